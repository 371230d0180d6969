"""U-Net kernels at the edges of their shapes, against the oracle.

The weight gradients walk segments of an x line (up to 64 nodes, a multiple of 16 in
shared memory) and the convolutions tiles of 16 or 32 nodes: lines just below, at and
above those lengths, lines of one node on the coarse grids, odd grids.  The check and its
tolerances are those of test_gpu_unet.py.
"""
import pytest

import test_gpu_unet as T
import workloads as W

pytestmark = pytest.mark.gpu

P, D = W.PERIODIC, W.DIRICHLET
MESHES = [(1, [64, 1, 1, 3], [P]), (1, [65, 1, 1, 5], [P]), (1, [129, 1, 1, 4], [P]), (1, [2, 1, 1, 37], [D]),
          (2, [17, 3, 1, 5], [P, P]), (2, [5, 33, 1, 2], [D, P]), (3, [18, 3, 2, 3], [D, P, P])]


@pytest.mark.parametrize("d,n_el,bc", MESHES)
def test_forward_and_gradients_at_shape_edges(d, n_el, bc):
    T.test_unet_forward_and_gradients_match_oracle("", lambda: W.random_mesh(d, n_el, bc, seed=9, with_potential=False))

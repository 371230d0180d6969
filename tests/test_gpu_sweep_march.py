"""Crank-Nicolson sweep at the edges of its kernels' shapes, against the oracle.

The banded march shares a system of x nodes between 8 to 256 lanes, two nodes each: the
numbers of x nodes here are the last of one lane count and the first of the next, one
node, and the longest axis taken; 3+1 meshes pair two systems per frequency.  Time steps
above half the x spacing take the refined form.  The plane FFTs take periodic lengths of
every radix (16, 8, 4, 2, 3, 5, other primes) and a plane too large for two buffers.

Tolerance as in test_gpu_precond.py: eps32 x N_t x 10^2 gives rel. L2 <= 1e-4 and
max |dz| <= 1e-3 max |z|; a wrong neighbour, factor or twiddle gives O(1).
"""
import numpy as np
import pytest

import workloads as W
from _helpers import max_rel, oracle_mesh, rel_l2

pytestmark = pytest.mark.gpu
P, D = W.PERIODIC, W.DIRICHLET


def _check(d, n_el, bc, with_v):
    import torch
    from oracle import operator as OOP, precond as PC
    from paper_2103_14588_gb300 import binding as B
    w = W.random_mesh(d, n_el, bc, seed=7, with_potential=False)
    if with_v:
        vx = np.random.default_rng(3).uniform(-0.5, 1.5, n_el[0])
        w.V = np.tile(vx, (n_el[1] if d > 1 else 1) * (n_el[2] if d > 2 else 1))
    om = oracle_mesh(w)
    A, _ = OOP.split(om, OOP.assemble(om, w.m, w.V), w.psi0)
    Mc = PC.crank_nicolson_sweep(A.tocsr(), om.nt, om.n_spatial_nodes * om.nc)[0]
    v = W.random_complex(om.n_unknowns, 5).astype(np.complex64)
    ref = Mc(v.astype(np.complex128))
    with B.Mesh.from_workload(w) as mesh:
        vd = torch.from_numpy(v).cuda()
        zd = torch.full_like(vd, complex("nan+nanj"))
        B.dst_precond_apply(mesh.handle, B.DST_PRECOND_CN_SWEEP, vd, zd)
        got = zd.cpu().numpy()
    assert np.all(np.isfinite(got))
    assert rel_l2(got, ref) <= 1e-4, rel_l2(got, ref)
    assert max_rel(got, ref) <= 1e-3


@pytest.mark.parametrize("nodes,nt", [(1, 3), (2, 3), (15, 12), (16, 3), (17, 9), (32, 30), (33, 3), (64, 40), (65, 3),
                                      (128, 50), (129, 3), (256, 4), (257, 3), (365, 3)])
def test_march_lane_counts(nodes, nt):
    _check(1, [nodes + 1, 1, 1, nt], [D], True)


@pytest.mark.parametrize("d,n_el,with_v", [(2, [18, 9, 1, 5], True), (2, [35, 3, 1, 30], False), (2, [66, 2, 1, 3], True),
                                           (3, [4, 1, 2, 3], True), (3, [18, 3, 3, 12], True), (3, [34, 2, 5, 3], False),
                                           (3, [67, 3, 1, 3], True)])
def test_march_frequencies_and_pairs(d, n_el, with_v):
    _check(d, n_el, [D, P, P][:d], with_v)


@pytest.mark.parametrize("n_el", [[16, 32, 1, 3], [48, 6, 1, 3], [96, 5, 1, 3], [45, 14, 1, 3], [7, 11, 1, 3], [29, 13, 1, 3],
                                  [1, 9, 1, 3], [116, 114, 1, 3]])
def test_fft_radices_and_layouts(n_el):
    _check(2, n_el, [P, P], False)

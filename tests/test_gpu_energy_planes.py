"""Energy per layer where the FFT's planes change form, against the oracle's numpy FFT.

1+1 meshes take x lines of several layers as a plane, as many as divide the layers, and the second
pass of a 3+1 mesh z lines that divide a layer's (y, x) plane: up to 32 lines and 1024 nodes,
while 304 CTAs are left.  Meshes on either side of those: lines by 32, by less, alone, z axes of
one node and of more than 512, odd and prime lengths, planes of few nodes (radices of four
in place of 16).  Tolerance as in test_gpu_observables.py: 1e-11 of the largest |E|.
"""
import numpy as np
import pytest

import workloads as W
from _helpers import oracle_mesh

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("d,n_el", [(1, [24, 1, 1, 310]), (1, [16, 1, 1, 4896]), (1, [512, 1, 1, 305]),
                                    (1, [512, 1, 1, 306]), (1, [37, 1, 1, 331]), (2, [12, 10, 1, 305]), (2, [7, 5, 1, 304]), (3, [8, 8, 8, 20]),
                                    (3, [12, 10, 9, 16]), (3, [5, 7, 11, 31]), (3, [11, 13, 6, 60]), (3, [4, 4, 1, 40]),
                                    (3, [2, 3, 520, 3]), (3, [32, 3, 32, 7]), (3, [1, 1, 12, 200])])
def test_energy(d, n_el):
    import torch
    from oracle import observables as OB
    from paper_2103_14588_gb300 import binding as B
    w = W.random_mesh(d, n_el, [W.PERIODIC] * d, seed=d + 70, with_potential=False)
    om = oracle_mesh(w)
    psi = W.random_complex(om.n_unknowns, 8).reshape(om.unknown_shape)
    ref = OB.energy(om, psi, w.m)
    with B.Mesh.from_workload(w) as mesh:
        out = torch.full((om.nt,), float("nan"), dtype=torch.float64, device="cuda")
        B.dst_energy(mesh.handle, torch.from_numpy(psi).cuda(), out)
        got = out.cpu().numpy()
    assert np.all(np.abs(got - ref) <= 1e-11 * np.abs(ref).max()), np.abs(got - ref).max() / np.abs(ref).max()

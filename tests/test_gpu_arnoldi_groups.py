"""FP64 Arnoldi projection and update over every group size of basis vectors.

The kernels take eight vectors at a time and the rest in exact groups of 1 to 7, slices of
256 entries per CTA up to 608 CTAs, and sum few partials in the kernel.  Error bounds of
sums of n products in FP64 whatever their order: |h_j| (n + 8) eps ||v_j|| ||w||; update
(4 nvec + 8) eps (|w_i| + sum_j |V_ji| |h_j|) per entry; ||w||^2 relative (n + 8) eps.
"""
import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu
EPS = np.finfo(np.float64).eps


@pytest.mark.parametrize("n", [1, 255, 257, 4099, 155649])
@pytest.mark.parametrize("nvec", [1, 2, 3, 4, 5, 6, 7, 8, 9, 15, 23, 30, 64])
def test_projection_and_update(n, nvec):
    import torch
    from paper_2103_14588_gb300 import binding as B
    V = W.random_complex(n * nvec, 1).reshape(nvec, n)
    w = W.random_complex(n, 2)
    Vd, wd = torch.from_numpy(V).cuda(), torch.from_numpy(w).cuda()
    h = torch.empty(nvec, dtype=torch.complex128, device="cuda")
    nrm2 = torch.empty(1, dtype=torch.float64, device="cuda")
    B.dst_arnoldi_project(n, nvec, Vd, wd, h)
    ref = V.conj() @ w
    hh = h.cpu().numpy()
    assert np.all(np.abs(hh - ref) <= (n + 8) * EPS * np.linalg.norm(V, axis=1) * np.linalg.norm(w))
    B.dst_arnoldi_update(n, nvec, Vd, h, wd, nrm2)
    got = wd.cpu().numpy()
    assert np.all(np.abs(got - (w - hh @ V)) <= (4 * nvec + 8) * EPS * (np.abs(w) + np.abs(hh) @ np.abs(V)))
    true = np.vdot(got, got).real
    assert abs(nrm2.item() - true) <= (n + 8) * EPS * true

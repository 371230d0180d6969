"""The FP64 Gram-Schmidt step of a solve: sums finished in the kernel, gated second pass.

Up to 2048 partial sums the last CTA of the projection adds them up (and those of ||w||^2),
above that a second kernel; the update's norm is always summed by its last CTA.  Both passes
of a step count on the same counters, which every kernel leaves at zero.  The numbers of
CTAs (n / 256, 608 at most) and vectors here lie on both sides of 2048.  Error bounds as in
test_gpu_arnoldi_groups.py: |h_j| (n + 8) eps ||v_j|| ||w||, update (4 nvec + 8) eps per entry
and pass, ||w||^2 relative (n + 8) eps.
"""
import ctypes

import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu
EPS = np.finfo(np.float64).eps


@pytest.mark.parametrize("n,nvec", [(1, 1), (300, 5), (4099, 30), (8192, 64), (8193, 63), (17408, 30), (17700, 30),
                                    (155649, 3), (155649, 4), (200000, 9)])
@pytest.mark.parametrize("kind", ["random", "mixture", "span"])
def test_step(n, nvec, kind):
    import torch
    from paper_2103_14588_gb300 import binding as B
    V = W.random_complex(n * nvec, 1).reshape(nvec, n)
    V /= np.linalg.norm(V, axis=1)[:, None] * np.sqrt(nvec)
    w = W.random_complex(n, 2)
    if kind == "span":              # orthonormal rows, w their sum and little else: the first pass leaves next to nothing
        V = np.linalg.qr(V.T)[0].T.copy()
        w = np.sum(V, axis=0) + 1e-3 * w / np.linalg.norm(w)
    elif kind == "mixture":         # a part of w in the span: either side of the second pass's limit
        w = np.sum(V, axis=0) * nvec + 1e-3 * w / np.linalg.norm(w)
    elif n == 1:
        w = w * 0 + 1.0
        V = V * 0.1
    Vd, wd = torch.from_numpy(V).cuda(), torch.from_numpy(w).cuda()
    h = torch.full((2 * nvec,), complex("nan+nanj"), dtype=torch.complex128, device="cuda")
    rec = torch.full((8,), float("nan"), dtype=torch.float64, device="cuda")
    st = torch.cuda.current_stream().cuda_stream
    p = lambda t: ctypes.c_void_p(t.data_ptr())          # noqa: E731
    assert B.library().dst_testing_fp64_step(n, nvec, p(Vd), p(wd), p(h), p(rec), st) == 0
    hh, r, got = h.cpu().numpy(), rec.cpu().numpy(), wd.cpu().numpy()
    vn, wn = np.linalg.norm(V, axis=1), np.linalg.norm(w)
    h1, h2 = hh[:nvec], hh[nvec:]
    assert np.all(np.abs(h1 - V.conj() @ w) <= (n + 8) * EPS * vn * wn)
    assert abs(r[3] - wn * wn) <= (n + 8) * EPS * wn * wn
    w1 = w - h1 @ V
    ran = np.vdot(w1, w1).real < 0.5 * r[3]
    assert r[6] == (1.0 if ran else 0.0)
    tol = (4 * nvec + 8) * EPS * (np.abs(w) + np.abs(h1) @ np.abs(V))
    if ran:
        slack = vn * np.linalg.norm(tol)                  # h2 sees the rounding of the first update
        assert np.all(np.abs(h2 - V.conj() @ w1) <= (n + 8) * EPS * vn * np.linalg.norm(w1) + slack)
        assert np.all(np.abs(got - (w1 - h2 @ V)) <= 2 * tol)
    else:
        assert not h2.any()
        assert np.all(np.abs(got - w1) <= tol)
    true = np.vdot(got, got).real
    assert abs(r[0] - true) <= (n + 8) * EPS * true
    assert ran or kind != "span"

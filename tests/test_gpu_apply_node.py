"""Operator apply where the launch chooses between its kernels.

Small meshes against the oracle over what the lane-per-number kernel takes: every kind of
axis (an open axis's end elements are missing), one and two elements along an axis, no
potential, an x-only and a general one, one layer and layer counts around a chunk.  Its sums
differ from the oracle's only in their order: FP64 rel. L2 <= 1e-14 (up to 81 terms of
alternating signs, ~20 eps), FP32 <= 2e-6 (~20 eps).

Meshes on both sides of 2^19 unknowns, where the tiled kernels take over: the FP32 apply
against the FP64 one of the same mesh (<= 2e-6), and the FP64 apply of a vector against the sum
of the applies of its two halves (linearity, <= 1e-14), whichever kernels they take.
"""
import numpy as np
import pytest

import workloads as W
from _helpers import oracle_mesh, rel_l2

pytestmark = pytest.mark.gpu
P, O, D = W.PERIODIC, W.OPEN, W.DIRICHLET

SMALL = [(1, [1, 1, 1, 1], [P]), (1, [2, 1, 1, 2], [P]), (1, [1, 1, 1, 3], [O]), (1, [33, 1, 1, 65], [O]),
         (1, [2, 1, 1, 5], [D]), (2, [1, 2, 1, 3], [P, P]), (2, [3, 1, 1, 2], [O, O]), (2, [17, 9, 1, 7], [D, O]),
         (2, [5, 6, 1, 33], [P, D]), (3, [1, 1, 1, 2], [P, P, P]), (3, [2, 1, 3, 3], [O, O, P]),
         (3, [5, 4, 3, 4], [D, P, O]), (3, [3, 6, 2, 9], [O, D, D])]


def _potential(w, kind, d, n_el):
    if kind == "none":
        w.V = None
    elif kind == "x":
        w.V = np.tile(np.random.default_rng(2).uniform(-1, 2, n_el[0]), (n_el[1] if d > 1 else 1) * (n_el[2] if d > 2 else 1))


def _apply(B, torch, mesh, x, prec):
    xd = torch.from_numpy(x).cuda()
    yd = torch.full_like(xd, complex("nan+nanj"))
    B.dst_apply_operator(mesh.handle, prec, xd, yd)
    return yd.cpu().numpy()


@pytest.mark.parametrize("kind", ["none", "x", "general"])
@pytest.mark.parametrize("d,n_el,bc", SMALL)
def test_small_meshes_match_oracle(d, n_el, bc, kind):
    import torch
    from oracle import operator as OOP
    from paper_2103_14588_gb300 import binding as B
    w = W.random_mesh(d, n_el, bc, seed=31)
    _potential(w, kind, d, n_el)
    om = oracle_mesh(w)
    A, _ = OOP.split(om, OOP.assemble(om, w.m, w.V), w.psi0)
    x = W.random_complex(om.n_unknowns, 4)
    ref = A @ x
    with B.Mesh.from_workload(w) as mesh:
        assert rel_l2(_apply(B, torch, mesh, x, B.DST_FP64), ref) <= 1e-14
        assert rel_l2(_apply(B, torch, mesh, x.astype(np.complex64), B.DST_FP32), ref) <= 2e-6


LARGE = [(1, [509, 1, 1, 515], [P]), (1, [513, 1, 1, 512], [P]), (1, [514, 1, 1, 513], [D]), (1, [600, 1, 1, 500], [O]),
         (2, [65, 63, 1, 64], [P, P]), (2, [67, 65, 1, 61], [D, P]), (2, [70, 61, 1, 70], [P, O]),
         (3, [20, 19, 18, 17], [D, P, P]), (3, [21, 19, 18, 20], [D, P, P]), (3, [33, 29, 31, 37], [P, D, P])]


@pytest.mark.parametrize("kind", ["none", "x", "general"])
@pytest.mark.parametrize("d,n_el,bc", LARGE)
def test_both_sides_of_the_tiled_kernels(d, n_el, bc, kind):
    import torch
    from paper_2103_14588_gb300 import binding as B
    w = W.random_mesh(d, n_el, bc, seed=32)
    _potential(w, kind, d, n_el)
    with B.Mesh.from_workload(w) as mesh:
        x = W.random_complex(mesh.n_unknowns, 6).astype(np.complex64).astype(np.complex128)
        half = np.arange(x.size) % 3 == 0
        y = _apply(B, torch, mesh, x, B.DST_FP64)
        y2 = _apply(B, torch, mesh, np.where(half, x, 0), B.DST_FP64) + _apply(B, torch, mesh, np.where(half, 0, x), B.DST_FP64)
        assert np.all(np.isfinite(y)) and rel_l2(y2, y) <= 1e-14
        for v in range(B.dst_get_apply_variant(mesh.handle, B.DST_FP32)[1]):
            B.dst_set_apply_variant(mesh.handle, B.DST_FP32, v)
            assert rel_l2(_apply(B, torch, mesh, x.astype(np.complex64), B.DST_FP32), y) <= 2e-6

"""Rounding of the Crank-Nicolson sweep, against the oracle's FP64 sweep.

A layer's solve in FP32 (u = 2^-24) adds a few u to a solution of steady norm, and the
march carries those errors on without damping: after N_t layers about 2 u sqrt(N_t) of
them, and the plane FFTs another 2 u or so.  48 layers: 9e-7 from the march, 1e-6 in all.
Time steps of many spacings, heavy masses and high potentials must not add to that: what a
step forms in FP32 must be no larger than the solution itself.
"""
import numpy as np
import pytest

import workloads as W
from _helpers import oracle_mesh, rel_l2

pytestmark = pytest.mark.gpu
P, D = W.PERIODIC, W.DIRICHLET
H, NT = 0.25, 48


def _error(d, n, bc, ratio, m, V, hy=1.0):
    """Relative L2 error at spacing H (H hy along y, z) and time step ratio H."""
    import torch
    from oracle import operator as OOP, precond as PC
    from paper_2103_14588_gb300 import binding as B
    n_el = [n] + [n if k < d else 1 for k in (1, 2)] + [NT]
    w = W.random_mesh(d, n_el, bc, seed=7, with_potential=False)
    w.lo, w.hi = [0.0] * 4, [n * H, n * H * hy, n * H * hy, NT * ratio * H]
    w.m, w.V = m, None if V is None else np.broadcast_to(V, (n_el[2], n_el[1], n_el[0])).ravel().copy()
    om = oracle_mesh(w)
    A, _ = OOP.split(om, OOP.assemble(om, w.m, w.V), w.psi0)
    exact = PC.crank_nicolson_sweep(A.tocsr(), om.nt, om.n_spatial_nodes * om.nc)[0]
    errors = []
    with B.Mesh.from_workload(w) as mesh:
        for seed in (1, 2):
            v = W.random_complex(om.n_unknowns, seed).astype(np.complex64)
            vd = torch.from_numpy(v).cuda()
            zd = torch.empty_like(vd)
            B.dst_precond_apply(mesh.handle, B.DST_PRECOND_CN_SWEEP, vd, zd)
            errors.append(rel_l2(zd.cpu().numpy(), exact(v.astype(np.complex128))))
    return max(errors)


@pytest.mark.parametrize("d,n", [(1, 64), (2, 12)])
@pytest.mark.parametrize("ratio,m,V", [(0.25, 1.0, 3.0), (0.25, 1.0, 1000.0), (1.0, 1.0, 1000.0), (2.0, 30.0, None), (4.0, 1.0, 3.0),
                                       (10.0, 1.0, 3.0), (10.0, 0.0, None), (40.0, 1.0, 3.0)])
def test_periodic(d, n, ratio, m, V):
    assert _error(d, n, [P] * d, ratio, m, V) <= 1e-6


# An elimination along x in order, solve by solve, is within 1.6e-6 on these meshes (the
# chain of 2 n_x products per layer in place of the two solves' worth above).
@pytest.mark.parametrize("d,n,ratio,m,V,hy", [(1, 64, 0.45, 30.0, None, 1.0), (1, 64, 0.25, 1.0, 100.0, 1.0),
                                              (2, 16, 0.45, 30.0, None, 10.0), (2, 16, 0.25, 1.0, 100.0, 0.1),
                                              (2, 16, 0.1, 0.0, None, 0.03), (3, 8, 0.25, 0.0, None, 0.1),
                                              (3, 8, 0.25, 1.0, 1000.0, 1.0), (1, 64, 4.0, 1.1, 2.5, 1.0)])
def test_dirichlet(d, n, ratio, m, V, hy):
    step = None if V is None else np.where(np.arange(n) >= n // 2, V, 0.0)
    assert _error(d, n, [D, P, P][:d], ratio, m, step, hy) <= 1.6e-6

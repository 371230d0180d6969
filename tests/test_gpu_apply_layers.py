"""Operator applies on meshes of very many time layers.

A tile shape has more chunks there than a grid's y extent takes (65535).  Every shape computes
an output from the same neighbours, so FP64 agrees bit for bit with the default shape, and FP32
agrees with the FP64 apply to 20 eps32: an output is a sum of at most 27 products whose
partial sums stay within a few times the largest (rel. L2).
"""
import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu
P, D = W.PERIODIC, W.DIRICHLET


@pytest.mark.parametrize("d,n_el,bc", [(1, [2, 1, 1, 524289], [P]), (1, [4, 1, 1, 524300], [D]), (2, [2, 2, 1, 262150], [P, D]),
                                       (2, [3, 2, 1, 524290], [P, P])])
def test_many_layers(d, n_el, bc):
    import torch
    from paper_2103_14588_gb300 import binding as B
    w = W.random_mesh(d, n_el, bc, seed=3, with_potential=False)
    with B.Mesh.from_workload(w) as mesh:
        assert mesh.n_unknowns >= 1 << 19
        x = torch.from_numpy(W.random_complex(mesh.n_unknowns, 4).astype(np.complex64)).cuda()
        x64 = x.to(torch.complex128)
        ref = torch.empty_like(x64)
        B.dst_apply_operator(mesh.handle, B.DST_FP64, x64, ref)
        for v in range(B.dst_get_apply_variant(mesh.handle, B.DST_FP32)[1]):
            B.dst_set_apply_variant(mesh.handle, B.DST_FP32, v)
            B.dst_set_apply_variant(mesh.handle, B.DST_FP64, v)
            y, y64 = torch.full_like(x, complex("nan+nanj")), torch.full_like(x64, complex("nan+nanj"))
            B.dst_apply_operator(mesh.handle, B.DST_FP64, x64, y64)
            assert torch.equal(torch.view_as_real(y64), torch.view_as_real(ref))
            B.dst_apply_operator(mesh.handle, B.DST_FP32, x, y)
            err = torch.linalg.vector_norm(y - ref) / torch.linalg.vector_norm(ref)
            assert err.item() <= 20 * np.finfo(np.float32).eps
        B.dst_tune_apply(mesh.handle)

"""FP32 vectors that start at an odd entry of their buffer (8-byte, not 16-byte aligned).

The preconditioners and the U-Net take such vectors; the kernels that load 16 bytes at a
time must not be handed them.  The same call on aligned buffers is the reference: the
sweep may take another kernel instance (rel. L2 <= 1e-4, the tolerance against the oracle
in test_gpu_precond.py; a shifted entry gives O(1)), the U-Net's values are the same.
"""
import numpy as np
import pytest

import workloads as W
from _helpers import rel_l2

pytestmark = pytest.mark.gpu
P, D = W.PERIODIC, W.DIRICHLET


def _odd(t):
    import torch
    buf = torch.full((t.numel() + 1,), complex("nan+nanj"), dtype=t.dtype, device="cuda")
    buf[1:].copy_(t)
    assert buf[1:].data_ptr() % 16 == 8
    return buf[1:]


@pytest.mark.parametrize("d,n_el,bc", [(1, [20, 1, 1, 9], [D]), (1, [21, 1, 1, 6], [P]), (2, [18, 9, 1, 5], [D, P]),
                                       (2, [12, 10, 1, 5], [P, P]), (3, [18, 5, 4, 4], [D, P, P])])
@pytest.mark.parametrize("learned", [False, True])
def test_preconditioner(d, n_el, bc, learned):
    import torch
    from paper_2103_14588_gb300 import binding as B
    w = W.random_mesh(d, n_el, bc, seed=7, with_potential=False)
    with B.Mesh.from_workload(w) as mesh:
        net = B.UNet(mesh.handle)
        net.set_params((0.1 * np.random.default_rng(2).standard_normal(net.num_params)).astype(np.float32))
        kind = B.DST_PRECOND_CN_SWEEP
        if learned:
            B.dst_set_learned_precond(mesh.handle, net)
            kind = B.DST_PRECOND_CN_LEARNED
        v = torch.from_numpy(W.random_complex(mesh.n_unknowns, 5).astype(np.complex64)).cuda()
        ref = torch.empty_like(v)
        B.dst_precond_apply(mesh.handle, kind, v, ref)
        for vi, zi in ((_odd(v), torch.empty_like(v)), (v, _odd(v)), (_odd(v), _odd(v))):
            zi.fill_(complex("nan+nanj"))
            B.dst_precond_apply(mesh.handle, kind, vi, zi)
            assert rel_l2(zi.cpu().numpy(), ref.cpu().numpy()) <= 1e-4
        B.dst_set_learned_precond(mesh.handle, None)
        net.close()


def test_unet():
    import torch
    from paper_2103_14588_gb300 import binding as B
    w = W.random_mesh(2, [9, 7, 1, 6], [P, P], seed=4, with_potential=False)
    with B.Mesh.from_workload(w) as mesh:
        net = B.UNet(mesh.handle)
        net.set_params((0.1 * np.random.default_rng(2).standard_normal(net.num_params)).astype(np.float32))
        x, t = (torch.from_numpy(W.random_complex(mesh.n_unknowns, k).astype(np.complex64)).cuda() for k in (5, 6))
        ref = torch.empty_like(x)
        net.forward(x, ref)
        y = _odd(x)
        net.forward(_odd(x), y)
        assert torch.equal(y, ref)
        # a result at a 4-byte boundary
        raw = torch.zeros(2 * x.numel() + 1, dtype=torch.float32, device="cuda")
        net.forward(x.data_ptr(), raw[1:].data_ptr(), stream=torch.cuda.current_stream().cuda_stream)
        assert torch.equal(raw[1:], torch.view_as_real(ref).reshape(-1))
        loss, grad = net.loss_grad(x, t)
        loss2, grad2 = net.loss_grad(_odd(x), _odd(t))
        assert loss == loss2 and np.array_equal(grad, grad2)
        net.close()

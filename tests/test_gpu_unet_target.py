"""The U-Net's training target at any float of its buffer (4-byte aligned): the same loss and
gradients as from an aligned one, whose values it holds (the same arithmetic, bit for bit)."""
import ctypes

import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu
P = W.PERIODIC


@pytest.mark.parametrize("d,n_el", [(1, [21, 1, 1, 6]), (2, [9, 7, 1, 6]), (3, [5, 4, 3, 4])])
@pytest.mark.parametrize("offset", [1, 2, 3])
def test_target_at_any_float(d, n_el, offset):
    import torch
    from paper_2103_14588_gb300 import binding as B
    w = W.random_mesh(d, n_el, [P] * d, seed=4, with_potential=False)
    with B.Mesh.from_workload(w) as mesh:
        net = B.UNet(mesh.handle)
        net.set_params((0.1 * np.random.default_rng(2).standard_normal(net.num_params)).astype(np.float32))
        x, t = (torch.from_numpy(W.random_complex(mesh.n_unknowns, k).astype(np.complex64)).cuda() for k in (5, 6))
        loss, grad = net.loss_grad(x, t)
        raw = torch.full((2 * t.numel() + offset,), float("nan"), dtype=torch.float32, device="cuda")
        raw[offset:].copy_(torch.view_as_real(t).reshape(-1))
        got, g = ctypes.c_double(), np.empty_like(grad)
        assert B.library().dst_unet_loss_grad(net.handle, x.data_ptr(), raw[offset:].data_ptr(), ctypes.byref(got),
                                              g.ctypes.data, torch.cuda.current_stream().cuda_stream) == 0
        assert got.value == loss and np.array_equal(g, grad)
        net.close()

"""Sweeps and U-Net gradients of meshes of several sizes from two threads at once.

The kernels' dynamic shared memory differs between the meshes while its limit belongs to
the function, so one thread's smaller mesh must not lower it under the other's launch.
Every call gives what it gives alone (the kernels sum in a fixed order).
"""
import threading

import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu
P, D = W.PERIODIC, W.DIRICHLET


def _both(jobs):
    errors = []

    def guard(job):
        try:
            job()
        except Exception as e:                              # reported by the main thread
            errors.append(repr(e))
    threads = [threading.Thread(target=guard, args=(j,)) for j in jobs]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not errors, errors


def test_sweeps_of_two_sizes():
    import torch
    from paper_2103_14588_gb300 import binding as B
    meshes = [B.Mesh.from_workload(W.random_mesh(3, n, [D, P, P], seed=7, with_potential=False)) for n in
              ([18, 4, 4, 4], [32, 4, 4, 4])]                # both 16 lanes per system

    def job(mesh):
        def run():
            stream = torch.cuda.Stream()
            with torch.cuda.stream(stream):
                v = torch.from_numpy(W.random_complex(mesh.n_unknowns, 5).astype(np.complex64)).cuda()
                ref, z = torch.empty_like(v), torch.empty_like(v)
                for i in range(200):
                    B.dst_precond_apply(mesh.handle, B.DST_PRECOND_CN_SWEEP, v, ref if i == 0 else z)
                stream.synchronize()
                assert torch.equal(z, ref)
        return run
    _both([job(m) for m in meshes])


def test_unet_gradients_of_two_sizes():
    import torch
    from paper_2103_14588_gb300 import binding as B
    meshes = [B.Mesh.from_workload(W.random_mesh(2, n, [P, P], seed=7, with_potential=False)) for n in
              ([6, 6, 1, 4], [60, 6, 1, 4])]

    def job(mesh):
        def run():
            net = B.UNet(mesh.handle)
            net.set_params((0.1 * np.random.default_rng(2).standard_normal(net.num_params)).astype(np.float32))
            stream = torch.cuda.Stream()
            with torch.cuda.stream(stream):
                x, t = (torch.from_numpy(W.random_complex(mesh.n_unknowns, k).astype(np.complex64)).cuda() for k in (5, 6))
                loss, grad = net.loss_grad(x, t)
                for _ in range(50):
                    again, g = net.loss_grad(x, t)
                    assert again == loss and np.array_equal(g, grad)
            net.close()
        return run
    _both([job(m) for m in meshes])

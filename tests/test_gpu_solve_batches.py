"""Steps that an FP64 solve enqueues past the one that meets its tolerance.

A batch between two host synchronisations is no longer than what the call has taken before it
(half of that from 2^16 unknowns on), two steps at first: of all enqueued steps at
least half (two thirds) count.  The enqueued steps are the operator applies but the
residuals before and after the cycle; ending tolerances are taken from the solve's start.
"""
import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,nt", [(24, 24), (64, 64), (256, 200), (360, 300)])
def test_few_steps_run_in_vain(n, nt):
    import torch
    from paper_2103_14588_gb300 import binding as B
    w = W.random_mesh(1, [n, 1, 1, nt], [W.PERIODIC], seed=5, with_potential=False)
    large = 2 * n * nt >= 1 << 16
    with B.Mesh.from_workload(w) as mesh:
        start = torch.from_numpy(W.random_complex(mesh.n_unknowns, 6)).cuda()
        psi = start.clone()
        opts = {"restart": 30, "max_iters": 0, "rtol": 1e-12, "use_initial_guess": 1}
        r = B.dst_solve(mesh.handle, opts, psi)["rel_resid_true"]
        seen = set()
        for f in (0.95, 0.8, 0.6, 0.4, 0.3, 0.2, 0.15):
            psi.copy_(start)
            st = B.dst_solve(mesh.handle, dict(opts, max_iters=1000, rtol=r * f), psi)
            assert st["status"] == 0
            if st["restarts"] != 1:
                continue
            seen.add(st["iters"])
            steps = st["kernel_launches"][0] - 2
            assert steps <= (max(2, st["iters"] * 3 // 2 + 1) if large else max(2, 2 * st["iters"])), (st["iters"], steps)
        assert seen

"""The tensor search of the element-wise kernels against the oracle, at table
sizes on either side of what one round of it probes (32 entries) and two
(1024), with runs of empty tensors at both ends and in the middle."""
from __future__ import annotations

import numpy as np
import pytest
import torch

import oracle
from paper_2606_30634_gb300 import dpo, synth
from parity_util import TOL_ONE_STEP, rel_err

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [1, 2, 32, 33, 1024, 1025, 2100])
def test_clipped_step_over_many_tensors(cuda_device, n):
    numels = [0 if i % 11 == 0 and n > 2 else 1 + (37 * i) % 61 for i in range(n)]
    total, seed = sum(numels), 0x7AB + n
    offs = np.concatenate([[0], np.cumsum(numels)])
    x0 = synth.host_normal(seed, synth.STREAM_INIT, 0, 0, total, 0.02)
    g = synth.host_normal(seed, synth.STREAM_GRAD, 1, 0, total, 1e-3, synth.F32)
    norm = float(np.linalg.norm(g.astype(np.float64)))
    opt = dpo.DelayedAdamW(numels, param_dtype=dpo.DPO_F32, grad_dtype=dpo.DPO_F32, ef=True,
                           max_grad_norm=0.5 * norm, device=cuda_device, x0=torch.from_numpy(x0))
    try:
        for i, k in enumerate(numels):
            if k:
                opt.grads(i).copy_(torch.from_numpy(g[offs[i]:offs[i + 1]]))
        opt.step()
        hp = oracle.HParams(ef_lambda=1.0, max_grad_norm=0.5 * norm).as_f32()
        ref = oracle.DelayedOptimizer([x0.astype(np.float64)], hp, ef=True, x_store=oracle.F32,
                                      stash_store=oracle.F32)
        ref.step(g.astype(np.float64), tag=ref.read_weights()[1])
        cat = lambda a: torch.cat([opt.view(a, i) for i in range(n)]).cpu().numpy()
        assert rel_err(cat(opt.master), ref.x) <= TOL_ONE_STEP
        assert rel_err(cat(opt.m), ref.m) <= TOL_ONE_STEP
        assert dpo.dpo_get_flags(opt.ctx)[1] == pytest.approx(norm, rel=1e-6)
    finally:
        opt.close()


def test_empty_tensors_do_not_change_the_launch(cuda_device):
    """A clipped step of more than one wave is launched by how many tensors a
    thread passes over; empty ones are not passed over."""
    def ctas(numels):
        opt = dpo.DelayedAdamW(numels, ef=True, stash_dtype=dpo.DPO_BF16, max_grad_norm=1.0,
                               device=cuda_device)
        try:
            return dpo.dpo_launch_config(opt.ctx)[0]
        finally:
            opt.close()

    n = 1 << 20
    one = ctas([n])
    assert ctas([n] + [0] * 200) == one == ctas([n // 63] * 63)
    assert ctas([n // 64] * 64) == n // 8 // 128 > one

"""The tensor search of the element-wise kernels against the oracle, at table
sizes on either side of what one round of it probes (32 entries) and two
(1024), with runs of empty tensors at both ends and in the middle; and the
launches by set size: one packet per thread or persistent CTAs for the step,
one to eight packets per thread for the norm pass."""
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


@pytest.mark.parametrize("dtype", [dpo.DPO_F32, dpo.DPO_BF16])
@pytest.mark.parametrize("pkts", [32768, 32769, 65537, 131073, 262145])
def test_norm_pass_at_each_width(cuda_device, pkts, dtype):
    """Sets on either side of where a thread of the norm pass takes 1, 2, 4 and
    (bf16) 8 packets per round, three ragged tensors: the norm of the clipped step,
    and dpo_grad_sqnorm's sum, against fp64."""
    n = 8 * pkts - 3
    numels = [n // 3, 11, n - n // 3 - 11]
    opt = dpo.DelayedAdamW(numels, grad_dtype=dtype, max_grad_norm=0.5, device=cuda_device)
    try:
        gen = torch.Generator(device=cuda_device).manual_seed(pkts)
        for i, k in enumerate(numels):
            opt.grads(i).copy_(torch.randn(k, device=cuda_device, generator=gen).mul_(1e-3))
        want = sum(float(opt.grads(i).double().square().sum()) for i in range(3))
        acc = torch.zeros(1, dtype=torch.float64, device=cuda_device)
        opt.grad_sqnorm(acc)
        opt.step()
        # each packet's squares in fp32: 2^-24 each, and as much per Kahan sum
        assert acc.item() == pytest.approx(want, rel=1e-6)
        _, norm, clip = dpo.dpo_get_flags(opt.ctx)
        assert norm == pytest.approx(want ** 0.5, rel=1e-6)
        assert clip == pytest.approx(0.5 / (want ** 0.5 + 1e-6), rel=1e-6)
    finally:
        opt.close()


def test_one_packet_per_thread_equals_persistent_ctas(cuda_device):
    """A flat set at the last size of one packet per thread (ten CTAs' packets per
    SM) and one element past it, which persistent CTAs take: the shared elements
    end up the same, bit for bit, over three calls."""
    sms = torch.cuda.get_device_properties(cuda_device).multi_processor_count
    n = 10 * sms * 128 * 8

    def run(numel, ctas):
        gen = torch.Generator(device=cuda_device).manual_seed(3)
        x0 = torch.randn(n + 1, device=cuda_device, generator=gen)[:numel]
        opt = dpo.DelayedAdamW([numel], ef=True, stash_dtype=dpo.DPO_BF16, x0=x0,
                               device=cuda_device)
        try:
            assert dpo.dpo_launch_config(opt.ctx)[0] == ctas
            for _ in range(3):
                opt.grads(0).copy_(torch.randn(n + 1, device=cuda_device,
                                               generator=gen)[:numel].mul_(1e-3))
                opt.step()
            torch.cuda.synchronize()
            return [opt.view(a, 0)[:n].clone() for a in (opt.master, opt.m, opt.v, opt.ef,
                                                         opt.stash, opt.param)]
        finally:
            opt.close()

    for a, b in zip(run(n, 10 * sms), run(n + 1, 3 * sms)):
        assert torch.equal(a, b)

"""dpo_grad_norm_noalloc at the sizes where its chunking changes: empty, one
element, one chunk and one past it (a round of a CTA's loads: 8192 fp32 or
16384 bf16 elements), many chunks with a ragged last one; twice in a row, a
larger buffer between, so no sum of another call is read."""
from __future__ import annotations

import pytest
import torch

from paper_2606_30634_gb300 import dpo

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dtype", [dpo.DPO_F32, dpo.DPO_BF16])
@pytest.mark.parametrize("n", [0, 1, 8191, 8192, 8193, 16384, 16385, 999_999])
def test_norm_at_chunk_edges(cuda_device, n, dtype):
    tdt = torch.float32 if dtype == dpo.DPO_F32 else torch.bfloat16
    gen = torch.Generator(device=cuda_device).manual_seed(n)
    g = torch.randn(max(n, 1), device=cuda_device, generator=gen).mul_(1e-3).to(tdt)[:n]
    big = torch.ones(5_000_000, device=cuda_device, dtype=tdt)
    want = float(g.double().square().sum().sqrt())
    norm = torch.zeros(1, dtype=torch.float64, device=cuda_device)
    clip = torch.zeros(1, dtype=torch.float32, device=cuda_device)
    for _ in range(2):
        dpo.dpo_grad_norm_noalloc(big, big.numel(), dtype, 1.0, norm, clip)
        dpo.dpo_grad_norm_noalloc(g.data_ptr() if n else None, n, dtype, 0.25 * want, norm, clip)
        assert norm.item() == pytest.approx(want, rel=1e-6, abs=0)
        # min(1, max_norm / (norm + 1e-6)), and 1 for max_norm = 0
        assert clip.item() == pytest.approx(0.25 * want / (want + 1e-6) if n else 1.0, rel=1e-6)

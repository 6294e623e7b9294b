"""The line engine's panel loop: enough arrays that every resident CTA takes at
least three panels in every pass (the panel buffer reloaded, both barrier
phases, the row stores of the spectral direction's last pass awaited).  The
batch repeats five arrays, so every copy must have the bits of the first five,
and those must match the oracle."""
import numpy as np
import pytest

from paper_2609_28519_gb300 import inputs

pytestmark = pytest.mark.gpu

# lines of n points that an SM's resident CTAs hold at most, over the directions
RESIDENT = {64: 12 * 32, 128: 6 * 32, 192: 8 * 32, 256: 4 * 32, 384: 6 * 16, 512: 4 * 16, 768: 3 * 16, 1024: 3 * 16,
            1536: 3 * 8, 2048: 2 * 8, 4096: 8}


@pytest.mark.parametrize("n", sorted(RESIDENT))
def test_three_panels_per_cta_replicated(oracle_mod, cuda_dev, n):
    import torch
    from paper_2609_28519_gb300 import Plan
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    m = 192 if n <= 128 else 64
    for h, w in ((n, m), (m, n)):
        batch = 11 + max(-(-3 * sms * RESIDENT[w] // h), -(-3 * sms * RESIDENT[h] // w))
        base = inputs.uniform(23 * h + w, 5, h, w)
        lam = inputs.random_diagonal(n + m, h, w)
        plan = Plan(h, w, kind=15, path="fp32")
        plan.set_chunk_bytes(4 * batch * h * w)
        plan.set_spectral(lam)
        x = torch.from_numpy(base).to(cuda_dev).repeat(batch // 5 + 1, 1, 1)[:batch].contiguous()
        refs = {"forward": oracle_mod.forward(base, 0), "inverse": oracle_mod.inverse(base, 0),
                "roundtrip": base.astype(np.float64), "spectral": oracle_mod.spectral(base, lam)}
        idx = torch.arange(batch, device=cuda_dev) % 5
        for kind, ref in refs.items():
            y = plan.execute(kind, x)
            assert torch.equal(y, y[:5][idx]), (h, w, kind)
            scale = float(np.max(np.abs(lam))) if kind == "spectral" else 1.0
            got = oracle_mod.metrics(y[:5].cpu().numpy() / scale, ref / scale, base)
            assert got["nonfinite"] == 0 and got["e_rel_max"] <= oracle_mod.ERR_REL_TOL, (h, w, kind, got)
            assert got["max_abs_ratio_max"] <= oracle_mod.MAX_ABS_TOL, (h, w, kind, got)
        assert plan.device_status() == 0
        plan.close()

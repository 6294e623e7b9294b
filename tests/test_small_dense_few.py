"""The on-chip dense route's form for calls of few arrays: bit for bit the
products of the other form, around the count where the route changes over."""
import pytest

from paper_2609_28519_gb300 import inputs

pytestmark = pytest.mark.gpu


# output quads per warp 1, 2 and 4, one and two blocks of 16 terms, odd heights, one array per CTA and many
@pytest.mark.parametrize("h,w", [(1, 4), (3, 12), (7, 20), (9, 8), (24, 24), (31, 36), (33, 4), (40, 40), (63, 52)])
def test_few_arrays_equal_many(cuda_dev, h, w):
    import torch
    from paper_2609_28519_gb300 import Plan
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    plan = Plan(h, w, kind=15)
    plan.set_spectral(inputs.random_diagonal(h + w, h, w))
    over = 6144 * sms // (h * w) + 1  # the first count above the line
    x = torch.from_numpy(inputs.uniform(13 * h + w, 5, h, w)).to(cuda_dev)
    many = x.repeat(-(-over // 5), 1, 1)
    for kind in ("forward", "inverse", "roundtrip", "spectral"):
        y = plan.execute(kind, many)
        assert torch.equal(y, y[:5].repeat(len(many) // 5, 1, 1)), kind
        for count in (1, 2, sms - 1, sms + 1, 2 * sms + 3, over - 1):
            if count < over:
                assert torch.equal(plan.execute(kind, many[:count].contiguous()), y[:count]), (kind, count)

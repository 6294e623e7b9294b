"""Forms of one kernel that a call's sizes choose between, each against the
FP64 oracle with the parity bars of the other GPU tests (relative L2 <= 1e-6,
max-abs <= 4e-6 * scale)."""
import numpy as np
import pytest

from paper_2609_28519_gb300 import inputs

pytestmark = pytest.mark.gpu

KINDS = ["forward", "inverse", "roundtrip", "spectral"]


def _ref(o, kind, x, norm, lam):
    if kind == "forward":
        return o.forward(x, norm)
    if kind == "inverse":
        return o.inverse(x, norm)
    if kind == "spectral":
        return o.spectral(x, lam)
    return x.astype(np.float64)


def _check(o, got, kind, x, norm, lam, tag):
    ref = _ref(o, kind, x, norm, lam)
    if kind == "spectral":
        sc = float(np.max(np.abs(lam)))
        got, ref = got / sc, ref / sc
    m = o.metrics(got, ref, x, output_relative=(norm == 1 and kind in ("forward", "inverse")))
    assert m["nonfinite"] == 0, tag
    assert m["e_rel_max"] <= o.ERR_REL_TOL, (tag, m["e_rel_max"])
    assert m["max_abs_ratio_max"] <= o.MAX_ABS_TOL, (tag, m["max_abs_ratio_max"])


@pytest.mark.parametrize("n", [64, 128, 192, 256, 384, 512, 768, 1024, 1536, 2048, 4096])
@pytest.mark.parametrize("norm", [0, 1])
def test_lines_many_and_few_panels(oracle_mod, cuda_dev, n, norm):
    """The line engine on a batch of more panels than SMs in both passes and on
    its single arrays (fewer panels: the short-chain form from 256 points on),
    lines of n points along h and along w, every direction."""
    import torch
    from paper_2609_28519_gb300 import Plan
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    for (h, w) in ((n, 192), (192, n)):
        batch = max(1, -(-33 * sms // min(h, w)))  # at least 32 lines per SM and pass
        one = inputs.uniform(7 * n + h, 2, h, w)
        plan = Plan(h, w, kind=15, norm=norm)
        lam = inputs.random_diagonal(n + 3, h, w)
        plan.set_spectral(lam)
        x = torch.zeros(batch, h, w, device=cuda_dev)
        x[0], x[batch - 1] = torch.from_numpy(one[0]), torch.from_numpy(one[1])
        for kind in KINDS:
            many = plan.execute(kind, x)
            few = torch.cat([plan.execute(kind, x[i:i + 1].contiguous()) for i in (0, batch - 1)])
            torch.cuda.synchronize()
            assert plan.device_status() == 0
            _check(oracle_mod, many[[0, batch - 1]].cpu().numpy(), kind, one, norm, lam, ("many", h, w, kind))
            _check(oracle_mod, few.cpu().numpy(), kind, one, norm, lam, ("few", h, w, kind))
        plan.close()


# odd and even heights, half lengths at and around the chunk of 16 and the tile
# of 64 pairs, one and several tiles, line counts that end inside a block
DENSE_SHAPES = [(65, 68), (66, 64), (1, 68), (2, 72), (31, 96), (33, 100), (95, 128), (97, 132), (127, 136), (128, 72),
                (129, 256), (130, 260), (257, 68), (255, 512), (300, 388), (5, 1028)]


@pytest.mark.parametrize("h,w", DENSE_SHAPES)
@pytest.mark.parametrize("norm", [0, 1])
def test_dense_passes_edges(oracle_mod, cuda_dev, h, w, norm):
    """The half products of the dense passes, every direction."""
    import torch
    from paper_2609_28519_gb300 import Plan
    batch = 3
    x = inputs.uniform(31 * h + w, batch, h, w)
    plan = Plan(h, w, kind=15, norm=norm)
    assert plan.info().variant == 2
    lam = inputs.random_diagonal(h + w, h, w)
    plan.set_spectral(lam)
    for kind in KINDS:
        y = plan.execute(kind, torch.from_numpy(x).to(cuda_dev))
        _check(oracle_mod, y.cpu().numpy(), kind, x, norm, lam, (h, w, kind))


# output quads per warp 1, 2 and 4 on either axis, sums of one and two blocks
# of 16, odd heights, widths whose half is no multiple of 4, one and many arrays
SMALL_SHAPES = [(1, 4), (2, 4), (3, 12), (7, 20), (9, 8), (15, 28), (17, 36), (31, 64), (33, 4), (34, 60), (64, 12),
                (63, 52), (64, 4), (16, 44)]


@pytest.mark.parametrize("h,w", SMALL_SHAPES)
@pytest.mark.parametrize("batch", [1, 333])
def test_small_dense_edges(oracle_mod, cuda_dev, h, w, batch):
    """The half products of the on-chip dense route, every direction."""
    import torch
    from paper_2609_28519_gb300 import Plan
    x = inputs.uniform(17 * h + w + batch, batch, h, w)
    plan = Plan(h, w, kind=15)
    lam = inputs.random_diagonal(h * w, h, w)
    plan.set_spectral(lam)
    for kind in KINDS:
        y = plan.execute(kind, torch.from_numpy(x).to(cuda_dev))
        _check(oracle_mod, y.cpu().numpy(), kind, x, 0, lam, (h, w, batch, kind))


@pytest.mark.parametrize("h,w", [(256, 384), (384, 256), (512, 768), (128, 1280)])
@pytest.mark.parametrize("norm", [0, 1])
def test_tensor_passes_half_and_whole(oracle_mod, cuda_dev, h, w, norm):
    """Tensor-core passes with half products (multiples of 256) on one axis and
    the whole operator (other multiples of 128) on the other, or on both."""
    import torch
    from paper_2609_28519_gb300 import Plan
    x = inputs.uniform(h * 5 + w, 3, h, w)
    plan = Plan(h, w, kind=15, norm=norm, path="split_tc")
    lam = inputs.random_diagonal(h + 1, h, w)
    plan.set_spectral(lam)
    for kind in KINDS:
        y = plan.execute(kind, torch.from_numpy(x).to(cuda_dev))
        _check(oracle_mod, y.cpu().numpy(), kind, x, norm, lam, (h, w, kind))

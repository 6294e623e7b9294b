"""The tensor-core passes by their number of BF16 terms, against the arithmetic
that the path names say: every operand in one, two or three BF16 terms, the
products of terms whose orders sum to at most the last one's."""
import numpy as np
import pytest

from paper_2609_28519_gb300 import inputs

pytestmark = pytest.mark.gpu


def _operator(n, inverse):
    k, j = np.arange(n)[:, None], np.arange(n)[None, :]
    q = np.cos(np.pi * ((2 * j + 1) * k % (4 * n)) / (2 * n)) * np.sqrt(2.0 / n)
    q[0] = np.sqrt(1.0 / n)
    return q.T if inverse else q


def _terms(x, count):
    import torch
    out = []
    for _ in range(count):
        t = torch.from_numpy(x).to(torch.bfloat16).double().numpy()
        out.append(t)
        x = x - t
    return out


def _pass(x, m, count):
    """x m^T along the rows in `count` terms, summed in 64 bits."""
    xs, ms = _terms(x, count), _terms(m, count)
    return sum(xs[i] @ ms[j].T for i in range(count) for j in range(count - i))


def _emulated(x, inverse, count):
    h, w = x.shape[-2:]
    y = _pass(x, _operator(w, inverse), count).astype(np.float32).astype(np.float64)
    return np.swapaxes(_pass(np.ascontiguousarray(np.swapaxes(y, -1, -2)), _operator(h, inverse), count), -1, -2)


def _rel(y, ref):
    return float(np.linalg.norm(y - ref) / np.linalg.norm(ref))


@pytest.mark.parametrize("h,w", [(256, 256), (256, 384), (512, 256), (128, 192)])
@pytest.mark.parametrize("path,count,top", [("bf16", 1, 256), ("split_hilo", 2, 65536)])
@pytest.mark.parametrize("kind", ["forward", "inverse"])
def test_one_and_two_terms_lose_no_more_than_the_operands(cuda_dev, h, w, path, count, top, kind):
    """Whole numbers that the terms hold exactly and uniform values: the error is
    that of the emulated arithmetic (2% for the order of the sums and the tensor
    cores' accumulation; sums of two operands, in as many terms, lose 15%)."""
    import torch
    from paper_2609_28519_gb300 import Plan
    plan = Plan(h, w, path=path)
    whole = np.random.default_rng(h + w).integers(0, top, (4, h, w)).astype(np.float32) - top / 2
    for x in (whole, inputs.uniform(h * w, 4, h, w)):
        inv = kind == "inverse"
        ref = _operator(h, inv) @ x.astype(np.float64) @ _operator(w, inv).T
        got = plan.execute(kind, torch.from_numpy(x).to(cuda_dev)).cpu().numpy()
        assert _rel(got, ref) <= 1.02 * _rel(_emulated(x.astype(np.float64), inv, count), ref)


@pytest.mark.parametrize("h,w", [(256, 256), (256, 640), (1024, 512)])
def test_three_terms_in_place(cuda_dev, h, w):
    import torch
    from paper_2609_28519_gb300 import Plan
    plan = Plan(h, w, kind=15, path="split_tc")
    plan.set_spectral(inputs.random_diagonal(5, h, w))
    x = torch.from_numpy(inputs.uniform(h + w, 3, h, w)).to(cuda_dev)
    for kind in ("forward", "inverse", "roundtrip", "spectral"):
        y, z = plan.execute(kind, x), x.clone()
        plan.execute(kind, z, z)
        assert torch.equal(y, z), kind


@pytest.mark.parametrize("h,w", [(256, 256), (256, 384), (768, 512), (1024, 1024)])
def test_narrow_items_equal_the_wide_ones(cuda_dev, h, w):
    """A call of few row tiles takes items of half the width, the same sums: one
    array alone is bit for bit what it is in a batch that fills the chip."""
    import torch
    from paper_2609_28519_gb300 import Plan
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    plan = Plan(h, w, kind=15, path="split_tc")
    plan.set_spectral(inputs.random_diagonal(9, h, w))
    x = torch.from_numpy(inputs.uniform(h + 2 * w, 2, h, w)).to(cuda_dev)
    many = x.repeat(-(-128 * sms // min(h, w)), 1, 1)
    for kind in ("forward", "inverse", "roundtrip", "spectral"):
        y = plan.execute(kind, many)
        assert torch.equal(y, plan.execute(kind, x).repeat(len(many) // 2, 1, 1)), kind
        assert torch.equal(y[1], plan.execute(kind, x[1:].contiguous())[0]), kind
    assert plan.device_status() == 0

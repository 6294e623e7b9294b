"""Values near the ends of the FP32 range without range protection: where the
exact result is representable and the direct sums (or the transforms that the
kernels replaced) reached it, the kernels reach it too.

Half products add mirrored values before any weight, FFT steps add a whole line
before the scale: both are checked with the arrays that meet their limit first.
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _plan(h, w, path, kinds=15):
    from paper_2609_28519_gb300 import Plan
    plan = Plan(h, w, kind=kinds, path=path)
    plan.set_spectral(np.ones((h, w)))
    return plan


def _mirrored(h, w, sign):
    """Two equal (or opposite) values mirrored in a row, two in a column."""
    x = np.zeros((2, h, w))
    x[0, h // 3, w // 3], x[0, h // 3, w - 1 - w // 3] = 1.0, sign
    x[1, h // 4, w // 3] += 1.0
    x[1, h - 1 - h // 4, w // 3] += sign
    return x


def _operator(n):
    k, j = np.arange(n)[:, None], np.arange(n)[None, :]
    q = np.cos(np.pi * ((2 * j + 1) * k % (4 * n)) / (2 * n)) * np.sqrt(2.0 / n)
    q[0] = np.sqrt(1.0 / n)
    return q


# the on-chip dense route, the dense passes (one and several tiles, odd heights), the tensor-core passes
@pytest.mark.parametrize("h,w,path", [(12, 12, "fp32"), (7, 20, "fp32"), (48, 60, "fp32"), (100, 100, "fp32"),
                                      (97, 132, "fp32"), (256, 256, "split_tc"), (256, 512, "split_tc")])
@pytest.mark.parametrize("sign", [1.0, -1.0])
def test_half_products_of_mirrored_large_values(cuda_dev, h, w, path, sign):
    """2^127.4 twice, whose sum is above FLT_MAX: no output is."""
    import torch
    plan = _plan(h, w, path)
    x = (_mirrored(h, w, sign) * 2.0 ** 127.4).astype(np.float32)
    ref = _operator(h) @ x.astype(np.float64) @ _operator(w).T
    xd = torch.from_numpy(x).to(cuda_dev)
    got = plan.forward(xd).cpu().numpy().astype(np.float64)
    assert np.all(np.isfinite(got))
    assert np.linalg.norm(got / 2.0 ** 120 - ref / 2.0 ** 120) <= 1e-6 * np.linalg.norm(ref / 2.0 ** 120)
    for kind in ("roundtrip", "spectral"):
        got = plan.execute(kind, xd).cpu().numpy().astype(np.float64)
        assert np.linalg.norm(got / 2.0 ** 120 - x / 2.0 ** 120) <= 1e-6 * np.linalg.norm(x / 2.0 ** 120), kind


# log2 of the amplitude that the kernels replaced took to finite results, halves of a binade: constant
# arrays and the middle cosine, round trip; +-1 signs, forward and spectral
LIMITS = [(128, 128, 121.0, 122.0, 122.5), (64, 128, 121.0, 122.0, 122.5), (128, 64, 121.0, 122.0, 122.5),
          (192, 192, 118.5, 121.0, 121.5), (256, 256, 118.0, 121.0, 121.5), (384, 384, 117.5, 120.0, 121.0),
          (512, 512, 117.0, 120.0, 121.0), (768, 768, 116.5, 119.0, 120.5), (1024, 1024, 116.0, 119.0, 120.0)]


@pytest.mark.parametrize("h,w,const,cos,sign", LIMITS)
def test_lines_reach_the_range_of_the_kernels_replaced(cuda_dev, h, w, const, cos, sign):
    import torch
    plan = _plan(h, w, "fp32")
    wave = lambda n: np.cos(np.pi * (2 * np.arange(n) + 1) * (n // 3) / (2 * n))
    signs = np.random.default_rng(h + w).integers(0, 2, (h, w)) * 2.0 - 1.0
    for name, x, e, kinds in (("const", np.ones((h, w)), const, ("roundtrip",)),
                              ("cos", np.outer(wave(h), wave(w)), cos, ("roundtrip",)),
                              ("signs", signs, sign, ("forward", "roundtrip", "spectral"))):
        xd = torch.from_numpy((x * 0.99 * 2.0 ** e).astype(np.float32)[None]).to(cuda_dev)
        for kind in kinds:
            assert torch.isfinite(plan.execute(kind, xd)).all(), (name, kind)

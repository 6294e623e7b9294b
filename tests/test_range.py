"""Values near the ends of the FP32 range without range protection: where the
exact result is representable and the direct sums reached it, half products,
which add mirrored values before any weight, reach it too.
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

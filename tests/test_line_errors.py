"""Errors of the FP32 line kernels (the line engine and the on-chip kernels of
sides 64 and 128) against 64 bits: relative L2 over about a million values, on
many arrays at once and on one array a call, which run different forms.

The bounds are the errors that the four-step engine and the recursion in one
thread, which these kernels replaced, had on the same inputs, plus 1% for the
sampling of the rounding errors themselves (their relative standard deviation
at a million values is about 0.1%, on fewer values of one array a call 0.3%).
"""
import numpy as np
import pytest

from paper_2609_28519_gb300 import inputs

pytestmark = pytest.mark.gpu

# shape: forward, inverse, round trip, spectral (orthonormal); forward, inverse (unnormalized); 1e-7
REPLACED = {
    (64, 256): (1.613, 1.613, 2.143, 2.602, 1.451, 1.456),
    (192, 256): (1.542, 1.539, 2.209, 2.327, 1.545, 1.546),
    (384, 256): (1.815, 1.819, 2.309, 2.963, 1.613, 1.614),
    (512, 256): (1.711, 1.710, 2.433, 2.713, 1.624, 1.625),
    (768, 256): (1.640, 1.646, 2.394, 2.478, 1.658, 1.662),
    (1024, 256): (1.878, 1.885, 2.562, 3.068, 1.695, 1.697),
    (1536, 256): (1.930, 1.934, 2.531, 3.172, 1.733, 1.736),
    (2048, 256): (1.865, 1.865, 2.723, 3.003, 1.770, 1.774),
    (4096, 256): (2.024, 2.025, 2.795, 3.324, 1.827, 1.825),
    (256, 256): (1.723, 1.727, 2.285, 2.774, 1.548, 1.554),
    (192, 192): (1.480, 1.474, 2.142, 2.177, 1.543, 1.540),
    (768, 768): (1.651, 1.648, 2.496, 2.416, 1.771, 1.773),
    (64, 128): (1.380, 1.376, 1.909, 2.159, 1.286, 1.287),
    (128, 64): (1.381, 1.381, 1.908, 2.160, 1.284, 1.289),
    (128, 128): (1.347, 1.346, 2.002, 2.054, 1.344, 1.346),
}
CALLS = [("forward", 0), ("inverse", 0), ("roundtrip", 0), ("spectral", 0), ("forward", 1), ("inverse", 1)]


def _operator(n, norm, inverse):
    k, j = np.arange(n)[:, None], np.arange(n)[None, :]
    q = np.cos(np.pi * ((2 * j + 1) * k % (4 * n)) / (2 * n))
    s = np.full((n, 1), np.sqrt(2.0 / n) if norm == 0 else 2.0)
    s[0] = np.sqrt(1.0 / n) if norm == 0 else (1.0 if inverse else 2.0)
    return (q * s).T if inverse else q * s


def _exact(kind, x, norm, lam):
    h, w = x.shape[-2:]
    x = x.astype(np.float64)
    if kind == "roundtrip":
        return x
    if kind == "spectral":
        y = _operator(h, 0, False) @ x @ _operator(w, 0, False).T * lam
        return _operator(h, 0, True) @ y @ _operator(w, 0, True).T
    inv = kind == "inverse"
    return _operator(h, norm, inv) @ x @ _operator(w, norm, inv).T


def measure(make_plan, h, w):
    """Relative L2 of every call: (all arrays in one call, one array a call)."""
    import torch
    b = max(1, (1 << 20) // (h * w))
    x = inputs.uniform(101 * h + w, b, h, w)
    lam = inputs.random_diagonal(h + w, h, w)
    xd = torch.from_numpy(x).cuda()
    got = {}
    for norm in (0, 1):
        plan = make_plan(h, w, norm)
        plan.set_spectral(lam)
        for kind, nrm in CALLS:
            if nrm != norm:
                continue
            ref = _exact(kind, x, norm, lam)
            # enough copies for more panels than SMs
            many = plan.execute(kind, xd.repeat(max(1, 16384 // (min(h, w) * b)), 1, 1))[:b]
            few = torch.cat([plan.execute(kind, xd[i:i + 1]) for i in range(b)])
            torch.cuda.synchronize()
            assert plan.device_status() == 0
            got[kind, norm] = [float(np.linalg.norm(y.cpu().numpy() - ref) / np.linalg.norm(ref)) for y in (many, few)]
        plan.close()
    return got


@pytest.mark.parametrize("h,w", list(REPLACED))
def test_errors_are_no_larger_than_of_the_kernels_replaced(cuda_dev, h, w):
    from paper_2609_28519_gb300 import Plan
    got = measure(lambda r, c, norm: Plan(r, c, kind=15, norm=norm), h, w)
    for call, bound in zip(CALLS, REPLACED[h, w]):
        assert max(got[call]) <= 1.01e-7 * bound, (call, got[call], bound)

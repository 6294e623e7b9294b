"""What a user of this library has it do, as timed cases.

Every case goes through the public binding: a plan (or a ragged plan) made
once, device tensors in, preallocated device tensors out.  Three families:

* ``batch``   contiguous arrays of one shape (``Plan.execute``), from one
  array to 512 MiB, on the default path or the split-BF16 tensor-core path;
* ``image``   the blocks of an image through the tiled view
  (``Plan.execute_tiled``);
* ``ragged``  arrays of mixed shapes in one call (``Ragged.execute``).

``listed()`` holds the workloads the repository's benchmark is quoted on (the
8 x 8 batch, the phase-unwrapping image, the square sweep, the ragged batch
and the large arrays) with the other routes a user meets: a whole-image
Poisson solve, sides that are no power of two, the tensor-core path.
``draw()`` spreads further cases over the same families.
"""
import math

import numpy as np
import torch

from paper_2609_28519_gb300 import FORWARD, INVERSE, ROUNDTRIP, Plan, Ragged

SPECTRAL = 8
KIND_BITS = {"forward": FORWARD, "inverse": INVERSE, "roundtrip": ROUNDTRIP, "spectral": SPECTRAL}

# shapes of the mixed batch: squares and rectangles, small blocks to whole images
MIXED_SHAPES = [(8, 8), (16, 16), (32, 32), (64, 64), (128, 128), (256, 256), (64, 256), (128, 512), (768, 1024)]
LINE_SIDES = [64, 128, 192, 256, 384, 512, 768, 1024, 1536, 2048, 4096]


def listed():
    return [
        # the smallest call: a codec's worth of 8 x 8 blocks, bound by launches and host work
        _batch("blocks8", 8, 8, 1024, "forward,inverse,roundtrip"),
        # phase unwrapping on blocks: a 2048 x 2048 image as 16 x 16 blocks, forward then inverse
        {"name": "image16", "family": "image", "img_rows": 2048, "img_cols": 2048, "rows": 16, "cols": 16,
         "kinds": "forward,inverse", "norm": "ortho", "path": "auto", "protect": False},
        # the square sweep at 512 MiB a direction: middle and upper block sizes
        _batch("square64", 64, 64, 32768, "forward,inverse,roundtrip"),
        _batch("square128", 128, 128, 8192, "forward,inverse,roundtrip"),
        _batch("square256", 256, 256, 2048, "forward,inverse,roundtrip"),
        # whole-image least-squares phase unwrapping: a stack of 1024 x 1024 images, the Poisson diagonal
        _batch("poisson1024", 1024, 1024, 16, "spectral"),
        # large whole arrays
        _batch("large4096", 4096, 4096, 4, "forward,inverse"),
        # one rectangle of 3 * 2^8 columns: a single image, too few lines to fill the chip
        _batch("single1024x768", 1024, 768, 1, "forward,inverse"),
        # mixed shapes in one call
        {"name": "ragged4096", "family": "ragged", "count": 4096, "shape_seed": 4, "kinds": "forward,inverse",
         "norm": "ortho"},
        # sides with other factors: small arrays, and arrays beyond the on-chip route
        _batch("small26x32", 26, 32, 80659, "forward,inverse"),
        _batch("other100", 100, 100, 6711, "forward,inverse", norm="none"),
        # the dense-contraction path on the tensor cores
        _batch("tensor1024", 1024, 1024, 16, "forward,inverse", path="split_tc"),
    ]


def _batch(name, rows, cols, count, kinds, norm="ortho", path="auto", protect=False):
    return {"name": name, "family": "batch", "rows": rows, "cols": cols, "count": count, "kinds": kinds,
            "norm": norm, "path": path, "protect": protect}


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    family = rng.choice(["fused", "ring", "lines", "lines", "image", "ragged", "small", "other", "tensor"])
    kinds = rng.choice(["forward,inverse", "forward,inverse", "forward,inverse,roundtrip", "roundtrip", "inverse",
                        "spectral"])
    norm = rng.choice(["ortho", "ortho", "none"])
    protect = rng.random() < 0.1
    most = 1 << 26  # elements
    if family == "ragged":
        return {"family": "ragged", "count": _log_int(rng, 40, 2500), "shape_seed": rng.randrange(1 << 20),
                "kinds": rng.choice(["forward,inverse", "roundtrip"]), "norm": norm}
    if family == "image":
        r, c = rng.choice([8, 16, 32, 64, 24]), rng.choice([8, 16, 32, 64, 40])
        return {"family": "image", "img_rows": r * _log_int(rng, 3, 4096 // r), "img_cols": c * _log_int(rng, 3, 4096 // c),
                "rows": r, "cols": c, "kinds": kinds, "norm": norm, "path": "auto", "protect": protect}
    path = "auto"
    if family == "fused":
        r, c = rng.choice([8, 16, 32]), rng.choice([8, 16, 32])
    elif family == "ring":
        r, c = rng.choice([64, 128]), rng.choice([64, 128])
    elif family == "lines":
        r, c = rng.choice(LINE_SIDES), rng.choice(LINE_SIDES)
        if r <= 128 and c <= 128:
            c = rng.choice(LINE_SIDES[2:])
    elif family == "small":
        r, c = rng.randint(3, 64), 4 * rng.randint(1, 16)
    elif family == "other":
        r, c = _log_int(rng, 65, 1300), 4 * _log_int(rng, 17, 480)
        most = min(most, 6_000_000_000 // (r + c))  # a dense product: n multiply-adds a value and pass
    else:
        r = c = rng.choice([16, 32, 64, 128, 256, 512, 1024])
        path, norm = "split_tc", "ortho"
        most = min(most, 30_000_000_000 // (r + c))
    lo = min(max(r * c, 1 << 14), most)
    count = max(1, _log_int(rng, lo, max(lo, most)) // (r * c))
    return _batch_case(r, c, count, kinds, norm, path, protect)


def _batch_case(rows, cols, count, kinds, norm, path, protect):
    c = _batch("", rows, cols, count, kinds, norm, path, protect)
    del c["name"]
    return c


# ------------------------------------------------------------------ inputs
def _shapes(case):
    idx = np.random.default_rng(case["shape_seed"]).integers(0, len(MIXED_SHAPES), size=case["count"])
    return [MIXED_SHAPES[int(i)] for i in idx]


def _offsets(shapes):
    return np.concatenate([[0], np.cumsum([r * c for r, c in shapes])]).astype(np.int64)


def _poisson(h, w):
    """Inverse eigenvalues of the 5-point Laplacian with reflecting borders, 0 for the constant."""
    k, l = np.arange(h, dtype=np.float64)[:, None], np.arange(w, dtype=np.float64)[None, :]
    ev = 2.0 * np.cos(np.pi * k / h) + 2.0 * np.cos(np.pi * l / w) - 4.0
    ev[0, 0] = 1.0
    lam = 1.0 / ev
    lam[0, 0] = 0.0
    return lam


def _input(case, seed):
    g = torch.Generator(device="cuda").manual_seed(seed)
    if case["family"] == "image":
        h, w = case["img_rows"], case["img_cols"]
        # Gaussian noise on a smooth ramp, as a wrapped-phase gradient has
        ramp = torch.arange(h, device="cuda", dtype=torch.float32)[:, None] + torch.arange(w, device="cuda", dtype=torch.float32)
        return torch.randn(h, w, generator=g, device="cuda") + 0.01 * ramp
    if case["family"] == "ragged":
        n = int(_offsets(_shapes(case))[-1])
        return torch.rand(n, generator=g, device="cuda").mul_(2.0).sub_(1.0)
    shape = (case["count"], case["rows"], case["cols"])
    if max(case["rows"], case["cols"]) > 256 or "spectral" in case["kinds"]:
        return torch.randn(shape, generator=g, device="cuda")
    return torch.rand(shape, generator=g, device="cuda").mul_(2.0).sub_(1.0)


def prepare(case, seed):
    kinds = case["kinds"].split(",")
    bits = sum(KIND_BITS[k] for k in kinds)
    x = _input(case, seed)
    state = {"case": case, "kinds": kinds, "x": x, "out": {k: torch.empty_like(x) for k in kinds}}
    if case["family"] == "ragged":
        state["plan"] = Ragged(_shapes(case), kind=bits, norm=case["norm"])
        return state
    plan = Plan(case["rows"], case["cols"], kind=bits, norm=case["norm"], path=case["path"])
    if "spectral" in kinds:
        plan.set_spectral(_poisson(case["rows"], case["cols"]))
    if case["protect"]:
        plan.set_range_protection(True)
    state["plan"] = plan
    return state


def run(state):
    """The case's directions in order; the inverse takes the forward's spectrum where there is one."""
    plan, out = state["plan"], state["out"]
    call = plan.execute_tiled if state["case"]["family"] == "image" else plan.execute
    for k in state["kinds"]:
        src = out["forward"] if k == "inverse" and "forward" in out else state["x"]
        call(k, src, out[k])
    return out


def work(case):
    """One read and one write of every value a direction; the multiply-adds of the dense product on that path."""
    n, mult = 0, 0
    if case["family"] == "ragged":
        n = int(_offsets(_shapes(case))[-1])
    elif case["family"] == "image":
        n = case["img_rows"] * case["img_cols"]
    else:
        n = case["count"] * case["rows"] * case["cols"]
        if case["path"] == "split_tc":
            mult = n * (case["rows"] + case["cols"])
    passes = sum(2 if k in ("roundtrip", "spectral") else 1 for k in case["kinds"].split(","))
    return {"bytes": 8 * n * len(case["kinds"].split(",")), "flops": 2 * mult * passes}


# ------------------------------------------------------------------ 64 bits
def _op(n, norm, inverse):
    """The n x n matrix of Eq. 1 (orthonormal), or of the unnormalized REDFT pair, in 64 bits."""
    k = torch.arange(n, device="cuda", dtype=torch.int64)[:, None]
    j = torch.arange(n, device="cuda", dtype=torch.int64)[None, :]
    q = torch.cos(((2 * j + 1) * k % (4 * n)).double() * (math.pi / (2 * n)))
    s = torch.full((n, 1), math.sqrt(2.0 / n) if norm == "ortho" else 2.0, device="cuda", dtype=torch.float64)
    if norm == "ortho":
        s[0] = math.sqrt(1.0 / n)
    elif inverse:
        s[0] = 1.0
    q = q * s
    return q.t().contiguous() if inverse else q


def _sandwich(x, norm, inverse, lam=None):
    """M_h X M_w^T of every array of x (batch, h, w), in 64 bits, a slice of the batch at a time."""
    h, w = x.shape[-2:]
    out = torch.empty(x.shape, device="cuda", dtype=torch.float64)
    mh, mw = _op(h, norm, inverse), _op(w, norm, inverse)
    step = max(1, (1 << 27) // (h * w))
    for b in range(0, x.shape[0], step):
        y = torch.matmul(mh, torch.matmul(x[b:b + step].double(), mw.t()))
        if lam is not None:
            y = torch.matmul(_op(h, norm, True), torch.matmul(y * lam, _op(w, norm, True).t()))
        out[b:b + step] = y
    return out


def _exact_arrays(kind, x, norm, forward_first):
    h, w = x.shape[-2:]
    if kind == "forward":
        return _sandwich(x, norm, False)
    if kind == "roundtrip":
        return x.double()
    if kind == "spectral":
        return _sandwich(x, "ortho", False, torch.from_numpy(_poisson(h, w)).to("cuda"))
    if forward_first:  # the pair's factor: 1 orthonormal, 2n an axis unnormalized
        return x.double() * (1.0 if norm == "ortho" else 4.0 * h * w)
    return _sandwich(x, norm, True)


def exact(case, seed):
    x, kinds, norm = _input(case, seed), case["kinds"].split(","), case["norm"]
    got = {}
    for k in kinds:
        first = "forward" in kinds
        if case["family"] == "image":
            h, w = case["rows"], case["cols"]
            r, c = case["img_rows"] // h, case["img_cols"] // w
            b = x.view(r, h, c, w).transpose(1, 2).reshape(r * c, h, w)
            got[k] = _exact_arrays(k, b, norm, first).view(r, c, h, w).transpose(1, 2).reshape(r * h, c * w)
        elif case["family"] == "ragged":
            shapes = _shapes(case)
            off = _offsets(shapes)
            got[k] = torch.empty(x.numel(), device="cuda", dtype=torch.float64)
            for (h, w) in sorted(set(shapes)):
                at = [int(off[i]) for i, s in enumerate(shapes) if s == (h, w)]
                y = _exact_arrays(k, torch.stack([x[o:o + h * w].view(h, w) for o in at]), norm, first)
                for o, a in zip(at, y):
                    got[k][o:o + h * w] = a.reshape(-1)
        else:
            got[k] = _exact_arrays(k, x, norm, first)
    return got

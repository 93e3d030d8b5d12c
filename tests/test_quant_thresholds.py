"""The quantizer kernel's int2 codes by thresholds on the bf16 inputs (CPU).

The kernel finds, for each group, the smallest bf16 value that reaches code 1,
2 and 3 and counts how many of the three an element passes. Here the same
steps in numpy are compared with the oracle's quantizer for every finite bf16
value: random fp16 scales and zero-points, and the relations where a
threshold lies near zero, where bf16 values are denser than fp32 differences.
This pins the argument only; the kernel's own codes are compared with the
oracle's in test_gpu_kernels (test_quantize_codes_at_their_edges and the
parity cases).
"""
import numpy as np
import pytest

from oracle import quant as oquant

BITS16 = np.arange(1 << 16, dtype=np.uint32)
ALL = (BITS16 << 16).view(np.float32)
FINITE = ALL[np.isfinite(ALL)]


def _bf16(x):
    u = np.float32(x).view(np.uint32)
    return (((u + 0x7FFF + ((u >> 16) & 1)) >> 16) << 16).astype(np.uint32) if np.isfinite(x) else u


def _of_order(o):
    b = (o & 0x7FFF) if o & 0x8000 else (~o & 0xFFFF)
    return np.uint32(b << 16).view(np.float32)


def _threshold(z, t_min):
    reaches = lambda x: np.float32(x) - z >= t_min  # noqa: E731
    u = int(_bf16(z + t_min))
    f = lambda v: np.uint32(v & 0xFFFFFFFF).view(np.float32)  # noqa: E731
    inside = bool(reaches(f(u)))
    nxt = f(u + (0x10000 if inside == bool(u & 0x80000000) else -0x10000))
    if u << 1 & 0xFFFFFFFF and bool(reaches(nxt)) != inside:
        return f(u) if inside else nxt
    lo, hi = 0x007F, 0xFF80
    while hi - lo > 1:
        mid = (lo + hi) >> 1
        lo, hi = (lo, mid) if reaches(_of_order(mid)) else (mid, hi)
    return _of_order(hi)


def _pairs(kind, n, rng):
    for _ in range(n):
        s = np.float16(0)
        while s == 0 or not np.isfinite(s):
            s = rng.integers(1, 0x7C00, dtype=np.uint16).view(np.float16) if kind != "normal" \
                else np.float16(abs(rng.standard_normal()) + 1e-3)
        if kind == "random":
            z = rng.integers(0, 1 << 16, dtype=np.uint16).view(np.float16)
        elif kind == "normal":
            z = np.float16(-1.5 * float(s) * (1 + 0.2 * rng.standard_normal()))
        else:   # a threshold at or next to zero
            z = np.float16(-float(rng.choice([0.5, 1.5, 2.5, 0.0])) * float(s))
            z = (z.view(np.uint16) + np.uint16(rng.integers(0, 3))).view(np.float16)
        if np.isfinite(z):
            yield s, np.float16(z + np.float16(0))


@pytest.mark.parametrize("kind", ["random", "normal", "near_zero"])
def test_threshold_codes_match_the_quantizer(kind):
    rng = np.random.default_rng(len(kind))
    with np.errstate(over="ignore", invalid="ignore"):
        for s16, z16 in _pairs(kind, 60, rng):
            s, z = np.float32(s16), np.float32(z16)
            t = [np.nextafter(np.float32(0.5) * s, np.float32(np.inf)), np.float32(1.5) * s,
                 np.nextafter(np.float32(2.5) * s, np.float32(np.inf))]
            got = sum((FINITE >= _threshold(z, x)).astype(np.uint8) for x in t)
            want = oquant._codes(FINITE, s16, z16, 2)
            bad = np.flatnonzero(got != want)
            assert bad.size == 0, (s16, z16, FINITE[bad[:4]], got[bad[:4]], want[bad[:4]])

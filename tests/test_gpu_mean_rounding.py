"""The float32 merged mean on the GPU, bit by bit against exact rational arithmetic.

Every A token of a sample merges into its first B token (their keys agree, the other B keys are orthogonal), so a merged
row is sum s_t x_t / sum s_t over one to five tokens.  The kernel forms the sum in float-float (about 44 bits of the
largest partial sum, so of sum |s_t x_t|) and the quotient to about 45 bits, with exact ties kept: the result is the
correctly rounded quotient unless that lies within 2^-40 sum |s_t x_t| / sum s_t of a rounding midpoint without being one."""
import os
import sys
from fractions import Fraction

import numpy as np
import pytest
import torch

sys.path.insert(0, os.path.dirname(os.path.abspath(__file__)))

from paper_2607_02612_gb300 import runner  # noqa: E402

pytestmark = pytest.mark.gpu

N, DIM = 9, 32   # CLS, four B tokens (1, 3, 5, 7) and four A tokens (2, 4, 6, 8)


def merged_rows(x, sizes, r):
    """Output rows of B token 1 of every sample: x [B, N, DIM], sizes [B, N] float32, r [B]."""
    B = x.shape[0]
    keys = np.zeros((B, N, 16), np.float32)
    keys[:, 0, 15] = 1
    keys[:, 2::2, 0] = keys[:, 1, 0] = 1                          # every A token like the first B token
    for k, pos in enumerate((3, 5, 7)):
        keys[:, pos, 1 + k] = 1
    offsets = np.arange(B + 1, dtype=np.int32) * N
    b = runner.device_batch("f32", offsets, x.reshape(B * N, DIM), keys.reshape(B * N, 16), sizes.reshape(-1), None)
    f = runner.Fusion(B)
    o = f.merge(b, torch.from_numpy(np.asarray(r, np.int32)).cuda())
    assert int(f.status.item()) == 0
    out, offs, keep = o["x"].cpu().numpy(), o["offsets"].cpu().numpy(), o["keep_idx"].cpu().numpy()
    assert (keep[offs[:-1] + 1] == offsets[:-1] + 1).all()
    return out[offs[:-1] + 1]


def rounded(q):
    """(q to nearest even as float32, the distance of q from the nearest rounding midpoint); no overflow."""
    if q == 0:
        return np.float32(0), None
    a, e = abs(q), 0
    while a >= Fraction(2) ** (e + 1):
        e += 1
    while a < Fraction(2) ** e:
        e -= 1
    ulp = Fraction(2) ** (max(e, -126) - 23)
    n = a / ulp
    f = n.numerator // n.denominator
    up = n - f > Fraction(1, 2) or (n - f == Fraction(1, 2) and f % 2)
    v = (f + up) * ulp
    return np.float32(float(v if q > 0 else -v)), abs(n - f - Fraction(1, 2)) * ulp


def check(x, sizes, r, slack=2.0 ** -40):
    got = merged_rows(x, sizes, r)
    wrong = skipped = 0
    for i in range(x.shape[0]):
        group = [1] + [2, 4, 6, 8][:r[i]]                         # equal similarities: the lowest positions first
        s = [Fraction(float(sizes[i, t])) for t in group]
        den = sum(s)
        for c in range(DIM):
            terms = [w * Fraction(float(x[i, t, c])) for w, t in zip(s, group)]
            want, margin = rounded(sum(terms) / den)
            if margin is not None and 0 < margin < Fraction(slack) * sum(abs(v) for v in terms) / den:
                skipped += 1
            else:
                wrong += got[i, c] != want
    assert wrong == 0, f"{wrong} of {x.shape[0] * DIM} means are not the rounded quotient"
    assert skipped <= x.shape[0] * DIM // 100
    return got


@pytest.mark.parametrize("kind", ["integers", "floats", "wide", "tiny", "huge"])
def test_means_are_correctly_rounded(kind):
    rng = np.random.default_rng(len(kind))
    B = 120
    x = rng.standard_normal((B, N, DIM)).astype(np.float32)
    sizes = rng.integers(1, 5, (B, N)).astype(np.float32)
    if kind == "floats":                                          # sums of sizes that are not floats
        sizes = (1 + 3 * rng.random((B, N))).astype(np.float32)
    elif kind == "wide":                                          # sources far apart
        x *= (2.0 ** rng.integers(-12, 13, x.shape)).astype(np.float32)
    elif kind in ("tiny", "huge"):                                # past the short division's range, 2^-40 to 2^40
        x *= np.float32(2.0 ** (-60 if kind == "tiny" else 60))
    check(x, sizes, rng.integers(1, 5, B))


def test_ties_go_to_even_and_zeros_stay():
    """(x_1 + 2 x_2) / 3 halfway between two floats: x_2 in [1.9, 2), x_1 in [0.5, 1) with a bit more."""
    rng = np.random.default_rng(1)
    B, ulp = 120, 2.0 ** -23
    x = rng.standard_normal((B, N, DIM)).astype(np.float32)
    sizes = np.ones((B, N), np.float32)
    sizes[:, 2] = 2
    mid = 1.55 + rng.integers(0, 1 << 17, (B, DIM)) * ulp
    mid = np.round(mid / ulp) * ulp + ulp / 2
    x2 = (1.9 + rng.integers(0, 1 << 17, (B, DIM)) * ulp).astype(np.float32)
    x1 = 3 * mid - 2 * x2.astype(np.float64)
    assert (x1 == x1.astype(np.float32)).all() and (x1 < 1).all()
    x[:, 1], x[:, 2] = x1.astype(np.float32), x2
    x[::7, 1], x[::7, 2] = 2.0, -1.0                              # a sum of zero
    got = check(x, sizes, np.ones(B, np.int64))
    assert (got[::7] == 0).all()
    ties = got[1::7].astype(np.float64)
    assert ((ties / ulp).astype(np.int64) % 2 == 0).all()


def test_subnormal_means():
    """Means below the normal range: within one of their units (products there are not exact)."""
    rng = np.random.default_rng(2)
    B = 40
    x = (rng.standard_normal((B, N, DIM)) * 2.0 ** -135).astype(np.float32)
    sizes = rng.integers(1, 5, (B, N)).astype(np.float32)
    r = rng.integers(1, 5, B)
    got = merged_rows(x, sizes, r).astype(np.float64)
    for i in range(B):
        group = [1] + [2, 4, 6, 8][:r[i]]
        s = sizes[i, group].astype(np.float64)
        want = (s[:, None] * x[i, group].astype(np.float64)).sum(0) / s.sum()
        assert np.abs(got[i] - want).max() <= len(group) * 2.0 ** -149

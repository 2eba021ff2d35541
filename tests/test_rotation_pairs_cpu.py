"""The split behind the tensor-core rotation, restated in numpy: x = hi + lo with hi a
multiple of 2^u, u = 1 - l + k, both halves binary16, and every signed sum of the 2^l
halves of a block exact in fp32 when the block's sum of |x| is below 2^(25 - l + k) and x
is a multiple of 2^(k - 24); and for k > 0 the list of what rounding to that grid takes off."""
import numpy as np
import pytest

F16, F32 = np.float16, np.float32


def split(x, l, k):
    c = F16(2.0 ** (11 - l + k))
    m = np.minimum(np.abs(x), c)
    r = (m + c).astype(F16) - c
    lo = np.where(np.signbit(x), -(m - r), m - r).astype(F16)
    return (x - lo).astype(F16), lo


def fwht(v):
    h, n = 1, v.shape[-1]
    while h < n:
        w = v.reshape(-1, n // (2 * h), 2, h)
        v = np.concatenate([w[:, :, :1] + w[:, :, 1:], w[:, :, :1] - w[:, :, 1:]], axis=2).reshape(v.shape)
        h *= 2
    return v


# The kernel takes rows whose sum of |x| is below 2^22 this way, so k is at most l - 3.
@pytest.mark.parametrize("l,k", [(l, k) for l in (0, 1, 4, 5, 6, 7, 8, 10, 11, 12) for k in (0, 1, 4, 7, 9)
                                 if k <= max(0, l - 3)])
def test_split_sums_are_exact(l, k):
    n = 1 << l
    rng = np.random.default_rng(100 * l + k)
    rows = [rng.standard_normal(n), rng.standard_normal(n) * 1e-4, np.full(n, 1.0), rng.standard_normal(n) * 20]
    rows[1][0] = 300.0
    top = min(2.0 ** (25 - l + k), 2.0 ** 22)
    tried = 0
    for row in rows:
        for scale in (1.0, 0.5 * top / max(np.abs(row).sum(), 1e-9), 0.99 * top / max(np.abs(row).sum(), 1e-9)):
            x = np.clip(row * scale, -65504, 65504).astype(F16)
            # onto the grid of 2^(k - 24)
            x = (np.round(x.astype(np.float64) * 2.0 ** (24 - k)) * 2.0 ** (k - 24)).astype(F16)
            if not np.abs(x.astype(np.float64)).sum() < top:
                continue
            tried += 1
            hi, lo = split(x, l, k)
            assert np.array_equal(hi.astype(np.float64) + lo, x.astype(np.float64))
            u = 2.0 ** (1 - l + k)
            assert np.all(np.abs(lo.astype(np.float64)) <= u / 2) and np.all(hi.astype(np.float64) % u == 0)
            for part in (hi, lo):
                got = fwht(part.astype(F32)[None])[0]
                assert got.dtype == F32 and np.array_equal(got.astype(np.float64), fwht(part.astype(np.float64)[None])[0])
            # one fp32 addition rounds the exact sum correctly
            S = fwht(x.astype(np.float64)[None])[0]   # exact: below 2^53 units of 2^-24
            assert np.array_equal(fwht(hi.astype(F32)[None])[0] + fwht(lo.astype(F32)[None])[0], S.astype(F32))
    assert tried


def test_grid_test_of_large_sums():
    """m = min(|x|, 2^(k - 14)): (m + c) - c = m in binary16 exactly when x is a multiple of
    2^(k - 24), for every finite binary16."""
    x = np.arange(0, 0x7C00, dtype=np.uint16).view(F16)
    for k in range(1, 8):
        c = F16(2.0 ** (k - 14))
        m = np.minimum(np.abs(x), c)
        ok = ((m + c).astype(F16) - c).astype(F16) == m
        assert np.array_equal(ok, (x.astype(np.float64) * 2.0 ** (24 - k)) % 1.0 == 0)


def to_grid(x, k):
    """x rounded to multiples of 2^(k - 24) (binary16), and what that took off."""
    c = F16(2.0 ** (k - 14))
    m = np.minimum(np.abs(x), c)
    d = (m - ((m + c).astype(F16) - c).astype(F16)).astype(F16)
    d = np.where(np.signbit(x), -d, d).astype(F16)
    return (x - d).astype(F16), d


def test_rounding_to_the_grid():
    """For every finite binary16: on the grid, at most half a step off, and exactly undone by
    an integer number n of 2^-24, |n| <= 2^(k - 1)."""
    x = np.arange(0, 0x7C00, dtype=np.uint16).view(F16)
    x = np.concatenate([x, -x])
    for k in range(1, 10):
        g, d = to_grid(x, k)
        g64, n = g.astype(np.float64), d.astype(np.float64) * 2.0 ** 24
        assert np.array_equal(g64 + n * 2.0 ** -24, x.astype(np.float64))
        assert np.all(g64 * 2.0 ** (24 - k) % 1.0 == 0) and np.all(n % 1.0 == 0) and np.all(np.abs(n) <= 2 ** (k - 1))


@pytest.mark.parametrize("l,k", [(12, 1), (12, 4), (12, 9), (11, 8), (10, 7), (8, 3)])
def test_listed_remainders_correct_the_sums_exactly(l, k):
    n = 1 << l
    rng = np.random.default_rng(7 * l + k)
    top = 2.0 ** (25 - l + k)
    parity = np.array([bin(v).count("1") & 1 for v in range(n)])
    for share in (0.51, 0.99):
        x = (rng.standard_normal(n) * (share * top / n / 0.8)).astype(F16)
        x[rng.choice(n, 40, replace=False)] = (rng.standard_normal(40) * 2.0 ** (k - 16)).astype(F16)   # fine values
        x[0] = F16(min(65504.0, max(0.0, share * top - np.abs(x[1:].astype(np.float64)).sum())))
        assert np.abs(x.astype(np.float64)).sum() < top
        on, d = to_grid(x, k)
        entries = np.flatnonzero(d)
        assert 0 < entries.size <= 63
        hi, lo = split(on, l, k)
        h, o = fwht(hi.astype(F32)[None])[0], fwht(lo.astype(F32)[None])[0]
        f = h + o
        bv = f - h
        rem = (h - (f - bv)) + (o - bv)
        for i in entries:
            rem = rem + np.where(parity[np.arange(n) & i], -d[i], d[i]).astype(F32)
        assert f.dtype == rem.dtype == F32
        S = fwht(x.astype(np.float64)[None])[0]
        assert np.array_equal(f.astype(np.float64) + rem, S) and np.array_equal(f + rem, S.astype(F32))


def test_exchange_has_no_bank_conflicts():
    """The eight lanes of a quarter warp touch eight different 16-byte columns, writing and
    reading, and the granules of a unit are a permutation."""
    def granule(i):
        return (i >> 1) ^ ((i >> 4) & 1) ^ ((((i >> 8) ^ (i >> 5)) & 1) << 1) ^ (((i >> 9) & 1) << 2)
    assert sorted(granule(i) for i in range(0, 1024, 2)) == list(range(512))
    def quarters(index):
        for q4 in range(4):
            assert len({granule(index(lane)) % 8 for lane in range(8 * q4, 8 * q4 + 8)}) == 8
    for const in range(0, 32):   # in-thread element bits 2, 5, 6, 7 of a writer
        low = ((const & 1) << 2) | ((const >> 1 & 1) << 5) | ((const >> 2 & 3) << 6)
        quarters(lambda lane: low | ((lane >> 2 & 1) << 1) | ((lane >> 3) << 3) | ((lane & 3) << 8))
    for R in (8, 4, 2):          # readers: runs of R, 16 bytes at a time
        for e in range(0, R, 2):
            for c in range(4):
                quarters(lambda lane: (256 * c + R * lane + e) % 1024)

"""The GICP sums' conversion-free rounding, in binary32 arithmetic on the CPU.

A term x (|x| < 2^20) enters the sums as rint(2^24 x), split as hi 2^22 + lo by
adding 1.5 x 2^23 (which leaves the rounded integer in the low bits of the
binary32 sum).  Checked against float64 rint on random magnitudes, ties and the
bounds; the remainder has to be exact, and 32 lanes' biased bits have to add up
to the sums in wrapping 32-bit arithmetic."""
import numpy as np

MAGIC, BIAS = np.float32(12582912.0), 0x4B400000


def _split(x):
    x = x.astype(np.float32)
    t = (np.float64(4) * x + np.float64(MAGIC)).astype(np.float32)       # one rounding
    hf = t - MAGIC
    rest64 = x.astype(np.float64) * 2.0 ** 24 - hf.astype(np.float64) * 2.0 ** 22
    rest = rest64.astype(np.float32)
    assert np.array_equal(rest.astype(np.float64), rest64)               # the remainder is exact
    return t.view(np.int32), (rest + MAGIC).view(np.int32)


def test_terms_round_as_rint():
    rng = np.random.default_rng(2)
    x = rng.uniform(-1, 1, 400000) * 2.0 ** rng.integers(-40, 21, 400000)
    ties = (rng.integers(-2 ** 22, 2 ** 22, 50000) + 0.5) * 2.0 ** -24
    x = np.concatenate([x, ties, [0.0, -0.0, 2.0 ** 20 - 0.0625, -(2.0 ** 20) + 0.0625, 0.125, -0.125]]).astype(np.float32)
    x = x[np.abs(x) < 2.0 ** 20]
    h, l = _split(x)
    got = (h.astype(np.int64) - BIAS) * 2 ** 22 + (l.astype(np.int64) - BIAS)
    assert np.array_equal(got, np.rint(x.astype(np.float64) * 2.0 ** 24).astype(np.int64))


def test_wrapped_sums_of_32_lanes():
    rng = np.random.default_rng(4)
    x = (rng.choice([-1, 1], (2000, 32)) * rng.uniform(0, 1, (2000, 32)) * 2.0 ** rng.integers(-20, 21, (2000, 1))).astype(np.float32)
    x[:8] = np.float32(2.0 ** 20 - 0.0625)
    x[8:16] = -x[:8]
    h, l = (v.view(np.uint32) for v in _split(x))
    sums = [((v.sum(1, dtype=np.uint64) - np.uint64(32 * BIAS)) & np.uint64(0xFFFFFFFF)).astype(np.uint32).view(np.int32)
            for v in (h, l)]
    got = sums[0].astype(np.int64) * 2 ** 22 + sums[1]
    assert np.array_equal(got, np.rint(x.astype(np.float64) * 2.0 ** 24).astype(np.int64).sum(1))

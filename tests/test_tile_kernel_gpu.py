"""The tile compression kernel's ways through a block, bit for bit against the
oracle: warps ranked by match and by shared atomics, alone and in one block
(few and many distinct keys), and values that take a fallback candidate, in
blocks wide and narrow enough for that to move the field's code width."""
import numpy as np
import pytest

from tests.test_parity_gpu import assert_parity, gpz  # noqa: F401  (the fixture)

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("F", [1, 3, 6])
@pytest.mark.parametrize("n", [7, 255, 257, 1024, 4 * 1024 + 129])
@pytest.mark.parametrize("G", [1, 3])
def test_rank_ways(gpz, oracle, F, n, G):  # noqa: F811
    """A quarter of each block constant, a quarter a slow ramp, the rest
    uniform: the first 32 particles of a warp have 1 to 32 distinct keys."""
    rng = np.random.default_rng(1000 * F + n + G)
    x = rng.random((F, n)) * 100.0
    pos = np.arange(n) % 1024
    x[:, pos < 256] = 40.0
    ramp = (pos >= 256) & (pos < 512)
    x[:, ramp] = 100.0 * pos[ramp] / 1024.0
    assert_parity(gpz, oracle, x.astype(np.float32), 1e-2, 0, G)


def first_candidate_failures(x, eb):
    """Values of one block whose first candidate fails (fp32, one field; the
    multiply-adds rounded once, through float64, whose products are exact)."""
    f32, f64 = np.float32, np.float64
    s = f32(eb * 1.96875)
    inv = f32(1.0 / f64(s))
    chk = np.nextafter(f32(eb * (1.0 - 2.0 ** -22)), f32(0))
    mn = x.min()
    q = np.floor((f64(1) * (x - mn).astype(f32) * f64(inv) + 0.5).astype(f32))
    xh = (q.astype(f64) * f64(s) + f64(mn)).astype(f32)
    return int((np.abs(x - xh) > chk).sum())


@pytest.mark.parametrize("codes", [1, 2, 4, 33, 1000])
@pytest.mark.parametrize("n", [1024, 3 * 1024 + 77])
@pytest.mark.parametrize("offset,eb", [(9000.0, 8e-4), (5000.0, 3e-4), (130.0, 1.1e-5)])
def test_fallback_candidates(gpz, oracle, codes, n, offset, eb):  # noqa: F811
    """Values so far from zero that their rounding is a good part of the
    bound, spread over `codes` steps."""
    rng = np.random.default_rng(codes + n)
    x = (offset + rng.random((3, n)) * codes * 2.0 * eb).astype(np.float32)
    x[2] = rng.random(n).astype(np.float32) * 1e-2  # one field without them
    if codes >= 33:
        assert sum(first_candidate_failures(x[0, k:k + 1024], eb) for k in range(0, n, 1024)) > 0
    for mode in (0, 1):
        assert_parity(gpz, oracle, x, eb if mode == 0 else eb / (2.0 * eb * codes), mode, 3)


@pytest.mark.parametrize("offset", [1, 2, 3])
@pytest.mark.parametrize("F,mode", [(1, 0), (3, 1), (6, 1), (8, 0)])
@pytest.mark.parametrize("n", [1, 2, 5, 1023, 1024, 1025, 1026, 1027, 1029, 2047, 2 * 1024 + 2])
def test_unaligned_rows(gpz, oracle, offset, F, mode, n):  # noqa: F811
    """Fields 1 to 3 words past a 16-byte boundary, at the sizes where the
    array's first and last 16-byte units are cut (a last block of one to three
    values may not fill its first unit)."""
    x = (np.random.default_rng(n + offset).random((F, n)) * 100.0).astype(np.float32)
    assert_parity(gpz, oracle, x, 1e-2 if mode == 0 else 1e-4, mode, 3, offset=offset)

"""The 64-bit form's ways for a block, absolute bounds included: coded by the
fast kernel, stored raw by it (a value that is not finite), left to the general
kernel (values beyond the reach of its fixed point, which the first 512 values
of a field may already show).  Bit for bit against the oracle."""
import numpy as np
import pytest

from tests.test_wide_gpu import check_parity, gpz  # noqa: F401  (the fixture)

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("F", [1, 3, 6, 8])
@pytest.mark.parametrize("n", [5, 255, 256, 1023, 1024, 2 * 1024 + 300])
@pytest.mark.parametrize("mode", [0, 1])
@pytest.mark.parametrize("kind", ["nan_first", "inf_last", "nan_later", "far_first", "far_last", "wide_later",
                                  "nan_late", "wide_late"])
def test_block_routes(gpz, oracle, F, n, mode, kind):  # noqa: F811
    rng = np.random.default_rng(F * 1000 + n)
    x = rng.random((F, n)) * 100.0
    eb = 1e-9
    if kind == "nan_first":
        x[F - 1, ::700] = np.nan
    elif kind == "inf_last":
        x[0, -1] = -np.inf
    elif kind == "nan_later":
        x[F // 2, 260::1024] = np.nan
    elif kind == "far_first":  # |x| beyond 2^45 bounds from the first value on
        x[0] += 1e5
    elif kind == "far_last":
        x[F - 1, -1] = 1e5
    elif kind == "wide_later":  # a range beyond 2^40 steps
        x[0, 257::1024] = 3e3
    elif kind == "nan_late":  # behind the 512 values that tell most blocks
        x[F - 1, 600::1024] = np.nan
    else:
        x[0, 600::1024] = 3e3
    check_parity(gpz, oracle, x, eb if mode == 0 else 1e-12, mode, 3)


@pytest.mark.parametrize("F", [1, 4, 6])
@pytest.mark.parametrize("n", [1, 255, 1024, 1024 + 513])
def test_constant_fields(gpz, oracle, F, n):  # noqa: F811
    """Fields of one value per block, negative zero among them, with and without
    others beside them; streams whose blocks have hardly any words."""
    x = np.full((F, n), -2.5)
    x[F - 1] = -0.0
    check_parity(gpz, oracle, x, 1e-12, 0, 3)
    x[0] = np.random.default_rng(n).random(n)
    check_parity(gpz, oracle, x, 1e-12, 0, 3)

"""The fold of a range pass over its CTAs' extremes: every field count, one CTA
to the whole grid's, the extremes of each field in a block of their own and
some fields without a value; bit for bit against the oracle."""
import numpy as np
import pytest
import torch

from tests.test_parity_gpu import assert_parity, gpz  # noqa: F401  (the fixture)

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("F", range(1, 9))
@pytest.mark.parametrize("blocks", [0, 1, 9, 1300])
def test_range_fold(gpz, oracle, F, blocks):  # noqa: F811
    n = 1024 * blocks + 3
    rng = np.random.default_rng(100 * F + blocks)
    x = rng.random((F, n)).astype(np.float32)
    for f in range(F):
        lo, hi = rng.permutation(n)[:2]
        x[f, lo], x[f, hi] = -1.0 - f, 2.0 + f
    if F in (3, 7):
        x[1] = np.nan   # a field without a value
        x[F - 1] = -0.0
    assert_parity(gpz, oracle, x, 1e-3, 1, 3)
    if n <= 10 * 1024:  # the same pass over interleaved records
        s, _ = gpz.compress_aos(torch.from_numpy(np.ascontiguousarray(x.T)).cuda().view(-1), F, 1e-3, 1)
        rs, _ = oracle.compress(x, 1e-3, 1, 3)
        assert np.array_equal(s.cpu().numpy(), rs)

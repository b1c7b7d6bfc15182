"""The decoder's two groups of four positions per thread at the edges of its
halves, for records of at most 64 bits, up to 128 and wider, with few and many
runs, as fields and as interleaved records: bit for bit against the oracle."""
import numpy as np
import pytest
import torch

from tests.test_parity_gpu import assert_parity, gpz  # noqa: F401  (the fixture)

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("F,eb", [(1, 1e-2), (3, 1e-2), (6, 1e-2), (6, 1e-4), (8, 1e-5)])
@pytest.mark.parametrize("n", [4, 509, 512, 513, 517, 1024, 1024 + 515])
def test_group_edges(gpz, oracle, F, eb, n):  # noqa: F811
    rng = np.random.default_rng(F * 10000 + n)
    x = (rng.random((F, n)) * 100.0).astype(np.float32)
    if n > 600:
        x[:3, :400] = 1.0  # one long run
    s, _, o = assert_parity(gpz, oracle, x, eb, 0, 3)
    rec = gpz.decompress_aos(torch.from_numpy(s.copy()).cuda(), F, n)
    assert np.array_equal(rec.cpu().numpy().view(np.uint32), o.T.copy().view(np.uint32))

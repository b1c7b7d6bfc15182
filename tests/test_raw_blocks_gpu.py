"""Blocks stored raw, in every form of output, at block sizes around what a
thread takes at once and what the decoder stages (all of a block of up to four
fields, a part of a wider one): the values come back bit for bit."""
import numpy as np
import pytest
import torch

from tests.test_parity_gpu import assert_parity, gpz  # noqa: F401  (the fixture)

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("F", [1, 3, 4, 5, 8])
@pytest.mark.parametrize("n", [1, 2, 5, 127, 129, 1023, 1024, 1024 + 700])
@pytest.mark.parametrize("offset", [0, 1])
@pytest.mark.parametrize("mode", [0, 1])
def test_raw_blocks(gpz, oracle, F, n, offset, mode):  # noqa: F811
    x = np.random.default_rng(F * 10000 + n).standard_normal((F, n)).astype(np.float32)
    x[0, -1] = -0.0
    x[F - 1, ::600] = np.inf
    s, _, o = assert_parity(gpz, oracle, x, 1e-2, mode, 3, offset=offset)
    bits = x.view(np.uint32)
    assert np.array_equal(o.view(np.uint32), bits)
    st = torch.from_numpy(s.copy()).cuda()
    rec = torch.zeros(n * F + 1, device="cuda")
    for at in (0, 1):  # compressed from records, one word past a 16-byte boundary too
        rec[at:at + n * F] = torch.from_numpy(x.T.copy()).cuda().view(-1)
        assert torch.equal(gpz.compress_aos(rec[at:at + n * F], F, 1e-2, mode, 3)[0], st)
    assert np.array_equal(gpz.decompress_aos(st, F, n).cpu().numpy().view(np.uint32), bits.T)
    assert np.array_equal(gpz.decompress_f64(st, F, n).cpu().numpy().view(np.uint64), x.astype(np.float64).view(np.uint64))
    out = torch.zeros(n * F + 1, device="cuda")  # records one word past a 16-byte boundary
    status = gpz.lib.gpz_decompress_aos(st.data_ptr(), st.numel(), out[1:].data_ptr(), F, n, None, 0, None)
    assert status == gpz.OK
    assert np.array_equal(out[1:].cpu().numpy().view(np.uint32).reshape(n, F), bits.T)

"""Calls one behind the other on one stream, enqueued and replayed from a CUDA graph,
each on a workspace left full of ones: dependent launches and the clearing of
what a call counts in hold together across calls, and give the oracle's stream and values."""
import numpy as np
import pytest
import torch

from tests.test_parity_gpu import gpz  # noqa: F401  (the fixture)

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("graph", [False, True])
@pytest.mark.parametrize("offset", [0, 1])
@pytest.mark.parametrize("flags", [0, 1])
@pytest.mark.parametrize("F,n,mode,eb", [(3, 1, 0, 1e-2), (3, 5000, 0, 1e-2), (6, 70 * 1024 + 3, 1, 1e-4),
                                         (1, 300 * 1024, 1, 1e-3)])
def test_calls_on_a_used_workspace(gpz, oracle, F, n, mode, eb, flags, offset, graph):  # noqa: F811
    rng = np.random.default_rng(F * 1000 + n % 97)
    x = (rng.random((F, n)) * 100.0).astype(np.float32)
    rs, _ = oracle.compress(x, eb, mode, 3)
    rv = oracle.decompress(rs, F, n)
    hold = torch.zeros(F, ((n + 3) & ~3) + 4, dtype=torch.float32, device="cuda")
    hold[:, offset:offset + n] = torch.from_numpy(x).cuda()
    fields = [hold[f, offset:offset + n] for f in range(F)]
    c = gpz.Compressor(n, F, eb, mode, 3, flags=flags)
    d = gpz.Decompressor(n, F)

    def calls():
        c.ws.fill_(255)
        d.ws.fill_(255)
        c(fields, sync=False)
        d(c.out, rs.size, check=False)

    torch.cuda.synchronize()
    s = torch.cuda.Stream()
    with torch.cuda.stream(s):
        calls()
        s.synchronize()
        if graph:
            g = torch.cuda.CUDAGraph()
            with torch.cuda.graph(g, stream=s):
                calls()
            again = g.replay
        else:
            again = calls
        for _ in range(3):
            c.out.zero_()
            d.out.zero_()
            again()
            s.synchronize()
            assert gpz.gpz_sync_status(c.ws) == 0 and gpz.gpz_sync_status(d.ws) == 0
            assert int(c.d_size.item()) == rs.size and np.array_equal(c.out[:rs.size].cpu().numpy(), rs)
            assert np.array_equal(d.out[:, :n].cpu().numpy().view(np.uint32), rv.view(np.uint32))


@pytest.mark.parametrize("mode,eb", [(0, 1e-2), (1, 1e-3)])
def test_records_from_a_graph(gpz, oracle, mode, eb):  # noqa: F811
    F, n = 4, 9 * 1024 + 5
    x = (np.random.default_rng(5).random((F, n)) * 50.0).astype(np.float32)
    rs, _ = oracle.compress(x, eb, mode, 3)
    rec = torch.from_numpy(np.ascontiguousarray(x.T)).cuda()
    p = gpz.make_params(F, eb, mode, 3)
    out = torch.empty(gpz.gpz_bound_size(n, F), dtype=torch.uint8, device="cuda")
    ws = torch.empty(gpz.gpz_compress_aos_workspace_size(n, F), dtype=torch.uint8, device="cuda")

    def call():
        ws.fill_(255)
        assert gpz.lib.gpz_compress_aos(rec.data_ptr(), n, p, out.data_ptr(), out.numel(), None, None, None,
                                        ws.data_ptr(), ws.numel(), gpz._stream_handle(None)) == 0

    s = torch.cuda.Stream()
    with torch.cuda.stream(s):
        call()
        s.synchronize()
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g, stream=s):
            call()
        for _ in range(2):
            out.zero_()
            g.replay()
            s.synchronize()
            assert np.array_equal(out[:rs.size].cpu().numpy(), rs)

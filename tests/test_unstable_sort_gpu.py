"""What becomes of a block whose sorted order fails its check (gpz_test.h: every
encoded block treated so): the general kernel redoes it, once, and the stream and
permutation are the ordinary ones.  Fields of any alignment, records, doubles
and a batch; keys ranked by match and by shared atomics; blocks that took
fallback candidates before their sort failed."""
import ctypes as C

import numpy as np
import pytest
import torch

from tests.test_fallback_routes_gpu import EB, blocks
from tests.test_parity_gpu import gpz  # noqa: F401  (the fixture)

pytestmark = pytest.mark.gpu

NB = 64  # the list's 64 words end where the next section begins
FIELDS, RECORDS, WIDE, BATCH = range(4)


def data(kind):
    if kind == "fallback":
        return blocks("coded", NB, 5), EB
    n = (NB - 1) * 1024 + 333
    rng = np.random.default_rng(6)
    x = rng.random((3, n)) * 100.0
    if kind == "runs":
        x[:, :] = np.repeat(x[:, ::64], 64, axis=1)[:, :n]
    return x.astype(np.float32), 1e-2


@pytest.mark.parametrize("kind", ["spread", "runs", "fallback"])
@pytest.mark.parametrize("form,offset,mode", [(FIELDS, 0, 0), (FIELDS, 0, 1), (FIELDS, 1, 0), (FIELDS, 1, 1),
                                              (RECORDS, 0, 0), (WIDE, 0, 0), (BATCH, 0, 0), (BATCH, 1, 1)])
def test_failed_checks_go_to_the_general_kernel_once(gpz, oracle, form, offset, mode, kind):  # noqa: F811
    x, eb = data(kind)
    n = x.shape[1]
    if mode == 1:
        eb = [eb / float(x[f].max() - x[f].min()) for f in range(3)]
    if form == WIDE:
        x = x.astype(np.float64)
        ref, rperm, _ = oracle.compress_wide(x, eb, mode, 3)
    else:
        ref, rperm = oracle.compress(x, eb, mode, 3)
    buf = torch.zeros((3, n + 4), dtype=torch.float64 if form == WIDE else torch.float32, device="cuda")
    buf[:, offset:offset + n] = torch.from_numpy(x)
    fields = [buf[f, offset:offset + n] for f in range(3)]
    if form == RECORDS:
        fields = [torch.from_numpy(x.T.copy()).cuda()]
    cap = gpz.gpz_bound_size_wide(n, 3)
    out = torch.zeros(cap, dtype=torch.uint8, device="cuda")
    perm = torch.zeros(n, dtype=torch.int32, device="cuda")
    ws = torch.empty(int(gpz.lib.gpz_test_unstable_sort_workspace_size(n)), dtype=torch.uint8, device="cuda")
    size, listed = C.c_uint64(0), C.c_uint32(0)
    status = gpz.lib.gpz_test_unstable_sort(
        form, (C.c_void_p * 3)(*[f.data_ptr() for f in fields]), n, C.byref(gpz.make_params(3, eb, mode, 3)),
        out.data_ptr(), cap, C.byref(size), perm.data_ptr(), ws.data_ptr(), ws.numel(), C.byref(listed),
        torch.cuda.current_stream().cuda_stream)
    assert status == gpz.OK
    assert listed.value == NB
    got = out[:size.value].cpu().numpy()
    assert got.size == ref.size and np.array_equal(got, ref)
    assert np.array_equal(perm.cpu().numpy().astype(np.uint32), rperm)

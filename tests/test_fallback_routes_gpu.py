"""Blocks whose first candidates do not suffice, by what becomes of them: coded in
place, left to the general kernel (a fallback candidate could change the code
width) or stored raw (no candidate passes).  Which of these a block takes is
worked out here from the format's rule in numpy."""
import numpy as np
import pytest
import torch

from tests.test_parity_gpu import gpz  # noqa: F401  (the fixture)

BLOCK = 1024
EB = 0.5
STEP = EB * 1.96875
BITS = 18  # codes of 18 bits: their fp32 quotients err by up to 2^-7 of a step


def route(x, eb):
    """One block of one field: "first", "coded", "general" or "raw" (multiply-adds
    rounded once through float64, whose products are exact)."""
    f32, f64 = np.float32, np.float64
    s = f32(eb * 1.96875)
    inv = f32(1.0 / f64(s))
    chk = f32(eb * (1.0 - 2.0 ** -22))
    if f64(chk) > eb * (1.0 - 2.0 ** -22):
        chk = np.nextafter(chk, f32(0))
    mn = x.min()
    q = np.floor(((x - mn).astype(f64) * f64(inv) + 0.5).astype(f32)).astype(f64)

    def ok(c):
        return np.abs(x - (c * f64(s) + f64(mn)).astype(f32)) <= chk

    fail = ~ok(q)
    down = fail & (q > 0) & ok(q - 1)
    up = fail & ~down & ok(q + 1)
    if (fail & ~down & ~up).any():
        return "raw"
    width = int(q.max()).bit_length()
    if (down & (q == (1 << width) >> 1)).any() or (up & (q == (1 << width) - 1)).any():
        return "general"
    return "coded" if fail.any() else "first"


def blocks(kind, count, seed):
    """[3, 1024 * count] fp32 values whose first field takes the route in every
    block; the other fields' first candidates pass."""
    rng = np.random.default_rng(seed)
    x = rng.random((3, count * BLOCK)) * 50.0
    for b in range(count):
        at = slice(b * BLOCK, (b + 1) * BLOCK)
        while True:
            if kind == "coded":
                v = rng.random(BLOCK) * 0.9 * 2 ** BITS * STEP
            elif kind == "general":  # around the step where the codes get their last bit
                v = (2 ** (BITS - 1) - 0.5 + 0.04 * (rng.random(BLOCK) - 0.5)) * STEP
            else:  # four times the codes: the values' own rounding is a good part of the bound
                v = rng.random(BLOCK) * 0.9 * 2 ** (BITS + 2) * STEP
            v[7], v[900] = 0.0, 0.9 * 2 ** BITS * STEP
            if route(v.astype(np.float32), EB) == kind:
                break
        x[0, at] = v
    return x.astype(np.float32)


def test_routes_are_reached():
    for kind in ("coded", "general", "raw"):
        x = blocks(kind, 3, 1)
        for f in range(3):
            for b in range(3):
                assert route(x[f, b * BLOCK:(b + 1) * BLOCK], EB) == (kind if f == 0 else "first")


def counts(ws):
    words = ws[:64].view(torch.int32).cpu().numpy()
    return int(words[3]), int(words[6])  # warps with fallback candidates, blocks listed


@pytest.mark.gpu
@pytest.mark.parametrize("kind", ["coded", "general", "raw"])
@pytest.mark.parametrize("offset", [0, 1])
@pytest.mark.parametrize("mode", [0, 1])
def test_a_block_is_listed_once_and_only_when_left(gpz, oracle, kind, offset, mode):  # noqa: F811
    """64 blocks: the list, one word per block, ends where the slots begin."""
    nb = 64
    x = blocks(kind, nb, 2)
    n = x.shape[1]
    eb = [EB / float(x[f].max() - x[f].min()) for f in range(3)] if mode else EB
    buf = torch.zeros(3, n + 8, device="cuda")
    buf[:, offset:offset + n] = torch.from_numpy(x)
    c = gpz.Compressor(n, 3, eb, mode, 3, want_perm=True)
    size = c([buf[f, offset:offset + n] for f in range(3)])
    warps, listed = counts(c.ws)
    ref, perm = oracle.compress(x, eb, mode, 3)
    assert np.array_equal(c.out[:size].cpu().numpy(), ref)
    assert np.array_equal(c.perm[:n].cpu().numpy().astype(np.uint32), perm)
    if mode == 0:  # the bound, and so every block's route, is the one worked out
        assert listed == (0 if kind == "coded" else nb)
        assert nb <= warps <= 4 * nb


@pytest.mark.gpu
@pytest.mark.parametrize("kind", ["coded", "general", "raw"])
@pytest.mark.parametrize("offset", [0, 1, 2, 3])
def test_routes_in_records_and_batches(gpz, oracle, kind, offset):  # noqa: F811
    """The same blocks as records, and as a chunk of a batch beside one that
    takes the ordinary way, from every word of a 16-byte unit."""
    x = blocks(kind, 5, 3 + offset)[:, :5 * BLOCK - 100]
    n = x.shape[1]
    ref, perm = oracle.compress(x, EB, 0, 3)
    rec = torch.zeros(3 * n + 4, device="cuda")
    rec[offset:offset + 3 * n] = torch.from_numpy(x.T.copy()).cuda().view(-1)
    got, p = gpz.compress_aos(rec[offset:offset + 3 * n], 3, EB, 0, 3, want_perm=True)
    assert np.array_equal(got.cpu().numpy(), ref)
    assert np.array_equal(p.cpu().numpy().astype(np.uint32), perm)
    y = (np.random.default_rng(7).random((3, 3000)) * 50.0).astype(np.float32)
    chunks, refs = [], []
    for v, at in ((y, 0), (x, offset)):
        buf = torch.zeros(3, v.shape[1] + 8, device="cuda")
        buf[:, at:at + v.shape[1]] = torch.from_numpy(v)
        chunks.append(([buf[f, at:at + v.shape[1]] for f in range(3)], gpz.make_params(3, EB, 0, 3)))
        refs.append(oracle.compress(v, EB, 0, 3)[0])
    c = gpz.BatchCompressor(chunks)
    c()
    assert c.status()[0] == gpz.OK
    for s, r in zip(c.streams(), refs):
        assert np.array_equal(s.cpu().numpy(), r)

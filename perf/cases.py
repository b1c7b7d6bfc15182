"""The workloads this library's speed is judged by, each through its public entry points.

A case is a dict of plain values; ``listed()`` gives the fixed ones and
``draw(rng)`` more of the same ranges.  The data is drawn by the package's own
generators (``paper_2508_10305_gb300.synth``): points uniform in a box, a
cosmology-like snapshot (positions, then velocities) and a LiDAR-like scan.

``api`` names the entry points of a case:

  call      compress() / decompress(): one-shot calls that allocate their
            buffers and wait for the result, as a script or notebook does;
  held      Compressor / Decompressor objects whose buffers are held, as a
            simulation's output step or a reader of many snapshots does; the
            calls are enqueued only (the size stays on the device);
  records   gpz_compress_aos / gpz_decompress_aos: interleaved point records;
  fp64      gpz_compress_f64 / gpz_decompress_f64: doubles whose bound fp32 can hold;
  wide      gpz_compress_wide / gpz_decompress_wide: doubles at a bound it cannot
            (these three with buffers the program keeps, as a C program does);
  batch     batched plans (gpz_batch_*, BatchDecompressor) over many arrays.

``op`` is "compress" (write), "decompress" (read) or "both": one snapshot is
written and a stored one read, as a restart or a rewriting tool does.  The
stored stream is made in ``prepare``.
"""
import ctypes as C
import math

import torch

from paper_2508_10305_gb300 import gpz, synth

HEADER_WORDS = 16
BLOCK = 1024


def _case(name, api, op, data, n, F, eb, rel, perm=False, chunks=0, seg_bits=3):
    c = {"api": api, "op": op, "data": data, "n": int(n), "fields": int(F), "eb": float(eb), "relative": bool(rel),
         "perm": bool(perm), "chunks": int(chunks), "seg_bits": int(seg_bits)}
    if name:
        c["name"] = name
    return c


def listed():
    return [
        # the smallest arrays of the batched workload, called one at a time: latency and launches
        _case("call_10k", "call", "both", "uniform", 10007, 3, 1e-2, False),
        # the small configuration: a million points in a box, absolute bound
        _case("box_1m", "held", "both", "uniform", 1000000, 3, 1e-2, False),
        # the headline snapshot: 64M particles, positions and velocities, relative bound
        _case("snapshot_64m_write", "held", "compress", "cosmology", 1 << 26, 6, 1e-4, True),
        _case("snapshot_64m_read", "held", "decompress", "cosmology", 1 << 26, 6, 1e-4, True),
        # an airborne scan: 200M points in acquisition order, absolute bound of a millimetre
        _case("scan_200m_write", "held", "compress", "lidar", 200000000, 3, 1e-3, False),
        _case("scan_200m_read", "held", "decompress", "lidar", 200000000, 3, 1e-3, False),
        # a snapshot of whatever size the run has (rows of an [F, n] array then start
        # anywhere), written with the permutation, e.g. to reorder particle ids
        _case("odd_10m_write", "held", "compress", "cosmology", 9999991, 6, 1e-3, True, perm=True),
        _case("odd_10m_read", "held", "decompress", "cosmology", 9999991, 6, 1e-3, True),
        # point records as they lie in a file
        _case("records_16m", "records", "both", "lidar", 16777259, 3, 1e-3, False),
        # a solver's doubles, at a bound fp32 can hold and at one it cannot
        _case("fp64_8m", "fp64", "both", "cosmology", 1 << 23, 6, 1e-4, True),
        _case("wide_4m", "wide", "both", "cosmology", 4000037, 6, 1e-12, True),
        # many arrays of 10 thousand to 4 million particles in a few launches
        _case("batch_128", "batch", "both", "mixed", 4000000, 6, 1e-4, True, chunks=128),
    ]


def _log_uniform(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    api = rng.choice(["call", "held", "held", "held", "held", "records", "fp64", "wide", "batch"])
    if api == "batch":
        return _case(None, "batch", "both", "mixed", _log_uniform(rng, 20000, 4000000), 6,
                     rng.choice([1e-3, 1e-4]), True, chunks=rng.randint(8, 128))
    data = rng.choice(["uniform", "cosmology", "lidar"])
    if api in ("fp64", "wide"):
        data = rng.choice(["uniform", "cosmology"])
    F = {"uniform": 3, "lidar": 3, "cosmology": rng.choice([3, 4, 6, 6])}[data]
    hi = {"call": 10 ** 6, "held": 6 * 10 ** 7, "records": 3 * 10 ** 7, "fp64": 10 ** 7, "wide": 4 * 10 ** 6}[api]
    n = _log_uniform(rng, 10 ** 4, hi)
    if rng.random() < 0.4:
        n = (n + 3) // 4 * 4
    if api == "wide":
        rel, eb = True, rng.choice([1e-11, 1e-12])
    elif data == "cosmology":
        rel, eb = True, rng.choice([1e-3, 1e-4, 1e-5])
    else:
        rel, eb = False, rng.choice([1e-2, 1e-3])
    op = rng.choice(["compress", "decompress"]) if api == "held" else "both"
    return _case(None, api, op, data, n, F, eb, rel, perm=op != "decompress" and api == "held" and rng.random() < 0.3,
                 seg_bits=rng.choice([3, 3, 3, 2]))


# ----------------------------------------------------------------------------- inputs

def _draw_data(data, n, F, seed, dev):
    """[F, n] float32."""
    if data == "uniform":
        return synth.uniform_box_torch(n, seed=seed, device=dev)[:F]
    if data == "lidar":
        return synth.lidar(n, seed=seed, device=dev)
    halos = max(4, int(round(20000 * n / 2 ** 26)))
    x = synth.cosmology(n, seed=seed, n_halos=halos, device=dev)
    return x if F == 6 else x[:F].contiguous()


def _mode(case):
    return gpz.EB_REL if case["relative"] else gpz.EB_ABS


def _chunk_sizes(case):
    """The batch's particle counts: log-uniform, the same for every seed."""
    return [int(v) for v in synth.chunk_sizes(case["chunks"], 10000, case["n"], seed=4)]


def _chunk_fields(case, c):
    return 3 if c % 2 else 6


def _batch_data(case, seed, dev):
    """The chunks' [F, n] views of one pool per field count, each starting on a
    128-byte boundary: 3 fields uniform in a box, 6 fields of a snapshot."""
    sizes = _chunk_sizes(case)
    out = [None] * len(sizes)
    for F in (3, 6):
        idx = [c for c in range(len(sizes)) if _chunk_fields(case, c) == F]
        if not idx:
            continue
        pad = [-(-sizes[c] // 32) * 32 for c in idx]
        pool = _draw_data("uniform" if F == 3 else "cosmology", sum(pad), F, seed, dev)
        o = 0
        for c, p in zip(idx, pad):
            out[c] = pool[:, o:o + sizes[c]]
            o += p
    return out


class _Held:
    """Buffers a C or Python program keeps for its own calls of one shape: the
    stream buffer, the workspaces, the size word and the decoded values."""

    def __init__(self, api, n, F, dev, shape, dtype):
        L = gpz.lib
        cap, cws, dws = {
            "records": (L.gpz_bound_size, L.gpz_compress_aos_workspace_size, L.gpz_decompress_aos_workspace_size),
            "fp64": (L.gpz_bound_size_wide, L.gpz_compress_f64_workspace_size, L.gpz_decompress_f64_workspace_size),
            "wide": (L.gpz_bound_size_wide, L.gpz_compress_wide_workspace_size, lambda n, F: 256)}[api]
        self.capacity = int(cap(n, F))
        self.stream = torch.zeros(self.capacity, dtype=torch.uint8, device=dev)
        self.size = torch.zeros(1, dtype=torch.int64, device=dev)
        self.ws = torch.empty(max(int(cws(n, F)), 256), dtype=torch.uint8, device=dev)
        self.dws = torch.empty(max(int(dws(n, F)), 256), dtype=torch.uint8, device=dev)
        self.values = torch.empty(shape, dtype=dtype, device=dev)
        self.used = (C.c_double * F)()


def _pointers(x):
    return (C.c_void_p * x.shape[0])(*[x[f].data_ptr() for f in range(x.shape[0])])


def _check(status, where):
    if status != gpz.OK:
        raise gpz.GpzError(status, where)


def _write(st):
    """One compression of st["x"] into st["held"] (enqueued; the size stays on the device)."""
    case, h, x = st["case"], st["held"], st["x"]
    call = {"records": gpz.lib.gpz_compress_aos, "fp64": gpz.lib.gpz_compress_f64,
            "wide": gpz.lib.gpz_compress_wide}[case["api"]]
    inp = x.data_ptr() if case["api"] == "records" else _pointers(x)
    used = () if case["api"] == "records" else (h.used,)
    _check(call(inp, case["n"], C.byref(st["params"]), h.stream.data_ptr(), h.capacity, h.size.data_ptr(), None, None,
                h.ws.data_ptr(), h.ws.numel(), *used, torch.cuda.current_stream().cuda_stream), call.__name__)


def _read(st):
    case, h = st["case"], st["held"]
    call = {"records": gpz.lib.gpz_decompress_aos, "fp64": gpz.lib.gpz_decompress_f64,
            "wide": gpz.lib.gpz_decompress_wide}[case["api"]]
    out = h.values.data_ptr() if case["api"] == "records" else _pointers(h.values)
    _check(call(st["stored"].data_ptr(), st["stored"].numel(), out, case["fields"], case["n"], h.dws.data_ptr(),
                h.dws.numel(), torch.cuda.current_stream().cuda_stream), call.__name__)


def _prepare_batch(case, st, seed, dev):
    """Two plans over the chunks, their streams and decoded values in pools."""
    xs = _batch_data(case, seed, dev)
    caps = [gpz.gpz_bound_size(x.shape[1], x.shape[0]) for x in xs]
    place = [0]
    for c in caps:
        place.append(place[-1] + -(-c // 256) * 256)
    streams = torch.zeros(place[-1], dtype=torch.uint8, device=dev)
    descs = []
    for c, x in enumerate(xs):
        d = gpz.gpz_compress_chunk()
        for f in range(x.shape[0]):
            d.fields[f] = x[f].data_ptr()
        # every other pair of chunks at a ten times coarser bound
        d.params = gpz.make_params(x.shape[0], case["eb"] * (10.0 if c & 2 else 1.0), _mode(case), case["seg_bits"])
        d.n, d.out, d.out_capacity = x.shape[1], streams.data_ptr() + place[c], caps[c]
        descs.append(d)
    status, comp = gpz.gpz_batch_create_compress(descs)
    _check(status, "gpz_batch_create_compress")
    ws = torch.empty(gpz.gpz_batch_workspace_size(comp), dtype=torch.uint8, device=dev)
    sizes = torch.zeros(len(xs), dtype=torch.int64, device=dev)
    _check(gpz.gpz_batch_run(comp, ws, ws.numel(), sizes, True), "gpz_batch_run")
    stored = [streams[place[c]:place[c] + v].clone() for c, v in enumerate(sizes.tolist())]
    pads = [-(-x.shape[1] // 32) * 32 for x in xs]
    values = torch.zeros(sum(p * x.shape[0] for p, x in zip(pads, xs)), dtype=torch.float32, device=dev)
    outs, o = [], 0
    for p, x in zip(pads, xs):
        outs.append(values[o:o + p * x.shape[0]].view(x.shape[0], p))
        o += p * x.shape[0]
    dec = gpz.BatchDecompressor([(s, s.numel(), x.shape[0], x.shape[1]) for s, x in zip(stored, xs)], device=dev, outs=outs)
    st.update(x=xs, comp=_Plan(comp), ws=ws, sizes=sizes, streams=streams, stored=stored, dec=dec, values=values)


class _Plan:
    def __init__(self, handle):
        self.handle = handle

    def __del__(self):
        gpz.gpz_batch_destroy(self.handle)


def prepare(case, seed):
    dev = torch.device("cuda")
    api, op, n, F = case["api"], case["op"], case["n"], case["fields"]
    eb, mode, G = case["eb"], _mode(case), case["seg_bits"]
    st = {"case": case}
    if api == "batch":
        _prepare_batch(case, st, seed, dev)
        return st
    x = _draw_data(case["data"], n, F, seed, dev)
    st["params"] = gpz.make_params(F, eb, mode, G)
    if api == "call":
        st["x"] = x
        st["stored"] = gpz.compress(x, eb, mode, G)[0].clone()
        st["file"] = torch.zeros(gpz.gpz_bound_size(n, F), dtype=torch.uint8, device=dev)
    elif api == "held":
        if op != "decompress":
            st["x"] = [x[f] for f in range(F)]
            st["comp"] = gpz.Compressor(n, F, eb, mode, G, want_perm=case["perm"], device=dev)
            st["comp"].out.zero_()
        if op != "compress":
            c = st.get("comp") or gpz.Compressor(n, F, eb, mode, G, device=dev)
            size = c([x[f] for f in range(F)])
            st["stored"] = c.out[:size].clone()
            st["dec"] = gpz.Decompressor(n, F, device=dev)
    else:
        if api == "records":
            st["x"] = x.t().contiguous()
        else:  # doubles near the fp32 values, not on them
            g = torch.Generator(device=dev)
            g.manual_seed(seed + 1)
            near = 1.0 + 1e-8 * torch.rand(x.shape, generator=g, device=dev, dtype=torch.float64)
            st["x"] = x.to(torch.float64) * near
        st["held"] = _Held(api, n, F, dev, st["x"].shape, st["x"].dtype)
        _write(st)
        st["stored"] = st["held"].stream[:int(st["held"].size.item())].clone()
    return st


def run(state):
    case = state["case"]
    api, op, n, F = case["api"], case["op"], case["n"], case["fields"]
    if api == "batch":
        _check(gpz.gpz_batch_run(state["comp"].handle, state["ws"], state["ws"].numel(), state["sizes"], True),
               "gpz_batch_run")
        state["dec"]()
        return {"streams": state["streams"], "sizes": state["sizes"], "fields": state["values"]}
    if api == "call":
        stream, _ = gpz.compress(state["x"], case["eb"], _mode(case), case["seg_bits"])
        state["file"][:stream.numel()] = stream  # the program's own copy
        return {"stream": state["file"], "size": stream.numel(), "fields": gpz.decompress(state["stored"], F, n)}
    if api == "held":
        out = {}
        if op != "decompress":
            comp = state["comp"]
            comp(state["x"], sync=False)
            out["stream"], out["size"] = comp.out, comp.d_size
            if case["perm"]:
                out["perm"] = comp.perm
        if op != "compress":
            out["fields"] = state["dec"](state["stored"], state["stored"].numel(), check=False)
        return out
    _write(state)
    _read(state)
    held = state["held"]
    out = {"stream": held.stream, "size": held.size, "fields": held.values}
    if api != "records":
        out["bounds"] = list(held.used)
    return out


# ----------------------------------------------------------------------------- necessary work

def _bits_per_value(case, data, eb):
    """Typical coded bits per value of the generators at a bound."""
    if case["api"] == "wide":
        return 35.4 + 3.32 * math.log10(1e-12 / eb)
    if data == "cosmology":
        return {1e-2: 3.3, 1e-3: 5.6, 1e-4: 8.9, 1e-5: 12.2}.get(eb, 8.9)
    if data == "lidar":
        return {1e-2: 7.9, 1e-3: 11.0}.get(eb, 11.0)
    # uniform: the range in steps of about 2 eb, less the segment bits the runs carry
    span = 1.0 if case["relative"] else 256.0
    return math.log2(span / (1.97 * eb)) - 1.8


def work(case):
    """Bytes: the values read (or written) once and the stream written (or
    read) once.  Flops: a subtraction and a multiply-add per coded value, a
    multiply-add per decoded one."""
    wide = case["api"] in ("fp64", "wide")
    if case["api"] == "batch":
        parts = [(v * _chunk_fields(case, c), "uniform" if _chunk_fields(case, c) == 3 else "cosmology",
                  case["eb"] * (10.0 if c & 2 else 1.0)) for c, v in enumerate(_chunk_sizes(case))]
    else:
        parts = [(case["n"] * case["fields"], case["data"], case["eb"])]
    values = sum(p[0] for p in parts)
    stream = sum(p[0] * _bits_per_value(case, p[1], p[2]) / 8.0 for p in parts)
    ways = 2 if case["op"] == "both" else 1
    nbytes = ways * (values * (8.0 if wide else 4.0) + stream)
    if case["perm"]:
        nbytes += 4.0 * case["n"]
    flops = values * ({"both": 5.0, "compress": 3.0, "decompress": 2.0}[case["op"]])
    return {"bytes": int(nbytes), "flops": int(flops)}


# ----------------------------------------------------------------------------- 64-bit values

def _bits_at(words, pos, width):
    """`width` (tensor, <= 53) bits at bit position pos of an int64 array of 32-bit words."""
    wi, sh = pos >> 5, pos & 31
    last = words.numel() - 1
    w0 = words[wi.clamp(max=last)]
    w1 = words[(wi + 1).clamp(max=last)]
    w2 = words[(wi + 2).clamp(max=last)]
    v = (w0 >> sh) | (w1 << (32 - sh))
    # the third word's bits start at bit 64 - sh
    v = v | torch.where(sh > 0, w2 << (64 - sh).clamp(max=63), torch.zeros_like(w2))
    return v & ((torch.ones_like(v) << width) - 1)


def _reconstruct(stream, n, F, wide=False):
    """[F, n] float64: the values a stream stands for, min + code * step in 64
    bits, by plain tensor operations on the stream's words."""
    words = stream.view(torch.int32).to(torch.int64) & 0xFFFFFFFF
    dev = words.device
    P = min(F, 3)
    G = int(words[3])
    nb = -(-n // BLOCK)
    ext = (4 if wide else 2) * F
    head = words[HEADER_WORDS:HEADER_WORDS + ext]

    def doubles(w):
        return ((w[..., 1::2] << 32) | w[..., 0::2]).contiguous().view(torch.float64)

    def floats(w):
        return torch.where(w >= 1 << 31, w - (1 << 32), w).to(torch.int32).view(torch.float32).to(torch.float64)

    step = doubles(head)[1::2] if wide else floats(head[1::2])
    table = words[HEADER_WORDS + ext:HEADER_WORDS + ext + nb + 1]
    base = HEADER_WORDS + ext + nb + 1
    out = torch.empty((F, nb * BLOCK), dtype=torch.float64, device=dev)
    j = torch.arange(BLOCK, device=dev)
    k = torch.arange(512, device=dev)
    mw = 2 if wide else 1
    hdr = 1 + mw * F + (F + 3) // 4
    for lo in range(0, nb, 2048):
        off = table[lo:min(lo + 2048, nb)] + base
        B = off.numel()
        blocks = torch.arange(lo, lo + B, device=dev)
        nbk = torch.where(blocks == nb - 1, n - (nb - 1) * BLOCK, BLOCK)
        mode = words[off]
        raw = (mode & 1) == 1
        U, wd, wc = (mode >> 1) & 0x7FF, (mode >> 12) & 31, (mode >> 17) & 31
        U = torch.where(raw, 1, U)
        wd, wc = torch.where(raw, 0, wd), torch.where(raw, 0, wc)
        at = lambda i: words[(off[:, None] + i).clamp(max=words.numel() - 1)]
        mins = at(1 + torch.arange(mw * F, device=dev))
        mins = doubles(mins) if wide else floats(mins)
        wb = at(1 + mw * F + torch.arange((F + 3) // 4, device=dev))
        bits = torch.stack([(wb[:, f >> 2] >> (8 * (f & 3))) & 0xFF for f in range(F)])
        bits = torch.where(raw[None, :], 0, bits)
        g = torch.stack([bits[f].clamp(max=G) if f < P else torch.zeros_like(bits[f]) for f in range(F)])
        wf = bits - g
        W = wf.sum(0)
        dstart = (off + hdr) * 32
        cstart = dstart + (U * wd + 31) // 32 * 32
        rstart = cstart + (U * wc + 31) // 32 * 32
        live = k[None, :] < U[:, None]
        delta = torch.where(live, _bits_at(words, dstart[:, None] + k * wd[:, None], wd[:, None].expand(B, 512)), 0)
        count = torch.where(live, _bits_at(words, cstart[:, None] + k * wc[:, None], wc[:, None].expand(B, 512)), 0)
        ids, ends = delta.cumsum(1), count.cumsum(1)
        run = torch.searchsorted(ends, j.expand(B, BLOCK).contiguous(), right=True).clamp(max=511)
        key = ids.gather(1, run)
        pos = rstart[:, None] + j * W[:, None]
        for f in range(F - 1, -1, -1):
            q = _bits_at(words, pos, wf[f][:, None].expand(B, BLOCK))
            pos = pos + wf[f][:, None]
            if f < P:
                q = q | ((key & ((1 << g[f]) - 1)[:, None]) << wf[f][:, None])
                key = key >> g[f][:, None]
            v = mins[:, f, None] + q.to(torch.float64) * step[f]
            if bool(raw.any()):
                p = (off[:, None] + 1 + mw * (f * nbk[:, None] + j)).clamp(max=words.numel() - mw)
                r = ((words[p + 1] << 32) | words[p]).view(torch.float64) if wide else floats(words[p])
                v = torch.where(raw[:, None], r, v)
            out[f, lo * BLOCK:(lo + B) * BLOCK] = v.reshape(-1)
    return out[:, :n]


def _bounds64(x, case):
    """The bounds the fp64 entry points work with."""
    out = []
    for f in range(x.shape[0]):
        eb = case["eb"] * float(x[f].max() - x[f].min()) if case["relative"] else case["eb"]
        if case["api"] == "fp64":
            eb -= float((x[f] - x[f].to(torch.float32).to(torch.float64)).abs().max())
        out.append(eb)
    return out


def exact(case, seed):
    """What run returns, in 64 bits: the values the stored streams stand for.
    Streams, sizes and permutations are whole numbers: None."""
    api, op, n, F = case["api"], case["op"], case["n"], case["fields"]
    if op == "compress":
        return None
    st = prepare(case, seed)
    if api == "batch":
        values = torch.zeros(st["values"].shape, dtype=torch.float64, device=st["values"].device)
        o = 0
        for s, x in zip(st["stored"], st["x"]):
            f, m = x.shape
            pad = -(-m // 32) * 32
            values[o:o + f * pad].view(f, pad)[:, :m] = _reconstruct(s, m, f)
            o += f * pad
        return {"streams": None, "sizes": None, "fields": values}
    v = _reconstruct(st["stored"], n, F, wide=api == "wide")
    out = {"fields": v.t().contiguous() if api == "records" else v}
    if op == "both":
        out["stream"], out["size"] = None, None
    if api in ("fp64", "wide"):
        out["bounds"] = _bounds64(st["x"], case)
    return out

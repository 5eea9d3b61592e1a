"""The decodes that the framework is measured on, and how to run one of them.

Codes and frames are the seeded stand-ins of `paper_2508_03567_gb300.inputs`: regular
(d_v, d_c) codes over GF(q), codewords of random information symbols, BPSK over AWGN,
drawn on the GPU.  A program keeps its code handle (and, for a mixed batch, its output
buffers and workspace) and hands new frames to it; that is what `prepare` returns.
"""
from __future__ import annotations

import torch

from paper_2508_03567_gb300 import binding, inputs

DEV = "cuda"
CHUNK = 2048          # frames generated at a time
ITERS_STOPPED = 8     # iterations a frame is counted with in work() when it may stop early


def _minmax(name, q, n, dv, dc, frames, lo, hi, iters=20, stop=True, bits=8):
    return dict(name=name, path="minmax", q=q, n=n, dv=dv, dc=dc, frames=frames, iters=iters, stop=stop, bits=bits,
                ebn0_lo=lo, ebn0_hi=hi)


def _fftspa(name, q, n, dv, dc, frames, lo, hi, iters=20, stop=True, app=False):
    return dict(name=name, path="fftspa", q=q, n=n, dv=dv, dc=dc, frames=frames, iters=iters, stop=stop, app=app,
                ebn0_lo=lo, ebn0_hi=hi)


def listed():
    return [
        # one frame of the benchmark's code as it comes off a receiver: nothing but latency
        _minmax("gf64 one frame", 64, 576, 2, 4, 1, 2.0, 2.0),
        # one middling request of the serving loop (1 to 256 frames), fewer frames than the chip has room for
        _minmax("gf64 request", 64, 576, 2, 4, 96, 1.5, 3.5, iters=30),
        # the benchmark's code at throughput: a long recording, 1.5 to 2.5 dB
        _minmax("gf64 batch", 64, 576, 2, 4, 16384, 1.5, 2.5),
        # the same code with the wider messages that take reliabilities of a wider range
        _minmax("gf64 batch 16-bit", 64, 576, 2, 4, 4096, 1.5, 2.5, bits=16),
        # the short GF(4) code: 1000 frames, ten fixed iterations, a call of a few microseconds
        _minmax("gf4 short code", 4, 48, 2, 4, 1000, 3.0, 3.0, iters=10, stop=False),
        # the longest code of the set, a small field
        _minmax("gf16 batch", 16, 1024, 2, 4, 4096, 1.5, 3.5, iters=30),
        # the (3, 6) code: three edges to a variable, an odd number of frames
        _minmax("gf32 batch", 32, 600, 3, 6, 2999, 1.5, 3.5, iters=30),
        # a few frames of the largest field
        _minmax("gf256 request", 256, 128, 2, 8, 17, 1.5, 3.5, iters=30),
        # the largest field at throughput, the benchmark's rate-2/3 code
        _minmax("gf256 batch", 256, 384, 2, 6, 4096, 2.5, 2.5),
        # what the serving loop launches: requests of four codes in one call
        dict(name="mixed batch", path="batch", iters=30, stop=True, ebn0_lo=1.5, ebn0_hi=3.5,
             jobs="16,1024,2,4,260 64,576,2,4,2749 32,600,3,6,196 256,128,2,8,2210"),
        # the second decoder on the benchmark's code and channel
        _fftspa("fft-spa gf64 batch", 64, 576, 2, 4, 8192, 1.5, 2.5),
        # the second decoder inside a larger receiver: some frames, a few iterations, soft outputs
        _fftspa("fft-spa gf16 soft", 16, 1024, 2, 4, 200, 2.0, 3.0, iters=5, stop=False, app=True),
    ]


# (d_v, d_c) pairs and the code lengths of each field order, short to long
_DEGREES = ((2, 4), (2, 4), (2, 6), (3, 6), (2, 8))
_LENGTHS = {2: (64, 1536), 4: (48, 1024), 8: (64, 1024), 16: (64, 1024), 32: (64, 768), 64: (64, 640), 128: (96, 384),
            256: (96, 384)}


def _spread(rng, lo, hi):
    """A whole number between lo and hi, spread over the logarithm."""
    return max(lo, min(hi, int(round(lo * (hi / lo) ** rng.random()))))


def _draw_code(rng, orders):
    q = rng.choice(orders)
    dv, dc = rng.choice(_DEGREES)
    lo, hi = _LENGTHS[q]
    n = _spread(rng, max(lo, 16 * dc), hi)
    step = dc // 2 if dv == 2 else dc // 3      # n d_v is a multiple of d_c
    return q, n // step * step, dv, dc


def _most_frames(q, n, dv, dc):
    """Frames that cost no more than the largest listed case: by the symbols of all messages, fields below
    GF(16) as GF(16)."""
    return max(8, min(60000, int(2048 * 1152 * 64 / (n * dv * max(q, 16)))))


def draw(rng):
    kind = rng.random()
    lo = round(rng.uniform(1.5, 2.5), 2)
    hi = round(lo + rng.choice((0.0, 1.0)), 2)
    iters = rng.choice((10, 20, 30))
    if kind < 0.15:
        jobs = []
        for _ in range(rng.randint(2, 6)):
            q, n, dv, dc = _draw_code(rng, (4, 8, 16, 32, 64, 64, 128, 256))
            jobs.append("%d,%d,%d,%d,%d" % (q, n, dv, dc, _spread(rng, 1, max(2, _most_frames(q, n, dv, dc) // 8))))
        return dict(path="batch", iters=iters, stop=True, ebn0_lo=lo, ebn0_hi=hi, jobs=" ".join(jobs))
    q, n, dv, dc = _draw_code(rng, (2, 4, 8, 16, 32, 64, 64, 64, 128, 256, 256))
    frames = _spread(rng, 1, _most_frames(q, n, dv, dc))
    if kind < 0.4:
        if rng.random() < 0.5:
            c = _fftspa("", q, n, dv, dc, min(frames, 2000), lo, hi, iters=rng.randint(1, 6), stop=False, app=True)
        else:
            c = _fftspa("", q, n, dv, dc, frames, lo, hi, iters=iters)
    else:
        c = _minmax("", q, n, dv, dc, frames, lo, hi, iters=iters, stop=rng.random() < 0.8,
                    bits=16 if rng.random() < 0.15 else 8)
    del c["name"]
    return c


# ---------------------------------------------------------------- codes and frames
_codes: dict[tuple, inputs.Code] = {}


def _code(q, n, dv, dc):
    key = (q, n, dv, dc)
    if key not in _codes:
        _codes[key] = inputs.make_regular_code(q, n, dv, dc, seed=q * 10007 + n * 31 + dv * 7 + dc)
    return _codes[key]


def _frames(code, frames, lo, hi, seed, make):
    """`make` (quantized reliabilities or channel probabilities) of `frames` random codewords."""
    g = torch.Generator(device=DEV)
    g.manual_seed(seed)
    out = None
    for f0 in range(0, frames, CHUNK):
        nf = min(CHUNK, frames - f0)
        info = torch.randint(0, code.q, (nf, code.k), generator=g, device=DEV)
        noise = torch.randn((nf, code.n, code.p), generator=g, device=DEV, dtype=torch.float64)
        eb = lo + (hi - lo) * torch.rand((nf,), generator=g, device=DEV, dtype=torch.float64)
        part = make(code, inputs.encode(code, info), noise, eb)
        if out is None:
            out = torch.empty((frames, code.n, code.q), dtype=part.dtype, device=DEV)
        out[f0:f0 + nf] = part
    return out


def _jobs(case):
    return [tuple(int(v) for v in j.split(",")) for j in case["jobs"].split()]


def prepare(case, seed):
    lo, hi = case["ebn0_lo"], case["ebn0_hi"]
    if case["path"] == "batch":
        decs, jobs = [], []
        for k, (q, n, dv, dc, frames) in enumerate(_jobs(case)):
            code = _code(q, n, dv, dc)
            dec = binding.Decoder.from_code(code)
            gamma = _frames(code, frames, lo, hi, seed * 64 + k, inputs.quantized_reliabilities)
            out = (torch.empty((frames, n), dtype=torch.uint8, device=DEV),
                   torch.empty((frames,), dtype=torch.int32, device=DEV),
                   torch.empty((frames,), dtype=torch.uint8, device=DEV))
            decs.append(dec)
            jobs.append((dec.handle, gamma, frames, case["iters"], int(case["stop"]), *out))
        ws = torch.empty(binding.nbldpc_decode_batch_workspace_size(jobs), dtype=torch.uint8, device=DEV)
        return dict(case=case, decs=decs, jobs=jobs, ws=ws)
    code = _code(case["q"], case["n"], case["dv"], case["dc"])
    dec = binding.Decoder.from_code(code)
    fft = case["path"] == "fftspa"
    if not fft and case["bits"] == 16:
        dec.set_message_bits(16)
    x = _frames(code, case["frames"], lo, hi, seed,
                inputs.channel_probabilities if fft else inputs.quantized_reliabilities)
    return dict(case=case, dec=dec, x=x)


def run(state):
    case = state["case"]
    if case["path"] == "batch":
        binding.nbldpc_decode_batch(state["jobs"], state["ws"])
        return [list(j[5:]) for j in state["jobs"]]
    if case["path"] == "fftspa":
        return list(state["dec"].fftspa_decode(state["x"], case["iters"], int(case["stop"]), want_app=case["app"]))
    return list(state["dec"].decode(state["x"], case["iters"], int(case["stop"])))


# ---------------------------------------------------------------- work
def _work(path, q, n, dv, dc, frames, iters, stop, app=False):
    """Every frame's input read and its outputs written once; the additions, products, minima and maxima of the
    algorithm (min-max: 3 (d_c - 2) convolutions of q^2 pairs for a check, as Alg. 2 counts them)."""
    p, m, its = q.bit_length() - 1, n * dv // dc, min(iters, ITERS_STOPPED) if stop else iters
    nbytes = frames * (n * q * (4 if path == "fftspa" else 1) + n + 5 + (4 * n * q if app else 0))
    if path == "fftspa":
        ops = n * dv * q * (2 * p + dc + dv + 2)
    else:
        ops = m * 3 * (dc - 2) * q * q * 2 + n * q * (2 * dv + 2)
    return nbytes, frames * its * ops


def work(case):
    if case["path"] == "batch":
        parts = [_work("minmax", *j, case["iters"], case["stop"]) for j in _jobs(case)]
    else:
        parts = [_work(case["path"], case["q"], case["n"], case["dv"], case["dc"], case["frames"], case["iters"],
                       case["stop"], case.get("app", False))]
    return {"bytes": sum(b for b, _ in parts), "flops": sum(f for _, f in parts)}


# ---------------------------------------------------------------- 64-bit values
def exact(case, seed):
    """The a-posteriori vectors of the second decoder (Alg. 1) in 64 bits.  Decided symbols, iteration counts and
    flags are whole numbers and have no value here; the min-max decoder returns nothing else."""
    if case["path"] != "fftspa" or not case["app"] or case["stop"]:
        return None
    code = _code(case["q"], case["n"], case["dv"], case["dc"])
    q, p = code.q, code.p
    prob = _frames(code, case["frames"], case["ebn0_lo"], case["ebn0_hi"], seed, inputs.channel_probabilities).double()
    # h x for every coefficient h and symbol x (carry-less product modulo the primitive polynomial)
    x = torch.arange(q)
    h = torch.from_numpy(code.coef.astype("int64"))[:, None]
    acc, a = torch.zeros((h.shape[0], q), dtype=torch.int64), h.clone()
    for i in range(p):
        acc ^= ((x >> i) & 1)[None, :] * a
        a <<= 1
        a = torch.where(a >= q, a ^ code.poly, a)
    mul = acc.to(DEV)                                                 # [edges, q]
    col = torch.from_numpy(code.col_idx.astype("int64")).to(DEV)
    m, dc, dv = code.m, case["dc"], case["dv"]
    edges_of = torch.argsort(col, stable=True).reshape(code.n, dv)    # regular: d_v edges to a variable
    had = torch.ones((1, 1), dtype=torch.float64)
    for _ in range(p):
        had = torch.cat([torch.cat([had, had], 1), torch.cat([had, -had], 1)], 0)
    had = had.to(DEV)
    app = torch.empty_like(prob)
    part = max(1, (1 << 26) // (code.nnz * q))                        # frames at a time
    for f0 in range(0, prob.shape[0], part):
        pr = prob[f0:f0 + part]
        nf = pr.shape[0]
        u = pr[:, col]                                                # [f, edges, q]
        z = pr
        for _ in range(case["iters"]):
            # u'(h x) = u(x), transform, product over the other edges, inverse transform, v'(x) = v(h x)
            w = (torch.zeros_like(u).scatter_(2, mul.expand_as(u), u) @ had).reshape(nf, m, dc, q)
            o = torch.stack([w[:, :, [k for k in range(dc) if k != j]].prod(2) for j in range(dc)], 2)
            v = (o.reshape(nf, code.nnz, q) @ had / q).gather(2, mul.expand_as(u)).clamp_min(0.0)
            t = v[:, edges_of]                                        # [f, n, d_v, q]
            z = pr * t.prod(2)
            for k in range(dv):
                e = pr * t[:, :, [j for j in range(dv) if j != k]].prod(2)
                s = e.sum(-1, keepdim=True)
                u[:, edges_of[:, k]] = torch.where(s > 0, e / s, torch.full_like(e, 1.0 / q))
        s = z.sum(-1, keepdim=True)
        app[f0:f0 + part] = torch.where(s > 0, z / s, torch.full_like(z, 1.0 / q))
    return [None, None, None, app]

"""GPU parity of the split-frame kernels: a small batch decodes each frame on a
cluster of blocks (the rule is in split_shape, csrc/nbldpc.cu).  Bar: bit-exact
against the oracle, and the same outputs as the one-block-per-frame kernels,
which a handle with a pinned tuning (nbldpc_code_set_tuning) keeps."""
import os

import numpy as np
import pytest
import torch

import oracle
from paper_2508_03567_gb300 import binding, inputs as I

pytestmark = pytest.mark.gpu
THREADS = os.cpu_count() or 4


def irregular(q, n, m, seed, dmax):
    """Rows of degree 2..dmax dealt from shuffled columns (every column used, degrees even to one
    or two), random coefficients."""
    rng = np.random.default_rng(seed)
    deal = np.concatenate([rng.permutation(n) for _ in range(m * dmax // n + 2)])
    h = np.zeros((m, n), np.int64)
    at = 0
    for r in range(m):
        d = 2 + (r * 7 + seed) % (dmax - 1)
        cols = np.unique(deal[at:at + d])
        if cols.size < 2:
            cols = np.array([deal[at], (deal[at] + 1) % n])
        h[r, cols] = 1
        at += d
    for c in np.nonzero(~h.any(0))[0]:
        h[c % m, c] = 1
    h *= rng.integers(1, q, h.shape)
    return I.code_from_dense(h, q, I.PRIMITIVE_POLY[q])


# fewer checks than ranks, rows and columns that do not divide by the ranks, ragged degrees
CODES = [("tiny", 16, 8, 5), ("ragged", 8, 70, 33), ("ragged", 32, 61, 31), ("ragged", 64, 45, 19), ("ragged", 128, 30, 13),
         ("ragged", 256, 26, 9), ("regular", 8, 64, 4), ("regular", 16, 100, 4), ("regular", 64, 576, 4),
         ("regular", 256, 128, 8)]


def make(kind, q, n, x):
    if kind == "regular":
        return I.make_regular_code(q, n, 2, x, seed=q + n)
    return irregular(q, n, x, q + n, 4 if kind == "tiny" else 6)


@pytest.mark.parametrize("bits", [8, 16])
@pytest.mark.parametrize("kind,q,n,x", CODES)
def test_small_batches_match_the_oracle_and_the_one_block_kernels(kind, q, n, x, bits):
    code = make(kind, q, n, x)
    rng = np.random.default_rng(3 * q + n)
    dec, one = binding.Decoder.from_code(code), binding.Decoder.from_code(code)
    if bits == 16:
        dec.set_message_bits(16)
        one.set_message_bits(16)
    one.set_tuning(*one.tuning())
    for frames in (1, 3, 25, 70, 130):          # every cluster size and block size of the rule
        g = rng.integers(0, 48, (frames, code.n, q)).astype(np.uint8)
        g[np.arange(frames)[:, None], np.arange(code.n)[None, :], rng.integers(0, q, (frames, code.n))] = 0
        g[0] = rng.choice(np.array([0, 255], np.uint8), g[0].shape)
        gd = torch.as_tensor(g).cuda()
        for iters, early in ((6, 1), (3, 0), (0, 1), (0, 0)):
            got = [t.cpu().numpy() for t in dec.decode(gd, iters, early)]
            ref = [t.cpu().numpy() for t in one.decode(gd, iters, early)]
            k = min(frames, 8)
            want = oracle.decode(code, g[:k], iters, early, threads=THREADS, cap=65535 if bits == 16 else 255)
            for name, a, b, w in zip(("symbols", "iterations", "ok"), got, ref, want):
                assert np.array_equal(a, b), f"{name}: {frames} frames, {iters} iterations, early {early}"
                assert np.array_equal(a[:k], w), f"{name} against the oracle: {frames} frames, {iters} iterations"


@pytest.mark.parametrize("q,n,m,dmax", [(2, 500, 140, 6), (4, 400, 110, 10), (8, 300, 210, 6), (16, 161, 101, 4),
                                        (32, 97, 53, 8), (64, 61, 31, 4), (128, 40, 17, 6), (256, 33, 14, 8),
                                        (64, 650, 390, 7), (256, 200, 110, 8)])
def test_small_fftspa_batches_match_the_one_block_kernel(q, n, m, dmax):
    """Same arithmetic in the same order: the frames of a small batch (cluster of blocks) equal, bit
    for bit and with their a-posteriori vectors, the same frames inside a batch of 240 (one block
    per frame; in the last two codes only some of the message rows fit its shared memory)."""
    code = irregular(q, n, m, q + n, dmax)
    assert np.bincount(code.col_idx, minlength=n).max() <= 8
    rng = np.random.default_rng(q)
    p = rng.dirichlet(np.full(q, 0.05), (240, n)).astype(np.float32) + np.float32(1e-6)
    p[0, 0] = 0.0                                # a vector without positive entries
    p[1] = rng.choice(np.array([0.0, 1.0], np.float32), p[1].shape)
    pd = torch.as_tensor(p).cuda()
    dec = binding.Decoder.from_code(code)
    for iters, early in ((5, 1), (2, 0), (0, 1)):
        ref = [t.cpu().numpy() for t in dec.fftspa_decode(pd, iters, early, want_app=True)]
        for frames in (1, 2, 30, 100, 220):
            got = [t.cpu().numpy() for t in dec.fftspa_decode(pd[:frames].contiguous(), iters, early, want_app=True)]
            for name, a, b in zip(("symbols", "iterations", "ok", "app"), got, ref):
                assert np.array_equal(a, b[:frames]), f"{name}: {frames} frames, {iters} iterations, early {early}"


def test_split_decode_replays_from_a_cuda_graph():
    code = I.workload_code("gf64_n576_dv2_dc4")
    dec = binding.Decoder.from_code(code)
    g = I.make_batch(code, 2.0, 5, 9).gamma.cuda()
    sym = torch.empty((9, code.n), dtype=torch.uint8, device="cuda")
    its, ok = torch.empty(9, dtype=torch.int32, device="cuda"), torch.empty(9, dtype=torch.uint8, device="cuda")
    ws = dec.workspace(9, "cuda")
    s = torch.cuda.Stream()
    s.wait_stream(torch.cuda.current_stream())
    binding.nbldpc_decode(dec.handle, g, 9, 20, 1, sym, its, ok, ws, stream=s)
    s.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=s):
        binding.nbldpc_decode(dec.handle, g, 9, 20, 1, sym, its, ok, ws, stream=s)
    g.copy_(I.make_batch(code, 1.5, 6, 9).gamma.cuda())
    graph.replay()
    torch.cuda.synchronize()
    for a, w in zip((sym, its, ok), oracle.decode(code, g.cpu().numpy(), 20, 1, threads=THREADS)):
        assert np.array_equal(a.cpu().numpy(), w)


@pytest.mark.parametrize("frames", [(1, 0, 3, 2, 1, 2, 1, 2), (9, 20, 0, 11, 7, 12, 5, 6), (150, 140, 160, 150, 30, 150, 60, 100)])
@pytest.mark.parametrize("early", [0, 1])
def test_mixed_batches_of_every_field_order(frames, early):
    """Ragged codes of every field order in one batch: a few frames (each on a cluster), and more than
    the one-block kernel holds at once (several frames to a slot, the code description changing
    under it); every job equals the oracle."""
    rng = np.random.default_rng(sum(frames))
    jobs, keep = [], []
    for k, q in enumerate((2, 4, 8, 16, 32, 64, 128, 256)):
        n, m, dmax = (24, 9, 6) if q >= 128 else (40, 19, 4) if q == 64 else (61, 31, 6)
        code = irregular(q, n, m, 5 * q, dmax)
        f = frames[k]
        g = rng.integers(0, 48, (f, code.n, q)).astype(np.uint8)
        if f:
            g[np.arange(f)[:, None], np.arange(code.n)[None, :], rng.integers(0, q, (f, code.n))] = 0
        dec, gd = binding.Decoder.from_code(code), torch.as_tensor(g).cuda()
        out = (torch.empty((f, code.n), dtype=torch.uint8, device="cuda"),
               torch.empty(f, dtype=torch.int32, device="cuda"), torch.empty(f, dtype=torch.uint8, device="cuda"))
        keep.append((code, g, dec, gd, out))
        jobs.append((dec.handle, gd, f, 4 + k % 3, early, *out))
    ws = torch.empty(binding.nbldpc_decode_batch_workspace_size(jobs), dtype=torch.uint8, device="cuda")
    before = binding.nbldpc_kernel_launch_count()
    binding.nbldpc_decode_batch(jobs, ws)
    torch.cuda.synchronize()
    assert binding.nbldpc_kernel_launch_count() == before + 1
    for k, (code, g, dec, gd, out) in enumerate(keep):
        if g.shape[0]:
            want = oracle.decode(code, g, 4 + k % 3, early, threads=THREADS)
            for name, a, w in zip(("symbols", "iterations", "ok"), out, want):
                assert np.array_equal(a.cpu().numpy(), w), f"q={code.q}: {name}"

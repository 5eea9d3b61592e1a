"""Which kernel a call takes (nbldpc_decode_cluster_blocks and its siblings), and
parity on the routes that the size rules choose between.  Bar: bit-exact
against the oracle."""
import os

import numpy as np
import pytest
import torch

import oracle
from paper_2508_03567_gb300 import binding, inputs as I
from test_gpu_split import irregular

pytestmark = pytest.mark.gpu
THREADS = os.cpu_count() or 4


def sms():
    return torch.cuda.get_device_properties(0).multi_processor_count


def random_gamma(code, frames, seed):
    """Random reliabilities with a zero per vector: frames that run to their last iteration."""
    rng = np.random.default_rng(seed)
    g = rng.integers(0, 48, (frames, code.n, code.q)).astype(np.uint8)
    if frames:
        g[np.arange(frames)[:, None], np.arange(code.n)[None, :], rng.integers(0, code.q, (frames, code.n))] = 0
    return g


def batch(specs, iters, early, setup=None):
    """Jobs of (code, gamma) pairs, each with a handle of its own (setup(k, decoder) tunes it)."""
    jobs, keep = [], []
    for k, (code, g) in enumerate(specs):
        dec, gd, f = binding.Decoder.from_code(code), torch.as_tensor(g).cuda(), g.shape[0]
        if setup:
            setup(k, dec)
        out = (torch.empty((f, code.n), dtype=torch.uint8, device="cuda"),
               torch.empty(f, dtype=torch.int32, device="cuda"), torch.empty(f, dtype=torch.uint8, device="cuda"))
        keep.append((dec, gd, out))
        jobs.append((dec.handle, gd, f, iters, early, *out))
    return jobs, keep


def check_batch(specs, jobs, keep, iters, early):
    ws = torch.empty(binding.nbldpc_decode_batch_workspace_size(jobs), dtype=torch.uint8, device="cuda")
    binding.nbldpc_decode_batch(jobs, ws)
    torch.cuda.synchronize()
    for (code, g), (_, _, out) in zip(specs, keep):
        if g.shape[0]:
            want = oracle.decode(code, g, iters, early, threads=THREADS)
            for name, a, w in zip(("symbols", "iterations", "ok"), out, want):
                assert np.array_equal(a.cpu().numpy(), w), f"q={code.q}: {name}"


# total frames, as a share of the SMs, of every cluster size and block size that the rule of mixed
# batches knows for codes with at least 1024 check-node lanes: 16 x 384, 8 x 384, 8 x 256, 8 x 128
@pytest.mark.parametrize("share,blocks", [(0.08, 16), (0.3, 8), (0.6, 8), (2.0, 8)])
def test_mixed_batches_on_every_cluster_shape(share, blocks):
    total = int(share * sms())
    codes = [I.workload_code("gf64_n576_dv2_dc4"), irregular(256, 61, 27, 261, 7), I.workload_code("gf16_n1024_dv2_dc4"),
             irregular(4, 61, 31, 20, 10)]
    counts = [total - 3 * (total // 4), total // 4, total // 4, total // 4]
    specs = [(c, random_gamma(c, f, 7 * c.q + total)) for c, f in zip(codes, counts)]
    jobs, keep = batch(specs, 4, 1)
    assert binding.nbldpc_decode_batch_cluster_blocks(jobs) == blocks
    check_batch(specs, jobs, keep, 4, 1)


def test_small_batches_take_the_cluster_kernels():
    """The sizes that test_gpu_split.py decodes reach the kernels that it is about."""
    for q, n, x in ((16, 100, 4), (64, 576, 4), (256, 128, 8)):
        dec = binding.Decoder.from_code(I.make_regular_code(q, n, 2, x, seed=q + n))
        for bits in (8, 16):
            dec.set_message_bits(bits)
            assert [binding.nbldpc_decode_cluster_blocks(dec.handle, f, 1) > 0 for f in (1, 3, 25)] == [True] * 3
            assert binding.nbldpc_decode_cluster_blocks(dec.handle, 60000, 1) == 0
        assert binding.nbldpc_fftspa_cluster_blocks(dec.handle, 60000, 1) == 0
    dec = binding.Decoder.from_code(I.workload_code("gf64_n576_dv2_dc4"))
    assert binding.nbldpc_fftspa_cluster_blocks(dec.handle, 1, 1) > 0


def test_fftspa_clusters_do_not_depend_on_the_minmax_schedule():
    """The Table 1 schedule is a setting of the min-max check-node pass: one FFT-SPA frame decodes on
    a cluster before and after it."""
    dec = binding.Decoder.from_code(I.workload_code("gf64_n576_dv2_dc4"))
    want = binding.nbldpc_fftspa_cluster_blocks(dec.handle, 1, 1)
    assert want > 0
    binding.nbldpc_code_set_cnp_schedule(dec.handle, binding.NBLDPC_CNP_TABLE1)
    assert binding.nbldpc_fftspa_cluster_blocks(dec.handle, 1, 1) == want
    assert binding.nbldpc_decode_cluster_blocks(dec.handle, 1, 1) == 0      # no Table 1 cluster kernel


def test_a_pinned_code_keeps_a_mixed_batch_on_the_one_block_kernel():
    """nbldpc_code_set_tuning holds for batches of every size: no cluster, and the pinned frames per
    block.  Only a job that has frames counts."""
    specs = [(I.workload_code("gf64_n576_dv2_dc4"), random_gamma(I.workload_code("gf64_n576_dv2_dc4"), 5, 1)),
             (I.workload_code("gf16_n1024_dv2_dc4"), random_gamma(I.workload_code("gf16_n1024_dv2_dc4"), 4, 2))]
    jobs, keep = batch(specs, 4, 1)
    assert binding.nbldpc_decode_batch_cluster_blocks(jobs) > 0
    slot = max(-(-c.nnz * c.q // 256) * 256 for c, _ in specs)
    for fpb in (1, 2):
        jobs, keep = batch(specs, 4, 1, lambda k, dec: dec.set_tuning(1, fpb))
        assert binding.nbldpc_decode_batch_cluster_blocks(jobs) == 0
        # nine frames in blocks of fpb slots
        assert binding.nbldpc_decode_batch_workspace_size(jobs) == 256 + -(-9 // fpb) * fpb * slot
        check_batch(specs, jobs, keep, 4, 1)
    empty = [(specs[0][0], specs[0][1][:0]), specs[0], specs[1]]
    jobs, keep = batch(empty, 4, 1, lambda k, dec: dec.set_tuning(1, 1) if k == 0 else None)
    assert binding.nbldpc_decode_batch_cluster_blocks(jobs) > 0
    check_batch(empty, jobs, keep, 4, 1)


@pytest.mark.parametrize("q,n", [(4, 48), (8, 512), (16, 1024), (32, 600), (64, 576), (128, 96), (256, 96)])
def test_a_handle_that_was_never_tuned_forgets_its_past_modes(q, n):
    """To 16-bit messages, or to the Table 1 schedule, and back: the launch shape of a new handle.
    A tuning that was set keeps its layout bit only, as before."""
    code = I.make_regular_code(q, n, 2, 4, seed=q + n)
    dec = binding.Decoder.from_code(code)

    def shape():
        return (dec.tuning(), binding.nbldpc_decode_workspace_size(dec.handle, 5000),
                [binding.nbldpc_decode_cluster_blocks(dec.handle, f, e) for f in (1, 60, 300) for e in (0, 1)])
    new = shape()
    dec.set_message_bits(16)
    assert dec.tuning()[0] == new[0][0] & 1
    dec.set_message_bits(8)
    assert shape() == new
    binding.nbldpc_code_set_cnp_schedule(dec.handle, binding.NBLDPC_CNP_TABLE1)
    assert dec.tuning()[0] == new[0][0] & 1
    binding.nbldpc_code_set_cnp_schedule(dec.handle, binding.NBLDPC_CNP_MINIMAL)
    assert shape() == new
    g = random_gamma(code, 40, q)
    got = [t.cpu().numpy() for t in dec.decode(torch.as_tensor(g).cuda(), 4, 0)]
    for a, w in zip(got, oracle.decode(code, g, 4, 0, threads=THREADS)):
        assert np.array_equal(a, w)
    dec.set_tuning(*new[0])
    dec.set_message_bits(16)
    dec.set_message_bits(8)
    assert dec.tuning()[0] == new[0][0] & 1


def test_gf4_checks_above_degree_8_in_mixed_batches():
    """The mixed-code kernels' group form of q = 4 (their register form ends at check degree 8): beside a
    GF(64) code on clusters, and on the one-block kernel."""
    small = irregular(4, 61, 31, 20, 10)
    assert np.diff(small.row_ptr).max() > 8
    for early, counts, cluster in ((1, (9, 20), True), (0, (600, 30), False), (0, (90, 0), False)):
        specs = [(small, random_gamma(small, counts[0], 5)),
                 (I.workload_code("gf64_n576_dv2_dc4"), random_gamma(I.workload_code("gf64_n576_dv2_dc4"), counts[1], 6))]
        jobs, keep = batch(specs, 4, early)
        assert (binding.nbldpc_decode_batch_cluster_blocks(jobs) > 0) == cluster
        check_batch(specs, jobs, keep, 4, early)


@pytest.mark.parametrize("early,frames", [(1, 8), (0, 130)])
def test_the_variant_of_a_code_does_not_change_a_mixed_batch(early, frames):
    """Mixed-code kernels have one form per field order: any variant, on clusters (no code tuned by hand)
    and on the one-block kernel, gives the oracle's outputs."""
    codes = [irregular(256, 61, 27, 261, 7), irregular(128, 61, 27, 133, 7), irregular(64, 61, 31, 69, 5),
             irregular(16, 61, 31, 21, 6)]
    specs = [(c, random_gamma(c, frames, 11 * c.q)) for c in codes]
    for variants in (None, (0, 0, 0, 0), (4, 4, 4, 1), (5, 1, 2, 2)):
        def tune(k, dec):
            if variants:
                dec.set_tuning(variants[k], 1)
        jobs, keep = batch(specs, 3, early, tune)
        assert (binding.nbldpc_decode_batch_cluster_blocks(jobs) > 0) == (variants is None and early == 1)
        check_batch(specs, jobs, keep, 3, early)


@pytest.mark.parametrize("q,n", [(32, 13936), (16, 13940)])
def test_the_largest_codes_leave_no_room_for_unused_tables(q, n):
    """Regular (2,4) codes within 100 bytes of the block's shared memory in the group form (15 n bytes of
    description, n of decisions, the groups' scratch): it stages no table of the register form.  The
    same code with 16-bit messages and under the Table 1 schedule, against the oracle."""
    code = I.make_regular_code(q, n, 2, 4, seed=q, encoder=False)
    dec = binding.Decoder.from_code(code)
    g = random_gamma(code, 3, q)
    gd = torch.as_tensor(g).cuda()
    for a, w in zip(dec.decode(gd, 4, 1), oracle.decode(code, g, 4, 1, threads=THREADS)):
        assert np.array_equal(a.cpu().numpy(), w)
    binding.nbldpc_code_set_cnp_schedule(dec.handle, binding.NBLDPC_CNP_TABLE1)
    for a, w in zip(dec.decode(gd, 4, 0), oracle.decode(code, g, 4, 0, threads=THREADS)):
        assert np.array_equal(a.cpu().numpy(), w)
    binding.nbldpc_code_set_cnp_schedule(dec.handle, binding.NBLDPC_CNP_MINIMAL)
    dec.set_message_bits(16)
    for a, w in zip(dec.decode(gd, 4, 0), oracle.decode(code, g, 4, 0, threads=THREADS, cap=65535)):
        assert np.array_equal(a.cpu().numpy(), w)


def one_heavy_check(q, n, m, seed, heavy=60):
    """Checks of degree 3, and one of degree `heavy`."""
    rng = np.random.default_rng(seed)
    h = np.zeros((m, n), np.int64)
    for r in range(m):
        d = heavy if r == m // 2 else 3
        h[r, (3 * r + np.arange(d)) % n] = rng.integers(1, q, d)
    return I.code_from_dense(h, q, I.PRIMITIVE_POLY[q])


@pytest.mark.parametrize("q,n,tunings", [(16, 1024, ((2, 1), (3, 2), (3, 4))), (32, 600, ((3, 1), (2, 2))),
                                         (8, 512, ((2, 1), (3, 2), (2, 4), (2, 8))),
                                         (16, 64, ((3, 4), (2, 8))), (32, 64, ((3, 2), (2, 4)))])
def test_resident_tunings_of_the_register_form(q, n, tunings):
    """Variants 2 and 3 at every frames-per-block whose messages fit, also where a frame has more checks
    than its share of the block's threads (n >= 512), or its checks want more scratch than is left (n =
    64: lanes without a check at 4 and 8 frames): taken, and equal to the oracle."""
    code = one_heavy_check(q, n, 40, q) if n == 64 else I.make_regular_code(q, n, 2, 4, seed=q + n)
    dec = binding.Decoder.from_code(code)
    g = random_gamma(code, 21, q + n)
    gd = torch.as_tensor(g).cuda()
    for v, fpb in tunings:
        dec.set_tuning(v, fpb)
        assert dec.tuning() == (v, fpb)
        for iters, early in ((4, 1), (2, 0)):
            want = oracle.decode(code, g, iters, early, threads=THREADS)
            for a, w in zip(dec.decode(gd, iters, early), want):
                assert np.array_equal(a.cpu().numpy(), w), f"variant {v}, {fpb} frames per block"


def test_mixed_batch_of_a_code_whose_register_scratch_does_not_fit():
    """32 checks, one of degree 34, eight frames to a block: the register form's scratch (31 KB a frame)
    does not fit eight times, the group form's does, and the batch takes it."""
    code = one_heavy_check(32, 34, 32, 7, heavy=34)
    assert code.m == 32 and np.diff(code.row_ptr).max() == 34
    frames = 13 * sms()                             # more than the group form is taken for anyway
    specs = [(code, random_gamma(code, frames, 8))]
    jobs, keep = batch(specs, 3, 0)
    check_batch(specs, jobs, keep, 3, 0)
    assert binding.nbldpc_decode_batch_workspace_size(jobs) % (8 * (-(-code.nnz * 32 // 256) * 256)) == 256


@pytest.mark.parametrize("q,n,dv,dc", [(8, 64, 2, 4), (16, 64, 2, 4), (16, 100, 2, 4), (16, 128, 2, 8), (32, 64, 2, 4),
                                       (32, 96, 3, 6), (32, 160, 2, 4), (32, 128, 2, 4)])
def test_short_codes_at_every_number_of_frames(q, n, dv, dc):
    """The form and the frames per block of an untuned handle follow the frames of a call: on each side of
    the limits (cluster limits, frames per SM, the whole chip), through
    nbldpc_decode and nbldpc_decode_noalloc, the oracle's outputs; a workspace of the largest call
    serves every smaller one."""
    code = I.make_regular_code(q, n, dv, dc, seed=q + n)
    dec = binding.Decoder.from_code(code)
    frames = [1, sms() // 3, sms(), sms() + 1, 3 * sms(), 3 * sms() + 1, 8 * sms(), 16 * sms(), 16 * sms() + 1, 37 * sms()]
    need = [binding.nbldpc_decode_workspace_size(dec.handle, f) for f in frames]
    assert need == sorted(need)
    g = random_gamma(code, frames[-1], q + n)
    gd = torch.as_tensor(g).cuda()
    want = {es: oracle.decode(code, g, 3, es, threads=THREADS) for es in (0, 1)}
    for f in reversed(frames):
        for es in (0, 1):
            got = dec.decode(gd[:f], 3, es)                 # (the workspace of the largest call)
            for a, w in zip(got, want[es]):
                assert np.array_equal(a.cpu().numpy(), w[:f]), f"{f} frames, early {es}"
            out = [torch.empty_like(t) for t in got]
            binding.nbldpc_decode_noalloc(dec.handle, gd, f, 3, es, *out)
            for a, b in zip(out, got):
                assert torch.equal(a, b), f"noalloc: {f} frames, early {es}"


def test_short_codes_take_the_group_form_until_the_chip_is_full():
    """Message slots in the workspace: the group form of GF(16) N=64 and GF(32) N=64.  A GF(16) N=1024
    code, and a tuning that was set, keep the register form, which has none."""
    for q in (16, 32):
        code = I.make_regular_code(q, 64, 2, 4, seed=q + 64)
        dec = binding.Decoder.from_code(code)
        slot = -(-code.nnz * q // 256) * 256
        assert dec.tuning()[0] == 3
        assert binding.nbldpc_decode_workspace_size(dec.handle, 2 * sms()) == 256 + 2 * sms() * slot
        dec.set_tuning(*dec.tuning())
        assert binding.nbldpc_decode_workspace_size(dec.handle, 2 * sms()) == 256
    dec = binding.Decoder.from_code(I.workload_code("gf16_n1024_dv2_dc4"))
    assert binding.nbldpc_decode_workspace_size(dec.handle, 5000) == 256


def test_fftspa_clusters_of_the_lane_per_edge_form_follow_the_tasks():
    """A warp task holds up to 32 edges: short GF(2) and GF(4) codes, whose few tasks leave most ranks
    without work, keep one block per frame, and no cluster has more blocks than the code has tasks."""
    for q, n, dv, dc, clusters in ((2, 64, 2, 4, False), (2, 200, 3, 6, False), (4, 48, 2, 4, False),
                                   (4, 200, 2, 4, False), (4, 1024, 2, 4, True), (2, 1536, 2, 4, True),
                                   (8, 120, 2, 12, False), (16, 240, 2, 12, True), (64, 192, 2, 12, True)):
        dec = binding.Decoder.from_code(I.make_regular_code(q, n, dv, dc, seed=q + n))
        assert (binding.nbldpc_fftspa_cluster_blocks(dec.handle, 1, 1) > 0) == clusters, (q, n, dc)
    code = irregular(32, 40, 6, 55, 20)            # six checks, one above degree 8: few tasks
    assert np.diff(code.row_ptr).max() > 8
    dec = binding.Decoder.from_code(code)
    assert 2 <= binding.nbldpc_fftspa_cluster_blocks(dec.handle, 1, 1) <= 6
    p = np.random.default_rng(16).dirichlet(np.full(32, 0.05), (300, code.n)).astype(np.float32) + np.float32(1e-6)
    pd = torch.as_tensor(p).cuda()
    ref = dec.fftspa_decode(pd, 4, 0, want_app=True)
    got = dec.fftspa_decode(pd[:5].contiguous(), 4, 0, want_app=True)
    for a, b in zip(got, ref):
        assert torch.equal(a, b[:5])


@pytest.mark.parametrize("q,n,want", [(64, 256, (16, 8, 8, 4, 0)), (128, 128, (16, 8, 8, 4, 0)), (128, 96, (16, 8, 8, 0, 0)),
                                      (256, 128, (16, 8, 8, 4, 0))])
def test_fftspa_clusters_of_fixed_iterations_take_one_wave(q, n, want):
    """Without early stop the frames' clusters run side by side or not at all: the more frames, the fewer
    blocks; outputs as inside a large batch."""
    code = I.make_regular_code(q, n, 2, 4, seed=q + n)
    dec = binding.Decoder.from_code(code)
    counts = [1, sms() // 8, sms() // 5, sms() // 3, sms() // 2]
    assert tuple(binding.nbldpc_fftspa_cluster_blocks(dec.handle, f, 0) for f in counts) == want
    p = np.random.default_rng(q).dirichlet(np.full(q, 0.05), (2 * sms(), code.n)).astype(np.float32) + np.float32(1e-6)
    pd = torch.as_tensor(p).cuda()
    ref = dec.fftspa_decode(pd, 3, 0, want_app=True)
    for f in counts:
        got = dec.fftspa_decode(pd[:f].contiguous(), 3, 0, want_app=True)
        for a, b in zip(got, ref):
            assert torch.equal(a, b[:f])


@pytest.mark.parametrize("early,per_sm", [(1, 1), (1, 5), (1, 30), (0, 2), (0, 3), (0, 9)])
@pytest.mark.parametrize("family", ["all", "small", "wide"])
def test_mixed_batches_on_both_one_block_kernels(family, early, per_sm):
    """Frames per SM on each side of the limits between the two-block kernel (paths in line) and the
    three-block one (a function per field order), for the mixes that have limits of their own; ragged
    codes below the sizes that take clusters, several frames to a slot at the largest."""
    fields = {"all": (2, 4, 8, 16, 32, 64, 128, 256), "small": (2, 4, 8), "wide": (128, 256)}[family]
    frames = per_sm * sms() // len(fields) + 1
    specs = []
    for q in fields:
        n, m, dmax = (24, 9, 6) if q >= 128 else (40, 19, 4) if q == 64 else (61, 31, 6)
        code = irregular(q, n, m, 5 * q, dmax)
        specs.append((code, random_gamma(code, frames, q + per_sm)))
    jobs, keep = batch(specs, 3, early, lambda k, dec: dec.set_tuning(0, 1 + (per_sm > 9)) if k == 0 else None)
    assert binding.nbldpc_decode_batch_cluster_blocks(jobs) == 0
    check_batch(specs, jobs, keep, 3, early)


@pytest.mark.parametrize("early", [0, 1])
@pytest.mark.parametrize("n,dc,per_sm", [(64, 4, 2), (64, 4, 13), (128, 4, 2), (128, 4, 4), (280, 8, 4)])
def test_mixed_batches_of_short_gf32_codes(n, dc, per_sm, early):
    """Group form and register form of GF(32) in a mixed batch (32, 64 and 70 checks), on each side of the
    limits in frames, beside a GF(4) code that shares the frame slots: the oracle's outputs."""
    codes = [I.make_regular_code(32, n, 2, dc, seed=32 + n), irregular(4, 61, 31, 20, 6)]
    specs = [(c, random_gamma(c, per_sm * sms() + 1, n + dc)) for c in codes]
    jobs, keep = batch(specs, 2, early)
    check_batch(specs, jobs, keep, 2, early)


def test_mixed_batches_leave_the_clusters_where_frames_fill_the_chip():
    """Frames per SM up to which a batch of one code decodes on clusters, by field, check-node lanes and check
    degree."""
    for q, n, dv, dc, per_sm in ((16, 1024, 2, 4, 0.625), (32, 600, 3, 6, 2), (32, 128, 2, 4, 0.75), (64, 576, 2, 4, 4),
                                 (64, 144, 2, 4, 1.5), (128, 256, 2, 4, 3), (256, 192, 2, 4, 3), (256, 192, 2, 6, 2.5),
                                 (256, 280, 2, 8, 1.5)):
        code = I.make_regular_code(q, n, dv, dc, seed=q + n, encoder=False)
        dec = binding.Decoder.from_code(code)
        for frames, cluster in ((int(per_sm * sms()), True), (int(per_sm * sms()) + 1, False)):
            job = (dec.handle, None, frames, 10, 1, None, None, None)
            assert (binding.nbldpc_decode_batch_cluster_blocks([job]) > 0) == cluster, (q, n, dc, frames)
            job = (dec.handle, None, frames, 10, 0, None, None, None)
            assert (binding.nbldpc_decode_batch_cluster_blocks([job]) > 0) == (frames <= 3 * sms() // 8)


def test_frames_of_small_fields_on_clusters_for_the_sake_of_a_few():
    """Many GF(8) frames as long as half of a GF(16) frame keep one block each with a few of those; many short
    GF(4) frames follow a few GF(256) frames, which take a hundred times as long, onto clusters."""
    a = [I.workload_code("gf16_n1024_dv2_dc4"), I.make_regular_code(8, 512, 2, 4, seed=520)]
    b = [I.workload_code("gf256_n128_dv2_dc8"), irregular(4, 61, 31, 20, 6)]
    for codes, counts, cluster in ((a, (5, 0), True), (a, (5, 30), True), (a, (sms() // 3, sms() // 3), False),
                                   (a, (5, 2 * sms()), False), (b, (3, sms()), True)):
        specs = [(c, random_gamma(c, f, f + c.q)) for c, f in zip(codes, counts)]
        jobs, keep = batch(specs, 3, 1)
        assert (binding.nbldpc_decode_batch_cluster_blocks(jobs) > 0) == cluster, counts
        check_batch(specs, jobs, keep, 3, 1)


def test_gf4_codes_at_eight_frames_per_block():
    """One warp per frame: regular and ragged codes that the one-warp kernels serve (up to 32 checks of degree
    <= 4, columns of degree <= 2), and the nearest codes that they do not (33 checks, degree 5, a column of
    degree 3): the oracle's outputs at few and many frames."""
    ragged = [irregular(4, 61, 32, 9, 4), irregular(4, 61, 33, 9, 4), irregular(4, 61, 30, 10, 5)]
    assert [(c.m, int(np.diff(c.row_ptr).max())) for c in ragged] == [(32, 4), (33, 4), (30, 5)]
    codes = [I.workload_code("gf4_n48_dv2_dc4"), *ragged, I.make_regular_code(4, 60, 3, 6, seed=64)]
    assert [int(np.bincount(c.col_idx).max()) for c in codes] == [2, 2, 2, 2, 3]
    for code in codes:
        dec = binding.Decoder.from_code(code)
        g = random_gamma(code, 9 * sms(), code.n + code.m)
        gd = torch.as_tensor(g).cuda()
        for v in (2, 3):
            dec.set_tuning(v, 8)
            for frames, iters, early in ((1, 5, 1), (13, 2, 0), (9 * sms(), 3, 1), (9 * sms(), 0, 0)):
                want = oracle.decode(code, g[:frames], iters, early, threads=THREADS)
                for a, w in zip(dec.decode(gd[:frames].contiguous(), iters, early), want):
                    assert np.array_equal(a.cpu().numpy(), w), (code.m, v, frames)

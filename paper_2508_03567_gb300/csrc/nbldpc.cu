// C ABI of the GB300 NB-LDPC decoders (declarations and contracts in
// include/nbldpc.h), min-max side: argument validation, GF tables, code upload
// (with the FFT-SPA blob section), launch planning, mixed batches, the
// autotuner, host-buffer and non-allocating decodes, stream-ordered launches
// of the min-max kernels.  FFT-SPA decodes are in fftspa_host.cu.
#include "nbldpc.h"

#include <algorithm>
#include <cstdio>
#include <cstring>
#include <new>
#include <vector>

#include "host_internal.h"
#include "mma_kernels.cuh"

static_assert(nbldpc::kMaxJobs == NBLDPC_MAX_BATCH_JOBS, "job table size");
static_assert(sizeof(nbldpc::LaunchParams<0>) < 32000 && sizeof(nbldpc::SplitBatchParams) < 32000, "kernel parameter space");

std::atomic<uint64_t> nbldpc_host::g_launches{0};
std::mutex nbldpc_host::g_attr_mu;

using namespace nbldpc_host;

namespace {

constexpr int kThreads = 256;

// Field tables by repeated multiplication by x modulo the primitive
// polynomial; fails unless x generates all q-1 non-zero elements.
bool build_field(int q, uint32_t poly, std::vector<uint8_t>& exp2, std::vector<uint8_t>& lg) {
  int p = 0;
  while ((1 << p) < q) ++p;
  if ((poly >> p) != 1u) return false;
  exp2.assign(2 * q, 0);
  lg.assign(q, 0);
  std::vector<int> seen(q, 0);
  uint32_t v = 1;
  for (int i = 0; i < q - 1; ++i) {
    if (seen[v]) return false;
    seen[v] = 1;
    exp2[i] = (uint8_t)v;
    lg[v] = (uint8_t)i;
    v <<= 1;
    if (v & (uint32_t)q) v ^= poly;
  }
  if (v != 1u) return false;
  for (int i = q - 1; i < 2 * q; ++i) exp2[i] = exp2[i % (q - 1)];
  return true;
}

}  // namespace

namespace nbldpc {   // defined in kernels.cu, one translation unit per field order
const void* kernel_q0(int v, int mb, int t1, int dreg);
const void* kernel_q0_wide();
const void* kernel_q2(int v, int mb, int t1, int dreg);
const void* kernel_q4(int v, int mb, int t1, int dreg);
const void* kernel_q8(int v, int mb, int t1, int dreg);
const void* kernel_q16(int v, int mb, int t1, int dreg);
const void* kernel_q32(int v, int mb, int t1, int dreg);
const void* kernel_q64(int v, int mb, int t1, int dreg);
const void* kernel_q128(int v, int mb, int t1, int dreg);
const void* kernel_q256(int v, int mb, int t1, int dreg);
const void* split_kernel_q0();
const void* split_kernel_q8(int mb, int dreg);
const void* split_kernel_q16(int mb, int dreg);
const void* split_kernel_q32(int mb, int dreg);
const void* split_kernel_q64(int mb, int dreg);
const void* split_kernel_q128(int mb, int dreg);
const void* split_kernel_q256(int mb, int dreg);
}  // namespace nbldpc

namespace {

// Kernel mode: 1 = 8-bit messages, 2 = 16-bit messages, 3 = 8-bit messages with
// the Table 1 check-node schedule (each a separate kernel instantiation).
int kmode(const nbldpc_code* c) { return c->mb == 2 ? 2 : (c->cnp_schedule == NBLDPC_CNP_TABLE1 ? 3 : 1); }

// kernel compiled for one field order, variant (bit 0: layout; bit 1: messages
// resident in shared memory; bit 2: pruned convolutions), kernel mode and the
// code's regular check degree (dreg: 0 when the rows differ, -1 for a register form
// with fewer lanes than threads, -1 or -4 for a GF(4) code in the one-warp form; a field order may have a kernel for it), or for every
// field order (q = 0, mode 1; v = -1 at three blocks an SM, -2 at two)
const void* kernel_for(int q, int v, int km, int dreg = 0) {
  const int mb = km == 2 ? 2 : 1, t1 = km == 3 ? 1 : 0;
  switch (q) {
    case 0: return v == -2 ? nbldpc::kernel_q0_wide() : nbldpc::kernel_q0(-1, mb, t1, 0);
    case 2: return nbldpc::kernel_q2(v, mb, t1, dreg);
    case 4: return nbldpc::kernel_q4(v, mb, t1, dreg);
    case 8: return nbldpc::kernel_q8(v, mb, t1, dreg);
    case 16: return nbldpc::kernel_q16(v, mb, t1, dreg);
    case 32: return nbldpc::kernel_q32(v, mb, t1, dreg);
    case 64: return nbldpc::kernel_q64(v, mb, t1, dreg);
    case 128: return nbldpc::kernel_q128(v, mb, t1, dreg);
    case 256: return nbldpc::kernel_q256(v, mb, t1, dreg);
  }
  return nullptr;
}

// the regular check degree that selects a specialised kernel (see kernel_for), else 0
int kernel_dreg(int q, int v, int km, int dreg) {
  return ((q == 64 || q == 4) && km == 1 && v >= 2 && v <= 3 && dreg == 4) ? 4 : 0;
}

// kernel that decodes a frame on a cluster of blocks (minimal schedule), null where
// split_shape never takes it; q = 0: mixed codes, 8-bit messages
const void* split_kernel_for(int q, int mb, int dreg) {
  switch (q) {
    case 0: return nbldpc::split_kernel_q0();
    case 8: return nbldpc::split_kernel_q8(mb, dreg);
    case 16: return nbldpc::split_kernel_q16(mb, dreg);
    case 32: return nbldpc::split_kernel_q32(mb, dreg);
    case 64: return nbldpc::split_kernel_q64(mb, dreg);
    case 128: return nbldpc::split_kernel_q128(mb, dreg);
    case 256: return nbldpc::split_kernel_q256(mb, dreg);
  }
  return nullptr;
}

int mixed_layout(int q) { return q >= 16 && q <= 64 ? 1 : 0; }   // as in mma_kernels.cuh

template <int Q> int lanes(int v) { return v ? nbldpc::Geo<Q, 1>::G : nbldpc::Geo<Q, 0>::G; }

int group_lanes(int q, int v) {
  switch (q) {
    case 2: return lanes<2>(v);
    case 4: return lanes<4>(v);
    case 8: return lanes<8>(v);
    case 16: return lanes<16>(v);
    case 32: return lanes<32>(v);
    case 64: return lanes<64>(v);
    case 128: return lanes<128>(v);
    case 256: return lanes<256>(v);
  }
  return 0;
}

int group_bytes(int q, int dmax, int mb, bool pr) {
  switch (q) {
    case 2: return nbldpc::group_scratch_bytes<2>(dmax, mb);
    case 4: return nbldpc::group_scratch_bytes<4>(dmax, mb);
    case 8: return nbldpc::group_scratch_bytes<8>(dmax, mb);
    case 16: return nbldpc::group_scratch_bytes<16>(dmax, mb);
    case 32: return nbldpc::group_scratch_bytes<32>(dmax, mb);
    case 64: return nbldpc::group_scratch_bytes<64>(dmax, mb, pr);
    case 128: return nbldpc::group_scratch_bytes<128>(dmax, mb, pr);
    case 256: return nbldpc::group_scratch_bytes<256>(dmax, mb, pr);
  }
  return 0;
}

// Every kernel may use up to the opt-in shared memory of the device (set once
// per device and kernel; occupancy still follows the bytes of each launch).
bool g_attr_done[64][91] = {};

// per field order: 3 kernel modes x 2 layouts, the 2 resident-message kernels,
// then the 2 pruned-convolution kernels; after them the 2 GF(64) and the 2 GF(4)
// resident kernels of check degree 4 and the GF(8), GF(16), GF(32) ones of few lanes
int kernel_slot(int q, int v, int km, int dreg) {
  if (q == 0) return v == -2 ? 88 : 0;
  if (kernel_dreg(q, v, km, dreg)) return (q == 64 ? 81 : 83) + (v & 1);
  if (dreg < 0) return q == 4 ? (dreg == -4 ? 90 : 89) : 85 + nbldpc::ilog2(q) - 3;
  return 1 + 10 * (nbldpc::ilog2(q) - 1) + ((v & 4) ? 8 + (v & 1) : (v & 2) ? 6 + (v & 1) : 2 * (km - 1) + (v & 1));
}

int prepare_kernel(int q, int v, int km, int dreg, int dev, int smem_optin) {
  std::lock_guard<std::mutex> lk(g_attr_mu);
  if (dev < 0 || dev >= 64) return NBLDPC_ERR_CUDA;
  const void* k = kernel_for(q, v, km, dreg);
  if (!k) return NBLDPC_ERR_UNSUPPORTED;
  bool& done = g_attr_done[dev][kernel_slot(q, v, km, dreg)];
  if (!done) {
    if (cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, smem_optin) != cudaSuccess)
      return NBLDPC_ERR_CUDA;
    done = true;
  }
  return NBLDPC_OK;
}

// Largest cluster of split-frame blocks (16, 8, 4 or 2) that the device runs for a field
// order and message width; 0 when there is none.  The kernel attributes are set and the
// device asked once (-1: asked, none).
int g_split_max[64][9][3] = {};

int split_max(int q, int mb, int dreg, int dev, int smem_optin) {
  std::lock_guard<std::mutex> lk(g_attr_mu);
  if (dev < 0 || dev >= 64) return 0;
  // (the third: 8-bit GF(64) messages and checks of degree 4)
  int& mx = g_split_max[dev][q ? nbldpc::ilog2(q) : 0][q == 64 && mb == 1 && dreg == 4 ? 2 : mb - 1];
  if (mx == 0) {
    const void* k = split_kernel_for(q, mb, dreg);
    mx = k ? split_kernel_prepare(k, nbldpc::kResidentThreads, smem_optin) : 0;
    if (mx == 0) mx = -1;
  }
  return mx < 0 ? 0 : mx;
}

struct CodeNeeds {       // what one code asks of a frame slot
  int q, variant, mb, dmax, blob, perm, n;   // blob: staged sections; perm: the register form's selectors
  size_t msg;
  int dreg;              // regular check degree (0: the rows differ)
  int m;
  bool warp4;            // a GF(4) code that one warp decodes alone
};

// GF(4) codes a single warp decodes alone (one-warp frame slots: at most 32
// checks of degree <= 4, columns of degree <= 2): GF(4) N=48 (2,4) 17-18 us per
// 1,000-frame decode at 8 frames per block against 24.5 at 4.
bool warp4_code(const nbldpc_code* c) { return c->q == 4 && c->m <= 32 && c->dmax <= 4 && c->vmax <= 2; }

CodeNeeds needs_of(const nbldpc_code* c, int variant, int mb) {
  return CodeNeeds{c->q, variant, mb, c->dmax, c->off.perm, c->off.bytes - c->off.perm, c->n,
                   round_up((size_t)c->nnz * c->q * mb, 256), c->dreg, c->m, warp4_code(c)};
}

// Field orders whose resident-message kernels take the register form of the check-node
// pass (one lane per check).
bool reg_form(int q) { return q == 8 || q == 16 || q == 32; }

// Threads of a frame slot of those kernels: the checks in as few rounds as `most` threads
// allow, and no more threads than these rounds need.
int reg_threads(int m, int most = nbldpc::kResidentThreads) {
  const int rounds = (m + most - 1) / most;
  return (int)round_up((size_t)(m + rounds - 1) / rounds, 32);
}

int reg_scratch(int q, int nthr, int dmax) {
  return q == 8 ? nbldpc::reg_scratch_bytes<8>(nthr, dmax)
                : q == 16 ? nbldpc::reg_scratch_bytes<16>(nthr, dmax) : nbldpc::reg_scratch_bytes<32>(nthr, dmax);
}

// Whether a code takes the register form in the mixed-code kernel: its scratch must leave
// three blocks on an SM.
bool mixed_reg(int q, int nthr, int dmax) { return reg_form(q) && reg_scratch(q, nthr, dmax) <= 32768; }

// Plan a launch of kernel (kq, kv, kernel mode km) with fpb frame slots per block for a set of codes.
// Variants 2 and 3 keep each frame's messages in shared memory: blocks of
// nbldpc::kResidentThreads threads (1, 2 or 4 frame slots) or of 256 threads with
// 8 one-warp slots (q = 8, 16, 32: no more threads a slot than its checks need, and as
// many of them with a check as their scratch leaves room for), no message slots in the workspace.
// mixed: the mixed-code kernel's (kq = 0) register form has its scratch and selectors beside the group
// form's, so that a launch may take either; without them where both do not fit.
int make_plan(int kq, int kv, int km, int fpb, const CodeNeeds* cs, int nc, Plan* out, bool mixed = true) {
  int dev = 0, sms = 0, optin = 0;
  if (cudaGetDevice(&dev) != cudaSuccess ||
      cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess ||
      cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev) != cudaSuccess)
    return NBLDPC_ERR_CUDA;
  const bool resident = kv >= 0 && (kv & 2);
  const bool reg = resident && reg_form(kq);
  const int most = resident && fpb != 8 ? nbldpc::kResidentThreads : kThreads;
  if (fpb < 1 || most % fpb) return NBLDPC_ERR_ARG;
  if (resident && km != 1) return NBLDPC_ERR_UNSUPPORTED;
  int nthr = most / fpb;
  if (nthr < 32 || nthr % 32) return NBLDPC_ERR_UNSUPPORTED;
  if (reg) nthr = std::min(nthr, reg_threads(cs[0].m, nthr));
  Plan pl{};
  pl.fpb = fpb;
  pl.threads = fpb * nthr;
  int scratch = 0;
  for (int i = 0; i < nc; ++i) {
    const int G = group_lanes(cs[i].q, cs[i].variant & 1);
    if (G > nthr) return NBLDPC_ERR_UNSUPPORTED;
    int s = reg ? reg_scratch(cs[i].q, nthr, cs[i].dmax)
                      : (nthr / G) * group_bytes(cs[i].q, cs[i].dmax, cs[i].mb, kq == 0 ? cs[i].q >= 128 : (kv & 4) != 0);
    const bool either = kq == 0 && mixed && mixed_reg(cs[i].q, nthr, cs[i].dmax);
    if (either) s = std::max(s, reg_scratch(cs[i].q, nthr, cs[i].dmax));
    if (s > scratch) scratch = s;
    const int blob = cs[i].blob + (reg || either ? cs[i].perm : 0);
    if (blob > pl.blob_cap) pl.blob_cap = blob;
    if (cs[i].n > pl.n_cap) pl.n_cap = cs[i].n;
    if (cs[i].msg > pl.slot_bytes) pl.slot_bytes = cs[i].msg;
  }
  pl.blob_cap = (int)round_up((size_t)pl.blob_cap, 16);
  pl.n_cap = (int)round_up((size_t)pl.n_cap, 16);
  const int fixed = pl.blob_cap + pl.n_cap + nbldpc::ctl_bytes(kq);
  if (kq == 0 && mixed && fpb * (int)round_up((size_t)(fixed + scratch), 16) > optin)
    return make_plan(kq, kv, km, fpb, cs, nc, out, false);
  pl.mixed_reg = kq == 0 && mixed;
  if (reg) {
    pl.lanes = nthr;
    const int row = reg_scratch(kq, 1, cs[0].dmax);   // a lane's scratch
    const int room = optin / fpb / 16 * 16 - (int)round_up((size_t)fixed, 16) - (int)round_up(pl.slot_bytes, 16);
    if (scratch > room) {
      pl.lanes = room < row ? 0 : std::min(nthr, room / 16 * 16 / row);
      if (pl.lanes < 1) return NBLDPC_ERR_UNSUPPORTED;
      scratch = pl.lanes * row;
    }
  }
  pl.slot_smem = (int)round_up((size_t)(fixed + scratch), 16);
  if (resident) {   // the messages follow the slot's scratch
    pl.xs_off = pl.slot_smem;
    pl.slot_smem += (int)round_up(pl.slot_bytes, 16);
    pl.slot_bytes = 0;
  }
  pl.smem = fpb * pl.slot_smem;
  if (pl.smem > optin) return NBLDPC_ERR_UNSUPPORTED;
  const bool w4 = kq == 4 && resident && nthr == 32 && cs[0].warp4;
  const int dreg = pl.dreg = reg ? (pl.lanes < nthr ? -1 : 0)
                             : w4 ? (cs[0].dreg == 4 ? -4 : -1) : (kq != 0 && nc == 1) ? cs[0].dreg : 0;
  int st = prepare_kernel(kq, kv, km, dreg, dev, optin);
  if (st != NBLDPC_OK) return st;
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&pl.per_sm, kernel_for(kq, kv, km, dreg), pl.threads, pl.smem) !=
      cudaSuccess)
    return NBLDPC_ERR_CUDA;
  if (pl.per_sm < 1) return NBLDPC_ERR_UNSUPPORTED;
  pl.grid_max = pl.per_sm * sms;
  *out = pl;
  return NBLDPC_OK;
}

// Variant when nothing better is known: the one measured fastest for the
// benchmark codes on GB300 (GF(8) to GF(64): layout 1 from GF(16) on, with the
// messages in shared memory; GF(4): layout 0 with the messages in shared
// memory; GF(128), GF(256): pruned convolutions, layout 0 (GF(256) (2,6) N=384:
// 3.2x the dense kernel; GF(128) (2,4) N=256: 35.6 against 41.1 ms); otherwise
// layout 0).
int default_variant(int q) { return q >= 128 ? 4 : (q >= 16 && q <= 64) ? 3 : q >= 4 ? 2 : 0; }

// Frame slots per block when nothing better is known: enough threads per slot
// for the checks and variable nodes of one frame, at least one warp.
int default_fpb(const nbldpc_code* c) {
  if (warp4_code(c)) return 8;
  const int G = group_lanes(c->q, default_variant(c->q) & 1);
  const int work = c->m * G;
  int fpb = 1;
  while (fpb < 8 && kThreads / (2 * fpb) >= 32 && kThreads / (2 * fpb) >= work && kThreads / (2 * fpb) >= G) fpb *= 2;
  return fpb;
}

int configure(nbldpc_code* c, int variant, int fpb) {
  Plan pl{};
  const CodeNeeds need = needs_of(c, variant, c->mb);
  const int st = make_plan(c->q, variant, kmode(c), fpb, &need, 1, &pl);
  if (st != NBLDPC_OK) return st;
  c->variant = variant;
  c->plan = pl;
  c->has_group = false;
  // (the limit serves the FFT-SPA clusters too, which the min-max settings do not touch)
  int optin = 0;
  if (cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, c->device) != cudaSuccess) optin = 0;
  c->smem_optin = optin;
  c->split_max = kmode(c) != 3 && optin > 0 ? split_max(c->q, c->mb, c->dreg, c->device, optin) : 0;
  return NBLDPC_OK;
}

// The register form (q = 8, 16, 32) with the frames per block that keep most threads of an
// SM resident, the larger of equals (GF(16) N=100: 4 frames 845 us, 2 frames 887; GF(32)
// (2,8) N=508, where two frames leave 8 warps: 1 frame 7.87 ms, 2 frames 8.99).  q = 32 with
// a fifth of the lanes without a check stays in the group form (N=96, 48 checks on 64 lanes:
// 2.93 ms against 2.74; N=128, 64 checks: 2.44 against 2.85).
int configure_reg(nbldpc_code* c, int variant) {
  const int nthr = reg_threads(c->m), rounds = (c->m + nthr - 1) / nthr;
  if (c->q == 32 && 5 * c->m <= 4 * nthr * rounds) return NBLDPC_ERR_UNSUPPORTED;
  const CodeNeeds need = needs_of(c, variant, c->mb);
  int best = 0, most = 0;
  for (int fpb = 1; fpb <= 8 && fpb * nthr <= nbldpc::kResidentThreads; fpb *= 2) {
    Plan pl{};
    const int st = make_plan(c->q, variant, kmode(c), fpb, &need, 1, &pl);
    if (st == NBLDPC_ERR_CUDA) return st;
    if (st == NBLDPC_OK && pl.lanes == nthr && pl.per_sm * pl.threads >= most) {
      most = pl.per_sm * pl.threads;
      best = fpb;
    }
  }
  return best ? configure(c, variant, best) : NBLDPC_ERR_UNSUPPORTED;
}

// Frames up to which an untuned GF(16) or GF(32) handle decodes in the group form.  A lane per
// check takes long with few checks, and a chip that is not full does not make up for it; the
// group form spreads a check over 8 (q = 16) or 16 lanes.  The limits are frames per SM, from
// sweeps of 20 to 16,000 frames over codes of 32 to 512 checks on GB300 (us per decode of up to
// 30 iterations with early stop, group form against register form with the frames per block
// of choose_plan):
//  - GF(16): N=64, 100 / 1,300 / 4,000 frames 75 / 140 / 253 against 126 / 158 / 255; N=96 (3,6),
//    152 / 1,300 / 2,700 frames 185 / 340 / 535 against 197 / 436 / 560; N=128 (64 checks), 300
//    frames 160 against 128.
//  - GF(32): N=64, 600 / 4,000 / 16,000 frames 199 / 541 / 1,689 against 449 / 781 / 1,743; N=128,
//    1,300 / 8,000 frames 522 / 1,766 against 649 / 1,652; N=256 (128 checks), 600 frames 725
//    against 610.
//  - Fixed iterations fill the chip sooner: N=64, 100 / 600 frames 29 / 52 against 47 / 48 at
//    GF(16), 50 / 111 against 152 / 156 at GF(32); GF(32) N=160, 450 / 600 frames 197 / 250
//    against 236 / 235; 32 checks of degree 4 and 8, 1,900 frames 320 and 743 against 300 and 936.
int group_frames(const nbldpc_code* c, int early_stop) {
  int per_sm = 0;
  if (c->q == 16 && c->m <= 50) per_sm = early_stop ? 16 : c->m <= 32 ? 3 : 1;
  if (c->q == 32) {
    if (c->m <= 32) per_sm = early_stop ? 1 << 16 : c->n <= 2 * c->m ? 12 : 18;
    else if (c->m <= 100) per_sm = early_stop ? 36 : 3;
    else if (c->m < 192) per_sm = early_stop ? 0 : 1;
  }
  return per_sm * (c->plan.grid_max / c->plan.per_sm);
}

// The launch shape of a handle that nobody tuned, for its message width and schedule.
// Minimal schedule, 8 bits: the resident-message form (384-thread blocks of 1, 2 or 4 frames)
// where it fits shared memory, otherwise the same layout with the messages in the workspace.
int configure_default(nbldpc_code* c) {
  const int v = default_variant(c->q), fpb = default_fpb(c);
  if (kmode(c) != 1) return configure(c, v & 1, reg_form(c->q) || v == 0 ? fpb : 1);
  int st = NBLDPC_ERR_UNSUPPORTED;
  if (reg_form(c->q)) {
    st = configure_reg(c, v);
    if (st == NBLDPC_OK && group_frames(c, 0) + group_frames(c, 1) > 0) {
      const CodeNeeds need = needs_of(c, v & 1, c->mb);
      const int st2 = make_plan(c->q, v & 1, 1, fpb, &need, 1, &c->group);
      if (st2 == NBLDPC_ERR_CUDA) return st2;
      c->has_group = st2 == NBLDPC_OK;
    }
  } else if (v >= 2) st = configure(c, v, (v & 2) && fpb > 4 && !warp4_code(c) ? 4 : fpb);
  return st == NBLDPC_ERR_UNSUPPORTED ? configure(c, v & 1, fpb) : st;
}

// The launch shape after a change of the message width or the schedule: a tuning that was set or
// measured keeps the layout (resident messages serve 8-bit codes and the minimal schedule only),
// any other handle has the default of its new mode, whatever it was before.
int configure_mode(nbldpc_code* c) {
  if (!c->tuned) return configure_default(c);
  const int v = kmode(c) == 1 ? c->variant : c->variant & 1;
  return configure(c, v, v == c->variant ? c->plan.fpb : reg_form(c->q) && !c->pinned ? default_fpb(c) : 1);
}

// The one-block launch shape of a call: a tuning that was set or measured as it is.  An untuned
// handle's frames share blocks only as long as that leaves three blocks to two SMs (GF(16)
// N=100, 300 frames 127 us in blocks of one frame, 159 in blocks of four; 10 fixed iterations of
// 900 frames of N=64 86 us in blocks of one, 60 in blocks of four).
Plan choose_plan(const nbldpc_code* c, int frames, int early_stop, int* variant) {
  *variant = c->variant;
  if (c->has_group && frames <= group_frames(c, early_stop)) {
    *variant = c->variant & 1;
    return c->group;
  }
  Plan pl = c->plan;
  if (c->tuned || pl.lanes == 0) return pl;
  const int sms = pl.grid_max / pl.per_sm;
  while (pl.fpb > 1 && 2 * frames < 3 * pl.fpb * sms) {
    pl.fpb /= 2;
    pl.threads /= 2;
    pl.smem /= 2;
    pl.grid_max *= 2;
  }
  return pl;
}

// Enough for `frames` frames and any smaller number, with and without early stop.
size_t decode_ws_bytes(const nbldpc_code* c, int frames) {
  size_t most = ws_bytes(c->plan, frames);
  if (c->has_group)
    most = std::max(most, ws_bytes(c->group, std::min(frames, std::max(group_frames(c, 0), group_frames(c, 1)))));
  return most;
}

nbldpc::JobDesc job_desc(const nbldpc_code* c, const uint8_t* gamma, int frames, int max_iters, int early_stop,
                         uint8_t* sym, int32_t* iters, uint8_t* ok, int item_begin, bool count = true) {
  nbldpc::JobDesc j{};
  j.blob = c->blob_dev;
  j.off = c->off;
  j.gamma = gamma;
  j.out_sym = sym;
  j.out_iters = iters;
  j.out_ok = ok;
  j.q = c->q;
  j.n = c->n;
  j.m = c->m;
  j.dmax = c->dmax;
  j.work = count ? c->work_counter : nullptr;
  j.vmax = c->vmax;
  j.perm_at = c->off.perm;
  j.key16 = (255 * (c->vmax + 1) + 1) * c->q <= 65536 ? 1 : 0;
  j.group_bytes = group_bytes(c->q, c->dmax, c->mb, false);
  j.frames = frames;
  j.max_iters = max_iters;
  j.early_stop = early_stop ? 1 : 0;
  j.item_begin = item_begin;
  return j;
}

// Queue the counter reset (not needed when every frame has its own slot) and the
// persistent kernel (grid blocks) on st.
template <int N>
int launch_plan(const void* kernel, const Plan& pl, nbldpc::LaunchParamsOf<N>& lp, int grid, void* counter, uint8_t* msg,
                cudaStream_t st) {
  if (lp.total_items == 0 || grid < 1) return NBLDPC_OK;
  lp.counter = reinterpret_cast<unsigned int*>(counter);
  lp.msg = msg;
  lp.slot_bytes = pl.slot_bytes;
  lp.fpb = pl.fpb;
  lp.slot_smem = pl.slot_smem;
  lp.blob_cap = pl.blob_cap;
  lp.n_cap = pl.n_cap;
  lp.xs_off = pl.xs_off;
  // no more frames than frame slots: slot s takes frame s, no counter to reset
  lp.static_items = (long long)lp.total_items <= (long long)grid * pl.fpb ? 1 : 0;
  cudaError_t e = cudaSuccess;
  if (!lp.static_items) {
    e = cudaMemsetAsync(counter, 0, sizeof(unsigned int), st);
    if (e != cudaSuccess) return NBLDPC_ERR_CUDA;
  }
  void* args[] = {&lp};
  e = cudaLaunchKernel(kernel, dim3(grid), dim3(pl.threads), args, (size_t)pl.smem, st);
  if (e != cudaSuccess) return NBLDPC_ERR_CUDA;
  g_launches.fetch_add(1, std::memory_order_relaxed);
  return NBLDPC_OK;
}

// ---- frames split over the blocks of a cluster ------------------------------
// Shape of a split launch: ranks per frame, threads per rank, shared memory of a rank.
struct SplitShape {
  int size = 0, threads = 0, smem = 0;
  nbldpc::SplitLayout lay{};
};

// What a rank of a mixed batch keeps behind its sections (its job and SplitCtx).
constexpr size_t kSplitTail = (sizeof(nbldpc::JobDesc) + 15) / 16 * 16 + (sizeof(nbldpc::SplitCtx) + 15) / 16 * 16;

// Lay out a rank's shared memory; size 0 when it does not fit the device.
SplitShape split_layout(const nbldpc_code* c, int size, int threads) {
  SplitShape s;
  const int G = group_lanes(c->q, mixed_layout(c->q));
  s.lay.cpc = (c->m + size - 1) / size;
  s.lay.npc = (c->n + size - 1) / size;
  const long long edges_r = std::min<long long>(c->nnz, (long long)s.lay.cpc * c->dmax);
  const long long edges_n = std::min<long long>(c->nnz, (long long)s.lay.npc * c->vmax);
  // Every section on a 128-byte line, all banks, unless the padding costs a resident block: where the
  // scratch of two groups of a warp starts in the middle of a line, their vectors meet in the banks (GF(32)
  // (3,6) N=600, 25 frames: 345 us, 335 on lines; but 225 frames of GF(256) (2,8) N=156 and 9 of N=280 in
  // one batch 5,040 us with three blocks an SM, 3,767 with four).
  auto lay_out = [&](size_t line) {
    size_t o = round_up((size_t)c->off.perm, line);
    auto take = [&](size_t bytes) { const size_t at = o; o = round_up(o + bytes, line); return (int)at; };
    s.lay.chat_off = take((size_t)c->n);
    s.lay.flag_off = take(2 * nbldpc::kMaxSplit * sizeof(int));
    s.lay.row_off = take((size_t)edges_n * sizeof(void*));
    s.lay.gam_off = take((size_t)s.lay.npc * c->q);
    s.lay.scratch_off = take((size_t)(threads / G) * group_bytes(c->q, c->dmax, c->mb, c->mb == 1 && c->q >= 128));
    s.lay.x_off = take((size_t)edges_r * c->q * c->mb);
    return o;
  };
  auto blocks = [&](size_t smem) { return ((size_t)c->smem_optin + 1024) / (smem + kSplitTail + 1024); };
  const size_t tight = lay_out(16), lines = lay_out(128);
  const size_t o = lines > (size_t)c->smem_optin || blocks(lines) < blocks(tight) ? lay_out(16) : lines;
  if (o > (size_t)c->smem_optin) return SplitShape{};
  s.size = size;
  s.threads = threads;
  s.smem = (int)o;
  return s;
}

// Threads of the split-frame blocks of one shape that an SM holds (80 registers a thread).
int split_resident(const nbldpc_code* c, const SplitShape& s) {
  const int by_smem = (c->smem_optin + 1024) / (s.smem + 1024), by_regs = 65536 / (80 * s.threads);
  return std::min(by_smem, by_regs) * s.threads;
}

// The split shape of a batch, or size 0 for the one-block-per-frame kernels.
//
// One block per frame leaves SMs idle below their number, and with early stop
// it leaves them idle at the end of a batch, when the last frames run all their
// iterations (a GF(64) N=576 frame: 56 us an iteration on one SM, 6.4 us on
// 16).  Measured on GB300, us per decode of up to 20 or 30 iterations, one
// block per frame against this rule: GF(64) N=576, 1 / 96 / 200 frames
// 1085 / 1142 / 1915 against 158 / 494 / 794; GF(256) (2,6) N=384 6080 / 6609 /
// 8330 against 502 / 2206 / 4519; GF(256) (2,8) N=128, 17 frames 2135 against
// 464; GF(32) N=600 (register form), 1 / 96 / 450 frames 814 / 814 / 1612
// against 151 / 436 / 1357; GF(16) N=1024, 1 / 48 frames 213 / 215 against
// 97 / 175.
//  - More ranks and threads for fewer frames, so that the SMs are filled and the
//    frame's chain of passes is as short as they allow.
//  - No more 128-thread ranks than the frame has check-node lanes for.
//  - q <= 8 stays (GF(8) N=512, one frame 83 against 109: the passes are shorter
//    than the cluster's barriers), but for the 16-bit messages of q = 8.
//  - GF(16) codes of one 256-thread block per frame keep it (N=64: 75 us against 99 to 110); the
//    few ranks of short GF(32) codes have a thread per lane up to one frame per SM (N=96 (3,6),
//    152 frames: 318 us with 128 threads, 245 with 256).
//  - The register form (q = 16, 32) is fast enough alone from 5/8 frame per SM on at
//    q = 16 (200 frames of N=1024 351 against 346, of N=444 251 against 284), from
//    three on at q = 32 (700 frames 1960 against 1985); 3/8 and 5/8 without early stop
//    (96 frames of GF(16) 126 against 158, 152 of GF(32) 431 against 446).
//  - Up to twice the frames that the one-block kernels hold at once when frames
//    stop early (beyond it the tail is short and the ranks' barriers cost 2-5 %);
//    half of them where the ranks fill an SM less than three quarters as full
//    (GF(256): 400 frames of N=384 12.9 ms against 15.6); a third when
//    every frame runs the same iterations (no tail: 1000 frames 7.1 ms against 7.7).
//  - 16-bit messages: as many frames as the one-block kernels hold, half at q = 8
//    (GF(64) N=576, 1 / 96 / 450 frames 1548 / 1629 / 3643 against 165 / 564 / 1890;
//    GF(256) N=384, 200 frames 26.3 against 12.1 ms; GF(8) N=512, 200 frames
//    217 against 167).
SplitShape split_shape(const nbldpc_code* c, int frames, int early_stop) {
  if (c->split_max == 0 || c->pinned) return SplitShape{};
  const long long slots = (long long)c->plan.grid_max * c->plan.fpb;
  if (frames > 2 * slots) return SplitShape{};
  const int sms = c->plan.grid_max / c->plan.per_sm;
  const int G = group_lanes(c->q, mixed_layout(c->q));
  int size = frames <= sms / 8 ? 16 : 8;
  int threads = frames <= 3 * sms / 8 ? 384 : frames <= 3 * sms / 4 ? 256 : 128;
  size = std::min(size, c->split_max);
  if (c->has_group && c->q == 16 && c->m * G <= 256) return SplitShape{};
  while (size > 2 && (long long)size * 128 > (long long)c->m * G * 5 / 4) size /= 2;
  if (c->has_group && size < 8 && threads == 128 && frames <= sms) threads = 256;
  const int cpc = (c->m + size - 1) / size;
  const int pair = c->mb == 1 && c->q >= 128 && frames <= 3 * sms / 8 ? 2 : 1;   // two warps to a check
  threads = std::min(threads, std::max(128, (int)round_up((size_t)cpc * G * pair, 32)));
  SplitShape s = split_layout(c, size, threads);
  while (s.size == 0 && threads > 64) s = split_layout(c, size, threads = (threads - 1) / 64 * 64);
  if (s.size == 0) return s;
  long long most = early_stop ? 2 * slots : slots / 3;
  if (c->mb == 2) most = std::min(most, c->q == 8 ? slots / 2 : slots);
  else if (reg_form(c->q) && (c->variant & 2))
    most = c->q == 16 ? (early_stop ? 5 : 3) * sms / 8 : early_stop ? 3 * sms : 5 * sms / 8;
  else if (4 * split_resident(c, s) < 3 * c->plan.per_sm * c->plan.threads) most = std::min(most, slots / 2);
  return frames <= most ? s : SplitShape{};
}

int launch_split(const nbldpc_code* c, const SplitShape& s, const nbldpc::JobDesc& job, cudaStream_t st) {
  nbldpc::SplitParams p{job, s.size, s.lay};
  return split_launch(split_kernel_for(c->q, c->mb, c->dreg), job.frames, s.size, s.threads, s.smem, &p, st);
}

// choose: the kernel follows the number of frames (not while the autotuner times a tuning)
int launch(const nbldpc_code* c, const uint8_t* gamma, int frames, int max_iters, int early_stop, uint8_t* sym,
           int32_t* iters, uint8_t* ok, void* ws, cudaStream_t st, bool count = true, bool choose = true) {
  if (frames == 0) return NBLDPC_OK;
  int variant = c->variant;
  Plan pl = c->plan;
  if (choose) {
    const SplitShape s = split_shape(c, frames, early_stop);
    if (s.size) return launch_split(c, s, job_desc(c, gamma, frames, max_iters, early_stop, sym, iters, ok, 0, count), st);
    pl = choose_plan(c, frames, early_stop, &variant);
  }
  nbldpc::LaunchParamsOf<1> lp{};
  lp.jobs[0] = job_desc(c, gamma, frames, max_iters, early_stop, sym, iters, ok, 0, count);
  lp.jobs[0].reg = pl.lanes;
  lp.njobs = 1;
  lp.total_items = frames;
  return launch_plan(kernel_for(c->q, variant, kmode(c), pl.dreg), pl, lp, grid_for(pl, frames), ws,
                     reinterpret_cast<uint8_t*>(ws) + 256, st);
}

// ---- non-allocating decode (nbldpc_decode_noalloc) -------------------------
// Fixed scratch for callers that cannot allocate: frame counter + message slots.
static __device__ __align__(256) unsigned char g_noalloc_scratch[NBLDPC_NOALLOC_SCRATCH_BYTES];

// Device address of g_noalloc_scratch in the current device's context.  Looked
// up on every call (a cheap table lookup once the module is loaded), so the
// address stays right after a context is torn down and re-created; host code
// must not use the symbol itself, which names a host-side stand-in.
int noalloc_scratch(void** out) {
  void* p = nullptr;
  if (cudaGetSymbolAddress(&p, g_noalloc_scratch) != cudaSuccess || !p) return NBLDPC_ERR_CUDA;
  *out = p;
  return NBLDPC_OK;
}

bool valid_outputs(const uint8_t* gamma, const uint8_t* sym, const int32_t* iters, const uint8_t* ok) {
  return gamma && sym && iters && ok && aligned(gamma, 16) && aligned(iters, 4);
}

}  // namespace

extern "C" {

int nbldpc_decode_noalloc(const nbldpc_code* c, const uint8_t* gamma_dev, int frames, int max_iters,
                          int early_stop, uint8_t* out_sym_dev, int32_t* out_iters_dev, uint8_t* out_ok_dev,
                          void* cuda_stream) {
  if (!c || frames < 0 || max_iters < 0) return NBLDPC_ERR_ARG;
  if (frames == 0) return NBLDPC_OK;
  if (!valid_outputs(gamma_dev, out_sym_dev, out_iters_dev, out_ok_dev)) return NBLDPC_ERR_ARG;
  int st = check_device(c);
  if (st != NBLDPC_OK) return st;
  int variant = 0;
  const Plan pl = choose_plan(c, frames, early_stop, &variant);
  const size_t per_block = (size_t)pl.fpb * pl.slot_bytes;   // 0 when the messages stay in shared memory
  if (256 + per_block > (size_t)NBLDPC_NOALLOC_SCRATCH_BYTES) return NBLDPC_ERR_UNSUPPORTED;
  int grid = grid_for(pl, frames);
  if (per_block) {
    const int fit = (int)(((size_t)NBLDPC_NOALLOC_SCRATCH_BYTES - 256) / per_block);
    if (grid > fit) grid = fit;
  }
  st = cuda_status(cudaGetLastError());
  if (st != NBLDPC_OK) return st;
  const SplitShape sp = split_shape(c, frames, early_stop);
  if (sp.size)
    return launch_split(c, sp,
                        job_desc(c, gamma_dev, frames, max_iters, early_stop, out_sym_dev, out_iters_dev, out_ok_dev, 0),
                        reinterpret_cast<cudaStream_t>(cuda_stream));
  void* scratch = nullptr;
  st = noalloc_scratch(&scratch);
  if (st != NBLDPC_OK) return st;
  // the array keeps the previous call's contents: the frame counter is cleared in launch_plan
  nbldpc::LaunchParamsOf<1> lp{};
  lp.jobs[0] = job_desc(c, gamma_dev, frames, max_iters, early_stop, out_sym_dev, out_iters_dev, out_ok_dev, 0);
  lp.jobs[0].reg = pl.lanes;
  lp.njobs = 1;
  lp.total_items = frames;
  return launch_plan(kernel_for(c->q, variant, kmode(c), pl.dreg), pl, lp, grid, scratch,
                     reinterpret_cast<uint8_t*>(scratch) + 256,
                     reinterpret_cast<cudaStream_t>(cuda_stream));
}

const char* nbldpc_status_string(int status) {
  switch (status) {
    case NBLDPC_OK: return "ok";
    case NBLDPC_ERR_ARG: return "invalid argument";
    case NBLDPC_ERR_POLY: return "field order not a power of two in [2,256] or polynomial not primitive";
    case NBLDPC_ERR_H: return "malformed parity-check matrix";
    case NBLDPC_ERR_CUDA: return "CUDA error";
    case NBLDPC_ERR_NOMEM: return "out of memory";
    case NBLDPC_ERR_TIMEOUT: return "device-side wait timed out";
    case NBLDPC_ERR_UNSUPPORTED: return "code outside the supported limits";
  }
  return "unknown status";
}

uint64_t nbldpc_kernel_launch_count(void) { return g_launches.load(); }

int nbldpc_code_create(int q, uint32_t prim_poly, int n_cols, int n_rows, const int32_t* row_ptr,
                       const int32_t* col_idx, const uint8_t* coef, nbldpc_code** out) {
  if (!out) return NBLDPC_ERR_ARG;
  *out = nullptr;
  if (!row_ptr || !col_idx || !coef || n_cols <= 0 || n_rows <= 0) return NBLDPC_ERR_ARG;
  if (q < 2 || q > 256 || (q & (q - 1))) return NBLDPC_ERR_POLY;
  std::vector<uint8_t> exp2, lg;
  if (!build_field(q, prim_poly, exp2, lg)) return NBLDPC_ERR_POLY;
  if (row_ptr[0] != 0) return NBLDPC_ERR_H;
  for (int r = 0; r < n_rows; ++r)
    if (row_ptr[r + 1] - row_ptr[r] < 2) return NBLDPC_ERR_H;
  const int64_t nnz64 = row_ptr[n_rows];
  if (n_cols >= 65535 || nnz64 >= 65535) return NBLDPC_ERR_UNSUPPORTED;
  const int nnz = (int)nnz64;
  std::vector<int> vdeg(n_cols, 0), last(n_cols, -1);
  int dmax = 0;
  for (int r = 0; r < n_rows; ++r) {
    const int d = row_ptr[r + 1] - row_ptr[r];
    if (d > dmax) dmax = d;
    for (int e = row_ptr[r]; e < row_ptr[r + 1]; ++e) {
      const int c = col_idx[e];
      if (c < 0 || c >= n_cols || coef[e] == 0 || coef[e] >= q || last[c] == r) return NBLDPC_ERR_H;
      last[c] = r;
      ++vdeg[c];
    }
  }
  int vmax = 0;
  for (int c = 0; c < n_cols; ++c) {
    if (vdeg[c] < 1) return NBLDPC_ERR_H;
    if (vdeg[c] > vmax) vmax = vdeg[c];
  }
  if (dmax > 64 || vmax > 64) return NBLDPC_ERR_UNSUPPORTED;

  // code blob: exp2 | log | row_ptr u16 | edge_lh u8 | edge_lhi u8 | edge_col u16 | vn_ptr u16 | vn_edge u16
  nbldpc::CodeBlob off{};
  size_t o = 0;
  auto take = [&](size_t bytes) { const size_t at = o; o = round_up(o + bytes, 16); return (int)at; };
  off.exp2 = take(2 * (size_t)q);
  off.log = take((size_t)q);
  off.row_ptr = take(2 * ((size_t)n_rows + 1));
  off.edge_lh = take((size_t)nnz);
  off.edge_lhi = take((size_t)nnz);
  off.edge_col = take(2 * (size_t)nnz);
  off.vn_ptr = take(2 * ((size_t)n_cols + 1));
  off.vn_edge = take(2 * (size_t)nnz);
  const int perm_row = q == 8 ? nbldpc::PermRow<8>::bytes : q == 16 ? nbldpc::PermRow<16>::bytes
                     : q == 32 ? nbldpc::PermRow<32>::bytes : 0;
  off.perm = (int)o;
  off.bytes = (int)(o + round_up((size_t)perm_row * (q - 1), 16));
  // FFT-SPA section: warp tasks pack consecutive checks with at most 32 edges in all
  std::vector<uint16_t> tasks;
  for (int r = 0; r < n_rows;) {
    tasks.push_back((uint16_t)r);
    int edges = 0;
    while (r < n_rows && edges + (row_ptr[r + 1] - row_ptr[r]) <= 32) edges += row_ptr[r + 1] - row_ptr[r], ++r;
    if (edges == 0) ++r;   // a check of degree > 32: its own task (such codes are rejected for q <= 64)
  }
  tasks.push_back((uint16_t)n_rows);
  const int pbits = [&] { int b = 0; while ((1 << b) < q) ++b; return b; }();
  off.edge_row = take(2 * (size_t)nnz);
  off.task_c0 = take(2 * tasks.size());
  off.at_log = take((size_t)(q - 1) * pbits);
  off.fft_bytes = (int)o;
  off.perm_src = take((size_t)perm_row * (q - 1));
  std::vector<unsigned char> blob(o, 0);
  {
    uint16_t* er = reinterpret_cast<uint16_t*>(&blob[off.edge_row]);
    for (int r = 0; r < n_rows; ++r)
      for (int e = row_ptr[r]; e < row_ptr[r + 1]; ++e) er[e] = (uint16_t)r;
    memcpy(&blob[off.task_c0], tasks.data(), 2 * tasks.size());
    // at_log[lc][i] = M_c^T e_i for c = x^lc: bit k is bit i of c x^k
    uint8_t* at = &blob[off.at_log];
    for (int lc = 0; lc < q - 1; ++lc)
      for (int i = 0; i < pbits; ++i) {
        int a = 0;
        for (int k = 0; k < pbits; ++k) a |= ((exp2[lc + k] >> i) & 1) << k;
        at[lc * pbits + i] = (uint8_t)a;
      }
  }
  // selectors of "byte y is byte h y of the row" for h = x^lh (PermRow): nibbles of the low
  // three bits of h y, then one mask word per four bytes for bit 3 and for bit 4
  for (int lh = 0; perm_row && lh < q - 1; ++lh)
    for (int y = 0; y < q; ++y) {
      unsigned char* t = &blob[off.perm_src + (size_t)lh * perm_row];
      const int i = y ? exp2[lg[y] + lh] : 0;
      t[y / 2] |= (unsigned char)((i & 7) << (4 * (y & 1)));
      const int sel = q == 8 ? nbldpc::PermRow<8>::sel_bytes : 16;
      if (q >= 16 && (i & 8)) t[sel + y] = 0xFF;
      if (q >= 32 && (i & 16)) t[sel + q + y] = 0xFF;
    }
  memcpy(&blob[off.exp2], exp2.data(), 2 * (size_t)q);
  memcpy(&blob[off.log], lg.data(), (size_t)q);
  uint16_t* rp = reinterpret_cast<uint16_t*>(&blob[off.row_ptr]);
  uint16_t* ec = reinterpret_cast<uint16_t*>(&blob[off.edge_col]);
  uint8_t* elh = &blob[off.edge_lh];
  uint8_t* elhi = &blob[off.edge_lhi];
  uint16_t* vp = reinterpret_cast<uint16_t*>(&blob[off.vn_ptr]);
  uint16_t* ve = reinterpret_cast<uint16_t*>(&blob[off.vn_edge]);
  for (int r = 0; r <= n_rows; ++r) rp[r] = (uint16_t)row_ptr[r];
  for (int e = 0; e < nnz; ++e) {
    ec[e] = (uint16_t)col_idx[e];
    elh[e] = lg[coef[e]];
    elhi[e] = (uint8_t)((q - 1 - lg[coef[e]]) % (q - 1));
  }
  vp[0] = 0;
  for (int c = 0; c < n_cols; ++c) vp[c + 1] = (uint16_t)(vp[c] + vdeg[c]);
  std::vector<int> fill(n_cols, 0);
  for (int e = 0; e < nnz; ++e) {
    const int c = col_idx[e];
    ve[vp[c] + fill[c]++] = (uint16_t)e;
  }

  nbldpc_code* c = new (std::nothrow) nbldpc_code();
  if (!c) return NBLDPC_ERR_NOMEM;
  c->q = q;
  c->p = 0;
  while ((1 << c->p) < q) ++c->p;
  c->n = n_cols;
  c->m = n_rows;
  c->nnz = nnz;
  c->dmax = dmax;
  c->vmax = vmax;
  c->dreg = dmax;                      // regular check degree, or 0 when the rows differ
  for (int r = 0; r < n_rows; ++r)
    if (row_ptr[r + 1] - row_ptr[r] != dmax) c->dreg = 0;
  c->ntasks = (int)tasks.size() - 1;
  c->poly = prim_poly;
  c->off = off;
  if (cudaGetDevice(&c->device) != cudaSuccess) { delete c; return NBLDPC_ERR_CUDA; }
  cudaError_t e = cudaMalloc(reinterpret_cast<void**>(&c->blob_dev), o);
  if (e != cudaSuccess) { delete c; return e == cudaErrorMemoryAllocation ? NBLDPC_ERR_NOMEM : NBLDPC_ERR_CUDA; }
  e = cudaMemcpy(c->blob_dev, blob.data(), o, cudaMemcpyHostToDevice);
  int st = cuda_status(e);
  if (st == NBLDPC_OK) st = configure_default(c);
  if (st == NBLDPC_OK) {
    c->fft_status = fft_configure(c, row_ptr);
    if (c->fft_status == NBLDPC_ERR_CUDA) st = NBLDPC_ERR_CUDA;
  }
  if (st != NBLDPC_OK) {
    cudaFree(c->blob_dev);
    delete c;
    return st;
  }
  *out = c;
  return NBLDPC_OK;
}

void nbldpc_code_destroy(nbldpc_code* c) {
  if (!c) return;
  for (auto& ev : c->ev)
    if (ev) cudaEventDestroy(ev);
  if (c->side) cudaStreamDestroy(c->side);
  if (c->blob_dev) cudaFree(c->blob_dev);
  delete c;
}

int nbldpc_code_info(const nbldpc_code* c, int* q, int* n, int* m, int* nnz) {
  if (!c) return NBLDPC_ERR_ARG;
  if (q) *q = c->q;
  if (n) *n = c->n;
  if (m) *m = c->m;
  if (nnz) *nnz = c->nnz;
  return NBLDPC_OK;
}

int nbldpc_code_get_tuning(const nbldpc_code* c, int* variant, int* frames_per_block) {
  if (!c) return NBLDPC_ERR_ARG;
  if (variant) *variant = c->variant;
  if (frames_per_block) *frames_per_block = c->plan.fpb;
  return NBLDPC_OK;
}

int nbldpc_code_set_tuning(nbldpc_code* c, int variant, int frames_per_block) {
  if (!c || variant < 0 || variant > 7 || frames_per_block < 1 || frames_per_block > 8 ||
      (frames_per_block & (frames_per_block - 1)))
    return NBLDPC_ERR_ARG;
  const int st = check_device(c);
  if (st != NBLDPC_OK) return st;
  const int st2 = configure(c, variant, frames_per_block);
  if (st2 == NBLDPC_OK) c->pinned = c->tuned = true;
  return st2;
}

int nbldpc_code_set_message_bits(nbldpc_code* c, int bits) {
  if (!c || (bits != 8 && bits != 16)) return NBLDPC_ERR_ARG;
  if (bits == 16 && c->cnp_schedule == NBLDPC_CNP_TABLE1) return NBLDPC_ERR_UNSUPPORTED;
  if (check_device(c) != NBLDPC_OK) return check_device(c);
  const int old = c->mb;
  c->mb = bits / 8;
  const int st = configure_mode(c);
  if (st != NBLDPC_OK) c->mb = old;
  return st;
}

int nbldpc_code_get_message_bits(const nbldpc_code* c, int* bits) {
  if (!c || !bits) return NBLDPC_ERR_ARG;
  *bits = 8 * c->mb;
  return NBLDPC_OK;
}

int nbldpc_code_set_cnp_schedule(nbldpc_code* c, int schedule) {
  if (!c || (schedule != NBLDPC_CNP_MINIMAL && schedule != NBLDPC_CNP_TABLE1)) return NBLDPC_ERR_ARG;
  if (schedule == NBLDPC_CNP_TABLE1 && c->mb != 1) return NBLDPC_ERR_UNSUPPORTED;
  if (check_device(c) != NBLDPC_OK) return check_device(c);
  const int old = c->cnp_schedule;
  c->cnp_schedule = schedule;
  const int st = configure_mode(c);
  if (st != NBLDPC_OK) c->cnp_schedule = old;
  return st;
}

int nbldpc_code_get_cnp_schedule(const nbldpc_code* c, int* schedule) {
  if (!c || !schedule) return NBLDPC_ERR_ARG;
  *schedule = c->cnp_schedule;
  return NBLDPC_OK;
}

int nbldpc_code_set_work_counter(nbldpc_code* c, unsigned long long* counter_dev) {
  if (!c || (counter_dev && !aligned(counter_dev, 8))) return NBLDPC_ERR_ARG;
  c->work_counter = counter_dev;
  return NBLDPC_OK;
}

int nbldpc_decode_workspace_size(const nbldpc_code* c, int frames, size_t* bytes) {
  if (!c || !bytes || frames < 0) return NBLDPC_ERR_ARG;
  *bytes = decode_ws_bytes(c, frames);
  return NBLDPC_OK;
}

int nbldpc_decode(const nbldpc_code* c, const uint8_t* gamma_dev, int frames, int max_iters, int early_stop,
                  uint8_t* out_sym_dev, int32_t* out_iters_dev, uint8_t* out_ok_dev, void* workspace_dev,
                  size_t workspace_bytes, void* cuda_stream) {
  if (!c || frames < 0 || max_iters < 0) return NBLDPC_ERR_ARG;
  if (frames == 0) return NBLDPC_OK;
  if (!valid_outputs(gamma_dev, out_sym_dev, out_iters_dev, out_ok_dev) || !workspace_dev) return NBLDPC_ERR_ARG;
  if (!aligned(workspace_dev, 16)) return NBLDPC_ERR_ARG;
  if (workspace_bytes < decode_ws_bytes(c, frames)) return NBLDPC_ERR_ARG;
  int st = check_device(c);
  if (st != NBLDPC_OK) return st;
  st = cuda_status(cudaGetLastError());
  if (st != NBLDPC_OK) return st;
  return launch(c, gamma_dev, frames, max_iters, early_stop, out_sym_dev, out_iters_dev, out_ok_dev,
                workspace_dev, reinterpret_cast<cudaStream_t>(cuda_stream));
}

int nbldpc_decode_cluster_blocks(const nbldpc_code* c, int frames, int early_stop, int* blocks) {
  if (!c || !blocks || frames < 0) return NBLDPC_ERR_ARG;
  *blocks = frames ? split_shape(c, frames, early_stop).size : 0;
  return NBLDPC_OK;
}

// ---- mixed-code batches -----------------------------------------------------
// Frame slots per block with enough threads each for a check a thread.
static int reg_fpb(const nbldpc_code* c) {
  int fpb = 1;
  while (fpb < 8 && kThreads / (2 * fpb) >= std::max(32, c->m)) fpb *= 2;
  return fpb;
}

// Whether a job may take the register form in the mixed-code kernels: GF(32) codes of up to 100 checks
// for more frames than an untuned handle decodes in the group form, and with a check for four fifths
// of the lanes (1,000 frames of GF(32) N=64 and 2,000 of GF(4) N=100: 416 us against 265; 2,106 of
// (2,8) N=280, 70 checks on 128 lanes, fixed iterations 2,011 against 1,608).
static bool batch_reg(const nbldpc_job& j) {
  const nbldpc_code* c = j.code;
  if (!reg_form(c->q)) return false;
  return c->q != 32 || c->m > 100 ||
         (j.frames > group_frames(c, j.early_stop) && 5 * c->m > 4 * (kThreads / reg_fpb(c)));
}

// Frame slots per block that suit a job in the mixed-code kernels: the pinned count, or (register
// form) enough threads per slot for the checks, or the group form's default.
static int batch_fpb(const nbldpc_job& j) {
  if (j.code->pinned || !reg_form(j.code->q)) return j.code->plan.fpb;
  return batch_reg(j) ? reg_fpb(j.code) : default_fpb(j.code);
}

// Time (us) of a frame's longest decode alone on a block: ns per edge and iteration as measured on
// GB300 (20 frames, two-block kernel: GF(4) N=400 5.0 us an iteration, GF(8) N=512 4.4, GF(16) N=1024
// 12.7, GF(32) N=600 52, GF(64) N=576 65, GF(128) N=256 127, GF(256) (2,8) N=128 107), and 1.5 us.
static double frame_us(const nbldpc_job& j) {
  static const double ns[9] = {0, 6, 5, 6, 10, 30, 56, 250, 420};
  return j.max_iters * (1.5 + 1e-3 * ns[nbldpc::ilog2(j.code->q)] * j.code->nnz);
}

// Convolution work of a frame's longest decode (pruned convolutions as a tenth).
static double frame_work(const nbldpc_job& j) {
  const nbldpc_code* c = j.code;
  return (double)j.max_iters * c->nnz * c->q * c->q * (c->q >= 128 ? 0.1 : 1.0);
}

// Whether a code that has frames in the batch was tuned by hand: the batch then keeps the one-block
// kernel and the smallest frames-per-block value among its codes.
static bool any_pinned(const nbldpc_job* jobs, int n_jobs) {
  for (int i = 0; i < n_jobs; ++i)
    if (jobs[i].frames > 0 && jobs[i].code->pinned) return true;
  return false;
}

static int batch_plan(const nbldpc_job* jobs, int n_jobs, Plan* pl, int* total) {
  if (!jobs || n_jobs < 1 || n_jobs > NBLDPC_MAX_BATCH_JOBS) return NBLDPC_ERR_ARG;
  CodeNeeds need[NBLDPC_MAX_BATCH_JOBS];
  int fpb = 8;
  long long t = 0;
  for (int i = 0; i < n_jobs; ++i) {
    const nbldpc_code* c = jobs[i].code;
    if (!c || jobs[i].frames < 0 || jobs[i].max_iters < 0) return NBLDPC_ERR_ARG;
    const int st = check_device(c);
    if (st != NBLDPC_OK) return st;
    if (kmode(c) != 1) return NBLDPC_ERR_UNSUPPORTED;   // mixed-code launches: 8-bit messages, minimal schedule
    need[i] = needs_of(c, mixed_layout(c->q), 1);
    need[i].blob = c->off.edge_col;   // the mixed-code kernel stages no edge_col or variable-node view
    fpb = std::min(fpb, batch_fpb(jobs[i]));
    t += jobs[i].frames;
  }
  if (t > 0x7FFFFFFF) return NBLDPC_ERR_ARG;
  *total = (int)t;
  // few frames: a block each (GF(4) N=48 and GF(8) N=100, 200 frames each: 100 us at two a block, 92 at one),
  // unless a code's frames per block are pinned
  const nbldpc_code* c0 = jobs[0].code;
  const Plan& pl0 = c0->plan;
  if (t <= 3LL * (pl0.grid_max / pl0.per_sm) && !any_pinned(jobs, n_jobs)) fpb = 1;
  const int st = prepare_kernel(0, -2, 1, 0, c0->device, c0->smem_optin);
  return st != NBLDPC_OK ? st : make_plan(0, -1, 1, fpb, need, n_jobs, pl);
}

// Shape of a mixed batch whose frames are each decoded on a cluster (size 0: one block per frame
// slot): the ranks and threads of split_shape, the jobs' layouts one over the other.  Frames count
// by their time against the longest ones' (an eighth at least; five times that for q <= 8, which a
// cluster hardly shortens: 565 frames of GF(8) and GF(4) codes and 5 of GF(32) N=728 647 us on
// clusters, 358 on one block each; but 406 of GF(4) N=194 with one of GF(256) N=180 and 75 others 499
// and 1438): one block per frame ends with the longest frames alone.  Taken with early stop (the
// serving loop's groups) up to a number of such frames per SM that follows the widest field: q = 16
// 5/8; q = 32 two, below 1200 check-node lanes 3/4; q = 64 four and q = 128 three, below 1200 lanes
// one and a half; q = 256 three, two and a half above check degree 4 and one and a half from 8 on;
// without early stop 3/8; and eight frames of any kind.  Not for q <= 8 alone, nor past 3/8 where the
// longest frames have fewer than 1024 lanes, nor there for q <= 32 at all (and no more 128-thread
// ranks than lanes).  Measured on GB300, us per batch, the faster one-block kernel against this: 60 /
// 240 / 450 frames of GF(64) N=576, GF(16) N=1024 and GF(256) N=128 in equal parts 2746 / 3455 / 3878
// against 795 / 1444 / 2399; one frame of GF(64) 1243 against 179; 580 of GF(64) 2854 against 2558;
// beyond the limits 823 of GF(32) N=716 1100 against 1421, 947 of GF(128) N=138 1582 against 2020,
// 263 of GF(256) (2,8) N=280 3132 against 4940, 213 of two GF(32) codes of 1184 lanes 300 against 372.
static int batch_split(const nbldpc_job* jobs, int n_jobs, int total, const Plan& pl, nbldpc::SplitBatchParams* p,
                       SplitShape* out) {
  if (any_pinned(jobs, n_jobs)) return 0;
  const nbldpc_code* c0 = jobs[0].code;
  const int sms = pl.grid_max / pl.per_sm;
  bool stop = true;
  int q_most = 0, lanes = 0, degree = 0;       // widest field; the longest frames' check-node lanes and degree
  double longest = 0.0, like_longest = 0.0;
  for (int i = 0; i < n_jobs; ++i)
    if (jobs[i].frames > 0) {
      stop = stop && jobs[i].early_stop;
      q_most = std::max(q_most, jobs[i].code->q);
      if (frame_us(jobs[i]) >= longest) {
        longest = frame_us(jobs[i]);
        lanes = jobs[i].code->m * group_lanes(jobs[i].code->q, mixed_layout(jobs[i].code->q));
        degree = jobs[i].code->dmax;
      }
    }
  if (q_most <= 8 || total > 8 * sms) return 0;
  for (int i = 0; i < n_jobs; ++i) {
    const double like = longest > 0.0 ? frame_us(jobs[i]) / longest : 1.0;
    like_longest += jobs[i].frames * std::min(1.0, std::max(0.125, jobs[i].code->q <= 8 ? 5 * like : like));
  }
  const int most_frames = !stop          ? 3 * sms / 8
                          : q_most <= 16  ? 5 * sms / 8
                          : q_most <= 32  ? (lanes < 1200 ? 3 * sms / 4 : 2 * sms)
                          : q_most <= 128 ? (lanes < 1200 ? 3 * sms / 2 : q_most <= 64 ? 4 * sms : 3 * sms)
                          : degree <= 4   ? 3 * sms
                                          : (degree < 8 ? 5 : 3) * sms / 2;
  if (like_longest > most_frames || (lanes < 1024 && (q_most <= 32 || total > 3 * sms / 8))) return 0;
  const int most = split_max(0, 1, 0, c0->device, c0->smem_optin);
  int size = std::min(total <= sms / 8 ? 16 : 8, most);
  while (size > 2 && (long long)size * 128 > (long long)lanes * 5 / 4) size /= 2;
  if (size < 2) return 0;
  for (int threads = total <= 3 * sms / 8 ? 384 : total <= 3 * sms / 4 ? 256 : 128; threads >= 64; threads -= 64) {
    SplitShape all;
    bool fits = true;
    for (int i = 0; i < n_jobs && fits; ++i) {
      const SplitShape s = split_layout(jobs[i].code, size, threads);
      fits = s.size != 0;
      p->lay[i] = s.lay;
      all.smem = std::max(all.smem, s.smem);
    }
    if (!fits) continue;
    all.size = size;
    all.threads = threads;
    p->job_off = all.smem;
    p->sc_off = p->job_off + (int)round_up(sizeof(nbldpc::JobDesc), 16);
    all.smem = p->sc_off + (int)round_up(sizeof(nbldpc::SplitCtx), 16);
    if (all.smem > c0->smem_optin) continue;
    *out = all;
    return size;
  }
  return 0;
}

// Whether a mixed batch takes the two-block kernel with its paths in line.  It decodes a frame 5 to 30 %
// sooner (see decode_mixed_call), the three-block kernel has more of them side by side; three to a
// block of rounds (frame slots of three blocks an SM), measured on GB300, us per batch, two against
// three blocks:
//  - With early stop the last frames decide until the chip has been full six times over: GF(64) N=576,
//    1,100 / 1,400 / 6,000 frames 4,406 / 5,520 / 19,957 against 4,537 / 5,686 / 19,672; GF(64) N=88,
//    N=522 and N=232, 2,123 in all 2,340 against 2,791; GF(256) N=384, 2,000 39.4 against 39.2 ms; 532
//    of GF(16) N=716, GF(64) N=126 and others 1,333 against 1,541.
//  - Fields up to GF(16) gain little from it: where their rounds are not fewer than four thirds of the
//    other kernel's, the third block wins (GF(8) (3,6) N=580, 361 frames 220 against 164; GF(2) N=534,
//    1,290 697 against 612; GF(16) N=308, 818 553 against 512, four GF(16) codes, 1,643 1,383 against 1,297;
//    20 of GF(16) N=64 and 30 of GF(8) N=100 64 against 78), but for GF(16) frames that the three blocks
//    take at once (436 of N=216 and N=272 266 against 319).
//  - Fixed iterations: up to two and a half frames per SM (GF(64) N=576, 300 frames 939 against 979; 399
//    of four GF(64) codes 649 against 730; GF(256) N=177, 416 2,982 against 2,588), and for GF(128) and
//    GF(256) where rounds allow (GF(256) N=384, 600 frames 6,973 against 8,427).
static bool batch_wide(const nbldpc_job* jobs, int n_jobs, int total, const Plan& pl) {
  bool stop = true;
  double small = 0.0, q16 = 0.0, middle = 0.0, large = 0.0;   // work up to GF(8), of GF(16), up to GF(64), above
  for (int i = 0; i < n_jobs; ++i) {
    if (jobs[i].frames == 0) continue;
    stop = stop && jobs[i].early_stop;
    const int q = jobs[i].code->q;
    (q <= 8 ? small : q == 16 ? q16 : q <= 64 ? middle : large) += jobs[i].frames * frame_work(jobs[i]);
  }
  const long long want = (total + pl.fpb - 1) / pl.fpb, sms = pl.grid_max / pl.per_sm;
  const long long two = (want + 2 * sms - 1) / (2 * sms), three = (want + pl.grid_max - 1) / pl.grid_max;
  const bool fewer = three <= 3 && 3 * two < 4 * three;
  if (small + q16 > middle + large) return fewer || (q16 > small && stop && three == 1);
  if (stop) return three <= 6;
  return 2 * want <= 5 * sms || (large > small + q16 + middle && fewer);
}

int nbldpc_decode_batch_workspace_size(const nbldpc_job* jobs, int n_jobs, size_t* bytes) {
  if (!bytes) return NBLDPC_ERR_ARG;
  Plan pl{};
  int total = 0;
  const int st = batch_plan(jobs, n_jobs, &pl, &total);
  if (st != NBLDPC_OK) return st;
  *bytes = ws_bytes(pl, total);
  return NBLDPC_OK;
}

int nbldpc_decode_batch_cluster_blocks(const nbldpc_job* jobs, int n_jobs, int* blocks) {
  if (!blocks) return NBLDPC_ERR_ARG;
  Plan pl{};
  int total = 0;
  const int st = batch_plan(jobs, n_jobs, &pl, &total);
  if (st != NBLDPC_OK) return st;
  nbldpc::SplitBatchParams sp{};
  SplitShape shape;
  *blocks = total > 0 ? batch_split(jobs, n_jobs, total, pl, &sp, &shape) : 0;
  return NBLDPC_OK;
}

int nbldpc_decode_batch(const nbldpc_job* jobs, int n_jobs, void* workspace_dev, size_t workspace_bytes,
                        void* cuda_stream) {
  Plan pl{};
  int total = 0;
  int st = batch_plan(jobs, n_jobs, &pl, &total);
  if (st != NBLDPC_OK) return st;
  if (!workspace_dev || !aligned(workspace_dev, 16) || workspace_bytes < ws_bytes(pl, total)) return NBLDPC_ERR_ARG;
  nbldpc::LaunchParams<0> lp{};
  int begin = 0;
  // The jobs with the longest frames first, so that they are not the ones that end the launch.
  int order[NBLDPC_MAX_BATCH_JOBS];
  for (int i = 0; i < n_jobs; ++i) order[i] = i;
  std::stable_sort(order, order + n_jobs, [&](int a, int b) { return frame_work(jobs[a]) > frame_work(jobs[b]); });
  nbldpc_job sorted[NBLDPC_MAX_BATCH_JOBS];
  for (int i = 0; i < n_jobs; ++i) sorted[i] = jobs[order[i]];
  jobs = sorted;
  for (int i = 0; i < n_jobs; ++i) {
    const nbldpc_job& j = jobs[i];
    if (j.frames > 0 && !valid_outputs(j.gamma_dev, j.out_sym_dev, j.out_iters_dev, j.out_ok_dev))
      return NBLDPC_ERR_ARG;
    lp.jobs[i] = job_desc(j.code, j.gamma_dev, j.frames, j.max_iters, j.early_stop, j.out_sym_dev, j.out_iters_dev,
                          j.out_ok_dev, begin);
    begin += j.frames;
  }
  lp.njobs = n_jobs;
  lp.total_items = total;
  st = cuda_status(cudaGetLastError());
  if (st != NBLDPC_OK) return st;
  if (total > 0) {
    nbldpc::SplitBatchParams sp{};
    SplitShape shape;
    if (batch_split(jobs, n_jobs, total, pl, &sp, &shape)) {
      memcpy(sp.jobs, lp.jobs, sizeof(sp.jobs));   // (perm_at, reg: the one-block kernel's, set below)
      sp.njobs = n_jobs;
      sp.size = shape.size;
      return split_launch(split_kernel_for(0, 1, 0), total, shape.size, shape.threads, shape.smem, &sp,
                          reinterpret_cast<cudaStream_t>(cuda_stream));
    }
  }
  for (int i = 0; i < n_jobs; ++i) {
    const nbldpc_code* c = jobs[i].code;
    lp.jobs[i].perm_at = c->off.edge_col;          // it stages no edge_col or variable-node view
    // a lane per check takes long with few checks: only when they fill half the slot's lanes or other
    // frames fill the SM (100 frames of GF(32) N=64 and 200 of GF(4) N=100: 312 us against 109)
    const int nthr = pl.threads / pl.fpb;
    const bool fills = 2 * c->m >= nthr || total > pl.grid_max * pl.fpb;
    const bool reg = pl.mixed_reg && mixed_reg(c->q, nthr, c->dmax) && fills && batch_reg(jobs[i]);
    lp.jobs[i].reg = reg || (c->q == 64 && c->dreg == 4) ? nthr : 0;
  }
  const bool wide = batch_wide(jobs, n_jobs, total, pl);
  const int grid = std::min(grid_for(pl, total), wide ? 2 * (pl.grid_max / pl.per_sm) : pl.grid_max);
  return launch_plan(kernel_for(0, wide ? -2 : -1, 1), pl, lp, grid, workspace_dev,
                     reinterpret_cast<uint8_t*>(workspace_dev) + 256, reinterpret_cast<cudaStream_t>(cuda_stream));
}

// ---- autotuner ----------------------------------------------------------------
constexpr int kTuneReps = 3;         // timed decodes per candidate (the fastest counts)
static size_t tune_outputs(const nbldpc_code* c, int frames) {
  return round_up((size_t)frames * c->n, 256) + round_up((size_t)frames * 4, 256) + round_up((size_t)frames, 256);
}

int nbldpc_code_autotune_workspace_size(const nbldpc_code* c, int frames, size_t* bytes) {
  if (!c || !bytes || frames < 1) return NBLDPC_ERR_ARG;
  size_t mx = 0;
  for (int v = 0; v < 8; ++v)
    for (int fpb = 1; fpb <= 8; fpb *= 2) {
      Plan pl{};
      const CodeNeeds need = needs_of(c, v, c->mb);
      if (make_plan(c->q, v, kmode(c), fpb, &need, 1, &pl) != NBLDPC_OK) continue;
      const size_t w = ws_bytes(pl, frames);
      if (w > mx) mx = w;
    }
  *bytes = tune_outputs(c, frames) + mx;
  return NBLDPC_OK;
}

int nbldpc_code_autotune(nbldpc_code* c, const uint8_t* gamma_dev, int frames, int max_iters, void* workspace_dev,
                         size_t workspace_bytes, void* cuda_stream, nbldpc_tune_result* results, int max_results,
                         int* n_results) {
  if (!c || !gamma_dev || frames < 1 || max_iters < 1 || !workspace_dev || !aligned(gamma_dev, 16) ||
      !aligned(workspace_dev, 256))
    return NBLDPC_ERR_ARG;
  int st = check_device(c);
  if (st != NBLDPC_OK) return st;
  size_t need = 0;
  st = nbldpc_code_autotune_workspace_size(c, frames, &need);
  if (st != NBLDPC_OK) return st;
  if (workspace_bytes < need) return NBLDPC_ERR_ARG;
  cudaStream_t s = reinterpret_cast<cudaStream_t>(cuda_stream);
  unsigned char* w = reinterpret_cast<unsigned char*>(workspace_dev);
  uint8_t* sym = w;
  int32_t* its = reinterpret_cast<int32_t*>(w + round_up((size_t)frames * c->n, 256));
  uint8_t* okb = w + round_up((size_t)frames * c->n, 256) + round_up((size_t)frames * 4, 256);
  void* dws = w + tune_outputs(c, frames);
  cudaEvent_t e0 = nullptr, e1 = nullptr;
  if (cudaEventCreate(&e0) != cudaSuccess || cudaEventCreate(&e1) != cudaSuccess) return NBLDPC_ERR_CUDA;
  const int v_old = c->variant, f_old = c->plan.fpb;
  int best_v = v_old, best_f = f_old, count = 0;
  float best = 3.4e38f;
  st = NBLDPC_OK;
  for (int v = 0; v < 8 && st == NBLDPC_OK; ++v)
    for (int fpb = 1; fpb <= 8 && st == NBLDPC_OK; fpb *= 2) {
      if (configure(c, v, fpb) != NBLDPC_OK) continue;
      // one untimed decode, then the fastest of kTuneReps timed decodes with fixed iterations
      // (pairs within 1-2 % of each other would otherwise swap places from run to run)
      st = launch(c, gamma_dev, frames, max_iters, 0, sym, its, okb, dws, s, false, false);
      if (st != NBLDPC_OK) break;
      float ms = 3.4e38f;
      for (int rep = 0; rep < kTuneReps && st == NBLDPC_OK; ++rep) {
        float t = 0.f;
        if (cudaEventRecord(e0, s) != cudaSuccess) { st = NBLDPC_ERR_CUDA; break; }
        st = launch(c, gamma_dev, frames, max_iters, 0, sym, its, okb, dws, s, false, false);
        if (st != NBLDPC_OK) break;
        if (cudaEventRecord(e1, s) != cudaSuccess || cudaEventSynchronize(e1) != cudaSuccess ||
            cudaEventElapsedTime(&t, e0, e1) != cudaSuccess) {
          st = NBLDPC_ERR_CUDA;
          break;
        }
        if (t < ms) ms = t;
      }
      if (st != NBLDPC_OK) break;
      if (results && count < max_results) results[count] = nbldpc_tune_result{v, fpb, ms};
      ++count;
      if (ms < best) { best = ms; best_v = v; best_f = fpb; }
    }
  cudaEventDestroy(e0);
  cudaEventDestroy(e1);
  const int st2 = st == NBLDPC_OK ? configure(c, best_v, best_f)
                                  : c->tuned ? configure(c, v_old, f_old) : configure_default(c);
  if (st == NBLDPC_OK && st2 == NBLDPC_OK) c->tuned = true;
  if (n_results) *n_results = count;
  return st != NBLDPC_OK ? st : st2;
}

int nbldpc_decode_host_workspace_size(const nbldpc_code* c, int chunk_frames, size_t* bytes) {
  if (!c || !bytes || chunk_frames <= 0) return NBLDPC_ERR_ARG;
  *bytes = 2 * host_chunk_bytes(c, chunk_frames, (size_t)c->n * c->q, decode_ws_bytes(c, chunk_frames));
  return NBLDPC_OK;
}

int nbldpc_decode_host(const nbldpc_code* cc, const uint8_t* gamma_host, int frames, int max_iters, int early_stop,
                       uint8_t* out_sym_host, int32_t* out_iters_host, uint8_t* out_ok_host, int chunk_frames,
                       void* workspace_dev, size_t workspace_bytes, void* cuda_stream) {
  nbldpc_code* c = const_cast<nbldpc_code*>(cc);
  if (!c || frames < 0 || max_iters < 0 || chunk_frames <= 0) return NBLDPC_ERR_ARG;
  if (frames == 0) return NBLDPC_OK;
  const int st = check_device(c);
  if (st != NBLDPC_OK) return st;
  const size_t per = host_chunk_bytes(c, chunk_frames, (size_t)c->n * c->q, decode_ws_bytes(c, chunk_frames));
  return host_chunks(c, gamma_host, (size_t)c->n * c->q, frames, out_sym_host, out_iters_host, out_ok_host,
                     chunk_frames, workspace_dev, workspace_bytes, per, cuda_stream,
                     [&](const void* in, int nf, uint8_t* sy, int32_t* it, uint8_t* okb, void* ws, cudaStream_t s) {
                       return launch(c, reinterpret_cast<const uint8_t*>(in), nf, max_iters, early_stop, sy, it, okb,
                                     ws, s);
                     });
}

}  // extern "C"

// C ABI of the GB300 NB-LDPC decoders, FFT-SPA side (Alg. 1; declarations and
// contracts in include/nbldpc.h): the launch shape of a code (check-node form,
// degree buckets, block size, shared memory, message slot), stream-ordered
// launches of the FFT-SPA kernels, device- and host-buffer entry points.
#include "nbldpc.h"

#include <algorithm>

#include "fftspa_kernels.cuh"
#include "host_internal.h"

static_assert(sizeof(nbldpc::FftParams) < 4000, "kernel parameter space");

using namespace nbldpc_host;

namespace nbldpc {   // defined in fftspa.cu, one translation unit per field order
const void* fft_kernel_q2(int dc, int dv, int form, int* threads);
const void* fft_kernel_q4(int dc, int dv, int form, int* threads);
const void* fft_kernel_q8(int dc, int dv, int form, int* threads);
const void* fft_kernel_q16(int dc, int dv, int form, int* threads);
const void* fft_kernel_q32(int dc, int dv, int form, int* threads);
const void* fft_kernel_q64(int dc, int dv, int form, int* threads);
const void* fft_kernel_q128(int dc, int dv, int form, int* threads);
const void* fft_kernel_q256(int dc, int dv, int form, int* threads);
}  // namespace nbldpc

namespace {

// Shared memory left to the L1 cache when the message rows do not all fit.  Measured on
// GB300 (8, 16, 24, 48 KB, us): GF(64) N=576, 4096 frames of 10 iterations 7247, 7288,
// 7317, 7404; GF(256) (2,8) N=128, 1000 frames 1735, 1765, 1816, 1921.
constexpr int kFftL1 = 8192;

const void* fft_kernel_for(int q, int dc, int dv, int form, int* threads = nullptr) {
  switch (q) {
    case 2: return nbldpc::fft_kernel_q2(dc, dv, form, threads);
    case 4: return nbldpc::fft_kernel_q4(dc, dv, form, threads);
    case 8: return nbldpc::fft_kernel_q8(dc, dv, form, threads);
    case 16: return nbldpc::fft_kernel_q16(dc, dv, form, threads);
    case 32: return nbldpc::fft_kernel_q32(dc, dv, form, threads);
    case 64: return nbldpc::fft_kernel_q64(dc, dv, form, threads);
    case 128: return nbldpc::fft_kernel_q128(dc, dv, form, threads);
    case 256: return nbldpc::fft_kernel_q256(dc, dv, form, threads);
  }
  return nullptr;
}

// Largest field order whose codes take the lane-per-edge check-node form at
// every check degree (compile-time tuning knob).  Measured on GB300 (Mbit/s,
// lane per edge against distributed with 4 elements per lane): GF(4) (2,4)
// N=48 1336 vs 1117, GF(8) (2,4) N=512 1441 vs 1467, GF(16) (2,4) N=1024
// 1432 vs 1759, GF(32) (3,6) N=600 408 vs 588.
#ifndef NBLDPC_FFT_LANE_MAXQ
#define NBLDPC_FFT_LANE_MAXQ 4
#endif

// device, log2(q) - 1, check-node form, column-degree bucket: the kernels' attributes are
// set; the largest cluster of the split-frame kernel (0: not asked, -1: none)
bool g_fft_attr_done[64][8][3][3][2] = {};
int g_fft_split_max[64][8][3][3] = {};

}  // namespace

// Launch shape of the FFT-SPA kernel for a code: check-node form and degree
// buckets, block size (one frame per SM), shared memory (code blob, decisions,
// control word, and for the lane-per-edge form one transformed vector per
// lane, then message rows), resident blocks, message slot of nnz * q floats.
int nbldpc_host::fft_configure(nbldpc_code* c, const int32_t* row_ptr) {
  // check-node form: lane per edge (dc 0: check degree <= 32) for small fields
  // and for q <= 64 codes with a check of degree > 8; otherwise the
  // distributed form with the check degree bucket 4 or 8
  const bool lane_form = c->q <= NBLDPC_FFT_LANE_MAXQ || (c->q <= 64 && c->dmax > 8);
  const int dc = lane_form ? (c->dmax <= 32 ? 0 : -1) : (c->dmax <= 4 ? 4 : (c->dmax <= 8 ? 8 : -1));
  const int dv = c->vmax <= 2 ? 2 : (c->vmax <= 4 ? 4 : (c->vmax <= 8 ? 8 : 0));
  if (dc < 0 || !dv) return NBLDPC_ERR_UNSUPPORTED;
  int threads = 0;
  if (!fft_kernel_for(c->q, dc, dv, 0, &threads)) return NBLDPC_ERR_UNSUPPORTED;
  int dev = 0, sms = 0, optin = 0;
  if (cudaGetDevice(&dev) != cudaSuccess ||
      cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess ||
      cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev) != cudaSuccess)
    return NBLDPC_ERR_CUDA;
  if (dev < 0 || dev >= 64) return NBLDPC_ERR_CUDA;
  Plan pl{};
  pl.fpb = 1;
  pl.threads = threads;
  pl.blob_cap = (int)round_up((size_t)c->off.fft_bytes, 16);
  pl.n_cap = (int)round_up((size_t)c->n, 16);
  const int w_area = dc == 0 ? threads * c->q * (int)sizeof(float) : 0;   // one transformed vector per lane
  pl.slot_smem = pl.smem = (int)round_up((size_t)(pl.blob_cap + pl.n_cap + 16), 256) + w_area;
  if (pl.smem > optin) return NBLDPC_ERR_UNSUPPORTED;
  // the rest of the shared memory holds message rows: all of them, or those of the first
  // checks, whole warps of them
  const int row_bytes = c->q * (int)sizeof(float);
  const long long room = optin - pl.smem;
  int rows = c->nnz;
  if ((long long)rows * row_bytes > room) {
    const long long most = std::max(0LL, (room - kFftL1) / row_bytes);
    const int step = dc == 0 ? 1 : 32 / (c->q == 256 ? 32 : c->q / 4);   // checks of a warp
    int r = 0;
    while (r + step <= c->m && row_ptr[r + step] <= most) r += step;
    rows = row_ptr[r];
  }
  pl.xs_off = pl.smem;
  pl.smem += (int)round_up((size_t)rows * row_bytes, 16);
  c->fft_res_edges = rows;
  c->fft_form = rows == c->nnz ? 1 : 0;
  const void* k = fft_kernel_for(c->q, dc, dv, c->fft_form);
  {
    std::lock_guard<std::mutex> lk(g_attr_mu);
    const int iq = nbldpc::ilog2(c->q) - 1, ic = dc == 0 ? 0 : (dc == 4 ? 1 : 2), iv = dv == 2 ? 0 : (dv == 4 ? 1 : 2);
    bool& done = g_fft_attr_done[dev][iq][ic][iv][c->fft_form];
    int& split = g_fft_split_max[dev][iq][ic][iv];
    if (!done) {
      if (cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, optin) != cudaSuccess)
        return NBLDPC_ERR_CUDA;
      if (split == 0) split = split_kernel_prepare(fft_kernel_for(c->q, dc, dv, 2), threads, optin);
      if (split == 0) split = -1;
      done = true;
    }
    c->fft_split_max = split < 0 ? 0 : split;
    c->fft_split_threads = threads;
  }
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&pl.per_sm, k, pl.threads, pl.smem) != cudaSuccess)
    return NBLDPC_ERR_CUDA;
  if (pl.per_sm < 1) return NBLDPC_ERR_UNSUPPORTED;
  pl.grid_max = pl.per_sm * sms;
  pl.slot_bytes = round_up((size_t)c->nnz * c->q * sizeof(float), 256);
  c->fft_plan = pl;
  c->fft_dc = dc;
  c->fft_dv = dv;
  return NBLDPC_OK;
}

namespace {

// Shape of a split launch (see nbldpc.cu): ranks per frame, threads per rank, shared memory of a rank.
struct FftSplitShape {
  int size = 0, threads = 0, smem = 0;
  nbldpc::FftSplitParams p{};
};

// Lay out a rank's shared memory; size 0 when it does not fit the device.
FftSplitShape fft_split_layout(const nbldpc_code* c, int size, int threads) {
  FftSplitShape s;
  const bool lane_form = c->fft_dc == 0;
  s.p.size = size;
  s.p.cpc = ((lane_form ? c->ntasks : c->m) + size - 1) / size;
  s.p.npc = (c->n + size - 1) / size;
  // a warp task holds at most 32 edges
  const long long edges_r = std::min<long long>(c->nnz, (long long)s.p.cpc * (lane_form ? 32 : c->dmax));
  const long long edges_n = std::min<long long>(c->nnz, (long long)s.p.npc * c->vmax);
  size_t o = round_up((size_t)c->off.fft_bytes, 16);
  auto take = [&](size_t bytes) { const size_t at = o; o = round_up(o + bytes, 256); return (int)at; };
  s.p.chat_off = take((size_t)c->n);
  s.p.flag_off = take(2 * nbldpc::kMaxSplit * sizeof(int));
  s.p.row_off = take((size_t)edges_n * sizeof(void*));
  s.p.w_off = take(lane_form ? (size_t)threads * c->q * sizeof(float) : 0);
  s.p.x_off = take((size_t)edges_r * c->q * sizeof(float));
  if (o > (size_t)c->smem_optin) return FftSplitShape{};
  s.size = size;
  s.threads = threads;
  s.smem = (int)o;
  return s;
}

// The split shape of a batch, or size 0 for the one-block-per-frame kernel.
//
// The one-block kernel gives a frame one SM.  A cluster shortens a frame's
// passes, but the variable-node pass then reads the other ranks' rows: at
// throughput it is slower (GF(64) N=576, 4096 frames: 5.5 ms against 8.2 ms at
// best), so it serves batches that leave SMs idle.  Measured on GB300, us per
// decode of up to 20 iterations with early stop, one block against this rule:
// GF(64) N=576, 1 / 48 / 200 frames 284 / 336 / 579 against 72 / 175 / 501; GF(16)
// N=1024, 1 / 96 / 200 frames 283 / 285 / 343 against 97 / 182 / 293; GF(256) N=384,
// 1 / 96 / 200 frames 1851 / 1851 / 2190 against 257 / 832 / 1668.
//  - The fewer check-node lanes a frame has, the fewer frames: from 2000 on, one and
//    a half frames per SM; from 1024 on, 3/8 (GF(256) (2,8) N=128, 48 frames:
//    499 against 301; 96 frames 519 against 550); from 400 on, and in the lane-per-edge form, 1/8
//    (GF(4) N=1024, one frame: 113 against 75; 96 frames 130 against 161), none below
//    (GF(16) N=100, one frame: 72 against 80).  A lane of the lane-per-edge form has q products
//    and sums a pass: from 1024 lanes on at q <= 4 (GF(4) N=48, N=200, N=500, one frame:
//    39, 44 and 69 against 60, 62 and 66; GF(2) N=200 (3,6) 51 against 72), from 512 on at
//    GF(8) and GF(16) ((2,12) N=120, 320 lanes: 75 and 98 against 93 and 103; GF(16) N=240, 640
//    lanes: 165 against 107), any number for wider fields (GF(32) (2,12) N=120: 188 against 126).
//  - Equal iterations for every frame have no tail to shorten, so a second wave of
//    clusters costs its whole time: 16 ranks up to a tenth of a frame per SM, 8 up to a
//    quarter, 4 up to 3/8 (one block, these, and 16 / 8 / 8 ranks, 5 iterations: GF(128)
//    N=128, 19 / 42 / 57 frames 69, 47, 71 / 70, 66, 87 / 70, 70, 91; GF(64) N=256 70, 47,
//    71 / 71, 63, 87 / 71, 66, 91; GF(256) (2,8) N=128 133, 77, 116 / 133, 105, 145 / 135,
//    115, 155; below 2000 lanes at q = 128 none past a quarter: N=96 55, 60, 78), none above
//    (96 frames of GF(64) N=576: 164 against 229), and for q <= 32 between one frame per SM
//    and four thirds, which the one-block kernel takes in two waves (200 frames of GF(32)
//    N=600, 5 iterations: 276 against 260).
FftSplitShape fft_split_shape(const nbldpc_code* c, int frames, int early_stop) {
  if (c->fft_split_max == 0) return FftSplitShape{};
  const bool lane_form = c->fft_dc == 0;
  const int sms = c->fft_plan.grid_max / c->fft_plan.per_sm;
  const int lanes = lane_form ? 32 * c->ntasks : c->m * (c->q == 256 ? 32 : c->q / 4);
  if (lanes < (!lane_form ? 400 : c->q <= 4 ? 1024 : c->q <= 16 ? 512 : 0)) return FftSplitShape{};
  const int few = lane_form || lanes < 1024 ? sms / 8 : 3 * sms / 8;
  const bool more = !lane_form && lanes >= 2000 && (early_stop ? frames <= 3 * sms / 2
                                                 : c->q <= 32 && frames > sms && frames <= 4 * sms / 3);
  if (frames > few && !more) return FftSplitShape{};
  int size = frames <= sms / 8 ? 16 : frames <= 3 * sms / 4 ? 8 : 4;
  int threads = c->q == 64 || c->q == 128 ? c->fft_split_threads / 2 : 256;
  if (!early_stop && frames <= 3 * sms / 8) {
    size = frames <= sms / 10 ? 16 : frames <= sms / 4 ? 8 : 4;
    if (size == 4) threads = 256;
    if (size == 4 && c->q == 128 && lanes < 2000) return FftSplitShape{};
  }
  if (lane_form || lanes < 1024) {
    size = 8;
    threads = lane_form ? 256 : 128;
  }
  if (lane_form)
    while (size > c->ntasks) size /= 2;
  size = std::min(size, c->fft_split_max);
  if (size < 2) return FftSplitShape{};
  FftSplitShape s = fft_split_layout(c, size, threads);
  while (s.size == 0 && threads > 64) s = fft_split_layout(c, size, threads = (threads - 1) / 64 * 64);
  return s;
}

int fft_launch(const nbldpc_code* c, const float* prob, int frames, int max_iters, int early_stop, uint8_t* sym,
               int32_t* iters, uint8_t* ok, float* app, void* ws, cudaStream_t st) {
  const Plan& pl = c->fft_plan;
  nbldpc::FftParams fp{};
  fp.job.ntasks = c->ntasks;
  fp.job.blob = c->blob_dev;
  fp.job.off = c->off;
  fp.job.prob = prob;
  fp.job.out_sym = sym;
  fp.job.out_iters = iters;
  fp.job.out_ok = ok;
  fp.job.out_app = app;
  fp.job.q = c->q;
  fp.job.n = c->n;
  fp.job.m = c->m;
  fp.job.frames = frames;
  fp.job.max_iters = max_iters;
  fp.job.early_stop = early_stop ? 1 : 0;
  FftSplitShape sp = fft_split_shape(c, frames, early_stop);
  if (sp.size) {
    sp.p.job = fp.job;
    return split_launch(fft_kernel_for(c->q, c->fft_dc, c->fft_dv, 2), frames, sp.size, sp.threads, sp.smem, &sp.p, st);
  }
  fp.counter = reinterpret_cast<unsigned int*>(ws);
  fp.msg = reinterpret_cast<float*>(reinterpret_cast<uint8_t*>(ws) + 256);
  fp.slot_floats = pl.slot_bytes / sizeof(float);
  fp.blob_cap = pl.blob_cap;
  fp.n_cap = pl.n_cap;
  fp.w_off = (int)round_up((size_t)(pl.blob_cap + pl.n_cap + 16), 256);
  fp.x_off = pl.xs_off;
  fp.res_edges = c->fft_res_edges;
  cudaError_t e = cudaMemsetAsync(ws, 0, sizeof(unsigned int), st);
  if (e != cudaSuccess) return NBLDPC_ERR_CUDA;
  void* args[] = {&fp};
  e = cudaLaunchKernel(fft_kernel_for(c->q, c->fft_dc, c->fft_dv, c->fft_form), dim3(grid_for(pl, frames)), dim3(pl.threads),
                       args, (size_t)pl.smem, st);
  if (e != cudaSuccess) return NBLDPC_ERR_CUDA;
  g_launches.fetch_add(1, std::memory_order_relaxed);
  return NBLDPC_OK;
}

}  // namespace

extern "C" {

// ---- FFT-SPA decoding ----------------------------------------------------------
int nbldpc_fftspa_workspace_size(const nbldpc_code* c, int frames, size_t* bytes) {
  if (!c || frames < 0 || !bytes) return NBLDPC_ERR_ARG;
  if (c->fft_status != NBLDPC_OK) return c->fft_status;
  *bytes = ws_bytes(c->fft_plan, frames);
  return NBLDPC_OK;
}

int nbldpc_fftspa_cluster_blocks(const nbldpc_code* c, int frames, int early_stop, int* blocks) {
  if (!c || !blocks || frames < 0) return NBLDPC_ERR_ARG;
  if (c->fft_status != NBLDPC_OK) return c->fft_status;
  *blocks = frames ? fft_split_shape(c, frames, early_stop).size : 0;
  return NBLDPC_OK;
}

int nbldpc_fftspa_decode(const nbldpc_code* c, const float* prob_dev, int frames, int max_iters, int early_stop,
                         uint8_t* out_sym_dev, int32_t* out_iters_dev, uint8_t* out_ok_dev, float* out_app_dev,
                         void* workspace_dev, size_t workspace_bytes, void* cuda_stream) {
  if (!c || frames < 0 || max_iters < 0) return NBLDPC_ERR_ARG;
  if (c->fft_status != NBLDPC_OK) return c->fft_status;
  if (frames == 0) return NBLDPC_OK;
  if (!prob_dev || !out_sym_dev || !out_iters_dev || !out_ok_dev || !workspace_dev) return NBLDPC_ERR_ARG;
  if (!aligned(prob_dev, 16) || !aligned(out_iters_dev, 4) || !aligned(workspace_dev, 16)) return NBLDPC_ERR_ARG;
  if (out_app_dev && !aligned(out_app_dev, 16)) return NBLDPC_ERR_ARG;
  if (workspace_bytes < ws_bytes(c->fft_plan, frames)) return NBLDPC_ERR_ARG;
  int st = check_device(c);
  if (st != NBLDPC_OK) return st;
  st = cuda_status(cudaGetLastError());
  if (st != NBLDPC_OK) return st;
  return fft_launch(c, prob_dev, frames, max_iters, early_stop, out_sym_dev, out_iters_dev, out_ok_dev, out_app_dev,
                    workspace_dev, reinterpret_cast<cudaStream_t>(cuda_stream));
}

int nbldpc_fftspa_decode_host_workspace_size(const nbldpc_code* c, int chunk_frames, size_t* bytes) {
  if (!c || !bytes || chunk_frames <= 0) return NBLDPC_ERR_ARG;
  if (c->fft_status != NBLDPC_OK) return c->fft_status;
  *bytes = 2 * host_chunk_bytes(c, chunk_frames, (size_t)c->n * c->q * sizeof(float),
                                ws_bytes(c->fft_plan, chunk_frames));
  return NBLDPC_OK;
}

int nbldpc_fftspa_decode_host(const nbldpc_code* cc, const float* prob_host, int frames, int max_iters,
                              int early_stop, uint8_t* out_sym_host, int32_t* out_iters_host, uint8_t* out_ok_host,
                              int chunk_frames, void* workspace_dev, size_t workspace_bytes, void* cuda_stream) {
  nbldpc_code* c = const_cast<nbldpc_code*>(cc);
  if (!c || frames < 0 || max_iters < 0 || chunk_frames <= 0) return NBLDPC_ERR_ARG;
  if (c->fft_status != NBLDPC_OK) return c->fft_status;
  if (frames == 0) return NBLDPC_OK;
  const int st = check_device(c);
  if (st != NBLDPC_OK) return st;
  const size_t fbytes = (size_t)c->n * c->q * sizeof(float);
  const size_t per = host_chunk_bytes(c, chunk_frames, fbytes, ws_bytes(c->fft_plan, chunk_frames));
  return host_chunks(c, prob_host, fbytes, frames, out_sym_host, out_iters_host, out_ok_host, chunk_frames,
                     workspace_dev, workspace_bytes, per, cuda_stream,
                     [&](const void* in, int nf, uint8_t* sy, int32_t* it, uint8_t* okb, void* ws, cudaStream_t s) {
                       return fft_launch(c, reinterpret_cast<const float*>(in), nf, max_iters, early_stop, sy, it, okb,
                                         nullptr, ws, s);
                     });
}

}  // extern "C"

// Min-max (MMA) decoding of non-binary LDPC codes over GF(2^p): device code
// for sm_103a.  One persistent block decodes one frame at a time, running the
// flooding schedule of Alg. 2 (check-node F/B/beta pass, variable-node pass,
// decision and syndrome) until the syndrome is zero or I_max is reached, then
// takes the next frame from a global counter.
//
// Message vectors (q reliabilities in 0..255) travel between the passes as q
// bytes per Tanner-graph edge in a per-block global slot that stays resident
// in L1/L2.  Inside the check-node pass a vector lives in shared memory as q
// 16-bit values, so that the min-max convolution (see mm_conv) runs on packed
// max.u16x2 / min.u16x2 instructions, two symbols per instruction; the
// variable-node pass also works on 16-bit pairs held in 32-bit registers.
//
// Min-max convolution (Alg. 2, F/B/beta equations, with the coefficient
// permutation applied to the inputs):
//     C(x) = min over y of max(A(y), B(x ^ y)),   x, y in GF(2^p).
#pragma once

#include <cstdint>
#include <type_traits>

#include <cuda_runtime.h>

namespace nbldpc {

// ---------------------------------------------------------------- primitives
__device__ __forceinline__ uint32_t vmax2(uint32_t a, uint32_t b) {
  uint32_t d;
  asm("max.u16x2 %0, %1, %2;" : "=r"(d) : "r"(a), "r"(b));
  return d;
}
__device__ __forceinline__ uint32_t vmin2(uint32_t a, uint32_t b) {
  uint32_t d;
  asm("min.u16x2 %0, %1, %2;" : "=r"(d) : "r"(a), "r"(b));
  return d;
}

// max of two packed pairs on the FMA pipe instead of the ALU pipe:
// max(a, b) = b + relu(a - b).  The operands are 16-bit integers 0..255; read
// as fp16 they are subnormal numbers (k * 2^-24), whose differences and sums
// below 2^11 are exact in fp16, so the result is the integer maximum bit for
// bit.  Used for part of the maxima so the two pipes share the work.
__device__ __forceinline__ uint32_t vmax2_fma(uint32_t a, uint32_t b) {
  uint32_t t, d;
  const uint32_t neg1 = 0xBC00BC00u;   // (-1.0, -1.0) in f16x2
  asm("fma.rn.relu.f16x2 %0, %1, %2, %3;" : "=r"(t) : "r"(b), "r"(neg1), "r"(a));
  asm("add.rn.f16x2 %0, %1, %2;" : "=r"(d) : "r"(t), "r"(b));
  return d;
}

// ---------------------------------------------------------------- geometry
// Bytes of one variable node's q-byte rows that each lane of the variable-node
// pass handles (q / VBPL lanes per node).  Wide lanes put several nodes in
// flight per warp and shorten the shuffle reductions; measured on GB300 the
// 4-byte lanes of GF(64) left that pass latency-bound (8 bytes: +10 %, 16
// bytes: +3 % more).
#ifndef NBLDPC_VBPL_64
#define NBLDPC_VBPL_64 16
#endif
#ifndef NBLDPC_VBPL_256
#define NBLDPC_VBPL_256 16
#endif
template <int Q> struct VnpBytes {
  static constexpr int v = Q == 2 ? 2 : Q == 4 ? 4 : Q == 8 ? 8 : Q == 64 ? NBLDPC_VBPL_64
                         : Q == 256 ? NBLDPC_VBPL_256 : Q >= 16 && Q <= 32 ? 16 : 8;
};

// LB: lane bits of x (the shuffle offset d runs over them); SB: lane bits that
// split the register part of y between lanes.  XB = p - LB register bits of x
// per lane, TB = XB - SB register bits of y per lane.  Each field order has
// two layouts (variant 0 and 1: two ways of splitting the q x q work between
// the lanes of a group and their registers); the autotuner picks one per code.
template <int Q, int V> struct Layout;
template <> struct Layout<2, 0>   { static constexpr int LB = 1, SB = 0; };
template <> struct Layout<2, 1>   { static constexpr int LB = 1, SB = 0; };
template <> struct Layout<4, 0>   { static constexpr int LB = 1, SB = 0; };
template <> struct Layout<4, 1>   { static constexpr int LB = 2, SB = 0; };
template <> struct Layout<8, 0>   { static constexpr int LB = 1, SB = 1; };
template <> struct Layout<8, 1>   { static constexpr int LB = 2, SB = 0; };
template <> struct Layout<16, 0>  { static constexpr int LB = 2, SB = 1; };
template <> struct Layout<16, 1>  { static constexpr int LB = 3, SB = 0; };
template <> struct Layout<32, 0>  { static constexpr int LB = 2, SB = 2; };
template <> struct Layout<32, 1>  { static constexpr int LB = 3, SB = 1; };
template <> struct Layout<64, 0>  { static constexpr int LB = 3, SB = 2; };
template <> struct Layout<64, 1>  { static constexpr int LB = 3, SB = 1; };
template <> struct Layout<128, 0> { static constexpr int LB = 4, SB = 1; };
template <> struct Layout<128, 1> { static constexpr int LB = 5, SB = 0; };
template <> struct Layout<256, 0> { static constexpr int LB = 5, SB = 0; };
template <> struct Layout<256, 1> { static constexpr int LB = 4, SB = 1; };

constexpr int ilog2(int v) { return v <= 1 ? 0 : 1 + ilog2(v >> 1); }

// bytes of one 16-bit message vector in shared memory (NBLDPC_VPAD: padding
// that shifts consecutive vectors to other banks)
#ifndef NBLDPC_VPAD
#define NBLDPC_VPAD 0
#endif
template <int Q> __host__ __device__ constexpr int vec_bytes() { return (2 * Q + 15) / 16 * 16 + NBLDPC_VPAD; }

template <int Q_, int V_> struct Geo {
  static constexpr int Q = Q_, V = V_;
  static constexpr int P = ilog2(Q);
  static constexpr int LB = Layout<Q, V>::LB, SB = Layout<Q, V>::SB;
  static constexpr int XB = P - LB;             // register bits of x
  static constexpr int TB = XB - SB;            // register bits of y
  static constexpr int G = 1 << (LB + SB);      // lanes per convolution group
  static constexpr int DN = 1 << LB;            // x values per register slot (lane part)
  static constexpr int DS = DN / 2;             // shuffle steps (even offsets d = 2*ds)
  static constexpr int XN = 1 << XB;            // accumulators per lane
  static constexpr int AWN = 1 << TB;           // packed A words per lane
  static constexpr int DC = (DS * XN <= 32) ? DS : (32 / XN >= 1 ? 32 / XN : 1);  // steps per B chunk
  static constexpr int OPL = 1 << TB;           // outputs per lane
  static constexpr int W = Q / 2;               // 32-bit words per vector
  static constexpr int PW = (W + G - 1) / G;    // permutation words per lane
  static constexpr int BPL = Q / G;             // bytes per lane when a group writes q bytes
  static constexpr int VB = vec_bytes<Q>();     // bytes per 16-bit vector in smem
  // variable-node pass: VG lanes per variable node, VBPL bytes (VBPL/2 packed words) each
  static constexpr int VBPL = VnpBytes<Q>::v;
  static constexpr int VG = Q / VBPL;
  static constexpr int VW = VBPL / 2;
  static_assert(LB >= 1 && TB >= 0 && XB == SB + TB, "layout");
  static_assert(G <= 32 && G * OPL == Q, "group covers the field");
  static_assert(DS % DC == 0, "chunking");
  static_assert(BPL == 1 || BPL == 2 || BPL == 4 || BPL == 8, "byte lanes");
};

// Of the XN * AWN maxima of one shuffle step, FmaEighths eighths use
// vmax2_fma (the rest the ALU pipe, which also takes every minimum).  Measured
// on GB300: 3/8 is best for q <= 64 (GF(64) step: 5/16 435.6, 6/16 437.5,
// 7/16 434.9, 8/16 430.4 Mbit/s; again with the current frame decoder: 2/8
// and 4/8 2-3 % slower than 3/8); 3/8 for q >= 128 too since the
// convolution's chunk loop is rolled (GF(256) (2,6) N=384, layout 0: 0 to
// 5/8 at 162.2, 150.2, 145.0, 142.5, 148.7, 167.5 ms; before the loop was
// rolled 1/8 was best).
#ifndef NBLDPC_FMA_EIGHTHS
#define NBLDPC_FMA_EIGHTHS 3
#endif
#ifndef NBLDPC_FMA_EIGHTHS_WIDE
#define NBLDPC_FMA_EIGHTHS_WIDE 3
#endif
template <int Q> struct FmaEighths {
  static constexpr int v = Q >= 128 ? NBLDPC_FMA_EIGHTHS_WIDE : NBLDPC_FMA_EIGHTHS;
};
template <class g> struct FmaMax { static constexpr int v = (g::XN * g::AWN * FmaEighths<g::Q>::v) / 8; };

// Lane constants of the convolution, computed once per thread.
struct ConvLane {
  int a_off;      // word index of the lane's first packed A word
  uint32_t sel;   // byte_perm selector: identity, or swap of the 16-bit halves on odd lanes
  int c_off;      // 16-bit index of the lane's first output
};

template <class g> __device__ __forceinline__ ConvLane conv_lane(int s, int l) {
  ConvLane c;
  c.a_off = (((s << g::TB) * g::DN) + (l & ~1)) >> 1;
  c.sel = (l & 1) ? 0x1032u : 0x3210u;
  c.c_off = (s << g::TB) * g::DN + l;
  return c;
}

// ---------------------------------------------------------------- convolution
// C = A (*) B: C(x) = min_y max(A(y), B(x ^ y)); vectors are q 16-bit values
// in natural order (element v at 16-bit index v).  A group of G lanes; lane
// (s, l) owns x = xh * DN + l for the XN values of xh and the y values with
// register part yr in [s * 2^TB, (s + 1) * 2^TB).  A packed A word pairs the
// lane positions (l, l ^ 1), so offset d = 2*ds reaches lane positions l ^ d
// and l ^ d ^ 1 in one shuffle, and the matching B values B(j*DN + d),
// B(j*DN + d + 1) form one natural 32-bit word whatever the parity of x, read
// by all lanes from the same shared-memory address.  Accumulator slot r holds
// xh = r ^ (s << TB), which makes the B register index r ^ t independent of
// the lane and lets the final reduce-scatter keep and send fixed slots.
// Inputs and output must not alias; the caller syncs the group afterwards.
//
// When the shuffle steps span several chunks of B registers (q >= 128), the
// chunk loop is kept rolled (NBLDPC_CONV_ROLL): the fully unrolled q = 256
// convolution, inlined at each call site, no longer fits the instruction
// cache.  The rolled form starts the accumulators at the maximum and shuffles
// at offset 0 in the first step, so every step has the same code.
#ifndef NBLDPC_CONV_ROLL
#define NBLDPC_CONV_ROLL 1
#endif
template <class g> __device__ __forceinline__ void load_b_chunk(const uint32_t* __restrict__ B, int c0,
                                                                uint32_t (&bl)[g::DC][g::XN]) {
#pragma unroll
  for (int j = 0; j < g::XN; ++j) {
    const uint32_t* row = B + j * g::DS + c0;
    if constexpr (g::DC % 4 == 0) {
#pragma unroll
      for (int dd = 0; dd < g::DC; dd += 4) {
        const uint4 v = *reinterpret_cast<const uint4*>(row + dd);
        bl[dd][j] = v.x; bl[dd + 1][j] = v.y; bl[dd + 2][j] = v.z; bl[dd + 3][j] = v.w;
      }
    } else if constexpr (g::DC % 2 == 0) {
#pragma unroll
      for (int dd = 0; dd < g::DC; dd += 2) {
        const uint2 v = *reinterpret_cast<const uint2*>(row + dd);
        bl[dd][j] = v.x; bl[dd + 1][j] = v.y;
      }
    } else {
#pragma unroll
      for (int dd = 0; dd < g::DC; ++dd) bl[dd][j] = row[dd];
    }
  }
}

template <class g, bool FMA_MAX>
__device__ __forceinline__ void mm_conv(const uint32_t* __restrict__ A, const uint32_t* __restrict__ B,
                                        uint16_t* __restrict__ C, const ConvLane& ln, unsigned gmask) {
  uint32_t aown[g::AWN];
#pragma unroll
  for (int t = 0; t < g::AWN; ++t) aown[t] = __byte_perm(A[ln.a_off + t * g::DS], 0, ln.sel);
  uint32_t acc[g::XN];

  if constexpr (NBLDPC_CONV_ROLL && g::DS / g::DC > 1) {
#pragma unroll
    for (int r = 0; r < g::XN; ++r) acc[r] = 0xFFFFFFFFu;
#pragma unroll 1
    for (int c0 = 0; c0 < g::DS; c0 += g::DC) {
      uint32_t bl[g::DC][g::XN];
      load_b_chunk<g>(B, c0, bl);
#pragma unroll
      for (int dd = 0; dd < g::DC; ++dd) {
        const int d = 2 * (c0 + dd);
        uint32_t a[g::AWN];
#pragma unroll
        for (int t = 0; t < g::AWN; ++t) a[t] = __shfl_xor_sync(gmask, aown[t], d);
#pragma unroll
        for (int r = 0; r < g::XN; ++r)
#pragma unroll
          for (int t = 0; t < g::AWN; ++t) {
            const uint32_t m = (FMA_MAX && r * g::AWN + t < FmaMax<g>::v) ? vmax2_fma(a[t], bl[dd][r ^ t])
                                                                : vmax2(a[t], bl[dd][r ^ t]);
            acc[r] = vmin2(acc[r], m);
          }
      }
    }
  } else {
#pragma unroll
  for (int c0 = 0; c0 < g::DS; c0 += g::DC) {
    uint32_t bl[g::DC][g::XN];
    load_b_chunk<g>(B, c0, bl);
#pragma unroll
    for (int dd = 0; dd < g::DC; ++dd) {
      const int d = 2 * (c0 + dd);
      uint32_t a[g::AWN];
#pragma unroll
      for (int t = 0; t < g::AWN; ++t) a[t] = (d == 0) ? aown[t] : __shfl_xor_sync(gmask, aown[t], d);
#pragma unroll
      for (int r = 0; r < g::XN; ++r)
#pragma unroll
        for (int t = 0; t < g::AWN; ++t) {
          const uint32_t m = (FMA_MAX && r * g::AWN + t < FmaMax<g>::v) ? vmax2_fma(a[t], bl[dd][r ^ t])
                                                              : vmax2(a[t], bl[dd][r ^ t]);
          acc[r] = (d == 0 && t == 0) ? m : vmin2(acc[r], m);
        }
    }
  }
  }
  // reduce-scatter over the SB lane bits: keep slot r, receive the partner's r | 2^c
#pragma unroll
  for (int b = g::SB - 1; b >= 0; --b) {
    const int c = g::TB + b;
#pragma unroll
    for (int r = 0; r < (1 << c); ++r)
      acc[r] = vmin2(acc[r], __shfl_xor_sync(gmask, acc[r | (1 << c)], 1 << (g::LB + b)));
  }
#pragma unroll
  for (int r = 0; r < g::OPL; ++r) C[ln.c_off + r * g::DN] = (uint16_t)vmin2(acc[r], acc[r] >> 16);
}

// ---------------------------------------------------------------- pruned convolution
// The same C = A (*) B, visiting only the y that can decide a minimum.  For any
// bound T >= max_x C(x), a y with A(y) > T gives max(A(y), B(x ^ y)) > C(x) for
// every x, so C(x) = min over {y : A(y) <= T} of max(A(y), B(x ^ y)), and the
// same holds with the roles of A and B exchanged (C is symmetric in them).
// T is found in phases: the entries of the chosen side with value <= hi are
// folded in, M = max_x of the partial result is an upper bound of max_x C(x)
// (a partial minimum is never below the full one), and the phases stop as soon
// as M <= hi; otherwise hi moves towards M.  The result is C exactly, with no
// approximation; the work is the number of entries folded in, about
// 17 of 256 for the GF(256) decoder's vectors instead of 256.
//
// One group of 32 lanes (one warp, so every branch below is warp-uniform).
// Vectors are q bytes; lane L owns x = L * OPL + k (k < OPL), kept as OPL/2 packed
// pairs.  For y = L' * OPL + i, x ^ y = (L ^ L') * OPL + (k ^ i): one aligned vector
// load of block L ^ L' from copy i of the other side, whose blocks are permuted by
// k -> k ^ i (OPL copies, written once per convolution).  The entries of a phase are
// compacted into a list of records (value << 16 | byte offset of copy and block), so
// that folding two of them in is a list load, two block loads and the maxima and
// minima, with no search (a quarter of the maxima on the FMA pipe at q = 256).  Bound by
// the ALU pipe (70 % busy): about 120 instructions a phase and 13 an entry.  Measured on
// GB300 against finding an entry by ffs over a ballot and its value by shuffle, in eight
// loops a phase: GF(256) (2,6) N=384, 4096 frames 52.1 against 46.9 ms; GF(256) (2,8)
// N=128, 3000 frames 19.5 against 17.1 (the byte vectors also leave three blocks an SM);
// GF(128) (2,4) N=256, 8192 frames 38.0 against 36.0.
// tprev: prediction of max_x C(x) (the previous convolution's maximum); it
// picks the side with fewer entries below it and the first phase's bound.
// tmp: kPrTmp<q> bytes of scratch.
// Returns max_x C(x); with folded non-null, adds the number of entries folded in
// (each entry is q pairs (x, y)).  C may be A or B: both are read before C is written.
#ifndef NBLDPC_PRUNE_BACK
#define NBLDPC_PRUNE_BACK 1          // first phase: hi = tprev - NBLDPC_PRUNE_BACK (4: 47.7 ms, -1: 47.7)
#endif
#ifndef NBLDPC_PRUNE_PHASES
#define NBLDPC_PRUNE_PHASES 6        // after this many phases hi jumps to M
#endif
constexpr int kPrList = 64;          // records of the list (a longer phase is folded in parts)
template <int Q> constexpr int kPrTmp = (Q / 32) * 2 * Q + (kPrList + 2) * 4 + 8;

template <int NW> __device__ __forceinline__ void load_words(const unsigned char* p, uint32_t (&w)[NW]) {
  if constexpr (NW == 4) {
    const uint4 v = *reinterpret_cast<const uint4*>(p);
    w[0] = v.x; w[1] = v.y; w[2] = v.z; w[3] = v.w;
  } else if constexpr (NW == 2) {
    const uint2 v = *reinterpret_cast<const uint2*>(p);
    w[0] = v.x; w[1] = v.y;
  } else {
    w[0] = *reinterpret_cast<const uint32_t*>(p);
  }
}
template <int NW> __device__ __forceinline__ void store_words(unsigned char* p, const uint32_t (&w)[NW]) {
  if constexpr (NW == 4) *reinterpret_cast<uint4*>(p) = make_uint4(w[0], w[1], w[2], w[3]);
  else if constexpr (NW == 2) *reinterpret_cast<uint2*>(p) = make_uint2(w[0], w[1]);
  else *reinterpret_cast<uint32_t*>(p) = w[0];
}

template <class g>
__device__ __forceinline__ int pr_conv(const uint8_t* A, const uint8_t* B, uint8_t* C, unsigned char* tmp, int lane,
                                       int tprev, int* folded) {
  constexpr int OPL = g::Q / 32, NW = OPL / 2;
  constexpr int BB = 2 * OPL, CB = 2 * g::Q;         // bytes of a block and of a copy
  static_assert(g::G == 32 && OPL >= 2 && NW <= 4, "one warp per convolution");
  uint32_t* list = reinterpret_cast<uint32_t*>(tmp + OPL * CB);
  // the lane's bytes of both sides (OPL bytes in one or two words), and as 16-bit pairs
  uint32_t a8[2] = {0u, 0u}, b8[2] = {0u, 0u};
  if constexpr (OPL == 8) {
    const uint2 x = *reinterpret_cast<const uint2*>(A + lane * 8), y = *reinterpret_cast<const uint2*>(B + lane * 8);
    a8[0] = x.x; a8[1] = x.y; b8[0] = y.x; b8[1] = y.y;
  } else if constexpr (OPL == 4) {
    a8[0] = *reinterpret_cast<const uint32_t*>(A + lane * 4);
    b8[0] = *reinterpret_cast<const uint32_t*>(B + lane * 4);
  } else {
    a8[0] = *reinterpret_cast<const uint16_t*>(A + lane * 2);
    b8[0] = *reinterpret_cast<const uint16_t*>(B + lane * 2);
  }
  uint32_t a[NW], b[NW];
#pragma unroll
  for (int w = 0; w < NW; ++w) {
    a[w] = __byte_perm(a8[w >> 1], 0, (w & 1) ? 0x4342 : 0x4140);
    b[w] = __byte_perm(b8[w >> 1], 0, (w & 1) ? 0x4342 : 0x4140);
  }
  // side: fewer entries <= tprev.  Per 16-bit half, 0x8000 + t - v has bit 15
  // set exactly when v <= t (values and t below 2^15: no borrow between halves)
  const uint32_t kt = 0x80008000u + (uint32_t)tprev * 0x10001u;
  int ca = 0, cb = 0;
#pragma unroll
  for (int w = 0; w < NW; ++w) {
    ca += __popc((kt - a[w]) & 0x80008000u);
    cb += __popc((kt - b[w]) & 0x80008000u);
  }
  const unsigned cc = __reduce_add_sync(0xFFFFFFFFu, (unsigned)(ca | (cb << 16)));
  const bool swap = (cc >> 16) < (cc & 0xFFFFu);
  const uint32_t e0 = swap ? b8[0] : a8[0], e1 = swap ? b8[1] : a8[1];   // the entries' values
  uint32_t left[NW];                   // entries still to fold in (0x4000 added once listed)
#pragma unroll
  for (int w = 0; w < NW; ++w) {
    left[w] = swap ? b[w] : a[w];
    b[w] = swap ? a[w] : b[w];         // the other side
  }
  // copies of the other side
  const int lane_off = lane * BB;
#pragma unroll
  for (int i = 0; i < OPL; i += 2) {
    uint32_t t[NW];
#pragma unroll
    for (int w = 0; w < NW; ++w) t[w] = b[w ^ (i >> 1)];
    store_words<NW>(tmp + i * CB + lane_off, t);
#pragma unroll
    for (int w = 0; w < NW; ++w) t[w] = __byte_perm(t[w], 0, 0x1032);
    store_words<NW>(tmp + (i + 1) * CB + lane_off, t);
  }
  const unsigned lt = (1u << lane) - 1u;
  uint32_t acc[NW];
#pragma unroll
  for (int w = 0; w < NW; ++w) acc[w] = 0xFFFFFFFFu;
  int hi = max(tprev - NBLDPC_PRUNE_BACK, 0), M = 0, total = 0;
  for (int phase = 1;; ++phase) {
    // entries <= hi not yet listed: element 2 w at bit 12 + w, element 2 w + 1 at bit 28 + w
    const uint32_t kh = 0x80008000u + (uint32_t)min(hi, 0x3FFF) * 0x10001u;
    uint32_t mm = 0;
#pragma unroll
    for (int w = 0; w < NW; ++w) {
      const uint32_t m = (kh - left[w]) & 0x80008000u;
      left[w] |= m >> 1;
      mm |= m >> (3 - w);
    }
    int n = 0;                         // records in the list
    for (;;) {
      const unsigned bal = __ballot_sync(0xFFFFFFFFu, mm != 0);
      if (mm) {
        const int bit = 31 - __clz(mm);
        mm ^= 1u << bit;
        const int i = ((bit & 15) - 12) * 2 + (bit >> 4);
        const uint32_t v = __byte_perm(e0, e1, 0x8880 + i) & 0xFFu;
        list[n + __popc(bal & lt)] = (v << 16) | (uint32_t)(i * CB + lane_off);
      }
      n += __popc(bal);
      if (bal && n <= kPrList - 32) continue;
      total += n;
      __syncwarp();                    // (and, the first time, the copies are complete)
      if (n & 1) {                     // an odd list ends with its last record twice
        if (lane == 0) list[n] = list[n - 1];
        __syncwarp();
      }
      for (int k = 0; k < n; k += 2) {
        const uint2 r = *reinterpret_cast<const uint2*>(list + k);
        uint32_t v0[NW], v1[NW];
        load_words<NW>(tmp + ((r.x ^ (uint32_t)lane_off) & 0xFFFFu), v0);
        load_words<NW>(tmp + ((r.y ^ (uint32_t)lane_off) & 0xFFFFu), v1);
        const uint32_t u0 = __byte_perm(r.x, 0, 0x3232), u1 = __byte_perm(r.y, 0, 0x3232);
#pragma unroll
        for (int w = 0; w < NW; ++w)
          acc[w] = w < NW / 4 ? __vimin3_u16x2(acc[w], vmax2_fma(v0[w], u0), vmax2_fma(v1[w], u1))
                           : __vimin3_u16x2(acc[w], vmax2(v0[w], u0), vmax2(v1[w], u1));
      }
      if (!bal) break;
      n = 0;
      __syncwarp();
    }
    uint32_t mx = acc[0];
#pragma unroll
    for (int w = 1; w < NW; ++w) mx = vmax2(mx, acc[w]);
    M = (int)__reduce_max_sync(0xFFFFFFFFu, max(mx & 0xFFFFu, mx >> 16));
    if (M <= hi || hi >= 255) break;                        // (the second: every entry folded in)
    if (M == 0xFFFF) hi = 2 * hi + 8;                       // nothing folded in yet
    else if (phase >= NBLDPC_PRUNE_PHASES) hi = M;
    else hi = min(M, max(hi + 2, (hi + M + 1) >> 1));
  }
  if (folded) *folded += total;
  uint32_t c8[2] = {0u, 0u};
#pragma unroll
  for (int w = 0; w < NW; w += 2) c8[w >> 1] = __byte_perm(acc[w], NW > 1 ? acc[w | 1] : 0u, 0x6420);
  if constexpr (OPL == 8) *reinterpret_cast<uint2*>(C + lane * 8) = make_uint2(c8[0], c8[1]);
  else if constexpr (OPL == 4) *reinterpret_cast<uint32_t*>(C + lane * 4) = c8[0];
  else *reinterpret_cast<uint16_t*>(C + lane * 2) = (uint16_t)c8[0];
  return M;
}

// ---------------------------------------------------------------- parameters
struct CodeBlob {           // offsets (bytes) into the code blob
  int exp2, log, row_ptr, edge_lh, edge_lhi, edge_col, vn_ptr, vn_edge;   // (in this order)
  // q = 8, 16, 32: byte selectors of every multiplication (PermRow), bytes - perm of them;
  // staged at `perm` behind the sections above where the register form runs, from perm_src
  // behind the FFT-SPA section
  int perm, perm_src;
  int bytes;                  // the sections above and the selectors
  // FFT-SPA section, from `perm` on (the min-max kernels do not stage it): check of each
  // edge, first check of each warp task, transposed-multiplication basis
  int edge_row, task_c0, at_log, fft_bytes;
};

// One code and the frames to decode with it.  (The mixed-code kernel reads edge_col and
// the variable-node view from the blob in global memory, through L1, and stages the rest.)
struct JobDesc {
  const unsigned char* blob;  // code description (device)
  CodeBlob off;
  const uint8_t* gamma;       // [frames][n][q]
  uint8_t* out_sym;           // [frames][n]
  int32_t* out_iters;         // [frames]
  uint8_t* out_ok;            // [frames]
  int q, n, m, dmax, vmax;    // field order, columns, rows, largest row and column degree
  int perm_at;                // where the permutation selectors are staged, behind the other staged sections
  int reg;                    // q = 8, 16, 32: lanes that take a check each in the register form of the
                              // check-node pass (the slot's threads, or D = -1 fewer; mixed-code kernel:
                              // 0, the group form); q = 64 in the mixed-code kernel: not 0 when every
                              // check has degree 4
  int key16;                  // (255 * (max column degree + 1) + 1) * q <= 65536: 16-bit argmin keys
  int group_bytes;            // per-group shared scratch for this code
  int frames, max_iters, early_stop;
  int item_begin;             // index of this job's first frame in the launch's work list
  unsigned long long* work;   // optional: adds the (x, y) pairs the convolutions visit (null: no count)
};

// Copy the sections of the code description that the min-max kernels read to shared memory:
// [0, common) bytes, then (perm: the register form, their only reader) the permutation selectors.
__device__ __forceinline__ void stage_blob(unsigned char* sblob, const JobDesc& job, int common_bytes, bool perm, int tid,
                                           int nthr) {
  for (int i = tid; i < common_bytes / 16; i += nthr)
    reinterpret_cast<uint4*>(sblob)[i] = reinterpret_cast<const uint4*>(job.blob)[i];
  if (perm)
    for (int i = tid; i < (job.off.bytes - job.off.perm) / 16; i += nthr)
      reinterpret_cast<uint4*>(sblob + common_bytes)[i] = reinterpret_cast<const uint4*>(job.blob + job.off.perm_src)[i];
}

constexpr int kMaxJobs = 32;

// One launch: up to N jobs whose frames form one work list, served by
// persistent blocks of `fpb` frame slots each.  Single-code launches pass the one
// job alone: a table of 32 is 7 KB of kernel parameters to copy on every launch.
template <int N> struct LaunchParamsOf {
  JobDesc jobs[N];
  int njobs, total_items;
  unsigned int* counter;      // next work item
  uint8_t* msg;               // message slots, one per (block, frame slot)
  size_t slot_bytes;
  int fpb;                    // frame slots per block (blockDim / fpb threads each)
  int slot_smem;              // shared bytes per frame slot
  int blob_cap, n_cap;        // largest code blob and N among the jobs
  int xs_off;                 // resident launches: shared-memory offset of the slot's messages
  int static_items;           // 1: no more items than frame slots; slot s takes item s (no counter)
};
template <int QSEL> using LaunchParams = LaunchParamsOf<QSEL == 0 ? kMaxJobs : 1>;

// Control words of a frame slot, then (mixed-code kernel) a copy of its job.
__host__ __device__ constexpr int ctl_bytes(int qsel) {
  return 16 + (qsel == 0 ? (int)(sizeof(JobDesc) + 15) / 16 * 16 : 0);
}

// Threads of a block whose frame keeps its messages in shared memory (two
// blocks per SM: the same 24 warps as three 256-thread blocks).
constexpr int kResidentThreads = 384;


// Check-node permutation by scatter from registers (q >= 16) instead of staging
// the incoming rows in shared memory and gathering them.
template <int Q> __host__ __device__ constexpr bool scatter_perm() { return Q >= 16; }

// per-group shared scratch: the d incoming rows (q symbols of mb bytes each;
// not with the scatter permutation) and 2*dmax+1 16-bit vectors: P_0..P_{d-1},
// F_1..F_{d-2}, two B vectors and the middle beta R.  Pruned convolutions: the
// vectors are bytes, B_j takes the place of P_j and the middle beta that of F_{j-1},
// and the copies and the list of pr_conv follow.
template <int Q> __host__ __device__ constexpr int group_scratch_bytes(int dmax, int mb = 1, bool pr = false) {
  return pr ? ((2 * dmax - 2) * Q + kPrTmp<Q> + 15) / 16 * 16
            : (scatter_perm<Q>() ? 0 : ((dmax * Q * mb + 15) / 16) * 16) + (2 * dmax + 1) * vec_bytes<Q>();
}

// named barrier over the threads of one frame slot (ids 1..fpb)
__device__ __forceinline__ void slot_sync(int id, int nthreads) {
  asm volatile("bar.sync %0, %1;" ::"r"(id), "r"(nthreads) : "memory");
}
__device__ __forceinline__ int slot_sync_or(int id, int nthreads, int pred) {
  int r;
  asm volatile(
      "{\n\t.reg .pred p, q;\n\tsetp.ne.s32 p, %1, 0;\n\tbar.red.or.pred q, %2, %3, p;\n\t"
      "selp.s32 %0, 1, 0, q;\n\t}"
      : "=r"(r)
      : "r"(pred), "r"(id), "r"(nthreads)
      : "memory");
  return r;
}

template <int N> __device__ __forceinline__ void store_bytes(uint8_t* p, const int (&v)[N]) {
  if constexpr (N == 1) {
    *p = (uint8_t)v[0];
  } else if constexpr (N == 2) {
    *reinterpret_cast<uint16_t*>(p) = (uint16_t)(v[0] | (v[1] << 8));
  } else if constexpr (N == 4) {
    *reinterpret_cast<uint32_t*>(p) = (uint32_t)(v[0] | (v[1] << 8) | (v[2] << 16) | (v[3] << 24));
  } else {
    uint2 w;
    w.x = (uint32_t)(v[0] | (v[1] << 8) | (v[2] << 16) | (v[3] << 24));
    w.y = (uint32_t)(v[4] | (v[5] << 8) | (v[6] << 16) | (v[7] << 24));
    *reinterpret_cast<uint2*>(p) = w;
  }
}

// NB bytes -> NB/2 words of two 16-bit values (byte 2i in the low half of word i)
template <int NB> __device__ __forceinline__ void load_pairs(const uint8_t* p, uint32_t (&w)[NB / 2]) {
  if constexpr (NB == 2) {
    w[0] = __byte_perm(*reinterpret_cast<const uint16_t*>(p), 0, 0x4140);
  } else if constexpr (NB == 4) {
    const uint32_t x = *reinterpret_cast<const uint32_t*>(p);
    w[0] = __byte_perm(x, 0, 0x4140); w[1] = __byte_perm(x, 0, 0x4342);
  } else if constexpr (NB == 8) {
    const uint2 x = *reinterpret_cast<const uint2*>(p);
    w[0] = __byte_perm(x.x, 0, 0x4140); w[1] = __byte_perm(x.x, 0, 0x4342);
    w[2] = __byte_perm(x.y, 0, 0x4140); w[3] = __byte_perm(x.y, 0, 0x4342);
  } else {
    const uint4 x = *reinterpret_cast<const uint4*>(p);
    w[0] = __byte_perm(x.x, 0, 0x4140); w[1] = __byte_perm(x.x, 0, 0x4342);
    w[2] = __byte_perm(x.y, 0, 0x4140); w[3] = __byte_perm(x.y, 0, 0x4342);
    w[4] = __byte_perm(x.z, 0, 0x4140); w[5] = __byte_perm(x.z, 0, 0x4342);
    w[6] = __byte_perm(x.w, 0, 0x4140); w[7] = __byte_perm(x.w, 0, 0x4342);
  }
}

// inverse of load_pairs (every 16-bit value must be <= 255)
template <int NB> __device__ __forceinline__ void store_pairs(uint8_t* p, const uint32_t (&w)[NB / 2]) {
  if constexpr (NB == 2) {
    *reinterpret_cast<uint16_t*>(p) = (uint16_t)__byte_perm(w[0], 0, 0x4420);
  } else if constexpr (NB == 4) {
    *reinterpret_cast<uint32_t*>(p) = __byte_perm(w[0], w[1], 0x6420);
  } else if constexpr (NB == 8) {
    uint2 x;
    x.x = __byte_perm(w[0], w[1], 0x6420);
    x.y = __byte_perm(w[2], w[3], 0x6420);
    *reinterpret_cast<uint2*>(p) = x;
  } else {
    uint4 x;
    x.x = __byte_perm(w[0], w[1], 0x6420);
    x.y = __byte_perm(w[2], w[3], 0x6420);
    x.z = __byte_perm(w[4], w[5], 0x6420);
    x.w = __byte_perm(w[6], w[7], 0x6420);
    *reinterpret_cast<uint4*>(p) = x;
  }
}

// N bytes, or N 16-bit values, to N ints (vector loads of at most 16 bytes)
template <int N> __device__ __forceinline__ void load_ints(const uint8_t* p, int (&v)[N]) {
  uint32_t w[N / 2];
  load_pairs<N>(p, w);
#pragma unroll
  for (int i = 0; i < N / 2; ++i) {
    v[2 * i] = (int)(w[i] & 0xFFFFu);
    v[2 * i + 1] = (int)(w[i] >> 16);
  }
}
template <int N> __device__ __forceinline__ void load_ints(const uint16_t* p, int (&v)[N]) {
  uint32_t w[N / 2];
  if constexpr (N == 8) {
    const uint4 t = *reinterpret_cast<const uint4*>(p);
    w[0] = t.x; w[1] = t.y; w[2] = t.z; w[3] = t.w;
  } else if constexpr (N == 4) {
    const uint2 t = *reinterpret_cast<const uint2*>(p);
    w[0] = t.x; w[1] = t.y;
  } else {
    w[0] = *reinterpret_cast<const uint32_t*>(p);
  }
#pragma unroll
  for (int i = 0; i < N / 2; ++i) {
    v[2 * i] = (int)(w[i] & 0xFFFFu);
    v[2 * i + 1] = (int)(w[i] >> 16);
  }
}
template <int N> __device__ __forceinline__ void store_u16(uint16_t* p, const int (&v)[N]) {
  uint32_t w[N / 2];
#pragma unroll
  for (int i = 0; i < N / 2; ++i) w[i] = __byte_perm((uint32_t)v[2 * i], (uint32_t)v[2 * i + 1], 0x5410);
  if constexpr (N == 8) *reinterpret_cast<uint4*>(p) = make_uint4(w[0], w[1], w[2], w[3]);
  else if constexpr (N == 4) *reinterpret_cast<uint2*>(p) = make_uint2(w[0], w[1]);
  else *reinterpret_cast<uint32_t*>(p) = w[0];
}

template <int G> __device__ __forceinline__ int group_min(int v, unsigned gmask) {
#pragma unroll
  for (int o = 1; o < G; o <<= 1) v = min(v, __shfl_xor_sync(gmask, v, o));
  return v;
}

template <int G> __device__ __forceinline__ void group_sync(unsigned gmask) {
  if constexpr (G > 1) __syncwarp(gmask);
}

template <int G> __device__ __forceinline__ unsigned group_mask(int lane) {
  return (G == 32) ? 0xFFFFFFFFu : (((1u << G) - 1u) << (lane & ~(G - 1)));
}

// ---------------------------------------------------------------- q = 4 in registers
// C(x) = min_y max(A(y), B(x ^ y)) on 4-symbol vectors held as two words of
// 16-bit values, (v0, v1) and (v2, v3): B ^ 1 swaps the halves of each word,
// B ^ 2 swaps the words.
__device__ __forceinline__ uint2 conv4(uint2 a, uint2 b) {
  const uint32_t a0 = __byte_perm(a.x, 0, 0x1010), a1 = __byte_perm(a.x, 0, 0x3232);
  const uint32_t a2 = __byte_perm(a.y, 0, 0x1010), a3 = __byte_perm(a.y, 0, 0x3232);
  const uint32_t s0 = __byte_perm(b.x, 0, 0x1032), s1 = __byte_perm(b.y, 0, 0x1032);
  return make_uint2(vmin2(vmin2(vmax2(a0, b.x), vmax2(a1, s0)), vmin2(vmax2(a2, b.y), vmax2(a3, s1))),
                    vmin2(vmin2(vmax2(a0, b.y), vmax2(a1, s1)), vmin2(vmax2(a2, b.x), vmax2(a3, s0))));
}


// ---------------------------------------------------------------- q = 8, 16, 32 in registers
// One lane per check: a message vector is W = q / 2 words of 16-bit pairs (or q / 4
// words of bytes) in the lane's registers.  y's register part picks the words and
// its lowest bit swaps their halves, so every index is static: a convolution is
// W * q maxima and minima with no shuffle and no shared memory, and the pass is bound
// by the ALU pipe (80 % busy at GF(16) N=1024; the 8- and 16-lane groups spent as
// much on shuffles, vector loads and stores, and group barriers).  Resident-message
// kernels only.  Measured on GB300, group form against this: GF(16) (2,4) N=1024,
// 4096 frames 4.60 against 2.21 ms; GF(8) (2,4) N=512, 8192 frames 2.10 against 0.89 ms;
// GF(32) (3,6) N=600, 2999 frames 9.24 against 7.79 ms.
template <int Q> __host__ __device__ constexpr bool reg_form() { return Q == 8 || Q == 16 || Q == 32; }

// C(x) = min_y max(A(y), B(x ^ y)) (B's halves are swapped for the odd y and back).
// Two y at a time, so that their two minima are one three-operand instruction (one
// at a time the compiler kept two: GF(32) N=600 10 % slower).  Half of the maxima on
// the FMA pipe (GF(16) N=1024, 0 to 4 eighths: 2.49, 2.42, 2.34, 2.31, 2.25 ms).
// q = 32 keeps the loop over the lowest bit of y rolled (500 instructions a turn).
template <int W>
__device__ __forceinline__ void conv_reg(const uint32_t (&A)[W], uint32_t (&B)[W], uint32_t (&C)[W]) {
  constexpr int F = W / 2;             // words whose maxima run on the FMA pipe (see FmaEighths)
#pragma unroll
  for (int w = 0; w < W; ++w) C[w] = 0xFFFFFFFFu;
#pragma unroll(W >= 16 ? 1 : 2)
  for (int half = 0; half < 2; ++half) {
    const uint32_t sel = half ? 0x3232u : 0x1010u;
#pragma unroll
    for (int i = 0; i < W; i += 2) {
      const uint32_t a0 = __byte_perm(A[i], 0, sel), a1 = __byte_perm(A[i + 1], 0, sel);
#pragma unroll
      for (int w = 0; w < W; ++w) {
        const uint32_t m0 = w < F ? vmax2_fma(a0, B[w ^ i]) : vmax2(a0, B[w ^ i]);
        const uint32_t m1 = w < F ? vmax2_fma(a1, B[w ^ i ^ 1]) : vmax2(a1, B[w ^ i ^ 1]);
        C[w] = __vimin3_u16x2(C[w], m0, m1);
      }
    }
#pragma unroll
    for (int w = 0; w < W; ++w) B[w] = __byte_perm(B[w], 0, 0x1032);
  }
}

// Byte selectors of "element y of the result is element h y of the argument" for
// the q / 4 words of a row: a selector among the eight bytes of a word pair for
// each word, and masks that choose between the pairs (bit 3 of h y, then bit 4).
template <int Q> struct PermRow {
  static constexpr int NB = Q / 4;
  static constexpr int sel_bytes = Q == 8 ? 4 : Q == 16 ? 16 : 16;   // NB 16-bit selectors (q = 16: padded)
  static constexpr int masks = Q == 8 ? 0 : Q == 16 ? 1 : 2;
  static constexpr int bytes = sel_bytes + masks * Q;
};

template <int Q>
__device__ __forceinline__ void gather_row(const uint32_t (&r)[Q / 4], uint32_t (&o)[Q / 4], const uint8_t* t) {
  constexpr int NB = Q / 4;
  uint32_t s[NB / 2];
  if constexpr (Q == 8) {
    s[0] = *reinterpret_cast<const uint32_t*>(t);
  } else if constexpr (Q == 16) {
    const uint2 v = *reinterpret_cast<const uint2*>(t);
    s[0] = v.x; s[1] = v.y;
  } else {
    const uint4 v = *reinterpret_cast<const uint4*>(t);
    s[0] = v.x; s[1] = v.y; s[2] = v.z; s[3] = v.w;
  }
  const uint32_t* m = reinterpret_cast<const uint32_t*>(t + PermRow<Q>::sel_bytes);
  uint32_t mk[PermRow<Q>::masks ? PermRow<Q>::masks * NB : 1];
  if constexpr (Q >= 16) {
#pragma unroll
    for (int i = 0; i < PermRow<Q>::masks * NB; i += 4) {
      const uint4 v = *reinterpret_cast<const uint4*>(m + i);
      mk[i] = v.x; mk[i + 1] = v.y; mk[i + 2] = v.z; mk[i + 3] = v.w;
    }
  }
#pragma unroll
  for (int w = 0; w < NB; ++w) {
    const uint32_t sl = (w & 1) ? s[w / 2] >> 16 : s[w / 2];      // (the permute reads 16 bits of it)
    uint32_t v = __byte_perm(r[0], r[1], sl);
    if constexpr (Q >= 16) {
      const uint32_t v1 = __byte_perm(r[2], r[3], sl);
      v = (v & ~mk[w]) | (v1 & mk[w]);
    }
    if constexpr (Q >= 32) {
      const uint32_t v2 = __byte_perm(r[4], r[5], sl), v3 = __byte_perm(r[6], r[7], sl);
      const uint32_t u = (v2 & ~mk[w]) | (v3 & mk[w]);
      v = (v & ~mk[NB + w]) | (u & mk[NB + w]);
    }
    o[w] = v;
  }
}

// a row of Q bytes to and from Q / 4 words
template <int Q> __device__ __forceinline__ void load_row(const uint8_t* p, uint32_t (&r)[Q / 4]) {
  if constexpr (Q == 8) {
    const uint2 v = *reinterpret_cast<const uint2*>(p);
    r[0] = v.x; r[1] = v.y;
  } else {
#pragma unroll
    for (int i = 0; i < Q / 16; ++i) {
      const uint4 v = reinterpret_cast<const uint4*>(p)[i];
      r[4 * i] = v.x; r[4 * i + 1] = v.y; r[4 * i + 2] = v.z; r[4 * i + 3] = v.w;
    }
  }
}
template <int Q> __device__ __forceinline__ void store_row(uint8_t* p, const uint32_t (&r)[Q / 4]) {
  if constexpr (Q == 8) {
    *reinterpret_cast<uint2*>(p) = make_uint2(r[0], r[1]);
  } else {
#pragma unroll
    for (int i = 0; i < Q / 16; ++i)
      reinterpret_cast<uint4*>(p)[i] = make_uint4(r[4 * i], r[4 * i + 1], r[4 * i + 2], r[4 * i + 3]);
  }
}
template <int NB> __device__ __forceinline__ void unpack_row(const uint32_t (&r)[NB], uint32_t (&v)[2 * NB]) {
#pragma unroll
  for (int i = 0; i < NB; ++i) {
    v[2 * i] = __byte_perm(r[i], 0, 0x4140);
    v[2 * i + 1] = __byte_perm(r[i], 0, 0x4342);
  }
}
template <int NB> __device__ __forceinline__ void pack_row(const uint32_t (&v)[2 * NB], uint32_t (&r)[NB]) {
#pragma unroll
  for (int i = 0; i < NB; ++i) r[i] = __byte_perm(v[2 * i], v[2 * i + 1], 0x6420);
}

// shared scratch of nthr lanes: F_1..F_{d-3} of each lane's check, as bytes
template <int Q> __host__ __device__ constexpr int reg_scratch_bytes(int nthr, int dmax) {
  return dmax > 3 ? nthr * (dmax - 3) * Q : 0;
}

// ---------------------------------------------------------------- q = 4, one warp per frame
// A frame of a small GF(4) code (at most 32 checks of degree <= kW4Deg, columns
// of degree <= 2) decoded by one warp with no block barrier: lane r owns check r
// and keeps its edges' alpha and beta rows (4 bytes each) in registers; the
// permutation and de-permutation byte selectors and the GF(4) products of its
// edges are set up once per frame; beta goes to the slot's message area (one
// word per edge) only for the variable-node step of the other edge's owner.
// Each edge's owner computes its variable node's sum, decision and next alpha,
// so every variable node is handled by the lanes of its (one or two) edges.
// The arithmetic is that of the other forms (Alg. 2): the same convolutions,
// the same min-normalization, saturation at 255 and lowest-symbol argmin.
// Returns false, having done nothing, when the code is outside these limits.
// DW = 4: every check has degree 4 (the per-iteration loops need no degree tests).
constexpr int kW4Deg = 4;
template <int DW>
__device__ __forceinline__ bool decode_frame_warp4(const JobDesc& job, int frame, uint8_t* X,
                                                   const unsigned char* sblob, const unsigned char* cold, int lane) {
  if (job.m > 32 || job.dmax > kW4Deg || job.vmax > 2) return false;
  const uint8_t* exp2 = sblob + job.off.exp2;
  const uint8_t* glog = sblob + job.off.log;
  const uint16_t* row_ptr = reinterpret_cast<const uint16_t*>(sblob + job.off.row_ptr);
  const uint16_t* edge_col = reinterpret_cast<const uint16_t*>(cold + job.off.edge_col);
  const uint8_t* edge_lh = sblob + job.off.edge_lh;
  const uint8_t* edge_lhi = sblob + job.off.edge_lhi;
  const uint16_t* vn_ptr = reinterpret_cast<const uint16_t*>(cold + job.off.vn_ptr);
  const uint16_t* vn_edge = reinterpret_cast<const uint16_t*>(cold + job.off.vn_edge);
  const uint8_t* gam = job.gamma + (size_t)frame * job.n * 4;
  const bool mine = lane < job.m;
  const int e0 = mine ? row_ptr[lane] : 0, d = mine ? row_ptr[lane + 1] - e0 : 0;
  // degree of the per-iteration loops: the lanes without a check compute on zeros and store nothing
  const int dd = DW > 0 ? DW : d;
  // per edge j < d: gamma row of its column, selectors, products, the other edge (-1: none)
  uint32_t gr[kW4Deg], psel[kW4Deg], bsel[kW4Deg], mt[kW4Deg], al[kW4Deg], be[kW4Deg];
  int oe[kW4Deg], col[kW4Deg];
  bool first_owner[kW4Deg];
#pragma unroll
  for (int j = 0; j < kW4Deg; ++j) {
    gr[j] = psel[j] = bsel[j] = mt[j] = al[j] = be[j] = 0u;
    oe[j] = -1;
    col[j] = 0;
    first_owner[j] = false;
    if (j < d) {
      const int e = e0 + j, c = edge_col[e];
      col[j] = c;
      gr[j] = *reinterpret_cast<const uint32_t*>(gam + (size_t)c * 4);
      // P_j(y) = alpha_j(h^-1 y) as the 16-bit pairs (P(0), P(1)), (P(2), P(3))
      const int lhinv = edge_lhi[e];
      const uint32_t s1 = exp2[lhinv], s2 = exp2[lhinv + 1], s3 = s1 ^ s2;
      psel[j] = (0x4040u | (s1 << 8)) | ((0x4040u | s2 | (s3 << 8)) << 16);
      // beta_j(a) = R(h a): byte a from the 16-bit value R(h a) of the pairs R
      const int lh = edge_lh[e];
      const int i1 = exp2[lh], i2 = exp2[lh + 1], i3 = i1 ^ i2;
      bsel[j] = (uint32_t)((((i1 >> 1) << 2) | ((i1 & 1) << 1)) << 4) |
                (uint32_t)((((i2 >> 1) << 2) | ((i2 & 1) << 1)) << 8) |
                (uint32_t)((((i3 >> 1) << 2) | ((i3 & 1) << 1)) << 12);
      // h c for c = 0..3, two bits each (syndrome)
      mt[j] = (uint32_t)exp2[lh] << 2 | (uint32_t)exp2[glog[2] + lh] << 4 | (uint32_t)exp2[glog[3] + lh] << 6;
      const int k0 = vn_ptr[c], k1 = vn_ptr[c + 1];
      first_owner[j] = vn_edge[k0] == e;
      for (int k = k0; k < k1; ++k)
        if (vn_edge[k] != e) oe[j] = vn_edge[k];
      al[j] = gr[j];                             // alpha^(0) = gamma
    }
  }
  const bool counting = job.work != nullptr;
  unsigned long long work = 0;
  // decisions from the sums S = gamma + the incoming betas (lowest symbol on ties), and the syndrome
  uint32_t cw = 0;                               // decisions of the lane's edges, two bits each
  auto decide = [&](int j, uint32_t s0, uint32_t s1) {
    const uint32_t kw = vmin2(s0 * 4u + 0x10000u, s1 * 4u + 0x30002u);
    const uint32_t key = min(kw & 0xFFFFu, kw >> 16);
    cw |= (key & 3u) << (2 * j);
  };
  auto syndrome_ok = [&]() -> bool {
    uint32_t sy = 0;
#pragma unroll
    for (int j = 0; j < kW4Deg; ++j)
      if (j < d) sy ^= (mt[j] >> (2 * ((cw >> (2 * j)) & 3u))) & 3u;   // (mt is 0 past d)
    return __all_sync(0xFFFFFFFFu, sy == 0);
  };
  auto unpack = [](uint32_t r, uint32_t& lo, uint32_t& hi) {
    lo = __byte_perm(r, 0, 0x4140);
    hi = __byte_perm(r, 0, 0x4342);
  };
  // c^(0) = argmin gamma
#pragma unroll
  for (int j = 0; j < kW4Deg; ++j)
    if (j < d) {
      uint32_t g0, g1;
      unpack(gr[j], g0, g1);
      decide(j, g0, g1);
    }
  const bool es = job.early_stop != 0;
  bool ok = (es || job.max_iters == 0) ? syndrome_ok() : false;
  int iters = 0;
  if (!(es && ok)) {
    for (int k = 1; k <= job.max_iters; ++k) {
      // check-node pass (the register form of one check)
      if (counting && d > 2) work += 16ull * 3 * (d - 2);
      uint2 P[kW4Deg], F[kW4Deg], Plast = make_uint2(0u, 0u);
#pragma unroll
      for (int j = 0; j < kW4Deg; ++j) {
        P[j] = make_uint2(0u, 0u);
        F[j] = make_uint2(0u, 0u);
        if (j < dd) {
          P[j].x = __byte_perm(al[j], 0, psel[j] & 0xFFFFu);
          P[j].y = __byte_perm(al[j], 0, psel[j] >> 16);
          Plast = P[j];
        }
      }
      F[0] = P[0];
      uint2 Flast = F[0];
#pragma unroll
      for (int j = 1; j < kW4Deg - 1; ++j)
        if (j <= dd - 2) {
          F[j] = conv4(F[j - 1], P[j]);
          Flast = F[j];
        }
      uint2 Bc = Plast;
      uint2 R[kW4Deg];
#pragma unroll
      for (int j = 0; j < kW4Deg; ++j) R[j] = make_uint2(0u, 0u);
#pragma unroll
      for (int j = kW4Deg - 2; j >= 1; --j) {
        if (j <= dd - 2) {
          R[j] = conv4(F[j - 1], Bc);
          Bc = conv4(Bc, P[j]);
        }
      }
#pragma unroll
      for (int j = 0; j < kW4Deg; ++j) {
        if (j < dd) {
          // beta_0 = B_1, beta_{d-1} = F_{d-2}, else the middle R_j
          const uint2 r = j == 0 ? Bc : (j == dd - 1 ? Flast : R[j]);
          be[j] = __byte_perm(r.x, r.y, bsel[j]);
          if (mine) reinterpret_cast<uint32_t*>(X)[e0 + j] = be[j];
        }
      }
      __syncwarp();
      // variable-node step of each of the lane's edges: S = gamma + beta_e + beta_other;
      // alpha_e = min(255, (S - beta_e) - min (S - beta_e))
      const bool decide_now = es || k == job.max_iters;
      if (decide_now) cw = 0;
#pragma unroll
      for (int j = 0; j < kW4Deg; ++j) {
        if (j < dd) {
          uint32_t t0, t1, b0, b1;
          unpack(gr[j], t0, t1);
          if (oe[j] >= 0) {
            unpack(reinterpret_cast<const uint32_t*>(X)[oe[j]], b0, b1);
            t0 += b0;
            t1 += b1;
          }
          if (decide_now) {
            unpack(be[j], b0, b1);
            decide(j, t0 + b0, t1 + b1);
          }
          const uint32_t mw = vmin2(t0, t1);
          const uint32_t mm = min(mw & 0xFFFFu, mw >> 16) * 0x10001u;
          al[j] = __byte_perm(vmin2(t0 - mm, 0x00FF00FFu), vmin2(t1 - mm, 0x00FF00FFu), 0x6420);
        }
      }
      __syncwarp();
      iters = k;
      if (decide_now) ok = syndrome_ok();
      if (es && ok) break;
    }
  }
#pragma unroll
  for (int j = 0; j < kW4Deg; ++j)
    if (j < d && first_owner[j]) job.out_sym[(size_t)frame * job.n + col[j]] = (uint8_t)((cw >> (2 * j)) & 3u);
  if (lane == 0) {
    job.out_iters[frame] = iters;
    job.out_ok[frame] = ok ? 1 : 0;
  }
  if (counting && work) atomicAdd(job.work, work);
  return true;
}

// ---------------------------------------------------------------- one frame on several SMs
// A thread-block cluster decodes one frame: rank k of the cluster owns the
// checks [k * cpc, (k + 1) * cpc) with the message rows of their edges, and the
// columns [k * npc, (k + 1) * npc) with their reliabilities and decisions, all
// in its shared memory.  The check-node pass is local to a rank; the variable-
// node pass and the syndrome reach the other ranks' rows and decisions through
// distributed shared memory, with one cluster barrier after each pass.
struct SplitCtx {
  int rank, size;
  int r0, r1, n0, n1;         // the rank's checks and columns
  int e0;                     // first edge of the rank's checks
  int t0, t1;                 // the rank's warp tasks (FFT-SPA, lane-per-edge form)
  int npc;                    // columns per rank
  const uint8_t* gam;         // the rank's reliability rows (shared memory)
  uint8_t* const* vrow;       // message row of each edge of the rank's columns, in column order
  int* flags;                 // [2][kMaxSplit] syndrome flags of the ranks
};
constexpr int kMaxSplit = 16;

__device__ __forceinline__ void cluster_barrier() {
  asm volatile("barrier.cluster.arrive.release;\n\tbarrier.cluster.wait.acquire;" ::: "memory");
}
// address of this rank's shared-memory object p in rank r's shared memory
template <class T> __device__ __forceinline__ T* at_rank(T* p, int r) {
  uint64_t d;
  asm("mapa.u64 %0, %1, %2;" : "=l"(d) : "l"(p), "r"(r));
  return reinterpret_cast<T*>(d);
}

// ---------------------------------------------------------------- one frame
// Decodes frame `frame` of `job` with the nthr threads of one frame slot
// (slot thread index stid, named barrier bar_id).  sblob holds the job's code
// description, chat[n] the decisions, scratch the per-group buffers; X is the
// slot's message area ([nnz][q] bytes); cold: where edge_col and the variable-node view
// of the description are (sblob, or the blob in global memory).
// q = 4 codes of check degree <= kRegDeg take the register form of the check-node pass
// (8-bit messages, minimal schedule).  PR: the check-node convolutions are pruned
// (pr_conv; 32-lane groups, 8-bit messages, minimal schedule).  W4: a GF(4) frame slot of one warp may take the one-warp form
// (decode_frame_warp4; resident-message kernels, which have the registers for it).
// D > 0: every check of the code has degree D (a compile-time loop bound and
// vector layout; 0: the degrees are read per check; -1: so they are, and not every
// lane of the slot has room for a check in the register form).  SP: the threads are those of
// one rank of a cluster that decodes the frame together (sc; X then holds the
// message rows of the rank's own edges).
template <class g, int MB, bool T1, bool PR = false, bool W4 = false, int D = 0, bool SP = false>
__device__ __forceinline__ void decode_frame(const JobDesc& job, int frame, uint8_t* Xown, const unsigned char* sblob,
                                             const unsigned char* cold, uint8_t* chat, unsigned char* scratch,
                                             int stid, int nthr, int bar_id, const SplitCtx* sc = nullptr) {
  constexpr int Q = g::Q;
  constexpr int PW = g::PW;
  constexpr int RS = Q * MB;                 // bytes of one message row
  constexpr bool kScatter = scatter_perm<Q>();
  static_assert(MB == 1 || MB == 2, "message bytes");
  static_assert(!PR || (g::G == 32 && MB == 1 && !T1), "pruned convolutions: 32-lane groups, 8-bit, minimal");
  if constexpr (Q == 4 && MB == 1 && !T1 && W4) {
    // one warp per frame: a slot of 32 threads
    if (nthr == 32 && decode_frame_warp4<D == 4 ? 4 : 0>(job, frame, Xown, sblob, cold, stid)) return;
  }
  // pairs (x, y) the convolutions visit in this frame (counted when job.work is set)
  const bool counting = job.work != nullptr;
  unsigned long long work = 0;
  const uint8_t* exp2 = sblob + job.off.exp2;        // x^(i mod (q-1)), i < 2(q-1)
  const uint8_t* glog = sblob + job.off.log;         // log_x(v), v >= 1
  const uint16_t* row_ptr = reinterpret_cast<const uint16_t*>(sblob + job.off.row_ptr);
  const uint16_t* edge_col = reinterpret_cast<const uint16_t*>(cold + job.off.edge_col);
  const uint8_t* edge_lh = sblob + job.off.edge_lh;    // log_x(h) of each edge
  const uint8_t* edge_lhi = sblob + job.off.edge_lhi;  // log_x(h^-1) of each edge
  const uint16_t* vn_ptr = reinterpret_cast<const uint16_t*>(cold + job.off.vn_ptr);
  const uint16_t* vn_edge = reinterpret_cast<const uint16_t*>(cold + job.off.vn_edge);

  const int lane = threadIdx.x & 31;
  // check-node groups (G lanes per check)
  const int grp = stid / g::G, ngroups = nthr / g::G;
  const int gl = stid % g::G;
  const unsigned gmask = group_mask<g::G>(lane);
  const ConvLane cl = conv_lane<g>(gl >> g::LB, gl & (g::DN - 1));
  // variable-node groups (VG lanes per variable node)
  // (16-bit messages keep at most 8 symbols per lane: their rows are read symbol by symbol)
  constexpr int VBPL = (MB == 2 && g::VBPL > 8) ? 8 : g::VBPL, VG = Q / VBPL, VW = VBPL / 2;
  const int vgrp = stid / VG, nvgroups = nthr / VG;
  const int vgl = stid % VG;
  const unsigned vmask = group_mask<VG>(lane);
  constexpr bool kGammaRegs = Q <= 16 && MB == 1;
  uint32_t gcache[kGammaRegs ? VW : 1];

  // lane constants for the gather permutation (staged rows): logarithms of the
  // symbols this lane gathers, packed 8 bits per symbol; the zero symbol, which
  // every multiplication fixes, is flagged separately.
  uint32_t py_log0 = 0, py_log1 = 0, py_nz0 = 0;   // word i: bits [8i, 8i+8)
  if constexpr (!kScatter) {
#pragma unroll
    for (int i = 0; i < PW; ++i) {
      const int w = gl + i * g::G;
      if (w < g::W) {
        if (w) { py_log0 |= (uint32_t)glog[2 * w] << (8 * i); py_nz0 |= 1u << i; }
        py_log1 |= (uint32_t)glog[2 * w + 1] << (8 * i);
      }
    }
  }
  // de-permutation: log of the first symbol this lane writes (-1 for symbol 0)
  const int da_log0 = gl ? (int)glog[gl * g::BPL] : -1;

  unsigned char* gs = scratch + (size_t)grp * (PR ? group_scratch_bytes<Q>(job.dmax, 1, true) : job.group_bytes);
  uint8_t* stage = gs;                                                   // [dmax][q * MB] bytes (staged rows)
  const int dm = D > 0 ? D : job.dmax;
  unsigned char* vecs = gs + (kScatter ? 0 : ((dm * RS + 15) / 16) * 16);
  using Sym = std::conditional_t<PR, uint8_t, uint16_t>;     // a vector's elements
  constexpr int VB = PR ? Q : g::VB;
  auto vec = [&](int i) { return reinterpret_cast<uint32_t*>(vecs + (size_t)i * VB); };
  auto vec16 = [&](int i) { return reinterpret_cast<Sym*>(vecs + (size_t)i * VB); };
  // vectors: P_j = vec(j) (j < dmax), F_j = vec(dmax + j - 1) (1 <= j <= d-2),
  // B ping-pong = vec(2 dmax - 2), vec(2 dmax - 1), R = vec(2 dmax) (neither if PR)
  const int vF = dm - 1, vB = 2 * dm - 2, vR = 2 * dm;
  const uint8_t* gam = job.gamma + (size_t)frame * job.n * Q;
  // rows are addressed by edge number: a rank's area starts with the row of its first edge
  uint8_t* X = SP ? Xown - (ptrdiff_t)sc->e0 * RS : Xown;
  const int r_first = SP ? sc->r0 : 0, r_last = SP ? sc->r1 : job.m;
  const int n_first = SP ? sc->n0 : 0, n_last = SP ? sc->n1 : job.n;
  // reliabilities of the columns of the variable-node pass, message row of entry k of
  // the column-ordered edge list, decision of column c
  const uint8_t* vgam = SP ? sc->gam - (ptrdiff_t)n_first * Q : gam;
  const int k_first = SP ? vn_ptr[n_first] : 0;
  auto vn_row = [&](int k) -> uint8_t* {
    if constexpr (SP) return sc->vrow[k - k_first];
    else return X + (size_t)vn_edge[k] * RS;
  };
  auto decision = [&](int c) -> int {
    if constexpr (SP) return *at_rank(chat + c, c / sc->npc);
    else return chat[c];
  };
  // end of a pass: its messages and decisions are visible to every thread of the frame
  auto pass_sync = [&]() {
    if constexpr (SP) cluster_barrier();
    else slot_sync(bar_id, nthr);
  };

    // ---- variable-node pass (Alg. 2, VNP and hard decision):
    //   S(a) = gamma(a) + sum over edges of beta(a);  c = argmin S (lowest a)
    //   alpha_e(a) = min(255, (S - beta_e)(a) - min_b (S - beta_e)(b))
    // Values are 16-bit halves of 32-bit words: every sum stays below 2^16
    // (at most 255 * (column degree + 1)), so plain 32-bit adds and
    // subtractions never carry or borrow across the halves.
    // 16-bit messages: the same pass on 32-bit sums, one symbol per register.  A lane's
    // symbols of a row move as one vector access: symbol by symbol (and with the rows
    // staged and gathered in the check-node pass) 4096 frames took 17.1 ms at GF(64)
    // N=576, 12.1 at GF(16) N=1024 and 5.5 at GF(8) N=512, against 14.5, 4.7 and 1.35.
    auto vnp_wide = [&](bool first, bool want_alpha) {
      constexpr int NB = VBPL;
      for (int vn = n_first + vgrp; vn < n_last; vn += nvgroups) {
        int S[NB];
        load_ints<NB>(vgam + (ptrdiff_t)vn * Q + vgl * NB, S);
        const int k0 = vn_ptr[vn], k1 = vn_ptr[vn + 1];
        if (!first) {
          for (int k = k0; k < k1; ++k) {
            int b[NB];
            load_ints<NB>(reinterpret_cast<const uint16_t*>(vn_row(k)) + vgl * NB, b);
#pragma unroll
            for (int i = 0; i < NB; ++i) S[i] += b[i];
          }
        }
        int key = 0x7FFFFFFF;
#pragma unroll
        for (int i = 0; i < NB; ++i) key = min(key, (S[i] << 8) | (vgl * NB + i));
        key = group_min<VG>(key, vmask);
        if (vgl == 0) chat[vn] = (uint8_t)(key & 0xFF);
        if (!first && want_alpha) {
          for (int k = k0; k < k1; ++k) {
            uint16_t* row = reinterpret_cast<uint16_t*>(vn_row(k)) + vgl * NB;
            int t[NB];
            load_ints<NB>(row, t);
            int mn = 0x7FFFFFFF;
#pragma unroll
            for (int i = 0; i < NB; ++i) { t[i] = S[i] - t[i]; mn = min(mn, t[i]); }
            mn = group_min<VG>(mn, vmask);
#pragma unroll
            for (int i = 0; i < NB; ++i) t[i] = min(65535, t[i] - mn);
            store_u16<NB>(row, t);
          }
        }
      }
    };

    // 16-bit messages of q < 16 start from alpha^(0) = gamma widened into every edge row
    auto init_wide = [&]() {
      const int first = SP ? row_ptr[r_first] * Q : 0, last = row_ptr[r_last] * Q;
      for (int i = first + stid; i < last; i += nthr) {
        const int e = i / Q, a = i % Q;
        reinterpret_cast<uint16_t*>(X)[i] = gam[(size_t)edge_col[e] * Q + a];
      }
    };

    // q <= 16 with every variable node in one pass of the slot's lanes: each lane
    // keeps its node's gamma words in registers from the first pass on (the later
    // passes then start without a global-memory load)
    const bool gamma_regs = kGammaRegs && n_last - n_first <= nvgroups;
    auto vnp = [&](bool first, bool want_alpha) {
      // symbol values of this lane's packed words: (a, a + 1), a = vgl * VBPL + 2 i
      const uint32_t vsym0 = (uint32_t)(vgl * VBPL) * 0x10001u + 0x10000u;
      for (int vn = n_first + vgrp; vn < n_last; vn += nvgroups) {
        uint32_t S[VW];
        if (gamma_regs && !first) {
#pragma unroll
          for (int i = 0; i < VW; ++i) S[i] = gcache[i];
        } else {
          load_pairs<VBPL>(vgam + (ptrdiff_t)vn * Q + vgl * VBPL, S);
          if (gamma_regs) {
#pragma unroll
            for (int i = 0; i < VW; ++i) gcache[i] = S[i];
          }
        }
        const int k0 = vn_ptr[vn], k1 = vn_ptr[vn + 1];
        if (!first) {
          for (int k = k0; k < k1; ++k) {
            uint32_t b[VW];
            load_pairs<VBPL>(vn_row(k) + vgl * VBPL, b);
#pragma unroll
            for (int i = 0; i < VW; ++i) S[i] += b[i];
          }
        }
        int key;
        if (job.key16) {        // key = S * q + a fits 16 bits: minimum value, lowest symbol
          uint32_t kw = S[0] * (uint32_t)Q + vsym0;
#pragma unroll
          for (int i = 1; i < VW; ++i) kw = vmin2(kw, S[i] * (uint32_t)Q + (vsym0 + 0x20002u * i));
          key = (int)min(kw & 0xFFFFu, kw >> 16);
          key = group_min<VG>(key, vmask);
          if (vgl == 0) chat[vn] = (uint8_t)(key & (Q - 1));
        } else {
          key = 0x7FFFFFFF;
#pragma unroll
          for (int i = 0; i < VW; ++i) {
            const uint32_t sy = vsym0 + 0x20002u * i;
            key = min(key, (int)(((S[i] & 0xFFFFu) << 8) | (sy & 0xFFFFu)));
            key = min(key, (int)(((S[i] >> 16) << 8) | (sy >> 16)));
          }
          key = group_min<VG>(key, vmask);
          if (vgl == 0) chat[vn] = (uint8_t)(key & 0xFF);
        }
        if (!first && want_alpha) {
          for (int k = k0; k < k1; ++k) {
            uint8_t* row = vn_row(k) + vgl * VBPL;
            uint32_t t[VW];
            load_pairs<VBPL>(row, t);
#pragma unroll
            for (int i = 0; i < VW; ++i) t[i] = S[i] - t[i];
            uint32_t mw = t[0];
#pragma unroll
            for (int i = 1; i < VW; ++i) mw = vmin2(mw, t[i]);
            int mn = (int)min(mw & 0xFFFFu, mw >> 16);
            mn = group_min<VG>(mn, vmask);
            const uint32_t mm = (uint32_t)mn * 0x10001u;
#pragma unroll
            for (int i = 0; i < VW; ++i) t[i] = vmin2(t[i] - mm, 0x00FF00FFu);
            store_pairs<VBPL>(row, t);
          }
        }
      }
    };

    // ---- syndrome of chat over all checks (slot-wide, cluster-wide for SP)
    int flag_set = 0;
    auto syndrome_ok = [&]() -> bool {
      int bad = 0;
      for (int r = r_first + stid; r < r_last; r += nthr) {
        int sy = 0;
        for (int e = row_ptr[r]; e < row_ptr[r + 1]; ++e) {
          const int c = decision(edge_col[e]);
          if (c) sy ^= exp2[glog[c] + edge_lh[e]];
        }
        bad |= sy;
      }
      bad = slot_sync_or(bar_id, nthr, bad);
      if constexpr (SP) {      // every rank's flag to every rank; two sets, so that a late reader's stays
        if (stid < sc->size) at_rank(sc->flags + flag_set * kMaxSplit + sc->rank, stid)[0] = bad;
        cluster_barrier();
        for (int k = 0; k < sc->size; ++k) bad |= sc->flags[flag_set * kMaxSplit + k];
        flag_set ^= 1;
      }
      return bad == 0;
    };

    // ---- check-node pass (Alg. 2, F & B matrices and beta), one group per check
    constexpr int CH = RS / 16 > 0 ? RS / 16 : 1;        // 16-byte pieces of one row
    // scatter permutation: piece c of the check (edges e0 ..) holds symbols
    // a = 16 part + k (k < 16) of edge j = c / CH, part = c % CH, and
    // P_j(h_j a) = alpha_j(a) with h (16 part + k) = h (16 part) ^ h k, both
    // XOR sums of the h x^b = exp2[log h + b] (16-bit messages: 8 symbols a piece)
    auto scatter_piece = [&](bool first, int e0, int c, unsigned char* base) {
      const int j = c / CH, part = c - j * CH;
      const int lh = edge_lh[e0 + j];
      const int h1 = exp2[lh], h2 = exp2[lh + 1], h4 = exp2[lh + 2];
      Sym* Pv = reinterpret_cast<Sym*>(base + (size_t)j * VB);
      if constexpr (MB == 2) {
        int v[8];
        if (first) load_ints<8>(gam + (size_t)edge_col[e0 + j] * Q + part * 8, v);
        else load_ints<8>(reinterpret_cast<const uint16_t*>(X + (size_t)(e0 + j) * RS) + part * 8, v);
        int yb = 0;
#pragma unroll
        for (int b = 3; b < g::P; ++b)
          if ((part >> (b - 3)) & 1) yb ^= exp2[lh + b];
#pragma unroll
        for (int k = 0; k < 8; ++k)
          Pv[yb ^ ((k & 1) ? h1 : 0) ^ ((k & 2) ? h2 : 0) ^ ((k & 4) ? h4 : 0)] = (uint16_t)v[k];
      } else {
        // gamma on the first pass, else the edge's message row (through one pointer: a separate
        // read-only load of gamma measured 2 % slower at GF(64))
        const uint8_t* src = first ? gam + (size_t)edge_col[e0 + j] * Q : X + (size_t)(e0 + j) * Q;
        const uint4 v = reinterpret_cast<const uint4*>(src)[part];
        const int h8 = exp2[lh + 3];
        int yb = 0;
#pragma unroll
        for (int b = 4; b < g::P; ++b)
          if ((part >> (b - 4)) & 1) yb ^= exp2[lh + b];
        const uint32_t w[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
        for (int k = 0; k < 16; ++k) {
          const int y = yb ^ ((k & 1) ? h1 : 0) ^ ((k & 2) ? h2 : 0) ^ ((k & 4) ? h4 : 0) ^ ((k & 8) ? h8 : 0);
          Pv[y] = (Sym)__byte_perm(w[k >> 2], 0, 0x4440 | (k & 3));
        }
      }
    };
    // predictions of max_x C(x), one per kind of convolution (F, B, beta): each
    // kind's maxima follow their own distribution
    int tpred[3] = {24, 24, 24};
    auto conv = [&](const uint32_t* A, const uint32_t* B, Sym* C, int kind) {
      if constexpr (PR) {
        int folded = 0;
        tpred[kind] = pr_conv<g>(reinterpret_cast<const uint8_t*>(A), reinterpret_cast<const uint8_t*>(B), C,
                                 vecs + (size_t)(2 * dm - 2) * VB, gl, tpred[kind], counting ? &folded : nullptr);
        if (counting && gl == 0) work += (unsigned long long)folded * Q;
      } else {
        mm_conv<g, MB == 1>(A, B, C, cl, gmask);
        if (counting && gl == 0) work += (unsigned long long)Q * Q;
      }
    };
    auto cnp = [&](bool first) {
      for (int r = r_first + grp; r < r_last; r += ngroups) {
        const int e0 = row_ptr[r], d = D > 0 ? D : row_ptr[r + 1] - e0;
        if constexpr (kScatter) {
          for (int c = gl; c < d * CH; c += g::G) scatter_piece(first, e0, c, vecs);
        } else {
          // stage incoming alpha rows (alpha^(0) = gamma on the first pass)
          if constexpr (MB == 2) {
            constexpr int CB = RS / CH;                      // chunks of CB bytes
            for (int i = gl; i < d * CH; i += g::G) {
              const int j = i / CH, c = i % CH;
              const uint8_t* src = X + (size_t)(e0 + j) * RS + c * CB;
              uint8_t* dst = stage + j * RS + c * CB;
              if constexpr (CB == 16) *reinterpret_cast<uint4*>(dst) = *reinterpret_cast<const uint4*>(src);
              else if constexpr (CB == 8) *reinterpret_cast<uint2*>(dst) = *reinterpret_cast<const uint2*>(src);
              else *reinterpret_cast<uint32_t*>(dst) = *reinterpret_cast<const uint32_t*>(src);
            }
          } else {
            for (int i = gl; i < d * Q; i += g::G) {
              const int j = i / Q, c = i % Q;
              const uint8_t* src = first ? gam + (size_t)edge_col[e0 + j] * Q : X + (size_t)(e0 + j) * Q;
              stage[i] = src[c];
            }
          }
          group_sync<g::G>(gmask);
          // permutation: P_j(y) = alpha_j(h_j^-1 y), 16-bit natural order
          for (int j = 0; j < d; ++j) {
            const int lhinv = edge_lhi[e0 + j];
            const uint8_t* a = stage + j * RS;
            const uint16_t* a16 = reinterpret_cast<const uint16_t*>(a);
            uint32_t* P = vec(j);
#pragma unroll
            for (int i = 0; i < PW; ++i) {
              const int w = gl + i * g::G;
              if (PW * g::G == g::W || w < g::W) {
                const int s0 = (py_nz0 >> i) & 1 ? exp2[((py_log0 >> (8 * i)) & 0xFF) + lhinv] : 0;
                const int s1 = exp2[((py_log1 >> (8 * i)) & 0xFF) + lhinv];
                if constexpr (MB == 2) P[w] = (uint32_t)a16[s0] | ((uint32_t)a16[s1] << 16);
                else P[w] = (uint32_t)a[s0] | ((uint32_t)a[s1] << 16);
              }
            }
          }
        }
        group_sync<g::G>(gmask);
        // beta_j(a) = R_j(h_j a), written over the edge's message row; the lane's
        // symbols are a0 + i (a0 = gl * BPL, i < BPL) and h (a0 + i) = h a0 ^ h i
        auto depermute = [=](const Sym* R16, int e) {
          const int lh = edge_lh[e];
          const int base = da_log0 >= 0 ? (int)exp2[da_log0 + lh] : 0;
          int hb[3] = {0, 0, 0};
#pragma unroll
          for (int b = 0; b < 3; ++b)
            if ((1 << b) < g::BPL) hb[b] = exp2[lh + b];
          int out[g::BPL];
#pragma unroll
          for (int i = 0; i < g::BPL; ++i)
            out[i] = R16[base ^ ((i & 1) ? hb[0] : 0) ^ ((i & 2) ? hb[1] : 0) ^ ((i & 4) ? hb[2] : 0)];
          if constexpr (MB == 2) {
            uint16_t* row = reinterpret_cast<uint16_t*>(X + (size_t)e * RS) + gl * g::BPL;
            if constexpr (g::BPL == 1) row[0] = (uint16_t)out[0];
            else store_u16<g::BPL>(row, out);
          } else {
            store_bytes<g::BPL>(X + (size_t)e * Q + gl * g::BPL, out);
          }
        };
        // forward: F_0 = P_0, F_j = F_{j-1} (*) P_j
        int fprev = 0;                                     // vector index of F_{j-1}
        for (int j = 1; j <= d - 2; ++j) {
          conv(vec(fprev), vec(j), vec16(vF + j), 0);
          group_sync<g::G>(gmask);
          fprev = vF + j;
        }
        depermute(vec16(fprev), e0 + d - 1);               // beta_{d-1} from F_{d-2}
        if constexpr (T1) {          // Table 1 schedule: F_{d-1} into the scratch vector, unused
          mm_conv<g, MB == 1>(vec(fprev), vec(d - 1), vec16(vR), cl, gmask);
          if (counting && gl == 0) work += (unsigned long long)Q * Q;
          group_sync<g::G>(gmask);
        }
        // backward: B_{d-1} = P_{d-1}; beta_j from F_{j-1} (*) B_{j+1}; B_j = B_{j+1} (*) P_j
        int bcur = d - 1;
        int pp = 0;
        for (int j = d - 2; j >= 1; --j) {
          const int fj = (j == 1) ? 0 : vF + j - 1;
          const int ro = PR ? fj : vR;
          conv(vec(fj), vec(bcur), vec16(ro), 2);
          group_sync<g::G>(gmask);
          depermute(vec16(ro), e0 + j);
          const int bn = PR ? j : vB + pp;
          conv(vec(bcur), vec(j), vec16(bn), 1);
          group_sync<g::G>(gmask);
          bcur = bn;
          pp ^= 1;
        }
        depermute(vec16(bcur), e0);                        // beta_0 from B_1
        if constexpr (T1)            // Table 1 schedule: B_0 into the scratch vector, unused
        {
          mm_conv<g, MB == 1>(vec(bcur), vec(0), vec16(vR), cl, gmask);
          if (counting && gl == 0) work += (unsigned long long)Q * Q;
        }
        group_sync<g::G>(gmask);
      }
    };

    // ---- check-node pass of a rank with at least two warps to a check (pruned, one warp
    // per convolution): the F chain on one warp and the B chain on the other, then each
    // every second middle beta, so that a check is 3/2 (d - 2) convolutions long and not
    // 3 (d - 2) (GF(256) (2,8) N=128, 17 frames: 889 us against 702).  P and F are in
    // the first warp's scratch, B in the second's.
    auto cnp_pair = [&](bool first) {
      if constexpr (PR && SP) {
        const int r = r_first + (grp >> 1), half = grp & 1;
        if (r >= r_last) return;
        auto pair_sync = [&]() { slot_sync(bar_id + 1 + (grp >> 1), 64); };
        const int e0 = row_ptr[r], d = row_ptr[r + 1] - e0;
        const int gb = group_scratch_bytes<Q>(job.dmax, 1, true);
        unsigned char* pf = scratch + (size_t)(grp & ~1) * gb;      // P_j, F_j
        unsigned char* pb = pf + gb;                                // B_j
        unsigned char* tmp = vecs + (size_t)(2 * dm - 2) * VB;      // this warp's
        auto depermute = [&](const Sym* R, int e) {                 // as in cnp: beta(a) = R(h a)
          const int lh = edge_lh[e], base = da_log0 >= 0 ? (int)exp2[da_log0 + lh] : 0;
          const int h1 = exp2[lh], h2 = exp2[lh + 1], h4 = exp2[lh + 2];
          int out[g::BPL];
#pragma unroll
          for (int i = 0; i < g::BPL; ++i)
            out[i] = R[base ^ ((i & 1) ? h1 : 0) ^ ((i & 2) ? h2 : 0) ^ ((i & 4) ? h4 : 0)];
          store_bytes<g::BPL>(X + (size_t)e * Q + gl * g::BPL, out);
        };
        auto at = [&](unsigned char* base, int i) { return reinterpret_cast<Sym*>(base + (size_t)i * VB); };
        auto convp = [&](const Sym* A, const Sym* B, Sym* C, int kind) {
          int folded = 0;
          tpred[kind] = pr_conv<g>(A, B, C, tmp, gl, tpred[kind], counting ? &folded : nullptr);
          if (counting && gl == 0) work += (unsigned long long)folded * Q;
          __syncwarp();
        };
        for (int c = gl + 32 * half; c < d * CH; c += 64) scatter_piece(first, e0, c, pf);
        pair_sync();
        if (half == 0) {
          const Sym* f = at(pf, 0);
          for (int j = 1; j <= d - 2; ++j) {
            convp(f, at(pf, j), at(pf, vF + j), 0);
            f = at(pf, vF + j);
          }
          depermute(f, e0 + d - 1);
        } else {
          const Sym* b = at(pf, d - 1);
          for (int j = d - 2; j >= 1; --j) {
            convp(b, at(pf, j), at(pb, j), 1);
            b = at(pb, j);
          }
          depermute(b, e0);
        }
        pair_sync();
        for (int j = 1 + half; j <= d - 2; j += 2) {
          Sym* f = at(pf, j == 1 ? 0 : vF + j - 1);
          convp(f, j == d - 2 ? at(pf, d - 1) : at(pb, j + 1), f, 2);
          depermute(f, e0 + j);
        }
      }
    };

    // ---- check-node pass for q = 4 in registers: one lane per check (checks of
    // degree <= kRegDeg).  A 4-symbol vector is two words of 16-bit values,
    // (v0, v1), (v2, v3); the coefficient permutations are byte permutes of the
    // 4-byte rows and the 16-pair convolutions use no shared memory, so the
    // pass has no memory round trip between its steps (at q = 4 the group form
    // is a chain of short shared-memory dependencies).
    constexpr int kRegDeg = 8;
    auto cnp_regs4 = [&](bool first) {
      // beta_e(a) = R(h a): byte a of the row from the 16-bit value R(i), i = h a, of the words R
      auto store_beta = [&](int e, uint2 R) {
        const int lh = edge_lh[e];
        const int i1 = exp2[lh], i2 = exp2[lh + 1], i3 = i1 ^ i2;
        const uint32_t sel = (uint32_t)((((i1 >> 1) << 2) | ((i1 & 1) << 1)) << 4) |
                             (uint32_t)((((i2 >> 1) << 2) | ((i2 & 1) << 1)) << 8) |
                             (uint32_t)((((i3 >> 1) << 2) | ((i3 & 1) << 1)) << 12);
        *reinterpret_cast<uint32_t*>(X + (size_t)e * 4) = __byte_perm(R.x, R.y, sel);
      };
      for (int r = r_first + stid; r < r_last; r += nthr) {
        const int e0 = row_ptr[r], d = row_ptr[r + 1] - e0;
        if (counting && d > 2) work += 16ull * 3 * (d - 2);
        // The last P and F are tracked as the loops run (Plast = P_{d-1}, Flast =
        // F_{d-2}): picking them out afterwards by "j == d - 1" turns into an indexed
        // access, which sends the arrays to local memory.
        uint2 P[kRegDeg], F[kRegDeg], Plast = make_uint2(0u, 0u);
#pragma unroll
        for (int j = 0; j < kRegDeg; ++j) {
          P[j] = make_uint2(0u, 0u);
          F[j] = make_uint2(0u, 0u);
          if (j < d) {
            // P_j(y) = alpha_j(h^-1 y): (alpha(0), alpha(h^-1)), (alpha(h^-1 2), alpha(h^-1 3))
            const int e = e0 + j;
            const uint32_t row = first ? *reinterpret_cast<const uint32_t*>(gam + (size_t)edge_col[e] * 4)
                                       : *reinterpret_cast<const uint32_t*>(X + (size_t)e * 4);
            const int lhinv = edge_lhi[e];
            const uint32_t s1 = exp2[lhinv], s2 = exp2[lhinv + 1], s3 = s1 ^ s2;
            P[j].x = __byte_perm(row, 0, 0x4040u | (s1 << 8));
            P[j].y = __byte_perm(row, 0, 0x4040u | s2 | (s3 << 8));
            Plast = P[j];
          }
        }
        // forward: F_0 = P_0, F_j = F_{j-1} (*) P_j; beta_{d-1} = F_{d-2}
        F[0] = P[0];
        uint2 Flast = F[0];
#pragma unroll
        for (int j = 1; j < kRegDeg - 1; ++j)
          if (j <= d - 2) {
            F[j] = conv4(F[j - 1], P[j]);
            Flast = F[j];
          }
        store_beta(e0 + d - 1, Flast);
        // backward: B_{d-1} = P_{d-1}; beta_j = F_{j-1} (*) B_{j+1}; B_j = B_{j+1} (*) P_j; beta_0 = B_1
        uint2 Bc = Plast;
#pragma unroll
        for (int j = kRegDeg - 2; j >= 1; --j) {
          if (j <= d - 2) {
            store_beta(e0 + j, conv4(F[j - 1], Bc));
            Bc = conv4(Bc, P[j]);
          }
        }
        store_beta(e0, Bc);
      }
    };

    // ---- check-node pass for q = 8, 16, 32 in registers: one lane per check of any
    // degree.  The lane reads an edge's row when it needs P_j (beta_j overwrites it only
    // after that) and parks F_1..F_{d-3} as bytes in the slot's shared scratch.  At q = 32
    // beta_j and B_j share one convolution's code: with three in line, frames in different
    // passes evicted each other's instructions (N=96: no_instruction 2.3 stalls per issue,
    // 3.33 ms against 2.91; with a single one for F_j too, N=600 was 5 % slower).
    auto cnp_reg = [&](bool first) {
      if constexpr (reg_form<Q>()) {
        constexpr int W = Q / 2, NB = Q / 4;
        const uint8_t* perm = sblob + job.perm_at;
        auto load_p = [&](int e, uint32_t (&P)[W]) {       // P_j(y) = alpha_j(h^-1 y)
          uint32_t r[NB], o[NB];
          load_row<Q>(first ? gam + (size_t)edge_col[e] * Q : X + (size_t)e * Q, r);
          gather_row<Q>(r, o, perm + edge_lhi[e] * PermRow<Q>::bytes);
          unpack_row<NB>(o, P);
        };
        auto store_packed = [&](int e, const uint32_t (&r)[NB]) {   // beta_j(a) = R(h a)
          uint32_t o[NB];
          gather_row<Q>(r, o, perm + edge_lh[e] * PermRow<Q>::bytes);
          store_row<Q>(X + (size_t)e * Q, o);
        };
        auto store_beta = [&](int e, const uint32_t (&R)[W]) {
          uint32_t r[NB];
          pack_row<NB>(R, r);
          store_packed(e, r);
        };
        // (a stride from the job costs up to 10 % where the pass is short: GF(16) N=64, 9,000 frames
        // 330 us against 300, so launches with all lanes have a kernel without it)
        const int lanes = D < 0 ? job.reg : nthr;
        if (D < 0 && stid >= lanes) return;
        uint8_t* fs = scratch + (size_t)stid * Q;                // F_j of this lane: fs + (j - 1) * lanes * Q
        for (int r = r_first + stid; r < r_last; r += lanes) {
          const int e0 = row_ptr[r], d = D > 0 ? D : row_ptr[r + 1] - e0;
          if (counting && d > 2) work += (unsigned long long)Q * Q * 3 * (d - 2);
          uint32_t a[W], b[W], c[W];
          // forward: F_0 = P_0, F_j = F_{j-1} (*) P_j
          load_p(e0, a);
#pragma unroll 1
          for (int j = 1; j <= d - 2; ++j) {
            load_p(e0 + j, b);
            conv_reg<W>(a, b, c);
            if (j <= d - 3) {
              uint32_t f[NB];
              pack_row<NB>(c, f);
              store_row<Q>(fs + (size_t)(j - 1) * lanes * Q, f);
            }
#pragma unroll
            for (int w = 0; w < W; ++w) a[w] = c[w];
          }
          load_p(e0 + d - 1, b);                                 // B_{d-1} = P_{d-1}
          store_beta(e0 + d - 1, a);                             // beta_{d-1} = F_{d-2}
          // backward: beta_j = F_{j-1} (*) B_{j+1}, B_j = B_{j+1} (*) P_j
#pragma unroll 1
          for (int j = d - 2; j >= 1; --j) {
            if (j == 1) {
              load_p(e0, a);
            } else {
              uint32_t f[NB];
              load_row<Q>(fs + (size_t)(j - 2) * lanes * Q, f);
              unpack_row<NB>(f, a);
            }
            uint32_t be[NB];
#pragma unroll(W >= 16 ? 1 : 2)
            for (int s = 0; s < 2; ++s) {
              if (s) {
                load_p(e0 + j, a);
                store_packed(e0 + j, be);
              }
              conv_reg<W>(b, a, c);
              if (!s) pack_row<NB>(c, be);
            }
#pragma unroll
            for (int w = 0; w < W; ++w) b[w] = c[w];
          }
          store_beta(e0, b);                                     // beta_0 = B_1
        }
      }
    };

    // ---- decode one frame.  Without early stop only the final decision is
    // tested, so the stop test runs once, after the last iteration.
    const bool es = job.early_stop != 0;
    if constexpr (MB == 2) vnp_wide(true, false); else vnp(true, false);   // c^(0) = argmin gamma
    pass_sync();
    bool ok = (es || job.max_iters == 0) ? syndrome_ok() : false;
    int iters = 0;
    if (!(es && ok)) {
      if constexpr (MB == 2 && !kScatter) {
        init_wide();
        pass_sync();
      }
      for (int k = 1; k <= job.max_iters; ++k) {
        if constexpr (Q == 4 && MB == 1 && !T1) {
          if (job.dmax <= kRegDeg) cnp_regs4(k == 1); else cnp(k == 1);
        } else if constexpr (reg_form<Q>() && MB == 1 && !T1 && W4) {
          cnp_reg(k == 1);
        } else if constexpr (PR && SP) {
          if (2 * (r_last - r_first) <= ngroups) cnp_pair(k == 1); else cnp(k == 1);
        } else {
          cnp((MB == 1 || kScatter) && k == 1);
        }
        pass_sync();
        if constexpr (MB == 2) vnp_wide(false, k < job.max_iters); else vnp(false, k < job.max_iters);
        pass_sync();
        iters = k;
        if (es || k == job.max_iters) ok = syndrome_ok();
        if (es && ok) break;
      }
    }
    for (int i = n_first + stid; i < n_last; i += nthr) job.out_sym[(size_t)frame * job.n + i] = chat[i];
    if (counting && work) atomicAdd(job.work, work);
    if (stid == 0 && (!SP || sc->rank == 0)) {
      job.out_iters[frame] = iters;
      job.out_ok[frame] = ok ? 1 : 0;
    }
}

// ---------------------------------------------------------------- the kernel
// Persistent blocks of fpb frame slots; every slot takes work items (a frame
// of one job) from a global counter until the list is exhausted.  QSEL = q,
// VSEL = variant compiles the path of one field order and layout (single-code
// launches); QSEL = 0, VSEL = -1 or -2 compiles every field order (mixed-code launches).
// Resident 256-thread blocks per SM the register allocation must allow: the
// q >= 128 paths need more than 85 registers per thread without spilling.
#ifndef NBLDPC_MINB_64
#define NBLDPC_MINB_64 4
#endif
#ifndef NBLDPC_MINB_WIDE
#define NBLDPC_MINB_WIDE 2
#endif
// The pruned kernels fit 80 registers without spilling: three 256-thread blocks
// per SM hide more of their shuffle and shared-memory latency (GF(256) (2,6)
// N=384: 119.8 ms at two blocks, 103.8 at three, 106.5 at four).
#ifndef NBLDPC_MINB_PRUNE
#define NBLDPC_MINB_PRUNE 3
#endif
// The mixed-code kernel (QSEL = 0) has no dense q >= 128 path and comes in two forms: VSEL = -1
// for batches that fill the chip, three blocks at 80 registers with a function per field order,
// VSEL = -2 for the others, two blocks with every path in line.
template <int QSEL, int VSEL> struct MinBlocks {
  static constexpr int v = QSEL == 0 ? (VSEL == -2 ? 2 : 3) : QSEL >= 128 ? NBLDPC_MINB_WIDE
                         : (QSEL == 64 ? (VSEL == 1 ? 3 : NBLDPC_MINB_64) : 4);
};

// The mixed-code kernels' form of field order Q: the default layout, with pruned
// convolutions for q >= 128; SP: the split-frame kernel's.
template <int Q> __host__ __device__ constexpr int mixed_layout() { return Q >= 16 && Q <= 64 ? 1 : 0; }

// Where a frame slot of a mixed-code launch keeps its things in shared memory (byte
// offsets); X: its message area there (SP), else its global slot.
struct MixedSlot {
  int job, blob, chat, scratch, x, sc;
  uint8_t* X;
};

// It takes offsets, so that its accesses are shared-memory ones.
template <int Q, bool REG, bool SP, int D>
__device__ __forceinline__ void decode_mixed_inline(const MixedSlot& m, int frame, int stid, int nthr, int bar_id) {
  extern __shared__ __align__(16) unsigned char smem[];
  const JobDesc& job = *reinterpret_cast<const JobDesc*>(smem + m.job);
  uint8_t* X = SP ? smem + m.x : m.X;
  decode_frame<Geo<Q, mixed_layout<Q>()>, 1, false, (Q >= 128), REG, D, SP>(
      job, frame, X, smem + m.blob, SP ? smem + m.blob : job.blob, smem + m.chat, smem + m.scratch, stid, nthr, bar_id,
      reinterpret_cast<const SplitCtx*>(smem + m.sc));
}

// As a function: at 80 registers, in line, the persistent kernel's frame loop kept a dozen registers
// across every path and the paths spilled.  A call costs 5 to 30 % of a frame's time, also without a
// spill: us per iteration of 20 frames, as a function and in line at 128 registers: GF(8) N=100 3.0
// and 2.4, GF(32) N=64 4.6 and 3.9, GF(64) N=576 69 and 65, GF(128) N=256 171 and 127, GF(256) (2,8)
// N=128 132 and 107.
template <int Q, bool REG, bool SP, int D>
__device__ __noinline__ void decode_mixed_call(MixedSlot m, int frame, int stid, int nthr, int bar_id) {
  decode_mixed_inline<Q, REG, SP, D>(m, frame, stid, nthr, bar_id);
}

template <bool CALL, int Q, bool REG, bool SP, int D = 0>
__device__ __forceinline__ void decode_mixed(const MixedSlot& m, int frame, int stid, int nthr, int bar_id) {
  if constexpr (CALL) decode_mixed_call<Q, REG, SP, D>(m, frame, stid, nthr, bar_id);
  else decode_mixed_inline<Q, REG, SP, D>(m, frame, stid, nthr, bar_id);
}

template <bool SP, bool CALL>
__device__ __forceinline__ void decode_any(const JobDesc& job, const MixedSlot& m, int frame, int stid, int nthr,
                                           int bar_id) {
  if constexpr (!SP) {
    if (job.reg) {
      if (job.q == 64) decode_mixed<CALL, 64, false, SP, 4>(m, frame, stid, nthr, bar_id);
      else if (job.q == 8) decode_mixed<CALL, 8, true, SP>(m, frame, stid, nthr, bar_id);
      else if (job.q == 16) decode_mixed<CALL, 16, true, SP>(m, frame, stid, nthr, bar_id);
      else decode_mixed<CALL, 32, true, SP>(m, frame, stid, nthr, bar_id);
      return;
    }
  }
  switch (job.q) {
    case 2: decode_mixed<CALL, 2, false, SP>(m, frame, stid, nthr, bar_id); break;
    case 4: decode_mixed<CALL, 4, !SP, SP>(m, frame, stid, nthr, bar_id); break;
    case 8: decode_mixed<CALL, 8, false, SP>(m, frame, stid, nthr, bar_id); break;
    case 16: decode_mixed<CALL, 16, false, SP>(m, frame, stid, nthr, bar_id); break;
    case 32: decode_mixed<CALL, 32, false, SP>(m, frame, stid, nthr, bar_id); break;
    case 64: decode_mixed<CALL, 64, false, SP>(m, frame, stid, nthr, bar_id); break;
    case 128: decode_mixed<CALL, 128, false, SP>(m, frame, stid, nthr, bar_id); break;
    default: decode_mixed<CALL, 256, false, SP>(m, frame, stid, nthr, bar_id); break;
  }
}

// MB: message bytes per symbol (1: 8-bit messages; 2: 16-bit, single-field kernels only).
// T1: the Table 1 check-node schedule (3 d_c - 4 convolutions; single-field kernels only).
// XS: the frames' messages stay in shared memory (8-bit messages, single-field
// kernels; at most kResidentThreads threads, see make_plan).
// PR: pruned check-node convolutions (single-field kernels whose layout has
// 32-lane groups; 8-bit messages, minimal schedule).  D > 0: every check has
// degree D (single-field kernels; see decode_frame).  QSEL = 4, D = -1 or -4: the one-warp form alone,
// for codes that it serves in slots of 32 threads (-4: every check of degree 4).  A kernel of its own:
// beside the other forms a 1,000-frame decode of N=48 took 7.8 us, 7.4 alone.
template <int QSEL, int VSEL, int MB, bool T1 = false, bool XS = false, bool PR = false, int D = 0>
__global__ void __launch_bounds__(XS ? kResidentThreads : 256, XS ? 2 : PR ? NBLDPC_MINB_PRUNE : MinBlocks<QSEL, VSEL>::v)
    mma_decode_kernel(const __grid_constant__ LaunchParams<QSEL> p) {
  static_assert(!XS || (QSEL >= 2 && MB == 1 && !T1), "resident messages: 8-bit, minimal schedule, one field");
  static_assert(!PR || (QSEL >= 2 && MB == 1 && !T1), "pruned convolutions: 8-bit, minimal schedule, one field");
  extern __shared__ __align__(16) unsigned char smem[];
  const int nthr = blockDim.x / p.fpb;
  const int slot = threadIdx.x / nthr, stid = threadIdx.x % nthr;
  const int bar_id = 1 + slot;
  unsigned char* base = smem + (size_t)slot * p.slot_smem;
  unsigned char* sblob = base;
  uint8_t* chat = base + p.blob_cap;
  volatile int* ctl = reinterpret_cast<volatile int*>(base + p.blob_cap + p.n_cap);
  constexpr int kCtl = ctl_bytes(QSEL);
  constexpr bool kW4 = QSEL == 4 && D < 0;
  unsigned char* scratch = base + p.blob_cap + p.n_cap + kCtl;
  JobDesc* sjob = reinterpret_cast<JobDesc*>(base + p.blob_cap + p.n_cap + 16);   // (QSEL = 0)
  uint8_t* X = XS ? base + p.xs_off : p.msg + ((size_t)blockIdx.x * p.fpb + slot) * p.slot_bytes;
  int staged = -1;

  // a launch with no more items than frame slots assigns them statically (the
  // host then skips the counter reset)
  int static_item = p.static_items ? (int)blockIdx.x * p.fpb + slot : -1;
  for (;;) {
    if (stid == 0) ctl[0] = static_item >= 0 ? static_item : (int)atomicAdd(p.counter, 1u);
    if (static_item >= 0) static_item = p.total_items;
    slot_sync(bar_id, nthr);
    const int item = ctl[0];
    if (item >= p.total_items) break;
    int j = 0;
    if constexpr (QSEL == 0)
      while (j + 1 < p.njobs && item >= p.jobs[j + 1].item_begin) ++j;
    // single-field launches carry one job: static parameter offsets
    const JobDesc& job = (QSEL == 0) ? p.jobs[j] : p.jobs[0];
    const int frame = item - job.item_begin;
    if (j != staged) {      // stage the code description (GF tables, H, variable-node view)
      stage_blob(sblob, job, job.perm_at, QSEL == 0 ? job.reg != 0 : XS && reg_form<QSEL>(), stid, nthr);
      if constexpr (QSEL == 0) {
        for (int i = stid; i < (int)(sizeof(JobDesc) / 4); i += nthr)
          reinterpret_cast<uint32_t*>(sjob)[i] = reinterpret_cast<const uint32_t*>(&job)[i];
      }
      staged = j;
      slot_sync(bar_id, nthr);
    }
    if constexpr (kW4)
      decode_frame_warp4<D == -4 ? 4 : 0>(job, frame, X, sblob, sblob, stid);
    else if constexpr (QSEL != 0)
      decode_frame<Geo<QSEL, VSEL>, MB, T1, PR, XS && QSEL != 4, D>(job, frame, X, sblob, sblob, chat, scratch, stid, nthr,
                                                                    bar_id);
    else
      decode_any<false, VSEL == -1>(*sjob,
                        MixedSlot{(int)(reinterpret_cast<unsigned char*>(sjob) - smem), (int)(sblob - smem),
                                  (int)(chat - smem), (int)(scratch - smem), 0, 0, X},
                        frame, stid, nthr, bar_id);
    slot_sync(bar_id, nthr);
  }
}

// ---------------------------------------------------------------- the kernels of split frames
// One cluster per frame (grid: frames * cluster size).  Shared memory of a rank:
// code blob | decisions (indexed by column) | flags | row table | reliabilities of
// its columns | check-node scratch | message rows of its edges.
struct SplitLayout {
  int cpc, npc;               // checks and columns per rank
  int chat_off, flag_off, row_off, gam_off, scratch_off, x_off;
};
struct SplitParams {          // one code
  JobDesc job;
  int size;                   // ranks per frame
  SplitLayout lay;
};
struct SplitBatchParams {     // mixed codes; the jobs' frames form one list
  JobDesc jobs[kMaxJobs];
  SplitLayout lay[kMaxJobs];
  int njobs, size;
  int job_off, sc_off;        // the rank's copies of its job and SplitCtx in shared memory
};

// Set up this rank of a frame's cluster (code description, reliabilities, row table); rs:
// bytes of a message row.
__device__ __forceinline__ void split_setup(const JobDesc& job, const SplitLayout& p, int frame, int rank, int size,
                                            int q, int rs, unsigned char* smem, SplitCtx& sc) {
  const int tid = threadIdx.x, nthr = blockDim.x;
  stage_blob(smem, job, job.off.perm, false, tid, nthr);
  sc.rank = rank;
  sc.size = size;
  sc.r0 = min(rank * p.cpc, job.m);
  sc.r1 = min(sc.r0 + p.cpc, job.m);
  sc.n0 = min(rank * p.npc, job.n);
  sc.n1 = min(sc.n0 + p.npc, job.n);
  sc.npc = p.npc;
  sc.flags = reinterpret_cast<int*>(smem + p.flag_off);
  uint8_t** vrow = reinterpret_cast<uint8_t**>(smem + p.row_off);
  sc.vrow = vrow;
  uint8_t* sgam = smem + p.gam_off;
  sc.gam = sgam;
  const uint8_t* src = job.gamma + ((size_t)frame * job.n + sc.n0) * q;   // (gamma is 16-byte aligned)
  const int bytes = (sc.n1 - sc.n0) * q;
  if (q >= 16) {
    for (int i = tid; i < bytes / 16; i += nthr)
      reinterpret_cast<uint4*>(sgam)[i] = reinterpret_cast<const uint4*>(src)[i];
  } else {
    for (int i = tid; i < bytes / 2; i += nthr)
      reinterpret_cast<uint16_t*>(sgam)[i] = reinterpret_cast<const uint16_t*>(src)[i];
  }
  __syncthreads();
  const uint16_t* row_ptr = reinterpret_cast<const uint16_t*>(smem + job.off.row_ptr);
  const uint16_t* vn_ptr = reinterpret_cast<const uint16_t*>(smem + job.off.vn_ptr);
  const uint16_t* vn_edge = reinterpret_cast<const uint16_t*>(smem + job.off.vn_edge);
  const uint16_t* edge_row = reinterpret_cast<const uint16_t*>(job.blob + job.off.edge_row);
  sc.e0 = row_ptr[sc.r0];
  uint8_t* X = smem + p.x_off;
  for (int k = vn_ptr[sc.n0] + tid; k < vn_ptr[sc.n1]; k += nthr) {
    const int e = vn_edge[k], owner = edge_row[e] / p.cpc;
    vrow[k - vn_ptr[sc.n0]] = at_rank(X, owner) + (size_t)(e - row_ptr[owner * p.cpc]) * rs;
  }
  cluster_barrier();           // the row table is complete, and every rank of the cluster runs
}

// D: as in decode_frame.
template <int Q, int V, int MB, bool PR, int D = 0>
__global__ void __launch_bounds__(kResidentThreads, 2) mma_split_kernel(const __grid_constant__ SplitParams p) {
  extern __shared__ __align__(16) unsigned char smem[];
  const int rank = blockIdx.x % p.size, frame = blockIdx.x / p.size;
  SplitCtx sc;
  split_setup(p.job, p.lay, frame, rank, p.size, Q, Q * MB, smem, sc);
  decode_frame<Geo<Q, V>, MB, false, PR, false, D, true>(p.job, frame, smem + p.lay.x_off, smem, smem,
                                                               smem + p.lay.chat_off, smem + p.lay.scratch_off,
                                                               threadIdx.x, blockDim.x, 1, &sc);
}

// 8-bit messages, minimal schedule.  (A template, so that only the mixed-code unit compiles it.)
template <int QSEL>
__global__ void __launch_bounds__(kResidentThreads, 2) mma_split_batch_kernel(const __grid_constant__ SplitBatchParams p) {
  extern __shared__ __align__(16) unsigned char smem[];
  const int rank = blockIdx.x % p.size, item = blockIdx.x / p.size;
  int j = 0;
  while (j + 1 < p.njobs && item >= p.jobs[j + 1].item_begin) ++j;
  const JobDesc& job = p.jobs[j];
  const SplitLayout& lay = p.lay[j];
  const int frame = item - job.item_begin;
  JobDesc* sjob = reinterpret_cast<JobDesc*>(smem + p.job_off);
  for (int i = threadIdx.x; i < (int)(sizeof(JobDesc) / 4); i += blockDim.x)
    reinterpret_cast<uint32_t*>(sjob)[i] = reinterpret_cast<const uint32_t*>(&job)[i];
  SplitCtx sc;
  split_setup(job, lay, frame, rank, p.size, job.q, job.q, smem, sc);
  if (threadIdx.x == 0) *reinterpret_cast<SplitCtx*>(smem + p.sc_off) = sc;
  __syncthreads();
  decode_any<true, true>(*sjob, MixedSlot{p.job_off, 0, lay.chat_off, lay.scratch_off, lay.x_off, p.sc_off, nullptr}, frame,
                   threadIdx.x, blockDim.x, 1);
}

}  // namespace nbldpc

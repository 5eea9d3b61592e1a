// One translation unit per kernel family, so the field orders compile in
// parallel: built with -DNBLDPC_KQ=q for the two layout variants of field
// order q (single-code launches), or -DNBLDPC_KQ=0 for the kernels that
// serve every field order (mixed-code launches; with -DNBLDPC_MIXED_WIDE the one
// for batches that do not fill the chip).
#include "mma_kernels.cuh"

#ifndef NBLDPC_KQ
#error "NBLDPC_KQ must name the field order (or 0)"
#endif

#define NBLDPC_CAT2(a, b) a##b
#define NBLDPC_CAT(a, b) NBLDPC_CAT2(a, b)

namespace nbldpc {

// pruned-convolution kernel of one layout, if that layout has 32-lane groups
// (a template, so that the layouts without them are never instantiated)
template <int Q> const void* pruned_kernel(int layout) {
  if constexpr (Geo<Q, 0>::G == 32)
    if (layout == 0) return reinterpret_cast<const void*>(&mma_decode_kernel<Q, 0, 1, false, false, true>);
  if constexpr (Geo<Q, 1>::G == 32)
    if (layout == 1) return reinterpret_cast<const void*>(&mma_decode_kernel<Q, 1, 1, false, false, true>);
  return nullptr;
}

#ifdef NBLDPC_MIXED_WIDE
// Address of the mixed-code kernel for batches that do not fill the chip (two blocks an SM).
const void* kernel_q0_wide() { return reinterpret_cast<const void*>(&mma_decode_kernel<0, -2, 1>); }
#else
// Address of the decode kernel for variant v (bit 0: layout; bit 1: messages
// resident in shared memory; bit 2: pruned convolutions, layouts of 32-lane
// groups only, not with bit 1), mb-byte messages and the check-node schedule t1
// (1: Table 1's 3 d_c - 4 convolutions, 8-bit messages only) of this unit's
// field order; dreg: the code's check degree when all are equal (GF(4) and
// GF(64) have resident-message kernels for degree 4), else 0, or -1 for the register form
// with fewer lanes than threads, -1 or -4 for GF(4) codes that a warp decodes alone; null
// when there is none.
const void* NBLDPC_CAT(kernel_q, NBLDPC_KQ)(int v, int mb, int t1, int dreg) {
  (void)dreg;
#if NBLDPC_KQ == 0
  (void)v;
  return (mb == 1 && !t1) ? reinterpret_cast<const void*>(&mma_decode_kernel<0, -1, 1>) : nullptr;
#else
  if (v & 4) {
    if (mb != 1 || t1 || (v & 2)) return nullptr;
    return pruned_kernel<NBLDPC_KQ>(v & 1);
  }
  if (v >= 2) {
    if (mb != 1 || t1) return nullptr;
#if NBLDPC_KQ == 4
    if (dreg < 0)    // the one-warp form alone
      return dreg == -4 ? reinterpret_cast<const void*>(&mma_decode_kernel<4, 0, 1, false, true, false, -4>)
                        : reinterpret_cast<const void*>(&mma_decode_kernel<4, 0, 1, false, true, false, -1>);
#endif
#if NBLDPC_KQ == 64 || NBLDPC_KQ == 4
    // every check of degree 4 (the regular (2,4) codes): a compile-time check degree
    if (dreg == 4)
      return (v & 1) ? reinterpret_cast<const void*>(&mma_decode_kernel<NBLDPC_KQ, 1, 1, false, true, false, 4>)
                     : reinterpret_cast<const void*>(&mma_decode_kernel<NBLDPC_KQ, 0, 1, false, true, false, 4>);
#endif
#if NBLDPC_KQ == 8 || NBLDPC_KQ == 16 || NBLDPC_KQ == 32
    // (one lane per check: the layouts of the group form do not differ here)
    return dreg < 0 ? reinterpret_cast<const void*>(&mma_decode_kernel<NBLDPC_KQ, 0, 1, false, true, false, -1>)
                    : reinterpret_cast<const void*>(&mma_decode_kernel<NBLDPC_KQ, 0, 1, false, true>);
#else
    return (v & 1) ? reinterpret_cast<const void*>(&mma_decode_kernel<NBLDPC_KQ, 1, 1, false, true>)
                   : reinterpret_cast<const void*>(&mma_decode_kernel<NBLDPC_KQ, 0, 1, false, true>);
#endif
  }
  if (t1) {
    if (mb != 1) return nullptr;
    return v ? reinterpret_cast<const void*>(&mma_decode_kernel<NBLDPC_KQ, 1, 1, true>)
             : reinterpret_cast<const void*>(&mma_decode_kernel<NBLDPC_KQ, 0, 1, true>);
  }
  if (mb == 2)
    return v ? reinterpret_cast<const void*>(&mma_decode_kernel<NBLDPC_KQ, 1, 2>)
             : reinterpret_cast<const void*>(&mma_decode_kernel<NBLDPC_KQ, 0, 2>);
  return v ? reinterpret_cast<const void*>(&mma_decode_kernel<NBLDPC_KQ, 1, 1>)
           : reinterpret_cast<const void*>(&mma_decode_kernel<NBLDPC_KQ, 0, 1>);
#endif
}

#if NBLDPC_KQ == 0
// Address of the mixed-code kernel that decodes each frame on a cluster of blocks.
const void* split_kernel_q0() { return reinterpret_cast<const void*>(&mma_split_batch_kernel<0>); }
#endif

#if NBLDPC_KQ >= 8
// Address of the kernel that decodes a frame on a cluster of blocks, for mb-byte
// messages (minimal schedule): the layout and the convolutions of the default variant
// (GF(8): 16-bit messages only); dreg as in kernel_q (GF(64), degree 4).
const void* NBLDPC_CAT(split_kernel_q, NBLDPC_KQ)(int mb, int dreg) {
  (void)dreg;
  constexpr int Q = NBLDPC_KQ, V = (Q >= 16 && Q <= 64) ? 1 : 0;
  if (mb == 2) return reinterpret_cast<const void*>(&mma_split_kernel<Q, V, 2, false>);
#if NBLDPC_KQ == 64
  if (dreg == 4) return reinterpret_cast<const void*>(&mma_split_kernel<Q, V, 1, false, 4>);
#endif
#if NBLDPC_KQ == 8
  return nullptr;
#else
  return reinterpret_cast<const void*>(&mma_split_kernel<Q, V, 1, (Q >= 128)>);
#endif
}
#endif
#endif  // NBLDPC_MIXED_WIDE

}  // namespace nbldpc

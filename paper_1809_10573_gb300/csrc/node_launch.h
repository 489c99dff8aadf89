// Host-side launch rules shared by the per-level node kernels (node.cu) and the batch (batch.cu).
#pragma once

#include <cuda_runtime.h>

#include <algorithm>

#include "idbf_internal.h"

namespace idbf {
namespace node {

inline int num_sms() {
  int dev = 0, sms = 152;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  return sms;
}

// Slices per node: levels of few nodes are cut until the grid holds about `per_sm` CTAs per SM, in
// slices of at least 16 rows (or columns).
inline int slices(int64_t ctas, int span, int per_sm) {
  const int64_t want = (int64_t)per_sm * num_sms();
  const int64_t n = (want + ctas - 1) / ctas;
  return (int)std::max<int64_t>(1, std::min<int64_t>(std::min<int64_t>(n, 8), span / 16));
}

// what a forward node of a level is cut by: rows of its blocks (V, S) or output positions (U)
inline int fwd_span(const LevelInfo& li) { return li.kind == KIND_U ? li.max_out : li.max_rows_pair; }

// Threads of a forward CTA, TR rows per thread: one row tile per thread in the tallest node; shorter ones split their columns (sized by the mean
// node instead, the nodes of a level differing several times over, the double-float apply of one
// vector takes 865 against 691 us for the FIO at N = 2^16; with twice the threads, more nodes wait:
// NUFFT N = 100003, 9 vectors, 2365 against 1796 us)
inline int fwd_threads(const LevelInfo& li, int TR, int nsl, int ntmax) {
  const int nt = ((li.max_rows_pair / nsl + TR - 1) / TR + 31) / 32 * 32;
  return std::max(nsl > 1 ? std::min(256, ntmax) : 64, std::min(ntmax, nt));
}

// The fewest right-hand-side blocks of at most `cap` columns, as even as possible: block width.
inline int even_block(int64_t R, int cap) {
  const int64_t nblk = (R + cap - 1) / cap;
  return (int)((R + nblk - 1) / nblk);
}

// FP64's block width, 3, 4, 5 or 7 (or R): the FP64 pipe is the bound, so the fewest right-hand sides
// past R are computed, and of those widths the narrowest, whose more numerous CTAs balance better over
// the SMs (NUFFT N = 30011, 18 vectors: 2.61 ms with 3, 2.88 with 6; the factors' re-reads come from L2).
// Blocks of 6 and 8 fit nothing that blocks of 3 and 4 do not.
inline int fitting_block(int64_t R) {
  if (R <= 3) return (int)R;
  int best = 3;
  for (const int w : {4, 5, 7})
    if (w <= R && (R + w - 1) / w * w < (R + best - 1) / best * best) best = w;
  return best;
}

// Launch on a stream whose previous launch was a level kernel of the same apply (after): the
// grid may begin while that one drains (programmatic dependent launch); else an ordinary launch.
template <class... A>
cudaError_t launch_after(void (*kern)(A...), bool after, int64_t grid, int nt, size_t sm, cudaStream_t st, A... args) {
  cudaLaunchConfig_t c = {};
  c.gridDim = dim3((unsigned)grid);
  c.blockDim = dim3((unsigned)nt);
  c.dynamicSmemBytes = sm;
  c.stream = st;
  cudaLaunchAttribute at;
  at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at.val.programmaticStreamSerializationAllowed = 1;
  c.attrs = &at;
  c.numAttrs = after ? 1 : 0;
  return cudaLaunchKernelEx(&c, kern, args...);
}

}  // namespace node
}  // namespace idbf

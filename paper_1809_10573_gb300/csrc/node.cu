// Launches of the node kernels (node_kernels.cuh): one butterfly level, forward or adjoint, for
// any number of right-hand sides in every CUDA-core arithmetic.
#include <cuda_runtime.h>

#include <algorithm>

#include "idbf_internal.h"
#include "node_kernels.cuh"

namespace idbf {
namespace node {

// The right-hand-side blocks of a slice are adjacent CTAs, so that their reads of the factors meet
// in L2; with a single block the factors are read once and marked for early eviction.
template <class P, int RB, int TR, int U, int NTMAX, int MINB, bool STREAM>
__global__ void __launch_bounds__(NTMAX, MINB)
    k_node_fwd(DevLevel d, const typename P::mat_t* __restrict__ mat, IO<typename P::vec_t> io, int max_in, int max_out,
               int max_rows, int max_cols, int max_rows_pair, int nblk, int nsl) {
  extern __shared__ __align__(16) unsigned char smem[];
  const unsigned unit = blockIdx.x / (unsigned)nblk;
  fwd_body<P, RB, TR, U, STREAM>(d, mat, io, max_in, max_out, max_rows, max_cols, max_rows_pair,
                                 (int64_t)(unit / (unsigned)nsl), (int)(unit % (unsigned)nsl), nsl,
                                 (int)(blockIdx.x % (unsigned)nblk) * RB, smem);
}

template <class P, int RB, int TC, int LR, int U, int NTMAX, int MINB, bool STREAM>
__global__ void __launch_bounds__(NTMAX, MINB)
    k_node_adj(DevLevel d, const typename P::mat_t* __restrict__ mat, IO<typename P::vec_t> io, int max_in, int max_out,
               int max_rows, int max_cols_pair, int nblk, int nsl) {
  extern __shared__ __align__(16) unsigned char smem[];
  const unsigned unit = blockIdx.x / (unsigned)nblk;
  adj_body<P, RB, TC, LR, U, STREAM>(d, mat, io, max_in, max_out, max_rows, max_cols_pair,
                                     (int64_t)(unit / (unsigned)nsl), (int)(unit % (unsigned)nsl), nsl,
                                     (int)(blockIdx.x % (unsigned)nblk) * RB, smem);
}

static int num_sms() {
  int dev = 0, sms = 152;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  return sms;
}

// Slices per node: levels of few nodes are cut until the grid holds about four CTAs per SM, in
// slices of at least 16 rows (or columns).
static int slices(int64_t ctas, int span) {
  const int64_t want = 4ll * num_sms();
  const int64_t n = (want + ctas - 1) / ctas;
  return (int)std::max<int64_t>(1, std::min<int64_t>(std::min<int64_t>(n, 8), span / 16));
}

static constexpr size_t kSmemCap = 220 * 1024;

template <class P, int RB, int TR, int U, int NTMAX, int MINB>
static idbf_status fwd_launch(Plan* p, int l, const void* mat, const IO<typename P::vec_t>& io, cudaStream_t st) {
  const LevelInfo& li = p->lv[l];
  const size_t sm = fwd_smem<P, RB>(li.max_in, li.max_out, li.max_rows, li.max_cols, li.max_rows_pair, li.kind == KIND_U);
  if (sm > kSmemCap) return IDBF_EUNSUPPORTED;
  const int nblk = (io.R + RB - 1) / RB;
  const int nsl = slices((int64_t)p->m * nblk, li.kind == KIND_U ? li.max_out : li.max_rows_pair);
  // one row tile per thread in the tallest node; shorter ones split their columns
  int nt = ((li.max_rows_pair / nsl + TR - 1) / TR + 31) / 32 * 32;
  nt = std::max(nsl > 1 ? std::min(256, NTMAX) : 64, std::min(NTMAX, nt));
  auto go = [&](auto kern) -> idbf_status {
    if (sm > 48 * 1024) IDBF_CUDA_TRY(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm));
    kern<<<(unsigned)((int64_t)p->m * nsl * nblk), nt, sm, st>>>(p->level(l), (const typename P::mat_t*)mat, io, li.max_in,
                                                                li.max_out, li.max_rows, li.max_cols, li.max_rows_pair,
                                                                nblk, nsl);
    IDBF_CUDA_TRY(cudaGetLastError());
    return IDBF_OK;
  };
  return nblk == 1 ? go(k_node_fwd<P, RB, TR, U, NTMAX, MINB, true>) : go(k_node_fwd<P, RB, TR, U, NTMAX, MINB, false>);
}

template <class P, int RB, int TC, int LR, int U, int NTMAX, int MINB>
static idbf_status adj_launch(Plan* p, int l, const void* mat, const IO<typename P::vec_t>& io, cudaStream_t st) {
  const LevelInfo& li = p->lv[l];
  const size_t sm = adj_smem<P, RB>(li.max_in, li.max_out, li.max_rows, li.max_cols_pair, li.kind == KIND_V);
  if (sm > kSmemCap) return IDBF_EUNSUPPORTED;
  const int nblk = (io.R + RB - 1) / RB;
  const int cols = li.kind == KIND_S ? li.max_cols : li.max_cols_pair;
  const int nsl = slices((int64_t)p->m * nblk, li.kind == KIND_V ? li.max_in : cols);
  const int tile = 32 / LR * TC;  // columns of a warp's tile
  int nt = ((cols / nsl + tile - 1) / tile + 1) / 2 * 32;  // two tiles per warp in the widest node
  nt = std::max(64, std::min(NTMAX, nt));
  auto go = [&](auto kern) -> idbf_status {
    if (sm > 48 * 1024) IDBF_CUDA_TRY(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm));
    kern<<<(unsigned)((int64_t)p->m * nsl * nblk), nt, sm, st>>>(p->level(l), (const typename P::mat_t*)mat, io, li.max_in,
                                                                li.max_out, li.max_rows, li.max_cols_pair, nblk, nsl);
    IDBF_CUDA_TRY(cudaGetLastError());
    return IDBF_OK;
  };
  return nblk == 1 ? go(k_node_adj<P, RB, TC, LR, U, NTMAX, MINB, true>) : go(k_node_adj<P, RB, TC, LR, U, NTMAX, MINB, false>);
}

// The fewest right-hand-side blocks of at most `cap` columns, as even as possible: block width.
static int even_block(int R, int cap) {
  const int nblk = (R + cap - 1) / cap;
  return (R + nblk - 1) / nblk;
}

template <class P>
static idbf_status fwd_level(Plan* p, int l, const void* mat, const IO<typename P::vec_t>& io, cudaStream_t st) {
  idbf_status s = IDBF_EUNSUPPORTED;
  // wide blocks whose operands do not fit in shared memory fall through to narrower ones
  if constexpr (std::is_same<P, FP32P>::value) {
    const int w = even_block(io.R, 16);
    if (w > 12) s = fwd_launch<P, 16, 2, 4, 256, 2>(p, l, mat, io, st);
    if (s == IDBF_EUNSUPPORTED && w > 8) s = fwd_launch<P, 12, 2, 4, 256, 2>(p, l, mat, io, st);
    if (s == IDBF_EUNSUPPORTED && w > 6) s = fwd_launch<P, 8, 2, 4, 256, 2>(p, l, mat, io, st);
    if (s == IDBF_EUNSUPPORTED && w > 4) s = fwd_launch<P, 6, 2, 4, 256, 3>(p, l, mat, io, st);
    if (s == IDBF_EUNSUPPORTED && w > 2) s = fwd_launch<P, 4, 2, 4, 256, 3>(p, l, mat, io, st);
    if (s == IDBF_EUNSUPPORTED && w > 1) s = fwd_launch<P, 2, 1, 8, 384, 2>(p, l, mat, io, st);
    if (s == IDBF_EUNSUPPORTED) s = fwd_launch<P, 1, 1, 8, 512, 2>(p, l, mat, io, st);
  } else if constexpr (std::is_same<P, FP64P>::value || std::is_same<P, FP64S32P>::value) {
    const int w = even_block(io.R, 8);
    if (w > 4) s = fwd_launch<P, 8, 1, 2, 256, 2>(p, l, mat, io, st);
    if (s == IDBF_EUNSUPPORTED && w > 2) s = fwd_launch<P, 4, 1, 4, 256, 2>(p, l, mat, io, st);
    if (s == IDBF_EUNSUPPORTED && w > 1) s = fwd_launch<P, 2, 1, 4, 256, 2>(p, l, mat, io, st);
    if (s == IDBF_EUNSUPPORTED) s = fwd_launch<P, 1, 1, 4, 512, 2>(p, l, mat, io, st);
  } else {
    const int w = even_block(io.R, 4);
    if (w > 3) s = fwd_launch<P, 4, 1, 2, 256, 2>(p, l, mat, io, st);
    if (s == IDBF_EUNSUPPORTED && w > 2) s = fwd_launch<P, 3, 1, 2, 256, 2>(p, l, mat, io, st);
    if (s == IDBF_EUNSUPPORTED && w > 1) s = fwd_launch<P, 2, 1, 4, 256, 2>(p, l, mat, io, st);
    if (s == IDBF_EUNSUPPORTED) s = fwd_launch<P, 1, 1, 4, 512, 2>(p, l, mat, io, st);
  }
  return s;
}

template <class P>
static idbf_status adj_level(Plan* p, int l, const void* mat, const IO<typename P::vec_t>& io, cudaStream_t st) {
  idbf_status s = IDBF_EUNSUPPORTED;
  if constexpr (std::is_same<P, FP32P>::value) {
    const int w = even_block(io.R, 16);
    if (w > 8) s = adj_launch<P, 16, 2, 4, 2, 256, 2>(p, l, mat, io, st);
    if (s == IDBF_EUNSUPPORTED && w > 4) s = adj_launch<P, 8, 4, 8, 1, 256, 2>(p, l, mat, io, st);
    if (s == IDBF_EUNSUPPORTED && w > 2) s = adj_launch<P, 4, 4, 8, 2, 256, 3>(p, l, mat, io, st);
    if (s == IDBF_EUNSUPPORTED && w > 1) s = adj_launch<P, 2, 4, 8, 2, 256, 3>(p, l, mat, io, st);
    if (s == IDBF_EUNSUPPORTED) s = adj_launch<P, 1, 4, 16, 2, 256, 4>(p, l, mat, io, st);
  } else if constexpr (std::is_same<P, FP64P>::value) {
    const int w = even_block(io.R, 8);
    if (w > 4) s = adj_launch<P, 8, 1, 8, 2, 256, 2>(p, l, mat, io, st);
    if (s == IDBF_EUNSUPPORTED && w > 2) s = adj_launch<P, 4, 2, 8, 2, 256, 2>(p, l, mat, io, st);
    if (s == IDBF_EUNSUPPORTED && w > 1) s = adj_launch<P, 2, 2, 8, 2, 256, 2>(p, l, mat, io, st);
    if (s == IDBF_EUNSUPPORTED) s = adj_launch<P, 1, 2, 8, 4, 256, 3>(p, l, mat, io, st);
  } else {
    const int w = even_block(io.R, 4);
    if (w > 3) s = adj_launch<P, 4, 1, 8, 2, 256, 2>(p, l, mat, io, st);
    if (s == IDBF_EUNSUPPORTED && w > 2) s = adj_launch<P, 3, 1, 8, 2, 256, 2>(p, l, mat, io, st);
    if (s == IDBF_EUNSUPPORTED && w > 1) s = adj_launch<P, 2, 2, 8, 2, 256, 2>(p, l, mat, io, st);
    if (s == IDBF_EUNSUPPORTED) s = adj_launch<P, 1, 2, 8, 4, 256, 3>(p, l, mat, io, st);
  }
  return s;
}

template <class P>
static IO<typename P::vec_t> make_io(const LevelIO& q) {
  using V = typename P::vec_t;
  IO<V> io;
  io.x = (const V*)q.x;
  io.ldx = q.ldx;
  io.y = (V*)q.y;
  io.ldy = q.ldy;
  io.win = (const V*)q.win;
  io.wout = (V*)q.wout;
  io.R = q.R;
  return io;
}

}  // namespace node

idbf_status node_fwd(Plan* p, Arith a, int l, const LevelIO& q, cudaStream_t st) {
  using namespace node;
  switch (a) {
    case ARITH_FP64: return fwd_level<FP64P>(p, l, p->lmat[IDBF_STORE_C128][l], make_io<FP64P>(q), st);
    case ARITH_DF64: return fwd_level<DF64P>(p, l, p->lmat[IDBF_STORE_DF64][l], make_io<DF64P>(q), st);
    case ARITH_FP32: return fwd_level<FP32P>(p, l, p->lmat[IDBF_STORE_C64][l], make_io<FP32P>(q), st);
    case ARITH_FP64_C64: return fwd_level<FP64S32P>(p, l, p->lmat[IDBF_STORE_C128][l], make_io<FP64S32P>(q), st);
    case ARITH_DF64_C64: return fwd_level<DF64S32P>(p, l, p->lmat[IDBF_STORE_DF64][l], make_io<DF64S32P>(q), st);
  }
  return IDBF_EINVAL;
}

idbf_status node_adj(Plan* p, Arith a, int l, const LevelIO& q, cudaStream_t st) {
  using namespace node;
  switch (a) {
    case ARITH_FP64: return adj_level<FP64P>(p, l, p->lmat[IDBF_STORE_C128][l], make_io<FP64P>(q), st);
    case ARITH_DF64: return adj_level<DF64P>(p, l, p->lmat[IDBF_STORE_DF64][l], make_io<DF64P>(q), st);
    case ARITH_FP32: return adj_level<FP32P>(p, l, p->lmat[IDBF_STORE_C64][l], make_io<FP32P>(q), st);
    default: return IDBF_EINVAL;
  }
}

}  // namespace idbf

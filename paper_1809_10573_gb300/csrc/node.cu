// Launches of the node kernels (node_kernels.cuh): one butterfly level, forward or adjoint, for
// any number of right-hand sides in every CUDA-core arithmetic.
#include <cuda_runtime.h>

#include <algorithm>

#include "idbf_internal.h"
#include "node_kernels.cuh"
#include "node_launch.h"

namespace idbf {
namespace node {

// The right-hand-side blocks of a slice are adjacent CTAs, so that their reads of the factors meet
// in L2, where the first of them asks for the whole node (9 vectors FP32, N = 2^16: 988 against
// 1090 us without). With a single block (STREAM) the factors are read once and marked for early
// eviction; asking for them ahead costs there (one vector FP32 J_0, N = 2^17: 311 against 278 us).
template <class P, int RB, int TR, int U, int NTMAX, int MINB, bool STREAM>
__global__ void __launch_bounds__(NTMAX, MINB)
    k_node_fwd(DevLevel d, const typename P::mat_t* __restrict__ mat, IO<typename P::vec_t> io, int max_in, int max_out,
               int max_rows, int max_cols, int max_rows_pair, int nblk, int nsl) {
  extern __shared__ __align__(16) unsigned char smem[];
  next_may_begin();
  const unsigned unit = blockIdx.x / (unsigned)nblk;
  fwd_body<P, RB, TR, U, STREAM>(d, mat, io, max_in, max_out, max_rows, max_cols, max_rows_pair,
                                 (int64_t)(unit / (unsigned)nsl), (int)(unit % (unsigned)nsl), nsl,
                                 (int)(blockIdx.x % (unsigned)nblk) * RB, io.R, smem, [] { wait_for_inputs(); });
}

template <class P, int RB, int TC, int LR, int U, int NTMAX, int MINB, bool STREAM>
__global__ void __launch_bounds__(NTMAX, MINB)
    k_node_adj(DevLevel d, const typename P::mat_t* __restrict__ mat, IO<typename P::vec_t> io, int max_in, int max_out,
               int max_rows, int max_cols_pair, int nblk, int nsl) {
  extern __shared__ __align__(16) unsigned char smem[];
  next_may_begin();
  const unsigned unit = blockIdx.x / (unsigned)nblk;
  adj_body<P, RB, TC, LR, U, STREAM>(d, mat, io, max_in, max_out, max_rows, max_cols_pair,
                                     (int64_t)(unit / (unsigned)nsl), (int)(unit % (unsigned)nsl), nsl,
                                     (int)(blockIdx.x % (unsigned)nblk) * RB, smem);
}

static constexpr size_t kSmemCap = 220 * 1024;

template <class P, int RB, int TR, int U, int NTMAX, int MINB>
static idbf_status fwd_launch(Plan* p, int l, const void* mat, const IO<typename P::vec_t>& io, bool after, cudaStream_t st) {
  const LevelInfo& li = p->lv[l];
  const size_t sm = fwd_smem<P, RB>(li.max_in, li.max_out, li.max_rows, li.max_cols, li.max_rows_pair, li.kind == KIND_U);
  if (sm > kSmemCap) return IDBF_EUNSUPPORTED;
  const int nblk = (io.R + RB - 1) / RB;
  const int nsl = slices((int64_t)p->m * nblk, fwd_span(li), 4);
  const int nt = fwd_threads(li, TR, nsl, NTMAX);
  auto go = [&](auto kern) -> idbf_status {
    if (sm > 48 * 1024) IDBF_CUDA_TRY(allow_smem(kern, kSmemCap));
    IDBF_CUDA_TRY(launch_after(kern, after, (int64_t)p->m * nsl * nblk, nt, sm, st, p->level(l),
                               (const typename P::mat_t*)mat, io, li.max_in, li.max_out, li.max_rows, li.max_cols,
                               li.max_rows_pair, nblk, nsl));
    return IDBF_OK;
  };
  return nblk == 1 ? go(k_node_fwd<P, RB, TR, U, NTMAX, MINB, true>) : go(k_node_fwd<P, RB, TR, U, NTMAX, MINB, false>);
}

template <class P, int RB, int TC, int LR, int U, int NTMAX, int MINB>
static idbf_status adj_launch(Plan* p, int l, const void* mat, const IO<typename P::vec_t>& io, bool after, cudaStream_t st) {
  const LevelInfo& li = p->lv[l];
  const size_t sm = adj_smem<P, RB>(li.max_in, li.max_out, li.max_rows, li.max_cols_pair, li.kind == KIND_V);
  if (sm > kSmemCap) return IDBF_EUNSUPPORTED;
  const int nblk = (io.R + RB - 1) / RB;
  const int cols = li.kind == KIND_S ? li.max_cols : li.max_cols_pair;
  const int nsl = slices((int64_t)p->m * nblk, li.kind == KIND_V ? li.max_in : cols, 4);
  const int tile = 32 / LR * TC;  // columns of a warp's tile
  // three column tiles per warp in the widest node: few warps for short blocks, so that more nodes
  // are resident (dft N = 40960, 9 vectors FP32: 268 us against 330 with two tiles of the mean node)
  int nt = ((cols + tile - 1) / tile + 2) / 3 * 32;
  nt = std::max(nsl > 1 ? NTMAX : 64, std::min(NTMAX, nt));
  auto go = [&](auto kern) -> idbf_status {
    if (sm > 48 * 1024) IDBF_CUDA_TRY(allow_smem(kern, kSmemCap));
    IDBF_CUDA_TRY(launch_after(kern, after, (int64_t)p->m * nsl * nblk, nt, sm, st, p->level(l),
                               (const typename P::mat_t*)mat, io, li.max_in, li.max_out, li.max_rows, li.max_cols_pair,
                               nblk, nsl));
    return IDBF_OK;
  };
  return nblk == 1 ? go(k_node_adj<P, RB, TC, LR, U, NTMAX, MINB, true>) : go(k_node_adj<P, RB, TC, LR, U, NTMAX, MINB, false>);
}

// Kernel instances: right-hand sides per CTA; rows (or columns) per thread; columns (or rows) in
// flight; threads per CTA and CTAs per SM the registers allow for.
template <class P>
static idbf_status fwd_level(Plan* p, int l, const void* mat, const IO<typename P::vec_t>& io, bool after, cudaStream_t st) {
  idbf_status s = IDBF_EUNSUPPORTED;
  // wide blocks whose operands do not fit in shared memory fall through to narrower ones
  if constexpr (std::is_same<P, FP32P>::value) {
    // eight right-hand sides per CTA and one row per thread, three CTAs of 256 threads per SM: the sums
    // and their totals fit in the registers (two rows per thread spill 532 bytes at 192 x 4 threads; 32
    // vectors, N = 2^16: 1764 us, 2030 with two rows and 128 x 4, 2190 with 192 x 3)
    const int w = even_block(io.R, 8);
    if (w > 6) s = fwd_launch<P, 8, 1, 4, 256, 3>(p, l, mat, io, after, st);
    if (s == IDBF_EUNSUPPORTED && w > 4) s = fwd_launch<P, 6, 1, 4, 256, 3>(p, l, mat, io, after, st);
    if (s == IDBF_EUNSUPPORTED && w > 2) s = fwd_launch<P, 4, 1, 4, 256, 3>(p, l, mat, io, after, st);
    if (s == IDBF_EUNSUPPORTED && w > 1) s = fwd_launch<P, 2, 1, 8, 384, 2>(p, l, mat, io, after, st);
    if (s == IDBF_EUNSUPPORTED) s = fwd_launch<P, 1, 1, 6, 384, 3>(p, l, mat, io, after, st);
  } else if constexpr (std::is_same<P, FP64P>::value || std::is_same<P, FP64S32P>::value) {
    // bound by the FP64 pipe: widths that leave few lanes multiplying for right-hand sides past R
    const int w = fitting_block(io.R);
    if (w > 5) s = fwd_launch<P, 7, 1, 2, 256, 2>(p, l, mat, io, after, st);
    if (s == IDBF_EUNSUPPORTED && w > 4) s = fwd_launch<P, 5, 1, 4, 256, 2>(p, l, mat, io, after, st);
    if (s == IDBF_EUNSUPPORTED && w > 3) s = fwd_launch<P, 4, 1, 4, 256, 2>(p, l, mat, io, after, st);
    if (s == IDBF_EUNSUPPORTED && w > 2) s = fwd_launch<P, 3, 1, 4, 256, 2>(p, l, mat, io, after, st);
    if (s == IDBF_EUNSUPPORTED && w > 1) s = fwd_launch<P, 2, 1, 4, 256, 2>(p, l, mat, io, after, st);
    // one vector: fewer resident CTAs than registers allow, for the same balance (FIO N = 2^16 1.50 ms
    // against 1.60 with 64 registers; J_0 624 against 655 us)
    if (s == IDBF_EUNSUPPORTED && p->lv[l].max_rows_pair <= 192) s = fwd_launch<P, 1, 1, 8, 256, 3>(p, l, mat, io, after, st);
    if (s == IDBF_EUNSUPPORTED) s = fwd_launch<P, 1, 1, 7, 384, 2>(p, l, mat, io, after, st);
  } else {
    const int w = even_block(io.R, 4);
    if (w > 3) s = fwd_launch<P, 4, 1, 2, 256, 2>(p, l, mat, io, after, st);
    if (s == IDBF_EUNSUPPORTED && w > 2) s = fwd_launch<P, 3, 1, 2, 256, 2>(p, l, mat, io, after, st);
    if (s == IDBF_EUNSUPPORTED && w > 1) s = fwd_launch<P, 2, 1, 4, 256, 2>(p, l, mat, io, after, st);
    if (s == IDBF_EUNSUPPORTED) s = fwd_launch<P, 1, 1, 4, 384, 2>(p, l, mat, io, after, st);
  }
  return s;
}

template <class P>
static idbf_status adj_level(Plan* p, int l, const void* mat, const IO<typename P::vec_t>& io, bool after, cudaStream_t st) {
  idbf_status s = IDBF_EUNSUPPORTED;
  if constexpr (std::is_same<P, FP32P>::value) {
    // sixteen right-hand sides, one column per lane: with the totals two columns need more than the 128
    // registers of two CTAs (32 vectors, N = 2^16: 2115 us; 1815 without totals, with errors 10 to 50 %
    // larger). Eight: a column over eight lanes without totals is 10 % faster, with errors 5 to 20 % larger
    const int w = even_block(io.R, 16);
    if (w > 8) s = adj_launch<P, 16, 1, 4, 2, 256, 2>(p, l, mat, io, after, st);
    if (s == IDBF_EUNSUPPORTED && w > 4) s = adj_launch<P, 8, 1, 4, 2, 192, 4>(p, l, mat, io, after, st);
    if (s == IDBF_EUNSUPPORTED && w > 2) s = adj_launch<P, 4, 2, 8, 2, 256, 3>(p, l, mat, io, after, st);
    if (s == IDBF_EUNSUPPORTED && w > 1) s = adj_launch<P, 2, 4, 8, 2, 256, 3>(p, l, mat, io, after, st);
    if (s == IDBF_EUNSUPPORTED) s = adj_launch<P, 1, 4, 16, 2, 256, 4>(p, l, mat, io, after, st);
  } else if constexpr (std::is_same<P, FP64P>::value) {
    const int w = fitting_block(io.R);
    if (w > 5) s = adj_launch<P, 7, 1, 8, 2, 256, 2>(p, l, mat, io, after, st);
    if (s == IDBF_EUNSUPPORTED && w > 4) s = adj_launch<P, 5, 1, 8, 2, 256, 2>(p, l, mat, io, after, st);
    if (s == IDBF_EUNSUPPORTED && w > 3) s = adj_launch<P, 4, 2, 8, 2, 256, 2>(p, l, mat, io, after, st);
    if (s == IDBF_EUNSUPPORTED && w > 2) s = adj_launch<P, 3, 2, 8, 2, 256, 2>(p, l, mat, io, after, st);
    if (s == IDBF_EUNSUPPORTED && w > 1) s = adj_launch<P, 2, 2, 8, 2, 256, 2>(p, l, mat, io, after, st);
    // one vector: four sums of single columns (two columns of two sums are 2 % faster, N = 2^12..2^16, with
    // 2-8 % larger errors)
    if (s == IDBF_EUNSUPPORTED) s = adj_launch<P, 1, 1, 8, 4, 256, 3>(p, l, mat, io, after, st);
  } else {
    const int w = even_block(io.R, 4);
    if (w > 3) s = adj_launch<P, 4, 1, 8, 2, 256, 2>(p, l, mat, io, after, st);
    if (s == IDBF_EUNSUPPORTED && w > 2) s = adj_launch<P, 3, 1, 8, 2, 256, 2>(p, l, mat, io, after, st);
    if (s == IDBF_EUNSUPPORTED && w > 1) s = adj_launch<P, 2, 2, 8, 2, 256, 2>(p, l, mat, io, after, st);
    if (s == IDBF_EUNSUPPORTED) s = adj_launch<P, 1, 2, 8, 2, 256, 3>(p, l, mat, io, after, st);
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
    case ARITH_FP64: return fwd_level<FP64P>(p, l, p->lmat[IDBF_STORE_C128][l], make_io<FP64P>(q), q.after, st);
    case ARITH_DF64: return fwd_level<DF64P>(p, l, p->lmat[IDBF_STORE_DF64][l], make_io<DF64P>(q), q.after, st);
    case ARITH_FP32: return fwd_level<FP32P>(p, l, p->lmat[IDBF_STORE_C64][l], make_io<FP32P>(q), q.after, st);
    case ARITH_FP64_C64: return fwd_level<FP64S32P>(p, l, p->lmat[IDBF_STORE_C128][l], make_io<FP64S32P>(q), q.after, st);
    case ARITH_DF64_C64: return fwd_level<DF64S32P>(p, l, p->lmat[IDBF_STORE_DF64][l], make_io<DF64S32P>(q), q.after, st);
  }
  return IDBF_EINVAL;
}

idbf_status node_adj(Plan* p, Arith a, int l, const LevelIO& q, cudaStream_t st) {
  using namespace node;
  switch (a) {
    case ARITH_FP64: return adj_level<FP64P>(p, l, p->lmat[IDBF_STORE_C128][l], make_io<FP64P>(q), q.after, st);
    case ARITH_DF64: return adj_level<DF64P>(p, l, p->lmat[IDBF_STORE_DF64][l], make_io<DF64P>(q), q.after, st);
    case ARITH_FP32: return adj_level<FP32P>(p, l, p->lmat[IDBF_STORE_C64][l], make_io<FP32P>(q), q.after, st);
    default: return IDBF_EINVAL;
  }
}

}  // namespace idbf

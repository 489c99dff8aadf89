// Per-node bodies of the level kernels, forward and adjoint, for any number of right-hand sides.
//
// A CTA computes one slice of one node for a block of RB right-hand sides. The node's input
// vectors are staged once in shared memory as operands; the factor blocks are read straight from
// global memory into registers (a warp reads consecutive rows of a column), several columns ahead,
// with no barrier between a node's first and last column, so that the loads of all resident CTAs
// overlap freely and the memory system, or the FMA pipes, set the time. Every thread keeps a
// small tile of the result in registers (rows or columns x right-hand sides).
//
// What bounds it: with one right-hand side the factor bytes (HBM) or the FP64 pipe; with many,
// the FMA pipes.
#pragma once

#include "level_kernels.cuh"

namespace idbf {
namespace node {

// double-float vectors between levels stay in the double-float format for any number of
// right-hand sides
template <class P>
using BndOf = Bnd<P, std::is_same<P, DF64P>::value>;

// operands of one element (RB right-hand sides) are padded by 16 bytes when a row of them is a
// multiple of 64 bytes, so that lanes reading neighbouring elements hit different banks
template <class P, int RB>
__host__ __device__ constexpr int op_pitch() {
  using G = typename P::gv_t;
  return (RB * sizeof(G)) % 64 == 0 && RB > 1 ? RB + (int)(16 / sizeof(G)) : RB;
}

// How the terms of a row (or column) are added up, so that the rounding error does not grow with its
// length:
//   FOLD  terms after which the running sums are folded into totals beside them: double-float, and
//         complex64, where a fold is a small part of the arithmetic;
//   K     independent sums that take the columns (rows) in turn and meet at the end: FP64, whose pipe
//         is the bound and which folds would load further (one sum for one vector forward, whose rows
//         are cut over the most lanes), and the complex64 adjoint of one or two vectors, whose lanes
//         hold few rows.
// Errors against the FP64 apply, FIO N = 2^16, with single chains and now: complex64 4 vectors 7.8e-7
// and 3.8e-7, 32 vectors 7.7e-7 and 3.9e-7, their adjoint 4.3e-7 and 3.5e-7, 5.5e-7 and 3.6e-7; double-float 4
// vectors 4.1e-14 (folds of 16 terms) and 2.9e-14, adjoint 1.85e-14 and 1.72e-14.
template <class P, int RB, bool ADJ>
struct Chains {
  static constexpr bool DF = std::is_same<typename P::part_t, float4>::value;
  static constexpr bool F64 = std::is_same<typename P::part_t, double2>::value;
  static constexpr int K = F64 ? (RB > 1 ? 2 : ADJ ? 4 : 1) : !DF && ADJ && RB <= 2 ? 2 : 1;
  static constexpr int FOLD = DF ? (ADJ ? 2 : RB <= 2 ? 4 : 8) : K > 1 || F64 ? 0 : !ADJ && RB == 4 ? 8 : 4;
};

// The RB operands of one element and the sums they enter. In general operand rb is element rb of the
// row and a sum is the policy's accumulator; complex64 with an even RB packs the right-hand sides in
// pairs, a row holding (re, re, im, im) per pair and a sum being two f32x2: each complex
// multiply-add of a pair is four packed FMAs, in the order of FP32P::mac on either lane, and the
// pairs' real and imaginary parts come out of one 16-byte load as packed registers.
template <class P, int RB, int K, bool TOT, bool PACKED = std::is_same<P, FP32P>::value && RB % 2 == 0>
struct Sums {
  using G = typename P::gv_t;
  using M = typename P::mat_t;
  struct ops_t { G g[RB]; };
  typename P::acc_t a[K][RB];
  __device__ static __forceinline__ void put(G* row, int rb, const G& v) { row[rb] = v; }
  __device__ static __forceinline__ G get(const G* row, int rb) { return row[rb]; }
  __device__ static __forceinline__ void load(ops_t& o, const G* row) {
#pragma unroll
    for (int i = 0; i < RB; ++i) o.g[i] = row[i];
  }
  __device__ __forceinline__ void init() {
#pragma unroll
    for (int k = 0; k < K; ++k)
#pragma unroll
      for (int i = 0; i < RB; ++i) P::init(a[k][i]);
  }
  __device__ __forceinline__ void mac(int u, const M& m, const ops_t& o) {  // into sum u mod K
#pragma unroll
    for (int i = 0; i < RB; ++i) {
      // double-float, three vectors and more: the registers of a second error sum cost 10 %
      if constexpr (std::is_same<typename P::part_t, float4>::value && RB > 2) P::mac_narrow(a[u % K][i], m, o.g[i]);
      else P::mac(a[u % K][i], m, o.g[i]);
    }
  }
  __device__ __forceinline__ void macc(int u, const M& m, const ops_t& o) {  // conj(m)
#pragma unroll
    for (int i = 0; i < RB; ++i) P::macc(a[u % K][i], m, o.g[i]);
  }
  __device__ __forceinline__ void fold() {
    if constexpr (K == 1) {
#pragma unroll
      for (int i = 0; i < RB; ++i) P::flush(a[0][i]);
    }
  }
  __device__ __forceinline__ void parts(typename P::part_t (&pr)[RB]) {
#pragma unroll
    for (int i = 0; i < RB; ++i) {
#pragma unroll
      for (int k = 0; k < K; ++k) P::flush(a[k][i]);
#pragma unroll
      for (int h = 1; h < K; h *= 2)
#pragma unroll
        for (int k = 0; k + h < K; k += 2 * h) P::combine(a[k][i], P::part(a[k + h][i]));
      pr[i] = P::part(a[0][i]);
    }
  }
};
template <class P, int RB, int K, bool TOT>
struct Sums<P, RB, K, TOT, true> {
  using G = float2;
  struct ops_t { ulonglong2 g[RB / 2]; };
  f32x2 re[K][RB / 2], im[K][RB / 2];
  f32x2 tre[TOT ? RB / 2 : 1], tim[TOT ? RB / 2 : 1];  // totals
  __device__ static __forceinline__ void put(G* row, int rb, const G& v) {
    float* f = (float*)row + (rb >> 1) * 4 + (rb & 1);
    f[0] = v.x;
    f[2] = v.y;
  }
  __device__ static __forceinline__ G get(const G* row, int rb) {
    const float* f = (const float*)row + (rb >> 1) * 4 + (rb & 1);
    return make_float2(f[0], f[2]);
  }
  __device__ static __forceinline__ void load(ops_t& o, const G* row) {
#pragma unroll
    for (int i = 0; i < RB / 2; ++i) o.g[i] = ((const ulonglong2*)row)[i];
  }
  __device__ __forceinline__ void init() {
#pragma unroll
    for (int i = 0; i < RB / 2; ++i) {
#pragma unroll
      for (int k = 0; k < K; ++k) re[k][i] = im[k][i] = 0ull;
      if (TOT) tre[TOT ? i : 0] = tim[TOT ? i : 0] = 0ull;
    }
  }
  __device__ __forceinline__ void mac(int u, const float2& m, const ops_t& o) {
    const f32x2 mx = pk2(m.x, m.x), my = pk2(m.y, m.y), ny = pk2(-m.y, -m.y);
    const int k = u % K;
#pragma unroll
    for (int i = 0; i < RB / 2; ++i) {
      re[k][i] = fma2(mx, o.g[i].x, re[k][i]);
      im[k][i] = fma2(mx, o.g[i].y, im[k][i]);
      re[k][i] = fma2(ny, o.g[i].y, re[k][i]);
      im[k][i] = fma2(my, o.g[i].x, im[k][i]);
    }
  }
  __device__ __forceinline__ void macc(int u, const float2& m, const ops_t& o) { mac(u, make_float2(m.x, -m.y), o); }
  __device__ __forceinline__ void fold() {
    if constexpr (TOT) {
#pragma unroll
      for (int i = 0; i < RB / 2; ++i) {
        tre[i] = add2(tre[i], re[0][i]);
        tim[i] = add2(tim[i], im[0][i]);
        re[0][i] = im[0][i] = 0ull;
      }
    }
  }
  __device__ __forceinline__ void parts(float2 (&pr)[RB]) {
    static_assert(K == 1 || (K == 2 && !TOT), "one sum, or two that meet in one addition");
    fold();
#pragma unroll
    for (int i = 0; i < RB / 2; ++i) {
      const float2 r = upk2(TOT ? tre[TOT ? i : 0] : K == 1 ? re[0][i] : add2(re[0][i], re[K - 1][i]));
      const float2 m = upk2(TOT ? tim[TOT ? i : 0] : K == 1 ? im[0][i] : add2(im[0][i], im[K - 1][i]));
      pr[2 * i] = make_float2(r.x, m.x);
      pr[2 * i + 1] = make_float2(r.y, m.y);
    }
  }
};

// the share of slice sl of nsl of both blocks of a node, by two threads of the CTA
template <class M>
__device__ __forceinline__ void prefetch_blocks(const M* mat, const int64_t (&mov)[2], const int (&rows)[2],
                                                const int (&cols)[2], int sl, int nsl) {
  if (threadIdx.x < 2) {
    const int c = threadIdx.x;
    const int64_t n = (int64_t)(c ? rows[1] : rows[0]) * (c ? cols[1] : cols[0]);
    const int64_t a = n * sl / nsl, b = n * (sl + 1) / nsl;
    prefetch_l2(mat + (c ? mov[1] : mov[0]) + a, (b - a) * (int64_t)sizeof(M));
  }
}

// Sums the partial sums pr[0 .. RB-1] of the S (1, 2, 4 or 8) neighbouring lanes of a group: lane s
// ends with the sums of the right-hand sides rb = s mod S, in slots rb & ~(S-1). Each step trades
// half of what is left with the lane one bit away, so S lanes exchange RB (1 - 1/S) values each
// instead of RB log2 S (shuffles run at a quarter of the FMA rate). Where a slot has no partner
// (RB odd, or fewer right-hand sides than lanes) both lanes keep the sum.
template <class P, int RB>
__device__ __forceinline__ void lane_sum(typename P::part_t (&pr)[RB], int S, int s) {
#pragma unroll
  for (int o = 1; o < 8; o <<= 1) {
    if (o >= S) break;
    const bool up = s & o;
#pragma unroll
    for (int i = 0; i < RB; ++i) {
      if (i & (2 * o - 1)) continue;
      const int q = i + o;
      if (q < RB) pr[i] = P::add_lane(up ? pr[q < RB ? q : 0] : pr[i], up ? pr[i] : pr[q < RB ? q : 0], o);
      else pr[i] = P::add_lane(pr[i], pr[i], o);
    }
  }
}

// ---------------------------------------------------------------------------------------------
// Forward. Work of slice sl of nsl of node j:
//   V and S levels: the rows [T sl / nsl, T (sl+1) / nsl) of the T = rows_0 + rows_1 output rows;
//   U levels: the output positions [t sl / nsl, t (sl+1) / nsl) of t = concat(out_0, out_1); the
//     rows of block c that land there are consecutive, because the lists p_c ascend.
// A thread takes TR rows (ntile apart, so that a warp reads consecutive rows) and all RB
// right-hand sides; when the slice has fewer row tiles than half the CTA, the columns are dealt to
// S = 2, 4 or 8 neighbouring lanes, which add their sums by shuffles. U levels collect the
// products in shared memory (res) and add the two terms of every position at the end.
template <class P, int RB>
__host__ __device__ constexpr size_t fwd_smem(int max_in, int max_out, int max_rows, int max_cols, int max_rows_pair,
                                              bool u_level) {
  using B = typename BndOf<P>::b_t;
  size_t n = ((size_t)max_in * op_pitch<P, RB>() * sizeof(typename P::gv_t) + 15) & ~(size_t)15;
  if (u_level) n += (size_t)max_rows_pair * RB * sizeof(B);
  n += 2 * (size_t)max_cols * sizeof(int32_t);                              // operand of every column
  n += 2 * (size_t)(u_level ? max_out : max_rows) * sizeof(int32_t);       // V: q lists; U: term of every position
  return (n + 15) & ~(size_t)15;
}

// wait() returns, in every thread, once the inputs may be read; everything before it reads the node's
// description and factors only.
template <class P, int RB, int TR, int U, bool STREAM, class W>
__device__ __forceinline__ void fwd_body(const DevLevel& d, const typename P::mat_t* __restrict__ mat,
                                         const IO<typename P::vec_t>& io, int max_in, int max_out, int max_rows,
                                         int max_cols, int max_rows_pair, int64_t j, int sl, int nsl, int r0,
                                         int r1, unsigned char* smem, W wait) {
  using G = typename P::gv_t;
  using M = typename P::mat_t;
  using BP = BndOf<P>;
  using B = typename BP::b_t;
  using CH = Chains<P, RB, false>;
  using SM = Sums<P, RB, CH::K, CH::FOLD != 0>;
  constexpr int PITCH = op_pitch<P, RB>();
  const int tid = threadIdx.x, nt = blockDim.x, lane = tid & 31;
  const int nrb = min(RB, r1 - r0);  // right-hand sides r0 .. r1-1
  const bool ulev = d.kind == KIND_U;
  G* opd = (G*)smem;
  B* res = (B*)(smem + (((size_t)max_in * PITCH * sizeof(G) + 15) & ~(size_t)15));
  int32_t* kix = (int32_t*)(res + (ulev ? (size_t)max_rows_pair * RB : 0));  // [2][max_cols]
  int32_t* aux = kix + 2 * max_cols;  // V: q lists [2][max_rows]; U: terms [2][max_out]
  __shared__ int s_ra[2], s_rb[2];    // U: rows of each block in this slice

  // ---- the node: everything here is independent of the input vectors
  const int rowsv[2] = {d.rows[2 * j], d.rows[2 * j + 1]};
  const int colsv[2] = {d.cols[2 * j], d.cols[2 * j + 1]};
  const int64_t mov[2] = {d.moff[2 * j], d.moff[2 * j + 1]};
  if (!STREAM && r0 == 0) prefetch_blocks(mat, mov, rowsv, colsv, sl, nsl);
  int l0, l1;
  int64_t i0 = 0, i1 = 0;
  if (d.lev == 0) {
    l0 = leaf_len(d, j);
    l1 = 0;
    i0 = leaf_start(d, j);
  } else {
    l0 = d.in_len[2 * j];
    l1 = d.in_len[2 * j + 1];
    i0 = d.in_off[2 * j];
    i1 = d.in_off[2 * j + 1];
  }
  int ra[2], rn[2];      // first row and number of rows of each block in this slice
  int e0 = 0, e1 = 0;    // U: output positions of this slice
  if (!ulev) {
    const int tot = rowsv[0] + rowsv[1];
    const int g0 = (int)((int64_t)tot * sl / nsl), g1 = (int)((int64_t)tot * (sl + 1) / nsl);
    ra[0] = min(g0, rowsv[0]);
    rn[0] = min(g1, rowsv[0]) - ra[0];
    ra[1] = max(g0 - rowsv[0], 0);
    rn[1] = max(g1 - rowsv[0], 0) - ra[1];
    if (d.kind == KIND_V) {
#pragma unroll
      for (int c = 0; c < 2; ++c) {
        const int32_t* ix = d.idx + d.ioff[2 * j + c];
        for (int i = tid; i < rn[c]; i += nt) aux[c * max_rows + ra[c] + i] = ix[ra[c] + i];
        for (int k = tid; k < colsv[c]; k += nt) kix[c * max_cols + k] = ix[rowsv[c] + k] * PITCH;
      }
    } else {
#pragma unroll
      for (int c = 0; c < 2; ++c)
        for (int k = tid; k < colsv[c]; k += nt) kix[c * max_cols + k] = k * PITCH;
    }
  } else {
    const int tl = l0 + rowsv[0];  // |t| = |q_0| + |p_0|
    e0 = (int)((int64_t)tl * sl / nsl);
    e1 = (int)((int64_t)tl * (sl + 1) / nsl);
    if (tid < 2) {
      s_ra[tid] = rowsv[tid];
      s_rb[tid] = rowsv[tid];
    }
    __syncthreads();
#pragma unroll
    for (int c = 0; c < 2; ++c) {
      const int lc = c ? l1 : l0;
      const int32_t* ix = d.idx + d.ioff[2 * j + c];
      for (int i = tid; i < lc; i += nt) {
        const int e = ix[i];
        if (e >= e0 && e < e1) aux[c * max_out + e - e0] = i;
      }
      for (int r = tid; r < rowsv[c]; r += nt) {
        const int e = ix[lc + r];
        if (e >= e0 && e < e1) aux[c * max_out + e - e0] = ~r;
        if (nsl > 1) {
          const int ep = r > 0 ? ix[lc + r - 1] : -1;
          if (e >= e0 && ep < e0) s_ra[c] = r;
          if (e >= e1 && ep < e1) s_rb[c] = r;
        }
      }
      for (int k = tid; k < colsv[c]; k += nt) kix[c * max_cols + k] = ((c ? l0 : 0) + k) * PITCH;
    }
  }
  if (ulev) {
    __syncthreads();
#pragma unroll
    for (int c = 0; c < 2; ++c) {
      ra[c] = nsl > 1 ? s_ra[c] : 0;
      rn[c] = (nsl > 1 ? s_rb[c] : rowsv[c]) - ra[c];
    }
  }
  const int nt0 = (rn[0] + TR - 1) / TR, T = nt0 + (rn[1] + TR - 1) / TR;
  const int maxc = max(colsv[0], colsv[1]);
  // Four columns per lane at least (eight: double-float, FIO N = 2^12, one vector 68 us against 63, 2^14 221
  // against 218), in FP64 with one vector eight, whose lanes' sums load its pipe (NUFFT N = 11331: 136 us,
  // 177 with four).
  int S = 1;
  while (S < 8 && 2 * S * T <= nt && maxc >= (CH::F64 && RB == 1 ? 16 : 8) * S) S *= 2;
  int64_t obv[2] = {0, 0};
  if (!ulev) {
    obv[0] = d.out_off[out_seg_id(d, j, 0)];
    obv[1] = d.out_off[out_seg_id(d, j, 1)];
  }

  // ---- this thread's row tile and its first columns
  const int s = tid & (S - 1);
  int c, rt, ntc, cols, rbeg, rcnt, step, off;
  const M* Mc;
  int roff[TR];
  M mv[U][TR];
  auto load = [&](int u, M (&m)[TR]) {
#pragma unroll
    for (int i = 0; i < TR; ++i) {
      const M* q = Mc + (off + u * step + roff[i]);
      m[i] = STREAM ? __ldcs(q) : __ldg(q);
    }
  };
  auto begin = [&](int w) {  // tile w / S (none past the last: no columns); the entries of its first U columns
    const bool active = w < T * S;
    const int tile = active ? w / S : 0;
    c = tile >= nt0;
    rt = tile - (c ? nt0 : 0);
    ntc = c ? T - nt0 : nt0;
    const int rows = c ? rowsv[1] : rowsv[0];
    cols = active ? (c ? colsv[1] : colsv[0]) : 0;
    rbeg = c ? ra[1] : ra[0];
    rcnt = active ? (c ? rn[1] : rn[0]) : 0;
    Mc = mat + (c ? mov[1] : mov[0]) + rbeg;
#pragma unroll
    for (int i = 0; i < TR; ++i) roff[i] = min(rt + i * ntc, max(rcnt - 1, 0));
    step = S * rows;
    off = s * rows;
#pragma unroll
    for (int u = 0; u < U; ++u)
      if (s + u * S < cols) load(u, mv[u]);
  };
  begin(tid);

  // ---- inputs -> operands
  wait();
  if (d.lev == 0) {
    for (int i = tid; i < l0 * RB; i += nt) {
      const int rb = i / l0, e = i - rb * l0;
      SM::put(opd + e * PITCH, rb, P::cvt(rb < nrb ? io.x[i0 + e + (int64_t)(r0 + rb) * io.ldx] : P::zero()));
    }
  } else {
    const B* winb = (const B*)io.win;
    for (int i = tid; i < (l0 + l1) * RB; i += nt) {
      const int e = i / RB, rb = i - e * RB;
      const int64_t o = e < l0 ? i0 + e : i1 + (e - l0);
      SM::put(opd + e * PITCH, rb, BP::g_of(rb < nrb ? winb[o * io.R + r0 + rb] : BP::zero()));
    }
  }
  __syncthreads();

  // ---- block products
  B* woutb = (B*)io.wout;
  for (int w = tid; w - lane < T * S; w += nt) {
    if (w != tid) begin(w);
    const int32_t* kc = kix + c * max_cols;
    SM acc[TR];
#pragma unroll
    for (int i = 0; i < TR; ++i) acc[i].init();
    auto mac = [&](int k, int u, const M (&m)[TR]) {
      typename SM::ops_t g;
      SM::load(g, opd + kc[k]);
#pragma unroll
      for (int i = 0; i < TR; ++i) acc[i].mac(u, m[i], g);
    };
    int k = s, since = 0;
    for (; k + (U - 1) * S < cols; k += U * S) {
      // an entry's register takes the entry U columns on as soon as it is consumed
#pragma unroll
      for (int u = 0; u < U; ++u) {
        mac(k + u * S, u, mv[u]);
        if (k + (U + u) * S < cols) load(U + u, mv[u]);
      }
      off += U * step;
      since += U;
      if (CH::FOLD > 0 && since >= CH::FOLD) {
#pragma unroll
        for (int i = 0; i < TR; ++i) acc[i].fold();
        since = 0;
      }
    }
#pragma unroll
    for (int u = 0; u < U - 1; ++u)
      if (k + u * S < cols) mac(k + u * S, u, mv[u]);
#pragma unroll
    for (int i = 0; i < TR; ++i) {
      typename P::part_t pr[RB];
      acc[i].parts(pr);
      lane_sum<P, RB>(pr, S, s);
      const int rr = rt + i * ntc;
      if (rr >= rcnt) continue;
#pragma unroll
      for (int ib = 0; ib < RB; ++ib) {
        if (ib & (S - 1)) continue;
        const int rb = ib | s;
        if (rb >= RB) continue;
        B v = BP::of_part(pr[ib]);
        if (ulev) {
          res[((size_t)(c ? rn[0] : 0) + rr) * RB + rb] = v;
        } else if (rb < nrb) {
          if (d.kind == KIND_V) v = BP::add(v, BP::b_of_g(SM::get(opd + aux[c * max_rows + rbeg + rr] * PITCH, rb)));
          woutb[((c ? obv[1] : obv[0]) + rbeg + rr) * io.R + r0 + rb] = v;
        }
      }
    }
  }
  if (!ulev) return;

  // ---- U levels: the two terms of every output position
  __syncthreads();
  const int ne = e1 - e0;
  auto term = [&](int c, int e, int rb) -> B {
    const int t = aux[c * max_out + e];
    return t >= 0 ? BP::b_of_g(SM::get(opd + ((c ? l0 : 0) + t) * PITCH, rb)) : res[((c ? rn[0] : 0) + ~t - ra[c]) * RB + rb];
  };
  if (d.lev == d.L) {
    const int64_t y0 = leaf_start(d, j) + e0;
    for (int i = tid; i < ne * nrb; i += nt) {
      const int rb = i / ne, e = i - rb * ne;
      io.y[y0 + e + (int64_t)(r0 + rb) * io.ldy] = BP::v_of(BP::add(term(0, e, rb), term(1, e, rb)));
    }
  } else {
    const int64_t s0 = out_seg_id(d, j, 0), s1 = out_seg_id(d, j, 1);
    const int len0 = d.out_len[s0];
    const int64_t b0 = d.out_off[s0], b1 = d.out_off[s1];
    for (int i = tid; i < ne * RB; i += nt) {
      const int e = i / RB, rb = i - e * RB;
      if (rb >= nrb) continue;
      const int64_t off = e0 + e < len0 ? b0 + e0 + e : b1 + (e0 + e - len0);
      woutb[off * io.R + r0 + rb] = BP::add(term(0, e, rb), term(1, e, rb));
    }
  }
}

// ---------------------------------------------------------------------------------------------
// Adjoint: reads the forward outputs v of node j and writes its forward inputs. An output is a
// column of a block: sum_r conj(M_c(r, i)) g_c[r]. LR neighbouring lanes take the rows of a column
// r = lane, lane + LR, ... (consecutive entries), the 32 / LR lane groups of a warp different
// columns, TC columns per lane; the LR partial sums meet by shuffles.
// Slices: U and S levels a range of columns; V levels a range of input positions [e0, e1) (the
// columns of block c that land there are consecutive, because the lists p_c ascend).
template <class P, int RB>
__host__ __device__ constexpr size_t adj_smem(int max_in, int max_out, int max_rows, int max_cols_pair, bool v_level) {
  using B = typename BndOf<P>::b_t;
  size_t n = ((size_t)max_out * op_pitch<P, RB>() * sizeof(typename P::gv_t) + 15) & ~(size_t)15;
  if (v_level) n += (size_t)max_cols_pair * RB * sizeof(B) + 2 * (size_t)max_in * sizeof(int32_t);
  n += 2 * (size_t)max_rows * sizeof(int32_t);  // operand of every row
  return (n + 15) & ~(size_t)15;
}

template <class P, int RB, int TC, int LR, int U, bool STREAM>
__device__ __forceinline__ void adj_body(const DevLevel& d, const typename P::mat_t* __restrict__ mat,
                                         const IO<typename P::vec_t>& io, int max_in, int max_out, int max_rows,
                                         int max_cols_pair, int64_t j, int sl, int nsl, int r0, unsigned char* smem) {
  using G = typename P::gv_t;
  using M = typename P::mat_t;
  using BP = BndOf<P>;
  using B = typename BP::b_t;
  using CH = Chains<P, RB, true>;
  using SM = Sums<P, RB, CH::K, CH::FOLD != 0>;
  constexpr int PITCH = op_pitch<P, RB>();
  constexpr int CG = 32 / LR, CT = CG * TC;  // lane groups of a warp, columns of a warp's tile
  const int tid = threadIdx.x, nt = blockDim.x, lane = tid & 31, warp = tid >> 5, nw = nt >> 5;
  const int lr = lane & (LR - 1), cg = lane / LR;
  const int nrb = min(RB, io.R - r0);
  const bool vlev = d.kind == KIND_V;
  G* opd = (G*)smem;
  B* res = (B*)(smem + (((size_t)max_out * PITCH * sizeof(G) + 15) & ~(size_t)15));
  int32_t* gix = (int32_t*)(res + (vlev ? (size_t)max_cols_pair * RB : 0));  // [2][max_rows]
  int32_t* aux = gix + 2 * max_rows;                                          // V: terms [2][max_in]
  __shared__ int s_ia[2], s_ib[2];  // V: columns of each block in this slice

  const int rowsv[2] = {d.rows[2 * j], d.rows[2 * j + 1]};
  const int colsv[2] = {d.cols[2 * j], d.cols[2 * j + 1]};
  const int64_t mov[2] = {d.moff[2 * j], d.moff[2 * j + 1]};
  if (!STREAM && r0 == 0) prefetch_blocks(mat, mov, rowsv, colsv, sl, nsl);
  int o0len, o1len = 0;
  int64_t b0, b1 = 0;
  if (d.lev == d.L) {
    o0len = leaf_len(d, j);
    b0 = leaf_start(d, j);
  } else {
    const int64_t s0 = out_seg_id(d, j, 0), s1 = out_seg_id(d, j, 1);
    o0len = d.out_len[s0];
    o1len = d.out_len[s1];
    b0 = d.out_off[s0];
    b1 = d.out_off[s1];
  }
  int ia[2] = {0, 0}, in[2] = {colsv[0], colsv[1]};  // first column and number of columns of each block
  int e0 = 0, e1 = 0;
  if (vlev) {
    const int nin = rowsv[0] + colsv[0];
    e0 = (int)((int64_t)nin * sl / nsl);
    e1 = (int)((int64_t)nin * (sl + 1) / nsl);
    if (tid < 2) {
      s_ia[tid] = colsv[tid];
      s_ib[tid] = colsv[tid];
    }
    __syncthreads();
#pragma unroll
    for (int c = 0; c < 2; ++c) {
      const int32_t* ix = d.idx + d.ioff[2 * j + c];
      for (int r = tid; r < rowsv[c]; r += nt) {
        const int e = ix[r];
        if (e >= e0 && e < e1) aux[c * max_in + e - e0] = r;
        gix[c * max_rows + r] = ((c ? o0len : 0) + r) * PITCH;
      }
      for (int i = tid; i < colsv[c]; i += nt) {
        const int e = ix[rowsv[c] + i];
        if (e >= e0 && e < e1) aux[c * max_in + e - e0] = ~i;
        if (nsl > 1) {
          const int ep = i > 0 ? ix[rowsv[c] + i - 1] : -1;
          if (e >= e0 && ep < e0) s_ia[c] = i;
          if (e >= e1 && ep < e1) s_ib[c] = i;
        }
      }
    }
  } else {
    const int tot = d.kind == KIND_S ? colsv[0] : colsv[0] + colsv[1];
    const int g0 = (int)((int64_t)tot * sl / nsl), g1 = (int)((int64_t)tot * (sl + 1) / nsl);
    ia[0] = min(g0, colsv[0]);
    in[0] = min(g1, colsv[0]) - ia[0];
    ia[1] = max(g0 - colsv[0], 0);
    in[1] = max(g1 - colsv[0], 0) - ia[1];
#pragma unroll
    for (int c = 0; c < 2; ++c) {
      const int32_t* ix = d.kind == KIND_U ? d.idx + d.ioff[2 * j + c] + colsv[c] : nullptr;
      for (int r = tid; r < rowsv[c]; r += nt) gix[c * max_rows + r] = (ix ? ix[r] : (c ? o0len : 0) + r) * PITCH;
    }
  }
  // ---- inputs -> operands
  wait_for_inputs();
  if (d.lev == d.L) {
    for (int i = tid; i < o0len * RB; i += nt) {
      const int rb = i / o0len, e = i - rb * o0len;
      SM::put(opd + e * PITCH, rb, P::cvt(rb < nrb ? io.x[b0 + e + (int64_t)(r0 + rb) * io.ldx] : P::zero()));
    }
  } else {
    const B* winb = (const B*)io.win;
    for (int i = tid; i < (o0len + o1len) * RB; i += nt) {
      const int e = i / RB, rb = i - e * RB;
      const int64_t off = e < o0len ? b0 + e : b1 + (e - o0len);
      SM::put(opd + e * PITCH, rb, BP::g_of(rb < nrb ? winb[off * io.R + r0 + rb] : BP::zero()));
    }
  }
  __syncthreads();
  if (vlev) {
#pragma unroll
    for (int c = 0; c < 2; ++c) {
      ia[c] = nsl > 1 ? s_ia[c] : 0;
      in[c] = (nsl > 1 ? s_ib[c] : colsv[c]) - ia[c];
    }
  }
  const bool slev = d.kind == KIND_S;
  const int nt0 = (in[0] + CT - 1) / CT, T = nt0 + (slev ? 0 : (in[1] + CT - 1) / CT);
  int64_t ib0 = 0, ib1 = 0;
  int len0 = 0;
  if (d.lev > 0) {
    len0 = d.in_len[2 * j];
    ib0 = d.in_off[2 * j];
    ib1 = d.in_off[2 * j + 1];
  }
  B* woutb = (B*)io.wout;
  for (int w = warp; w < T; w += nw) {
    const int c = w >= nt0;
    const int i_first = (w - (c ? nt0 : 0)) * CT + cg;  // this lane's first column within the slice
    const int icnt = c ? in[1] : in[0], ibeg = c ? ia[1] : ia[0];
    SM acc[TC];
#pragma unroll
    for (int t = 0; t < TC; ++t) acc[t].init();
    int coff[TC];
#pragma unroll
    for (int t = 0; t < TC; ++t) coff[t] = ibeg + min(i_first + t * CG, icnt - 1);
    for (int bc = c; bc <= (slev ? 1 : c); ++bc) {  // S levels: both blocks have the same columns
      const int rows = bc ? rowsv[1] : rowsv[0];
      const M* Mc = mat + (bc ? mov[1] : mov[0]);
      const int32_t* gc = gix + bc * max_rows;
      int base[TC];
#pragma unroll
      for (int t = 0; t < TC; ++t) base[t] = coff[t] * rows;
      int r = lr, since = 0;
      auto load = [&](int u, M (&mv)[TC]) {
#pragma unroll
        for (int t = 0; t < TC; ++t) {
          const M* q = Mc + (base[t] + r + u * LR);
          mv[t] = STREAM ? __ldcs(q) : __ldg(q);
        }
      };
      auto mac = [&](int u, const M (&mv)[TC]) {
        typename SM::ops_t g;
        SM::load(g, opd + gc[r + u * LR]);
#pragma unroll
        for (int t = 0; t < TC; ++t) acc[t].macc(u, mv[t], g);
      };
      M mv[U][TC];
#pragma unroll
      for (int u = 0; u < U; ++u)
        if (r + u * LR < rows) load(u, mv[u]);
      for (; r + (U - 1) * LR < rows; r += U * LR) {
#pragma unroll
        for (int u = 0; u < U; ++u) {
          mac(u, mv[u]);
          if (r + (U + u) * LR < rows) load(U + u, mv[u]);
        }
        since += U;
        if (CH::FOLD > 0 && since >= CH::FOLD) {
#pragma unroll
          for (int t = 0; t < TC; ++t) acc[t].fold();
          since = 0;
        }
      }
#pragma unroll
      for (int u = 0; u < U - 1; ++u)
        if (r + u * LR < rows) mac(u, mv[u]);
    }
    __syncwarp();
#pragma unroll
    for (int t = 0; t < TC; ++t) {
      typename P::part_t pr[RB];
      acc[t].parts(pr);
      lane_sum<P, RB>(pr, LR < 8 ? LR : 8, lr & 7);
      if constexpr (LR == 16) {
#pragma unroll
        for (int rb = 0; rb < RB; ++rb) pr[rb] = P::add_lane(pr[rb], pr[rb], 8);
      }
      const int ii = i_first + t * CG;
      if (ii >= icnt || lr >= 8) continue;
      const int i = ibeg + ii;
      constexpr int LS = LR < 8 ? LR : 8;
#pragma unroll
      for (int ib = 0; ib < RB; ib += LS) {
        const int rb = ib | lr;
        if (rb >= RB) continue;
        B v = BP::of_part(pr[ib]);
        if (vlev) {
          res[((c ? in[0] : 0) + ii) * RB + rb] = v;
        } else if (rb < nrb) {
          if (slev) {
            woutb[(i < len0 ? ib0 + i : ib1 + (i - len0)) * io.R + r0 + rb] = v;
          } else {  // U: forward input segment c gets v[q_c] + res_c
            const int q = d.idx[d.ioff[2 * j + c] + i];
            woutb[((c ? ib1 : ib0) + i) * io.R + r0 + rb] = BP::add(BP::b_of_g(SM::get(opd + q * PITCH, rb)), v);
          }
        }
      }
    }
  }
  if (!vlev) return;

  // ---- V levels: the two terms of every input position
  __syncthreads();
  const int ne = e1 - e0;
  auto term = [&](int c, int e, int rb) -> B {
    const int t = aux[c * max_in + e];
    return t >= 0 ? BP::b_of_g(SM::get(opd + ((c ? o0len : 0) + t) * PITCH, rb)) : res[((c ? in[0] : 0) + ~t - ia[c]) * RB + rb];
  };
  if (d.lev == 0) {
    const int64_t y0 = leaf_start(d, j) + e0;
    for (int i = tid; i < ne * nrb; i += nt) {
      const int rb = i / ne, e = i - rb * ne;
      io.y[y0 + e + (int64_t)(r0 + rb) * io.ldy] = BP::v_of(BP::add(term(0, e, rb), term(1, e, rb)));
    }
  } else {
    for (int i = tid; i < ne * RB; i += nt) {
      const int e = i / RB, rb = i - e * RB;
      if (rb >= nrb) continue;
      const int f = e0 + e;
      woutb[(f < len0 ? ib0 + f : ib1 + (f - len0)) * io.R + r0 + rb] = BP::add(term(0, e, rb), term(1, e, rb));
    }
  }
}

}  // namespace node
}  // namespace idbf

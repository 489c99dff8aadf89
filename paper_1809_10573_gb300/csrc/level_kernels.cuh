// What the level kernels share: the arithmetic policies, the format of the vectors between levels, the
// launch overlap, and the warp-per-node forward body of one vector (the node kernels' bodies are in
// node_kernels.cuh). Three policies:
//   FP64P - complex128 factors and vectors, FP64 FMA;
//   DF64P - factors stored as double-float pairs (hi, lo) of binary32, complex128 vectors;
//           products formed exactly with FMA (Dekker's product), sums accumulated with Knuth's
//           TwoSum in chunks (the compensated dot product of Ogita, Rump and Oishi, "Accurate sum
//           and dot product", SIAM J. Sci. Comput. 26, 2005) and folded into a normalised
//           double-float total (Joldes, Muller and Popescu, "Tight and rigorous error bounds for
//           basic building blocks of double-word arithmetic", ACM TOMS 44, 2017);
//   FP32P - complex64 factors and vectors, FP32 FMA, running sums folded into totals.
#pragma once

#include <cuda_runtime.h>

#include <type_traits>

#include "idbf_internal.h"

namespace idbf {

// ---- pairs of binary32 lanes -------------------------------------------------------------------
// add / mul / fma.rn.f32x2 work on two binary32 values in one 64-bit register: the same FP32-pipe
// time per value as the scalar forms (about 116 lanes per clock and SM either way, measured), but
// half the issue slots.
using f32x2 = unsigned long long;
__device__ __forceinline__ f32x2 pk2(float a, float b) {
  f32x2 r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b));
  return r;
}
__device__ __forceinline__ float2 upk2(f32x2 v) {
  float2 r;
  asm("mov.b64 {%0, %1}, %2;" : "=f"(r.x), "=f"(r.y) : "l"(v));
  return r;
}
__device__ __forceinline__ f32x2 fma2(f32x2 a, f32x2 b, f32x2 c) {
  f32x2 r;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
  return r;
}
__device__ __forceinline__ f32x2 add2(f32x2 a, f32x2 b) {
  f32x2 r;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}

// ---------------------------------------------------------------------------------------------
// arithmetic policies
struct FP64P {
  using mat_t = double2;
  using vec_t = double2;
  using gv_t = double2;
  struct acc_t { double re, im; };
  static constexpr int CHUNK = 16;
  __device__ static __forceinline__ mat_t ld(const mat_t* p) { return __ldcs(p); }
  __device__ static __forceinline__ gv_t cvt(vec_t v) { return v; }
  __device__ static __forceinline__ void init(acc_t& a) { a.re = 0.0; a.im = 0.0; }
  __device__ static __forceinline__ void mac(acc_t& a, const mat_t& m, const gv_t& g) {
    a.re = fma(m.x, g.x, a.re);
    a.re = fma(-m.y, g.y, a.re);
    a.im = fma(m.x, g.y, a.im);
    a.im = fma(m.y, g.x, a.im);
  }
  __device__ static __forceinline__ void macc(acc_t& a, const mat_t& m, const gv_t& g) {  // conj(m) g
    a.re = fma(m.x, g.x, a.re);
    a.re = fma(m.y, g.y, a.re);
    a.im = fma(m.x, g.y, a.im);
    a.im = fma(-m.y, g.x, a.im);
  }
  __device__ static __forceinline__ void flush(acc_t&) {}
  __device__ static __forceinline__ vec_t fin(const acc_t& a) { return make_double2(a.re, a.im); }
  __device__ static __forceinline__ vec_t add(vec_t a, vec_t b) { return make_double2(a.x + b.x, a.y + b.y); }
  __device__ static __forceinline__ vec_t zero() { return make_double2(0.0, 0.0); }
  using part_t = double2;  // a flushed accumulator, for combining partial sums
  __device__ static __forceinline__ part_t part(const acc_t& a) { return make_double2(a.re, a.im); }
  // a partial sum plus one of lane (lane xor o)
  __device__ static __forceinline__ part_t add_lane(const part_t& keep, const part_t& send, int o) {
    return make_double2(keep.x + __shfl_xor_sync(0xffffffffu, send.x, o), keep.y + __shfl_xor_sync(0xffffffffu, send.y, o));
  }
  __device__ static __forceinline__ vec_t fin_part(const part_t& p) { return p; }
  __device__ static __forceinline__ void combine(acc_t& a, const part_t& b) { a.re += b.x; a.im += b.y; }
};

struct FP32P {
  using mat_t = float2;
  using vec_t = float2;
  using gv_t = float2;
  // (re, im) takes the running terms; flush folds it into the total (tr, ti), so that a long sum rounds
  // like a sum of short ones
  struct acc_t { float re, im, tr, ti; };
  static constexpr int CHUNK = 16;
  __device__ static __forceinline__ mat_t ld(const mat_t* p) { return __ldcs(p); }
  __device__ static __forceinline__ gv_t cvt(vec_t v) { return v; }
  __device__ static __forceinline__ void init(acc_t& a) { a.re = a.im = a.tr = a.ti = 0.f; }
  __device__ static __forceinline__ void mac(acc_t& a, const mat_t& m, const gv_t& g) {
    a.re = fmaf(m.x, g.x, a.re);
    a.re = fmaf(-m.y, g.y, a.re);
    a.im = fmaf(m.x, g.y, a.im);
    a.im = fmaf(m.y, g.x, a.im);
  }
  __device__ static __forceinline__ void macc(acc_t& a, const mat_t& m, const gv_t& g) {
    a.re = fmaf(m.x, g.x, a.re);
    a.re = fmaf(m.y, g.y, a.re);
    a.im = fmaf(m.x, g.y, a.im);
    a.im = fmaf(-m.y, g.x, a.im);
  }
  __device__ static __forceinline__ void flush(acc_t& a) {
    a.tr += a.re;
    a.ti += a.im;
    a.re = a.im = 0.f;
  }
  __device__ static __forceinline__ vec_t fin(const acc_t& a) { return make_float2(a.tr, a.ti); }
  __device__ static __forceinline__ vec_t add(vec_t a, vec_t b) { return make_float2(a.x + b.x, a.y + b.y); }
  __device__ static __forceinline__ vec_t zero() { return make_float2(0.f, 0.f); }
  using part_t = float2;
  __device__ static __forceinline__ part_t part(const acc_t& a) { return make_float2(a.tr, a.ti); }
  // a partial sum plus one of lane (lane xor o)
  __device__ static __forceinline__ part_t add_lane(const part_t& keep, const part_t& send, int o) {
    return make_float2(keep.x + __shfl_xor_sync(0xffffffffu, send.x, o), keep.y + __shfl_xor_sync(0xffffffffu, send.y, o));
  }
  __device__ static __forceinline__ vec_t fin_part(const part_t& p) { return p; }
  __device__ static __forceinline__ void combine(acc_t& a, const part_t& b) { a.tr += b.x; a.ti += b.y; }
};

// ---- double-float helpers (round-to-nearest intrinsics: never contracted into FMA) ----------
__device__ __forceinline__ void two_sum(float a, float b, float& s, float& e) {
  s = __fadd_rn(a, b);
  const float bb = __fsub_rn(s, a);
  e = __fadd_rn(__fsub_rn(a, __fsub_rn(s, bb)), __fsub_rn(b, bb));
}
__device__ __forceinline__ void fast_two_sum(float a, float b, float& s, float& e) {
  s = __fadd_rn(a, b);
  e = __fsub_rn(b, __fsub_rn(s, a));
}
// (hi, lo) += (s, c): the "sloppy" double-word addition (TwoSum of the high parts, the low
// parts added, then renormalised with Fast2Sum).
__device__ __forceinline__ void dw_accumulate(float& hi, float& lo, float s, float c) {
  float t, e;
  two_sum(hi, s, t, e);
  e = __fadd_rn(e, __fadd_rn(lo, c));
  fast_two_sum(t, e, hi, lo);
}
// The same with the error of the low parts' sum kept too (the "accurate" double-word addition), for
// the additions that are few: lanes' partial sums and the two terms of an output.
__device__ __forceinline__ void dw_add(float& hi, float& lo, float s, float c) {
  float t, e, u, v;
  two_sum(hi, s, t, e);
  two_sum(lo, c, u, v);
  fast_two_sum(t, __fadd_rn(e, u), hi, lo);
  fast_two_sum(hi, __fadd_rn(lo, v), hi, lo);
}
// s + c + d += a * b for double-float a = (ah, al), b = (bh, bl): the product of the high parts is
// split exactly (p + e, e = fma(ah, bh, -p)), the cross terms ah bl + al bh enter e, and p enters the
// running sum through TwoSum. The errors of the sum (c) and of the products (d) are added up apart:
// one rounding per term less than in a common sum.
__device__ __forceinline__ void dot2_step(float& s, float& c, float& d, float ah, float al, float bh, float bl) {
  const float p = __fmul_rn(ah, bh);
  float e = __fmaf_rn(ah, bh, -p);
  e = __fmaf_rn(ah, bl, e);
  e = __fmaf_rn(al, bh, e);
  float t, err;
  two_sum(s, p, t, err);
  s = t;
  c = __fadd_rn(c, err);
  d = __fadd_rn(d, e);
}

// The same with the errors of the sum and of the products in one sum c: a register less.
__device__ __forceinline__ void dot2_step(float& s, float& c, float ah, float al, float bh, float bl) {
  const float p = __fmul_rn(ah, bh);
  float e = __fmaf_rn(ah, bh, -p);
  e = __fmaf_rn(ah, bl, e);
  e = __fmaf_rn(al, bh, e);
  float t, err;
  two_sum(s, p, t, err);
  s = t;
  c = __fadd_rn(c, __fadd_rn(err, e));
}

struct DF64P {
  using mat_t = float4;   // (re_hi, re_lo, im_hi, im_lo)
  using vec_t = double2;
  using gv_t = float4;
  struct acc_t { float sr, cr, dr, si, ci, di, hr, lr, hi, li; };
  static constexpr int CHUNK = 16;  // terms between two folds of the warp-per-node kernel
  __device__ static __forceinline__ mat_t ld(const mat_t* p) { return __ldcs(p); }
  __device__ static __forceinline__ gv_t cvt(vec_t v) {
    const float rh = (float)v.x, ih = (float)v.y;
    return make_float4(rh, (float)(v.x - (double)rh), ih, (float)(v.y - (double)ih));
  }
  __device__ static __forceinline__ void init(acc_t& a) {
    a.sr = a.cr = a.dr = a.si = a.ci = a.di = 0.f;
    a.hr = a.lr = a.hi = a.li = 0.f;
  }
  __device__ static __forceinline__ void mac(acc_t& a, const mat_t& m, const gv_t& g) {
    dot2_step(a.sr, a.cr, a.dr, m.x, m.y, g.x, g.y);
    dot2_step(a.sr, a.cr, a.dr, -m.z, -m.w, g.z, g.w);
    dot2_step(a.si, a.ci, a.di, m.x, m.y, g.z, g.w);
    dot2_step(a.si, a.ci, a.di, m.z, m.w, g.x, g.y);
  }
  __device__ static __forceinline__ void mac_narrow(acc_t& a, const mat_t& m, const gv_t& g) {  // d is not used
    dot2_step(a.sr, a.cr, m.x, m.y, g.x, g.y);
    dot2_step(a.sr, a.cr, -m.z, -m.w, g.z, g.w);
    dot2_step(a.si, a.ci, m.x, m.y, g.z, g.w);
    dot2_step(a.si, a.ci, m.z, m.w, g.x, g.y);
  }
  __device__ static __forceinline__ void macc(acc_t& a, const mat_t& m, const gv_t& g) {
    dot2_step(a.sr, a.cr, a.dr, m.x, m.y, g.x, g.y);
    dot2_step(a.sr, a.cr, a.dr, m.z, m.w, g.z, g.w);
    dot2_step(a.si, a.ci, a.di, m.x, m.y, g.z, g.w);
    dot2_step(a.si, a.ci, a.di, -m.z, -m.w, g.x, g.y);
  }
  __device__ static __forceinline__ void flush(acc_t& a) {
    dw_accumulate(a.hr, a.lr, a.sr, __fadd_rn(a.cr, a.dr));
    dw_accumulate(a.hi, a.li, a.si, __fadd_rn(a.ci, a.di));
    a.sr = a.cr = a.dr = a.si = a.ci = a.di = 0.f;
  }
  __device__ static __forceinline__ vec_t fin(const acc_t& a) {
    return make_double2((double)a.hr + (double)a.lr, (double)a.hi + (double)a.li);
  }
  __device__ static __forceinline__ vec_t add(vec_t a, vec_t b) { return make_double2(a.x + b.x, a.y + b.y); }
  __device__ static __forceinline__ vec_t zero() { return make_double2(0.0, 0.0); }
  using part_t = float4;  // (re_hi, re_lo, im_hi, im_lo) of a flushed accumulator
  __device__ static __forceinline__ part_t part(const acc_t& a) { return make_float4(a.hr, a.lr, a.hi, a.li); }
  // a partial sum plus one of lane (lane xor o)
  __device__ static __forceinline__ part_t add_lane(const part_t& keep, const part_t& send, int o) {
    part_t r = keep;
    const float hr = __shfl_xor_sync(0xffffffffu, send.x, o), lr = __shfl_xor_sync(0xffffffffu, send.y, o);
    const float hi = __shfl_xor_sync(0xffffffffu, send.z, o), li = __shfl_xor_sync(0xffffffffu, send.w, o);
    dw_add(r.x, r.y, hr, lr);
    dw_add(r.z, r.w, hi, li);
    return r;
  }
  __device__ static __forceinline__ vec_t fin_part(const part_t& p) {
    return make_double2((double)p.x + (double)p.y, (double)p.z + (double)p.w);
  }
  __device__ static __forceinline__ void combine(acc_t& a, const part_t& b) {
    dw_accumulate(a.hr, a.lr, b.x, b.y);
    dw_accumulate(a.hi, a.li, b.z, b.w);
  }
};

// The middle factor S^h of the split-precision tensor form (IDBF_MODE_TF32X3_S64): complex64
// vectors on both sides, as on the tensor-core levels around it, with the products and sums in
// FP64 (C128 storage of S^h) or in double-float (DF64 storage). Each FP32 input is exact in the
// wider format; the output is rounded to FP32 once.
struct FP64S32P : FP64P {
  using vec_t = float2;
  __device__ static __forceinline__ gv_t cvt(vec_t v) { return make_double2((double)v.x, (double)v.y); }
  __device__ static __forceinline__ vec_t narrow(gv_t g) { return make_float2((float)g.x, (float)g.y); }
  __device__ static __forceinline__ vec_t fin_part(const part_t& p) { return make_float2((float)p.x, (float)p.y); }
  __device__ static __forceinline__ vec_t fin(const acc_t& a) { return make_float2((float)a.re, (float)a.im); }
  __device__ static __forceinline__ vec_t add(vec_t a, vec_t b) { return make_float2(a.x + b.x, a.y + b.y); }
  __device__ static __forceinline__ vec_t zero() { return make_float2(0.f, 0.f); }
};
struct DF64S32P : DF64P {
  using vec_t = float2;
  __device__ static __forceinline__ gv_t cvt(vec_t v) { return make_float4(v.x, 0.f, v.y, 0.f); }
  __device__ static __forceinline__ vec_t narrow(gv_t g) { return make_float2(g.x, g.z); }
  __device__ static __forceinline__ vec_t fin_part(const part_t& p) {
    return make_float2((float)((double)p.x + (double)p.y), (float)((double)p.z + (double)p.w));
  }
  __device__ static __forceinline__ vec_t fin(const acc_t& a) {
    return make_float2((float)((double)a.hr + (double)a.lr), (float)((double)a.hi + (double)a.li));
  }
  __device__ static __forceinline__ vec_t add(vec_t a, vec_t b) { return make_float2(a.x + b.x, a.y + b.y); }
  __device__ static __forceinline__ vec_t zero() { return make_float2(0.f, 0.f); }
};

// Vectors between levels. With DF set the double-float policy keeps them in its own format, (re_hi,
// re_lo, im_hi, im_lo) floats (16 bytes, like complex128), so that gathering a level's operands, adding
// its pass-through terms and writing its outputs take no FP64 arithmetic (GB300 issues FP64 at a small
// fraction of the FP32 rate); only the first level converts the complex128 x and the last the
// complex128 y. A pair holds 48 bits of the 53, as much as the operands of the products; with
// complex128 between levels the errors are within 4 % of these, and nine vectors at N = 40960 take 880
// us against 763. Otherwise the boundary vectors are the policy's vec_t.
template <class P, bool DF>
struct Bnd {
  using b_t = typename P::vec_t;
  __device__ static __forceinline__ b_t of_v(typename P::vec_t v) { return v; }
  __device__ static __forceinline__ typename P::vec_t v_of(b_t b) { return b; }
  __device__ static __forceinline__ typename P::gv_t g_of(b_t b) { return P::cvt(b); }
  __device__ static __forceinline__ b_t b_of_g(const typename P::gv_t& g) {
    if constexpr (std::is_same<b_t, typename P::gv_t>::value) return g;
    else return P::narrow(g);
  }
  __device__ static __forceinline__ b_t of_acc(const typename P::acc_t& a) { return P::fin(a); }
  __device__ static __forceinline__ b_t of_part(const typename P::part_t& a) { return P::fin_part(a); }
  __device__ static __forceinline__ b_t add(b_t a, b_t b) { return P::add(a, b); }
  __device__ static __forceinline__ b_t zero() { return P::zero(); }
};
template <>
struct Bnd<DF64P, true> {
  using b_t = float4;
  __device__ static __forceinline__ b_t of_v(double2 v) { return DF64P::cvt(v); }  // exact split
  __device__ static __forceinline__ double2 v_of(b_t b) {  // exact: 48 bits in a double
    return make_double2((double)b.x + (double)b.y, (double)b.z + (double)b.w);
  }
  __device__ static __forceinline__ float4 g_of(b_t b) { return b; }
  __device__ static __forceinline__ b_t b_of_g(const float4& g) { return g; }
  // a flushed accumulator: its (hi, lo) pairs, of the value fin() rounds exactly into a double
  __device__ static __forceinline__ b_t of_acc(const DF64P::acc_t& a) { return DF64P::part(a); }
  __device__ static __forceinline__ b_t of_part(const float4& a) { return a; }
  __device__ static __forceinline__ b_t add(b_t a, b_t b) {
    dw_add(a.x, a.y, b.x, b.y);
    dw_add(a.z, a.w, b.z, b.w);
    return a;
  }
  __device__ static __forceinline__ b_t zero() { return make_float4(0.f, 0.f, 0.f, 0.f); }
};
static_assert(sizeof(Bnd<DF64P, true>::b_t) == sizeof(DF64P::vec_t), "boundary elements keep their size");

template <class P> constexpr int fmt_of();
template <> constexpr int fmt_of<FP64P>() { return IDBF_STORE_C128; }
template <> constexpr int fmt_of<DF64P>() { return IDBF_STORE_DF64; }
template <> constexpr int fmt_of<FP32P>() { return IDBF_STORE_C64; }
template <> constexpr int fmt_of<FP64S32P>() { return IDBF_STORE_C128; }
template <> constexpr int fmt_of<DF64S32P>() { return IDBF_STORE_DF64; }

// ---------------------------------------------------------------------------------------------
// the vectors of a level
template <class V>
struct IO {
  const V* x;  // user input (forward: level 0; adjoint: level L)
  int64_t ldx;
  V* y;        // user output (forward: level L; adjoint: level 0)
  int64_t ldy;
  const V* win;  // workspace boundary read
  V* wout;       // workspace boundary written
  int R;
};

__device__ __forceinline__ int64_t out_seg_id(const DevLevel& d, int64_t j, int c) {
  return (j / d.H) * 2 * d.H + j % d.H + c * d.H;
}

namespace node {
// Asks for `bytes` at p (rounded out to 16-byte granules, which the arenas' tails allow) in L2: one
// instruction streams a whole block from HBM while the CTA is still loading its index lists and
// inputs, so that the product loop's loads meet L2 latency instead of HBM latency.
__device__ __forceinline__ void prefetch_l2(const void* p, int64_t bytes) {
  const uintptr_t a = (uintptr_t)p & ~(uintptr_t)15;
  const uint32_t n = (uint32_t)((((uintptr_t)p + bytes + 15) & ~(uintptr_t)15) - a);
  if (bytes > 0) asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(a), "r"(n) : "memory");
}
// A level's launch may begin while the previous level still runs (launch_after in node.cu): what
// comes before wait_for_inputs reads the factors only. next_may_begin lets the following launch
// begin once every CTA of this one has started.
__device__ __forceinline__ void wait_for_inputs() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void next_may_begin() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
}  // namespace node

// ---------------------------------------------------------------------------------------------
// Warp-per-node forward body, one right-hand side, for levels of short blocks (the outer levels
// of the butterfly: leaves and their neighbours). Every phase of a node (inputs, gathered operands,
// block products, combination) is done by one warp with __syncwarp between phases, so a CTA has
// as many nodes in flight as it has warps and no phase waits for another warp. Lanes cover the
// rows of a block, RPL rows each (rows <= 32 RPL); a column of a block is read by the warp as
// consecutive entries. Shared memory per warp: u[max_in] (inputs), g[2][gcap] (gathered
// operands), t[max_out] (row-ID accumulation of a U level).
template <class P>
__host__ __device__ constexpr size_t warp_node_smem(int max_in, int gcap, int max_out) {
  return (((size_t)max_in * sizeof(typename P::vec_t) + 2 * (size_t)gcap * sizeof(typename P::gv_t) +
           (size_t)max_out * sizeof(typename P::vec_t)) + 15) & ~(size_t)15;
}

template <class P, int RPL>
__device__ __forceinline__ void fwd_node_warp(const DevLevel& d, const typename P::mat_t* __restrict__ mat,
                                              const IO<typename P::vec_t>& io, int max_in, int gcap, int64_t j,
                                              unsigned char* wsm) {
  using V = typename P::vec_t;
  using G = typename P::gv_t;
  using M = typename P::mat_t;
  using BP = Bnd<P, std::is_same<P, DF64P>::value>;
  using B = typename BP::b_t;
  V* u = (V*)wsm;
  B* ub = (B*)u;  // the inputs of a level > 0, in the boundary format
  G* g = (G*)(u + max_in);
  B* t = (B*)(g + 2 * (size_t)gcap);
  const B* winb = (const B*)io.win;
  B* woutb = (B*)io.wout;
  const int lane = threadIdx.x & 31;

  // inputs -> u
  int l0, l1;
  if (d.lev == 0) {
    l0 = d.n0;
    l1 = 0;
    for (int e = lane; e < l0; e += 32) u[e] = io.x[j * d.n0 + e];
  } else {
    l0 = d.in_len[2 * j];
    l1 = d.in_len[2 * j + 1];
    const int64_t o0 = d.in_off[2 * j], o1 = d.in_off[2 * j + 1];
    for (int e = lane; e < l0 + l1; e += 32) ub[e] = winb[(e < l0 ? o0 + e : o1 + (e - l0)) * io.R];
  }
  const bool lev0 = d.lev == 0;
  auto gin = [&](int e) -> G { return lev0 ? P::cvt(u[e]) : BP::g_of(ub[e]); };
  auto bin = [&](int e) -> B { return lev0 ? BP::of_v(u[e]) : ub[e]; };
  const int rowsv[2] = {d.rows[2 * j], d.rows[2 * j + 1]};
  const int colsv[2] = {d.cols[2 * j], d.cols[2 * j + 1]};
  const int64_t mov[2] = {d.moff[2 * j], d.moff[2 * j + 1]};
  const int32_t* ixv[2] = {d.idx + d.ioff[2 * j], d.idx + d.ioff[2 * j + 1]};
  __syncwarp();

  // gathered operands -> g
  if (d.kind == KIND_V) {
#pragma unroll
    for (int c = 0; c < 2; ++c)
      for (int k = lane; k < colsv[c]; k += 32) g[c * gcap + k] = gin(ixv[c][rowsv[c] + k]);
  } else if (d.kind == KIND_S) {
    for (int e = lane; e < l0 + l1; e += 32) g[e] = gin(e);
  } else {
    for (int e = lane; e < l0; e += 32) g[e] = gin(e);
    for (int e = lane; e < l1; e += 32) g[gcap + e] = gin(l0 + e);
  }
  __syncwarp();

  // block products: lane owns rows lane + 32 i
  B res[2][RPL];
#pragma unroll
  for (int c = 0; c < 2; ++c) {
    const int rows = rowsv[c], cols = colsv[c];
    const M* Mc = mat + mov[c];
    const G* gc = g + (d.kind == KIND_S ? 0 : c * gcap);
    // two accumulators per row (even and odd columns): two independent dependency chains
    typename P::acc_t acc0[RPL], acc1[RPL];
#pragma unroll
    for (int i = 0; i < RPL; ++i) {
      P::init(acc0[i]);
      P::init(acc1[i]);
    }
    auto pair = [&](int kk) {  // columns kk (into acc0) and kk + 1 (into acc1)
      const G g0 = gc[kk], g1 = gc[kk + 1];
#pragma unroll
      for (int i = 0; i < RPL; ++i) {
        const int r = lane + 32 * i;
        if (r < rows) {
          P::mac(acc0[i], P::ld(Mc + (int64_t)kk * rows + r), g0);
          P::mac(acc1[i], P::ld(Mc + (int64_t)(kk + 1) * rows + r), g1);
        }
      }
    };
    int k = 0;
    for (; k + 2 * P::CHUNK <= cols; k += 2 * P::CHUNK) {
#pragma unroll 4
      for (int q = 0; q < 2 * P::CHUNK; q += 2) pair(k + q);
#pragma unroll
      for (int i = 0; i < RPL; ++i) {
        P::flush(acc0[i]);
        P::flush(acc1[i]);
      }
    }
    for (; k + 1 < cols; k += 2) pair(k);
    if (k < cols) {
      const G g0 = gc[k];
#pragma unroll
      for (int i = 0; i < RPL; ++i) {
        const int r = lane + 32 * i;
        if (r < rows) P::mac(acc0[i], P::ld(Mc + (int64_t)k * rows + r), g0);
      }
    }
#pragma unroll
    for (int i = 0; i < RPL; ++i) {
      P::flush(acc0[i]);
      P::flush(acc1[i]);
      P::combine(acc0[i], P::part(acc1[i]));
      res[c][i] = BP::of_acc(acc0[i]);
    }
    if (d.kind != KIND_U) {
      const int64_t ob = d.out_off[out_seg_id(d, j, c)];
#pragma unroll
      for (int i = 0; i < RPL; ++i) {
        const int r = lane + 32 * i;
        if (r >= rows) continue;
        B v = res[c][i];
        if (d.kind == KIND_V) v = BP::add(v, bin(ixv[c][r]));
        woutb[(ob + r) * io.R] = v;
      }
    }
  }
  if (d.kind != KIND_U) return;
  // row-ID level: t[q_c] = in_c, t[p_c] = res_c, block 0 first (q_0, p_0 partition t), then
  // block 1 adds (q_1, p_1 also a partition)
  const int tl = l0 + rowsv[0];
  for (int e = lane; e < l0; e += 32) t[ixv[0][e]] = bin(e);
#pragma unroll
  for (int i = 0; i < RPL; ++i) {
    const int r = lane + 32 * i;
    if (r < rowsv[0]) t[ixv[0][l0 + r]] = res[0][i];
  }
  __syncwarp();
  for (int e = lane; e < l1; e += 32) {
    B* dst = &t[ixv[1][e]];
    *dst = BP::add(*dst, bin(l0 + e));
  }
#pragma unroll
  for (int i = 0; i < RPL; ++i) {
    const int r = lane + 32 * i;
    if (r < rowsv[1]) {
      B* dst = &t[ixv[1][l1 + r]];
      *dst = BP::add(*dst, res[1][i]);
    }
  }
  __syncwarp();
  if (d.lev == d.L) {
    for (int e = lane; e < tl; e += 32) io.y[j * d.n0 + e] = BP::v_of(t[e]);
  } else {
    const int64_t s0 = out_seg_id(d, j, 0), s1 = out_seg_id(d, j, 1);
    const int len0 = d.out_len[s0];
    const int64_t b0 = d.out_off[s0], b1 = d.out_off[s1];
    for (int e = lane; e < tl; e += 32) woutb[(e < len0 ? b0 + e : b1 + (e - len0)) * io.R] = t[e];
  }
}

}  // namespace idbf

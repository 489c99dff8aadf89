// The items of the batch's persistent launch: how an operator's right-hand sides are cut into items
// and an item's into passes of the node body, and the shared memory those passes take. The kernel and
// the code that sizes its launch share these rules.
#pragma once

#include <algorithm>
#include <type_traits>

#include "idbf_internal.h"
#include "node_kernels.cuh"

namespace idbf {
namespace bat {

template <class P>
__host__ __device__ constexpr int max_rb() {
  return std::is_same<P, FP32P>::value ? 32 : std::is_same<P, FP64P>::value ? 16 : 8;
}
// Right-hand sides that one pass of the body holds: 2 in FP64 and 4 else (8 in FP64 and FP32 spill in the
// kernel's 128 registers; 24 operators of N = 2^9 .. 2^14, 4 per item: FP64 11.3 against 12.2 ms, but 10.3 with
// items of one; FP32 2710 against 2570 us).
template <class P>
__host__ __device__ constexpr int pass_rb() {
  return std::is_same<P, FP64P>::value ? 2 : 4;
}

// The body's width for an item of at most w right-hand sides in one pass: calls f with it.
template <class P, class F>
__host__ __device__ __forceinline__ void at_width(int w, F f) {
  using std::integral_constant;
  if constexpr (pass_rb<P>() > 2) {
    if constexpr (std::is_same<P, DF64P>::value) {
      if (w == 3) return f(integral_constant<int, 3>(), integral_constant<int, 1>(), integral_constant<int, 2>());
    }
    if (w > 2) return f(integral_constant<int, 4>(), integral_constant<int, 1>(), integral_constant<int, 2>());
  }
  if (w > 1) return f(integral_constant<int, 2>(), integral_constant<int, 1>(), integral_constant<int, 4>());
  return f(integral_constant<int, 1>(), integral_constant<int, 1>(), integral_constant<int, 4>());
}

// Right-hand sides per pass of an item of n: as few passes as the registers allow, as even as possible.
template <class P>
__host__ __device__ constexpr int pass_width(int n) {
  const int passes = (n + pass_rb<P>() - 1) / pass_rb<P>();
  return (n + passes - 1) / passes;
}

template <class P>
size_t node_smem(const LevelInfo& li, int pw) {
  size_t n = 0;
  at_width<P>(pw, [&](auto rb, auto, auto) {
    n = node::fwd_smem<P, decltype(rb)::value>(li.max_in, li.max_out, li.max_rows, li.max_cols, li.max_rows_pair,
                                               li.kind == KIND_U);
  });
  return n;
}

// The shared memory of any item of an operator with R right-hand sides in items of `width`. The last
// item may be shorter and yet run a wider body: double-float, R = 9 in items of five: 5 vectors take
// two passes of three, the last 4 one pass of four.
template <class P>
size_t items_smem(const LevelInfo& li, int64_t R, int width) {
  const int last = (int)((R - 1) % width) + 1;
  return std::max(node_smem<P>(li, pass_width<P>((int)std::min<int64_t>(width, R))), node_smem<P>(li, pass_width<P>(last)));
}

}  // namespace bat
}  // namespace idbf

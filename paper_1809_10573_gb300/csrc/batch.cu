// An uneven batch of IDBF applies (operators of different N, each with its own number of
// right-hand sides) as one CUDA graph, in one of two forms (a tile, autotuned).
//
// Level launches: every width of right-hand-side block in the batch is a chain of launches, one per
// level, each over all operators of that width; the chains run side by side, and a launch begins
// (index lists, factor reads) while its predecessor drains. Each launch has the shared memory, the
// threads and the registers of its own level and width.
//
// Persistent launch: work items (operator, level, run of nodes, block of right-hand sides) are
// queued in the order of the levels (all level-0 items of every operator, then all level-1 items,
// ...), and persistent CTAs take them from the queue with an atomic counter. Before starting an
// item of level l, a CTA waits until every item of level l-1 of the same operator has finished (a
// per-(operator, level) completion counter). Those items are earlier in the queue, so they have
// already been taken by CTAs that are running, and the wait ends: there is no cycle, whatever the
// number of resident CTAs. (A CTA holds one item ahead of the one it computes; of all unfinished items
// the earliest in the queue is always one being computed.) Every wait is bounded in time; on a
// timeout the item runs all the same (its results are invalid) and is counted as done, bit 0 of the
// status word is set, and idbf_batch_sync_status reports IDBF_ETIMEOUT.
//
// Each node is computed by node::fwd_body, the body of the per-level kernels (node_kernels.cuh).
#include <cuda_runtime.h>
#include <string.h>

#include <algorithm>
#include <new>
#include <type_traits>
#include <vector>

#include "batch_items.cuh"
#include "idbf_internal.h"
#include "node_kernels.cuh"
#include "node_launch.h"

namespace idbf {
namespace bat {

struct OpLevel {
  DevLevel d;
  const void* mat;
  int max_in, max_out, max_rows, max_cols, max_rows_pair, pad;
};
struct OpDesc {
  int L, R, level_base;
  int width;  // right-hand sides per item
  void* ws0;
  void* ws1;
};
struct Item {
  int op, level, node0, nodes, r0, pad;
};
struct LevelItem {  // a CTA of a level launch: slice sl of nsl of each of `nodes` nodes
  int op, node0, nodes, r0, sl, nsl;
};

__device__ __forceinline__ uint64_t gtimer() {
  uint64_t t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}

constexpr int NTMAX = 256;
constexpr size_t kSmemCap = 200 * 1024;  // per CTA

// Tiles: right-hand sides per work item (rb; above the body's width in several passes), threads per
// CTA of the persistent launch, or 0 for level launches, one chain of launches per width of the
// batch's operators: with rb = 8 in the instances of the per-level kernels (most CTAs resident),
// with rb = 16 in instances of more registers per CTA, whose tall nodes finish sooner, with rb = 4 in
// narrow ones, of which a small batch has fewer chains. In FP32 ten operators of N = 2^10 .. 2^11 take 149
// us with rb = 4, 156 with 16, 169 with 8, and 24 of N = 2^9 .. 2^14 1475, 1195 and 1132 us. FP64, bound by
// its pipe, prefers persistent launches of one right-hand side per item (the same batches: 1030 and
// 10310 us with 128 threads, 1114 and 12150 with 256, 1090 and 10860 as level launches).
struct Tile {
  int rb, nt;
  bool wide;  // FP32 and FP64 only
};
constexpr Tile kTiles[] = {{1, 256, false}, {4, 256, false}, {8, 128, false}, {8, 0, false},
                           {8, 256, true},  {16, 0, true},   {32, 256, true}, {16, 128, true},
                           {4, 0, false},   {1, 128, false}};
constexpr int kNumTiles = 10;
// One node at one width. Not inlined: the widths of a precision share the kernel's registers.
// dep: the completion counter that the item waits for (nullptr: no wait).
struct Dep {
  const volatile int* done;
  int need;
  uint64_t limit_ns;
  int* status;
};
template <class P, int RB, int TR, int U>
__device__ __noinline__ void batch_node(const OpLevel& ol, const IO<typename P::vec_t>& io, int64_t j, int r, int r1,
                                        unsigned char* smem, const Dep& dep) {
  node::fwd_body<P, RB, TR, U, false>(
      ol.d, (const typename P::mat_t*)ol.mat, io, ol.max_in, ol.max_out, ol.max_rows, ol.max_cols, ol.max_rows_pair, j, 0, 1,
      r, r1, smem, [&] {
        if (!dep.done) return;
        if (threadIdx.x == 0) {
          if (*dep.done < dep.need) {
            const uint64_t t0 = gtimer();
            while (*dep.done < dep.need) {
              if (gtimer() - t0 > dep.limit_ns) {
                atomicOr(dep.status, 1);
                break;
              }
            }
          }
          __threadfence();  // acquire: the previous level's outputs are visible
        }
        __syncthreads();
      });
}

// W: the widest pass, 1 for items of one right-hand side (three CTAs of 256 threads per SM) or the
// policy's.
template <class P, int W>
__global__ void __launch_bounds__(NTMAX, W == 1 ? 3 : 2)
    k_batch(const OpDesc* __restrict__ ops, const OpLevel* __restrict__ lv, const Item* __restrict__ items, int nitems,
            const void* const* xs, void* const* ys, const int64_t* lds, int* head, int* done,
            const int* __restrict__ target, int* status, uint64_t limit_ns) {
  using V = typename P::vec_t;
  using M = typename P::mat_t;
  extern __shared__ __align__(16) unsigned char smem[];
  __shared__ int sidx;
  __shared__ OpLevel ol;  // the item's level and vectors
  __shared__ IO<V> io;
  if (threadIdx.x == 0) sidx = atomicAdd(head, 1);
  for (;;) {
    __syncthreads();
    const int i = sidx;
    if (i >= nitems) break;
    const Item w = items[i];
    const OpDesc od = ops[w.op];
    const int li = od.level_base + w.level;
    __syncthreads();  // every thread has read sidx and is past the previous item's shared memory
    static_assert(sizeof(OpLevel) % 4 == 0, "copied in words");
    if (threadIdx.x >= 32 && threadIdx.x < 64)
      for (int q = threadIdx.x - 32; q < (int)(sizeof(OpLevel) / 4); q += 32) ((uint32_t*)&ol)[q] = ((const uint32_t*)(lv + li))[q];
    if (threadIdx.x == 32) {
      io.x = (const V*)xs[w.op];
      io.ldx = lds[w.op];
      io.y = (V*)ys[w.op];
      io.ldy = lds[w.op];
      io.R = od.R;
      io.win = w.level > 0 ? (const V*)(w.level & 1 ? od.ws0 : od.ws1) : nullptr;
      io.wout = w.level < od.L ? (V*)(w.level & 1 ? od.ws1 : od.ws0) : nullptr;
    }
    if (threadIdx.x == 0) {
      const int nxt = atomicAdd(head, 1);
      sidx = nxt;
      if (nxt < nitems) {  // the next item's blocks (contiguous over a run of nodes) into L2
        const Item nw = items[nxt];
        const OpLevel& nl = lv[ops[nw.op].level_base + nw.level];
        const int64_t a = nl.d.moff[2 * nw.node0], e = 2 * (int64_t)(nw.node0 + nw.nodes) - 1;
        const int64_t n = nl.d.moff[e] + (int64_t)nl.d.rows[e] * nl.d.cols[e] - a;
        if (nw.r0 == 0 && n * (int64_t)sizeof(M) < (1 << 22)) node::prefetch_l2((const M*)nl.mat + a, n * (int64_t)sizeof(M));
      }
    }
    __syncthreads();
    {
      // only the item's first node and pass wait, after their index lists and first factor columns
      // are on their way
      Dep dep = {w.level > 0 ? done + (li - 1) : nullptr, w.level > 0 ? target[li - 1] : 0, limit_ns, status};
      const int r1 = min(od.R, w.r0 + od.width);
      const int pw = pass_width<P>(r1 - w.r0);
      for (int n = 0; n < w.nodes; ++n)
        for (int r = w.r0; r < r1; r += pw) {
          if (n || r != w.r0) __syncthreads();
          if constexpr (W == 1)
            batch_node<P, 1, 1, 4>(ol, io, (int64_t)(w.node0 + n), r, r + 1, smem, dep);
          else
            at_width<P>(pw, [&](auto rb, auto tr, auto u) {
              batch_node<P, decltype(rb)::value, decltype(tr)::value, decltype(u)::value>(
                  ol, io, (int64_t)(w.node0 + n), r, min(r + pw, r1), smem, dep);
            });
          dep.done = nullptr;
        }
    }
    __threadfence();  // release: this item's outputs before its completion count
    __syncthreads();
    if (threadIdx.x == 0) atomicAdd(done + li, 1);
  }
}

// One level of the operators of one width: a CTA per item. Everything before the body's
// wait_for_inputs (the item, its level's description, the factors) is independent of the previous
// level's launch.
template <class P, int RB, int TR, int U, int NTL, int MINB>
__global__ void __launch_bounds__(NTL, MINB)
    k_batch_level(const LevelItem* __restrict__ items, const OpDesc* __restrict__ ops, const OpLevel* __restrict__ lv,
                  int level, const void* const* xs, void* const* ys, const int64_t* lds) {
  using V = typename P::vec_t;
  extern __shared__ __align__(16) unsigned char smem[];
  __shared__ OpLevel ol;
  __shared__ IO<V> io;
  __shared__ LevelItem it;
  node::next_may_begin();
  if (threadIdx.x < 32) {
    const LevelItem q = items[blockIdx.x];
    const OpDesc od = ops[q.op];
    const uint32_t* src = (const uint32_t*)(lv + od.level_base + level);
    for (int w = threadIdx.x; w < (int)(sizeof(OpLevel) / 4); w += 32) ((uint32_t*)&ol)[w] = src[w];
    if (threadIdx.x == 0) {
      it = q;
      io.x = (const V*)xs[q.op];
      io.ldx = lds[q.op];
      io.y = (V*)ys[q.op];
      io.ldy = lds[q.op];
      io.R = od.R;
      io.win = level > 0 ? (const V*)(level & 1 ? od.ws0 : od.ws1) : nullptr;
      io.wout = level < od.L ? (V*)(level & 1 ? od.ws1 : od.ws0) : nullptr;
    }
  }
  __syncthreads();
  for (int n = 0; n < it.nodes; ++n) {
    if (n) __syncthreads();
    node::fwd_body<P, RB, TR, U, false>(ol.d, (const typename P::mat_t*)ol.mat, io, ol.max_in, ol.max_out, ol.max_rows,
                                        ol.max_cols, ol.max_rows_pair, (int64_t)(it.node0 + n), it.sl, it.nsl, it.r0,
                                        min(it.r0 + RB, io.R), smem, [] { node::wait_for_inputs(); });
  }
}

// right-hand sides that a level launch's instance holds in registers
template <class P>
constexpr int level_rb() {
  return std::is_same<P, DF64P>::value ? 4 : 8;
}

// The instances of the level launches, as the per-level kernels of node.cu: calls f with
// (right-hand sides, rows per thread, columns in flight, threads, CTAs per SM) for items of w
// right-hand sides.
template <class P, class F>
void at_level_width(int w, bool few, F f) {
#define IDBF_W(RB, TR, U, NT, MB)                                                                              \
  return f(std::integral_constant<int, RB>(), std::integral_constant<int, TR>(), std::integral_constant<int, U>(), \
           std::integral_constant<int, NT>(), std::integral_constant<int, MB>())
  if constexpr (std::is_same<P, FP32P>::value) {
    if (w > 6 && few) IDBF_W(8, 1, 4, 256, 2);
    if (w > 6) IDBF_W(8, 1, 4, 256, 3);
    if (w > 4) IDBF_W(6, 1, 4, 256, 3);
    if (w > 2) IDBF_W(4, 1, 4, 256, 3);
    if (w > 1) IDBF_W(2, 1, 8, 256, 3);
    IDBF_W(1, 1, 6, 256, 4);
  } else if constexpr (std::is_same<P, FP64P>::value) {
    if (w > 5) IDBF_W(7, 1, 2, 256, 2);
    if (w > 4) IDBF_W(5, 1, 4, 256, 2);
    if (w > 3) IDBF_W(4, 1, 4, 256, 2);
    if (w > 2) IDBF_W(3, 1, 4, 256, 2);
    if (w > 1) IDBF_W(2, 1, 4, 256, 2);
    IDBF_W(1, 1, 8, 256, 3);
  } else {
    if (w > 3) IDBF_W(4, 1, 2, 256, 2);
    if (w > 2) IDBF_W(3, 1, 2, 256, 2);
    if (w > 1) IDBF_W(2, 1, 4, 256, 2);
    IDBF_W(1, 1, 4, 256, 3);
  }
#undef IDBF_W
}

}  // namespace bat
}  // namespace idbf

using namespace idbf;

struct idbf_batch_s {
  int device = 0, nops = 0, mode = 0, fmt = 0;
  std::vector<idbf_plan> plans;
  std::vector<int64_t> R;
  std::vector<void*> ws;
  bat::OpDesc* d_ops = nullptr;
  bat::OpLevel* d_lv = nullptr;
  int nlevels_total = 0;
  bat::Item* d_items = nullptr;
  int nitems = 0;
  int* d_counters = nullptr;  // head, then done[nlevels_total]
  int* d_target = nullptr;
  int* d_status = nullptr;
  void** d_ptrs = nullptr;    // xs[nops], ys[nops], then lds[nops] (int64)
  int tile = 1, rb = 4, npi = 1;  // tile: index into bat::kTiles
  std::vector<bat::OpDesc> h_ops; // host copy of the operator table (the item widths change with the tile)
  size_t smem = 0;
  int ctas = 0;
  uint64_t limit_ns = 2000000000ull;
  int debug_extra = 0;  // fault injection: added to the first operator's level-0 completion target
  int64_t split_n = INT64_MAX;  // operators with N >= split_n run through idbf_apply, not the launch
  bool split_auto = true;       // idbf_batch_autotune chooses split_n
  std::vector<char> sep;        // per operator: runs through idbf_apply
  cudaGraph_t graph = nullptr;
  cudaGraphExec_t exec = nullptr;
  cudaStream_t cap = nullptr;
  // level launches (tiles with nt = 0): every width of the batch is a chain of launches, one per
  // level, of its own stream during the capture
  struct LevelLaunch {
    int width, level, first, count, nt;
    size_t smem;
  };
  std::vector<LevelLaunch> level_launches;  // by width, then level
  bat::LevelItem* d_litems = nullptr;
  std::vector<cudaStream_t> side;           // capture streams of the second and later widths
  cudaEvent_t ev_fork = nullptr;
  std::vector<cudaEvent_t> ev_join;
};

namespace {

void free_layout(idbf_batch_s* b) {
  if (b->exec) cudaGraphExecDestroy(b->exec);
  if (b->graph) cudaGraphDestroy(b->graph);
  b->exec = nullptr;
  b->graph = nullptr;
  if (b->d_items) cudaFree(b->d_items);
  if (b->d_litems) cudaFree(b->d_litems);
  b->d_litems = nullptr;
  b->level_launches.clear();
  if (b->d_target) cudaFree(b->d_target);
  if (b->d_counters) cudaFree(b->d_counters);
  b->d_items = nullptr;
  b->d_target = nullptr;
  b->d_counters = nullptr;
}

// The fault injection of idbf_batch_debug_set_wait needs the persistent launch's waits: while it is
// set, tiles of level launches run as a persistent one.
bool level_launched(const idbf_batch_s* b) { return bat::kTiles[b->tile].nt == 0 && b->debug_extra == 0; }
int persistent_threads(const idbf_batch_s* b) { return bat::kTiles[b->tile].nt ? bat::kTiles[b->tile].nt : bat::NTMAX; }

// The launches of every width and level and their items, for the current tile.
template <class P>
idbf_status plan_levels(idbf_batch_s* b, std::vector<bat::LevelItem>& items) {
  const int cap = std::min(b->rb, bat::level_rb<P>());
  constexpr bool kFp64 = std::is_same<P, FP64P>::value;
  std::vector<int> widths;  // instance widths in use
  std::vector<int> cls(b->nops, 0);
  int maxL = 0;
  for (int o = 0; o < b->nops; ++o) {
    if (b->sep[o]) continue;
    int w = 0;
    const int want = kFp64 ? node::fitting_block(b->R[o]) : node::even_block(b->R[o], cap);
    bat::at_level_width<P>(want, b->rb > 8, [&](auto rb, auto, auto, auto, auto) { w = decltype(rb)::value; });
    cls[o] = w;
    if (std::find(widths.begin(), widths.end(), w) == widths.end()) widths.push_back(w);
    maxL = std::max(maxL, b->plans[o]->p.L);
  }
  std::sort(widths.begin(), widths.end(), [](int x, int y) { return x > y; });
  // few nodes on a level over the whole batch: cut them as the single apply does. FP64 counts each
  // operator's nodes alone, and cuts to one CTA per SM: its chains share one slow pipe and end together
  // only in small items, but every slice repeats a node's preparation (24 operators of N = 2^9 .. 2^14: 10860
  // us, with two CTAs 11210, four 11680; double-float and complex64, whose chains fill one another's
  // gaps, lose by counts of their own: 421 us against 316 and 199 against 154 for five operators of
  // N = 1024 .. 8192)
  std::vector<int64_t> nodes(maxL + 1, 0);
  for (int o = 0; o < b->nops; ++o)
    for (int l = 0; !b->sep[o] && l <= b->plans[o]->p.L; ++l)
      nodes[l] += (int64_t)b->plans[o]->p.m * ((b->R[o] + cls[o] - 1) / cls[o]);
  for (const int w : widths)
    for (int l = 0; l <= maxL; ++l) {
      idbf_batch_s::LevelLaunch q{w, l, (int)items.size(), 0, 0, 0};
      for (int o = 0; o < b->nops; ++o) {
        const Plan& p = b->plans[o]->p;
        if (b->sep[o] || cls[o] != w || l > p.L) continue;
        const LevelInfo& li = p.lv[l];
        const int nsl = node::slices(kFp64 ? (int64_t)p.m * ((b->R[o] + w - 1) / w) : nodes[l], node::fwd_span(li), kFp64 ? 1 : 4);
        bat::at_level_width<P>(w, b->rb > 8, [&](auto rb, auto tr, auto, auto ntl, auto) {
          q.smem = std::max(q.smem, node::fwd_smem<P, decltype(rb)::value>(li.max_in, li.max_out, li.max_rows, li.max_cols,
                                                                            li.max_rows_pair, li.kind == KIND_U));
          q.nt = std::max(q.nt, node::fwd_threads(li, decltype(tr)::value, nsl, decltype(ntl)::value));
        });
        // the right-hand-side blocks of a slice are adjacent, so that their reads meet in L2
        const int npi = nsl > 1 ? 1 : b->npi;
        for (int n0 = 0; n0 < p.m; n0 += npi)
          for (int sl = 0; sl < nsl; ++sl)
            for (int64_t r0 = 0; r0 < b->R[o]; r0 += w)
              items.push_back({o, n0, std::min(npi, p.m - n0), (int)r0, sl, nsl});
      }
      q.count = (int)items.size() - q.first;
      if (q.smem > bat::kSmemCap) return IDBF_EUNSUPPORTED;
      if (q.count > 0) b->level_launches.push_back(q);
    }
  return IDBF_OK;
}

template <class P>
idbf_status launch_levels(idbf_batch_s* b, cudaStream_t st) {
  const void* const* xs = (const void* const*)b->d_ptrs;
  void* const* ys = (void* const*)(b->d_ptrs + b->nops);
  const int64_t* lds = (const int64_t*)(b->d_ptrs + 2 * b->nops);
  IDBF_CUDA_TRY(cudaEventRecord(b->ev_fork, st));
  int chain = -1, width = 0;
  cudaStream_t cs = st;
  auto join = [&]() -> cudaError_t {  // the chain that just ended rejoins the main stream
    if (chain <= 0) return cudaSuccess;
    const cudaError_t e = cudaEventRecord(b->ev_join[chain - 1], cs);
    return e != cudaSuccess ? e : cudaStreamWaitEvent(st, b->ev_join[chain - 1], 0);
  };
  for (size_t k = 0; k < b->level_launches.size(); ++k) {
    const auto& q = b->level_launches[k];
    const bool first = q.width != width;
    if (first) {
      if (++chain > 0) {
        if ((int)b->side.size() < chain) {
          cudaStream_t s = nullptr;
          cudaEvent_t ev = nullptr;
          IDBF_CUDA_TRY(cudaStreamCreateWithFlags(&s, cudaStreamNonBlocking));
          const cudaError_t e = cudaEventCreateWithFlags(&ev, cudaEventDisableTiming);
          if (e != cudaSuccess) cudaStreamDestroy(s);
          IDBF_CUDA_TRY(e);
          b->side.push_back(s);
          b->ev_join.push_back(ev);
        }
        cs = b->side[chain - 1];
        IDBF_CUDA_TRY(cudaStreamWaitEvent(cs, b->ev_fork, 0));
      }
      width = q.width;
    }
    cudaError_t e = cudaSuccess;
    bat::at_level_width<P>(q.width, b->rb > 8, [&](auto rb, auto tr, auto u, auto ntl, auto mb) {
      auto kern = bat::k_batch_level<P, decltype(rb)::value, decltype(tr)::value, decltype(u)::value, decltype(ntl)::value,
                                     decltype(mb)::value>;
      if (q.smem > 48 * 1024) e = allow_smem(kern, bat::kSmemCap);
      if (e == cudaSuccess)
        e = node::launch_after(kern, !first, (int64_t)q.count, q.nt, q.smem, cs, (const bat::LevelItem*)b->d_litems + q.first,
                               (const bat::OpDesc*)b->d_ops, (const bat::OpLevel*)b->d_lv, q.level, xs, ys, lds);
    });
    IDBF_CUDA_TRY(e);
    const bool last = k + 1 == b->level_launches.size() || b->level_launches[k + 1].width != width;
    if (last) IDBF_CUDA_TRY(join());
  }
  return IDBF_OK;
}

// the instance of the persistent kernel for the current tile
template <class P>
auto* batch_kernel(const idbf_batch_s* b) {
  return b->rb == 1 ? bat::k_batch<P, 1> : bat::k_batch<P, bat::pass_rb<P>()>;
}

template <class P>
idbf_status launch_batch(idbf_batch_s* b, cudaStream_t st) {
  const auto kern = batch_kernel<P>(b);
  if (b->smem > 48 * 1024) IDBF_CUDA_TRY(allow_smem(kern, bat::kSmemCap));
  const void* const* xs = (const void* const*)b->d_ptrs;
  void* const* ys = (void* const*)(b->d_ptrs + b->nops);
  const int64_t* lds = (const int64_t*)(b->d_ptrs + 2 * b->nops);
  IDBF_CUDA_TRY(cudaMemsetAsync(b->d_counters, 0, sizeof(int) * (1 + b->nlevels_total), st));
  kern<<<b->ctas, persistent_threads(b), b->smem, st>>>(b->d_ops, b->d_lv, b->d_items, b->nitems, xs, ys, lds, b->d_counters,
                                                        b->d_counters + 1, b->d_target, b->d_status, b->limit_ns);
  IDBF_CUDA_TRY(cudaGetLastError());
  return IDBF_OK;
}

// shared memory per CTA: the largest node of any level of any operator
template <class P>
size_t smem_for(idbf_batch_s* b) {
  size_t sm = 0;
  for (int o = 0; o < b->nops; ++o) {
    if (b->sep[o]) continue;
    for (const LevelInfo& li : b->plans[o]->p.lv) sm = std::max(sm, bat::items_smem<P>(li, b->R[o], b->h_ops[o].width));
  }
  return sm;
}

template <class P>
int occupancy(idbf_batch_s* b) {
  int n = 0;
  const auto kern = batch_kernel<P>(b);
  if (b->smem > 48 * 1024) allow_smem(kern, bat::kSmemCap);
  cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, kern, persistent_threads(b), b->smem);
  return std::max(n, 1);
}

// calls FN<P>(args...) for the batch's arithmetic
#define IDBF_BATCH_DISPATCH(FN, ...)                            \
  (b->mode == IDBF_MODE_FP64   ? FN<FP64P>(__VA_ARGS__)         \
   : b->mode == IDBF_MODE_DF64 ? FN<DF64P>(__VA_ARGS__)         \
                               : FN<FP32P>(__VA_ARGS__))

idbf_status launch(idbf_batch_s* b, cudaStream_t st) {
  return level_launched(b) ? IDBF_BATCH_DISPATCH(launch_levels, b, st) : IDBF_BATCH_DISPATCH(launch_batch, b, st);
}

bool tile_valid(int mode, int tile) {
  if (tile < 0 || tile >= bat::kNumTiles) return false;
  const bat::Tile t = bat::kTiles[tile];
  switch (mode) {
    case IDBF_MODE_FP64: return t.rb <= bat::max_rb<FP64P>();
    case IDBF_MODE_DF64: return t.rb <= bat::max_rb<DF64P>() && !t.wide;
    default: return t.rb <= bat::max_rb<FP32P>();
  }
}

// The launches of one batch apply as a graph.
idbf_status capture(idbf_batch_s* b) {
  IDBF_CUDA_TRY(cudaStreamBeginCapture(b->cap, cudaStreamCaptureModeThreadLocal));
  idbf_status s = launch(b, b->cap);
  cudaGraph_t g = nullptr;
  const cudaError_t e = cudaStreamEndCapture(b->cap, &g);
  if (s != IDBF_OK) { if (g) cudaGraphDestroy(g); return s; }
  if (e != cudaSuccess) { set_cuda_error(e); return IDBF_ECUDA; }
  b->graph = g;
  IDBF_CUDA_TRY(cudaGraphInstantiate(&b->exec, g, 0));
  return IDBF_OK;
}

// Queue of items, completion targets and the captured graph for the current (rb, npi).
idbf_status layout(idbf_batch_s* b) {
  free_layout(b);
  if (!tile_valid(b->mode, b->tile)) return IDBF_EUNSUPPORTED;
  b->rb = bat::kTiles[b->tile].rb;
  b->sep.assign(b->nops, 0);
  for (int o = 0; o < b->nops; ++o) b->sep[o] = b->plans[o]->p.N >= b->split_n ? 1 : 0;
  for (int o = 0; o < b->nops; ++o) b->h_ops[o].width = node::even_block(b->R[o], b->rb);
  IDBF_CUDA_TRY(cudaMemcpy(b->d_ops, b->h_ops.data(), sizeof(bat::OpDesc) * b->nops, cudaMemcpyHostToDevice));
  if (level_launched(b)) {
    std::vector<bat::LevelItem> li;
    const idbf_status s = IDBF_BATCH_DISPATCH(plan_levels, b, li);
    if (s != IDBF_OK) return s;
    b->nitems = (int)li.size();
    b->smem = 0;
    b->ctas = b->nitems;
    if (b->nitems == 0) return IDBF_OK;
    IDBF_CUDA_TRY(cudaMalloc((void**)&b->d_litems, sizeof(bat::LevelItem) * li.size()));
    IDBF_CUDA_TRY(cudaMemcpy(b->d_litems, li.data(), sizeof(bat::LevelItem) * li.size(), cudaMemcpyHostToDevice));
    return capture(b);
  }
  std::vector<bat::Item> items;
  std::vector<int> target(b->nlevels_total, 0);
  int maxL = 0, base = 0;
  std::vector<int> lbase(b->nops);
  for (int o = 0; o < b->nops; ++o) {
    lbase[o] = base;
    base += b->plans[o]->p.L + 1;
    maxL = std::max(maxL, b->plans[o]->p.L);
  }
  for (int l = 0; l <= maxL; ++l)
    for (int o = 0; o < b->nops; ++o) {
      const Plan& p = b->plans[o]->p;
      if (l > p.L || b->sep[o]) continue;
      // the right-hand-side blocks of a run of nodes are neighbours in the queue, so the
      // blocks' second and later reads of the factors come from L2
      const int rbl = b->h_ops[o].width;
      for (int n0 = 0; n0 < p.m; n0 += b->npi)
        for (int r0 = 0; r0 < b->R[o]; r0 += rbl) {
          bat::Item it;
          it.op = o;
          it.level = l;
          it.node0 = n0;
          it.nodes = std::min(b->npi, p.m - n0);
          it.r0 = r0;
          it.pad = 0;
          items.push_back(it);
          ++target[lbase[o] + l];
        }
    }
  b->nitems = (int)items.size();
  if (b->debug_extra > 0 && b->nlevels_total > 0) target[0] += b->debug_extra;
  if (b->nitems == 0) {  // every operator runs through idbf_apply: no persistent launch
    b->smem = 0;
    b->ctas = 0;
    return IDBF_OK;
  }
  b->smem = IDBF_BATCH_DISPATCH(smem_for, b);
  if (b->smem == 0 || b->smem > bat::kSmemCap) return IDBF_EUNSUPPORTED;
  const int occ = IDBF_BATCH_DISPATCH(occupancy, b);
  int sms = 152;
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, b->device);
  b->ctas = std::max(1, std::min(occ * sms, b->nitems));
  IDBF_CUDA_TRY(cudaMalloc((void**)&b->d_items, sizeof(bat::Item) * std::max(1, b->nitems)));
  IDBF_CUDA_TRY(cudaMalloc((void**)&b->d_target, sizeof(int) * b->nlevels_total));
  IDBF_CUDA_TRY(cudaMalloc((void**)&b->d_counters, sizeof(int) * (1 + b->nlevels_total)));
  IDBF_CUDA_TRY(cudaMemcpy(b->d_items, items.data(), sizeof(bat::Item) * b->nitems, cudaMemcpyHostToDevice));
  IDBF_CUDA_TRY(cudaMemcpy(b->d_target, target.data(), sizeof(int) * b->nlevels_total, cudaMemcpyHostToDevice));
  return capture(b);
}

}  // namespace

extern "C" {

idbf_status idbf_batch_create(const idbf_plan* plans, int32_t nops, const int64_t* nrhs, int32_t mode, idbf_batch* out) {
  if (!out) return IDBF_EINVAL;
  *out = nullptr;
  if (!plans || !nrhs || nops < 1 || nops > (1 << 16)) return IDBF_EINVAL;
  if (mode != IDBF_MODE_FP64 && mode != IDBF_MODE_DF64 && mode != IDBF_MODE_FP32) return IDBF_EINVAL;
  const int fmt = mode == IDBF_MODE_FP64 ? IDBF_STORE_C128 : mode == IDBF_MODE_DF64 ? IDBF_STORE_DF64 : IDBF_STORE_C64;
  int dev = 0;
  cudaGetDevice(&dev);
  for (int o = 0; o < nops; ++o) {
    if (!plans[o] || nrhs[o] < 1 || nrhs[o] > (1 << 16) || plans[o]->p.device != dev) return IDBF_EINVAL;
    if (!plans[o]->p.has_format(fmt) || plans[o]->p.uneven) return IDBF_EUNSUPPORTED;
  }
  idbf_batch_s* b = new (std::nothrow) idbf_batch_s();
  if (!b) return IDBF_ENOMEM;
  b->device = dev;
  b->nops = nops;
  b->mode = mode;
  b->fmt = fmt;
  b->plans.assign(plans, plans + nops);
  b->R.assign(nrhs, nrhs + nops);
  std::vector<bat::OpDesc> ods(nops);
  std::vector<bat::OpLevel> lvs;
  idbf_status s = IDBF_OK;
  for (int o = 0; o < nops && s == IDBF_OK; ++o) {
    const Plan& p = plans[o]->p;
    const size_t half = (size_t)p.max_seg_total * nrhs[o] * 16;
    void* w = nullptr;
    cudaError_t e = cudaMalloc(&w, 2 * half);
    if (e != cudaSuccess) { set_cuda_error(e); s = IDBF_ENOMEM; break; }
    b->ws.push_back(w);
    ods[o].L = p.L;
    ods[o].R = (int)nrhs[o];
    ods[o].level_base = (int)lvs.size();
    ods[o].width = 1;
    ods[o].ws0 = w;
    ods[o].ws1 = (char*)w + half;
    for (int l = 0; l <= p.L; ++l) {
      const LevelInfo& li = p.lv[l];
      bat::OpLevel ol;
      ol.d = p.level(l);
      ol.mat = p.lmat[fmt][l];
      ol.max_in = li.max_in;
      ol.max_out = li.max_out;
      ol.max_rows = li.max_rows;
      ol.max_cols = li.max_cols;
      ol.max_rows_pair = li.max_rows_pair;
      ol.pad = 0;
      lvs.push_back(ol);
    }
  }
  b->nlevels_total = (int)lvs.size();
  if (s == IDBF_OK) {
    cudaError_t e = cudaMalloc((void**)&b->d_ops, sizeof(bat::OpDesc) * nops);
    if (e == cudaSuccess) e = cudaMalloc((void**)&b->d_lv, sizeof(bat::OpLevel) * lvs.size());
    if (e == cudaSuccess) e = cudaMalloc((void**)&b->d_ptrs, sizeof(void*) * 3 * nops);
    if (e == cudaSuccess) e = cudaMalloc((void**)&b->d_status, sizeof(int));
    if (e == cudaSuccess) e = cudaMemcpy(b->d_lv, lvs.data(), sizeof(bat::OpLevel) * lvs.size(), cudaMemcpyHostToDevice);
    b->h_ops = ods;
    if (e == cudaSuccess) e = cudaMemset(b->d_status, 0, sizeof(int));
    if (e == cudaSuccess) e = cudaStreamCreateWithFlags(&b->cap, cudaStreamNonBlocking);
    if (e == cudaSuccess) e = cudaEventCreateWithFlags(&b->ev_fork, cudaEventDisableTiming);
    if (e != cudaSuccess) { set_cuda_error(e); s = e == cudaErrorMemoryAllocation ? IDBF_ENOMEM : IDBF_ECUDA; }
  }
  if (s == IDBF_OK) {
    // default tile: the largest preferred one whose shared memory fits
    static const int pref_df[] = {3, 2, 1, 0}, pref_other[] = {5, 4, 3, 1, 0};
    const int* pref = mode == IDBF_MODE_DF64 ? pref_df : pref_other;
    const int npref = mode == IDBF_MODE_DF64 ? 4 : 5;
    for (int k = 0; k < npref; ++k) {
      b->tile = pref[k];
      s = layout(b);
      if (s != IDBF_EUNSUPPORTED) break;
    }
  }
  if (s != IDBF_OK) {
    idbf_batch_destroy(b);
    return s;
  }
  *out = b;
  return IDBF_OK;
}

idbf_status idbf_batch_apply(idbf_batch b, const void* const* x, void* const* y, const int64_t* ld, void* stream) {
  if (!b || !x || !y || !ld) return IDBF_EINVAL;
  int cur = -1;
  cudaGetDevice(&cur);
  if (cur != b->device) return IDBF_EINVAL;
  std::vector<void*> tab(3 * b->nops);
  for (int o = 0; o < b->nops; ++o) {
    if (!x[o] || !y[o] || ld[o] < b->plans[o]->p.N) return IDBF_EINVAL;
    tab[o] = (void*)x[o];
    tab[b->nops + o] = y[o];
    memcpy(&tab[2 * b->nops + o], &ld[o], sizeof(int64_t));
  }
  cudaStream_t st = (cudaStream_t)stream;
  // after a layout that failed there is no graph; without one, every operator must be above the split
  if (!b->exec && std::find(b->sep.begin(), b->sep.end(), (char)0) != b->sep.end()) return IDBF_ECUDA;
  if (b->exec) {
    // pageable source: the copy is staged before the call returns, so tab may go out of scope
    IDBF_CUDA_TRY(cudaMemcpyAsync(b->d_ptrs, tab.data(), sizeof(void*) * tab.size(), cudaMemcpyHostToDevice, st));
    IDBF_CUDA_TRY(cudaGraphLaunch(b->exec, st));
  }
  // the operators above the split: their own per-level kernels, after the persistent launch
  for (int o = 0; o < b->nops; ++o) {
    if (!b->sep[o]) continue;
    const idbf_status s = idbf_apply(b->plans[o], x[o], y[o], b->R[o], ld[o], b->mode, stream);
    if (s != IDBF_OK) return s;
  }
  return IDBF_OK;
}

idbf_status idbf_batch_autotune(idbf_batch b, const void* const* x, void* const* y, const int64_t* ld, int32_t reps,
                                void* stream, float* best_ms) {
  if (!b || reps < 1) return IDBF_EINVAL;
  cudaStream_t st = (cudaStream_t)stream;
  cudaEvent_t e0, e1;
  cudaEventCreate(&e0);
  cudaEventCreate(&e1);
  float best = 1e30f;
  int btile = b->tile, bnpi = b->npi;
  int64_t bsplit = b->split_n;
  idbf_status s = IDBF_OK;
  // time the current layout (a warm-up launch, then reps launches); EUNSUPPORTED layouts are skipped
  auto trial = [&]() {
    idbf_status r = layout(b);
    if (r == IDBF_EUNSUPPORTED) return;
    if (r != IDBF_OK) { s = r; return; }
    if ((s = idbf_batch_apply(b, x, y, ld, stream)) != IDBF_OK) return;
    cudaEventRecord(e0, st);
    for (int k = 0; k < reps && s == IDBF_OK; ++k) s = idbf_batch_apply(b, x, y, ld, stream);
    cudaEventRecord(e1, st);
    cudaEventSynchronize(e1);
    float ms = 0.f;
    cudaEventElapsedTime(&ms, e0, e1);
    ms /= reps;
    if (s == IDBF_OK && ms < best) {
      best = ms;
      btile = b->tile;
      bnpi = b->npi;
      bsplit = b->split_n;
    }
  };
  // every tiling at the current split
  auto tilings = [&]() {
    const int npis[3] = {1, 2, 4};
    for (int a = 0; a < bat::kNumTiles && s == IDBF_OK; ++a)
      for (int c = 0; c < 3 && s == IDBF_OK; ++c) {
        if (!tile_valid(b->mode, a)) continue;
        b->tile = a;
        b->npi = npis[c];
        trial();
      }
  };
  if (b->split_auto) {
    b->split_n = INT64_MAX;
    bsplit = INT64_MAX;
  }
  tilings();
  // then, with the best tiling, every split: all operators in the persistent launch, or those of
  // N >= n for each N of the batch through their own per-level kernels; the tilings again if the
  // best split changed
  const int64_t split0 = bsplit;
  if (s == IDBF_OK && b->split_auto) {
    std::vector<int64_t> cand = {INT64_MAX};
    for (const idbf_plan pl : b->plans) cand.push_back(pl->p.N);
    std::sort(cand.begin(), cand.end());
    cand.erase(std::unique(cand.begin(), cand.end()), cand.end());
    for (const int64_t c : cand) {
      if (s != IDBF_OK) break;
      b->tile = btile;
      b->npi = bnpi;
      b->split_n = c;
      trial();
    }
  }
  if (s == IDBF_OK && bsplit != split0) {
    b->split_n = bsplit;
    tilings();
  }
  cudaEventDestroy(e0);
  cudaEventDestroy(e1);
  b->tile = btile;
  b->npi = bnpi;
  b->split_n = bsplit;
  if (s == IDBF_OK) s = layout(b);
  if (best_ms) *best_ms = best;
  return s;
}

idbf_status idbf_batch_set_split(idbf_batch b, int64_t min_separate_n) {
  if (!b || min_separate_n < 0) return IDBF_EINVAL;
  if (min_separate_n == 0) {  // the autotuner chooses; until then every operator stays in the launch
    b->split_auto = true;
    if (b->split_n == INT64_MAX) return IDBF_OK;
    b->split_n = INT64_MAX;
    return layout(b);
  }
  const int64_t old = b->split_n;
  b->split_n = min_separate_n;
  idbf_status s = layout(b);
  if (s == IDBF_EUNSUPPORTED) {
    b->split_n = old;
    const idbf_status r = layout(b);
    return r == IDBF_OK ? s : r;
  }
  b->split_auto = false;
  return s;
}

idbf_status idbf_batch_split(idbf_batch b, int64_t* min_separate_n, int32_t* separate_ops) {
  if (!b) return IDBF_EINVAL;
  if (min_separate_n) *min_separate_n = b->split_n;
  if (separate_ops) {
    int32_t n = 0;
    for (const char c : b->sep) n += c ? 1 : 0;
    *separate_ops = n;
  }
  return IDBF_OK;
}

idbf_status idbf_batch_set_tiling(idbf_batch b, int32_t tile, int32_t nodes_per_item) {
  if (!b || tile < 0 || tile >= bat::kNumTiles) return IDBF_EINVAL;
  if (nodes_per_item != 1 && nodes_per_item != 2 && nodes_per_item != 4) return IDBF_EINVAL;
  if (!tile_valid(b->mode, tile)) return IDBF_EUNSUPPORTED;
  const int old_tile = b->tile, old_npi = b->npi;
  b->tile = tile;
  b->npi = nodes_per_item;
  idbf_status s = layout(b);
  if (s == IDBF_EUNSUPPORTED) {
    b->tile = old_tile;
    b->npi = old_npi;
    const idbf_status r = layout(b);
    return r == IDBF_OK ? s : r;
  }
  return s;
}

idbf_status idbf_batch_debug_set_wait(idbf_batch b, uint64_t limit_ns, int32_t extra_target) {
  if (!b || limit_ns == 0 || extra_target < 0) return IDBF_EINVAL;
  const uint64_t old_limit = b->limit_ns;
  const int old_extra = b->debug_extra;
  b->limit_ns = limit_ns;
  b->debug_extra = extra_target;
  const idbf_status s = layout(b);  // the limit and the targets are captured in the graph
  if (s == IDBF_EUNSUPPORTED) {     // the persistent launch does not fit where level launches do
    b->limit_ns = old_limit;
    b->debug_extra = old_extra;
    const idbf_status r = layout(b);
    return r == IDBF_OK ? s : r;
  }
  return s;
}

idbf_status idbf_batch_info(idbf_batch b, int32_t* rhs_per_item, int32_t* nodes_per_item, int32_t* items, int32_t* ctas) {
  if (!b) return IDBF_EINVAL;
  if (rhs_per_item) *rhs_per_item = b->rb;
  if (nodes_per_item) *nodes_per_item = b->npi;
  if (items) *items = b->nitems;
  if (ctas) *ctas = b->ctas;
  return IDBF_OK;
}

idbf_status idbf_batch_sync_status(idbf_batch b, void* stream) {
  if (!b) return IDBF_EINVAL;
  int v = 0;
  cudaStream_t st = (cudaStream_t)stream;
  IDBF_CUDA_TRY(cudaMemcpyAsync(&v, b->d_status, sizeof(int), cudaMemcpyDeviceToHost, st));
  IDBF_CUDA_TRY(cudaStreamSynchronize(st));
  idbf_status res = IDBF_OK;
  if (v) {
    IDBF_CUDA_TRY(cudaMemset(b->d_status, 0, sizeof(int)));
    res = IDBF_ETIMEOUT;
  }
  // the operators applied through idbf_apply report their own bounded waits
  for (int o = 0; o < b->nops; ++o) {
    if (!b->sep[o]) continue;
    const idbf_status r = idbf_sync_status(b->plans[o], stream);
    if (r != IDBF_OK && res == IDBF_OK) res = r;
  }
  return res;
}

void idbf_batch_destroy(idbf_batch b) {
  if (!b) return;
  int cur = 0;
  cudaGetDevice(&cur);
  if (cur != b->device) cudaSetDevice(b->device);
  cudaDeviceSynchronize();
  free_layout(b);
  for (void* w : b->ws) cudaFree(w);
  if (b->d_ops) cudaFree(b->d_ops);
  if (b->d_lv) cudaFree(b->d_lv);
  if (b->d_ptrs) cudaFree(b->d_ptrs);
  if (b->d_status) cudaFree(b->d_status);
  if (b->cap) cudaStreamDestroy(b->cap);
  for (cudaStream_t q : b->side) cudaStreamDestroy(q);
  for (cudaEvent_t q : b->ev_join) cudaEventDestroy(q);
  if (b->ev_fork) cudaEventDestroy(b->ev_fork);
  if (cur != b->device) cudaSetDevice(cur);
  delete b;
}

}  // extern "C"

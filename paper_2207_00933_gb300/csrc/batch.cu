// Batched recursion level: many queries (bins of possibly different
// circuits, uneven active-qubit counts) reconstructed together: the merges of
// all of them in one launch, then their contraction steps in one persistent
// launch.  (A single query's one launch keeps its merges in the work list.)
//
// The host flattens every query's contraction bands and tiles into one work
// list ordered by dependency level.  Persistent CTAs claim items in list order
// from a global head counter, ahead of the item they work on while many are
// left.  Every tensor has a completion counter; an item waits (bounded) until
// the counters of its input tensors reach their expected item counts, does its
// work, then bumps the counter of the tensor it wrote.  An item only ever waits
// for items earlier in the list, and every CTA works through its claims in
// order, so the earliest unfinished item always runs and the schedule cannot
// deadlock.  The last CTA to leave re-arms the head and the counters, so the
// same launch can be replayed (e.g. from a CUDA graph).  On a wait timeout the
// kernel raises an abort flag that makes every CTA drain quickly and records an
// error code.
//
// Bound: the latency of its items (operands, map entries and counters from
// L2), so three CTAs per SM although the 64 x 64 tiles then spill.  256 queries
// of 10 to 20 active qubits over four circuits (165 MB of bins, 863 MB of
// states merged from L2): 162 us, 66 of them the merges (180 with two CTAs per
// SM, 158 with four, where longer shared indices lose: 64 queries of K = 64
// steps 210, 197 and 200 us, 179 since a list's last items are claimed late and
// a 64-deep stage's stores spread over the banks);
// one launch with a merge block or a 32 x 32 tile per item took 833 us.
#include "device_ops.cuh"

namespace sqc {

namespace {

__device__ __forceinline__ uint64_t global_ns() {
  uint64_t t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}

__device__ __forceinline__ unsigned ld_acquire(const unsigned* p) {
  unsigned v;
  asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return v;
}

// Per-query FP64 probability sum over the final step's tiles: each tile
// stores its partial (the warps' sums in red, added in warp order), the last
// one adds them into *total in a fixed order.  Run by one warp while the rest
// of the CTA goes on to the next item.
__device__ __forceinline__ void finish_query_total(const double* red, const BatchStep& st, int64_t tile,
                                                   double* total) {
  const int lane = threadIdx.x & 31;
  int last = 0;
  if (lane == 0) {
    double s = 0.0;
    for (int w = 0; w < kOpThreads / 32; ++w) s += red[w];
    st.partials[tile] = s;
    __threadfence();
    last = atomicAdd(st.counter, 1u) == unsigned(st.ntiles - 1);
  }
  if (!__shfl_sync(0xffffffffu, last, 0)) return;
  __threadfence();
  double s = 0.0;
  for (int64_t i = lane; i < st.ntiles; i += 32) s += static_cast<volatile double*>(st.partials)[i];
  for (int off = 16; off > 0; off >>= 1) s += __shfl_down_sync(0xffffffffu, s, off);
  if (lane == 0) {
    *total = s;
    *st.counter = 0u;
  }
}

template <int BM, int BN, int TM, int TN, bool CH, int BK>
__device__ __forceinline__ double run_tile(const BatchStep& st, int64_t tile, float* smem, void* C) {
  const int64_t tiles_n = (st.a.N + BN - 1) / BN;
  const int tn_shift = __ffsll(tiles_n) - 1;
  const int64_t m0 = (tile >> tn_shift) * BM;
  const int64_t n0 = (tile & (tiles_n - 1)) * BN;
  // operands written by other CTAs of this launch: read from L2, not
  // through the read-only path
  return gemm_tile<BM, BN, TM, TN, CH, BK, kOpThreads, true>(st.a, m0, n0, smem, smem + BK * (BM + 4), C);
}

// Items per CTA at the end of a list that are not claimed ahead (1, 2, 4: 256
// queries 169, 163, 164 us; 64 with the pyramid 195, 190, 190).
constexpr int64_t kLead = 2;

__global__ void __launch_bounds__(kOpThreads, kBatchCtasPerSm) batch_kernel(BatchLaunch L) {
  pdl_wait();      // the previous kernel on the stream has completed
  pdl_trigger();   // the next one may start launching
  extern __shared__ __align__(16) float smem[];
  __shared__ MergeDesc md;
  __shared__ __align__(16) BatchItem items[2];
  __shared__ double red[kOpThreads / 32];
  __shared__ bool is_last;
  __shared__ int skip;                        // -1: no more items
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  // While the list is long, items are claimed ahead, so that an item's number
  // and contents are on their way while the one before it is worked on.  Its
  // last kLead items per CTA (all of a short list) are claimed when the CTA is
  // free: claimed ahead they would wait behind the item at hand while other
  // CTAs are idle.  Every CTA works through its claims in list order, so the
  // earliest unfinished item is never held up by a later one and the schedule
  // still cannot deadlock.
  auto claim = [&]() -> int64_t {
    return int64_t(atomicAdd(reinterpret_cast<unsigned long long*>(L.head), 1ull));
  };
  constexpr int64_t kNone = -1;
  const int64_t ahead_to = L.n_items - kLead * int64_t(gridDim.x);   // items before it are claimed ahead
  int64_t id = 0, next = kNone;               // thread 0: this item's number and the next one's
  if (threadIdx.x == 0) {
    id = claim();
    if (id < ahead_to) next = claim();
    if (id < L.n_items) items[0] = L.items[id];
  }
  for (int p = 0;; p ^= 1) {
    const BatchItem& item = items[p];
    if (threadIdx.x == 0) {
      skip = -1;
      if (id < L.n_items) {
        // wait for the input tensors (bounded; abort on timeout)
        unsigned want[2], have[2];
#pragma unroll
        for (int k = 0; k < 2; ++k) {
          const int dep = k ? item.dep1 : item.dep0;
          want[k] = dep < 0 ? 0u : __ldg(L.expected + dep);
          have[k] = dep < 0 ? 0u : ld_acquire(L.counts + dep);
        }
        for (int k = 0; k < 2; ++k) {
          const int dep = k ? item.dep1 : item.dep0;
          uint32_t i = 0;
          uint64_t t0 = 0;
          while (have[k] < want[k]) {
            if (*static_cast<volatile int*>(L.abort)) break;     // another CTA gave up: drain
            if ((++i & 31) == 0) {
              const uint64_t now = global_ns();
              if (t0 == 0) {
                t0 = now;
              } else if (now - t0 > L.wait_ns) {
                atomicExch(L.abort, 1);
                atomicExch(L.err, 1);
                break;
              }
            }
            if (i > 32) __nanosleep(64);
            have[k] = ld_acquire(L.counts + dep);
          }
        }
        skip = *static_cast<volatile int*>(L.abort) ? 1 : 0;    // one decision for the whole CTA
      }
    }
    __syncthreads();
    const int sk = skip;
    if (sk < 0) break;
    int64_t after = kNone;
    if (threadIdx.x == 0 && next != kNone) {
      if (next < L.n_items) {
        const char* src = reinterpret_cast<const char*>(L.items + next);
        const uint32_t dst = uint32_t(__cvta_generic_to_shared(&items[p ^ 1]));
        asm volatile("cp.async.ca.shared.global [%0], [%1], 16;" ::"r"(dst), "l"(src) : "memory");
        asm volatile("cp.async.ca.shared.global [%0], [%1], 16;" ::"r"(dst + 16), "l"(src + 16) : "memory");
      }
      if (next < ahead_to) after = claim();
    }
    const BatchStep* sums = nullptr;          // a last step with a probability sum
    if (!sk) {
      if (item.type == kItemMerge) {
        static_assert(sizeof(MergeDesc) % 8 == 0 && sizeof(MergeDesc) / 8 <= kOpThreads, "a thread per word");
        if (threadIdx.x < sizeof(MergeDesc) / 8)
          reinterpret_cast<uint64_t*>(&md)[threadIdx.x] = reinterpret_cast<const uint64_t*>(L.mdescs + item.idx)[threadIdx.x];
        __syncthreads();
        for (int b = 0; b < item.count; ++b) {
          if (md.tiled) merge_tile(md, item.tile + b, smem);
          else merge_block(md, item.tile + b);
          if (md.tiled) __syncthreads();
        }
      } else {
        const BatchStep& st = L.steps[item.idx];
        // a single-query launch names its output and probability sum per
        // run; a batch baked them into its steps
        void* C = st.from_launch ? L.out : st.a.C;
        double* total = st.from_launch ? L.total : st.total;
        double mine;
        if (st.band > 0) {
          const int64_t cols = st.a.N / band_cols(st.a);
          const int c_shift = __ffsll(cols) - 1;
          const int64_t m0 = (item.tile >> c_shift) * st.band, n0 = (item.tile & (cols - 1)) * band_cols(st.a);
          // the FP32 groups of the probability check are the tile's
          if (st.cfg == 2) mine = gemm_band<8, true>(st.a, m0, n0, st.band, smem, C);
          else if (st.cfg == 1 || st.cfg == 4) mine = gemm_band<4, true>(st.a, m0, n0, st.band, smem, C);
          else mine = gemm_band<2, true>(st.a, m0, n0, st.band, smem, C);
        } else switch (st.cfg) {
          case 0: mine = run_tile<32, 32, 2, 2, false, 16>(st, item.tile, smem, C); break;
          case 1: mine = run_tile<64, 64, 4, 4, false, 16>(st, item.tile, smem, C); break;
          case 2: mine = run_tile<128, 64, 8, 4, false, 16>(st, item.tile, smem, C); break;
          case 3: mine = run_tile<32, 32, 2, 2, false, 64>(st, item.tile, smem, C); break;
          case 4: mine = run_tile<64, 64, 4, 4, false, 64>(st, item.tile, smem, C); break;
          case 5: mine = run_tile<32, 32, 2, 2, true, 16>(st, item.tile, smem, C); break;
          default: mine = run_tile<64, 64, 4, 4, true, 16>(st, item.tile, smem, C); break;
        }
        if (st.a.partials && total) {
          for (int off = 16; off > 0; off >>= 1) mine += __shfl_down_sync(0xffffffffu, mine, off);
          if (lane == 0) red[warp] = mine;
          sums = &st;
        }
      }
    }
    __syncthreads();
    if (warp == 1) {
      if (sums) finish_query_total(red, *sums, item.tile, sums->from_launch ? L.total : sums->total);
      if (lane == 0 && item.out >= 0) {
        __threadfence();
        atomicAdd(L.counts + item.out, 1u);
      }
    }
    if (threadIdx.x == 0) {
      asm volatile("cp.async.wait_all;" ::: "memory");
      if (sk) {
        id = L.n_items;                       // after an abort: drain
      } else if (next != kNone) {
        id = next;
        next = after;
      } else {
        id = claim();
        if (id < L.n_items) items[p ^ 1] = L.items[id];
      }
    }
  }
  // the last CTA out re-arms the schedule for the next launch
  if (threadIdx.x == 0) {
    __threadfence();
    is_last = atomicAdd(L.done, 1u) == gridDim.x - 1;
  }
  __syncthreads();
  if (is_last) {
    __threadfence();
    for (int64_t i = threadIdx.x; i < L.n_slots; i += blockDim.x) L.counts[i] = 0u;
    if (threadIdx.x == 0) {
      *L.head = 0ull;
      *L.done = 0u;
      *L.abort = 0;
    }
  }
}

// The merges of a level, one work item (some blocks of one descriptor) per
// CTA.  On their own because they need 32 registers where the steps' kernel
// needs 80: eight CTAs per SM cover the descriptor and item loads and the short
// chains of each sum, where that one holds three.  The price: a level whose
// merges take longer than its steps has no steps to hide them (16 queries with
// runs of 2^12 states and more over 16 MB: 54 + 30 us, 64 us together in one
// list).  With the long merges in the list, 256 queries took 163-197 us for
// 162.  The states come from L2
// (the resident tensors of a level's circuits fit it), so L2 bandwidth is the
// bound.
template <bool TILED>
__global__ void __launch_bounds__(256) batch_merge_kernel(const BatchItem* __restrict__ items,
                                                          const MergeDesc* __restrict__ mdescs) {
  pdl_wait();      // the previous kernel on the stream has completed
  pdl_trigger();   // the next one may start launching
  __shared__ MergeDesc d;
  __shared__ __align__(16) float tile[TILED ? kMergeTileFloats : 4];
  const BatchItem it = items[blockIdx.x];
  static_assert(sizeof(BatchItem) == 32, "fetched as two 16-byte words");
  static_assert(sizeof(MergeDesc) % 8 == 0 && sizeof(MergeDesc) / 8 <= 256, "one word per thread");
  if (threadIdx.x < sizeof(MergeDesc) / 8)
    reinterpret_cast<uint64_t*>(&d)[threadIdx.x] = reinterpret_cast<const uint64_t*>(mdescs + it.idx)[threadIdx.x];
  __syncthreads();
  for (int b = 0; b < it.count; ++b) {
    if (TILED && d.tiled) {
      merge_tile(d, it.tile + b, tile);
      __syncthreads();
    } else {
      merge_block(d, it.tile + b);
    }
  }
}

}  // namespace

cudaError_t launch_batch_merges(const BatchItem* items, int64_t n, const MergeDesc* mdescs, bool tiled,
                                cudaStream_t s) {
  if (n <= 0) return cudaSuccess;
  return launch_k(tiled ? batch_merge_kernel<true> : batch_merge_kernel<false>, dim3(unsigned(n)), dim3(256), 0, s,
                  false, items, mdescs);
}

int batch_smem_bytes() {
  // largest tile stage among the configurations above (64x64 with BK = 64)
  // and a band's rows
  constexpr int f = gemm_tile_smem_floats<64, 64, 64>();
  return int(sizeof(float)) * (f > kBandSmemFloats ? f : kBandSmemFloats);
}

cudaError_t batch_configure() {
  return cudaFuncSetAttribute(batch_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, batch_smem_bytes());
}

cudaError_t launch_batch(const BatchLaunch& L, int grid, cudaStream_t s) {
  if (L.n_items <= 0) return cudaSuccess;
  return launch_k(batch_kernel, dim3(unsigned(grid)), dim3(kOpThreads), size_t(batch_smem_bytes()), s, false, L);
}

// Tile configuration ids of the batch kernel for one step, under a tile
// policy: 0 = by occupancy (the default), 1 = small tiles (32 x 32: the
// most work items, best balance for many uneven queries), 2 = large tiles
// (64 x 64 or 128 x 64 wherever a step has enough of them: fewer operand
// reloads).  Every configuration sums each bin in the same order, so the
// bins do not depend on the policy.
int batch_tile_cfg(int64_t M, int64_t N, int64_t K, bool chunked, int64_t chunk, int64_t* bm, int64_t* bn,
                   int policy) {
  auto tiles = [&](int64_t a, int64_t b) { return ((M + a - 1) / a) * ((N + b - 1) / b); };
  (void)chunk;
  const bool deep = K >= 64;
  if (policy == 1) {
    *bm = 32; *bn = 32;
    return chunked ? 5 : (deep ? 3 : 0);
  }
  if (policy == 2) {
    if (chunked) {
      if (tiles(64, 64) >= 4) { *bm = 64; *bn = 64; return 6; }
      *bm = 32; *bn = 32;
      return 5;
    }
    if (!deep && tiles(128, 64) >= 16) { *bm = 128; *bn = 64; return 2; }
    if (tiles(64, 64) >= 4) { *bm = 64; *bn = 64; return deep ? 4 : 1; }
    *bm = 32; *bn = 32;
    return deep ? 3 : 0;
  }
  if (chunked) {
    if (tiles(64, 64) >= 64) { *bm = 64; *bn = 64; return 6; }
    *bm = 32; *bn = 32;
    return 5;
  }
  if (tiles(128, 64) >= 152 && !deep) { *bm = 128; *bn = 64; return 2; }
  if (tiles(64, 64) >= 64) { *bm = 64; *bn = 64; return deep ? 4 : 1; }
  *bm = 32; *bn = 32;
  return deep ? 3 : 0;
}

}  // namespace sqc

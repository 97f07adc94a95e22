// States merging (Section 4, Algorithm 2): for every subcircuit,
//
//   T_i[e][b] = sum_{x : zoom bits of x fixed, active bits of x = b} A_i[e][x]
//
// One launch covers all subcircuits of a query (a descriptor per
// subcircuit, a contiguous CTA range per descriptor).  It is an HBM-bound
// streaming reduction: with the recursion's roles the merged data qubits are
// the low bits of the bit-reversed storage index, so each bin is a
// contiguous run read with 128-bit loads, `lanes` threads per bin and a
// shuffle tree.  Other role patterns take the generic bit-deposit path.
// The result goes straight into the layout the first contraction step reads
// (rowmap/colmap), in FP32, FP64 or as three BF16 planes.
#include "device_ops.cuh"

namespace sqc {

namespace {

// Persistent: CTAs walk the blocks of all descriptors in order; a CTA
// reads a descriptor (and where the next one starts) only when it crosses
// into it.  Warp 0 does: a lane per descriptor finds the one that holds the
// block, a lane per word copies it, a round trip each (one thread that walked
// the descriptors and copied the 160 bytes through its 32 registers took 1-1.4
// us more per launch: 286 MB 60.0 -> 57.8 us; blocks of 13 and 16 wires into 2^20
// bins, merge and step, 14.3 -> 13.0).
// TILED: some descriptor is (a kernel of its own: the tiles' registers would
// cost the others occupancy).
template <bool TILED>
__global__ void __launch_bounds__(256) merge_kernel(const MergeDesc* __restrict__ descs, int n,
                                                    int64_t total_blocks) {
  pdl_wait();      // the previous kernel on the stream has completed
  pdl_trigger();   // the next one may start launching
  static_assert(sizeof(MergeDesc) % 8 == 0 && sizeof(MergeDesc) / 8 <= 32 && kMaxMerge <= 64, "a lane per word");
  __shared__ MergeDesc d;
  __shared__ __align__(16) float tile[TILED ? kMergeTileFloats : 4];
  __shared__ int64_t next_begin;
  if (threadIdx.x == 0) next_begin = 0;
  __syncthreads();
  for (int64_t blk = blockIdx.x; blk < total_blocks; blk += gridDim.x) {
    if (threadIdx.x < 32 && blk >= next_begin) {
      // the last descriptor that begins at or before blk (block_begin ascends)
      const int lane = threadIdx.x;
      const int64_t b0 = lane < n ? descs[lane].block_begin : total_blocks;
      const int64_t b1 = lane + 32 < n ? descs[lane + 32].block_begin : total_blocks;
      const int i = __popc(__ballot_sync(0xffffffffu, b0 <= blk)) + __popc(__ballot_sync(0xffffffffu, b1 <= blk)) - 1;
      if (lane < int(sizeof(MergeDesc) / 8))
        reinterpret_cast<uint64_t*>(&d)[lane] = reinterpret_cast<const uint64_t*>(descs + i)[lane];
      if (lane == ((i + 1) & 31)) next_begin = i + 1 < 32 ? b0 : (i + 1 < 64 ? b1 : total_blocks);
    }
    __syncthreads();
    if (TILED && d.tiled) merge_tile(d, blk - d.block_begin, tile);
    else merge_block(d, blk - d.block_begin);
    __syncthreads();
  }
}

// The merge of a query with few outputs over long runs (thousands of states
// per bin, as the first recursions over a wide circuit have): one warp per
// output as merge_block has it, but the run's 16-byte words go through each
// lane's own slots of a ring in shared memory (cp.async, three rounds of four
// words ahead), and the CTAs are small, so that a thousand warps keep HBM
// busy.  The additions are merge_sum's, in its order.
//
// Bound: HBM.  59 subcircuits, 1200 outputs of 2^10-2^15 states (123 MB):
// 28.6 us, against 73 us with merge_block's four words in flight per lane on
// 154 CTAs.
constexpr int kLongWarps = 2;
constexpr int kLongRounds = 4;                    // rounds of four words in the ring
__global__ void __launch_bounds__(32 * kLongWarps) merge_long_kernel(const MergeDesc* __restrict__ descs, int n,
                                                                     int64_t total) {
  pdl_wait();      // the previous kernel on the stream has completed
  pdl_trigger();   // the next one may start launching
  __shared__ float4 ring[kLongWarps][kLongRounds][4][32];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  int64_t o = int64_t(blockIdx.x) * kLongWarps + warp;
  if (o >= total) return;
  int i = 0;
  for (; i + 1 < n; ++i) {                        // the descriptor that holds output o
    const int64_t cnt = descs[i].warps ? descs[i].rows << descs[i].a : 0;
    if (o < cnt) break;
    o -= cnt;
  }
  const MergeDesc& d = descs[i];
  const int64_t e = o >> d.a;
  const uint32_t b = uint32_t(o & ((int64_t(1) << d.a) - 1));
  const float4* src = reinterpret_cast<const float4*>(merge_row(d, e) + (d.zoom_val | (b << d.m))) + lane;
  const uint32_t rounds = (1u << d.m) / (4u * 128u);
  const uint64_t off = d.rowmap[e] + d.colmap[b];
  auto request = [&](uint32_t r) {
    if (r < rounds) {
#pragma unroll
      for (int q = 0; q < 4; ++q)
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(uint32_t(__cvta_generic_to_shared(
                         &ring[warp][r % kLongRounds][q][lane]))),
                     "l"(src + size_t(r) * 128 + q * 32)
                     : "memory");
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
  };
  for (uint32_t r = 0; r < kLongRounds - 1; ++r) request(r);
  float acc = 0.f;
  for (uint32_t r = 0; r < rounds; ++r) {
    request(r + kLongRounds - 1);
    asm volatile("cp.async.wait_group %0;" ::"n"(kLongRounds - 1) : "memory");
    const float4(&w)[4][32] = ring[warp][r % kLongRounds];
    const float4 q0 = w[0][lane], q1 = w[1][lane], q2 = w[2][lane], q3 = w[3][lane];
    acc += (((q0.x + q0.y) + (q0.z + q0.w)) + ((q1.x + q1.y) + (q1.z + q1.w))) +
           (((q2.x + q2.y) + (q2.z + q2.w)) + ((q3.x + q3.y) + (q3.z + q3.w)));
  }
#pragma unroll
  for (int o2 = 16; o2 > 0; o2 >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o2);
  if (lane == 0) store_out_f(d.dst, d.kind, d.plane_stride, off, acc * pow2_to_float(d.alpha));
}

// Up to ten levels of the merge pyramids of several subcircuits.  A level is
// pairwise sums of the level below, and rows are powers of two long, so a
// pyramid is the pairwise reduction of one flat array: a CTA takes 1024
// consecutive values, four per thread -- two levels in registers, five by
// shuffles, three over the warps -- and writes its share of every level.
//
// Bound: HBM (4 bytes read and about 4 written per value).  The pyramids of
// two circuits of 5 and 6 subcircuits (72 MB of outputs): 4 launches, against
// 22 of a kernel that halved in shared memory, two barriers per level.
__global__ void __launch_bounds__(256) pyramid_kernel(PyramidLaunch L) {
  pdl_wait();      // the previous kernel on the stream has completed
  pdl_trigger();   // the next one may start launching
  __shared__ float wsum[8];
  int di = 0;
#pragma unroll
  for (int i = 1; i < kAttrPerLaunch; ++i)
    if (i < L.n && L.d[i].block_begin <= int64_t(blockIdx.x)) di = i;
  const PyramidDesc& d = L.d[di];
  const int64_t blk = int64_t(blockIdx.x) - d.block_begin;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int64_t len = d.V << (d.n - d.s);           // values of the level read
  const int64_t i4 = blk * 256 + threadIdx.x;
  // level s + l of the pyramid
  auto level = [&](int l) -> float* {
    return d.pyr + d.V * ((int64_t(1) << d.n) - (int64_t(1) << (d.n - d.s - l + 1)));
  };
  float4 q = make_float4(0.f, 0.f, 0.f, 0.f);
  if (4 * i4 + 3 < len) q = __ldg(reinterpret_cast<const float4*>(d.src) + i4);
  else if (4 * i4 < len) { q.x = d.src[4 * i4]; q.y = d.src[4 * i4 + 1]; }   // len == 2
  const float x = q.x + q.y, y = q.z + q.w;
  if (4 * i4 + 3 < len) *reinterpret_cast<float2*>(level(1) + 2 * i4) = make_float2(x, y);
  else if (4 * i4 < len) level(1)[2 * i4] = x;
  float v = x + y;
  if (d.c >= 2 && i4 < (len >> 2)) level(2)[i4] = v;
#pragma unroll
  for (int l = 3; l <= 7; ++l) {
    v += __shfl_down_sync(0xffffffffu, v, 1 << (l - 3));
    const int64_t i = i4 >> (l - 2);
    if (d.c >= l && (lane & ((1 << (l - 2)) - 1)) == 0 && i < (len >> l)) level(l)[i] = v;
  }
  if (d.c < 8) return;
  if (lane == 0) wsum[warp] = v;
  __syncthreads();
  if (warp == 0) {
    v = lane < 8 ? wsum[lane] : 0.f;
#pragma unroll
    for (int l = 8; l <= 10; ++l) {
      v += __shfl_down_sync(0xffffffffu, v, 1 << (l - 8));
      const int64_t i = (blk * 8 + lane) >> (l - 7);
      if (d.c >= l && lane < 8 && (lane & ((1 << (l - 7)) - 1)) == 0 && i < (len >> l)) level(l)[i] = v;
    }
  }
}

}  // namespace

cudaError_t launch_pyramids(PyramidDesc* d, int n, int* launches, cudaStream_t s) {
  // pass by pass (ten levels each), every subcircuit that has levels left
  for (int lev = 0;; lev += kPyramidLevelsPerPass) {
    PyramidLaunch L{};
    int64_t blocks = 0;
    bool any = false;
    auto flush = [&]() -> cudaError_t {
      if (L.n == 0) return cudaSuccess;
      const cudaError_t e = launch_k(pyramid_kernel, dim3(unsigned(blocks)), dim3(256), 0, s, false, L);
      *launches += 1;
      L.n = 0;
      blocks = 0;
      return e;
    };
    for (int i = 0; i < n; ++i) {
      if (lev >= d[i].n) continue;
      any = true;
      PyramidDesc t = d[i];
      t.s = lev;
      t.c = t.n - lev < kPyramidLevelsPerPass ? t.n - lev : kPyramidLevelsPerPass;
      if (lev > 0) t.src = t.pyr + t.V * ((int64_t(1) << t.n) - (int64_t(1) << (t.n - lev + 1)));
      t.block_begin = blocks;
      const int64_t nb = ((t.V << (t.n - lev)) + 1023) / 1024;
      if (L.n > 0 && blocks + nb > 0x7fffffff) {
        const cudaError_t e = flush();
        if (e != cudaSuccess) return e;
        t.block_begin = 0;
      }
      L.d[L.n++] = t;
      blocks += nb;
      if (L.n == kAttrPerLaunch) {
        const cudaError_t e = flush();
        if (e != cudaSuccess) return e;
      }
    }
    const cudaError_t e = flush();
    if (e != cudaSuccess || !any) return e;
  }
}

cudaError_t launch_merge_long(const MergeDesc* d_descs, int n, int64_t total_outputs, cudaStream_t s) {
  if (n <= 0 || total_outputs <= 0) return cudaSuccess;
  const int64_t grid = (total_outputs + kLongWarps - 1) / kLongWarps;
  return launch_k(merge_long_kernel, dim3(unsigned(grid)), dim3(32 * kLongWarps), 0, s, false, d_descs, n,
                  total_outputs);
}

cudaError_t launch_merge_blocks(const MergeDesc* d_descs, int n, int64_t total_blocks, bool tiled, cudaStream_t s) {
  if (n <= 0 || total_blocks <= 0) return cudaSuccess;
  // 8 CTAs of 256 threads per SM
  const int64_t grid = total_blocks < 152 * 8 ? total_blocks : 152 * 8;
  return launch_k(tiled ? merge_kernel<true> : merge_kernel<false>, dim3(unsigned(grid)), dim3(256), 0, s, false, d_descs, n, total_blocks);
}

}  // namespace sqc

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
// into it.
// TILED: some descriptor is (a kernel of its own: the tiles' registers would
// cost the others occupancy).
template <bool TILED>
__global__ void __launch_bounds__(256) merge_kernel(const MergeDesc* __restrict__ descs, int n,
                                                    int64_t total_blocks) {
  pdl_wait();      // the previous kernel on the stream has completed
  pdl_trigger();   // the next one may start launching
  __shared__ MergeDesc d;
  __shared__ __align__(16) float tile[TILED ? kMergeTileFloats : 4];
  __shared__ int cur;
  __shared__ int64_t next_begin;
  if (threadIdx.x == 0) {
    cur = -1;
    next_begin = 0;
  }
  __syncthreads();
  for (int64_t blk = blockIdx.x; blk < total_blocks; blk += gridDim.x) {
    if (threadIdx.x == 0 && blk >= next_begin) {
      int i = cur < 0 ? 0 : cur;
      while (i + 1 < n && descs[i + 1].block_begin <= blk) ++i;
      d = descs[i];
      cur = i;
      next_begin = i + 1 < n ? descs[i + 1].block_begin : total_blocks;
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
    const int64_t cnt = descs[i].rows << descs[i].a;
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

// Levels s+1 .. s+c of the merge pyramid from level s: a CTA takes chunks
// of 2^c consecutive values of one row, halves them c times in shared
// memory (pairwise sums) and writes every level's share.
__global__ void __launch_bounds__(256) pyramid_kernel(const float* __restrict__ src, float* pyr, int64_t V, int n,
                                                      int s, int c) {
  pdl_wait();      // the previous kernel on the stream has completed
  pdl_trigger();   // the next one may start launching
  __shared__ float buf[1 << kPyramidLevelsPerPass];
  const int C = 1 << c;
  const int row_shift = n - s - c;                   // chunks per row = 2^row_shift
  const int64_t total = V << row_shift;
  for (int64_t b = blockIdx.x; b < total; b += gridDim.x) {
    const int64_t e = b >> row_shift;
    const int64_t ch = b & ((int64_t(1) << row_shift) - 1);
    const float* in = src + (e << (n - s)) + (ch << c);
    for (int i = threadIdx.x; i < C; i += blockDim.x) buf[i] = in[i];
    __syncthreads();
    for (int l = 1; l <= c; ++l) {
      const int half = C >> l;
      const int m = s + l;
      float* out = pyr + V * ((int64_t(1) << n) - (int64_t(1) << (n - m + 1))) + (e << (n - m)) + (ch << (c - l));
      float t[(1 << kPyramidLevelsPerPass) / 2 / 256];
#pragma unroll
      for (int k = 0; k < int(sizeof(t) / sizeof(float)); ++k) {
        const int i = int(threadIdx.x) + k * 256;
        t[k] = i < half ? buf[2 * i] + buf[2 * i + 1] : 0.f;
      }
      __syncthreads();
#pragma unroll
      for (int k = 0; k < int(sizeof(t) / sizeof(float)); ++k) {
        const int i = int(threadIdx.x) + k * 256;
        if (i < half) {
          buf[i] = t[k];
          out[i] = t[k];
        }
      }
      __syncthreads();
    }
  }
}

}  // namespace

cudaError_t launch_pyramid(const float* A, float* pyr, int64_t V, int n, cudaStream_t s) {
  for (int lev = 0; lev < n;) {
    const int c = n - lev < kPyramidLevelsPerPass ? n - lev : kPyramidLevelsPerPass;
    const float* src = lev == 0 ? A : pyr + V * ((int64_t(1) << n) - (int64_t(1) << (n - lev + 1)));
    const int64_t total = V << (n - lev - c);
    const int64_t grid = total < 152 * 8 ? total : 152 * 8;
    cudaError_t e = launch_k(pyramid_kernel, dim3(unsigned(grid)), dim3(256), 0, s, false, src, pyr, V, n, lev, c);
    if (e != cudaSuccess) return e;
    lev += c;
  }
  return cudaSuccess;
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

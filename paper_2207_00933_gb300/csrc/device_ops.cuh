// Device-side bodies shared by the per-step kernels and the persistent
// batched kernel: one merge CTA-block and one SIMT contraction tile.
#pragma once
#include <type_traits>

#include "common.cuh"

namespace sqc {

// One lane's share of the sum over output (row of A, bin b) of descriptor d:
// every lanes-th 16-byte word of the run (or every lanes-th value).
__device__ __forceinline__ float merge_sum(const MergeDesc& d, const float* row, uint32_t b, uint32_t lane,
                                           uint32_t lanes) {
  float acc = 0.f;
  const uint32_t run = 1u << d.m;
  if (d.fast) {
    const float* src = row + (d.zoom_val | (b << d.m));
    if (run >= 4u * lanes) {
      // four independent 16-byte loads in flight per lane and round
      const float4* s4 = reinterpret_cast<const float4*>(src);
      const uint32_t nv = run / 4;
      uint32_t r = lane;
#pragma unroll 2
      for (; r + 3u * lanes < nv; r += 4u * lanes) {
        const float4 q0 = __ldg(s4 + r), q1 = __ldg(s4 + r + lanes);
        const float4 q2 = __ldg(s4 + r + 2u * lanes), q3 = __ldg(s4 + r + 3u * lanes);
        acc += (((q0.x + q0.y) + (q0.z + q0.w)) + ((q1.x + q1.y) + (q1.z + q1.w))) +
               (((q2.x + q2.y) + (q2.z + q2.w)) + ((q3.x + q3.y) + (q3.z + q3.w)));
      }
      for (; r < nv; r += lanes) {
        const float4 q = __ldg(s4 + r);
        acc += (q.x + q.y) + (q.z + q.w);
      }
    } else {
      for (uint32_t r = lane; r < run; r += lanes) acc += __ldg(src + r);
    }
  } else {
    // the merged bits of r spread over mer_mask: the next r of the lane by one
    // addition whose carries run over the other bits (a deposit per state, a
    // step per merged bit, was most of the loop: 16 outputs of 2^16 states in a
    // one-launch query 1151 -> 357 us)
    const float* src = row + (deposit(b, d.act_mask) | d.zoom_val);
    const uint32_t gaps = ~d.mer_mask, step = deposit(lanes, d.mer_mask);
    uint32_t x = deposit(lane, d.mer_mask);
#pragma unroll 4
    for (uint32_t r = lane; r < run; r += lanes) {
      acc += __ldg(src + x);
      x = ((x | gaps) + step) & ~gaps;
    }
  }
  return acc;
}

// Row of A that descriptor row e reads.
__device__ __forceinline__ const float* merge_row(const MergeDesc& d, int64_t e) {
  const int64_t er = d.rowsel ? int64_t(d.rowsel[e]) + d.row_add : e;
  return d.A + (er << d.n);
}

// The sums of a turned tile (merge_tile) over runs of 2^MB states: 2^MB / 4
// lanes per output, one 16-byte word each, so that a warp reads whole lines,
// and U rows' loads in flight per thread.  The additions are merge_sum's (one
// lane), in its order.
template <int MB, int U>
__device__ __forceinline__ void merge_tile_rows(const MergeDesc& d, const float* const* rows, uint32_t bin0, int nr,
                                                float alpha, float* tile) {
  constexpr int SB = kMergeTileBins + 1, L = MB > 2 ? 1 << (MB - 2) : 1, RP = 4 / L;
  const int sub = threadIdx.x & (L - 1), bin = (threadIdx.x / L) & 63, rg = threadIdx.x / (64 * L);
  const uint32_t at = (d.zoom_val | ((bin0 + bin) << MB)) + 4 * sub;
  for (int r0 = rg; r0 < nr; r0 += RP * U) {
    float4 w[U];
#pragma unroll
    for (int u = 0; u < U; ++u) {
      w[u] = make_float4(0.f, 0.f, 0.f, 0.f);
      const int r = r0 + RP * u;
      if (r >= nr) continue;
      const float* src = rows[r] + at;
      if constexpr (MB == 0) {
        w[u].x = __ldg(src);
      } else if constexpr (MB == 1) {
        const float2 t = __ldg(reinterpret_cast<const float2*>(src));
        w[u].x = t.x; w[u].y = t.y;
      } else {
        w[u] = __ldg(reinterpret_cast<const float4*>(src));
      }
    }
#pragma unroll
    for (int u = 0; u < U; ++u) {
      float acc = 0.f;
      if constexpr (MB == 0) {
        acc += w[u].x;
      } else if constexpr (MB == 1) {
        acc += w[u].x;
        acc += w[u].y;
      } else {
        float t = (w[u].x + w[u].y) + (w[u].z + w[u].w);
        if constexpr (MB == 4) {                     // ((0) + (1)) + ((2) + (3))
          t += __shfl_xor_sync(0xffffffffu, t, 1);
          t += __shfl_xor_sync(0xffffffffu, t, 2);
          acc += t;
        } else if constexpr (MB == 3) {              // (0) + (1)
          const float o = __shfl_xor_sync(0xffffffffu, t, 1);
          acc += t;
          acc += o;
        } else {
          acc += t;
        }
      }
      const int r = r0 + RP * u;
      if (sub == 0 && r < nr) tile[r * SB + bin] = acc * alpha;
    }
  }
}

// One tile of up to 32 rows x 64 bins of a descriptor whose rows are
// consecutive in the destination while its bins lie a whole operand row
// apart (a contraction operand: the shared cut edges innermost).  Bins are
// read along A's rows, the sums turned in shared memory, and consecutive rows
// written as 16-byte words: written as they are read, every 4-byte (BF16: 2-
// byte) value would touch a sector of its own.  smem: kMergeTileFloats.
// Bound: HBM.  256 rows x 4096 bins of one value and of 16 (71 MB): into FP32
// operands 29 -> 21 us, into BF16 planes 62 -> 23 us; 64 rows x 4096 bins of
// two and of 16 values, FP32, 12.9 -> 10.3 us.
constexpr int kMergeTileFloats = kMergeTileRows * (kMergeTileBins + 1) + 2 * kMergeTileRows + 2 * kMergeTileBins;
__device__ __forceinline__ void merge_tile(const MergeDesc& d, int64_t blk, float* smem) {
  constexpr int SB = kMergeTileBins + 1;
  const float** rows = reinterpret_cast<const float**>(smem);              // [kMergeTileRows]
  uint64_t* cols = reinterpret_cast<uint64_t*>(smem + 2 * kMergeTileRows);  // [kMergeTileBins]
  float* tile = smem + 2 * kMergeTileRows + 2 * kMergeTileBins;
  const int lr = d.rows < kMergeTileRows ? __ffsll(d.rows) - 1 : 5;      // log2 of the tile's rows
  const int nr = 1 << lr;
  const int64_t bt = blk & ((int64_t(1) << (d.a - 6)) - 1), rt = blk >> (d.a - 6);
  const uint32_t bin0 = uint32_t(bt) * kMergeTileBins;
  __shared__ uint64_t base;
  const int tid = threadIdx.x;
  if (tid < nr) {
    const int nbits = __ffsll(d.rows) - 1;
    const int64_t r = (rt << lr) + tid;                                  // r-th row in destination order
    int64_t e = 0;
    for (int j = 0; j < nbits; ++j) e |= ((r >> j) & 1) << d.rowbit[j];
    rows[tid] = merge_row(d, e);
    if (tid == 0) base = d.rowmap[e];
  } else if (tid >= 64 && tid < 64 + kMergeTileBins) {
    cols[tid - 64] = d.colmap[bin0 + tid - 64];
  }
  __syncthreads();
  const float alpha = pow2_to_float(d.alpha);
  if (d.fast && d.m <= 4) {
    switch (d.m) {
      case 0: merge_tile_rows<0, 8>(d, rows, bin0, nr, alpha, tile); break;
      case 1: merge_tile_rows<1, 8>(d, rows, bin0, nr, alpha, tile); break;
      case 2: merge_tile_rows<2, 8>(d, rows, bin0, nr, alpha, tile); break;
      case 3: merge_tile_rows<3, 8>(d, rows, bin0, nr, alpha, tile); break;
      default: merge_tile_rows<4, 8>(d, rows, bin0, nr, alpha, tile); break;
    }
  } else {
    for (int r = tid >> 6; r < nr; r += 4) tile[r * SB + (tid & 63)] = merge_sum(d, rows[r], bin0 + (tid & 63), 0, 1) * alpha;
  }
  __syncthreads();
  if (d.kind == OUT_F32) {
    for (int i = tid; i < (nr * kMergeTileBins) >> 2; i += 256) {
      const int r = 4 * (i & ((nr >> 2) - 1)), c = i >> (lr - 2);
      const float* t = tile + r * SB + c;
      float* p = static_cast<float*>(d.dst) + base + cols[c] + r;
      *reinterpret_cast<float4*>(p) = make_float4(t[0], t[SB], t[2 * SB], t[3 * SB]);
    }
  } else {                                           // OUT_BF16X3
    for (int i = tid; i < (nr * kMergeTileBins) >> 3; i += 256) {
      const int r = 8 * (i & ((nr >> 3) - 1)), c = i >> (lr - 3);
      const float* t = tile + r * SB + c;
      uint32_t w[3][4];
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        __nv_bfloat16 h[2][3];
#pragma unroll
        for (int u = 0; u < 2; ++u) {                // as store_out_f splits a value
          const float f = t[(2 * q + u) * SB];
          h[u][0] = __float2bfloat16_rn(f);
          const float r1 = f - __bfloat162float(h[u][0]);
          h[u][1] = __float2bfloat16_rn(r1);
          h[u][2] = __float2bfloat16_rn(r1 - __bfloat162float(h[u][1]));
        }
#pragma unroll
        for (int p = 0; p < 3; ++p)
          w[p][q] = uint32_t(__bfloat16_as_ushort(h[0][p])) | uint32_t(__bfloat16_as_ushort(h[1][p])) << 16;
      }
      __nv_bfloat16* o = static_cast<__nv_bfloat16*>(d.dst) + base + cols[c] + r;
#pragma unroll
      for (int p = 0; p < 3; ++p)
        *reinterpret_cast<uint4*>(o + p * d.plane_stride) = make_uint4(w[p][0], w[p][1], w[p][2], w[p][3]);
    }
  }
}

// One CTA-block of the merge of descriptor d (Section 4, Algorithm 2):
// blk is the block index relative to the descriptor's first block.
__device__ __forceinline__ void merge_block(const MergeDesc& d, int64_t blk) {
  const int lanes = d.lanes;                       // power of two
  const int lshift = __ffs(lanes) - 1;
  const int64_t o = (blk << (8 - lshift)) + (threadIdx.x >> lshift);
  const int lane = threadIdx.x & (lanes - 1);
  const int64_t total = d.rows << d.a;
  const bool valid = o < total;
  float acc = 0.f;
  if (valid) acc = merge_sum(d, merge_row(d, o >> d.a), uint32_t(o & ((int64_t(1) << d.a) - 1)), lane, lanes);
  for (int off = lanes >> 1; off > 0; off >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, off);
  if (valid && lane == 0) {
    const int64_t e = o >> d.a;
    const uint32_t b = uint32_t(o & ((int64_t(1) << d.a) - 1));
    store_out_f(d.dst, d.kind, d.plane_stride, d.rowmap[e] + d.colmap[b], acc * pow2_to_float(d.alpha));
  }
}

// Shared memory (floats) one SIMT tile needs for its A and B stages.
template <int BM, int BN, int kBK>
constexpr int gemm_tile_smem_floats() {
  return kBK * (BM + 4) + kBK * (BN + 4);
}

// Operand load: through the read-only path, or from L2 only (CG) for
// operands that other CTAs of the same launch wrote.
template <bool CG>
__device__ __forceinline__ float ld_operand(const float* p) {
  if constexpr (CG) return __ldcg(p);
  else return __ldg(p);
}

// A thread's TM x TN FP32 outputs (first row row0, first column c0), scaled and
// written through the layout maps; returns the FP64 sum of the FP32 sums of its
// GR x GC groups.
template <int TM, int TN, int GR = TM, int GC = TN>
__device__ __forceinline__ double store_tile_f32(const GemmArgs& a, const float (&acc)[TM][TN], int64_t row0,
                                                 int64_t c0, float alpha_f, void* Cout) {
  static_assert(TM % GR == 0 && TN % GC == 0 && (GC == TN || GC % 4 == 0), "whole groups");
  double sum = 0.0;
  float group[TN / GC] = {};
  // every map entry before the first store: the compiler may not move a load
  // over a store that might alias it, and one round trip per row is what the
  // epilogue then takes
  constexpr int kC = TN % 4 == 0 ? TN / 4 : TN;
  uint64_t rb[TM], cb[kC];
#pragma unroll
  for (int i = 0; i < TM; ++i) rb[i] = row0 + i < a.M ? __ldg(a.rowmap + row0 + i) : 0;
  const bool vec = a.vec4 && (TN % 4) == 0 && c0 + TN <= a.N;
#pragma unroll
  for (int j = 0; j < kC; ++j) {
    const int64_t col = c0 + j * (TN / kC);
    cb[j] = col < a.N ? __ldg(a.colmap + col) : 0;
  }
#pragma unroll
  for (int i = 0; i < TM; ++i) {
    const uint64_t rbase = rb[i];
    if (row0 + i >= a.M) {
      // (no such row)
    } else if (vec) {
#pragma unroll
      for (int j = 0; j + 3 < TN; j += 4) {
        float4 q;
        q.x = acc[i][j] * alpha_f; q.y = acc[i][j + 1] * alpha_f;
        q.z = acc[i][j + 2] * alpha_f; q.w = acc[i][j + 3] * alpha_f;
        group[j / GC] += (q.x + q.y) + (q.z + q.w);
        float4* dst = reinterpret_cast<float4*>(static_cast<float*>(Cout) + rbase + cb[j / 4]);
        if (a.accumulate) {
          const float4 o = *dst;
          q.x += o.x; q.y += o.y; q.z += o.z; q.w += o.w;
        }
        *dst = q;
      }
    } else {
#pragma unroll
      for (int j = 0; j < TN; ++j) {
        const int64_t col = c0 + j;
        if (col >= a.N) continue;
        const float v = acc[i][j] * alpha_f;
        group[j / GC] += v;
        float* dst = static_cast<float*>(Cout) + rbase + (kC == TN ? cb[j < kC ? j : 0] : __ldg(a.colmap + col));
        *dst = a.accumulate ? *dst + v : v;
      }
    }
    if ((i + 1) % GR == 0) {
#pragma unroll
      for (int j = 0; j < TN / GC; ++j) {
        sum += double(group[j]);
        group[j] = 0.f;
      }
    }
  }
  return sum;
}

// One BM x BN tile (origin m0, n0) of C = A B^T (Section 6.1) on NT threads
// (256 unless a launch gives the whole CTA to one tile), epilogue through
// the layout maps into Cout (the step's own output, or the one a
// single-query launch names); returns this thread's sum of the values it
// wrote (for the probability check).  smem_a / smem_b: kBK x (BM+4) and
// kBK x (BN+4) floats of shared memory.  CG: read the operands from L2 (they
// were written earlier in the same launch).
template <int BM, int BN, int TM, int TN, bool CHUNKED, int kBK, int NT = kOpThreads, bool CG = false>
__device__ __forceinline__ double gemm_tile(const GemmArgs& a, int64_t m0, int64_t n0, float* smem_a,
                                            float* smem_b, void* Cout) {
  constexpr int kThreads = NT;
  static_assert((BM / TM) * (BN / TN) == kThreads, "tile shape");
  constexpr int TX = BN / TN;
  float (*As)[BM + 4] = reinterpret_cast<float (*)[BM + 4]>(smem_a);
  float (*Bs)[BN + 4] = reinterpret_cast<float (*)[BN + 4]>(smem_b);

  const int tid = threadIdx.x;
  const int tx = tid % TX, ty = tid / TX;

  // alpha is a power of two: scaling an FP32 partial by it is exact
  const float alpha_f = pow2_to_float(a.alpha);
  float acc[TM][TN];
  double acc64[CHUNKED ? TM : 1][CHUNKED ? TN : 1];
#pragma unroll
  for (int i = 0; i < TM; ++i)
#pragma unroll
    for (int j = 0; j < TN; ++j) acc[i][j] = 0.f;
  if constexpr (CHUNKED) {
#pragma unroll
    for (int i = 0; i < TM; ++i)
#pragma unroll
      for (int j = 0; j < TN; ++j) acc64[i][j] = 0.0;
  }

  // A stage's operands: 16-byte words along the shared index, both operands'
  // loads in flight before their shared-memory stores (one memory round trip
  // per stage; four-byte loads in groups of four took up to eight).  A shared
  // index of 1 (an outer product) has no such words.
  constexpr int kQ = kBK / 4;
  constexpr int kLA = (BM * kQ + kThreads - 1) / kThreads;
  constexpr int kLB = (BN * kQ + kThreads - 1) / kThreads;
  auto ld4 = [](const float* p) -> float4 {
    if constexpr (CG) return __ldcg(reinterpret_cast<const float4*>(p));
    else return __ldg(reinterpret_cast<const float4*>(p));
  };
  // Row and first shared index of word i: a warp takes 8 rows x 4 words, whose
  // transposed stores meet in two lanes per bank (2 rows x 16 words, for a
  // stage of 64, in eight: 128 x 128 outputs of K = 256 with their merge 17.1
  // us, 14.8 so; 64 queries of K = 64 steps 189 -> 179).
  static_assert(BM % 8 == 0 && BN % 8 == 0 && kQ % 4 == 0, "whole warps of words");
  auto row_of = [](int i) -> int { return ((i >> 2) & 7) + 8 * ((i >> 5) / (kQ / 4)); };
  auto k_of = [](int i) -> int { return 4 * ((i & 3) + 4 * ((i >> 5) % (kQ / 4))); };
  for (int64_t k0 = 0; k0 < a.K; k0 += kBK) {
    if (a.K >= 4) {
      float4 ra[kLA], rb[kLB];
#pragma unroll
      for (int u = 0; u < kLA; ++u) {
        const int i = tid + u * kThreads, r = row_of(i), kk = k_of(i);
        ra[u] = make_float4(0.f, 0.f, 0.f, 0.f);
        if (i < BM * kQ && m0 + r < a.M && k0 + kk < a.K) ra[u] = ld4(a.A + (m0 + r) * a.K + k0 + kk);
      }
#pragma unroll
      for (int u = 0; u < kLB; ++u) {
        const int i = tid + u * kThreads, r = row_of(i), kk = k_of(i);
        rb[u] = make_float4(0.f, 0.f, 0.f, 0.f);
        if (i < BN * kQ && n0 + r < a.N && k0 + kk < a.K) rb[u] = ld4(a.B + (n0 + r) * a.K + k0 + kk);
      }
#pragma unroll
      for (int u = 0; u < kLA; ++u) {
        const int i = tid + u * kThreads, r = row_of(i), kk = k_of(i);
        if (i < BM * kQ) {
          As[kk][r] = ra[u].x; As[kk + 1][r] = ra[u].y; As[kk + 2][r] = ra[u].z; As[kk + 3][r] = ra[u].w;
        }
      }
#pragma unroll
      for (int u = 0; u < kLB; ++u) {
        const int i = tid + u * kThreads, r = row_of(i), kk = k_of(i);
        if (i < BN * kQ) {
          Bs[kk][r] = rb[u].x; Bs[kk + 1][r] = rb[u].y; Bs[kk + 2][r] = rb[u].z; Bs[kk + 3][r] = rb[u].w;
        }
      }
    } else {
      for (int i = tid; i < BM * kBK; i += kThreads) {
        const int r = i % BM, kk = i / BM;
        As[kk][r] = kk == 0 && m0 + r < a.M ? ld_operand<CG>(a.A + m0 + r) : 0.f;
      }
      for (int i = tid; i < BN * kBK; i += kThreads) {
        const int r = i % BN, kk = i / BN;
        Bs[kk][r] = kk == 0 && n0 + r < a.N ? ld_operand<CG>(a.B + n0 + r) : 0.f;
      }
    }
    __syncthreads();
#pragma unroll
    for (int kk = 0; kk < kBK; ++kk) {
      float af[TM], bf[TN];
#pragma unroll
      for (int i = 0; i < TM; ++i) af[i] = As[kk][ty * TM + i];
#pragma unroll
      for (int j = 0; j < TN; ++j) bf[j] = Bs[kk][tx * TN + j];
#pragma unroll
      for (int i = 0; i < TM; ++i)
#pragma unroll
        for (int j = 0; j < TN; ++j) acc[i][j] = fmaf(af[i], bf[j], acc[i][j]);
    }
    __syncthreads();
    if constexpr (CHUNKED) {
      const int64_t done = k0 + kBK;
      if ((done & (a.chunk - 1)) == 0 || done >= a.K) {
#pragma unroll
        for (int i = 0; i < TM; ++i)
#pragma unroll
          for (int j = 0; j < TN; ++j) {
            acc64[i][j] += f2d(acc[i][j] * alpha_f);
            acc[i][j] = 0.f;
          }
      }
    }
  }

  // FP32 outputs are scaled and summed in FP32; only FP64 outputs use the
  // FP64 pipe per element
  if constexpr (!CHUNKED)
    if (a.kind == OUT_F32) return store_tile_f32<TM, TN>(a, acc, m0 + ty * TM, n0 + tx * TN, alpha_f, Cout);
  float sum_f = 0.f;
  double sum_d = 0.0;
  uint64_t rb[TM], cb[TN];                 // map entries before any store, as above
#pragma unroll
  for (int i = 0; i < TM; ++i) rb[i] = m0 + ty * TM + i < a.M ? __ldg(a.rowmap + m0 + ty * TM + i) : 0;
#pragma unroll
  for (int j = 0; j < TN; ++j) cb[j] = n0 + tx * TN + j < a.N ? __ldg(a.colmap + n0 + tx * TN + j) : 0;
#pragma unroll
  for (int i = 0; i < TM; ++i) {
    const int64_t row = m0 + ty * TM + i;
    if (row >= a.M) continue;
    const uint64_t rbase = rb[i];
    const int64_t c0 = n0 + tx * TN;
#pragma unroll
    for (int j = 0; j < TN; ++j) {
      const int64_t col = c0 + j;
      if (col >= a.N) continue;
      double v;
      if constexpr (CHUNKED) v = acc64[i][j]; else v = f2d(acc[i][j] * alpha_f);
      if (a.kind == OUT_F64) sum_d += v; else sum_f += float(v);
      if (a.accumulate && a.kind == OUT_F64) {
        double* dst = static_cast<double*>(Cout) + rbase + cb[j];
        *dst += v;                          // slices add up in FP64
      } else if (a.accumulate && a.kind == OUT_F32) {
        float* dst = static_cast<float*>(Cout) + rbase + cb[j];
        *dst += float(v);
      } else {
        store_out(Cout, a.kind, a.plane_stride, rbase + cb[j], v);
      }
    }
  }
  return sum_d + double(sum_f);
}

// Two FP32 multiply-adds in one instruction (each rounded as fmaf does).
__device__ __forceinline__ void fma2(float2& d, float2 a, float2 b) {
  unsigned long long& dd = reinterpret_cast<unsigned long long&>(d);
  asm("fma.rn.f32x2 %0, %1, %2, %0;"
      : "+l"(dd)
      : "l"(reinterpret_cast<unsigned long long&>(a)), "l"(reinterpret_cast<unsigned long long&>(b)));
}

// The same tile of a long shared index (K a multiple of kPipeK, whole tiles:
// M a multiple of BM, N of BN; FP32 output), for steps that are bound by the
// FP32 units: the next stage's operands (16-byte loads) travel in registers,
// A during the first half of the current stage and B during the second, into
// the other shared-memory buffer (one CTA barrier per stage), and the
// multiply-adds are issued two columns at a time.  k runs upwards as in
// gemm_tile, so the values are the same bit for bit.  The probability check's
// FP32 groups are G x G outputs, those of the plain tile in its place: 4 x 4
// where 64 x 64 tiles would run (2^21 outputs: 128 tiles of 128 x 128 are too
// few), 8 x 8 beyond.  B's columns lie in
// shared memory with the two float4 halves of a thread's 8 columns apart, so
// that a warp's 16-byte reads do not collide.  128 threads with 8 x 8 outputs
// each, three CTAs per SM.  (Measured and not kept: 16 x 8 outputs a thread,
// two CTAs per SM, 1.4% faster at 4096 x 4096 x 256 and 11% slower at
// 4096 x 2048 x 256; A doubled in shared memory to save the register moves,
// 13% slower.)
// 4096 x 4096 x 256: 164 us, 52 TFLOP/s of the 75 that packed multiply-adds
// reach from registers (gemm_tile's unbuffered stages and scalar loads: 218
// us).  Before the epilogue read its map entries first it took 178 us, 4096 x
// 2048 x 256 131 -> 95 us and 4096 x 2048 x 64 47 -> 37 us.
constexpr int kPipeK = 16;
template <int BM, int BN>
constexpr int gemm_pipe_smem_floats() {
  return 2 * kPipeK * (BM + 4 + BN + 4);
}
constexpr int kPipeThreads = 128;
template <int BM, int BN, int TM, int TN, int G, bool CG = false>
__device__ __forceinline__ double gemm_tile_pipe(const GemmArgs& a, int64_t m0, int64_t n0, float* smem,
                                                 void* Cout) {
  constexpr int NT = kPipeThreads, TX = BN / TN;
  static_assert((BM / TM) * TX == NT && TM % 8 == 0 && TN % 4 == 0 && TN <= 8, "tile shape");
  constexpr int SA = BM + 4, SB = BN + 4, kStage = kPipeK * (SA + SB);
  constexpr int kQ = kPipeK / 4;                     // float4 per row and stage
  constexpr int LA = BM * kQ / NT, LB = BN * kQ / NT;
  static_assert(LA * NT == BM * kQ && LB * NT == BN * kQ, "whole loads");
  const int tid = threadIdx.x, tx = tid % TX, ty = tid / TX;
  const float* A = a.A + m0 * a.K;
  const float* B = a.B + n0 * a.K;
  auto ld4 = [](const float* p) -> float4 {
    if constexpr (CG) return __ldcg(reinterpret_cast<const float4*>(p));
    else return __ldg(reinterpret_cast<const float4*>(p));
  };
  // position of column c in a row of the B stage
  auto bpos = [](int c) -> int { return TN == 8 ? ((c >> 2) & 1) * (BN / 2) + (c >> 3) * 4 + (c & 3) : c; };
  constexpr int LR = LA > LB ? LA : LB;
  float4 r[LR];                                      // one operand of the next stage on its way
  auto fetch = [&](const float* P, auto cnt, int64_t k0) {
#pragma unroll
    for (int u = 0; u < cnt.value; ++u) {
      const int i = tid + u * NT;
      r[u] = ld4(P + int64_t(i / kQ) * a.K + k0 + 4 * (i % kQ));
    }
  };
  auto put_a = [&](float* st) {
#pragma unroll
    for (int u = 0; u < LA; ++u) {
      const int i = tid + u * NT;
      float* p = st + 4 * (i % kQ) * SA + i / kQ;
      p[0] = r[u].x; p[SA] = r[u].y; p[2 * SA] = r[u].z; p[3 * SA] = r[u].w;
    }
  };
  auto put_b = [&](float* st) {
#pragma unroll
    for (int u = 0; u < LB; ++u) {
      const int i = tid + u * NT;
      float* p = st + kPipeK * SA + 4 * (i % kQ) * SB + bpos(i / kQ);
      p[0] = r[u].x; p[SB] = r[u].y; p[2 * SB] = r[u].z; p[3 * SB] = r[u].w;
    }
  };
  const std::integral_constant<int, LA> la{};
  const std::integral_constant<int, LB> lb{};
  float2 acc[TM][TN / 2];
#pragma unroll
  for (int i = 0; i < TM; ++i)
#pragma unroll
    for (int j = 0; j < TN / 2; ++j) acc[i][j] = make_float2(0.f, 0.f);
  auto multiply = [&](const float* sa, const float* sb) {   // half a stage
#pragma unroll
    for (int kk = 0; kk < kPipeK / 2; ++kk) {
      float4 af[TM / 4], bf[TN / 4];
#pragma unroll
      for (int i = 0; i < TM / 4; ++i) af[i] = *reinterpret_cast<const float4*>(sa + kk * SA + 4 * i);
#pragma unroll
      for (int j = 0; j < TN / 4; ++j) bf[j] = *reinterpret_cast<const float4*>(sb + kk * SB + j * (BN / 2));
#pragma unroll
      for (int i = 0; i < TM; ++i) {
        const float x = reinterpret_cast<const float*>(af)[i];
#pragma unroll
        for (int j = 0; j < TN / 2; ++j) fma2(acc[i][j], make_float2(x, x), reinterpret_cast<const float2*>(bf)[j]);
      }
    }
  };
  fetch(A, la, 0);
  put_a(smem);
  fetch(B, lb, 0);
  put_b(smem);
  __syncthreads();
  int cur = 0;
  for (int64_t k0 = 0; k0 < a.K; k0 += kPipeK) {
    const bool more = k0 + kPipeK < a.K;
    const float* st = smem + cur * kStage;
    float* next = smem + (cur ^ 1) * kStage;
    const float* sa = st + ty * TM;
    const float* sb = st + kPipeK * SA + 4 * tx;
    if (more) fetch(A, la, k0 + kPipeK);
    multiply(sa, sb);
    if (more) {
      put_a(next);
      fetch(B, lb, k0 + kPipeK);
    }
    multiply(sa + kPipeK / 2 * SA, sb + kPipeK / 2 * SB);
    if (more) put_b(next);
    __syncthreads();
    cur ^= 1;
  }
  return store_tile_f32<TM, TN, G, G>(a, reinterpret_cast<const float(&)[TM][TN]>(acc), m0 + ty * TM, n0 + tx * TN,
                                      pow2_to_float(a.alpha), Cout);
}


// The probability check of a thread whose FP32 pair has left the finite range
// (an infinite bin, whose TwoSum error is NaN, or a sum beyond FP32's largest
// value): the same groups again, from the outputs the thread has written, in
// FP64 as gemm_tile adds them.  Rare, out of line.
template <int G, int R>
__device__ __noinline__ double band_sum_again(const float* out, const uint64_t* roff, int first, int step, int bm) {
  double sum = 0.0;
  for (int r0 = first; r0 < bm; r0 += step)
    for (int r = r0; r < r0 + R; r += G) {
      float g0 = 0.f, g1 = 0.f;
      for (int g = 0; g < G; ++g) {
        const float4 v = *reinterpret_cast<const float4*>(out + roff[r + g]);
        if constexpr (G == 2) {
          g0 = (g0 + v.x) + v.y;
          g1 = (g1 + v.z) + v.w;
        } else {
          g0 += (v.x + v.y) + (v.z + v.w);
        }
      }
      sum += double(g0);
      if constexpr (G == 2) sum += double(g1);
    }
  return sum;
}

// Bands: steps of a short shared index (K = 1, 4 or 16) with contiguous output
// columns (vec4) and FP32 output write far more than they read or multiply.
// In plain tiles a thread stores a few values after a chain of dependent
// memory round trips; a band's thread owns four columns and walks down the
// band's rows, 16 bytes stored per row.  k runs upwards, with the zero term
// that a shared index below the plain tile's stage of 16 gets there (it turns
// -0 into +0): the values are the same bit for bit.  The probability check's
// FP32 groups are the plain tile's too: G rows x 4 columns, or (G = 2) 2 x 2.
//
// Threads: CT = columns / 4 across the columns, 256 / CT row groups.
// K <= 4: a thread's four B rows stay in registers; A's rows are read from
// shared memory, each value doubled, so that two columns' multiply-adds are
// one instruction.  smem: 2 bm K floats and bm 8-byte offsets.
template <int K, int G, bool CG>
__device__ __forceinline__ double gemm_band_k(const GemmArgs& a, int64_t m0, int64_t n0, int bm, float* smem,
                                              void* Cout) {
  const int bn = band_cols(a), ct = bn >> 2, ct_log2 = __ffs(ct) - 1;
  const int tid = threadIdx.x, col = 4 * (tid & (ct - 1)), rg = tid >> ct_log2, nrg = kOpThreads >> ct_log2;
  float2* xs = reinterpret_cast<float2*>(smem);                       // [bm][K], doubled
  uint64_t* roff = reinterpret_cast<uint64_t*>(smem + 2 * bm * K);    // [bm]
  const uint64_t coff = __ldg(a.colmap + n0 + col);
  float2 y[K][2];
  {
    const float* Y = a.B + (n0 + col) * K;
    if constexpr (K >= 4) {
#pragma unroll
      for (int q = 0; q < K / 4; ++q) {
        float4 w[4];
#pragma unroll
        for (int c = 0; c < 4; ++c) {
          const float4* p = reinterpret_cast<const float4*>(Y + c * K) + q;
          if constexpr (CG) w[c] = __ldcg(p); else w[c] = __ldg(p);
        }
        y[4 * q][0] = make_float2(w[0].x, w[1].x); y[4 * q][1] = make_float2(w[2].x, w[3].x);
        y[4 * q + 1][0] = make_float2(w[0].y, w[1].y); y[4 * q + 1][1] = make_float2(w[2].y, w[3].y);
        y[4 * q + 2][0] = make_float2(w[0].z, w[1].z); y[4 * q + 2][1] = make_float2(w[2].z, w[3].z);
        y[4 * q + 3][0] = make_float2(w[0].w, w[1].w); y[4 * q + 3][1] = make_float2(w[2].w, w[3].w);
      }
    } else {
      y[0][0] = make_float2(ld_operand<CG>(Y), ld_operand<CG>(Y + 1));
      y[0][1] = make_float2(ld_operand<CG>(Y + 2), ld_operand<CG>(Y + 3));
    }
  }
  for (int i = tid; i < bm * K; i += kOpThreads) {
    const float x = ld_operand<CG>(a.A + m0 * K + i);
    xs[i] = make_float2(x, x);
  }
  for (int i = tid; i < bm; i += kOpThreads) roff[i] = __ldg(a.rowmap + m0 + i);
  __syncthreads();
  const float alpha = pow2_to_float(a.alpha);
  float* out = static_cast<float*>(Cout) + coff;
  float s_hi = 0.f, s_lo = 0.f;
  for (int r0 = rg * G; r0 < bm; r0 += nrg * G) {
    float g0 = 0.f, g1 = 0.f;
#pragma unroll
    for (int g = 0; g < G; ++g) {
      const float2* x = xs + (r0 + g) * K;
      float2 c0 = make_float2(0.f, 0.f), c1 = make_float2(0.f, 0.f);
      if constexpr (K >= 4) {
#pragma unroll
        for (int k = 0; k < K; k += 2) {
          const float4 w = *reinterpret_cast<const float4*>(x + k);
          fma2(c0, make_float2(w.x, w.y), y[k][0]);
          fma2(c1, make_float2(w.x, w.y), y[k][1]);
          fma2(c0, make_float2(w.z, w.w), y[k + 1][0]);
          fma2(c1, make_float2(w.z, w.w), y[k + 1][1]);
        }
      } else {
        fma2(c0, x[0], y[0][0]);
        fma2(c1, x[0], y[0][1]);
      }
      if constexpr (K < 16) {
        fma2(c0, make_float2(0.f, 0.f), make_float2(0.f, 0.f));
        fma2(c1, make_float2(0.f, 0.f), make_float2(0.f, 0.f));
      }
      const float4 v = make_float4(c0.x * alpha, c0.y * alpha, c1.x * alpha, c1.y * alpha);
      *reinterpret_cast<float4*>(out + roff[r0 + g]) = v;
      if constexpr (G == 2) {
        g0 = (g0 + v.x) + v.y;
        g1 = (g1 + v.z) + v.w;
      } else {
        g0 += (v.x + v.y) + (v.z + v.w);
      }
    }
    two_sum_add(s_hi, s_lo, g0);
    if constexpr (G == 2) two_sum_add(s_hi, s_lo, g1);
  }
  const double sum = isfinite(s_hi) ? double(s_hi) + double(s_lo) : band_sum_again<G, G>(out, roff, rg * G, nrg * G, bm);
  __syncthreads();                                   // the next band may reuse the shared memory
  return sum;
}
// K = 16: both operands in shared memory, k-major; 8 rows x 4 columns per
// thread and round, the multiply-adds of two rows in one instruction (four B
// rows of 16 in registers were loaded a line per lane, and took longer than
// the stores).  smem: 16 (bm + 4) + 16 (bn + 4) floats and bm offsets.
template <int G, bool CG>
__device__ __forceinline__ double gemm_band_16(const GemmArgs& a, int64_t m0, int64_t n0, int bm, float* smem,
                                               void* Cout) {
  const int bn = band_cols(a), ct = bn >> 2, ct_log2 = __ffs(ct) - 1;
  const int tid = threadIdx.x, col = 4 * (tid & (ct - 1)), rg = tid >> ct_log2, nrg = kOpThreads >> ct_log2;
  const int sx = bm + 4, sy = bn + 4;
  float* xs = smem;                                                   // [16][sx]
  float* ys = smem + 16 * sx;                                         // [16][sy]
  uint64_t* roff = reinterpret_cast<uint64_t*>(ys + 16 * sy);         // [bm]
  const uint64_t coff = __ldg(a.colmap + n0 + col);
  auto ld4 = [](const float* p) -> float4 {
    if constexpr (CG) return __ldcg(reinterpret_cast<const float4*>(p));
    else return __ldg(reinterpret_cast<const float4*>(p));
  };
  const float* X = a.A + m0 * 16;
  const float* Y = a.B + n0 * 16;
  // four 16-byte words in flight per thread (each row is four of them)
  auto stage = [&](const float* src, int rows, float* dst, int stride) {
    for (int i0 = tid; i0 < rows * 4; i0 += 4 * kOpThreads) {
      float4 w[4];
#pragma unroll
      for (int u = 0; u < 4; ++u)
        if (i0 + u * kOpThreads < rows * 4) w[u] = ld4(src + 4 * (i0 + u * kOpThreads));
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        const int i = i0 + u * kOpThreads;
        if (i < rows * 4) {
          float* p = dst + 4 * (i & 3) * stride + (i >> 2);
          p[0] = w[u].x; p[stride] = w[u].y; p[2 * stride] = w[u].z; p[3 * stride] = w[u].w;
        }
      }
    }
  };
  stage(X, bm, xs, sx);
  stage(Y, bn, ys, sy);
  for (int i = tid; i < bm; i += kOpThreads) roff[i] = __ldg(a.rowmap + m0 + i);
  __syncthreads();
  const float alpha = pow2_to_float(a.alpha);
  float* out = static_cast<float*>(Cout) + coff;
  float s_hi = 0.f, s_lo = 0.f;
  for (int r0 = rg * 8; r0 < bm; r0 += nrg * 8) {
    float2 acc[4][4];                                // [row pair][column]
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
      for (int c = 0; c < 4; ++c) acc[i][c] = make_float2(0.f, 0.f);
#pragma unroll 4
    for (int k = 0; k < 16; ++k) {
      const float4 y = *reinterpret_cast<const float4*>(ys + k * sy + col);
      const float4 x0 = *reinterpret_cast<const float4*>(xs + k * sx + r0);
      const float4 x1 = *reinterpret_cast<const float4*>(xs + k * sx + r0 + 4);
      const float2 xp[4] = {make_float2(x0.x, x0.y), make_float2(x0.z, x0.w), make_float2(x1.x, x1.y),
                            make_float2(x1.z, x1.w)};
      const float yc[4] = {y.x, y.y, y.z, y.w};
#pragma unroll
      for (int c = 0; c < 4; ++c)
#pragma unroll
        for (int i = 0; i < 4; ++i) fma2(acc[i][c], xp[i], make_float2(yc[c], yc[c]));
    }
    float g0 = 0.f, g1 = 0.f;
#pragma unroll
    for (int r = 0; r < 8; ++r) {
      float v[4];
#pragma unroll
      for (int c = 0; c < 4; ++c) v[c] = (r & 1 ? acc[r >> 1][c].y : acc[r >> 1][c].x) * alpha;
      *reinterpret_cast<float4*>(out + roff[r0 + r]) = make_float4(v[0], v[1], v[2], v[3]);
      if constexpr (G == 2) {
        g0 = (g0 + v[0]) + v[1];
        g1 = (g1 + v[2]) + v[3];
      } else {
        g0 += (v[0] + v[1]) + (v[2] + v[3]);
      }
      if ((r + 1) % G == 0) {
        two_sum_add(s_hi, s_lo, g0);
        if constexpr (G == 2) two_sum_add(s_hi, s_lo, g1);
        g0 = g1 = 0.f;
      }
    }
  }
  const double sum = isfinite(s_hi) ? double(s_hi) + double(s_lo) : band_sum_again<G, 8>(out, roff, rg * 8, nrg * 8, bm);
  __syncthreads();                                   // the next band may reuse the shared memory
  return sum;
}

template <int G, bool CG>
__device__ __forceinline__ double gemm_band(const GemmArgs& a, int64_t m0, int64_t n0, int bm, float* smem,
                                            void* Cout) {
  if (a.K == 16) return gemm_band_16<G, CG>(a, m0, n0, bm, smem, Cout);
  if (a.K == 4) return gemm_band_k<4, G, CG>(a, m0, n0, bm, smem, Cout);
  return gemm_band_k<1, G, CG>(a, m0, n0, bm, smem, Cout);
}

}  // namespace sqc

// One contraction step of the compute graph in FP32 on the SIMT cores
// (Section 6.1: contracting two tensors over their shared cut edges is the
// matrix product C = A B^T with both operands K-contiguous).
//
// Register-tiled: a CTA computes a BM x BN tile with 256 threads, each a
// TM x TN block of outputs, staging BK = 16 columns of A and B through
// shared memory.  The epilogue scales by alpha (2^-K on the last step),
// writes every element to rowmap[i] + colmap[j] of its destination (the
// layout the next step reads, or the canonical bin order), in FP32, FP64
// or three BF16 planes, and adds the written values into per-CTA FP64
// partial sums that the last CTA reduces in a fixed order (the probability
// check).  With `chunk` > 0 the shared index is summed in FP32 chunks of
// `chunk` terms that are added up in FP64 registers (the cross-chunk sum).
#include "device_ops.cuh"

namespace sqc {

namespace {

constexpr int kThreads = kOpThreads;

template <int BM, int BN, int TM, int TN, bool CHUNKED, int kBK>
__global__ void __launch_bounds__(kThreads, 2) gemm_simt_kernel(GemmArgs a) {
  pdl_wait();      // the previous kernel on the stream has completed
  pdl_trigger();   // the next one may start launching
  __shared__ __align__(16) float As[kBK * (BM + 4)];
  __shared__ __align__(16) float Bs[kBK * (BN + 4)];
  __shared__ double red[kThreads / 32];
  // M, N, BM, BN are powers of two: tile coordinates by shifts (64-bit
  // division is a long software sequence)
  const int64_t tiles_n = (a.N + BN - 1) / BN;
  const int tn_shift = __ffsll(tiles_n) - 1;
  const int64_t tile = int64_t(blockIdx.y) * gridDim.x + blockIdx.x;
  const int64_t m0 = (tile >> tn_shift) * BM;
  const int64_t n0 = (tile & (tiles_n - 1)) * BN;
  const double mysum = gemm_tile<BM, BN, TM, TN, CHUNKED, kBK>(a, m0, n0, As, Bs, a.C);
  if (a.partials) finish_total(mysum, a.partials, a.counter, a.total, red);
}

template <int BM, int BN, int TM, int TN, int G>
__global__ void __launch_bounds__(kPipeThreads, 3) gemm_pipe_kernel(GemmArgs a) {
  pdl_wait();      // the previous kernel on the stream has completed
  pdl_trigger();   // the next one may start launching
  extern __shared__ __align__(16) float smem[];
  __shared__ double red[kPipeThreads / 32];
  const int tn_shift = __ffsll(a.N / BN) - 1;
  const int64_t tile = blockIdx.x;
  const int64_t m0 = (tile >> tn_shift) * BM;
  const int64_t n0 = (tile & ((int64_t(1) << tn_shift) - 1)) * BN;
  const double mysum = gemm_tile_pipe<BM, BN, TM, TN, G>(a, m0, n0, smem, a.C);
  if (a.partials) finish_total(mysum, a.partials, a.counter, a.total, red);
}

// Steps of at most 1024 outputs and 16 shared terms, one after the other in
// one CTA: what a long chain of narrow subcircuits contracts to (a 59-block
// chain has 55 such steps in a row).  A launch each costs the host and the
// GPU about 3 us; here an output is one round of loads from L2 (both operand
// rows and the two map entries together), its multiply-adds and a store, and a
// thread's outputs follow each other: one round per 256 outputs of a step.  k
// runs upwards with gemm_tile's zero term below 16: the values are the same bit
// for bit.  Bound: the latency of L2.
__global__ void __launch_bounds__(kThreads) gemm_small_run_kernel(const __grid_constant__ SmallRun r) {
  pdl_wait();      // the previous kernel on the stream has completed
  pdl_trigger();   // the next one may start launching
  for (int i = 0; i < r.n; ++i) {
    const SmallStep& st = r.s[i];
    const int nl = st.n_log2, outs = 1 << (st.m_log2 + nl), K = 1 << st.k_log2;
    // (a step's output is none of its operands; the barrier below orders it
    // before the next step's loads)
    for (int o = threadIdx.x; o < outs; o += kThreads) {
      const int row = o >> nl, col = o & ((1 << nl) - 1);
      const uint64_t at = __ldg(st.rowmap + row) + __ldg(st.colmap + col);
      float acc = 0.f;
      if (K >= 4) {
        const float4* a = reinterpret_cast<const float4*>(st.A + row * K);
        const float4* b = reinterpret_cast<const float4*>(st.B + col * K);
        if (K == 16) {
          float4 x[4], y[4];
#pragma unroll
          for (int q = 0; q < 4; ++q) {
            x[q] = __ldcg(a + q);
            y[q] = __ldcg(b + q);
          }
#pragma unroll
          for (int q = 0; q < 4; ++q) {
            acc = fmaf(x[q].x, y[q].x, acc);
            acc = fmaf(x[q].y, y[q].y, acc);
            acc = fmaf(x[q].z, y[q].z, acc);
            acc = fmaf(x[q].w, y[q].w, acc);
          }
        } else {
          const float4 x = __ldcg(a), y = __ldcg(b);
          acc = fmaf(x.x, y.x, acc);
          acc = fmaf(x.y, y.y, acc);
          acc = fmaf(x.z, y.z, acc);
          acc = fmaf(x.w, y.w, acc);
          acc = fmaf(0.f, 0.f, acc);
        }
      } else {
        acc = fmaf(__ldcg(st.A + row), __ldcg(st.B + col), acc);
        acc = fmaf(0.f, 0.f, acc);
      }
      store_out_f(st.C, st.kind, st.plane_stride, at, acc);
    }
    __syncthreads();
  }
}

// Bands of a short shared index (gemm_band), one per CTA.
template <int G>
__global__ void __launch_bounds__(kThreads, 2) gemm_band_kernel(GemmArgs a, int bm) {
  pdl_wait();      // the previous kernel on the stream has completed
  pdl_trigger();   // the next one may start launching
  __shared__ __align__(16) float smem[kBandSmemFloats];
  __shared__ double red[kThreads / 32];
  const int bn = band_cols(a);
  const int c_shift = __ffsll(a.N / bn) - 1;
  const int64_t tile = blockIdx.x;
  const int64_t m0 = (tile >> c_shift) * bm, n0 = (tile & ((int64_t(1) << c_shift) - 1)) * bn;
  const double mysum = gemm_band<G, false>(a, m0, n0, bm, smem, a.C);
  if (a.partials) finish_total(mysum, a.partials, a.counter, a.total, red);
}

template <int G>
cudaError_t launch_band(const GemmArgs& a, int bm, cudaStream_t s) {
  return launch_k(gemm_band_kernel<G>, dim3(unsigned((a.M / bm) * (a.N / band_cols(a)))), dim3(kThreads), 0, s,
                  false, a, bm);
}

template <int BM, int BN, int TM, int TN, int G>
cudaError_t launch_pipe(const GemmArgs& a, cudaStream_t s) {
  return launch_k(gemm_pipe_kernel<BM, BN, TM, TN, G>, dim3(unsigned((a.M / BM) * (a.N / BN))), dim3(kPipeThreads),
                  sizeof(float) * gemm_pipe_smem_floats<BM, BN>(), s, false, a);
}

template <int BM, int BN, int TM, int TN, bool CH, int BK = 16>
cudaError_t launch_cfg(const GemmArgs& a, cudaStream_t s) {
  const int64_t tiles = ((a.M + BM - 1) / BM) * ((a.N + BN - 1) / BN);
  const int64_t gx = tiles < 65535 ? tiles : 65535;
  const int64_t gy = (tiles + gx - 1) / gx;
  if (gx * gy != tiles) {
    // tiles is a product of powers of two: gx = 65535 never divides it, so
    // fall back to an exact power-of-two split
    int64_t x = 32768;
    while (tiles % x) x >>= 1;
    return launch_k(gemm_simt_kernel<BM, BN, TM, TN, CH, BK>, dim3(unsigned(x), unsigned(tiles / x)), dim3(kThreads),
                    0, s, false, a);
  }
  return launch_k(gemm_simt_kernel<BM, BN, TM, TN, CH, BK>, dim3(unsigned(gx), unsigned(gy)), dim3(kThreads), 0, s,
                  false, a);
}

}  // namespace

namespace {
constexpr int64_t kBandLeast = int64_t(1) << 18;
}

cudaError_t gemm_simt_configure() {
  constexpr int smem = int(sizeof(float)) * gemm_pipe_smem_floats<128, 64>();
  const cudaError_t e =
      cudaFuncSetAttribute(gemm_pipe_kernel<128, 64, 8, 8, 8>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
  if (e != cudaSuccess) return e;
  return cudaFuncSetAttribute(gemm_pipe_kernel<128, 64, 8, 8, 4>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
}

cudaError_t launch_gemm_small_run(const SmallRun& r, cudaStream_t s) {
  if (r.n <= 0) return cudaSuccess;
  return launch_k(gemm_small_run_kernel, dim3(1), dim3(kThreads), 0, s, false, r);
}

cudaError_t launch_gemm_simt(const GemmArgs& a, cudaStream_t s) {
  if (a.M <= 0 || a.N <= 0 || a.K <= 0) return cudaErrorInvalidValue;
  const bool chunked = a.chunk > 0;
  const bool wide = !chunked && a.kind == OUT_F32;
  auto tiles = [&](int bm, int bn) { return ((a.M + bm - 1) / bm) * ((a.N + bn - 1) / bn); };
  const int64_t want = 152;   // at least one full wave of CTAs
  // bands (shared index up to 16, contiguous columns) once two per SM have
  // 1024 outputs each; the FP32 groups of the probability check stay those of
  // the plain tile the step would take
  const int64_t outs = a.M * a.N;
  if (wide && outs >= kBandLeast) {
    int64_t per = kBandOutputs;
    while (per > 1024 && outs / per < 2 * want) per >>= 1;
    const int g = tiles(128, 128) >= want ? 8 : (tiles(64, 64) >= want ? 4 : 2);
    const int bm = band_rows(a, g, per);
    if (bm > 0 && (a.M / bm) * (a.N / band_cols(a)) <= 0x7fffffff)
      return g == 8 ? launch_band<8>(a, bm, s) : (g == 4 ? launch_band<4>(a, bm, s) : launch_band<2>(a, bm, s));
  }
  // the pipelined form: whole tiles (M, N, K are powers of two) for every SM,
  // two stages or more -- with a single stage there is nothing to overlap --
  // and 16-byte aligned operands
  const int64_t pipe_tiles = (a.M / 128) * (a.N / 64);
  if (wide && a.K >= 2 * kPipeK && pipe_tiles >= want && pipe_tiles <= 0x7fffffff &&
      ((reinterpret_cast<uintptr_t>(a.A) | reinterpret_cast<uintptr_t>(a.B)) & 15) == 0)
    return tiles(128, 128) >= want ? launch_pipe<128, 64, 8, 8, 8>(a, s) : launch_pipe<128, 64, 8, 8, 4>(a, s);
  if (wide && tiles(128, 128) >= want) return launch_cfg<128, 128, 8, 8, false>(a, s);
  if (!wide && tiles(128, 64) >= want) {
    if (chunked) return launch_cfg<128, 64, 8, 4, true>(a, s);
    return launch_cfg<128, 64, 8, 4, false>(a, s);
  }
  // small steps: few CTAs, so stage up to 64 shared-index columns per
  // round (fewer dependent load rounds)
  const bool deep = a.K >= 64 && (!chunked || a.chunk % 64 == 0);
  if (tiles(64, 64) >= want) {
    if (chunked) return deep ? launch_cfg<64, 64, 4, 4, true, 64>(a, s) : launch_cfg<64, 64, 4, 4, true>(a, s);
    return deep ? launch_cfg<64, 64, 4, 4, false, 64>(a, s) : launch_cfg<64, 64, 4, 4, false>(a, s);
  }
  if (chunked) return deep ? launch_cfg<32, 32, 2, 2, true, 64>(a, s) : launch_cfg<32, 32, 2, 2, true>(a, s);
  return deep ? launch_cfg<32, 32, 2, 2, false, 64>(a, s) : launch_cfg<32, 32, 2, 2, false>(a, s);
}

}  // namespace sqc

// fp32 GEMM on the CUDA cores, used by fp32 models (the tiny workload):
// acc[M, N] = A[M, K] * B[N, K]^T with the same fused epilogues as the tensor
// core path.
//
// One 128-thread block per TM x 64 output tile (TM = 32, or 16 when 32-row
// tiles would leave SMs idle).  The GEMMs of this path are a few hundred rows
// by a few hundred columns, so a launch is paced by one block's K loop and its
// shared-memory reads: K advances 64 at a time through a cp.async ring; a warp
// owns TM / 4 whole rows, so that its reads of A are one address for all lanes,
// and a lane two columns.  Every output is one FMA chain in the order of k: a
// result depends neither on the tile nor on the number of rows.  (K split over
// thread groups of the block was 8 % faster over a generation, but its sums
// differ in the last bit, which moves tokens between nearly equal confidences.)
// Weights (b_weights) start loading ahead of the grid dependency.  Rows of the
// stage are padded to 68 floats: the eight column addresses of a quarter-warp's
// float4 reads fall into different banks.  16-row tiles run six stages, one
// block per SM: a launch that starts while its predecessor's last blocks run
// otherwise packs three blocks onto the first SMs that come free.  512 rows,
// events around each launch: W_down and W_o (N 256, K 1024 and 256) 15.5 us on
// average, QKV (N 768, K 256) 16.2, GLU (N 2 x 1024, K 256) 26, fusion hidden
// (N 1280, K 512) 42; with 64 x 64 tiles and 16 columns of K per synchronous
// step the residual projections took 77 us, QKV 33, GLU 37, fusion hidden 71.
// Eight warps of half as many columns: 10.9 -> 12.2 ms a generation.
// EPI_GLU tiles hold 32 gate and 32 up columns; EPI_QKV needs head_dim <= 64.
#include "kernels.h"

namespace tadm {
namespace {
constexpr int TN = 64, TK = 64, LDK = TK + 4, NT = 128;

struct SmemSrc {
  static constexpr bool kStaged = false;
  __device__ bool staged() const { return false; }
  __device__ void store64(int, int, const float (&)[32], const float (&)[32]) {}
  const float* row;  // accumulator row in shared memory
  __device__ __forceinline__ void load(int chunk, float (&v)[32]) {
#pragma unroll
    for (int i = 0; i < 32; ++i) v[i] = row[32 * chunk + i];
  }
};

__device__ __forceinline__ void cp_async(float* dst, const float* src, int bytes, bool ok, bool wide) {
  const int n = ok ? bytes : 0;   // 0: the destination is zero-filled
  if (wide) asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(smem_u32(dst)), "l"(src), "r"(n) : "memory");
  else asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"(smem_u32(dst)), "l"(src), "r"(n) : "memory");
}
__device__ __forceinline__ void cp_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_wait() { asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory"); }

template <int TM>
struct SimtCfg {
  static constexpr int STAGES = TM == 16 ? 6 : 3;
  static constexpr int FLOATS = STAGES * (TM + TN) * LDK;
};

// VEC: rows of A and B are 16-byte aligned and K % 4 == 0 (16-byte copies); otherwise 4-byte copies.
template <int EPI, int TM, bool VEC>
__global__ void __launch_bounds__(NT, TM == 16 ? 1 : 2) gemm_simt_kernel(const float* __restrict__ A, const float* __restrict__ B, int M,
                                                       int K, int lda, int ldb, int tiles_n, int n_rows_b, int b_split,
                                                       int b_early, EpiParams ep) {
  constexpr int STAGES = SimtCfg<TM>::STAGES, RM = TM / (NT / 32);
  extern __shared__ __align__(16) float smem[];
  const int tid = threadIdx.x, m0 = blockIdx.x / tiles_n * TM, nb = blockIdx.x % tiles_n;
  const int ksteps = (K + TK - 1) / TK;
  constexpr int W = VEC ? 4 : 1, CPR = TK / W;      // copies per row of a stage
  float* sA = smem;                                 // [STAGES][TM][LDK]
  float* sB = smem + STAGES * TM * LDK;             // [STAGES][TN][LDK]
  // A thread copies the same columns of every RPC-th row of a stage: its source is one pointer that steps by whole
  // rows.  With a row, a column and a 64-bit product per copy the copies' own instructions paced the kernel: 4096 x 4095
  // x 1023 (4-byte copies) 1589 -> 979 us, 4096 x 4096 x 512 514 -> 470, a fp32 generation of the tiny model 10.6 -> 10.0 ms.
  constexpr int RPC = NT / CPR;                     // rows that the block covers at a time
  const int r_in = tid / CPR, c_in = tid % CPR * W;
  auto load_a = [&](int ks) {
    float* dst = sA + (ks % STAGES) * TM * LDK + r_in * LDK + c_in;
    const int gk = ks * TK + c_in;
    const float* src = A + static_cast<size_t>(m0 + r_in) * lda + gk;
    const int rows = gk < K ? M - m0 - r_in : 0;    // rows of this thread's column that exist
#pragma unroll
    for (int r = 0; r < TM; r += RPC) {
      cp_async(dst + r * LDK, r < rows ? src : A, 4 * W, r < rows, VEC);
      src += static_cast<size_t>(RPC) * lda;
    }
  };
  auto load_b = [&](int ks) {
    float* dst = sB + (ks % STAGES) * TN * LDK + r_in * LDK + c_in;
    const int gk = ks * TK + c_in;
    // GLU: the tile's first half are gate rows, its second half their up rows
    const int n0 = b_split > 0 ? nb * (TN / 2) : nb * TN, up = b_split > 0 ? b_split - TN / 2 : 0;
    const float* src = B + static_cast<size_t>(n0 + r_in) * ldb + gk;
#pragma unroll
    for (int r = 0; r < TN; r += RPC) {
      const int gn = n0 + r_in + r + (r >= TN / 2 ? up : 0);
      const bool ok = gn < n_rows_b && gk < K;
      const float* p = r >= TN / 2 ? src + static_cast<ptrdiff_t>(up) * ldb : src;
      cp_async(dst + r * LDK, ok ? p : B, 4 * W, ok, VEC);
      src += static_cast<size_t>(RPC) * ldb;
    }
  };
  if (b_early) {
    for (int s = 0; s < STAGES - 1 && s < ksteps; ++s) load_b(s);
  }
  pdl_enter();
  for (int s = 0; s < STAGES - 1; ++s) {
    if (s < ksteps) {
      if (!b_early) load_b(s);
      load_a(s);
    }
    cp_commit();
  }
  // warp w owns rows RM w .. RM w + RM - 1 of the tile, its lane l columns l and l + 32
  const int warp = tid >> 5, lane = tid & 31;
  float acc[RM][2];
#pragma unroll
  for (int i = 0; i < RM; ++i) acc[i][0] = acc[i][1] = 0.0f;
  for (int ks = 0; ks < ksteps; ++ks) {
    cp_wait<STAGES - 2>();
    __syncthreads();                                // stage ks has landed; stage ks - 1 has been read by all
    if (ks + STAGES - 1 < ksteps) {
      load_b(ks + STAGES - 1);
      load_a(ks + STAGES - 1);
    }
    cp_commit();
    const float* a0 = sA + (ks % STAGES) * TM * LDK + RM * warp * LDK;
    const float* b0 = sB + (ks % STAGES) * TN * LDK + lane * LDK;
#pragma unroll
    for (int kk = 0; kk < TK; kk += 4) {
      float4 a[RM], b[2];
#pragma unroll
      for (int j = 0; j < 2; ++j) b[j] = *reinterpret_cast<const float4*>(b0 + 32 * j * LDK + kk);
#pragma unroll
      for (int i = 0; i < RM; ++i) a[i] = *reinterpret_cast<const float4*>(a0 + i * LDK + kk);
#pragma unroll
      for (int i = 0; i < RM; ++i)
#pragma unroll
        for (int j = 0; j < 2; ++j) {
          acc[i][j] = fmaf(a[i].x, b[j].x, acc[i][j]);
          acc[i][j] = fmaf(a[i].y, b[j].y, acc[i][j]);
          acc[i][j] = fmaf(a[i].z, b[j].z, acc[i][j]);
          acc[i][j] = fmaf(a[i].w, b[j].w, acc[i][j]);
        }
    }
  }
  if constexpr (EPI == EPI_RESID) {                 // element-wise, coalesced
#pragma unroll
    for (int i = 0; i < RM; ++i)
#pragma unroll
      for (int j = 0; j < 2; ++j) {
        const int m = m0 + RM * warp + i, n = nb * TN + lane + 32 * j;
        if (m < M && n < ep.N) {
          float* x = ep.resid + static_cast<size_t>(m) * ep.ldr + n;
          *x += ep.bias ? acc[i][j] + ld_param(ep.bias, ep.bias_bf16, n) : acc[i][j];
        }
      }
  }
  if constexpr (EPI == EPI_RESID) return;
  cp_wait<0>();
  __syncthreads();                                  // the stages are free: the tile goes over them
  constexpr int LDC = TN + 1;
  static_assert(TM * LDC <= SimtCfg<TM>::FLOATS, "the output tile fits the stages");
  float* sC = smem;
#pragma unroll
  for (int i = 0; i < RM; ++i)
#pragma unroll
    for (int j = 0; j < 2; ++j) sC[(RM * warp + i) * LDC + lane + 32 * j] = acc[i][j];
  __syncthreads();
  // the tile's 64 columns of a row go to one thread, or to two where the epilogue's columns are independent
  constexpr int NS = (EPI == EPI_STORE || EPI == EPI_SILU || EPI == EPI_ADD || EPI == EPI_FUSION1 || EPI == EPI_FUSION2 ||
                      EPI == EPI_PA_UP) ? 2 : 1;
  if (tid < TM * NS) {
    SmemSrc src{sC + (tid % TM) * LDC};
    epilogue_row<EPI>(ep, m0 + tid % TM, nb, TN, src, tid / TM, NS);
  }
}

template <int EPI, int TM, bool VEC>
cudaError_t launch_tile(const GemmCall& g, int dev, int tiles_n, int b_split, int n_rows_b, const EpiParams& ep,
                        cudaStream_t s) {
  constexpr int smem = SimtCfg<TM>::FLOATS * 4;
  static PerDevice ready;
  cudaError_t e = cudaSuccess;
  if (ready.get(dev, [&] {
        e = cudaFuncSetAttribute(gemm_simt_kernel<EPI, TM, VEC>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
        return e == cudaSuccess ? 1 : 0;
      }) <= 0)
    return e;
  const unsigned grid = static_cast<unsigned>(tiles_n) * static_cast<unsigned>((g.M + TM - 1) / TM);
  launch_pdl(gemm_simt_kernel<EPI, TM, VEC>, grid, NT, smem, s, static_cast<const float*>(g.A),
             static_cast<const float*>(g.B), g.M, g.K, g.lda, g.ldb, tiles_n, n_rows_b, b_split, g.b_weights ? 1 : 0, ep);
  return cudaGetLastError();
}

template <int EPI>
cudaError_t launch(const GemmCall& g, int tiles_n, int b_split, int n_rows_b, const EpiParams& ep, cudaStream_t s) {
  int dev = 0;
  const int n_sms = current_sms(&dev);
  const bool vec = g.K % 4 == 0 && g.lda % 4 == 0 && g.ldb % 4 == 0 &&
                   ((reinterpret_cast<uintptr_t>(g.A) | reinterpret_cast<uintptr_t>(g.B)) & 15) == 0;
  // 16-row tiles until 32-row tiles alone put a block on every SM (512 x 256: 64 against 128 blocks)
  const bool tall = static_cast<int64_t>(tiles_n) * ((g.M + 31) / 32) >= n_sms;
  if (vec)
    return tall ? launch_tile<EPI, 32, true>(g, dev, tiles_n, b_split, n_rows_b, ep, s)
                : launch_tile<EPI, 16, true>(g, dev, tiles_n, b_split, n_rows_b, ep, s);
  return launch_tile<EPI, 32, false>(g, dev, tiles_n, b_split, n_rows_b, ep, s);
}
}  // namespace

int gemm_simt_tiles_n(int N, int epi) { return epi == EPI_GLU ? (N + 31) / 32 : (N + 63) / 64; }

const char* gemm_simt(const GemmCall& g, cudaStream_t s) {
  if (g.M <= 0 || g.N <= 0 || g.K <= 0) return nullptr;
  const bool glu = g.epi == EPI_GLU;
  if (glu && g.N % 32) return "GLU GEMM (fp32) needs the FFN width to be a multiple of 32";
  if (g.epi == EPI_QKV && TN % g.ep.head_dim) return "fp32 path needs head_dim dividing 64";
  if (g.epi == EPI_PA_GATE && g.N > TN) return "fp32 gate GEMM needs N <= 64";
  const int tiles_n = gemm_simt_tiles_n(g.N, g.epi);
  EpiParams ep = g.ep;
  ep.M = g.M;
  ep.N = g.N;
  ep.n_tiles = tiles_n;
  const int b_split = glu ? g.N : 0;
  const int n_rows_b = glu ? 2 * g.N : g.N;
  cudaError_t e;
  switch (g.epi) {
    case EPI_STORE: e = launch<EPI_STORE>(g, tiles_n, b_split, n_rows_b, ep, s); break;
    case EPI_RESID: e = launch<EPI_RESID>(g, tiles_n, b_split, n_rows_b, ep, s); break;
    case EPI_QKV: e = launch<EPI_QKV>(g, tiles_n, b_split, n_rows_b, ep, s); break;
    case EPI_GLU: e = launch<EPI_GLU>(g, tiles_n, b_split, n_rows_b, ep, s); break;
    case EPI_FUSION1: e = launch<EPI_FUSION1>(g, tiles_n, b_split, n_rows_b, ep, s); break;
    case EPI_FUSION2: e = launch<EPI_FUSION2>(g, tiles_n, b_split, n_rows_b, ep, s); break;
    case EPI_LMHEAD: e = launch<EPI_LMHEAD>(g, tiles_n, b_split, n_rows_b, ep, s); break;
    case EPI_PA_UP: e = launch<EPI_PA_UP>(g, tiles_n, b_split, n_rows_b, ep, s); break;
    case EPI_SILU: e = launch<EPI_SILU>(g, tiles_n, b_split, n_rows_b, ep, s); break;
    case EPI_ADD: e = launch<EPI_ADD>(g, tiles_n, b_split, n_rows_b, ep, s); break;
    case EPI_PA_GATE: e = launch<EPI_PA_GATE>(g, tiles_n, b_split, n_rows_b, ep, s); break;
    default: return "unknown epilogue";
  }
  return e == cudaSuccess ? nullptr : cudaGetErrorString(e);
}

}  // namespace tadm

// Split-K reduction for the tcgen05 GEMM: sums the fp32 partials of the K
// slices in slice order (deterministic) and runs the GEMM's own epilogue on
// that sum, in one launch with coalesced reads: element-wise for the epilogues
// whose outputs depend on one column (GLU: a gate and an up column), a warp
// per head row for QKV (QK-norm, RoPE, cache write), a warp per row for the
// paired-attention gate.  The output head, whose partials need whole 128-column
// runs of a row, takes two launches: the sum into slice 0, then the epilogue,
// one thread per (output row, half of a 256-column tile).  Outputs that are not
// 16-byte aligned are not split (splitk_takes).
// With two launches for every epilogue the reductions took 15 us for the QKV
// projection of a 32-row block step, 9 us for its GLU and 20 us for the gate of
// 256 rows (16 to 64 blocks, rows read by one lane each).  With one launch each
// a batch-1 block step 542 -> 496 us, a 27 B block step 1108 -> 1060 us.
#include "kernels.h"

namespace tadm {
namespace {

// row of slice 0 at a tile's first column
struct PartSrc {
  static constexpr bool kStaged = false;
  const float* row;
  __device__ __forceinline__ void load(int chunk, float (&v)[32]) {
    const float4* p = reinterpret_cast<const float4*>(row + 32 * chunk);
#pragma unroll
    for (int q = 0; q < 8; ++q) {
      const float4 t = p[q];
      v[4 * q] = t.x; v[4 * q + 1] = t.y; v[4 * q + 2] = t.z; v[4 * q + 3] = t.w;
    }
  }
};

// Output head, phase 2: the epilogue on slice 0.  Block: 32 rows x the two
// column halves of a tile (the two partials that the tensor-core path writes).
__global__ void __launch_bounds__(64) splitk_head_kernel(EpiParams ep, const float* __restrict__ part, int ldp) {
  pdl_enter();
  const int m = blockIdx.x * 32 + (threadIdx.x & 31), nb = blockIdx.y;
  if (m >= ep.M) return;
  PartSrc src{part + static_cast<size_t>(m) * ldp + nb * 256};
  epilogue_row<EPI_LMHEAD>(ep, m, nb, 256, src, threadIdx.x >> 5, 2);
}

// Output head, phase 1: slice 0 <- sum of all slices in slice order, one float4 per thread.
__global__ void __launch_bounds__(256) splitk_sum_kernel(float* __restrict__ part, size_t stride, size_t n4,
                                                         int splits) {
  pdl_enter();
  const size_t i = blockIdx.x * static_cast<size_t>(blockDim.x) + threadIdx.x;
  if (i >= n4) return;
  float4* p = reinterpret_cast<float4*>(part);
  float4 a = p[i];
  for (int ks = 1; ks < splits; ++ks) {
    const float4 t = p[i + ks * (stride / 4)];
    a.x += t.x; a.y += t.y; a.z += t.z; a.w += t.w;
  }
  p[i] = a;
}

// four consecutive elements at element offset `off` of a bf16 or fp32 array (8- / 16-byte aligned)
__device__ __forceinline__ float4 ld4(const void* base, int bf, size_t off) {
  if (!bf) return *reinterpret_cast<const float4*>(static_cast<const float*>(base) + off);
  const uint2 u = *reinterpret_cast<const uint2*>(static_cast<const bf16*>(base) + off);
  const float2 a = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&u.x));
  const float2 b = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&u.y));
  return make_float4(a.x, a.y, b.x, b.y);
}
__device__ __forceinline__ void st4(void* base, int bf, size_t off, const float4& v) {
  if (!bf) {
    *reinterpret_cast<float4*>(static_cast<float*>(base) + off) = v;
    return;
  }
  __nv_bfloat162 a = __floats2bfloat162_rn(v.x, v.y), b = __floats2bfloat162_rn(v.z, v.w);
  *reinterpret_cast<uint2*>(static_cast<bf16*>(base) + off) =
      make_uint2(*reinterpret_cast<uint32_t*>(&a), *reinterpret_cast<uint32_t*>(&b));
}
template <class F>
__device__ __forceinline__ float4 map4(const float4& a, F f) { return make_float4(f(a.x), f(a.y), f(a.z), f(a.w)); }
__device__ __forceinline__ float4 add4(const float4& a, const float4& b) {
  return make_float4(a.x + b.x, a.y + b.y, a.z + b.z, a.w + b.w);
}
__device__ __forceinline__ float4 mul4(const float4& a, const float4& b) {
  return make_float4(a.x * b.x, a.y * b.y, a.z * b.z, a.w * b.w);
}
__device__ __forceinline__ float4 slice_sum(const float* p, size_t stride, int splits) {
  float4 a = *reinterpret_cast<const float4*>(p);
  for (int ks = 1; ks < splits; ++ks) a = add4(a, *reinterpret_cast<const float4*>(p + ks * stride));
  return a;
}

// Element-wise epilogues in one launch: each thread sums four consecutive
// columns of one row over the slices in slice order, then runs the epilogue on
// them, with coalesced 16-byte accesses.
// The epilogue's other inputs (residual, base, gate, bias) are read ahead of the
// grid dependency: their writers ran before the GEMM whose partials this kernel
// waits for, and that GEMM writes nothing else.
template <int EPI>
__global__ void __launch_bounds__(256) splitk_elem_kernel(EpiParams ep, const float* __restrict__ part, size_t stride,
                                                          int ldp, int splits) {
  const int n4 = ep.N / 4;
  const size_t i = blockIdx.x * static_cast<size_t>(blockDim.x) + threadIdx.x;
  const bool on = i < static_cast<size_t>(ep.M) * n4;
  const int m = on ? static_cast<int>(i / n4) : 0, n = on ? static_cast<int>(i % n4) * 4 : 0;
  const size_t row = static_cast<size_t>(m);
  float4 x = make_float4(0.0f, 0.0f, 0.0f, 0.0f), b = x, g = x;
  float gs = 0.0f;
  if constexpr (EPI == EPI_RESID || EPI == EPI_FUSION1 || EPI == EPI_FUSION2) {
    if (on && ep.bias) b = ld4(ep.bias, ep.bias_bf16, n);
  }
  if constexpr (EPI == EPI_RESID) {
    if (on) x = ld4(ep.resid, 0, row * ep.ldr + n);
  } else if constexpr (EPI == EPI_ADD || EPI == EPI_FUSION2 || EPI == EPI_PA_UP) {
    if (on) x = ld4(ep.base, 0, row * ep.ldb + n);
    if constexpr (EPI == EPI_FUSION2)
      if (on) g = ld4(ep.gate, ep.out_bf16, row * ep.ldg + n);
    if constexpr (EPI == EPI_PA_UP)
      if (on) gs = static_cast<const float*>(ep.gate)[m] * ep.rowscale[m];
  }
  pdl_enter();
  if (!on) return;
  if constexpr (EPI == EPI_GLU) {   // a tile's 256 columns: 128 gate columns, then their up columns
    const float* p = part + row * ldp + (n / 128) * 256 + n % 128;
    const float4 ga = slice_sum(p, stride, splits), u = slice_sum(p + 128, stride, splits);
    const bool tanh = ep.glu != 0;
    st4(ep.out, ep.out_bf16, row * ep.ldo + n,
        mul4(map4(ga, [&](float v) { return tanh ? gelu_tanh_f(v) : silu_f(v); }), u));
    return;
  }
  float4 a = slice_sum(part + row * ldp + n, stride, splits);
  if constexpr (EPI == EPI_RESID || EPI == EPI_FUSION1 || EPI == EPI_FUSION2) {
    if (ep.bias) a = add4(a, b);
  }
  if constexpr (EPI == EPI_RESID) {
    st4(ep.resid, 0, row * ep.ldr + n, add4(x, a));
  } else if constexpr (EPI == EPI_STORE) {
    st4(ep.out, ep.out_bf16, row * ep.ldo + n, a);
  } else if constexpr (EPI == EPI_SILU) {
    st4(ep.out, ep.out_bf16, row * ep.ldo + n, map4(a, [](float v) { return silu_f(v); }));
  } else if constexpr (EPI == EPI_ADD) {
    a = add4(x, a);
    st4(ep.out, 0, row * ep.ldo + n, a);
    if (ep.out2) st4(ep.out2, ep.out_bf16, row * ep.ldo2 + n, a);
  } else if constexpr (EPI == EPI_FUSION1) {
    if (n < ep.d_split) st4(ep.out, ep.out_bf16, row * ep.ldo + n, map4(a, [](float v) { return sigmoid_f(v); }));
    else st4(ep.out2, ep.out_bf16, row * ep.ldo2 + n - ep.d_split, map4(a, [](float v) { return gelu_erf_f(v); }));
  } else if constexpr (EPI == EPI_FUSION2) {
    st4(ep.out, 0, row * ep.ldo + n, add4(x, mul4(g, a)));
  } else if constexpr (EPI == EPI_PA_UP) {
    st4(ep.out, 0, row * ep.ldo + n, add4(x, map4(a, [&](float v) { return gs * v; })));
  }
}

// true when the element-wise kernel serves this epilogue (aligned rows, N % 4 == 0)
bool elem_ok(int epi, const EpiParams& ep, int ldp) {
  if (ep.N % 4 || ldp % 4) return false;
  auto al = [](const void* p, int ld) { return ld % 4 == 0 && (reinterpret_cast<uintptr_t>(p) & 15) == 0; };
  const bool bias = !ep.bias || al(ep.bias, 0);
  switch (epi) {
    case EPI_RESID: return al(ep.resid, ep.ldr) && bias;
    case EPI_STORE:
    case EPI_SILU:
    case EPI_GLU: return al(ep.out, ep.ldo);
    case EPI_ADD: return al(ep.out, ep.ldo) && al(ep.base, ep.ldb) && (!ep.out2 || al(ep.out2, ep.ldo2));
    case EPI_FUSION1: return al(ep.out, ep.ldo) && al(ep.out2, ep.ldo2) && ep.d_split % 4 == 0 && bias;
    case EPI_FUSION2: return al(ep.out, ep.ldo) && al(ep.base, ep.ldb) && al(ep.gate, ep.ldg) && bias;
    case EPI_PA_UP: return al(ep.out, ep.ldo) && al(ep.base, ep.ldb);
    default: return false;
  }
}

// QKV epilogue on the slice sums: a block takes 8 rows of one head, one per
// warp; a lane holds the rotate-half pairs (i, i + HD / 2) of HD / 64
// consecutive dims i, so partials, Q and K move in whole lines.  V rows cross
// shared memory and leave transposed, 8 positions of a dim at a time.
template <int HD>
__global__ void __launch_bounds__(256) splitk_qkv_kernel(EpiParams ep, const float* __restrict__ part, size_t stride,
                                                         int ldp, int splits) {
  constexpr int P = HD / 64, H2 = HD / 2, RB = 8;
  __shared__ bf16 sv[HD][RB + 2];
  __shared__ __align__(16) float sr[RB][HD];       // a warp's row, for QK-norm
  const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int gh = blockIdx.y, m0 = blockIdx.x * RB;
  int region = 2, head = gh - ep.n_heads - ep.n_kv_heads;
  if (gh < ep.n_heads) { region = 0; head = gh; }
  else if (gh < ep.n_heads + ep.n_kv_heads) { region = 1; head = gh - ep.n_heads; }
  const void* gain = region == 0 ? ep.q_gain : region == 1 ? ep.k_gain : nullptr;
  const int rr = w, m = m0 + rr;
  const int b = m / ep.R, r = m - b * ep.R, pos = ep.ctx + r;
  float2 cs[P];                                    // constant table, often no longer in L2: read while the GEMM runs
#pragma unroll
  for (int t = 0; t < P; ++t)
    cs[t] = ep.rope && region < 2 && m < ep.M ? ep.rope_tab[static_cast<size_t>(lane * P + t) * ep.rope_npos + pos]
                                              : make_float2(1.0f, 0.0f);
  pdl_enter();
  if (m < ep.M) {                                  // uniform across the warp
    const float* p = part + static_cast<size_t>(m) * ldp + gh * HD + lane * P;
    float a[P], c[P];
#pragma unroll
    for (int t = 0; t < P; ++t) a[t] = c[t] = 0.0f;
#pragma unroll 8
    for (int ks = 0; ks < splits; ++ks) {
      const float* q = p + ks * stride;
      if constexpr (P == 2) {
        const float2 x = *reinterpret_cast<const float2*>(q), y = *reinterpret_cast<const float2*>(q + H2);
        a[0] += x.x; a[1] += x.y; c[0] += y.x; c[1] += y.y;
      } else {
        a[0] += q[0];
        c[0] += q[H2];
      }
    }
    if (region == 2) {
#pragma unroll
      for (int t = 0; t < P; ++t) {
        sv[lane * P + t][rr] = __float2bfloat16_rn(a[t]);
        sv[H2 + lane * P + t][rr] = __float2bfloat16_rn(c[t]);
      }
    }
    if (gain) {
      // squares in column order, as the epilogue of an unsplit GEMM adds them: the row crosses shared memory and every
      // lane runs the same chain (hd dependent FMAs on broadcast reads)
      float* row = sr[w];
#pragma unroll
      for (int t = 0; t < P; ++t) {
        row[lane * P + t] = a[t];
        row[H2 + lane * P + t] = c[t];
      }
      __syncwarp();
      float ss = 0.0f;
#pragma unroll 8
      for (int n = 0; n < HD; n += 4) {
        const float4 x = *reinterpret_cast<const float4*>(row + n);
        ss = fmaf(x.w, x.w, fmaf(x.z, x.z, fmaf(x.y, x.y, fmaf(x.x, x.x, ss))));
      }
      const float inv = rsqrtf(ss / static_cast<float>(HD) + ep.qk_eps);
#pragma unroll
      for (int t = 0; t < P; ++t) {
        a[t] *= inv * ld_param(gain, ep.bias_bf16, lane * P + t);
        c[t] *= inv * ld_param(gain, ep.bias_bf16, H2 + lane * P + t);
      }
    }
    if (ep.rope && region < 2) {
#pragma unroll
      for (int t = 0; t < P; ++t) {
        const float x = a[t], y = c[t];
        a[t] = x * cs[t].x - y * cs[t].y;
        c[t] = y * cs[t].x + x * cs[t].y;
      }
    }
    bf16* dst = region == 0
                    ? static_cast<bf16*>(ep.q) + ((static_cast<size_t>(b) * ep.n_heads + head) * ep.R + r) * HD
                    : static_cast<bf16*>(ep.k) + ((static_cast<size_t>(b) * ep.n_kv_heads + head) * ep.kv_stride + pos) * HD;
    if (region < 2) {
      if constexpr (P == 2) {
        *reinterpret_cast<__nv_bfloat162*>(dst + 2 * lane) = __floats2bfloat162_rn(a[0], a[1]);
        *reinterpret_cast<__nv_bfloat162*>(dst + H2 + 2 * lane) = __floats2bfloat162_rn(c[0], c[1]);
      } else {
        dst[lane] = __float2bfloat16_rn(a[0]);
        dst[H2 + lane] = __float2bfloat16_rn(c[0]);
      }
    }
  }
  if (region != 2) return;                         // uniform across the block
  __syncthreads();
  for (int i = threadIdx.x; i < HD * RB; i += 256) {
    const int d = i / RB, rr = i % RB, m = m0 + rr;
    if (m >= ep.M) continue;
    const int b = m / ep.R, pos = ep.ctx + m - b * ep.R;
    static_cast<bf16*>(ep.v)[((static_cast<size_t>(b) * ep.n_kv_heads + head) * HD + d) * ep.kv_stride + pos] = sv[d][rr];
  }
}

// Paired-attention gate on the slice sums: one warp per row (N <= 256 columns,
// N % 4 == 0).  The lanes sum the slices and take the SiLU, whole lines at a
// time; one lane adds the products in column order, as the epilogue of an
// unsplit GEMM does, so that the gate's order of sums is the same on both
// paths (256 dependent FMAs, under 1 us).
constexpr int kGateCols = 256;
__global__ void __launch_bounds__(256) splitk_gate_kernel(EpiParams ep, const float* __restrict__ part, size_t stride,
                                                          int ldp, int splits) {
  __shared__ float2 term[8][kGateCols];             // (SiLU of the column, its weight)
  pdl_enter();
  const int m = blockIdx.x * 8 + (threadIdx.x >> 5), lane = threadIdx.x & 31;
  if (m >= ep.M) return;                            // uniform across the warp
  float2* t = term[threadIdx.x >> 5];
  for (int n = 4 * lane; n < ep.N; n += 128) {
    const float4 a = slice_sum(part + static_cast<size_t>(m) * ldp + n, stride, splits);
    t[n] = make_float2(silu_f(a.x), ld_param(ep.vec, ep.bias_bf16, n));
    t[n + 1] = make_float2(silu_f(a.y), ld_param(ep.vec, ep.bias_bf16, n + 1));
    t[n + 2] = make_float2(silu_f(a.z), ld_param(ep.vec, ep.bias_bf16, n + 2));
    t[n + 3] = make_float2(silu_f(a.w), ld_param(ep.vec, ep.bias_bf16, n + 3));
  }
  __syncwarp();
  if (lane != 0) return;
  float s = 0.0f;
#pragma unroll 16
  for (int n = 0; n < ep.N; ++n) s = fmaf(t[n].x, t[n].y, s);
  static_cast<float*>(ep.out)[m] = sigmoid_f(s + ld_param(ep.bias, ep.bias_bf16, 0));
}

template <int EPI>
cudaError_t launch_elem(const EpiParams& ep, const float* part, size_t stride, int ldp, int splits, cudaStream_t s) {
  const size_t n = static_cast<size_t>(ep.M) * (ep.N / 4);
  launch_pdl(splitk_elem_kernel<EPI>, static_cast<unsigned>((n + 255) / 256), 256, 0, s, ep, part, stride, ldp, splits);
  return cudaGetLastError();
}

cudaError_t launch_qkv(const EpiParams& ep, const float* part, size_t stride, int ldp, int splits, cudaStream_t s) {
  const dim3 grid((ep.M + 7) / 8, ep.n_heads + 2 * ep.n_kv_heads);
  if (ep.head_dim == 64) launch_pdl(splitk_qkv_kernel<64>, grid, 256, 0, s, ep, part, stride, ldp, splits);
  else launch_pdl(splitk_qkv_kernel<128>, grid, 256, 0, s, ep, part, stride, ldp, splits);
  return cudaGetLastError();
}

cudaError_t launch_head(const EpiParams& ep, float* part, size_t stride, int ldp, int splits, int n_tiles_n,
                        cudaStream_t s) {
  const size_t n4 = static_cast<size_t>(ep.M) * ldp / 4;
  launch_pdl(splitk_sum_kernel, static_cast<unsigned>((n4 + 255) / 256), 256, 0, s, part, stride, n4, splits);
  launch_pdl(splitk_head_kernel, dim3((ep.M + 31) / 32, n_tiles_n), 64, 0, s, ep, part, ldp);
  return cudaGetLastError();
}
}  // namespace

bool splitk_takes(int epi, const EpiParams& ep, int ldp) {
  switch (epi) {
    case EPI_LMHEAD: return true;
    case EPI_QKV: return ep.out_bf16 && (ep.head_dim == 64 || ep.head_dim == 128);
    case EPI_PA_GATE: return ep.N % 4 == 0 && ep.N <= kGateCols;
    default: return elem_ok(epi, ep, ldp);
  }
}

const char* splitk_reduce(int epi, const EpiParams& ep, float* part, size_t stride, int ldp, int splits, int n_tiles_n,
                          cudaStream_t s, int* launches) {
  if (!splitk_takes(epi, ep, ldp)) return "split-K reduction of an output that it does not take";
  *launches = epi == EPI_LMHEAD ? 2 : 1;
  cudaError_t e;
  switch (epi) {
    case EPI_STORE: e = launch_elem<EPI_STORE>(ep, part, stride, ldp, splits, s); break;
    case EPI_RESID: e = launch_elem<EPI_RESID>(ep, part, stride, ldp, splits, s); break;
    case EPI_QKV: e = launch_qkv(ep, part, stride, ldp, splits, s); break;
    case EPI_GLU: e = launch_elem<EPI_GLU>(ep, part, stride, ldp, splits, s); break;
    case EPI_FUSION1: e = launch_elem<EPI_FUSION1>(ep, part, stride, ldp, splits, s); break;
    case EPI_FUSION2: e = launch_elem<EPI_FUSION2>(ep, part, stride, ldp, splits, s); break;
    case EPI_LMHEAD: e = launch_head(ep, part, stride, ldp, splits, n_tiles_n, s); break;
    case EPI_PA_UP: e = launch_elem<EPI_PA_UP>(ep, part, stride, ldp, splits, s); break;
    case EPI_SILU: e = launch_elem<EPI_SILU>(ep, part, stride, ldp, splits, s); break;
    case EPI_ADD: e = launch_elem<EPI_ADD>(ep, part, stride, ldp, splits, s); break;
    case EPI_PA_GATE:
      launch_pdl(splitk_gate_kernel, (ep.M + 7) / 8, 256, 0, s, ep, part, stride, ldp, splits);
      e = cudaGetLastError();
      break;
    default: return "unknown epilogue";
  }
  return e == cudaSuccess ? nullptr : cudaGetErrorString(e);
}

}  // namespace tadm

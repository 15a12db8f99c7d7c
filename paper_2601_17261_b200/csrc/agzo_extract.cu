// The two products of Algorithm 1 (SubspaceExtract) with X on CUDA cores in fp32, for any dtype,
// pitch and size; the tensor-core path (agzo_extract_tc.cu) replaces them when the layer's shape
// allows it.  qr(Y) is in agzo_panel_qr.cu.
//
// Ypart[s] = X_s^T T_s per token slab s (summed in slab order later, so the result does not
// depend on scheduling), and T = X Q.
#include "agzo_common.cuh"

namespace agzo {

// ------------------------------------------------------------------ Omega -> T
// Local token t is row row0 + t of the test matrix of the whole batch: element e of the stream is
// (row0 + t) * r + k, so the Philox blocks that cover the local rows are walked, whatever row0 is.
__global__ void fill_omega_kernel(const DevLayer* __restrict__ layers, int l0, uint64_t seed, long long row0) {
  chain_wait();
  if (short_launch()) chain_next();
  const DevLayer& L = layers[l0 + blockIdx.y];
  const long long n = (long long)L.m * L.r;
  const long long e0 = row0 * L.r;
  const long long b_end = (e0 + n + 3) >> 2;
  for (long long b = (e0 >> 2) + blockIdx.x * (long long)blockDim.x + threadIdx.x; b < b_end;
       b += (long long)gridDim.x * blockDim.x) {
    const float4 g = gaussian_block((uint64_t)b, L.layer_id, kTagOmega, seed);
    const float gv[4] = {g.x, g.y, g.z, g.w};
#pragma unroll
    for (int lane = 0; lane < 4; ++lane) {
      const long long e = 4 * b + lane - e0;
      if (e >= 0 && e < n) L.T[e] = gv[lane];
    }
  }
}

cudaError_t launch_fill_omega(const ExtractWave& w, uint64_t seed, cudaStream_t s) {
  const long long nb = (((long long)w.max_m * w.max_r + 3) >> 2) + 1;
  int gx = (int)((nb + 255) / 256);
  if (gx > 512) gx = 512;
  if (gx < 1) gx = 1;
  return launch_chained(fill_omega_kernel, dim3(gx, w.l1 - w.l0), 256, 0, 0, s, w.d_layers, w.l0, seed, w.omega_row0);
}

// ------------------------------------------------------------------ four consecutive columns of one row of X
// kind of access a layer's X allows: 16-byte fp32, 8-byte bf16, or element by element
enum XKind : int { X_F32_VEC = 0, X_BF16_VEC = 1, X_SCALAR = 2 };
__device__ __forceinline__ int x_kind(const DevLayer& L) {
  const uintptr_t p = reinterpret_cast<uintptr_t>(L.X);
  if ((L.d_in & 3) != 0 || (L.ldx & 3) != 0) return X_SCALAR;
  if (L.x_dtype == AGZO_F32) return (p & 15u) == 0 ? X_F32_VEC : X_SCALAR;
  return (p & 7u) == 0 ? X_BF16_VEC : X_SCALAR;
}
// zero beyond d_in; `ok` false: zeros
template <int KIND>
__device__ __forceinline__ float4 load_x4(const DevLayer& L, long long t, int d, bool ok) {
  float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
  if (!ok || d >= L.d_in) return v;
  if constexpr (KIND == X_F32_VEC) {
    return __ldg(reinterpret_cast<const float4*>(reinterpret_cast<const float*>(L.X) + t * L.ldx + d));
  } else if constexpr (KIND == X_BF16_VEC) {
    const uint2 u = __ldg(reinterpret_cast<const uint2*>(reinterpret_cast<const __nv_bfloat16*>(L.X) + t * L.ldx + d));
    return make_float4(__uint_as_float(u.x << 16), __uint_as_float(u.x & 0xFFFF0000u), __uint_as_float(u.y << 16),
                       __uint_as_float(u.y & 0xFFFF0000u));
  } else {
    float e[4];
#pragma unroll
    for (int c = 0; c < 4; ++c) {
      const long long at = t * L.ldx + d + c;
      e[c] = d + c >= L.d_in ? 0.f
             : L.x_dtype == AGZO_BF16 ? __bfloat162float(reinterpret_cast<const __nv_bfloat16*>(L.X)[at])
                                      : reinterpret_cast<const float*>(L.X)[at];
    }
    return make_float4(e[0], e[1], e[2], e[3]);
  }
}

constexpr int kXThreads = 256, kXWarps = kXThreads / 32;
constexpr int kXCols = 128;              // columns of one row that a warp reads at a time, four per lane

// ------------------------------------------------------------------ Ypart[s][k][d] = sum_{t in slab s} X[t][d] T[t][k]
// CTA = 128 columns x token slab; a lane keeps 4 columns x RC ranks in registers, the eight warps split the tokens of
// the slab (their sums are added pairwise at the end, in a fixed order), T comes from shared memory as broadcasts.
// Ranks above RC are further passes over the slab, from L2.
// Bound by X (HBM, or L2 where neighbouring layers read the same buffer) for RC <= 8.  The form before this one gave a
// thread one column and all tokens of the slab, one 2- or 4-byte load at a time, and always 16 ranks: 14 fp32 layers of 4000
// tokens (328 MB), r = 8: 289 us per product, now 115; one 512 x 256 layer, r = 4: 60 us, now 3.4.
constexpr int kXtTokens = 128;           // tokens of T staged at a time
template <int RC, int KIND>
__device__ __forceinline__ void xt_t_body(const DevLayer& L, float* sT, float* sRed, int d0, int slab) {
  constexpr int U = 4;                   // tokens in flight per warp
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int d = d0 + 4 * lane, r = L.r;
  const int t_begin = slab * L.slab_rows, t_end = min(L.m, t_begin + L.slab_rows);
  for (int k0 = 0; k0 < r; k0 += RC) {
    const int kc = min(RC, r - k0);
    float acc[RC][4];
#pragma unroll
    for (int k = 0; k < RC; ++k)
#pragma unroll
      for (int c = 0; c < 4; ++c) acc[k][c] = 0.f;
    for (int tb = t_begin; tb < t_end; tb += kXtTokens) {
      float4 x[U];                       // the first rows of the chunk are on their way while T is staged
      const int n = min(kXtTokens, t_end - tb);
#pragma unroll
      for (int u = 0; u < U; ++u) x[u] = load_x4<KIND>(L, tb + warp + u * kXWarps, d, warp + u * kXWarps < n);
      __syncthreads();
      for (int i = threadIdx.x; i < n * RC; i += kXThreads) {
        const int tt = i / RC, k = i - tt * RC;
        sT[i] = k < kc ? L.T[(long long)(tb + tt) * r + k0 + k] : 0.f;
      }
      __syncthreads();
      for (int t0 = warp; t0 < n; t0 += U * kXWarps) {
        float4 nx[U];
#pragma unroll
        for (int u = 0; u < U; ++u) {
          const int t = t0 + (U + u) * kXWarps;
          nx[u] = load_x4<KIND>(L, tb + t, d, t < n);
        }
#pragma unroll
        for (int u = 0; u < U; ++u) {
          const int t = min(t0 + u * kXWarps, n - 1);          // x is zero beyond n
#pragma unroll
          for (int k4 = 0; k4 < RC; k4 += 4) {
            const float4 v = *reinterpret_cast<const float4*>(sT + t * RC + k4);
            const float tv[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
            for (int k = 0; k < 4; ++k) {
              acc[k4 + k][0] = fmaf(x[u].x, tv[k], acc[k4 + k][0]);
              acc[k4 + k][1] = fmaf(x[u].y, tv[k], acc[k4 + k][1]);
              acc[k4 + k][2] = fmaf(x[u].z, tv[k], acc[k4 + k][2]);
              acc[k4 + k][3] = fmaf(x[u].w, tv[k], acc[k4 + k][3]);
            }
          }
          x[u] = nx[u];
        }
      }
    }
    // the warps' sums, halving: 4..7 onto 0..3, 2..3 onto 0..1, 1 onto 0
#pragma unroll
    for (int half = kXWarps / 2; half >= 1; half >>= 1) {
      __syncthreads();
      if (warp >= half && warp < 2 * half) {
#pragma unroll
        for (int k = 0; k < RC; ++k)
          *reinterpret_cast<float4*>(sRed + (((warp - half) * RC + k) * 32 + lane) * 4) =
              make_float4(acc[k][0], acc[k][1], acc[k][2], acc[k][3]);
      }
      __syncthreads();
      if (warp < half) {
#pragma unroll
        for (int k = 0; k < RC; ++k) {
          const float4 v = *reinterpret_cast<const float4*>(sRed + ((warp * RC + k) * 32 + lane) * 4);
          acc[k][0] += v.x; acc[k][1] += v.y; acc[k][2] += v.z; acc[k][3] += v.w;
        }
      }
    }
    if (warp == 0) {
      float* out = L.Ypart + slab * L.ypart_stride + (long long)k0 * L.d_in + d;
#pragma unroll
      for (int k = 0; k < RC; ++k) {
        if (k >= kc) break;
        if (KIND != X_SCALAR) {
          if (d < L.d_in)
            *reinterpret_cast<float4*>(out + (long long)k * L.d_in) = make_float4(acc[k][0], acc[k][1], acc[k][2], acc[k][3]);
        } else {
#pragma unroll
          for (int c = 0; c < 4; ++c)
            if (d + c < L.d_in) out[(long long)k * L.d_in + c] = acc[k][c];
        }
      }
    }
  }
}

template <int RC>
__global__ void __launch_bounds__(kXThreads, 2) xt_t_kernel(const DevLayer* __restrict__ layers, int l0) {
  const DevLayer& L = layers[l0 + blockIdx.z];
  const int slab = blockIdx.y, d0 = blockIdx.x * kXCols;
  chain_wait();
  if (short_launch()) chain_next();
  if (slab >= L.slabs || d0 >= L.d_in) return;
  __shared__ __align__(16) float sT[kXtTokens * RC];
  __shared__ __align__(16) float sRed[kXWarps / 2 * RC * kXCols];
  const int kind = x_kind(L);
  if (kind == X_F32_VEC) xt_t_body<RC, X_F32_VEC>(L, sT, sRed, d0, slab);
  else if (kind == X_BF16_VEC) xt_t_body<RC, X_BF16_VEC>(L, sT, sRed, d0, slab);
  else xt_t_body<RC, X_SCALAR>(L, sT, sRed, d0, slab);
}

cudaError_t launch_xt_t(const ExtractWave& w, cudaStream_t s) {
  const dim3 grid((w.max_din + kXCols - 1) / kXCols, w.max_slabs, w.l1 - w.l0);
  const auto kernel = w.max_r <= 4 ? xt_t_kernel<4> : w.max_r <= 8 ? xt_t_kernel<8> : xt_t_kernel<16>;
  return launch_chained(kernel, grid, kXThreads, 0, 0, s, w.d_layers, w.l0);
}

// ------------------------------------------------------------------ T[t][k] = sum_d X[t][d] Q[k][d]   (Q = rows of V)
// A warp takes four tokens, its lanes four columns each; Q passes through shared memory 512 columns at a time, so that
// a 16-byte read of it serves 16 multiply-adds (as many cycles of the FMA pipes as the read takes of shared memory).
// The lanes' sums are added by halving exchanges (a lane ends up with RC / 8 of them).  Same bound as X^T T; before: one column per lane and load, 16 ranks always, 713 us and 15 us
// on the two examples above, now 95 and 3.1.
constexpr int kXqChunk = 512, kXqTokens = 4;
template <int RC, int KIND>
__device__ __forceinline__ void x_q_body(const DevLayer& L, float* sQ, int t0) {
  constexpr int TOK = kXqTokens;
  const int lane = threadIdx.x & 31, r = L.r, d_in = L.d_in;
  const bool v_vec = (d_in & 3) == 0 && (L.ldv & 3) == 0 && (reinterpret_cast<uintptr_t>(L.V) & 15u) == 0;
  for (int k0 = 0; k0 < r; k0 += RC) {
    const int kc = min(RC, r - k0);
    float acc[TOK * RC];
#pragma unroll
    for (int i = 0; i < TOK * RC; ++i) acc[i] = 0.f;
    for (int c0 = 0; c0 < d_in; c0 += kXqChunk) {
      const int nc = min(kXqChunk, d_in - c0);
      float4 x[TOK];                     // the first columns of the chunk are on their way while Q is staged
#pragma unroll
      for (int t = 0; t < TOK; ++t) x[t] = load_x4<KIND>(L, t0 + t, c0 + 4 * lane, t0 + t < L.m);
      __syncthreads();
      if (v_vec) {
        for (int i = threadIdx.x; i < RC * (kXqChunk / 4); i += kXThreads) {
          const int k = i / (kXqChunk / 4), c = 4 * (i - k * (kXqChunk / 4));
          *reinterpret_cast<float4*>(sQ + k * kXqChunk + c) =
              k < kc && c < nc ? *reinterpret_cast<const float4*>(L.V + (long long)(k0 + k) * L.ldv + c0 + c)
                               : make_float4(0.f, 0.f, 0.f, 0.f);
        }
      } else {
        for (int i = threadIdx.x; i < RC * kXqChunk; i += kXThreads) {
          const int k = i / kXqChunk, c = i - k * kXqChunk;
          sQ[i] = k < kc && c < nc ? L.V[(long long)(k0 + k) * L.ldv + c0 + c] : 0.f;
        }
      }
      __syncthreads();
      for (int c = 4 * lane; c - 4 * lane < nc; c += kXCols) {
        float4 nx[TOK];
        const bool more = c - 4 * lane + kXCols < nc;
#pragma unroll
        for (int t = 0; t < TOK; ++t) nx[t] = load_x4<KIND>(L, t0 + t, c0 + c + kXCols, more && t0 + t < L.m);
#pragma unroll
        for (int k = 0; k < RC; ++k) {
          const float4 q = *reinterpret_cast<const float4*>(sQ + k * kXqChunk + c);
#pragma unroll
          for (int t = 0; t < TOK; ++t)
            acc[t * RC + k] = fmaf(x[t].w, q.w, fmaf(x[t].z, q.z, fmaf(x[t].y, q.y, fmaf(x[t].x, q.x, acc[t * RC + k]))));
        }
#pragma unroll
        for (int t = 0; t < TOK; ++t) x[t] = nx[t];
      }
    }
    int at = 0;                          // first of the sums this lane keeps
    constexpr int N = TOK * RC;
#pragma unroll
    for (int o = 16, n = N / 2; o >= 1; o >>= 1, n >>= 1) {
      const bool up = (lane & o) != 0;
      if (n >= 1) {
#pragma unroll
        for (int i = 0; i < N / 2; ++i)
          if (i < n) {
            const float send = up ? acc[i] : acc[i + n], keep = up ? acc[i + n] : acc[i];
            acc[i] = keep + __shfl_xor_sync(0xffffffffu, send, o);
          }
        at += up ? n : 0;
      } else {
        acc[0] += __shfl_xor_sync(0xffffffffu, acc[0], o);
      }
    }
    constexpr int kKeep = N >= 32 ? N / 32 : 1;
    if (N >= 32 || (lane & (32 / (N < 32 ? N : 32) - 1)) == 0) {
#pragma unroll
      for (int i = 0; i < kKeep; ++i) {
        const int t = t0 + (at + i) / RC, k = (at + i) % RC;
        if (t < L.m && k < kc) L.T[(long long)t * r + k0 + k] = acc[i];
      }
    }
  }
}

template <int RC>
__global__ void __launch_bounds__(kXThreads, 2) x_q_kernel(const DevLayer* __restrict__ layers, int l0) {
  const DevLayer& L = layers[l0 + blockIdx.y];
  chain_wait();
  if (short_launch()) chain_next();
  if ((int)blockIdx.x * kXWarps * kXqTokens >= L.m) return;
  __shared__ __align__(16) float sQ[RC * kXqChunk];
  const int t0 = ((int)blockIdx.x * kXWarps + (threadIdx.x >> 5)) * kXqTokens;
  const int kind = x_kind(L);
  if (kind == X_F32_VEC) x_q_body<RC, X_F32_VEC>(L, sQ, t0);
  else if (kind == X_BF16_VEC) x_q_body<RC, X_BF16_VEC>(L, sQ, t0);
  else x_q_body<RC, X_SCALAR>(L, sQ, t0);
}

cudaError_t launch_x_q(const ExtractWave& w, cudaStream_t s) {
  const dim3 grid((w.max_m + kXWarps * kXqTokens - 1) / (kXWarps * kXqTokens), w.l1 - w.l0);
  const auto kernel = w.max_r <= 4 ? x_q_kernel<4> : w.max_r <= 8 ? x_q_kernel<8> : x_q_kernel<16>;
  return launch_chained(kernel, grid, kXThreads, 0, 0, s, w.d_layers, w.l0);
}

// Y[k][d] = sum_s Ypart[s][k][d] in slab order, on its own: token-sharded extraction sums Y over
// the ranks before the panel QR reads it
__global__ void __launch_bounds__(256) sum_slabs_kernel(const DevLayer* __restrict__ layers, int l0, int after_fused) {
  const DevLayer& L = layers[l0 + blockIdx.y];
  chain_wait();
  if (short_launch()) chain_next();
  const int nparts = y_parts(L, after_fused);
  const long long n = (long long)L.r * L.d_in;
  for (long long i = blockIdx.x * 256ll + threadIdx.x; i < n; i += (long long)gridDim.x * 256) {
    float y = 0.f;
    for (int s = 0; s < nparts; ++s) y += L.Ypart[s * L.ypart_stride + i];
    L.Y[i] = y;
  }
}

cudaError_t launch_sum_slabs(const ExtractWave& w, cudaStream_t s) {
  long long blocks = ((long long)w.max_r * w.max_din + 255) / 256;
  if (blocks > 256) blocks = 256;
  return launch_chained(sum_slabs_kernel, dim3((unsigned)blocks, w.l1 - w.l0), 256, 0, 0, s, w.d_layers, w.l0, w.after_fused);
}

}  // namespace agzo

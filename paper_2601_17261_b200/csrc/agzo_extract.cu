// The two products of Algorithm 1 (SubspaceExtract) with X on CUDA cores in fp32, for any dtype,
// pitch and size; the tensor-core path (agzo_extract_tc.cu) replaces them when the layer's shape
// allows it, and the products in fp32 precision (agzo_extract_split.cu) where those are estimated the faster ones.  qr(Y) is in agzo_panel_qr.cu.
//
// Ypart[s] = X_s^T T_s per token slab s (summed in slab order later, so the result does not
// depend on scheduling), and T = X Q.
#include "agzo_common.cuh"

namespace agzo {

// ------------------------------------------------------------------ Omega -> T
// Local token t is row row0 + t of the test matrix of the whole batch: element e of the stream is
// (row0 + t) * r + k, so the Philox blocks that cover the local rows are walked, whatever row0 is.
__global__ void fill_omega_kernel(const DevLayer* layers, int l0, uint64_t seed, long long row0, DevStatus* status, int region) {
  chain_wait();
  if (short_launch()) chain_next();
  if (blockIdx.x + blockIdx.y == 0 && threadIdx.x == 0) wave_begins(status, region);
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

cudaError_t launch_fill_omega(const ExtractWave& w, uint64_t seed, DevStatus* d_status, cudaStream_t s) {
  const long long nb = (((long long)w.max_m * w.max_r + 3) >> 2) + 1;
  int gx = (int)((nb + 255) / 256);
  if (gx > 512) gx = 512;
  if (gx < 1) gx = 1;
  return launch_chained(fill_omega_kernel, dim3(gx, w.l1 - w.l0), 256, 0, 0, s, w.d_layers, w.l0, seed, w.omega_row0, d_status, w.region);
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
// Row t (below m), columns d .. d + 3.  The vector kinds read four columns inside the row whatever d is: for uses where what
// they are multiplied with is zero there, or the product is not stored.  The scalar kind returns zeros beyond d_in.
template <int KIND>
__device__ __forceinline__ float4 load_x4_at(const DevLayer& L, int t, int d) {
  float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
  if constexpr (KIND != X_SCALAR) d = min(d, L.d_in - 4);
  const long long at = (long long)t * L.ldx + d;
  if constexpr (KIND == X_F32_VEC) {
    const float* p = reinterpret_cast<const float*>(L.X) + at;
    asm("ld.global.nc.L1::no_allocate.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "l"(p));
  } else if constexpr (KIND == X_BF16_VEC) {
    const __nv_bfloat16* p = reinterpret_cast<const __nv_bfloat16*>(L.X) + at;
    uint2 u;
    asm("ld.global.nc.L1::no_allocate.v2.u32 {%0, %1}, [%2];" : "=r"(u.x), "=r"(u.y) : "l"(p));
    v = make_float4(__uint_as_float(u.x << 16), __uint_as_float(u.x & 0xFFFF0000u), __uint_as_float(u.y << 16),
                    __uint_as_float(u.y & 0xFFFF0000u));
  } else {
    float e[4];
#pragma unroll
    for (int c = 0; c < 4; ++c)
      e[c] = d + c >= L.d_in ? 0.f
             : L.x_dtype == AGZO_BF16 ? __bfloat162float(reinterpret_cast<const __nv_bfloat16*>(L.X)[at + c])
                                      : reinterpret_cast<const float*>(L.X)[at + c];
    v = make_float4(e[0], e[1], e[2], e[3]);
  }
  return v;
}
// zeros beyond d_in, and where `ok` is false
template <int KIND>
__device__ __forceinline__ float4 load_x4(const DevLayer& L, int t, int d, bool ok) {
  return ok && d < L.d_in ? load_x4_at<KIND>(L, t, d) : make_float4(0.f, 0.f, 0.f, 0.f);
}

constexpr int kXThreads = 256, kXWarps = kXThreads / 32;
constexpr int kXCols = 128;              // columns of one row that a warp reads at a time, four per lane

// ------------------------------------------------------------------ Ypart[s][k][d] = sum_{t in slab s} X[t][d] T[t][k]
// CTA = 128 columns x token slab; a lane keeps 4 columns x RC ranks in registers, the eight warps split the tokens of
// the slab (their sums are added pairwise at the end, in a fixed order), T comes from shared memory as broadcasts.
// Ranks above RC are further passes over the slab, from L2.
// Bound by X (HBM, or L2 where neighbouring layers read the same buffer) for RC <= 8.  The form before this one gave a
// thread one column and all tokens of the slab, one 2- or 4-byte load at a time, and always 16 ranks: 14 fp32 layers of 4000
// tokens (328 MB), r = 8: 289 us per product, now 71; one 512 x 256 layer, r = 4: 60 us, now 3.4.
constexpr int kXtTokens = 128;           // tokens of T staged at a time
template <int RC, int KIND>
__device__ __forceinline__ void xt_t_body(const DevLayer& L, float* sT, float* sRed, int d0, int slab) {
  constexpr int U = RC <= 8 ? 8 : 4;     // tokens in flight per warp
  // Above rank 8 the pass is bound by its multiply-adds: two columns per instruction, T side by side twice as their operand
  // (4096 x 2048, r = 16: 38 -> 29 us per product; at r = 8 the wider operand reads cost more than they save: 71 -> 78 us)
  constexpr bool kPacked = RC > 8;
  constexpr int kDup = kPacked ? 2 : 1;
  constexpr int kStage = kXtTokens * RC / kXThreads;     // values of T per thread and chunk
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int d = d0 + 4 * lane, r = L.r;
  const int rows = cc_rows(L.m, L.cc_slabs), t_begin = slab * rows, t_end = min(L.m, t_begin + rows);
  for (int k0 = 0; k0 < r; k0 += RC) {
    const int kc = min(RC, r - k0);
    float acc[RC][4];
    uint64_t acc2[kPacked ? RC : 1][2];
#pragma unroll
    for (int k = 0; k < RC; ++k) {
#pragma unroll
      for (int c = 0; c < 4; ++c) acc[k][c] = 0.f;
      if (kPacked) acc2[k][0] = acc2[k][1] = 0;
    }
    // Both streams run ahead: a chunk's T is fetched into registers while the chunk before it is worked on, and the next U
    // rows of X while the current ones are used, across chunks too; T is zero beyond the slab, where X is read at its last row.
    float tv[kStage];
    auto fetch_t = [&](int tb) {
#pragma unroll
      for (int j = 0; j < kStage; ++j) {
        const int i = threadIdx.x + j * kXThreads, tt = i / RC, k = i - tt * RC;
        tv[j] = tb + tt < t_end && k < kc ? L.T[(long long)(tb + tt) * r + k0 + k] : 0.f;
      }
    };
    float4 x[U];
    if (k0 > 0) fetch_t(t_begin);
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int t = t_begin + warp + u * kXWarps;
      x[u] = load_x4_at<KIND>(L, min(t, t_end - 1), d);
    }
    if (k0 == 0) {                       // the first rows of X are on their way: now for the predecessor's T (one 256 x 256
                                         // fp32 layer of 512 tokens: a step 59.9 -> 54.0 us; with x_q's)
      chain_wait();
      if (short_launch()) chain_next();
      fetch_t(t_begin);
    }
    for (int tb = t_begin; tb < t_end; tb += kXtTokens) {
      __syncthreads();
#pragma unroll
      for (int j = 0; j < kStage; ++j) {
        const int i = threadIdx.x + j * kXThreads;
        if (kPacked) *reinterpret_cast<float2*>(sT + 2 * i) = make_float2(tv[j], tv[j]);
        else sT[i] = tv[j];
      }
      __syncthreads();
      if (tb + kXtTokens < t_end) fetch_t(tb + kXtTokens);
      const int rounds = (min(kXtTokens, t_end - tb) + kXWarps - 1) / kXWarps;
#pragma unroll 1
      for (int i0 = 0; i0 < rounds; i0 += U) {        // rows warp + 8 (i0 + u) of the chunk
        const float* st = sT + kDup * (warp + i0 * kXWarps) * RC;
#pragma unroll
        for (int u = 0; u < U; ++u) {
          const float4 xu = x[u];
          const int next = tb + warp + (i0 + U + u) * kXWarps;     // zero beyond the slab
          x[u] = load_x4_at<KIND>(L, min(next, t_end - 1), d);
          if constexpr (kPacked) {
            const uint64_t xa = pack_f32x2(xu.x, xu.y), xb = pack_f32x2(xu.z, xu.w);
#pragma unroll
            for (int k = 0; k < RC; k += 2) {
              const ulonglong2 v = *reinterpret_cast<const ulonglong2*>(st + 2 * (u * kXWarps * RC + k));
              acc2[k][0] = fma_f32x2(xa, v.x, acc2[k][0]);
              acc2[k][1] = fma_f32x2(xb, v.x, acc2[k][1]);
              acc2[k + 1][0] = fma_f32x2(xa, v.y, acc2[k + 1][0]);
              acc2[k + 1][1] = fma_f32x2(xb, v.y, acc2[k + 1][1]);
            }
          } else
#pragma unroll
          for (int k4 = 0; k4 < RC; k4 += 4) {
            const float4 v = *reinterpret_cast<const float4*>(st + u * kXWarps * RC + k4);
            const float tk[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
            for (int k = 0; k < 4; ++k) {
              acc[k4 + k][0] = fmaf(xu.x, tk[k], acc[k4 + k][0]);
              acc[k4 + k][1] = fmaf(xu.y, tk[k], acc[k4 + k][1]);
              acc[k4 + k][2] = fmaf(xu.z, tk[k], acc[k4 + k][2]);
              acc[k4 + k][3] = fmaf(xu.w, tk[k], acc[k4 + k][3]);
            }
          }
        }
      }
    }
    if (kPacked) {
#pragma unroll
      for (int k = 0; k < RC; ++k) {
        unpack_f32x2(acc2[k][0], acc[k][0], acc[k][1]);
        unpack_f32x2(acc2[k][1], acc[k][2], acc[k][3]);
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
  if (slab >= L.cc_slabs || d0 >= L.d_in) return;
  __shared__ __align__(16) float sT[kXtTokens * RC * (RC > 8 ? 2 : 1)];
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
// A warp takes four tokens, its lanes four columns each, so that a 16-byte read of Q serves 16 multiply-adds.  Q is read
// through L1, which X passes by (no_allocate), so it is fetched about once per SM, and the warps run without barriers.  The
// lanes' sums are added by halving exchanges (a lane ends up with RC / 8 of them).  Same bound as X^T T; with one column per
// lane and load, and always 16 ranks: 713 us and 15 us on the two examples above, now 94 and 3.
constexpr int kXqTokens = 4;
template <bool VVEC>
__device__ __forceinline__ float4 load_q4(const float* p, int left) {
  if constexpr (VVEC) {
    return left > 0 ? *reinterpret_cast<const float4*>(p) : make_float4(0.f, 0.f, 0.f, 0.f);
  } else {
    float4 q = make_float4(0.f, 0.f, 0.f, 0.f);
    if (left > 0) q.x = p[0];
    if (left > 1) q.y = p[1];
    if (left > 2) q.z = p[2];
    if (left > 3) q.w = p[3];
    return q;
  }
}

// SPLIT = 2: two neighbouring warps take half of the columns each and the sums meet in sPart (launches of so few tokens
// that the SMs would have fewer than eight warps)
template <int RC, int SPLIT, int KIND, bool VVEC>
__device__ __forceinline__ void x_q_body(const DevLayer& L, int t0, float* sPart) {
  constexpr int TOK = kXqTokens;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, r = L.r;
  const int half = SPLIT == 2 ? warp & 1 : 0;
  const int blocks = (L.d_in + kXCols - 1) / kXCols;
  const int c_begin = half * ((blocks + 1) / 2) * kXCols;
  const int d_end = SPLIT == 2 && half == 0 ? min(L.d_in, (blocks + 1) / 2 * kXCols) : L.d_in;
  for (int k0 = 0; k0 < r; k0 += RC) {
    const int kc = min(RC, r - k0);
    const float* V = L.V + (long long)k0 * L.ldv;
    float acc[TOK * RC];
#pragma unroll
    for (int i = 0; i < TOK * RC; ++i) acc[i] = 0.f;
    float4 x[TOK];
#pragma unroll
    for (int t = 0; t < TOK; ++t) x[t] = load_x4<KIND>(L, t0 + t, c_begin + 4 * lane, t0 + t < L.m);
    if (k0 == 0) {                       // the first columns of X are on their way: now for the predecessor's Q
      chain_wait();
      if (short_launch()) chain_next();
    }
    for (int c = c_begin + 4 * lane; c - 4 * lane < d_end; c += kXCols) {
      float4 nx[TOK];
#pragma unroll
      for (int t = 0; t < TOK; ++t) nx[t] = load_x4<KIND>(L, t0 + t, c + kXCols, t0 + t < L.m);
#pragma unroll
      for (int k = 0; k < RC; ++k) {
        const float4 q = load_q4<VVEC>(V + (long long)min(k, kc - 1) * L.ldv + c, L.d_in - c);   // ranks beyond kc are not stored
#pragma unroll
        for (int t = 0; t < TOK; ++t)
          acc[t * RC + k] = fmaf(x[t].w, q.w, fmaf(x[t].z, q.z, fmaf(x[t].y, q.y, fmaf(x[t].x, q.x, acc[t * RC + k]))));
      }
#pragma unroll
      for (int t = 0; t < TOK; ++t) x[t] = nx[t];
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
    if constexpr (SPLIT == 2) {
      __syncthreads();                   // the previous ranks' sums have been used
      if (half == 1) {
#pragma unroll
        for (int i = 0; i < kKeep; ++i) sPart[(warp >> 1) * 32 * kKeep + i * 32 + lane] = acc[i];
      }
      __syncthreads();
      if (half == 1) continue;
#pragma unroll
      for (int i = 0; i < kKeep; ++i) acc[i] += sPart[(warp >> 1) * 32 * kKeep + i * 32 + lane];
    }
    if (N >= 32 || (lane & (32 / (N < 32 ? N : 32) - 1)) == 0) {
#pragma unroll
      for (int i = 0; i < kKeep; ++i) {
        const int t = t0 + (at + i) / RC, k = (at + i) % RC;
        if (t < L.m && k < kc) L.T[(long long)t * r + k0 + k] = acc[i];
      }
    }
  }
}

template <int RC, int SPLIT>
__global__ void __launch_bounds__(kXThreads, 2) x_q_kernel(const DevLayer* __restrict__ layers, int l0) {
  const DevLayer& L = layers[l0 + blockIdx.y];
  constexpr int kGroups = kXWarps / SPLIT;               // token groups per CTA
  if ((int)blockIdx.x * kGroups * kXqTokens >= L.m) return;
  __shared__ float sPart[SPLIT == 2 ? kGroups * 32 * (RC / 8 > 1 ? RC / 8 : 1) : 1];
  const int t0 = ((int)blockIdx.x * kGroups + (int)(threadIdx.x >> 5) / SPLIT) * kXqTokens;
  const bool v_vec = (L.d_in & 3) == 0 && (L.ldv & 3) == 0 && (reinterpret_cast<uintptr_t>(L.V) & 15u) == 0;
  const int kind = v_vec ? x_kind(L) : X_SCALAR;
  if (kind == X_F32_VEC) x_q_body<RC, SPLIT, X_F32_VEC, true>(L, t0, sPart);
  else if (kind == X_BF16_VEC) x_q_body<RC, SPLIT, X_BF16_VEC, true>(L, t0, sPart);
  else x_q_body<RC, SPLIT, X_SCALAR, false>(L, t0, sPart);
}

template <int SPLIT>
cudaError_t launch_x_q_split(const ExtractWave& w, cudaStream_t s) {
  const int per = kXWarps / SPLIT * kXqTokens;
  const dim3 grid((w.max_m + per - 1) / per, w.l1 - w.l0);
  const auto kernel = w.max_r <= 4 ? x_q_kernel<4, SPLIT> : w.max_r <= 8 ? x_q_kernel<8, SPLIT> : x_q_kernel<16, SPLIT>;
  return launch_chained(kernel, grid, kXThreads, 0, 0, s, w.d_layers, w.l0);
}
cudaError_t launch_x_q(const ExtractWave& w, cudaStream_t s) {
  const bool few = (long long)w.max_m * (w.l1 - w.l0) <= (long long)w.sm_count * kXWarps * kXqTokens;
  return few ? launch_x_q_split<2>(w, s) : launch_x_q_split<1>(w, s);
}

// Y[k][d] = sum_s Ypart[s][k][d] in slab order, on its own: token-sharded extraction sums Y over
// the ranks before the panel QR reads it
__global__ void __launch_bounds__(256) sum_slabs_kernel(const DevLayer* __restrict__ layers, int l0, int after_fused) {
  const DevLayer& L = layers[l0 + blockIdx.y];
  chain_wait();                          // releases nobody: the caller's all-reduce follows
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

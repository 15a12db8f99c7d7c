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
  fill_omega_kernel<<<dim3(gx, w.l1 - w.l0), 256, 0, s>>>(w.d_layers, w.l0, seed, w.omega_row0);
  return cudaGetLastError();
}

__device__ __forceinline__ float load_x(const DevLayer& L, long long t, int d) {
  return L.x_dtype == AGZO_BF16
             ? __bfloat162float(reinterpret_cast<const __nv_bfloat16*>(L.X)[t * L.ldx + d])
             : reinterpret_cast<const float*>(L.X)[t * L.ldx + d];
}

// ------------------------------------------------------------------ Ypart[s][k][d] = sum_{t in slab s} X[t][d] T[t][k]
// block: 256 threads = 256 columns d; grid (d chunks, slabs, layers).  Rank handled in chunks of 16.
constexpr int kXtTokens = 32;
__global__ void __launch_bounds__(256) xt_t_kernel(const DevLayer* __restrict__ layers, int l0) {
  const DevLayer& L = layers[l0 + blockIdx.z];
  const int slab = blockIdx.y;
  if (slab >= L.slabs) return;
  const int d0 = blockIdx.x * 256;
  if (d0 >= L.d_in) return;
  const int d = d0 + threadIdx.x;
  const bool d_ok = d < L.d_in;
  const int t_begin = slab * L.slab_rows;
  const int t_end = min(L.m, t_begin + L.slab_rows);
  __shared__ float sT[kXtTokens][16];
  const int r = L.r;
  for (int k0 = 0; k0 < r; k0 += 16) {
    const int kc = min(16, r - k0);
    float acc[16];
#pragma unroll
    for (int k = 0; k < 16; ++k) acc[k] = 0.f;
    for (int tb = t_begin; tb < t_end; tb += kXtTokens) {
      __syncthreads();
      for (int i = threadIdx.x; i < kXtTokens * 16; i += 256) {
        const int tt = i >> 4, k = i & 15;
        sT[tt][k] = (tb + tt < t_end && k < kc) ? L.T[(long long)(tb + tt) * r + k0 + k] : 0.f;
      }
      __syncthreads();
      if (d_ok) {
        const int nt = min(kXtTokens, t_end - tb);
        for (int tt = 0; tt < nt; ++tt) {
          const float x = load_x(L, tb + tt, d);
#pragma unroll
          for (int k = 0; k < 16; ++k) acc[k] = fmaf(x, sT[tt][k], acc[k]);
        }
      }
    }
    if (d_ok) {
      float* out = L.Ypart + ((long long)slab * r + k0) * L.d_in + d;
      for (int k = 0; k < kc; ++k) out[(long long)k * L.d_in] = acc[k];
    }
  }
}

cudaError_t launch_xt_t(const ExtractWave& w, cudaStream_t s) {
  dim3 grid((w.max_din + 255) / 256, w.max_slabs, w.l1 - w.l0);
  xt_t_kernel<<<grid, 256, 0, s>>>(w.d_layers, w.l0);
  return cudaGetLastError();
}

// ------------------------------------------------------------------ T[t][k] = sum_d X[t][d] Q[k][d]   (Q = rows of V)
// one warp per token; Q streamed through shared memory in column chunks.
constexpr int kXqCols = 256;
constexpr int kXqWarps = 8;
__global__ void __launch_bounds__(256) x_q_kernel(const DevLayer* __restrict__ layers, int l0) {
  const DevLayer& L = layers[l0 + blockIdx.y];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int tokens_per_block = kXqWarps * 4;
  const int t0 = blockIdx.x * tokens_per_block;
  if (t0 >= L.m) return;
  __shared__ float sQ[16][kXqCols + 1];
  const int r = L.r;
  for (int k0 = 0; k0 < r; k0 += 16) {
    const int kc = min(16, r - k0);
    float acc[4][16];
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
      for (int k = 0; k < 16; ++k) acc[i][k] = 0.f;
    for (int c0 = 0; c0 < L.d_in; c0 += kXqCols) {
      __syncthreads();
      for (int i = threadIdx.x; i < 16 * kXqCols; i += 256) {
        const int k = i / kXqCols, c = i - k * kXqCols;
        sQ[k][c] = (k < kc && c0 + c < L.d_in) ? L.V[(long long)(k0 + k) * L.ldv + c0 + c] : 0.f;
      }
      __syncthreads();
      const int nc = min(kXqCols, L.d_in - c0);
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const int t = t0 + warp * 4 + i;
        if (t < L.m) {
          for (int c = lane; c < nc; c += 32) {
            const float x = load_x(L, t, c0 + c);
#pragma unroll
            for (int k = 0; k < 16; ++k) acc[i][k] = fmaf(x, sQ[k][c], acc[i][k]);
          }
        }
      }
    }
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const int t = t0 + warp * 4 + i;
#pragma unroll
      for (int k = 0; k < 16; ++k) {
        float v = acc[i][k];
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
        if (lane == 0 && t < L.m && k < kc) L.T[(long long)t * r + k0 + k] = v;
      }
    }
  }
}

cudaError_t launch_x_q(const ExtractWave& w, cudaStream_t s) {
  dim3 grid((w.max_m + kXqWarps * 4 - 1) / (kXqWarps * 4), w.l1 - w.l0);
  x_q_kernel<<<grid, 256, 0, s>>>(w.d_layers, w.l0);
  return cudaGetLastError();
}

// Y[k][d] = sum_s Ypart[s][k][d] in slab order, on its own: token-sharded extraction sums Y over
// the ranks before the panel QR reads it
__global__ void __launch_bounds__(256) sum_slabs_kernel(const DevLayer* __restrict__ layers, int l0, int after_fused) {
  const DevLayer& L = layers[l0 + blockIdx.y];
  const int nparts = y_parts(L, after_fused);
  const long long n = (long long)L.r * L.d_in;
  for (long long i = blockIdx.x * 256ll + threadIdx.x; i < n; i += (long long)gridDim.x * 256) {
    float y = 0.f;
    for (int s = 0; s < nparts; ++s) y += L.Ypart[(long long)s * n + i];
    L.Y[i] = y;
  }
}

cudaError_t launch_sum_slabs(const ExtractWave& w, cudaStream_t s) {
  long long blocks = ((long long)w.max_r * w.max_din + 255) / 256;
  if (blocks > 256) blocks = 256;
  sum_slabs_kernel<<<dim3((unsigned)blocks, w.l1 - w.l0), 256, 0, s>>>(w.d_layers, w.l0, w.after_fused);
  return cudaGetLastError();
}

}  // namespace agzo

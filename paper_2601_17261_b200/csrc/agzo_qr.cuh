// Pieces of the panel QR (Gram products, Cholesky and inverse, apply, all in double on the FP64 tensor cores) that the panel-QR
// kernels and the resident extraction share.
#pragma once

#include "agzo_common.cuh"
#include "agzo_ptx.cuh"

namespace agzo {
namespace qr {

using namespace ptx;

constexpr int kQrThreads = 256;
constexpr int kQrWarps = kQrThreads / 32;
constexpr int kQrChunk = 128;            // columns of Y that are staged together
constexpr int kQrMaxCluster = 16;         // beyond the portable 8: asked for, and used only where the device grants it
constexpr int kBlk = 8;                  // block of the factorisation = tile of the FP64 tensor cores
// up to here the slice stays in shared memory from load to apply, with two CTAs per SM
constexpr size_t kQrResidentSmem = 112 * 1024;

__device__ __forceinline__ void dmma_m8n8k4(double& c0, double& c1, double a, double b) {
  asm volatile("mma.sync.aligned.m8n8k4.row.col.f64.f64.f64.f64 {%0, %1}, {%2}, {%3}, {%0, %1};"
               : "+d"(c0), "+d"(c1) : "d"(a), "d"(b));
}
__device__ __forceinline__ double ld_cluster_f64(uint32_t addr) {
  double v;
  asm volatile("ld.shared::cluster.f64 %0, [%1];" : "=d"(v) : "r"(addr) : "memory");
  return v;
}

// Sizes of an instantiation.  NT: 8-row tiles of the panel (the wave's largest rank, rounded up).
template <int NT>
struct QrCfg {
  static constexpr int r8 = 8 * NT;
  static constexpr int tiles = NT * (NT + 1) / 2;          // 8 x 8 tiles of the upper triangle of S
  static constexpr int my_tiles = NT <= 4 ? tiles : 10;    // ... of them per warp, at most
  static constexpr int ksplit = NT <= 4 ? kQrWarps : 2;    // warps that split the columns (eight tile rows: four sets of tiles)
  static constexpr int ap = r8 + 1;                        // pitch of S / R in doubles
  static constexpr int mp = (r8 + 15) / 16 * 16 + 4;       // pitch of M in doubles
  static constexpr size_t g_bytes = (size_t)tiles * 64 * 8;
  static constexpr size_t am_bytes = (size_t)r8 * (ap + mp) * 8;
  static constexpr size_t p_bytes = NT <= 4 ? (size_t)kQrWarps * tiles * 64 * 8 : 0;
  static constexpr size_t u_bytes = am_bytes > p_bytes ? am_bytes : p_bytes;   // warps' partial sums, then S/R and M
  static constexpr size_t fixed = g_bytes + u_bytes;
};
// pitch of the staged columns in floats: 12 beyond a multiple of 32, so that the 8 x 4 elements of a Gram fragment
// fall into 32 banks and an apply fragment's into 28
__host__ __device__ inline int qr_pitch(int cols) { return cols + 12; }

// Which tiles of the upper triangle a warp of set H works on.  Eight tile rows are split into four sets that touch few
// different tile rows each (a fragment is converted to double once per set): the two triangles of ten tiles and the
// two halves, eight tiles each, of the square between them.
template <int NT, int H>
__device__ constexpr bool qr_tile_mine(int bi, int bj) {
  return NT <= 4 ? true
                 : (H == 0 ? bj < 4 : H == 3 ? bi >= 4 : (bi < 4 && bj >= 4 && (bi < 2) == (H == 1)));
}
template <int NT, int H>
__device__ constexpr bool qr_row_used(int b) {
  return NT <= 4 ? true : (H == 0 ? b < 4 : H == 3 ? b >= 4 : (b >= 4 || (b < 2) == (H == 1)));
}

// Gram products of `steps` groups of four columns, this warp taking every ksplit-th group.  Fragments (PTX ISA, m8n8k4
// .f64): lane l holds A[l / 4][l % 4], B[l % 4][l / 4] and D[l / 4][2 (l % 4) + {0, 1}]; with A = Y[8 bi ..][c ..] and
// B = Y[8 bj ..][c ..]^T both operands are the element (l / 4, l % 4) of a row block of the staged columns.
template <int NT, int H>
__device__ __forceinline__ void qr_gram(const float* sY, int pitch, int steps, int k0, double (&acc)[QrCfg<NT>::my_tiles][2]) {
  const int lane = threadIdx.x & 31, fr = lane >> 2, fc = lane & 3;
  const float* base = sY + fr * pitch + fc;
#pragma unroll 2
  for (int ks = k0; ks < steps; ks += QrCfg<NT>::ksplit) {
    double f[NT];
#pragma unroll
    for (int b = 0; b < NT; ++b)
      if (qr_row_used<NT, H>(b)) f[b] = (double)base[8 * b * pitch + 4 * ks];
    int t = 0;
#pragma unroll
    for (int bi = 0; bi < NT; ++bi)
#pragma unroll
      for (int bj = bi; bj < NT; ++bj)
        if (qr_tile_mine<NT, H>(bi, bj)) { dmma_m8n8k4(acc[t][0], acc[t][1], f[bi], f[bj]); ++t; }
  }
}

// adds this warp's sums to a Gram share (this lane's two elements of every tile of the warp)
template <int NT, int H>
__device__ __forceinline__ void qr_add_share(double* g, const double (&acc)[QrCfg<NT>::my_tiles][2], bool first) {
  int t = 0, n = 0;
#pragma unroll
  for (int bi = 0; bi < NT; ++bi)
#pragma unroll
    for (int bj = bi; bj < NT; ++bj, ++t)
      if (qr_tile_mine<NT, H>(bi, bj)) {
        double2* p = reinterpret_cast<double2*>(g + t * 64);
        double2 v = first ? make_double2(0.0, 0.0) : *p;
        v.x += acc[n][0]; v.y += acc[n][1];
        *p = v;
        ++n;
      }
}

// Stages columns [d0, d0 + ncols) of Y (ncols a multiple of 128; zero beyond d_in and beyond row r) into sY.
// from_y: read L.Y as it is; else the sum of the partial sums, which is also written to L.Y when `keep` is set.
__device__ __forceinline__ void qr_load(const DevLayer& L, float* sY, int pitch, int r8, int d0, int ncols, int nparts,
                                        bool from_y, bool keep) {
  const int r = L.r, d_in = L.d_in;
  const long long part = L.ypart_stride;
  const float* src0 = from_y ? L.Y : L.Ypart;
  const int np = from_y ? 1 : nparts;
  if ((d_in & 3) == 0) {
    const int vrow = ncols >> 2, nvec = r8 * vrow;
    constexpr int U = 4, P = 4;                      // 16 independent loads before the first use
    for (int i0 = threadIdx.x; i0 < nvec; i0 += U * kQrThreads) {
      float4 v[U];
      const float* src[U];
      bool live[U];
      int at[U], col[U], row[U];
#pragma unroll
      for (int u = 0; u < U; ++u) {
        const int i = i0 + u * kQrThreads;
        row[u] = i / vrow;
        col[u] = d0 + 4 * (i - row[u] * vrow);
        at[u] = row[u] * pitch + (col[u] - d0);
        live[u] = i < nvec && row[u] < r && col[u] < d_in;
        src[u] = src0 + (long long)row[u] * d_in + col[u];
        v[u] = make_float4(0.f, 0.f, 0.f, 0.f);
      }
      for (int s0 = 0; s0 < np; s0 += P) {
        float4 t[U][P];
#pragma unroll
        for (int u = 0; u < U; ++u)
#pragma unroll
          for (int s = 0; s < P; ++s)
            t[u][s] = live[u] && s0 + s < np ? __ldcg(reinterpret_cast<const float4*>(src[u] + (s0 + s) * part))
                                             : make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
        for (int u = 0; u < U; ++u)
#pragma unroll
          for (int s = 0; s < P; ++s) { v[u].x += t[u][s].x; v[u].y += t[u][s].y; v[u].z += t[u][s].z; v[u].w += t[u][s].w; }
      }
#pragma unroll
      for (int u = 0; u < U; ++u) {
        if (i0 + u * kQrThreads >= nvec) continue;
        *reinterpret_cast<float4*>(sY + at[u]) = v[u];
        if (keep && live[u]) *reinterpret_cast<float4*>(L.Y + (long long)row[u] * d_in + col[u]) = v[u];
      }
    }
  } else {
    for (int i = threadIdx.x; i < r8 * ncols; i += kQrThreads) {
      const int k = i / ncols, c = i - k * ncols, d = d0 + c;
      float y = 0.f;
      if (k < r && d < d_in) {
        for (int s = 0; s < np; ++s) y += __ldcg(src0 + s * part + (long long)k * d_in + d);
        if (keep) L.Y[(long long)k * d_in + d] = y;
      }
      sY[k * pitch + c] = y;
    }
  }
}

// Diagonal block kb (8 x 8) of the factorisation by one warp, every lane on the whole block in registers: the chain is
// then four times (rsqrt, multiply, multiply-add) with no exchange between lanes.  D = R_kk^-1 goes to the block of M
// (zero below the diagonal): lane j takes row j, which goes through the elimination with the block instead of a back
// substitution after it.  kLive: the columns that can be live, four where no rank of the launch is larger (one 256 x 256 layer, r = 4: step 52 -> 49 us; as a
// branch between the pivots it cost r = 8 1 % of a step of small layers).
// A pivot with R_kk <= kRankTol * ||y_k|| (what is left of column k after the columns before it are projected out,
// against the column's own length) marks a dependent column, which becomes zero.  The test is scale-free per column: the
// columns of Y = H (H^T Q) carry squared singular values, so a short column is normal and says nothing about dependence.
template <int NT, int kLive = kBlk>
__device__ __forceinline__ void qr_factor_block(const double* A, double* M, const double* own, int kb, int r, DevStatus* status,
                                                bool report) {
  constexpr int ap = QrCfg<NT>::ap, mp = QrCfg<NT>::mp;
  const int lane = threadIdx.x & 31, j = lane & 7;
  const int o = kb * kBlk;
  double a[kLive][kLive];                     // the upper triangle is used
  double b[kLive];                           // e_j under the same elimination: column j of R^-T, which is row j of D
#pragma unroll
  for (int i = 0; i < kLive; ++i)
#pragma unroll
    for (int c = i; c < kLive; ++c) a[i][c] = A[(o + i) * ap + o + c];
#pragma unroll
  for (int i = 0; i < kLive; ++i) b[i] = i == j ? 1.0 : 0.0;
  bool any_bad = false;
  // two pivots at a time: with d1 = a_kk and det = d1 a_22 - a_12^2 both reciprocal roots start together
  // (1 / R_22 = sqrt(d1) / sqrt(det)); what a subtraction loses in det it loses in a_22 - R_12^2 as well
#pragma unroll
  for (int k = 0; k < kLive; k += 2) {
    const double d1 = a[k][k], a12 = a[k][k + 1], a22 = a[k + 1][k + 1];
    const double det = fma(d1, a22, -(a12 * a12));
    const double r1 = rsqrt(d1), rd = rsqrt(det);
    const bool live1 = o + k < r, live2 = o + k + 1 < r;
    const bool bad1 = !(d1 > 0.0) || d1 <= kRankTol * kRankTol * own[o + k];
    const double i1 = (live1 && !bad1) ? r1 : 0.0;
    const double d2 = bad1 ? a22 : det * (r1 * r1);
    const bool bad2 = !(d2 > 0.0) || d2 <= kRankTol * kRankTol * own[o + k + 1];
    double i2 = (d1 * r1) * rd;
    if (bad1) i2 = rsqrt(a22);
    if (!live2 || bad2) i2 = 0.0;
    any_bad = any_bad || (live1 && bad1) || (live2 && bad2);
#pragma unroll
    for (int c = k + 1; c < kLive; ++c) a[k][c] *= i1;
#pragma unroll
    for (int c = k + 2; c < kLive; ++c) a[k + 1][c] = (a[k + 1][c] - a[k][k + 1] * a[k][c]) * i2;
    b[k] *= i1;
    b[k + 1] = (b[k + 1] - a[k][k + 1] * b[k]) * i2;
#pragma unroll
    for (int i = k + 2; i < kLive; ++i) {
#pragma unroll
      for (int c = i; c < kLive; ++c) a[i][c] = (a[i][c] - a[k][i] * a[k][c]) - a[k + 1][i] * a[k + 1][c];
      b[i] = (b[i] - a[k][i] * b[k]) - a[k + 1][i] * b[k + 1];
    }
  }
  if (any_bad && report && lane == 0) atomicExch(&status->rank_deficient, 1);
  if (lane < kBlk) {
#pragma unroll
    for (int i = 0; i < kBlk; ++i) M[(o + j) * mp + o + i] = i < kLive ? b[i < kLive ? i : 0] : 0.0;
  }
}

// One 8 x 8 tile  C += sign P Q  of doubles in shared memory, k from 0 to kdim - 1:
// element (i, k) of P at p[k * pk + i * pi], element (k, j) of Q at q[k * qk + j].
__device__ __forceinline__ void dtile(double& c0, double& c1, const double* p, int pk, int pi, const double* q, int qk, int kdim,
                                      double sign) {
  const int lane = threadIdx.x & 31, fr = lane >> 2, fc = lane & 3;
#pragma unroll 2
  for (int k = 0; k < kdim; k += 4) dmma_m8n8k4(c0, c1, sign * p[(k + fc) * pk + fr * pi], q[(k + fc) * qk + fr]);
}

// Block (i, j), i < j, of M = R^-1 by one warp, the blocks of M left of column j and D_j being known:
// M_ij = -(sum_{i <= l < j} M_il R_lj) D_j.  The sum passes through the block (j, i) below the diagonal of A, which nothing
// else uses.
template <int NT>
__device__ __forceinline__ void qr_inverse_block(double* A, double* M, int i, int j) {
  constexpr int ap = QrCfg<NT>::ap, mp = QrCfg<NT>::mp;
  const int lane = threadIdx.x & 31, fr = lane >> 2, fc = lane & 3;
  double* t = A + kBlk * j * ap + kBlk * i;
  double c0 = 0.0, c1 = 0.0;
  dtile(c0, c1, M + kBlk * i * mp + kBlk * i, 1, mp, A + kBlk * i * ap + kBlk * j, ap, kBlk * (j - i), 1.0);
  t[fr * ap + 2 * fc] = c0; t[fr * ap + 2 * fc + 1] = c1;
  __syncwarp();
  c0 = c1 = 0.0;
  dtile(c0, c1, t, 1, ap, M + kBlk * j * mp + kBlk * j, mp, kBlk, -1.0);
  double* m = M + (kBlk * i + fr) * mp + kBlk * j + 2 * fc;
  m[0] = c0; m[1] = c1;
}

// S (upper triangle in A) -> M = R^-1 (upper triangle) in blocks of 8: one warp factors the diagonal block, the rest of
// the block row, the trailing update and the off-diagonal blocks of M are tiles on the FP64 tensor cores.  Column kb - 1
// of M is made by the other warps while warp 0 factors block kb.  Up to 16 columns one warp does it all.  (One thread
// arrangement over the whole matrix with a barrier per pivot, the form before this one, took 63 us at r = 64; this 15.)
// kOneWarp: by the calling warp alone, for its own lanes (__syncwarp); else by the eight warps of the block together.
template <int NT, int kLive, bool kOneWarp>
__device__ __forceinline__ void qr_factor_by(double* A, double* M, const double* own, int r, DevStatus* status, bool report) {
  constexpr int ap = QrCfg<NT>::ap, mp = QrCfg<NT>::mp;
  const int warp = kOneWarp ? 0 : (int)(threadIdx.x >> 5), lane = threadIdx.x & 31, fr = lane >> 2, fc = lane & 3;
  const int nb = (r + kBlk - 1) / kBlk;
  constexpr int workers = kOneWarp ? 1 : kQrWarps;
  auto sync = [&]() { if (kOneWarp) __syncwarp(); else __syncthreads(); };
  for (int kb = 0; kb < nb; ++kb) {
    const int o = kb * kBlk;
    if (warp == 0) qr_factor_block<NT, kLive>(A, M, own, kb, r, status, report);
    if (!kOneWarp && warp > 0)
      for (int i = warp - 1; i < kb - 1; i += kQrWarps - 1) qr_inverse_block<NT>(A, M, i, kb - 1);
    sync();
    const int ntr = nb - 1 - kb;                            // tiles to the right of the block
    for (int t = warp; t < ntr; t += workers) {             // R_k. = R_kk^-T A_k. in place, a tile per warp
      double* p = A + o * ap + o + kBlk * (t + 1);
      double c0 = 0.0, c1 = 0.0;
      dtile(c0, c1, M + o * mp + o, mp, 1, p, ap, kBlk, 1.0);
      __syncwarp();
      p[fr * ap + 2 * fc] = c0; p[fr * ap + 2 * fc + 1] = c1;
    }
    sync();
    int t = 0;                                              // A_ij -= R_ki^T R_kj on the tiles of the upper triangle
    for (int bi = 0; bi < ntr; ++bi)
      for (int bj = bi; bj < ntr; ++bj, ++t) {
        if (t % workers != warp) continue;
        double* p = A + (o + kBlk * (bi + 1) + fr) * ap + o + kBlk * (bj + 1) + 2 * fc;
        double c0 = p[0], c1 = p[1];
        dtile(c0, c1, A + o * ap + o + kBlk * (bi + 1), ap, 1, A + o * ap + o + kBlk * (bj + 1), ap, kBlk, -1.0);
        p[0] = c0; p[1] = c1;
      }
    sync();
  }
  for (int i = warp; i < nb - 1; i += workers) qr_inverse_block<NT>(A, M, i, nb - 1);
  sync();
}
template <int NT, int kLive = kBlk>
__device__ __forceinline__ void qr_factor(double* A, double* M, const double* own, int r, DevStatus* status, bool report) {
  if constexpr (NT <= 2) {
    if (threadIdx.x < 32) qr_factor_by<NT, kLive, true>(A, M, own, r, status, report);
    __syncthreads();
  } else {
    qr_factor_by<NT, kLive, false>(A, M, own, r, status, report);
  }
}

// Q = Y M in place on `ncols` staged columns: Q^T (r x 8 columns) = M^T Y in 8 x 8 tiles, A[k][j] = M[j][k], K = j up
// to the tile's last k (M is upper triangular).  A warp owns whole 8-column strips, so it may overwrite them.
template <int NT>
__device__ __forceinline__ void qr_apply(float* sY, int pitch, const double* M, int ncols) {
  constexpr int mp = QrCfg<NT>::mp;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, fr = lane >> 2, fc = lane & 3;
  constexpr int kSp = 2;                          // strips at a time: independent chains for the FP64 pipe
  for (int s0 = warp * kSp; s0 < ncols / 8; s0 += kQrWarps * kSp) {
    double acc[kSp][NT][2];
#pragma unroll
    for (int sp = 0; sp < kSp; ++sp)
#pragma unroll
      for (int kt = 0; kt < NT; ++kt) acc[sp][kt][0] = acc[sp][kt][1] = 0.0;
#pragma unroll
    for (int j0 = 0; j0 < 8 * NT; j0 += 4) {
      double b[kSp];
#pragma unroll
      for (int sp = 0; sp < kSp; ++sp) b[sp] = (double)sY[(j0 + fc) * pitch + 8 * (s0 + sp) + fr];
      const double* ma = M + (j0 + fc) * mp + fr;
#pragma unroll
      for (int kt = 0; kt < NT; ++kt)
        if (8 * kt + 7 >= j0) {
          const double a = ma[8 * kt];
#pragma unroll
          for (int sp = 0; sp < kSp; ++sp) dmma_m8n8k4(acc[sp][kt][0], acc[sp][kt][1], a, b[sp]);
        }
    }
    __syncwarp();
#pragma unroll
    for (int sp = 0; sp < kSp; ++sp)
#pragma unroll
      for (int kt = 0; kt < NT; ++kt)
        *reinterpret_cast<float2*>(sY + (8 * kt + fr) * pitch + 8 * (s0 + sp) + 2 * fc) =
            make_float2((float)acc[sp][kt][0], (float)acc[sp][kt][1]);
  }
}

}  // namespace qr
}  // namespace agzo

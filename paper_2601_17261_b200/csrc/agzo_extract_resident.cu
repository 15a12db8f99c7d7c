// Algorithm 1 in one launch for inputs that fit the chip's shared memory.
//
// A small extraction is a chain of 3 K + 3 dependent kernels of 3 to 5 us each, most of which is hand-over: launch, set-up, X
// from L2, the panels through global memory.  Here X is loaded once and stays: a CTA keeps tb x cb blocks of 128 tokens x 128
// columns in the layout that tcgen05.mma reads as X (T = X Q) and as X^T (Y = X^T T), and the operands never leave the chip's
// shared memory either.  The cj CTAs that cover the columns of the same tokens lie in one cluster:
//   T = X Q    every CTA's sums over its columns (TMEM) meet through distributed shared memory; groups of eight tokens are
//              added up in rank order by the CTA that owns them and sent to the T operand of all
//   Y = X^T T  a CTA's sums over its tokens go to global memory (L2) as a partial sum, all CTAs of the unit meet (in a cluster
//              barrier where the unit is one cluster, else at a counter), and the ni partial sums of the CTA's columns are
//              added in order; where ni x columns is large a CTA adds up ni-th of them only and the sums meet once more
//   qr(Y)      the Gram matrix, factor and Q = Y M as in the panel QR (agzo_qr.cuh): shares of the Gram matrix through
//              distributed shared memory, every CTA factoring for itself, a warp per layer
// Operands are fp32 quantities carried as bf16 parts side by side in N: two parts (16 bits) as in the tensor-core products,
// three (24 bits) where the CUDA-core products would run, X in fp32 as three planes with the six products down to 2^-24.
// Accumulation is fp32, over at most 128 tb tokens or 128 cb columns before the sums leave TMEM.
//
// What bounds it is the chain of synchronisations of a round: a cluster barrier 0.2 us, all CTAs of a unit at a counter 1.3, the
// partial sums of Y from L2 1.2, the exchange of T 1.4 and the Gram matrix with its exchange 2 (both read from the peers between
// barriers; sent, 0.3 to 0.9 less together), the factor 0.5 to 2.4.  Against the chain of launches, K = 3: without workspace 4096 x 2048, r = 16 158 -> 85 us;
// 8000 x 256 bf16, r = 8 83 -> 51; 1500 x 515 fp32, r = 5 97 -> 51; 613 x 1024 bf16, three layers of r = 8 53 -> 48.
#include "agzo_qr.cuh"
#include "agzo_resident.cuh"

#include <algorithm>
#include <vector>

namespace agzo {

namespace {

using namespace qr;
using namespace ptx;

constexpr int kThreads = kQrThreads, kWarps = kQrWarps;
constexpr int kBlock = 128;                     // tokens, columns of a block
constexpr int kSlotBytes = 16 * 1024;           // [128 tokens][64 columns] bf16, 128-byte swizzle
constexpr int kShareElems = QrCfg<2>::tiles * 64;
constexpr int kAmBytes = (int)QrCfg<2>::am_bytes;
constexpr size_t kMaxSmem = 226 * 1024;

struct ResShared {
  uint64_t mma;
  uint64_t gram_in, t_in, t_full;      // what the peers send has come: shares of S, partial T, the T operand
  uint32_t tmem_base;
  int failed;
  DevStatus st;
  signed char row_of[64];        // panel rank -> row of the staged Y
  double own[kResMaxLayers][16];
};

__device__ __forceinline__ uint32_t swz(int i, int j) { return (uint32_t)((i >> 3) * 1024 + (i & 7) * 128 + ((j ^ (i & 7)) << 4)); }

__device__ __forceinline__ uint32_t bf16_pair(float a, float b) {
  const __nv_bfloat162 v = __floats2bfloat162_rn(a, b);
  return *reinterpret_cast<const uint32_t*>(&v);
}
// v -> its bf16 parts, each what the ones before it leave over; with three of them all 24 bits
template <int N>
__device__ __forceinline__ void split8(const float (&v)[8], uint4 (&out)[N]) {
  float rest[8];
#pragma unroll
  for (int i = 0; i < 8; ++i) rest[i] = v[i];
#pragma unroll
  for (int p = 0; p < N; ++p) {
    uint32_t w[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      w[i] = bf16_pair(rest[2 * i], rest[2 * i + 1]);
      rest[2 * i] -= __uint_as_float(w[i] << 16);
      rest[2 * i + 1] -= __uint_as_float(w[i] & 0xffff0000u);
    }
    out[p] = make_uint4(w[0], w[1], w[2], w[3]);
  }
}
template <int N>
__device__ __forceinline__ void split1(float v, __nv_bfloat16 (&out)[N]) {
#pragma unroll
  for (int p = 0; p < N; ++p) {
    out[p] = __float2bfloat16_rn(v);
    v -= __bfloat162float(out[p]);
  }
}

__device__ __forceinline__ void cp_async16(uint32_t dst, const void* src, uint32_t bytes) {      // zeros beyond `bytes`
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(src), "r"(bytes) : "memory");
}
__device__ __forceinline__ float4 ld_cluster_f4(uint32_t addr) {
  float4 v;
  asm volatile("ld.shared::cluster.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "r"(addr) : "memory");
  return v;
}
__device__ __forceinline__ void st_cluster_u4(uint32_t addr, uint4 v) {
  asm volatile("st.shared::cluster.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(addr), "r"(v.x), "r"(v.y), "r"(v.z), "r"(v.w) : "memory");
}

// ------------------------------------------------------------------ X into shared memory
// Tokens [t0, t0 + 128 tb), columns [col0, col0 + 128 cb) as bf16 planes, zero beyond m and d.
template <int PLANES>
__device__ __forceinline__ void load_x(const ResidentUnit& U, uint8_t* sX, int plane, int t0, int col0, int tb, int cb) {
  const int per_row = cb * 16, n = tb * kBlock * per_row;          // pieces of eight columns
  const int m = U.m, d = U.d;
  const long long ldx = U.ldx;
  auto place = [&](int t, int c8) {
    return (uint32_t)(((t >> 7) * 2 * cb + (c8 >> 3)) * kSlotBytes + (t & 127) * 128 + (((c8 & 7) ^ (t & 7)) << 4));
  };
  if (PLANES == 1 && U.x_vec) {
    const __nv_bfloat16* X = reinterpret_cast<const __nv_bfloat16*>(U.X);
    const uint32_t base = smem_u32(sX);
#pragma unroll 1
    for (int i = threadIdx.x; i < n; i += kThreads) {
      const int t = i / per_row, c8 = i - t * per_row, gt = t0 + t, gc = col0 + 8 * c8;
      const bool in = gt < m && gc < d;
      cp_async16(base + place(t, c8), in ? X + gt * ldx + gc : X, in ? 16u : 0u);
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
    return;
  }
  constexpr int kU = 4;
#pragma unroll 1
  for (int i0 = threadIdx.x; i0 < n; i0 += kU * kThreads) {
    float v[kU][8];
#pragma unroll
    for (int u = 0; u < kU; ++u) {
      const int i = i0 + u * kThreads, t = i / per_row, gt = t0 + t, gc = col0 + 8 * (i - t * per_row);
#pragma unroll
      for (int c = 0; c < 8; ++c) v[u][c] = 0.f;
      if (i >= n || gt >= m) continue;
      const long long at = gt * ldx + gc;
      if (PLANES == 3 && U.x_vec) {
        const float* X = reinterpret_cast<const float*>(U.X);
#pragma unroll
        for (int h = 0; h < 2; ++h)
          if (gc + 4 * h < d) {
            const float4 x = *reinterpret_cast<const float4*>(X + at + 4 * h);
            v[u][4 * h] = x.x; v[u][4 * h + 1] = x.y; v[u][4 * h + 2] = x.z; v[u][4 * h + 3] = x.w;
          }
      } else {
#pragma unroll
        for (int c = 0; c < 8; ++c)
          if (gc + c < d)
            v[u][c] = PLANES == 3 ? reinterpret_cast<const float*>(U.X)[at + c]
                                  : __bfloat162float(reinterpret_cast<const __nv_bfloat16*>(U.X)[at + c]);
      }
    }
#pragma unroll
    for (int u = 0; u < kU; ++u) {
      const int i = i0 + u * kThreads, t = i / per_row;
      if (i >= n) break;
      uint4 part[PLANES];
      split8<PLANES>(v[u], part);
#pragma unroll
      for (int p = 0; p < PLANES; ++p) *reinterpret_cast<uint4*>(sX + p * plane + place(t, i - t * per_row)) = part[p];
    }
  }
}

// ------------------------------------------------------------------ Omega into the T operand
// Rows of the test matrix of this CTA's tokens (see fill_omega_kernel for the stream); the CTAs of a row each make all of them.
template <int PARTS>
__device__ __forceinline__ void fill_omega(const ResidentUnit& U, uint8_t* sT, int t0, int tb, unsigned long long seed) {
  const int tokens = min(tb * kBlock, U.m - t0), NB = U.NB, NP = U.NP;
  if (tokens <= 0) return;
#pragma unroll 1
  for (int l = 0; l < U.n_layers; ++l) {
    const int r = U.layer[l].r, off = U.layer[l].off;
    const unsigned id = U.layer[l].layer_id;
    const unsigned long long b0 = (unsigned long long)t0 * r / 4;       // t0 is a multiple of 128
#pragma unroll 1
    for (int b = threadIdx.x; 4 * b < tokens * r; b += kThreads) {
      const float4 g = gaussian_block(b0 + b, id, kTagOmega, seed);
      const float v[4] = {g.x, g.y, g.z, g.w};
      int t = 4 * b / r, k = 4 * b - t * r;
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        __nv_bfloat16 part[PARTS];
        split1<PARTS>(v[e], part);
        uint8_t* box = sT + (size_t)(t >> 6) * NB * 128 + (t & 7) * 2;
        if (t < tokens) {
#pragma unroll
          for (int p = 0; p < PARTS; ++p) *reinterpret_cast<__nv_bfloat16*>(box + swz(p * NP + off + k, (t & 63) >> 3)) = part[p];
        }
        if (++k == r) { k = 0; ++t; }
      }
    }
  }
}

__device__ __forceinline__ void tmem_ld8_issue(uint32_t taddr, uint32_t (&r)[8]) {
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7])
               : "r"(taddr));
}
// Eight ranks' sums of this lane's row from TMEM: `chunks` accumulators of NB columns, in each the parts' columns; the parts are
// added from the smallest
template <int PARTS>
__device__ __forceinline__ void tmem_sum8(uint32_t at, int NP, int NB, int chunks, float (&v)[8]) {
  float s[PARTS][8];
#pragma unroll
  for (int p = 0; p < PARTS; ++p)
#pragma unroll
    for (int k = 0; k < 8; ++k) s[p][k] = 0.f;
  constexpr int kC = PARTS == 3 ? 2 : 1;
#pragma unroll 1
  for (int c = 0; c < chunks; c += kC) {
    uint32_t z[kC][PARTS][8];
#pragma unroll
    for (int x = 0; x < kC; ++x)
#pragma unroll
      for (int p = 0; p < PARTS; ++p) tmem_ld8_issue(at + (uint32_t)((c + x) * NB + p * NP), z[x][p]);
    tmem_ld_wait();
#pragma unroll
    for (int x = 0; x < kC; ++x)
#pragma unroll
      for (int p = 0; p < PARTS; ++p)
#pragma unroll
        for (int k = 0; k < 8; ++k) s[p][k] += __uint_as_float(z[x][p][k]);
  }
#pragma unroll
  for (int k = 0; k < 8; ++k) {
    v[k] = s[PARTS - 1][k];
#pragma unroll
    for (int p = PARTS - 2; p >= 0; --p) v[k] += s[p][k];
  }
}

// All CTAs of a unit meet, and what they wrote to global memory before is visible after.  Where the unit is one cluster, the
// cluster's barrier; else a counter (Meeting).  A CTA that has given up waiting says so in the counter while the meeting still lacks
// somebody, so that whoever completes it or finds it complete sees that too: all of them have sh->failed set from there on.  (One that
// starts only then takes what it finds for the count of earlier launches; the others say so again at the next meeting.)
// What is done when a wait runs out, and the meeting itself, are out of line: a round's code is larger than the instruction cache as
// it is, and every line of it costs (mean of 77 calls of 27 to 130 us 61.1 -> 62.2 us with this in the rounds, 61.0 out of line).
struct Meeting {
  unsigned long long* counter;
  int n;                          // CTAs
  bool first;
  unsigned phase, failures;       // what it showed before the launch (thread 0)
};
// arrives and waits for the phase; whether a wait of this CTA's or another's has run out
__device__ __noinline__ bool meet(unsigned long long* counter, unsigned long long add, unsigned phase, unsigned failures, bool failed,
                                  unsigned long long wait_ns) {
  if (failed) add += kMeetingFailure;
  asm volatile("red.release.gpu.global.add.u64 [%0], %1;" ::"l"(counter), "l"(add) : "memory");
  if (failed) return true;
  const unsigned long long t_start = global_ns();
#pragma unroll 1
  for (;;) {
    unsigned long long got;
    asm volatile("ld.acquire.gpu.global.u64 %0, [%1];" : "=l"(got) : "l"(counter) : "memory");
    if (meeting_phase(got) == phase) return meeting_failures(got) != failures;
    if (global_ns() - t_start > wait_ns && atomicCAS(counter, got, got + kMeetingFailure) == got) return true;
  }
}
__device__ __forceinline__ void unit_barrier(Meeting& m, int clusters, int cs, const ResidentParams& P, ResShared* sh) {
  if (clusters == 1) {
    __syncwarp();
    if (cs > 1) cluster_sync_all(); else __syncthreads();
    return;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    const unsigned long long add = meeting_increment(m.n, m.first, m.phase);
    m.phase ^= 1u;
    if (meet(m.counter, add, m.phase, m.failures, sh->failed != 0, P.wait_ns)) sh->failed = 1;
  }
  __syncthreads();
}
// A product or a sum that did not come: known to the n CTAs of the cluster where that is all of the unit, else to the others by the next
// meeting.  By every lane whose wait ran out: near the limit it can be one warp's, or one lane's, and not the first one's.
__device__ __noinline__ void product_failed(ResShared* sh, int n) {
  sh->failed = 1;
#pragma unroll 1
  for (int c = 0; c < n; ++c) st_cluster_u32(mapa_shared(smem_u32(&sh->failed), (uint32_t)c), 1u);
}
// V = 0, with which a pass changes nothing: the strips of the CTA in row i whose first column is col0
__device__ __noinline__ void zero_strips(const ResidentUnit& U, int i, int col0) {
  const int lane = threadIdx.x & 31;
  for (int l = 0; l < U.n_layers; ++l)
    for (int s0 = threadIdx.x >> 5; s0 < U.cb * 8; s0 += kWarps) {
      const int c = 16 * s0 + (lane & 15);
      if (s0 % U.ni != i || c >= U.d - col0) continue;
      for (int k = lane >> 4; k < U.layer[l].r; k += 2) U.layer[l].V[col0 + k * U.layer[l].ldv + c] = 0.f;
    }
}

// Gram products of one layer's rows of the staged Y, by `split` warps of which this is number `me`
template <int NT>
__device__ __forceinline__ void gram_layer(const float* y, int pitch, int steps, int me, int split, double* part) {
  const int lane = threadIdx.x & 31, fr = lane >> 2, fc = lane & 3, el = fr * 8 + 2 * fc;
  double acc[QrCfg<NT>::tiles][2];
#pragma unroll
  for (int t = 0; t < QrCfg<NT>::tiles; ++t) acc[t][0] = acc[t][1] = 0.0;
  const float* base = y + fr * pitch + fc;
#pragma unroll 4
  for (int ks = me; ks < steps; ks += split) {
    double f[NT];
#pragma unroll
    for (int b = 0; b < NT; ++b) f[b] = (double)base[8 * b * pitch + 4 * ks];
    int t = 0;
#pragma unroll
    for (int bi = 0; bi < NT; ++bi)
#pragma unroll
      for (int bj = bi; bj < NT; ++bj, ++t) dmma_m8n8k4(acc[t][0], acc[t][1], f[bi], f[bj]);
  }
#pragma unroll
  for (int t = 0; t < QrCfg<NT>::tiles; ++t) *reinterpret_cast<double2*>(part + me * kShareElems + t * 64 + el) = make_double2(acc[t][0], acc[t][1]);
}
// Q = Y M of 16 columns of one layer (first column c0 of the CTA's), a warp: into the operand Q as bf16 parts, or (V) out
template <int NT, int PARTS>
__device__ __forceinline__ void apply_strips(const float* y, int pitch, const double* M, int c0, int r, uint8_t* sQ, int NB, int NP,
                                             int off, float* V, long long ldv, int live_cols) {
  constexpr int mp = QrCfg<NT>::mp;
  const int lane = threadIdx.x & 31, fr = lane >> 2, fc = lane & 3;
  double acc[2][NT][2];
#pragma unroll
  for (int sp = 0; sp < 2; ++sp)
#pragma unroll
    for (int kt = 0; kt < NT; ++kt) acc[sp][kt][0] = acc[sp][kt][1] = 0.0;
#pragma unroll
  for (int j0 = 0; j0 < 8 * NT; j0 += 4) {
    double b[2];
#pragma unroll
    for (int sp = 0; sp < 2; ++sp) b[sp] = (double)y[(j0 + fc) * pitch + c0 + 8 * sp + fr];
#pragma unroll
    for (int kt = 0; kt < NT; ++kt)
      if (8 * kt + 7 >= j0) {
        const double a = M[(j0 + fc) * mp + fr + 8 * kt];
#pragma unroll
        for (int sp = 0; sp < 2; ++sp) dmma_m8n8k4(acc[sp][kt][0], acc[sp][kt][1], a, b[sp]);
      }
  }
#pragma unroll
  for (int sp = 0; sp < 2; ++sp)
#pragma unroll
    for (int kt = 0; kt < NT; ++kt) {
      const int k = 8 * kt + fr, c = c0 + 8 * sp + 2 * fc;
      if (k >= r) continue;
      float a = (float)acc[sp][kt][0], b = (float)acc[sp][kt][1];
      if (V) {
        float* out = V + k * ldv + c;
        if (c + 1 < live_cols && (reinterpret_cast<uintptr_t>(out) & 7u) == 0) {
          *reinterpret_cast<float2*>(out) = make_float2(a, b);
        } else {
          if (c < live_cols) out[0] = a;
          if (c + 1 < live_cols) out[1] = b;
        }
      } else {
        uint8_t* box = sQ + (size_t)(c >> 6) * NB * 128 + (c & 7) * 2;
#pragma unroll
        for (int p = 0; p < PARTS; ++p) {
          const uint32_t w = bf16_pair(a, b);
          *reinterpret_cast<uint32_t*>(box + swz(p * NP + off + k, (c & 63) >> 3)) = w;
          a -= __uint_as_float(w << 16);
          b -= __uint_as_float(w & 0xffff0000u);
        }
      }
    }
}
// One product of this CTA's blocks: nd accumulators side by side, each the sum over `boxes` pieces of 64 of the contracted
// dimension (all of them; with three parts an accumulator per piece, since the tensor core truncates what it accumulates: the
// pieces' sums are added with rounding).  Planes of X go from the smallest, for the same reason.
template <int PLANES, int PARTS>
__device__ __forceinline__ void issue_product(uint32_t go, uint32_t tmem, uint32_t ax, uint32_t plane, uint32_t ab, int nd, int boxes,
                                              uint32_t d_step, uint32_t box_step, uint32_t box_pair, uint32_t lbo, uint32_t kk_step,
                                              int a_mn, int NB, int NP) {
  const int n_plane[3] = {NB, (2 * NP + 15) & ~15, (NP + 15) & ~15};     // operand rows that a plane of X meets
  uint32_t d = tmem;
#pragma unroll 1
  for (int b = 0; b < nd; ++b) {
    uint32_t acc = 0u;
#pragma unroll 1
    for (int h = 0; h < boxes; ++h) {
      const uint64_t bd = smem_desc(ab + (uint32_t)(h * NB * 128), 0, 1024);
      const uint32_t x0 = ax + (uint32_t)b * d_step + (uint32_t)(h >> 1) * box_pair + (uint32_t)(h & 1) * box_step;
#pragma unroll
      for (int p = PLANES - 1; p >= 0; --p) {
        const uint64_t xd = smem_desc(x0 + (uint32_t)p * plane, lbo, 1024);
        const uint32_t idesc = instr_desc(128, n_plane[p], a_mn, 0), idesc_all = instr_desc(128, NB, a_mn, 0);
#pragma unroll
        for (int kk = 0; kk < 4; ++kk) {       // an accumulator's first instruction writes all of its columns
          mma_bf16_if(go, d, xd + (uint64_t)(kk_step * kk), bd + (uint64_t)(2 * kk), p == PLANES - 1 && kk == 0 ? idesc_all : idesc, acc);
          acc = 1u;
        }
      }
      if (PARTS == 3) { d += (uint32_t)NB; acc = 0u; }
    }
    if (PARTS != 3) d += (uint32_t)NB;
  }
}
// Row and column in S of element i of a share (tiles of the upper triangle)
template <int NT>
__device__ __forceinline__ void share_place(int i, int* row, int* col) {
  int t = i >> 6, bi = 0;
  while (t >= NT - bi) { t -= NT - bi; ++bi; }
  *row = 8 * bi + ((i & 63) >> 3);
  *col = 8 * (bi + t) + (i & 7);
}
// element i of a share -> S
template <int NT>
__device__ __forceinline__ void place_share(double* A, double* own, int i, double v) {
  int row, col;
  share_place<NT>(i, &row, &col);
  A[row * QrCfg<NT>::ap + col] = v;
  if (row == col) own[row] = v;
}
// Bytes of Y, with which the pieces of T that the warps send take turns
__host__ __device__ constexpr int push_front(int y_bytes, int parts) { return y_bytes > kWarps * parts * 256 ? y_bytes : kWarps * parts * 256; }

// PUSH: what a cluster's CTAs exchange is sent (st.async, counted on the receiver's barrier) into buffers that nothing else uses at the
// time: a way instead of a barrier of the cluster, a round trip, and for T another barrier.  512 x 256 fp32, r = 4 35.3 -> 32.2 us, the
// layers of a block of width 1024 with 613 tokens 45.3 -> 42.7 on the mean.  No buffer is sent to before its owner is done with it: a
// CTA sends its shares of a round only after the exchange of T of the last one (or a meeting), which its peers' sums of the shares before
// precede, and partial T only after the exchange of the shares.  Otherwise it is read from the peers between barriers (resident_plan).
template <int PLANES, int PARTS, bool PUSH>
__global__ void __launch_bounds__(kThreads, 1) resident_extract_kernel(const __grid_constant__ ResidentParams P) {
  extern __shared__ __align__(1024) uint8_t smem_raw[];
  __shared__ ResShared sh;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int cs = P.cs, cluster = (int)blockIdx.x / cs, rank = (int)blockIdx.x - cluster * cs;
  int unit = 0;
  while (unit + 1 < P.n_units && cluster >= P.unit[unit + 1].cluster0) ++unit;
  const ResidentUnit& U = P.unit[unit];
  const int cj = U.cj, j = rank % cj, row0 = rank - j, ni = U.ni, i = (cluster - U.cluster0) * (cs / cj) + rank / cj;
  const int cb = U.cb, tb = U.tb, NB = U.NB, NP = U.NP, ranks = U.ranks, nl = U.n_layers, clusters = U.clusters;
  const int ncols = cb * kBlock, col0 = j * ncols, cols_pad = cj * ncols, t0 = i * tb * kBlock, pitch = qr_pitch(ncols);
  Meeting meeting{P.counters + U.counter, clusters * cs, i == 0 && j == 0, 0u, 0u};
  // no meeting of this launch is complete before this CTA has arrived; asked for here, where nothing waits for it (a launch of several
  // clusters per unit does not start before the kernel in front is done; beside the loads of X: twenty calls of the entry without
  // workspace 53.8 -> 54.6 us on the mean)
  const unsigned long long met = clusters > 1 && tid == 0 ? __ldcg(meeting.counter) : 0ull;

  const int plane = tb * cb * 2 * kSlotBytes;
  uint8_t* sX = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
  // Q [2 cb boxes][NB][64 columns] and T [2 tb boxes][NB][64 tokens] take turns in one place: T is written, by the peers too,
  // after the product that reads Q, and Q after the one that reads T
  uint8_t* sQ = sX + PLANES * plane;
  uint8_t* sT = sQ;
  int n_share = 0;                                       // elements of the shares of all layers
#pragma unroll 1
  for (int l = 0; l < nl; ++l) n_share += U.layer[l].r <= 8 ? 64 : kShareElems;
  const int n_gram = U.sub ? cs : cj, gram0 = U.sub ? 0 : row0;          // CTAs whose shares are added up, the first of them
  const bool wide = U.sub && clusters > 1;               // the clusters' shares meet in global memory
  // shares of S, one layer's after another's; those of all CTAs where they are sent
  double* sG = reinterpret_cast<double*>(sQ + max(cb, tb) * 2 * NB * 128);
  uint8_t* sAM = reinterpret_cast<uint8_t*>(sG + (PUSH ? n_gram * n_share : nl * kShareElems));      // [layer] S / R and M
  uint8_t* sU = sAM + nl * kAmBytes;
  float* sY = reinterpret_cast<float*>(sU);              // [rows][pitch] ...
  double* sPart = reinterpret_cast<double*>(sY + (size_t)U.rows * pitch);        // ... and [layer][warp] shares of S; or
  float* sEx = reinterpret_cast<float*>(sU);             // [rank group][128 tb tokens][8] partial T ...
  __nv_bfloat16* sStage = reinterpret_cast<__nv_bfloat16*>(sEx + (size_t)tb * kBlock * NP);    // ... and pieces to send
  if (PUSH) {                          // partial T [CTA][token group of mine][8][NP] take turns with the warps' shares, pieces with Y
    sStage = reinterpret_cast<__nv_bfloat16*>(sU) + warp * (PARTS * 128);
    sPart = reinterpret_cast<double*>(sU + push_front(U.rows * pitch * 4, PARTS));
    sEx = reinterpret_cast<float*>(sPart);
  }

  const int y_chunks = PARTS == 3 ? 2 * tb : 1, t_chunks = PARTS == 3 ? 2 * cb : 1;
  uint32_t ncol = 32;
  while ((int)ncol < max(cb * y_chunks, tb * t_chunks) * NB) ncol <<= 1;
  if (tid == 0) {
    mbar_init(&sh.mma, 1);
    mbar_init(&sh.gram_in, 1);
    mbar_init(&sh.t_in, 1);
    mbar_init(&sh.t_full, 1);
    sh.failed = 0;
    sh.st = DevStatus{};
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 1) tmem_alloc(&sh.tmem_base, ncol);
  if (tid < 64) {
    int row = -1;
#pragma unroll 1
    for (int l = 0; l < nl; ++l)
      if (tid >= U.layer[l].off && tid < U.layer[l].off + U.layer[l].r) row = U.layer[l].row + tid - U.layer[l].off;
    sh.row_of[tid] = (signed char)row;
  }
  // operand rows beyond the ranks stay zero
#pragma unroll 1
  for (int k = tid; k < max(cb, tb) * 2 * NB * 8; k += kThreads) reinterpret_cast<uint4*>(sQ)[k] = make_uint4(0u, 0u, 0u, 0u);
  __syncthreads();
  if (PUSH && cs > 1) asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");      // my barriers can be sent to
  if (!(PLANES == 1 && U.x_vec)) fill_omega<PARTS>(U, sT, t0, tb, P.seed);      // needs nothing from before the launch
  chain_wait();
  load_x<PLANES>(U, sX, plane, t0, col0, tb, cb);
  if (PLANES == 1 && U.x_vec) fill_omega<PARTS>(U, sT, t0, tb, P.seed);         // while X arrives
  asm volatile("cp.async.wait_all;" ::: "memory");
  meeting.phase = meeting_phase(met);
  meeting.failures = meeting_failures(met);
  if (clusters > 1 && tid == 0 && meeting.first && P.late_ns) {
    const unsigned long long t_late = global_ns() + P.late_ns;
    while (global_ns() < t_late) {}
  }

  const uint32_t tmem = sh.tmem_base;
  const uint32_t go = elect_one();
  const uint32_t ax = smem_u32(sX), aq = smem_u32(sQ), at = smem_u32(sT);
  const int q = warp & 3, half = warp >> 2, groups = NP / 8;
  const uint32_t lanes = (uint32_t)(q * 32) << 16;
  const int gram_split = U.gram_split;
  uint32_t mma_par = 0, gram_par = 0, t_par = 0;
  // element e of the shares of all layers: layer l, element x of its tiles
  auto share_at = [&](int e, int* l, int* x) {
    *l = 0;
#pragma unroll 1
    for (;; ++*l) {
      const int n = U.layer[*l].r <= 8 ? 64 : kShareElems;
      if (e < n) break;
      e -= n;
    }
    *x = e;
  };
  // PUSH: this thread's two elements of the shares (at most 512 for 24 ranks in four layers), where they come from and go to
  const bool has_pair = PUSH && 2 * tid < n_share;
  const double* pair_src = sPart;
  double *pair_dst = nullptr, *pair_diag = nullptr;
  bool diag_second = false;
  if (has_pair) {
    int l, x, row, col;
    share_at(2 * tid, &l, &x);
    pair_src = sPart + l * gram_split * kShareElems + x;
    double* A = reinterpret_cast<double*>(sAM + l * kAmBytes);
    if (U.layer[l].r <= 8) { share_place<1>(x, &row, &col); pair_dst = A + row * QrCfg<1>::ap + col; }
    else { share_place<2>(x, &row, &col); pair_dst = A + row * QrCfg<2>::ap + col; }
    diag_second = row == col + 1;
    if (row == col || diag_second) pair_diag = &sh.own[l][row];
  }
  auto place_pair = [&](double2 v) {
    pair_dst[0] = v.x;
    pair_dst[1] = v.y;
    if (pair_diag) *pair_diag = diag_second ? v.y : v.x;
  };
  const int own = tb * (kBlock / 8) / cj;                // token groups whose T is added up here: j, j + cj, ... (cj divides 16)
  __syncwarp();
  if (PUSH && cs > 1) asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
  const int width = U.sub ? (i < ni ? max(0, min(U.sub, ncols - i * U.sub)) : 0) : ncols;     // columns of Y that are added up here
  const int c_first = U.sub ? i * U.sub : 0;
  const bool direct = ni == 1;

  for (int round = 0;; ++round) {
    const bool last = round == P.K;
    // Partial sums that every CTA adds up for itself: a CTA that is a round ahead must not write over what another still reads; two
    // rounds ahead none can be
    float* ypart = U.ypart + (U.sub == 0 && (round & 1) ? (long long)ni * ranks * cols_pad : 0ll);
    // ---------------------------------------------------------------- Y = X^T T of this CTA's tokens
    fence_proxy_async();
    tc_fence_before();
    __syncthreads();
    if (warp == 0) {
      tc_fence_after();
      issue_product<PLANES, PARTS>(go, tmem, ax, (uint32_t)plane, at, cb, 2 * tb, 2 * kSlotBytes, kSlotBytes / 2,
                                   (uint32_t)(2 * cb * kSlotBytes), kSlotBytes, 128u, 1, NB, NP);
      mma_commit_if(go, &sh.mma);
    }
    if (!mbar_wait(&sh.mma, mma_par)) product_failed(&sh, clusters == 1 ? cs : 1);
    mma_par ^= 1u;
    tc_fence_after();
    if (i < ni)
#pragma unroll 1
      for (int b = 0, it = 0; b < cb; ++b)
#pragma unroll 1
        for (int k0 = 0; k0 < NP; k0 += 8, ++it) {
          if ((it & 1) != half) continue;
          float v[8];
          tmem_sum8<PARTS>(tmem + lanes + (uint32_t)(b * y_chunks * NB + k0), NP, NB, y_chunks, v);
          const int c = b * kBlock + 32 * q + lane;
          float* out = ypart + ((long long)i * ranks + k0) * cols_pad + col0 + c;
#pragma unroll
          for (int k = 0; k < 8; ++k)
            if (k0 + k < ranks) {
              if (direct) sY[sh.row_of[k0 + k] * pitch + c] = v[k];
              else out[k * cols_pad] = v[k];
            }
        }
    // ---------------------------------------------------------------- the sum over the tokens' CTAs, this CTA's columns
#pragma unroll 1
    for (int l = 0; l < nl; ++l) {                                     // rows between the layers
      const int r = U.layer[l].r, pad = -r & 7;
      float4* y = reinterpret_cast<float4*>(sY + (U.layer[l].row + r) * pitch);
#pragma unroll 1
      for (int k = tid; k < pad * (pitch / 4); k += kThreads) y[k] = make_float4(0.f, 0.f, 0.f, 0.f);
    }
    if (!direct) {
      unit_barrier(meeting, clusters, cs, P, &sh);
      const long long part = (long long)ranks * cols_pad;
      if (U.sub == 0) {              // a warp per rank and 128 columns, three of them and five partial sums in flight
        constexpr int kE = 3, kP = 5;
        const int n_items = ranks * cb;
#pragma unroll 1
        for (int i0 = warp; i0 < n_items; i0 += kE * kWarps) {
          const float* src[kE];
          float* dst[kE];
          float4 sum[kE];
#pragma unroll
          for (int e = 0; e < kE; ++e) {
            const int it = min(i0 + e * kWarps, n_items - 1), k = it / cb, c = (it - k * cb) * kBlock + 4 * lane;
            src[e] = ypart + (long long)k * cols_pad + col0 + c;
            dst[e] = sY + sh.row_of[k] * pitch + c;
            sum[e] = make_float4(0.f, 0.f, 0.f, 0.f);
          }
#pragma unroll 1
          for (int s0 = 0; s0 < ni; s0 += kP) {
            float4 t[kE][kP];
#pragma unroll
            for (int e = 0; e < kE; ++e)
#pragma unroll
              for (int x = 0; x < kP; ++x)
                t[e][x] = i0 + e * kWarps < n_items && s0 + x < ni ? __ldcg(reinterpret_cast<const float4*>(src[e] + (s0 + x) * part))
                                                                   : make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
            for (int e = 0; e < kE; ++e)
#pragma unroll
              for (int x = 0; x < kP; ++x) { sum[e].x += t[e][x].x; sum[e].y += t[e][x].y; sum[e].z += t[e][x].z; sum[e].w += t[e][x].w; }
          }
#pragma unroll
          for (int e = 0; e < kE; ++e)
            if (i0 + e * kWarps < n_items) *reinterpret_cast<float4*>(dst[e]) = sum[e];
        }
      } else {                       // few columns, many partial sums: four neighbouring lanes share a sum
        const int v4 = width / 4;
#pragma unroll 1
        for (int e0 = 0; e0 < ranks * v4 * 4; e0 += kThreads) {
          const int e = (e0 + tid) >> 2, g = tid & 3, k = v4 ? e / v4 : 0, c = 4 * (e - k * v4);
          const bool live = e < ranks * v4;
          const float* src = ypart + (long long)k * cols_pad + col0 + c_first + c;
          float4 sum = make_float4(0.f, 0.f, 0.f, 0.f);
          constexpr int kP = 8;
          const int lo = g * ni / 4, hi = (g + 1) * ni / 4;
#pragma unroll 1
          for (int s0 = lo; s0 < hi; s0 += kP) {
            float4 t[kP];
#pragma unroll
            for (int x = 0; x < kP; ++x)
              t[x] = live && s0 + x < hi ? __ldcg(reinterpret_cast<const float4*>(src + (s0 + x) * part)) : make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
            for (int x = 0; x < kP; ++x) { sum.x += t[x].x; sum.y += t[x].y; sum.z += t[x].z; sum.w += t[x].w; }
          }
#pragma unroll
          for (int o = 1; o < 4; o <<= 1) {
            sum.x += __shfl_xor_sync(0xffffffffu, sum.x, o); sum.y += __shfl_xor_sync(0xffffffffu, sum.y, o);
            sum.z += __shfl_xor_sync(0xffffffffu, sum.z, o); sum.w += __shfl_xor_sync(0xffffffffu, sum.w, o);
          }
          if (live && g == 0) {
            *reinterpret_cast<float4*>(sY + sh.row_of[k] * pitch + c) = sum;
            *reinterpret_cast<float4*>(U.y + (long long)k * cols_pad + col0 + c_first + c) = sum;
          }
        }
      }
    }
    __syncthreads();
    // ---------------------------------------------------------------- Gram matrix of every layer
    {
      const int l = warp / gram_split, me = warp - l * gram_split;
      if (l < nl) {
        const float* y = sY + U.layer[l].row * pitch;
        double* part = sPart + l * gram_split * kShareElems;
        if (U.layer[l].r <= 8) gram_layer<1>(y, pitch, width / 4, me, gram_split, part);
        else gram_layer<2>(y, pitch, width / 4, me, gram_split, part);
      }
    }
    __syncthreads();
    if constexpr (PUSH) {
      if (has_pair) {
        double2 v[kWarps], sum = make_double2(0.0, 0.0);
#pragma unroll
        for (int w = 0; w < kWarps; ++w)
          v[w] = w < gram_split ? *reinterpret_cast<const double2*>(pair_src + w * kShareElems) : make_double2(0.0, 0.0);
#pragma unroll
        for (int w = 0; w < kWarps; ++w) { sum.x += v[w].x; sum.y += v[w].y; }
        if (n_gram == 1) {
          place_pair(sum);
        } else {
          const uint32_t to = smem_u32(sG + (rank - gram0) * n_share + 2 * tid), bar = smem_u32(&sh.gram_in);
          const uint32_t w[4] = {(uint32_t)__double2loint(sum.x), (uint32_t)__double2hiint(sum.x), (uint32_t)__double2loint(sum.y),
                                 (uint32_t)__double2hiint(sum.y)};
#pragma unroll 1
          for (int c = 0; c < n_gram; ++c) st_async_u4(mapa_shared(to, (uint32_t)(gram0 + c)), w, mapa_shared(bar, (uint32_t)(gram0 + c)));
        }
      }
      if (n_gram > 1) {
        if (tid == 0) mbar_expect_tx(&sh.gram_in, (uint32_t)(n_gram * n_share * 8));
        if (!mbar_wait_cluster(&sh.gram_in, gram_par)) product_failed(&sh, clusters == 1 ? cs : 1);
        gram_par ^= 1u;
        if (has_pair) {
          double2 v[8], sum = make_double2(0.0, 0.0);
#pragma unroll
          for (int c = 0; c < 8; ++c)
            v[c] = c < n_gram ? *reinterpret_cast<const double2*>(sG + c * n_share + 2 * tid) : make_double2(0.0, 0.0);
#pragma unroll
          for (int c = 0; c < 8; ++c) { sum.x += v[c].x; sum.y += v[c].y; }
          place_pair(sum);
        }
      }
    } else {
#pragma unroll 1
      for (int e = tid; e < n_share; e += kThreads) {
        int l, x;
        share_at(e, &l, &x);
        double v[kWarps], sum = 0.0;
#pragma unroll
        for (int w = 0; w < kWarps; ++w) v[w] = w < gram_split ? sPart[(l * gram_split + w) * kShareElems + x] : 0.0;
#pragma unroll
        for (int w = 0; w < kWarps; ++w) sum += v[w];
        sG[e] = sum;
      }
      __syncwarp();
      if (cs > 1) cluster_sync_all(); else __syncthreads();
      {
        auto place = [&](int e, double v) {
          int l, x;
          share_at(e, &l, &x);
          double* A = reinterpret_cast<double*>(sAM + l * kAmBytes);
          if (U.layer[l].r <= 8) place_share<1>(A, sh.own[l], x, v); else place_share<2>(A, sh.own[l], x, v);
        };
        if (!wide || rank == 0)
#pragma unroll 1
          for (int e = tid; e < n_share; e += kThreads) {
            double v[8], sum = 0.0;
#pragma unroll
            for (int c = 0; c < 8; ++c) v[c] = c < n_gram ? ld_cluster_f64(mapa_shared(smem_u32(sG + e), (uint32_t)(gram0 + c))) : 0.0;
#pragma unroll
            for (int c = 0; c < 8; ++c) sum += v[c];
            if (wide) U.gshare[(cluster - U.cluster0) * n_share + e] = sum; else place(e, sum);
          }
        if (wide) {
          unit_barrier(meeting, clusters, cs, P, &sh);
#pragma unroll 1
          for (int e = tid; e < n_share; e += kThreads) {
            double sum = 0.0;
            constexpr int kP = 16;
#pragma unroll 1
            for (int s0 = 0; s0 < clusters; s0 += kP) {
              double t[kP];
#pragma unroll
              for (int c = 0; c < kP; ++c) t[c] = s0 + c < clusters ? __ldcg(U.gshare + (s0 + c) * n_share + e) : 0.0;
#pragma unroll
              for (int c = 0; c < kP; ++c) sum += t[c];
            }
            place(e, sum);
          }
        }
      }
    }
    __syncthreads();
    // ---------------------------------------------------------------- factor, a warp per layer; Y of all columns meanwhile
    if (warp < nl) {
      const int r = U.layer[warp].r;
      double* A = reinterpret_cast<double*>(sAM + warp * kAmBytes);
      const bool report = i == 0 && j == 0;
      if (r <= 4) qr_factor_by<1, 4, true>(A, A + QrCfg<1>::r8 * QrCfg<1>::ap, sh.own[warp], r, &sh.st, report);
      else if (r <= 8) qr_factor_by<1, 8, true>(A, A + QrCfg<1>::r8 * QrCfg<1>::ap, sh.own[warp], r, &sh.st, report);
      else qr_factor_by<2, 8, true>(A, A + QrCfg<2>::r8 * QrCfg<2>::ap, sh.own[warp], r, &sh.st, report);
    } else if (U.sub) {
      const int v4 = ncols / 4, first = tid - 32 * nl, step = kThreads - 32 * nl;
#pragma unroll 1
      for (int e0 = first; e0 < ranks * v4; e0 += 4 * step) {
        float4 t[4];
#pragma unroll
        for (int x = 0; x < 4; ++x) {
          const int e = e0 + x * step, k = e / v4;
          if (e < ranks * v4) t[x] = __ldcg(reinterpret_cast<const float4*>(U.y + (long long)k * cols_pad + col0) + (e - k * v4));
        }
#pragma unroll
        for (int x = 0; x < 4; ++x) {
          const int e = e0 + x * step, k = e / v4;
          if (e < ranks * v4) *reinterpret_cast<float4*>(sY + sh.row_of[k] * pitch + 4 * (e - k * v4)) = t[x];
        }
      }
    }
    __syncthreads();
    // ---------------------------------------------------------------- Q = Y M: the operand, or V (whose strips the rows of CTAs share)
#pragma unroll 1
    for (int l = 0; l < nl; ++l) {
      const int r = U.layer[l].r, off = U.layer[l].off;
      const double* A = reinterpret_cast<const double*>(sAM + l * kAmBytes);
      const float* y = sY + U.layer[l].row * pitch;
      float* V = last ? U.layer[l].V + col0 : nullptr;
#pragma unroll 1
      for (int s0 = warp; s0 < cb * 8; s0 += kWarps) {
        if (last && s0 % ni != i) continue;
        if (r <= 8) apply_strips<1, PARTS>(y, pitch, A + QrCfg<1>::r8 * QrCfg<1>::ap, 16 * s0, r, sQ, NB, NP, off, V, U.layer[l].ldv, U.d - col0);
        else apply_strips<2, PARTS>(y, pitch, A + QrCfg<2>::r8 * QrCfg<2>::ap, 16 * s0, r, sQ, NB, NP, off, V, U.layer[l].ldv, U.d - col0);
      }
    }
    if (last) break;
    // ---------------------------------------------------------------- T = X Q over this CTA's columns
    fence_proxy_async();
    tc_fence_before();
    __syncthreads();
    if (warp == 0) {
      tc_fence_after();
      issue_product<PLANES, PARTS>(go, tmem, ax, (uint32_t)plane, aq, tb, 2 * cb, (uint32_t)(2 * cb * kSlotBytes), kSlotBytes,
                                   2 * kSlotBytes, 0u, 2u, 0, NB, NP);
      mma_commit_if(go, &sh.mma);
    }
    if (!mbar_wait(&sh.mma, mma_par)) product_failed(&sh, clusters == 1 ? cs : 1);
    mma_par ^= 1u;
    tc_fence_after();
#pragma unroll 1
    for (int b = 0, it = 0; b < tb; ++b)
#pragma unroll 1
      for (int g = 0; g < groups; ++g, ++it) {
        if ((it & 1) != half) continue;
        float v[8];
        tmem_sum8<PARTS>(tmem + lanes + (uint32_t)(b * t_chunks * NB + 8 * g), NP, NB, t_chunks, v);
        const int t = b * kBlock + 32 * q + lane;
        if (cj == 1) {
          uint8_t* box = sT + (size_t)(t >> 6) * NB * 128 + (t & 7) * 2;
#pragma unroll
          for (int k = 0; k < 8; ++k) {
            __nv_bfloat16 part[PARTS];
            split1<PARTS>(v[k], part);
#pragma unroll
            for (int p = 0; p < PARTS; ++p) *reinterpret_cast<__nv_bfloat16*>(box + swz(p * NP + 8 * g + k, (t & 63) >> 3)) = part[p];
          }
        } else if (PUSH) {                                    // to the CTA that adds up this token's group
          const int c = (t >> 3) & (cj - 1), o = (t >> 3) / cj;
          const uint32_t to = mapa_shared(smem_u32(sEx + ((size_t)((j * own + o) * 8 + (t & 7)) * NP + 8 * g)), (uint32_t)(row0 + c));
          const uint32_t bar = mapa_shared(smem_u32(&sh.t_in), (uint32_t)(row0 + c));
          st_async_f4(to, make_float4(v[0], v[1], v[2], v[3]), bar);
          st_async_f4(to + 16u, make_float4(v[4], v[5], v[6], v[7]), bar);
        } else {
          float4* out = reinterpret_cast<float4*>(sEx + ((size_t)g * tb * kBlock + t) * 8);
          out[0] = make_float4(v[0], v[1], v[2], v[3]);
          out[1] = make_float4(v[4], v[5], v[6], v[7]);
        }
      }
    if (PUSH && cj > 1) {
      if (tid == 0) {
        mbar_expect_tx(&sh.t_in, (uint32_t)(tb * kBlock * NP * 4));
        mbar_expect_tx(&sh.t_full, (uint32_t)(tb * (kBlock / 8) * PARTS * NP * 16));
      }
      if (!mbar_wait_cluster(&sh.t_in, t_par)) product_failed(&sh, clusters == 1 ? cs : 1);
      // lane = (one of two pieces, token of the group, half of a rank group): four ranks of a token; a warp sends what it has split
#pragma unroll 1
      for (int e = tid; e < own * 16 * groups; e += kThreads) {
        const int x = (e >> 1) & 7, kh = e & 1, og = e >> 4, o = og / groups, g = og - o * groups;
        const float* src = sEx + (size_t)(o * 8 + x) * NP + 8 * g + 4 * kh;
        float4 z[8], sum = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
        for (int c = 0; c < 8; ++c)
          z[c] = c < cj ? *reinterpret_cast<const float4*>(src + (size_t)c * own * 8 * NP) : make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
        for (int c = 0; c < 8; ++c) { sum.x += z[c].x; sum.y += z[c].y; sum.z += z[c].z; sum.w += z[c].w; }
        const float v[4] = {sum.x, sum.y, sum.z, sum.w};
#pragma unroll
        for (int k = 0; k < 4; ++k) {
          __nv_bfloat16 part[PARTS];
          split1<PARTS>(v[k], part);
#pragma unroll
          for (int p = 0; p < PARTS; ++p) sStage[(((lane >> 4) * PARTS + p) * 8 + 4 * kh + k) * 8 + x] = part[p];
        }
        __syncwarp();
        // 16 PARTS pieces of eight tokens of an operand row, to every CTA of the row
#pragma unroll 1
        for (int n = lane; n < 16 * PARTS; n += 32) {
          const int h = n / (8 * PARTS), p = (n >> 3) - h * PARTS, og_n = ((e - lane) >> 4) + h, o_n = og_n / groups;
          const int row = p * NP + 8 * (og_n - o_n * groups) + (n & 7), tg = j + o_n * cj;
          const uint32_t to = at + (uint32_t)((tg >> 3) * NB * 128) + swz(row, tg & 7), bar = smem_u32(&sh.t_full);
          const uint4 u = *reinterpret_cast<const uint4*>(sStage + n * 8);
          const uint32_t w[4] = {u.x, u.y, u.z, u.w};
#pragma unroll 1
          for (int c = 0; c < cj; ++c)
            st_async_u4(mapa_shared(to, (uint32_t)(row0 + c)), w, mapa_shared(bar, (uint32_t)(row0 + c)));
        }
        __syncwarp();
      }
      if (!mbar_wait_cluster(&sh.t_full, t_par)) product_failed(&sh, clusters == 1 ? cs : 1);
      t_par ^= 1u;
    } else if (cj > 1) {
      __syncwarp();
      cluster_sync_all();                                    // every CTA's partial T is in its shared memory
      const int n_groups = tb * (kBlock / 8), mine = (n_groups - j + cj - 1) / cj;      // token groups j, j + cj, ...
      // lane = (token of the group, half of a rank group): four ranks of a token, all sources in flight
#pragma unroll 1
      for (int e = tid; e < mine * 16 * groups; e += kThreads) {
        const int x = (e >> 1) & 7, kh = e & 1, og = e >> 4, o = og / groups, g = og - o * groups;
        const uint32_t src = smem_u32(sEx + ((size_t)g * tb * kBlock + (j + o * cj) * 8 + x) * 8 + 4 * kh);
        float4 z[8], sum = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
        for (int c = 0; c < 8; ++c)
          z[c] = c < cj ? ld_cluster_f4(mapa_shared(src, (uint32_t)(row0 + c))) : make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
        for (int c = 0; c < 8; ++c) { sum.x += z[c].x; sum.y += z[c].y; sum.z += z[c].z; sum.w += z[c].w; }
        const float v[4] = {sum.x, sum.y, sum.z, sum.w};
#pragma unroll
        for (int k = 0; k < 4; ++k) {
          __nv_bfloat16 part[PARTS];
          split1<PARTS>(v[k], part);
#pragma unroll
          for (int p = 0; p < PARTS; ++p) sStage[((size_t)o * PARTS * NP + p * NP + 8 * g + 4 * kh + k) * 8 + x] = part[p];
        }
      }
      __syncthreads();
      {                                                      // a warp per destination, pieces of eight tokens of an operand row
        const int c = warp % cj, first = lane + 32 * (warp / cj), step = 32 * (kWarps / cj);
        const uint32_t dst = mapa_shared(at, (uint32_t)(row0 + c));
#pragma unroll 1
        for (int o = 0; o < mine; ++o) {
          const int tg = j + o * cj;
          const uint32_t box = dst + (uint32_t)((tg >> 3) * NB * 128);
#pragma unroll 1
          for (int row = first; row < PARTS * NP; row += step)
            st_cluster_u4(box + swz(row, tg & 7), *reinterpret_cast<const uint4*>(sStage + ((size_t)o * PARTS * NP + row) * 8));
        }
      }
      __syncwarp();
      cluster_sync_all();                                    // the T operand is complete
    }
  }

  tc_fence_before();
  __syncwarp();
  if (cs > 1) cluster_sync_all(); else __syncthreads();      // nobody leaves while a peer may read its share
  if (sh.failed) {                                           // a wait has run out and the sums are not whole
    zero_strips(U, i, col0);
    if (PUSH) let_land();
  }
  if (tid == 0) {
    if (sh.failed && P.status) report_timeout(P.status, 5);
    if (i == 0 && j == 0) {
      if (P.status && sh.st.rank_deficient) atomicExch(&P.status->rank_deficient, 1);
      if (P.flag) *P.flag = sh.failed ? 2 : sh.st.rank_deficient;
    }
  }
  if (warp == 1) { tc_fence_after(); tmem_dealloc(tmem, ncol); }
}

using ResKernel = void (*)(const ResidentParams);
ResKernel res_kernel(int planes, int parts, bool push) {
  if (push) return planes == 3 ? resident_extract_kernel<3, 3, true> : parts == 3 ? resident_extract_kernel<1, 3, true> : resident_extract_kernel<1, 2, true>;
  return planes == 3 ? resident_extract_kernel<3, 3, false> : parts == 3 ? resident_extract_kernel<1, 3, false> : resident_extract_kernel<1, 2, false>;
}

// Warps of a layer's Gram products: all of them between the layers, fewer where their sums would not fit beside X
int gram_split(const ResidentUnit& u) { return u.n_layers == 1 ? (u.cb * u.tb >= 4 ? 4 : 8) : u.n_layers == 2 ? 4 : 2; }

// Shared memory of a CTA
size_t res_smem(const ResidentUnit& u, int planes, int parts) {
  const size_t x = (size_t)planes * u.tb * u.cb * 2 * kSlotBytes, ops = (size_t)std::max(u.cb, u.tb) * 2 * u.NB * 128;
  const size_t y = (size_t)u.rows * qr_pitch(u.cb * kBlock) * 4 + (size_t)u.n_layers * gram_split(u) * kShareElems * 8;
  const size_t own = (size_t)(u.tb * (kBlock / 8) + u.cj - 1) / u.cj;
  const size_t ex = u.cj == 1 ? 0 : (size_t)u.tb * kBlock * u.NP * 4 + own * parts * u.NP * 16;
  return x + ops + (size_t)u.n_layers * (kShareElems * 8 + kAmBytes) + std::max(y, ex) + 1024;
}

// ... of one that is sent what its cluster exchanges (sub is known by then)
size_t push_smem(const ResidentUnit& u, int planes, int parts, int cs) {
  const size_t x = (size_t)planes * u.tb * u.cb * 2 * kSlotBytes, ops = (size_t)std::max(u.cb, u.tb) * 2 * u.NB * 128;
  size_t share = 0;
  for (int l = 0; l < u.n_layers; ++l) share += u.layer[l].r <= 8 ? 64 : kShareElems;
  const size_t front = push_front(u.rows * qr_pitch(u.cb * kBlock) * 4, parts);
  const size_t part = (size_t)u.n_layers * gram_split(u) * kShareElems * 8, ex = u.cj == 1 ? 0 : (size_t)u.tb * kBlock * u.NP * 4;
  return x + ops + (u.sub ? cs : u.cj) * share * 8 + (size_t)u.n_layers * kAmBytes + front + std::max(part, ex) + 1024;
}

// One way to lay a unit out over clusters of cs CTAs, and what a round of it is estimated to take (us)
struct Shape {
  int cj, cb, tb, ni, clusters, sub;
  double cost;
};

// The estimate that puts layouts in order: what it picks takes 0.6 % longer than the best of the layouts that were measured beside it
// (geometric mean over 1236 units; a unit of several clusters pays most for meeting).
Shape shape_of(const ResidentUnit& u, int planes, int cs, int cj, int cb, int tb) {
  Shape s{cj, cb, tb, 0, 0, 0, 0.0};
  const int blocks_m = (u.m + kBlock - 1) / kBlock, per = cs / cj;
  s.ni = (blocks_m + tb - 1) / tb;
  s.clusters = (s.ni + per - 1) / per;
  double cycles = 0.0;                 // of a product's instructions for 16 of the contracted dimension, all planes of X
  for (int p = 0; p < planes; ++p) cycles += 32.0 + (double)(p == 0 ? u.NB : (3 - p) * u.NP) / 4.0;
  int groups = 0, rank = 0;
  for (int l = 0; l < u.n_layers; ++l) { groups += (u.layer[l].r + 7) / 8; rank = std::max(rank, u.layer[l].r); }
  s.cost = 1.3 + 2.6 * (2.0 * tb * cb * 8 * cycles / 1900.0) + (cj > 1 ? 1.1 : 0.0) + 0.54 * cb * groups + 0.41 * (cb + tb) * (u.NP / 8) +
           (rank > 4 ? 0.2 : 0.0) + (rank > 8 ? 1.4 : 0.0);
  if (s.ni > 1) {
    const double kb = (double)u.ranks * cb * kBlock * 4.0 / 60e3;      // a partial sum of the CTA's columns
    // all of the columns: five partial sums of 24 rows of 128 columns a trip to L2
    const double all = 0.45 * ((u.ranks * cb + 23) / 24) * ((s.ni + 4) / 5) + 0.1 * s.ni * kb, part = (s.clusters > 1 ? 3.2 : 1.2) + kb;
    s.cost += s.clusters > 1 ? 3.4 : 1.2;
    if (part < all) s.sub = ((cb * kBlock + s.ni - 1) / s.ni + 3) & ~3;
    s.cost += std::min(part, all);
  }
  return s;
}

// Shapes for all units on clusters of cs CTAs within the device's clusters: from the fewest clusters on, the slowest unit gets more.
bool lay_out(const std::vector<ResidentUnit>& units, int planes, int parts, int cs, int cap, std::vector<Shape>* out, double* slowest) {
  std::vector<std::vector<Shape>> ways(units.size());
  out->assign(units.size(), Shape{});
  int used = 0;
  for (size_t n = 0; n < units.size(); ++n) {
    ResidentUnit u = units[n];
    const int blocks_d = (u.d + kBlock - 1) / kBlock, blocks_m = (u.m + kBlock - 1) / kBlock;
    for (int cj = 1; cj <= cs; cj *= 2) {
      const int cb = (blocks_d + cj - 1) / cj;
      if (cj > 1 && cb == (blocks_d + cj / 2 - 1) / (cj / 2)) break;          // CTAs without columns
      for (int tb = 1; tb <= 8 && tb <= blocks_m && cb * tb <= 8; ++tb) {
        u.cj = cj; u.cb = cb; u.tb = tb;
        if ((parts == 3 ? 2 * cb * tb : std::max(cb, tb)) * u.NB > 512 || res_smem(u, planes, parts) > kMaxSmem) break;
        const Shape s = shape_of(u, planes, cs, cj, cb, tb);
        if (s.clusters <= cap) ways[n].push_back(s);
      }
    }
    if (ways[n].empty()) return false;
    const Shape* best = nullptr;
    for (const Shape& s : ways[n])
      if (!best || s.clusters < best->clusters || (s.clusters == best->clusters && s.cost < best->cost)) best = &s;
    (*out)[n] = *best;
    used += best->clusters;
    if (used > cap) return false;
  }
  for (;;) {
    size_t worst = 0;
    for (size_t n = 1; n < units.size(); ++n)
      if ((*out)[n].cost > (*out)[worst].cost) worst = n;
    const Shape* next = nullptr;
    for (const Shape& s : ways[worst])
      if (s.cost < (*out)[worst].cost - 0.05 && used - (*out)[worst].clusters + s.clusters <= cap &&
          (!next || s.clusters < next->clusters || (s.clusters == next->clusters && s.cost < next->cost)))
        next = &s;
    *slowest = (*out)[worst].cost;
    if (!next) return true;
    used += next->clusters - (*out)[worst].clusters;
    (*out)[worst] = *next;
  }
}

size_t up256(size_t x) { return (x + 255) / 256 * 256; }

bool same_x(const agzo_layer& a, const agzo_layer& b) {
  return a.X == b.X && a.ldx == b.ldx && a.m == b.m && a.d_in == b.d_in && a.x_dtype == b.x_dtype;
}

}  // namespace

cudaError_t resident_init(int sm_count, ResidentCaps* caps) {
  for (int k = 0; k < 6; ++k) {
    const void* f = (const void*)res_kernel(k % 3 == 2 ? 3 : 1, k % 3 == 0 ? 2 : 3, k >= 3);
    cudaError_t e = cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kMaxSmem);
    if (e != cudaSuccess) return e;
  }
  for (int cs = 1; cs <= 8; cs *= 2) {
    cudaLaunchConfig_t cfg{};
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = (unsigned)cs;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    cfg.gridDim = dim3((unsigned)(sm_count / cs * cs));
    cfg.blockDim = dim3(kThreads);
    cfg.dynamicSmemBytes = kMaxSmem;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    int n = 0;
    if (cudaOccupancyMaxActiveClusters(&n, (const void*)res_kernel(3, 3, true), &cfg) != cudaSuccess) { cudaGetLastError(); n = 0; }
    caps->clusters[cs] = n;
  }
  caps->sm_count = sm_count;
  return cudaSuccess;
}

bool resident_plan(const ResidentCaps& caps, const agzo_layer* L, int n, bool share_inputs, bool two_parts, ResidentLaunch* out) {
  if (caps.sm_count == 0 || n < 1) return false;
  const int planes = L[0].x_dtype == AGZO_F32 ? 3 : 1, parts = planes == 1 && two_parts ? 2 : 3;
  // what does not fit whatever the layout is refused before anything is laid out
  const size_t chip = (size_t)caps.sm_count * kMaxSmem;
  std::vector<ResidentUnit> units;
  size_t bytes = 0;
  for (int k = 0; k < n;) {
    const agzo_layer& a = L[k];
    ResidentUnit u{};
    u.X = a.X; u.ldx = a.ldx; u.m = a.m; u.d = a.d_in;
    const int per16 = a.x_dtype == AGZO_F32 ? 4 : 8;
    u.x_vec = (reinterpret_cast<uintptr_t>(a.X) & 15u) == 0 && a.ldx % per16 == 0 && a.d_in % per16 == 0;
    for (; k < n; ++k) {
      const agzo_layer& b = L[k];
      if (!b.X || b.m < 1 || b.r > kResMaxRank || (b.x_dtype == AGZO_F32 ? 3 : 1) != planes) return false;
      if (u.n_layers > 0 && (!share_inputs || !same_x(a, b))) break;
      if (u.ranks + b.r > kResMaxPanel || u.n_layers == kResMaxLayers) return false;
      u.layer[u.n_layers++] = ResidentLayer{b.V, b.ldv, b.layer_id, b.r, u.ranks, u.rows};
      u.ranks += b.r;
      u.rows += (b.r + 7) & ~7;
    }
    u.NP = (u.ranks + 7) & ~7;
    u.NB = (parts * u.NP + 15) & ~15;
    bytes += (size_t)((u.m + kBlock - 1) / kBlock) * ((u.d + kBlock - 1) / kBlock) * 2 * kSlotBytes * planes;
    if ((int)units.size() == kResMaxUnits || bytes > chip) return false;
    units.push_back(u);
  }
  std::vector<Shape> shapes, best;
  double slowest = 0.0, least = 0.0;
  int cs = 0;
  for (int c = 8; c >= 1; c /= 2)
    if (caps.clusters[c] > 0 && lay_out(units, planes, parts, c, caps.clusters[c], &shapes, &slowest) && (cs == 0 || slowest < least)) {
      cs = c; least = slowest; best = shapes;
    }
  if (cs == 0) return false;
  ResidentParams& p = out->p;
  p = ResidentParams{};
  p.n_units = (int)units.size();
  p.wait_ns = ptx::kWaitCapNs;
  p.cs = cs;
  out->planes = planes; out->parts = parts;
  out->n_clusters = 0; out->grid_wide = false; out->smem = 0;
  size_t sent = 0;
  int most_sent = 0, most_clusters = 0;
  bool wide = false;
  for (size_t k = 0; k < units.size(); ++k) {
    ResidentUnit& u = units[k];
    const Shape& s = best[k];
    u.cj = s.cj; u.cb = s.cb; u.tb = s.tb; u.ni = s.ni; u.sub = s.sub; u.gram_split = gram_split(u);
    u.clusters = s.clusters; u.cluster0 = out->n_clusters; u.counter = (int)k;
    out->n_clusters += s.clusters;
    out->grid_wide = out->grid_wide || s.clusters > 1;
    out->smem = std::max(out->smem, res_smem(u, planes, parts));
    sent = std::max(sent, push_smem(u, planes, parts, cs));
    wide = wide || (u.sub && u.clusters > 1);
    most_clusters = std::max(most_clusters, u.clusters);
    if (u.cj > 1) most_sent = std::max(most_sent, u.tb * u.NP * (16 * parts + 32));
    p.unit[k] = u;
  }
  // Kernel times of 196 lists, read from the peers -> sent.  Units of one cluster: all faster or even, by 6 % on the mean and up to 23 %
  // (613 x 280 and smaller; 3 x 128 tokens a CTA 40.1 -> 32.6 us).  Of several, which also meet at a counter: 3 % up to five clusters; from
  // six on 3 % while a CTA gets up to 1024 messages of 16 bytes for T (two parts: ranks up to 8 on 256 tokens, 16 on 128), beyond those
  // the receiver's counting of them takes what the barriers did (2560: 88.5 -> 91.1 us, 3840: 77.7 -> 82.3).  Where the clusters' shares
  // meet in global memory, the round trip is hidden behind that meeting already: 4096 x 2048, r = 16 84.0 -> 87.5.
  out->push = cs > 1 && !wide && sent <= kMaxSmem && (most_clusters <= 5 || most_sent <= 1024);
  if (out->push) out->smem = sent;
  resident_bind(out, nullptr);
  return true;
}

// ------------------------------------------------------------------ which kernels are the faster ones
// Both sides as K + 1 times what every round has, K times what only those with T = X Q have, and the rest.  Weighted least squares over
// 1800 units of one X and 230 lists of several, 32 to 8192 tokens, 32 to 4096 columns, one to four layers of ranks 1 to 16, K = 0, 1
// and 3, all types and alignments.  The resident kernel is estimated to 4.6 % rms, the others to 4 to 6 % (8 % element by element).
struct Rounds { double once, every, power; };

Rounds resident_rounds(const ResidentUnit& u, int planes, int parts) {
  int groups = 0, rank = 0;
  for (int l = 0; l < u.n_layers; ++l) { groups += (u.layer[l].r + 7) / 8; rank = std::max(rank, u.layer[l].r); }
  double cycles = 0.0;                 // of a product's instructions for 16 of the contracted dimension, all planes of X
  for (int p = 0; p < planes; ++p) cycles += 32.0 + (double)(p == 0 ? u.NB : (3 - p) * u.NP) / 4.0;
  const double blocks = u.tb * u.cb, panel = 0.01 * u.ranks * u.cb;
  Rounds t;
  t.once = (0.41 * planes + (u.x_vec ? 0.0 : 1.89)) * blocks;                    // X
  t.every = 1.2 + 3.1 * (8.0 * blocks * cycles / 1900.0) + 0.56 * u.cb * groups + (rank > 4 ? 0.84 : 0.0) + (rank > 8 ? 2.0 : 0.0) +
            0.53 * (u.n_layers - 1);
  if (u.ni > 1) t.every += 0.73;
  if (u.clusters > 1) t.every += 0.49;
  if (u.sub) t.every += (u.clusters > 1 ? 2.92 : 1.43) + 1.08 * panel;
  else if (u.ni > 1) t.every += 0.48 * ((u.ranks * u.cb + 23) / 24) * ((u.ni + 4) / 5) + 0.26 * u.ni * panel;
  t.power = 0.71 + (u.cj > 1 ? 2.35 : 0.0) + 0.39 * u.tb * (u.NP / 8) * (parts == 3 ? 1.5 * u.cb : 1.0);
  return t;
}
// The chain of launches, for the unit alone.  By kernels: tensor-core products, fp32 products on bf16 and on fp32 in 16- or 8-byte
// pieces, element by element.  m, d in thousands, md in millions; r4, r8: ranks above 4, 8; more: md per further layer on the X, which
// the fp32 products read once per layer.
struct ChainFit {
  double once;
  double every, every_r4, every_r8, every_m, every_d, every_md, every_r8_d, every_r8_md, every_more;
  double power, power_m, power_d, power_md, power_r4_d, power_r8_d, power_r8_md, power_more;
};
constexpr ChainFit kChain[3] = {
    {3.66, 4.37, 1.35, 3.82, 0.83, 0.39, 0.39, 0.0, 0.86, 0.54, 3.49, 0.45, 1.74, 0.0, 0.91, 4.58, 0.93, 0.50},
    {4.15, 4.19, 1.44, 3.46, 0.84, 0.36, 0.62, 0.0, 1.15, 0.93, 4.08, 0.33, 1.10, 0.0, 0.29, 2.68, 3.96, 0.66},
    {4.54, 8.34, 2.90, 6.87, 2.38, 0.98, 0.71, 0.39, 0.96, 1.49, 3.80, 0.79, 5.78, 0.22, 7.01, 10.14, 1.62, 2.26}};

Rounds other_rounds(const ResidentUnit& u, int planes, bool two_parts) {
  int rank = 0;
  for (int l = 0; l < u.n_layers; ++l) rank = std::max(rank, u.layer[l].r);
  const double m = 1e-3 * u.m, d = 1e-3 * u.d, md = m * d, r4 = rank > 4, r8 = rank > 8;
  if (two_parts) {
    const double group = u.n_layers > 1 ? md : 0.0;
    return Rounds{4.14, 4.55 + 0.66 * r4 + (2.12 + 0.41 * d) * r8 + 1.17 * m + 0.37 * d + 0.024 * u.ranks + 0.07 * group,
                  4.94 + 0.67 * d + 0.37 * md + 0.019 * u.ranks + 0.32 * group};
  }
  const bool in_pieces = u.d % 4 == 0 && u.ldx % 4 == 0 && (reinterpret_cast<uintptr_t>(u.X) & (planes == 3 ? 15u : 7u)) == 0;
  const ChainFit& f = kChain[!in_pieces ? 2 : planes == 3 ? 1 : 0];
  const double more = md * (u.n_layers - 1);
  return Rounds{f.once,
                f.every + f.every_r4 * r4 + f.every_r8 * r8 + f.every_m * m + f.every_d * d + f.every_md * md + (f.every_r8_d * d + f.every_r8_md * md) * r8 +
                    f.every_more * more,
                f.power + f.power_m * m + f.power_d * d + f.power_md * md + f.power_r4_d * d * r4 + (f.power_r8_d * d + f.power_r8_md * md) * r8 +
                    f.power_more * more};
}

// Over those lists the rule takes the slower kernels by more than 2 % for 1.6, 1.3 and 0.5 % of them (K = 0, 1, 3; at most 25, 8 and 6 %
// slower) and leaves 1 to 12 % of the logarithm of what the faster kernel each time would gain.  An estimate without the rounds apart,
// fitted before the partial sums of several column blocks were read together and without bf16 on the fp32 kernels: 23, 11 and 4.7 %.
bool resident_pays(const ResidentLaunch& plan, int K, bool fresh) {
  // Below 2^-109 an fp32 value's third part is no bf16 number any more.  With a power step such inputs underflow whatever the kernel,
  // without one the fp32 products keep them (2^-118 of N(0, 1): 5e-9 against 64 bits, the parts 9e-6): they stay there.
  if (K == 0 && plan.planes == 3) return false;
  double here = 0.0, there = 0.0, most = 0.0, all = 0.0;
  int layers = 0;
  for (int k = 0; k < plan.p.n_units; ++k) {
    const ResidentUnit& u = plan.p.unit[k];
    const Rounds a = resident_rounds(u, plan.planes, plan.parts), b = other_rounds(u, plan.planes, plan.parts == 2);
    const double md = 1e-6 * u.m * (double)u.d;
    here = std::max(here, a.once + (K + 1) * a.every + K * a.power);
    there = std::max(there, b.once + (K + 1) * b.every + K * b.power);
    most = std::max(most, md);
    all += md;
    layers += u.n_layers;
  }
  here += plan.grid_wide ? 8.43 : 5.65;
  if (plan.p.n_units > 1) {            // their launches serve all units, which share the SMs
    const bool two_parts = plan.parts == 2;
    const int more = std::min(layers - 1, 8);
    there += (two_parts ? 0.19 : plan.planes == 3 ? 0.74 : 0.59) * (2 * K + 1) * (all - most) + (two_parts ? 0.13 : plan.planes == 3 ? 0.09 : 0.18) * (K + 1) * more;
  }
  if (fresh) there += 1.3;
  return here < 0.97 * there;
}

void resident_bind(ResidentLaunch* plan, char* scratch) {
  size_t at = 0;
  auto take = [&](size_t bytes) { char* p = scratch ? scratch + at : nullptr; at += up256(bytes); return p; };
  for (int k = 0; k < plan->p.n_units; ++k) {
    ResidentUnit& u = plan->p.unit[k];
    const size_t panel = (size_t)u.ranks * u.cj * u.cb * kBlock * 4;
    if (u.ni > 1) u.ypart = reinterpret_cast<float*>(take(u.ni * panel * (u.sub ? 1 : 2)));
    if (u.sub) {
      u.y = reinterpret_cast<float*>(take(panel));
      u.gshare = reinterpret_cast<double*>(take((size_t)u.clusters * u.n_layers * kShareElems * 8));
    }
  }
  plan->scratch = at;
}

cudaError_t launch_resident(const ResidentLaunch& plan, cudaStream_t s) {
  cudaLaunchConfig_t cfg{};
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = (unsigned)plan.p.cs;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  if (plan.grid_wide) {                // its CTAs wait for one another: all resident at once, or no launch
    attr[1].id = cudaLaunchAttributeCooperative;
    attr[1].val.cooperative = 1;
  } else {
    attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[1].val.programmaticStreamSerializationAllowed = 1;
  }
  cfg.gridDim = dim3((unsigned)(plan.n_clusters * plan.p.cs));
  cfg.blockDim = dim3(kThreads);
  cfg.dynamicSmemBytes = plan.smem;
  cfg.stream = s;
  cfg.attrs = attr;
  cfg.numAttrs = 2;
  return cudaLaunchKernelEx(&cfg, res_kernel(plan.planes, plan.parts, plan.push), plan.p);
}

bool resident_refused(cudaError_t e) {
  if (e != cudaErrorCooperativeLaunchTooLarge && e != cudaErrorLaunchOutOfResources && e != cudaErrorNotSupported) return false;
  cudaGetLastError();
  return true;
}

}  // namespace agzo

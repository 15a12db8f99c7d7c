// qr(Y) of Algorithm 1 for the panels of a wave: Q = Y R^-1 with the unique R that has a positive diagonal
// (S = Y^T Y = R^T R).  With the Gram matrix and the factor in double this is as accurate in fp32 as a Householder QR
// for cond(Y) well below 1e7.
//
// Up to rank 32 (panel_qr_kernel) one launch per round, a thread-block cluster of C CTAs per layer, CTA c owning a
// contiguous slice of the columns d of Y (r x d_in):
//   load    Y = sum of the partial sums that the last product left, in order, into shared memory
//   gram    the slice's share of S on the FP64 tensor cores (mma.sync m8n8k4: true double multiply-adds; tcgen05
//           has no FP64 form), the warps splitting the columns, partial sums added in a fixed order
//   -- every CTA sends its share to all (st.async, counted on the receiver's barrier) and adds the C shares in rank order; above rank 16,
//      or where shared memory has no room for them, they are read from the peers after a cluster barrier --
//   factor  Cholesky and M = R^-1, by every CTA for itself (what it costs is a dependent chain, so doing it C
//           times takes no longer than doing it once and saves a second exchange)
//   apply   Q = Y M on the FP64 tensor cores, from the slice that is still in shared memory, and out: V (fp32) after
//           the last round, the bf16 hi/lo operand panel of the next product before it
// What bounds it is the latency of that chain (load, gram, exchange, r pivots).  The three kernels it replaced (Gram per
// 512 columns, one factorisation block per layer, apply per 128 columns) handed Y, the Gram shares and M over through
// global memory: r = 8, d_in = 1024, one layer 24 -> 10.3 us per round; r = 16, d_in = 4096 44 -> 20 us.
//
// Above rank 32 the FP64 products (r^2 d_in multiply-adds each) weigh more than the chain and layers of a wave differ
// in d_in, so three launches cut the work evenly: Gram per 512 columns, factorisation per layer, apply per 128 columns.
#include "agzo_qr.cuh"

namespace agzo {

namespace {

using namespace qr;
using namespace ptx;

// Q of columns [d0, d0 + ncols) out: V rows (fp32) and / or the bf16 hi/lo rows of the next product's operand
__device__ __forceinline__ void qr_store(const DevLayer& L, const float* sY, int pitch, int d0, int ncols, bool to_v, bool to_qb) {
  const int r = L.r, d_in = L.d_in;
  const int rows = to_qb ? L.prow_n : r;
  __nv_bfloat16* hi_rows = L.Qb + (long long)L.grp_off * d_in;
  __nv_bfloat16* lo_rows = hi_rows + (long long)L.NP * d_in;
  if ((d_in & 3) == 0 && (L.ldv & 3) == 0 && (reinterpret_cast<uintptr_t>(L.V) & 15u) == 0) {
    const int vrow = ncols >> 2;
    for (int i = threadIdx.x; i < rows * vrow; i += kQrThreads) {
      const int k = i / vrow, c = 4 * (i - k * vrow), d = d0 + c;
      if (d >= d_in) continue;
      const float4 q = k < r ? *reinterpret_cast<const float4*>(sY + k * pitch + c) : make_float4(0.f, 0.f, 0.f, 0.f);
      if (to_v && k < r) *reinterpret_cast<float4*>(L.V + (long long)k * L.ldv + d) = q;
      if (to_qb) {
        const __nv_bfloat162 h0 = __floats2bfloat162_rn(q.x, q.y), h1 = __floats2bfloat162_rn(q.z, q.w);
        const __nv_bfloat162 l0 = __floats2bfloat162_rn(q.x - __low2float(h0), q.y - __high2float(h0));
        const __nv_bfloat162 l1 = __floats2bfloat162_rn(q.z - __low2float(h1), q.w - __high2float(h1));
        uint2 h, l;
        h.x = *reinterpret_cast<const uint32_t*>(&h0); h.y = *reinterpret_cast<const uint32_t*>(&h1);
        l.x = *reinterpret_cast<const uint32_t*>(&l0); l.y = *reinterpret_cast<const uint32_t*>(&l1);
        *reinterpret_cast<uint2*>(hi_rows + (long long)k * d_in + d) = h;
        *reinterpret_cast<uint2*>(lo_rows + (long long)k * d_in + d) = l;
      }
    }
  } else {
    for (int i = threadIdx.x; i < rows * ncols; i += kQrThreads) {
      const int k = i / ncols, c = i - k * ncols, d = d0 + c;
      if (d >= d_in) continue;
      const float q = k < r ? sY[k * pitch + c] : 0.f;
      if (to_v && k < r) L.V[(long long)k * L.ldv + d] = q;
      if (to_qb) {
        const __nv_bfloat16 hi = __float2bfloat16_rn(q);
        hi_rows[(long long)k * d_in + d] = hi;
        lo_rows[(long long)k * d_in + d] = __float2bfloat16_rn(q - __bfloat162float(hi));
      }
    }
  }
}

// A wait for what the peers send has run out: known to all C CTAs of the cluster, and to the round that stores V
__device__ __noinline__ void qr_wait_failed(int* failed, int C, DevStatus* status) {
  if ((threadIdx.x & 31) == 0 && atomicExch(failed, 1) == 0) report_timeout(status, 8);
  if ((int)(threadIdx.x & 31) < C) st_cluster_u32(mapa_shared(smem_u32(failed), threadIdx.x & 31u), 1u);
}
// V = 0 in columns [d0, d0 + ncols)
__device__ __noinline__ void qr_zero(const DevLayer& L, int d0, int ncols) {
  for (int i = threadIdx.x; i < L.r * ncols; i += kQrThreads) {
    const int k = i / ncols, d = d0 + i - k * ncols;
    if (d < L.d_in) L.V[(long long)k * L.ldv + d] = 0.f;
  }
}

// kResident: the CTA's whole slice stays in shared memory from load to apply; otherwise it is staged 128 columns at
// a time and read a second time (from L.Y, through L2) for the apply.
template <int NT, bool kResident, int kLive, bool kSend>
__global__ void __launch_bounds__(kQrThreads, 2) panel_qr_kernel(const DevLayer* __restrict__ layers, int l0, int C, int pitch,
                                                                 int y_reduced, int after_fused, int last, unsigned* published,
                                                                 DevStatus* status, int region, unsigned wait_ns, unsigned missing) {
  static_assert(NT <= 4, "larger ranks take the three launches");
  using Cfg = QrCfg<NT>;
  // the layer's record comes into shared memory before the wait: read in place, each of its lines would cost the chain a
  // trip to L2 where it is first touched
  __shared__ __align__(16) unsigned char record[sizeof(DevLayer)];
  static_assert(sizeof(DevLayer) % 8 == 0, "copied in words of eight bytes");
  for (int i = threadIdx.x; i < (int)(sizeof(DevLayer) / 8); i += kQrThreads)
    reinterpret_cast<unsigned long long*>(record)[i] =
        __ldcg(reinterpret_cast<const unsigned long long*>(layers + l0 + (int)blockIdx.x / C) + i);
  __shared__ uint64_t shares_in;
  __shared__ int failed;                 // a wait of this wave has run out
  if (threadIdx.x == 0) {
    failed = 0;
    if (kSend) {
      mbar_init(&shares_in, 1);
      asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
  }
  __syncthreads();
  if (kSend) asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");        // my barrier can be sent to
  const DevLayer& L = *reinterpret_cast<const DevLayer*>(record);
  const int rank = (int)cluster_ctarank();
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  extern __shared__ __align__(16) unsigned char qr_smem[];
  double* sU = reinterpret_cast<double*>(qr_smem);                       // warps' partial sums, then S / R and M
  double* sG = reinterpret_cast<double*>(qr_smem + Cfg::u_bytes);        // this CTA's share of S, [tile][8][8]
  float* sY = reinterpret_cast<float*>(qr_smem + Cfg::fixed);            // [r8][pitch]
  double* sIn = reinterpret_cast<double*>(qr_smem + Cfg::fixed + (size_t)Cfg::r8 * pitch * sizeof(float));      // kSend: the C shares
  double* A = sU;
  double* M = sU + Cfg::r8 * Cfg::ap;
  __shared__ double own[AGZO_MAX_RANK];
  const int r = L.r, nparts = y_parts(L, after_fused);
  const int cpc = (L.gchunks + C - 1) / C;
  const int ch0 = rank * cpc, nch = max(0, min(cpc, L.gchunks - ch0));
  const int d0 = ch0 * kQrChunk;

  chain_wait();
  if (!last && short_launch()) chain_next();
  if (published && blockIdx.x == 0 && tid == 0) *published = 0u;
  int timeouts = 0, before = 0;          // asked for here, compared behind the Gram products
  if (last && tid == 0) { timeouts = __ldcg(&status->timeout); before = __ldcg(&status->before[region]); }
  double acc[Cfg::my_tiles][2];
#pragma unroll
  for (int t = 0; t < Cfg::my_tiles; ++t) acc[t][0] = acc[t][1] = 0.0;
  if (kResident) {
    qr_load(L, sY, pitch, Cfg::r8, d0, nch * kQrChunk, nparts, y_reduced != 0, false);
    __syncthreads();
    qr_gram<NT, 0>(sY, pitch, nch * kQrChunk / 4, warp, acc);
  } else {
    for (int ch = 0; ch < nch; ++ch) {
      __syncthreads();
      qr_load(L, sY, pitch, Cfg::r8, d0 + ch * kQrChunk, kQrChunk, nparts, y_reduced != 0, y_reduced == 0);
      __syncthreads();
      qr_gram<NT, 0>(sY, pitch, kQrChunk / 4, warp, acc);
    }
  }
  // the warps' sums into this CTA's share of S, in warp order; fragment element (l / 4, 2 (l % 4) + x) of a tile
  const int el = (lane >> 2) * 8 + 2 * (lane & 3);
#pragma unroll
  for (int t = 0; t < Cfg::tiles; ++t)
    *reinterpret_cast<double2*>(sU + (warp * Cfg::tiles + t) * 64 + el) = make_double2(acc[t][0], acc[t][1]);
  if (timeouts != before) failed = 1;
  __syncthreads();
  auto place = [&](int i, double v) {
    int t = i >> 6, bi = 0;
    while (t >= NT - bi) { t -= NT - bi; ++bi; }
    const int row = 8 * bi + ((i & 63) >> 3), col = 8 * (bi + t) + (i & 7);
    A[row * Cfg::ap + col] = v;
    if (row == col) own[row] = v;
  };
  if constexpr (kSend) {
    constexpr int kPairs = Cfg::tiles * 32;
    static_assert(kPairs <= kQrThreads, "two elements a thread");
    __syncwarp();
    asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
    if (tid == 0) mbar_expect_tx(&shares_in, (uint32_t)(C * Cfg::tiles * 64 * 8) + missing);
    if (tid < kPairs) {
      double2 sum = make_double2(0.0, 0.0);
#pragma unroll
      for (int w = 0; w < kQrWarps; ++w) {
        const double2 v = *reinterpret_cast<const double2*>(sU + w * Cfg::tiles * 64 + 2 * tid);
        sum.x += v.x;
        sum.y += v.y;
      }
      const uint32_t to = smem_u32(sIn + rank * Cfg::tiles * 64 + 2 * tid), bar = smem_u32(&shares_in);
      const uint32_t w[4] = {(uint32_t)__double2loint(sum.x), (uint32_t)__double2hiint(sum.x), (uint32_t)__double2loint(sum.y),
                             (uint32_t)__double2hiint(sum.y)};
#pragma unroll 4
      for (int c = 0; c < C; ++c) st_async_u4(mapa_shared(to, (uint32_t)c), w, mapa_shared(bar, (uint32_t)c));
    }
    __syncthreads();                        // the warps' sums are read: S takes their place
    if (!mbar_wait_cluster_warp(&shares_in, 0, wait_ns)) qr_wait_failed(&failed, C, status);
    if (tid < kPairs) {
      double2 v[kQrMaxCluster], sum = make_double2(0.0, 0.0);
#pragma unroll
      for (int c = 0; c < kQrMaxCluster; ++c)
        v[c] = c < C ? *reinterpret_cast<const double2*>(sIn + c * Cfg::tiles * 64 + 2 * tid) : make_double2(0.0, 0.0);
#pragma unroll
      for (int c = 0; c < kQrMaxCluster; ++c) { sum.x += v[c].x; sum.y += v[c].y; }
      place(2 * tid, sum.x);
      place(2 * tid + 1, sum.y);
    }
  } else {
    for (int i = tid; i < Cfg::tiles * 64; i += kQrThreads) {
      double s = 0.0;
#pragma unroll
      for (int w = 0; w < kQrWarps; ++w) s += sU[w * Cfg::tiles * 64 + i];
      sG[i] = s;
    }
    __syncwarp();
    cluster_sync_all();                       // every CTA's share is in its shared memory
    for (int i = tid; i < Cfg::tiles * 64; i += kQrThreads) {
      double v[kQrMaxCluster], sum = 0.0;
#pragma unroll
      for (int c = 0; c < kQrMaxCluster; ++c) v[c] = c < C ? ld_cluster_f64(mapa_shared(smem_u32(sG + i), (uint32_t)c)) : 0.0;
#pragma unroll
      for (int c = 0; c < kQrMaxCluster; ++c) sum += v[c];
      place(i, sum);
    }
  }
  __syncthreads();
  asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");   // done with the peers' shares, or they have come
  qr_factor<NT, kLive>(A, M, own, r, status, rank == 0);

  const bool to_v = last || !L.Qb, to_qb = !last && L.Qb;
  if (kResident) {
    qr_apply<NT>(sY, pitch, M, nch * kQrChunk);
    __syncthreads();
    qr_store(L, sY, pitch, d0, nch * kQrChunk, to_v, to_qb);
  } else {
    for (int ch = 0; ch < nch; ++ch) {
      __syncthreads();
      qr_load(L, sY, pitch, Cfg::r8, d0 + ch * kQrChunk, kQrChunk, nparts, true, false);
      __syncthreads();
      qr_apply<NT>(sY, pitch, M, kQrChunk);
      __syncthreads();
      qr_store(L, sY, pitch, d0 + ch * kQrChunk, kQrChunk, to_v, to_qb);
    }
  }
  __syncwarp();
  asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");   // nobody leaves while a peer may read its share
  if (failed) {
    if (last) qr_zero(L, d0, nch * kQrChunk);
    if (kSend) let_land();
  }
}

// ------------------------------------------------------------------ ranks above 32: three launches
constexpr int kGramGroup = 4;            // 128-column chunks per CTA of the Gram launch

// In global memory a share of S is the nt (nt + 1) / 2 tiles of the layer's own rank (nt = r / 8, rounded up), row by
// row; M, once it is known, takes the place of the first share.
__host__ __device__ inline int qr_share_elems(int r) { const int nt = (r + 7) >> 3; return nt * (nt + 1) / 2 * 64; }
__device__ __forceinline__ void qr_tile_of(int t, int nt, int* bi, int* bj) {
  int b = 0;
  while (t >= nt - b) { t -= nt - b; ++b; }
  *bi = b; *bj = b + t;
}

// Gram share of up to 512 columns of a layer, and their Y = sum of the partial sums.  Two warps split the columns of
// each of the four tile sets; a scheduler's two warps have 18 tiles between them.
__global__ void __launch_bounds__(kQrThreads, 2) panel_gram_kernel(const DevLayer* __restrict__ layers, int l0, int y_reduced,
                                                                   int after_fused) {
  using Cfg = QrCfg<8>;
  const DevLayer& L = layers[l0 + blockIdx.y];
  chain_wait();
  if (short_launch()) chain_next();
  const int ch0 = blockIdx.x * kGramGroup;
  if (ch0 >= L.gchunks) return;
  const int nch = min(kGramGroup, L.gchunks - ch0), nparts = y_parts(L, after_fused);
  extern __shared__ __align__(16) unsigned char qr_smem[];
  float* sY = reinterpret_cast<float*>(qr_smem);           // [64][pitch], then the share of S
  const int pitch = qr_pitch(kQrChunk);
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int set = (warp + 2 * (warp >> 2)) & 3, turn0 = warp >> 2;
  double acc[Cfg::my_tiles][2];
#pragma unroll
  for (int t = 0; t < Cfg::my_tiles; ++t) acc[t][0] = acc[t][1] = 0.0;
  for (int ch = 0; ch < nch; ++ch) {
    __syncthreads();
    qr_load(L, sY, pitch, Cfg::r8, (ch0 + ch) * kQrChunk, kQrChunk, nparts, y_reduced != 0, y_reduced == 0);
    __syncthreads();
    if (set == 0) qr_gram<8, 0>(sY, pitch, kQrChunk / 4, turn0, acc);
    else if (set == 1) qr_gram<8, 1>(sY, pitch, kQrChunk / 4, turn0, acc);
    else if (set == 2) qr_gram<8, 2>(sY, pitch, kQrChunk / 4, turn0, acc);
    else qr_gram<8, 3>(sY, pitch, kQrChunk / 4, turn0, acc);
  }
  static_assert(Cfg::g_bytes <= (size_t)Cfg::r8 * (kQrChunk + 12) * 4, "the share of S fits the staging buffer");
  double* sG = reinterpret_cast<double*>(qr_smem);
  const int el = (lane >> 2) * 8 + 2 * (lane & 3);
  __syncthreads();                        // the staged columns have been used: their place takes the sums
  for (int turn = 0; turn < Cfg::ksplit; ++turn) {
    if (turn0 == turn) {
      if (set == 0) qr_add_share<8, 0>(sG + el, acc, turn == 0);
      else if (set == 1) qr_add_share<8, 1>(sG + el, acc, turn == 0);
      else if (set == 2) qr_add_share<8, 2>(sG + el, acc, turn == 0);
      else qr_add_share<8, 3>(sG + el, acc, turn == 0);
    }
    __syncthreads();
  }
  const int nt = (L.r + 7) >> 3, n2 = qr_share_elems(L.r) / 2;
  double2* out = reinterpret_cast<double2*>(L.Gpart) + (size_t)blockIdx.x * n2;
  for (int i = tid; i < n2; i += kQrThreads) {
    int bi, bj;
    qr_tile_of(i >> 5, nt, &bi, &bj);
    out[i] = reinterpret_cast<const double2*>(sG)[(bi * 8 - bi * (bi - 1) / 2 + bj - bi) * 32 + (i & 31)];
  }
}

// One CTA per layer: S = sum of its shares in order, factorisation, M out
__global__ void __launch_bounds__(kQrThreads) panel_factor_kernel(const DevLayer* __restrict__ layers, int l0, DevStatus* status) {
  using Cfg = QrCfg<8>;
  const DevLayer& L = layers[l0 + blockIdx.x];
  extern __shared__ __align__(16) unsigned char qr_smem[];
  double* A = reinterpret_cast<double*>(qr_smem);
  double* M = A + Cfg::r8 * Cfg::ap;
  __shared__ double own[AGZO_MAX_RANK];
  const int tid = threadIdx.x, r = L.r;
  chain_wait();
  if (short_launch()) chain_next();
  const int nsh = (L.gchunks + kGramGroup - 1) / kGramGroup;
  const int nt = (r + 7) >> 3, ne = qr_share_elems(r);
  constexpr int kPer = (Cfg::tiles * 64 + kQrThreads - 1) / kQrThreads;
  double sum[kPer];
#pragma unroll
  for (int u = 0; u < kPer; ++u) sum[u] = 0.0;
  for (int s0 = 0; s0 < nsh; s0 += 2) {
    double v[2][kPer];
#pragma unroll
    for (int s = 0; s < 2; ++s)
#pragma unroll
      for (int u = 0; u < kPer; ++u) {
        const int i = tid + u * kQrThreads;
        v[s][u] = s0 + s < nsh && i < ne ? __ldcg(L.Gpart + (size_t)(s0 + s) * ne + i) : 0.0;
      }
#pragma unroll
    for (int s = 0; s < 2; ++s)
#pragma unroll
      for (int u = 0; u < kPer; ++u) sum[u] += v[s][u];
  }
#pragma unroll
  for (int u = 0; u < kPer; ++u) {
    const int i = tid + u * kQrThreads;
    if (i >= ne) break;
    int bi, bj;
    qr_tile_of(i >> 6, nt, &bi, &bj);
    const int row = 8 * bi + ((i & 63) >> 3), col = 8 * bj + (i & 7);
    A[row * Cfg::ap + col] = sum[u];
    if (row == col) own[row] = sum[u];
  }
  __syncthreads();
  qr_factor<8>(A, M, own, r, status, true);
  for (int i = tid; i < ne; i += kQrThreads) {
    int bi, bj;
    qr_tile_of(i >> 6, nt, &bi, &bj);
    L.Gpart[i] = M[(8 * bi + ((i & 63) >> 3)) * Cfg::mp + 8 * bj + (i & 7)];
  }
}

// Q = Y M on 128 columns of a layer
__global__ void __launch_bounds__(kQrThreads, 2) panel_apply_kernel(const DevLayer* __restrict__ layers, int l0, int last,
                                                                    unsigned* published, const DevStatus* status, int region) {
  using Cfg = QrCfg<8>;
  const DevLayer& L = layers[l0 + blockIdx.y];
  const int d0 = blockIdx.x * kQrChunk;
  chain_wait();
  if (!last && short_launch()) chain_next();
  if (published && blockIdx.x == 0 && blockIdx.y == 0 && threadIdx.x == 0) *published = 0u;
  if (d0 >= L.d_in) return;
  const bool failed = last && wave_failed(status, region);
  extern __shared__ __align__(16) unsigned char qr_smem[];
  double* M = reinterpret_cast<double*>(qr_smem);
  float* sY = reinterpret_cast<float*>(M + Cfg::r8 * Cfg::mp);
  const int pitch = qr_pitch(kQrChunk);
  for (int i = threadIdx.x; i < Cfg::r8 * Cfg::mp; i += kQrThreads) M[i] = 0.0;   // tiles below the diagonal, rows beyond r
  __syncthreads();
  const int nt = (L.r + 7) >> 3, n2 = qr_share_elems(L.r) / 2;
  constexpr int kPer = (Cfg::tiles * 32 + kQrThreads - 1) / kQrThreads;
  double2 v[kPer];
#pragma unroll
  for (int u = 0; u < kPer; ++u) {
    const int i = threadIdx.x + u * kQrThreads;
    v[u] = i < n2 ? __ldcg(reinterpret_cast<const double2*>(L.Gpart) + i) : make_double2(0.0, 0.0);
  }
#pragma unroll
  for (int u = 0; u < kPer; ++u) {
    const int i = threadIdx.x + u * kQrThreads;
    if (i >= n2) break;
    int bi, bj;
    qr_tile_of(i >> 5, nt, &bi, &bj);
    *reinterpret_cast<double2*>(M + (8 * bi + ((i & 31) >> 2)) * Cfg::mp + 8 * bj + 2 * (i & 3)) = v[u];
  }
  qr_load(L, sY, pitch, Cfg::r8, d0, kQrChunk, 1, true, false);
  __syncthreads();
  qr_apply<8>(sY, pitch, M, kQrChunk);
  __syncthreads();
  if (failed) qr_zero(L, d0, kQrChunk); else qr_store(L, sY, pitch, d0, kQrChunk, last || !L.Qb, !last && L.Qb);
}

// The extraction's last round takes back the number of its last power step (DevStatus::panel_ready): a replayed graph gives the
// same numbers again and must not find its own there from the replay before.
unsigned* published_at(const ExtractWave& w, bool last, DevStatus* d_status) { return last ? d_status->panel_ready + w.region : nullptr; }

// CTAs per layer: eight, for up to eight layers sixteen, while the launch is a chain of latencies (two 8B-shaped blocks from
// hooks, one group per launch: 3000 -> 2848 us per iteration with sixteen); with so many layers that eight each would queue for
// the SMs (two CTAs each), four or two, since every CTA repeats the factorisation (r = 8, d_in = 2048, 196 layers: 44.5 /
// 27.7 / 26.1 us with 8 / 4 / 2; r = 16, d_in = 4096, 70 layers: 43.5 / 28.3 / 55.1 us; 35 layers 28.7 / 27.4 / 51.5), but
// never so few that the widest layer's slice leaves shared memory where eight would keep it (the 55 us above).
template <int NT>
size_t qr_smem(int slice) { return QrCfg<NT>::fixed + (size_t)QrCfg<NT>::r8 * qr_pitch(slice) * sizeof(float); }

template <int NT, int kLive = kBlk>
cudaError_t launch_qr(const ExtractWave& w, bool last, DevStatus* d_status, cudaStream_t s) {
  const int nl = w.l1 - w.l0;
  auto slice_of = [&](int c) { return (w.max_gchunks + c - 1) / c * kQrChunk; };
  int C = nl <= 8 && w.qr_wide ? 16 : nl <= 40 ? 8 : nl <= 80 ? 4 : 2;
  while (C < 8 && qr_smem<NT>(slice_of(C)) > kQrResidentSmem) C *= 2;
  if (C > w.max_gchunks) C = w.max_gchunks;
  const bool resident = qr_smem<NT>(slice_of(C)) <= kQrResidentSmem;
  const int slice = resident ? slice_of(C) : kQrChunk;
  size_t smem = qr_smem<NT>(slice);
  auto* kernel = resident ? panel_qr_kernel<NT, true, kLive, false> : panel_qr_kernel<NT, false, kLive, false>;
  // Sending (up to rank 16, whose C shares are 24 KB at most) leaves out a barrier's wait and a round trip: 120 lists 0.5 % on the mean, eight
  // 1024 x 1024 layers, r = 8 141.9 -> 139.5 us, two 8B-shaped blocks from hooks 2806 -> 2789.
  if constexpr (NT <= 2)
    if (smem + C * QrCfg<NT>::g_bytes <= kQrResidentSmem) {
      smem += C * QrCfg<NT>::g_bytes;
      kernel = resident ? panel_qr_kernel<NT, true, kLive, true> : panel_qr_kernel<NT, false, kLive, true>;
    }
  return launch_chained(kernel, dim3((unsigned)(C * nl)), kQrThreads, smem, C, s, w.d_layers, w.l0, C, qr_pitch(slice), w.y_reduced,
                        w.after_fused, last ? 1 : 0, published_at(w, last, d_status), d_status, w.region, w.missing ? kMissingWaitNs : (unsigned)kWaitCapNs,
                        w.missing ? 1u : 0u);
}

constexpr size_t kGramSmem = (size_t)64 * (kQrChunk + 12) * sizeof(float);
constexpr size_t kFactorSmem = QrCfg<8>::am_bytes;
constexpr size_t kApplySmem = (size_t)64 * QrCfg<8>::mp * sizeof(double) + kGramSmem;

cudaError_t launch_qr_large(const ExtractWave& w, bool last, DevStatus* d_status, cudaStream_t s) {
  const unsigned nl = (unsigned)(w.l1 - w.l0);
  cudaError_t e = launch_chained(panel_gram_kernel, dim3((unsigned)((w.max_gchunks + kGramGroup - 1) / kGramGroup), nl), kQrThreads,
                                 kGramSmem, 0, s, w.d_layers, w.l0, w.y_reduced, w.after_fused);
  if (e == cudaSuccess) e = launch_chained(panel_factor_kernel, dim3(nl), kQrThreads, kFactorSmem, 0, s, w.d_layers, w.l0, d_status);
  if (e == cudaSuccess)
    e = launch_chained(panel_apply_kernel, dim3((unsigned)w.max_gchunks, nl), kQrThreads, kApplySmem, 0, s, w.d_layers, w.l0,
                       last ? 1 : 0, published_at(w, last, d_status), d_status, w.region);
  return e;
}

template <typename K>
cudaError_t allow_smem(K* kernel, size_t bytes) {
  return cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
}
template <typename K>
bool allow_wide(K* kernel) {
  if (cudaFuncSetAttribute(kernel, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) != cudaSuccess) return false;
  cudaLaunchConfig_t cfg{};
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = 16;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  cfg.gridDim = dim3(16);
  cfg.blockDim = dim3(kQrThreads);
  cfg.dynamicSmemBytes = kQrResidentSmem;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  int n = 0;
  return cudaOccupancyMaxActiveClusters(&n, kernel, &cfg) == cudaSuccess && n > 0;
}

}  // namespace

cudaError_t panel_qr_init(bool* wide) {
  cudaError_t e = cudaSuccess;
  *wide = true;
  auto allow = [&](auto* kernel) {
    if (e == cudaSuccess) e = allow_smem(kernel, kQrResidentSmem);
    *wide = *wide && allow_wide(kernel);
  };
  allow(panel_qr_kernel<1, true, 4, false>); allow(panel_qr_kernel<1, false, 4, false>); allow(panel_qr_kernel<1, true, kBlk, false>);
  allow(panel_qr_kernel<1, false, kBlk, false>); allow(panel_qr_kernel<2, true, kBlk, false>); allow(panel_qr_kernel<2, false, kBlk, false>);
  allow(panel_qr_kernel<4, true, kBlk, false>); allow(panel_qr_kernel<4, false, kBlk, false>);
  allow(panel_qr_kernel<1, true, 4, true>); allow(panel_qr_kernel<1, false, 4, true>); allow(panel_qr_kernel<1, true, kBlk, true>);
  allow(panel_qr_kernel<1, false, kBlk, true>); allow(panel_qr_kernel<2, true, kBlk, true>); allow(panel_qr_kernel<2, false, kBlk, true>);
  cudaGetLastError();
  if (e == cudaSuccess) e = allow_smem(panel_factor_kernel, kFactorSmem);
  if (e == cudaSuccess) e = allow_smem(panel_apply_kernel, kApplySmem);
  return e;
}

int panel_qr_launches(int max_r) { return max_r > 32 ? 3 : 1; }

// Scratch of a layer for the three-launch form, which a wave with a larger rank takes for all its layers
size_t panel_gram_bytes(int d_in, int r, int max_r) {
  if (panel_qr_launches(max_r) == 1) return 0;
  const size_t groups = (size_t)((d_in + kGramGroup * kQrChunk - 1) / (kGramGroup * kQrChunk));
  return groups * qr_share_elems(r) * sizeof(double);
}

cudaError_t launch_panel_qr(const ExtractWave& w, bool last, DevStatus* d_status, cudaStream_t s) {
  if (w.max_r <= 4) return launch_qr<1, 4>(w, last, d_status, s);
  if (w.max_r <= 8) return launch_qr<1>(w, last, d_status, s);
  if (w.max_r <= 16) return launch_qr<2>(w, last, d_status, s);
  if (w.max_r <= 32) return launch_qr<4>(w, last, d_status, s);
  return launch_qr_large(w, last, d_status, s);
}

}  // namespace agzo

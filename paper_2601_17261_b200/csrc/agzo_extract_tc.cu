// Tensor-core path of Algorithm 1's two products with X on sm_100a: TMA-fed shared-memory
// tiles, tcgen05.mma with fp32 accumulators in TMEM, one elected thread issuing.
//
//   x_q :  T  = H^T Q = X Q        M = 128 tokens, N = NB, K = d_in   (A = X tile, K-major)
//   xt_t:  Y  = H T   = X^T T      M = 128 columns of X, N = NB, K = tokens
//                                  (A = the same kind of X tile read as an MN-major operand)
//
// X is bf16 and exact; Q and T are fp32 quantities, so each is split as hi + lo in bf16 and
// the two parts sit side by side as extra N columns (N = NB = 2*NP, NP = r rounded up to 8):
// the products are exact, the accumulation is fp32, and the column groups are summed in the
// epilogue.  The kernels are HBM-bound (about r flop per byte of X), so the doubled N is free.
//
// Operand panels: Qb [NB][d_in] bf16 (written by the panel-QR apply kernel) and
// Tt [NB][m_pad] bf16 (T transposed; written by x_q's epilogue or by the Omega fill), both
// K-major B operands.  Every wait on an mbarrier is bounded; a wait that runs out sets the
// status word and the CTA leaves through the common exit (TMEM freed).
#include <cuda.h>

#include <cstring>

#include "agzo_ptx.cuh"
#include "agzo_tc.cuh"

namespace agzo {

namespace {

using namespace ptx;

// Threads of a CTA that works on MB blocks of 128 rows: warp 0 TMA producer, warp 1 MMA issuer, then four epilogue warps
// per block.
constexpr int tc_threads(int mb) { return 64 + 128 * mb; }
constexpr int kBoxK = 64;              // elements per 128-byte swizzle row
constexpr int kTileBytes = 64 * kBoxK * 2;   // one [64 rows][64 elems] bf16 box = 8 KiB
constexpr size_t kMinSmem = 80 * 1024;  // keeps at most 2 CTAs per SM: 2 * 256 TMEM columns fit

// One block per CTA (two CTAs per SM) while the operand panel is small.  A panel of NB rows is fetched through L2 once per
// block of X, NB / 128 bytes per byte of X; from about one byte per byte on, the path from L2 into the SMs is what the
// sweep waits for (r = 64, q + k in one panel of 256 rows: 5.1 TB/s of X, 11.7 TB/s into the SMs).  Two blocks per CTA (one
// CTA per SM) then share each fetch.  Extraction, one / two blocks: four 8B-shaped blocks with shared inputs r = 24 4174 / 3751 us,
// r = 64 5920 / 5272; 20 0.6B-shaped blocks r = 16 1808 / 1670; panels of up to 64 rows 3005 / 3001 (r = 16 without shared inputs).
constexpr int kTwoBlockRows = 96;      // panel rows from which a launch takes two blocks per CTA

struct TcShared {
  uint64_t full[8];
  uint64_t empty[8];
  uint64_t accum;
  uint32_t tmem_base;
  int failed;
};

__device__ __forceinline__ uint32_t pow2_cols(int n) {
  uint32_t c = 32;
  while ((int)c < n) c <<= 1;
  return c;
}

__device__ __forceinline__ void split_bf16(float v, __nv_bfloat16* hi, __nv_bfloat16* lo) {
  const __nv_bfloat16 h = __float2bfloat16_rn(v);
  *hi = h;
  *lo = __float2bfloat16_rn(v - __bfloat162float(h));
}

__device__ __forceinline__ float4 ld_cluster_f4(uint32_t addr) {
  float4 v;
  asm volatile("ld.shared::cluster.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "r"(addr) : "memory");
  return v;
}

// Eight ranks of a token of T out, as bf16 hi and lo parts (Tt is [NB][m_pad], tokens contiguous): `hi` is where the first
// rank's hi part goes, its lo part follows `lo_off` elements after
__device__ __forceinline__ void put_t8(__nv_bfloat16* hi, long long lo_off, long long m_pad, const float (&v)[8]) {
#pragma unroll
  for (int j = 0; j < 8; ++j) {
    __nv_bfloat16 h, l;
    split_bf16(v[j], &h, &l);
    hi[j * m_pad] = h;
    hi[j * m_pad + lo_off] = l;
  }
}

// ---------------------------------------------------------------- T = X Q  (Tt = T^T as bf16 hi/lo)
// One cluster of CK CTAs per tile of 128 * MB tokens of one layer; grid = (max token tiles * CK, layers in the wave).
// CK > 1 (MB = 1 only): launches with fewer token tiles than the device has room for split the columns over the CTAs of a
// cluster; their sums of T meet through distributed shared memory, CTA c adding (in rank order) and writing the ranks
// 8 c .. 8 c + 7, 8 (c + CK) ...  Four 0.6B-shaped blocks, 613 tokens, r = 8, a call per group: 1465 -> 1186 us.
template <int MB>
__global__ void __launch_bounds__(tc_threads(MB)) tc_x_q_kernel(const DevLayer* __restrict__ layers, int l0, DevStatus* status,
                                                                int stages, int skip_fused, int CK) {
  // CTA rows are handed out in the order the scheduler starts them: the layers with the longest
  // token rows (largest d_in, longest CTAs) go first so that the wave does not end on them
  const int li = l0 + layers[l0 + blockIdx.y].xq_order;
  const DevLayer& L = layers[li];
  const int rank = CK > 1 ? (int)cluster_ctarank() : 0;
  const int t0 = ((int)blockIdx.x / CK) * 128 * MB;
  if (t0 >= L.m || (skip_fused && L.fz_C) || L.grp_role == 2) return;
  extern __shared__ __align__(1024) uint8_t smem_raw[];
  uint8_t* tiles = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
  __shared__ TcShared sh;
  const int NB = L.NB, NP = L.NP;                     // operand rows: the whole group's for a leader
  const int a_bytes = 2 * MB * kTileBytes;            // [128 MB tokens][64 d]
  const int b_bytes = NB * kBoxK * 2;                 // [NB][64 d]
  const int stage_bytes = a_bytes + ((b_bytes + 1023) & ~1023);
  const int nk_all = (L.d_in + kBoxK - 1) / kBoxK;
  const int kb = rank * nk_all / CK, nk = (rank + 1) * nk_all / CK - kb;   // this CTA's k-steps
  const int nblk = min(MB, (L.m - t0 + 127) / 128);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const uint8_t* maps = reinterpret_cast<const uint8_t*>(L.tmaps);
  const void* map_x = maps;            // X  [m][d_in], box 64 x 64
  const void* map_q = maps + 128;      // Qb [NB][d_in], box 64 x NB
  const uint32_t ncols = pow2_cols(MB * NB);

  if (threadIdx.x == 0) {
    for (int s = 0; s < stages; ++s) { mbar_init(&sh.full[s], 1); mbar_init(&sh.empty[s], 1); }
    mbar_init(&sh.accum, 1);
    sh.failed = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  }
  if (warp == 1) tmem_alloc(&sh.tmem_base, ncols);
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = sh.tmem_base;
  const uint32_t step_tx = nblk * 2 * kTileBytes + b_bytes;
  // With one row block per CTA the ring's first tiles of X are on their way before the panel that the predecessor writes
  // is waited for (a step of small shapes through forward hooks, 613 tokens, r = 8: 1124 -> 1081 us).  With two the same
  // was slower (eight 8B blocks, r = 64: 11.86 -> 12.07 ms at best).
  const int pre = MB == 1 ? min(stages, nk) : 0;
  if (MB == 1 && threadIdx.x == 0) {
    tmap_acquire(map_x);
    for (int k = 0; k < pre; ++k) {
      mbar_expect_tx(&sh.full[k], step_tx);
      for (int x = 0; x < 2 * nblk; ++x) tma_load_2d(tiles + (size_t)k * stage_bytes + x * kTileBytes, map_x, (kb + k) * kBoxK, t0 + 64 * x, &sh.full[k]);
    }
  }
  chain_wait();
  const long long m_pad = L.m_pad, lo_off = NP * m_pad;
  const bool early = short_launch();
  if (early) chain_next();

  if (warp == 0) {
    if (lane == 0) {
      tmap_acquire(map_x);
      tmap_acquire(map_q);
      // With four or more stages, two k-steps are issued together, box by box: the two 128-byte
      // pieces of a token row then reach the memory system back to back (256 contiguous bytes per
      // row instead of 128; 8B shapes, r = 16: T = X Q 20.6 -> 17.6 ms per step).  With three
      // stages waiting for two free ones at a time costs more than it brings.
      bool ok = true;
      int issued = 0;            // k-steps whose loads have been issued
      const int group = stages >= 4 ? 2 : 1;
      for (int k = 0; k < pre; ++k)
        tma_load_2d(tiles + (size_t)k * stage_bytes + a_bytes, map_q, (kb + k) * kBoxK, 0, &sh.full[k]);
      issued = pre;
      for (int k = pre; k < nk && ok; k += group) {
        const int n2 = min(group, nk - k);
        uint8_t* a[2];
        uint64_t* bar[2];
        for (int u = 0; u < n2; ++u) {
          const int kk = k + u, s = kk % stages;
          if (kk >= stages && !mbar_wait(&sh.empty[s], ((kk / stages) - 1) & 1)) { sh.failed = 1; ok = false; break; }
          a[u] = tiles + (size_t)s * stage_bytes;
          bar[u] = &sh.full[s];
          mbar_expect_tx(bar[u], step_tx);
        }
        if (!ok) break;
        for (int x = 0; x < 2 * nblk; ++x)
          for (int u = 0; u < n2; ++u) tma_load_2d(a[u] + x * kTileBytes, map_x, (kb + k + u) * kBoxK, t0 + 64 * x, bar[u]);
        for (int u = 0; u < n2; ++u) tma_load_2d(a[u] + a_bytes, map_q, (kb + k + u) * kBoxK, 0, bar[u]);
        issued = k + n2;
      }
      if (!ok || sh.failed) {    // leaving early: the copies in flight must land before the CTA goes away
        for (int k = issued > stages ? issued - stages : 0; k < issued; ++k) mbar_wait(&sh.full[k % stages], (k / stages) & 1);
      }
    }
  } else if (warp == 1) {
    // all lanes run the loop and one elected lane issues: the descriptors stay warp-uniform (see mma_bf16_if)
    const uint32_t go = elect_one();
    const uint32_t idesc = instr_desc(128, NB, 0, 0), tiles_addr = smem_u32(tiles);
    uint32_t s = 0, par = 0, acc = 0u;
    for (int k = 0; k < nk; ++k) {
      if (!mbar_wait_warp(&sh.full[s], par)) { sh.failed = 1; break; }
      tc_fence_after();
      const uint32_t a = tiles_addr + s * (uint32_t)stage_bytes;
      const uint64_t bd = smem_desc(a + (uint32_t)a_bytes, 0, 1024);
#pragma unroll
      for (int x = 0; x < MB; ++x) {
        if (x >= nblk) break;
        const uint64_t ad = smem_desc(a + (uint32_t)(x * 2 * kTileBytes), 0, 1024);
#pragma unroll
        for (int kk = 0; kk < kBoxK / 16; ++kk)          // 16 columns = 32 bytes = 2 descriptor units further
          mma_bf16_if(go, tmem + (uint32_t)(x * NB), ad + (uint64_t)(2 * kk), bd + (uint64_t)(2 * kk), idesc, kk > 0 ? 1u : acc);
      }
      acc = 1u;
      mma_commit_if(go, &sh.empty[s]);       // the stage is free once these MMAs have read it
      if (++s == (uint32_t)stages) { s = 0; par ^= 1u; }
    }
    mma_commit_if(go, &sh.accum);            // arrives when every MMA issued so far is done
  } else {
    // epilogue: TMEM lane i of this warp's quarter = token 32 q + lane of the block
    const int q = warp & 3, blk = (warp - 2) >> 2;
    const bool ok = mbar_wait(&sh.accum, 0);
    tc_fence_after();
    if (!early) chain_next();
    if (!ok) sh.failed = 1;
    const int row = q * 32 + lane, t = t0 + 128 * blk + row;
    __nv_bfloat16* out = L.Tb + t;
    if (ok && blk < nblk) {
      for (int k0 = 0; k0 < NP; k0 += 8) {
        float hi[8], lo[8];
        const uint32_t col = tmem + ((uint32_t)(q * 32) << 16) + (uint32_t)(blk * NB + k0);
        tmem_ld8(col, hi);
        tmem_ld8(col + (uint32_t)NP, lo);
#pragma unroll
        for (int j = 0; j < 8; ++j) hi[j] += lo[j];
        if (CK > 1) {            // the pipeline's stages are idle: they take the partial sums, [rank group][token][8]
          float4* p = reinterpret_cast<float4*>(tiles) + ((k0 >> 3) * 128 + row) * 2;
          p[0] = make_float4(hi[0], hi[1], hi[2], hi[3]);
          p[1] = make_float4(hi[4], hi[5], hi[6], hi[7]);
        } else if (t < L.m) {
          put_t8(out + k0 * m_pad, lo_off, m_pad, hi);
        }
      }
    }
  }
  if (MB == 1 && CK > 1) {
    __syncwarp();
    cluster_sync_all();          // every CTA's partial sums are in its shared memory
    const int q = warp & 3, row = q * 32 + lane, t = t0 + row;
    if (warp >= 2 && t < L.m) {
      for (int g = rank; g < NP / 8; g += CK) {
        float v[8] = {};
        const uint32_t at = smem_u32(tiles) + (uint32_t)((g * 128 + row) * 32);
        for (int c = 0; c < CK; ++c) {
          const uint32_t src = mapa_shared(at, (uint32_t)c);
          const float4 x = ld_cluster_f4(src), y = ld_cluster_f4(src + 16);
          v[0] += x.x; v[1] += x.y; v[2] += x.z; v[3] += x.w;
          v[4] += y.x; v[5] += y.y; v[6] += y.z; v[7] += y.w;
        }
        put_t8(L.Tb + t + 8 * g * m_pad, lo_off, m_pad, v);
      }
    }
    __syncwarp();
    cluster_sync_all();          // nobody leaves while a peer reads its sums
  }
  tc_fence_before();
  __syncthreads();
  if (sh.failed && threadIdx.x == 0) report_timeout(status, 1);
  if (warp == 1) { tc_fence_after(); tmem_dealloc(tmem, ncols); }
}

// ---------------------------------------------------------------- Ypart[s] = X_s^T T_s
// One CTA per (128 * MB columns of X, token slab) of one layer.  grid = (column chunks, slabs, layers).
template <int MB>
__global__ void __launch_bounds__(tc_threads(MB)) tc_xt_t_kernel(const DevLayer* __restrict__ layers, int l0, DevStatus* status,
                                                                 int stages, int skip_fused) {
  const DevLayer& L = layers[l0 + blockIdx.z];
  const int d0 = blockIdx.x * 128 * MB;
  const int slab = blockIdx.y;
  if (d0 >= L.d_in || slab >= L.slabs || (skip_fused && L.fz_C) || L.grp_role == 2) return;
  extern __shared__ __align__(1024) uint8_t smem_raw[];
  uint8_t* tiles = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
  __shared__ TcShared sh;
  const int NB = L.NB;
  const int a_bytes = 2 * MB * kTileBytes;            // two [64 tokens][64 d] boxes per block of 128 columns
  const int b_bytes = NB * kBoxK * 2;                 // [NB][64 tokens]
  const int stage_bytes = a_bytes + ((b_bytes + 1023) & ~1023);
  const int nblk = min(MB, (L.d_in - d0 + 127) / 128);
  const int t_begin = slab * L.slab_rows;
  const int t_end = min(L.m, t_begin + L.slab_rows);
  const int nk = (t_end - t_begin + kBoxK - 1) / kBoxK;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const uint8_t* maps = reinterpret_cast<const uint8_t*>(L.tmaps);
  const void* map_x = maps;            // X  [m][d_in], box 64 x 64
  const void* map_t = maps + 256;      // Tt [NB][m],   box 64 x NB
  const uint32_t ncols = pow2_cols(MB * NB);

  if (threadIdx.x == 0) {
    for (int s = 0; s < stages; ++s) { mbar_init(&sh.full[s], 1); mbar_init(&sh.empty[s], 1); }
    mbar_init(&sh.accum, 1);
    sh.failed = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  }
  if (warp == 1) tmem_alloc(&sh.tmem_base, ncols);
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = sh.tmem_base;
  const uint32_t step_tx = nblk * 2 * kTileBytes + b_bytes;
  const int pre = MB == 1 ? min(stages, nk) : 0;       // as in tc_x_q_kernel
  if (MB == 1 && threadIdx.x == 0) {
    tmap_acquire(map_x);
    for (int k = 0; k < pre; ++k) {
      mbar_expect_tx(&sh.full[k], step_tx);
      for (int x = 0; x < 2 * nblk; ++x) tma_load_2d(tiles + (size_t)k * stage_bytes + x * kTileBytes, map_x, d0 + 64 * x, t_begin + k * kBoxK, &sh.full[k]);
    }
  }
  chain_wait();
  const bool early = short_launch();
  if (early) chain_next();

  if (warp == 0) {
    if (lane == 0) {
      tmap_acquire(map_x);
      tmap_acquire(map_t);
      for (int k = 0; k < pre; ++k)
        tma_load_2d(tiles + (size_t)k * stage_bytes + a_bytes, map_t, t_begin + k * kBoxK, 0, &sh.full[k]);
      int issued = pre;
      for (int k = pre; k < nk; ++k) {
        const int s = k % stages;
        if (k >= stages && !mbar_wait(&sh.empty[s], ((k / stages) - 1) & 1)) { sh.failed = 1; break; }
        uint8_t* a = tiles + (size_t)s * stage_bytes;
        const int tk = t_begin + k * kBoxK;
        mbar_expect_tx(&sh.full[s], step_tx);
        for (int x = 0; x < 2 * nblk; ++x) tma_load_2d(a + x * kTileBytes, map_x, d0 + 64 * x, tk, &sh.full[s]);
        tma_load_2d(a + a_bytes, map_t, tk, 0, &sh.full[s]);
        issued = k + 1;
      }
      if (sh.failed) {           // leaving early: the copies in flight must land before the CTA goes away
        for (int k = issued > stages ? issued - stages : 0; k < issued; ++k) mbar_wait(&sh.full[k % stages], (k / stages) & 1);
      }
    }
  } else if (warp == 1) {
    const uint32_t go = elect_one();
    const uint32_t idesc = instr_desc(128, NB, 1, 0), tiles_addr = smem_u32(tiles);     // A is MN-major: the X tile as X^T
    uint32_t s = 0, par = 0, acc = 0u;
    for (int k = 0; k < nk; ++k) {
      if (!mbar_wait_warp(&sh.full[s], par)) { sh.failed = 1; break; }
      tc_fence_after();
      const uint32_t a = tiles_addr + s * (uint32_t)stage_bytes;
      const uint64_t bd = smem_desc(a + (uint32_t)a_bytes, 0, 1024);
#pragma unroll
      for (int x = 0; x < MB; ++x) {
        if (x >= nblk) break;
        const uint64_t ad = smem_desc(a + (uint32_t)(x * 2 * kTileBytes), kTileBytes, 1024);
#pragma unroll
        for (int kk = 0; kk < kBoxK / 16; ++kk)
          // 16 tokens = two 8-row swizzle atoms = 2048 bytes = 128 descriptor units further down the X boxes
          mma_bf16_if(go, tmem + (uint32_t)(x * NB), ad + (uint64_t)(128 * kk), bd + (uint64_t)(2 * kk), idesc, kk > 0 ? 1u : acc);
      }
      acc = 1u;
      mma_commit_if(go, &sh.empty[s]);
      if (++s == (uint32_t)stages) { s = 0; par ^= 1u; }
    }
    mma_commit_if(go, &sh.accum);
  } else {
    const int q = warp & 3, blk = (warp - 2) >> 2;
    const bool ok = mbar_wait(&sh.accum, 0);
    tc_fence_after();
    if (!early) chain_next();
    if (!ok) sh.failed = 1;
    const int d = d0 + 128 * blk + q * 32 + lane;
    if (ok && blk < nblk) {
      const int r = L.pr, NP = L.NP;
      float* out = L.Ypart + slab * L.ypart_stride + d;
      for (int k0 = 0; k0 < NP; k0 += 8) {
        float hi[8], lo[8];
        const uint32_t col = tmem + ((uint32_t)(q * 32) << 16) + (uint32_t)(blk * NB + k0);
        tmem_ld8(col, hi);
        tmem_ld8(col + (uint32_t)NP, lo);
        if (d < L.d_in) {
#pragma unroll
          for (int j = 0; j < 8; ++j)
            if (k0 + j < r) out[(long long)(k0 + j) * L.d_in] = hi[j] + lo[j];
        }
      }
    }
  }
  tc_fence_before();
  __syncthreads();
  if (sh.failed && threadIdx.x == 0) report_timeout(status, 2);
  if (warp == 1) { tc_fence_after(); tmem_dealloc(tmem, ncols); }
}

// ---------------------------------------------------------------- Omega -> Tt (hi/lo), pads zero
// Tt is [NB][m_pad] with the tokens contiguous, Omega's stream is row-major over (token, k): a
// thread takes kTok neighbouring tokens and the eight consecutive k of group blockIdx.z, so that for every
// k a warp writes 32 kTok neighbouring tokens.  Local token t is row row0 + t of the whole batch's
// test matrix (see fill_omega_kernel).
// Bound by the instructions of the generator: two tokens a thread make four-byte stores and independent chains, and no division
// per unit: 196 layers, 8192 tokens, r = 8 49 -> 37 us, 50 layers, 16384 tokens, r = 16 43 -> 32;
// one where two would leave SMs without work.
template <int kTok>
__global__ void __launch_bounds__(256) tc_fill_omega_kernel(const DevLayer* layers, int l0, uint64_t seed,
                                                            long long row0, DevStatus* status, int region) {
  chain_wait();
  if (short_launch()) chain_next();
  if (blockIdx.x + blockIdx.y + blockIdx.z == 0 && threadIdx.x == 0) wave_begins(status, region);
  const DevLayer& L = layers[l0 + blockIdx.y];
  const int g = (int)blockIdx.z, r = L.r, rows = L.prow_n;
  const int t0 = (int)(blockIdx.x * 256 + threadIdx.x) * kTok;
  if (8 * g >= rows || t0 >= L.m) return;
  const int nv = min(8, r - 8 * g);                 // live k of this group (the rest is padding)
  float v[kTok][8];
#pragma unroll
  for (int i = 0; i < kTok; ++i) {
#pragma unroll
    for (int u = 0; u < 8; ++u) v[i][u] = 0.f;
    if (nv <= 0 || t0 + i >= L.m) continue;
    const long long e_first = (row0 + t0 + i) * r + 8 * g;
    const uint64_t b0 = (uint64_t)(e_first >> 2);
    const int off = (int)(e_first & 3);
    const int nblk = (off + nv + 3) >> 2;           // at most three Philox blocks, two where r is a multiple of four
    const float4 none = make_float4(0.f, 0.f, 0.f, 0.f);
    const float4 ga = gaussian_block(b0, L.layer_id, kTagOmega, seed);
    const float4 gb = nblk > 1 ? gaussian_block(b0 + 1, L.layer_id, kTagOmega, seed) : none;
    const float4 gc = nblk > 2 ? gaussian_block(b0 + 2, L.layer_id, kTagOmega, seed) : none;
    const float x[12] = {ga.x, ga.y, ga.z, ga.w, gb.x, gb.y, gb.z, gb.w, gc.x, gc.y, gc.z, gc.w};
#pragma unroll
    for (int u = 0; u < 8; ++u) {
      const float y = off == 0 ? x[u] : off == 1 ? x[u + 1] : off == 2 ? x[u + 2] : x[u + 3];
      v[i][u] = u < nv ? y : 0.f;
    }
  }
  __nv_bfloat16* hi_rows = L.Tb + (long long)(L.grp_off + 8 * g) * L.m_pad + t0;
  __nv_bfloat16* lo_rows = hi_rows + (long long)L.NP * L.m_pad;
#pragma unroll
  for (int u = 0; u < 8; ++u) {
    if (8 * g + u >= rows) break;
    __nv_bfloat16 h[kTok], l[kTok];
#pragma unroll
    for (int i = 0; i < kTok; ++i) split_bf16(v[i][u], &h[i], &l[i]);
    const long long at = (long long)u * L.m_pad;
    if (kTok == 2) {        // the pitch is a multiple of eight: the second token is inside the row, beyond m a zero
      *reinterpret_cast<__nv_bfloat162*>(hi_rows + at) = __nv_bfloat162(h[0], h[kTok - 1]);
      *reinterpret_cast<__nv_bfloat162*>(lo_rows + at) = __nv_bfloat162(l[0], l[kTok - 1]);
    } else {
      hi_rows[at] = h[0];
      lo_rows[at] = l[0];
    }
  }
}

// ---------------------------------------------------------------- the bounded wait, on its own
__global__ void debug_wait_kernel(DevStatus* status) {
  __shared__ uint64_t bar;
  if (threadIdx.x == 0) {
    mbar_init(&bar, 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  __syncthreads();
  if (threadIdx.x == 0 && !mbar_wait(&bar, 0)) report_timeout(status, 100);     // nobody arrives: the wait runs out
}

typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                  const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                                  CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

bool encode_2d(void* fn, void* out, const void* base, uint64_t inner, uint64_t outer, uint64_t pitch_bytes,
               uint32_t box_inner, uint32_t box_outer) {
  CUtensorMap m;
  const cuuint64_t dims[2] = {inner, outer};
  const cuuint64_t strides[1] = {pitch_bytes};
  const cuuint32_t box[2] = {box_inner, box_outer};
  const cuuint32_t es[2] = {1, 1};
  CUresult r = reinterpret_cast<EncodeTiledFn>(fn)(&m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void*>(base),
                                                   dims, strides, box, es, CU_TENSOR_MAP_INTERLEAVE_NONE,
                                                   // 256-byte promotion: the neighbouring 128 bytes of a row are
                                                   // what the next box of the same rows reads
                                                   CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                                                   CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  if (r != CUDA_SUCCESS) return false;
  std::memcpy(out, &m, sizeof(m));
  return true;
}

int np_of(int r) { return (r + 7) & ~7; }
long long mpad_of(int m) { return ((long long)m + 7) & ~7ll; }
size_t up256(size_t x) { return (x + 255) / 256 * 256; }

int stage_bytes(int NB, int mb) { return mb * 2 * kTileBytes + ((NB * kBoxK * 2 + 1023) & ~1023); }
int stages_for(int NB, int mb) {
  int s = (mb == 1 ? 96 : 220) * 1024 / stage_bytes(NB, mb);
  if (s > 8) s = 8;
  if (s < 2) s = 2;
  return s;
}
size_t smem_for(int NB, int mb, int stages) {
  const size_t b = (size_t)stage_bytes(NB, mb) * stages + 1024, least = mb == 1 ? kMinSmem : 120 * 1024;   // two, one CTA per SM
  return b < least ? least : b;
}

// What a product's launch has to serve: the layers that stand for themselves or lead a group
struct ProductShape {
  int max_nb = 0, min_nk = 1 << 30;
  long long tiles = 0;      // blocks of 128 tokens, or of 128 columns times slabs
};
template <typename F>
ProductShape product_shape(const ExtractWave& w, const DevLayer* h_dev, bool skip_fused, F tiles_of) {
  ProductShape p;
  for (int i = w.l0; i < w.l1; ++i) {
    const DevLayer& D = h_dev[i];
    if (D.grp_role == 2 || (skip_fused && D.fz_C)) continue;
    p.max_nb = D.NB > p.max_nb ? D.NB : p.max_nb;
    const int nk = (D.d_in + kBoxK - 1) / kBoxK;
    p.min_nk = nk < p.min_nk ? nk : p.min_nk;
    p.tiles += tiles_of(D);
  }
  return p;
}

}  // namespace

bool tc_encode_bf16_2d(const TcState& st, void* out, const void* base, uint64_t inner, uint64_t outer,
                       uint64_t pitch_bytes, uint32_t box_inner, uint32_t box_outer) {
  if (!st.encode_fn) return false;
  return encode_2d(st.encode_fn, out, base, inner, outer, pitch_bytes, box_inner, box_outer);
}

cudaError_t tc_init(TcState* st, int device) {
  st->device = device;
  st->available = false;
  st->encode_fn = nullptr;
  void* fn = nullptr;
  cudaDriverEntryPointQueryResult q;
  cudaError_t e = cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &fn, cudaEnableDefault, &q);
  if (e != cudaSuccess || q != cudaDriverEntryPointSuccess || !fn) {
    cudaGetLastError();
    return cudaSuccess;   // the CUDA-core path still works
  }
  int major = 0;
  cudaDeviceGetAttribute(&major, cudaDevAttrComputeCapabilityMajor, device);
  st->encode_fn = fn;
  st->available = major == 10;
  if (st->available) {
    for (const void* k : {(const void*)tc_x_q_kernel<1>, (const void*)tc_x_q_kernel<2>, (const void*)tc_xt_t_kernel<1>,
                          (const void*)tc_xt_t_kernel<2>})
      if (e == cudaSuccess) e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, 226 * 1024);
    if (e == cudaSuccess) e = rmw_tc_init();
    if (e == cudaSuccess) {
      int sms = 0;
      e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, device);
      if (e == cudaSuccess) e = fused_init(sms, &st->fused);
    }
    if (e != cudaSuccess) { cudaGetLastError(); st->available = false; }
  }
  return cudaSuccess;
}

cudaError_t launch_debug_wait(DevStatus* d_status, cudaStream_t s) {
  debug_wait_kernel<<<1, 32, 0, s>>>(d_status);
  return cudaGetLastError();
}

bool tc_eligible(const agzo_layer& a) {
  return a.X && a.x_dtype == AGZO_BF16 && (reinterpret_cast<uintptr_t>(a.X) & 15u) == 0 && a.ldx % 8 == 0 &&
         a.d_in % 8 == 0 && a.d_in >= 128 && a.m >= 256 && a.r >= 1 && a.r <= AGZO_MAX_RANK;
}

int tc_operand_rows(int r) { return 2 * np_of(r); }

size_t tc_panel_bytes(const agzo_layer& a, int ranks) {
  const size_t rows = (size_t)tc_operand_rows(ranks);
  return up256(rows * (size_t)a.d_in * 2) + up256(rows * (size_t)mpad_of(a.m) * 2);
}

void tc_set_panels(const agzo_layer& a, DevLayer* D, char* p, int ranks, int off, bool last) {
  D->NP = np_of(ranks);
  D->NB = 2 * D->NP;
  D->m_pad = mpad_of(a.m);
  D->Qb = reinterpret_cast<__nv_bfloat16*>(p);
  D->Tb = reinterpret_cast<__nv_bfloat16*>(p + up256((size_t)D->NB * (size_t)a.d_in * 2));
  D->pr = ranks;
  D->grp_off = off;
  D->prow_n = last ? D->NP - off : a.r;
}

bool tc_encode_maps(const TcState& st, const DevLayer& D, void* host_maps) {
  if (!st.encode_fn) return false;
  uint8_t* out = static_cast<uint8_t*>(host_maps);
  // X [m][ldx]: inner = d_in, outer = m; one box = 64 columns x 64 tokens
  if (!encode_2d(st.encode_fn, out, D.X, (uint64_t)D.d_in, (uint64_t)D.m, (uint64_t)D.ldx * 2, 64, 64)) return false;
  const uint32_t nb = (uint32_t)D.NB;       // a group leader's descriptors cover the panel of the whole group
  // Qb [nb][d_in]: box = 64 columns x nb rows
  if (!encode_2d(st.encode_fn, out + 128, D.Qb, (uint64_t)D.d_in, (uint64_t)nb, (uint64_t)D.d_in * 2, 64, nb))
    return false;
  // Tt [nb][m_pad]: inner extent is the true m so that the padding is read as zero
  if (!encode_2d(st.encode_fn, out + 256, D.Tb, (uint64_t)D.m, (uint64_t)nb, (uint64_t)D.m_pad * 2, 64, nb))
    return false;
  return true;
}

cudaError_t tc_fill_omega(const TcState&, const ExtractWave& w, const DevLayer*, uint64_t seed, DevStatus* d_status, cudaStream_t s) {
  const unsigned nl = (unsigned)(w.l1 - w.l0), groups = (unsigned)((w.max_r + 14) >> 3);   // padding rows of a panel included
  const bool pairs = (long long)w.max_m * groups * nl >= 2ll * w.sm_count * 2048;
  const unsigned per = pairs ? 512 : 256;
  return launch_chained(pairs ? tc_fill_omega_kernel<2> : tc_fill_omega_kernel<1>, dim3(((unsigned)w.max_m + per - 1) / per, nl, groups),
                        256, 0, 0, s, w.d_layers, w.l0, seed, w.omega_row0, d_status, w.region);
}

cudaError_t tc_xt_t(const TcState&, const ExtractWave& w, const DevLayer* h_dev, DevStatus* d_status,
                    bool skip_fused, cudaStream_t s) {
  const ProductShape p = product_shape(w, h_dev, skip_fused, [](const DevLayer& D) { return (long long)D.gchunks * D.slabs; });
  const int mb = p.max_nb >= kTwoBlockRows && p.tiles >= 4 * w.sm_count ? 2 : 1;
  const int stages = stages_for(p.max_nb, mb);
  const dim3 grid((w.max_din + 128 * mb - 1) / (128 * mb), w.max_slabs, w.l1 - w.l0);
  return launch_chained(mb == 1 ? tc_xt_t_kernel<1> : tc_xt_t_kernel<2>, grid, tc_threads(mb), smem_for(p.max_nb, mb, stages), 0, s,
                        w.d_layers, w.l0, d_status, stages, skip_fused ? 1 : 0);
}

cudaError_t tc_x_q(const TcState&, const ExtractWave& w, const DevLayer* h_dev, DevStatus* d_status,
                   bool skip_fused, cudaStream_t s) {
  const ProductShape p = product_shape(w, h_dev, skip_fused, [](const DevLayer& D) { return (long long)(D.m + 127) / 128; });
  const int mb = p.max_nb >= kTwoBlockRows && p.tiles >= 4 * w.sm_count ? 2 : 1;
  int ck = 1;       // CTAs per token tile: up to two per SM, and at least two k-steps each
  while (mb == 1 && ck < 8 && p.tiles * ck <= w.sm_count && p.min_nk >= 4 * ck) ck *= 2;
  const int stages = stages_for(p.max_nb, mb);
  const dim3 grid((w.max_m + 128 * mb - 1) / (128 * mb) * ck, w.l1 - w.l0);
  return launch_chained(mb == 1 ? tc_x_q_kernel<1> : tc_x_q_kernel<2>, grid, tc_threads(mb), smem_for(p.max_nb, mb, stages),
                        ck > 1 ? ck : 0, s, w.d_layers, w.l0, d_status, stages, skip_fused ? 1 : 0, ck);
}

}  // namespace agzo

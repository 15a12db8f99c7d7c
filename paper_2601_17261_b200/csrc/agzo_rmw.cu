// In-place low-rank passes of Algorithm 2: W <- W + c * R A^T with R regenerated from the
// Philox counter inside the kernel (Eq. agzo-perturb).  One grouped launch covers every
// layer of the call; a tile is tile_rows x kTileCols of one layer's W.
//
// HBM-bound for r <= 16: each weight is read once and written once (16-byte accesses, 128 bytes
// in flight per thread at all times); R for the tile's rows is generated once into shared memory
// and the tile's slice of A^T lives in registers, so neither R nor Delta ever reaches DRAM.
// Measured (one pass over six 8B-shaped blocks, bf16, 4.6 GB, copy rate 6541 GB/s): r = 1 6289 GB/s (6182 with loads
// issued a sub-block at a time and after R), r = 4 6326 (5614), r = 8 5625 (4740); 28 0.6B-shaped blocks r = 4 6246 (5317), fp32
// r = 8 6194 (4448); eight 1024 x 1024 master/compute pairs, r = 8: 37 -> 9.7 us; one fp32 256 x 256 layer 16 -> 3 us.
#include "agzo_common.cuh"

namespace agzo {

constexpr int kRmwThreads = 256;
constexpr int kTileCols = kRmwTileCols;   // 64 threads x 8 consecutive columns
constexpr int kTileRows = kRmwMaxTileRows;   // largest tile (shared memory is sized for it)
constexpr int kRowLanes = 4;     // thread groups that take different rows
constexpr int kRowsInFlight = 8; // rows per thread per sub-block
constexpr int kSubRows = kRowLanes * kRowsInFlight;
// rows whose loads a thread keeps in flight: 128 bytes
template <int MODE> constexpr int rows_ahead() { return MODE == RMW_BF16 ? 8 : 4; }

__device__ __forceinline__ float bf16lo(uint32_t u) { return __uint_as_float(u << 16); }
__device__ __forceinline__ float bf16hi(uint32_t u) { return __uint_as_float(u & 0xFFFF0000u); }
__device__ __forceinline__ uint32_t pack_bf16(float a, float b) {
  __nv_bfloat162 p = __floats2bfloat162_rn(a, b);   // RNE, a in the low half
  return *reinterpret_cast<uint32_t*>(&p);
}
__device__ __forceinline__ float round_to_bf16(float a) {
  return __bfloat162float(__float2bfloat16_rn(a));
}

// ------------------------------------------------------------------ tile I/O (16-byte accesses)
// Eight consecutive weights of one row, kept in their storage format until they are used
// (a bf16 row segment is four registers, not eight).
template <int MODE> struct Raw8 { float4 a, b; };
template <> struct Raw8<RMW_BF16> { uint4 q; };

template <int MODE>
__device__ __forceinline__ void load8(const DevLayer& L, long long row, int col, Raw8<MODE>& w) {
  if constexpr (MODE == RMW_BF16) {
    const __nv_bfloat16* p = reinterpret_cast<const __nv_bfloat16*>(L.W) + row * L.ldw + col;
    w.q = __ldcs(reinterpret_cast<const uint4*>(p));
  } else {
    const float* p = reinterpret_cast<const float*>(L.W) + row * L.ldw + col;
    w.a = __ldcs(reinterpret_cast<const float4*>(p));
    w.b = __ldcs(reinterpret_cast<const float4*>(p) + 1);
  }
}

template <int MODE>
__device__ __forceinline__ void unpack8(const Raw8<MODE>& r, float (&w)[8]) {
  if constexpr (MODE == RMW_BF16) {
    w[0] = bf16lo(r.q.x); w[1] = bf16hi(r.q.x); w[2] = bf16lo(r.q.y); w[3] = bf16hi(r.q.y);
    w[4] = bf16lo(r.q.z); w[5] = bf16hi(r.q.z); w[6] = bf16lo(r.q.w); w[7] = bf16hi(r.q.w);
  } else {
    w[0] = r.a.x; w[1] = r.a.y; w[2] = r.a.z; w[3] = r.a.w;
    w[4] = r.b.x; w[5] = r.b.y; w[6] = r.b.z; w[7] = r.b.w;
  }
}

template <int MODE>
__device__ __forceinline__ void store8(const DevLayer& L, long long row, int col, const float (&w)[8]) {
  if (MODE == RMW_BF16 || MODE == RMW_PAIR_COMPUTE || MODE == RMW_PAIR_UPDATE) {
    __nv_bfloat16* p = (MODE == RMW_BF16)
                           ? reinterpret_cast<__nv_bfloat16*>(L.W) + row * L.ldw + col
                           : reinterpret_cast<__nv_bfloat16*>(L.W16) + row * L.ldw16 + col;
    uint4 q;
    q.x = pack_bf16(w[0], w[1]); q.y = pack_bf16(w[2], w[3]);
    q.z = pack_bf16(w[4], w[5]); q.w = pack_bf16(w[6], w[7]);
    __stcs(reinterpret_cast<uint4*>(p), q);
  }
  if (MODE == RMW_F32 || MODE == RMW_PAIR_UPDATE) {
    float* p = reinterpret_cast<float*>(L.W) + row * L.ldw + col;
    __stcs(reinterpret_cast<float4*>(p), make_float4(w[0], w[1], w[2], w[3]));
    __stcs(reinterpret_cast<float4*>(p) + 1, make_float4(w[4], w[5], w[6], w[7]));
  }
}

// ------------------------------------------------------------------ R for the rows of a tile
// sG[DUP * (row_local * RS + k)] = R[row0 + row_local][k], DUP = 2: twice, side by side (an operand of the packed
// multiply-adds); columns r..RS-1 are zero.
template <int DUP>
__device__ __forceinline__ void generate_G(float* sG, int RS, int r, long long row0, int nrows,
                                           uint32_t layer_id, uint64_t seed) {
  const long long e_first = row0 * r;
  const long long e_last = e_first + (long long)nrows * r;
  const long long b_first = e_first >> 2;
  const int nb = (int)(((e_last - 1) >> 2) - b_first + 1);
  for (int i = threadIdx.x; i < nb; i += kRmwThreads) {
    const long long b = b_first + i;
    const float4 g = gaussian_block<false>((uint64_t)b, layer_id, kTagG, seed);
    const float gv[4] = {g.x, g.y, g.z, g.w};
#pragma unroll
    for (int lane = 0; lane < 4; ++lane) {
      const long long e = 4 * b + lane;
      if (e >= e_first && e < e_last) {
        const int local = (int)(e - e_first);
        const int rl = local / r;
        const int at = rl * RS + (local - rl * r);
        if (DUP == 2) *reinterpret_cast<float2*>(sG + 2 * at) = make_float2(gv[lane], gv[lane]);
        else sG[at] = gv[lane];
      }
    }
  }
  if (RS > r) {
    const int pad = RS - r;
    for (int i = threadIdx.x; i < nrows * pad; i += kRmwThreads) {
      const int rl = i / pad;
      const int at = rl * RS + r + (i - rl * pad);
      if (DUP == 2) *reinterpret_cast<float2*>(sG + 2 * at) = make_float2(0.f, 0.f);
      else sG[at] = 0.f;
    }
  }
}

// ------------------------------------------------------------------ r <= 16: A^T slice in registers
// A thread's weights of a tile: eight columns, rows ry, ry + 4, ...  The loads of the first rows are issued before R is
// generated, and every row that has been written is followed by the load of the row `rows_ahead` further on.
template <int RC, int MODE>
struct TileReg {
  static constexpr int kAhead = rows_ahead<MODE>();
  uint64_t v[RC][4];
  Raw8<MODE> raw[kAhead];
  int col, ry;
  bool live;

  __device__ __forceinline__ void begin(const DevLayer& L, int row0, int nrows, int col0) {
    col = col0 + (threadIdx.x & 63) * 8;
    ry = threadIdx.x >> 6;
    live = col < L.d_in;                 // d_in is a multiple of 8 on this path
    if (!live) return;
#pragma unroll
    for (int j = 0; j < kAhead; ++j)
      if (ry + j * kRowLanes < nrows) load8<MODE>(L, (long long)(row0 + ry + j * kRowLanes), col, raw[j]);
#pragma unroll
    for (int k = 0; k < RC; ++k) {
      float4 a = make_float4(0.f, 0.f, 0.f, 0.f), b = a;
      if (k < L.r) {
        const float* p = L.V + (long long)k * L.ldv + col;
        a = __ldcg(reinterpret_cast<const float4*>(p));
        b = __ldcg(reinterpret_cast<const float4*>(p) + 1);
      }
      v[k][0] = pack_f32x2(a.x, a.y); v[k][1] = pack_f32x2(a.z, a.w);
      v[k][2] = pack_f32x2(b.x, b.y); v[k][3] = pack_f32x2(b.z, b.w);
    }
  }

  __device__ __forceinline__ void run(const DevLayer& L, const float* sG, int row0, int nrows, float coef) {
    if (!live) return;
    const uint64_t c2 = pack_f32x2(coef, coef);
    for (int sb = ry; sb < nrows; sb += kAhead * kRowLanes) {
#pragma unroll
      for (int j = 0; j < kAhead; ++j) {
        const int rl = sb + j * kRowLanes;
        if (rl >= nrows) break;
        uint64_t z[4] = {0, 0, 0, 0};
        const float* g = sG + 2 * rl * RC;
        if constexpr (RC == 1) {
          const uint64_t g2 = *reinterpret_cast<const uint64_t*>(g);
#pragma unroll
          for (int c = 0; c < 4; ++c) z[c] = fma_f32x2(g2, v[0][c], z[c]);
        } else {
#pragma unroll
          for (int k = 0; k < RC; k += 2) {          // k ascending, fixed order
            const ulonglong2 g2 = *reinterpret_cast<const ulonglong2*>(g + 2 * k);
#pragma unroll
            for (int c = 0; c < 4; ++c) z[c] = fma_f32x2(g2.x, v[k][c], z[c]);
#pragma unroll
            for (int c = 0; c < 4; ++c) z[c] = fma_f32x2(g2.y, v[k + 1][c], z[c]);
          }
        }
        float w[8], o[8];
        unpack8<MODE>(raw[j], w);
#pragma unroll
        for (int c = 0; c < 4; ++c) unpack_f32x2(fma_f32x2(c2, z[c], pack_f32x2(w[2 * c], w[2 * c + 1])), o[2 * c], o[2 * c + 1]);
        store8<MODE>(L, (long long)(row0 + rl), col, o);
        const int next = rl + kAhead * kRowLanes;
        if (next < nrows) load8<MODE>(L, (long long)(row0 + next), col, raw[j]);
      }
    }
  }
};

// ------------------------------------------------------------------ 16 < r <= 64: A^T slice in shared memory
template <int MODE>
__device__ __forceinline__ void tile_body_smem(const DevLayer& L, const float* sG, const float* sV,
                                               int RS, int row0, int nrows, int col0, float coef) {
  const int cx = threadIdx.x & 63;
  const int ry = threadIdx.x >> 6;
  const int col = col0 + cx * 8;
  if (col >= L.d_in) return;
  const float* sv = sV + cx * 8;

  for (int sb = 0; sb < nrows; sb += kSubRows) {
    Raw8<MODE> raw[kRowsInFlight];
    float z[kRowsInFlight][8];
#pragma unroll
    for (int j = 0; j < kRowsInFlight; ++j) {
      const int rl = sb + ry + j * kRowLanes;
      if (rl < nrows) load8<MODE>(L, (long long)(row0 + rl), col, raw[j]);
#pragma unroll
      for (int c = 0; c < 8; ++c) z[j][c] = 0.f;
    }
    for (int k4 = 0; k4 < RS; k4 += 4) {
      float4 g4[kRowsInFlight];
#pragma unroll
      for (int j = 0; j < kRowsInFlight; ++j) {
        const int rl = min(sb + ry + j * kRowLanes, nrows - 1);
        g4[j] = *reinterpret_cast<const float4*>(sG + rl * RS + k4);
      }
#pragma unroll
      for (int kk = 0; kk < 4; ++kk) {
        const float4 va = *reinterpret_cast<const float4*>(sv + (k4 + kk) * kTileCols);
        const float4 vb = *reinterpret_cast<const float4*>(sv + (k4 + kk) * kTileCols + 4);
        const float vv[8] = {va.x, va.y, va.z, va.w, vb.x, vb.y, vb.z, vb.w};
#pragma unroll
        for (int j = 0; j < kRowsInFlight; ++j) {
          const float gk = kk == 0 ? g4[j].x : kk == 1 ? g4[j].y : kk == 2 ? g4[j].z : g4[j].w;
#pragma unroll
          for (int c = 0; c < 8; ++c) z[j][c] = fmaf(gk, vv[c], z[j][c]);
        }
      }
    }
#pragma unroll
    for (int j = 0; j < kRowsInFlight; ++j) {
      const int rl = sb + ry + j * kRowLanes;
      if (rl < nrows) {
        float w[8], o[8];
        unpack8<MODE>(raw[j], w);
#pragma unroll
        for (int c = 0; c < 8; ++c) o[c] = fmaf(coef, z[j][c], w[c]);
        store8<MODE>(L, (long long)(row0 + rl), col, o);
      }
    }
  }
}

// the layer of a tile: the last entry of the prefix that is <= tile.  A warp looks at 32 entries at a time (a binary
// search is a chain of log2(layers) dependent loads, paid by every tile); all 32 lanes must call it.
__device__ __forceinline__ int find_layer(const int* tile_start, int n_layers, int tile) {
  const int lane = threadIdx.x & 31;
  int lo = 0, n = n_layers;
  while (n > 1) {
    const int step = (n + 31) >> 5;
    const int at = lo + lane * step;
    const unsigned le = __ballot_sync(0xffffffffu, lane * step < n && tile_start[at] <= tile);
    const int last = 31 - __clz(le);           // entry `lo` always qualifies
    n = min(step, n - last * step);
    lo += last * step;
  }
  return lo;
}

// one 16-byte piece of the record per thread
__device__ __forceinline__ void fetch_layer(DevLayer* dst, const DevLayer* src) {
  static_assert(sizeof(DevLayer) % 16 == 0 && sizeof(DevLayer) / 16 <= kRmwThreads, "one piece per thread");
  if (threadIdx.x < sizeof(DevLayer) / 16)
    reinterpret_cast<uint4*>(dst)[threadIdx.x] = reinterpret_cast<const uint4*>(src)[threadIdx.x];
}

__device__ __forceinline__ int effective_mode(const DevLayer& L, int pair_update) {
  return (L.rmw_mode == RMW_PAIR_COMPUTE && pair_update) ? RMW_PAIR_UPDATE : L.rmw_mode;
}

// Persistent CTAs stride over the tiles of all layers.  A kernel instance serves the layers
// whose storage mode is MODE and whose pointers allow 16-byte accesses; other tiles are
// skipped (another instance, or the generic kernel, takes them).
template <int RC, int MODE>
__global__ void __launch_bounds__(kRmwThreads, (RC <= 8 ? 2 : 1))
rmw_reg_kernel(const DevLayer* layers, const int* tile_start,
               int n_layers, int total_tiles, int tile_rows, uint64_t seed, PassCoef coef_of,
               int pair_update) {
  extern __shared__ __align__(16) float smem[];
  __shared__ DevLayer sL;
  float* sG = smem;
  chain_wait();
  const float coef = coef_of.value();
  for (int tile = blockIdx.x; tile < total_tiles; tile += gridDim.x) {
    const int li = find_layer(tile_start, n_layers, tile);
    __syncthreads();   // previous tile is done with sG and sL
    fetch_layer(&sL, layers + li);
    __syncthreads();
    const DevLayer& L = sL;
    if (!L.vec_ok || effective_mode(L, pair_update) != MODE) continue;
    const int t = tile - L.tile0;
    const int tr = t / L.tiles_c, tc = t - tr * L.tiles_c;
    const int row0 = tr * tile_rows, col0 = tc * kTileCols;
    const int nrows = min(tile_rows, L.d_out - row0);
    TileReg<RC, MODE> body;
    body.begin(L, row0, nrows, col0);
    generate_G<2>(sG, RC, L.r, row0, nrows, L.layer_id, seed);
    __syncthreads();
    body.run(L, sG, row0, nrows, coef);
  }
}

template <int MODE>
__global__ void __launch_bounds__(kRmwThreads, 1)
rmw_smem_kernel(const DevLayer* layers, const int* tile_start,
                int n_layers, int total_tiles, int tile_rows, int max_rs, uint64_t seed, PassCoef coef_of,
                int pair_update) {
  extern __shared__ __align__(16) float smem[];
  __shared__ DevLayer sL;
  float* sG = smem;                              // [kTileRows][RS]
  float* sV = smem + kTileRows * max_rs;         // [RS][kTileCols]
  chain_wait();
  const float coef = coef_of.value();
  for (int tile = blockIdx.x; tile < total_tiles; tile += gridDim.x) {
    const int li = find_layer(tile_start, n_layers, tile);
    __syncthreads();
    fetch_layer(&sL, layers + li);
    __syncthreads();
    const DevLayer& L = sL;
    if (!L.vec_ok || effective_mode(L, pair_update) != MODE) continue;
    const int RS = (L.r + 3) & ~3;
    const int t = tile - L.tile0;
    const int tr = t / L.tiles_c, tc = t - tr * L.tiles_c;
    const int row0 = tr * tile_rows, col0 = tc * kTileCols;
    const int nrows = min(tile_rows, L.d_out - row0);
    generate_G<1>(sG, RS, L.r, row0, nrows, L.layer_id, seed);
    for (int i = threadIdx.x; i < RS * kTileCols; i += kRmwThreads) {
      const int k = i / kTileCols, c = i - k * kTileCols;
      sV[i] = (k < L.r && col0 + c < L.d_in) ? __ldcg(L.V + (long long)k * L.ldv + col0 + c) : 0.f;
    }
    __syncthreads();
    tile_body_smem<MODE>(L, sG, sV, RS, row0, nrows, col0, coef);
  }
}

// Any pitch, alignment, storage mode and rank, element by element: layers that the vector kernels cannot take.  A thread has two columns
// of the tile, 256 apart, and eight rows at a time: their weights are asked for, R's products formed meanwhile, sixteen ranks of A^T in
// registers at a time (read again for every eight rows where there are more).  Five 1500 x 1500 fp32 layers, r = 16, with a row at a time and
// A^T from L2 for each of its products: 132 us, now 43; twelve 2047 x 2047 pairs, r = 16, 475 -> 216.
constexpr int kGenRows = 8, kGenRanks = 16;
__global__ void __launch_bounds__(kRmwThreads)
rmw_generic_kernel(const DevLayer* layers, const int* tile_start,
                   int n_layers, int total_tiles, int tile_rows, uint64_t seed, PassCoef coef_of,
                   int pair_update) {
  __shared__ __align__(16) float sG[32 * AGZO_MAX_RANK];
  __shared__ DevLayer sL;
  chain_wait();
  const float coef = coef_of.value();
  for (int tile = blockIdx.x; tile < total_tiles; tile += gridDim.x) {
    const int li = find_layer(tile_start, n_layers, tile);
    __syncthreads();
    fetch_layer(&sL, layers + li);
    __syncthreads();
    const DevLayer& L = sL;
    if (L.vec_ok) continue;
    const int mode = effective_mode(L, pair_update);
    const int r = L.r, RS = (r + kGenRanks - 1) / kGenRanks * kGenRanks;       // zero beyond r
    const int t = tile - L.tile0;
    const int tr = t / L.tiles_c, tc = t - tr * L.tiles_c;
    const int row0 = tr * tile_rows, col0 = tc * kTileCols;
    const int nrows = min(tile_rows, L.d_out - row0);
    const __nv_bfloat16* Wb = reinterpret_cast<const __nv_bfloat16*>(L.W);
    const float* Wf = reinterpret_cast<const float*>(L.W);
    for (int sb = 0; sb < nrows; sb += 32) {
      const int nr = min(32, nrows - sb);
      __syncthreads();
      generate_G<1>(sG, RS, r, row0 + sb, nr, L.layer_id, seed);
      __syncthreads();
      for (int c = threadIdx.x; c < kTileCols; c += kRmwThreads) {
        const int col = col0 + c;
        if (col >= L.d_in) break;
        for (int r0 = 0; r0 < nr; r0 += kGenRows) {
          const long long at = (long long)(row0 + sb + r0) * L.ldw + col;
          float w[kGenRows], z[kGenRows];
#pragma unroll
          for (int j = 0; j < kGenRows; ++j) {
            z[j] = 0.f;
            w[j] = r0 + j >= nr ? 0.f : mode == RMW_BF16 ? __bfloat162float(Wb[at + j * L.ldw]) : Wf[at + j * L.ldw];
          }
          for (int k0 = 0; k0 < r; k0 += kGenRanks) {
            float v[kGenRanks];
#pragma unroll
            for (int k = 0; k < kGenRanks; ++k) v[k] = k0 + k < r ? L.V[(long long)(k0 + k) * L.ldv + col] : 0.f;
#pragma unroll
            for (int j = 0; j < kGenRows; ++j) {
              const float4* g = reinterpret_cast<const float4*>(sG + (r0 + j < nr ? r0 + j : 0) * RS + k0);
#pragma unroll
              for (int k = 0; k < kGenRanks; k += 4) {           // k ascending, fixed order
                const float4 q = g[k / 4];
                z[j] = fmaf(q.x, v[k], z[j]); z[j] = fmaf(q.y, v[k + 1], z[j]);
                z[j] = fmaf(q.z, v[k + 2], z[j]); z[j] = fmaf(q.w, v[k + 3], z[j]);
              }
            }
          }
#pragma unroll
          for (int j = 0; j < kGenRows; ++j) {
            if (r0 + j >= nr) break;
            const float o = fmaf(coef, z[j], w[j]);
            if (mode == RMW_BF16) reinterpret_cast<__nv_bfloat16*>(L.W)[at + j * L.ldw] = __float2bfloat16_rn(o);
            if (mode == RMW_F32 || mode == RMW_PAIR_UPDATE) reinterpret_cast<float*>(L.W)[at + j * L.ldw] = o;
            if (mode == RMW_PAIR_COMPUTE || mode == RMW_PAIR_UPDATE)
              reinterpret_cast<__nv_bfloat16*>(L.W16)[(long long)(row0 + sb + r0 + j) * L.ldw16 + col] = __float2bfloat16_rn(o);
          }
        }
      }
    }
  }
}

struct RmwArgs {
  const DevLayer* d_layers; const int* d_tile_start; int n_layers, total_tiles, tile_rows;
  uint64_t seed; PassCoef coef; int pair_update; int sm_count;
};

// A pass of one tile per CTA may start beside its predecessor.  A longer one may not: CTAs that take their places one by
// one while the panel QR runs out drift apart and the pass loses the locality of its row segments (rank-1 pass over eight
// 8B-shaped blocks behind the extraction: 970 us, 1190 us when started early).
static int starts_early(int total_tiles, int grid) { return total_tiles <= grid ? 1 : 0; }

template <int RC, int MODE>
static cudaError_t launch_reg(const RmwArgs& a, cudaStream_t s) {
  const int per_sm = RC <= 8 ? 2 : 1;
  const int grid = a.total_tiles < a.sm_count * per_sm ? a.total_tiles : a.sm_count * per_sm;
  const size_t smem = (size_t)a.tile_rows * RC * 2 * sizeof(float);
  return launch_kernel(rmw_reg_kernel<RC, MODE>, dim3(grid), kRmwThreads, smem, 0, starts_early(a.total_tiles, grid), s, a.d_layers, a.d_tile_start, a.n_layers,
                        a.total_tiles, a.tile_rows, a.seed, a.coef, a.pair_update);
}

template <int MODE>
static cudaError_t launch_mode(const RmwArgs& a, int max_r, cudaStream_t s) {
  if (max_r <= 1) return launch_reg<1, MODE>(a, s);
  if (max_r <= 2) return launch_reg<2, MODE>(a, s);
  if (max_r <= 4) return launch_reg<4, MODE>(a, s);
  if (max_r <= 8) return launch_reg<8, MODE>(a, s);
  if (max_r <= 16) return launch_reg<16, MODE>(a, s);
  const int max_rs = (max_r + 3) & ~3;
  const size_t smem = ((size_t)kTileRows * max_rs + (size_t)max_rs * kTileCols) * sizeof(float);
  const int grid = a.total_tiles < a.sm_count ? a.total_tiles : a.sm_count;
  return launch_kernel(rmw_smem_kernel<MODE>, dim3(grid), kRmwThreads, smem, 0, starts_early(a.total_tiles, grid), s, a.d_layers, a.d_tile_start, a.n_layers,
                        a.total_tiles, a.tile_rows, max_rs, a.seed, a.coef, a.pair_update);
}

cudaError_t launch_rmw(const DevLayer* d_layers, const int* d_tile_start, int n_layers,
                       int total_tiles, int tile_rows, int slow_rows, int max_r, int fast_mode_mask, bool any_slow,
                       uint64_t seed, PassCoef coef, bool pair_update, int sm_count, cudaStream_t s) {
  if (total_tiles <= 0) return cudaSuccess;
  RmwArgs a{d_layers, d_tile_start, n_layers, total_tiles, tile_rows, seed, coef, pair_update ? 1 : 0, sm_count};
  cudaError_t e = cudaSuccess;
  if (pair_update && (fast_mode_mask & (1 << RMW_PAIR_COMPUTE)))
    fast_mode_mask = (fast_mode_mask & ~(1 << RMW_PAIR_COMPUTE)) | (1 << RMW_PAIR_UPDATE);
  if (e == cudaSuccess && (fast_mode_mask & (1 << RMW_BF16))) e = launch_mode<RMW_BF16>(a, max_r, s);
  if (e == cudaSuccess && (fast_mode_mask & (1 << RMW_F32))) e = launch_mode<RMW_F32>(a, max_r, s);
  if (e == cudaSuccess && (fast_mode_mask & (1 << RMW_PAIR_COMPUTE))) e = launch_mode<RMW_PAIR_COMPUTE>(a, max_r, s);
  if (e == cudaSuccess && (fast_mode_mask & (1 << RMW_PAIR_UPDATE))) e = launch_mode<RMW_PAIR_UPDATE>(a, max_r, s);
  if (e == cudaSuccess && any_slow) {
    const int grid = total_tiles < sm_count * 4 ? total_tiles : sm_count * 4;
    e = launch_kernel(rmw_generic_kernel, dim3(grid), kRmwThreads, 0, 0, starts_early(total_tiles, grid), s, d_layers, d_tile_start, n_layers, total_tiles,
                       slow_rows, seed, coef, pair_update ? 1 : 0);
  }
  return e;
}

cudaError_t rmw_init() {
  const int smem = (int)(((size_t)kTileRows * 64 + (size_t)64 * kTileCols) * sizeof(float));
  cudaError_t e = cudaFuncSetAttribute(rmw_smem_kernel<RMW_BF16>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
  if (e == cudaSuccess) e = cudaFuncSetAttribute(rmw_smem_kernel<RMW_F32>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
  if (e == cudaSuccess) e = cudaFuncSetAttribute(rmw_smem_kernel<RMW_PAIR_COMPUTE>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
  if (e == cudaSuccess) e = cudaFuncSetAttribute(rmw_smem_kernel<RMW_PAIR_UPDATE>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
  return e;
}

// ------------------------------------------------------------------ dense direction (second case of Eq. agzo-perturb)
// w <- w + c u, u ~ N(0, I) from (seed, layer_id, tag 2), element e = word e & 3 of block e >> 2.
// Scalar form: any pointer, blocks [b_first, b_end).
template <typename T>
__global__ void dense_kernel(T* w, long long n, long long b_first, uint64_t seed, uint32_t layer_id, float scale,
                             const float* d_scale) {
  chain_wait();
  const float c = d_scale ? scale * __ldcg(d_scale) : scale;
  const long long nb = (n + 3) >> 2;
  for (long long b = b_first + blockIdx.x * (long long)blockDim.x + threadIdx.x; b < nb;
       b += (long long)gridDim.x * blockDim.x) {
    const float4 g = gaussian_block((uint64_t)b, layer_id, kTagDense, seed);
    const float gv[4] = {g.x, g.y, g.z, g.w};
#pragma unroll
    for (int lane = 0; lane < 4; ++lane) {
      const long long e = 4 * b + lane;
      if (e < n) w[e] = (T)fmaf(c, gv[lane], (float)w[e]);
    }
  }
}

// Vector form for 16-byte aligned vectors: a thread takes eight consecutive elements (two Philox blocks), one 16-byte load and
// store for bf16, two for fp32.  A long vector is bound by the arithmetic of one Philox + Box-Muller normal per weight, not by HBM
// (67 M weights: 142 us with logf, sqrtf and sincospif, 119 with one pair of normals after another and a grid that stays resident, 97 now; HBM would
// allow 41); a short one by its launch, so the normals are made, and the weights asked for as far as L2, before the kernel waits
// for its predecessor.  Every thread has one step: with a share of the vector per resident thread the scheduler runs some warps far ahead
// of others, and the SM ends on few (121 -> 109 us for that alone, 105 with 32-bit block numbers).
// hi: upper word of the block numbers, the same in the whole launch, so that what the first two rounds of Philox make of it is made once.
template <typename T>
__global__ void __launch_bounds__(256) dense_vec_kernel(T* w, uint32_t n8, uint32_t hi, uint64_t seed, uint32_t layer_id, float scale,
                                                        const float* d_scale) {
  const uint32_t g = blockIdx.x * 256u + threadIdx.x;
  if (g < n8) asm volatile("prefetch.global.L2 [%0];" ::"l"(w + 8 * (size_t)g));
  const uint64_t b = (uint64_t)hi << 32 | 2u * g;
  const float4 ga = gaussian_block(b, layer_id, kTagDense, seed), gb = gaussian_block(b | 1u, layer_id, kTagDense, seed);
  chain_wait();
  if (g >= n8) return;
  const float c = d_scale ? scale * __ldcg(d_scale) : scale;
  const float u[8] = {ga.x, ga.y, ga.z, ga.w, gb.x, gb.y, gb.z, gb.w};
  if constexpr (sizeof(T) == 2) {
    uint4* p = reinterpret_cast<uint4*>(w) + g;
    const uint4 v = *p;
    const uint32_t in[4] = {v.x, v.y, v.z, v.w};
    uint32_t out[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      const float w0 = __uint_as_float(in[k] << 16), w1 = __uint_as_float(in[k] & 0xFFFF0000u);
      __nv_bfloat162 r = __floats2bfloat162_rn(fmaf(c, u[2 * k], w0), fmaf(c, u[2 * k + 1], w1));
      out[k] = *reinterpret_cast<uint32_t*>(&r);
    }
    *p = make_uint4(out[0], out[1], out[2], out[3]);
  } else {
    float4* p = reinterpret_cast<float4*>(w) + 2 * (size_t)g;
    float4 a = p[0], b2 = p[1];
    a.x = fmaf(c, u[0], a.x); a.y = fmaf(c, u[1], a.y); a.z = fmaf(c, u[2], a.z); a.w = fmaf(c, u[3], a.w);
    b2.x = fmaf(c, u[4], b2.x); b2.y = fmaf(c, u[5], b2.y); b2.z = fmaf(c, u[6], b2.z); b2.w = fmaf(c, u[7], b2.w);
    p[0] = a; p[1] = b2;
  }
}

template <typename T>
cudaError_t launch_dense_t(T* w, long long n, uint64_t seed, uint32_t layer_id, float scale, const float* d_scale,
                           int sm_count, cudaStream_t s) {
  const long long cap = (long long)sm_count * 8;      // eight resident blocks of 256 threads per SM
  long long n8 = 0;
  if ((reinterpret_cast<uintptr_t>(w) & 15u) == 0) n8 = n >> 3;
  constexpr long long kLaunch8 = 1ll << 31;           // steps of a launch: 2^32 blocks, which share their upper word
  for (long long at = 0; at < n8; at += kLaunch8) {
    const uint32_t steps = (uint32_t)(n8 - at < kLaunch8 ? n8 - at : kLaunch8);
    cudaError_t e = launch_chained(dense_vec_kernel<T>, dim3((steps + 255u) / 256u), 256, 0, 0, s, w + 8 * at, steps,
                                   (uint32_t)(at / kLaunch8), seed, layer_id, scale, d_scale);
    if (e != cudaSuccess) return e;
  }
  if (8 * n8 < n) {                                    // the rest: blocks from 2 n8 on
    const long long nb = ((n + 3) >> 2) - 2 * n8;
    const int grid = (int)((nb + 255) / 256 < cap ? (nb + 255) / 256 : cap);
    return launch_chained(dense_kernel<T>, dim3(grid), 256, 0, 0, s, w, n, 2 * n8, seed, layer_id, scale, d_scale);
  }
  return cudaSuccess;
}

cudaError_t launch_dense(void* w, long long n, int dtype, uint64_t seed, uint32_t layer_id,
                         float scale, const float* d_scale, int sm_count, cudaStream_t s) {
  if (n <= 0) return cudaSuccess;
  if (dtype == AGZO_BF16)
    return launch_dense_t<__nv_bfloat16>((__nv_bfloat16*)w, n, seed, layer_id, scale, d_scale, sm_count, s);
  return launch_dense_t<float>((float*)w, n, seed, layer_id, scale, d_scale, sm_count, s);
}

// ------------------------------------------------------------------ Gaussian right factor (LOZO comparison)
__global__ void fill_basis_kernel(const DevLayer* layers, uint64_t seed) {
  chain_wait();
  const DevLayer& L = layers[blockIdx.y];
  const long long n = (long long)L.r * L.d_in;
  const long long nb = (n + 3) >> 2;
  for (long long b = blockIdx.x * (long long)blockDim.x + threadIdx.x; b < nb;
       b += (long long)gridDim.x * blockDim.x) {
    const float4 g = gaussian_block((uint64_t)b, L.layer_id, kTagBasis, seed);
    const float gv[4] = {g.x, g.y, g.z, g.w};
#pragma unroll
    for (int lane = 0; lane < 4; ++lane) {
      const long long e = 4 * b + lane;
      if (e < n) {
        const long long k = e / L.d_in;
        L.V[k * L.ldv + (e - k * L.d_in)] = gv[lane];
      }
    }
  }
}

cudaError_t launch_fill_basis(const DevLayer* d_layers, int n_layers, int max_elems, uint64_t seed, cudaStream_t s) {
  if (n_layers <= 0) return cudaSuccess;
  int gx = (max_elems / 4 + 255) / 256;
  if (gx < 1) gx = 1;
  if (gx > 64) gx = 64;
  return launch_chained(fill_basis_kernel, dim3((unsigned)gx, (unsigned)n_layers), 256, 0, 0, s, d_layers, seed);
}

// ------------------------------------------------------------------ scalars (Algorithm 2, step 3)
__global__ void ghat_kernel(const double* fp, const double* fo, float eps, int mode, float* g) {
  chain_wait();
  const double d = *fp - *fo;
  *g = (float)(mode == 0 ? d / (2.0 * (double)eps) : d / (double)eps);
}
cudaError_t launch_ghat(const double* fp, const double* fo, float eps, int mode, float* g, cudaStream_t s) {
  return launch_chained(ghat_kernel, dim3(1), 1, 0, 0, s, fp, fo, eps, mode, g);
}

// ------------------------------------------------------------------ test exports
__global__ void debug_early_copy_kernel(const uint4* src, uint4* dst, uint64_t n16) {
  for (uint64_t i = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; i < n16; i += (uint64_t)gridDim.x * blockDim.x) dst[i] = __ldcg(src + i);
  chain_wait();
}
cudaError_t launch_debug_early_copy(const void* src, void* dst, uint64_t n16, int sm_count, cudaStream_t s) {
  if (n16 == 0) return cudaSuccess;
  const uint64_t cap = (uint64_t)sm_count;
  const unsigned grid = (unsigned)((n16 + 255) / 256 < cap ? (n16 + 255) / 256 : cap);
  return launch_chained(debug_early_copy_kernel, dim3(grid), 256, 0, 0, s, static_cast<const uint4*>(src), static_cast<uint4*>(dst), n16);
}
__global__ void debug_philox_kernel(uint64_t seed, uint32_t layer, uint32_t tag, uint64_t first,
                                    uint64_t n, uint32_t* out) {
  for (uint64_t i = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; i < n;
       i += (uint64_t)gridDim.x * blockDim.x) {
    const uint64_t e = first + i;
    const uint4 w = philox4x32_10(e >> 2, layer, tag, seed);
    const uint32_t wv[4] = {w.x, w.y, w.z, w.w};
    out[i] = wv[e & 3];
  }
}
__global__ void debug_gauss_kernel(uint64_t seed, uint32_t layer, uint32_t tag, uint64_t first,
                                   uint64_t n, float* out) {
  for (uint64_t i = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; i < n;
       i += (uint64_t)gridDim.x * blockDim.x) {
    const uint64_t e = first + i;
    const float4 g = gaussian_block(e >> 2, layer, tag, seed);
    const float gv[4] = {g.x, g.y, g.z, g.w};
    out[i] = gv[e & 3];
  }
}
__global__ void debug_normal_parts_kernel(uint32_t first, uint32_t n, float4* out) {
  for (uint32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) out[i] = normal_parts(first + i);
}
cudaError_t launch_debug_normal_parts(uint32_t first, uint32_t n, float* out, int sm_count, cudaStream_t s) {
  if (n == 0) return cudaSuccess;
  const uint32_t cap = (uint32_t)sm_count * 8, want = (n + 255) / 256;
  debug_normal_parts_kernel<<<want < cap ? want : cap, 256, 0, s>>>(first, n, reinterpret_cast<float4*>(out));
  return cudaGetLastError();
}
cudaError_t launch_debug_philox(uint64_t seed, uint32_t layer, uint32_t tag, uint64_t first,
                                uint64_t n, uint32_t* out, int sm_count, cudaStream_t s) {
  if (n == 0) return cudaSuccess;
  const uint64_t cap = (uint64_t)sm_count * 8;
  const int grid = (int)((n + 255) / 256 < cap ? (n + 255) / 256 : cap);
  debug_philox_kernel<<<grid, 256, 0, s>>>(seed, layer, tag, first, n, out);
  return cudaGetLastError();
}
cudaError_t launch_debug_gauss(uint64_t seed, uint32_t layer, uint32_t tag, uint64_t first,
                               uint64_t n, float* out, int sm_count, cudaStream_t s) {
  if (n == 0) return cudaSuccess;
  const uint64_t cap = (uint64_t)sm_count * 8;
  const int grid = (int)((n + 255) / 256 < cap ? (n + 255) / 256 : cap);
  debug_gauss_kernel<<<grid, 256, 0, s>>>(seed, layer, tag, first, n, out);
  return cudaGetLastError();
}

}  // namespace agzo

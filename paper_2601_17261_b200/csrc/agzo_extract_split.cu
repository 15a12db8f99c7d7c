// The two products of Algorithm 1 in fp32 precision on the tensor cores: for fp32 activations, and for bf16 ones that the
// TMA kernels (agzo_extract_tc.cu) do not take.
//
// An fp32 number is three bf16 parts; X becomes three planes on its way from registers into shared memory, Q and T three operand
// rows each, and of their nine products the six down to 2^-24 are formed (the splitting of G. Henry, P. T. P. Tang and A. Heinecke,
// "Leveraging the bfloat16 artificial intelligence datatype for higher-precision computations", ARITH 2019).  bf16 X is one plane.  The
// tensor core truncates when it accumulates, so an accumulator covers 64 of the contracted dimension only, the smallest plane
// first; the accumulators are added up in registers, with rounding, the three parts' columns apart until the end.
//
// A persistent CTA per SM walks over work items: 128 tokens and all columns of a unit for T = X Q, 128 columns and a token slab for
// Y = X^T T; a unit is the layers that read one X, up to 24 ranks of them.  16 loader warps in two groups take turns at steps of 64 of the
// contracted dimension: eight 16-byte loads per thread, each register asked for again as soon as it has been converted, so that 32 to
// 64 KB are in flight; a warp per four ranks makes the operand's rows, one issues the products, eight take the accumulators in.
// A step of 32 KB of fp32 takes 1400 to 1800 cycles, of which the copy rate would allow 1400: what bounds it is the round trip of a stage
// (converted, multiplied, free again) through the two or three others there is room for; leaving out the loads, the conversion or the products
// changes little.  All units of a launch run the widest one's instance; with NP = 16 and 24 (928 and 992 threads) a thread has 64 registers, and the
// instances of X^T T on fp32 spill 28 and 24 bytes, those of NP = 24 on bf16 4 (X^T T) and 8 (X Q).
// Two fp32 blocks of 0.6B shape (229 MB), 4000 tokens, r = 8: X^T T 67 -> 57 us, X Q 93 -> 68, the step 692 -> 590;
// r = 16 on 4000 x 3072, two layers, K = 1: 133 -> 100 us for the extraction; 5000 x 1001 in bf16, r = 8: 226 -> 122.
// Error against 64 bits, 172 bases of 60 lists: 1.2e-7 root mean square, the CUDA-core kernels 1.4e-7.
// Units go from the widest to the narrowest in T = X Q and back in Y = X^T T, so that what is left of X in L2 serves the next product.
#include "agzo_split.cuh"

#include <algorithm>
#include <mutex>
#include <vector>

#include "agzo_ptx.cuh"

namespace agzo {

namespace {

using namespace ptx;

constexpr int kLoadGroups = 2, kGroupWarps = 8, kEpiWarps = 8;
constexpr int kLoadWarps = kLoadGroups * kGroupWarps;
constexpr int kMmaWarp = kLoadWarps + kEpiWarps, kOpWarp0 = kMmaWarp + 1;
constexpr int kStep = 64;                        // of the contracted dimension
constexpr int kPlaneBytes = 16 * 1024;           // 128 x 64 bf16
constexpr int kAcc = 4;                          // accumulators in TMEM
constexpr int kMaxStages = 4;
constexpr int kMaxSplit = 4;                     // CTAs of a cluster that share an item of T = X Q

template <int NP, int PLANES, bool XQ> struct Cfg {
  static constexpr int NB = (3 * NP + 15) & ~15;           // operand rows, columns of an accumulator
  static constexpr int op_warps = NP / 4, threads = (kOpWarp0 + op_warps) * 32;
  static constexpr int stage_bytes = PLANES * kPlaneBytes + (NB * 128 + 1023) / 1024 * 1024;
  static constexpr int peer_bytes = XQ ? kEpiWarps * 32 * NP / 2 * 4 : 0;    // sums of T of another CTA of the cluster
  static constexpr int fit = (225 * 1024 - (kMaxSplit - 1) * peer_bytes) / stage_bytes, stages = fit < kMaxStages ? fit : kMaxStages;
  static constexpr size_t smem = (size_t)stages * stage_bytes + 1024;       // and the sums of the peers that there are
  static constexpr uint32_t tmem_cols = kAcc * NB <= 128 ? 128u : kAcc * NB <= 256 ? 256u : 512u;
};

struct Shared {
  uint64_t full[kMaxStages], empty[kMaxStages], acc_full[kAcc], acc_empty[kAcc];
  uint64_t sums_in, sums_out;    // of the other CTAs are here; this one's may be sent
  uint32_t tmem_base;
  int failed;
};

__device__ __forceinline__ uint32_t bf16_pair(float a, float b) {
  const __nv_bfloat162 v = __floats2bfloat162_rn(a, b);
  return *reinterpret_cast<const uint32_t*>(&v);
}

// A work item: its unit, and 128 rows (tokens of T = X Q, columns of Y = X^T T) times the range [k_begin, k_end) of the contracted dimension
struct Item {
  int unit, row0, k_begin, k_end, slab;
};
template <bool XQ, int N>
__device__ __forceinline__ Item item_of(const SplitUnits<N>& U, int it) {
  // the last unit that starts at or before it: 32 at a time
  const int lane = threadIdx.x & 31;
  Item x;
  x.unit = 0;
  for (int b = 0; b < U.n_units; b += 32) {
    const int k = b + lane;
    const unsigned before = __ballot_sync(0xffffffffu, k < U.n_units && U.unit[k < U.n_units ? k : 0].item0 <= it);
    if (!before) break;
    x.unit = b + 31 - __clz(before);
  }
  const SplitUnit& s = U.unit[x.unit];
  const int local = it - s.item0;
  if (XQ) {                               // the CTAs of a cluster take a share of the columns each
    const int n = (s.d_in + kStep - 1) / kStep, c = U.split > 1 ? (int)cluster_ctarank() : 0;
    x.row0 = 128 * local;
    x.k_begin = c * n / U.split * kStep; x.k_end = min(s.d_in, (c + 1) * n / U.split * kStep);
    x.slab = 0;
  } else {                                // slabs from the last on, all columns of one after another
    const int blocks = (s.d_in + 127) / 128, s_back = local / blocks;
    x.slab = s.slabs - 1 - s_back;
    x.row0 = 128 * (local - s_back * blocks);
    x.k_begin = x.slab * s.slab_rows;
    x.k_end = min(s.m, x.k_begin + s.slab_rows);
  }
  return x;
}
// items of this CTA or cluster, back and forth over them: i-th one, or -1
template <int N>
__device__ __forceinline__ int nth_item(const SplitUnits<N>& U, int i) {
  const int G = (int)gridDim.x / U.split, id = (int)blockIdx.x / U.split, b = (i & 1) ? G - 1 - id : id;
  const long long it = (long long)i * G + b;
  return it < U.n_items ? (int)it : -1;
}
__device__ __forceinline__ int steps_of(const Item& x) { return (x.k_end - x.k_begin + kStep - 1) / kStep; }
// the layer of panel rank k of a unit, and which rank of that layer it is
__device__ __forceinline__ int layer_of(const SplitUnit& s, int k, int* kl) {
  int l = 0, left = s.k0 + k;
#pragma unroll
  for (int x = 0; x < kSplitMaxLayers - 1; ++x)
    if (l == x && left >= s.layer[x].r) { left -= s.layer[x].r; ++l; }
  *kl = left;
  return l;
}

// The steps of a CTA, one after another over its items; a loader group takes every kLoadGroups-th
template <bool XQ, int N>
struct Walk {
  int i, it, step, n_steps;
  Item x;
  __device__ __forceinline__ void open(const SplitUnits<N>& U) {
    if (it >= 0) { x = item_of<XQ>(U, it); n_steps = steps_of(x); }
  }
  __device__ __forceinline__ void start(const SplitUnits<N>& U) {
    i = 0; step = 0; n_steps = 0;
    it = nth_item(U, 0);
    open(U);
    advance(U, 0);
  }
  // by n steps, over items without any; whether the item changed
  __device__ __forceinline__ bool advance(const SplitUnits<N>& U, int n) {
    step += n;
    bool moved = false;
    while (it >= 0 && step >= n_steps) {
      step -= n_steps;
      it = nth_item(U, ++i);
      open(U);
      moved = true;
    }
    return moved;
  }
};

// what a loader thread reads of X: four columns of a row, in fp32 or bf16
template <int PLANES> struct X4;
template <> struct X4<3> { float4 v; };
template <> struct X4<1> { uint2 v; };

template <int PLANES> struct Elem;
template <> struct Elem<3> { using type = float; };
template <> struct Elem<1> { using type = unsigned short; };
// as one access, or element by element with zeros from the left-th on
__device__ __forceinline__ X4<3> fetch_x(const float* p) {
  X4<3> r;
  asm volatile("ld.global.nc.L1::no_allocate.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(r.v.x), "=f"(r.v.y), "=f"(r.v.z), "=f"(r.v.w) : "l"(p));
  return r;
}
__device__ __forceinline__ X4<1> fetch_x(const unsigned short* p) {
  X4<1> r;
  asm volatile("ld.global.nc.L1::no_allocate.v2.u32 {%0, %1}, [%2];" : "=r"(r.v.x), "=r"(r.v.y) : "l"(p));
  return r;
}
__device__ __forceinline__ X4<3> fetch_x(const float* p, int left) {
  X4<3> r;
  r.v = make_float4(left > 0 ? p[0] : 0.f, left > 1 ? p[1] : 0.f, left > 2 ? p[2] : 0.f, left > 3 ? p[3] : 0.f);
  return r;
}
__device__ __forceinline__ X4<1> fetch_x(const unsigned short* p, int left) {
  X4<1> r;
  const uint32_t a = left > 0 ? p[0] : 0u, b = left > 1 ? p[1] : 0u, c = left > 2 ? p[2] : 0u, d = left > 3 ? p[3] : 0u;
  r.v = make_uint2(a | b << 16, c | d << 16);
  return r;
}
__device__ __forceinline__ void st_shared_v2(uint32_t at, uint32_t a, uint32_t b) {
  asm volatile("st.shared.v2.b32 [%0], {%1, %2};" ::"r"(at), "r"(a), "r"(b) : "memory");
}
// a - its bf16 pair, both numbers
__device__ __forceinline__ uint64_t less_pair(uint64_t v, uint32_t pair) {
  return fma_f32x2(pack_f32x2(__uint_as_float(pair << 16), __uint_as_float(pair & 0xffff0000u)), pack_f32x2(-1.f, -1.f), v);
}
__device__ __forceinline__ uint32_t bf16_pair(uint64_t v) {
  float a, b;
  unpack_f32x2(v, a, b);
  return bf16_pair(a, b);
}
// into the planes, plane p at `at` + p kPlaneBytes
template <int PLANES>
__device__ __forceinline__ void put_x(const X4<PLANES>& x, uint32_t at) {
  if constexpr (PLANES == 1) {
    st_shared_v2(at, x.v.x, x.v.y);
  } else {
    uint64_t v = pack_f32x2(x.v.x, x.v.y), w = pack_f32x2(x.v.z, x.v.w);
#pragma unroll
    for (int p = 0; p < 3; ++p) {
      const uint32_t a = bf16_pair(v), b = bf16_pair(w);
      st_shared_v2(at + (uint32_t)(p * kPlaneBytes), a, b);
      if (p < 2) { v = less_pair(v, a); w = less_pair(w, b); }
    }
  }
}

__device__ __forceinline__ void mbar_arrive_remote(uint32_t bar) {
  asm volatile("mbarrier.arrive.release.cluster.shared::cluster.b64 _, [%0];" ::"r"(bar) : "memory");
}
// H consecutive fp32 columns of this warp's 32 TMEM lanes; issues the loads only
template <int H>
__device__ __forceinline__ void tmem_ld_cols(uint32_t at, uint32_t (&z)[H]) {
  static_assert(H == 4 || H == 8 || H == 12, "");
  if constexpr (H >= 8)
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
                 : "=r"(z[0]), "=r"(z[1]), "=r"(z[2]), "=r"(z[3]), "=r"(z[4]), "=r"(z[5]), "=r"(z[6]), "=r"(z[7])
                 : "r"(at));
  if constexpr (H != 8)
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x4.b32 {%0, %1, %2, %3}, [%4];"
                 : "=r"(z[H - 4]), "=r"(z[H - 3]), "=r"(z[H - 2]), "=r"(z[H - 1])
                 : "r"(at + (uint32_t)(H - 4)));
}

template <int NP, int PLANES, bool XQ, int N>
__global__ void __launch_bounds__(Cfg<NP, PLANES, XQ>::threads, 1) split_product_kernel(const __grid_constant__ SplitUnits<N> U, DevStatus* status) {
  extern __shared__ __align__(1024) uint8_t smem_raw[];
  __shared__ Shared sh;
  using C = Cfg<NP, PLANES, XQ>;
  constexpr int NB = C::NB, kStages = C::stages, kStageBytes = C::stage_bytes;
  const uint32_t tiles = (smem_u32(smem_raw) + 1023u) & ~1023u;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (threadIdx.x == 0) {
    for (int s = 0; s < kStages; ++s) { mbar_init(&sh.full[s], kGroupWarps + C::op_warps + (U.split == 1 ? U.missing : 0u)); mbar_init(&sh.empty[s], 1); }
    for (int b = 0; b < kAcc; ++b) { mbar_init(&sh.acc_full[b], 1); mbar_init(&sh.acc_empty[b], kEpiWarps); }
    mbar_init(&sh.sums_in, 1);
    mbar_init(&sh.sums_out, kEpiWarps);
    sh.failed = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    fence_proxy_async();
  }
  if (warp == kMmaWarp) tmem_alloc(&sh.tmem_base, C::tmem_cols);
  tc_fence_before();
  __syncthreads();
  if (XQ && U.split > 1) cluster_sync_all();               // the barriers are ready for the peers
  tc_fence_after();
  const uint32_t tmem = sh.tmem_base;

  if (warp < kLoadWarps) {
    // ---------------------------------------------------------------- loaders
    const int group = warp / kGroupWarps, w = warp % kGroupWarps, tid = w * 32 + lane;
    // T = X Q: 16 lanes to a row of 64 columns, rows 16 apart; Y = X^T T: a warp to a row of 128 columns, rows 8 apart
    constexpr int kRowStep = XQ ? 16 : 8;
    const int row = XQ ? tid >> 4 : tid >> 5, c4 = XQ ? tid & 15 : tid & 31;
    const uint32_t place = (uint32_t)((XQ ? 0 : (c4 >> 4) * (kPlaneBytes / 2)) + row * 128 + ((((c4 & 15) >> 1) ^ (row & 7)) << 4) + (c4 & 1) * 8);
    using T = typename Elem<PLANES>::type;
    Walk<XQ, N> at;
    at.start(U);
    at.advance(U, group);
    X4<PLANES> v[8];
    // of the item: X at this thread's first row and column of the step, the steps between rows and between this group's turns
    const T* x = nullptr;
    long long row_step = 0, turn = 0;
    bool vec = false, whole = false;       // whole: all rows and columns of the item's 128 are inside
    auto open = [&]() {
      const SplitUnit& L = U.unit[at.x.unit];
      vec = L.vec != 0;
      whole = vec && at.x.row0 + 128 <= L.rows;
      row_step = kRowStep * L.ldx;
      turn = kLoadGroups * (XQ ? (long long)kStep : kStep * L.ldx);
      const int k0 = at.x.k_begin + at.step * kStep;
      x = reinterpret_cast<const T*>(L.X) + (XQ ? (long long)(at.x.row0 + row) * L.ldx + k0 + 4 * c4 : (long long)(k0 + row) * L.ldx + at.x.row0 + 4 * c4);
    };
    // a step that ends an item or the matrix: rows of X beyond m are read as the last one (nothing of them is stored in T, or they meet zeros
    // in Y), and so are columns beyond d_in
    auto fetch_edge = [&](int u) {
      const SplitUnit& L = U.unit[at.x.unit];
      const int k0 = at.x.k_begin + at.step * kStep, d_in = L.d_in;
      const int r = min((XQ ? at.x.row0 : k0) + row + kRowStep * u, L.m - 1);
      const int c = (XQ ? k0 : at.x.row0) + 4 * c4, left = d_in - c;
      const T* p = reinterpret_cast<const T*>(L.X) + r * L.ldx;
      v[u] = vec ? fetch_x(p + min(c, d_in - 4)) : fetch_x(p + (left > 0 ? c : 0), left);
    };
    auto inside = [&]() { return whole && at.x.k_begin + at.step * kStep + kStep <= at.x.k_end; };
    if (at.it >= 0) {
      open();
#pragma unroll
      for (int u = 0; u < 8; ++u) fetch_edge(u);
    }
    uint32_t s = (uint32_t)(group % kStages), par = 1;     // first round of a stage: free
    while (at.it >= 0) {
      if (!mbar_wait_warp(&sh.empty[s], par, U.wait_ns)) { sh.failed = 1; break; }
      const uint32_t dst = tiles + s * (uint32_t)kStageBytes;
      const bool moved = at.advance(U, kLoadGroups);
      const bool more = at.it >= 0;
      if (!moved) x += turn; else if (more) open();
      const uint32_t put = dst + place;
      if (more && inside()) {
        const T* p = x;
#pragma unroll
        for (int u = 0; u < 8; ++u) {
          put_x<PLANES>(v[u], put + (uint32_t)(u * kRowStep * 128));
          v[u] = fetch_x(p);
          p += row_step;
        }
      } else {
#pragma unroll
        for (int u = 0; u < 8; ++u) {
          put_x<PLANES>(v[u], put + (uint32_t)(u * kRowStep * 128));
          if (more) fetch_edge(u);
        }
      }
      __syncwarp();
      if (lane == 0) mbar_arrive(&sh.full[s]);
      s += kLoadGroups;
      if (s >= (uint32_t)kStages) { s -= kStages; par ^= 1u; }
    }
  } else if (warp == kMmaWarp) {
    // ---------------------------------------------------------------- products
    const uint32_t go = elect_one();
    constexpr int n1 = (2 * NP + 15) & ~15, n2 = (NP + 15) & ~15;
    const uint32_t id0 = instr_desc(128, NB, XQ ? 0 : 1, 0), id1 = instr_desc(128, n1, XQ ? 0 : 1, 0), id2 = instr_desc(128, n2, XQ ? 0 : 1, 0);
    uint32_t s = 0, par = 0, b = 0, bpar = 1;
    bool ok = true;
    for (int i = 0, it; ok && (it = nth_item(U, i)) >= 0; ++i) {
      const int n = __shfl_sync(0xffffffffu, steps_of(item_of<XQ>(U, it)), 0);      // which the compiler knows to be uniform
      for (int k = 0; k < n; ++k) {
        if (!mbar_wait_warp(&sh.full[s], par, U.wait_ns) || !mbar_wait_warp(&sh.acc_empty[b], bpar, U.wait_ns)) { sh.failed = 1; ok = false; break; }
        fence_proxy_async();
        tc_fence_after();
        const uint32_t a = tiles + s * (uint32_t)kStageBytes, d = tmem + b * (uint32_t)NB;
        const uint64_t bd = smem_desc(a + (uint32_t)(PLANES * kPlaneBytes), 0, 1024);
#pragma unroll
        for (int p = PLANES - 1; p >= 0; --p) {
          const uint64_t ad = smem_desc(a + (uint32_t)(p * kPlaneBytes), XQ ? 0 : kPlaneBytes / 2, 1024);
#pragma unroll
          for (int kk = 0; kk < kStep / 16; ++kk) {       // an accumulator's first instruction writes all of its columns
            const bool first = p == PLANES - 1 && kk == 0;
            mma_bf16_if(go, d, ad + (uint64_t)((XQ ? 2 : 128) * kk), bd + (uint64_t)(2 * kk), first || p == 0 ? id0 : p == 1 ? id1 : id2,
                        first ? 0u : 1u);
          }
        }
        mma_commit_if(go, &sh.empty[s]);
        mma_commit_if(go, &sh.acc_full[b]);
        if (++s == (uint32_t)kStages) { s = 0; par ^= 1u; }
        if (++b == (uint32_t)kAcc) { b = 0; bpar ^= 1u; }
      }
    }
  } else if (warp >= kOpWarp0) {
    // ---------------------------------------------------------------- operand rows 4 e to 4 e + 3, two of the contracted dimension per lane
    const int e = warp - kOpWarp0;
    uint32_t op_place[4];
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const int row = 4 * e + j;
      op_place[j] = tiles + (uint32_t)(PLANES * kPlaneBytes + row * 128 + (((lane >> 2) ^ (row & 7)) << 4) + (lane & 3) * 4);
    }
    Walk<XQ, N> at;
    const float* op[4];                    // source of a row; where the four ranks are one layer's (quad) the first one serves
    int op_step[4];                        // from one of the contracted dimension to the next, 0: no such rank
    bool quad = false;
    long long op_row = 0;                  // between the ranks of a quad
    float o[4][2];
    auto open = [&]() {
      const SplitUnit& s = U.unit[at.x.unit];
      const long long k0 = at.x.k_begin + 2 * lane;
      quad = s.quads != 0 && 4 * e < s.np;
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        op_step[j] = 0;
        op[j] = nullptr;
        if (4 * e + j >= s.np) continue;
        int k;
        const SplitLayer& L = s.layer[layer_of(s, 4 * e + j, &k)];
        op_step[j] = XQ ? 1 : L.r;
        op[j] = L.src + (XQ ? k * L.ldv : (long long)k) + k0 * op_step[j];
        if (j == 0) op_row = L.ldv;
      }
    };
    auto fetch = [&]() {
      const int left = at.x.k_end - (at.x.k_begin + at.step * kStep + 2 * lane);
      if (quad && left > 1) {
        if constexpr (XQ) {
#pragma unroll
          for (int j = 0; j < 4; ++j) {
            const float2 z = *reinterpret_cast<const float2*>(op[0] + j * op_row);
            o[j][0] = z.x; o[j][1] = z.y;
          }
        } else {
          const float4 a = *reinterpret_cast<const float4*>(op[0]), b = *reinterpret_cast<const float4*>(op[0] + op_step[0]);
          o[0][0] = a.x; o[1][0] = a.y; o[2][0] = a.z; o[3][0] = a.w;
          o[0][1] = b.x; o[1][1] = b.y; o[2][1] = b.z; o[3][1] = b.w;
        }
      } else {
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          const bool any = op_step[j] != 0;
          o[j][0] = any && left > 0 ? op[j][0] : 0.f;
          o[j][1] = any && left > 1 ? op[j][op_step[j]] : 0.f;
        }
      }
    };
    uint32_t s = 0, par = 1;
    at.start(U);
    chain_wait();
    if (e == 0 && short_launch()) chain_next();
    if (at.it >= 0) { open(); fetch(); }
    while (at.it >= 0) {
      if (!mbar_wait_warp(&sh.empty[s], par, U.wait_ns)) { sh.failed = 1; break; }
      const uint32_t dst = s * (uint32_t)kStageBytes;
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        uint64_t z = pack_f32x2(o[j][0], o[j][1]);
#pragma unroll
        for (int p = 0; p < 3; ++p) {
          const uint32_t a = bf16_pair(z);
          asm volatile("st.shared.b32 [%0], %1;" ::"r"(op_place[j] + dst + (uint32_t)(p * NP * 128)), "r"(a) : "memory");
          if (p < 2) z = less_pair(z, a);
        }
      }
      __syncwarp();
      if (lane == 0) mbar_arrive(&sh.full[s]);
      if (++s == (uint32_t)kStages) { s = 0; par ^= 1u; }
      const bool moved = at.advance(U, 1);
      if (at.it < 0) break;
      if (moved) {
        open();
      } else {
#pragma unroll
        for (int j = 0; j < 4; ++j) op[j] += kStep * op_step[j];
      }
      fetch();
    }
  } else {
    // ---------------------------------------------------------------- accumulators: this warp's 32 rows, half of the ranks
    constexpr int H = NP / 2;
    const int q = warp & 3, half = (warp - kLoadWarps) >> 2;
    const uint32_t lanes = tmem + ((uint32_t)(q * 32) << 16) + (uint32_t)(half * H);
    uint32_t b = 0, par = 0;
    bool ok = true;
    chain_wait();                          // what it writes, the kernel before may still read
    for (int i = 0, it; ok && (it = nth_item(U, i)) >= 0; ++i) {
      const Item x = item_of<XQ>(U, it);
      const int n = steps_of(x);
      uint64_t sum[3][H / 2];
#pragma unroll
      for (int p = 0; p < 3; ++p)
#pragma unroll
        for (int k = 0; k < H / 2; ++k) sum[p][k] = 0;
      for (int k = 0; k < n; ++k) {
        if (!mbar_wait_warp(&sh.acc_full[b], par, U.wait_ns)) { ok = false; break; }
        tc_fence_after();
        // two parts at a time, for want of registers
        uint32_t z[2][H];
#pragma unroll
        for (int p = 0; p < 2; ++p) tmem_ld_cols<H>(lanes + b * (uint32_t)NB + (uint32_t)(p * NP), z[p]);
        tmem_ld_wait();
#pragma unroll
        for (int p = 0; p < 2; ++p)
#pragma unroll
          for (int c = 0; c < H; c += 2)
            sum[p][c / 2] = add_f32x2(sum[p][c / 2], pack_f32x2(__uint_as_float(z[p][c]), __uint_as_float(z[p][c + 1])));
        tmem_ld_cols<H>(lanes + b * (uint32_t)NB + (uint32_t)(2 * NP), z[0]);
        tmem_ld_wait();
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(&sh.acc_empty[b]);
        if (++b == (uint32_t)kAcc) { b = 0; par ^= 1u; }
#pragma unroll
        for (int c = 0; c < H; c += 2)
          sum[2][c / 2] = add_f32x2(sum[2][c / 2], pack_f32x2(__uint_as_float(z[0][c]), __uint_as_float(z[0][c + 1])));
      }
      if (!ok) break;
      float y[H];
#pragma unroll
      for (int c = 0; c < H; c += 2) unpack_f32x2(add_f32x2(add_f32x2(sum[2][c / 2], sum[1][c / 2]), sum[0][c / 2]), y[c], y[c + 1]);
      const SplitUnit& s = U.unit[x.unit];
      if (XQ && U.split > 1) {             // rank 0 adds the others' sums to its own, in rank order
        const uint32_t rank = cluster_ctarank(), mine = (uint32_t)((warp - kLoadWarps) * 32 + lane) * 16u, piece = kEpiWarps * 32 * 16;
        const uint32_t peers = tiles + (uint32_t)(kStages * kStageBytes);
        if (rank != 0) {
          if (i > 0 && !mbar_wait_cluster_warp(&sh.sums_out, (uint32_t)(i - 1) & 1u, U.wait_ns)) { ok = false; break; }
          const uint32_t dst = mapa_shared(peers + (rank - 1u) * C::peer_bytes + mine, 0), bar = mapa_shared(smem_u32(&sh.sums_in), 0);
#pragma unroll
          for (int c = 0; c < H; c += 4) st_async_f4(dst + (uint32_t)(c / 4) * piece, make_float4(y[c], y[c + 1], y[c + 2], y[c + 3]), bar);
          continue;
        }
        if (warp == kLoadWarps && lane == 0) mbar_expect_tx(&sh.sums_in, (uint32_t)(U.split - 1) * C::peer_bytes + U.missing);
        if (!mbar_wait_cluster_warp(&sh.sums_in, (uint32_t)i & 1u, U.wait_ns)) { ok = false; break; }
        for (int p = 0; p < U.split - 1; ++p)
#pragma unroll
          for (int c = 0; c < H; c += 4) {
            float4 z;
            asm volatile("ld.shared.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(z.x), "=f"(z.y), "=f"(z.z), "=f"(z.w)
                         : "r"(peers + (uint32_t)(p * C::peer_bytes) + (uint32_t)(c / 4) * piece + mine) : "memory");
            y[c] += z.x; y[c + 1] += z.y; y[c + 2] += z.z; y[c + 3] += z.w;
          }
        __syncwarp();
        if (lane > 0 && lane < U.split) mbar_arrive_remote(mapa_shared(smem_u32(&sh.sums_out), (uint32_t)lane));
      }
      const int r = x.row0 + 32 * q + lane;
      if (r < s.rows) {
        int kl, l = layer_of(s, half * H, &kl);
#pragma unroll
        for (int c = 0; c < H; ++c) {
          if (half * H + c >= s.np) break;
          const SplitLayer& L = s.layer[l];
          if (XQ) L.dst[(long long)r * L.r + kl] = y[c];
          else L.dst[x.slab * L.slab + (long long)kl * s.d_in + r] = y[c];
          if (++kl == L.r) { kl = 0; ++l; }
        }
      }
    }
    if (!ok) sh.failed = 1;
  }
  tc_fence_before();
  __syncthreads();
  if (XQ && U.split > 1) cluster_sync_all();               // nobody leaves while a peer sends to it
  if (sh.failed) let_land();
  if (sh.failed && threadIdx.x == 0) report_timeout(status, XQ ? 6 : 7);
  if (warp == kMmaWarp) { tc_fence_after(); tmem_dealloc(tmem, C::tmem_cols); }
}

template <int N> using Kernel = void (*)(const SplitUnits<N>, DevStatus*);
template <int NP, int N> Kernel<N> kernel_np(int planes, bool xq) {
  if (planes == 3) return xq ? split_product_kernel<NP, 3, true, N> : split_product_kernel<NP, 3, false, N>;
  return xq ? split_product_kernel<NP, 1, true, N> : split_product_kernel<NP, 1, false, N>;
}
template <int N> Kernel<N> kernel_of(int np, int planes, bool xq) {
  return np <= 8 ? kernel_np<8, N>(planes, xq) : np <= 16 ? kernel_np<16, N>(planes, xq) : kernel_np<24, N>(planes, xq);
}
// Shared memory is asked for only where it is used: the operands' sources come through L1, which has the rest (the peers' places in a launch
// without clusters: T = X Q of two fp32 blocks of 0.6B shape, r = 8, 65 -> 72 us)
template <int NP, int PLANES> size_t smem_at(int split) {
  return split > 0 ? Cfg<NP, PLANES, true>::smem + (size_t)(split - 1) * Cfg<NP, PLANES, true>::peer_bytes : Cfg<NP, PLANES, false>::smem;
}
template <int NP> size_t smem_np(int planes, int split) { return planes == 3 ? smem_at<NP, 3>(split) : smem_at<NP, 1>(split); }
int threads_of(int np) { return np <= 8 ? Cfg<8, 1, true>::threads : np <= 16 ? Cfg<16, 1, true>::threads : Cfg<24, 1, true>::threads; }
// split: CTAs that share an item of T = X Q, 0 for Y = X^T T
size_t smem_of(int np, int planes, int split) { return np <= 8 ? smem_np<8>(planes, split) : np <= 16 ? smem_np<16>(planes, split) : smem_np<24>(planes, split); }

// CTAs that share an item of T = X Q: where the items do not fill the device, clusters of two or four take the columns between them.  Returns
// the steps of the CTA that has most; the exchange counts as two, as six where the cluster has items before it, which then wait for accumulators
// (an extraction with K = 3, alone / shared: 4000 x 1024 fp32, r = 8, 93 / 79 us in fours; 5000 x 1001 bf16, r = 8, 158 / 124 in pairs; T = X Q of two
// fp32 blocks of 0.6B shape, at most 64 steps alone and 50 in pairs: 72 / 78 us).  Units from the widest on.
struct XqUnit { int m, d_in; };
int clusters_of(int split, int sm_count) { return split == 4 ? sm_count / 4 * 7 / 8 : sm_count / split; }     // fours lie inside GPCs of no multiple of four SMs
int most_steps(const std::vector<XqUnit>& units, int sm_count, int* split) {
  int least = -1, items = 0;
  for (const XqUnit& u : units) items += (u.m + 127) / 128;
  std::vector<int> load;
  for (int c = 1; c <= kMaxSplit; c *= 2) {
    const int G = clusters_of(c, sm_count);
    if (G < 1 || (c > 1 && items > 8 * G)) break;
    load.assign((size_t)G, 0);
    int it = 0, most = 0;
    for (const XqUnit& u : units)
      for (int e = (u.m + 127) / 128; e > 0; --e, ++it) {
        const int round = it / G, b = it % G;
        int& l = load[(size_t)((round & 1) ? G - 1 - b : b)];
        l += ((u.d_in + kStep - 1) / kStep + c - 1) / c + (c == 1 ? 0 : l == 0 ? 2 : 6);
        most = std::max(most, l);
      }
    if (least < 0 || most < least) { least = most; *split = c; }
  }
  return least;
}

// Units of the wave: the layers that read one X, at most four at a time, their ranks cut into panels of about equal size
std::vector<SplitUnit> units_of(const ExtractWave& w, const DevLayer* dev, bool share, bool xq) {
  std::vector<SplitUnit> units;
  for (int l = w.l0; l < w.l1;) {
    const DevLayer& a = dev[l];
    int n = 1, ranks = a.r;
    while (share && n < kSplitMaxLayers && l + n < w.l1 && split_same_x(a, dev[l + n])) ranks += dev[l + n++].r;
    SplitUnit u{};
    u.X = a.X; u.ldx = a.ldx; u.m = a.m; u.d_in = a.d_in; u.slabs = a.slabs; u.slab_rows = a.slab_rows;
    u.rows = xq ? a.m : a.d_in;
    u.vec = a.d_in % 4 == 0 && a.ldx % 4 == 0 && (reinterpret_cast<uintptr_t>(a.X) & (a.x_dtype == AGZO_F32 ? 15u : 7u)) == 0;
    // panels of whole fours
    const int panels = (ranks + kSplitMaxRanks - 1) / kSplitMaxRanks, per = ((ranks + panels - 1) / panels + 3) & ~3;
    for (int p = 0; p < ranks; p += per) {
      int first = l, k0 = p;
      while (k0 >= dev[first].r) k0 -= dev[first++].r;
      u.k0 = (short)k0; u.np = (short)std::min(per, ranks - p);
      for (int k = 0; k < kSplitMaxLayers; ++k) {
        u.layer[k] = SplitLayer{};
        if (first + k >= l + n) continue;
        const DevLayer& D = dev[first + k];
        u.layer[k] = SplitLayer{xq ? D.V : D.T, xq ? D.T : D.Ypart, D.ldv, D.ypart_stride, D.r, 0};
      }
      u.quads = 1;
      for (int k = l; k < l + n; ++k)
        if (dev[k].r % 4 != 0 || (xq && (dev[k].ldv % 2 != 0 || (reinterpret_cast<uintptr_t>(dev[k].V) & 7u) != 0))) u.quads = 0;
      units.push_back(u);
    }
    l += n;
  }
  return units;
}

// The kernel's shared-memory limit, set when it is first used in a CUDA context (it ends with the context): few programs use more than two
cudaError_t allow_smem(const void* kernel, size_t smem) {
  struct Known { unsigned long long context; std::vector<const void*> kernels; };
  static std::mutex mu;
  static Known known[kMaxDevices];
  int device = -1;
  cudaError_t e = cudaGetDevice(&device);
  if (e != cudaSuccess) return e;
  const unsigned long long id = current_context_id(device);
  std::lock_guard<std::mutex> lock(mu);
  Known* k = device < kMaxDevices && id != 0 ? known + device : nullptr;
  if (k && k->context != id) { k->context = id; k->kernels.clear(); }
  if (k && std::find(k->kernels.begin(), k->kernels.end(), kernel) != k->kernels.end()) return cudaSuccess;
  e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e == cudaSuccess && k) k->kernels.push_back(kernel);
  return e;
}

template <int N>
cudaError_t launch_units(const std::vector<SplitUnit>& units, size_t first, int np, int planes, bool xq, int sm_count, bool missing, DevStatus* status, cudaStream_t s) {
  SplitUnits<N> U;
  U.n_units = (int)std::min((size_t)N, units.size() - first);
  long long items = 0;
  for (int k = 0; k < U.n_units; ++k) {
    U.unit[k] = units[first + k];
    SplitUnit& u = U.unit[k];
    u.item0 = (int)items;
    items += xq ? (u.m + 127) / 128 : (long long)((u.d_in + 127) / 128) * u.slabs;
  }
  if (items > 0x3fffffff) return cudaErrorInvalidValue;
  U.n_items = (int)items;
  U.split = 1;
  U.wait_ns = missing ? kMissingWaitNs : (unsigned)kWaitCapNs;
  U.missing = missing ? 1 : 0;
  if (xq) {
    std::vector<XqUnit> shapes;
    for (int k = 0; k < U.n_units; ++k) shapes.push_back(XqUnit{U.unit[k].m, U.unit[k].d_in});
    most_steps(shapes, sm_count, &U.split);
  }
  const long long groups = std::min(items, (long long)clusters_of(U.split, sm_count));
  const Kernel<N> kernel = kernel_of<N>(np, planes, xq);
  const size_t smem = smem_of(np, planes, xq ? U.split : 0);
  const cudaError_t e = allow_smem((const void*)kernel, smem_of(np, planes, xq ? kMaxSplit : 0));
  if (e != cudaSuccess) return e;
  return launch_chained(kernel, dim3((unsigned)(groups * U.split)), threads_of(np), smem, U.split > 1 ? U.split : 0, s, U, status);
}

cudaError_t launch(const ExtractWave& w, const DevLayer* dev, bool share, bool xq, DevStatus* status, cudaStream_t s) {
  std::vector<SplitUnit> units = units_of(w, dev, share, xq);
  int np = 0;
  for (const SplitUnit& u : units) np = std::max(np, (int)u.np);
  const int planes = dev[w.l0].x_dtype == AGZO_F32 ? 3 : 1;
  std::stable_sort(units.begin(), units.end(), [](const SplitUnit& a, const SplitUnit& b) { return a.d_in > b.d_in; });
  if (!xq) std::reverse(units.begin(), units.end());
  if (units.size() <= kSplitFewUnits) return launch_units<kSplitFewUnits>(units, 0, np, planes, xq, w.sm_count, w.missing != 0, status, s);
  for (size_t at = 0; at < units.size(); at += kSplitMaxUnits) {
    const cudaError_t e = launch_units<kSplitMaxUnits>(units, at, np, planes, xq, w.sm_count, w.missing != 0, status, s);
    if (e != cudaSuccess) return e;
  }
  return cudaSuccess;
}

}  // namespace

bool split_same_x(const DevLayer& a, const DevLayer& b) {
  return a.X == b.X && a.ldx == b.ldx && a.m == b.m && a.d_in == b.d_in && a.x_dtype == b.x_dtype && a.slabs == b.slabs && a.slab_rows == b.slab_rows;
}

bool split_pays(const agzo_layer* L, const std::vector<int>& which, bool share, int sm_count) {
  std::vector<XqUnit> units;
  long long blocks = 0;
  int max_m = 0, max_d = 0, max_r = 0;
  double wide = 0.0;                     // operand rows beyond those of eight ranks, 1 for 24
  double there = 0.0;                    // microseconds of two products X^T T and one X Q
  double x_bytes = 0.0;
  for (int k : which) max_r = std::max(max_r, L[k].r);
  const bool r4 = max_r > 4, r8 = max_r > 8;
  const int passes = (max_r + 15) / 16;
  bool any_scalar = false;
  for (size_t i = 0; i < which.size();) {
    const agzo_layer& a = L[which[i]];
    if (a.x_dtype != L[which[0]].x_dtype) return false;
    int n = 1, ranks = a.r;
    for (; share && n < kSplitMaxLayers && i + n < which.size() && which[i + n] == which[i] + n; ++n) {
      const agzo_layer& b = L[which[i + n]];
      if (a.X != b.X || a.ldx != b.ldx || a.m != b.m || a.d_in != b.d_in || a.x_dtype != b.x_dtype) break;
      ranks += b.r;
    }
    i += n;
    const int panels = (ranks + kSplitMaxRanks - 1) / kSplitMaxRanks;
    for (int p = 0; p < panels; ++p) units.push_back(XqUnit{a.m, a.d_in});
    wide = std::max(wide, (((ranks + panels - 1) / panels + 7) / 8 - 1) / 2.0);
    blocks += (long long)panels * ((a.d_in + 127) / 128);
    max_m = std::max(max_m, a.m); max_d = std::max(max_d, a.d_in);
    const bool f32 = a.x_dtype == AGZO_F32, scalar = a.d_in % 4 != 0 || a.ldx % 4 != 0 || (reinterpret_cast<uintptr_t>(a.X) & (f32 ? 15u : 7u)) != 0;
    any_scalar = any_scalar || scalar;
    x_bytes += (f32 ? 4.0 : 2.0) * a.m * (double)a.d_in;
    const double md = 1e-6 * n * a.m * (double)a.d_in;
    there += md * (scalar ? 2.0 * (1.96 + 0.48 * r4 + 5.30 * (passes - 1)) + 1.70 + 2.43 * r4 + 2.48 * r8 + 4.92 * (passes - 1)
                   : f32 ? 2.0 * (0.21 + 0.31 * r4 + 0.64 * r8 + 1.19 * (passes - 1)) + 1.29 + 0.47 * r8 + 1.82 * (passes - 1)
                         : 2.0 * 0.12 * r4 + 0.82 + 0.55 * r4);
  }
  if (units.empty()) return false;
  there += 0.75 + 1e-3 * max_d * (6.75 * r8 * passes + 10.9 * any_scalar) + 2.0 * 0.79e-3 * max_m;
  std::stable_sort(units.begin(), units.end(), [](const XqUnit& a, const XqUnit& b) { return a.d_in > b.d_in; });
  int split = 1;
  const int rows = split_slab_rows(max_m, blocks, sm_count);
  const long long slabs = (max_m + rows - 1) / rows, rounds = (slabs * blocks + sm_count - 1) / sm_count;
  const double here = 2.0 * (1.17 + 0.13 * wide) * (double)(rounds * (rows / kStep)) + 0.85 * most_steps(units, sm_count, &split);
  // Inputs that stay in L2 between the products serve fp32 rows of whole 16-byte pieces at ranks up to 8, where the CUDA-core products wait for memory,
  // sooner than `there` has it: a layer of 7858 x 828, r = 3, 21.7 here and 24.3 there by estimate, takes 101 and 81 us.  From 100 MB on they don't.
  const bool in_l2 = x_bytes < 100e6 && !any_scalar && L[which[0]].x_dtype == AGZO_F32;
  const double line = !in_l2 || max_r > 8 ? 1.0 : max_r <= 4 ? 0.8 : 0.92;
  return here < line * there;
}

bool split_takes(const ExtractWave& w, const DevLayer* dev, int K) {
  for (int l = w.l0; l < w.l1; ++l)
    if (dev[l].x_dtype != dev[w.l0].x_dtype || dev[l].Qb) return false;
  return dev[w.l0].x_dtype == AGZO_BF16 || K > 0;
}

cudaError_t launch_split_xt_t(const ExtractWave& w, const DevLayer* dev, bool share, DevStatus* status, cudaStream_t s) {
  return launch(w, dev, share, false, status, s);
}
cudaError_t launch_split_x_q(const ExtractWave& w, const DevLayer* dev, bool share, DevStatus* status, cudaStream_t s) {
  return launch(w, dev, share, true, status, s);
}

}  // namespace agzo

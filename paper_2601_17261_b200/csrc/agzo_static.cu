// Allocation-free variant of Algorithm 1 for one layer: the scratch that the extraction
// kernels need lives in a fixed array inside the loaded library image instead of a workspace
// the caller would have to allocate.
//
// Who needs this: code that may not call cudaMalloc at the point where it wants a subspace --
// a forward hook running while another framework owns the allocator (or while a memory pool is
// frozen), a callback invoked from a context where allocation would synchronise the device, a
// process whose memory budget is fixed up front.  Such a caller still owns X and V; it simply
// has nowhere to get a workspace from.
#include <mutex>

#include "agzo_common.cuh"
#include "agzo_ptx.cuh"
#include "agzo_resident.cuh"
#include "agzo_split.cuh"

namespace {

constexpr size_t kStaticScratchBytes = 4u << 20;   // 4 MiB, held by every GPU that loads the library

// The name below is a host-side handle for the symbol, not a device address: kernels must be
// given the address that cudaGetSymbolAddress returns for the current device.
static __device__ __align__(256) unsigned char g_static_scratch[kStaticScratchBytes];
// What the resident kernel needs where the problem fits the limit above (a partial sum of Y per row of CTAs), and its counter, which
// a launch leaves as good as it found it.
constexpr size_t kResidentScratchBytes = 5u << 20;
static __device__ __align__(256) unsigned char g_resident_scratch[kResidentScratchBytes];
static __device__ unsigned long long g_resident_counter;

// Looked up once per CUDA context: the address and the kernels' limits end with it (cudaDeviceReset).
struct Scratch {
  unsigned long long context;
  void* addr;
  bool qr_wide;
  int sm_count;
  agzo::ResidentCaps resident;
  void* resident_addr;
  void* resident_counter;
};
std::mutex g_mu;
Scratch g_scratch[agzo::kMaxDevices] = {};

cudaError_t scratch_of_current_device(Scratch* out) {
  int dev = -1;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  if (dev < 0 || dev >= agzo::kMaxDevices) return cudaErrorInvalidDevice;
  const unsigned long long id = agzo::current_context_id(dev);
  std::lock_guard<std::mutex> lock(g_mu);
  Scratch& known = g_scratch[dev];
  if (!known.addr || id == 0 || known.context != id) {
    Scratch fresh{};
    fresh.context = id;
    e = cudaGetSymbolAddress(&fresh.addr, g_static_scratch);   // with that device current
    if (e == cudaSuccess) e = cudaGetSymbolAddress(&fresh.resident_addr, g_resident_scratch);
    if (e == cudaSuccess) e = cudaGetSymbolAddress(&fresh.resident_counter, g_resident_counter);
    if (e == cudaSuccess) e = agzo::panel_qr_init(&fresh.qr_wide);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&fresh.sm_count, cudaDevAttrMultiProcessorCount, dev);
    if (e == cudaSuccess) e = agzo::resident_init(fresh.sm_count, &fresh.resident);
    if (e != cudaSuccess) return e;
    known = fresh;
  }
  *out = known;
  return cudaSuccess;
}

inline size_t up256(size_t x) { return (x + 255) / 256 * 256; }

// The array is shared by all calls and keeps the previous call's contents: the layer record is
// rewritten and the status word cleared here; every other slice is fully overwritten by the
// kernels before it is read.
__global__ void static_begin_kernel(agzo::DevLayer rec, agzo::DevLayer* dst, agzo::DevStatus* st) {
  agzo::chain_wait();      // an earlier call may still read the record; the kernels after it read it before they wait,
                           // so they are not allowed to start early (no chain_next)
  *dst = rec;
  st->rank_deficient = 0;
  st->timeout = 0;
  st->where = 0;
  st->pad = 0;
}

// 2: a wait ran out, and the last panel QR has left V = 0
__global__ void static_end_kernel(const agzo::DevStatus* st, int32_t* flag) {
  agzo::chain_wait();
  *flag = st->timeout ? 2 : st->rank_deficient;
}

}  // namespace

namespace {

// route: 0 = the faster kernels, 1 = the chain, 2 = the resident kernel, whose waits for other blocks end after wait_ns
agzo_status extract_static(const void* X, int64_t ldx, int32_t x_dtype, int32_t m, int32_t d_in, int32_t r, int32_t K, uint64_t seed,
                           uint32_t layer_id, float* V, int64_t ldv, int32_t* d_rank_deficient, int route, unsigned long long wait_ns,
                           void* stream) {
  using namespace agzo;
  if (!X || !V || m < 1 || d_in < 1 || r < 1 || r > AGZO_MAX_RANK || r > d_in || r > m ||
      ldx < d_in || ldv < d_in || K < 0 || K > 16)
    return AGZO_ERR_INVALID_ARG;
  if (x_dtype != AGZO_BF16 && x_dtype != AGZO_F32) return AGZO_ERR_UNSUPPORTED;
  const size_t es = x_dtype == AGZO_BF16 ? 2 : 4;
  if ((reinterpret_cast<uintptr_t>(X) & (es - 1)) || (reinterpret_cast<uintptr_t>(V) & 3u))
    return AGZO_ERR_INVALID_ARG;

  // token slabs of the X^T T product.  What the array admits is decided with slabs of at least 256 tokens; inside that
  // limit the slabs are as short as the room left over allows, down to what fills the GPU.
  int slab_rows = (m + 31) / 32;
  slab_rows = (slab_rows + 31) / 32 * 32;
  if (slab_rows < 256) slab_rows = 256;
  int slabs = (m + slab_rows - 1) / slab_rows;
  const size_t gch = ((size_t)d_in + 127) / 128;
  const size_t R = (size_t)r, D = (size_t)d_in, M = (size_t)m;
  const size_t need = 512 + up256(M * R * 4) + up256((size_t)slabs * R * D * 4) + up256(R * D * 4) +
                      up256(gch * R * R * 8) + up256(R * R * 8);
  if (need > kStaticScratchBytes) return AGZO_ERR_WORKSPACE;   // problem too large for the fixed array
  Scratch scratch;
  if (scratch_of_current_device(&scratch) != cudaSuccess) return AGZO_ERR_CUDA;
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  agzo_layer a{};
  a.X = X; a.ldx = ldx; a.x_dtype = x_dtype; a.m = m; a.d_in = d_in; a.r = r; a.layer_id = layer_id;
  a.V = V; a.ldv = ldv;
  if (route != 1) {
    ResidentLaunch plan;      // K = 0: a block that comes too late to the only meeting would not see that others have given up
    if (resident_plan(scratch.resident, &a, 1, false, false, &plan) && plan.scratch <= kResidentScratchBytes &&
        !(plan.grid_wide && K == 0) && (route == 2 || resident_pays(plan, K, true))) {
      resident_bind(&plan, static_cast<char*>(scratch.resident_addr));
      plan.p.K = K;
      plan.p.wait_ns = wait_ns;
      plan.p.late_ns = wait_ns < ptx::kWaitCapNs ? wait_ns + 100000 : 0;
      plan.p.seed = seed;
      plan.p.flag = d_rank_deficient;
      plan.p.counters = static_cast<unsigned long long*>(scratch.resident_counter);
      const cudaError_t e = launch_resident(plan, s);
      if (e == cudaSuccess) return AGZO_OK;
      if (!resident_refused(e)) return AGZO_ERR_CUDA;
    }
    if (route == 2) return AGZO_ERR_UNSUPPORTED;
  }
  const bool split = (K > 0 || x_dtype == AGZO_BF16) && split_pays(&a, std::vector<int>{0}, true, scratch.sm_count);
  const long long panels = (r + kSplitMaxRanks - 1) / kSplitMaxRanks;
  for (int rows = split ? split_slab_rows(m, (long long)gch * panels, scratch.sm_count) : cc_slab_rows(m, (long long)gch, scratch.sm_count);; rows += 32) {      // ends at 256 tokens per slab at the latest
    const size_t n = ((size_t)m + rows - 1) / rows;
    if (need - up256((size_t)slabs * R * D * 4) + up256(n * R * D * 4) <= kStaticScratchBytes) { slab_rows = rows; slabs = (int)n; break; }
  }

  unsigned char* p = static_cast<unsigned char*>(scratch.addr);
  DevLayer* d_rec = reinterpret_cast<DevLayer*>(p);
  DevStatus* d_status = reinterpret_cast<DevStatus*>(p + 384);
  p += 512;
  DevLayer rec{};
  rec.X = X; rec.V = V; rec.ldx = ldx; rec.ldv = ldv;
  rec.x_dtype = x_dtype; rec.d_in = d_in; rec.m = m; rec.r = r; rec.layer_id = layer_id;
  rec.slabs = rec.cc_slabs = slabs; rec.slab_rows = slab_rows; rec.gchunks = (int)gch;
  rec.T = reinterpret_cast<float*>(p);      p += up256(M * R * 4);
  rec.ypart_stride = (long long)r * d_in;
  rec.Ypart = reinterpret_cast<float*>(p);  p += up256((size_t)slabs * R * D * 4);
  rec.Y = reinterpret_cast<float*>(p);      p += up256(R * D * 4);
  rec.Gpart = reinterpret_cast<double*>(p);     // used above rank 32 only; never more than the two terms in r^2 of the limit there
  static_assert(sizeof(DevLayer) <= 384, "layer record must fit its slot");

  if (launch_chained(static_begin_kernel, dim3(1), 1, 0, 0, s, rec, d_rec, d_status) != cudaSuccess) return AGZO_ERR_CUDA;

  ExtractWave w{};
  w.d_layers = d_rec;
  w.l0 = 0; w.l1 = 1;
  w.sm_count = scratch.sm_count;
  w.qr_wide = scratch.qr_wide ? 1 : 0;
  w.max_m = m; w.max_din = d_in; w.max_r = r; w.max_slabs = slabs; w.max_gchunks = (int)gch;
  if (launch_fill_omega(w, seed, d_status, s) != cudaSuccess) return AGZO_ERR_CUDA;     // Omega
  const auto xt_t = [&] { return split ? launch_split_xt_t(w, &rec, true, d_status, s) : launch_xt_t(w, s); };
  const auto x_q = [&] { return split ? launch_split_x_q(w, &rec, true, d_status, s) : launch_x_q(w, s); };
  if (xt_t() != cudaSuccess) return AGZO_ERR_CUDA;                            // Y <- H Omega
  for (int k = 0; k < K; ++k) {
    if (launch_panel_qr(w, false, d_status, s) != cudaSuccess) return AGZO_ERR_CUDA;  // Q <- qr(Y)
    if (x_q() != cudaSuccess) return AGZO_ERR_CUDA;
    if (xt_t() != cudaSuccess) return AGZO_ERR_CUDA;                          // Y <- H (H^T Q)
  }
  if (launch_panel_qr(w, true, d_status, s) != cudaSuccess) return AGZO_ERR_CUDA;    // A <- qr(Y)
  if (d_rank_deficient) {
    if (launch_chained(static_end_kernel, dim3(1), 1, 0, 0, s, d_status, d_rank_deficient) != cudaSuccess) return AGZO_ERR_CUDA;
  }
  return AGZO_OK;
}

}  // namespace

extern "C" agzo_status agzo_extract_subspace_static(const void* X, int64_t ldx, int32_t x_dtype,
                                                    int32_t m, int32_t d_in, int32_t r, int32_t K,
                                                    uint64_t seed, uint32_t layer_id, float* V,
                                                    int64_t ldv, int32_t* d_rank_deficient,
                                                    void* stream) {
  return extract_static(X, ldx, x_dtype, m, d_in, r, K, seed, layer_id, V, ldv, d_rank_deficient, 0, agzo::ptx::kWaitCapNs, stream);
}

extern "C" agzo_status agzo_debug_extract_static(const void* X, int64_t ldx, int32_t x_dtype, int32_t m, int32_t d_in, int32_t r,
                                                 int32_t K, uint64_t seed, uint32_t layer_id, float* V, int64_t ldv,
                                                 int32_t* d_rank_deficient, int32_t route, int64_t wait_ns, void* stream) {
  if (route < 0 || route > 2 || wait_ns < 0 || (unsigned long long)wait_ns > agzo::ptx::kWaitCapNs) return AGZO_ERR_INVALID_ARG;
  return extract_static(X, ldx, x_dtype, m, d_in, r, K, seed, layer_id, V, ldv, d_rank_deficient, route, (unsigned long long)wait_ns, stream);
}

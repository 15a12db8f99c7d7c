// C ABI of the AGZO library: context, host-side validation, workspace planning and the
// sequencing of Algorithm 1 / Algorithm 2 over the grouped kernels.
#include <cuda.h>

#include <algorithm>
#include <cstdio>
#include <cstring>
#include <mutex>
#include <new>
#include <vector>

#include "agzo_common.cuh"
#include "agzo_resident.cuh"
#include "agzo_split.cuh"
#include "agzo_tc.cuh"

using namespace agzo;

namespace {

constexpr uint32_t kMagic = 0xA620B200u;
constexpr size_t kAlign = 256;
constexpr size_t kHeaderBytes = 256;          // DevStatus, and from kCountersAt on the counters of the resident extraction
constexpr size_t kCountersAt = 128;
static_assert(sizeof(DevStatus) <= kCountersAt && kCountersAt + kResMaxUnits * sizeof(unsigned long long) <= kHeaderBytes, "header");
constexpr int64_t kDefaultWaveBytes = 8ll << 30;
constexpr int64_t kL2ResidentWaveBytes = 64ll << 20;   // a wave's X up to this size is still in L2 at its next sweep

inline size_t align_up(size_t x, size_t a = kAlign) { return (x + a - 1) / a * a; }

struct Plan {
  std::vector<DevLayer> dev;       // one per layer, scratch pointers filled
  std::vector<int> tile_start;     // n + 1
  std::vector<int> wave_end;       // exclusive end index of each extraction wave
  std::vector<int> wave_region;    // scratch region (= helper stream) of each wave, -1 = nothing to do
  // the Y panels of a wave's layers lie one after another at the end of the wave's scratch, so that a
  // token-sharded run can sum all of them over the ranks in one call
  std::vector<float*> wave_y;
  std::vector<size_t> wave_y_count;   // floats, alignment gaps included
  int regions = 1;
  int total_tiles = 0;
  int tile_rows = kRmwMaxTileRows, slow_rows = 32;     // of layers on the vector path, and of the others
  int max_r = 0;
  int cc_max_r = 0;                // largest rank among layers on the vector path
  int fast_mode_mask = 0;          // storage modes present among layers on the vector path
  bool any_slow = false;           // some layer needs the scalar kernel
  bool has_extract = false;
  bool split = false;              // products in parts (agzo_split.cuh) for the waves that they can serve
  // tensor-core in-place pass: work items per layer (prefix, n + 1), zero-length for other layers
  std::vector<int> item_start;
  int total_items = 0;
  int max_rp = 0;
  int max_b_bytes = 0;   // largest B operand area of a tensor-core pass item
  bool staged_r = false;           // the tensor-core pass copies R tiles that a fill kernel wrote to scratch
  int max_row_tiles = 0;
  size_t image_bytes = 0;
};

constexpr int kRmwTcMinRank = 5;   // where the option has not been set

struct PlanOpts {
  int64_t wave_bytes;
  int extract_path;      // 0 auto, 1 CUDA-core only, 2 tensor-core required
  int rmw_path;          // 0 auto, 1 CUDA-core only, 2 tensor cores wherever a layer allows it
  int rmw_tc_min_rank;   // auto: layers with r >= this use the tensor-core pass; 0: kRmwTcMinRank, and lists of few weights the CUDA-core pass
  int rmw_tc_panels;     // column panels per work item of the tensor-core pass (1 or 2)
  int rmw_stage_r;       // 0: stage R in scratch when some rank exceeds 16; 1: never; 2: always
  bool tc_available;
  int extract_fused;     // 1: power steps of eligible layers run in the fused single-pass kernel; 2: also on
                         // cluster sizes that leave much of the device idle
  bool share_inputs;     // consecutive layers with the same X are served by one sweep
  int extract_regions;   // 1: waves run one after another; 2: alternate waves use two scratch regions
                         // and two helper streams, so one wave's small kernels overlap the other's sweeps
  int split;             // the products that the TMA kernels do not take run in parts on the tensor cores: 0 never, 1 where that pays, 2 always
  int sm_count;          // of the device; when sizing without one, any number will do
  const FusedCaps* fused_caps;   // what the device holds of the fused kernel; null when sizing without a device
};

}  // namespace

struct agzo_ctx {
  uint32_t magic;
  int device;
  int sm_count;
  char* ws;
  size_t ws_bytes;
  int last_cuda;
  int extract_path;        // 0 auto, 1 CUDA-core only, 2 tensor-core required
  int rmw_path;            // 0 auto, 1 CUDA-core only, 2 tensor cores wherever possible
  int rmw_tc_min_rank;
  int rmw_tc_slots;        // ring slots of the tensor-core pass, 0 = as many as fit
  int rmw_tc_inflight;     // loads in flight per CTA, 0 = by rank
  int rmw_tc_panels;       // column panels per work item (1 or 2), 0 = by rank
  int rmw_stage_r;         // 0 auto, 1 never, 2 always
  int64_t wave_bytes;
  int extract_streams;     // 1 or 2 (see PlanOpts::extract_regions)
  int extract_fused;       // 0 off, 1 fused power-step kernel where it pays, 2 wherever a layer's shape allows it
  int share_inputs;        // 1: consecutive layers with the same X share the sweeps over it
  int extract_split;       // products that the TMA kernels do not take, in bf16 parts on the tensor cores: 1 where that is faster, 2 always, 0 never
  int extract_resident;    // 1: inputs that fit the chip's shared memory are extracted by one kernel where that is faster; 2: always; 0: never
  // the layer list that extraction last looked at for that kernel, and what came of it
  std::vector<agzo_layer> resident_cached;
  bool resident_known, resident_ok;
  int resident_admitted;   // whether the other kernels would take the list in this workspace: 1, 0, -1 not looked at yet
  ResidentLaunch resident;
  // staged R images in scratch: valid for this seed until the plan changes or extraction uses the scratch
  bool rimg_valid;
  uint64_t rimg_seed;
  cudaStream_t rimg_stream;   // stream the images were written on: another stream refills them
  agzo_allreduce_fn allreduce;   // token-sharded extraction: sums a wave's Y panels over the ranks
  void* allreduce_user;
  int64_t token_offset;    // global index of this rank's first token
  cudaStream_t aux[2];     // helper streams of extraction, forked from and joined to the caller's stream
  cudaEvent_t fork_ev, join_ev[2];
  // descriptors last uploaded
  std::vector<agzo_layer> cached;
  bool cached_valid;
  Plan plan;
  // the tables as they were built, and pinned staging for those too large for a kernel's parameters
  std::vector<char> h_tables;
  void* h_stage;
  size_t h_stage_bytes;
  bool h_stage_busy;       // a copy out of h_stage may still be under way (stage_ev tells)
  cudaEvent_t stage_ev;
  bool stage_pending;
  cudaStream_t stage_stream;  // stream of the last table upload: a call on another stream waits for stage_ev
  unsigned long long tables_capture;   // the capture that holds that upload, 0: it was made outside of any
  bool tables_captured;    // a captured call reads the tables of a list without weights (see prepare)
  TcState tc;
  ResidentCaps resident_caps;
  // measurement aid: event pairs around the launches of one kernel class
  int debug_fail_step_call;   // test option: the n-th internal call of agzo_step fails on the host, 0 = off
  int debug_missing_class;       // test option: in launches of this kernel class a wait runs out (ExtractWave::missing), 0 = off
  int debug_refuse_resident;  // test option: launches of the resident kernel end as if the device had refused them
  int time_class;
  std::vector<cudaEvent_t> events;   // pairs: start, stop
  size_t events_used;
  int64_t launches;
  unsigned power_steps;    // fused power steps issued so far: the number that tells one from the one before it
};

namespace {

// What is asked of a device and set for its kernels is the same for every agzo_ctx: done once per CUDA context, since the
// kernels' limits end with the context (cudaDeviceReset).
cudaError_t device_init(int device, TcState* tc, ResidentCaps* resident) {
  struct Known { unsigned long long id; TcState st; ResidentCaps resident; };
  static std::mutex mu;
  static Known known[kMaxDevices];
  const unsigned long long id = current_context_id(device);
  std::lock_guard<std::mutex> lock(mu);
  Known* k = device < kMaxDevices ? known + device : nullptr;
  if (k && id != 0 && k->id == id) { *tc = k->st; *resident = k->resident; return cudaSuccess; }
  TcState st;
  ResidentCaps rc;
  cudaError_t e = panel_qr_init(&st.qr_wide);
  if (e == cudaSuccess) e = rmw_init();
  if (e == cudaSuccess) e = tc_init(&st, device);
  if (e == cudaSuccess && st.available) e = resident_init(st.fused.sm_count, &rc);
  if (e != cudaSuccess) return e;
  if (k) { k->id = id; k->st = st; k->resident = rc; }
  *tc = st;
  *resident = rc;
  return cudaSuccess;
}

#define CU(ctx, expr)                              \
  do {                                             \
    cudaError_t e__ = (expr);                      \
    if (e__ != cudaSuccess) {                      \
      (ctx)->last_cuda = (int)e__;                 \
      return AGZO_ERR_CUDA;                        \
    }                                              \
  } while (0)

// Launch bookkeeping: counts every kernel-launching call and, for the class being timed,
// brackets it with an event pair on the stream.
struct Timed {
  agzo_ctx* c;
  cudaStream_t s;
  bool on;
  Timed(agzo_ctx* ctx, int cls, cudaStream_t st, int n_kernels = 1) : c(ctx), s(st), on(false) {
    c->launches += n_kernels;
    if (c->time_class != cls) return;
    if (c->events_used + 2 > c->events.size()) {
      for (int i = 0; i < 2; ++i) {
        cudaEvent_t e = nullptr;
        if (cudaEventCreate(&e) != cudaSuccess) return;
        c->events.push_back(e);
      }
    }
    on = cudaEventRecord(c->events[c->events_used], s) == cudaSuccess;
  }
  ~Timed() {
    if (!on) return;
    cudaEventRecord(c->events[c->events_used + 1], s);
    c->events_used += 2;
  }
};

bool aligned16(const void* p) { return (reinterpret_cast<uintptr_t>(p) & 15u) == 0; }

enum Need { NEED_RMW = 1, NEED_EXTRACT = 2 };

agzo_status validate(const agzo_layer* L, int n, int need) {
  if (n < 0 || n > AGZO_MAX_LAYERS) return AGZO_ERR_INVALID_ARG;
  if (n > 0 && !L) return AGZO_ERR_INVALID_ARG;
  for (int i = 0; i < n; ++i) {
    const agzo_layer& a = L[i];
    if (a.reserved != 0) return AGZO_ERR_INVALID_ARG;
    if (a.d_in < 1 || a.d_out < 0) return AGZO_ERR_INVALID_ARG;
    if (a.r < 1 || a.r > AGZO_MAX_RANK || a.r > a.d_in) return AGZO_ERR_INVALID_ARG;
    if (!a.V || a.ldv < a.d_in || (reinterpret_cast<uintptr_t>(a.V) & 3u)) return AGZO_ERR_INVALID_ARG;
    if (need & NEED_RMW) {
      if (a.d_out < 1) return AGZO_ERR_INVALID_ARG;
      if (a.w_dtype != AGZO_BF16 && a.w_dtype != AGZO_F32) return AGZO_ERR_UNSUPPORTED;
      if (!a.W || a.ldw < a.d_in) return AGZO_ERR_INVALID_ARG;
      const size_t es = a.w_dtype == AGZO_BF16 ? 2 : 4;
      if (reinterpret_cast<uintptr_t>(a.W) & (es - 1)) return AGZO_ERR_INVALID_ARG;
      if (a.W16) {
        if (a.w_dtype != AGZO_F32) return AGZO_ERR_UNSUPPORTED;
        if (a.ldw16 < a.d_in || (reinterpret_cast<uintptr_t>(a.W16) & 1u)) return AGZO_ERR_INVALID_ARG;
      }
    }
    if (need & NEED_EXTRACT) {
      if (a.x_dtype != AGZO_BF16 && a.x_dtype != AGZO_F32) return AGZO_ERR_UNSUPPORTED;
      if (!a.X || a.m < 1 || a.ldx < a.d_in || a.r > a.m) return AGZO_ERR_INVALID_ARG;
      const size_t es = a.x_dtype == AGZO_BF16 ? 2 : 4;
      if (reinterpret_cast<uintptr_t>(a.X) & (es - 1)) return AGZO_ERR_INVALID_ARG;
    }
  }
  return AGZO_OK;
}

bool has_x(const agzo_layer& a) { return a.X != nullptr && a.m >= 1; }
bool same_input(const agzo_layer& a, const agzo_layer& b) {
  return a.X == b.X && a.ldx == b.ldx && a.m == b.m && a.d_in == b.d_in && a.x_dtype == b.x_dtype;
}

// Token slabs of the X^T T product.  CUDA-core kernels: cc_slab_rows.  Tensor-core kernels: slabs of 2048 tokens (32 pipeline
// steps per CTA) when the layer has that many.  When the call's layers fill the grid by their column blocks alone (long_slabs), a slab is up to
// 16384 tokens: every slab costs a partial Y (r x d_in floats written, and read again by the
// panel QR), and the CTAs' pipelines start and drain less often.
constexpr int kLongSlabColumnBlocks = 1024;   // 128-column blocks over all layers from which slabs are long
// blocks: 128-column blocks over the call's layers on the CUDA-core path, or (split) over the units of the products in parts; 0 = the most
// slabs the layer can get (sizing).
void slab_shape(const agzo_layer& a, bool tc, bool long_slabs, long long blocks, bool split, int sm_count, int* slabs, int* slab_rows) {
  int rows;
  if (tc) {
    rows = a.m >= 8192 ? (long_slabs ? (a.m < 16384 ? a.m : 16384) : 2048) : (a.m + 3) / 4;
    rows = (rows + 127) / 128 * 128;      // whole tiles of every tensor-core kernel (64 or 128 tokens)
    if (rows < 256) rows = 256;
  } else if (blocks > 0) {
    rows = split ? split_slab_rows(a.m, blocks, sm_count) : cc_slab_rows(a.m, blocks, sm_count);
  } else {
    const int most = (a.m + kCcMinSlabRows - 1) / kCcMinSlabRows;
    *slabs = most < kCcMaxSlabs ? most : kCcMaxSlabs;
    *slab_rows = 0;
    return;
  }
  *slab_rows = rows;
  *slabs = (a.m + rows - 1) / rows;
}


constexpr size_t kMapBytes = 512;   // four TMA descriptors per layer
// device tables after the header: layer records | tile prefix and item prefix (n + 1 ints each) | TMA descriptors
size_t prefix_bytes(int n) { return align_up((size_t)2 * (n + 1) * sizeof(int)); }
size_t table_bytes(int n) {
  return align_up((size_t)n * sizeof(DevLayer)) + prefix_bytes(n) + align_up((size_t)n * kMapBytes);
}
size_t maps_offset(int n) { return kHeaderBytes + align_up((size_t)n * sizeof(DevLayer)) + prefix_bytes(n); }

// Builds the device records.  ws == nullptr: only sizes are computed (scratch_needed).
agzo_status build_plan(const agzo_layer* L, int n, char* ws, size_t ws_bytes, const PlanOpts& opts,
                       Plan* plan, size_t* scratch_needed) {
  const int64_t wave_bytes = opts.wave_bytes;
  const int extract_path = opts.extract_path;
  const bool tc_available = opts.tc_available;
  plan->dev.assign(n, DevLayer{});
  plan->tile_start.assign(n + 1, 0);
  plan->wave_end.clear();
  plan->wave_region.clear();
  plan->wave_y.clear();
  plan->wave_y_count.clear();
  const int regions = opts.extract_regions == 2 ? 2 : 1;
  plan->regions = regions;
  plan->max_r = 0;
  plan->cc_max_r = 0;
  plan->fast_mode_mask = 0;
  plan->any_slow = false;
  plan->has_extract = false;
  plan->item_start.assign(n + 1, 0);
  plan->total_items = 0;
  plan->max_rp = 0;
  plan->max_b_bytes = 0;
  const size_t base = kHeaderBytes + table_bytes(n);
  const size_t scratch_all = ws ? (ws_bytes > base ? ws_bytes - base : 0) : (size_t)-1;
  const size_t scratch_cap = ws ? scratch_all / regions / kAlign * kAlign : (size_t)-1;   // per region
  int real_waves = 0;
  size_t max_wave_scratch = 0;

  // Which layers take the tensor-core pass, and whether their R operands are staged in scratch
  // (ranks above 16): the operand image of every 128-row tile of every such layer, laid out from
  // the start of the scratch area (which extraction uses at other times).
  // 16-byte accesses possible for every operand of the CUDA-core pass
  auto vector_rows = [&](const agzo_layer& a) {
    const size_t es = a.w_dtype == AGZO_BF16 ? 2 : 4;
    bool vec = a.W && aligned16(a.W) && (a.ldw * es) % 16 == 0 && a.d_in % 8 == 0 && aligned16(a.V) && a.ldv % 4 == 0;
    if (a.W16) vec = vec && aligned16(a.W16) && (a.ldw16 * 2) % 16 == 0;
    return vec;
  };
  // A list of few weights, which L2 holds between the passes, is a matter of set-up, of which the tensor-core pass has more: where it
  // would take over at its own rank it does so from 32 M weights up to rank 8, from 3 M up to rank 16 (CUDA cores / tensor cores, us per pass:
  // 0.8 M r = 8 4.8 / 8.6, r = 16 5.0 / 8.5; 8.4 M r = 8 9.5 / 10.9, r = 16 13.0 / 11.2; 31 M r = 5 23.4 / 27.2, r = 8 23.5 / 25.0; 50 M r = 5
  // 41.3 / 40.7, r = 8 43.4 / 37.9).
  bool few_weights = false;
  if (opts.rmw_path == 0 && opts.rmw_tc_min_rank == 0) {
    int64_t weights = 0;
    int max_r = 0;
    for (int i = 0; i < n; ++i)
      if (rmw_tc_eligible(L[i])) {
        weights += (int64_t)L[i].d_out * L[i].d_in;
        max_r = std::max(max_r, L[i].r);
      }
    few_weights = weights <= (max_r <= 8 ? 32000000ll : max_r <= 16 ? 3000000ll : 0ll);
  }
  const int tc_min_rank = opts.rmw_tc_min_rank ? opts.rmw_tc_min_rank : kRmwTcMinRank;
  std::vector<char> vector_path((size_t)n), tc_pass((size_t)n);      // of the in-place passes
  for (int i = 0; i < n; ++i) {
    vector_path[i] = vector_rows(L[i]);
    // from rank 3 on the element-by-element kernel is no alternative where the vector kernels cannot run
    tc_pass[i] = tc_available && opts.rmw_path != 1 && rmw_tc_eligible(L[i]) &&
                 (opts.rmw_path == 2 || (L[i].r >= tc_min_rank && !few_weights) || (L[i].r >= 3 && !vector_path[i]));
  }
  {
    size_t img = 0;
    int max_tiles = 0, max_rp_all = 0;
    for (int i = 0; i < n; ++i) {
      if (!tc_pass[i]) continue;
      img += rmw_tc_image_bytes(L[i]);
      max_tiles = std::max(max_tiles, (L[i].d_out + 127) / 128);
      max_rp_all = std::max(max_rp_all, (L[i].r + 7) & ~7);
    }
    const size_t room = ws ? (ws_bytes > base ? ws_bytes - base : 0) : (size_t)-1;
    const bool want = opts.rmw_stage_r == 2 || (opts.rmw_stage_r == 0 && max_rp_all > 16);
    plan->staged_r = want && img > 0 && img <= room;
    plan->max_row_tiles = max_tiles;
    plan->image_bytes = want ? img : 0;
  }
  // Rows per tile of the CUDA-core pass.  The CTAs, all resident, take tiles in turn, so a pass lasts as many rounds as the one with most
  // tiles has, each a tile's rows and what setting up a tile costs beside them (R, the slice of A^T, the record; with the slice in shared memory as
  // many rows again as there are ranks): 32 rows above rank 8, 22 where there are 16-bit weights, five or six of fp32; where there are several
  // rounds, CTAs have drifted apart by half a tile at the end.  Multiples of eight, the tallest of the cheapest.
  // From 100 MB of fp32 weights on (ranks up to 4, strips of 512 columns all in use) and 250 MB of bf16 the memory sets the time whatever
  // the rounds, and takes it best in tiles of 32 and of 128 rows (bf16 lists of more than 640 MB at ranks 3 and 4 of 256, as below: the same on a cool
  // chip, 903 and 899 us for 28 1.7B-shaped blocks, r = 4, but with the power cap active, where the set-up's work costs clock, 947 and 920; ranks 1 and
  // 2 keep 128: r = 2 875 / 898 and 890 / 884).
  // Measured on 1377 lists of up to 700 MB at every height and 1148 of up to 4.4 GB at ten: on the mean 1.6 % above the best height (with 2 to 12 rows
  // for the set-up and without the two lines 2.4); of those above 6 us four are more than 3 % slower than at the height that gives each CTA sixteen
  // tiles, of at least 32 rows (33 without: two fp32 0.6B-shaped blocks, r = 1, 51 us at 224 rows, 44 at 32; thirty bf16 1024 x 1024, r = 1, 24.6 at
  // 24 rows, 15.3 at 256).
  // Other lists of more than 640 MB: the tallest tiles of which each CTA gets sixteen, for rank 1, whose set-up
  // is least, half as tall.
  // The element-by-element kernel has heights of its own (32 rows at most): one 1001 x 1001 layer among four fp32 8B-shaped blocks, r = 8,
  // 1162 us per pass with one height for both, now 998.
  auto height = [&](bool slow) {
    struct Strip { int d_out, n; };
    std::vector<Strip> strips;             // 512 columns wide, by height
    int best = slow ? 32 : kRmwMaxTileRows;
    int max_r = 0;
    int64_t bytes = 0, weights = 0, strip_rows = 0;
    bool any_f32 = false, any_bf16 = false, any_pair = false;
    for (int i = 0; i < n; ++i) {
      if (!L[i].W || tc_pass[i] || (vector_path[i] != 0) == slow) continue;
      const int count = (L[i].d_in + kRmwTileCols - 1) / kRmwTileCols;
      max_r = std::max(max_r, L[i].r);
      const int64_t size = (int64_t)L[i].d_out * L[i].d_in;
      weights += size;
      strip_rows += (int64_t)count * L[i].d_out;
      bytes += size * ((L[i].w_dtype == AGZO_BF16 ? 2 : 4) + (L[i].W16 ? 2 : 0));
      (L[i].w_dtype == AGZO_BF16 ? any_bf16 : L[i].W16 ? any_pair : any_f32) = true;
      auto same = std::find_if(strips.begin(), strips.end(), [&](const Strip& s) { return s.d_out == L[i].d_out; });
      if (same != strips.end()) same->n += count; else strips.push_back(Strip{L[i].d_out, count});
    }
    const long long ctas = (slow ? 4ll : max_r <= 8 ? 2ll : 1ll) * opts.sm_count;       // element by element: four on an SM
    const int setup = slow ? (max_r == 1 ? 3 : std::min(12, 3 + 3 * max_r)) * (any_bf16 || max_r > 8 ? 2 : 1)
                           : max_r > 8 ? 64 : any_bf16 || any_pair ? 44 : std::min(12, std::max(9, 3 + 3 * max_r));
    long long least = -1;
    auto tiles_of = [&](int rows) {
      long long tiles = 0;
      for (const Strip& s : strips) tiles += (long long)s.n * ((s.d_out + rows - 1) / rows);
      return tiles;
    };
    const bool few_ranks = !slow && max_r <= 4;
    const bool large = bytes > (640ll << 20);
    if (few_ranks && !any_bf16 && !any_pair && bytes >= (100ll << 20) && 100 * weights >= 98 * strip_rows * kRmwTileCols) return 32;
    if (few_ranks && any_bf16 && !any_f32 && !any_pair && bytes >= (250ll << 20) && !(large && max_r >= 3)) return 128;
    if (large) {
      best = slow ? 32 : max_r == 1 ? kRmwMaxTileRows / 2 : kRmwMaxTileRows;
      while (best > 32 && tiles_of(best) < 32ll * opts.sm_count) best /= 2;
      return best;
    }
    for (int rows = slow ? 32 : kRmwMaxTileRows; rows >= 8 && !strips.empty(); rows -= 8) {
      const long long rounds = (tiles_of(rows) + ctas - 1) / ctas;
      const long long cost = rounds * (2 * rows + setup + (max_r > 16 ? 2 * max_r : 0)) + (rounds > 1 ? rows : 0);     // in half rows
      if (least < 0 || cost < least) { least = cost; best = rows; }
    }
    return best;
  };
  plan->tile_rows = height(false);
  plan->slow_rows = height(true);
  // A list with fewer items than three quarters of the SMs gets shorter ones (one 4096 x 4096 layer, r = 64: 64 items of eight
  // row tiles 23.7 us, 128 of four 16.5, 256 of two 20.3; r = 8: 128 of four 14.5, 256 of two 16.7).
  int halvings = 0;
  for (; halvings < 3; ++halvings) {
    long long count = 0;
    for (int i = 0; i < n && 4 * count < 3ll * opts.sm_count; ++i) {
      if (!tc_pass[i]) continue;
      DevLayer D{};
      rmw_tc_shape(L[i], opts.rmw_tc_panels, plan->staged_r, halvings, &D);
      count += (long long)D.rtc_panels * D.rtc_chunks;
    }
    if (4 * count >= 3ll * opts.sm_count || count == 0) break;
  }
  // Where the items make a few rounds over the SMs, the last one is mostly empty: the list's last layers get shorter items still, as many
  // layers and as short as leave the CTA with most to do the least (row tiles of 128 x 256, an item's set-up counted as one: two 0.6B-shaped
  // blocks, r = 8, with all items half as high 25.8 -> 35 us).  Four 0.6B-shaped blocks, r = 8, 52.4 -> 48.0 us per pass, three, r = 64, 54.0 -> 42.8,
  // five 2048 x 2048 layers, r = 12, 24.8 -> 19.5; 23 of 45 lists unchanged, none slower.
  // Layers of one shape have the same items, in runs of equal ones, and the layers before the first that gets shorter ones have the same
  // in all the tries: 9 us for 28 layers of 0.6B shape, 3 for seven of 8B shape; item by item it took 45 and 115.
  int fine_from = n, fine_halvings = 0;
  {
    std::vector<int> which;
    long long count = 0;
    const long long limit = 10ll * opts.sm_count;
    for (int i = 0; i < n && count <= limit; ++i) {
      if (!tc_pass[i]) continue;
      DevLayer D{};
      rmw_tc_shape(L[i], opts.rmw_tc_panels, plan->staged_r, halvings, &D);
      which.push_back(i);
      count += (long long)D.rtc_panels * D.rtc_chunks;
    }
    if (count > opts.sm_count && count <= limit) {
      struct Run { float load; int n; };
      struct Items { int layer; std::vector<Run> runs[3]; };         // of the layer and those of its shape, by halvings more
      struct Load { std::vector<float> cta; int next; };
      auto add_run = [](std::vector<Run>& v, float load, int n) {
        if (!v.empty() && v.back().load == load) v.back().n += n; else if (n > 0) v.push_back(Run{load, n});
      };
      std::vector<Items> items;
      std::vector<int> items_of;                                     // of which[p]
      for (int i : which) {
        const agzo_layer& a = L[i];
        size_t k = 0;
        while (k < items.size() && (L[items[k].layer].d_out != a.d_out || L[items[k].layer].d_in != a.d_in || L[items[k].layer].r != a.r)) ++k;
        items_of.push_back((int)k);
        if (k < items.size()) continue;
        items.emplace_back();
        items[k].layer = i;
        for (int more = 0; more < 3; ++more) {
          DevLayer D{};
          rmw_tc_shape(a, opts.rmw_tc_panels, plan->staged_r, halvings + more, &D);
          const int row_tiles = (a.d_out + 127) / 128, cols = D.rtc_np * D.rtc_cw;
          for (int c = 0; c < D.rtc_chunks; ++c) {
            const float high = (float)std::min(D.rtc_chunk_blocks, row_tiles - c * D.rtc_chunk_blocks);
            add_run(items[k].runs[more], 1.f + high * (float)cols / 256.f, D.rtc_panels - 1);
            add_run(items[k].runs[more], 1.f + high * (float)(a.d_in - (D.rtc_panels - 1) * cols) / 256.f, 1);
          }
        }
      }
      const int G = opts.sm_count;
      auto add = [&](Load& l, const std::vector<Run>& runs) {        // in turn to the CTAs
        for (const Run& run : runs) {
          const float rounds = (float)(run.n / G) * run.load;
          const int rest = run.n % G, upto = std::min(rest, G - l.next);
          float* c = l.cta.data();
          if (rounds > 0.f)
            for (int x = 0; x < G; ++x) c[x] += rounds;
          for (int x = 0; x < upto; ++x) c[l.next + x] += run.load;
          for (int x = 0; x < rest - upto; ++x) c[x] += run.load;
          l.next = (l.next + rest) % G;
        }
      };
      auto most = [](const Load& l) { return *std::max_element(l.cta.begin(), l.cta.end()); };
      Load all{std::vector<float>((size_t)G, 0.f), 0}, tried;
      std::vector<Load> before;                                      // load ahead of which[p], from the last 24 layers on
      const size_t first = which.size() > 24 ? which.size() - 24 : 0;
      for (size_t p = 0; p < which.size(); ++p) {
        if (p >= first) before.push_back(all);
        add(all, items[items_of[p]].runs[0]);
      }
      float least = 0.97f * most(all), sum = 0.f;
      for (float l : all.cta) sum += l;
      for (size_t k = 1; k <= before.size() && least * (float)G > sum; k += k < 4 ? 1 : k / 2)      // none can do better than share it evenly
        for (int more = 1; more <= 2; ++more) {
          const size_t from = which.size() - k;
          tried = before[from - first];
          for (size_t p = from; p < which.size(); ++p) add(tried, items[items_of[p]].runs[more]);
          const float m = most(tried);
          if (m < least) { least = m; fine_from = which[from]; fine_halvings = more; }
        }
    }
  }
  size_t img_off = 0;
  int tiles = 0;
  long long items = 0;
  for (int i = 0; i < n; ++i) {
    const agzo_layer& a = L[i];
    DevLayer& D = plan->dev[i];
    D.W = a.W; D.W16 = a.W16; D.X = a.X; D.V = a.V;
    D.ldw = a.ldw; D.ldw16 = a.ldw16; D.ldx = a.ldx; D.ldv = a.ldv;
    D.w_dtype = a.w_dtype; D.x_dtype = a.x_dtype;
    D.d_out = a.d_out; D.d_in = a.d_in; D.m = a.m; D.r = a.r;
    D.layer_id = a.layer_id;
    D.rmw_mode = a.W16 ? RMW_PAIR_COMPUTE : (a.w_dtype == AGZO_BF16 ? RMW_BF16 : RMW_F32);
    const bool vec = vector_path[i] != 0;
    D.vec_ok = vec ? 1 : 0;
    // bf16 weights of sufficient rank go through the tensor-core pass and get no CUDA-core tiles
    const bool tc_rmw = tc_pass[i] != 0;
    plan->item_start[i] = (int)items;
    if (tc_rmw) {
      rmw_tc_shape(a, opts.rmw_tc_panels, plan->staged_r, halvings + (i >= fine_from ? fine_halvings : 0), &D);
      if (plan->staged_r && ws) {
        D.rimg = reinterpret_cast<unsigned char*>(ws + base + img_off);
        D.rimg_tile_bytes = (int)(rmw_tc_image_bytes(a) / (size_t)((a.d_out + 127) / 128));
      }
      img_off += rmw_tc_image_bytes(a);
      D.rtc_item0 = (int)items;
      items += (long long)D.rtc_panels * D.rtc_chunks;
      if (items > 0x7fffffff) return AGZO_ERR_INVALID_ARG;
      if (D.rtc_rp > plan->max_rp) plan->max_rp = D.rtc_rp;
      plan->max_b_bytes = std::max(plan->max_b_bytes, rmw_tc_b_bytes(D));
      if (ws) D.wmap = ws + maps_offset(n) + (size_t)i * kMapBytes + 384;
    } else if (a.W) {
      if (vec) {
        plan->fast_mode_mask |= 1 << D.rmw_mode;
        plan->cc_max_r = std::max(plan->cc_max_r, a.r);
      } else {
        plan->any_slow = true;
      }
    }
    D.tile0 = tiles;
    D.tiles_c = (a.d_in + kRmwTileCols - 1) / kRmwTileCols;
    const int rows = vec ? plan->tile_rows : plan->slow_rows;
    D.tiles_r = (a.W && !tc_rmw) ? (a.d_out + rows - 1) / rows : 0;
    plan->tile_start[i] = tiles;
    const long long nt = (long long)D.tiles_c * D.tiles_r;
    if (tiles + nt > 0x7fffffff) return AGZO_ERR_INVALID_ARG;
    tiles += (int)nt;
    if (a.r > plan->max_r) plan->max_r = a.r;
  }
  plan->tile_start[n] = tiles;
  plan->total_tiles = tiles;
  plan->item_start[n] = (int)items;
  plan->total_items = (int)items;

  // extraction waves: consecutive layers whose activations fit the wave budget and whose
  // scratch fits the workspace
  auto on_tc = [&](const agzo_layer& a) { return extract_path != 1 && tc_available && tc_eligible(a); };
  // the fused power step for a layer, or for layers on one X taken as one layer of `ranks` ranks
  auto with_ranks = [](agzo_layer a, int ranks) { a.r = ranks; return a; };
  auto fuses = [&](const agzo_layer& a, int ranks) {
    return opts.extract_fused && extract_path != 3 && on_tc(a) && ranks <= 16 &&
           fused_eligible(opts.fused_caps, with_ranks(a, ranks), opts.extract_fused == 2);
  };
  long long column_blocks = 0, cc_blocks = 0;
  for (int k = 0; k < n; ++k)
    if (has_x(L[k]))
      (on_tc(L[k]) ? column_blocks : cc_blocks) += (L[k].d_in + 127) / 128;
  plan->split = false;
  if (opts.split && cc_blocks > 0) {
    std::vector<int> which;
    for (int k = 0; k < n; ++k)
      if (has_x(L[k]) && !on_tc(L[k])) which.push_back(k);
    plan->split = opts.split == 2 || split_pays(L, which, opts.share_inputs, opts.sm_count);
  }
  long long split_blocks = 0;
  if (plan->split) {                       // its units are panels of the layers on one X
    for (int k = 0; k < n;) {
      int run = 1, all = L[k].r;
      while (opts.share_inputs && has_x(L[k]) && k + run < n && has_x(L[k + run]) && same_input(L[k], L[k + run])) all += L[k + run++].r;
      if (has_x(L[k]) && !on_tc(L[k])) split_blocks += (long long)((L[k].d_in + 127) / 128) * ((all + kSplitMaxRanks - 1) / kSplitMaxRanks);
      k += run;
    }
  }
  const bool long_slabs_any = column_blocks >= kLongSlabColumnBlocks;
  int extract_max_r = 0;
  for (int k = 0; k < n; ++k)
    if (has_x(L[k])) extract_max_r = std::max(extract_max_r, L[k].r);
  // scratch of a layer that does not depend on its slabs: T, Y and, where the call has a rank whose panel QR uses them, the Gram shares
  auto layer_need = [&](const agzo_layer& a, bool tc) {
    return (tc ? 0 : align_up((size_t)a.m * a.r * 4)) + align_up((size_t)a.r * a.d_in * 4) + align_up(panel_gram_bytes(a.d_in, a.r, extract_max_r));
  };
  auto ypart_bytes = [&](int parts, int ranks, int d_in) { return align_up((size_t)parts * ranks * (size_t)d_in * 4); };
  // Of the tokens seen last, for either kernel: the layers of a call mostly have as many, and trying the counts takes 0.2 us each time, three times a
  // layer (a list of 64 layers: 65 -> 30 us, with both kernels' counts 101 -> 31; two fp32 0.6B-shaped blocks, a new state's first step 655 -> 644)
  struct { int m, slabs, rows; } seen[2] = {};
  auto slabs_of = [&](const agzo_layer& a, bool tc, bool split, int* slabs, int* slab_rows) {
    if (!tc && seen[split].m == a.m) {
      *slabs = seen[split].slabs; *slab_rows = seen[split].rows;
    } else {
      slab_shape(a, tc, long_slabs_any, !ws ? 0 : split ? split_blocks : cc_blocks, split, opts.sm_count, slabs, slab_rows);
      if (!tc) seen[split] = {a.m, *slabs, *slab_rows};
    }
    // a workspace of less than agzo_workspace_bytes takes fewer slabs on the CUDA-core path, as long as one is left
    for (int want = *slabs; ws && !tc && want > 1 && ypart_bytes(*slabs, a.r, a.d_in) + layer_need(a, tc) > scratch_cap;) {
      --want;
      *slab_rows = ((a.m + want - 1) / want + 31) / 32 * 32;
      *slabs = (a.m + *slab_rows - 1) / *slab_rows;
    }
  };
  // partial sums of Y that a unit's last product can leave: slabs, or shares of a fused launch
  auto parts_of = [&](const agzo_layer& a, bool tc, bool fused, int ranks) {
    int slabs, slab_rows;
    slabs_of(a, tc, false, &slabs, &slab_rows);
    if (!tc && plan->split) {              // either product
      int split_slabs;
      slabs_of(a, tc, true, &split_slabs, &slab_rows);
      slabs = std::max(slabs, split_slabs);
    }
    if (!fused) return slabs;
    const int C = ws ? fused_cluster_size(opts.fused_caps, with_ranks(a, ranks), opts.extract_fused == 2) : fused_min_cluster(a);
    return std::max(slabs, fused_parts_bound(a, C));
  };
  int i = 0;
  while (i < n) {
    if (!has_x(L[i])) {
      ++i;
      plan->wave_end.push_back(i); plan->wave_region.push_back(-1);
      plan->wave_y.push_back(nullptr); plan->wave_y_count.push_back(0);
      continue;
    }
    const int region = real_waves++ % regions;
    plan->has_extract = true;
    size_t used = 0, used_y = 0;    // scratch of the wave so far; the part of it that is Y panels
    int64_t xbytes = 0;
    int j = i;
    const bool wave_tc = on_tc(L[i]);
    while (j < n && has_x(L[j])) {
      const bool tc = on_tc(L[j]);
      if (tc != wave_tc) break;      // a wave runs on one kind of kernel
      // A unit is one layer, or a run of consecutive layers that read the same X.  A run of at most 16 ranks in all takes
      // the fused power step as one layer of that many ranks; a larger one the two sweeps, which serve it with two
      // reads of X per step where fusing it layer by layer would read X once for each (unless fusing is forced).
      int glen = 1, ranks = L[j].r;
      bool fused = tc && fuses(L[j], ranks);
      if (tc && opts.share_inputs) {
        int run = 1, all = ranks;
        while (j + run < n && has_x(L[j + run]) && same_input(L[j], L[j + run])) all += L[j + run++].r;
        if (run > 1 && fuses(L[j], all)) {
          glen = run; ranks = all; fused = true;
        } else if (run > 1 && !(fused && opts.extract_fused == 2)) {
          fused = false;
          while (glen < run && tc_operand_rows(ranks + L[j + glen].r) <= 256 &&
                 !(opts.extract_fused == 2 && fuses(L[j + glen], L[j + glen].r)))
            ranks += L[j + glen++].r;
        }
      }
      auto unit_need = [&]() {
        size_t b = ypart_bytes(parts_of(L[j], tc, fused, ranks), ranks, L[j].d_in);
        for (int g = 0; g < glen; ++g) b += layer_need(L[j + g], tc);
        if (tc) b += tc_panel_bytes(L[j], ranks);
        return b;
      };
      size_t need = unit_need();
      const int64_t xb = (int64_t)L[j].m * L[j].d_in * (L[j].x_dtype == AGZO_BF16 ? 2 : 4);
      if (j > i && (used + need > scratch_cap || xbytes + xb > wave_bytes)) break;
      if (used + need > scratch_cap && glen > 1) {   // the group alone does not fit: fall back to single layers
        glen = 1;
        ranks = L[j].r;
        fused = false;
        need = unit_need();
      }
      if (used + need > scratch_cap) return AGZO_ERR_WORKSPACE;
      // carve
      size_t need_y = 0;
      for (int g = 0; g < glen; ++g) need_y += align_up((size_t)L[j + g].r * (size_t)L[j + g].d_in * 4);
      if (ws) {
        char* p = ws + base + (size_t)region * scratch_cap + (used - used_y);
        float* ypart = reinterpret_cast<float*>(p);
        p += ypart_bytes(parts_of(L[j], tc, fused, ranks), ranks, L[j].d_in);
        int off = 0;
        for (int g = 0; g < glen; ++g) {
          DevLayer& D = plan->dev[j + g];
          const agzo_layer& a = L[j + g];
          slabs_of(a, tc, false, &D.slabs, &D.slab_rows);
          D.cc_slabs = D.slabs;
          if (!tc && plan->split) slabs_of(a, tc, true, &D.slabs, &D.slab_rows);
          D.gchunks = (a.d_in + 127) / 128;
          D.Ypart = ypart + (size_t)off * a.d_in;
          D.ypart_stride = (long long)ranks * a.d_in;
          off += a.r;
          if (!tc) { D.T = reinterpret_cast<float*>(p); p += align_up((size_t)a.m * a.r * 4); }
          D.Gpart = reinterpret_cast<double*>(p); p += align_up(panel_gram_bytes(a.d_in, a.r, extract_max_r));
        }
        off = 0;
        for (int g = 0; tc && g < glen; ++g) {
          DevLayer& D = plan->dev[j + g];
          tc_set_panels(L[j + g], &D, p, ranks, off, g == glen - 1);
          off += L[j + g].r;
          D.grp_role = glen == 1 ? 0 : (g == 0 ? 1 : 2);
          D.tmaps = ws + maps_offset(n) + (size_t)(j + g) * kMapBytes;
          // the power steps of this unit run fused (X read once per step) where its shape allows
          const agzo_layer all = with_ranks(L[j], ranks);
          D.fz_C = fused ? fused_cluster_size(opts.fused_caps, all, opts.extract_fused == 2) : 0;
          D.fz_slice = fused ? fused_slice_cols(opts.fused_caps, all, opts.extract_fused == 2) : 0;
        }
      }
      used += need;
      used_y += need_y;
      xbytes += xb;
      j += glen;
    }
    if (used > max_wave_scratch) max_wave_scratch = used;
    {   // the Y panels follow everything else of the wave
      char* y0 = ws ? ws + base + (size_t)region * scratch_cap + (used - used_y) : nullptr;
      char* y = y0;
      for (int k = i; k < j && ws; ++k) {
        plan->dev[k].Y = reinterpret_cast<float*>(y);
        y += align_up((size_t)L[k].r * (size_t)L[k].d_in * 4);
      }
      plan->wave_y.push_back(reinterpret_cast<float*>(y0));
      plan->wave_y_count.push_back(used_y / 4);
    }
    {   // order in which T = X Q takes the wave's layers: largest d_in first (stable)
      std::vector<int> ord(j - i);
      for (int k = 0; k < j - i; ++k) ord[k] = k;
      std::stable_sort(ord.begin(), ord.end(), [&](int a, int b) { return L[i + a].d_in > L[i + b].d_in; });
      for (int k = 0; k < j - i; ++k) plan->dev[i + k].xq_order = ord[k];
    }
    if (ws) {
      // A wave whose activations stay in L2 from one sweep to the next gains nothing from the fused kernel
      // (its point is that X crosses HBM once per power step): such a wave takes the two sweeps throughout.
      if (opts.extract_fused != 2 && xbytes <= kL2ResidentWaveBytes)
        for (int k = i; k < j; ++k) plan->dev[k].fz_C = 0;
      // the fused kernel's launches of this wave, one per cluster size: who works on which tiles
      if (opts.fused_caps)
        for (int C = 1; C <= 16; ++C) fused_plan_shares(*opts.fused_caps, plan->dev.data(), i, j, C);
    }
    plan->wave_end.push_back(j);
    plan->wave_region.push_back(region);
    i = j;
  }
  if (scratch_needed) {
    *scratch_needed = max_wave_scratch * regions + (regions > 1 ? kAlign : 0);
    if (plan->image_bytes > *scratch_needed) *scratch_needed = plan->image_bytes;
  }
  return AGZO_OK;
}

bool same_layers(const agzo_ctx* c, const agzo_layer* L, int n) {
  return c->cached_valid && (int)c->cached.size() == n &&
         (n == 0 || std::memcmp(c->cached.data(), L, (size_t)n * sizeof(agzo_layer)) == 0);
}

DevLayer* dev_layers(agzo_ctx* c) { return reinterpret_cast<DevLayer*>(c->ws + kHeaderBytes); }
int* dev_tiles(agzo_ctx* c, int n) {
  return reinterpret_cast<int*>(c->ws + kHeaderBytes + align_up((size_t)n * sizeof(DevLayer)));
}
int* dev_items(agzo_ctx* c, int n) { return dev_tiles(c, n) + (n + 1); }
DevStatus* dev_status(agzo_ctx* c) { return reinterpret_cast<DevStatus*>(c->ws); }

// Tables of up to 30 KiB (36 layers) travel as the parameters of a kernel that writes them to the workspace: the launch
// takes its copy, so the host neither waits for an earlier upload nor keeps a buffer, and the stream stays a chain of
// kernels.  A forward hook that extracts one group of layers per call uploads once per call; with a pinned buffer the host
// waited there for the previous call's kernels.  The kernels after it read the tables before they wait for their
// predecessor, so this one does not let them start early.
constexpr int kTableThreads = 256, kTableCtas = 8;
template <int BYTES> struct TableBlob { uint4 d[BYTES / 16]; };
template <int BYTES>
__global__ void __launch_bounds__(kTableThreads) table_kernel(const __grid_constant__ TableBlob<BYTES> blob, uint4* dst, int n16) {
  chain_wait();
  for (int i = blockIdx.x * kTableThreads + threadIdx.x; i < n16; i += gridDim.x * kTableThreads) dst[i] = blob.d[i];
}
template <int BYTES>
cudaError_t launch_table(const char* t, size_t bytes, char* dst, cudaStream_t s) {
  TableBlob<BYTES> blob;
  std::memcpy(&blob, t, bytes);
  const int n16 = (int)(bytes / 16), ctas = std::min(kTableCtas, (n16 + kTableThreads - 1) / kTableThreads);
  return launch_chained(table_kernel<BYTES>, dim3((unsigned)ctas), kTableThreads, 0, 0, s, blob, reinterpret_cast<uint4*>(dst), n16);
}
constexpr size_t kTableParamBytes = 30 * 1024;
cudaError_t upload_as_parameters(const std::vector<char>& t, char* dst, cudaStream_t s) {
  if (t.size() <= 3 * 1024) return launch_table<3 * 1024>(t.data(), t.size(), dst, s);
  if (t.size() <= 10 * 1024) return launch_table<10 * 1024>(t.data(), t.size(), dst, s);
  for (size_t at = 0; at < t.size(); at += kTableParamBytes) {
    const cudaError_t e = launch_table<(int)kTableParamBytes>(t.data() + at, std::min(kTableParamBytes, t.size() - at), dst + at, s);
    if (e != cudaSuccess) return e;
  }
  return cudaSuccess;
}

// A number of the capture that the stream takes part in, 0 outside of any
unsigned long long capture_of(cudaStream_t s) {
  cudaStreamCaptureStatus st = cudaStreamCaptureStatusNone;
  unsigned long long id = 0;
  if (cudaStreamGetCaptureInfo(s, &st, &id) != cudaSuccess) { cudaGetLastError(); return 0; }
  return st == cudaStreamCaptureStatusActive ? id : 0;
}

PlanOpts plan_opts(const agzo_ctx* c, int regions) {
  return PlanOpts{c->wave_bytes, c->extract_path, c->rmw_path, c->rmw_tc_min_rank, c->rmw_tc_panels, c->rmw_stage_r,
                  c->tc.available, c->extract_fused, c->share_inputs != 0, regions, c->extract_path == 0 ? c->extract_split : 0, c->sm_count, &c->tc.fused};
}

bool any_weights(const agzo_layer* L, int n) {
  for (int i = 0; i < n; ++i)
    if (L[i].W) return true;
  return false;
}

// Makes the device tables describe `L`; uploads only when the descriptors changed.  An upload that is captured is a node of the
// graph: the tables are in place for the rest of that capture and for nobody else.
agzo_status prepare(agzo_ctx* c, const agzo_layer* L, int n, cudaStream_t s) {
  if (!c->tables_captured && !any_weights(L, n)) c->tables_captured = capture_of(s) != 0;
  if (same_layers(c, L, n) && (c->tables_capture == 0 || c->tables_capture == capture_of(s))) {
    // the tables were uploaded on another stream: this one must not read them before they have landed
    if (c->stage_pending && s != c->stage_stream) CU(c, cudaStreamWaitEvent(s, c->stage_ev, 0));
    return AGZO_OK;
  }
  c->rimg_valid = false;
  if (kHeaderBytes + table_bytes(n) > c->ws_bytes) return AGZO_ERR_WORKSPACE;
  Plan plan;
  PlanOpts opts = plan_opts(c, c->allreduce ? 1 : c->extract_streams);    // the ranks' sums run in wave order on the caller's stream
  agzo_status st = build_plan(L, n, c->ws, c->ws_bytes, opts, &plan, nullptr);
  if (st == AGZO_ERR_WORKSPACE && opts.extract_regions == 2) {   // a workspace sized for one region
    opts.extract_regions = 1;
    st = build_plan(L, n, c->ws, c->ws_bytes, opts, &plan, nullptr);
  }
  if (st != AGZO_OK) return st;
  const size_t lb = align_up((size_t)n * sizeof(DevLayer));
  const size_t tb = prefix_bytes(n) + (size_t)n * kMapBytes;
  if (n > 0) {
    c->h_tables.assign(lb + tb, 0);      // both multiples of 16
    char* hs = c->h_tables.data();
    std::memcpy(hs, plan.dev.data(), (size_t)n * sizeof(DevLayer));
    std::memcpy(hs + lb, plan.tile_start.data(), (size_t)(n + 1) * sizeof(int));
    std::memcpy(hs + lb + (size_t)(n + 1) * sizeof(int), plan.item_start.data(), (size_t)(n + 1) * sizeof(int));
    char* hmaps = hs + lb + prefix_bytes(n);
    for (int i = 0; i < n; ++i) {
      if (plan.dev[i].Qb && plan.dev[i].grp_role != 2 &&
          !tc_encode_maps(c->tc, plan.dev[i], hmaps + (size_t)i * kMapBytes))
        return AGZO_ERR_UNSUPPORTED;
      if (plan.dev[i].wmap && !rmw_tc_encode_map(c->tc, plan.dev[i], hmaps + (size_t)i * kMapBytes + 384))
        return AGZO_ERR_UNSUPPORTED;
    }
    c->cached_valid = false;             // until the upload is on its way
    const unsigned long long capture = capture_of(s);
    if (lb + tb <= kTableParamBytes || capture != 0) {       // a copy that is captured would find the pinned buffer rewritten
      c->launches += (int64_t)((lb + tb + kTableParamBytes - 1) / kTableParamBytes);
      CU(c, upload_as_parameters(c->h_tables, c->ws + kHeaderBytes, s));
    } else {
      if (c->h_stage_busy) CU(c, cudaEventSynchronize(c->stage_ev));
      c->h_stage_busy = false;
      if (lb + tb > c->h_stage_bytes) {
        if (c->h_stage) CU(c, cudaFreeHost(c->h_stage));
        c->h_stage = nullptr;
        c->h_stage_bytes = 0;
        CU(c, cudaMallocHost(&c->h_stage, (lb + tb) * 2));
        c->h_stage_bytes = (lb + tb) * 2;
      }
      std::memcpy(c->h_stage, hs, lb + tb);
      CU(c, cudaMemcpyAsync(c->ws + kHeaderBytes, c->h_stage, lb + tb, cudaMemcpyHostToDevice, s));
      c->h_stage_busy = true;
    }
    c->tables_capture = capture;
    c->stage_pending = capture == 0;     // inside a capture the graph's edges order it
    if (c->stage_pending) CU(c, cudaEventRecord(c->stage_ev, s));
    c->stage_stream = s;
  }
  c->plan = std::move(plan);
  c->cached.assign(L, L + n);
  c->cached_valid = true;
  return AGZO_OK;
}

// Whether the resident kernel extracts this list: c->resident is its launch then.  It takes part of the scratch area, at its
// end, and leaves the tables of the list that was prepared last alone.  prepared: the tables are this list's.  What a list that goes to
// the other kernels pays for the question is the layouts (1 us on the host); whether those would take the list, half a microsecond more
// that their own planning repeats, is asked last.
bool plan_resident(agzo_ctx* c, const agzo_layer* L, int n, int K, bool prepared) {
  // an option that asks for one of the other paths, cuts the list into waves or times their kernels is meant for those
  const bool times_others = c->time_class != AGZO_KC_NONE && c->time_class != AGZO_KC_RMW && c->time_class != AGZO_KC_RMW_TC &&
                            c->time_class != AGZO_KC_RESIDENT;
  if (times_others || !c->extract_resident || c->allreduce || c->extract_path != 0 || c->extract_fused != 1 || c->wave_bytes != kDefaultWaveBytes) return false;
  if (!c->resident_known || c->resident_cached.size() != (size_t)n ||
      std::memcmp(c->resident_cached.data(), L, (size_t)n * sizeof(agzo_layer)) != 0) {
    bool two_parts = c->tc.available;
    for (int i = 0; i < n && two_parts; ++i) two_parts = tc_eligible(L[i]);
    c->resident_ok = resident_plan(c->resident_caps, L, n, c->share_inputs != 0, two_parts, &c->resident);
    c->resident_admitted = -1;
    c->resident_cached.assign(L, L + n);
    c->resident_known = true;
  }
  if (!c->resident_ok || (c->extract_resident != 2 && !resident_pays(c->resident, K, !any_weights(L, n)))) return false;
  // a workspace that the other kernels would refuse is refused by all
  if (c->resident_admitted < 0) {
    Plan others;
    c->resident_admitted = prepared || (kHeaderBytes + table_bytes(n) <= c->ws_bytes &&
                                        build_plan(L, n, c->ws, c->ws_bytes, plan_opts(c, 1), &others, nullptr) == AGZO_OK);
  }
  if (!c->resident_admitted) return false;
  const size_t tables = kHeaderBytes + (c->cached_valid ? table_bytes((int)c->cached.size()) : 0);
  const size_t end = c->ws_bytes & ~(kAlign - 1), need = align_up(c->resident.scratch);
  if (end < tables || end - tables < need) return false;
  resident_bind(&c->resident, c->ws + end - need);
  return true;
}

agzo_status check_ctx(agzo_ctx* c) {
  if (!c || c->magic != kMagic) return AGZO_ERR_STATE;
  int dev = -1;
  if (cudaGetDevice(&dev) != cudaSuccess || dev != c->device) {
    if (cudaSetDevice(c->device) != cudaSuccess) return AGZO_ERR_CUDA;
  }
  return AGZO_OK;
}

agzo_status rmw_pass(agzo_ctx* c, const agzo_layer* L, int n, uint64_t seed, PassCoef coef,
                     bool pair_update, cudaStream_t s) {
  agzo_status st = validate(L, n, NEED_RMW);
  if (st != AGZO_OK) return st;
  if (n == 0) return AGZO_OK;
  st = prepare(c, L, n, s);
  if (st != AGZO_OK) return st;
  if (c->plan.total_items > 0) {
    // the passes of one step share the seed, hence R: the images a pass staged serve the next ones
    const bool fill = c->plan.staged_r && !(c->rimg_valid && c->rimg_seed == seed && c->rimg_stream == s);
    c->rimg_valid = false;
    Timed t(c, AGZO_KC_RMW_TC, s, fill ? 2 : 1);
    CU(c, launch_rmw_tc(dev_layers(c), dev_items(c, n), n, c->plan.total_items, c->plan.max_rp, c->plan.max_r,
                        c->plan.max_b_bytes, c->plan.max_row_tiles, c->plan.staged_r, fill, c->rmw_tc_slots,
                        c->rmw_tc_inflight, seed, coef, dev_status(c), c->sm_count, s));
    if (c->plan.staged_r) { c->rimg_valid = true; c->rimg_seed = seed; c->rimg_stream = s; }
  }
  if (c->plan.total_tiles > 0) {
    Timed t(c, AGZO_KC_RMW, s);
    CU(c, launch_rmw(dev_layers(c), dev_tiles(c, n), n, c->plan.total_tiles, c->plan.tile_rows, c->plan.slow_rows, c->plan.cc_max_r,
                     c->plan.fast_mode_mask, c->plan.any_slow, seed, coef, pair_update, c->sm_count, s));
  }
  return AGZO_OK;
}

}  // namespace

namespace agzo {

unsigned long long current_context_id(int device) {
  typedef CUresult (*GetIdFn)(CUcontext, unsigned long long*);
  static const GetIdFn get_id = [] {
    void* fn = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPoint("cuCtxGetId", &fn, cudaEnableDefault, &q) != cudaSuccess || q != cudaDriverEntryPointSuccess) {
      cudaGetLastError();
      fn = nullptr;
    }
    return reinterpret_cast<GetIdFn>(fn);
  }();
  unsigned long long id = 0;
  if (!get_id) return 0;
  if (get_id(nullptr, &id) == CUDA_SUCCESS) return id;
  // no context on this thread yet (or one that a reset has ended): the device's primary one
  if (cudaSetDevice(device) != cudaSuccess || get_id(nullptr, &id) != CUDA_SUCCESS) return 0;
  return id;
}

}  // namespace agzo

// =================================================================== C ABI
extern "C" {

const char* agzo_status_string(agzo_status s) {
  switch (s) {
    case AGZO_OK: return "ok";
    case AGZO_ERR_INVALID_ARG: return "invalid argument";
    case AGZO_ERR_UNSUPPORTED: return "unsupported dtype or mode";
    case AGZO_ERR_CUDA: return "CUDA runtime error";
    case AGZO_ERR_WORKSPACE: return "workspace missing, misaligned or too small";
    case AGZO_ERR_STATE: return "invalid context";
    case AGZO_ERR_TIMEOUT: return "device-side wait ran out";
    case AGZO_ERR_CALLBACK: return "callback failed (loss or all-reduce)";
    case AGZO_WARN_RANK_DEFICIENT: return "rank-deficient activation panel";
  }
  return "unknown status";
}

int agzo_last_cuda_error(const agzo_ctx* ctx) { return ctx ? ctx->last_cuda : 0; }

agzo_status agzo_workspace_bytes(const agzo_layer* h_layers, int n, size_t* h_bytes) {
  if (!h_bytes) return AGZO_ERR_INVALID_ARG;
  agzo_status st = validate(h_layers, n, 0);
  if (st != AGZO_OK) return st;
  // large enough for either kind of extraction kernel (the "extract_path" option may pick
  // the CUDA-core kernels, whose slabs are shaped differently)
  Plan plan;
  size_t scratch = 0, scratch_cc = 0;
  st = build_plan(h_layers, n, nullptr, 0, PlanOpts{kDefaultWaveBytes, 0, 0, 3, 0, 0, true, 0, false, 2, 0, 148, nullptr}, &plan, &scratch);
  if (st != AGZO_OK) return st;
  st = build_plan(h_layers, n, nullptr, 0, PlanOpts{kDefaultWaveBytes, 1, 1, 0, 1, 1, false, 0, false, 2, 0, 148, nullptr}, &plan, &scratch_cc);
  if (st != AGZO_OK) return st;
  if (scratch_cc > scratch) scratch = scratch_cc;
  // ... and for the fused power step, whose layers keep room for one partial sum of Y per share of a launch
  st = build_plan(h_layers, n, nullptr, 0, PlanOpts{kDefaultWaveBytes, 0, 0, 3, 0, 0, true, 2, false, 2, 0, 148, nullptr}, &plan, &scratch_cc);
  if (st != AGZO_OK) return st;
  if (scratch_cc > scratch) scratch = scratch_cc;
  *h_bytes = kHeaderBytes + table_bytes(n) + scratch + kAlign;
  return AGZO_OK;
}

agzo_status agzo_create(agzo_ctx** out, int device, void* workspace, size_t workspace_bytes) {
  if (!out) return AGZO_ERR_INVALID_ARG;
  *out = nullptr;
  if (!workspace || (reinterpret_cast<uintptr_t>(workspace) & (kAlign - 1)) ||
      workspace_bytes < kHeaderBytes)
    return AGZO_ERR_WORKSPACE;
  int count = 0;
  if (cudaGetDeviceCount(&count) != cudaSuccess || device < 0 || device >= count)
    return AGZO_ERR_CUDA;
  agzo_ctx* c = new (std::nothrow) agzo_ctx();
  if (!c) return AGZO_ERR_INVALID_ARG;
  c->magic = kMagic;
  c->device = device;
  c->ws = static_cast<char*>(workspace);
  c->ws_bytes = workspace_bytes;
  c->last_cuda = 0;
  c->extract_path = 0;
  c->rmw_path = 0;
  c->rmw_tc_min_rank = 0;   // kRmwTcMinRank: 8B shapes, six blocks, one pass, CUDA cores / tensor cores: r = 1 736 / 786 us, r = 4 732 / 783,
                            // r = 6 822 / 780, r = 8 823 / 783, r = 16 1471 / 770; 0.6B shapes r = 4 282 / 302, r = 6 331 / 316
  c->rmw_tc_slots = 0;
  c->rmw_tc_inflight = 0;
  c->rmw_tc_panels = 0;
  c->rmw_stage_r = 0;
  c->wave_bytes = kDefaultWaveBytes;
  c->extract_streams = 2;
  c->extract_fused = 1;
  c->allreduce = nullptr;
  c->rimg_valid = false;
  c->rimg_seed = 0;
  c->rimg_stream = nullptr;
  c->stage_stream = nullptr;
  c->allreduce_user = nullptr;
  c->token_offset = 0;
  c->share_inputs = 1;
  c->extract_resident = 1;
  c->extract_split = 1;
  c->resident_known = c->resident_ok = false;
  c->resident_admitted = -1;
  c->aux[0] = c->aux[1] = nullptr;
  c->fork_ev = c->join_ev[0] = c->join_ev[1] = nullptr;
  c->cached_valid = false;
  c->tables_capture = 0;
  c->tables_captured = false;
  c->h_stage = nullptr;
  c->h_stage_bytes = 0;
  c->h_stage_busy = false;
  c->stage_pending = false;
  c->stage_ev = nullptr;
  c->time_class = 0;
  c->debug_fail_step_call = 0;
  c->debug_missing_class = 0;
  c->debug_refuse_resident = 0;
  c->events_used = 0;
  c->launches = 0;
  c->power_steps = 0;
  cudaError_t e = cudaSetDevice(device);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&c->sm_count, cudaDevAttrMultiProcessorCount, device);
  if (e == cudaSuccess) e = cudaEventCreateWithFlags(&c->stage_ev, cudaEventDisableTiming);
  for (int k = 0; k < 2 && e == cudaSuccess; ++k) {
    e = cudaStreamCreateWithFlags(&c->aux[k], cudaStreamNonBlocking);
    if (e == cudaSuccess) e = cudaEventCreateWithFlags(&c->join_ev[k], cudaEventDisableTiming);
  }
  if (e == cudaSuccess) e = cudaEventCreateWithFlags(&c->fork_ev, cudaEventDisableTiming);
  if (e == cudaSuccess) e = cudaMemset(c->ws, 0, kHeaderBytes);
  if (e == cudaSuccess) e = cudaDeviceSynchronize();
  if (e == cudaSuccess) e = device_init(device, &c->tc, &c->resident_caps);
  if (e != cudaSuccess) {
    if (c->stage_ev) cudaEventDestroy(c->stage_ev);
    if (c->fork_ev) cudaEventDestroy(c->fork_ev);
    for (int k = 0; k < 2; ++k) {
      if (c->join_ev[k]) cudaEventDestroy(c->join_ev[k]);
      if (c->aux[k]) cudaStreamDestroy(c->aux[k]);
    }
    delete c;
    return AGZO_ERR_CUDA;
  }
  *out = c;
  return AGZO_OK;
}

agzo_status agzo_destroy(agzo_ctx* ctx) {
  if (!ctx || ctx->magic != kMagic) return AGZO_ERR_STATE;
  if (ctx->stage_pending) cudaEventSynchronize(ctx->stage_ev);
  if (ctx->h_stage) cudaFreeHost(ctx->h_stage);
  if (ctx->stage_ev) cudaEventDestroy(ctx->stage_ev);
  if (ctx->fork_ev) cudaEventDestroy(ctx->fork_ev);
  for (int k = 0; k < 2; ++k) {
    if (ctx->aux[k]) cudaStreamSynchronize(ctx->aux[k]);
    if (ctx->join_ev[k]) cudaEventDestroy(ctx->join_ev[k]);
    if (ctx->aux[k]) cudaStreamDestroy(ctx->aux[k]);
  }
  for (cudaEvent_t e : ctx->events) cudaEventDestroy(e);
  ctx->magic = 0;
  delete ctx;
  return AGZO_OK;
}

agzo_status agzo_set_option(agzo_ctx* ctx, const char* name, int64_t value) {
  if (!ctx || ctx->magic != kMagic) return AGZO_ERR_STATE;
  if (!name) return AGZO_ERR_INVALID_ARG;
  if (std::strcmp(name, "extract_path") == 0) {
    if (value < 0 || value > 3) return AGZO_ERR_INVALID_ARG;
    ctx->extract_path = (int)value;
  } else if (std::strcmp(name, "rmw_path") == 0) {
    if (value < 0 || value > 2) return AGZO_ERR_INVALID_ARG;
    ctx->rmw_path = (int)value;
  } else if (std::strcmp(name, "rmw_tc_min_rank") == 0) {
    if (value < 1 || value > AGZO_MAX_RANK) return AGZO_ERR_INVALID_ARG;
    ctx->rmw_tc_min_rank = (int)value;
  } else if (std::strcmp(name, "rmw_tc_inflight") == 0) {
    if (value < 0 || value > 64) return AGZO_ERR_INVALID_ARG;
    ctx->rmw_tc_inflight = (int)value;
    return AGZO_OK;
  } else if (std::strcmp(name, "rmw_stage_r") == 0) {
    if (value < 0 || value > 2) return AGZO_ERR_INVALID_ARG;
    ctx->rmw_stage_r = (int)value;
  } else if (std::strcmp(name, "rmw_tc_panels") == 0) {
    if (value < 0 || value > 2) return AGZO_ERR_INVALID_ARG;
    ctx->rmw_tc_panels = (int)value;
  } else if (std::strcmp(name, "rmw_tc_slots") == 0) {
    if (value < 0 || value > 64) return AGZO_ERR_INVALID_ARG;
    ctx->rmw_tc_slots = (int)value;
    return AGZO_OK;
  } else if (std::strcmp(name, "share_inputs") == 0) {
    if (value < 0 || value > 1) return AGZO_ERR_INVALID_ARG;
    ctx->share_inputs = (int)value;
  } else if (std::strcmp(name, "extract_resident") == 0) {
    if (value < 0 || value > 2) return AGZO_ERR_INVALID_ARG;
    ctx->extract_resident = (int)value;
    return AGZO_OK;
  } else if (std::strcmp(name, "extract_split") == 0) {
    if (value < 0 || value > 2) return AGZO_ERR_INVALID_ARG;
    ctx->extract_split = (int)value;
  } else if (std::strcmp(name, "extract_fused") == 0) {
    if (value < 0 || value > 2) return AGZO_ERR_INVALID_ARG;
    ctx->extract_fused = (int)value;
  } else if (std::strcmp(name, "extract_streams") == 0) {
    if (value < 1 || value > 2) return AGZO_ERR_INVALID_ARG;
    ctx->extract_streams = (int)value;
  } else if (std::strcmp(name, "wave_bytes") == 0) {
    if (value < 0) return AGZO_ERR_INVALID_ARG;
    ctx->wave_bytes = value;
  } else if (std::strcmp(name, "debug_fail_step_call") == 0) {
    if (value < 0 || value > 16) return AGZO_ERR_INVALID_ARG;
    ctx->debug_fail_step_call = (int)value;
    return AGZO_OK;
  } else if (std::strcmp(name, "debug_missing_class") == 0) {
    if (value != 0 && value != AGZO_KC_XT_T && value != AGZO_KC_X_Q && value != AGZO_KC_PANEL_QR) return AGZO_ERR_INVALID_ARG;
    ctx->debug_missing_class = (int)value;
    return AGZO_OK;
  } else if (std::strcmp(name, "debug_refuse_resident") == 0) {
    if (value < 0 || value > 1) return AGZO_ERR_INVALID_ARG;
    ctx->debug_refuse_resident = (int)value;
    return AGZO_OK;
  } else if (std::strcmp(name, "time_kernel_class") == 0) {
    if (value < 0 || value > AGZO_KC_RESIDENT) return AGZO_ERR_INVALID_ARG;
    ctx->time_class = (int)value;
    return AGZO_OK;
  } else {
    return AGZO_ERR_INVALID_ARG;
  }
  ctx->cached_valid = ctx->resident_known = false;   // the plans depend on the options
  return AGZO_OK;
}

agzo_status agzo_set_allreduce(agzo_ctx* ctx, agzo_allreduce_fn fn, void* user, int64_t token_offset) {
  if (!ctx || ctx->magic != kMagic) return AGZO_ERR_STATE;
  if (token_offset < 0 || (!fn && token_offset != 0)) return AGZO_ERR_INVALID_ARG;
  ctx->allreduce = fn;
  ctx->allreduce_user = user;
  ctx->token_offset = token_offset;
  ctx->cached_valid = false;   // the number of scratch regions depends on it
  return AGZO_OK;
}

agzo_status agzo_read_counters(agzo_ctx* ctx, double* h_ms, int64_t* h_timed, int64_t* h_total) {
  agzo_status st = check_ctx(ctx);
  if (st != AGZO_OK) return st;
  double ms = 0.0;
  for (size_t i = 0; i + 1 < ctx->events_used; i += 2) {
    CU(ctx, cudaEventSynchronize(ctx->events[i + 1]));
    float t = 0.f;
    CU(ctx, cudaEventElapsedTime(&t, ctx->events[i], ctx->events[i + 1]));
    ms += (double)t;
  }
  if (h_ms) *h_ms = ms;
  if (h_timed) *h_timed = (int64_t)(ctx->events_used / 2);
  if (h_total) *h_total = ctx->launches;
  ctx->events_used = 0;
  ctx->launches = 0;
  return AGZO_OK;
}

agzo_status agzo_query_cluster_capacity(agzo_ctx* ctx, int32_t* h_clusters) {
  agzo_status st = check_ctx(ctx);
  if (st != AGZO_OK) return st;
  if (!h_clusters) return AGZO_ERR_INVALID_ARG;
  for (int C = 0; C <= 16; ++C) h_clusters[C] = ctx->tc.available ? fused_resident_clusters(ctx->tc.fused, C) : 0;
  return AGZO_OK;
}

agzo_status agzo_query_fused(agzo_ctx* ctx, const agzo_layer* h_layers, int n, int32_t* h_cluster, void* stream) {
  agzo_status st = check_ctx(ctx);
  if (st != AGZO_OK) return st;
  if (!h_cluster || n < 0) return AGZO_ERR_INVALID_ARG;
  st = validate(h_layers, n, 0);
  if (st != AGZO_OK) return st;
  if (n == 0) return AGZO_OK;
  st = prepare(ctx, h_layers, n, static_cast<cudaStream_t>(stream));
  if (st != AGZO_OK) return st;
  for (int i = 0; i < n; ++i) h_cluster[i] = ctx->plan.dev[i].fz_C;
  return AGZO_OK;
}

agzo_status agzo_query_resident(agzo_ctx* ctx, const agzo_layer* h_layers, int n, int K, int32_t* h_units, int32_t* h_count) {
  agzo_status st = check_ctx(ctx);
  if (st != AGZO_OK) return st;
  if (!h_units || !h_count || K < 0 || K > 16) return AGZO_ERR_INVALID_ARG;
  st = validate(h_layers, n, NEED_EXTRACT);
  if (st != AGZO_OK) return st;
  *h_count = 0;
  if (n == 0 || !plan_resident(ctx, h_layers, n, K, false)) return AGZO_OK;
  const ResidentLaunch& r = ctx->resident;
  for (int k = 0; k < r.p.n_units; ++k) {
    const ResidentUnit& u = r.p.unit[k];
    const int32_t v[8] = {r.p.cs, u.cj, u.cb, u.tb, u.ni, u.clusters, u.sub, r.parts};
    std::memcpy(h_units + 8 * k, v, sizeof(v));
  }
  *h_count = r.p.n_units;
  return AGZO_OK;
}

agzo_status agzo_poll(agzo_ctx* ctx, void* stream) {
  agzo_status st = check_ctx(ctx);
  if (st != AGZO_OK) return st;
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  DevStatus h{};
  CU(ctx, cudaMemcpyAsync(&h, dev_status(ctx), sizeof(h), cudaMemcpyDeviceToHost, s));
  CU(ctx, cudaMemsetAsync(dev_status(ctx), 0, sizeof(DevStatus), s));
  CU(ctx, cudaStreamSynchronize(s));
  if (h.timeout) return AGZO_ERR_TIMEOUT;
  if (h.rank_deficient) return AGZO_WARN_RANK_DEFICIENT;
  return AGZO_OK;
}

agzo_status agzo_extract_subspace(agzo_ctx* ctx, const agzo_layer* h_layers, int n, uint64_t seed,
                                  int K, void* stream) {
  agzo_status st = check_ctx(ctx);
  if (st != AGZO_OK) return st;
  if (K < 0 || K > 16) return AGZO_ERR_INVALID_ARG;
  st = validate(h_layers, n, NEED_EXTRACT);
  if (st != AGZO_OK) return st;
  if (n == 0) return AGZO_OK;
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  if (ctx->extract_path >= 2)
    for (int i = 0; i < n; ++i)
      if (!ctx->tc.available || !tc_eligible(h_layers[i])) return AGZO_ERR_UNSUPPORTED;
  // A list with weights gets its tables here, whichever kernels extract it: the passes read them.  One without gets them where it
  // takes the other kernels; but once calls that read such a list's tables have been captured, every use of the list outside the
  // capture leaves them in place for the graph.
  const bool tables = any_weights(h_layers, n) || (ctx->tables_captured && capture_of(s) == 0);
  if (tables && (st = prepare(ctx, h_layers, n, s)) != AGZO_OK) return st;
  if (plan_resident(ctx, h_layers, n, K, tables)) {
    // it reads no tables, so an upload that another stream has under way is not waited for (a capturing stream could not)
    ctx->rimg_valid = false;
    ResidentParams& p = ctx->resident.p;
    p.K = K;
    p.seed = seed;
    p.status = dev_status(ctx);
    p.flag = nullptr;
    p.counters = reinterpret_cast<unsigned long long*>(ctx->ws + kCountersAt);
    cudaError_t e;
    {
      Timed t(ctx, AGZO_KC_RESIDENT, s);
      e = ctx->debug_refuse_resident ? cudaErrorCooperativeLaunchTooLarge : launch_resident(ctx->resident, s);
    }
    if (e == cudaSuccess) return AGZO_OK;
    ctx->launches -= 1;      // refused: not a launch, and no time of one
    if (ctx->time_class == AGZO_KC_RESIDENT && ctx->events_used >= 2) ctx->events_used -= 2;
    ctx->resident_ok = false;
    if (!resident_refused(e)) { ctx->last_cuda = (int)e; return AGZO_ERR_CUDA; }
  }
  if (!tables && (st = prepare(ctx, h_layers, n, s)) != AGZO_OK) return st;
  ctx->rimg_valid = false;   // extraction takes the scratch area

  const Plan& P = ctx->plan;
  // With two scratch regions, alternate waves run on two helper streams forked from the
  // caller's stream: the short, latency-bound kernels of one wave (panel QR) overlap the
  // other wave's sweeps over X.  Everything is joined back before the call returns.
  int n_real = 0;
  for (int rg : P.wave_region) n_real += rg >= 0;
  const bool forked = P.regions == 2 && n_real >= 2;
  if (forked) {
    CU(ctx, cudaEventRecord(ctx->fork_ev, s));
    for (int k = 0; k < 2; ++k) CU(ctx, cudaStreamWaitEvent(ctx->aux[k], ctx->fork_ev, 0));
  }
  auto run_waves = [&]() -> agzo_status {
    int l0 = 0;
    for (size_t wv = 0; wv < P.wave_end.size(); ++wv) {
      const int l1 = P.wave_end[wv];
      ExtractWave w{};
      w.d_layers = dev_layers(ctx);
      w.l0 = l0; w.l1 = l1;
      w.omega_row0 = ctx->allreduce ? ctx->token_offset : 0;
      w.y_reduced = ctx->allreduce ? 1 : 0;
      w.qr_wide = ctx->tc.qr_wide ? 1 : 0;
      w.sm_count = ctx->sm_count;
      w.region = P.wave_region[wv] == 1 ? 1 : 0;
      bool all_tc = ctx->extract_path != 1;
      for (int i = l0; i < l1; ++i) {
        const DevLayer& D = P.dev[i];
        if (D.m > w.max_m) w.max_m = D.m;
        if (D.d_in > w.max_din) w.max_din = D.d_in;
        if (D.r > w.max_r) w.max_r = D.r;
        if (D.slabs > w.max_slabs) w.max_slabs = D.slabs;
        if (D.gchunks > w.max_gchunks) w.max_gchunks = D.gchunks;
        if (!D.Qb) all_tc = false;
      }
      l0 = l1;
      if (w.max_m == 0 || P.wave_region[wv] < 0) continue;
      cudaStream_t ws = forked ? ctx->aux[P.wave_region[wv]] : s;
      DevStatus* dst = dev_status(ctx);
      auto panel_qr = [&](bool last) -> cudaError_t {
        Timed t(ctx, AGZO_KC_PANEL_QR, ws, panel_qr_launches(w.max_r));
        w.missing = ctx->debug_missing_class == AGZO_KC_PANEL_QR;
        return launch_panel_qr(w, last, dst, ws);
      };
      // token-sharded run: Y = sum over ranks of X_p^T T_p, all panels of the wave in one call
      auto sum_over_ranks = [&]() -> agzo_status {
        if (!ctx->allreduce) return AGZO_OK;
        {
          Timed t(ctx, AGZO_KC_PANEL_QR, ws);
          CU(ctx, launch_sum_slabs(w, ws));
        }
        if (ctx->allreduce(ctx->allreduce_user, ws, P.wave_y[wv], P.wave_y_count[wv]) != 0) return AGZO_ERR_CALLBACK;
        return AGZO_OK;
      };
      // products of this wave in parts: layers of one dtype, and for fp32 a power step (see split_takes)
      const bool split = !all_tc && P.split && split_takes(w, P.dev.data(), K);
      if (!all_tc && !split) {
        w.after_fused = 2;
        w.max_slabs = 0;
        for (int i = w.l0; i < w.l1; ++i) w.max_slabs = std::max(w.max_slabs, P.dev[i].cc_slabs);
      }
      auto omega = [&]() -> cudaError_t {
        Timed t(ctx, AGZO_KC_OMEGA, ws);
        return all_tc ? tc_fill_omega(ctx->tc, w, P.dev.data(), seed, dst, ws) : launch_fill_omega(w, seed, dst, ws);
      };
      // layers served by the fused power-step kernel, by cluster size; the rest take T = X Q, Y = X^T T
      unsigned fz_classes = 0;
      bool any_unfused = false;
      for (int i = w.l0; i < w.l1; ++i) {
        if (all_tc && P.dev[i].fz_C) fz_classes |= 1u << P.dev[i].fz_C; else any_unfused = true;
      }
      auto xt_t = [&](bool skip_fused) -> cudaError_t {       // Y <- H T
        Timed t(ctx, all_tc ? AGZO_KC_TC_XT_T : AGZO_KC_XT_T, ws);
        w.missing = ctx->debug_missing_class == AGZO_KC_XT_T;
        if (split) return launch_split_xt_t(w, P.dev.data(), ctx->share_inputs != 0, dst, ws);
        return all_tc ? tc_xt_t(ctx->tc, w, P.dev.data(), dst, skip_fused, ws) : launch_xt_t(w, ws);
      };
      auto x_q = [&]() -> cudaError_t {        // T <- H^T Q
        Timed t(ctx, all_tc ? AGZO_KC_TC_X_Q : AGZO_KC_X_Q, ws);
        w.missing = ctx->debug_missing_class == AGZO_KC_X_Q;
        if (split) return launch_split_x_q(w, P.dev.data(), ctx->share_inputs != 0, dst, ws);
        return all_tc ? tc_x_q(ctx->tc, w, P.dev.data(), dst, true, ws) : launch_x_q(w, ws);
      };
      auto power_fused = [&]() -> cudaError_t {              // Y <- H (H^T Q) in one pass
        // a launch per cluster size, the largest clusters first; they touch different layers and run into one another
        unsigned left = fz_classes;
        const unsigned step = ++ctx->power_steps;
        for (int C = 16; C >= 1; --C) {
          if (!(left & (1u << C))) continue;
          left &= ~(1u << C);
          Timed t(ctx, AGZO_KC_FUSED_POWER, ws);
          const bool follows = (fz_classes >> (C + 1)) != 0;
          cudaError_t e = launch_fused_power_step(ctx->tc.fused, w, P.dev.data(), C, follows, left != 0, step, dst, ws);
          if (e != cudaSuccess) return e;
        }
        return cudaSuccess;
      };
      agzo_status sr;
      CU(ctx, omega());                        // Omega
      CU(ctx, xt_t(false));                    // Y <- H Omega
      for (int k = 0; k < K; ++k) {
        if ((sr = sum_over_ranks()) != AGZO_OK) return sr;
        CU(ctx, panel_qr(false));              // Q <- qr(Y)
        if (fz_classes) {
          CU(ctx, power_fused());
          w.after_fused = 1;                   // their partial sums are now one per share, not one per slab
        }
        if (any_unfused) {
          CU(ctx, x_q());
          CU(ctx, xt_t(true));                 // Y <- H (H^T Q)
        }
      }
      if ((sr = sum_over_ranks()) != AGZO_OK) return sr;
      CU(ctx, panel_qr(true));                 // A <- qr(Y)
    }
    return AGZO_OK;
  };
  st = run_waves();
  if (forked) {   // join also when a launch failed: the caller's stream must not run ahead of the helpers
    for (int k = 0; k < 2; ++k) {
      cudaError_t e = cudaEventRecord(ctx->join_ev[k], ctx->aux[k]);
      if (e == cudaSuccess) e = cudaStreamWaitEvent(s, ctx->join_ev[k], 0);
      if (e != cudaSuccess && st == AGZO_OK) { ctx->last_cuda = (int)e; st = AGZO_ERR_CUDA; }
    }
  }
  return st;
}

agzo_status agzo_perturb(agzo_ctx* ctx, const agzo_layer* h_layers, int n, uint64_t seed,
                         float scale, void* stream) {
  agzo_status st = check_ctx(ctx);
  if (st != AGZO_OK) return st;
  return rmw_pass(ctx, h_layers, n, seed, pass_coef(scale), false, static_cast<cudaStream_t>(stream));
}

agzo_status agzo_restore(agzo_ctx* ctx, const agzo_layer* h_layers, int n, uint64_t seed,
                         float scale, void* stream) {
  agzo_status st = check_ctx(ctx);
  if (st != AGZO_OK) return st;
  // a master/compute pair is restored by rewriting W16 = bf16(W): coefficient 0 on the pair path
  bool any_pair = false, any_plain = false;
  for (int i = 0; h_layers && i < n; ++i) (h_layers[i].W16 ? any_pair : any_plain) = true;
  if (any_pair && any_plain) return AGZO_ERR_UNSUPPORTED;
  const float c = any_pair ? 0.0f : -scale;
  return rmw_pass(ctx, h_layers, n, seed, pass_coef(c), false, static_cast<cudaStream_t>(stream));
}

agzo_status agzo_update(agzo_ctx* ctx, const agzo_layer* h_layers, int n, uint64_t seed, float lr,
                        const float* d_ghat, void* stream) {
  agzo_status st = check_ctx(ctx);
  if (st != AGZO_OK) return st;
  if (!d_ghat) return AGZO_ERR_INVALID_ARG;
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  st = validate(h_layers, n, NEED_RMW);
  if (st != AGZO_OK) return st;
  if (n == 0) return AGZO_OK;
  return rmw_pass(ctx, h_layers, n, seed, pass_coef(d_ghat, 0.f, lr, 2), true, s);
}

agzo_status agzo_ghat(agzo_ctx* ctx, const double* d_f_plus, const double* d_f_other, float eps,
                      int mode, float* d_ghat, void* stream) {
  agzo_status st = check_ctx(ctx);
  if (st != AGZO_OK) return st;
  if (!d_f_plus || !d_f_other || !d_ghat || !(eps > 0.f) || (mode != 0 && mode != 1))
    return AGZO_ERR_INVALID_ARG;
  ctx->launches += 1;
  CU(ctx, launch_ghat(d_f_plus, d_f_other, eps, mode, d_ghat, static_cast<cudaStream_t>(stream)));
  return AGZO_OK;
}

agzo_status agzo_restore_update(agzo_ctx* ctx, const agzo_layer* h_layers, int n, uint64_t seed,
                                float eps, float lr, int mode, const float* d_ghat, void* stream) {
  agzo_status st = check_ctx(ctx);
  if (st != AGZO_OK) return st;
  if (!d_ghat || (mode != 0 && mode != 1)) return AGZO_ERR_INVALID_ARG;
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  st = validate(h_layers, n, NEED_RMW);
  if (st != AGZO_OK) return st;
  if (n == 0) return AGZO_OK;
  bool any_pair = false, any_plain = false;
  for (int i = 0; i < n; ++i) (h_layers[i].W16 ? any_pair : any_plain) = true;
  if (any_pair && any_plain) return AGZO_ERR_UNSUPPORTED;
  // a pair's master was never perturbed: only the update term applies to it
  return rmw_pass(ctx, h_layers, n, seed, pass_coef(d_ghat, eps, lr, any_pair ? 2 : mode), true, s);
}

agzo_status agzo_step(agzo_ctx* ctx, const agzo_layer* h_layers, int n, const agzo_params* p,
                      agzo_loss_fn loss, void* user, double* d_losses2, float* d_ghat,
                      void* stream) {
  agzo_status st = check_ctx(ctx);
  if (st != AGZO_OK) return st;
  if (!p || !loss || !d_losses2 || !d_ghat || !(p->eps > 0.f) || (p->mode != 0 && p->mode != 1) || p->K < 0 ||
      p->K > 16)
    return AGZO_ERR_INVALID_ARG;
  st = validate(h_layers, n, NEED_RMW | NEED_EXTRACT);
  if (st != AGZO_OK) return st;
  bool any_pair = false, any_plain = false;
  for (int i = 0; i < n; ++i) (h_layers[i].W16 ? any_pair : any_plain) = true;
  if (any_pair && any_plain) return AGZO_ERR_UNSUPPORTED;
  double* d_fplus = d_losses2;
  double* d_fother = d_losses2 + 1;
  float* d_g = d_ghat;

  // The library knows where the weights sit at every moment: W0 + outstanding * Delta.  Whatever
  // fails after the first pass -- the callback or one of the library's own calls -- the inverse of
  // the outstanding perturbation is applied before the error is returned.
  float outstanding = 0.f;
  int call = 0;     // internal calls of this step, counted for the host-side fault injection of the tests
  auto injected = [&]() { return ++call == ctx->debug_fail_step_call; };
  auto fail = [&](agzo_status why) {
    if (outstanding != 0.f) agzo_restore(ctx, h_layers, n, p->seed, outstanding, stream);
    return why;
  };

  // step 1: unperturbed forward (fills X), then Algorithm 1 per layer
  if (loss(user, stream, 0, d_fother) != 0) return AGZO_ERR_CALLBACK;
  st = injected() ? AGZO_ERR_CUDA : agzo_extract_subspace(ctx, h_layers, n, p->seed, p->K, stream);
  if (st != AGZO_OK) return st;
  // step 2: W + eps*Delta
  st = injected() ? AGZO_ERR_CUDA : agzo_perturb(ctx, h_layers, n, p->seed, p->eps, stream);
  if (st != AGZO_OK) return st;
  outstanding = p->eps;
  if (loss(user, stream, 1, d_fplus) != 0) return fail(AGZO_ERR_CALLBACK);
  if (p->mode == 0) {
    // a pair is always rebuilt from the untouched master, so its flip is -eps, not -2 eps
    st = injected() ? AGZO_ERR_CUDA
                    : agzo_perturb(ctx, h_layers, n, p->seed, any_pair ? -p->eps : -2.0f * p->eps, stream);
    if (st != AGZO_OK) return fail(st);
    outstanding = -p->eps;
    if (loss(user, stream, 2, d_fother) != 0) return fail(AGZO_ERR_CALLBACK);
  }
  st = injected() ? AGZO_ERR_CUDA : agzo_ghat(ctx, d_fplus, d_fother, p->eps, p->mode, d_g, stream);
  if (st != AGZO_OK) return fail(st);
  // step 3: restore and update in one pass
  st = injected() ? AGZO_ERR_CUDA
                  : agzo_restore_update(ctx, h_layers, n, p->seed, p->eps, p->lr, p->mode, d_g, stream);
  if (st != AGZO_OK) return fail(st);
  return AGZO_OK;
}

agzo_status agzo_fill_gaussian_basis(agzo_ctx* ctx, const agzo_layer* h_layers, int n, uint64_t seed,
                                     void* stream) {
  agzo_status st = check_ctx(ctx);
  if (st != AGZO_OK) return st;
  st = validate(h_layers, n, 0);
  if (st != AGZO_OK) return st;
  if (n == 0) return AGZO_OK;
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  st = prepare(ctx, h_layers, n, s);
  if (st != AGZO_OK) return st;
  int max_elems = 0;
  for (int i = 0; i < n; ++i) max_elems = std::max(max_elems, h_layers[i].r * h_layers[i].d_in);
  ctx->launches += 1;
  CU(ctx, launch_fill_basis(dev_layers(ctx), n, max_elems, seed, s));
  return AGZO_OK;
}

agzo_status agzo_perturb_dense(agzo_ctx* ctx, void* w, int64_t n_elems, int dtype, uint64_t seed,
                               uint32_t layer_id, float scale, const float* d_scale, void* stream) {
  agzo_status st = check_ctx(ctx);
  if (st != AGZO_OK) return st;
  if (n_elems < 0 || (n_elems > 0 && !w)) return AGZO_ERR_INVALID_ARG;
  if (dtype != AGZO_BF16 && dtype != AGZO_F32) return AGZO_ERR_UNSUPPORTED;
  ctx->launches += 1;
  CU(ctx, launch_dense(w, n_elems, dtype, seed, layer_id, scale, d_scale, ctx->sm_count,
                       static_cast<cudaStream_t>(stream)));
  return AGZO_OK;
}

agzo_status agzo_debug_philox(agzo_ctx* ctx, uint64_t seed, uint32_t layer_id, uint32_t tag,
                              uint64_t first, uint64_t n, uint32_t* d_words, void* stream) {
  agzo_status st = check_ctx(ctx);
  if (st != AGZO_OK) return st;
  if (n > 0 && !d_words) return AGZO_ERR_INVALID_ARG;
  CU(ctx, launch_debug_philox(seed, layer_id, tag, first, n, d_words, ctx->sm_count, static_cast<cudaStream_t>(stream)));
  return AGZO_OK;
}

agzo_status agzo_debug_gaussian(agzo_ctx* ctx, uint64_t seed, uint32_t layer_id, uint32_t tag,
                                uint64_t first, uint64_t n, float* d_vals, void* stream) {
  agzo_status st = check_ctx(ctx);
  if (st != AGZO_OK) return st;
  if (n > 0 && !d_vals) return AGZO_ERR_INVALID_ARG;
  CU(ctx, launch_debug_gauss(seed, layer_id, tag, first, n, d_vals, ctx->sm_count, static_cast<cudaStream_t>(stream)));
  return AGZO_OK;
}

agzo_status agzo_debug_normal_parts(agzo_ctx* ctx, uint32_t first, uint32_t n, float* d_parts, void* stream) {
  agzo_status st = check_ctx(ctx);
  if (st != AGZO_OK) return st;
  if ((n > 0 && !d_parts) || !aligned16(d_parts)) return AGZO_ERR_INVALID_ARG;
  if (first > (1u << 24) || n > (1u << 24) - first) return AGZO_ERR_INVALID_ARG;
  CU(ctx, launch_debug_normal_parts(first, n, d_parts, ctx->sm_count, static_cast<cudaStream_t>(stream)));
  return AGZO_OK;
}

agzo_status agzo_debug_early_copy(agzo_ctx* ctx, const void* src, void* dst, uint64_t bytes, void* stream) {
  agzo_status st = check_ctx(ctx);
  if (st != AGZO_OK) return st;
  if (bytes > 0 && (!src || !dst)) return AGZO_ERR_INVALID_ARG;
  if ((bytes & 15u) || !aligned16(src) || !aligned16(dst)) return AGZO_ERR_INVALID_ARG;
  CU(ctx, launch_debug_early_copy(src, dst, bytes / 16, ctx->sm_count, static_cast<cudaStream_t>(stream)));
  return AGZO_OK;
}

agzo_status agzo_debug_fused_split(const int32_t* h_tiles, int n, int clusters, int32_t* h_tile0, int32_t* h_first,
                                   int32_t* h_parts, int32_t* h_share_begin, int32_t* h_shares) {
  if (n < 0 || clusters < 1 || (n > 0 && (!h_tiles || !h_tile0 || !h_first || !h_parts)) || !h_share_begin || !h_shares)
    return AGZO_ERR_INVALID_ARG;
  long long total = 0;
  for (int i = 0; i < n; ++i) {
    if (h_tiles[i] < 0) return AGZO_ERR_INVALID_ARG;
    total += h_tiles[i];
  }
  if (total > (1ll << 30)) return AGZO_ERR_INVALID_ARG;
  int base = 0, rem = 0;
  const int G = fused_split(h_tiles, n, clusters, h_tile0, h_first, h_parts, &base, &rem);
  for (int k = 0; k <= G; ++k) h_share_begin[k] = fused_share_begin(k, base, rem);
  *h_shares = G;
  return AGZO_OK;
}

agzo_status agzo_debug_meeting(int32_t n, int32_t first, uint32_t phase, uint64_t value, uint64_t* h_increment, uint32_t* h_phase,
                               uint32_t* h_failures) {
  if (n < 1 || phase > 1 || !h_increment || !h_phase || !h_failures) return AGZO_ERR_INVALID_ARG;
  *h_increment = meeting_increment(n, first != 0, phase);
  *h_phase = meeting_phase(value);
  *h_failures = meeting_failures(value);
  return AGZO_OK;
}

agzo_status agzo_debug_tile_rows(const agzo_layer* h_layers, int n, int sm_count, int32_t* h_rows) {
  if (sm_count < 1 || !h_rows) return AGZO_ERR_INVALID_ARG;
  agzo_status st = validate(h_layers, n, 0);
  if (st != AGZO_OK) return st;
  Plan plan;
  st = build_plan(h_layers, n, nullptr, 0, PlanOpts{kDefaultWaveBytes, 0, 0, 0, 0, 0, true, 0, false, 2, 0, sm_count, nullptr}, &plan, nullptr);
  if (st != AGZO_OK) return st;
  h_rows[0] = plan.tile_rows;
  h_rows[1] = plan.slow_rows;
  return AGZO_OK;
}

agzo_status agzo_debug_wait_timeout(agzo_ctx* ctx, void* stream) {
  agzo_status st = check_ctx(ctx);
  if (st != AGZO_OK) return st;
  if (!ctx->tc.available) return AGZO_ERR_UNSUPPORTED;
  CU(ctx, launch_debug_wait(dev_status(ctx), static_cast<cudaStream_t>(stream)));
  return AGZO_OK;
}

}  // extern "C"

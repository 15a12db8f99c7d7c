// Products of Algorithm 1 in fp32 precision on the tensor cores: host interface (agzo_extract_split.cu).
#pragma once

#include <vector>

#include "agzo_common.cuh"

namespace agzo {

constexpr int kSplitMaxRanks = 24;       // of a unit: three parts each, 36 sums per thread and half of them
constexpr int kSplitMaxLayers = 4;       // of a unit
// Units of a launch.  The list is a kernel parameter, where every warp finds an item's shapes and pointers without a trip to memory.
constexpr int kSplitFewUnits = 16, kSplitMaxUnits = 150;

struct SplitLayer {
  const float* src;      // T = X Q: V; Y = X^T T: T
  float* dst;            // T; Ypart
  long long ldv;         // of V
  long long slab;        // between partial sums of Y
  int r, pad;
};
// Layers that read one X, or some ranks of them: from rank k0 of the first layer on, np ranks
struct SplitUnit {
  const void* X;
  long long ldx;
  int m, d_in, slabs, slab_rows;
  int item0, rows;       // first work item; T = X Q: m, Y = X^T T: d_in
  short k0, np;
  short vec;             // accesses of X that are aligned: four columns (1), or element by element (0)
  short quads;           // ranks 4 k to 4 k + 3 of the panel are one layer's, and their source is aligned
  SplitLayer layer[kSplitMaxLayers];
};
template <int N> struct SplitUnits {
  int n_units, n_items, split;           // split: CTAs that share an item (T = X Q)
  unsigned wait_ns, missing, pad;        // limit of a wait; a test's: 1: a barrier expects more than comes
  SplitUnit unit[N];
};
static_assert(sizeof(SplitUnits<kSplitMaxUnits>) + sizeof(void*) <= 32764, "kernel parameters");

// Token slabs of Y = X^T T for `units` units of 128 columns on the device: whole steps of 64, the SMs' last items starting
// together; a step is about 0.7 us, an item's start 1.5 steps, a slab costs the panel QR 0.2 us.
inline int split_slab_rows(int m, long long blocks, int sm_count) {
  long long best = -1;
  int best_rows = m;
  for (int n = 1; n <= kCcMaxSlabs; ++n) {
    const int rows = ((m + n - 1) / n + 63) / 64 * 64;
    const long long slabs = (m + rows - 1) / rows, rounds = (slabs * blocks + sm_count - 1) / sm_count;
    const long long cost = rounds * (20 * (rows / 64) + 30) + 6 * slabs;
    if (best < 0 || cost < best) { best = cost; best_rows = rows; }
  }
  return best_rows;
}
// Whether they are estimated to be the faster ones for the layers `which` of L (ascending): two products X^T T and one X Q.  Both sides fitted
// to 820 lists of one to 21 layers, 64 to 12000 tokens and 64 to 4096 columns, ranks 1 to 64, all types and alignments, K = 0, 1 and 3.
// Of 1000 others (one to seven inputs of 1 to 600 MB in all, four fifths of them fp32, K = 3, the resident kernel off) the rule gains a factor of 1.498 on
// the mean (1.505 with the faster side each time) and takes the slower side by more than 3 % for seven (at most 10 %).  The CUDA cores keep ranks up to
// 4 on layers with an X of their own (their products are at 80 % of the copy rate there, where a step of these takes 0.6 us at best) and lists
// that do not fill the device.
bool split_pays(const agzo_layer* L, const std::vector<int>& which, bool share, int sm_count);
// Whether the wave's products can run here with a power step or K = 0: below 2^-109 an fp32 value's third part is no bf16 number any
// more; with a power step such inputs underflow whatever the kernel, without one the CUDA cores keep them.
bool split_takes(const ExtractWave& w, const DevLayer* dev, int K);
bool split_same_x(const DevLayer& a, const DevLayer& b);     // one unit, also by their slabs
// dev: host copy of all layers' records; share: layers on one X are one unit
cudaError_t launch_split_xt_t(const ExtractWave& w, const DevLayer* dev, bool share, DevStatus* status, cudaStream_t s);
cudaError_t launch_split_x_q(const ExtractWave& w, const DevLayer* dev, bool share, DevStatus* status, cudaStream_t s);

}  // namespace agzo

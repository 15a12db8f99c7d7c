// Algorithm 1 for small inputs in one launch, X resident in shared memory: host interface.
#pragma once

#include "agzo_common.cuh"

namespace agzo {

constexpr int kResMaxUnits = 12;        // units (runs of layers on one X) of a launch
constexpr int kResMaxLayers = 4;        // layers of a unit
constexpr int kResMaxRank = 16;         // rank of a layer
// Ranks of a unit.  Beyond, the sweeps over X are what takes the time and their chain has more SMs for them: two layers of rank 16 on
// 2000 x 1024 80 us here and 73 there, on 613 x 2048 82 and 69, three on 2000 x 1024 96 and 82 (the other way about only where X is
// tall and narrow: two on 8000 x 512 84 and 109); three of rank 8 on 613 x 1024 51 and 53.
constexpr int kResMaxPanel = 24;

struct ResidentLayer {
  float* V;
  long long ldv;
  unsigned layer_id;
  int r;
  int off;               // first rank in the unit's panel
  int row;               // first row of the staged Y (layers start at multiples of 8)
};
// Layers that read one X.  The X of a unit is cut into blocks of 128 tokens x 128 columns; a CTA keeps tb x cb of them.  The
// cj CTAs side by side cover the columns, ni such rows the tokens; a cluster holds whole rows.
struct ResidentUnit {
  const void* X;
  long long ldx;
  int x_vec, m, d;                      // x_vec: rows of X in 16-byte pieces
  int n_layers, ranks, NP, NB;          // ranks of the panel, rounded up to 8; operand rows (parts x NP, rounded up to 16)
  int rows;                             // rows of the staged Y
  int cb, tb, cj, ni;
  int gram_split;                       // warps per layer of the Gram products
  int cluster0, clusters;               // clusters of the launch that work on this unit
  int sub;                              // columns of Y that a CTA adds up for the unit, 0: all of its cb blocks for itself
  int counter;                          // index of the unit's counter
  float* ypart;                         // [ni][ranks][cj cb 128] partial sums of Y; twice, by turns, where sub = 0
  float* y;                             // [ranks][cj cb 128], where sub > 0
  double* gshare;                       // [clusters][layers][192], where sub > 0
  ResidentLayer layer[kResMaxLayers];
};
struct ResidentParams {
  int n_units, cs, K;
  unsigned long long wait_ns;           // limit of a wait for the other CTAs of a unit
  unsigned long long late_ns;           // a test's: how late the unit's first CTA comes to the first meeting
  unsigned long long seed;
  DevStatus* status;                    // may be null
  int* flag;                            // may be null: set to whether a column was dependent, to 2 where a wait ran out
  unsigned long long* counters;         // one per unit
  ResidentUnit unit[kResMaxUnits];
};

// The counter at which n CTAs meet: bit 31 turns with the last arrival whatever the order, and the low bits are as they were then,
// so nothing has to be set back.  Launches that overlap against the rules (two streams without an order) spoil one another's
// results, but when they are over the counter serves the next one again.  The upper half counts waits that ran out; a meeting that
// turns the bit back to zero borrows one from it until it is complete (bits 31 and 30 are both set then, and only then).
__host__ __device__ constexpr unsigned long long meeting_increment(int n, bool first, unsigned phase) {
  return first ? (phase ? 0ull - (1ull << 31) : 1ull << 31) - (unsigned long long)(n - 1) : 1ull;
}
constexpr unsigned long long kMeetingFailure = 1ull << 32;
__host__ __device__ constexpr unsigned meeting_phase(unsigned long long v) { return (unsigned)(v >> 31) & 1u; }
__host__ __device__ constexpr unsigned meeting_failures(unsigned long long v) { return (unsigned)(v >> 32) + (((unsigned)v >> 30) == 3u ? 1u : 0u); }

struct ResidentCaps {
  int sm_count = 0;
  int clusters[9] = {};                 // resident clusters of 1, 2, 4 and 8 CTAs, by size; 0: not usable
};
struct ResidentLaunch {
  ResidentParams p;
  int planes, parts;                    // bf16 planes of X (1: bf16, 3: fp32), parts of the operands Q and T
  int n_clusters;
  bool push;                            // the CTAs of a cluster send one another what they exchange
  bool grid_wide;                       // some unit has several clusters, which wait for one another
  size_t smem;
  size_t scratch;                       // bytes behind ypart, y and gshare
};

cudaError_t resident_init(int sm_count, ResidentCaps* caps);      // once per device
// Plans one launch for the layers; false where the resident kernel does not take them.  two_parts: the products of every layer
// would run on the tensor-core path, whose operands are two bf16 parts; else they are three (24 bits, as the CUDA-core path's fp32).
bool resident_plan(const ResidentCaps& caps, const agzo_layer* layers, int n, bool share_inputs, bool two_parts, ResidentLaunch* out);
// It is estimated to be the faster one.  fresh: the others would have the list's tables or records to write first.
bool resident_pays(const ResidentLaunch& plan, int K, bool fresh);
// points the plan at its scratch (256-byte aligned, out->scratch bytes)
void resident_bind(ResidentLaunch* plan, char* scratch);
cudaError_t launch_resident(const ResidentLaunch& plan, cudaStream_t s);
// The launch was refused for want of SMs (a context that has been given a part of the device): the other kernels serve the call.
// Clears the runtime's last error then.
bool resident_refused(cudaError_t e);

}  // namespace agzo

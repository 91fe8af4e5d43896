// snn_internal.h -- device descriptors shared by the host runtime (snn_host.cpp)
// and the kernels (snn_kernels.cu).  Not part of the public ABI.
#pragma once
#include <cstddef>
#include <cstdint>

#include <cuda_runtime.h>

namespace snn {

constexpr int kK = 1250;          // neurons per module (Sec. 2.2)
constexpr int kNPop = 3;          // F, B, I
constexpr int kZTab = 4096;       // Gaussian quantile table size (12-bit index)
constexpr int kPoisMax = 16;      // external events per neuron and step are capped at 16
constexpr int kMaxM = 2048;       // out-degree limit
constexpr uint32_t kMaxWindow = 1024;   // steps of a window at most
constexpr int kNeuronAlign = 128; // neuron arrays padded to a multiple of 128

// status bits written by kernels
constexpr uint32_t kStatusRasterOverflow = 2u;
constexpr uint32_t kStatusBarrier = 4u;   // a grid barrier ran out of its polling limit

// Time window of one graph replay (device memory, rewritten by the host
// before every replay so that captured graphs stay valid).
struct alignas(16) NetWin {
  uint32_t t0;          // absolute step of the window's first step
  uint32_t t_end;       // exclusive absolute step at which the network stops
  uint32_t bin0;        // first rate bin of the window (t0 / bin_steps)
  uint32_t t0_slot;     // t0 mod D
  uint32_t pad[4];
};

// Baked into the kernels of step k of a window when the window is captured
// (windows of one graph all start at the same t0 mod nbuf): k mod D, from
// which a kernel finds the slot of step t0 + k with the window's t0_slot and
// no division, and the input buffer of step t0 + k itself, known before the
// window is read.
struct StepMod {
  uint32_t slot;        // k mod D
  uint32_t buf;         // (t0 + k) mod nbuf
  uint32_t overlapped;  // update of step t0 + k: launched to overlap the delivery pass before it
                        // (programmatic dependent launch; its input buffer is read after griddepcontrol.wait)
};

// Recording header of a network (device memory, zeroed at every window start).
// The barrier words of the persistent kernel lie 128 bytes behind it.
struct alignas(16) RecHeader {
  uint32_t cursor;        // raster entries appended in this window
  uint32_t status;        // kStatus* bits
  uint32_t pad[2];
};

// Static description of a network.  Passed by value as a kernel parameter for
// a single network and stored in a device table for several.
struct alignas(16) NetDev {
  // --- sizes
  uint32_t N;           // neurons
  uint32_t N_pad;       // padded to kNeuronAlign
  uint32_t G, gx;       // modules, grid width
  uint32_t M;           // out-degree
  uint32_t M_pad;       // padded to a multiple of 8
  uint32_t D;           // spike-history slots = n_delay + kmin
  uint32_t fmt;         // 0 = f32 weights, 1 = i16 weights
  uint32_t row_bytes;   // bytes of one row: M_pad keys then M_pad weights
  uint32_t bin_steps;
  uint32_t key0, key1;  // Philox key (seed)
  uint32_t slot;        // index of this network in a batch
  uint32_t rec_cap;     // raster entries per window
  uint32_t rates_bins;  // bins in the rate window
  uint32_t n_delay;     // largest delay in steps
  uint32_t os;          // u16 entries per row of the delay-group table (multiple of 8)
  uint32_t kmin;        // smallest delay: steps per exchange period (delivery after steps t with (t + 1) % kmin == 0)
  uint32_t nbuf;        // input buffers = 2 kmin (the input of step t is buffer t % nbuf)
  uint32_t pad1;

  // --- per population constants (Eq. 2 propagators, Table S1)
  float vth[kNPop];
  alignas(16) uint32_t thr[kNPop][kPoisMax];   // Poisson CDF thresholds, scaled by 2^20 (read four at a time)
  // two 16-byte loads per population: {P_VV, P_Vc, P_cc, E} and {V_th, V_r,
  // alpha, refractory steps (bits)}
  float4 pa[kNPop], pb[kNPop];

  // --- device arrays
  float *V;             // [N_pad]
  float *c;             // [N_pad]
  uint8_t *ref;         // [N_pad]
  // Synaptic input of step t (2^-16 mV): acc[t % nbuf][n], accumulated by
  // reductions during the delivery pass before step t, cleared by the update.
  // The persistent kernel has kMaxVisit more behind hist, zero between windows.
  int32_t *acc;         // [nbuf][N_pad], directly followed by hist
  uint32_t *cnt;        // [D] spikes of the step with slot t mod D
  uint32_t *hist;       // [D][N_pad] their ids, in the order they were appended
  uint8_t *rows;        // [N][row_bytes]
  const uint16_t *offs; // [N][os] delay groups: records with delay <= d end at offs[s * os + d]
  const int32_t *amp;   // [3][kZTab] external amplitudes, 2^-16 mV
  const NetWin *win;    // current window
  RecHeader *rec;       // recording header
  unsigned long long *rec_entries;  // [rec_cap] (slot << 48 | k << 32 | id)
  uint32_t *rates;      // [rates_bins][G][3] window counts
  unsigned long long *ext_acc;      // [N_pad / 128] external events per 128-neuron group
};

static_assert(offsetof(NetDev, thr) % 16 == 0 && offsetof(NetDev, pa) % 16 == 0 && offsetof(NetDev, pb) % 16 == 0 &&
                  sizeof(NetDev) % 16 == 0 && sizeof(NetWin) % 16 == 0,
              "16-byte loads of the descriptor tables");

// Construction-time inputs.
struct BuildDev {
  const uint32_t *cdf;  // [G][G-1] module thresholds
  const float *ztab;    // [kZTab]
  float J[kNPop][kNPop];
  float sig[kNPop][kNPop];
  uint32_t n_delay;     // delays uniform on min_delay..n_delay
  uint32_t min_delay;
};

// ---- launchers (snn_kernels.cu) -------------------------------------------
cudaError_t prepare_kernels();
cudaError_t launch_build_rows(const NetDev &h_nd, const BuildDev &bd, cudaStream_t s);
cudaError_t launch_init_state(const NetDev &nd, cudaStream_t s);
// Persisting L2 access-policy window attached to a launch (bytes == 0: none).
struct L2Window {
  void *base = nullptr;
  size_t bytes = 0;
  float hit_ratio = 0.0f;
};
// pdl: launched with programmatic stream serialization (overlaps the previous kernel).
cudaError_t launch_update(const NetDev &nd, uint32_t k, StepMod km, int block, int groups, const L2Window &l2,
                          bool pdl, cudaStream_t s);
cudaError_t launch_deliver(const NetDev &nd, uint32_t k, StepMod km, uint32_t lanes, int warps, int blocks,
                           const L2Window &l2, bool pdl, cudaStream_t s);

// Persistent kernel: steps between two visits of a live spike, at most; kmin = 1
// networks have visit + 2 input buffers.
constexpr uint32_t kMaxVisit = 4;
// Tiles of one launch at most: a block's shared memory holds the state of fewer
// than 128, on 152 SMs.  Grids above hold no further input buffers (64x64 modules:
// 82 MB); a constant, so that snn_footprint needs no device.
constexpr uint32_t kRunMaxTiles = 128u * 152u;

// Persistent kernel: a window of steps of one or more networks in one launch
// (snn_run.cu).
struct RunArgs {
  NetDev nd;                  // single network: its descriptor and window
  NetWin win;
  const NetDev *nets;         // several networks: device tables [n_nets]
  const NetWin *wins;
  const uint32_t *tile_pre;   // [n_nets + 1] 128-neuron tiles before each network
  uint32_t n_nets;
  uint32_t n_tiles;           // tiles of all networks
  uint32_t steps;             // steps of the window (the longest of the networks)
  uint32_t nd_max;            // largest delay of the networks
  uint32_t kmin;              // smallest delay, the same for all networks
  uint32_t visit;             // steps between two visits of a live spike (1 in the period form)
  uint32_t fifo;              // live spikes of one ring that a block holds in shared memory (power of two)
  uint32_t nt;                // tiles of a block, at most
  uint32_t drives;            // external drives kept per neuron: kmin or less in the period form, else 1 or 2
  uint32_t pre;               // records of a new spike's row prefetched (multiple of 8)
  // {grid barrier count, last step (+1) that overflowed a live list, lists not taken over}, zero at launch
  uint32_t *bar;
  uint32_t *status;           // status word of a network that advances
  // t0 mod kmin, the same for all networks that advance (those that have stopped: any).  Last: among the fields above it
  // moved what every step reads, 4x4 modules 2.375 us a step instead of 2.361
  uint32_t phase;
};
struct RunShape {
  int blocks = 0, threads = 0;
  int form = 0;               // RunForm
  uint32_t fifo = 0, nt = 0, visit = 1, drives = 1;
  uint32_t tables = 0;        // networks whose descriptors fit in shared memory beside the rest
  size_t smem = 0;
};
// blocks == 0: too many tiles for one launch.  `part`: the drives of part of an exchange period will do.
RunShape run_shape(uint32_t n_tiles, uint32_t kmin, int max_threads, uint32_t n_nets, bool part);
cudaError_t launch_run(const RunArgs &a, const RunShape &sh, const L2Window &l2, cudaStream_t s);
cudaError_t prepare_run_kernels();
// Delivery keeps each warp's segment prefix in registers, in chunks of 32
// delays: one chunk up to n_delay 32, else kMaxPreChunks (n_delay <= 256).
constexpr uint32_t kMaxPreChunks = 8;
inline uint32_t pre_chunks(uint32_t n_delay) { return n_delay <= 32u ? 1u : kMaxPreChunks; }
// u16 entries per row of the delay-group table
inline uint32_t offs_stride(uint32_t n_delay) { return (n_delay + 1u + 7u) & ~7u; }
int device_sm_count();

}  // namespace snn

// ---- host helpers shared by the host translation units (snn_host.cpp) ----
#include <string>
#include <vector>
struct snn_params;
namespace snn {
void module_thresholds(const snn_params &p, std::vector<uint32_t> &out);   // Eq. 1 thresholds [G][G-1]
void gaussian_table(std::vector<float> &ztab);                             // Phi^-1((i + 0.5) / 4096)
void build_inputs(const snn_params &p, BuildDev &bd);                      // efficacy means and spreads
}  // namespace snn
int snn_validate_params(const snn_params &p);   // SNN_OK or an error code (message set)
int snn_fail(int code, const std::string &msg);  // set the thread's last error, return code

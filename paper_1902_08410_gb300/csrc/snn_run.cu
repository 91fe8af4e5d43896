// snn_run.cu -- persistent kernel: a window of time steps of one or more
// networks in one cooperative launch, one block per SM.
//
// The two-kernel path pays two dependent launches per step and, per (spike,
// delay) segment, the chain count -> list -> delay-group table -> records.
// Here
//   * a block owns every gridDim-th 128-neuron tile, so that neighbouring tiles,
//     and with them the modules of a wave front, spread over all SMs; their
//     state and external drive stay in shared memory;
//   * a block keeps the live spikes of its own tiles in shared memory, with a
//     position in each spike's row: a row is ordered by delay, so the records due
//     are the first ones from that position.  No per-step count, spike list or
//     delay-group table is read;
//   * a spike's row is visited every few steps and several delay groups are
//     delivered at a time, into as many input buffers: a group is 56 records on
//     average, and reading each by itself costs DRAM an activation per 200 bytes
//     and the SM more instructions to get at the records than to deliver them;
//   * the grid meets once per step, or once per exchange period or part of one.  Between
//     arriving and waiting a block records its spikes, draws the next external
//     drive and visits its live spikes; only the update and the delay-1 records
//     of its new spikes stand between two barriers.
//
// What bounds it: small networks, the grid barrier and two L2 or DRAM round trips
// a step (4x4 modules: 5.3 us a step as two kernels, 2.5 us here); larger ones,
// the visits and draws between two barriers.  Cycles of a step at 24x24 modules
// and 8.7 Hz (17.8 us as two kernels in the default shape, 10.1-11.3 us here):
// update 3000, records of new spikes 2900, visits and draws 9900, waiting for the
// block's other warps and the other blocks 3900; at 4x4 200, 1500, 1200 and 3600.
// The reductions by themselves are not the bound: 0.8e11 a second at 24x24, 1e11
// with two such networks, where L2 took 2e11 to 3.7e11 scattered ones.  (64
// networks of 2.3M neurons in all: 78 us as one kernel per step, 53 us here.)
// Measured beside it: one delay group per visit, 13-15 us at 24x24; whole modules
// per block with the records of the own module summed in shared memory, 17 us
// (blocks whose modules are active hold up the grid).
//
// A window starts from the spike lists in global memory (hist, cnt) and leaves
// its own last n_delay steps there, so the other launch paths can go on from
// it.  Spikes that find the block's live list full go to the global lists at
// once; while such spikes (or lists too long to take over at the start) are
// alive, every warp also takes (spike, delay) segments from them.
#include <algorithm>
#include <cstdint>

#include "snn_device.cuh"
#include "snn_internal.h"

namespace snn {

constexpr int kRunThreads = 640;
constexpr uint32_t kPendCap = 1024;      // neurons with two or more external events listed per step and block
// Barrier polls (about a microsecond each) before giving up.  The time that other streams' kernels hold SMs does not
// count: a cooperative launch starts when all its blocks can be resident (it waited 25 s behind a kernel on four SMs).
constexpr uint32_t kSpinLimit = 1u << 22;

// Live spike: id (24 bits) | step of the window + 512 (12) | position in the row (12) | network (16).
// A spike of a window before is at most 254 steps old at the window's start.
static_assert(kMaxM < (1 << 12) && kMaxWindow + 512u <= (1u << 12), "fields of a live spike");
__device__ __forceinline__ unsigned long long live_pack(uint32_t id, int kts, uint32_t p, uint32_t net) {
  return (unsigned long long)(id | ((p & 0xFFu) << 24)) |
         ((unsigned long long)((p >> 8) | ((uint32_t)(kts + 512) << 4) | (net << 16)) << 32);
}
__device__ __forceinline__ void live_unpack(unsigned long long e, uint32_t &id, int &kts, uint32_t &p, uint32_t &net) {
  const uint32_t lo = (uint32_t)e, hi = (uint32_t)(e >> 32);
  id = lo & 0xFFFFFFu;
  p = (lo >> 24) | ((hi & 0xFu) << 8);
  kts = (int)((hi >> 4) & 0xFFFu) - 512;
  net = hi >> 16;
}

// Neurons of one step's drive with more than one external event: index in the drives << 5 | events.
struct Pending {
  uint32_t n;
  uint32_t list[kPendCap];
};

struct RunShared {
  NetDev nd;                          // single network
  // Live spikes by (step of the spike mod visit): ring c holds those visited after the steps k = c mod visit.
  uint32_t tail[kMaxVisit];           // appended so far (may pass head + capacity within a step)
  uint32_t base[kMaxVisit];           // the same before this step
  uint32_t head[kMaxVisit];           // first entry that may still be alive
  struct {
    uint32_t next, draw;              // next live spike, (tile, step) unit
  } ctr[2];                           // of this interval and, cleared ahead, the next
  uint32_t abort;
  uint32_t end_k;                     // next step of the window at which a network has stopped before the others
  int last_list;                      // latest step (of the window) with spikes in the global lists still to deliver
  int lo_list;                        // first step (of the window) the global lists are read from
  unsigned long long live0;
  uint32_t tail_at[512];              // tail of the ring of step k after it, at k mod 512 (above n_delay + visit)
  Pending pend[2];
};

// MULTI: one network (its descriptor a kernel parameter), several, or several
// whose descriptors are copied to shared memory.  From global memory every
// interval reads them anew, a round trip per tile and visit: 16 networks of 4x4
// modules 8.2 us a step, 7.5 from shared memory; 4 of 16x16 21.7, 20.1; a batch
// that leaves no room for them is 2% faster with a kernel of its own.
enum RunNets : int { kOne = 0, kSeveral = 1, kTables = 2 };

template <int MULTI>
__device__ __forceinline__ const NetDev &net_of(const NetDev *nets, const RunShared &s, uint32_t net) {
  if constexpr (MULTI) return nets[net];
  else return s.nd;
}
template <int MULTI>
__device__ __forceinline__ NetWin win_of(const RunArgs &a, const NetWin *wins, uint32_t net) {
  if constexpr (MULTI) return wins[net];
  else return a.win;
}
__device__ __forceinline__ bool pass_after(const NetDev &nd, uint32_t t) { return nd.kmin == 1u || (t + 1u) % nd.kmin == 0u; }

// Forms of the kernel (all networks of a launch have the same smallest delay
// kmin, and the same phase of its period).
//   kAhead   kmin = 1.  After step k the spikes of steps k, k - visit,
//            k - 2 visit, ... are visited and their records for steps k + 2 ..
//            k + visit + 1 delivered, between arriving at the grid barrier and
//            waiting for it (the records for step k + 1 were delivered at the
//            visit before, or before the barrier when the spike is new).
//            visit + 2 input buffers rotate: step k uses buffer k mod (visit +
//            2), cleared by its update, and is next added to from step k + 1 on,
//            after the barrier that ends step k.
//   kPeriod  kmin > 1.  The grid meets once per exchange period of kmin steps
//            (where only the drives of part of a period fit, after each part);
//            all live spikes are visited before the meeting that ends a period.
//            2 kmin input buffers: the
//            updates of a period read and clear its own, the pass after it adds
//            into those of the next kmin steps.
enum RunForm { kAhead, kPeriod };

// Buffer r of the rotation, counted in N_pad entries from acc.  kAhead places 0
// and 1 where the other paths have the inputs of the window's first two steps,
// acc[t0 mod 2] and acc[(t0 + 1) mod 2] (flip = t0 mod 2); the rest lie behind
// the D spike lists that follow acc.  kPeriod: buffer t mod nbuf (flip = gap = 0).
__device__ __forceinline__ uint32_t buffer_at(uint32_t r, uint32_t flip, uint32_t gap) { return r < 2u ? r ^ flip : r + gap; }
// kAhead: r = k mod (visit + 2), k a step of the window that starts at t0.
template <int FORM>
__device__ __forceinline__ int32_t *input_of(const NetDev &nd, uint32_t t0, uint32_t k, uint32_t r) {
  const uint32_t b = FORM == kAhead ? buffer_at(r, t0 & 1u, nd.D) : (t0 + k) % nd.nbuf;
  return nd.acc + (size_t)b * nd.N_pad;
}

// Where the records of a spike go: a record of delay d into buffer off + d of a
// rotation of n (off may be negative; off + d is in 1 .. 2 n - 1 for those due).
struct Due {
  int off;
  uint32_t n, flip, gap;
};
// Records due after step k (relative to a window that starts at t0) of a spike `age` steps old.
template <int FORM>
__device__ __forceinline__ Due due_at(const RunArgs &a, const NetDev &nd, uint32_t t0, uint32_t k, uint32_t r, int age) {
  if constexpr (FORM == kAhead) return Due{(int)r - age, a.visit + 2u, t0 & 1u, nd.D};
  else return Due{(int)((t0 + k) % nd.nbuf) - age, nd.nbuf, 0u, 0u};
}

// Reduce the records of source s from position p whose delay is at most dlim;
// returns the position behind them.  Whole warp, 32 U records in flight.  The
// records of a row are ordered by delay: those due are the first ones from p.
template <int U>
__device__ __forceinline__ uint32_t deliver_front(const NetDev &nd, uint32_t s, uint32_t p, uint32_t dlim, const Due &to) {
  const uint32_t lane = lane_id(), M = nd.M, N_pad = nd.N_pad;
  const uint8_t *row = nd.rows + (size_t)s * nd.row_bytes;
  const bool i16 = nd.fmt != 0u;
  int32_t *acc = nd.acc;
  while (p < M) {
    const uint32_t i0 = p + lane;
    const uint32_t *kp = reinterpret_cast<const uint32_t *>(row) + i0;
    const uint8_t *wp = row + (size_t)nd.M_pad * 4u + (size_t)i0 * (i16 ? 2u : 4u);
    uint32_t k[U];
    int32_t v[U];
#pragma unroll
    for (int u = 0; u < U; ++u) k[u] = ld_rec_u32_if(i0 + 32u * u < M, kp + 32 * u, 0xFFFFFFFFu);
    if (i16) {
#pragma unroll
      for (int u = 0; u < U; ++u) v[u] = ld_rec_s16_if(i0 + 32u * u < M, reinterpret_cast<const int16_t *>(wp) + 32 * u);
    } else {
#pragma unroll
      for (int u = 0; u < U; ++u)
        v[u] = (int32_t)ld_rec_u32_if(i0 + 32u * u < M, reinterpret_cast<const uint32_t *>(wp) + 32 * u, 0u);
    }
    uint32_t n = 0;
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const uint32_t d = k[u] >> 24;
      const bool due = d <= dlim;
      n += __popc(__ballot_sync(0xFFFFFFFFu, due));
      if (due) {
        uint32_t b = (uint32_t)(to.off + (int)d);
        if (b >= to.n) b -= to.n;
        b = buffer_at(b, to.flip, to.gap);
        red_add_s32(acc + (size_t)(b * N_pad + (k[u] & 0xFFFFFFu)),
                    i16 ? v[u] * 64 : __float2int_rn(__fmul_rn(__int_as_float(v[u]), 65536.0f)));
      }
    }
    p += n;
    if (n < 32u * U) break;
  }
  return p;
}

// Raster entry and rate count of one spike (the position in the raster is given).
__device__ __forceinline__ void record_at(const NetDev &nd, const NetWin &w, uint32_t pos, uint32_t id, uint32_t k) {
  if (pos < nd.rec_cap)
    nd.rec_entries[pos] = ((unsigned long long)nd.slot << 48) | ((unsigned long long)k << 32) | id;
  else
    atomicOr(&nd.rec->status, kStatusRasterOverflow);
  const uint32_t bin = (w.t0 + k) / nd.bin_steps - w.bin0;
  const uint32_t m = id / (uint32_t)kK;
  red_add_u32(nd.rates + ((size_t)bin * nd.G + m) * 3u + pop_of_local(id - m * (uint32_t)kK), 1u);
}

// Append to the global list of step ts (absolute).
__device__ __forceinline__ void list_append(const NetDev &nd, uint32_t ts, uint32_t id) {
  const uint32_t slot = ts % nd.D;
  const uint32_t pos = atomicAdd(nd.cnt + slot, 1u);
  nd.hist[(size_t)slot * nd.N_pad + pos] = id;
}

// Spikes that found the live list full (mask of each lane): delivered up to
// delay dlim here (0: not now) and appended to the global list of their step.
// Whole warp.
static __device__ __noinline__ void spill_spikes(const RunArgs &a, const NetDev &nd, const NetWin &w, uint32_t n0,
                                                 uint32_t mask, uint32_t k, uint32_t dlim, Due to) {
  const uint32_t lane = lane_id();
#pragma unroll 1
  for (uint32_t q = 0; q < 4u; ++q) {
    uint32_t bits = __ballot_sync(0xFFFFFFFFu, (mask >> q) & 1u);
    while (bits) {
      const uint32_t id = __shfl_sync(0xFFFFFFFFu, n0, __ffs(bits) - 1) + q;
      bits &= bits - 1u;
      if (dlim) deliver_front<2>(nd, id, 0u, dlim, to);
      if (lane == 0) {
        list_append(nd, w.t0 + k, id);
        record_at(nd, w, atomicAdd(&nd.rec->cursor, 1u), id, k);
        atomicMax(a.bar + 1, k + 1u);
      }
    }
  }
}

// Segments of the global lists' spikes of steps lo <= ts - t < before (relative
// to t) in the pass after step t, this warp is number wi of wn.  `one`: the input of step t + 1 where it is not buffer
// (t + 1) mod nbuf.
static __device__ __noinline__ void deliver_lists(const NetDev &nd, uint32_t t, int lo, int before, uint32_t wi, uint32_t wn,
                                                  int32_t *one) {
  const uint32_t lane = lane_id();
  for (uint32_t j = 0; j < nd.kmin; ++j) {
    const uint32_t T = t + 1u + j, Tm = T % nd.D;
    int32_t *acc_T = one ? one : nd.acc + (size_t)(T % nd.nbuf) * nd.N_pad;
    constexpr int NCH = (int)kMaxPreChunks;
    WarpPrefix<NCH> P;
    uint32_t run = 0;
#pragma unroll
    for (int c = 0; c < NCH; ++c) {
      const uint32_t d = 32u * c + lane + 1u;
      const int rel = (int)(j + 1u) - (int)d;   // step of the spike, relative to t
      const bool use = d >= nd.kmin && d <= nd.n_delay && rel >= lo && rel < before;
      uint32_t x = use ? ld_cg_u32(nd.cnt + slot_back(Tm, d, nd.D)) : 0u;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const uint32_t y = __shfl_up_sync(0xFFFFFFFFu, x, o);
        if (lane >= (uint32_t)o) x += y;
      }
      P.base[c] = run;
      P.incl[c] = x + run;
      run = __shfl_sync(0xFFFFFFFFu, P.incl[c], 31);
    }
    P.total = run;
    deliver_segments<NCH>(nd, P, Tm, acc_T, wi, wn, 32u);
  }
}

// Network and first neuron of tile g of the table.
template <int MULTI>
__device__ __forceinline__ uint2 tile_at(const RunArgs &a, uint32_t g) {
  if constexpr (!MULTI) return make_uint2(0u, g * 128u);
  uint32_t lo = 0, hi = a.n_nets;   // last network with tile_pre <= g
  while (hi - lo > 1u) {
    const uint32_t mid = (lo + hi) >> 1;
    if (a.tile_pre[mid] <= g) lo = mid; else hi = mid;
  }
  return make_uint2(lo, (g - a.tile_pre[lo]) * 128u);
}

// Grid barrier: thread 0 arrives; later it waits until every block has
// arrived `met` times (a bounded number of polls, then s.abort).
__device__ __forceinline__ void grid_arrive(const RunArgs &a) {
  __threadfence();
  atomicAdd(a.bar, 1u);
}
__device__ __forceinline__ void grid_wait(const RunArgs &a, RunShared &s, uint32_t met) {
  const uint32_t want = met * gridDim.x;
  uint32_t got, spins = 0;
  while (true) {
    asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(got) : "l"(a.bar) : "memory");
    if ((int)(got - want) >= 0) break;
    if (++spins > kSpinLimit) {
      s.abort = 1u;
      break;
    }
  }
}

template <int N>
struct Width {
  static constexpr int n = N;
};

// MULTI: several networks (device tables).
template <int MULTI, int FORM>
__global__ void __launch_bounds__(kRunThreads, 1) k_run(const __grid_constant__ RunArgs a) {
  extern __shared__ __align__(128) uint8_t smem[];
  __shared__ RunShared s;
  constexpr bool PERIOD = FORM == kPeriod;
  const uint32_t nt = blockIdx.x < a.n_tiles ? (a.n_tiles - 1u - blockIdx.x) / gridDim.x + 1u : 0u;
  const bool deep = !PERIOD && a.drives == 2u;   // drives are drawn two steps ahead
  const uint32_t P = a.drives;                   // drives kept per tile
  const uint32_t C = PERIOD ? 1u : a.visit, cap = a.fifo;
  // live spikes of ring c at c * cap
  unsigned long long *live = reinterpret_cast<unsigned long long *>(smem);
  uint2 *s_tile = reinterpret_cast<uint2 *>(live + C * cap);
  uint32_t *s_ext = reinterpret_cast<uint32_t *>(s_tile + a.nt);
  // (8 + 4) nt bytes behind the 16-byte aligned lists, rounded up to 16
  int4 *s_I = reinterpret_cast<int4 *>(smem + ((C * cap * 8u + a.nt * 12u + 15u) & ~15u));
  float4 *s_V = reinterpret_cast<float4 *>(s_I + a.nt * P * 32u);
  float4 *s_c = s_V + a.nt * 32u;
  uint32_t *s_ref = reinterpret_cast<uint32_t *>(s_c + a.nt * 32u);
  const uint32_t tid = threadIdx.x, warp = tid >> 5, lane = lane_id(), nw = blockDim.x >> 5;
  // descriptors and windows of several networks, in shared memory where they fit: a barrier ends what L1 holds of them
  const NetDev *nets = MULTI == kTables ? reinterpret_cast<const NetDev *>(s_ref + a.nt * 32u) : a.nets;   // 16-byte aligned
  const NetWin *wins = MULTI == kTables ? reinterpret_cast<const NetWin *>(nets + a.n_nets) : a.wins;

  // ---- prologue
  if constexpr (!MULTI) {
    const uint32_t *src = reinterpret_cast<const uint32_t *>(&a.nd);
    uint32_t *dst = reinterpret_cast<uint32_t *>(&s.nd);
    for (uint32_t i = tid; i < sizeof(NetDev) / 4; i += blockDim.x) dst[i] = src[i];
  }
  if constexpr (MULTI == kTables) {
    uint4 *dst = reinterpret_cast<uint4 *>(s_ref + a.nt * 32u);
    const uint32_t n = a.n_nets * (uint32_t)(sizeof(NetDev) / 16u), m = a.n_nets * (uint32_t)(sizeof(NetWin) / 16u);
    for (uint32_t i = tid; i < n + m; i += blockDim.x)
      dst[i] = i < n ? reinterpret_cast<const uint4 *>(a.nets)[i] : reinterpret_cast<const uint4 *>(a.wins)[i - n];
  }
  if (tid == 0) {
    for (uint32_t c = 0; c < kMaxVisit; ++c) s.tail[c] = s.base[c] = s.head[c] = 0u;
    for (uint32_t i = 0; i < 2u; ++i) s.ctr[i].next = s.ctr[i].draw = s.pend[i].n = 0u;
    s.abort = 0u;
    s.live0 = 0ull;
    s.last_list = -100000;
    s.lo_list = 0;
    s.end_k = 0xFFFFFFFFu;
  }
  for (uint32_t j = tid; j < nt; j += blockDim.x) {
    s_tile[j] = tile_at<MULTI>(a, blockIdx.x + j * gridDim.x);
    s_ext[j] = 0u;
  }
  __syncthreads();
  for (uint32_t j = warp; j < nt; j += nw) {
    const uint2 tile = s_tile[j];
    const NetDev &nd = net_of<MULTI>(nets, s, tile.x);
    const uint32_t i4 = (tile.y >> 2) + lane;
    s_V[j * 32u + lane] = ld_cg_f4(reinterpret_cast<const float4 *>(nd.V) + i4);
    s_c[j * 32u + lane] = ld_cg_f4(reinterpret_cast<const float4 *>(nd.c) + i4);
    s_ref[j * 32u + lane] = ld_cg_u32(reinterpret_cast<const uint32_t *>(nd.ref) + i4);
  }
  // Spikes of earlier windows that are still alive: the steps from the first
  // one the next pass reaches.  One (network, delay slot) per thread; the lists
  // are dealt over the blocks.  When a block's share may not fit its rings, the
  // blocks meet to learn whether any did not; then all are delivered from the
  // global lists.
  uint32_t met = 0;   // grid barriers passed
  auto each_slot = [&](auto &&use) {
    for (uint32_t i = tid; i < a.n_nets * a.nd_max; i += blockDim.x) {
      const uint32_t net = MULTI ? i / a.nd_max : 0u, back = i - net * a.nd_max + 1u;   // step t0 - back
      const NetDev &nd = net_of<MULTI>(nets, s, net);
      const NetWin w = win_of<MULTI>(a, wins, net);
      if (w.t0 >= w.t_end || back > w.t0) continue;
      const uint32_t tp = w.t0 + (nd.kmin - 1u - w.t0 % nd.kmin);   // first pass of the window
      if (tp + 1u > w.t0 - back + nd.n_delay) continue;
      use(nd, net, i, back, (w.t0 - back) % nd.D, tp - (w.t0 - back));
    }
  };
  unsigned long long sum = 0;
  each_slot([&](const NetDev &nd, uint32_t, uint32_t, uint32_t, uint32_t slot, uint32_t) { sum += ld_cg_u32(nd.cnt + slot); });
  if (sum) atomicAdd(&s.live0, sum);
  __syncthreads();
  // `reach`: the pass before the first one reached the inputs up to that delay (a spike it has not seen has no delay
  // that short)
  each_slot([&](const NetDev &nd, uint32_t net, uint32_t i, uint32_t back, uint32_t slot, uint32_t reach) {
    const uint32_t n = ld_cg_u32(nd.cnt + slot), c = (C - back % C) % C;
    for (uint32_t e = (blockIdx.x + gridDim.x - (i * 61u) % gridDim.x) % gridDim.x; e < n; e += gridDim.x) {
      const uint32_t id = ld_cg_u32(nd.hist + (size_t)slot * nd.N_pad + e), at = atomicAdd(&s.tail[c], 1u);
      if (at < cap / 2u) live[c * cap + at] = live_pack(id, -(int)back, nd.offs[(size_t)id * nd.os + reach], net);
    }
  });
  __syncthreads();
  if (s.live0 / gridDim.x + (unsigned long long)a.n_nets * a.nd_max > cap / 2u) {   // may be more than half a ring
    ++met;
    if (tid == 0) {
      for (uint32_t c = 0; c < C; ++c)
        if (s.tail[c] > cap / 2u) atomicOr(a.bar + 2, 1u);
      grid_arrive(a);
      grid_wait(a, s, met);
      if (ld_cg_u32(a.bar + 2)) {
        for (uint32_t c = 0; c < C; ++c) s.tail[c] = 0u;
        s.last_list = -1;
        s.lo_list = -512;
      }
    }
    __syncthreads();
  }
  if (tid < C) s.tail_at[(tid - C) & 511u] = s.base[tid] = s.tail[tid];   // as if of the ring's last step before 0

  // live spikes of networks whose window has lo .. hi steps, into the lists their next window starts from
  auto leave = [&](uint32_t lo, uint32_t hi) {
    for (uint32_t c = 0; c < C; ++c)
      for (uint32_t e = s.head[c] + tid, n = min(s.tail[c], s.head[c] + cap); e < n; e += blockDim.x) {
        uint32_t id, p, net;
        int kts;
        live_unpack(live[c * cap + (e & (cap - 1u))], id, kts, p, net);
        if (kts < 0) continue;   // in the lists already
        const NetDev &nd = net_of<MULTI>(nets, s, net);
        const NetWin w = win_of<MULTI>(a, wins, net);
        const uint32_t adv = w.t_end - w.t0;
        if (adv >= lo && adv <= hi && w.t0 + (uint32_t)kts + nd.n_delay >= w.t_end)
          list_append(nd, w.t0 + (uint32_t)kts, id);
      }
  };
  auto find_end = [&](uint32_t k) {
    for (uint32_t i = tid; i < a.n_nets; i += blockDim.x) {
      const uint32_t adv = wins[i].t_end - wins[i].t0;
      if (adv > k && adv < a.steps) atomicMin(&s.end_k, adv);
    }
  };
  auto next_end = [&](uint32_t k) {
    __syncthreads();
    if (tid == 0) s.end_k = 0xFFFFFFFFu;
    __syncthreads();
    find_end(k);
    __syncthreads();
  };
  if constexpr (MULTI) find_end(0u);

  // The records of live entry e of ring c for the steps of the window up to
  // `upto`, after step k.  Whole warp, 32 U records in flight.
  auto visit = [&](auto U, uint32_t c, uint32_t e, uint32_t k, uint32_t r, uint32_t upto) {
    unsigned long long *at = live + c * cap + (e & (cap - 1u));
    uint32_t id, p, net;
    int kts;
    live_unpack(*at, id, kts, p, net);
    const NetDev &nd = net_of<MULTI>(nets, s, net);
    const NetWin w = win_of<MULTI>(a, wins, net);
    const uint32_t adv = w.t_end - w.t0;
    // kAhead: nothing beyond the first step after the network's window
    const int dlim = (int)(PERIOD ? upto : min(upto, adv)) - kts;
    if (PERIOD ? k >= adv : dlim <= 0) return;
    const uint32_t q = deliver_front<decltype(U)::n>(nd, id, p, (uint32_t)min(dlim, 254),
                                                     due_at<FORM>(a, nd, w.t0, k, r, (int)k - kts));
    if (q != p && lane == 0) *at = live_pack(id, kts, q, net);
  };

  // The entries [from, to) of ring c as they come, their records for steps up to `upto`, after step k.
  auto visit_all = [&](uint32_t c, uint32_t from, uint32_t to, uint32_t k, uint32_t r, uint32_t upto, uint32_t ci) {
    while (true) {
      uint32_t e = 0;
      if (lane == 0) e = atomicAdd(&s.ctr[ci].next, 1u);
      e = from + __shfl_sync(0xFFFFFFFFu, e, 0);
      if (e >= to) break;
      visit(Width<8>{}, c, e, k, r, upto);
    }
  };

  // External drive of the block's tiles at steps k .. k + L - 1 into s_I: (tile,
  // step) units taken as they come
  auto draw = [&](uint32_t k, uint32_t L, uint32_t ci, Pending &pend) {
    const uint32_t units = nt * L;
    while (true) {
      uint32_t u = 0;
      if (lane == 0) u = atomicAdd(&s.ctr[ci].draw, 1u);
      u = __shfl_sync(0xFFFFFFFFu, u, 0);
      if (u >= units) break;
      const uint32_t i = PERIOD ? u / nt : 0u, j = PERIOD ? u - i * nt : u;
      const uint2 tile = s_tile[j];
      const NetDev &nd = net_of<MULTI>(nets, s, tile.x);
      const NetWin w = win_of<MULTI>(a, wins, tile.x);
      const uint32_t t = w.t0 + k + i;
      if (t >= w.t_end) continue;
      const uint32_t n0 = tile.y + lane * 4u, slot = PERIOD ? j * P + i : (deep ? j * 2u + (k & 1u) : j);
      int p0, p1;
      pair_pops(n0, p0, p1);
      uint32_t kx[4];
      const int4 I = first_drive(nd, n0, t, p0, p1, kx);
      s_I[slot * 32u + lane] = I;
      uint32_t ext = 0;
      if (n0 < nd.N) ext = kx[0] + kx[1];
      if (n0 + 2u < nd.N) ext += kx[2] + kx[3];
      ext = __reduce_add_sync(0xFFFFFFFFu, ext);
      if (lane == 0) {
        if constexpr (PERIOD) atomicAdd(&s_ext[j], ext);
        else s_ext[j] += ext;
      }
#pragma unroll
      for (int q = 0; q < 4; ++q)
        if (kx[q] > 1u) {
          const uint32_t at = atomicAdd(&pend.n, 1u), n = slot * 128u + lane * 4u + q;
          if (at < kPendCap)
            pend.list[at] = (n << 5) | kx[q];
          else
            reinterpret_cast<int32_t *>(s_I)[n] += extra_sum(nd, q < 2 ? p0 : p1, kx[q], n0 + q, t);
        }
    }
  };
  // events after the first of the listed neurons, one neuron per thread (the last warps first)
  auto draw_more = [&](uint32_t k, const Pending &pend) {
    const uint32_t np = min(pend.n, kPendCap);
    for (uint32_t x = (nw - 1u - warp) * 32u + lane; x < np; x += blockDim.x) {
      const uint32_t e = pend.list[x], at = e >> 5, kx = e & 31u;
      const uint32_t slot = at >> 7, j = PERIOD ? slot / P : slot >> (deep ? 1 : 0), i = PERIOD ? slot - j * P : 0u;
      const uint2 tile = s_tile[j];
      const NetDev &nd = net_of<MULTI>(nets, s, tile.x);
      const uint32_t n = tile.y + (at & 127u);
      reinterpret_cast<int32_t *>(s_I)[at] +=
          extra_sum(nd, pop_of_local(n % (uint32_t)kK), kx, n, win_of<MULTI>(a, wins, tile.x).t0 + k + i);
    }
  };
  const uint32_t phase0 = PERIOD ? a.phase : 0u;
  auto interval = [&](uint32_t k) {   // steps until the grid meets again
    return PERIOD ? min(min(a.kmin - (phase0 + k) % a.kmin, P), a.steps - k) : 1u;
  };
  __syncthreads();
  draw(0u, interval(0u), (met & 1u) ^ 1u, s.pend[0]);
  if constexpr (!PERIOD) {   // up to the steps that the first visit of each ring leaves out
    for (uint32_t c = 0; c < C; ++c)
      for (uint32_t e = warp; e < s.base[c]; e += nw) visit(Width<8>{}, c, e, 0u, 0u, c + 1u);
  }
  __syncthreads();
  draw_more(0u, s.pend[0]);
  if (deep) {
    if (tid == 0) s.ctr[(met & 1u) ^ 1u].draw = 0u;
    __syncthreads();
    if (1u < a.steps) draw(1u, 1u, (met & 1u) ^ 1u, s.pend[1]);
  }
  __syncthreads();
  if (tid == 0) s.pend[0].n = 0u;
  __syncthreads();

  uint32_t rk = 0, ck = 0;   // k mod (visit + 2), k mod visit
  for (uint32_t k = 0; k < a.steps && !s.abort;) {
    const uint32_t L = interval(k), kl = k + L - 1u;   // steps of this interval, its last step
    const uint32_t ring = PERIOD ? 0u : ck, ci = met & 1u;
    const uint32_t base = s.base[ring], head = s.head[ring];
    unsigned long long *rlive = live + ring * cap;
    if constexpr (MULTI) {
      if (k == s.end_k) {   // networks that stopped: no block reads their lists any more
        leave(k, k);
        next_end(k);
      }
    }

    // the list counts of the steps after a pass start at zero (not read or appended to before the next barrier)
    if (warp == nw - 1u)
      for (uint32_t net = blockIdx.x + lane * gridDim.x; net < a.n_nets; net += gridDim.x * 32u) {
        const NetDev &nd = net_of<MULTI>(nets, s, net);
        const NetWin w = win_of<MULTI>(a, wins, net);
        const uint32_t t = w.t0 + kl;
        if (t < w.t_end && pass_after(nd, t))
          for (uint32_t i = 0; i < nd.kmin; ++i) nd.cnt[(t + 1u + i) % nd.D] = 0u;
      }

    // ---- update of the block's tiles
    for (uint32_t j = warp; j < nt; j += nw) {
      const uint2 tile = s_tile[j];
      const NetDev &nd = net_of<MULTI>(nets, s, tile.x);
      const NetWin w = win_of<MULTI>(a, wins, tile.x);
      if (w.t0 + k >= w.t_end) continue;
      const uint32_t n0 = tile.y + lane * 4u, i4 = n0 >> 2;
      constexpr uint32_t IN = PERIOD ? 4u : 1u;   // steps whose inputs are loaded together
      const uint32_t Ln = PERIOD ? min(L, w.t_end - w.t0 - k) : 1u;
      int4 I[IN];
      auto load = [&](uint32_t i0) {
#pragma unroll
        for (uint32_t i = 0; i < IN; ++i)
          I[i] = i0 + i < Ln ? ld_cg_i4(reinterpret_cast<const int4 *>(input_of<FORM>(nd, w.t0, k + i0 + i, rk)) + i4)
                             : make_int4(0, 0, 0, 0);
      };
      load(0u);
      int p0, p1;
      pair_pops(n0, p0, p1);
      float4 V = s_V[j * 32u + lane], c = s_c[j * 32u + lane];
      uint32_t ref = s_ref[j * 32u + lane];
      for (uint32_t i0 = 0; i0 < Ln; i0 += IN) {
        if (i0) load(i0);
#pragma unroll
        for (uint32_t i = 0; i < IN; ++i) {
          if (i0 + i >= Ln) break;
          const uint32_t ki = k + i0 + i;
          int4 E = s_I[(PERIOD ? j * P + i0 + i : (deep ? j * 2u + (k & 1u) : j)) * 32u + lane];
          if (I[i].x | I[i].y | I[i].z | I[i].w) {
            reinterpret_cast<int4 *>(input_of<FORM>(nd, w.t0, ki, rk))[i4] = make_int4(0, 0, 0, 0);
            E.x += I[i].x;
            E.y += I[i].y;
            E.z += I[i].z;
            E.w += I[i].w;
          }
          const uint32_t mask = run_step4(nd, n0, p0, p1, V, c, ref, E);
          if (__any_sync(0xFFFFFFFFu, mask)) {
            uint32_t r = __popc(mask), tot = r;   // rank of the lane's spikes
#pragma unroll
            for (uint32_t o = 1; o < 32u; o <<= 1) {
              const uint32_t y = __shfl_up_sync(0xFFFFFFFFu, tot, o);
              if (lane >= o) tot += y;
            }
            r = tot - r;
            tot = __shfl_sync(0xFFFFFFFFu, tot, 31);
            uint32_t e = 0;
            if (lane == 0) e = atomicAdd(&s.tail[ring], tot);
            e = __shfl_sync(0xFFFFFFFFu, e, 0) + r;
            uint32_t full = 0;
#pragma unroll
            for (uint32_t q = 0; q < 4u; ++q)
              if ((mask >> q) & 1u) {
                if (e - head < cap) {
                  const uint32_t id = n0 + q;
                  rlive[e & (cap - 1u)] = live_pack(id, (int)ki, 0u, tile.x);
                  // the first records are next
                  const uint8_t *row = nd.rows + (size_t)id * nd.row_bytes;
                  bulk_prefetch_l2(row, min(a.pre * 4u, nd.M_pad * 4u));
                  bulk_prefetch_l2(row + (size_t)nd.M_pad * 4u, min(a.pre, nd.M_pad) * (nd.fmt ? 2u : 4u));
                } else {
                  full |= 1u << q;
                }
                ++e;
              }
            if (__any_sync(0xFFFFFFFFu, full)) {
              // the pass that ends the interval reaches steps up to kl + kmin
              const uint32_t age = kl - ki;
              spill_spikes(a, nd, w, n0, full, ki, w.t0 + kl < w.t_end && pass_after(nd, w.t0 + kl) ? age + nd.kmin : 0u,
                           due_at<FORM>(a, nd, w.t0, kl, rk, (int)age));
            }
          }
        }
      }
      s_V[j * 32u + lane] = V;
      s_c[j * 32u + lane] = c;
      s_ref[j * 32u + lane] = ref;
    }
    __syncthreads();

    if constexpr (MULTI && PERIOD) {
      if (s.end_k <= kl) {   // networks that stop inside the period: they have no pass now, so nobody reads their lists
        leave(k + 1u, kl);
        next_end(kl);
      }
    }

    // ---- delivery before the barrier
    const uint32_t tail = min(s.tail[ring], head + cap);
    const bool more = k + L < a.steps;
    // Visits wait for records and reductions, the draws for issue slots: half of the warps begin with each.
    auto visit_and_draw = [&](bool visits, uint32_t upto) {
      for (uint32_t i = 0; i < 2u; ++i) {
        if ((i ^ warp) & 1u) {
          const uint32_t kd = deep ? k + 2u : k + L;
          if (kd < a.steps) draw(kd, interval(kd), ci, s.pend[PERIOD ? ci : kd & 1u]);
        } else {
          if (visits) visit_all(ring, head, tail, kl, rk, upto, ci);
        }
      }
    };
    if constexpr (PERIOD) {
      visit_and_draw((phase0 + kl + 1u) % a.kmin == 0u, kl + a.kmin);
    } else {
      for (uint32_t e = base + warp; e < tail; e += nw) visit(Width<3>{}, ring, e, k, rk, k + 1u);
    }
    if (s.last_list >= (int)kl + 1 - (int)a.nd_max) {   // global lists hold live spikes (block-uniform)
      const uint32_t gw = blockIdx.x * nw + warp, total = gridDim.x * nw;
      auto lists = [&](const NetDev &nd, const NetWin &w, uint32_t wi, uint32_t wn) {
        if (w.t0 + kl < w.t_end && pass_after(nd, w.t0 + kl))
          deliver_lists(nd, w.t0 + kl, s.lo_list - (int)kl, (int)k - (int)kl, wi, wn,
                        PERIOD ? nullptr : input_of<FORM>(nd, w.t0, k + 1u, rk + 1u == a.visit + 2u ? 0u : rk + 1u));
      };
      if constexpr (!MULTI) {
        lists(s.nd, a.win, gw, total);
      } else {
        // warps are dealt to the networks in proportion to their tiles, one at least
        auto first = [&](uint32_t net) { return (uint32_t)((unsigned long long)a.tile_pre[net] * total / a.n_tiles); };
        uint32_t net = tile_at<MULTI>(a, (uint32_t)((unsigned long long)gw * a.n_tiles / total)).x;
        while (net > 0u && max(first(net - 1u) + 1u, first(net)) > gw) --net;   // the first network with this warp
        for (; net < a.n_nets && first(net) <= gw; ++net) {
          const uint32_t lo = first(net), hi = max(lo + 1u, first(net + 1u));
          if (hi > gw) lists(nets[net], wins[net], gw - lo, hi - lo);
        }
      }
    }
    if (tid == 0) {   // last used before the barrier before
      s.ctr[ci ^ 1u].next = s.ctr[ci ^ 1u].draw = 0u;
      s.pend[PERIOD ? ci ^ 1u : (k + (deep ? 2u : 1u)) & 1u].n = 0u;
    }
    __syncthreads();

    // ---- arrive; record, visit and draw; wait
    ++met;
    if (tid == 0) {
      grid_arrive(a);
      for (uint32_t i = k; i <= kl; ++i) s.tail_at[i & 511u] = tail;
      s.tail[ring] = s.base[ring] = tail;
      // spikes of steps <= kl + 1 - nd_max have delivered every delay; in the period form those of the whole
      // exchange period of that step, once its pass is done
      const int done = (int)kl - (int)((a.nd_max + C - 2u) / C * C);
      if (done >= (int)ring - (int)C && (!PERIOD || (phase0 + kl + 1u) % a.kmin == 0u))
        s.head[ring] = s.tail_at[(uint32_t)done & 511u];
    }
    if (warp == nw - 1u) {
      for (uint32_t e0 = base; e0 < tail; e0 += 32u) {
        const uint32_t e = e0 + lane;
        uint32_t id = 0, p, net = 0;
        int kts = 0;
        if (e < tail) live_unpack(rlive[e & (cap - 1u)], id, kts, p, net);
        uint32_t at = 0;
        if constexpr (MULTI) {
          if (e < tail) at = atomicAdd(&nets[net].rec->cursor, 1u);
        } else {
          if (lane == 0) at = atomicAdd(&s.nd.rec->cursor, min(32u, tail - e0));
          at = __shfl_sync(0xFFFFFFFFu, at, 0) + lane;
        }
        if (e < tail) record_at(net_of<MULTI>(nets, s, net), win_of<MULTI>(a, wins, net), at, id, (uint32_t)kts);
      }
    }
    if constexpr (PERIOD) {
      if (more) draw_more(k + L, s.pend[ci]);
    } else if (more) {
      if (deep) draw_more(k + 1u, s.pend[(k + 1u) & 1u]);   // drawn in the last interval
      visit_and_draw(true, k + C + 1u);
      if (!deep) {
        __syncthreads();
        draw_more(k + 1u, s.pend[(k + 1u) & 1u]);
      }
    }
    if (tid == 0) {
      grid_wait(a, s, met);
      const uint32_t over = ld_cg_u32(a.bar + 1);
      if (over) s.last_list = max(s.last_list, (int)over - 1);
    }
    __syncthreads();
    k += L;
    rk = rk + 1u == a.visit + 2u ? 0u : rk + 1u;
    ck = ck + 1u == C ? 0u : ck + 1u;
  }

  // ---- epilogue: live spikes, external events, inputs and state back to global memory
  if (s.abort) {
    if (tid == 0) atomicOr(a.status, kStatusBarrier);
    return;
  }
  leave(a.steps, a.steps);
  for (uint32_t j = tid; j < nt; j += blockDim.x) {
    const uint2 tile = s_tile[j];
    if (s_ext[j]) net_of<MULTI>(nets, s, tile.x).ext_acc[tile.y >> 7] += s_ext[j];
  }
  for (uint32_t j = warp; j < nt; j += nw) {
    const uint2 tile = s_tile[j];
    const NetDev &nd = net_of<MULTI>(nets, s, tile.x);
    const NetWin w = win_of<MULTI>(a, wins, tile.x);
    const uint32_t n0 = tile.y + lane * 4u, i4 = n0 >> 2;
    if (n0 >= nd.N) continue;
    if constexpr (!PERIOD) {   // the input of the next step goes where the other paths read it
      const uint32_t adv = w.t_end - w.t0;
      int4 *from = reinterpret_cast<int4 *>(input_of<FORM>(nd, w.t0, adv, adv % (a.visit + 2u))) + i4;
      int4 *to = reinterpret_cast<int4 *>(nd.acc + (size_t)(w.t_end & 1u) * nd.N_pad) + i4;
      if (from != to) {
        *to = ld_cg_i4(from);
        *from = make_int4(0, 0, 0, 0);
      }
    }
    reinterpret_cast<float4 *>(nd.V)[i4] = s_V[j * 32u + lane];
    reinterpret_cast<float4 *>(nd.c)[i4] = s_c[j * 32u + lane];
    reinterpret_cast<uint32_t *>(nd.ref)[i4] = s_ref[j * 32u + lane];
  }
}

// ---------------------------------------------------------------------------
// Shape and launch
// ---------------------------------------------------------------------------
// Shared memory of a block with nt tiles: live lists, tile table, and per
// neuron `drives` drives (4 bytes each), V, c and the refractory counter.
static size_t run_smem(uint32_t drives, uint32_t nt, uint32_t entries) {
  return (((size_t)entries * 8u + (size_t)nt * 12u + 15u) & ~(size_t)15u) + (size_t)nt * 128u * (4u * drives + 9u);
}

// Dynamic shared memory of a block: the opt-in maximum less the static part.
static size_t run_smem_budget() {
  static const size_t budget = [] {
    int dev = 0, optin = 0;
    if (cudaGetDevice(&dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev) != cudaSuccess || optin <= 0)
      optin = 200 * 1024;
    return std::min<size_t>((size_t)optin, 227u * 1024u) - sizeof(RunShared) - 1024u;
  }();
  return budget;
}

using RunKernel = void (*)(RunArgs);

static RunKernel run_kernel(int nets, int form) {
  if (form == kPeriod)
    return nets == kOne ? k_run<kOne, kPeriod> : (nets == kSeveral ? k_run<kSeveral, kPeriod> : k_run<kTables, kPeriod>);
  return nets == kOne ? k_run<kOne, kAhead> : (nets == kSeveral ? k_run<kSeveral, kAhead> : k_run<kTables, kAhead>);
}

cudaError_t prepare_run_kernels() {
  for (int nets : {kOne, kSeveral, kTables})
    for (int form : {kAhead, kPeriod}) {
      cudaError_t e = cudaFuncSetAttribute(run_kernel(nets, form), cudaFuncAttributeMaxDynamicSharedMemorySize,
                                           (int)run_smem_budget());
      if (e != cudaSuccess) return e;
    }
  return cudaSuccess;
}

// One block per SM, or per tile where there are fewer tiles; 640 threads (96
// registers, no spills; 1024: 4-10% more time a step from 4x4 to 40x40 modules,
// 512: 8% more from 16x16 on) but fewer for a few tiles, where the block barriers
// cost more than further warps give.  The form fits as long as the state and `kmin` drives per
// neuron stay in shared memory (2.35M neurons at kmin = 1); what does not fit
// takes two kernels per step (64x64 modules: 80 us a step, against 125 and 217 us
// in two forms of this kernel with the state in global memory).
// `part`: a set that has too many drives for its whole exchange period keeps
// those of up to 16 steps and 1024 live spikes at least, and the grid meets
// within the period.  us a step of all networks, as two kernels side by side and
// so: four of 8x8 modules with smallest delay 100 15.6 and 3.2, eight of 4x4 with
// 254 24 and 2.4, six of 16x16 with 100 25 and 16.  Room for four steps' drives is
// the line: two of 22x22 with 20 (five) 17.1 and 16.0, two of 20x20 (six) 16.1 and
// 16.1, but two of 24x24 with 10 (three) 20.6 and 28, two of 28x28 (two) 25 and 33.
RunShape run_shape(uint32_t n_tiles, uint32_t kmin, int max_threads, uint32_t n_nets, bool part) {
  RunShape sh;
  const uint32_t sms = (uint32_t)std::max(1, device_sm_count());
  sh.blocks = (int)std::max(1u, std::min(sms, n_tiles));
  sh.nt = (n_tiles + (uint32_t)sh.blocks - 1u) / (uint32_t)sh.blocks;
  sh.threads = sh.nt <= 4u ? 256 : (sh.nt <= 12u ? 512 : kRunThreads);
  sh.threads = std::min(sh.threads, std::max(64, max_threads));
  sh.form = kmin > 1u ? kPeriod : kAhead;
  sh.visit = sh.form == kAhead ? kMaxVisit : 1u;
  const size_t budget = run_smem_budget();
  sh.fifo = 512u;
  // Drives a step further ahead where they fit: the neurons with several external events are then completed beside
  // the visits instead of behind a block barrier.
  sh.drives = sh.form == kPeriod ? kmin : (run_smem(2u, sh.nt, sh.visit * sh.fifo) <= budget ? 2u : 1u);
  if (part && sh.form == kPeriod && run_smem(kmin, sh.nt, sh.fifo) > budget) {
    sh.fifo = 1024u;
    sh.drives = std::min(kmin, 16u);
    while (sh.drives > 4u && run_smem(sh.drives, sh.nt, sh.fifo) > budget) --sh.drives;
  }
  const size_t tables = n_nets > 1u ? n_nets * (sizeof(NetDev) + sizeof(NetWin)) : 0u;
  sh.tables = tables && run_smem(sh.drives, sh.nt, sh.visit * sh.fifo) + tables <= budget ? n_nets : 0u;
  const size_t fixed = sh.tables ? tables : 0u;
  while (sh.fifo < 8192u / sh.visit && run_smem(sh.drives, sh.nt, sh.visit * sh.fifo * 2u) + fixed <= budget)
    sh.fifo *= 2u;
  sh.smem = run_smem(sh.drives, sh.nt, sh.visit * sh.fifo) + fixed;
  if (sh.smem > budget || n_tiles > kRunMaxTiles) sh.blocks = 0;   // too many tiles per block, or in all
  return sh;
}

cudaError_t launch_run(const RunArgs &args, const RunShape &sh, const L2Window &l2, cudaStream_t s) {
  if (sh.blocks < 1) return cudaErrorInvalidValue;
  RunArgs a = args;
  a.pre = 64u * (sh.form == kAhead ? sh.visit + 1u : 4u);
  a.fifo = sh.fifo;
  a.nt = sh.nt;
  a.visit = sh.visit;
  a.drives = sh.drives;
  const int nets = a.n_nets < 2u ? kOne : (sh.tables >= a.n_nets ? kTables : kSeveral);
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)sh.blocks);
  cfg.blockDim = dim3((unsigned)sh.threads);
  cfg.dynamicSmemBytes = sh.smem;
  cfg.stream = s;
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeCooperative;   // every block resident: the grid barrier can be met
  attr[0].val.cooperative = 1;
  unsigned n = 1;
  if (l2.bytes) {
    attr[n].id = cudaLaunchAttributeAccessPolicyWindow;
    attr[n].val.accessPolicyWindow.base_ptr = l2.base;
    attr[n].val.accessPolicyWindow.num_bytes = l2.bytes;
    attr[n].val.accessPolicyWindow.hitRatio = l2.hit_ratio;
    attr[n].val.accessPolicyWindow.hitProp = cudaAccessPropertyPersisting;
    attr[n].val.accessPolicyWindow.missProp = cudaAccessPropertyStreaming;
    ++n;
  }
  cfg.attrs = attr;
  cfg.numAttrs = n;
  return cudaLaunchKernelEx(&cfg, run_kernel(nets, sh.form), a);
}

}  // namespace snn

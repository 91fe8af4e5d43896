// snn_kernels.cu -- sm_103a kernels of the DPSNN-style grid simulation.
//
// Arithmetic contract (identical on every path, no FMA contraction: the
// dynamics use explicit __fmul_rn/__fadd_rn and the file is built with
// -fmad=false):
//   Eq. 2 over one step for neuron n at step t:
//     I  = synaptic input of step t (int32, 2^-16 mV), cleared once read
//     w  = word (n mod 4) of Philox4x32-10(key = seed, ctr = (n div 4, t, 1, 0))
//     k  = #{j < 16 : (w >> 12) >= thr[pop][j]}     (Poisson count, Sec. 2.1)
//     I += amp[pop][z_e] for the k external events: z_0 = w & 0xFFF, z_e (e >= 1)
//          = top 12 bits of half (e-1) mod 8 of Philox(seed, (n, t, 3, (e-1) div 8))
//     ref > 0 : ref -= 1, V = V_r                    (refractory clamp, Sec. 2.2)
//     else    : V = (E + (P_VV*(V-E) + P_Vc*c)) + I*2^-16; spike if V > V_th
//     c = P_cc*c (+ alpha when the neuron fired)
//   Delivery (Sec. 2.1.1): a spike of source s at step t reaches the target of
//   each record (d, target, w) of s's row at step t + d: the record's
//   fixed-point weight is added to the target's input of step t + d (int32
//   reductions, so the sum does not depend on order).
//
// Delay-major delivery.  A row is stored grouped by delay (Sec. 2.1), with the
// end of each delay group in a small table (offs).  Delays run from kmin to
// n_delay.  A delivery pass follows every kmin-th step t (the paper's exchange
// step equals the minimum delay): it produces the inputs of steps t + 1 ..
// t + kmin, for each of them adding, for d = kmin..n_delay, the delay-d group
// of every spike of step T - d.  Every record handled lands in one of the
// next kmin steps, so the input needs only kmin + 1 int32 buffers per neuron
// (the one being read is never written); 2 kmin are kept, so that windows
// starting at the same step mod 2 kmin share one captured graph, instead of a
// ring of n_delay + 1 slots.  They stay in L2.  The spikes of the last
// n_delay + kmin steps are kept per step slot in `hist`.
#include <algorithm>
#include <cstdint>

#include "snn_device.cuh"
#include "snn_internal.h"

namespace snn {

// State of 4 consecutive neurons n0..n0+3 (n0 % 4 == 0, n0 < N_pad).
struct Group4 {
  float4 V, c;
  uint32_t ref;   // 4 x u8
  int4 I;         // synaptic input of the step
};

__device__ __forceinline__ void load_state4(const NetDev &nd, uint32_t n0, Group4 &g) {
  const uint32_t i4 = n0 >> 2;
  g.V = ld_cg_f4(reinterpret_cast<const float4 *>(nd.V) + i4);
  g.c = ld_cg_f4(reinterpret_cast<const float4 *>(nd.c) + i4);
  g.ref = ld_cg_u32(reinterpret_cast<const uint32_t *>(nd.ref) + i4);
}

// Input buffer of the step (buffer `buf` = t % nbuf).  It is cleared by integrate4
// after the neuron state is stored: a store right behind the load to the same
// address held every later load of the warp back.
__device__ __forceinline__ void load_input4(const NetDev &nd, uint32_t n0, uint32_t buf, Group4 &g) {
  g.I = ld_cg_i4(reinterpret_cast<const int4 *>(nd.acc + (size_t)buf * nd.N_pad) + (n0 >> 2));
}

// External drive of 4 neurons at step t: adds the drive to I and the number of
// external events of the live neurons to n_ext.  Reads only the parameters and
// the amplitude table.
__device__ __forceinline__ void drive4(const NetDev &nd, uint32_t n0, uint32_t t, int p0, int p1, int32_t (&I)[4],
                                       uint32_t &n_ext) {
  uint32_t kx[4];
  const int4 E = first_drive(nd, n0, t, p0, p1, kx);
  I[0] += E.x;
  I[1] += E.y;
  I[2] += E.z;
  I[3] += E.w;
  extra_events_warp(nd, n0, t, kx, I);
  if (n0 < nd.N) n_ext += kx[0] + kx[1];
  if (n0 + 2u < nd.N) n_ext += kx[2] + kx[3];
}

// Advance the 4 neurons of g by one step (Eq. 2) with total input I (the
// external drive plus the buffer g.I), store the state and clear input buffer
// `buf`; returns the 4-bit spike mask.  Integer input: the order in which the
// drive and the buffer are summed does not change the result.
__device__ __forceinline__ uint32_t integrate4(const NetDev &nd, uint32_t n0, uint32_t buf, int p0, int p1, Group4 &g,
                                               const int32_t (&I)[4]) {
  const uint32_t mask =
      run_step4(nd, n0, p0, p1, g.V, g.c, g.ref, make_int4(I[0] + g.I.x, I[1] + g.I.y, I[2] + g.I.z, I[3] + g.I.w));
  if (n0 < nd.N) {
    const uint32_t i4 = n0 >> 2;
    reinterpret_cast<float4 *>(nd.V)[i4] = g.V;
    reinterpret_cast<float4 *>(nd.c)[i4] = g.c;
    reinterpret_cast<uint32_t *>(nd.ref)[i4] = g.ref;
    if (g.I.x | g.I.y | g.I.z | g.I.w)
      reinterpret_cast<int4 *>(nd.acc + (size_t)buf * nd.N_pad)[i4] = make_int4(0, 0, 0, 0);
  }
  return mask;
}

// Slot (t mod D) of step t = t0 + k from the window's residue and the step's,
// without a division.
__device__ __forceinline__ uint32_t step_slot(const NetDev &nd, const NetWin &w, StepMod km) {
  const uint32_t tm = w.t0_slot + km.slot;
  return tm >= nd.D ? tm - nd.D : tm;
}

// Warp-level recording of the warp's spikes over G groups (all 32 lanes
// active; in group g lane L owns neurons n0[g]..n0[g]+3, and the warp's 32
// lanes cover one aligned 128-neuron tile).  Appends raster entries and the
// step's spike list (`hist`) with one returning atomic each per warp, counts
// rates with fire-and-forget reductions, adds each tile's external events to
// that tile's slot and prefetches into L2 the delay-group table and the first
// records of every spiking neuron's row.
template <int G>
__device__ __forceinline__ void record_warp(const NetDev &nd, const uint32_t (&mask)[G], const uint32_t (&n0)[G],
                                            const uint32_t (&n_ext)[G], uint32_t t, uint32_t slot, uint32_t k,
                                            uint32_t bin0) {
  const uint32_t lane = lane_id();
  const uint32_t lt = (1u << lane) - 1u;
  uint32_t before[G], wtot = 0;
#pragma unroll
  for (int g = 0; g < G; ++g) {
    before[g] = wtot;
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const uint32_t b = __ballot_sync(0xFFFFFFFFu, (mask[g] >> q) & 1u);
      before[g] += __popc(b & lt);
      wtot += __popc(b);
    }
    uint32_t ext = n_ext[g];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) ext += __shfl_xor_sync(0xFFFFFFFFu, ext, o);
    const uint32_t tile = __shfl_sync(0xFFFFFFFFu, n0[g], 0) >> 7;
    if (lane == 0 && ext) red_add_u64(nd.ext_acc + tile, ext);   // slot owned by this warp
  }
  if (wtot == 0) return;
  uint32_t gbase = 0, hbase = 0;
  if (lane == 0) {
    gbase = atomicAdd(&nd.rec->cursor, wtot);
    hbase = atomicAdd(nd.cnt + slot, wtot);
  }
  gbase = __shfl_sync(0xFFFFFFFFu, gbase, 0);
  hbase = __shfl_sync(0xFFFFFFFFu, hbase, 0);
  if (lane == 0 && gbase + wtot > nd.rec_cap) atomicOr(&nd.rec->status, kStatusRasterOverflow);
  const unsigned long long tag = ((unsigned long long)nd.slot << 48) | ((unsigned long long)k << 32);
  const uint32_t bin = t / nd.bin_steps - bin0;
  const uint32_t wb = nd.fmt ? 2u : 4u;
  const uint32_t pre_keys = min(256u, nd.M_pad * 4u), pre_w = min(256u, nd.M_pad * wb);
  uint32_t *hist = nd.hist + (size_t)slot * nd.N_pad;
#pragma unroll
  for (int g = 0; g < G; ++g) {
    uint32_t pos = before[g];
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      if ((mask[g] >> q) & 1u) {
        const uint32_t id = n0[g] + q;
        // the delivery reads this row's delay groups over the next steps
        const uint8_t *row = nd.rows + (size_t)id * nd.row_bytes;
        bulk_prefetch_l2(nd.offs + (size_t)id * nd.os, nd.os * 2u);
        bulk_prefetch_l2(row, pre_keys);
        bulk_prefetch_l2(row + (size_t)nd.M_pad * 4u, pre_w);
        if (gbase + pos < nd.rec_cap) nd.rec_entries[gbase + pos] = tag | id;
        hist[hbase + pos] = id;
        const uint32_t m = id / (uint32_t)kK;
        red_add_u32(nd.rates + ((size_t)bin * nd.G + m) * 3u + pop_of_local(id - m * (uint32_t)kK), 1u);
        ++pos;
      }
    }
  }
}

// The counts of the slots the next kmin steps append to (none of them read by
// the pass after step t).
__device__ __forceinline__ void clear_next_counts(const NetDev &nd, uint32_t t) {
  for (uint32_t i = threadIdx.x; i < nd.kmin; i += blockDim.x) nd.cnt[(t + 1u + i) % nd.D] = 0u;
}

// Target step T = t + 1 + j of the pass after step t: its slot T mod D and its
// input buffer T mod nbuf, from tm = t mod D and tb = t mod nbuf (j < kmin < D,
// kmin < nbuf = 2 kmin: one wrap at most).
__device__ __forceinline__ void target_of(const NetDev &nd, uint32_t tm, uint32_t tb, uint32_t j, uint32_t &Tm,
                                          int32_t *&acc_T) {
  Tm = tm + 1u + j;
  Tm = Tm >= nd.D ? Tm - nd.D : Tm;
  uint32_t b = tb + 1u + j;
  b = b >= nd.nbuf ? b - nd.nbuf : b;
  acc_T = nd.acc + (size_t)b * nd.N_pad;
}

// ---------------------------------------------------------------------------
// Kernel: initial state (V uniform on [0, V_th) from Philox stream 2).
// ---------------------------------------------------------------------------
__global__ void k_init_state(const __grid_constant__ NetDev nd) {
  const uint32_t n = blockIdx.x * blockDim.x + threadIdx.x;
  if (n >= nd.N_pad) return;
  float v = 0.0f;
  if (n < nd.N) {
    const uint4 r = philox4x32_10(n, 0u, 2u, 0u, nd.key0, nd.key1);
    const float u = __fmul_rn(__uint2float_rn(r.x >> 8), 1.0f / 16777216.0f);
    v = __fmul_rn(nd.vth[pop_of_local(n % (uint32_t)kK)], u);
  }
  nd.V[n] = v;
  nd.c[n] = 0.0f;
  nd.ref[n] = 0;
}

// ---------------------------------------------------------------------------
// Kernel: synapse rows (Eq. 1 module choice, uniform target within the module,
// uniform delay, Gaussian efficacy), each row ordered by key (delay << 24 |
// target), records with equal keys in draw order: grouped by delay and sorted
// by target within a delay, so that the lanes of one delivery instruction
// often update the same 32-byte sector of the input buffer.
// Grid (G, y): block (m, y) builds rows of module m, `rows` of them.  One warp
// per row at a time.
//
// Sorting uses that the draws are uniform by construction: with F = the value of
// the module's cumulative threshold interval at lt / 1250 of its width (lt =
// target within the module), (delay, F) grows with the key and is uniform, so a
// monotone map of it to 512 buckets leaves 2.2 draws to a bucket.  Draws are
// counted per bucket, placed in any order, and each finds its rank among the few
// of its bucket by (key, draw index).  The bucket ends are the delay groups.
//
// Bound by instruction issue (0.6 per cycle) at the 16 warps that their 12 KB each
// leave per SM; the rows written are 6% of the HBM rate.  24x24 modules, packed
// records: 20.8 ms with a 4-pass radix sort by match and a binary search over the
// modules, 16.6 ms with three passes and a guide table (the match instructions
// alone kept their pipe busy 68% of the time), 11.8 ms here (1024 buckets, 15
// warps: 12.1 ms; 2048, 13 warps: 14.1 ms).
// ---------------------------------------------------------------------------
constexpr int kBuildWarpsMax = 16;
constexpr uint32_t kGuideBits = 10;      // guide to the module thresholds
constexpr uint32_t kBuckets = 512;       // per row, at least 254 delays

// Shared memory of one building warp: keys (u32), bucket counters (u16 pairs),
// then quantile indices, buckets and a permutation (u16), rounded up to 16 bytes.
__host__ __device__ inline uint32_t build_warp_bytes(uint32_t M_pad) {
  return (M_pad * 10u + kBuckets * 2u + 15u) & ~15u;
}

// Bytes of shared memory before the staged CDF: the quantile table, the
// efficacy means and spreads (s_js[0] = J, s_js[1] = sigma, [target][source])
// and the guide.
constexpr uint32_t kGuideBytes = (((1u << kGuideBits) + 1u) * 2u + 15u) & ~15u;
constexpr uint32_t kBuildTableBytes = kZTab * 4u + 128u + kGuideBytes;

// Efficacy of a synapse from a population-sp source on population tp with
// quantile index z: J + sigma * z-quantile, clamped so it keeps J's sign.
__device__ __forceinline__ float synapse_weight(const float *s_js, const float *s_z, int sp, uint32_t tp, uint32_t z) {
  const float J = s_js[tp * kNPop + sp];
  float w = __fadd_rn(J, __fmul_rn(s_js[kNPop * kNPop + tp * kNPop + sp], s_z[z]));
  if (J > 0.0f && w < 0.0f) w = 0.0f;
  if (J < 0.0f && w > 0.0f) w = 0.0f;
  return w;
}

__global__ void __launch_bounds__(kBuildWarpsMax * 32) k_build_rows(const __grid_constant__ NetDev nd,
                                                                  const __grid_constant__ BuildDev bd, uint32_t rows,
                                                                  uint32_t cdf_in_smem) {
  extern __shared__ __align__(128) uint8_t smem[];
  float *s_z = reinterpret_cast<float *>(smem);                       // kZTab
  float *s_js = s_z + kZTab;                                          // J, sigma
  uint16_t *s_guide = reinterpret_cast<uint16_t *>(smem + kZTab * 4u + 128u);
  uint32_t *s_cdf = reinterpret_cast<uint32_t *>(smem + kBuildTableBytes);   // G-1 (if staged)
  const uint32_t Gm1 = nd.G - 1u;
  const uint32_t cdf_words = cdf_in_smem ? ((Gm1 + 3u) & ~3u) : 0u;
  uint8_t *warp_base = reinterpret_cast<uint8_t *>(s_cdf + cdf_words);
  const uint32_t warp = threadIdx.x >> 5, lane = lane_id();
  const uint32_t per_warp = build_warp_bytes(nd.M_pad);
  uint32_t *w_key = reinterpret_cast<uint32_t *>(warp_base + (size_t)warp * per_warp);
  uint32_t *w_cnt = w_key + nd.M_pad;                                  // kBuckets counters, two per word
  uint16_t *w_z = reinterpret_cast<uint16_t *>(w_cnt + kBuckets / 2u);   // quantile index | population << 12
  uint16_t *w_b = w_z + nd.M_pad;                                       // bucket
  uint16_t *w_perm = w_b + nd.M_pad;                                    // draws by bucket

  const uint32_t m = blockIdx.x;
  for (uint32_t i = threadIdx.x; i < (uint32_t)kZTab; i += blockDim.x) s_z[i] = bd.ztab[i];
  if (threadIdx.x < (uint32_t)(kNPop * kNPop)) {
    s_js[threadIdx.x] = bd.J[threadIdx.x / kNPop][threadIdx.x % kNPop];
    s_js[kNPop * kNPop + threadIdx.x] = bd.sig[threadIdx.x / kNPop][threadIdx.x % kNPop];
  }
  const uint32_t *cdf_row = bd.cdf + (size_t)m * Gm1;
  if (cdf_in_smem)
    for (uint32_t i = threadIdx.x; i < Gm1; i += blockDim.x) s_cdf[i] = cdf_row[i];
  __syncthreads();
  const uint32_t *T = cdf_in_smem ? s_cdf : cdf_row;
  // guide[h]: thresholds at or below h 2^22; a draw u with u >> 22 = h has between guide[h] and guide[h + 1] of them
  for (uint32_t h = threadIdx.x; h <= (1u << kGuideBits); h += blockDim.x) {
    uint32_t lo = 0, hi = Gm1;
    if (h == (1u << kGuideBits)) lo = Gm1;
    const uint32_t at = h << (32u - kGuideBits);
    while (lo < hi) {
      const uint32_t mid = (lo + hi) >> 1;
      if (at < T[mid]) hi = mid; else lo = mid + 1u;
    }
    s_guide[h] = (uint16_t)lo;
  }
  // the source module's own draws: lo_loc <= u < T[m] (no bound above for the last module)
  const uint32_t lo_loc = m == 0u ? 0u : T[m - 1u];
  const uint32_t w_loc = m == Gm1 ? 0xFFFFFFFFu - lo_loc : T[m] - lo_loc;   // one short for the last module:
                                                                            // the search finds it too
  __syncthreads();

  const uint32_t M = nd.M, Mp = nd.M_pad, n_del = bd.n_delay - bd.min_delay + 1u;
  const uint32_t per_delay = kBuckets / n_del;   // buckets of one delay
  const uint32_t n_warps = blockDim.x >> 5;
  const uint32_t l_end = min((uint32_t)kK, (blockIdx.y + 1u) * rows);
  auto bucket_end = [&](uint32_t b) { return (w_cnt[b >> 1] >> (16u * (b & 1u))) & 0xFFFFu; };   // once placed
  for (uint32_t l = blockIdx.y * rows + warp; l < l_end; l += n_warps) {
    const uint32_t s = m * (uint32_t)kK + l;
    const int sp = pop_of_local(l);
    for (uint32_t i = lane; i < kBuckets / 2u; i += 32u) w_cnt[i] = 0u;
    __syncwarp();
    // 1. draw the M synapses of row s, four per lane at a time
    for (uint32_t j0 = 0; j0 < M; j0 += 128u) {
      uint4 r[4];
      uint32_t lo[4], hi[4];
#pragma unroll
      for (uint32_t u = 0; u < 4u; ++u) {
        const uint32_t j = j0 + 32u * u + lane;
        r[u] = philox4x32_10(s, j, 0u, 0u, nd.key0, nd.key1);
        const bool local = sp == 2 || r[u].x - lo_loc < w_loc;
        lo[u] = hi[u] = m;
        if (!local && j < M) {
          const uint32_t h = r[u].x >> (32u - kGuideBits);
          lo[u] = s_guide[h];
          hi[u] = s_guide[h + 1u];
        }
      }
      while (true) {
        bool more = false;
#pragma unroll
        for (uint32_t u = 0; u < 4u; ++u) {
          if (lo[u] < hi[u]) {
            const uint32_t mid = (lo[u] + hi[u]) >> 1;
            if (r[u].x < T[mid]) hi[u] = mid; else lo[u] = mid + 1u;
          }
          more |= lo[u] < hi[u];
        }
        if (!__any_sync(0xFFFFFFFFu, more)) break;
      }
#pragma unroll
      for (uint32_t u = 0; u < 4u; ++u) {
        const uint32_t j = j0 + 32u * u + lane;
        if (j < M) {
          const uint32_t mt = lo[u], lt = __umulhi(r[u].y, (uint32_t)kK), d = __umulhi(r[u].z, n_del);
          // thresholds below and above the module (inhibitory rows: their module is the whole interval)
          const uint32_t t0 = sp == 2 || mt == 0u ? 0u : T[mt - 1u];
          const uint32_t t1 = sp == 2 || mt == Gm1 ? 0xFFFFFFFFu : T[mt];
          const uint32_t F = t0 + __umulhi(t1 - t0, lt * 3435973u);   // 3435973 = floor(2^32 / 1250)
          const uint32_t b = d * per_delay + __umulhi(F, per_delay);
          w_key[j] = ((d + bd.min_delay) << 24) | (mt * (uint32_t)kK + lt);
          w_z[j] = (uint16_t)((r[u].w >> 20) | ((uint32_t)pop_of_local(lt) << 12));
          w_b[j] = (uint16_t)b;
          atomicAdd(&w_cnt[b >> 1], 1u << (16u * (b & 1u)));
        }
      }
    }
    __syncwarp();
    // 2. starts of the buckets: exclusive scan of the counts, two per word
    {
      constexpr uint32_t W = kBuckets / 64u;   // words per lane
      uint4 v[W / 4u];
      uint32_t sum = 0;
#pragma unroll
      for (uint32_t q = 0; q < W / 4u; ++q) {
        v[q] = reinterpret_cast<const uint4 *>(w_cnt)[lane * (W / 4u) + q];
        sum += v[q].x + v[q].y + v[q].z + v[q].w;   // both halves at once: neither carries (at most M)
      }
      sum = (sum & 0xFFFFu) + (sum >> 16);
      uint32_t incl = sum;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const uint32_t y = __shfl_up_sync(0xFFFFFFFFu, incl, o);
        if (lane >= (uint32_t)o) incl += y;
      }
      uint32_t run = incl - sum;
      auto start = [&](uint32_t &x) {
        const uint32_t low = x & 0xFFFFu, high = x >> 16;
        x = run | ((run + low) << 16);
        run += low + high;
      };
#pragma unroll
      for (uint32_t q = 0; q < W / 4u; ++q) {
        start(v[q].x);
        start(v[q].y);
        start(v[q].z);
        start(v[q].w);
        reinterpret_cast<uint4 *>(w_cnt)[lane * (W / 4u) + q] = v[q];
      }
    }
    __syncwarp();
    // 3. place the draws, those of a bucket in any order; the counters end at the buckets' ends
    for (uint32_t j = lane; j < M; j += 32u) {
      const uint32_t b = w_b[j], sh = 16u * (b & 1u);
      w_perm[(atomicAdd(&w_cnt[b >> 1], 1u << sh) >> sh) & 0xFFFFu] = (uint16_t)j;
    }
    __syncwarp();
    // 4. write the row, each record at its rank within its bucket; padding records zero
    uint8_t *row = nd.rows + (size_t)s * nd.row_bytes;
    uint32_t *okey = reinterpret_cast<uint32_t *>(row);
    uint8_t *ow = row + (size_t)Mp * 4u;
    for (uint32_t p = lane; p < Mp; p += 32u) {
      uint32_t key = 0u, at = p;
      float w = 0.0f;
      if (p < M) {
        const uint32_t j = w_perm[p], b = w_b[j], z = w_z[j];
        key = w_key[j];
        at = b ? bucket_end(b - 1u) : 0u;
        for (uint32_t q = at, end = bucket_end(b); q < end; ++q) {
          const uint32_t i = w_perm[q], k = w_key[i];
          at += (k < key || (k == key && i < j)) ? 1u : 0u;
        }
        w = synapse_weight(s_js, s_z, sp, z >> 12, z & 0xFFFu);
      }
      okey[at] = key;
      if (nd.fmt) {
        int q = __float2int_rn(__fmul_rn(w, 1024.0f));
        q = q > 32767 ? 32767 : (q < -32768 ? -32768 : q);
        reinterpret_cast<int16_t *>(ow)[at] = (int16_t)q;
      } else {
        reinterpret_cast<float *>(ow)[at] = w;
      }
    }
    // 5. delay groups of the row: records with delay <= d end at offs[d]
    if (nd.offs) {
      uint16_t *orow = const_cast<uint16_t *>(nd.offs) + (size_t)s * nd.os;
      for (uint32_t d = lane; d < nd.os; d += 32u)
        orow[d] = (uint16_t)(d < bd.min_delay ? 0u
                                              : (d < bd.n_delay ? bucket_end((d - bd.min_delay + 1u) * per_delay - 1u) : M));
    }
    __syncwarp();
  }
}

// ---------------------------------------------------------------------------
// Kernel: neuron update + recording (two-kernel path).  No block barrier:
// spikes are appended per warp.
// ---------------------------------------------------------------------------
// Each thread advances G groups of 4 neurons; group g of block b covers the
// neuron range ((b * G + g) * BLOCK + thread) * 4, so every warp owns whole
// aligned 128-neuron tiles.
// The neuron state is final when the kernel starts: either the kernel before
// it has finished, or (km.overlapped) it is a delivery pass launched after the
// previous update, which it waited for before letting this kernel start.  The
// state loads are issued first, then the external drive (which reads no state)
// is computed; without overlap the input buffer is loaded with the state, with
// it only after griddepcontrol.wait (the pass writes that buffer).  The trigger
// that follows the wait lets the delivery pass after this step start on older
// spikes.
// One group per thread is capped at 48 registers (40 resident warps per SM), so
// that a 720k-neuron grid (37 warps per SM) runs in a single wave; at 5.12M
// neurons 64 registers and 32 warps take the same 34.6 us, 40 registers and 48
// warps 40.7.  There the state and inputs (133 MB a step, about the size of L2)
// bound it; the branchless step with two parameter loads per pair of neurons
// brought it from 39.2 us (a loop over the thresholds and seven parameter loads
// per neuron).
template <int BLOCK, int G>
__global__ void __launch_bounds__(BLOCK, G == 1 ? 1280 / BLOCK : 1) k_update(const __grid_constant__ NetDev nd,
                                                                           uint32_t k, StepMod km) {
  uint32_t n0[G];
  bool live[G];
  bool any = false;
#pragma unroll
  for (int g = 0; g < G; ++g) {
    const uint32_t tile0 = ((blockIdx.x * G + g) * BLOCK + (threadIdx.x & ~31u)) * 4u;
    n0[g] = ((blockIdx.x * G + g) * BLOCK + threadIdx.x) * 4u;
    live[g] = tile0 < nd.N_pad;     // whole warps: N_pad is a multiple of 128
    any |= live[g];
  }
  if (!any) return;
  const NetWin w = *nd.win;   // written before the window's first kernel
  const uint32_t t = w.t0 + k;
  if (t >= w.t_end) return;
  Group4 st4[G];
#pragma unroll
  for (int g = 0; g < G; ++g)
    if (live[g]) {
      load_state4(nd, n0[g], st4[g]);
      if (!km.overlapped) load_input4(nd, n0[g], km.buf, st4[g]);
    }
  int32_t I[G][4];
  int p0[G], p1[G];
  uint32_t n_ext[G];
#pragma unroll
  for (int g = 0; g < G; ++g) {
    I[g][0] = I[g][1] = I[g][2] = I[g][3] = 0;
    n_ext[g] = 0;
    if (live[g]) {
      pair_pops(n0[g], p0[g], p1[g]);
      drive4(nd, n0[g], t, p0[g], p1[g], I[g], n_ext[g]);
    }
  }
  pdl_wait();      // the previous kernel (and everything before it) is complete
  pdl_trigger();
  const uint32_t slot = step_slot(nd, w, km), buf = km.buf;
  uint32_t mask[G];
#pragma unroll
  for (int g = 0; g < G; ++g) {
    mask[g] = 0;
    if (live[g] && km.overlapped) load_input4(nd, n0[g], buf, st4[g]);
  }
#pragma unroll
  for (int g = 0; g < G; ++g)
    if (live[g]) mask[g] = integrate4(nd, n0[g], buf, p0[g], p1[g], st4[g], I[g]);
  // record per group whose tile is live (warp-uniform)
  if (live[G - 1]) {
    record_warp<G>(nd, mask, n0, n_ext, t, slot, k, w.bin0);
  } else {
#pragma unroll
    for (int g = 0; g < G; ++g) {
      if (live[g]) {
        const uint32_t m1[1] = {mask[g]}, a1[1] = {n0[g]}, e1[1] = {n_ext[g]};
        record_warp<1>(nd, m1, a1, e1, t, slot, k, w.bin0);
      }
    }
  }
}

// ---------------------------------------------------------------------------
// Kernel: delivery pass after step t (two-kernel path).  Every warp takes
// segments of every target step of the pass.  Launched with programmatic
// dependent launch after the update of step t: the segments of older spikes
// (steps before t, complete before that update started) are delivered first,
// while the update may still run; after griddepcontrol.wait the step's own
// spikes (their delay-kmin group, into the input of step t + kmin).  The
// trigger after the wait lets the next update load its state and compute its
// drive while the pass finishes.
// ---------------------------------------------------------------------------
// One prefix chunk (n_delay <= 32) fits in 40 registers: three 512-thread
// blocks per SM.
template <int NCH>
__global__ void __launch_bounds__(512, NCH == 1 ? 3 : 2) k_deliver(const __grid_constant__ NetDev nd, uint32_t k, StepMod km,
                                                  uint32_t lanes) {
  const NetWin w = *nd.win;   // written before the window's first kernel
  const uint32_t t = w.t0 + k;
  if (t >= w.t_end) return;
  const uint32_t warp = threadIdx.x >> 5, lane = lane_id();
  const uint32_t gpw = 32u / lanes, grp = lane / lanes, sub = lane % lanes;
  const uint32_t nwarps = gridDim.x * (blockDim.x >> 5);
  const uint32_t gw = blockIdx.x * (blockDim.x >> 5) + warp;
  const uint32_t first = gw * gpw + grp, stride = nwarps * gpw;
  const uint32_t tm = step_slot(nd, w, km), tb = km.buf;
  for (uint32_t j = 0; j < nd.kmin; ++j) {
    uint32_t Tm;
    int32_t *acc_T;
    target_of(nd, tm, tb, j, Tm, acc_T);
    WarpPrefix<NCH> P;   // each warp its own prefix, in registers
    warp_prefix<NCH>(nd, P, Tm, j, true);
    deliver_segments<NCH>(nd, P, Tm, acc_T, gw * gpw, stride, lanes);
  }
  pdl_wait();       // the update of step t is complete: its spike list is final
  pdl_trigger();
  {
    const uint32_t kmin = nd.kmin;
    uint32_t Tm;
    int32_t *acc_T;
    target_of(nd, tm, tb, kmin - 1u, Tm, acc_T);
    const uint32_t *ids = nd.hist + (size_t)tm * nd.N_pad;
    // the list's first entry of this group is loaded together with the count
    // (entries past the count are stale ids, in bounds and unused)
    const uint32_t s0 = first < nd.N_pad ? ld_cg_u32(ids + first) : 0u;
    const uint32_t n = ld_cg_u32(nd.cnt + tm);
    for (uint32_t i = first; i < n; i += stride) {
      const uint32_t s = i == first ? s0 : ld_cg_u32(ids + i);
      const uint16_t *o = nd.offs + (size_t)s * nd.os;
      const uint32_t a = o[kmin - 1u], b = o[kmin];
      if (sub == 0) prefetch_next_group(nd, s, o, kmin, b);
      add_records(nd, acc_T, s, a, b, sub, lanes);
    }
  }
  if (blockIdx.x == 0) clear_next_counts(nd, t);
}

// ---------------------------------------------------------------------------
// Launchers
// ---------------------------------------------------------------------------
int device_sm_count() {
  int dev = 0, sms = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) return 0;
  if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) return 0;
  return sms;
}

static bool valid_lanes(uint32_t lanes) { return lanes == 4 || lanes == 8 || lanes == 16 || lanes == 32; }

// Dynamic shared memory of one construction block: the device's opt-in
// maximum per block (227 KB on sm_103), never above 227 KB.
static size_t build_smem_budget() {
  static size_t cached = 0;
  if (cached) return cached;
  int dev = 0, optin = 0;
  size_t b = 200u * 1024u;
  if (cudaGetDevice(&dev) == cudaSuccess &&
      cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev) == cudaSuccess && optin > 0)
    b = std::min<size_t>((size_t)optin, 227u * 1024u);
  cached = b;
  return b;
}

cudaError_t prepare_kernels() {
  return cudaFuncSetAttribute(k_build_rows, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)build_smem_budget());
}

cudaError_t launch_init_state(const NetDev &nd, cudaStream_t s) {
  const uint32_t threads = 256;
  const uint32_t blocks = (nd.N_pad + threads - 1) / threads;
  k_init_state<<<blocks, threads, 0, s>>>(nd);
  return cudaGetLastError();
}

cudaError_t launch_build_rows(const NetDev &h_nd, const BuildDev &bd, cudaStream_t s) {
  const uint32_t Gm1 = h_nd.G - 1u;
  const uint32_t cdf_in_smem = (Gm1 <= 12288u) ? 1u : 0u;
  const size_t per_warp = build_warp_bytes(h_nd.M_pad);
  const size_t fixed = (size_t)kBuildTableBytes + (cdf_in_smem ? (((size_t)Gm1 + 3u) & ~(size_t)3u) * 4u : 0u);
  const size_t budget = build_smem_budget();
  if (fixed + per_warp > budget) return cudaErrorInvalidValue;
  const uint32_t warps = (uint32_t)std::min<size_t>(kBuildWarpsMax, (budget - fixed) / per_warp);
  const size_t smem = fixed + per_warp * (size_t)warps;
  // Rows per block (a multiple of its warps, one block per SM): the fewest
  // rounds of rows over all waves, one round more per block for its tables.
  const uint32_t sms = (uint32_t)std::max(1, device_sm_count());
  uint32_t best = 0xFFFFFFFFu, rows = warps;
  for (uint32_t rounds = 1; rounds <= ((uint32_t)kK + warps - 1u) / warps; ++rounds) {
    const uint32_t y = ((uint32_t)kK + rounds * warps - 1u) / (rounds * warps);
    const unsigned long long waves = ((unsigned long long)h_nd.G * y + sms - 1u) / sms;
    const uint32_t cost = (uint32_t)std::min<unsigned long long>(waves * (rounds + 1u), 0xFFFFFFFEull);
    if (cost < best) {
      best = cost;
      rows = rounds * warps;
    }
  }
  dim3 grid(h_nd.G, ((uint32_t)kK + rows - 1u) / rows);
  k_build_rows<<<grid, warps * 32u, smem, s>>>(h_nd, bd, rows, cdf_in_smem);
  return cudaGetLastError();
}

// Launch with an optional persisting L2 access-policy window.
// Launch with an optional persisting L2 access-policy window and, with `pdl`,
// programmatic stream serialization (the kernel may start once every block of
// the previous kernel has passed griddepcontrol.launch_dependents).
template <typename... Args>
static cudaError_t launch_ex(void (*kernel)(Args...), dim3 grid, dim3 block, size_t smem, const L2Window &l2,
                             bool pdl, cudaStream_t s, Args... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = block;
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cudaLaunchAttribute attr[2];
  unsigned n = 0;
  if (pdl) {
    attr[n].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[n].val.programmaticStreamSerializationAllowed = 1;
    ++n;
  }
  if (l2.bytes) {
    attr[n].id = cudaLaunchAttributeAccessPolicyWindow;
    attr[n].val.accessPolicyWindow.base_ptr = l2.base;
    attr[n].val.accessPolicyWindow.num_bytes = l2.bytes;
    attr[n].val.accessPolicyWindow.hitRatio = l2.hit_ratio;
    attr[n].val.accessPolicyWindow.hitProp = cudaAccessPropertyPersisting;
    attr[n].val.accessPolicyWindow.missProp = cudaAccessPropertyStreaming;
    ++n;
  }
  cfg.attrs = n ? attr : nullptr;
  cfg.numAttrs = n;
  return cudaLaunchKernelEx(&cfg, kernel, args...);
}

cudaError_t launch_update(const NetDev &nd, uint32_t k, StepMod km, int block, int groups, const L2Window &l2,
                          bool pdl, cudaStream_t s) {
  const uint32_t per_block = (uint32_t)block * 4u * (uint32_t)groups;
  const uint32_t blocks = (nd.N_pad + per_block - 1) / per_block;
#define SNN_UPD(B, G) \
  if (block == B && groups == G) return launch_ex(k_update<B, G>, dim3(blocks), dim3(B), 0, l2, pdl, s, nd, k, km);
  SNN_UPD(64, 1) SNN_UPD(128, 1) SNN_UPD(128, 2) SNN_UPD(128, 4)
  SNN_UPD(256, 1) SNN_UPD(256, 2) SNN_UPD(256, 4)
  SNN_UPD(512, 1) SNN_UPD(512, 2)
#undef SNN_UPD
  return cudaErrorInvalidValue;
}

cudaError_t launch_deliver(const NetDev &nd, uint32_t k, StepMod km, uint32_t lanes, int warps, int blocks,
                           const L2Window &l2, bool pdl, cudaStream_t s) {
  if (warps < 1 || warps > 16 || blocks < 1 || !valid_lanes(lanes)) return cudaErrorInvalidValue;
  if (pre_chunks(nd.n_delay) == 1u)
    return launch_ex(k_deliver<1>, dim3((unsigned)blocks), dim3(warps * 32), 0, l2, pdl, s, nd, k, km, lanes);
  if (nd.n_delay <= 32u * kMaxPreChunks)
    return launch_ex(k_deliver<kMaxPreChunks>, dim3((unsigned)blocks), dim3(warps * 32), 0, l2, pdl, s, nd, k, km,
                     lanes);
  return cudaErrorInvalidValue;
}

}  // namespace snn

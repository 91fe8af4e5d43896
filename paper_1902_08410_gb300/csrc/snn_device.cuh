// snn_device.cuh -- device primitives shared by the kernels (snn_kernels.cu,
// snn_run.cu): counter-based draws, memory operations, the neuron update and
// the reduction of synapse records.
#pragma once
#include <cstdint>

#include "snn_internal.h"

namespace snn {

// ---------------------------------------------------------------------------
// Philox4x32-10 (Salmon et al., SC'11): ten rounds, Weyl key schedule.
// ---------------------------------------------------------------------------
__device__ __forceinline__ uint4 philox4x32_10(uint32_t c0, uint32_t c1, uint32_t c2, uint32_t c3,
                                               uint32_t k0, uint32_t k1) {
#pragma unroll
  for (int r = 0; r < 10; ++r) {
    const uint32_t lo0 = 0xD2511F53u * c0;
    const uint32_t hi0 = __umulhi(0xD2511F53u, c0);
    const uint32_t lo1 = 0xCD9E8D57u * c2;
    const uint32_t hi1 = __umulhi(0xCD9E8D57u, c2);
    const uint32_t n0 = hi1 ^ c1 ^ k0;
    const uint32_t n2 = hi0 ^ c3 ^ k1;
    c0 = n0;
    c1 = lo1;
    c2 = n2;
    c3 = lo0;
    k0 += 0x9E3779B9u;
    k1 += 0xBB67AE85u;
  }
  return make_uint4(c0, c1, c2, c3);
}

__device__ __forceinline__ int pop_of_local(uint32_t local) { return local < 250u ? 0 : (local < 1000u ? 1 : 2); }

__device__ __forceinline__ uint32_t lane_id() { return threadIdx.x & 31u; }

// Fire-and-forget prefetch of [src, src + bytes) into L2 (16-byte aligned
// address, size a multiple of 16).
__device__ __forceinline__ void bulk_prefetch_l2(const void *src, uint32_t bytes) {
  asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(src), "r"(bytes) : "memory");
}

// Prefetch the byte range [p, p + bytes) widened to 16-byte boundaries; the
// caller guarantees the widened range lies inside one allocation.
__device__ __forceinline__ void prefetch_range_l2(const uint8_t *p, uint32_t bytes) {
  if (bytes == 0) return;
  const uintptr_t a0 = reinterpret_cast<uintptr_t>(p) & ~uintptr_t(15);
  const uintptr_t a1 = (reinterpret_cast<uintptr_t>(p) + bytes + 15u) & ~uintptr_t(15);
  bulk_prefetch_l2(reinterpret_cast<const void *>(a0), (uint32_t)(a1 - a0));
}

// Programmatic dependent launch: wait for the previous kernel in the stream
// (no-op when launched without the attribute), then let the next one launch.
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void pdl_trigger() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

// ---------------------------------------------------------------------------
// Fire-and-forget global reductions (no value returned, no scoreboard wait).
// ---------------------------------------------------------------------------
__device__ __forceinline__ void red_add_s32(int32_t *addr, int32_t v) {
  asm volatile("red.relaxed.gpu.global.add.s32 [%0], %1;" ::"l"(addr), "r"(v) : "memory");
}
__device__ __forceinline__ void red_add_u32(uint32_t *addr, uint32_t v) {
  asm volatile("red.relaxed.gpu.global.add.u32 [%0], %1;" ::"l"(addr), "r"(v) : "memory");
}
__device__ __forceinline__ void red_add_u64(unsigned long long *addr, unsigned long long v) {
  asm volatile("red.relaxed.gpu.global.add.u64 [%0], %1;" ::"l"(addr), "l"(v) : "memory");
}

// L2-only loads (never served from L1) of data that other kernels of the
// stream write: the neuron state and input buffers, and the spike lists and
// counts, which the update of a step appends to while an overlapping delivery
// pass reads older slots of the same arrays.  L1 stays for the amplitude table.
__device__ __forceinline__ float4 ld_cg_f4(const float4 *p) {
  float4 v;
  asm volatile("ld.global.cg.v4.f32 {%0, %1, %2, %3}, [%4];"
               : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w)
               : "l"(p));
  return v;
}
__device__ __forceinline__ int4 ld_cg_i4(const int4 *p) {
  int4 v;
  asm volatile("ld.global.cg.v4.s32 {%0, %1, %2, %3}, [%4];"
               : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w)
               : "l"(p));
  return v;
}
__device__ __forceinline__ uint32_t ld_cg_u32(const uint32_t *p) {
  uint32_t v;
  asm volatile("ld.global.cg.u32 %0, [%1];" : "=r"(v) : "l"(p));
  return v;
}
// Read-only loads of synapse records, not kept in L1 (each is used once).
// The predicate is inside the instruction, with a value for lanes without it: a
// conditional around a load became a branch that waits for each load before the
// next is issued (6x6 modules, packed records: 5.2 us a step, 4.3 us so; the f32
// loads are as fast either way).
__device__ __forceinline__ uint32_t ld_rec_u32_if(bool on, const uint32_t *p, uint32_t other) {
  uint32_t v;
  asm volatile(
      "{\n\t.reg .pred q;\n\tsetp.ne.u32 q, %2, 0;\n\tmov.b32 %0, %3;\n\t"
      "@q ld.global.nc.L1::no_allocate.u32 %0, [%1];\n\t}"
      : "=&r"(v) : "l"(p), "r"((uint32_t)on), "r"(other));
  return v;
}
__device__ __forceinline__ int32_t ld_rec_s16_if(bool on, const int16_t *p) {
  int32_t v;
  asm volatile(
      "{\n\t.reg .pred q;\n\tsetp.ne.u32 q, %2, 0;\n\tmov.b32 %0, 0;\n\t"
      "@q ld.global.nc.L1::no_allocate.s16 %0, [%1];\n\t}"
      : "=&r"(v) : "l"(p), "r"((uint32_t)on));
  return v;
}

// ---------------------------------------------------------------------------
// Neuron update (Eq. 2 over one step, Poisson drive) of 4 consecutive neurons.
// ---------------------------------------------------------------------------
// Amplitudes of external events e0..k-1 of neuron n at step t (2^-16 mV), one
// Philox draw per 8 events; only the rare tail e0 = 9 comes through here.
static __device__ __noinline__ int32_t extra_amplitudes(const NetDev &nd, int pop, uint32_t e0, uint32_t k, uint32_t n,
                                                 uint32_t t) {
  const int32_t *ap = nd.amp + pop * kZTab;
  int32_t I = 0;
  uint4 q = make_uint4(0, 0, 0, 0);
  for (uint32_t e = e0; e < k; ++e) {
    const uint32_t i = (e - 1u) & 7u;
    if (e == e0 || i == 0) q = philox4x32_10(n, t, 3u, (e - 1u) >> 3, nd.key0, nd.key1);
    const uint32_t w = i >> 1;
    const uint32_t word = (w == 0) ? q.x : ((w == 1) ? q.y : ((w == 2) ? q.z : q.w));
    const uint32_t half = (i & 1u) ? (word >> 16) : (word & 0xFFFFu);
    I += __ldg(ap + (half >> 4));
  }
  return I;
}

// Amplitudes of events 1..k-1 (k >= 2) of neuron n: events 1..8 come from the
// halves of one draw and their table loads are independent.
__device__ __forceinline__ int32_t extra_sum(const NetDev &nd, int pop, uint32_t k, uint32_t n, uint32_t t) {
  const int32_t *ap = nd.amp + pop * kZTab;
  const uint4 R = philox4x32_10(n, t, 3u, 0u, nd.key0, nd.key1);
  const uint32_t h[8] = {R.x & 0xFFFFu, R.x >> 16, R.y & 0xFFFFu, R.y >> 16,
                         R.z & 0xFFFFu, R.z >> 16, R.w & 0xFFFFu, R.w >> 16};
  int32_t I = 0;
#pragma unroll
  for (uint32_t j = 0; j < 8u; ++j)
    if (j + 1u < k) I += __ldg(ap + (h[j] >> 4));
  if (k > 9u) I += extra_amplitudes(nd, pop, 9u, k, n, t);
  return I;
}

// Events 1..k-1 of every neuron of the warp's 128-neuron tile that received
// more than one external event this step (about 1.4% of neurons at 0.18
// expected events).  The pending (lane, q) pairs are numbered q-major by
// ballots and lane i serves pair i, so a warp pays one draw and one table
// round trip instead of one per neuron and event; sums return by shuffle.
// Called by whole warps (all 32 lanes).
__device__ __forceinline__ void extra_events_warp(const NetDev &nd, uint32_t n0, uint32_t t, const uint32_t (&kx)[4],
                                                  int32_t (&Iv)[4]) {
  if (!__any_sync(0xFFFFFFFFu, kx[0] > 1u || kx[1] > 1u || kx[2] > 1u || kx[3] > 1u)) return;   // most warps
  const uint32_t lane = lane_id(), lt = (1u << lane) - 1u;
  uint32_t bal[4], idx[4], cnt[4], total = 0;
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    bal[q] = __ballot_sync(0xFFFFFFFFu, kx[q] > 1u);
    idx[q] = total + __popc(bal[q] & lt);
    cnt[q] = total;
    total += __popc(bal[q]);
  }
  if (total == 0u) return;
  const uint32_t packed = kx[0] | (kx[1] << 8) | (kx[2] << 16) | (kx[3] << 24);   // each count <= 16
  const uint32_t tile0 = n0 - lane * 4u;
  for (uint32_t s = 0; s < total; s += 32u) {
    const uint32_t i = s + lane;
    uint32_t q = 0, owner = 0;
    if (i < total) {
      q = (i >= cnt[1] ? 1u : 0u) + (i >= cnt[2] ? 1u : 0u) + (i >= cnt[3] ? 1u : 0u);
      uint32_t b = (q == 0u) ? bal[0] : ((q == 1u) ? bal[1] : ((q == 2u) ? bal[2] : bal[3]));
      const uint32_t base = (q == 0u) ? 0u : ((q == 1u) ? cnt[1] : ((q == 2u) ? cnt[2] : cnt[3]));
      for (uint32_t r = base; r < i; ++r) b &= b - 1u;   // drop the lower set bits: rank i - base
      owner = (uint32_t)(__ffs(b) - 1);
    }
    const uint32_t pk = __shfl_sync(0xFFFFFFFFu, packed, owner);
    int32_t acc = 0;
    if (i < total) {
      const uint32_t n = tile0 + owner * 4u + q;
      acc = extra_sum(nd, pop_of_local(n % (uint32_t)kK), (pk >> (8u * q)) & 0xFFu, n, t);
    }
#pragma unroll
    for (int qq = 0; qq < 4; ++qq) {
      const int32_t v = __shfl_sync(0xFFFFFFFFu, acc, idx[qq] & 31u);
      if (kx[qq] > 1u && idx[qq] - s < 32u) Iv[qq] += v;
    }
  }
}


// Populations of the pairs (n0, n0 + 1) and (n0 + 2, n0 + 3), n0 % 4 == 0: all
// population and module boundaries (250, 1000, 1250) are even.
__device__ __forceinline__ void pair_pops(uint32_t n0, int &p0, int &p1) {
  const uint32_t l0 = n0 % (uint32_t)kK;
  const uint32_t l1 = (l0 + 2u == (uint32_t)kK) ? 0u : l0 + 2u;
  p0 = pop_of_local(l0);
  p1 = pop_of_local(l1);
}

// Number of thresholds <= u (thresholds ascend), u = w >> 12.
__device__ __forceinline__ uint32_t events_of(const NetDev &nd, int pop, const uint4 &th, uint32_t w) {
  const uint32_t u = w >> 12;
  uint32_t k = (u >= th.x ? 1u : 0u) + (u >= th.y ? 1u : 0u) + (u >= th.z ? 1u : 0u);
  if (u >= th.w) {
    k = 4u;
    while (k < (uint32_t)kPoisMax && u >= nd.thr[pop][k]) ++k;
  }
  return k;
}

// External drive of 4 neurons at step t without the events after each neuron's
// first (kx counts them all).
__device__ __forceinline__ int4 first_drive(const NetDev &nd, uint32_t n0, uint32_t t, int p0, int p1, uint32_t (&kx)[4]) {
  const uint4 R = philox4x32_10(n0 >> 2, t, 1u, 0u, nd.key0, nd.key1);
  const uint4 t0 = *reinterpret_cast<const uint4 *>(nd.thr[p0]);
  const uint4 t1 = *reinterpret_cast<const uint4 *>(nd.thr[p1]);
  kx[0] = events_of(nd, p0, t0, R.x);
  kx[1] = events_of(nd, p0, t0, R.y);
  kx[2] = events_of(nd, p1, t1, R.z);
  kx[3] = events_of(nd, p1, t1, R.w);
  const int32_t *a0 = nd.amp + p0 * kZTab, *a1 = nd.amp + p1 * kZTab;
  int4 I = make_int4(0, 0, 0, 0);
  if (kx[0]) I.x = __ldg(a0 + (R.x & 0xFFFu));
  if (kx[1]) I.y = __ldg(a0 + (R.y & 0xFFFu));
  if (kx[2]) I.z = __ldg(a1 + (R.z & 0xFFFu));
  if (kx[3]) I.w = __ldg(a1 + (R.w & 0xFFFu));
  return I;
}

// Eq. 2 over one step (every operation rounded once; no branches).
__device__ __forceinline__ bool run_step(const float4 &pa, const float4 &pb, float &V, float &c, uint32_t &ref, int32_t I,
                                         bool live) {
  const float c_old = c;
  const float b = __fmul_rn(pa.x, __fsub_rn(V, pa.w));
  const float f = __fadd_rn(b, __fmul_rn(pa.y, c_old));
  const float g = __fadd_rn(pa.w, f);
  const float vn = __fadd_rn(g, __fmul_rn(__int2float_rn(I), 1.0f / 65536.0f));
  const bool held = ref > 0u;
  const bool spike = live && !held && vn > pb.x;
  V = (held || spike) ? pb.y : vn;
  ref = held ? ref - 1u : (spike ? __float_as_uint(pb.w) : 0u);
  float cn = __fmul_rn(pa.z, c_old);
  if (spike) cn = __fadd_rn(cn, pb.z);
  c = cn;
  return spike;
}

__device__ __forceinline__ uint32_t run_step4(const NetDev &nd, uint32_t n0, int p0, int p1, float4 &V, float4 &c, uint32_t &ref,
                                              const int4 &I) {
  const float4 a0 = nd.pa[p0], b0 = nd.pb[p0], a1 = nd.pa[p1], b1 = nd.pb[p1];
  uint32_t r0 = ref & 0xFFu, r1 = (ref >> 8) & 0xFFu, r2 = (ref >> 16) & 0xFFu, r3 = ref >> 24;
  const bool l0 = n0 < nd.N, l1 = n0 + 2u < nd.N;   // N is even
  uint32_t mask = 0;
  if (run_step(a0, b0, V.x, c.x, r0, I.x, l0)) mask |= 1u;
  if (run_step(a0, b0, V.y, c.y, r1, I.y, l0)) mask |= 2u;
  if (run_step(a1, b1, V.z, c.z, r2, I.z, l1)) mask |= 4u;
  if (run_step(a1, b1, V.w, c.w, r3, I.w, l1)) mask |= 8u;
  ref = r0 | (r1 << 8) | (r2 << 16) | (r3 << 24);
  return mask;
}

// ---------------------------------------------------------------------------
// Delay-major delivery (Sec. 2.1.1).  A delivery pass follows the update of
// every step t with (t + 1) % kmin == 0 (kmin = the smallest delay: the spikes
// of kmin consecutive steps are delivered together, the paper's exchange step
// equal to the minimum delay).  It produces the inputs of the next kmin steps
// T = t + 1 .. t + kmin: for each T, the delay-d group (kmin <= d <= n_delay)
// of every spike of step T - d, one segment per (spike, d).  Segments are
// spread over all warps of the grid, `lanes` lanes per segment, and their
// records are reduced straight into the input buffer of T.
// ---------------------------------------------------------------------------
// Slot of step T - d, Tm = T mod D, 1 <= d < D.
__device__ __forceinline__ uint32_t slot_back(uint32_t Tm, uint32_t d, uint32_t D) { return Tm >= d ? Tm - d : Tm + D - d; }

// Segment prefix of one target step, held in registers across the warp:
// lane l of chunk c stands for delay d = 32 c + l + 1, with incl[c] = the
// spikes of steps T - d' summed over kmin <= d' <= d (0 below kmin; past
// n_delay it stays at the total) and base[c] = the sum below the chunk.
// NCH = chunks of 32 delays (n_delay <= 32 NCH).  No shared memory.
template <int NCH>
struct WarpPrefix {
  uint32_t incl[NCH];
  uint32_t base[NCH];
  uint32_t total;
};

// T = t + 1 + j with Tm = T mod D; the spikes of step t itself are left out
// when skip_current.  The count loads of all chunks are issued first.
template <int NCH>
__device__ __forceinline__ void warp_prefix(const NetDev &nd, WarpPrefix<NCH> &P, uint32_t Tm, uint32_t j,
                                            bool skip_current) {
  const uint32_t lane = lane_id();
  const uint32_t D = nd.D, dmax = nd.n_delay, kmin = nd.kmin;
  uint32_t v[NCH];
#pragma unroll
  for (int c = 0; c < NCH; ++c) {
    const uint32_t d = 32u * c + lane + 1u;
    const bool use = d >= kmin && d <= dmax && !(skip_current && d == j + 1u);
    v[c] = use ? ld_cg_u32(nd.cnt + slot_back(Tm, d, D)) : 0u;
  }
  uint32_t run = 0;
#pragma unroll
  for (int c = 0; c < NCH; ++c) {
    uint32_t x = v[c];
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
}

// The delay d of segment g of this lane's group (smallest d with prefix > g)
// and the prefix below it; d = 0 when g >= the total.  Called by whole warps:
// every group's g is tested against a chunk with one ballot.
template <int NCH>
__device__ __forceinline__ void find_delay(const WarpPrefix<NCH> &P, uint32_t g, uint32_t lanes, uint32_t &d,
                                           uint32_t &below) {
  const uint32_t lane = lane_id(), grp = lane / lanes, gpw = 32u / lanes;
  d = 0;
  below = 0;
#pragma unroll
  for (int c = 0; c < NCH; ++c) {
    uint32_t first = 32u;   // this group's first lane of the chunk with prefix > g
    for (uint32_t q = 0; q < gpw; ++q) {
      const uint32_t gq = __shfl_sync(0xFFFFFFFFu, g, q * lanes);
      const uint32_t bal = __ballot_sync(0xFFFFFFFFu, P.incl[c] > gq);
      if (grp == q && bal) first = (uint32_t)(__ffs(bal) - 1);
    }
    const uint32_t prev = __shfl_sync(0xFFFFFFFFu, P.incl[c], (first - 1u) & 31u);
    if (d == 0 && first < 32u) {
      d = 32u * c + first + 1u;
      below = first ? prev : P.base[c];
    }
  }
}

// Prefetch into L2 the next delay group (after record b) of source s's row.
__device__ __forceinline__ void prefetch_next_group(const NetDev &nd, uint32_t s, const uint16_t *o, uint32_t d,
                                                    uint32_t b) {
  if (d >= nd.n_delay) return;
  const uint32_t c2 = o[d + 1u];
  if (c2 <= b) return;
  const uint32_t wb = nd.fmt ? 2u : 4u;
  const uint8_t *row = nd.rows + (size_t)s * nd.row_bytes;
  prefetch_range_l2(row + (size_t)b * 4u, (c2 - b) * 4u);
  prefetch_range_l2(row + (size_t)nd.M_pad * 4u + (size_t)b * wb, (c2 - b) * wb);
}

// Reduce the records [a, b) of source s's row into `acc_T`, `lanes` lanes
// (this lane is `sub`), the loads of four records per lane issued first.
__device__ __forceinline__ void add_records(const NetDev &nd, int32_t *acc_T, uint32_t s, uint32_t a, uint32_t b,
                                            uint32_t sub, uint32_t lanes) {
  const uint8_t *row = nd.rows + (size_t)s * nd.row_bytes;
  const uint32_t *keys = reinterpret_cast<const uint32_t *>(row);
  const uint8_t *wrow = row + (size_t)nd.M_pad * 4u;
  const bool i16 = nd.fmt != 0u;
  for (uint32_t r = a + sub; r < b; r += 4u * lanes) {
    uint32_t kk[4];
    int32_t vv[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) kk[u] = ld_rec_u32_if(r + (uint32_t)u * lanes < b, keys + r + (uint32_t)u * lanes, 0u);
    if (i16) {
#pragma unroll
      for (int u = 0; u < 4; ++u)
        vv[u] = ld_rec_s16_if(r + (uint32_t)u * lanes < b, reinterpret_cast<const int16_t *>(wrow) + r + (uint32_t)u * lanes);
    } else {
#pragma unroll
      for (int u = 0; u < 4; ++u)
        vv[u] = (int32_t)ld_rec_u32_if(r + (uint32_t)u * lanes < b,
                                       reinterpret_cast<const uint32_t *>(wrow) + r + (uint32_t)u * lanes, 0u);
    }
#pragma unroll
    for (int u = 0; u < 4; ++u)
      if (r + (uint32_t)u * lanes < b)
        red_add_s32(acc_T + (kk[u] & 0xFFFFFFu),
                    i16 ? vv[u] * 64 : __float2int_rn(__fmul_rn(__int_as_float(vv[u]), 65536.0f)));
  }
}

// Segments of the target step with slot Tm (prefix P): the warp takes
// segments wbase .. wbase + 32 / lanes - 1, then the same plus stride, ...,
// one per group of `lanes` lanes (this lane is `sub` of group grp).
template <int NCH>
__device__ __forceinline__ void deliver_segments(const NetDev &nd, const WarpPrefix<NCH> &P, uint32_t Tm,
                                                 int32_t *acc_T, uint32_t wbase, uint32_t stride, uint32_t lanes) {
  const uint32_t D = nd.D;
  const uint32_t lane = lane_id(), grp = lane / lanes, sub = lane % lanes;
  for (uint32_t gb = wbase; gb < P.total; gb += stride) {   // warp-uniform
    const uint32_t g = gb + grp;
    uint32_t d, below;
    find_delay<NCH>(P, g, lanes, d, below);
    if (d == 0) continue;   // g past the total (last round)
    const uint32_t s = ld_cg_u32(nd.hist + (size_t)slot_back(Tm, d, D) * nd.N_pad + (g - below));
    const uint16_t *o = nd.offs + (size_t)s * nd.os;
    add_records(nd, acc_T, s, o[d - 1u], o[d], sub, lanes);
  }
}

}  // namespace snn

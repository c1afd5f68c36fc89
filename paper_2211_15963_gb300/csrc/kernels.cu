// Hot-path kernels for sm_103a.
//
//   k_update   one Euler step of every neuron (Methods, capacitance-voltage
//              equation and Eq. 2; Supplementary Sec. 3, Eqs. 3 and 5 with
//              the refractory reset), the Poisson background drawn from
//              Philox4x64-10, spike compaction into the spike ring,
//              and region spike counts; k_update<true> also integrates the
//              background OU current (Eq. 1) and applies the per-neuron
//              injected-current factors; k_update<., true> reads four
//              accumulator channels (two weights per edge) instead of the
//              two classes.
//   k_close / the first blocks of k_update: the per-bin Balloon-Windkessel
//              step (Extended Data Table 4) and the BOLD sample, a region on
//              two lanes.
//   push delivery (Supplementary Algorithm 2) into the ring of fixed-point
//              accumulators, by the engine's mode (engine.h): k_update adds
//              the edges of the spikes it emits that come due soon (or all),
//              k_windows those of earlier spikes due in the next few steps,
//              k_deliver those due in one step.  In each, a warp lays the
//              segments of its 32 spikes end to end so that consecutive lanes
//              read consecutive edge records; with two weights per edge an
//              edge adds both to the channel pair of the source's class with
//              one 64-bit atomic.
//
// The kernels find their iteration through a StepRef (a base word in device
// memory plus an offset), so a captured CUDA graph of steps is valid for any
// aligned step.
//
// The FP32 neuron arithmetic is written with explicit round-to-nearest
// intrinsics in a fixed order so that no operation is fused or reordered; the
// library is also built with -fmad=false.
#include <cuda_runtime.h>

#include "engine.h"

namespace dbn {

namespace {

constexpr unsigned kFull = 0xffffffffu;

// (philox4x64_10 is in engine.h: the host draws with it too)

__device__ __forceinline__ int find_region(const int32_t* __restrict__ ro, int R, int32_t li) {
  int lo = 0, hi = R - 1;
  while (lo < hi) {
    int mid = (lo + hi + 1) >> 1;
    if (__ldg(ro + mid) <= li) lo = mid; else hi = mid - 1;
  }
  return lo;
}

// Edge records stream through the delivery once (a spike's row is read in a
// few short segments, one per delay, spread over up to D steps), while the
// accumulators of the step are its working set: the record loads carry an
// L2 evict-first policy and the accumulator reductions an evict-last one
// (PTX createpolicy / .L2::cache_hint).
#ifndef DBNET_L2_HINTS
#define DBNET_L2_HINTS 1
#endif
// 32-edge chunks of a warp's walk whose record loads are issued before the
// first of their atomics (memory-level parallelism of the walk): two measured
// 97.8 / 129.5 us a step at 5 M neurons and for the 64-member ensemble, four
// 99.1 / 131.4, eight 104.6 / 138.5.  A lone spike's row takes four at once:
// nothing else covers its latency.
#ifndef DBNET_WALK_CHUNKS
#define DBNET_WALK_CHUNKS 2
#endif
constexpr int kLoneU = 4;
constexpr int kWalkU = DBNET_WALK_CHUNKS;
constexpr int kSegGroup = 32;  // spikes per transposition group of the segment-ring copy
constexpr int kTileWarps = kTile / 128;  // warps of an update tile, 128 neurons each
constexpr int kMaxPhases = 8;  // rank phases of the arrival items (see k_deliver)

__device__ __forceinline__ unsigned long long l2_policy_first() {
  unsigned long long p = 0;
#if DBNET_L2_HINTS
  asm("createpolicy.fractional.L2::evict_first.b64 %0, 1.0;" : "=l"(p));
#endif
  return p;
}
__device__ __forceinline__ unsigned long long l2_policy_last() {
  unsigned long long p = 0;
#if DBNET_L2_HINTS
  asm("createpolicy.fractional.L2::evict_last.b64 %0, 1.0;" : "=l"(p));
#endif
  return p;
}
__device__ __forceinline__ uint32_t ld_stream_u32(const uint32_t* a, unsigned long long pol) {
#if DBNET_L2_HINTS
  uint32_t v;
  asm("ld.global.nc.L2::cache_hint.u32 %0, [%1], %2;" : "=r"(v) : "l"(a), "l"(pol));
  return v;
#else
  (void)pol;
  return __ldg(a);
#endif
}
__device__ __forceinline__ uint2 ld_stream_u64(const uint2* a, unsigned long long pol) {
#if DBNET_L2_HINTS
  uint2 v;
  asm("ld.global.nc.L2::cache_hint.v2.u32 {%0, %1}, [%2], %3;" : "=r"(v.x), "=r"(v.y) : "l"(a), "l"(pol));
  return v;
#else
  (void)pol;
  return __ldg(a);
#endif
}
__device__ __forceinline__ void red_add_s32(int* a, int v, unsigned long long pol) {
#if DBNET_L2_HINTS
  asm volatile("red.global.add.L2::cache_hint.s32 [%0], %1, %2;" ::"l"(a), "r"(v), "l"(pol));
#else
  (void)pol;
  atomicAdd(a, v);
#endif
}
__device__ __forceinline__ void red_add_u64(unsigned long long* a, unsigned long long v,
                                            unsigned long long pol) {
#if DBNET_L2_HINTS
  asm volatile("red.global.add.L2::cache_hint.u64 [%0], %1, %2;" ::"l"(a), "l"(v), "l"(pol));
#else
  (void)pol;
  atomicAdd(a, v);
#endif
}

// Forward-Euler step of the hemodynamic model for one region (FP64), from
// its two powers fout = v^(1/alpha) and oe = (1 - rho)^(1/f).
__device__ double bw_euler(double* x, double z, const InstDesc& d, double fout, double oe) {
  const double s = x[0], f = x[1], v = x[2], q = x[3];
  const double E = 1.0 - oe;
  const double ds = z - d.kappa * s - d.gamma * (f - 1.0);
  const double dv = (f - fout) / d.tau;
  const double dq = (f * E / d.rho - fout * q / v) / d.tau;
  const double h = d.h_bw;
  const double s2 = s + h * ds, f2 = f + h * s, v2 = v + h * dv, q2 = q + h * dq;
  x[0] = s2;
  x[1] = f2;
  x[2] = v2;
  x[3] = q2;
  const double k1 = 7.0 * d.rho, k2 = 2.0, k3 = 2.0 * d.rho - 0.2;
  return d.V0 * (k1 * (1.0 - q2) + k2 * (1.0 - q2 / v2) + k3 * (1.0 - v2));
}

__global__ void __launch_bounds__(kTile / 4) k_init_state(EngineDev e, int inst, int first_tile) {
  const InstDesc& d = e.insts[inst];
  const int64_t gi0 = (int64_t)(first_tile + blockIdx.x) * kTile + threadIdx.x * 4;
  const int32_t li0 = (int32_t)(gi0 - d.base);
  float v4[4] = {0.f, 0.f, 0.f, 0.f};
  float b4[4] = {0.f, 0.f, 0.f, 0.f};  // background OU current starts at its mean
  unsigned long long c[4] = {0ull, (unsigned long long)(li0 >> 2), 1ull, 0ull};
  philox4x64_10(c, d.seed, d.net_id);
  int r = li0 < d.N ? find_region(d.region_offsets, d.R, li0) : 0;
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    const int32_t li = li0 + k;
    if (li < d.N) {
      while (li >= d.rc[r].end) ++r;
      const RegionConst& p = d.rc[r];
      const float u = __fmul_rn(__ull2float_rn(c[k] >> 40), 5.9604644775390625e-08f);  // 2^-24
      const float span = __fsub_rn(p.Vth, p.Vreset);
      v4[k] = __fadd_rn(p.Vreset, __fmul_rn(span, u));
      if (p.ext & kExtOU) b4[k] = p.ou_mu;
    }
  }
  *reinterpret_cast<float4*>(e.V + gi0) = make_float4(v4[0], v4[1], v4[2], v4[3]);
  if (e.Ibg) *reinterpret_cast<float4*>(e.Ibg + gi0) = make_float4(b4[0], b4[1], b4[2], b4[3]);
#pragma unroll
  for (int u = 0; u < 4; ++u)
    *reinterpret_cast<float4*>(e.J + u * e.stride + gi0) = make_float4(0.f, 0.f, 0.f, 0.f);
  *reinterpret_cast<uint32_t*>(e.ref + gi0) = 0u;
  // accumulators: int2 per neuron, or int4 (acc[2i], acc[2i + 1]) with four
  // channels, in every slot of the ring
  const int words = e.four ? 4 : 2;
  for (int a = 0; a < e.acc_slots; ++a) {
    int2* slot = e.acc + (size_t)a * (size_t)e.stride * (e.four ? 2 : 1);
    for (int k = 0; k < words; ++k)
      *reinterpret_cast<int4*>(slot + (e.four ? 2 : 1) * gi0 + 2 * k) = make_int4(0, 0, 0, 0);
  }
}

__device__ __forceinline__ unsigned long long step_of(const StepRef& sr) {
  return (sr.base ? *reinterpret_cast<const volatile unsigned long long*>(sr.base) : 0ull) + sr.off;
}

// Close the bins that ended with iteration g - 1, each once: the
// Balloon-Windkessel step with that bin's activity, and the BOLD sample when
// the bin ends a TR.  Warps w, w + n, ... of the caller take 16 regions each,
// a region on two lanes that compute one of its two powers (a power is some
// 3 us of dependent FP64 operations, and on small networks everybody waits
// for them).  Called by whole warps.
__device__ void close_regions(const EngineDev& e, unsigned long long g, int w, int n) {
  const int lane = threadIdx.x & 31;
  for (int first = w * 16; first < e.total_R; first += n * 16) {
    const int gr = first + (lane >> 1);
    int k = -1;
    long long nk = 0;
    if (gr < e.total_R) {
      k = e.region_inst[gr];
      if (k >= 0 && !e.dyn[k].active) k = -1;  // unused region slot, or retired
      if (k >= 0) {
        const InstDesc& dk = e.insts[k];
        nk = (long long)(g - 1ull - dk.g0);  // step just completed
        if (g <= dk.g0 || nk >= dk.n_end || (nk + 1) % dk.spb != 0 || e.closed[gr] >= (long long)g) k = -1;
      }
    }
    if (!__any_sync(kFull, k >= 0)) continue;
    const InstDesc& dk = e.insts[k < 0 ? 0 : k];
    double a = 1.0, x = 1.0;
    if (k >= 0) {
      a = (lane & 1) ? 1.0 - dk.rho : e.bw[4 * gr + 2];
      x = 1.0 / ((lane & 1) ? e.bw[4 * gr + 1] : dk.alpha);
    }
    const double p = pow(a, x);
    const double other = __shfl_xor_sync(kFull, p, 1);
    if (k < 0 || (lane & 1)) continue;
    const int r = gr - dk.rbase;
    const double nr = (double)(dk.rc[r].end - dk.rc[r].start);
    int32_t* const cnt = e.cnt + ((nk / dk.spb) & 1) * e.cnt_stride + gr;  // that bin's
    const double z = dk.z_scale * (double)*cnt / nr;
    *cnt = 0;
    const double y = bw_euler(e.bw + 4 * gr, z, dk, p, other);
    e.ylast[gr] = y;
    const long long b = (nk + 1) / dk.spb;  // bins completed
    if (b % dk.bins_per_tr == 0) {
      const long long sidx = b / dk.bins_per_tr - 1;
      if (sidx < dk.bold_cap) dk.bold[sidx * dk.R + r] = y;
    }
    e.closed[gr] = (long long)g;
  }
}

__global__ void k_close(EngineDev e, unsigned long long g) {
  close_regions(e, g, (blockIdx.x * blockDim.x + threadIdx.x) >> 5, (gridDim.x * blockDim.x) >> 5);
}

__global__ void k_set_base(unsigned long long* base, unsigned long long g) { *base = g; }

// Standard normal from one Philox word (Box-Muller): u1 = (high 32 bits + 1)
// 2^-32 in (0, 1], u2 = low 32 bits 2^-32, sqrt(-2 ln u1) cos(2 pi u2) in FP32.
__device__ __forceinline__ float normal_from_word(unsigned long long w) {
  const float u1 = __double2float_rn(((double)(uint32_t)(w >> 32) + 1.0) * 2.3283064365386963e-10);
  const float u2 = __double2float_rn((double)(uint32_t)w * 2.3283064365386963e-10);
  return sqrtf(-2.0f * logf(u1)) * cospif(2.0f * u2);
}

// The accumulator slot of iteration a, and where it lies.  ANY: the ring may be
// other than a power of two (at most 256 slots); the update's variants without
// the kExt* terms leave that out (nest_4m_1ms 49.8 against 49.6 ms, 64 members
// 131.3 against 130.7) and such engines take the variants with them.
template <bool ANY>
__device__ __forceinline__ uint32_t acc_slot(const EngineDev& e, unsigned long long a) {
  const uint32_t n = (uint32_t)e.acc_slots;
  if (!ANY || (n & (n - 1u)) == 0u) return (uint32_t)a & (n - 1u);
  return ((uint32_t)(a >> 32) % n * (0xFFFFFFFFu % n + 1u) + (uint32_t)a % n) % n;
}
template <bool ANY>
__device__ __forceinline__ int2* acc_of(const EngineDev& e, unsigned long long g) {
  return e.acc + (size_t)acc_slot<ANY>(e, g) * (size_t)e.stride * (e.four ? 2 : 1);
}

// a / b for step counts: in 32 bits while they fit
__device__ __forceinline__ long long div_steps(long long a, int b) {
  return (unsigned long long)a >> 32 ? a / b : (long long)((uint32_t)a / (uint32_t)b);
}

__device__ __forceinline__ uint32_t edge_delay(const uint32_t* col, const uint8_t* dl, int shift,
                                               int64_t e) {
  return dl ? (uint32_t)__ldg(dl + e) : (__ldg(col + e) >> shift);
}

// first edge in [lo, hi) whose delay is >= d (rows are sorted by delay)
__device__ int64_t first_delay_at_least(const uint32_t* col, const uint8_t* dl, int shift,
                                        int64_t lo, int64_t hi, uint32_t d) {
  while (lo < hi) {
    const int64_t mid = (lo + hi) >> 1;
    if (edge_delay(col, dl, shift, mid) < d) lo = mid + 1; else hi = mid;
  }
  return lo;
}

// What the walk needs of an instance.
struct EdgeView {
  const uint16_t* rec;
  const uint32_t* col;
  const uint16_t* w;
  const uint8_t* delay;
  int64_t base;
  uint32_t tmask;
  int32_t shift, two_w;
  float two_S;
  __device__ __forceinline__ explicit EdgeView(const InstDesc& d)
      : rec(d.rec), col(d.col), w(d.w), delay(d.delay), base(d.base), tmask(d.tmask), shift(d.shift),
        two_w(d.two_w), two_S(d.two_S) {}
};

// One edge's additions: word and weights of a record of v, of a spike with
// this key (handed on at a step with low bits key >> 1, class key & 1).
//
// FOUR: four accumulator channels per neuron; an edge adds its two weights
// (the one weight twice for one-weight records) to the channel pair of the
// source's class with one 64-bit atomic.  Every channel sum stays below 2^31
// (the fixed-point scale is chosen so), so the low word never carries into
// the high one.
template <bool FOUR>
__device__ __forceinline__ void add_edge(const EngineDev& e, const EdgeView& v, uint32_t word, uint32_t wts,
                                         uint32_t key, unsigned long long pol_acc) {
  const uint32_t slot = ((key >> 1) + (word >> v.shift)) & ((uint32_t)e.acc_slots - 1u);
  const size_t at = (size_t)slot * (size_t)e.stride + (size_t)v.base + (word & v.tmask);
  const int q = __float2int_rn(__fmul_rn(__uint_as_float(wts << 16), v.two_S));
  if (FOUR) {
    const int q2 = __float2int_rn(__fmul_rn(__uint_as_float(wts & 0xFFFF0000u), v.two_S));
    red_add_u64(reinterpret_cast<unsigned long long*>(e.acc) + 2 * at + (key & 1u),
                ((unsigned long long)(uint32_t)q2 << 32) | (uint32_t)q, pol_acc);
  } else {
    red_add_s32(reinterpret_cast<int*>(e.acc) + 2 * at + (key & 1u), q, pol_acc);
  }
}

// Record ei of v: its word and its two weights (the one weight twice).
template <bool FOUR>
__device__ __forceinline__ void load_edge(const EdgeView& v, int64_t ei, uint32_t& word, uint32_t& wts,
                                          unsigned long long pol_rec) {
  if (FOUR && v.two_w) {  // 8-byte record: word, weight | second weight << 16
    const uint2 r4 = ld_stream_u64(reinterpret_cast<const uint2*>(v.rec) + ei, pol_rec);
    word = r4.x;
    wts = r4.y;
  } else if (v.rec) {
    // 6-byte record at byte 6 ei: two aligned words cover it (the record
    // array carries 8 bytes of padding at its end)
    const size_t byte = 6 * (size_t)ei;
    const uint32_t* w4 = reinterpret_cast<const uint32_t*>(
        reinterpret_cast<const unsigned char*>(v.rec) + (byte & ~size_t(3)));
    const uint32_t w0 = ld_stream_u32(w4, pol_rec), w1 = ld_stream_u32(w4 + 1, pol_rec);
    const uint32_t sh = (uint32_t)(byte & 3u) * 8u;  // 0 or 16
    word = __funnelshift_r(w0, w1, sh);
    const uint32_t wb = (w1 >> sh) & 0xFFFFu;
    wts = wb | (wb << 16);
  } else {
    word = __ldg(v.col + ei) | ((uint32_t)__ldg(v.delay + ei) << v.shift);
    const uint32_t wb = __ldg(v.w + ei);
    wts = wb | (wb << 16);
  }
}

// Adds the warp's segments -- nseg edge records from e0 on, of a row of
// instance inst (UNI: the first) whose spike was handed on at a step with low
// bits key >> 1 and has class key & 1 -- each edge into the accumulator slot
// of its arrival step.  The segments are laid end to end: consecutive lanes
// take consecutive records (coalesced), and kWalkU chunks of 32 records are
// loaded before the first of their reductions.  A chunk's owners come from
// one word: the lanes whose segment starts in the chunk set its bit (a warp
// OR), and a record belongs to the item whose rank among the non-empty ones
// is the number of starts up to it; the items lie by rank in s_item (32 a
// warp), so that an owner's data is one 16-byte read.  (A shuffle search per
// chunk took 5 + 5 shuffles and more than twice the instructions, and the
// walk is bound by its issue slots.)  Called by the whole warp.
template <bool FOUR, bool UNI>
__device__ __forceinline__ void walk_segments(const EngineDev& e, const InstDesc* insts, int4* s_item,
                                              int64_t e0, uint32_t nseg, int inst, uint32_t key,
                                              unsigned long long pol_rec, unsigned long long pol_acc) {
  const int lane = threadIdx.x & 31;
  uint32_t incl = nseg;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const uint32_t x = __shfl_up_sync(kFull, incl, o);
    if (lane >= o) incl += x;
  }
  const uint32_t total = __shfl_sync(kFull, incl, 31);
  if (total == 0u) return;
  const uint32_t ex = incl - nseg;
  const unsigned full = __ballot_sync(kFull, nseg != 0u);
  if (nseg != 0u) {
    const int64_t b = e0 - (int64_t)ex;  // record of edge fi of the walk: b + fi
    s_item[__popc(full & ((1u << lane) - 1u))] = make_int4((int)(uint32_t)b, (int)(b >> 32), (int)key, inst);
  }
  __syncwarp();
  const unsigned upto = 0xffffffffu >> (31 - lane);  // this lane and those before
  const EdgeView v0(insts[0]);
  int begun = -1;  // items that start before the chunk, less one
  for (uint32_t f = 0; f < total; f += 32u * kWalkU) {  // warp-uniform
    uint32_t tg[kWalkU], wv[kWalkU], ky[kWalkU];
    int ic[kWalkU];
#pragma unroll
    for (int u = 0; u < kWalkU; ++u) {
      const uint32_t at = ex - (f + 32u * u);
      const unsigned starts = __reduce_or_sync(kFull, nseg != 0u && at < 32u ? 1u << at : 0u);
      const int owner = begun + __popc(starts & upto);
      begun += __popc(starts);
      const uint32_t fi = f + 32u * u + lane;
      ky[u] = 0u;
      ic[u] = -1;
      if (fi < total) {
        const int4 it = s_item[owner];
        ky[u] = (uint32_t)it.z;
        ic[u] = UNI ? 0 : it.w;
        const int64_t ei = (int64_t)(((uint64_t)(uint32_t)it.y << 32) | (uint32_t)it.x) + (int64_t)fi;
        const EdgeView v(UNI ? v0 : EdgeView(insts[ic[u]]));
        load_edge<FOUR>(v, ei, tg[u], wv[u], pol_rec);
      }
    }
#pragma unroll
    for (int u = 0; u < kWalkU; ++u) {
      if (ic[u] < 0) continue;
      add_edge<FOUR>(e, UNI ? v0 : EdgeView(insts[ic[u]]), tg[u], wv[u], ky[u], pol_acc);
    }
  }
  __syncwarp();  // s_item is read
}

// Row j of the segment table: a header with the row's first and last edge,
// then the counts.  One look-up per item reads both from one DRAM page.
__device__ __forceinline__ const unsigned char* seg_row(const InstDesc& dd, int64_t j) {
  return static_cast<const unsigned char*>(dd.seg) + j * (int64_t)dd.seg_bytes;
}
// Edges of a row of delay <= d, for 1 <= d <= dmax, from its table row.
__device__ __forceinline__ uint32_t edges_up_to(const InstDesc& dd, const unsigned char* row, int d) {
  return dd.seg_kind == kSeg16 ? (uint32_t)__ldg(reinterpret_cast<const uint16_t*>(row + kSegHead) + d - 1)
                               : __ldg(reinterpret_cast<const uint32_t*>(row + kSegHead) + d - 1);
}

// Region constants of a thread's four neurons: one region's for all (ONE), or
// each neuron's own.
// HELD: they may lie in shared memory (the resident steppers), else they are
// read through the L1's read-only path.
template <bool ONE, bool HELD>
struct QuadConst {
  const RegionConst* p;  // the tile's first region
  int r[ONE ? 1 : 4];    // the neurons' regions, counted from it
  __device__ __forceinline__ const RegionConst& of(int k) const { return ONE ? *p : p[r[ONE ? 0 : k]]; }
  template <class T>
  static __device__ __forceinline__ T ld(const T* a) {
    return HELD ? *a : __ldg(a);
  }
  // the regions of neurons li0 .. li0 + m - 1
  __device__ __forceinline__ void find(int32_t li0, int m) {
    int at = 0;
#pragma unroll
    for (int k = 0; k < (ONE ? 0 : 4); ++k) {
      if (k < m)
        while (li0 + k >= ld(&p[at].end)) ++at;
      r[ONE ? 0 : k] = at;
    }
  }
};

// What the membrane step of a thread's four neurons leaves: bit k of spk and
// cls for a spike of neuron k and its inhibitory class.
struct QuadSpikes {
  unsigned spk = 0, cls = 0;
};

// A step's random draws of the thread's four neurons: what the background
// drive adds to AMPA and NMDA, and the normals of the OU current where the
// instance has it.  They depend on the step alone.
struct QuadDraw {
  int dq[4];
  float xi[4];
};
template <bool EXT, bool ONE, bool HELD>
__device__ __forceinline__ QuadDraw quad_draw(const InstDesc& d, const QuadConst<ONE, HELD>& rc, int32_t li0,
                                              long long n) {
  QuadDraw o;
  unsigned long long x[4] = {(unsigned long long)n, (unsigned long long)(li0 >> 2), 0ull, 0ull};
  philox4x64_10(x, d.seed, d.net_id);
  // background: Poisson count by integer inversion of 32 Philox bits (the
  // thresholds are non-decreasing: count them up to the first miss)
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    const RegionConst& p = rc.of(k);
    const uint32_t uu = (uint32_t)(x[k] >> 32);
    const int n_thr = rc.ld(&p.n_thr);
    int c = 0;
    while (c < n_thr && uu >= rc.ld(&p.thr[c])) ++c;
    o.dq[k] = c * rc.ld(&p.q_ext);
  }
  if (EXT && (d.ext & kExtOU)) {  // the OU noise: stream 4
    unsigned long long xo[4] = {(unsigned long long)n, (unsigned long long)(li0 >> 2), 4ull, 0ull};
    philox4x64_10(xo, d.seed, d.net_id);
#pragma unroll
    for (int k = 0; k < 4; ++k) o.xi[k] = normal_from_word(xo[k]);
  }
  return o;
}

// State of the thread's four neurons.
struct QuadState {
  float4 V, J[4], B;  // B: the background current, where the instance has it
  uchar4 ref;
};
__device__ __forceinline__ void quad_load(const EngineDev& e, int64_t gi0, QuadState& q) {
  // (state is streamed once per step: evict-first, so that the delivery's
  // working set keeps the L2)
  q.V = __ldcs(reinterpret_cast<const float4*>(e.V + gi0));
#pragma unroll
  for (int u = 0; u < 4; ++u) q.J[u] = __ldcs(reinterpret_cast<const float4*>(e.J + u * e.stride + gi0));
  q.ref = __ldcs(reinterpret_cast<const uchar4*>(e.ref + gi0));
}

// One Euler step of the thread's four neurons (m of them exist).  The traces
// go channel by channel over the four, so that only one channel's constants
// are live at a time.  HELD: the state stays in q (the resident steppers);
// else each vector is stored as soon as it is updated.
template <bool EXT, bool FOUR, bool ONE, bool HELD>
__device__ __forceinline__ QuadSpikes quad_step(const EngineDev& e, const InstDesc& d, const QuadConst<ONE, HELD>& rc,
                                                int m, int64_t gi0, int32_t li0, const QuadDraw& draw,
                                                QuadState& q, const int4 (&A)[FOUR ? 4 : 2]) {
  const float v[4] = {q.V.x, q.V.y, q.V.z, q.V.w};
  float Isyn[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
  for (int u = 0; u < 4; ++u) {  // the membrane sees the old V and traces
    const float jo[4] = {q.J[u].x, q.J[u].y, q.J[u].z, q.J[u].w};
    float jn[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      const RegionConst& p = rc.of(k);
      const float gj = __fmul_rn(rc.ld(&p.g[u]), jo[k]);
      const float dv = __fsub_rn(rc.ld(&p.Vu[u]), v[k]);
      Isyn[k] = __fadd_rn(Isyn[k], __fmul_rn(gj, dv));
      // traces: decay, then this step's arrivals
      const int4 Ak = FOUR ? A[k] : A[k >> 1];
      const int a = FOUR ? (u == 0 ? Ak.x : u == 1 ? Ak.y : u == 2 ? Ak.z : Ak.w)
                         : ((k & 1) ? (u < 2 ? Ak.z : Ak.w) : (u < 2 ? Ak.x : Ak.y));
      const float xu = __fmul_rn(__int2float_rn(u < 2 ? a + draw.dq[k] : a), d.inv_two_S);
      jn[k] = __fadd_rn(__fmul_rn(rc.ld(&p.dec[u]), jo[k]), xu);
    }
    // (the last neurons of an instance: the padding keeps its values)
    q.J[u] = make_float4(jn[0], m > 1 ? jn[1] : jo[1], m > 2 ? jn[2] : jo[2], m > 3 ? jn[3] : jo[3]);
    if (!HELD) __stcs(reinterpret_cast<float4*>(e.J + u * e.stride + gi0), q.J[u]);
  }
  // the background current and the injected-current factors, only where the
  // instance has them (a request server's engine runs this variant for
  // every request)
  const bool ou = EXT && (d.ext & kExtOU), het = EXT && (d.ext & kExtHet);
  float4 F4 = make_float4(1.f, 1.f, 1.f, 1.f);
  if (ou && !HELD) q.B = __ldcs(reinterpret_cast<const float4*>(e.Ibg + gi0));
  if (het) F4 = __ldg(reinterpret_cast<const float4*>(e.fext + gi0));
  float ib[4] = {q.B.x, q.B.y, q.B.z, q.B.w};
  const float fe[4] = {F4.x, F4.y, F4.z, F4.w};
  float vo[4];
  int rr[4] = {q.ref.x, q.ref.y, q.ref.z, q.ref.w};
  QuadSpikes out;
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    vo[k] = v[k];
    if (k >= m) continue;
    const RegionConst& p = rc.of(k);
    const float4 M = rc.ld(reinterpret_cast<const float4*>(&p.dtC));     // dtC gL VL Vth
    const float4 Q = rc.ld(reinterpret_cast<const float4*>(&p.Vreset));  // Vreset Iext n_ref q_ext
    const float leak = __fmul_rn(M.y, __fsub_rn(v[k], M.z));
    float I = __fsub_rn(Isyn[k], leak);
    float4 OUc = make_float4(0.f, 0.f, 0.f, 0.f);  // mu, dt/tau, sigma sqrt(2 dt/tau), bits
    if (EXT && d.ext) OUc = rc.ld(reinterpret_cast<const float4*>(&p.ou_mu));
    const int xb = __float_as_int(OUc.w);
    // injected current, scaled by the neuron's factor where heterogeneous
    const float ie = (EXT && (xb & kExtHet)) ? __fmul_rn(Q.y, fe[k]) : Q.y;
    I = __fadd_rn(I, ie);
    if (EXT && (xb & kExtOU)) I = __fadd_rn(I, ib[k]);  // I_bg before this step
    const float vn = __fadd_rn(v[k], __fmul_rn(I, M.x));
    if (EXT && (xb & kExtOU)) {  // Eq. 1, Euler-Maruyama
      const float t1 = __fmul_rn(__fsub_rn(OUc.x, ib[k]), OUc.y);
      ib[k] = __fadd_rn(ib[k], t1);
      ib[k] = __fadd_rn(ib[k], __fmul_rn(OUc.z, draw.xi[k]));
    }
    // refractory clamp, threshold, reset
    if (rr[k] > 0) {
      vo[k] = Q.x;
      rr[k] -= 1;
    } else if (vn >= M.w) {
      vo[k] = Q.x;
      rr[k] = __float_as_int(Q.z);
      out.spk |= 1u << k;
      if (li0 + k >= rc.ld(&p.exc_end)) out.cls |= 1u << k;
    } else {
      vo[k] = vn;
    }
  }
  q.V = make_float4(vo[0], vo[1], vo[2], vo[3]);
  q.ref = make_uchar4((unsigned char)rr[0], (unsigned char)rr[1], (unsigned char)rr[2], (unsigned char)rr[3]);
  if (ou) q.B = make_float4(ib[0], ib[1], ib[2], ib[3]);
  if (!HELD) {
    __stcs(reinterpret_cast<float4*>(e.V + gi0), q.V);
    __stcs(reinterpret_cast<uchar4*>(e.ref + gi0), q.ref);
    if (ou) __stcs(reinterpret_cast<float4*>(e.Ibg + gi0), q.B);
  }
  return out;
}

// A warp's place: its tile's instance and regions, and its lanes' neurons.
struct WarpPlace {
  int inst, r0, nr, m;  // m: neurons of the thread that exist
  int64_t gi0;
  int32_t li0;
};

// What a block keeps of a tile in shared memory while its state is held: a
// barrier between steps empties the L1, and every constant would come from
// the L2 again.
constexpr int kHeldRegions = 8;
struct HeldTile {
  InstDesc d;
  RegionConst rc[kHeldRegions];
  int64_t row0;             // first edge of the tile's rows, -1: not held
  uint32_t row[kTile + 1];  // and of each row, from there
};
// The spikes of a warp's neurons in iteration g (step n of the instance):
// counts, ring append, and the edges that are due soon.  Called by the whole
// warp; s_item has 32 entries per warp of the block.
template <bool FOUR>
__device__ __forceinline__ void warp_spikes(const EngineDev& e, const InstDesc& d, const WarpPlace& w,
                                            unsigned long long g, long long n, QuadSpikes qs, int4* s_item,
                                            const HeldTile* held = nullptr) {
  const int lane = threadIdx.x & 31;
  const unsigned spk = qs.spk, cls_bits = qs.cls;
  if (!__any_sync(kFull, spk != 0)) return;
  const int nsp = __popc(spk);
  int ps = nsp;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int t = __shfl_up_sync(kFull, ps, o);
    if (lane >= o) ps += t;
  }
  const int total = __shfl_sync(kFull, ps, 31);
  // the step at which these spikes are handed on: this step, or with spike
  // binning the last step of its bin
  const long long bin = div_steps(n, d.spb);
  const unsigned long long rel = d.bin_sp ? d.g0 + (unsigned long long)((bin + 1) * d.spb - 1) : g;
  const int slot = e.mode == kAtEmission ? 0
                   : (int)((rel >> 32) ? rel % (unsigned long long)e.D : (uint32_t)rel % (uint32_t)e.D);
  int32_t* const cnt = e.cnt + (bin & 1) * e.cnt_stride + d.rbase + w.r0;
  uint32_t hbase = 0;
  unsigned long long rbase = 0;
  if (lane == 31) {
    if (e.mode != kAtEmission) hbase = atomicAdd(e.hcount + slot, (uint32_t)ps);
    atomicAdd(&e.dyn[w.inst].spikes, (unsigned long long)ps);
    if (d.raster_cap > 0) rbase = atomicAdd(&e.dyn[w.inst].raster_count, (unsigned long long)ps);
    if (w.nr == 1) atomicAdd(cnt, ps);
  }
  hbase = __shfl_sync(kFull, hbase, 31);
  rbase = __shfl_sync(kFull, rbase, 31);
  // the longest delay whose edges this warp adds: up to the end of the window
  // in which the spikes are handed on, or every delay
  const int dnow = e.mode == kAtEmission ? d.dmax
                   : e.push_now ? min(e.wmask - (int)((unsigned)rel & (unsigned)e.wmask), d.dmax)
                                : 0;
  unsigned long long ev = 0;
  // spike i of the warp goes to lane i mod 32: its owner by a shuffle search
  // over the inclusive counts, its neuron the owner's bit of that rank
  for (int i0 = 0; i0 < total; i0 += 32) {
    const int i = i0 + lane;
    int o = 0;
#pragma unroll
    for (int step = 16; step > 0; step >>= 1) {
      const int v = __shfl_sync(kFull, ps, o + step - 1);
      if (v <= i) o += step;
    }
    o = o < 32 ? o : 31;
    unsigned bits = __shfl_sync(kFull, spk, o);
    const unsigned inh = __shfl_sync(kFull, cls_bits, o);
    int rank = i - (__shfl_sync(kFull, ps, o) - __popc(bits));
    const int rk = w.nr == 1 ? 0 : -1;
    int64_t e0 = 0;
    uint32_t nseg = 0, key = 0;
    int k = 0;
    if (i < total) {
      while (rank-- > 0) bits &= bits - 1u;
      k = __ffs(bits) - 1;
      const int32_t lo = w.li0 - lane * 4 + o * 4 + k;  // the neuron
      const unsigned cl = (inh >> k) & 1u;
      if (e.mode != kAtEmission) {
        const uint64_t pos = (uint64_t)hbase + (uint32_t)i;
        if (pos < (uint64_t)e.hist_cap)
          e.hist[(size_t)slot * (size_t)e.hist_cap + pos] = (uint32_t)(d.base + lo) | (cl << 31);
        else
          atomicOr(e.flags, kFlagHistOverflow);
      }
      if (d.raster_cap > 0 && rbase + (unsigned)i < (unsigned long long)d.raster_cap) {
        d.raster_step[rbase + (unsigned)i] = (int32_t)n;
        d.raster_id[rbase + (unsigned)i] = lo;
      }
      if (rk < 0) {
        int r = 0;
        while (lo >= __ldg(&d.rc[w.r0 + r].end)) ++r;
        atomicAdd(cnt + r, 1);
      }
      if (dnow > 0) {
        key = ((uint32_t)rel << 1) | cl;
        if (e.mode == kAtEmission) {  // the whole row
          if (held && held->row0 >= 0) {
            const uint32_t* row = held->row + (lo & (kTile - 1));  // (an instance starts on a tile)
            e0 = held->row0 + row[0];
            nseg = row[1] - row[0];
          } else {
            e0 = __ldg(d.row_ptr + lo);
            nseg = (uint32_t)(__ldg(d.row_ptr + lo + 1) - e0);
          }
          ev += nseg;
        } else {
          const unsigned char* row = seg_row(d, lo);
          e0 = __ldg(reinterpret_cast<const longlong2*>(row)).x;
          nseg = edges_up_to(d, row, dnow);
        }
      }
    }
    if (dnow <= 0) continue;
    if (total == 1) {  // most often: lane 0 has it, the lanes take its records in turn
      e0 = __shfl_sync(kFull, e0, 0);
      nseg = __shfl_sync(kFull, nseg, 0);
      key = __shfl_sync(kFull, key, 0);
      const EdgeView v(d);
      const unsigned long long first = l2_policy_first(), last = l2_policy_last();
      for (uint32_t f = lane; f < nseg; f += 32u * kLoneU) {
        uint32_t word[kLoneU], wts[kLoneU];
#pragma unroll
        for (int u = 0; u < kLoneU; ++u)
          if (f + 32u * u < nseg) load_edge<FOUR>(v, e0 + f + 32u * u, word[u], wts[u], first);
#pragma unroll
        for (int u = 0; u < kLoneU; ++u)
          if (f + 32u * u < nseg) add_edge<FOUR>(e, v, word[u], wts[u], key, last);
      }
      __syncwarp();
      continue;
    }
    walk_segments<FOUR, true>(e, &d, s_item + (threadIdx.x >> 5) * 32, e0, nseg, 0, key, l2_policy_first(),
                              l2_policy_last());
  }
  if (e.mode == kAtEmission) {  // the synaptic events of these spikes
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) ev += __shfl_down_sync(kFull, ev, o);
    if (lane == 0 && ev) atomicAdd(e.events, ev);
  }
}

// One warp's 128 neurons of a tile, in the iteration sr names.
//
// EXT: also the kExt* terms of the instances that have them: the background
// OU current and the per-neuron injected-current factor.  FOUR: the
// accumulators hold four channels per neuron (two weights per edge); the
// background drive adds to both AMPA and NMDA.
//
// Bound: the state's traffic (58 bytes a neuron and step) on large networks,
// the latency of the loads on small ones.  The warps of a tile share
// nothing, so the kernel has no block barrier: a warp's region constants
// come through the L1 (one 176-byte row, the same for most warps of an SM),
// its Philox rounds run under its state loads, and a warp without spikes
// ends after its stores.  A tile inside one region (most) reads its
// constants once for four neurons.  Measured against blocks of 256 that
// staged constants in shared memory behind a barrier, one neuron after the
// other: 51.0 us against 59.8 us at 5 M neurons (5.7 TB/s of 290 MB),
// 25.9 against 30.1 us at 2 M.  Seven blocks of 128 (72 registers) beat six
// (53.2 us) and eight (64 registers, spills: 51.3 us, and 56.1 against
// 53.2 us with 50,000 spikes a step); an L2 prefetch of the state 304 to
// 1,216 tiles ahead changed nothing.
template <bool EXT, bool FOUR>
__device__ __forceinline__ void update_warp(const EngineDev& e, const StepRef& sr, int tile, int warp,
                                            int4* s_item) {
  // state loads first: they depend only on the tile, and the arrays cover
  // every padded tile
  WarpPlace w;
  w.gi0 = (int64_t)tile * kTile + warp * 128 + (threadIdx.x & 31) * 4;
  QuadState q;
  quad_load(e, w.gi0, q);
  const int4 ti = __ldg(e.tile_info + tile);  // instance, first region, regions touched
  // this step's arrivals: one int4 per neuron (AMPA, NMDA, GABA_A, GABA_B)
  // or per two (E, I of each), from the accumulator slot of this iteration
  const unsigned long long g = step_of(sr);
  constexpr int kA = FOUR ? 4 : 2;
  int4* const accs = reinterpret_cast<int4*>(acc_of<EXT>(e, g)) + (FOUR ? w.gi0 : w.gi0 / 2);
  int4 A[kA];
#pragma unroll
  for (int k = 0; k < kA; ++k) A[k] = __ldcg(accs + k);

  if (sr.next && threadIdx.x == 0) *sr.next = g + 1ull;
  if (ti.x < 0) return;  // unused tile
  w.inst = ti.x;
  w.r0 = ti.y;
  w.nr = ti.z;
  const InstDesc& d = e.insts[w.inst];
  const long long n = (long long)(g - d.g0);
  if (e.dyn[w.inst].active == 0 || n >= d.n_end) return;
  w.li0 = (int32_t)(w.gi0 - d.base);
  w.m = d.N - w.li0 < 4 ? d.N - w.li0 : 4;
  const QuadConst<true, false> one{d.rc + w.r0, {0}};
  QuadConst<false, false> each{d.rc + w.r0, {0, 0, 0, 0}};
  QuadSpikes qs;
  if (w.m > 0) {
#pragma unroll
    for (int k = 0; k < kA; ++k) accs[k] = make_int4(0, 0, 0, 0);
    if (w.nr == 1) {  // the whole tile lies in one region
      qs = quad_step<EXT, FOUR, true, false>(e, d, one, w.m, w.gi0, w.li0, quad_draw<EXT>(d, one, w.li0, n), q, A);
    } else {
      each.find(w.li0, w.m);
      qs = quad_step<EXT, FOUR, false, false>(e, d, each, w.m, w.gi0, w.li0, quad_draw<EXT>(d, each, w.li0, n), q, A);
    }
  }
  warp_spikes<FOUR>(e, d, w, g, n, qs, s_item);
}

// Programmatic dependent launch: the kernels of a step are launched while
// their predecessor still runs, wait here for its end and its writes, and let
// their successor be launched in turn once all their blocks have started
// (nothing, on an ordinary launch).
__device__ __forceinline__ void step_after() {
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  asm volatile("griddepcontrol.wait;" ::: "memory");
}

// Blocks of the update that close bins: a warp for 16 regions.
__host__ __device__ __forceinline__ int close_blocks(const EngineDev& e) {
  return (e.total_R + 16 * (kUpdThreads / 32) - 1) / (16 * (kUpdThreads / 32));
}

template <bool EXT, bool FOUR>
__global__ void __launch_bounds__(kUpdThreads, 7) k_update(EngineDev e, StepRef sr) {
  step_after();
  const int n_close = close_blocks(e);
  if ((int)blockIdx.x < n_close) {  // close the bins that ended with the previous iteration
    close_regions(e, step_of(sr), blockIdx.x * (kUpdThreads / 32) + (threadIdx.x >> 5), n_close * (kUpdThreads / 32));
    return;
  }
  const int w = (blockIdx.x - n_close) * (kUpdThreads / 32) + (threadIdx.x >> 5);
  __shared__ int4 s_item[kUpdThreads];
  update_warp<EXT, FOUR>(e, sr, w / kTileWarps, w % kTileWarps, s_item);
}

// Stage one of resolving an item (spike k of the ring slot of step g - d,
// delay d, due now; or, in the emission range, spike k of step g - 1 and one
// of its long delays d): everything that needs no other load -- the ring
// entry and, from the delay-major segment ring, the row start and the two
// segment counts -- and the accumulator slot its edges go to.
struct ItemLoads {
  uint32_t ent, d, slot, k, aslot;
  int64_t r0;
  uint32_t a, b;
  bool ring;
};

// FOUR: the engine keeps four accumulator channels per neuron; an edge adds
// its two weights (the one weight twice for one-weight records) to the
// channel pair of the source's class with one 64-bit atomic.  Every channel
// sum stays below 2^31 (the fixed-point scale is chosen so), so the low word
// never carries into the high one.  SINGLE: the engine holds one instance
// (a network, or the allocation-free run), so every spike's descriptor is
// the first.
// part: kPartAll does the whole delivery of iteration g.  The pipelined
// schedule splits it: kPartLong, the arrival items of delays >= 2, which
// read only spikes of steps <= g - 2 and so run beside the update of
// iteration g - 1; then kPartShort after that update: the ring bookkeeping,
// the segment-ring copy of step g - 1's spikes, the delay-1 items and the
// emission items.
// Per-step delivery's loads of the spike and segment rings: through the
// read-only path where an entry was written by a launch that has ended
// (k_deliver is launched plainly, never as a programmatic dependent); from the
// L2 (coherent, never a stale L1 line) in the persistent stepper, whose own
// blocks wrote them earlier in the launch.
template <bool PERSIST, typename T>
__device__ __forceinline__ T ld_ring(const T* p) {
  if (PERSIST) return __ldcg(p);
  return __ldg(p);
}

// The delivery of the iteration sr names, as block bid of nblk; the block's
// threads call it together.
template <bool FOUR, bool SINGLE, bool PERSIST>
__device__ __forceinline__ void deliver_body(const EngineDev& e, const StepRef& sr, int part, int bid,
                                             int nblk) {
  // arrival items of phase q and delay bucket i start at s_phase[q] +
  // s_pre[q][i]; bucket i holds ranks [q c/Q, (q+1) c/Q) of the c spikes
  // handed on at g - i - 1
  __shared__ unsigned long long s_pre[kMaxPhases][256];
  __shared__ unsigned long long s_wsum[kMaxPhases][kDelThreads / 32];
  __shared__ unsigned long long s_phase[kMaxPhases + 1];
  __shared__ uint32_t s_cnt[256];
  __shared__ __align__(16) uint16_t s_tab[256 * kSegGroup];  // [delay][spike] of a copy group
  __shared__ const uint4* s_row[kSegGroup];
  __shared__ int32_t s_nq[kSegGroup];
  __shared__ long long s_r0[kSegGroup];
  const unsigned long long g = step_of(sr);
  const int D = e.D;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int gtid = bid * blockDim.x + threadIdx.x;
  const bool do_short = part != kPartLong, do_long = part != kPartShort;
  // the slot that the updates from this iteration on fill (a bin later with
  // spike binning) was last read by the previous iteration; the slot handed
  // on at g - 1 gets its long delays now, at emission, when d_emit allows
  const unsigned long long s1 = (g + (unsigned long long)D - 1ull) % (unsigned long long)D;
  if (gtid == 0 && do_short) {
    e.hcount[(g + (unsigned long long)e.bin_lead) % (unsigned long long)D] = 0u;
    if (e.slot_emit) e.slot_emit[s1] = (uint16_t)e.d_emit;
  }
  // The leading nA blocks copy the row start and segment counts of the
  // previous step's spikes into the delay-major ring and take no items; nA
  // follows that step's spike count, the same in every block.
  unsigned long long c1 = 0;
  int nA = 0;
  // delay-major planes the later arrival items read: delays below d_emit
  const int planes = e.dcap < e.d_emit - 1 ? e.dcap : e.d_emit - 1;
  if (e.seg_cap > 0 && g >= 1ull && planes > 1 && do_short) {
    c1 = e.hcount[s1];
    if (c1 > (unsigned long long)e.hist_cap) c1 = (unsigned long long)e.hist_cap;
    if (c1 > (unsigned long long)e.seg_cap) c1 = (unsigned long long)e.seg_cap;
    const unsigned long long want = (c1 + kSegGroup - 1) / kSegGroup;
    // at most a 32nd of the grid: the copy overlaps the item blocks' work
    const int most = nblk >= 64 ? nblk / 32 : 1;  // the host launches >= 2 blocks
    nA = want < (unsigned long long)most ? (int)want : most;
  }
  if (bid < nA) {
    // Groups of 32 spikes: their segment-table rows are loaded at once (one
    // 16-byte vector of 8 delays per task, consecutive lanes on consecutive
    // spikes), transposed in shared memory to [delay][spike], and stored
    // plane by plane, 64 contiguous bytes per delay.
    const size_t cap = (size_t)e.seg_cap;
    const int dcap = e.dcap;
    const int nq_all = (planes + 7) >> 3;
    for (unsigned long long k0 = (unsigned long long)bid * kSegGroup; k0 < c1;
         k0 += (unsigned long long)nA * kSegGroup) {
      if (threadIdx.x < kSegGroup) {
        const unsigned long long k = k0 + threadIdx.x;
        const uint4* row = nullptr;
        int nq = 0;
        long long r0 = 0;
        if (k < c1) {
          const uint32_t ent = ld_ring<PERSIST>(e.hist + s1 * (unsigned long long)e.hist_cap + k);
          const int64_t gidx = (int64_t)(ent & 0x7FFFFFFFu);
          const int inst = SINGLE ? 0 : e.tile_info[gidx / kTile].x;
          if (inst >= 0) {
            const InstDesc& dd = e.insts[inst];
            if (dd.seg_kind == kSeg16) {
              const int64_t j = gidx - dd.base;
              r0 = __ldg(dd.row_ptr + j);
              row = reinterpret_cast<const uint4*>(seg_row(dd, j) + kSegHead);
              nq = (dd.dmax + 7) >> 3;
            }
          }
        }
        s_row[threadIdx.x] = row;
        s_nq[threadIdx.x] = nq;
        s_r0[threadIdx.x] = r0;
      }
      __syncthreads();
      for (int t = threadIdx.x; t < kSegGroup * nq_all; t += kDelThreads) {
        const int ks = t & (kSegGroup - 1), q = t / kSegGroup;
        const uint4 v = q < s_nq[ks] ? __ldg(s_row[ks] + q) : make_uint4(0u, 0u, 0u, 0u);
        const uint32_t wd[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
        for (int i = 0; i < 8; ++i)
          s_tab[(8 * q + i) * kSegGroup + ks] = (uint16_t)(wd[i >> 1] >> ((i & 1) * 16));
      }
      __syncthreads();
      // k0 + 31 < seg_cap (a multiple of 32): whole groups stay in the ring
      for (int t = threadIdx.x; t < planes * (kSegGroup / 2); t += kDelThreads) {
        const int dl = t / (kSegGroup / 2), w = t % (kSegGroup / 2);
        const uint32_t pair = *reinterpret_cast<const uint32_t*>(&s_tab[dl * kSegGroup + 2 * w]);
        uint32_t* H = reinterpret_cast<uint32_t*>(e.hseg + (s1 * (size_t)dcap + dl) * cap + k0);
        H[w] = pair;
      }
      if (threadIdx.x < kSegGroup) e.hr0[s1 * cap + k0 + threadIdx.x] = s_r0[threadIdx.x];
      __syncthreads();
    }
    return;
  }
  const int bB = bid - nA, nB = nblk - nA;  // item blocks

  // spikes handed on at step g - d for d = threadIdx.x + 1, and their
  // exclusive prefix
  const int dlim = e.dmax;
  unsigned long long c = 0;
  const int dme = threadIdx.x + 1;
  if (dme <= dlim && g >= (unsigned long long)dme && (dme == 1 ? do_short : do_long)) {
    const unsigned long long sl = (g - dme) % (unsigned long long)D;
    // delays at or above the threshold in force when that slot was handed
    // on went out at emission
    const int thr = dme == 1 ? e.d_emit : (e.slot_emit ? (int)e.slot_emit[sl] : D + 1);
    if (dme < thr) {
      const unsigned long long h = e.hcount[sl];
      c = h < (unsigned long long)e.hist_cap ? h : (unsigned long long)e.hist_cap;
    }
  }
  // Phases: the update appends each step's spikes roughly in tile order, so
  // a spike's rank in its slot follows its region.  Taking the items rank
  // phase by rank phase (phase q: ranks [q c/Q, (q+1) c/Q) of every delay's
  // slot) keeps the warps in flight on a narrow band of regions, so the
  // within-region edges (most of them) add into a slice of the accumulators
  // that stays in the L2 even when all of them do not fit (Q = 1 when they
  // do).
  const int Q = e.phases;
  s_cnt[threadIdx.x] = (uint32_t)c;
  unsigned long long incl[kMaxPhases], own[kMaxPhases];
#pragma unroll
  for (int q = 0; q < kMaxPhases; ++q) {
    own[q] = q < Q ? (q + 1ull) * c / (unsigned long long)Q - q * c / (unsigned long long)Q : 0ull;
    incl[q] = own[q];
    if (q < Q) {  // block-uniform
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const unsigned long long t = __shfl_up_sync(kFull, incl[q], o);
        if (lane >= o) incl[q] += t;
      }
    }
    if (lane == 31) s_wsum[q][warp] = incl[q];
  }
  __syncthreads();
  if (threadIdx.x < kMaxPhases) {  // warp offsets within each phase
    unsigned long long acc = 0;
    for (int w = 0; w < kDelThreads / 32; ++w) {
      const unsigned long long t = s_wsum[threadIdx.x][w];
      s_wsum[threadIdx.x][w] = acc;
      acc += t;
    }
    s_phase[threadIdx.x + 1] = acc;  // the phase's total, summed below
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    s_phase[0] = 0ull;
    for (int q = 0; q < kMaxPhases; ++q) s_phase[q + 1] += s_phase[q];
  }
#pragma unroll
  for (int q = 0; q < kMaxPhases; ++q) s_pre[q][threadIdx.x] = s_wsum[q][warp] + incl[q] - own[q];
  __syncthreads();
  const int nd = dlim < kDelThreads ? dlim : kDelThreads;  // delay buckets d = 1..nd
  // the emission range: every spike handed on at g - 1 times its delays
  // d_emit..dlim, spike-major so that consecutive lanes take consecutive
  // delays of one row (its segments lie end to end)
  const unsigned long long W_arr = s_phase[Q];
  const int ne = e.d_emit <= dlim ? dlim - e.d_emit + 1 : 0;
  unsigned long long c1e = 0;
  if (ne > 0 && g >= 1ull && do_short) {
    c1e = e.hcount[s1];
    if (c1e > (unsigned long long)e.hist_cap) c1e = (unsigned long long)e.hist_cap;
  }
  const unsigned long long W = W_arr + c1e * (unsigned long long)ne;
  const unsigned long long acc_elems = (unsigned long long)e.stride * (FOUR ? 2 : 1);
  const uint32_t aslot_now = acc_slot<true>(e, g), aslot_last = acc_slot<true>(e, g - 1ull);
  __syncthreads();

  const unsigned long long pol_rec = l2_policy_first(), pol_acc = l2_policy_last();
  const size_t cap = (size_t)e.seg_cap;
  // stage one: bucket (delay) by binary search over the prefix, then the
  // loads that need nothing else
  auto stage_one = [&](unsigned long long t, ItemLoads& p) {
    p.d = 0u;
    p.ring = false;
    if (t >= W) return;
    if (t >= W_arr) {  // emission: spike k of step g - 1, delay d, into slot g - 1 + d
      const unsigned long long te = t - W_arr;
      p.k = (uint32_t)(te / (unsigned long long)ne);
      p.d = (uint32_t)e.d_emit + (uint32_t)(te % (unsigned long long)ne);
      p.slot = (uint32_t)s1;
      p.aslot = aslot_last + p.d;  // (the ring is longer than any delay)
      if (p.aslot >= (uint32_t)e.acc_slots) p.aslot -= (uint32_t)e.acc_slots;
      p.ent = ld_ring<PERSIST>(e.hist + (size_t)p.slot * (size_t)e.hist_cap + p.k);
      return;
    }
    p.aslot = aslot_now;
    int q = 0;  // the phase: the largest q < Q with s_phase[q] <= t
    for (int step = kMaxPhases / 2; step > 0; step >>= 1)
      if (q + step < Q && s_phase[q + step] <= t) q += step;
    const unsigned long long tq = t - s_phase[q];
    int lo = 0, hi = nd - 1;
    while (lo < hi) {
      const int mid = (lo + hi + 1) >> 1;
      if (s_pre[q][mid] <= tq) lo = mid; else hi = mid - 1;
    }
    p.d = (uint32_t)lo + 1u;
    p.k = (uint32_t)((unsigned long long)q * s_cnt[lo] / (unsigned long long)Q + (tq - s_pre[q][lo]));
    p.slot = (uint32_t)((g - p.d) % (unsigned long long)D);
    p.ent = ld_ring<PERSIST>(e.hist + (size_t)p.slot * (size_t)e.hist_cap + p.k);
    if (p.d >= 2u && p.k < cap && g - p.d >= e.since) {  // from the delay-major ring (coalesced across lanes)
      p.ring = true;
      p.r0 = ld_ring<PERSIST>(e.hr0 + p.slot * cap + p.k);
      const uint16_t* H = e.hseg + ((size_t)p.slot * (size_t)e.dcap) * cap + p.k;
      p.a = ld_ring<PERSIST>(H + (size_t)(p.d - 2u) * cap);
      p.b = ld_ring<PERSIST>(H + (size_t)(p.d - 1u) * cap);
    }
  };
  // stage two: the item's edge segment [e0, e0 + nseg) from the stage-one
  // loads, or by the graph's own tables when the ring does not hold it
  // The synaptic events of a spike (its out-degree: Supp. Alg. 2 pushes
  // every out-edge once) are counted at its delay-1 item, which every spike
  // handed on has exactly once (arrival, or emission when every delay goes
  // at emission); the spikes handed on at the last step, not yet reached by
  // a delivery, are added when the counters are read (k_pending_events).
  unsigned long long ev = 0;
  auto stage_two = [&](const ItemLoads& p, int64_t& e0, uint32_t& nseg, int& inst, uint32_t& cls) {
    e0 = 0;
    nseg = 0u;
    inst = 0;
    cls = 0u;
    if (p.d == 0u) return;
    cls = p.aslot << 1;  // the accumulator slot travels with the class bit
    const int64_t gidx = (int64_t)(p.ent & 0x7FFFFFFFu);
    cls |= p.ent >> 31;
    if (!SINGLE) {
      inst = e.tile_info[gidx / kTile].x;
      if (inst < 0) {  // never for a listed spike: tiles are reused D steps late
        inst = 0;
        return;
      }
    }
    const InstDesc& dd = e.insts[inst];
    const uint32_t d = p.d;
    const int64_t j = gidx - dd.base;
    if (d == 1u) ev += (unsigned long long)(__ldg(dd.row_ptr + j + 1) - __ldg(dd.row_ptr + j));
    if ((int32_t)d > dd.dmax) return;
    int64_t r0, a, b;
    if (dd.seg_kind == kSeg16 && p.ring) {
      r0 = p.r0;
      a = (int64_t)p.a;
      b = (int64_t)p.b;
    } else if (dd.seg_kind == kSeg16) {
      r0 = __ldg(dd.row_ptr + j);
      const uint16_t* T = reinterpret_cast<const uint16_t*>(seg_row(dd, j) + kSegHead);
      a = d >= 2 ? (int64_t)__ldg(T + d - 2) : 0;
      b = (int64_t)__ldg(T + d - 1);
    } else if (dd.seg_kind == kSeg32) {
      r0 = __ldg(dd.row_ptr + j);
      const uint32_t* T = reinterpret_cast<const uint32_t*>(seg_row(dd, j) + kSegHead);
      a = d >= 2 ? (int64_t)__ldg(T + d - 2) : 0;
      b = (int64_t)__ldg(T + d - 1);
    } else {
      r0 = __ldg(dd.row_ptr + j);
      const int64_t r1 = __ldg(dd.row_ptr + j + 1);
      a = first_delay_at_least(dd.col, dd.delay, dd.shift, r0, r1, d) - r0;
      b = first_delay_at_least(dd.col, dd.delay, dd.shift, r0 + a, r1, d + 1) - r0;
    }
    nseg = (uint32_t)(b - a);
    e0 = r0 + a;
  };

  const unsigned long long wstride = (unsigned long long)nB * blockDim.x;
  const unsigned long long wbase = (unsigned long long)bB * blockDim.x + warp * 32;
  ItemLoads pend;
  stage_one(wbase + lane, pend);
  for (unsigned long long b0 = wbase; b0 < W; b0 += wstride) {  // warp-uniform
    int64_t e0;
    uint32_t nseg, cls;
    int inst;
    stage_two(pend, e0, nseg, inst, cls);
    // the next batch's loads fly while this batch's edges are walked
    stage_one(b0 + wstride + lane, pend);
    // the warp's segments laid end to end; consecutive lanes take
    // consecutive edges (coalesced), the owning item found by a shuffle search
    uint32_t incl = nseg;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const uint32_t x = __shfl_up_sync(kFull, incl, o);
      if (lane >= o) incl += x;
    }
    const uint32_t total = __shfl_sync(kFull, incl, 31);
    const uint32_t ex = incl - nseg;
    // instance (23 bits) | accumulator slot << 23 (8 bits) | class << 31
    const int icls = inst | (int)((cls >> 1) << 23) | (int)((cls & 1u) << 31);
    for (uint32_t f = 0; f < total; f += 32u * kWalkU) {  // warp-uniform
      uint32_t tg[kWalkU], wv[kWalkU];
      int ic[kWalkU];
      bool ok[kWalkU];
#pragma unroll
      for (int u = 0; u < kWalkU; ++u) {
        ok[u] = false;
        if (f + 32u * u < total) {  // warp-uniform
          const uint32_t fi = f + 32u * u + lane;
          int L = 0;
#pragma unroll
          for (int step = 16; step > 0; step >>= 1) {
            const int cand = L + step < 32 ? L + step : 31;
            const uint32_t v = __shfl_sync(kFull, ex, cand);
            if (L + step < 32 && v <= fi) L = cand;
          }
          const int64_t q0 = __shfl_sync(kFull, e0, L);
          const uint32_t qx = __shfl_sync(kFull, ex, L);
          ic[u] = __shfl_sync(kFull, icls, L);
          if (fi < total) {
            const InstDesc& dd = e.insts[SINGLE ? 0 : (ic[u] & 0x7FFFFF)];
            const int64_t ei = q0 + (int64_t)(fi - qx);
            if (FOUR && dd.two_w) {  // 8-byte record: word, weight | second weight << 16
              const uint2 r4 = ld_stream_u64(reinterpret_cast<const uint2*>(dd.rec) + ei, pol_rec);
              tg[u] = r4.x & dd.tmask;
              wv[u] = r4.y;
            } else if (dd.rec) {
              // 6-byte record at byte 6 ei: two aligned words cover it (the
              // record array carries 8 bytes of padding at its end)
              const size_t byte = 6 * (size_t)ei;
              const uint32_t* w4 = reinterpret_cast<const uint32_t*>(
                  reinterpret_cast<const unsigned char*>(dd.rec) + (byte & ~size_t(3)));
              const uint32_t w0 = ld_stream_u32(w4, pol_rec), w1 = ld_stream_u32(w4 + 1, pol_rec);
              const uint32_t sh = (uint32_t)(byte & 3u) * 8u;  // 0 or 16
              tg[u] = __funnelshift_r(w0, w1, sh) & dd.tmask;
              const uint32_t wb = (w1 >> sh) & 0xFFFFu;
              wv[u] = wb | (wb << 16);
            } else {
              tg[u] = __ldg(dd.col + ei) & dd.tmask;
              const uint32_t wb = __ldg(dd.w + ei);
              wv[u] = wb | (wb << 16);
            }
            ok[u] = true;
          }
        }
      }
#pragma unroll
      for (int u = 0; u < kWalkU; ++u) {
        if (!ok[u]) continue;
        const InstDesc& dd = e.insts[SINGLE ? 0 : (ic[u] & 0x7FFFFF)];
        const uint32_t qc = (uint32_t)ic[u] >> 31;
        int2* const accs = e.acc + (size_t)(((uint32_t)ic[u] >> 23) & 0xFFu) * acc_elems;
        const int q = __float2int_rn(__fmul_rn(__uint_as_float(wv[u] << 16), dd.two_S));
        if (FOUR) {
          const int q2 = __float2int_rn(__fmul_rn(__uint_as_float(wv[u] & 0xFFFF0000u), dd.two_S));
          unsigned long long* accp = reinterpret_cast<unsigned long long*>(accs) +
                                     2 * (size_t)(dd.base + (int64_t)tg[u]) + qc;
          red_add_u64(accp, ((unsigned long long)(uint32_t)q2 << 32) | (uint32_t)q, pol_acc);
        } else {
          int* accp = reinterpret_cast<int*>(accs + dd.base) + qc;
          red_add_s32(accp + 2 * (size_t)tg[u], q, pol_acc);
        }
      }
    }
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) ev += __shfl_down_sync(kFull, ev, o);
  if (lane == 0 && ev) atomicAdd(e.events, ev);
}

// A row in the bounds ring: first edge (47 bits), class, instance (16 bits).
constexpr unsigned long long kRowMask = (1ull << 47) - 1ull;
constexpr unsigned long long kNoRow = ~0ull;

// Windows delivery's loads of the spike and bounds rings and their counts.
// Never through the read-only path: the update that writes them may still run
// when these kernels start as its programmatic dependents, or is a part of the
// same launch in the persistent stepper.  Ordinary loads see the writes of the
// grids that griddepcontrol.wait waited for, and neighbouring items share
// sectors in the L1 (with loads from the L2: hmda_64x100k 130.4 -> 131.0 ms);
// the persistent stepper's blocks read from the L2.
template <bool PERSIST, typename T>
__device__ __forceinline__ T ld_step(const T* p) {
  return PERSIST ? __ldcg(p) : *p;
}

// The window bounds of step g - 1's spikes into the ring, one warp per spike,
// warps w0, w0 + n, ...: for the spike of rank k, its row into hr0[slot][k],
// and into hseg[slot][j][k] the number of its edges with delay below the
// first of window j (of W delays; the first window starts at the next
// multiple of W).  The items of later windows then read 12 bytes next to
// their neighbours' each, where the row and table look-ups of an item are
// three random DRAM accesses: at the 37 G a second measured for those, they
// cost more than the edges (of a window kernel of 285 us for 21.6 M edges,
// 128 us were left without its edge reads and reductions).  Counts the
// synaptic events of those spikes: the out-degree of each, once (Supp. Alg. 2
// pushes every out-edge once).
template <bool PERSIST>
__device__ __forceinline__ void copy_bounds(const EngineDev& e, unsigned long long g, uint32_t w0, uint32_t n,
                                            unsigned long long& ev) {
  if (g == 0ull) return;
  const int lane = threadIdx.x & 31;
  const uint32_t sl = (uint32_t)((g - 1ull) % (unsigned long long)e.D);
  const uint32_t h = ld_step<PERSIST>(e.hcount + sl);
  const uint32_t c = (int64_t)h < e.hist_cap ? h : (uint32_t)e.hist_cap, cap = (uint32_t)e.seg_cap;
  const int W = e.wmask + 1;
  const int first = W - (int)((unsigned)(g - 1ull) & (unsigned)e.wmask);  // delay at the next window's start
  for (uint32_t k = w0; k < c; k += n) {
    const uint32_t ent = ld_step<PERSIST>(e.hist + (size_t)sl * (size_t)e.hist_cap + k);
    const int64_t gidx = (int64_t)(ent & 0x7FFFFFFFu);
    const int inst = e.n_inst == 1 ? 0 : e.tile_info[gidx / kTile].x;
    unsigned long long packed = kNoRow;
    if (inst >= 0) {
      const InstDesc& dd = e.insts[inst];
      const unsigned char* row = seg_row(dd, gidx - dd.base);
      if (dd.seg_kind == kSeg16 && k < cap)
        for (int j = lane; j < e.dcap; j += 32) {
          const int d = first + j * W - 1;  // the last delay before window j
          e.hseg[(sl * (size_t)e.dcap + j) * cap + k] =
              (uint16_t)(d < 1 ? 0u : edges_up_to(dd, row, d < dd.dmax ? d : dd.dmax));
        }
      const longlong2 r = __ldg(reinterpret_cast<const longlong2*>(row));
      if (lane == 0) ev += (unsigned long long)(r.y - r.x);
      if (dd.seg_kind == kSeg16)
        packed = (unsigned long long)r.x | ((unsigned long long)(ent >> 31) << 47) | ((unsigned long long)inst << 48);
    }
    if (lane == 0 && k < cap) reinterpret_cast<unsigned long long*>(e.hr0)[sl * (size_t)cap + k] = packed;
  }
}

// kWindows: the arrivals of steps g .. g + W - 1, W = wmask + 1, from the
// spikes handed on before step g, as block bid of nblk; the block's threads
// call it together.  Bucket t holds the spikes of step g - 1 - t, and an item
// (a spike of bucket t) is the segment of its row with delays t + 1 .. t + W.
//
// Bound: random DRAM accesses (some 37 G a second measured) and the
// reductions into the accumulators (212 G/s while they lie in the L2, 34 to
// 58 G/s beyond).  A window of W delays reads a row in pieces W times as long
// as one step's would be, W times less often, so the items and the sectors
// that hold a piece's few records fall with W, and the accumulators grow with
// it: W = 4 / 2 / 1 measured 33.8 / 35.0 / 43.2 us a step at 2 M neurons and
// in-degree 1,000 (16 MB of accumulators per step; 45.3 us with one delay per
// step and kernel), 49.9 / 45.2 / 50.9 us at 5 M and 400 (40 MB; 60.2 us).
template <bool FOUR, bool SINGLE, bool PERSIST>
__device__ __forceinline__ void deliver_windows(const EngineDev& e, unsigned long long g, int bid, int nblk) {
  // items of phase q and bucket t start at s_pre[q][t] of the phase
  __shared__ uint32_t s_pre[kMaxPhases][256];
  __shared__ uint32_t s_wsum[kMaxPhases][kDelThreads / 32];
  __shared__ uint32_t s_items[kMaxPhases];     // of the phase
  __shared__ uint32_t s_unit[kMaxPhases + 1];  // warp units before the phase
  __shared__ uint32_t s_cnt[256];
  __shared__ int4 s_item[kDelThreads];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const unsigned long long D = (unsigned long long)e.D;
  const int W = e.wmask + 1;
  // the slots that the updates of this window fill (a bin later with spike
  // binning): their spikes' last arrivals lie before step g
  if (bid == 0 && (int)threadIdx.x < W && !e.keep_counts)
    e.hcount[(g + (unsigned long long)e.bin_lead + threadIdx.x) % D] = 0u;
  const uint32_t top = (uint32_t)((g + D - 1ull) % D);  // ring slot of step g - 1
  const auto ring_of = [&](int t) {                     // and of step g - 1 - t
    return top >= (uint32_t)t ? top - (uint32_t)t : top + (uint32_t)D - (uint32_t)t;
  };
  unsigned long long ev = 0;
  // buckets t0 .. t0 + nb - 1 at a time, so that their spikes count in 32 bits
  // (all of them at once up to some 20 M neurons)
  const int n_buckets = e.dmax;
  const int at_once = (int)min((long long)n_buckets, 0xFFFFFFC0ll / (long long)e.hist_cap);
  for (int t0 = 0; t0 < n_buckets; t0 += at_once) {
  const int nb = min(at_once, n_buckets - t0);
  uint32_t c = 0;
  const int tme = threadIdx.x;
  if (tme < nb && g >= (unsigned long long)(t0 + tme) + 1ull) {
    const uint32_t sl = ring_of(t0 + tme);
    const uint32_t h = ld_step<PERSIST>(e.hcount + sl);
    c = (int64_t)h < e.hist_cap ? h : (uint32_t)e.hist_cap;
  }
  // Phases: the update appends each step's spikes roughly in tile order, so
  // a spike's rank in its slot follows its region.  Taking the items rank
  // phase by rank phase (phase q: ranks [q c/Q, (q+1) c/Q) of every slot)
  // keeps the warps in flight on a narrow band of regions, so the
  // within-region edges (most of them) add into a slice of the accumulators
  // that stays in the L2 even when all of them do not fit.
  const int Qb = e.phases > 1 ? 3 : 0, Q = 1 << Qb;
  s_cnt[threadIdx.x] = c;
  uint32_t incl[kMaxPhases], own[kMaxPhases];
#pragma unroll
  for (int q = 0; q < kMaxPhases; ++q) {
    own[q] = q < Q ? (uint32_t)(((q + 1ull) * c >> Qb) - ((unsigned long long)q * c >> Qb)) : 0u;
    incl[q] = own[q];
    if (q < Q) {  // block-uniform
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const uint32_t t = __shfl_up_sync(kFull, incl[q], o);
        if (lane >= o) incl[q] += t;
      }
    }
    if (lane == 31) s_wsum[q][warp] = incl[q];
  }
  __syncthreads();
  if (threadIdx.x < kMaxPhases) {  // warp offsets within each phase
    uint32_t acc = 0;
    for (int w = 0; w < kDelThreads / 32; ++w) {
      const uint32_t t = s_wsum[threadIdx.x][w];
      s_wsum[threadIdx.x][w] = acc;
      acc += t;
    }
    s_items[threadIdx.x] = acc;
  }
  __syncthreads();
  // items per unit: 32, or fewer when that would leave some warps with one and
  // others with two (100 -> 93 us a step at 4 M neurons with 50,000 spikes of
  // 100 edges)
  uint32_t all = 0;
  for (int q = 0; q < Q; ++q) all += s_items[q];
  int ub = 5;
  while (ub > 0 && (all >> ub) < 2u * (uint32_t)nblk * (kDelThreads / 32)) --ub;
  if (threadIdx.x == 0) {
    s_unit[0] = 0u;
    for (int q = 0; q < kMaxPhases; ++q) s_unit[q + 1] = s_unit[q] + ((s_items[q] + (1u << ub) - 1u) >> ub);
  }
#pragma unroll
  for (int q = 0; q < kMaxPhases; ++q) s_pre[q][threadIdx.x] = s_wsum[q][warp] + incl[q] - own[q];
  __syncthreads();
  const uint32_t n_units = s_unit[kMaxPhases];
  const unsigned long long pol_rec = l2_policy_first(), pol_acc = l2_policy_last();

  // A unit of 8 to 32 items is four runs of consecutive ones, a quarter of
  // the phase apart: the buckets hold segments of very different lengths
  // (short delays within a region, long ones across), so every unit gets an
  // even share, and a run's bounds lie side by side in the ring.
  struct Item {
    unsigned long long row;  // packed row of the bounds ring, kNoRow: not there
    uint32_t a, b, k;
    int t;  // bucket, -1: none
  };
  const uint32_t cap = (uint32_t)e.seg_cap;
  auto fetch = [&](uint32_t u) {
    Item it{kNoRow, 0u, 0u, 0u, -1};
    if (u >= n_units || lane >= (1 << ub)) return it;
    int q = 0;  // the phase: the largest q < Q with s_unit[q] <= u
    for (int step = kMaxPhases / 2; step > 0; step >>= 1)
      if (q + step < Q && s_unit[q + step] <= u) q += step;
    const uint32_t U = s_unit[q + 1] - s_unit[q], v = u - s_unit[q];
    const int rb = ub >= 3 ? ub - 2 : ub;  // a run's length, or the unit's
    const uint32_t x = ((uint32_t)lane >> rb) * (U << rb) + (v << rb) + (lane & ((1 << rb) - 1));
    if (x >= s_items[q]) return it;
    int lo = 0;  // the bucket: the largest with s_pre[q][lo] <= x
#pragma unroll
    for (int step = 128; step > 0; step >>= 1)
      if (lo + step < nb && s_pre[q][lo + step] <= x) lo += step;
    it.k = (uint32_t)((unsigned long long)q * s_cnt[lo] >> Qb) + (x - s_pre[q][lo]);
    it.t = t0 + lo;
    if (it.t > 0 && it.k < cap && g - 1ull - (unsigned long long)it.t >= e.since) {  // window it.t / W of its slot
      const size_t sl = ring_of(it.t);
      const uint16_t* B = e.hseg + (sl * (size_t)e.dcap + (uint32_t)it.t / (uint32_t)W) * cap + it.k;
      it.row = ld_step<PERSIST>(reinterpret_cast<const unsigned long long*>(e.hr0) + sl * cap + it.k);
      it.a = ld_step<PERSIST>(B);
      it.b = ld_step<PERSIST>(B + cap);
    }
    return it;
  };
  // an item's segment: from the ring, or from its row of the segment table
  auto resolve = [&](const Item& it, int64_t& e0, uint32_t& n, int& inst, uint32_t& key) {
    e0 = 0;
    n = 0u;
    inst = 0;
    key = 0u;
    if (it.t < 0) return;
    const int d0 = it.t + 1;
    key = (uint32_t)(g - (unsigned long long)d0) << 1;
    if (it.row != kNoRow) {
      e0 = (int64_t)(it.row & kRowMask) + it.a;
      n = it.b - it.a;
      inst = SINGLE ? 0 : (int)(it.row >> 48);
      key |= (uint32_t)(it.row >> 47) & 1u;
      return;
    }
    const uint32_t ent = ld_step<PERSIST>(e.hist + (size_t)ring_of(it.t) * (size_t)e.hist_cap + it.k);
    const int64_t gidx = (int64_t)(ent & 0x7FFFFFFFu);
    key |= ent >> 31;
    if (!SINGLE) {
      inst = e.tile_info[gidx / kTile].x;
      if (inst < 0) {  // never for a listed spike: tiles are reused D steps late
        inst = 0;
        return;
      }
    }
    const InstDesc& dd = e.insts[inst];
    const int d1 = it.t + W < dd.dmax ? it.t + W : dd.dmax;
    const unsigned char* row = seg_row(dd, gidx - dd.base);
    const longlong2 r = __ldg(reinterpret_cast<const longlong2*>(row));
    if (cap == 0u && it.t < W && g - (unsigned long long)d0 >= e.since) ev += (unsigned long long)(r.y - r.x);
    if (d0 > d1) return;
    const uint32_t a = d0 >= 2 ? edges_up_to(dd, row, d0 - 1) : 0u;
    e0 = r.x + a;
    n = (d1 == dd.dmax ? (uint32_t)(r.y - r.x) : edges_up_to(dd, row, d1)) - a;
  };
  const uint32_t stride = (uint32_t)nblk * (kDelThreads / 32);
  uint32_t u = (uint32_t)bid * (kDelThreads / 32) + warp;
  Item next = fetch(u);
  for (; u < n_units; u += stride) {  // warp-uniform
    const Item it = next;
    next = fetch(u + stride);  // its loads fly while this unit's edges are walked
    int64_t e0;
    uint32_t n, key;
    int inst;
    resolve(it, e0, n, inst, key);
    walk_segments<FOUR, SINGLE>(e, e.insts, s_item + warp * 32, e0, n, inst, key, pol_rec, pol_acc);
  }
  __syncthreads();
  }
  if (e.seg_cap > 0)
    copy_bounds<PERSIST>(e, g, (uint32_t)bid * (kDelThreads / 32) + warp, (uint32_t)nblk * (kDelThreads / 32), ev);
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) ev += __shfl_down_sync(kFull, ev, o);
  if (lane == 0 && ev) atomicAdd(e.events, ev);
}

// kWindows, inside a window: the edges of the spikes handed on at step g - 1
// that come due by the window's end, the start of their rows.  A warp takes 32
// of the spikes, or fewer when that would leave warps without one; four
// dependent loads (count, ring entry, table row, records) bound it.
template <bool FOUR, bool SINGLE, bool PERSIST>
__device__ __forceinline__ void deliver_rest(const EngineDev& e, unsigned long long g, int bid, int nblk,
                                             int4* s_item) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int left = e.wmask + 1 - (int)((unsigned)g & (unsigned)e.wmask);  // steps to the window's end
  const uint32_t sl = (uint32_t)((g - 1ull) % (unsigned long long)e.D);
  const uint32_t h = ld_step<PERSIST>(e.hcount + sl);
  const uint32_t c = (int64_t)h < e.hist_cap ? h : (uint32_t)e.hist_cap;
  const uint32_t warps = (uint32_t)nblk * (kDelThreads / 32);
  int ub = 5;
  while (ub > 0 && (c >> ub) < 2u * warps) --ub;
  const uint32_t n_units = (uint32_t)(((unsigned long long)c + (1u << ub) - 1u) >> ub);
  for (uint32_t u = (uint32_t)bid * (kDelThreads / 32) + warp; u < n_units; u += warps) {
    const uint32_t k = (u << ub) + lane;
    int64_t e0 = 0;
    uint32_t nseg = 0, key = 0;
    int inst = 0;
    if (lane < (1 << ub) && k < c) {
      const uint32_t ent = ld_step<PERSIST>(e.hist + (size_t)sl * (size_t)e.hist_cap + k);
      const int64_t gidx = (int64_t)(ent & 0x7FFFFFFFu);
      if (!SINGLE) inst = e.tile_info[gidx / kTile].x;
      if (inst >= 0) {
        const InstDesc& dd = e.insts[inst];
        const unsigned char* row = seg_row(dd, gidx - dd.base);
        const longlong2 r = __ldg(reinterpret_cast<const longlong2*>(row));
        e0 = r.x;
        nseg = left < dd.dmax ? edges_up_to(dd, row, left) : (uint32_t)(r.y - r.x);
        key = ((uint32_t)(g - 1ull) << 1) | (ent >> 31);
      } else {
        inst = 0;
      }
    }
    walk_segments<FOUR, SINGLE>(e, e.insts, s_item + warp * 32, e0, nseg, inst, key, l2_policy_first(),
                                l2_policy_last());
  }
  if (e.seg_cap == 0) return;
  unsigned long long ev = 0;
  copy_bounds<PERSIST>(e, g, (uint32_t)bid * (kDelThreads / 32) + warp, warps, ev);
  if (lane == 0 && ev) atomicAdd(e.events, ev);
}

template <bool FOUR, bool SINGLE>
__global__ void __launch_bounds__(kDelThreads, 4) k_windows(EngineDev e, StepRef sr) {
  step_after();
  deliver_windows<FOUR, SINGLE, false>(e, step_of(sr), blockIdx.x, gridDim.x);
}

template <bool FOUR, bool SINGLE>
__global__ void __launch_bounds__(kDelThreads, 4) k_rest(EngineDev e, StepRef sr) {
  __shared__ int4 s_item[kDelThreads];
  step_after();
  deliver_rest<FOUR, SINGLE, false>(e, step_of(sr), blockIdx.x, gridDim.x, s_item);
}

template <bool FOUR, bool SINGLE>
__global__ void __launch_bounds__(kDelThreads, 4) k_deliver(EngineDev e, StepRef sr, int part) {
  deliver_body<FOUR, SINGLE, false>(e, sr, part, blockIdx.x, gridDim.x);
}

__device__ __forceinline__ unsigned long long global_ns() {
  unsigned long long t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}

__device__ __forceinline__ unsigned ld_acquire_u32(const unsigned* a) {
  unsigned v;
  asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(a) : "memory");
  return v;
}

__device__ __forceinline__ void red_release_add_u32(unsigned* a, unsigned v) {
  asm volatile("red.release.gpu.global.add.u32 [%0], %1;" ::"l"(a), "r"(v) : "memory");
}

// Grid-wide barrier of a cooperative launch.  After a block barrier (which
// orders the block's earlier writes before thread 0's), thread 0 of every
// block adds one to *count with device-scope release semantics and polls it
// with acquire loads until it reaches target (the blocks of the grid times
// the barriers passed, counting this one); the block barrier after the wait
// orders the block's later reads after the acquire.  The wait is bounded:
// after limit_ns of the global timer, or as soon as another block has given
// up (kFlagTimeout set in *flags), it gives up too, sets kFlagTimeout, and
// every thread of the block gets false.
__device__ __forceinline__ void grid_arrive(unsigned* count) {
  __syncthreads();
  if (threadIdx.x == 0) red_release_add_u32(count, 1u);
}

__device__ bool grid_wait(unsigned* count, unsigned target, unsigned long long limit_ns, unsigned* flags) {
  __shared__ int s_ok;
  if (threadIdx.x == 0) {
    int ok = 1;
    const unsigned long long t0 = global_ns();
    for (unsigned spin = 0; (int)(ld_acquire_u32(count) - target) < 0; ++spin) {
      if ((spin & 15u) != 15u) continue;  // the flag and the clock every 16 polls
      if (*reinterpret_cast<volatile unsigned*>(flags) & kFlagTimeout) {
        ok = 0;
        break;
      }
      if (global_ns() - t0 > limit_ns) {
        atomicOr(flags, kFlagTimeout);
        ok = 0;
        break;
      }
    }
    s_ok = ok;
  }
  __syncthreads();
  return s_ok != 0;
}

__device__ __forceinline__ bool grid_barrier(unsigned* count, unsigned target, unsigned long long limit_ns,
                                             unsigned* flags) {
  grid_arrive(count);
  return grid_wait(count, target, limit_ns, flags);
}

// Whether the instance of a tile (its tile_info) has steps to run from
// iteration g0 on.  Where not, nothing of it is read: a server may have given
// its constants and graph to the next request while a launch is in flight.
__device__ __forceinline__ bool runs_from(const EngineDev& e, const int4& ti, unsigned long long g0) {
  return ti.x >= 0 && e.dyn[ti.x].active != 0 && (long long)(g0 - e.insts[ti.x].g0) < e.insts[ti.x].n_end;
}

// by the tile's 256 threads, a block barrier after it; g0: the launch's first
// iteration
__device__ __forceinline__ void held_load(const EngineDev& e, int tile, unsigned long long g0, HeldTile& h) {
  if (tile >= e.n_tiles) return;
  const int4 ti = __ldg(e.tile_info + tile);
  if (!runs_from(e, ti, g0)) return;
  const InstDesc& d = e.insts[ti.x];
  const int t = threadIdx.x % (kTile / 4);
  const uint32_t* from = reinterpret_cast<const uint32_t*>(&d);
  for (int w = t; w < (int)(sizeof(InstDesc) / 4); w += kTile / 4) reinterpret_cast<uint32_t*>(&h.d)[w] = from[w];
  if (e.mode == kAtEmission) {
    const int32_t lo = (int32_t)((int64_t)tile * kTile - d.base);
    const int rows = d.N - lo < kTile ? d.N - lo : kTile;
    const int64_t r0 = d.row_ptr[lo];
    const bool fits = (unsigned long long)(d.row_ptr[lo + rows] - r0) < (1ull << 32);
    if (t == 0) h.row0 = fits ? r0 : -1;
    for (int k = t; k <= rows; k += kTile / 4) h.row[k] = (uint32_t)(d.row_ptr[lo + k] - r0);
  }
  if (ti.z > kHeldRegions) return;
  from = reinterpret_cast<const uint32_t*>(d.rc + ti.y);
  for (int w = t; w < ti.z * (int)(sizeof(RegionConst) / 4); w += kTile / 4)
    reinterpret_cast<uint32_t*>(h.rc)[w] = from[w];
}

// A warp's 128 neurons with their state in registers over many steps.
template <bool EXT, bool FOUR>
struct HeldWarp {
  WarpPlace w;
  QuadState q;
  QuadConst<true, true> one;
  QuadConst<false, true> each;
  QuadDraw draw;
  const InstDesc* d;
  const HeldTile* tile;
  bool ou;

  __device__ __forceinline__ HeldWarp(const EngineDev& e, int t, int warp, unsigned long long g0, const HeldTile& h)
      : tile(&h) {
    w.inst = -1;
    w.m = w.r0 = w.nr = 0;
    w.li0 = 0;
    w.gi0 = (int64_t)t * kTile + warp * 128 + (threadIdx.x & 31) * 4;
    if (t < e.n_tiles) {
      quad_load(e, w.gi0, q);
      const int4 ti = __ldg(e.tile_info + t);
      if (runs_from(e, ti, g0)) w.inst = ti.x;
      w.r0 = ti.y;
      w.nr = ti.z;
    }
    d = &h.d;
    ou = false;
    if (w.inst >= 0) {
      one.p = each.p = w.nr <= kHeldRegions ? h.rc : d->rc + w.r0;
      w.li0 = (int32_t)(w.gi0 - d->base);
      w.m = d->N - w.li0 < 4 ? d->N - w.li0 : 4;
      if (w.nr > 1) each.find(w.li0, w.m);
      ou = EXT && (d->ext & kExtOU);
      if (ou) q.B = __ldcs(reinterpret_cast<const float4*>(e.Ibg + w.gi0));
    }
  }
  // the random draws of iteration g
  __device__ __forceinline__ void prepare(unsigned long long g) {
    if (w.m <= 0) return;
    const long long n = (long long)(g - d->g0);
    draw = w.nr == 1 ? quad_draw<EXT>(*d, one, w.li0, n) : quad_draw<EXT>(*d, each, w.li0, n);
  }
  // iteration g, prepared; the whole warp
  __device__ __forceinline__ void step(const EngineDev& e, unsigned long long g, int4* s_item) {
    if (w.inst < 0) return;  // warp-uniform, as the next
    const long long n = (long long)(g - d->g0);
    if (n >= d->n_end) return;
    QuadSpikes qs;
    if (w.m > 0) {
      constexpr int kA = FOUR ? 4 : 2;
      int4* const accs = reinterpret_cast<int4*>(acc_of<false>(e, g)) + (FOUR ? w.gi0 : w.gi0 / 2);
      int4 A[kA];
#pragma unroll
      for (int k = 0; k < kA; ++k) A[k] = __ldcg(accs + k);
#pragma unroll
      for (int k = 0; k < kA; ++k) accs[k] = make_int4(0, 0, 0, 0);
      qs = w.nr == 1 ? quad_step<EXT, FOUR, true, true>(e, *d, one, w.m, w.gi0, w.li0, draw, q, A)
                     : quad_step<EXT, FOUR, false, true>(e, *d, each, w.m, w.gi0, w.li0, draw, q, A);
    }
    __syncwarp();
    warp_spikes<FOUR>(e, *d, w, g, n, qs, s_item, tile);
  }
  __device__ __forceinline__ void store(const EngineDev& e) {
    if (w.m <= 0) return;
    __stcs(reinterpret_cast<float4*>(e.V + w.gi0), q.V);
#pragma unroll
    for (int u = 0; u < 4; ++u) __stcs(reinterpret_cast<float4*>(e.J + u * e.stride + w.gi0), q.J[u]);
    __stcs(reinterpret_cast<uchar4*>(e.ref + w.gi0), q.ref);
    if (ou) __stcs(reinterpret_cast<float4*>(e.Ibg + w.gi0), q.B);
  }
};

// The persistent stepper: iterations g0 .. g0 + nsteps - 1 in one
// cooperative launch, each the delivery where the mode has one (the whole
// grid) and the update (tiles dealt round robin over the blocks), with a grid
// barrier after each.  The same device functions as the launched step do
// the work, so the results are identical bit for bit; a barrier that gives
// up ends the launch (kFlagTimeout stays set for the host).
template <bool EXT, bool FOUR, bool SINGLE, bool PER_STEP, bool HELD>
__global__ void __launch_bounds__(kDelThreads, 2)
    k_persist(EngineDev e, unsigned long long g0, int nsteps, unsigned* count,
              unsigned long long limit_ns) {
  __shared__ int4 s_item[kDelThreads];
  const int warp = threadIdx.x >> 5;
  unsigned target = 0;
  __shared__ HeldTile s_tile;
  if (HELD) {
    held_load(e, blockIdx.x, g0, s_tile);
    __syncthreads();
  }
  HeldWarp<EXT, FOUR> h(e, HELD ? (int)blockIdx.x : e.n_tiles, warp, g0, s_tile);
  if (HELD) h.prepare(g0);
  for (int s = 0; s < nsteps; ++s) {
    const unsigned long long g = g0 + (unsigned long long)s;
    const StepRef sr{nullptr, g, nullptr};
    const bool due = PER_STEP || (e.mode == kWindows && (!e.push_now || ((unsigned)g & (unsigned)e.wmask) == 0u));
    if (due) {
      if (PER_STEP) deliver_body<FOUR, SINGLE, true>(e, sr, kPartAll, blockIdx.x, gridDim.x);
      else if (((unsigned)g & (unsigned)e.wmask) == 0u)
        deliver_windows<FOUR, SINGLE, true>(e, g, blockIdx.x, gridDim.x);
      else deliver_rest<FOUR, SINGLE, true>(e, g, blockIdx.x, gridDim.x, s_item);
      target += gridDim.x;
      if (!grid_barrier(count, target, limit_ns, e.flags)) return;
    }
    // the last blocks: the first ones have the most tiles
    close_regions(e, g, (gridDim.x - 1 - blockIdx.x) * (kDelThreads / 32) + warp, gridDim.x * (kDelThreads / 32));
    target += gridDim.x;
    if (HELD) {
      h.step(e, g, s_item);
      grid_arrive(count);
      h.prepare(g + 1ull);  // under the barrier
      if (!grid_wait(count, target, limit_ns, e.flags)) return;
    } else {
      for (int t = blockIdx.x; t < e.n_tiles; t += gridDim.x)
        update_warp<EXT, FOUR>(e, sr, t, warp, s_item);
      if (!grid_barrier(count, target, limit_ns, e.flags)) return;
    }
  }
  if (HELD) h.store(e);
}

// The resident stepper of small networks (kAtEmission, at most 64 tiles):
// iterations g0 .. g0 + nsteps - 1 in one launch of one thread-block cluster
// of at most 16 blocks, each holding the state of its THREADS / 256 tiles in
// registers.  A step is the arrivals' load from the L2, the membrane step,
// the rows of the step's spikes and one hardware cluster barrier, under which
// the next step's random draws are made; nothing else leaves the registers,
// and nothing is launched between steps.
//
// Bound: the latency of that chain, not traffic.  4.4 us a step at 10,000
// neurons and 8 spikes a step (2.0 the arrivals, the membrane step and the
// barrier, some 2 the spikes' rows, 0.4 the bins), 6.6 at 30,000 and 9.1 at
// 60,000 (four tiles a block: 64 registers, spills); with a launch per step
// 7.4, 12.4 and 14, and 13.2, 25 and 27 with two.  The grid barrier of the
// persistent stepper costs 1.1 to 1.2 us by itself.  Constants and row starts
// in registers' reach (HeldTile) took 0.6 us off, a region's two powers on two
// lanes and the short way for a lone spike 0.7.  The warps of all blocks close
// the bins, 16 regions each: with those of one block 1,000 regions of ten
// neurons took 18.5 us a step, now 9.3 (1 ms steps: 110, now 36.8).
template <bool EXT, bool FOUR, int THREADS>
__global__ void __launch_bounds__(THREADS, 1) k_resident(EngineDev e, unsigned long long g0, int nsteps) {
  __shared__ int4 s_item[THREADS];
  const int warp = threadIdx.x >> 5;
  __shared__ HeldTile s_tile[THREADS / (kTile / 4)];
  const int tile = blockIdx.x * (THREADS / (kTile / 4)) + warp / kTileWarps;
  held_load(e, tile, g0, s_tile[warp / kTileWarps]);
  __syncthreads();
  HeldWarp<EXT, FOUR> h(e, tile, warp % kTileWarps, g0, s_tile[warp / kTileWarps]);
  // the last blocks close the bins, for they have the fewest tiles
  const auto close = [&](unsigned long long g) {
    close_regions(e, g, (gridDim.x - 1 - blockIdx.x) * (THREADS / 32) + warp, gridDim.x * (THREADS / 32));
  };
  h.prepare(g0);
  for (int s = 0; s < nsteps; ++s) {
    const unsigned long long g = g0 + (unsigned long long)s;
    h.step(e, g, s_item);
    close(g);
    __syncwarp();
    asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
    h.prepare(g + 1ull);
    __syncwarp();
    asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
  }
  close(g0 + (unsigned long long)nsteps);
  h.store(e);
}

// The grid barrier alone, rounds times, with extra arrivals expected per
// round that no block makes when extra > 0 (the wait then runs out).
__global__ void k_barrier_probe(unsigned* count, unsigned extra, int rounds,
                                unsigned long long limit_ns, unsigned* flags) {
  unsigned target = 0;
  for (int r = 0; r < rounds; ++r) {
    target += gridDim.x + extra;
    if (!grid_barrier(count, target, limit_ns, flags)) return;
  }
}

// BF16 bit pattern of staged weight e (float32 rounded to nearest even, or
// taken as given), with the rounding and range checks of ingest.
__device__ __forceinline__ uint16_t staged_bf16(const void* w_in, int32_t w_dtype, int64_t e,
                                                unsigned& err, unsigned& wmax) {
  uint16_t wb;
  if (w_dtype == 1) {
    wb = static_cast<const uint16_t*>(w_in)[e];
  } else {
    const float f = static_cast<const float*>(w_in)[e];
    const uint32_t u = __float_as_uint(f);
    const uint32_t r = u + 0x7FFFu + ((u >> 16) & 1u);  // round to nearest even
    wb = (uint16_t)(r >> 16);
    if ((uint32_t)wb << 16 != u) err |= kErrRounded;
  }
  const uint32_t wu = (uint32_t)wb << 16;
  const float wf = __uint_as_float(wu);
  if (!(wf >= 0.0f) || isinf(wf)) err |= kErrWeight;
  else wmax = max(wmax, wu);
  return wb;
}

// Ingest rows [j0, j1) of a graph from staging arrays that hold its edges
// from e_base on: warp per source row.  Checks every edge (target range,
// delay >= 1 and non-decreasing within the row, weights finite and
// non-negative after rounding to BF16), counts in-degrees, and writes
//   rec[3e .. 3e+2] = word low 16 bits, word high 16 bits, BF16 weight
//   (word: target | delay << shift, the delay's bits that fit)
//   (with second weights w2_in: rec[4e .. 4e+3], the second weight last)
//   row j of the segment table: first and last edge, then for k < dmax the
//   number of edges with delay <= k + 1
// (the segment table must be zero on entry; entries below the row's first
// delay stay zero).
__global__ void k_ingest(int32_t N, int32_t j0, int32_t j1, int64_t e_base,
                         const int64_t* __restrict__ row_ptr, const int32_t* __restrict__ col_in,
                         const void* __restrict__ w_in, const void* __restrict__ w2_in,
                         int32_t w_dtype, const uint8_t* __restrict__ delay_in,
                         uint16_t* __restrict__ rec, int32_t shift,
                         int32_t dmax, int32_t seg_bytes, void* seg, int32_t kind,
                         int32_t* indeg, unsigned* wmax_bits, unsigned* err) {
  const int lane = threadIdx.x & 31;
  const int64_t warp = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const int64_t nwarps = ((int64_t)gridDim.x * blockDim.x) >> 5;
  unsigned my_err = 0, my_wmax = 0;
  for (int64_t j = j0 + warp; j < j1; j += nwarps) {
    const int64_t a = row_ptr[j] - e_base, b = row_ptr[j + 1] - e_base;
    for (int64_t e = a + lane; e < b; e += 32) {
      const int32_t t = col_in[e];
      const unsigned d = delay_in[e];
      if (t < 0 || t >= N) my_err |= kErrTarget;
      if (d < 1u) my_err |= kErrDelayRange;
      if (e > a && delay_in[e - 1] > d) my_err |= kErrDelayOrder;
      const uint16_t wb = staged_bf16(w_in, w_dtype, e, my_err, my_wmax);
      const uint32_t tu = (uint32_t)t | (shift < 32 ? (uint32_t)d << shift : 0u);
      if (w2_in) {
        const uint16_t wb2 = staged_bf16(w2_in, w_dtype, e, my_err, my_wmax);
        reinterpret_cast<uint2*>(rec)[e_base + e] = make_uint2(tu, (uint32_t)wb | ((uint32_t)wb2 << 16));
      } else {
        uint16_t* r3 = rec + 3 * (e_base + e);
        r3[0] = (uint16_t)(tu & 0xFFFFu);
        r3[1] = (uint16_t)(tu >> 16);
        r3[2] = wb;
      }
      if (t >= 0 && t < N) atomicAdd(indeg + t, 1);
    }
    // segment counts: edge p closes the delays from its own to the next edge's
    const int64_t n = b - a;
    unsigned char* row = static_cast<unsigned char*>(seg) + j * (int64_t)seg_bytes;
    if (lane == 0) *reinterpret_cast<longlong2*>(row) = make_longlong2(row_ptr[j], row_ptr[j + 1]);
    uint16_t* T16 = reinterpret_cast<uint16_t*>(row + kSegHead);
    uint32_t* T32 = reinterpret_cast<uint32_t*>(row + kSegHead);
    for (int64_t p = lane; p < n; p += 32) {
      const int dp = (int)delay_in[a + p];
      const int dn = p + 1 < n ? (int)delay_in[a + p + 1] : dmax + 1;
      const int k0 = dp - 1 > 0 ? dp - 1 : 0;
      const int k1 = dn - 2 < dmax - 1 ? dn - 2 : dmax - 1;  // malformed rows fail creation
      for (int k = k0; k <= k1; ++k) {
        if (kind == kSeg16) T16[k] = (uint16_t)(p + 1);
        else T32[k] = (uint32_t)(p + 1);
      }
    }
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    my_err |= __shfl_xor_sync(kFull, my_err, o);
    my_wmax = max(my_wmax, __shfl_xor_sync(kFull, my_wmax, o));
  }
  if (lane == 0) {
    if (my_err) atomicOr(err, my_err);
    atomicMax(wmax_bits, my_wmax);
  }
}

// Out-degree sum of the spikes handed on at steps [r0, r1] (the ones no
// delivery has reached yet when the counters are read), into *out.
__global__ void k_pending_events(EngineDev e, long long r0, long long r1, unsigned long long* out) {
  unsigned long long ev = 0;
  for (long long r = r0 < 0 ? 0 : r0; r <= r1; ++r) {
    const unsigned long long slot = (unsigned long long)r % (unsigned long long)e.D;
    unsigned long long c = e.hcount[slot];
    if (c > (unsigned long long)e.hist_cap) c = (unsigned long long)e.hist_cap;
    for (unsigned long long k = (unsigned long long)blockIdx.x * blockDim.x + threadIdx.x; k < c;
         k += (unsigned long long)gridDim.x * blockDim.x) {
      const uint32_t ent = e.hist[slot * (unsigned long long)e.hist_cap + k];
      const int64_t gidx = (int64_t)(ent & 0x7FFFFFFFu);
      const int inst = e.n_inst == 1 ? 0 : e.tile_info[gidx / kTile].x;
      if (inst < 0) continue;
      const InstDesc& dd = e.insts[inst];
      const int64_t j = gidx - dd.base;
      ev += (unsigned long long)(dd.row_ptr[j + 1] - dd.row_ptr[j]);
    }
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) ev += __shfl_down_sync(kFull, ev, o);
  if ((threadIdx.x & 31) == 0 && ev) atomicAdd(out, ev);
}

__global__ void k_max_reduce(const int32_t* __restrict__ a, int64_t n, unsigned* out) {
  unsigned m = 0;
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n;
       i += (int64_t)gridDim.x * blockDim.x)
    m = max(m, (unsigned)a[i]);
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) m = max(m, __shfl_xor_sync(kFull, m, o));
  if ((threadIdx.x & 31) == 0) atomicMax(out, m);
}

int g_deliver_grid = 0;

}  // namespace

void launch_init_state(const EngineDev& e, int inst, int n_tiles_inst, int first_tile,
                       cudaStream_t s) {
  if (n_tiles_inst > 0) k_init_state<<<n_tiles_inst, kTile / 4, 0, s>>>(e, inst, first_tile);
}

namespace {

// A step kernel's launch.  Up to 2,048 tiles it need not wait for its
// predecessor on the stream to end (step_after in the kernel does): that
// took a step of 2 M neurons from 54.7 to 53.1 us and one of 500,000 in
// columns from 19.2 to 18.4; at 4 and 5 M neurons it cost one of 98 us 1.2.
// Per-step delivery keeps plain launches: its kernels' shares are what the
// autotuner compares, a candidate by itself.
template <class... Par, class... Arg>
void launch_after(void (*k)(Par...), int grid, int threads, cudaStream_t s, const EngineDev& e, Arg... arg) {
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3(grid);
  cfg.blockDim = dim3(threads);
  cfg.stream = s;
  cudaLaunchAttribute at{};
  at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at.val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = &at;
  cfg.numAttrs = e.mode != kPerStep && e.n_tiles <= 2048 ? 1 : 0;
  cudaLaunchKernelEx(&cfg, k, e, arg...);  // (errors by cudaGetLastError, as for <<<>>>)
}

}  // namespace

// The update's variant with the kExt* terms: they act only on instances that
// have them, and it takes accumulator rings of any length.
static bool ext_variant(const EngineDev& e) { return e.any_ext || (e.acc_slots & (e.acc_slots - 1)) != 0; }

void launch_update(const EngineDev& e, StepRef sr, cudaStream_t s) {
  const int blocks = e.n_tiles * (kTile / 4 / kUpdThreads) + close_blocks(e);
  if (e.four) {
    if (ext_variant(e)) launch_after(k_update<true, true>, blocks, kUpdThreads, s, e, sr);
    else launch_after(k_update<false, true>, blocks, kUpdThreads, s, e, sr);
  } else {
    if (ext_variant(e)) launch_after(k_update<true, false>, blocks, kUpdThreads, s, e, sr);
    else launch_after(k_update<false, false>, blocks, kUpdThreads, s, e, sr);
  }
}

void launch_close(const EngineDev& e, unsigned long long g, cudaStream_t s) {
  const int blocks = (e.total_R + 63) / 64;  // a warp for 16 regions
  k_close<<<blocks > 0 ? blocks : 1, 128, 0, s>>>(e, g);
}

void launch_set_base(unsigned long long* base, unsigned long long g, cudaStream_t s) {
  k_set_base<<<1, 1, 0, s>>>(base, g);
}

int deliver_grid() {
  if (g_deliver_grid == 0) {
    int dev = 0, sms = 0, occ = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, k_deliver<false, true>, kDelThreads, 0);
    if (occ < 1) occ = 1;
    g_deliver_grid = sms * occ;
  }
  return g_deliver_grid;
}

void launch_deliver(const EngineDev& e, int grid, StepRef sr, cudaStream_t s, int part) {
  if (grid < 2) grid = 2;  // with a segment ring, block 0 may take no items
  if (e.n_inst == 1) {
    if (e.four) k_deliver<true, true><<<grid, kDelThreads, 0, s>>>(e, sr, part);
    else k_deliver<false, true><<<grid, kDelThreads, 0, s>>>(e, sr, part);
  } else {
    if (e.four) k_deliver<true, false><<<grid, kDelThreads, 0, s>>>(e, sr, part);
    else k_deliver<false, false><<<grid, kDelThreads, 0, s>>>(e, sr, part);
  }
}

void launch_windows(const EngineDev& e, int grid, StepRef sr, bool first, cudaStream_t s) {
  auto go = [&](auto kw, auto kr) {
    launch_after(first ? kw : kr, grid, kDelThreads, s, e, sr);
  };
  if (e.n_inst == 1) {
    if (e.four) go(k_windows<true, true>, k_rest<true, true>);
    else go(k_windows<false, true>, k_rest<false, true>);
  } else {
    if (e.four) go(k_windows<true, false>, k_rest<true, false>);
    else go(k_windows<false, false>, k_rest<false, false>);
  }
}

namespace {

// f(kernel) for the engine's variant of the stepper; held: a block for every
// tile keeps its state (not per step)
template <bool EXT, bool FOUR, class F>
auto with_persist(const EngineDev& e, bool held, F&& f) {
  const bool one = e.n_inst == 1;
  if (e.mode == kPerStep)
    return one ? f(k_persist<EXT, FOUR, true, true, false>) : f(k_persist<EXT, FOUR, false, true, false>);
  if (held)
    return one ? f(k_persist<EXT, FOUR, true, false, true>) : f(k_persist<EXT, FOUR, false, false, true>);
  return one ? f(k_persist<EXT, FOUR, true, false, false>) : f(k_persist<EXT, FOUR, false, false, false>);
}
template <class F>
auto with_persist(const EngineDev& e, bool held, F&& f) {
  const bool ext = ext_variant(e);
  if (e.four) return ext ? with_persist<true, true>(e, held, f) : with_persist<false, true>(e, held, f);
  return ext ? with_persist<true, false>(e, held, f) : with_persist<false, false>(e, held, f);
}

}  // namespace

int persist_max_grid(const EngineDev& e) {
  int dev = 0, sms = 0, occ = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  int least = 1 << 20;  // of both variants: which one runs depends on the tiles in use
  for (bool held : {false, true}) {
    const cudaError_t r = with_persist(e, held, [&](auto k) {
      return cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, k, kDelThreads, 0);
    });
    if (r != cudaSuccess) return 0;
    least = occ < least ? occ : least;
  }
  return sms * least;
}

cudaError_t launch_persist(const EngineDev& e, int grid, unsigned long long g0, int nsteps,
                           unsigned* count, unsigned long long limit_ns, cudaStream_t s) {
  if (e.mode == kAtEmission) grid = grid < e.n_tiles ? grid : e.n_tiles;  // no work for more
  else if (grid < 2) grid = 2;  // with a segment ring, block 0 may take no items
  const cudaError_t r = cudaMemsetAsync(count, 0, sizeof(unsigned), s);
  if (r != cudaSuccess) return r;
  EngineDev ea = e;
  void* args[] = {&ea, &g0, &nsteps, &count, &limit_ns};
  return with_persist(e, grid >= e.n_tiles, [&](auto k) {
    return cudaLaunchCooperativeKernel(k, dim3(grid), dim3(kDelThreads), args, 0, s);
  });
}

namespace {

// The resident stepper's variant for the engine's tiles: threads per block
// (256, 512 or 1,024) and blocks (a power of two, the cluster).
template <bool EXT, bool FOUR, class F>
cudaError_t with_resident(const EngineDev& e, F&& f) {
  int blocks = 1;
  const int per = e.n_tiles <= kClusterBlocks ? 1 : e.n_tiles <= 2 * kClusterBlocks ? 2 : 4;
  while (blocks * per < e.n_tiles) blocks *= 2;
  if (per == 1) return f(k_resident<EXT, FOUR, 256>, blocks, 256);
  if (per == 2) return f(k_resident<EXT, FOUR, 512>, blocks, 512);
  return f(k_resident<EXT, FOUR, 1024>, blocks, 1024);
}
template <class F>
cudaError_t with_resident(const EngineDev& e, F&& f) {
  if (e.four) return e.any_ext ? with_resident<true, true>(e, f) : with_resident<false, true>(e, f);
  return e.any_ext ? with_resident<true, false>(e, f) : with_resident<false, false>(e, f);
}

}  // namespace

bool resident_fits(const EngineDev& e) {
  if (e.mode != kAtEmission || e.n_tiles < 1 || e.n_tiles > kResidentTiles) return false;
  int clusters = 0;
  const cudaError_t r = with_resident(e, [&](auto k, int blocks, int threads) {
    cudaError_t a = cudaFuncSetAttribute(k, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
    if (a != cudaSuccess) return a;
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3(blocks);
    cfg.blockDim = dim3(threads);
    cudaLaunchAttribute at{};
    at.id = cudaLaunchAttributeClusterDimension;
    at.val.clusterDim.x = blocks;
    at.val.clusterDim.y = at.val.clusterDim.z = 1;
    cfg.attrs = &at;
    cfg.numAttrs = 1;
    return cudaOccupancyMaxActiveClusters(&clusters, k, &cfg);
  });
  if (r != cudaSuccess) cudaGetLastError();  // not a failure of the engine
  return r == cudaSuccess && clusters > 0;
}

cudaError_t launch_resident(const EngineDev& e, unsigned long long g0, int nsteps, cudaStream_t s) {
  return with_resident(e, [&](auto k, int blocks, int threads) {
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3(blocks);
    cfg.blockDim = dim3(threads);
    cfg.stream = s;
    cudaLaunchAttribute at{};
    at.id = cudaLaunchAttributeClusterDimension;
    at.val.clusterDim.x = blocks;
    at.val.clusterDim.y = at.val.clusterDim.z = 1;
    cfg.attrs = &at;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, k, e, g0, nsteps);
  });
}

cudaError_t launch_barrier_probe(int grid, unsigned extra, int rounds, unsigned long long limit_ns,
                                 unsigned* count, unsigned* flags, cudaStream_t s) {
  cudaError_t r = cudaMemsetAsync(count, 0, sizeof(unsigned), s);
  if (r != cudaSuccess) return r;
  void* args[] = {&count, &extra, &rounds, &limit_ns, &flags};
  return cudaLaunchCooperativeKernel(k_barrier_probe, dim3(grid), dim3(32), args, 0, s);
}

void launch_ingest(int32_t N, int32_t j0, int32_t j1, int64_t e_base, const int64_t* row_ptr,
                   const int32_t* col_in, const void* w_in, const void* w2_in, int32_t w_dtype,
                   const uint8_t* delay_in, uint16_t* rec, int32_t shift, int32_t dmax,
                   int32_t seg_bytes, void* seg, int32_t seg_kind, int32_t* indeg, unsigned* wmax_bits, unsigned* err,
                   cudaStream_t s) {
  int64_t blocks = ((int64_t)(j1 - j0) * 32 + 255) / 256;
  if (blocks > 152 * 64) blocks = 152 * 64;
  if (blocks < 1) blocks = 1;
  k_ingest<<<(int)blocks, 256, 0, s>>>(N, j0, j1, e_base, row_ptr, col_in, w_in, w2_in, w_dtype,
                                       delay_in, rec, shift, dmax, seg_bytes, seg, seg_kind, indeg,
                                       wmax_bits, err);
}

void launch_pending_events(const EngineDev& e, unsigned long long g, unsigned long long* out,
                           cudaStream_t s) {
  if (g == 0 || e.mode == kAtEmission) return;
  const long long window = ((long long)g - 1) & ~(long long)(e.mode == kWindows && !e.seg_cap ? e.wmask : 0);
  launch_count_events(e, window > (long long)e.since ? window : (long long)e.since, (long long)g - 1 + e.bin_lead,
                      out, s);
}

void launch_count_events(const EngineDev& e, long long r0, long long r1, unsigned long long* out, cudaStream_t s) {
  if (r1 >= r0) k_pending_events<<<152, 256, 0, s>>>(e, r0, r1, out);
}

void launch_hand_over(const EngineDev& e, int grid, unsigned long long g, cudaStream_t s) {
  EngineDev f = e;  // one window as long as the accumulator ring
  f.mode = kWindows;
  f.wmask = e.acc_slots - 1;
  f.seg_cap = 0;
  f.phases = 1;
  f.keep_counts = 1;
  f.since = g - 1ull;  // the spikes of step g - 1 are not counted yet
  launch_windows(f, grid, StepRef{nullptr, g, nullptr}, true, s);
}

void launch_max_reduce(const int32_t* a, int64_t n, unsigned* out, cudaStream_t s) {
  int64_t blocks = (n + 255) / 256;
  if (blocks > 152 * 8) blocks = 152 * 8;
  if (blocks < 1) blocks = 1;
  k_max_reduce<<<(int)blocks, 256, 0, s>>>(a, n, out);
}


}  // namespace dbn

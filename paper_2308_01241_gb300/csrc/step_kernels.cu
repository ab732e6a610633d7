// step_kernels.cu -- the kernels of one simulation step and their launchers,
// but for the delivery (deliver.cu).
//
//   neuron_update  Eq. 1 by explicit Euler (sections III.B, VI.A), Poisson drive,
//                  threshold / reset / refractory; spike bits by warp ballot
//   spike_compact  ascending spike ids from the bits: per-block counts,
//                  prefix sums, popc ranks ("collect spikes sequence", V.B)
//   bold_step      Balloon-Windkessel per voxel (section V.E, Friston 2000)
//
// Every floating-point operation of the neuron update is an explicit
// round-to-nearest intrinsic, in the order the header dtb.h states, so no
// multiply-add is ever fused and the result is bit-identical to the C oracle.
#include <cuda_runtime.h>
#include <stdint.h>

#include <mutex>

#include "device_launch.h"
#include "dtb_device.cuh"
#include "dtb_launch.h"

namespace dtb {
namespace {

__device__ __forceinline__ float fsub(float a, float b) { return __fsub_rn(a, b); }
__device__ __forceinline__ float fadd(float a, float b) { return __fadd_rn(a, b); }
__device__ __forceinline__ float fmul(float a, float b) { return __fmul_rn(a, b); }

// Two neurons' values in one 64-bit register pair: the packed FP32 operations
// round each half like the scalar ones and take one issue slot for both.
typedef unsigned long long f2;
__device__ __forceinline__ f2 pk(float a, float b) {
  f2 d;
  asm("mov.b64 %0, {%1, %2};" : "=l"(d) : "f"(a), "f"(b));
  return d;
}
__device__ __forceinline__ f2 dup(float a) { return pk(a, a); }
__device__ __forceinline__ void unpk(f2 v, float& a, float& b) { asm("mov.b64 {%0, %1}, %2;" : "=f"(a), "=f"(b) : "l"(v)); }
__device__ __forceinline__ f2 add2(f2 a, f2 b) {
  f2 d;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
  return d;
}
__device__ __forceinline__ f2 sub2(f2 a, f2 b) {
  f2 d;
  asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
  return d;
}
__device__ __forceinline__ f2 mul2(f2 a, f2 b) {
  f2 d;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
  return d;
}
__device__ __forceinline__ f2 fma2(f2 a, f2 b, f2 c) {
  f2 d;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
  return d;
}

// A product that a later sum must not absorb: packed mul and add are fused
// into one multiply-add even with contraction off, so the product is itself a
// multiply-add of -0, which changes no bit of it.  The -0 comes from a
// register whose value the compiler does not know.
__device__ __forceinline__ f2 neg_zero(const DevNet& g) {
  return dup(__uint_as_float(0x80000000u | (uint32_t)((uint64_t)g.npad >> 63)));
}
__device__ __forceinline__ f2 prod2(f2 a, f2 b, f2 nz) { return fma2(a, b, nz); }

constexpr float kAccScale = 1.52587890625e-05f;  // 2^-16

// k = #{m < M : u >= T_m}.  T is ascending, so past the first threshold u is
// below, none of the later ones counts: three compares cover all but a
// fraction P(K >= 3) (1e-3 at 2 kHz x 0.1 ms) of the draws.
__device__ __forceinline__ int32_t poisson_low(const DevNet& g, uint32_t u) {
  int32_t k = (g.M > 0 && u >= g.T[0]) ? 1 : 0;
  if (g.M > 1 && u >= g.T[1]) k = 2;
  if (g.M > 2 && u >= g.T[2]) k = 3;
  return k;
}
__device__ __forceinline__ int32_t poisson_high(const DevNet& g, uint32_t u) {
  int32_t k = 0;
#pragma unroll 1
  for (int m = 3; m < g.M; m++) k += (u >= g.T[m]) ? 1 : 0;
  return k;
}

// One neuron, one step, in two parts that touch disjoint state:
//   j part: consume the arrivals A[] of a step and its Poisson count k,
//           j_u <- dJ_u j_u + a_u;
//   V part: V from V and j (the j of the start of the step), OU current,
//           refractory period and threshold; returns the spike.
// The plain step of the paper's order is V part then j part at the same t.
// Applying the j part of step t-1 right before the V part of step t gives
// the same numbers (each operation sees the same operands).
template <int NCH>
__device__ __forceinline__ void update_j(const DevNet& g, const VoxConst& c, float (&jj)[4], const int32_t (&A)[NCH],
                                         int32_t k) {
#pragma unroll
  for (int q = 0; q < 4; q++) {
    int32_t in = A[NCH == 2 ? q / 2 : q % NCH];
    if (q == 0) in += k * g.w_ext;
    jj[q] = fadd(fmul(c.dJ[q], jj[q]), fmul(__int2float_rn(in), kAccScale));
  }
}

// The OU current's Euler-Maruyama step; the normal is the centred sum of the
// four words of one Philox call.
__device__ __forceinline__ float ou_step(const DevNet& g, float I, int64_t i, int64_t t) {
  const uint4 r = philox4x32_10(make_uint4((uint32_t)i, (uint32_t)t, (uint32_t)((uint64_t)t >> 32), kTagOU), g.key0,
                                g.key1);
  const long long S = (long long)((unsigned long long)r.x + r.y + r.z + r.w) - (1LL << 33);
  const float xi = fmul(__ll2float_rn(S), g.ou_xi);
  return fadd(fadd(fmul(g.ou_d, I), g.ou_c), fmul(g.ou_s, xi));
}

// Membrane potential after one step, before the threshold (OU: I is the
// current of the start of the step).
template <bool OU>
__device__ __forceinline__ float membrane(const VoxConst& c, float V, const float (&jj)[4], float I) {
  float s = 0.0f;
#pragma unroll
  for (int q = 0; q < 4; q++) s = fadd(s, fmul(fmul(c.kU[q], jj[q]), fsub(V, c.E[q])));
  float Vn = fsub(V, fmul(c.kL, fsub(V, c.EL)));
  Vn = fsub(Vn, s);
  Vn = fadd(Vn, c.kI);
  if (OU) Vn = fadd(Vn, fmul(c.kO, I));
  return Vn;
}

// Refractory period, threshold and reset of neuron q of a quad: its byte of
// ref4, its potential; true when it fires.
__device__ __forceinline__ bool threshold(float Vth, float Vreset, uint32_t ref_steps, float& V, uint32_t& ref4, int q) {
  const bool refr = (ref4 & (0xFFu << (8 * q))) != 0;
  const bool over = V >= Vth;
  if (refr || over) V = Vreset;
  const bool spike = over && !refr;
  if (refr) ref4 -= 1u << (8 * q);
  if (spike) ref4 += ref_steps << (8 * q);  // the byte is 0 here
  return spike;
}

// Four neighbouring neurons of one voxel: receptor-major gating variables.
struct Quad {
  float V[4], J[4][4], I[4];
  uint32_t ref4;
};

// The j part of four neurons, two per packed operation.  The scaled input
// 2^-16 * in is exact, so one fused multiply-add rounds like the separate
// product and sum.
template <int NCH>
__device__ __forceinline__ void quad_j(const DevNet& g, const VoxConst& c, Quad& s, const int4 (&A4)[NCH],
                                       const int32_t (&k)[4]) {
  const f2 sc = dup(kAccScale);
  const float4 dJ = *reinterpret_cast<const float4*>(c.dJ);
  const f2 d[4] = {dup(dJ.x), dup(dJ.y), dup(dJ.z), dup(dJ.w)};
#pragma unroll
  for (int p = 0; p < 2; p++) {
    f2 a[4];
#pragma unroll
    for (int q = 0; q < 4; q++) {
      if (NCH == 2 && q == 3) {
        a[3] = a[2];
        continue;
      }
      const int4 A = A4[NCH == 2 ? q / 2 : q % NCH];
      int32_t x = p ? A.z : A.x, y = p ? A.w : A.y;
      if (q == 0) {
        x += k[2 * p] * g.w_ext;
        y += k[2 * p + 1] * g.w_ext;
      }
      a[q] = pk(__int2float_rn(x), __int2float_rn(y));
    }
#pragma unroll
    for (int q = 0; q < 4; q++) {
      const f2 j = fma2(a[q], sc, mul2(d[q], pk(s.J[q][2 * p], s.J[q][2 * p + 1])));
      unpk(j, s.J[q][2 * p], s.J[q][2 * p + 1]);
    }
  }
}

// The V part of four neurons; returns their spike bits.
template <bool OU>
__device__ __forceinline__ uint32_t quad_v(const DevNet& g, const VoxConst& c, Quad& s, int64_t i0, int64_t t) {
  const float4 kU4 = *reinterpret_cast<const float4*>(c.kU), E4 = *reinterpret_cast<const float4*>(c.E);
  const float4 b = *reinterpret_cast<const float4*>(&c.kL);      // kL, EL, kI, Vth
  const float4 r = *reinterpret_cast<const float4*>(&c.Vreset);  // Vreset, ref_steps, kO
  const float kU[4] = {kU4.x, kU4.y, kU4.z, kU4.w}, E[4] = {E4.x, E4.y, E4.z, E4.w};
  const f2 nz = neg_zero(g);
  const f2 V[2] = {pk(s.V[0], s.V[1]), pk(s.V[2], s.V[3])};
  f2 sum[2] = {0ull, 0ull};  // {0.0f, 0.0f}
#pragma unroll
  for (int q = 0; q < 4; q++) {
    const f2 k = dup(kU[q]), e = dup(E[q]);
#pragma unroll
    for (int p = 0; p < 2; p++)
      sum[p] = add2(sum[p], prod2(mul2(k, pk(s.J[q][2 * p], s.J[q][2 * p + 1])), sub2(V[p], e), nz));
  }
  const f2 kL = dup(b.x), EL = dup(b.y), kI = dup(b.z), kO = dup(r.z);
#pragma unroll
  for (int p = 0; p < 2; p++) {
    f2 Vn = sub2(V[p], prod2(kL, sub2(V[p], EL), nz));
    Vn = sub2(Vn, sum[p]);
    Vn = add2(Vn, kI);
    if (OU) Vn = add2(Vn, prod2(kO, pk(s.I[2 * p], s.I[2 * p + 1]), nz));
    unpk(Vn, s.V[2 * p], s.V[2 * p + 1]);
  }
  uint32_t nib = 0;
#pragma unroll
  for (int q = 0; q < 4; q++) {
    if (OU) s.I[q] = ou_step(g, s.I[q], i0 + q, t);
    if (threshold(b.w, r.x, (uint32_t)__float_as_int(r.y), s.V[q], s.ref4, q)) nib |= 1u << q;
  }
  return nib;
}

__device__ __forceinline__ VoxConst load_vc(const VoxConst* p) {
  VoxConst c;
  const float4* s = reinterpret_cast<const float4*>(p);
  float4* d = reinterpret_cast<float4*>(&c);
#pragma unroll
  for (int q = 0; q < 5; q++) d[q] = __ldg(s + q);
  return c;
}

template <typename T>
__device__ __forceinline__ T pick(const T (&a)[4], int q) {
  const T lo = q & 1 ? a[1] : a[0], hi = q & 1 ? a[3] : a[2];
  return q & 2 ? hi : lo;
}
template <typename T>
__device__ __forceinline__ void put(T (&a)[4], int q, T x) {
#pragma unroll
  for (int k = 0; k < 4; k++)
    if (k == q) a[k] = x;
}

// Four neurons of different voxels (v: the first one's): one after the other,
// each with its own voxel's constants.
template <int NCH, bool OU>
__device__ __forceinline__ uint32_t quad_mixed(const DevNet& g, Quad& s, const int4 (&A4)[NCH], const int32_t (&k)[4],
                                               int64_t i0, int64_t t, int32_t v, bool do_v, bool do_j, bool j_first) {
  uint32_t nib = 0;
#pragma unroll 1
  for (int q = 0; q < 4; q++) {
    while (v + 1 < g.nv && g.vstart[v + 1] <= i0 + q) v++;
    const VoxConst c = load_vc(g.vc + v);
    float V = pick(s.V, q), I = OU ? pick(s.I, q) : 0.0f;
    float J[4] = {pick(s.J[0], q), pick(s.J[1], q), pick(s.J[2], q), pick(s.J[3], q)};
    int32_t A[NCH];
#pragma unroll
    for (int cc = 0; cc < NCH; cc++) {
      const int32_t a[4] = {A4[cc].x, A4[cc].y, A4[cc].z, A4[cc].w};
      A[cc] = pick(a, q);
    }
    if (j_first) update_j<NCH>(g, c, J, A, pick(k, q));
    if (do_v) {
      V = membrane<OU>(c, V, J, I);
      if (OU) I = ou_step(g, I, i0 + q, t);
      if (threshold(c.Vth, c.Vreset, (uint32_t)c.ref_steps, V, s.ref4, q)) nib |= 1u << q;
    }
    if (do_j && !j_first) update_j<NCH>(g, c, J, A, pick(k, q));
    put(s.V, q, V);
    if (OU) put(s.I, q, I);
#pragma unroll
    for (int u = 0; u < 4; u++) put(s.J[u], q, J[u]);
  }
  return nib;
}

// Persistent, TMA-fed neuron update.  A CTA of 256 threads owns the tiles
// blockIdx.x, blockIdx.x + gridDim.x, ... of 1024 neurons each.  One thread
// streams each tile's state rows (V, j[4], ref, the ring slot's NCH rows:
// 29 KB for two channels) into a ring of S shared-memory stages with 1D bulk
// copies, S tiles ahead of the compute; every thread then updates its four
// consecutive neurons from shared memory and writes V, j, ref, zeroed
// accumulators and spike bits straight to HBM with 128-bit stores.  One
// Philox call per thread gives the four neurons' drive words.  Spike bits:
// 4-bit nibbles OR-ed across groups of 8 lanes into 32-bit words (word w
// holds neurons 32w .. 32w+31); one spike count per tile.  With the OU drive
// the stage also carries the tile's OU currents (4 KB more).
//
// Bins mode (BINS): there is no dense accumulator.  A CTA owns the regions
// blockIdx.x, blockIdx.x + gridDim.x, ... of kRegionTiles consecutive tiles.
// At the start of a region its threads add the region's bin of arrival events
// into an int32 [NCH][kRegionNeurons] array in shared memory (exact integer
// sums, any order); each neuron then takes its arrivals from that array and
// clears them.  The bin (up to kEvBufWords words) is staged in shared memory
// by one bulk copy issued a region ahead, so adding it waits on no global
// load.  Three resident CTAs per SM (two stages each) let one CTA add its
// region's events while the others stream tiles.
//
// What bounds it: not bytes (at 5M neurons 0.21 GB take 31 us at the copy
// rate; the kernel takes 46) but issue slots and the latency of 24 warps per SM.
// So the four neurons of a thread go through packed FP32 operations two by
// two, the body of a call is an instance of its own without mode tests, and
// no barrier holds a tile's warps together (only a region's two, in bins mode):
// step 73.6 -> 70.0 us at 5M neurons, 7 Hz; 39.4 -> 36.1 us at 1M, 15 Hz.
template <int NCH, bool OU, bool BINS>
struct Stage {
  // bins mode stages V, ref (and I) and loads each thread's j straight into
  // registers, so that three CTAs fit on an SM
  static constexpr uint32_t kV = 0, kJ = 4096, kRef = BINS ? 4096 : kJ + 4 * 4096, kAcc = kRef + 1024;
  static constexpr uint32_t kI = kAcc + (BINS ? 0 : NCH * 4096);
  static constexpr uint32_t kNit = kI + (OU ? 4096 : 0);  // bins mode: work items per neuron (1 B each)
  static constexpr uint32_t kBytes = kNit + (BINS ? kNeuronsPerBlock : 0);  // one tile
  // bins mode: the region's arrival sums and its staged bin sit in front of the stages
  static constexpr uint32_t kRegionAcc = BINS ? NCH * kRegionNeurons * 4 : 0;
  static constexpr uint32_t kFront = BINS ? kRegionAcc + kEvBufWords * 4 : 0;
  static constexpr uint32_t bytes(int S) { return kFront + S * kBytes; }
};
// Counts a warp's arrival at a stage (its reads of the stage come before).
__device__ __forceinline__ uint32_t taken_add(uint32_t* p) {
  uint32_t old;
  asm volatile("atom.acq_rel.cta.shared::cta.add.u32 %0, [%1], 1;" : "=r"(old) : "r"(smem_u32(p)) : "memory");
  return old;
}

// A warp's spiking neurons (id, or -1 for a lane without one) on the delivery's
// list of step t: queue mode, the chunks of their rows; ring mode, their rows in
// pieces of kItemEvents synapses.
__device__ __forceinline__ void list_work(const DevNet& g, int32_t id, int64_t t, int lane) {
  const bool rows = g.row_list != nullptr;
  int64_t cb = 0, len = 0;
  if (id >= 0) {
    const int64_t* p = (rows ? g.row_ptr : g.chunk_base) + id;
    cb = __ldg(p);
    len = __ldg(p + 1) - cb;
  }
  const int nc = (int)(rows ? (len + kItemEvents - 1) / kItemEvents : len);
  int end = nc;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int y = __shfl_up_sync(0xFFFFFFFFu, end, o);
    if (lane >= o) end += y;
  }
  uint32_t base = 0;
  if (lane == 31 && end > 0) base = atomicAdd(g.chunk_cnt + t % 3, (uint32_t)end);
  base = __shfl_sync(0xFFFFFFFFu, base, 31) + (uint32_t)(end - nc);
  const int64_t at = (t & 1) * g.list_cap + base;
  if (rows) {
    for (int k = 0; k < nc; k++)
      g.row_list[at + k] = make_ulonglong2((unsigned long long)(cb + (int64_t)k * kItemEvents),
                                           row_piece(id, (int)min(len - (int64_t)k * kItemEvents, (int64_t)kItemEvents)));
  } else {
    for (int k = 0; k < nc; k++) g.chunk_list[at + k] = (uint32_t)(cb + k);
  }
}
constexpr int kSpikeList = 1024;  // spikes of a CTA held in shared memory until its end

constexpr int kMaxRegionsPerCta = 128;  // bins mode: the launcher keeps grid * 128 >= regions

// upd: kUpdFull (V part then j part of step t), kUpdJV (j part of step t-1,
// then V part of step t), kUpdV (V part of step t only), kUpdJ (j part of
// step t only).  The j part consumes the arrivals of its step x: slot x mod D
// of the ring, slot x mod 2 of the event-queue mode's accumulator, or the
// bins of parity x mod 2 in bins mode.  BODY: kUpdJV at compile time (every
// step of a call but its first); the other modes share one instance.
template <int NCH, int S, bool OU, bool BINS, bool BODY>
__global__ void __launch_bounds__(kUpdateThreads, BINS || (NCH == 2 && !OU) ? 3 : 2)
    neuron_update_kernel(DevNet g, int32_t t_rel, int32_t upd) {
  using St = Stage<NCH, OU, BINS>;
  constexpr int kThr = kUpdateThreads, kWarps = kThr / 32;
  constexpr int kSlots = 8;  // tiles whose counts can be under way: warps are at most S <= 4 tiles apart
  extern __shared__ __align__(128) unsigned char smem[];
  unsigned char* stages = smem + St::kFront;
  int32_t* racc = reinterpret_cast<int32_t*>(smem);  // bins mode: [NCH][kRegionNeurons]
  uint32_t* ebuf = reinterpret_cast<uint32_t*>(smem + St::kRegionAcc);  // bins mode: staged bin
  __shared__ uint64_t bar[S];    // stage k % S holds my k-th tile
  __shared__ uint32_t s_taken[S];  // warps that have taken what they need from the stage, over all its tiles
  __shared__ uint64_t ebar;                          // bins mode: the staged bin landed
  __shared__ uint32_t s_rcnt[BINS ? kMaxRegionsPerCta : 1];  // bins mode: events in my regions' bins
  // the tiles' constants, in a ring of their own: it is deep enough that a
  // refill never meets a warp still reading, so no thread holds them in registers
  __shared__ __align__(16) VoxConst s_vc[kSlots];
  __shared__ int32_t s_spk[BINS ? 1 : kSpikeList];  // ring and queue modes: the CTA's spikes
  __shared__ int s_nspk;
  __shared__ uint32_t s_done[kSlots];   // warps done with the tile << 28 | its spikes
  __shared__ uint32_t s_items[kSlots];  // its delivery work items
  const int64_t t = *g.t_base + t_rel;
  const bool do_v = BODY || upd != kUpdJ, do_j = BODY || upd != kUpdV, j_first = BODY || upd == kUpdJV;
  const int64_t x = j_first ? t - 1 : t;  // the step whose arrivals the j part consumes
  const int64_t np = g.npad;
  int32_t* acc_slot = BINS ? nullptr : g.ring + (g.mode ? (x & 1) : x % g.D) * NCH * np;
  const int ntile = g.nblk;
  // n_mine: my tiles
  int n_mine, r_mine = 0;
  if (BINS) {  // whole regions; only the network's last one may be short
    const int nreg = g.n_reg;
    r_mine = (int)blockIdx.x < nreg ? (nreg - 1 - (int)blockIdx.x) / (int)gridDim.x + 1 : 0;
    const int r_last = (int)blockIdx.x + (r_mine - 1) * (int)gridDim.x;
    n_mine = r_mine ? (r_mine - 1) * kRegionTiles + min(kRegionTiles, ntile - r_last * kRegionTiles) : 0;
  } else {
    n_mine = (int)blockIdx.x < ntile ? (ntile - 1 - (int)blockIdx.x) / (int)gridDim.x + 1 : 0;
  }
  // my k-th tile
  auto tile_of = [&](int k) {
    return BINS ? ((int)blockIdx.x + (k / kRegionTiles) * (int)gridDim.x) * kRegionTiles + k % kRegionTiles
                : (int)blockIdx.x + k * (int)gridDim.x;
  };
  const int tid = threadIdx.x, lane = tid & 31;
  const bool spilled = do_j && g.mode && g.spill_dirty[x % g.D] == spill_mark(x);
  // the queue of step x is in the accumulator or the bins by now; it is empty
  // again for the deliveries of step x + 1 on, which come after this kernel
  if (do_j && g.mode && blockIdx.x == 0 && tid < g.n_sub) g.qcnt[((x % g.D) * g.n_sub + tid) * kQcntStride] = 0;

  // state is read and written once per step: it makes room for the accumulators
  // and queues, unless all of it fits (then it is the synapses that pass through)
  const uint64_t once = !BINS && g.keep_state ? l2_evict_normal() : l2_evict_first();
  auto issue = [&](int k) {  // one thread: bulk loads of my k-th tile into stage k % S
    uint64_t* b = &bar[k % S];
    const int tl = tile_of(k);
    const int64_t base = (int64_t)tl * kNeuronsPerBlock;
    unsigned char* st = stages + (size_t)(k % S) * St::kBytes;
    mbar_expect_tx(b, St::kBytes + (uint32_t)sizeof(VoxConst));
    bulk_g2s_hint(st + St::kV, g.V + base, 4096, b, once);
    if (!BINS) {
#pragma unroll
      for (int q = 0; q < 4; q++) bulk_g2s_hint(st + St::kJ + q * 4096, g.j + q * np + base, 4096, b, once);
    }
    bulk_g2s_hint(st + St::kRef, g.ref + base, 1024, b, once);
    if (!BINS) {
#pragma unroll
      for (int c = 0; c < NCH; c++) bulk_g2s_hint(st + St::kAcc + c * 4096, acc_slot + c * np + base, 4096, b, once);
    }
    if (OU) bulk_g2s_hint(st + St::kI, g.Iou + base, 4096, b, once);
    bulk_g2s(&s_vc[k % kSlots], g.tile_vc + tl, sizeof(VoxConst), b);
    if (BINS) bulk_g2s_hint(st + St::kNit, g.nitem + base, kNeuronsPerBlock, b, once);
  };
  // bins mode: the bin of my m-th region, parity of step x
  const int par = (int)(x & 1);
  const int ew = g.ev8 ? 2 : 1;
  auto bin_of = [&](int m) {
    return g.bins + ((int64_t)par * g.n_reg + (int)blockIdx.x + m * (int)gridDim.x) * g.bcap * ew;
  };
  auto issue_ev = [&](int m) {  // one thread: bulk copy of my m-th region's bin (up to kEvBufWords words)
    const uint32_t words = min(s_rcnt[m] * (uint32_t)ew, (uint32_t)kEvBufWords);
    const uint32_t bytes = (words * 4u + 15u) & ~15u;  // within the bin: its size is a multiple of 16 bytes
    mbar_expect_tx(&ebar, bytes);
    if (bytes) bulk_g2s_hint(ebuf, bin_of(m), bytes, &ebar, once);
  };

  if (tid == 0) {
#pragma unroll
    for (int q = 0; q < S; q++) {
      mbar_init(&bar[q], 1);
      s_taken[q] = 0;
    }
    if (BINS) mbar_init(&ebar, 1);
    fence_mbar_init();
  }
  if (tid < kSlots) {
    s_done[tid] = 0;
    s_items[tid] = 0;
  }
  const bool listing = !BINS && do_v;
  if (tid == 0) {
    s_nspk = 0;
    if (listing && blockIdx.x == 0) g.chunk_cnt[(t + 1) % 3] = 0;
  }
  if (BINS) {
    int4* z = reinterpret_cast<int4*>(racc);
    for (int q = tid; q < NCH * kRegionNeurons / 4; q += kThr) z[q] = make_int4(0, 0, 0, 0);
    if (do_j)
      for (int m = tid; m < r_mine; m += kThr)
        s_rcnt[m] = (uint32_t)min(g.bcnt[((int64_t)par * g.n_reg + (int)blockIdx.x + m * (int)gridDim.x) * kBcntStride],
                                  (unsigned long long)g.bcap);
  }
  __syncthreads();
  if (tid == 0) {
    if (BINS && do_j && r_mine > 0) issue_ev(0);
    for (int k = 0; k < S && k < n_mine; k++) issue(k);
  }

  bool bad = false;            // this warp gave up waiting
  int ev_pending = BINS && do_j && r_mine > 0 ? 0 : -1;  // tid 0: the region whose staged bin is in flight
  uint32_t ph = 1u;
  for (int k = 0, sg = S - 1; k < n_mine; k++) {
    sg = sg == S - 1 ? 0 : sg + 1;  // tile k's stage and the phase of its barrier
    if (sg == 0) ph ^= 1u;
    const int tile = tile_of(k);
    const int64_t i0 = (int64_t)tile * kNeuronsPerBlock + tid * 4;
    if (BINS && do_j && k % kRegionTiles == 0) {
      // the region's arrivals of step x into shared memory; racc is all zero
      // here (cleared at the start and by every tile's consumers, which the
      // barrier waits for).  A warp that gave up still meets the others here.
      const int m = k / kRegionTiles;
      if (!__syncthreads_and(!bad && mbar_wait_bounded(&ebar, (uint32_t)m & 1u))) {
        if (tid == 0) atomicOr(g.err, 1);
        bad = true;
        break;
      }
      ev_pending = -1;
      const int cnt = (int)s_rcnt[m];
      const int nbuf = min(cnt, kEvBufWords / ew);
      const uint32_t* evg = bin_of(m);
      const int32_t wfmt = g.wfmt, wsh = g.wshift;
      for (int e = tid; e < cnt; e += kThr) {
        uint32_t a, c;
        if (ew == 1) {
          a = e < nbuf ? ebuf[e] : __ldcs(evg + e);
          c = a >> 16;
        } else {
          const uint2 v = e < nbuf ? reinterpret_cast<const uint2*>(ebuf)[e]
                                   : __ldcs(reinterpret_cast<const uint2*>(evg) + e);
          a = v.x;
          c = v.y;
        }
        atomicAdd(racc + ((a >> kRegionShift) & 3u) * kRegionNeurons + (a & (kRegionNeurons - 1)),
                  decode_weight(c, wfmt, wsh));
      }
      __syncthreads();
      if (tid == 0) {
        // the bin is free for the step two later; the staging buffer for the next region
        g.bcnt[((int64_t)par * g.n_reg + (int)blockIdx.x + m * (int)gridDim.x) * kBcntStride] = 0;
        if (m + 1 < r_mine) {
          fence_proxy_async_smem();
          issue_ev(m + 1);
          ev_pending = m + 1;
        }
      }
    }
    float4 J4[4];
    if (BINS) {  // bins mode: my four neurons' j rows, loaded while the stage is in flight
#pragma unroll
      for (int q = 0; q < 4; q++) J4[q] = ld_hint(reinterpret_cast<const float4*>(g.j + q * np + i0), once);
    }
    // the drive words depend only on (i, x): drawn while the loads are in flight
    int32_t kp[4] = {0, 0, 0, 0};
    if (do_j) {
      const uint4 r = philox4x32_10(
          make_uint4((uint32_t)(i0 >> 2), (uint32_t)x, (uint32_t)((uint64_t)x >> 32), kTagDrive), g.key0, g.key1);
      const uint32_t u[4] = {r.x, r.y, r.z, r.w};
#pragma unroll
      for (int q = 0; q < 4; q++) kp[q] = poisson_low(g, u[q]);
      if (g.M > 3 && max(max(u[0], u[1]), max(u[2], u[3])) >= g.T[2]) {
#pragma unroll
        for (int q = 0; q < 4; q++) kp[q] += poisson_high(g, u[q]);
      }
    }
    // every warp waits for the stage by itself: no barrier per tile, so a warp
    // held up by a spike or a voxel boundary does not hold the others
    if (!bad) {
      bad = !__all_sync(0xFFFFFFFFu, mbar_wait_bounded(&bar[sg], ph));
      if (bad && lane == 0) atomicOr(g.err, 1);
    }
    if (bad) continue;  // gave up: only the barriers of the regions to come
    const unsigned char* st = stages + (size_t)sg * St::kBytes;
    // everything this tile takes from the stage, into registers; then the
    // stage is handed back and refilled while the neurons are updated
    const float4 V4 = reinterpret_cast<const float4*>(st + St::kV)[tid];
    if (!BINS) {
#pragma unroll
      for (int q = 0; q < 4; q++) J4[q] = reinterpret_cast<const float4*>(st + St::kJ + q * 4096)[tid];
    }
    Quad s;
    s.ref4 = reinterpret_cast<const uint32_t*>(st + St::kRef)[tid];
    int4 A4[NCH];
    if (!BINS) {
#pragma unroll
      for (int cc = 0; cc < NCH; cc++) A4[cc] = reinterpret_cast<const int4*>(st + St::kAcc + cc * 4096)[tid];
    }
    const float4 I4 = OU ? reinterpret_cast<const float4*>(st + St::kI)[tid] : make_float4(0.f, 0.f, 0.f, 0.f);
    const uint32_t ni4 = BINS ? reinterpret_cast<const uint32_t*>(st + St::kNit)[tid] : 0u;
    const VoxConst* vc = &s_vc[k % kSlots];
    const bool first_vox = tid * 4 + 3 < vc->n_first;
    __syncwarp();
    // the warp that is the last one to take its part refills the stage
    if (lane == 0 && taken_add(&s_taken[sg]) % kWarps == kWarps - 1 && k + S < n_mine) {
      fence_proxy_async_smem();  // the stage's generic reads before the async refill
      issue(k + S);
    }
    if (BINS) {
      const int off = (k % kRegionTiles) * kNeuronsPerBlock + tid * 4;
#pragma unroll
      for (int cc = 0; cc < NCH; cc++) {
        int4* p = reinterpret_cast<int4*>(racc + cc * kRegionNeurons + off);
        A4[cc] = *p;
        if (do_j) *p = make_int4(0, 0, 0, 0);
      }
    }
    if (spilled) {  // event-queue and bins modes after a queue or bin overflowed: the spill slot adds in (rare)
      int32_t* sp = g.spill + (x % g.D) * NCH * np + i0;
#pragma unroll
      for (int cc = 0; cc < NCH; cc++) {
        const int4 y = *reinterpret_cast<const int4*>(sp + cc * np);
        *reinterpret_cast<int4*>(sp + cc * np) = make_int4(0, 0, 0, 0);
        A4[cc] = make_int4(A4[cc].x + y.x, A4[cc].y + y.y, A4[cc].z + y.z, A4[cc].w + y.w);
      }
    }
    s.V[0] = V4.x; s.V[1] = V4.y; s.V[2] = V4.z; s.V[3] = V4.w;
    s.I[0] = I4.x; s.I[1] = I4.y; s.I[2] = I4.z; s.I[3] = I4.w;
#pragma unroll
    for (int q = 0; q < 4; q++) {
      s.J[q][0] = J4[q].x; s.J[q][1] = J4[q].y; s.J[q][2] = J4[q].z; s.J[q][3] = J4[q].w;
    }
    // constants: the tile's copy when my four neurons lie in its first voxel
    // (no global load), else looked up
    int32_t v = 0;
    bool mixed = false;
    if (!first_vox) {
      v = g.blk_vox[tile];
      while (v + 1 < g.nv && g.vstart[v + 1] <= i0) v++;
      mixed = v + 1 < g.nv && g.vstart[v + 1] <= i0 + 3;
      vc = g.vc + v;
    }
    uint32_t nib = 0;
    if (!mixed) {
      if (j_first) quad_j<NCH>(g, *vc, s, A4, kp);
      if (do_v) nib = quad_v<OU>(g, *vc, s, i0, t);
      if (do_j && !j_first) quad_j<NCH>(g, *vc, s, A4, kp);
    } else {
      nib = quad_mixed<NCH, OU>(g, s, A4, kp, i0, t, v, do_v, do_j, j_first);
    }
    if (i0 + 3 >= g.n) nib &= i0 >= g.n ? 0u : (1u << (g.n - i0)) - 1u;  // padding never fires
    if (do_v) {
      st_hint(reinterpret_cast<float4*>(g.V + i0), make_float4(s.V[0], s.V[1], s.V[2], s.V[3]), once);
      st_hint(reinterpret_cast<uint32_t*>(g.ref + i0), s.ref4, once);
      if (OU) st_hint(reinterpret_cast<float4*>(g.Iou + i0), make_float4(s.I[0], s.I[1], s.I[2], s.I[3]), once);
    }
    if (do_j) {
#pragma unroll
      for (int q = 0; q < 4; q++)
        st_hint(reinterpret_cast<float4*>(g.j + q * np + i0), make_float4(s.J[q][0], s.J[q][1], s.J[q][2], s.J[q][3]),
                once);
      if (!BINS) {
        // all of them, also where nothing had arrived: a sector of which one
        // thread's half is written is read again before it leaves the cache
        // (clearing only what was not zero: 18.5 us a step for 18.2 at 1M
        // neurons, 30.4 for 29.8 at 2M, 81.3 for 74.5 at 4M in ring mode)
#pragma unroll
        for (int cc = 0; cc < NCH; cc++)
          st_hint(reinterpret_cast<float4*>(acc_slot + cc * np + i0), make_float4(0.f, 0.f, 0.f, 0.f), once);
      }
    }
    // spike bits, and the tile's spikes and work items: the warp that is the
    // last one done with the tile stores them.  Most warps of 128 neurons have
    // no spike (p = 0.9 at 7 Hz, 0.7 at 30 Hz).
    uint32_t word = 0;
    int cnt = 0;
    if (__any_sync(0xFFFFFFFFu, nib != 0)) {
      word = nib << (4 * (lane & 7));
      word |= __shfl_xor_sync(0xFFFFFFFFu, word, 1);
      word |= __shfl_xor_sync(0xFFFFFFFFu, word, 2);
      word |= __shfl_xor_sync(0xFFFFFFFFu, word, 4);
      int nit = 0;  // delivery work items of my spiking neurons
      if (listing) {  // the spikes wait for the CTA's end, where their lookups run side by side
        int rank = 0;
        const int mine = __popc(nib);
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
          const int y = __shfl_up_sync(0xFFFFFFFFu, mine + rank, o);
          if (lane >= o) rank += y;
        }
        int at = 0;
        if (lane == 31) at = atomicAdd(&s_nspk, mine + rank);
        at = __shfl_sync(0xFFFFFFFFu, at, 31);
        const int all = __shfl_sync(0xFFFFFFFFu, mine + rank, 31);
        if (at + all <= kSpikeList) {
          at += rank;
#pragma unroll
          for (int q = 0; q < 4; q++)
            if ((nib >> q) & 1u) s_spk[at++] = (int32_t)i0 + q;
        } else {  // no room left (rare): listed here, and the slots marked empty
          for (int k = at + lane; k < min(at + all, kSpikeList); k += 32) s_spk[k] = -1;
#pragma unroll 1
          for (int q = 0; q < 4; q++) list_work(g, (nib >> q) & 1u ? (int32_t)i0 + q : -1, t, lane);
        }
      }
      cnt = __reduce_add_sync(0xFFFFFFFFu, __popc(nib));
      if (BINS) {
#pragma unroll
        for (int q = 0; q < 4; q++)
          if ((nib >> q) & 1u) {
            if (g.nitem_ok) {
              nit += (int)((ni4 >> (8 * q)) & 0xFFu);
            } else {
              const int64_t len = g.row_ptr[i0 + q + 1] - g.row_ptr[i0 + q];
              nit += (int)((len + kItemEvents - 1) / kItemEvents);
            }
          }
        nit = __reduce_add_sync(0xFFFFFFFFu, nit);
        if (lane == 0) atomicAdd(&s_items[k % kSlots], (uint32_t)nit);
      }
    }
    if ((lane & 7) == 0) g.flags[i0 >> 5] = word;  // i0 of lane 8q is the first neuron of word q
    if (lane == 0) {
      __threadfence_block();  // my items before my arrival
      const uint32_t old = atomicAdd(&s_done[k % kSlots], (1u << 28) | (uint32_t)cnt);
      if (old >> 28 == kWarps - 1) {
        __threadfence_block();
        g.blk_cnt[tile] = (int32_t)(old & 0xFFFFu) + cnt;
        if (BINS) {
          g.blk_items[tile] = (int32_t)s_items[k % kSlots];
          s_items[k % kSlots] = 0;
        }
        s_done[k % kSlots] = 0;
      }
    }
  }
  // gave up (any warp): let the copies still in flight land before the CTA exits
  const bool gave_up = __syncthreads_or(bad);
  if (listing) {
    const int n_spk = min(s_nspk, kSpikeList);
    for (int k = tid & ~31; k < n_spk; k += kThr) list_work(g, k + lane < n_spk ? s_spk[k + lane] : -1, t, lane);
  }
  if (gave_up && tid == 0) {
    for (int q = 0; q < S; q++) {
      const uint32_t full = s_taken[q] / kWarps;  // tiles of this stage that every warp took
      if (q + (int)full * S < n_mine) (void)mbar_wait_bounded(&bar[q], full & 1u);
    }
    if (ev_pending >= 0) (void)mbar_wait_bounded(&ebar, (uint32_t)ev_pending & 1u);
  }
}

// ==== end of the neuron update ====  A recorded DRAM traffic of the update
// kernel is keyed by a hash of this file up to this line and of dtb_device.cuh.
__device__ __forceinline__ int warp_incl_scan(int x, int lane) {
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int y = __shfl_up_sync(0xFFFFFFFFu, x, o);
    if (lane >= o) x += y;
  }
  return x;
}

// Work items of neuron id's row (ceil(len / kItemEvents)), from the per-neuron
// byte when every row fits in it, else from the row bounds.
__device__ __forceinline__ int items_of(const DevNet& g, int32_t id) {
  if (g.nitem_ok) return (int)__ldg(g.nitem + id);
  const int64_t len = __ldg(g.row_ptr + id + 1) - __ldg(g.row_ptr + id);
  return (int)((len + kItemEvents - 1) / kItemEvents);
}

// Block-wide exclusive scan of one value per thread (256 threads); returns the
// thread's exclusive prefix and sets *total.  Two barriers; s holds 8 ints.
__device__ __forceinline__ int block_excl_scan(int x, int* s, int* total) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int inc = warp_incl_scan(x, lane);
  if (lane == 31) s[warp] = inc;
  __syncthreads();
  int before = 0, all = 0;
#pragma unroll
  for (int k = 0; k < 8; k++) {
    const int v = s[k];
    if (k < warp) before += v;
    all += v;
  }
  __syncthreads();
  *total = all;
  return before + inc - x;
}

// Compaction: CTA = tile of 64 neuron blocks (65,536 neurons, 2,048 spike-bit
// words).  Thread i owns words 8i .. 8i+7, so thread order is neuron order and
// one block scan ranks the ids.  The tile's base offsets are sums of all
// earlier blocks' counts, re-read from L2 by every CTA: no inter-CTA waiting.
// Work items are then built in rounds of up to kRound spikes: the round's ids
// go to shared memory in rank order, one thread per spike looks up its item
// count, a block scan places the items, and one thread per item (its spike
// found by binary search over the scan) looks up its chunk's run table.  No
// thread walks a chain of lookups per spike or per item, so a tile with a
// crowded word or a row of many items costs a few memory latencies, not one
// per spike.
// In the queue and ring modes the update lists the delivery's work and no work
// items are built here.
//
// BESIDE: the instance of the networks whose compaction runs beside an update,
// with the update's division of an SM's memory; the other keeps its own, which
// leaves it more L1 (20M neurons, 30 Hz: 18.4 us alone for 23.2 all shared, and
// the step, with the deliveries' division also their own, 381 for 401).
template <bool BESIDE>
__global__ void __launch_bounds__(256) spike_compact_kernel(DevNet g, int32_t t_rel) {
  constexpr int kWords = 8;    // spike-bit words per thread
  constexpr int kRound = 1024; // spikes per round of item building
  const int tile = blockIdx.x;
  const int b0 = tile * kCompactBlocksPerTile;
  const int words = min(kCompactBlocksPerTile, g.nblk - b0) * 32;  // a multiple of kWords
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  // steps alternate between two copies of the spike list and its count (the BOLD
  // step reads one while the next compaction writes the other) and of the log's
  // position: this step's is read, the next one's written by the last tile
  const int par = g.t_base ? (int)((*g.t_base + t_rel) & 1) : 0;
  int32_t* spk = g.spk + par * g.spk_par;
  const bool with_items = g.items != nullptr;
  // the log's bookkeeping is one thread's; what it needs is loaded here, ahead
  // of the chain of lookups that the kernel's time consists of
  const bool keeps_log = tile == (int)gridDim.x - 1 && threadIdx.x == 0 && g.step_off != nullptr;
  int64_t log_pos = 0;
  int32_t log_step = 0;
  if (keeps_log) {
    log_pos = g.log_pos[par];
    log_step = *g.call_steps;
  }
  __shared__ int s_part[8], s_ipart[8], s_scan[8];
  __shared__ int32_t s_id[kRound];
  __shared__ int s_it[kRound + 1];

  uint32_t w[kWords];
  const int w0 = tid * kWords;
  if (w0 < words) {
    const uint4* f = reinterpret_cast<const uint4*>(g.flags + (int64_t)b0 * 32 + w0);
    const uint4 x = f[0], y = f[1];
    w[0] = x.x; w[1] = x.y; w[2] = x.z; w[3] = x.w;
    w[4] = y.x; w[5] = y.y; w[6] = y.z; w[7] = y.w;
  } else {
#pragma unroll
    for (int k = 0; k < kWords; k++) w[k] = 0u;
  }

  // the counts of all earlier blocks (b0 is a multiple of 64): 16-byte loads,
  // several in flight per thread, so that the last tiles (tens of thousands
  // of earlier blocks) do not wait on a chain of L2 round trips
  int part = 0, ipart = 0;
  {
    const int4* c4 = reinterpret_cast<const int4*>(g.blk_cnt);
    const int4* i4 = reinterpret_cast<const int4*>(g.blk_items);
    const int n4 = b0 >> 2;
#pragma unroll 4
    for (int q = tid; q < n4; q += 256) {
      const int4 v = c4[q];
      part += (v.x + v.y) + (v.z + v.w);
      if (with_items) {
        const int4 u = i4[q];
        ipart += (u.x + u.y) + (u.z + u.w);
      }
    }
  }
  part = __reduce_add_sync(0xFFFFFFFFu, part);
  ipart = __reduce_add_sync(0xFFFFFFFFu, ipart);
  if (lane == 0) {
    s_part[warp] = part;
    s_ipart[warp] = ipart;
  }

  const int32_t id0 = (b0 * 32 + w0) * 32;  // first neuron of this thread's words
  int c = 0;
#pragma unroll
  for (int k = 0; k < kWords; k++) c += __popc(w[k]);
  int tot;
  const int r0 = block_excl_scan(c, s_scan, &tot);  // its barriers also publish s_part, s_ipart
  int base = 0, ibase = 0;
#pragma unroll
  for (int k = 0; k < 8; k++) {
    base += s_part[k];
    ibase += s_ipart[k];
  }

  if (c) {
    const int64_t lp = g.log_cap ? g.log_pos[par] : 0;
    int pos = base + r0;
#pragma unroll
    for (int k = 0; k < kWords; k++)
      for (uint32_t bits = w[k]; bits; bits &= bits - 1) {
        const int32_t id = id0 + 32 * k + __ffs(bits) - 1;
        spk[pos] = id;
        if (lp + pos < g.log_cap) g.log_ids[lp + pos] = id;
        pos++;
      }
  }

  int itot = 0;
  if (with_items) {
    for (int lo = 0; lo < tot; lo += kRound) {
      const int nr = min(kRound, tot - lo);
      // this round's ids in rank order
      if (c && r0 < lo + kRound && r0 + c > lo) {
        int r = r0;
#pragma unroll
        for (int k = 0; k < kWords; k++)
          for (uint32_t bits = w[k]; bits; bits &= bits - 1, r++)
            if (r >= lo && r < lo + kRound) s_id[r - lo] = id0 + 32 * k + __ffs(bits) - 1;
      }
      __syncthreads();
      // item counts, four spikes per thread (consecutive, for the scan), loads in flight together
      int cnt[4], sum = 0;
#pragma unroll
      for (int q = 0; q < 4; q++) {
        const int j = 4 * tid + q;
        cnt[q] = j < nr ? items_of(g, s_id[j]) : 0;
      }
#pragma unroll
      for (int q = 0; q < 4; q++) sum += cnt[q];
      int rtot;
      int e = block_excl_scan(sum, s_scan, &rtot);
#pragma unroll
      for (int q = 0; q < 4; q++) {
        const int j = 4 * tid + q;
        if (j < nr) s_it[j] = e;
        e += cnt[q];
      }
      if (tid == 0) s_it[nr] = rtot;
      __syncthreads();
      // one thread per item of the round
      for (int j = tid; j < rtot; j += 256) {
        int lo_k = 0, hi_k = nr - 1;  // the last spike whose first item is <= j
        while (lo_k < hi_k) {
          const int mid = (lo_k + hi_k + 1) >> 1;
          if (s_it[mid] <= j) lo_k = mid;
          else hi_k = mid - 1;
        }
        const int32_t id = s_id[lo_k];
        const int64_t q = j - s_it[lo_k];
        const int64_t rb = __ldg(g.row_ptr + id), len = __ldg(g.row_ptr + id + 1) - rb;
        const int64_t cb = g.run_ptr ? __ldg(g.chunk_base + id) : 0;
        WorkItem it;
        it.e0 = rb + q * kItemEvents;
        it.len = (int32_t)min(len - q * kItemEvents, (int64_t)kItemEvents);
        it.src = id;
        it.rp0 = 0;
        it.nr = 0;
        it.pad = 0;
        if (g.run_ptr) {  // the chunk's run table, so that delivery needs no further lookup
          it.rp0 = __ldg(g.run_ptr + cb + q);
          it.nr = (int32_t)(__ldg(g.run_ptr + cb + q + 1) - it.rp0);
        }
        g.items[ibase + itot + j] = it;
      }
      itot += rtot;
      __syncthreads();  // s_id and s_it are rewritten by the next round
    }
  }
  if (tile == gridDim.x - 1 && tid == 0) {
    const int total = base + tot;
    g.n_spk[par] = total;
    if (keeps_log) {
      log_pos += total;
      if (log_pos > g.log_cap) {
        log_pos = g.log_cap;
        *g.log_trunc = 1;
      }
      g.step_off[log_step + 1] = log_pos;
      g.log_pos[par ^ 1] = log_pos;
      *g.call_steps = log_step + 1;
    }
    if (with_items) *g.n_items = ibase + itot;
    if (g.spikes) atomicAdd(g.spikes, (unsigned long long)total);
  }
}

__device__ __forceinline__ int lower_bound(const int32_t* a, int n, int32_t x) {
  int lo = 0, hi = n;
  while (lo < hi) {
    const int mid = (lo + hi) >> 1;
    if (a[mid] < x) lo = mid + 1; else hi = mid;
  }
  return lo;
}

// Balloon-Windkessel, one Euler step of one voxel's state s, f, v, q at input z (Hz).
__device__ __forceinline__ float bold_euler(const BoldConst& b, float z, float& s, float& f, float& vv, float& q) {
  const float fout = powf(vv, b.inv_alpha);
  const float Ef = 1.0f - expf(b.ln_1mE0 / f);
  const float ds = b.eps * z - s * b.inv_tau_s - (f - 1.0f) * b.inv_tau_f;
  const float df = s;
  const float dv = (f - fout) * b.inv_tau_0;
  const float dq = (f * Ef * b.inv_E0 - fout * q / vv) * b.inv_tau_0;
  s += b.dt_s * ds;
  f += b.dt_s * df;
  vv += b.dt_s * dv;
  q += b.dt_s * dq;
  return b.V0 * (b.k1 * (1.0f - q) + b.k2 * (1.0f - q / vv) + b.k3 * (1.0f - vv));
}

// Balloon-Windkessel, one thread per voxel.  z = spikes / (n_v * dt) in Hz,
// counted by binary search of the voxel's id range in the ascending list.
template <bool BESIDE>  // as for the compaction
__global__ void bold_step_kernel(DevNet g, int32_t t_rel) {
  const int v = blockIdx.x * blockDim.x + threadIdx.x;
  const int64_t t = *g.t_base + t_rel;
  if (v >= g.nv) return;
  const int n_spk = g.n_spk[t & 1];
  const int32_t* spk = g.spk + (t & 1) * g.spk_par;
  const int cnt = lower_bound(spk, n_spk, g.vstart[v + 1]) - lower_bound(spk, n_spk, g.vstart[v]);
  g.vox_spikes[v] += (unsigned long long)cnt;
  const float z = (float)cnt * g.inv_nvox[v];
  const int nv = g.nv;
  float s = g.bold[v], f = g.bold[nv + v], vv = g.bold[2 * nv + v], q = g.bold[3 * nv + v];
  const float y = bold_euler(g.bc, z, s, f, vv, q);
  g.bold[v] = s;
  g.bold[nv + v] = f;
  g.bold[2 * nv + v] = vv;
  g.bold[3 * nv + v] = q;
  g.bold[4 * nv + v] = y;
  if (g.bold_every > 0 && (t + 1) % g.bold_every == 0) {
    const int64_t idx = (t + 1) / g.bold_every - 1;
    g.bold_log[(idx % g.bold_cap) * nv + v] = y;
  }
}

// ---- networks of at most kSmallBlocks blocks: a call in one CTA ----
//
// A step of a network of a few thousand neurons is a chain of dependent
// launches: 6.9 us a step for 1,000 neurons with 100 synapses each, whose
// arithmetic takes well under one (2.8 us with this kernel).  Here one CTA runs
// all the steps of a call with V, j and the refractory counters in registers
// (four neurons per thread); only the delay ring, the synapses and the BOLD state
// are in global memory.  One barrier a step:
//   before it  j part of step t - 1 and V part of step t; the spikes go to a
//              list in shared memory with their rows' bounds;
//   barrier    the list is complete, and what step t - 1 delivered is visible;
//   after it   the arrivals of step t are fetched for the next iteration (they
//              were all delivered by step t - 1) and the list's rows are
//              delivered, a warp each; helper warps without neurons advance the
//              spike log and the BOLD step as well.
// What bounds a step is the chain of one trip to L2 for the rows, one for the
// sums, and the neuron's own arithmetic.
constexpr int kSmallBlocks = 3;

__device__ __forceinline__ int32_t synapse_weight(const DevNet& g, int64_t e, int32_t src) {
  switch (g.wfmt) {
    case 0: return decode_weight(weight_code<0>(g.w, e, 0), 0, g.wshift);
    case 1: return decode_weight(weight_code<1>(g.w, e, 0), 1, g.wshift);
    case 2: return decode_weight(weight_code<2>(g.w, e, 0), 2, g.wshift);
    default: return decode_weight(weight_code<3>(g.w, e, g.wshift + (g.row_shift ? g.row_shift[src] : 0)), 3, g.wshift);
  }
}

// Dynamic shared memory: spike list and rows, two copies (a list is read after
// its step's barrier and written again before the barrier two steps on); counts,
// bits and voxel counts [nv], three copies (step k clears those of step k + 2,
// which nobody touches between the barriers around it).
struct SmallSmem {
  static constexpr int kN = kSmallBlocks * kNeuronsPerBlock;
  static constexpr size_t kRow = 0;                          // int64 [2][kN] row starts
  static constexpr size_t kLen = kRow + 2 * kN * 8;          // int32 [2][kN] row lengths
  static constexpr size_t kId = kLen + 2 * kN * 4;           // int32 [2][kN] ids, in no order
  static constexpr size_t kBits = kId + 2 * kN * 4;          // uint32 [3][kN / 32]
  static constexpr size_t kVox = kBits + 3 * (kN / 32) * 4;  // int32 [3][nv]
  static constexpr size_t bytes(int nv) { return kVox + 3 * (size_t)nv * 4; }
};

template <int NCH, bool OU, int MAXT>
__global__ void __launch_bounds__(MAXT, 1) small_steps_kernel(DevNet g, int32_t n_steps) {
  using L = SmallSmem;
  extern __shared__ __align__(16) unsigned char ssm[];
  int64_t* s_row = reinterpret_cast<int64_t*>(ssm + L::kRow);
  int32_t* s_len = reinterpret_cast<int32_t*>(ssm + L::kLen);
  int32_t* s_id = reinterpret_cast<int32_t*>(ssm + L::kId);
  uint32_t* s_bits = reinterpret_cast<uint32_t*>(ssm + L::kBits);
  int32_t* s_vox = reinterpret_cast<int32_t*>(ssm + L::kVox);
  __shared__ int s_n[3];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int nthr = g.nblk * kUpdateThreads, nwarp = nthr / 32;  // with neurons
  const int nhelp = (int)blockDim.x - nthr;                      // threads without
  const bool helper = tid >= nthr;
  const int nv = g.nv;
  const int64_t np = g.npad, t0 = *g.t_base;
  const int64_t i0 = (int64_t)tid * 4;
  // my neurons
  Quad s = {};
  if (!helper) {
    const float4 v = *reinterpret_cast<const float4*>(g.V + i0);
    s.V[0] = v.x; s.V[1] = v.y; s.V[2] = v.z; s.V[3] = v.w;
#pragma unroll
    for (int q = 0; q < 4; q++) {
      const float4 j = *reinterpret_cast<const float4*>(g.j + q * np + i0);
      s.J[q][0] = j.x; s.J[q][1] = j.y; s.J[q][2] = j.z; s.J[q][3] = j.w;
    }
    s.ref4 = *reinterpret_cast<const uint32_t*>(g.ref + i0);
    const float4 I = OU ? *reinterpret_cast<const float4*>(g.Iou + i0) : make_float4(0.f, 0.f, 0.f, 0.f);
    s.I[0] = I.x; s.I[1] = I.y; s.I[2] = I.z; s.I[3] = I.w;
  }
  // voxel of my first neuron, from the coarse table (from the first voxel on, a call
  // on 3,000 voxels began with up to 3,000 dependent loads: 232 us for one of one step)
  int32_t v0 = g.coarse[min(i0, g.n - 1) >> g.coarse_shift];
  while (!helper && v0 + 1 < nv && g.vstart[v0 + 1] <= i0) v0++;
  const bool mixed = v0 + 1 < nv && g.vstart[v0 + 1] <= i0 + 3;
  // BOLD: a helper's first voxel (from the last thread on) in registers, further
  // ones through memory
  const int my_vox = helper ? (int)blockDim.x - 1 - tid : nv;
  float bs = 0.f, bf = 1.f, bv = 1.f, bq = 1.f, by = 0.f;
  unsigned long long vox_total = 0;
  if (my_vox < nv) {
    bs = g.bold[my_vox]; bf = g.bold[nv + my_vox]; bv = g.bold[2 * nv + my_vox]; bq = g.bold[3 * nv + my_vox];
    by = g.bold[4 * nv + my_vox];
  }
  int64_t log_pos = g.log_pos[t0 & 1];
  const int32_t cs0 = *g.call_steps;
  bool trunc = false;
  unsigned long long events = 0, spikes = 0;
  for (int k = tid; k < 3 * nv; k += (int)blockDim.x) s_vox[k] = 0;
  for (int k = tid; k < 3 * L::kN / 32; k += (int)blockDim.x) s_bits[k] = 0;
  if (tid < 3) s_n[tid] = 0;
  __syncthreads();

  int32_t slot = (int32_t)(t0 % g.D);  // of step t
  int4 A4[NCH];                        // arrivals of the step before
#pragma unroll
  for (int cc = 0; cc < NCH; cc++) A4[cc] = make_int4(0, 0, 0, 0);
  bool sent = false;                   // this warp delivered in the step before
  auto j_part = [&](int64_t x) {
    const uint4 r = philox4x32_10(make_uint4((uint32_t)(i0 >> 2), (uint32_t)x, (uint32_t)((uint64_t)x >> 32), kTagDrive),
                                  g.key0, g.key1);
    const uint32_t u[4] = {r.x, r.y, r.z, r.w};
    int32_t kp[4];
#pragma unroll
    for (int q = 0; q < 4; q++) {
      kp[q] = poisson_low(g, u[q]);
      if (g.M > 3 && u[q] >= g.T[2]) kp[q] += poisson_high(g, u[q]);
    }
    if (!mixed) quad_j<NCH>(g, g.vc[v0], s, A4, kp);
    else (void)quad_mixed<NCH, false>(g, s, A4, kp, i0, x, v0, false, true, false);
  };
  auto fetch = [&](int32_t sl) {  // my neurons' sums of slot sl, which are cleared
#pragma unroll
    for (int cc = 0; cc < NCH; cc++) {
      int4* p = reinterpret_cast<int4*>(g.ring + ((int64_t)sl * NCH + cc) * np + i0);
      A4[cc] = __ldcg(p);
      if (A4[cc].x | A4[cc].y | A4[cc].z | A4[cc].w) __stcg(p, make_int4(0, 0, 0, 0));
    }
  };
  for (int32_t k = 0, c = 0; k < n_steps; k++, c = c == 2 ? 0 : c + 1) {  // c: copy k mod 3
    const int64_t t = t0 + k;
    const int par = k & 1;
    uint32_t* bits = s_bits + c * (L::kN / 32);
    int32_t* vox = s_vox + c * nv;
    if (k > 0 && !helper) j_part(t - 1);
    uint32_t nib = 0;
    if (helper) {
    } else if (!mixed) {
      nib = quad_v<OU>(g, g.vc[v0], s, i0, t);
    } else {
      const int32_t none[4] = {0, 0, 0, 0};
      nib = quad_mixed<NCH, OU>(g, s, A4, none, i0, t, v0, true, false, false);
    }
    if (i0 + 3 >= g.n) nib &= i0 >= g.n ? 0u : (1u << (g.n - i0)) - 1u;  // padding never fires
    if (nib) {
      atomicOr(&bits[tid >> 3], nib << (4 * (tid & 7)));
      int at = atomicAdd(&s_n[c], __popc(nib));
#pragma unroll
      for (int q = 0; q < 4; q++)
        if ((nib >> q) & 1u) {
          const int32_t id = (int32_t)i0 + q;
          const int64_t a = __ldg(g.row_ptr + id);
          s_id[par * L::kN + at] = id;
          s_row[par * L::kN + at] = a;
          s_len[par * L::kN + at] = (int32_t)(__ldg(g.row_ptr + id + 1) - a);
          int32_t v = v0;
          while (v + 1 < nv && g.vstart[v + 1] <= id) v++;
          atomicAdd(&vox[v], 1);
          at++;
        }
    }
    if (sent) __threadfence();  // my deliveries of step t - 1 before the barrier
    __syncthreads();
    const int n = s_n[c];
    sent = warp < n;
    if (!helper) fetch(slot);
    // rows of the list, a warp each (long ones are walked by their warp)
    for (int l = warp; l < n; l += (int)(blockDim.x >> 5)) {
      const int64_t a = s_row[par * L::kN + l];
      const int len = s_len[par * L::kN + l];
      const int32_t src = s_id[par * L::kN + l];
      if (lane == 0) events += (unsigned long long)len;
      for (int e0 = lane; e0 < len; e0 += 128) {
        uint32_t wd[4];
        int32_t wa[4], dd[4];
#pragma unroll
        for (int u = 0; u < 4; u++) {
          const bool in = e0 + 32 * u < len;
          const int64_t e = a + (in ? e0 + 32 * u : 0);
          wd[u] = __ldg(g.word + e);
          wa[u] = synapse_weight(g, e, src);
          dd[u] = in ? (int32_t)__ldg(g.syn_delay + e) : 0;
        }
#pragma unroll
        for (int u = 0; u < 4; u++) {
          if (dd[u] == 0) continue;
          int32_t sl = slot + dd[u];
          if (sl >= g.D) sl -= g.D;
          atomicAdd(g.ring + ((int64_t)sl * NCH + (wd[u] >> 30)) * np + (wd[u] & 0x3FFFFFFFu), wa[u]);
        }
      }
    }
    // the spike log: a spike's rank is the number of bits below its own
    if (warp == nwarp) {
      for (int l = lane; l < n; l += 32) {
        const int32_t id = s_id[par * L::kN + l];
        int rank = __popc(bits[id >> 5] & ((1u << (id & 31)) - 1u));
        for (int w = 0; w < (id >> 5); w++) rank += __popc(bits[w]);
        if (log_pos + rank < g.log_cap) g.log_ids[log_pos + rank] = id;
      }
      log_pos += n;
      if (log_pos > g.log_cap) {
        log_pos = g.log_cap;
        trunc = true;
      }
      if (lane == 0) g.step_off[cs0 + k + 1] = log_pos;
      spikes += (unsigned long long)n;
    }
    // BOLD
    const bool sample = g.bold_every > 0 && (t + 1) % g.bold_every == 0;
    float* row = sample ? g.bold_log + (((t + 1) / g.bold_every - 1) % g.bold_cap) * nv : nullptr;
    if (my_vox < nv) {
      const int fired = vox[my_vox];
      vox_total += (unsigned long long)fired;
      by = bold_euler(g.bc, (float)fired * g.inv_nvox[my_vox], bs, bf, bv, bq);
      if (row) row[my_vox] = by;
    }
    for (int v = my_vox + nhelp; v < nv; v += nhelp) {
      const int fired = vox[v];
      g.vox_spikes[v] += (unsigned long long)fired;
      float a = g.bold[v], b = g.bold[nv + v], d = g.bold[2 * nv + v], q = g.bold[3 * nv + v];
      const float y = bold_euler(g.bc, (float)fired * g.inv_nvox[v], a, b, d, q);
      g.bold[v] = a; g.bold[nv + v] = b; g.bold[2 * nv + v] = d; g.bold[3 * nv + v] = q; g.bold[4 * nv + v] = y;
      if (row) row[v] = y;
    }
    // clear the copies of step k + 2
    const int c2 = c == 0 ? 2 : c - 1;
    if (helper) {
      if (tid == nthr) s_n[c2] = 0;
      for (int w = tid - nthr; w < L::kN / 32; w += nhelp) s_bits[c2 * (L::kN / 32) + w] = 0;
      for (int v = tid - nthr; v < nv; v += nhelp) s_vox[c2 * nv + v] = 0;
    }
    slot = slot + 1 == g.D ? 0 : slot + 1;
  }
  if (!helper) {
    j_part(t0 + n_steps - 1);
    // the state back
    *reinterpret_cast<float4*>(g.V + i0) = make_float4(s.V[0], s.V[1], s.V[2], s.V[3]);
#pragma unroll
    for (int q = 0; q < 4; q++)
      *reinterpret_cast<float4*>(g.j + q * np + i0) = make_float4(s.J[q][0], s.J[q][1], s.J[q][2], s.J[q][3]);
    *reinterpret_cast<uint32_t*>(g.ref + i0) = s.ref4;
    if (OU) *reinterpret_cast<float4*>(g.Iou + i0) = make_float4(s.I[0], s.I[1], s.I[2], s.I[3]);
  }
  if (my_vox < nv) {
    g.bold[my_vox] = bs; g.bold[nv + my_vox] = bf; g.bold[2 * nv + my_vox] = bv; g.bold[3 * nv + my_vox] = bq;
    g.bold[4 * nv + my_vox] = by;
    g.vox_spikes[my_vox] += vox_total;
  }
  if (lane == 0 && events) atomicAdd(g.events, events);
  if (tid < 3) g.chunk_cnt[tid] = 0;  // the lists of a network that is stepped by the other kernels next
  if (tid == nthr) {
    g.log_pos[0] = g.log_pos[1] = log_pos;
    if (trunc) *g.log_trunc = 1;
    *g.call_steps = cs0 + n_steps;
    *g.spikes += spikes;
    *g.t_base = t0 + n_steps;
  }
}

__global__ void advance_kernel(int64_t* t_base, int32_t k) { *t_base += k; }

// After a j-only update of step t: its arrivals' spill slot is consumed.
__global__ void spill_clear_kernel(DevNet g, int32_t t_rel) {
  if (g.mode) g.spill_dirty[(*g.t_base + t_rel) % g.D] = 0;
}

__global__ void begin_call_kernel(DevNet g) {
  g.log_pos[0] = g.log_pos[1] = 0;
  *g.call_steps = 0;
  *g.log_trunc = 0;
  g.step_off[0] = 0;
}

template <int NCH, int S, bool OU, bool BINS, bool BODY>
cudaError_t launch_update(const DevNet& g, int32_t t_rel, cudaStream_t st, int blocks_per_sm, int32_t upd) {
  using St = Stage<NCH, OU, BINS>;
  static DeviceLaunch cache[kMaxDevices];  // per instance and device
  static std::mutex mu;
  const int smem = (int)St::bytes(S);
  DeviceLaunch dl;
  cudaError_t e0 = device_launch(cache, mu, [&](DeviceLaunch& d) {
    cudaError_t e = cudaFuncSetAttribute(neuron_update_kernel<NCH, S, OU, BINS, BODY>,
                                         cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
    if (e == cudaSuccess) e = share_sm_division(neuron_update_kernel<NCH, S, OU, BINS, BODY>);
    if (e != cudaSuccess) return e;
    int per = 0;
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, neuron_update_kernel<NCH, S, OU, BINS, BODY>, kUpdateThreads,
                                                      smem);
    d.per_sm = per > 0 ? per : 1;
    return e;
  }, &dl);
  if (e0 != cudaSuccess) return e0;
  const int sms = dl.sms, max_per_sm = dl.per_sm;
  const int per = blocks_per_sm > 0 && blocks_per_sm < max_per_sm ? blocks_per_sm : max_per_sm;
  const int grid = sms * per;  // persistent grid: SMs x resident CTAs
  const int units = BINS ? g.n_reg : g.nblk;  // regions or tiles
  int blocks = grid < units ? grid : units;
  if (BINS && blocks * kMaxRegionsPerCta < units) blocks = (units + kMaxRegionsPerCta - 1) / kMaxRegionsPerCta;
  neuron_update_kernel<NCH, S, OU, BINS, BODY><<<blocks, kUpdateThreads, smem, st>>>(g, t_rel, upd);
  return cudaGetLastError();
}

template <int NCH, int S, bool OU, bool BINS>
cudaError_t launch_update_mode(const DevNet& g, int32_t t_rel, cudaStream_t st, int blocks_per_sm, int32_t upd) {
  return upd == kUpdJV ? launch_update<NCH, S, OU, BINS, true>(g, t_rel, st, blocks_per_sm, upd)
                       : launch_update<NCH, S, OU, BINS, false>(g, t_rel, st, blocks_per_sm, upd);
}

// Stages: 2..4 with two channels, 2..3 with four.
template <bool OU, bool BINS>
cudaError_t launch_update_ou(const DevNet& g, int32_t t_rel, cudaStream_t st, int stages, int blocks_per_sm,
                             int32_t upd) {
  if (g.nch == 2) {
    if (stages == 2) return launch_update_mode<2, 2, OU, BINS>(g, t_rel, st, blocks_per_sm, upd);
    if (stages == 4) return launch_update_mode<2, 4, OU, BINS>(g, t_rel, st, blocks_per_sm, upd);
    return launch_update_mode<2, 3, OU, BINS>(g, t_rel, st, blocks_per_sm, upd);
  }
  if (stages == 3) return launch_update_mode<4, 3, OU, BINS>(g, t_rel, st, blocks_per_sm, upd);
  return launch_update_mode<4, 2, OU, BINS>(g, t_rel, st, blocks_per_sm, upd);
}

}  // namespace

cudaError_t launch_neuron_update(const DevNet& g, int32_t t_rel, cudaStream_t st, int stages, int blocks_per_sm,
                                 int32_t upd) {
  if (g.mode == kModeBins)
    return g.ou ? launch_update_ou<true, true>(g, t_rel, st, stages, blocks_per_sm, upd)
                : launch_update_ou<false, true>(g, t_rel, st, stages, blocks_per_sm, upd);
  return g.ou ? launch_update_ou<true, false>(g, t_rel, st, stages, blocks_per_sm, upd)
              : launch_update_ou<false, false>(g, t_rel, st, stages, blocks_per_sm, upd);
}

// Voxels may be empty, so there can be more of them than neurons: the voxel
// counts have room in shared memory for one voxel per neuron.
bool small_network(const DevNet& g) { return g.nblk <= kSmallBlocks && g.nv <= SmallSmem::kN; }

int small_warps(const DevNet& g) { return g.nblk == 1 ? 16 : 32; }

cudaError_t launch_small_steps(const DevNet& g, int32_t n_steps, cudaStream_t st) {
  static DeviceLaunch cache[kMaxDevices];
  static std::mutex mu;
  DeviceLaunch dl;
  const int most = (int)SmallSmem::bytes(SmallSmem::kN);  // a voxel per neuron
  const cudaError_t e = device_launch(cache, mu, [&](DeviceLaunch& d) {
    cudaError_t r = cudaSuccess;
    for (const void* f : {(const void*)small_steps_kernel<2, false, 512>, (const void*)small_steps_kernel<2, true, 512>,
                          (const void*)small_steps_kernel<4, false, 512>, (const void*)small_steps_kernel<4, true, 512>,
                          (const void*)small_steps_kernel<2, false, 1024>, (const void*)small_steps_kernel<2, true, 1024>,
                          (const void*)small_steps_kernel<4, false, 1024>, (const void*)small_steps_kernel<4, true, 1024>})
      if (r == cudaSuccess) r = cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, most);
    d.per_sm = 1;
    return r;
  }, &dl);
  if (e != cudaSuccess) return e;
  const size_t smem = SmallSmem::bytes(g.nv);
  const bool few = g.nblk == 1;  // half the threads with twice the registers each, none of them spilled
  auto run = [&](auto kernel) { kernel<<<1, 32 * small_warps(g), smem, st>>>(g, n_steps); };
  if (g.nch == 2) {
    if (g.ou) few ? run(small_steps_kernel<2, true, 512>) : run(small_steps_kernel<2, true, 1024>);
    else few ? run(small_steps_kernel<2, false, 512>) : run(small_steps_kernel<2, false, 1024>);
  } else {
    if (g.ou) few ? run(small_steps_kernel<4, true, 512>) : run(small_steps_kernel<4, true, 1024>);
    else few ? run(small_steps_kernel<4, false, 512>) : run(small_steps_kernel<4, false, 1024>);
  }
  return cudaGetLastError();
}

cudaError_t prepare_step_kernels() {
  return share_sm_division(spike_compact_kernel<true>, bold_step_kernel<true>, advance_kernel, begin_call_kernel,
                           spill_clear_kernel);
}

cudaError_t launch_spike_compact(const DevNet& g, int32_t t_rel, cudaStream_t st) {
  if (g.beside) spike_compact_kernel<true><<<g.ntiles, 256, 0, st>>>(g, t_rel);
  else spike_compact_kernel<false><<<g.ntiles, 256, 0, st>>>(g, t_rel);
  return cudaGetLastError();
}

cudaError_t launch_spill_clear(const DevNet& g, int32_t t_rel, cudaStream_t st) {
  spill_clear_kernel<<<1, 1, 0, st>>>(g, t_rel);
  return cudaGetLastError();
}

cudaError_t launch_bold_step(const DevNet& g, int32_t t_rel, cudaStream_t st) {
  const int blocks = (g.nv + 127) / 128;
  if (g.beside) bold_step_kernel<true><<<blocks, 128, 0, st>>>(g, t_rel);
  else bold_step_kernel<false><<<blocks, 128, 0, st>>>(g, t_rel);
  return cudaGetLastError();
}

cudaError_t launch_advance(const DevNet& g, int32_t k, cudaStream_t st) {
  advance_kernel<<<1, 1, 0, st>>>(g.t_base, k);
  return cudaGetLastError();
}

cudaError_t launch_begin_call(const DevNet& g, cudaStream_t st) {
  begin_call_kernel<<<1, 1, 0, st>>>(g);
  return cudaGetLastError();
}

}  // namespace dtb

// setup_kernels.cu -- kernels run once per network (initial state, synapse
// table validation and int32 overflow bound) and the Philox test hook.
#include <cuda_runtime.h>
#include <stdint.h>

#include "dtb_device.cuh"
#include "dtb_launch.h"

namespace dtb {
namespace {

// V0 = Vreset + (Vth - Vreset) * ((word >> 8) * 2^-24), word = Philox({i/4, 0, 0, INIT})[i mod 4].
__global__ void init_voltage_kernel(DevNet g, uint32_t k0, uint32_t k1) {
  const int64_t i0 = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) * 4;
  if (i0 >= g.npad) return;
  const uint4 r = philox4x32_10(make_uint4((uint32_t)(i0 >> 2), 0u, 0u, kTagInit), k0, k1);
  const uint32_t rq[4] = {r.x, r.y, r.z, r.w};
  float out[4];
  int32_t v = g.blk_vox[i0 / kNeuronsPerBlock];
#pragma unroll
  for (int q = 0; q < 4; q++) {
    while (v + 1 < g.nv && g.vstart[v + 1] <= i0 + q) v++;
    const VoxConst* c = g.vc + v;
    const float u = __fmul_rn((float)(rq[q] >> 8), 5.9604644775390625e-08f);  // 2^-24, exact
    const float span = __fsub_rn(c->Vth, c->Vreset);
    out[q] = __fadd_rn(c->Vreset, __fmul_rn(span, u));
  }
  *reinterpret_cast<float4*>(g.V + i0) = make_float4(out[0], out[1], out[2], out[3]);
}

template <int WFMT>
__device__ __forceinline__ int64_t acc_weight(const DevNet& g, int64_t e, int shift) {
  if (WFMT == 0) return (int64_t)reinterpret_cast<const int16_t*>(g.w)[e] * ((int64_t)1 << shift);
  if (WFMT == 1) return (int64_t)reinterpret_cast<const int32_t*>(g.w)[e] * ((int64_t)1 << shift);
  if (WFMT == 2) {
    const uint32_t b = (uint32_t)reinterpret_cast<const unsigned short*>(g.w)[e] << 16;
    const float x = __fmul_rn(__uint_as_float(b), 65536.0f);
    if (!(fabsf(x) < 2147483520.0f)) return (int64_t)1 << 40;
    return (int64_t)__float2int_rn(x);
  }
  return (int64_t)reinterpret_cast<const signed char*>(g.w)[e] * ((int64_t)1 << shift);
}

// Warp per row.  Rows must be ascending and within [0, nnz]; every entry's
// target < n and class < nch; |w_acc| summed per (target, channel).
template <int WFMT>
__global__ void check_kernel(DevNet g, unsigned long long* insum, int* bad) {
  const int lane = threadIdx.x & 31;
  const int64_t gw = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const int64_t nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
  for (int64_t s = gw; s < g.n; s += nw) {
    const int64_t r0 = g.row_ptr[s], r1 = g.row_ptr[s + 1];
    if (r1 < r0) {
      if (lane == 0) atomicOr(bad, 1);
      continue;
    }
    const int shift = WFMT == 3 ? g.wshift + (g.row_shift ? g.row_shift[s] : 0) : g.wshift;
    if (WFMT == 3 && shift > 30 && r1 > r0) {  // a shifted int8 weight must stay an int32
      if (lane == 0) atomicOr(bad, 4);
      continue;
    }
    for (int64_t e = r0 + lane; e < r1; e += 32) {
      const uint32_t wd = g.word[e];
      const int64_t tgt = wd & 0x3FFFFFFFu;
      const int32_t c = (int32_t)(wd >> 30);
      if (tgt >= g.n || c >= g.nch) {
        atomicOr(bad, 2);
        continue;
      }
      int64_t w = acc_weight<WFMT>(g, e, shift);
      if (w > 2147483647LL || w < -2147483648LL) {
        atomicOr(bad, 4);
        continue;
      }
      if (w < 0) w = -w;
      atomicAdd(insum + (int64_t)c * g.npad + tgt, (unsigned long long)w);
    }
  }
}

// Warp per row: the delay of every synapse, delay[vox(source)][vox(target)].
// Work items per neuron, ceil(row length / kItemEvents), one byte each; a
// count above 255 sets *too_long.
__global__ void item_count_kernel(DevNet g, uint8_t* out, int32_t* too_long) {
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < g.npad; i += stride) {
    int64_t c = 0;
    if (i < g.n) c = (g.row_ptr[i + 1] - g.row_ptr[i] + kItemEvents - 1) / kItemEvents;
    if (c > 255) {
      atomicOr(too_long, 1);
      c = 255;
    }
    out[i] = (uint8_t)c;
  }
}

__global__ void delay_fill_kernel(DevNet g, uint8_t* out) {
  const int lane = threadIdx.x & 31;
  const int64_t gw = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const int64_t nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
  for (int64_t s = gw; s < g.n; s += nw) {
    const uint8_t* drow = g.delay + (int64_t)voxel_of(g, (int32_t)s) * g.nv;
    const int64_t r0 = g.row_ptr[s], r1 = g.row_ptr[s + 1];
    for (int64_t e = r0 + lane; e < r1; e += 32) out[e] = drow[voxel_of(g, (int32_t)(g.word[e] & 0x3FFFFFFFu))];
  }
}

// Bitonic sort of 32 * R keys held by one warp, element i = r * 32 + lane in
// register r of lane `lane`: distances below 32 exchange across lanes,
// larger ones inside a lane.  Ascending.
template <int R>
__device__ __forceinline__ void warp_bitonic_sort(unsigned long long (&v)[R], int lane) {
#pragma unroll
  for (int k = 2; k <= 32 * R; k <<= 1) {
#pragma unroll
    for (int j = k >> 1; j > 0; j >>= 1) {
      if (j >= 32) {
        const int jj = j >> 5;
#pragma unroll
        for (int r = 0; r < R; r++) {
          if ((r & jj) == 0) {
            const bool asc = ((r * 32) & k) == 0;  // k >= 64 > lane: bit k of i is bit k of r * 32
            const unsigned long long a = v[r], b = v[r | jj];
            const bool sw = asc ? (a > b) : (a < b);
            v[r] = sw ? b : a;
            v[r | jj] = sw ? a : b;
          }
        }
      } else {
        const bool lower = (lane & j) == 0;  // my element has the lower index of its pair
#pragma unroll
        for (int r = 0; r < R; r++) {
          const bool asc = (((r * 32) | lane) & k) == 0;
          const unsigned long long o = __shfl_xor_sync(0xFFFFFFFFu, v[r], j);
          const bool take_min = lower == asc;
          v[r] = take_min ? (o < v[r] ? o : v[r]) : (o > v[r] ? o : v[r]);
        }
      }
    }
  }
}

// Run key of a synapse: the arrival step's queue for delay d > 1, the target
// region's bin for delay 1 in bins mode (every delay-1 event shares one key in
// the event-queue mode).
__device__ __forceinline__ uint32_t synapse_run_key(uint32_t word, uint32_t d, bool bins) {
  if (d > 1) return d;
  return bins ? (kRunRegion | ((word & 0x3FFFFFFFu) >> kRegionShift)) : kRunRegion;
}

// Heads of a chunk's runs, one 32-element round of a warp after the other: an
// element starts a run when its key differs from its left neighbour's, or in
// the queue mode when the run of a longer delay reaches kMaxRun elements.
struct RunHeads {
  uint32_t last = 0xFFFFFFFFu;  // key of the element before this round
  int start = 0;                // where the run that reaches into this round began
  __device__ __forceinline__ unsigned round(uint32_t k, bool valid, int pos, int lane, bool split) {
    uint32_t left = __shfl_up_sync(0xFFFFFFFFu, k, 1);
    if (lane == 0) left = last;
    const unsigned diff = __ballot_sync(0xFFFFFFFFu, valid && k != left);
    const unsigned mine = diff & (0xFFFFFFFFu >> (31 - lane));
    const int from = mine ? pos - lane + 31 - __clz(mine) : start;  // first element of my stretch of one key
    const bool cut = split && valid && !(k & kRunRegion) && (pos - from) % kMaxRun == 0;
    const unsigned heads = diff | __ballot_sync(0xFFFFFFFFu, cut);
    last = __shfl_sync(0xFFFFFFFFu, k, 31);
    start = __shfl_sync(0xFFFFFFFFu, from, 31);
    return heads;
  }
};

// Warp per row: every synapse as a packed record, each chunk of kItemEvents
// synapses (one delivery work item) sorted by delay (from the voxel-pair
// table) and target, so that its events wait in few places (runs).
// counts[chunk_base[row] + k] receives the chunk's runs.  A record is (word,
// weight code | delay << 16) until run_fill replaces the second word; 32-bit
// weights leave no room for the delay, which run_fill then looks up again (a
// buffer of the delays was another byte per synapse on top of all the rest).
// A sort key is delay | target | class | weight code, or for 32-bit weights the
// place in the chunk, from which the weight is read again.
// The order of a row's synapses changes no result: the sums are exact integers.
template <int WFMT>
__global__ void __launch_bounds__(256) pack_fill_kernel(DevNet g, uint2* out, int32_t* counts) {
  constexpr int R = kItemEvents / 32;
  const int lane = threadIdx.x & 31;
  const bool bins = g.mode == kModeBins;
  const int64_t gw = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const int64_t nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
  if (gw == 0 && lane == 0) out[g.nnz] = make_uint2(0u, 0u);
  for (int64_t s = gw; s < g.n; s += nw) {
    const uint8_t* drow = g.delay + (int64_t)voxel_of(g, (int32_t)s) * g.nv;
    const int shift = WFMT == 3 ? g.wshift + (g.row_shift ? g.row_shift[s] : 0) : g.wshift;
    const int64_t r0 = g.row_ptr[s], r1 = g.row_ptr[s + 1];
    int64_t chunk = g.chunk_base[s];
    for (int64_t c0 = r0; c0 < r1; c0 += kItemEvents, chunk++) {
      unsigned long long v[R];
#pragma unroll
      for (int r = 0; r < R; r++) {
        const int64_t e = c0 + r * 32 + lane;
        v[r] = ~0ull;  // padding sorts last
        if (e < r1) {
          const uint32_t wd = g.word[e];
          const uint32_t d = drow[voxel_of(g, (int32_t)(wd & 0x3FFFFFFFu))];
          const uint32_t low = WFMT == 1 ? (uint32_t)(r * 32 + lane) : weight_code<WFMT>(g.w, e, shift);
          v[r] = ((unsigned long long)d << 48) | ((unsigned long long)(wd & 0x3FFFFFFFu) << 18) |
                 ((unsigned long long)(wd >> 30) << 16) | (unsigned long long)low;
        }
      }
      warp_bitonic_sort<R>(v, lane);
      int runs = 0;
      RunHeads rh;
#pragma unroll
      for (int r = 0; r < R; r++) {
        const int64_t e = c0 + r * 32 + lane;
        const bool valid = e < r1;
        const uint32_t word = (uint32_t)((v[r] >> 18) & 0x3FFFFFFFu) | ((uint32_t)((v[r] >> 16) & 3u) << 30);
        const uint32_t d = (uint32_t)(v[r] >> 48) & 0xFFu;
        const uint32_t k = valid ? synapse_run_key(word, d, bins) : 0xFFFFFFFFu;
        runs += __popc(rh.round(k, valid, r * 32 + lane, lane, !bins));
        if (valid) {
          const uint32_t low = (uint32_t)(v[r] & 0xFFFFu);
          out[e] = make_uint2(word, WFMT == 1 ? (uint32_t)decode_weight(weight_code<1>(g.w, c0 + low, 0), 1, g.wshift)
                                              : low | (d << 16));
        }
      }
      if (lane == 0) counts[chunk] = runs;
    }
  }
}

// Warp per row, after pack_fill and the run pointers: every chunk's run
// records (key | start << 14 | (length - 1) << 23) at runs[run_ptr[chunk]..];
// in bins mode each packed record's run index above its weight code, in the
// queue mode its accumulator value, and the chunk's info.
__global__ void __launch_bounds__(256) run_fill_kernel(DevNet g, uint2* pack, const int64_t* run_ptr, uint32_t* runs,
                                                       ChunkInfo* info) {
  const int lane = threadIdx.x & 31;
  const bool bins = g.mode == kModeBins, wide = g.wfmt == 1;
  const int64_t gw = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const int64_t nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
  for (int64_t s = gw; s < g.n; s += nw) {
    const uint8_t* drow = g.delay + (int64_t)voxel_of(g, (int32_t)s) * g.nv;
    const int64_t r0 = g.row_ptr[s], r1 = g.row_ptr[s + 1];
    int64_t chunk = g.chunk_base[s];
    for (int64_t c0 = r0; c0 < r1; c0 += kItemEvents, chunk++) {
      const int n = (int)min((int64_t)kItemEvents, r1 - c0);
      uint32_t* out = runs + run_ptr[chunk];
      RunHeads rh;
      int before = 0;  // runs that start before this round
      int n1 = 0;      // synapses of delay 1
      for (int p = 0; p < n; p += 32) {
        const int64_t e = c0 + p + lane;
        const bool valid = p + lane < n;
        const uint2 rec = valid ? pack[e] : make_uint2(0u, 0u);
        const uint32_t d = !wide ? (rec.y >> 16) & 0xFFu : valid ? drow[voxel_of(g, (int32_t)(rec.x & 0x3FFFFFFFu))] : 0u;
        const uint32_t k = valid ? synapse_run_key(rec.x, d, bins) : 0xFFFFFFFFu;
        const unsigned heads = rh.round(k, valid, p + lane, lane, !bins);
        const int idx = before + __popc(heads & (0xFFFFFFFFu >> (31 - lane))) - 1;
        if ((heads >> lane) & 1u) out[idx] = k | ((uint32_t)(p + lane) << 14);
        if (valid && !wide)
          pack[e].y = bins ? (rec.y & 0xFFFFu) | ((uint32_t)idx << 16)
                           : (uint32_t)decode_weight(rec.y & 0xFFFFu, g.wfmt, g.wshift);
        before += __popc(heads);
        n1 += __popc(__ballot_sync(0xFFFFFFFFu, valid && (k & kRunRegion)));
      }
      if (info && lane == 0) info[chunk] = chunk_info(c0, n, n1, run_ptr[chunk], before);
      __syncwarp();
      // lengths: up to the next run's start
      for (int r0_ = 0; r0_ < before; r0_ += 32) {
        const int r = r0_ + lane;
        uint32_t mine = 0;
        int next = n;
        if (r < before) {
          mine = out[r];
          if (r + 1 < before) next = run_start(out[r + 1]);
        }
        __syncwarp();
        if (r < before) out[r] = mine | ((uint32_t)(next - run_start(mine) - 1) << 23);
        __syncwarp();
      }
    }
  }
}

__global__ void max_kernel(const unsigned long long* a, int64_t m, unsigned long long* out) {
  unsigned long long best = 0;
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < m; i += (int64_t)gridDim.x * blockDim.x)
    best = a[i] > best ? a[i] : best;
  for (int o = 16; o > 0; o >>= 1) {
    const unsigned long long x = __shfl_xor_sync(0xFFFFFFFFu, best, o);
    best = x > best ? x : best;
  }
  if ((threadIdx.x & 31) == 0) atomicMax(out, best);
}

// One block row per (slot, channel) pair; int64 sums by two's-complement adds.
__global__ void ring_sums_kernel(DevNet g, unsigned long long* sums) {
  const int64_t pair = blockIdx.y;
  const int32_t* row = g.ring + pair * g.npad;
  long long acc = 0;
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < g.n; i += (int64_t)gridDim.x * blockDim.x)
    acc += row[i];
  for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xFFFFFFFFu, acc, o);
  if ((threadIdx.x & 31) == 0) atomicAdd(sums + pair, (unsigned long long)acc);
}

__global__ void ring_gather_kernel(DevNet g, const int64_t* idx, int64_t m, int32_t* out) {
  const int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  const int64_t per = (int64_t)g.D * g.nch;
  if (k >= m * per) return;
  const int64_t r = k / per, sc = k - r * per;  // sc = slot * nch + c
  out[k] = g.ring[sc * g.npad + idx[r]];
}

// ---- queue and bins modes: the dense ring view of the pending events ----
// Queue x holds what arrives at the step congruent to x: runs of synapses in the
// queue mode, events in bins mode.  In the queue mode slot t mod D (t = the next
// step to run) is the accumulator's and its queue is drained (x_acc; -1 in bins
// mode).
// Test hook of the counters: every queue (blockIdx.y < nq = D * n_sub) and, in
// bins mode, every bin (blockIdx.y = nq + parity * n_reg + region) gets its unused
// entries filled with placeholders of weight 0 (target 0, class 0, weight code
// 0; a queued run is the one record past the last synapse), then its count set
// to value (>= its capacity).
__global__ void preset_counters_kernel(DevNet g, unsigned long long value) {
  const int64_t y = blockIdx.y, nq = (int64_t)g.D * g.n_sub;
  const bool queue = y < nq;
  const int64_t cap = queue ? g.qcap : g.bcap;
  unsigned long long* cnt = queue ? g.qcnt + y * kQcntStride : g.bcnt + (y - nq) * kBcntStride;
  const int64_t used = (int64_t)min(*cnt, (unsigned long long)cap);
  for (int64_t i = used + (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < cap; i += (int64_t)gridDim.x * blockDim.x) {
    if (queue) g.q[y * g.qcap + i] = g.mode == kModeBins ? 0ull : run_desc(g.nnz, 1);
    else if (g.ev8) reinterpret_cast<uint2*>(g.bins)[(y - nq) * g.bcap + i] = make_uint2(0u, 0u);
    else g.bins[(y - nq) * g.bcap + i] = 0u;
  }
}

__global__ void set_counters_kernel(DevNet g, unsigned long long value) {
  const int64_t y = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  const int64_t nb = g.mode == kModeBins ? 2 * (int64_t)g.n_reg : 0;
  const int64_t nq = (int64_t)g.D * g.n_sub;
  if (y < nq) g.qcnt[y * kQcntStride] = value;
  else if (y < nq + nb) g.bcnt[(y - nq) * kBcntStride] = value;
}

// Every pending event of step x's queues: f(class, target, weight).  Queue mode:
// the step's queues are read side by side, by every kSubQueues-th block each, and
// eight lanes share a run, whose records are loaded all at once (one queue after
// the other and a run per thread, the dense view of 20,000 neurons took 190 us
// where one queue of events had taken 120).
template <typename F>
__device__ __forceinline__ void for_queued(const DevNet& g, int32_t x, F&& f) {
  const int64_t s = (int64_t)x * g.n_sub + blockIdx.x % (unsigned)g.n_sub;
  const int64_t cnt = (int64_t)min(g.qcnt[s * kQcntStride], (unsigned long long)g.qcap);
  const unsigned long long* q = g.q + s * g.qcap;
  const int64_t me = (int64_t)(blockIdx.x / (unsigned)g.n_sub) * blockDim.x + threadIdx.x;
  const int64_t all = (int64_t)(gridDim.x / (unsigned)g.n_sub) * blockDim.x;
  if (g.mode == kModeBins) {
    for (int64_t i = me; i < cnt; i += all) {
      const uint2 e = reinterpret_cast<const uint2*>(q)[i];
      f(e.x >> 30, e.x & 0x3FFFFFFFu, decode_weight(e.y, g.wfmt, g.wshift));
    }
    return;
  }
  constexpr int kPer = kMaxRun / 8;  // records of a run per lane
  const int gl = threadIdx.x & 7;
  unsigned long long next = me / 8 < cnt ? q[me / 8] : 0ull;
  for (int64_t i = me / 8; i < cnt; i += all / 8) {
    const unsigned long long d = next;
    if (i + all / 8 < cnt) next = q[i + all / 8];
    const uint2* rec = g.syn_pack + desc_first(d);
    uint2 e[kPer];
#pragma unroll
    for (int u = 0; u < kPer; u++)
      if (gl + 8 * u < desc_len(d)) e[u] = rec[gl + 8 * u];
#pragma unroll
    for (int u = 0; u < kPer; u++)
      if (gl + 8 * u < desc_len(d)) f(e[u].x >> 30, e[u].x & 0x3FFFFFFFu, (int32_t)e[u].y);
  }
}

__global__ void queue_to_dense_kernel(DevNet g, int32_t* dense, int32_t x_acc) {
  const int32_t x = blockIdx.y;
  if (x == x_acc) return;
  for_queued(g, x, [&](uint32_t c, uint32_t tgt, int32_t w) {
    atomicAdd(dense + ((int64_t)x * g.nch + c) * g.npad + tgt, w);
  });
}

__global__ void queue_sums_kernel(DevNet g, unsigned long long* sums, int32_t x_acc) {
  const int32_t x = blockIdx.y;
  if (x == x_acc) return;
  long long acc[4] = {0, 0, 0, 0};
  for_queued(g, x, [&](uint32_t c, uint32_t, int32_t w) { acc[c] += w; });
  for (int c = 0; c < 4; c++) {
    long long a = acc[c];
    for (int o = 16; o > 0; o >>= 1) a += __shfl_xor_sync(0xFFFFFFFFu, a, o);
    if ((threadIdx.x & 31) == 0 && a != 0 && c < g.nch) atomicAdd(sums + x * g.nch + c, (unsigned long long)a);
  }
}

// out [m][D][nch]: map [n] gives the row of a requested neuron (or -1).
__global__ void queue_gather_kernel(DevNet g, const int32_t* map, int32_t* out, int32_t x_acc) {
  const int32_t x = blockIdx.y;
  if (x == x_acc) return;
  for_queued(g, x, [&](uint32_t c, uint32_t tgt, int32_t w) {
    const int32_t r = map[tgt];
    if (r >= 0) atomicAdd(out + ((int64_t)r * g.D + x) * g.nch + c, w);
  });
}

// Bins mode: between calls the bins of parity x mod 2 hold the delay-1 events
// of the last delivery, due at step x (the next step to run, ring slot x mod D).
// The three views of the dense ring add them in: into a dense ring, into the
// per-slot sums, into the gathered entries of the neurons in map.
__device__ __forceinline__ void bin_event(const DevNet& g, const uint32_t* bin, int64_t e, uint32_t& loc,
                                          int32_t& w) {
  if (g.ev8) {
    const uint2 v = reinterpret_cast<const uint2*>(bin)[e];
    loc = v.x;
    w = decode_weight(v.y, g.wfmt, g.wshift);
  } else {
    const uint32_t v = bin[e];
    loc = v & 0xFFFFu;
    w = decode_weight(v >> 16, g.wfmt, g.wshift);
  }
}

__global__ void bins_view_kernel(DevNet g, int64_t x, int32_t* dense, unsigned long long* sums, const int32_t* map,
                                 int32_t* out) {
  const int r = blockIdx.y;
  const int par = (int)(x & 1);
  const int32_t slot = (int32_t)(x % g.D);
  const int ew = g.ev8 ? 2 : 1;
  const int64_t cnt = (int64_t)min(g.bcnt[((int64_t)par * g.n_reg + r) * kBcntStride], (unsigned long long)g.bcap);
  const uint32_t* bin = g.bins + ((int64_t)par * g.n_reg + r) * g.bcap * ew;
  long long acc[4] = {0, 0, 0, 0};
  for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < cnt; e += (int64_t)gridDim.x * blockDim.x) {
    uint32_t loc;
    int32_t w;
    bin_event(g, bin, e, loc, w);
    const uint32_t cls = (loc >> kRegionShift) & 3u;
    const int64_t tgt = (int64_t)r * kRegionNeurons + (loc & (kRegionNeurons - 1));
    if (dense) atomicAdd(dense + ((int64_t)slot * g.nch + cls) * g.npad + tgt, w);
    if (sums) acc[cls] += w;
    if (map) {
      const int32_t row = map[tgt];
      if (row >= 0) atomicAdd(out + ((int64_t)row * g.D + slot) * g.nch + cls, w);
    }
  }
  if (sums)
    for (int c = 0; c < 4; c++) {
      long long a = acc[c];
      for (int o = 16; o > 0; o >>= 1) a += __shfl_xor_sync(0xFFFFFFFFu, a, o);
      if ((threadIdx.x & 31) == 0 && a != 0 && c < g.nch) atomicAdd(sums + slot * g.nch + c, (unsigned long long)a);
    }
}

__global__ void acc_gather_kernel(DevNet g, const int64_t* idx, int64_t m, int32_t* out, int32_t x_acc) {
  const int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (k >= m * g.nch) return;
  const int64_t r = k / g.nch;
  const int32_t c = (int32_t)(k - r * g.nch);
  out[(r * g.D + x_acc) * g.nch + c] += g.ring[(int64_t)c * g.npad + idx[r]];
}

__global__ void add_kernel(int32_t* dst, const int32_t* src, int64_t n) {
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
    dst[i] += src[i];
}

__global__ void map_kernel(const int64_t* idx, int64_t m, int32_t* map) {
  const int64_t r = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (r < m) map[idx[r]] = (int32_t)r;
}

__global__ void philox_kernel(const uint4* ctr, const uint2* key, uint4* out, int64_t n) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) out[i] = philox4x32_10(ctr[i], key[i].x, key[i].y);
}

}  // namespace

cudaError_t launch_init_voltage(const DevNet& g, uint64_t init_seed, cudaStream_t st) {
  const int64_t threads = g.npad / 4;
  init_voltage_kernel<<<(unsigned)((threads + 255) / 256), 256, 0, st>>>(g, (uint32_t)init_seed,
                                                                          (uint32_t)(init_seed >> 32));
  return cudaGetLastError();
}

cudaError_t launch_check_synapses(const DevNet& g, unsigned long long* insum, int* bad,
                                  unsigned long long* max_insum, cudaStream_t st) {
  int dev = 0, sms = 1;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  const int blocks = sms * 8;
  switch (g.wfmt) {
    case 0: check_kernel<0><<<blocks, 256, 0, st>>>(g, insum, bad); break;
    case 1: check_kernel<1><<<blocks, 256, 0, st>>>(g, insum, bad); break;
    case 2: check_kernel<2><<<blocks, 256, 0, st>>>(g, insum, bad); break;
    default: check_kernel<3><<<blocks, 256, 0, st>>>(g, insum, bad); break;
  }
  max_kernel<<<blocks, 256, 0, st>>>(insum, (int64_t)g.nch * g.npad, max_insum);
  return cudaGetLastError();
}

cudaError_t launch_ring_sums(const DevNet& g, unsigned long long* sums, cudaStream_t st) {
  dim3 grid(64, (unsigned)(g.D * g.nch));
  ring_sums_kernel<<<grid, 256, 0, st>>>(g, sums);
  return cudaGetLastError();
}

cudaError_t launch_ring_gather(const DevNet& g, const int64_t* idx, int64_t m, int32_t* out, cudaStream_t st) {
  const int64_t total = m * g.D * g.nch;
  if (total <= 0) return cudaSuccess;
  ring_gather_kernel<<<(unsigned)((total + 255) / 256), 256, 0, st>>>(g, idx, m, out);
  return cudaGetLastError();
}

// Blocks of 256 threads over the queues, D rows of a multiple of n_sub.
static dim3 queue_grid(const DevNet& g) {
  const int64_t per = (g.qcap + 1023) / 1024;
  const int64_t x = g.mode == kModeBins ? 64 : (int64_t)g.n_sub * (per < 8 ? per : 8);
  return dim3((unsigned)x, (unsigned)g.D);
}

cudaError_t launch_queue_to_dense(const DevNet& g, int32_t* dense, int32_t x_acc, cudaStream_t st) {
  queue_to_dense_kernel<<<queue_grid(g), 256, 0, st>>>(g, dense, x_acc);
  return cudaGetLastError();
}

cudaError_t launch_bins_view(const DevNet& g, int64_t x, int32_t* dense, unsigned long long* sums,
                             const int32_t* map, int32_t* out, cudaStream_t st) {
  if (g.mode != kModeBins || g.n_reg < 1) return cudaSuccess;
  bins_view_kernel<<<dim3(8, (unsigned)g.n_reg), 256, 0, st>>>(g, x, dense, sums, map, out);
  return cudaGetLastError();
}

cudaError_t launch_add(int32_t* dst, const int32_t* src, int64_t n, cudaStream_t st) {
  add_kernel<<<1024, 256, 0, st>>>(dst, src, n);
  return cudaGetLastError();
}

cudaError_t launch_preset_counters(const DevNet& g, unsigned long long value, cudaStream_t st) {
  const int64_t rows = (int64_t)g.D * g.n_sub + (g.mode == kModeBins ? 2 * (int64_t)g.n_reg : 0);
  preset_counters_kernel<<<dim3(8, (unsigned)rows), 256, 0, st>>>(g, value);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  set_counters_kernel<<<(unsigned)((rows + 255) / 256), 256, 0, st>>>(g, value);  // after every fill has read its count
  return cudaGetLastError();
}

cudaError_t launch_queue_sums(const DevNet& g, unsigned long long* sums, int32_t x_acc, cudaStream_t st) {
  queue_sums_kernel<<<queue_grid(g), 256, 0, st>>>(g, sums, x_acc);
  return cudaGetLastError();
}

cudaError_t launch_queue_gather(const DevNet& g, const int64_t* idx, int64_t m, int32_t* map, int32_t* out,
                                int32_t x_acc, cudaStream_t st) {
  // map: int32 [n], all -1 on entry.  out starts as the spill ring's entries.
  {
    DevNet sp = g;
    sp.ring = g.spill;
    const int64_t total = m * g.D * g.nch;
    ring_gather_kernel<<<(unsigned)((total + 255) / 256), 256, 0, st>>>(sp, idx, m, out);
  }
  map_kernel<<<(unsigned)((m + 255) / 256), 256, 0, st>>>(idx, m, map);
  queue_gather_kernel<<<queue_grid(g), 256, 0, st>>>(g, map, out, x_acc);
  if (x_acc >= 0) acc_gather_kernel<<<(unsigned)((m * g.nch + 255) / 256), 256, 0, st>>>(g, idx, m, out, x_acc);
  return cudaGetLastError();
}

// The bounded wait of the neuron update's pipeline on an mbarrier: with
// arrive = 0 nothing ever arrives, so the wait gives up after max_cycles and
// the kernel reports it in *status (1); with arrive = 1 the barrier completes
// first and *status is 0.  No asynchronous copy is involved.
__global__ void bounded_wait_kernel(long long max_cycles, int32_t arrive, int32_t* status) {
  __shared__ uint64_t bar;
  mbar_init(&bar, 1);
  fence_mbar_init();
  if (arrive) asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(&bar)) : "memory");
  *status = mbar_wait_bounded(&bar, 0, max_cycles) ? 0 : 1;
}

cudaError_t launch_bounded_wait(long long max_cycles, int32_t arrive, int32_t* status, cudaStream_t st) {
  bounded_wait_kernel<<<1, 1, 0, st>>>(max_cycles, arrive, status);
  return cudaGetLastError();
}

cudaError_t launch_item_count(const DevNet& g, uint8_t* out, int32_t* too_long, cudaStream_t st) {
  int dev = 0, sms = 1;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  item_count_kernel<<<sms * 4, 256, 0, st>>>(g, out, too_long);
  return cudaGetLastError();
}

cudaError_t launch_delay_fill(const DevNet& g, uint8_t* out, cudaStream_t st) {
  int dev = 0, sms = 1;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  delay_fill_kernel<<<sms * 8, 256, 0, st>>>(g, out);
  return cudaGetLastError();
}

cudaError_t launch_pack_fill(const DevNet& g, uint2* out, int32_t* counts, cudaStream_t st) {
  int dev = 0, sms = 1;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  switch (g.wfmt) {
    case 0: pack_fill_kernel<0><<<sms * 8, 256, 0, st>>>(g, out, counts); break;
    case 1: pack_fill_kernel<1><<<sms * 8, 256, 0, st>>>(g, out, counts); break;
    case 2: pack_fill_kernel<2><<<sms * 8, 256, 0, st>>>(g, out, counts); break;
    default: pack_fill_kernel<3><<<sms * 8, 256, 0, st>>>(g, out, counts); break;
  }
  return cudaGetLastError();
}

cudaError_t launch_run_fill(const DevNet& g, uint2* pack, const int64_t* run_ptr, uint32_t* runs, ChunkInfo* info,
                            cudaStream_t st) {
  int dev = 0, sms = 1;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  run_fill_kernel<<<sms * 8, 256, 0, st>>>(g, pack, run_ptr, runs, info);
  return cudaGetLastError();
}

cudaError_t launch_philox(const uint32_t* ctr, const uint32_t* key, uint32_t* out, int64_t n, cudaStream_t st) {
  if (n <= 0) return cudaSuccess;
  philox_kernel<<<(unsigned)((n + 255) / 256), 256, 0, st>>>(reinterpret_cast<const uint4*>(ctr),
                                                              reinterpret_cast<const uint2*>(key),
                                                              reinterpret_cast<uint4*>(out), n);
  return cudaGetLastError();
}

}  // namespace dtb

// deliver.cu -- spike delivery: the outgoing synapse rows of the spiking
// neurons into the pending sums of their arrival steps (J sums of section
// V.B), in the ring layout (every synapse event is one int32 reduction into the
// dense ring) and the queue layout (runs of synapses wait in the queue of their
// arrival step, then they are reduced into the accumulator of that step).  The
// bins layout is in bins.cu.
#include <cuda_runtime.h>
#include <stdint.h>

#include <algorithm>
#include <mutex>

#include "device_launch.h"
#include "dtb_device.cuh"
#include "dtb_launch.h"

namespace dtb {
namespace {

template <int WFMT>
__device__ __forceinline__ int32_t stored_weight(const void* w, int64_t e, int shift) {
  if (WFMT == 0) return (int32_t)__ldg(reinterpret_cast<const int16_t*>(w) + e) * (1 << shift);
  if (WFMT == 1) return __ldg(reinterpret_cast<const int32_t*>(w) + e) * (1 << shift);
  if (WFMT == 2) {
    const uint32_t b = (uint32_t)__ldg(reinterpret_cast<const unsigned short*>(w) + e) << 16;
    return __float2int_rn(__fmul_rn(__uint_as_float(b), 65536.0f));
  }
  return (int32_t)__ldg(reinterpret_cast<const signed char*>(w) + e) * (1 << shift);
}

// Ring delivery: one warp per piece of a spiking row (up to 512 synapses;
// grid-stride over the list that the neuron update left, so nothing waits for
// the compaction), lanes stride over the piece, four synapses in flight per lane.
// The add is a fire-and-forget reduction at L2, so the order of adds does not
// matter.
template <int WFMT, int NCH>
__global__ void __launch_bounds__(256, 8) spike_deliver_kernel(DevNet g, int32_t t_rel) {
  const int64_t t = *g.t_base + t_rel;
  const int32_t tm = (int32_t)(t % g.D);
  const int n_list = (int)g.chunk_cnt[t % 3];
  const ulonglong2* list = g.row_list + (t & 1) * g.list_cap;
  const int lane = threadIdx.x & 31;
  const int64_t gw = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const int64_t nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
  const int64_t np = g.npad;
  unsigned long long ev = 0;
  __shared__ unsigned long long s_ev;  // one events atomic per block, not per warp
  if (threadIdx.x == 0) s_ev = 0;
  __syncthreads();
  for (int64_t ii = gw; ii < n_list; ii += nw) {
    const ulonglong2 piece = list[ii];
    const int32_t s = (int32_t)(uint32_t)piece.y;
    const int64_t r0 = (int64_t)piece.x, r1 = r0 + (int64_t)(piece.y >> 32);
    ev += (unsigned long long)(r1 - r0);
    const int shift = WFMT == 3 ? g.wshift + (g.row_shift ? g.row_shift[s] : 0) : g.wshift;
    for (int64_t e0 = r0 + lane; e0 < r1; e0 += 4 * 32) {
      uint32_t wd[4];
      int32_t wa[4];
      int32_t dd[4];
#pragma unroll
      for (int u = 0; u < 4; u++) {
        const int64_t e = e0 + u * 32;
        wd[u] = e < r1 ? __ldg(g.word + e) : 0xFFFFFFFFu;
        wa[u] = e < r1 ? stored_weight<WFMT>(g.w, e, shift) : 0;
        dd[u] = e < r1 ? (int32_t)__ldg(g.syn_delay + e) : 0;
      }
#pragma unroll
      for (int u = 0; u < 4; u++) {
        if (wd[u] == 0xFFFFFFFFu) continue;
        const int32_t tgt = (int32_t)(wd[u] & 0x3FFFFFFFu);
        const int32_t cls = (int32_t)(wd[u] >> 30);
        int32_t sl = tm + dd[u];
        if (sl >= g.D) sl -= g.D;
        atomicAdd(g.ring + ((int64_t)sl * NCH + cls) * np + tgt, wa[u]);
      }
    }
  }
  if (lane == 0 && ev) atomicAdd(&s_ev, ev);
  __syncthreads();
  if (threadIdx.x == 0 && s_ev) atomicAdd(g.events, s_ev);
}

// A run beyond its queue's capacity goes event by event into the dense spill
// slot sl of its arrival step (exact int32 adds).
__device__ __noinline__ void spill_run(const DevNet& g, int32_t sl, int32_t mark, int64_t e, int len) {
  for (int q = 0; q < len; q++) {
    const uint2 r = g.syn_pack[e + q];
    atomicAdd(g.spill + ((int64_t)sl * g.nch + (r.x >> 30)) * g.npad + (r.x & 0x3FFFFFFFu), (int32_t)r.y);
  }
  g.spill_dirty[sl] = mark;
}

// Queue delivery.  A row's synapses lie in chunks of kItemEvents, each sorted by
// delay and target at creation and cut into runs of one arrival step (run
// tables, dtb_device.cuh); the neuron update leaves the list of the chunks whose
// neurons fired.  The delivery touches the synapses of delay 1 only; of a longer
// run it queues one 8-byte record, the place and length of the run, and the
// synapses are read once, at their arrival step.  (Queueing every event cost an
// 8-byte read, an 8-byte write and another 8-byte read per synapse; a run of 5
// to 40 synapses is now one 8-byte record.)
// A CTA takes batches of 8 chunks, one per warp:
//   1. one run per lane; the longer runs are counted per arrival step in shared
//      memory (the count is the run's place in the batch);
//   2. one global atomic per arrival step of the batch reserves a range of the
//      CTA's queue of that step; meanwhile the delay-1 synapses are reduced into
//      the accumulator of step t + 1;
//   3. every run record goes to its queue.
// What bounds it is latency, with few CTAs resident beside the neuron update, so
// every load is issued ahead of its use: the delay-1 records before the count,
// the next batch's runs, the chunk info of the one after and the list entry of
// the third before the barrier.
constexpr int kPushThreads = 256, kPushWarps = kPushThreads / 32;

__global__ void __launch_bounds__(kPushThreads, 4) spike_push_kernel(DevNet g, int32_t t_rel) {
  __shared__ int hist[256];                 // runs of the batch per delay
  __shared__ unsigned long long base[256];  // their reserved start in the queue
  __shared__ unsigned long long s_ev;
  const int64_t t = *g.t_base + t_rel;
  const int32_t tm = (int32_t)(t % g.D);
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int n = (int)g.chunk_cnt[t % 3];
  const uint32_t* list = g.chunk_list + (t & 1) * g.list_cap;
  int32_t* acc1 = g.ring + ((t + 1) & 1) * (int64_t)g.nch * g.npad;  // arrivals of step t + 1
  const unsigned long long qcap = (unsigned long long)g.qcap;
  const int sub = (int)blockIdx.x % kSubQueues;
  unsigned long long ev = 0;
  hist[tid] = 0;
  if (tid == 0) s_ev = 0;
  const int step = (int)gridDim.x * kPushWarps;
  constexpr uint32_t kNone = 0xFFFFFFFFu;
  auto entry = [&](int i) -> uint32_t { return i < n ? list[i] : kNone; };
  auto info_of = [&](uint32_t c) -> ulonglong2 {  // none: no synapse, no run
    return c != kNone ? __ldg(reinterpret_cast<const ulonglong2*>(g.chunks) + c) : make_ulonglong2(0ull, 0ull);
  };
  auto runs_of = [&](ulonglong2 c, uint32_t (&x)[2]) {
    const uint32_t* rt = g.runs + (c.y & kLow44);
    const int nr = (int)(c.y >> 44);
#pragma unroll
    for (int h = 0; h < 2; h++) x[h] = lane + 32 * h < nr ? __ldg(rt + lane + 32 * h) : kRunNone;
  };
  int i = (int)blockIdx.x * kPushWarps + warp;
  ulonglong2 cur = info_of(entry(i)), nxt = info_of(entry(i + step));
  uint32_t c2 = entry(i + 2 * step);
  uint32_t x[2];
  runs_of(cur, x);
  __syncthreads();  // hist is clear
  for (int b = (int)blockIdx.x * kPushWarps; b < n; b += step, i += step) {
    const int64_t e0 = (int64_t)(cur.x & kLow44);
    const int n1 = (int)(cur.x >> 54), nr = (int)(cur.y >> 44);
    const uint2* rec = g.syn_pack + e0;
    uint2 r[8];
#pragma unroll
    for (int u = 0; u < 8; u++) r[u] = lane + 32 * u < n1 ? __ldcs(rec + lane + 32 * u) : make_uint2(0u, 0u);
    uint32_t off = 0;  // the two runs' places in the batch, 16 bits each
#pragma unroll
    for (int h = 0; h < 2; h++)
      if (!(run_key(x[h]) & kRunRegion)) off |= (uint32_t)atomicAdd(&hist[run_key(x[h])], 1) << (16 * h);
    uint32_t xn[2];
    runs_of(nxt, xn);
    const ulonglong2 nn = info_of(c2);
    c2 = entry(i + 3 * step);
    if (lane == 0) ev += (cur.x >> 44) & 1023u;
    __syncthreads();
    const int h = hist[tid];  // 256 threads, 256 delays
    unsigned long long got = 0;
    if (h) {
      int32_t sl = tm + tid;
      if (sl >= g.D) sl -= g.D;
      got = atomicAdd(g.qcnt + ((int64_t)sl * kSubQueues + sub) * kQcntStride, (unsigned long long)h);
      hist[tid] = 0;
    }
#pragma unroll
    for (int u = 0; u < 8; u++)
      if (lane + 32 * u < n1)
        atomicAdd(acc1 + (int64_t)(r[u].x >> 30) * g.npad + (r[u].x & 0x3FFFFFFFu), (int32_t)r[u].y);
    for (int j = lane + 256; j < n1; j += 32) {  // more than 256 of delay 1
      const uint2 v = __ldcs(rec + j);
      atomicAdd(acc1 + (int64_t)(v.x >> 30) * g.npad + (v.x & 0x3FFFFFFFu), (int32_t)v.y);
    }
    if (h) base[tid] = got;
    __syncthreads();
    auto queue_run = [&](uint32_t run, unsigned long long p, int64_t qi, int32_t sl) {
      if (p < qcap) g.q[qi * g.qcap + (int64_t)p] = run_desc(e0 + run_start(run), run_len(run));
      else spill_run(g, sl, spill_mark(t + run_key(run)), e0 + run_start(run), run_len(run));
    };
#pragma unroll
    for (int v = 0; v < 2; v++) {
      const uint32_t key = run_key(x[v]);
      if (key & kRunRegion) continue;
      int32_t sl = tm + (int32_t)key;
      if (sl >= g.D) sl -= g.D;
      queue_run(x[v], base[key] + ((off >> (16 * v)) & 0xFFFFu), (int64_t)sl * kSubQueues + sub, sl);
    }
    for (int k = lane + 64; k < nr; k += 32) {  // beyond 64 runs of a chunk: one by one (rare)
      const uint32_t run = __ldg(g.runs + (cur.y & kLow44) + k);
      int32_t sl = tm + (int32_t)run_key(run);
      if (sl >= g.D) sl -= g.D;
      const int64_t qi = (int64_t)sl * kSubQueues + sub;
      queue_run(run, atomicAdd(g.qcnt + qi * kQcntStride, 1ull), qi, sl);
    }
    cur = nxt;
    nxt = nn;
    x[0] = xn[0];
    x[1] = xn[1];
  }
  if (lane == 0 && ev) atomicAdd(&s_ev, ev);
  __syncthreads();
  if (tid == 0 && s_ev) atomicAdd(g.events, s_ev);
}

// Windows of 32 consecutive events over up to 32 runs of at least one event, one
// warp: lane l holds run l (start: events of the runs before it; recs: its
// first record minus start).  Returns the record of event p + lane (the caller
// masks the tail).
__device__ __forceinline__ int64_t window_record(int p, int lane, bool has, int start, int64_t recs) {
  const int d = start - p;
  const unsigned heads = __reduce_or_sync(0xFFFFFFFFu, has && d >= 0 && d < 32 ? 1u << d : 0u);
  const int before = __popc(__ballot_sync(0xFFFFFFFFu, has && d < 0));
  const int owner = before + __popc(heads & (0xFFFFFFFFu >> (31 - lane))) - 1;
  return __shfl_sync(0xFFFFFFFFu, recs, owner) + p + lane;
}

// Queue mode: the runs queued for arrival step t + 1 into that step's
// accumulator.  A warp takes groups of at most kDrainRuns runs of at most
// kMaxRun synapses (so no warp is held long by a few long runs: without the
// bounds the slowest warps took half of the kernel's time) and walks their
// synapses in windows of 32: one 8-byte load and one int32 reduction per
// synapse, four windows in flight.  The neuron update that consumes the
// accumulator empties the queue.
constexpr int kDrainRuns = 4;

__global__ void __launch_bounds__(256, 6) drain_kernel(DevNet g, int32_t t_rel) {
  const int64_t t = *g.t_base + t_rel;
  const int32_t x = (int32_t)((t + 1) % g.D);
  const int64_t np = g.npad;
  int32_t* acc = g.ring + ((t + 1) & 1) * g.nch * np;  // the accumulator of step t + 1
  const int lane = threadIdx.x & 31;
  // every kSubQueues-th warp serves one of the step's queues
  const int all = (int)((gridDim.x * blockDim.x) >> 5), me = (int)((blockIdx.x * blockDim.x + threadIdx.x) >> 5);
  const int64_t qi = (int64_t)x * kSubQueues + me % kSubQueues;
  const int64_t cnt = (int64_t)min(g.qcnt[qi * kQcntStride], (unsigned long long)g.qcap);
  const unsigned long long* q = g.q + qi * g.qcap;
  const int64_t nw = all / kSubQueues, gw = me / kSubQueues;
  const int per = (int)min((int64_t)kDrainRuns, max((int64_t)1, cnt / nw));
  for (int64_t i0 = gw * per; i0 < cnt; i0 += nw * per) {
    const bool has = lane < per && i0 + lane < cnt;
    const unsigned long long d = has ? __ldcs(q + i0 + lane) : 0ull;
    const int len = has ? desc_len(d) : 0;
    int end = len;
#pragma unroll
    for (int o = 1; o < kDrainRuns; o <<= 1) {
      const int y = __shfl_up_sync(0xFFFFFFFFu, end, o);
      if (lane >= o) end += y;
    }
    const int total = __shfl_sync(0xFFFFFFFFu, end, kDrainRuns - 1);
    const int64_t recs = desc_first(d) - (end - len);
    for (int p0 = 0; p0 < total; p0 += 128) {
      uint2 r[4];
#pragma unroll
      for (int u = 0; u < 4; u++) {
        const int p = p0 + 32 * u;
        r[u] = make_uint2(0u, 0u);
        if (p < total) {
          const int64_t e = window_record(p, lane, has, end - len, recs);
          if (p + lane < total) r[u] = __ldcs(g.syn_pack + e);
        }
      }
#pragma unroll
      for (int u = 0; u < 4; u++)
        if (p0 + 32 * u + lane < total)
          atomicAdd(acc + (int64_t)(r[u].x >> 30) * np + (r[u].x & 0x3FFFFFFFu), (int32_t)r[u].y);
    }
  }
}

// CTAs of a kernel without dynamic shared memory that fit the device at once.
template <typename K>
cudaError_t resident_ctas(K kernel, int threads, DeviceLaunch (&cache)[kMaxDevices], std::mutex& mu, DeviceLaunch* dl) {
  return device_launch(cache, mu, [&](DeviceLaunch& d) {
    int per = 0;
    const cudaError_t r = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, kernel, threads, 0);
    d.per_sm = per > 0 ? per : 1;
    return r;
  }, dl);
}

template <int NCH>
cudaError_t launch_ring(const DevNet& g, int32_t t_rel, int blocks, cudaStream_t st) {
  switch (g.wfmt) {
    case 0: spike_deliver_kernel<0, NCH><<<blocks, 256, 0, st>>>(g, t_rel); break;
    case 1: spike_deliver_kernel<1, NCH><<<blocks, 256, 0, st>>>(g, t_rel); break;
    case 2: spike_deliver_kernel<2, NCH><<<blocks, 256, 0, st>>>(g, t_rel); break;
    default: spike_deliver_kernel<3, NCH><<<blocks, 256, 0, st>>>(g, t_rel); break;
  }
  return cudaGetLastError();
}

}  // namespace

cudaError_t launch_spike_deliver(const DevNet& g, int32_t t_rel, int blocks, cudaStream_t st) {
  if (g.mode == kModeBins) return launch_bins_deliver(g, t_rel, blocks, st);
  if (g.mode == kModeQueue) {
    static DeviceLaunch cache[kMaxDevices];
    static std::mutex mu;
    DeviceLaunch dl;
    const cudaError_t e = resident_ctas(spike_push_kernel, kPushThreads, cache, mu, &dl);
    if (e != cudaSuccess) return e;
    spike_push_kernel<<<std::min(blocks, dl.sms * dl.per_sm), kPushThreads, 0, st>>>(g, t_rel);
    return cudaGetLastError();
  }
  return g.nch == 2 ? launch_ring<2>(g, t_rel, blocks, st) : launch_ring<4>(g, t_rel, blocks, st);
}

cudaError_t launch_drain(const DevNet& g, int32_t t_rel, int blocks, cudaStream_t st) {
  if (g.mode != kModeQueue) return cudaSuccess;
  static DeviceLaunch cache[kMaxDevices];
  static std::mutex mu;
  DeviceLaunch dl;
  const cudaError_t e = resident_ctas(drain_kernel, 256, cache, mu, &dl);
  if (e != cudaSuccess) return e;
  drain_kernel<<<std::min(blocks, dl.sms * dl.per_sm), 256, 0, st>>>(g, t_rel);
  return cudaGetLastError();
}

cudaError_t prepare_deliver_kernels() {
  return share_sm_division(spike_push_kernel, drain_kernel, spike_deliver_kernel<0, 2>, spike_deliver_kernel<1, 2>,
                           spike_deliver_kernel<2, 2>, spike_deliver_kernel<3, 2>, spike_deliver_kernel<0, 4>,
                           spike_deliver_kernel<1, 4>, spike_deliver_kernel<2, 4>, spike_deliver_kernel<3, 4>);
}

int deliver_blocks_per_sm() {
  int n = 0;
  cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, spike_deliver_kernel<0, 2>, 256, 0);
  return n > 0 ? n : 1;
}

}  // namespace dtb

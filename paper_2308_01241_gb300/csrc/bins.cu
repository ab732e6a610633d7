// bins.cu -- bins delivery: events of delay 1 straight into the bins of their
// target regions, longer ones through the event queue of their arrival step,
// which is sorted into the bins one step before that step.
#include <cuda_runtime.h>
#include <stdint.h>

#include <mutex>

#include "device_launch.h"
#include "dtb_device.cuh"
#include "dtb_launch.h"

namespace dtb {
namespace {

// Bins delivery of 32-bit weights.  A CTA takes batches of kQBatch work items
// (one warp per item).  Each lane loads its up to 16 synapses of the item in
// one round (lane l holds synapses l, l + 32, ...), so one memory latency
// covers the item.  Every event then has a key: the arrival step's queue
// (delay d > 1), or for delay-1 events the target region's bin of step t + 1
// (their targets lie in the source's voxel: a window of kWin regions around
// the source region, per warp).
//   pass 1: the 32 synapses a warp holds in one round form runs of equal keys
//           (consecutive lanes); the run's first lane adds the run's length to
//           the key's batch count in shared memory and learns the run's offset
//           among the batch's events of that key;
//   then:   one global atomic per key of the batch reserves the key's range of
//           its queue or bin, and a block scan places the keys' events one
//           after the other in a shared-memory staging buffer;
//   pass 2: every event goes to its staging slot; then consecutive threads
//           write the staged events out, so that each key's run goes to its
//           queue or bin in coalesced stores.
// Events at or beyond a queue's or bin's capacity are added into the dense
// spill ring instead.  Delay-1 events outside a warp's window reserve one by
// one.  Three barriers per batch.
constexpr int kQBatch = 8;
constexpr int kWin = 64;

// Exclusive scan of a[0 .. n) into out by the 256 threads of a CTA, each a
// contiguous chunk of at most 4 (n <= 1024); returns the total.  a is read
// before the scan's barrier only, so callers may change it afterwards.
__device__ __forceinline__ int deliver_block_scan(const int* a, int* out, int n, int* s_warp) {
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int per = (n + 255) / 256;
  const int r0 = tid * per;
  int v[4];
  int sum = 0;
#pragma unroll
  for (int q = 0; q < 4; q++) {
    v[q] = q < per && r0 + q < n ? a[r0 + q] : 0;
    sum += v[q];
  }
  int x = sum;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int y = __shfl_up_sync(0xFFFFFFFFu, x, o);
    if (lane >= o) x += y;
  }
  if (lane == 31) s_warp[warp] = x;
  __syncthreads();
  int before = 0, total = 0;
#pragma unroll
  for (int w = 0; w < 8; w++) {
    const int t = s_warp[w];
    before += w < warp ? t : 0;
    total += t;
  }
  int run = before + x - sum;
#pragma unroll
  for (int q = 0; q < 4; q++)
    if (q < per && r0 + q < n) {
      out[r0 + q] = run;
      run += v[q];
    }
  return total;
}

template <int NCH>
__global__ void __launch_bounds__(256, 3) spike_deliver_bins32_kernel(DevNet g, int32_t t_rel) {
  constexpr int kPer = kItemEvents / 32;  // synapses of an item per lane
  constexpr int kDelayKeys = 256;         // keys 0 .. 255: the queue of arrival step t + key
  constexpr int kKeys = kDelayKeys + kQBatch * kWin;  // then warp w's window region r: 256 + w * kWin + r
  constexpr int kStage = kQBatch * kItemEvents;
  extern __shared__ __align__(16) unsigned char dsm[];
  uint2* stage = reinterpret_cast<uint2*>(dsm);                           // [kStage] staged events
  unsigned short* skey = reinterpret_cast<unsigned short*>(stage + kStage);  // [kStage] their keys
  int* hist = reinterpret_cast<int*>(skey + kStage);                      // [kKeys] events per key in the batch
  int* sbase = hist + kKeys;                                              // [kKeys] staging offset of each key
  unsigned int* gbase = reinterpret_cast<unsigned int*>(sbase + kKeys);   // [kKeys] reserved start (clamped to capacity)
  __shared__ int s_warp[8];
  __shared__ int s_wlo[2][kQBatch];  // bins mode: first region of each warp's window, by batch parity
  __shared__ unsigned long long s_ev;  // one events atomic per block, not per warp
  const int64_t t = *g.t_base + t_rel;
  const int32_t tm = (int32_t)(t % g.D);
  const int32_t n_items = *g.n_items;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int64_t np = g.npad;
  const long long qcap = g.qcap;
  unsigned long long ev = 0;
  if (threadIdx.x == 0) s_ev = 0;
  for (int k = threadIdx.x; k < kKeys; k += blockDim.x) hist[k] = 0;
  const int par1 = (int)((t + 1) & 1);  // bins mode: parity of step t + 1
  unsigned long long* bc1 = g.bcnt + (int64_t)par1 * g.n_reg * kBcntStride;
  uint2* bins1 = reinterpret_cast<uint2*>(g.bins) + (int64_t)par1 * g.n_reg * g.bcap;
  const uint64_t once = l2_evict_first();  // a row is read once per spike
  __syncthreads();
  const int nbatch = (n_items + kQBatch - 1) / kQBatch;
  int bp = 0;  // batch parity
  for (int b = blockIdx.x; b < nbatch; b += gridDim.x, bp ^= 1) {
    const int ii = b * kQBatch + warp;
    const bool has = ii < n_items;
    // the whole item in registers: lane holds synapses lane + 32 u
    uint32_t wd[kPer];
    uint8_t dl[kPer];             // delay (0: no synapse); weights are re-read where they are needed
    uint32_t off2[kPer / 2];      // two 16-bit offsets per word: an event's place among its key's batch events
#pragma unroll
    for (int u = 0; u < kPer; u++) {
      wd[u] = 0u;
      dl[u] = 0;
    }
    int len = 0, wlo = 0;
    if (has) {
      const WorkItem item = g.items[ii];
      len = item.len;
      wlo = max((item.src >> kRegionShift) - kWin / 2, 0);
      if (lane == 0) ev += (unsigned long long)len;
      const uint32_t* wrow = g.word + item.e0;
      const uint8_t* drow = g.syn_delay + item.e0;
#pragma unroll
      for (int u = 0; u < kPer; u++) {
        const int j = lane + 32 * u;
        const bool in = j < len;
        wd[u] = in ? ldg_hint(wrow + j, once) : 0u;
        dl[u] = in ? __ldg(drow + j) : (uint8_t)0;
      }
    }
    if (lane == 0) s_wlo[bp][warp] = wlo;
    // pass 1: runs of equal keys -> one shared atomic per run
#pragma unroll
    for (int u = 0; u < kPer; u++) {
      const uint32_t d = dl[u];
      const int32_t tgt = (int32_t)(wd[u] & 0x3FFFFFFFu);
      int key = -1;
      if (d > 1) {
        key = (int)d;
      } else if (d == 1) {
        const int w = (tgt >> kRegionShift) - wlo;
        if (w >= 0 && w < kWin) {
          key = kDelayKeys + warp * kWin + w;
        } else {  // outside the window: reserve alone (rare)
          const int r = tgt >> kRegionShift;
          const int64_t pos = (int64_t)min(atomicAdd(bc1 + (int64_t)r * kBcntStride, 1ull), (unsigned long long)g.bcap);
          const uint32_t loc = (uint32_t)(tgt & (kRegionNeurons - 1)) | ((wd[u] >> 30) << kRegionShift);
          const uint32_t code = weight_code<1>(g.w, g.items[ii].e0 + lane + 32 * u, 0);
          if (pos < g.bcap) {
            bins1[(int64_t)r * g.bcap + pos] = make_uint2(loc, code);
          } else {
            int32_t sl = tm + 1;
            if (sl >= g.D) sl -= g.D;
            atomicAdd(g.spill + ((int64_t)sl * NCH + (wd[u] >> 30)) * np + tgt, decode_weight(code, 1, g.wshift));
            g.spill_dirty[sl] = spill_mark(t + 1);
          }
        }
      }
      const int left = __shfl_up_sync(0xFFFFFFFFu, key, 1);
      const bool head = key >= 0 && (lane == 0 || left != key);
      const unsigned heads = __ballot_sync(0xFFFFFFFFu, head);
      const unsigned ends = heads | __ballot_sync(0xFFFFFFFFu, key < 0);
      int run_off = 0;
      if (head) {
        const unsigned above = lane == 31 ? 0u : (ends >> (lane + 1)) << (lane + 1);
        const int nb = above ? __ffs(above) - 1 : 32;
        run_off = atomicAdd(&hist[key], nb - lane);
      }
      const int my_head = 31 - __clz(heads & (0xFFFFFFFFu >> (31 - lane)));
      const int o = __shfl_sync(0xFFFFFFFFu, run_off, my_head & 31) + (lane - my_head);
      const uint32_t o16 = key >= 0 ? (uint32_t)o : 0u;
      if (u & 1) off2[u >> 1] |= o16 << 16;
      else off2[u >> 1] = o16;
    }
    __syncthreads();
    // reservations of the batch's keys and their places in the staging buffer
    const int total = deliver_block_scan(hist, sbase, kKeys, s_warp);
    for (int k = threadIdx.x; k < kKeys; k += blockDim.x) {
      const int h = hist[k];
      if (h > 0) {
        if (k < kDelayKeys) {
          int32_t sl = tm + k;
          if (sl >= g.D) sl -= g.D;
          const unsigned long long p = atomicAdd(g.qcnt + sl * kQcntStride, (unsigned long long)h);
          if (p + (unsigned long long)h > (unsigned long long)qcap) g.spill_dirty[sl] = spill_mark(t + k);  // the tail spills
          gbase[k] = (unsigned int)min(p, (unsigned long long)qcap);
        } else {
          const int w = k - kDelayKeys;
          const int r = s_wlo[bp][w / kWin] + w % kWin;
          gbase[k] = (unsigned int)min(atomicAdd(bc1 + (int64_t)r * kBcntStride, (unsigned long long)h),
                                       (unsigned long long)g.bcap);
        }
        hist[k] = 0;  // for the next batch (every warp is past its pass 1)
      }
    }
    __syncthreads();
    // pass 2a: every keyed event into its staging slot
    if (has) {
#pragma unroll
      for (int u = 0; u < kPer; u++) {
        const uint32_t d = dl[u];
        if (d == 0) continue;
        const int32_t tgt = (int32_t)(wd[u] & 0x3FFFFFFFu);
        int key;
        if (d > 1) {
          key = (int)d;
        } else {
          const int w = (tgt >> kRegionShift) - wlo;
          if (w < 0 || w >= kWin) continue;
          key = kDelayKeys + warp * kWin + w;
        }
        const int at = sbase[key] + (int)((off2[u >> 1] >> (16 * (u & 1))) & 0xFFFFu);
        const uint32_t v = weight_code<1>(g.w, g.items[ii].e0 + lane + 32 * u, 0);
        stage[at] = make_uint2(d == 1 ? (uint32_t)(tgt & (kRegionNeurons - 1)) | ((wd[u] >> 30) << kRegionShift) : wd[u], v);
        skey[at] = (unsigned short)key;
      }
    }
    __syncthreads();
    // pass 2b: consecutive threads write each key's run out
    for (int i = threadIdx.x; i < total; i += blockDim.x) {
      const int key = skey[i];
      const uint2 e = stage[i];
      const int64_t pos = (int64_t)gbase[key] + (i - sbase[key]);
      if (key < kDelayKeys) {
        int32_t sl = tm + key;
        if (sl >= g.D) sl -= g.D;
        if (pos < qcap) {
          reinterpret_cast<uint2*>(g.q)[(int64_t)sl * qcap + pos] = e;
        } else {
          atomicAdd(g.spill + ((int64_t)sl * NCH + (e.x >> 30)) * np + (e.x & 0x3FFFFFFFu),
                    decode_weight(e.y, 1, g.wshift));
        }
      } else {
        const int w = key - kDelayKeys;
        const int r = s_wlo[bp][w / kWin] + w % kWin;
        if (pos < g.bcap) {
          bins1[(int64_t)r * g.bcap + pos] = e;
        } else {
          int32_t sl = tm + 1;
          if (sl >= g.D) sl -= g.D;
          const int64_t tg = (int64_t)r * kRegionNeurons + (e.x & (kRegionNeurons - 1));
          atomicAdd(g.spill + ((int64_t)sl * NCH + ((e.x >> kRegionShift) & 3u)) * np + tg,
                    decode_weight(e.y, 1, g.wshift));
          g.spill_dirty[sl] = spill_mark(t + 1);
        }
      }
    }
  }
  if (lane == 0 && ev) atomicAdd(&s_ev, ev);
  __syncthreads();
  if (threadIdx.x == 0 && s_ev) atomicAdd(g.events, s_ev);
}

// Bins delivery over the run tables (16-bit weight codes: packed records whose
// chunks are sorted by delay and target).  A CTA takes batches of kQBatch work
// items, one warp per item (one chunk), in a two-stage pipeline: while the
// events of batch b go out, batch b + 1 is counted and reserved.
//   pass 1: the warp's lanes take the chunk's runs (a few dozen); each run
//           adds its length to its key's batch count in shared memory, which
//           returns the run's offset among the batch's events of that key
//           (keys: the queue of arrival step t + d, or the bin of a target
//           region of step t + 1 inside the warp's window of kWin regions; a
//           delay-1 run outside the window reserves its own range and is
//           written right away).  The first run of a key puts the key on the
//           batch's list of active keys;
//   reservation: one thread per active key reserves the key's range with one
//           global atomic;
//   pass 2: every event's record names its run; its position is the key's
//           reserved start + the run's offset + its place in the run.
//           Consecutive events of a run go to consecutive positions.
// Iteration b: load batch b's records; pass 1 of batch b + 1; load the first
// run entries of batch b + 2; barrier; issue the reservations of batch b + 1;
// pass 2 of batch b; store the reserved positions of batch b + 1; barrier.
// So a batch's record and run loads and its reservation round trip overlap
// the other batch's work instead of adding up.  Every per-key and per-run
// array is double-buffered by batch parity; the work items (two ahead) rotate
// through three shared slots.
struct RunsSmem {
  static constexpr int kKeys = 256 + kQBatch * kWin;
  static constexpr size_t kHist = 0;                                           // int [2][kKeys]
  static constexpr size_t kPtr = kHist + 2 * kKeys * 4;                        // u64 [2][kKeys]
  static constexpr size_t kRoom = kPtr + 2 * kKeys * 8;                        // u32 [2][kKeys]
  static constexpr size_t kRinfo = kRoom + 2 * kKeys * 4;                      // u32 [2][kQBatch][kItemEvents]
  static constexpr size_t kActive = kRinfo + 2 * kQBatch * kItemEvents * 4;    // u16 [2][kKeys]
  static constexpr size_t kBytes = kActive + 2 * kKeys * 2;
};

// Rare paths of the run-table delivery, kept out of line so that the unrolled
// per-event code stays small.  An event beyond its queue's or bin's capacity
// goes into the dense spill slot sl of its arrival step (exact int32 add).
template <int WFMT, int NCH>
__device__ __noinline__ void spill_event(const DevNet& g, int32_t sl, uint32_t word, uint32_t code, int32_t mark) {
  atomicAdd(g.spill + ((int64_t)sl * NCH + (word >> 30)) * g.npad + (word & 0x3FFFFFFFu), decode_weight(code, WFMT, g.wshift));
  g.spill_dirty[sl] = mark;
}

// A delay-1 run whose target region lies outside the warp's window: its own
// range of the region's bin of step t + 1, written right away.
template <int WFMT, int NCH>
__device__ __forceinline__ void direct_run(const DevNet& g, const uint2* prow, int start, int len, int region,
                                        unsigned long long* bc1, uint32_t* bins1, int32_t s1, int32_t mark) {
  const int64_t p0 = (int64_t)atomicAdd(bc1 + (int64_t)region * kBcntStride, (unsigned long long)len);
  for (int q = 0; q < len; q++) {
    const uint2 e = prow[start + q];
    const uint32_t tgt = e.x & 0x3FFFFFFFu, code = e.y & 0xFFFFu;
    const uint32_t loc = (tgt & (kRegionNeurons - 1)) | ((e.x >> 30) << kRegionShift);
    if (p0 + q < g.bcap) bins1[(int64_t)region * g.bcap + p0 + q] = loc | (code << 16);
    else spill_event<WFMT, NCH>(g, s1, e.x, code, mark);
  }
}

template <int WFMT, int NCH>
__global__ void __launch_bounds__(256, 3) spike_deliver_runs_kernel(DevNet g, int32_t t_rel) {
  using L = RunsSmem;
  constexpr int kPer = kItemEvents / 32;
  constexpr int kDelayKeys = 256;
  constexpr int kKeys = L::kKeys;
  constexpr uint32_t kDirect = 1023u;  // a delay-1 run written in pass 1
  extern __shared__ __align__(16) unsigned char dsm[];
  int* hist = reinterpret_cast<int*>(dsm + L::kHist);
  unsigned long long* kptr = reinterpret_cast<unsigned long long*>(dsm + L::kPtr);  // key's reserved start (address)
  unsigned int* kroom = reinterpret_cast<unsigned int*>(dsm + L::kRoom);  // positions left in its queue or bin
  uint32_t* rinfo = reinterpret_cast<uint32_t*>(dsm + L::kRinfo);  // per run: key | (offset - start + 512) << 10
  unsigned short* active = reinterpret_cast<unsigned short*>(dsm + L::kActive);
  __shared__ int n_active[2];
  __shared__ int s_wlo[2][kQBatch];
  __shared__ __align__(16) WorkItem s_item[3][kQBatch];
  __shared__ unsigned long long s_ev;
  const int64_t t = *g.t_base + t_rel;
  const int32_t tm = (int32_t)(t % g.D);
  const int32_t n_items = *g.n_items;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const long long qcap = g.qcap;
  unsigned long long ev = 0;
  if (tid == 0) {
    s_ev = 0;
    n_active[0] = n_active[1] = 0;
  }
  for (int k = tid; k < 2 * kKeys; k += 256) hist[k] = 0;
  const int par1 = (int)((t + 1) & 1);  // bins mode: parity of step t + 1
  unsigned long long* bc1 = g.bcnt + (int64_t)par1 * g.n_reg * kBcntStride;
  uint32_t* bins1 = g.bins + (int64_t)par1 * g.n_reg * g.bcap;  // 4-byte events (16-bit codes)
  const uint64_t once = l2_evict_first();  // a row is read once per spike
  const int nbatch = (n_items + kQBatch - 1) / kQBatch;
  const int G = (int)gridDim.x;

  // the warp's work item of batch b, one 4-byte word per lane (len 0: none)
  auto item_word = [&](int b) -> int32_t {
    const int i = b * kQBatch + warp;
    return (lane < 8 && b < nbatch && i < n_items) ? reinterpret_cast<const int32_t*>(g.items + i)[lane] : 0;
  };
  auto put_item = [&](int slot, int32_t w) {
    if (lane < 8) reinterpret_cast<int32_t*>(&s_item[slot][warp])[lane] = w;
    __syncwarp();
  };

  // pass 1 of a batch of parity p whose item sits in slot sl
  constexpr int kRunsAhead = 2;  // run entries per lane loaded one iteration ahead of pass 1
  auto pass1 = [&](int sl, int p, const uint32_t (&rr)[kRunsAhead]) {
    const WorkItem& it = s_item[sl][warp];
    const int len = it.len;
    int wlo = 0;
    if (len > 0) {
      wlo = max((it.src >> kRegionShift) - kWin / 2, 0);
      const uint2* prow = g.syn_pack + it.e0;
      const int64_t rp0 = it.rp0;
      const int nr = it.nr;
      int* hp = hist + p * kKeys;
      uint32_t* ri = rinfo + (p * kQBatch + warp) * kItemEvents;
      unsigned short* act = active + p * kKeys;
      auto take_run = [&](int r, uint32_t run) {
        const uint32_t key = run_key(run);
        const int start = run_start(run), Ln = run_len(run);
        uint32_t ki;
        if (key & kRunRegion) {
          const int region = (int)(key & (kRunRegion - 1u));
          const int w = region - wlo;
          if (w >= 0 && w < kWin) {
            ki = (uint32_t)(kDelayKeys + warp * kWin + w);
          } else {  // outside the window: its own range, written now (rare)
            ki = kDirect;
            direct_run<WFMT, NCH>(g, prow, start, Ln, region, bc1, bins1, tm + 1 >= g.D ? tm + 1 - g.D : tm + 1,
                                    spill_mark(t + 1));
          }
        } else {
          ki = key;  // the queue of arrival step t + key
        }
        int off = 0;
        if (ki < (uint32_t)kKeys) {
          off = atomicAdd(&hp[ki], Ln);
          if (off == 0) act[atomicAdd(&n_active[p], 1)] = (unsigned short)ki;  // the key's first run
        }
        ri[r] = ki | ((uint32_t)(off - start + 512) << 10);
      };
#pragma unroll
      for (int q = 0; q < kRunsAhead; q++)
        if (lane + 32 * q < nr) take_run(lane + 32 * q, rr[q]);
      for (int r = lane + 32 * kRunsAhead; r < nr; r += 32) take_run(r, __ldg(g.runs + rp0 + r));
    }
    if (lane == 0) s_wlo[p][warp] = wlo;
  };

  // the counter a key of a batch of parity p reserves on
  auto key_counter = [&](int k, int p) -> unsigned long long* {
    if (k < kDelayKeys) {
      int32_t sl = tm + k;
      if (sl >= g.D) sl -= g.D;
      return g.qcnt + sl * kQcntStride;
    }
    const int w = k - kDelayKeys;
    return bc1 + (int64_t)(s_wlo[p][w / kWin] + w % kWin) * kBcntStride;
  };
  // the reserved start of a key (h events from position got on) for pass 2
  auto store_key = [&](int k, int p, unsigned long long got, int h) {
    if (k < kDelayKeys) {
      int32_t sl = tm + k;
      if (sl >= g.D) sl -= g.D;
      if (got + (unsigned long long)h > (unsigned long long)qcap) g.spill_dirty[sl] = spill_mark(t + k);  // the tail spills
      const unsigned long long p0 = min(got, (unsigned long long)qcap);
      kptr[p * kKeys + k] = reinterpret_cast<unsigned long long>(reinterpret_cast<uint2*>(g.q) + (int64_t)sl * qcap + (int64_t)p0);
      kroom[p * kKeys + k] = (unsigned int)((unsigned long long)qcap - p0);
    } else {
      const int w = k - kDelayKeys;
      const int r = s_wlo[p][w / kWin] + w % kWin;
      const unsigned long long p0 = min(got, (unsigned long long)g.bcap);
      kptr[p * kKeys + k] = reinterpret_cast<unsigned long long>(bins1 + (int64_t)r * g.bcap + (int64_t)p0);
      kroom[p * kKeys + k] = (unsigned int)((unsigned long long)g.bcap - p0);
    }
  };

  // pass 2 of a batch of parity p: every event to its place
  auto pass2 = [&](int len, const uint2 (&rec)[kPer], int p) {
    const uint32_t* ri = rinfo + (p * kQBatch + warp) * kItemEvents;
    const unsigned long long* kp = kptr + p * kKeys;
    const unsigned int* kr = kroom + p * kKeys;
#pragma unroll
    for (int u = 0; u < kPer; u++) {
      const int pos = lane + 32 * u;
      if (pos >= len) continue;
      const uint2 e = rec[u];
      const uint32_t info = ri[(e.y >> 16) & 511u];
      const uint32_t ki = info & 1023u;
      const uint32_t o = (info >> 10) + (uint32_t)pos - 512u;  // >= 0: a run's offset + the place in it
      if (ki >= (uint32_t)kKeys) continue;  // kDirect: written in pass 1
      if (o < kr[ki]) {
        if (ki < (uint32_t)kDelayKeys) {
          reinterpret_cast<uint2*>(kp[ki])[o] = make_uint2(e.x, e.y & 0xFFFFu);
        } else {  // bins event: local target | class << 12 | code << 16
          reinterpret_cast<uint32_t*>(kp[ki])[o] =
              (e.x & (kRegionNeurons - 1)) | ((e.x >> (30 - kRegionShift)) & (3u << kRegionShift)) | (e.y << 16);
        }
      } else {  // beyond the capacity: the spill ring of the arrival step (rare)
        const int32_t d = ki < (uint32_t)kDelayKeys ? (int32_t)ki : 1;
        int32_t sl = tm + d;
        if (sl >= g.D) sl -= g.D;
        spill_event<WFMT, NCH>(g, sl, e.x, e.y & 0xFFFFu, spill_mark(t + d));
      }
    }
  };

  // The first iteration has no current batch (slot 0 stays empty): it only
  // counts and reserves the CTA's first batch.
  put_item(0, 0);
  put_item(1, item_word((int)blockIdx.x));
  // the first runs of the next pass-1 batch, loaded an iteration ahead (its item
  // is the one two batches ahead, loaded at the start of the iteration before)
  uint32_t rn[kRunsAhead];
  auto load_runs = [&](int64_t rp0, int nr) {
#pragma unroll
    for (int q = 0; q < kRunsAhead; q++) rn[q] = lane + 32 * q < nr ? __ldg(g.runs + rp0 + lane + 32 * q) : 0u;
  };
  load_runs(s_item[1][warp].rp0, s_item[1][warp].len > 0 ? s_item[1][warp].nr : 0);
  __syncthreads();  // hist and n_active are clear
  int b = (int)blockIdx.x - G, bp = 1, sc = 0;  // batch, its parity, the slot of its item
  for (; b < nbatch; b += G, bp ^= 1, sc = sc == 2 ? 0 : sc + 1) {
    const int bn = b + G, p1 = bp ^ 1;
    const int sn = sc == 2 ? 0 : sc + 1, snn = sn == 2 ? 0 : sn + 1;
    // batch b's records, and the item two batches ahead
    const int len = s_item[sc][warp].len;
    uint2 rec[kPer];
    {
      const uint2* prow = g.syn_pack + s_item[sc][warp].e0;
#pragma unroll
      for (int u = 0; u < kPer; u++) {
        const int j = lane + 32 * u;
        rec[u] = j < len ? ldg_hint(prow + j, once) : make_uint2(0u, 0u);
      }
    }
    const int32_t wnn = item_word(bn + G);
    if (bn < nbatch) pass1(sn, p1, rn);
    {  // the runs of batch bn + G from its item's words (rp0: words 2-3, len: 4, nr: 6)
      const uint32_t lo = (uint32_t)__shfl_sync(0xFFFFFFFFu, wnn, 2), hi = (uint32_t)__shfl_sync(0xFFFFFFFFu, wnn, 3);
      const int lenn = __shfl_sync(0xFFFFFFFFu, wnn, 4), nrn = __shfl_sync(0xFFFFFFFFu, wnn, 6);
      load_runs((int64_t)(((uint64_t)hi << 32) | lo), lenn > 0 ? nrn : 0);
    }
    __syncthreads();
    // reservations of batch b + 1: a thread's first key stays in flight until
    // after pass 2 of batch b; further keys (more than 256) are stored now
    int rk = -1, rh = 0;
    unsigned long long rg = 0;
    if (bn < nbatch) {
      const int na = n_active[p1];
      if (tid < na) {
        rk = active[p1 * kKeys + tid];
        rh = hist[p1 * kKeys + rk];
        hist[p1 * kKeys + rk] = 0;
        rg = atomicAdd(key_counter(rk, p1), (unsigned long long)rh);
      }
      for (int a = tid + 256; a < na; a += 256) {
        const int k = active[p1 * kKeys + a];
        const int h = hist[p1 * kKeys + k];
        hist[p1 * kKeys + k] = 0;
        store_key(k, p1, atomicAdd(key_counter(k, p1), (unsigned long long)h), h);
      }
    }
    if (tid == 0) n_active[bp] = 0;  // batch b's list is done; pass 1 of batch b + 2 fills it
    if (len > 0) {
      if (lane == 0) ev += (unsigned long long)len;
      pass2(len, rec, bp);
    }
    if (rk >= 0) store_key(rk, p1, rg, rh);
    put_item(snn, wnn);
    __syncthreads();
  }
  if (lane == 0 && ev) atomicAdd(&s_ev, ev);
  __syncthreads();
  if (threadIdx.x == 0 && s_ev) atomicAdd(g.events, s_ev);
}

// Dynamic shared memory of the ballot delivery.
constexpr int kDeliverSmem = kQBatch * kItemEvents * (8 + 2) + (256 + kQBatch * kWin) * 12;

// Bins mode: sorts the queue of arrival step x = t + t_rel by target region
// into the bins of parity x mod 2, which the neuron update of step x then
// sums in shared memory.  A CTA takes tiles of kBinThreads * kPer events:
//   1. every event gets its rank among the tile's events of its region from a
//      shared-memory histogram;
//   2. one global atomic per region of the tile reserves a contiguous range of
//      that region's bin, and a block scan of the histogram gives each
//      region's offset in the tile;
//   3. the events are placed in shared memory in region order, then written
//      out by consecutive threads, so that a region's run of the tile goes to
//      its bin in coalesced stores (scattered stores of single events from
//      many warps into the same sectors were the kernel's bottleneck).
// A bin that is full sends the rest of its events into the dense spill slot
// of step x (exact int32 adds), as a full queue does.
constexpr int kBinThreads = 1024;

// Exclusive scan of a[0 .. n) into out (in place allowed, n <= 16 * kBinThreads),
// each thread a contiguous chunk; returns the total to every thread.
__device__ __forceinline__ uint32_t bin_block_scan(const uint32_t* a, uint32_t* out, int n, uint32_t* s_warp) {
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int per = (n + kBinThreads - 1) / kBinThreads;
  const int r0 = tid * per, r1 = min(r0 + per, n);
  uint32_t sum = 0;
  for (int r = r0; r < r1; r++) sum += a[r];
  uint32_t x = sum;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const uint32_t y = __shfl_up_sync(0xFFFFFFFFu, x, o);
    if (lane >= o) x += y;
  }
  if (lane == 31) s_warp[warp] = x;
  __syncthreads();
  if (warp == 0) {
    uint32_t w = lane < kBinThreads / 32 ? s_warp[lane] : 0u;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const uint32_t y = __shfl_up_sync(0xFFFFFFFFu, w, o);
      if (lane >= o) w += y;
    }
    s_warp[lane] = w;  // inclusive warp totals
  }
  __syncthreads();
  uint32_t run = (warp ? s_warp[warp - 1] : 0u) + x - sum;
  for (int r = r0; r < r1; r++) {
    const uint32_t v = a[r];
    out[r] = run;
    run += v;
  }
  return s_warp[kBinThreads / 32 - 1];
}

template <bool EV8>
__global__ void __launch_bounds__(kBinThreads, 1) bin_kernel(DevNet g, int32_t t_rel) {
  // events per thread and tile; a 16-bit code leaves room for the rank in
  // the upper half of the event's second word
  constexpr int kPer = EV8 ? 8 : 20;
  constexpr int kTile = kBinThreads * kPer;
  extern __shared__ __align__(16) uint32_t bsm[];
  const int nreg = g.n_reg;
  uint32_t* hist = bsm;                  // [n_reg] events of the tile per region
  uint32_t* base = bsm + nreg;           // [n_reg] start of the tile's range in each bin
  uint32_t* loff = bsm + 2 * nreg;       // [n_reg] start of each region's run in the sorted tile
  uint32_t* sev = bsm + ((3 * nreg + 3) & ~3);  // [kTile] the tile's events in region order (EV8: [kTile][2]), 16-byte aligned
  unsigned short* sreg = reinterpret_cast<unsigned short*>(sev + kTile * (EV8 ? 2 : 1));  // [kTile] their regions
  __shared__ uint32_t s_warp[32];
  const int64_t x = *g.t_base + t_rel;
  const int32_t slot = (int32_t)(x % g.D);
  const int par = (int)(x & 1);
  const int64_t cnt = (int64_t)min(g.qcnt[slot * kQcntStride], (unsigned long long)g.qcap);
  const uint2* q = reinterpret_cast<const uint2*>(g.q) + (int64_t)slot * g.qcap;
  unsigned long long* bc = g.bcnt + (int64_t)par * nreg * kBcntStride;
  uint32_t* bins = g.bins + (int64_t)par * nreg * g.bcap * (EV8 ? 2 : 1);
  const int64_t bcap = g.bcap;
  const int tid = threadIdx.x;
  for (int r = tid; r < nreg; r += kBinThreads) hist[r] = 0u;
  __syncthreads();
  for (int64_t b0 = (int64_t)blockIdx.x * kTile; b0 < cnt; b0 += (int64_t)gridDim.x * kTile) {
    const int n_tile = (int)min((int64_t)kTile, cnt - b0);
    uint2 e[kPer];
    uint32_t rk[EV8 ? kPer : 1];
#pragma unroll
    for (int u = 0; u < kPer; u++) {
      const int64_t i = b0 + u * kBinThreads + tid;
      e[u] = i < cnt ? __ldcs(q + i) : make_uint2(0xFFFFFFFFu, 0u);  // all-ones id: no event
    }
#pragma unroll
    for (int u = 0; u < kPer; u++) {
      if (e[u].x == 0xFFFFFFFFu) continue;
      const uint32_t k = atomicAdd(&hist[(e[u].x & 0x3FFFFFFFu) >> kRegionShift], 1u);
      if (EV8) rk[u] = k;
      else e[u].y = (e[u].y & 0xFFFFu) | (k << 16);  // k < kTile < 2^16
    }
    __syncthreads();
    // reservations, and each region's offset in the tile; the histogram is
    // cleared for the next tile
    {  // all of this thread's reservations in flight at once (kMaxRegions / kBinThreads per thread at most)
      constexpr int kRegPer = kMaxRegions / kBinThreads;
      unsigned long long got[kRegPer];
#pragma unroll
      for (int q = 0; q < kRegPer; q++) {
        const int r = tid + q * kBinThreads;
        const uint32_t h = r < nreg ? hist[r] : 0u;
        got[q] = h ? atomicAdd(bc + (int64_t)r * kBcntStride, (unsigned long long)h) : 0ull;
      }
#pragma unroll
      for (int q = 0; q < kRegPer; q++) {
        const int r = tid + q * kBinThreads;
        if (r < nreg) base[r] = (uint32_t)min(got[q], (unsigned long long)bcap);
      }
    }
    (void)bin_block_scan(hist, loff, nreg, s_warp);
    __syncthreads();
    for (int r = tid; r < nreg; r += kBinThreads) hist[r] = 0u;
#pragma unroll
    for (int u = 0; u < kPer; u++) {
      if (e[u].x == 0xFFFFFFFFu) continue;
      const uint32_t tgt = e[u].x & 0x3FFFFFFFu, cls = e[u].x >> 30;
      const uint32_t r = tgt >> kRegionShift;
      const uint32_t loc = (tgt & (kRegionNeurons - 1)) | (cls << kRegionShift);
      const uint32_t at = loff[r] + (EV8 ? rk[u] : (e[u].y >> 16));
      if (EV8) reinterpret_cast<uint2*>(sev)[at] = make_uint2(loc, e[u].y);
      else sev[at] = loc | (e[u].y << 16);
      sreg[at] = (unsigned short)r;
    }
    __syncthreads();
    for (int i = tid; i < n_tile; i += kBinThreads) {
      const uint32_t r = sreg[i];
      const int64_t pos = (int64_t)base[r] + (i - (int)loff[r]);
      if (pos < bcap) {
        if (EV8) reinterpret_cast<uint2*>(bins)[(int64_t)r * bcap + pos] = reinterpret_cast<const uint2*>(sev)[i];
        else bins[(int64_t)r * bcap + pos] = sev[i];
      } else {
        const uint32_t loc = EV8 ? reinterpret_cast<const uint2*>(sev)[i].x : (sev[i] & 0xFFFFu);
        const uint32_t code = EV8 ? reinterpret_cast<const uint2*>(sev)[i].y : (sev[i] >> 16);
        const uint32_t cls = (loc >> kRegionShift) & 3u;
        const int64_t tgt = (int64_t)r * kRegionNeurons + (loc & (kRegionNeurons - 1));
        atomicAdd(g.spill + ((int64_t)slot * g.nch + cls) * g.npad + tgt, decode_weight(code, g.wfmt, g.wshift));
        g.spill_dirty[slot] = spill_mark(x);
      }
    }
    __syncthreads();  // base, loff and the sorted tile are rewritten by the next tile
  }
}

// Dynamic shared memory set once per device; the grid is at most the CTAs that
// fit at once (the kernels stride over batches).
template <typename K>
cudaError_t launch_batches(K kernel, int smem, DeviceLaunch (&cache)[kMaxDevices], std::mutex& mu, const DevNet& g,
                           int32_t t_rel, int blocks, cudaStream_t st) {
  DeviceLaunch dl;
  cudaError_t e = device_launch(cache, mu, [&](DeviceLaunch& d) {
    cudaError_t r = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
    if (r != cudaSuccess) return r;
    int per = 0;
    r = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, kernel, 256, smem);
    d.per_sm = per > 0 ? per : 1;
    return r;
  }, &dl);
  if (e != cudaSuccess) return e;
  const int most = dl.sms * dl.per_sm;
  kernel<<<blocks < most ? blocks : most, 256, smem, st>>>(g, t_rel);
  return cudaGetLastError();
}

template <int C>
cudaError_t launch_deliver_32(const DevNet& g, int32_t t_rel, int blocks, cudaStream_t st) {
  static DeviceLaunch cache[kMaxDevices];
  static std::mutex mu;
  return launch_batches(spike_deliver_bins32_kernel<C>, kDeliverSmem, cache, mu, g, t_rel, blocks, st);
}

template <int W, int C>
cudaError_t launch_deliver_runs(const DevNet& g, int32_t t_rel, int blocks, cudaStream_t st) {
  static DeviceLaunch cache[kMaxDevices];
  static std::mutex mu;
  return launch_batches(spike_deliver_runs_kernel<W, C>, (int)RunsSmem::kBytes, cache, mu, g, t_rel, blocks, st);
}

}  // namespace

cudaError_t launch_bins_deliver(const DevNet& g, int32_t t_rel, int blocks, cudaStream_t st) {
  if (g.wfmt == 1) {
    return g.nch == 2 ? launch_deliver_32<2>(g, t_rel, blocks, st) : launch_deliver_32<4>(g, t_rel, blocks, st);
  }
  if (g.nch == 2) {
    switch (g.wfmt) {
      case 0: return launch_deliver_runs<0, 2>(g, t_rel, blocks, st);
      case 2: return launch_deliver_runs<2, 2>(g, t_rel, blocks, st);
      default: return launch_deliver_runs<3, 2>(g, t_rel, blocks, st);
    }
  }
  switch (g.wfmt) {
    case 0: return launch_deliver_runs<0, 4>(g, t_rel, blocks, st);
    case 2: return launch_deliver_runs<2, 4>(g, t_rel, blocks, st);
    default: return launch_deliver_runs<3, 4>(g, t_rel, blocks, st);
  }
}

cudaError_t launch_bin(const DevNet& g, int32_t t_rel, cudaStream_t st) {
  if (g.mode != kModeBins) return cudaSuccess;
  static DeviceLaunch cache[kMaxDevices];
  static std::mutex mu;
  // histogram, reservations and offsets per region; the sorted tile (16K
  // one-word or 8K two-word events) and its regions (2 bytes each)
  const int tile_bytes = 20 * kBinThreads * 4 + 20 * kBinThreads * 2;
  const int smem = 4 * ((3 * g.n_reg + 3) & ~3) + tile_bytes;
  DeviceLaunch dl;
  cudaError_t e0 = device_launch(cache, mu, [&](DeviceLaunch& d) {
    const int most = 12 * kMaxRegions + tile_bytes;
    cudaError_t e = cudaFuncSetAttribute(bin_kernel<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, most);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(bin_kernel<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, most);
    d.per_sm = 1;
    return e;
  }, &dl);
  if (e0 != cudaSuccess) return e0;
  const int blocks = dl.sms;  // one CTA of kBinThreads per SM
  if (g.ev8) bin_kernel<true><<<blocks, kBinThreads, smem, st>>>(g, t_rel);
  else bin_kernel<false><<<blocks, kBinThreads, smem, st>>>(g, t_rel);
  return cudaGetLastError();
}

}  // namespace dtb

// Device side of the what-if placement simulator, shared by the kernel
// translation units (gmgsim_full.cu, gmgsim_inc.cu, gmgsim_kernels.cu).
//
// One warp simulates one candidate placement (Algorithm 1 evaluates the
// candidate partitions "in parallel"; here every warp of a persistent grid
// takes candidates k = warp, warp + W, ...).  Inside a warp the simulation
// is the event-driven loop of Sec. 3.3.3 restated as one ordered sweep:
//
//   READY(r_i, i)  op i's last input has arrived (Sec. 3.3.2 ready time).
//                  Taking READY keys in (r, id) order and starting each op
//                  at s_i = max(r_i, accelerator free time) makes every queue
//                  run its ops in (ready time, id) order, one at a time
//                  (Sec. 3.3.2, Sec. 3.5.1) -- exactly "an idle queue starts
//                  the ready op with the earliest ready time".
//   FREE / ALLOC   HBM events of the copies of an op's output: the op's own
//                  buffer at s_i, a receive buffer on every other accelerator
//                  of a successor at f_i (Recv before Send, Sec. 3.5.2), each
//                  released by its last listed consumer there (Sec. 3.3.2).
//
// READY ops are taken many at a time (Sim::run): every pending op has a lower
// bound of its finish, and all pending ops with a ready time below the smallest
// of these bounds are started together, one per lane -- nothing that they make
// ready can precede any of them.  What bounds the kernels is the chain of
// dependent instructions and loads per batch, and the issue slots that all warps
// share; DRAM is idle.  On the prefill graph (3,088 ops, 8 accelerators) it is
// 2.5 to 3 ops a batch and 172 warp instructions an op, against 333 for one key
// at a time.  With at most 32 accelerators the lanes hold the pending ops, one
// each (prefill, 4,096 placements, 4.74 ms -> 3.09; as keys in shared memory
// instead: 4.5); with more, where more ops than lanes are pending, they are 64-bit
// keys in a pool in shared memory (256 accelerators, 4,096 placements, 128 ms ->
// 81).  What does not fit goes to a warp-cooperative 32-ary min-heap.  Ops
// without predecessors come in when they are due: their keys are pre-sorted on
// the host.
//
// HBM events are appended to a per-warp log in O(1).  Every event produced
// while handling READY(r, .) happens at a time >= r, so once the next READY
// key has time T, every logged event with time < T is final and no later
// event can precede it.  Such events are drained in batches.  Their order
// matters only on an accelerator whose peak they can raise: there they are sorted
// by (time, frees before allocs, op) and applied in order, which gives the peaks
// and the first capacity violation (Sec. 3.4.2 OOM discard) exactly; elsewhere
// their sum is added (apply_due).
//
// Lanes also fan out over successor lists (readiness, transfer arrivals,
// distinct receiving accelerators via __match_any_sync) and predecessor
// lists (ready-time maxima, last-consumer releases).
//
// No wait in these kernels depends on another block.  The two warps of a pair
// (kRole) meet at named barriers of their block, and each message of one has its
// counterpart in the other, whatever the candidate's status.  The only loop whose
// trip count is not bounded by the data is the event loop, capped at g.max_iter
// iterations (status GMG_SIM_LOOP).

#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include <type_traits>

#include "gmg_layout.h"

namespace gsim {
namespace {

constexpr unsigned kFullMask = 0xffffffffu;
constexpr uint64_t kKeyMax = ~0ull;
constexpr int64_t kI64Max = 0x7fffffffffffffffll;

__device__ __forceinline__ uint64_t warp_min_u64(uint64_t v) {
  const uint32_t hi = (uint32_t)(v >> 32), lo = (uint32_t)v;
  const uint32_t mh = __reduce_min_sync(kFullMask, hi);
  const uint32_t ml = __reduce_min_sync(kFullMask, hi == mh ? lo : 0xffffffffu);
  return ((uint64_t)mh << 32) | ml;
}

__device__ __forceinline__ uint64_t warp_max_u64(uint64_t v) {
  const uint32_t hi = (uint32_t)(v >> 32), lo = (uint32_t)v;
  const uint32_t mh = __reduce_max_sync(kFullMask, hi);
  const uint32_t ml = __reduce_max_sync(kFullMask, hi == mh ? lo : 0u);
  return ((uint64_t)mh << 32) | ml;
}

__device__ __forceinline__ unsigned lane_id() { return threadIdx.x & 31u; }
__device__ __forceinline__ uint32_t lanes_below() { return (1u << lane_id()) - 1u; }

// Bulk prefetch of [p, p + bytes) into L2 (no completion to wait for), 32 KB
// pieces spread over the warp.  p is 16-byte aligned; a ragged tail below 16
// bytes is left out.  Single-warp kernels that walk the graph serially start
// with it, so that their dependent loads hit L2 instead of DRAM.
__device__ __forceinline__ void warp_prefetch_l2(const void* p, int64_t bytes) {
  const uint64_t a = (uint64_t)__cvta_generic_to_global(p);
  constexpr int64_t kPiece = 1 << 15;
  for (int64_t o = (int64_t)lane_id() * kPiece; o < bytes; o += 32 * kPiece) {
    const int64_t left = bytes - o;
    const uint32_t sz = (uint32_t)((left < kPiece ? left : kPiece) & ~int64_t(15));
    if (sz) asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" :: "l"(a + o), "r"(sz) : "memory");
  }
}

// The next candidate of a launch that hands them out one at a time (uniform).
__device__ __forceinline__ int64_t take_candidate(uint32_t* next_k) {
  uint32_t k = 0;
  if (lane_id() == 0) k = atomicAdd(next_k, 1u);
  return (int64_t)__shfl_sync(kFullMask, k, 0);
}

// Warp copy of `bytes` rounded up to a multiple of 16 between 16-byte
// aligned buffers (both must extend to the rounded size), kDepth 16-byte
// loads in flight per lane (a single-warp kernel takes a deeper pipeline:
// nothing else hides its load latency).
template <int kDepth = 4>
__device__ __forceinline__ void warp_copy16(void* dst, const void* src, int64_t bytes) {
  const int64_t nv = (bytes + 15) >> 4;
  uint4* d = static_cast<uint4*>(dst);
  const uint4* s = static_cast<const uint4*>(src);
  int64_t i = lane_id();
  for (; i + 32 * (kDepth - 1) < nv; i += 32 * kDepth) {
    uint4 v[kDepth];
#pragma unroll
    for (int u = 0; u < kDepth; ++u) v[u] = s[i + 32 * u];
#pragma unroll
    for (int u = 0; u < kDepth; ++u) d[i + 32 * u] = v[u];
  }
  for (; i < nv; i += 32) d[i] = s[i];
}

// 16-byte pieces of an OpRec, loaded through the read-only path.
__device__ __forceinline__ longlong2 op_durbytes(const OpRec* ops, uint32_t i) {
  return __ldg(reinterpret_cast<const longlong2*>(ops + i));
}
struct RelPred {
  int64_t rel;
  uint32_t pred_off, npred;
};
struct XqSucc {
  int64_t xq;
  uint32_t succ_off, nsucc;
};
__device__ __forceinline__ RelPred op_relpred(const OpRec* ops, uint32_t i) {
  const uint4 v = __ldg(reinterpret_cast<const uint4*>(ops + i) + 1);
  return RelPred{(int64_t)(((uint64_t)v.y << 32) | v.x), v.z, v.w};
}
__device__ __forceinline__ XqSucc op_xqsucc(const OpRec* ops, uint32_t i) {
  const uint4 v = __ldg(reinterpret_cast<const uint4*>(ops + i) + 2);
  return XqSucc{(int64_t)(((uint64_t)v.y << 32) | v.x), v.z, v.w};
}
// (succ_off, nsucc, pred_off, npred) from two pieces, for code that needs both lists.
__device__ __forceinline__ uint4 op_lists(const OpRec* ops, uint32_t i) {
  const XqSucc a = op_xqsucc(ops, i);
  const RelPred b = op_relpred(ops, i);
  return make_uint4(a.succ_off, a.nsucc, b.pred_off, b.npred);
}
__device__ __forceinline__ uint4 op_cons(const OpRec* ops, uint32_t i) {
  return __ldg(reinterpret_cast<const uint4*>(ops + i) + 3);  // cons_off, ncons, req, flags
}

// The codecs' parameters stay in the launch parameters (constant bank).
struct KeyCodec {
  const DevGmg& g;
  template <typename TM>
  __device__ __forceinline__ uint64_t make(TM t, uint32_t cls, uint32_t op) const {
    using U = typename std::make_unsigned<TM>::type;
    return ((uint64_t)(U)t << (g.ib + 2)) | ((uint64_t)cls << g.ib) | (uint64_t)op;
  }
  __device__ __forceinline__ int64_t time(uint64_t k) const { return (int64_t)(k >> (g.ib + 2)); }
  __device__ __forceinline__ uint64_t time_floor(int64_t t) const { return (uint64_t)t << (g.ib + 2); }
  __device__ __forceinline__ uint32_t cls(uint64_t k) const { return (uint32_t)(k >> g.ib) & 3u; }
  __device__ __forceinline__ uint32_t op(uint64_t k) const { return (uint32_t)k & g.opmask; }
};

// READY keys of the pool: time, op id, then qb bits that hold how far the op's
// finish is from its ready time at least (floating point, rounded down: qb - 5
// bits of mantissa below a 5-bit exponent; qb = 0 where the key has no room,
// then the distance is taken as 1).  These bits are the lowest, so they never
// change the order of two keys.
struct ReadyCodec {
  const DevGmg& g;
  __device__ __forceinline__ uint32_t enc(uint32_t x) const {  // x >= 1
    const int m = g.qb - 5;
    const int e = max(0, 32 - m - __clz(x));
    return ((uint32_t)e << m) | (x >> e);
  }
  template <typename TM>
  __device__ __forceinline__ uint64_t make(TM t, uint32_t op, TM least) const {
    using U = typename std::make_unsigned<TM>::type;
    const uint32_t x = sizeof(TM) > 4 && least > (TM)0x7fffffff ? 0x7fffffffu : (uint32_t)least;
    return ((uint64_t)(U)t << g.qsh) | ((uint64_t)op << g.qb) | (g.qb ? enc(x) : 0u);
  }
  __device__ __forceinline__ int64_t time(uint64_t k) const { return (int64_t)(k >> g.qsh); }
  __device__ __forceinline__ uint32_t op(uint64_t k) const { return (uint32_t)(k >> g.qb) & g.opmask; }
  // The earliest finish of the key's op.
  __device__ __forceinline__ int64_t bound(uint64_t k) const {
    if (g.qb == 0) return time(k) + 1;
    const int m = g.qb - 5;
    const uint32_t q = (uint32_t)k & ((1u << g.qb) - 1u);
    return time(k) + (int64_t)((q & ((1u << m) - 1u)) << (q >> m));
  }
};

__device__ __forceinline__ int64_t warp_sum_i64(int64_t v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(kFullMask, v, o);
  return v;
}

// ---------------------------------------------------------------------------
// READY keys: warp-cooperative 32-ary min-heap.  Slots [0, qs) are in shared
// memory (qs >= 33, so the root and its children always are), the rest in
// the warp's global scratch.  All lanes call every method with the same
// arguments; lane 0 performs the stores.
// ---------------------------------------------------------------------------
struct ReadyHeap {
  const SimParams& P;
  uint64_t* sk;
  uint8_t* sl;  // the warp's scratch slot
  int size;

  __device__ __forceinline__ uint64_t* kp(int i) const {
    return i < P.qs ? sk + i : reinterpret_cast<uint64_t*>(sl + P.off_qk) + (i - P.qs);
  }
  __device__ __forceinline__ uint64_t top() const { return size > 0 ? sk[0] : kKeyMax; }

  __device__ void sift_down(int pos, uint64_t x) {
    const unsigned lane = lane_id();
    while (true) {
      const int c0 = pos * 32 + 1;
      if (c0 >= size) break;
      const int idx = c0 + (int)lane;
      uint64_t ck = kKeyMax;
      if (idx < size) ck = c0 == 1 ? sk[idx] : *kp(idx);
      const uint64_t m = warp_min_u64(ck);
      if (m >= x) break;
      const int src = __ffs(__ballot_sync(kFullMask, ck == m)) - 1;
      if (lane == 0) *kp(pos) = m;
      pos = c0 + src;
    }
    if (lane == 0) *kp(pos) = x;
    __syncwarp();
  }

  __device__ void pop() {
    const int n = --size;
    if (n == 0) return;
    const uint64_t x = *kp(n);
    sift_down(0, x);
  }

  __device__ bool push(uint64_t key) {
    if (size >= P.qcap) return false;
    int pos = size++;
    while (pos > 0) {
      const int par = (pos - 1) >> 5;
      const uint64_t pk = *kp(par);
      if (pk <= key) break;
      if (lane_id() == 0) *kp(pos) = pk;
      pos = par;
    }
    if (lane_id() == 0) *kp(pos) = key;
    __syncwarp();
    return true;
  }

  __device__ void heapify() {
    if (size < 2) return;
    for (int pos = (size - 2) / 32; pos >= 0; --pos) {
      const uint64_t x = *kp(pos);
      __syncwarp();
      sift_down(pos, x);
    }
  }
};

// ---------------------------------------------------------------------------
// HBM event log: unordered 8-byte entries -- (accelerator << g.ds) | key when
// the accelerator id fits above the key, else the key with the accelerator
// in a side byte array.  Slots [0, ms) are in shared memory, the rest in
// global scratch.
// ---------------------------------------------------------------------------
struct MemLog {
  const SimParams& P;
  uint64_t* sk;
  uint8_t* sd;
  uint8_t* sl;  // the warp's scratch slot
  int n;

  __device__ __forceinline__ uint64_t* kp(int i) const {
    return i < P.ms ? sk + i : reinterpret_cast<uint64_t*>(sl + P.off_mk) + (i - P.ms);
  }
  __device__ __forceinline__ uint8_t* dp(int i) const { return i < P.ms ? sd + i : sl + P.off_md + (i - P.ms); }
};

// ---------------------------------------------------------------------------
// Per-accelerator state.  Free times: a shared array of the kernel's time
// type.  Live bytes: a shared array (the drain updates it a batch at a time).
// Peak bytes: a shared array, or with more than 32 accelerators (!kPkShared) an
// array in the warp's global scratch (only raised by atomicMax and read where an
// allocation may exceed it).
// ---------------------------------------------------------------------------
// kParts: a drain's sums cover 2^kParts parts of its time.
template <bool kPkShared, typename TM, int kParts>
struct Devices {
  TM* fr;       // shared [D]
  int64_t* lv;  // shared [D]
  int64_t* pk;  // [D], shared or global
  uint32_t* acc;   // shared [(4 << kParts) * D], zero between drains (kPkShared)
  uint32_t* over;  // shared [8] (!kPkShared)
  int D;
  __device__ void setup(const DevGmg& g, uint8_t* sm, int64_t* pk_global) {
    D = g.D;
    if (kPkShared) {  // sums of a drain by accelerator, else a bit set of accelerators
      acc = reinterpret_cast<uint32_t*>(sm);
      sm += (16 << kParts) * (size_t)D;
    } else {
      over = reinterpret_cast<uint32_t*>(sm);
      sm += 32;
    }
    lv = reinterpret_cast<int64_t*>(sm);
    pk = kPkShared ? lv + D : pk_global;  // a compile-time fact of the instance
    fr = reinterpret_cast<TM*>(lv + (kPkShared ? 2 * D : D));
  }
  __device__ void reset_free(const DevGmg& g) {
    for (int d = lane_id(); d < D; d += 32) fr[d] = (TM)g.avail0[d];
    __syncwarp();
  }
  __device__ void reset_bytes(const DevGmg& g) {
    const unsigned l = lane_id();
    for (int d = l; d < D; d += 32) {
      lv[d] = g.base[d];
      pk[d] = g.base[d];
      if (kPkShared)
        for (int w = 0; w < 1 << kParts; ++w) reinterpret_cast<uint4*>(acc)[(d << kParts) + w] = make_uint4(0u, 0u, 0u, 0u);
    }
    __syncwarp();
  }
  // One event at a time (used when accelerator ids do not fit in the sort key).
  __device__ __forceinline__ bool alloc(int d, int64_t b, int64_t cap) {
    const int64_t v = lv[d] + b;
    const int64_t p = pk[d];
    __syncwarp();
    if (lane_id() == 0) {
      lv[d] = v;
      if (v > p) pk[d] = v;
    }
    __syncwarp();
    return v > cap;
  }
  __device__ __forceinline__ void release(int d, int64_t b) {
    const int64_t v = lv[d] - b;
    __syncwarp();
    if (lane_id() == 0) lv[d] = v;
    __syncwarp();
  }
  __device__ void save_free(int64_t* dst) const {
    for (int d = lane_id(); d < D; d += 32) dst[d] = (int64_t)fr[d];
  }
  __device__ void save_bytes(int64_t* dst) const {
    for (int d = lane_id(); d < D; d += 32) {
      dst[D + d] = lv[d];
      dst[2 * D + d] = kPkShared ? pk[d] : __ldcg(pk + d);
    }
  }
  __device__ void load_free(const int64_t* src) {
    for (int d = lane_id(); d < D; d += 32) fr[d] = (TM)src[d];
    __syncwarp();
  }
  __device__ void load_bytes(const int64_t* src) {
    for (int d = lane_id(); d < D; d += 32) {
      lv[d] = src[D + d];
      pk[d] = src[2 * D + d];
      if (kPkShared)
        for (int w = 0; w < 1 << kParts; ++w) reinterpret_cast<uint4*>(acc)[(d << kParts) + w] = make_uint4(0u, 0u, 0u, 0u);
    }
    __syncwarp();
  }
  // Largest final free time over the accelerators whose free time moved past
  // their initial availability (0 if none).  Uniform result.
  __device__ int64_t max_busy(const DevGmg& g) const {
    uint64_t m = 0;
    for (int d = lane_id(); d < D; d += 32) {
      const int64_t f = (int64_t)fr[d];
      if (f > g.avail0[d]) m = (uint64_t)f > m ? (uint64_t)f : m;
    }
    return (int64_t)warp_max_u64(m);
  }
  __device__ void write_peak(int64_t* dst) const {
    for (int d = lane_id(); d < D; d += 32) dst[d] = kPkShared ? pk[d] : __ldcg(pk + d);
  }
};

// Shared-memory carve-up per warp: READY pool, heap head, event-log head, sort
// area, accelerator state.
struct WarpSmem {
  uint64_t* pool;   // [pool]
  uint32_t* oplog;  // [opcap]
  uint64_t* heap;   // [qs]
  uint64_t* logk;   // [ms]
  uint64_t* sortk;  // [P.sortcap]
  uint8_t* logd;    // [ms]
  uint8_t* sortd;   // [P.sortcap]
  uint8_t* fstk;    // [pool]
  uint8_t* dev;     // accelerator state (P.dev_bytes)
};

__device__ __forceinline__ size_t align16(size_t x) { return (x + 15) & ~(size_t)15; }

__device__ __forceinline__ WarpSmem carve_smem(uint8_t* smem, const SimParams& P, unsigned wib) {
  // the side bytes (accelerator of a log entry) are left out where the
  // accelerator is inside the entry and shared memory is tight (P.no_side)
  const size_t side = P.no_side ? 0 : 1;
  const size_t head = align16((size_t)P.pool * 9 + (size_t)P.qs * 8 + (size_t)P.ms * (8 + side) +
                              (size_t)P.sortcap * (8 + side) + (size_t)P.opcap * 4);
  const size_t per = head + (size_t)P.dev_bytes + (size_t)P.pair_bytes;
  uint8_t* b = smem + per * wib;
  WarpSmem w;
  w.pool = reinterpret_cast<uint64_t*>(b);
  w.heap = w.pool + P.pool;
  w.logk = w.heap + P.qs;
  w.sortk = w.logk + P.ms;
  w.logd = reinterpret_cast<uint8_t*>(w.sortk + P.sortcap);
  w.sortd = w.logd + P.ms * side;
  w.oplog = reinterpret_cast<uint32_t*>(w.sortd + P.sortcap * side);
  w.fstk = reinterpret_cast<uint8_t*>(w.oplog + P.opcap);
  w.dev = b + head;
  return w;
}

// ---------------------------------------------------------------------------
// One warp's simulator.
// ---------------------------------------------------------------------------
// kT32: every time of the graph is below 2^32 - 1 (the host's bound), so ready,
// start, finish, free and arrival times are carried as uint32 (bytes, scores
// and outputs stay int64).
// kTypes: the graph has several accelerator types (durations per (type, op)).
// kNarrow: at most 32 accelerators.
// kPool: pending READY ops are keys in a pool in shared memory (the pure-latency
// kernels of more than 32 accelerators, where more ops are pending than a warp
// has lanes), else each lane holds one.
// kParts: a drain's sums cover 2^kParts parts of its time (at most 32 accelerators).
// kHot: the sweep reads compact 16-byte records (duration, transfer time, flags,
// both CSR lists) instead of the 64-byte ones -- kHotGlobal through the
// read-only path, kHotShared from the CTA's shared-memory copy (staged by
// sim_full_staged_kernel).
constexpr int kHotNone = 0, kHotGlobal = 1, kHotShared = 2;
// kRole: a candidate may have two warps (few candidates: what counts is then the
// time of one simulation, and nothing in the sweep depends on the HBM
// accounting).  kSweep starts the ops and hands them over in batches, kAccount
// generates and applies their HBM events and writes the results; kBoth does
// both in one warp.  (One warp / two, ms: 14 placements of the prefill graph 1.84 /
// 1.41, 2,048 2.07 / 1.53, 2,048 of a decode graph of 49,408 ops 65.7 / 31.3.)
constexpr int kBoth = 0, kSweep = 1, kAccount = 2;

// What the sweep hands over: n started ops (in the buffer of the same index) and
// what to do once their events are generated.
struct Hand {
  int64_t t;       // drain limit, time of the checkpoint, or the candidate
  int64_t score, nev;
  int32_t n, flags;
  int32_t iters, status;
  int32_t ck, pad;
};
constexpr int kHandDrain = 1, kHandEnd = 2, kHandCheckpoint = 4, kHandKeep = 8, kHandResume = 16, kHandQuit = 32;

// Named barriers of a pair, a block of 64 threads: full 0, full 1, empty 0, empty
// 1.  The ids are immediates: an id in a register would make every block claim
// all 16 barriers, and an SM has 64 (measured: 4 blocks instead of 14).
__device__ __forceinline__ void pair_sync(int id) {
  __syncwarp();
  if (id == 0) asm volatile("barrier.sync 0, 64;" ::: "memory");
  else if (id == 1) asm volatile("barrier.sync 1, 64;" ::: "memory");
  else if (id == 2) asm volatile("barrier.sync 2, 64;" ::: "memory");
  else asm volatile("barrier.sync 3, 64;" ::: "memory");
}
__device__ __forceinline__ void pair_arrive(int id) {
  __threadfence_block();
  __syncwarp();
  if (id == 0) asm volatile("barrier.arrive 0, 64;" ::: "memory");
  else if (id == 1) asm volatile("barrier.arrive 1, 64;" ::: "memory");
  else if (id == 2) asm volatile("barrier.arrive 2, 64;" ::: "memory");
  else asm volatile("barrier.arrive 3, 64;" ::: "memory");
}

template <bool kNarrow, int kMode, bool kKey, bool kT32 = false, bool kTypes = false, int kHot = kHotNone,
          bool kPool = !kNarrow, int kRole = kBoth, int kParts = kPartsLog>
struct Sim {
  static_assert(kHot == kHotNone || (kT32 && !kTypes), "compact records: 32-bit times, one type");
  using tm_t = typename std::conditional<kT32, uint32_t, int64_t>::type;
  const SimParams& P;
  const DevGmg& g;
  static constexpr int kSlots = kReadyPoolWide / 32;  // pool slots per lane (kPool)
  static constexpr bool kCompact = kHot != kHotNone, kKeyed = kKey, kPooled = kPool;
  static constexpr int kRoleOf = kRole;
  static constexpr tm_t kNever = kT32 ? (tm_t)0xffffffffu : (tm_t)kI64Max;  // later than every time
  struct Pending {
    tm_t r, e, dur;  // ready time, earliest finish (both kNever: empty), duration
    uint32_t op;
    int d;           // its accelerator
  };
  KeyCodec kc;      // HBM log entries (and the arbitrated simulators' READY keys)
  ReadyCodec rq;    // READY keys of the pool
  ReadyHeap q;      // READY keys beyond the pool (the lanes)
  Pending pd;       // !kPool: this lane's pending op
  uint64_t* pool;   // kPool: shared [32 * kSlots], pending READY keys (kKeyMax = empty)
  uint8_t* fstk;    // shared [32 * kSlots]: the empty slots, a stack of nfree
  uint64_t* bounce; // kPool: shared [48], a batch's keys and slots on their way to its lanes (the sort
                    // area, free between drains; of a pair's sweep its own)
  int nfree;
  MemLog log;
  uint64_t* sortk;
  uint8_t* sortd;
  tm_t drained;     // every event before this time is applied, none after it
  uint32_t* oplog;  // ops started since the last HBM-event generation (a pair: two buffers, oplog and hands of index hb)
  Hand* hands;      // shared [2]
  int hb;
  int opn;
  Devices<kNarrow, tm_t, kParts> dv;
  const uint8_t* row;
  tm_t* fbuf;       // finish times (scratch)
  uint8_t* sl;      // the warp's scratch slot (the less used arrays in it are found from the launch parameters)
  __device__ __forceinline__ tm_t* holdb() const { return reinterpret_cast<tm_t*>(sl + P.off_hold); }  // [N] latest outgoing arrival of the op's output
  __device__ __forceinline__ uint32_t* bits() const { return reinterpret_cast<uint32_t*>(sl + P.off_bits); }
  __device__ __forceinline__ int64_t* creq() const { return reinterpret_cast<int64_t*>(sl + P.off_creq); }
  // incremental resume
  const int64_t* rb;
  const int64_t* fb;
  tm_t Tc, T0;
  // running results
  int rootptr;
  uint64_t rkey;    // root_keys[rootptr], kKeyMax past the end
  int64_t score, nev;   // each lane's share, summed at the end
  int64_t readypops;
  int32_t iters;        // ops started (loop guard; the event count of a full run)
  int64_t last_t;       // latest READY time handled, kept in base mode only (checkpoints)
  int32_t vflag, vop, vdev, status;
  int64_t vt;
  // base checkpoints
  int ck, next_ck;
  // staged GMG (kHotShared): shared copies
  const uint4* sh_hot;      // per op {dur, xq | flags << 29, succ_off | nsucc << 24, pred_off | npred << 24}
  const uint32_t* sh_rel;   // per op release
  const uint32_t* sh_succ;  // successor lists
  const uint32_t* sh_pred;  // predecessor lists (hold bits included)

  __device__ Sim(const SimParams& p) : P(p), g(p.g), kc{p.g}, rq{p.g}, q{p}, log{p} {}
  __device__ __forceinline__ uint64_t lowmask() const { return kKey ? g.keymask : kKeyMax; }  // key of a log entry

  // Started ops are those with a finish time: every finish time is >= 1, the
  // finish array is zeroed per candidate, and the sweep marks a join whose READY
  // key is queued with kQueued.
  static constexpr tm_t kQueued = (tm_t)-1;
  static __device__ __forceinline__ bool started(tm_t f) { return kT32 ? (uint32_t)f - 1u < 0xfffffffeu : f > 0; }
  // The low 32 bits of a base-snapshot time (little-endian int64).
  static __device__ __forceinline__ tm_t base_time(const int64_t* a, uint32_t x) {
    if (kT32) return (tm_t)__ldg(reinterpret_cast<const uint32_t*>(a) + 2 * (size_t)x);
    return (tm_t)__ldg(a + x);
  }
  // Duration of op i on accelerator d: by the accelerator's type when the
  // graph has several (Sec. 3.3.1 keeps one operator estimate per (type,
  // operator)), else the op record's dur (dflt).
  __device__ __forceinline__ int64_t dur_of(uint32_t i, int d, int64_t dflt) const {
    if (kTypes) return __ldg(g.durt + (size_t)i * g.ntypes + __ldg(g.dtype + d));
    return dflt;
  }
  // Finish time of a simulated op (incremental candidates start from
  // fill_fin: ops started before the resume point keep their base finish).
  __device__ __forceinline__ tm_t fin(uint32_t x) const { return fbuf[x]; }

  // Transfer estimator of one output over link d -> e (d != e), Sec. 3.3.1.
  __device__ __forceinline__ tm_t xfer(int d, int e, int64_t bytes, int64_t xq) const {
    if (g.uniform) return (tm_t)xq + (tm_t)g.lat0;
    const longlong2* L = reinterpret_cast<const longlong2*>(g.links + (d * g.D + e));
    const longlong2 a = __ldg(L), b = __ldg(L + 1);
    LinkRec l;
    l.magic = (uint64_t)a.x;
    l.bw = a.y;
    l.lat = b.x;
    l.shift = (int32_t)(b.y & 0xffffffff);
    return (tm_t)(ceil_div_link(bytes, l) + l.lat);
  }

  // Latest arrival of p's output at another accelerator (or f_p): the
  // earliest its source copy may be released.  Per lane.
  __device__ tm_t lane_hold(uint32_t p, tm_t fp, int dp) const {
    const int64_t pb = op_durbytes(g.ops, p).y;
    const XqSucc ps = op_xqsucc(g.ops, p);
    const int64_t pxq = ps.xq;
    tm_t h = fp;
    for (uint32_t u = 0; u < ps.nsucc; ++u) {
      const int du = row[__ldg(g.succ + ps.succ_off + u)];
      if (du != dp) {
        const tm_t a = fp + xfer(dp, du, pb, pxq);
        h = a > h ? a : h;
      }
    }
    return h;
  }


  __device__ __forceinline__ tm_t warp_min_t(tm_t v) const {
    if (kT32) return (tm_t)__reduce_min_sync(kFullMask, (unsigned)v);
    return (tm_t)warp_min_u64((uint64_t)v);  // times are >= 0
  }

  __device__ __forceinline__ void load_root() {
    rkey = rootptr < g.nroots ? __ldg(g.root_keys + rootptr) : kKeyMax;
  }

  // Every lane with `want` logs (key, dev).  Uniform call.
  __device__ __forceinline__ void log_event(bool want, uint64_t key, int dev) {
    const uint32_t b = __ballot_sync(kFullMask, want);
    const int cnt = __popc(b);
    const int pos = log.n + __popc(b & lanes_below());
    if (kKey && log.n + 32 <= P.ms) {
      // fast path: every lane's slot is in shared memory
      if (want) log.sk[pos] = ((uint64_t)(dev & 0xff) << g.ds) | key;
      log.n += cnt;
      return;
    }
    if (cnt == 0 || status) return;
    if (log.n + cnt > P.mcap) {
      status = GMG_SIM_QUEUE;
      return;
    }
    if (want) {
      *log.kp(pos) = kKey ? (((uint64_t)(dev & 0xff) << g.ds) | key) : key;
      if (!kKey) *log.dp(pos) = (uint8_t)dev;
    }
    log.n += cnt;
  }

  // Zero this candidate's finish times (16-byte stores; the array is padded).
  __device__ void zero_fin() {
    uint4* v = reinterpret_cast<uint4*>(fbuf);
    const int nv = (int)((sizeof(tm_t) * (size_t)g.n + 15) / 16);
    for (int x = lane_id(); x < nv; x += 32) v[x] = make_uint4(0u, 0u, 0u, 0u);
    __syncwarp();
  }

  // An incremental candidate's finish times at the resume point T_c: the
  // base finish of every op started before it (base ready time < T_c), zero
  // for the others and for the padding.  Four ops in flight per lane.
  __device__ void fill_fin() {
    const int n = g.n;
    const int np = (int)((sizeof(tm_t) * (size_t)n + 15) / 16 * 16 / sizeof(tm_t));
    int x = (int)lane_id();
    for (; x + 96 < np; x += 128) {
      tm_t v[4];
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        const int i = x + 32 * u;
        const bool in = i < n;
        const tm_t r = in ? base_time(rb, (uint32_t)i) : Tc;
        const tm_t f = in ? base_time(fb, (uint32_t)i) : 0;
        v[u] = r < Tc ? f : 0;
      }
#pragma unroll
      for (int u = 0; u < 4; ++u) fbuf[x + 32 * u] = v[u];
    }
    for (; x < np; x += 32) {
      const bool in = x < n;
      const tm_t r = in ? base_time(rb, (uint32_t)x) : Tc;
      fbuf[x] = r < Tc ? base_time(fb, (uint32_t)x) : 0;
    }
    __syncwarp();
  }

  __device__ void reset_common() {
    const unsigned lane = lane_id();
    if constexpr (kRole != kAccount) {
      zero_fin();
      for (int r = lane; r < g.R; r += 32) creq()[r] = 0;
      dv.reset_free(g);
      q.size = 0;
      if constexpr (kPool) empty_pool(0);
      else pd.r = pd.e = kNever;
      rootptr = 0;
      load_root();
      score = 0;
      iters = nev = readypops = 0;
      last_t = -1;
    }
    if constexpr (kRole != kSweep) {
      dv.reset_bytes(g);
      log.n = 0;
      drained = 0;
      vflag = 0;
      vop = vdev = -1;
      vt = -1;
    }
    opn = 0;
    status = GMG_SIM_OK;
    __syncwarp();
  }

  // -------------------------------------------------------------------------
  // HBM events of the ops started since the last generation, one op per lane
  // (Sec. 3.3.2 residency, Recv before Send of Sec. 3.5.2): the op's own
  // output allocated at s; a receive copy on every other accelerator of a
  // successor allocated at f (released on arrival if no listed consumer is
  // there); the own copy released at the latest outgoing arrival if no
  // listed consumer is local; and for every held input whose last local
  // consumer this op is, that copy released at f (an own copy not before its
  // producer's outgoing arrivals).  Ops on one accelerator finish in the
  // order they start, so "last consumer here" compares finish times and can
  // be decided any time after the op started.
  //
  // Bounded by the chain of dependent loads (record, list entries, placement
  // and finish times of the ops on them): the first two entries of both lists
  // -- all that most ops have -- are loaded side by side, one level after the
  // other, and a lane's events are written together.
  // -------------------------------------------------------------------------

  // One event of this lane in the making: appended by log_lanes.
  __device__ __forceinline__ uint64_t entry(tm_t t, uint32_t cls, uint32_t op, int dev) const {
    const uint64_t k = kc.make(t, cls, op);
    return kKey ? ((uint64_t)(dev & 0xff) << g.ds) | k : k;
  }
  template <int kMax>
  __device__ __forceinline__ void log_lanes(const uint64_t (&ev)[kMax], const int (&dev)[kMax], uint32_t want) {
    const unsigned lane = lane_id();
    const int c = __popc(want);
    int at = c;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int y = __shfl_up_sync(kFullMask, at, o);
      if ((int)lane >= o) at += y;
    }
    const int total = __shfl_sync(kFullMask, at, 31);
    at += log.n - c;
    if (log.n + total <= P.ms) {
#pragma unroll
      for (int x = 0; x < kMax; ++x)
        if ((want >> x) & 1u) {
          log.sk[at] = ev[x];
          if (!kKey) log.sd[at] = (uint8_t)dev[x];
          ++at;
        }
    } else {
      if (status) return;
      if (log.n + total > P.mcap) {
        status = GMG_SIM_QUEUE;
        return;
      }
#pragma unroll
      for (int x = 0; x < kMax; ++x)
        if ((want >> x) & 1u) {
          *log.kp(at) = ev[x];
          if (!kKey) *log.dp(at) = (uint8_t)dev[x];
          ++at;
        }
    }
    log.n += total;
  }

  // Whether op x (ending at f on d) is the last listed consumer on d of its
  // predecessor: ps is the predecessor's entry in x's list.
  __device__ __forceinline__ bool releases(uint32_t x, int d, tm_t f, const uint2 ps) const {
    if (!(ps.x & kHoldBit)) return false;
    const uint32_t sb = ps.y;
    if (sb == kSibNone) return true;
    if (sb != kSibMany) {
      if (row[sb & ~kSibLater] != d) return true;
      if (sb & kSibLater) return false;  // the other consumer finishes later
      const tm_t fs = fin(sb);
      return started(fs) && fs < f;
    }
    const uint32_t p = ps.x & kIdMask;
    const XqSucc px = op_xqsucc(g.ops, p);
    const uint4 pcs = op_cons(g.ops, p);
    const bool all = (pcs.w & kAllCons) != 0;
    const uint32_t* lst = all ? g.succ + px.succ_off : g.cons + pcs.x;
    const uint32_t nl = all ? px.nsucc : pcs.y;
    for (uint32_t w = 0; w < nl; ++w) {
      const uint32_t c = __ldg(lst + w);
      const tm_t fc = c != x ? fin(c) : 0;
      if (c != x && row[c] == d && !(started(fc) && fc < f)) return false;
    }
    return true;
  }
  // When p's copy on d that an op ending at f there releases is freed (p's own
  // copy: not before its outgoing arrivals, recorded when p's events were
  // generated; p started before this op).
  __device__ __forceinline__ tm_t freed_at(uint32_t p, int d, tm_t f) const {
    if (row[p] != d) return f;
    const tm_t h = (kMode == kInc && base_time(rb, p) < Tc) ? lane_hold(p, fin(p), d) : holdb()[p];
    return h > f ? h : f;
  }
  // A listed consumer of x on accelerator e?
  __device__ __forceinline__ bool consumer_on(const uint4& cs, int e) const {
    for (uint32_t w = 0; w < cs.y; ++w)
      if (row[__ldg(g.cons + cs.x + w)] == e) return true;
    return false;
  }

  __device__ void generate() {
    const unsigned lane = lane_id();
    for (int c0 = 0; c0 < opn; c0 += 32) {
      const int idx = c0 + (int)lane;
      const bool v = idx < opn;
      const uint32_t x = v ? oplog[idx] : 0u;
      Start s;
      s.nsucc = 0;
      s.flags = kAllCons;
      s.dur = s.xq = 0;
      s.bytes = 0;
      s.succ_off = 0;
      uint32_t pred_off = 0, npred = 0;
      int d = 0;
      tm_t f = 0;
      if (v) {
        d = row[x];
        f = fbuf[x];
        if constexpr (kHot != kHotNone) {
          const uint4 h = hot(x);
          s.dur = (tm_t)h.x;
          s.xq = (tm_t)(h.y & 0x1fffffffu);
          s.flags = h.y >> 29;
          s.succ_off = h.z & 0xffffffu;
          s.nsucc = h.z >> 24;
          pred_off = h.w & 0xffffffu;
          npred = h.w >> 24;
        } else {
          s = start_of(x, d);
          const RelPred rp = op_relpred(g.ops, x);
          pred_off = rp.pred_off;
          npred = rp.npred;
        }
      }
      // list entries, then what they point at, side by side
      int du[2] = {d, d};
      uint2 ps[2] = {make_uint2(0u, 0u), make_uint2(0u, 0u)};
#pragma unroll
      for (int u = 0; u < 2; ++u) {
        if ((uint32_t)u < npred) ps[u] = __ldg(g.predsib + pred_off + u);
        if ((uint32_t)u < s.nsucc) du[u] = row[succ_at(s.succ_off + u)];
      }
      const bool all = (s.flags & kAllCons) != 0;
      uint64_t ev[6];
      int dev[6];
      uint32_t want = v ? 1u : 0u;
      dev[0] = d;
      ev[0] = entry(f - s.dur, kAlloc, x, d);
      // receive copies, one per distinct remote accelerator
      tm_t hold = f;
      bool localc = false;
#pragma unroll
      for (int u = 0; u < 2; ++u) {
        dev[1 + u] = du[u];
        ev[1 + u] = entry(f, kAlloc, x, du[u]);
        if ((uint32_t)u < s.nsucc) {
          if (du[u] == d) {
            localc = true;
          } else if (u == 0 || du[1] != du[0]) {
            want |= 2u << u;
            const tm_t a = f + (kHot != kHotNone ? s.xq + (tm_t)g.lat0 : xfer(d, du[u], s.bytes, s.xq));
            hold = a > hold ? a : hold;
          }
        }
      }
      if (__any_sync(kFullMask, s.nsucc > 2u || !all)) {
        // longer lists, and copies that nobody listed holds
        const uint32_t maxs = __reduce_max_sync(kFullMask, s.nsucc);
        const uint4 cs = v && !all ? op_cons(g.ops, x) : make_uint4(0u, 0u, 0u, 0u);
        for (uint32_t u = 0; u < maxs; ++u) {
          bool first = false;
          int e = d;
          tm_t a = f;
          if (u < s.nsucc) {
            e = row[succ_at(s.succ_off + u)];
            first = e != d;
            localc = localc || e == d;
            for (uint32_t w = 0; w < u && first; ++w) first = row[succ_at(s.succ_off + w)] != e;
            if (first) {
              a = f + (kHot != kHotNone ? s.xq + (tm_t)g.lat0 : xfer(d, e, s.bytes, s.xq));
              hold = a > hold ? a : hold;
            }
          }
          if (u >= 2u) log_event(first, kc.make(f, kAlloc, x), e);
          log_event(first && !all && !consumer_on(cs, e), kc.make(a, kFree, x), e);
        }
        if (v && !all) localc = consumer_on(cs, d);
      }
      if (v && !localc) want |= 8u;
      dev[3] = d;
      ev[3] = entry(hold, kFree, x, d);
      if (v) holdb()[x] = hold;
      __syncwarp();
      // releases of the inputs this op holds
#pragma unroll
      for (int u = 0; u < 2; ++u) {
        const uint32_t p = ps[u].x & kIdMask;
        dev[4 + u] = d;
        ev[4 + u] = 0;
        if (releases(x, d, f, ps[u])) {
          want |= 16u << u;
          ev[4 + u] = entry(freed_at(p, d, f), kFree, p, d);
        }
      }
      log_lanes<6>(ev, dev, want);
      if (__any_sync(kFullMask, npred > 2u)) {
        const uint32_t maxp = __reduce_max_sync(kFullMask, npred);
        for (uint32_t u = 2; u < maxp; ++u) {
          bool rel = false;
          tm_t t = f;
          uint32_t p = 0;
          if (u < npred) {
            const uint2 e = __ldg(g.predsib + pred_off + u);
            p = e.x & kIdMask;
            rel = releases(x, d, f, e);
            if (rel) t = freed_at(p, d, f);
          }
          log_event(rel, kc.make(t, kFree, p), d);
        }
      }
    }
    opn = 0;
    __syncwarp();
  }

  // Apply sorted events one at a time (accelerator ids not in the key).
  __device__ void apply_serial(int m) {
    for (int e = 0; e < m; ++e) {
      const uint64_t k = sortk[e];
      const int dev = sortd[e];
      const uint32_t op = kc.op(k);
      const int64_t b = __ldg(g.bytes + op);
      if (kc.cls(k) == kFree) {
        dv.release(dev, b);
      } else if (dv.alloc(dev, b, __ldg(g.cap + dev))) {
        const int64_t t = kc.time(k);
        if (!vflag || (t == vt && (int32_t)op == vop && dev < vdev)) {
          vflag = 1;
          vt = t;
          vop = (int32_t)op;
          vdev = dev;
        }
      }
    }
    __syncwarp();
  }

  // Apply 32 consecutive events of the (accelerator, time, class, op) order,
  // one per lane (v: lane holds an event).  Each accelerator's events are
  // contiguous, so a segmented warp scan of the byte deltas gives the live
  // bytes after every event; allocations raise the accelerator's peak; the
  // smallest (time, op, accelerator) allocation over capacity is kept in
  // vmin.
  __device__ __forceinline__ void apply_chunk(uint64_t key, bool v, uint64_t& vmin) {
    const unsigned lane = lane_id();
    const uint64_t tmask = (1ull << g.tb) - 1ull;
    const int dev = v ? (int)(key >> g.ds) : -1 - (int)lane;
    const uint32_t op = (uint32_t)(key & g.opmask);
    const bool isalloc = v && kc.cls(key) == kAlloc;
    int64_t delta = 0;
    if (v) {
      const int64_t b = __ldg(g.bytes + op);
      delta = isalloc ? b : -b;
    }
    int64_t s = delta;
#pragma unroll
    for (int off = 1; off < 32; off <<= 1) {
      const int64_t o = __shfl_up_sync(kFullMask, s, off);
      const int od = __shfl_up_sync(kFullMask, dev, off);
      if ((int)lane >= off && od == dev) s += o;
    }
    const int64_t live = (v ? dv.lv[dev] : 0) + s;
    const int nd = __shfl_down_sync(kFullMask, dev, 1);
    const bool last = v && (lane == 31 || nd != dev);
    const bool over = isalloc && live > __ldg(g.cap + dev);
    const uint64_t vk = over ? ((((key >> (g.ib + 2)) & tmask) << (g.ib + 8)) | ((uint64_t)op << 8) |
                                (uint64_t)dev)
                             : kKeyMax;
    const uint64_t cm = warp_min_u64(vk);
    vmin = cm < vmin ? cm : vmin;
    __syncwarp();
    // live bytes are never negative; in shared memory most do not raise the peak
    if (isalloc && (!kNarrow || live > dv.pk[dev]))
      atomicMax(reinterpret_cast<unsigned long long*>(dv.pk + dev), (unsigned long long)live);
    if (last) dv.lv[dev] = live;
    __syncwarp();
  }

  // every event of a drain is later than every event already applied, so
  // an earlier violation stands
  __device__ __forceinline__ void settle_violation(uint64_t vmin) {
    if (!vflag && vmin != kKeyMax) {
      vflag = 1;
      vt = (int64_t)(vmin >> (g.ib + 8));
      vop = (int32_t)((vmin >> 8) & g.opmask);
      vdev = (int32_t)(vmin & 0xffu);
    }
  }

  __device__ void apply_segmented(int m) {
    uint64_t vmin = kKeyMax;
    for (int c0 = 0; c0 < m; c0 += 32) {
      const int idx = c0 + (int)lane_id();
      const bool v = idx < m;
      apply_chunk(v ? sortk[idx] : 0ull, v, vmin);
    }
    settle_violation(vmin);
  }

  // Sort and apply m extracted events of accelerators whose order matters.
  // may_violate: one of them may exceed its capacity -- then equal times are
  // told apart by op id (the whole entry is the sort key), else the order of
  // equal times of one kind does not matter and 32 bits hold the key.  The staged
  // kernel keeps to one way: it serves the many candidates of small graphs, whose
  // warps run all of this code all the time, and both ways at once overflow the
  // instruction cache (386 ops, 8 accelerators, 4,096 placements: 588 -> 547 us,
  // 1,544 ops 1,909 -> 1,514; through L1 the prefill graph would lose, 3.06 -> 3.10).
  __device__ __forceinline__ void apply_ordered(int m, bool may_violate, tm_t span) {
    constexpr int kDevBits = kNarrow ? 5 : 8;
    if (kHot != kHotShared && !may_violate && m <= 32 && (span >> (32 - kDevBits - 6)) == 0) {
      apply_short(m);
    } else {
      sort_area(m);
      apply_segmented(m);
    }
  }

  // m <= 32 events, none of which exceeds a capacity: sorted in registers by
  // (accelerator, time since the last drain, frees first, position) in 32 bits,
  // then a prefix sum of the byte changes, less its value where the
  // accelerator's events begin, gives the live bytes after each.  (A bitonic
  // network over the 64-bit entries takes three times the instructions.)
  __device__ __forceinline__ void apply_short(int m) {
    constexpr int kDevBits = kNarrow ? 5 : 8;
    const int lane = (int)lane_id();
    const bool v = lane < m;
    uint32_t a = 0xffffffffu;
    int64_t delta = 0;
    if (v) {
      const uint64_t x = sortk[lane];
      const bool al = kc.cls(x) == kAlloc;
      const tm_t t = (tm_t)((x & lowmask()) >> (g.ib + 2)) - drained;
      delta = __ldg(g.bytes + (uint32_t)(x & g.opmask));
      if (!al) delta = -delta;
      a = ((uint32_t)(x >> g.ds) << (32 - kDevBits)) | ((uint32_t)t << 6) | (al ? 32u : 0u) | (uint32_t)lane;
    }
#pragma unroll
    for (int k = 2; k <= 32; k <<= 1) {
#pragma unroll
      for (int j = k >> 1; j > 0; j >>= 1) {
        const uint32_t o = __shfl_xor_sync(kFullMask, a, j);
        const bool keep_min = ((lane & j) == 0) == ((lane & k) == 0);
        a = keep_min ? (o < a ? o : a) : (o < a ? a : o);
      }
    }
    delta = __shfl_sync(kFullMask, delta, (int)(a & 31u));
    if (!v) delta = 0;
    const int dev = v ? (int)(a >> (32 - kDevBits)) : -1 - lane;
    int64_t s = delta;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int64_t y = __shfl_up_sync(kFullMask, s, o);
      if (lane >= o) s += y;
    }
    const int dl = __shfl_up_sync(kFullMask, dev, 1), dr = __shfl_down_sync(kFullMask, dev, 1);
    const uint32_t heads = __ballot_sync(kFullMask, lane == 0 || dl != dev);
    const int head = 31 - __clz(heads & (lanes_below() | (1u << lane)));
    const int64_t before = __shfl_sync(kFullMask, s - delta, head);
    const int64_t live = (v ? dv.lv[dev] : 0) + s - before;
    __syncwarp();
    if (v && (a & 32u) && (!kNarrow || live > dv.pk[dev]))
      atomicMax(reinterpret_cast<unsigned long long*>(dv.pk + dev), (unsigned long long)live);
    if (v && (lane == 31 || dr != dev)) dv.lv[dev] = live;
    __syncwarp();
  }

  // Extracted events are not summed up but ordered: sizes that the 24-bit halves
  // would not hold; and the staged kernel on one or two accelerators, where nearly
  // every drain can raise a peak (386 ops, 4,096 placements: 574 -> 549 us on two,
  // on eight 547 -> 563).
  __device__ __forceinline__ bool unsummed() const { return (kHot == kHotShared && g.D <= 2) || g.big_bytes; }

  // Apply the m events just extracted.  Their order matters only on an
  // accelerator whose peak they can raise (without a violation so far the peak
  // is within the capacity).  An upper bound of its live bytes is cheap: with at
  // most 32 accelerators extract() has summed up what is allocated and freed on
  // each in every part (2^kParts of them) of the time since the last drain, and within one
  // the live bytes are at most those at its start plus all its allocations; with
  // more (few events each) the whole drain is one such interval.  Everywhere
  // else the sums are enough.  (Prefill graph: 1.6 events an op are ordered with
  // one bound per drain, fewer with quarters; without the wide sort networks that
  // no drain then needs, 4,096 placements 3.66 ms -> 3.22.)
  __device__ __forceinline__ void apply_due(int m, tm_t span) {
    const unsigned lane = lane_id();
    uint32_t fail = 0u;
    bool viol = false;
    if constexpr (kNarrow) {
      if (unsummed()) {
        apply_ordered(m, true, span);
        return;
      }
      bool over = false;
      if ((int)lane < g.D) {
        uint4* q4 = reinterpret_cast<uint4*>(dv.acc) + (lane << kParts);
        const int64_t l0 = dv.lv[lane], peak = dv.pk[lane];
        int64_t l = l0, top = 0;
#pragma unroll
        for (int w = 0; w < 1 << kParts; ++w) {
          const uint4 x = q4[w];
          q4[w] = make_uint4(0u, 0u, 0u, 0u);
          const int64_t most = l + (int64_t)(((uint64_t)x.y << 24) + x.x);
          top = most > top ? most : top;
          l = most - (int64_t)(((uint64_t)x.w << 24) + x.z);
        }
        over = top > peak;
        if (!over) dv.lv[lane] = l;
        else viol = top > __ldg(g.cap + lane);
      }
      fail = __ballot_sync(kFullMask, over);
      if (fail == 0u) return;
    } else {
      // extract() has added the allocations to the live bytes
      if (lane < 8u) dv.over[lane] = 0u;
      __syncwarp();
      for (int c0 = 0; c0 < m; c0 += 32) {
        const int idx = c0 + (int)lane;
        if (idx < m) {
          const uint64_t e = sortk[idx];
          const int dev = (int)(e >> g.ds);
          if (kc.cls(e) == kAlloc && dv.lv[dev] > __ldcg(dv.pk + dev)) {
            atomicOr(dv.over + (dev >> 5), 1u << (dev & 31));
            viol = viol || dv.lv[dev] > __ldg(g.cap + dev);
          }
        }
      }
      __syncwarp();
    }
    viol = __any_sync(kFullMask, viol);
    // the other accelerators' events leave; with more than 32 accelerators
    // their frees are applied, and where the order matters the allocations are
    // taken back
    int keep = 0;
    for (int c0 = 0; c0 < m; c0 += 32) {
      const int idx = c0 + (int)lane;
      const bool v = idx < m;
      const uint64_t e = v ? sortk[idx] : 0ull;
      const int dev = (int)(e >> g.ds);
      bool k;
      if constexpr (kNarrow) {
        k = v && ((fail >> dev) & 1u);
      } else {
        k = v && ((dv.over[dev >> 5] >> (dev & 31)) & 1u);
        if (v && k == (kc.cls(e) == kAlloc))
          atomicAdd(reinterpret_cast<unsigned long long*>(dv.lv + dev),
                    (unsigned long long)-__ldg(g.bytes + (uint32_t)(e & g.opmask)));
      }
      const uint32_t bk = __ballot_sync(kFullMask, k);
      if (k) sortk[keep + __popc(bk & lanes_below())] = e;  // at most idx: in place
      keep += __popc(bk);
      __syncwarp();
    }
    if (keep) apply_ordered(keep, viol, span);
  }

  __device__ int count_below(uint64_t kmax) const {
    int c = 0;
    for (int c0 = 0; c0 < log.n; c0 += 32) {
      const int idx = c0 + (int)lane_id();
      const bool take = idx < log.n && (*log.kp(idx) & lowmask()) < kmax;
      c += __popc(__ballot_sync(kFullMask, take));
    }
    return c;
  }

  // Move the logged events whose key part is < kmax to the sort area (their
  // number is known to fit) and compact the rest; returns their number.  Sums
  // them up for apply_due on the way: with at most 32 accelerators what is
  // allocated and freed per accelerator and part of the time since the last
  // drain (parts of 2^wsh), each as sums of the low 24 and of the higher 24
  // bits of the sizes (32-bit shared atomics; at most 256 events), with more the
  // allocations into the live bytes.
  __device__ int extract(uint64_t kmax, int wsh) {
    const unsigned lane = lane_id();
    const bool side = !kKey;
    int m = 0, keep = 0;
    const int n = log.n;
    for (int c0 = 0; c0 < n; c0 += 32) {
      const int idx = c0 + (int)lane;
      const bool v = idx < n;
      uint64_t e = kKeyMax;
      uint8_t dv8 = 0;
      if (v) {
        if (idx < P.ms) {
          e = log.sk[idx];
          if (side) dv8 = log.sd[idx];
        } else {
          e = *log.kp(idx);
          if (side) dv8 = *log.dp(idx);
        }
      }
      const bool take = v && (e & lowmask()) < kmax;
      const uint32_t bt = __ballot_sync(kFullMask, take);
      const uint32_t bk = __ballot_sync(kFullMask, v && !take);
      if (take) {
        const int pos = m + __popc(bt & lanes_below());
        sortk[pos] = e;
        if (side) sortd[pos] = dv8;
        if constexpr (kKey) {
          const uint64_t b = (uint64_t)__ldg(g.bytes + (uint32_t)(e & g.opmask));
          const bool al = kc.cls(e) == kAlloc;
          const int dev = (int)(e >> g.ds);
          if constexpr (kNarrow) {
            const tm_t t = (tm_t)((e & lowmask()) >> (g.ib + 2)) - drained;
            const int w = min((int)(t >> wsh), (1 << kParts) - 1);
            uint32_t* a = dv.acc + 4 * ((dev << kParts) + w) + (al ? 0 : 2);
            if (!unsummed()) {
              atomicAdd(a, (uint32_t)b & 0xffffffu);
              atomicAdd(a + 1, (uint32_t)(b >> 24));
            }
          } else if (al) {
            atomicAdd(reinterpret_cast<unsigned long long*>(dv.lv + dev), (unsigned long long)b);
          }
        }
      } else if (v) {
        const int pos = keep + __popc(bk & lanes_below());  // pos <= idx: in place
        *log.kp(pos) = e;
        if (side) *log.dp(pos) = dv8;
      }
      m += __popc(bt);
      keep += __popc(bk);
      __syncwarp();
    }
    log.n = keep;
    return m;
  }

  // Bitonic sort of sortk[0, m) (and the side bytes alongside), padded to a
  // power of two >= 32.
  __device__ void sort_area(int m) {
    const unsigned lane = lane_id();
    const bool side = !kKey;
    int p2 = 32;
    while (p2 < m) p2 <<= 1;
    for (int x = m + (int)lane; x < p2; x += 32) sortk[x] = kKeyMax;
    __syncwarp();
    for (int k = 2; k <= p2; k <<= 1) {
      for (int j = k >> 1; j > 0; j >>= 1) {
        for (int t = lane; t < (p2 >> 1); t += 32) {
          const int i = ((t & ~(j - 1)) << 1) | (t & (j - 1));
          const int l = i + j;
          const uint64_t a = sortk[i], b = sortk[l];
          const bool asc = (i & k) == 0;
          if ((a > b) == asc) {
            sortk[i] = b;
            sortk[l] = a;
            if (side) {
              const uint8_t da = sortd[i], db = sortd[l];
              sortd[i] = db;
              sortd[l] = da;
            }
          }
        }
        __syncwarp();
      }
    }
  }

  // Apply every logged event that can no longer be preceded (time < t_next).
  __device__ __forceinline__ void drain(int64_t t_next) {
    generate();
    drain_log(t_next);
  }
  __device__ __forceinline__ void drain_log(int64_t t_next) {
    const uint64_t lim = t_next == kI64Max ? kKeyMax : kc.time_floor(t_next);
    // the time since the last drain, and parts of it (the last drain of all has one
    // interval)
    const tm_t span = t_next == kI64Max ? kNever : (tm_t)t_next - drained;
    int wsh = 8 * (int)sizeof(tm_t) - 1;
    if (span < ((tm_t)1 << 30)) wsh = max(0, 32 - __clz((uint32_t)span) - kParts);
    while (log.n > 0) {
      uint64_t kmax = lim;
      if (log.n > P.sortcap) {
        const int due = count_below(lim);
        if (due == 0) break;
        if (due > P.sortcap) {
          // Rare: more due events than the sort area.  Bisect a key bound
          // with at most P.sortcap events below it (at most n_dev <= P.sortcap
          // events share a key part).
          uint64_t lo = kKeyMax;
          for (int c0 = 0; c0 < log.n; c0 += 32) {
            const int idx = c0 + (int)lane_id();
            const uint64_t kk = idx < log.n ? (*log.kp(idx) & lowmask()) : kKeyMax;
            lo = kk < lo ? kk : lo;
          }
          lo = warp_min_u64(lo) + 1;  // 1 <= count_below(lo) <= P.sortcap
          uint64_t hi = lim;          // count_below(hi) > P.sortcap
          while (hi - lo > 1) {
            const uint64_t mid = lo + (hi - lo) / 2;
            if (count_below(mid) <= P.sortcap) lo = mid;
            else hi = mid;
          }
          kmax = lo;
        }
      }
      const int m = extract(kmax, wsh);
      if (m == 0) break;
      if (kKey) {
        apply_due(m, span);
      } else {
        sort_area(m);
        apply_serial(m);
      }
      if (kmax == lim) break;
    }
    drained = (tm_t)t_next;
  }

  __device__ void maybe_checkpoint(int64_t next_t, uint64_t held = kKeyMax);
  __device__ void save_accounts(int c, int64_t tn, bool keep);

  // -------------------------------------------------------------------------
  // The event loop (Sec. 3.3.3), many READY keys at a time.  Let lim be the
  // smallest earliest finish over every pending key.  A key pushed later is the
  // successor of a pending op (or of one that such an op makes ready), so its
  // ready time is >= lim: the pending keys with a time below lim are exactly the
  // next ones in key order, and none of them can make an op ready that precedes
  // another of them.  They are started together, one op per lane, each
  // accelerator's ops in key order, which gives the starts of handling them one
  // at a time.  An op's earliest finish is max(ready time, its accelerator's
  // free time when it was queued) + duration: free times only grow.
  //
  // What bounds the sweep is the chain of dependent instructions and loads per
  // op (record, successors, their placement and predecessors) and, one key at a
  // time, the extraction of the minimum; a batch pays each once for all its ops
  // and finds its keys with one reduction.
  // -------------------------------------------------------------------------
  __device__ __forceinline__ uint64_t outside_min() const {
    const uint64_t top = q.top();
    return rkey < top ? rkey : top;
  }
  __device__ __forceinline__ tm_t key_time(uint64_t k) const { return k == kKeyMax ? kNever : (tm_t)rq.time(k); }
  // Removes the smallest key outside the pool (root list or heap).
  __device__ __forceinline__ void take_outside(uint64_t x) {
    if (x == rkey) {
      ++rootptr;
      load_root();
    } else {
      __syncwarp();
      q.pop();
    }
  }
  // ---- a candidate's two warps ------------------------------------------------
  // The sweep owns buffer hb; handing it over, it waits until the other one is
  // free (two batches ahead at most).
  __device__ __forceinline__ void hand_over(int64_t t, int flags, int n) {
    if (lane_id() == 0) {
      Hand& h = hands[hb];
      h.t = t;
      h.flags = flags;
      h.n = n;
      h.ck = ck;
    }
    pair_arrive(hb);
    opn = 0;
    if (flags & kHandQuit) return;
    hb ^= 1;
    oplog += hb ? P.opcap : -P.opcap;
    pair_sync(2 + hb);
  }
  // The candidate's end: the other warp finishes it from these results.
  __device__ __forceinline__ void hand_end() {
    const int64_t sc = warp_sum_i64(score), ne = warp_sum_i64(nev);
    if (lane_id() == 0) {
      Hand& h = hands[hb];
      h.t = kI64Max;
      h.flags = kHandEnd;
      h.n = opn;
      h.score = sc;
      h.nev = ne;
      h.iters = iters;
      h.status = status;
    }
    pair_arrive(hb);
    pair_sync(2 + hb);  // the buffer stays this warp's
  }
  // One batch handed over (kAccount); returns its flags.
  __device__ __forceinline__ int take_hand(Hand& h) {
    pair_sync(hb);
    h = hands[hb];
    return h.flags;
  }
  __device__ __forceinline__ void free_hand() {
    pair_arrive(2 + hb);
    hb ^= 1;
    oplog += hb ? P.opcap : -P.opcap;
  }
  // Everything handed over up to the candidate's end, whose results are then
  // this warp's.
  __device__ __forceinline__ void account() {
    while (true) {
      Hand h;
      const int flags = take_hand(h);
      const bool end = (flags & kHandEnd) != 0;
      opn = h.n;
      if (end && h.status != GMG_SIM_OK) status = h.status;
      if (status == GMG_SIM_OK) generate();
      opn = 0;
      if (!end) free_hand();
      if (status == GMG_SIM_OK) drain_log(h.t);
      if (kMode == kBase && (flags & kHandCheckpoint)) save_accounts(h.ck, h.t, (flags & kHandKeep) != 0);
      if (end) {
        score = lane_id() == 0 ? h.score : 0;
        nev = lane_id() == 0 ? h.nev : 0;
        iters = h.iters;
        return;
      }
    }
  }
  __device__ __forceinline__ void done() { pair_arrive(2 + hb); }

  __device__ void run() {
    if (status) return;
    if constexpr (kPool) run_pool();
    else run_lanes();
  }

  // What starting an op needs of its record, and the record of a successor.
  struct Start {
    tm_t dur, xq;
    int64_t bytes;
    uint32_t succ_off, nsucc, flags;
    int32_t req;
  };
  __device__ __forceinline__ uint4 hot(uint32_t i) const { return kHot == kHotShared ? sh_hot[i] : __ldg(g.st_hot + i); }
  __device__ __forceinline__ uint32_t succ_at(uint32_t k) const {
    return kHot == kHotShared ? sh_succ[k] : __ldg(g.succ + k);
  }
  __device__ __forceinline__ uint32_t pred_at(uint32_t k) const {
    return (kHot == kHotShared ? sh_pred[k] : __ldg(g.pred + k)) & kIdMask;
  }
  __device__ __forceinline__ Start start_of(uint32_t i, int d) const {
    Start s;
    if constexpr (kHot != kHotNone) {
      const uint4 h = hot(i);
      s.dur = (tm_t)h.x;
      s.xq = (tm_t)(h.y & 0x1fffffffu);
      s.flags = h.y >> 29;
      s.succ_off = h.z & 0xffffffu;
      s.nsucc = h.z >> 24;
      s.bytes = 0;
      s.req = 0;  // read when the op ends a request
    } else {
      const longlong2 db = op_durbytes(g.ops, i);
      const XqSucc xs = op_xqsucc(g.ops, i);
      const uint4 cs = op_cons(g.ops, i);
      s.bytes = db.y;
      s.xq = (tm_t)xs.xq;
      s.succ_off = xs.succ_off;
      s.nsucc = xs.nsucc;
      s.req = (int32_t)cs.z;
      s.flags = cs.w;
      s.dur = (tm_t)dur_of(i, d, db.x);
    }
    return s;
  }
  // The time that p's output takes to dj (p on dp, another accelerator).
  __device__ __forceinline__ tm_t sends(uint32_t p, int dp, int dj) const {
    if constexpr (kHot != kHotNone) return (tm_t)(hot(p).y & 0x1fffffffu) + (tm_t)g.lat0;
    return xfer(dp, dj, op_durbytes(g.ops, p).y, op_xqsucc(g.ops, p).xq);
  }

  // The op started by this lane (i on d, ending at f) reaches its successor j:
  // ready once every predecessor has started, at the latest arrival over all of
  // them (Sec. 3.3.2).
  struct Reached {
    uint32_t j;
    int d;
    tm_t r, dur;
    bool rdy, join;
  };
  __device__ __forceinline__ Reached reach(uint32_t i, int d, tm_t f, const Start& s, uint32_t u) const {
    Reached x;
    x.j = succ_at(s.succ_off + u);
    x.d = row[x.j];
    uint32_t npred, pred_off;
    if constexpr (kHot != kHotNone) {
      const uint4 h = hot(x.j);
      x.dur = (tm_t)h.x;
      npred = h.w >> 24;
      pred_off = h.w & 0xffffffu;
      x.r = (tm_t)(kHot == kHotShared ? sh_rel[x.j] : __ldg(g.st_rel + x.j));
    } else {
      const RelPred jp = op_relpred(g.ops, x.j);
      x.dur = (tm_t)dur_of(x.j, x.d, op_durbytes(g.ops, x.j).x);
      npred = jp.npred;
      pred_off = jp.pred_off;
      x.r = (tm_t)jp.rel;
    }
    tm_t arr = f;
    if (x.d != d) arr += kHot != kHotNone ? s.xq + (tm_t)g.lat0 : xfer(d, x.d, s.bytes, s.xq);
    x.r = x.r > arr ? x.r : arr;
    x.rdy = true;
    x.join = npred > 1;
    if (npred == 2u) {  // one other predecessor: its loads side by side
      const tm_t fj = fin(x.j);  // nonzero: queued already, by another lane of this batch
      const uint32_t p0 = pred_at(pred_off), p1 = pred_at(pred_off + 1u);
      const uint32_t p = p0 == i ? p1 : p0;
      const tm_t a = fin(p);
      const int dp = row[p];
      const tm_t b = a + (dp != x.d ? sends(p, dp, x.d) : (tm_t)0);
      x.rdy = started(a) && fj == 0;
      x.r = b > x.r ? b : x.r;
    } else if (x.join) {
      const tm_t fj = fin(x.j);
      for (uint32_t t = 0; t < npred; ++t) {
        const uint32_t p = pred_at(pred_off + t);
        if (p == i) continue;
        tm_t a = fin(p);
        const int dp = row[p];
        if (!started(a)) {
          x.rdy = false;
          break;
        }
        if (dp != x.d) a += sends(p, dp, x.d);
        x.r = a > x.r ? a : x.r;
      }
      x.rdy = x.rdy && fj == 0;
    }
    return x;
  }
  // A join whose inputs several lanes complete is queued once.  Uniform call.
  __device__ __forceinline__ void claim(Reached& x) {
    const uint32_t jm = __ballot_sync(kFullMask, x.rdy && x.join);
    if (jm == 0u) return;
    if (jm & (jm - 1u)) {
      const uint32_t grp = __match_any_sync(kFullMask, x.rdy && x.join ? x.j : ~lane_id());
      if (x.join && __ffs(grp) - 1 != (int)lane_id()) x.rdy = false;
    }
    if (x.rdy && x.join) fbuf[x.j] = kQueued;
    __syncwarp();
  }
  // Op i of this lane started, ready at r and ending at f (act: the lanes that
  // started one).  Uniform call.
  __device__ __forceinline__ void record(bool v, uint32_t act, uint32_t i, tm_t r, tm_t f, const Start& s) {
    if (v) {
      fbuf[i] = f;
      if (s.flags & kReqSink) {
        const int32_t req = kHot != kHotNone ? (int32_t)op_cons(g.ops, i).z : s.req;
        atomicMax(reinterpret_cast<unsigned long long*>(creq() + req), (unsigned long long)f);
      }
      if (kMode == kBase) {
        P.base.rb[i] = r;
        P.base.fb[i] = f;
      }
      oplog[opn + __popc(act & lanes_below())] = i;
      if (s.flags & kScored) score += (int64_t)f;
      if (kMode == kInc && r >= T0) ++nev;
    }
    opn += __popc(act);
    if (kMode == kBase) {
      const int64_t lt = (int64_t)warp_max_u64(v ? (uint64_t)r : 0ull);
      last_t = lt > last_t ? lt : last_t;
      readypops += __popc(act);
    }
  }
  __device__ __forceinline__ bool count_started(int m) {
    iters += m;
    if (iters <= (int32_t)g.max_iter) return true;
    status = GMG_SIM_LOOP;
    return false;
  }

  // A batch of one op, started by lane src: its successors side by side, one per
  // lane from src on (whose place is free), instead of one after the other.  Each
  // is reached once, so none needs to be claimed.  (Graphs with little in
  // parallel start one op at a time: one request of 386 ops on 2 accelerators,
  // 4,096 placements, 634 -> 603 us; the prefill graph 3.21 -> 3.06 ms.  Where all
  // warps have room to wait the exchange costs more than it gives: the sweep warps
  // of pairs, decode 31.2 -> 31.7 ms, and the pool, wide 81.6 -> 84.5 ms, do without;
  // so do the 64-byte records, two types on 16 accelerators 3.82 -> 3.96 ms.)
  template <class B_>
  __device__ __forceinline__ void spread(B_& B, int src, uint32_t& u, uint32_t& step) const {
    B.i = __shfl_sync(kFullMask, B.i, src);
    B.d = __shfl_sync(kFullMask, B.d, src);
    B.f = __shfl_sync(kFullMask, B.f, src);
    B.s.succ_off = __shfl_sync(kFullMask, B.s.succ_off, src);
    B.s.nsucc = __shfl_sync(kFullMask, B.s.nsucc, src);
    B.s.xq = __shfl_sync(kFullMask, B.s.xq, src);
    if constexpr (kHot == kHotNone) B.s.bytes = __shfl_sync(kFullMask, B.s.bytes, src);
    u = (lane_id() - (uint32_t)src) & 31u;
    step = 32;
  }

  // ---- one pending op per lane, in registers --------------------------------
  __device__ __forceinline__ void hold_op(tm_t r, uint32_t op) {
    pd.r = r;
    pd.op = op;
    pd.d = row[op];
    if constexpr (kHot != kHotNone) pd.dur = (tm_t)hot(op).x;
    else pd.dur = (tm_t)dur_of(op, pd.d, op_durbytes(g.ops, op).x);
    pd.e = earliest(r, pd.d, pd.dur);
  }
  __device__ __forceinline__ tm_t earliest(tm_t r, int d, tm_t dur) const {
    const tm_t fd = dv.fr[d];
    return (r > fd ? r : fd) + dur;
  }
  __device__ __forceinline__ uint64_t held_key() const {
    return pd.r == kNever ? kKeyMax : rq.make(pd.r, pd.op, (tm_t)(pd.e - pd.r));
  }
  __device__ __forceinline__ bool precedes(tm_t ra, uint32_t ia, tm_t rb_, uint32_t ib_) const {
    return ra < rb_ || (ra == rb_ && ia < ib_);
  }

  // The smallest key outside the lanes, and its time (kNever: none).
  struct Outside {
    uint64_t k;
    tm_t r;
  };
  __device__ __forceinline__ void look_outside(Outside& o) const {
    o.k = outside_min();
    o.r = key_time(o.k);
  }

  // Whether this lane's pending op starts now: those before lim, the smallest
  // earliest finish (and `until`, a time that no start may pass).  Keys outside
  // the lanes that are due (rare: every root once, the heap only after the lanes
  // were all taken) come into empty lanes first.  Each lowers lim by its own bound,
  // so all that come in start now: no root waits in a lane, where it would take the
  // place of an op that the caller's queue_cap counts.
  __device__ __forceinline__ bool starts(tm_t lim, tm_t until, Outside& o) {
    if (o.r >= lim) return pd.r < lim;
    uint32_t fm = __ballot_sync(kFullMask, pd.r == kNever);
    bool fresh = false;
    while (fm && o.r < lim) {
      const int dst = __ffs(fm) - 1;
      fm &= fm - 1u;
      if ((int)lane_id() == dst) {
        pd.r = o.r;
        pd.op = rq.op(o.k);
        fresh = true;
      }
      const tm_t e = (tm_t)rq.bound(o.k);
      lim = e < lim ? e : lim;
      take_outside(o.k);
      look_outside(o);
    }
    if (fresh) hold_op(pd.r, pd.op);
    lim = warp_min_t(pd.e);
    lim = lim < until ? lim : until;
    bool act = pd.r < lim;
    if (o.r < lim) {
      // no empty lane (or a bound below the finish that it stands for): only keys
      // before the next outside one; if there is none
      // it changes places with the last key of the lanes
      act = act && precedes(pd.r, pd.op, o.r, rq.op(o.k));
      if (!__any_sync(kFullMask, act)) {
        const uint64_t mine = held_key();
        const uint64_t last = warp_max_u64(mine);
        const uint64_t x = o.k;
        take_outside(x);
        // the heap keeps one entry beyond its limit for this; in use (a successor of
        // x may have taken the lane since), the next such op finds none.  (Testing
        // for one op too many in every batch: prefill 3.25 -> 3.40 ms.)
        if (!q.push(last)) status = GMG_SIM_QUEUE;
        act = mine == last;
        if (act) hold_op((tm_t)rq.time(x), rq.op(x));
        look_outside(o);
      }
    }
    return act;
  }

  // The ops started together: this lane's (v) and the lanes' (b); ord: its place
  // among the batch's ops of its accelerator, last: the largest of these.
  struct Batch {
    bool v;
    uint32_t b, i;
    int d, ord, last;
    tm_t f;
    Start s;
  };
  // Start the lanes' ops with act; false if the iteration limit is passed.
  __device__ __forceinline__ bool start_held(bool act, Batch& B) {
    B.v = act;
    B.b = __ballot_sync(kFullMask, act);
    const int m = __popc(B.b);
    if (!count_started(m)) return false;
    B.i = pd.op;
    B.d = pd.d;
    const tm_t r = pd.r;
    B.s.nsucc = 0;
    B.s.flags = 0;
    B.f = 0;
    B.ord = B.last = 0;
    tm_t fd = 0;
    if (act) {
      B.s = start_of(B.i, B.d);
      fd = dv.fr[B.d];
    }
    // every accelerator starts its ops of the batch in key order
    bool shared = false;
    if (m > 1) {
      if constexpr (kNarrow) {
        shared = __popc(__reduce_or_sync(kFullMask, act ? 1u << B.d : 0u)) < m;
      } else {
        const uint32_t grp = __match_any_sync(kFullMask, act ? (uint32_t)B.d : 256u + lane_id());
        shared = __any_sync(kFullMask, (grp & (grp - 1u)) != 0u);
      }
    }
    if (shared) {
      int ord = 0;
      for (uint32_t o = B.b; o; o &= o - 1u) {
        const int src = __ffs(o) - 1;
        const tm_t ro = __shfl_sync(kFullMask, r, src);
        const uint32_t io = __shfl_sync(kFullMask, B.i, src);
        const int dd = __shfl_sync(kFullMask, B.d, src);
        ord += act && dd == B.d && precedes(ro, io, r, B.i) ? 1 : 0;
      }
      const int last = (int)__reduce_max_sync(kFullMask, (unsigned)ord);
      for (int t = 0; t < last; ++t) {
        if (act && ord == t) {
          B.f = earliest(r, B.d, pd.dur);
          dv.fr[B.d] = B.f;
        }
        __syncwarp();
      }
      act = act && ord == last;  // the others have theirs
      if (act) fd = dv.fr[B.d];
      B.ord = ord;
      B.last = last;
    }
    if (act) {
      B.f = (r > fd ? r : fd) + pd.dur;
      dv.fr[B.d] = B.f;
    }
    record(B.v, B.b, B.i, r, B.f, B.s);
    if (B.v) pd.r = pd.e = kNever;
    __syncwarp();
    return true;
  }

  // Ops that became ready (at most one per lane) become pending: in this lane if
  // it is empty, else in another empty one, else in the heap.
  __device__ __forceinline__ void place(Reached& x, Outside& o) {
    tm_t e = kNever;
    if (x.rdy) {
      e = earliest(x.r, x.d, x.dur);
      if (pd.r == kNever) {
        pd.r = x.r;
        pd.e = e;
        pd.dur = x.dur;
        pd.op = x.j;
        pd.d = x.d;
        x.rdy = false;
      }
    }
    uint32_t more = __ballot_sync(kFullMask, x.rdy);
    while (more) {
      const int src = __ffs(more) - 1;
      more &= more - 1u;
      const uint32_t fm = __ballot_sync(kFullMask, pd.r == kNever);
      const tm_t r = __shfl_sync(kFullMask, x.r, src), te = __shfl_sync(kFullMask, e, src),
                 dur = __shfl_sync(kFullMask, x.dur, src);
      const uint32_t j = __shfl_sync(kFullMask, x.j, src);
      const int d = __shfl_sync(kFullMask, x.d, src);
      if (fm) {
        if ((int)lane_id() == __ffs(fm) - 1) {
          pd.r = r;
          pd.e = te;
          pd.dur = dur;
          pd.op = j;
          pd.d = d;
        }
      } else {
        if (32 + q.size >= P.pend_cap || !q.push(rq.make(r, j, (tm_t)(te - r)))) status = GMG_SIM_QUEUE;
        look_outside(o);
      }
    }
  }

  __device__ void run_lanes() {
    Outside o;
    look_outside(o);
    while (true) {
      if (kMode == kBase && readypops >= next_ck) {
        const tm_t t = warp_min_t(pd.r);
        const tm_t tn = t < o.r ? t : o.r;
        if (tn != kNever) maybe_checkpoint((int64_t)tn, held_key());
      }
      const tm_t lim = warp_min_t(pd.e);
      const bool end = lim == kNever && o.r == kNever;
      if (end || opn >= P.drain_trigger) {  // the only copy of this code: it is large
        const tm_t t = warp_min_t(pd.r);
        const int64_t tn = end ? kI64Max : (int64_t)(t < o.r ? t : o.r);
        if constexpr (kRole == kBoth) drain(tn);
        else if (!end) hand_over(tn, kHandDrain, opn);
        if (end || status) break;
      }
      Batch B;
      if (!start_held(starts(lim, kNever, o), B)) break;
      uint32_t u = 0, step = 1;
      const bool one = kRole == kBoth && kCompact && (B.b & (B.b - 1u)) == 0u;
      if (one) spread(B, __ffs(B.b) - 1, u, step);
      for (; __any_sync(kFullMask, u < B.s.nsucc); u += step) {
        Reached x;
        x.rdy = x.join = false;
        x.j = 0;
        x.d = 0;
        x.r = x.dur = 0;
        if (u < B.s.nsucc) x = reach(B.i, B.d, B.f, B.s, u);
        if (!one) claim(x);
        place(x, o);
      }
      if (status) break;
    }
  }

  // ---- pending ops as keys in a pool in shared memory -------------------------

  // Slots [from, 32 * kSlots) are empty.
  __device__ void empty_pool(int from) {
    for (int x = (int)lane_id(); x < 32 * kSlots; x += 32) {
      if (x >= from) pool[x] = kKeyMax;
      fstk[x] = (uint8_t)(32 * kSlots - 1 - x);
    }
    nfree = 32 * kSlots - from;
    __syncwarp();
  }
  __device__ __forceinline__ uint64_t pool_min() const {
    uint64_t m = kKeyMax;
#pragma unroll
    for (int s = 0; s < kSlots; ++s) {
      const uint64_t k = pool[32 * s + lane_id()];
      m = k < m ? k : m;
    }
    return warp_min_u64(m);
  }
  __device__ __forceinline__ uint64_t next_key() const {
    const uint64_t m = pool_min(), x = outside_min();
    return m < x ? m : x;
  }

  // The pending ops that start now: those before lim, the smallest earliest finish
  // (and `until`, a time that no start may pass); returns their number m, and in
  // the first m lanes their keys and pool slots.
  __device__ __forceinline__ int startable(tm_t until, uint64_t& key, int& slot) {
    const unsigned lane = lane_id();
    uint64_t k[kSlots];
    tm_t lim = kNever;
#pragma unroll
    for (int s = 0; s < kSlots; ++s) {
      k[s] = pool[32 * s + lane];
      const tm_t e = k[s] == kKeyMax ? kNever : (tm_t)rq.bound(k[s]);
      lim = e < lim ? e : lim;
    }
    lim = warp_min_t(lim);
    lim = lim < until ? lim : until;
    // keys outside the pool that are due come in (rare: the roots once each,
    // the heap only after the pool was full), as far as they are among the 32 that
    // can start now: no root waits in the pool, where it would count as one of the
    // ops that the caller's queue_cap limits
    uint64_t x = outside_min();
    uint64_t kb = kKeyMax;  // keys below kb are started
    uint64_t in = 0;        // one above the last key that came in
    if (key_time(x) < lim) {
      __syncwarp();
      while (key_time(x) < lim) {
        int c = 0;  // the pool's keys before x
#pragma unroll
        for (int s = 0; s < kSlots; ++s) c += __popc(__ballot_sync(kFullMask, pool[32 * s + lane] < x));
        if (c >= 32 || (nfree == 0 && c > 0)) {
          kb = x;
          break;
        }
        int slot;
        if (nfree > 0) {
          slot = fstk[--nfree];
          take_outside(x);
        } else {
          // full, and x is the next key of all: it changes places with the pool's
          // last key
          uint64_t mx = 0;
          int ms = 0;
#pragma unroll
          for (int s = 0; s < kSlots; ++s) {
            const uint64_t y = pool[32 * s + lane];
            if (y > mx) {
              mx = y;
              ms = 32 * s + (int)lane;
            }
          }
          const uint64_t last = warp_max_u64(mx);
          slot = __shfl_sync(kFullMask, ms, __ffs(__ballot_sync(kFullMask, mx == last)) - 1);
          take_outside(x);
          if (!q.push(last)) status = GMG_SIM_QUEUE;  // (one entry beyond the heap's limit is for this)
        }
        if (lane == 0) pool[slot] = x;
        in = x + 1;
        __syncwarp();
        const tm_t e = (tm_t)rq.bound(x);
        lim = e < lim ? e : lim;
        x = outside_min();
      }
#pragma unroll
      for (int s = 0; s < kSlots; ++s) k[s] = pool[32 * s + lane];
    }
    const uint64_t lb = (uint64_t)lim << g.qsh;
    kb = lb < kb ? lb : kb;
    int m = 0;
    uint32_t b[kSlots];
#pragma unroll
    for (int s = 0; s < kSlots; ++s) {
      b[s] = __ballot_sync(kFullMask, k[s] < kb);
      m += __popc(b[s]);
    }
    if (m > 32) {
      // more keys than lanes: those up to the last that came in (32 at most), else
      // a bound with 16 to 32 keys below it (or at least one)
      uint64_t lo = in ? in : pool_min() + 1, hi = in ? in : kb;
      m = 0;
      while (m < 16 && hi - lo > 1) {
        const uint64_t mid = lo + (hi - lo) / 2;
        int c = 0;
#pragma unroll
        for (int s = 0; s < kSlots; ++s) c += __popc(__ballot_sync(kFullMask, k[s] < mid));
        if (c <= 32) {
          lo = mid;
          m = c;
        } else {
          hi = mid;
        }
      }
      m = 0;
#pragma unroll
      for (int s = 0; s < kSlots; ++s) {
        b[s] = __ballot_sync(kFullMask, k[s] < lo);
        m += __popc(b[s]);
      }
    }
    // one key per lane, through shared memory
    int at = 0;
    __syncwarp();
#pragma unroll
    for (int s = 0; s < kSlots; ++s) {
      if ((b[s] >> lane) & 1u) {
        const int pos = at + __popc(b[s] & lanes_below());
        bounce[pos] = k[s];
        reinterpret_cast<uint32_t*>(bounce + 32)[pos] = (uint32_t)(32 * s) + lane;
      }
      at += __popc(b[s]);
    }
    __syncwarp();
    key = kKeyMax;
    slot = 0;
    if ((int)lane < m) {
      key = bounce[lane];
      slot = (int)reinterpret_cast<const uint32_t*>(bounce + 32)[lane];
    }
    return m;
  }

  // The ops started together: this lane's (v), its place among the batch's ops of
  // its accelerator (ord) and the largest of these.
  struct WideBatch {
    bool v;
    uint32_t i;
    int d, ord, last;
    tm_t f;
    Start s;
  };
  // Start the batch's ops (lanes below m: a key) and record them for HBM-event
  // generation.
  __device__ __forceinline__ void start_keys(uint64_t key, int m, WideBatch& B) {
    const unsigned lane = lane_id();
    const bool v = key != kKeyMax;
    const uint32_t i = rq.op(key);
    const tm_t r = (tm_t)rq.time(key);
    int d = 0;
    tm_t f = 0;
    Start& s = B.s;
    s.nsucc = 0;
    s.flags = 0;
    s.dur = 0;
    if (v) {
      d = row[i];
      s = start_of(i, d);
    }
    // every accelerator starts its ops of the batch in key order
    int ord = 0, maxord = 0;
    if (m > 1) {
      const uint32_t grp = __match_any_sync(kFullMask, v ? (uint32_t)d : 256u + lane);
      uint32_t o = grp & ~(1u << lane);
      while (__any_sync(kFullMask, o != 0u)) {
        const uint64_t ok = __shfl_sync(kFullMask, key, o ? __ffs(o) - 1 : (int)lane);
        if (ok < key) ++ord;
        o &= o - 1u;
        maxord = 1;
      }
      if (maxord) maxord = (int)__reduce_max_sync(kFullMask, (unsigned)ord);
    }
    for (int t = 0; t <= maxord; ++t) {
      if (v && ord == t) {
        f = earliest(r, d, s.dur);
        dv.fr[d] = f;
      }
      __syncwarp();
    }
    record(v, __ballot_sync(kFullMask, v), i, r, f, s);
    __syncwarp();
    B.v = v;
    B.i = i;
    B.d = d;
    B.f = f;
    B.ord = ord;
    B.last = maxord;
  }

  // Keys of ready ops (per lane) to empty slots, or to the heap.
  __device__ __forceinline__ void spill(bool want, uint64_t nk) {
    const uint32_t more = __ballot_sync(kFullMask, want);
    if (more == 0u) return;
    const int c = __popc(more), have = nfree < c ? nfree : c;
    const int rank = __popc(more & lanes_below());
    if (want && rank < have) pool[fstk[nfree - 1 - rank]] = nk;
    nfree -= have;
    uint32_t rest = __ballot_sync(kFullMask, want && rank >= have);
    while (rest) {
      const int src = __ffs(rest) - 1;
      rest &= rest - 1;
      if (!q.push(__shfl_sync(kFullMask, nk, src))) status = GMG_SIM_QUEUE;
    }
    __syncwarp();
  }
  __device__ __forceinline__ void free_slots(bool gone, int slot) {
    const uint32_t gm = __ballot_sync(kFullMask, gone);
    if (gone) {
      pool[slot] = kKeyMax;
      fstk[nfree + __popc(gm & lanes_below())] = (uint8_t)slot;
    }
    nfree += __popc(gm);
    __syncwarp();
  }

  __device__ void run_pool() {
    while (true) {
      // counted between batches: the started ops' slots are free again, or their
      // successors'
      const int pending = 32 * kSlots - nfree + q.size;
      if (pending > P.pend_cap) {
        status = GMG_SIM_QUEUE;
        break;
      }
      if (kMode == kBase && readypops >= next_ck) {
        const uint64_t nk = next_key();
        if (nk != kKeyMax) maybe_checkpoint(rq.time(nk));
      }
      const bool end = pending == 0 && rkey == kKeyMax;
      if (end || opn >= P.drain_trigger) {  // the only copy of this code: it is large
        const int64_t tn = end ? kI64Max : rq.time(next_key());
        if constexpr (kRole == kBoth) drain(tn);
        else if (!end) hand_over(tn, kHandDrain, opn);
        if (end || status) break;
      }
      uint64_t key;
      int slot;
      const int m = startable(kNever, key, slot);
      if (!count_started(m)) break;
      start_batch(key, slot, m);
      if (status) break;
    }
  }

  // Start the batch's ops and queue the successors they make ready: a lane's
  // first takes its own slot, further ones take empty slots.
  __device__ __forceinline__ void start_batch(uint64_t key, int slot, int m) {
    WideBatch B;
    start_keys(key, m, B);
    bool kept = false;
    for (uint32_t u = 0; __any_sync(kFullMask, u < B.s.nsucc); ++u) {
      Reached x;
      x.rdy = x.join = false;
      x.j = 0;
      x.d = 0;
      x.r = x.dur = 0;
      if (u < B.s.nsucc) x = reach(B.i, B.d, B.f, B.s, u);
      claim(x);
      uint64_t nk = kKeyMax;
      if (x.rdy) {
        nk = rq.make(x.r, x.j, (tm_t)(earliest(x.r, x.d, x.dur) - x.r));
        if (!kept) {
          pool[slot] = nk;
          kept = true;
          x.rdy = false;
        }
      }
      spill(x.rdy, nk);
    }
    free_slots(B.v && !kept, slot);
  }

  __device__ void write_invalid(int64_t k, int32_t st) {
    const DevOut& o = P.out;
    const unsigned lane = lane_id();
    if (lane == 0) {
      o.makespan[k] = 0;
      o.score[k] = kI64Max;
      o.status[k] = st;
      o.viol_flag[k] = 0;
      o.viol_op[k] = -1;
      o.viol_dev[k] = -1;
      o.viol_time[k] = -1;
      o.sla_miss[k] = 0;
      o.events[k] = 0;
    }
    for (int d = lane; d < g.D; d += 32) o.peak[k * g.D + d] = 0;
    if (o.req_done)
      for (int r = lane; r < g.R; r += 32) o.req_done[k * g.R + r] = 0;
    const int ts = trace_slot(k);
    if (ts >= 0)
      for (int x = lane; x < g.n; x += 32) {
        o.trace_start[(int64_t)ts * g.n + x] = 0;
        o.trace_finish[(int64_t)ts * g.n + x] = 0;
      }
  }

  __device__ int trace_slot(int64_t k) const {
    if (P.n_trace == 0) return -1;
    int ts = -1;
    for (int t = lane_id(); t < P.n_trace; t += 32)
      if (P.trace_k[t] == k) ts = t;
    return __reduce_max_sync(kFullMask, ts);
  }

  __device__ void finish(int64_t k) {
    if (status != GMG_SIM_OK) {
      write_invalid(k, status);
      return;
    }
    const DevOut& o = P.out;
    const unsigned lane = lane_id();
    int32_t miss = 0;
    for (int r = lane; r < g.R; r += 32) {
      const int64_t c = __ldcg(creq() + r);  // raised by atomics
      miss += c > __ldg(g.deadline + r) ? 1 : 0;
      if (o.req_done) o.req_done[k * g.R + r] = c;
    }
    miss = (int32_t)__reduce_add_sync(kFullMask, (unsigned)miss);
    dv.write_peak(o.peak + k * g.D);
    // The makespan is the latest finish, i.e. the largest final free time over
    // the accelerators that ran an op (an op finishes after its accelerator's
    // initial availability).
    const int64_t mk = dv.max_busy(g);
    const int64_t sc = warp_sum_i64(score);
    const int64_t ne = kMode == kFull ? (int64_t)iters : warp_sum_i64(nev);
    if (lane == 0) {
      o.makespan[k] = mk;
      o.score[k] = vflag ? kI64Max : sc;
      o.status[k] = GMG_SIM_OK;
      o.viol_flag[k] = vflag;
      o.viol_op[k] = vop;
      o.viol_dev[k] = vdev;
      o.viol_time[k] = vt;
      o.sla_miss[k] = miss;
      o.events[k] = ne;
    }
    const int ts = trace_slot(k);
    if (ts >= 0)
      for (int x = lane; x < g.n; x += 32) {
        const int64_t fx = (int64_t)fin((uint32_t)x);
        o.trace_finish[(int64_t)ts * g.n + x] = fx;
        o.trace_start[(int64_t)ts * g.n + x] = fx - dur_of((uint32_t)x, row[x], op_durbytes(g.ops, (uint32_t)x).x);
      }
  }

  // Any placement byte >= D?  (16-byte coalesced loads of the row.)
  __device__ bool row_has_bad_device(const uint8_t* rw) const {
    if (g.D >= 256) return false;
    const unsigned lane = lane_id();
    const uint32_t dd = (uint32_t)g.D * 0x01010101u;
    bool bad = false;
    for (int c = lane * 16; c < g.n; c += 512) {
      const uint4 v = *reinterpret_cast<const uint4*>(rw + c);
      const uint32_t w[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
      for (int h = 0; h < 4; ++h) {
        uint32_t ge = __vcmpgeu4(w[h], dd);
        const int first = c + 4 * h;
        if (first + 4 > g.n) {
          const int keep = g.n - first;  // bytes of this word inside the row
          ge = keep <= 0 ? 0u : (ge & (0xffffffffu >> (8 * (4 - keep))));
        }
        bad |= ge != 0u;
      }
    }
    return __any_sync(kFullMask, bad);
  }
};

// Base-mode checkpoint: at a time boundary T_c (nothing at the next key's
// time next_t handled yet), save the complete simulator state -- accelerator state,
// READY heap, event log, partial results; the ops started by then are those
// with base ready time < T_c.  An incremental candidate whose resume time T0
// is >= T_c restarts there.  The events before T_c are applied first: what is
// left in the log is small.  (Checkpoints every few ops generate events before
// the sweep's own drain is due; without a drain of their own the log of an 8 x
// 32-layer graph, one checkpoint per 12 ops, kept every event: 24 ms for the base
// and 21 ms for a late candidate instead of 2.7 and 0.09.)
template <bool kNarrow, int kMode, bool kKey, bool kT32, bool kTypes, int kHot, bool kPool, int kRole, int kParts>
__device__ void Sim<kNarrow, kMode, kKey, kT32, kTypes, kHot, kPool, kRole, kParts>::maybe_checkpoint(int64_t tn, uint64_t held) {
  if (kMode != kBase) return;
  const DevBase& B = P.base;
  if (ck >= B.nck || readypops < next_ck) return;
  if (tn <= last_t) return;
  const unsigned lane = lane_id();
  if constexpr (kRole == kBoth) {
    generate();
    drain_log(tn);
  }
  // the pool's keys (or the keys that the lanes hold) follow the heap's
  const uint32_t hm = __ballot_sync(kFullMask, held != kKeyMax);
  const int nready = q.size + (kPool ? 32 * kSlots - nfree : __popc(hm));
  const bool keep = nready <= B.ckq;
  if (keep) {
    int64_t* sc = B.ck_scalars + (int64_t)ck * 8;
    uint64_t* qk = B.ck_qkey + (int64_t)ck * B.ckq;
    if constexpr (kPool) {
      int at = q.size;
#pragma unroll
      for (int s = 0; s < kSlots; ++s) {
        const uint64_t k = pool[32 * s + lane];
        const uint32_t b = __ballot_sync(kFullMask, k != kKeyMax);
        if (k != kKeyMax) qk[at + __popc(b & lanes_below())] = k;
        at += __popc(b);
      }
    } else if (held != kKeyMax) {
      qk[q.size + __popc(hm & lanes_below())] = held;
    }
    const int64_t total = warp_sum_i64(score);
    if (lane == 0) {
      sc[0] = nready;
      sc[1] = rootptr;
      sc[2] = total;
    }
    dv.save_free(B.ck_dev + (int64_t)ck * 3 * g.D);
    for (int r = lane; r < g.R; r += 32) B.ck_creq[(int64_t)ck * g.R + r] = __ldcg(creq() + r);
    for (int x = lane; x < q.size; x += 32) qk[x] = *q.kp(x);
  }
  if constexpr (kRole == kBoth) save_accounts(ck, tn, keep);
  else hand_over(tn, kHandCheckpoint | (keep ? kHandKeep : 0), opn);
  ++ck;
  next_ck += B.stride_pops;
  __syncwarp();
}

// The accounting's part of checkpoint c at time tn (keep: the sweep's part is
// saved): live and peak bytes, the event log, the first violation.
template <bool kNarrow, int kMode, bool kKey, bool kT32, bool kTypes, int kHot, bool kPool, int kRole, int kParts>
__device__ void Sim<kNarrow, kMode, kKey, kT32, kTypes, kHot, kPool, kRole, kParts>::save_accounts(int c, int64_t tn, bool keep) {
  const DevBase& B = P.base;
  const unsigned lane = lane_id();
  if (keep && log.n <= B.ckm) {
    int64_t* sc = B.ck_scalars + (int64_t)c * 8;
    if (lane == 0) {
      B.ck_time[c] = tn;
      sc[3] = (int64_t)drained;
      sc[4] = vflag;
      sc[5] = vt;
      sc[6] = ((int64_t)vop << 32) | (uint32_t)vdev;
      sc[7] = log.n;
    }
    dv.save_bytes(B.ck_dev + (int64_t)c * 3 * g.D);
    for (int x = lane; x < log.n; x += 32) {
      B.ck_mkey[(int64_t)c * B.ckm + x] = *log.kp(x);
      if (!kKey) B.ck_mdev[(int64_t)c * B.ckm + x] = *log.dp(x);
    }
  } else if (lane == 0) {
    B.ck_time[c] = kI64Max;
  }
  __syncwarp();
}

// Results of the base placement (after its last drain).
template <class S_>
__device__ __forceinline__ void write_base(S_& S, const DevBase& B) {
  const unsigned lane = lane_id();
  if (lane == 0) B.status[0] = S.status;
  if (S.status != GMG_SIM_OK) return;
  int32_t miss = 0;
  for (int r = lane; r < S.g.R; r += 32) {
    const int64_t c = __ldcg(S.creq() + r);
    B.res_creq[r] = c;
    miss += c > __ldg(S.g.deadline + r) ? 1 : 0;
  }
  miss = (int32_t)__reduce_add_sync(kFullMask, (unsigned)miss);
  S.dv.write_peak(B.res_peak);
  const int64_t makespan = S.dv.max_busy(S.g);
  const int64_t score = warp_sum_i64(S.score);
  if (lane == 0) {
    int64_t* rs = B.res_scalars;
    rs[0] = makespan;
    rs[1] = S.vflag ? kI64Max : score;
    rs[2] = S.vflag;
    rs[3] = S.vop;
    rs[4] = S.vdev;
    rs[5] = S.vt;
    rs[6] = miss;
  }
}

template <bool kNarrow, int kMode, bool kKey, bool kT32, bool kTypes, int kHot, bool kPool, int kRole, int kParts>
__device__ void setup_slot(Sim<kNarrow, kMode, kKey, kT32, kTypes, kHot, kPool, kRole, kParts>& S, const SimParams& P, unsigned wib,
                           int64_t slot, uint8_t* smem) {
  uint8_t* sl = P.scratch + slot * P.slot_bytes;
  const WarpSmem w = carve_smem(smem, P, wib);
  S.pool = w.pool;
  S.fstk = w.fstk;
  S.nfree = 0;
  S.q.sk = w.heap;
  S.q.sl = sl;
  S.log.sl = sl;
  S.q.size = 0;
  S.log.sk = w.logk;
  S.log.sd = w.logd;
  S.log.n = 0;
  S.sortk = w.sortk;
  S.bounce = w.sortk;
  S.sortd = w.sortd;
  S.oplog = w.oplog;
  S.opn = 0;
  using tm_t = typename Sim<kNarrow, kMode, kKey, kT32, kTypes, kHot, kPool, kRole, kParts>::tm_t;
  S.fbuf = reinterpret_cast<tm_t*>(sl + P.off_f);
  S.sl = sl;
  S.dv.setup(P.g, w.dev, P.off_pk >= 0 ? reinterpret_cast<int64_t*>(sl + P.off_pk) : nullptr);
  S.T0 = 0;
  S.Tc = 0;
  S.ck = 0;
  S.hb = 0;
  if constexpr (kRole != kBoth) {  // behind the accelerator state: the second buffer is P.opcap entries after the first
    uint8_t* c = w.dev + P.dev_bytes;
    S.hands = reinterpret_cast<Hand*>(c);
    S.oplog = reinterpret_cast<uint32_t*>(c + 2 * sizeof(Hand) + 8 * 48);
    S.bounce = reinterpret_cast<uint64_t*>(c + 2 * sizeof(Hand));
    // buffer 1 starts free
    if (kRole == kAccount) pair_arrive(3);
  }
}

// Leaving: the sweep takes the last arrival that nothing has waited for.
template <class S_>
__device__ __forceinline__ void leave_pair(S_& S) { pair_sync(2 + (S.hb ^ 1)); }

}  // namespace
}  // namespace gsim

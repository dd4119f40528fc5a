// sim_batch / sim_incremental with arbitrated transfers (Sec. 3.5.2,
// "Tensor Transfer Arbitration") for 33 to 256 accelerators.  The same
// simulation as gmgsim_arb.cu (same events, same arbitration order, same
// HBM accounting); what differs is where an accelerator's transfer state
// lives.  With more accelerators than lanes it sits in tables in shared memory
// that the lanes stride over (a = lane, lane + 32, ...): the transfer that a is
// sending, a's list of entries that have arrived but not started, and its list
// of started ops whose intents are to come (both lists linked through per-op
// arrays in the warp's scratch).  Pending READY ops are held by the lanes,
// as in the pure-latency simulation of at most 32 accelerators (every event
// looks at them, and the pool's scan is longer).
//
// The next completion and the next intent are one pass over two of the tables;
// the arbiter takes, per lane, the first entry that can start among the lane's
// accelerators, and the smallest (finish time, op) over the warp.  (With the
// tables in global scratch and a queue per accelerator pair, each event was a
// chain of L2 loads: 64 accelerators, 6,208 ops, 1,024 placements 56.6 ms -> 40.7.)
//
// The HBM-event generation and the input counting are the narrow kernel's
// (gmg_arb_events.h).  Every loop is bounded by the graph: completions by the
// number of transfers, intents by the number of ops.
#include <algorithm>

#include "gmg_arbw.h"
#include "gmg_arb_events.h"

namespace gsim {
namespace {

template <bool kT32, bool kTypes, int kHot>
struct ArbWSim : ArbEvents<ArbWSim<kT32, kTypes, kHot>, Sim<false, kFull, true, kT32, kTypes, kHot, false>> {
  using Base = ArbEvents<ArbWSim<kT32, kTypes, kHot>, Sim<false, kFull, true, kT32, kTypes, kHot, false>>;
  using tm_t = typename Base::tm_t;
  using Reached = typename Base::Reached;
  using Outside = typename Base::Outside;
  using Batch = typename Base::Batch;
  using Base::g;
  using Base::P;
  using Base::row;
  using Base::status;
  using Base::add_input;
  using Base::kNever;
  using Base::sl;
  using Base::warp_min_t;
  static constexpr int kDevBits = 8;
  const ArbWParams& A;
  // shared, per accelerator a: the transfer that a is sending (completion, kNever:
  // none; its entry), and a's list of entries (transfers) in (intent time,
  // producer, destination) order that have not started -- first and last -- and of
  // started ops whose intents are to come, in finish order: first, its finish
  // time (kNever: none), last
  tm_t* xd;
  tm_t* fu;
  uint32_t* xe;
  int32_t* eh;
  int32_t* et;
  int32_t* uh;
  int32_t* ut;
  uint32_t* rb;      // shared [8] busy receivers
  int32_t xev;       // transfer events handled (loop guard)

  __device__ ArbWSim(const ArbWParams& a) : Base(a.P), A(a) {}

  template <typename T>
  __device__ __forceinline__ T* at(int64_t off) const { return reinterpret_cast<T*>(sl + off); }
  __device__ __forceinline__ int32_t* cnt() const { return at<int32_t>(A.off_cnt); }
  __device__ __forceinline__ tm_t* rmax() const { return at<tm_t>(A.off_rmax); }
  __device__ __forceinline__ int32_t* refs() const { return at<int32_t>(A.off_refs); }
  __device__ __forceinline__ int32_t* nextop() const { return at<int32_t>(A.off_nextop); }
  // entry k of op p (k = p's successor offset + 0, 1, ...): p << 8 | destination,
  // and the next entry of its accelerator
  __device__ __forceinline__ uint32_t* xent() const { return at<uint32_t>(A.off_xent); }
  __device__ __forceinline__ int32_t* xnext() const { return at<int32_t>(A.off_xnext); }
  __device__ __forceinline__ uint32_t* lb() const { return at<uint32_t>(A.off_lb); }

  __device__ void setup_arb(uint8_t* smem_warp) {
    const int D = g.D;
    xd = reinterpret_cast<tm_t*>(smem_warp);
    fu = xd + D;
    this->dtime = fu + D;
    xe = reinterpret_cast<uint32_t*>(this->dtime + kArrivals);
    eh = reinterpret_cast<int32_t*>(xe + D);
    et = eh + D;
    uh = et + D;
    ut = uh + D;
    rb = reinterpret_cast<uint32_t*>(ut + D);
    this->dlog = rb + 8;
  }

  __device__ void reset_arb() {
    const unsigned lane = lane_id();
    const int D = g.D;
    this->reset_common();
    uint4* c4 = reinterpret_cast<uint4*>(cnt());
    const int nv = (int)((4 * (size_t)g.n + 15) / 16);
    for (int x = lane; x < nv; x += 32) c4[x] = make_uint4(0u, 0u, 0u, 0u);
    for (int a = lane; a < D; a += 32) {
      xd[a] = kNever;
      fu[a] = kNever;
      eh[a] = et[a] = uh[a] = ut[a] = -1;
    }
    if (A.shared_links)
      for (int x = lane; x < (D * D + 31) / 32; x += 32) lb()[x] = 0u;
    if (lane < 8) rb[lane] = 0u;
    this->dn = 0;
    xev = 0;
    __syncwarp();
  }

  __device__ __forceinline__ uint2 succs(uint32_t p) const {  // {offset, number}
    if constexpr (kHot != kHotNone) {
      const uint32_t z = this->hot(p).z;
      return make_uint2(z & 0xffffffu, z >> 24);
    }
    const XqSucc xs = op_xqsucc(g.ops, p);
    return make_uint2(xs.succ_off, xs.nsucc);
  }

  // The batch's ops start; local successors get this input; an op with remote
  // successors joins the end of its accelerator's list of coming ones.
  __device__ __forceinline__ void start_ops(Batch& B, Outside& o) {
    for (int t = 0; t <= B.last; ++t) {  // ops of one accelerator in turn
      const bool mine = B.v && B.ord == t;
      const uint32_t ns = mine ? B.s.nsucc : 0u;
      int rem = 0;
      for (uint32_t u = 0; __any_sync(kFullMask, u < ns); ++u) {
        Reached x;
        x.rdy = x.join = false;
        x.j = 0;
        x.d = 0;
        x.r = x.dur = 0;
        if (u < ns) {
          const uint32_t j = this->succ_at(B.s.succ_off + u);
          const int dj = row[j];
          if (dj == B.d) {
            x = add_input(j, dj, B.f);
          } else {  // a new destination?
            bool first = true;
            for (uint32_t w = 0; w < u && first; ++w) first = row[this->succ_at(B.s.succ_off + w)] != dj;
            rem += first ? 1 : 0;
          }
        }
        this->place(x, o);
      }
      if (mine) {
        refs()[B.i] = 1 + rem;
        this->holdb()[B.i] = B.f;
        if (rem) {
          if (uh[B.d] < 0) {
            uh[B.d] = (int32_t)B.i;
            fu[B.d] = B.f;
          } else {
            nextop()[ut[B.d]] = (int32_t)B.i;
          }
          ut[B.d] = (int32_t)B.i;
        }
      }
      __syncwarp();
    }
  }

  // The transfer sent by accelerator src completes at time t.
  __device__ __forceinline__ void transfer_done(int src, tm_t t, Outside& o) {
    const unsigned lane = lane_id();
    const uint32_t en = xe[src];
    const uint32_t p = en >> 8;
    const int e = (int)(en & 0xffu);
    __syncwarp();
    if (lane == 0) {
      xd[src] = kNever;
      rb[e >> 5] &= ~(1u << (e & 31));
      if (A.shared_links) {
        const uint32_t lid = __ldg(A.link + src * g.D + e);
        lb()[lid >> 5] &= ~(1u << (lid & 31u));
      }
    }
    const uint2 sc = succs(p);
    for (uint32_t c0 = 0; c0 < sc.y; c0 += 32) {
      const uint32_t u = c0 + lane;
      Reached x;
      x.rdy = x.join = false;
      x.j = 0;
      x.d = 0;
      x.r = x.dur = 0;
      if (u < sc.y) {
        const uint32_t j = this->succ_at(sc.x + u);
        if (row[j] == e) x = add_input(j, e, t);
      }
      this->place(x, o);
    }
    this->template log_arrival<kDevBits>(p, e, t);
    __syncwarp();
  }

  // The intents of accelerator a's first coming op arrive (per lane): one entry
  // per remote accelerator of its successors, in destination order, at the end of
  // a's list.
  __device__ __forceinline__ void intents_arrive(int a) {
    const uint32_t p = (uint32_t)uh[a];
    const uint2 sc = succs(p);
    int32_t tail = et[a];
    int after = -1;
    for (uint32_t k = 0;; ++k) {
      int e = 256;  // the next destination
      for (uint32_t u = 0; u < sc.y; ++u) {
        const int d = row[this->succ_at(sc.x + u)];
        if (d != a && d > after && d < e) e = d;
      }
      if (e == 256) break;
      after = e;
      const int32_t x = (int32_t)(sc.x + k);
      xent()[x] = (p << 8) | (uint32_t)e;
      if (tail >= 0) xnext()[tail] = x;
      else eh[a] = x;
      tail = x;
    }
    et[a] = tail;
    if (uh[a] == ut[a]) {
      uh[a] = ut[a] = -1;
      fu[a] = kNever;
    } else {
      const int32_t nh = nextop()[p];
      uh[a] = nh;
      fu[a] = this->fbuf[nh];
    }
  }

  // Start every pending intent whose endpoints and link are free, in (intent
  // time, producer, destination) order: every lane offers the first that can
  // start among its accelerators, a warp minimum over (finish time, op) picks the
  // next.  An offer stands until its destination (or, with shared links,
  // anything) is taken.
  __device__ __forceinline__ void arbitrate(tm_t t) {
    const unsigned lane = lane_id();
    const int D = g.D;
    const bool links = A.shared_links != 0;
    uint64_t key = kKeyMax;  // (finish time, op) offered
    int32_t ox = -1, oprev = -1;
    int oa = 0, oe = 0;
    bool scan = true;
    while (true) {
      if (scan) {
        key = kKeyMax;
        for (int a = (int)lane; a < D; a += 32) {
          if (eh[a] < 0 || xd[a] != kNever) continue;
          int32_t prev = -1;
          int32_t guard = 0;
          for (int32_t x = eh[a];; x = xnext()[x]) {
            const uint32_t en = xent()[x];
            const int e = (int)(en & 0xffu);
            bool free = !((rb[e >> 5] >> (e & 31)) & 1u);
            if (free && links) {
              const uint32_t lid = __ldg(A.link + a * D + e);
              free = !((lb()[lid >> 5] >> (lid & 31u)) & 1u);
            }
            if (free) {
              const uint64_t k = ((uint64_t)this->fin(en >> 8) << g.ib) | (en >> 8);
              if (k < key) {
                key = k;
                ox = x;
                oprev = prev;
                oa = a;
                oe = e;
              }
              break;
            }
            if (x == et[a] || ++guard > g.n_edges) break;
            prev = x;
          }
        }
      }
      const uint64_t best = warp_min_u64(key);
      if (best == kKeyMax) break;
      const int sel = __ffs(__ballot_sync(kFullMask, key == best)) - 1;
      const int src = __shfl_sync(kFullMask, oa, sel), e = __shfl_sync(kFullMask, oe, sel);
      const uint32_t p = (uint32_t)best & g.opmask;
      const tm_t done = t + this->sends(p, src, e);
      __syncwarp();
      if ((int)lane == sel) {
        xd[src] = done;
        xe[src] = (p << 8) | (uint32_t)e;
        rb[e >> 5] |= 1u << (e & 31);
        if (links) {
          const uint32_t lid = __ldg(A.link + src * D + e);
          lb()[lid >> 5] |= 1u << (lid & 31u);
        }
        // the entry leaves the list
        const bool tail = ox == et[src];
        const int32_t nx = tail ? -1 : xnext()[ox];
        if (oprev < 0) eh[src] = nx;
        else if (!tail) xnext()[oprev] = nx;
        if (tail) et[src] = oprev;
      }
      __syncwarp();
      scan = (int)lane == sel || (key != kKeyMax && (links || oe == e));
      this->log_event(lane == 0, this->kc.make(t, kAlloc, p), e);
    }
  }

  // The event loop: transfer events at a time (completions, then new intents,
  // then the arbiter), then the READY ops before the next one that the others
  // cannot delay.
  __device__ void run() {
    if (status) return;
    const unsigned lane = lane_id();
    const int D = g.D;
    const int32_t xlim = A.xcap + g.n + 2;
    Outside o;
    this->look_outside(o);
    while (true) {
      tm_t tx = kNever;
      for (int a = (int)lane; a < D; a += 32) {
        const tm_t x = xd[a], f = fu[a];
        tx = x < tx ? x : tx;
        tx = f < tx ? f : tx;
      }
      tx = warp_min_t(tx);
      tm_t lim = warp_min_t(this->pd.e);
      const bool end = lim == kNever && o.r == kNever && tx == kNever;
      if (end || this->opn >= P.drain_trigger || this->dn > kArrivals - 32) {  // the only copy of this code
        const tm_t r = warp_min_t(this->pd.r);
        tm_t tn = r < o.r ? r : o.r;
        tn = tx < tn ? tx : tn;
        this->template drain<kDevBits>(end ? kI64Max : (int64_t)tn);
        if (end || status) break;
      }
      lim = lim < tx ? lim : tx;
      const bool act = this->starts(lim, tx, o);
      if (__any_sync(kFullMask, act)) {
        Batch B;
        if (!this->start_held(act, B)) break;
        start_ops(B, o);
      } else {
        // completions first, 32 at most at a time; then everything else at tx
        int done = 0;
        bool more = false;
        for (int a0 = 0; a0 < D && !more; a0 += 32) {
          const int a = a0 + (int)lane;
          uint32_t dm = __ballot_sync(kFullMask, a < D && xd[a] == tx);
          for (; dm && !more; dm &= dm - 1u) {
            if (done == 32) {
              more = true;
            } else {
              transfer_done(a0 + __ffs(dm) - 1, tx, o);
              ++done;
            }
          }
        }
        int arrived = 0;
        if (!more) {
          for (int a = (int)lane; a < D; a += 32)
            if (fu[a] == tx) {
              intents_arrive(a);
              ++arrived;
            }
          __syncwarp();
          arbitrate(tx);
        }
        const int events = done + (int)__reduce_add_sync(kFullMask, (unsigned)arrived);
        xev += events;
        if (xev > xlim || events == 0) {
          status = GMG_SIM_LOOP;
          break;
        }
      }
      if (status) break;
    }
  }
};

// kBlocks per SM: 4 (128 registers a thread) while that holds all candidates,
// else 6 (80).  Ms on 64 accelerators, 6,208 ops, 6 blocks / 4: 1,024 placements
// 46.4 / 40.6, 2,400 52.1 / 45.7, 3,600 60.8 / 86.7.
template <bool kT32, bool kTypes, int kHot, int kBlocks>
__global__ void __launch_bounds__(128, kBlocks) sim_arbw_kernel(const __grid_constant__ ArbWParams A) {
  extern __shared__ __align__(16) uint8_t smem[];
  const unsigned wib = threadIdx.x >> 5;
  const int64_t slot = (int64_t)blockIdx.x * (blockDim.x >> 5) + wib;
  const int64_t nslots = (int64_t)gridDim.x * (blockDim.x >> 5);
  ArbWSim<kT32, kTypes, kHot> S(A);
  setup_slot(S, A.P, wib, slot, smem);
  S.setup_arb(smem + A.smem_std + (size_t)wib * A.smem_arb);
  for (int64_t k = slot; k < A.P.K; k += nslots) {
    S.row = A.P.place + k * A.P.ld;
    if (A.pre_status) {
      const int32_t st = A.pre_status[k];
      if (st != GMG_SIM_OK) {
        S.write_invalid(k, st);
        continue;
      }
    }
    if (S.row_has_bad_device(S.row)) {
      S.write_invalid(k, GMG_SIM_BADDEV);
      continue;
    }
    S.reset_arb();
    S.run();
    S.finish(k);
  }
}

}  // namespace

// Instances by (32-bit times, accelerator types; compact records wherever the
// graph has them).
template <int kBlocks>
const void* arbw_ptr(const DevGmg& g) {
  if (g.hot_ok) return (const void*)sim_arbw_kernel<true, false, kHotGlobal, kBlocks>;
  if (g.t32)
    return g.ntypes >= 2 ? (const void*)sim_arbw_kernel<true, true, kHotNone, kBlocks>
                         : (const void*)sim_arbw_kernel<true, false, kHotNone, kBlocks>;
  return g.ntypes >= 2 ? (const void*)sim_arbw_kernel<false, true, kHotNone, kBlocks>
                       : (const void*)sim_arbw_kernel<false, false, kHotNone, kBlocks>;
}
const void* arbw_kernel_ptr(const DevGmg& g, bool few) { return few ? arbw_ptr<4>(g) : arbw_ptr<6>(g); }

// Every instance may ask for the shared memory that the device has.
cudaError_t set_arbw_smem_limit() {
  int dev = 0, optin = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
  DevGmg g{};
  for (int c = 0; c < 16 && e == cudaSuccess; ++c) {
    g.hot_ok = c & 1;
    g.t32 = (c >> 1) & 1;
    g.ntypes = c & 4 ? 2 : 0;
    e = cudaFuncSetAttribute(arbw_kernel_ptr(g, (c & 8) != 0), cudaFuncAttributeMaxDynamicSharedMemorySize, optin);
  }
  return e;
}

cudaError_t launch_arbw(const ArbWParams& A, int grid, int block, size_t smem, cudaStream_t st) {
  void* args[] = {const_cast<ArbWParams*>(&A)};
  return cudaLaunchKernel(arbw_kernel_ptr(A.P.g, A.few != 0), dim3(grid), dim3(block), args, smem, st);
}

}  // namespace gsim

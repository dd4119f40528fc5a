// Parts shared by the two arbitrated-transfer simulators (gmgsim_arb.cu, at
// most 32 accelerators with transfer state in lane registers; gmgsim_arbw.cu,
// 33 to 256 accelerators with it in per-warp tables): counting an op's inputs
// as they arrive, the holds on a producer's own copy, and the HBM events of
// the ops started since the last generation (Sec. 3.5.2: a receive buffer is
// allocated when its transfer starts, a producer's copy is released once its
// last local consumer has finished and every outgoing transfer has arrived).
//
// ArbEvents<Self, SimBase> sits between the pure-latency simulator SimBase and
// the kernel's own simulator Self, which provides the per-op scratch arrays
// cnt() (inputs present), rmax() (latest arrival so far) and refs() (holds
// left on the op's own copy).
#pragma once

#include "gmgsim_sim.cuh"

namespace gsim {
namespace {

constexpr int kArrivals = kArbArrivals;

template <class Self, class SimBase>
struct ArbEvents : SimBase {
  using tm_t = typename SimBase::tm_t;
  __device__ explicit ArbEvents(const SimParams& p) : SimBase(p) {}
  __device__ __forceinline__ const Self& self() const { return *static_cast<const Self*>(this); }

  // One more input of op j (on accelerator d) present at time a (per lane);
  // ready if it was the last.
  __device__ __forceinline__ typename SimBase::Reached add_input(uint32_t j, int d, tm_t a) const {
    typename SimBase::Reached x;
    x.j = j;
    x.d = d;
    x.join = false;
    int32_t* cp = self().cnt() + j;
    tm_t* mp = self().rmax() + j;
    uint32_t npred;
    if constexpr (SimBase::kCompact) {
      const uint4 h = this->hot(j);
      x.dur = (tm_t)h.x;
      npred = h.w >> 24;
      x.r = (tm_t)__ldg(this->g.st_rel + j);
    } else {
      const RelPred jp = op_relpred(this->g.ops, j);
      x.dur = (tm_t)this->dur_of(j, d, op_durbytes(this->g.ops, j).x);
      npred = jp.npred;
      x.r = (tm_t)jp.rel;
    }
    tm_t m = a;
    x.rdy = npred == 1u;
    if (npred > 1u) {
      const int32_t c = *cp + 1;
      const tm_t o = *mp;
      m = c > 1 && o > a ? o : a;
      *cp = c;
      *mp = m;
      x.rdy = (uint32_t)c == npred;
    }
    x.r = x.r > m ? x.r : m;
    return x;
  }

  // One hold on op p's own copy ends at time v (per lane); true if it was the
  // last: the copy is then released at h.
  __device__ __forceinline__ bool drop_hold(uint32_t p, tm_t v, tm_t& h) {
    int32_t* rp = self().refs() + p;
    const tm_t o = this->holdb()[p];
    const int32_t left = *rp - 1;
    *rp = left;
    h = o > v ? o : v;
    this->holdb()[p] = h;
    return left == 0;
  }

  // HBM events of the ops started since the last generation, one op per
  // lane: the own copy allocated at s; the op's local hold on its own copy
  // ends at f if no listed consumer is local; every held input whose last
  // local listed consumer this op is gets released at f (a receive copy) or
  // loses its local hold (the producer's own copy).  One op ends the local hold
  // on a copy, so no two lanes touch the same one.  Loads side by side as in the
  // pure-latency simulation.
  __device__ __forceinline__ void generate() {
    const unsigned lane = lane_id();
    for (int c0 = 0; c0 < this->opn; c0 += 32) {
      const int idx = c0 + (int)lane;
      const bool v = idx < this->opn;
      const uint32_t x = v ? this->oplog[idx] : 0u;
      typename SimBase::Start s;
      s.nsucc = 0;
      s.flags = kAllCons;
      s.dur = 0;
      s.succ_off = 0;
      uint32_t pred_off = 0, npred = 0;
      int d = 0;
      tm_t f = 0;
      if (v) {
        d = this->row[x];
        f = this->fbuf[x];
        if constexpr (SimBase::kCompact) {
          const uint4 h = this->hot(x);
          s.dur = (tm_t)h.x;
          s.flags = h.y >> 29;
          s.succ_off = h.z & 0xffffffu;
          s.nsucc = h.z >> 24;
          pred_off = h.w & 0xffffffu;
          npred = h.w >> 24;
        } else {
          s = this->start_of(x, d);
          const RelPred rp = op_relpred(this->g.ops, x);
          pred_off = rp.pred_off;
          npred = rp.npred;
        }
      }
      bool localc = false;
      uint2 ps[2] = {make_uint2(0u, 0u), make_uint2(0u, 0u)};
#pragma unroll
      for (int u = 0; u < 2; ++u) {
        if ((uint32_t)u < npred) ps[u] = __ldg(this->g.predsib + pred_off + u);
        if ((uint32_t)u < s.nsucc) localc = localc || this->row[this->succ_at(s.succ_off + u)] == d;
      }
      if (!(s.flags & kAllCons)) {
        localc = this->consumer_on(op_cons(this->g.ops, x), d);
      } else {
        for (uint32_t u = 2; u < s.nsucc && !localc; ++u) localc = this->row[this->succ_at(s.succ_off + u)] == d;
      }
      uint64_t ev[4];
      int dev[4] = {d, d, d, d};
      uint32_t want = v ? 1u : 0u;
      ev[0] = this->entry(f - s.dur, kAlloc, x, d);
      tm_t h = f;
      if (v && !localc && drop_hold(x, f, h)) want |= 2u;
      ev[1] = this->entry(h, kFree, x, d);
#pragma unroll
      for (int u = 0; u < 2; ++u) {
        const uint32_t p = ps[u].x & kIdMask;
        tm_t t = f;
        if (this->releases(x, d, f, ps[u]) && (this->row[p] != d || drop_hold(p, f, t))) want |= 4u << u;
        ev[2 + u] = this->entry(t, kFree, p, d);
      }
      this->template log_lanes<4>(ev, dev, want);
      if (__any_sync(kFullMask, npred > 2u)) {
        const uint32_t maxp = __reduce_max_sync(kFullMask, npred);
        for (uint32_t u = 2; u < maxp; ++u) {
          bool rel = false;
          tm_t t = f;
          uint32_t p = 0;
          if (u < npred) {
            const uint2 e = __ldg(this->g.predsib + pred_off + u);
            p = e.x & kIdMask;
            rel = this->releases(x, d, f, e) && (this->row[p] != d || drop_hold(p, f, t));
          }
          this->log_event(rel, this->kc.make(t, kFree, p), d);
        }
      }
    }
    this->opn = 0;
    __syncwarp();
  }

  // Transfers that arrived since the last generation wait in a list (dlog: the
  // producer and the destination; dtime; drained before it has no room for 32 more),
  // so that what they end is looked up for
  // all of them at once, one per lane: one hold on the sender's copy; the receive
  // copy is released on arrival if no listed consumer is there.
  uint32_t* dlog;  // shared [kArrivals]
  tm_t* dtime;     // shared [kArrivals]
  int dn;
  template <int kDevBits>
  __device__ __forceinline__ void log_arrival(uint32_t p, int e, tm_t t) {
    if (lane_id() == 0) {
      dlog[dn] = (p << kDevBits) | (uint32_t)e;
      dtime[dn] = t;
    }
    ++dn;
  }
  template <int kDevBits>
  __device__ __forceinline__ void arrivals() {
    const unsigned lane = lane_id();
    __syncwarp();
    for (int c0 = 0; c0 < dn; c0 += 32) {
      const int idx = c0 + (int)lane;
      const bool v = idx < dn;
      const uint32_t x = v ? dlog[idx] : 0u;
      const uint32_t p = x >> kDevBits;
      const int e = (int)(x & ((1u << kDevBits) - 1u));
      const tm_t t = v ? dtime[idx] : 0;
      const uint4 cs = v ? op_cons(this->g.ops, p) : make_uint4(0u, 0u, 0u, kAllCons);
      const int dp = v ? this->row[p] : 0;
      uint32_t want = v && !(cs.w & kAllCons) && !this->consumer_on(cs, e) ? 1u : 0u;
      // transfers of one producer one after the other
      const uint32_t grp = __match_any_sync(kFullMask, v ? p : ~lane);
      const int ord = __popc(grp & lanes_below());
      const int last = (int)__reduce_max_sync(kFullMask, (unsigned)ord);
      tm_t h = 0;
      for (int r = 0; r <= last; ++r) {
        if (v && ord == r && drop_hold(p, t, h)) want |= 2u;
        __syncwarp();
      }
      const uint64_t ev[2] = {this->entry(t, kFree, p, e), this->entry(h, kFree, p, dp)};
      const int dev[2] = {e, dp};
      this->template log_lanes<2>(ev, dev, want);
    }
    dn = 0;
    __syncwarp();
  }

  template <int kDevBits>
  __device__ __forceinline__ void drain(int64_t t_next) {
    generate();
    arrivals<kDevBits>();
    this->drain_log(t_next);
  }
};

}  // namespace
}  // namespace gsim

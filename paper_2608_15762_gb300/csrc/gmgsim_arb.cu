// sim_batch with arbitrated transfers (Sec. 3.5.2, "Tensor Transfer
// Arbitration"): one warp per candidate, as in the pure-latency simulation,
// with two more kinds of event.
//
//   INTENT(f_p, p)     producer p finished; its output is wanted on every
//                      distinct remote accelerator e of p's successors: one
//                      intent per e joins the FIFO queue of the pair (dev p, e).
//   DONE(c, p, e)      the transfer arrived: the sender's endpoint, e's
//                      receiving endpoint and the pair's link are free again;
//                      p's successors on e have one more input present.
//
// Lane a keeps accelerator a's side of both.  An accelerator sends one transfer
// at a time, so lane a holds the completion time of the transfer it is sending,
// if any.  Its ops finish in the order they start, so those with remote
// successors form one list in finish order, linked through a per-op array: first
// the ops whose intents have arrived and are not all on their way, then those
// whose intents are to come.  The next DONE and the next INTENT are warp minima
// over the lanes.
//
// After the last INTENT / DONE of a time t the arbiter starts, in (intent time,
// producer, destination) order, every pending intent whose sending endpoint,
// receiving endpoint and link are all free (the communication graph of Sec.
// 3.5.2; the selection rule among conflicting intents is this FIFO greedy
// one).  An intent's time is its producer's finish time, so lane a's first list
// entry with a destination that it can send to is its earliest, and a warp
// minimum over (finish time, op) picks the next.  A started transfer allocates
// its receive buffer and lasts the transfer estimate.  When no two ordered pairs
// share a link id, a busy link implies a busy sender and the link state is not
// kept.
//
// What bounds the kernel is the chain of dependent steps and loads per event, one
// event time after the other.  So READY ops start many at a time, as in the
// pure-latency simulation, and stop at the next event; an entry is a producer and
// a bit mask of its destinations, not a record per intent in a queue per pair; an
// arrival's consumer lookups, needed for HBM accounting only, wait and are done
// for a warp of arrivals side by side.  Prefill graph, 8 accelerators, 2,048
// placements: 15.3 ms -> 9.6.
//
// Readiness: an op's inputs are counted as they become present -- a local
// predecessor's output when that predecessor starts (its finish time is then
// known), a remote one when its transfer is DONE -- and the op becomes READY
// at the latest arrival once all are there.  Transfer events at a time are
// handled before READY keys at that time (a DONE can make an op ready then).
//
// HBM events: an op's own copy is released once two holds are gone -- its
// last local listed consumer has finished (or the op itself, if none) and
// every outgoing transfer has arrived -- at the later of those times; a
// receive copy is allocated when its transfer starts and released by its last
// listed consumer there (or on arrival if none).  Every such event is logged
// at a time no earlier than the sweep's, so the batched drain of the
// pure-latency simulation applies unchanged.
//
// Requires at most 32 accelerators (endpoint sets are warp bit masks) and an
// accelerator id that fits beside the packed key.  Every loop is bounded by
// the graph: DONEs by the number of transfers, INTENTs by the number of ops.
#include <algorithm>

#include "gmg_arb.h"
#include "gmg_arb_events.h"

namespace gsim {
namespace {

// kMode: kFull (sim_batch), kBase (the arbitrated base snapshot: records
// ready and finish times and checkpoints), kInc (candidates resumed from it).
template <bool kT32, bool kTypes, int kMode = kFull, int kHot = kHotNone>
struct ArbSim : ArbEvents<ArbSim<kT32, kTypes, kMode, kHot>, Sim<true, kMode, true, kT32, kTypes, kHot>> {
  using Base = ArbEvents<ArbSim<kT32, kTypes, kMode, kHot>, Sim<true, kMode, true, kT32, kTypes, kHot>>;
  using tm_t = typename Base::tm_t;
  using Reached = typename Base::Reached;
  using Outside = typename Base::Outside;
  using Batch = typename Base::Batch;
  using Base::g;
  using Base::P;
  using Base::pd;
  using Base::row;
  using Base::status;
  using Base::add_input;
  using Base::arrivals;
  using Base::generate;
  using Base::kNever;
  using Base::place;
  using Base::sl;
  using Base::warp_min_t;
  static constexpr int kDevBits = 5;
  const ArbParams& A;
  // The warp's shared area: busy links (32 words), then the arrivals waiting for
  // the next generation (gmg_arb_events.h).
  uint8_t* sm;
  int32_t xev;     // transfer events handled (loop guard)
  uint32_t recvm;  // accelerators whose receiving endpoint is busy
  // lane a: accelerator a's side of the transfers
  tm_t xd;         // completion of the transfer a is sending (kNever: none)
  uint32_t xdp;    // its producer << 5 | its destination
  // a's started ops with remote successors that are not all on their way yet, in
  // finish order (linked through nextop): those whose intents have arrived from
  // ah to al, the coming ones from uh to lt (-1: none; lt is the last of both)
  int32_t ah, uh;
  tm_t fu;         // finish time of uh (kNever: none)
  // (al, lt, the destinations left of ah and its finish time, used on changes
  // only, are the lane's words in the shared area: registers are scarce)
  __device__ __forceinline__ int32_t& al() const { return reinterpret_cast<int32_t*>(sm + 128)[lane_id()]; }
  __device__ __forceinline__ int32_t& lt() const { return reinterpret_cast<int32_t*>(sm + 256)[lane_id()]; }
  __device__ __forceinline__ uint32_t& hm() const { return reinterpret_cast<uint32_t*>(sm + 384)[lane_id()]; }
  __device__ __forceinline__ tm_t& hf() const { return reinterpret_cast<tm_t*>(sm + 512)[lane_id()]; }

  __device__ ArbSim(const ArbParams& a) : Base(a.P), A(a) {}

  template <typename T>
  __device__ __forceinline__ T* at(int64_t off) const { return reinterpret_cast<T*>(sl + off); }
  __device__ __forceinline__ int32_t* cnt() const { return at<int32_t>(A.off_cnt); }      // [N] inputs present (joins)
  __device__ __forceinline__ tm_t* rmax() const { return at<tm_t>(A.off_rmax); }          // [N] latest arrival
  __device__ __forceinline__ int32_t* refs() const { return at<int32_t>(A.off_refs); }    // [N] holds left
  __device__ __forceinline__ uint32_t* rmask() const { return at<uint32_t>(A.off_rmask); }  // [N] destinations left
  __device__ __forceinline__ int32_t* nextop() const { return at<int32_t>(A.off_nextop); }  // [N] list link
  __device__ __forceinline__ uint32_t* lbits() const { return reinterpret_cast<uint32_t*>(sm); }

  __device__ void setup_arb(uint8_t* smem_warp) {
    sm = smem_warp;
    this->dtime = reinterpret_cast<tm_t*>(sm + 768);
    this->dlog = reinterpret_cast<uint32_t*>(sm + 768 + 8 * kArrivals);
  }

  __device__ void reset_arb() {
    const unsigned lane = lane_id();
    this->reset_common();
    uint4* c4 = reinterpret_cast<uint4*>(cnt());
    const int nv = (int)((4 * (size_t)g.n + 15) / 16);
    for (int x = lane; x < nv; x += 32) c4[x] = make_uint4(0u, 0u, 0u, 0u);
    lbits()[lane] = 0u;
    this->dn = 0;
    xev = 0;
    recvm = 0u;
    xd = kNever;
    xdp = 0u;
    ah = uh = -1;
    al() = lt() = -1;
    fu = kNever;
    __syncwarp();
  }

  // Lane a: op p, ending at f, joins the end of a's list.
  __device__ __forceinline__ void append(uint32_t p, tm_t f) {
    if (lt() >= 0) nextop()[lt()] = (int32_t)p;
    if (uh < 0) {
      uh = (int32_t)p;
      fu = f;
    }
    lt() = (int32_t)p;
  }

  // READY ops: start them; local successors get this input; an op with remote
  // successors joins its accelerator's list.
  __device__ __forceinline__ void start_ops(Batch& B, Outside& o) {
    const unsigned lane = lane_id();
    uint32_t remote = 0u;
    // ops of one accelerator (which may feed one local successor) in turn
    for (int t = 0; t <= B.last; ++t) {
      const uint32_t ns = B.ord == t ? B.s.nsucc : 0u;
      for (uint32_t u = 0; __any_sync(kFullMask, u < ns); ++u) {
        Reached x;
        x.rdy = x.join = false;
        x.j = 0;
        x.d = 0;
        x.r = x.dur = 0;
        if (u < ns) {
          const uint32_t j = this->succ_at(B.s.succ_off + u);
          const int dj = row[j];
          if (dj == B.d) x = add_input(j, dj, B.f);
          else remote |= 1u << dj;
        }
        place(x, o);
      }
      __syncwarp();
    }
    if (B.v) {
      refs()[B.i] = 1 + __popc(remote);
      this->holdb()[B.i] = B.f;
      if (remote) rmask()[B.i] = remote;
    }
    const uint32_t rem = __ballot_sync(kFullMask, B.v && remote);
    for (int t = 0; t <= B.last; ++t)
      for (uint32_t m = B.last ? __ballot_sync(kFullMask, ((rem >> lane) & 1u) && B.ord == t) : rem; m; m &= m - 1u) {
        const int src = __ffs(m) - 1;
        const uint32_t p = __shfl_sync(kFullMask, B.i, src);
        const tm_t f = __shfl_sync(kFullMask, B.f, src);
        if ((int)lane == __shfl_sync(kFullMask, B.d, src)) append(p, f);
      }
    __syncwarp();
  }

  // The transfer sent by lane src completes at time t.
  __device__ __forceinline__ void transfer_done(int src, tm_t t, Outside& o) {
    const unsigned lane = lane_id();
    const uint32_t pe = __shfl_sync(kFullMask, xdp, src);
    const uint32_t p = pe >> kDevBits;
    const int e = (int)(pe & 31u);
    if ((int)lane == src) xd = kNever;
    recvm &= ~(1u << e);
    if (A.shared_links) {
      const uint32_t lid = __ldg(A.link + src * g.D + e);
      if (lane == 0) lbits()[lid >> 5] &= ~(1u << (lid & 31u));
      __syncwarp();
    }
    // p's successors on e have this input now
    uint32_t off, ns;
    if constexpr (kHot != kHotNone) {
      const uint4 h = this->hot(p);
      off = h.z & 0xffffffu;
      ns = h.z >> 24;
    } else {
      const XqSucc xs = op_xqsucc(g.ops, p);
      off = xs.succ_off;
      ns = xs.nsucc;
    }
    for (uint32_t c0 = 0; c0 < ns; c0 += 32) {
      const uint32_t u = c0 + lane;
      Reached x;
      x.rdy = x.join = false;
      x.j = 0;
      x.d = 0;
      x.r = x.dur = 0;
      if (u < ns) {
        const uint32_t j = this->succ_at(off + u);
        if (row[j] == e) x = add_input(j, e, t);
      }
      place(x, o);
    }
    __syncwarp();
    this->template log_arrival<kDevBits>(p, e, t);
  }

  // Start every pending intent whose endpoints and link are free, in (intent
  // time, producer, destination) order: each free accelerator offers the first
  // destination that it can send to of the first op in its list that has one, and
  // a warp minimum over (finish time, op) picks the next to start.  An offer
  // stands until its destination (or, with shared links, anything) is taken.
  __device__ __forceinline__ void arbitrate(tm_t t) {
    const int lane = (int)lane_id();
    const int D = g.D;
    const bool links = A.shared_links != 0;
    int32_t cp = -1, prev = -1;  // the op offered, the one before it in the list
    uint32_t cm = 0u;            // its destinations left
    tm_t cf = kNever;
    int ce = 0;
    bool scan = xd == kNever && ah >= 0;
    while (true) {
      if (scan) {
        cp = ah;
        cm = hm();
        cf = hf();
        prev = -1;
        for (int32_t guard = 0;; ++guard) {
          uint32_t c = cm & ~recvm;
          if (links) {
            uint32_t ok = 0u;
            while (c) {
              const int e = __ffs(c) - 1;
              c &= c - 1u;
              const uint32_t lid = __ldg(A.link + lane * D + e);
              if (!((lbits()[lid >> 5] >> (lid & 31u)) & 1u)) {
                ok = 1u << e;
                break;
              }
            }
            c = ok;
          }
          if (c) {
            ce = __ffs(c) - 1;
            break;
          }
          if (cp == al() || guard > g.n) {
            cp = -1;
            break;
          }
          prev = cp;
          cp = nextop()[cp];
          cm = rmask()[cp];
          cf = this->fin((uint32_t)cp);
        }
      }
      const uint64_t key = cp >= 0 ? ((uint64_t)cf << g.ib) | (uint32_t)cp : kKeyMax;
      const uint64_t best = warp_min_u64(key);
      if (best == kKeyMax) break;
      const int src = __ffs(__ballot_sync(kFullMask, key == best)) - 1;
      const int e = __shfl_sync(kFullMask, ce, src);
      const uint32_t p = (uint32_t)best & g.opmask;
      const tm_t done = t + this->sends(p, src, e);
      recvm |= 1u << e;
      if (links) {
        const uint32_t lid = __ldg(A.link + src * D + e);
        if (lane == 0) lbits()[lid >> 5] |= 1u << (lid & 31u);
        __syncwarp();
      }
      if (lane == src) {
        xd = done;
        xdp = (p << kDevBits) | (uint32_t)e;
        const uint32_t left = cm & ~(1u << e);
        if (left) {
          rmask()[p] = left;
          if (cp == ah) hm() = left;
        } else {  // leaves the list
          const bool tail = cp == lt();
          const int32_t nx = tail ? -1 : nextop()[cp];
          if (cp == ah) {
            ah = cp == al() ? -1 : nx;
            if (ah >= 0) {
              hm() = rmask()[ah];
              hf() = this->fin((uint32_t)ah);
            } else {
              al() = -1;
            }
          } else {
            if (!tail) nextop()[prev] = nx;
            if (cp == al()) al() = prev;
          }
          if (tail) lt() = prev;
        }
      }
      scan = cp >= 0 && lane != src && (links || ce == e);
      if (lane == src) cp = -1;
      __syncwarp();
      this->log_event(lane == 0, this->kc.make(t, kAlloc, p), e);
    }
  }

  // The event loop: transfer events at a time (completions, then new intents,
  // then the arbiter), then the READY ops before the next one that the others
  // cannot delay.
  __device__ void run() {
    if (status) return;
    const unsigned lane = lane_id();
    const int32_t xlim = A.xcap + g.n + 2;
    Outside o;
    this->look_outside(o);
    while (true) {
      const tm_t td = warp_min_t(xd), ti = warp_min_t(fu);
      const tm_t tx = td < ti ? td : ti;
      tm_t lim = warp_min_t(pd.e);
      const bool end = lim == kNever && o.r == kNever && tx == kNever;
      // (at most 32 transfers complete at one time)
      if (end || this->opn >= P.drain_trigger || this->dn > kArrivals - 32) {  // the only copy of this code
        const tm_t r = warp_min_t(pd.r);
        tm_t tn = r < o.r ? r : o.r;
        tn = tx < tn ? tx : tn;
        this->template drain<kDevBits>(end ? kI64Max : (int64_t)tn);
        if (end || status) break;
      }
      lim = lim < tx ? lim : tx;
      if (kMode == kBase && this->readypops >= this->next_ck) {
        // READY ops start now (the next comes before every transfer event)
        const tm_t r = warp_min_t(pd.r);
        if ((r < o.r ? r : o.r) < tx) arb_checkpoint(o);
      }
      const bool act = this->starts(lim, tx, o);
      if (__any_sync(kFullMask, act)) {
        Batch B;
        if (!this->start_held(act, B)) break;
        start_ops(B, o);
      } else {
        uint32_t dm = __ballot_sync(kFullMask, xd == tx);
        const bool arrives = fu == tx;
        const int events = __popc(dm) + __popc(__ballot_sync(kFullMask, arrives));
        xev += events;
        if (xev > xlim || events == 0) {
          status = GMG_SIM_LOOP;
          break;
        }
        for (; dm; dm &= dm - 1u) transfer_done(__ffs(dm) - 1, tx, o);
        if (arrives) {
          if (ah < 0) {
            ah = uh;
            hm() = rmask()[uh];
            hf() = tx;
          }
          al() = uh;
          uh = uh == lt() ? -1 : nextop()[uh];
          fu = uh < 0 ? kNever : this->fin((uint32_t)uh);
        }
        arbitrate(tx);
        if (kMode == kBase) this->last_t = (int64_t)tx;
      }
      if (status) break;
    }
  }

  // -------------------------------------------------------------------------
  // Arbitrated base snapshot.  A checkpoint is taken right before READY ops
  // whose smallest time T_c is past every event handled so far: every transfer
  // event and arbitration before T_c is done (transfer events at a time come
  // before READY ops at that time), nothing at T_c or later is.  The simulation
  // part is the base snapshot's (Sim::maybe_checkpoint, after this simulator's
  // own event generation); the arbiter's part goes to the checkpoint's arena.
  // -------------------------------------------------------------------------
  __device__ void arb_checkpoint(const Outside& o) {
    const DevBase& B = P.base;
    if (this->ck >= B.nck || this->readypops < this->next_ck) return;
    const tm_t r = warp_min_t(pd.r);
    const tm_t tn = r < o.r ? r : o.r;
    if ((int64_t)tn <= this->last_t) return;
    generate();  // the simulation checkpoint then finds no started op left to generate
    this->template arrivals<kDevBits>();
    this->drain_log((int64_t)tn);
    const int c = this->ck;
    this->maybe_checkpoint((int64_t)tn, this->held_key());
    if (this->ck > c && B.ck_time[c] != kI64Max) save_arb(c);
  }

  __device__ uint8_t* arena(int c) const { return A.ck.arena + (int64_t)c * A.ck.bytes; }

  // The base runs with 64-bit times, so every per-op array has the arena's
  // element size and is copied as bytes (each region of the slot and of the
  // arena is padded to 256 bytes).
  __device__ void save_arb(int c) {
    static_assert(kMode != kBase || !kT32, "the base snapshot keeps 64-bit times");
    const unsigned lane = lane_id();
    uint8_t* a = arena(c);
    const ArbCk& K = A.ck;
    const int64_t n = g.n;
    warp_copy16<16>(a + K.off_cnt, cnt(), 4 * n);
    warp_copy16<16>(a + K.off_rmax, rmax(), 8 * n);
    warp_copy16<16>(a + K.off_refs, refs(), 4 * n);
    warp_copy16<16>(a + K.off_rmask, rmask(), 4 * n);
    warp_copy16<16>(a + K.off_nextop, nextop(), 4 * n);
    warp_copy16<16>(a + K.off_hold, this->holdb(), 8 * n);
    int64_t* ls = reinterpret_cast<int64_t*>(a + K.off_lanes) + 7 * lane;
    ls[0] = (int64_t)xd;
    ls[1] = xdp;
    ls[2] = ah;
    ls[3] = al();
    ls[4] = uh;
    ls[5] = lt();
    ls[6] = (int64_t)fu;
    int64_t* w = reinterpret_cast<int64_t*>(a + K.off_warp);
    if (lane == 0) {
      w[0] = xev;
      w[1] = recvm;
    }
    reinterpret_cast<uint32_t*>(w + 2)[lane] = lbits()[lane];
    __syncwarp();
  }

  // A base time (int64) in this kernel's time type; the base's "never" maps
  // to this kernel's.
  static __device__ __forceinline__ tm_t narrow_time(int64_t v) {
    return v >= (int64_t)kNever ? kNever : (tm_t)v;
  }

  // An arena's 64-bit times into this kernel's time type, four loads in
  // flight per lane.
  static __device__ void narrow_times(tm_t* dst, const int64_t* src, int n) {
    int x = (int)lane_id();
    for (; x + 96 < n; x += 128) {
      const int64_t a = src[x], b = src[x + 32], c = src[x + 64], e = src[x + 96];
      dst[x] = narrow_time(a);
      dst[x + 32] = narrow_time(b);
      dst[x + 64] = narrow_time(c);
      dst[x + 96] = narrow_time(e);
    }
    for (; x < n; x += 32) dst[x] = narrow_time(src[x]);
  }

  __device__ void restore_arb(int c) {
    const unsigned lane = lane_id();
    const uint8_t* a = arena(c);
    const ArbCk& K = A.ck;
    const int64_t n = g.n;
    warp_copy16(cnt(), a + K.off_cnt, 4 * n);
    warp_copy16(refs(), a + K.off_refs, 4 * n);
    warp_copy16(rmask(), a + K.off_rmask, 4 * n);
    warp_copy16(nextop(), a + K.off_nextop, 4 * n);
    if (kT32) {
      narrow_times(rmax(), reinterpret_cast<const int64_t*>(a + K.off_rmax), g.n);
      narrow_times(this->holdb(), reinterpret_cast<const int64_t*>(a + K.off_hold), g.n);
    } else {
      warp_copy16(rmax(), a + K.off_rmax, 8 * n);
      warp_copy16(this->holdb(), a + K.off_hold, 8 * n);
    }
    const int64_t* w = reinterpret_cast<const int64_t*>(a + K.off_warp);
    xev = (int32_t)w[0];
    recvm = (uint32_t)w[1];
    lbits()[lane] = reinterpret_cast<const uint32_t*>(w + 2)[lane];
    const int64_t* ls = reinterpret_cast<const int64_t*>(a + K.off_lanes) + 7 * lane;
    xd = narrow_time(ls[0]);
    xdp = (uint32_t)ls[1];
    ah = (int32_t)ls[2];
    al() = (int32_t)ls[3];
    uh = (int32_t)ls[4];
    lt() = (int32_t)ls[5];
    fu = narrow_time(ls[6]);
    this->dn = 0;
    __syncwarp();
    // an op whose intents have arrived finished before T0: the moves change
    // nothing about it
    hm() = ah >= 0 ? rmask()[ah] : 0u;
    hf() = ah >= 0 ? this->fin((uint32_t)ah) : kNever;
  }

  // Remote accelerators of p's successors under placement rw (uniform).
  __device__ uint32_t remote_set(uint32_t p, const uint8_t* rw) const {
    const XqSucc xs = op_xqsucc(g.ops, p);
    const int dp = rw[p];
    uint32_t m = 0u;
    for (uint32_t u = lane_id(); u < xs.nsucc; u += 32) {
      const int dj = rw[__ldg(g.succ + xs.succ_off + u)];
      if (dj != dp) m |= 1u << dj;
    }
    return __reduce_or_sync(kFullMask, m);
  }

  // A listed consumer of p on p's accelerator under placement rw (uniform).
  __device__ bool local_consumer(uint32_t p, const uint8_t* rw) const {
    const uint4 cs = op_cons(g.ops, p);
    const XqSucc xs = op_xqsucc(g.ops, p);
    const bool all = (cs.w & kAllCons) != 0;
    const uint32_t* lst = all ? g.succ + xs.succ_off : g.cons + cs.x;
    const uint32_t nl = all ? xs.nsucc : cs.y;
    const int dp = rw[p];
    bool f = false;
    for (uint32_t u = lane_id(); u < nl; u += 32) f |= rw[__ldg(lst + u)] == dp;
    return __any_sync(kFullMask, f);
  }

  // Op p (started before the resume point, finishing at or after it) among the
  // coming ones of its accelerator d's list, kept in finish order: insert
  // (want) or remove.  Uniform call; lane d owns the list's ends.
  __device__ void list_set(uint32_t p, int d, bool want) {
    const unsigned lane = lane_id();
    const int32_t a = __shfl_sync(kFullMask, al(), d);  // the link of the last arrived op leads to the first coming one
    int32_t h = __shfl_sync(kFullMask, uh, d);
    int32_t t = __shfl_sync(kFullMask, lt(), d);
    int32_t* nxp = nextop();
    const tm_t fp = this->fin(p);
    int32_t prev = a, cur = h;
    bool found = false;
    for (int guard = 0; cur >= 0 && guard <= g.n; ++guard) {
      if (cur == (int32_t)p) {
        found = true;
        break;
      }
      if (this->fin((uint32_t)cur) > fp) break;
      prev = cur;
      cur = cur == t ? -1 : nxp[cur];
    }
    if (want == found) return;
    const bool first = cur == h;  // (also with no coming op)
    if (want) {  // link p between prev and cur
      if (lane == 0) {
        nxp[p] = cur;
        if (prev >= 0) nxp[prev] = (int32_t)p;
      }
      if (first) h = (int32_t)p;
      if (cur < 0) t = (int32_t)p;
    } else {  // unlink p (cur == p)
      const int32_t after = (int32_t)p == t ? -1 : nxp[p];
      if (lane == 0 && prev >= 0) nxp[prev] = after;
      if (first) h = after;
      if (t == (int32_t)p) t = prev;
    }
    __syncwarp();
    if ((int)lane == d) {
      uh = h;
      lt() = t;
      fu = h < 0 ? kNever : this->fin((uint32_t)h);
    }
    __syncwarp();
  }

  // One incremental candidate resumed from the arbitrated base snapshot.
  // Results equal the full arbitrated simulation of the moved placement
  // (Sec. 3.5.2); the fix-ups below are what the moves change in the state
  // at the checkpoint T_c <= T0: a moved op's inputs counted so far (only
  // predecessors local under the new placement and already started count; no
  // remote one has finished) and its READY key; and for every predecessor p
  // of a moved op that started before T_c (it finishes at or after T0, so
  // none of its intents, transfers or receive buffers exist yet): its remote
  // set, the holds on its copy, its place in its accelerator's list of coming
  // intents, and whether its copy's release is already logged.
  __device__ void inc_candidate(int64_t k, uint8_t* crow) {
    const DevBase& B = P.base;
    const unsigned lane = lane_id();
    const int32_t m0 = P.move_off[k], m1 = P.move_off[k + 1];
    const int32_t nm = m1 - m0;
    // validate the move list (range, then an op moved twice)
    bool bad = false, dup = false;
    for (int32_t m = m0 + (int32_t)lane; m < m1; m += 32)
      bad |= P.move_op[m] < 0 || P.move_op[m] >= g.n || P.move_dev[m] >= g.D;
    bad = __any_sync(kFullMask, bad);
    if (!bad)
      for (int32_t m = m0 + (int32_t)lane; m < m1; m += 32)
        for (int32_t m2 = m + 1; m2 < m1 && !dup; ++m2) dup = P.move_op[m2] == P.move_op[m];
    dup = __any_sync(kFullMask, dup);
    if (B.status[0] != GMG_SIM_OK) {
      this->write_invalid(k, GMG_SIM_BADBASE);
      return;
    }
    if (bad || dup) {
      this->write_invalid(k, bad ? GMG_SIM_MOVE_RANGE : GMG_SIM_MOVE_DUP);
      return;
    }
    warp_copy16(crow, B.row, B.ld);
    __syncwarp();
    uint64_t t0 = kKeyMax;
    for (int t = lane; t < nm; t += 32) {
      const int32_t op = P.move_op[m0 + t];
      const uint8_t dvc = P.move_dev[m0 + t];
      crow[op] = dvc;
      if (dvc != B.row[op]) {
        const RelPred rp = op_relpred(g.ops, (uint32_t)op);
        uint64_t tx = (uint64_t)rp.rel;
        if (rp.npred) {
          tx = kKeyMax;
          for (uint32_t u = 0; u < rp.npred; ++u) {
            const uint64_t fp = (uint64_t)B.fb[__ldg(g.pred + rp.pred_off + u) & kIdMask];
            tx = fp < tx ? fp : tx;
          }
        }
        t0 = tx < t0 ? tx : t0;
      }
    }
    t0 = warp_min_u64(t0);
    __syncwarp();
    row = crow;
    const DevOut& o = P.out;
    if (t0 == kKeyMax) {  // no effective move: the base results
      const int64_t* rs = B.res_scalars;
      if (lane == 0) {
        o.makespan[k] = rs[0];
        o.score[k] = rs[1];
        o.status[k] = GMG_SIM_OK;
        o.viol_flag[k] = (int32_t)rs[2];
        o.viol_op[k] = (int32_t)rs[3];
        o.viol_dev[k] = (int32_t)rs[4];
        o.viol_time[k] = rs[5];
        o.sla_miss[k] = (int32_t)rs[6];
        o.events[k] = 0;
      }
      for (int d = lane; d < g.D; d += 32) o.peak[k * g.D + d] = B.res_peak[d];
      if (o.req_done)
        for (int r = lane; r < g.R; r += 32) o.req_done[k * g.R + r] = B.res_creq[r];
      const int ts = this->trace_slot(k);
      if (ts >= 0)
        for (int x = lane; x < g.n; x += 32) {
          o.trace_finish[(int64_t)ts * g.n + x] = B.fb[x];
          o.trace_start[(int64_t)ts * g.n + x] =
              B.fb[x] - this->dur_of((uint32_t)x, B.row[x], op_durbytes(g.ops, (uint32_t)x).x);
        }
      return;
    }
    this->T0 = (tm_t)t0;
    int best = -1;
    for (int c = lane; c < B.nck; c += 32)
      if (B.ck_time[c] <= (int64_t)t0) best = c;
    const int c = __reduce_max_sync(kFullMask, best);
    const int64_t* sc = B.ck_scalars + (int64_t)c * 8;
    const int qsz = (int)sc[0];
    const int msz = (int)sc[7];
    if (qsz + nm > P.pend_cap - 32 || msz + nm > P.mcap) {
      this->write_invalid(k, GMG_SIM_QUEUE);
      return;
    }
    // the simulation state of checkpoint c
    this->Tc = (tm_t)B.ck_time[c];
    this->drained = (tm_t)sc[3];
    this->rootptr = (int)sc[1];
    this->load_root();
    this->score = lane == 0 ? sc[2] : 0;  // lanes add up their ops' finishes
    this->vflag = (int32_t)sc[4];
    this->vt = sc[5];
    this->vop = (int32_t)(sc[6] >> 32);
    this->vdev = (int32_t)(sc[6] & 0xffffffff);
    this->iters = 0;
    this->nev = 0;
    this->readypops = 0;
    this->last_t = -1;
    status = GMG_SIM_OK;
    pd.r = pd.e = kNever;
    this->opn = 0;
    this->dv.load_free(B.ck_dev + (int64_t)c * 3 * g.D);
    this->dv.load_bytes(B.ck_dev + (int64_t)c * 3 * g.D);
    for (int r = lane; r < g.R; r += 32) this->creq()[r] = B.ck_creq[(int64_t)c * g.R + r];
    this->fill_fin();
    restore_arb(c);
    // READY keys, except those of moved ops (recomputed below): the lanes' go
    // through the sort area (free between drains), the others to the heap
    auto queue = [&](int n, uint64_t key) {
      if (n < 32) this->sortk[n] = key;
      else *this->q.kp(n - 32) = key;
    };
    int nq = 0;
    for (int c0 = 0; c0 < qsz; c0 += 32) {
      const int x = c0 + (int)lane;
      const bool v = x < qsz;
      const uint64_t key = v ? B.ck_qkey[(int64_t)c * B.ckq + x] : 0ull;
      const uint32_t op = this->rq.op(key);
      // (a moved op without predecessors keeps its ready time)
      const bool keep = v && (crow[op] == B.row[op] || op_relpred(g.ops, op).npred == 0u);
      const uint32_t bal = __ballot_sync(kFullMask, keep);
      if (keep) queue(nq + __popc(bal & lanes_below()), key);
      nq += __popc(bal);
    }
    // logged HBM events, except the release of a moved op's predecessor's own
    // copy (regenerated below if it is due)
    int outn = 0;
    for (int c0 = 0; c0 < msz; c0 += 32) {
      const int x = c0 + (int)lane;
      const bool v = x < msz;
      const uint64_t e = v ? B.ck_mkey[(int64_t)c * B.ckm + x] : 0ull;
      bool keep = v;
      if (v && this->kc.cls(e) == kFree) {
        const uint32_t op = this->kc.op(e);
        const int dev = (int)(e >> g.ds);
        if (dev == B.row[op]) {
          const XqSucc xs = op_xqsucc(g.ops, op);
          for (uint32_t u = 0; u < xs.nsucc && keep; ++u) {
            const uint32_t j = __ldg(g.succ + xs.succ_off + u);
            keep = crow[j] == B.row[j];
          }
        }
      }
      const uint32_t bal = __ballot_sync(kFullMask, keep);
      if (keep) *this->log.kp(outn + __popc(bal & lanes_below())) = e;
      outn += __popc(bal);
    }
    this->log.n = outn;
    __syncwarp();
    // every effective move: the moved op's inputs, its predecessors' state
    for (int32_t t = 0; t < nm; ++t) {
      const uint32_t x = (uint32_t)P.move_op[m0 + t];
      if (crow[x] == B.row[x]) continue;
      const RelPred rp = op_relpred(g.ops, x);
      // inputs of x present so far: started predecessors local under crow
      int32_t cx = 0;
      uint64_t rx = 0;
      for (uint32_t u = lane; u < rp.npred; u += 32) {
        const uint32_t p = __ldg(g.pred + rp.pred_off + u) & kIdMask;
        if (this->base_time(this->rb, p) < this->Tc && crow[p] == crow[x]) {
          ++cx;
          const uint64_t fp = (uint64_t)this->base_time(this->fb, p);
          rx = fp > rx ? fp : rx;
        }
      }
      cx = (int32_t)__reduce_add_sync(kFullMask, (uint32_t)cx);
      rx = warp_max_u64(rx);
      if (lane == 0) {
        cnt()[x] = cx;
        rmax()[x] = (tm_t)rx;
      }
      if (rp.npred > 0 && (uint32_t)cx == rp.npred) {
        const tm_t rel = (tm_t)rp.rel;
        const tm_t rj = rel > (tm_t)rx ? rel : (tm_t)rx;
        if (lane == 0) queue(nq, this->rq.make(rj, x, (tm_t)1));
        ++nq;
      }
      // started predecessors: remote set, holds, FIFO, own copy's release;
      // each predecessor once, by its first moved successor in this list
      for (uint32_t u = 0; u < rp.npred; ++u) {
        const uint32_t p = __ldg(g.pred + rp.pred_off + u) & kIdMask;
        if (this->base_time(this->rb, p) >= this->Tc) continue;
        bool first = true;
        for (int32_t t2 = 0; t2 < t && first; ++t2) {
          const uint32_t x2 = (uint32_t)P.move_op[m0 + t2];
          if (crow[x2] == B.row[x2]) continue;
          const RelPred r2 = op_relpred(g.ops, x2);
          for (uint32_t u2 = 0; u2 < r2.npred; ++u2)
            if ((__ldg(g.pred + r2.pred_off + u2) & kIdMask) == p) {
              first = false;
              break;
            }
        }
        if (!first) continue;
        const uint32_t rc = remote_set(p, crow);
        const bool lc = local_consumer(p, crow);
        const int dp = crow[p];
        const int32_t holds = 1 + __popc(rc) - (lc ? 0 : 1);
        const tm_t fp = this->fin(p);
        if (lane == 0) {
          rmask()[p] = rc;
          refs()[p] = holds;
          this->holdb()[p] = fp;
        }
        __syncwarp();
        list_set(p, dp, rc != 0u);
        this->log_event(lane == 0 && holds == 0, this->kc.make(fp, kFree, p), dp);
      }
    }
    __syncwarp();
    if ((int)lane < nq && lane < 32u) {
      const uint64_t key = this->sortk[lane];
      this->hold_op((tm_t)this->rq.time(key), this->rq.op(key));
    }
    this->q.size = nq > 32 ? nq - 32 : 0;
    this->q.heapify();
    run();
    this->finish(k);
  }
};

// 96 registers a thread, 5 blocks per SM (kArbBlocks): at 72 and 7 blocks the
// spills cost more than the two blocks give (prefill graph, ms, 7 blocks / 5: 2,048
// placements 12.7 / 9.6, 3,000 15.0 / 10.6) -- unless they save a second wave: 6
// blocks where they hold all placements and 5 do not (5 / 6, 3,500 placements: 98
// ops on 2 accelerators 0.49 / 0.33 ms, 3,088 ops on 8 17.8 / 12.1), 7 where 6 do not
// and the graph has 1,024 ops and 12 accelerators at most (5 / 7, 4,096 placements:
// 386 ops on 8 accelerators 2.24 / 2.00, 772 4.41 / 4.17, 3,088 18.7 / 19.2, 392 in
// four requests 2.28 / 2.27; 392 and 772 ops on 16 accelerators 2.35 / 2.47 and 4.55 /
// 4.58, 386 on 32 2.33 / 2.65).  Resumed candidates are handed out one by one and gain
// nothing from it (3,500 on 8 accelerators, 3,088 ops, 5 / 6 / 7: 10.6 / 13.5 / 14.2).
template <bool kT32, bool kTypes, int kHot, int kBlocks>
__global__ void __launch_bounds__(128, kBlocks) sim_arb_kernel(const __grid_constant__ ArbParams A) {
  extern __shared__ __align__(16) uint8_t smem[];
  const unsigned wib = threadIdx.x >> 5;
  const int64_t slot = (int64_t)blockIdx.x * (blockDim.x >> 5) + wib;
  const int64_t nslots = (int64_t)gridDim.x * (blockDim.x >> 5);
  ArbSim<kT32, kTypes, kFull, kHot> S(A);
  setup_slot(S, A.P, wib, slot, smem);
  S.setup_arb(smem + A.smem_std + (size_t)wib * A.smem_arb);
  for (int64_t k = slot; k < A.P.K; k += nslots) {
    S.row = A.P.place + k * A.P.ld;
    if (A.pre_status) {
      const int32_t ps = A.pre_status[k];
      if (ps != GMG_SIM_OK) {
        S.write_invalid(k, ps);
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

// The arbitrated base snapshot: the base placement simulated once (64-bit
// times) with checkpoints of the simulation and the arbiter.
template <bool kTypes>
__global__ void __launch_bounds__(32, 1) sim_arb_base_kernel(const __grid_constant__ ArbParams A) {
  extern __shared__ __align__(16) uint8_t smem[];
  ArbSim<false, kTypes, kBase> S(A);
  setup_slot(S, A.P, 0, 0, smem);
  S.setup_arb(smem + A.smem_std);
  const DevBase& B = A.P.base;
  const unsigned lane = lane_id();
  warp_prefetch_l2(A.P.g.ws, A.P.g.ws_bytes);
  for (int c = lane * 16; c < B.ld; c += 512)
    *reinterpret_cast<uint4*>(B.row + c) = *reinterpret_cast<const uint4*>(A.P.place + c);
  for (int c = lane; c < B.nck; c += 32) B.ck_time[c] = kI64Max;
  S.row = A.P.place;
  __syncwarp();
  if (S.row_has_bad_device(A.P.place)) {
    if (lane == 0) B.status[0] = GMG_SIM_BADDEV;
    return;
  }
  S.reset_arb();
  S.ck = 0;
  S.next_ck = 0;
  {  // checkpoint 0: the initial state
    const typename ArbSim<false, kTypes, kBase>::Outside none{kKeyMax, 0};
    S.arb_checkpoint(none);
  }
  S.run();
  write_base(S, B);
}

// Incremental candidates resumed from the arbitrated base snapshot.
template <bool kT32, bool kTypes, int kHot>
__global__ void __launch_bounds__(128, kArbBlocks) sim_arb_inc_kernel(const __grid_constant__ ArbParams A) {
  extern __shared__ __align__(16) uint8_t smem[];
  const unsigned wib = threadIdx.x >> 5;
  const int64_t slot = (int64_t)blockIdx.x * (blockDim.x >> 5) + wib;
  ArbSim<kT32, kTypes, kInc, kHot> S(A);
  setup_slot(S, A.P, wib, slot, smem);
  S.setup_arb(smem + A.smem_std + (size_t)wib * A.smem_arb);
  S.rb = A.P.base.rb;
  S.fb = A.P.base.fb;
  uint8_t* crow = A.P.scratch + slot * A.P.slot_bytes + A.P.off_row;
  for (int64_t k = take_candidate(A.P.next_k); k < A.P.K; k = take_candidate(A.P.next_k)) S.inc_candidate(k, crow);
}

// One warp per incremental candidate: check the move list (an op or device
// out of range, then an op moved twice), copy the base row, apply the moves.
// A base row with a device out of range makes every candidate BADBASE.
__global__ void __launch_bounds__(128) expand_moves_kernel(const uint8_t* base_row, const int32_t* base_status,
                                                           int32_t ld, int32_t n, int32_t D, const int32_t* off,
                                                           const int32_t* op, const uint8_t* dev, int32_t K,
                                                           uint8_t* rows, int32_t* status) {
  const unsigned lane = lane_id();
  const int64_t w0 = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const int64_t nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
  // Only a base row with a device out of range invalidates the moved rows;
  // the base's own (pure-latency) simulation status -- a queue or loop limit
  // of that run -- says nothing about the arbitrated simulations of the
  // moved placements, which run in full.
  const bool base_ok = *base_status != GMG_SIM_BADDEV;
  for (int64_t k = w0; k < K; k += nw) {
    const int32_t a = off[k], b = off[k + 1];
    int32_t st = base_ok ? GMG_SIM_OK : GMG_SIM_BADBASE;
    if (st == GMG_SIM_OK) {
      bool bad = false;
      for (int32_t m = a + (int32_t)lane; m < b; m += 32) bad |= op[m] < 0 || op[m] >= n || dev[m] >= D;
      if (__any_sync(kFullMask, bad)) st = GMG_SIM_MOVE_RANGE;
    }
    if (st == GMG_SIM_OK) {
      bool dup = false;
      for (int32_t m = a + (int32_t)lane; m < b; m += 32)
        for (int32_t m2 = m + 1; m2 < b && !dup; ++m2) dup = op[m2] == op[m];
      if (__any_sync(kFullMask, dup)) st = GMG_SIM_MOVE_DUP;
    }
    uint8_t* rw = rows + k * (int64_t)ld;
    warp_copy16(rw, base_row, ld);
    __syncwarp();
    if (st == GMG_SIM_OK)
      for (int32_t m = a + (int32_t)lane; m < b; m += 32) rw[op[m]] = dev[m];
    if (lane == 0) status[k] = st;
    __syncwarp();
  }
}

}  // namespace

cudaError_t launch_expand_moves(const uint8_t* base_row, const int32_t* base_status, int32_t ld, int32_t n,
                                int32_t D, const int32_t* off, const int32_t* op, const uint8_t* dev, int32_t K,
                                uint8_t* rows, int32_t* status, cudaStream_t st) {
  const int blocks = (int)std::min<int64_t>(((int64_t)K + 3) / 4, 152 * 16);
  expand_moves_kernel<<<std::max(blocks, 1), 128, 0, st>>>(base_row, base_status, ld, n, D, off, op, dev, K,
                                                           rows, status);
  return cudaGetLastError();
}

// Instances by (32-bit times, accelerator types; compact records wherever the
// graph has them).
template <int kBlocks>
const void* arb_ptr(const DevGmg& g) {
  if (g.hot_ok) return (const void*)sim_arb_kernel<true, false, kHotGlobal, kBlocks>;
  if (g.t32)
    return g.ntypes >= 2 ? (const void*)sim_arb_kernel<true, true, kHotNone, kBlocks>
                         : (const void*)sim_arb_kernel<true, false, kHotNone, kBlocks>;
  return g.ntypes >= 2 ? (const void*)sim_arb_kernel<false, true, kHotNone, kBlocks>
                       : (const void*)sim_arb_kernel<false, false, kHotNone, kBlocks>;
}
const void* arb_kernel_ptr(const DevGmg& g, int blocks) {
  return blocks == 7 ? arb_ptr<7>(g) : blocks == 6 ? arb_ptr<6>(g) : arb_ptr<kArbBlocks>(g);
}
const void* arb_inc_kernel_ptr(const DevGmg& g) {
  if (g.hot_ok) return (const void*)sim_arb_inc_kernel<true, false, kHotGlobal>;
  if (g.t32)
    return g.ntypes >= 2 ? (const void*)sim_arb_inc_kernel<true, true, kHotNone>
                         : (const void*)sim_arb_inc_kernel<true, false, kHotNone>;
  return g.ntypes >= 2 ? (const void*)sim_arb_inc_kernel<false, true, kHotNone>
                       : (const void*)sim_arb_inc_kernel<false, false, kHotNone>;
}
const void* arb_base_kernel_ptr(bool types) {
  return types ? (const void*)sim_arb_base_kernel<true> : (const void*)sim_arb_base_kernel<false>;
}

cudaError_t launch_arb(const ArbParams& A, int grid, int block, size_t smem, cudaStream_t st) {
  void* args[] = {const_cast<ArbParams*>(&A)};
  return cudaLaunchKernel(arb_kernel_ptr(A.P.g, A.blocks), dim3(grid), dim3(block), args, smem, st);
}

cudaError_t launch_arb_base(bool types, const ArbParams& A, size_t smem, cudaStream_t st) {
  void* args[] = {const_cast<ArbParams*>(&A)};
  return cudaLaunchKernel(arb_base_kernel_ptr(types), dim3(1), dim3(32), args, smem, st);
}

cudaError_t launch_arb_inc(const ArbParams& A, int grid, int block, size_t smem, cudaStream_t st) {
  void* args[] = {const_cast<ArbParams*>(&A)};
  return cudaLaunchKernel(arb_inc_kernel_ptr(A.P.g), dim3(grid), dim3(block), args, smem, st);
}

}  // namespace gsim

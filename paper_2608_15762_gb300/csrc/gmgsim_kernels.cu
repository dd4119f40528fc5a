// The base-snapshot kernel, select_best and the launchers of every kernel
// (called from the host translation unit).
#include "gmgsim_sim.cuh"

namespace gsim {
namespace {

// ---------------------------------------------------------------------------
// base_create: simulate the base placement once, recording resume points.
// ---------------------------------------------------------------------------
// The base placement is kept for the candidates.
__device__ __forceinline__ void copy_base_row(const SimParams& P) {
  const DevBase& B = P.base;
  for (int c = (int)lane_id() * 16; c < B.ld; c += 512)
    *reinterpret_cast<uint4*>(B.row + c) = *reinterpret_cast<const uint4*>(P.place + c);
  __syncwarp();
}

template <class S_>
__device__ __forceinline__ void sweep_base(S_& S, const SimParams& P) {
  S.row = P.place;
  S.reset_common();
  if (S.row_has_bad_device(P.place)) S.status = GMG_SIM_BADDEV;
  S.ck = 0;
  S.next_ck = 0;
  // checkpoint 0: the initial state, valid for every resume time >= 0
  if (S.status == GMG_SIM_OK) S.maybe_checkpoint(0);
  S.run();
}

template <bool kNarrow, bool kTypes>
__global__ void __launch_bounds__(32, 1) sim_base_kernel(const __grid_constant__ SimParams P) {
  extern __shared__ __align__(16) uint8_t smem[];
  Sim<kNarrow, kBase, false, false, kTypes, kHotNone> S(P);
  setup_slot(S, P, 0, 0, smem);
  warp_prefetch_l2(P.g.ws, P.g.ws_bytes);
  copy_base_row(P);
  for (int c = lane_id(); c < P.base.nck; c += 32) P.base.ck_time[c] = kI64Max;
  __syncwarp();
  sweep_base(S, P);
  write_base(S, P.base);
}

// The same by two warps, the sweep and the HBM accounting: graphs whose accelerator
// ids fit into the event key.
template <bool kNarrow, bool kT32, bool kTypes, int kHot>
__global__ void __launch_bounds__(64, 1) sim_base_pair_kernel(const __grid_constant__ SimParams P) {
  extern __shared__ __align__(16) uint8_t smem[];
  if (threadIdx.x < 32) {
    Sim<kNarrow, kBase, true, kT32, kTypes, kHot, !kNarrow, kSweep> S(P);
    setup_slot(S, P, 0, 0, smem);
    sweep_base(S, P);
    S.hand_end();
    leave_pair(S);
  } else {
    Sim<kNarrow, kBase, true, kT32, kTypes, kHot, !kNarrow, kAccount> S(P);
    setup_slot(S, P, 0, 0, smem);
    warp_prefetch_l2(P.g.ws, P.g.ws_bytes);
    for (int c = lane_id(); c < P.base.nck; c += 32) P.base.ck_time[c] = kI64Max;
    copy_base_row(P);
    S.row = P.place;
    S.reset_common();
    S.account();
    write_base(S, P.base);
    S.done();
  }
}

// ---------------------------------------------------------------------------
// select_best (Algorithm 1, BestRecordedCandidateResult): block argmin of
// (mode ? sla_miss : 0, score, k) over eligible candidates, then a one-block
// final argmin; one block alone for few candidates.
// ---------------------------------------------------------------------------
struct Rank {
  int64_t a;  // sla_miss (mode 1) or 0; INT64_MAX = not eligible
  int64_t s;  // score
  int64_t k;
};

__device__ __forceinline__ bool rank_less(const Rank& x, const Rank& y) {
  if (x.a != y.a) return x.a < y.a;
  if (x.s != y.s) return x.s < y.s;
  return x.k < y.k;
}

__device__ Rank block_argmin(Rank r) {
  __shared__ Rank part[32];
  for (int o = 16; o > 0; o >>= 1) {
    Rank t;
    t.a = __shfl_down_sync(kFullMask, r.a, o);
    t.s = __shfl_down_sync(kFullMask, r.s, o);
    t.k = __shfl_down_sync(kFullMask, r.k, o);
    if (rank_less(t, r)) r = t;
  }
  const unsigned w = threadIdx.x >> 5;
  if (lane_id() == 0) part[w] = r;
  __syncthreads();
  if (w == 0) {
    const unsigned nw = blockDim.x >> 5;
    r = lane_id() < nw ? part[lane_id()] : Rank{kI64Max, kI64Max, kI64Max};
    for (int o = 16; o > 0; o >>= 1) {
      Rank t;
      t.a = __shfl_down_sync(kFullMask, r.a, o);
      t.s = __shfl_down_sync(kFullMask, r.s, o);
      t.k = __shfl_down_sync(kFullMask, r.k, o);
      if (rank_less(t, r)) r = t;
    }
  }
  return r;
}

__device__ __forceinline__ Rank best_of(const int32_t* status, const int32_t* viol, const int64_t* score,
                                        const int32_t* miss, int32_t K, int32_t mode) {
  Rank r{kI64Max, kI64Max, kI64Max};
  for (int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; k < K;
       k += (int64_t)gridDim.x * blockDim.x) {
    if (status[k] != GMG_SIM_OK || viol[k] != 0) continue;
    const Rank c{mode ? (int64_t)miss[k] : 0, score[k], k};
    if (rank_less(c, r)) r = c;
  }
  return block_argmin(r);
}

__device__ __forceinline__ void write_best(const Rank& r, int64_t* best) {
  const bool none = r.k == kI64Max;
  best[0] = none ? -1 : r.k;
  best[1] = none ? kI64Max : r.s;
}

__global__ void __launch_bounds__(256) select_partial_kernel(const int32_t* status, const int32_t* viol,
                                                             const int64_t* score, const int32_t* miss,
                                                             int32_t K, int32_t mode, Rank* part) {
  const Rank r = best_of(status, viol, score, miss, K, mode);
  if (threadIdx.x == 0) part[blockIdx.x] = r;
}

__global__ void __launch_bounds__(256) select_final_kernel(const Rank* part, int32_t nparts, int64_t* best) {
  Rank r{kI64Max, kI64Max, kI64Max};
  for (int i = threadIdx.x; i < nparts; i += blockDim.x)
    if (rank_less(part[i], r)) r = part[i];
  r = block_argmin(r);
  if (threadIdx.x == 0) write_best(r, best);
}

// Up to kSelectOne candidates: one block does both (a second launch costs more
// than the few rows that each thread goes through: one / two launches in a graph,
// us, 256 candidates 2.4 / 4.4, 1,024 3.4 / 4.6, 2,048 4.0 / 4.4, 4,096 5.3 / 4.7,
// 8,192 7.4 / 4.7).
__global__ void __launch_bounds__(1024) select_one_kernel(const int32_t* status, const int32_t* viol,
                                                          const int64_t* score, const int32_t* miss, int32_t K,
                                                          int32_t mode, int64_t* best) {
  const Rank r = best_of(status, viol, score, miss, K, mode);
  if (threadIdx.x == 0) write_best(r, best);
}
constexpr int32_t kSelectOne = 2048;

}  // namespace

// ---------------------------------------------------------------------------
// Launchers (called from the host translation unit).
// ---------------------------------------------------------------------------
size_t select_rank_bytes() { return sizeof(Rank); }

const void* full_kernel_ptr(const DevGmg& g);  // gmgsim_full.cu
const void* full_pair_kernel_ptr(const DevGmg& g);
const void* inc_kernel_ptr(const DevGmg& g);  // gmgsim_inc.cu
const void* inc_pair_kernel_ptr(const DevGmg& g);

// One warp (64-bit times): graphs whose accelerator ids do not fit into the event
// key.
template <bool N>
const void* base_ptr(bool types) {
  return types ? (const void*)sim_base_kernel<N, true> : (const void*)sim_base_kernel<N, false>;
}
const void* base_kernel_ptr(const DevGmg& g) {
  return g.D <= 32 ? base_ptr<true>(g.ntypes >= 2) : base_ptr<false>(g.ntypes >= 2);
}
// Two warps: all others, by (at most 32 accelerators, 32-bit times, accelerator
// types; compact records wherever the graph has them, only with 32-bit times).
template <bool N, bool T32>
const void* base_pair_ptr(bool types) {
  return types ? (const void*)sim_base_pair_kernel<N, T32, true, kHotNone>
               : (const void*)sim_base_pair_kernel<N, T32, false, kHotNone>;
}
template <bool N>
const void* base_pair_ptr_n(const DevGmg& g) {
  if (g.hot_ok) return (const void*)sim_base_pair_kernel<N, true, false, kHotGlobal>;
  return g.t32 ? base_pair_ptr<N, true>(g.ntypes >= 2) : base_pair_ptr<N, false>(g.ntypes >= 2);
}
const void* base_pair_kernel_ptr(const DevGmg& g) { return g.D <= 32 ? base_pair_ptr_n<true>(g) : base_pair_ptr_n<false>(g); }

cudaError_t set_smem_limits(int smem) {
  DevGmg g{};
  for (int c = 0; c < 48; ++c) {
    g.D = c % 3 == 0 ? 16 : c % 3 == 1 ? 32 : 33;
    g.dev_key = (c / 3) & 1;
    g.t32 = (c / 6) & 1;
    g.ntypes = (c / 12) & 1 ? 2 : 0;
    g.hot_ok = (c / 24) & 1;
    const void* fns[] = {full_kernel_ptr(g),      inc_kernel_ptr(g),      base_kernel_ptr(g),
                         full_pair_kernel_ptr(g), inc_pair_kernel_ptr(g), base_pair_kernel_ptr(g)};
    for (const void* f : fns) {
      const cudaError_t e = cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
      if (e != cudaSuccess) return e;
    }
  }
  return cudaSuccess;
}

// A kernel instance's launch through its pointer (the instance is chosen by
// the graph's flags).
static cudaError_t launch_ptr(const void* fn, const SimParams& P, int grid, int block, size_t smem,
                              cudaStream_t st) {
  void* args[] = {const_cast<SimParams*>(&P)};
  return cudaLaunchKernel(fn, dim3(grid), dim3(block), args, smem, st);
}

// pair: two warps per candidate, a block of their own.
cudaError_t launch_full(bool pair, const SimParams& P, int grid, int block, size_t smem, cudaStream_t st) {
  return launch_ptr(pair ? full_pair_kernel_ptr(P.g) : full_kernel_ptr(P.g), P, grid, block, smem, st);
}

cudaError_t launch_inc(bool pair, const SimParams& P, int grid, int block, size_t smem, cudaStream_t st) {
  return launch_ptr(pair ? inc_pair_kernel_ptr(P.g) : inc_kernel_ptr(P.g), P, grid, block, smem, st);
}

cudaError_t launch_base(bool pair, const SimParams& P, size_t smem, cudaStream_t st) {
  return launch_ptr(pair ? base_pair_kernel_ptr(P.g) : base_kernel_ptr(P.g), P, 1, pair ? 64 : 32, smem, st);
}

cudaError_t launch_select(const int32_t* status, const int32_t* viol, const int64_t* score,
                          const int32_t* miss, int32_t K, int32_t mode, void* tmp, int nparts,
                          int64_t* best, cudaStream_t st) {
  if (K <= kSelectOne) {
    const int threads = K <= 32 ? 32 : (K + 31) / 32 * 32;
    select_one_kernel<<<1, threads < 1024 ? threads : 1024, 0, st>>>(status, viol, score, miss, K, mode, best);
    return cudaGetLastError();
  }
  Rank* part = reinterpret_cast<Rank*>(tmp);
  select_partial_kernel<<<nparts, 256, 0, st>>>(status, viol, score, miss, K, mode, part);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  select_final_kernel<<<1, 256, 0, st>>>(part, nparts, best);
  return cudaGetLastError();
}

}  // namespace gsim

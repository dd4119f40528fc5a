// Online linear estimators (Sec. 3.3.1): batched least-squares refits from
// executor feedback and the integer duration / link tables they produce for
// the simulation.  The C ABI is declared in include/gmgest.h.
//
// est_update, in two launches:
//  1. one warp per chunk of 32 to 512 consecutive sample rows (enough chunks to
//     fill the GPU, long enough that the reduction is a small part): for every
//     estimator with rows in the chunk, lane l sums rows l, l+32, ... into the
//     upper triangle of X^T X and X^T y (fp64); a fixed tree combines the lanes
//     and the totals go to the caller's buffer.  Estimator e's part of chunk c is
//     entry c + e (each chunk and each estimator begins one, in order), so an
//     estimator's entries are consecutive and no prefix of chunk counts is needed;
//  2. per estimator, its entries are added in a fixed order -- by one warp, or by
//     eight that share them -- and one warp adds the result to the running
//     statistics and refits by a Cholesky solve of the normal equations, lane i
//     holding row i.
// Every sum has a fixed order, so results do not depend on scheduling.  F
// (<= 8) is a template parameter so the per-sample arrays stay in registers.
//
// The first launch is bound by fp64 instructions (an SM issues two fp64 lanes a
// clock): F(F+1)/2 + F multiply-adds per row cannot go.  The tree halves the
// values that a lane carries with every step: 31 additions a lane for up to 32
// values instead of 5 for each value.  458,752 rows
// of 5 features: 44.5 -> 22.8 us (fp64 floor 15); the second launch, 28 estimators of 64
// entries: 26.5 -> 11.8 us.

#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>

#include "../../include/gmgest.h"

namespace gest {
namespace {

constexpr unsigned kFullMask = 0xffffffffu;
constexpr double kPivotRel = 1e-12;   // pivot threshold relative to its own diagonal entry
constexpr int64_t kMaxTicks = int64_t(1) << 40;
constexpr int32_t kMinChunk = 32, kMaxChunk = 512;  // sample rows per warp in the first launch
// Warps that fill 152 SMs (12 each).  An update, us, with 912 / 1,824 / 3,648: 28
// estimators of 5 features, 60,000 rows 18.3 / 18.9 / 21.4, 458,752 rows 34.5 / 30.7 /
// 34.9, 2,000,000 (512 rows a warp in each) 94.3 / 94.5 / 94.8; 64 of 2 features,
// 60,000 rows 12.2 / 13.1 / 15.8, 458,752 rows 16.4 / 15.2 / 18.9.
constexpr int64_t kChunks = 1824;
constexpr int kFitWarps = 8;       // warps per estimator in the second launch when it has many entries

size_t align256(size_t x) { return (x + 255) & ~(size_t)255; }

// State layout (each array 256-byte aligned): G [E][F(F+1)/2] upper triangle
// row-major, h [E][F], n [E], beta [E][F], fitted [E] (int32).
struct Layout {
  size_t g, h, n, beta, fitted, total;
};

Layout layout(int32_t E, int32_t F) {
  Layout L;
  const size_t tri = (size_t)F * (F + 1) / 2;
  size_t o = 0;
  L.g = o;
  o = align256(o + 8 * tri * (size_t)E);
  L.h = o;
  o = align256(o + 8 * (size_t)F * E);
  L.n = o;
  o = align256(o + 8 * (size_t)E);
  L.beta = o;
  o = align256(o + 8 * (size_t)F * E);
  L.fitted = o;
  o = align256(o + 4 * (size_t)E);
  L.total = o;
  return L;
}

struct State {
  double* g;
  double* h;
  double* n;
  double* beta;
  int32_t* fitted;
};

State view(void* d_state, int32_t E, int32_t F) {
  const Layout L = layout(E, F);
  uint8_t* b = static_cast<uint8_t*>(d_state);
  return State{reinterpret_cast<double*>(b + L.g), reinterpret_cast<double*>(b + L.h),
               reinterpret_cast<double*>(b + L.n), reinterpret_cast<double*>(b + L.beta),
               reinterpret_cast<int32_t*>(b + L.fitted)};
}

// The lanes' totals of the values v[0..N): lane l gets the total of value l (and
// of value 32 + l in the second word).  Step by step a lane passes half of the
// values that it carries to the lane across and adds its own half's: the same
// pairwise tree (distance 16, 8, ..., 1) for every value.
template <int N>
__device__ __forceinline__ double reduce_to_lanes(double (&v)[32]) {
  const int lane = threadIdx.x & 31;
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    const bool up = (lane & o) != 0;
#pragma unroll
    for (int i = 0; i < o; ++i) {
      const double give = up ? v[i] : v[i + o];
      const double keep = up ? v[i + o] : v[i];
      v[i] = keep + __shfl_xor_sync(kFullMask, give, o);
    }
  }
  return v[0];
}

// One warp per chunk of rows: entry c + e = [T triangle | F] of estimator e's rows.
template <int F>
__global__ void __launch_bounds__(128) est_partial_kernel(int32_t E, int32_t S, int32_t chunk,
                                                          const int32_t* __restrict__ off,
                                                          const double* __restrict__ x,
                                                          const double* __restrict__ y,
                                                          double* __restrict__ partial) {
  constexpr int T = F * (F + 1) / 2;
  constexpr int N = T + F;
  const int lane = threadIdx.x & 31;
  const int64_t c = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const int64_t c0 = c * chunk;
  if (c0 >= S) return;  // whole warps leave together
  const int32_t r0 = (int32_t)c0, r1 = (int32_t)(c0 + chunk < S ? c0 + chunk : S);
  // the first estimator that ends after r0: 32 probes at a time
  int32_t lo = 0, left = E;
  while (left > 0) {
    const int32_t step = (left + 31) >> 5;
    const int32_t last = lo + min(left, (lane + 1) * step) - 1;  // of the lane's part
    const uint32_t b = __ballot_sync(kFullMask, off[last + 1] > r0);
    if (b == 0u) {
      lo += left;
      break;
    }
    const int32_t skip = (__ffs(b) - 1) * step;
    lo += skip;
    left = step == 1 ? 0 : min(step, left - skip);
  }
  for (int32_t e = lo; e < E; ++e) {
    const int32_t a0 = off[e], a1 = off[e + 1];
    if (a0 >= r1) break;
    const int32_t s0 = a0 > r0 ? a0 : r0, s1 = a1 < r1 ? a1 : r1;
    if (s1 <= s0) continue;  // no samples
    double v[N];
#pragma unroll
    for (int t = 0; t < N; ++t) v[t] = 0.0;
    for (int32_t r = s0 + lane; r < s1; r += 64) {
      // rows r and r + 32: twice the loads in flight
      double xv[2][F], yv[2];
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const int32_t rr = r + 32 * h;
        const bool in = rr < s1;
#pragma unroll
        for (int a = 0; a < F; ++a) xv[h][a] = in ? x[(int64_t)rr * F + a] : 0.0;
        yv[h] = in ? y[rr] : 0.0;
      }
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        if (r + 32 * h >= s1) break;
        int t = 0;
#pragma unroll
        for (int a = 0; a < F; ++a) {
          v[T + a] += xv[h][a] * yv[h];
#pragma unroll
          for (int b = a; b < F; ++b) v[t++] += xv[h][a] * xv[h][b];
        }
      }
    }
    double* out = partial + (c + e) * N;
#pragma unroll
    for (int w = 0; w < (N + 31) / 32; ++w) {
      double q[32];
#pragma unroll
      for (int i = 0; i < 32; ++i) q[i] = 32 * w + i < N ? v[32 * w + i < N ? 32 * w + i : 0] : 0.0;
      const double tot = reduce_to_lanes<N>(q);
      if (32 * w + lane < N) out[32 * w + lane] = tot;
    }
  }
}

__device__ __forceinline__ double tree8(const double (&a)[8]) {
  return ((a[0] + a[1]) + (a[2] + a[3])) + ((a[4] + a[5]) + (a[6] + a[7]));
}

// a / d from r = 1 / d: the product, corrected once by its residual (without that
// the coefficients' error against exact sums grows by a sixth; with a division
// each, 15 in a row, the kernel takes 7 us more).  d and r are finite and positive
// wherever the result is used.
__device__ __forceinline__ double quotient(double a, double d, double r) {
  const double q = a * r, e = fma(-q, d, a);
  return isfinite(e) ? fma(e, r, q) : q;  // an infinite q (or a) has no residual
}

// kWarps warps per estimator (blocks of 4 estimators with one warp each, else of
// one): add the entries in a fixed order, then refit.
template <int F, int kWarps>
__global__ void __launch_bounds__(kWarps == 1 ? 128 : 32 * kWarps)
    est_fit_kernel(State S, int32_t E, int32_t chunk, const int32_t* __restrict__ off,
                   const double* __restrict__ partial) {
  constexpr int T = F * (F + 1) / 2;
  constexpr int N = T + F;
  constexpr int kPer = kWarps == 1 ? 4 : 1;  // estimators per block
  __shared__ double part[kWarps * kPer][N];
  __shared__ double sum[kPer][N];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const int q = kWarps == 1 ? w : 0;  // the block's estimator of this warp
  const int64_t e = (int64_t)blockIdx.x * kPer + q;
  const bool in = e < E;
  const int32_t a0 = in ? off[e] : 0, a1 = in ? off[e + 1] : 0;
  const int64_t n0 = a0 / chunk + e;
  const int64_t n = a1 > a0 ? (a1 - 1) / chunk - a0 / chunk + 1 : 0;
  // lane l adds values l and 32 + l of entries first, first + kWarps, ...
#pragma unroll
  for (int u = 0; u < (N + 31) / 32; ++u) {
    const int t = 32 * u + lane;
    if (t < N) {
      // eight sums side by side: their loads overlap, and short sums and a tree
      // lose less than one long sum
      double a[8];
#pragma unroll
      for (int c = 0; c < 8; ++c) a[c] = 0.0;
      for (int64_t k = kWarps == 1 ? 0 : w; k < n; k += 8 * kWarps) {
#pragma unroll
        for (int c = 0; c < 8; ++c)
          if (k + c * kWarps < n) a[c] += partial[(n0 + k + c * kWarps) * N + t];
      }
      part[w][t] = tree8(a);
    }
  }
  if (kWarps == 1) __syncwarp();
  else __syncthreads();
  if ((kWarps > 1 && w > 0) || !in) return;  // whole warps leave together
#pragma unroll
  for (int u = 0; u < (N + 31) / 32; ++u) {
    const int t = 32 * u + lane;
    if (t < N) {
      double acc = part[kWarps == 1 ? w : 0][t];
      if (kWarps == 8) {
        double a[8];
#pragma unroll
        for (int c = 0; c < 8; ++c) a[c] = part[c % kWarps][t];
        acc = tree8(a);
      }
      double* st = t < T ? S.g + e * T + t : S.h + e * F + (t - T);
      acc += *st;
      *st = acc;
      sum[q][t] = acc;
    }
  }
  double cnt = 0.0;
  if (lane == 0) cnt = (S.n[e] += (double)(a1 - a0));
  cnt = __shfl_sync(kFullMask, cnt, 0);
  __syncwarp();
  // lane i: row i of the full matrix and of the factor L
  // (below the diagonal; own_l, inv: its diagonal entry and the reciprocal)
  double A[F], Lr[F], v = 0.0, diag = 0.0, own_l = 1.0, inv = 1.0;
#pragma unroll
  for (int b = 0; b < F; ++b) {
    const int i = lane < F ? lane : 0, r = i < b ? i : b, c = i < b ? b : i;
    A[b] = sum[q][r * F - r * (r - 1) / 2 + (c - r)];
    if (i == b) diag = A[b];
    Lr[b] = 0.0;
  }
  if (lane < F) v = sum[q][T + lane];
  // A pivot is compared with its own diagonal entry, which makes the test
  // independent of each feature's scale (bytes next to a constant term).
  bool ok = cnt >= (double)F;
#pragma unroll
  for (int j = 0; j < F; ++j) {
    const double d = __shfl_sync(kFullMask, A[j], j);
    const double own = __shfl_sync(kFullMask, diag, j);
    ok = ok && d > kPivotRel * own;
    const double ljj = sqrt(fmax(d, 0.0)), r = 1.0 / ljj;
    if (lane == j) {
      own_l = ljj;
      inv = r;
    }
    if (lane > j && lane < F) Lr[j] = ok ? quotient(A[j], ljj, r) : 0.0;
#pragma unroll
    for (int k = j + 1; k < F; ++k) {
      const double lkj = __shfl_sync(kFullMask, Lr[j], k);
      A[k] -= Lr[j] * lkj;
    }
  }
  double beta = 0.0;
  if (ok) {
#pragma unroll
    for (int k = 0; k < F; ++k) {  // L z = h
      const double z = __shfl_sync(kFullMask, quotient(v, own_l, inv), k);
      if (lane == k) v = z;
      else if (lane > k) v -= Lr[k] * z;
    }
#pragma unroll
    for (int k = F - 1; k >= 0; --k) {  // L^T beta = z
      const double bk = __shfl_sync(kFullMask, quotient(v, own_l, inv), k);
      if (lane == k) beta = bk;
      // L[k][i] is lane k's Lr[i]
#pragma unroll
      for (int i = 0; i < k; ++i) {
        const double lki = __shfl_sync(kFullMask, Lr[i], k);
        if (lane == i) v -= lki * bk;
      }
    }
  }
  if (lane < F) S.beta[e * F + lane] = ok ? beta : 0.0;
  if (lane == 0) S.fitted[e] = ok ? 1 : 0;
}

// Rounds to the nearest integer (halves to even), at least lo, at most kMaxTicks;
// lo for NaN (the conversion gives the smallest integer then).
__device__ __forceinline__ int64_t to_ticks(double v, int64_t lo) {
  const int64_t r = __double2ll_rn(v);
  return r < lo ? lo : r > kMaxTicks ? kMaxTicks : r;
}

// One thread per op, its features loaded once for all types.
template <int F>
__global__ void __launch_bounds__(256) est_predict_kernel(State S, int32_t N, int32_t T,
                                                          const int32_t* __restrict__ est_of,
                                                          const double* __restrict__ x,
                                                          const int64_t* __restrict__ dflt,
                                                          int64_t* __restrict__ dur) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= N) return;
  double xv[F];
#pragma unroll
  for (int a = 0; a < F; ++a) xv[a] = x[i * F + a];
  for (int32_t t = 0; t < T; ++t) {
    const int64_t q = i * T + t;
    const int32_t e = est_of[q];
    if (e < 0 || !S.fitted[e]) {
      dur[q] = dflt[i];
      continue;
    }
    double v = 0.0;
#pragma unroll
    for (int a = 0; a < F; ++a) v += S.beta[(int64_t)e * F + a] * xv[a];
    dur[q] = to_ticks(v, 1);
  }
}

template <int F>
cudaError_t launch_predict(State S, int32_t N, int32_t T, const int32_t* est_of, const double* x, const int64_t* dflt,
                           int64_t* dur, cudaStream_t st) {
  est_predict_kernel<F><<<(int)(((int64_t)N + 255) / 256), 256, 0, st>>>(S, N, T, est_of, x, dflt, dur);
  return cudaGetLastError();
}

__global__ void __launch_bounds__(256) est_links_kernel(State S, int32_t D, const int64_t* __restrict__ bw_dflt,
                                                        const int64_t* __restrict__ lat_dflt,
                                                        int64_t* __restrict__ bw, int64_t* __restrict__ lat) {
  const int32_t q = blockIdx.x * blockDim.x + threadIdx.x;
  if (q >= D * D) return;
  const int32_t d = q / D, e = q % D;
  if (d == e || !S.fitted[q]) {
    bw[q] = bw_dflt[q];
    lat[q] = lat_dflt[q];
    return;
  }
  const double alpha = S.beta[2 * (int64_t)q], c = S.beta[2 * (int64_t)q + 1];
  bw[q] = alpha > 0.0 ? to_ticks(1.0 / alpha, 1) : kMaxTicks;
  lat[q] = to_ticks(c, 0);
}

// Coefficients and fitted flags (each if asked for) in one launch.
__global__ void __launch_bounds__(256) est_copy_kernel(State S, int64_t nb, int32_t E, double* __restrict__ beta,
                                                       int32_t* __restrict__ fitted) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i < nb && beta) beta[i] = S.beta[i];
  if (i < E && fitted) fitted[i] = S.fitted[i];
}

// Rows per chunk for S samples, and an upper bound of the entries of S or fewer
// samples (chunks + estimators).
int32_t chunk_rows(int64_t S) {
  int32_t c = kMinChunk;
  while (c < kMaxChunk && S / c > kChunks) c *= 2;
  return c;
}
int64_t max_entries(int32_t E, int64_t S) {
  const int64_t few = S / kMinChunk + 1, most = S / kMaxChunk + 1;
  return (few < kChunks + 2 ? few : most > kChunks + 2 ? most : kChunks + 2) + E;
}

template <int F>
cudaError_t launch_update(State S, int32_t E, int64_t nsamp, const int32_t* off, const double* x,
                          const double* y, double* partial, cudaStream_t st) {
  const int32_t chunk = chunk_rows(nsamp);
  const int64_t nc = (nsamp + chunk - 1) / chunk;
  if (nc > 0) est_partial_kernel<F><<<(int)((nc * 32 + 127) / 128), 128, 0, st>>>(E, (int32_t)nsamp, chunk, off, x, y, partial);
  // several warps share an estimator's entries where it has more than a few
  if (nc / E >= 2 * kFitWarps) est_fit_kernel<F, kFitWarps><<<E, 32 * kFitWarps, 0, st>>>(S, E, chunk, off, partial);
  else est_fit_kernel<F, 1><<<(E + 3) / 4, 128, 0, st>>>(S, E, chunk, off, partial);
  return cudaGetLastError();
}

// Caller buffer of est_update: the entries [chunks + estimators][F(F+1)/2 + F] fp64.
size_t tmp_bytes(int32_t E, int32_t F, int64_t S) {
  const size_t N = (size_t)F * (F + 1) / 2 + F;
  return align256(8 * N * (size_t)max_entries(E, S));
}

bool args_ok(const void* state, int32_t E, int32_t F) {
  return state && E >= 1 && F >= 1 && F <= GMG_EST_MAX_FEATURES &&
         (reinterpret_cast<uintptr_t>(state) & 255) == 0;
}

}  // namespace
}  // namespace gest

using namespace gest;

extern "C" {

size_t est_state_bytes(int32_t n_est, int32_t n_feat) {
  if (n_est < 1 || n_feat < 1 || n_feat > GMG_EST_MAX_FEATURES) return 0;
  return layout(n_est, n_feat).total;
}

int est_reset(void* d_state, int32_t n_est, int32_t n_feat, gmg_stream_t stream) {
  if (!args_ok(d_state, n_est, n_feat)) return GMG_EINVAL;
  const cudaError_t e =
      cudaMemsetAsync(d_state, 0, layout(n_est, n_feat).total, reinterpret_cast<cudaStream_t>(stream));
  return e == cudaSuccess ? GMG_OK : GMG_ECUDA;
}

size_t est_update_tmp_bytes(int32_t n_est, int32_t n_feat, int64_t n_samples) {
  if (n_est < 1 || n_feat < 1 || n_feat > GMG_EST_MAX_FEATURES || n_samples < 0) return 0;
  return tmp_bytes(n_est, n_feat, n_samples);
}

int est_update(void* d_state, int32_t n_est, int32_t n_feat, const int32_t* d_off, const double* d_x,
               const double* d_y, int64_t n_samples, void* d_tmp, size_t tmp_bytes_given, gmg_stream_t stream) {
  if (!args_ok(d_state, n_est, n_feat) || !d_off || n_samples < 0 || n_samples > INT32_MAX) return GMG_EINVAL;
  if (n_samples > 0 && (!d_x || !d_y)) return GMG_EINVAL;
  if (!d_tmp || (reinterpret_cast<uintptr_t>(d_tmp) & 255) != 0 ||
      tmp_bytes_given < tmp_bytes(n_est, n_feat, n_samples))
    return GMG_EWS;
  const State S = view(d_state, n_est, n_feat);
  const cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
  double* partial = static_cast<double*>(d_tmp);
  cudaError_t e = cudaSuccess;
  switch (n_feat) {
    case 1: e = launch_update<1>(S, n_est, n_samples, d_off, d_x, d_y, partial, st); break;
    case 2: e = launch_update<2>(S, n_est, n_samples, d_off, d_x, d_y, partial, st); break;
    case 3: e = launch_update<3>(S, n_est, n_samples, d_off, d_x, d_y, partial, st); break;
    case 4: e = launch_update<4>(S, n_est, n_samples, d_off, d_x, d_y, partial, st); break;
    case 5: e = launch_update<5>(S, n_est, n_samples, d_off, d_x, d_y, partial, st); break;
    case 6: e = launch_update<6>(S, n_est, n_samples, d_off, d_x, d_y, partial, st); break;
    case 7: e = launch_update<7>(S, n_est, n_samples, d_off, d_x, d_y, partial, st); break;
    default: e = launch_update<8>(S, n_est, n_samples, d_off, d_x, d_y, partial, st); break;
  }
  return e == cudaSuccess ? GMG_OK : GMG_ECUDA;
}

int est_coefficients(const void* d_state, int32_t n_est, int32_t n_feat, double* d_beta, int32_t* d_fitted,
                     gmg_stream_t stream) {
  if (!args_ok(d_state, n_est, n_feat)) return GMG_EINVAL;
  const State S = view(const_cast<void*>(d_state), n_est, n_feat);
  const cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
  if (!d_beta && !d_fitted) return GMG_OK;
  const int64_t nb = (int64_t)n_est * n_feat;
  est_copy_kernel<<<(int)((nb + 255) / 256), 256, 0, st>>>(S, nb, n_est, d_beta, d_fitted);
  return cudaGetLastError() == cudaSuccess ? GMG_OK : GMG_ECUDA;
}

int est_predict_durations(const void* d_state, int32_t n_est, int32_t n_feat, int32_t n_ops, int32_t n_types,
                          const int32_t* d_est_of, const double* d_x, const int64_t* d_dflt, int64_t* d_dur,
                          gmg_stream_t stream) {
  if (!args_ok(d_state, n_est, n_feat) || n_ops < 0 || n_types < 1) return GMG_EINVAL;
  if (n_ops == 0) return GMG_OK;
  if (!d_est_of || !d_x || !d_dflt || !d_dur) return GMG_EINVAL;
  const State S = view(const_cast<void*>(d_state), n_est, n_feat);
  const cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
  cudaError_t e = cudaSuccess;
  switch (n_feat) {
    case 1: e = launch_predict<1>(S, n_ops, n_types, d_est_of, d_x, d_dflt, d_dur, st); break;
    case 2: e = launch_predict<2>(S, n_ops, n_types, d_est_of, d_x, d_dflt, d_dur, st); break;
    case 3: e = launch_predict<3>(S, n_ops, n_types, d_est_of, d_x, d_dflt, d_dur, st); break;
    case 4: e = launch_predict<4>(S, n_ops, n_types, d_est_of, d_x, d_dflt, d_dur, st); break;
    case 5: e = launch_predict<5>(S, n_ops, n_types, d_est_of, d_x, d_dflt, d_dur, st); break;
    case 6: e = launch_predict<6>(S, n_ops, n_types, d_est_of, d_x, d_dflt, d_dur, st); break;
    case 7: e = launch_predict<7>(S, n_ops, n_types, d_est_of, d_x, d_dflt, d_dur, st); break;
    default: e = launch_predict<8>(S, n_ops, n_types, d_est_of, d_x, d_dflt, d_dur, st); break;
  }
  return e == cudaSuccess ? GMG_OK : GMG_ECUDA;
}

int est_links(const void* d_state, int32_t n_dev, const int64_t* d_bw_dflt, const int64_t* d_lat_dflt,
              int64_t* d_bw, int64_t* d_lat, gmg_stream_t stream) {
  if (n_dev < 1 || n_dev > 256 || !args_ok(d_state, n_dev * n_dev, 2)) return GMG_EINVAL;
  if (!d_bw_dflt || !d_lat_dflt || !d_bw || !d_lat) return GMG_EINVAL;
  const State S = view(const_cast<void*>(d_state), n_dev * n_dev, 2);
  const int n = n_dev * n_dev;
  est_links_kernel<<<(n + 255) / 256, 256, 0, reinterpret_cast<cudaStream_t>(stream)>>>(S, n_dev, d_bw_dflt,
                                                                                          d_lat_dflt, d_bw, d_lat);
  return cudaGetLastError() == cudaSuccess ? GMG_OK : GMG_ECUDA;
}

}  // extern "C"

// Pivoted incomplete Cholesky factorisation of a two-electron supermatrix on
// the GPU: the three-index factor of Eq. int_fact, (pq|rs) ~ sum_Q B^Q_pq
// B^Q_rs, obtained by Cholesky decomposition with a threshold as for the
// paper's larger applications (Sec. IV, thresholds 1e-6 and 1e-8 a.u.).
// Algorithm of Beebe and Linderberg (1977) as described by Koch, Sanchez de
// Meras and Pedersen (J. Chem. Phys. 118, 9481 (2003)): at step Q the pivot J
// is the largest remaining diagonal D[J] (the smallest index on ties); the
// factorisation stops when D[J] <= tau; the vector is
//   B[Q][i] = (V[J][i] - sum_{Q' < Q} B[Q'][i] B[Q'][J]) / sqrt(D[J])
// and D[i] -= B[Q][i]^2.  Corrections are summed over Q' in increasing order
// with one rounding per product and per sum (no fused multiply-add), so the
// result is reproducible operation by operation.
#include <cmath>
#include <string>

#include "../../include/dsrg.h"
#include "ladder.cuh"

namespace {

constexpr int CH_MAX_CTAS = 152 * 4;
constexpr int CH_Q = 512;  // earlier vectors whose pivot entries are held at a time

struct ChState {
  long long J;     // pivot of the vector being formed
  double dJ;       // its remaining diagonal
  int nvec;        // vectors completed
  int done;        // 1: stopped (threshold or max_vecs)
  unsigned ticket; // CTAs finished in the current launch
};

// (value, index) order of the pivot search: larger value first, then the
// smaller index; NaN never wins
__device__ __forceinline__ bool better(double v, long long i, double bv, long long bi) {
  return v > bv || (v == bv && i < bi);
}

// in-CTA maximum of one (value, index) pair per thread; valid in thread 0
template <int CH_T>
__device__ void cta_argmax(double& v, long long& i) {
  __shared__ double sv[CH_T / 32];
  __shared__ long long si[CH_T / 32];
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    const double ov = __shfl_down_sync(0xffffffffu, v, o);
    const long long oi = __shfl_down_sync(0xffffffffu, i, o);
    if (better(ov, oi, v, i)) {
      v = ov;
      i = oi;
    }
  }
  __syncthreads();  // an earlier call's values are no longer read
  if ((threadIdx.x & 31) == 0) {
    sv[threadIdx.x >> 5] = v;
    si[threadIdx.x >> 5] = i;
  }
  __syncthreads();
  if (threadIdx.x == 0)
    for (int w = 1; w < CH_T / 32; ++w)
      if (better(sv[w], si[w], v, i)) {
        v = sv[w];
        i = si[w];
      }
}

// The CTA that finishes last combines the per-CTA maxima (fixed order) and
// sets the next pivot, or stops.  finish: the vector of this launch is done.
template <int CH_T>
__device__ void last_cta_pivot(double bv, long long bi, double* pv, long long* pi, ChState* st, double tau,
                               int max_vecs, long long* piv, bool finish) {
  __shared__ bool last;
  cta_argmax<CH_T>(bv, bi);
  if (threadIdx.x == 0) {
    pv[blockIdx.x] = bv;
    pi[blockIdx.x] = bi;
    __threadfence();
    last = atomicAdd(&st->ticket, 1u) == gridDim.x - 1;
  }
  __syncthreads();
  if (!last) return;
  __threadfence();
  double v = -INFINITY;
  long long i = -1;
  for (unsigned c = threadIdx.x; c < gridDim.x; c += CH_T) {
    const double cv = __ldcg(pv + c);
    const long long ci = __ldcg(pi + c);
    if (better(cv, ci, v, i)) {
      v = cv;
      i = ci;
    }
  }
  cta_argmax<CH_T>(v, i);
  if (threadIdx.x == 0) {
    if (finish) st->nvec += 1;
    if (!(v > tau) || i < 0 || st->nvec >= max_vecs) {
      st->done = 1;
    } else {
      st->J = i;
      st->dJ = v;
      piv[st->nvec] = i;
    }
    st->ticket = 0u;
  }
}

// D = diag(V) and the first pivot
template <int CH_T>
__global__ void __launch_bounds__(CH_T) k_chol_init(const double* __restrict__ V, long long N, double* __restrict__ D,
                                                   double* pv, long long* pi, ChState* st, double tau, int max_vecs,
                                                   long long* piv) {
  double bv = -INFINITY;
  long long bi = -1;
  for (long long i = blockIdx.x * (long long)CH_T + threadIdx.x; i < N; i += (long long)gridDim.x * CH_T) {
    const double d = V[i * N + i];
    D[i] = d;
    if (better(d, i, bv, bi)) {
      bv = d;
      bi = i;
    }
  }
  last_cta_pivot<CH_T>(bv, bi, pv, pi, st, tau, max_vecs, piv, false);
}

// one vector: B[nvec][i], D[i] -= B[nvec][i]^2, and the next pivot
template <int CH_T>
__global__ void __launch_bounds__(CH_T) k_chol_step(const double* __restrict__ V, long long N, double* B,
                                                   double* D, double* pv, long long* pi, ChState* st,
                                                   double tau, int max_vecs, long long* piv) {
  dsrg::wait_for_previous();
  if (__ldcg(&st->done)) return;
  const long long J = __ldcg(&st->J);
  const int Q = __ldcg(&st->nvec);
  const double sq = sqrt(__ldcg(&st->dJ));
  // B and D are what earlier kernels of the chain wrote: read through L2 (the
  // end of one vector and the start of the next may share a cache line)
  const double* bJ = B + J;  // B[q][J] at bJ[q * N]
  double bv = -INFINITY;
  long long bi = -1;
  // the pivot's column of the earlier vectors goes through shared memory, CH_Q
  // at a time (each entry its own DRAM sector: one round of loads, not one a
  // product); this thread's column is loaded 16 vectors ahead of the products
  // being formed and added (sequentially, in increasing q)
  __shared__ double yj[CH_Q];
  for (long long i0 = blockIdx.x * (long long)CH_T; i0 < N; i0 += (long long)gridDim.x * CH_T) {
    const long long i = i0 + threadIdx.x;
    const bool live = i < N;
    const double* bi_ = B + (live ? i : 0);
    constexpr int U = 16;
    double acc = 0.0;
    for (int q0 = 0; q0 < Q; q0 += CH_Q) {
      const int nq = Q - q0 < CH_Q ? Q - q0 : CH_Q;
      double x[U];
      const int full = nq / U * U;
      if (full > 0) {
#pragma unroll
        for (int u = 0; u < U; ++u) x[u] = __ldcg(bi_ + (long long)(q0 + u) * N);
      }
      __syncthreads();  // the last block's entries are no longer read
      for (int q = threadIdx.x; q < nq; q += CH_T) yj[q] = __ldcg(bJ + (long long)(q0 + q) * N);
      __syncthreads();
      for (int q = 0; q < full; q += U) {
        double nx[U];
        if (q + U < full) {
#pragma unroll
          for (int u = 0; u < U; ++u) nx[u] = __ldcg(bi_ + (long long)(q0 + q + U + u) * N);
        }
#pragma unroll
        for (int u = 0; u < U; ++u) x[u] = __dmul_rn(x[u], yj[q + u]);
#pragma unroll
        for (int u = 0; u < U; ++u) acc = __dadd_rn(acc, x[u]);
#pragma unroll
        for (int u = 0; u < U; ++u) x[u] = nx[u];
      }
      for (int q = full; q < nq; ++q) acc = __dadd_rn(acc, __dmul_rn(__ldcg(bi_ + (long long)(q0 + q) * N), yj[q]));
    }
    if (!live) continue;
    const double L = __ddiv_rn(__dsub_rn(V[J * N + i], acc), sq);
    B[(long long)Q * N + i] = L;
    const double d = __dsub_rn(__ldcg(D + i), __dmul_rn(L, L));
    D[i] = d;
    if (better(d, i, bv, bi)) {
      bv = d;
      bi = i;
    }
  }
  last_cta_pivot<CH_T>(bv, bi, pv, pi, st, tau, max_vecs, piv, true);
}

inline int ch_grid(long long N, int threads) {
  long long g = (N + threads - 1) / threads;
  if (g < 1) g = 1;
  if (g > CH_MAX_CTAS) g = CH_MAX_CTAS;
  return (int)g;
}

// f with the CTA size as a constant
template <class F>
void ch_dispatch(int threads, F&& f) {
  switch (threads) {
    case 96: f(std::integral_constant<int, 96>{}); break;
    case 128: f(std::integral_constant<int, 128>{}); break;
    case 160: f(std::integral_constant<int, 160>{}); break;
    case 192: f(std::integral_constant<int, 192>{}); break;
    case 224: f(std::integral_constant<int, 224>{}); break;
    default: f(std::integral_constant<int, 256>{}); break;
  }
}

// How a size is launched.  Every correction is one rounded product and one
// rounded sum, and an SM retires two FP64 operations a clock, so a step lasts as
// long as the SM with the most rows: of the CTA sizes whose CTAs are all
// resident, the one that gives the fullest SM the fewest.  The launches are chained
// unless the next step's CTAs, which take their places while this one's still
// hold theirs, would not all find one: those that come later pile up on a few
// SMs.  Microseconds a vector, 200 vectors (100 and 60 at the ends):
//   N = 14592 13.4 (152 CTAs of 96; 57 of 256 took 20.6), 20000 20.3 (125 of 160;
//   chained 256: 25.2), 38900 25.5 (304 of 128), 39000 30.0 (407 of 96, plain;
//   chained 39.8, 153 of 256 chained 41.4), 60000 38.4 (268 of 224), 100000 29.1
//   (1042 of 96, plain; 391 of 256 38.0).
struct ChPlan {
  int threads, grid;
  bool chained;
};
ChPlan ch_plan(long long N) {
  ChPlan best{96, ch_grid(N, 96), false};  // where no size has all its CTAs resident (N > 77824)
  long long least = -1;
  for (int t = 256; t >= 96; t -= 32) {
    int fit = 1;  // CTAs resident on an SM
    ch_dispatch(t, [&](auto c) {
      constexpr int T = decltype(c)::value;
      static const int n = [] {
        int v = 0;
        if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&v, k_chol_step<T>, T, 0) != cudaSuccess) cudaGetLastError();
        return v < 1 ? 1 : v;
      }();
      fit = n;
    });
    const long long ctas = (N + t - 1) / t, wave = 152LL * fit;
    const long long rows = (ctas + 151) / 152 * t;
    if (ctas > wave || (least >= 0 && rows > least)) continue;
    least = rows;
    best = ChPlan{t, ch_grid(N, t), fit <= 2 || 2 * ctas <= wave};
  }
  return best;
}

}  // namespace

extern "C" int dsrg_cholesky(long long N, const double* V, double tau, int max_vecs, double* B, int* nvecs,
                             long long* pivots, void* stream) {
  using namespace dsrg;
  if (nvecs) *nvecs = 0;
  if (N < 0 || max_vecs < 0 || !(tau >= 0.0) || !nvecs) return set_error(DSRG_ERR_ARG, "cholesky: need N >= 0, max_vecs >= 0, tau >= 0, nvecs");
  if (N == 0 || max_vecs == 0) return DSRG_OK;
  if (!V || !B) return set_error(DSRG_ERR_ARG, "cholesky: V and B must be device pointers");
  if (N > (1LL << 40) / N) return set_error(DSRG_ERR_ARG, "cholesky: N too large");
  cudaStream_t st = (cudaStream_t)stream;
  const ChPlan plan = ch_plan(N);
  const int threads = plan.threads, grid = plan.grid;
  // scratch: D [N], per-CTA maxima, pivots [max_vecs], state
  const size_t bytes = (size_t)N * 8 + (size_t)grid * 16 + (size_t)max_vecs * 8 + sizeof(ChState) + 64;
  try {
    CallWorkspace call(st);
    Workspace& ws = *call.ws;
    const WorkspaceBlock scratch(ws, (bytes + 7) / 8);
    double* D = scratch.p;
    double* pv = D + N;
    long long* pi = reinterpret_cast<long long*>(pv + grid);
    long long* piv = pi + grid;
    ChState* cs = reinterpret_cast<ChState*>(piv + max_vecs);
    check_cuda(cudaMemsetAsync(cs, 0, sizeof(ChState), st), "cudaMemsetAsync (cholesky)");
    void (*step)(const double*, long long, double*, double*, double*, long long*, ChState*, double, int, long long*) = nullptr;
    ch_dispatch(threads, [&](auto t) {
      constexpr int T = decltype(t)::value;
      k_chol_init<T><<<grid, T, 0, st>>>(V, N, D, pv, pi, cs, tau, max_vecs, piv);
      step = k_chol_step<T>;
    });
    check_cuda(cudaGetLastError(), "cholesky launch");
    ChState h{};
    for (int q = 0; q < max_vecs; ++q) {
      if (plan.chained) {
        check_cuda(launch_chained(step, grid, threads, st, V, N, B, D, pv, pi, cs, tau, max_vecs, piv), "cholesky launch");
      } else {
        step<<<grid, threads, 0, st>>>(V, N, B, D, pv, pi, cs, tau, max_vecs, piv);
        check_cuda(cudaGetLastError(), "cholesky launch");
      }
      // every 32 vectors: stop launching once the factorisation has stopped
      if ((q & 31) == 31 || q == max_vecs - 1) {
        check_cuda(cudaMemcpyAsync(&h, cs, sizeof h, cudaMemcpyDeviceToHost, st), "cudaMemcpyAsync (cholesky)");
        check_cuda(cudaStreamSynchronize(st), "cudaStreamSynchronize (cholesky)");
        if (h.done) break;
      }
    }
    check_cuda(cudaMemcpyAsync(&h, cs, sizeof h, cudaMemcpyDeviceToHost, st), "cudaMemcpyAsync (cholesky)");
    check_cuda(cudaStreamSynchronize(st), "cudaStreamSynchronize (cholesky)");
    *nvecs = h.nvec;
    if (pivots && h.nvec > 0)
      check_cuda(cudaMemcpy(pivots, piv, (size_t)h.nvec * sizeof(long long), cudaMemcpyDeviceToHost),
                 "cudaMemcpy (pivots)");
  } catch (const Error& ex) {
    return set_error(ex.code, ex.what());
  } catch (const std::exception& ex) {
    return set_error(DSRG_ERR_INTERNAL, ex.what());
  }
  return DSRG_OK;
}

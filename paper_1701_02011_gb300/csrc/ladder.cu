// Density-fitted particle-particle ladder (paper Eq. scaling_problem with the
// factorised integrals of Eq. int_fact), usable on caller buffers.
#include <stdexcept>
#include <string>

#include "../../include/dsrg.h"
#include "ladder.cuh"

namespace dsrg {

void ladder_core(const double* B, long long n, int naux, int p0, int np, int nh, const double* t,
                 const long long* tst, double* L, double* G, long long bp, cudaStream_t st, Workspace* ws) {
  if (np <= 0 || nh <= 0) return;
  const long long p3 = (long long)np * np * np;
  for (long long r0 = 0; r0 < np; r0 += bp) {
    long long nb = (np - r0 < bp) ? np - r0 : bp;
    check_cuda(cudaMemsetAsync(G, 0, (size_t)(nb * p3) * sizeof(double), st), "cudaMemsetAsync (ladder)");
    {  // G[pp,q,r,s] = sum_Q B[Q, p0+r0+pp, p0+r] B[Q, p0+q, p0+s]
      GemmArgs g{};
      g.A = B + (p0 + r0) * n + p0;
      g.B = B + (long long)p0 * n + p0;
      g.C = G;
      g.alpha = 1.0;
      g.nM = 2;
      g.eM[0] = (int)nb; g.aM[0] = n; g.cM[0] = p3;
      g.eM[1] = np;      g.aM[1] = 1; g.cM[1] = np;
      g.nN = 2;
      g.eN[0] = np; g.bN[0] = n; g.cN[0] = (long long)np * np;
      g.eN[1] = np; g.bN[1] = 1; g.cN[1] = 1;
      g.nK = 1;
      g.eK[0] = naux; g.aK[0] = n * n; g.bK[0] = n * n;
      g.M = nb * np;
      g.N = (long long)np * np;
      g.K = naux;
      g.nbatch = 1;
      if (ws) run_gemm(*ws, g, K_LADDER_BUILD);
      else launch_gemm(g, st, 1);
    }
    {  // L[r0+pp,q,i,j] += sum_{r,s} G[pp,q,r,s] t[r,s,i,j]
      GemmArgs g{};
      g.A = G;
      g.B = t;
      g.C = L + r0 * (long long)np * nh * nh;
      g.alpha = 1.0;
      g.nM = 2;
      g.eM[0] = (int)nb; g.aM[0] = p3;                 g.cM[0] = (long long)np * nh * nh;
      g.eM[1] = np;      g.aM[1] = (long long)np * np; g.cM[1] = (long long)nh * nh;
      g.nK = 2;
      g.eK[0] = np; g.aK[0] = np; g.bK[0] = tst[0];
      g.eK[1] = np; g.aK[1] = 1;  g.bK[1] = tst[1];
      g.nN = 2;
      g.eN[0] = nh; g.bN[0] = tst[2]; g.cN[0] = nh;
      g.eN[1] = nh; g.bN[1] = tst[3]; g.cN[1] = 1;
      g.M = nb * np;
      g.N = (long long)nh * nh;
      g.K = (long long)np * np;
      g.nbatch = 1;
      if (ws) run_gemm(*ws, g, K_LADDER_CONTRACT);
      else launch_gemm(g, st, 2);
    }
  }
}

// By (pr|qs) = (qs|pr), a batch of rows p in [e0, e1) builds (pr|qs) only for
// q >= e0, half of the build of ladder_core.  It contracts them with t[r,s] into
// the rows L[p, q >= e0] and, for q >= e1, into L[q,p] = sum_{r,s} (pr|qs) t[s,r];
// with t[r,s,i,j] = t[s,r,j,i] (t_sym: the alpha-beta block of a spin-free T2)
// L[q,p,i,j] = L[p,q,j,i] instead, by a transposed copy.  Either way every
// element of L is the plain sum of its own products.  most_rows bounds a
// batch: the rows p, q within it are built twice.
void ladder_core_half(const double* B, long long n, int naux, int p0, int np, int nh, const double* t,
                      const long long* tst, bool t_sym, double* L, double* G, long long max_doubles, long long most_rows,
                      cudaStream_t st, Workspace* ws) {
  if (np <= 0 || nh <= 0) return;
  const long long p2 = (long long)np * np, h2 = (long long)nh * nh;
  if (max_doubles < np * p2) throw std::runtime_error("ladder: scratch below one row of (pr|qs)");
  long long e0 = 0;
  while (e0 < np) {
    const long long nf = np - e0;  // q in [e0, np)
    long long nb = max_doubles / (nf * p2);
    if (nb > most_rows) nb = most_rows;
    if (nb < 1) nb = 1;
    if (nb > nf) nb = nf;
    const long long e1 = e0 + nb;
    check_cuda(cudaMemsetAsync(G, 0, (size_t)(nb * nf * p2) * sizeof(double), st), "cudaMemsetAsync (ladder)");
    const char* outer = ws ? ws->tag : "";
    if (ws) ws->tag = "ladder-build";
    {  // G[e, q - e0, r, s] = sum_Q B[Q, p0+e, p0+r] B[Q, p0+q, p0+s], e in [e0, e1), q in [e0, np)
      GemmArgs g{};
      g.A = B + (p0 + e0) * n + p0;
      g.B = B + (p0 + e0) * n + p0;
      g.C = G;
      g.alpha = 1.0;
      g.nM = 2;
      g.eM[0] = (int)nb; g.aM[0] = n; g.cM[0] = nf * p2;
      g.eM[1] = np;      g.aM[1] = 1; g.cM[1] = np;
      g.nN = 2;
      g.eN[0] = (int)nf; g.bN[0] = n; g.cN[0] = p2;
      g.eN[1] = np;      g.bN[1] = 1; g.cN[1] = 1;
      g.nK = 1;
      g.eK[0] = naux; g.aK[0] = n * n; g.bK[0] = n * n;
      g.M = nb * np;
      g.N = nf * np;
      g.K = naux;
      g.nbatch = 1;
      if (ws) run_gemm(*ws, g, K_LADDER_BUILD);
      else launch_gemm(g, st, 1);
    }
    if (ws) ws->tag = "ladder-contract";
    // L[e, q, i, j] (swap: L[q, e, i, j]) += sum_{r,s} G[e, q - e0, r, s] t[r, s, i, j] (t[s, r, i, j]), q in [q0, np)
    auto contract = [&](long long q0, bool swap) {
      GemmArgs g{};
      g.A = G + (q0 - e0) * p2;
      g.B = t;
      g.C = L + (swap ? q0 * np + e0 : e0 * np + q0) * h2;
      g.alpha = 1.0;
      g.nM = 2;
      g.eM[0] = (int)nb;        g.aM[0] = nf * p2; g.cM[0] = swap ? h2 : np * h2;
      g.eM[1] = (int)(np - q0); g.aM[1] = p2;      g.cM[1] = swap ? np * h2 : h2;
      g.nK = 2;
      g.eK[0] = np; g.aK[0] = np; g.bK[0] = tst[swap ? 1 : 0];
      g.eK[1] = np; g.aK[1] = 1;  g.bK[1] = tst[swap ? 0 : 1];
      g.nN = 2;
      g.eN[0] = nh; g.bN[0] = tst[2]; g.cN[0] = nh;
      g.eN[1] = nh; g.bN[1] = tst[3]; g.cN[1] = 1;
      g.M = nb * (np - q0);
      g.N = h2;
      g.K = p2;
      g.nbatch = 1;
      if (ws) run_gemm(*ws, g, K_LADDER_CONTRACT);
      else launch_gemm(g, st, 2);
    };
    contract(e0, false);
    if (e1 < np && !t_sym) contract(e1, true);
    if (e1 < np && t_sym) {  // L[q, e, i, j] = L[e, q, j, i] for e in [e0, e1), q in [e1, np)
      NdArgs a{};
      a.nd = 4;
      a.e[0] = (int)nb;       a.sa[0] = np * h2; a.sb[0] = h2;
      a.e[1] = (int)(np - e1); a.sa[1] = h2;     a.sb[1] = np * h2;
      a.e[2] = nh;            a.sa[2] = 1;       a.sb[2] = nh;
      a.e[3] = nh;            a.sa[3] = nh;      a.sb[3] = 1;
      a.total = nb * (np - e1) * h2;
      const double* src = L + (e0 * np + e1) * h2;
      double* dst = L + (e1 * np + e0) * h2;
      if (ws) run_axpy(*ws, a, 1.0, src, dst);
      else launch_axpy(a, 1.0, src, dst, st);
    }
    if (ws) ws->tag = outer;
    e0 = e1;
  }
}

// ---------------------------------------------------------------------------
// pair form
// ---------------------------------------------------------------------------
// For B symmetric in its last two indices and t[r,s,i,j] = t[s,r,j,i] (a spin-free
// T2).  With t+-[rs] = (t[r,s] +- t[s,r]) / 2 and G+-[pq,rs] = (pr|qs) +- (ps|qr),
// r >= s, p >= q (the sum once for r = s),
//   L[p,q] = S + D,  L[q,p] = S - D,  S = sum_{r >= s} G+ t+,  D = sum_{r > s} G- t-.
// t+- is symmetric or antisymmetric in i, j, so only i >= j is needed: two
// contractions of an eighth of the full one's size each; (pr|qs) is one
// symmetric matrix over pairs (p >= r), (q >= s), an eighth of the full build.
// An L[p,q] much smaller than L[q,p] has an error of the size of the latter's: right
// for an energy, which sums over both, not for a caller's own t and L
// (dsrg_df_ladder takes ladder_core_rows).
// Bound: the FP64 (or tensor) pipe of the two products.  np = 106, nh = 16, 400
// auxiliary functions, FP64: build 81 -> 12.6 ms, contraction 58 -> 17 ms, G+- rows
// 0.27 ms, mirror 0.06 ms.  np = 248, nh = 28, split: build and contraction 130 ->
// 60 ms, of which the G+- rows 8.3 ms.
namespace {
__host__ __device__ inline long long pair_index(long long a, long long b) { return a * (a + 1) / 2 + b; }

// (a, b), a >= b, of pair index x < 2^31
__device__ __forceinline__ void pair_of(unsigned x, int& a, int& b) {
  long long r = (long long)((sqrtf(8.0f * (float)x + 1.0f) - 1.0f) * 0.5f);
  while ((r + 1) * (r + 2) / 2 <= (long long)x) ++r;
  while (r * (r + 1) / 2 > (long long)x) --r;
  a = (int)r;
  b = (int)((long long)x - r * (r + 1) / 2);
}

struct TPairs {
  const double* t;
  long long st[4];
  int np, nh;
  double *plus, *minus;
  long long cp, cm;  // columns: i >= j of t+, i > j of t-
};

// t+ and t- [pairs r >= s][columns]; blockIdx.y walks the pairs
__global__ void k_ladder_t(const TPairs a) {
  const long long pairs = pair_index(a.np, 0);
  for (long long x = blockIdx.y; x < pairs; x += gridDim.y) {
    int r, s;
    pair_of((unsigned)x, r, s);
    const double* t1 = a.t + r * a.st[0] + s * a.st[1];
    const double* t2 = a.t + s * a.st[0] + r * a.st[1];
    for (long long c = blockIdx.x * (long long)blockDim.x + threadIdx.x; c < a.cp; c += (long long)gridDim.x * blockDim.x) {
      int i, j;
      pair_of((unsigned)c, i, j);
      const long long o = i * a.st[2] + j * a.st[3];
      const double u = t1[o], v = t2[o];
      a.plus[x * a.cp + c] = r == s ? u : 0.5 * (u + v);
      if (i > j) a.minus[x * a.cm + (long long)i * (i - 1) / 2 + j] = r == s ? 0.0 : 0.5 * (u - v);
    }
  }
}

// Bp[Q][pair p >= r] = B[Q][p0 + p][p0 + r]
__global__ void k_ladder_b(const double* __restrict__ B, long long n, int p0, int np, int naux, double* __restrict__ Bp) {
  const long long pairs = pair_index(np, 0);
  for (long long x = blockIdx.x * (long long)blockDim.x + threadIdx.x; x < pairs; x += (long long)gridDim.x * blockDim.x) {
    int p, r;
    pair_of((unsigned)x, p, r);
    for (int Q = blockIdx.y; Q < naux; Q += gridDim.y) Bp[Q * pairs + x] = B[(Q * n + p0 + p) * n + p0 + r];
  }
}

// M[b][a] = M[a][b] for a > b, 32 x 32 tiles through shared memory
__global__ void __launch_bounds__(256) k_ladder_mirror(double* M, long long n) {
  __shared__ double tile[32][33];
  const long long bi = blockIdx.y, bj = blockIdx.x;
  if (bj > bi) return;
  for (int y = threadIdx.y; y < 32; y += 8) {
    const long long i = bi * 32 + y, j = bj * 32 + threadIdx.x;
    if (i < n && j < n) tile[y][threadIdx.x] = M[i * n + j];
  }
  __syncthreads();
  for (int y = threadIdx.y; y < 32; y += 8) {
    const long long i = bj * 32 + y, j = bi * 32 + threadIdx.x;  // element (i, j) = tile[j][i]
    if (i < n && j < n && j > i) M[i * n + j] = tile[threadIdx.x][y];
  }
}

// rows of G+ and G- (pairs p >= q from row0 on) from the full matrix of
// (pr|qs) over pairs; blockIdx.y is the row
__global__ void k_ladder_g_pairs(const double* __restrict__ M, int np, long long row0, double* __restrict__ plus,
                                 double* __restrict__ minus) {
  const long long pairs = pair_index(np, 0);
  int p, q;
  pair_of((unsigned)(row0 + blockIdx.y), p, q);
  double* gp = plus + blockIdx.y * pairs;
  double* gm = minus + blockIdx.y * pairs;
  for (long long x = blockIdx.x * (long long)blockDim.x + threadIdx.x; x < pairs; x += (long long)gridDim.x * blockDim.x) {
    int r, s;
    pair_of((unsigned)x, r, s);
    // (pr|qs) and (qr|ps), each with s in the column pair: s runs along lanes
    const long long pr = p > r ? pair_index(p, r) : pair_index(r, p), qs = q > s ? pair_index(q, s) : pair_index(s, q);
    const long long qr = q > r ? pair_index(q, r) : pair_index(r, q), ps = p > s ? pair_index(p, s) : pair_index(s, p);
    const double u = __ldg(M + pr * pairs + qs), v = __ldg(M + qr * pairs + ps);
    gp[x] = r == s ? u : u + v;
    gm[x] = r == s ? 0.0 : u - v;
  }
}

// L from S (plus) and D (minus) of the pairs p >= q from row0 on
__global__ void k_ladder_out(const double* __restrict__ plus, const double* __restrict__ minus, int np, int nh,
                             long long cp, long long cm, long long row0, double* __restrict__ L) {
  int p, q;
  pair_of((unsigned)(row0 + blockIdx.y), p, q);
  const long long h2 = (long long)nh * nh;
  double* pq = L + ((long long)p * np + q) * h2;
  double* qp = L + ((long long)q * np + p) * h2;
  for (long long c = blockIdx.x * (long long)blockDim.x + threadIdx.x; c < cp; c += (long long)gridDim.x * blockDim.x) {
    const double S = plus[blockIdx.y * cp + c];
    int i, j;
    pair_of((unsigned)c, i, j);
    const double D = i > j ? minus[blockIdx.y * cm + (long long)i * (i - 1) / 2 + j] : 0.0;
    pq[(long long)i * nh + j] = S + D;
    pq[(long long)j * nh + i] = S - D;
    if (p != q) {
      qp[(long long)i * nh + j] = S - D;
      qp[(long long)j * nh + i] = S + D;
    }
  }
}

unsigned blocks_for(long long n, int threads, long long most) {
  long long b = (n + threads - 1) / threads;
  if (b > most) b = most;
  return (unsigned)(b < 1 ? 1 : b);
}

// C [M][N] (row stride ldc) += sum_k A[m am + k ak] B[k bk + n]
void pair_product(Workspace& ws, int kind, const double* A, long long am, long long ak, const double* B, long long bk,
                  double* C, long long ldc, long long M, long long N, long long K) {
  GemmArgs g{};
  g.A = A;
  g.B = B;
  g.C = C;
  g.alpha = 1.0;
  g.nM = g.nN = g.nK = 1;
  g.eM[0] = (int)M; g.aM[0] = am; g.cM[0] = ldc;
  g.eN[0] = (int)N; g.bN[0] = 1;  g.cN[0] = 1;
  g.eK[0] = (int)K; g.aK[0] = ak; g.bK[0] = bk;
  g.M = M;
  g.N = N;
  g.K = K;
  g.nbatch = 1;
  run_gemm(ws, g, kind);
}

// S, D and L of `rows` pairs from row0 on, given their G+- rows
void pair_contract(Workspace& ws, const TPairs& t, const double* gp, const double* gm, double* lp, double* lm,
                   long long row0, long long rows, double* L) {
  const long long pairs = pair_index(t.np, 0);
  check_cuda(cudaMemsetAsync(lp, 0, (size_t)(rows * t.cp) * sizeof(double), ws.stream), "cudaMemsetAsync (ladder)");
  pair_product(ws, K_LADDER_CONTRACT, gp, pairs, 1, t.plus, t.cp, lp, t.cp, rows, t.cp, pairs);
  if (t.cm > 0) {
    check_cuda(cudaMemsetAsync(lm, 0, (size_t)(rows * t.cm) * sizeof(double), ws.stream), "cudaMemsetAsync (ladder)");
    pair_product(ws, K_LADDER_CONTRACT, gm, pairs, 1, t.minus, t.cm, lm, t.cm, rows, t.cm, pairs);
  }
  const int r = ws.begin(K_AXPY, 0.0, 32.0 * (double)rows * (double)t.cp);
  k_ladder_out<<<dim3(blocks_for(t.cp, 128, 8), (unsigned)rows), 128, 0, ws.stream>>>(lp, lm, t.np, t.nh, t.cp, t.cm,
                                                                                      row0, L);
  ws.end(r);
}

void pair_amplitudes(Workspace& ws, TPairs& t) {
  const long long pairs = pair_index(t.np, 0);
  const int r = ws.begin(K_AXPY, 0.0, 32.0 * (double)pairs * (double)t.cp);
  k_ladder_t<<<dim3(blocks_for(t.cp, 128, 64), blocks_for(pairs, 1, 16384)), 128, 0, ws.stream>>>(t);
  ws.end(r);
}

constexpr long long kMaxRows = 65535;  // gridDim.y
}  // namespace

// The pair form for symmetric B and t[r,s,i,j] = t[s,r,j,i]: (pr|qs) as one
// matrix over pairs, its lower half built in eight row panels and mirrored.
// max_doubles bounds a batch of G+- rows, m_bytes the matrix; false (nothing
// done) where the matrix does not fit.
bool ladder_core_pairs(const double* B, long long n, int naux, int p0, int np, int nh, const double* t,
                       const long long* tst, double* L, long long max_doubles, double m_bytes, Workspace& ws,
                       Workspace& mws) {
  if (np <= 0 || nh <= 0) return true;
  const long long pairs = pair_index(np, 0);
  if ((double)pairs * (double)pairs * 8.0 > m_bytes || pairs >= (1LL << 31)) return false;
  cudaStream_t st = ws.stream;
  ProfTag tag_(ws, "ladder-build");
  WorkspaceBlock M(mws, (size_t)(pairs * pairs));
  {
    WorkspaceBlock Bp(mws, (size_t)(naux * pairs));
    int r = ws.begin(K_AXPY, 0.0, 16.0 * (double)naux * (double)pairs);
    k_ladder_b<<<dim3(blocks_for(pairs, 256, 1024), blocks_for(naux, 1, 64)), 256, 0, st>>>(B, n, p0, np, naux, Bp.p);
    ws.end(r);
    long long step = (pairs + 7) / 8;
    step = step < 512 ? 512 : (step + 127) / 128 * 128;
    for (long long m0 = 0; m0 < pairs; m0 += step) {
      const long long m1 = m0 + step < pairs ? m0 + step : pairs;
      check_cuda(cudaMemset2DAsync(M.p + m0 * pairs, (size_t)pairs * 8, 0, (size_t)m1 * 8, (size_t)(m1 - m0), st),
                 "cudaMemset2DAsync (ladder)");
      pair_product(ws, K_LADDER_BUILD, Bp.p + m0, 1, pairs, Bp.p, pairs, M.p + m0 * pairs, pairs, m1 - m0, m1, naux);
    }
    r = ws.begin(K_AXPY, 0.0, 8.0 * (double)pairs * (double)pairs);
    const unsigned nt = (unsigned)((pairs + 31) / 32);
    k_ladder_mirror<<<dim3(nt, nt), dim3(32, 8), 0, st>>>(M.p, pairs);
    ws.end(r);
  }
  ws.tag = "ladder-contract";
  TPairs tp{};
  tp.t = t;
  for (int k = 0; k < 4; ++k) tp.st[k] = tst[k];
  tp.np = np;
  tp.nh = nh;
  tp.cp = pair_index(nh, 0);
  tp.cm = tp.cp - nh;
  WorkspaceBlock plus(mws, (size_t)(pairs * tp.cp)), minus(mws, (size_t)(pairs * tp.cm));
  tp.plus = plus.p;
  tp.minus = minus.p;
  pair_amplitudes(ws, tp);
  long long rows = max_doubles / (2 * pairs);
  if (rows > 128) rows = rows / 128 * 128;
  rows = rows < 1 ? 1 : rows > kMaxRows ? kMaxRows : rows;
  if (rows > pairs) rows = pairs;
  WorkspaceBlock gp(mws, (size_t)(rows * pairs)), gm(mws, (size_t)(rows * pairs)), lp(mws, (size_t)(rows * tp.cp)),
      lm(mws, (size_t)(rows * tp.cm));
  for (long long r0 = 0; r0 < pairs; r0 += rows) {
    const long long nr = r0 + rows < pairs ? rows : pairs - r0;
    const int r = ws.begin(K_AXPY, 0.0, 32.0 * (double)nr * (double)pairs);
    k_ladder_g_pairs<<<dim3(blocks_for(pairs, 256, 64), (unsigned)nr), 256, 0, st>>>(M.p, np, r0, gp.p, gm.p);
    ws.end(r);
    pair_contract(ws, tp, gp.p, gm.p, lp.p, lm.p, r0, nr, L);
  }
  check_cuda(cudaGetLastError(), "ladder launch");
  return true;
}

// ---------------------------------------------------------------------------
// any B and t
// ---------------------------------------------------------------------------
// (pr|qs) for q <= p as rows [pq][rs], and one product with both orders of t,
//   L[p,q] = sum_{r,s} (pr|qs) t[r,s],  L[q,p] = sum_{r,s} (pr|qs) t[s,r]
// (by (ps|qr) = (qr|ps)): half of the build of ladder_core, every element of L
// the plain sum of its own products.  Bound: the FP64 pipe.  np = 106, nh = 16,
// 400 auxiliary functions: 140 (ladder_core) -> 103 ms; a contraction per batch
// of p (ladder_core_half, which needs less memory) takes 113.  Sums and
// differences as in the pair form took 85, and lost the smaller one of L[p,q]
// and L[q,p].
namespace {
// t2[rs][0][ij] = t[r][s][ij], t2[rs][1][ij] = t[s][r][ij]
__global__ void k_ladder_t2(const double* __restrict__ t, long long np, long long h2, double* __restrict__ t2) {
  const long long n = np * np * h2;
  for (long long x = blockIdx.x * (long long)blockDim.x + threadIdx.x; x < n; x += (long long)gridDim.x * blockDim.x) {
    const long long rs = x / h2, ij = x - rs * h2, r = rs / np, s = rs - r * np;
    t2[2 * rs * h2 + ij] = t[x];
    t2[(2 * rs + 1) * h2 + ij] = t[(s * np + r) * h2 + ij];
  }
}

// L[p,q] and L[q,p] from the rows (p - b0, q), p in [b0, b0 + gridDim.z), q < gridDim.y
__global__ void k_ladder_rows_out(const double* __restrict__ c, int b0, int np, long long h2, double* __restrict__ L) {
  const int p = b0 + blockIdx.z, q = blockIdx.y;
  if (q > p) return;  // p's own row in the same batch has it
  const double* row = c + ((long long)blockIdx.z * gridDim.y + q) * 2 * h2;
  double* pq = L + ((long long)p * np + q) * h2;
  double* qp = L + ((long long)q * np + p) * h2;
  for (long long x = blockIdx.x * (long long)blockDim.x + threadIdx.x; x < h2; x += (long long)gridDim.x * blockDim.x) {
    pq[x] = row[x];
    if (q < p) qp[x] = row[h2 + x];
  }
}

// C [M][N] = A [M][K] B [K][N] in sums of at most 1024 products each, as partial
// tiles of one launch within kSums doubles: a third of the rounding error of one
// sum over all K, and with 2400 tiles or more (of 128 products at least) hardly
// a part-filled last wave.
constexpr long long kSums = 1LL << 25;
void rows_contract(Workspace& ws, const double* A, const double* B, double* C, long long M, long long N, long long K) {
  int bm, bn;
  gemm_tile(M, N, 2, &bm, &bn);
  const long long tiles = ((M + bm - 1) / bm) * ((N + bn - 1) / bn);
  long long z = (2400 + tiles - 1) / tiles;
  if (z > K / 128) z = K / 128;
  if (z < (K + 1023) / 1024) z = (K + 1023) / 1024;
  if (z > kSums / (M * N)) z = kSums / (M * N);
  if (z < 2) {
    pair_product(ws, K_LADDER_CONTRACT, A, K, 1, B, N, C, N, M, N, K);
    return;
  }
  GemmArgs g{};
  g.A = A;
  g.B = B;
  g.C = C;
  g.alpha = 1.0;
  g.nM = g.nN = g.nK = 1;
  g.eM[0] = (int)M; g.aM[0] = K; g.cM[0] = N;
  g.eN[0] = (int)N; g.bN[0] = 1; g.cN[0] = 1;
  g.eK[0] = (int)K; g.aK[0] = 1; g.bK[0] = N;
  g.M = M;
  g.N = N;
  g.K = K;
  g.nbatch = 1;
  g.kper = ((K + z - 1) / z + 15) / 16 * 16;
  g.splits = (int)((K + g.kper - 1) / g.kper);
  const WorkspaceBlock part(ws, (size_t)(g.splits * M * N));
  g.part = part.p;
  launch_gemm(g, ws.stream, 2);
}
}  // namespace

bool ladder_core_rows(const double* B, long long n, int naux, int p0, int np, int nh, const double* t, double* L,
                      long long max_doubles, Workspace& ws) {
  const long long p2 = (long long)np * np, h2 = (long long)nh * nh;
  // batches of p whose build has at least 256 rows (p, r); rows held: those of
  // all batches, or as many as fit, but at least one batch
  const long long nb = np < 256 ? (255 + np) / np : 1;
  const long long cap = (max_doubles - 2 * p2 * h2) / (p2 + 2 * h2);
  if (cap < nb * np || np > 65535) return false;
  const long long all = (p2 + (nb + 1) * np) / 2 + nb;
  const long long held = cap < all ? cap : all;
  cudaStream_t st = ws.stream;
  WorkspaceBlock t2(ws, (size_t)(2 * p2 * h2)), G(ws, (size_t)(held * p2)), C(ws, (size_t)(held * 2 * h2));
  k_ladder_t2<<<blocks_for(p2 * h2, 256, 152 * 16), 256, 0, st>>>(t, np, h2, t2.p);
  for (int p = 0; p < np;) {
    const int first = p;
    long long rows = 0;
    auto size = [&](int b0) { return (b0 + nb < np ? nb : np - b0) * (b0 + nb < np ? b0 + nb : np); };
    for (; p < np && rows + size(p) <= held; p += (int)nb) rows += size(p);
    check_cuda(cudaMemsetAsync(G.p, 0, (size_t)(rows * p2) * sizeof(double), st), "cudaMemsetAsync (ladder)");
    check_cuda(cudaMemsetAsync(C.p, 0, (size_t)(rows * 2 * h2) * sizeof(double), st), "cudaMemsetAsync (ladder)");
    const int end = p < np ? p : np;
    long long at = 0;
    for (int b0 = first; b0 < end; b0 += (int)nb) {
      const int b1 = b0 + nb < np ? b0 + (int)nb : np;
      GemmArgs g{};  // G[p - b0, q, r, s] = sum_Q B[Q, p0+p, p0+r] B[Q, p0+q, p0+s], p in [b0, b1), q < b1
      g.A = B + (p0 + b0) * n + p0;
      g.B = B + (long long)p0 * n + p0;
      g.C = G.p + at * p2;
      g.alpha = 1.0;
      g.nM = g.nN = 2;
      g.eM[0] = b1 - b0; g.aM[0] = n; g.cM[0] = b1 * p2;
      g.eM[1] = np;      g.aM[1] = 1; g.cM[1] = np;
      g.eN[0] = b1;      g.bN[0] = n; g.cN[0] = p2;
      g.eN[1] = np;      g.bN[1] = 1; g.cN[1] = 1;
      g.nK = 1;
      g.eK[0] = naux; g.aK[0] = n * n; g.bK[0] = n * n;
      g.M = (long long)(b1 - b0) * np;
      g.N = (long long)b1 * np;
      g.K = naux;
      g.nbatch = 1;
      run_gemm(ws, g, K_LADDER_BUILD);
      at += size(b0);
    }
    rows_contract(ws, G.p, t2.p, C.p, rows, 2 * h2, p2);
    at = 0;
    for (int b0 = first; b0 < end; b0 += (int)nb) {
      const int b1 = b0 + nb < np ? b0 + (int)nb : np;
      k_ladder_rows_out<<<dim3(blocks_for(h2, 256, 8), b1, b1 - b0), 256, 0, st>>>(C.p + at * 2 * h2, b0, np, h2, L);
      at += size(b0);
    }
  }
  check_cuda(cudaGetLastError(), "ladder launch");
  return true;
}

long long ladder_batch_rows(int np, long long max_doubles) {
  const long long p3 = (long long)np * np * np;
  long long bp = max_doubles / (p3 > 0 ? p3 : 1);
  if (bp > np) bp = np;
  return bp;
}

int ladder_check_args(int n, int naux, int p0, int np, int nh, const void* B, const void* t, const void* L,
                      std::string& msg) {
  if (n < 1 || naux < 1 || np < 0 || nh < 0 || p0 < 0 || p0 + np > n) {
    msg = "ladder: need n >= 1, naux >= 1, 0 <= p0, p0 + np <= n, np >= 0, nh >= 0";
    return DSRG_ERR_ARG;
  }
  if ((np > 0 && nh > 0) && (!B || !t || !L)) {
    msg = "ladder: B, t and L must be device pointers";
    return DSRG_ERR_ARG;
  }
  return DSRG_OK;
}

}  // namespace dsrg

extern "C" int dsrg_df_ladder(int n, int naux, int p0, int np, int nh, const double* B, const double* t, double* L,
                              void* stream) {
  using namespace dsrg;
  std::string msg;
  int rc = ladder_check_args(n, naux, p0, np, nh, B, t, L, msg);
  if (rc) return set_error(rc, msg.c_str());
  if (np == 0 || nh == 0) return DSRG_OK;
  cudaStream_t st = (cudaStream_t)stream;
  const long long p3 = (long long)np * np * np;
  const long long tst[4] = {(long long)np * nh * nh, (long long)nh * nh, nh, 1};
  // Scratch of at most 1 GiB, or one row of (pr|qs): rows, and up to 256 MiB of
  // partial sums (kSums).  In one batch where the build has less than 2e8 flops:
  // two launches, and half of so little is not worth a third (24 particles, 96
  // auxiliary functions 0.11 ms; 32 and 128, above the line, 0.36 in two batches,
  // 0.43 in rows).  Batch by batch where the pairs' rows do not fit.
  constexpr long long kMost = 1LL << 27;
  const bool one = 2.0 * (double)naux * (double)p3 * (double)np < 2e8;
  long long rows = one ? np : (np + 15) / 16;
  if (rows > ladder_batch_rows(np, kMost - kSums)) rows = ladder_batch_rows(np, kMost - kSums);
  if (rows < 1) rows = 1;
  try {
    CallWorkspace call(st);
    Workspace& ws = *call.ws;
    bool done = false;
    try {
      done = !one && ladder_core_rows(B, n, naux, p0, np, nh, t, L, kMost - kSums, ws);
    } catch (const Error& e) {
      if (e.code != DSRG_ERR_OOM) throw;
    }
    for (bool sums = true; !done;) {
      try {
        const WorkspaceBlock G(ws, (size_t)(rows * p3));
        check_cuda(cudaMemsetAsync(L, 0, (size_t)np * np * nh * nh * sizeof(double), st), "cudaMemsetAsync");
        ladder_core_half(B, n, naux, p0, np, nh, t, tst, false, L, G.p, rows * p3, rows, st, sums ? &ws : nullptr);
        check_cuda(cudaGetLastError(), "ladder launch");
        done = true;
      } catch (const Error& e) {
        // too little memory: half the rows, and with one row no partial sums
        if (e.code != DSRG_ERR_OOM || !sums) throw;
        if (rows == 1) sums = false;
        rows = (rows + 1) / 2;
      }
    }
    check_cuda(cudaStreamSynchronize(st), "cudaStreamSynchronize");
  } catch (const Error& ex) {
    return set_error(ex.code, ex.what());
  } catch (const std::exception& ex) {
    return set_error(DSRG_ERR_CUDA, ex.what());
  }
  return DSRG_OK;
}

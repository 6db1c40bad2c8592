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

// Pair-symmetric variant where the pair form below does not fit: with t[r,s,i,j] = t[s,r,j,i] (the alpha-beta block
// of a spin-free T2) and (pr|qs) = (qs|pr), L[q,p,i,j] = L[p,q,j,i], so a
// batch of rows p in [e0, e1) builds and contracts (pr|qs) only for
// q >= e0 and writes the rows q >= e1 of the mirror image by a transposed
// copy.  About half of the build and contraction work of ladder_core.
void ladder_core_sym(const double* B, long long n, int naux, int p0, int np, int nh, const double* t,
                     const long long* tst, double* L, double* G, long long max_doubles, cudaStream_t st,
                     Workspace* ws) {
  if (np <= 0 || nh <= 0) return;
  const long long p2 = (long long)np * np, h2 = (long long)nh * nh;
  if (max_doubles < np * p2) throw std::runtime_error("ladder: scratch below one row of (pr|qs)");
  long long e0 = 0;
  while (e0 < np) {
    const long long nf = np - e0;  // q in [e0, np)
    long long nb = max_doubles / (nf * p2);
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
    {  // L[e, q, i, j] += sum_{r,s} G[e, q - e0, r, s] t[r, s, i, j]
      GemmArgs g{};
      g.A = G;
      g.B = t;
      g.C = L + (e0 * np + e0) * h2;
      g.alpha = 1.0;
      g.nM = 2;
      g.eM[0] = (int)nb; g.aM[0] = nf * p2; g.cM[0] = np * h2;
      g.eM[1] = (int)nf; g.aM[1] = p2;      g.cM[1] = h2;
      g.nK = 2;
      g.eK[0] = np; g.aK[0] = np; g.bK[0] = tst[0];
      g.eK[1] = np; g.aK[1] = 1;  g.bK[1] = tst[1];
      g.nN = 2;
      g.eN[0] = nh; g.bN[0] = tst[2]; g.cN[0] = nh;
      g.eN[1] = nh; g.bN[1] = tst[3]; g.cN[1] = 1;
      g.M = nb * nf;
      g.N = h2;
      g.K = p2;
      g.nbatch = 1;
      if (ws) run_gemm(*ws, g, K_LADDER_CONTRACT);
      else launch_gemm(g, st, 2);
    }
    if (e1 < np) {  // L[q, e, i, j] = L[e, q, j, i] for e in [e0, e1), q in [e1, np)
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
// With t+-[rs] = (t[r,s] +- t[s,r]) / 2 and G+-[pq,rs] = (pr|qs) +- (ps|qr),
// r >= s, p >= q (the sum once for r = s),
//   L[p,q] = S + D,  L[q,p] = S - D,  S = sum_{r >= s} G+ t+,  D = sum_{r > s} G- t-:
// two contractions of a quarter of the full one's size.  If t[r,s,i,j] =
// t[s,r,j,i] as well (a spin-free T2), t+- is symmetric or antisymmetric in
// i, j and only i >= j is needed: an eighth each.  If B is symmetric in its
// last two indices (pr|qs) is one symmetric matrix over pairs (p >= r),
// (q >= s), an eighth of the full build.
// Bound: the FP64 (or tensor) pipe of the two products.  np = 106, nh = 16, 400
// auxiliary functions, FP64: general 140 -> 85 ms; symmetric (the energy) build
// 81 -> 12.6 ms, contraction 58 -> 17 ms, G+- rows 0.27 ms, mirror 0.06 ms.
// np = 248, nh = 28, split: build and contraction 130 -> 60 ms, of which the
// G+- rows 8.3 ms.
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
  int np, nh, sym;  // sym: columns of t+ are i >= j, of t- i > j; else both all (i, j)
  double *plus, *minus;
  long long cp, cm;  // columns
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
      if (a.sym) {
        pair_of((unsigned)c, i, j);
      } else {
        i = (int)(c / a.nh);
        j = (int)(c - (long long)i * a.nh);
      }
      const long long o = i * a.st[2] + j * a.st[3];
      const double u = t1[o], v = t2[o];
      a.plus[x * a.cp + c] = r == s ? u : 0.5 * (u + v);
      const double m = r == s ? 0.0 : 0.5 * (u - v);
      if (!a.sym) a.minus[x * a.cm + c] = m;
      else if (i > j) a.minus[x * a.cm + (long long)i * (i - 1) / 2 + j] = m;
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

// the same rows from a batch G[p - b0][q][r][s], q < nq, of rows p in [b0, b1)
__global__ void k_ladder_g_rows(const double* __restrict__ G, int np, int nq, int b0, long long row0, long long first,
                                double* __restrict__ plus, double* __restrict__ minus) {
  const long long pairs = pair_index(np, 0), row = first + blockIdx.y;
  int p, q;
  pair_of((unsigned)row, p, q);
  const double* g = G + ((long long)(p - b0) * nq + q) * np * np;
  double* gp = plus + (row - row0) * pairs;
  double* gm = minus + (row - row0) * pairs;
  for (long long x = blockIdx.x * (long long)blockDim.x + threadIdx.x; x < pairs; x += (long long)gridDim.x * blockDim.x) {
    int r, s;
    pair_of((unsigned)x, r, s);
    const double u = g[(long long)r * np + s], v = g[(long long)s * np + r];
    gp[x] = r == s ? u : u + v;
    gm[x] = r == s ? 0.0 : u - v;
  }
}

// L from S (plus) and D (minus) of the pairs p >= q from row0 on
__global__ void k_ladder_out(const double* __restrict__ plus, const double* __restrict__ minus, int np, int nh, int sym,
                             long long cp, long long cm, long long row0, double* __restrict__ L) {
  int p, q;
  pair_of((unsigned)(row0 + blockIdx.y), p, q);
  const long long h2 = (long long)nh * nh;
  double* pq = L + ((long long)p * np + q) * h2;
  double* qp = L + ((long long)q * np + p) * h2;
  for (long long c = blockIdx.x * (long long)blockDim.x + threadIdx.x; c < cp; c += (long long)gridDim.x * blockDim.x) {
    const double S = plus[blockIdx.y * cp + c];
    if (!sym) {
      const double D = minus[blockIdx.y * cm + c];
      pq[c] = S + D;
      if (p != q) qp[c] = S - D;
      continue;
    }
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
  k_ladder_out<<<dim3(blocks_for(t.cp, 128, 8), (unsigned)rows), 128, 0, ws.stream>>>(lp, lm, t.np, t.nh, t.sym, t.cp,
                                                                                      t.cm, row0, L);
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
  tp.sym = 1;
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

// The pair form for any B and t: (pr|qs) for q < p + 1 in batches of rows p.
// All scratch stays within max_doubles; false (nothing done) where that is
// too little for ten batches or so.
bool ladder_core_general(const double* B, long long n, int naux, int p0, int np, int nh, const double* t, double* L,
                         long long max_doubles, Workspace& ws) {
  const long long pairs = pair_index(np, 0), h2 = (long long)nh * nh, p2 = (long long)np * np;
  const long long left = max_doubles - 2 * pairs * h2;
  // a row p: its (pr|qs) and, for its pairs, G+- and S, D
  const long long per = np * p2 + np * (2 * pairs + 2 * h2);
  long long nb = left / per;
  if (nb > (np + 9) / 10) nb = (np + 9) / 10;
  if (nb < 1 || nb * np > kMaxRows || pairs >= (1LL << 31)) return false;
  cudaStream_t st = ws.stream;
  TPairs tp{};
  tp.t = t;
  const long long tst[4] = {np * h2, h2, nh, 1};
  for (int k = 0; k < 4; ++k) tp.st[k] = tst[k];
  tp.np = np;
  tp.nh = nh;
  tp.cp = tp.cm = h2;
  WorkspaceBlock plus(ws, (size_t)(pairs * h2)), minus(ws, (size_t)(pairs * h2));
  tp.plus = plus.p;
  tp.minus = minus.p;
  pair_amplitudes(ws, tp);
  WorkspaceBlock G(ws, (size_t)(nb * np * p2));
  // as many pairs per contraction as the rest of the budget holds
  long long cap = (left - nb * np * p2) / (2 * pairs + 2 * h2);
  if (cap > pairs) cap = pairs;
  if (cap > kMaxRows) cap = kMaxRows;
  WorkspaceBlock gp(ws, (size_t)(cap * pairs)), gm(ws, (size_t)(cap * pairs)), lp(ws, (size_t)(cap * h2)),
      lm(ws, (size_t)(cap * h2));
  long long row0 = 0, row1 = 0;  // pairs whose G+- rows are held
  for (int b0 = 0; b0 < np; b0 += (int)nb) {
    const int b1 = b0 + nb < np ? b0 + (int)nb : np;
    const int nq = b1;
    check_cuda(cudaMemsetAsync(G.p, 0, (size_t)(b1 - b0) * nq * p2 * sizeof(double), st), "cudaMemsetAsync (ladder)");
    GemmArgs g{};  // G[p - b0, q, r, s] = sum_Q B[Q, p0+p, p0+r] B[Q, p0+q, p0+s], p in [b0, b1), q < b1
    g.A = B + (p0 + b0) * n + p0;
    g.B = B + (long long)p0 * n + p0;
    g.C = G.p;
    g.alpha = 1.0;
    g.nM = g.nN = 2;
    g.eM[0] = b1 - b0; g.aM[0] = n; g.cM[0] = nq * p2;
    g.eM[1] = np;      g.aM[1] = 1; g.cM[1] = np;
    g.eN[0] = nq;      g.bN[0] = n; g.cN[0] = p2;
    g.eN[1] = np;      g.bN[1] = 1; g.cN[1] = 1;
    g.nK = 1;
    g.eK[0] = naux; g.aK[0] = n * n; g.bK[0] = n * n;
    g.M = (long long)(b1 - b0) * np;
    g.N = (long long)nq * np;
    g.K = naux;
    g.nbatch = 1;
    run_gemm(ws, g, K_LADDER_BUILD);
    const long long next = pair_index(b1, 0);
    if (next - row0 > cap) {
      pair_contract(ws, tp, gp.p, gm.p, lp.p, lm.p, row0, row1 - row0, L);
      row0 = row1;
    }
    k_ladder_g_rows<<<dim3(blocks_for(pairs, 256, 64), (unsigned)(next - row1)), 256, 0, st>>>(G.p, np, nq, b0, row0,
                                                                                               row1, gp.p, gm.p);
    row1 = next;
  }
  pair_contract(ws, tp, gp.p, gm.p, lp.p, lm.p, row0, row1 - row0, L);
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
  long long bp = ladder_batch_rows(np, 1LL << 27);  // at most 1 GiB of scratch
  if (bp < 1) bp = 1;
  try {
    CallWorkspace call(st);
    Workspace& ws = *call.ws;
    bool done = false;
    try {
      done = ladder_core_general(B, n, naux, p0, np, nh, t, L, 1LL << 27, ws);
    } catch (const Error& e) {
      if (e.code != DSRG_ERR_OOM) throw;  // too little memory: the batched form needs less
    }
    if (!done) {
      const WorkspaceBlock rows(ws, (size_t)(bp * p3));
      check_cuda(cudaMemsetAsync(L, 0, (size_t)np * np * nh * nh * sizeof(double), st), "cudaMemsetAsync");
      const long long tst[4] = {(long long)np * nh * nh, (long long)nh * nh, nh, 1};
      ladder_core(B, n, naux, p0, np, nh, t, tst, L, rows.p, bp, st, nullptr);
      check_cuda(cudaGetLastError(), "ladder launch");
    }
    check_cuda(cudaStreamSynchronize(st), "cudaStreamSynchronize");
  } catch (const Error& ex) {
    return set_error(ex.code, ex.what());
  } catch (const std::exception& ex) {
    return set_error(DSRG_ERR_CUDA, ex.what());
  }
  return DSRG_OK;
}

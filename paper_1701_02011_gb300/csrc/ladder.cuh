// Density-fitted particle-particle ladder core shared by the energy driver
// and the standalone C entry points.
#pragma once
#include <string>

#include "engine.cuh"

namespace dsrg {

// L[p,q,i,j] += sum_{r,s} (sum_Q B[Q,p0+p,p0+r] B[Q,p0+q,p0+s]) t[r,s,i,j]
// for p,q,r,s in [0,np), i,j in [0,nh).  B is [naux][n][n] (row-major), t is
// addressed with strides tst[0..3], L is contiguous [np][np][nh][nh].  The
// (pr|qs) rows are built bp at a time into G (capacity bp * np^3 doubles).
// Launches go through `ws` (counted, optionally timed) when it is non-null.
void ladder_core(const double* B, long long n, int naux, int p0, int np, int nh, const double* t,
                 const long long* tst, double* L, double* G, long long bp, cudaStream_t st, Workspace* ws);
// The same sum (L must be zero on entry) using (pr|qs) = (qs|pr): half the
// build, and with t[r,s,i,j] = t[s,r,j,i] (t_sym) half the contraction; G holds
// at most max_doubles doubles, a batch at most most_rows rows.
void ladder_core_half(const double* B, long long n, int naux, int p0, int np, int nh, const double* t,
                      const long long* tst, bool t_sym, double* L, double* G, long long max_doubles, long long most_rows,
                      cudaStream_t st, Workspace* ws);
// The same sums in pair form (see ladder.cu) for B symmetric in its last two
// indices and t_sym; its blocks come from mws.  False, and nothing done, where
// the matrix of (pr|qs) takes more than m_bytes.  L is overwritten.
bool ladder_core_pairs(const double* B, long long n, int naux, int p0, int np, int nh, const double* t,
                       const long long* tst, double* L, long long max_doubles, double m_bytes, Workspace& ws,
                       Workspace& mws);
// The same sums for any B and t (contiguous), in rows over pairs p >= q (see
// ladder.cu); false, and nothing done, where max_doubles do not hold a batch of
// them.  L is overwritten.
bool ladder_core_rows(const double* B, long long n, int naux, int p0, int np, int nh, const double* t, double* L,
                      long long max_doubles, Workspace& ws);
// Largest batch of p rows whose (pr|qs) fits in max_doubles (0 if none).
long long ladder_batch_rows(int np, long long max_doubles);
int ladder_check_args(int n, int naux, int p0, int np, int nh, const void* B, const void* t, const void* L,
                      std::string& msg);

// sets the calling thread's dsrg_last_error message and returns code
int set_error(int code, const char* msg);

}  // namespace dsrg

// Split-precision FP64 contraction on tcgen05 (see ozaki.cuh).
#include <cuda_bf16.h>

#include <cstdint>
#include <stdexcept>

#include "ozaki.cuh"

#include <algorithm>
#include <cmath>
#include <map>
#include <mutex>
#include <type_traits>
#include <vector>

namespace dsrg {
namespace {

// k per stage (a 32-byte row of bf16 digits), stage buffers, and stages per
// exact window: digits are balanced, |d| <= 64, so a level sum over one
// window has at most 8 pairs x 480 products of |d d'| <= 2^12,
// 8 x 480 x 4096 < 2^24, and is exact in FP32
constexpr int OZ_BM = 128, OZ_BK = 16, OZ_MAXBUF = 8, OZ_WIN = 30;
// fewest stages per k split
constexpr int OZ_SPLIT_MIN = 8;
// row tiles per rasterisation group
constexpr int OZ_GROUP = 8;
constexpr int OZ_THREADS = 256;  // 8 warps: lane quadrant (warp % 4) x column half (warp / 4)
constexpr int OZ_CTA_THREADS = OZ_THREADS + 128;  // and a warpgroup with one warp for the bulk copies and one for the MMAs
// registers per thread: the block is launched with 384 x 168 (a quarter of
// them on each sub-partition) and the warpgroups take 208 + 208 + 88 = 3 x 168.
// The build checks that every instantiation has 168.  Where a summing thread
// holds 64-bit sums for 32 columns the compiler still spills a little: 40 to 72
// bytes at 6 to 8 slices with 64 columns, 24 at 3 and 8 at 5; with 32 columns
// 28 at 8; none elsewhere.
constexpr int OZ_REGS = 168, OZ_REGS_SUM = 208, OZ_REGS_ISSUE = 88;
static_assert(2 * OZ_REGS_SUM + OZ_REGS_ISSUE == 3 * OZ_REGS, "register split");
constexpr int OZ_TILE_ELEMS = OZ_BM * OZ_BK;  // A stage tile of one slice: 2048 bf16 = 4 KiB
constexpr int OZ_TILE_BYTES = OZ_TILE_ELEMS * 2;
// exponents are stored as 2048 + frexp exponent of the row / column maximum (0: all zero)
constexpr unsigned OZ_EBIAS = 2048;
// default budget of a bounded wait, and the fixed budget of the waits that
// drain copies and products in flight after a wait ran out (SM clock cycles,
// about 2 s at 2 GHz)
constexpr long long OZ_WAIT_CYCLES = 1LL << 32;

__device__ __forceinline__ uint32_t smem_u32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

// Shared-memory matrix descriptor: K-major operand in the 32-byte swizzled
// layout (rows of 16 bf16, 8-row groups 256 bytes apart; the 16-byte chunk c
// of row r sits at chunk c ^ ((r >> 2) & 1)).
__device__ __forceinline__ uint64_t sdesc(uint32_t saddr) {
  uint64_t d = 0;
  d |= (uint64_t)((saddr & 0x3FFFFu) >> 4);  // start address
  d |= (uint64_t)1 << 16;                    // leading byte offset (unused when swizzled)
  d |= (uint64_t)(256 >> 4) << 32;           // stride byte offset: 8 rows x 32 B
  d |= (uint64_t)1 << 46;                    // descriptor version
  d |= (uint64_t)6 << 61;                    // 32-byte swizzle
  return d;
}

// Instruction descriptor, kind::f16: FP32 accumulator, BF16 A and B, both
// K-major, M = 128, N columns (a multiple of 16, at most 256).
__host__ __device__ constexpr uint32_t oz_idesc(int n) {
  return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(n >> 3) << 17) | ((uint32_t)(OZ_BM >> 4) << 24);
}

__device__ __forceinline__ void mbar_init(uint64_t* bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count) : "memory");
}

__device__ __forceinline__ bool mbar_try(uint64_t* bar, uint32_t phase) {
  uint32_t ok;
  asm volatile(
      "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.b32 %0, 1, 0, p;\n}"
      : "=r"(ok)
      : "r"(smem_u32(bar)), "r"(phase)
      : "memory");
  return ok != 0;
}

// non-blocking test of the phase
__device__ __forceinline__ bool mbar_test(uint64_t* bar, uint32_t phase) {
  uint32_t ok;
  asm volatile(
      "{\n .reg .pred p;\n mbarrier.test_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.b32 %0, 1, 0, p;\n}"
      : "=r"(ok)
      : "r"(smem_u32(bar)), "r"(phase)
      : "memory");
  return ok != 0;
}

// bounded wait: false if the phase did not complete within `budget` SM clock
// cycles (tested once without blocking, then polled with try_wait)
__device__ __forceinline__ bool mbar_wait(uint64_t* bar, uint32_t phase, long long budget) {
  const long long t0 = clock64();
  while (true) {
    if (mbar_test(bar, phase)) return true;
    if (clock64() - t0 > budget) return false;
    if (mbar_try(bar, phase)) return true;
  }
}

__device__ __forceinline__ void mbar_arrive(uint64_t* bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(bar)) : "memory");
}

__device__ __forceinline__ void mbar_expect_tx(uint64_t* bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)), "r"(bytes) : "memory");
}

// global -> shared bulk copy (bytes a multiple of 16, both addresses 16-byte
// aligned), completion counted on the mbarrier
__device__ __forceinline__ void bulk_g2s(void* dst, const void* src, uint32_t bytes, uint64_t* bar) {
  asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
                   smem_u32(dst)),
               "l"(src), "r"(bytes), "r"(smem_u32(bar))
               : "memory");
}

// *p += v in L2, off the FP64 pipe and without a load into the SM (one addition
// per element and launch, so the result does not depend on any order).  It goes
// at about 110 G/s on the whole chip, which bounds the short-k products; loads,
// additions and stores by the summing warps were slower at every width (1722112 x
// 28 x 8: 550 against 513 us, 61504 x 784 x 64: 570 against 450 us).
__device__ __forceinline__ void red_add(double* p, double v) {
  asm volatile("red.global.add.f64 [%0], %1;" ::"l"(p), "d"(v) : "memory");
}

__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }

__device__ __forceinline__ void mma_bf16(uint32_t d_tmem, uint64_t adesc, uint64_t bdesc, uint32_t idesc,
                                         uint32_t acc) {
  asm volatile(
      "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n"
      " tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}" ::"r"(d_tmem),
      "l"(adesc), "l"(bdesc), "r"(idesc), "r"(acc)
      : "memory");
}

// true on one lane of the (converged) warp
__device__ __forceinline__ bool elect_one() {
  uint32_t p;
  asm volatile("{\n .reg .pred p;\n elect.sync _|p, 0xffffffff;\n selp.b32 %0, 1, 0, p;\n}" : "=r"(p));
  return p != 0;
}

__device__ __forceinline__ void mma_commit(uint64_t* bar) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(smem_u32(bar))
               : "memory");
}

// 16 consecutive TMEM columns of this thread's lane
__device__ __forceinline__ void tmem_ld16(uint32_t taddr, uint32_t* r) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15}, "
      "[%16];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]),
        "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
      : "r"(taddr)
      : "memory");
}
__device__ __forceinline__ void tmem_wait_ld() { asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory"); }

__device__ __forceinline__ long long c_offset32(unsigned lin, int nd, const FastDiv* f, const long long* st) {
  long long o = 0;
  for (int d = nd - 1; d >= 0; --d) {
    const unsigned q = fast_div(lin, f[d]);
    o += (long long)(lin - q * f[d].d) * st[d];
    lin = q;
  }
  return o;
}

struct OzArgs {
  const __nv_bfloat16* As;  // [MT][KT][S] tiles
  const __nv_bfloat16* Bs;  // [NT][KT][S] tiles
  const int* ea;            // [MT*128]
  const int* fb;            // [NT*BN]
  const unsigned* sq;       // [2] largest sum of squared digits of 16 k, A and B
  int S, MT, NT, KT;
  long long M, N;
  double alpha;
  // alpha = +-2^alpha_exp (its effect is on sign and exponent) unless alpha_fma
  // or alpha_zero; split-k partials carry no alpha
  int alpha_exp;
  bool alpha_neg, alpha_fma, alpha_zero;
  double* C;
  // C offsets: row m -> decoded with (nM, eM, cM), column n -> (nN, eN, cN)
  int nM, nN;
  int eM[4], eN[4];
  FastDiv fM[4], fN[4];  // divisors of eM, eN
  long long cM[4], cN[4];
  int rowfast;  // C's row index has the smaller stride (epilogue writes along rows)
  int* status;
  long long wait_cycles;  // budget of each bounded wait (clock cycles)
  // split over k tiles: split z covers [z*ktper, (z+1)*ktper) and writes its
  // scaled partial tile to part[z][MT*128][NT*BN] instead of C
  int splits, ktper;
  double* part;
  unsigned tiles;   // MT * NT * splits < 2^31
  FastDiv f_z, f_group, f_full, f_tail;  // divisors of the work list (oz_tile)
  int nbuf;         // stage buffers
};

__device__ __forceinline__ long long c_offset(long long lin, int nd, const int* ext, const long long* st) {
  long long o = 0;
  for (int d = nd - 1; d >= 0; --d) {
    long long q = lin / ext[d];
    o += (lin - q * ext[d]) * st[d];
    lin = q;
  }
  return o;
}

// barrier 2: the tile's warps and the two that write its tables.  Every one
// of them passes it once per tile, whatever happened before.
__device__ __forceinline__ void table_sync() { asm volatile("bar.sync 2, %0;" ::"n"(OZ_THREADS + 64) : "memory"); }
// barrier 1 over the 8 warps of the tile; whether every thread's pred was true
__device__ __forceinline__ bool tile_sync_and(bool pred) {
  uint32_t r;
  asm volatile(
      "{\n .reg .pred p, q;\n setp.ne.u32 p, %1, 0;\n bar.red.and.pred q, 1, %2, p;\n selp.u32 %0, 1, 0, q;\n}"
      : "=r"(r)
      : "r"((uint32_t)pred), "n"(OZ_THREADS)
      : "memory");
  return r != 0;
}

// Digit pairs (t, u), t + u <= S + 1, of one stage into the accumulators of
// their levels t + u (one thread), for the A slices t = LO .. HI.  For a fixed
// t the levels t + 1 .. S + 1 are adjacent in TMEM and the B slices
// 1 .. S + 1 - t adjacent in shared memory, so one MMA of N = BN (S + 1 - t)
// columns (pieces of at most 256) covers them and reads A_t once.  FRESH (the
// first stage of a window): t = 1, whose MMAs cover every level, comes first
// and overwrites.  Otherwise the slices run downwards, so that a stage ends
// with its widest MMAs.  dA / dB describe the first A / B tile of the stage's
// buffer (the descriptors differ only in the start-address field, bytes / 16).
template <int BN, int S, int LO, int HI, bool FRESH>
__device__ __forceinline__ void oz_issue(uint32_t tm, uint64_t dA, uint64_t dB) {
  constexpr int B_TILE_BYTES = BN * OZ_BK * 2;
  constexpr int UMAX = 256 / BN;
#pragma unroll
  for (int i = LO; i <= HI; ++i) {
    const int t = FRESH ? i : HI - (i - LO);
#pragma unroll
    for (int u0 = 1; u0 <= S + 1 - t; u0 += UMAX) {
      const int nu = (S + 1 - t) - u0 + 1 < UMAX ? (S + 1 - t) - u0 + 1 : UMAX;
      mma_bf16(tm + (uint32_t)((t + u0 - 2) * BN), dA + (uint64_t)(((t - 1) * OZ_TILE_BYTES) >> 4),
               dB + (uint64_t)(((u0 - 1) * B_TILE_BYTES) >> 4), oz_idesc(nu * BN), FRESH && t == 1 ? 0u : 1u);
    }
  }
}

// tile `lin` of the work list -> (k split z, row tile, column tile).  Grouped
// rasterisation: consecutive tiles walk the columns of a group of OZ_GROUP row
// tiles, so the CTAs running together share their digit tiles in L2.
__device__ __forceinline__ void oz_tile(const OzArgs& a, unsigned lin, int& z, int& mt, int& nt) {
  const unsigned zz = fast_div(lin, a.f_z), l = lin - zz * a.f_z.d;
  const unsigned grp = fast_div(l, a.f_group), within = l - grp * a.f_group.d;
  const bool tail = (int)(grp + 1) * OZ_GROUP > a.MT;
  const FastDiv& f = tail ? a.f_tail : a.f_full;  // row tiles of this group
  const unsigned c = fast_div(within, f);
  z = (int)zz;
  mt = (int)(grp * OZ_GROUP + within - c * f.d);
  nt = (int)c;
}

// (top 2^SH + bot) 2^k, negated if flip, as a double, assembled with integer
// instructions and rounded to nearest (bits beyond the 64th are dropped): the
// FP64 pipe has two lanes a clock.  No branches, so that several elements
// overlap (with branches a 128 x 32 tile's 16 elements a lane took 8400 clocks);
// odd is set where the result is subnormal or out of range (oz_value_odd).
template <int SH>
__device__ __forceinline__ double oz_value(long long top, long long bot, int k, bool flip, bool& odd) {
  // 128-bit two's complement hi:lo = (top << SH) + bot, then its magnitude
  unsigned long long lo = (unsigned long long)top << SH;
  long long hi = top >> (SH ? 64 - SH : 63);
  lo += (unsigned long long)bot;
  hi += (bot >> 63) + (lo < (unsigned long long)bot ? 1 : 0);
  const unsigned long long neg = (unsigned long long)(hi >> 63);
  lo ^= neg;
  hi ^= (long long)neg;
  lo -= neg;
  hi += neg && lo == 0 ? 1 : 0;
  // its leading 64 bits m in [2^63, 2^64), value m 2^e
  const bool wide = hi != 0;
  const unsigned long long H = wide ? (unsigned long long)hi : lo, L = wide ? lo : 0ULL;
  const int n = __clzll((long long)H) & 63;
  const unsigned long long m = (H << n) | ((L >> 1) >> (63 - n));
  const int ex = k + (wide ? 64 : 0) - n + 63 + 1023;
  const unsigned long long r = (m >> 11) + ((m >> 10) & 1ULL);  // in [2^52, 2^53]
  // the leading bit of r adds one to ex - 1
  const unsigned long long bits = ((unsigned long long)(unsigned)(ex - 1) << 52) + r;
  const unsigned long long sign = (neg ^ (flip ? ~0ULL : 0ULL)) & (1ULL << 63);
  odd = odd || (H != 0 && (ex <= 0 || ex >= 2046));
  return __longlong_as_double((long long)(H == 0 ? 0ULL : bits | sign));
}

// the same where it is subnormal or out of range: scaled in exact steps but the last
template <int SH>
__device__ __noinline__ double oz_value_odd(long long top, long long bot, int k, bool flip) {
  // |top 2^SH + bot| < 2^96: two halves, each exact in its own double
  const long long t = top >> 20, u = ((top & 0xFFFFF) << SH) + bot;
  double v = 0.0;
  for (int part = 0; part < 2; ++part) {
    double w = (double)(part ? u : t);
    for (int s = (part ? 0 : SH + 20) + k; s != 0;) {
      const int d = s > 1000 ? 1000 : s < -1000 ? -1000 : s;
      w *= __longlong_as_double((long long)(d + 1023) << 52);
      s -= d;
    }
    v += w;
  }
  return flip ? -v : v;
}

// Bounded wait that also gives up once another role of the CTA has.
__device__ __forceinline__ bool oz_wait(uint64_t* bar, uint32_t phase, long long budget, volatile int* stop) {
  if (mbar_test(bar, phase)) return true;
  const long long t0 = clock64();
  while (true) {
    if (clock64() - t0 > budget || *stop) {
      *stop = 1;
      return false;
    }
    if (mbar_try(bar, phase)) return true;
  }
}

constexpr int OZ_EPC = 8;                  // columns per warp staged at a time in the epilogue
constexpr int OZ_STAGE_LD = OZ_EPC + 1;    // padded against bank conflicts
constexpr int OZ_STAGE_BYTES = (OZ_THREADS / 32) * 32 * OZ_STAGE_LD * 8;
constexpr int OZ_STATIC_BYTES = 6144;     // more than the static tables and barriers take

// Stages per exact window: the level sums over the window must stay within
// 2^24.  With m the largest sum of squared digits (all slices) over any row's
// 16 k of an operand (oz_digits measures it), a level sum over one stage, and
// any part of it, is at most sqrt(mA mB) by Cauchy and Schwarz, once over k
// and once over the digit pairs of the level.  Digits of real data are spread
// over [-64, 64], about a third of the square of the largest, so windows are
// about 2.5 times as long as the OZ_WIN stages that hold for any digits.
__device__ __forceinline__ int oz_window(const OzArgs& a) {
  const float p = sqrtf((float)a.sq[0]) * sqrtf((float)a.sq[1]);
  const float w = 16777216.0f * 0.9999f / fmaxf(p, 1.0f);
  const int n = (int)fminf(w, 1048576.0f);
  return n > OZ_WIN ? n : OZ_WIN;
}

// stages whose level sums stay within 2^22, by the same bound
__device__ __forceinline__ int oz_quick(const OzArgs& a) {
  const float p = sqrtf((float)a.sq[0]) * sqrtf((float)a.sq[1]);
  return (int)fminf(4194304.0f * 0.9999f / fmaxf(p, 1.0f), 1048576.0f);
}

// Adds a window's level sums to top and bot.  QUICK (sums within 2^22): a sum
// becomes an integer by an addition of 1.5 2^23, whose bit pattern carries it
// in the low bits (the constant is taken off at the end); the conversion
// instruction, needed above that, runs at an eighth of the rate.
template <int BN, int S, int NCH, int CH, bool QUICK>
__device__ __forceinline__ void oz_sum(uint32_t taddr, long long (&top)[NCH][CH], long long (&bot)[NCH][CH]) {
  constexpr int CT = (S + 1) / 2;
  constexpr int MAGIC = 0x4B400000;  // 1.5 2^23
  long long bias_top = 0, bias_bot = 0;
#pragma unroll
  for (int c = 0; c < S; ++c) {
    if (c < CT) bias_top += (long long)MAGIC << (7 * (CT - 1 - c));
    else bias_bot += (long long)MAGIC << (7 * (S - 1 - c));
  }
  // chunks of CH columns, PER of them per wait (level by level)
  constexpr int PER = BN == 32 ? 2 : 1;
#pragma unroll
  for (int i0 = 0; i0 < S * NCH; i0 += PER) {
    uint32_t acc[PER][CH];
#pragma unroll
    for (int i = i0; i < i0 + PER && i < S * NCH; ++i)
      tmem_ld16(taddr + (uint32_t)(i / NCH * BN + i % NCH * CH), acc[i - i0]);
    tmem_wait_ld();
#pragma unroll
    for (int i = i0; i < i0 + PER && i < S * NCH; ++i) {
      const int c = i / NCH, j = i % NCH;
#pragma unroll
      for (int q = 0; q < CH; ++q) {
        const float f = __uint_as_float(acc[i - i0][q]);
        const int v = QUICK ? __float_as_int(f + __int_as_float(MAGIC)) : __float2int_rn(f);
        if (c < CT) top[j][q] += (long long)v * (1 << (7 * (CT - 1 - c)));
        else bot[j][q] += (long long)v * (1 << (7 * (S - 1 - c)));
      }
    }
  }
  if (QUICK) {
#pragma unroll
    for (int j = 0; j < NCH; ++j)
#pragma unroll
      for (int q = 0; q < CH; ++q) {
        top[j][q] -= bias_top;
        bot[j][q] -= bias_bot;
      }
  }
}

// Persistent CTAs: each walks the 128 x BN tiles of C (and k splits)
// blockIdx.x, blockIdx.x + gridDim.x, ...  Four roles run concurrently:
//  * warp 8 (lane 0) issues two bulk copies per 16-k stage (the S digit tiles
//    of A and of B are contiguous) into a ring of nbuf buffers;
//  * warp 9 (lane 0) issues the stage's MMAs as soon as its data are there;
//  * warps 10 and 11 write the tiles' tables of C offsets and exponents;
//  * warps 0-7 (warp w: TMEM lanes 32 (w % 4) .., column half w / 4) take the
//    level sums of every exact window (oz_window) out of TMEM into two 64-bit
//    integers per element, then write the tile while the next tile's MMAs run.
// Every level c = t + u has its own TMEM accumulator (S levels x BN columns);
// a window's level sums are exact integers below 2^24 in FP32, so the integer
// sums are exact: top = levels 2 .. CT + 1 in units of 2^(-7 (CT + 1)), bot =
// the rest in units of 2^(-7 (S + 1)).
// Bound: the tensor pipe.  One CTA per tile with the fold in float-float and
// 2 S copies per stage took 24.3 / 26.6 ms at 8192^3 (6 / 7 slices): 25 ms
// of it were the copies alone (14 copies of 2-4 KB a stage), 21 ms the MMAs
// alone (a shared issue thread).  Now 11.0 / 14.4 ms, 2090 / 2140 TFLOP/s
// executed (above the measured bf16 burst rate of a library GEMM); 4096^3 at 8
// slices 4.2 -> 2.4 ms.  Short contractions are bound by the write-back of C: the
// reductions in L2 (red_add).
template <int BN, int S>
__global__ void __launch_bounds__(OZ_CTA_THREADS, 1) k_ozaki_mma(const OzArgs a) {
  constexpr uint32_t TMEM_COLS = 512;
  constexpr int B_TILE_BYTES = BN * OZ_BK * 2;
  constexpr int STAGE_BYTES = S * (OZ_TILE_BYTES + B_TILE_BYTES);
  constexpr int HALF = BN / 2;               // columns per warp
  constexpr int CH = 16, NCH = HALF / CH;    // TMEM columns per load
  constexpr int CT = (S + 1) / 2, SH = 7 * (S - CT);  // levels in top; unit of top over that of bot
  // sets of accumulators: with two, the MMAs of the next window (or tile) run
  // while this one's sums are read
  constexpr int NACC = 2 * S * BN <= (int)TMEM_COLS ? 2 : 1;
  static_assert(S * BN <= (int)TMEM_COLS && HALF % CH == 0, "tile");
  extern __shared__ unsigned char oz_smem_raw[];
  unsigned char* smem = (unsigned char*)(((uintptr_t)oz_smem_raw + 1023) & ~(uintptr_t)1023);
  __shared__ uint64_t bar_full[OZ_MAXBUF], bar_free[OZ_MAXBUF], bar_acc[NACC], bar_read[NACC], bar_drain;
  __shared__ uint32_t tmem_base;
  __shared__ long long colC[2][BN], rowC[2][OZ_BM];  // C offsets and exponents of a tile and the next
  __shared__ int colE[2][BN], rowE[2][OZ_BM];
  __shared__ volatile int stop;  // a bounded wait ran out
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int nbuf = a.nbuf;

  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&tmem_base)),
                 "r"(TMEM_COLS)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  if (tid == 0) {
    for (int i = 0; i < nbuf; ++i) {
      mbar_init(&bar_full[i], 1);
      mbar_init(&bar_free[i], 1);
    }
    for (int i = 0; i < NACC; ++i) {
      mbar_init(&bar_acc[i], 1);
      mbar_init(&bar_read[i], OZ_THREADS / 32);
    }
    mbar_init(&bar_drain, 1);
    stop = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tm = tmem_base;

  if (warp >= OZ_THREADS / 32) {
    asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(OZ_REGS_ISSUE));
    if (warp == OZ_THREADS / 32 && lane == 0) {
      // ---- copies
      int b = 0;
      uint32_t lap = 0;  // times the ring has been walked
      bool ok = true;
      for (unsigned lin = blockIdx.x; ok && lin < a.tiles; lin += gridDim.x) {
        int z, mt, nt;
        oz_tile(a, lin, z, mt, nt);
        const int kt0 = z * a.ktper, kt1 = kt0 + a.ktper < a.KT ? kt0 + a.ktper : a.KT;
        const __nv_bfloat16* pa = a.As + ((size_t)mt * a.KT + kt0) * (S * OZ_TILE_ELEMS);
        const __nv_bfloat16* pb = a.Bs + ((size_t)nt * a.KT + kt0) * (S * BN * OZ_BK);
        for (int kt = kt0; kt < kt1; ++kt, pa += S * OZ_TILE_ELEMS, pb += S * BN * OZ_BK) {
          // the MMAs of the buffer's last use have completed
          if (lap > 0 && !oz_wait(&bar_free[b], (lap - 1) & 1, a.wait_cycles, &stop)) {
            ok = false;
            break;
          }
          unsigned char* base = smem + (size_t)b * STAGE_BYTES;
          mbar_expect_tx(&bar_full[b], (uint32_t)STAGE_BYTES);
          bulk_g2s(base, pa, S * OZ_TILE_BYTES, &bar_full[b]);
          bulk_g2s(base + S * OZ_TILE_BYTES, pb, S * B_TILE_BYTES, &bar_full[b]);
          if (++b == nbuf) {
            b = 0;
            ++lap;
          }
        }
      }
      // before the shared memory is released every copy issued has landed
      // (with the fixed default budget; immediate unless a wait ran out)
      for (int i = 0; i < nbuf; ++i) {
        const uint32_t n = lap + (i < b ? 1u : 0u);  // copies issued into buffer i
        if (n > 0) mbar_wait(&bar_full[i], (n - 1) & 1, OZ_WAIT_CYCLES);
      }
    }
    if (warp == OZ_THREADS / 32 + 1) {
      // ---- MMAs (the whole warp walks the stages, one elected lane issues)
      const uint64_t descA0 = sdesc(smem_u32(smem)), descB0 = sdesc(smem_u32(smem + S * OZ_TILE_BYTES));
      const int window = oz_window(a);
      int b = 0;                     // buffer of the next stage
      uint32_t ph = 0, win = 0;      // its phase; windows issued
      uint64_t dA = descA0, dB = descB0;
      bool there = false;            // its data are known to be there
      // one stage.  The tensor queue holds only a few MMAs, so the next
      // stage's barrier is tested between this stage's, and the stage ends
      // with wide ones: bookkeeping behind narrow ones left the pipe idle
      // (8192^3: 13.4 -> 11.8 ms at 6 slices, 15.9 -> 14.9 ms at 7)
      auto stage = [&](auto fresh) {
        constexpr bool FRESH = decltype(fresh)::value;
        constexpr int MID = S > 2 ? 2 : S;  // A slices 1 .. MID are the wide half
        if (!there && !__all_sync(0xffffffffu, oz_wait(&bar_full[b], ph, a.wait_cycles, &stop))) return false;
        uint64_t* const free = &bar_free[b];
        const uint64_t cA = dA, cB = dB;
        if (++b == nbuf) {
          b = 0;
          ph ^= 1;
        }
        dA = descA0 + (uint64_t)((uint32_t)(b * STAGE_BYTES) >> 4);
        dB = descB0 + (uint64_t)((uint32_t)(b * STAGE_BYTES) >> 4);
        const uint32_t acc = NACC == 2 ? tm + (win & 1) * (uint32_t)(S * BN) : tm;
        if (elect_one()) {
          if (FRESH) oz_issue<BN, S, 1, MID, FRESH>(acc, cA, cB);
          else oz_issue<BN, S, MID + 1, S, FRESH>(acc, cA, cB);
        }
        const bool next = mbar_test(&bar_full[b], ph);
        if (elect_one()) {
          if (FRESH) oz_issue<BN, S, MID + 1, S, FRESH>(acc, cA, cB);
          else oz_issue<BN, S, 1, MID, FRESH>(acc, cA, cB);
          mma_commit(free);  // the buffer is free once these complete
        }
        there = __all_sync(0xffffffffu, next);
        return true;
      };
      bool ok = true;
      for (unsigned lin = blockIdx.x; ok && lin < a.tiles; lin += gridDim.x) {
        const int z = (int)fast_div(lin, a.f_z);
        const int kt0 = z * a.ktper;
        int left = (kt0 + a.ktper < a.KT ? kt0 + a.ktper : a.KT) - kt0;
        while (ok && left > 0) {
          // the level sums of these accumulators' last window have been read
          const uint32_t set = win % NACC, use = win / NACC;
          if (use > 0 && !__all_sync(0xffffffffu, oz_wait(&bar_read[set], (use - 1) & 1, a.wait_cycles, &stop))) {
            ok = false;
            break;
          }
          tc_fence_after();
          const int n = left < window ? left : window;
          left -= n;
          ok = stage(std::true_type{});
          for (int i = 1; ok && i < n; ++i) ok = stage(std::false_type{});
          if (ok && elect_one()) mma_commit(&bar_acc[set]);  // completes once every MMA issued so far has
          ++win;
        }
      }
      // every MMA issued has completed before TMEM is released
      __syncwarp();
      if (elect_one()) mma_commit(&bar_drain);
      mbar_wait(&bar_drain, 0, OZ_WAIT_CYCLES);
    }
    if (warp >= OZ_THREADS / 32 + 2) {
      // ---- tables: C offsets and exponents of a tile's rows and columns, one
      // tile ahead of the summing warps (which spent 1200 clocks a tile on them)
      const int t0 = tid - (OZ_THREADS + 64);
      int tb = 0;
      for (unsigned lin = blockIdx.x; lin < a.tiles; lin += gridDim.x, tb ^= 1) {
        int z, mt, nt;
        oz_tile(a, lin, z, mt, nt);
        for (int i = t0; i < BN + OZ_BM; i += 64) {
          if (i < BN) {
            const long long n = (long long)nt * BN + i;
            colE[tb][i] = a.fb[n] - (int)OZ_EBIAS;
            colC[tb][i] = a.splits > 1 ? n : n < a.N ? c_offset32((unsigned)n, a.nN, a.fN, a.cN) : -1;
          } else {
            const long long m = (long long)mt * OZ_BM + i - BN;
            rowE[tb][i - BN] = a.ea[m] - (int)OZ_EBIAS;
            rowC[tb][i - BN] = a.splits > 1 ? ((long long)z * a.MT * OZ_BM + m) * ((long long)a.NT * BN)
                               : m < a.M   ? c_offset32((unsigned)m, a.nM, a.fM, a.cM)
                                           : -1;
          }
        }
        table_sync();
      }
    }
    __syncwarp();
  } else {
    // ---- level sums and C
    asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(OZ_REGS_SUM));
    const int quad = warp & 3, half = warp >> 2;
    const int row = quad * 32 + lane;
    const uint32_t taddr = tm + ((uint32_t)(quad * 32) << 16) + (uint32_t)(half * HALF);
    double* stg = reinterpret_cast<double*>(smem + (size_t)nbuf * STAGE_BYTES) + warp * 32 * OZ_STAGE_LD;
    uint32_t win = 0;
    const int window = oz_window(a), quick = oz_quick(a);
    int tb = 0;  // tables of this tile
    bool ok = true;
    for (unsigned lin = blockIdx.x; lin < a.tiles; lin += gridDim.x, tb ^= 1) {
      int z, mt, nt;
      oz_tile(a, lin, z, mt, nt);
      const int kt0 = z * a.ktper;
      int left = (kt0 + a.ktper < a.KT ? kt0 + a.ktper : a.KT) - kt0;
      // a warp whose rows or columns all lie outside C sums and writes nothing
      const bool used = (long long)nt * BN + half * HALF < a.N && (long long)mt * OZ_BM + quad * 32 < a.M;
      table_sync();  // this tile's tables are written, the last one's may be overwritten
      if (!ok) continue;
      double* const out = a.splits > 1 ? a.part : a.C;
      const long long keep = a.alpha_zero ? 0LL : ~0LL;  // alpha = 0 adds zeros
      // element u of a lane in a group of OZ_EPC columns: along the columns of
      // rows 4 u + lane / 8, or along the rows of column u
      auto place = [&](int c0, int u) -> long long {
        const long long fix = a.rowfast ? rowC[tb][quad * 32 + lane] : colC[tb][c0 + lane % OZ_EPC];
        const long long var = a.rowfast ? colC[tb][c0 + u] : rowC[tb][quad * 32 + u * (32 / OZ_EPC) + lane / OZ_EPC];
        return fix >= 0 && var >= 0 ? fix + var : -1;
      };
      const double* const sp =
          stg + (a.rowfast ? lane * OZ_STAGE_LD : lane / OZ_EPC * OZ_STAGE_LD + lane % OZ_EPC);
      const int sstep = a.rowfast ? 1 : 32 / OZ_EPC * OZ_STAGE_LD;
      constexpr int NG = HALF / OZ_EPC;
      long long top[NCH][CH], bot[NCH][CH];
#pragma unroll
      for (int j = 0; j < NCH; ++j)
#pragma unroll
        for (int q = 0; q < CH; ++q) top[j][q] = bot[j][q] = 0;
      for (; left > 0; left -= window, ++win) {
        // one thread polls, the others sleep at the barrier
        const uint32_t set = win % NACC;
        if (tid == 0) ok = oz_wait(&bar_acc[set], (win / NACC) & 1, a.wait_cycles, &stop);
        ok = tile_sync_and(ok);
        if (!ok) break;
        tc_fence_after();
        const int n = left < window ? left : window;
        if (used) {
          const uint32_t t = taddr + set * (uint32_t)(S * BN);
          if (n <= quick) oz_sum<BN, S, NCH, CH, true>(t, top, bot);
          else oz_sum<BN, S, NCH, CH, false>(t, top, bot);
        }
        // the accumulators are read; the next window may overwrite them
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(&bar_read[set]);
      }
      if (!ok) continue;
      // alpha 2^(ea[m] + fb[n] + 2 - 7 (S + 1)) (top 2^SH + bot), OZ_EPC columns at
      // a time through this warp's staging rows, so that consecutive lanes
      // touch consecutive elements of C (or of the split-k partial)
      if (used) {
        const int em = rowE[tb][row] + 2 - 7 * (S + 1) + a.alpha_exp;
#pragma unroll
        for (int g = 0; g < NG; ++g) {
          const int c0 = half * HALF + g * OZ_EPC;
          bool odd = false;
#pragma unroll
          for (int q = 0; q < OZ_EPC; ++q)
            stg[lane * OZ_STAGE_LD + q] =
                oz_value<SH>(top[g * OZ_EPC / CH][g * OZ_EPC % CH + q], bot[g * OZ_EPC / CH][g * OZ_EPC % CH + q],
                             em + colE[tb][c0 + q], a.alpha_neg, odd);
          if (__any_sync(0xffffffffu, odd)) {
#pragma unroll
            for (int q = 0; q < OZ_EPC; ++q)
              stg[lane * OZ_STAGE_LD + q] = oz_value_odd<SH>(top[g * OZ_EPC / CH][g * OZ_EPC % CH + q],
                                                             bot[g * OZ_EPC / CH][g * OZ_EPC % CH + q],
                                                             em + colE[tb][c0 + q], a.alpha_neg);
          }
          __syncwarp();
          if (a.alpha_fma) {
            // alpha t + C rounded once, as where alpha is a power of two, by
            // loads a few elements ahead (61504 x 784 x 64, 7 slices: 687 us, one
            // by one 1003; a reduction in L2, 485, would round alpha t first)
            constexpr int AHEAD = 4;
#pragma unroll
            for (int u0 = 0; u0 < OZ_EPC; u0 += AHEAD) {
              long long o[AHEAD];
              double c[AHEAD];
#pragma unroll
              for (int u = 0; u < AHEAD; ++u) {
                o[u] = place(c0, u0 + u);
                c[u] = o[u] >= 0 ? a.C[o[u]] : 0.0;
              }
#pragma unroll
              for (int u = 0; u < AHEAD; ++u)
                if (o[u] >= 0) a.C[o[u]] = fma(a.alpha, sp[(u0 + u) * sstep], c[u]);
            }
          } else {
#pragma unroll
            for (int u = 0; u < OZ_EPC; ++u) {
              const long long o = place(c0, u);
              const double t = sp[u * sstep];
              if (o >= 0) {
                if (a.splits > 1) out[o] = t;
                else red_add(out + o, __longlong_as_double(__double_as_longlong(t) & keep));
              }
            }
          }
          __syncwarp();
        }
      }
    }
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 0) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tm), "r"(TMEM_COLS)
                              : "memory");
  if (stop && tid == 0) atomicExch(a.status, 1);
}

// C[m, n] += alpha * sum_z part[z][m][n] (z in order)
template <int BN>
__global__ void k_ozaki_reduce(const OzArgs a) {
  const long long Mp = (long long)a.MT * OZ_BM, ldp = (long long)a.NT * BN;
  const long long total = a.M * a.N;
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < total;
       i += (long long)gridDim.x * blockDim.x) {
    const long long m = i / a.N, n = i - m * a.N;
    double s = 0.0;
    for (int z = 0; z < a.splits; ++z) s += a.part[((long long)z * Mp + m) * ldp + n];
    a.C[c_offset(m, a.nM, a.eM, a.cM) + c_offset(n, a.nN, a.eN, a.cN)] += a.alpha * s;
  }
}

// The same sum with one warp per output element, for many splits over few
// outputs (one thread would chain hundreds of dependent loads): lane l adds
// z = l, l + 32, ... in order, then a fixed shuffle tree combines the lanes.
template <int BN>
__global__ void k_ozaki_reduce_warp(const OzArgs a) {
  const long long Mp = (long long)a.MT * OZ_BM, ldp = (long long)a.NT * BN;
  const long long total = a.M * a.N;
  const int lane = threadIdx.x & 31;
  const long long wid = (blockIdx.x * (long long)blockDim.x + threadIdx.x) >> 5;
  const long long nw = ((long long)gridDim.x * blockDim.x) >> 5;
  for (long long i = wid; i < total; i += nw) {
    const long long m = i / a.N, n = i - m * a.N;
    double s = 0.0;
    for (int z = lane; z < a.splits; z += 32) s += a.part[((long long)z * Mp + m) * ldp + n];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) s += __shfl_down_sync(0xffffffffu, s, o);
    if (lane == 0) a.C[c_offset(m, a.nM, a.eM, a.cM) + c_offset(n, a.nN, a.eN, a.cN)] += a.alpha * s;
  }
}

// ---------------------------------------------------------------------------
// operand preparation
// ---------------------------------------------------------------------------
struct OzPack {
  const double* src;
  int nR, nK;
  int eR[4], eK[4];
  long long sR[4], sK[4];
  long long R, K;      // logical sizes (both < 2^31)
  int T, KT;           // tiles along rows (TR each) and k (64 each)
  int TR;              // rows per tile: 128 (A) or BN (B)
  int S;
  int vec;             // 1: every full 8-group is 64 contiguous, 16-byte aligned bytes; 2: 32-byte aligned
  FastDiv fR[4], fK[4];  // divisors of eR, eK
};

// whether pack_load8 may read a full k group with 32-byte (2) or 16-byte (1)
// loads: unit innermost k stride, groups that never cross a carry of the k
// multi-index (innermost extent a multiple of 8), every other stride a
// multiple of 4 (2) and the base aligned, so every group starts on a boundary
inline int pack_vec_ok(const OzPack& p) {
  if (p.nK < 1 || p.sK[p.nK - 1] != 1 || p.eK[p.nK - 1] % 8 != 0) return 0;
  for (int v = 2; v > 0; --v) {
    bool ok = reinterpret_cast<uintptr_t>(p.src) % (16 * v) == 0;
    for (int d = 0; d < p.nK - 1; ++d) ok = ok && p.sK[d] % (2 * v) == 0;
    for (int d = 0; d < p.nR; ++d) ok = ok && p.sR[d] % (2 * v) == 0;
    if (ok) return v;
  }
  return 0;
}

// Operand preparation runs in two passes over the padded operand viewed as
// rows x (8-element k groups).  Work item i is one (row r, group q); when the
// source's innermost k index is contiguous the groups of a row are adjacent
// items (reads coalesce along k), otherwise the rows are (reads coalesce along
// the row index).
//   pass 1: eu[r] = 2048 + max over k of the binary exponent ex with
//           |x| < 2^ex (frexp), 0 for an all-zero row (eu zeroed beforehand);
//   pass 2: the S balanced 7-bit digits of x 2^(-e) go to the swizzled tiles,
//           eight bf16 (16 bytes) per store.
constexpr int PACK_T = 256;

// Everything below works on the bit patterns with integer instructions: the
// FP64 pipe of this SM is narrow, and even a comparison with 0.0 runs there.
__device__ __forceinline__ unsigned exp_code(long long bits) {
  if ((bits << 1) == 0) return 0u;  // +-0
  const int be = (int)((bits >> 52) & 0x7FF);
  return (unsigned)((be ? be - 1022 : -1022) + (int)OZ_EBIAS);
}

// work item i -> (row r, group q); i, Rpad, Q < 2^32
__device__ __forceinline__ void pack_item(unsigned i, const FastDiv& fQ, const FastDiv& fR, bool kfast, unsigned& r,
                                          unsigned& q) {
  if (kfast) {
    r = fast_div(i, fQ);
    q = i - r * fQ.d;
  } else {
    q = fast_div(i, fR);
    r = i - q * fR.d;
  }
}

// bit patterns of the (up to) 8 source values of group q of row r; zero
// outside R x K
__device__ __forceinline__ void pack_load8(const OzPack& p, unsigned r, unsigned q, long long x[8]) {
  const unsigned k0 = q * 8u;
#pragma unroll
  for (int j = 0; j < 8; ++j) x[j] = 0;
  if (r >= (unsigned long long)p.R || k0 >= (unsigned long long)p.K) return;
  const long long* src = reinterpret_cast<const long long*>(p.src);
  long long roff = 0;
  {
    unsigned lin = r;
    for (int d = p.nR - 1; d >= 0; --d) {
      const unsigned qd = fast_div(lin, p.fR[d]);
      roff += (long long)(lin - qd * p.fR[d].d) * p.sR[d];
      lin = qd;
    }
  }
  // multi-index of k0, then step through the next 7 with carries
  int idx[4];
  long long off = 0;
  {
    unsigned lin = k0;
    for (int d = p.nK - 1; d >= 0; --d) {
      const unsigned qd = fast_div(lin, p.fK[d]);
      idx[d] = (int)(lin - qd * p.fK[d].d);
      off += (long long)idx[d] * p.sK[d];
      lin = qd;
    }
  }
  if (p.vec == 2 && k0 + 8 <= (unsigned long long)p.K) {
    // one full sector per lane and load: with 16-byte loads at a 64-byte
    // stride the row-maximum pass read 3.7 TB/s
    const long long* v = src + roff + off;
#pragma unroll
    for (int h = 0; h < 2; ++h)
      asm volatile("ld.global.v4.b64 {%0, %1, %2, %3}, [%4];"
                   : "=l"(x[4 * h]), "=l"(x[4 * h + 1]), "=l"(x[4 * h + 2]), "=l"(x[4 * h + 3])
                   : "l"(v + 4 * h));
    return;
  }
  if (p.vec && k0 + 8 <= (unsigned long long)p.K) {
    const longlong2* v = reinterpret_cast<const longlong2*>(src + roff + off);
#pragma unroll
    for (int h = 0; h < 4; ++h) {
      const longlong2 t = v[h];
      x[2 * h] = t.x;
      x[2 * h + 1] = t.y;
    }
    return;
  }
  const int last = p.nK - 1;
#pragma unroll
  for (int j = 0; j < 8; ++j) {
    if (k0 + j >= (unsigned long long)p.K) break;
    x[j] = src[roff + off];
    if (j == 7) break;
    int d = last;
    ++idx[d];
    off += p.sK[d];
    while (idx[d] == p.eK[d] && d > 0) {
      off -= (long long)p.eK[d] * p.sK[d];
      idx[d] = 0;
      --d;
      ++idx[d];
      off += p.sK[d];
    }
  }
}

// Both operands of a product in one launch: blockIdx.y selects A (0) or B (1).
struct PackPass {
  OzPack p[2];
  unsigned* eu[2];
  __nv_bfloat16* dst[2];
  int kfast[2];
  FastDiv fQ[2], fR[2];
  unsigned W[2];
  unsigned* sq;  // [2] (pass 2 and the one-pass form)
  int lpr[2];    // one-pass form: lanes per row, 0: one thread per row
};

// Each warp walks one contiguous range of steps of 32 work items, and each lane
// keeps the maximum of its current row in a register.  When lanes move to
// another row, those that leave the same row combine their maxima and one of
// them issues the atomic max: with k along the lanes a warp crosses a row's end
// every few steps, and an atomic per lane (6 million for 61504 x 784) held the
// pass at 3.8 TB/s.
__global__ void __launch_bounds__(PACK_T) k_ozaki_rowexp(const PackPass pp) {
  const int o = blockIdx.y;
  const OzPack& p = pp.p[o];
  unsigned* eu = pp.eu[o];
  const int kfast = pp.kfast[o];
  const FastDiv fQ = pp.fQ[o], fR = pp.fR[o];
  const unsigned W = pp.W[o];
  const unsigned lane = threadIdx.x & 31;
  const unsigned long long warps = (unsigned long long)gridDim.x * (PACK_T / 32);
  const unsigned long long steps = (W + 31ULL) / 32;  // of 32 items; W is a multiple of 32 when rows are along the lanes
  const unsigned long long per = (steps + warps - 1) / warps;
  const unsigned long long lo = (blockIdx.x * (unsigned long long)(PACK_T / 32) + (threadIdx.x >> 5)) * per;
  const unsigned long long hi = lo + per < steps ? lo + per : steps;
  unsigned held = ~0u, hv = 0;  // row (none: ~0) and the maximum so far
  // lanes with `go` send (held, hv); a warp-wide step
  auto flush = [&](bool go) {
    go = go && hv;
    const unsigned mask = __ballot_sync(0xffffffffu, go);
    if (!mask) return;
    const int lead = __ffs(mask) - 1;
    const unsigned r0 = __shfl_sync(0xffffffffu, held, lead);
    if (__all_sync(0xffffffffu, !go || held == r0)) {
      const unsigned m = __reduce_max_sync(0xffffffffu, go ? hv : 0u);
      if ((int)lane == lead) atomicMax(eu + r0, m);
    } else if (go) {
      atomicMax(eu + held, hv);
    }
  };
  for (unsigned long long t = lo; t < hi; ++t) {
    unsigned rr = ~0u, v = 0;
    const unsigned long long i = t * 32 + lane;
    if (i < W) {
      // along k: item i is (row, group); along the rows: step t is the 32 rows
      // of a block at one group, the groups of a block in a row
      unsigned q;
      if (kfast) {
        pack_item((unsigned)i, fQ, fR, true, rr, q);
      } else {
        const unsigned rb = fast_div((unsigned)t, fQ);
        q = (unsigned)t - rb * fQ.d;
        rr = rb * 32 + lane;
      }
      if (rr < (unsigned long long)p.R) {
        long long x[8];
        pack_load8(p, rr, q, x);
#pragma unroll
        for (int j = 0; j < 8; ++j) v = max(v, exp_code(x[j]));
      }
    }
    const bool moved = rr != held;
    if (__any_sync(0xffffffffu, moved)) {
      flush(moved);
      if (moved) {
        held = rr;
        hv = 0;
      }
    }
    hv = max(hv, v);
  }
  flush(true);
}

// S balanced base-128 digits of each element: V = round(x 2^(7S - 1 - e)),
// |V| <= 2^(7S - 1) (|x| < 2^e, e the row / column exponent), written as
// V = sum_t d_t 128^(S - t) with |d_t| <= 64, so x = 2^(e + 1) sum_t d_t 2^(-7t);
// the digits are extracted from the lowest up with balanced remainders and
// stored as bf16 (exact: |d| <= 64).  One call: group q of row r, S 16-byte
// stores (one per slice tile); returns the sum of the squared digits.
template <int S>
__device__ __forceinline__ int digits_item(const OzPack& p, const long long (&x)[8], int e, __nv_bfloat16* dst,
                                            unsigned r, unsigned q) {
  const long long tile_elems = (long long)p.TR * OZ_BK;
  constexpr int F = 7 * S - 1;
  int dg[S][8];
#pragma unroll
  for (int j = 0; j < 8; ++j) {
    long long V = 0;
    const long long bits = x[j];
    if ((bits << 1) != 0) {
      const int be = (int)((bits >> 52) & 0x7FF);
      unsigned long long m = (unsigned long long)(bits & ((1LL << 52) - 1));
      int E;
      if (be) {
        m |= 1ULL << 52;
        E = be - 1075;
      } else {
        E = -1074;
      }
      const int sh_ = E + F - e;  // |x| 2^(F - e) = m 2^sh < 2^F
      unsigned long long v;
      if (sh_ >= 0) v = sh_ < 12 ? (m << sh_) : 0;
      else if (-sh_ >= 64) v = 0;
      else v = (m >> (-sh_)) + ((m >> (-sh_ - 1)) & 1ULL);  // to nearest, ties away from zero
      V = bits < 0 ? -(long long)v : (long long)v;
    }
    // V = hi 2^28 + lo, 0 <= lo < 2^28: a digit depends only on the running
    // value mod 128, so the (at most) four lowest digits come from lo in
    // 32-bit arithmetic (lo - d >= 0 stays exact), then the carry joins the
    // upper part for the rest
    constexpr int NL = S - 1 < 4 ? S - 1 : 4;
    int lo = (int)(V & 0xFFFFFFFLL), hi = (int)(V >> 28);
#pragma unroll
    for (int k = 0; k < NL; ++k) {
      const int d = ((lo + 64) & 127) - 64;
      dg[S - 1 - k][j] = d;
      lo = (lo - d) >> 7;
    }
    hi = lo + hi * (1 << (28 - 7 * NL));
#pragma unroll
    for (int k = NL; k < S - 1; ++k) {
      const int d = ((hi + 64) & 127) - 64;
      dg[S - 1 - k][j] = d;
      hi = (hi - d) >> 7;
    }
    dg[0][j] = hi;  // |hi| <= 64 here
  }
  int sq = 0;
  const unsigned tr = r / p.TR, rr = r - tr * p.TR;  // TR is 32, 64 or 128
  const int tk = (int)(q >> 1), chunk = (int)(q & 1);   // two 8-element chunks per 16-k row
  const long long within = (long long)rr * OZ_BK + ((chunk ^ ((rr >> 2) & 1)) << 3);
#pragma unroll
  for (int t = 1; t <= S; ++t) {
    uint32_t w[4];
#pragma unroll
    for (int h = 0; h < 4; ++h) {
      // |d| <= 64: exact in float and in bf16, so the conversion is exact
      sq += dg[t - 1][2 * h] * dg[t - 1][2 * h] + dg[t - 1][2 * h + 1] * dg[t - 1][2 * h + 1];
      const __nv_bfloat162 b2 = __floats2bfloat162_rn((float)dg[t - 1][2 * h], (float)dg[t - 1][2 * h + 1]);
      w[h] = *reinterpret_cast<const uint32_t*>(&b2);
    }
    const long long tile = ((long long)tr * p.KT + tk) * S + (t - 1);  // the S tiles of a stage are adjacent
    *reinterpret_cast<uint4*>(dst + tile * tile_elems + within) = make_uint4(w[0], w[1], w[2], w[3]);
  }
  return sq;
}

// A 16-k row of a digit tile is 32 bytes, one DRAM sector, filled by its two
// 8-element groups, and the two halves are written by neighbouring lanes:
// along k the groups of a row are consecutive items anyway; along rows item
// i takes row (i / 2) mod rows and group 2 ((i / 2) / rows) + i mod 2.  (With
// rows alone along the lanes, the second half of every sector followed a
// whole pass over the rows later, after the sector had left L2: each
// half-sector write then cost a read-modify-write in DRAM, and the digit pass
// moved 2-4x its bytes.)
template <int S>
__global__ void __launch_bounds__(PACK_T) k_ozaki_digits(const PackPass pp) {
  const int o = blockIdx.y;
  const OzPack& p = pp.p[o];
  const unsigned* eu = pp.eu[o];
  __nv_bfloat16* dst = pp.dst[o];
  const int kfast = pp.kfast[o];
  const FastDiv fQ = pp.fQ[o], fR = pp.fR[o];
  const unsigned W = pp.W[o];
  const unsigned stride = gridDim.x * PACK_T;
  int most = 0;  // largest sum of squared digits of one row's 16 k (the window rule)
  for (unsigned long long base = blockIdx.x * PACK_T; base < W; base += stride) {
    const unsigned i = (unsigned)base + threadIdx.x;
    int sq = 0;
    if (base + threadIdx.x < W) {
      unsigned r, q;
      if (kfast) {
        pack_item(i, fQ, fR, true, r, q);
      } else {
        const unsigned j = i >> 1, tk = fast_div(j, fR);
        r = j - tk * fR.d;
        q = 2u * tk + (i & 1u);
      }
      long long x[8];
      pack_load8(p, r, q, x);
      sq = digits_item<S>(p, x, r < (unsigned long long)p.R ? (int)eu[r] - (int)OZ_EBIAS : 0, dst, r, q);
    }
    // items 2 j and 2 j + 1 are the halves of one row's 16 k
    sq += __shfl_xor_sync(0xffffffffu, sq, 1);
    most = sq > most ? sq : most;
  }
  most = __reduce_max_sync(0xffffffffu, most);
  __shared__ int part[PACK_T / 32];
  if ((threadIdx.x & 31) == 0) part[threadIdx.x >> 5] = most;
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int w = 1; w < PACK_T / 32; ++w) most = part[w] > most ? part[w] : most;
    if (most > 0) atomicMax(pp.sq + o, (unsigned)most);
  }
}

// Both passes in one for k up to PACK_SHORT: the exponent of a row is known
// before its digits are cut.  Lanes along k (a row's groups in `lpr` adjacent
// lanes, each group loaded once), or where the rows are the contiguous
// direction and many, one thread per row, which reads it twice.  The window
// rule gets the bound that holds for any digits (one window, and the quick
// sums for k up to 112 at 8 slices).  Every padded row is written, so nothing
// is cleared beforehand: one launch in place of three.
constexpr int PACK_SHORT = 256, PACK_ROWS = 4096;
template <int S>
__global__ void __launch_bounds__(PACK_T) k_ozaki_pack_short(const PackPass pp) {
  const int o = blockIdx.y;
  const OzPack& p = pp.p[o];
  unsigned* eu = pp.eu[o];
  __nv_bfloat16* dst = pp.dst[o];
  const unsigned rows = (unsigned)p.T * (unsigned)p.TR, groups = (unsigned)p.KT * (OZ_BK / 8);
  if (blockIdx.x == 0 && threadIdx.x == 0) pp.sq[o] = (unsigned)(OZ_BK * S * 64 * 64);
  const unsigned long long t0 = blockIdx.x * (unsigned long long)PACK_T + threadIdx.x;
  const unsigned long long stride = (unsigned long long)gridDim.x * PACK_T;
  if (pp.lpr[o]) {
    const unsigned lpr = (unsigned)pp.lpr[o], sh = 31 - __clz(lpr), q = (unsigned)t0 & (lpr - 1);
    // rows is a multiple of 32, so whole warps leave the loop together
    for (unsigned long long t = t0; t < (unsigned long long)rows << sh; t += stride) {
      const unsigned r = (unsigned)(t >> sh);
      long long x[8];
      pack_load8(p, r, q, x);  // zero beyond the operand
      unsigned c = 0;
#pragma unroll
      for (int j = 0; j < 8; ++j) c = max(c, exp_code(x[j]));
      for (unsigned d = lpr >> 1; d > 0; d >>= 1) c = max(c, __shfl_xor_sync(0xffffffffu, c, d));
      if (q < groups) digits_item<S>(p, x, (int)c - (int)OZ_EBIAS, dst, r, q);
      if (q == 0) eu[r] = c;
    }
  } else {
    for (unsigned long long r = t0; r < rows; r += stride) {
      unsigned c = 0;
      for (unsigned q = 0; q < groups; ++q) {
        long long x[8];
        pack_load8(p, (unsigned)r, q, x);
#pragma unroll
        for (int j = 0; j < 8; ++j) c = max(c, exp_code(x[j]));
      }
      for (unsigned q = 0; q < groups; ++q) {
        long long x[8];
        pack_load8(p, (unsigned)r, q, x);
        digits_item<S>(p, x, (int)c - (int)OZ_EBIAS, dst, (unsigned)r, q);
      }
      eu[r] = c;
    }
  }
}

inline int oz_pack_grid(long long n) {
  long long b = (n + PACK_T - 1) / PACK_T;
  if (b < 1) b = 1;
  if (b > 152 * 32) b = 152 * 32;
  return (int)b;
}

// rows or k along the coalesced direction of the source (see the pack kernels)
inline int pack_kfast(const OzPack& p) {
  if (p.nK > 0 && p.sK[p.nK - 1] == 1) return 1;
  if (p.nR > 0 && p.sR[p.nR - 1] == 1) return 0;
  return 1;
}

inline int oz_grid(long long n) {
  long long b = (n + 255) / 256;
  if (b < 1) b = 1;
  if (b > 152 * 16) b = 152 * 16;
  return (int)b;
}

// stage buffers that fit beside the staging rows and the static tables
int oz_buffers(int S, int BN) {
  const int stage = S * (OZ_TILE_BYTES + BN * OZ_BK * 2);
  const int n = (227 * 1024 - OZ_STATIC_BYTES - 1024 - OZ_STAGE_BYTES) / stage;
  return n < OZ_MAXBUF ? n : OZ_MAXBUF;
}

size_t oz_smem_bytes(int S, int BN, int nbuf) {
  return (size_t)nbuf * S * (OZ_TILE_BYTES + BN * OZ_BK * 2) + OZ_STAGE_BYTES + 1024;
}

// the largest dynamic shared memory any launch of a kernel asks for, set once
// per device (kept out of the launch path, which may be captured)
template <int BN, int S>
void oz_smem_attribute() {
  static std::mutex mu;
  static bool done[64] = {};
  int dev = 0;
  check_cuda(cudaGetDevice(&dev), "cudaGetDevice");
  std::lock_guard<std::mutex> lock(mu);
  if (dev < 0 || dev >= 64 || done[dev]) return;
  check_cuda(cudaFuncSetAttribute(k_ozaki_mma<BN, S>, cudaFuncAttributeMaxDynamicSharedMemorySize, 227 * 1024 - OZ_STATIC_BYTES),
             "cudaFuncSetAttribute (ozaki)");
  // the kernel's register split draws on exactly this launch total
  cudaFuncAttributes fa{};
  check_cuda(cudaFuncGetAttributes(&fa, k_ozaki_mma<BN, S>), "cudaFuncGetAttributes (ozaki)");
  if (fa.numRegs != OZ_REGS) throw std::runtime_error("split-precision kernel: unexpected register count");
  done[dev] = true;
}

template <int BN, int S>
void oz_launch_bn_s(const OzArgs& a, cudaStream_t st) {
  // at least 120 KiB so that one CTA (one TMEM allocation) occupies an SM
  size_t smem = oz_smem_bytes(S, BN, a.nbuf);
  if (smem < 120 * 1024) smem = 120 * 1024;
  oz_smem_attribute<BN, S>();
  const unsigned grid = (unsigned)(a.tiles < 152 ? a.tiles : 152);
  k_ozaki_mma<BN, S><<<grid, OZ_CTA_THREADS, smem, st>>>(a);
}

template <int BN>
void oz_launch_bn(OzArgs a, int MT, int NT, cudaStream_t st) {
  const long long tiles = (long long)MT * NT * a.splits;
  if (tiles >= (1LL << 31)) throw std::runtime_error("split-precision contraction: too many tiles");
  a.tiles = (unsigned)tiles;
  a.f_z = make_fastdiv((unsigned)(MT * NT));
  a.f_group = make_fastdiv((unsigned)(OZ_GROUP * NT));
  a.f_full = make_fastdiv((unsigned)(MT < OZ_GROUP ? MT : OZ_GROUP));
  a.f_tail = make_fastdiv((unsigned)(MT % OZ_GROUP ? MT % OZ_GROUP : OZ_GROUP));
  a.nbuf = oz_buffers(a.S, BN);
  switch (a.S) {
    case 1: oz_launch_bn_s<BN, 1>(a, st); break;
    case 2: oz_launch_bn_s<BN, 2>(a, st); break;
    case 3: oz_launch_bn_s<BN, 3>(a, st); break;
    case 4: oz_launch_bn_s<BN, 4>(a, st); break;
    case 5: oz_launch_bn_s<BN, 5>(a, st); break;
    case 6: oz_launch_bn_s<BN, 6>(a, st); break;
    case 7: oz_launch_bn_s<BN, 7>(a, st); break;
    default: oz_launch_bn_s<BN, 8>(a, st); break;
  }
  if (a.splits > 1) {
    // few outputs, many splits: a warp per output keeps loads in flight
    if (a.splits >= 32 && a.M * a.N < 152LL * 256)
      k_ozaki_reduce_warp<BN><<<oz_grid(a.M * a.N * 32), 256, 0, st>>>(a);
    else
      k_ozaki_reduce<BN><<<oz_grid(a.M * a.N), 256, 0, st>>>(a);
  }
}

void oz_launch_mma(const OzArgs& a, int MT, int NT, int BN, cudaStream_t st) {
  if (BN == 32) oz_launch_bn<32>(a, MT, NT, st);
  else oz_launch_bn<64>(a, MT, NT, st);
}
}  // namespace

int ozaki_status(cudaStream_t st, const int* flag) {
  int v = 0;
  check_cuda(cudaMemcpyAsync(&v, flag, sizeof(int), cudaMemcpyDeviceToHost, st), "status");
  check_cuda(cudaStreamSynchronize(st), "sync");
  return v;
}

bool ozaki_supported(const GemmArgs& g) {
  // packing indexes (padded rows) x (8-element k groups) with 32 bits
  const long long big = g.M > g.N ? g.M : g.N;
  const long long rows = (big + OZ_BM - 1) / OZ_BM * OZ_BM, groups = (g.K + OZ_BK - 1) / OZ_BK * (OZ_BK / 8);
  return g.M < (1LL << 31) && g.N < (1LL << 31) && g.K < (1LL << 31) && rows * groups < (1LL << 32);
}

namespace {
// tile width (0: the rule below) and k-split mode (0: rule, 1: none, 2: twice the rule)
struct OzChoice {
  int bn = 0;
  int split_mode = 0;
};

void ozaki_run(Workspace& ws, const GemmArgs& g0, int S, int kind, const OzChoice& ch) {
  if (g0.M <= 0 || g0.N <= 0 || g0.K <= 0) return;
  if (g0.nbatch != 1) throw std::runtime_error("split-precision contraction needs nbatch == 1");
  if (S < 1 || S > kOzakiMaxSlices) throw std::runtime_error("split-precision slices must be 1..8");
  if (!ozaki_supported(g0)) throw std::runtime_error("split-precision contraction too large for 32-bit packing");
  // orient so that the longer output side runs along the 128-row A tiles:
  // C^T = B^T A^T just exchanges the roles of the operands
  const bool swap = g0.N > g0.M;
  OzPack pa{}, pb{};
  OzArgs a{};
  auto fill = [&](OzPack& p, const double* src, int nR, const int* eR, const long long* sR) {
    p.src = src;
    p.nR = nR;
    p.nK = g0.nK;
    for (int d = 0; d < 4; ++d) {
      p.eR[d] = eR[d];
      p.sR[d] = sR[d];
      p.eK[d] = g0.eK[d];
    }
    p.K = g0.K;
    p.S = S;
    for (int d = 0; d < 4; ++d) {
      p.fR[d] = make_fastdiv(d < nR ? (unsigned)eR[d] : 1u);
      p.fK[d] = make_fastdiv(d < g0.nK ? (unsigned)g0.eK[d] : 1u);
    }
  };
  long long M, N;
  if (!swap) {
    fill(pa, g0.A, g0.nM, g0.eM, g0.aM);
    for (int d = 0; d < 4; ++d) pa.sK[d] = g0.aK[d];
    fill(pb, g0.B, g0.nN, g0.eN, g0.bN);
    for (int d = 0; d < 4; ++d) pb.sK[d] = g0.bK[d];
    M = g0.M;
    N = g0.N;
    a.nM = g0.nM;
    a.nN = g0.nN;
    for (int d = 0; d < 4; ++d) {
      a.eM[d] = g0.eM[d];
      a.cM[d] = g0.cM[d];
      a.eN[d] = g0.eN[d];
      a.cN[d] = g0.cN[d];
    }
  } else {
    fill(pa, g0.B, g0.nN, g0.eN, g0.bN);
    for (int d = 0; d < 4; ++d) pa.sK[d] = g0.bK[d];
    fill(pb, g0.A, g0.nM, g0.eM, g0.aM);
    for (int d = 0; d < 4; ++d) pb.sK[d] = g0.aK[d];
    M = g0.N;
    N = g0.M;
    a.nM = g0.nN;
    a.nN = g0.nM;
    for (int d = 0; d < 4; ++d) {
      a.eM[d] = g0.eN[d];
      a.cM[d] = g0.cN[d];
      a.eN[d] = g0.eM[d];
      a.cN[d] = g0.cM[d];
    }
  }
  pa.vec = pack_vec_ok(pa);
  pb.vec = pack_vec_ok(pb);
  // 64 columns per tile, or 32 where the output is narrow or gives fewer tiles
  // than SMs (257 x 131 x 700: 18 -> 10 us)
  const long long wide = (M + OZ_BM - 1) / OZ_BM * ((N + 63) / 64);
  int BN = ch.bn ? ch.bn : N <= 32 || wide < 152 ? 32 : 64;
  const int MT = (int)((M + OZ_BM - 1) / OZ_BM), NT = (int)((N + BN - 1) / BN);
  const int KT = (int)((g0.K + OZ_BK - 1) / OZ_BK);
  pa.R = M;
  pa.T = MT;
  pa.TR = OZ_BM;
  pa.KT = KT;
  pb.R = N;
  pb.T = NT;
  pb.TR = BN;
  pb.KT = KT;
  // spread a short output over more CTAs by splitting the k tiles
  int splits = 1, ktper = KT;
  const long long ctas = (long long)MT * NT;
  if (ch.split_mode != 1 && ctas < 2 * 152 && KT >= 2 * OZ_SPLIT_MIN) {
    long long sp = (2 * 152 + ctas - 1) / ctas;
    if (ch.split_mode == 2) sp *= 2;
    if (sp > KT / OZ_SPLIT_MIN) sp = KT / OZ_SPLIT_MIN;
    if (sp >= 2) {
      ktper = (KT + (int)sp - 1) / (int)sp;
      splits = (KT + ktper - 1) / ktper;
    }
  }
  // a tile's integer sums stay within 64 bits for any digits up to 2^26 k: at 8
  // slices the lower half holds 5 pairs of 2^12 a k in units of 2^21, and less
  constexpr int KT_MOST = 1 << 22;
  if (ktper > KT_MOST) {
    ktper = KT_MOST;
    splits = (KT + ktper - 1) / ktper;
  }
  cudaStream_t st = ws.stream;
  const size_t nA = (size_t)S * MT * KT * OZ_TILE_ELEMS, nB = (size_t)S * NT * KT * BN * OZ_BK;
  const WorkspaceBlock bufA(ws, (nA + 3) / 4), bufB(ws, (nB + 3) / 4);  // bf16 digit tiles in double-sized blocks
  const size_t nE = (size_t)MT * OZ_BM + (size_t)NT * BN;
  const WorkspaceBlock bufE(ws, (nE + 2 + 1) / 2);
  const WorkspaceBlock part(ws, splits > 1 ? (size_t)splits * MT * OZ_BM * NT * BN : 0);
  int* ea = (int*)bufE.p;
  int* fb = ea + (size_t)MT * OZ_BM;
  // algorithmic bytes: each operand element read twice (8 B each; once in the
  // one-pass form), S bf16 digits written
  int r = ws.begin(K_OZAKI_PACK, 0.0,
                   ((g0.K <= PACK_SHORT ? 8.0 : 16.0) + 2.0 * S) * (double)(M + N) * (double)g0.K);
  if (r >= 0) {
    ws.recs[r].m = M;
    ws.recs[r].n = N;
    ws.recs[r].k = g0.K;
  }
  PackPass pp{};
  long long w1max = 1, w2max = 1;
  PackPass pd{};
  pd.sq = (unsigned*)ea + nE;
  for (int o = 0; o < 2; ++o) {
    const OzPack& p = o ? pb : pa;
    const long long rows = (long long)p.T * p.TR;
    const long long q1 = (p.K + 7) / 8, q2 = (long long)p.KT * (OZ_BK / 8);
    pp.p[o] = pd.p[o] = p;
    pp.eu[o] = pd.eu[o] = (unsigned*)(o ? fb : ea);
    pp.dst[o] = pd.dst[o] = (__nv_bfloat16*)(o ? bufB.p : bufA.p);
    pp.kfast[o] = pd.kfast[o] = pack_kfast(p);
    pp.fR[o] = pd.fR[o] = make_fastdiv((unsigned)rows);
    pp.fQ[o] = make_fastdiv((unsigned)q1);
    pd.fQ[o] = make_fastdiv((unsigned)q2);
    pp.W[o] = (unsigned)(rows * q1);
    pd.W[o] = (unsigned)(rows * q2);
    w1max = std::max(w1max, rows * q1);
    w2max = std::max(w2max, rows * q2);
  }
  if (g0.K <= PACK_SHORT) {
    unsigned lpr = 1;
    while (lpr < (unsigned)KT * (OZ_BK / 8)) lpr *= 2;
    long long wmax = 1;
    for (int o = 0; o < 2; ++o) {
      const OzPack& p = o ? pb : pa;
      const long long rows = (long long)p.T * p.TR;
      pd.lpr[o] = pd.kfast[o] || rows < PACK_ROWS ? (int)lpr : 0;
      wmax = std::max(wmax, pd.lpr[o] ? rows * lpr : rows);
    }
    const dim3 gs((unsigned)oz_pack_grid(wmax), 2);
    switch (S) {
      case 1: k_ozaki_pack_short<1><<<gs, PACK_T, 0, st>>>(pd); break;
      case 2: k_ozaki_pack_short<2><<<gs, PACK_T, 0, st>>>(pd); break;
      case 3: k_ozaki_pack_short<3><<<gs, PACK_T, 0, st>>>(pd); break;
      case 4: k_ozaki_pack_short<4><<<gs, PACK_T, 0, st>>>(pd); break;
      case 5: k_ozaki_pack_short<5><<<gs, PACK_T, 0, st>>>(pd); break;
      case 6: k_ozaki_pack_short<6><<<gs, PACK_T, 0, st>>>(pd); break;
      case 7: k_ozaki_pack_short<7><<<gs, PACK_T, 0, st>>>(pd); break;
      default: k_ozaki_pack_short<8><<<gs, PACK_T, 0, st>>>(pd); break;
    }
  } else {
    check_cuda(cudaMemsetAsync(ea, 0, (nE + 2) * sizeof(int), st), "cudaMemsetAsync (exponents)");
    k_ozaki_rowexp<<<dim3((unsigned)oz_pack_grid(w1max), 2), PACK_T, 0, st>>>(pp);
    const dim3 g2((unsigned)oz_pack_grid(w2max), 2);
    switch (S) {
      case 1: k_ozaki_digits<1><<<g2, PACK_T, 0, st>>>(pd); break;
      case 2: k_ozaki_digits<2><<<g2, PACK_T, 0, st>>>(pd); break;
      case 3: k_ozaki_digits<3><<<g2, PACK_T, 0, st>>>(pd); break;
      case 4: k_ozaki_digits<4><<<g2, PACK_T, 0, st>>>(pd); break;
      case 5: k_ozaki_digits<5><<<g2, PACK_T, 0, st>>>(pd); break;
      case 6: k_ozaki_digits<6><<<g2, PACK_T, 0, st>>>(pd); break;
      case 7: k_ozaki_digits<7><<<g2, PACK_T, 0, st>>>(pd); break;
      default: k_ozaki_digits<8><<<g2, PACK_T, 0, st>>>(pd); break;
    }
    ws.launches += 1;  // two pack kernels (begin() counts one; the memset is not a kernel)
  }
  ws.end(r);
  a.As = (const __nv_bfloat16*)bufA.p;
  a.Bs = (const __nv_bfloat16*)bufB.p;
  a.ea = ea;
  a.fb = fb;
  a.sq = (const unsigned*)ea + nE;
  a.S = S;
  a.MT = MT;
  a.NT = NT;
  a.KT = KT;
  a.M = M;
  a.N = N;
  a.alpha = g0.alpha;
  {
    int e = 0;
    const double f = std::frexp(g0.alpha, &e);  // +-0.5 for a power of two
    const bool pow2 = std::fabs(f) == 0.5 && e > -500 && e < 500;
    a.alpha_zero = g0.alpha == 0.0 && splits <= 1;  // the tuner's: timed as the power of two it stands for
    a.alpha_fma = !pow2 && !a.alpha_zero && splits <= 1;
    a.alpha_exp = pow2 && splits <= 1 ? e - 1 : 0;
    a.alpha_neg = pow2 && splits <= 1 && f < 0.0;
  }
  for (int d = 0; d < 4; ++d) {
    a.fM[d] = make_fastdiv(d < a.nM ? (unsigned)a.eM[d] : 1u);
    a.fN[d] = make_fastdiv(d < a.nN ? (unsigned)a.eN[d] : 1u);
  }
  a.C = g0.C;
  a.status = ws.oz_status;
  a.wait_cycles = ws.wait_cycles > 0 ? ws.wait_cycles : OZ_WAIT_CYCLES;
  a.splits = splits;
  a.ktper = ktper;
  a.part = part.p;
  a.rowfast = (a.nM > 0 && a.nN > 0 && a.cM[a.nM - 1] < a.cN[a.nN - 1]) || (a.nN == 0 && a.nM > 0) ? 1 : 0;
  // timed as the tensor-core kernel whatever the contraction (kind is the
  // step it belongs to); flops: the FP64 product it computes, executed:
  // digit pairs with t + u <= S + 1 over the padded tiles
  (void)kind;
  const double pairs = (double)S * (S + 1) / 2.0;
  r = ws.begin(K_OZAKI_MMA, 2.0 * (double)M * (double)N * (double)g0.K, 0.0,
               2.0 * pairs * (double)MT * OZ_BM * (double)NT * BN * (double)KT * OZ_BK);
  if (r >= 0) {
    ws.recs[r].m = M;
    ws.recs[r].n = N;
    ws.recs[r].k = g0.K;
  }
  oz_launch_mma(a, MT, NT, BN, st);
  ws.end(r);
  if (splits > 1) ws.launches++;
}

}  // namespace

// Tile width and k split of a split product: fixed rules, or with ws.tune the
// fastest of a few candidates, timed once per (M, N, K, slices) and device on
// the caller's operands with alpha = 0 (C keeps its values bit for bit) and
// cached for the process.  No timing while the stream is being captured.
namespace {
struct OzKey {
  long long M, N, K;
  int S, dev;
  bool operator<(const OzKey& o) const {
    if (M != o.M) return M < o.M;
    if (N != o.N) return N < o.N;
    if (K != o.K) return K < o.K;
    if (S != o.S) return S < o.S;
    return dev < o.dev;
  }
};
std::mutex g_tune_mu;
std::map<OzKey, OzChoice> g_tune;

OzChoice choose(Workspace& ws, const GemmArgs& g0, int S, int kind) {
  OzChoice def;
  if (!ws.tune) return def;
  int dev = 0;
  check_cuda(cudaGetDevice(&dev), "cudaGetDevice");
  const OzKey key{g0.M, g0.N, g0.K, S, dev};
  {
    std::lock_guard<std::mutex> lock(g_tune_mu);
    auto it = g_tune.find(key);
    if (it != g_tune.end()) return it->second;
  }
  int stored[2];
  if (tune_cache_lookup("tile", g0.M, g0.N, g0.K, S, 2, stored)) {
    OzChoice c;
    c.bn = stored[0];
    c.split_mode = stored[1];
    if (c.bn == 32 || c.bn == 64) {
      std::lock_guard<std::mutex> lock(g_tune_mu);
      g_tune[key] = c;
      return c;
    }
  }
  cudaStreamCaptureStatus cs = cudaStreamCaptureStatusNone;
  check_cuda(cudaStreamIsCapturing(ws.stream, &cs), "cudaStreamIsCapturing");
  if (cs != cudaStreamCaptureStatusNone) return def;
  // candidates: tile widths up to about twice the shorter output side, and
  // the k-split rule, no split, twice the rule when the rule splits
  const long long nshort = g0.M < g0.N ? g0.M : g0.N;
  const long long KT = (g0.K + OZ_BK - 1) / OZ_BK;
  std::vector<OzChoice> cands;
  for (int bn : {32, 64}) {
    if (bn != 32 && bn / 2 >= nshort) continue;
    const long long big = g0.M > g0.N ? g0.M : g0.N;
    const long long ctas = ((big + OZ_BM - 1) / OZ_BM) * ((nshort + bn - 1) / bn);
    const bool splits = ctas < 2 * 152 && KT >= 2 * OZ_SPLIT_MIN;
    for (int sm = 0; sm < (splits ? 3 : 1); ++sm) {
      OzChoice c;
      c.bn = bn;
      c.split_mode = sm;
      cands.push_back(c);
    }
  }
  GemmArgs gz = g0;
  gz.alpha = 0.0;
  const TimingScope ts(ws);
  OzChoice best = def;
  float best_ms = 1e30f;
  for (const OzChoice& c : cands) {
    ozaki_run(ws, gz, S, kind, c);  // first run: packing buffers, caches
    check_cuda(cudaEventRecord(ts.e0, ws.stream), "cudaEventRecord");
    ozaki_run(ws, gz, S, kind, c);
    check_cuda(cudaEventRecord(ts.e1, ws.stream), "cudaEventRecord");
    check_cuda(cudaEventSynchronize(ts.e1), "cudaEventSynchronize");
    float ms = 0.f;
    check_cuda(cudaEventElapsedTime(&ms, ts.e0, ts.e1), "cudaEventElapsedTime");
    if (ms < best_ms) {
      best_ms = ms;
      best = c;
    }
  }
  const int v[2] = {best.bn, best.split_mode};
  tune_cache_store("tile", g0.M, g0.N, g0.K, S, 2, v);
  std::lock_guard<std::mutex> lock(g_tune_mu);
  g_tune[key] = best;
  return best;
}
}  // namespace

void ozaki_gemm(Workspace& ws, const GemmArgs& g0, int S, int kind) {
  if (g0.M <= 0 || g0.N <= 0 || g0.K <= 0) return;
  ozaki_run(ws, g0, S, kind, choose(ws, g0, S, kind));
}

}  // namespace dsrg

// ---------------------------------------------------------------------------
// C entry point
// ---------------------------------------------------------------------------
#include "../../include/dsrg.h"

namespace dsrg {
int set_error(int code, const char* msg);
}

extern "C" int dsrg_split_gemm(long long M, long long N, long long K, const double* A, long long lda, const double* B,
                               long long ldb, double* C, long long ldc, double alpha, int slices, void* stream) {
  using namespace dsrg;
  if (M < 0 || N < 0 || K < 0 || M >= (1LL << 31) || N >= (1LL << 31) || K >= (1LL << 31))
    return set_error(DSRG_ERR_ARG, "split gemm: sizes must be in [0, 2^31)");
  if (slices < 1 || slices > kOzakiMaxSlices) return set_error(DSRG_ERR_ARG, "split gemm: slices must be 1..8");
  if (M == 0 || N == 0 || K == 0) return DSRG_OK;
  if (!A || !B || !C) return set_error(DSRG_ERR_ARG, "split gemm: NULL pointer");
  cudaStream_t st = (cudaStream_t)stream;
  try {
    CallWorkspace call(st);
    Workspace& ws = *call.ws;
    const WorkspaceBlock flag(ws, 1);
    ws.oz_status = reinterpret_cast<int*>(flag.p);
    check_cuda(cudaMemsetAsync(ws.oz_status, 0, sizeof(int), st), "status reset");
    GemmArgs g{};
    g.A = A;
    g.B = B;
    g.C = C;
    g.alpha = alpha;
    g.nM = 1;
    g.eM[0] = (int)M;
    g.aM[0] = lda;
    g.cM[0] = ldc;
    g.nN = 1;
    g.eN[0] = (int)N;
    g.bN[0] = 1;
    g.cN[0] = 1;
    g.nK = 1;
    g.eK[0] = (int)K;
    g.aK[0] = 1;
    g.bK[0] = ldb;
    g.M = M;
    g.N = N;
    g.K = K;
    g.nbatch = 1;
    ozaki_gemm(ws, g, slices, K_OZAKI_MMA);
    check_cuda(cudaGetLastError(), "split gemm launch");
    if (ozaki_status(st, ws.oz_status))
      return set_error(DSRG_ERR_TIMEOUT, "split gemm: a bounded wait in the kernel ran out");
  } catch (const Error& e) {
    return set_error(e.code, e.what());
  } catch (const std::exception& e) {
    return set_error(DSRG_ERR_INTERNAL, e.what());
  }
  return DSRG_OK;
}

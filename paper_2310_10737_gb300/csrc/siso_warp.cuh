// siso_warp.cuh -- one warp decodes one component word with soft-output GRAND.
//
// arXiv 2310.10737 (SOGRAND):
//   Sec. III-B  GRAND query loop, membership H x = 0, even-code parity skip;
//   Sec. IV     Corollary: APP of every list word and of "not in the list",
//               phi = (2^k-1)/(2^n-1) (parity class: 2^(n-1) in place of 2^n);
//   Sec. V-B    SISO in/out (L_Ch + L_A -> L_APP, L_E) and eq. LLRi.
// Query order: 1-line ORBGRAND (cited by the paper), cost(z) = sum of the
// reliability ranks in z + c |z|, ties by Hamming weight then lexicographic
// rank vector; c from an exact integer least-squares line through the sorted
// reliabilities quantised to 1/256.
//
// Warp mapping: lane l holds bits l, l+32, ... (NPL per lane).  The word's
// |lambda| are bitonic-sorted across the warp (32-bit keys of |lambda| and the
// index, so ties fall to the lower index; the exact order is restored where
// the key's dropped bits decide) and the H columns are permuted into rank order
// in shared memory.  The query order depends only on (n, c, parity class), so
// it is read from a flattened table, in chunks of 32 consecutive queries: lane
// j takes query q0 + j, XORs its pattern's H columns (those of a shared prefix
// at once) into the syndrome of y and reports a hit; __ballot_sync + __ffs
// keep the hits in query order, so list, stop point and query count are those
// of a sequential decoder.
//
// Remaining mass.  The Corollary needs the mass of the unqueried patterns of
// the parity class, i.e. the class total minus the queried mass.  Every
// pattern mass is the product of per-rank factors t_e = exp(-|lambda_e|)
// (one FP32 value per rank), and the queried masses are formed and summed in
// double-float (an unevaluated pair of floats: Knuth's TwoSum and the
// FMA-based exact product), so the difference is exact for those factors up
// to about 2^-46 of the operands.  It is taken in FP32 when the remainder is
// at least 2% of the operands, in double-float when it is at least 2^-26 of
// them; below that (the list has taken nearly all the mass) the kernel sums
// the unqueried patterns directly (all terms positive): patterns of cost above
// the stop level C* by a dynamic programme over the ranks (cost-indexed,
// parity-split, a pattern is added to the tail the moment one more rank lifts
// it over C*), plus the unqueried rest of level C* from the table.  There the
// masses are cost-scaled by exp(gamma * cost) so that every factor stays <= 1;
// if the scaled total still falls below 2^-60 (all dominant terms underflow)
// or overflows, the same computation is redone in an extended-range float
// (FP32 mantissa + int exponent).
#pragma once
#include <cuda_runtime.h>
#include <math_constants.h>

#include <cstdint>

#include "sg_common.h"

namespace sg {

#ifdef SG_PHASE_PROFILE
// [0] prologue cycles [1] query-loop cycles [2] remainder cycles [3] soft-output
// cycles [4] words [5] query chunks [6] DP words [7] DP ranks [8] XF fallbacks
// Every translation unit has its own copy of the counters (no relocatable
// device code), so each registers a reader that sogrand_debug_phase sums.
__device__ unsigned long long g_phase[16];
#define SG_PROF(i, v) atomicAdd(&g_phase[i], (unsigned long long)(v))
typedef int (*PhaseReader)(unsigned long long *acc, int reset);
void phase_register(PhaseReader r);
namespace {
int phase_read_here(unsigned long long *acc, int reset) {
  unsigned long long v[16];
  if (cudaMemcpyFromSymbol(v, g_phase, sizeof(v)) != cudaSuccess) return 1;
  for (int i = 0; i < 16; i++) acc[i] += v[i];
  if (reset) {
    unsigned long long z[16] = {0};
    if (cudaMemcpyToSymbol(g_phase, z, sizeof(z)) != cudaSuccess) return 1;
  }
  return 0;
}
struct PhaseHook {
  PhaseHook() { phase_register(phase_read_here); }
} phase_hook_;
}  // namespace
#else
#define SG_PROF(i, v) ((void)0)
#endif

constexpr unsigned FULL = 0xffffffffu;
constexpr float LOG2E_F = 1.4426950408889634f;
constexpr float LN2_F = 0.6931471805599453f;

__host__ __device__ constexpr int align16(int x) { return (x + 15) & ~15; }

// ----------------------------------------------------------------------------
// double-float: value = h + l, |l| <= ulp(h) / 2 after df_norm.  Rounded
// intrinsics keep the compiler from contracting the error terms.
// ----------------------------------------------------------------------------
struct DF {
  float h, l;
};
__device__ __forceinline__ DF df_two_sum(float a, float b) {  // Knuth: s + err == a + b exactly
  const float s = __fadd_rn(a, b);
  const float bb = __fsub_rn(s, a);
  return {s, __fadd_rn(__fsub_rn(a, __fsub_rn(s, bb)), __fsub_rn(b, bb))};
}
__device__ __forceinline__ DF df_norm(float h, float l) {  // |h| >= |l| (Dekker's fast two-sum)
  const float s = __fadd_rn(h, l);
  return {s, __fsub_rn(l, __fsub_rn(s, h))};
}
__device__ __forceinline__ DF df_add(DF a, DF b) {
  const DF s = df_two_sum(a.h, b.h), t = df_two_sum(a.l, b.l);
  const DF r = df_norm(s.h, __fadd_rn(s.l, t.h));
  return df_norm(r.h, __fadd_rn(r.l, t.l));
}
// a + b for a, b >= 0 (no cancellation: one TwoSum on the high parts)
__device__ __forceinline__ DF df_add_pos(DF a, DF b) {
  const DF s = df_two_sum(a.h, b.h);
  return df_norm(s.h, __fadd_rn(s.l, __fadd_rn(a.l, b.l)));
}
__device__ __forceinline__ DF df_mul(DF a, DF b) {  // the FMA gives the exact error of a.h * b.h
  const float p = __fmul_rn(a.h, b.h);
  return df_norm(p, fmaf(a.h, b.l, fmaf(a.l, b.h, fmaf(a.h, b.h, -p))));
}
__device__ __forceinline__ DF df_mul_f(DF a, float b) {
  const float p = __fmul_rn(a.h, b);
  return df_norm(p, fmaf(a.l, b, fmaf(a.h, b, -p)));
}
// running sum of nonnegative terms: the low part collects the exact rounding
// errors (the larger high part first: Dekker's fast two-sum, the same exact
// error as Knuth's)
__device__ __forceinline__ void df_acc(DF &a, DF x) {
  const float hi = fmaxf(a.h, x.h), lo = fminf(a.h, x.h);
  const float s = __fadd_rn(hi, lo);
  const float err = __fsub_rn(lo, __fsub_rn(s, hi));
  a.h = s;
  a.l = __fadd_rn(a.l, __fadd_rn(err, x.l));
}
// The warp butterflies that run once per word are loops, unrolled only where
// the kernel's code leaves room in the instruction cache (ROOMY, siso_word).
template <bool ROOMY>
__device__ __forceinline__ DF df_warp_sum(DF x) {  // x >= 0; lane 0's result broadcast (warp-uniform)
  x = df_norm(x.h, x.l);
#pragma unroll(ROOMY ? 5 : 1)
  for (int d = 16; d > 0; d >>= 1)
    x = df_add_pos(x, DF{__shfl_xor_sync(0xffffffffu, x.h, d), __shfl_xor_sync(0xffffffffu, x.l, d)});
  return {__shfl_sync(0xffffffffu, x.h, 0), __shfl_sync(0xffffffffu, x.l, 0)};
}

// ----------------------------------------------------------------------------
// extended-range float: value = m * 2^e, m in [1, 2) (or 0)
// ----------------------------------------------------------------------------
struct XF {
  float m;
  int e;
};
constexpr int XF_ZERO_E = -(1 << 29);

__device__ __forceinline__ XF xf_zero() { return {0.f, XF_ZERO_E}; }
__device__ __forceinline__ XF xf_one() { return {1.f, 0}; }
__device__ __forceinline__ XF xf_norm(float m, int e) {
  if (m == 0.f) return xf_zero();
  int b = __float_as_int(m);
  int ex = ((b >> 23) & 0xff) - 127;
  return {__int_as_float((b & 0x807fffff) | (127 << 23)), e + ex};
}
__device__ __forceinline__ XF xf_mul(XF a, XF b) { return xf_norm(a.m * b.m, a.e + b.e); }
__device__ __forceinline__ XF xf_add(XF a, XF b) {
  if (a.e < b.e) {
    XF t = a;
    a = b;
    b = t;
  }
  int d = b.e - a.e;
  if (d < -40) return a;
  float m = a.m + b.m * __int_as_float((127 + d) << 23);
  return xf_norm(m, a.e);
}
__device__ __forceinline__ XF xf_from_log2(float x) {
  if (!(x > -1e30f)) return xf_zero();
  float f = floorf(x);
  return xf_norm(exp2f(x - f), (int)f);
}
__device__ __forceinline__ float xf_log2(XF a) { return a.m == 0.f ? -CUDART_INF_F : (float)a.e + log2f(a.m); }

// Number policies for the remaining-mass computation.
struct FOps {  // plain FP32, cost-scaled
  using T = float;
  static __device__ __forceinline__ T zero() { return 0.f; }
  static __device__ __forceinline__ T one() { return 1.f; }
  static __device__ __forceinline__ T add(T a, T b) { return a + b; }
  static __device__ __forceinline__ T mul(T a, T b) { return a * b; }
  static __device__ __forceinline__ T fma(T a, T b, T c) { return fmaf(a, b, c); }
  static __device__ __forceinline__ T from_log2(float x) { return exp2f(x); }
  static __device__ __forceinline__ T from_float(float x) { return x; }
  static __device__ __forceinline__ T shfl(T a, int src) { return __shfl_sync(FULL, a, src); }
  static __device__ __forceinline__ T shfl_down(T a, int d) { return __shfl_down_sync(FULL, a, d); }
  static __device__ __forceinline__ T shfl_xor(T a, int d) { return __shfl_xor_sync(FULL, a, d); }
};
struct XOps {  // extended range, unscaled
  using T = XF;
  static __device__ __forceinline__ T zero() { return xf_zero(); }
  static __device__ __forceinline__ T one() { return xf_one(); }
  static __device__ __forceinline__ T add(T a, T b) { return xf_add(a, b); }
  static __device__ __forceinline__ T mul(T a, T b) { return xf_mul(a, b); }
  static __device__ __forceinline__ T fma(T a, T b, T c) { return xf_add(xf_mul(a, b), c); }
  static __device__ __forceinline__ T from_log2(float x) { return xf_from_log2(x); }
  static __device__ __forceinline__ T from_float(float x) { return xf_norm(x, 0); }
  static __device__ __forceinline__ T shfl(T a, int src) {
    return {__shfl_sync(FULL, a.m, src), __shfl_sync(FULL, a.e, src)};
  }
  static __device__ __forceinline__ T shfl_down(T a, int d) {
    return {__shfl_down_sync(FULL, a.m, d), __shfl_down_sync(FULL, a.e, d)};
  }
  static __device__ __forceinline__ T shfl_xor(T a, int d) {
    return {__shfl_xor_sync(FULL, a.m, d), __shfl_xor_sync(FULL, a.e, d)};
  }
};

// ----------------------------------------------------------------------------
// per-warp shared-memory scratch
// ----------------------------------------------------------------------------
// H column and mass factor t = exp(-|lambda|) of one reliability rank, read
// together in the query loop
template <class SYN>
struct RankRec {
  SYN h;
  float t;
};
// |lambda| of one reliability rank and the bit it belongs to, read together
// when a listed word is recorded
struct RankBit {
  float a;
  int bit;
};

// Shared memory of a block: one area per warp (below), then a tail: the lock
// word of the block's remaining-mass area with the lock's poll limit (16
// bytes) and one 16-byte tally slot per warp (summed pattern weights,
// extended-range words), flushed to global counters when the warp exits; then
// (unless the launch puts it in global memory) the remaining-mass area for the
// whole block (the cost DP, needed by about 1% of component decodings or
// fewer).
constexpr int TAIL_BYTES = 16 + 16 * WARPS_PER_BLOCK;

template <int NPL, class SYN>
struct Layout {
  static constexpr int NT = 32 * NPL;
  static constexpr int NM = (NT + 63) / 64;
  static constexpr int o_rb = 0;                                      // RankBit[NT] |lambda| and bit, by rank
  static constexpr int o_hr = o_rb + 8 * NT;  // RankRec[NT + 1] H column + mass factor, by rank; [n] neutral
  static constexpr int o_cw = align16(o_hr + (int)sizeof(RankRec<SYN>) * (NT + 1));  // u64[LMAX][NM] listed codewords
  static constexpr int o_lp = o_cw + 8 * LMAX * NM;                   // float[LMAX] log p(z)/p(0)
  static constexpr int o_wl = o_lp + 4 * LMAX;                        // float[LMAX] APP of each listed word
  static constexpr int o_w = align16(o_wl + 4 * LMAX);                // u64[NT][NM] words of a frame (check)
  // During a word the frame-check area is free: its first 32 bytes hold the
  // word's context (product kernels) and then float[NT] the word's lambda.
  // (A separate area would cost 1 KB per block, which moved the shared-memory
  // carveout of the 8-block schedule up a step and shrank L1 by a quarter.)
  static constexpr int o_lam = o_w + 32;
  static constexpr int HEAD = NPL + 5;  // words after lambda: see Scratch::headv
  static_assert(32 + 4 * NT + 4 * HEAD <= 8 * NT * NM, "lambda and the word head fit in the frame-check area");
  // Prefix records of the query loop (uint4[FAST_SLOTS]); or, where a chunk is
  // tested from the 16-byte entries, uint4[32], the next chunk's entries.
  static constexpr int o_pf = align16(o_w + 8 * NT * NM);
  static constexpr int warp_bytes = o_pf + 16 * (sizeof(SYN) == 4 ? FAST_SLOTS : 32);
  // block area (sized for the 8-byte XF policy): sfac[NT+1], fu[NT+1], fb[NT+1], ek[J] (float), he[J], ho[J]
  static __host__ __device__ int dp_bytes(int jm) { return align16(24 * (NT + 1) + 20 * jm + 32); }
  // a block of WARPS_PER_BLOCK warps: their areas, the tail and the remaining-mass area
  static __host__ __device__ int block_bytes(int jm) { return WARPS_PER_BLOCK * warp_bytes + TAIL_BYTES + dp_bytes(jm); }
};

// A typed pointer to a shared-memory address.  The scratch is carried as 32-bit
// shared addresses: a generic pointer handed to an out-of-line function is
// read with generic loads and 64-bit address arithmetic.
template <class T>
__device__ __forceinline__ T *sptr(unsigned addr) {
  return reinterpret_cast<T *>(__cvta_shared_to_generic((size_t)addr));
}

// A warp's view of the block's scratch: its own area, the block's tail
// (lock word and tally slots, shared memory) and the block's remaining-mass
// area (shared or global memory).  Only the base addresses are kept; every
// array is a fixed offset from them.
template <int NPL, class SYN>
struct Scratch {
  using LY = Layout<NPL, SYN>;
  unsigned base;      // this warp's area (shared address)
  unsigned tl;        // the block's tail (shared address): lock word and poll limit, then the warps' tally slots
  unsigned char *dp;  // the block's remaining-mass area
  __device__ void bind(unsigned char *warp_area, unsigned char *dp_area, unsigned char *tail_area) {
    base = (unsigned)__cvta_generic_to_shared(warp_area);
    dp = dp_area;
    tl = (unsigned)__cvta_generic_to_shared(tail_area);
  }
  __device__ RankBit *rb() const { return sptr<RankBit>(base + LY::o_rb); }
  // |lambda| log2(e) of rank e
  __device__ float l2(int e) const { return __fmul_rn(rb()[e].a, LOG2E_F); }
  __device__ RankRec<SYN> *hr() const { return sptr<RankRec<SYN>>(base + LY::o_hr); }
  __device__ uint64_t *cw() const { return sptr<uint64_t>(base + LY::o_cw); }
  __device__ unsigned *cw32() const { return sptr<unsigned>(base + LY::o_cw); }
  __device__ float *lp() const { return sptr<float>(base + LY::o_lp); }
  __device__ float *wl() const { return sptr<float>(base + LY::o_wl); }
  __device__ uint4 *pf() const { return sptr<uint4>(base + LY::o_pf); }
  __device__ uint4 *prec() const { return sptr<uint4>(base + LY::o_pf); }
  __device__ uint64_t *W() const { return sptr<uint64_t>(base + LY::o_w); }
  // lambda by bit, kept here during the search and read back (volatile) for
  // the soft output, so that it holds no registers while the search runs
  __device__ float *lamv() const { return sptr<float>(base + LY::o_lam); }
  __device__ float lam_at(int i) const { return *sptr<const volatile float>(base + LY::o_lam + 4 * i); }
  // after lambda: the word's hard decision words (NPL) and 1-line parameter,
  // then (threshold rule) which class totals are known, and they
  __device__ unsigned *headv() const { return sptr<unsigned>(base + LY::o_lam + 4 * LY::NT); }
  __device__ unsigned head_at(int k) const { return *sptr<const volatile unsigned>(base + LY::o_lam + 4 * LY::NT + 4 * k); }
  __device__ unsigned char *tail() const { return dp; }
  __device__ int *lock() const { return sptr<int>(tl); }
  // this warp's tally slot: [0] summed pattern weights, [1] extended-range words
  __device__ unsigned long long *tally() const { return sptr<unsigned long long>(tl + 16) + 2 * (threadIdx.x >> 5); }
};

// The block's remaining-mass area is taken by one warp at a time.  Its holder
// runs a bounded computation that waits for nothing, so the wait ends; the
// bound (lock[1] polls, about 4 s by default) only keeps a broken state from
// spinning for ever: the warp then proceeds without the lock and reports it
// (returns false).
__device__ __forceinline__ bool dp_lock(int *lock, int lane) {
  unsigned nap = 32;
  long long tries = 0;
  const long long limit = *reinterpret_cast<volatile int *>(lock + 1);
  bool ok = true;
#pragma unroll 1
  for (;;) {
    int got = 0;
    if (lane == 0) got = atomicCAS(lock, 0, 1) == 0;
    if (__shfl_sync(0xffffffffu, got, 0)) break;
    if (++tries > limit) {
      ok = false;
      break;
    }
    __nanosleep(nap);
    if (nap < 1024) nap <<= 1;
  }
  __threadfence_block();
  return ok;
}
__device__ __forceinline__ void dp_unlock(int *lock, bool held, int lane) {
  __syncwarp();
  __threadfence_block();
  if (lane == 0 && held) atomicExch(lock, 0);
}

// ----------------------------------------------------------------------------
// warp helpers
// ----------------------------------------------------------------------------
// Bitonic sort of the warp's 32 * NPL 32-bit keys, ascending, lane l holding
// sorted positions l NPL .. l NPL + NPL - 1 (blocked: exchanges at distances
// below NPL stay inside a lane's registers, 15 of 21 stages take shuffles for
// 64 keys and 15 of 28 for 128).  Every merge starts by comparing position p
// with p ^ (size - 1), so that the lower position always keeps the smaller
// key: a stage is a shuffle, a minimum or maximum by one bit of the lane, and
// no direction.  Unrolled: 64 keys take about 130 instructions, where 64-bit
// keys sorted in loops with a direction took 600 of a word's 3000.
template <int NPL>
__device__ __forceinline__ void warp_sort_blocked(unsigned (&v)[NPL], int lane) {
  constexpr int N = 32 * NPL;
#pragma unroll
  for (int size = 2; size <= N; size <<= 1) {
#pragma unroll
    for (int j = size >> 1; j > 0; j >>= 1) {
      const bool flip = j == (size >> 1);
      if (j >= NPL) {  // partners in other lanes
        const bool low = (lane & (j / NPL)) == 0;
        unsigned o[NPL];
#pragma unroll
        for (int k = 0; k < NPL; k++)
          o[k] = flip ? __shfl_xor_sync(FULL, v[NPL - 1 - k], size / NPL - 1) : __shfl_xor_sync(FULL, v[k], j / NPL);
#pragma unroll
        for (int k = 0; k < NPL; k++) v[k] = low ? min(v[k], o[k]) : max(v[k], o[k]);
      } else {
#pragma unroll
        for (int k = 0; k < NPL; k++) {
          const int kp = flip ? k ^ (size - 1) : k ^ j;
          if (k < kp) {
            const unsigned lo = min(v[k], v[kp]), hi = max(v[k], v[kp]);
            v[k] = lo;
            v[kp] = hi;
          }
        }
      }
    }
  }
}

// Exact order of the rank records where truncated keys left neighbours
// descending: odd-even transposition on |lambda| (equal values keep their
// order, the lower bit first).  0.02%, 0.16% and 1.3% of 32-, 64- and 128-bit
// words at 3 dB need it, a pass or two each.
template <int NPL>
__device__ __forceinline__ void fix_rank_order(RankBit *rb, int n, int lane) {
  int moved;
  do {
    moved = 0;
#pragma unroll 1
    for (int ph = 0; ph < 2; ph++) {
#pragma unroll
      for (int x = 0; x < (NPL + 1) / 2; x++) {
        const int p = 2 * (lane + 32 * x) + ph;
        if (p + 1 < n) {
          const RankBit u = rb[p], v = rb[p + 1];
          if (u.a > v.a) {
            rb[p] = v;
            rb[p + 1] = u;
            moved = 1;
          }
        }
      }
      __syncwarp();
    }
  } while (__any_sync(FULL, moved));
}

__device__ __forceinline__ float warp_min_f(float x) {
#pragma unroll
  for (int d = 16; d > 0; d >>= 1) x = fminf(x, __shfl_xor_sync(FULL, x, d));
  return x;
}

// floor(v * 256 + 1/2) for v >= 0, saturating at 2^20 - 1.  Exact in FP32:
// v * 256 is a power-of-two scaling, and below the saturation point the sum
// with 1/2 needs no rounding (x < 2^20 has an ulp of at most 2^-4).
__device__ __forceinline__ int quant256(float v) { return __float2int_rd(fminf(fmaf(v, 256.f, 0.5f), 1048575.5f)); }

// 1-line ORBGRAND parameter: intercept/slope of the least-squares line through
// (r, a_r), r = 1..n, rounded half up, clamped to [0, c_max]; 0 if the slope
// is not positive.  With sy = sum a_r, sxy = sum r a_r and B = 2 sxy -
// (n + 1) sy (the slope is 6 B / (n (n^2 - 1))), intercept / slope + 1/2 =
// (sy (n^2 - 1) - 3 n B) / (6 B) exactly, so the parameter is the number of
// c = 1 .. c_max with 6 B c <= sy (n^2 - 1) - 3 n B: one candidate a lane,
// counted by a ballot (the quotient by floating-point estimate and exact
// correction was four times the instructions).  |sxy| < 2^34, so every
// product fits 64 bits.  All lanes get the same value.
template <int NPL>
__device__ __forceinline__ int one_line_c(unsigned sy, int64_t sxy, int n, int c_max, int lane) {
  const int64_t B = 2 * sxy - (int64_t)(n + 1) * sy;
  if (B <= 0) return 0;
  const int64_t den = 6 * B, top = (int64_t)sy * (n * n - 1) - 3 * n * B;
  int c = 0;
#pragma unroll 1
  for (int k = 0; k < NPL; k++) {
    const int cand = lane + 1 + 32 * k;
    const unsigned ok = __ballot_sync(FULL, cand <= c_max && den * cand <= top);
    c += __popc(ok);
    if (ok != FULL) break;  // the candidates that pass are the smallest ones
  }
  return c;
}

// rank k (0-based position in the pattern) of a table entry: byte k + 1
template <int K>
__device__ __forceinline__ int ent_rank(const uint4 &e) {
  constexpr int B = K + 1;
  const unsigned wd = (B >> 2) == 0 ? e.x : (B >> 2) == 1 ? e.y : (B >> 2) == 2 ? e.z : e.w;
  return (wd >> (8 * (B & 3))) & 0xff;
}

// XOR of the rank-ordered H columns of a pattern and its mass relative to
// p(0), the product of its ranks' factors, in double-float (0 for the zero
// pattern).  The loop runs to the warp's largest weight; a shorter pattern's
// extra bytes name the neutral record hr[n] (H column 0, factor 1: the XOR
// and the products are exact no-ops).  Ranks go in pairs: both records are
// loaded before either is used (two shared-memory loads in flight, half the
// branches), and the pair's second rank past the weight is the neutral
// record (2-3% faster than one rank at a time; fours were slower).
template <class SYN>
__device__ __forceinline__ SYN ent_syndrome(const uint4 &e, int w, int wmax, const RankRec<SYN> *hr, DF &mass) {
  SYN s = 0;
  float mh = 1.f, ml = 0.f;
  const auto mul = [&](float t) {
    const float p = __fmul_rn(mh, t);
    ml = fmaf(ml, t, fmaf(mh, t, -p));
    mh = p;
  };
#define SG_R2(K)                                       \
  if (K < wmax) {                                      \
    const RankRec<SYN> v0 = hr[ent_rank<K>(e)];        \
    const RankRec<SYN> v1 = hr[ent_rank<K + 1>(e)];    \
    s ^= v0.h ^ v1.h;                                  \
    mul(v0.t);                                         \
    mul(v1.t);                                         \
  }
  SG_R2(0) SG_R2(2) SG_R2(4) SG_R2(6) SG_R2(8) SG_R2(10) SG_R2(12)
#undef SG_R2
  if (14 < wmax) {
    const RankRec<SYN> v = hr[ent_rank<14>(e)];
    s ^= v.h;
    mul(v.t);
  }
  mass = w > 0 ? DF{mh, ml} : DF{0.f, 0.f};
  return s;
}

// sum over the pattern's ranks of |lambda| log2(e)
template <int NPL, class SYN>
__device__ __forceinline__ float ent_sum(const uint4 &e, int w, const Scratch<NPL, SYN> &sc) {
  float s = 0.f;
#define SG_S(K) \
  if (K < w) s += sc.l2(ent_rank<K>(e));
  SG_S(0) SG_S(1) SG_S(2) SG_S(3) SG_S(4) SG_S(5) SG_S(6) SG_S(7)
  SG_S(8) SG_S(9) SG_S(10) SG_S(11) SG_S(12) SG_S(13) SG_S(14)
#undef SG_S
  return s;
}

// ----------------------------------------------------------------------------
// remaining mass: tail over cost > Cs (DP) + unqueried rest of level Cs
// ----------------------------------------------------------------------------
// The rank DP: he/ho hold the head masses of cost j = 0..Cs by parity, in the
// block's remaining-mass area; rank e lifts cost j by d_e = e + 1 + c.  Slots
// of 32 costs, one cost a lane.  Every term is accumulated before the rank's
// update, by ascending slots below a stop level of 128 (FP32) and by
// descending ones otherwise.  Rolled and short: it runs for fewer than 1% of
// the words, inside the words' kernels.
template <class Ops>
__device__ __forceinline__ void dp_ranks(int Cs, int c, int R0, int cls, const typename Ops::T *sfac,
                                         const typename Ops::T *fu, const typename Ops::T *fb, const float *ek,
                                         typename Ops::T g_even, typename Ops::T g_odd, typename Ops::T *he,
                                         typename Ops::T *ho, int lane, typename Ops::T &acc) {
  using T = typename Ops::T;
  constexpr bool SCALED = sizeof(T) == 4;
  const int nslot = (Cs + 32) >> 5;
#pragma unroll 1
  for (int t = 0; t < nslot; t++) {
    const int j = 32 * t + lane;
    if (j <= Cs) {
      he[j] = j == 0 ? Ops::one() : Ops::zero();
      ho[j] = Ops::zero();
    }
  }
  __syncwarp();
  const bool ascending = SCALED && Cs < 128;
#pragma unroll 1
  for (int e = 0; e <= R0; e++) {
    // e < R0: rank e joins the heads; e == R0: the high ranks (d_e > Cs) join every head
    const bool high = e == R0;
    const int d = e + 1 + c;
    const T s = high ? Ops::one() : sfac[e];
    const T fe = high ? g_even : fb[e + 1];
    const T fo = high ? g_odd : Ops::add(Ops::one(), fu[e + 1]);
#pragma unroll 1
    for (int t = 0; t < nslot; t++) {
      const int j = 32 * (ascending || high ? t : nslot - 1 - t) + lane;
      if (j <= Cs && (high || j > Cs - d)) {
        T w = s;
        if constexpr (SCALED) {
          const T k = Ops::from_float(ek[high ? j : j + d - Cs]);
          w = high ? k : Ops::mul(w, k);
        }
        const T a = he[j], b = ho[j];
        T term;
        if (cls == 0)
          term = Ops::fma(a, fe, Ops::mul(b, fo));
        else if (cls == 1)
          term = Ops::fma(a, fo, Ops::mul(b, fe));
        else
          term = Ops::mul(Ops::add(a, b), Ops::add(fo, fe));
        acc = Ops::fma(w, term, acc);
      }
    }
    __syncwarp();
    if (high) break;
    // slots from the top, so every read of he/ho[j - d] sees the values
    // before this rank (a slot's reads are separated from its writes)
#pragma unroll 1
    for (int sl = nslot - 1; sl >= 0; sl--) {
      const int j = sl * 32 + lane;
      const bool upd = j <= Cs && j >= d;
      T ne = Ops::zero(), no = Ops::zero();
      if (upd) {
        ne = Ops::fma(s, ho[j - d], he[j]);
        no = Ops::fma(s, he[j - d], ho[j]);
      }
      __syncwarp();
      if (upd) {
        he[j] = ne;
        ho[j] = no;
      }
      __syncwarp();
    }
#ifdef SG_PHASE_PROFILE
    if (lane == 0) SG_PROF(7, 1);
#endif
  }
}

// The (scaled) remaining mass summed over the warp.  With FOps every mass
// carries the factor 2^(g2 * Cs) (g2 = gamma log2 e); with XOps g2 = 0.
// `ent` and `cost` are the word's order, `tc` its entries, `qs` the last queried pattern.
// The products with g2 are rounded by themselves (__fmul_rn): left to the
// compiler, each kernel that this is inlined into fused some of them with the
// subtraction that follows, and the same word's mass came out differently with
// and without the threshold rule (by a unit or two in the last place of its
// logarithm).
template <class Ops, int NPL, class SYN>
__device__ __forceinline__ typename Ops::T remaining_scaled(const Scratch<NPL, SYN> &sc, const uint4 *ent,
                                                            const uint16_t *cost, int tc, int qs, int n, int c,
                                                            int cls, int Cs, float g2, int lane) {
  using T = typename Ops::T;
  constexpr int NT = 32 * NPL;
  T *sfac = reinterpret_cast<T *>(sc.tail());
  T *fu = sfac + NT + 1;
  T *fb = fu + NT + 1;
  float *ek = reinterpret_cast<float *>(fb + NT + 1);
  T *he = reinterpret_cast<T *>(ek + align16(4 * (Cs + 1)) / 4);
  T *ho = he + (Cs + 1);
  constexpr bool SCALED = sizeof(T) == 4;
  const int R0 = min(max(Cs - c, 0), n);  // ranks e < R0 can sit inside a pattern of cost <= Cs
  const float g2Cs = __fmul_rn(g2, (float)Cs);

  // --- unqueried rest of level Cs (the table stores every level completely)
  T acc = Ops::zero();
  for (int q0 = qs + 1; q0 < tc; q0 += 32) {
    const int q = q0 + lane;
    bool in = false;
    if (q < tc) in = __ldg(cost + q) == (uint16_t)Cs;
    if (in) {
      const uint4 e = __ldg(ent + q);
      const float s2 = ent_sum<NPL, SYN>(e, e.x & 0xff, sc);
      acc = Ops::add(acc, Ops::from_log2(__fsub_rn(g2Cs, s2)));
    }
    if (!__all_sync(FULL, in)) break;  // costs are nondecreasing
  }

  // --- per-rank factors and suffix products F_e = prod_{e' >= e} (1 + y t_e')
  //     kept as (u, b) = (even part - 1, odd part); lanes own ranks
  //     lane*NPL .. lane*NPL+NPL-1.
  {
    T lu[NPL], lb[NPL];
    T u = Ops::zero(), b = Ops::zero();
#pragma unroll
    for (int k = NPL - 1; k >= 0; k--) {
      const int e = lane * NPL + k;
      T t = Ops::zero();
      if (e < n) {
        t = Ops::from_log2(-sc.l2(e));
        // factor used by the tail: low ranks t * 2^(g2 d_e), high ranks t * 2^(g2 Cs)
        const float d = (float)(e + 1 + c);
        sfac[e] = Ops::from_log2(__fsub_rn(e < R0 ? __fmul_rn(g2, d) : g2Cs, sc.l2(e)));
      }
      const T nu = Ops::fma(b, t, u);
      const T nb = Ops::fma(u, t, Ops::add(b, t));
      u = nu;
      b = nb;
      lu[k] = u;
      lb[k] = b;
    }
    T su = u, sb = b;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
      const T ou = Ops::shfl_down(su, d), ob = Ops::shfl_down(sb, d);
      if (lane + d < 32) {
        const T nu = Ops::add(Ops::add(su, ou), Ops::fma(su, ou, Ops::mul(sb, ob)));
        const T nb = Ops::add(Ops::add(sb, ob), Ops::fma(su, ob, Ops::mul(sb, ou)));
        su = nu;
        sb = nb;
      }
    }
    T xu = Ops::shfl_down(su, 1), xb = Ops::shfl_down(sb, 1);
    if (lane == 31) {
      xu = Ops::zero();
      xb = Ops::zero();
    }
#pragma unroll
    for (int k = 0; k < NPL; k++) {
      const int e = lane * NPL + k;
      if (e < n) {
        fu[e] = Ops::add(Ops::add(lu[k], xu), Ops::fma(lu[k], xu, Ops::mul(lb[k], xb)));
        fb[e] = Ops::add(Ops::add(lb[k], xb), Ops::fma(lu[k], xb, Ops::mul(lb[k], xu)));
      }
    }
    if (lane == 0) {
      fu[n] = Ops::zero();
      fb[n] = Ops::zero();
    }
  }
  if constexpr (SCALED)
#pragma unroll 1
    for (int j0 = 0; j0 <= Cs; j0 += 32)
      if (j0 + lane <= Cs) ek[j0 + lane] = exp2f(-g2 * (float)(j0 + lane));
  __syncwarp();

  // --- high ranks (d_e > Cs): G_P = sum_e sfac_e * F_{e+1} (parity of the
  //     pattern {e} + any higher subset), reduced over the warp
  T g_even = Ops::zero(), g_odd = Ops::zero();
#pragma unroll 1
  for (int e0 = R0; e0 < n; e0 += 32) {
    const int e = e0 + lane;
    if (e < n) {
      const T s = sfac[e];
      g_odd = Ops::fma(s, Ops::add(Ops::one(), fu[e + 1]), g_odd);
      g_even = Ops::fma(s, fb[e + 1], g_even);
    }
  }
#pragma unroll
  for (int d = 16; d > 0; d >>= 1) {
    g_even = Ops::add(g_even, Ops::shfl_xor(g_even, d));
    g_odd = Ops::add(g_odd, Ops::shfl_xor(g_odd, d));
  }

  // --- low ranks in ascending order: tail contributions and the cost DP
  dp_ranks<Ops>(Cs, c, R0, cls, sfac, fu, fb, ek, g_even, g_odd, he, ho, lane, acc);
#pragma unroll
  for (int d = 16; d > 0; d >>= 1) acc = Ops::add(acc, Ops::shfl_xor(acc, d));
  __syncwarp();
  return acc;
}

// Class total of the nonzero patterns in double-float: prod_e (1 + y t_e) as
// (even part - 1, odd part) = (u, b), lanes own ranks lane*NPL ..
// lane*NPL+NPL-1, then a tree over the warp whose root (lane 0's chain) is
// broadcast.  Every term is nonnegative, so the additions need no
// cancellation handling.  Joining two nodes takes the same operations for u
// as for b on other operands, and a level of the tree needs at most 16
// joins: lanes 0-15 form the u parts and lanes 16-31 the b parts, so a level
// is 47 double-float instructions instead of 94, executed and fetched.
template <int NPL, class SYN>
__device__ __forceinline__ DF class_total_df(const Scratch<NPL, SYN> &sc, int n, int cls, int lane) {
  DF u = {0.f, 0.f}, b = {lane * NPL < n ? sc.hr()[lane * NPL].t : 0.f, 0.f};
#pragma unroll 1
  for (int k = 1; k < NPL; k++) {
    const int e = lane * NPL + k;
    if (e < n) {
      const float t = sc.hr()[e].t;
      const DF nu = df_add_pos(u, df_mul_f(b, t));
      const DF nb = df_add_pos(df_add_pos(b, DF{t, 0.f}), df_mul_f(u, t));
      u = nu;
      b = nb;
    }
  }
  const bool odd = lane >= 16;
  DF v = odd ? b : u, w = odd ? u : b;  // own part, other part of the own node
  DF vo, wo;                            // the same parts of the node to join
#pragma unroll 1
  for (int d = 16; d > 0; d >>= 1) {
    if (d == 16) {  // every lane still holds both parts of its own node
      const DF xu = {__shfl_xor_sync(FULL, u.h, 16), __shfl_xor_sync(FULL, u.l, 16)};
      const DF xb = {__shfl_xor_sync(FULL, b.h, 16), __shfl_xor_sync(FULL, b.l, 16)};
      if (odd) {  // this lane's node is the upper one of the pair (lane - 16, lane)
        vo = b;
        wo = u;
        v = xb;
        w = xu;
      } else {
        vo = xu;
        wo = xb;
      }
    } else {
      w = DF{__shfl_xor_sync(FULL, v.h, 16), __shfl_xor_sync(FULL, v.l, 16)};
      vo = DF{__shfl_xor_sync(FULL, v.h, d), __shfl_xor_sync(FULL, v.l, d)};
      wo = DF{__shfl_xor_sync(FULL, w.h, d), __shfl_xor_sync(FULL, w.l, d)};
    }
    // u: (u + ou) + (u ou + b ob);  b: (b + ob) + (u ob + b ou)
    const DF pu = odd ? w : v, pb = odd ? v : w;
    v = df_add_pos(df_add_pos(v, vo), df_add_pos(df_mul(pu, vo), df_mul(pb, wo)));
  }
  u = DF{__shfl_sync(FULL, v.h, 0), __shfl_sync(FULL, v.l, 0)};
  b = DF{__shfl_sync(FULL, v.h, 16), __shfl_sync(FULL, v.l, 16)};
  return cls == 0 ? u : (cls == 1 ? b : df_add_pos(u, b));
}

// The unqueried patterns summed directly: the cost DP of remaining_scaled
// under the block's lock, again in the extended range when every FP32-scaled
// term of the dominant part underflows.  It runs for 0.04-0.9% of the
// component words; inlined all the same, because an out-of-line call keeps
// the whole word's values in the registers that calls preserve (63 spill
// loads a word at 40 registers) and leaves the compiler unsure that the warp
// comes back converged.
// Returns log2 of the mass and flags: bit 0 when the extended-range sum was
// needed, bit 1 when the block's remaining-mass area could not be locked.
struct Remaining {
  float lr2;
  int flags;
};
template <int NPL, class SYN>
__device__ __forceinline__ Remaining remaining_log2_dp(const Scratch<NPL, SYN> &sc, const uint4 *ent,
                                                       const uint16_t *cost, int tc, int qs, int n, int c, int cls,
                                                       int lane) {
#ifdef SG_PHASE_PROFILE
  if (lane == 0) SG_PROF(6, 1);
#endif
  const int Cs = __ldg(cost + qs);
  const int R0 = min(max(Cs - c, 0), n);
  float g = CUDART_INF_F;
#pragma unroll 1
  for (int e0 = 0; e0 < R0; e0 += 32) {
    const int e = e0 + lane;
    if (e < R0) g = fminf(g, sc.l2(e) / (float)(e + 1 + c));
  }
  g = __shfl_sync(FULL, warp_min_f(g), 0);
  if (!(g < CUDART_INF_F)) g = 0.f;
  const bool held = dp_lock(sc.lock(), lane);
  Remaining out = {0.f, 0};
  const float tot =
      __shfl_sync(FULL, remaining_scaled<FOps, NPL, SYN>(sc, ent, cost, tc, qs, n, c, cls, Cs, g, lane), 0);
  if (tot >= 0x1p-60f && tot < CUDART_INF_F) {
    out.lr2 = fmaf(-g, (float)Cs, log2f(tot));  // one rounding of a difference of two large terms
  } else {
    out.flags = 1;
#ifdef SG_PHASE_PROFILE
    if (lane == 0) SG_PROF(8, 1);
#endif
    out.lr2 = __shfl_sync(
        FULL, xf_log2(remaining_scaled<XOps, NPL, SYN>(sc, ent, cost, tc, qs, n, c, cls, Cs, 0.f, lane)), 0);
  }
  dp_unlock(sc.lock(), held, lane);
  if (!held) out.flags |= 2;
  return out;
}

// log2 of the remaining (unqueried) mass relative to p(0^n|r); warp-uniform.
// tq is the queried mass of the nonzero patterns (double-float, summed over
// the warp, the same value in every lane).  The class total minus tq is used
// when it is well conditioned: in FP32 when the difference is at least 2% of
// the operands (FP32 rounding of about 4e-6 of them moves it by at most 2e-4
// relative), in double-float when it is at least 2^-26 of them (rounding of a
// few 2^-46 moves it by at most about 1e-5 relative).  Otherwise the
// unqueried patterns are summed directly.  KEEP: the class totals are kept
// with the word's head (the threshold rule asks at every listed word).
template <bool KEEP, bool ROOMY, int NPL, class SYN>
__device__ __forceinline__ Remaining remaining_log2(const Scratch<NPL, SYN> &sc, const uint4 *ent,
                                                    const uint16_t *cost, int tc, int qs, int n, int cls, int lane,
                                                    DF tq) {
  // class total of the nonzero patterns: prod_e (1 + y t_e) as (even - 1, odd)
  unsigned *kept = sc.headv() + NPL + 1;  // [0] bit 0: [3] is known, bit 1: [1], [2] are
  const unsigned known = KEEP ? __shfl_sync(FULL, sc.head_at(NPL + 1), 0) : 0u;
  float enz;
  if (KEEP && known != 0) {
    enz = __uint_as_float(sc.head_at(NPL + 4));
  } else {
    float u = 0.f, b = 0.f;
#pragma unroll
    for (int k = 0; k < NPL; k++) {
      const int e = lane * NPL + k;
      if (e < n) {
        const float t = sc.hr()[e].t;
        const float nu = fmaf(b, t, u), nb = fmaf(u, t, b + t);
        u = nu;
        b = nb;
      }
    }
#pragma unroll(ROOMY ? 5 : 1)
    for (int d = 16; d > 0; d >>= 1) {
      const float ou = __shfl_xor_sync(FULL, u, d), ob = __shfl_xor_sync(FULL, b, d);
      const float nu = (u + ou) + fmaf(u, ou, b * ob);
      const float nb = (b + ob) + fmaf(u, ob, b * ou);
      u = nu;
      b = nb;
    }
    // the butterfly's fused products round differently per lane: take lane
    // 0's value so the branches below are warp-uniform
    enz = __shfl_sync(FULL, cls == 0 ? u : (cls == 1 ? b : u + b), 0);
    if (KEEP) {
      __syncwarp();
      if (lane == 0) {
        kept[0] = 1u;
        kept[3] = __float_as_uint(enz);
      }
      __syncwarp();
    }
  }
  const float tqf = tq.h + tq.l;
  const float r = enz - tqf;
  if (enz > 0x1p-60f && enz < 0x1p60f) {
    // the hardware log2 (about 2^-22 relative): far inside the soft output's tolerance
    if (r > 0.02f * (enz + tqf)) return {__log2f(r), 0};
    DF E;
    if (KEEP && (known & 2u) != 0) {
      E = DF{__uint_as_float(sc.head_at(NPL + 2)), __uint_as_float(sc.head_at(NPL + 3))};
    } else {
      E = class_total_df<NPL, SYN>(sc, n, cls, lane);
      if (KEEP) {
        if (lane == 0) {
          kept[0] = 3u;
          kept[1] = __float_as_uint(E.h);
          kept[2] = __float_as_uint(E.l);
        }
        __syncwarp();
      }
    }
    const DF R = df_add(E, DF{-tq.h, -tq.l});
#ifdef SG_PHASE_PROFILE
    if (lane == 0) SG_PROF(R.h > 0x1p-26f * (E.h + tq.h) ? 12 : 13, 1);
#endif
    if (R.h > 0x1p-26f * (E.h + tq.h)) return {__log2f(R.h + R.l), 0};
  }
  return remaining_log2_dp<NPL, SYN>(sc, ent, cost, tc, qs, n, (int)sc.head_at(NPL), cls, lane);
}

// numerically safe log(exp(a) + exp(b)) (natural log, -inf aware)
__device__ __forceinline__ float lse(float a, float b) {
  const float mx = fmaxf(a, b), mn = fminf(a, b);
  if (mx == -CUDART_INF_F) return mx;
  return mx + log1pf(expf(mn - mx));
}
__device__ __forceinline__ float softplus(float z) { return fmaxf(z, 0.f) + log1pf(expf(-fabsf(z))); }

// ----------------------------------------------------------------------------
// one word
// ----------------------------------------------------------------------------
template <int NPL, class SYN>
struct WordHead {
  unsigned yb[NPL];  // hard decision, bits lane + 32k
  int par;           // parity of y
  SYN s0;            // syndrome of y
  int c;             // 1-line parameter
};

// Hard decision, parity, syndrome of y, reliability ranks (scratch rb/hr) and
// the 1-line parameter.  The caller has stored lambda in sc.lamv().  Returns
// false (and leaves the head undefined) if any input is not finite.
template <int NPL, class SYN>
__device__ __forceinline__ bool siso_prologue(const DevCode &code, const Scratch<NPL, SYN> &sc, const float (&lam)[NPL],
                                              int lane, WordHead<NPL, SYN> &h) {
  const int n = code.n;
  const SYN *hcol = reinterpret_cast<const SYN *>(code.hcol);  // 8-byte columns: the low half serves 32-bit syndromes
  constexpr int HS = 8 / sizeof(SYN);
  bool bad = false;
#pragma unroll
  for (int k = 0; k < NPL; k++)
    if (lane + 32 * k < n && !(fabsf(lam[k]) < CUDART_INF_F)) bad = true;
  if (__any_sync(FULL, bad)) return false;

  int ones = 0;
  SYN s0p = 0;
#pragma unroll
  for (int k = 0; k < NPL; k++) {
    const int i = lane + 32 * k;
    const bool one = (i < n) && lam[k] < 0.f;  // lambda = 0 -> bit 0
    h.yb[k] = __ballot_sync(FULL, one);
    ones += __popc(h.yb[k]);
    if (one) s0p ^= __ldg(hcol + i * HS);
  }
  h.par = ones & 1;
  if (sizeof(SYN) == 4) {
    h.s0 = (SYN)__reduce_xor_sync(FULL, (unsigned)s0p);
  } else {
    const unsigned lo_ = __reduce_xor_sync(FULL, (unsigned)(uint64_t)s0p);
    const unsigned hi_ = __reduce_xor_sync(FULL, (unsigned)((uint64_t)s0p >> 32));
    h.s0 = (SYN)(((uint64_t)hi_ << 32) | lo_);
  }

  // reliability ranks: sort (|lambda|, index) ascending, on 32-bit keys of
  // |lambda| (its lowest LOGN - 1 mantissa bits dropped) and the index; equal
  // values are in index order, and neighbours that the dropped bits would
  // order otherwise are found by comparing the exact values and exchanged
  constexpr int LOGN = NPL == 1 ? 5 : (NPL == 2 ? 6 : 7);
  unsigned key[NPL];
#pragma unroll
  for (int k = 0; k < NPL; k++) {
    const int i = lane + 32 * k;
    key[k] = i < n ? (((__float_as_uint(lam[k]) << 1) >> LOGN) << LOGN) | i : 0xffffffffu;
  }
  warp_sort_blocked<NPL>(key, lane);
  __syncwarp();  // lambda is in shared memory (siso_word)
  float a[NPL];
  bool wrong = false;
#pragma unroll
  for (int k = 0; k < NPL; k++) {
    const int bit = key[k] & (32 * NPL - 1);
    a[k] = fabsf(sc.lamv()[bit]);
    sc.rb()[lane * NPL + k] = RankBit{a[k], bit};
    if (k > 0 && lane * NPL + k < n) wrong = wrong || a[k - 1] > a[k];
  }
  const float next = __shfl_down_sync(FULL, a[0], 1);
  if (lane < 31 && lane * NPL + NPL < n) wrong = wrong || a[NPL - 1] > next;
  if (__any_sync(FULL, wrong)) {
    __syncwarp();
    fix_rank_order<NPL>(sc.rb(), n, lane);
  }
  unsigned sy = 0, sxy = 0;  // a lane's share: below 2^22 and 2^29
#pragma unroll
  for (int k = 0; k < NPL; k++) {
    const int e = lane * NPL + k;  // sorted position (blocked layout)
    if (e < n) {
      const RankBit r = sc.rb()[e];
      sc.hr()[e] = RankRec<SYN>{__ldg(hcol + r.bit * HS), exp2f(-__fmul_rn(r.a, LOG2E_F))};
      const unsigned qa = (unsigned)quant256(r.a);
      sy += qa;
      sxy += qa * (e + 1);
    }
  }
  // the sum of sy is below 2^27; that of sxy (below 2^34) is taken in two parts
  sy = __reduce_add_sync(FULL, sy);
  const int64_t sxyw = ((int64_t)__reduce_add_sync(FULL, sxy >> 16) << 16) + __reduce_add_sync(FULL, sxy & 0xffffu);
  h.c = one_line_c<NPL>(sy, sxyw, n, code.c_max, lane);
  if (lane == 0) sc.hr()[n] = RankRec<SYN>{(SYN)0, 1.f};  // neutral record for unused entry bytes
  __syncwarp();
  return true;
}

// rank mask (bit r = rank r + 1) of a table entry
template <int NM>
__device__ __forceinline__ void ent_mask(const uint4 &e, uint64_t (&m)[NM]) {
  const int w = e.x & 0xff;
#pragma unroll
  for (int x = 0; x < NM; x++) m[x] = 0;
#define SG_M(K)                                           \
  if (K < w) {                                            \
    const int r = ent_rank<K>(e);                         \
    _Pragma("unroll") for (int x = 0; x < NM; x++) {      \
      if ((r >> 6) == x) m[x] |= 1ull << (r & 63);        \
    }                                                     \
  }
  SG_M(0) SG_M(1) SG_M(2) SG_M(3) SG_M(4) SG_M(5) SG_M(6) SG_M(7)
  SG_M(8) SG_M(9) SG_M(10) SG_M(11) SG_M(12) SG_M(13) SG_M(14)
#undef SG_M
}

// ----------------------------------------------------------------------------
// the query order enumerated by the lanes (instead of read from the table)
// ----------------------------------------------------------------------------
// 1-line ORBGRAND (Sec. III-B) queries the patterns in order of cost = sum of
// ranks + c * weight; the patterns of one cost and weight w are the
// partitions of m = cost - c w into w distinct parts <= n (rank sets), taken
// in lexicographic order of the ascending rank vector.  Pattern o of such a
// group is found part by part: with the parts so far summing to m - m', wl
// parts left and each part above the last one (at least a0), part a is taken
// if o is below the number of ways to finish after it, and otherwise o drops
// by that number and a grows.  The ways to finish after a are the
// (wl - 1)-subsets of {a+1..n} with sum m' - a, i.e. (subtracting a from
// each) the (wl - 1)-subsets of {1..n-a} with sum m' - wl a, read from the
// table of subset counts.  The last two parts follow in closed form: the
// pairs {a, m' - a} in order of a, from max(a0, m' - n).  The pattern is
// written as a table entry (weight byte, 0-based rank bytes, n in the unused
// bytes) into the lane's 16-byte slot and read back.
__device__ __forceinline__ uint4 unrank_entry(const int32_t *scnt, int sc_w, int sc_m, int n, int w, int m, int o,
                                              uint4 *slot) {
  unsigned char *b = reinterpret_cast<unsigned char *>(slot);
  const unsigned nn = (unsigned)n * 0x01010101u;
  *slot = make_uint4((nn & ~0xffu) | (unsigned)w, nn, nn, nn);
  int lo = 1;
#pragma unroll 1
  for (int i = 0; i < w - 2; i++) {
    const int wl = w - i;
    int a = lo;
#pragma unroll 1
    for (; a < n; a++) {  // bounded: for an index inside the group the count is reached by a = n - 1
      const int mm = m - wl * a;
      const int cnt = mm < 0 ? 0 : __ldg(scnt + ((n - a) * sc_w + (wl - 1)) * sc_m + mm);
      if (o < cnt) break;
      o -= cnt;
    }
    b[1 + i] = (unsigned char)(a - 1);
    m -= a;
    lo = a + 1;
  }
  // (the clamps keep every rank byte a valid record index, n the neutral one,
  // whatever the arguments; for an offset inside its group they change nothing)
  if (w >= 2) {
    const int a = max(lo, m - n) + o;
    b[w - 1] = (unsigned char)min(max(a - 1, 0), n);
    b[w] = (unsigned char)min(max(m - a - 1, 0), n);
  } else if (w == 1) {
    b[1] = (unsigned char)min(max(m - 1, 0), n);
  }
  return *slot;
}

// The group window of the lane-enumerated order: the group holding query q
// (warp-uniform: its index g, start gx and record gy) and, for a chunk of 32
// queries q .. q + 31, each lane's group and its offset there, from one
// coalesced load of the next 32 group records (group starts after q are at
// least q + 1, and at most 32 of them fall in q + 1 .. q + 32) and a bit mask
// of the groups that start inside the chunk.  Order (c, class) owns groups
// g0 .. ge - 1.
struct GroupWindow {
  const uint2 *grp;
  int g, ge;
  unsigned gx, gy;
  __device__ __forceinline__ void init(const uint2 *grp_, int g0, int ge_) {
    grp = grp_;
    g = g0;
    ge = ge_;
    gx = 0u;
    gy = g < ge ? __ldg(&grp[g].y) : 0u;
  }
  // lane's pattern for query q + lane (an empty entry for lane >= lim), then
  // the window moves on to the group holding q + 32
  __device__ __forceinline__ uint4 chunk(int q, int lim, int lane, const int32_t *scnt, int sc_w, int sc_m, int n,
                                         uint4 *slot) {
    const int gi = g + 1 + lane;
    const uint2 r = gi < ge ? __ldg(grp + gi) : make_uint2(0x7fffffffu, 0u);
    const int d = (int)r.x - q;
    const unsigned starts = __reduce_or_sync(FULL, d < 32 ? 1u << d : 0u);  // groups starting in the chunk
    const unsigned upto = lane == 31 ? 0xffffffffu : ((2u << lane) - 1u);
    const int rg = __popc(starts & upto);  // groups started after q and at or before q + lane
    const unsigned sx = __shfl_sync(FULL, r.x, rg > 0 ? rg - 1 : 0);
    const unsigned sy = __shfl_sync(FULL, r.y, rg > 0 ? rg - 1 : 0);
    const unsigned my = rg > 0 ? sy : gy;
    const int mo = q + lane - (int)(rg > 0 ? sx : gx);
    uint4 e = make_uint4(0u, 0u, 0u, 0u);
    if (lane < lim) e = unrank_entry(scnt, sc_w, sc_m, n, (int)(my >> 16), (int)(my & 0xffffu), mo, slot);
    const int adv = __popc(__ballot_sync(FULL, d <= 32));
    if (adv > 0) {
      gx = __shfl_sync(FULL, r.x, adv - 1);
      gy = __shfl_sync(FULL, r.y, adv - 1);
      g += adv;
    }
    return e;
  }
};

// The canonical query order for one input (test hook): writes the first
// max_q rank masks (NM words each); returns how many were written.
template <int NPL, class SYN>
__device__ int trace_word(const DevCode &code, const Scratch<NPL, SYN> &sc, const float (&lam)[NPL], int lane,
                          int max_q, uint64_t *out, int *c_out) {
  constexpr int NM = (32 * NPL + 63) / 64;
  WordHead<NPL, SYN> h;
#pragma unroll
  for (int k = 0; k < NPL; k++) sc.lamv()[lane + 32 * k] = lam[k];
  if (!siso_prologue<NPL, SYN>(code, sc, lam, lane, h)) return -1;
  const DevOrder &O = code.ord;
  const int ti = h.c * O.ncls + (code.even ? h.par : 0);
  const int tb = __ldg(O.base + ti), tc = __ldg(O.count + ti);
  const int qn = min(max_q, tc);
  if (code.ord_lanes) {  // the order as the lanes enumerate it
    GroupWindow W;
    W.init(code.grp.grp, __ldg(code.grp.gbase + ti), __ldg(code.grp.gbase + ti + 1));
    for (int q0 = 0; q0 < qn; q0 += 32) {
      const uint4 e = W.chunk(q0, min(32, qn - q0), lane, code.grp.scnt, code.grp.sc_w, code.grp.sc_m, code.n,
                              sc.pf() + lane);
      if (q0 + lane < qn) {
        uint64_t m[NM];
        ent_mask<NM>(e, m);
#pragma unroll
        for (int x = 0; x < NM; x++) out[(size_t)(q0 + lane) * NM + x] = m[x];
      }
    }
  } else {
    for (int q = lane; q < qn; q += 32) {
      uint64_t m[NM];
      ent_mask<NM>(__ldg(O.ent + tb + q), m);
#pragma unroll
      for (int x = 0; x < NM; x++) out[(size_t)q * NM + x] = m[x];
    }
  }
  if (c_out && lane == 0) *c_out = h.c;
  return qn;
}

// Threshold rule: whether the predicted probability that the list misses the
// codeword, e^M / (e^M + sum_l e^lp_l), is below thr.  With s = sum_l
// e^(lp_l - M) that is thr (1 + s) > 1.  The hardware exponential gives s to
// about 1e-5, so outside a band around 1 it decides; inside, the accurate
// functions do (they took about 60 instructions a list word, at every list
// word).  Their sum is taken in the log domain and is itself off by up to an
// ulp of M a list word (16 of them: 1e-6 |M|), so the band grows with |M|.
// Thresholds below the smallest normal number, where s overflows and the
// probability is a denormal, are left to them altogether.
__device__ __forceinline__ bool thr_reached(const float *lp, int nhit, float M, float thr) {
  float s = 1.f;
#pragma unroll 1
  for (int l = 0; l < nhit; l++) s += __expf(lp[l] - M);
  const float x = thr * s;
  const float band = thr >= 0x1p-126f ? fmaf(fabsf(M), 2e-6f, 1e-3f) : CUDART_INF_F;
  if (x > 1.f + band || x < 1.f - band) return x > 1.f;
  float D = M;
#pragma unroll 1
  for (int l = 0; l < nhit; l++) D = lse(D, lp[l]);
  return expf(M - D) < thr;
}

// eq. LLRi in the log domain for a bit whose linear sums underflowed (out of line: rare)
template <int NPL, class SYN>
__device__ __noinline__ float lapp_logdomain(const Scratch<NPL, SYN> &sc, int nhit, float M, float x, int i) {
  constexpr int NM = (32 * NPL + 63) / 64;
  float b0 = M - softplus(-x), b1 = M - softplus(x);
  const uint64_t bitm = 1ull << (i & 63);
  for (int l = 0; l < nhit; l++) {
    if (sc.cw()[l * NM + (i >> 6)] & bitm)
      b1 = lse(b1, sc.lp()[l]);
    else
      b0 = lse(b0, sc.lp()[l]);
  }
  return b0 - b1;
}

// Record list words l0 .. l1 - 1 of a search from their query indices (lane l
// holds hq of list word l): the codeword y + z in bit order (sc.cw()) and
// log p(z)/p(0) = -sum |lambda| over z (sc.lp()).  Two words at a time, 16
// lanes each: lane k of a half takes the pattern's k-th rank from the order
// table `ent` (one byte load; lane 15 the weight).  Without the threshold
// rule the list is recorded once, after the search.  The sum's butterfly adds
// the same values in the same order as one over 32 lanes whose upper half
// holds zeros.
template <int NPL, class SYN>
__device__ __forceinline__ void record_list(const Scratch<NPL, SYN> &sc, const uint4 *ent, int hq, int l0, int l1,
                                            int lane) {
  constexpr int NM = (32 * NPL + 63) / 64;
  const int k = lane & 15;
  int l = l0 + (lane >> 4);
  const auto load = [&]() {  // list word l's byte of this lane
    const int q = __shfl_sync(FULL, hq, l & 31);
    return l < l1 ? (int)__ldg(reinterpret_cast<const uint8_t *>(ent + q) + ((k + 1) & 15)) : 0;
  };
  int nxt = load();
  const int xw = lane & (2 * NM - 1);
  const unsigned yw = xw < NPL ? sc.head_at(xw) : 0u;  // this lane's word of y
#pragma unroll
  for (int i = lane; i < LMAX * 2 * NM; i += 32)
    if (i >= l0 * 2 * NM && i < l1 * 2 * NM) sc.cw32()[i] = yw;
  __syncwarp();
#pragma unroll 1
  for (; l0 < l1; l0 += 2) {
    const int at = l, v = nxt;
    l += 2;
    nxt = load();
    const int w = __shfl_sync(FULL, v, lane | 15);  // 0 past the list
    RankBit rb = {0.f, 0};
    if (k < w) {
      rb = sc.rb()[v];
      atomicXor(sc.cw32() + at * 2 * NM + (rb.bit >> 5), 1u << (rb.bit & 31));
    }
#pragma unroll
    for (int d = 8; d > 0; d >>= 1) rb.a += __shfl_xor_sync(FULL, rb.a, d);
    if (k == 0 && at < l1) sc.lp()[at] = -rb.a;
  }
  __syncwarp();
}

// ----------------------------------------------------------------------------
// the search
// ----------------------------------------------------------------------------
// Chunks of 32 queries, lane j testing query q0 + j; hits are taken in query
// order until L codewords are listed, the cap is reached or the threshold rule
// applies.
//
// Prefix records.  A pattern of weight w costs a byte extract, a record load,
// an XOR and a three-operation product for every rank.  In 1-line ORBGRAND
// order the patterns of many consecutive queries share their low ranks:
// without its last two ranks, the first thousand queries' patterns have only
// 32 different prefixes, and without the last three the first nine thousand
// have 64.  So the word first computes each prefix's record {syndrome of y XOR
// its H columns, mass in double-float, weight} once, one lane each, and then
// every query costs one 16-byte record, two (three) rank records and one
// compact 4-byte entry {slot, ranks}, read a chunk ahead into a register (the
// 16-byte entries cost four times the L2 traffic).  The factors are multiplied
// in the same ascending order, so masses are bit for bit those of the
// rank-by-rank product.  A word starts in the two-rank form (one 32-lane build
// step), goes on in the three-rank form (two build steps), and past that, and
// for a last partial chunk, tests the 16-byte entries rank by rank
// (ent_syndrome).  64-bit syndromes leave no room for the record in 16 bytes
// and always take the last form.

struct FalseTag {
  static constexpr bool value = false;
};
struct TrueTag {
  static constexpr bool value = true;
};

// Where the query loop takes its patterns and when it stops.
enum : int {
  MODE_TABLE = 0,  // the order tables, no threshold rule
  MODE_LANES = 1,  // enumerated by the lanes (DevCode::ord_lanes), no threshold rule
  MODE_THR = 2     // the order tables, the threshold rule asked at every listed word
};

// Compute the records of `count` prefix slots.
template <int NPL, class SYN>
__device__ __forceinline__ void build_prefixes(const Scratch<NPL, SYN> &sc, SYN s0, const uint2 *slots, int count,
                                               int lane) {
  __syncwarp();  // every lane is done with the previous records
#pragma unroll 1
  for (int i0 = 0; i0 < count; i0 += 32) {  // count is a multiple of 32
    uint2 d = __ldg(slots + i0 + lane);
    const int len = d.x & 15, w = len + ((d.x >> 4) & 15);
    const int longest = (int)__reduce_max_sync(FULL, (unsigned)len);
    unsigned h = (unsigned)s0;
    float mh = w > 0 ? 1.f : 0.f, ml = 0.f;  // the zero pattern has no queried mass
#pragma unroll 1
    for (int k = 0; k < longest; k++) {
      d.x = __funnelshift_r(d.x, d.y, 8);
      d.y >>= 8;
      if (k < len) {
        const RankRec<SYN> v = sc.hr()[d.x & 0xff];
        h ^= (unsigned)v.h;
        const float p = __fmul_rn(mh, v.t);
        ml = fmaf(ml, v.t, fmaf(mh, v.t, -p));
        mh = p;
      }
    }
    sc.prec()[i0 + lane] = make_uint4(h, __float_as_uint(mh), __float_as_uint(ml), (unsigned)w);
  }
  __syncwarp();
}

// lam[k] is bit lane + 32k of the SISO input lambda = fl32(L_Ch + L_A)
// (the caller loads it; entries past n are ignored).  L_APP is handed to
// emit(k, x, lapp, listed) for k = 0 .. NPL - 1 in turn: bit lane + 32k, its
// lambda x and whether the word's list holds a word (else lapp = x), after
// begin().  res gets the per-word results (before the first emit); the list (in query order) is
// left in the scratch: sc.cw() (codewords, natural bit order), sc.lp() (log
// p(z)/p(0)) and sc.wl() (APP of each word).  res.flags collects
// the remaining-mass flags (bit 0: extended range; bit 1: the block's
// remaining-mass area could not be locked).
//
// Loops whose trip count differs between lanes are avoided throughout: after
// one the compiler no longer knows the warp to be converged, and every later
// shuffle and vote of the kernel pays for a check (about 135 instructions a
// word when only the rarely run remaining-mass sums had such loops).
//
// What bounds a word is instruction fetch and issue: a word runs about two
// thousand instructions once each around a short query loop, and the warps of
// an SM are in different phases of their words, so the whole word's code
// competes for the SM's instruction cache.  Everything that runs once per word
// is therefore written for few instructions: lanes share what a single lane
// could do (list words' APPs, candidates of the 1-line parameter), and loops
// over the list and over a lane's bits stay rolled.  ROOMY: the kernel has
// little other code (k_decode), and the per-word sums are unrolled (2% faster
// there; in the batched kernel they pushed the code past the instruction cache,
// 4% slower).
template <int NPL, class SYN, int MODE, bool ROOMY, class Begin, class Emit>
__device__ __forceinline__ void siso_word(const DevCode &code, const SisoParams &P, const Scratch<NPL, SYN> &sc,
                                          const float (&lam)[NPL], int lane, WordResult &res, Begin begin, Emit emit) {
  using LY = Layout<NPL, SYN>;
  constexpr int NM = (32 * NPL + 63) / 64;
  const int n = code.n;
#ifdef SG_PHASE_PROFILE
  const long long t0 = clock64();
#endif
#pragma unroll
  for (int k = 0; k < NPL; k++) sc.lamv()[lane + 32 * k] = lam[k];  // each lane reads back its own
  WordHead<NPL, SYN> h;
  res.flags = res.wsum = res.nhit = 0;
  res.queries = -1;
  res.pmiss = 1.f;
  if (!siso_prologue<NPL, SYN>(code, sc, lam, lane, h)) {
    begin();
#pragma unroll 1
    for (int k = 0; k < NPL; k++) {
      const float x = sc.lam_at(lane + 32 * k);
      emit(k, x, x, false);
    }
    return;
  }
#ifdef SG_PHASE_PROFILE
  const long long t1 = clock64();
#endif

  // the order of (c, class)
  const DevOrder &O = code.ord;
  const int cls = code.even ? h.par : -1;
  const int ti = h.c * O.ncls + (code.even ? h.par : 0);
  if (lane == 0) {
#pragma unroll
    for (int k = 0; k < NPL; k++) sc.headv()[k] = h.yb[k];
    sc.headv()[NPL] = (unsigned)h.c;
    if (MODE == MODE_THR) sc.headv()[NPL + 1] = 0u;  // the class totals are not known yet
  }
  __syncwarp();
  const int tb = __ldg(O.base + ti), tc = __ldg(O.count + ti);
  const int qlim = min(P.cap, tc);
  const uint4 *ent = O.ent + tb;

  int q = 0, nhit = 0;    // the chunk's first query, the list
  int hq = 0;             // lane l: the query index of list word l
  int wacc = 0;           // this lane's share of the summed pattern weights
  DF tmass = {0.f, 0.f};  // and of the queried mass (nonzero patterns)
  GroupWindow win;
  if constexpr (MODE == MODE_LANES)
    win.init(code.grp.grp, __ldg(code.grp.gbase + ti), __ldg(code.grp.gbase + ti + 1));
  // zone 0: two-rank form, 1: three-rank form, 2: 16-byte entries (or the lanes' patterns), 3: the end
  int zone = -1, qe = 0;
  unsigned hm = 0;  // the current chunk's hits still to take
  int lim = 32, w = 0;
  DF mass = {0.f, 0.f};
  const uint4 *e4 = O.e4 + (size_t)ti * O.e4_stride + lane;
  uint4 e = make_uint4(0u, 0u, 0u, 0u), en = e;  // this lane's entries of the current group of chunks and the next
  // takes the chunk's hits in order: the lane of the one the search leaves at, or -1
  const auto take = [&]() {
    do {
      const int at = __ffs(hm) - 1;
      hm &= hm - 1;
      if (lane == nhit) hq = q + at;
      nhit++;
      if (MODE == MODE_THR || nhit >= P.L) return at;
    } while (hm != 0);
    return -1;
  };
  const auto queried = [&]() {  // the whole chunk has been queried
    wacc += w;
    df_acc(tmass, mass);
    q += lim;
  };
  int listed = 0;  // list words recorded so far
  float M;         // log (R phi), natural
#ifdef SG_PHASE_PROFILE
  long long t2 = 0;
#endif
#pragma unroll 1
  for (;;) {
    // the search proper: to the hit that completes the list (MODE_THR: to the
    // next hit), or to the end
    int hl = -1;
    if (MODE == MODE_THR && hm != 0) {
      hl = take();
      goto left;
    }
#pragma unroll 1
    for (;;) {
      if (q >= qe) {
        zone++;
        if (zone >= 3) break;
        lim = 32;
        qe = qlim;
        if (MODE != MODE_LANES && zone == 2)
          en = __ldg(ent + min(q + lane, tc - 1));
        if (zone < 2) {
          qe = 0;
          if constexpr (MODE != MODE_LANES && sizeof(SYN) == 4) {
            const int2 z = __ldg(O.zones + ti);
            qe = min(zone ? z.y : z.x, qlim & ~127);
            if (q < qe) {
              e = __ldg(e4 + (q >> 2));
              en = __ldg(e4 + (q >> 2) + 32);
              build_prefixes<NPL, SYN>(sc, h.s0, O.slots + ti * (FAST_SLOTS2 + FAST_SLOTS) + (zone ? FAST_SLOTS2 : 0),
                                       zone ? FAST_SLOTS : FAST_SLOTS2, lane);
            }
          }
        }
      } else if (MODE != MODE_LANES && sizeof(SYN) == 4 && zone < 2) {
        // full chunks, two at a time: the record of each entry's prefix, then
        // its last ranks.  Both chunks are tested before either is taken, so
        // a warp alone on its SM waits for one chunk's loads and products, not
        // two.  (MODE_THR can resume at a pair's second chunk.)
        const unsigned prec = sc.base + LY::o_pf, hr = sc.base + LY::o_hr;
        const auto test = [&](unsigned cur, auto three, DF &m, int &wt) {
          const uint4 r = *sptr<const uint4>(prec + 16 * __byte_perm(cur, 0u, 0x4440));
          unsigned s = r.x;
          m = DF{__uint_as_float(r.y), __uint_as_float(r.z)};
          wt = (int)r.w;
          const auto rank = [&](unsigned byte) {
            const RankRec<SYN> v = *sptr<const RankRec<SYN>>(hr + 8 * byte);
            s ^= (unsigned)v.h;
            const float p = __fmul_rn(m.h, v.t);
            m.l = fmaf(m.l, v.t, fmaf(m.h, v.t, -p));
            m.h = p;
          };
          rank(__byte_perm(cur, 0u, 0x4441));
          rank(__byte_perm(cur, 0u, 0x4442));
          if constexpr (decltype(three)::value) rank(cur >> 24);
          return s;
        };
        const auto pairs = [&](auto three) {  // whether the search leaves
#pragma unroll 1
          do {
            DF ma, mb;
            int wa, wb;
            const unsigned sa = test(e.x, three, ma, wa), sb = test(e.y, three, mb, wb);
            const unsigned ha = __ballot_sync(FULL, sa == 0), hb = __ballot_sync(FULL, sb == 0);
            if (MODE != MODE_THR || (q & 32) == 0) {
              if (ha != 0) {
                hm = ha;
                mass = ma;
                w = wa;
                hl = take();
                if (hl >= 0) return true;
              }
              wacc += wa;
              df_acc(tmass, ma);
              q += 32;
            }
            e.x = e.z;
            e.y = e.w;
            if ((q & 64) != 0) {  // the next group of entries
              e = en;
              en = __ldg(e4 + (q >> 2) + 64 - ((q >> 2) & 31));
            }
            if (hb != 0) {
              hm = hb;
              mass = mb;
              w = wb;
              hl = take();
              if (hl >= 0) return true;
            }
            wacc += wb;
            df_acc(tmass, mb);
            q += 32;
          } while (q < qe);
          return false;
        };
        // a loop for each form: a predicated third rank would cost the
        // two-rank form its instructions
        if (zone == 0) {
          if (pairs(FalseTag{})) goto left;
        } else {
          if (pairs(TrueTag{})) goto left;
        }
      } else {
        // rank by rank, the entries read a chunk ahead
#pragma unroll 1
        do {
          lim = min(32, qlim - q);
          uint4 ee;
          if constexpr (MODE == MODE_LANES) {
            ee = win.chunk(q, lim, lane, code.grp.scnt, code.grp.sc_w, code.grp.sc_m, n, sc.pf() + lane);
          } else {
            // an empty entry past the end (selected, not branched to: a branch
            // on the lane here costs the kernel its proof of convergence)
            ee.x = lane < lim ? en.x : 0u;
            ee.y = lane < lim ? en.y : 0u;
            ee.z = lane < lim ? en.z : 0u;
            ee.w = lane < lim ? en.w : 0u;
            en = __ldg(ent + min(q + 32 + lane, tc - 1));
          }
          w = ee.x & 0xff;
          const int wmax = (int)__reduce_max_sync(FULL, (unsigned)w);
          const SYN s = ent_syndrome<SYN>(ee, w, wmax, sc.hr(), mass) ^ h.s0;
          hm = __ballot_sync(FULL, lane < lim && s == 0);
          if (hm != 0) {
            hl = take();
            if (hl >= 0) goto left;
          }
          queried();  // lanes past lim hold an empty entry
        } while (q < qlim);
      }
    }
  left:
#ifdef SG_PHASE_PROFILE
    if (t2 == 0) t2 = clock64();
#endif
    // the list is complete, or the order or the cap ended
    const bool fin = nhit >= P.L || zone >= 3;
    record_list<NPL, SYN>(sc, ent, hq, listed, nhit, lane);
    listed = nhit;
    // the queries made up to here: qn, their mass `part`
    const int qn = hl >= 0 ? q + hl + 1 : q;
    DF part = tmass;
    if (lane <= hl) df_acc(part, mass);
    Remaining rem = {-CUDART_INF_F, 0};
    // when the whole parity class has been queried nothing remains
    if (!(fin && qn >= tc && tc == O.class_size) && !P.forney)
      rem = remaining_log2<MODE == MODE_THR, ROOMY, NPL, SYN>(sc, ent, O.cost + tb, tc, qn - 1, n, cls, lane,
                                                       df_warp_sum<ROOMY>(part));
    res.flags |= rem.flags;
    M = fmaf(rem.lr2, LN2_F, code.log_phi);
    if (MODE != MODE_THR || fin || thr_reached(sc.lp(), nhit, M, P.thr)) {
      if (lane <= hl) wacc += w;
      q = qn;
      break;
    }
    if (hm == 0) queried();  // that was the chunk's last hit
  }
#ifdef SG_PHASE_PROFILE
  if (lane == 0) SG_PROF(5, (q + 31) / 32);
  const long long t3 = clock64();
#endif
  res.wsum = (int32_t)__reduce_add_sync(FULL, (unsigned)wacc);
  res.queries = q;
  res.nhit = nhit;
  // log(R phi + sum_l p_l), all relative to p(0): max plus log of a sum
  // (lane l takes list word l; the terms are added in list order).  The
  // hardware exponential and logarithm (relative errors near 2^-21 over
  // these ranges) keep L_APP within about 1e-5 of the exact formula, far
  // inside the soft output's tolerance; no decision is taken on them.
  const float lp = lane < nhit ? sc.lp()[lane] : -CUDART_INF_F;
  // log masses are <= 0: the largest has the smallest magnitude bits
  const float mx = fmaxf(M, -__uint_as_float(__reduce_min_sync(FULL, __float_as_uint(-lp) & 0x7fffffffu)));
  float sum = M == -CUDART_INF_F ? 0.f : __expf(M - mx);
  const float el = __expf(lp - mx);
#pragma unroll 1
  for (int l = 0; l < nhit; l++) sum += __shfl_sync(FULL, el, l);
  const float D = mx + __logf(sum);
  const float pm = M == -CUDART_INF_F ? 0.f : __expf(M - D);
  if (nhit > 0) res.pmiss = pm;
  // APP of each listed word (list weights relative to the normaliser)
  const float wl = __expf(lp - D);
  if (lane < nhit) sc.wl()[lane] = wl;
  // eq. LLRi: the miss term, then each listed word adds its APP to the side
  // of its bit
  begin();
#pragma unroll(ROOMY ? NPL : 1)
  for (int k = 0; k < NPL; k++) {
    const float x = sc.lam_at(lane + 32 * k);
    // sigma(x) and sigma(-x) without cancellation
    const float ex = __expf(-fabsf(x));
    const float sp = __fdividef(1.f, 1.f + ex), sn = ex * sp;  // sigma(|x|), sigma(-|x|)
    float a0 = pm * (x >= 0.f ? sp : sn);                       // miss term, bit 0
    float a1 = pm * (x >= 0.f ? sn : sp);                       // miss term, bit 1
#pragma unroll 1
    for (int l = 0; l < nhit; l++) {
      const float wlv = __shfl_sync(FULL, wl, l);
      if ((sc.cw32()[l * 2 * NM + k] >> lane) & 1u)
        a1 += wlv;
      else
        a0 += wlv;
    }
    // both sums lie in (1e-30, 1 + 1e-6]: __fdividef's range
    float lapp = x;
    if (nhit > 0)
      lapp = (a0 > 1e-30f && a1 > 1e-30f) ? __logf(__fdividef(a0, a1))
                                          : lapp_logdomain<NPL, SYN>(sc, nhit, M, x, lane + 32 * k);
    emit(k, x, lapp, nhit > 0);
  }
  __syncwarp();
#ifdef SG_PHASE_PROFILE
  const long long t4 = clock64();
  if (lane == 0) {
    SG_PROF(0, t1 - t0);
    SG_PROF(1, t2 - t1);
    SG_PROF(2, t3 - t2);
    SG_PROF(3, t4 - t3);
    SG_PROF(4, 1);
  }
#endif
}

}  // namespace sg

// kernels.cuh -- __global__ kernels and their launchers (instantiated per lane
// width in inst_npl*.cu).
//
//   k_decode        sogrand_decode: warp-per-word SISO over many independent
//                   component words (Sec. V-B, Fig. siso);
//   k_trace         test hook: the canonical query order of one word;
//   k_product_half  one half iteration of block turbo decoding (Sec. VI,
//                   steps 1/2): every row (odd half) or column (even half) of
//                   every running frame is decoded with lambda = L_Ch +
//                   alpha L_E(previous half) and its L_E and hard decision are
//                   stored;
//   k_product_check hard decision of the whole frame: every row and every
//                   column must satisfy H x = 0 (Sec. VI), else continue.
#pragma once
#include <algorithm>

#include "launch.h"
#include "siso_warp.cuh"

namespace sg {

constexpr int TPB = 32 * WARPS_PER_BLOCK;

// Resident blocks per SM that a schedule's kernels are compiled for.  Schedule
// 8 takes 64 registers a thread; schedule 12 (its name: the second value of
// sogrand_code_schedule) 56 registers, which is 9 blocks.  The launch is bound
// by issue and the instruction cache, not by latency that more warps would
// hide, and more blocks leave less L1 (eBCH(64,57)^2, 20,000 frames: 21.0 ms
// at 7 blocks, 20.3 at 8, 20.1 at 9, 21.3 at 10; at 12 the code also spills).
__host__ __device__ constexpr int resident_blocks(int minb) { return minb == 12 ? 9 : minb; }

// The warp's index in its block, broadcast so that the compiler knows it to be
// the same in every lane: the words' control flow is then provably uniform
// and needs no divergence handling around its shuffles and votes.
__device__ __forceinline__ int warp_index() { return __shfl_sync(FULL, (int)(threadIdx.x >> 5), 0); }

// dynamic shared memory of one block of a single-code kernel
template <int NPL, class SYN>
__host__ __device__ inline int block_scratch_bytes(int jmax) {
  return Layout<NPL, SYN>::block_bytes(jmax);
}

// The block's tail (lock word of its remaining-mass area and the warps'
// tally slots) in shared memory after the warps' areas (`wstride` bytes
// each); the remaining-mass area after the tail, or the block's own slice of
// a global region when the launch passes one.  The area serves about 1% of
// component decodings or fewer; in global memory it leaves the SM's on-chip
// memory to L1, which holds the hot query-order entries (a block of a long
// code kept 14 KB of shared memory for it).
__device__ __forceinline__ unsigned char *block_tail(unsigned char *smem, int wstride) {
  return smem + WARPS_PER_BLOCK * wstride;
}
__device__ __forceinline__ unsigned char *block_dp_area(unsigned char *smem, int wstride, unsigned char *dp_global,
                                                        int dp_stride) {
  return dp_global ? dp_global + (size_t)blockIdx.x * dp_stride : block_tail(smem, wstride) + TAIL_BYTES;
}

// Bind warp `warp`'s view: its area in shared memory (`wstride` bytes a warp),
// the block's remaining-mass area `dpb` and tail `tl`.
template <int NPL, class SYN>
__device__ __forceinline__ void bind_scratch(Scratch<NPL, SYN> &sc, unsigned char *smem, int warp, int wstride,
                                             unsigned char *dpb, unsigned char *tl) {
  sc.bind(smem + warp * wstride, dpb, tl);
}

// Clear the block's remaining-mass lock and store its poll limit (every
// thread of the block calls this).  P.lock_preheld starts the block with the
// lock taken, as if a warp held it and never released it.
__device__ __forceinline__ void init_block_lock(unsigned char *tl, const SisoParams &P) {
  if (threadIdx.x == 0) {
    int *lock = reinterpret_cast<int *>(tl);
    lock[0] = P.lock_preheld ? 1 : 0;
    lock[1] = P.lock_polls;
  }
  __syncthreads();
}

// ---------------------------------------------------------------------------
// MODE: where the query loop takes its patterns and whether the threshold rule
// applies; kernels of their own, so that the code and register allocation of
// each are not shaped by the others'.
template <int NPL, class SYN, int MINB, int MODE>
__global__ void __launch_bounds__(TPB, resident_blocks(MINB)) k_decode(const __grid_constant__ DevCode code,
                                                      const __grid_constant__ SisoParams P,
                                                      const __grid_constant__ DecodeArgs a) {
  extern __shared__ __align__(16) unsigned char smem[];
  using LY = Layout<NPL, SYN>;
  constexpr int NM = (32 * NPL + 63) / 64;
  const int warp = warp_index(), lane = threadIdx.x & 31;
  unsigned char *tl = block_tail(smem, LY::warp_bytes);
  init_block_lock(tl, P);
  Scratch<NPL, SYN> sc;
  bind_scratch(sc, smem, warp, LY::warp_bytes, tl + TAIL_BYTES, tl);
  const int n = code.n;
  const int64_t nwarps = (int64_t)gridDim.x * WARPS_PER_BLOCK;
  for (int64_t w = (int64_t)blockIdx.x * WARPS_PER_BLOCK + warp; w < a.n_words; w += nwarps) {
    const size_t base = (size_t)w * n;
    float lam[NPL];
#pragma unroll
    for (int k = 0; k < NPL; k++) {
      const int i = lane + 32 * k;
      float x = 0.f;
      if (i < n) {
        x = __ldg(a.llr_ch + base + i);
        if (a.llr_a) x = __fadd_rn(x, __ldg(a.llr_a + base + i));
      }
      lam[k] = x;
    }
    WordResult res;
    siso_word<NPL, SYN, MODE, true>(code, P, sc, lam, lane, res, [] {}, [&](int k, float x, float lapp, bool listed) {
      const int i = lane + 32 * k;
      if (i < n) {
        if (a.llr_app) a.llr_app[base + i] = lapp;
        if (a.llr_ext) a.llr_ext[base + i] = listed ? __fsub_rn(lapp, x) : 0.f;
        if (a.hard) a.hard[base + i] = lapp < 0.f ? 1 : 0;
      }
    });
    if (lane == 0) {
      if (a.p_miss) a.p_miss[w] = res.pmiss;
      if (a.queries) a.queries[w] = res.queries;
      if (a.list_count) a.list_count[w] = res.nhit;
      if ((res.flags & 1) && a.xf_count) atomicAdd(a.xf_count, 1);
      if (a.wsum) atomicAdd(a.wsum, (unsigned long long)res.wsum);
    }
    if (a.list_words || a.list_app) {
      const int l = lane;
      if (l < P.L) {  // L <= 16
        if (a.list_words)
#pragma unroll
          for (int wd = 0; wd < NM; wd++)
            a.list_words[((size_t)w * P.L + l) * NM + wd] = l < res.nhit ? sc.cw()[l * NM + wd] : 0ull;
        if (a.list_app) a.list_app[(size_t)w * P.L + l] = l < res.nhit ? sc.wl()[l] : 0.f;
      }
    }
    __syncwarp();
  }
}

template <int NPL, class SYN>
__global__ void k_trace(const DevCode code, const float *lam_in, int max_q, uint64_t *out, int32_t *count,
                        int32_t *c_out) {
  extern __shared__ __align__(16) unsigned char smem[];
  using LY = Layout<NPL, SYN>;
  const int lane = threadIdx.x & 31;
  unsigned char *tl = block_tail(smem, LY::warp_bytes);
  init_block_lock(tl, SisoParams{1, 1, 0.f});
  Scratch<NPL, SYN> sc;
  bind_scratch(sc, smem, 0, LY::warp_bytes, tl + TAIL_BYTES, tl);
  float lam[NPL];
#pragma unroll
  for (int k = 0; k < NPL; k++) {
    const int i = lane + 32 * k;
    lam[k] = i < code.n ? lam_in[i] : 0.f;
  }
  const int q = trace_word<NPL, SYN>(code, sc, lam, lane, max_q, out, c_out);
  if (lane == 0) *count = q;
}

// ---------------------------------------------------------------------------
// product codes
// ---------------------------------------------------------------------------
enum : int32_t { F_RUN = 0, F_DECODED = 1, F_MAXIT = 2, F_BAD_PENDING = 3, F_BAD = 4 };

// Loads that must see writes made by other SMs during the same kernel (the
// persistent form) bypass L1.
template <bool COHERENT>
__device__ __forceinline__ float ld_state(const float *p) {
  if constexpr (COHERENT) return __ldcg(p);
  return *p;
}
template <bool COHERENT>
__device__ __forceinline__ uint64_t ld_state(const uint64_t *p) {
  if constexpr (COHERENT) return __ldcg(reinterpret_cast<const unsigned long long *>(p));
  return *p;
}

// Per-warp tallies live in the warp's shared slot (not in registers, which
// the search needs) and reach the global counters once, when the warp exits.
__device__ __forceinline__ void tally_clear(unsigned long long *slot, int lane) {
  if (lane == 0) slot[0] = slot[1] = 0ull;
  __syncwarp();
}
__device__ __forceinline__ void tally_flush(const unsigned long long *slot, unsigned long long *wsum, int32_t *xf_count,
                                            int lane) {
  __syncwarp();
  if (lane != 0) return;
  if (wsum && slot[0]) atomicAdd(wsum, slot[0]);
  if (xf_count && slot[1]) atomicAdd(xf_count, (int32_t)slot[1]);
}

// A word's context (frame, word, kind of half, list index) is kept at the
// start of the frame-check area sc.W(), which nothing else uses during a word
// (the word's lambda follows it), and read back after the search: the
// registers that held it are free while the search runs.
struct WordCtx {
  int32_t f, li, wd, rows;
  // persistent form: the queries and the largest query count of the words
  // decoded since the frame's counters were last brought up to date
  int32_t qmax, words;
  int64_t queries;
};
static_assert(sizeof(WordCtx) <= 32, "the word's lambda follows the context in the frame-check area");

// Offset of bit i of word wd in its frame of rows of nr bits: a row, a column
// or (diag) a wrapped diagonal.
__device__ __forceinline__ int bit_offset(int i, int wd, int nr, bool rows, bool diag) {
  int r = rows ? wd : i;
  if (diag && !rows) {
    r = wd + i;
    if (r >= nr) r -= nr;
  }
  return r * nr + ((rows || diag) ? i : wd);
}

// One component word of frame f (a row, or a column or diagonal): lambda =
// L_Ch + fl32(alpha L_E) (L_A = 0 in the first half), SOGRAND, then L_E and
// the hard decision of L_APP are stored and the query counters updated.
// `code` is the code of this half's words (the row code in a row half, the
// column code in a column half).  GEN: the frame is a.nc rows of a.nr bits
// and the second set of words may be wrapped diagonals (a.diag); otherwise
// it is a square code.n x code.n frame with columns as the second set.
// Returns the word's query count (-1: non-finite input).
template <int NPL, class SYN, bool COHERENT, bool GEN, int MODE>
__device__ __forceinline__ int product_word(const DevCode &code, const SisoParams &P, const ProductArgs &a,
                                            const Scratch<NPL, SYN> &sc, int f, int li, int wd, bool rows, bool first,
                                            int lane) {
  constexpr int NM = (32 * NPL + 63) / 64;
#ifdef SG_PHASE_PROFILE
  const long long t0 = clock64();
#endif
  const int n = code.n, nr = GEN ? a.nr : n, fsz = nr * (GEN ? a.nc : n);
  const bool diag = GEN && a.diag;
  // the word's bits lie `step` positions apart for every 32 (a wrapped diagonal's do not)
  const auto position = [&](int k, int w, bool r) {
    if (diag) return bit_offset(lane + 32 * k, w, nr, r, diag);
    return (r ? w * nr + lane : lane * nr + w) + k * (r ? 32 : 32 * nr);
  };
  float lam[NPL];
  {
    const size_t fb = (size_t)f * fsz;
    const float *ch = a.llr_ch + fb, *le = a.le + fb;
    float ext[NPL];
#pragma unroll
    for (int k = 0; k < NPL; k++) {
      const int i = lane + 32 * k;
      lam[k] = ext[k] = 0.f;
      if (i < n) {
        const int pos = position(k, wd, rows);
        lam[k] = __ldg(ch + pos);
        if (!first) ext[k] = ld_state<COHERENT>(le + pos);
      }
    }
    if (!first)  // L_A = alpha L_E
#pragma unroll
      for (int k = 0; k < NPL; k++) lam[k] = __fadd_rn(lam[k], __fmul_rn(a.alpha, ext[k]));
  }
  WordResult res;
  if (lane == 0) *reinterpret_cast<int4 *>(sc.W()) = make_int4(f, li, wd, rows);
  __syncwarp();
  const volatile WordCtx *vc = reinterpret_cast<const volatile WordCtx *>(sc.W());
  // where the word's L_E and hard decision go, set once the search has ended
  float *le = nullptr;
  unsigned *hb = nullptr;
  size_t at = 0;
  siso_word<NPL, SYN, MODE, false>(
      code, P, sc, lam, lane, res,
      [&]() {
        f = vc->f;
        wd = vc->wd;
        rows = vc->rows != 0;
        le = a.le + (size_t)f * fsz;
        at = (size_t)f * (GEN ? a.hbw : n) + wd;
        hb = reinterpret_cast<unsigned *>(a.hb + at * NM);
      },
      [&](int k, float x, float lapp, bool listed) {
        const bool in = lane + 32 * k < n;
        if (in) le[position(k, wd, rows)] = listed ? __fsub_rn(lapp, x) : 0.f;
        const unsigned h = __ballot_sync(FULL, in && lapp < 0.f);
        if (lane == 0) hb[k] = h;
      });
  if (lane == 0) {
    if (NPL & 1) hb[NPL] = 0u;  // the upper half of the last u64
    if (a.wq) a.wq[at] = res.queries;
    if (res.queries >= 0) {
      if constexpr (COHERENT) {
        WordCtx *c = reinterpret_cast<WordCtx *>(sc.W());
        c->queries += res.queries;
        c->qmax = max(c->qmax, res.queries);
      } else {
        atomicAdd(reinterpret_cast<unsigned long long *>(a.queries + f), (unsigned long long)res.queries);
        atomicMax(a.hmax + f, res.queries);
      }
      sc.tally()[0] += (unsigned long long)res.wsum;
    }
    if (res.flags) {
      sc.tally()[1] += res.flags & 1;
      if ((res.flags & 2) && a.ctrl) atomicExch(a.ctrl + CTRL_ERROR, 2);  // stops a persistent launch: reported as a timeout
    }
  }
  __syncwarp();
#ifdef SG_PHASE_PROFILE
  if (lane == 0) {
    SG_PROF(10, clock64() - t0);
    SG_PROF(11, 1);
  }
#endif
  return res.queries;
}

// Hard decision of frame f after a half: W holds its words (rows after an
// odd half, columns after an even one): xc.n words of wc.n bits, wc the code
// of these words and xc the code across them.  Every word is a codeword of wc
// iff parity(word & H_wc row t) = 0 for all t; every word of the other
// orientation is a codeword of xc iff, for every t, the XOR of the words
// selected by H_xc row t is zero (bit-sliced, no transpose).  Warp-uniform.
//
// The frame check and frame_finish run once per frame and half, after the
// half's last word, on a warp whose SM is busy with words: they are kept short
// (rolled loops, no per-bit divisions) because their code evicts the words'
// from the instruction cache.
template <int NPL>
__device__ __forceinline__ bool frame_valid(const DevCode &wc, const DevCode &xc, const uint64_t *W, int lane) {
  constexpr int NM = (32 * NPL + 63) / 64, W32 = 2 * NM;  // 32-bit words of a word, as stored (NPL of them used)
  const int nw = xc.n;  // words in W
  const unsigned *Ws = reinterpret_cast<const unsigned *>(W);
  unsigned own[NPL][NPL];  // [k]: this lane's words lane + 32 k
  uint64_t hx[NPL];        // their columns in the code across
#pragma unroll
  for (int k = 0; k < NPL; k++) {
    const int wd = lane + 32 * k;
    hx[k] = wd < nw ? __ldg(xc.hcol + wd) : 0ull;
#pragma unroll
    for (int j = 0; j < NPL; j++) own[k][j] = wd < nw ? Ws[wd * W32 + j] : 0u;
  }
  const unsigned *hrow = reinterpret_cast<const unsigned *>(wc.hrow);
  unsigned bad = 0;
#pragma unroll 1
  for (int t0 = 0; t0 < wc.m; t0 += 32) {
    unsigned row[NPL];  // lane t holds check t0 + t
#pragma unroll
    for (int j = 0; j < NPL; j++) row[j] = t0 + lane < wc.m ? __ldg(hrow + (t0 + lane) * W32 + j) : 0u;
#pragma unroll 1
    for (int t = 0; t < 32 && t0 + t < wc.m; t++) {
      unsigned acc[NPL] = {};
#pragma unroll
      for (int j = 0; j < NPL; j++) {
        const unsigned r = __shfl_sync(FULL, row[j], t);
#pragma unroll
        for (int k = 0; k < NPL; k++) acc[k] ^= own[k][j] & r;
      }
#pragma unroll
      for (int k = 0; k < NPL; k++) bad |= __popc(acc[k]) & 1;
    }
  }
  bool ok = !__any_sync(FULL, bad);
#pragma unroll 1
  for (int t = 0; t < xc.m && ok; t++) {
    unsigned acc[NPL] = {};
#pragma unroll
    for (int k = 0; k < NPL; k++)
      if ((hx[k] >> t) & 1ull)
#pragma unroll
        for (int j = 0; j < NPL; j++) acc[j] ^= own[k][j];
    unsigned any = 0;
#pragma unroll
    for (int j = 0; j < NPL; j++) any |= __reduce_xor_sync(FULL, acc[j]);
    ok = any == 0;
  }
  return ok;
}

// QC-GLDPC frame check: W holds the n words of the last half (rows, or the
// wrapped diagonals after a diagonal half).  Each must be a codeword, and so
// must each word of the other set, whose syndrome is gathered bit by bit:
// after a row half diagonal x has bit j = bit j of row (x + j) mod n; after a
// diagonal half row x has bit j = bit j of diagonal (x - j) mod n.
template <int NPL>
__device__ __forceinline__ bool frame_valid_diag(const DevCode &code, const uint64_t *W, bool rows, int lane) {
  constexpr int NM = (32 * NPL + 63) / 64;
  const int n = code.n;
  bool ok = true;
#pragma unroll 1
  for (int x0 = 0; x0 < n; x0 += 32) {
    const int x = min(x0 + lane, n - 1);
    uint64_t own = 0, other = 0;  // syndromes of word x and of word x of the other set
    int w = x;                    // (x + j) mod n after rows, (x - j) mod n after diagonals
#pragma unroll 1
    for (int j = 0; j < n; j++) {
      const uint64_t h = __ldg(code.hcol + j);
      if ((W[x * NM + (j >> 6)] >> (j & 63)) & 1ull) own ^= h;
      if ((W[w * NM + (j >> 6)] >> (j & 63)) & 1ull) other ^= h;
      w += rows ? 1 : n - 1;
      if (w >= n) w -= n;
    }
    ok = ok && (own | other) == 0;
  }
  return __all_sync(FULL, ok);
}

// Write the frame's decision as row-major bits and its status.  W holds the
// words of the last half: rows (bit j of word i is bit (i, j)), columns
// (bit i of word j is bit (i, j)) or, for a QC-GLDPC, wrapped diagonals (bit j
// of word (i - j) mod n is bit (i, j)).
// Columns are turned into rows first (a ballot collects one row of 32
// columns), so a byte of the output is a shift of its row when rows start on
// byte boundaries.
template <int NPL>
__device__ __forceinline__ void frame_finish(const ProductArgs &a, int64_t f, bool rows, int half, int status,
                                             uint64_t *W, int lane) {
  constexpr int NM = (32 * NPL + 63) / 64, W32 = 2 * NM;
  const int nr = a.nr, nc = a.nc, nbits = nr * nc;
  const int nbytes = (nbits + 7) / 8;
  uint8_t *out = a.bits + (size_t)f * nbytes;
  unsigned *Ws = reinterpret_cast<unsigned *>(W);
  const bool diag = !rows && a.diag;
  if (!rows && !diag) {
    unsigned own[NPL][NPL];  // [k]: columns lane + 32 k
#pragma unroll
    for (int k = 0; k < NPL; k++)
#pragma unroll
      for (int j = 0; j < NPL; j++) own[k][j] = lane + 32 * k < nr ? Ws[(lane + 32 * k) * W32 + j] : 0u;
    __syncwarp();
#pragma unroll
    for (int j = 0; j < NPL; j++) {
#pragma unroll 1
      for (int i = 32 * j; i < 32 * j + 32 && i < nc; i++) {
#pragma unroll
        for (int k = 0; k < NPL; k++) {
          const unsigned row = __ballot_sync(FULL, own[k][j] & 1u);
          own[k][j] >>= 1;
          if (lane == k) Ws[i * W32 + k] = row;
        }
      }
    }
    __syncwarp();
  }
  const bool aligned = (nr & 7) == 0 && !diag;
#pragma unroll 1
  for (int b0 = 0; b0 < nbytes; b0 += 32) {
    const int by = min(b0 + lane, nbytes - 1);
    int i = by * 8 / nr, j = by * 8 - i * nr;
    unsigned v = 0;
    if (aligned) {
      v = Ws[i * W32 + (j >> 5)] >> (j & 31);
    } else {
#pragma unroll 1
      for (int t = 0; t < 8; t++) {
        if (i < nc) {
          int w = i;
          if (diag) {
            w = i - j;
            if (w < 0) w += nr;
          }
          v |= ((Ws[w * W32 + (j >> 5)] >> (j & 31)) & 1u) << t;
        }
        if (++j == nr) {
          j = 0;
          i++;
        }
      }
    }
    if (b0 + lane < nbytes) out[by] = (uint8_t)v;
  }
  if (lane == 0) {
    a.half_iters[f] = half;
    a.status[f] = (uint8_t)status;
  }
  __syncwarp();
}

// ---- plain form: one launch per half iteration, then a check launch ----
template <int NPL, class SYN, int MINB, bool GEN, int MODE>
__global__ void __launch_bounds__(TPB, resident_blocks(MINB))
    k_product_half(const __grid_constant__ DevCode rowc, const __grid_constant__ DevCode colc,
                   const __grid_constant__ SisoParams P, const __grid_constant__ ProductArgs a, int half) {
  extern __shared__ __align__(16) unsigned char smem[];
  using LY = Layout<NPL, SYN>;
  const int warp = warp_index(), lane = threadIdx.x & 31;
  unsigned char *tl = block_tail(smem, LY::warp_bytes);
  init_block_lock(tl, P);
  Scratch<NPL, SYN> sc;
  bind_scratch(sc, smem, warp, LY::warp_bytes, tl + TAIL_BYTES, tl);
  const bool rows = (half & 1) != 0;
  const DevCode &code = GEN && !rows ? colc : rowc;  // the code of this half's words
  const int n = rows ? a.nc : a.nr;                  // words per frame in this half
  const int64_t items = a.n_frames * n;
  const int64_t nwarps = (int64_t)gridDim.x * WARPS_PER_BLOCK;
  tally_clear(sc.tally(), lane);
  for (int64_t it = (int64_t)blockIdx.x * WARPS_PER_BLOCK + warp; it < items; it += nwarps) {
    const int64_t f = it / n;
    int wd = (int)(it - f * n);
    const int32_t fs = __ldg(a.fstate + f);
    if (fs != F_RUN && fs != F_BAD_PENDING) continue;  // finished frames only: a flag raised during
                                                        // this half must not change which words run
    const int q = product_word<NPL, SYN, false, GEN, MODE>(code, P, a, sc, (int)f, 0, wd, rows, half == 1, lane);
    if (lane == 0 && q < 0) atomicExch(a.fstate + f, (int32_t)F_BAD_PENDING);
  }
  tally_flush(sc.tally(), a.wsum, a.xf_count, lane);
}

// One warp per frame.
template <int NPL, class SYN>
__global__ void __launch_bounds__(TPB) k_product_check(const DevCode rowc, const DevCode colc, const ProductArgs a,
                                                       int half) {
  constexpr int NM = (32 * NPL + 63) / 64;
  constexpr int NT = 32 * NPL;
  __shared__ uint64_t words_s[WARPS_PER_BLOCK][NT * NM];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int64_t nwarps = (int64_t)gridDim.x * WARPS_PER_BLOCK;
  const bool rows = (half & 1) != 0;
  const DevCode &wc = rows ? rowc : colc, &xc = rows ? colc : rowc;
  const int n = xc.n;  // words of the last half
  for (int64_t f = (int64_t)blockIdx.x * WARPS_PER_BLOCK + warp; f < a.n_frames; f += nwarps) {
    const int32_t st = a.fstate[f];
    if (st != F_RUN && st != F_BAD_PENDING) continue;
    uint64_t *W = words_s[warp];
    for (int x = lane; x < n * NM; x += 32) W[x] = a.hb[(size_t)f * a.hbw * NM + x];
    __syncwarp();
    const bool ok = a.diag ? frame_valid_diag<NPL>(wc, W, rows, lane) : frame_valid<NPL>(wc, xc, W, lane);
    const bool bad = st == F_BAD_PENDING;
    const bool finish = bad || ok || half >= a.max_half;
    if (lane == 0) {
      a.par_queries[f] += a.hmax[f];
      a.hmax[f] = 0;
    }
    if (!finish) {
      if (lane == 0 && a.active) atomicAdd(a.active, 1);
      __syncwarp();
      continue;
    }
    frame_finish<NPL>(a, f, rows, half, bad ? 2 : (ok ? 0 : 1), W, lane);
    if (lane == 0) a.fstate[f] = bad ? F_BAD : (ok ? F_DECODED : F_MAXIT);
    __syncwarp();
  }
}

// ---- persistent forms: one launch decodes the whole batch ----

// Lane 0 of a warp publishes and observes the list with release/acquire
// operations at GPU scope; __syncwarp orders the other lanes' accesses before
// (release) or after (acquire) lane 0's, so no lane runs a full fence.
__device__ __forceinline__ int32_t ld_acquire_gpu(const int32_t *p) {
  int32_t v;
  asm volatile("ld.acquire.gpu.global.b32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return v;
}
__device__ __forceinline__ void st_release_gpu(int32_t *p, int32_t v) {
  asm volatile("st.release.gpu.global.b32 [%0], %1;" ::"l"(p), "r"(v) : "memory");
}
__device__ __forceinline__ int32_t atom_add_acq_rel_gpu(int32_t *p, int32_t x) {
  int32_t old;
  asm volatile("atom.acq_rel.gpu.global.add.s32 %0, [%1], %2;" : "=r"(old) : "l"(p), "r"(x) : "memory");
  return old;
}

// A filled slot of the frame-half list holds +v for an odd half and -v for an
// even one, v = 2 (list entry + 1) + 1 for a frame's first half and
// 2 (list entry + 1) for a later one.  The slot itself says which kind of half
// it is, so a ticket that the half skips (codes of different lengths) is
// recognised even after the frame has moved on, and a word needs no look at
// its frame's counters before it starts.
__device__ __forceinline__ int32_t slot_value(int li, int half) {
  const int v = 2 * (li + 1) + (half == 1);
  return (half & 1) ? v : -v;
}

// Wait until slot `slot` of the frame-half list is filled.  Returns its signed
// value, or 0 when the list is done (every frame finished or parked) or the
// launch's error word is set.  The wait backs off exponentially and gives up
// after max_spin microseconds of sleep for every word that a warp draws at
// once (what it waits for may be all the words of another warp's run, decoded
// one after the other), setting the error word.  All reads of
// shared state are made by lane 0 and broadcast, so the whole warp takes the
// same branch.
__device__ __forceinline__ int sched_wait(const ProductArgs &a, int slot, int lane, int *waited) {
  const bool real = slot < a.n_frames * a.max_half;  // a frame has at most max_half halves
  int v = 0;
  long long slept = 0;  // nanoseconds
  unsigned nap = 64;
  for (;;) {
    int stop = 0;
    if (lane == 0) {
      if (real) v = ld_acquire_gpu(a.queue + slot);
      // an error, or every frame finished and this ticket has no work
      const volatile int32_t *ctrl = a.ctrl;
      if (ctrl[CTRL_ERROR] != 0)
        stop = 1;
      else if (v == 0)
        stop = ctrl[CTRL_DONE] >= a.n_frames;
    }
    stop = __shfl_sync(FULL, stop, 0);
    v = __shfl_sync(FULL, v, 0);
    if (stop) return 0;
    if (v != 0) break;
    *waited = 1;
    if (slept > (long long)a.max_spin * 1000 * a.run) {
      if (lane == 0) atomicExch(a.ctrl + CTRL_ERROR, 1);
      return 0;
    }
    __nanosleep(nap);
    slept += nap;
    if (nap < 8192) nap <<= 1;
  }
  __syncwarp();  // after lane 0's acquire: the warp reads the frame's state for this half
  return v;
}

// After the last word of a half of frame f (list entry li): check the frame
// and finish it, park it (a serving epoch ran out: its state stays for the
// next launch) or append its next half.  `words` is the shared address of the
// warp's frame-check area.
template <int NPL, bool GEN>
__device__ __forceinline__ void frame_after_half(const DevCode &wc, const DevCode &xc, const ProductArgs &a, int f, int li,
                                              unsigned words, int lane) {
  constexpr int NM = (32 * NPL + 63) / 64;
  uint64_t *W = sptr<uint64_t>(words);
  const int n = xc.n;  // words of this half
  __syncwarp();  // after lane 0's acquire of the frame's word count: the other words' results
  const uint64_t *hb = a.hb + (size_t)f * (GEN ? a.hbw : n) * NM;
#pragma unroll 1
  for (int x0 = 0; x0 < n * NM; x0 += 32)
    if (x0 + lane < n * NM) W[x0 + lane] = ld_state<true>(hb + x0 + lane);
  const int half = __ldcg(a.half_cur + f), bad = __ldcg(a.bad + f);
  const int stop = a.half_stop ? __ldcg(a.half_stop + f) : a.max_half;
  __syncwarp();
  const bool rows = (half & 1) != 0;
  const bool ok = (GEN && a.diag) ? frame_valid_diag<NPL>(wc, W, rows, lane) : frame_valid<NPL>(wc, xc, W, lane);
  if (lane == 0) {
    a.par_queries[f] += __ldcg(a.hmax + f);
    a.hmax[f] = 0;
  }
  if (bad || ok || half >= a.max_half) {
    frame_finish<NPL>(a, f, rows, half, bad ? 2 : (ok ? 0 : 1), W, lane);
    if (lane == 0) atomicAdd(a.ctrl + CTRL_DONE, 1);
  } else if (lane == 0) {
    a.half_cur[f] = half + 1;
    a.done_words[f] = 0;
    if (half >= stop) {  // parked: resumes at half + 1 in a later launch
      atomicAdd(a.ctrl + CTRL_DONE, 1);
    } else {
      const int t = atomicAdd(a.ctrl + CTRL_SLOTS, 1);  // < nslots: every frame appends at most max_half - 1 times
      st_release_gpu(a.queue + t, slot_value(li, half + 1));
    }
  }
  __syncwarp();
}

// Frame-halves are appended to a list (a.queue, see slot_value); the first F
// slots hold every frame's current half.  Warps draw runs of global word
// tickets T (a.run of them, one once the warp has had to wait): slot T / slot_n,
// word T mod slot_n.  The warp that completes a frame's last word of a half runs
// the frame check and either finishes the frame or appends it for its next half.
// A warp whose slot is not filled yet waits with exponential back-off (the
// tickets of its run then lie in slots that are not reserved yet or about to be
// stored, so it holds back no word that another warp waits for); all waits are
// bounded (a.max_spin * a.run microseconds of accumulated sleep without progress):
// the kernel then records an error and every warp returns.  GEN: two codes or
// wrapped diagonals (the code of a word is chosen per half); otherwise a
// square product code whose words all use rowc, with no selection of a code
// and its geometry in every word.
template <int NPL, class SYN, int MINB, bool GEN, int MODE>
__global__ void __launch_bounds__(TPB, resident_blocks(MINB))
    k_product_persistent(const __grid_constant__ DevCode rowc, const __grid_constant__ DevCode colc,
                         const __grid_constant__ SisoParams P, const __grid_constant__ ProductArgs a) {
  extern __shared__ __align__(16) unsigned char smem[];
  using LY = Layout<NPL, SYN>;
  const int warp = warp_index(), lane = threadIdx.x & 31;
  unsigned char *tl = block_tail(smem, LY::warp_bytes);
  init_block_lock(tl, P);
  Scratch<NPL, SYN> sc;
  bind_scratch(sc, smem, warp, LY::warp_bytes, block_dp_area(smem, LY::warp_bytes, a.dp_area, a.dp_stride), tl);
  const int slot_n = GEN ? max(a.nr, a.nc) : rowc.n;  // tickets per list slot: the most words in a half
  tally_clear(sc.tally(), lane);
  if (lane == 0) atomicAdd(a.ctrl + CTRL_WARPS, 1);  // one more active warp
  int waited = 0;
  int ticket = 0, left = 0;  // the next ticket and how many more of its run are this warp's
  int slot = -1, v = 0;      // the slot last waited for and its value
  WordCtx *ctx = reinterpret_cast<WordCtx *>(sc.W());
  for (;;) {
    if (left == 0) {
      // Drain: a warp leaves once the unfinished frames cannot use it (each has
      // at most slot_n words in flight), so the SMs go to other work sharing
      // the GPU (the parallel kernels of the mixed form); the warps that stay
      // can always take every word that becomes available.  Decided before a
      // ticket is drawn (a drawn ticket is always decoded), and only once the
      // warp has had to wait for work: while the list runs ahead of the
      // tickets the check is skipped.
      int leave = 0;
      if (waited && lane == 0) {
        const int64_t need = (a.n_frames - (int64_t)__ldcg(a.ctrl + CTRL_DONE)) * slot_n;
        if ((int64_t)__ldcg(a.ctrl + CTRL_WARPS) - 1 >= need) {
          if ((int64_t)atomicSub(a.ctrl + CTRL_WARPS, 1) - 1 >= need)
            leave = 1;
          else
            atomicAdd(a.ctrl + CTRL_WARPS, 1);
        }
      }
      if (__shfl_sync(FULL, leave, 0)) {
        // this block has begun to leave: a decoder launched as a programmatic
        // dependent of this one may start (no effect otherwise)
        asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
        break;
      }
      left = waited ? 1 : a.run;
      if (lane == 0) ticket = atomicAdd(a.ctrl + CTRL_TICKETS, left);
      ticket = __shfl_sync(FULL, ticket, 0);
    }
    const int at = ticket / slot_n, w = ticket - at * slot_n;
    ticket++;
    left--;
    if (at != slot) {
      slot = at;
      v = sched_wait(a, slot, lane, &waited);
      if (v == 0) break;
      if (lane == 0) {
        ctx->qmax = ctx->words = 0;
        ctx->queries = 0;
      }
      __syncwarp();
    }
    const bool rows = v > 0;  // the slot's half is odd: a row half
    const DevCode &code = GEN ? (rows ? rowc : colc) : rowc, &xcode = GEN ? (rows ? colc : rowc) : rowc;
    const int n = xcode.n;  // words in this half
    // (a ticket past this half's words, of codes of different lengths, has no
    // word; decided from the slot, since the frame may already be in its next half)
    if (!GEN || w < n) {
      const int li = ((rows ? v : -v) >> 1) - 1;  // list index
      const int f = a.frame_list ? a.frame_list[li] : li;
      const int q = product_word<NPL, SYN, true, GEN, MODE>(code, P, a, sc, f, li, w, rows, rows && (v & 1), lane);
      if (lane == 0) {
        ctx->words++;
        if (q < 0) atomicExch(a.bad + ctx->f, 1);
      }
      __syncwarp();  // every lane's L_E and hard decision, then lane 0 releases them
      // the frame's counters once for the words of it that were drawn together
      if (left == 0 || w == n - 1) {
        int last = 0;
        if (lane == 0) {
          const int fr = ctx->f, words = ctx->words;
          atomicAdd(reinterpret_cast<unsigned long long *>(a.queries + fr), (unsigned long long)ctx->queries);
          atomicMax(a.hmax + fr, ctx->qmax);
          last = atom_add_acq_rel_gpu(a.done_words + fr, words) + words == n;  // acquire: the frame's other words
          ctx->qmax = ctx->words = 0;
          ctx->queries = 0;
        }
        if (__shfl_sync(FULL, last, 0)) {
          const volatile WordCtx *vc = ctx;
          const int fr = vc->f, fl = vc->li;
          frame_after_half<NPL, GEN>(code, xcode, a, fr, fl, sc.base + LY::o_w, lane);
          slot = -1;  // the frame check has used the words' context
        }
      }
    }
  }
  tally_flush(sc.tally(), a.wsum, a.xf_count, lane);
}

// list and counters of the persistent form: every frame queued for half 1
static __global__ void k_persistent_init(const ProductArgs a) {
  const int64_t F = a.n_frames;
  const int64_t slots = F * (int64_t)a.max_half;
  int32_t *queue = a.queue;
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < slots; i += (int64_t)gridDim.x * blockDim.x) {
    if (i >= F) queue[i] = 0;
    if (i < F) {
      int64_t f = i;
      bool fresh = true;
      if (a.frame_list) {
        const int32_t e = a.frame_list[i];
        fresh = e < 0;
        f = fresh ? -(int64_t)e - 1 : (int64_t)e;
        if (fresh) a.frame_list[i] = (int32_t)f;
      }
      if (fresh) {
        a.half_cur[f] = 1;
        a.bad[f] = 0;
        a.queries[f] = 0;
        a.par_queries[f] = 0;
        if (a.frame_list) a.status[f] = 255;  // in progress until the frame finishes
      }
      a.done_words[f] = 0;
      a.hmax[f] = 0;
      if (a.half_stop) a.half_stop[f] = a.half_cur[f] + a.epoch_halves - 1;
      queue[i] = slot_value((int)i, a.half_cur[f]);
    }
  }
  if (blockIdx.x == 0 && threadIdx.x == 0) {
    a.ctrl[CTRL_SLOTS] = (int32_t)F;  // next slot to reserve
    a.ctrl[CTRL_TICKETS] = 0;           // word tickets drawn
    a.ctrl[CTRL_DONE] = 0;           // frames finished
    a.ctrl[CTRL_ERROR] = 0;           // error
    a.ctrl[CTRL_WARPS] = 0;           // active warps
  }
}

// ---------------------------------------------------------------------------
// launchers
// ---------------------------------------------------------------------------
inline int sm_count() {
  static int sms = 0;
  if (!sms) {
    int dev = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (sms <= 0) sms = 1;
  }
  return sms;
}

template <class K>
inline int grid_for(K kernel, int smem, int64_t warps_needed) {
  int occ = 0;
  cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, kernel, TPB, smem);
  if (occ < 1) occ = 1;
  int64_t blocks = (warps_needed + WARPS_PER_BLOCK - 1) / WARPS_PER_BLOCK;
  int64_t cap = (int64_t)sm_count() * occ;
  if (blocks > cap) blocks = cap;
  if (blocks < 1) blocks = 1;
  return (int)blocks;
}

// The schedule a launch runs: the code's, except that schedule 12's kernels
// (56 registers) are used only when the launch has more words than the 8-block
// grid has warps; a smaller batch gains nothing from the extra warps and
// decodes each word faster at 64 registers.
inline int launch_minb(int minb, int64_t words) {
  return (minb == 12 && words > (int64_t)sm_count() * 8 * WARPS_PER_BLOCK) ? 12 : 8;
}

template <class K>
inline cudaError_t set_smem(K kernel, int smem) {
  if (smem > 48 * 1024) return cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
  return cudaSuccess;
}

template <int NPL, class SYN>
cudaError_t launch_decode(const DevCode &code, const SisoParams &P, const DecodeArgs &a, cudaStream_t s) {
  if (a.n_words <= 0) return cudaSuccess;
  const int smem = block_scratch_bytes<NPL, SYN>(code.jmax);
  const bool eight = launch_minb(code.minb, a.n_words) == 8, lanes = code.ord_lanes;
  auto kern = P.thr > 0.f ? (eight ? k_decode<NPL, SYN, 8, MODE_THR> : k_decode<NPL, SYN, 12, MODE_THR>)
              : lanes     ? (eight ? k_decode<NPL, SYN, 8, MODE_LANES> : k_decode<NPL, SYN, 12, MODE_LANES>)
                          : (eight ? k_decode<NPL, SYN, 8, MODE_TABLE> : k_decode<NPL, SYN, 12, MODE_TABLE>);
  cudaError_t e = set_smem(kern, smem);
  if (e != cudaSuccess) return e;
  const int grid = grid_for(kern, smem, a.n_words);
  kern<<<grid, TPB, smem, s>>>(code, P, a);
  return cudaGetLastError();
}

template <int NPL, class SYN>
cudaError_t launch_trace(const DevCode &code, const float *lam, int max_q, uint64_t *out, int32_t *count,
                         int32_t *c_out, cudaStream_t s) {
  const int smem = block_scratch_bytes<NPL, SYN>(code.jmax);
  auto kern = k_trace<NPL, SYN>;
  cudaError_t e = set_smem(kern, smem);
  if (e != cudaSuccess) return e;
  kern<<<1, 32, smem, s>>>(code, lam, max_q, out, count, c_out);
  return cudaGetLastError();
}

template <int NPL, class SYN, bool GEN>
cudaError_t launch_product_half(const DevCode &rowc, const DevCode &colc, const SisoParams &P, const ProductArgs &a,
                                int half, cudaStream_t s) {
  const int smem = block_scratch_bytes<NPL, SYN>(std::max(rowc.jmax, colc.jmax));
  const int64_t items = a.n_frames * ((half & 1) ? a.nc : a.nr);
  const int minb = launch_minb(rowc.minb, items);
  auto kern = P.thr > 0.f ? (minb == 8 ? k_product_half<NPL, SYN, 8, GEN, MODE_THR> : k_product_half<NPL, SYN, 12, GEN, MODE_THR>)
                          : (minb == 8 ? k_product_half<NPL, SYN, 8, GEN, MODE_TABLE> : k_product_half<NPL, SYN, 12, GEN, MODE_TABLE>);
  cudaError_t e = set_smem(kern, smem);
  if (e != cudaSuccess) return e;
  kern<<<grid_for(kern, smem, items), TPB, smem, s>>>(rowc, colc, P, a, half);
  return cudaGetLastError();
}

template <int NPL, class SYN>
cudaError_t launch_product_check(const DevCode &rowc, const DevCode &colc, const ProductArgs &a, int half,
                                 cudaStream_t s) {
  auto kern = k_product_check<NPL, SYN>;
  kern<<<grid_for(kern, 0, a.n_frames), TPB, 0, s>>>(rowc, colc, a, half);
  return cudaGetLastError();
}

template <int NPL, class SYN>
cudaError_t launch_product_init(const DevCode &code, const ProductArgs &a, cudaStream_t s) {
  (void)code;
  cudaError_t e = cudaMemsetAsync(a.fstate, 0, sizeof(int32_t) * a.n_frames, s);
  if (e == cudaSuccess) e = cudaMemsetAsync(a.hmax, 0, sizeof(int32_t) * a.n_frames, s);
  if (e == cudaSuccess && a.queries) e = cudaMemsetAsync(a.queries, 0, sizeof(int64_t) * a.n_frames, s);
  if (e == cudaSuccess && a.par_queries) e = cudaMemsetAsync(a.par_queries, 0, sizeof(int64_t) * a.n_frames, s);
  return e;
}

template <int NPL, class SYN, bool GEN>
cudaError_t launch_product_persistent(const DevCode &rowc, const DevCode &colc, const SisoParams &P,
                                      const ProductArgs &a_, cudaStream_t s, int part) {
  ProductArgs a = a_;
  if (a.n_frames <= 0) return cudaSuccess;
  cudaError_t e = cudaSuccess;
  if (part == PERSISTENT_ALL || part == PERSISTENT_INIT) {
    k_persistent_init<<<(int)std::min<int64_t>((a.n_frames + 255) / 256, 4096), 256, 0, s>>>(a);
    e = cudaGetLastError();
    if (e != cudaSuccess || part == PERSISTENT_INIT) return e;
  }
  // with a global remaining-mass region only the warps' areas are shared memory
  const int smem = a.dp_area ? WARPS_PER_BLOCK * Layout<NPL, SYN>::warp_bytes + TAIL_BYTES
                             : block_scratch_bytes<NPL, SYN>(std::max(rowc.jmax, colc.jmax));
  const int64_t words = a.n_frames * std::max(a.nr, a.nc);  // the most words of one half
  // the lanes-enumerated order: the square geometry only (GEN reads the table)
  const bool eight = launch_minb(rowc.minb, words) == 8, lanes = !GEN && rowc.ord_lanes;
  constexpr int ML = GEN ? MODE_TABLE : MODE_LANES;
  auto kern = P.thr > 0.f ? (eight ? k_product_persistent<NPL, SYN, 8, GEN, MODE_THR> : k_product_persistent<NPL, SYN, 12, GEN, MODE_THR>)
              : lanes     ? (eight ? k_product_persistent<NPL, SYN, 8, GEN, ML> : k_product_persistent<NPL, SYN, 12, GEN, ML>)
                          : (eight ? k_product_persistent<NPL, SYN, 8, GEN, MODE_TABLE> : k_product_persistent<NPL, SYN, 12, GEN, MODE_TABLE>);
  e = set_smem(kern, smem);
  if (e != cudaSuccess) return e;
  int occ = 0;
  cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, kern, TPB, smem);
  if (occ < 1) occ = 1;
  // every block resident at once, no more warps than words of the batch
  const int64_t want = (words + WARPS_PER_BLOCK - 1) / WARPS_PER_BLOCK;
  int64_t cap = (int64_t)sm_count() * occ;
  if (a.grid_cap > 0 && a.grid_cap < cap) cap = a.grid_cap;
  if (a.dp_area && a.dp_blocks < cap) cap = a.dp_blocks;  // one slice of the region per block
  const int grid = (int)std::max<int64_t>(1, std::min<int64_t>(cap, want));
  // Tickets drawn at once: up to 8 while every warp has at least 8 such runs
  // in the first half alone, else fewer, so that a small batch spreads over
  // all warps.  A run saves the draw, the look at the list and the release of
  // the finished words for all but one of its words: with one ticket a draw
  // the ticket counter's L2 line took three accesses a word and bound the
  // launch (eBCH(64,57)^2, 20,000 frames: 26.7 ms at runs of 1, 23.1 at 2,
  // 22.1 at 4, 21.6 at 8).
  const int64_t per_warp = words / ((int64_t)grid * WARPS_PER_BLOCK);
  a.run = per_warp >= 64 ? 8 : (per_warp >= 32 ? 4 : (per_warp >= 16 ? 2 : 1));
  if (part == PERSISTENT_DECODE_PDL) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(grid);
    cfg.blockDim = dim3(TPB);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kern, rowc, colc, P, a);
  }
  kern<<<grid, TPB, smem, s>>>(rowc, colc, P, a);
  return cudaGetLastError();
}

#define SG_INSTANTIATE(NPL, SYN)                                                                                 \
  template cudaError_t launch_decode<NPL, SYN>(const DevCode &, const SisoParams &, const DecodeArgs &,          \
                                               cudaStream_t);                                                    \
  template cudaError_t launch_trace<NPL, SYN>(const DevCode &, const float *, int, uint64_t *, int32_t *,        \
                                              int32_t *, cudaStream_t);                                          \
  template cudaError_t launch_product_half<NPL, SYN, false>(const DevCode &, const DevCode &, const SisoParams &, \
                                                            const ProductArgs &, int, cudaStream_t);             \
  template cudaError_t launch_product_check<NPL, SYN>(const DevCode &, const DevCode &, const ProductArgs &, int, \
                                                      cudaStream_t);                                             \
  template cudaError_t launch_product_init<NPL, SYN>(const DevCode &, const ProductArgs &, cudaStream_t);           \
  template cudaError_t launch_product_persistent<NPL, SYN, false>(const DevCode &, const DevCode &,              \
                                                                  const SisoParams &, const ProductArgs &,       \
                                                                  cudaStream_t, int);

// Launchers of the general geometry (two codes, or wrapped diagonals), in
// translation units of their own so that they compile in parallel.
#define SG_INSTANTIATE_GEN(NPL, SYN)                                                                             \
  template cudaError_t launch_product_half<NPL, SYN, true>(const DevCode &, const DevCode &, const SisoParams &,  \
                                                           const ProductArgs &, int, cudaStream_t);              \
  template cudaError_t launch_product_persistent<NPL, SYN, true>(const DevCode &, const DevCode &,               \
                                                                 const SisoParams &, const ProductArgs &,        \
                                                                 cudaStream_t, int);

}  // namespace sg

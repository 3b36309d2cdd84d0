// sg_common.h -- types shared by the host and device halves of libsogrand.
// Internal to the library; the public interface is include/sogrand.h.
#pragma once
#include <cuda_runtime.h>

#include <cstdint>

namespace sg {

constexpr int NMAX = 128;      // longest component code
constexpr int LMAX = 16;       // longest list a decode may request
constexpr int WMAXT = 64;      // most Hamming weights a query-order table may reach
constexpr int WENT = 15;       // most ranks one table entry holds
constexpr int WARPS_PER_BLOCK = 4;
// Schedules: the per-word kernels are compiled for 8 resident blocks per SM
// (64 registers a thread, schedule 8) and for 9 (56 registers, schedule 12); a
// launch never has more than MAX_BLOCKS_PER_SM blocks resident on an SM.
constexpr int MAX_BLOCKS_PER_SM = 9;

// Query order of one code, flattened per 1-line parameter c and parity class.
// For every c in [0, c_max] and class (the parity of y for an even code, or
// the single class of all patterns) the patterns are stored in query order:
// increasing cost = sum of ranks + c * weight, ties by weight, then by the
// ascending rank vector in lexicographic order.  Each order is stored up to
// the query cap it was built for and then to the end of that cost level.
struct DevOrder {
  const uint4 *ent;       // [total] byte 0: Hamming weight w; bytes 1..w: ranks (0-based, ascending)
  const uint16_t *cost;   // [total] cost of each pattern
  const int32_t *base;    // [(c_max+1) * ncls] first entry of order (c, class)
  const int32_t *count;   // [(c_max+1) * ncls] entries stored for (c, class)
  int32_t ncls;           // 2 for an even code (class = parity of y), else 1
  int32_t class_size;     // patterns in one class (saturated): count == class_size means the whole class
  // The head of every order again, a pattern as its prefix and its last ranks
  // (see siso_word's search): order (c, class) = ti owns e4[ti * e4_stride ...]
  // and slots[ti * (FAST_SLOTS2 + FAST_SLOTS) ...].
  // e4: one 32-bit entry a query, byte 0: prefix slot; bytes 1..3: the last
  // ranks (0-based; n where there is none).  Groups of four chunks, lane j's
  // four entries together (uint4 [group][lane]): one load serves four chunks,
  // and a warp alone on its SM, which waits out the L2 latency for every load,
  // waits once in 128 queries.
  const uint4 *e4;
  const uint2 *slots;     // byte 0: prefix length | ranks after it << 4; bytes 1..7: the prefix's ranks
  const int2 *zones;      // [ti] queries in two-rank form (slots 0..31) and, from there, in three-rank form up to .y (multiples of 128)
  int32_t e4_stride;      // in uint4
};

// Prefix slots of the two-rank and the three-rank form, and the longest prefix.
// In query order the first 32 prefixes reach about 1000 queries when the last
// two ranks are split off, and 64 about 9000 when the last three are (c = 0;
// further for c > 0, where heavy patterns come later).
constexpr int FAST_SLOTS2 = 32, FAST_SLOTS = 64, FAST_PREFIX = 7;
constexpr int FAST_QUERIES = 16384;  // most queries of an order kept in these forms

// The same orders as groups, for lanes that enumerate their patterns instead
// of reading DevOrder::ent (DevCode::ord_lanes): a group is the run of
// patterns of one cost and one Hamming weight w, i.e. the w-subsets of the
// ranks {1..n} with rank sum m = cost - c w, in lexicographic order.
struct DevGroups {
  const uint2 *grp;       // [groups] x: first entry of the group within its order; y: m | w << 16
  const int32_t *gbase;   // [(c_max+1) * ncls + 1] first group of order (c, class)
  const int32_t *scnt;    // [(n+1) * sc_w * sc_m] w-subsets of {1..N} with sum m at (N, w, m), saturated
  int32_t sc_w, sc_m;     // extents of scnt in w and m
};

struct DevCode {
  int32_t n, k, m;       // length, dimension, parity checks (m = n - k)
  int32_t even;          // 1: even code, search restricted to the parity of y
  int32_t c_max;         // clamp of the 1-line parameter
  float log_phi;         // log((2^k-1)/(2^(n-1)-1)) (even) or log((2^k-1)/(2^n-1))
  const uint64_t *hcol;  // [n] syndrome contribution of bit i (bit t = H[t][i])
  const uint64_t *hrow;  // [m][nm] rows of H as bit masks over the n positions
  DevOrder ord;
  int32_t jmax;          // largest stored cost + 2 (bounds the remaining-mass DP)
  int32_t minb;          // schedule: 8 or 12 (resident_blocks in kernels.cuh)
  int32_t dp_global;     // schedule: the batched forms keep the remaining-mass area in global memory
  int32_t ord_lanes;     // 1: the lanes enumerate the query order (loop without the threshold rule)
  DevGroups grp;         // the order's groups (used with ord_lanes)
};

struct SisoParams {
  int32_t L;
  int32_t cap;
  float thr;
  int32_t forney = 0;            // 1: Forney's list-only normalisation (the mass outside the list taken as 0)
  int32_t lock_polls = 1 << 22;  // polls of the block's remaining-mass lock before a warp gives up on it
  int32_t lock_preheld = 0;      // 1: blocks start with that lock taken (test of the bound)
};

// Per-word results that the callers write out.
struct WordResult {
  int32_t queries;       // -1: invalid input
  int32_t nhit;
  float pmiss;
  int32_t wsum;          // sum of the Hamming weights of the queried patterns
  int32_t flags;         // remaining mass: bit 0 extended range used, bit 1 its area could not be locked
};

}  // namespace sg

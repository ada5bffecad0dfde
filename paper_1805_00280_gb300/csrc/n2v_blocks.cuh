// The step through sampled blocks: membership in the longer list by a search of
// its samples and one 32-byte block.
//
// col is read in blocks of eight entries (32 bytes: one DRAM sector where col lies on
// 32 bytes, as an allocation does; on 16, which suffices, parts of two), and the
// auxiliary buffer keeps the first entry of every block, samples[i] = col[8 i]
// (built by n2v_graph_load; half a byte for each entry of col).  The block that
// can hold x is found among a row's samples, an eighth of the row, and whether it
// holds x takes eight compares.  So a step reads the shorter list, the samples
// beside its keys, and only those blocks of the longer list that a key falls
// into: neighbouring keys share a block when the lists are of like length, and
// when they are not most blocks are never read.
//
// Measured (GB300, R-MAT 24, p = 2, q = 0.5): staging the whole longer list read
// 55 KB of lists a step; the blocks move 28 KB of DRAM (5.65 TB/s) and run 262,144-walk
// launches in 56 ms against 132 ms.  Hashed sets of every row (one 32-byte bucket
// a key, an eighth of the instructions) were built and measured as well: DRAM gives
// 64 bytes for each random 32, 71 KB a step, and the same launches took 155 ms.
//
// A row starts and ends inside a block as a rule.  Entries of the neighbouring
// rows there are told apart by their index, in the row's first and last block
// only.
#pragma once

#include <algorithm>
#include <type_traits>

#include "n2v_step.cuh"

namespace n2v {

// A row as its blocks: block i holds the row's positions [8 i - head, 8 i + 8 - head).
struct BlockRow {
  const int32_t* __restrict__ smp;  // smp[i]: first entry of block i + 1, i < n1
  const int32_t* __restrict__ blk;  // block i at blk + 8 i
  const int32_t* __restrict__ top;  // every eighth sample: top[i], i < n2, the first entry of group i + 1
  int n1;    // samples inside the row (its blocks are 0 .. n1)
  int n2;    // of them, first of a group of eight blocks (64 entries, aligned in col)
  int up;    // group i starts at block 8 i - up
  int head;  // entries of block 0 before the row
  int len;
  int cut;                           // the block that reaches past the end of col, or -1
  const int32_t* __restrict__ tail;  // its copy
};

__device__ __forceinline__ BlockRow block_row(const GraphView& g, int64_t b, int d) {
  BlockRow r;
  const int64_t f = b >> 3;
  r.smp = g.samples + f + 1;
  r.blk = g.col + 8 * f;
  r.n1 = (int)(((b + d - 1) >> 3) - f);
  r.top = g.top + (f >> 3) + 1;
  r.n2 = (int)(((f + r.n1) >> 3) - (f >> 3));
  r.up = (int)(f & 7);
  r.head = (int)(b & 7);
  r.len = d;
  r.cut = f + r.n1 == g.cut_block ? r.n1 : -1;
  r.tail = g.tail;
  return r;
}

struct Block {
  int32_t s[8];
};

__device__ __forceinline__ Block block_at(const int32_t* p) {
  const int4 x = __ldg((const int4*)p), y = __ldg((const int4*)p + 1);
  return Block{{x.x, x.y, x.z, x.w, y.x, y.y, y.z, y.w}};
}
// Block i of the row (0 <= i <= n1).
__device__ __forceinline__ Block block_load(const BlockRow& r, int i) {
  return block_at(i == r.cut ? r.tail : r.blk + 8ll * i);
}

__device__ __forceinline__ bool block_has(const Block& b, int32_t x) {
  return b.s[0] == x || b.s[1] == x || b.s[2] == x || b.s[3] == x || b.s[4] == x || b.s[5] == x || b.s[6] == x ||
         b.s[7] == x;
}

// Position in the row of an x that block i holds as the row's own.
__device__ __forceinline__ int block_pos(const BlockRow& r, int i, const Block& b, int32_t x) {
  const unsigned at = (unsigned)(8 * i - r.head);
  unsigned p = 0;
#pragma unroll
  for (int j = 0; j < 8; ++j)
    if (b.s[j] == x && at + j < (unsigned)r.len) p = at + j;
  return (int)p;
}

// First position of the row whose entry is >= x, given the block of x (the number
// of samples <= x).
__device__ __forceinline__ int block_lower_bound(const BlockRow& r, int i, const int32_t* __restrict__ row, int32_t x) {
  const int lo = max(0, 8 * i - r.head), hi = min(r.len, 8 * i + 8 - r.head);
  return lo + lower_bound32(row + lo, hi - lo, x);
}

// The block of x, given its group i (the number of top samples <= x): eight samples in
// one load.
__device__ __forceinline__ int block_in_group(const BlockRow& r, int i, int32_t x) {
  const int i0 = 8 * i - r.up;  // the group's first block (before the row's, for i = 0)
  const Block s = block_at(r.smp + (i0 - 1));
  unsigned m = 0;
#pragma unroll
  for (int j = 1; j < 8; ++j) m |= s.s[j] <= x ? 1u << j : 0u;
  // blocks 1 .. n1 only: samples of other rows do not count
  if (i0 < 0) m &= 0xffffffffu << (1 - i0);
  if (i0 + 7 > r.n1) m &= (2u << (r.n1 - i0)) - 1u;
  return max(i0, 0) + __popc(m);
}

// Blocks of N keys of one lane: the number of samples in [from, n1) at or below
// each, plus from (N searches side by side).
template <int N>
__device__ __forceinline__ void block_search(const int32_t* __restrict__ smp, int n1, int from, const int32_t (&x)[N],
                                             int (&node)[N]) {
#pragma unroll
  for (int e = 0; e < N; ++e) node[e] = from;
  const int n = n1 - from;
  if (n <= 0) return;
  for (int st = 1 << (31 - __clz(n)); st > 0; st >>= 1) {
#pragma unroll
    for (int e = 0; e < N; ++e) {
      const int at = node[e] + st;
      if (at <= n1 && __ldg(smp + at - 1) <= x[e]) node[e] = at;
    }
  }
}

// Parameters of a job that the steps share.
struct StepArgs {
  uint32_t a_p, a_q;
  uint64_t inv_q;  // floor((2^64 - 1) / a_q)
  uint64_t seed;
};

// ---------------------------------------------------------------------------
// One lane, one step whose weights do not depend on N(t): the first step and an
// approximated one (static weights: t < 0), and every step at q = 1 (a_q is one),
// where each neighbour but t weighs w alone.  t's index in N(v) takes one binary
// search (none when p = 1 too), the rest is the static prefix with one jump at t.
// T and r carry the common factor one = 2^16, which r drops again:
// floor(floor(u 2^16 W / 2^64) / 2^16) = floor(u W / 2^64).
// Measured, R-MAT 20, p = q = 1, 51.7M steps: 129 ms through the two lists,
// 1.2 ms here.
template <bool W>
__device__ __forceinline__ int32_t first_order_step(const GraphView& g, int64_t bv, int dv, int32_t t, uint64_t u,
                                                    uint32_t a_p) {
  const int32_t* __restrict__ nv = g.col + bv;
  int pt = dv;  // index of t in N(v), dv when it is not there or weighs like the others
  if (t >= 0 && a_p != kAlphaOne) {
    pt = lower_bound32(nv, dv, t);
    if (pt < dv && __ldg(nv + pt) != t) pt = dv;
  }
  uint64_t wt = 0, c0 = 0;  // w(v, t), and C just before t
  if (pt < dv) {
    wt = W ? (uint64_t)__ldg(g.w + bv + pt) : 1ull;
    c0 = (W ? __ldg(g.wpre + bv + pt) - wt : (uint64_t)pt) << 16;
  }
  const uint64_t jump = ((uint64_t)a_p - (uint64_t)kAlphaOne) * wt;  // modulo 2^64
  const uint64_t T = ((W ? __ldg(g.wpre + bv + dv - 1) : (uint64_t)dv) << 16) + jump;
  if (W && T == 0) return -1;
  uint64_t r = scale_draw(u, T);
  if (pt < dv && r >= c0) {
    if (r - c0 < (uint64_t)a_p * wt) return t;  // inside t's share
    r -= jump;
  }
  const uint64_t m = r >> 16;  // first j with W_j > m
  N2V_CHECK(g, m < (W ? __ldg(g.wpre + bv + dv - 1) : (uint64_t)dv));
  if (!W) return __ldg(nv + m);
  int lo = 0, n = dv - 1;  // (the last position has W_j > m)
  while (n > 0) {
    const int half = n >> 1;
    if (__ldg(g.wpre + bv + lo + half) <= m) {
      lo += half + 1;
      n -= half + 1;
    } else {
      n = half;
    }
  }
  return __ldg(nv + lo);
}

// ---------------------------------------------------------------------------
// One lane, one step (k >= 1), 1 <= deg v <= kLaneDeg: N(v) and N(t) are merged four
// entries against four, one aligned 16-byte load for each four, and the hits are kept
// as a bit mask.  Thirty-two walkers of a warp go side by side, so a step of 20
// neighbours costs a warp about a dozen rounds for 32 steps, where the warp-wide form
// below pays its fixed cost once for each.  When N(t) is much the longer list, the
// lane goes to the next four of it that can hold a neighbour of v by a search of the
// samples.
// Bound: L1, whose every 16 bytes here belong to another line.  Measured (ER, 8M steps
// of 20 neighbours): 1.62 ms with one look-up of samples and block for each
// neighbour (112 sectors a step, L1 91% busy), 0.89 ms merged.
// A lane with a longer N(t) than it can merge keeps only the shortest N(v): up to 64
// R-MAT 20 (4, .25) took 120 ms, up to 8 114 ms.
constexpr int kLaneDeg = 64, kJumpDeg = 8;

// The longest N(t) that is merged four by four; behind it the lane searches.
__device__ __forceinline__ int lane_reach(int dv) { return 4 * dv + 16; }

// Entries 4 k .. 4 k + 3 of the aligned quads that hold the row [b, b + d) (k = 0 holds
// its first entry); none in the place of other rows' entries.
__device__ __forceinline__ int4 lane_quad(const GraphView& g, int64_t b, int d, int k, int32_t none) {
  const int64_t q = (b >> 2) + k;
  // (the quad that the end of col cuts is in the copy of its block)
  const int32_t* p = (q >> 1) == g.cut_block ? g.tail + 4 * (int)(q & 1) : g.col + 4 * q;
  int4 x = __ldg((const int4*)p);
  const unsigned at = (unsigned)(4 * k - (int)(b & 3));
  if (at >= (unsigned)d) x.x = none;
  if (at + 1 >= (unsigned)d) x.y = none;
  if (at + 2 >= (unsigned)d) x.z = none;
  if (at + 3 >= (unsigned)d) x.w = none;
  return x;
}

template <bool W>
__device__ __forceinline__ int32_t lane_block_step(const GraphView& g, int64_t bv, int dv, int64_t bt, int dt,
                                                   int32_t t, uint64_t u, const StepArgs& A) {
  const int32_t* __restrict__ nv = g.col + bv;
  const uint64_t d1 = (uint64_t)kAlphaOne - (uint64_t)A.a_q, d2 = (uint64_t)A.a_p - (uint64_t)A.a_q;
  uint64_t hits = 0;
  int pt = kLaneDeg;  // index of t in N(v)
  const int vlast = (int)(((bv + dv - 1) >> 2) - (bv >> 2)), tlast = (int)(((bt + dt - 1) >> 2) - (bt >> 2));
  const bool jump = dt > lane_reach(dv);
  int vi = 0, ti = 0;
  int4 X = lane_quad(g, bv, dv, 0, -1), Y = lane_quad(g, bt, dt, 0, -2);
  for (;;) {
    const int at = 4 * vi - (int)(bv & 3);  // position of X.x (below 0: another row's)
    const unsigned m = (X.x == Y.x || X.x == Y.y || X.x == Y.z || X.x == Y.w ? 1u : 0u) |
                       (X.y == Y.x || X.y == Y.y || X.y == Y.z || X.y == Y.w ? 2u : 0u) |
                       (X.z == Y.x || X.z == Y.y || X.z == Y.z || X.z == Y.w ? 4u : 0u) |
                       (X.w == Y.x || X.w == Y.y || X.w == Y.z || X.w == Y.w ? 8u : 0u);
    hits |= at >= 0 ? (uint64_t)m << at : (uint64_t)(m >> -at);
    if (X.x == t || X.y == t || X.z == t || X.w == t) pt = at + (X.x == t ? 0 : X.y == t ? 1 : X.z == t ? 2 : 3);
    const int32_t vmax = max(max(X.x, X.y), max(X.z, X.w)), tmax = max(max(Y.x, Y.y), max(Y.z, Y.w));
    const bool next_v = vmax <= tmax || ti == tlast;
    if (next_v && vi == vlast) break;
    int k = (next_v ? vi : ti) + 1;
    if (jump && !next_v) {
      // the first of v's four that Y does not reach, and the block that can hold it
      const int32_t y[1] = {X.x > tmax ? X.x : X.y > tmax ? X.y : X.z > tmax ? X.z : X.w};
      int node[1];
      const BlockRow rt = block_row(g, bt, dt);
      block_search<1>(rt.smp, rt.n1, 0, y, node);
      k = min(tlast, max(k, (int)(2 * ((bt >> 3) + node[0]) - (bt >> 2))));
    }
    N2V_CHECK(g, k > (next_v ? vi : ti) && k <= (next_v ? vlast : tlast));
    const int4 Z = lane_quad(g, next_v ? bv : bt, next_v ? dv : dt, k, next_v ? -1 : -2);
    if (next_v) {
      X = Z;
      vi = k;
    } else {
      Y = Z;
      ti = k;
    }
  }
  N2V_CHECK(g, pt == kLaneDeg || (pt >= 0 && pt < dv && __ldg(nv + pt) == t));
  N2V_CHECK(g, dv > 63 || (hits >> dv) == 0);
  if (pt < kLaneDeg) hits &= ~(1ull << pt);  // t weighs 1/p whatever N(t) holds
  if (!W) {
    const uint64_t T = (uint64_t)A.a_q * (uint64_t)dv + d1 * (uint64_t)__popcll(hits) + (pt < kLaneDeg ? d2 : 0ull);
    const uint64_t r = scale_draw(u, T);
    int lo = 0, n = dv - 1;  // the last position has C = T > r
    while (n > 0) {
      const int half = n >> 1, j = lo + half;
      const uint64_t C = (uint64_t)A.a_q * (uint64_t)(j + 1) + d1 * (uint64_t)__popcll(hits & (~0ull >> (63 - j))) +
                         (pt <= j ? d2 : 0ull);
      if (C <= r) {
        lo = j + 1;
        n -= half + 1;
      } else {
        n = half;
      }
    }
    return __ldg(nv + lo);
  }
  uint64_t T = (uint64_t)A.a_q * __ldg(g.wpre + bv + dv - 1);
  for (uint64_t m = hits; m; m &= m - 1) T += d1 * (uint64_t)__ldg(g.w + bv + (__ffsll((long long)m) - 1));
  if (pt < kLaneDeg) T += d2 * (uint64_t)__ldg(g.w + bv + pt);
  if (T == 0) return -1;
  const uint64_t r = scale_draw(u, T);
  uint64_t C = 0;
  int j = 0;
  for (; j < dv - 1; ++j) {
    const uint32_t a = j == pt ? A.a_p : ((hits >> j) & 1ull ? kAlphaOne : A.a_q);
    C += (uint64_t)__ldg(g.w + bv + j) * a;
    if (C > r) break;
  }
  return __ldg(nv + j);
}

// ---------------------------------------------------------------------------
// Whole warp, one step (k >= 1, both degrees at least 1).  The keys are the
// shorter list, in chunks of 32 and batches of four chunks.  The samples of the
// longer list that lie between a batch's first and last key are staged in shared
// memory (kWin at most; they follow on from the batch before, so each sample is
// read once), every key finds its block there by a fixed-depth search, and the
// batch's 128 blocks are loaded together.  Keys of a batch that spans more
// samples search them in global memory.
//
// As in warp_step, C_j = a_q W_j + D_j, and T = a_q W_last + D_last needs only
// how many keys hit (or the weights they hit).  What is kept of a chunk is its
// ballot of hits and the block of its first key (with weights, also the sum over
// its hits), not a list of positions.  When the chunks are more than the records,
// one record keeps the total of a group of chunks, and the group that holds the
// answer is gone through once more.
//
//   keys N(v), blocks of N(t): a key's index is its position, so C at the end of
//     every chunk is known and the answer's chunk, then its lane, is found by
//     ballots;
//   keys N(t), blocks of N(v): a hit's position in N(v) is its lower bound there.
//     It is taken for the first key of each chunk (one lane each, inside the
//     recorded block), then for the 32 keys of the answer's chunk only.
//
// t itself (weight 1/p) is never counted as a hit: its part of D is added where
// a position is at or behind it.
//
// Bound: instruction issue while the graph's hot lists stay in L2, DRAM beyond.  The
// size of the code is part of it, since the warps of an SM are all over it: at 2,500
// instructions a kernel waits for none, at 3,300 a seventh of the time, at 4,600 it
// takes twice as long (R-MAT 20).  A separate form for one batch in registers saved a
// fifth of WeC-20's instructions and was slower for that reason.
constexpr int kWin = 128;         // staged samples per warp
constexpr int32_t kNoKey = -2;    // in the place of a key past the end: below every vertex, equal to none

// Shared memory of one warp: cap record words, cap more (the blocks of the first
// keys; with weights the records take both), kWin samples.
__host__ __device__ __forceinline__ int block_records(const LaunchCfg& L) {
  return L.smem_specials < 256 ? L.smem_specials : 256;
}
__host__ __device__ __forceinline__ int block_smem_words(const LaunchCfg& L) { return 2 * block_records(L) + kWin; }

template <bool W>
struct BlockStep {
  // Chunks of a batch.  With weights two: four are 4,200 instructions and 300 bytes of spills,
  // and weighted R-MAT 23 took 160 ms instead of 143 ms; without, two cost R-MAT 24 133 ms
  // instead of 117 ms.
  static constexpr int kB = W ? 2 : 4;
  using Sum = typename std::conditional<W, uint64_t, uint32_t>::type;  // of hits, or of their weights
  const GraphView& g;
  const StepArgs& A;
  const int64_t bv, bt;
  const int dv, dt;
  const int32_t t;
  const int lane;
  uint32_t* rec;
  const int cap;
  const int32_t* __restrict__ nv;
  const int32_t* __restrict__ nt;
#ifdef N2V_STATS
  bool keys_v = false, searched = false;  // the keys are N(v); a batch was searched in global memory
#endif

  __device__ __forceinline__ int records() const { return W ? cap >> 1 : cap; }
  // record i: total, ballot and first key's block
  __device__ __forceinline__ void put_total(int i, Sum s) {
    if (W) *(uint64_t*)(rec + 4 * i) = s;
    else rec[i] = (uint32_t)s;
  }
  __device__ __forceinline__ Sum total_at(int i, int group) const {
    if (W) return (Sum) * (const uint64_t*)(rec + 4 * i);
    return group == 1 ? (Sum)__popc(rec[i]) : (Sum)rec[i];
  }
  __device__ __forceinline__ uint32_t ballot_at(int i) const { return W ? rec[4 * i + 2] : rec[i]; }
  __device__ __forceinline__ uint32_t& block_of(int i) { return W ? rec[4 * i + 3] : rec[cap + i]; }

  // static prefix of the positions before p
  __device__ __forceinline__ uint64_t w_before(int p) const {
    return W ? (p > 0 ? __ldg(g.wpre + bv + p - 1) : 0ull) : (uint64_t)p;
  }
  // a_q times it
  __device__ __forceinline__ uint64_t base_before(int p) const {
    return W ? (uint64_t)A.a_q * w_before(p) : (uint64_t)A.a_q * (uint32_t)p;
  }
  // D of hits that number (weigh) s
  __device__ __forceinline__ uint64_t part_of(Sum s) const {
    const int32_t d1 = (int32_t)kAlphaOne - (int32_t)A.a_q;
    return W ? (uint64_t)(int64_t)d1 * s : (uint64_t)((int64_t)d1 * (int32_t)s);
  }

  // first position in [lo, hi) of N(v) with an entry >= x (hi if none)
  __device__ __forceinline__ int pos_of(int lo, int hi, int32_t x) const { return lo + lower_bound32(nv + lo, hi - lo, x); }

  // The search of one staged level: p points at the first staged sample not yet known to
  // be at or below the key.
  template <int ST, int NE>
  __device__ __forceinline__ static void level(uint32_t (&p)[NE], const int32_t (&x)[NE]) {
    int32_t s[NE];
#pragma unroll
    for (int e = 0; e < NE; ++e) asm volatile("ld.shared.s32 %0, [%1+%2];" : "=r"(s[e]) : "r"(p[e]), "n"(4 * (ST - 1)));
#pragma unroll
    for (int e = 0; e < NE; ++e)
      asm("{\n .reg .pred q;\n setp.le.s32 q, %1, %2;\n @q add.u32 %0, %0, %3;\n}"
          : "+r"(p[e])
          : "r"(s[e]), "r"(x[e]), "n"(4 * ST));
  }

  // Number of the first n staged samples (n < kWin, ascending, larger ones behind them) at
  // or below each key: a search of the 2^d - 1 >= n first slots.
  template <int NE>
  __device__ __forceinline__ void search_staged(const int32_t* win, int n, const int32_t (&x)[NE], int (&count)[NE]) const {
    const uint32_t w0 = smem_addr(win);
    uint32_t p[NE];
#pragma unroll
    for (int e = 0; e < NE; ++e) p[e] = w0;
    if (n >= 32) {
      if (n >= 64) level<64>(p, x);
      level<32>(p, x);
    }
    if (n >= 8) {
      if (n >= 16) level<16>(p, x);
      level<8>(p, x);
    }
    level<4>(p, x);
    level<2>(p, x);
    level<1>(p, x);
#pragma unroll
    for (int e = 0; e < NE; ++e) count[e] = (int)((p[e] - w0) >> 2);
  }

#ifdef N2V_CHECKED
  // i is the number of the n samples at or below x (a place past the end has no key).
  __device__ void check_found(const int32_t* __restrict__ smp, int n, int i, int32_t x) const {
    N2V_CHECK(g, i >= 0 && i <= n);
    if (x == kNoKey || i < 0 || i > n) return;
    N2V_CHECK(g, i == 0 || __ldg(smp + i - 1) <= x);
    N2V_CHECK(g, i == n || __ldg(smp + i) > x);
  }
#endif

  // Compare keys and blocks; the lane's first key is keys[i0], the others 32 apart.  With edges, a
  // block may be the row's first or last one and a match there an entry of a neighbouring row:
  // then the row's own entries are searched (rare, and one copy of it).
  template <int NE>
  __device__ __forceinline__ void match(const BlockRow& r, bool edges, const int32_t* __restrict__ keys, int i0,
                                        const int (&node)[NE], const int32_t (&x)[NE], const Block (&bl)[NE],
                                        bool (&in)[NE]) const {
#pragma unroll
    for (int e = 0; e < NE; ++e) in[e] = block_has(bl[e], x[e]);
    if (!edges) return;
    unsigned check = 0;
#pragma unroll
    for (int e = 0; e < NE; ++e) check |= in[e] && (node[e] == 0 || node[e] == r.n1 || g.loops) ? 1u << e : 0u;
    if (check) {
      const int32_t* __restrict__ row = r.blk + r.head;
      unsigned no = 0;
#pragma unroll 1
      for (; check; check &= check - 1) {
        const int e = __ffs(check) - 1;
        const int32_t y = __ldg(keys + i0 + 32 * e);
        const int p = lower_bound32(row, r.len, y);
        // t itself is no hit (only a graph with self-loops has t in N(t))
        if (p >= r.len || __ldg(row + p) != y || y == t) no |= 1u << e;
      }
#pragma unroll
      for (int e = 0; e < NE; ++e) in[e] = in[e] && !((no >> e) & 1u);
    }
  }

  // State of a pass over the keys.
  struct Pass {
    const int32_t* __restrict__ keys;  // this lane's key of chunk 0
    int nk;
    int32_t kmax;          // the last key
    const int32_t* __restrict__ smp;  // what is staged: the samples, or the top ones
    int n;                 // of the row
    bool far;              // the top ones
    int stage;             // staged for a batch at first: 64 or 128; 0: searched in global memory
    int from;              // of them, at or below every key still to come
    int group;             // chunks that share one record (1, or a multiple of four)
    int left, gi;          // of the current group: chunks to come, and its record
    int pt;                // index of the key equal to t that this lane saw, or -1
    int32_t nx[kB], ns[4];  // the next batch's keys and samples
    uint32_t w[kB];        // with weights: those of the last batch's hits (this lane's),
    int owed;              // and its record
    Sum sum;               // hits so far (with weights: this lane's share of their weights)
  };

  __device__ __forceinline__ void fetch(Pass& P, const BlockRow& r, int c) const {
    const int32_t* k = P.keys + 32 * c;
    const int n = P.nk - 32 * c;
#pragma unroll
    for (int e = 0; e < kB; ++e) P.nx[e] = 32 * e < n - lane ? __ldg(k + 32 * e) : kNoKey;
    const int32_t* q = P.smp + P.from + lane;
    const int m = P.n - P.from - lane;
    P.ns[0] = 0 < m ? __ldg(q) : INT32_MAX;
    P.ns[1] = 32 < m ? __ldg(q + 32) : INT32_MAX;
    if (P.stage > 64) {
      P.ns[2] = 64 < m ? __ldg(q + 64) : INT32_MAX;
      P.ns[3] = 96 < m ? __ldg(q + 96) : INT32_MAX;
    }
  }

  // One batch: chunks c .. c + kB - 1 (with weights, c at the end only settles the last one).
  __device__ __forceinline__ void batch(Pass& P, const BlockRow& r, int c, int c1, bool vk) {
    int32_t* win = (int32_t*)(rec + 2 * cap);
    int32_t x[kB];
    int node[kB];
    Block b[kB];
    bool edges = P.from == 0 || g.loops;  // a key may lie in the row's first or last block
    if (!W || c < c1) {
#pragma unroll
      for (int e = 0; e < kB; ++e) x[e] = P.nx[e];
      // the batch's largest key
      const int32_t last = P.nk - 32 * c >= 32 * kB ? __shfl_sync(kFull, x[kB - 1], 31) : P.kmax;
      int below = 0;  // staged samples at or below the last key
      if (!W || P.stage) {
        win[lane] = P.ns[0];
        win[32 + lane] = P.ns[1];
        below = (P.ns[0] <= last ? 1 : 0) + (P.ns[1] <= last ? 1 : 0);
        if (P.stage > 64) {
          win[64 + lane] = P.ns[2];
          win[96 + lane] = P.ns[3];
          below += (P.ns[2] <= last ? 1 : 0) + (P.ns[3] <= last ? 1 : 0);
        }
        below = __reduce_add_sync(kFull, below);
        __syncwarp();
      }
      N2V_CHECK(g, below <= P.stage && P.stage <= kWin && P.from >= 0 && P.from + below <= P.n);
      if (below < P.stage) {
        search_staged(win, below, x, node);
#pragma unroll
        for (int e = 0; e < kB; ++e) node[e] += P.from;
        P.from += below;
      } else {
#ifdef N2V_STATS
        searched = true;
#endif
        block_search<kB>(P.smp, P.n, P.from, x, node);
        P.from = __shfl_sync(kFull, node[kB - 1], 31);  // (of use only before a further batch)
        edges = true;
      }
      edges = edges || P.from == P.n;
#ifdef N2V_CHECKED
      for (int e = 0; e < kB; ++e) check_found(P.smp, P.n, node[e], x[e]);
#endif
      if (!W && P.far) {
#pragma unroll
        for (int e = 0; e < kB; ++e) node[e] = block_in_group(r, node[e], x[e]);
      }
#ifdef N2V_CHECKED
      for (int e = 0; e < kB; ++e) check_found(r.smp, r.n1, node[e], x[e]);
#endif
#pragma unroll
      for (int e = 0; e < kB; ++e) b[e] = block_load(r, node[e]);
      if (32 * (c + kB) < P.nk) fetch(P, r, c + kB);
    }
    if (W) {
      settle(P);
      if (c >= c1) return;
    }
    bool has_t = false;
#pragma unroll
    for (int e = 0; e < kB; ++e) has_t = has_t || x[e] == t;
    if (has_t) {
#pragma unroll
      for (int e = 0; e < kB; ++e) P.pt = x[e] == t ? 32 * (c + e) + lane : P.pt;
    }
    bool in[kB];
    match(r, edges, P.keys, 32 * c, node, x, b, in);
    const Sum before = P.sum;
    uint32_t word[kB];
#pragma unroll
    for (int e = 0; e < kB; ++e) {
      word[e] = __ballot_sync(kFull, in[e]);
      if (!W) {
        P.sum += __popc(word[e]);
      } else {  // (the weights are waited for in settle, behind the next batch's loads)
        const int at = vk ? 32 * (c + e) + lane : block_pos(r, node[e], b[e], x[e]);
        N2V_CHECK(g, !in[e] || (at >= 0 && at < dv && __ldg(nv + at) == x[e]));
        P.w[e] = in[e] ? __ldg(g.w + bv + at) : 0u;
        if (P.group == 1 && lane == 0) {
          rec[4 * (P.gi + e) + 2] = word[e];
          block_of(P.gi + e) = (uint32_t)node[e];
        }
      }
    }
    P.owed = P.gi;
    N2V_CHECK(g, P.gi >= 0 && P.gi + (P.group == 1 ? kB : 1) <= records());
    if (P.group == 1) {
      if (!W && lane == 0) {
        if (kB == 4) {
          *(uint4*)(rec + P.gi) = make_uint4(word[0], word[1], word[2 % kB], word[3 % kB]);
          *(uint4*)(rec + cap + P.gi) =
              make_uint4((uint32_t)node[0], (uint32_t)node[1], (uint32_t)node[2 % kB], (uint32_t)node[3 % kB]);
        } else {
          *(uint2*)(rec + P.gi) = make_uint2(word[0], word[1]);
          *(uint2*)(rec + cap + P.gi) = make_uint2((uint32_t)node[0], (uint32_t)node[1]);
        }
      }
      P.gi += kB;
    } else {  // the batch adds to its group's record
      if (lane == 0) {
        if (P.left == P.group) {
          block_of(P.gi) = (uint32_t)node[0];
          put_total(P.gi, 0);
        }
        if (!W) rec[P.gi] += P.sum - before;
      }
      P.left -= kB;
      if (P.left <= 0) {
        P.left = P.group;
        ++P.gi;
      }
    }
    __syncwarp();  // the staged samples are read before the next batch's are written
  }

  // With weights: add the last batch's to the sum and to its records (before the first batch,
  // nothing, to a record that comes to be written).
  __device__ __forceinline__ void settle(Pass& P) {
#pragma unroll
    for (int e = 0; e < kB; ++e) {
      P.sum += P.w[e];
      // the chunk's weights, in two halves that cannot overflow
      Sum cs = (Sum)__reduce_add_sync(kFull, P.w[e] & 0xffffu) +
               ((Sum)__reduce_add_sync(kFull, P.w[e] >> 16) << (W ? 16 : 0));
      if (lane == 0) {
        if (P.group == 1) put_total(P.owed + e, cs);
        else put_total(P.owed, total_at(P.owed, 2) + cs);
      }
    }
  }

  // Look chunks [c0, c1) of the keys up in the longer list; the samples before `from`
  // are at or below every key.  c1 - c0 is a multiple of four unless c1 ends the keys.
  // Leaves a record for each group of chunks and returns the number of hits (with
  // weights: this lane's share of their weights).
  __device__ __forceinline__ Sum look_up(bool vk, const BlockRow& r, int from, int c0, int c1, int group, int* pt) {
    Pass P;
    P.keys = (vk ? nv : nt) + lane;
    P.nk = vk ? dv : dt;
    P.kmax = __ldg((vk ? nv : nt) + P.nk - 1);
    // samples beside a batch: sixteen times the ratio of the lists (128 keys), with weights eight
    // times (64 keys)
    const int beside = r.len >> 3, nb = (P.nk + 32 * kB - 1) / (32 * kB);
    // Without weights the top samples are staged beyond the ratio 4, and a key's group of eight
    // samples is one more load; beyond 64 a batch's window outgrows the staging area and is
    // searched in global memory.  (R-MAT 24: 116.5 ms with the samples themselves at every ratio,
    // 111 ms so.)  With weights the 150 instructions of that cost more than they give (weighted
    // R-MAT 23 138 ms against 125 ms): there the samples are staged up to the ratio 16 and searched
    // in global memory beyond.
    P.far = !W && beside > 64 * nb;
    P.smp = P.far ? r.top : r.smp;
    P.n = P.far ? r.n2 : r.n1;
    P.stage = beside <= 48 * nb || (P.far && beside <= 8 * 48 * nb) ? 64 : W && beside > 128 * nb ? 0 : 128;
    P.from = P.far ? (from + r.up) >> 3 : from;
    P.group = group;
    P.left = group;
    P.gi = 0;
    P.sum = 0;
    P.pt = -1;
    P.owed = 0;
#pragma unroll
    for (int e = 0; e < kB; ++e) P.w[e] = 0;
    fetch(P, r, c0);
#pragma unroll 1
    for (int c = c0; c < c1 + (W ? kB : 0); c += kB) batch(P, r, c, c1, vk);
    if (W) __syncwarp();
    *pt = P.pt;
    return P.sum;
  }

  // Where a search of the hits ends: at the chosen position, or (keys N(t)) at the last hit
  // with C at or below r just before it, with D up to there.
  struct Found {
    int pos;
    bool chosen;
    bool hit;  // pos is a hit
    int pos_t;
    uint64_t D, t_part, r;
  };

#ifdef N2V_STATS
  // As the generator modes of warp_step: steps with keys searched in global memory (0, 1), or in
  // staged samples only (2, 3); keys N(v) are modes 0 and 3, and sh counts the keys.
  __device__ __forceinline__ void stat(long long t_enter) const {
    const int sh = keys_v ? dv : dt, lg = keys_v ? dt : dv;
    const int m = searched ? (keys_v ? 0 : 1) : (keys_v ? 3 : 2);
    if (lane == 0) {
      N2V_STAT(kStatMode + 4 * m, 1);
      N2V_STAT(kStatMode + 4 * m + 1, clock64() - t_enter);
      N2V_STAT(kStatMode + 4 * m + 2, sh);
      N2V_STAT(kStatMode + 4 * m + 3, lg);
    }
  }
#endif

  __device__ __forceinline__ uint64_t part_of_t(int pos_t) const {
    return pos_t >= 0 ? ((uint64_t)A.a_p - (uint64_t)A.a_q) * (W ? (uint64_t)__ldg(g.w + bv + pos_t) : 1ull) : 0ull;
  }

  // The chosen position in N(v), or -1 when T == 0.
  __device__ __forceinline__ int run(uint64_t u) {
    // keys N(v) give positions without a search: also when they are the longer list but one batch
    const bool vk = dv <= max(dt, 32 * kB);
#ifdef N2V_STATS
    keys_v = vk;
#endif
    const BlockRow row = vk ? block_row(g, bt, dt) : block_row(g, bv, dv);
    const Found f = search(u, vk, row);
    N2V_CHECK(g, f.pos >= -1 && f.pos < dv);
    return f.chosen ? f.pos : behind(f.pos, f.hit, f.D, f.pos_t, f.t_part, f.r);
  }

  __device__ __forceinline__ Found search(uint64_t u, bool vk, const BlockRow& row) {
    const int nk = vk ? dv : dt;
    // t's position in N(v), -1 when it is not there (keys N(v) have it on the way)
    int pos_t = vk ? -1 : warp_find(t);
    uint64_t t_part = 0;  // (1/p - 1/q) w(v, t) when t is in N(v)
    int c0 = 0, c1 = (nk + 31) >> 5;           // the chunks that can hold the answer
    uint64_t D = 0;                            // the hits' part of D before chunk c0
    int plo = 0, phi = dv;                     // keys N(t): positions of the first keys of c0 and c1
    uint64_t r = 0;
    int from = 0;                              // samples at or below every key from c0 on
    for (bool first = true;; first = false) {
      const int nc = c1 - c0;
      int group = 1;
      if (nc > records()) group = ((nc + records() - 1) / records() + 3) & ~3;  // (a multiple of a batch)
      const int n = (nc + group - 1) / group;
      int pt;
      const Sum part = look_up(vk, row, from, c0, c1, group, &pt);
      if (first) {
        if (vk) pos_t = __reduce_max_sync(kFull, pt);
        t_part = part_of_t(pos_t);
        const Sum all = W ? (Sum)warp_sum_u64(part) : part;
        const uint64_t T = base_before(dv) + part_of(all) + t_part;
        if (W && T == 0) return Found{-1, true};
        r = scale_draw(u, T);
      }
      // the last record that the answer can lie in: C at or below r just before it (keys N(v):
      // before its first key; keys N(t): before the first position its first key can have)
      int pick = 0, npl = plo, nph = phi;
      uint64_t Dp = D;
      for (int i0 = 0; i0 < n; i0 += 32) {
        const int i = i0 + lane;
        const Sum x = i < n ? total_at(i, group) : (Sum)0;
        const Sum incl = W ? (Sum)warp_incl_scan_u64(x, lane) : (Sum)warp_incl_scan_u32((uint32_t)x, lane);
        int p = plo;
        bool before = i == 0;
        if (i > 0 && i < n) {
          p = 32 * (c0 + group * i);
          if (!vk) p = block_lower_bound(row, (int)block_of(i), nv, __ldg(nt + p));
          before = base_before(p) + D + part_of((Sum)(incl - x)) + (pos_t >= 0 && pos_t < p ? t_part : 0ull) <= r;
        }
        const unsigned m = __ballot_sync(kFull, before);
        const int f = 31 - __clz(m);  // -1: none of these
        const Sum excl = __shfl_sync(kFull, (Sum)(incl - x), f & 31), all = __shfl_sync(kFull, incl, 31);
        const int pf = __shfl_sync(kFull, p, f & 31), pn = __shfl_sync(kFull, p, (f + 1) & 31);
        if (f >= 0) {
          pick = i0 + f;
          Dp = D + part_of(excl);
          npl = pf;
        }
        if (f < 31) {  // the next record's first key bounds the answer
          if (i0 + f + 1 < n) nph = pn;
          break;
        }
        D += part_of(all);
      }
      D = Dp;
      plo = npl;
      phi = nph;
      if (group == 1) return in_chunk(vk, c0 + pick, ballot_at(pick), D, pos_t, t_part, plo, phi, r);
      from = (int)block_of(pick);
      c1 = min(c1, c0 + group * (pick + 1));
      c0 += group * pick;
      __syncwarp();  // every lane has read the records before they are written again
    }
  }

  // Position of x in N(v), or -1: the warp narrows the list 32-fold with each load.
  __device__ __forceinline__ int warp_find(int32_t x) const {
    int lo = 0, n = dv;  // the first entry >= x is in [lo, lo + n]
    while (n > 32) {
      const int step = (n + 31) >> 5, i = lo + min((lane + 1) * step, n) - 1;
      const unsigned m = __ballot_sync(kFull, __ldg(nv + i) < x);
      const int f = __popc(m);  // the first f probes are below x
      const int at = f * step;
      if (at >= n) return -1;
      lo += at;
      n = min(step, n - at);
    }
    const unsigned m = __ballot_sync(kFull, lane < n && __ldg(nv + lo + lane) == x);
    return m ? lo + __ffs(m) - 1 : -1;
  }

  // The chosen position, given that it lies in chunk c of the keys (its hits: word; D before
  // it), or, keys N(t), in [plo, phi) from the first key of c on.
  __device__ __forceinline__ Found in_chunk(bool vk, int c, uint32_t word, uint64_t D, int pos_t, uint64_t t_part,
                                          int plo, int phi, uint64_t r) {
    const bool hit = (word >> lane) & 1u;
    int p = 32 * c + lane;
    bool live = p < dv;
    if (!vk) {
      if (hit) p = pos_of(plo, phi, __ldg(nt + p));
      N2V_CHECK(g, !hit || (p >= plo && p < phi && __ldg(nv + p) == __ldg(nt + 32 * c + lane)));
      live = hit;
    }
    Sum incl, own = 1;
    if (W) {
      own = hit ? (Sum)__ldg(g.w + bv + p) : (Sum)0;
      incl = (Sum)warp_incl_scan_u64(own, lane);
    } else {
      incl = (Sum)__popc(word & (0xffffffffu >> (31 - lane)));
    }
    // keys N(v): is C at this key at or below r?  keys N(t): is C just before this hit?
    const int q = vk ? p + 1 : p;
    const bool below = live && base_before(q) + D + part_of(vk ? incl : (Sum)(incl - own)) +
                                       (pos_t >= 0 && pos_t < q ? t_part : 0ull) <= r;
    const unsigned m = __ballot_sync(kFull, below);
    const int f = 31 - __clz(m);
    N2V_CHECK(g, c >= 0 && 32 * c < (vk ? dv : dt) && plo >= 0 && plo <= phi && phi <= dv);
    if (vk) return Found{min(32 * c + f + 1, dv - 1), true};
    int prev = plo - 1;
    if (m) {
      prev = __shfl_sync(kFull, p, f);
      D += part_of(__shfl_sync(kFull, incl, f));
    }
    return Found{prev, false, m != 0u, pos_t, D, t_part, r};
  }

  // The chosen position, given that it is prev (a hit, if hit) or behind it and before the
  // next hit, and the hits' part D of D up to there.
  __device__ __forceinline__ int behind(int prev, bool hit, uint64_t D, int pos_t, uint64_t t_part, uint64_t r) const {
    if (hit && base_before(prev + 1) + D + (pos_t >= 0 && pos_t < prev ? t_part : 0ull) > r) return prev;
    // behind prev every weight is the default, but for t
    bool passed = pos_t >= 0 && pos_t <= prev;
    if (passed) D += t_part;
    for (;;) {
      const int j = first_above(prev, r - D);
      if (pos_t < 0 || passed || j < pos_t) {
        N2V_CHECK(g, j > prev && j < dv);
        return j;
      }
      // t lies in (prev, j], and nothing before it is above r
      if (base_before(pos_t + 1) + D + t_part > r) return pos_t;
      D += t_part;
      prev = pos_t;
      passed = true;
    }
  }

  // First position behind prev whose a_q W exceeds x (the last one if none does).
  __device__ __forceinline__ int first_above(int prev, uint64_t x) const {
    const uint64_t m = div_by(x, A.a_q, A.inv_q);
    if (W) return (int)warp_first_above_u64(g.wpre + bv, prev + 1, dv - 1, m, lane);
    const int j = m > (uint64_t)(dv - 1) ? dv - 1 : (int)m;
    return min(dv - 1, max(j, prev + 1));
  }
};

// ---------------------------------------------------------------------------
// Do most steps stay on their lanes?  Walks visit vertices about in proportion to
// their degree, so the question is how many of the entries of col belong to rows
// of at most kLaneDeg entries.
// Every first step does, and every step at q = 1 (blocks_step).
inline bool lane_walks(const n2v_graph_info& info, int32_t l, uint32_t a_q) {
  if (l == 1 || a_q == kAlphaOne) return true;
  int64_t small = 0;
  for (int i = 1; i < 34 && ((int64_t)1 << i) <= kLaneDeg; ++i) small += info.deg_hist[i] * (((int64_t)3 << i) / 4);
  return 2 * small > info.nnz;
}

// How many walkers a warp takes next of `count`, of which `counter` are taken, where the launch
// does not say it (LaunchCfg::take).  Warp-wide steps of one warp's walkers run one after
// another, so the fewer walkers a warp has, the more warps share the job: half of what is left
// is spread evenly over the warps, up to 32 each.  A small job then runs on as many warps as it
// has walkers, and a large one ends on warps that finish together.
// Measured against 32 a warp throughout: 999 walks on R-MAT 20 7.5 -> 0.67 ms,
// 524,288 on R-MAT 24 in two launches 167 -> 126 ms, 40 mixed serving jobs on R-MAT
// 22 25.9 -> 9.0 ms.
__device__ __forceinline__ int grab_size(int64_t count, const unsigned long long* counter) {
  const int64_t warps = (int64_t)gridDim.x * (kPersistThreads / 32);
  const int64_t left = count - (int64_t)*(const volatile unsigned long long*)counter;
  return (int)max((int64_t)1, min((int64_t)32, left / (2 * warps)));
}

// Where steps stay on their lanes 32 walkers cost a warp no more than one, and the launch fixes the
// walkers that a warp takes: a job is only spread so that one round of the warps takes it, and a
// job of one short step a walker not at all.  Warps then do not read the counter, which costs the
// others as much as their own turn at it.
// Measured, one step from 131,072 vertices of R-MAT 20: 85 us by grab_size, 11 us; from 8,192 of a
// path 14.7 us by an even spread with a look at the counter, 10.1 us without, 8.4 us by 32.
inline int lane_take(int64_t walkers, int32_t l, int64_t warps) {
  return l == 1 ? 32 : (int)std::min<int64_t>(32, (walkers + warps - 1) / warps);
}

// ---------------------------------------------------------------------------
// One step of up to 32 walkers, one per lane.  On its lane: the first step, an
// approximated step, every step at q = 1 and the steps that are short enough; the
// others one after another by the whole warp.
template <bool W, bool APPROX>
__device__ __forceinline__ int32_t blocks_step(const GraphView& g, bool alive, int32_t t, int32_t v, int k, uint64_t wid,
                                               const WalkJob& J, const StepArgs& A, int thr, uint32_t* rec, int cap,
                                               int lane) {
  enum { kDone, kLane, kMid, kWarp };
  int how = kDone;
  int32_t x = -1;
  uint64_t u = 0;
  int64_t bv = 0, bt = 0;
  int dv = 0, dt = 0;
#ifdef N2V_STATS
  const long long t_lane = clock64();
#endif
  if (alive) {
    bv = g.rp[v];
    dv = (int)(g.rp[v + 1] - bv);
    const bool two = k > 0 && (A.a_q != kAlphaOne || APPROX);  // N(t) plays a part
    if (two) {
      bt = g.rp[t];
      dt = (int)(g.rp[t + 1] - bt);
    }
    u = philox_draw(A.seed, wid, (uint32_t)k);
    const bool fixed = k == 0 || (APPROX && approx_here(J, k, dv, dt));
    if (dv == 0) {
      // a dead end
    } else if (fixed || A.a_q == kAlphaOne) {
      x = first_order_step<W>(g, bv, dv, fixed ? -1 : t, u, fixed ? kAlphaOne : A.a_p);
    } else if (dv <= min(thr, kLaneDeg) && dt <= lane_reach(dv)) {
      how = kLane;
    } else {
      how = thr > 0 && dv <= (dt <= lane_reach(dv) ? kLaneDeg : kJumpDeg) ? kMid : kWarp;
    }
  }
  // other steps of up to kLaneDeg neighbours stay on their lanes when enough lanes have one
  const bool together = __popc(__ballot_sync(kFull, how == kMid)) >= 8;
  if (how == kLane || (together && how == kMid)) {
    x = lane_block_step<W>(g, bv, dv, bt, dt, t, u, A);
    how = kDone;
  }
  __syncwarp();
#ifdef N2V_STATS
  {
    const unsigned mx = __reduce_max_sync(kFull, (unsigned)min(clock64() - t_lane, 0xffffffffll));
    const bool any_alive = __any_sync(kFull, alive);  // every lane votes
    if (lane == 0 && any_alive) {
      N2V_STAT(k == 0 ? kStatFirst : kStatLaneSteps, 1);
      N2V_STAT(k == 0 ? kStatFirstCycles : kStatLaneCycles, mx);
    }
  }
#endif
  unsigned wm = __ballot_sync(kFull, how != kDone);
  while (wm) {
    const int src = __ffs(wm) - 1;
    wm &= wm - 1;
    // (a shuffle from one lane: the compiler knows these to be the same in every lane and keeps
    // them in uniform registers; through shared memory they cost the step 130 bytes of spills)
    const int64_t bv_ = __shfl_sync(kFull, bv, src), bt_ = __shfl_sync(kFull, bt, src);
    BlockStep<W> st{g, A, bv_, bt_, __shfl_sync(kFull, dv, src), __shfl_sync(kFull, dt, src),
                    __shfl_sync(kFull, t, src), lane, rec, cap, g.col + bv_, g.col + bt_};
#ifdef N2V_STATS
    const long long t_enter = clock64();
#endif
    const int j = st.run(__shfl_sync(kFull, u, src));
#ifdef N2V_STATS
    st.stat(t_enter);
#endif
    if (lane == src) x = j < 0 ? -1 : __ldg(g.col + bv + j);
    __syncwarp();
  }
  return x;
}

}  // namespace n2v

// The walk over a cell's survivors shared by the particle-step kernels (one
// simulation and batched): a warp takes a run of consecutive ids of one cell,
// draws their offset and creation words, counts who stays and who moves, and
// hands out the pair events.
//
// Ids of a cell are consecutive and lie bucket after bucket (column after
// column), so the warp goes through them in windows of 128 ids, lane l taking
// the quad 4 l .. 4 l + 3 of the window (one Philox call per quad and word
// kind).  The columns are looked up 32 at a time: lane l holds column 32 b + l
// of the current block b (its inclusive id prefix, move threshold and sign),
// so a bucket's data reach the warp by shuffles and no row is staged in shared
// memory; the per-block prefixes `bp` written by the per-cell scan give the
// block of any id.  Three cases, chosen per window by uniform tests:
//   - every id of the window in one bucket (92 % of the windows of a 1e8
//     particle state with 450 non-empty buckets a cell): the stretch of such
//     windows runs with the bucket's data in uniform values, two instructions
//     per particle beside the generator, one warp reduction per stretch;
//   - otherwise up to kFewBuckets buckets of more than kLaneBucket ids in the
//     window are counted under quad masks, bucket by bucket;
//   - and the others from the offset words in shared memory: each by the lane
//     that holds its column, or, if one has more than kLaneBucket ids, by as many
//     lanes as there are for each column.
// The counts then go out together, with neighbouring columns' additions coalesced.
//
// What bounds it: instruction issue and the wide multiplier.  The two calls of a
// quad take 34 wide multiplications (4 cycles each on a scheduler) and as many
// XORs; a one-bucket window takes 104 instructions (with creation words), a
// mixed one several hundred.  Measured (ncu, 1.08e8 particles, 3555 occupied
// cells with 450 non-empty buckets each): k_step 352 -> 201 us, 275e6 -> 140e6
// warp instructions, against the form that staged each row in shared memory
// and gave every lane a run of ids of its own (nearly every warp iteration
// then met a lane that changed its bucket); drift only, 1e7 particles on 2000
// cells: 34 -> 20 us.  The generator alone takes 111 us for the calls of the first.
// Rows of 64 columns that are all held by a few dozen ids are what that form did
// best: 16384 such cells, two steps, drift only, mean bucket 20, 50 and 130: 213,
// 368 and 675 us there, here 334, 478 and 805 us with every larger bucket under
// masks and 228, 402 and 758 us as it is.
#pragma once

#include "wmc_batch_ranges.cuh"
#include "wmc_device.cuh"

namespace wmc {

// With 4, 8, 16 and 32: 16384 cells, four steps 1320, 1238, 1207 and 1207 us; 2000
// cells, twenty steps 306, 306, 305 and 312 us; 512 simulations, four steps 3346,
// 3286, 3263 and 3300 us; 38 simulations of 2.5e7 scattered particles, four steps
// 1379, 1274, 1163 and 1147 us.
constexpr uint32_t kLaneBucket = 16;
// A bucket under masks takes some forty instructions of the whole warp, shared-out
// lanes about as many for all buckets and five more for every four ids of a lane's:
// with 1 instead of 2, buckets of 130 ids (above) 829 instead of 758 us; with all
// windows' lanes shared out also where no bucket is large, 400 small simulations
// 1148 instead of 1110 us.
constexpr int kFewBuckets = 2;

// Move entry of a column: bits 1-2 drift direction + 1, bits 8-31 the crossing
// threshold on the offset word w (move_threshold).  A right-moving column's
// particles move iff w > th, a left-moving one's iff not, a resting one's never.
// (Thresholds act on the 24 offset bits, so their low byte is all ones.)
constexpr uint32_t kMoveNever = 0xffffff02u;
__device__ __forceinline__ uint32_t move_entry(float d) {
  if (d > 0.f) return ((uint32_t)(first_offset_reaching(d, 1.f) - 1) << 8) | 4u;
  const int j = d < 0.f ? first_offset_reaching(d, 0.f) : 0;
  return j ? (uint32_t)(j - 1) << 8 : kMoveNever;
}
// Drift direction of a move entry: -1, 0, 1.
__device__ __forceinline__ int move_dir(uint32_t e) { return (int)((e >> 1) & 3u) - 1; }
// Which of a quad's words move under entry e (4 bits; higher bits undefined).
__device__ __forceinline__ uint32_t move_bits(const uint4& w, uint32_t e) {
  const uint32_t th = e | 255u;
  const uint32_t m = (uint32_t)(w.x > th) | ((uint32_t)(w.y > th) << 1) | ((uint32_t)(w.z > th) << 2) |
                     ((uint32_t)(w.w > th) << 3);
  return (e & 6u) == 0u ? ~m : m;
}

// 4-bit mask of the elements j of a quad with j < d (d may be <= 0 or >= 4).
__device__ __forceinline__ uint32_t first_mask(int d) { return (1u << min(max(d, 0), 4)) - 1u; }

// The walk takes a cell as a type C with
//   row(col), xm(col): signed count and move entry of a column;
//   bp(b): inclusive id prefix of 32-column block b;
//   n_M(): columns;  off: first id - A, where A is the first id rounded down to
//   a multiple of 4 (id offsets are relative to A);
//   gen, rej: whether any of the cells i - 1, i, i + 1 has an event threshold,
//   and the largest such threshold less one.
// (Accessors, so that a cell's pointers need not stay in registers during the
// draws.)

// The column block a warp holds: lane l's column 32 b + l.
struct WalkBlock {
  int b;         // -1: nothing loaded yet
  uint32_t E;    // id offset just past the bucket
  uint32_t e;    // move entry, with bit 0 = negative count, bit 3 = not empty
  uint32_t end;  // E of the last column (uniform)
  uint32_t grp;  // prefix of block 32 (b / 32) + l
  int pn;        // the next block's count and entry, asked for ahead
  uint32_t pe;
};

__device__ __forceinline__ void walk_begin(WalkBlock& k) {
  k.b = -1;
  k.end = 0u;
  k.grp = 0u;
}

// Moves on to the block holding the id at offset x (at or after k.end, before
// the cell's last).  In a sparse row the ids of one window lie in many blocks:
// the block prefixes stay in the warp and the next block is always under way.
template <class C>
__device__ __forceinline__ void walk_load(const C& c, uint32_t x, WalkBlock& k, int lane) {
  const int n_M = c.n_M(), NB = (n_M + 31) >> 5;
  const uint32_t rel = x - c.off;
  int g = k.b & ~31;
  unsigned above;
  while (!(above = __ballot_sync(0xffffffffu, k.grp > rel))) {
    g += 32;
    k.grp = g + lane < NB ? c.bp(g + lane) : 0xffffffffu;
  }
  const int j = __ffs(above) - 1, nb = g + j;
  k.end = c.off + __shfl_sync(0xffffffffu, k.grp, j);
  uint32_t start = __shfl_sync(0xffffffffu, k.grp, j ? j - 1 : 0);
  if (j == 0) start = g ? c.bp(g - 1) : 0u;
  int col = (nb << 5) + lane;
  int n = k.pn;
  uint32_t e = k.pe;
  if (k.b < 0 || nb != k.b + 1) {
    n = col < n_M ? c.row(col) : 0;
    e = col < n_M ? c.xm(col) : kMoveNever;
  }
  k.b = nb;
  col += 32;
  k.pn = col < n_M ? c.row(col) : 0;
  k.pe = col < n_M ? c.xm(col) : kMoveNever;
  uint32_t incl = n < 0 ? 0u - (uint32_t)n : (uint32_t)n;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const uint32_t u = __shfl_up_sync(0xffffffffu, incl, o);
    if (lane >= o) incl += u;
  }
  // the block ends where its prefix says, whatever the row holds: the walk always advances
  k.E = lane == 31 ? k.end : min(c.off + start + incl, k.end);
  k.e = e | (n < 0 ? 1u : 0u) | (n != 0 ? 8u : 0u);
}

// ---------------------------------------------------------------- sparse rows
// Where a window's ids lie in many column blocks, a few in each, going from block to
// block is one chain of shuffles after the other, about 1000 cycles a block; there
// every lane takes a block of its own and goes through that block's buckets.  Two
// steps of 9 cells x 4096 columns, one in ten with a particle, and of 3000 x 1026:
// 191 and 157 us with each row staged in shared memory, 211 and 194 us from block to
// block, 180 and 154 us; 16384 cells, four steps 1190 -> 1175 us.
constexpr int kManyBlocks = 12;
constexpr uint32_t kFewIds = 128 / kManyBlocks;  // of one block; with more it is not looked at

struct WalkSparse {
  unsigned mask;         // columns of the lane's block not yet handed out
  uint32_t run, lo, hi;  // id offset of the next one; the ids of the window in the block
  int col0;
};

// From offset x, the end of block k, on: whether the ids before wend lie in many
// blocks of the present 32.  If so they are all taken (x moves past them), and k is
// left so that walk_load looks for x anew.
template <class C>
__device__ __forceinline__ bool sparse_begin(const C& c, uint32_t& x, uint32_t wend, WalkBlock& k, int lane,
                                             WalkSparse& s) {
  const uint32_t before = __shfl_up_sync(0xffffffffu, k.grp, 1);  // (lane 0's block is not ahead)
  const uint32_t lo = max(before + c.off, x), hi = min(k.grp < 0xffffffffu - c.off ? k.grp + c.off : 0xffffffffu, wend);
  const unsigned in = __ballot_sync(0xffffffffu, lane && before != 0xffffffffu && lo < hi);
  if (__popc(in) < kManyBlocks) return false;
  const int n_M = c.n_M(), g = k.b & ~31;
  s.mask = 0u;
#pragma unroll 1
  for (unsigned m = in; m;) {
    int b[4], n[4];
#pragma unroll
    for (int u = 0; u < 4; ++u, m &= m - 1u) {
      b[u] = __ffs(m) - 1;
      const int col = ((g + b[u]) << 5) + lane;
      n[u] = m && col < n_M ? c.row(col) : 0;
    }
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const unsigned held = __ballot_sync(0xffffffffu, n[u] != 0);
      if (lane == b[u]) s.mask = held;
    }
  }
  s.run = before + c.off;
  s.lo = lo;
  s.hi = hi;
  s.col0 = (g + lane) << 5;
  const int last = 31 - __clz(in);
  x = __shfl_sync(0xffffffffu, hi, last);
  k.b = g + last - 2;  // (neither the next block nor the one that is still under way)
  k.end = x;
  return true;
}

// The lane's next bucket, its ids [from, to) in the window (none: to = from), its
// column and entry; false when no lane has one.
template <class C>
__device__ __forceinline__ bool sparse_next(const C& c, WalkSparse& s, int& col, uint32_t& e, uint32_t& from,
                                            uint32_t& to) {
  if (!__any_sync(0xffffffffu, s.mask != 0u)) return false;
  from = to = 0u;
  col = 0;
  e = kMoveNever;
  if (s.mask) {
    col = s.col0 + __ffs(s.mask) - 1;
    s.mask &= s.mask - 1u;
    const int n = c.row(col);
    from = max(s.run, s.lo);
    s.run += n < 0 ? 0u - (uint32_t)n : (uint32_t)n;
    to = max(from, min(s.run, s.hi));
    e = c.xm(col) | (n < 0 ? 1u : 0u);
    if (s.run >= s.hi) s.mask = 0u;
  }
  return true;
}

// Low word of R[i]: ids are 32-bit (the plan refuses a larger population).
__device__ __forceinline__ uint32_t id_prefix(const unsigned long long* __restrict__ R, int i) {
  return __ldg(reinterpret_cast<const uint32_t*>(R + i));  // (little-endian)
}

// ---------------------------------------------------------------- cells of a work range
// The work of a step is measured in windows of 128 ids; an occupied cell counts
// for more by its chains of dependent loads (units_of_cell): U[0..n] is the
// prefix of these units over the cells.
struct CellWork {
  int i;
  uint32_t u0, u1;  // the cell's units [U[i], U[i + 1])
};

// The cell holding unit u (U[lo] <= u < U[n]): the warp narrows the range of
// cells by 32 a round.
__device__ __forceinline__ CellWork cell_of_unit(const uint32_t* __restrict__ U, int n, uint32_t u, int lane,
                                                 int lo = 0) {
  int hi = n;
  while (hi - lo > 1) {
    const int step = (hi - lo + 31) >> 5, p = lo + (lane + 1) * step;
    lo += __popc(__ballot_sync(0xffffffffu, p < hi && __ldg(U + p) <= u)) * step;
    hi = min(hi, lo + step);
  }
  CellWork c;
  c.i = lo;
  c.u0 = __ldg(U + lo);
  c.u1 = __ldg(U + lo + 1);
  return c;
}

// The next cell with work after c (one exists: c.u1 < U[n]).
__device__ __forceinline__ CellWork next_cell(const uint32_t* __restrict__ U, int n, const CellWork& c, int lane) {
  const int p = c.i + 2 + lane;
  const uint32_t v = __ldg(U + min(p, n));
  const unsigned m = __ballot_sync(0xffffffffu, v > c.u1);
  if (!m) return cell_of_unit(U, n, c.u1, lane, min(c.i + 33, n - 1));
  const int j = __ffs(m) - 1;
  CellWork d;
  d.i = c.i + 1 + j;
  d.u0 = c.u1;
  d.u1 = __shfl_sync(0xffffffffu, v, j);
  return d;
}

// First window at or after unit u of a cell with t survivors: its windows are
// its last units.
__device__ __forceinline__ uint32_t window_of_unit(const CellWork& c, uint32_t t, uint32_t u) {
  const uint32_t w0 = c.u1 - windows_of_cell(t);
  return u > w0 ? u - w0 : 0u;
}

// The schedule of work ranges over the warps, in units: the first n_warps
// ranges are one per warp, later ones come from a ticket.  Up to kSingleRound
// units a warp everything goes out at once in equal shares (2000 cells, 1e7
// particles: 15.4 us a step against 21 us in rounds of 4).  Beyond, rounds of
// kMaxRange units, then halves of what is left down to kMinRange, so that the
// SMs finish together.  (First ranges of a warp's whole half share, 86 units on
// 1e8 particles, took single warps up to 390 of 340 us: the SM favours its
// older warps, which go on to new ranges while a starved one sits on its
// share; a range of 16 costs 1 % more instructions than one of 32.)
constexpr uint32_t kMinRange = 4, kSingleRound = 24;

struct RangeSchedule {
  uint32_t total;     // units
  uint32_t n_warps;
  uint32_t start, size, ticket;  // current round: first unit, units a range, first ticket

  __device__ __forceinline__ RangeSchedule(uint32_t units, uint32_t warps, uint32_t most = kMaxRange,
                                           uint32_t single = kSingleRound)
      : total(units), n_warps(warps), start(0u), ticket(0u) {
    size = units <= single * warps ? (units + warps - 1u) / warps : most;
    if (units > single * warps) fit();
  }
  // halves the range size while a round of it would take more than half of what is left
  __device__ __forceinline__ void fit() {
    while (size > kMinRange && 2u * size * n_warps > total - start) size >>= 1;
  }
  // unit range of ticket n (tickets of one warp increase); false past the end
  __device__ __forceinline__ bool range(uint32_t n, uint32_t& w0, uint32_t& w1) {
    while (n - ticket >= n_warps) {
      if (!more()) return false;
      start += size * n_warps;
      ticket += n_warps;
      fit();
    }
    const uint32_t at = (n - ticket) * size;
    if (at >= total - start) return false;
    w0 = start + at;
    w1 = min(w0 + size, total);
    return true;
  }
  // whether any ticket after the current round has work
  __device__ __forceinline__ bool more() const { return total - start > size * n_warps; }
};

// ---------------------------------------------------------------- the walk
// Candidate quads of a warp: a quad whose smallest creation word may create a
// pair in one of the three cells is queued with its column, and its words are
// drawn again and tested where the events are completed, 32 quads at a time.
constexpr int kWalkQueue = 160;

// The pair kernels' items: quads, or (split 2) their ids where the threads are
// enough, item e then being id e % 4 of quad e / 4.
__device__ __forceinline__ unsigned pairs_split(unsigned n, unsigned threads) { return n <= threads / 4u ? 2u : 0u; }
__device__ __forceinline__ uint4 pairs_item(const uint4* pairs, unsigned e, unsigned split) {
  uint4 ev = pairs[e >> split];
  if (split) ev.z &= 0xffffu | (1u << (16u + (e & 3u)));
  return ev;
}

// Walks the ids at offsets [r0, r1) of cell c (r0 a multiple of 4, ids before
// the cell's first excluded).  draw(offset / 4, gen, wr, wg) gives the quad's
// offset words and, if gen, its creation words; count(k, e, stay, move) takes
// a bucket's counts from one lane (e: its move entry, bit 0 set if negative);
// push(who, me, offset / 4, k, e, ids) queues the quads of the lanes `who`
// (warp-collective; adds to nq); flush() empties the queue; words: 32 uint4 of
// the warp's shared memory.
template <class C, class Draw, class Count, class Push, class Flush>
__device__ __forceinline__ void walk_ids(const C& c, uint32_t r0, uint32_t r1, int lane, uint4* words,
                                         const int& nq, Draw draw, Count count, Push push, Flush flush) {
  const uint32_t g0 = r0 > c.off ? r0 : c.off;
  if (g0 >= r1) return;
  const bool gen = c.gen;
  const uint32_t rej = c.rej;  // gen: a word above it creates no pair anywhere
  WalkBlock B;
  walk_begin(B);
  uint32_t a = r0;
#pragma unroll 1
  while (a < r1) {
    if (nq > kWalkQueue - 128) flush();  // (a window queues each of its ids at most once)
    uint32_t x = a > g0 ? a : g0;
    if (x >= B.end) walk_load(c, x, B, lane);
    int j = __ffs(__ballot_sync(0xffffffffu, B.E > x)) - 1;
    uint32_t Ej = __shfl_sync(0xffffffffu, B.E, j);
    const uint32_t stop = Ej < r1 ? Ej : r1;
    if (x == a && stop - a >= 128u) {
      // whole windows of one bucket
      const uint32_t e = __shfl_sync(0xffffffffu, B.e, j), th = e | 255u;
      const int k = min((B.b << 5) + j, c.n_M() - 1);
      const uint32_t end = a + ((stop - a) & ~127u), from = a;
      uint32_t above = 0u;
      if (gen) {
#pragma unroll 1
        do {
          const uint32_t q = (a >> 2) + (uint32_t)lane;
          uint4 wr, wg;
          draw(q, true, wr, wg);
          above += (wr.x > th) + (wr.y > th);
          above += (wr.z > th) + (wr.w > th);
          const bool cand = min(min(wg.x, wg.y), min(wg.z, wg.w)) <= rej;
          const unsigned who = __ballot_sync(0xffffffffu, cand);
          a += 128u;
          if (who) {
            push(who, cand, q, k, e, 0xfu);
            if (nq > kWalkQueue - 128) break;
          }
        } while (a < end);
      } else {
#pragma unroll 1
        do {
          uint4 wr, wg;
          draw((a >> 2) + (uint32_t)lane, false, wr, wg);
          above += (wr.x > th) + (wr.y > th);
          above += (wr.z > th) + (wr.w > th);
          a += 128u;
        } while (a < end);
      }
      const uint32_t tot = __reduce_add_sync(0xffffffffu, above), all = a - from;
      const uint32_t mv = (e & 6u) == 0u ? all - tot : tot;
      if (lane == 0) count(k, e, all - mv, mv);
      continue;
    }
    // a window with several buckets, or cut by the range's ends, block by block: one
    // or two large buckets are counted by the warp, the others from the offset
    // words in shared memory by the lane or lanes of each column
    const uint32_t qa = a + 4u * (uint32_t)lane;
    const uint32_t wend = a + 128u < r1 ? a + 128u : r1;
    uint4 wr, wg = make_uint4(0u, 0u, 0u, 0u);
    draw(qa >> 2, gen, wr, wg);
    const unsigned cand = __ballot_sync(0xffffffffu, gen && min(min(wg.x, wg.y), min(wg.z, wg.w)) <= rej);
    while (true) {
      const uint32_t lim = B.end < wend ? B.end : wend;
      // the ids [from, to) of this window in the lane's bucket
      uint32_t from = __shfl_up_sync(0xffffffffu, B.E, 1);
      from = lane && from > x ? from : x;
      const uint32_t to = B.E < lim ? B.E : lim;
      const uint32_t cnt = to > from ? to - from : 0u;
      uint32_t own = cnt, mv = 0u, most = __reduce_max_sync(0xffffffffu, cnt);
      unsigned big = __ballot_sync(0xffffffffu, cnt > kLaneBucket);
      const int k = min((B.b << 5) + lane, c.n_M() - 1);
      if (big && __popc(big) <= kFewBuckets) {
        if (cnt > kLaneBucket) own = 0u;
#pragma unroll 1
        while (big) {
          j = __ffs(big) - 1;
          big &= big - 1u;
          const uint32_t f = __shfl_sync(0xffffffffu, from, j), t = __shfl_sync(0xffffffffu, to, j),
                         e = __shfl_sync(0xffffffffu, B.e, j);
          const uint32_t inb = first_mask((int)(t - qa)) & ~first_mask((int)(f - qa));
          const uint32_t m = __reduce_add_sync(0xffffffffu, (uint32_t)__popc(move_bits(wr, e) & inb));
          if (lane == j) mv = m;
          if (cand) {
            const bool me = (cand >> lane) & 1u && inb != 0u;
            push(__ballot_sync(0xffffffffu, me), me, qa >> 2, min((B.b << 5) + j, c.n_M() - 1), e, inb);
          }
        }
        most = __reduce_max_sync(0xffffffffu, own);
      }
      if (most) {  // (what follows leaves the words read)
        words[lane] = wr;
        __syncwarp();
        const uint32_t* w = reinterpret_cast<const uint32_t*>(words);
        uint32_t above = 0u;
        if (most <= kLaneBucket) {
          const uint32_t th = B.e | 255u;
          w += from - a;
#pragma unroll
          for (uint32_t t0 = 0; t0 < kLaneBucket; t0 += 4) {
            if (t0 && most <= t0) break;
#pragma unroll
            for (uint32_t t = t0; t < t0 + 4; ++t)
              if (t < own) above += w[t] > th;
          }
        } else {
          // columns j0 .. j0 + 2^(5 - s) - 1 hold them: 2^s lanes count each
          const unsigned held = __ballot_sync(0xffffffffu, own != 0u);
          const int j0 = __ffs(held) - 1, s = __clz(31 - __clz(held) - j0) - 27, src = j0 + (lane >> s);
          const uint32_t n = __shfl_sync(0xffffffffu, own, src), th = __shfl_sync(0xffffffffu, B.e, src) | 255u;
          w += __shfl_sync(0xffffffffu, from, src) - a;
#pragma unroll 1
          for (uint32_t t = (uint32_t)lane & ((1u << s) - 1u); t < n; t += 4u << s)
#pragma unroll
            for (uint32_t u = 0; u < 4; ++u)
              if (t + (u << s) < n) above += w[t + (u << s)] > th;
          __syncwarp();
#pragma unroll 1
          for (int o = 1 << s >> 1; o; o >>= 1) above += __shfl_xor_sync(0xffffffffu, above, o);
          above = __shfl_sync(0xffffffffu, above, (lane - j0) << s);
        }
        __syncwarp();
        if (own) mv = (B.e & 6u) == 0u ? own - above : above;
        // candidate quads with ids in this block: their ids in the lanes' buckets
        const unsigned span = (0xffffffffu << ((x - a) >> 2)) & (0xffffffffu >> (31u - ((lim - 1u - a) >> 2)));
#pragma unroll 1
        for (unsigned cd = cand & span; cd; cd &= cd - 1u) {
          const uint32_t q0 = a + 4u * (uint32_t)(__ffs(cd) - 1);
          const uint32_t in = first_mask((int)(from + own - q0)) & ~first_mask((int)(from - q0));
          const bool me = own && in;
          const unsigned who = __ballot_sync(0xffffffffu, me);
          if (who) push(who, me, q0 >> 2, k, B.e, in);
        }
      }
      if (cnt) count(k, B.e, cnt - mv, mv);
      if (lim == wend) break;
      const uint32_t part = lim - x;
      x = lim;
      if (WalkSparse sp; part <= kFewIds && sparse_begin(c, x, wend, B, lane, sp)) {
        words[lane] = wr;
        __syncwarp();
        const uint32_t* w = reinterpret_cast<const uint32_t*>(words);
        int ks;
        uint32_t e, f, t;
#pragma unroll 1
        while (sparse_next(c, sp, ks, e, f, t)) {
          uint32_t above = 0u;
#pragma unroll 1
          for (uint32_t q = f; q < t; ++q) above += w[q - a] > (e | 255u);
          if (f < t) {
            const uint32_t m = (e & 6u) == 0u ? t - f - above : above;
            count(ks, e, t - f - m, m);
          }
#pragma unroll 1
          for (unsigned cd = cand; cd; cd &= cd - 1u) {
            const uint32_t q0 = a + 4u * (uint32_t)(__ffs(cd) - 1);
            const uint32_t ids = f < t ? first_mask((int)(t - q0)) & ~first_mask((int)(f - q0)) : 0u;
            const unsigned who = __ballot_sync(0xffffffffu, ids != 0u);
            if (who) push(who, ids != 0u, q0 >> 2, ks, e, ids);
          }
        }
        __syncwarp();
        if (x == wend) break;
      }
      walk_load(c, x, B, lane);
    }
    a += 128u;
  }
}

}  // namespace wmc

// One step of the postulate (Sec. 2.1) over the survivors of a net histogram:
// free drift, absorption, pair creation with probability gamma dt and momentum
// p' ~ V_W^+ / gamma, and the signed histogram of parents and children (whose
// summation is the annihilation of rule 2).
//
// The survivors are never stored: after annihilation every particle of bucket
// (i, M) carries the same cell, momentum and sign, and its offset is a Philox
// draw of its id, so the histogram and the id prefix describe the ensemble
// exactly.  Two kernels:
//   k_step   -- each warp takes ranges of consecutive ids (RangeSchedule) and
//               walks them cell by cell (walk_ids): parents are counted per
//               bucket and added to the next histogram with one reduction per
//               bucket run; quads that may hold a pair event are queued;
//   k_pairs  -- one thread per queued quad: its words again, the event tests,
//               and per event the PICK draw, p' from the coarse CDF of the
//               cell's kernel row, and the two children.
// When the quads do not fit the queue, k_pairs finds them by a second walk, so
// any rate is handled.
#include "wmc_walk.cuh"

namespace wmc {

constexpr int kStepBlocks = 4;
struct StepArgs {
  const int32_t* hist_in;
  int32_t* hist_out;
  const unsigned long long* R;
  const uint32_t* U;          // prefix of the cells' work units
  const uint32_t* bp;         // id prefixes of the rows' 32-column blocks
  const int* row_map;
  const float* VWh;           // kernel rows [rows][Q/2]
  const long long* ccdf;      // coarse CDF [rows][kCdfBlocks]
  const int* scale;           // fixed-point scale of each row
  const unsigned long long* thr_cell;
  const uint32_t* xm;         // move entries of the columns
  uint4* pairs;               // queued quads (quad_events)
  unsigned pair_cap;
  DevHeader* hdr;
  int n_x, n_M, Q, r0, child_wrap;
  uint32_t sim, k0, k1, t;
  int t_from_device;
  PhiloxKeys K;               // round keys of (k0, k1)
};

// p' of the pair created by particle id (column k, sign sgn) in cell c and the
// children c (k + M', +sgn), (k - M', -sgn); rows follow the cell index or the
// occupied list as the kernel stage laid them out.
__device__ __forceinline__ void pair_children(const StepArgs& a, int rows_by_cell, uint32_t id, uint32_t t, int c,
                                              int k, int sgn, unsigned long long& pairs, unsigned long long& dropped,
                                              long long& drop_signed) {
  const int n_M = a.n_M, h = a.Q / 2;
  const int orow = rows_by_cell ? c : __ldg(a.row_map + c);
  const uint4 wp = philox4x32_10k(make_uint4(id, t, kPurposePick, a.sim), a.K);
  const unsigned long long U2 = ((unsigned long long)(wp.x >> 5) << 26) | (unsigned long long)(wp.y >> 6);
  const float* vrow = a.VWh + (size_t)orow * h;
  const long long* crow = a.ccdf + (size_t)orow * kCdfBlocks;
  const int sc = __ldg(a.scale + orow);
  const int kp = sample_coarse_row(vrow, crow, sc, a.Q, a.r0, n_M, U2);
  ++pairs;
  const int Mp = kp - n_M / 2;
  const int kc2[2] = {k + Mp, k - Mp};
  const int sc2[2] = {sgn, -sgn};
#pragma unroll
  for (int q = 0; q < 2; ++q) {
    int kc = kc2[q];
    if (kc < 0 || kc >= n_M) {
      if (!a.child_wrap) {
        ++dropped;
        drop_signed += sc2[q];
        continue;
      }
      kc = ((kc % n_M) + n_M) % n_M;
    }
    atomicAdd(a.hist_out + (size_t)c * n_M + kc, sc2[q]);
  }
}

// The pair events of one queued quad -- {id / 4, cell, column | sign bit << 12
// | ids << 16, -}: its words are drawn again, its ids of the column tested against the threshold of the
// cell they end in, and each event completed.
__device__ __forceinline__ void quad_events(const StepArgs& a, int rows_by_cell, uint32_t t, const uint4& ev,
                                            unsigned long long& pairs, unsigned long long& dropped,
                                            long long& drop_signed) {
  const int i = (int)ev.y, k = (int)(ev.z & 4095u);
  const uint32_t e = __ldg(a.xm + k);
  const int dir = move_dir(e);
  uint4 wr = make_uint4(ev.x, t - 1u, kPurposeRepos, a.sim), wg = make_uint4(ev.x, t, kPurposeGen, a.sim);
  philox4x32_10_x2k(wr, wg, a.K);
  const unsigned long long t_st = __ldg(a.thr_cell + i);
  const unsigned long long t_mv = (unsigned)(i + dir) < (unsigned)a.n_x ? __ldg(a.thr_cell + i + dir) : 0ull;
  const uint32_t mvb = move_bits(wr, e), u4[4] = {wg.x, wg.y, wg.z, wg.w};
  uint32_t m = 0u;
#pragma unroll
  for (int j = 0; j < 4; ++j) m |= (uint32_t)((unsigned long long)u4[j] < ((mvb >> j) & 1u ? t_mv : t_st)) << j;
  m &= ev.z >> 16;
  while (m) {
    const int j = __ffs(m) - 1;
    m &= m - 1u;
    pair_children(a, rows_by_cell, 4u * ev.x + (uint32_t)j, t, i + ((mvb >> j) & 1u ? dir : 0), k,
                       (ev.z >> 12) & 1u ? -1 : 1, pairs, dropped, drop_signed);
  }
}

// Sums five per-thread counters over the block into the header (one atomic each).
__device__ __forceinline__ void block_counters(DevHeader* hdr, unsigned long long pairs, unsigned long long absorbed,
                                               long long abs_signed, unsigned long long dropped,
                                               long long drop_signed) {
  __shared__ unsigned long long s_red[5][kStepWarps];
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  unsigned long long vals[5] = {pairs, absorbed, (unsigned long long)abs_signed, dropped,
                                (unsigned long long)drop_signed};
#pragma unroll
  for (int j = 0; j < 5; ++j) {
    unsigned long long v = vals[j];
#pragma unroll
    for (int off = 16; off; off >>= 1) v += __shfl_down_sync(0xffffffffu, v, off);
    if (lane == 0) s_red[j][wid] = v;
  }
  __syncthreads();
  if (threadIdx.x < 5) {
    unsigned long long v = 0;
    for (int w = 0; w < kStepWarps; ++w) v += s_red[threadIdx.x][w];
    if (v) {
      unsigned long long* dst[5] = {&hdr->pairs, &hdr->absorbed, reinterpret_cast<unsigned long long*>(&hdr->absorbed_signed),
                                    &hdr->dropped, reinterpret_cast<unsigned long long*>(&hdr->dropped_signed)};
      atomicAdd(dst[threadIdx.x], v);
    }
  }
}

// A cell of one simulation for the walk.
struct StepCell {
  const int32_t* hist;
  const uint32_t* bpa;
  const uint32_t* xma;
  int nM, i;
  uint32_t off, rej;
  bool gen;
  __device__ __forceinline__ int n_M() const { return nM; }
  __device__ __forceinline__ int row(int col) const { return __ldg(hist + (size_t)i * nM + col); }
  __device__ __forceinline__ uint32_t bp(int b) const { return __ldg(bpa + (size_t)i * ((nM + 31) >> 5) + b); }
  __device__ __forceinline__ uint32_t xm(int col) const { return __ldg(xma + col); }
};

// The ids of a range of work units [w0, w1), cell by cell, through walk_ids.
// COUNT: the step proper (parents counted, absorbed particles too); otherwise
// only the quads that may hold events are queued.  queue: kWalkQueue entries
// of the warp and 32 more for the walk's words.
template <bool COUNT, class Flush>
__device__ __forceinline__ void walk_range(const StepArgs& a, uint32_t t, uint32_t w0, uint32_t w1, int lane,
                                           uint4* queue, int& nq, Flush flush) {
  const int n_M = a.n_M;
  CellWork cell = cell_of_unit(a.U, a.n_x, w0, lane);
#pragma unroll 1
  while (true) {
    const int i = cell.i;
    const uint32_t first = id_prefix(a.R, i), last = id_prefix(a.R, i + 1);
    const uint32_t A = first & ~3u, qA = A >> 2;
    StepCell c{a.hist_in, a.bp, a.xm, n_M, i, first & 3u};
    const unsigned long long thr_m = i > 0 ? __ldg(a.thr_cell + i - 1) : 0ull, thr_0 = __ldg(a.thr_cell + i),
                             thr_p = i + 1 < a.n_x ? __ldg(a.thr_cell + i + 1) : 0ull;
    const unsigned long long tmax = max(thr_0, max(thr_m, thr_p));
    c.gen = tmax != 0ull;
    c.rej = (uint32_t)(tmax - 1ull);
    // v particles' net sign (n of them) to column k of cell i + d, or out of the domain
    auto add = [&](int k, int d, int v, uint32_t n) {
      if (!COUNT) return;
      if ((unsigned)(i + d) < (unsigned)a.n_x) {
        atomicAdd(a.hist_out + (size_t)(i + d) * n_M + k, v);
      } else {  // (edge cells only)
        atomicAdd(&a.hdr->absorbed, (unsigned long long)n);
        atomicAdd(reinterpret_cast<unsigned long long*>(&a.hdr->absorbed_signed), (unsigned long long)(long long)v);
      }
    };
    walk_ids(
        c, window_of_unit(cell, last - first, w0) << 7, min(last - A, window_of_unit(cell, last - first, w1) << 7),
        lane, queue + kWalkQueue, nq,
        [&](uint32_t q, bool gen, uint4& wr, uint4& wg) {
          wr = make_uint4(qA + q, t - 1u, kPurposeRepos, a.sim);
          if (gen) {
            wg = make_uint4(qA + q, t, kPurposeGen, a.sim);
            philox4x32_10_x2k(wr, wg, a.K);
          } else {
            wr = philox4x32_10k(wr, a.K);
          }
        },
        [&](int k, uint32_t e, uint32_t stay, uint32_t move) {
          if (stay) add(k, 0, e & 1u ? -(int)stay : (int)stay, stay);
          if (move) add(k, move_dir(e), e & 1u ? -(int)move : (int)move, move);
        },
        [&](unsigned who, bool me, uint32_t q, int k, uint32_t e, uint32_t ids) {
          if (me)
            queue[nq + __popc(who & ((1u << lane) - 1u))] =
                make_uint4(qA + q, (uint32_t)i, (uint32_t)k | ((e & 1u) << 12) | (ids << 16), 0u);
          nq += __popc(who);
        },
        flush);
    if (cell.u1 >= w1) break;
    cell = next_cell(a.U, a.n_x, cell, lane);
  }
}

__global__ __launch_bounds__(kStepThreads, kStepBlocks) void k_step(const __grid_constant__ StepArgs a) {
  __shared__ uint4 s_queue[kStepWarps][kWalkQueue + 32];
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  uint4* queue = s_queue[wid];
  const uint32_t t = a.t_from_device ? a.hdr->step : a.t;
  // (n_items = 0: the plan refused the population)
  const uint32_t total = a.hdr->n_items ? __ldg(a.U + a.n_x) : 0u;
  int nq = 0;  // queued quads (uniform)
  // the warp's queue to the global one; what does not fit there is dropped,
  // and the pair kernel, which sees the count, finds all quads again
  auto flush = [&]() {
    __syncwarp();
    unsigned qb = 0u;
    if (lane == 0) qb = atomicAdd(&a.hdr->pair_count, (unsigned)nq);
    qb = __shfl_sync(0xffffffffu, qb, 0);
    for (int e = lane; e < nq; e += 32)
      if (qb + (unsigned)e < a.pair_cap) a.pairs[qb + (unsigned)e] = queue[e];
    __syncwarp();
    nq = 0;
  };
  // consecutive ranges go to different SMs
  RangeSchedule sched(total, gridDim.x * kStepWarps);
  uint32_t ticket = (uint32_t)wid * gridDim.x + blockIdx.x, w0, w1;
  while (sched.range(ticket, w0, w1)) {
    const bool more = sched.more();
    uint32_t nxt = 0u;
    if (lane == 0 && more) nxt = atomicAdd(&a.hdr->item_ticket, 1u);  // consumed at the end of this range
    walk_range<true>(a, t, w0, w1, lane, queue, nq, flush);
    if (!more) break;
    ticket = sched.n_warps + __shfl_sync(0xffffffffu, nxt, 0);
  }
  if (nq) flush();
  if (blockIdx.x == 0 && threadIdx.x == 0 && a.hdr->n_items > 0) atomicAdd(&a.hdr->particle_steps, a.hdr->population);
}

// All quads of the step that may hold events, found by a second walk and
// completed from the warps' queues: the pair kernel's path when they did not
// fit the global queue (pair_cap quads).
__device__ __noinline__ void rewalk_events(const StepArgs& a, uint32_t t, uint4* queue, unsigned long long& pairs,
                                           unsigned long long& dropped, long long& drop_signed) {
  const int lane = threadIdx.x & 31;
  const int rows_by_cell = (int)a.hdr->rows_by_cell;
  const uint32_t total = a.hdr->n_items ? __ldg(a.U + a.n_x) : 0u;
  constexpr uint32_t kUnits = 32;
  int nq = 0;
  auto flush = [&]() {
    __syncwarp();
    for (int e = lane; e < nq; e += 32) quad_events(a, rows_by_cell, t, queue[e], pairs, dropped, drop_signed);
    __syncwarp();
    nq = 0;
  };
  const uint32_t stride = gridDim.x * kStepWarps * kUnits;
  for (uint32_t w0 = (blockIdx.x * kStepWarps + (threadIdx.x >> 5)) * kUnits; w0 < total; w0 += stride)
    walk_range<false>(a, t, w0, min(w0 + kUnits, total), lane, queue, nq, flush);
  if (nq) flush();
}

// The queued quads of the step: a thread for each of a quad's four ids while the
// grid has that many, so that no thread draws and samples two events one after
// the other; one thread per quad beyond.  24 cells of 1026 columns, 18000 events
// in 16000 quads: 24.5 us by quads, 15.1 us by ids.  The last block to finish resets
// the queue and the range ticket for the next step.
__global__ __launch_bounds__(kStepThreads, 4) void k_pairs(const __grid_constant__ StepArgs a) {
  const int rows_by_cell = (int)a.hdr->rows_by_cell;
  const uint32_t t = a.t_from_device ? a.hdr->step : a.t;
  const unsigned n = a.hdr->pair_count;
  // the blocks that have work (or block 0) count themselves done; the others
  // leave at once, whether they see the count or its reset
  const unsigned split = pairs_split(n, gridDim.x * kStepThreads), items = n << split;
  const unsigned blocks =
      n > a.pair_cap ? gridDim.x : min(gridDim.x, max(1u, (items + kStepThreads - 1) / kStepThreads));
  if (blockIdx.x >= blocks) return;
  unsigned long long pairs = 0, dropped = 0;
  long long drop_signed = 0;
  if (n <= a.pair_cap) {
    for (unsigned e = blockIdx.x * kStepThreads + threadIdx.x; e < items; e += blocks * kStepThreads)
      quad_events(a, rows_by_cell, t, pairs_item(a.pairs, e, split), pairs, dropped, drop_signed);
  } else {
    __shared__ uint4 s_queue[kStepWarps][kWalkQueue + 32];
    rewalk_events(a, t, s_queue[threadIdx.x >> 5], pairs, dropped, drop_signed);
  }
  block_counters(a.hdr, pairs, 0ull, 0ll, dropped, drop_signed);
  __syncthreads();
  if (threadIdx.x == 0) {
    __threadfence();
    if (atomicAdd(&a.hdr->pairs_done, 1u) == blocks - 1u) {
      a.hdr->pair_count = 0u;
      a.hdr->item_ticket = 0u;
      a.hdr->pairs_done = 0u;
      __threadfence();
    }
  }
}

int step_grid() {
  static int cached[8] = {0};
  int dev = 0;
  cudaGetDevice(&dev);
  const int slot = dev & 7;
  if (cached[slot] > 0) return cached[slot];
  int per_sm = 0;
  cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_step, kStepThreads, 0);
  if (per_sm < 1) per_sm = 1;
  int g = per_sm * num_sms();
  if (g > kMaxStepBlocks) g = kMaxStepBlocks;
  cached[slot] = g;
  return g;
}

void prepare_step() { (void)step_grid(); }

cudaError_t launch_step(const wmc_params& p, const View& v, const int32_t* hist_in, uint32_t t, int t_from_device,
                        int32_t* hist_out, cudaStream_t s) {
  const Layout L = layout(p);
  StepArgs a;
  a.hist_in = hist_in;
  a.hist_out = hist_out;
  a.R = v.R;
  a.U = v.U;
  a.bp = v.bp;
  a.row_map = v.row_map;
  a.VWh = v.VWh;
  a.ccdf = v.ccdf;
  a.scale = v.scale;
  a.thr_cell = v.thr_cell;
  a.xm = v.xm;
  a.pairs = v.pairs;
  a.pair_cap = L.pair_cap;
  a.hdr = v.hdr;
  a.n_x = p.n_x;
  a.n_M = p.n_M;
  a.Q = p.Q;
  a.r0 = ((-(p.n_M / 2)) % p.Q + p.Q) % p.Q;
  a.child_wrap = p.child_wrap;
  a.sim = p.sim;
  a.k0 = (uint32_t)(p.seed & 0xffffffffu);
  a.k1 = (uint32_t)(p.seed >> 32);
  a.K = philox_keys(a.k0, a.k1);
  a.t = t;
  a.t_from_device = t_from_device;
  const int grid = step_grid();
  cudaError_t e = step_timing_record(s, false);
  if (e != cudaSuccess) return e;
  k_step<<<grid, kStepThreads, 0, s>>>(a);
  e = cudaGetLastError();
  if (e == cudaSuccess) e = step_timing_record(s, true);
  if (e != cudaSuccess) return e;
  // one thread per queued event (the count is on the device: surplus blocks exit)
  const unsigned pair_blocks = (L.pair_cap + kStepThreads - 1) / kStepThreads;
  k_pairs<<<pair_blocks < 8u * (unsigned)num_sms() ? pair_blocks : 8u * (unsigned)num_sms(), kStepThreads, 0, s>>>(a);
  return cudaGetLastError();
}

// ---------------------------------------------------------------- explicit survivors
// One warp per range of work units, cell by cell: lane l writes the ids 4 l ..
// 4 l + 3 of a window (one Philox call) as one vector per array (cell 16 B,
// offset 16 B, momentum 8 B, sign 4 B) where the quad lies inside the cell,
// else id by id.  Bound by the 11 B written per particle; 1e7 particles on 2000
// cells: 180 -> 45 us (one thread per run of ids, a call per id and single
// stores before; the writes alone would take 16 us).
// SPARSE: rows wide enough for a window in more than kManyBlocks column blocks. 3000
// cells of 1026 columns, one in ten with a particle: 54 us with rows staged in shared
// memory, 61 us from block to block, 21 us; the code costs denser states of such rows
// up to 10 % (12 registers), so narrower ones do without.
template <bool SPARSE>
__global__ __launch_bounds__(kStepThreads) void k_materialize(const int32_t* __restrict__ hist,
                                                              const unsigned long long* __restrict__ R,
                                                              const uint32_t* __restrict__ U,
                                                              const uint32_t* __restrict__ bp,
                                                              const uint32_t* __restrict__ xm, DevHeader* hdr, int n_x,
                                                              int n_M, uint32_t sim, PhiloxKeys K, uint32_t t,
                                                              int32_t* __restrict__ cell, float* __restrict__ f,
                                                              int16_t* __restrict__ M, int8_t* __restrict__ sign,
                                                              long long capacity, int vec_ok) {
  __shared__ uint4 s_words[SPARSE ? kStepWarps : 1][32];
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  if ((long long)hdr->population > capacity) {
    if (blockIdx.x == 0 && threadIdx.x == 0) atomicOr(&hdr->flags, WMC_FLAG_CAPACITY);
    return;
  }
  const uint32_t id_base = (uint32_t)hdr->id_base;
  const uint32_t total = hdr->n_items ? __ldg(U + n_x) : 0u, n_warps = gridDim.x * kStepWarps;
  const bool vec = vec_ok && (id_base & 3u) == 0u;  // a quad's place in the arrays is a multiple of 4
  const uint32_t size = max((total + n_warps - 1u) / n_warps, 1u);
  const uint32_t wn = (uint32_t)wid * gridDim.x + blockIdx.x;
  if (wn >= (total + size - 1u) / size) return;
  const uint32_t w0 = wn * size, w1 = min(w0 + size, total);
  const int h = n_M / 2;
  CellWork cw = cell_of_unit(U, n_x, w0, lane);
#pragma unroll 1
  while (true) {
    const uint32_t first = id_prefix(R, cw.i), last = id_prefix(R, cw.i + 1), A = first & ~3u;
    const StepCell c{hist, bp, xm, n_M, cw.i, first & 3u, 0u, false};
    WalkBlock B;
    walk_begin(B);
    const uint32_t r1 = min(last - A, window_of_unit(cw, last - first, w1) << 7);
#pragma unroll 1
    for (uint32_t a = window_of_unit(cw, last - first, w0) << 7; a < r1; a += 128u) {
      const uint32_t qa = a + 4u * (uint32_t)lane, wend = min(a + 128u, r1);
      const uint4 w = philox4x32_10k(make_uint4((A + qa) >> 2, t, kPurposeRepos, sim), K);
      int ck[4] = {0, 0, 0, 0};
      uint32_t neg = 0u, have = 0u;
      uint32_t x = max(a, c.off);  // ids before x have their columns
      if (x >= B.end) walk_load(c, x, B, lane);
      const int j0 = __ffs(__ballot_sync(0xffffffffu, B.E > x)) - 1;
      if (x == a && wend - a == 128u && __shfl_sync(0xffffffffu, B.E, j0) >= wend) {  // one bucket
        const int k = min((B.b << 5) + j0, n_M - 1);
        ck[0] = ck[1] = ck[2] = ck[3] = k;
        neg = __shfl_sync(0xffffffffu, B.e, j0) & 1u ? 0xfu : 0u;
        have = 0xfu;
        x = wend;
      }
#pragma unroll 1
      while (x < wend) {
        if (x >= B.end) walk_load(c, x, B, lane);
        const uint32_t lim = min(B.end, wend);
        const unsigned nz = __ballot_sync(0xffffffffu, (B.e & 8u) != 0u);
        const uint32_t from = max(qa, x);
        int jl = 0;
#pragma unroll
        for (int s = 16; s; s >>= 1) {
          const uint32_t e = __shfl_sync(0xffffffffu, B.E, jl + s - 1);
          if (e <= from) jl += s;
        }
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          const uint32_t id = qa + (uint32_t)j;
          const bool on = id >= x && id < lim;
          const uint32_t e = __shfl_sync(0xffffffffu, B.E, jl);
          if (on && e <= id) jl = (__ffs(nz & (0xfffffffeu << jl)) - 1) & 31;
          const uint32_t en = __shfl_sync(0xffffffffu, B.e, jl);
          if (on) {
            ck[j] = min((B.b << 5) + jl, n_M - 1);
            neg |= (en & 1u) << j;
            have |= 1u << j;
          }
        }
        const uint32_t part = lim - x;
        x = lim;
        if (WalkSparse sp; SPARSE && x < wend && part <= kFewIds && sparse_begin(c, x, wend, B, lane, sp)) {
          s_words[wid][lane] = w;  // id by id, by the lane of its block
          __syncwarp();
          const uint32_t* words = reinterpret_cast<const uint32_t*>(s_words[wid]);
          int k;
          uint32_t e, q0, q1;
#pragma unroll 1
          while (sparse_next(c, sp, k, e, q0, q1)) {
#pragma unroll 1
            for (uint32_t q = q0; q < q1; ++q) {
              const long long o = (long long)(A + q) - (long long)id_base;
              cell[o] = cw.i;
              f[o] = (float)(words[q - a] >> 8) * 0x1p-24f;
              M[o] = (int16_t)(k - h);
              sign[o] = (int8_t)(e & 1u ? -1 : 1);
            }
          }
          __syncwarp();
        }
      }
      const long long o = (long long)(A + qa) - (long long)id_base;
      const float fv[4] = {(float)(w.x >> 8) * 0x1p-24f, (float)(w.y >> 8) * 0x1p-24f, (float)(w.z >> 8) * 0x1p-24f,
                           (float)(w.w >> 8) * 0x1p-24f};
      if (vec && have == 0xfu) {
        *reinterpret_cast<int4*>(cell + o) = make_int4(cw.i, cw.i, cw.i, cw.i);
        *reinterpret_cast<float4*>(f + o) = make_float4(fv[0], fv[1], fv[2], fv[3]);
        *reinterpret_cast<short4*>(M + o) =
            make_short4((short)(ck[0] - h), (short)(ck[1] - h), (short)(ck[2] - h), (short)(ck[3] - h));
        *reinterpret_cast<char4*>(sign + o) = make_char4(neg & 1u ? -1 : 1, neg & 2u ? -1 : 1, neg & 4u ? -1 : 1,
                                                         neg & 8u ? -1 : 1);
      } else {
#pragma unroll
        for (int j = 0; j < 4; ++j)
          if ((have >> j) & 1u) {
            cell[o + j] = cw.i;
            f[o + j] = fv[j];
            M[o + j] = (int16_t)(ck[j] - h);
            sign[o + j] = (int8_t)((neg >> j) & 1u ? -1 : 1);
          }
      }
    }
    if (cw.u1 >= w1) break;
    cw = next_cell(U, n_x, cw, lane);
  }
}

cudaError_t launch_materialize(const wmc_params& p, const View& v, const int32_t* hist, uint32_t t, int32_t* cell,
                               float* f, int16_t* M, int8_t* sign, long long capacity, cudaStream_t s) {
  const auto aligned = [](const void* q, uintptr_t n) { return (reinterpret_cast<uintptr_t>(q) & (n - 1)) == 0; };
  const int vec_ok = aligned(cell, 16) && aligned(f, 16) && aligned(M, 8) && aligned(sign, 4);
  const auto k = p.n_M > 32 * kManyBlocks ? k_materialize<true> : k_materialize<false>;
  k<<<6 * num_sms(), kStepThreads, 0, s>>>(
      hist, v.R, v.U, v.bp, v.xm, v.hdr, p.n_x, p.n_M, p.sim,
      philox_keys((uint32_t)(p.seed & 0xffffffffu), (uint32_t)(p.seed >> 32)), t, cell, f, M, sign, capacity, vec_ok);
  return cudaGetLastError();
}

}  // namespace wmc

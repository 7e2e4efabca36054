// Batched form: many independent simulations of uneven size advanced together,
// one launch per phase for the whole batch (and the step pair captured in a
// CUDA graph).  Each simulation keeps its own parameters, potential, net
// histogram and Philox stream (counter word 3 = its sim index); its results
// are bit-identical to running it alone.
//
// Cells of all simulations are concatenated (global cell c = cell_off[s] + i);
// per-cell arrays (survivors, id prefix, reach bits, row map, thresholds) are
// indexed by global cell, and the survivor-id prefix, work units and occupied
// list come from one scan over all cells (three passes: block sums, a scan of
// the block sums, and the final block scan).  Ids restart at 0 in every
// simulation: id = G[c] - G[cell_off[s]] + (offset within the cell).
//
// The largest range of ids a warp takes at a time is a run-time parameter
// (ids per lane) chosen by wmc_batch_autotune; the results do not depend on it.
#include <string.h>

#include <mutex>
#include <type_traits>
#include <vector>

#include "wmc_graph_slots.cuh"
#include "wmc_walk.cuh"

namespace wmc {

namespace {

struct SimDesc {
  int n_x, Q, n_M, bc, wrap, h, log2_nM, Kp, Np;
  uint32_t sim, k0, k1;
  float c;
  float pad;
  double dt, d1;
  long long cell_off, hist_off, tab_off, sine_off;
};

constexpr int kScanCells = 1024;  // cells per block of the batch scan
constexpr int kScanThreads = 256;
constexpr int kBatchMaxH = 128;   // warp-per-row kernel: Q <= 256
constexpr int kBatchRowWarps = 8;
constexpr int kScanned = 4;       // counters of the scan: survivors, work items, needed cells, work units

struct BatchLayout {
  size_t header, descs, sim_base, cell_sim, T, G, U, bp, nbk, reach, row_map, thr_cell, occ, live, pairs, blk, cdf,
      xm, sine, total;
  long long n_cells, hist_elems, tab_elems, sine_elems, max_items;
  unsigned pair_cap;
  int n_blk, H, NM, NB;  // NB: 32-column blocks of the widest row
};

int ceil_log2_host(int n) {
  int L = 0;
  while ((1 << L) < n) ++L;
  return L;
}

size_t al256(size_t x) { return (x + 255) & ~(size_t)255; }

bool batch_ok(const wmc_params* ps, int n) {
  if (!ps || n < 1 || n > (1 << 20)) return false;
  for (int s = 0; s < n; ++s) {
    if (!params_ok(&ps[s])) return false;
    if (ps[s].Q / 2 > kBatchMaxH) return false;
  }
  return true;
}

BatchLayout batch_layout(const wmc_params* ps, int n) {
  BatchLayout L;
  L.n_cells = 0;
  L.hist_elems = 0;
  L.tab_elems = 0;
  L.sine_elems = 0;
  L.H = 1;
  L.NM = 2;
  for (int s = 0; s < n; ++s) {
    const int h = ps[s].Q / 2;
    const int Kp = ((h - 1 + 31) / 32) * 32 > 0 ? ((h - 1 + 31) / 32) * 32 : 32;
    const int Np = ((h + 63) / 64) * 64;
    L.n_cells += ps[s].n_x;
    L.hist_elems += (long long)ps[s].n_x * ps[s].n_M;
    L.tab_elems += ps[s].n_M;
    L.sine_elems += (long long)Kp * Np;
    if (h > L.H) L.H = h;
    if (ps[s].n_M > L.NM) L.NM = ps[s].n_M;
  }
  L.n_blk = (int)((L.n_cells + kScanCells - 1) / kScanCells);
  L.max_items = 2 * L.n_cells + (1ll << 23);
  const size_t nc = (size_t)L.n_cells;
  size_t o = 0;
  L.header = o; o = al256(o + sizeof(DevHeader));
  L.descs = o; o = al256(o + sizeof(SimDesc) * n);
  L.sim_base = o; o = al256(o + sizeof(unsigned long long) * n);
  L.cell_sim = o; o = al256(o + sizeof(int) * nc);
  L.T = o; o = al256(o + sizeof(unsigned long long) * nc);
  L.G = o; o = al256(o + sizeof(unsigned long long) * (nc + 1));
  L.U = o; o = al256(o + sizeof(uint32_t) * (nc + 1));
  L.NB = (L.NM + 31) / 32;
  L.bp = o; o = al256(o + sizeof(uint32_t) * nc * (size_t)L.NB);
  L.nbk = o; o = al256(o + nc);
  L.reach = o; o = al256(o + nc);
  L.row_map = o; o = al256(o + sizeof(int) * nc);
  L.thr_cell = o; o = al256(o + sizeof(unsigned long long) * nc);
  L.occ = o; o = al256(o + sizeof(int) * nc);
  L.live = o; o = al256(o + sizeof(int) * nc);
  // one entry per quad that may hold a pair event (if they are more, the pair
  // kernel walks the ids again instead)
  {
    const long long want = L.hist_elems / 8;
    L.pair_cap = (unsigned)(want < (1ll << 21) ? (1ll << 21) : (want > (1ll << 23) ? (1ll << 23) : want));
  }
  L.pairs = o; o = al256(o + sizeof(uint4) * (size_t)L.pair_cap);
  L.blk = o; o = al256(o + sizeof(unsigned long long) * kScanned * (size_t)(L.n_blk + 1));
  L.cdf = o; o = al256(o + sizeof(long long) * nc * (size_t)L.NM);
  L.xm = o; o = al256(o + sizeof(uint32_t) * (size_t)L.tab_elems);
  L.sine = o; o = al256(o + sizeof(float) * (size_t)L.sine_elems);
  L.total = o;
  return L;
}

struct BatchView {
  DevHeader* hdr;
  SimDesc* descs;
  unsigned long long *sim_base, *T, *G, *thr_cell, *blk;
  int *cell_sim, *row_map, *occ, *live;
  unsigned char *reach, *nbk;
  uint4* pairs;
  float* sine;
  long long* cdf;
  uint32_t *U, *bp, *xm;
};

BatchView batch_view(const BatchLayout& L, void* ws) {
  char* b = static_cast<char*>(ws);
  BatchView v;
  v.hdr = reinterpret_cast<DevHeader*>(b + L.header);
  v.descs = reinterpret_cast<SimDesc*>(b + L.descs);
  v.sim_base = reinterpret_cast<unsigned long long*>(b + L.sim_base);
  v.cell_sim = reinterpret_cast<int*>(b + L.cell_sim);
  v.T = reinterpret_cast<unsigned long long*>(b + L.T);
  v.G = reinterpret_cast<unsigned long long*>(b + L.G);
  v.reach = reinterpret_cast<unsigned char*>(b + L.reach);
  v.row_map = reinterpret_cast<int*>(b + L.row_map);
  v.thr_cell = reinterpret_cast<unsigned long long*>(b + L.thr_cell);
  v.occ = reinterpret_cast<int*>(b + L.occ);
  v.live = reinterpret_cast<int*>(b + L.live);
  v.U = reinterpret_cast<uint32_t*>(b + L.U);
  v.bp = reinterpret_cast<uint32_t*>(b + L.bp);
  v.nbk = reinterpret_cast<unsigned char*>(b + L.nbk);
  v.pairs = reinterpret_cast<uint4*>(b + L.pairs);
  v.blk = reinterpret_cast<unsigned long long*>(b + L.blk);
  v.cdf = reinterpret_cast<long long*>(b + L.cdf);
  v.xm = reinterpret_cast<uint32_t*>(b + L.xm);
  v.sine = reinterpret_cast<float*>(b + L.sine);
  return v;
}

// simulation owning element e of a concatenation with offsets off[0..n)
__device__ __forceinline__ int owner(const SimDesc* __restrict__ d, int n, long long e, int which) {
  int lo = 0, hi = n;
  while (hi - lo > 1) {
    const int mid = (lo + hi) >> 1;
    const long long o = which == 0 ? d[mid].cell_off : (which == 1 ? d[mid].tab_off : d[mid].sine_off);
    if (o <= e) lo = mid; else hi = mid;
  }
  return lo;
}

// ---------------------------------------------------------------- set-up
__global__ void k_b_init(const SimDesc* __restrict__ d, int n, long long n_cells, long long tab_elems,
                         long long sine_elems, int* __restrict__ cell_sim, uint32_t* __restrict__ xm,
                         float* __restrict__ sine, DevHeader* hdr) {
  const long long tid = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  const long long nt = (long long)gridDim.x * blockDim.x;
  if (tid == 0) {
    DevHeader z = {};
    z.magic = kMagic;
    *hdr = z;
  }
  for (long long c = tid; c < n_cells; c += nt) cell_sim[c] = owner(d, n, c, 0);
  for (long long e = tid; e < tab_elems; e += nt) {
    const SimDesc& s = d[owner(d, n, e, 1)];
    const int k = (int)(e - s.tab_off);
    xm[e] = move_entry(__double2float_rn((double)(k - s.n_M / 2) * s.d1));
  }
  for (long long e = tid; e < sine_elems; e += nt) {
    const SimDesc& s = d[owner(d, n, e, 2)];
    const long long q = e - s.sine_off;
    sine[e] = sine_entry_n1(s.Q, (int)(q / s.Np), (int)(q % s.Np));
  }
}

// ---------------------------------------------------------------- per-cell scan
// Per cell: survivors, survivor prefixes of the row's 32-column blocks and the
// number of non-empty ones, reach bits, and a zeroed row of the next histogram.
// A warp takes RPW cells; between the steps of a run (rows_known) it passes over
// the cells that can hold no particle -- those the last step did not need -- and
// zeroes only the rows that were occupied.  Memory-bound for many cells: 512
// simulations, 1.06e6 cells, a third of them occupied, 119 us (every row read
// 240 us, and 106 us for clearing the next histograms).  Few cells are a chain
// of latencies instead, eight rows of a warp one after the other 15 us for
// 13000 to 19000 cells, so below kManyCells a warp takes one.
constexpr int kRowsPerWarp = 8;
constexpr long long kManyCells = 1ll << 16;

__device__ __forceinline__ void b_row(const int32_t* __restrict__ hist, const SimDesc* __restrict__ d,
                                      const int* __restrict__ cell_sim, long long c, int NB,
                                      unsigned long long* __restrict__ T, uint32_t* __restrict__ bp,
                                      unsigned char* __restrict__ nbk, unsigned char* __restrict__ reach,
                                      int32_t* __restrict__ out, bool clear) {
  const int lane = threadIdx.x & 31;
  const SimDesc& s = d[__ldg(cell_sim + c)];
  const long long i = c - s.cell_off;
  const int n_M = s.n_M;
  const int32_t* row = hist + s.hist_off + i * n_M;
  int32_t* zrow = out + s.hist_off + i * n_M;
  uint32_t* bpr = bp + (size_t)c * NB;
  // the drift D[M] = fl32(M d1), d1 > 0, has the sign of M: a column right of
  // the centre drifts right, left of it left (a D that rounds to zero only
  // marks a neighbour that needs its kernel anyway, which changes no result)
  unsigned long long a = 0;
  unsigned bits = 0;
  int nb = 0;
  uint32_t before = 0u;  // survivors of the blocks done (modulo 2^32: a larger cell is refused by the scan)
  if ((n_M & 3) == 0 && ((reinterpret_cast<uintptr_t>(row) | reinterpret_cast<uintptr_t>(zrow)) & 15) == 0) {
    const int4* row4 = reinterpret_cast<const int4*>(row);
    int4* z4 = reinterpret_cast<int4*>(zrow);
    const int nq = n_M >> 2;
    for (int q0 = 0; q0 < nq; q0 += 64) {
      int4 v[2];
#pragma unroll
      for (int u = 0; u < 2; ++u) {
        const int q = q0 + 32 * u + lane;
        v[u] = q < nq ? __ldg(row4 + q) : make_int4(0, 0, 0, 0);
        if (clear && q < nq) z4[q] = make_int4(0, 0, 0, 0);
      }
#pragma unroll
      for (int u = 0; u < 2; ++u) {
        const int q = q0 + 32 * u + lane;
        if (q0 + 32 * u >= nq) break;
        uint32_t p = 0u;
        if (__any_sync(0xffffffffu, (v[u].x | v[u].y | v[u].z | v[u].w) != 0)) {
          const int nv[4] = {v[u].x, v[u].y, v[u].z, v[u].w};
#pragma unroll
          for (int e = 0; e < 4; ++e)
            if (nv[e]) {
              const int M = 4 * q + e - n_M / 2;
              const uint32_t m = nv[e] < 0 ? 0u - (uint32_t)nv[e] : (uint32_t)nv[e];
              a += m;
              p += m;
              bits |= 1u | (M > 0 ? 2u : 0u) | (M < 0 ? 4u : 0u);
            }
#pragma unroll
          for (int o = 1; o < 8; o <<= 1) p += __shfl_xor_sync(0xffffffffu, p, o);
          nb += __popc(__ballot_sync(0xffffffffu, p != 0u && (lane & 7) == 0));
          uint32_t w = __shfl_up_sync(0xffffffffu, p, 8);
          if (lane >= 8) p += w;
          w = __shfl_up_sync(0xffffffffu, p, 16);
          if (lane >= 16) p += w;
        }
        if ((lane & 7) == 0 && q < nq) bpr[q >> 3] = before + p;
        before += __shfl_sync(0xffffffffu, p, 31);
      }
    }
  } else {
    for (int k0 = 0; k0 < n_M; k0 += 32) {
      const int k = k0 + lane;
      const int nv = k < n_M ? __ldg(row + k) : 0;
      if (clear && k < n_M) zrow[k] = 0;
      const uint32_t m = nv < 0 ? 0u - (uint32_t)nv : (uint32_t)nv;
      if (nv) {
        const int M = k - n_M / 2;
        a += m;
        bits |= 1u | (M > 0 ? 2u : 0u) | (M < 0 ? 4u : 0u);
      }
      before += __reduce_add_sync(0xffffffffu, m);
      nb += __any_sync(0xffffffffu, nv != 0);
      if (lane == 0) bpr[k0 >> 5] = before;
    }
  }
#pragma unroll
  for (int off = 16; off; off >>= 1) {
    a += __shfl_down_sync(0xffffffffu, a, off);
    bits |= __shfl_down_sync(0xffffffffu, bits, off);
  }
  if (lane == 0) {
    T[c] = a;
    reach[c] = (unsigned char)bits;
    nbk[c] = (unsigned char)nb;
  }
}

template <int RPW>
__global__ void k_b_rows(const int32_t* __restrict__ hist, const SimDesc* __restrict__ d,
                         const int* __restrict__ cell_sim, long long n_cells, int NB,
                         unsigned long long* __restrict__ T, uint32_t* __restrict__ bp,
                         unsigned char* __restrict__ nbk, unsigned char* __restrict__ reach,
                         int32_t* __restrict__ out, const int* __restrict__ row_map, const DevHeader* hdr) {
  const long long c0 = ((blockIdx.x * (long long)blockDim.x + threadIdx.x) >> 5) * RPW;
  const int lane = threadIdx.x & 31;
  if (c0 >= n_cells) return;
  const bool known = hdr->rows_known != 0u;
  const long long c = c0 + lane;
  const bool in = lane < RPW && c < n_cells;
  const bool clear = in && (!known || T[c] != 0ull), read = in && (!known || row_map[c] >= 0);
  if (in && !read) {  // (its row of the next histogram is zero)
    T[c] = 0ull;
    reach[c] = 0;
  }
  const unsigned clears = __ballot_sync(0xffffffffu, clear);
  for (unsigned m = __ballot_sync(0xffffffffu, read); m; m &= m - 1u) {
    const int j = __ffs(m) - 1;
    b_row(hist, d, cell_sim, c0 + j, NB, T, bp, nbk, reach, out, (clears >> j) & 1u);
  }
}

// kernel needed at cell c: occupied, or a neighbour of the same simulation
// drifts into it
__device__ __forceinline__ int b_needs(const unsigned char* __restrict__ reach, const SimDesc* __restrict__ d,
                                       const int* __restrict__ cell_sim, long long c) {
  const SimDesc& s = d[__ldg(cell_sim + c)];
  const long long i = c - s.cell_off;
  return (reach[c] & 1) || (i > 0 && (reach[c - 1] & 2)) || (i + 1 < s.n_x && (reach[c + 1] & 4));
}

__device__ __forceinline__ int b_items(unsigned long long t, int chunk) {
  return t ? (int)((t + 3 + chunk - 1) / chunk) : 0;
}

// block-wide exclusive scan of kScanned counters (256 threads)
__device__ __forceinline__ void block_scan(unsigned long long (&x)[kScanned], unsigned long long* sh /*kScanned x 8*/,
                                           unsigned long long (&tot)[kScanned]) {
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
#pragma unroll
  for (int j = 0; j < kScanned; ++j) {
    unsigned long long in = x[j];
#pragma unroll
    for (int off = 1; off < 32; off <<= 1) {
      const unsigned long long u = __shfl_up_sync(0xffffffffu, in, off);
      if (lane >= off) in += u;
    }
    if (lane == 31) sh[8 * j + wid] = in;
    x[j] = in - x[j];
  }
  __syncthreads();
#pragma unroll
  for (int j = 0; j < kScanned; ++j) {
    tot[j] = 0;
    for (int w = 0; w < 8; ++w) {
      if (w == wid) x[j] += tot[j];
      tot[j] += sh[8 * j + w];
    }
  }
}

constexpr int kCellsPerThread = kScanCells / kScanThreads;

// the counters of cell c added to x
__device__ __forceinline__ void scan_cell(unsigned long long t, int need, uint32_t nb, int chunk,
                                          unsigned long long (&x)[kScanned]) {
  x[0] += t;
  x[1] += b_items(t, chunk);
  x[2] += need;
  x[3] += units_of_cell(t, nb);
}

__global__ __launch_bounds__(kScanThreads) void k_b_scan1(const unsigned long long* __restrict__ T,
                                                          const unsigned char* __restrict__ reach,
                                                          const unsigned char* __restrict__ nbk,
                                                          const SimDesc* __restrict__ d,
                                                          const int* __restrict__ cell_sim, long long n_cells,
                                                          int chunk, unsigned long long* __restrict__ blk) {
  __shared__ unsigned long long sh[8 * kScanned];
  const long long c0 = (long long)blockIdx.x * kScanCells + threadIdx.x * kCellsPerThread;
  unsigned long long x[kScanned] = {}, tot[kScanned];
  for (int q = 0; q < kCellsPerThread; ++q) {
    const long long cc = c0 + q;
    if (cc >= n_cells) break;
    scan_cell(T[cc], b_needs(reach, d, cell_sim, cc), nbk[cc], chunk, x);
  }
  block_scan(x, sh, tot);
  if (threadIdx.x == 0)
    for (int j = 0; j < kScanned; ++j) blk[kScanned * blockIdx.x + j] = tot[j];
}

// single block: exclusive scan of the block sums, totals to the header
__global__ __launch_bounds__(kScanThreads) void k_b_scan2(unsigned long long* __restrict__ blk, int n_blk,
                                                          long long max_items, DevHeader* hdr, int advance_step) {
  __shared__ unsigned long long sh[8 * kScanned];
  __shared__ unsigned long long carry[kScanned];
  if (threadIdx.x < kScanned) carry[threadIdx.x] = 0;
  __syncthreads();
  for (int base = 0; base < n_blk; base += kScanThreads) {
    const int q = base + threadIdx.x;
    unsigned long long x[kScanned] = {}, tot[kScanned];
    if (q < n_blk)
      for (int j = 0; j < kScanned; ++j) x[j] = blk[kScanned * q + j];
    block_scan(x, sh, tot);
    if (q < n_blk)
      for (int j = 0; j < kScanned; ++j) blk[kScanned * q + j] = x[j] + carry[j];
    __syncthreads();
    if (threadIdx.x == 0)
      for (int j = 0; j < kScanned; ++j) carry[j] += tot[j];
    __syncthreads();
  }
  if (threadIdx.x == 0) {
    const int ok = (long long)carry[1] <= max_items && carry[3] < (1ull << 32);
    hdr->n_items = ok ? (int)carry[1] : 0;
    hdr->n_occ = (int)carry[2];
    hdr->n_live = 0;
    hdr->population = 0;  // summed per simulation by k_b_simbase
    if (!ok) atomicOr(&hdr->flags, WMC_FLAG_CAPACITY);
    if (advance_step) {
      hdr->step += 1u;
      hdr->rows_known = 1u;
    }
  }
}

__global__ __launch_bounds__(kScanThreads) void k_b_scan3(
    const unsigned long long* __restrict__ T, const unsigned char* __restrict__ reach,
    const unsigned char* __restrict__ nbk, const SimDesc* __restrict__ d, const int* __restrict__ cell_sim,
    long long n_cells, int chunk, const unsigned long long* __restrict__ blk, unsigned long long* __restrict__ G,
    uint32_t* __restrict__ U, int* __restrict__ occ, int* __restrict__ row_map,
    unsigned long long* __restrict__ thr_cell, DevHeader* hdr) {
  __shared__ unsigned long long sh[8 * kScanned];
  const long long c0 = (long long)blockIdx.x * kScanCells + threadIdx.x * kCellsPerThread;
  unsigned long long x[kScanned] = {}, tot[kScanned];
  for (int q = 0; q < kCellsPerThread; ++q) {
    const long long cc = c0 + q;
    if (cc >= n_cells) break;
    scan_cell(T[cc], b_needs(reach, d, cell_sim, cc), nbk[cc], chunk, x);
  }
  block_scan(x, sh, tot);
#pragma unroll
  for (int j = 0; j < kScanned; ++j) x[j] += blk[kScanned * blockIdx.x + j];
  for (int q = 0; q < kCellsPerThread; ++q) {
    const long long cc = c0 + q;
    if (cc >= n_cells) break;
    const unsigned long long t = T[cc];
    const int need = b_needs(reach, d, cell_sim, cc);
    G[cc] = x[0];
    U[cc] = (uint32_t)x[3];
    if (t > 0x7fffffffull) {  // a cell's ids must fit the 31-bit row-local offsets
      atomicOr(&hdr->flags, WMC_FLAG_CAPACITY);
      hdr->n_items = 0;
    }
    if (need) {
      occ[x[2]] = (int)cc;
      row_map[cc] = (int)x[2];
    } else {
      row_map[cc] = -1;
    }
    thr_cell[cc] = 0ull;
    scan_cell(t, need, nbk[cc], chunk, x);
  }
  if (blockIdx.x == gridDim.x - 1 && threadIdx.x == 0) {
    G[n_cells] = blk[kScanned * blockIdx.x] + tot[0];
    U[n_cells] = (uint32_t)(blk[kScanned * blockIdx.x + 3] + tot[3]);
  }
}

// per simulation: first id offset and population
__global__ void k_b_simbase(const SimDesc* __restrict__ d, int n, const unsigned long long* __restrict__ G,
                            unsigned long long* __restrict__ base, DevHeader* hdr) {
  const int s = blockIdx.x * blockDim.x + threadIdx.x;
  if (s >= n) return;
  const unsigned long long b0 = G[d[s].cell_off], b1 = G[d[s].cell_off + d[s].n_x];
  base[s] = b0;
  const unsigned long long P = b1 - b0;
  atomicAdd(&hdr->population, P);
  if (P >= (1ull << 32)) {  // ids of one simulation are 32-bit
    atomicOr(&hdr->flags, WMC_FLAG_CAPACITY);
    hdr->n_items = 0;
  }
}

// ---------------------------------------------------------------- kernel rows
// The needed cells that see a potential: a cell whose window differences all
// vanish has an exactly zero row and creates no pair, so its row is not built
// (its threshold is zero already).  One thread per needed cell.
__global__ __launch_bounds__(256) void k_b_live(const float* __restrict__ V, const SimDesc* __restrict__ d,
                                                const int* __restrict__ cell_sim, const int* __restrict__ occ,
                                                int* __restrict__ live, DevHeader* hdr) {
  const int n_rows = hdr->n_occ, lane = threadIdx.x & 31;
  const int stride = gridDim.x * blockDim.x;
  for (int r0 = blockIdx.x * blockDim.x + threadIdx.x - lane; r0 < n_rows; r0 += stride) {
    const int row = r0 + lane;
    bool on = false;
    if (row < n_rows) {
      const int cg = __ldg(occ + row);
      const SimDesc& s = d[__ldg(cell_sim + cg)];
      const float* Vs = V + s.cell_off;
      const int i = (int)(cg - s.cell_off), n_x = s.n_x, bc = s.bc, h = s.h;
      for (int m = 1; m < h && !on; m += 8) {  // eight differences in flight
#pragma unroll
        for (int u = 0; u < 8; ++u)
          if (m + u < h)
            on |= __fsub_rn(pot(Vs, n_x, bc, (long long)i + m + u), pot(Vs, n_x, bc, (long long)i - m - u)) != 0.f;
      }
    }
    const unsigned who = __ballot_sync(0xffffffffu, on);
    if (who) {
      int at = 0;
      if (lane == 0) at = atomicAdd(&hdr->n_live, __popc(who));
      at = __shfl_sync(0xffffffffu, at, 0);
      if (on) live[at + __popc(who & ((1u << lane) - 1u))] = row;
    }
  }
}

// One warp per such cell (LIVE), or per needed cell with the same test inside
// where there are few: FP32 contraction with the simulation's own window and
// sine matrix (read through L1), then the fixed-point CDF and event threshold
// of the row.  With a warp per needed cell, most of them flat, the rows took
// 171 us of 512 simulations' step, a chain of dependent loads each, 48 us by the
// list; for 19000 cells the list's own kernel takes 13 us, so it is made from
// kManyCells cells on.
template <int C, bool LIVE>
__global__ __launch_bounds__(kBatchRowWarps * 32) void k_b_kernel_rows(
    const float* __restrict__ V, const SimDesc* __restrict__ d, const int* __restrict__ cell_sim,
    const int* __restrict__ occ, const int* __restrict__ live, DevHeader* __restrict__ hdr,
    const float* __restrict__ sine, int NM, long long* __restrict__ cdf, unsigned long long* __restrict__ thr_cell) {
  __shared__ float s_buf[kBatchRowWarps][2 * 32 * C];
  const int n_rows = LIVE ? hdr->n_live : hdr->n_occ;
  const int wid = threadIdx.x >> 5, lane = threadIdx.x & 31;
  float* s_row = s_buf[wid];
  float* s_dv = s_buf[wid] + 32 * C;
  for (int l = blockIdx.x * kBatchRowWarps + wid; l < n_rows; l += gridDim.x * kBatchRowWarps) {
    const int row = LIVE ? __ldg(live + l) : l;
    const int cg = __ldg(occ + row);
    const SimDesc& s = d[__ldg(cell_sim + cg)];
    const int i = (int)(cg - s.cell_off), h = s.h, Q = s.Q, n_M = s.n_M;
    const float* Vs = V + s.cell_off;
    const float* B = sine + s.sine_off;
#pragma unroll
    for (int q = 0; q < C; ++q) {
      const int m = lane + 1 + 32 * q;
      s_dv[m - 1] = m <= h - 1 ? __fsub_rn(pot(Vs, s.n_x, s.bc, (long long)i + m), pot(Vs, s.n_x, s.bc, (long long)i - m))
                               : 0.f;
    }
    if (!LIVE) {
      bool nz = false;
#pragma unroll
      for (int q = 0; q < C; ++q) nz |= s_dv[lane + 32 * q] != 0.f;
      if (!__any_sync(0xffffffffu, nz)) continue;
    }
    __syncwarp();
    float sacc[C], eacc[C];
#pragma unroll
    for (int cc = 0; cc < C; ++cc) sacc[cc] = eacc[cc] = 0.f;
    for (int m0 = 1; m0 <= h - 1; m0 += 32) {
      float part[C];
#pragma unroll
      for (int cc = 0; cc < C; ++cc) part[cc] = 0.f;
      const int m1 = min(m0 + 32, h);
      for (int m = m0; m < m1; ++m) {
        const float dv = s_dv[m - 1];
        const float* brow = B + (size_t)(m - 1) * s.Np;
#pragma unroll
        for (int cc = 0; cc < C; ++cc) {
          const int r = lane + 32 * cc;
          if (r < h) part[cc] = fmaf(dv, __ldg(brow + r), part[cc]);
        }
      }
#pragma unroll
      for (int cc = 0; cc < C; ++cc) two_sum_acc(sacc[cc], eacc[cc], part[cc]);
    }
#pragma unroll
    for (int cc = 0; cc < C; ++cc) {
      const int r = lane + 32 * cc;
      if (r < h) s_row[r] = __fmul_rn(s.c, __fadd_rn(sacc[cc], eacc[cc]));
    }
    __syncwarp();
    const int r0 = ((-(n_M / 2)) % Q + Q) % Q;
    auto xres = [&](int rr) { return positive_part_smem(s_row, Q, rr); };
    double g;
    int sc;
    long long tot;
    warp_row_cdf(xres, Q, r0, n_M, s.log2_nM, lane, cdf + (size_t)row * NM, g, sc, tot, false);
    if (lane == 0) thr_cell[cg] = g > 0.0 ? event_threshold(g, s.dt, &hdr->flags) : 0ull;
    __syncwarp();
  }
}

// ---------------------------------------------------------------- step
struct BatchStepArgs {
  const int32_t* hist_in;
  int32_t* hist_out;
  const SimDesc* d;
  const int* cell_sim;
  const unsigned long long* G;
  const unsigned long long* sim_base;
  const uint32_t* U;
  const uint32_t* bp;
  const int* row_map;
  const long long* cdf;
  const unsigned long long* thr_cell;
  const uint32_t* xm;
  uint4* pairs;
  unsigned pair_cap;
  DevHeader* hdr;
  int NM, NB, n_cells;
  uint32_t max_range;  // work units of the schedule's largest ranges
};

// The walk and the pair events of wmc_step.cu on the concatenated cells: the
// work units of all simulations are one sequence, so a warp's range may run
// from one simulation into the next.
constexpr int kBStepWarps = 8;
// Units a warp up to which everything goes out at once (RangeSchedule).  Units of
// several simulations differ more in cost than those of one, whole windows of a
// bucket beside scattered ones with events: 28 simulations, 4.8e6 particles and
// 12 units a warp, took 445 us for three steps in ranges of 16 and less, 519 us
// in equal shares; 512 simulations are far above either.
constexpr uint32_t kBSingleRound = 8;

// One thread's share of the step's counters.
struct PairCounters {
  unsigned long long pairs = 0, dropped = 0;
  long long drop_signed = 0;
};

// The pair events of one queued quad {id / 4, cell, column | sign bit << 12 |
// ids << 16, -}.
__device__ __forceinline__ void b_quad_events(const BatchStepArgs& a, uint32_t t, const uint4& ev, PairCounters& pc) {
  const int cg = (int)ev.y, k = (int)(ev.z & 4095u);
  const SimDesc& S = a.d[__ldg(a.cell_sim + cg)];
  const int n_M = S.n_M, i = (int)(cg - S.cell_off);
  const uint32_t sim = S.sim, k0 = S.k0, k1 = S.k1;
  const uint32_t e = __ldg(a.xm + S.tab_off + k);
  const int dir = move_dir(e);
  uint4 wr = make_uint4(ev.x, t - 1u, kPurposeRepos, sim), wg = make_uint4(ev.x, t, kPurposeGen, sim);
  philox4x32_10_x2(wr, wg, k0, k1);
  const unsigned long long t_st = __ldg(a.thr_cell + cg);
  const unsigned long long t_mv = (unsigned)(i + dir) < (unsigned)S.n_x ? __ldg(a.thr_cell + cg + dir) : 0ull;
  const uint32_t mvb = move_bits(wr, e), u4[4] = {wg.x, wg.y, wg.z, wg.w};
  uint32_t m = 0u;
#pragma unroll
  for (int j = 0; j < 4; ++j) m |= (uint32_t)((unsigned long long)u4[j] < ((mvb >> j) & 1u ? t_mv : t_st)) << j;
  m &= ev.z >> 16;
  while (m) {
    const int j = __ffs(m) - 1;
    m &= m - 1u;
    // p' from the PICK draw of this id, children into the cell it ended in
    const int dd = (mvb >> j) & 1u ? dir : 0;
    const int orow = __ldg(a.row_map + cg + dd);
    const uint4 wp = philox4x32_10(make_uint4(4u * ev.x + (uint32_t)j, t, kPurposePick, sim), k0, k1);
    const unsigned long long U2 = ((unsigned long long)(wp.x >> 5) << 26) | (unsigned long long)(wp.y >> 6);
    const int Mp = sample_cdf_row(a.cdf + (size_t)orow * a.NM, n_M, U2) - n_M / 2;
    ++pc.pairs;
    const int sgn = (ev.z >> 12) & 1u ? -1 : 1;
    const int kc2[2] = {k + Mp, k - Mp}, sc2[2] = {sgn, -sgn};
    int32_t* out = a.hist_out + S.hist_off + (size_t)(i + dd) * n_M;
#pragma unroll
    for (int q = 0; q < 2; ++q) {
      int kc = kc2[q];
      if (kc < 0 || kc >= n_M) {
        if (!S.wrap) {
          ++pc.dropped;
          pc.drop_signed += sc2[q];
          continue;
        }
        kc = ((kc % n_M) + n_M) % n_M;
      }
      atomicAdd(out + kc, sc2[q]);
    }
  }
}

// A cell of some simulation for the walk: its pointers in the warp's shared
// memory, so that the draws keep their registers.
struct BatchRow {
  const int32_t* row;
  const uint32_t* bp;
  const uint32_t* xm;
  int32_t* out;  // the cell's row of the next histogram
  int n_M, i, n_x, cg;
};

struct BatchCell {
  const BatchRow* r;
  uint32_t off, rej;
  bool gen;
  __device__ __forceinline__ int n_M() const { return r->n_M; }
  __device__ __forceinline__ int row(int col) const { return __ldg(r->row + col); }
  __device__ __forceinline__ uint32_t bp(int b) const { return __ldg(r->bp + b); }
  __device__ __forceinline__ uint32_t xm(int col) const { return __ldg(r->xm + col); }
};

// The ids of the work units [w0, w1), cell by cell.  COUNT: parents counted,
// absorbed particles too; otherwise only the quads that may hold events are
// queued.
template <bool COUNT, class Flush>
__device__ __forceinline__ void b_walk_range(const BatchStepArgs& a, uint32_t t, uint32_t w0, uint32_t w1, int lane,
                                             uint4* queue, BatchRow* br, int& nq, Flush flush) {
  CellWork cell = cell_of_unit(a.U, a.n_cells, w0, lane);
#pragma unroll 1
  while (true) {
    const int cg = cell.i, sidx = __ldg(a.cell_sim + cg);
    const SimDesc& S = a.d[sidx];
    const int i = (int)(cg - S.cell_off);
    const uint32_t sim = S.sim, k0 = S.k0, k1 = S.k1;
    const uint32_t sb = id_prefix(a.sim_base, sidx);
    const uint32_t first = id_prefix(a.G, cg) - sb, last = id_prefix(a.G, cg + 1) - sb;
    const uint32_t A = first & ~3u, qA = A >> 2;
    __syncwarp();
    if (lane == 0) {
      const int n_M = S.n_M;
      const long long at = S.hist_off + (long long)i * n_M;
      br->row = a.hist_in + at;
      br->bp = a.bp + (size_t)cg * a.NB;
      br->xm = a.xm + S.tab_off;
      br->out = a.hist_out + at;
      br->n_M = n_M;
      br->i = i;
      br->n_x = S.n_x;
      br->cg = cg;
    }
    __syncwarp();
    BatchCell c{br, first & 3u};
    const unsigned long long thr_m = i > 0 ? __ldg(a.thr_cell + cg - 1) : 0ull, thr_0 = __ldg(a.thr_cell + cg),
                             thr_p = i + 1 < S.n_x ? __ldg(a.thr_cell + cg + 1) : 0ull;
    const unsigned long long tmax = max(thr_0, max(thr_m, thr_p));
    c.gen = tmax != 0ull;
    c.rej = (uint32_t)(tmax - 1ull);
    auto add = [&](int k, int dd, int v, uint32_t n) {
      if (!COUNT) return;
      if ((unsigned)(br->i + dd) < (unsigned)br->n_x) {
        atomicAdd(br->out + dd * br->n_M + k, v);
      } else {  // (edge cells only)
        atomicAdd(&a.hdr->absorbed, (unsigned long long)n);
        atomicAdd(reinterpret_cast<unsigned long long*>(&a.hdr->absorbed_signed), (unsigned long long)(long long)v);
      }
    };
    walk_ids(
        c, window_of_unit(cell, last - first, w0) << 7, min(last - A, window_of_unit(cell, last - first, w1) << 7),
        lane, queue + kWalkQueue, nq,
        [&](uint32_t q, bool gen, uint4& wr, uint4& wg) {
          wr = make_uint4(qA + q, t - 1u, kPurposeRepos, sim);
          if (gen) {
            wg = make_uint4(qA + q, t, kPurposeGen, sim);
            philox4x32_10_x2(wr, wg, k0, k1);
          } else {
            wr = philox4x32_10(wr, k0, k1);
          }
        },
        [&](int k, uint32_t e, uint32_t stay, uint32_t move) {
          if (stay) add(k, 0, e & 1u ? -(int)stay : (int)stay, stay);
          if (move) add(k, move_dir(e), e & 1u ? -(int)move : (int)move, move);
        },
        [&](unsigned who, bool me, uint32_t q, int k, uint32_t e, uint32_t ids) {
          if (me)
            queue[nq + __popc(who & ((1u << lane) - 1u))] =
                make_uint4(qA + q, (uint32_t)br->cg, (uint32_t)k | ((e & 1u) << 12) | (ids << 16), 0u);
          nq += __popc(who);
        },
        flush);
    if (cell.u1 >= w1) break;
    cell = next_cell(a.U, a.n_cells, cell, lane);
  }
}

__global__ __launch_bounds__(kBStepWarps * 32, 4) void k_b_step(const __grid_constant__ BatchStepArgs a) {
  __shared__ uint4 s_queue[kBStepWarps][kWalkQueue + 32];
  __shared__ BatchRow s_row[kBStepWarps];
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  uint4* queue = s_queue[wid];
  const uint32_t t = a.hdr->step;
  const uint32_t total = a.hdr->n_items ? __ldg(a.U + a.n_cells) : 0u;
  int nq = 0;
  auto flush = [&]() {  // (what does not fit is found again by the pair kernel)
    __syncwarp();
    unsigned qb = 0u;
    if (lane == 0) qb = atomicAdd(&a.hdr->pair_count, (unsigned)nq);
    qb = __shfl_sync(0xffffffffu, qb, 0);
    for (int e = lane; e < nq; e += 32)
      if (qb + (unsigned)e < a.pair_cap) a.pairs[qb + (unsigned)e] = queue[e];
    __syncwarp();
    nq = 0;
  };
  RangeSchedule sched(total, gridDim.x * kBStepWarps, a.max_range, kBSingleRound);
  uint32_t ticket = (uint32_t)wid * gridDim.x + blockIdx.x, w0, w1;
  while (sched.range(ticket, w0, w1)) {
    const bool more = sched.more();
    uint32_t nxt = 0u;
    if (lane == 0 && more) nxt = atomicAdd(&a.hdr->item_ticket, 1u);  // consumed at the end of this range
    b_walk_range<true>(a, t, w0, w1, lane, queue, s_row + wid, nq, flush);
    if (!more) break;
    ticket = sched.n_warps + __shfl_sync(0xffffffffu, nxt, 0);
  }
  if (nq) flush();
  if (blockIdx.x == 0 && threadIdx.x == 0 && a.hdr->n_items > 0) atomicAdd(&a.hdr->particle_steps, a.hdr->population);
}

// All quads that may hold events, by a second walk (they did not fit the queue).
__device__ __noinline__ void b_rewalk_events(const BatchStepArgs& a, uint32_t t, uint4* queue, BatchRow* br, PairCounters& pc) {
  const int lane = threadIdx.x & 31;
  const uint32_t total = a.hdr->n_items ? __ldg(a.U + a.n_cells) : 0u;
  constexpr uint32_t kUnits = 32;
  int nq = 0;
  auto flush = [&]() {
    __syncwarp();
    for (int e = lane; e < nq; e += 32) b_quad_events(a, t, queue[e], pc);
    __syncwarp();
    nq = 0;
  };
  const uint32_t stride = gridDim.x * kBStepWarps * kUnits;
  for (uint32_t w0 = (blockIdx.x * kBStepWarps + (threadIdx.x >> 5)) * kUnits; w0 < total; w0 += stride)
    b_walk_range<false>(a, t, w0, min(w0 + kUnits, total), lane, queue, br, nq, flush);
  if (nq) flush();
}

// The queued quads of the step, by ids or by quads as in the single form.  The last
// block to finish resets the queue and the range ticket for the next step.
__global__ __launch_bounds__(kBStepWarps * 32, 4) void k_b_pairs(const __grid_constant__ BatchStepArgs a) {
  __shared__ uint4 s_queue[kBStepWarps][kWalkQueue + 32];
  __shared__ BatchRow s_row[kBStepWarps];
  __shared__ unsigned long long s_red[3][kBStepWarps];
  const uint32_t t = a.hdr->step;
  const unsigned n = a.hdr->pair_count;
  // (blocks without work leave at once and are not counted)
  const unsigned split = pairs_split(n, gridDim.x * blockDim.x), items = n << split;
  const unsigned blocks = n > a.pair_cap ? gridDim.x : min(gridDim.x, max(1u, (items + blockDim.x - 1) / blockDim.x));
  if (blockIdx.x >= blocks) return;
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  PairCounters pc;
  if (n <= a.pair_cap) {
    for (unsigned e = blockIdx.x * blockDim.x + threadIdx.x; e < items; e += blocks * blockDim.x)
      b_quad_events(a, t, pairs_item(a.pairs, e, split), pc);
  } else {
    b_rewalk_events(a, t, s_queue[wid], s_row + wid, pc);
  }
  const unsigned long long vals[3] = {pc.pairs, pc.dropped, (unsigned long long)pc.drop_signed};
#pragma unroll
  for (int j = 0; j < 3; ++j) {
    unsigned long long v = vals[j];
#pragma unroll
    for (int off = 16; off; off >>= 1) v += __shfl_down_sync(0xffffffffu, v, off);
    if (lane == 0) s_red[j][wid] = v;
  }
  __syncthreads();
  if (threadIdx.x < 3) {
    unsigned long long v = 0;
    for (int w = 0; w < kBStepWarps; ++w) v += s_red[threadIdx.x][w];
    unsigned long long* dst[3] = {&a.hdr->pairs, &a.hdr->dropped,
                                  reinterpret_cast<unsigned long long*>(&a.hdr->dropped_signed)};
    if (v) atomicAdd(dst[threadIdx.x], v);
  }
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

// Start of a run: the step number, and nothing known about the caller's buffers.
__global__ void k_b_set_step(DevHeader* hdr, uint32_t step) {
  hdr->step = step;
  hdr->rows_known = 0u;
}

// ---------------------------------------------------------------- host driver
int b_step_grid() {
  static int cached[8] = {0};
  int dev = 0;
  cudaGetDevice(&dev);
  int& grid = cached[dev & 7];
  if (grid > 0) return grid;
  int per_sm = 0;
  cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_b_step, kBStepWarps * 32, 0);
  if (per_sm < 1) per_sm = 1;
  grid = per_sm * num_sms();
  return grid;
}

cudaError_t b_one_step(const BatchLayout& L, const BatchView& v, int n, const float* V, const int32_t* in,
                       int32_t* out, int per_thread, int grid, cudaStream_t s) {
  const long long nc = L.n_cells;
  const int chunk = 32 * per_thread;  // ids per work item as counted in n_items
  const bool many = nc >= kManyCells;
  const long long row_warps = many ? (nc + kRowsPerWarp - 1) / kRowsPerWarp : nc;
  const unsigned row_blocks = (unsigned)((row_warps * 32 + 255) / 256);
  if (many)
    k_b_rows<kRowsPerWarp><<<row_blocks, 256, 0, s>>>(in, v.descs, v.cell_sim, nc, L.NB, v.T, v.bp, v.nbk, v.reach, out,
                                                      v.row_map, v.hdr);
  else
    k_b_rows<1><<<row_blocks, 256, 0, s>>>(in, v.descs, v.cell_sim, nc, L.NB, v.T, v.bp, v.nbk, v.reach, out, v.row_map,
                                           v.hdr);
  k_b_scan1<<<L.n_blk, kScanThreads, 0, s>>>(v.T, v.reach, v.nbk, v.descs, v.cell_sim, nc, chunk, v.blk);
  k_b_scan2<<<1, kScanThreads, 0, s>>>(v.blk, L.n_blk, L.max_items, v.hdr, 1);
  k_b_scan3<<<L.n_blk, kScanThreads, 0, s>>>(v.T, v.reach, v.nbk, v.descs, v.cell_sim, nc, chunk, v.blk, v.G, v.U, v.occ,
                                             v.row_map, v.thr_cell, v.hdr);
  k_b_simbase<<<(n + 127) / 128, 128, 0, s>>>(v.descs, n, v.G, v.sim_base, v.hdr);
  const int rows_blocks = (int)((nc + kBatchRowWarps - 1) / kBatchRowWarps);
  const int rb = rows_blocks < 8 * num_sms() ? rows_blocks : 8 * num_sms();
  auto rows = [&](auto live) {
    constexpr bool LIVE = decltype(live)::value;
    const auto k = L.H <= 32 ? k_b_kernel_rows<1, LIVE> : (L.H <= 64 ? k_b_kernel_rows<2, LIVE> : k_b_kernel_rows<4, LIVE>);
    k<<<rb, kBatchRowWarps * 32, 0, s>>>(V, v.descs, v.cell_sim, v.occ, v.live, v.hdr, v.sine, L.NM, v.cdf, v.thr_cell);
  };
  if (many) {
    const int live_blocks = (int)((nc + 255) / 256);
    k_b_live<<<live_blocks < rb ? live_blocks : rb, 256, 0, s>>>(V, v.descs, v.cell_sim, v.occ, v.live, v.hdr);
    rows(std::true_type{});
  } else {
    rows(std::false_type{});
  }
  BatchStepArgs a;
  a.hist_in = in;
  a.hist_out = out;
  a.d = v.descs;
  a.cell_sim = v.cell_sim;
  a.G = v.G;
  a.sim_base = v.sim_base;
  a.U = v.U;
  a.bp = v.bp;
  a.row_map = v.row_map;
  a.cdf = v.cdf;
  a.thr_cell = v.thr_cell;
  a.xm = v.xm;
  a.pairs = v.pairs;
  a.pair_cap = L.pair_cap;
  a.hdr = v.hdr;
  a.NM = L.NM;
  a.NB = L.NB;
  a.n_cells = (int)nc;
  a.max_range = batch_max_range(per_thread);
  k_b_step<<<grid, kBStepWarps * 32, 0, s>>>(a);
  const unsigned pair_blocks = (L.pair_cap + kBStepWarps * 32 - 1) / (kBStepWarps * 32);
  const unsigned pair_most = 8u * (unsigned)num_sms();
  k_b_pairs<<<pair_blocks < pair_most ? pair_blocks : pair_most, kBStepWarps * 32, 0, s>>>(a);
  return cudaGetLastError();
}

// Executable graphs of the step pair a -> b -> a for the last few
// configurations used, as in the single form: a caller that goes from one batch
// to another and back does not recapture (a pass over 58 small simulations,
// three batches in turn: most of its 430 us was capture and instantiation).
constexpr int kBatchGraphs = 4;
struct BatchGraphKey {
  std::vector<wmc_params> ps;
  const void *V = nullptr, *a = nullptr, *b = nullptr, *ws = nullptr;
  int per = 0;
  cudaStream_t stream = nullptr;
};
struct BatchGraphs {
  std::mutex mu;
  GraphSlots<BatchGraphKey, cudaGraphExec_t, kBatchGraphs> slots;
};
BatchGraphs g_bgraph;

}  // namespace
}  // namespace wmc

using namespace wmc;

extern "C" {

size_t wmc_batch_workspace_size(const wmc_params* ps, int32_t n_sims) {
  if (!batch_ok(ps, n_sims)) return 0;
  return batch_layout(ps, n_sims).total;
}

wmc_status wmc_batch_layout(const wmc_params* ps, int32_t n_sims, int64_t* cell_off, int64_t* hist_off) {
  if (!batch_ok(ps, n_sims) || !cell_off || !hist_off) return WMC_ERR_ARG;
  long long c = 0, h = 0;
  for (int s = 0; s < n_sims; ++s) {
    cell_off[s] = c;
    hist_off[s] = h;
    c += ps[s].n_x;
    h += (long long)ps[s].n_x * ps[s].n_M;
  }
  cell_off[n_sims] = c;
  hist_off[n_sims] = h;
  return WMC_OK;
}

wmc_status wmc_batch_init(const wmc_params* ps, int32_t n_sims, void* ws, size_t ws_bytes, wmc_stream_t stream) {
  if (!batch_ok(ps, n_sims) || !ws || ((uintptr_t)ws & 255)) return WMC_ERR_ARG;
  const BatchLayout L = batch_layout(ps, n_sims);
  if (ws_bytes < L.total) return WMC_ERR_ARG;
  std::vector<SimDesc> d(n_sims);
  long long c = 0, h = 0, tb = 0, sn = 0;
  for (int s = 0; s < n_sims; ++s) {
    const wmc_params& p = ps[s];
    SimDesc& x = d[s];
    memset(&x, 0, sizeof(x));
    x.n_x = p.n_x;
    x.Q = p.Q;
    x.n_M = p.n_M;
    x.bc = p.bc_potential;
    x.wrap = p.child_wrap;
    x.h = p.Q / 2;
    x.log2_nM = ceil_log2_host(p.n_M);
    x.Kp = ((x.h - 1 + 31) / 32) * 32 > 0 ? ((x.h - 1 + 31) / 32) * 32 : 32;
    x.Np = ((x.h + 63) / 64) * 64;
    x.sim = p.sim;
    x.k0 = (uint32_t)(p.seed & 0xffffffffu);
    x.k1 = (uint32_t)(p.seed >> 32);
    x.c = (float)(-2.0 / (kHbarEVs * (double)p.Q));
    x.dt = p.dt_s;
    x.d1 = ((kHbarJs * kPi) * p.dt_s) / ((p.mass_kg * (double)p.Q) * (p.dx_m * p.dx_m));
    x.cell_off = c;
    x.hist_off = h;
    x.tab_off = tb;
    x.sine_off = sn;
    c += p.n_x;
    h += (long long)p.n_x * p.n_M;
    tb += p.n_M;
    sn += (long long)x.Kp * x.Np;
  }
  const BatchView v = batch_view(L, ws);
  cudaStream_t s = (cudaStream_t)stream;
  // set-up copy of the descriptors (synchronous: the host vector is temporary)
  if (cudaMemcpyAsync(v.descs, d.data(), sizeof(SimDesc) * n_sims, cudaMemcpyHostToDevice, s) != cudaSuccess)
    return WMC_ERR_CUDA;
  if (cudaStreamSynchronize(s) != cudaSuccess) return WMC_ERR_CUDA;
  k_b_init<<<512, 256, 0, s>>>(v.descs, n_sims, L.n_cells, L.tab_elems, L.sine_elems, v.cell_sim, v.xm, v.sine,
                               v.hdr);
  (void)b_step_grid();
  return cudaGetLastError() == cudaSuccess ? WMC_OK : WMC_ERR_CUDA;
}

wmc_status wmc_batch_run(const wmc_params* ps, int32_t n_sims, const float* V, int32_t* hist_a, int32_t* hist_b,
                         uint32_t t_first, int32_t n_steps, int32_t per_thread, int32_t use_graph, void* ws,
                         wmc_stream_t stream) {
  NvtxRange nvtx("wmc_batch_run");
  if (!batch_ok(ps, n_sims) || !V || !hist_a || !hist_b || hist_a == hist_b || !ws || n_steps < 0 || t_first == 0)
    return WMC_ERR_ARG;
  if (per_thread == 0) per_thread = 16;
  if (!valid_per_thread(per_thread)) return WMC_ERR_ARG;
  if (n_steps == 0) return WMC_OK;
  const BatchLayout L = batch_layout(ps, n_sims);
  const BatchView v = batch_view(L, ws);
  cudaStream_t s = (cudaStream_t)stream;
  const int grid = b_step_grid();
  k_b_set_step<<<1, 1, 0, s>>>(v.hdr, t_first - 1u);
  if (cudaGetLastError() != cudaSuccess) return WMC_ERR_CUDA;
  const int pairs = n_steps / 2;
  if (use_graph && s != nullptr && pairs > 0) {
    std::lock_guard<std::mutex> lock(g_bgraph.mu);
    int dev = 0;
    cudaGetDevice(&dev);
    const unsigned long long ctx = current_context_id();
    auto* hit = g_bgraph.slots.find(dev, ctx, [&](const BatchGraphKey& k) {
      return (int)k.ps.size() == n_sims && k.V == V && k.a == hist_a && k.b == hist_b && k.ws == ws &&
             k.per == per_thread && k.stream == s && memcmp(k.ps.data(), ps, sizeof(wmc_params) * n_sims) == 0;
    });
    if (!hit) {
      auto& slot = g_bgraph.slots.take([](cudaGraphExec_t e) { cudaGraphExecDestroy(e); });
      cudaGraph_t graph = nullptr;
      if (cudaStreamBeginCapture(s, cudaStreamCaptureModeThreadLocal) != cudaSuccess) return WMC_ERR_CUDA;
      cudaError_t e = b_one_step(L, v, n_sims, V, hist_a, hist_b, per_thread, grid, s);
      if (e == cudaSuccess) e = b_one_step(L, v, n_sims, V, hist_b, hist_a, per_thread, grid, s);
      const cudaError_t e2 = cudaStreamEndCapture(s, &graph);
      if (e != cudaSuccess || e2 != cudaSuccess) {
        if (graph) cudaGraphDestroy(graph);
        return WMC_ERR_CUDA;
      }
      cudaGraphExec_t exec = nullptr;
      e = cudaGraphInstantiate(&exec, graph, 0);
      cudaGraphDestroy(graph);
      if (e != cudaSuccess) return WMC_ERR_CUDA;
      hit = g_bgraph.slots.fill(slot, BatchGraphKey{{ps, ps + n_sims}, V, hist_a, hist_b, ws, per_thread, s}, exec, dev, ctx);
    }
    for (int q = 0; q < pairs; ++q)
      if (cudaGraphLaunch(hit->exec, s) != cudaSuccess) return WMC_ERR_CUDA;
  } else {
    for (int q = 0; q < pairs; ++q) {
      if (b_one_step(L, v, n_sims, V, hist_a, hist_b, per_thread, grid, s) != cudaSuccess) return WMC_ERR_CUDA;
      if (b_one_step(L, v, n_sims, V, hist_b, hist_a, per_thread, grid, s) != cudaSuccess) return WMC_ERR_CUDA;
    }
  }
  if (n_steps & 1) {
    if (b_one_step(L, v, n_sims, V, hist_a, hist_b, per_thread, grid, s) != cudaSuccess) return WMC_ERR_CUDA;
    if (cudaMemcpyAsync(hist_a, hist_b, sizeof(int32_t) * (size_t)L.hist_elems, cudaMemcpyDeviceToDevice, s) !=
        cudaSuccess)
      return WMC_ERR_CUDA;
  }
  return WMC_OK;
}

wmc_status wmc_batch_autotune(const wmc_params* ps, int32_t n_sims, const float* V, int32_t* hist, int32_t* scratch,
                              uint32_t t, void* ws, int32_t* best_per_thread, wmc_stream_t stream) {
  if (!batch_ok(ps, n_sims) || !V || !hist || !scratch || hist == scratch || !ws || !best_per_thread || t == 0)
    return WMC_ERR_ARG;
  const BatchLayout L = batch_layout(ps, n_sims);
  const BatchView v = batch_view(L, ws);
  cudaStream_t s = (cudaStream_t)stream;
  const int grid = b_step_grid();
  cudaEvent_t e0, e1;
  if (cudaEventCreate(&e0) != cudaSuccess || cudaEventCreate(&e1) != cudaSuccess) return WMC_ERR_CUDA;
  float best = 1e30f;
  int best_per = kTuneCandidates[0];
  for (int r = 0; r < 2; ++r) {  // second round measures warm
    for (const int per : kTuneCandidates) {
      k_b_set_step<<<1, 1, 0, s>>>(v.hdr, t - 1u);
      cudaEventRecord(e0, s);
      if (b_one_step(L, v, n_sims, V, hist, scratch, per, grid, s) != cudaSuccess) return WMC_ERR_CUDA;
      cudaEventRecord(e1, s);
      if (cudaEventSynchronize(e1) != cudaSuccess) return WMC_ERR_CUDA;
      float ms = 0.f;
      cudaEventElapsedTime(&ms, e0, e1);
      if (r == 1 && ms < best) {
        best = ms;
        best_per = per;
      }
    }
  }
  cudaEventDestroy(e0);
  cudaEventDestroy(e1);
  *best_per_thread = best_per;
  return WMC_OK;
}

wmc_status wmc_batch_get_counters(const wmc_params* ps, int32_t n_sims, const void* ws, wmc_counters* out,
                                  wmc_stream_t stream) {
  if (!batch_ok(ps, n_sims) || !ws || !out) return WMC_ERR_ARG;
  const BatchLayout L = batch_layout(ps, n_sims);
  DevHeader h;
  const char* b = static_cast<const char*>(ws);
  cudaError_t e = cudaMemcpyAsync(&h, b + L.header, sizeof(h), cudaMemcpyDeviceToHost, (cudaStream_t)stream);
  if (e == cudaSuccess) e = cudaStreamSynchronize((cudaStream_t)stream);
  if (e != cudaSuccess) return WMC_ERR_CUDA;
  out->population = h.population;
  out->particle_steps = h.particle_steps;
  out->pairs = h.pairs;
  out->absorbed = h.absorbed;
  out->absorbed_signed = h.absorbed_signed;
  out->dropped = h.dropped;
  out->dropped_signed = h.dropped_signed;
  out->n_occ = h.n_occ;
  out->n_items = h.n_items;
  out->flags = h.flags;
  out->step = h.step;
  return h.magic == kMagic ? WMC_OK : WMC_ERR_ARG;
}

}  // extern "C"

// The trained N = 2 network of Sec. 2.3: Eq. (kernel_ML) with N = 2 (one cosine
// factor), its weights learnt by stochastic gradient descent on a
// mean-squared-error loss against exact kernels, one example per step.
//
// Reduced units (kernels times hbar Q / 2, V in eV):
//   y(i, j) = cos(pi j / Q) sum_{d in D(i)} W[d] (wv1 V(i + d) + wv2 V(i + d + 1))
//                                         sin(2 pi j / Q (wt1 d + wt2 (d + 1))),
// D(i) = {d in [-h, h - 1] : i + d even}: the absolute cell pairs (2q, 2q + 1),
// 2q = i + d, inside the window [i - h, i + h]; W indexed by d + h.  The
// parameters are one vector [W[0 .. Q-1], wv1, wv2, wt1, wt2]; at W = -1,
// wv = (1, 1), wt = (1/2, 1/2) the model is the analytic N = 2 network.
//
// Loss of one example: mean over i in [0, n_x), j in [1, h) of (y - t)^2;
// gradient, with G(i, d) = sum_j dL/dy c_j sin(.), H(i, d) = sum_j dL/dy c_j
// phi_j cos(.), phi_j = 2 pi j / Q, P = wv1 V(i+d) + wv2 V(i+d+1):
//   dW[d] = sum_i P G,  dwv1 = sum W V(i+d) G,  dwv2 = sum W V(i+d+1) G,
//   dwt1 = sum W P H d, dwt2 = sum W P H (d + 1).
//
// k_n2_train: one cluster of CTAs per training run (runs differ in learning
// rate; they train on the same examples in the same order), the whole SGD loop
// inside it.  The rows of an example are cut into up to eight parts, by n_x
// alone, and the parts shared out over the CTAs; each CTA builds the phase tables
// (sincospif of the current wt) for itself, its residuals and its share of the
// gradient; the shares are exchanged through distributed shared memory with one
// cluster barrier per step and every CTA adds them, so all of them make the same
// update.  Every sum is taken within a part and then over the parts in pairs, in
// an order that does not depend on the number of CTAs: a run's result is the same
// beside any other runs and on any GPU.
// k_n2_eval: the trained model's rows, in 1/s, for given parameters.
#include <cooperative_groups.h>

#include "wmc_device.cuh"

namespace wmc {

namespace {

constexpr float kPiF = 3.14159265358979f;  // pi rounded to FP32
constexpr int kN2Threads = 512;
constexpr int kN2Warps = kN2Threads / 32;
constexpr int kN2MaxParts = 8;  // parts of the rows, and CTAs of a cluster

// Parts of the rows: as many as hold four row pairs each.
__host__ __device__ inline int n2_parts(int n_x) {
  int P = 1;
  while (2 * P <= kN2MaxParts && n_x / 2 >= 4 * 2 * P) P *= 2;
  return P;
}

// Sizes of k_n2_train with the rows over C CTAs.  Rows and pair offsets are
// held by parity (row i meets the offsets dd = d + h of parity (i + h) mod 2):
// G groups of four row pairs, part c of P the groups [G c / P, G (c + 1) / P), up
// to Mp row pairs per CTA, and h offsets padded to hp, a multiple of four, for
// 16-byte loads.
struct N2Shape {
  int h, hp, G, Mp, parts;  // parts: of one CTA
  __host__ __device__ N2Shape(int n_x, int Q, int C)
      : h(Q / 2), hp((Q / 2 + 3) & ~3), G((n_x / 2 + 3) / 4), Mp(4 * ((G + C - 1) / C)), parts(n2_parts(n_x) / C) {}
  // sin and phi-weighted cos tables [h][2][hp]; W P [h][2][Mp], later the sums of
  // the groups, [Mp / 4][2][hp] of the W gradient and as many of the other four;
  // residuals [2][h][Mp]; V of the rows' windows; cos(pi j / Q); parameters; the
  // exchanged sums, two buffers; the loss of the groups [Mp / 4][2][hp / 4]
  __host__ __device__ size_t table() const { return (size_t)h * 2 * hp; }
  __host__ __device__ size_t rows() const { return (size_t)h * 2 * Mp; }
  __host__ __device__ size_t window() const { return (size_t)2 * Mp + 2 * h + 4; }
  __host__ __device__ size_t exchanged() const { return (size_t)2 * h + 5 * parts; }
  __host__ __device__ size_t losses() const { return (size_t)(Mp / 4) * 2 * (hp / 4); }
  __host__ __device__ size_t floats() const {
    return 2 * table() + 2 * rows() + ((window() + 3) & ~(size_t)3) + hp + (2 * h + 4) + 2 * exchanged() + losses();
  }
};

// Sum over the parts in pairs (entries past the last are zero): the sum of
// aligned runs of parts, then of the runs' sums, is the same sum.
__device__ __forceinline__ float n2_pairwise(float (&x)[kN2MaxParts]) {
#pragma unroll
  for (int w = 1; w < kN2MaxParts; w *= 2)
#pragma unroll
    for (int c = 0; c < kN2MaxParts; c += 2 * w) x[c] += x[c + w];
  return x[0];
}

__device__ __forceinline__ float n2_pot(const float* __restrict__ V, int n_x, int bc, int l) {
  if (l >= 0 && l < n_x) return __ldg(V + l);
  if (!bc) return 0.f;
  return __ldg(V + (l < 0 ? 0 : n_x - 1));
}

}  // namespace

// A thread's tile is 4 rows (of one parity) x 4 columns of the residuals, then
// 4 rows x 4 offsets of the gradient sums: 16 and 32 FMAs for 5 and 3 loads of
// shared memory (one load per FMA, 40 k shared-memory cycles a step, bound the
// form with one output per thread at 36 us a step on one SM).  256 cells, Q =
// 64, three runs: 6.9 us a step with eight CTAs per run.  There a CTA has 64
// tiles, so two of its sixteen warps do the residuals and the gradient sums, with
// little to hide their latency: by clock stamps 2800 and 4500 of 14600 cycles a
// step, the tables 2800, W P 1500, the sums and their exchange 3000.  152 runs
// of one CTA each: 20.8 us a step (19.8 with sums whose order followed the
// number of CTAs).
__global__ __launch_bounds__(kN2Threads) void k_n2_train(int n_x, int Q, int bc, int n_ex, const float* __restrict__ Vs,
                                                          const float* __restrict__ VW, float scale, int epochs,
                                                          const int* __restrict__ order, const float* __restrict__ lr,
                                                          float* __restrict__ params, float* __restrict__ loss_out) {
  namespace cg = cooperative_groups;
  extern __shared__ __align__(16) float sm_n2[];
  cg::cluster_group cluster = cg::this_cluster();
  const int C = (int)cluster.num_blocks(), rank = (int)cluster.block_rank();
  const int run = blockIdx.x / C;
  const N2Shape z(n_x, Q, C);
  // exchanged sums: dW, then dwv, dwt and the loss of each of the CTA's parts
  const int h = z.h, hp = z.hp, Mp = z.Mp, n_parts = z.parts, NV = (int)z.exchanged();
  const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
  float* sS = sm_n2;              // [h][2][hp]: sin of offset dd (parity, dd / 2) at column j
  float* sC = sS + z.table();     // phi_j times the cosines
  float* sWP = sC + z.table();    // [h][2][Mp]: W P of pair k of the rows of each parity
  float* sR = sWP + z.rows();     // [2][h][Mp]: residuals times (2 / n_out) cos(pi j / Q)
  float* sV = sR + z.rows();      // V(i0 - h + q)
  float* sCJ = sV + ((z.window() + 3) & ~(size_t)3);
  float* sP = sCJ + hp;           // parameters
  float* sX = sP + (Q + 4);       // exchanged sums, by step parity
  float* sL = sX + 2 * NV;        // the groups' losses
  // this CTA's groups of row pairs, its row pairs and its first row
  const int g0 = (int)((long long)z.G * rank / C), RG = (int)((long long)z.G * (rank + 1) / C) - g0;
  const int m_n = min(4 * RG, n_x / 2 - 4 * g0), i0 = 8 * g0;
  float* sGp = sWP;               // the W gradient of the groups, once W P has been used
  // their sums for dwv1, dwv2, dwt1, dwt2 (one column: in the place of the residuals, which no sum reads)
  float* sG4 = h > 1 ? sGp + (size_t)RG * 2 * hp : sR;
  // first group of each of the CTA's parts (and the end of the last), and log2 of their number
  __shared__ int s_first[kN2MaxParts + 1];
  if (tid <= n_parts) s_first[tid] = (int)((long long)z.G * (rank * n_parts + tid) / (C * n_parts)) - g0;
  const int log_parts = __ffs(n_parts) - 1;
  const float rate = __ldg(lr + run);
  float* prm = params + (size_t)run * (Q + 4);
  for (int q = tid; q < Q + 4; q += kN2Threads) sP[q] = prm[q];
  for (int j = tid; j < h; j += kN2Threads) sCJ[j] = cospif((float)j / (float)Q);
  for (size_t q = tid; q < 2 * z.table(); q += kN2Threads) sS[q] = 0.f;  // (the padding stays zero)
  const float inv_n = 2.f / (float)((long long)n_x * (h - 1));  // d(mean of squares)/dy = inv_n r
  const int JG = hp / 4;  // groups of four columns or offsets
  const int n_tasks = 2 * RG * JG;
  __syncthreads();
  int step = 0;
  // what the rounding of this thread's parameter has left out so far in this call
  // (the sizes that are accepted have Q <= 222, so a thread holds one at most).
  // 300 steps of 256 cells, Q = 64: parameters 4.4e-7 -> 2e-8 from FP64, no time.
  float low = 0.f;
  for (int ep = 0; ep < epochs; ++ep) {
    float ep_loss = 0.f;
    for (int s = 0; s < n_ex; ++s, ++step) {
      const int ex = __ldg(order + (size_t)ep * n_ex + s);
      const float* V = Vs + (size_t)ex * n_x;
      const float* T = VW + (size_t)ex * n_x * h;
      const float wv1 = sP[Q], wv2 = sP[Q + 1], wt1 = sP[Q + 2], wt2 = sP[Q + 3];
      // phase tables of the current wt, the potential and W P
      for (int q = tid; q < 2 * m_n + 2 * h + 1; q += kN2Threads) sV[q] = n2_pot(V, n_x, bc, i0 - h + q);
      for (int q = tid; q < Q * h; q += kN2Threads) {
        const int j = q / Q, dd = q % Q, d = dd - h;
        float sv, cv;
        sincospif(2.f * (float)j / (float)Q * (wt1 * (float)d + wt2 * (float)(d + 1)), &sv, &cv);
        const size_t at = ((size_t)j * 2 + (dd & 1)) * hp + (dd >> 1);
        sS[at] = sv;
        sC[at] = cv * (2.f * (float)j / (float)Q) * kPiF;
      }
      __syncthreads();
      for (int q = tid; q < h * 2 * Mp; q += kN2Threads) {  // pair k of row i0 + 2 m + p
        const int m = q % Mp, p = (q / Mp) & 1, k = q / (2 * Mp);
        const int dd = 2 * k + ((i0 + p + h) & 1), at = 2 * m + p + dd;  // sV[at] = V(i + d)
        sWP[q] = m < m_n ? sP[dd] * fmaf(wv1, sV[at], wv2 * sV[at + 1]) : 0.f;
      }
      __syncthreads();
      // residuals
      for (int t = tid; t < n_tasks; t += kN2Threads) {
        const int rg = t % RG, jg = (t / RG) % JG, p = t / (RG * JG);
        const int pd = (i0 + p + h) & 1;  // parity of the rows' offsets
        float tv[4][4];  // targets, asked for before the sums
#pragma unroll
        for (int b = 0; b < 4; ++b)
#pragma unroll
          for (int a = 0; a < 4; ++a) {
            const int m = 4 * rg + a, j = 4 * jg + b;
            tv[a][b] = m < m_n && j < h ? __ldg(T + (size_t)(i0 + 2 * m + p) * h + j) : 0.f;
          }
        float acc[4][4];
#pragma unroll
        for (int a = 0; a < 4; ++a)
#pragma unroll
          for (int b = 0; b < 4; ++b) acc[a][b] = 0.f;
        const float* wp = sWP + (size_t)p * Mp + 4 * rg;
        const float* st = sS + (size_t)pd * hp;
        int jb[4];
#pragma unroll
        for (int b = 0; b < 4; ++b) jb[b] = min(4 * jg + b, h - 1) * 2 * hp;
#pragma unroll 4
        for (int k = 0; k < h; ++k) {
          const float4 w4 = *reinterpret_cast<const float4*>(wp + (size_t)k * 2 * Mp);
          const float wa[4] = {w4.x, w4.y, w4.z, w4.w};
#pragma unroll
          for (int b = 0; b < 4; ++b) {
            const float sv = st[jb[b] + k];
#pragma unroll
            for (int a = 0; a < 4; ++a) acc[a][b] = fmaf(wa[a], sv, acc[a][b]);
          }
        }
        float part = 0.f;
#pragma unroll
        for (int b = 0; b < 4; ++b) {
          const int j = 4 * jg + b;
          if (j < h) {
            float4 r4;
            float* rv = reinterpret_cast<float*>(&r4);
            const float cj = sCJ[j];
#pragma unroll
            for (int a = 0; a < 4; ++a) {
              const float r = j > 0 && 4 * rg + a < m_n ? fmaf(cj, acc[a][b], -tv[a][b] * scale) : 0.f;
              part = fmaf(r, r, part);
              rv[a] = r * cj * inv_n;
            }
            *reinterpret_cast<float4*>(sR + ((size_t)p * h + j) * Mp + 4 * rg) = r4;
          }
        }
        sL[(rg * 2 + p) * JG + jg] = part;
      }
      __syncthreads();
      // gradient sums of 4 rows x 4 offsets
      for (int t = tid; t < n_tasks; t += kN2Threads) {
        const int rg = t % RG, dg = (t / RG) % JG, p = t / (RG * JG);
        const int pd = (i0 + p + h) & 1;
        float G[4][4], H[4][4];
#pragma unroll
        for (int a = 0; a < 4; ++a)
#pragma unroll
          for (int b = 0; b < 4; ++b) G[a][b] = H[a][b] = 0.f;
        const float* rp = sR + (size_t)p * h * Mp + 4 * rg;
        const size_t tb = (size_t)pd * hp + 4 * dg;
#pragma unroll 2
        for (int j = 1; j < h; ++j) {
          const float4 r4 = *reinterpret_cast<const float4*>(rp + (size_t)j * Mp);
          const float4 s4 = *reinterpret_cast<const float4*>(sS + tb + (size_t)j * 2 * hp);
          const float4 c4 = *reinterpret_cast<const float4*>(sC + tb + (size_t)j * 2 * hp);
          const float ra[4] = {r4.x, r4.y, r4.z, r4.w}, sb[4] = {s4.x, s4.y, s4.z, s4.w}, cb[4] = {c4.x, c4.y, c4.z, c4.w};
#pragma unroll
          for (int a = 0; a < 4; ++a)
#pragma unroll
            for (int b = 0; b < 4; ++b) {
              G[a][b] = fmaf(ra[a], sb[b], G[a][b]);
              H[a][b] = fmaf(ra[a], cb[b], H[a][b]);
            }
        }
        float4 g4;
        float* gw = reinterpret_cast<float*>(&g4);
        float gv1 = 0.f, gv2 = 0.f, gt1 = 0.f, gt2 = 0.f;
#pragma unroll
        for (int b = 0; b < 4; ++b) {
          const int dd = 2 * (4 * dg + b) + pd, d = dd - h;
          gw[b] = 0.f;
          if (4 * dg + b < h) {
            const float Wd = sP[dd];
#pragma unroll
            for (int a = 0; a < 4; ++a) {
              const int m = 4 * rg + a;
              if (m < m_n) {
                const float Va = sV[2 * m + p + dd], Vb = sV[2 * m + p + dd + 1];
                const float P = fmaf(wv1, Va, wv2 * Vb);
                gw[b] = fmaf(P, G[a][b], gw[b]);
                gv1 = fmaf(Wd * Va, G[a][b], gv1);
                gv2 = fmaf(Wd * Vb, G[a][b], gv2);
                gt1 = fmaf(Wd * P * H[a][b], (float)d, gt1);
                gt2 = fmaf(Wd * P * H[a][b], (float)(d + 1), gt2);
              }
            }
          }
        }
        // (each offset belongs to one row parity, so a slot has one writer)
        *reinterpret_cast<float4*>(sGp + ((size_t)rg * 2 + pd) * hp + 4 * dg) = g4;
        *reinterpret_cast<float4*>(sG4 + ((size_t)rg * 2 + pd) * hp + 4 * dg) = make_float4(gv1, gv2, gt1, gt2);
      }
      __syncthreads();
      // this CTA's sums: dW over its parts, an offset per thread, and the other
      // five of each part by one warp
      float* mine = sX + (step & 1) * NV;
      if (const int q = tid; q < Q) {
        const float* gp = sGp + (size_t)(q & 1) * hp + (q >> 1);
        float v = 0.f, s1 = 0.f, s2 = 0.f, s4 = 0.f;  // runs of one, two and four parts waiting for their neighbours
        int rg = 0;
#pragma unroll 1
        for (int c = 0; c < n_parts; ++c) {
          v = 0.f;
#pragma unroll 4
          for (const int end = s_first[c + 1]; rg < end; ++rg) v += gp[(size_t)rg * 2 * hp];
          if (!(c & 1)) {
            s1 = v;
            continue;
          }
          v = s1 + v;
          if (!(c & 2)) {
            s2 = v;
            continue;
          }
          v = s2 + v;
          if (!(c & 4)) s4 = v;
          else v = s4 + v;
        }
        mine[q] = v;
      }
      if (const int c = kN2Warps - 1 - wid; c < n_parts) {
        float v5[5] = {0.f, 0.f, 0.f, 0.f, 0.f};
        for (int e = s_first[c] * 2 * JG + lane; e < s_first[c + 1] * 2 * JG; e += 32) {
          const float4 v = *reinterpret_cast<const float4*>(sG4 + 4 * e);
          v5[0] += v.x, v5[1] += v.y, v5[2] += v.z, v5[3] += v.w, v5[4] += sL[e];
        }
#pragma unroll
        for (int off = 16; off > 0; off >>= 1)
#pragma unroll
          for (int u = 0; u < 5; ++u) v5[u] += __shfl_down_sync(0xffffffffu, v5[u], off);
        if (lane == 0)
          for (int u = 0; u < 5; ++u) mine[Q + 5 * c + u] = v5[u];
      }
      // every CTA's sums are there; the other buffer serves the next step, so
      // that no CTA overwrites sums another still reads
      if (C > 1) cluster.sync();
      else __syncthreads();
      if (const int q = tid; q < Q + 5) {
        // dW from every CTA, the others from every part; without branches, so that
        // all loads are under way before the first sum (700 cycles a step otherwise)
        float x[kN2MaxParts];
        const int n = q < Q ? C : C * n_parts, shift = q < Q ? 0 : log_parts;
#pragma unroll
        for (int c = 0; c < kN2MaxParts; ++c) {
          const int u = min(c, n - 1);
          x[c] = *(cluster.map_shared_rank(mine, u >> shift) + q + 5 * (u & ((1 << shift) - 1)));
        }
#pragma unroll
        for (int c = 0; c < kN2MaxParts; ++c) x[c] = c < n ? x[c] : 0.f;
        const float v = n2_pairwise(x);
        if (q < Q + 4) {
          const float old = sP[q], up = fmaf(-rate, v, low);
          const float now = __fadd_rn(old, up), d = __fsub_rn(now, old);
          sP[q] = now;
          low = __fadd_rn(__fsub_rn(old, __fsub_rn(now, d)), __fsub_rn(up, d));
        } else {
          ep_loss += v * (0.5f * inv_n);
        }
      }
      __syncthreads();
    }
    if (rank == 0 && tid == Q + 4 && loss_out) loss_out[(size_t)run * epochs + ep] = ep_loss / (float)n_ex;
  }
  if (rank == 0)
    for (int q = tid; q < Q + 4; q += kN2Threads) prm[q] = sP[q];
  if (C > 1) cluster.sync();  // no CTA leaves while another reads its shared memory
}

// Rows of the trained model in 1/s: row = potential b, cell i (b n_x + i),
// columns j = 0 .. h - 1; one block per row group stages the phase tables.
__global__ __launch_bounds__(256) void k_n2_eval(int n_x, int Q, int bc, long long rows, const float* __restrict__ V,
                                                 const float* __restrict__ prm, float inv_scale,
                                                 float* __restrict__ out) {
  extern __shared__ float sm_e[];
  const int h = Q / 2;
  float* sS = sm_e;            // [Q][h]
  float* sP = sS + (size_t)Q * h;
  for (int q = threadIdx.x; q < Q + 4; q += blockDim.x) sP[q] = __ldg(prm + q);
  __syncthreads();
  const float wv1 = sP[Q], wv2 = sP[Q + 1], wt1 = sP[Q + 2], wt2 = sP[Q + 3];
  for (int q = threadIdx.x; q < Q * h; q += blockDim.x) {
    const int d = q / h - h, j = q % h;
    sS[q] = sinpif(2.f * (float)j / (float)Q * (wt1 * (float)d + wt2 * (float)(d + 1)));
  }
  __syncthreads();
  const long long total = rows * h;
  for (long long q = blockIdx.x * (long long)blockDim.x + threadIdx.x; q < total;
       q += (long long)gridDim.x * blockDim.x) {
    const long long row = q / h;
    const int j = (int)(q % h), i = (int)(row % n_x);
    const float* Vb = V + (size_t)(row / n_x) * n_x;
    float acc = 0.f;
    const int d0 = ((i - h) & 1) == 0 ? -h : -h + 1;
    for (int k = 0; k < h; ++k) {
      const int d = d0 + 2 * k;
      const float P = fmaf(wv1, n2_pot(Vb, n_x, bc, i + d), wv2 * n2_pot(Vb, n_x, bc, i + d + 1));
      acc = fmaf(sP[d + h] * P, sS[(d + h) * h + j], acc);
    }
    out[q] = j ? cospif((float)j / (float)Q) * acc * inv_scale : 0.f;
  }
}

}  // namespace wmc

using namespace wmc;

extern "C" {

wmc_status wmc_n2_train(const wmc_params* p, int32_t n_examples, const float* V, const float* VW, int32_t epochs,
                        const int32_t* order, int32_t n_runs, const float* lr, float* params, float* loss,
                        wmc_stream_t stream) {
  if (!params_ok(p) || n_examples <= 0 || epochs < 0 || n_runs < 0 || !V || !VW || !order || !lr || !params)
    return WMC_ERR_ARG;
  if (p->n_x % 2 != 0) return WMC_ERR_ARG;
  // the sizes one CTA's shared memory holds with whole tables and rows
  const size_t h = (size_t)p->Q / 2;
  if (sizeof(float) * (2 * (size_t)p->Q * h + 2 * (size_t)p->n_x * h + (size_t)(p->n_x + p->Q + 2) + h +
                       (size_t)(2 * p->Q + 4) + 192) > 200 * 1024)
    return WMC_ERR_UNSUPPORTED;
  if (n_runs == 0 || epochs == 0) return WMC_OK;
  // CTAs per run: as many as the SMs hold for all runs, with at least one part each
  int C = 1;
  while (2 * C <= n2_parts(p->n_x) && (long long)n_runs * 2 * C <= num_sms()) C *= 2;
  const size_t sm = sizeof(float) * N2Shape(p->n_x, p->Q, C).floats();
  if (sm > 48 * 1024 && raise_smem_limit(reinterpret_cast<const void*>(k_n2_train), sm) != cudaSuccess)
    return WMC_ERR_CUDA;
  const float scale = (float)(kHbarEVs * (double)p->Q / 2.0);
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)(n_runs * C));
  cfg.blockDim = dim3(kN2Threads);
  cfg.dynamicSmemBytes = sm;
  cfg.stream = (cudaStream_t)stream;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = (unsigned)C;
  at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, k_n2_train, p->n_x, p->Q, p->bc_potential, n_examples, V, VW, scale, epochs, order, lr,
                            params, loss) == cudaSuccess
             ? WMC_OK
             : WMC_ERR_CUDA;
}

wmc_status wmc_n2_eval(const wmc_params* p, const float* params, const float* V, int32_t n_pot, float* VWh,
                       wmc_stream_t stream) {
  if (!params_ok(p) || !params || !V || !VWh || n_pot < 0) return WMC_ERR_ARG;
  const long long rows = (long long)n_pot * p->n_x;
  if (rows == 0) return WMC_OK;
  const int h = p->Q / 2;
  const size_t sm = sizeof(float) * ((size_t)p->Q * h + (size_t)(p->Q + 4));
  if (sm > 200 * 1024) return WMC_ERR_UNSUPPORTED;
  if (sm > 48 * 1024 &&
      raise_smem_limit(reinterpret_cast<const void*>(k_n2_eval), sm) != cudaSuccess)
    return WMC_ERR_CUDA;
  long long blocks = (rows * h + 255) / 256;
  if (blocks > 8LL * num_sms()) blocks = 8LL * num_sms();
  const float inv_scale = (float)(2.0 / (kHbarEVs * (double)p->Q));
  k_n2_eval<<<(unsigned)blocks, 256, sm, (cudaStream_t)stream>>>(p->n_x, p->Q, p->bc_potential, rows, V, params,
                                                                 inv_scale, VWh);
  return cudaGetLastError() == cudaSuccess ? WMC_OK : WMC_ERR_CUDA;
}

}  // extern "C"

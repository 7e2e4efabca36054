// Wigner-kernel contraction on the 5th-generation tensor cores (tcgen05):
// the precision forms of wmc_kernel_eval (BF16, FP16, FP16 hi/lo split, 3xTF32).
//
//   VWh[row][r] = c * sum_{m=1}^{h-1} A[row][m] S[m][r],  A[row][m] = V(i+m) - V(i-m)
//
// The sine matrix S is precomputed once per workspace as operand images in
// global memory (BF16, FP16 hi, FP16 lo, TF32 hi, TF32 lo) in 16 KB blocks of
// 128 rows in the layout below; A is generated on chip from the potential
// and never written to global memory.  Three kernels:
//   - k_kernel_eval_tc_ta<BF16 | FP16, N>: warp-specialised (16 builder /
//     epilogue warps, one MMA-issuing thread, one bulk-copy thread), the whole
//     A operand of a 128-row tile in tensor memory, B streamed through a deep
//     ring of shared-memory stages, M = N = 128, two TMEM accumulator buffers
//     so that the epilogue of one column tile overlaps the MMAs of the next
//     (K <= 512);
//   - k_rows_split<FP16 | TF32>: the hi/lo split forms, three MMAs per K step
//     (hi x hi, hi x lo, lo x hi), A through a ring of TMEM stages, each K
//     block's main product in its own accumulator;
//   - k_kernel_eval_tc: a per-tile kernel with both operands streamed, for
//     BF16 / FP16 windows wider than the tensor-memory form holds.
// Shared-memory operands use the K-major 128-byte swizzled layout: rows of
// 128 bytes (64 16-bit or 32 TF32 values), 8-row atoms 1024 bytes apart, the
// 16-byte chunks of row r XOR-swizzled by r % 8; shared-memory blocks are
// aligned to 1024 bytes.  Accumulation is FP32 in TMEM; the epilogue reads
// the accumulators with tcgen05.ld and combines and scales them in FP32.
//
// Every wait is bounded (about one second of SM clock); on a timeout the CTA
// sets WMC_FLAG_TIMEOUT, stops issuing work, lets its copies and MMAs in
// flight complete (bounded again) and still frees its tensor memory.
#include <cuda_bf16.h>
#include <cuda_fp16.h>

#include "wmc_device.cuh"
#include "wmc_ta_ring.cuh"

namespace wmc {

namespace {

constexpr int TM = 128, TN = 128, TK = 64;
constexpr uint32_t kSBO = 1024, kKStepBytes = 32;  // atom stride; bytes per K step of 16
constexpr uint32_t kTileBytes = TN * TK * 2;  // one 128 x 64 16-bit operand image
constexpr long long kWaitCycles = 2000000000ll;

__device__ __forceinline__ uint32_t smem_u32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

__device__ __forceinline__ void mbar_init(uint64_t* bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count) : "memory");
}

__device__ __forceinline__ void mbar_expect_tx(uint64_t* bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)), "r"(bytes)
               : "memory");
}

// One probe of the phase of the given parity.  While the phase is incomplete
// the thread may sleep in hardware for up to kSuspendNs nanoseconds (woken
// when the phase completes) instead of spinning on the barrier word.
constexpr uint32_t kSuspendNs = 100000;
__device__ __forceinline__ bool mbar_try_wait(uint64_t* bar, uint32_t parity) {
  uint32_t done;
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2, %3;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(done)
      : "r"(smem_u32(bar)), "r"(parity), "r"(kSuspendNs)
      : "memory");
  return done != 0;
}

// Waits for the phase of the given parity; false after about a second.
__device__ __forceinline__ bool mbar_wait(uint64_t* bar, uint32_t parity) {
  const long long t0 = clock64();
  while (!mbar_try_wait(bar, parity))
    if (clock64() - t0 > kWaitCycles) return false;
  return true;
}

__device__ __forceinline__ void bulk_g2s(void* dst, const void* src, uint32_t bytes, uint64_t* bar) {
  asm volatile(
      "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
          smem_u32(dst)),
      "l"(src), "r"(bytes), "r"(smem_u32(bar))
      : "memory");
}

__device__ __forceinline__ void fence_proxy_async_smem() { asm volatile("fence.proxy.async.shared::cta;" ::: "memory"); }
__device__ __forceinline__ void fence_mbar_init() { asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }

__device__ __forceinline__ void tmem_alloc(uint32_t* slot, uint32_t ncols) {
  asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(slot)), "r"(ncols)
               : "memory");
  asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
}

__device__ __forceinline__ void tmem_dealloc(uint32_t taddr, uint32_t ncols) {
  asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(taddr), "r"(ncols) : "memory");
}

// K-major shared-memory matrix descriptor (version 1) of the 128-byte swizzled
// layout: 8-row atoms of 128-byte rows (64 16-bit K values) 1024 bytes apart
// (SBO), the 16-byte chunks of row r XOR-swizzled by r % 8; a K step of 16
// values advances the start address by 32 bytes inside the atom.
__device__ __forceinline__ uint64_t smem_desc(uint32_t addr) {
  return (uint64_t)((addr & 0x3FFFFu) >> 4) | (1ull << 16) | ((uint64_t)(kSBO >> 4) << 32) | (1ull << 46) |
         (2ull << 61);
}

// Dynamic shared memory rounded up to the 1024-byte alignment the swizzled
// atoms need (launches request kSmemAlignPad extra bytes).
constexpr uint32_t kSmemAlignPad = 1024;
__device__ __forceinline__ uint8_t* align_smem(uint8_t* p) {
  const uint32_t a = smem_u32(p);
  return p + (((a + 1023u) & ~1023u) - a);
}

// Instruction descriptor of kind::f16: D FP32, A and B of one 16-bit format
// (0 FP16, 1 BF16), both K-major, M = 128, N = 128.
__host__ __device__ constexpr uint32_t idesc_f16(uint32_t fmt) {
  return (1u << 4) | (fmt << 7) | (fmt << 10) | ((uint32_t)(TN >> 3) << 17) | ((uint32_t)(TM >> 4) << 24);
}

__device__ __forceinline__ void mma_f16(uint32_t d_tmem, uint64_t adesc, uint64_t bdesc, uint32_t idesc,
                                        uint32_t accumulate) {
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "setp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}" ::"r"(d_tmem),
      "l"(adesc), "l"(bdesc), "r"(idesc), "r"(accumulate)
      : "memory");
}

// x rounded to TF32 (nearest, ties away from zero), as FP32 bits with the low
// 13 mantissa bits zero.
__device__ __forceinline__ uint32_t to_tf32(float x) {
  uint32_t r;
  asm("cvt.rna.tf32.f32 %0, %1;" : "=r"(r) : "f"(x));
  return r;
}

__device__ __forceinline__ void mma_commit(uint64_t* bar) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(smem_u32(bar))
               : "memory");
}

__device__ __forceinline__ void tmem_wait16(uint32_t* r);

// 16 consecutive 32-bit columns of this thread's TMEM lane.
__device__ __forceinline__ void tmem_ld16(uint32_t taddr, float* v) {
  uint32_t r[16];
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, "
      "%15}, [%16];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]),
        "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
      : "r"(taddr));
  tmem_wait16(r);
#pragma unroll
  for (int q = 0; q < 16; ++q) v[q] = __uint_as_float(r[q]);
}

// Split form of tmem_ld16: the load is issued into r, and tmem_wait16 waits
// for all loads in flight while naming r as read-write, so that no use of r
// can be scheduled before the wait.
__device__ __forceinline__ void tmem_ld16_issue(uint32_t taddr, uint32_t* r) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, "
      "%15}, [%16];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]),
        "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
      : "r"(taddr));
}

__device__ __forceinline__ void tmem_wait16(uint32_t* r) {
  asm volatile("tcgen05.wait::ld.sync.aligned;"
               : "+r"(r[0]), "+r"(r[1]), "+r"(r[2]), "+r"(r[3]), "+r"(r[4]), "+r"(r[5]), "+r"(r[6]), "+r"(r[7]),
                 "+r"(r[8]), "+r"(r[9]), "+r"(r[10]), "+r"(r[11]), "+r"(r[12]), "+r"(r[13]), "+r"(r[14]), "+r"(r[15])
               :
               : "memory");
}

// 16 consecutive 32-bit columns of this thread's TMEM lane from registers;
// tmem_wait_st waits until this thread's stores are complete.
__device__ __forceinline__ void tmem_st16(uint32_t taddr, const uint32_t* r) {
  asm volatile(
      "tcgen05.st.sync.aligned.32x32b.x16.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, "
      "%15, %16};" ::"r"(taddr),
      "r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7]), "r"(r[8]), "r"(r[9]),
      "r"(r[10]), "r"(r[11]), "r"(r[12]), "r"(r[13]), "r"(r[14]), "r"(r[15])
      : "memory");
}

__device__ __forceinline__ void tmem_wait_st() { asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory"); }

// kind::f16 MMA with the A operand in tensor memory: M = 128 rows in the 128
// lanes, each 32-bit column holding two consecutive K values (the lower K in
// the low half), K = 16 over 8 columns starting at a_tmem.
__device__ __forceinline__ void mma_f16_ta(uint32_t d_tmem, uint32_t a_tmem, uint64_t bdesc, uint32_t idesc,
                                           uint32_t accumulate) {
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "setp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], [%1], %2, %3, p;\n\t}" ::"r"(d_tmem),
      "r"(a_tmem), "l"(bdesc), "r"(idesc), "r"(accumulate)
      : "memory");
}

__device__ __forceinline__ float potential_at(const float* __restrict__ V, int n_x, int bc, long long l) {
  if (l >= 0 && l < n_x) return __ldg(V + l);
  if (!bc) return 0.f;
  return __ldg(V + (l < 0 ? 0 : n_x - 1));
}

// Byte offset of element (row, k) of a 128 x 64 K-major operand block in the
// 128-byte swizzled layout (row r at 128 r, chunk k / 8 stored at chunk
// (k / 8) ^ (r % 8)); blocks of consecutive rows concatenate.
__host__ __device__ __forceinline__ uint32_t core_offset(int row, int k) {
  return (uint32_t)(row * 128 + ((((k >> 3) ^ (row & 7)) & 7) << 4) + (k & 7) * 2);
}

__device__ __forceinline__ uint16_t to_bits(float x, int prec) {
  if (prec == WMC_BF16) return __bfloat16_as_ushort(__float2bfloat16_rn(x));
  return __half_as_ushort(__float2half_rn(x));
}

__device__ __forceinline__ float from_bits(uint16_t b, int prec) {
  if (prec == WMC_BF16) return __bfloat162float(__ushort_as_bfloat16(b));
  return __half2float(__ushort_as_half(b));
}

}  // namespace

// ---------------------------------------------------------------- operand images
// img[(nt * KB + kb)] is the 128 x 64 image of S[m = kb*64 + k + 1][r = nt*128 + n]
// (zero outside m < h, r < h), rounded to BF16 (img_bf16), FP16 (img_hi) and the
// FP16 residual scaled by 2^11 (img_lo).
__global__ void k_init_tc_images(int Q, int KB, int NT, uint16_t* __restrict__ img_bf16,
                                 uint16_t* __restrict__ img_hi, uint16_t* __restrict__ img_lo, int net) {
  const long long total = (long long)NT * KB * TN * TK;
  for (long long q = blockIdx.x * (long long)blockDim.x + threadIdx.x; q < total;
       q += (long long)gridDim.x * blockDim.x) {
    const int blk = (int)(q / (TN * TK));
    const int e = (int)(q % (TN * TK));
    const int n = e / TK, k = e % TK;
    const int nt = blk / KB, kb = blk % KB;
    const int kk = kb * TK + k, r = nt * TN + n;
    const float v = net == 2 ? sine_entry_n2(Q, kk, r) : sine_entry_n1(Q, kk, r);
    const size_t off = (size_t)blk * (kTileBytes / 2) + core_offset(n, k) / 2;
    img_bf16[off] = __bfloat16_as_ushort(__float2bfloat16_rn(v));
    const __half hi = __float2half_rn(v);
    img_hi[off] = __half_as_ushort(hi);
    img_lo[off] = __half_as_ushort(__float2half_rn((v - __half2float(hi)) * 2048.f));
  }
}

// The same sine matrix as TF32 hi/lo pairs (hi = tf32(v), lo = tf32(v - hi)),
// in 128 x 32 blocks of the swizzled layout (four 4-byte values per chunk).
__global__ void k_init_tc_images32(int Q, int KB32, int NT, uint32_t* __restrict__ img_hi,
                                   uint32_t* __restrict__ img_lo, int transposed) {
  const long long total = (long long)NT * KB32 * TN * 32;
  for (long long q = blockIdx.x * (long long)blockDim.x + threadIdx.x; q < total;
       q += (long long)gridDim.x * blockDim.x) {
    const int blk = (int)(q / (TN * 32));
    const int e = (int)(q % (TN * 32));
    const int n = e / 32, k = e % 32;
    const int nt = blk / KB32, kb = blk % KB32;
    // transposed (the adjoint's B): S[m][r] at n = m - 1, k = r
    const float v = transposed ? sine_entry_n1(Q, nt * TN + n, kb * 32 + k) : sine_entry_n1(Q, kb * 32 + k, nt * TN + n);
    // chunk k / 4 of row n, value k % 4 in it
    const size_t off = (size_t)blk * (kTileBytes / 4) + (core_offset(n, (k >> 2) * 8) >> 2) + (k & 3);
    const uint32_t hi = to_tf32(v);
    img_hi[off] = hi;
    img_lo[off] = to_tf32(v - __uint_as_float(hi));
  }
}

// ---------------------------------------------------------------- contraction
// Two pipeline stages: while the tensor cores run the MMAs of K block kb from
// stage kb % 2, the threads build the A operand of block kb + 1 into the other
// stage and thread 0 has already started the copy of its B operand(s); a
// stage is rewritten only after the MMAs that read it have completed (one
// mbarrier per stage for the copies, one for the MMA commits).  When the
// tile's 128 rows are 128 consecutive cells of one potential, the potential
// window they need is staged in shared memory once and the A operand is built
// from it without branches.
constexpr int kStages = 2;

__host__ __device__ constexpr size_t tc_smem_bytes(int h) {
  return kSmemAlignPad + (size_t)4 * kTileBytes + sizeof(float) * (size_t)(TM + 2 * h);
}

template <int PREC>
__global__ __launch_bounds__(128, 1) void k_kernel_eval_tc(const float* __restrict__ V, int n_x, int bc, int Q,
                                                           const int* __restrict__ occ,
                                                           const int* __restrict__ n_occ_dev, int n_occ_host,
                                                           const uint16_t* __restrict__ img_b, int KB, float c,
                                                           float* __restrict__ VWh, unsigned int* __restrict__ flags) {
  constexpr int kind_fmt = PREC == WMC_BF16 ? 1 : 0;
  constexpr uint32_t kCols = 256u;
  constexpr uint32_t idesc = idesc_f16(kind_fmt);
  extern __shared__ __align__(1024) uint8_t smem_raw[];
  uint8_t* smem = align_smem(smem_raw);
  uint8_t* sA[kStages] = {smem, smem + kTileBytes};
  uint8_t* sB[kStages] = {smem + 2 * kTileBytes, smem + 3 * kTileBytes};
  float* sV = reinterpret_cast<float*>(smem + 4 * kTileBytes);
  __shared__ __align__(8) uint64_t bar_tma[kStages];
  __shared__ __align__(8) uint64_t bar_mma[kStages];
  __shared__ uint32_t tmem_slot;
  __shared__ int s_abort, s_cell0;

  const int n_rows = n_occ_dev ? *n_occ_dev : n_occ_host;
  const int row0 = blockIdx.x * TM, col0 = blockIdx.y * TN;
  const int h = Q / 2;
  if (row0 >= n_rows || col0 >= h) return;  // uniform over the CTA, before any allocation
  const int tid = threadIdx.x, warp = tid >> 5;

  if (warp == 0) tmem_alloc(&tmem_slot, kCols);
  if (tid == 0) {
    for (int q = 0; q < kStages; ++q) {
      mbar_init(&bar_tma[q], 1);
      mbar_init(&bar_mma[q], 1);
    }
    fence_mbar_init();
    s_abort = 0;
  }

  // this thread's row: occ == nullptr means implicit rows over consecutive
  // potentials (row r is cell r % n_x of potential r / n_x)
  const int my_row = row0 + tid;
  const bool valid = my_row < n_rows;
  const int cell = valid ? (occ ? __ldg(occ + my_row) : my_row % n_x) : 0;
  const int pot_idx = (occ || !valid) ? 0 : my_row / n_x;
  const float* Vr = V + (size_t)pot_idx * n_x;
  if (tid == 0) s_cell0 = cell;
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = tmem_slot;
  const uint32_t accA = tmem, accB = tmem + (uint32_t)TN;
  const int pot0 = (occ || row0 >= n_rows) ? 0 : row0 / n_x;
  const bool contig = __syncthreads_and(valid && cell == s_cell0 + tid && pot_idx == pot0) != 0;
  if (contig) {
    const float* V0 = V + (size_t)pot0 * n_x;
    for (int q = tid; q < TM + 2 * h; q += blockDim.x) sV[q] = potential_at(V0, n_x, bc, (long long)s_cell0 - h + q);
  }

  const int half_kb = (KB + 1) / 2;
  const uint16_t* imgB_tile = img_b + (size_t)blockIdx.y * KB * (kTileBytes / 2);

  auto issue_copy = [&](int kb, int st) {
    mbar_expect_tx(&bar_tma[st], kTileBytes);
    bulk_g2s(sB[st], imgB_tile + (size_t)kb * (kTileBytes / 2), kTileBytes, &bar_tma[st]);
  };
  // this thread's A row of K block kb: window terms m = kb*64 + k + 1
  auto build_A = [&](int kb, int st) {
    if (contig) __syncthreads();  // the window is staged (first use) / keeps warps aligned
#pragma unroll
    for (int k8 = 0; k8 < TK / 8; ++k8) {
      uint32_t hw[4];
#pragma unroll
      for (int e = 0; e < 8; e += 2) {
        uint16_t hb[2];
#pragma unroll
        for (int u = 0; u < 2; ++u) {
          const int m = kb * TK + k8 * 8 + e + u + 1;
          float dv = 0.f;
          if (m <= h - 1) {
            if (contig) dv = __fsub_rn(sV[tid + h + m], sV[tid + h - m]);
            else if (valid)
              dv = __fsub_rn(potential_at(Vr, n_x, bc, (long long)cell + m), potential_at(Vr, n_x, bc, (long long)cell - m));
          }
          hb[u] = to_bits(dv, PREC);
        }
        hw[e / 2] = (uint32_t)hb[0] | ((uint32_t)hb[1] << 16);
      }
      const uint32_t off = core_offset(tid, k8 * 8);
      *reinterpret_cast<uint4*>(sA[st] + off) = make_uint4(hw[0], hw[1], hw[2], hw[3]);
    }
  };

  if (tid == 0) issue_copy(0, 0);
  build_A(0, 0);
  for (int kb = 0; kb < KB; ++kb) {
    const int st = kb & 1;
    const uint32_t ph = (uint32_t)((kb >> 1) & 1);
    fence_proxy_async_smem();
    __syncthreads();  // A of block kb is in stage st
    if (s_abort) break;
    if (tid == 0) {
      if (!mbar_wait(&bar_tma[st], ph)) {
        atomicOr(flags, WMC_FLAG_TIMEOUT);
        s_abort = 1;
      } else {
        tc_fence_after();
        const uint32_t acc = kb < half_kb ? accA : accB;
        const int first = kb == 0 || kb == half_kb;
#pragma unroll
        for (int s = 0; s < TK / 16; ++s) {
          const uint64_t a_hi = smem_desc(smem_u32(sA[st]) + s * kKStepBytes);
          const uint64_t b_hi = smem_desc(smem_u32(sB[st]) + s * kKStepBytes);
          mma_f16(acc, a_hi, b_hi, idesc, (first && s == 0) ? 0u : 1u);
        }
        mma_commit(&bar_mma[st]);
        // the other stage is free once the MMAs of block kb - 1 are done
        if (kb + 1 < KB) {
          if (kb >= 1 && !mbar_wait(&bar_mma[st ^ 1], (uint32_t)(((kb - 1) >> 1) & 1))) {
            atomicOr(flags, WMC_FLAG_TIMEOUT);
            s_abort = 1;
          } else {
            issue_copy(kb + 1, st ^ 1);
          }
        }
      }
    }
    if (kb + 1 < KB) {
      if (kb >= 1 && !mbar_wait(&bar_mma[st ^ 1], (uint32_t)(((kb - 1) >> 1) & 1))) s_abort = 1;
      build_A(kb + 1, st ^ 1);
    }
  }
  // all MMAs of the tile done (commits complete in order)
  if (tid == 0 && !s_abort && !mbar_wait(&bar_mma[(KB - 1) & 1], (uint32_t)(((KB - 1) >> 1) & 1))) {
    atomicOr(flags, WMC_FLAG_TIMEOUT);
    s_abort = 1;
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();

  if (!s_abort) {
    // epilogue: lane (warp 32 w + l) of TMEM holds tile row 32 w + l
    const int row = row0 + warp * 32 + (tid & 31);
    const uint32_t lane_base = (uint32_t)(warp * 32) << 16;
    const bool has_B = KB > half_kb;
    for (int cc = 0; cc < TN; cc += 16) {
      float a[16], b[16];
      tmem_ld16(accA + lane_base + (uint32_t)cc, a);
      if (has_B) tmem_ld16(accB + lane_base + (uint32_t)cc, b);
      if (row < n_rows) {
        float* out = VWh + (size_t)row * h + col0 + cc;
#pragma unroll
        for (int q = 0; q < 16; ++q) {
          if (col0 + cc + q >= h) break;
          float v = a[q];
          if (has_B) v = __fadd_rn(v, b[q]);
          out[q] = __fmul_rn(c, v);
        }
      }
    }
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 0) tmem_dealloc(tmem, kCols);
}

// ---------------------------------------------------------------- warp-specialised forms
// Roles of the form below (608 threads): warps 0-15 build
// the A operand and then run the epilogue, warp 16 has one thread issue the
// MMAs, warp 17 one thread stream the B operand images.  The epilogue warp w
// reads TMEM lane quadrant w % 4 and transposes each 32 x 16 piece through
// shared memory, so that global stores are whole 64-byte row segments.
constexpr int kWsBuilders = 512;

constexpr int kWsStageFloats = 32 * 16;  // epilogue staging per warp: 32 rows x 16 columns

// AND of pred over the kWsBuilders builder threads (named barrier 1).
__device__ __forceinline__ bool builders_and(bool pred) {
  uint32_t r;
  asm volatile(
      "{\n\t.reg .pred q, p;\n\t"
      "setp.ne.u32 q, %1, 0;\n\t"
      "barrier.cta.red.and.pred p, 1, %2, q;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(r)
      : "r"((uint32_t)pred), "n"(kWsBuilders)
      : "memory");
  return r != 0;
}

__device__ __forceinline__ void builders_sync() { asm volatile("barrier.cta.sync 1, %0;" ::"n"(kWsBuilders) : "memory"); }

template <int PREC>
__device__ __forceinline__ uint32_t pack2(float a, float b) {
  if (PREC == WMC_BF16) {
    const __nv_bfloat162 v = __floats2bfloat162_rn(a, b);
    return *reinterpret_cast<const uint32_t*>(&v);
  } else {
    const __half2 v = __floats2half2_rn(a, b);
    return *reinterpret_cast<const uint32_t*>(&v);
  }
}

// Cells the rows of a 128-row tile may span for their potential window (span
// + 2 h values) to be staged in shared memory; beyond, every term is read from
// the potential itself.  Scattered lists of every second cell still fit.
constexpr int kWindowSpan = 640;

// N consecutive terms kk = k0 .. of the A operand of one row.  w[m] = V(cell + m).
template <int NET, int N>
__device__ __forceinline__ void a_run_window(const float* w, int h, int cell, int k0, float (&dv)[N]) {
  if (NET == 1) {
    if (k0 + N <= h - 1) {
#pragma unroll
      for (int e = 0; e < N; ++e) dv[e] = __fsub_rn(w[k0 + e + 1], w[-(k0 + e + 1)]);
    } else {
#pragma unroll
      for (int e = 0; e < N; ++e) {
        const int m = k0 + e + 1;
        dv[e] = 0.f;
        if (m <= h - 1) dv[e] = __fsub_rn(w[m], w[-m]);
      }
    }
  } else {
    // a pair to the right of the cell where i + u is even, else its mirror to the left
#pragma unroll
    for (int e = 0; e < N; ++e) {
      const int u = k0 + e;
      dv[e] = 0.f;
      if (u <= h - 1) {
        const bool right = ((cell + u) & 1) == 0;
        const int at = right ? u : -u - 1;
        const float s = __fadd_rn(w[at], w[at + 1]);
        dv[e] = right ? s : -s;
      }
    }
  }
}

// ---------------------------------------------------------------- A in tensor memory
// BF16 / FP16, K <= 512: one CTA per 128 rows and a run of 128-column tiles.
// The whole A operand of the row tile lives in tensor memory (up to 8 blocks
// of 64 K values, 32 columns each, at columns 0 .. 255), built once and used
// by every column tile; two 128-column FP32 accumulator buffers at columns
// 256 and 384 let the epilogue of tile j overlap the MMAs of tile j + 1; the
// shared memory holds a ring of kTaStages B stages (128 columns x two 64-K
// blocks each), so the tensor core reads only B from shared memory and the ring
// covers a copy round trip.  Builder warp w writes TMEM lanes 32 (w % 4) ..
// + 31 (one row of the tile per thread) for the K blocks kb = w / 4 (mod 4):
// its row's entries, packed in pairs, by tcgen05.st, then arrives on
// a_ready[kb].  Two threads issue the MMAs, one the even and one the odd column
// tiles: each waits for a_ready (its first tile), each B stage of its tiles (by
// the barrier of that filling, wmc_ta_ring.cuh) and its drained accumulator
// buffer, and commits each stage and each tile.  Every wait is bounded; on a
// timeout an abort flag makes all roles drain to the final barrier, after which
// TMEM is freed.
// What bounds it: building A, then the commits between the MMAs (with one
// issuing thread and a commit per K block they ran at a third of the pipe's
// rate).  BF16, 16384 cells at Q = 1024: 22.8 -> 19.0 us with two issuers and
// stages of two blocks; N = 2, FP16, 3600 cells: 57 -> 12.7 us, its terms no
// longer chosen by divergent branches.
constexpr int kTaThreads = kWsBuilders + 96;
constexpr uint32_t kTaStageBytes = 2 * kTileBytes;
static_assert((kTaMaxKB * TK + 1 + TN - 1) / TN <= kTaMaxTiles, "h <= kTaMaxKB TK + 1 columns");
constexpr uint32_t kTaAccCol = 256;

__host__ __device__ constexpr size_t ta_window_floats(int h) {
  return (size_t)kWindowSpan + 2 * (size_t)h + 4 > (size_t)(kWsBuilders / 32) * kWsStageFloats
             ? (size_t)kWindowSpan + 2 * (size_t)h + 4
             : (size_t)(kWsBuilders / 32) * kWsStageFloats;
}

__host__ __device__ constexpr size_t ta_smem_bytes(int h) {
  return kSmemAlignPad + (size_t)kTaStages * kTaStageBytes + sizeof(float) * ta_window_floats(h);
}

template <int PREC, int NET>
__global__ __launch_bounds__(kTaThreads, 1) void k_kernel_eval_tc_ta(const float* __restrict__ V, int n_x, int bc,
                                                                     int Q, const int* __restrict__ occ,
                                                                     const int* __restrict__ n_occ_dev, int n_occ_host,
                                                                     const uint16_t* __restrict__ img_b, int KB,
                                                                     int NT, int n_split, float c,
                                                                     float* __restrict__ VWh,
                                                                     unsigned int* __restrict__ flags) {
  constexpr uint32_t idesc = idesc_f16(PREC == WMC_BF16 ? 1u : 0u);  // M = N = 128
  constexpr int STG = kTaStages;
  constexpr uint32_t n_cols = 512;
  extern __shared__ __align__(1024) uint8_t smem_raw[];
  uint8_t* smem = align_smem(smem_raw);
  uint8_t* sB = smem;                                                     // STG stages of two 128 x 64 blocks
  float* sV = reinterpret_cast<float*>(sB + (size_t)STG * kTaStageBytes);  // window, then epilogue staging
  __shared__ __align__(8) uint64_t a_ready[kTaMaxKB];
  __shared__ __align__(8) uint64_t b_full[kTaFills], b_empty[kTaStages];
  __shared__ __align__(8) uint64_t acc_full[2], acc_empty[2];
  __shared__ __align__(8) uint64_t drain[2];
  __shared__ int s_min[kWsBuilders / 32], s_max[kWsBuilders / 32];
  __shared__ uint32_t tmem_slot;
  __shared__ volatile int s_abort;

  const int n_rows = n_occ_dev ? *n_occ_dev : n_occ_host;
  const int row0 = blockIdx.x * TM;
  const int h = Q / 2;
  if (row0 >= n_rows) return;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  // this CTA's 128-column tiles: [nt_begin, nt_begin + n_my)
  const int nt_begin = (int)(((long long)blockIdx.y * NT) / n_split);
  const int n_my = (int)(((long long)(blockIdx.y + 1) * NT) / n_split) - nt_begin;
  const int KP = (KB + 1) / 2, n_tiles = n_my * KP;  // stages of a column tile, and of all

  if (warp == 0) tmem_alloc(&tmem_slot, n_cols);
  if (tid == 0) {
    for (int q = 0; q < KB; ++q) mbar_init(&a_ready[q], 4);  // one arrival per lane-quarter warp
    for (int q = 0; q < n_tiles; ++q) mbar_init(&b_full[q], 1);
    for (int q = 0; q < STG; ++q) mbar_init(&b_empty[q], 1);
    for (int q = 0; q < 2; ++q) {
      mbar_init(&acc_full[q], 1);
      mbar_init(&acc_empty[q], kWsBuilders / 32);  // one arrival per epilogue warp
    }
    for (int q = 0; q < 2; ++q) mbar_init(&drain[q], 1);
    fence_mbar_init();
    s_abort = 0;
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = tmem_slot;

  if (warp == kWsBuilders / 32 + 1) {
    // ---- B producer
    if (lane == 0) {
      int issued = 0;
      for (int t = 0; t < n_tiles && !s_abort; ++t) {
        const int st = ta_stage(t);
        uint64_t* full = &b_full[ta_full_bar(t)];
        if (t >= STG && !mbar_wait(&b_empty[st], ta_empty_parity(t))) {
          atomicOr(flags, WMC_FLAG_TIMEOUT);
          s_abort = 1;
          break;
        }
        const int nt = nt_begin + t / KP, kb = 2 * (t % KP);
        const uint32_t bytes = kb + 1 < KB ? kTaStageBytes : kTileBytes;
        mbar_expect_tx(full, bytes);
        bulk_g2s(sB + (size_t)st * kTaStageBytes, img_b + ((size_t)nt * KB + kb) * (kTileBytes / 2), bytes, full);
        issued = t + 1;
      }
      if (s_abort)  // let the copies still in flight land before the CTA exits (bounded)
        for (int t = max(0, issued - STG); t < issued; ++t)
          (void)mbar_wait(&b_full[ta_full_bar(t)], ta_full_parity(t));
    }
  } else if (warp == kWsBuilders / 32 || warp == kWsBuilders / 32 + 2) {
    // ---- MMA issuers: one thread the even column tiles (accumulator 0), one the
    // odd ones, so that one's waits and commits pass behind the other's MMAs
    const int buf = warp == kWsBuilders / 32 ? 0 : 1;
    if (lane == 0) {
      for (int j = buf; j < n_my && !s_abort; j += kTaIssuers) {
        if (j >= 2 && !mbar_wait(&acc_empty[buf], (uint32_t)(((j - 2) >> 1) & 1))) {
          atomicOr(flags, WMC_FLAG_TIMEOUT);
          s_abort = 1;
          break;
        }
        tc_fence_after();
        const uint32_t acc = tmem + kTaAccCol + (uint32_t)(buf * TN);
        for (int kb = 0; kb < KB; ++kb) {
          const int t = j * KP + kb / 2, st = ta_stage(t);
          if ((j < 2 && !mbar_wait(&a_ready[kb], 0u)) ||
              ((kb & 1) == 0 && !mbar_wait(&b_full[ta_full_bar(t)], ta_full_parity(t)))) {
            atomicOr(flags, WMC_FLAG_TIMEOUT);
            s_abort = 1;
            break;
          }
          tc_fence_after();
          const uint32_t b_base = smem_u32(sB + (size_t)st * kTaStageBytes + (kb & 1) * kTileBytes);
#pragma unroll
          for (int s4 = 0; s4 < TK / 16; ++s4)
            mma_f16_ta(acc, tmem + (uint32_t)(kb * (TK / 2) + s4 * 8), smem_desc(b_base + s4 * kKStepBytes), idesc,
                       (kb == 0 && s4 == 0) ? 0u : 1u);
          if (((kb & 1) || kb + 1 == KB) && t + STG < n_tiles) mma_commit(&b_empty[st]);  // (a stage filled again)
        }
        if (s_abort) break;
        mma_commit(&acc_full[buf]);
      }
      if (s_abort) {  // drain the MMAs already issued before TMEM is freed (bounded)
        mma_commit(&drain[buf]);
        (void)mbar_wait(&drain[buf], 0u);
      }
    }
  } else {
    // ---- A builders (warps 0-15), then the epilogue
    // this thread's row of the tile = its TMEM lane (rows past the end repeat the last)
    const int quad = warp & 3, kp = warp >> 2;
    const int row = min(row0 + 32 * quad + lane, n_rows - 1);
    const int cell = occ ? __ldg(occ + row) : row % n_x;
    const int pot0 = occ ? 0 : row0 / n_x, pot_i = occ ? 0 : row / n_x;
    // the cells of the tile's rows, and whether their window can be staged
    int lo = __reduce_min_sync(0xffffffffu, cell), hi = __reduce_max_sync(0xffffffffu, cell);
    if (lane == 0) {
      s_min[warp] = lo;
      s_max[warp] = hi;
    }
    const bool one_pot = builders_and(pot_i == pot0);
    lo = min(min(s_min[0], s_min[1]), min(s_min[2], s_min[3]));
    hi = max(max(s_max[0], s_max[1]), max(s_max[2], s_max[3]));
    const bool window = one_pot && hi - lo < kWindowSpan;
    if (window) {
      const float* V0 = V + (size_t)pot0 * n_x;
      const int n = hi - lo + 1 + 2 * h;
      constexpr int kU = 4;  // loads issued together
      for (int q0 = tid; q0 < n; q0 += kU * kWsBuilders) {
        float v[kU];
#pragma unroll
        for (int u = 0; u < kU; ++u) {
          const int q = q0 + u * kWsBuilders;
          v[u] = q < n ? potential_at(V0, n_x, bc, (long long)lo - h + q) : 0.f;
        }
#pragma unroll
        for (int u = 0; u < kU; ++u)
          if (q0 + u * kWsBuilders < n) sV[q0 + u * kWsBuilders] = v[u];
      }
      builders_sync();
    }
    const float* w = sV + h + (cell - lo);
    const float* Vr = V + (size_t)pot_i * n_x;
    const uint32_t lane_base = (uint32_t)(quad * 32) << 16;
#pragma unroll 1
    for (int kb = kp; kb < KB; kb += 4) {
#pragma unroll 1
      for (int hf = 0; hf < 2; ++hf) {  // 32 K values, 16 columns
        float dv[32];
        const int k0 = kb * TK + 32 * hf;
        if (window) {
          a_run_window<NET, 32>(w, h, cell, k0, dv);
        } else {
#pragma unroll
          for (int e = 0; e < 32; ++e) dv[e] = a_term<NET>(Vr, n_x, bc, h, cell, k0 + e);
        }
        uint32_t wv[16];
#pragma unroll
        for (int e = 0; e < 16; ++e) wv[e] = pack2<PREC>(dv[2 * e], dv[2 * e + 1]);
        tmem_st16(tmem + lane_base + (uint32_t)(kb * (TK / 2) + 16 * hf), wv);
      }
      tmem_wait_st();
      tc_fence_before();
      __syncwarp();
      if (lane == 0)
        asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(&a_ready[kb])) : "memory");
    }
    // epilogue of each column tile: warp w reads lanes 32 (w % 4) .. + 31, columns 32 (w / 4) .. + 31
    const int cq = warp >> 2;
    float* stg = sV + warp * kWsStageFloats;
    const bool vec_ok = (h & 3) == 0 && (reinterpret_cast<uintptr_t>(VWh) & 15) == 0;
    for (int j = 0; j < n_my; ++j) {
      const int buf = j & 1;
      // lane 0 waits for the tile; the decision is warp-uniform because the
      // TMEM loads below are warp-collective
      int okw = 1;
      if (lane == 0) okw = !s_abort && mbar_wait(&acc_full[buf], (uint32_t)((j >> 1) & 1));
      const bool ok = __shfl_sync(0xffffffffu, okw, 0) != 0;
      if (!ok) {
        if (lane == 0) atomicOr(flags, WMC_FLAG_TIMEOUT);
        s_abort = 1;
        break;
      }
      tc_fence_after();
      constexpr int NP = TN / 64;  // pieces of 16 columns per warp
      uint32_t rg2[2][16];
      const uint32_t tbase = tmem + kTaAccCol + (uint32_t)(buf * TN) + lane_base + (uint32_t)(cq * (TN / 4));
      tmem_ld16_issue(tbase, rg2[0]);
      tmem_wait16(rg2[0]);
#pragma unroll
      for (int hf = 0; hf < NP; ++hf) {
        if (hf + 1 < NP) tmem_ld16_issue(tbase + (uint32_t)((hf + 1) * 16), rg2[(hf + 1) & 1]);
        const uint32_t* a = rg2[hf & 1];
        const int col0 = (nt_begin + j) * TN + cq * (TN / 4) + hf * 16;
        // row `lane` of the piece; its four 16-byte groups are XOR-swizzled by
        // (row / 2) % 4, so that the row-wise writes and the group-wise reads
        // below are free of bank conflicts
#pragma unroll
        for (int g = 0; g < 4; ++g)
          *reinterpret_cast<float4*>(stg + lane * 16 + 4 * (g ^ ((lane >> 1) & 3))) =
              make_float4(__fmul_rn(c, __uint_as_float(a[4 * g])), __fmul_rn(c, __uint_as_float(a[4 * g + 1])),
                          __fmul_rn(c, __uint_as_float(a[4 * g + 2])), __fmul_rn(c, __uint_as_float(a[4 * g + 3])));
        __syncwarp();
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          const int r2 = 8 * i + (lane >> 2), g = lane & 3;
          const float4 v = *reinterpret_cast<const float4*>(stg + r2 * 16 + 4 * (g ^ ((r2 >> 1) & 3)));
          const int grow = row0 + quad * 32 + r2, gcol = col0 + 4 * g;
          if (grow < n_rows && gcol < h) {
            float* out = VWh + (size_t)grow * h + gcol;
            if (vec_ok) {
              *reinterpret_cast<float4*>(out) = v;
            } else {
              out[0] = v.x;
              if (gcol + 1 < h) out[1] = v.y;
              if (gcol + 2 < h) out[2] = v.z;
              if (gcol + 3 < h) out[3] = v.w;
            }
          }
        }
        __syncwarp();
        if (hf + 1 < NP) tmem_wait16(rg2[(hf + 1) & 1]);
      }
      tc_fence_before();
      __syncwarp();
      if (lane == 0)
        asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(&acc_empty[buf])) : "memory");
    }
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 0) {
    tc_fence_after();
    tmem_dealloc(tmem, n_cols);
  }
}

// ---------------------------------------------------------------- split forms
// FP16 hi/lo split: A = A_hi + 2^-11 A_lo, B = B_hi + 2^-11 B_lo, and
//   A B ~ A_hi B_hi + 2^-11 (A_hi B_lo + A_lo B_hi)
// (the A_lo B_lo term is below FP32 rounding).  3xTF32 (TF32 = true) is the
// same with TF32 parts and no scaling (TF32 keeps the FP32 exponent range):
// A = A_hi + A_lo with A_hi = tf32(A), A_lo = tf32(A - A_hi).  An operand block
// holds 128 rows x 64 FP16 or x 32 TF32 values.  The tensor core's FP32
// accumulation does not round to nearest: its error grows with the number of
// MMAs accumulated into one TMEM accumulator.  So the A_hi B_hi product of
// every K block goes to an accumulator of its own, drained into FP32 registers
// (round to nearest); the cross terms, 2^-11 smaller, share one over all of K.
//
// One persistent CTA per SM takes a run of consecutive 128 x 128 tiles (the
// column tiles of a row tile follow each other) and keeps four stages working
// at once across K blocks and tiles:
//   - warps 0-7 build A, one row and half a K block per thread, into a ring of
//     two TMEM stages (32 columns hi, 32 lo);
//   - warp 17 streams the (hi, lo) blocks of B through kSpStages of shared
//     memory;
//   - warps 16 and 18 issue 12 MMAs per K block (N = 128, A from TMEM): the
//     main products into two alternating TMEM accumulators, the cross terms into
//     a third;
//   - warps 8-15 drain the main accumulator of each K block, 64 columns per
//     warp, and write the tile.
// What bounds it: the MMA pipe and its hand-overs.  An MMA of this shape takes
// 82 cycles with A in TMEM (86 with A in shared memory, where the builders'
// stores, the copies and the MMA's own reads would also exceed the 128 B/cycle
// of shared memory), and each commit holds up the MMAs behind it by about 165,
// so a K block takes about 1860 cycles here.  The form before built passes of
// four K blocks in shared memory and drained each pass before it built the
// next, 3400 cycles a block: 16384 cells at Q = 1024 (3xTF32) 111 -> 63 us, 3600
// occupied cells in the step 47 -> 22 us, 262144 rows at Q = 256 155 -> 78 us,
// the adjoint contraction over the same rows 277 -> 130 us (half of it the builders and the stores).
constexpr int kSpStages = 5;
// K blocks whose barriers are in use at once: more than the longest look-back,
// kSpStages blocks, so that no waiter meets a barrier two phases on.
constexpr int kSpRing = 8;
static_assert(kSpRing > kSpStages, "a barrier comes round only after every waiter has seen it");
constexpr int kSpBuilders = 256, kSpThreads = 19 * 32;
constexpr uint32_t kSpAccX = 2 * TN, kSpA = 3 * TN;  // TMEM columns: main 0, main 1, cross, A ring

// NET = 3, the adjoint contraction Abar = c Gbar S^T of the differentiation
// form: A is Gbar[row][r] = gVW[row][r] + g_gamma[row] dgamma/dVWh[row][r]
// (K = h columns r), formed by the builders from these rows; the B image
// holds S[m][r] at (n = m - 1, k = r).
struct DenseA {
  const float* gVW;      // [rows][h] or null
  const float* VWh;      // [rows][h], the forward rows (sign of each entry)
  const float* g_gamma;  // [rows] or null
  int ca, cb, cr0;       // momentum grid: n_M = ca Q + cb, cr0 = -n_M/2 mod Q
};

// number of momentum indices M of the grid with M = r (mod Q)
__device__ __forceinline__ int grid_count_tc(int r, int Q, int a, int b, int r0) {
  int off = r - r0;
  if (off < 0) off += Q;
  return a + (off < b ? 1 : 0);
}

__host__ __device__ constexpr size_t split_window_floats(int h) { return (size_t)kWindowSpan + 2 * (size_t)h + 4; }

// Tiles whose rows fit no window (cells too far apart, or of more than one
// potential): in the STAGED form every builder warp fetches 16 terms of each of its
// 32 rows at a time by coalesced loads and hands them to the rows' threads through
// kRowStage floats of shared memory.  Where the windows leave no room for it, that
// is the tile's own window buffer, which is then large enough.
constexpr int kRowStage = 32 * 16;  // floats per builder warp
constexpr int kRowStageOwn = 8 * kRowStage;
__host__ __device__ constexpr bool split_row_stage_apart(int h) {
  return kSmemAlignPad + (size_t)kSpStages * 2 * kTileBytes + sizeof(float) * 8 * kWsStageFloats +
             sizeof(float) * (2 * split_window_floats(h) + kRowStageOwn) <=
         226 * 1024;
}
static_assert([] {
  for (int h = 1; h <= 2048; ++h)
    if (!split_row_stage_apart(h) && split_window_floats(h) < kRowStageOwn + 4) return false;
  return true;
}(), "a window buffer holds the row stages where they have no room of their own");

// NET = 3: the rows of gVW and VWh of a K block (128 x 32) pass through
// kDenseStages buffers of shared memory each, padded to 36 floats a row; fewer
// B stages make room.
constexpr int kDenseStages = 3, kDensePitch = 36;
__host__ __device__ constexpr int split_stages(int net) { return net == 3 ? 3 : kSpStages; }

__host__ __device__ constexpr size_t split_smem_bytes(int h, int net, bool staged) {
  return kSmemAlignPad + (size_t)split_stages(net) * 2 * kTileBytes + sizeof(float) * 8 * kWsStageFloats +
         sizeof(float) * (net == 3 ? (size_t)2 * kDenseStages * TM * kDensePitch
                                   : 2 * split_window_floats(h) + (staged && split_row_stage_apart(h) ? kRowStageOwn : 0));
}

// N consecutive terms kk = k0 .. of the A operand for the 32 rows of a warp (cell,
// and base = where its potential begins: the lane's row), dv those of the lane's
// own row.  Lanes 0-15 load the 16 terms of one row and lanes 16-31 those of the
// next, consecutive cells each; a row's 16-byte groups go to stg XOR-swizzled by
// (row / 2) % 4, so that the row's thread reads them without bank conflicts.
template <int NET, int N>
__device__ __forceinline__ void a_run_rows(const float* __restrict__ V, int n_x, int bc, int h, int cell, int base,
                                           int k0, float* stg, float (&dv)[N]) {
  static_assert(N % 16 == 0, "");
  const int lane = threadIdx.x & 31, l = lane & 15, second = lane >> 4;
  const int last = NET == 1 ? h - 2 : h - 1;  // last term that is not zero
#pragma unroll
  for (int q = 0; q < N; q += 16) {
    const int t = k0 + q + l;
    if (k0 + q > last) {  // (uniform)
#pragma unroll
      for (int e = 0; e < 16; ++e) dv[q + e] = 0.f;
      continue;
    }
    __syncwarp();  // the stage's last terms are read
#pragma unroll 1
    for (int j0 = 0; j0 < 16; j0 += 8) {
      float va[8], vb[8];  // sixteen loads under way together, without branches
      uint32_t left = 0u;
#pragma unroll
      for (int j = 0; j < 8; ++j) {
        const int row = 2 * (j0 + j) + second;
        const int c = __shfl_sync(0xffffffffu, cell, row), b = __shfl_sync(0xffffffffu, base, row);
        const bool right = NET == 1 || ((c + t) & 1) == 0;
        const int a0 = NET == 1 ? c + t + 1 : (right ? c + t : c - t - 1), a1 = NET == 1 ? c - t - 1 : a0 + 1;
        const float x0 = __ldg(V + (b + min(max(a0, 0), n_x - 1))), x1 = __ldg(V + (b + min(max(a1, 0), n_x - 1)));
        va[j] = (unsigned)a0 < (unsigned)n_x || bc ? x0 : 0.f;
        vb[j] = (unsigned)a1 < (unsigned)n_x || bc ? x1 : 0.f;
        if (NET == 2) left |= (right ? 0u : 1u) << j;
      }
#pragma unroll
      for (int j = 0; j < 8; ++j) {
        float d = NET == 1 ? __fsub_rn(va[j], vb[j]) : __fadd_rn(va[j], vb[j]);
        if (NET == 2 && ((left >> j) & 1u)) d = -d;
        stg[(2 * (j0 + j) + second) * 16 + (((l >> 2) ^ ((j0 + j) & 3)) << 2) + (l & 3)] = t <= last ? d : 0.f;
      }
    }
    __syncwarp();
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      const float4 x = *reinterpret_cast<const float4*>(stg + lane * 16 + 4 * (e ^ ((lane >> 1) & 3)));
      dv[q + 4 * e] = x.x, dv[q + 4 * e + 1] = x.y, dv[q + 4 * e + 2] = x.z, dv[q + 4 * e + 3] = x.w;
    }
  }
}

__device__ __forceinline__ void mma_tf32_ta(uint32_t d_tmem, uint32_t a_tmem, uint64_t bdesc, uint32_t idesc,
                                            uint32_t accumulate) {
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "setp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::1.kind::tf32 [%0], [%1], %2, %3, p;\n\t}" ::"r"(d_tmem),
      "r"(a_tmem), "l"(bdesc), "r"(idesc), "r"(accumulate)
      : "memory");
}

__device__ __forceinline__ void mbar_arrive(uint64_t* bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(bar)) : "memory");
}

// Four bytes of global memory to shared memory, zero if not in; waited for by
// cp_async_wait.
__device__ __forceinline__ void cp_async4(float* dst, const float* src, bool in) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"(smem_u32(dst)), "l"(src), "r"(in ? 4 : 0)
               : "memory");
}
__device__ __forceinline__ void cp_async16(float* dst, const float* src, bool in) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(smem_u32(dst)), "l"(src), "r"(in ? 16 : 0)
               : "memory");
}
__device__ __forceinline__ void cp_async_wait() { asm volatile("cp.async.wait_all;" ::: "memory"); }

// Reductions over the kSpBuilders builder threads (named barrier 1; every
// builder thread takes part).
__device__ __forceinline__ void sp_builders_sync() {
  asm volatile("barrier.cta.sync 1, %0;" ::"n"(kSpBuilders) : "memory");
}

// The row tile a CTA builds from: whether its window is staged, and the row of
// this thread.
struct SplitRows {
  bool window;
  int cell0;   // first cell of the window's rows
  int cell;    // this thread's row: cell and potential (clamped to a valid row)
  int pot;
};

template <bool TF32, int NET, bool STAGED>
__global__ __launch_bounds__(kSpThreads, 1) void k_rows_split(
    const float* __restrict__ V, int n_x, int bc, int Q, const int* __restrict__ occ,
    const int* __restrict__ n_occ_dev, int n_occ_host, const void* __restrict__ img_hi_v,
    const void* __restrict__ img_lo_v, int KB, int NT, float c, float* __restrict__ VWh,
    unsigned int* __restrict__ flags, DenseA dense) {
  // FP16 x FP16 -> FP32 (format 0) or TF32 x TF32 -> FP32 (format 2)
  constexpr uint32_t idesc = idesc_f16(TF32 ? 2u : 0u);
  constexpr int KBLK = TF32 ? 32 : TK;   // K values per operand block
  constexpr int EPT = KBLK / 2;          // values a builder thread makes of one block
  constexpr int STG = split_stages(NET);
  constexpr float kLoScale = TF32 ? 1.f : 0x1p-11f;
  const uint8_t* img_hi = static_cast<const uint8_t*>(img_hi_v);
  const uint8_t* img_lo = static_cast<const uint8_t*>(img_lo_v);
  extern __shared__ __align__(1024) uint8_t smem_raw[];
  uint8_t* sB = align_smem(smem_raw);                                             // stages of (B_hi, B_lo)
  float* s_stage = reinterpret_cast<float*>(sB + (size_t)STG * 2 * kTileBytes);  // output staging, per drain warp
  float* s_win = s_stage + 8 * kWsStageFloats;  // two windows (NET = 3: the rows' buffers)
  // of K block g, index g % kSpRing: its operands are there; its MMAs are complete
  __shared__ __align__(8) uint64_t full[kSpRing], done[kSpRing];
  __shared__ __align__(8) uint64_t acc_empty[2], x_empty, drain[2];
  __shared__ uint32_t tmem_slot;
  __shared__ volatile int s_abort;
  __shared__ int s_min[8], s_max[8];
  __shared__ __align__(16) float s_cnt[NET == 3 ? 2 * kAdjMaxH : 4];

  const int n_rows = n_occ_dev ? *n_occ_dev : n_occ_host;
  const int h = Q / 2;
  const long long n_tiles = (long long)((n_rows + TM - 1) / TM) * NT;
  // this CTA's tiles [t0, t0 + n_my); row tile t / NT, column tile t % NT
  const long long t0 = n_tiles * blockIdx.x / gridDim.x;
  const int n_my = (int)(n_tiles * (blockIdx.x + 1) / gridDim.x - t0);
  if (n_my <= 0) return;  // uniform over the CTA, before any allocation
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;

  if (warp == 0) tmem_alloc(&tmem_slot, 512u);
  if (tid == 0) {
    for (int q = 0; q < kSpRing; ++q) {
      mbar_init(&full[q], kSpBuilders / 32 + 1);  // the builder warps, and the B producer with its bytes
      mbar_init(&done[q], 2);                     // both MMA threads
    }
    for (int q = 0; q < 2; ++q) {
      mbar_init(&acc_empty[q], 8);
      mbar_init(&drain[q], 1);
    }
    mbar_init(&x_empty, 8);
    fence_mbar_init();
    s_abort = 0;
  }
  if (NET == 3)
    for (int r = tid; r < h; r += kSpThreads) {
      s_cnt[r] = r ? (float)grid_count_tc(r, Q, dense.ca, dense.cb, dense.cr0) : 0.f;
      s_cnt[kAdjMaxH + r] = r ? (float)grid_count_tc(Q - r, Q, dense.ca, dense.cb, dense.cr0) : 0.f;
    }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = tmem_slot;
  const int n_blocks = n_my * KB;  // K blocks of this CTA, numbered through its tiles
  // a failed wait (about a second): every role stops working
  auto give_up = [&]() {
    atomicOr(flags, WMC_FLAG_TIMEOUT);
    s_abort = 1;
  };
  auto wait_full = [&](int g) { return mbar_wait(&full[g % kSpRing], (uint32_t)((g / kSpRing) & 1)); };
  auto wait_done = [&](int g) { return mbar_wait(&done[g % kSpRing], (uint32_t)((g / kSpRing) & 1)); };

  if (warp == 17) {
    // ---- B producer
    if (lane == 0) {
      int issued = 0;
      for (int g = 0; g < n_blocks && !s_abort; ++g) {
        const int st = g % STG;
        if (g >= STG && !wait_done(g - STG)) {
          give_up();
          break;
        }
        uint8_t* dst = sB + (size_t)st * 2 * kTileBytes;
        const int ct = (int)((t0 + g / KB) % NT);
        const size_t off = ((size_t)ct * KB + g % KB) * kTileBytes;  // bytes
        mbar_expect_tx(&full[g % kSpRing], 2 * kTileBytes);
        bulk_g2s(dst, img_hi + off, kTileBytes, &full[g % kSpRing]);
        bulk_g2s(dst + kTileBytes, img_lo + off, kTileBytes, &full[g % kSpRing]);
        issued = g + 1;
      }
      if (s_abort)  // let the copies still in flight land before the CTA exits (bounded: the builders,
                    // who give up too, may leave their arrivals out)
        for (int g = max(0, issued - STG); g < issued; ++g) (void)wait_full(g);
    }
  } else if (warp == 16 || warp == 18) {
    // ---- MMA issuers: one thread the main products, one the cross terms.  An
    // MMA holds its thread for 65 cycles and more, and a wait on a barrier that
    // is ready takes 130: one thread for both needed 2100 cycles a block for
    // 1000 cycles of MMAs.
    const bool is_main = warp == 16;
    if (lane == 0) {
      int kb = 0, tile = 0;
      for (int g = 0; g < n_blocks && !s_abort; ++g) {
        const int ab = g & 1;
        if (!wait_full(g) || (is_main ? g >= 2 && !mbar_wait(&acc_empty[ab], (uint32_t)(((g >> 1) & 1) ^ 1))
                                      : kb == 0 && tile > 0 && !mbar_wait(&x_empty, (uint32_t)((tile - 1) & 1)))) {
          give_up();
          break;
        }
        tc_fence_after();
        const uint32_t ah = tmem + kSpA + (uint32_t)(ab * 64), al = ah + 32u;
        const uint32_t bh = smem_u32(sB + (size_t)(g % STG) * 2 * kTileBytes), bl = bh + kTileBytes;
        if (is_main) {
          const uint32_t acc_m = tmem + (uint32_t)(ab * TN);
#pragma unroll
          for (int s4 = 0; s4 < 4; ++s4) {
            const uint64_t d = smem_desc(bh + s4 * kKStepBytes);
            if (TF32) mma_tf32_ta(acc_m, ah + s4 * 8, d, idesc, s4 ? 1u : 0u);
            else mma_f16_ta(acc_m, ah + s4 * 8, d, idesc, s4 ? 1u : 0u);
          }
        } else {
          const uint32_t acc_x = tmem + kSpAccX;
#pragma unroll
          for (int s4 = 0; s4 < 4; ++s4) {
            const uint64_t dh = smem_desc(bh + s4 * kKStepBytes), dl = smem_desc(bl + s4 * kKStepBytes);
            const uint32_t more = (kb == 0 && s4 == 0) ? 0u : 1u;
            if (TF32) {
              mma_tf32_ta(acc_x, ah + s4 * 8, dl, idesc, more);
              mma_tf32_ta(acc_x, al + s4 * 8, dh, idesc, 1u);
            } else {
              mma_f16_ta(acc_x, ah + s4 * 8, dl, idesc, more);
              mma_f16_ta(acc_x, al + s4 * 8, dh, idesc, 1u);
            }
          }
        }
        mma_commit(&done[g % kSpRing]);
        if (++kb == KB) {
          kb = 0;
          ++tile;
        }
      }
      if (s_abort) {  // drain the MMAs already issued before TMEM is freed (bounded)
        uint64_t* mine = &drain[is_main ? 0 : 1];
        mma_commit(mine);
        (void)mbar_wait(mine, 0u);
      }
    }
  } else if (warp < 8) {
    // ---- A builders: thread = row 32 (warp % 4) + lane of the tile, K half warp / 4
    const int quad = warp & 3, half = warp >> 2;
    const int rr = 32 * quad + lane;
    const uint32_t a_base = tmem + kSpA + ((uint32_t)(quad * 32) << 16) + (uint32_t)(half * 16);
    bool ok = true;  // (a thread that gave up keeps to the barriers)
    // the rows of a row tile: this thread's cell and whether the tile's window
    // can be staged; starts the copies of the window (every builder thread)
    auto rows_of = [&](int rt, float* win) {
      SplitRows r;
      const int row = min(rt * TM + rr, n_rows - 1);
      r.cell = occ ? __ldg(occ + row) : row % n_x;
      r.pot = occ ? 0 : row / n_x;
      r.window = false;
      r.cell0 = 0;
      if (NET != 3) {
        int lo = r.cell, hi = r.cell;
        if (occ) {
          lo = __reduce_min_sync(0xffffffffu, lo);
          hi = __reduce_max_sync(0xffffffffu, hi);
          if (lane == 0) {
            s_min[warp] = lo;
            s_max[warp] = hi;
          }
          sp_builders_sync();
          lo = min(min(s_min[0], s_min[1]), min(s_min[2], s_min[3]));
          hi = max(max(s_max[0], s_max[1]), max(s_max[2], s_max[3]));
          sp_builders_sync();
          r.window = hi - lo < kWindowSpan;
        } else {
          lo = (rt * TM) % n_x;
          const int last = min(rt * TM + TM, n_rows) - 1;
          hi = last % n_x;
          r.window = (rt * TM) / n_x == last / n_x;  // one potential
        }
        r.cell0 = lo;
        if (r.window) {
          const float* Vp = V + (size_t)((occ ? 0 : (rt * TM) / n_x)) * n_x;
          const int n = hi - lo + 1 + 2 * h;
          for (int q = tid; q < n; q += kSpBuilders) {
            const long long l = (long long)lo - h + q;
            const bool in = l >= 0 && l < n_x;
            cp_async4(win + q, Vp + (in ? l : (l < 0 ? 0 : n_x - 1)), in || bc);
          }
        }
      }
      return r;
    };
    const size_t wf = split_window_floats(h);
    SplitRows cur = rows_of((int)(t0 / NT), s_win);
    cp_async_wait();
    sp_builders_sync();
    int wb = 0;
    // NET = 3: the rows of gVW and VWh come by 16-byte copies, eight threads a
    // row (128 bytes), kDenseStages - 1 blocks ahead: 32 rows read by one warp's
    // own loads, 16 bytes of each, took 192 us for 262144 rows of 128 columns.
    const bool dense_vec = NET == 3 && (h & 3) == 0 &&
                           ((reinterpret_cast<uintptr_t>(dense.gVW) | reinterpret_cast<uintptr_t>(dense.VWh)) & 15) == 0;
    constexpr size_t kDenseBuf = (size_t)TM * kDensePitch;
    int cd_rt = (int)(t0 / NT), cd_kb = 0, cd_ct = (int)(t0 % NT);  // the next block to copy
    auto copy_dense = [&](int g) {
      if (g < n_blocks) {
        const int r0 = tid >> 3, col = 4 * (tid & 7), k0 = cd_kb * KBLK;
        float* dst = s_win + (size_t)(g % kDenseStages) * 2 * kDenseBuf + r0 * kDensePitch + col;
        size_t o = (size_t)(cd_rt * TM + r0) * h + k0 + col;
        const int left = k0 + col < h ? n_rows - cd_rt * TM - r0 : 0;  // rows from r0 on
#pragma unroll
        for (int q = 0; q < TM / 32; ++q, o += 32 * (size_t)h) {
          const bool in = 32 * q < left;
          if (dense.gVW) cp_async16(dst + 32 * q * kDensePitch, dense.gVW + (in ? o : 0), in);
          if (dense.g_gamma) cp_async16(dst + kDenseBuf + 32 * q * kDensePitch, dense.VWh + (in ? o : 0), in);
        }
        if (++cd_kb == KB) {
          cd_kb = 0;
          if (++cd_ct == NT) {
            cd_ct = 0;
            ++cd_rt;
          }
        }
      }
      asm volatile("cp.async.commit_group;" ::: "memory");
    };
    if (dense_vec)
      for (int g = 0; g < kDenseStages - 1; ++g) copy_dense(g);
    for (int tile = 0; tile < n_my; ++tile) {
      const int rt = (int)((t0 + tile) / NT);
      // the next tile's window on its way while this tile is built
      const bool last = tile + 1 == n_my, same = last || (int)((t0 + tile + 1) / NT) == rt;
      SplitRows nxt = cur;
      if (!same) nxt = rows_of(rt + 1, s_win + (wb ^ 1) * wf);
      const float* w = s_win + wb * wf + h + (cur.cell - cur.cell0);
      const float* Vr = NET == 3 ? nullptr : V + (size_t)cur.pot * n_x;
#pragma unroll 1
      for (int kb = 0; kb < KB; ++kb) {
        const int g = tile * KB + kb, ab = g & 1;
        const int k0 = kb * KBLK + half * EPT;
        float dv[EPT];
        if (NET == 3) {
          const int row = rt * TM + rr;
          const bool on = row < n_rows;
          const float gg = on && dense.g_gamma ? __ldg(dense.g_gamma + row) : 0.f;
          float graw[EPT], vraw[EPT];
          if (dense_vec) {
            // this block's rows have arrived, and every thread has read the last block's
            asm volatile("cp.async.wait_group %0;" ::"n"(kDenseStages - 2) : "memory");
            sp_builders_sync();
            copy_dense(g + kDenseStages - 1);
            const float* src = s_win + (size_t)(g % kDenseStages) * 2 * kDenseBuf + rr * kDensePitch + half * EPT;
#pragma unroll
            for (int q = 0; q < EPT / 4; ++q) {
              const float4 a = dense.gVW ? *reinterpret_cast<const float4*>(src + 4 * q) : make_float4(0.f, 0.f, 0.f, 0.f);
              const float4 b = dense.g_gamma ? *reinterpret_cast<const float4*>(src + kDenseBuf + 4 * q)
                                             : make_float4(0.f, 0.f, 0.f, 0.f);
              graw[4 * q] = a.x, graw[4 * q + 1] = a.y, graw[4 * q + 2] = a.z, graw[4 * q + 3] = a.w;
              vraw[4 * q] = b.x, vraw[4 * q + 1] = b.y, vraw[4 * q + 2] = b.z, vraw[4 * q + 3] = b.w;
            }
          } else {
            const size_t o = (size_t)row * h + k0;
#pragma unroll
            for (int e = 0; e < EPT; ++e) {
              const bool in = on && k0 + e < h;
              graw[e] = in && dense.gVW ? __ldg(dense.gVW + o + e) : 0.f;
              vraw[e] = in && dense.g_gamma ? __ldg(dense.VWh + o + e) : 0.f;
            }
          }
          if (gg == 0.f) {
#pragma unroll
            for (int e = 0; e < EPT; ++e) dv[e] = graw[e];
          } else if (k0 + EPT <= h) {
            // multiplicities four columns at a time (the same for every lane)
#pragma unroll
            for (int q = 0; q < EPT / 4; ++q) {
              const int at = NET == 3 ? k0 + 4 * q : 0;
              const float4 cp = *reinterpret_cast<const float4*>(s_cnt + at);
              const float4 cn = *reinterpret_cast<const float4*>(s_cnt + (NET == 3 ? kAdjMaxH : 0) + at);
              const float p4[4] = {cp.x, cp.y, cp.z, cp.w}, n4[4] = {cn.x, cn.y, cn.z, cn.w};
#pragma unroll
              for (int e = 0; e < 4; ++e) {
                const float x = vraw[4 * q + e];
                const float dg = x > 0.f ? p4[e] : (x < 0.f ? -n4[e] : 0.f);
                dv[4 * q + e] = __fadd_rn(graw[4 * q + e], __fmul_rn(gg, dg));
              }
            }
            if (k0 == 0) dv[0] = graw[0];  // (column 0 counts nowhere, whatever gg is)
          } else {
#pragma unroll
            for (int e = 0; e < EPT; ++e) {
              const int r = k0 + e;
              float v = graw[e];
              if (r > 0 && r < h) {
                const float x = vraw[e];
                const float dg = x > 0.f ? s_cnt[NET == 3 ? r : 0] : (x < 0.f ? -s_cnt[NET == 3 ? kAdjMaxH + r : 0] : 0.f);
                v = __fadd_rn(v, __fmul_rn(gg, dg));
              }
              dv[e] = v;
            }
          }
        } else if (cur.window) {
          a_run_window<NET == 3 ? 1 : NET, EPT>(w, h, cur.cell, k0, dv);
        } else if (STAGED) {
          float* stg = s_win + (split_row_stage_apart(h) ? 2 * wf : ((wb * wf + 3) & ~(size_t)3)) + warp * kRowStage;
          a_run_rows<NET == 3 ? 1 : NET, EPT>(V, n_x, bc, h, cur.cell, cur.pot * n_x, k0, stg, dv);
        } else {
#pragma unroll
          for (int e = 0; e < EPT; ++e) dv[e] = a_term<NET == 3 ? 1 : NET>(Vr, n_x, bc, h, cur.cell, k0 + e);
        }
        uint32_t hi[16], lo[16];
        if (TF32) {
#pragma unroll
          for (int e = 0; e < 16; ++e) {
            hi[e] = to_tf32(dv[e]);
            lo[e] = to_tf32(__fsub_rn(dv[e], __uint_as_float(hi[e])));
          }
        } else {
#pragma unroll
          for (int e = 0; e < 16; ++e) {
            const float x = dv[TF32 ? 0 : 2 * e], y = dv[TF32 ? 0 : 2 * e + 1];
            hi[e] = pack2<WMC_FP16>(x, y);
            lo[e] = pack2<WMC_FP16>(__fmul_rn(__fsub_rn(x, from_bits((uint16_t)(hi[e] & 0xffffu), WMC_FP16)), 2048.f),
                                    __fmul_rn(__fsub_rn(y, from_bits((uint16_t)(hi[e] >> 16), WMC_FP16)), 2048.f));
          }
        }
        if (ok && g >= 2) {
          ok = !s_abort && wait_done(g - 2);
          if (!ok) give_up();
        }
        ok = __all_sync(0xffffffffu, ok);  // (the TMEM stores are warp-collective)
        if (ok) {
          tc_fence_after();
          tmem_st16(a_base + (uint32_t)(ab * 64), hi);
          tmem_st16(a_base + (uint32_t)(ab * 64 + 32), lo);
          tmem_wait_st();
          tc_fence_before();
          __syncwarp();
          if (lane == 0) mbar_arrive(&full[g % kSpRing]);
        }
      }
      if (!same) {
        cp_async_wait();
        sp_builders_sync();
        wb ^= 1;
        cur = nxt;
      }
    }
  } else {
    // ---- drain and output: warp 8 + w reads lanes 32 (w % 4) .. + 31, columns 64 (w / 4) .. + 63
    const int dw = warp - 8, quad = dw & 3, ch = dw >> 2;
    const uint32_t t_base = tmem + ((uint32_t)(quad * 32) << 16) + (uint32_t)(ch * 64);
    float* stg = s_stage + dw * kWsStageFloats;
    const bool vec_ok = (h & 3) == 0 && (reinterpret_cast<uintptr_t>(VWh) & 15) == 0;
    bool ok = true;
    for (int tile = 0; tile < n_my && ok; ++tile) {
      float sacc[64];  // sum over the K blocks drained so far of A_hi B_hi
#pragma unroll
      for (int q = 0; q < 64; ++q) sacc[q] = 0.f;
      for (int kb = 0; kb < KB; ++kb) {
        const int g = tile * KB + kb, ab = g & 1;
        int okw = 1;
        if (lane == 0) okw = !s_abort && wait_done(g);
        if (__shfl_sync(0xffffffffu, okw, 0) == 0) {  // warp-uniform: the TMEM loads are warp-collective
          if (lane == 0) give_up();
          ok = false;
          break;
        }
        tc_fence_after();
        uint32_t r[2][16];
        tmem_ld16_issue(t_base + (uint32_t)(ab * TN), r[0]);
        tmem_ld16_issue(t_base + (uint32_t)(ab * TN) + 16u, r[1]);
        tmem_wait16(r[0]);
        tmem_wait16(r[1]);
#pragma unroll
        for (int q = 0; q < 32; ++q) sacc[q] = __fadd_rn(sacc[q], __uint_as_float(r[q >> 4][q & 15]));
        tmem_ld16_issue(t_base + (uint32_t)(ab * TN) + 32u, r[0]);
        tmem_ld16_issue(t_base + (uint32_t)(ab * TN) + 48u, r[1]);
        tmem_wait16(r[0]);
        tmem_wait16(r[1]);
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(&acc_empty[ab]);
#pragma unroll
        for (int q = 0; q < 32; ++q) sacc[32 + q] = __fadd_rn(sacc[32 + q], __uint_as_float(r[q >> 4][q & 15]));
      }
      if (!ok) break;
      // v = c (sum of the block products + 2^-11 x cross); every MMA of the tile is complete
#pragma unroll
      for (int p = 0; p < 4; ++p) {
        float x[16];
        tmem_ld16(t_base + kSpAccX + (uint32_t)(16 * p), x);
#pragma unroll
        for (int q = 0; q < 16; ++q)
          sacc[16 * p + q] = __fmul_rn(c, __fadd_rn(sacc[16 * p + q], __fmul_rn(x[q], kLoScale)));
      }
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(&x_empty);
      const int row0 = (int)((t0 + tile) / NT) * TM + quad * 32;
      const int col00 = (int)((t0 + tile) % NT) * TN + ch * 64;
#pragma unroll
      for (int p = 0; p < 4; ++p) {
        const int col0 = col00 + 16 * p;
        if (col0 < h) {  // uniform
          // 32 rows x 16 columns through shared memory, so that stores are whole 64-byte row segments
#pragma unroll
          for (int q = 0; q < 4; ++q)
            *reinterpret_cast<float4*>(stg + lane * 16 + 4 * (q ^ ((lane >> 1) & 3))) =
                make_float4(sacc[16 * p + 4 * q], sacc[16 * p + 4 * q + 1], sacc[16 * p + 4 * q + 2],
                            sacc[16 * p + 4 * q + 3]);
          __syncwarp();
#pragma unroll
          for (int i = 0; i < 4; ++i) {
            const int r2 = 8 * i + (lane >> 2), q = lane & 3;
            const float4 v = *reinterpret_cast<const float4*>(stg + r2 * 16 + 4 * (q ^ ((r2 >> 1) & 3)));
            const int grow = row0 + r2, gcol = col0 + 4 * q;
            if (grow < n_rows && gcol < h) {
              float* out = VWh + (size_t)grow * h + gcol;
              if (vec_ok) {
                *reinterpret_cast<float4*>(out) = v;
              } else {
                out[0] = v.x;
                if (gcol + 1 < h) out[1] = v.y;
                if (gcol + 2 < h) out[2] = v.z;
                if (gcol + 3 < h) out[3] = v.w;
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
  if (warp == 0) {
    tc_fence_after();
    tmem_dealloc(tmem, 512u);
  }
}

// ---------------------------------------------------------------- host side
struct TcImages {
  int KB, NT, KB32, KB2;     // 16-bit K blocks (64 values), column tiles, TF32 K blocks (32 values), N = 2 K blocks
  int KBa;                   // the adjoint's TF32 K blocks (K = h), Q <= 256 only (else 0)
  size_t bytes_per_image;    // NT * KB * kTileBytes (BF16, FP16 hi, FP16 lo)
  size_t bytes_per_image32;  // NT * KB32 * kTileBytes (TF32 hi, TF32 lo)
  size_t bytes_per_image2;   // NT * KB2 * kTileBytes (N = 2 network: BF16, FP16 hi, FP16 lo)
  size_t bytes_per_imagea;   // NT * KBa * kTileBytes (adjoint, TF32 hi, TF32 lo)
};

static int g_h(const wmc_params& p) { return p.Q / 2; }

static TcImages tc_geometry(const wmc_params& p) {
  TcImages g;
  const int h = p.Q / 2;
  g.KB = (h - 1 + TK - 1) / TK;
  if (g.KB < 1) g.KB = 1;
  g.NT = (h + TN - 1) / TN;
  g.KB32 = (h - 1 + 31) / 32;
  if (g.KB32 < 1) g.KB32 = 1;
  g.KB2 = (h + TK - 1) / TK;  // the N = 2 network's K = h pair offsets
  g.bytes_per_image = (size_t)g.NT * g.KB * kTileBytes;
  g.bytes_per_image32 = (size_t)g.NT * g.KB32 * kTileBytes;
  g.bytes_per_image2 = (size_t)g.NT * g.KB2 * kTileBytes;
  g.KBa = h <= kAdjMaxH ? (h + 31) / 32 : 0;
  g.bytes_per_imagea = (size_t)g.NT * g.KBa * kTileBytes;
  return g;
}

size_t tc_images_bytes(const wmc_params& p) {
  const TcImages g = tc_geometry(p);
  return 3 * g.bytes_per_image + 2 * g.bytes_per_image32 + 3 * g.bytes_per_image2 + 2 * g.bytes_per_imagea;
}

static const uint8_t* adjoint_images(const void* images, const TcImages& g) {
  return static_cast<const uint8_t*>(images) + 3 * g.bytes_per_image + 2 * g.bytes_per_image32 +
         3 * g.bytes_per_image2;
}

cudaError_t launch_init_tc_images(const wmc_params& p, void* images, cudaStream_t s) {
  const TcImages g = tc_geometry(p);
  uint16_t* base = static_cast<uint16_t*>(images);
  const size_t n16 = g.bytes_per_image / 2;
  k_init_tc_images<<<256, 256, 0, s>>>(p.Q, g.KB, g.NT, base, base + n16, base + 2 * n16, 1);
  uint32_t* b32 = reinterpret_cast<uint32_t*>(static_cast<uint8_t*>(images) + 3 * g.bytes_per_image);
  k_init_tc_images32<<<256, 256, 0, s>>>(p.Q, g.KB32, g.NT, b32, b32 + g.bytes_per_image32 / 4, 0);
  uint16_t* b2 = reinterpret_cast<uint16_t*>(static_cast<uint8_t*>(images) + 3 * g.bytes_per_image +
                                             2 * g.bytes_per_image32);
  const size_t n2 = g.bytes_per_image2 / 2;
  k_init_tc_images<<<256, 256, 0, s>>>(p.Q, g.KB2, g.NT, b2, b2 + n2, b2 + 2 * n2, 2);
  if (g.KBa) {
    uint32_t* ba = reinterpret_cast<uint32_t*>(const_cast<uint8_t*>(adjoint_images(images, g)));
    k_init_tc_images32<<<256, 256, 0, s>>>(p.Q, g.KBa, g.NT, ba, ba + g.bytes_per_imagea / 4, 1);
  }
  return cudaGetLastError();
}

// One persistent CTA per SM, fewer if there are fewer tiles.
template <bool TF32, int NET, bool STAGED>
static cudaError_t launch_split_as(const float* V, int n_x, int bc, int Q, const int* occ, const int* n_occ_dev,
                                   int n_occ_host, int max_rows, const void* img_hi, const void* img_lo, int KB, int NT,
                                   float c, float* out, unsigned int* flags, const DenseA& dense, cudaStream_t s) {
  const size_t sm = split_smem_bytes(Q / 2, NET, STAGED);
  const cudaError_t e = raise_smem_limit(reinterpret_cast<const void*>(k_rows_split<TF32, NET, STAGED>), sm);
  if (e != cudaSuccess) return e;
  const long long tiles = (long long)((max_rows + TM - 1) / TM) * NT;
  const unsigned grid = (unsigned)(tiles < num_sms() ? tiles : num_sms());
  k_rows_split<TF32, NET, STAGED><<<grid, kSpThreads, sm, s>>>(V, n_x, bc, Q, occ, n_occ_dev, n_occ_host, img_hi,
                                                               img_lo, KB, NT, c, out, flags, dense);
  return cudaGetLastError();
}

// The staged form where tiles may be without a window: lists from the host that
// leave cells out, of domains that no window spans, and rows over several
// potentials that tiles straddle.  With each thread reading its own row in such
// tiles (the plain form), a load touched 32 lines, and they ran up to 1.75 times as
// long as in the kernel that built passes of four K blocks: 37 random cells, Q =
// 2048, 3xTF32: 108 us there, 118 us plain, 60 us staged; 9000 permuted cells of
// 20000, Q = 1024, FP16 split: 240, 162 and 64 us, of the N = 2 network 172, 267 and
// 70 us; 33 x 700 rows, FP16 split: 148, 202 and 97 us.  Where all tiles have windows
// the staged form costs 3xTF32 more (16384 cells at Q = 1024 66.3 against 64.1 us,
// FP16 split nothing), and in the step loop its shared memory costs the kernels
// around it 20 us a step.  So the occupied lists of a step and lists of every cell
// take the plain form, and 3xTF32 lists of at least a quarter of the cells too: if
// they ascend, 128 of them span some 512 cells and have windows (in any order, 9000
// of 20000: 157 us plain, 71 us staged).  That exception ends where the kernel's
// shared memory leaves an L1 that does not hold the potential: 4500 permuted cells
// of 9001 at Q = 2048 took 240 us in the kernel before, 351 us plain, 127 us staged,
// against 3 to 5 % on lists that ascend.
template <bool TF32, int NET>
static cudaError_t launch_split(const float* V, int n_x, int bc, int Q, const int* occ, const int* n_occ_dev,
                                int n_occ_host, int max_rows, const void* img_hi, const void* img_lo, int KB, int NT,
                                float c, float* out, unsigned int* flags, const DenseA& dense, cudaStream_t s) {
  if (NET != 3) {
    const bool uncached = split_smem_bytes(Q / 2, NET, false) > 192 * 1024 && n_x > 7 * 1024;
    const bool left_out = (TF32 && !uncached ? 4ll : 1ll) * n_occ_host < n_x;
    if (occ ? !n_occ_dev && left_out && n_x > kWindowSpan : max_rows > n_x && n_x % TM != 0)
      return launch_split_as<TF32, NET, NET != 3>(V, n_x, bc, Q, occ, n_occ_dev, n_occ_host, max_rows, img_hi, img_lo, KB,
                                                  NT, c, out, flags, dense, s);
  }
  return launch_split_as<TF32, NET, false>(V, n_x, bc, Q, occ, n_occ_dev, n_occ_host, max_rows, img_hi, img_lo, KB, NT,
                                           c, out, flags, dense, s);
}

// Abar = c Gbar S^T on the 3xTF32 split kernel (NET = 3), rows = n_pot n_x
// implicit rows; Q <= 256.
cudaError_t launch_adjoint_abar_tc(const wmc_params& p, int rows, const float* VWh, const float* gVW,
                                   const float* g_gamma, const void* images, float* Abar, unsigned int* flags,
                                   cudaStream_t s) {
  const TcImages g = tc_geometry(p);
  if (!g.KBa) return cudaErrorNotSupported;
  if (rows <= 0) return cudaSuccess;
  const uint8_t* ba = adjoint_images(images, g);
  DenseA d;
  d.gVW = gVW;
  d.VWh = VWh;
  d.g_gamma = g_gamma;
  d.ca = p.n_M / p.Q;
  d.cb = p.n_M - d.ca * p.Q;
  d.cr0 = ((-(p.n_M / 2)) % p.Q + p.Q) % p.Q;
  const float c = (float)(-2.0 / (kHbarEVs * (double)p.Q));
  return launch_split<true, 3>(nullptr, rows, 0, p.Q, nullptr, nullptr, rows, rows, ba, ba + g.bytes_per_imagea, g.KBa,
                               g.NT, c, Abar, flags, d, s);
}

// The form behind a requested precision: WMC_FP32 takes the 3xTF32 split
// kernel (N = 1 network, where its shared memory holds the window) for
// Q > 256, and for Q >= 128 when the rows fill a wave of 128-row tiles on
// every SM (rows > 0: the row entry points; measured 2.4x faster than the
// CUDA cores at Q = 256 over 262144 rows, error 1.6e-7 against 2.2e-7);
// else the CUDA-core form.  WMC_FP32_SIMT is always the CUDA-core form.  The
// result is the internal code: WMC_FP32 then always means the CUDA cores.
int resolve_precision(const wmc_params& p, int prec, int net, long long rows) {
  if (prec == WMC_FP32_SIMT) return WMC_FP32;
  if (prec != WMC_FP32 || net != 1) return prec;
  if (p.Q <= 256 && !(p.Q >= 128 && rows >= (long long)TM * num_sms())) return prec;
  return WMC_TF32X3;
}

// The N = 2 network (net = 2) runs on the warp-specialised BF16 / FP16 and
// FP16-split kernels with its own operand images and A builder; other forms
// return cudaErrorNotSupported for it.
template <int NET>
static cudaError_t launch_tc_net(const wmc_params& p, int prec, const float* V, const int* occ, const int* n_occ_dev,
                                 int n_occ_host, int max_rows, const uint16_t* base, int KB, const TcImages& g,
                                 float* VWh, unsigned int* flags, cudaStream_t s);

cudaError_t launch_kernel_eval_tc(const wmc_params& p, int prec, const float* V, const int* occ, const int* n_occ_dev,
                                  int n_occ_host, int max_rows, const void* images, float* VWh, unsigned int* flags,
                                  cudaStream_t s, int net) {
  if (max_rows <= 0) return cudaSuccess;
  const TcImages g = tc_geometry(p);
  if (net == 2) {
    const uint16_t* b2 = reinterpret_cast<const uint16_t*>(static_cast<const uint8_t*>(images) +
                                                           3 * g.bytes_per_image + 2 * g.bytes_per_image32);
    return launch_tc_net<2>(p, prec, V, occ, n_occ_dev, n_occ_host, max_rows, b2, g.KB2, g, VWh, flags, s);
  }
  const uint16_t* base = static_cast<const uint16_t*>(images);
  if (prec == WMC_BF16 || prec == WMC_FP16 || prec == WMC_FP16_SPLIT) {
    const cudaError_t e = launch_tc_net<1>(p, prec, V, occ, n_occ_dev, n_occ_host, max_rows, base, g.KB, g, VWh,
                                           flags, s);
    if (e != cudaErrorNotSupported) return e;
  }
  const size_t n16 = g.bytes_per_image / 2;
  const float c = (float)(-2.0 / (kHbarEVs * (double)p.Q));
  dim3 grid((max_rows + TM - 1) / TM, g.NT);
  if (prec == WMC_BF16) {
    const size_t sm = tc_smem_bytes(g_h(p));
    raise_smem_limit(reinterpret_cast<const void*>(k_kernel_eval_tc<WMC_BF16>), sm);
    k_kernel_eval_tc<WMC_BF16><<<grid, 128, sm, s>>>(V, p.n_x, p.bc_potential, p.Q, occ, n_occ_dev, n_occ_host,
                                                     base, g.KB, c, VWh, flags);
  } else if (prec == WMC_FP16) {
    const size_t sm = tc_smem_bytes(g_h(p));
    raise_smem_limit(reinterpret_cast<const void*>(k_kernel_eval_tc<WMC_FP16>), sm);
    k_kernel_eval_tc<WMC_FP16><<<grid, 128, sm, s>>>(V, p.n_x, p.bc_potential, p.Q, occ, n_occ_dev, n_occ_host,
                                                     base + n16, g.KB, c, VWh, flags);
  } else if (prec == WMC_TF32X3) {
    const uint8_t* b32 = reinterpret_cast<const uint8_t*>(images) + 3 * g.bytes_per_image;
    return launch_split<true, 1>(V, p.n_x, p.bc_potential, p.Q, occ, n_occ_dev, n_occ_host, max_rows, b32,
                                 b32 + g.bytes_per_image32, g.KB32, g.NT, c, VWh, flags, DenseA{}, s);
  } else {
    return cudaErrorInvalidValue;
  }
  return cudaGetLastError();
}

template <int NET>
static cudaError_t launch_tc_net(const wmc_params& p, int prec, const float* V, const int* occ, const int* n_occ_dev,
                                 int n_occ_host, int max_rows, const uint16_t* base, int KB, const TcImages& g,
                                 float* VWh, unsigned int* flags, cudaStream_t s) {
  const size_t n16 = (size_t)g.NT * KB * kTileBytes / 2;
  const float c = (float)(-2.0 / (kHbarEVs * (double)p.Q));
  const int row_tiles = (max_rows + TM - 1) / TM;
  if ((prec == WMC_BF16 || prec == WMC_FP16) && KB <= kTaMaxKB && ta_smem_bytes(g_h(p)) <= 226 * 1024) {
    // A in tensor memory.  The 128-column tiles are split over grid.y by the
    // factor that minimises waves x per-CTA work, with the fixed part of a CTA
    // (set-up and building A) counted as three column tiles.
    const uint16_t* img = prec == WMC_BF16 ? base : base + n16;
    const long long sms = num_sms();
    int n_split = 1;
    long long best = -1;
    for (int ns = 1; ns <= g.NT; ns *= 2) {
      const long long waves = ((long long)row_tiles * ns + sms - 1) / sms;
      const long long cost = waves * (3 + (long long)((g.NT + ns - 1) / ns));
      if (best < 0 || cost < best) {
        best = cost;
        n_split = ns;
      }
    }
    const size_t sm = ta_smem_bytes(g_h(p));
    const void* fn = prec == WMC_BF16 ? reinterpret_cast<const void*>(k_kernel_eval_tc_ta<WMC_BF16, NET>)
                                      : reinterpret_cast<const void*>(k_kernel_eval_tc_ta<WMC_FP16, NET>);
    const cudaError_t e = raise_smem_limit(fn, sm);
    if (e != cudaSuccess) return e;
    const dim3 grid(row_tiles, n_split);
    if (prec == WMC_BF16)
      k_kernel_eval_tc_ta<WMC_BF16, NET><<<grid, kTaThreads, sm, s>>>(V, p.n_x, p.bc_potential, p.Q, occ, n_occ_dev,
                                                                      n_occ_host, img, KB, g.NT, n_split, c, VWh,
                                                                      flags);
    else
      k_kernel_eval_tc_ta<WMC_FP16, NET><<<grid, kTaThreads, sm, s>>>(V, p.n_x, p.bc_potential, p.Q, occ, n_occ_dev,
                                                                      n_occ_host, img, KB, g.NT, n_split, c, VWh,
                                                                      flags);
    return cudaGetLastError();
  }
  if (prec == WMC_FP16_SPLIT)
    return launch_split<false, NET>(V, p.n_x, p.bc_potential, p.Q, occ, n_occ_dev, n_occ_host, max_rows, base + n16,
                                    base + 2 * n16, KB, g.NT, c, VWh, flags, DenseA{}, s);
  return cudaErrorNotSupported;
}

}  // namespace wmc

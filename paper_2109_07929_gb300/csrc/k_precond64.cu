// FP64 form of the preconditioner apply z = P^-1 r (eqs. P, block, M; Section 3.2).
//
// In the Kronecker eigenbasis of G_t = I (x) G_r and G_b = G_c (x) I the operator P is a
// 2x2 block per mode (i', k'): [[mu_k' + a1, -a1], [-a2, nu_i' + a2]].  The apply is four
// dense transforms per layer with a per-mode 2x2 inverse in the middle:
//   T1^T = (X Q_r)^T,  X_hat = Q_c^T X Q_r,  Y_hat = modes^-1 X_hat,
//   E^T = (Y_hat Q_r^T)^T,  Z = Q_c Y_hat Q_r^T,
// each one the block-transposed GEMM O[blk][c][r] = sum_k A[blk][r][k] Bm[c][k].  This file
// holds it with FP64 results; the mixed-precision form lives in k_precond_tc.cu.
//
// The FP64 pipe gives 1.05 TFLOP/s, so the GEMM runs on the BF16 tensor cores, after Ozaki,
// Ogita, Oishi and Rump ("Error-free transformations of matrix multiplication by using fast
// routines of matrix multiplication and its applications", Numer. Algorithms 59, 2012) and its
// tensor-core form by Mukunoki, Ozaki, Ogita and Imamura (ISC 2020): every row of A and of Bm is
// scaled by a power of two and cut into 8 slices of signed 7-bit digits,
//   x = 2^(e + 2) sum_s a_s 128^-(s + 1),   |a_s| <= 64,   2^e <= row maximum < 2^(e + 1),
// which BF16 holds exactly; products of digits are integers of at most 2^12, so that the FP32
// accumulators of the tensor core hold exactly what the up to 8 slice products of one weight
// d = s + t sum over K <= 512 (8 x 512 x 2^12 = 2^24); and the sums of weights 0 .. 7 (36 of the
// 64 slice products) are joined to one FP64 result per 512 of K, rounded once.
//
// What is lost, per product of entries and in units of 2^(ea + eb): the 28 products of weights 8
// and up, at most 7.1 x 2^-54 (seven of weight 8 with 2^-54 each), and the rounding of the two
// entries to multiples of 2^(e - 54), at most 2 x 2^-54: below 9.1 x 2^-54 = 2^-50.8, and 1.1 x
// 2^-54 in the mean square over evenly spread digits.  So the error is relative to the maxima of
// the rows, not to the entries: one 2^-20 of its row's maximum keeps 35 bits, one below 2^-56
// none, where a chain of FMAs keeps 53 of each and rounds at 2^-53 of its partial sums.  The
// apply's error in the norm falls all the same (96 x 160 to 40 x 600, random, spike, one-column,
// graded, decaying and smooth right-hand sides, a from 2e-5 to 5: 2.7e-16 to 8.2e-16 of |z|, the
// chain's 7.2e-16 to 2.1e-15); single components move both ways: in a spike's far field and a
// few of a smooth z up to 6 times the chain's error, most others below it.
// One apply (four transforms), against the FMA kernel: 512 x 512, 4 vectors 520 us (8300),
// 1024 x 1024 933 us (16500), 64 x 64 135 us (324), 16 x 16 110 us (126).
#include <cuda.h>

#include <algorithm>

#include "bits.cuh"
#include "mca_internal.cuh"
#include "precond_tc.h"
#include "tc_ptx.cuh"

namespace mca {

namespace {

using namespace tc;

constexpr int kSlices = 8;        // digits per entry
constexpr int kDigit = 7;         // bits per digit
constexpr int kOzM = 128;         // output rows per tile (TMEM lanes)
constexpr int kOzN = 64;          // output columns per tile: 8 accumulators fill the TMEM
constexpr int kOzK = 32;          // K per stage (64-byte rows, 64-byte swizzle)
constexpr int kOzThreads = 256;
constexpr int kOzA = kOzM * kOzK * 2, kOzB = kOzN * kOzK * 2;      // one slice's tile
constexpr int kOzStage = kSlices * (kOzA + kOzB);                  // 96 KB
constexpr int kOzStages = 2;
constexpr int kOzBar = kOzStages * kOzStage;
constexpr int kOzSmem = kOzBar + 256 + 1024;
constexpr int kOzKMax = 512;      // largest K whose 8 products per weight FP32 sums hold exactly
constexpr int kBadRow = 0x7FFFFFFF;   // exponent of a row with an infinity or a NaN, which has
                                      // no slices: its results are the plain FP64 sums
constexpr int kZeroRow = -0x7FFFFFFF; // and of a row of zeros

// Row slicing: a warp per row, `rows` of them (of the batch at hand; the operand holds
// plane / Kp).  out[s][row][k] (BF16, K padded to Kp with zeros) and exps[row].  Row r of block
// blk = 2 b + layer starts at A + b a.bs + layer a.ls + r a.ld.  Integer arithmetic only: the
// entry's mantissa shifted to a 56-bit fixed-point number in units of 2^(e - 54), its digits
// taken from the low end with a carry.
__global__ void __launch_bounds__(256)
k_slice_rows(const double* __restrict__ A, BlkAddr a, int R, int K, int Kp, int rows,
             size_t plane, const VecCtl* __restrict__ ctl, __nv_bfloat16* __restrict__ out,
             int* __restrict__ exps) {
  const int row = blockIdx.x * 8 + (threadIdx.x >> 5), lane = threadIdx.x & 31;
  if (row >= rows) return;
  const int blk = row / R, r = row - blk * R, b = blk >> 1;
  if (ctl != nullptr && !ctl[b].gm_active) return;
  const double* x = A + (size_t)b * a.bs + (size_t)(blk & 1) * a.ls + (size_t)r * a.ld;
  uint32_t top = 0;                                  // largest |high word| of the row
  bool any = false;
#pragma unroll 4
  for (int k = lane; k < K; k += 32) {
    const uint32_t hi = (uint32_t)__double2hiint(x[k]) & 0x7FFFFFFFu;
    top = max(top, hi);
    any |= (hi | (uint32_t)__double2loint(x[k])) != 0u;
  }
  top = __reduce_max_sync(0xffffffffu, top);
  any = __any_sync(0xffffffffu, any);
  // rows near the bottom of the FP64 range are lifted by 2^512 first
  const bool low = any && (top >> 20) < 128u;
  const bool bad = (top >> 20) == 0x7FFu;
  if (low) {
    top = 0;
    for (int k = lane; k < K; k += 32)
      top = max(top, (uint32_t)__double2hiint(x[k] * 0x1p+512) & 0x7FFFFFFFu);
    top = __reduce_max_sync(0xffffffffu, top);
  }
  const int E = (int)(top >> 20);                    // biased exponent of the largest entry
  if (lane == 0) exps[row] = bad ? kBadRow : (any ? E - 1023 - (low ? 512 : 0) : kZeroRow);
  __nv_bfloat16* o = out + (size_t)row * Kp;
  for (int k0 = 2 * lane; k0 < Kp; k0 += 64) {
    uint32_t w[kSlices] = {};
#pragma unroll
    for (int q = 0; q < 2; ++q) {
      const int k = k0 + q;
      double v = (k < K && !bad) ? x[k] : 0.0;
      if (low) v *= 0x1p+512;
      const uint32_t hi = (uint32_t)__double2hiint(v);
      const int ex = (int)((hi >> 20) & 0x7FFu), sh = E - ex;
      if (ex == 0 || sh > 57) continue;              // zero, or below half a unit
      unsigned long long f = ((unsigned long long)((hi & 0xFFFFFu) | 0x100000u) << 34) |
                             ((unsigned long long)(uint32_t)__double2loint(v) << 2);
      if (sh > 0) f = (f + (1ull << (sh - 1))) >> sh;
      // digits in [-64, 63] from the low end; the last one is what is left, at most 64
      uint32_t part = (uint32_t)f & 0xFFFFFFFu;
      const uint32_t high = (uint32_t)(f >> 28);
      const uint32_t sg = hi & 0x80000000u;
#pragma unroll
      for (int s = kSlices - 1; s >= 0; --s) {
        if (s == 3) part += high;
        const int d = (s > 0) ? (int)((part + 64u) & 127u) - 64 : (int)part;
        part = (uint32_t)((int)part - d) >> kDigit;
        const float g = __uint_as_float(0x4B400000u + (uint32_t)d) - 12582912.f;
        const uint32_t h = (__float_as_uint(g) ^ (d != 0 ? sg : 0u)) >> 16;
        w[s] |= h << (16 * q);
      }
    }
#pragma unroll
    for (int s = 0; s < kSlices; ++s)
      *reinterpret_cast<uint32_t*>(o + s * plane + k0) = w[s];
  }
}

// 8 columns of this warp's 32 TMEM lanes, without the wait
__device__ __forceinline__ void tmem_ld8(uint32_t taddr, uint32_t (&v)[8]) {
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
               : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]),
                 "=r"(v[6]), "=r"(v[7])
               : "r"(taddr));
}

// sum_q acc[q] 128^(3 - q), an integer below 2^51, as FP64: added up in two 32-bit words and
// read through the bits of 1.5 2^52 + v
__device__ __forceinline__ double join4(int a0, int a1, int a2, int a3) {
  const long long v = ((long long)a0 << 21) + ((long long)a1 << 14) + ((long long)a2 << 7) + a3;
  return __longlong_as_double(0x4338000000000000LL + v) - 6755399441055744.0;
}

// x 2^e with the exponent added on the integer pipe
__device__ __forceinline__ double scale2(double x, int e) {
  const uint32_t hi = (uint32_t)__double2hiint(x);
  const int ex = (int)((hi >> 20) & 0x7FFu);
  if (ex == 0) return x;                             // (x is an integer sum: zero)
  if (ex + e >= 1 && ex + e <= 2046)
    return __hiloint2double((int)(hi + ((uint32_t)e << 20)), __double2loint(x));
  return scalbn(x, e);
}

struct OzArgs {
  int R, C, K0, K1;          // output rows per block, columns, this launch's K range
  const int *ea, *eb;        // exponents of A's rows (all blocks) and of Bm's
  const double *A, *Bm;      // the operands themselves, K entries a row
  BlkAddr a;
  int K;
  double* O;
  BlkAddr o;
  const VecCtl* ctl;
  int* err;
};

// One 128 x 64 output tile per CTA: 8 accumulators (one per weight) fill the TMEM; thread 0
// streams both operands' 8 slices with one TMA box each (96 KB per 32 of K, two stages),
// thread 32 issues the 36 slice products of a stage, and the 8 warps join the accumulators.
// Bound: shared-memory reads of the operands (N = 64: 6 KB per MMA of 32 clocks' work; 512 x 512,
// 4 vectors: 65 % of their rate, the tensor pipe active 35 %) and a second wave two thirds full.
// ADD: a later K range, added to O.
template <bool ADD>
__global__ void __launch_bounds__(kOzThreads, 1)
k_gemm_sliced(const __grid_constant__ CUtensorMap tmA, const __grid_constant__ CUtensorMap tmB,
              OzArgs p) {
  const int blk = blockIdx.z, b = blk >> 1;
  if (p.ctl != nullptr && !p.ctl[b].gm_active) return;
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>(
      (reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
  uint64_t* full = reinterpret_cast<uint64_t*>(smem + kOzBar);
  uint64_t* empty = full + kOzStages;
  uint64_t* accum = empty + kOzStages;
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(accum + 1);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int r0 = blockIdx.x * kOzM, c0 = blockIdx.y * kOzN;
  const int nkb = (p.K1 - p.K0 + kOzK - 1) / kOzK;
  if (threadIdx.x == 0) {
    for (int s = 0; s < kOzStages; ++s) {
      mbar_init(&full[s], 1);
      mbar_init(&empty[s], 1);
    }
    mbar_init(accum, 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                     smem_u32(tmem_slot)),
                 "r"((uint32_t)(kSlices * kOzN))
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *tmem_slot;
  if (threadIdx.x == 0) {
    for (int kb = 0; kb < nkb; ++kb) {
      const int s = kb % kOzStages;
      if (!mbar_wait(&empty[s], ((uint32_t)(kb / kOzStages) & 1u) ^ 1u)) {
        record_error(p.err, MCA_ERR_TIMEOUT);
        break;
      }
      uint8_t* st = smem + s * kOzStage;
      mbar_expect_tx(&full[s], (uint32_t)kOzStage);
      const int k0 = p.K0 + kb * kOzK;
      tma_load_3d(st, &tmA, k0, blk * p.R + r0, 0, &full[s]);
      tma_load_3d(st + kSlices * kOzA, &tmB, k0, c0, 0, &full[s]);
    }
  } else if (threadIdx.x == 32) {
    constexpr uint32_t idesc = idesc_bf16(kOzM, kOzN);
    bool ok = true;
    for (int kb = 0; kb < nkb; ++kb) {
      const int s = kb % kOzStages;
      if (!mbar_wait(&full[s], (uint32_t)(kb / kOzStages) & 1u)) {
        record_error(p.err, MCA_ERR_TIMEOUT);
        ok = false;
        break;
      }
      tc_fence_after();
      const uint8_t* sa = smem + s * kOzStage;
      const uint8_t* sb = sa + kSlices * kOzA;
#pragma unroll
      for (int kk = 0; kk < kOzK / 16; ++kk) {
#pragma unroll
        for (int i = 0; i < kSlices; ++i) {
          const uint64_t ad = sw64_desc(sa + i * kOzA + kk * 32);
#pragma unroll
          for (int j = 0; i + j < kSlices; ++j)
            umma(tmem + (uint32_t)((i + j) * kOzN), ad, sw64_desc(sb + j * kOzB + kk * 32), idesc,
                 (kb > 0 || kk > 0 || i > 0) ? 1u : 0u);
        }
      }
      umma_commit(&empty[s]);
    }
    if (ok) umma_commit(accum);
  }
  __syncwarp();
  const bool have = __syncthreads_and(mbar_wait(accum, 0) ? 1 : 0) != 0;
  if (!have && threadIdx.x == 0) record_error(p.err, MCA_ERR_TIMEOUT);
  if (have) {
    tc_fence_after();
    const int q = warp & 3, half = warp >> 2;
    const int r = r0 + q * 32 + lane;
    const bool rok = r < p.R;
    const int ea = rok ? p.ea[blk * p.R + r] : kZeroRow;
    const double* A = p.A + (size_t)b * p.a.bs + (size_t)(blk & 1) * p.a.ls + (size_t)r * p.a.ld;
    double* O = p.O + (size_t)b * p.o.bs + (size_t)(blk & 1) * p.o.ls + r;
    const uint32_t base = tmem + ((uint32_t)(q * 32) << 16) + (uint32_t)(half * 32);
#pragma unroll 1
    for (int cc = 0; cc < 4; ++cc) {
      uint32_t v[kSlices][8];
#pragma unroll
      for (int d = 0; d < kSlices; ++d) tmem_ld8(base + d * kOzN + cc * 8, v[d]);
      asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
      for (int j = 0; j < 8; ++j) {
        const int c = c0 + half * 32 + cc * 8 + j;
        if (c >= p.C || !rok) continue;
        double* dst = O + (size_t)c * p.o.ld;
        if (ea == kBadRow) {                           // (in the first K range)
          if (ADD) continue;
          const double* q = p.Bm + (size_t)c * p.K;
          double x = 0.0;
#pragma unroll 1
          for (int k = 0; k < p.K; ++k) x = fma(A[k], q[k], x);
          *dst = x;
          continue;
        }
        const int eb = p.eb[c];
        int t[kSlices];
#pragma unroll
        for (int d = 0; d < kSlices; ++d) t[d] = __float2int_rn(__uint_as_float(v[d][j]));
        // 2^(ea + eb + 4) sum_d t_d 128^-(d + 2)
        const double hi = join4(t[0], t[1], t[2], t[3]), lo = join4(t[4], t[5], t[6], t[7]);
        double x = fma(lo, 0x1p-28, hi);
        x = (ea == kZeroRow || eb == kZeroRow) ? 0.0 : scale2(x, ea + eb + 4 - 5 * kDigit);
        *dst = ADD ? *dst + x : x;
      }
    }
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 1) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem),
                 "r"((uint32_t)(kSlices * kOzN))
                 : "memory");
  }
}

// [y_t; y_b] = (1/det) [[nu + a2, a1], [a2, mu + a1]] [x_t; x_b],
// det = mu nu + mu a2 + nu a1 = (mu + a1)(nu + a2) - a1 a2, with a1 = a2 = a.
__global__ void k_modes_2x2(double* __restrict__ Xh, const double* __restrict__ mu,
                            const double* __restrict__ nu, int m, int n,
                            const VecCtl* __restrict__ ctl, int kidx) {
  const int b = blockIdx.y;
  if (!ctl[b].gm_active) return;
  const double a = ctl[b].a;
  // scale of the unnormalised input basis vector (kidx < 0: none)
  const double sc = (kidx >= 0) ? ctl[b].s[kidx] : 1.0;
  const size_t mn = (size_t)m * n;
  double* xt = Xh + (size_t)b * 2 * mn;
  double* xb = xt + mn;
  for (size_t e = blockIdx.x * (size_t)blockDim.x + threadIdx.x; e < mn;
       e += (size_t)gridDim.x * blockDim.x) {
    const int ip = (int)(e / n), kp = (int)(e - (size_t)ip * n);
    const double M = mu[kp], N = nu[ip];
    const double f = sc / (M * N + M * a + N * a);
    const double u = xt[e], v = xb[e];
    xt[e] = ((N + a) * u + a * v) * f;
    xb[e] = (a * u + (M + a) * v) * f;
  }
}

}  // namespace

size_t sliced_elems(size_t rows, int K) {
  return kSlices * rows * ((size_t)(K + kOzK - 1) / kOzK * kOzK);
}

int make_sliced(SlicedOperand* op, __nv_bfloat16* buf, int* exps, int rows, int K, bool is_a) {
  op->buf = buf;
  op->exps = exps;
  op->rows = rows;
  op->K = K;
  op->Kp = (K + kOzK - 1) / kOzK * kOzK;
  if (!tc::make_map_slices(&op->map, buf, op->Kp, rows, kSlices, is_a ? kOzM : kOzN))
    return MCA_ERR_UNSUPPORTED;
  for (auto kern : {k_gemm_sliced<false>, k_gemm_sliced<true>})
    if (cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, kOzSmem) !=
        cudaSuccess)
      return MCA_ERR_CUDA;
  return MCA_OK;
}

void launch_slice_rows(const double* A, BlkAddr a, int R, const SlicedOperand& op, int rows,
                       const VecCtl* ctl, cudaStream_t s) {
  k_slice_rows<<<(rows + 7) / 8, 256, 0, s>>>(A, a, R, op.K, op.Kp, rows,
                                              (size_t)op.rows * op.Kp, ctl, op.buf, op.exps);
}

int launch_gemm_sliced(const SlicedOperand& A, const SlicedOperand& Bm, const double* A64,
                       BlkAddr a, const double* Bm64, double* O, BlkAddr o, int B, int R, int C,
                       const VecCtl* ctl, int* err, cudaStream_t s) {
  const dim3 grid((R + kOzM - 1) / kOzM, (C + kOzN - 1) / kOzN, 2 * B);
  int launches = 0;
  for (int k0 = 0; k0 < A.Kp; k0 += kOzKMax, ++launches) {
    const OzArgs p{R, C, k0, std::min(A.Kp, k0 + kOzKMax), A.exps, Bm.exps, A64, Bm64, a,
                   A.K, O, o, ctl, err};
    if (k0 == 0)
      k_gemm_sliced<false><<<grid, kOzThreads, kOzSmem, s>>>(A.map, Bm.map, p);
    else
      k_gemm_sliced<true><<<grid, kOzThreads, kOzSmem, s>>>(A.map, Bm.map, p);
  }
  return launches;
}

void launch_modes_2x2_f64(double* Xh, const double* mu, const double* nu, int m, int n,
                          const VecCtl* ctl, int B, int kidx, cudaStream_t s) {
  const size_t mn = (size_t)m * n;
  int nb = (int)((mn + 255) / 256);
  if (nb > 1216) nb = 1216;
  k_modes_2x2<<<dim3(nb, B), 256, 0, s>>>(Xh, mu, nu, m, n, ctl, kidx);
}

}  // namespace mca

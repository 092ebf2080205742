// The paper's own evaluation of the preconditioner (Section 3.2, eqs. block, Mhat,
// G2hat, M-1hat, 2matrix1-4) and the two comparison preconditioners of its Table 1
// (Jacobi, none), all in FP64 on CUDA cores.
//
// Block inversion with B = -a1 I (eq. block):
//   z_t = M^-1 (r_b + (G_b + a2 I) r_t / a1),   z_b = ((G_t + a1 I) z_t - r_t) / a1,
// with the Schur complement approximated as M_hat = (G_2 / a1) (x) G_1 (eq. Mhat, the
// whole G_2 divided by a1), so M_hat^-1 W = a1 G_2^-1 W G_1^-1 on the row-major m x n grid
// W (eq. 2matrix4): tridiagonal solves along every column (G_2 = G_c + a2 I) and then
// along every row (G_1 = G_r + a1 I).  G_b + a2 I is G_2 along the columns, so
// M_hat^-1 (r_b + G_2 r_t / a1) = (a1 G_2^-1 r_b + r_t) G_1^-1, and with G_t + a1 I = G_1 along
// the rows z_b = ((a1 G_2^-1 r_b + r_t) - r_t) / a1: the same z is
//   z_b = G_2^-1 r_b,   z_t = (r_t + a1 z_b) G_1^-1,
// one solve per layer, without the two operator applies and their cancellation (z_b's error
// falls from 5e-10 to 6e-16 relative at 1024 x 1024).
//
// A tridiagonal solve T x = w, T = tridiag(-g, d_j + a, -g) = L U with pivots piv_j, is two
// first-order recurrences,
//   y_j = w_j + q_{j-1} y_{j-1},   x_j = q_j x_{j+1} + y_j / piv_j,   q_j = g / piv_j,
// and one thread per row or column walking them was a chain of 2 n loads and FP64
// operations with 4096 threads on the chip.  Each line is cut into 32 chunks instead: a chunk
// runs its recurrence from a zero carry, the 32 carries are combined by a scan with
// precomputed products of q, and every entry gets its share of the carry (product of the
// chunk's q up to it, also precomputed) in one FMA: 5 FP64 instructions per entry and solve
// against 3, with 32 times the threads.  All products are of factors 0 < q < 1, so nothing
// is amplified.  The factors depend on a only and are built once per GMRES cycle, in closed
// form.
// Bound: the FP64 pipe (13 instructions per cell; busy 79 % in the columns, 82 % in the rows).
// 1024 x 1024, 4 vectors, per apply: 1330 us (factor 460, columns 502, rows 273, stencils 97),
// now 115 (51 and 64) and the factors 30 us once per cycle.
#include "mca_internal.cuh"

namespace mca {

namespace {

constexpr int kT = 256;
constexpr int kChunks = 32;

// Factors of one line operator of `len` nodes in chunks of L = ceil(len / 32): arrays of 32 L
// doubles, entry (chunk c, k) at index [k][c] for the row operator (a warp's lanes are a
// row's chunks) or [c][k] = node order for the column operator:
//   lo   q_{j-1} (0 at a chunk's start: the carry enters through ylo)
//   ylo  (product of q_{i-1}, i = chunk start .. j) / piv_j
//   ip   1 / piv_j
//   q    q_j (0 at a chunk's end)
//   xhi  product of q_i, i = j .. chunk end
// then the scans' factors, 5 x 32 each: level s of the forward scan multiplies the carry of
// chunk c - 2^s by the products of chunks c - 2^s + 1 .. c, the backward scan mirrored.
struct LineFac {
  const double *lo, *ylo, *ip, *q, *xhi, *fwd, *bwd;
};

__host__ __device__ __forceinline__ int chunk_len(int len) {
  return (len + kChunks - 1) / kChunks;
}

__device__ __forceinline__ LineFac line_fac(const double* base, int len) {
  const size_t N = (size_t)kChunks * chunk_len(len);
  return LineFac{base, base + N, base + 2 * N, base + 3 * N, base + 4 * N, base + 5 * N,
                 base + 5 * N + 5 * kChunks};
}

__host__ __device__ __forceinline__ size_t line_fac_size(int len) {
  return 5 * (size_t)kChunks * chunk_len(len) + 10 * kChunks;
}

// One block per vector: half of its threads the row operator G_1 (over j), half the column
// operator G_2 (over i).  The pivots are a continued fraction, piv_j = d_j + a - g^2 /
// piv_{j-1}, which one thread walked at 0.45 us a step.  Inside a line all d_j are 2 g, so the
// leading minors p_j (of T / g) have a closed form: with 4 sinh^2(t / 2) = a / g and
// s = (g_first + a) / g,
//   p_j = s sinh((j + 1) t) / sinh t + cosh((j + 1/2) t) / cosh(t / 2),
// and p_j - p_{j-1} = s cosh((j + 1/2) t) / cosh(t / 2) + 2 tanh(t / 2) sinh(j t), sums of
// positive terms.  Taking out e^{j t} leaves decaying exponentials only (C and S below), and
// q_j = p_{j-1} / p_j = 1 - (p_j - p_{j-1}) / p_j for every j at once.  The subtraction keeps
// the formula's own roundings, which are alike for all j and would act like a change of a by
// eps g / a, far below an ulp of q; where q < 1/2 (a not small against g) the quotient of two
// p is the accurate form.  The last node, with its own diagonal, takes one step of the
// recurrence.  Lines of up to kWalk nodes walk the recurrence: the exponentials take about as long
// as eight of its steps (one apply by closed form and walking: 1 x 1 55 and 46 us, 8 x 8 60 and 49).
constexpr int kWalk = 8;
constexpr int kFacT = 256;
__global__ void __launch_bounds__(kFacT)
k_mhat_factor(int m, int n, Grid gr, const VecCtl* __restrict__ ctl, double* __restrict__ fac,
              size_t fstride) {
  const int b = blockIdx.x;
  if (!ctl[b].gm_active) return;
  const int which = threadIdx.x / (kFacT / 2), t = threadIdx.x & (kFacT / 2 - 1);
  const double a = ctl[b].a;
  const int len = which == 0 ? n : m;
  const double g = which == 0 ? gr.gt : gr.gb;
  const double g_first = which == 0 ? gr.g_src : gr.g_bt;
  const double g_last = which == 0 ? gr.g_tr : gr.g_sense;
  double* base = fac + (size_t)b * fstride + (which == 0 ? 0 : line_fac_size(n));
  const int L = chunk_len(len);
  const size_t N = (size_t)kChunks * L;
  double *lo = base, *ylo = base + N, *ip = base + 2 * N, *q = base + 3 * N,
         *xhi = base + 4 * N, *fwd = base + 5 * N, *bwd = fwd + 5 * kChunks;
  const double inv_g = 1.0 / g;
  // q in node order, in xhi for now
  if (len <= kWalk) {
    if (t == 0) {
      double qj = 0.0;
      for (int j = 0; j < len; ++j) {
        const double d = ((j > 0) ? g : g_first) + ((j < len - 1) ? g : g_last) + a;
        qj = g / fma(-g, qj, d);
        xhi[j] = qj;
      }
    }
  } else {
    const double th = 2.0 * asinh(0.5 * sqrt(a * inv_g)), et = exp(-th);
    const double s = (g_first + a) * inv_g, sl = (g_last + a) * inv_g;
    const double cc = 1.0 / (1.0 + et), ce = s / expm1(-2.0 * th), ct = expm1(-th) * cc;
    auto C = [&](int j) { return cc * (1.0 + exp(-(2.0 * j + 1.0) * th)); };
    auto S = [&](int j) { return fma(ce, expm1(-2.0 * (j + 1) * th), C(j)); };
    auto one_minus_q = [&](int j) { return fma(s, C(j), ct * expm1(-2.0 * j * th)) / S(j); };
    for (int j = t; j < len; j += kFacT / 2) {
      double qj;
      if (j < len - 1) {
        const double x = one_minus_q(j);
        qj = (x <= 0.5) ? 1.0 - x : ((j == 0) ? 1.0 / (1.0 + s) : et * S(j - 1) / S(j));
      } else {
        qj = 1.0 / (sl + one_minus_q(j - 1));
      }
      xhi[j] = qj;
    }
  }
  __syncthreads();
  if (t >= kChunks) return;
  // chunk c: its q, the one before it, then the running products
  const int c = t;
  const int j0 = c * L, j1 = (j0 + L < len) ? j0 + L : len;
  const size_t o0 = which == 0 ? (size_t)c : (size_t)j0, os = which == 0 ? kChunks : 1;
  double qm = (j0 > 0 && j0 < len) ? xhi[j0 - 1] : 0.0;
  size_t o = o0;
#pragma unroll 4
  for (int j = j0; j < j1; ++j, o += os) q[o] = xhi[j];
  __syncwarp();                            // xhi is free
  double prod = 1.0;
  o = o0;
#pragma unroll 4
  for (int j = j0; j < j1; ++j, o += os) {
    const double qj = q[o], iv = qj * inv_g;
    prod *= qm;
    lo[o] = (j == j0) ? 0.0 : qm;
    ip[o] = iv;
    ylo[o] = prod * iv;
    qm = qj;
  }
  double fc = (j0 < j1) ? prod : 0.0;      // carry factor of the whole chunk, forward
  double back = 1.0;
#pragma unroll 4
  for (int j = j1 - 1; j >= j0; --j) {
    o -= os;
    back *= q[o];
    xhi[o] = back;
    if (j == j1 - 1) q[o] = 0.0;
  }
  double bc = (j0 < j1) ? back : 0.0;      // and backward
  for (int k = (j1 > j0 ? j1 - j0 : 0); k < L; ++k) {      // unused slots of the last chunks
    const size_t e = o0 + k * os;
    lo[e] = ylo[e] = ip[e] = q[e] = xhi[e] = 0.0;
  }
#pragma unroll
  for (int s = 0; s < 5; ++s) {
    const int o = 1 << s;
    fwd[s * kChunks + c] = (c >= o) ? fc : 0.0;
    bwd[s * kChunks + c] = (c + o < kChunks) ? bc : 0.0;
    const double f2 = __shfl_up_sync(0xffffffffu, fc, o);
    const double b2 = __shfl_down_sync(0xffffffffu, bc, o);
    if (c >= o) fc *= f2;
    if (c + o < kChunks) bc *= b2;
  }
}

// Value that enters chunk `lane` from its left (right): inclusive scan of the chunks' own end
// values v with the factors f (5 x 32), then shifted by one.  Lanes without a partner keep v
// (their factor is zero, which an infinite v would turn into NaN).
__device__ __forceinline__ double carry_left(double v, const double* __restrict__ f, int lane) {
#pragma unroll
  for (int s = 0; s < 5; ++s) {
    const double w = fma(f[s * kChunks + lane], __shfl_up_sync(0xffffffffu, v, 1 << s), v);
    v = (lane >= (1 << s)) ? w : v;
  }
  v = __shfl_up_sync(0xffffffffu, v, 1);
  return lane == 0 ? 0.0 : v;
}
__device__ __forceinline__ double carry_right(double v, const double* __restrict__ f, int lane) {
#pragma unroll
  for (int s = 0; s < 5; ++s) {
    const double w = fma(f[s * kChunks + lane], __shfl_down_sync(0xffffffffu, v, 1 << s), v);
    v = (lane + (1 << s) < kChunks) ? w : v;
  }
  v = __shfl_down_sync(0xffffffffu, v, 1);
  return lane == kChunks - 1 ? 0.0 : v;
}

// z_b = sc G_2^-1 r_b along every column (sc: the scale of the unnormalised input basis
// vector).  A block takes 16 columns (128-byte rows) x 32 chunks; the carries are scanned by
// 16 warps, one column each.  The three passes over a chunk go through z_b (in L2).
constexpr int kCols = 16;
__global__ void __launch_bounds__(kCols * kChunks)
k_mhat_cols(int m, int n, const double* __restrict__ r, size_t rstride, double* __restrict__ z,
            size_t zstride, const double* __restrict__ fac, size_t fstride,
            const VecCtl* __restrict__ ctl, int kidx) {
  const int b = blockIdx.y;
  if (!ctl[b].gm_active) return;
  const double sc = (kidx >= 0) ? ctl[b].s[kidx] : 1.0;
  const int tj = threadIdx.x & (kCols - 1), c = threadIdx.x / kCols;
  const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int j = blockIdx.x * kCols + tj;
  const bool col = j < n;
  const LineFac f = line_fac(fac + (size_t)b * fstride + line_fac_size(n), m);
  const int L = chunk_len(m), i0 = c * L, i1 = min(i0 + L, m);
  const double* rb = r + (size_t)b * rstride + (size_t)m * n + j;
  double* u = z + (size_t)b * zstride + (size_t)m * n + j;
  __shared__ double ends[kChunks][kCols + 1];
  double y = 0.0;
  if (col) {
#pragma unroll 8
    for (int i = i0; i < i1; ++i) {
      y = fma(f.lo[i], y, sc * rb[(size_t)i * n]);
      u[(size_t)i * n] = y;
    }
  }
  ends[c][tj] = y;
  __syncthreads();
  ends[lane][w] = carry_left(ends[lane][w], f.fwd, lane);
  __syncthreads();
  double carry = ends[c][tj];
  double x = 0.0;
  if (col) {
#pragma unroll 8
    for (int i = i1 - 1; i >= i0; --i) {
      x = fma(f.q[i], x, fma(f.ylo[i], carry, f.ip[i] * u[(size_t)i * n]));
      u[(size_t)i * n] = x;
    }
  }
  __syncthreads();
  ends[c][tj] = x;
  __syncthreads();
  ends[lane][w] = carry_right(ends[lane][w], f.bwd, lane);
  __syncthreads();
  carry = ends[c][tj];
  if (col) {
#pragma unroll 8
    for (int i = i0; i < i1; ++i) u[(size_t)i * n] = fma(f.xhi[i], carry, u[(size_t)i * n]);
  }
}

// z_t = (sc r_t + a1 z_b) G_1^-1 along every row.  A warp takes a row, staged in shared memory
// with chunk `lane` at lane S (S odd: the lanes' walks hit different banks).
__global__ void __launch_bounds__(kT)
k_mhat_rows(int m, int n, const double* __restrict__ r, size_t rstride, double* __restrict__ z,
            size_t zstride, const double* __restrict__ fac, size_t fstride,
            const VecCtl* __restrict__ ctl, int kidx, FastDiv by_len) {
  const int b = blockIdx.y;
  if (!ctl[b].gm_active) return;
  extern __shared__ double row_smem[];
  const double a = ctl[b].a;
  const double sc = (kidx >= 0) ? ctl[b].s[kidx] : 1.0;
  const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int i = blockIdx.x * (blockDim.x >> 5) + w;
  if (i >= m) return;
  const LineFac f = line_fac(fac + (size_t)b * fstride, n);
  const int L = chunk_len(n), S = L | 1;
  double* s = row_smem + (size_t)w * kChunks * S;
  auto at = [&](int j) {
    const int c = (int)by_len.quot((uint32_t)j);
    return c * S + (j - c * L);
  };
  double* zt = z + (size_t)b * zstride + (size_t)i * n;
  const double* zb = zt + (size_t)m * n;
  const double* rt = r + (size_t)b * rstride + (size_t)i * n;
#pragma unroll 4
  for (int j = lane; j < n; j += 32) s[at(j)] = fma(a, zb[j], sc * rt[j]);
  __syncwarp();
  double* sl = s + lane * S;
  const int cnt = max(0, min(L, n - lane * L));
  double y = 0.0;
#pragma unroll 4
  for (int k = 0; k < cnt; ++k) {
    y = fma(f.lo[k * kChunks + lane], y, sl[k]);
    sl[k] = y;
  }
  double carry = carry_left(y, f.fwd, lane);
  double x = 0.0;
#pragma unroll 4
  for (int k = cnt - 1; k >= 0; --k) {
    const int o = k * kChunks + lane;
    x = fma(f.q[o], x, fma(f.ylo[o], carry, f.ip[o] * sl[k]));
    sl[k] = x;
  }
  carry = carry_right(x, f.bwd, lane);
#pragma unroll 4
  for (int k = 0; k < cnt; ++k) sl[k] = fma(f.xhi[k * kChunks + lane], carry, sl[k]);
  __syncwarp();
#pragma unroll 4
  for (int j = lane; j < n; j += 32) zt[j] = s[at(j)];
}

// Jacobi: z = r / diag(J), diag(J) = wire diagonal + D; none: z = r.
__global__ void k_jacobi(Grid gr, const double* __restrict__ D, const double* __restrict__ r,
                         size_t rstride, double* __restrict__ z, size_t zstride, int none,
                         const VecCtl* __restrict__ ctl, int kidx) {
  const int b = blockIdx.y;
  if (ctl && !ctl[b].gm_active) return;
  const double sc = (ctl && kidx >= 0) ? ctl[b].s[kidx] : 1.0;
  const int m = gr.m, n = gr.n, mn = m * n;
  const double* rb = r + (size_t)b * rstride;
  double* zb = z + (size_t)b * zstride;
  const double* Db = D + (size_t)b * mn;
  for (int c = blockIdx.x * kT + threadIdx.x; c < mn; c += gridDim.x * kT) {
    if (none) {
      zb[c] = sc * rb[c];
      zb[mn + c] = sc * rb[mn + c];
      continue;
    }
    const int i = c / n, j = c - i * n;
    const double dt = (j == 0) ? gr.dt0 : ((j == n - 1) ? gr.dtl : gr.dtm);
    const double db = (i == 0) ? gr.db0 : ((i == m - 1) ? gr.dbl : gr.dbm);
    zb[c] = sc * rb[c] / (dt + Db[c]);
    zb[mn + c] = sc * rb[mn + c] / (db + Db[c]);
  }
}

// a row of 16384 nodes takes 131 KB
constexpr int kRowSmemMax = 220 * 1024;

int nblocks(size_t count) {
  size_t nb = (count + kT - 1) / kT;
  if (nb > 1216) nb = 1216;
  return nb < 1 ? 1 : (int)nb;
}

}  // namespace

size_t mhat_fac_size(int m, int n) { return line_fac_size(n) + line_fac_size(m); }

cudaError_t mhat_configure() {
  return cudaFuncSetAttribute(k_mhat_rows, cudaFuncAttributeMaxDynamicSharedMemorySize,
                              kRowSmemMax);
}

int precond_mhat(const Grid& gr, const double* r, size_t rstride, double* z, size_t zstride,
                 int B, const VecCtl* ctl, double* fac, int kidx, cudaStream_t s) {
  const int m = gr.m, n = gr.n;
  const size_t fstride = mhat_fac_size(m, n);
  // a cycle's a is fixed: its first iteration (and a single apply) builds the factors
  if (kidx <= 0) {
    k_mhat_factor<<<B, kFacT, 0, s>>>(m, n, gr, ctl, fac, fstride);
    count_launches(1);
  }
  k_mhat_cols<<<dim3((n + kCols - 1) / kCols, B), kCols * kChunks, 0, s>>>(
      m, n, r, rstride, z, zstride, fac, fstride, ctl, kidx);
  // rows per block: as many as half an SM's shared memory holds, eight at most
  const size_t row = (size_t)kChunks * (chunk_len(n) | 1) * sizeof(double);
  int rows = (int)(kRowSmemMax / 2 / row);
  rows = rows < 1 ? 1 : (rows > kT / 32 ? kT / 32 : rows);
  k_mhat_rows<<<dim3((m + rows - 1) / rows, B), 32 * rows, rows * row, s>>>(
      m, n, r, rstride, z, zstride, fac, fstride, ctl, kidx, FastDiv(chunk_len(n)));
  count_launches(2);
  return cudaGetLastError() == cudaSuccess ? MCA_OK : MCA_ERR_CUDA;
}

int precond_jacobi(const Grid& gr, const double* D, const double* r, size_t rstride, double* z,
                   size_t zstride, int B, bool none, const VecCtl* ctl, int kidx,
                   cudaStream_t s) {
  const size_t mn = (size_t)gr.m * gr.n;
  k_jacobi<<<dim3(nblocks(mn), B), kT, 0, s>>>(gr, D, r, rstride, z, zstride, none ? 1 : 0, ctl,
                                               kidx);
  count_launches(1);
  return cudaGetLastError() == cudaSuccess ? MCA_OK : MCA_ERR_CUDA;
}

}  // namespace mca

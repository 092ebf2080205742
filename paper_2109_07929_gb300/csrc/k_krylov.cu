// Flexible GMRES kernels (Section 4: GMRES on each Newton system; right preconditioned,
// Saad, Iterative Methods for Sparse Linear Systems, Alg. 9.6): classical Gram-Schmidt in
// FP64 with a second pass when a running estimate of the loss of orthogonality asks for
// it (the Daniel-Gragg-Kaufman-Stewart selective reorthogonalisation), Givens rotations
// on the Hessenberg column, back substitution and the solution update dx = Z y.
//
// Per iteration k the orthogonalisation runs as
//   pass 1 (fused into the Jacobian apply): h1 = V^T w
//   pass 2: u = w - V h1 (the next basis vector) and ||u||^2 in the same sweep
//   only when the estimate asks for it:
//   pass 3: h2 = V^T u;  pass 4: u <- u - V h2 and ||u||^2
// The estimate follows u = (I - V V^T) w: if V^T V = I + E with |E| <= delta, then
// |V^T u| <= delta |V^T w| plus rounding of order nk eps |w|, so the new vector keeps a
// loss of about (sqrt(nk) delta + c nk eps) / rho with rho = |u| / |w| (the cancellation
// of the pass, |w|^2 = |u|^2 + |h1|^2).  While that stays below kOrthTol the second pass
// is skipped; the GMRES residual estimate is then exact up to a factor 1 + O(k kOrthTol).
// All reductions are two-level (per-block partials, then one fixed-order sum per vector),
// hence deterministic.
#include <algorithm>

#include "bits.cuh"
#include "mca_internal.cuh"
#include "solver_dev.cuh"

namespace mca {

namespace {

constexpr int kThreads = 256;

template <int KP>
__device__ __forceinline__ void block_store_partials(double (&acc)[KP], int nk,
                                                     double* __restrict__ part, int b,
                                                     int nblk, int vb) {
  __shared__ double red[kThreads / 32][KP];
  const int wv = threadIdx.x >> 5, l = threadIdx.x & 31;
  const double tot = warp_sum_scatter<KP>(acc);
  if (warp_scatter_writer<KP>(l)) red[wv][warp_scatter_index<KP>(l)] = tot;
  __syncthreads();
  if (threadIdx.x < nk && threadIdx.x < KP) {
    double s = 0.0;
#pragma unroll
    for (int q = 0; q < kThreads / 32; ++q) s += red[q][threadIdx.x];
    part[((size_t)b * 32 + threadIdx.x) * nblk + vb] = s;
    __threadfence();
  }
}

// True in every thread of the block that finished last among the launch's blocks of vector
// b (its partial sums are then all visible); the counter is reset by the caller.
__device__ __forceinline__ bool last_block(unsigned int* cnt, int b) {
  __shared__ bool last;
  __syncthreads();
  if (threadIdx.x == 0) last = (atomicAdd(&cnt[b], 1u) == gridDim.x - 1);
  __syncthreads();
  if (last) __threadfence();
  return last;
}

// h[b][j] = sum over blocks of part[b][j][:] for j < nk (kHStride; nothing behind them).
__global__ void k_reduce_dots(const double* __restrict__ part, int nblk, int nk,
                              double* __restrict__ h, const VecCtl* __restrict__ ctl) {
  const int b = blockIdx.x;
  if (ctl != nullptr && !ctl[b].gm_active) return;
  const int wv = threadIdx.x >> 5, l = threadIdx.x & 31;
  for (int j = wv; j < nk; j += kThreads / 32) {
    double s = 0.0;
    for (int t = l; t < nblk; t += 32) s += part[((size_t)b * 32 + j) * nblk + t];
    s = warp_sum(s);
    if (l == 0) h[(size_t)b * kHStride + j] = s;
  }
}

// The reductions below follow one summation order, whatever the launch shape: nblk blocks of
// kThreads accumulators per vector (vec_nblk; the Jacobian apply: residual_nblk), accumulator
// (v, t) adding the entries v kThreads + t + k nblk kThreads in order; then a butterfly over
// each 32 accumulators, the warps of a block in order, and the blocks' partial sums by 32 lanes
// and a butterfly.  Results (and with them the rounding of the BF16 preconditioner's inputs) do
// not depend on how many accumulators a thread holds.

// pass 3 (marked vectors only): partial dots <V_j, u> of the new vector u, reduced by the
// last block into h2_j = s_j <V_j, u>.  Most launches find no marked vector and only end their
// blocks, so a launch has a quarter of the summation's blocks, each taking them in turn, where
// that leaves the eight per SM that reside, and for few vectors as many as do: with a quarter
// of the blocks the pass and its update took 352 us for one vector of 1024 x 1024 (long cycles,
// Jacobi preconditioner; now 233) and 50 us at 64 x 64 (now 34).
// ZS: the Newton step from V = 0, whose v_0 is stored in the first column of the top layer
// only (the residual's sparse_f); its other entries are not read, and the last block also
// subtracts h2_0 v_0 from u (see subtract_sparse_v0), in place of the update pass.
template <int KP, bool ZS = false>
__global__ void __launch_bounds__(kThreads)
k_reorth_dots(double* u, const double* __restrict__ V, size_t vstride, size_t n2, int nk,
              double* __restrict__ part, int nblk, const VecCtl* __restrict__ ctl,
              unsigned int* cnt, double* h2, int ncols) {
  const int b = blockIdx.y;
  if (!ctl[b].gm_active || !ctl[b].reorth) return;
  double* ub = u + (size_t)b * vstride;
  const double* Vb = V + (size_t)b * vstride;
  const int N2 = (int)n2;
  const int mn = N2 / 2, n = ncols;
  for (int vb = blockIdx.x; vb < nblk; vb += gridDim.x) {
    double acc[KP];
#pragma unroll
    for (int j = 0; j < KP; ++j) acc[j] = 0.0;
    for (int e = vb * kThreads + threadIdx.x; e < N2; e += nblk * kThreads) {
      const double x = ub[e];
      const bool v0 = !ZS || (e < mn && e % n == 0);
#pragma unroll
      for (int j = 0; j < KP; ++j)
        if (j < nk && (!ZS || j > 0 || v0)) acc[j] = fma(Vb[(size_t)j * n2 + e], x, acc[j]);
    }
    block_store_partials<KP>(acc, nk, part, b, nblk, vb);
    __syncthreads();
  }
  if (last_block(cnt, b)) {
    reduce_rows(part, b, nblk, nk, h2, ctl[b].s);
    if (threadIdx.x == 0) cnt[b] = 0;
    if (ZS) subtract_sparse_v0(ub, Vb, h2 + (size_t)b * kHStride, mn, n);
  }
}

// Passes 2 and 4: out <- w - sum_j hc_j v_j over j = j0 .. nk - 1 (the next, unnormalised
// basis vector, with its BF16 copy for the tensor-core preconditioner), then the partial
// ||out||^2; the last block of each vector runs the phase's control step (UpdPhase).  j0 = 1
// in the Newton step from V = 0, where the dots' last block has subtracted the sparse v_0.
//
// Bound: the FP64 pipe from three vectors on, HBM below.  A predicated-off FMA takes its
// turn on that pipe like any other, so the number of vectors NK is exact: 1 .. 8, or any
// (NK = 0) in groups of four and a rest by cases (at 1024 x 1024, 16 vectors, three of
// them took as long as four, 312 us; now 239).  Entries go in
// pairs (16-byte loads; n2 is even, so every vector starts on a 16-byte boundary): half a
// block takes one block of the summation, two accumulators per thread.  Two pairs are in
// flight per thread, all their loads issued before the first store (out may alias w, so the
// compiler cannot move loads of the next trip above the stores): G = 1 the next trip of the
// same accumulators, G = 2 (when the accumulators have one trip or two) another block of
// the summation.  With one entry per thread and a butterfly per warp the reduction and the
// coefficients took more FP64 instructions than the update itself (256 x 256, 8 vectors,
// nk = 1 and 2: 34 and 38 us, now 16 and 20).
// (layer, i, j) of a pair comes from one multiply-and-shift quotient.
template <int N>
__device__ __forceinline__ void subtract(const double* __restrict__ v, size_t n2,
                                         const double* hj, uint32_t p, double2& x) {
#pragma unroll
  for (int j = 0; j < N; ++j) {
    const double2 t = reinterpret_cast<const double2*>(v + (size_t)j * n2)[p];
    x.x = fma(-hj[j], t.x, x.x);
    x.y = fma(-hj[j], t.y, x.y);
  }
}

// the same for two pairs, with both pairs' loads of a vector together
template <int N>
__device__ __forceinline__ void subtract2(const double* __restrict__ v, size_t n2,
                                          const double* hj, uint32_t p, uint32_t q, double2& x,
                                          double2& y) {
#pragma unroll
  for (int j = 0; j < N; ++j) {
    const double2* vj = reinterpret_cast<const double2*>(v + (size_t)j * n2);
    const double2 t = vj[p], u = vj[q];
    x.x = fma(-hj[j], t.x, x.x);
    x.y = fma(-hj[j], t.y, x.y);
    y.x = fma(-hj[j], u.x, y.x);
    y.y = fma(-hj[j], u.y, y.y);
  }
}

template <int NK, int G>
__global__ void __launch_bounds__(kThreads, NK <= 4 ? 4 : 3)
k_update_norm(int phase, const double* w, size_t wstride, const double* __restrict__ V,
              size_t vstride, size_t n2, int nk, int j0, const double* __restrict__ hc,
              double* __restrict__ part, int nblk, VecCtl* ctl, unsigned int* cnt,
              const double* __restrict__ h1, int restart, int32_t* host_flags, double* out,
              size_t ostride, __nv_bfloat16* __restrict__ xbf, int mp, int np, int m, int n,
              FastDiv by_n) {
  const int b = blockIdx.y;
  if (phase != UPD_PLAIN && (!ctl[b].gm_active || (phase == UPD_REORTH && !ctl[b].reorth)))
    return;
  const double* hs = hc + (size_t)b * kHStride + 32 + j0;      // their scaled coefficients
  double hj[NK > 0 ? NK : 1];
  __shared__ double hsh[32];
  if constexpr (NK > 0) {
#pragma unroll
    for (int j = 0; j < NK; ++j) hj[j] = hs[j];
  } else {
    if ((int)threadIdx.x < nk - j0) hsh[threadIdx.x] = hs[threadIdx.x];
    __syncthreads();
  }
  const double2* wb = reinterpret_cast<const double2*>(w + (size_t)b * wstride);
  double2* ob = reinterpret_cast<double2*>(out + (size_t)b * ostride);
  const double* Vb = V + (size_t)b * vstride + (size_t)j0 * n2;
  __nv_bfloat16* xb = xbf ? xbf + (size_t)b * 2 * mp * np : nullptr;
  const uint32_t mn = (uint32_t)(n2 / 2), P = mn;      // P pairs = m n
  const bool even = (n & 1) == 0;                      // no pair crosses a row
  // position of entry e < 2 m n in the padded BF16 copy, and its column
  auto pad = [&](uint32_t e, uint32_t& j) {
    const uint32_t l = (e >= mn) ? 1u : 0u;
    const uint32_t cell = e - l * mn;
    const uint32_t i = by_n.quot(cell);
    j = cell - i * (uint32_t)n;
    return (l * (uint32_t)mp + i) * (uint32_t)np + j;
  };
  auto finish = [&](uint32_t p, double2 x, double (&acc)[2]) {
    ob[p] = x;
    if (xb != nullptr) {
      uint32_t j;
      const uint32_t o = pad(2 * p, j);
      const __nv_bfloat16 b0 = d2bf16_bits(x.x), b1 = d2bf16_bits(x.y);
      if (even) {
        *reinterpret_cast<__nv_bfloat162*>(xb + o) = __nv_bfloat162(b0, b1);
      } else {
        xb[o] = b0;
        xb[(j + 1 < (uint32_t)n) ? o + 1 : pad(2 * p + 1, j)] = b1;
      }
    }
    acc[0] = fma(x.x, x.x, acc[0]);
    acc[1] = fma(x.y, x.y, acc[1]);
  };
  auto one = [&](uint32_t p, double (&acc)[2]) {
    double2 x = wb[p];
    if constexpr (NK > 0) {
      subtract<NK>(Vb, n2, hj, p, x);
    } else {
      for (int j = 0; j < nk - j0; ++j) subtract<1>(Vb + (size_t)j * n2, n2, hsh + j, p, x);
    }
    finish(p, x, acc);
  };
  auto two = [&](uint32_t p, uint32_t q, double (&accp)[2], double (&accq)[2]) {
    double2 x = wb[p], y = wb[q];
    if constexpr (NK > 0) {
      subtract2<NK>(Vb, n2, hj, p, q, x, y);
    } else {
      int j = 0;
      const double* vj = Vb;
      for (; j + 4 <= nk - j0; j += 4, vj += 4 * n2) subtract2<4>(vj, n2, hsh + j, p, q, x, y);
      switch (nk - j0 - j) {
        case 1: subtract2<1>(vj, n2, hsh + j, p, q, x, y); break;
        case 2: subtract2<2>(vj, n2, hsh + j, p, q, x, y); break;
        case 3: subtract2<3>(vj, n2, hsh + j, p, q, x, y); break;
        default: break;
      }
    }
    finish(p, x, accp);
    finish(q, y, accq);
  };
  constexpr uint32_t kHalf = kThreads / 2;             // pairs of one block of the summation
  const uint32_t half = threadIdx.x / kHalf;
  const uint32_t vb0 = 2 * G * blockIdx.x + half;      // G = 2: also vb0 + 2
  const uint32_t st = (uint32_t)nblk * kHalf;
  double acc[G][2] = {};
  uint32_t p = vb0 * kHalf + (threadIdx.x & (kHalf - 1));
  if constexpr (G == 1) {
    if (vb0 < (uint32_t)nblk) {
      for (; p + st < P; p += 2 * st) two(p, p + st, acc[0], acc[0]);
      if (p < P) one(p, acc[0]);
    }
  } else {
    const bool second = vb0 + 2 < (uint32_t)nblk;
    if (vb0 < (uint32_t)nblk) {
      for (; p < P; p += st) {
        const uint32_t q = p + 2 * kHalf;
        if (second && q < P) two(p, q, acc[0], acc[1]);
        else one(p, acc[0]);
      }
    }
  }
  // the butterfly over 32 accumulators, which sit in 16 lanes (two each): its first levels
  // halve what a lane holds, its last level joins the two
  const int lane = threadIdx.x & 31, wv = threadIdx.x >> 5;
  double t0 = acc[0][0], t1 = acc[0][1];
  if constexpr (G == 2) {
    const bool up = (lane & 8) != 0;
    const double s0 = up ? acc[0][0] : acc[1][0], s1 = up ? acc[0][1] : acc[1][1];
    t0 = (up ? acc[1][0] : acc[0][0]) + __shfl_xor_sync(0xffffffffu, s0, 8);
    t1 = (up ? acc[1][1] : acc[0][1]) + __shfl_xor_sync(0xffffffffu, s1, 8);
  }
  constexpr int kFirst = (G == 2) ? 4 : 8;
  {
    const bool up = (lane & kFirst) != 0;
    t0 = (up ? t1 : t0) + __shfl_xor_sync(0xffffffffu, up ? t0 : t1, kFirst);
  }
#pragma unroll
  for (int o = kFirst / 2; o > 0; o >>= 1) t0 += __shfl_xor_sync(0xffffffffu, t0, o);
  t0 += __shfl_xor_sync(0xffffffffu, t0, kFirst);
  __shared__ double red[G][2][kThreads / 32];
  if ((lane & 7) == 0 && (G == 2 || (lane & 8) == 0))
    red[G == 2 ? (lane >> 3) & 1 : 0][half][(wv & 3) * 2 + (lane >> 4)] = t0;
  __syncthreads();
  if (threadIdx.x < 2 * G) {
    const int g = threadIdx.x >> 1, hf = threadIdx.x & 1;
    const int vb = 2 * (G * (int)blockIdx.x + g) + hf;
    double s = 0.0;
#pragma unroll
    for (int q = 0; q < kThreads / 32; ++q) s += red[g][hf][q];
    if (vb < nblk) part[(size_t)b * 32 * nblk + vb] = s;
    __threadfence();
  }
  if (phase == UPD_PLAIN) return;
  if (last_block(cnt, b)) {
    __shared__ GsShared gs;
    __shared__ double ps[kMaxVecBlocks];
    for (int t = threadIdx.x; t < nblk; t += kThreads)
      ps[t] = __ldcg(&part[(size_t)b * 32 * nblk + t]);
    if (threadIdx.x == 0) cnt[b] = 0;
    __syncthreads();
    if (threadIdx.x < 32) {
      double s = 0.0;
      for (int t = threadIdx.x; t < nblk; t += 32) s += ps[t];
      s = warp_sum(s);
      if (threadIdx.x == 0) gs.hn2 = s;
    }
    gram_schmidt_control(ctl[b], phase, hc + (size_t)b * kHStride, h1 + (size_t)b * kHStride, nk,
                         restart, host_flags ? host_flags + b : nullptr, gs);
  }
}

__device__ __forceinline__ double widen(double x) { return x; }
__device__ __forceinline__ double widen(float x) { return f2d_bits(x); }

__device__ __forceinline__ double2 widen2(const double* z, uint32_t p) {
  return reinterpret_cast<const double2*>(z)[p];
}
__device__ __forceinline__ double2 widen2(const float* z, uint32_t p) {
  const float2 v = reinterpret_cast<const float2*>(z)[p];
  return make_double2(f2d_bits(v.x), f2d_bits(v.y));
}

// x <- x + sum_j y_j z_j over the finished cycle (Z in FP64 or FP32), entries in pairs
// (W = 2, x on a 16-byte boundary) or one by one.  Bound: the FP64 pipe (k FMAs per entry).
template <typename ZT, int W>
__global__ void __launch_bounds__(kThreads)
k_update_x(double* __restrict__ x, const ZT* __restrict__ Z, size_t zstride, size_t n2,
           const VecCtl* __restrict__ ctl) {
  const int b = blockIdx.y;
  const VecCtl& c = ctl[b];
  if (!c.newton_active) return;
  const int kd = c.k_done;
  __shared__ double ys[MCA_KMAX];
  if (threadIdx.x < MCA_KMAX) ys[threadIdx.x] = (threadIdx.x < kd) ? c.y[threadIdx.x] : 0.0;
  __syncthreads();
  double* xb = x + (size_t)b * n2;
  const ZT* Zb = Z + (size_t)b * zstride;
  const uint32_t st = gridDim.x * kThreads, N = (uint32_t)(n2 / W);
  uint32_t e = blockIdx.x * kThreads + threadIdx.x;
  if constexpr (W == 2) {
    double2* x2 = reinterpret_cast<double2*>(xb);
    for (; e + st < N; e += 2 * st) {          // two independent pairs per trip
      double2 s0 = x2[e], s1 = x2[e + st];
      const ZT* zj = Zb;
      for (int j = 0; j < kd; ++j, zj += n2) {
        const double2 z0 = widen2(zj, e), z1 = widen2(zj, e + st);
        s0.x = fma(ys[j], z0.x, s0.x);
        s0.y = fma(ys[j], z0.y, s0.y);
        s1.x = fma(ys[j], z1.x, s1.x);
        s1.y = fma(ys[j], z1.y, s1.y);
      }
      x2[e] = s0;
      x2[e + st] = s1;
    }
    for (; e < N; e += st) {
      double2 s0 = x2[e];
      const ZT* zj = Zb;
      for (int j = 0; j < kd; ++j, zj += n2) {
        const double2 z0 = widen2(zj, e);
        s0.x = fma(ys[j], z0.x, s0.x);
        s0.y = fma(ys[j], z0.y, s0.y);
      }
      x2[e] = s0;
    }
  } else {
    for (; e < N; e += st) {
      double s = xb[e];
      const ZT* zj = Zb;
      for (int j = 0; j < kd; ++j, zj += n2) s = fma(ys[j], widen(zj[e]), s);
      xb[e] = s;
    }
  }
}

// Start of a stand-alone linear solve: beta = ||rhs|| from the norm partials, stop at
// rtol * beta.
__global__ void k_gmres_init(const double* __restrict__ part_norm, int nblk, VecCtl* ctl,
                             double rtol, int first) {
  const int b = blockIdx.x;
  double s = 0.0;
  for (int t = threadIdx.x; t < nblk; t += 32) s += part_norm[((size_t)b * 32) * nblk + t];
  s = warp_sum(s);
  if (threadIdx.x == 0) {
    VecCtl& c = ctl[b];
    const double beta = sqrt(s);
    if (first) {
      c.ynorm = beta;                      // ||rhs|| of the linear system
      c.tol_abs = rtol * beta;
      c.gmres_iters = 0;
    }
    c.g[0] = beta;
    c.s[0] = 1.0;
    c.orth = 0.0;
    c.reorth = 0;
    c.reorth_mask = 0u;
    c.res_est = beta;
    c.k_done = 0;
    c.newton_active = 1;
    c.status = MCA_OK;
    c.gm_active = (beta > c.tol_abs && beta > 0.0) ? 1 : 0;
  }
}

__global__ void k_sub(const double* __restrict__ a, const double* __restrict__ b,
                      double* __restrict__ out, size_t n2) {
  const size_t off = (size_t)blockIdx.y * n2;
  for (size_t e = blockIdx.x * (size_t)blockDim.x + threadIdx.x; e < n2;
       e += (size_t)gridDim.x * blockDim.x)
    out[off + e] = a[off + e] - b[off + e];
}

__global__ void k_report(const VecCtl* __restrict__ ctl, const double* __restrict__ kcl,
                         const int* __restrict__ err, HostReport* rep, int B) {
  for (int b = threadIdx.x; b < B; b += blockDim.x) {
    const VecCtl& c = ctl[b];
    HostReport r;
    r.status = c.status;
    r.newton_iters = c.newton_iters;
    r.gmres_iters = c.gmres_iters;
    r.k_done = c.k_done;
    r.fnorm = c.fnorm;
    r.ynorm = c.ynorm;
    r.kcl = kcl ? kcl[b] : 0.0;
    r.res_est = c.res_est;
    rep[b] = r;
  }
  if (threadIdx.x == 0) rep[B].status = *err;
  __threadfence_system();
}

}  // namespace

void launch_report(const VecCtl* ctl, const double* kcl, const int* err, HostReport* rep,
                   int B, cudaStream_t s) {
  k_report<<<1, 128, 0, s>>>(ctl, kcl, err, rep, B);
}

void launch_gmres_init(const double* part_norm, int nblk, VecCtl* ctl, int B, double rtol,
                       int first, cudaStream_t s) {
  k_gmres_init<<<B, 32, 0, s>>>(part_norm, nblk, ctl, rtol, first);
}

void launch_sub(const double* a, const double* b, double* out, size_t n2, int B,
                cudaStream_t s) {
  int nb = (int)((n2 + kThreads - 1) / kThreads);
  if (nb > 1216) nb = 1216;
  k_sub<<<dim3(nb, B), kThreads, 0, s>>>(a, b, out, n2);
}

int vec_nblk(size_t n2, int B) {
  constexpr size_t kGridBlocks = 152 * 32;
  size_t nb = (n2 + kThreads - 1) / kThreads;
  const size_t want = (kGridBlocks + B - 1) / (size_t)(B < 1 ? 1 : B);
  if (nb > want) nb = want;
  if (nb > kMaxVecBlocks) nb = kMaxVecBlocks;
  return nb < 1 ? 1 : (int)nb;
}

void launch_reduce_dots(const double* part, int nblk, int nk, double* h, int B,
                        const VecCtl* ctl, cudaStream_t s) {
  k_reduce_dots<<<B, kThreads, 0, s>>>(part, nblk, nk, h, ctl);
}

void launch_reorth_dots(double* u, const double* V, size_t vstride, size_t n2, int nk,
                        double* part, int nblk, int B, const VecCtl* ctl, unsigned int* cnt,
                        double* h2, cudaStream_t s, bool zs, int ncols) {
  constexpr int kResident = 8 * 152;
  const int turns = std::max(1, std::min(4, nblk * B / kResident));
  const dim3 grid((nblk + turns - 1) / turns, B);
#define MCA_CALL(KP_)                                                                        \
  do {                                                                                       \
    if (zs)                                                                                  \
      k_reorth_dots<KP_, true><<<grid, kThreads, 0, s>>>(u, V, vstride, n2, nk, part, nblk,  \
                                                         ctl, cnt, h2, ncols);               \
    else                                                                                     \
      k_reorth_dots<KP_, false><<<grid, kThreads, 0, s>>>(u, V, vstride, n2, nk, part, nblk, \
                                                          ctl, cnt, h2, ncols);              \
  } while (0)
  if (nk <= 2) MCA_CALL(2);
  else if (nk <= 4) MCA_CALL(4);
  else if (nk <= 8) MCA_CALL(8);
  else if (nk <= 16) MCA_CALL(16);
  else MCA_CALL(32);
#undef MCA_CALL
}

void launch_update_norm(int phase, const double* w, size_t wstride, const double* V,
                        size_t vstride, size_t n2, int nk, const double* hc, double* part,
                        int nblk, int B, VecCtl* ctl, unsigned int* cnt, const double* h1,
                        int restart, int32_t* host_flags, double* out, size_t ostride,
                        __nv_bfloat16* xbf, int mp, int np, int m, int n, cudaStream_t s,
                        bool zs) {
  // two blocks of the summation per block, or four when their accumulators see at most two
  // entries each (then a thread would otherwise have one pair in flight)
  const bool four = n2 <= 2 * (size_t)nblk * kThreads;
  const dim3 grid(four ? (nblk + 3) / 4 : (nblk + 1) / 2, B);
  const FastDiv by_n(n);
  const int j0 = zs ? 1 : 0;
#define MCA_CALL(NK_)                                                                       \
  do {                                                                                      \
    if (four)                                                                               \
      k_update_norm<NK_, 2><<<grid, kThreads, 0, s>>>(                                      \
          phase, w, wstride, V, vstride, n2, nk, j0, hc, part, nblk, ctl, cnt, h1, restart, \
          host_flags, out, ostride, xbf, mp, np, m, n, by_n);                               \
    else                                                                                    \
      k_update_norm<NK_, 1><<<grid, kThreads, 0, s>>>(                                      \
          phase, w, wstride, V, vstride, n2, nk, j0, hc, part, nblk, ctl, cnt, h1, restart, \
          host_flags, out, ostride, xbf, mp, np, m, n, by_n);                               \
  } while (0)
  switch (nk - j0) {
    case 1: MCA_CALL(1); break;
    case 2: MCA_CALL(2); break;
    case 3: MCA_CALL(3); break;
    case 4: MCA_CALL(4); break;
    case 5: MCA_CALL(5); break;
    case 6: MCA_CALL(6); break;
    case 7: MCA_CALL(7); break;
    case 8: MCA_CALL(8); break;
    default: MCA_CALL(0); break;
  }
#undef MCA_CALL
}

template <typename ZT>
void update_x(double* x, const ZT* Z, size_t zstride, size_t n2, VecCtl* ctl, int B,
              cudaStream_t s) {
  // one block per SM slot at most, four entries per thread at least
  int nb = (int)((n2 + 4 * kThreads - 1) / (4 * kThreads));
  if (nb > 608) nb = 608;
  const dim3 grid(nb, B);
  if ((reinterpret_cast<uintptr_t>(x) & 15) == 0)
    k_update_x<ZT, 2><<<grid, kThreads, 0, s>>>(x, Z, zstride, n2, ctl);
  else
    k_update_x<ZT, 1><<<grid, kThreads, 0, s>>>(x, Z, zstride, n2, ctl);
}

void launch_update_x(double* x, const double* Z, size_t zstride, size_t n2, VecCtl* ctl,
                       int B, cudaStream_t s) {
  update_x(x, Z, zstride, n2, ctl, B, s);
}

void launch_update_x(double* x, const float* Z, size_t zstride, size_t n2, VecCtl* ctl,
                       int B, cudaStream_t s) {
  update_x(x, Z, zstride, n2, ctl, B, s);
}

}  // namespace mca

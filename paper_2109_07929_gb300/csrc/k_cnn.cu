// Learned warm start: kernels of the convolutional network that predicts the nonlinear
// correction V* - V_lin of a crossbar's node voltages from its conductance map, its input
// vector and the state V_lin after the first Newton step (the linear-circuit solve), and
// of its training on solves the method itself produces.  Not part of the paper (a
// throughput pattern layered on top of the Newton solve, which remains the judge of the
// guess: mca_solve_from).
//
// Layout: activations and gradients NHWC BF16 with 32 channels ([n][y][x][c], 64 bytes per
// pixel; channels beyond a layer's count are zero), FP32 accumulation in TMEM.  A layer is
// a K x K convolution with dilation d and zero padding d (K - 1) / 2 (output size = input
// size), plus bias and an optional leaky ReLU (slope 0.1).
//
// Convolutions are implicit GEMMs on the tcgen05 tensor cores, each in two forms:
//   forward  out[p][co] = sum_t sum_ci W[t][co][ci] x[p + off_t][ci].  k_conv_taps (32 output
//            channels, K >= 5): four taps' weights are the rows (M = 4 x 32), the pixels of an
//            input row the columns, and the drain adds the four taps' shifted rows.
//            k_conv_tc (16 output channels, small kernels, and where taps_faster finds it the
//            faster one): a CTA owns 128 pixels of one image row (M = 128, TMEM lane =
//            pixel) and all output channels (N = 16 or 32); per kernel row ky one pipeline
//            stage holds the shifted input row segment (128 + (K - 1) d pixels, out-of-range
//            pixels read as zero: the padding) in the K-major layout without swizzle, whose
//            16-byte pixel rows let the K taps of that row start at any pixel offset of the
//            same segment, plus the row's K weight tiles; two MMAs (K = 16 channels each) per
//            tap accumulate;
//   backward data is the same operation on the output gradient with the taps flipped and
//            the channel roles swapped (mca_cnn_prep_weights builds both weight tiles), with
//            the activation derivative of the layer below applied in the epilogue;
//   weight gradient gW[t][co][ci] = sum_p gz[p][co] x[p + off_t][ci], K = pixels, both
//            operands straight from the NHWC tensors as MN-major tiles.  k_wgrad_rows (K from 5
//            to 13): rows of the gradient against rows of the input, all taps of a kernel row
//            at once.  k_conv_wgrad_tc (the other kernel sizes, and where wgrad_rows_faster
//            finds it the faster one): M = 4 taps x 32 input
//            channels, N = 32 output channels, 64 consecutive pixels of a row per stage, a CTA
//            covers one group of 4 taps over a block of rows.  Both write FP32 partial sums
//            that a second kernel adds in a fixed order.
// Every mbarrier wait is bounded; an expired wait sets the module's error flag (read and
// cleared by mca_cnn_check) and the CTA leaves after freeing its TMEM.
#include <cuda.h>
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <mutex>

#include "mca_internal.cuh"
#include "precond_tc.h"
#include "tc_ptx.cuh"

namespace mca {

namespace {

using namespace tc;

constexpr int kC = 32;                 // channels of every activation tensor (padded)
constexpr int kPix = 128;              // pixels per forward tile (accumulator rows)
constexpr int kWgPix = 64;             // pixels per weight-gradient stage (K)
constexpr int kWgTaps = 4;             // taps per weight-gradient CTA (M = 4 x 32)
constexpr int kWgRows = 16;            // image rows per weight-gradient CTA
constexpr int kWgStages = 4;
constexpr int kMaxK = 15;

// module error flag (bounded waits that expired), read and cleared by mca_cnn_check
__device__ int g_cnn_err;

__device__ __forceinline__ float leaky(float z) { return z > 0.f ? z : 0.1f * z; }

// Pipeline plan of one convolution (host-computed): a stage is one kernel row ky, holding
// the input row segment as 4 chunks of 8 channels (each nbox TMA boxes of wbox 16-byte
// pixel rows, lbo bytes per chunk) and the row's K weight tiles.
struct ConvPlan {
  int wbox, nbox, lbo;
  int wrows, nwbox;     // weight rows per TMA box, boxes per kernel row (K COUT rows)
  int a_bytes, b_bytes, stage, stages;
  int smem;             // dynamic shared memory: the stages, a guard tail, barriers
};

constexpr int kConvBarBytes = 512;

template <int COUT>
ConvPlan conv_plan(int K, int d) {
  ConvPlan p{};
  const int wseg = kPix + (K - 1) * d;
  p.nbox = (wseg + 255) / 256;
  p.wbox = ((wseg + p.nbox - 1) / p.nbox + 7) / 8 * 8;
  p.lbo = p.nbox * p.wbox * 16;
  p.a_bytes = (4 * p.lbo + 1023) / 1024 * 1024;
  // the K weight tiles of a kernel row are consecutive rows of the weight tensor: one or
  // two boxes (at most 256 rows each, whole 8-row swizzle atoms)
  p.nwbox = (K * COUT + 255) / 256;
  p.wrows = ((K * COUT + p.nwbox - 1) / p.nwbox + 7) / 8 * 8;
  p.b_bytes = (p.nwbox * p.wrows * kC * 2 + 1023) / 1024 * 1024;
  p.stage = p.a_bytes + p.b_bytes;
  // the furthest byte an A descriptor can reach from its stage, also if the hardware took
  // the two strides the other way round (16 row groups lbo apart): every such address stays
  // inside the allocation
  const int reach = 18 * p.lbo + (K - 1) * d * 16 + 256;
  const int tail = reach > p.stage ? reach - p.stage : 0;
  int st = (220 * 1024 - tail - kConvBarBytes - 1024) / p.stage;
  if (st > K) st = K;
  p.stages = st;
  p.smem = st * p.stage + tail + kConvBarBytes + 1024;
  return p;
}

struct ConvArgs {
  int N, H, W;          // images, rows, columns
  int K, d, r;          // kernel size, dilation, radius (K - 1) / 2
  int cout;             // output channels written (the rest of the 32 are zero)
  const float* bias;    // forward: per output channel (NULL: none)
  int act;              // forward: leaky ReLU on the output; backward: times act'(yprev)
  int backward;         // 0 forward, 1 backward data
  const __nv_bfloat16* yprev;   // backward: NHWC32 output of the layer below (for act')
  __nv_bfloat16* out;   // NHWC32 BF16 output (may be NULL)
  float* out32;         // [N][H][W][cout] FP32 output (may be NULL)
  ConvPlan plan;
};

template <int COUT>
__global__ void __launch_bounds__(128, 1)
k_conv_tc(const __grid_constant__ CUtensorMap tmX, const __grid_constant__ CUtensorMap tmW,
          ConvArgs a) {
  const ConvPlan& P = a.plan;
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>(
      (reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
  uint64_t* full = reinterpret_cast<uint64_t*>(smem + P.smem - kConvBarBytes - 1024);
  uint64_t* empty = full + P.stages;
  uint64_t* accum = empty + P.stages;
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(accum + 1);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int x0 = blockIdx.x * kPix, y = blockIdx.y, n = blockIdx.z;
  const int S = P.stages;

  if (threadIdx.x == 0) {
    for (int s = 0; s < S; ++s) {
      mbar_init(&full[s], 1);
      mbar_init(&empty[s], 1);
    }
    mbar_init(accum, 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                     smem_u32(tmem_slot)), "r"(32u)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *tmem_slot;

  if (threadIdx.x == 0) {
    // ---------------- TMA producer: per kernel row, the input row segment (4 chunks of 8
    // channels) and the row's K weight tiles
    const uint32_t bytes = (uint32_t)(4 * P.nbox * P.wbox * 16 + P.nwbox * P.wrows * kC * 2);
    const int xs = x0 - a.r * a.d;
    for (int ky = 0; ky < a.K; ++ky) {
      const int s = ky % S;
      const uint32_t ph = (uint32_t)(ky / S) & 1u;
      if (!mbar_wait(&empty[s], ph ^ 1u)) {
        atomicCAS(&g_cnn_err, 0, MCA_ERR_TIMEOUT);
        break;
      }
      uint8_t* st = smem + s * P.stage;
      mbar_expect_tx(&full[s], bytes);
      const int yy = y + (ky - a.r) * a.d;
      for (int kc = 0; kc < 4; ++kc)
        for (int bx = 0; bx < P.nbox; ++bx)
          tma_load_4d(st + kc * P.lbo + bx * P.wbox * 16, &tmX, kc * 8, xs + bx * P.wbox, yy,
                      n, &full[s]);
      for (int bw = 0; bw < P.nwbox; ++bw)
        tma_load_2d(st + P.a_bytes + bw * P.wrows * kC * 2, &tmW, 0,
                    ky * a.K * COUT + bw * P.wrows, &full[s]);
    }
  } else if (threadIdx.x == 32) {
    // ---------------- MMA issuer: per tap (ky, kx) the window starting kx d pixels into
    // the row segment, two K = 16 steps (channel chunks 0-1 and 2-3)
    constexpr uint32_t idesc = idesc_bf16(kPix, COUT);
    bool ok = true;
    for (int ky = 0; ky < a.K; ++ky) {
      const int s = ky % S;
      const uint32_t ph = (uint32_t)(ky / S) & 1u;
      if (!mbar_wait(&full[s], ph)) {
        atomicCAS(&g_cnn_err, 0, MCA_ERR_TIMEOUT);
        ok = false;
        break;
      }
      tc_fence_after();
      const uint8_t* st = smem + s * P.stage;
      for (int kx = 0; kx < a.K; ++kx) {
#pragma unroll
        for (int kk = 0; kk < 2; ++kk)
          umma(tmem, kmajor_noswz_desc(st + kx * a.d * 16 + kk * 2 * P.lbo, P.lbo, 128),
               sw64_desc(st + P.a_bytes + kx * COUT * kC * 2 + kk * 32), idesc,
               (ky > 0 || kx > 0 || kk > 0) ? 1u : 0u);
      }
      umma_commit(&empty[s]);
    }
    if (ok) umma_commit(accum);
  }
  __syncwarp();

  // ---------------- epilogue: thread = TMEM lane = pixel x0 + 32 warp + lane
  const bool have = __syncthreads_and(mbar_wait(accum, 0) ? 1 : 0) != 0;
  if (!have && threadIdx.x == 0) atomicCAS(&g_cnn_err, 0, MCA_ERR_TIMEOUT);
  if (have) {
    tc_fence_after();
    const int x = x0 + warp * 32 + lane;
    uint32_t v[32];
    if (COUT == 32) {
      tmem_ld32(tmem + ((uint32_t)(warp * 32) << 16), v);
    } else {
      uint32_t h[16];
      tmem_ld16(tmem + ((uint32_t)(warp * 32) << 16), h);
#pragma unroll
      for (int c = 0; c < 16; ++c) v[c] = h[c];
#pragma unroll
      for (int c = 16; c < 32; ++c) v[c] = 0u;
    }
    if (x < a.W) {
      const size_t p = ((size_t)n * a.H + y) * a.W + x;
      float o[32];
      if (a.backward) {
        uint4 yp[4] = {};
        if (a.act && a.yprev) {
          const uint4* src = reinterpret_cast<const uint4*>(a.yprev + p * kC);
#pragma unroll
          for (int q = 0; q < 4; ++q) yp[q] = src[q];
        }
        const __nv_bfloat16* ypb = reinterpret_cast<const __nv_bfloat16*>(yp);
#pragma unroll
        for (int c = 0; c < 32; ++c) {
          float g = __uint_as_float(v[c]);
          if (a.act && a.yprev) g *= (__bfloat162float(ypb[c]) > 0.f) ? 1.f : 0.1f;
          o[c] = (c < a.cout) ? g : 0.f;
        }
      } else {
#pragma unroll
        for (int c = 0; c < 32; ++c) {
          float z = __uint_as_float(v[c]) + ((a.bias && c < a.cout) ? a.bias[c] : 0.f);
          if (a.act) z = leaky(z);
          o[c] = (c < a.cout) ? z : 0.f;
        }
      }
      if (a.out) {
        uint4 pk[4];
        uint32_t* w32 = reinterpret_cast<uint32_t*>(pk);
#pragma unroll
        for (int c = 0; c < 16; ++c) {
          const __nv_bfloat162 b2 = __floats2bfloat162_rn(o[2 * c], o[2 * c + 1]);
          w32[c] = *reinterpret_cast<const uint32_t*>(&b2);
        }
        uint4* dst = reinterpret_cast<uint4*>(a.out + p * kC);
#pragma unroll
        for (int q = 0; q < 4; ++q) dst[q] = pk[q];
      }
      if (a.out32) {
#pragma unroll
        for (int c = 0; c < 32; ++c)
          if (c < a.cout) a.out32[p * a.cout + c] = o[c];
      }
    }
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 1) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(32u)
                 : "memory");
  }
}

// ---- convolution with 32 output channels, weights as the M operand ----------------------
//
// k_conv_tc multiplies 128 pixels by 32 output channels per MMA: it reads 4 KB of pixels from
// shared memory for 16 clocks of work, and fills and drains its pipeline for every 128 pixels
// with the tensor core idle (347 TFLOP/s).  Here M holds 4 neighbouring taps of a kernel row x
// 32 output channels and N the pixels:
//   D_q[co][u] = sum_ky sum_g sum_ci W[ky][4 g + q][co][ci] x[y + (ky - r) d][b + u + 4 g d][ci]
// for q = 0 .. 3, b = x0 - r d: the taps of group g see a window shifted by 4 g d pixels (16-byte
// pixel rows without swizzle: any start), so that all groups add to one accumulator, and
//   out[co][x0 + p] = sum_q D_q[co][p + q d]
// is left to the epilogue: N = P + 3 d columns for P pixels.  Taps beyond the kernel row read
// as zero weights (TMA bounds), which an infinity or a NaN up to 3 d pixels outside a window turns
// into NaN: an output that comes out NaN is summed again over its own window (window_sum).
// Keeping those taps out by the MMA's lane mask took 806 us for the 32 images below, halving the
// weights of an overlapping last group in shared memory 1140.  Input rows outside the image are
// left out; as zeros they would still turn weights that are no numbers into NaN, so the drain
// looks at the weights of those kernel rows (once per CTA, while it waits) and sums the outputs
// of such channels again too.
// One persistent CTA per SM walks the tiles (P pixels of one image row): per stage, warp 0
// brings in a kernel row's weights (TMA) and 8 warps its input row, warp 1 issues 2 G MMAs of
// 128 x N x 16 into one of two accumulators, and 8 warps drain the other one, 64 pixels at a
// time.  The input rows go through 16-byte asynchronous copies: a TMA box of one 8-channel
// plane consists of 16-byte rows, and 700 of those per stage took three times its MMAs.
// Bound: no unit (tensor pipe active 31 %, L2 56 %), but the chain of a stage, copy, landing,
// MMAs and release: about 1300 clocks a stage against 430 of MMAs.  32 images of 256 x 256, 11 x
// 11, dilation 4: 1495 us, now 775 (one CTA per tile with the drain exposed: 1081; persistent with
// TMA input rows: 828).
constexpr int kTapM = 4;               // taps per M tile
constexpr int kTapPad = 36;            // floats per pixel of the epilogue's staging rows
constexpr int kTapChunk = 64;          // pixels drained at a time
constexpr int kTapMaxStages = 8;
constexpr int kTapDrain = 256;         // threads of the drain (warps 2 .. 9)
constexpr int kTapCopy = 256;          // threads of the input rows (warps 10 .. 17)
constexpr int kTapThreads = 64 + kTapDrain + kTapCopy;
constexpr int kTapStaging = kTapM * kTapChunk * kTapPad * 4;

struct TapPlan {
  int G, P, N;                         // tap groups, pixels per tile, accumulator columns
  int seg, lbo;                        // input row: pixels, bytes per plane of 8 channels
  int wb, rb, stage, stages;           // bytes of a stage's weights and input row
  int smem;
};

// False where the form does not fit.
bool tap_plan(int K, int d, int W, TapPlan& p) {
  if (K < 5) return false;             // a row of 1 or 3 taps would leave M mostly zero
  if (d > 256 / (kTapM - 1)) return false;             // (before the products below overflow)
  p.G = (K + kTapM - 1) / kTapM;
  long best = -1;
  for (int P = 16; P <= 240; P += 16) {
    const int N = (P + (kTapM - 1) * d + 15) / 16 * 16;
    if (N > 256) break;
    const long cost = (long)((W + P - 1) / P) * (N + 16);
    if (best < 0 || cost < best) {
      best = cost;
      p.P = P;
      p.N = N;
    }
  }
  if (best < 0) return false;
  p.seg = p.N + kTapM * (p.G - 1) * d;
  // planes 2 x 16 bytes apart modulo 128: the copies of two pixels' four planes hit
  // different banks
  p.lbo = ((p.seg + 5) / 8 * 8 + 2) * 16;
  p.rb = (4 * p.lbo + 1023) / 1024 * 1024;
  p.wb = p.G * kTapM * kC * kC * 2;
  p.stage = p.wb + p.rb;
  const int room = 224 * 1024 - kTapStaging;
  p.stages = room / p.stage < kTapMaxStages ? room / p.stage : kTapMaxStages;
  if (p.stages < 2) return false;
  p.smem = p.stages * p.stage + kTapStaging + 512 + 1024;
  return true;
}

// Which form of a convolution is the faster one, by the time (us) that each takes on `sms` SMs,
// fitted to 415 layers of 1 to 32 images (kernels 5 to 15, dilations up to where k_conv_tc ends;
// mean error 9 % and 12 %).  k_conv_taps: its stages' bytes, for the kernel rows inside the image
// (more where only two stages fit), and its drain per 64 pixels, over the waves of tiles; large
// dilations leave few pixels of its 256 columns (1024 x 1024, K = 5: d = 32 256 us against 307,
// d = 48 358 and 345, d = 70 1224 and 405), and one wave of wide tiles is mostly its pipeline's
// start (17 x 500, 2 images, K = 5: 12.8 us against 8.9).  k_conv_tc: K stages per tile of 128
// pixels, with the segment's length.  The line lies at 1.05, for the fit's own error: of the 415
// layers, one is then slower than in k_conv_tc (12.4 against 10.7 us), 32 with k_conv_taps alone.
bool taps_faster(const TapPlan& p, int n, int h, int w, int K, int d, int sms) {
  const double images_rows = (double)n * h;
  double inside = 0.0;                   // kernel rows inside the image, mean over its rows
  for (int ky = 0; ky < K; ++ky) inside += std::max(0, h - std::abs(ky - K / 2) * d) / (double)h;
  const double waves = std::ceil(images_rows * ((w + p.P - 1) / p.P) / sms);
  const double waves_tc = std::ceil(images_rows * ((w + kPix - 1) / kPix) / sms);
  const double kb = p.stage / 1024.0;
  const double taps = 6.5 + waves * (inside * kb * (p.stages > 2 ? 0.0156 : 0.0258) +
                                     0.8 * ((p.P + kTapChunk - 1) / kTapChunk)) + 0.23 * K;
  const double tc = 4.8 + waves_tc * (K * (0.67 + 0.045 * K) + 0.010 * (K - 1) * d);
  return 1.05 * taps <= tc;
}

struct TapArgs {
  int H, W, K, d, r;
  int xt, tiles;                       // tiles per image row and in all
  int cout;
  const __nv_bfloat16 *x, *w;          // w: [ky][kx][co][ci]
  const float* bias;
  int act, backward;
  const __nv_bfloat16* yprev;
  __nv_bfloat16* out;
  float* out32;
  TapPlan plan;
};

// The convolution's sum of channel co at pixel (y, x) of image n, without bias, term by term: for
// outputs in whose accumulators an infinity or a NaN has been.  Ends at a NaN.
__device__ __forceinline__ float window_sum(const TapArgs& a, int n, int y, int x, int co) {
  float s = 0.f;
#pragma unroll 1
  for (int ky = 0; ky < a.K; ++ky) {
    const int yy = y + (ky - a.r) * a.d;
    const bool row = yy >= 0 && yy < a.H;
#pragma unroll 1
    for (int kx = 0; kx < a.K && s == s; ++kx) {
      const int xx = x + (kx - a.r) * a.d;
      const bool in = row && xx >= 0 && xx < a.W;
      const __nv_bfloat16* px = a.x + (in ? (((size_t)n * a.H + yy) * a.W + xx) * kC : 0);
      const __nv_bfloat16* wt = a.w + ((size_t)(ky * a.K + kx) * kC + co) * kC;
#pragma unroll 1
      for (int ci = 0; ci < kC; ++ci)
        s = fmaf(in ? __bfloat162float(px[ci]) : 0.f, __bfloat162float(wt[ci]), s);
    }
  }
  return s;
}

// 16 bytes to shared memory, zeros when !ok (src must be readable memory either way)
__device__ __forceinline__ void copy16_async(uint32_t dst, const void* src, bool ok) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(src),
               "r"(ok ? 16 : 0)
               : "memory");
}

// At most LEFT of this thread's newest copy groups may still be in flight.
template <int LEFT>
__device__ __forceinline__ void copies_wait() {
  asm volatile("cp.async.wait_group %0;" ::"n"(LEFT) : "memory");
}

__global__ void __launch_bounds__(kTapThreads, 1)
k_conv_taps(const __grid_constant__ CUtensorMap tmW, const __grid_constant__ TapArgs a) {
  const TapPlan& P = a.plan;
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>(
      (reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
  const int S = P.stages;
  float* stg = reinterpret_cast<float*>(smem + S * P.stage);
  uint64_t* full = reinterpret_cast<uint64_t*>(smem + S * P.stage + kTapStaging);
  uint64_t* empty = full + kTapMaxStages;
  uint64_t* tfull = empty + kTapMaxStages;           // [2] accumulator complete
  uint64_t* tempty = tfull + 2;                      // [2] accumulator drained
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(tempty + 2);
  volatile uint32_t& dead = tmem_slot[1];            // a drain warp's wait gave up
  uint32_t* wbad = tmem_slot + 2;                    // channels without numbers per kernel row; any
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int d = a.d;
  // tile t: P pixels from x0 of row y of image n, and the kernel rows that meet the image
  auto decode = [&](int t, int& n, int& y, int& x0, int& k0, int& k1) {
    const int row = t / a.xt;
    x0 = (t - row * a.xt) * P.P;
    n = row / a.H;
    y = row - n * a.H;
    k0 = max(0, a.r - y / d);
    k1 = min(a.K - 1, a.r + (a.H - 1 - y) / d);
  };
  if (threadIdx.x <= kMaxK) wbad[threadIdx.x] = 0;
  if (threadIdx.x == 0) {
    dead = 0;
    for (int s = 0; s < S; ++s) {
      mbar_init(&full[s], 1 + kTapCopy);
      mbar_init(&empty[s], 1);
    }
    for (int q = 0; q < 2; ++q) {
      mbar_init(&tfull[q], 1);
      mbar_init(&tempty[q], kTapDrain / 32);
    }
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                     smem_u32(tmem_slot)), "r"(512u)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *tmem_slot;

  if (warp == 0) {
    if (lane == 0) {
      int it = 0;
      bool ok = true;
      for (int t = blockIdx.x; t < a.tiles && ok; t += gridDim.x) {
        int n, y, x0, k0, k1;
        decode(t, n, y, x0, k0, k1);
        for (int ky = k0; ky <= k1; ++ky, ++it) {
          const int s = it % S;
          if (!mbar_wait(&empty[s], ((uint32_t)(it / S) & 1u) ^ 1u)) {
            atomicCAS(&g_cnn_err, 0, MCA_ERR_TIMEOUT);
            ok = false;
            break;
          }
          uint8_t* st = smem + s * P.stage;
          mbar_expect_tx(&full[s], (uint32_t)P.wb);
          for (int g = 0; g < P.G; ++g)
            tma_load_4d(st + g * kTapM * kC * kC * 2, &tmW, 0, 0, g * kTapM, ky, &full[s]);
        }
      }
    }
  } else if (warp == 1) {
    if (lane == 0) {
      const uint32_t idesc = idesc_bf16(kTapM * kC, P.N);
      int it = 0, tl = 0;
      bool ok = true;
      for (int t = blockIdx.x; t < a.tiles && ok; t += gridDim.x, ++tl) {
        int n, y, x0, k0, k1;
        decode(t, n, y, x0, k0, k1);
        const int acc = tl & 1;
        if (!mbar_wait(&tempty[acc], ((uint32_t)(tl >> 1) & 1u) ^ 1u)) {
          atomicCAS(&g_cnn_err, 0, MCA_ERR_TIMEOUT);
          break;
        }
        tc_fence_after();
        const uint32_t dst = tmem + (uint32_t)(acc * 256);
        for (int ky = k0; ky <= k1; ++ky, ++it) {
          const int s = it % S;
          if (!mbar_wait(&full[s], (uint32_t)(it / S) & 1u)) {
            atomicCAS(&g_cnn_err, 0, MCA_ERR_TIMEOUT);
            ok = false;
            break;
          }
          tc_fence_after();
          const uint8_t* wt = smem + s * P.stage;
          const uint8_t* row = wt + P.wb;
          for (int g = 0; g < P.G; ++g) {
#pragma unroll
            for (int kk = 0; kk < 2; ++kk)
              umma(dst, sw64_desc(wt + g * kTapM * kC * kC * 2 + kk * 32),
                   kmajor_noswz_desc(row + kTapM * g * d * 16 + kk * 2 * P.lbo, P.lbo, 128), idesc,
                   (ky > k0 || g > 0 || kk > 0) ? 1u : 0u);
          }
          umma_commit(&empty[s]);
        }
        if (ok) umma_commit(&tfull[acc]);
      }
    }
  } else if (warp >= 2 + kTapDrain / 32) {
    // ---------------- input rows: pixel-major 16-byte copies into the four planes; a row is
    // reported one row later, when its copies have landed (the slot of row `it` is free once
    // row it - S is consumed, and S >= 2; reporting three rows later left the MMAs too few
    // rows ahead: 257 against 202 us per layer at 8 images of 256 x 256)
    const int tid = threadIdx.x - 64 - kTapDrain;
    constexpr int lag = 1;
    auto report = [&](int it) {
      asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
      asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(&full[it % S]))
                   : "memory");
    };
    int it = 0;
    bool ok = true;
    for (int t = blockIdx.x; t < a.tiles && ok; t += gridDim.x) {
      int n, y, x0, k0, k1;
      decode(t, n, y, x0, k0, k1);
      for (int ky = k0; ky <= k1; ++ky, ++it) {
        const int s = it % S;
        if (!mbar_wait(&empty[s], ((uint32_t)(it / S) & 1u) ^ 1u)) {
          atomicCAS(&g_cnn_err, 0, MCA_ERR_TIMEOUT);
          ok = false;
          break;
        }
        const uint32_t dst = smem_u32(smem + s * P.stage + P.wb);
        const __nv_bfloat16* src =
            a.x + ((size_t)n * a.H + (y + (ky - a.r) * d)) * a.W * kC;
        for (int e = tid; e < P.seg * 4; e += kTapCopy) {
          const int px = e >> 2, kc = e & 3, xx = x0 - a.r * d + px;
          const bool in = xx >= 0 && xx < a.W;
          copy16_async(dst + kc * P.lbo + px * 16, src + (size_t)(in ? xx : 0) * kC + kc * 8, in);
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
        if (it >= lag) {
          copies_wait<lag>();
          report(it - lag);
        }
      }
    }
    copies_wait<0>();                          // (also after a timeout: no copy outlives the CTA)
    if (ok)
      for (int r = it - lag > 0 ? it - lag : 0; r < it; ++r) report(r);
  } else {
    // ---------------- drain: 64 pixels at a time, the four taps' accumulators to shared memory
    // as [q][pixel][channel], shifted by q d (a warp reads the lanes of tap warp % 4), then one
    // thread per pixel and 8 channels adds them
    const int q = warp & 3, hf = (warp - 2) >> 2, tid = threadIdx.x - 64;
    const int pl = tid >> 2, c8 = (tid & 3) * 8;
    float bias[8];
#pragma unroll
    for (int c = 0; c < 8; ++c)
      bias[c] = (!a.backward && a.bias && c8 + c < a.cout) ? a.bias[c8 + c] : 0.f;
    const bool gate = a.backward && a.act && a.yprev;
    // the weights of kernel rows outside the image of any of the CTA's tiles: [0, lo), [hi, K)
    int lo = 0, hi = a.K;
    for (int t = blockIdx.x + lane * gridDim.x; t < a.tiles; t += 32 * gridDim.x) {
      int n, y, x0, k0, k1;
      decode(t, n, y, x0, k0, k1);
      lo = max(lo, k0);
      hi = min(hi, k1 + 1);
    }
    lo = __reduce_max_sync(0xffffffffu, lo);
    hi = __reduce_min_sync(0xffffffffu, hi);
    const int per_row = a.K * (kC * kC / 8);           // 16-byte pieces of a row's weights
    const int skip = (hi - lo) * per_row, all = (a.K - (hi - lo)) * per_row;
    constexpr int kLook = 8;                           // loads in flight per thread
    for (int e0 = tid; e0 < all; e0 += kLook * kTapDrain) {
      uint4 u[kLook];
#pragma unroll
      for (int q = 0; q < kLook; ++q) {
        const int e = min(e0 + q * kTapDrain, all - 1);
        u[q] = reinterpret_cast<const uint4*>(a.w)[e + (e >= lo * per_row ? skip : 0)];
      }
      uint32_t nan = 0;
#pragma unroll
      for (int q = 0; q < kLook; ++q) {
        const uint32_t v[4] = {u[q].x, u[q].y, u[q].z, u[q].w};
#pragma unroll
        for (int k = 0; k < 4; ++k)
          if ((v[k] & 0x7F80u) == 0x7F80u || (v[k] & 0x7F800000u) == 0x7F800000u) nan |= 1u << q;
      }
      for (; nan != 0; nan &= nan - 1) {
        int e = min(e0 + (__ffs(nan) - 1) * kTapDrain, all - 1);
        e += (e >= lo * per_row) ? skip : 0;
        atomicOr(&wbad[e / per_row], 1u << ((e >> 2) & (kC - 1)));
        wbad[kMaxK] = 1;
      }
    }
    int tl = 0;
    for (int t = blockIdx.x; t < a.tiles; t += gridDim.x, ++tl) {
      int n, y, x0, k0, k1;
      decode(t, n, y, x0, k0, k1);
      const int acc = tl & 1;
      const bool have = __all_sync(0xffffffffu,
                                   mbar_wait(&tfull[acc], (uint32_t)(tl >> 1) & 1u) ? 1 : 0) != 0;
      if (!have && lane == 0) {
        atomicCAS(&g_cnn_err, 0, MCA_ERR_TIMEOUT);
        dead = 1;
      }
      asm volatile("bar.sync 1, %0;" ::"n"(kTapDrain) : "memory");
      if (dead) break;                 // (all 8 warps: a wait that gave up)
      tc_fence_after();
      uint32_t bad = 0;                // channels whose weights outside the image are no numbers
      if (wbad[kMaxK])
        for (int ky = 0; ky < a.K; ++ky) bad |= (ky < k0 || ky > k1) ? wbad[ky] : 0u;
      for (int p0 = 0; p0 < P.P; p0 += kTapChunk) {
        const int p = p0 + pl, x = x0 + p;
        const bool in = p < P.P && x < a.W;
        const size_t px = ((size_t)n * a.H + y) * a.W + x;
        uint4 yp = {};
        if (gate && in) yp = *reinterpret_cast<const uint4*>(a.yprev + px * kC + c8);
        // columns p0 + q d .. + 63 of this tap, in 16-column blocks
        const int first = p0 + q * d;
        const int c1 = min(P.N, first + kTapChunk);
        for (int c0 = first / 16 * 16 + hf * 16; c0 < c1; c0 += 32) {
          uint32_t v[16];
          tmem_ld16(tmem + (uint32_t)(acc * 256 + c0) + ((uint32_t)(q * 32) << 16), v);
#pragma unroll
          for (int j = 0; j < 16; ++j) {
            const int u = c0 + j - first;
            if (u >= 0 && u < kTapChunk)
              stg[(q * kTapChunk + u) * kTapPad + lane] = __uint_as_float(v[j]);
          }
        }
        asm volatile("bar.sync 1, %0;" ::"n"(kTapDrain) : "memory");
        if (in) {
          float o[8] = {};
#pragma unroll
          for (int k = 0; k < kTapM; ++k) {
            const float4* src =
                reinterpret_cast<const float4*>(stg + (k * kTapChunk + pl) * kTapPad + c8);
            const float4 u = src[0], w = src[1];
            o[0] += u.x; o[1] += u.y; o[2] += u.z; o[3] += u.w;
            o[4] += w.x; o[5] += w.y; o[6] += w.z; o[7] += w.w;
          }
          const float any = ((o[0] + o[1]) + (o[2] + o[3])) + ((o[4] + o[5]) + (o[6] + o[7]));
          if (any != any || ((bad >> c8) & 0xFFu) != 0) {
#pragma unroll 1
            for (int c = 0; c < 8; ++c) {
              const float sum = window_sum(a, n, y, x, c8 + c);
#pragma unroll
              for (int k = 0; k < 8; ++k) o[k] = (k == c) ? sum : o[k];
            }
          }
          const __nv_bfloat16* ypb = reinterpret_cast<const __nv_bfloat16*>(&yp);
#pragma unroll
          for (int c = 0; c < 8; ++c) {
            if (gate) {
              o[c] *= (__bfloat162float(ypb[c]) > 0.f) ? 1.f : 0.1f;
            } else if (!a.backward) {
              o[c] += bias[c];
              if (a.act) o[c] = leaky(o[c]);
            }
            if (c8 + c >= a.cout) o[c] = 0.f;
          }
          if (a.out) {
            uint4 pk;
            uint32_t* w32 = reinterpret_cast<uint32_t*>(&pk);
#pragma unroll
            for (int c = 0; c < 4; ++c) {
              const __nv_bfloat162 b2 = __floats2bfloat162_rn(o[2 * c], o[2 * c + 1]);
              w32[c] = *reinterpret_cast<const uint32_t*>(&b2);
            }
            *reinterpret_cast<uint4*>(a.out + px * kC + c8) = pk;
          }
          if (a.out32) {
#pragma unroll
            for (int c = 0; c < 8; ++c)
              if (c8 + c < a.cout) a.out32[px * a.cout + c8 + c] = o[c];
          }
        }
        asm volatile("bar.sync 1, %0;" ::"n"(kTapDrain) : "memory");
      }
      tc_fence_before();
      __syncwarp();
      if (lane == 0)
        asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(&tempty[acc]))
                     : "memory");
    }
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 1) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(512u)
                 : "memory");
  }
}

// ---- weight gradient ------------------------------------------------------------------

struct WgLayout {
  static constexpr int A_TAP = kWgPix * kC * 2;                       // 4 KB per tap
  static constexpr int A_BYTES = kWgTaps * A_TAP;
  static constexpr int B_BYTES = kWgPix * kC * 2;
  static constexpr int STAGE = A_BYTES + B_BYTES;                     // 20 KB
  static constexpr int BAR_OFF = kWgStages * STAGE;
  static constexpr int SMEM = BAR_OFF + 256 + 1024;
};

struct WgArgs {
  int N, H, W, K, d, r;
  int rows_total;       // N * H
  int nxc;              // 64-pixel chunks per row
  float* part;          // [chunk][t][ci 32][co 32]
};

// CTA (group g of 4 taps, block of kWgRows image rows): D[(tap, ci)][co] accumulated over
// the block's pixels; A tile of tap tl = 64 pixels x 32 channels of the shifted input row
// (MN-major: the 32 channels of a pixel are one 64-byte row), B tile = the same pixels of
// the output gradient.
__global__ void __launch_bounds__(128, 2)
k_conv_wgrad_tc(const __grid_constant__ CUtensorMap tmX, const __grid_constant__ CUtensorMap tmG,
                WgArgs a) {
  using L = WgLayout;
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>(
      (reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
  uint64_t* full = reinterpret_cast<uint64_t*>(smem + L::BAR_OFF);
  uint64_t* empty = full + kWgStages;
  uint64_t* accum = empty + kWgStages;
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(accum + 1);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int g = blockIdx.x, chunk = blockIdx.y;
  const int T = a.K * a.K;
  const int t0 = g * kWgTaps;
  const int ntg = (T - t0 < kWgTaps) ? T - t0 : kWgTaps;
  const int row0 = chunk * kWgRows;
  const int nrows = (a.rows_total - row0 < kWgRows) ? a.rows_total - row0 : kWgRows;
  const int nsteps = nrows * a.nxc;

  if (threadIdx.x == 0) {
    for (int s = 0; s < kWgStages; ++s) {
      mbar_init(&full[s], 1);
      mbar_init(&empty[s], 1);
    }
    mbar_init(accum, 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                     smem_u32(tmem_slot)), "r"(32u)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *tmem_slot;

  if (threadIdx.x == 0) {
    for (int it = 0; it < nsteps; ++it) {
      const int s = it % kWgStages;
      const uint32_t ph = (uint32_t)(it / kWgStages) & 1u;
      if (!mbar_wait(&empty[s], ph ^ 1u)) {
        atomicCAS(&g_cnn_err, 0, MCA_ERR_TIMEOUT);
        break;
      }
      uint8_t* st = smem + s * L::STAGE;
      mbar_expect_tx(&full[s], (uint32_t)(ntg * L::A_TAP + L::B_BYTES));
      const int row = row0 + it / a.nxc;
      const int x0 = (it - (it / a.nxc) * a.nxc) * kWgPix;
      const int n = row / a.H, y = row - n * a.H;
      for (int tl = 0; tl < ntg; ++tl) {
        const int t = t0 + tl, ky = t / a.K, kx = t - ky * a.K;
        tma_load_4d(st + tl * L::A_TAP, &tmX, 0, x0 + (kx - a.r) * a.d, y + (ky - a.r) * a.d,
                    n, &full[s]);
      }
      tma_load_4d(st + L::A_BYTES, &tmG, 0, x0, y, n, &full[s]);
    }
  } else if (threadIdx.x == 32) {
    constexpr uint32_t idesc = idesc_bf16_mn(128, kC);
    bool ok = true;
    for (int it = 0; it < nsteps; ++it) {
      const int s = it % kWgStages;
      const uint32_t ph = (uint32_t)(it / kWgStages) & 1u;
      if (!mbar_wait(&full[s], ph)) {
        atomicCAS(&g_cnn_err, 0, MCA_ERR_TIMEOUT);
        ok = false;
        break;
      }
      tc_fence_after();
      const uint8_t* st = smem + s * L::STAGE;
      // K = 16 pixels per MMA: 16 rows of 64 bytes, two 8-row groups 512 bytes apart; the
      // A atoms along M (one per tap) are L::A_TAP apart; B is a single atom along N, so its
      // atom stride is never used (512 keeps every address inside the stage either way)
#pragma unroll
      for (int kk = 0; kk < kWgPix / 16; ++kk)
        umma(tmem, sw64_mn_desc(st + kk * 1024, L::A_TAP, 512),
             sw64_mn_desc(st + L::A_BYTES + kk * 1024, 512, 512), idesc,
             (it > 0 || kk > 0) ? 1u : 0u);
      umma_commit(&empty[s]);
    }
    if (ok && nsteps > 0) umma_commit(accum);
  }
  __syncwarp();

  const bool have = nsteps > 0 && __syncthreads_and(mbar_wait(accum, 0) ? 1 : 0) != 0;
  if (nsteps > 0 && !have && threadIdx.x == 0) atomicCAS(&g_cnn_err, 0, MCA_ERR_TIMEOUT);
  if (have) {
    tc_fence_after();
    // thread = TMEM lane = (tap warp, input channel lane)
    uint32_t v[32];
    tmem_ld32(tmem + ((uint32_t)(warp * 32) << 16), v);
    if (warp < ntg) {
      float4* dst = reinterpret_cast<float4*>(
          a.part + (((size_t)chunk * T + t0 + warp) * kC + lane) * kC);
#pragma unroll
      for (int q = 0; q < 8; ++q)
        dst[q] = make_float4(__uint_as_float(v[4 * q]), __uint_as_float(v[4 * q + 1]),
                             __uint_as_float(v[4 * q + 2]), __uint_as_float(v[4 * q + 3]));
    }
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 1) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(32u)
                 : "memory");
  }
}

// ---- weight gradient, rows against rows --------------------------------------------------
//
// k_conv_wgrad_tc brings 20 KB through shared memory per 64 pixels for 4 MMAs of 16 clocks'
// work (201 TFLOP/s).  Here a CTA owns one kernel column kx and
// multiplies 4 gradient rows y + j d (M = 4 x 32 output channels) by the K + 3 input rows
// y + (i - r) d shifted by (kx - r) d pixels (N = 32 (K + 3) input channels, at most the 512
// TMEM columns):
//   D[(j, co)][(i, ci)] = sum_x gz[y + j d][x][co] x[y + (i - r) d][x + (kx - r) d][ci],
// whose blocks i = j + ky are the four rows' parts of tap (ky, kx): 4 K of 4 (K + 3) blocks
// are used, and 72 KB per 64 pixels feed 900 clocks of MMAs (K = 11).  D accumulates over a
// share of the images' row blocks; the epilogue adds the four diagonals and writes one
// partial sum per CTA.  Gradient rows beyond the image, where the row blocks do not divide H,
// are kept out of D by the MMA's lane mask and not only by their zeros, which an infinity or a
// NaN in x would turn into NaN; D starts from zeros, so that every MMA can have a mask.
// Bound: the stages in flight, three of 72 KB (tensor pipe active 42 %, L2 41 %).  32 images of
// 256 x 256, 11 x 11, dilation 4, with the sums behind it: 2779 us per call, now 687.
constexpr int kWrJ = 4;                                 // gradient rows per CTA step
constexpr int kWrRow = kWgPix * kC * 2;                 // 64 pixels of a row: 4 KB
constexpr int kWrMaxK = 512 / kC - (kWrJ - 1);          // 13
constexpr int kWrStages = 3;                            // (2 where 3 do not fit: K = 13)
// Row-block chunks per partial sum, at most: 256 MMA steps per accumulator, as many as the
// other form takes on 256-pixel rows, and on narrower rows its number there, kWgRows rows of
// chunks (the tensor core's FP32 sums lose about a rounding per step.  32 images of 92 x 92,
// dilation 8, 11 x 11: relative error against FP64 2.0e-6 with up to 64, 1.1e-6 with up to
// 32; the other form's 1.4e-6)
constexpr int kWrItems = 64;

struct WrArgs {
  int H, K, d, r;
  int stages;
  int blocks;            // row blocks of one image
  int items;             // N * blocks * nxc
  int nxc;               // 64-pixel chunks per row
  float* part;           // [chunk][t][ci 32][co 32]
};

struct WrPlan {
  int blocks, nxc, items, chunks;
};

// nmax: partial sums that the scratch holds
WrPlan wgrad_rows_plan(int n, int h, int w, int K, int d, int nmax, int sms) {
  WrPlan p{};
  const int64_t period = (int64_t)kWrJ * d;          // image rows of d row blocks
  p.blocks = (int)(h / period * d + std::min<int64_t>(h % period, d));
  p.nxc = (w + kWgPix - 1) / kWgPix;
  p.items = n * p.blocks * p.nxc;
  const int most = std::min(kWrItems, kWgRows * p.nxc);
  p.chunks = (p.items + most - 1) / most;
  // whole waves of CTAs (one resides per SM), two at least: 11 images of 187 x 187, dilation 8,
  // 182 us per call with 33 chunks (2.4 waves), 158 with 41; 32 of 256 x 256, 717 and 685
  const int waves = std::max(2, (K * p.chunks + sms - 1) / sms);
  p.chunks = std::max(p.chunks, waves * sms / K);
  p.chunks = std::min(p.chunks, std::min(nmax, p.items));
  return p;
}

// Which form is the faster one, by the time (us) of each with its sums, fitted to 375 layers of 1
// to 32 images (kernels 5 to 13; mean error 13 % and 16 %): the steps of k_wgrad_rows' waves
// against the per-tap form's groups of four taps.  Images of fewer rows than four dilations leave
// most of a row block's gradient rows outside (27 images of 21 x 169, K = 5, d = 53: 88 us against
// 48; 12 of 12 x 15, K = 7, d = 32: 36 and 21).  The line lies at 1.1, for the fit's own error: of
// the 375 layers, three are then slower than in the per-tap form, by 6 % at most, 53 with
// k_wgrad_rows alone.
bool wgrad_rows_faster(const WrPlan& p, int n, int h, int w, int K, int nmax, int sms) {
  const int taps = K * K, steps = (p.items + p.chunks - 1) / p.chunks;
  const int waves = (K * p.chunks + sms - 1) / sms;
  const double rows = 13.7 + waves * (0.0577 * steps * (K + 7) + 0.296 * K) +
                      0.0011 * p.chunks * taps;
  const double share = (double)std::min<int64_t>(kWgRows, (int64_t)n * h) * p.nxc;
  const double groups = (double)((taps + kWgTaps - 1) / kWgTaps) * nmax;
  const double per_tap = 12.2 + share * (0.351 * groups / sms + 0.507) + 0.00164 * nmax * taps;
  return 1.1 * rows <= per_tap;
}

__global__ void __launch_bounds__(128, 1)
k_wgrad_rows(const __grid_constant__ CUtensorMap tmX, const __grid_constant__ CUtensorMap tmG,
             WrArgs a) {
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>(
      (reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
  const int rows = a.K + kWrJ - 1, stage = (rows + kWrJ) * kWrRow, S = a.stages;
  uint64_t* full = reinterpret_cast<uint64_t*>(smem + S * stage);
  uint64_t* empty = full + S;
  uint64_t* accum = empty + S;
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(accum + 1);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int kx = blockIdx.x, chunk = blockIdx.y;
  const int it0 = (int)((long long)a.items * chunk / gridDim.y);
  const int steps = (int)((long long)a.items * (chunk + 1) / gridDim.y) - it0;
  if (threadIdx.x == 0) {
    for (int s = 0; s < S; ++s) {
      mbar_init(&full[s], 1);
      mbar_init(&empty[s], 1);
    }
    mbar_init(accum, 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                     smem_u32(tmem_slot)), "r"(512u)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *tmem_slot;
  for (int c = 0; c < rows; ++c)
    tmem_zero32(tmem + (uint32_t)(c * kC) + ((uint32_t)(warp * 32) << 16));
  asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  // first gradient row of a row block, and the image n and pixel x0 of an item
  auto first_row = [&](int item, int& n, int& x0) {
    const int rb = item / a.nxc;
    x0 = (item - rb * a.nxc) * kWgPix;
    n = rb / a.blocks;
    const int blk = rb - n * a.blocks;
    return blk / a.d * kWrJ * a.d + blk % a.d;
  };
  if (threadIdx.x == 0) {
    for (int it = 0; it < steps; ++it) {
      const int s = it % S;
      if (!mbar_wait(&empty[s], ((uint32_t)(it / S) & 1u) ^ 1u)) {
        atomicCAS(&g_cnn_err, 0, MCA_ERR_TIMEOUT);
        break;
      }
      uint8_t* st = smem + s * stage;
      mbar_expect_tx(&full[s], (uint32_t)stage);
      int n, x0;
      const int y = first_row(it0 + it, n, x0);
      for (int j = 0; j < kWrJ; ++j)
        tma_load_4d(st + j * kWrRow, &tmG, 0, x0, y + j * a.d, n, &full[s]);
      for (int i = 0; i < rows; ++i)
        tma_load_4d(st + (kWrJ + i) * kWrRow, &tmX, 0, x0 + (kx - a.r) * a.d,
                    y + (i - a.r) * a.d, n, &full[s]);
    }
  } else if (threadIdx.x == 32) {
    const int n1 = rows * kC < 256 ? rows * kC : 256, n2 = rows * kC - n1;
    const uint32_t id1 = idesc_bf16_mn(128, n1), id2 = idesc_bf16_mn(128, n2 > 0 ? n2 : 32);
    bool ok = true;
    for (int it = 0; it < steps; ++it) {
      const int s = it % S;
      if (!mbar_wait(&full[s], (uint32_t)(it / S) & 1u)) {
        atomicCAS(&g_cnn_err, 0, MCA_ERR_TIMEOUT);
        ok = false;
        break;
      }
      tc_fence_after();
      const uint8_t* g = smem + s * stage;
      const uint8_t* x = g + kWrJ * kWrRow;
      int n, x0;
      const int y = first_row(it0 + it, n, x0);
      uint32_t off[kWrJ];
#pragma unroll
      for (int j = 0; j < kWrJ; ++j) off[j] = (y + j * a.d < a.H) ? 0u : 0xffffffffu;
#pragma unroll
      for (int kk = 0; kk < kWgPix / 16; ++kk) {
        const uint64_t ad = sw64_mn_desc(g + kk * 1024, kWrRow, 512);
        umma_lanes(tmem, ad, sw64_mn_desc(x + kk * 1024, kWrRow, 512), id1, 1u, off);
        if (n2 > 0)
          umma_lanes(tmem + 256, ad, sw64_mn_desc(x + 8 * kWrRow + kk * 1024, kWrRow, 512), id2,
                     1u, off);
      }
      umma_commit(&empty[s]);
    }
    if (ok && steps > 0) umma_commit(accum);
  }
  __syncwarp();
  const bool have = steps > 0 && __syncthreads_and(mbar_wait(accum, 0) ? 1 : 0) != 0;
  if (steps > 0 && !have && threadIdx.x == 0) atomicCAS(&g_cnn_err, 0, MCA_ERR_TIMEOUT);
  if (have || steps == 0) {
    tc_fence_after();
    float* stg = reinterpret_cast<float*>(smem);       // [j][ci][co]
    const size_t T = (size_t)a.K * a.K;
    for (int ky = 0; ky < a.K; ++ky) {
      uint32_t v[32] = {};
      if (have) tmem_ld32(tmem + (uint32_t)((warp + ky) * kC) + ((uint32_t)(warp * 32) << 16), v);
#pragma unroll
      for (int ci = 0; ci < kC; ++ci) stg[(warp * kC + ci) * kC + lane] = __uint_as_float(v[ci]);
      __syncthreads();
      float* dst = a.part + ((size_t)chunk * T + (size_t)ky * a.K + kx) * kC * kC;
      for (int e = threadIdx.x; e < kC * kC; e += 128)
        dst[e] = (stg[e] + stg[kC * kC + e]) + (stg[2 * kC * kC + e] + stg[3 * kC * kC + e]);
      __syncthreads();
    }
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 1) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(512u)
                 : "memory");
  }
}

// gw[co][ci][t] = sum over chunks of part[chunk][t][ci][co] (fixed order), co < cout,
// ci < cin: the master weight layout [cout][cin][K][K].
__global__ void k_wgrad_reduce(const float* __restrict__ part, int nchunk, int T, int cin,
                               int cout, float* __restrict__ gw) {
  const size_t total = (size_t)T * cin * cout;
  for (size_t e = blockIdx.x * (size_t)blockDim.x + threadIdx.x; e < total;
       e += (size_t)gridDim.x * blockDim.x) {
    const int co = (int)(e % cout);
    const size_t r = e / cout;
    const int ci = (int)(r % cin);
    const int t = (int)(r / cin);
    const size_t off = ((size_t)t * kC + ci) * kC + co;
    float s = 0.f;
    for (int c = 0; c < nchunk; ++c) s += part[(size_t)c * T * kC * kC + off];
    gw[((size_t)co * cin + ci) * T + t] = s;
  }
}

// Partial sums of the bias gradient gb[co] = sum_p gz[p][co]: block b sums its pixels.
__global__ void k_bias_grad_part(const __nv_bfloat16* __restrict__ gz, size_t npix, int cout,
                                 float* __restrict__ part) {
  __shared__ float red[8][kC];
  float acc[kC];
#pragma unroll
  for (int c = 0; c < kC; ++c) acc[c] = 0.f;
  for (size_t p = blockIdx.x * (size_t)blockDim.x + threadIdx.x; p < npix;
       p += (size_t)gridDim.x * blockDim.x) {
    const uint4* src = reinterpret_cast<const uint4*>(gz + p * kC);
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const uint4 u = src[q];
      const __nv_bfloat16* b = reinterpret_cast<const __nv_bfloat16*>(&u);
#pragma unroll
      for (int c = 0; c < 8; ++c) acc[q * 8 + c] += __bfloat162float(b[c]);
    }
  }
  const int w = threadIdx.x >> 5, l = threadIdx.x & 31;
#pragma unroll
  for (int c = 0; c < kC; ++c) {
    float v = acc[c];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    if (l == 0) red[w][c] = v;
  }
  __syncthreads();
  if (threadIdx.x < kC) {
    float s = 0.f;
    for (int q = 0; q < (int)(blockDim.x >> 5); ++q) s += red[q][threadIdx.x];
    part[(size_t)blockIdx.x * kC + threadIdx.x] = s;
  }
}

// gb[c] from the nb blocks' sums: 32 x 32 threads, thread (g, c) sums the blocks g, g + 32,
// ..., then one warp adds the 32 sums in order (one thread per channel over 4096 blocks took
// 92 us).
__global__ void __launch_bounds__(1024)
k_bias_grad_finish(const float* __restrict__ part, int nb, int cout, float* __restrict__ gb) {
  __shared__ float red[32][kC];
  const int c = threadIdx.x & 31, g = threadIdx.x >> 5;
  float s = 0.f;
  for (int b = g; b < nb; b += 32) s += part[(size_t)b * kC + c];
  red[g][c] = s;
  __syncthreads();
  if (g == 0 && c < cout) {
    float t = 0.f;
    for (int q = 0; q < 32; ++q) t += red[q][c];
    gb[c] = t;
  }
}

// BF16 operand tiles from the FP32 master weights w[co][ci][K][K]:
//   wf[t][co][ci] (forward, co padded to cout_mma rows, ci to 32),
//   wb[t][ci][co] = w[co][ci][T - 1 - t] (backward data: flipped taps, 32 x 32).
__global__ void k_prep_weights(const float* __restrict__ w, int cout, int cin, int T,
                               int cout_mma, __nv_bfloat16* __restrict__ wf,
                               __nv_bfloat16* __restrict__ wb) {
  const size_t nf = (size_t)T * cout_mma * kC, nb = (size_t)T * kC * kC;
  for (size_t e = blockIdx.x * (size_t)blockDim.x + threadIdx.x; e < nf + nb;
       e += (size_t)gridDim.x * blockDim.x) {
    if (e < nf) {
      const int ci = (int)(e % kC);
      const int co = (int)((e / kC) % cout_mma);
      const int t = (int)(e / ((size_t)kC * cout_mma));
      const float v = (co < cout && ci < cin) ? w[((size_t)co * cin + ci) * T + t] : 0.f;
      if (wf) wf[e] = __float2bfloat16_rn(v);
    } else {
      const size_t f = e - nf;
      const int co = (int)(f % kC);
      const int ci = (int)((f / kC) % kC);
      const int t = (int)(f / ((size_t)kC * kC));
      const float v = (co < cout && ci < cin) ? w[((size_t)co * cin + ci) * T + (T - 1 - t)] : 0.f;
      if (wb) wb[f] = __float2bfloat16_rn(v);
    }
  }
}

// Network input, NHWC32 BF16: channel 0 = log10(g) + 5 (log-uniform [1e-6, 1e-4] S maps to
// [-1, 1]), 1 = V_in[i] / vscale along row i, 2 = V_lin,t / vscale, 3 = V_lin,b * bscale /
// vscale, the rest zero.  Vector b uses map map_index[b] (NULL: map 0).
__global__ void k_features(const double* __restrict__ gmaps, const int* __restrict__ map_index,
                           const double* __restrict__ vin, const double* __restrict__ vlt,
                           const double* __restrict__ vlb, int m, int n, float vscale,
                           float bscale, __nv_bfloat16* __restrict__ x) {
  const int b = blockIdx.y;
  const size_t mn = (size_t)m * n;
  const double* g = gmaps + (map_index ? (size_t)map_index[b] : 0) * mn;
  const double* lt = vlt + (size_t)b * mn;
  const double* lb = vlb + (size_t)b * mn;
  for (size_t c = blockIdx.x * (size_t)blockDim.x + threadIdx.x; c < mn;
       c += (size_t)gridDim.x * blockDim.x) {
    const int i = (int)(c / n);
    float f[kC] = {};
    f[0] = (float)(log10(g[c]) + 5.0);
    f[1] = (float)(vin[(size_t)b * m + i] / vscale);
    f[2] = (float)(lt[c] / vscale);
    f[3] = (float)(lb[c] * bscale / vscale);
    uint4 pk[4];
    uint32_t* w32 = reinterpret_cast<uint32_t*>(pk);
#pragma unroll
    for (int q = 0; q < 16; ++q) {
      const __nv_bfloat162 b2 = __floats2bfloat162_rn(f[2 * q], f[2 * q + 1]);
      w32[q] = *reinterpret_cast<const uint32_t*>(&b2);
    }
    uint4* dst = reinterpret_cast<uint4*>(x + ((size_t)b * mn + c) * kC);
#pragma unroll
    for (int q = 0; q < 4; ++q) dst[q] = pk[q];
  }
}

// target[p][0..1] = (V* - V_lin) * (dscale_t, dscale_b) per node (FP32); the voltages of
// each layer are [nvec][m*n] arrays
__global__ void k_target(const double* __restrict__ st, const double* __restrict__ sb,
                         const double* __restrict__ lt, const double* __restrict__ lb, int mn,
                         float dst_t, float dst_b, float* __restrict__ target) {
  const size_t o0 = (size_t)blockIdx.y * mn;
  float* o = target + 2 * o0;
  for (int c = blockIdx.x * blockDim.x + threadIdx.x; c < mn; c += gridDim.x * blockDim.x) {
    o[2 * c] = (float)((st[o0 + c] - lt[o0 + c]) * dst_t);
    o[2 * c + 1] = (float)((sb[o0 + c] - lb[o0 + c]) * dst_b);
  }
}

// guess = V_lin + pred / dscale as an FP64 state [V_t ; V_b] (pred NULL: V_lin itself)
__global__ void k_guess(const float* __restrict__ pred, const double* __restrict__ lt,
                        const double* __restrict__ lb, int mn, float dst_t, float dst_b,
                        double* __restrict__ guess) {
  const size_t o0 = (size_t)blockIdx.y * mn;
  const float* p = pred ? pred + 2 * o0 : nullptr;
  double* o = guess + 2 * o0;
  for (int c = blockIdx.x * blockDim.x + threadIdx.x; c < mn; c += gridDim.x * blockDim.x) {
    o[c] = lt[o0 + c] + (p ? (double)p[2 * c] / dst_t : 0.0);
    o[mn + c] = lb[o0 + c] + (p ? (double)p[2 * c + 1] / dst_b : 0.0);
  }
}

// Mean squared error over npix pixels x 2 channels and its gradient gz = 2 (p - t) / count
// as NHWC32 BF16 (channels 2..31 zero); loss_part[block] partial sums.
__global__ void k_loss(const float* __restrict__ pred, const float* __restrict__ tgt, size_t npix,
                       __nv_bfloat16* __restrict__ gz, float* __restrict__ loss_part) {
  float s = 0.f;
  const float sc = 2.0f / (float)(2 * npix);
  for (size_t p = blockIdx.x * (size_t)blockDim.x + threadIdx.x; p < npix;
       p += (size_t)gridDim.x * blockDim.x) {
    const float r0 = pred[2 * p] - tgt[2 * p], r1 = pred[2 * p + 1] - tgt[2 * p + 1];
    s = fmaf(r0, r0, fmaf(r1, r1, s));
    if (gz) {
      uint4 pk[4] = {};
      const __nv_bfloat162 b2 = __floats2bfloat162_rn(sc * r0, sc * r1);
      pk[0].x = *reinterpret_cast<const uint32_t*>(&b2);
      uint4* dst = reinterpret_cast<uint4*>(gz + p * kC);
#pragma unroll
      for (int q = 0; q < 4; ++q) dst[q] = pk[q];
    }
  }
  __shared__ float red[8];
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = s;
  __syncthreads();
  if (threadIdx.x == 0) {
    float t = 0.f;
    for (int w = 0; w < (int)(blockDim.x >> 5); ++w) t += red[w];
    loss_part[blockIdx.x] = t;
  }
}

__global__ void k_loss_finish(const float* __restrict__ part, int nb, size_t count,
                              float* __restrict__ loss) {
  if (threadIdx.x == 0 && blockIdx.x == 0) {
    double s = 0.0;
    for (int b = 0; b < nb; ++b) s += part[b];
    *loss = (float)(s / (double)count);
  }
}

// Adam on the FP32 master weights (Kingma & Ba, bias-corrected).
__global__ void k_adam(float* __restrict__ w, const float* __restrict__ g, float* __restrict__ m1,
                       float* __restrict__ m2, size_t count, float lr, float b1, float b2,
                       float eps, float bc1, float bc2) {
  for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < count;
       i += (size_t)gridDim.x * blockDim.x) {
    const float gi = g[i];
    const float a = b1 * m1[i] + (1.f - b1) * gi;
    const float b = b2 * m2[i] + (1.f - b2) * gi * gi;
    m1[i] = a;
    m2[i] = b;
    w[i] -= lr * ((a / bc1) / (sqrtf(b / bc2) + eps));
  }
}

int grid1d(size_t count, int th) {
  size_t nb = (count + th - 1) / th;
  if (nb > 4096) nb = 4096;
  return nb < 1 ? 1 : (int)nb;
}

std::once_flag g_cfg_once;
cudaError_t g_cfg_err = cudaSuccess;

cudaError_t configure() {
  std::call_once(g_cfg_once, [] {
    cudaError_t e = cudaFuncSetAttribute(k_conv_tc<32>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         227 * 1024);
    if (e == cudaSuccess)
      e = cudaFuncSetAttribute(k_conv_tc<16>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                               227 * 1024);
    if (e == cudaSuccess)
      e = cudaFuncSetAttribute(k_conv_taps, cudaFuncAttributeMaxDynamicSharedMemorySize,
                               227 * 1024);
    if (e == cudaSuccess)
      e = cudaFuncSetAttribute(k_wgrad_rows, cudaFuncAttributeMaxDynamicSharedMemorySize,
                               227 * 1024);
    if (e == cudaSuccess)
      e = cudaFuncSetAttribute(k_conv_wgrad_tc, cudaFuncAttributeMaxDynamicSharedMemorySize,
                               WgLayout::SMEM);
    g_cfg_err = e;
  });
  return g_cfg_err;
}

cudaError_t sm_count(int* sms) {
  int dev = 0;
  const cudaError_t e = cudaGetDevice(&dev);
  return e != cudaSuccess ? e
                          : cudaDeviceGetAttribute(sms, cudaDevAttrMultiProcessorCount, dev);
}

int launch_status(const char* what) {
  const cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) {
    set_last_cuda_error(e, what, __FILE__, __LINE__);
    return MCA_ERR_CUDA;
  }
  return MCA_OK;
}

bool shape_ok(int n, int h, int w, int k, int d) {
  return n >= 1 && h >= 1 && w >= 1 && k >= 1 && k <= kMaxK && (k & 1) && d >= 1 &&
         (size_t)n * h * w < (1ull << 31) && (size_t)h * w * kC * 2 < (1ull << 40);
}

}  // namespace

}  // namespace mca

using namespace mca;

extern "C" {

int mca_cnn_conv(const uint16_t* x, int32_t n, int32_t h, int32_t w, const uint16_t* wt,
                 int32_t ksize, int32_t dilation, int32_t cout_mma, int32_t cout,
                 const float* bias, int32_t act, int32_t backward, const uint16_t* y_prev,
                 uint16_t* out, float* out32, void* stream) {
  clear_error_message();
  if (!x || !wt || !shape_ok(n, h, w, ksize, dilation) || (cout_mma != 16 && cout_mma != 32) ||
      cout < 1 || cout > cout_mma || (!out && !out32) || (backward && cout_mma != 32)) {
    set_error_message("mca_cnn_conv: bad arguments");
    return MCA_ERR_INVALID_ARG;
  }
  if (cudaError_t e = configure(); e != cudaSuccess) {
    set_last_cuda_error(e, "mca_cnn_conv configure", __FILE__, __LINE__);
    return MCA_ERR_CUDA;
  }
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  // what k_conv_tc's stages hold is what a layer may ask for, whichever form runs: a row segment
  // takes 64 bytes per pixel, 128 + (K - 1) d of them (compared in 64 bits: the plan's own
  // arithmetic has 32)
  const bool fits = (int64_t)(ksize - 1) * dilation <= 227 * 1024 / 64;
  const ConvPlan plan = !fits ? ConvPlan{} : (cout_mma == 32) ? conv_plan<32>(ksize, dilation)
                                                              : conv_plan<16>(ksize, dilation);
  if (plan.stages < 2 || plan.smem > 227 * 1024) {
    set_error_message("mca_cnn_conv: kernel size and dilation too large for one row segment");
    return MCA_ERR_INVALID_ARG;
  }
  int sms = 0;
  if (const cudaError_t e = sm_count(&sms); e != cudaSuccess) {
    set_last_cuda_error(e, "mca_cnn_conv device", __FILE__, __LINE__);
    return MCA_ERR_CUDA;
  }
  TapPlan tp{};
  if (cout_mma == 32 && tap_plan(ksize, dilation, w, tp) &&
      taps_faster(tp, n, h, w, ksize, dilation, sms)) {
    CUtensorMap tmW;
    if ((reinterpret_cast<uintptr_t>(x) & 15) != 0 ||
        !tc::make_map_taps(&tmW, wt, ksize, kC, kTapM)) {
      set_error_message("mca_cnn_conv: tensor map encoding failed");
      return MCA_ERR_UNSUPPORTED;
    }
    TapArgs a{};
    a.H = h; a.W = w; a.K = ksize; a.d = dilation; a.r = (ksize - 1) / 2;
    a.xt = (w + tp.P - 1) / tp.P;
    a.cout = cout; a.bias = bias; a.act = act; a.backward = backward;
    a.yprev = reinterpret_cast<const __nv_bfloat16*>(y_prev);
    a.out = reinterpret_cast<__nv_bfloat16*>(out);
    a.out32 = out32;
    a.x = reinterpret_cast<const __nv_bfloat16*>(x);
    a.w = reinterpret_cast<const __nv_bfloat16*>(wt);
    a.plan = tp;
    a.tiles = n * h * a.xt;            // (n h w < 2^31)
    k_conv_taps<<<a.tiles < sms ? a.tiles : sms, kTapThreads, tp.smem, s>>>(tmW, a);
    count_launches(1);
    return launch_status("mca_cnn_conv launch");
  }
  CUtensorMap tmX, tmW;
  if (!tc::make_map_nhwc32_k8(&tmX, x, w, h, n, plan.wbox) ||
      !tc::make_map(&tmW, wt, (uint64_t)ksize * ksize * cout_mma, kC, plan.wrows, kC)) {
    set_error_message("mca_cnn_conv: tensor map encoding failed");
    return MCA_ERR_UNSUPPORTED;
  }
  ConvArgs a{};
  a.plan = plan;
  a.N = n; a.H = h; a.W = w; a.K = ksize; a.d = dilation; a.r = (ksize - 1) / 2;
  a.cout = cout; a.bias = bias; a.act = act; a.backward = backward;
  a.yprev = reinterpret_cast<const __nv_bfloat16*>(y_prev);
  a.out = reinterpret_cast<__nv_bfloat16*>(out);
  a.out32 = out32;
  dim3 grid((w + kPix - 1) / kPix, h, n);
  if (cout_mma == 32)
    k_conv_tc<32><<<grid, 128, plan.smem, s>>>(tmX, tmW, a);
  else
    k_conv_tc<16><<<grid, 128, plan.smem, s>>>(tmX, tmW, a);
  count_launches(1);
  return launch_status("mca_cnn_conv launch");
}

int64_t mca_cnn_wgrad_scratch(int32_t n, int32_t h, int32_t w, int32_t ksize) {
  if (!shape_ok(n, h, w, ksize, 1)) return -1;
  const int64_t nchunk = ((int64_t)n * h + kWgRows - 1) / kWgRows;
  const int64_t nbias = grid1d((size_t)n * h * w, 256);
  return nchunk * ksize * ksize * kC * kC + nbias * kC;
}

int mca_cnn_conv_wgrad(const uint16_t* x, const uint16_t* gz, int32_t n, int32_t h, int32_t w,
                       int32_t ksize, int32_t dilation, int32_t cin, int32_t cout,
                       float* scratch, float* gw, float* gb, void* stream) {
  clear_error_message();
  if (!x || !gz || !scratch || !gw || !shape_ok(n, h, w, ksize, dilation) || cin < 1 ||
      cin > kC || cout < 1 || cout > kC) {
    set_error_message("mca_cnn_conv_wgrad: bad arguments");
    return MCA_ERR_INVALID_ARG;
  }
  if (cudaError_t e = configure(); e != cudaSuccess) {
    set_last_cuda_error(e, "mca_cnn_conv_wgrad configure", __FILE__, __LINE__);
    return MCA_ERR_CUDA;
  }
  CUtensorMap tmX, tmG;
  if (!tc::make_map_nhwc32(&tmX, x, w, h, n, kWgPix) ||
      !tc::make_map_nhwc32(&tmG, gz, w, h, n, kWgPix)) {
    set_error_message("mca_cnn_conv_wgrad: tensor map encoding failed");
    return MCA_ERR_UNSUPPORTED;
  }
  const int T = ksize * ksize;
  // beyond the image's sizes every dilation is the same (only the centre tap sees pixels); the
  // bound keeps the shifts within 32 bits
  const int d = std::min(dilation, std::max(h, w));
  // partial sums: the scratch holds one set per kWgRows image rows
  const int nmax = (int)(((int64_t)n * h + kWgRows - 1) / kWgRows);
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  int sms = 0;
  if (const cudaError_t e = sm_count(&sms); e != cudaSuccess) {
    set_last_cuda_error(e, "mca_cnn_conv_wgrad device", __FILE__, __LINE__);
    return MCA_ERR_CUDA;
  }
  const WrPlan rp = wgrad_rows_plan(n, h, w, ksize, d, nmax, sms);
  int nchunk;
  if (ksize >= 5 && ksize <= kWrMaxK && wgrad_rows_faster(rp, n, h, w, ksize, nmax, sms)) {
    WrArgs a{};
    a.H = h; a.K = ksize; a.d = d; a.r = (ksize - 1) / 2;
    a.blocks = rp.blocks;
    a.nxc = rp.nxc;
    a.items = rp.items;
    a.part = scratch;
    nchunk = rp.chunks;
    const int stage = (ksize + 2 * kWrJ - 1) * kWrRow;
    a.stages = kWrStages * stage <= 224 * 1024 ? kWrStages : 2;
    const int smem = a.stages * stage + 512 + 1024;
    k_wgrad_rows<<<dim3(ksize, nchunk), 128, smem, s>>>(tmX, tmG, a);
  } else {
    WgArgs a{};
    a.N = n; a.H = h; a.W = w; a.K = ksize; a.d = d; a.r = (ksize - 1) / 2;
    a.rows_total = n * h;
    a.nxc = (w + kWgPix - 1) / kWgPix;
    a.part = scratch;
    nchunk = nmax;
    dim3 grid((T + kWgTaps - 1) / kWgTaps, nchunk);
    k_conv_wgrad_tc<<<grid, 128, WgLayout::SMEM, s>>>(tmX, tmG, a);
  }
  k_wgrad_reduce<<<grid1d((size_t)T * cin * cout, 256), 256, 0, s>>>(scratch, nchunk, T, cin,
                                                                      cout, gw);
  count_launches(2);
  if (gb) {
    const size_t npix = (size_t)n * h * w;
    const int nb = std::min(grid1d(npix, 256), 8 * 152);
    float* pb = scratch + (size_t)nmax * T * kC * kC;
    k_bias_grad_part<<<nb, 256, 0, s>>>(reinterpret_cast<const __nv_bfloat16*>(gz), npix, cout, pb);
    k_bias_grad_finish<<<1, 1024, 0, s>>>(pb, nb, cout, gb);
    count_launches(2);
  }
  return launch_status("mca_cnn_conv_wgrad launch");
}

int mca_cnn_prep_weights(const float* w, int32_t cout, int32_t cin, int32_t ksize,
                         int32_t cout_mma, uint16_t* wf, uint16_t* wb, void* stream) {
  clear_error_message();
  if (!w || (!wf && !wb) || cout < 1 || cout > cout_mma || (cout_mma != 16 && cout_mma != 32) ||
      cin < 1 || cin > kC || ksize < 1 || ksize > kMaxK || !(ksize & 1)) {
    set_error_message("mca_cnn_prep_weights: bad arguments");
    return MCA_ERR_INVALID_ARG;
  }
  const int T = ksize * ksize;
  const size_t count = (size_t)T * cout_mma * kC + (size_t)T * kC * kC;
  k_prep_weights<<<grid1d(count, 256), 256, 0, static_cast<cudaStream_t>(stream)>>>(
      w, cout, cin, T, cout_mma, reinterpret_cast<__nv_bfloat16*>(wf),
      reinterpret_cast<__nv_bfloat16*>(wb));
  count_launches(1);
  return launch_status("mca_cnn_prep_weights launch");
}

int mca_cnn_features(const double* gmaps, const int32_t* map_index, const double* v_in,
                     const double* vlin_t, const double* vlin_b, int32_t nvec, int32_t m,
                     int32_t n, float vscale, float bscale, uint16_t* x, void* stream) {
  clear_error_message();
  if (!gmaps || !v_in || !vlin_t || !vlin_b || !x || nvec < 1 || m < 1 || n < 1 ||
      !(vscale > 0.f) ||
      !(bscale > 0.f)) {
    set_error_message("mca_cnn_features: bad arguments");
    return MCA_ERR_INVALID_ARG;
  }
  k_features<<<dim3(grid1d((size_t)m * n, 256), nvec), 256, 0, static_cast<cudaStream_t>(stream)>>>(
      gmaps, map_index, v_in, vlin_t, vlin_b, m, n, vscale, bscale,
      reinterpret_cast<__nv_bfloat16*>(x));
  count_launches(1);
  return launch_status("mca_cnn_features launch");
}

int mca_cnn_target(const double* vstar_t, const double* vstar_b, const double* vlin_t,
                   const double* vlin_b, int32_t nvec, int32_t m, int32_t n, float dscale_t,
                   float dscale_b, float* target, void* stream) {
  clear_error_message();
  if (!vstar_t || !vstar_b || !vlin_t || !vlin_b || !target || nvec < 1 || m < 1 || n < 1 ||
      !(dscale_t > 0.f) ||
      !(dscale_b > 0.f)) {
    set_error_message("mca_cnn_target: bad arguments");
    return MCA_ERR_INVALID_ARG;
  }
  k_target<<<dim3(grid1d((size_t)m * n, 256), nvec), 256, 0, static_cast<cudaStream_t>(stream)>>>(
      vstar_t, vstar_b, vlin_t, vlin_b, m * n, dscale_t, dscale_b, target);
  count_launches(1);
  return launch_status("mca_cnn_target launch");
}

int mca_cnn_guess(const float* pred, const double* vlin_t, const double* vlin_b, int32_t nvec,
                  int32_t m, int32_t n, float dscale_t, float dscale_b, double* guess,
                  void* stream) {
  clear_error_message();
  if (!vlin_t || !vlin_b || !guess || nvec < 1 || m < 1 || n < 1 || !(dscale_t > 0.f) ||
      !(dscale_b > 0.f)) {
    set_error_message("mca_cnn_guess: bad arguments");
    return MCA_ERR_INVALID_ARG;
  }
  k_guess<<<dim3(grid1d((size_t)m * n, 256), nvec), 256, 0, static_cast<cudaStream_t>(stream)>>>(
      pred, vlin_t, vlin_b, m * n, dscale_t, dscale_b, guess);
  count_launches(1);
  return launch_status("mca_cnn_guess launch");
}

int mca_cnn_loss(const float* pred, const float* target, int64_t npix, uint16_t* gz,
                 float* part, float* loss, void* stream) {
  clear_error_message();
  if (!pred || !target || !part || !loss || npix < 1) {
    set_error_message("mca_cnn_loss: bad arguments");
    return MCA_ERR_INVALID_ARG;
  }
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  const int nb = 256;
  k_loss<<<nb, 256, 0, s>>>(pred, target, (size_t)npix, reinterpret_cast<__nv_bfloat16*>(gz),
                            part);
  k_loss_finish<<<1, 32, 0, s>>>(part, nb, (size_t)npix * 2, loss);
  count_launches(2);
  return launch_status("mca_cnn_loss launch");
}

int mca_cnn_adam(float* w, const float* g, float* m1, float* m2, int64_t count, float lr,
                 float beta1, float beta2, float eps, int32_t step, void* stream) {
  clear_error_message();
  if (!w || !g || !m1 || !m2 || count < 1 || step < 1) {
    set_error_message("mca_cnn_adam: bad arguments");
    return MCA_ERR_INVALID_ARG;
  }
  const float bc1 = 1.f - powf(beta1, (float)step), bc2 = 1.f - powf(beta2, (float)step);
  k_adam<<<grid1d((size_t)count, 256), 256, 0, static_cast<cudaStream_t>(stream)>>>(
      w, g, m1, m2, (size_t)count, lr, beta1, beta2, eps, bc1, bc2);
  count_launches(1);
  return launch_status("mca_cnn_adam launch");
}

int mca_cnn_check(void* stream) {
  clear_error_message();
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  int e = 0;
  const int zero = 0;
  cudaError_t ce = cudaMemcpyFromSymbolAsync(&e, g_cnn_err, sizeof(int), 0,
                                             cudaMemcpyDeviceToHost, s);
  if (ce == cudaSuccess) ce = cudaStreamSynchronize(s);
  if (ce == cudaSuccess && e != 0)
    ce = cudaMemcpyToSymbolAsync(g_cnn_err, &zero, sizeof(int), 0, cudaMemcpyHostToDevice, s);
  if (ce == cudaSuccess) ce = cudaStreamSynchronize(s);
  if (ce != cudaSuccess) {
    set_last_cuda_error(ce, "mca_cnn_check", __FILE__, __LINE__);
    return MCA_ERR_CUDA;
  }
  if (e != 0) {
    set_error_message("a bounded wait of a network kernel expired");
    return e;
  }
  return MCA_OK;
}

}  // extern "C"

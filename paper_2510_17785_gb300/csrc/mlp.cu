// Learned Chebyshev intervals: per-patch features, a 16 -> 64 -> 64 -> 2 MLP
// with BF16 inference and FP32 training, all on the GPU.
//
// The paper has no learned component; its smoother is damped Jacobi.  The
// Chebyshev variant needs, for every patch j and p-level q, an interval for the
// spectrum of D^-1 A_{j,q}.  A 16-step Lanczos run per (patch, level) gives it
// (k_lanczos); the MLP predicts (log theta_max, log theta_min) of that run from
// geometric and coefficient features at a tiny fraction of the cost, and
// Lanczos remains the reference the predictions are checked against (tests)
// and the fallback.
//
// Features of patch j at degree q, from its 2^d cells, with J_c the Jacobian
// of cell c at its centre, s_c its singular values, d_c = det J_c,
// r_c = min over the cell's vertices of det J / d_c, k_c = log kappa_c,
// t_c = k_c + log d_c - 2 log(mean s_c):
//    0 q/8   1 2^d/8   2 max k - min k   3 mean |k - mean k|
//    4/5/6 max/mean/min of log(s_max/s_min)   7 log(max d / min d)
//    8/9 min/mean r   10 max t - min t   11 mean |t - mean t|
//   12 log(max s_max / min s_min)   13 (q/8)^2   14 max |log d - mean log d|
//   15 (number of p-levels below q)/4
//
// Network (standardised inputs and targets): relu(W1 x + b1) -> relu(W2 h + b2)
// -> W3 h + b3.  Parameters: W1 (64x16, row-major), b1, W2 (64x64), b2,
// W3 (2x64), b3 = 5378 floats.  Normalisation: 36 floats, mean/std of the 16
// inputs then mean/std of the 2 targets.
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstdint>
#include <numeric>
#include <type_traits>
#include <random>
#include <vector>

#include "../../include/pmg.h"
#include "device_guard.h"
#include "mlp.h"

namespace pmg {
namespace {

constexpr int NF = 16, NH = 64, NO = 2;
constexpr int OW1 = 0, OB1 = OW1 + NH * NF, OW2 = OB1 + NH, OB2 = OW2 + NH * NH, OW3 = OB2 + NH, OB3 = OW3 + NO * NH;
constexpr int NP = OB3 + NO;
static_assert(NP == PMG_MLP_NPARAM, "parameter count");

int grid_for(size_t work, int threads) {
  size_t g = (work + threads - 1) / threads;
  if (g > 152 * 32) g = 152 * 32;
  return (int)std::max<size_t>(g, 1);
}

// ---------------------------------------------------------------- features
// singular values of a dim x dim matrix from the eigenvalues of J^T J
// (2x2: closed form; 3x3 symmetric: trigonometric solution of the cubic)
template <int DIM>
__device__ void singular_values(const double J[3][3], double* s) {
  double M[3][3];
  for (int i = 0; i < DIM; ++i)
    for (int j = 0; j < DIM; ++j) {
      double v = 0.0;
      for (int k = 0; k < DIM; ++k) v += J[k][i] * J[k][j];
      M[i][j] = v;
    }
  if (DIM == 2) {
    const double tr = M[0][0] + M[1][1], det = M[0][0] * M[1][1] - M[0][1] * M[1][0];
    const double disc = sqrt(fmax(0.25 * tr * tr - det, 0.0));
    s[0] = sqrt(fmax(0.5 * tr + disc, 0.0));
    s[1] = sqrt(fmax(0.5 * tr - disc, 0.0));
  } else {
    const double p1 = M[0][1] * M[0][1] + M[0][2] * M[0][2] + M[1][2] * M[1][2];
    const double q = (M[0][0] + M[1][1] + M[2][2]) / 3.0;
    double e0, e1, e2;
    if (p1 == 0.0) {
      e0 = M[0][0];
      e1 = M[1][1];
      e2 = M[2][2];
      const double mx = fmax(e0, fmax(e1, e2)), mn = fmin(e0, fmin(e1, e2));
      e1 = e0 + e1 + e2 - mx - mn;
      e0 = mx;
      e2 = mn;
    } else {
      const double p2 = (M[0][0] - q) * (M[0][0] - q) + (M[1][1] - q) * (M[1][1] - q) +
                        (M[2][2] - q) * (M[2][2] - q) + 2.0 * p1;
      const double p = sqrt(p2 / 6.0);
      double B[3][3];
      for (int i = 0; i < 3; ++i)
        for (int j = 0; j < 3; ++j) B[i][j] = (M[i][j] - (i == j ? q : 0.0)) / p;
      const double detB = B[0][0] * (B[1][1] * B[2][2] - B[1][2] * B[2][1]) -
                          B[0][1] * (B[1][0] * B[2][2] - B[1][2] * B[2][0]) +
                          B[0][2] * (B[1][0] * B[2][1] - B[1][1] * B[2][0]);
      const double r = fmin(fmax(detB / 2.0, -1.0), 1.0);
      const double phi = acos(r) / 3.0;
      const double pi = 3.14159265358979323846;
      e0 = q + 2.0 * p * cos(phi);
      e2 = q + 2.0 * p * cos(phi + 2.0 * pi / 3.0);
      e1 = 3.0 * q - e0 - e2;
    }
    s[0] = sqrt(fmax(e0, 0.0));
    s[1] = sqrt(fmax(e1, 0.0));
    s[2] = sqrt(fmax(e2, 0.0));
  }
}

template <int DIM>
__device__ void jac(const double* X, const double* xi, double J[3][3]) {
  for (int i = 0; i < DIM; ++i)
    for (int j = 0; j < DIM; ++j) J[i][j] = 0.0;
  for (int v = 0; v < (1 << DIM); ++v)
    for (int j = 0; j < DIM; ++j) {
      double f = 1.0;
      for (int k = 0; k < DIM; ++k) {
        const int bit = (v >> k) & 1;
        f *= (k == j) ? (bit ? 1.0 : -1.0) : (bit ? xi[k] : 1.0 - xi[k]);
      }
      for (int i = 0; i < DIM; ++i) J[i][j] += X[v * DIM + i] * f;
    }
}

template <int DIM>
__device__ double det3(const double J[3][3]) {
  return DIM == 3 ? J[0][0] * (J[1][1] * J[2][2] - J[1][2] * J[2][1]) -
                        J[0][1] * (J[1][0] * J[2][2] - J[1][2] * J[2][0]) +
                        J[0][2] * (J[1][0] * J[2][1] - J[1][1] * J[2][0])
                  : J[0][0] * J[1][1] - J[0][1] * J[1][0];
}

template <int DIM>
__global__ void k_features(const double* __restrict__ coords, const double* __restrict__ kappa, int N, int q,
                           int n_below, int npatch, float* __restrict__ Xout) {
  const int j = blockIdx.x * blockDim.x + threadIdx.x;
  if (j >= npatch) return;
  constexpr int NC = 1 << DIM;
  const int Nv = N - 1;
  int v[3] = {1, 1, 1};
  {
    int rem = j;
    for (int ax = 0; ax < DIM; ++ax) { v[ax] = 1 + rem % Nv; rem /= Nv; }
  }
  double an[NC], dd[NC], rr[NC], kk[NC], tt[NC], smax[NC], smin[NC];
  for (int c = 0; c < NC; ++c) {
    int cc[3] = {0, 0, 0};
    for (int ax = 0; ax < DIM; ++ax) cc[ax] = v[ax] - 1 + ((c >> ax) & 1);
    double X[8 * 3];
    int cell = 0, cm = 1;
    for (int ax = 0; ax < DIM; ++ax) { cell += cc[ax] * cm; cm *= N; }
    for (int w = 0; w < (1 << DIM); ++w) {
      size_t id = 0, mul = 1;
      for (int ax = 0; ax < DIM; ++ax) { id += (size_t)(cc[ax] + ((w >> ax) & 1)) * mul; mul *= (N + 1); }
      for (int i = 0; i < DIM; ++i) X[w * DIM + i] = coords[id * DIM + i];
    }
    double J[3][3], xi[3] = {0.5, 0.5, 0.5};
    jac<DIM>(X, xi, J);
    double s[3];
    singular_values<DIM>(J, s);
    const double d = det3<DIM>(J);
    double rmin = 1e300;
    for (int w = 0; w < (1 << DIM); ++w) {
      double xw[3];
      for (int k = 0; k < DIM; ++k) xw[k] = (w >> k) & 1;
      double Jw[3][3];
      jac<DIM>(X, xw, Jw);
      rmin = fmin(rmin, det3<DIM>(Jw) / d);
    }
    double smean = 0.0;
    for (int k = 0; k < DIM; ++k) smean += s[k];
    smean /= DIM;
    smax[c] = s[0];
    smin[c] = s[DIM - 1];
    an[c] = log(s[0] / s[DIM - 1]);
    dd[c] = d;
    rr[c] = rmin;
    kk[c] = log(kappa[cell]);
    tt[c] = kk[c] + log(d) - 2.0 * log(smean);
  }
  auto mx = [&](const double* a) { double r = a[0]; for (int c = 1; c < NC; ++c) r = fmax(r, a[c]); return r; };
  auto mn = [&](const double* a) { double r = a[0]; for (int c = 1; c < NC; ++c) r = fmin(r, a[c]); return r; };
  auto mean = [&](const double* a) { double r = 0.0; for (int c = 0; c < NC; ++c) r += a[c]; return r / NC; };
  auto mad = [&](const double* a) {
    const double m = mean(a);
    double r = 0.0;
    for (int c = 0; c < NC; ++c) r += fabs(a[c] - m);
    return r / NC;
  };
  double ld[NC];
  for (int c = 0; c < NC; ++c) ld[c] = log(dd[c]);
  double ldm = mean(ld), ldmax = 0.0;
  for (int c = 0; c < NC; ++c) ldmax = fmax(ldmax, fabs(ld[c] - ldm));
  float* o = Xout + (size_t)j * NF;
  o[0] = (float)(q / 8.0);
  o[1] = (float)(NC / 8.0);
  o[2] = (float)(mx(kk) - mn(kk));
  o[3] = (float)mad(kk);
  o[4] = (float)mx(an);
  o[5] = (float)mean(an);
  o[6] = (float)mn(an);
  o[7] = (float)log(mx(dd) / mn(dd));
  o[8] = (float)mn(rr);
  o[9] = (float)mean(rr);
  o[10] = (float)(mx(tt) - mn(tt));
  o[11] = (float)mad(tt);
  o[12] = (float)log(mx(smax) / mn(smin));
  o[13] = (float)((q / 8.0) * (q / 8.0));
  o[14] = (float)ldmax;
  o[15] = (float)(n_below / 4.0);
}

// ------------------------------------------------------------ inference
// FP32 inference: one thread per sample, parameters in shared memory
__global__ void k_mlp_infer(const float* __restrict__ params, const float* __restrict__ norm,
                            const float* __restrict__ X, int64_t n, float* __restrict__ Y) {
  using W = float;
  __shared__ W w[NP];
  __shared__ float nm[36];
  for (int i = threadIdx.x; i < NP; i += blockDim.x) w[i] = (W)params[i];
  for (int i = threadIdx.x; i < 36; i += blockDim.x) nm[i] = norm[i];
  __syncthreads();
  for (int64_t s = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; s < n; s += (int64_t)gridDim.x * blockDim.x) {
    float x[NF];
    for (int i = 0; i < NF; ++i) {
      x[i] = (X[s * NF + i] - nm[i]) / nm[NF + i];
    }
    float h1[NH];
    for (int r = 0; r < NH; ++r) {
      float a = (float)w[OB1 + r];
      for (int i = 0; i < NF; ++i) a += (float)w[OW1 + r * NF + i] * x[i];
      h1[r] = fmaxf(a, 0.f);
    }
    float y0 = (float)w[OB3], y1 = (float)w[OB3 + 1];
    for (int r = 0; r < NH; ++r) {
      float a = (float)w[OB2 + r];
      for (int i = 0; i < NH; ++i) a += (float)w[OW2 + r * NH + i] * h1[i];
      a = fmaxf(a, 0.f);
      y0 += (float)w[OW3 + r] * a;
      y1 += (float)w[OW3 + NH + r] * a;
    }
    // back to (log theta_max, log theta_min)
    Y[s * NO] = y0 * nm[2 * NF + 2] + nm[2 * NF];
    Y[s * NO + 1] = y1 * nm[2 * NF + 3] + nm[2 * NF + 1];
  }
}

// BF16 inference on the tensor cores: one warp per tile of 16 samples, the
// three layers as mma.sync m16n8k16 products with BF16 operands and FP32
// accumulation (16x16 inputs x 16x64 W1^T, 16x64 x 64x64 W2^T, 16x64 x 64x8
// W3^T with W3 padded to 8 rows).  Weights, biases, inputs and the two hidden
// activations are BF16 values; sums are FP32.  Fragment layouts (PTX ISA,
// m16n8k16 with .bf16): lane = 4 g + t; A holds rows g and g + 8, columns
// 2t, 2t+1, 2t+8, 2t+9 of the 16x16 tile; B holds rows (k) 2t, 2t+1, 2t+8,
// 2t+9 of column (n) g; C/D holds rows g, g + 8 and columns 2t, 2t+1.  The
// C tiles 2k and 2k+1 of one layer are exactly the A tile k of the next, so
// activations never leave the registers.
constexpr int MW1 = NF / 2 + 4;     // words per W1 row in shared memory (padded: conflict-free B loads)
constexpr int MW2 = NH / 2 + 4;     // words per W2 / W3 row
constexpr int MMA_THREADS = 128;

__device__ __forceinline__ unsigned pack_bf16(float lo, float hi) {
  const __nv_bfloat162 v = __floats2bfloat162_rn(lo, hi);    // lo in the low half
  unsigned u;
  memcpy(&u, &v, 4);
  return u;
}

__device__ __forceinline__ void mma_bf16(float (&d)[4], const unsigned (&a)[4], unsigned b0, unsigned b1) {
  asm volatile(
      "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, "
      "{%0,%1,%2,%3};"
      : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
      : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}

// C tiles (n-tiles 0..7 of a 16x64 layer output) + bias, ReLU, rounded to BF16
// -> the four A tiles of the next layer
__device__ __forceinline__ void act_to_a(float (&c)[8][4], const float* bias, int t, unsigned (&a)[4][4]) {
#pragma unroll
  for (int nt = 0; nt < 8; ++nt) {
    const float b0 = bias[nt * 8 + 2 * t], b1 = bias[nt * 8 + 2 * t + 1];
    c[nt][0] = fmaxf(c[nt][0] + b0, 0.f);
    c[nt][1] = fmaxf(c[nt][1] + b1, 0.f);
    c[nt][2] = fmaxf(c[nt][2] + b0, 0.f);
    c[nt][3] = fmaxf(c[nt][3] + b1, 0.f);
  }
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    a[k][0] = pack_bf16(c[2 * k][0], c[2 * k][1]);
    a[k][1] = pack_bf16(c[2 * k][2], c[2 * k][3]);
    a[k][2] = pack_bf16(c[2 * k + 1][0], c[2 * k + 1][1]);
    a[k][3] = pack_bf16(c[2 * k + 1][2], c[2 * k + 1][3]);
  }
}

__global__ void __launch_bounds__(MMA_THREADS) k_mlp_infer_mma(const float* __restrict__ params,
                                                               const float* __restrict__ norm,
                                                               const float* __restrict__ X, int64_t n,
                                                               float* __restrict__ Y) {
  __shared__ unsigned w1[NH * MW1], w2[NH * MW2], w3[8 * MW2];
  __shared__ float bs[2 * NH + NO], nm[36];
  for (int i = threadIdx.x; i < NH * NF / 2; i += blockDim.x) {
    const int r = i / (NF / 2), c = i - r * (NF / 2);
    w1[r * MW1 + c] = pack_bf16(params[OW1 + 2 * i], params[OW1 + 2 * i + 1]);
  }
  for (int i = threadIdx.x; i < NH * NH / 2; i += blockDim.x) {
    const int r = i / (NH / 2), c = i - r * (NH / 2);
    w2[r * MW2 + c] = pack_bf16(params[OW2 + 2 * i], params[OW2 + 2 * i + 1]);
  }
  for (int i = threadIdx.x; i < 8 * NH / 2; i += blockDim.x) {
    const int r = i / (NH / 2), c = i - r * (NH / 2);
    w3[r * MW2 + c] = r < NO ? pack_bf16(params[OW3 + 2 * i], params[OW3 + 2 * i + 1]) : 0u;
  }
  // biases as BF16 values (the weights' precision), kept in FP32 registers
  for (int i = threadIdx.x; i < NH; i += blockDim.x) {
    bs[i] = __bfloat162float(__float2bfloat16_rn(params[OB1 + i]));
    bs[NH + i] = __bfloat162float(__float2bfloat16_rn(params[OB2 + i]));
  }
  if (threadIdx.x < NO) bs[2 * NH + threadIdx.x] = __bfloat162float(__float2bfloat16_rn(params[OB3 + threadIdx.x]));
  for (int i = threadIdx.x; i < 36; i += blockDim.x) nm[i] = norm[i];
  __syncthreads();
  const int lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3;
  const int64_t ntile = (n + 15) / 16;
  const int64_t warps = (int64_t)gridDim.x * (MMA_THREADS / 32);
  for (int64_t tile = blockIdx.x * (int64_t)(MMA_THREADS / 32) + (threadIdx.x >> 5); tile < ntile; tile += warps) {
    const int64_t s0 = tile * 16 + g, s1 = s0 + 8;      // the two samples (rows) of this thread
    // layer-1 A tile: standardised inputs, rounded to BF16
    auto xin = [&](int64_t s, int c) { return s < n ? (X[s * NF + c] - nm[c]) / nm[NF + c] : 0.f; };
    unsigned a[4];
    a[0] = pack_bf16(xin(s0, 2 * t), xin(s0, 2 * t + 1));
    a[1] = pack_bf16(xin(s1, 2 * t), xin(s1, 2 * t + 1));
    a[2] = pack_bf16(xin(s0, 2 * t + 8), xin(s0, 2 * t + 9));
    a[3] = pack_bf16(xin(s1, 2 * t + 8), xin(s1, 2 * t + 9));
    float c[8][4];
#pragma unroll
    for (int nt = 0; nt < 8; ++nt) {
      c[nt][0] = c[nt][1] = c[nt][2] = c[nt][3] = 0.f;
      const unsigned* wr = w1 + (nt * 8 + g) * MW1;
      mma_bf16(c[nt], a, wr[t], wr[t + 4]);
    }
    unsigned h[4][4];
    act_to_a(c, bs, t, h);
#pragma unroll
    for (int nt = 0; nt < 8; ++nt) {
      c[nt][0] = c[nt][1] = c[nt][2] = c[nt][3] = 0.f;
      const unsigned* wr = w2 + (nt * 8 + g) * MW2;
#pragma unroll
      for (int k = 0; k < 4; ++k) mma_bf16(c[nt], h[k], wr[k * 8 + t], wr[k * 8 + t + 4]);
    }
    act_to_a(c, bs + NH, t, h);
    float y[4] = {0.f, 0.f, 0.f, 0.f};
    const unsigned* wr = w3 + g * MW2;
#pragma unroll
    for (int k = 0; k < 4; ++k) mma_bf16(y, h[k], wr[k * 8 + t], wr[k * 8 + t + 4]);
    // columns 0 and 1 of the output tile sit in lanes with t = 0
    if (t == 0) {
      const float b0 = bs[2 * NH], b1 = bs[2 * NH + 1];
      if (s0 < n) {
        Y[s0 * NO] = (y[0] + b0) * nm[2 * NF + 2] + nm[2 * NF];
        Y[s0 * NO + 1] = (y[1] + b1) * nm[2 * NF + 3] + nm[2 * NF + 1];
      }
      if (s1 < n) {
        Y[s1 * NO] = (y[2] + b0) * nm[2 * NF + 2] + nm[2 * NF];
        Y[s1 * NO + 1] = (y[3] + b1) * nm[2 * NF + 3] + nm[2 * NF + 1];
      }
    }
  }
}

// predicted logs -> Chebyshev interval [lo, hi]
template <typename T>
__global__ void k_bounds_from_logs(const float* __restrict__ Y, int64_t n, double safety, double ratio,
                                   T* __restrict__ bounds, double* __restrict__ bounds64) {
  for (int64_t s = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; s < n; s += (int64_t)gridDim.x * blockDim.x) {
    const double tmax = exp((double)Y[s * 2]), tmin = exp((double)Y[s * 2 + 1]);
    const double hi = safety * tmax;
    const double lo = fmax(tmin, hi / ratio);
    bounds[2 * s] = T(lo);
    bounds[2 * s + 1] = T(hi);
    bounds64[2 * s] = lo;
    bounds64[2 * s + 1] = hi;
  }
}

// ------------------------------------------------------------- training
// One training step is two launches: k_mlp_grad runs forward and backward of
// the whole network for tiles of TS samples with every weight and activation
// in shared memory, one partial gradient per CTA; k_mlp_reduce sums the
// partials and applies Adam (or stores the gradient).  The network is tiny
// (5,378 parameters), so a step is bound by launches and by the latency of
// loading the weights (21 KB from L2 per CTA), not by its products; TS = 8
// spreads a batch of 256 over 32 SMs.  One launch per product, bias, activation
// and column sum (20 a step, the loss read back after each) took 254 us a step
// at batch 256, these two 29 us (18 steps of 1,750 samples: 4.58 ms, 0.52 ms).
constexpr int TS = 8;                    // samples per tile
constexpr int GRAD_THREADS = 256;
constexpr int GRAD_CTAS = 304;           // two CTAs per SM; more tiles are looped over
constexpr int NPART = NP + 2;            // a partial: the gradient, then the loss, padded to even
constexpr int P1 = NF + 1, P2 = NH + 1;  // row pitches of the weights (lanes read one column of 32 rows)
static_assert(GRAD_THREADS == 4 * NH && NF == 16 && NO == 2, "thread layout of k_mlp_grad");

int grad_ctas(int64_t b) { return (int)std::min<int64_t>((b + TS - 1) / TS, GRAD_CTAS); }

// partial gradient and loss of batch rows perm[i] (i without perm), i < b
__global__ void __launch_bounds__(GRAD_THREADS) k_mlp_grad(const float* __restrict__ P, const float* __restrict__ norm,
                                                           const float* __restrict__ X, const float* __restrict__ T,
                                                           const int* __restrict__ perm, int b, float asym,
                                                           float* __restrict__ part) {
  __shared__ float w1[NH * P1], w2[NH * P2], w3[NO * NH], bias[2 * NH + NO], nm[2 * NF + 2 * NO];
  __shared__ __align__(16) float x[TS][NF], h1[TS][NH], h2[TS][NH], g2[TS][NH], g1[TS][NH];
  __shared__ float tgt[TS][NO], gy[TS][NO], ls[TS];
  const int tid = threadIdx.x;
  for (int i = tid; i < NH * NF; i += GRAD_THREADS) w1[(i / NF) * P1 + i % NF] = P[OW1 + i];
#pragma unroll
  for (int i = tid; i < NH * NH; i += GRAD_THREADS) w2[(i / NH) * P2 + i % NH] = P[OW2 + i];
  if (tid < NO * NH) w3[tid] = P[OW3 + tid];
  if (tid < NH) bias[tid] = P[OB1 + tid];
  else if (tid < 2 * NH) bias[tid] = P[OB2 + tid - NH];
  else if (tid < 2 * NH + NO) bias[tid] = P[OB3 + tid - 2 * NH];
  if (tid < 2 * NF + 2 * NO) nm[tid] = norm[tid];

  // this thread's gradient entries: a 4 x 4 block of W2, four of W1, one of W3
  // (tid < 128), one bias (tid < 130), the loss (tid = 130)
  float aw2[4][4] = {}, aw1[4] = {}, aw3 = 0.f, ab = 0.f;
  const int r4 = (tid / 16) * 4, c4 = (tid % 16) * 4;     // W2 block
  const int r1 = tid / 4, c1 = (tid % 4) * 4;             // W1 entries
  const int h = tid % NH, s0 = (tid / NH) * (TS / 4);     // activations: unit h of TS / 4 samples
  const int ntile = (b + TS - 1) / TS;
  for (int tile = blockIdx.x; tile < ntile; tile += gridDim.x) {
    // rows of the batch in this tile; the rows a last tile lacks have zero
    // inputs and zero activations, so that no product of theirs can be NaN
    const int rows = min(TS, b - tile * TS);
    __syncthreads();
    if (tid < TS * (NF + NO)) {
      const int s = tid / (NF + NO), f = tid % (NF + NO), i = tile * TS + s;
      float v = 0.f;
      if (s < rows) {
        const size_t src = perm ? (size_t)perm[i] : (size_t)i;
        v = f < NF ? (X[src * NF + f] - nm[f]) / nm[NF + f]
                   : (T[src * NO + f - NF] - nm[2 * NF + f - NF]) / nm[2 * NF + NO + f - NF];
      }
      if (f < NF) x[s][f] = v;
      else tgt[s][f - NF] = v;
    }
    __syncthreads();
    float z[TS / 4];
#pragma unroll
    for (int j = 0; j < TS / 4; ++j) z[j] = 0.f;
#pragma unroll
    for (int k = 0; k < NF; ++k) {
      const float w = w1[h * P1 + k];
#pragma unroll
      for (int j = 0; j < TS / 4; ++j) z[j] += w * x[s0 + j][k];
    }
#pragma unroll
    for (int j = 0; j < TS / 4; ++j) h1[s0 + j][h] = s0 + j < rows ? fmaxf(z[j] + bias[h], 0.f) : 0.f;
    __syncthreads();
#pragma unroll
    for (int j = 0; j < TS / 4; ++j) z[j] = 0.f;
#pragma unroll 16
    for (int k = 0; k < NH; ++k) {
      const float w = w2[h * P2 + k];
#pragma unroll
      for (int j = 0; j < TS / 4; ++j) z[j] += w * h1[s0 + j][k];
    }
#pragma unroll
    for (int j = 0; j < TS / 4; ++j) h2[s0 + j][h] = s0 + j < rows ? fmaxf(z[j] + bias[NH + h], 0.f) : 0.f;
    __syncthreads();
    // output layer: a warp per sample, both outputs; GY = w (y - t) / b
    {
      const int s = tid / 32, l = tid % 32;
      float y0 = w3[l] * h2[s][l] + w3[l + 32] * h2[s][l + 32];
      float y1 = w3[NH + l] * h2[s][l] + w3[NH + l + 32] * h2[s][l + 32];
#pragma unroll
      for (int m = 16; m > 0; m >>= 1) {
        y0 += __shfl_xor_sync(0xffffffffu, y0, m);
        y1 += __shfl_xor_sync(0xffffffffu, y1, m);
      }
      if (l == 0) {
        const bool live = s < rows;
        y0 += bias[2 * NH];
        y1 += bias[2 * NH + 1];
        const float d0 = y0 - tgt[s][0], d1 = y1 - tgt[s][1];
        const float wt = y0 < tgt[s][0] ? asym : 1.f;
        gy[s][0] = live ? wt * d0 / b : 0.f;
        gy[s][1] = live ? d1 / b : 0.f;
        ls[s] = live ? (0.5f * wt * d0 * d0 + 0.5f * d1 * d1) / b : 0.f;
      }
    }
    __syncthreads();
#pragma unroll
    for (int j = 0; j < TS / 4; ++j) {
      const int s = s0 + j;
      const float g = gy[s][0] * w3[h] + gy[s][1] * w3[NH + h];
      g2[s][h] = h2[s][h] > 0.f ? g : 0.f;
    }
    __syncthreads();
#pragma unroll
    for (int j = 0; j < TS / 4; ++j) z[j] = 0.f;
#pragma unroll 16
    for (int k = 0; k < NH; ++k) {
      const float w = w2[k * P2 + h];
#pragma unroll
      for (int j = 0; j < TS / 4; ++j) z[j] += w * g2[s0 + j][k];
    }
#pragma unroll
    for (int j = 0; j < TS / 4; ++j) g1[s0 + j][h] = h1[s0 + j][h] > 0.f ? z[j] : 0.f;
    __syncthreads();
#pragma unroll
    for (int s = 0; s < TS; ++s) {
      const float4 ga = *reinterpret_cast<const float4*>(&g2[s][r4]);
      const float4 ha = *reinterpret_cast<const float4*>(&h1[s][c4]);
      const float4 xa = *reinterpret_cast<const float4*>(&x[s][c1]);
      const float g[4] = {ga.x, ga.y, ga.z, ga.w}, hv[4] = {ha.x, ha.y, ha.z, ha.w};
#pragma unroll
      for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) aw2[i][j] += g[i] * hv[j];
      const float gg = g1[s][r1];
      aw1[0] += gg * xa.x;
      aw1[1] += gg * xa.y;
      aw1[2] += gg * xa.z;
      aw1[3] += gg * xa.w;
      if (tid < 2 * NH) {
        aw3 += gy[s][tid / NH] * h2[s][h];
        ab += tid < NH ? g1[s][h] : g2[s][h];
      } else if (tid < 2 * NH + NO) {
        ab += gy[s][tid - 2 * NH];
      } else if (tid == 2 * NH + NO) {
        ab += ls[s];
      }
    }
  }
  float* out = part + (size_t)blockIdx.x * NPART;
#pragma unroll
  for (int i = 0; i < 4; ++i)
#pragma unroll
    for (int j = 0; j < 4; ++j) out[OW2 + (r4 + i) * NH + c4 + j] = aw2[i][j];
#pragma unroll
  for (int j = 0; j < 4; ++j) out[OW1 + r1 * NF + c1 + j] = aw1[j];
  if (tid < NO * NH) out[OW3 + tid] = aw3;
  if (tid < NH) out[OB1 + tid] = ab;
  else if (tid < 2 * NH) out[OB2 + tid - NH] = ab;
  else if (tid < 2 * NH + NO) out[OB3 + tid - 2 * NH] = ab;
  else if (tid == 2 * NH + NO) out[NP] = ab;
}

struct AdamArgs {
  float *p, *m, *v;                      // p NULL: the gradient is stored instead
  float lr, b1, b2, eps, c1, c2;
};

// entry i of the gradient (i = NP: the loss): eight threads each sum every
// eighth partial, their sums are added in a fixed order
__global__ void __launch_bounds__(256) k_mlp_reduce(const float* __restrict__ part, int nparts, AdamArgs o,
                                                    float* __restrict__ grad, float* __restrict__ loss) {
  __shared__ float red[8][33];
  const int l = threadIdx.x % 32, w = threadIdx.x / 32, i = blockIdx.x * 32 + l;
  float s = 0.f;
  if (i <= NP) {
#pragma unroll 4
    for (int k = w; k < nparts; k += 8) s += part[(size_t)k * NPART + i];
  }
  red[w][l] = s;
  __syncthreads();
  if (w != 0 || i > NP) return;
  float gi = 0.f;
#pragma unroll
  for (int k = 0; k < 8; ++k) gi += red[k][l];
  if (i == NP) {
    if (loss) *loss = gi;
  } else if (!o.p) {
    grad[i] = gi;
  } else {
    const float mi = o.b1 * o.m[i] + (1.f - o.b1) * gi;
    const float vi = o.b2 * o.v[i] + (1.f - o.b2) * gi * gi;
    o.m[i] = mi;
    o.v[i] = vi;
    o.p[i] -= o.lr * (mi / o.c1) / (sqrtf(vi / o.c2) + o.eps);
  }
}

// the events of the copies out of two host buffers
struct CopyEvents {
  cudaEvent_t ev[2] = {nullptr, nullptr};
  cudaError_t err = cudaSuccess;
  CopyEvents() {
    for (cudaEvent_t& x : ev)
      if (err == cudaSuccess) err = cudaEventCreateWithFlags(&x, cudaEventDisableTiming);
  }
  ~CopyEvents() {
    for (cudaEvent_t x : ev)
      if (x) cudaEventDestroy(x);
  }
  CopyEvents(const CopyEvents&) = delete;
  CopyEvents& operator=(const CopyEvents&) = delete;
};

// loss and gradient (or Adam step) of the standardised batch rows perm[0..b);
// a launch that fails says so itself, whatever error is pending on the thread
cudaError_t grad_step(const float* P, const float* norm, const float* X, const float* T, const int* perm, int b, float asym,
               float* part, const AdamArgs& o, float* grad, float* loss, cudaStream_t s) {
  const int ctas = grad_ctas(b);
  cudaLaunchConfig_t cfg = {};
  cfg.stream = s;
  cfg.gridDim = dim3(ctas);
  cfg.blockDim = dim3(GRAD_THREADS);
  const cudaError_t e = cudaLaunchKernelEx(&cfg, k_mlp_grad, P, norm, X, T, perm, b, asym, part);
  if (e != cudaSuccess) return e;
  cfg.gridDim = dim3((NP + 1 + 31) / 32);
  cfg.blockDim = dim3(256);
  return cudaLaunchKernelEx(&cfg, k_mlp_reduce, (const float*)part, ctas, o, grad, loss);
}

}  // namespace

// -------------------------------------------------------------- host API
int features_launch(int dim, const double* coords, const double* kappa, int N, int q, int n_below, int npatch,
                    float* X, cudaStream_t s) {
  if (npatch <= 0) return PMG_OK;
  if (dim == 2) k_features<2><<<grid_for(npatch, 128), 128, 0, s>>>(coords, kappa, N, q, n_below, npatch, X);
  else k_features<3><<<grid_for(npatch, 128), 128, 0, s>>>(coords, kappa, N, q, n_below, npatch, X);
  return cudaPeekAtLastError() == cudaSuccess ? PMG_OK : PMG_ERR_CUDA;
}

int mlp_infer_launch(const float* params, const float* norm, const float* X, int64_t n, int bf16, float* Y,
                     cudaStream_t s) {
  if (n <= 0) return PMG_OK;
  if (bf16) {
    const size_t tiles = ((size_t)n + 15) / 16;
    k_mlp_infer_mma<<<grid_for(tiles, MMA_THREADS / 32), MMA_THREADS, 0, s>>>(params, norm, X, n, Y);
  } else {
    k_mlp_infer<<<grid_for((size_t)n, 128), 128, 0, s>>>(params, norm, X, n, Y);
  }
  return cudaPeekAtLastError() == cudaSuccess ? PMG_OK : PMG_ERR_CUDA;
}

int bounds_from_logs_launch(const float* Y, int64_t n, double safety, double ratio, float* b32, double* b64,
                            cudaStream_t s) {
  if (n <= 0) return PMG_OK;
  k_bounds_from_logs<float><<<grid_for((size_t)n, 256), 256, 0, s>>>(Y, n, safety, ratio, b32, b64);
  return cudaPeekAtLastError() == cudaSuccess ? PMG_OK : PMG_ERR_CUDA;
}

// ---- training targets and normalisation ------------------------------------
// T[i] = (log theta_max, log theta_min) of patch i from its Ritz pair
// (theta_min, theta_max)
__global__ void k_log_targets(const double* __restrict__ ritz, int64_t n, float* __restrict__ T) {
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
    T[2 * i] = (float)log(ritz[2 * i + 1]);
    T[2 * i + 1] = (float)log(ritz[2 * i]);
  }
}

// column c of an n x cols row-major matrix: out[c] = mean, out[cols + c] =
// population standard deviation + 1e-6 (two passes in FP64, one block per
// column, fixed reduction order: deterministic)
__global__ void __launch_bounds__(256) k_col_stats(const float* __restrict__ A, int64_t n, int cols,
                                                   float* __restrict__ out) {
  __shared__ double red[256];
  const int c = blockIdx.x;
  double s = 0.0;
  for (int64_t i = threadIdx.x; i < n; i += 256) s += (double)A[i * cols + c];
  red[threadIdx.x] = s;
  __syncthreads();
  for (int w = 128; w > 0; w >>= 1) {
    if (threadIdx.x < w) red[threadIdx.x] += red[threadIdx.x + w];
    __syncthreads();
  }
  const double mean = red[0] / (double)n;
  __syncthreads();
  double v = 0.0;
  for (int64_t i = threadIdx.x; i < n; i += 256) {
    const double d = (double)A[i * cols + c] - mean;
    v += d * d;
  }
  red[threadIdx.x] = v;
  __syncthreads();
  for (int w = 128; w > 0; w >>= 1) {
    if (threadIdx.x < w) red[threadIdx.x] += red[threadIdx.x + w];
    __syncthreads();
  }
  if (threadIdx.x == 0) {
    out[c] = (float)mean;
    out[cols + c] = (float)(sqrt(red[0] / (double)n) + 1e-6);
  }
}

int targets_launch(const double* ritz, int64_t n, float* T, cudaStream_t s) {
  if (n <= 0) return PMG_OK;
  k_log_targets<<<grid_for((size_t)n, 256), 256, 0, s>>>(ritz, n, T);
  return cudaPeekAtLastError() == cudaSuccess ? PMG_OK : PMG_ERR_CUDA;
}

}  // namespace pmg

using namespace pmg;

extern "C" {

void pmg_mlp_init(uint64_t seed, float* params) {
  if (!params) return;
  // SplitMix64 counter stream (Steele, Lea and Flood 2014): u_i in [0, 1)
  auto u01 = [seed](uint64_t i) {
    uint64_t z = seed + (i + 1) * 0x9E3779B97F4A7C15ull;
    z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
    z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
    z ^= z >> 31;
    return (double)(z >> 11) * 0x1.0p-53;
  };
  const int rows[3] = {NH, NH, NO}, cols[3] = {NF, NH, NH}, woff[3] = {OW1, OW2, OW3}, boff[3] = {OB1, OB2, OB3};
  uint64_t ctr = 0;
  for (int l = 0; l < 3; ++l) {
    const double lim = std::sqrt(6.0 / cols[l]);
    for (int i = 0; i < rows[l] * cols[l]; ++i) params[woff[l] + i] = (float)((2.0 * u01(ctr++) - 1.0) * lim);
    for (int i = 0; i < rows[l]; ++i) params[boff[l] + i] = 0.f;
  }
}

int pmg_mlp_norm(int device, const float* X, const float* T, int64_t n, float* norm_host) {
  if (!X || !T || !norm_host || n <= 0) return PMG_ERR_ARG;
  pmg::DeviceGuard guard(device);
  if (guard.err != cudaSuccess) return PMG_ERR_CUDA;
  float* out = nullptr;
  if (cudaMalloc(&out, PMG_MLP_NNORM * sizeof(float)) != cudaSuccess) return PMG_ERR_CUDA;
  k_col_stats<<<NF, 256>>>(X, n, NF, out);
  k_col_stats<<<NO, 256>>>(T, n, NO, out + 2 * NF);
  cudaError_t e = cudaMemcpy(norm_host, out, PMG_MLP_NNORM * sizeof(float), cudaMemcpyDeviceToHost);
  cudaFree(out);
  return e == cudaSuccess ? PMG_OK : PMG_ERR_CUDA;
}

void pmg_default_train_options(pmg_train_opts* o) {
  if (!o) return;
  o->epochs = 200;
  o->batch = 1024;
  o->lr = 2e-3f;
  o->beta1 = 0.9f;
  o->beta2 = 0.999f;
  o->eps = 1e-8f;
  o->asym = 4.0f;
  o->seed = 0;
}

int pmg_mlp_grad(int device, const float* params, const float* norm, const float* X, const float* T, int n,
                 float asym, float* loss, float* grad, void* stream) {
  if (!params || !norm || !X || !T || !grad || n <= 0) return PMG_ERR_ARG;
  pmg::DeviceGuard guard(device);
  if (guard.err != cudaSuccess) return PMG_ERR_CUDA;
  cudaStream_t s = (cudaStream_t)stream;
  float* part = nullptr;
  if (cudaMalloc(&part, (size_t)grad_ctas(n) * NPART * sizeof(float)) != cudaSuccess) return PMG_ERR_CUDA;
  cudaError_t e = grad_step(params, norm, X, T, nullptr, n, asym, part, AdamArgs{}, grad, loss, s);
  const cudaError_t se = cudaStreamSynchronize(s);
  if (e == cudaSuccess) e = se;
  cudaFree(part);
  return e == cudaSuccess ? PMG_OK : PMG_ERR_CUDA;
}

int pmg_mlp_train(int device, float* params, const float* norm, const float* X, const float* T, int64_t n,
                  const pmg_train_opts* opt_in, float* loss_hist) {
  pmg_train_opts o;
  if (opt_in) o = *opt_in;
  else pmg_default_train_options(&o);
  if (!params || !norm || !X || !T || n <= 0 || o.batch <= 0 || o.epochs < 0) return PMG_ERR_ARG;
  pmg::DeviceGuard guard(device);
  if (guard.err != cudaSuccess) return PMG_ERR_CUDA;
  cudaStream_t s = nullptr;
  const int b = (int)std::min<int64_t>(o.batch, n);
  const int64_t nb = n / b;
  // the losses of up to E epochs stay on the device: the steps of E epochs
  // are queued without waiting for one
  const int64_t E = std::min<int64_t>(std::max<int64_t>(o.epochs, 1), std::max<int64_t>(1, (1 << 16) / nb));
  // one allocation: moments, partial gradients, losses, batch order
  const size_t n_part = (size_t)grad_ctas(b) * NPART, n_loss = (size_t)(E * nb);
  float* base = nullptr;
  if (cudaMalloc(&base, (2 * NP + n_part + n_loss + (size_t)n) * sizeof(float)) != cudaSuccess) return PMG_ERR_CUDA;
  float *m = base, *v = m + NP, *part = v + NP, *loss = part + n_part;
  int* perm = reinterpret_cast<int*>(loss + n_loss);
  // Epochs alternate between two host buffers for their order: the copy of a
  // pageable buffer may read it after the call returned (this GPU's CPU shares
  // its page tables), so a buffer is drawn into again only after its copy's
  // event.  That is two epochs back: the steps of one stay queued meanwhile.
  std::vector<int> order[2] = {std::vector<int>(n), std::vector<int>(n)};
  std::iota(order[1].begin(), order[1].end(), 0);
  CopyEvents copied;
  std::mt19937_64 rng(o.seed);
  int64_t step = 0;
  std::vector<float> lh(n_loss);
  cudaError_t e = copied.err;
  if (e == cudaSuccess) e = cudaMemsetAsync(m, 0, 2 * NP * sizeof(float), s);
  for (int ep = 0; ep < o.epochs && e == cudaSuccess; ++ep) {
    std::vector<int>&cur = order[ep % 2], &prev = order[1 - ep % 2];
    if (ep >= 2) e = cudaEventSynchronize(copied.ev[ep % 2]);
    if (e != cudaSuccess) break;
    std::copy(prev.begin(), prev.end(), cur.begin());
    std::shuffle(cur.begin(), cur.end(), rng);
    e = cudaMemcpyAsync(perm, cur.data(), n * sizeof(int), cudaMemcpyHostToDevice, s);
    if (e == cudaSuccess) e = cudaEventRecord(copied.ev[ep % 2], s);
    if (e != cudaSuccess) break;
    const int64_t slot = ep % E;
    for (int64_t bi = 0; bi < nb && e == cudaSuccess; ++bi) {
      ++step;
      const float c1 = 1.f - std::pow(o.beta1, (float)step), c2 = 1.f - std::pow(o.beta2, (float)step);
      e = grad_step(params, norm, X, T, perm + bi * b, b, o.asym, part,
                    AdamArgs{params, m, v, o.lr, o.beta1, o.beta2, o.eps, c1, c2}, nullptr, loss + slot * nb + bi, s);
    }
    if (e != cudaSuccess) break;
    if (loss_hist && (slot == E - 1 || ep == o.epochs - 1)) {
      e = cudaMemcpyAsync(lh.data(), loss, (size_t)((slot + 1) * nb) * sizeof(float), cudaMemcpyDeviceToHost, s);
      if (e == cudaSuccess) e = cudaStreamSynchronize(s);
      if (e != cudaSuccess) break;
      for (int64_t k = 0; k <= slot; ++k) {
        double tot = 0.0;
        for (int64_t bi = 0; bi < nb; ++bi) tot += lh[k * nb + bi];
        loss_hist[ep - slot + k] = (float)(tot / nb);
      }
    }
  }
  const cudaError_t se = cudaStreamSynchronize(s);
  if (e == cudaSuccess) e = se;
  cudaFree(base);
  return e == cudaSuccess ? PMG_OK : PMG_ERR_CUDA;
}

int pmg_mlp_predict(int device, const float* params, const float* norm, const float* X, int64_t n, int bf16,
                    float* Y, void* stream) {
  if (!params || !norm || !X || !Y || n < 0) return PMG_ERR_ARG;
  pmg::DeviceGuard guard(device);
  if (guard.err != cudaSuccess) return PMG_ERR_CUDA;
  return mlp_infer_launch(params, norm, X, n, bf16, Y, (cudaStream_t)stream);
}

}  // extern "C"

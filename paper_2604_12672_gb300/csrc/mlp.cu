// mlp.cu -- the temperature-guess network: FP32 training kernels (forward,
// backward, weight-gradient reduction, Adam) on EOS samples generated on the
// device, and BF16 tensor-core inference (mlp_dev.cuh).
//
// Training data: (log10 rho, log10 T, X_0) drawn uniformly in the stated
// ranges by a counter-based generator (SplitMix64, Steele, Lea & Flood 2014),
// e_int from the device EOS (eos_rt), inputs (log10 rho, log10 e_int, X_0),
// target log10 T, all mapped affinely onto [-1, 1].  Loss: mean squared error
// of the mapped target.
#include <cuda_runtime.h>
#include <math.h>
#include <stddef.h>
#include <stdint.h>
#include <string.h>

#include <algorithm>
#include <chrono>
#include <vector>

#include "eos_stellar.cuh"
#include "mlp_dev.cuh"
#include "phl.h"
#include "phl_internal.cuh"

using namespace phl::mlp;

struct phl_mlp {
  float *w = nullptr;       // FP32 master weights (NPARAM), device
  float *m = nullptr, *v = nullptr;   // Adam moments
  float *grad = nullptr;    // NPARAM
  uint2 *frag = nullptr;    // BF16 fragments (F_TOTAL)
  float *bias = nullptr;    // b1, b2 copies for inference (2 NH)
  float b3 = 0.0f;
  float c[4] = {6.0f, 18.0f, 0.5f, 8.75f}, s[4] = {1.0f, 1.0f, 2.0f, 1.0f};
  long adam_t = 0;
  int sms = phl::sm_count();
};

namespace phl {
namespace {

__host__ __device__ __forceinline__ uint64_t splitmix64(uint64_t z) {
  z += 0x9E3779B97F4A7C15ull;
  z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
  z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
  return z ^ (z >> 31);
}
__device__ __forceinline__ double uniform01(uint64_t seed, uint64_t i, int comp) {
  const uint64_t z = splitmix64(seed ^ splitmix64(3 * i + comp));
  return (double)(z >> 11) * (1.0 / 9007199254740992.0);
}

// EOS samples: x[3 n] (raw log10 rho, log10 e, X_0), t[n] raw log10 T.
__global__ void k_samples(eos::Table tab, long n, uint64_t seed, double lr0, double lr1, double lt0, double lt1,
                          double A0, double Z0, double A1, double Z1, float *x, float *t, int *fail) {
  const long i = blockIdx.x * (long)blockDim.x + threadIdx.x;
  if (i >= n) return;
  const double lr = lr0 + (lr1 - lr0) * uniform01(seed, i, 0);
  const double lt = lt0 + (lt1 - lt0) * uniform01(seed, i, 1);
  const double X0 = uniform01(seed, i, 2);
  const double rho = pow(10.0, lr), T = pow(10.0, lt);
  const double sa = X0 / A0 + (1.0 - X0) / A1;
  const double abar = 1.0 / sa, ye = X0 * Z0 / A0 + (1.0 - X0) * Z1 / A1;
  eos::EosOut<double> o;
  if (!eos::eos_rt<double>(tab, rho, T, abar, ye, o) || !(o.e > 0.0)) {
    atomicOr(fail, 1);
    x[3 * i] = x[3 * i + 1] = x[3 * i + 2] = 0.0f;
    t[i] = 0.0f;
    return;
  }
  x[3 * i] = (float)lr;
  x[3 * i + 1] = (float)log10(o.e);
  x[3 * i + 2] = (float)X0;
  t[i] = (float)lt;
}

// Apply the affine maps in place: x <- (x - c) s, t <- (t - c3) s3.
__global__ void k_normalise(long n, float *x, float *t, float4 c, float4 s) {
  const long i = blockIdx.x * (long)blockDim.x + threadIdx.x;
  if (i >= n) return;
  x[3 * i] = (x[3 * i] - c.x) * s.x;
  x[3 * i + 1] = (x[3 * i + 1] - c.y) * s.y;
  x[3 * i + 2] = (x[3 * i + 2] - c.z) * s.z;
  t[i] = (t[i] - c.w) * s.w;
}

// min / max of column 1 (log10 e) over the samples (positive floats order like
// their bit patterns)
__global__ void k_minmax_e(long n, const float *x, unsigned int *mn, unsigned int *mx) {
  unsigned int lo = 0x7f7fffffu, hi = 0u;
  for (long i = blockIdx.x * (long)blockDim.x + threadIdx.x; i < n; i += (long)gridDim.x * blockDim.x) {
    const unsigned int b = __float_as_uint(x[3 * i + 1]);
    lo = min(lo, b);
    hi = max(hi, b);
  }
  atomicMin(mn, lo);
  atomicMax(mx, hi);
}

// Loss and weight gradient in FP32 (weights in shared memory, rounded to BF16
// as in inference: straight-through gradient).  A block takes tiles of LG_S
// samples: first layer, second layer (64 x 64 times the tile), output and
// residual, the back-propagated errors (the transposed product) and the
// tile's weight gradient D2 H1^T, which stays in registers over the block's
// tiles and is added to grad at the end, once per block and entry (456 FP32
// additions at most; the loss goes to an FP64 sum tile by tile).
// Bound by FP32 issue: 12288 multiply-adds per sample in the three products.
// Each thread forms 8 x 4 (4 x 8 in the last) of a product from 16-byte
// shared-memory reads, 10.7 multiply-adds per read; one sample per thread had
// one read per four, and the activations and errors made a round trip of
// 1 KB per sample through memory to a second kernel.  65536 samples:
// 57 us instead of 84 + 53 (68 with the bias sums added once per warp).  The rows a thread takes are spread so that the
// eight lanes of a read phase fall into different banks (row stride 68).
constexpr int LG_T = 128, LG_S = 64, LG_LD = 68;
struct LossGradSmem {
  float w2[NH][LG_LD];   // W2[a][b]
  float h1[NH][LG_LD];   // h1[b][s]
  float d2[NH][LG_LD];   // d2[a][s]
  float w1[NH * NIN], b1[NH], b2[NH], w3[NH], b3;
  alignas(16) float x[NIN][LG_S];
  float t[LG_S];
  float row[LG_T / 32][6][NH];   // per warp: sums over the samples of d2, dy h2, d1, d1 x
  float gb3[LG_T / 32];          // and of dy
};
static_assert(offsetof(LossGradSmem, w2) % 16 == 0 && offsetof(LossGradSmem, h1) % 16 == 0 &&
                  offsetof(LossGradSmem, d2) % 16 == 0 && offsetof(LossGradSmem, x) % 16 == 0 && LG_LD % 4 == 0 &&
                  LG_S % 4 == 0,
              "rows read by float4");
constexpr size_t LG_SMEM = sizeof(LossGradSmem);

__device__ __forceinline__ float4 ld4(const float *p) { return *reinterpret_cast<const float4 *>(p); }
__device__ __forceinline__ float elem(const float4 &v, int i) { return i == 0 ? v.x : (i == 1 ? v.y : (i == 2 ? v.z : v.w)); }

__global__ void __launch_bounds__(LG_T, 3) k_loss_grad(const float *__restrict__ w, long nb,
                                                       const float *__restrict__ x, const float *__restrict__ t,
                                                       float inv_n, float *__restrict__ grad, double *loss) {
  extern __shared__ __align__(16) unsigned char lg_raw[];
  LossGradSmem &sm = *reinterpret_cast<LossGradSmem *>(lg_raw);
  const int tid = threadIdx.x, lane = tid & 31;
  // the weight matrices as the inference sees them, the biases in FP32; the
  // gradient updates the FP32 master weights
  auto bf = [](float v) { return __bfloat162float(__float2bfloat16_rn(v)); };
  for (int k = tid; k < NH * NH; k += LG_T) sm.w2[k / NH][k % NH] = bf(w[O_W2 + k]);
  for (int k = tid; k < NH * NIN; k += LG_T) sm.w1[k] = bf(w[O_W1 + k]);
  if (tid < NH) {
    sm.b1[tid] = w[O_B1 + tid];
    sm.b2[tid] = w[O_B2 + tid];
    sm.w3[tid] = bf(w[O_W3 + tid]);
  }
  if (tid == 0) sm.b3 = w[O_B3];
  const int rg = tid & 7, s4 = 4 * (tid >> 3);       // products 1, 2: row group, first of four samples
  const int gb = tid & 7, ga = tid >> 3;             // product 3: columns gb + 8 j, rows ga + 16 i
  float gw[4][8] = {}, gb3 = 0.0f;
  double r2 = 0.0;   // squared residuals: a tile's 16 of a warp in FP32, the tiles in FP64
  // per-row sums: over the warp's four sample groups, then into the warp's own
  // row of shared memory (48 registers less than keeping them per thread)
  float (*row)[NH] = sm.row[tid >> 5];
  for (int k = lane; k < 6 * NH; k += 32) (&row[0][0])[k] = 0.0f;
  __syncwarp();
  auto rows = [&](float v) {
    v += __shfl_xor_sync(0xffffffffu, v, 8);
    return v + __shfl_xor_sync(0xffffffffu, v, 16);
  };
  auto add_row = [&](float *dst, float v) {
    v = rows(v);
    if (lane < 8) *dst += v;
  };
  for (long s0 = (long)blockIdx.x * LG_S; s0 < nb; s0 += (long)gridDim.x * LG_S) {
    const int cnt = (int)min((long)LG_S, nb - s0);
    __syncthreads();   // the previous tile's readers are done
    for (int e = tid; e < NIN * LG_S; e += LG_T) sm.x[e % NIN][e / NIN] = e < NIN * cnt ? x[NIN * s0 + e] : 0.0f;
    if (tid < LG_S) sm.t[tid] = tid < cnt ? t[s0 + tid] : 0.0f;
    __syncthreads();
    {
      const int ss = tid & (LG_S - 1), b0 = (tid / LG_S) * (NH / 2);
      const float x0 = sm.x[0][ss], x1 = sm.x[1][ss], x2 = sm.x[2][ss];
      for (int b = b0; b < b0 + NH / 2; ++b)
        sm.h1[b][ss] = tanhf(sm.b1[b] + sm.w1[3 * b] * x0 + sm.w1[3 * b + 1] * x1 + sm.w1[3 * b + 2] * x2);
    }
    __syncthreads();
    {   // z[a][s] = b2 + sum_b W2[a][b] h1[b][s], rows a = rg + 8 i
      float z[8][4];
#pragma unroll
      for (int i = 0; i < 8; ++i)
#pragma unroll
        for (int q = 0; q < 4; ++q) z[i][q] = sm.b2[rg + 8 * i];
#pragma unroll 4
      for (int k = 0; k < NH; k += 4) {
        float4 h[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) h[q] = ld4(&sm.h1[k + q][s4]);
#pragma unroll
        for (int i = 0; i < 8; ++i) {
          const float4 a = ld4(&sm.w2[rg + 8 * i][k]);
#pragma unroll
          for (int kk = 0; kk < 4; ++kk)
#pragma unroll
            for (int q = 0; q < 4; ++q) z[i][q] += elem(a, kk) * elem(h[kk], q);
        }
      }
      float y[4] = {0.0f, 0.0f, 0.0f, 0.0f};
#pragma unroll
      for (int i = 0; i < 8; ++i)
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          z[i][q] = tanhf(z[i][q]);
          y[q] += sm.w3[rg + 8 * i] * z[i][q];
        }
      float dy[4], t2 = 0.0f;
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        for (int o = 1; o < 8; o <<= 1) y[q] += __shfl_xor_sync(0xffffffffu, y[q], o);
        const float r = s4 + q < cnt ? sm.b3 + y[q] - sm.t[s4 + q] : 0.0f;   // no contribution beyond the batch
        dy[q] = 2.0f * r * inv_n;
        t2 += r * r;
        gb3 += dy[q];
      }
      t2 = rows(t2);
      if (lane == 0) r2 += (double)t2;
#pragma unroll
      for (int i = 0; i < 8; ++i) {
        const float w3 = sm.w3[rg + 8 * i];
        float d[4], gb2 = 0.0f, gw3 = 0.0f;
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          d[q] = dy[q] * w3 * (1.0f - z[i][q] * z[i][q]);
          gb2 += d[q];
          gw3 += dy[q] * z[i][q];
        }
        add_row(&row[0][rg + 8 * i], gb2);
        add_row(&row[1][rg + 8 * i], gw3);
        *reinterpret_cast<float4 *>(&sm.d2[rg + 8 * i][s4]) = make_float4(d[0], d[1], d[2], d[3]);
      }
    }
    __syncthreads();
    {   // d1[b][s] = (1 - h1^2) sum_a W2[a][b] d2[a][s], rows b = 4 rg + i and 32 + 4 rg + i
      float d1[8][4] = {};
#pragma unroll 16
      for (int k = 0; k < NH; ++k) {
        const float4 a0 = ld4(&sm.w2[k][4 * rg]), a1 = ld4(&sm.w2[k][32 + 4 * rg]), d = ld4(&sm.d2[k][s4]);
#pragma unroll
        for (int i = 0; i < 4; ++i)
#pragma unroll
          for (int q = 0; q < 4; ++q) {
            d1[i][q] += elem(a0, i) * elem(d, q);
            d1[4 + i][q] += elem(a1, i) * elem(d, q);
          }
      }
      float4 xs[NIN];
#pragma unroll
      for (int c = 0; c < NIN; ++c) xs[c] = ld4(&sm.x[c][s4]);
#pragma unroll
      for (int i = 0; i < 8; ++i) {
        const int b = (i < 4 ? 0 : 28) + 4 * rg + i;
        const float4 h = ld4(&sm.h1[b][s4]);
        float gb1 = 0.0f, gw1[NIN] = {};
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          const float v = d1[i][q] * (1.0f - elem(h, q) * elem(h, q));
          gb1 += v;
#pragma unroll
          for (int c = 0; c < NIN; ++c) gw1[c] += v * elem(xs[c], q);
        }
        add_row(&row[2][b], gb1);
#pragma unroll
        for (int c = 0; c < NIN; ++c) add_row(&row[3 + c][b], gw1[c]);
      }
    }
    // dW2[a][b] += sum_s d2[a][s] h1[b][s]
#pragma unroll 4
    for (int k = 0; k < LG_S; k += 4) {
      float4 d[4];
#pragma unroll
      for (int i = 0; i < 4; ++i) d[i] = ld4(&sm.d2[ga + 16 * i][k]);
#pragma unroll
      for (int j = 0; j < 8; ++j) {
        const float4 h = ld4(&sm.h1[gb + 8 * j][k]);
#pragma unroll
        for (int kk = 0; kk < 4; ++kk)
#pragma unroll
          for (int i = 0; i < 4; ++i) gw[i][j] += elem(d[i], kk) * elem(h, kk);
      }
    }
  }
#pragma unroll
  for (int i = 0; i < 4; ++i)
#pragma unroll
    for (int j = 0; j < 8; ++j) atomicAdd(&grad[O_W2 + (ga + 16 * i) * NH + gb + 8 * j], gw[i][j]);
  // one addition per block and entry: more partial sums mean more roundings
  // against the full one (a warp each: 1.5 times the error against 64 bits)
  gb3 = rows(gb3);
  if (lane == 0) {
    sm.gb3[tid >> 5] = gb3;
    atomicAdd(loss, r2);
  }
  __syncthreads();
  static_assert(LG_T == 128, "four warps' sums");
  for (int k = tid; k < 6 * NH; k += LG_T) {
    const int m = k / NH, a = k % NH;
    const int o = m == 0 ? O_B2 + a : (m == 1 ? O_W3 + a : (m == 2 ? O_B1 + a : O_W1 + 3 * a + m - 3));
    atomicAdd(&grad[o], (sm.row[0][m][a] + sm.row[1][m][a]) + (sm.row[2][m][a] + sm.row[3][m][a]));
  }
  if (tid == 0) atomicAdd(&grad[O_B3], (sm.gb3[0] + sm.gb3[1]) + (sm.gb3[2] + sm.gb3[3]));
}

__global__ void k_adam(int n, float *w, float *m, float *v, const float *g, float lr, float b1, float b2, float eps,
                       float c1, float c2) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const float gi = g[i];
  const float mi = b1 * m[i] + (1.0f - b1) * gi, vi = b2 * v[i] + (1.0f - b2) * gi * gi;
  m[i] = mi;
  v[i] = vi;
  w[i] -= lr * (mi / c1) / (sqrtf(vi / c2) + eps);
}

// BF16 tensor-core inference over n samples of normalised inputs (x[3 n]).
__global__ void k_infer(phl::mlp::Dev M, long n, const float *__restrict__ x, float *__restrict__ y) {
  const long i = blockIdx.x * (long)blockDim.x + threadIdx.x;
  const bool in = i < n;
  const float xin[3] = {in ? x[3 * i] : 0.f, in ? x[3 * i + 1] : 0.f, in ? x[3 * i + 2] : 0.f};
  const int lane = threadIdx.x & 31;
  const float ylo = tile_forward(M, xin, 0);
  const float yhi = tile_forward(M, xin, 16);
  if (in) y[i] = lane < 16 ? ylo : yhi;
}

// Temperature guesses for the batch EOS: T = 10^(network output).
__global__ void k_guess(phl::mlp::Dev M, long n, const double *rho, const double *eint, const double *X0,
                        double Tlo, double Thi, double *T) {
  const long i = blockIdx.x * (long)blockDim.x + threadIdx.x;
  const bool in = i < n;
  const float lr = in ? (float)log10(rho[i]) : M.c[0];
  const float le = in ? (float)log10(fmax(eint[i], 1e-300)) : M.c[1];
  const float xx = in ? (float)X0[i] : M.c[2];
  const float lt = guess_log10T(M, lr, le, xx);
  if (in) T[i] = fmin(fmax(exp10((double)lt), Tlo), Thi);
}

phl_status cuda_status(cudaError_t e, const char *what) {
  return (phl_status)set_error(PHL_ECUDA, "%s: %s", what, cudaGetErrorString(e));
}

// BF16 fragments and bias copies from the FP32 master weights.
cudaError_t build_fragments(phl_mlp *M) {
  std::vector<float> w(NPARAM);
  cudaError_t e = cudaMemcpy(w.data(), M->w, NPARAM * sizeof(float), cudaMemcpyDeviceToHost);
  if (e != cudaSuccess) return e;
  auto bf = [](float f) -> uint32_t {   // round to nearest even
    uint32_t u;
    memcpy(&u, &f, 4);
    if ((u & 0x7f800000u) == 0x7f800000u) return u >> 16;
    u += 0x7fffu + ((u >> 16) & 1u);
    return u >> 16;
  };
  auto B = [&](int layer, int k, int n) -> float {   // B[k][n] = W[n][k]
    if (layer == 1) return (k < NIN) ? w[O_W1 + n * NIN + k] : 0.0f;
    if (layer == 2) return w[O_W2 + n * NH + k];
    return n == 0 ? w[O_W3 + k] : 0.0f;
  };
  std::vector<uint2> f(F_TOTAL);
  auto fill = [&](int layer, int off, int KT, int NT) {
    for (int kt = 0; kt < KT; ++kt)
      for (int nt = 0; nt < NT; ++nt)
        for (int lane = 0; lane < 32; ++lane) {
          const int g = lane >> 2, q = lane & 3, n = 8 * nt + g, k = 16 * kt + 2 * q;
          uint2 u;
          u.x = bf(B(layer, k, n)) | (bf(B(layer, k + 1, n)) << 16);
          u.y = bf(B(layer, k + 8, n)) | (bf(B(layer, k + 9, n)) << 16);
          f[off + (kt * NT + nt) * 32 + lane] = u;
        }
  };
  fill(1, F_L1, 1, 8);
  fill(2, F_L2, 4, 8);
  fill(3, F_L3, 4, 1);
  e = cudaMemcpy(M->frag, f.data(), F_TOTAL * sizeof(uint2), cudaMemcpyHostToDevice);
  if (e != cudaSuccess) return e;
  std::vector<float> b(2 * NH);
  for (int a = 0; a < NH; ++a) { b[a] = w[O_B1 + a]; b[NH + a] = w[O_B2 + a]; }
  e = cudaMemcpy(M->bias, b.data(), 2 * NH * sizeof(float), cudaMemcpyHostToDevice);
  M->b3 = w[O_B3];
  return e;
}

// grad <- d loss / d w over nb samples (normalised x, t on the device); loss
// (device double) receives the sum of squared residuals.
cudaError_t launch_loss_grad(phl_mlp *M, long nb, const float *x, const float *t, double *loss, cudaStream_t s) {
  const cudaError_t e = cudaFuncSetAttribute(k_loss_grad, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)LG_SMEM);
  if (e != cudaSuccess) return e;
  cudaMemsetAsync(M->grad, 0, NPARAM * sizeof(float), s);
  cudaMemsetAsync(loss, 0, sizeof(double), s);
  // three blocks fit an SM; a block's tiles share its weights and its sums
  const unsigned grid = (unsigned)std::min<long>((nb + LG_S - 1) / LG_S, 3L * M->sms);
  k_loss_grad<<<grid, LG_T, LG_SMEM, s>>>(M->w, nb, x, t, 1.0f / (float)nb, M->grad, loss);
  return cudaGetLastError();
}

}  // namespace

mlp::Dev mlp_view(const phl_mlp *M) {
  mlp::Dev d;
  d.frag = M->frag;
  d.b1 = M->bias;
  d.b2 = M->bias + NH;
  d.b3 = M->b3;
  for (int k = 0; k < 4; ++k) { d.c[k] = M->c[k]; d.s[k] = M->s[k]; }
  return d;
}

}  // namespace phl

using namespace phl;

extern "C" {

phl_status phl_mlp_create(unsigned long long seed, phl_mlp **out) {
  if (!out) return (phl_status)set_error(PHL_EINVAL, "phl_mlp_create: null out");
  *out = nullptr;
  phl_mlp *M = new phl_mlp();
  scratch_owner(1);
  cudaError_t e = cudaMalloc(&M->w, 4 * NPARAM * sizeof(float));
  if (e == cudaSuccess) e = cudaMalloc(&M->frag, F_TOTAL * sizeof(uint2));
  if (e == cudaSuccess) e = cudaMalloc(&M->bias, 2 * NH * sizeof(float));
  if (e != cudaSuccess) {
    phl_mlp_destroy(M);
    return (phl_status)set_error(PHL_ENOMEM, "phl_mlp_create: %s", cudaGetErrorString(e));
  }
  M->m = M->w + NPARAM;
  M->v = M->w + 2 * NPARAM;
  M->grad = M->w + 3 * NPARAM;
  // Glorot-uniform initial weights from SplitMix64, zero biases
  std::vector<float> w(NPARAM, 0.0f);
  auto u = [&](long i) { return (double)(splitmix64(seed ^ splitmix64((uint64_t)i)) >> 11) / 9007199254740992.0; };
  const double l1 = sqrt(6.0 / (NIN + NH)), l2 = sqrt(6.0 / (2 * NH)), l3 = sqrt(6.0 / (NH + 1));
  for (int i = 0; i < NH * NIN; ++i) w[O_W1 + i] = (float)(l1 * (2 * u(i) - 1));
  for (int i = 0; i < NH * NH; ++i) w[O_W2 + i] = (float)(l2 * (2 * u(10000 + i) - 1));
  for (int i = 0; i < NH; ++i) w[O_W3 + i] = (float)(l3 * (2 * u(20000 + i) - 1));
  e = cudaMemcpy(M->w, w.data(), NPARAM * sizeof(float), cudaMemcpyHostToDevice);
  if (e == cudaSuccess) e = cudaMemset(M->m, 0, 2 * NPARAM * sizeof(float));
  if (e == cudaSuccess) e = build_fragments(M);
  if (e != cudaSuccess) {
    phl_mlp_destroy(M);
    return cuda_status(e, "phl_mlp_create");
  }
  *out = M;
  return PHL_OK;
}

void phl_mlp_destroy(phl_mlp *M) {
  if (!M) return;
  cudaFree(M->w);
  cudaFree(M->frag);
  cudaFree(M->bias);
  delete M;
  scratch_owner(-1);
}

phl_status phl_mlp_set_weights(phl_mlp *M, const float *w) {
  if (!M || !w) return (phl_status)set_error(PHL_EINVAL, "phl_mlp_set_weights: null argument");
  cudaError_t e = cudaMemcpy(M->w, w, NPARAM * sizeof(float), cudaMemcpyHostToDevice);
  if (e == cudaSuccess) e = cudaMemset(M->m, 0, 2 * NPARAM * sizeof(float));
  M->adam_t = 0;
  if (e == cudaSuccess) e = build_fragments(M);
  return e == cudaSuccess ? PHL_OK : cuda_status(e, "phl_mlp_set_weights");
}

phl_status phl_mlp_get_weights(const phl_mlp *M, float *w) {
  if (!M || !w) return (phl_status)set_error(PHL_EINVAL, "phl_mlp_get_weights: null argument");
  cudaError_t e = cudaMemcpy(w, M->w, NPARAM * sizeof(float), cudaMemcpyDeviceToHost);
  return e == cudaSuccess ? PHL_OK : cuda_status(e, "phl_mlp_get_weights");
}

phl_status phl_mlp_set_norm(phl_mlp *M, const double *c, const double *s) {
  if (!M || !c || !s) return (phl_status)set_error(PHL_EINVAL, "phl_mlp_set_norm: null argument");
  for (int k = 0; k < 4; ++k) {
    if (!(s[k] != 0.0) || !isfinite(c[k]) || !isfinite(s[k]))
      return (phl_status)set_error(PHL_EINVAL, "phl_mlp_set_norm: bad map");
    M->c[k] = (float)c[k];
    M->s[k] = (float)s[k];
  }
  return PHL_OK;
}

phl_status phl_mlp_get_norm(const phl_mlp *M, double *c, double *s) {
  if (!M || !c || !s) return (phl_status)set_error(PHL_EINVAL, "phl_mlp_get_norm: null argument");
  for (int k = 0; k < 4; ++k) { c[k] = M->c[k]; s[k] = M->s[k]; }
  return PHL_OK;
}

phl_status phl_mlp_loss_grad(phl_mlp *M, long n, const float *x, const float *t, double *loss, float *grad,
                             int where) {
  if (!M || n <= 0 || !x || !t || !loss || !grad)
    return (phl_status)set_error(PHL_EINVAL, "phl_mlp_loss_grad: bad arguments");
  const float *dx = x, *dt = t;
  CallScratch room;   // the loss sum, then the samples
  constexpr size_t HEAD = 256;
  cudaError_t e = room.get(HEAD + (where == PHL_HOST ? 4 * n * sizeof(float) : 0), 0);
  double *dloss = (double *)room.p;
  if (e == cudaSuccess && where == PHL_HOST) {
    float *tmp = (float *)((char *)room.p + HEAD);
    e = cudaMemcpy(tmp, x, 3 * n * sizeof(float), cudaMemcpyHostToDevice);
    if (e == cudaSuccess) e = cudaMemcpy(tmp + 3 * n, t, n * sizeof(float), cudaMemcpyHostToDevice);
    dx = tmp;
    dt = tmp + 3 * n;
  }
  if (e == cudaSuccess) e = launch_loss_grad(M, n, dx, dt, dloss, 0);
  double l = 0.0;
  if (e == cudaSuccess) e = cudaMemcpy(&l, dloss, sizeof(double), cudaMemcpyDeviceToHost);
  if (e == cudaSuccess)
    e = cudaMemcpy(grad, M->grad, NPARAM * sizeof(float),
                   where == PHL_HOST ? cudaMemcpyDeviceToHost : cudaMemcpyDeviceToDevice);
  if (e == cudaSuccess) e = cudaDeviceSynchronize();   // a copy within the device does not wait
  if (e != cudaSuccess) return cuda_status(e, "phl_mlp_loss_grad");
  *loss = l / (double)n;
  return PHL_OK;
}

phl_status phl_mlp_forward(const phl_mlp *M, long n, const float *x, float *y, int where) {
  if (!M || n <= 0 || !x || !y) return (phl_status)set_error(PHL_EINVAL, "phl_mlp_forward: bad arguments");
  const float *dx = x;
  float *dy = y;
  CallScratch room;
  cudaError_t e = cudaSuccess;
  if (where == PHL_HOST) {
    e = room.get(4 * n * sizeof(float), 0);
    float *tmp = (float *)room.p;
    if (e == cudaSuccess) e = cudaMemcpy(tmp, x, 3 * n * sizeof(float), cudaMemcpyHostToDevice);
    dx = tmp;
    dy = tmp + 3 * n;
  }
  if (e == cudaSuccess) {
    k_infer<<<(unsigned)((n + 127) / 128), 128>>>(mlp_view(M), n, dx, dy);
    e = cudaGetLastError();
  }
  if (e == cudaSuccess && where == PHL_HOST) e = cudaMemcpy(y, dy, n * sizeof(float), cudaMemcpyDeviceToHost);
  if (e == cudaSuccess) e = cudaDeviceSynchronize();
  return e == cudaSuccess ? PHL_OK : cuda_status(e, "phl_mlp_forward");
}

phl_status phl_mlp_guess_temperature(const phl_mlp *M, const phl_eos_table *tab, long n, const double *rho,
                           const double *eint, const double *X0, double *T, int where) {
  if (!M || !tab || n <= 0 || !rho || !eint || !X0 || !T)
    return (phl_status)set_error(PHL_EINVAL, "phl_mlp_guess_temperature: bad arguments");
  const eos::Table &t = *eos_table_view(tab);
  const double Tlo = exp(t.y0), Thi = exp(t.y0 + (t.ny - 1) * t.dy);
  const double *dr = rho, *de = eint, *dx = X0;
  double *dT = T;
  CallScratch room;
  cudaError_t e = cudaSuccess;
  if (where == PHL_HOST) {
    e = room.get(4 * n * sizeof(double), 0);
    double *tmp = (double *)room.p;
    if (e == cudaSuccess) e = cudaMemcpy(tmp, rho, n * 8, cudaMemcpyHostToDevice);
    if (e == cudaSuccess) e = cudaMemcpy(tmp + n, eint, n * 8, cudaMemcpyHostToDevice);
    if (e == cudaSuccess) e = cudaMemcpy(tmp + 2 * n, X0, n * 8, cudaMemcpyHostToDevice);
    dr = tmp; de = tmp + n; dx = tmp + 2 * n; dT = tmp + 3 * n;
  }
  if (e == cudaSuccess) {
    k_guess<<<(unsigned)((n + 127) / 128), 128>>>(mlp_view(M), n, dr, de, dx, Tlo, Thi, dT);
    e = cudaGetLastError();
  }
  if (e == cudaSuccess && where == PHL_HOST) e = cudaMemcpy(T, dT, n * 8, cudaMemcpyDeviceToHost);
  if (e == cudaSuccess) e = cudaDeviceSynchronize();
  return e == cudaSuccess ? PHL_OK : cuda_status(e, "phl_mlp_guess_temperature");
}

phl_status phl_mlp_train(phl_mlp *M, const phl_eos_table *tab, const phl_mlp_train_cfg *cfg,
                         phl_mlp_train_stats *st) {
  if (!M || !tab || !cfg || cfg->nsamples < 1000 || cfg->batch < 32 || cfg->epochs < 1 || !(cfg->lr > 0.0))
    return (phl_status)set_error(PHL_EINVAL, "phl_mlp_train: bad arguments");
  const auto t0 = std::chrono::steady_clock::now();
  const eos::Table &t = *eos_table_view(tab);
  const long n = cfg->nsamples;
  const long nval = std::max(1000L, n / 20), ntr = n - nval;
  float *x = nullptr, *tt = nullptr, *pred = nullptr;
  int *fail = nullptr;
  unsigned int *mm = nullptr;
  cudaError_t e = cudaMalloc(&x, 3 * n * sizeof(float));
  if (e == cudaSuccess) e = cudaMalloc(&tt, n * sizeof(float));
  if (e == cudaSuccess) e = cudaMalloc(&pred, nval * sizeof(float));
  if (e == cudaSuccess) e = cudaMalloc(&fail, sizeof(int));
  if (e == cudaSuccess) e = cudaMalloc(&mm, 2 * sizeof(unsigned int));
  CallScratch room;
  if (e == cudaSuccess) e = room.get(sizeof(double), 0);
  double *dloss = (double *)room.p;
  phl_status ret = PHL_OK;
  auto done = [&](phl_status r) {
    cudaFree(x); cudaFree(tt); cudaFree(pred); cudaFree(fail); cudaFree(mm);
    return r;
  };
  if (e != cudaSuccess) return done((phl_status)set_error(PHL_ENOMEM, "phl_mlp_train: %s", cudaGetErrorString(e)));
  cudaMemset(fail, 0, sizeof(int));
  const unsigned nbk = (unsigned)((n + 255) / 256);
  k_samples<<<nbk, 256>>>(t, n, cfg->seed, cfg->lrho[0], cfg->lrho[1], cfg->lT[0], cfg->lT[1], cfg->A[0], cfg->Z[0],
                          cfg->A[1], cfg->Z[1], x, tt, fail);
  const unsigned int init[2] = {0x7f7fffffu, 0u};
  cudaMemcpy(mm, init, sizeof(init), cudaMemcpyHostToDevice);
  k_minmax_e<<<4 * 152, 256>>>(n, x, mm, mm + 1);
  int f = 0;
  unsigned int hm[2];
  e = cudaMemcpy(&f, fail, sizeof(int), cudaMemcpyDeviceToHost);
  if (e == cudaSuccess) e = cudaMemcpy(hm, mm, sizeof(hm), cudaMemcpyDeviceToHost);
  if (e != cudaSuccess) return done(cuda_status(e, "phl_mlp_train samples"));
  if (f) return done((phl_status)set_error(PHL_EINVAL, "phl_mlp_train: sample range leaves the EOS table"));
  float emin, emax;
  memcpy(&emin, &hm[0], 4);
  memcpy(&emax, &hm[1], 4);
  // affine maps onto [-1, 1]
  M->c[0] = (float)(0.5 * (cfg->lrho[0] + cfg->lrho[1]));
  M->s[0] = (float)(2.0 / (cfg->lrho[1] - cfg->lrho[0]));
  M->c[1] = 0.5f * (emin + emax);
  M->s[1] = 2.0f / (emax - emin);
  M->c[2] = 0.5f;
  M->s[2] = 2.0f;
  M->c[3] = (float)(0.5 * (cfg->lT[0] + cfg->lT[1]));
  M->s[3] = (float)(2.0 / (cfg->lT[1] - cfg->lT[0]));
  k_normalise<<<nbk, 256>>>(n, x, tt, make_float4(M->c[0], M->c[1], M->c[2], M->c[3]),
                            make_float4(M->s[0], M->s[1], M->s[2], M->s[3]));
  // Adam on minibatches in sample order (the samples are i.i.d.); cosine-decayed rate
  const long nbat = std::max(1L, ntr / cfg->batch);
  const long total = nbat * cfg->epochs;
  double last = 0.0;
  long step = 0;
  for (int ep = 0; ep < cfg->epochs; ++ep) {
    double ep_loss = 0.0;
    std::vector<double> losses;
    for (long b = 0; b < nbat; ++b, ++step) {
      const long off = b * cfg->batch;
      e = launch_loss_grad(M, cfg->batch, x + 3 * off, tt + off, dloss, 0);
      if (e != cudaSuccess) return done(cuda_status(e, "phl_mlp_train"));
      ++M->adam_t;
      const float lr = (float)(cfg->lr * 0.5 * (1.0 + cos(3.141592653589793 * (double)step / (double)total)));
      const float b1 = 0.9f, b2 = 0.999f;
      const float c1 = 1.0f - powf(b1, (float)M->adam_t), c2 = 1.0f - powf(b2, (float)M->adam_t);
      k_adam<<<(NPARAM + 255) / 256, 256>>>(NPARAM, M->w, M->m, M->v, M->grad, lr, b1, b2, 1e-8f, c1, c2);
      if (b + 1 == nbat) {
        double l = 0.0;
        cudaMemcpy(&l, dloss, sizeof(double), cudaMemcpyDeviceToHost);
        ep_loss = l / (double)cfg->batch;
      }
    }
    last = ep_loss;
  }
  e = cudaDeviceSynchronize();
  if (e == cudaSuccess) e = build_fragments(M);
  if (e != cudaSuccess) return done(cuda_status(e, "phl_mlp_train"));
  // validation on the held-out samples with the BF16 inference kernel
  k_infer<<<(unsigned)((nval + 127) / 128), 128>>>(mlp_view(M), nval, x + 3 * ntr, pred);
  std::vector<float> hp(nval), ht(nval);
  e = cudaMemcpy(hp.data(), pred, nval * sizeof(float), cudaMemcpyDeviceToHost);
  if (e == cudaSuccess) e = cudaMemcpy(ht.data(), tt + ntr, nval * sizeof(float), cudaMemcpyDeviceToHost);
  if (e != cudaSuccess) return done(cuda_status(e, "phl_mlp_train validation"));
  double se = 0.0, mx = 0.0;
  for (long i = 0; i < nval; ++i) {
    const double d = fabs((double)hp[i] - (double)ht[i]) / M->s[3];   // in log10 T
    se += d * d;
    mx = std::max(mx, d);
  }
  if (st) {
    st->final_loss = last;
    st->val_rms_log10T = sqrt(se / (double)nval);
    st->val_max_log10T = mx;
    st->steps = step;
    st->seconds = std::chrono::duration<double>(std::chrono::steady_clock::now() - t0).count();
  }
  return done(ret);
}

}  // extern "C"

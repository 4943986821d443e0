// Learned frequency surrogate: the network f(x) = L x + s * MLP(x), its training (forward,
// backward, Adam, closed-form ridge fit of L) and inference. The paper has no counterpart;
// the model predicts the mode diagonal of eps~^-1 - 1 on the fine frequencies of the grid
// from its values on a coarse subset.
//
//   MLP(x) = W4 h3 + b4,  h3 = silu(W3 h2 + b3),  h2 = silu(W2 h1 + b2),  h1 = silu(W1 x + b1)
//
// Parameters: one fp32 vector, W1 [H][I], b1 [H], W2 [H][H], b2 [H], W3 [H][H], b3 [H],
// W4 [O][H], b4 [O], L [O][I], s [1] (row-major). Matrix products read bf16 copies of
// W1..W4 and accumulate in fp32; biases, L and s are used in fp32. Adam trains W1..b4;
// L and s come from gw_surrogate_fit_linear (ridge normal equations in FP64).
#include "gw_internal.h"

#include <cuda_bf16.h>

#include <algorithm>
#include <cmath>
#include <cstdint>
#include <string>
#include <vector>

using namespace gw;

namespace {

thread_local std::string g_mlp_err;

gw_status mfail(gw_status s, const std::string& m) {
  g_mlp_err = m;
  gw_set_last_error(m);
  return s;
}

#define MLP_CUDA(call)                                                                     \
  do {                                                                                     \
    cudaError_t e_ = (call);                                                               \
    if (e_ != cudaSuccess) return mfail(GW_ERR_CUDA, std::string(#call) + ": " + cudaGetErrorString(e_)); \
  } while (0)

#define MLP_TRY(x)               \
  do {                           \
    gw_status s_ = (x);          \
    if (s_ != GW_OK) return s_;  \
  } while (0)

struct Offs {
  long long W1, b1, W2, b2, W3, b3, W4, b4, L, s, P;
};

Offs offsets(int I, int H, int O) {
  Offs o{};
  long long p = 0;
  o.W1 = p; p += (long long)H * I;
  o.b1 = p; p += H;
  o.W2 = p; p += (long long)H * H;
  o.b2 = p; p += H;
  o.W3 = p; p += (long long)H * H;
  o.b3 = p; p += H;
  o.W4 = p; p += (long long)O * H;
  o.b4 = p; p += O;
  o.L = p; p += (long long)O * I;
  o.s = p; p += 1;
  o.P = p;
  return o;
}

// ---------------------------------------------------------------------------------------------
// Dense products of the network, fp32 on CUDA cores: sum_k A(m,k) B(k,n) in ascending k,
//   A(m,k) = TA ? A[k*lda + m] : A[m*lda + k]   (fp32)
//   B(k,n) = BT ? B[n*ldb + k] : B[k*ldb + n]   (fp32 or bf16, converted to fp32)
// with the layer's elementwise part in the epilogue:
//   MM_PLAIN  C = alpha acc + bias[n]
//   MM_SILU   C = acc + bias[n], X = silu(C)                        (forward layer)
//   MM_DSILU  C = alpha acc silu'(X)                                (backward through a layer)
//   MM_PART   C[z][m][0..N) = acc, C[z][m][N] = sum_k A(m,k) over k part z  (weight and bias gradients)
// BM x 64 tiles (BM 128 or 64), 256 threads with BM/16 x 4 outputs each, k steps of 16 staged through
// registers into two shared buffers. The FP32 units bound it: 8 x 4 outputs per thread need 3 128-bit
// shared loads per 32 FMAs. The gradients reduce over the rows of the data set, M x N is one layer's
// weights: the k range is split so that the chip is filled, and the parts are added in order.
// 16384 rows, 12-256-256-256-48: loss and gradient 10.6 ms with 64 x 64 tiles of 4 x 4, one block per
// output tile of a gradient and one thread per bias column; 0.74 ms now.
// ---------------------------------------------------------------------------------------------
__device__ __forceinline__ float to_f(float v) { return v; }
__device__ __forceinline__ float to_f(__nv_bfloat16 v) { return __bfloat162float(v); }
__device__ __forceinline__ float sigm(float z) { return 1.f / (1.f + expf(-z)); }

enum { MM_PLAIN, MM_SILU, MM_DSILU, MM_PART };

template <int BM, typename TB, bool TA, bool BT, int EPI>
__global__ void __launch_bounds__(256) k_mm(int M, int N, int K, int kpart, const float* __restrict__ A, int lda,
                                            const TB* __restrict__ B, int ldb, float* __restrict__ C, int ldc,
                                            float alpha, const float* __restrict__ bias, float* __restrict__ X) {
  constexpr int AR = BM / 16, TMR = BM / 16;   // A elements staged per thread, outputs along m per thread
  __shared__ __align__(16) float As[2][16][BM + 4];
  __shared__ __align__(16) float Bs[2][16][64 + 4];
  const int m0 = blockIdx.y * BM, n0 = blockIdx.x * 64;
  const int k0 = blockIdx.z * kpart, k1 = min(K, k0 + kpart);
  const int tid = threadIdx.x, tx = tid % 16, ty = tid / 16;
  float ra[AR], rb[4];
  auto fetch = [&](int kb) {
#pragma unroll
    for (int r = 0; r < AR; ++r) {
      const int e = tid + 256 * r;
      const int mm = TA ? e % BM : e / 16, kk = TA ? e / BM : e % 16;
      const int gm = m0 + mm, gk = kb + kk;
      ra[r] = (gm < M && gk < k1) ? (TA ? A[(long long)gk * lda + gm] : A[(long long)gm * lda + gk]) : 0.f;
    }
#pragma unroll
    for (int r = 0; r < 4; ++r) {
      const int e = tid + 256 * r;
      const int nn = BT ? e / 16 : e % 64, kk = BT ? e % 16 : e / 64;
      const int gn = n0 + nn, gk = kb + kk;
      rb[r] = (gn < N && gk < k1) ? to_f(BT ? B[(long long)gn * ldb + gk] : B[(long long)gk * ldb + gn]) : 0.f;
    }
  };
  auto stash = [&](int s) {
#pragma unroll
    for (int r = 0; r < AR; ++r) {
      const int e = tid + 256 * r;
      As[s][TA ? e / BM : e % 16][TA ? e % BM : e / 16] = ra[r];
    }
#pragma unroll
    for (int r = 0; r < 4; ++r) {
      const int e = tid + 256 * r;
      Bs[s][BT ? e % 16 : e / 64][BT ? e / 16 : e % 64] = rb[r];
    }
  };
  float acc[TMR][4] = {};
  float csum = 0.f;                            // MM_PART: sum over k of A(m0 + tid, k), tid < BM
  fetch(k0);
  stash(0);
  __syncthreads();
  int s = 0;
  for (int kb = k0; kb < k1; kb += 16) {
    const bool more = kb + 16 < k1;
    if (more) fetch(kb + 16);
#pragma unroll
    for (int kk = 0; kk < 16; ++kk) {
      float a[TMR], b[4];
#pragma unroll
      for (int i = 0; i < TMR; i += 4)
        *reinterpret_cast<float4*>(a + i) = *reinterpret_cast<const float4*>(&As[s][kk][4 * ty + 16 * i]);
      *reinterpret_cast<float4*>(b) = *reinterpret_cast<const float4*>(&Bs[s][kk][4 * tx]);
#pragma unroll
      for (int i = 0; i < TMR; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) acc[i][j] = fmaf(a[i], b[j], acc[i][j]);
    }
    if constexpr (EPI == MM_PART) {
      if (blockIdx.x == 0 && tid < BM)
#pragma unroll
        for (int kk = 0; kk < 16; ++kk) csum += As[s][kk][tid];
    }
    if (more) {
      stash(s ^ 1);
      __syncthreads();
      s ^= 1;
    }
  }
#pragma unroll
  for (int i = 0; i < TMR; ++i) {
    const int m = m0 + 4 * ty + 16 * (i & ~3) + (i & 3);
    if (m >= M) continue;
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const int n = n0 + 4 * tx + j;
      if (n >= N) continue;
      if constexpr (EPI == MM_PART) {
        C[((long long)blockIdx.z * M + m) * (N + 1) + n] = acc[i][j];
      } else if constexpr (EPI == MM_DSILU) {
        const float z = X[(long long)m * ldc + n], sg = sigm(z);
        C[(long long)m * ldc + n] = alpha * acc[i][j] * sg * (1.f + z * (1.f - sg));
      } else {
        float v = alpha * acc[i][j];
        if (bias) v += bias[n];
        C[(long long)m * ldc + n] = v;
        if constexpr (EPI == MM_SILU) X[(long long)m * ldc + n] = v * sigm(v);
      }
    }
  }
  if constexpr (EPI == MM_PART) {
    if (blockIdx.x == 0 && tid < BM && m0 + tid < M) C[((long long)blockIdx.z * M + m0 + tid) * (N + 1) + N] = csum;
  }
}

// 128-row tiles once they fill the chip (152 SMs), else 64-row ones (twice the blocks)
template <typename TB, bool BT, int EPI>
void mm(int M, int N, int K, const float* A, int lda, const TB* B, int ldb, float* C, int ldc, float alpha,
        const float* bias, float* X, cudaStream_t st) {
  if (M <= 0 || N <= 0) return;
  const int nn = (N + 63) / 64;
  if ((long long)nn * (M / 128) >= 152) {
    ++g_launch_count, k_mm<128, TB, false, BT, EPI><<<dim3(nn, (M + 127) / 128), 256, 0, st>>>(M, N, K, K, A, lda, B, ldb,
                                                                                             C, ldc, alpha, bias, X);
  } else {
    ++g_launch_count, k_mm<64, TB, false, BT, EPI><<<dim3(nn, (M + 63) / 64), 256, 0, st>>>(M, N, K, K, A, lda, B, ldb, C,
                                                                                          ldc, alpha, bias, X);
  }
}

// k parts of a gradient product: two blocks per SM, at least 256 rows each
int grad_parts(int M, int N, int K) {
  const int tiles = ((N + 63) / 64) * ((M + 127) / 128);
  return std::max(1, std::min((2 * 152) / tiles, K / 256));
}

// gW[m][n] = alpha sum_z part[z][m][n], gb[m] (may be NULL) = alpha times column N
__global__ void k_grad_sum(int M, int N, int parts, const float* __restrict__ part, float alpha, float* __restrict__ gW,
                           float* __restrict__ gb) {
  const long long n = (long long)M * (N + 1);
  for (long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x; e < n; e += (long long)gridDim.x * blockDim.x) {
    float v = 0.f;
    for (int z = 0; z < parts; ++z) v += part[z * n + e];
    const long long m = e / (N + 1);
    const int c = (int)(e % (N + 1));
    if (c < N) gW[m * N + c] = alpha * v;
    else if (gb) gb[m] = alpha * v;
  }
}

// ---------------------------------------------------------------------------------------------
// elementwise pieces
// ---------------------------------------------------------------------------------------------
// F = F + s G (F holds x L^T on entry); R = F - Y; dF = 2 R / (B n_out); loss += sum R^2 / (B n_out)
__global__ void k_mse(long long n, float inv, float s, float* __restrict__ F, const float* __restrict__ G,
                      const float* __restrict__ Y, float* __restrict__ dF, double* __restrict__ loss) {
  __shared__ double red[256];
  double acc = 0.0;
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
    const float f = F[i] + s * G[i];
    F[i] = f;
    if (!Y) continue;
    const float r = f - Y[i];
    if (dF) dF[i] = 2.f * r * inv;
    acc += (double)r * r;
  }
  red[threadIdx.x] = acc;
  __syncthreads();
  for (int h = 128; h > 0; h >>= 1) {
    if (threadIdx.x < h) red[threadIdx.x] += red[threadIdx.x + h];
    __syncthreads();
  }
  if (threadIdx.x == 0 && loss) atomicAdd(loss, red[0] * (double)inv);
}

// bf16 copies of the weight matrices (round to nearest even); other entries copied too
__global__ void k_to_bf16(long long n, const float* __restrict__ a, __nv_bfloat16* __restrict__ b) {
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x)
    b[i] = __float2bfloat16_rn(a[i]);
}

// Adam (Kingma & Ba, Algorithm 1) on theta[0 .. n), step t = *t_dev + 1; refreshes the bf16 copy
__global__ void k_adam(long long n, float* __restrict__ th, const float* __restrict__ g, float* __restrict__ m,
                       float* __restrict__ v, __nv_bfloat16* __restrict__ wb, const int* __restrict__ t_dev, float lr,
                       float b1, float b2, float eps) {
  const int t = *t_dev + 1;
  const float c1 = 1.f / (1.f - powf(b1, (float)t)), c2 = 1.f / (1.f - powf(b2, (float)t));
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
    const float gi = g[i];
    const float mi = b1 * m[i] + (1.f - b1) * gi;
    const float vi = b2 * v[i] + (1.f - b2) * gi * gi;
    m[i] = mi;
    v[i] = vi;
    const float w = th[i] - lr * (mi * c1) / (sqrtf(vi * c2) + eps);
    th[i] = w;
    wb[i] = __float2bfloat16_rn(w);
  }
}

// rows of the next batch: xb[i] = x[perm[step * B + i]], yb likewise
__global__ void k_gather(int B, int I, int O, const float* __restrict__ x, const float* __restrict__ y,
                         const int* __restrict__ perm, const int* __restrict__ step, float* __restrict__ xb,
                         float* __restrict__ yb) {
  const int i = blockIdx.x;
  const int r = perm[(long long)(*step) * B + i];
  for (int j = threadIdx.x; j < I; j += blockDim.x) xb[(long long)i * I + j] = x[(long long)r * I + j];
  for (int j = threadIdx.x; j < O; j += blockDim.x) yb[(long long)i * O + j] = y[(long long)r * O + j];
}

__global__ void k_tick(int* __restrict__ step, int* __restrict__ t) {
  ++*step;
  ++*t;
}

// FP64 normal equations of the ridge fit: G += x^T x, R += x^T y over a chunk of rows per block
__global__ void k_gram(long long n, int I, int O, const float* __restrict__ x, const float* __restrict__ y,
                       long long rows_per_block, double* __restrict__ G, double* __restrict__ R) {
  const long long r0 = blockIdx.x * rows_per_block, r1 = min(n, r0 + rows_per_block);
  const int outs = I * (I + O);
  for (int e = threadIdx.x; e < outs; e += blockDim.x) {
    const int i = e / (I + O), j = e % (I + O);
    double acc = 0.0;
    if (j < I) {
      for (long long r = r0; r < r1; ++r) acc += (double)x[r * I + i] * (double)x[r * I + j];
      atomicAdd(&G[i * I + j], acc);
    } else {
      const int o = j - I;
      for (long long r = r0; r < r1; ++r) acc += (double)x[r * I + i] * (double)y[r * O + o];
      atomicAdd(&R[i * O + o], acc);
    }
  }
}

// (G + lam 1) L^T = R by Cholesky in shared memory (I <= 64); writes L [O][I] (fp32) into theta.
// One block; status bit ST_NOT_PD if a pivot is not positive.
__global__ void k_ridge_solve(int I, int O, const double* __restrict__ G, const double* __restrict__ R, double lam,
                              float* __restrict__ Lout, int* __restrict__ status) {
  __shared__ double c[64][65];
  for (int e = threadIdx.x; e < I * I; e += blockDim.x) c[e / I][e % I] = G[e] + (e / I == e % I ? lam : 0.0);
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int j = 0; j < I; ++j) {
      double d = c[j][j];
      for (int k = 0; k < j; ++k) d -= c[j][k] * c[j][k];
      if (!(d > 0.0)) {
        atomicOr(status, ST_NOT_PD);
        d = 1e-300;
      }
      c[j][j] = sqrt(d);
      for (int i = j + 1; i < I; ++i) {
        double s = c[i][j];
        for (int k = 0; k < j; ++k) s -= c[i][k] * c[j][k];
        c[i][j] = s / c[j][j];
      }
    }
  }
  __syncthreads();
  for (int o = threadIdx.x; o < O; o += blockDim.x) {
    double z[64];
    for (int i = 0; i < I; ++i) {  // forward: C z = r
      double s = R[i * O + o];
      for (int k = 0; k < i; ++k) s -= c[i][k] * z[k];
      z[i] = s / c[i][i];
    }
    for (int i = I - 1; i >= 0; --i) {  // backward: C^T l = z
      double s = z[i];
      for (int k = i + 1; k < I; ++k) s -= c[k][i] * z[k];
      z[i] = s / c[i][i];
    }
    for (int i = 0; i < I; ++i) Lout[(long long)o * I + i] = (float)z[i];
  }
}

// sum of squared residuals of the linear map in FP64: sum (y - x L^T)^2
__global__ void k_lin_resid(long long n, int I, int O, const float* __restrict__ x, const float* __restrict__ y,
                            const float* __restrict__ L, double* __restrict__ out) {
  __shared__ double red[256];
  double acc = 0.0;
  for (long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x; e < n * O;
       e += (long long)gridDim.x * blockDim.x) {
    const long long r = e / O;
    const int o = (int)(e % O);
    double f = 0.0;
    for (int i = 0; i < I; ++i) f += (double)L[(long long)o * I + i] * (double)x[r * I + i];
    const double d = (double)y[e] - f;
    acc += d * d;
  }
  red[threadIdx.x] = acc;
  __syncthreads();
  for (int h = 128; h > 0; h >>= 1) {
    if (threadIdx.x < h) red[threadIdx.x] += red[threadIdx.x + h];
    __syncthreads();
  }
  if (threadIdx.x == 0) atomicAdd(out, red[0]);
}

inline int ew_grid(long long n) { return (int)std::min<long long>((n + 255) / 256, 152LL * 16); }

}  // namespace

namespace {
// residual targets of the MLP in FP64: yr = (y - x L^T) / s
__global__ void k_resid_targets(long long n, int I, int O, const float* __restrict__ x, const float* __restrict__ y,
                                const float* __restrict__ L, const float* __restrict__ s_dev, float* __restrict__ yr) {
  const double inv_s = 1.0 / (double)(*s_dev);
  for (long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x; e < n * O;
       e += (long long)gridDim.x * blockDim.x) {
    const long long r = e / O;
    const int o = (int)(e % O);
    double f = 0.0;
    for (int i = 0; i < I; ++i) f += (double)L[(long long)o * I + i] * (double)x[r * I + i];
    yr[e] = (float)(((double)y[e] - f) * inv_s);
  }
}

// loss += sum (G - Y)^2 / (B O) and dG = 2 (G - Y) / (B O)   (residual form, no linear part)
__global__ void k_mse_res(long long n, float inv, const float* __restrict__ G, const float* __restrict__ Y,
                          float* __restrict__ dG, double* __restrict__ loss) {
  __shared__ double red[256];
  double acc = 0.0;
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
    const float r = G[i] - Y[i];
    dG[i] = 2.f * r * inv;
    acc += (double)r * r;
  }
  red[threadIdx.x] = acc;
  __syncthreads();
  for (int h = 128; h > 0; h >>= 1) {
    if (threadIdx.x < h) red[threadIdx.x] += red[threadIdx.x + h];
    __syncthreads();
  }
  if (threadIdx.x == 0) atomicAdd(loss, red[0] * (double)inv);
}
}  // namespace

// ---------------------------------------------------------------------------------------------
// the model
// ---------------------------------------------------------------------------------------------
struct gw_surrogate_s {
  int I = 0, H = 0, O = 0;
  Offs off{};
  cudaStream_t st = nullptr;     // the model's own stream (non-blocking)
  cudaStream_t user = nullptr;   // the caller's stream, ordered against st by events
  cudaEvent_t ev_in = nullptr, ev_out = nullptr;
  float* th = nullptr;           // fp32 parameters [P]
  __nv_bfloat16* wb = nullptr;   // bf16 copy [P] (matrix entries are the ones used)
  float* grad = nullptr;         // [P]
  float *am = nullptr, *av = nullptr;  // Adam moments [P]
  int* d_ctr = nullptr;          // [0] batch index within the epoch, [1] Adam step count
  double* d_acc = nullptr;       // [0] loss accumulator, [1..] scratch
  int* d_status = nullptr;
  float h_s = 1.f;               // host copy of the output scale s
  // activations for up to cap rows
  int cap = 0;
  float *xb = nullptr, *yb = nullptr, *Z1 = nullptr, *H1 = nullptr, *Z2 = nullptr, *H2 = nullptr, *Z3 = nullptr,
        *H3 = nullptr, *G = nullptr, *F = nullptr, *dG = nullptr, *dA = nullptr, *dB = nullptr, *part = nullptr;
  std::vector<void*> allocs;
};

namespace {

gw_status salloc(gw_surrogate_s* m, void** p, size_t bytes) {
  ++::gw::g_alloc_count;
  cudaError_t e = cudaMalloc(p, std::max<size_t>(bytes, 16));
  if (e != cudaSuccess) {
    cudaGetLastError();
    return mfail(GW_ERR_NOMEM, "surrogate: cudaMalloc of " + std::to_string(bytes) + " bytes failed");
  }
  m->allocs.push_back(*p);
  return GW_OK;
}

template <typename T>
gw_status salloc_n(gw_surrogate_s* m, T** p, size_t n) {
  return salloc(m, reinterpret_cast<void**>(p), n * sizeof(T));
}

void sfree(gw_surrogate_s* m, void* p) {
  if (!p) return;
  cudaFree(p);
  auto it = std::find(m->allocs.begin(), m->allocs.end(), p);
  if (it != m->allocs.end()) m->allocs.erase(it);
}

gw_status ensure_cap(gw_surrogate_s* m, int rows) {
  if (rows <= m->cap) return GW_OK;
  float** bufs[] = {&m->xb, &m->yb, &m->Z1, &m->H1, &m->Z2, &m->H2, &m->Z3, &m->H3, &m->G, &m->F, &m->dG, &m->dA, &m->dB,
                    &m->part};
  for (float** b : bufs) {
    sfree(m, *b);
    *b = nullptr;
  }
  const size_t r = (size_t)rows;
  const size_t wI = m->I, wH = m->H, wO = m->O;
  MLP_TRY(salloc_n(m, &m->xb, r * wI));
  MLP_TRY(salloc_n(m, &m->yb, r * wO));
  MLP_TRY(salloc_n(m, &m->Z1, r * wH));
  MLP_TRY(salloc_n(m, &m->H1, r * wH));
  MLP_TRY(salloc_n(m, &m->Z2, r * wH));
  MLP_TRY(salloc_n(m, &m->H2, r * wH));
  MLP_TRY(salloc_n(m, &m->Z3, r * wH));
  MLP_TRY(salloc_n(m, &m->H3, r * wH));
  MLP_TRY(salloc_n(m, &m->G, r * wO));
  MLP_TRY(salloc_n(m, &m->F, r * wO));
  MLP_TRY(salloc_n(m, &m->dG, r * wO));
  MLP_TRY(salloc_n(m, &m->dA, r * wH));
  MLP_TRY(salloc_n(m, &m->dB, r * wH));
  // parts of the gradient products over up to `rows` rows
  size_t parts = 0;
  const int shapes[4][2] = {{m->O, m->H}, {m->H, m->H}, {m->H, m->I}, {m->O, m->I}};
  for (const auto& s : shapes)
    parts = std::max(parts, (size_t)grad_parts(s[0], s[1], rows) * s[0] * ((size_t)s[1] + 1));
  MLP_TRY(salloc_n(m, &m->part, parts));
  m->cap = rows;
  return GW_OK;
}

// G = MLP(x) (without the output scale s) for B rows of x; activations kept for backward
void forward_mlp(gw_surrogate_s* m, const float* x, int B, float* G, cudaStream_t st) {
  using W = __nv_bfloat16;
  const int I = m->I, H = m->H, O = m->O;
  const Offs& o = m->off;
  mm<W, true, MM_SILU>(B, H, I, x, I, m->wb + o.W1, I, m->Z1, H, 1.f, m->th + o.b1, m->H1, st);
  mm<W, true, MM_SILU>(B, H, H, m->H1, H, m->wb + o.W2, H, m->Z2, H, 1.f, m->th + o.b2, m->H2, st);
  mm<W, true, MM_SILU>(B, H, H, m->H2, H, m->wb + o.W3, H, m->Z3, H, 1.f, m->th + o.b3, m->H3, st);
  mm<W, true, MM_PLAIN>(B, O, H, m->H3, H, m->wb + o.W4, H, G, O, 1.f, m->th + o.b4, nullptr, st);
}

// gW[M][N] = alpha sum_r dZ[r][m] X[r][n], gb[m] = alpha sum_r dZ[r][m] over the B rows
void weight_grad(gw_surrogate_s* m, int M, int N, int B, const float* dZ, const float* X, float alpha, float* gW,
                 float* gb, cudaStream_t st) {
  const int parts = grad_parts(M, N, B), kpart = ((B + parts - 1) / parts + 15) / 16 * 16;
  const int used = (B + kpart - 1) / kpart;
  ++g_launch_count, k_mm<128, float, true, false, MM_PART><<<dim3((N + 63) / 64, (M + 127) / 128, used), 256, 0, st>>>(
      M, N, B, kpart, dZ, M, X, N, m->part, 0, 1.f, nullptr, nullptr);
  const long long n = (long long)M * (N + 1);
  ++g_launch_count, k_grad_sum<<<(int)std::min<long long>((n + 255) / 256, 152LL * 16), 256, 0, st>>>(M, N, used, m->part,
                                                                                                    alpha, gW, gb);
}

// gradients of the W/b parameters from dG = dLoss/d(MLP output) for the B rows of x (alpha
// scales every gradient, e.g. by s); fills m->grad[W1 .. b4]
void backward_mlp(gw_surrogate_s* m, const float* x, int B, const float* dG, float alpha, cudaStream_t st) {
  using W = __nv_bfloat16;
  const int I = m->I, H = m->H, O = m->O;
  const Offs& o = m->off;
  float* g = m->grad;
  weight_grad(m, O, H, B, dG, m->H3, alpha, g + o.W4, g + o.b4, st);
  mm<W, false, MM_DSILU>(B, H, O, dG, O, m->wb + o.W4, H, m->dA, H, alpha, nullptr, m->Z3, st);    // dZ3
  weight_grad(m, H, H, B, m->dA, m->H2, 1.f, g + o.W3, g + o.b3, st);
  mm<W, false, MM_DSILU>(B, H, H, m->dA, H, m->wb + o.W3, H, m->dB, H, 1.f, nullptr, m->Z2, st);   // dZ2
  weight_grad(m, H, H, B, m->dB, m->H1, 1.f, g + o.W2, g + o.b2, st);
  mm<W, false, MM_DSILU>(B, H, H, m->dB, H, m->wb + o.W2, H, m->dA, H, 1.f, nullptr, m->Z1, st);   // dZ1
  weight_grad(m, H, I, B, m->dA, x, 1.f, g + o.W1, g + o.b1, st);
}

gw_status begin(gw_surrogate_s* m) {
  MLP_CUDA(cudaEventRecord(m->ev_in, m->user));
  MLP_CUDA(cudaStreamWaitEvent(m->st, m->ev_in, 0));
  return GW_OK;
}

gw_status finish(gw_surrogate_s* m, const char* where) {
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return mfail(GW_ERR_CUDA, std::string(where) + ": " + cudaGetErrorString(e));
  MLP_CUDA(cudaEventRecord(m->ev_out, m->st));
  MLP_CUDA(cudaStreamWaitEvent(m->user, m->ev_out, 0));
  return GW_OK;
}

}  // namespace

namespace {

__global__ void k_scale_copy(long long n, float s, const float* __restrict__ a, float* __restrict__ b) {
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x)
    b[i] = s * a[i];
}

uint64_t splitmix64(uint64_t& x) {
  uint64_t z = (x += 0x9E3779B97F4A7C15ull);
  z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
  z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
  return z ^ (z >> 31);
}

bool dims_ok(const gw_surrogate_dims* d) {
  return d && d->n_in >= 1 && d->n_in <= 64 && d->n_hidden >= 1 && d->n_hidden <= 4096 && d->n_out >= 1 &&
         d->n_out <= 1024;
}

constexpr int kChunk = 8192;  // rows per forward pass of gw_surrogate_forward

}  // namespace

namespace gw {

// g = s * MLP(x) for n <= 4096 rows on stream st (used by the plan's surrogate pass)
gw_status sur_correction(gw_surrogate_s* m, const float* x, int n, float* g_out, cudaStream_t st) {
  if (n > 4096) return mfail(GW_ERR_ARG, "surrogate: too many modes for one pass");
  MLP_TRY(ensure_cap(m, std::max(n, 1)));
  forward_mlp(m, x, n, m->G, st);
  const long long no = (long long)n * m->O;
  ++g_launch_count, k_scale_copy<<<ew_grid(no), 256, 0, st>>>(no, m->h_s, m->G, g_out);
  return GW_OK;
}

int sur_n_in(const gw_surrogate_s* m) { return m->I; }
int sur_n_out(const gw_surrogate_s* m) { return m->O; }
const float* sur_linear(const gw_surrogate_s* m) { return m->th + m->off.L; }

}  // namespace gw

extern "C" {

gw_status gw_surrogate_param_count(const gw_surrogate_dims* dims, int64_t* count) {
  if (!dims_ok(dims) || !count) return mfail(GW_ERR_ARG, "surrogate: bad dims or NULL count");
  *count = offsets(dims->n_in, dims->n_hidden, dims->n_out).P;
  return GW_OK;
}

gw_status gw_surrogate_create(const gw_surrogate_dims* dims, const float* params, void* stream, gw_surrogate* out) {
  if (!out) return mfail(GW_ERR_ARG, "surrogate: out is NULL");
  *out = nullptr;
  if (!dims_ok(dims)) return mfail(GW_ERR_ARG, "surrogate: dims out of range (n_in 1..64, n_hidden 1..4096, n_out 1..1024)");
  if (!params) return mfail(GW_ERR_ARG, "surrogate: params is NULL");
  auto* m = new (std::nothrow) gw_surrogate_s();
  if (!m) return mfail(GW_ERR_NOMEM, "surrogate: host allocation failed");
  m->I = dims->n_in;
  m->H = dims->n_hidden;
  m->O = dims->n_out;
  m->off = offsets(m->I, m->H, m->O);
  m->user = static_cast<cudaStream_t>(stream);
  auto fail_destroy = [&](gw_status s) {
    gw_surrogate_destroy(m);
    return s;
  };
  if (cudaStreamCreateWithFlags(&m->st, cudaStreamNonBlocking) != cudaSuccess ||
      cudaEventCreateWithFlags(&m->ev_in, cudaEventDisableTiming) != cudaSuccess ||
      cudaEventCreateWithFlags(&m->ev_out, cudaEventDisableTiming) != cudaSuccess)
    return fail_destroy(mfail(GW_ERR_CUDA, "surrogate: stream/event creation failed"));
  const size_t P = (size_t)m->off.P;
  gw_status s;
  if ((s = salloc_n(m, &m->th, P)) != GW_OK || (s = salloc_n(m, &m->wb, P)) != GW_OK ||
      (s = salloc_n(m, &m->grad, P)) != GW_OK || (s = salloc_n(m, &m->am, P)) != GW_OK ||
      (s = salloc_n(m, &m->av, P)) != GW_OK || (s = salloc_n(m, &m->d_ctr, 4)) != GW_OK ||
      (s = salloc_n(m, &m->d_acc, 2 + (size_t)m->I * (m->I + m->O))) != GW_OK ||
      (s = salloc_n(m, &m->d_status, 1)) != GW_OK)
    return fail_destroy(s);
  if ((s = begin(m)) != GW_OK) return fail_destroy(s);
  cudaMemcpyAsync(m->th, params, P * sizeof(float), cudaMemcpyDeviceToDevice, m->st);
  cudaMemsetAsync(m->am, 0, P * sizeof(float), m->st);
  cudaMemsetAsync(m->av, 0, P * sizeof(float), m->st);
  cudaMemsetAsync(m->grad, 0, P * sizeof(float), m->st);
  cudaMemsetAsync(m->d_ctr, 0, 4 * sizeof(int), m->st);
  ++g_launch_count, k_to_bf16<<<ew_grid((long long)P), 256, 0, m->st>>>((long long)P, m->th, m->wb);
  float hs = 1.f;
  cudaMemcpyAsync(&hs, m->th + m->off.s, sizeof(float), cudaMemcpyDeviceToHost, m->st);
  if (cudaStreamSynchronize(m->st) != cudaSuccess) return fail_destroy(mfail(GW_ERR_CUDA, "surrogate: create failed"));
  m->h_s = hs;
  if ((s = finish(m, "gw_surrogate_create")) != GW_OK) return fail_destroy(s);
  *out = m;
  return GW_OK;
}

gw_status gw_surrogate_destroy(gw_surrogate m) {
  if (!m) return GW_OK;
  if (m->st) cudaStreamSynchronize(m->st);
  for (void* p : m->allocs) cudaFree(p);
  if (m->ev_in) cudaEventDestroy(m->ev_in);
  if (m->ev_out) cudaEventDestroy(m->ev_out);
  if (m->st) cudaStreamDestroy(m->st);
  delete m;
  return GW_OK;
}

gw_status gw_surrogate_get_params(gw_surrogate m, float* params) {
  if (!m || !params) return mfail(GW_ERR_ARG, "surrogate: NULL argument");
  MLP_TRY(begin(m));
  MLP_CUDA(cudaMemcpyAsync(params, m->th, (size_t)m->off.P * sizeof(float), cudaMemcpyDeviceToDevice, m->st));
  return finish(m, "gw_surrogate_get_params");
}

gw_status gw_surrogate_set_params(gw_surrogate m, const float* params) {
  if (!m || !params) return mfail(GW_ERR_ARG, "surrogate: NULL argument");
  MLP_TRY(begin(m));
  const long long P = m->off.P;
  MLP_CUDA(cudaMemcpyAsync(m->th, params, (size_t)P * sizeof(float), cudaMemcpyDeviceToDevice, m->st));
  ++g_launch_count, k_to_bf16<<<ew_grid(P), 256, 0, m->st>>>(P, m->th, m->wb);
  float hs = 1.f;
  MLP_CUDA(cudaMemcpyAsync(&hs, m->th + m->off.s, sizeof(float), cudaMemcpyDeviceToHost, m->st));
  MLP_CUDA(cudaStreamSynchronize(m->st));
  m->h_s = hs;
  return finish(m, "gw_surrogate_set_params");
}

gw_status gw_surrogate_forward(gw_surrogate m, const float* x, int64_t n, float* f, float* g) {
  if (!m || !x || (!f && !g) || n < 0) return mfail(GW_ERR_ARG, "surrogate: bad forward arguments");
  MLP_TRY(begin(m));
  const int I = m->I, O = m->O;
  MLP_TRY(ensure_cap(m, (int)std::min<int64_t>(std::max<int64_t>(n, 1), kChunk)));
  for (int64_t r0 = 0; r0 < n; r0 += kChunk) {
    const int B = (int)std::min<int64_t>(kChunk, n - r0);
    const float* xr = x + r0 * I;
    forward_mlp(m, xr, B, m->G, m->st);
    const long long no = (long long)B * O;
    if (g) ++g_launch_count, k_scale_copy<<<ew_grid(no), 256, 0, m->st>>>(no, m->h_s, m->G, g + r0 * O);
    if (f) {
      float* fr = f + r0 * O;
      mm<float, true, MM_PLAIN>(B, O, I, xr, I, m->th + m->off.L, I, fr, O, 1.f, nullptr, nullptr, m->st);
      ++g_launch_count, k_mse<<<ew_grid(no), 256, 0, m->st>>>(no, 0.f, m->h_s, fr, m->G, nullptr, nullptr, nullptr);
    }
  }
  return finish(m, "gw_surrogate_forward");
}

gw_status gw_surrogate_loss_grad(gw_surrogate m, const float* x, const float* y, int64_t n, double* loss,
                                 float* grad) {
  if (!m || !x || !y || !loss || !grad || n < 1 || n > 65536)
    return mfail(GW_ERR_ARG, "surrogate: bad loss_grad arguments (1 <= n <= 65536)");
  MLP_TRY(begin(m));
  const int I = m->I, O = m->O, B = (int)n;
  const Offs& o = m->off;
  MLP_TRY(ensure_cap(m, B));
  MLP_CUDA(cudaMemsetAsync(m->d_acc, 0, sizeof(double), m->st));
  forward_mlp(m, x, B, m->G, m->st);
  mm<float, true, MM_PLAIN>(B, O, I, x, I, m->th + o.L, I, m->F, O, 1.f, nullptr, nullptr, m->st);
  const long long no = (long long)B * O;
  ++g_launch_count, k_mse<<<ew_grid(no), 256, 0, m->st>>>(no, 1.f / (float)no, m->h_s, m->F, m->G, y, m->dG,
                                                          m->d_acc);
  backward_mlp(m, x, B, m->dG, m->h_s, m->st);
  weight_grad(m, O, I, B, m->dG, x, 1.f, m->grad + o.L, nullptr, m->st);
  MLP_CUDA(cudaMemsetAsync(m->grad + o.s, 0, sizeof(float), m->st));
  MLP_CUDA(cudaMemcpyAsync(grad, m->grad, (size_t)o.P * sizeof(float), cudaMemcpyDeviceToDevice, m->st));
  double h = 0.0;
  MLP_CUDA(cudaMemcpyAsync(&h, m->d_acc, sizeof(double), cudaMemcpyDeviceToHost, m->st));
  MLP_CUDA(cudaStreamSynchronize(m->st));
  *loss = h;
  return finish(m, "gw_surrogate_loss_grad");
}

gw_status gw_surrogate_fit_linear(gw_surrogate m, const float* x, const float* y, int64_t n, double ridge,
                                  double* rms) {
  if (!m || !x || !y || n < 1 || !(ridge >= 0.0)) return mfail(GW_ERR_ARG, "surrogate: bad fit_linear arguments");
  MLP_TRY(begin(m));
  const int I = m->I, O = m->O;
  double* G = m->d_acc + 2;
  double* R = G + (size_t)I * I;
  MLP_CUDA(cudaMemsetAsync(m->d_acc, 0, (2 + (size_t)I * (I + O)) * sizeof(double), m->st));
  MLP_CUDA(cudaMemsetAsync(m->d_status, 0, sizeof(int), m->st));
  const long long rpb = std::max<long long>(256, (n + 152 * 4 - 1) / (152 * 4));
  const int nblk = (int)((n + rpb - 1) / rpb);
  ++g_launch_count, k_gram<<<nblk, 256, 0, m->st>>>(n, I, O, x, y, rpb, G, R);
  ++g_launch_count, k_ridge_solve<<<1, 64, 0, m->st>>>(I, O, G, R, ridge * (double)n, m->th + m->off.L, m->d_status);
  ++g_launch_count, k_lin_resid<<<ew_grid(n * O), 256, 0, m->st>>>(n, I, O, x, y, m->th + m->off.L, m->d_acc);
  double ss = 0.0;
  int stt = 0;
  MLP_CUDA(cudaMemcpyAsync(&ss, m->d_acc, sizeof(double), cudaMemcpyDeviceToHost, m->st));
  MLP_CUDA(cudaMemcpyAsync(&stt, m->d_status, sizeof(int), cudaMemcpyDeviceToHost, m->st));
  MLP_CUDA(cudaStreamSynchronize(m->st));
  if (stt & ST_NOT_PD) return mfail(GW_ERR_NOT_PD, "surrogate: x^T x + ridge is not positive definite");
  const double r = std::sqrt(ss / ((double)n * O));
  const float s = (r > 0.0 && std::isfinite(r)) ? (float)r : 1.f;
  MLP_CUDA(cudaMemcpyAsync(m->th + m->off.s, &s, sizeof(float), cudaMemcpyHostToDevice, m->st));
  MLP_CUDA(cudaStreamSynchronize(m->st));
  m->h_s = s;
  if (rms) *rms = r;
  return finish(m, "gw_surrogate_fit_linear");
}

gw_status gw_surrogate_fit_moments(gw_surrogate m, const double* moments, double ridge) {
  if (!m || !moments || !(ridge >= 0.0)) return mfail(GW_ERR_ARG, "surrogate: bad fit_moments arguments");
  MLP_TRY(begin(m));
  const int I = m->I, O = m->O;
  double* G = m->d_acc + 2;
  double* R = G + (size_t)I * I;
  std::vector<double> h((size_t)I * (I + O));
  MLP_CUDA(cudaMemcpyAsync(h.data(), moments, h.size() * sizeof(double), cudaMemcpyDeviceToHost, m->st));
  MLP_CUDA(cudaMemcpy2DAsync(G, I * sizeof(double), moments, (I + O) * sizeof(double), I * sizeof(double), I,
                             cudaMemcpyDeviceToDevice, m->st));
  MLP_CUDA(cudaMemcpy2DAsync(R, O * sizeof(double), moments + I, (I + O) * sizeof(double), O * sizeof(double), I,
                             cudaMemcpyDeviceToDevice, m->st));
  MLP_CUDA(cudaMemsetAsync(m->d_status, 0, sizeof(int), m->st));
  MLP_CUDA(cudaStreamSynchronize(m->st));
  double tr = 0.0;
  for (int i = 0; i < I; ++i) tr += h[(size_t)i * (I + O) + i];
  ++g_launch_count, k_ridge_solve<<<1, 64, 0, m->st>>>(I, O, G, R, ridge * tr / I, m->th + m->off.L, m->d_status);
  int stt = 0;
  MLP_CUDA(cudaMemcpyAsync(&stt, m->d_status, sizeof(int), cudaMemcpyDeviceToHost, m->st));
  MLP_CUDA(cudaStreamSynchronize(m->st));
  if (stt & ST_NOT_PD) return mfail(GW_ERR_NOT_PD, "surrogate: the coarse moment matrix + ridge is not positive definite");
  return finish(m, "gw_surrogate_fit_moments");
}

gw_status gw_surrogate_fit_scale(gw_surrogate m, const float* x, const float* y, int64_t n, double* rms) {
  if (!m || !x || !y || n < 1) return mfail(GW_ERR_ARG, "surrogate: bad fit_scale arguments");
  MLP_TRY(begin(m));
  const int I = m->I, O = m->O;
  MLP_CUDA(cudaMemsetAsync(m->d_acc, 0, sizeof(double), m->st));
  ++g_launch_count, k_lin_resid<<<ew_grid(n * O), 256, 0, m->st>>>(n, I, O, x, y, m->th + m->off.L, m->d_acc);
  double ss = 0.0;
  MLP_CUDA(cudaMemcpyAsync(&ss, m->d_acc, sizeof(double), cudaMemcpyDeviceToHost, m->st));
  MLP_CUDA(cudaStreamSynchronize(m->st));
  const double r = std::sqrt(ss / ((double)n * O));
  const float sc = (r > 0.0 && std::isfinite(r)) ? (float)r : 1.f;
  MLP_CUDA(cudaMemcpyAsync(m->th + m->off.s, &sc, sizeof(float), cudaMemcpyHostToDevice, m->st));
  MLP_CUDA(cudaStreamSynchronize(m->st));
  m->h_s = sc;
  if (rms) *rms = r;
  return finish(m, "gw_surrogate_fit_scale");
}

gw_status gw_surrogate_train(gw_surrogate m, const float* x, const float* y, int64_t n, int32_t epochs, int32_t batch,
                             double lr, uint64_t seed, double* loss_hist) {
  if (!m || !x || !y || n < 1 || n > (int64_t)1 << 30 || epochs < 0 || batch < 1 || batch > 4096 || batch > n ||
      !(lr > 0.0))
    return mfail(GW_ERR_ARG, "surrogate: bad train arguments (1 <= batch <= min(n, 4096), lr > 0)");
  MLP_TRY(begin(m));
  const int I = m->I, O = m->O, B = batch;
  const int nb = (int)(n / B);  // the last n % batch rows of each shuffled epoch are skipped
  MLP_TRY(ensure_cap(m, B));
  float* yr = nullptr;
  int* perm = nullptr;
  MLP_TRY(salloc_n(m, &yr, (size_t)n * O));
  gw_status st = salloc_n(m, &perm, (size_t)n);
  cudaGraph_t graph = nullptr;
  cudaGraphExec_t exec = nullptr;
  auto cleanup = [&](gw_status s) {
    if (exec) cudaGraphExecDestroy(exec);
    if (graph) cudaGraphDestroy(graph);
    cudaStreamSynchronize(m->st);
    sfree(m, yr);
    sfree(m, perm);
    return s;
  };
  if (st != GW_OK) return cleanup(st);
  // residual targets of the MLP: yr = (y - x L^T) / s, in FP64
  ++g_launch_count, k_resid_targets<<<ew_grid(n * O), 256, 0, m->st>>>(n, I, O, x, y, m->th + m->off.L,
                                                                       m->th + m->off.s, yr);
  // one training step (gather, forward, loss, backward, Adam, counters) as a CUDA graph
  const unsigned long long c0 = g_launch_count;
  if (cudaStreamBeginCapture(m->st, cudaStreamCaptureModeThreadLocal) != cudaSuccess)
    return cleanup(mfail(GW_ERR_CUDA, "surrogate: stream capture failed to begin"));
  const long long no = (long long)B * O;
  ++g_launch_count, k_gather<<<B, 64, 0, m->st>>>(B, I, O, x, yr, perm, m->d_ctr, m->xb, m->yb);
  forward_mlp(m, m->xb, B, m->G, m->st);
  ++g_launch_count, k_mse_res<<<ew_grid(no), 256, 0, m->st>>>(no, 1.f / (float)no, m->G, m->yb, m->dG, m->d_acc);
  backward_mlp(m, m->xb, B, m->dG, 1.f, m->st);
  ++g_launch_count, k_adam<<<ew_grid(m->off.L), 256, 0, m->st>>>(m->off.L, m->th, m->grad, m->am, m->av, m->wb,
                                                                 m->d_ctr + 1, (float)lr, 0.9f, 0.999f, 1e-8f);
  ++g_launch_count, k_tick<<<1, 1, 0, m->st>>>(m->d_ctr, m->d_ctr + 1);
  cudaError_t ce = cudaStreamEndCapture(m->st, &graph);
  const unsigned long long per_step = g_launch_count - c0;
  g_launch_count = c0;
  if (ce != cudaSuccess || !graph) return cleanup(mfail(GW_ERR_CUDA, std::string("surrogate: capture: ") + cudaGetErrorString(ce)));
  if (cudaGraphInstantiate(&exec, graph, 0) != cudaSuccess)
    return cleanup(mfail(GW_ERR_CUDA, "surrogate: graph instantiation failed"));
  std::vector<int> hp((size_t)n);
  uint64_t state = seed;
  const double s2 = (double)m->h_s * m->h_s;
  for (int e = 0; e < epochs; ++e) {
    for (int64_t i = 0; i < n; ++i) hp[i] = (int)i;
    for (int64_t i = n - 1; i > 0; --i) {  // Fisher-Yates with splitmix64
      const int64_t j = (int64_t)(splitmix64(state) % (uint64_t)(i + 1));
      std::swap(hp[i], hp[j]);
    }
    if (cudaMemcpyAsync(perm, hp.data(), (size_t)n * sizeof(int), cudaMemcpyHostToDevice, m->st) != cudaSuccess ||
        cudaMemsetAsync(m->d_ctr, 0, sizeof(int), m->st) != cudaSuccess ||
        cudaMemsetAsync(m->d_acc, 0, sizeof(double), m->st) != cudaSuccess)
      return cleanup(mfail(GW_ERR_CUDA, "surrogate: epoch set-up failed"));
    for (int b = 0; b < nb; ++b) {
      if (cudaGraphLaunch(exec, m->st) != cudaSuccess) return cleanup(mfail(GW_ERR_CUDA, "surrogate: graph launch failed"));
    }
    g_launch_count += per_step * (unsigned long long)nb;
    double acc = 0.0;
    if (cudaMemcpyAsync(&acc, m->d_acc, sizeof(double), cudaMemcpyDeviceToHost, m->st) != cudaSuccess ||
        cudaStreamSynchronize(m->st) != cudaSuccess)
      return cleanup(mfail(GW_ERR_CUDA, "surrogate: training step failed"));
    if (loss_hist) loss_hist[e] = s2 * acc / std::max(nb, 1);
  }
  gw_status fs = finish(m, "gw_surrogate_train");
  return cleanup(fs);
}

}  // extern "C"

// FP64 inversion of the batched Hermitian positive definite eps~ (step c), A := A^{-1} - I, with its
// rank-32 updates on the FP16 tensor cores as products of integer digits.
//
// Method: block elimination over pivot blocks P of 32 indices, in place. With the Cholesky factor
// L of B_PP and W = L^{-1},
//   Y_i = B_iP W^H,  B_ij <- B_ij - Y_i Y_j^H (i, j not in P),  B_iP <- Y_i W,  B_PP <- -W^H W,
// for every P; B = -A^{-1} at the end. Rows behind the pivot hold the Schur complement and rows
// before it build up -A^{-1} from the rows of L^{-1}, so this is a Cholesky inversion (N^3/2 complex
// multiply-adds) whose every step is one rank-32 update of the whole triangle, with its pivots and its
// stability. (The same sweep with the explicit inverse, T_i = B_iP B_PP^{-1} and B_ij - T_i B_jP^H, needs
// one product less per row but loses a further factor of up to kappa: 4e-7 instead of 4e-10 at
// kappa = 2e7.) Only one triangle is kept: B = A^T, element (i, j), i >= j, at mem[j * N + i] (rows of B
// contiguous).
//
// Emulated FP64 products: each row of the two factors (32 complex = 64 reals) is scaled by a power
// of two to 55-bit integers and cut into 7 balanced base-256 digits, exact in FP16. Products of
// digits d1, d2 are summed in FP32 accumulators by order d1 + d2 = 0..6 (28 of the 49 pairs): at
// most 7 pairs x 64 terms x 2^14 < 2^23, so every sum is an exact integer. The seven sums are put
// together in 64-bit integers and rounded to FP64 once. The dropped orders, above 6, are typically 2^-51
// of the product of the two rows' largest elements (digits of random sign; 2^-45 if every digit were -128),
// the size of the rounding of an FP64 dot product of 64 terms of that size.
//
// Scaling: an element 2^m below its row's largest is known to m bits less, so the error of a matrix D A D,
// D diagonal, would grow with the spread of D (which it does not in FP64 elimination): 5e-13 at a spread
// of 1e4, 4e-11 at 1e6. Rows and columns are therefore scaled by powers of two of the diagonal first, which is
// exact and leaves 4e-16 at every spread (N = 200, against 5e-16 for FP64 Cholesky). Elements between rows
// whose diagonal is in [1, 4) are not touched. It costs 1% of a screening call (16 matrices of N = 1200 with a
// larger diagonal: 0.13 of 15.3 ms).
//
// Why: the chip does ~2 FP64 FMA per clock and SM (1.1 TFLOP/s by cuBLAS DGEMM) and the 4 N^3 flops
// of an inverse bound the screening by that; 28 FP16 products of the tensor cores are ~25 times
// faster than one FP64 one. What is left in FP64 is one addition per element and pivot block, and
// the factor of the 32 x 32 pivot blocks. Every size is spread over the whole chip (a CTA per 64 rows
// of a matrix). Measured against one block per matrix with FP64 FMAs throughout: 1152 matrices of
// N = 400 332 -> 47 ms, 32 of them 44 -> 2.1 ms, 16 of N = 1200 1004 -> 10.7 ms, 32 of N = 96 1.5 -> 0.4 ms;
// the error against a refined inverse is the same (N = 400: 3.7e-16 and 5.6e-16 before at kappa = 3,
// 4.7e-10 and 6.5e-10 before at kappa = 2e7). Two thirds of it are the updates, which take ~9 us per 64 x 64
// tile: the products need 2, the FP64 conversions and additions of the epilogue 3, the rest is latency
// (loads of B, the handover of the accumulators, the left operand at the start of a row block).
#include "gw_internal.h"
#include "tc_ptx.cuh"

#include <algorithm>

namespace gw {

namespace {

using namespace ptx;

constexpr int PB = 32;                   // pivot block
constexpr int ND = 7;                    // digits per operand
constexpr int TM = 64;                   // complex rows (and columns) of a tile
constexpr int A_PIECE = 128 * ROWB;      // 16 KB: one digit of the left operand, Re / Im rows stacked
constexpr int B_PIECE = TM * ROWB;       // 8 KB: one digit of the right operand
constexpr int SLOTS = 2 * ND;            // right-operand ring: two tiles
constexpr int OFF_B = ND * A_PIECE;
constexpr int OFF_BAR = OFF_B + SLOTS * B_PIECE;
constexpr int UPD_SMEM = OFF_BAR + 8 * (2 * SLOTS + ND + 5) + 16 + 1024;
static_assert(UPD_SMEM <= 232448, "shared memory budget");
constexpr int EPI_WARPS = 16;
constexpr int UPD_THREADS = (EPI_WARPS + 2) * 32;
constexpr int W_PLANE = 2 * PB * ROWB;   // one digit of W, Re / Im rows stacked (64 rows)
constexpr int R_PLANE = PB * ROWB;       // one digit of W^H as right rows
constexpr int E_BAD = 1 << 20;           // exponent of a row with an infinity or a NaN

// ---- splitting into digits----------------------------------------------------------------------

// exponent field of the largest of 8 doubles
__device__ __forceinline__ int max_field(const double (&v)[8]) {
  int m = 0;
#pragma unroll
  for (int j = 0; j < 8; ++j) m = max(m, (__double2hiint(v[j]) >> 20) & 0x7ff);
  return m;
}

// x as an integer multiple of 2^(field - 1022 - 55), offset by 128 in each of the lower six digits:
// byte k < 6 of the result is digit 6 - k plus 128, the rest digit 0
__device__ __forceinline__ long long to_digits(double x, int field) {
  const long long b = __double_as_longlong(x);
  const int e = (int)((b >> 52) & 0x7ff);
  long long m = (b & 0xfffffffffffffLL) | 0x10000000000000LL;
  const int s = e - field + 2;
  if (s >= 0) {
    m <<= s;
  } else {
    const int r = -s;
    m = r > 54 ? 0 : (m + (1LL << (r - 1))) >> r;
  }
  if (e == 0) m = 0;
  return (b < 0 ? -m : m) + 0x808080808080LL;
}

// digit d of 8 values as 8 FP16 integers
template <int D> __device__ __forceinline__ uint4 digit8(const long long (&y)[8]) {
  uint32_t o[4];
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    uint32_t u;
    if constexpr (D == 0) {
      const int a = (int)(y[2 * j] >> 48) + 128, b = (int)(y[2 * j + 1] >> 48) + 128;
      u = (uint32_t)a | ((uint32_t)b << 16);
    } else {
      constexpr int k = 6 - D;          // byte of the digit
      const uint32_t a = (uint32_t)(y[2 * j] >> (k >= 4 ? 32 : 0)), b = (uint32_t)(y[2 * j + 1] >> (k >= 4 ? 32 : 0));
      u = __byte_perm(a, b, (k & 3) | (((k & 3) + 4) << 8)) & 0x00ff00ffu;   // byte k of a, byte k of b
    }
    u |= 0x64006400u;                   // 1024 + (digit + 128)
    const __half2 h = __hsub2(*reinterpret_cast<const __half2*>(&u), __halves2half2(__ushort_as_half(0x6480), __ushort_as_half(0x6480)));
    o[j] = *reinterpret_cast<const uint32_t*>(&h);
  }
  return make_uint4(o[0], o[1], o[2], o[3]);
}

template <int D, typename F> __device__ __forceinline__ void each_digit(const long long (&y)[8], F&& f) {
  if constexpr (D < ND) {
    f(D, digit8<D>(y));
    each_digit<D + 1>(y, f);
  }
}
__device__ __forceinline__ uint4 neg8(uint4 v) {
  return make_uint4(v.x ^ 0x80008000u, v.y ^ 0x80008000u, v.z ^ 0x80008000u, v.w ^ 0x80008000u);
}

// 2^ex, 0 below the normal range and infinity above it
__device__ __forceinline__ double pow2(int ex) {
  return __hiloint2double(max(0, min(ex + 1023, 2047)) << 20, 0);
}

__host__ __device__ __forceinline__ int padded(int N) { return (N + TM - 1) / TM * TM; }

// per-matrix workspace: digits of Y as right rows (yb) and as stacked left rows (ya), of W as left
// rows, of W^H as right rows, the rows' exponents, and the scales of A
struct InvLayout {
  long long yb, ya, w, r, ey, ew, er, sc;   // byte offsets of the arrays over the batch
  long long bytes;
};
InvLayout inv_layout(int N, int batch) {
  const long long Nr = padded(N);
  InvLayout l;
  l.yb = 0;
  l.ya = l.yb + (long long)batch * ND * Nr * ROWB;
  l.w = l.ya + (long long)batch * ND * 2 * Nr * ROWB;
  l.r = l.w + (long long)batch * ND * W_PLANE;
  l.ey = l.r + (long long)batch * ND * R_PLANE;
  l.ew = l.ey + (long long)batch * Nr * 4;
  l.er = l.ew + (long long)batch * PB * 4;
  l.sc = l.er + (long long)batch * PB * 4;
  l.bytes = l.sc + (long long)batch * N * 4;
  return l;
}

// the 8 lanes of a row agree on its exponent field; returns the exponent kept with the digits
__device__ __forceinline__ int row_field(const double (&x)[8], int& e) {
  int f = max_field(x);
  for (int o = 1; o < 8; o <<= 1) f = max(f, __shfl_xor_sync(0xffffffffu, f, o));
  e = f == 2047 ? E_BAD : (f == 0 ? 0 : f - 1022);
  return f;
}

// ---- scaling: A_ij <- 2^(s_i + s_j) A_ij with s_i taking the diagonal to [1, 4) ------------------

__global__ void k_inv_exps(int N, const c128* __restrict__ Aall, long long stride, int* __restrict__ sc) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= N) return;
  const double d = Aall[blockIdx.y * stride + (long long)i * (N + 1)].re;
  sc[(long long)blockIdx.y * N + i] = d > 0.0 && isfinite(d) ? -(ilogb(d) >> 1) : 0;
}

// The kept triangle of A; elements with nothing to scale are not touched
__global__ void k_inv_scale(int N, c128* __restrict__ Aall, long long stride, const int* __restrict__ scall) {
  if (blockIdx.x < blockIdx.y) return;
  c128* A = Aall + blockIdx.z * stride;
  const int* sc = scall + (long long)blockIdx.z * N;
  const int j0 = blockIdx.y * 32, i = blockIdx.x * 32 + threadIdx.x;
  if (i >= N) return;
  const int si = sc[i];
  for (int j = j0 + threadIdx.y; j < min(N, j0 + 32); j += blockDim.y) {
    const int sj = sc[j];
    if (i >= j && (si | sj) != 0) {
      c128& a = A[(long long)j * N + i];
      a = c128{a.re * pow2(sj) * pow2(si), a.im * pow2(sj) * pow2(si)};   // (one after the other: no overflow)
    }
  }
}

// ---- pivot block: W = L^{-1}, B_PP <- -W^H W ----------------------------------------------------
//
// One block per matrix, one element of the 32 x 32 triangle per thread: element (i, j) is A_ij while
// the elimination is left of its column, l_ij at column j, then builds up W_ij until row i is reached.
// Every step is one complex multiply-add per element between two barriers; the FP64 units (2 FMA per
// clock and SM) bound it.
constexpr int PIV_THREADS = 544;         // 528 elements of the triangle

__global__ void __launch_bounds__(PIV_THREADS) k_inv_pivot(int N, int p, c128* __restrict__ Aall, long long stride,
                                                           uint8_t* __restrict__ wdig, uint8_t* __restrict__ rdig,
                                                           int* __restrict__ eW, int* __restrict__ eR,
                                                           int* __restrict__ status) {
  __shared__ double2 buf[PB][PB + 1];    // W, zero above the diagonal
  __shared__ double2 raw[PB], u[PB];
  const int b = blockIdx.x, t = threadIdx.x;
  c128* A = Aall + b * stride;
  const int pw = min(PB, N - p);
  int i = (int)((sqrtf(8.0f * t + 1.0f) - 1.0f) * 0.5f);
  while ((i + 1) * (i + 2) / 2 <= t) ++i;
  while (i * (i + 1) / 2 > t) --i;
  const int j = t - i * (i + 1) / 2;
  const bool own = i < PB;
  double2 v = make_double2(0.0, 0.0);
  if (own) {
    if (i < pw) {
      const c128 a = A[(long long)(p + j) * N + p + i];
      v = make_double2(a.re, i == j ? 0.0 : a.im);
    } else if (i == j) {
      v.x = 1.0;                         // beyond N: identity
    }
  }
  for (int k = 0; k < PB; ++k) {
    // column k of A (rows i >= k) and row k of W so far (columns j < k)
    if (own && j == k) raw[i] = v;
    if (own && i == k && j < k) raw[j] = v;
    __syncthreads();
    if (t < 32) {
      double d = raw[k].x;
      if (!(d > 0.0)) {
        if (t == 0) atomicOr(status, ST_NOT_PD);
        d = 1.0;
      }
      const double rs = 1.0 / sqrt(d);
      const double2 c = raw[t];
      u[t] = t == k ? make_double2(rs, 0.0) : make_double2(c.x * rs, c.y * rs);
    }
    __syncthreads();
    if (own && i >= k) {
      if (i == k) {
        v = u[j];                        // row k of W is done
      } else {
        const double2 a = u[i];
        double2 f = u[j];
        if (j > k) f.y = -f.y;
        if (j == k) v = make_double2(0.0, 0.0);
        v.x = fma(-a.x, f.x, fma(a.y, f.y, v.x));
        v.y = fma(-a.x, f.y, fma(-a.y, f.x, v.y));
        if (i == j) v.y = 0.0;
      }
    }
  }
  if (own) {
    if (i >= pw) v = make_double2(0.0, 0.0);
    buf[i][j] = v;
    if (i != j) buf[j][i] = make_double2(0.0, 0.0);
  }
  __syncthreads();
  if (own && i < pw) {
    double gr = 0.0, gi = 0.0;           // G_ij = sum_{k >= i} conj(W_ki) W_kj
    for (int k = i; k < PB; ++k) {
      const double2 a = buf[k][i], c = buf[k][j];
      gr = fma(a.x, c.x, fma(a.y, c.y, gr));
      gi = fma(a.x, c.y, fma(-a.y, c.x, gi));
    }
    A[(long long)(p + j) * N + p + i] = c128{-gr, i == j ? 0.0 : -gi};
  }
  if (t < 16 * PB) {                     // digits: rows of W as left rows, rows of W^H as right rows
    const int w = t >> 8, r = (t >> 3) & 31, part = (t >> 2) & 1, qr = t & 3;
    double x[8];
#pragma unroll
    for (int c = 0; c < 8; ++c) {
      const double2 z = w == 0 ? buf[r][8 * qr + c] : buf[8 * qr + c][r];
      x[c] = part ? (w == 0 ? z.y : -z.y) : z.x;
    }
    int e;
    const int f = row_field(x, e);
    if ((t & 7) == 0) (w == 0 ? eW : eR)[b * PB + r] = e;
    long long y[8];
#pragma unroll
    for (int c = 0; c < 8; ++c) y[c] = to_digits(x[c], f);
    if (w == 0) {
      const int m1 = (r >> 4) * 32 + (r & 15), m2 = m1 + 16;
      uint8_t* g = wdig + (long long)b * ND * W_PLANE;
      each_digit<0>(y, [&](int d, uint4 q) {
        *reinterpret_cast<uint4*>(g + d * W_PLANE + m1 * ROWB + (part * 4 + qr) * 16) = q;
        *reinterpret_cast<uint4*>(g + d * W_PLANE + m2 * ROWB + ((part ^ 1) * 4 + qr) * 16) = part ? q : neg8(q);
      });
    } else {
      uint8_t* g = rdig + (long long)b * ND * R_PLANE;
      each_digit<0>(y, [&](int d, uint4 q) {
        *reinterpret_cast<uint4*>(g + d * R_PLANE + r * ROWB + (part * 4 + qr) * 16) = q;
      });
    }
  }
}

// ---- shared pieces of the two product kernels ---------------------------------------------------

struct InvMaps {
  CUtensorMap yb, ya, w, r;
};

// 256 v_o + v_(o+1) of 16 columns. SMALL: |v| <= 2^22 (orders 0-3: at most 4 pairs x 2^20), converted by
// an exact addition of 1.5 2^23 whose bits hold the integer (the general conversion runs at a quarter rate)
template <bool SMALL, int STRIDE> __device__ __forceinline__ void ld_pair(uint32_t taddr, int (&v)[16]) {
  uint32_t r[16], s[16];
  tmem_ld16_nowait(taddr, r);
  tmem_ld16_nowait(taddr + STRIDE, s);
  tmem_wait_ld();
#pragma unroll
  for (int j = 0; j < 16; ++j) {
    const float x = __uint_as_float(r[j]), y = __uint_as_float(s[j]);
    if constexpr (SMALL)
      v[j] = __float_as_int(x + 12582912.0f) * 256 + __float_as_int(y + 12582912.0f) - 0x4b400000 * 257u;
    else
      v[j] = __float2int_rn(x) * 256 + __float2int_rn(y);
  }
}
// orders 0-3 of 16 columns (orders STRIDE columns apart): S = sum_o v_o 256^(3 - o)  (|S| < 2^45)
template <int STRIDE> __device__ __forceinline__ void high_orders(uint32_t tl, long long (&S)[16]) {
  int v[16], w[16];
  ld_pair<true, STRIDE>(tl, v);
  ld_pair<true, STRIDE>(tl + 2 * STRIDE, w);
#pragma unroll
  for (int j = 0; j < 16; ++j) S[j] = (long long)v[j] * 65536 + w[j];
}
// and orders 4-6: S <- (S 2^24 + sum_o v_o 256^(6 - o)) / 64  (|S| < 2^63)
template <int STRIDE> __device__ __forceinline__ void low_orders(uint32_t tl, long long (&S)[16]) {
  int v[16];
  uint32_t r[16];
  tmem_ld16_nowait(tl + 6 * STRIDE, r);
  ld_pair<false, STRIDE>(tl + 4 * STRIDE, v);
#pragma unroll
  for (int j = 0; j < 16; ++j)
    S[j] = (S[j] << 18) + (((long long)v[j] * 256 + __float2int_rn(__uint_as_float(r[j]))) >> 6);
}
// A lane of the upper half holds Im, of the lower half Re of the same row: for the column pair
// (2u, 2u + 1) the lower half keeps column 2u and the upper half 2u + 1, each with both parts
// (integers below 2^63, rounded to FP64 once)
__device__ __forceinline__ double2 trade(const long long s0, const long long s1, int h) {
  const long long got = __shfl_xor_sync(0xffffffffu, h ? s0 : s1, 16);
  return make_double2((double)(h ? got : s0), (double)(h ? s1 : got));
}
constexpr int E_SHIFT = 110 - 48 - 6;    // value = S 2^(e_left + e_right - E_SHIFT)

// ---- Y_i = B_iP W^H and its digits, 32 rows per CTA ---------------------------------------------
//
// The panel rows are read and cut straight into the right operand in shared memory, W is the left
// one (conj(Y_i) = W B_iP^H, so only W needs stacked rows), and the product's rows are cut again. The
// steps of a CTA follow one another, so two CTAs share an SM (110 KB and 256 TMEM columns each).
constexpr int YR = 32;                                       // rows per CTA
constexpr int Y_THREADS = 8 * YR;
constexpr int Y_PIECE = YR * ROWB;
constexpr int Y_OFF_B = ND * W_PLANE + W_PLANE;              // (the MMA reads 128 rows of a 64-row digit)
constexpr int Y_OFF_Z = Y_OFF_B + ND * Y_PIECE;
constexpr int Y_OFF_E = Y_OFF_Z + PB * (YR + 1) * 16;
constexpr int Y_OFF_BAR = Y_OFF_E + YR * 4;
constexpr int Y_SMEM = Y_OFF_BAR + 32 + 1024;
static_assert(2 * (Y_SMEM + 1024) <= 233472, "two blocks per SM");

__global__ void __launch_bounds__(Y_THREADS, 2) k_inv_y(const __grid_constant__ InvMaps maps, int N, int Nr, int p, int batch,
                                                        const c128* __restrict__ Aall, long long stride,
                                                        uint8_t* __restrict__ yb, uint8_t* __restrict__ ya,
                                                        const int* __restrict__ eW, int* __restrict__ eY,
                                                        int* __restrict__ status) {
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  double2* Z = reinterpret_cast<double2*>(smem + Y_OFF_Z);     // [32 panel columns][33 rows], then [32][32]
  int* eC = reinterpret_cast<int*>(smem + Y_OFF_E);
  uint64_t* wfull = reinterpret_cast<uint64_t*>(smem + Y_OFF_BAR);
  uint64_t* dfull = wfull + 1;
  uint32_t* tmem_p = reinterpret_cast<uint32_t*>(wfull + 2);
  const int t = threadIdx.x, warp = t / 32, lane = t % 32;
  const int blk = blockIdx.x / batch, b = blockIdx.x % batch;
  const int r0 = blk * YR, pw = min(PB, N - p);
  const c128* A = Aall + b * stride;
  if (t == 0) {
    mbar_init(wfull, 1);
    mbar_init(dfull, 1);
    fence_mbar_init();
    mbar_arrive_expect_tx(wfull, ND * W_PLANE);
    for (int d = 0; d < ND; ++d) tma_load_2d(smem + d * W_PLANE, &maps.w, wfull, 0, (b * ND + d) * 2 * PB);
  }
  if (warp == 1) {
    tmem_alloc(tmem_p, 256);
    tmem_relinquish();
  }
  for (int e = t; e < YR * PB; e += Y_THREADS) {
    // behind the pivot the panel runs along the rows, before it along the panel columns
    int r = e % YR, c = e / YR;
    if (r0 < p) {
      r = e / PB;
      c = e % PB;
    }
    const int i = r0 + r;
    double2 z = make_double2(0.0, 0.0);       // rows of P and beyond N: no update
    if (i < N && c < pw) {
      if (i >= p + PB) {
        const c128 a = A[(long long)(p + c) * N + i];
        z = make_double2(a.re, a.im);
      } else if (i < p) {
        const c128 a = A[(long long)i * N + p + c];
        z = make_double2(a.re, -a.im);
      }
    }
    Z[c * (YR + 1) + r] = z;
  }
  __syncthreads();
  const int r = t >> 3, part = (t >> 2) & 1, qr = t & 3;      // 8 threads per row: Re / Im, a quarter of the columns
  {
    double x[8];
#pragma unroll
    for (int c = 0; c < 8; ++c) {
      const double2 z = Z[(8 * qr + c) * (YR + 1) + r];
      x[c] = part ? z.y : z.x;
    }
    int e;
    const int f = row_field(x, e);
    if ((t & 7) == 0) eC[r] = e;
    long long y[8];
#pragma unroll
    for (int c = 0; c < 8; ++c) y[c] = to_digits(x[c], f);
    each_digit<0>(y, [&](int d, uint4 q) {
      *reinterpret_cast<uint4*>(smem + Y_OFF_B + d * Y_PIECE + swz(r, part * 4 + qr)) = q;
    });
    fence_proxy_async();
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *tmem_p;
  if (t == 0) {
    const uint32_t idesc = (1u << 4) | ((uint32_t)(YR >> 3) << 17) | ((uint32_t)(128 >> 4) << 24);
    const uint32_t abase = smem_u32(smem), bbase = abase + Y_OFF_B;
    if (mbar_wait(wfull, 0, status)) {
      tc_fence_after();
      for (int o = 0; o < ND; ++o)
        for (int d1 = 0; d1 <= o; ++d1) {
          const uint64_t dA = sdesc(abase + d1 * W_PLANE), dB = sdesc(bbase + (o - d1) * Y_PIECE);
#pragma unroll
          for (int kk = 0; kk < 4; ++kk)
            mma<false>(tmem + o * YR, dA + 2 * kk, dB + 2 * kk, idesc, (d1 == 0 && kk == 0) ? 0u : 1u);
        }
    }
    mma_commit(dfull);
  }
  __syncwarp();
  const bool ok = __all_sync(0xffffffffu, mbar_wait(dfull, 0, status));
  tc_fence_after();
  const int quad = warp & 3, cg = warp >> 2, h = lane >> 4;
  if (ok && quad < 2) {
    const uint32_t tl = tmem + ((uint32_t)(quad * 32) << 16) + cg * 16;
    const int pc = quad * 16 + (lane & 15);
    long long S[16];
    high_orders<YR>(tl, S);
    low_orders<YR>(tl, S);
    const int ew = eW[b * PB + pc] - E_SHIFT;
#pragma unroll
    for (int u = 0; u < 8; ++u) {
      const int c = cg * 16 + 2 * u + h;                       // row of the block
      const double2 z = trade(S[2 * u], S[2 * u + 1], h);
      const double f = pow2(ew + eC[c]);
      Z[c * PB + pc] = make_double2(f * z.x, -f * z.y);
    }
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  if (warp == 1) tmem_dealloc(tmem, 256);
  double x[8];
#pragma unroll
  for (int c = 0; c < 8; ++c) {
    const double2 z = Z[r * PB + 8 * qr + c];
    x[c] = part ? z.y : z.x;
  }
  int e;
  const int f = row_field(x, e);
  if ((t & 7) == 0) eY[(long long)b * Nr + r0 + r] = e;
  long long y[8];
#pragma unroll
  for (int c = 0; c < 8; ++c) y[c] = to_digits(x[c], f);
  const int r64 = r0 % TM + r, m1 = (r64 >> 4) * 32 + (r64 & 15), m2 = m1 + 16;
  const int nblk = Nr / TM;
  uint8_t* ob = yb + ((long long)b * ND * Nr + r0 + r) * ROWB + (part * 4 + qr) * 16;
  uint8_t* oa = ya + ((long long)b * ND * nblk + r0 / TM) * A_PIECE;
  each_digit<0>(y, [&](int d, uint4 q) {
    *reinterpret_cast<uint4*>(ob + (long long)d * Nr * ROWB) = q;
    uint8_t* o = oa + (long long)d * nblk * A_PIECE;
    *reinterpret_cast<uint4*>(o + m1 * ROWB + (part * 4 + qr) * 16) = q;
    *reinterpret_cast<uint4*>(o + m2 * ROWB + ((part ^ 1) * 4 + qr) * 16) = part ? q : neg8(q);
  });
}

// ---- the update of one row block ----------------------------------------------------------------
//
// One CTA per (matrix, block of 64 rows): tile 0 is the new panel B_iP = Y_i W, tiles 1 .. i + 1
// subtract Y_i Y_j^H from the column blocks j <= i. The left operand stays for the whole row block, the
// right one streams through a ring of two tiles. Left rows are stacked as 16 Re rows, 16 Im rows, ..., so
// a warp of the epilogue (32 TMEM lanes) holds both parts of its 16 rows and trades them by shuffles;
// rows of B are contiguous, so each half warp then updates 256 contiguous bytes.
// Roles: warp 0 TMA, warp 1 MMA, warps 2-17 epilogue. TMEM: order o at column 64 o; orders 0-3 and
// 4-6 are handed over separately so that the next tile's first orders run under the drain.
__global__ void __launch_bounds__(UPD_THREADS, 1) k_inv_update(const __grid_constant__ InvMaps maps, int N, int Nr, int p,
                                                               int batch, c128* __restrict__ Aall, long long stride,
                                                               const int* __restrict__ eY, const int* __restrict__ eR,
                                                               int* __restrict__ status) {
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  uint64_t* bars = reinterpret_cast<uint64_t*>(smem + OFF_BAR);
  uint64_t* bfull = bars;
  uint64_t* bempty = bars + SLOTS;
  uint64_t* afull = bars + 2 * SLOTS;    // [7] digits of the left operand
  uint64_t* dfull = afull + ND;          // [2] orders 0-3, orders 4-6 of a tile ready
  uint64_t* dempty = dfull + 2;          // [2] and drained
  uint64_t* done = dfull + 4;
  uint32_t* tmem_p = reinterpret_cast<uint32_t*>(dfull + 5);
  const int warp = threadIdx.x / 32, lane = threadIdx.x % 32;
  const int nblk = Nr / TM;
  const int bi = nblk - 1 - blockIdx.x / batch;                // longest row blocks first
  const int b = blockIdx.x % batch;
  if (threadIdx.x == 0) {
    for (int s = 0; s < SLOTS; ++s) {
      mbar_init(&bfull[s], 1);
      mbar_init(&bempty[s], 1);
    }
    for (int d = 0; d < ND; ++d) mbar_init(&afull[d], 1);
    for (int h = 0; h < 2; ++h) {
      mbar_init(&dfull[h], 1);
      mbar_init(&dempty[h], EPI_WARPS);
    }
    mbar_init(done, 1);
    fence_mbar_init();
  }
  if (warp == 1) {
    tmem_alloc(tmem_p, 512);
    tmem_relinquish();
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *tmem_p;
  const int ntile = bi + 2;

  if (warp == 0) {
    if (lane == 0) {
      int s = 0;
      uint32_t ph = 0;
      bool ok = true;
      for (int tt = 0; tt < ntile && ok; ++tt)
        for (int d = 0; d < ND; ++d) {
          if (tt == 0) {
            mbar_arrive_expect_tx(&afull[d], A_PIECE);
            tma_load_2d(smem + d * A_PIECE, &maps.ya, &afull[d], 0, ((b * ND + d) * nblk + bi) * 128);
          }
          if (!mbar_wait(&bempty[s], ph ^ 1u, status)) { ok = false; break; }
          uint8_t* dst = smem + OFF_B + s * B_PIECE;
          mbar_arrive_expect_tx(&bfull[s], tt == 0 ? R_PLANE : B_PIECE);
          if (tt == 0) tma_load_2d(dst, &maps.r, &bfull[s], 0, (b * ND + d) * PB);   // (columns 32-63 unused)
          else tma_load_2d(dst, &maps.yb, &bfull[s], 0, (b * ND + d) * Nr + (tt - 1) * TM);
          if (++s == SLOTS) { s = 0; ph ^= 1u; }
        }
    }
  } else if (warp == 1) {
    if (lane == 0) {
      const uint32_t idesc = (1u << 4) | ((uint32_t)(TM >> 3) << 17) | ((uint32_t)(128 >> 4) << 24);
      const uint32_t abase = smem_u32(smem), bbase = abase + OFF_B;
      bool ok = true;
      for (int tt = 0; tt < ntile && ok; ++tt) {
        const uint32_t bt = bbase + (tt & 1) * ND * B_PIECE;       // the ring holds two tiles
        const uint32_t ph = (tt >> 1) & 1;
        for (int o = 0; o < ND && ok; ++o) {
          if ((o == 0 || o == 4) && tt > 0 && !mbar_wait(&dempty[o == 4], (tt - 1) & 1, status)) { ok = false; break; }
          if (tt == 0 && !mbar_wait(&afull[o], 0, status)) { ok = false; break; }
          if (!mbar_wait(&bfull[(tt & 1) * ND + o], ph, status)) { ok = false; break; }
          tc_fence_after();
          for (int d1 = 0; d1 <= o; ++d1) {
            const uint64_t dA = sdesc(abase + d1 * A_PIECE), dB = sdesc(bt + (o - d1) * B_PIECE);
#pragma unroll
            for (int kk = 0; kk < 4; ++kk)
              mma<false>(tmem + o * TM, dA + 2 * kk, dB + 2 * kk, idesc, (d1 == 0 && kk == 0) ? 0u : 1u);
            if (o == ND - 1) mma_commit(&bempty[(tt & 1) * ND + o - d1]);   // the last use of this digit of the tile
          }
          if (o == 3) mma_commit(&dfull[0]);
          if (o == ND - 1) mma_commit(&dfull[1]);
        }
      }
      mma_commit(done);
      mbar_wait(done, 0, status);
    }
  } else {
    const int quad = warp & 3, cg = (warp - 2) >> 2;
    const int h = lane >> 4, row = bi * TM + quad * 16 + (lane & 15);
    const uint32_t tl = tmem + ((uint32_t)(quad * 32) << 16) + cg * 16;
    c128* A = Aall + b * stride;
    const int pw = min(PB, N - p);
    const bool rok = row < N && !(row >= p && row < p + PB);
    const int erow = eY[(long long)b * Nr + row] - E_SHIFT;
    const bool full_rows = bi * TM + quad * 16 + 16 <= p || bi * TM + quad * 16 >= p + PB;   // none of the warp's in P
    for (int tt = 0; tt < ntile; ++tt) {
      const bool panel = tt == 0;
      const bool active = !panel || cg < 2;           // the panel has 32 columns
      // the elements this thread updates: columns c0 + 2 u + h, u < 8
      const int c0 = panel ? cg * 16 : (tt - 1) * TM + cg * 16;
      c128* at = A + (long long)(c0 + h) * N + row;                // and every second column of B from there
      const int* et = panel ? eR + b * PB : eY + (long long)b * Nr;
      // whole tiles left of the diagonal and off the pivot block take every element
      unsigned live = 0;
      if (!panel && bi * TM + TM <= N && c0 + 16 <= bi * TM && (c0 >= p + PB || c0 + 16 <= p) && full_rows) {
        live = 0xffu;
      } else if (rok) {
#pragma unroll
        for (int u = 0; u < 8; ++u) {
          const int c = c0 + 2 * u + h;
          live |= (panel ? c < pw : c <= row && !(c >= p && c < p + PB)) ? 1u << u : 0u;
        }
      }
      c128 old[4];
      long long S[16];
      if (!__all_sync(0xffffffffu, mbar_wait(&dfull[0], tt & 1, status))) break;
      tc_fence_after();
      if (active) high_orders<TM>(tl, S);
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(&dempty[0]);
      if (!panel)
#pragma unroll
        for (int u = 0; u < 4; ++u)
          if (live & (1u << u)) old[u] = at[2LL * u * N];
      if (!__all_sync(0xffffffffu, mbar_wait(&dfull[1], tt & 1, status))) break;
      tc_fence_after();
      if (active) low_orders<TM>(tl, S);
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(&dempty[1]);
      if (active) {
#pragma unroll
        for (int g = 0; g < 2; ++g) {
#pragma unroll
          for (int v = 0; v < 4; ++v) {
            const int u = 4 * g + v, c = c0 + 2 * u + h;
            const double2 z = trade(S[2 * u], S[2 * u + 1], h);
            const double f = pow2(erow + et[c]);
            if (live & (1u << u)) {
              if (!panel) at[2LL * u * N] = c128{fma(-f, z.x, old[v].re), fma(-f, z.y, old[v].im)};
              else if (row >= p) A[(long long)(p + c) * N + row] = c128{f * z.x, f * z.y};
              else A[(long long)row * N + p + c] = c128{f * z.x, -f * z.y};
            }
            if (g == 0 && !panel && (live & (16u << v))) old[v] = at[2LL * (u + 4) * N];
          }
        }
      }
    }
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  if (warp == 1) tmem_dealloc(tmem, 512);
}

// A := -B - I in full from the kept triangle, the scales of A undone
__global__ void k_inv_finish(int N, c128* __restrict__ Aall, long long stride, const int* __restrict__ scall) {
  __shared__ c128 tt[32][33];
  if (blockIdx.x < blockIdx.y) return;
  c128* A = Aall + blockIdx.z * stride;
  const int* sc = scall + (long long)blockIdx.z * N;
  const int j0 = blockIdx.y * 32, i0 = blockIdx.x * 32;     // memory rows j, columns i >= j
  for (int r = threadIdx.y; r < 32; r += blockDim.y) {
    const int j = j0 + r, i = i0 + threadIdx.x;
    if (j < N && i < N && i >= j) {
      c128 v = A[(long long)j * N + i];
      const double fj = pow2(sc[j]), fi = pow2(sc[i]);
      v = c128{v.re * fj * fi, v.im * fj * fi};
      const c128 o = i == j ? c128{-v.re - 1.0, 0.0} : c128{-v.re, -v.im};
      A[(long long)j * N + i] = o;
      tt[r][threadIdx.x] = o;
    }
  }
  __syncthreads();
  for (int r = threadIdx.y; r < 32; r += blockDim.y) {
    const int i = i0 + r, j = j0 + threadIdx.x;
    if (j < N && i < N && i > j) {
      const c128 v = tt[threadIdx.x][r];
      A[(long long)i * N + j] = c128{v.re, -v.im};
    }
  }
}

}  // namespace

size_t inv_work_bytes(int N, int batch) { return (size_t)inv_layout(N, batch).bytes; }

gw_status launch_inv_minus_I(int N, c128* A, int batch, long long stride, void* work, int* status, cudaStream_t st,
                             std::string& err) {
  const InvLayout l = inv_layout(N, batch);
  uint8_t* w = static_cast<uint8_t*>(work);
  const int Nr = padded(N), nblk = Nr / TM;
  int* eY = reinterpret_cast<int*>(w + l.ey);
  int* eW = reinterpret_cast<int*>(w + l.ew);
  int* eR = reinterpret_cast<int*>(w + l.er);
  InvMaps maps;
  if (!tc_map_16bit(&maps.yb, w + l.yb, ROWB / 2, (long long)batch * ND * Nr, TM, err) ||
      !tc_map_16bit(&maps.ya, w + l.ya, ROWB / 2, (long long)batch * ND * 2 * Nr, 128, err) ||
      !tc_map_16bit(&maps.w, w + l.w, ROWB / 2, (long long)batch * ND * 2 * PB, 2 * PB, err) ||
      !tc_map_16bit(&maps.r, w + l.r, ROWB / 2, (long long)batch * ND * PB, PB, err))
    return GW_ERR_CUDA;
  cudaFuncSetAttribute(k_inv_y, cudaFuncAttributeMaxDynamicSharedMemorySize, Y_SMEM);
  cudaFuncSetAttribute(k_inv_update, cudaFuncAttributeMaxDynamicSharedMemorySize, UPD_SMEM);
  int* sc = reinterpret_cast<int*>(w + l.sc);
  const int nt = (N + 31) / 32;
  ++g_launch_count, k_inv_exps<<<dim3((N + 127) / 128, batch), 128, 0, st>>>(N, A, stride, sc);
  ++g_launch_count, k_inv_scale<<<dim3(nt, nt, batch), dim3(32, 8), 0, st>>>(N, A, stride, sc);
  for (int p = 0; p < N; p += PB) {
    ++g_launch_count, k_inv_pivot<<<batch, PIV_THREADS, 0, st>>>(N, p, A, stride, w + l.w, w + l.r, eW, eR, status);
    if (N <= PB) break;
    ++g_launch_count, k_inv_y<<<Nr / YR * batch, Y_THREADS, Y_SMEM, st>>>(maps, N, Nr, p, batch, A, stride, w + l.yb,
                                                                      w + l.ya, eW, eY, status);
    ++g_launch_count, k_inv_update<<<nblk * batch, UPD_THREADS, UPD_SMEM, st>>>(maps, N, Nr, p, batch, A, stride, eY, eR,
                                                                               status);
  }
  ++g_launch_count, k_inv_finish<<<dim3(nt, nt, batch), dim3(32, 8), 0, st>>>(N, A, stride, sc);
  return GW_OK;
}

}  // namespace gw

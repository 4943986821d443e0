// Step (a): LRI triple coefficients -> band-pair coefficients M^mu_{ab}(k, q).
//
// Eq. (AO_triple_split2): C~^mu_{ij}(k+q,k) = C~^{mu(0)}_{j(0),i(-k-q)} + C~^{mu(0)}_{i(0),j(k)},
// with C~_{i(0),j(R)}^{mu(0)} nonzero only for mu on the atom of i, and the
// Fourier sums of Eqs. (expan_coeff_FT1/2). Inserting this into Eq. (AO_MO_transform)
// and contracting the NAO index that is not on mu's atom first gives the
// half-transformed coefficients (computed once per k at plan time)
//     T1^mu_{ib}(k) = sum_R e^{i k.R} sum_j C~^{mu(0)}_{i(0),j(R)} c_{jb}(k),   i on atom(mu)
// and, because the stored C~(R) are real (real NAOs and ABFs), the second
// sector's transform is conj(T1). Then per (k, q):
//     M^mu_{ab}(k,q) = sum_{j in A(mu)} c_{jb}(k) conj(T1^mu_{ja}(k+q))
//                    + sum_{i in A(mu)} conj(c_{ia}(k+q)) T1^mu_{ib}(k),
// which is Eq. (AO_MO_transform) exactly, with n_b(A) instead of N_b terms per sum.
#include "gw_internal.h"
#include <cuda_bf16.h>

namespace gw {

template <typename T>
__global__ void k_lri_halfT(const __grid_constant__ LriGeom g, const double* __restrict__ ctil,
                            const c128* __restrict__ evec, cplx<T>* __restrict__ T1, int A) {
  const int nb_A = g.atom_nb[A], nx_A = g.atom_nx[A];
  const long long total = (long long)g.NK * nx_A * nb_A * g.NBd;
  for (long long idx = blockIdx.x * (long long)blockDim.x + threadIdx.x; idx < total;
       idx += (long long)gridDim.x * blockDim.x) {
    int b = (int)(idx % g.NBd);
    long long t = idx / g.NBd;
    int i = (int)(t % nb_A);
    t /= nb_A;
    int mu = (int)(t % nx_A);
    int k = (int)(t / nx_A);
    int k3 = k % g.nk[2], k2 = (k / g.nk[2]) % g.nk[1], k1 = k / (g.nk[1] * g.nk[2]);
    double acc_re = 0.0, acc_im = 0.0;
    const c128* ck = evec + (long long)k * g.NB * g.NBd;
    for (int r = 0; r < g.nR; ++r) {
      // phase e^{2 pi i k.R}, k = mesh point + offset in fractional coordinates
      double ph = 2.0 * (((double)k1 / g.nk[0] + g.koff[0]) * g.R[r][0] + ((double)k2 / g.nk[1] + g.koff[1]) * g.R[r][1] +
                         ((double)k3 / g.nk[2] + g.koff[2]) * g.R[r][2]);
      double s, c;
      sincospi(ph, &s, &c);
      const double* crow = ctil + g.ctil_off[A] + (((long long)r * nx_A + mu) * nb_A + i) * g.NB;
      double sr = 0.0, si = 0.0;
      for (int j = 0; j < g.NB; ++j) {
        c128 cj = ck[(long long)j * g.NBd + b];
        sr = fma(crow[j], cj.re, sr);
        si = fma(crow[j], cj.im, si);
      }
      acc_re += c * sr - s * si;
      acc_im += c * si + s * sr;
    }
    T1[g.t_off[A] + idx] = cplx<T>{(T)acc_re, (T)acc_im};
  }
}

template <typename T>
void launch_lri_halfT(const LriGeom& g, const double* ctil, const c128* evec, const cplx<T>* /*evec_t*/, cplx<T>* T1,
                      cudaStream_t st) {
  for (int A = 0; A < g.n_atoms; ++A) {
    long long total = (long long)g.NK * g.atom_nx[A] * g.atom_nb[A] * g.NBd;
    int blocks = (int)std::min<long long>((total + 255) / 256, 152LL * 64);
    ++::gw::g_launch_count, k_lri_halfT<T><<<blocks, 256, 0, st>>>(g, ctil, evec, T1, A);
  }
}
template void launch_lri_halfT<double>(const LriGeom&, const double*, const c128*, const c128*, c128*, cudaStream_t);

// fp32 (split-precision plans): the same sums with the Fourier sum over the lattice vectors taken first,
//   C(k)[(mu,i)][j] = sum_R e^{2 pi i k.R} C~(R)[(mu,i)][j]  (to 2^-46, rounded once),
//   T1[k] = C(k) . c(k), batched over as many k as the staging holds.
// One complex product per k instead of one per k and lattice vector onto T1: 64 k, 2 atoms of 200 ABFs and 39
// functions, 78 bands, 7 lattice vectors 8.8 -> 2.0 ms.
namespace {

// Ck[k - k0][e] for e < n (one atom's [(mu,i)][j]), LF_K consecutive k per block. The sums run in pairs of floats
// (products and additions with their rounding errors, 2^-46 of the terms): on the FP64 units, 2 multiply-adds
// per clock and SM, they took 2.7 ms of a plan of 64 k, 2 atoms, 200 ABFs, 39 functions, 78 bands, 7 vectors; 0.93 ms now.
constexpr int LF_K = 8;
struct Pair32 {
  float h = 0.f, l = 0.f;
  __device__ __forceinline__ void add(float xh, float xl, float ch, float cl) {   // += (xh + xl) (ch + cl)
    const float p = __fmul_rn(xh, ch);
    const float e = fmaf(xh, cl, fmaf(xl, ch, fmaf(xh, ch, -p)));
    const float s = __fadd_rn(h, p), b = __fsub_rn(s, h);
    l += __fadd_rn(__fsub_rn(h, __fsub_rn(s, b)), __fsub_rn(p, b)) + e;
    h = s;
  }
};
__global__ void __launch_bounds__(256) k_lri_fourier(const __grid_constant__ LriGeom g, int k0, int nk, long long n,
                                                     const double* __restrict__ ctil, c64* __restrict__ Ck) {
  __shared__ float4 ph[64][LF_K];      // cos and sin, each as a pair
  const int kb = blockIdx.y * LF_K;
  for (int i = threadIdx.x; i < g.nR * LF_K; i += blockDim.x) {
    const int r = i / LF_K, k = k0 + min(kb + i % LF_K, nk - 1);
    const int k3 = k % g.nk[2], k2 = (k / g.nk[2]) % g.nk[1], k1 = k / (g.nk[1] * g.nk[2]);
    const double x = 2.0 * (((double)k1 / g.nk[0] + g.koff[0]) * g.R[r][0] +
                            ((double)k2 / g.nk[1] + g.koff[1]) * g.R[r][1] +
                            ((double)k3 / g.nk[2] + g.koff[2]) * g.R[r][2]);
    double s, c;
    sincospi(x, &s, &c);
    const float ch = (float)c, sh = (float)s;
    ph[r][i % LF_K] = make_float4(ch, (float)(c - ch), sh, (float)(s - sh));
  }
  __syncthreads();
  for (long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x; e < n; e += (long long)gridDim.x * blockDim.x) {
    Pair32 re[LF_K], im[LF_K];
    for (int r = 0; r < g.nR; ++r) {
      const double x = ctil[r * n + e];
      const float xh = (float)x, xl = (float)(x - xh);
#pragma unroll
      for (int k = 0; k < LF_K; ++k) {
        const float4 f = ph[r][k];
        re[k].add(xh, xl, f.x, f.y);
        im[k].add(xh, xl, f.z, f.w);
      }
    }
#pragma unroll
    for (int k = 0; k < LF_K; ++k)
      if (kb + k < nk) Ck[(kb + k) * n + e] = c64{re[k].h + re[k].l, im[k].h + im[k].l};
  }
}

}  // namespace

template <>
void launch_lri_halfT<float>(const LriGeom& g, const double* ctil, const c128* evec, const c64* evec_t, c64* T1,
                             cudaStream_t st) {
  const long long per_k = (long long)g.NB * g.NBd;
  long long amax = 0;
  for (int A = 0; A < g.n_atoms; ++A) amax = std::max(amax, (long long)g.atom_nx[A] * g.atom_nb[A] * g.NB);
  const int kc = (int)std::max<long long>(1, std::min<long long>(g.NK, (256LL << 20) / (amax * (long long)sizeof(c64))));
  c64* Ck = nullptr;
  ++::gw::g_alloc_count;
  if (cudaMallocAsync(&Ck, sizeof(c64) * amax * kc, st) != cudaSuccess) {
    // fall back to the direct kernel (same sums, FP64 arithmetic) when the staging does not fit
    cudaGetLastError();
    for (int A = 0; A < g.n_atoms; ++A) {
      long long total = (long long)g.NK * g.atom_nx[A] * g.atom_nb[A] * g.NBd;
      int blocks = (int)std::min<long long>((total + 255) / 256, 152LL * 64);
      ++::gw::g_launch_count, k_lri_halfT<float><<<blocks, 256, 0, st>>>(g, ctil, evec, T1, A);
    }
    return;
  }
  for (int A = 0; A < g.n_atoms; ++A) {
    const long long rows = (long long)g.atom_nx[A] * g.atom_nb[A], n = rows * g.NB;
    for (int k0 = 0; k0 < g.NK; k0 += kc) {
      const int nk = std::min(kc, g.NK - k0);
      const dim3 grid((unsigned)std::min<long long>((n + 255) / 256, 1024), (nk + LF_K - 1) / LF_K);
      ++::gw::g_launch_count, k_lri_fourier<<<grid, 256, 0, st>>>(g, k0, nk, n, ctil + g.ctil_off[A], Ck);
      launch_zgemm<float>((int)rows, g.NBd, g.NB, c64{1, 0}, Ck, g.NB, n, OP_N, evec_t + k0 * per_k, g.NBd, per_k, OP_N,
                          c64{0, 0}, T1 + g.t_off[A] + k0 * rows * g.NBd, g.NBd, rows * g.NBd, nk, st);
    }
  }
  cudaFreeAsync(Ck, st);
}

// ---------------------------------------------------------------------------------------------
// M generation. One block per (row-k kk, block of MU ABFs); threads over (a, b) pairs.
// ---------------------------------------------------------------------------------------------
constexpr int MGEN_MU = 8;

__device__ __forceinline__ int aux_atom_of(const LriGeom& g, int mu) {
  int A = 0;
  while (A + 1 < g.n_atoms && mu >= g.atom_x0[A + 1]) ++A;
  return A;
}

template <typename T, typename Store>
__device__ __forceinline__ void mgen_body(const LriGeom& g, const cplx<T>* __restrict__ T1,
                                          const c128* __restrict__ evec, int q, int kk0, int mode, int a0, int na,
                                          int b0, int nb, Store store) {
  const int kk = blockIdx.x;
  int ktgt = g.ktab ? g.ktab[kk0 + kk] : kk0 + kk;
  int k3 = ktgt % g.nk[2], k2 = (ktgt / g.nk[2]) % g.nk[1], k1 = ktgt / (g.nk[1] * g.nk[2]);
  int q3 = q % g.nk[2], q2 = (q / g.nk[2]) % g.nk[1], q1 = q / (g.nk[1] * g.nk[2]);
  int kp;  // k' (b bands live here), k'+q (a bands live here)
  if (mode == MAP_K_IS_KK) {
    kp = ktgt;
  } else {
    kp = (((k1 - q1 + g.nk[0]) % g.nk[0]) * g.nk[1] + ((k2 - q2 + g.nk[1]) % g.nk[1])) * g.nk[2] +
         ((k3 - q3 + g.nk[2]) % g.nk[2]);
  }
  int p3 = kp % g.nk[2], p2 = (kp / g.nk[2]) % g.nk[1], p1 = kp / (g.nk[1] * g.nk[2]);
  int kpq = (((p1 + q1) % g.nk[0]) * g.nk[1] + ((p2 + q2) % g.nk[1])) * g.nk[2] + ((p3 + q3) % g.nk[2]);
  const c128* ck = evec + (long long)kp * g.NB * g.NBd;    // c(k')
  const c128* ckq = evec + (long long)kpq * g.NB * g.NBd;  // c(k'+q)
  const int mu_begin = blockIdx.y * MGEN_MU;
  const int mu_end = min(mu_begin + MGEN_MU, g.N);
  const int npair = na * nb;
  // (ABF, pair) flattened over the block's threads so that no lanes idle on a ragged pair count
  for (int idx = threadIdx.x; idx < (mu_end - mu_begin) * npair; idx += blockDim.x) {
    const int mu = mu_begin + idx / npair;
    const int p = idx % npair;
    const int A = aux_atom_of(g, mu);
    const int nbA = g.atom_nb[A], b0A = g.atom_b0[A];
    const int mul = mu - g.atom_x0[A];
    const cplx<T>* t1k = T1 + g.t_off[A] + (((long long)kp * g.atom_nx[A] + mul) * nbA) * g.NBd;
    const cplx<T>* t1kq = T1 + g.t_off[A] + (((long long)kpq * g.atom_nx[A] + mul) * nbA) * g.NBd;
    {
      const int a = a0 + p / nb, b = b0 + p % nb;
      T sr = 0, si = 0;
      for (int j = 0; j < nbA; ++j) {
        // c_{jb}(k') conj(T1^mu_{ja}(k'+q))
        c128 cjb = ck[(long long)(b0A + j) * g.NBd + b];
        cplx<T> t = t1kq[(long long)j * g.NBd + a];
        T cr = (T)cjb.re, ci = (T)cjb.im;
        sr += cr * t.re + ci * t.im;
        si += ci * t.re - cr * t.im;
        // conj(c_{ja}(k'+q)) T1^mu_{jb}(k')
        c128 cja = ckq[(long long)(b0A + j) * g.NBd + a];
        cplx<T> u = t1k[(long long)j * g.NBd + b];
        T dr = (T)cja.re, di = (T)cja.im;
        sr += dr * u.re + di * u.im;
        si += dr * u.im - di * u.re;
      }
      long long r = ((long long)kk * na + (p / nb)) * nb + (p % nb);
      store(r, mu, sr, si);
    }
  }
}

template <typename T>
__global__ void k_mgen(const __grid_constant__ LriGeom g, const cplx<T>* __restrict__ T1, const c128* __restrict__ evec, int q, int kk0, int mode,
                       int a0, int na, int b0, int nb, cplx<T>* __restrict__ out, long long s_r, long long s_mu) {
  mgen_body<T>(g, T1, evec, q, kk0, mode, a0, na, b0, nb, [&](long long r, int mu, T re, T im) {
    out[r * s_r + (long long)mu * s_mu] = cplx<T>{re, im};
  });
}

template <>
void launch_mgen<double>(const LriGeom& g, const c128* T1, const c128* evec, int q, int kk0, int nkk, MapMode mode, int a0,
                         int na, int b0, int nb, c128* out, long long s_r, long long s_mu, cudaStream_t st,
                         unsigned* /*absmax*/) {
  dim3 grid(nkk, (g.N + MGEN_MU - 1) / MGEN_MU);
  ++::gw::g_launch_count, k_mgen<double><<<grid, 256, 0, st>>>(g, T1, evec, q, kk0, (int)mode, a0, na, b0, nb, out, s_r, s_mu);
}

// fp32 rows (split-precision path), tiled: for one k' and one ABF mu the rows are a complex matrix
// product over K = 2 n_b(A),
//   M_ab = sum_j c_jb(k') conj(T1_ja(k'+q)) + sum_i conj(c_ia(k'+q)) T1_ib(k').
// A block takes one k', `mut` ABFs of one atom, 4 ta bands a and 4 tb bands b; a thread 4 x 4 outputs of
// one ABF (16 complex values from shared memory per 32 complex multiply-adds). The four operands are
// streamed in chunks of JC basis functions by cp.async (16 bytes where the rows allow it) into two
// buffers, whole rows by groups of lanes, so no index is divided in the copy.
// Bound: the T1 stream where one side has few bands (Sigma_c rows, chi0 of few occupied bands), else the
// FP32 units; it reaches a third of the first (issue slots 60% busy) and two thirds of the second. One
// kernel for every shape, measured against the kernels it replaces (streamed ones for at most 8 bands on
// the narrow side and 48 basis functions per atom, shared-memory and direct ones for the rest): chi0 rows of
// 36 x 264 bands, 75 basis functions, 4 k, 1600 ABFs 33.4 -> 2.8 ms; Sigma_c rows of 8 x 300 bands, one k
// 3.0 -> 0.19 ms, of 8 x 78 bands, 39 basis functions, 216 k, 400 ABFs 1.94 -> 1.42 ms; exchange rows (8 x 4
// bands) 104 -> 55 us per q. JC = 2: 4 and 8 hold more shared memory per block and are slower (exchange 73
// and 144 us).
constexpr int MT_JC = 2;
constexpr int MT_THREADS = 256;

struct MgenTile {
  int ta, tb, mut;       // 4-band tiles along a and b, ABFs per block
  int nba, nbb;          // blocks along a and b
  int pa, pb;            // row pitches of the a and b operands in shared memory (complex, even)
  int la, lb;            // log2 of the lanes that copy one row
};

// VEC complex values to shared memory, the first n of them from src and zeros for the rest
template <int VEC> __device__ __forceinline__ void cp_async_c64(float2* dst, const void* src, int n) {
  const uint32_t d = (uint32_t)__cvta_generic_to_shared(dst);
  const int bytes = 8 * max(0, min(n, VEC));
  if constexpr (VEC == 2)
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(d), "l"(src), "r"(bytes) : "memory");
  else
    asm volatile("cp.async.ca.shared.global [%0], [%1], 8, %2;" ::"r"(d), "l"(src), "r"(bytes) : "memory");
}

template <int VEC>
__global__ void __launch_bounds__(MT_THREADS, 3) k_mgen_tile(const __grid_constant__ LriGeom g, MgenTile s,
                                                          const c64* __restrict__ T1, const c64* __restrict__ evec,
                                                          int q, int kk0, int mode, int a0, int na, int b0, int nb,
                                                          c64* __restrict__ out, long long s_r, long long s_mu,
                                                          unsigned* __restrict__ absmax) {
  extern __shared__ __align__(16) float2 sm[];
  const int kk = blockIdx.x;
  int t = blockIdx.y, A = 0;
  for (; A + 1 < g.n_atoms; ++A) {
    const int nt = (g.atom_nx[A] + s.mut - 1) / s.mut;
    if (t < nt) break;
    t -= nt;
  }
  const int mul0 = t * s.mut, cnt = min(s.mut, g.atom_nx[A] - mul0);
  const int ktgt = g.ktab ? g.ktab[kk0 + kk] : kk0 + kk;
  const int k3 = ktgt % g.nk[2], k2 = (ktgt / g.nk[2]) % g.nk[1], k1 = ktgt / (g.nk[1] * g.nk[2]);
  const int q3 = q % g.nk[2], q2 = (q / g.nk[2]) % g.nk[1], q1 = q / (g.nk[1] * g.nk[2]);
  int kp = ktgt, kpq = ktgt;
  if (mode == MAP_K_IS_KK)
    kpq = (((k1 + q1) % g.nk[0]) * g.nk[1] + (k2 + q2) % g.nk[1]) * g.nk[2] + (k3 + q3) % g.nk[2];
  else
    kp = (((k1 - q1 + g.nk[0]) % g.nk[0]) * g.nk[1] + (k2 - q2 + g.nk[1]) % g.nk[1]) * g.nk[2] +
         (k3 - q3 + g.nk[2]) % g.nk[2];
  const int nbA = g.atom_nb[A], b0A = g.atom_b0[A];
  const int at0 = 4 * s.ta * (blockIdx.z % s.nba), bt0 = 4 * s.tb * (blockIdx.z / s.nba);   // first bands of the tile
  const int wa = min(4 * s.ta, na - at0), wb = min(4 * s.tb, nb - bt0);
  const c64* cK = evec + ((long long)kp * g.NB + b0A) * g.NBd + b0 + bt0;
  const c64* cQ = evec + ((long long)kpq * g.NB + b0A) * g.NBd + a0 + at0;
  const c64* tQ = T1 + g.t_off[A] + ((long long)kpq * g.atom_nx[A] + mul0) * nbA * g.NBd + a0 + at0;
  const c64* tK = T1 + g.t_off[A] + ((long long)kp * g.atom_nx[A] + mul0) * nbA * g.NBd + b0 + bt0;
  const long long slab = (long long)nbA * g.NBd;
  // one buffer: rows (m, j), m = 0 the eigenvectors, m = 1 .. mut the T1 slabs; a part then b part
  const int rows = (s.mut + 1) * MT_JC;
  const int buf = rows * (s.pa + s.pb);
  const int warp = threadIdx.x / 32, lane = threadIdx.x % 32, nwarp = blockDim.x / 32;
  // rows of `w` bands (of 4 tl) copied by groups of 2^lg lanes, so that narrow rows fill a warp too
  auto copy = [&](int j0, float2* dst, int pitch, int lg, int w, int width, const c64* ev, const c64* slabs) {
    const int sub = lane >> lg, c0 = VEC * (lane & ((1 << lg) - 1)), per = 32 >> lg;
    for (int r = warp * per + sub; r < rows; r += nwarp * per) {
      const int m = r / MT_JC, j = j0 + r % MT_JC;
      const bool ok = j < nbA && m <= cnt;
      const c64* src = (m == 0 ? ev : slabs + min(m - 1, cnt - 1) * slab) + (long long)min(j, nbA - 1) * g.NBd;
      for (int c = c0; c < width; c += VEC << lg)
        cp_async_c64<VEC>(dst + r * pitch + c, src + (c < w ? c : 0), ok ? w - c : 0);
    }
  };
  auto load = [&](int j0, float2* dst) {
    copy(j0, dst, s.pa, s.la, wa, 4 * s.ta, cQ, tQ);
    copy(j0, dst + rows * s.pa, s.pb, s.lb, wb, 4 * s.tb, cK, tK);
    asm volatile("cp.async.commit_group;" ::: "memory");
  };
  const int m = threadIdx.x % s.mut, rest = threadIdx.x / s.mut, tb = rest % s.tb, ta = rest / s.tb;
  const bool live = ta < s.ta && m < cnt;
  float ar[4][4] = {}, ai[4][4] = {};
  load(0, sm);
  int cur = 0;
  for (int j0 = 0; j0 < nbA; j0 += MT_JC) {
    const bool more = j0 + MT_JC < nbA;
    if (more) load(j0 + MT_JC, sm + (cur ^ 1) * buf);
    if (more) asm volatile("cp.async.wait_group 1;" ::: "memory");
    else asm volatile("cp.async.wait_group 0;" ::: "memory");
    __syncthreads();
    if (live) {
      const float2* pa = sm + cur * buf + 4 * ta;
      const float2* pb = sm + cur * buf + rows * s.pa + 4 * tb;
#pragma unroll
      for (int j = 0; j < MT_JC; ++j) {
        float2 c[4], u[4], d[4], x[4];
        auto four = [](float2 (&v)[4], const float2* p) {
          const float4 lo = reinterpret_cast<const float4*>(p)[0], hi = reinterpret_cast<const float4*>(p)[1];
          v[0] = make_float2(lo.x, lo.y);
          v[1] = make_float2(lo.z, lo.w);
          v[2] = make_float2(hi.x, hi.y);
          v[3] = make_float2(hi.z, hi.w);
        };
        four(d, pa + j * s.pa);                              // c_ja(k'+q)
        four(x, pa + ((m + 1) * MT_JC + j) * s.pa);          // T1_ja(k'+q)
        four(c, pb + j * s.pb);                              // c_jb(k')
        four(u, pb + ((m + 1) * MT_JC + j) * s.pb);          // T1_jb(k')
#pragma unroll
        for (int a = 0; a < 4; ++a)
#pragma unroll
          for (int b = 0; b < 4; ++b) {
            ar[a][b] = fmaf(c[b].x, x[a].x, fmaf(c[b].y, x[a].y, ar[a][b]));      // c conj(T1)
            ai[a][b] = fmaf(c[b].y, x[a].x, fmaf(-c[b].x, x[a].y, ai[a][b]));
            ar[a][b] = fmaf(d[a].x, u[b].x, fmaf(d[a].y, u[b].y, ar[a][b]));      // conj(c) T1
            ai[a][b] = fmaf(d[a].x, u[b].y, fmaf(-d[a].y, u[b].x, ai[a][b]));
          }
      }
    }
    __syncthreads();
    cur ^= 1;
  }
  float amax = 0.f;
  if (live) {
    c64* o = out + (long long)(g.atom_x0[A] + mul0 + m) * s_mu;
#pragma unroll
    for (int a = 0; a < 4; ++a) {
      const int ga = at0 + 4 * ta + a;
      if (ga >= na) continue;
#pragma unroll
      for (int b = 0; b < 4; ++b) {
        const int gb = bt0 + 4 * tb + b;
        if (gb >= nb) continue;
        o[(((long long)kk * na + ga) * nb + gb) * s_r] = c64{ar[a][b], ai[a][b]};
        amax = fmaxf(amax, fmaxf(fabsf(ar[a][b]), fabsf(ai[a][b])));
      }
    }
  }
  if (absmax) {
    // every thread gets here (whole warps); non-negative floats order like their bit patterns
    const unsigned mm = __reduce_max_sync(0xffffffffu, __float_as_uint(amax));
    if (lane == 0) atomicMax(absmax, mm);
  }
}

// Tile shape: blocks of at most 256 threads cut evenly along a and b, then as many ABFs as fit (4 where
// the output runs along the ABFs, so that neighbouring threads fill a 32-byte sector); more than 8 only to reach four warps
template <>
void launch_mgen<float>(const LriGeom& g, const c64* T1, const c64* evec, int q, int kk0, int nkk, MapMode mode, int a0,
                        int na, int b0, int nb, c64* out, long long s_r, long long s_mu, cudaStream_t st,
                        unsigned* absmax) {
  MgenTile s;
  const bool along_mu = s_mu == 1;
  const int qa = (na + 3) / 4, qb = (nb + 3) / 4, most = along_mu ? MT_THREADS / 4 : MT_THREADS;
  // the narrower side whole if it fits, the other one in equal blocks
  s.ta = std::min(qa, 16);
  s.tb = std::min(qb, 16);
  if (qa <= qb) s.tb = std::min(qb, std::max(1, most / s.ta));
  else s.ta = std::min(qa, std::max(1, most / s.tb));
  while (s.ta * s.tb > most) (s.ta > s.tb ? s.ta : s.tb) /= 2;
  s.nba = (qa + s.ta - 1) / s.ta;
  s.nbb = (qb + s.tb - 1) / s.tb;
  s.ta = (qa + s.nba - 1) / s.nba;
  s.tb = (qb + s.nbb - 1) / s.nbb;
  s.mut = along_mu ? 4 : 1;
  while (2 * s.mut * s.ta * s.tb <= MT_THREADS && (s.mut < 8 || (s.mut < 64 && s.mut * s.ta * s.tb < 128))) s.mut *= 2;
  s.pa = 4 * s.ta + 2;   // (16-byte rows)
  s.pb = 4 * s.tb + 2;
  // 16-byte copies where every row of the evec and T1 ranges starts on 16 bytes
  const int vec = (g.NBd % 2 == 0 && a0 % 2 == 0 && b0 % 2 == 0) ? 2 : 1;
  for (s.la = vec == 2 ? 1 : 2; s.la < 5 && (vec << s.la) < 4 * s.ta; ++s.la) {}
  for (s.lb = vec == 2 ? 1 : 2; s.lb < 5 && (vec << s.lb) < 4 * s.tb; ++s.lb) {}
  int tiles = 0;
  for (int A = 0; A < g.n_atoms; ++A) tiles += (g.atom_nx[A] + s.mut - 1) / s.mut;
  const int nt = (s.ta * s.tb * s.mut + 31) / 32 * 32;
  const size_t smem = 2 * sizeof(float2) * (size_t)(s.mut + 1) * MT_JC * (s.pa + s.pb);
  auto* kern = vec == 2 ? k_mgen_tile<2> : k_mgen_tile<1>;
  if (smem > 48 * 1024) cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  ++::gw::g_launch_count, kern<<<dim3(nkk, tiles, s.nba * s.nbb), nt, smem, st>>>(
      g, s, T1, evec, q, kk0, (int)mode, a0, na, b0, nb, out, s_r, s_mu, absmax);
}

}  // namespace gw

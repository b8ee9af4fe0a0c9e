// K5 + K6: RPA correlation energy (Sec. 2):
//
//   E_c = (1/2 pi) sum_q w_q sum_k W_k { ln det[1 - Pi(q, i omega_k)] + Tr Pi(q, i omega_k) },  Pi = chi0 V.
//
// With the Cholesky factor V(q) = L L^H, det(1 - chi0 V) = det(I - L^H chi0 L) (Sylvester) and
// A = I - L^H chi0 L is Hermitian positive definite (chi0 <= 0), so ln det A = 2 sum_i ln (L_A)_ii
// from a Cholesky factorisation A = L_A L_A^H, and Tr Pi = Tr(L^H chi0 L).  Per q: factor V;
// per (q, omega): W = chi0 L, A = I - L^H W (lower triangle), factor A.  The factorisations are
// right-looking and blocked (panel width NB): the diagonal block is factored in shared memory by
// one CTA per matrix, the panel below it by a triangular solve, and the trailing matrix is
// updated by a batched GEMM; every matrix of a batch advances panel by panel in step, so each
// launch has work from all of them.
//
// Two arithmetic routes for the dense GEMMs (W, L^H W and the trailing updates):
//   * native FP64 (complex GEMM on the FP64 pipe, k_zgemm.cu), for the small orders of the FP64 mode;
//   * digit-sliced on the BF16 tensor cores (k_ozgemm.cu, S digit planes, 8 in the FP64 mode): complex products as
//     2 x 2 real blocks [[Re, -Im], [Im, Re]], W produced transposed so that the second GEMM reads
//     it row by row.
// The diagonal blocks, the logarithms and the energy sum are FP64 in both, and so are the panel solves of V(q).  Those of
// I - L^H chi0 L are substitutions on the FP64 route and products with the inverse of the diagonal block on digit planes
// (8 for real matrices), which loses nothing: for I + c PSD of order 48 and norm 1 .. 1e12 the ln det is off by 2.7e-15,
// 4e-14, 3e-11, 4e-8, 2e-6 with substitution and 2.7e-15, 1.1e-13, 4e-11, 3e-8, 4e-7 so.
// On the FP64 route the q with q = -q (chi0 and, when checked, V real there) run every step in
// real arithmetic (A = I - L^T chi0 L, real GEMMs and a real Cholesky): a quarter of the flops.
#include <algorithm>
#include <cmath>
#include <cstring>
#include <vector>

#include "internal.h"
#include "ozgemm.h"
#include "rsqrt.h"
#include "tc.h"

namespace librpa {
namespace {

constexpr int NB = 64;

// ------------------------------------------------------------------ panel kernels (FP64 pipe)
// FP64 runs at two fused multiply-adds per cycle and SM on GB300, a warp's instruction taking ~64 cycles of its
// scheduler's share, so the panel kernels are bound by that pipe (a 64 x 64 complex factorisation is 87k
// cycles of it) and by how few FP64 instructions the serial chains take: columns go in blocks of 8, whose
// 8 x 8 triangle 64 threads factor, an element each, and every other product runs over many threads.
constexpr int KB = 8;   // columns per block

__device__ __forceinline__ void bar_64() { asm volatile("bar.sync 1, 64;" ::: "memory"); }   // threads 0..63

// element arithmetic: T = double2 (complex) or double
__device__ __forceinline__ void sub_mul_conj(double2 &c, double2 a, double2 b) {   // c -= a conj(b)
  c.x = fma(-a.x, b.x, fma(-a.y, b.y, c.x));
  c.y = fma(-a.y, b.x, fma(a.x, b.y, c.y));
}
__device__ __forceinline__ void sub_mul_conj(double &c, double a, double b) { c = fma(-a, b, c); }
__device__ __forceinline__ void sub_mul(double2 &c, double2 a, double2 b) {        // c -= a b
  c.x = fma(-a.x, b.x, fma(a.y, b.y, c.x));
  c.y = fma(-a.x, b.y, fma(-a.y, b.x, c.y));
}
__device__ __forceinline__ void sub_mul(double &c, double a, double b) { c = fma(-a, b, c); }
__device__ __forceinline__ double2 scaled(double2 a, double s) { return make_double2(a.x * s, a.y * s); }
__device__ __forceinline__ double scaled(double a, double s) { return a * s; }
__device__ __forceinline__ double2 sum(double2 a, double2 b) { return make_double2(a.x + b.x, a.y + b.y); }
__device__ __forceinline__ double sum(double a, double b) { return a + b; }
__device__ __forceinline__ double re_of(double2 a) { return a.x; }
__device__ __forceinline__ double re_of(double a) { return a; }
__device__ __forceinline__ void set_re(double2 &a, double x) { a = make_double2(x, 0.0); }
__device__ __forceinline__ void set_re(double &a, double x) { a = x; }

// Factor the NB x NB diagonal block at p0 of every matrix in place (lower triangle).  One CTA per
// matrix.  Adds sum ln d_j of the pivots d_j (= L_jj^2) to lndet[b] (of 2 ln L_jj, the square root's rounding is biased
// downwards for pivots just above 1, which the ln det adds up); sets info[b] = 1 on a non-positive pivot.
// inv (optional, [matrix][NB][NB]): receives L_pp^{-1} of the factored block (lower triangular, zero elsewhere), by
// blocks of 8 rows: Y_II = L_II^{-1}, Y_IJ = -Y_II sum_K L_IK Y_KJ.
// 64 x 64 complex: 268 -> ~75 us (with the inverse 390 -> ~150 us at 96 matrices) against one column at a time.
template <class T>
__global__ void __launch_bounds__(256) k_potrf_diag(T *const *mats, int n, int ld, int p0, double *lndet, int *info,
                                                    T *inv) {
  extern __shared__ __align__(16) unsigned char sm_potrf[];
  T *a = reinterpret_cast<T *>(sm_potrf);   // [NB][NB + 1] (and, with inv, a second such array)
  constexpr int lda = NB + 1;
  __shared__ double rinv[NB], piv[NB];
  __shared__ T colj[2][KB];
  __shared__ int bad;
  const int b = blockIdx.x, tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  T *M = mats[b];
  const int nb = min(NB, n - p0);
  // a ragged last block is completed with the unit matrix
  for (int e = tid; e < NB * NB; e += 256) {
    const int i = e / NB, j = e % NB;
    T v{};
    if (i < nb) {
      if (j <= i) v = M[(size_t)(p0 + i) * ld + p0 + j];
    } else if (i == j) {
      set_re(v, 1.0);
    }
    a[i * lda + j] = v;
  }
  if (tid == 0) bad = 0;
  __syncthreads();
  for (int j0 = 0; j0 < nb; j0 += KB) {
    if (tid < KB * KB) {   // the 8 x 8 triangle: thread = element (r, k)
      const int r = tid / KB, k = tid % KB;
      T e = a[(j0 + r) * lda + j0 + k], s{};   // s: the updates, added once
#pragma unroll
      for (int j = 0; j < KB; ++j) {
        T *col = colj[j & 1];   // column j before its scaling
        if (k == j) {
          e = sum(e, s);
          col[r] = e;
        }
        bar_64();
        double d = re_of(col[j]);
        const bool ok = d > 0.0 && isfinite(d);
        if (!ok) d = 1.0;
        const double ri = fast_rsqrt(d);
        if (k == j) {
          if (r == j) {
            set_re(e, sqrt_from(d, ri));
            rinv[j0 + j] = ri;
            piv[j0 + j] = d;
            if (!ok) bad = 1;
          } else {
            e = scaled(e, ri);
          }
        } else if (k > j && r >= k) {
          sub_mul_conj(s, scaled(col[r], ri), scaled(col[k], ri));
        }
      }
      if (k <= r) a[(j0 + r) * lda + j0 + k] = e;
    }
    __syncthreads();
    const int c0 = j0 + KB, m = NB - c0;   // the rows and columns left
    if (tid < m) {   // panel rows: x_j = (b_j - sum_{k<j} x_k conj(L_jk)) / L_jj
      T x[KB], *row = a + (c0 + tid) * lda + j0;
#pragma unroll
      for (int j = 0; j < KB; ++j) {
        x[j] = row[j];
#pragma unroll
        for (int k = 0; k < j; ++k) sub_mul_conj(x[j], x[k], a[(j0 + j) * lda + j0 + k]);
        x[j] = scaled(x[j], rinv[j0 + j]);
      }
#pragma unroll
      for (int j = 0; j < KB; ++j) row[j] = x[j];
    }
    __syncthreads();
    // trailing update a_ik -= sum_j a_ij conj(a_kj) in 2 x 2 tiles of the lower triangle; the sums apart: products
    // below the last place of a diagonal near 1 (high frequencies) would each be lost, always to the same side
    const int mt = m / 2, nt = mt * (mt + 1) / 2;
    for (int t = tid; t < nt; t += 256) {
      int ty = (int)((sqrtf(8.f * t + 1.f) - 1.f) * 0.5f);
      if (ty * (ty + 1) / 2 > t) --ty;
      if ((ty + 1) * (ty + 2) / 2 <= t) ++ty;
      const int tx = t - ty * (ty + 1) / 2, i = c0 + 2 * ty, k = c0 + 2 * tx;
      T c00{}, c01{}, c10{}, c11{};
#pragma unroll
      for (int j = 0; j < KB; ++j) {
        const T x0 = a[i * lda + j0 + j], x1 = a[(i + 1) * lda + j0 + j], y0 = a[k * lda + j0 + j],
                y1 = a[(k + 1) * lda + j0 + j];
        sub_mul_conj(c00, x0, y0);
        sub_mul_conj(c01, x0, y1);
        sub_mul_conj(c10, x1, y0);
        sub_mul_conj(c11, x1, y1);
      }
      T *row0 = a + i * lda + k, *row1 = row0 + lda;
      row0[0] = sum(row0[0], c00);
      if (tx < ty) row0[1] = sum(row0[1], c01);   // (the element above the diagonal stays)
      row1[0] = sum(row1[0], c10);
      row1[1] = sum(row1[1], c11);
    }
    __syncthreads();
  }
  for (int e = tid; e < nb * nb; e += 256) {
    const int i = e / nb, j = e % nb;
    if (j <= i) M[(size_t)(p0 + i) * ld + p0 + j] = a[i * lda + j];
  }
  if (warp == 0) {
    double l = 0.0;
    for (int j = lane; j < nb; j += 32) l += log(piv[j]);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) l += __shfl_xor_sync(0xffffffffu, l, o);
    if (lane == 0) {
      lndet[b] += l;
      if (bad) info[b] = 1;
    }
  }
  if (!inv) return;
  T *y = a + NB * lda;
  if (tid < 64) {   // Y_II: thread = column c of its block
    const int I = tid / KB, c = tid % KB;
    T v[KB];
#pragma unroll
    for (int i = 0; i < KB; ++i) {
      T s{};
      if (i == c) set_re(s, 1.0);
#pragma unroll
      for (int k = 0; k < i; ++k) sub_mul(s, a[(I * KB + i) * lda + I * KB + k], v[k]);   // v[k] = 0 for k < c
      v[i] = I * KB + i < nb ? scaled(s, rinv[I * KB + i]) : s;
    }
#pragma unroll
    for (int i = 0; i < KB; ++i) y[(I * KB + i) * lda + I * KB + c] = v[i];
  }
  __syncthreads();
  for (int I = 1; I < NB / KB; ++I) {
    // S_IJ = -sum_K L_IK Y_KJ, 2 I tasks of 32 elements (half of a block (I, J)): the warps w < I take tasks w and
    // 2 I - 1 - w, whose sums are equally long together
    if (warp < I) {
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const int t = h ? 2 * I - 1 - warp : warp, J = t >> 1;
        const int i = I * KB + (t & 1) * 4 + (lane >> 3), c = J * KB + (lane & 7);
        T s{};
        for (int k = J * KB; k < I * KB; ++k) sub_mul(s, a[i * lda + k], y[k * lda + c]);
        y[i * lda + c] = s;
      }
    }
    __syncthreads();
    // Y_IJ = Y_II S_IJ: an element per thread, written after every read
    T z[2];
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const int e = h * 256 + tid;
      z[h] = T{};
      if (e < KB * KB * I) {
        const int i = e & 7, c = e >> 3;
        for (int k = 0; k <= i; ++k) sub_mul(z[h], y[(I * KB + i) * lda + I * KB + k], y[(I * KB + k) * lda + c]);
      }
    }
    __syncthreads();
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const int e = h * 256 + tid;
      if (e < KB * KB * I) y[(I * KB + (e & 7)) * lda + (e >> 3)] = scaled(z[h], -1.0);
    }
    __syncthreads();
  }
  T *Y = inv + (size_t)b * NB * NB;
  for (int e = tid; e < NB * NB; e += 256) {
    const int i = e / NB, j = e % NB;
    Y[e] = j <= i && i < nb ? y[i * lda + j] : T{};
  }
}

// Panel solve by substitution: rows i >= p0 + nb, X L_pp^H = B  =>  x_j = (b_j - sum_{k<j} x_k conj(L_jk)) / L_jj, 16
// rows per CTA (so that the few matrices of V(q) fill the SMs), columns in blocks of 8.  Graphene slab, one
// matrix of order 2010: 465 -> ~45 us per panel against 64 rows per CTA, a row per thread.
constexpr int TR = 16;
template <class T>
__global__ void __launch_bounds__(128) k_trsm_panel(T *const *mats, int n, int ld, int p0) {
  extern __shared__ __align__(16) unsigned char sm_trsm[];
  constexpr int lda = NB + 1;
  T *L = reinterpret_cast<T *>(sm_trsm), *X = L + NB * lda;   // [NB][NB + 1], [TR][NB + 1]
  __shared__ double rinv[NB];
  T *M = mats[blockIdx.y];
  const int nb = min(NB, n - p0), r0 = p0 + nb + blockIdx.x * TR, rows = min(TR, n - r0), tid = threadIdx.x;
  for (int e = tid; e < NB * NB; e += 128) {
    const int i = e / NB, j = e % NB;
    L[i * lda + j] = i < nb && j <= i ? M[(size_t)(p0 + i) * ld + p0 + j] : T{};
  }
  for (int e = tid; e < TR * NB; e += 128) {
    const int i = e / NB, j = e % NB;
    X[i * lda + j] = i < rows && j < nb ? M[(size_t)(r0 + i) * ld + p0 + j] : T{};
  }
  if (tid < NB) rinv[tid] = tid < nb ? 1.0 / re_of(M[(size_t)(p0 + tid) * ld + p0 + tid]) : 1.0;
  __syncthreads();
  const int r = tid & (TR - 1), cg = tid / TR;   // row, and one of 8 columns in turn
  for (int j0 = 0; j0 < nb; j0 += KB) {
    T x[KB];
    if (cg == 0) {
#pragma unroll
      for (int j = 0; j < KB; ++j) {
        x[j] = X[r * lda + j0 + j];
#pragma unroll
        for (int k = 0; k < j; ++k) sub_mul_conj(x[j], x[k], L[(j0 + j) * lda + j0 + k]);
        x[j] = scaled(x[j], rinv[j0 + j]);
      }
#pragma unroll
      for (int j = 0; j < KB; ++j) X[r * lda + j0 + j] = x[j];
    }
    __syncthreads();
#pragma unroll
    for (int j = 0; j < KB; ++j) x[j] = X[r * lda + j0 + j];
    for (int c = j0 + KB + cg; c < nb; c += 128 / TR) {
      T s = X[r * lda + c];
#pragma unroll
      for (int j = 0; j < KB; ++j) sub_mul_conj(s, x[j], L[c * lda + j0 + j]);
      X[r * lda + c] = s;
    }
    __syncthreads();
  }
  for (int e = tid; e < rows * NB; e += 128) {
    const int i = e / NB, j = e % NB;
    if (j < nb) M[(size_t)(r0 + i) * ld + p0 + j] = X[i * lda + j];
  }
}

template <class T>
constexpr size_t potrf_smem(bool inv) { return (size_t)(inv ? 2 : 1) * NB * (NB + 1) * sizeof(T); }
template <class T>
constexpr size_t trsm_smem() { return (size_t)(NB + TR) * (NB + 1) * sizeof(T); }

template <class T>
void launch_potrf(T *const *mats, int B, int n, int ld, int p0, double *lndet, int *info, T *inv, cudaStream_t s) {
  LR_CUDA(cudaFuncSetAttribute(k_potrf_diag<T>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)potrf_smem<T>(true)));
  k_potrf_diag<T><<<B, 256, potrf_smem<T>(inv != nullptr), s>>>(mats, n, ld, p0, lndet, info, inv);
  ++launch_counter();
}
template <class T>
void launch_trsm(T *const *mats, int B, int n, int ld, int p0, int rest, cudaStream_t s) {
  LR_CUDA(cudaFuncSetAttribute(k_trsm_panel<T>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)trsm_smem<T>()));
  k_trsm_panel<T><<<dim3((unsigned)((rest + TR - 1) / TR), (unsigned)B), 128, trsm_smem<T>(), s>>>(mats, n, ld, p0);
  ++launch_counter();
}

// Zero the strict upper triangle (so a Cholesky factor can be used as a triangular operand).
__global__ void k_zero_upper(double2 *const *mats, int n, int ld) {
  double2 *M = mats[blockIdx.y];
  const size_t x = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (x >= (size_t)n * n) return;
  const int i = (int)(x / n), j = (int)(x % n);
  if (j > i) M[(size_t)i * ld + j] = make_double2(0.0, 0.0);
}

// Largest |V(-q) - conj V(q)| over the pairs q < -q (res[0]), largest |V(q)| (res[1]) and largest
// |Im V(q)| over the q = -q (res[2]), as the bit patterns of non-negative doubles (ordered like the
// values) for atomicMax.
__global__ void k_conj_check(const double2 *V, int n, int n1, int n2, int n3, unsigned long long *res) {
  const int q = blockIdx.y;
  const int a = q / (n2 * n3), b = (q / n3) % n2, c = q % n3;
  const int p = (((n1 - a) % n1) * n2 + (n2 - b) % n2) * n3 + (n3 - c) % n3;
  if (p < q) return;
  const bool self = p == q;
  const size_t nn = (size_t)n * n;
  const double2 *Vq = V + nn * q, *Vp = V + nn * p;
  double d = 0.0, m = 0.0;
  for (size_t x = (size_t)blockIdx.x * blockDim.x + threadIdx.x; x < nn; x += (size_t)gridDim.x * blockDim.x) {
    const double2 u = Vq[x], v = Vp[x];
    d = self ? fmax(d, fabs(u.y)) : fmax(d, fmax(fabs(v.x - u.x), fabs(v.y + u.y)));
    m = fmax(m, fmax(fabs(u.x), fabs(u.y)));
    if (isnan(u.x + u.y + v.x + v.y)) d = INFINITY;
  }
  for (int o = 16; o > 0; o >>= 1) {
    d = fmax(d, __shfl_xor_sync(0xffffffffu, d, o));
    m = fmax(m, __shfl_xor_sync(0xffffffffu, m, o));
  }
  if ((threadIdx.x & 31) == 0) {
    atomicMax(res + (self ? 2 : 0), (unsigned long long)__double_as_longlong(d));
    atomicMax(res + 1, (unsigned long long)__double_as_longlong(m));
  }
}

// ---------------------------------------------------------------------------------------
// Real route for the q with q = -q (time-reversal-invariant q: q.R is a multiple of pi for every
// lattice vector, so chi0(q, i omega) = sum_R (+-1) chi0(R, i omega) is real symmetric, and V(q)
// is real when V(-q) = conj V(q)).  There A = I - L^T chi0 L is real and every product runs in
// real arithmetic: a quarter of the complex flops.

// Lt = (Re L)^T, n x n, through 32 x 32 shared-memory tiles
__global__ void k_real_transpose(const double2 *L, int n, double *Lt) {
  __shared__ double t[32][33];
  const int r0 = blockIdx.y * 32, c0 = blockIdx.x * 32;
  for (int r = threadIdx.y; r < 32; r += 8) {
    const int gr = r0 + r, gc = c0 + threadIdx.x;
    if (gr < n && gc < n) t[r][threadIdx.x] = L[(size_t)gr * n + gc].x;
  }
  __syncthreads();
  for (int r = threadIdx.y; r < 32; r += 8) {
    const int gr = c0 + r, gc = r0 + threadIdx.x;   // Lt[gr][gc] = L[gc][gr]
    if (gr < n && gc < n) Lt[(size_t)gr * n + gc] = t[threadIdx.x][r];
  }
}

// real parts of n x n matrices, a row per CTA; eq (or NULL): element (i, j) times 2^-(eq[i] + eq[j])
__global__ void k_real_part(const double2 *src, int n, const int *eq, double *dst) {
  const size_t row = (size_t)blockIdx.x * n;
  const int ei = eq ? eq[blockIdx.x % n] : 0;
  for (int j = threadIdx.x; j < n; j += blockDim.x) {
    const double v = src[row + j].x;
    dst[row + j] = eq ? scale_pow2(v, -(ei + eq[j])) : v;
  }
}

// Equilibration of the 8-plane route.  A digit plane holds an element to 2^-63 of its row's largest, where FP64 holds
// every element to 53 bits of its own, so functions of widely different norms would lose the small ones (aux functions
// scaled over 2^30: ln det off by 4e-12, over 2^40 by 1e-8, against 1e-15 in FP64).  The integrand does not change under
// V -> D V D, chi0 -> D^-1 chi0 D^-1, so each V(q) is taken with D_i = 2^eq[i] that brings its diagonal into [1, 4):
// powers of two, exact, and L^H chi0 L is the same matrix.
// V: all matrices; the b-th taken is V[ql[b]].  eq[b][i]
__global__ void k_equil_expo(const double2 *V, const int *ql, int n, int *eq) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const double v = V[((size_t)ql[blockIdx.y] * n + i) * n + i].x;
  const int ex = biased_exp(v);
  eq[(size_t)blockIdx.y * n + i] = v > 0.0 && ex > 0 && ex < 2047 ? -((ex - 1023) >> 1) : 0;
}
__global__ void k_equil_copy(const double2 *V, const int *ql, int n, const int *eq, double2 *out) {   // a row per CTA
  const double2 *src = V + ((size_t)ql[blockIdx.y] * n + blockIdx.x) * n;
  double2 *dst = out + ((size_t)blockIdx.y * n + blockIdx.x) * n;
  eq += (size_t)blockIdx.y * n;
  const int ei = eq[blockIdx.x];
  for (int j = threadIdx.x; j < n; j += blockDim.x) {
    const double2 v = src[j];
    const int e = ei + eq[j];
    dst[j] = make_double2(scale_pow2(v.x, e), scale_pow2(v.y, e));
  }
}

struct RGemm {
  const double *A, *B;   // A [M][K] (lda), B [N][K] (ldb), row-major
  double *C;             // C [M][N] (ldc)
  int M, N, K, lda, ldb, ldc;
  double alpha, beta;
};
struct RTile {
  int e, m0, n0, k0;     // descriptor, output tile origin, first k (rows of A zero before it)
};

// C = alpha A B^T + beta C on the FP64 tensor cores (mma.sync m8n8k4 f64): one 64 x 64 tile per
// CTA, four warps with 32 x 32 warp tiles, K staged 16 at a time through shared memory from the
// tile's k0 (A is upper triangular in the ln det products, zero left of the tile's first row).
__global__ void __launch_bounds__(128) k_dgemm_tri(const RGemm *__restrict__ gs, const RTile *__restrict__ tiles) {
  constexpr int BM = 64, BN = 64, KS = 16, NT = 128;
  const RTile t = tiles[blockIdx.x];
  const RGemm g = gs[t.e];
  __shared__ double As[BM][KS + 1];
  __shared__ double Bs[BN][KS + 1];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int wm = warp >> 1, wn = warp & 1, gid = lane >> 2, tig = lane & 3;
  double acc[4][4][2];
#pragma unroll
  for (int r = 0; r < 4; ++r)
#pragma unroll
    for (int c = 0; c < 4; ++c) acc[r][c][0] = acc[r][c][1] = 0.0;
  for (int k0 = t.k0; k0 < g.K; k0 += KS) {
    for (int e = tid; e < BM * KS; e += NT) {
      const int row = e / KS, k = e % KS, gm = t.m0 + row, gk = k0 + k;
      As[row][k] = (gm < g.M && gk < g.K) ? g.A[(size_t)gm * g.lda + gk] : 0.0;
    }
    for (int e = tid; e < BN * KS; e += NT) {
      const int row = e / KS, k = e % KS, gn = t.n0 + row, gk = k0 + k;
      Bs[row][k] = (gn < g.N && gk < g.K) ? g.B[(size_t)gn * g.ldb + gk] : 0.0;
    }
    __syncthreads();
#pragma unroll
    for (int kk = 0; kk < KS; kk += 4) {
      double a[4], b[4];
#pragma unroll
      for (int r = 0; r < 4; ++r) a[r] = As[wm * 32 + r * 8 + gid][kk + tig];
#pragma unroll
      for (int c = 0; c < 4; ++c) b[c] = Bs[wn * 32 + c * 8 + gid][kk + tig];
#pragma unroll
      for (int r = 0; r < 4; ++r)
#pragma unroll
        for (int c = 0; c < 4; ++c)
          asm volatile("mma.sync.aligned.m8n8k4.row.col.f64.f64.f64.f64 {%0,%1}, {%2}, {%3}, {%0,%1};\n"
                       : "+d"(acc[r][c][0]), "+d"(acc[r][c][1])
                       : "d"(a[r]), "d"(b[c]));
    }
    __syncthreads();
  }
#pragma unroll
  for (int r = 0; r < 4; ++r) {
    const int gm = t.m0 + wm * 32 + r * 8 + gid;
    if (gm >= g.M) continue;
#pragma unroll
    for (int c = 0; c < 4; ++c)
#pragma unroll
      for (int hh = 0; hh < 2; ++hh) {
        const int gn = t.n0 + wn * 32 + c * 8 + tig * 2 + hh;
        if (gn >= g.N) continue;
        double *p = g.C + (size_t)gm * g.ldc + gn;
        const double v = g.alpha * acc[r][c][hh];
        *p = g.beta == 0.0 ? v : v + g.beta * *p;
      }
  }
}

// A = -L^T chi0 L on entry: trace[b] = -sum A_ii, then A_ii += 1 (real route).
__global__ void k_diag_shift_r(double *const *mats, int n, int ld, double *trace) {
  double *M = mats[blockIdx.x];
  double sv = 0.0;
  for (int i = threadIdx.x; i < n; i += blockDim.x) {
    double *p = M + (size_t)i * ld + i;
    sv -= *p;
    *p += 1.0;
  }
  __shared__ double red[256];
  red[threadIdx.x] = sv;
  __syncthreads();
  for (int w = blockDim.x / 2; w > 0; w >>= 1) {
    if (threadIdx.x < w) red[threadIdx.x] += red[threadIdx.x + w];
    __syncthreads();
  }
  if (threadIdx.x == 0) trace[blockIdx.x] = red[0];
}

// A = -L^H chi0 L on entry (lower triangle).  trace[b] = Re Tr(L^H chi0 L) = -sum Re A_ii;
// then A_ii += 1 (A = I - L^H chi0 L).  One CTA per matrix.
__global__ void k_diag_shift(double2 *const *mats, int n, int ld, double *trace) {
  double2 *M = mats[blockIdx.x];
  double s = 0.0;
  for (int i = threadIdx.x; i < n; i += blockDim.x) {
    double2 *p = M + (size_t)i * ld + i;
    s -= p->x;
    p->x += 1.0;
  }
  __shared__ double red[256];
  red[threadIdx.x] = s;
  __syncthreads();
  for (int w = blockDim.x / 2; w > 0; w >>= 1) {
    if (threadIdx.x < w) red[threadIdx.x] += red[threadIdx.x + w];
    __syncthreads();
  }
  if (threadIdx.x == 0) trace[blockIdx.x] = red[0];
}

// K6: E_c, per-q and per-omega parts from the per-(q, omega) ln det and trace.  w_q: per-q weights
// of the q sum, or nullptr for 1 / N_q.
__global__ void k_energy(const double *lndet, const double *trace, const double *w_omega, const double *w_q, int nq,
                         int nw, double *out /* [1 + nq + nw] */) {
  if (threadIdx.x != 0 || blockIdx.x != 0) return;
  const double uniform = 1.0 / (2.0 * M_PI * nq);
  double tot = 0.0;
  for (int k = 0; k < nw; ++k) out[1 + nq + k] = 0.0;
  for (int q = 0; q < nq; ++q) {
    const double pref = w_q ? w_q[q] / (2.0 * M_PI) : uniform;
    double sq = 0.0;
    for (int k = 0; k < nw; ++k) {
      const double f = pref * w_omega[k] * (lndet[q * nw + k] + trace[q * nw + k]);
      sq += f;
      out[1 + nq + k] += f;
    }
    out[1 + q] = sq;
    tot += sq;
  }
  out[0] = tot;
}

// Sliced-operand scratch of the tensor-core route.
struct TcScratch {
  oz::Sliced pa, pb;      // panel of the trailing updates (as A' and as B'^T)
  oz::Sliced pi;          // L_pp^{-H} of the panel solves (as B'^T)
  double2 *inv = nullptr; // [matrix][NB][NB]: L_pp^{-1} of every matrix's current diagonal block
  int *err = nullptr;
  int S = 0;
};

// Blocked Cholesky of `mats` (n x n, lower, in place, uniform stride when tc != nullptr), in step.
// inv_panel (tensor-core route, matrices whose diagonal blocks are well conditioned, such as
// I - L^H chi0 L >= I): the panel solve X L_pp^H = B as the product X = B L_pp^{-H} on the tensor
// cores, with L_pp^{-1} from the diagonal-block kernel; otherwise by substitution (FP64).
void potrf_batched(Handle &h, double2 *const *d_mats, const std::vector<double2 *> &mats, int n, int ld,
                   double *lndet, int *info, TcScratch *tc, bool inv_panel = false) {
  cudaStream_t s = h.stream;
  const int B = (int)mats.size();
  const bool use_inv = tc && inv_panel && tc->inv;
  const long long bstride = B > 1 ? (long long)(mats[1] - mats[0]) : 0;
  for (int p0 = 0; p0 < n; p0 += NB) {
    const int nb = std::min(NB, n - p0), rest = n - p0 - nb;
    const bool inv_now = use_inv && rest > 0;
    launch_potrf<double2>(d_mats, B, n, ld, p0, lndet, info, inv_now ? tc->inv : nullptr, s);
    if (rest <= 0) break;
    if (inv_now) {
      // X = B L_pp^{-H}: stacked real GEMM over the B matrices, K' = 2 nb, written over B
      double2 *P = mats[0] + (size_t)(p0 + nb) * ld + p0;
      oz::sliced_bind(tc->pa, tc->pa.digits, 2 * rest * B, 2 * nb, tc->S);
      oz::sliced_bind(tc->pi, tc->pi.digits, nb * B, 2 * nb, tc->S);
      oz::split_complex(P, ld, oz::OP_N, true, rest, nb, B, bstride, tc->pa, s);
      oz::split_complex(tc->inv, NB, oz::OP_H, false, nb, nb, B, (long long)NB * NB, tc->pi, s);
      oz::Out o;
      o.C = (double *)P;
      o.ldc = ld;
      o.batch_stride = bstride;
      o.mode = 1;
      o.alpha = 1.0;
      o.beta = 0.0;
      Handle::Timed tm{nullptr, nullptr, 8.0 * B * rest * 0.5 * nb * nb, 1};
      LR_CUDA(cudaEventCreate(&tm.a));
      LR_CUDA(cudaEventCreate(&tm.b));
      LR_CUDA(cudaEventRecord(tm.a, s));
      oz::gemm(tc->pa, tc->pi, 2 * rest, nb, B, o, 0, 0, 0, tc->err, s, h);
      LR_CUDA(cudaEventRecord(tm.b, s));
      tm.exec_flops = h.oz_exec_flops;
      h.timed.push_back(tm);
    } else {
      launch_trsm<double2>(d_mats, B, n, ld, p0, rest, s);
    }
    // algorithmic work: the lower triangle (with diagonal) of a rest x rest update of rank nb
    const double fl = 8.0 * B * (0.5 * rest * (rest + 1.0)) * nb;
    if (tc) {
      // A22 -= P P^H with P = A[p0+nb.., p0..p0+nb): stacked real GEMM, K' = 2 nb
      const double2 *P = mats[0] + (size_t)(p0 + nb) * ld + p0;
      oz::sliced_bind(tc->pa, tc->pa.digits, 2 * rest * B, 2 * nb, tc->S);
      oz::sliced_bind(tc->pb, tc->pb.digits, rest * B, 2 * nb, tc->S);
      oz::split_complex(P, ld, oz::OP_N, true, rest, nb, B, bstride, tc->pa, s);
      oz::split_complex(P, ld, oz::OP_H, false, rest, nb, B, bstride, tc->pb, s);
      oz::Out o;
      o.C = (double *)(mats[0] + (size_t)(p0 + nb) * ld + p0 + nb);
      o.ldc = ld;
      o.batch_stride = bstride;
      o.mode = 1;
      o.alpha = -1.0;
      o.beta = 1.0;
      Handle::Timed tm{nullptr, nullptr, fl, 1};
      LR_CUDA(cudaEventCreate(&tm.a));
      LR_CUDA(cudaEventCreate(&tm.b));
      LR_CUDA(cudaEventRecord(tm.a, s));
      oz::gemm(tc->pa, tc->pb, 2 * rest, rest, B, o, 0, 0, 2, tc->err, s, h);
      LR_CUDA(cudaEventRecord(tm.b, s));
      tm.exec_flops = h.oz_exec_flops;
      h.timed.push_back(tm);
      continue;
    }
    std::vector<ZGemm> batch;
    for (int b = 0; b < B; ++b) {
      ZGemm z{};
      double2 *M = mats[b];
      z.A = M + (size_t)(p0 + nb) * ld + p0;
      z.B = z.A;
      z.C = M + (size_t)(p0 + nb) * ld + p0 + nb;
      z.M = rest;
      z.N = rest;
      z.K = nb;
      z.lda = ld;
      z.ldb = ld;
      z.ldc = ld;
      z.alpha = make_double2(-1.0, 0.0);
      z.beta = make_double2(1.0, 0.0);
      batch.push_back(z);
    }
    ZGemmFlags f;
    f.transB = true;
    f.conjB = true;
    f.lower_only = true;
    zgemm_batched(batch, f, s, h, 1, fl);
  }
  LR_CUDA(cudaGetLastError());
}

// Batched real GEMMs (k_dgemm_tri) of one launch.  shape: 0 = every output tile, 1 = tiles on or
// above the diagonal (n0 >= m0), 2 = on or below (n0 <= m0); kfrom_row: K starts at the tile's
// first row (A zero left of its diagonal).  flops: algorithmic count for the stats.
void rgemm_batched(Handle &h, const std::vector<RGemm> &gs, int shape, bool kfrom_row, double flops) {
  constexpr int T = 64;
  std::vector<RTile> tiles;
  for (int e = 0; e < (int)gs.size(); ++e)
    for (int m0 = 0; m0 < gs[e].M; m0 += T)
      for (int n0 = 0; n0 < gs[e].N; n0 += T) {
        if ((shape == 1 && n0 < m0) || (shape == 2 && n0 > m0)) continue;
        tiles.push_back({e, m0, n0, kfrom_row ? m0 : 0});
      }
  if (tiles.empty()) return;
  const size_t b1 = gs.size() * sizeof(RGemm), b2 = tiles.size() * sizeof(RTile);
  const size_t off2 = (b1 + 255) / 256 * 256;
  static thread_local std::vector<char> host;
  host.resize(off2 + b2);
  std::memcpy(host.data(), gs.data(), b1);
  std::memcpy(host.data() + off2, tiles.data(), b2);
  h.ensure(h.rgemm_args, off2 + b2);
  cudaStream_t s = h.stream;
  LR_CUDA(cudaMemcpyAsync(h.rgemm_args.p, host.data(), off2 + b2, cudaMemcpyHostToDevice, s));
  const RGemm *dg = reinterpret_cast<const RGemm *>(h.rgemm_args.p);
  const RTile *dt = reinterpret_cast<const RTile *>((const char *)h.rgemm_args.p + off2);
  Handle::Timed tm{nullptr, nullptr, flops, 1};
  LR_CUDA(cudaEventCreate(&tm.a));
  LR_CUDA(cudaEventCreate(&tm.b));
  LR_CUDA(cudaEventRecord(tm.a, s));
  for (size_t t0 = 0; t0 < tiles.size(); t0 += 1u << 30) {
    const unsigned nb = (unsigned)std::min<size_t>(tiles.size() - t0, 1u << 30);
    k_dgemm_tri<<<nb, 128, 0, s>>>(dg, dt + t0);
    ++launch_counter();
  }
  LR_CUDA(cudaEventRecord(tm.b, s));
  h.timed.push_back(tm);
  LR_CUDA(cudaGetLastError());
}

// Blocked real Cholesky of `mats` (n x n, lower, in place), in step (as potrf_batched), of matrices
// I - L^T chi0 L >= I.  tc (tensor-core route, uniform matrix stride): the panels as products with the inverse
// diagonal block (as inv_panel of potrf_batched) and the trailing updates as digit-plane GEMMs; otherwise
// substitution and FP64 DMMA.
void potrf_batched_r(Handle &h, double *const *d_mats, const std::vector<double *> &mats, int n, int ld,
                     double *lndet, int *info, TcScratch *tc = nullptr) {
  cudaStream_t s = h.stream;
  const int B = (int)mats.size();
  const long long bstride = B > 1 ? (long long)(mats[1] - mats[0]) : 0;
  for (int p0 = 0; p0 < n; p0 += NB) {
    const int nb = std::min(NB, n - p0), rest = n - p0 - nb;
    double *inv = tc && rest > 0 ? (double *)tc->inv : nullptr;
    launch_potrf<double>(d_mats, B, n, ld, p0, lndet, info, inv, s);
    if (rest <= 0) break;
    if (tc) {
      // X = B L_pp^{-T} with 8 digit planes (the substitution it stands for is FP64), written over B
      double *P = mats[0] + (size_t)(p0 + nb) * ld + p0;
      oz::sliced_bind(tc->pa, tc->pa.digits, rest * B, nb, oz::S_WIDE);
      oz::sliced_bind(tc->pi, tc->pi.digits, nb * B, nb, oz::S_WIDE);
      oz::split_real(P, ld, false, rest, nb, B, bstride, tc->pa, s);
      oz::split_real(inv, NB, false, nb, nb, B, (long long)NB * NB, tc->pi, s);
      oz::Out o;
      o.C = P;
      o.ldc = ld;
      o.batch_stride = bstride;
      o.mode = 0;
      Handle::Timed tm{nullptr, nullptr, 2.0 * B * rest * 0.5 * nb * nb, 1};
      LR_CUDA(cudaEventCreate(&tm.a));
      LR_CUDA(cudaEventCreate(&tm.b));
      LR_CUDA(cudaEventRecord(tm.a, s));
      oz::gemm(tc->pa, tc->pi, rest, nb, B, o, 0, 0, 0, tc->err, s, h);
      LR_CUDA(cudaEventRecord(tm.b, s));
      tm.exec_flops = h.oz_exec_flops;
      h.timed.push_back(tm);
    } else {
      launch_trsm<double>(d_mats, B, n, ld, p0, rest, s);
    }
    const double fl = 2.0 * B * (0.5 * rest * (rest + 1.0)) * nb;
    if (tc) {
      // A22 -= P P^T on the lower tiles, P = A[p0+nb.., p0..p0+nb): one operand in both roles
      const double *P = mats[0] + (size_t)(p0 + nb) * ld + p0;
      oz::sliced_bind(tc->pa, tc->pa.digits, rest * B, nb, tc->S);
      oz::split_real(P, ld, false, rest, nb, B, bstride, tc->pa, s);
      oz::Out o;
      o.C = mats[0] + (size_t)(p0 + nb) * ld + p0 + nb;
      o.ldc = ld;
      o.batch_stride = bstride;
      o.mode = 0;
      o.alpha = -1.0;
      o.beta = 1.0;
      Handle::Timed tm{nullptr, nullptr, fl, 1};
      LR_CUDA(cudaEventCreate(&tm.a));
      LR_CUDA(cudaEventCreate(&tm.b));
      LR_CUDA(cudaEventRecord(tm.a, s));
      oz::gemm(tc->pa, tc->pa, rest, rest, B, o, 0, 0, 1, tc->err, s, h);
      LR_CUDA(cudaEventRecord(tm.b, s));
      tm.exec_flops = h.oz_exec_flops;
      h.timed.push_back(tm);
      continue;
    }
    // A22 -= P P^T on the lower tiles, P = A[p0+nb.., p0..p0+nb)
    std::vector<RGemm> batch;
    for (int b = 0; b < B; ++b) {
      double *M = mats[b];
      const double *P = M + (size_t)(p0 + nb) * ld + p0;
      batch.push_back(RGemm{P, P, M + (size_t)(p0 + nb) * ld + p0 + nb, rest, rest, nb, ld, ld, ld, -1.0, 1.0});
    }
    rgemm_batched(h, batch, 2, false, fl);
  }
  LR_CUDA(cudaGetLastError());
}

// digit planes of the ln det GEMMs: those of the mode, and 8 in the FP64 mode for matrices of order
// kWideMinN or more (-1: the FP64 pipes).  Both sides measured (1 k point, 8 frequencies, ms on the pipes / planes):
// N_aux 16 0.21 / 0.23, 32 0.31 / 0.30, 48 0.41 / 0.35, 96 1.20 / 0.75, 180 2.3 / 1.3, 340 5.3 / 2.6.  The line lies above the
// crossover: smaller matrices keep the arithmetic of the pipes at up to 0.5 ms more.
constexpr int kWideMinN = 96;
int ec_planes(const Handle &h) { return h.ec_S >= 0 ? h.ec_S : h.naux >= kWideMinN && !h.lean_ec ? oz::S_WIDE : -1; }

size_t al256(size_t b) { return (b + 255) / 256 * 256; }

// Workspace of the ln det stage: L[nq], W[nw], A[nw] (complex n x n), pointer tables,
// lndet/trace/info, output, and for the tensor-core route the digit planes.
struct EcLayout {
  size_t o_L, o_W, o_A, o_ptr, o_ld, o_tr, o_ldc, o_trc, o_inf, o_out, o_wo, o_wq, o_err;
  size_t o_sx = 0, o_sw = 0, o_sl = 0, o_slh = 0, o_pa = 0, o_pb = 0, o_inv = 0, o_pi = 0, o_eq = 0;
  size_t total = 0;
};

// q points factorised together: the q <= -q of the mesh (all q are computed in chunks of this
// size when V(q) turns out not to pair)
int ec_chunk(const Handle &h) {
  int c = 0;
  for (int q = 0; q < h.mesh.size(); ++q) c += q <= h.mesh.neg(q);
  return c;
}

EcLayout ec_layout(const Handle &h) {
  const int n = h.naux, nq = h.mesh.size(), nw = h.ntau, S = ec_planes(h), nc = ec_chunk(h);
  const size_t n2 = (size_t)n * n, mat = n2 * sizeof(double2);
  const int bmax = std::max(nq, nc * nw);
  EcLayout l;
  size_t off = 0;
  auto take = [&](size_t bytes) { const size_t o = off; off += al256(bytes); return o; };
  l.o_L = take(nq * mat);
  l.o_W = take(nw * mat);
  l.o_A = take((size_t)nc * nw * mat);   // the (q, omega) of a chunk are factorised in one batch
  l.o_ptr = take(((size_t)nq + (size_t)nc * nw + 8) * 8);
  l.o_ld = take(((size_t)nq * nw + nq) * 8);
  l.o_tr = take((size_t)nq * nw * 8);
  l.o_ldc = take((size_t)nq * nw * 8);
  l.o_trc = take((size_t)nq * nw * 8);
  l.o_inf = take((size_t)(nq + nq * nw) * 4);
  l.o_out = take((size_t)(1 + nq + nw) * 8);
  l.o_wo = take((size_t)nw * 8);
  l.o_wq = take((size_t)nq * 8);
  l.o_err = take(4);
  if (S >= 0) {
    l.o_sx = take(oz::sliced_bytes(nw * 2 * n, 2 * n, S));
    l.o_sw = take(oz::sliced_bytes(nw * n, 2 * n, S));
    l.o_sl = take(oz::sliced_bytes(n, 2 * n, S));
    l.o_slh = take(oz::sliced_bytes(2 * n, 2 * n, S));
    // panels and inverse diagonal blocks: complex ones with S planes, those of the real route with 8
    l.o_pa = take(std::max(oz::sliced_bytes(bmax * 2 * n, 2 * NB, S), oz::sliced_bytes(bmax * n, NB, oz::S_WIDE)));
    l.o_pb = take(oz::sliced_bytes(bmax * n, 2 * NB, S));
    l.o_inv = take((size_t)bmax * NB * NB * sizeof(double2));
    l.o_pi = take(std::max(oz::sliced_bytes(bmax * NB, 2 * NB, S), oz::sliced_bytes(bmax * NB, NB, oz::S_WIDE)));
  }
  if (S == oz::S_WIDE) l.o_eq = take((size_t)nq * (n + 1) * 4);
  l.total = off;
  return l;
}

}  // namespace

size_t ec_work_bytes(const Handle &h) { return ec_layout(h).total; }

int ec_run(Handle &h, double *ec, double *ec_q, double *ec_w) {
  const int n = h.naux, nq = h.mesh.size(), nw = h.ntau, S = ec_planes(h);
  const size_t n2 = (size_t)n * n;
  cudaStream_t s = h.stream;
  const size_t mat = n2 * sizeof(double2);
  const int nc = ec_chunk(h), bmax = std::max(nq, nc * nw);
  const EcLayout lay = ec_layout(h);
  const size_t o_L = lay.o_L, o_W = lay.o_W, o_A = lay.o_A, o_ptr = lay.o_ptr, o_ld = lay.o_ld, o_tr = lay.o_tr,
               o_inf = lay.o_inf, o_out = lay.o_out, o_wo = lay.o_wo, o_err = lay.o_err, o_sx = lay.o_sx,
               o_sw = lay.o_sw, o_sl = lay.o_sl, o_slh = lay.o_slh, o_pa = lay.o_pa, o_pb = lay.o_pb;
  h.ensure(h.work, lay.total);
  char *w = (char *)h.work.p;
  double2 *Lq = (double2 *)(w + o_L), *Wm = (double2 *)(w + o_W), *Am = (double2 *)(w + o_A);
  double2 **ptrs = (double2 **)(w + o_ptr);
  double *lndet = (double *)(w + o_ld), *trace = (double *)(w + o_tr), *out = (double *)(w + o_out);
  double *wo = (double *)(w + o_wo);
  int *info = (int *)(w + o_inf);
  int *err = (int *)(w + o_err);
  double *lndet_v = lndet + (size_t)nq * nw;   // scratch for the V(q) factorisations
  LR_CUDA(cudaMemsetAsync(lndet, 0, ((size_t)nq * nw + nq) * 8, s));
  LR_CUDA(cudaMemsetAsync(info, 0, (size_t)(nq + nq * nw) * 4, s));
  LR_CUDA(cudaMemsetAsync(err, 0, 4, s));
  LR_CUDA(cudaMemcpyAsync(wo, h.w_omega.data(), (size_t)nw * 8, cudaMemcpyHostToDevice, s));
  // per-q weights of the q sum (set_q_weights), else 1 / N_q; q of zero weight are not computed
  const bool weighted = !h.wq.empty();
  double *wqd = weighted ? (double *)(w + lay.o_wq) : nullptr;
  if (weighted) LR_CUDA(cudaMemcpyAsync(wqd, h.wq.data(), (size_t)nq * 8, cudaMemcpyHostToDevice, s));
  auto weight = [&](int q) { return weighted ? h.wq[q] : 1.0; };
  TcScratch tcs;
  TcScratch *tc = nullptr;
  oz::Sliced sx, sw, sl, slh;
  if (S >= 0) {
    tcs.S = S;
    tcs.err = err;
    oz::sliced_bind(tcs.pa, w + o_pa, bmax * 2 * n, 2 * NB, S);
    oz::sliced_bind(tcs.pb, w + o_pb, bmax * n, 2 * NB, S);
    oz::sliced_bind(tcs.pi, w + lay.o_pi, bmax * NB, 2 * NB, S);
    tcs.inv = (double2 *)(w + lay.o_inv);
    oz::sliced_bind(sx, w + o_sx, nw * 2 * n, 2 * n, S);
    oz::sliced_bind(sw, w + o_sw, nw * n, 2 * n, S);
    oz::sliced_bind(sl, w + o_sl, n, 2 * n, S);
    oz::sliced_bind(slh, w + o_slh, 2 * n, 2 * n, S);
    tc = &tcs;
  }
  // q <-> -q: chi0(R) is real, so chi0(-q) = conj chi0(q); when also V(-q) = conj V(q) (to 1e-12
  // of max |V|), the integrand of -q equals that of q (ln det and trace of complex-conjugate
  // matrices), and only q <= -q is computed.  The check runs once per set of V(q).
  // The same check gives the real route (section above) its condition: V(q) real at q = -q.
  if (h.vq_sym < 0 || h.vq_real < 0) {
    // 24 bytes at lndet (its region is at least 256 bytes long; it is cleared again below)
    unsigned long long *res = (unsigned long long *)(w + o_ld);
    LR_CUDA(cudaMemsetAsync(res, 0, 24, s));
    k_conj_check<<<dim3(64, (unsigned)nq), 256, 0, s>>>((const double2 *)h.d_vq.p, n, h.mesh.n1, h.mesh.n2,
                                                        h.mesh.n3, res);
    ++launch_counter();
    LR_CUDA(cudaGetLastError());
    double dm[3] = {0, 0, 0};
    LR_CUDA(cudaMemcpyAsync(dm, res, 24, cudaMemcpyDeviceToHost, s));
    LR_CUDA(cudaStreamSynchronize(s));
    h.vq_sym = dm[0] <= 1e-12 * dm[1] ? 1 : 0;
    h.vq_real = dm[2] <= 1e-12 * dm[1] ? 1 : 0;
    LR_CUDA(cudaMemsetAsync(lndet, 0, 24, s));
  }
  std::vector<int> qlist;
  for (int q = 0; q < nq; ++q) {
    const int p = h.mesh.neg(q);
    if (h.vq_sym == 1 ? q <= p && (weight(q) > 0 || weight(p) > 0) : weight(q) > 0) qlist.push_back(q);
  }
  const int nql = (int)qlist.size();
  // positions in qlist, the complex ones first, then those of the real route: the per-(q, omega)
  // ln det and trace are kept in this order until the end
  std::vector<int> order;
  auto real_q = [&](int q) { return h.vq_real == 1 && q == h.mesh.neg(q); };
  for (int qi = 0; qi < nql; ++qi)
    if (!real_q(qlist[qi])) order.push_back(qi);
  const int nx = (int)order.size();
  for (int qi = 0; qi < nql; ++qi)
    if (real_q(qlist[qi])) order.push_back(qi);
  // Cholesky of every V(q) computed, packed in qlist order (the batched factorisation needs a
  // uniform stride)
  std::vector<double2 *> lp(nql);
  int *eq = S == oz::S_WIDE ? (int *)(w + lay.o_eq) : nullptr;   // [qlist][n], then the qlist
  for (int i = 0; i < nql; ++i) {
    lp[i] = Lq + (size_t)i * n2;
    if (!eq) LR_CUDA(cudaMemcpyAsync(lp[i], (const char *)h.d_vq.p + (size_t)qlist[i] * mat, mat, cudaMemcpyDeviceToDevice, s));
  }
  if (eq) {
    int *ql = eq + (size_t)nq * n;
    LR_CUDA(cudaMemcpyAsync(ql, qlist.data(), nql * 4, cudaMemcpyHostToDevice, s));
    k_equil_expo<<<dim3((unsigned)((n + 255) / 256), (unsigned)nql), 256, 0, s>>>((const double2 *)h.d_vq.p, ql, n, eq);
    k_equil_copy<<<dim3((unsigned)n, (unsigned)nql), 256, 0, s>>>((const double2 *)h.d_vq.p, ql, n, eq, Lq);
    launch_counter() += 2;
    LR_CUDA(cudaGetLastError());
  }
  LR_CUDA(cudaMemcpyAsync(ptrs, lp.data(), nql * 8, cudaMemcpyHostToDevice, s));
  auto eq_of = [&](int qi) { return eq ? eq + (size_t)qi * n : nullptr; };
  potrf_batched(h, ptrs, lp, n, n, lndet_v, info, tc);
  {
    dim3 g((unsigned)((n2 + 255) / 256), (unsigned)nql);
    k_zero_upper<<<g, 256, 0, s>>>(ptrs, n, n);
    ++launch_counter();
  }
  const double2 *chi = (const double2 *)h.d_chi_qw.p;
  // A(q, omega) of the q of a chunk, packed: A[(pos - c0) * nw + k]; each chunk is factorised in
  // one lockstep batch
  double2 **aptr = ptrs + nq;
  double *lndet_c = (double *)(w + lay.o_ldc), *trace_c = (double *)(w + lay.o_trc);
  LR_CUDA(cudaMemsetAsync(lndet_c, 0, (size_t)nql * nw * 8, s));
  // algorithmic work (8 flops per complex MAC): A = -L^H W on the lower triangle,
  // sum_{i >= j} (n - i) MACs per matrix
  const double dn = n;
  const double fl_a = 8.0 * nw * (dn * (dn + 1) * (dn + 2) / 6);
  // A needs W only on and below its diagonal tiles (j >= k), sum_k (n - k)^2 MACs
  const double fl_w_lower = 8.0 * nw * (dn * (dn + 1) * (2 * dn + 1) / 6);
  for (int c0 = 0; c0 < nx; c0 += nc) {
    const int c1 = std::min(nx, c0 + nc);
    std::vector<double2 *> ap((size_t)(c1 - c0) * nw);
    for (size_t b = 0; b < ap.size(); ++b) ap[b] = Am + b * n2;
    LR_CUDA(cudaMemcpyAsync(aptr, ap.data(), ap.size() * 8, cudaMemcpyHostToDevice, s));
    for (int pos = c0; pos < c1; ++pos) {
      const int qi = order[pos], q = qlist[qi];
      double2 *Aq = Am + (size_t)(pos - c0) * nw * n2;
      if (S >= 0) {
        const double2 *L = Lq + (size_t)qi * n2;
        oz::split_complex(L, n, oz::OP_N, false, n, n, 1, 0, sl, s);     // B'^T of W = chi0 L
        oz::split_complex(L, n, oz::OP_H, true, n, n, 1, 0, slh, s);     // A' of L^H W
        oz::split_complex(chi + (size_t)q * nw * n2, n, oz::OP_N, true, n, n, nw, (long long)n2, sx, s,
                          eq_of(qi));
        // W^T, so that the second GEMM reads W column by column as rows.  A = -L^H W reads W only on
        // and below its diagonal tiles (k >= j): the tiles above are not computed and stay zero
        // (the digit planes of W's rows see zeros there)
        LR_CUDA(cudaMemsetAsync(Wm, 0, (size_t)nw * mat, s));
        oz::Out o1;
        o1.C = (double *)Wm;
        o1.ldc = n;
        o1.batch_stride = (long long)n2;
        o1.mode = 2;
        Handle::Timed t1{nullptr, nullptr, fl_w_lower, 1};
        LR_CUDA(cudaEventCreate(&t1.a));
        LR_CUDA(cudaEventCreate(&t1.b));
        LR_CUDA(cudaEventRecord(t1.a, s));
        oz::gemm(sx, sl, 2 * n, n, nw, o1, 0, 2, 2, err, s, h);
        LR_CUDA(cudaEventRecord(t1.b, s));
        t1.exec_flops = h.oz_exec_flops;
        h.timed.push_back(t1);
        oz::split_complex(Wm, n, oz::OP_T, false, n, n, nw, (long long)n2, sw, s);   // B'^T rows j: W[k][j]
        oz::Out o2;
        o2.C = (double *)Aq;
        o2.ldc = n;
        o2.batch_stride = (long long)n2;
        o2.mode = 1;
        o2.alpha = -1.0;
        Handle::Timed t2{nullptr, nullptr, fl_a, 1};
        LR_CUDA(cudaEventCreate(&t2.a));
        LR_CUDA(cudaEventCreate(&t2.b));
        LR_CUDA(cudaEventRecord(t2.a, s));
        oz::gemm(slh, sw, 2 * n, n, nw, o2, 1, 0, 2, err, s, h);
        LR_CUDA(cudaEventRecord(t2.b, s));
        t2.exec_flops = h.oz_exec_flops;
        h.timed.push_back(t2);
      } else {
        // W = chi0(q, omega) L_q  (L lower triangular: k >= j)
        std::vector<ZGemm> b1, b2;
        for (int k = 0; k < nw; ++k) {
          ZGemm z{};
          z.A = chi + ((size_t)q * nw + k) * n2;
          z.B = Lq + (size_t)qi * n2;
          z.C = Wm + k * n2;
          z.M = z.N = z.K = n;
          z.lda = z.ldb = z.ldc = n;
          z.alpha = make_double2(1.0, 0.0);
          z.beta = make_double2(0.0, 0.0);
          b1.push_back(z);
          ZGemm y{};
          y.A = Lq + (size_t)qi * n2;     // op(A) = L^H: stored [K][M], conjugated
          y.B = Wm + k * n2;
          y.C = Aq + k * n2;
          y.M = y.N = y.K = n;
          y.lda = y.ldb = y.ldc = n;
          y.alpha = make_double2(-1.0, 0.0);
          y.beta = make_double2(0.0, 0.0);
          b2.push_back(y);
        }
        ZGemmFlags f1;
        f1.kfrom = 2;
        f1.lower_only = true;   // the second GEMM reads W only on and below the diagonal tiles
        zgemm_batched(b1, f1, s, h, 1, fl_w_lower);
        ZGemmFlags f2;
        f2.transA = true;
        f2.conjA = true;
        f2.kfrom = 1;
        f2.lower_only = true;
        zgemm_batched(b2, f2, s, h, 1, fl_a);
      }
    }
    // A = I - L^H chi0 L of the chunk's (q, omega): trace, then one lockstep Cholesky of all
    k_diag_shift<<<(unsigned)ap.size(), 256, 0, s>>>(aptr, n, n, trace_c + (size_t)c0 * nw);
    ++launch_counter();
    potrf_batched(h, aptr, ap, n, n, lndet_c + (size_t)c0 * nw, info + nq + (size_t)c0 * nw, tc, true);
  }
  if (nql > nx) {
    // real route, all its (q, omega) in one lockstep batch, in the A region (real matrices take
    // half the room of complex ones): Ar[B] then Lt; W's region holds Re chi0 and W^T of one q
    const int nr = nql - nx;
    const size_t B = (size_t)nr * nw;
    double *Ar = (double *)Am, *Lt = Ar + B * n2;
    double *Xr = (double *)Wm, *WT = Xr + (size_t)nw * n2;
    std::vector<double *> ar(B);
    for (size_t b = 0; b < B; ++b) ar[b] = Ar + b * n2;
    double **rptr = reinterpret_cast<double **>(aptr);
    LR_CUDA(cudaMemcpyAsync(rptr, ar.data(), B * 8, cudaMemcpyHostToDevice, s));
    const unsigned nt = (unsigned)((n + 31) / 32);
    for (int r = 0; r < nr; ++r) {
      const int qi = order[nx + r], q = qlist[qi];
      k_real_transpose<<<dim3(nt, nt), dim3(32, 8), 0, s>>>(Lq + (size_t)qi * n2, n, Lt);
      k_real_part<<<(unsigned)(nw * n), 256, 0, s>>>(chi + (size_t)q * nw * n2, n, eq_of(qi), Xr);
      launch_counter() += 2;
      LR_CUDA(cudaGetLastError());
      if (S >= 0) {
        // W = Xr L on and below the diagonal tiles (W[k][j] = sum_l Xr[k][l] Lt[j][l], l >= j; the
        // tiles above stay zero), then A = -L^T W = -(Lt rows) . (W^T rows), l >= i, lower tiles
        double *Wr = WT;
        LR_CUDA(cudaMemsetAsync(Wr, 0, (size_t)nw * n2 * sizeof(double), s));
        oz::Sliced slt = sl, sxr = sx, swt = sw;
        oz::sliced_bind(slt, sl.digits, n, n, S);
        oz::sliced_bind(sxr, sx.digits, nw * n, n, S);
        oz::sliced_bind(swt, sw.digits, nw * n, n, S);
        oz::split_real(Lt, n, false, n, n, 1, 0, slt, s);
        oz::split_real(Xr, n, false, n, n, nw, (long long)n2, sxr, s);
        oz::Out o1;
        o1.C = Wr;
        o1.ldc = n;
        o1.batch_stride = (long long)n2;
        o1.mode = 0;
        Handle::Timed t1{nullptr, nullptr, fl_w_lower / 4, 1};
        LR_CUDA(cudaEventCreate(&t1.a));
        LR_CUDA(cudaEventCreate(&t1.b));
        LR_CUDA(cudaEventRecord(t1.a, s));
        oz::gemm(sxr, slt, n, n, nw, o1, 0, 1, 1, err, s, h);
        LR_CUDA(cudaEventRecord(t1.b, s));
        t1.exec_flops = h.oz_exec_flops;
        h.timed.push_back(t1);
        oz::split_real(Wr, n, true, n, n, nw, (long long)n2, swt, s);
        oz::Out o2;
        o2.C = Ar + (size_t)r * nw * n2;
        o2.ldc = n;
        o2.batch_stride = (long long)n2;
        o2.mode = 0;
        o2.alpha = -1.0;
        Handle::Timed t2{nullptr, nullptr, fl_a / 4, 1};
        LR_CUDA(cudaEventCreate(&t2.a));
        LR_CUDA(cudaEventCreate(&t2.b));
        LR_CUDA(cudaEventRecord(t2.a, s));
        oz::gemm(slt, swt, n, n, nw, o2, 1, 0, 1, err, s, h);
        LR_CUDA(cudaEventRecord(t2.b, s));
        t2.exec_flops = h.oz_exec_flops;
        h.timed.push_back(t2);
        continue;
      }
      // W^T = Lt Xr^T (= (chi0 L)^T) on and above the diagonal tiles; A = -Lt (W^T)^T = -L^T W on
      // and below them; Lt is upper triangular, so K starts at the tile's first row
      std::vector<RGemm> g1, g2;
      for (int k = 0; k < nw; ++k) {
        g1.push_back(RGemm{Lt, Xr + (size_t)k * n2, WT + (size_t)k * n2, n, n, n, n, n, n, 1.0, 0.0});
        g2.push_back(RGemm{Lt, WT + (size_t)k * n2, Ar + ((size_t)r * nw + k) * n2, n, n, n, n, n, n, -1.0, 0.0});
      }
      rgemm_batched(h, g1, 1, true, fl_w_lower / 4);
      rgemm_batched(h, g2, 2, true, fl_a / 4);
    }
    k_diag_shift_r<<<(unsigned)B, 256, 0, s>>>(rptr, n, n, trace_c + (size_t)nx * nw);
    ++launch_counter();
    potrf_batched_r(h, rptr, ar, n, n, lndet_c + (size_t)nx * nw, info + nq + (size_t)nx * nw, tc);
  }
  for (int pos = 0; pos < nql; ++pos) {   // to the flat (q, omega) order
    const int q = qlist[order[pos]];
    LR_CUDA(cudaMemcpyAsync(lndet + (size_t)q * nw, lndet_c + (size_t)pos * nw, nw * 8, cudaMemcpyDeviceToDevice, s));
    LR_CUDA(cudaMemcpyAsync(trace + (size_t)q * nw, trace_c + (size_t)pos * nw, nw * 8, cudaMemcpyDeviceToDevice, s));
  }
  for (int q : qlist) {   // the integrands of -q
    const int p = h.mesh.neg(q);
    if (p == q || h.vq_sym != 1) continue;
    LR_CUDA(cudaMemcpyAsync(lndet + (size_t)p * nw, lndet + (size_t)q * nw, nw * 8, cudaMemcpyDeviceToDevice, s));
    LR_CUDA(cudaMemcpyAsync(trace + (size_t)p * nw, trace + (size_t)q * nw, nw * 8, cudaMemcpyDeviceToDevice, s));
  }
  k_energy<<<1, 1, 0, s>>>(lndet, trace, wo, wqd, nq, nw, out);
  ++launch_counter();
  LR_CUDA(cudaGetLastError());
  std::vector<double> res(1 + nq + nw);
  std::vector<int> inf(nq + (size_t)nq * nw);
  int e_host = 0;
  LR_CUDA(cudaMemcpyAsync(res.data(), out, res.size() * 8, cudaMemcpyDeviceToHost, s));
  LR_CUDA(cudaMemcpyAsync(inf.data(), info, inf.size() * 4, cudaMemcpyDeviceToHost, s));
  LR_CUDA(cudaMemcpyAsync(&e_host, err, 4, cudaMemcpyDeviceToHost, s));
  LR_CUDA(cudaStreamSynchronize(s));
  if (e_host) return LIBRPA_E_TIMEOUT;
  for (int v : inf)
    if (v) return LIBRPA_E_NOT_PD;
  *ec = res[0];
  if (ec_q)
    for (int q = 0; q < nq; ++q) ec_q[q] = res[1 + q];
  if (ec_w)
    for (int k = 0; k < nw; ++k) ec_w[k] = res[1 + nq + k];
  // flop count of this stage (complex MAC = 8 real flops, real MAC = 2): per q (4/3 n^3 real for
  // the Cholesky of V), per (q, omega): W = chi0 L on the tiles A needs (n^3/3 MAC), L^H W lower
  // (n^3/6 MAC), Cholesky (n^3/6 MAC)
  const double n3 = (double)n * n * n;
  const double macs = n3 / 3 + n3 / 6 + n3 / 6;
  h.stats.flop_ec = nql * (8.0 * n3 / 6.0) + (double)nx * nw * 8.0 * macs + (double)(nql - nx) * nw * 2.0 * macs;
  return LIBRPA_OK;
}

}  // namespace librpa

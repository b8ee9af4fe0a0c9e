// O assembly of the chi0 contraction (k_chi0.cu) on the tensor cores.
//
// Per nu of V, O_nu[i][kap] is the sum of two products over K = 2 n_V:
//   term 1:  Lm[i][t] . Nt_nu[t][kap]   Lm = [A_UV(R) | B_UV(R)],  Nt = [N[G^occ]; N[G^vir]] at the union
//                                       column of kap
//   term 2:  LX_nu[i][t] . RG[t][kap]   LX = [X^A_nu | X^B_nu] (rows of U),  RG = [B_{V,kap}; A_{V,kap}](R1 - R)
// Every row of an operand (i or kap, over t) is scaled by a power of two 2^-E (E: its largest |value| < 2^E) and cut
// into S balanced base-256 digits x = sum_s d_s 2^{-7-8(s-1)}, |d_s| <= 128 (exact in BF16); the digit products
// of one diagonal s + t are summed exactly in FP32 (|sum| <= S * 32 * 2^14 <= 2^22), the diagonals folded into an
// integer per term, the two terms aligned to the larger scale and converted to FP64 once (8 planes: each
// term converted, then added).
//
// Two steps:
//   k_split_n, k_split_x: the digit planes of N and X, once per point (N serves every U that holds the union
//     column, X every tile of U).  HBM-bound.
//   k_oasm<S>: one CTA per (point, V, U, tile of 128 rows kap).  tcgen05.mma with the kap rows as M = 128, the
//     i of U as N (16 per plane, the planes stacked: plane s of A meets all S + 1 - s planes of B in one MMA of
//     N = 16 (S + 1 - s)), K = 32.  RG and Lm stay in shared memory; a TMA warp streams N and X planes of two nu at a
//     time (one box of 2 nu x S planes x 8 rows per row group, so a tile gathers U's columns from the union), one lane
//     issues the MMAs, 16 warps fold and store.
// The kernel is bound by the folding of the diagonal sums (integer and FP32 instructions) and by the
// L2 -> shared-memory traffic of the N planes, not by the MMAs.
#include <algorithm>
#include <cstring>
#include <type_traits>

#include "internal.h"
#include "oasm.h"
#include "tc.h"

namespace librpa {
namespace oasm {
namespace {

constexpr float kRintMagic = 12582912.0f;   // 1.5 * 2^23: (x + M) - M rounds |x| < 2^22 to an integer

// E with max |value| < 2^E from the largest |hi| (0 for an all-zero row), kept in [-100, 100]
__device__ __forceinline__ int tc_expo(float m) {
  if (!(m > 0.f)) return 0;
  const int be = (__float_as_int(m) >> 23) & 0xff;
  return min(100, max(-100, be - 126));
}
__device__ __forceinline__ float tc_pow2(int k) { return __int_as_float((k + 127) << 23); }   // |k| <= 126

// S digits of (h + l) 2^-E into d[] (sc7 = 2^{7-E}, sc15 = 2^{15-E})
template <int S>
__device__ __forceinline__ void tc_digits(float h, float l, float sc7, float sc15, float *d) {
  float t = h * sc7;
  float dd = (t + kRintMagic) - kRintMagic;
  float r = t - dd;
  d[0] = dd;
#pragma unroll
  for (int s = 1; s < S; ++s) {
    if (s == 2) r = fmaf(l, sc15, r);   // the low part, in units of the third digit
    t = r * 256.f;
    dd = (t + kRintMagic) - kRintMagic;
    r = t - dd;
    d[s] = dd;
  }
}

// The element type of the operands: (hi, lo) FP32 pairs with up to 5 planes (N and X arrive so from their GEMMs, G as
// FP64 turned into pairs; the low part joins the digits after the second, error below 2^-39 of the row
// maximum), FP64 numbers with 8 planes.  NANS: G or C holds an infinity or a NaN (known on the host); the exponent of a row
// with one is then 1025, as it always is with 8 planes (in every kernel this test costs 2% of the slab's SPLIT energy).
template <int S, bool NANS>
struct Elem {
  using T = float2;
  __device__ static T zero() { return make_float2(0.f, 0.f); }
  __device__ static T load(const double *p) { return *reinterpret_cast<const float2 *>(p); }
  __device__ static T from_g(double v) {
    const float h = __double2float_rn(v);
    return make_float2(h, __double2float_rn(v - (double)h));
  }
  using M = float;   // running maximum
  __device__ static M m0() { return 0.f; }
  __device__ static M mx(M m, T v) { return larger(m, fabsf(v.x)); }
  __device__ static M both(M m, int o) { return larger(m, __shfl_xor_sync(0xffffffffu, m, o)); }
  __device__ static int expo(M m) { return NANS && !(m < __int_as_float(0x7F800000)) ? 1025 : tc_expo(m); }
  __device__ static float larger(float a, float b) {
    if (!NANS) return fmaxf(a, b);
    return a != a || a > b ? a : b;   // NaN if either is
  }
  // digits of 8 elements, 16 bytes per plane
  __device__ static void digits8(const T *v, int E, uint4 *w) {
    const float sc7 = tc_pow2(7 - E), sc15 = tc_pow2(15 - E);
    float d[8][S];
#pragma unroll
    for (int q = 0; q < 8; ++q) tc_digits<S>(v[q].x, v[q].y, sc7, sc15, d[q]);
#pragma unroll
    for (int s = 0; s < S; ++s)
      w[s] = make_uint4(pack_bf16(d[0][s], d[1][s]), pack_bf16(d[2][s], d[3][s]), pack_bf16(d[4][s], d[5][s]),
                        pack_bf16(d[6][s], d[7][s]));
  }
};
template <bool NANS>
struct Elem<oz::S_WIDE, NANS> {
  using T = double;
  __device__ static T zero() { return 0.0; }
  __device__ static T load(const double *p) { return *p; }
  __device__ static T from_g(double v) { return v; }
  using M = int;
  __device__ static M m0() { return 0; }
  __device__ static M mx(M m, T v) { return max(m, biased_exp(v)); }
  __device__ static M both(M m, int o) { return max(m, __shfl_xor_sync(0xffffffffu, m, o)); }
  __device__ static int expo(M m) { return m - 1022; }   // 1025: the row holds an infinity or a NaN
  __device__ static void digits8(const T *v, int E, uint4 *w) {
    constexpr int S = oz::S_WIDE;
    unsigned *u = reinterpret_cast<unsigned *>(w);
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      float d0[S], d1[S];
      make_digits<S>(v[2 * q], E, d0);
      make_digits<S>(v[2 * q + 1], E, d1);
#pragma unroll
      for (int s = 0; s < S; ++s) u[4 * s + q] = pack_bf16(d0[s], d1[s]);
    }
  }
};

// Digit planes of N: laid out [(p, nu)][plane][union column][t], t = (g, j); row exponents [(p, nu)][union column].  Two lanes per row (16 t each), 16 consecutive
// columns per warp; block = 128 columns of one (p, nu).
template <int S, bool NANS>
__global__ void __launch_bounds__(256) k_split_n(OArgs a, const int *__restrict__ aux_atom, __nv_bfloat16 *dig,
                                                 int *expo) {
  using E_ = Elem<S, NANS>;
  const int p = blockIdx.x / a.naux, nug = blockIdx.x % a.naux, V = aux_atom[nug], nu = nug - a.aux_off[V];
  const int lane = threadIdx.x & 31, h = lane >> 4;
  const int col = blockIdx.y * 128 + (threadIdx.x >> 5) * 16 + (lane & 15);
  const int nV = a.n_ao[V], two = 2 * nV;
  const double *N0 = a.N + p * a.n_sz_p + a.n_off[V] + (size_t)nu * nV * a.m_all + col, *N1 = N0 + a.n_sz_g;
  const bool live = col < a.m_all;
  typename E_::T v[16];
  typename E_::M m = E_::m0();
#pragma unroll
  for (int q = 0; q < 16; ++q) {
    const int t = 16 * h + q;
    v[q] = E_::zero();
    if (live && t < two) v[q] = E_::load(t < nV ? N0 + (size_t)t * a.m_all : N1 + (size_t)(t - nV) * a.m_all);
    m = E_::mx(m, v[q]);
  }
  m = E_::both(m, 16);
  if (!live) return;
  const int E = E_::expo(m);
  const long long row = ((long long)p * a.naux + nug) * a.m_all + col;
  if (h == 0) expo[row] = E;
  __nv_bfloat16 *out = dig + (((size_t)p * a.naux + nug) * S * a.m_all + col) * 32 + 16 * h;
#pragma unroll
  for (int c = 0; c < 2; ++c) {
    uint4 w[S];
    E_::digits8(v + 8 * c, E, w);
#pragma unroll
    for (int s = 0; s < S; ++s) *reinterpret_cast<uint4 *>(out + (size_t)s * a.m_all * 32 + 8 * c) = w[s];
  }
}

// Digit planes of X: [(p, nu)][plane][16 U + i][t]; two lanes per row.  Rows i >= n_U are left as they are (the MMA
// columns they give are not read).
template <int S, bool NANS>
__global__ void __launch_bounds__(256) k_split_x(OArgs a, const int *__restrict__ aux_atom,
                                                 const int *__restrict__ ao_row, __nv_bfloat16 *dig, int *expo) {
  using E_ = Elem<S, NANS>;
  const int p = blockIdx.x / a.naux, nug = blockIdx.x % a.naux, V = aux_atom[nug], nu = nug - a.aux_off[V];
  const int lane = threadIdx.x & 31, h = lane >> 4;
  const int ao = blockIdx.y * 128 + (threadIdx.x >> 5) * 16 + (lane & 15);
  const int nV = a.n_ao[V], two = 2 * nV;
  const size_t ldx = (size_t)a.n_aux[V] * nV;
  const double *XB = a.X + p * a.x_sz_p + a.x_off[V] + ao * ldx + (size_t)nu * nV, *XA = XB + a.x_sz_g;
  const bool live = ao < a.nao;
  typename E_::T v[16];
  typename E_::M m = E_::m0();
#pragma unroll
  for (int q = 0; q < 16; ++q) {
    const int t = 16 * h + q;
    v[q] = E_::zero();
    if (live && t < two) v[q] = E_::load(t < nV ? XA + t : XB + (t - nV));
    m = E_::mx(m, v[q]);
  }
  m = E_::both(m, 16);
  if (!live) return;
  const int E = E_::expo(m);
  const long long row = ((long long)p * a.naux + nug) * (a.natoms * kMaxAo) + ao_row[ao];
  if (h == 0) expo[row] = E;
  __nv_bfloat16 *out = dig + (((size_t)p * a.naux + nug) * S * a.natoms * kMaxAo + ao_row[ao]) * 32 + 16 * h;
#pragma unroll
  for (int c = 0; c < 2; ++c) {
    uint4 w[S];
    E_::digits8(v + 8 * c, E, w);
#pragma unroll
    for (int s = 0; s < S; ++s) *reinterpret_cast<uint4 *>(out + (size_t)s * a.natoms * kMaxAo * 32 + 8 * c) = w[s];
  }
}

// ------------------------------------------------------------------ the products
constexpr int kEpi = 16, kThreads = 32 * (kEpi + 2);
__host__ __device__ constexpr int op_bytes(int S) { return kTileGroups * S * 512; }   // 128 rows: groups of 8 rows x S planes x 64 bytes
__host__ __device__ constexpr int x_bytes(int S) { return S * kMaxAo * 64; }          // S planes of 16 rows x 64 bytes
__host__ __device__ constexpr int static_size(int S) { return op_bytes(S) + x_bytes(S); }   // RG and Lm
// nu per stage: half the copies to issue, 64-byte rows fetched two nu at a time, where two stages fit (k_oasm of the graphene
// slab 1.08 -> 1.04 ms a point with 5 planes, 0.97 -> 0.92 with 3).
__host__ __device__ constexpr int nus(int S) { return S == oz::S_WIDE ? 1 : 2; }
__host__ __device__ constexpr int stage_size(int S) { return nus(S) * static_size(S); }
__host__ __device__ constexpr int ring(int S) { return S == 3 ? 3 : 2; }
__host__ __device__ constexpr int smem_size(int S) { return static_size(S) + ring(S) * stage_size(S) + 512; }
__host__ __device__ constexpr int slot_cols(int S) { return 2 * S * kMaxAo; }         // TMEM columns of one nu: two terms, S diagonals, 16 i
__host__ __device__ constexpr int slots(int S) { return 512 / slot_cols(S); }

// sum_d A_d 2^{8(N-1-d)} of N exact integer-valued FP32 diagonal sums (|A_d| <= 2^22): the bits of A_d + 1.5 2^23
// are A_d plus a constant, so the constants are subtracted from the sum once (mod 2^64)
template <int N>
__device__ __forceinline__ long long fold_sums(const uint32_t *a) {
  constexpr unsigned long long kOne = 0x4B400000ull;
  unsigned long long c = 0, T = 0;
#pragma unroll
  for (int d = 0; d < N; ++d) {
    const unsigned b = __float_as_uint(__uint_as_float(a[4 * d]) + kRintMagic);
    c += kOne << (8 * (N - 1 - d));
    T += (unsigned long long)b << (8 * (N - 1 - d));
  }
  return (long long)(T - c);
}

// element x of the two terms' sums r1, r2 ([diagonal][4] registers), scales 2^E1, 2^E2
template <int S>
__device__ __forceinline__ double combine(const uint32_t (&r1)[S][4], const uint32_t (&r2)[S][4], int x, int E1, int E2) {
  if constexpr (S == oz::S_WIDE) {
    return i96_to_f64(fold_sums<4>(&r1[0][x]), fold_sums<4>(&r1[4][x]), E1 - 14 - 56) +
           i96_to_f64(fold_sums<4>(&r2[0][x]), fold_sums<4>(&r2[4][x]), E2 - 14 - 56);
  } else {
    const long long T1 = fold_sums<S>(&r1[0][x]), T2 = fold_sums<S>(&r2[0][x]);
    // the smaller scale's sum rounded to the larger scale, half up
    const bool one = E1 >= E2;
    const long long big = one ? T1 : T2, small = one ? T2 : T1;
    const int E = max(E1, E2), sh = min(E - min(E1, E2), 62);
    const long long T = big + ((((small << 1) >> sh) + 1) >> 1);
    // the conversion on the FP64 pipe, which is idle otherwise (one instruction in place of ~25); the scales are
    // within 2^+-200 (tc_expo), far from the ends of the exponent range
    const long long bits = __double_as_longlong((double)T) + ((long long)(E - 14 - 8 * (S - 1)) << 52);
    return __longlong_as_double(T == 0 ? 0ll : bits);
  }
}

// NANS (see Elem; with 8 planes always): outputs of rows with the exponent 1025 are NaN, whatever their digits gave
template <int S, bool NANS>
__global__ void __launch_bounds__(kThreads, 1)
    k_oasm(OArgs a, Tables tb, const __grid_constant__ CUtensorMap nmap, const __grid_constant__ CUtensorMap xmap,
           const int *__restrict__ nexp, const int *__restrict__ xexp, int *rexp, int *err, uint64_t stall_ns) {
  using E_ = Elem<S, NANS>;
  constexpr int NST = ring(S), NSL = slots(S), SL = slot_cols(S);
  constexpr int NU = nus(S);
  constexpr uint32_t OPB = op_bytes(S), XB_ = x_bytes(S), FIXED = static_size(S), STAGE = stage_size(S);
  extern __shared__ uint8_t smem_raw[];
  __shared__ uint64_t full[NST], empty[NST], tfull[2][NSL], tempty[NSL], mdone, never;
  __shared__ uint32_t tmem_slot;
  __shared__ volatile int abort_flag;
  __shared__ int s_e1[kMaxAo], s_box[kTileGroups];
  __shared__ int s_groups;
  // U and its tiles run fastest: the CTAs in flight share the N planes of a few V in the L2
  const int uv = blockIdx.x / tb.max_tiles;
  const int U = uv % a.natoms, V = (uv / a.natoms) % a.natoms, p = uv / (a.natoms * a.natoms);
  const int tile = tb.tile_off[U] + (int)(blockIdx.x % tb.max_tiles);
  if (tile >= tb.tile_off[U + 1]) return;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int nU = a.n_ao[U], nV = a.n_ao[V], two = 2 * nV, nauxV = a.n_aux[V], mU = a.m[U];
  double *Ob = a.O + p * a.o_sz_p + a.o_off[U];
  const int ldo = o_pitch(nU, mU);
  if (a.zero) {   // under screening: a tile whose 64-column chunks are all exactly zero
    const Group g0 = tb.groups[(size_t)tile * kTileGroups];
    int k1 = g0.kap;
    for (int g = 0; g < kTileGroups; ++g) {
      const Group gg = tb.groups[(size_t)tile * kTileGroups + g];
      if (gg.live) k1 = gg.kap + gg.live;
    }
    const unsigned char *z = a.zero + ((size_t)(p * a.natoms + U) * a.natoms + V) * a.zero_chunks;
    bool all = true;
    for (int c = g0.kap / 64; c * 64 < k1; ++c) all = all && z[c];
    if (all) {
      const int w = k1 - g0.kap;
      for (long long e = tid; e < (long long)nauxV * nU * w; e += kThreads) {
        const int col = (int)(e % w);
        const long long r = e / w;
        Ob[(size_t)(a.aux_off[V] + r / nU) * ldo + (size_t)(r % nU) * mU + g0.kap + col] = 0.0;
      }
      return;
    }
  }
  uint8_t *smem = (uint8_t *)(((uintptr_t)smem_raw + 511) & ~(uintptr_t)511);   // 64-byte swizzle: 512-byte atoms
  uint8_t *sRG = smem, *sLm = smem + OPB;   // static operands, then the ring
  // exponent, packed and union column of the tile's rows, in the first stage until the epilogue has read them
  int *s_f2 = reinterpret_cast<int *>(smem + FIXED), *s_kap = s_f2 + 128, *s_urow = s_kap + 128;
  if (tid == 0) {
    for (int s = 0; s < NST; ++s) {
      mbar_init(&full[s], 1);
      mbar_init(&empty[s], 1);
    }
    for (int s = 0; s < NSL; ++s) {
      mbar_init(&tfull[0][s], 1);
      mbar_init(&tfull[1][s], 1);
      mbar_init(&tempty[s], 8);
    }
    mbar_init(&mdone, 1);
    mbar_init(&never, 1);
    abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == kEpi) tmem_alloc(&tmem_slot, 512);
  if (warp == kEpi + 1 && lane < kTileGroups) {   // the tile's row groups
    const Group g = tb.groups[(size_t)tile * kTileGroups + lane];
    s_box[lane] = g.live ? g.urow : -1;
    const unsigned m = __ballot_sync(0xffffu, g.live > 0);
    if (lane == 0) s_groups = __popc(m);
  }
  const Point pt = a.pts[p];
  const size_t n2 = (size_t)a.nao * a.nao;
  const double *GB = a.G + ((size_t)pt.itau * a.nR_stride) * n2;                 // G^occ(tau)
  const double *GA = a.G + a.g_gstride + ((size_t)pt.itau * a.nR_stride) * n2;   // G^vir(tau)
  const int aoU = a.ao_off[U], aoV = a.ao_off[V];
  // RG digits: four threads per row kap, 8 columns t each; 16-byte pieces swizzled as TMA would
  if (tid < 512) {
    const int r = tid >> 2, c = tid & 3;
    const Group g = tb.groups[(size_t)tile * kTileGroups + (r >> 3)];
    const bool live = (r & 7) < g.live;
    const int kc = g.kap + (r & 7);
    const int *kp = a.kap + 6 * (a.kap_off[U] + (live ? kc : 0));
    auto fold = [](int x, int nn) { int q = x % nn; return q < 0 ? q + nn : q; };
    const int iR = (fold(kp[1] - pt.R[0], a.n1) * a.n2 + fold(kp[2] - pt.R[1], a.n2)) * a.n3 + fold(kp[3] - pt.R[2], a.n3);
    typename E_::T v[8];
    typename E_::M m = E_::m0();
#pragma unroll
    for (int q = 0; q < 8; ++q) {
      const int t = 8 * c + q;
      v[q] = E_::zero();
      if (live && t < two)
        v[q] = E_::from_g((t < nV ? GB : GA)[(size_t)iR * n2 + (size_t)(aoV + (t < nV ? t : t - nV)) * a.nao + kp[4]]);
      m = E_::mx(m, v[q]);
    }
    m = E_::both(E_::both(m, 1), 2);
    const int E = E_::expo(m);
    if (c == 0) {
      s_f2[r] = E;
      s_kap[r] = live ? kc : -1;
      s_urow[r] = g.urow + (r & 7);
    }
    uint4 w[S];
    E_::digits8(v, E, w);
#pragma unroll
    for (int s = 0; s < S; ++s)
      *reinterpret_cast<uint4 *>(sRG + (r >> 3) * (S * 512) + s * 512 + (r & 7) * 64 + ((c ^ ((r >> 1) & 3)) << 4)) = w[s];
  }
  if (tid < 64) {   // Lm digits: rows i, planes of 16 rows one after the other
    const int i = tid >> 2, c = tid & 3;
    typename E_::T v[8];
    typename E_::M m = E_::m0();
#pragma unroll
    for (int q = 0; q < 8; ++q) {
      const int t = 8 * c + q;
      v[q] = E_::zero();
      if (i < nU && t < two)
        v[q] = E_::from_g((t < nV ? GA : GB)[(size_t)pt.iR * n2 + (size_t)(aoU + i) * a.nao + aoV + (t < nV ? t : t - nV)]);
      m = E_::mx(m, v[q]);
    }
    m = E_::both(E_::both(m, 1), 2);
    const int E = E_::expo(m);
    if (c == 0) s_e1[i] = E;
    uint4 w[S];
    E_::digits8(v, E, w);
#pragma unroll
    for (int s = 0; s < S; ++s)
      *reinterpret_cast<uint4 *>(sLm + s * 1024 + i * 64 + ((c ^ ((i >> 1) & 3)) << 4)) = w[s];
  }
  asm volatile("fence.proxy.async.shared::cta;" ::: "memory");   // the MMAs read what was stored here
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = tmem_slot;
  int kap = -1, f2 = 0, urow = 0;
  if (warp < kEpi) {
    const int r = (warp & 3) * 32 + lane;
    kap = s_kap[r];
    f2 = s_f2[r];
    urow = s_urow[r];
  }
  asm volatile("fence.proxy.async.shared::cta;" ::: "memory");   // the copies come after these reads
  __syncthreads();
  const long long nu0 = (long long)p * a.naux + a.aux_off[V];
  if (warp == kEpi) {
    if (elect_one()) {   // TMA producer: N rows of the tile's groups and the 16 X rows of U, per nu
      const int ng = s_groups;
      const int nblk = (nauxV + NU - 1) / NU;   // (the nu beyond V's last in a block are loaded, not used)
      int it = 0;
      for (; it < nblk; ++it) {
        const int st = it % NST;
        if (abort_flag || !mbar_wait(&empty[st], (uint32_t)(((it / NST) & 1) ^ 1), WAIT_NS, &abort_flag)) {
          abort_flag = 1;
          break;
        }
        uint8_t *sn = smem + FIXED + st * STAGE, *sx = sn + NU * OPB;
        mbar_expect_tx(&full[st], NU * ((uint32_t)ng * S * 512 + XB_));
        const int nu = (int)nu0 + it * NU;
        for (int g = 0; g < ng; ++g) tma_load_4d(sn + g * (NU * S * 512), &nmap, &full[st], 0, s_box[g], 0, nu);
        tma_load_4d(sx, &xmap, &full[st], 0, U * kMaxAo, 0, nu);
      }
      // after a failure: wait for the copies still in flight (the last NST issued stages)
      if (abort_flag)
        for (int i = it > NST ? it - NST : 0; i < it; ++i) mbar_wait(&full[i % NST], (uint32_t)((i / NST) & 1), WAIT_NS);
    }
  } else if (warp == kEpi + 1) {
    if (elect_one()) {   // MMA issuer
      if (stall_ns) {   // testing only: a barrier nothing arrives at
        mbar_wait(&never, 0, stall_ns, &abort_flag);
        abort_flag = 1;
      }
      const int ks = (two + 15) / 16;
      const uint32_t rg = smem_u32(sRG), lm = smem_u32(sLm);
      for (int it = 0; it < nauxV; ++it) {
        const int blk = it / NU, st = blk % NST, sl = it % NSL;
        if (it >= NSL && (abort_flag || !mbar_wait(&tempty[sl], (uint32_t)((it / NSL - 1) & 1), WAIT_NS, &abort_flag))) {
          abort_flag = 1;
          break;
        }
        if (abort_flag || !mbar_wait(&full[st], (uint32_t)((blk / NST) & 1), WAIT_NS, &abort_flag)) {
          abort_flag = 1;
          break;
        }
        tc_fence_after();
        const uint32_t s0 = smem_u32(smem + FIXED + st * STAGE), sn = s0 + it % NU * (S * 512), sx = s0 + NU * OPB + it % NU * XB_,
                       d = tmem + sl * SL;
        const uint64_t dn = smem_desc64(sn, NU * S * 512), dr = smem_desc64(rg, S * 512), dl = smem_desc64(lm), dx = smem_desc64(sx);
#pragma unroll
        for (int j = 0; j < 2; ++j) {
          if (j >= ks) break;
#pragma unroll
          for (int s = 0; s < S; ++s) {   // plane s of A by planes 0 .. S - 1 - s of B, into the diagonals s ..
            const uint32_t ide = idesc(kMaxAo * (S - s), false), o = (s * 512 + 32 * j) / 16;
            if (j == 0 && s == 0) {
              umma(d, dn, dl, ide, 0u);
              umma(d + S * kMaxAo, dr, dx, ide, 0u);
            } else {
              umma_add(d + s * kMaxAo, dn + o, dl + 2 * j, ide);
              umma_add(d + (S + s) * kMaxAo, dr + o, dx + 2 * j, ide);
            }
          }
        }
        if (it % NU == NU - 1) umma_commit(&empty[st]);
        umma_commit(&tfull[it & 1][sl]);
      }
      if (abort_flag) {   // after a failure: wait for the MMAs already issued
        umma_commit(&mdone);
        mbar_wait(&mdone, 0, WAIT_NS);
      }
    }
  } else {
    // epilogue: warps 0-7 the even nu, 8-15 the odd ones; thread = row kap, half of the i each.  A slot has a tfull barrier
    // for each of the two groups, which waits for every phase of its own: with an odd number of slots the groups take a
    // slot in turn, and of one barrier a group would wait for every other phase, the parity of the one before passing for it.
    const int grp = warp >> 3, quad = warp & 3, half = (warp >> 2) & 1;
    const bool any = __any_sync(0xffffffffu, kap >= 0);
    const int per = (nU + 1) / 2, c0 = half * per, c1 = min(nU, c0 + per);
    // exponents: of the lane's N row, and of row i = lane of Lm and X; those of the warp's next nu are fetched while
    // this one is folded
    const int i16 = lane & (kMaxAo - 1), e1_lane = s_e1[i16];
    const int *np_ = nexp + nu0 * a.m_all + urow, *xp_ = xexp + (nu0 * a.natoms + U) * kMaxAo + i16;
    auto next_f1 = [&](int i) { return kap >= 0 && i < nauxV ? np_[(size_t)i * a.m_all] : 0; };
    auto next_e2 = [&](int i) { return i < nauxV ? xp_[(size_t)i * a.natoms * kMaxAo] : 0; };
    int f1n = next_f1(grp), e2n = next_e2(grp);
    for (int it = grp; it < nauxV; it += 2) {
      const int sl = it % NSL, f1 = f1n;
      const int e_lane = (int)((unsigned)e1_lane << 16) | (e2n & 0xFFFF);   // both, one shuffle per i (|e| <= 1100)
      f1n = next_f1(it + 2);
      e2n = next_e2(it + 2);
      bool ok = !abort_flag && mbar_wait(&tfull[grp][sl], (uint32_t)(it / (NSL % 2 ? 2 * NSL : NSL) & 1), WAIT_NS, &abort_flag);
      ok = __all_sync(0xffffffffu, ok);
      if (!ok) {
        abort_flag = 1;
        break;
      }
      tc_fence_after();
      int emax = 0;   // upper word of the largest |output| of this lane: its biased exponent
      if (any) {
        const uint32_t tb0 = tmem + ((uint32_t)(32 * quad) << 16) + sl * SL;
        double *orow = Ob + (size_t)(a.aux_off[V] + it) * ldo + kap;
#pragma unroll 1
        for (int c = c0; c < c1; c += 4) {
          uint32_t r1[S][4], r2[S][4];
          int e[4];
#pragma unroll
          for (int d = 0; d < S; ++d) {
            tmem_ld(tb0 + d * kMaxAo + c, r1[d]);
            tmem_ld(tb0 + (S + d) * kMaxAo + c, r2[d]);
          }
#pragma unroll
          for (int x = 0; x < 4; ++x) e[x] = __shfl_sync(0xffffffffu, e_lane, c + x & (kMaxAo - 1));
#pragma unroll
          for (int d = 0; d < S; ++d) {
            tmem_ld_wait(r1[d]);
            tmem_ld_wait(r2[d]);
          }
          // N elements from x0 on, side by side (a branch per element would fold them one after the other); those
          // beyond c1 are not stored
          auto fold = [&](auto x0_, auto n_) {
            constexpr int x0 = decltype(x0_)::value, N = decltype(n_)::value;
            double o[N];
#pragma unroll
            for (int x = x0; x < x0 + N; ++x) {
              const int e1 = e[x] >> 16, e2 = (int)(short)e[x];
              o[x - x0] = combine<S>(r1, r2, x, e1 + f1, e2 + f2);
              if ((S == oz::S_WIDE || NANS) && max(max(e1, f1), max(e2, f2)) > 1024)
                o[x - x0] = __longlong_as_double(0x7FF8000000000000ll);
            }
#pragma unroll
            for (int x = x0; x < x0 + N; ++x)
              if (kap >= 0 && c + x < c1) {
                orow[(size_t)(c + x) * mU] = o[x - x0];
                emax = max(emax, __double2hiint(o[x - x0]) & 0x7FFFFFFF);
              }
          };
          using std::integral_constant;
          if constexpr (S == oz::S_WIDE) {   // (one at a time: the two-word sums of more do not fit the registers)
            fold(integral_constant<int, 0>(), integral_constant<int, 1>());
            if (c + 1 < c1) fold(integral_constant<int, 1>(), integral_constant<int, 1>());
            if (c + 2 < c1) fold(integral_constant<int, 2>(), integral_constant<int, 1>());
            if (c + 3 < c1) fold(integral_constant<int, 3>(), integral_constant<int, 1>());
          } else if (c + 2 < c1) {
            fold(integral_constant<int, 0>(), integral_constant<int, 4>());
          } else {
            fold(integral_constant<int, 0>(), integral_constant<int, 2>());
          }
        }
      }
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(&tempty[sl]);
      // the row (p, U, nu) of the final contraction's O operand
      emax = __reduce_max_sync(0xffffffffu, emax) >> 20;
      if (lane == 0 && emax > 0) atomicMax(rexp + ((size_t)p * a.natoms + U) * a.naux + a.aux_off[V] + it, emax - 1022);
    }
  }
  __syncthreads();
  if (abort_flag && tid == 0) atomicExch(err, 1);
  tc_fence_before();
  __syncthreads();
  if (warp == kEpi) tmem_dealloc(tmem, 512);
}

template <int S, bool NANS = false>
void launch(const OArgs &a, const Tables &t, int np, oz::Sliced &nd, oz::Sliced &xd, int *expo, int *err, uint64_t stall_ns,
            cudaStream_t s) {
  static_assert(smem_size(S) <= 227 * 1024, "k_oasm: shared memory");
  const unsigned rows = (unsigned)(np * a.naux);
  k_split_n<S, NANS><<<dim3(rows, (unsigned)((a.m_all + 127) / 128)), 256, 0, s>>>(
      a, t.aux_atom, (__nv_bfloat16 *)nd.digits, nd.expo);
  k_split_x<S, NANS><<<dim3(rows, (unsigned)((a.nao + 127) / 128)), 256, 0, s>>>(
      a, t.aux_atom, t.ao_row, (__nv_bfloat16 *)xd.digits, xd.expo);
  LR_CUDA(cudaFuncSetAttribute(k_oasm<S, NANS>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem_size(S)));
  k_oasm<S, NANS><<<(unsigned)t.max_tiles * (unsigned)(np * a.natoms * a.natoms), kThreads, smem_size(S), s>>>(
      a, t, oz::make_map_nested(nd.digits, a.m_all, S, (int)rows, 8, nus(S)),
      oz::make_map_nested(xd.digits, a.natoms * kMaxAo, S, (int)rows, kMaxAo, nus(S)), nd.expo, xd.expo, expo, err,
      stall_ns);
  launch_counter() += 3;
  LR_CUDA(cudaGetLastError());
}

}  // namespace

void run(int S, const OArgs &a, const Tables &t, int np, oz::Sliced &nd, oz::Sliced &xd, int *expo, int *err,
         bool nans, uint64_t stall_ns, cudaStream_t s) {
  oz::init();
  if (S == 3 && nans)
    launch<3, true>(a, t, np, nd, xd, expo, err, stall_ns, s);
  else if (S == 5 && nans)
    launch<5, true>(a, t, np, nd, xd, expo, err, stall_ns, s);
  else if (S == 3)
    launch<3>(a, t, np, nd, xd, expo, err, stall_ns, s);
  else if (S == 5)
    launch<5>(a, t, np, nd, xd, expo, err, stall_ns, s);
  else
    launch<oz::S_WIDE>(a, t, np, nd, xd, expo, err, stall_ns, s);
}

}  // namespace oasm
}  // namespace librpa

// FP64-accurate GEMM on the BF16 tensor cores of sm_103a (see ozgemm.h for the scheme).
//
// Operands are split once into BF16 digit planes (k_row_expo + k_digits, or k_plain for plain
// BF16); the GEMM kernel streams them with TMA (cp.async.bulk.tensor) into a shared-memory ring
// and multiplies every digit pair with tcgen05.mma (kind::f16, BF16 x BF16 -> FP32, M = 128, K = 16,
// planes stacked along N) into the TMEM accumulator of its diagonal; flush groups (the largest K range
// whose FP32 sums stay exact) are moved into exact int64 register sums, scaled by
// 2^(E_A + E_B - 14 - 8(S-1)) into FP64 at the end.  Every wait on an mbarrier is bounded by the
// global timer; on a timeout the kernel records the failure in *err, waits (bounded) for its own
// copies in flight, frees TMEM and returns.
#include <cuda.h>
#include <cudaTypedefs.h>

#include <algorithm>
#include <cmath>
#include <cstdint>
#include <cstring>
#include <map>
#include <mutex>
#include <string>
#include <tuple>
#include <type_traits>
#include <utility>

#include "internal.h"
#include "ozgemm.h"
#include "tc.h"

namespace librpa {
namespace oz {
namespace {

// ------------------------------------------------------------------ splitting

struct RealSrc {
  const double *p;
  long long ld, bstride;
  int rows_pb;
  bool trans;
  __device__ double get(int r, int k) const {
    const int b = r / rows_pb, rr = r % rows_pb;
    const double *q = p + b * bstride;
    return trans ? q[(long long)k * ld + rr] : q[(long long)rr * ld + k];
  }
};

struct CplxSrc {
  const double2 *p;
  long long ld, bstride;
  int rows_pb, op;
  bool as_a;
  __device__ double2 opget(const double2 *q, int i, int k) const {
    if (op == OP_N) return q[(long long)i * ld + k];
    if (op == OP_C) {
      const double2 z = q[(long long)i * ld + k];
      return make_double2(z.x, -z.y);
    }
    double2 z = q[(long long)k * ld + i];
    if (op == OP_H) z.y = -z.y;
    return z;
  }
  __device__ double get(int r, int kk) const {
    const int b = r / rows_pb, rr = r % rows_pb;
    const double2 *q = p + b * bstride;
    const int k = kk >> 1, cp = kk & 1;
    if (as_a) {
      const int i = rr >> 1, c = rr & 1;
      const double2 z = opget(q, i, k);
      return c == cp ? z.x : (c == 0 ? -z.y : z.y);
    }
    const double2 z = opget(q, k, rr);
    return cp ? z.y : z.x;
  }
};

// A'-form rows (as_a) of Z with element (i, k) times 2^-(eq[i] + eq[k])
struct CplxEqSrc {
  CplxSrc z;
  const int *eq;
  __device__ double get(int r, int kk) const {
    return scale_pow2(z.get(r, kk), -(eq[(r % z.rows_pb) >> 1] + eq[kk >> 1]));
  }
};

struct GatherDev {
  GatherSrc g;
  __device__ static int fold(int a, int n) {
    const int r = a % n;
    return r < 0 ? r + n : r;
  }
  __device__ double get(int r, int k) const {
    const int e = r / g.rows_per_entry, rr = r % g.rows_per_entry;
    const int V = e % g.natoms, gg = (e / g.natoms) % 2, p = e / (2 * g.natoms);
    if (k >= g.m[V]) return 0.0;
    const int *pt = g.pts + 5 * p;
    const int *c = g.lam + 6 * (g.lam_off[V] + k);
    int iR, row, col;
    if (g.kind == 0) {
      const int *u = g.uni + 6 * rr;
      iR = (fold(u[1] - pt[2] - c[1], g.n1) * g.n2 + fold(u[2] - pt[3] - c[2], g.n2)) * g.n3 +
           fold(u[3] - pt[4] - c[3], g.n3);
      row = c[5];
      col = u[5];
    } else {
      iR = (fold(pt[2] + c[1], g.n1) * g.n2 + fold(pt[3] + c[2], g.n2)) * g.n3 + fold(pt[4] + c[3], g.n3);
      row = rr;
      col = c[5];
    }
    const double *Gp = g.G + gg * g.g_gstride + ((long long)pt[1] * g.nR + iR) * g.nao * g.nao;
    return Gp[(long long)row * g.nao + col];
  }
};

struct RaggedSrc {
  const double *base;
  const long long *off;
  const int *Ke;
  int rows_pe;
  __device__ double get(int r, int k) const {
    const int e = r / rows_pe, rr = r % rows_pe;
    const int K = Ke[e];
    return k < K ? base[off[e] + (long long)rr * ((K + 1) & ~1) + k] : 0.0;
  }
};

// exponent of each row: one warp per row
template <class Src>
__global__ void k_row_expo(Src src, int rows, int K, int row0, int *expo) {
  const int w = (blockIdx.x * blockDim.x + threadIdx.x) >> 5, lane = threadIdx.x & 31;
  if (w >= rows) return;
  int m = 0;
  for (int k = lane; k < K; k += 32) m = max(m, biased_exp(src.get(w, k)));
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) m = max(m, __shfl_xor_sync(0xffffffffu, m, o));
  if (lane == 0) expo[row0 + w] = m - 1022;
}

// one row per blockIdx.x, 4 consecutive k per thread (kpad is a multiple of 8): the row's scale and
// source offsets are fetched once, each plane is written 8 bytes per thread
template <int S, class Src>
__global__ void __launch_bounds__(256) k_digits(Src src, int K, int kpad, int row0, long long plane, const int *expo,
                                                __nv_bfloat16 *dig) {
  const int r = blockIdx.x;
  const int k0 = (blockIdx.y * 256 + threadIdx.x) * 4;
  if (k0 >= kpad) return;
  const int E = expo[row0 + r];
  float d[4][S];
#pragma unroll
  for (int q = 0; q < 4; ++q) make_digits<S>(k0 + q < K ? src.get(r, k0 + q) : 0.0, E, d[q]);
  const long long o = ((long long)row0 + r) * kpad + k0;
#pragma unroll
  for (int s = 0; s < S; ++s) {
    const uint2 w = make_uint2(pack_bf16(d[0][s], d[1][s]), pack_bf16(d[2][s], d[3][s]));
    *reinterpret_cast<uint2 *>(dig + s * plane + o) = w;
  }
}

// Digit planes of ragged rows (the O operand): one block per row, 4 consecutive k per thread and pass, up to 3 passes'
// loads in flight before the first is split; rows start on 16 bytes (even pitch).  HBM-bound: 8 bytes read, 2 S written
// per element.
template <int S>
__global__ void __launch_bounds__(256) k_digits_ragged(RaggedSrc src, int kpad, long long plane, const int *__restrict__ expo,
                                                       __nv_bfloat16 *__restrict__ dig) {
  const int r = blockIdx.x, e = r / src.rows_pe, K = src.Ke[e], E = expo[r];
  const double *row = src.base + src.off[e] + (long long)(r % src.rows_pe) * ((K + 1) & ~1);
  __nv_bfloat16 *out = dig + (long long)r * kpad;
  for (int k1 = 0; k1 < kpad; k1 += 3 * 1024) {
    double2 v[3][2];
#pragma unroll
    for (int b = 0; b < 3; ++b)
#pragma unroll
      for (int q = 0; q < 2; ++q) {
        const int k = k1 + b * 1024 + threadIdx.x * 4 + 2 * q;
        v[b][q] = make_double2(0.0, 0.0);
        if (k < K) v[b][q] = __ldcs(reinterpret_cast<const double2 *>(row + k));
        if (k + 1 >= K) v[b][q].y = 0.0;   // the pad of an odd row
      }
#pragma unroll
    for (int b = 0; b < 3; ++b) {
      const int k = k1 + b * 1024 + threadIdx.x * 4;
      if (k >= kpad) break;
      float d[4][S];
      make_digits<S>(v[b][0].x, E, d[0]);
      make_digits<S>(v[b][0].y, E, d[1]);
      make_digits<S>(v[b][1].x, E, d[2]);
      make_digits<S>(v[b][1].y, E, d[3]);
#pragma unroll
      for (int s = 0; s < S; ++s)
        *reinterpret_cast<uint2 *>(out + s * plane + k) = make_uint2(pack_bf16(d[0][s], d[1][s]), pack_bf16(d[2][s], d[3][s]));
    }
  }
}

// Exponents and digit planes of gathered Green's-function rows in one pass: a warp per row, 4 consecutive k per lane and
// 128 per pass, kept in registers between the exponent and the split (NB passes, K <= 128 NB).  The lattice
// vectors come folded into the BvK cell and packed (GatherSrc::lamf, unif), so an element's cell is a few
// subtractions where folding took three integer divisions.
template <int S, int NB>
__global__ void __launch_bounds__(256) k_digits_gather(GatherSrc g, int rows, int K, int kpad, long long plane, int *expo,
                                                       __nv_bfloat16 *__restrict__ dig) {
  const int r = (blockIdx.x * 256 + threadIdx.x) >> 5, lane = threadIdx.x & 31;
  if (r >= rows) return;
  const int e = r / g.rows_per_entry, rr = r % g.rows_per_entry;
  const int V = e % g.natoms, gg = (e / g.natoms) % 2, p = e / (2 * g.natoms), mV = g.m[V];
  const int *pt = g.pts + 5 * p;
  const int2 *lam = g.lamf + g.lam_off[V];
  // kind 0: cell = fold(R1 - R_p) - fold(R2');  kind 1: fold(R_p) + fold(R2') = fold(R_p) - fold(-R2')
  int b0 = pt[2], b1 = pt[3], b2 = pt[4], fixed = rr;
  if (g.kind == 0) {
    const int2 u = g.unif[rr];
    b0 = (u.x & 255) - b0;
    b1 = (u.x >> 8 & 255) - b1;
    b2 = (u.x >> 16) - b2;
    b0 += b0 < 0 ? g.n1 : 0;
    b1 += b1 < 0 ? g.n2 : 0;
    b2 += b2 < 0 ? g.n3 : 0;
    fixed = u.y;
  }
  const double *G = g.G + gg * g.g_gstride + (long long)pt[1] * g.nR * g.nao * g.nao;
  double v[NB][4];
  int mx = 0;
#pragma unroll
  for (int b = 0; b < NB; ++b)
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const int k = b * 128 + lane * 4 + q;
      v[b][q] = 0.0;
      if (k < mV) {
        const int2 c = lam[k];
        int c0 = c.x & 255, c1 = c.x >> 8 & 255, c2 = c.x >> 16;
        if (g.kind == 0) {
          c0 = b0 - c0;
          c1 = b1 - c1;
          c2 = b2 - c2;
          c0 += c0 < 0 ? g.n1 : 0;
          c1 += c1 < 0 ? g.n2 : 0;
          c2 += c2 < 0 ? g.n3 : 0;
        } else {
          c0 += b0;
          c1 += b1;
          c2 += b2;
          c0 -= c0 >= g.n1 ? g.n1 : 0;
          c1 -= c1 >= g.n2 ? g.n2 : 0;
          c2 -= c2 >= g.n3 ? g.n3 : 0;
        }
        const int iR = (c0 * g.n2 + c1) * g.n3 + c2, row = g.kind == 0 ? c.y : fixed, col = g.kind == 0 ? fixed : c.y;
        v[b][q] = G[((long long)iR * g.nao + row) * g.nao + col];
      }
      mx = max(mx, biased_exp(v[b][q]));
    }
  mx = __reduce_max_sync(0xffffffffu, mx);
  const int E = mx - 1022;
  if (lane == 0) expo[r] = E;
#pragma unroll
  for (int b = 0; b < NB; ++b) {
    const int k = b * 128 + lane * 4;
    if (k >= kpad) break;
    float d[4][S];
#pragma unroll
    for (int q = 0; q < 4; ++q) make_digits<S>(v[b][q], E, d[q]);
#pragma unroll
    for (int s = 0; s < S; ++s)
      *reinterpret_cast<uint2 *>(dig + s * plane + (long long)r * kpad + k) =
          make_uint2(pack_bf16(d[0][s], d[1][s]), pack_bf16(d[2][s], d[3][s]));
  }
}

template <class Src>
__global__ void k_plain(Src src, int rows, int K, int kpad, int row0, __nv_bfloat16 *dig) {
  const long long x = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (x >= (long long)rows * kpad) return;
  const int r = (int)(x / kpad), k = (int)(x % kpad);
  dig[(long long)row0 * kpad + x] = __double2bfloat16(k < K ? src.get(r, k) : 0.0);
}

__device__ __forceinline__ float to_tf32(float f) {   // round to nearest, ties away
  uint32_t t;
  asm("cvt.rna.tf32.f32 %0, %1;" : "=r"(t) : "f"(f));
  return __uint_as_float(t);
}

// 3xTF32 split: plane 0 = tf32(x), plane 1 = tf32(x - plane 0)
template <class Src>
__global__ void k_split_tf32x3(Src src, int rows, int K, int kpad, int row0, long long plane, float *dig) {
  const long long x = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (x >= (long long)rows * kpad) return;
  const int r = (int)(x / kpad), k = (int)(x % kpad);
  const double v = k < K ? src.get(r, k) : 0.0;
  const float hi = to_tf32((float)v);
  const long long o = (long long)row0 * kpad + x;
  dig[o] = hi;
  dig[plane + o] = to_tf32((float)(v - (double)hi));
}

// plain TF32: the FP32 value rounded to the 10-bit TF32 mantissa (round to nearest, ties away)
template <class Src>
__global__ void k_plain_tf32(Src src, int rows, int K, int kpad, int row0, float *dig) {
  const long long x = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (x >= (long long)rows * kpad) return;
  const int r = (int)(x / kpad), k = (int)(x % kpad);
  dig[(long long)row0 * kpad + x] = to_tf32((float)(k < K ? src.get(r, k) : 0.0));
}

template <class Src>
void split_any(const Src &src, int rows, int K, int row0, Sliced &o, cudaStream_t s, bool expo_given = false) {
  if (row0 < 0 || row0 + rows > o.rows || K > o.kpad) throw Error{LIBRPA_E_ARG, "split: rows or K exceed the operand"};
  if (rows <= 0) return;
  const int kpad = o.kpad;
  const long long plane = (long long)o.rows * kpad;
  const long long n = (long long)rows * kpad;
  const unsigned g = (unsigned)((n + 255) / 256);
  if (o.S == S_TF32X3) {
    k_split_tf32x3<Src><<<g, 256, 0, s>>>(src, rows, K, kpad, row0, plane, (float *)o.digits);
    ++launch_counter();
    LR_CUDA(cudaGetLastError());
    return;
  }
  if (o.S == 0 || o.S == S_TF32) {
    if (o.S == 0)
      k_plain<Src><<<g, 256, 0, s>>>(src, rows, K, kpad, row0, (__nv_bfloat16 *)o.digits);
    else
      k_plain_tf32<Src><<<g, 256, 0, s>>>(src, rows, K, kpad, row0, (float *)o.digits);
    ++launch_counter();
    LR_CUDA(cudaGetLastError());
    return;
  }
  __nv_bfloat16 *dig = (__nv_bfloat16 *)o.digits;
  if (!expo_given) {
    k_row_expo<Src><<<(unsigned)(((long long)rows * 32 + 255) / 256), 256, 0, s>>>(src, rows, K, row0, o.expo);
    ++launch_counter();
  }
  const dim3 gd((unsigned)rows, (unsigned)((kpad + 1023) / 1024));
  switch (o.S) {
    case 1: k_digits<1, Src><<<gd, 256, 0, s>>>(src, K, kpad, row0, plane, o.expo, dig); break;
    case 2: k_digits<2, Src><<<gd, 256, 0, s>>>(src, K, kpad, row0, plane, o.expo, dig); break;
    case 3: k_digits<3, Src><<<gd, 256, 0, s>>>(src, K, kpad, row0, plane, o.expo, dig); break;
    case 4: k_digits<4, Src><<<gd, 256, 0, s>>>(src, K, kpad, row0, plane, o.expo, dig); break;
    case S_WIDE: k_digits<S_WIDE, Src><<<gd, 256, 0, s>>>(src, K, kpad, row0, plane, o.expo, dig); break;
    default: k_digits<5, Src><<<gd, 256, 0, s>>>(src, K, kpad, row0, plane, o.expo, dig); break;
  }
  ++launch_counter();
  LR_CUDA(cudaGetLastError());
}

// An output tile; c_n >= 0: only the K steps listed at chunks[c_off .. + c_n) are summed -- block-sparse operands,
// the others multiply exact zeros.  A listed step is 2 h + two: from half step h on (32 elements, 16 for
// TF32), both halves of a step (two = 1) or one.
// The host fills in what the producer and the MMA issuer need of the tile's entry, so that each reads one
// record per tile (and the next tile's ahead of time: a chain of two loads per tile was 10% of a short-K tile).
struct alignas(16) Tile {
  int e, m0, n0, c_off, c_n;
  int kbeg, nsteps, K;       // first k, steps, the entry's K
  int arow, brow, pair, pad;
};

__host__ __device__ constexpr uint32_t tmem_cols(int cols) { return cols <= 128 ? 128 : cols <= 256 ? 256 : 512; }
constexpr int PBK = 64;   // K per step: one 128-byte swizzle row of BF16 (32 TF32 values)
// Tile width BN of the S variant: the widest whose accumulators (S diagonals of BN columns) fit TMEM's 512 columns
// twice, so that one tile drains while the next fills; 5 planes also take 64 columns with one accumulator set
// (narrow outputs, see pick_bn).
__host__ __device__ constexpr int tile_bn(int S) { return S == S_WIDE ? 32 : S == 5 ? 48 : 64; }
__host__ __device__ constexpr int acc_cols(int S, int bn) { return (is_digits(S) ? S : 1) * bn; }
__host__ __device__ constexpr int acc_sets(int S, int bn) { return 2 * acc_cols(S, bn) <= 512 ? 2 : 1; }
// epilogue warps of the S variant
__host__ __device__ constexpr int epi_warps(int S) { return is_digits(S) ? 16 : 4; }
// columns of an epilogue warp, columns it stages at a time (what the shared memory beside the ring holds, pitch
// + 1), and the bytes of the staging area
__host__ __device__ constexpr int warp_cols(int S, int bn) { return bn * 4 / epi_warps(S); }
__host__ __device__ constexpr int stage_cols(int S, int bn) { return S == 5 && bn == 64 ? 8 : warp_cols(S, bn); }
__host__ __device__ constexpr int stage_bytes(int S, int bn) {
  return is_digits(S) ? epi_warps(S) * 32 * (stage_cols(S, bn) + 1) * 8 : 0;
}
// pipeline depths, what fits beside the staging area: slots of one A plane (128 rows x 128 bytes, 16 KB), and of
// all B planes
__host__ __device__ constexpr int a_slots(int S) {
  return S == S_WIDE ? 7 : !is_digits(S) ? 8 : S == 4 || S == 1 ? 5 : 6;
}
__host__ __device__ constexpr int b_slots(int S) { return planes(S) >= 3 ? 2 : is_digits(S) ? 2 * S - 1 + (S == 1) * 4 : 8 / planes(S); }
__host__ __device__ constexpr int ring_bytes(int S, int bn) {
  return a_slots(S) * BM * 128 + b_slots(S) * planes(S) * bn * 128;
}

// Position in a ring of N slots and the phase its barriers are in there.
template <int N>
struct Ring {
  int slot = 0;
  uint32_t phase = 0;
  bool wrapped = false;
  __device__ void next() {
    if (++slot == N) {
      slot = 0;
      phase ^= 1;
      wrapped = true;
    }
  }
  // for the drain after a failure: whether slot i was ever filled, and the phase of its last fill
  __device__ bool filled(int i) const { return wrapped || i < slot; }
  __device__ uint32_t last_phase(int i) const { return i < slot ? phase : phase ^ 1; }
};

// Operands of the entries of one launch that share them: tensor maps of the A and B digit planes
// (global memory, 128-byte aligned) and their row exponents.
struct alignas(128) MapPair {
  CUtensorMap a, b;
  const int *ea, *eb;
};

// Pipelined, warp-specialised kernel: CTA c takes tiles c, c + gridDim.x, ... (128 x BN output
// tiles of the launch's entries, sorted by decreasing K range on the host), keeping its barriers and
// TMEM across them (a persistent grid of one CTA per SM).
//   warp EW (one lane): TMA producer over two shared-memory rings of 128-byte rows (SWIZZLE_128B, K-major): all B
//     planes of a K step of 64 in one slot, the A planes one slot each, so that two steps fit where whole
//     steps of 5 planes (110 KB) would not.  (Rows of 64 bytes, a step of 32, moved 7 TB/s over the
//     chip, 25 bytes per cycle and SM, which bound every GEMM of the path.)  The rings run on across
//     tiles, so the next tile's loads overlap this tile's MMAs and epilogue;
//   warp EW + 1 (one lane): tcgen05.mma issuer; commits free a slot when its MMAs complete and, at
//     the end of a flush group, signal the epilogue; the next group (of this or the next tile) uses the
//     other accumulator set (or, with one set, starts once the epilogue has drained it).  The B planes lie one after the other in a
//     slot and the accumulators of consecutive diagonals in consecutive columns, so plane s of A
//     meets as many planes of B as 256 columns hold in one MMA: 5 MMAs per K step of 16 with 5 planes in
//     place of 15 of N = 48, and A read from shared memory 5 times instead of 15 (42 KB a step, below what the
//     MMAs' 368 cycles can take; one MMA per pair of planes held the tensor pipe at two thirds);
//   warps 0..EW-1: epilogue; warp w owns TMEM lanes 32 (w % 4) .. + 31 (= tile rows).  With EW = 16
//     (digit planes) warp w takes the (w / 4)-th quarter of the columns and after each flush group moves
//     the diagonal accumulators into exact int64 register sums (8 to 16 per thread, of two words each with 8
//     planes); with EW = 4 (plain BF16 / TF32, one group) each warp takes all columns into
//     registers.  The TMEM columns go back to the issuer before the values are converted and stored, so
//     conversion and stores overlap the next tile's MMAs.  The conversion (~30 integer instructions) is
//     bound by its latency: four warps per scheduler, 8 to 16 independent sums each.
// The epilogue of short-K tiles is bound by that chain and, in the trailing updates, by the FP64 pipe (two additions
// a cycle and SM), so it has no other FP64 instruction, reads the old outputs before it waits for the sums and stores
// whole sectors: 96 complex matrices of order 1946, K = 128: 7.0 -> 5.1 ms; N step of the slab 0.50 -> 0.44 ms.
// DIRECT: every tile has a single flush group (K up to 192 with 5 planes: the N and X steps, the trailing updates);
// outputs are then formed four columns at a time straight from TMEM, in a rolled loop, with no sums kept (a thread's
// columns unrolled are more instructions than the instruction cache holds).
// stall_ns > 0 (testing only): the MMA issuer first waits that long on an mbarrier nothing arrives
// at, so the CTA takes the bounded-wait failure path.  On any failure the CTA sets *err, stops
// issuing, waits (with the full limit) for the TMA copies and MMAs it has already issued, frees its
// TMEM and returns.
template <int S, int BN, bool DIRECT>
__global__ void __launch_bounds__(32 * (epi_warps(S) + 2), 1)
    k_ozgemm(const MapPair *__restrict__ maps, const Entry *__restrict__ entries, const Tile *__restrict__ tiles,
             const int *__restrict__ chunks, int ntiles, int *err, uint64_t stall_ns, int stage_in_ring) {
  constexpr bool TF = S == S_TF32 || S == S_TF32X3;   // kind::tf32
  constexpr bool PLAIN = !is_digits(S);                // one FP32 accumulator over all K
  constexpr bool WIDE = S == S_WIDE;                   // two-word sums
  constexpr int NP = planes(S);                        // planes per operand
  constexpr int NA = a_slots(S), NBS = b_slots(S);      // ring slots
  constexpr int KS = TF ? PBK / 2 : PBK;               // K elements per step (128 bytes per row)
  constexpr int KI = KS / 4;                           // K elements per MMA (32 bytes per row)
  constexpr uint32_t A_BYTES = BM * 128, B_BYTES = BN * 128;   // one plane
  // K steps per flush group: NP pairs x (64 G) x 2^14 <= 2^24 keeps the FP32 sums exact; plain
  // forms accumulate over the whole K in FP32
  constexpr int G = PLAIN ? (1 << 30) : 16 / NP;
  constexpr int EPI_WARPS = epi_warps(S), HALF = warp_cols(S, BN);   // HALF: columns per epilogue warp
  constexpr int kStack = 256 / BN;                     // B planes of one MMA: at most 256 columns
  constexpr int SETS = acc_sets(S, BN);                    // accumulator sets, one flush group each
  constexpr uint32_t SET_COLS = acc_cols(S, BN), TMEM_COLS = tmem_cols(SETS * acc_cols(S, BN));
  static_assert(SETS * acc_cols(S, BN) <= 512, "k_ozgemm: TMEM");
  extern __shared__ uint8_t smem_raw[];
  __shared__ uint64_t afull[NA], aempty[NA], bfull[NBS], bempty[NBS], tfull[SETS], tempty[SETS], mdone, never;
  __shared__ uint32_t tmem_slot;
  __shared__ volatile int abort_flag;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  uint8_t *smem = (uint8_t *)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
  uint8_t *sm_a = smem, *sm_b = smem + NA * A_BYTES;
  // the epilogue's staging area: in the rings when the CTA has a single tile (they are idle once its last MMA
  // completed), else after them
  uint8_t *stage_out = stage_in_ring ? smem : sm_b + NBS * NP * B_BYTES;
  if (tid == 0) {
#pragma unroll
    for (int s = 0; s < NA; ++s) {
      mbar_init(&afull[s], 1);
      mbar_init(&aempty[s], 1);
    }
#pragma unroll
    for (int s = 0; s < NBS; ++s) {
      mbar_init(&bfull[s], 1);
      mbar_init(&bempty[s], 1);
    }
#pragma unroll
    for (int b = 0; b < SETS; ++b) {
      mbar_init(&tfull[b], 1);
      mbar_init(&tempty[b], EPI_WARPS);
    }
    mbar_init(&mdone, 1);
    mbar_init(&never, 1);
    abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 0) tmem_alloc(&tmem_slot, TMEM_COLS);
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = tmem_slot;
  // first k of step i and, in `half`, whether only its first half is summed (a listed half step, see Tile)
  auto k_of = [&](const Tile &tl, int i, bool &half) {
    const int c = tl.c_n >= 0 ? chunks[tl.c_off + i] : 0;
    half = tl.c_n >= 0 && !(c & 1);
    return tl.c_n >= 0 ? (c >> 1) * (KS / 2) : tl.kbeg + i * KS;
  };
  const int stride = (int)gridDim.x;
  auto tile_at = [&](int t) { return tiles[t < ntiles ? t : 0]; };
  if (warp == EPI_WARPS) {
    if (elect_one()) {
      Ring<NA> ra;
      Ring<NBS> rb;
      Tile nx = tile_at(blockIdx.x);
      for (int t = blockIdx.x; t < ntiles && !abort_flag; t += stride) {
        const Tile tl = nx;
        nx = tile_at(t + stride);
        const MapPair *mp = maps + tl.pair;
        for (int i = 0; i < tl.nsteps && !abort_flag; ++i) {
          bool half;
          const int k0 = k_of(tl, i, half);
          if (!mbar_wait(&bempty[rb.slot], rb.phase ^ 1, WAIT_NS, &abort_flag)) {
            abort_flag = 1;
            break;
          }
          mbar_expect_tx(&bfull[rb.slot], NP * B_BYTES);
          tma_load_3d(sm_b + rb.slot * (NP * B_BYTES), &mp->b, &bfull[rb.slot], k0, tl.brow, 0);
          rb.next();
          for (int p = 0; p < NP; ++p) {
            if (!mbar_wait(&aempty[ra.slot], ra.phase ^ 1, WAIT_NS, &abort_flag)) {
              abort_flag = 1;
              break;
            }
            mbar_expect_tx(&afull[ra.slot], A_BYTES);
            tma_load_3d(sm_a + ra.slot * A_BYTES, &mp->a, &afull[ra.slot], k0, tl.arow, p);
            ra.next();
          }
        }
      }
      // after a failure: the copies of the last slots filled may still be in flight (earlier ones were consumed);
      // wait for each to land before the CTA exits
      if (abort_flag) {
        for (int i = 0; i < NA; ++i)
          if (ra.filled(i)) mbar_wait(&afull[i], ra.last_phase(i), WAIT_NS);
        for (int i = 0; i < NBS; ++i)
          if (rb.filled(i)) mbar_wait(&bfull[i], rb.last_phase(i), WAIT_NS);
      }
    }
  } else if (warp == EPI_WARPS + 1) {
    if (elect_one()) {
      if (stall_ns) {   // testing only: a barrier nothing arrives at
        mbar_wait(&never, 0, stall_ns, &abort_flag);
        abort_flag = 1;
      }
      Ring<NA> ra;
      Ring<NBS> rb;
      Ring<SETS> rt;   // accumulator sets, one flush group each
      Tile nx = tile_at(blockIdx.x);
      for (int t = blockIdx.x; t < ntiles && !abort_flag; t += stride) {
        const Tile tl = nx;
        nx = tile_at(t + stride);
        int c = 0;   // step of the group
        for (int i = 0; i < tl.nsteps && !abort_flag; ++i) {
          // a new group needs its accumulators drained by the epilogue (the group before in this set, any tile)
          if (c == 0 && !mbar_wait(&tempty[rt.slot], rt.phase ^ 1, WAIT_NS, &abort_flag)) {
            abort_flag = 1;
            break;
          }
          if (!mbar_wait(&bfull[rb.slot], rb.phase, WAIT_NS, &abort_flag)) {
            abort_flag = 1;
            break;
          }
          const uint32_t db0 = smem_u32(sm_b + rb.slot * (NP * B_BYTES)), tacc = tmem + (uint32_t)rt.slot * SET_COLS;
          // MMAs of the step: K columns past the operands' end hold zeros and are left out
          bool half;
          const int k0 = k_of(tl, i, half), nk = min(half ? 2 : 4, (tl.K - k0 + KI - 1) / KI);
          const uint64_t db = smem_desc128(db0);   // (address fields in units of 16 bytes)
#pragma unroll
          for (int s = 1; s <= NP; ++s) {
            if (!mbar_wait(&afull[ra.slot], ra.phase, WAIT_NS, &abort_flag)) {
              abort_flag = 1;
              break;
            }
            tc_fence_after();
            const uint64_t da = smem_desc128(smem_u32(sm_a + ra.slot * A_BYTES));
#pragma unroll
            for (int j = 0; j < 4; ++j) {   // 32 bytes of K per MMA
              if (j >= nk) break;
              // plain forms: one accumulator for all products, hi hi (and hi lo, lo hi of the 3xTF32 split);
              // digit planes: plane s of A by planes u .. u + w - 1 of B (N = BN w), into the diagonals s + u ..
              constexpr int kStep = PLAIN ? 1 : kStack;
#pragma unroll
              for (int u = 1; u + s <= NP + 1; u += kStep) {
                const int w = PLAIN ? 1 : NP + 2 - s - u < kStack ? NP + 2 - s - u : kStack;
                const uint32_t d = tacc + (PLAIN ? 0u : (uint32_t)(s + u - 2) * BN);
                const uint64_t dbu = db + ((u - 1) * B_BYTES + 32 * j) / 16;
                const bool first = j == 0 && s == 1 && (!PLAIN || u == 1);
                if constexpr (TF)
                  umma_tf32(d, da + 2 * j, dbu, idesc(BN, true), first && c == 0 ? 0u : 1u);
                else if (first)
                  umma(d, da + 2 * j, dbu, idesc(BN * w, false), c == 0 ? 0u : 1u);
                else
                  umma_add(d, da + 2 * j, dbu, idesc(BN * w, false));
              }
            }
            umma_commit(&aempty[ra.slot]);
            ra.next();
          }
          if (abort_flag) break;
          umma_commit(&bempty[rb.slot]);
          rb.next();
          if (++c == G || i == tl.nsteps - 1) {
            umma_commit(&tfull[rt.slot]);
            rt.next();
            c = 0;
          }
        }
      }
      // after a failure: wait until every MMA this thread issued has completed (they read the
      // shared-memory stages and write TMEM)
      if (abort_flag) {
        umma_commit(&mdone);
        mbar_wait(&mdone, 0, WAIT_NS);
      }
    }
  } else {
    const int quad = warp & 3, half = warp >> 2;   // TMEM lane quadrant, column half
    const uint32_t tbase0 = tmem + ((uint32_t)(32 * quad) << 16) + half * HALF;
    Ring<SETS> rt;   // accumulator sets, one flush group each
    for (int t = blockIdx.x; t < ntiles; t += stride) {
      const Tile &tl = tiles[t];
      const Entry &en = entries[tl.e];
      const Tile &tn = tiles[t + stride < ntiles ? t + stride : t];   // the next tile's record and exponents to the L1
      prefetch_l1(&tiles[t + 2 * stride < ntiles ? t + 2 * stride : t]);
      prefetch_l1(&entries[tn.e]);
      prefetch_l1(&maps[tn.pair].ea);
      const int nsteps = tl.nsteps;
      const int ngroups = (nsteps + G - 1) / G;
      const int m0 = tl.m0, n0 = tl.n0;
      const int eM = en.M, eN = en.N, mode = en.mode;
      const long long ldc = en.ldc;
      double *const C = en.C;
      const double alpha = en.alpha, beta = en.beta;
      // beta != 0, tested on its bits (a comparison of doubles per store held the FP64 pipe for a third of the N step)
      const bool upd = (__double_as_longlong(beta) << 1) != 0;
      const bool pow2 = en.alpha_shift != kNoShift;   // alpha = +-2^alpha_shift: folded into the exponent
      const int row = m0 + 32 * quad + lane;          // thread = tile row (the TMEM lane layout)
      const bool row_ok = row < eM;
      // output (row, col) at out_row(row) + col cstep
      const bool trans = mode == 2 || mode == 4;
      const long long cstep = mode == 4 ? ldc : mode == 2 ? 2 * ldc : mode == 1 ? 2 : 1;
      auto out_row = [&](int r_) {
        return trans ? C + r_ : mode == 1 ? C + 2 * (r_ >> 1) * ldc + (r_ & 1) : C + r_ * ldc;
      };
      // digit planes: exact sums of the diagonals, in units of the last one's scale (WIDE: the first four
      // diagonals in acch, in units of the fourth's, the last four in acc)
      long long acc[PLAIN || DIRECT ? 1 : HALF], acch[WIDE && !DIRECT ? HALF : 1];
      uint32_t fa[PLAIN ? HALF : 1];   // plain forms: the FP32 accumulators
      constexpr int SC = stage_cols(S, BN);
      const int cbase = n0 + half * HALF, nc = min(HALF, eN - cbase);   // nc: live columns of the warp (may be <= 0)
      const MapPair &mp = maps[tl.pair];
      const int ash = (pow2 ? en.alpha_shift : 0) - 14 - 8 * (S - 1);
      const int ea = PLAIN || !row_ok ? ash : mp.ea[tl.arow + 32 * quad + lane] + ash;
      // the exponents of the warp's columns, one per lane
      const int eb_lane = !PLAIN && lane < nc ? (mp.eb + tl.brow + half * HALF)[lane] : 0;
      auto eb = [&](int j) { return __shfl_sync(0xffffffffu, eb_lane, j); };
      const bool aneg = pow2 && alpha < 0.0;
      // a row or column with an infinity or a NaN has the exponent 1025 (finite ones at most 1024)
      const bool row_nan = ea - ash > 1024;
      // an output (FP64 bits, or in mode 3 the FP32 pair) from the exact sum lo, or hi 2^32 + lo (WIDE)
      auto value = [&](long long hi, long long lo, int e_b) {
        const int sh = ea + e_b;
        const bool nan = row_nan || e_b > 1024;
        float2 pr;
        if (!WIDE && mode == 3 && pow2) {
          pr = i64_to_f32x2(aneg ? -lo : lo, sh);
        } else {
          double v;
          if constexpr (WIDE)
            v = i96_to_f64(hi, lo, sh);
          else
            v = i64_to_f64(lo, sh);
          if (!pow2) {
            asm volatile("");   // a branch: FP64 instructions cost their place on the pipe even when predicated off
            v *= alpha;
          } else if (aneg) {
            v = -v;
          }
          if (nan) v = __longlong_as_double(0x7FF8000000000000ll);
          if (mode != 3) return __double_as_longlong(v);
          pr.x = __double2float_rn(v);
          pr.y = __double2float_rn(v - (double)pr.x);
        }
        if (nan) pr = make_float2(__uint_as_float(0x7FC00000u), 0.f);
        return (long long)(((unsigned long long)__float_as_uint(pr.y) << 32) | __float_as_uint(pr.x));
      };
      // row-major outputs go through the staging area: SC columns of RPI rows at a time, the components of a
      // complex element (rows 2 i, 2 i + 1) next to each other, so that every pass stores whole sectors
      constexpr int RPI = PLAIN ? 2 : 32 / SC, PASSES = 32 / RPI;
      static_assert(PLAIN || RPI % 2 == 0, "k_ozgemm: staging");
      long long *stg = reinterpret_cast<long long *>(stage_out) + warp * 32 * (SC + 1);
      const int lr = mode == 1 ? lane / (2 * SC) * 2 + (lane & 1) : lane / SC;   // the lane's row and column of a pass
      const int lc = mode == 1 ? lane % (2 * SC) >> 1 : lane % SC;
      const int rlive = lane < RPI * SC ? eM - (m0 + 32 * quad) - lr : 0;        // passes with RPI i < rlive
      auto out0 = [&](int cb) { return out_row(m0 + 32 * quad + lr) + (cbase + cb + lc) * cstep; };
      const long long step = RPI * ldc;
      auto store_rows = [&](int cb, auto &&old) {   // columns cb .. + SC of the warp, staged; old(i, q): *q before
        __syncwarp();
        double *q = out0(cb);
        const long long *sp = stg + lr * (SC + 1) + lc;
        if (cb + lc < nc) {
#pragma unroll
          for (int i = 0; i < PASSES; ++i, q += step) {
            if (RPI * i >= rlive) break;
            double v = __longlong_as_double(sp[i * RPI * (SC + 1)]);
            if (upd) {   // (modes 0 and 1)
              asm volatile("");
              v += beta * old(i, q);
            }
            *q = v;
          }
        }
        __syncwarp();
      };
      // updated outputs of a single group are read before its sums are waited for
      double old0[DIRECT ? PASSES : 1];
      if constexpr (DIRECT) {
        if (upd && !trans) {
          const double *q = out0(0);
#pragma unroll
          for (int i = 0; i < PASSES; ++i, q += step) old0[i] = RPI * i < rlive && lc < nc ? *q : 0.0;
        }
      }
      auto read0 = [&](int i, const double *) { return old0[DIRECT ? i : 0]; };
      auto read_now = [&](int, const double *q) { return *q; };
      if constexpr (!PLAIN && !DIRECT) {
#pragma unroll
        for (int j = 0; j < HALF; ++j) acc[j] = 0;
        if constexpr (WIDE) {
#pragma unroll
          for (int j = 0; j < HALF; ++j) acch[j] = 0;
        }
      }
      bool ok_all = true;
      for (int gi = 0; gi < ngroups; ++gi) {
        bool ok = !abort_flag && mbar_wait(&tfull[rt.slot], rt.phase, WAIT_NS, &abort_flag);
        const uint32_t tbase = tbase0 + (uint32_t)rt.slot * SET_COLS;
        ok = __all_sync(0xffffffffu, ok);
        if (!ok) {
          abort_flag = 1;
          ok_all = false;
          break;
        }
        tc_fence_after();
        if constexpr (!PLAIN) {
          if constexpr (DIRECT) {
#pragma unroll 1
            for (int c = 0; c < nc; c += 4) {
              uint32_t r[S][4];
              int e_b[4];
#pragma unroll
              for (int d = 0; d < S; ++d) tmem_ld(tbase + (uint32_t)d * BN + c, r[d]);
#pragma unroll
              for (int x = 0; x < 4; ++x) e_b[x] = eb(c + x);
#pragma unroll
              for (int d = 0; d < S; ++d) tmem_ld_wait(r[d]);
#pragma unroll
              for (int x = 0; x < 4; ++x) {
                long long o;
                if (!WIDE && mode == 3 && pow2) {
                  // FP32-pair outputs: the diagonal sums, integers below 2^24 times their powers of two, summed into an
                  // unevaluated FP32 pair by exact two-sums, renormalised and scaled by 2^sh
                  float hi = __uint_as_float(r[0][x]) * (float)(1ull << (8 * (S - 1))), lo = 0.f;   // exact
#pragma unroll
                  for (int d = 1; d < S; ++d) {
                    const float t = __uint_as_float(r[d][x]) * (float)(1ull << (8 * (S - 1 - d)));
                    const float sm = hi + t, bb = sm - hi;
                    lo += (hi - (sm - bb)) + (t - bb);
                    hi = sm;
                  }
                  const float sm = hi + lo;
                  lo = lo - (sm - hi);
                  hi = sm;
                  const int sh = ea + e_b[x], eh = (int)((__float_as_uint(hi) >> 23) & 0xFF);
                  const float sc = __uint_as_float(((uint32_t)(sh + 127) << 23) | (aneg ? 0x80000000u : 0u));
                  float2 pr = make_float2(hi * sc, lo * sc);
                  if ((unsigned)(sh + 126) > 253u || (hi != 0.f && (unsigned)(eh + sh - 1) > 253u)) {
                    asm volatile("");   // a branch: outside the FP32 range of a direct scaling, through FP64
                    const double dv = ldexp((double)hi + (double)lo, sh) * (aneg ? -1.0 : 1.0);
                    pr.x = __double2float_rn(dv);
                    pr.y = __double2float_rn(dv - (double)pr.x);
                  }
                  if (row_nan || e_b[x] > 1024) pr = make_float2(__uint_as_float(0x7FC00000u), 0.f);
                  o = (long long)(((unsigned long long)__float_as_uint(pr.y) << 32) | __float_as_uint(pr.x));
                } else {
                  long long hi = 0, lo = 0;
#pragma unroll
                  for (int d = 0; d < S; ++d) {
                    const int v = __float2int_rn(__uint_as_float(r[d][x]));
                    if (WIDE && d < 4)
                      hi += (long long)v * (1 << (8 * (3 - d) & 31));
                    else if (S == 5 && d == 0)
                      lo += (long long)((unsigned long long)(unsigned)v << 32);   // 2^32 v (mod 2^64)
                    else
                      lo += (long long)v * (1 << (8 * (S - 1 - d) & 31));
                  }
                  o = value(hi, lo, e_b[x]);
                }
                if (!trans) {
                  stg[lane * (SC + 1) + c + x] = o;
                } else if (row_ok && c + x < nc) {   // consecutive along the lanes
                  double *q = out_row(row) + (cbase + c + x) * cstep;
                  double v = __longlong_as_double(o);
                  if (upd) {
                    asm volatile("");
                    v += beta * *q;
                  }
                  *q = v;
                }
              }
            }
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(&tempty[rt.slot]);   // the accumulators may be overwritten now
            rt.next();
            if (!trans && nc > 0) store_rows(0, read0);
            break;
          }
          if constexpr (!DIRECT) {
          // one diagonal at a time, the next load in flight while this one is added
          constexpr int RB = 2;
          uint32_t r[RB][HALF];
          tmem_ld(tbase, r[0]);
#pragma unroll
          for (int d = 0; d < S; ++d) {
            tmem_ld_wait(r[d % RB]);
            if (d + 1 < S) tmem_ld(tbase + (uint32_t)(d + 1) * BN, r[(d + 1) % RB]);
#pragma unroll
            for (int j = 0; j < HALF; ++j) {
              const int v = __float2int_rn(__uint_as_float(r[d % RB][j]));
              if constexpr (WIDE) {
                if (d < 4)
                  acch[j] += (long long)v * (1 << (8 * (3 - d)));
                else
                  acc[j] += (long long)v * (1 << (8 * (7 - d)));
              } else if (S == 5 && d == 0) {
                acc[j] += (long long)((unsigned long long)(unsigned)v << 32);   // 2^32 v (mod 2^64)
              } else {
                acc[j] += (long long)v * (1 << (8 * (S - 1 - d) % 32));
              }
            }
          }
          }
        } else {
#pragma unroll
          for (int cb = 0; cb < HALF / 16; ++cb) {
            uint32_t r[16];
            tmem_ld(tbase + cb * 16, r);
            tmem_ld_wait(r);
#pragma unroll
            for (int j = 0; j < 16; ++j) fa[cb * 16 + j] = r[j];
          }
        }
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(&tempty[rt.slot]);   // the accumulators may be overwritten now
        rt.next();
      }
      if (!ok_all) break;
      if constexpr (DIRECT) {
        if (nsteps == 0 && nc > 0) {   // nothing to sum: zeros
          if (trans) {
            for (int j = 0; j < nc && row_ok; ++j) {
              double *q = out_row(row) + (cbase + j) * cstep;
              *q = !upd ? 0.0 : beta * *q;
            }
          } else {
#pragma unroll
            for (int j = 0; j < SC; ++j) stg[lane * (SC + 1) + j] = 0;
            store_rows(0, read0);
          }
        }
      } else if constexpr (PLAIN) {
        // plain forms: one FP32 sum per element, scaled in FP64 and stored from the registers,
        // thread = tile row
        if (row_ok) {
#pragma unroll
          for (int c = 0; c < HALF; ++c) {
            const int col = n0 + half * HALF + c;
            if (col >= eN) break;
            if (mode == 3 && pow2) {   // the FP32 sum times +-2^k: exact in FP32
              const float f = nsteps > 0 ? __uint_as_float(fa[c]) * (float)alpha : 0.f;
              reinterpret_cast<float2 *>(C)[(long long)row * ldc + col] = make_float2(f, 0.f);
              continue;
            }
            const double v = nsteps > 0 ? alpha * (double)__uint_as_float(fa[c]) : 0.0;
            if (mode == 3) {   // real, as an unevaluated pair of FP32 numbers (hi, lo)
              const float hi = __double2float_rn(v);
              reinterpret_cast<float2 *>(C)[(long long)row * ldc + col] =
                  make_float2(hi, __double2float_rn(v - (double)hi));
              continue;
            }
            double *p = out_row(row) + col * cstep;
            *p = !upd ? v : v + beta * *p;
          }
        }
      } else {
        if (nc <= 0) continue;
        // the values in place of the sums
#pragma unroll
        for (int j = 0; j < HALF; ++j) acc[j] = value(WIDE ? acch[WIDE ? j : 0] : 0, acc[j], eb(j));
        if (trans) {   // consecutive along the lanes (tile rows)
          if (row_ok) {
            double old[HALF];
            if (upd) {
#pragma unroll
              for (int j = 0; j < HALF; ++j)
                if (j < nc) old[j] = out_row(row)[(cbase + j) * cstep];
            }
#pragma unroll
            for (int j = 0; j < HALF; ++j)
              if (j < nc) {
                const double v = __longlong_as_double(acc[j]);
                out_row(row)[(cbase + j) * cstep] = !upd ? v : v + beta * old[j];
              }
          }
          continue;
        }
#pragma unroll
        for (int cb = 0; cb < HALF; cb += SC) {
          if (cb >= nc) break;   // the same for the whole warp
#pragma unroll
          for (int j = 0; j < SC; ++j) stg[lane * (SC + 1) + j] = acc[cb + j];
          store_rows(cb, read_now);
        }
      }
    }
  }
  __syncthreads();
  if (abort_flag && tid == 0) atomicExch(err, 1);
  tc_fence_before();
  __syncthreads();
  if (warp == 0) tmem_dealloc(tmem, TMEM_COLS);
}

PFN_cuTensorMapEncodeTiled_v12000 g_encode = nullptr;

// Tensor map of an operand's planes with boxes of 128 bytes (the swizzle width) x box_rows rows x box_planes planes.
CUtensorMap make_map(const Sliced &o, int box_rows, int box_planes) {
  CUtensorMap m;
  const cuuint64_t eb = (cuuint64_t)elem_bytes(o.S);
  const cuuint64_t dims[3] = {(cuuint64_t)o.kpad, (cuuint64_t)o.rows, (cuuint64_t)planes(o.S)};
  const cuuint64_t strides[2] = {(cuuint64_t)o.kpad * eb, (cuuint64_t)o.kpad * eb * (cuuint64_t)o.rows};
  const cuuint32_t box[3] = {(cuuint32_t)(128 / eb), (cuuint32_t)box_rows, (cuuint32_t)box_planes};
  const cuuint32_t estr[3] = {1, 1, 1};
  const CUtensorMapDataType dt = eb == 4 ? CU_TENSOR_MAP_DATA_TYPE_FLOAT32 : CU_TENSOR_MAP_DATA_TYPE_BFLOAT16;
  const CUresult r = g_encode(&m, dt, 3, o.digits, dims, strides, box, estr,
                              CU_TENSOR_MAP_INTERLEAVE_NONE,
                              CU_TENSOR_MAP_SWIZZLE_128B,
                              CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  if (r != CUDA_SUCCESS) throw Error{LIBRPA_E_CUDA, "cuTensorMapEncodeTiled failed: " + std::to_string((int)r)};
  return m;
}

}  // namespace

CUtensorMap make_map_nested(const void *digits, int rows, int planes, int outer, int box_rows, int box_outer) {
  CUtensorMap m;
  const cuuint64_t dims[4] = {32, (cuuint64_t)rows, (cuuint64_t)planes, (cuuint64_t)outer};
  const cuuint64_t strides[3] = {64, 64ull * rows, 64ull * rows * planes};
  const cuuint32_t box[4] = {32, (cuuint32_t)box_rows, (cuuint32_t)planes, (cuuint32_t)box_outer};
  const cuuint32_t estr[4] = {1, 1, 1, 1};
  const CUresult r = g_encode(&m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 4, const_cast<void *>(digits), dims, strides, box, estr,
                              CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_64B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                              CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  if (r != CUDA_SUCCESS) throw Error{LIBRPA_E_CUDA, "cuTensorMapEncodeTiled failed: " + std::to_string((int)r)};
  return m;
}

namespace {

// dynamic shared memory of k_ozgemm<S, BN>: the pipeline's stages and the epilogue's staging area, overlapping
// when every CTA has one tile
constexpr int gemm_smem(int S, int bn, bool in_ring) {
  return (in_ring ? (ring_bytes(S, bn) > stage_bytes(S, bn) ? ring_bytes(S, bn) : stage_bytes(S, bn))
                  : ring_bytes(S, bn) + stage_bytes(S, bn)) + 1024;
}

struct Launch {
  const MapPair *maps;
  const Entry *entries;
  const Tile *tiles;
  const int *chunks;
  int ntiles, grid, *err;
  uint64_t stall_ns;
  cudaStream_t s;
};

template <int S, int BN, bool DIRECT>
void launch_as(const Launch &l) {
  static_assert(gemm_smem(S, BN, false) <= 226 * 1024, "k_ozgemm: shared memory");
  const bool in_ring = l.grid >= l.ntiles;
  // one limit for every launch: host threads set it concurrently, and a launch's own size could
  // undercut another thread's launch
  LR_CUDA(cudaFuncSetAttribute(k_ozgemm<S, BN, DIRECT>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                               gemm_smem(S, BN, false)));
  k_ozgemm<S, BN, DIRECT><<<l.grid, 32 * (epi_warps(S) + 2), gemm_smem(S, BN, in_ring), l.s>>>(
      l.maps, l.entries, l.tiles, l.chunks, l.ntiles, l.err, l.stall_ns, in_ring);
}
// max_steps: of the launch's tiles
template <int S, int BN = tile_bn(S)>
void launch(const Launch &l, int max_steps) {
  if constexpr (is_digits(S)) {
    if constexpr (stage_cols(S, BN) == warp_cols(S, BN)) {
      if (max_steps <= 16 / planes(S)) return launch_as<S, BN, true>(l);
    }
  }
  launch_as<S, BN, false>(l);
}

// Tile width of a launch.  With 5 planes, 48 columns and two accumulator sets: the drain of a flush group
// (~3000 cycles) overlaps the next MMAs.  64 columns with one set where 48 would pad the outputs' columns by a third
// or more beyond them (the final contraction: 60 auxiliary functions an atom).
int pick_bn(int S, const std::vector<Entry> &entries) {
  if (S != 5) return tile_bn(S);
  double c48 = 0, c64 = 0;
  for (const Entry &e : entries) {
    const double w = (double)e.M * e.K;
    c48 += w * ((e.N + 47) / 48 * 48);
    c64 += w * ((e.N + 63) / 64 * 64);
  }
  return 4 * c64 <= 3 * c48 ? 64 : 48;
}

}  // namespace

void init() {
  static std::once_flag once;   // handles on several host threads (the serving loop) share it
  std::call_once(once, [] {
    void *fn = nullptr;
    cudaDriverEntryPointQueryResult q;
    cudaError_t e = cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &fn, 12000, cudaEnableDefault, &q);
    if (e == cudaSuccess && q == cudaDriverEntryPointSuccess && fn) g_encode = (PFN_cuTensorMapEncodeTiled_v12000)fn;
  });
  if (!g_encode) throw Error{LIBRPA_E_CUDA, "cuTensorMapEncodeTiled entry point not available"};
}

size_t sliced_bytes(int rows, int K, int S) {
  const size_t kpad = ((size_t)K + 7) / 8 * 8;
  const size_t dig = ((size_t)planes(S) * rows * kpad * elem_bytes(S) + 255) / 256 * 256;
  return dig + ((size_t)rows * 4 + 255) / 256 * 256;
}

void sliced_bind(Sliced &o, void *mem, int rows, int K, int S) {
  o.rows = rows;
  o.K = K;
  o.kpad = (K + 7) / 8 * 8;
  o.S = S;
  o.digits = mem;
  const size_t dig = ((size_t)planes(S) * rows * o.kpad * elem_bytes(S) + 255) / 256 * 256;
  o.expo = (int *)((char *)mem + dig);
}

void split_real(const double *src, long long ld, bool trans, int rows, int K, int batch, long long batch_stride,
                Sliced &out, cudaStream_t s, int row0) {
  RealSrc r{src, ld, batch_stride, rows, trans};
  split_any(r, rows * batch, K, row0, out, s);
}

void split_complex(const double2 *src, long long ld, Op op, bool as_a, int n_out, int n_k, int batch,
                   long long batch_stride, Sliced &out, cudaStream_t s, const int *eq) {
  const int rows_pb = as_a ? 2 * n_out : n_out;
  CplxSrc c{src, ld, batch_stride, rows_pb, (int)op, as_a};
  if (eq) {
    if (!as_a) throw Error{LIBRPA_E_ARG, "split_complex: scaled elements in the B' form"};
    split_any(CplxEqSrc{c, eq}, rows_pb * batch, 2 * n_k, 0, out, s);
    return;
  }
  split_any(c, rows_pb * batch, 2 * n_k, 0, out, s);
}

// calls f(integral_constant S) for the digit-plane count of an operand
template <class F>
void with_planes(int S, F &&f) {
  switch (S) {
    case 1: f(std::integral_constant<int, 1>()); break;
    case 2: f(std::integral_constant<int, 2>()); break;
    case 3: f(std::integral_constant<int, 3>()); break;
    case 4: f(std::integral_constant<int, 4>()); break;
    case 5: f(std::integral_constant<int, 5>()); break;
    default: f(std::integral_constant<int, S_WIDE>()); break;
  }
}

void split_gather(const GatherSrc &src, int rows, int K, Sliced &out, cudaStream_t s) {
  if (is_digits(out.S) && src.lamf && K <= 512) {
    if (rows > out.rows || K > out.kpad) throw Error{LIBRPA_E_ARG, "split: rows or K exceed the operand"};
    if (rows <= 0) return;
    const unsigned grid = (unsigned)(((long long)rows * 32 + 255) / 256);
    const long long plane = (long long)out.rows * out.kpad;
    __nv_bfloat16 *dig = (__nv_bfloat16 *)out.digits;
    with_planes(out.S, [&](auto c) {
      constexpr int S = decltype(c)::value;
      if (out.kpad <= 256)
        k_digits_gather<S, 2><<<grid, 256, 0, s>>>(src, rows, K, out.kpad, plane, out.expo, dig);
      else
        k_digits_gather<S, 4><<<grid, 256, 0, s>>>(src, rows, K, out.kpad, plane, out.expo, dig);
    });
    ++launch_counter();
    LR_CUDA(cudaGetLastError());
    return;
  }
  GatherDev g{src};
  split_any(g, rows, K, 0, out, s);
}

void split_ragged(const double *base, const long long *off, const int *Ke, int rows_per_entry, int n_entries,
                  int Kmax, Sliced &out, cudaStream_t s, bool expo_given) {
  RaggedSrc r{base, off, Ke, rows_per_entry};
  if (is_digits(out.S) && expo_given) {
    const int rows = rows_per_entry * n_entries;
    if (rows > out.rows || Kmax > out.kpad) throw Error{LIBRPA_E_ARG, "split: rows or K exceed the operand"};
    if (rows <= 0) return;
    with_planes(out.S, [&](auto c) {
      k_digits_ragged<decltype(c)::value><<<(unsigned)rows, 256, 0, s>>>(r, out.kpad, (long long)out.rows * out.kpad, out.expo,
                                                                       (__nv_bfloat16 *)out.digits);
    });
    ++launch_counter();
    LR_CUDA(cudaGetLastError());
    return;
  }
  split_any(r, rows_per_entry * n_entries, Kmax, 0, out, s, expo_given);
}

// out.expo[r] = -1022 (the exponent of an all-zero row) for rows [0, rows)
__global__ void k_expo_init(int *expo, int rows) {
  const int r = blockIdx.x * blockDim.x + threadIdx.x;
  if (r < rows) expo[r] = -1022;
}
void expo_init(Sliced &out, int rows, cudaStream_t s) {
  if (rows <= 0) return;
  k_expo_init<<<(unsigned)((rows + 255) / 256), 256, 0, s>>>(out.expo, rows);
  ++launch_counter();
  LR_CUDA(cudaGetLastError());
}

long long gemm_multi(const std::vector<std::pair<const Sliced *, const Sliced *>> &ops, const std::vector<Entry> &entries,
                     int *err, cudaStream_t s, Handle &h, DevBuf &args, const StageFn *stage_fn) {
  if (ops.empty()) return 0;
  const int S = ops[0].first->S, BN = pick_bn(S, entries);   // BN: tile width of this launch
  for (const auto &o : ops)
    if (o.first->S != S || o.second->S != S || S < 0 || S > S_WIDE)
      throw Error{LIBRPA_E_ARG, "oz::gemm: operand mismatch"};
  init();
  // tiles with their K range in stages; MMA flops issued: per tile BM x BN x (K rounded up to the
  // K step) per digit-plane product
  const double prods = is_digits(S) ? S * (S + 1) / 2.0 : S == S_TF32X3 ? 3.0 : 1.0;
  const int ks = elem_bytes(S) == 4 ? PBK / 2 : PBK;   // K elements per pipeline step
  const int kh = ks / 2;                               // the half steps that stage_fn lists
  std::vector<std::pair<int, Tile>> tk;
  std::vector<int> chunks, cl;
  double exec = 0;
  h.oz_exec_flops = 0;
  h.oz_alg_flops = 0;
  for (int e = 0; e < (int)entries.size(); ++e) {
    const Entry &en = entries[e];
    if (en.M <= 0 || en.N <= 0) continue;
    if (en.pair < 0 || en.pair >= (int)ops.size()) throw Error{LIBRPA_E_ARG, "oz::gemm: entry without operands"};
    const Sliced &a = *ops[en.pair].first, &b = *ops[en.pair].second;
    if (en.K > a.kpad || en.K > b.kpad || en.a_row0 < 0 || en.b_row0 < 0 || en.a_row0 + en.M > a.rows ||
        en.b_row0 + en.N > b.rows)
      throw Error{LIBRPA_E_ARG, "oz::gemm: entry outside its operands"};
    for (int m0 = 0; m0 < en.M; m0 += BM)
      for (int n0 = 0; n0 < en.N; n0 += BN) {
        // strictly above the diagonal: every column of the tile beyond every row (in output rows,
        // lower_div stacked rows per output row)
        if (en.lower_div > 0 && (long long)n0 * en.lower_div >= (long long)m0 + BM) continue;
        const int rows = std::min(BM, en.M - m0), cols = std::min(BN, en.N - n0);
        cl.clear();
        if (stage_fn && (*stage_fn)(e, m0, rows, n0, cols, kh, en.K, cl)) {
          double kk = 0;
          for (int c : cl) kk += std::min(kh, en.K - c * kh);
          h.oz_alg_flops += 2.0 * rows * cols * kk;
          exec += 2.0 * BM * BN * (double)cl.size() * kh * prods;
          const int c0 = (int)chunks.size();
          for (size_t i = 0; i < cl.size(); ++i) {   // neighbours share a step
            const bool two = i + 1 < cl.size() && cl[i + 1] == cl[i] + 1;
            chunks.push_back(2 * cl[i] + two);
            if (two) ++i;
          }
          const int n = (int)chunks.size() - c0;
          tk.push_back({n, Tile{e, m0, n0, c0, n, 0, n, en.K, en.a_row0 + m0, en.b_row0 + n0, en.pair, 0}});
          continue;
        }
        const int kbeg = (m0 * en.km + n0 * en.kn) / ks * ks;   // triangular operands: rounded down to the step
        const int nst = en.K > kbeg ? (en.K - kbeg + ks - 1) / ks : 0;
        tk.push_back({nst, Tile{e, m0, n0, 0, -1, kbeg, nst, en.K, en.a_row0 + m0, en.b_row0 + n0, en.pair, 0}});
        h.oz_alg_flops += 2.0 * rows * cols * std::max(0, en.K - kbeg);
        exec += 2.0 * BM * BN * (double)nst * ks * prods;
      }
  }
  if (tk.empty()) return 0;
  // Order of the tiles, which CTAs take round-robin.  Operands within the L2: the longest K ranges first, which
  // evens out the CTAs' work.  Larger ones (the ln det products of a slab: 160 MB of planes a matrix): entry by
  // entry in blocks of 12 x 12 tiles, about one per SM, whose A and B rows stay in the L2 while they are in work;
  // by K they ran column by column through every matrix and read 40 GB from DRAM (W at N_aux 2010, 16
  // frequencies: 6.3 ms against 2.4 ms of MMAs).
  double opbytes = 0;
  for (const auto &o : ops)
    opbytes += (double)planes(S) * elem_bytes(S) * o.first->kpad * ((double)o.first->rows + o.second->rows);
  if (opbytes <= 96e6) {
    std::stable_sort(tk.begin(), tk.end(), [](const std::pair<int, Tile> &x, const std::pair<int, Tile> &y) {
      return x.first > y.first;
    });
  } else {
    const int bm = 12 * BM, bn = 12 * BN;
    std::stable_sort(tk.begin(), tk.end(), [bm, bn](const std::pair<int, Tile> &x, const std::pair<int, Tile> &y) {
      const Tile &a = x.second, &b = y.second;
      return std::make_tuple(a.e, a.m0 / bm, a.n0 / bn, a.m0, a.n0) < std::make_tuple(b.e, b.m0 / bm, b.n0 / bn, b.m0, b.n0);
    });
  }
  std::vector<MapPair> mp(ops.size());
  for (size_t i = 0; i < ops.size(); ++i) {
    mp[i].a = make_map(*ops[i].first, BM, 1);
    mp[i].b = make_map(*ops[i].second, BN, planes(S));
    mp[i].ea = ops[i].first->expo;
    mp[i].eb = ops[i].second->expo;
  }
  auto al = [](size_t b) { return (b + 255) / 256 * 256; };
  const size_t b0 = mp.size() * sizeof(MapPair), off1 = al(b0), b1 = entries.size() * sizeof(Entry),
               off2 = off1 + al(b1), b2 = tk.size() * sizeof(Tile), off3 = off2 + al(b2),
               b3 = std::max<size_t>(1, chunks.size()) * sizeof(int);
  std::vector<char> host(off3 + b3);
  std::memcpy(host.data(), mp.data(), b0);
  std::memcpy(host.data() + off1, entries.data(), b1);
  // alpha = +-2^k goes into the epilogue's exponent arithmetic (every GEMM of the path), other
  // values are multiplied in FP64
  for (size_t e = 0; e < entries.size(); ++e) {
    Entry &en = reinterpret_cast<Entry *>(host.data() + off1)[e];
    int ex = 0;
    const double fr = std::frexp(std::fabs(en.alpha), &ex);
    en.alpha_shift = (en.alpha != 0.0 && fr == 0.5) ? ex - 1 : kNoShift;
  }
  Tile *ht = reinterpret_cast<Tile *>(host.data() + off2);
  for (size_t i = 0; i < tk.size(); ++i) ht[i] = tk[i].second;
  if (!chunks.empty()) std::memcpy(host.data() + off3, chunks.data(), chunks.size() * sizeof(int));
  if (s != h.stream) throw Error{LIBRPA_E_ARG, "oz::gemm: launch on a stream other than the handle's"};
  h.upload_async(args, host.data(), off3 + b3);
  const MapPair *dm = (const MapPair *)args.p;
  const Entry *de = (const Entry *)((const char *)args.p + off1);
  const Tile *dt = (const Tile *)((const char *)args.p + off2);
  const int *dc = (const int *)((const char *)args.p + off3);
  // a persistent grid of one CTA per SM (its shared memory and registers fill the SM): the ring and the
  // accumulators run on across its tiles
  int nsm = 0;
  LR_CUDA(cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, h.opts.device));
  const int nt = (int)tk.size(), grid = std::min(nt, nsm);
  const uint64_t stall = Handle::stall_ns(S == S_WIDE ? h.stalls_wide : h.stalls_left);   // testing only
  const Launch l{dm, de, dt, dc, nt, grid, err, stall, s};
  int ms = 0;
  for (const auto &x : tk) ms = std::max(ms, x.first);
  switch (S) {
    case 0: launch<0>(l, ms); break;
    case 1: launch<1>(l, ms); break;
    case 2: launch<2>(l, ms); break;
    case 3: launch<3>(l, ms); break;
    case 4: launch<4>(l, ms); break;
    case S_WIDE: launch<S_WIDE>(l, ms); break;
    case S_TF32: launch<S_TF32>(l, ms); break;
    case S_TF32X3: launch<S_TF32X3>(l, ms); break;
    case 5: BN == 64 ? launch<5, 64>(l, ms) : launch<5>(l, ms); break;
    default: throw Error{LIBRPA_E_ARG, "oz::gemm: no such operand form"};
  }
  ++launch_counter();
  LR_CUDA(cudaGetLastError());
  h.oz_exec_flops = exec;
  return nt;
}

long long gemm_grouped(const Sliced &a, const Sliced &b, const std::vector<Entry> &entries, int *err,
                       cudaStream_t s, Handle &h, DevBuf &args, const StageFn *stage_fn) {
  std::vector<Entry> es(entries);
  for (Entry &e : es) e.pair = 0;
  return gemm_multi({{&a, &b}}, es, err, s, h, args, stage_fn);
}

long long gemm(const Sliced &a, const Sliced &b, int M, int N, int batch, const Out &out, int km, int kn,
               int lower_div, int *err, cudaStream_t s, Handle &h) {
  if (a.K != b.K) throw Error{LIBRPA_E_ARG, "oz::gemm: K mismatch"};
  // an operand holding a single entry is shared by every batch entry
  const int a_pb = (batch > 1 && a.rows == M) ? 0 : a.rows / batch;
  const int b_pb = (batch > 1 && b.rows == N) ? 0 : b.rows / batch;
  std::vector<Entry> es(batch);
  for (int i = 0; i < batch; ++i) {
    Entry &e = es[i];
    e.a_row0 = i * a_pb;
    e.b_row0 = i * b_pb;
    e.M = M;
    e.N = N;
    e.K = a.K;
    e.km = km;
    e.kn = kn;
    e.lower_div = lower_div;
    e.C = out.C + (long long)i * out.batch_stride * (out.mode == 0 || out.mode == 4 ? 1 : 2);
    e.ldc = out.ldc;
    e.mode = out.mode;
    e.alpha = out.alpha;
    e.beta = out.beta;
  }
  return gemm_grouped(a, b, es, err, s, h, h.oz_args);
}

}  // namespace oz
}  // namespace librpa

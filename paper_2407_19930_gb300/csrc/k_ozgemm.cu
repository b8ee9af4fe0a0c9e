// FP64-accurate GEMM on the BF16 tensor cores of sm_103a (see ozgemm.h for the scheme).
//
// Operands are split once into BF16 digit planes (k_row_expo + k_digits, or k_plain for plain
// BF16); the GEMM kernel streams them with TMA (cp.async.bulk.tensor) into a shared-memory ring
// and multiplies every digit pair with tcgen05.mma (kind::f16, BF16 x BF16 -> FP32, M = 128,
// N = 64, K = 16) into the TMEM accumulator of its diagonal; flush groups (the largest K range
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
    return k < K ? base[off[e] + (long long)rr * K + k] : 0.0;
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
  int d[4][S];
#pragma unroll
  for (int q = 0; q < 4; ++q) make_digits<S>(k0 + q < K ? src.get(r, k0 + q) : 0.0, E, d[q]);
  const long long o = ((long long)row0 + r) * kpad + k0;
#pragma unroll
  for (int s = 0; s < S; ++s) {
    __nv_bfloat162 lo = __floats2bfloat162_rn((float)d[0][s], (float)d[1][s]);
    __nv_bfloat162 hi = __floats2bfloat162_rn((float)d[2][s], (float)d[3][s]);
    uint2 w;
    w.x = *reinterpret_cast<unsigned *>(&lo);
    w.y = *reinterpret_cast<unsigned *>(&hi);
    *reinterpret_cast<uint2 *>(dig + s * plane + o) = w;
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

// An output tile; c_n >= 0: only the K stages listed at chunks[c_off .. + c_n) (in units of the
// stage's K) are summed -- block-sparse operands, the others multiply exact zeros.
struct Tile {
  int e, m0, n0, c_off, c_n;
};

__host__ __device__ constexpr uint32_t tmem_cols(int cols) { return cols <= 128 ? 128 : cols <= 256 ? 256 : 512; }
constexpr int PBK = 32;   // K per stage: one 64-byte swizzle row of BF16 (16 TF32 values)
// pipeline depth: what fits in the shared memory beside the staging area (180 KB with 3 or 5 planes, 192 KB
// with 8)
__host__ __device__ constexpr int ring_stages(int S) {
  return S == S_WIDE ? 2 : S == 5 ? 3 : S == 4 ? 3 : S == 3 ? 5 : planes(S) == 2 ? 6 : 8;
}
// accumulator sets in TMEM: two where they fit (up to 4 planes), so that one is drained while the other fills
__host__ __device__ constexpr int acc_sets(int S) { return !is_digits(S) || S <= 4 ? 2 : 1; }
__host__ __device__ constexpr int acc_cols(int S) { return (is_digits(S) ? S : 1) * BN; }
// epilogue warps of the S variant
__host__ __device__ constexpr int epi_warps(int S) { return is_digits(S) ? 16 : 4; }
// columns the epilogue stages at a time (what the shared memory beside the ring holds), pitch + 1, and the
// bytes of its staging area
__host__ __device__ constexpr int stage_cols(int S) { return S == S_WIDE ? 4 : 8; }
__host__ __device__ constexpr int stage_bytes(int S) { return is_digits(S) ? epi_warps(S) * 32 * (stage_cols(S) + 1) * 8 : 0; }
// digit planes of B multiplied by one MMA: at most 256 columns
constexpr int kStack = 256 / BN;

// Operands of the entries of one launch that share them: tensor maps of the A and B digit planes
// (global memory, 128-byte aligned) and their row exponents.
struct alignas(128) MapPair {
  CUtensorMap a, b;
  const int *ea, *eb;
};

// Pipelined, warp-specialised kernel: CTA c takes tiles c, c + gridDim.x, ... (128 x 64 output
// tiles of the launch's entries, sorted by decreasing K range on the host), keeping its barriers and
// TMEM across them (a persistent grid of one CTA per SM).
//   warp EW (one lane): TMA producer over a ring of NST shared-memory stages (each the NP digit
//     planes of a 128 x 32 A slice and a 64 x 32 B slice, SWIZZLE_64B, K-major); the ring runs on
//     across tiles, so the next tile's loads overlap this tile's MMAs and epilogue;
//   warp EW + 1 (one lane): tcgen05.mma issuer; commits free a stage when its MMAs complete and, at
//     the end of a flush group, signal the epilogue; the next group (of this or the next tile) uses the
//     other accumulator set (up to 4 planes), or starts once the epilogue has drained the only one.  The B planes lie one after the other in a
//     stage and the accumulators of consecutive diagonals in consecutive columns, so plane s of A
//     meets up to four planes of B in one MMA of N = 256: 6 MMAs per K step of 16 with 5 planes in place of 15
//     of N = 64, and A read from shared memory 6 times instead of 15 (54 KB a step, below what the
//     MMAs' 480 cycles can take; at N = 64 the 90 KB held the tensor pipe at two thirds);
//   warps 0..EW-1: epilogue; warp w owns TMEM lanes 32 (w % 4) .. + 31 (= tile rows).  With EW = 16
//     (digit planes) warp w takes columns 16 (w / 4) .. + 15 and after each flush group moves the
//     diagonal accumulators into exact int64 register sums (16 per thread, of two words each with 8
//     planes); with EW = 4 (plain BF16 / TF32, one group) each warp takes all 64 columns into
//     registers.  The TMEM columns go back to the issuer before the values are converted and stored, so
//     conversion and stores overlap the next tile's MMAs.  The conversion (~30 integer instructions) is
//     bound by its latency: four warps per scheduler, 16 independent sums each.
// stall_ns > 0 (testing only): the MMA issuer first waits that long on an mbarrier nothing arrives
// at, so the CTA takes the bounded-wait failure path.  On any failure the CTA sets *err, stops
// issuing, waits (with the full limit) for the TMA copies and MMAs it has already issued, frees its
// TMEM and returns.
template <int S>
__global__ void __launch_bounds__(32 * (epi_warps(S) + 2), 1)
    k_ozgemm(const MapPair *__restrict__ maps, const Entry *__restrict__ entries, const Tile *__restrict__ tiles,
             const int *__restrict__ chunks, int ntiles, int *err, uint64_t stall_ns, int stage_in_ring) {
  constexpr bool TF = S == S_TF32 || S == S_TF32X3;   // kind::tf32
  constexpr bool PLAIN = !is_digits(S);                // one FP32 accumulator over all K
  constexpr bool WIDE = S == S_WIDE;                   // two-word sums
  constexpr int NP = planes(S);                        // planes per operand
  constexpr int NST = ring_stages(S);
  constexpr int KS = TF ? PBK / 2 : PBK;               // K elements per stage (64 bytes per row)
  constexpr uint32_t A_BYTES = BM * 64, B_BYTES = BN * 64;
  constexpr uint32_t STAGE = NP * (A_BYTES + B_BYTES);
  // K steps per flush group: NP pairs x (32 G) x 2^14 <= 2^24 keeps the FP32 sums exact; plain
  // forms accumulate over the whole K in FP32
  constexpr int G = PLAIN ? (1 << 30) : 32 / NP;
  constexpr int EPI_WARPS = epi_warps(S), HALF = BN * 4 / EPI_WARPS;   // HALF: columns per epilogue warp
  constexpr int SETS = acc_sets(S);                    // accumulator sets, one flush group each
  constexpr uint32_t SET_COLS = acc_cols(S), TMEM_COLS = tmem_cols(SETS * acc_cols(S));
  static_assert(SETS * acc_cols(S) <= 512, "k_ozgemm: TMEM");
  extern __shared__ uint8_t smem_raw[];
  __shared__ uint64_t full[NST], empty[NST], tfull[SETS], tempty[SETS], mdone, never;
  __shared__ uint32_t tmem_slot;
  __shared__ volatile int abort_flag;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  uint8_t *smem = (uint8_t *)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
  // the epilogue's staging area: in the pipeline's stages when the CTA has a single tile (they are
  // idle once its last MMA completed), else after them
  uint8_t *stage_out = stage_in_ring ? smem : smem + NST * STAGE;
  if (tid == 0) {
#pragma unroll
    for (int s = 0; s < NST; ++s) {
      mbar_init(&full[s], 1);
      mbar_init(&empty[s], 1);
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
  // K range of a tile: from (m0 km + n0 kn) rounded down to the stage size (triangular operands),
  // or the tile's list of stages
  auto steps_of = [&](const Entry &en, const Tile &tl, int &kbeg) {
    kbeg = (tl.m0 * en.km + tl.n0 * en.kn) / KS * KS;
    if (tl.c_n >= 0) return tl.c_n;
    return en.K > kbeg ? (en.K - kbeg + KS - 1) / KS : 0;
  };
  auto k_of = [&](const Tile &tl, int kbeg, int i) { return tl.c_n >= 0 ? chunks[tl.c_off + i] * KS : kbeg + i * KS; };
  if (warp == EPI_WARPS) {
    if (lane == 0) {
      long long it = 0;   // stages issued so far (all tiles)
      for (int t = blockIdx.x; t < ntiles && !abort_flag; t += gridDim.x) {
        const Tile tl = tiles[t];
        const Entry &en = entries[tl.e];
        const MapPair *mp = maps + en.pair;
        int kbeg;
        const int nsteps = steps_of(en, tl, kbeg);
        const int arow = en.a_row0 + tl.m0, brow = en.b_row0 + tl.n0;
        for (int i = 0; i < nsteps; ++i, ++it) {
          const int st = (int)(it % NST);
          if (abort_flag || !mbar_wait(&empty[st], (uint32_t)(((it / NST) & 1) ^ 1), WAIT_NS, &abort_flag)) {
            abort_flag = 1;
            break;
          }
          mbar_expect_tx(&full[st], STAGE);
          uint8_t *sa = smem + st * STAGE, *sb = sa + NP * A_BYTES;
          const int k0 = k_of(tl, kbeg, i);
#pragma unroll
          for (int p = 0; p < NP; ++p) tma_load_3d(sa + p * A_BYTES, &mp->a, &full[st], k0, arow, p);
#pragma unroll
          for (int p = 0; p < NP; ++p) tma_load_3d(sb + p * B_BYTES, &mp->b, &full[st], k0, brow, p);
        }
      }
      // after a failure: the copies of the last NST issued stages may still be in flight (earlier
      // ones were consumed); wait for each to land before the CTA exits
      if (abort_flag)
        for (long long i = it > NST ? it - NST : 0; i < it; ++i)
          mbar_wait(&full[i % NST], (uint32_t)((i / NST) & 1), WAIT_NS);
    }
  } else if (warp == EPI_WARPS + 1) {
    if (lane == 0) {
      if (stall_ns) {   // testing only: a barrier nothing arrives at
        mbar_wait(&never, 0, stall_ns, &abort_flag);
        abort_flag = 1;
      }
      long long it = 0, g = 0;   // stages consumed, flush groups committed (all tiles)
      for (int t = blockIdx.x; t < ntiles && !abort_flag; t += gridDim.x) {
        const Tile tl = tiles[t];
        int kbeg;
        const int nsteps = steps_of(entries[tl.e], tl, kbeg);
        for (int i = 0; i < nsteps; ++i, ++it) {
          const int st = (int)(it % NST), c = i % G;
          // a new group needs its accumulators drained by the epilogue (group g - SETS, any tile)
          if (c == 0 && g >= SETS &&
              (abort_flag || !mbar_wait(&tempty[g % SETS], (uint32_t)((g / SETS - 1) & 1), WAIT_NS, &abort_flag))) {
            abort_flag = 1;
            break;
          }
          if (abort_flag || !mbar_wait(&full[st], (uint32_t)((it / NST) & 1), WAIT_NS, &abort_flag)) {
            abort_flag = 1;
            break;
          }
          tc_fence_after();
          const uint32_t sa = smem_u32(smem + st * STAGE), sb = sa + NP * A_BYTES;
          const uint32_t tacc = tmem + (uint32_t)(g % SETS) * SET_COLS;
          if constexpr (PLAIN) {
            // one accumulator for all products: hi hi (and hi lo, lo hi of the 3xTF32 split)
#pragma unroll
            for (int s = 1; s <= NP; ++s)
#pragma unroll
              for (int u = 1; u + s <= NP + 1; ++u)
#pragma unroll
                for (int j = 0; j < 2; ++j) {   // two MMAs of 32 bytes of K per 64-byte row
                  const uint64_t da = smem_desc64(sa + (s - 1) * A_BYTES + 32 * j);
                  const uint64_t db = smem_desc64(sb + (u - 1) * B_BYTES + 32 * j);
                  const uint32_t accum = (c == 0 && j == 0 && s == 1 && u == 1) ? 0u : 1u;
                  if constexpr (TF)
                    umma_tf32(tacc, da, db, idesc(BN, true), accum);
                  else
                    umma(tacc, da, db, idesc(BN, false), accum);
                }
          } else {
            // plane s of A by planes u .. u + w - 1 of B (N = 64 w), into the diagonals s + u ..
#pragma unroll
            for (int j = 0; j < 2; ++j)
#pragma unroll
              for (int s = 1; s <= NP; ++s)
#pragma unroll
                for (int u = 1; u + s <= NP + 1; u += kStack) {
                  const int w = NP + 2 - s - u < kStack ? NP + 2 - s - u : kStack;
                  const uint64_t da = smem_desc64(sa + (s - 1) * A_BYTES + 32 * j);
                  const uint64_t db = smem_desc64(sb + (u - 1) * B_BYTES + 32 * j);
                  umma(tacc + (uint32_t)(s + u - 2) * BN, da, db, idesc(BN * w, false), (c == 0 && j == 0 && s == 1) ? 0u : 1u);
                }
          }
          umma_commit(&empty[st]);
          if (c == G - 1 || i == nsteps - 1) {
            umma_commit(&tfull[g % SETS]);
            ++g;
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
    long long g = 0;   // flush groups drained (all tiles)
    for (int t = blockIdx.x; t < ntiles; t += gridDim.x) {
      const Tile tl = tiles[t];
      const Entry &en = entries[tl.e];
      int kbeg;
      const int nsteps = steps_of(en, tl, kbeg);
      const int ngroups = (nsteps + G - 1) / G;
      const int m0 = tl.m0, n0 = tl.n0;
      // digit planes: exact sums of the diagonals, in units of the last one's scale (WIDE: the first four
      // diagonals in acch, in units of the fourth's, the last four in acc)
      long long acc[PLAIN ? 1 : HALF], acch[WIDE ? HALF : 1];
      uint32_t fa[PLAIN ? HALF : 1];   // plain forms: the FP32 accumulators
      // FP32-pair outputs of a tile with a single flush group (the short-K GEMMs of the chi0 steps): the
      // diagonal sums, integers below 2^24 times their powers of two, are summed into an unevaluated FP32
      // pair by exact two-sums, held in the halves of acc -- FP32 arithmetic instead of the integer
      // conversions
      const bool fpath = !PLAIN && !WIDE && ngroups == 1 && en.mode == 3 && en.alpha_shift != kNoShift;
      if constexpr (!PLAIN) {
#pragma unroll
        for (int j = 0; j < HALF; ++j) acc[j] = 0;
        if constexpr (WIDE) {
#pragma unroll
          for (int j = 0; j < HALF; ++j) acch[j] = 0;
        }
      }
      bool ok_all = true;
      for (int gi = 0; gi < ngroups; ++gi, ++g) {
        bool ok = !abort_flag && mbar_wait(&tfull[g % SETS], (uint32_t)((g / SETS) & 1), WAIT_NS, &abort_flag);
        const uint32_t tbase = tbase0 + (uint32_t)(g % SETS) * SET_COLS;
        ok = __all_sync(0xffffffffu, ok);
        if (!ok) {
          abort_flag = 1;
          ok_all = false;
          break;
        }
        tc_fence_after();
        if constexpr (!PLAIN) {
          // one diagonal at a time, the next load in flight while this one is added
          constexpr int CB = HALF / 16, RB = WIDE ? 1 : 2;
          uint32_t r[RB][16];
          if (!WIDE) tmem_ld16(tbase, r[0]);
#pragma unroll
          for (int l = 0; l < S * CB; ++l) {
            const int d = l / CB, cb = l % CB * 16;
            if (WIDE) tmem_ld16(tbase + (uint32_t)d * BN + cb, r[0]);
            tmem_ld_wait(r[l % RB]);
            if (!WIDE && l + 1 < S * CB)
              tmem_ld16(tbase + (uint32_t)((l + 1) / CB) * BN + (l + 1) % CB * 16, r[(l + 1) % RB]);
            if (!WIDE && fpath) {
#pragma unroll
              for (int j = 0; j < 16; ++j) {
                const float t = __uint_as_float(r[l % RB][j]) * (float)(1ull << (8 * (S - 1 - d)));   // exact
                const float hi = __int_as_float((int)(acc[cb + j] & 0xFFFFFFFFll));
                float lo = __int_as_float((int)(acc[cb + j] >> 32));
                const float sm = hi + t, bb = sm - hi;
                lo += (hi - (sm - bb)) + (t - bb);
                acc[cb + j] = ((long long)__float_as_int(lo) << 32) | (long long)(uint32_t)__float_as_int(sm);
              }
              continue;
            }
#pragma unroll
            for (int j = 0; j < 16; ++j) {
              const int v = __float2int_rn(__uint_as_float(r[l % RB][j]));
              if constexpr (WIDE) {
                if (d < 4)
                  acch[cb + j] += (long long)v * (1 << (8 * (3 - d)));
                else
                  acc[cb + j] += (long long)v * (1 << (8 * (7 - d)));
              } else if (S == 5 && d == 0) {
                acc[cb + j] += (long long)((unsigned long long)(unsigned)v << 32);   // 2^32 v (mod 2^64)
              } else {
                acc[cb + j] += (long long)v * (1 << (8 * (S - 1 - d) % 32));
              }
            }
          }
        } else {
#pragma unroll
          for (int cb = 0; cb < HALF / 16; ++cb) {
            uint32_t r[16];
            tmem_ld16(tbase + cb * 16, r);
            tmem_ld_wait(r);
#pragma unroll
            for (int j = 0; j < 16; ++j) fa[cb * 16 + j] = r[j];
          }
        }
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(&tempty[g % SETS]);   // the accumulators may be overwritten now
      }
      if (!ok_all) break;
      const int eM = en.M, eN = en.N, mode = en.mode;
      const long long ldc = en.ldc;
      double *const C = en.C;
      const double alpha = en.alpha, beta = en.beta;
      const bool pow2 = en.alpha_shift != kNoShift;   // alpha = +-2^alpha_shift: folded into the exponent
      const int row = m0 + 32 * quad + lane;          // thread = tile row (the TMEM lane layout)
      const bool row_ok = row < eM;
      auto at = [&](int r_, int c_) {   // one output element (modes 0, 1, 2, 4)
        return mode == 0   ? C + (long long)r_ * ldc + c_
               : mode == 1 ? C + 2 * ((long long)(r_ >> 1) * ldc + c_) + (r_ & 1)
               : mode == 4 ? C + (long long)c_ * ldc + r_
                           : C + 2 * ((long long)c_ * ldc + (r_ >> 1)) + (r_ & 1);
      };
      if constexpr (PLAIN) {
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
            double *p = at(row, col);
            *p = beta == 0.0 ? v : v + beta * *p;
          }
        }
      } else {
        constexpr int SC = stage_cols(S);
        const int cbase = n0 + half * HALF, nc = min(HALF, eN - cbase);   // nc: live columns of the warp
        if (nc <= 0) continue;
        const MapPair &mp = maps[en.pair];
        const int ash = (pow2 ? en.alpha_shift : 0) - 14 - 8 * (S - 1);
        const int ea = (row_ok ? mp.ea[en.a_row0 + row] : 0) + ash;
        const int *eb = mp.eb + en.b_row0 + cbase;
        const bool aneg = pow2 && alpha < 0.0;
        // a row or column with an infinity or a NaN has the exponent 1025 (finite ones at most 1024)
        const bool row_nan = ea - ash > 1024;
        // the values in place of the sums: FP64 bits, or (mode 3) the pair (hi, lo)
#pragma unroll
        for (int j = 0; j < HALF; ++j) {
          const int e_b = j < nc ? eb[j] : 0, sh = ea + e_b;
          float2 pr;
          if (fpath) {
            // renormalise the pair, then scale it by 2^sh (exact in the normal range)
            float hi = __int_as_float((int)(acc[j] & 0xFFFFFFFFll)), lo = __int_as_float((int)(acc[j] >> 32));
            const float sm = hi + lo;
            lo = lo - (sm - hi);
            hi = sm;
            const int eh = (int)((__float_as_uint(hi) >> 23) & 0xFF);
            const float sc = __uint_as_float((uint32_t)(sh + 127) << 23);
            pr = make_float2(hi * sc, lo * sc);
            if (!(sh >= -126 && sh <= 127 && (hi == 0.f || (eh + sh >= 1 && eh + sh <= 254)))) {
              const double dv = ldexp((double)hi + (double)lo, sh);   // outside the FP32 range: through FP64
              pr.x = __double2float_rn(dv);
              pr.y = __double2float_rn(dv - (double)pr.x);
            }
            if (aneg) pr = make_float2(-pr.x, -pr.y);
          } else if (!WIDE && mode == 3 && pow2) {
            pr = i64_to_f32x2(aneg ? -acc[j] : acc[j], sh);
          } else {
            double v;
            if constexpr (WIDE)
              v = i96_to_f64(acch[j], acc[j], sh);
            else
              v = i64_to_f64(acc[j], sh);
            if (!pow2)
              v *= alpha;
            else if (aneg)
              v = -v;
            if (row_nan || e_b > 1024) v = __longlong_as_double(0x7FF8000000000000ll);
            acc[j] = __double_as_longlong(v);
            if (mode == 3) {
              pr.x = __double2float_rn(v);
              pr.y = __double2float_rn(v - (double)pr.x);
            }
          }
          if (mode == 3) {
            if (row_nan || e_b > 1024) pr = make_float2(__uint_as_float(0x7FC00000u), 0.f);
            acc[j] = (long long)(((unsigned long long)__float_as_uint(pr.y) << 32) | __float_as_uint(pr.x));
          }
        }
        if (mode == 2 || mode == 4) {
          // transposed outputs: consecutive along the lanes (tile rows)
          if (row_ok) {
#pragma unroll
            for (int j0 = 0; j0 < HALF; j0 += 8) {
              double old[8];
              if (beta != 0.0) {
#pragma unroll
                for (int j = 0; j < 8; ++j)
                  if (j0 + j < nc) old[j] = *at(row, cbase + j0 + j);
              }
#pragma unroll
              for (int j = 0; j < 8; ++j)
                if (j0 + j < nc) {
                  const double v = __longlong_as_double(acc[j0 + j]);
                  *at(row, cbase + j0 + j) = beta == 0.0 ? v : v + beta * old[j];
                }
            }
          }
          continue;
        }
        // row-major outputs: through the staging area, lanes along SC columns of 32 / SC rows
        long long *stg = reinterpret_cast<long long *>(stage_out) + warp * 32 * (SC + 1);
        const int cl = lane % SC, rl = lane / SC, rbase = m0 + 32 * quad + rl;
#pragma unroll
        for (int cb = 0; cb < HALF / SC; ++cb) {
          if (cb * SC >= nc) break;   // the same for the whole warp
          const int col = cbase + cb * SC + cl;
          const bool col_ok = cb * SC + cl < nc;
          double old[SC];
          if (beta != 0.0) {
#pragma unroll
            for (int i = 0; i < SC; ++i)
              if (col_ok && rbase + i * (32 / SC) < eM) old[i] = *at(rbase + i * (32 / SC), col);
          }
#pragma unroll
          for (int j = 0; j < SC; ++j) stg[lane * (SC + 1) + j] = acc[cb * SC + j];
          __syncwarp();
#pragma unroll
          for (int i = 0; i < SC; ++i) {
            const int rr = rl + i * (32 / SC), grow = rbase + i * (32 / SC);
            if (!col_ok || grow >= eM) continue;
            const double v = __longlong_as_double(stg[rr * (SC + 1) + cl]);
            if (mode == 3)   // the 8 bytes hold the pair (hi, lo)
              C[(long long)grow * ldc + col] = v;
            else
              *at(grow, col) = beta == 0.0 ? v : v + beta * old[i];
          }
          __syncwarp();
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

}  // namespace

CUtensorMap make_map(const Sliced &o, int box_rows, int box_planes) {
  CUtensorMap m;
  const cuuint64_t eb = (cuuint64_t)elem_bytes(o.S);
  const cuuint64_t dims[3] = {(cuuint64_t)o.kpad, (cuuint64_t)o.rows, (cuuint64_t)planes(o.S)};
  const cuuint64_t strides[2] = {(cuuint64_t)o.kpad * eb, (cuuint64_t)o.kpad * eb * (cuuint64_t)o.rows};
  const cuuint32_t box[3] = {(cuuint32_t)(64 / eb), (cuuint32_t)box_rows, (cuuint32_t)box_planes};   // 64-byte rows
  const cuuint32_t estr[3] = {1, 1, 1};
  const CUtensorMapDataType dt = eb == 4 ? CU_TENSOR_MAP_DATA_TYPE_FLOAT32 : CU_TENSOR_MAP_DATA_TYPE_BFLOAT16;
  const CUresult r = g_encode(&m, dt, 3, o.digits, dims, strides, box, estr,
                              CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_64B,
                              CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  if (r != CUDA_SUCCESS) throw Error{LIBRPA_E_CUDA, "cuTensorMapEncodeTiled failed: " + std::to_string((int)r)};
  return m;
}

namespace {

// dynamic shared memory of k_ozgemm<S>: the pipeline's stages and the epilogue's staging area, overlapping
// when every CTA has one tile (the shared memory, and so the CTAs an SM holds at once, stay those
// of the stages alone)
constexpr int ring_bytes(int S) { return ring_stages(S) * planes(S) * (BM + BN) * 64; }
constexpr int gemm_smem(int S, bool in_ring) {
  return (in_ring ? (ring_bytes(S) > stage_bytes(S) ? ring_bytes(S) : stage_bytes(S)) : ring_bytes(S) + stage_bytes(S)) + 1024;
}

template <int S>
void launch(const MapPair *mp, const Entry *e, const Tile *t, const int *c, int ntiles, int grid, int *err,
            uint64_t stall_ns, cudaStream_t s) {
  static_assert(gemm_smem(S, false) <= 226 * 1024, "k_ozgemm: shared memory");
  const bool in_ring = grid >= ntiles;
  // one limit for every launch: host threads set it concurrently, and a launch's own size could
  // undercut another thread's launch
  LR_CUDA(cudaFuncSetAttribute(k_ozgemm<S>, cudaFuncAttributeMaxDynamicSharedMemorySize, gemm_smem(S, false)));
  k_ozgemm<S><<<grid, 32 * (epi_warps(S) + 2), gemm_smem(S, in_ring), s>>>(mp, e, t, c, ntiles, err, stall_ns, in_ring);
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
                   long long batch_stride, Sliced &out, cudaStream_t s) {
  const int rows_pb = as_a ? 2 * n_out : n_out;
  CplxSrc c{src, ld, batch_stride, rows_pb, (int)op, as_a};
  split_any(c, rows_pb * batch, 2 * n_k, 0, out, s);
}

void split_gather(const GatherSrc &src, int rows, int K, Sliced &out, cudaStream_t s) {
  GatherDev g{src};
  split_any(g, rows, K, 0, out, s);
}

void split_ragged(const double *base, const long long *off, const int *Ke, int rows_per_entry, int n_entries,
                  int Kmax, Sliced &out, cudaStream_t s, bool expo_given) {
  RaggedSrc r{base, off, Ke, rows_per_entry};
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
  const int S = ops[0].first->S;
  for (const auto &o : ops)
    if (o.first->S != S || o.second->S != S || S < 0 || S > S_WIDE)
      throw Error{LIBRPA_E_ARG, "oz::gemm: operand mismatch"};
  init();
  // tiles with their K range in stages; MMA flops issued: per tile BM x BN x (K rounded up to the
  // K step) per digit-plane product
  const double prods = is_digits(S) ? S * (S + 1) / 2.0 : S == S_TF32X3 ? 3.0 : 1.0;
  const int ks = elem_bytes(S) == 4 ? PBK / 2 : PBK;   // K elements per pipeline stage
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
        if (stage_fn && (*stage_fn)(e, m0, rows, n0, cols, ks, en.K, cl)) {
          double kk = 0;
          for (int c : cl) kk += std::min(ks, en.K - c * ks);
          h.oz_alg_flops += 2.0 * rows * cols * kk;
          tk.push_back({(int)cl.size(), Tile{e, m0, n0, (int)chunks.size(), (int)cl.size()}});
          chunks.insert(chunks.end(), cl.begin(), cl.end());
          exec += 2.0 * BM * BN * (double)cl.size() * ks * prods;
          continue;
        }
        const int kbeg = (m0 * en.km + n0 * en.kn) / ks * ks;   // as in the kernel
        const int nst = en.K > kbeg ? (en.K - kbeg + ks - 1) / ks : 0;
        tk.push_back({nst, Tile{e, m0, n0, 0, -1}});
        h.oz_alg_flops += 2.0 * rows * cols * std::max(0, en.K - kbeg);
        exec += 2.0 * BM * BN * (double)nst * ks * prods;
      }
  }
  if (tk.empty()) return 0;
  // the longest K ranges first: CTAs take tiles round-robin, so this evens out their work
  std::stable_sort(tk.begin(), tk.end(), [](const std::pair<int, Tile> &x, const std::pair<int, Tile> &y) {
    return x.first > y.first;
  });
  std::vector<MapPair> mp(ops.size());
  for (size_t i = 0; i < ops.size(); ++i) {
    mp[i].a = make_map(*ops[i].first, BM);
    mp[i].b = make_map(*ops[i].second, BN);
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
  // testing only: the handle's first opts.test_stall_gemms launches take the failure path
  uint64_t stall = 0;
  if (h.stalls_left > 0 && S != S_WIDE) {
    --h.stalls_left;
    stall = 100000;   // 100 us per CTA
  }
  switch (S) {
    case 0: launch<0>(dm, de, dt, dc, nt, grid, err, stall, s); break;
    case 1: launch<1>(dm, de, dt, dc, nt, grid, err, stall, s); break;
    case 2: launch<2>(dm, de, dt, dc, nt, grid, err, stall, s); break;
    case 3: launch<3>(dm, de, dt, dc, nt, grid, err, stall, s); break;
    case 4: launch<4>(dm, de, dt, dc, nt, grid, err, stall, s); break;
    case S_WIDE: launch<S_WIDE>(dm, de, dt, dc, nt, grid, err, stall, s); break;
    case S_TF32: launch<S_TF32>(dm, de, dt, dc, nt, grid, err, stall, s); break;
    case S_TF32X3: launch<S_TF32X3>(dm, de, dt, dc, nt, grid, err, stall, s); break;
    default: launch<5>(dm, de, dt, dc, nt, grid, err, stall, s); break;
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

// O assembly of the chi0 contraction on the tensor cores (k_oasm.cu).
#pragma once

#include <cuda_runtime.h>

#include "ozgemm.h"

namespace librpa {

// A (R, tau) point of the contraction.
struct Point {
  int iR, itau;
  int R[3];
};

// Row pitch of O_U (rows nu, columns (i, kap)): n_U m_U rounded up to even, so that rows start on 16 bytes.
__host__ __device__ constexpr int o_pitch(int n, int m) { return (n * m + 1) & ~1; }

// Operands of the O assembly: O^nu_{ik}(K R1) for every (point, U, V), written as O_U[nu][(i, kap)].
struct OArgs {
  const double *G;       // [2][ntau][nR][nao][nao]
  size_t g_gstride;
  int nR_stride, nao, natoms, naux, n1, n2, n3;
  const Point *pts;
  const int *n_ao, *n_aux, *ao_off, *aux_off, *m;
  const int *kap;            // per-U column table {K, R0, R1, R2, ao(K)+k, union column}
  const long long *kap_off;
  const double *N;           // [P][2][sum_V n_aux_V n_V M_all]
  const long long *n_off;
  long long n_sz_g, n_sz_p;
  int m_all;
  const double *X;           // [P][2][sum_V nao n_aux_V n_V]
  const long long *x_off;
  long long x_sz_g, x_sz_p;
  double *O;                 // [P][sum_U naux n_U m_U]
  const long long *o_off;
  long long o_sz_p;
  // under screening: 1 where the O block is exactly zero ([P][U][V][64-column chunk], zero_chunks of them), else
  // NULL
  const unsigned char *zero;
  int zero_chunks;
};

namespace oasm {

// Rows of U's packed columns in groups of up to 8 that are consecutive union columns, 16 groups to a tile of 128 rows.
struct Group {
  int urow, kap, live;   // first union column, first packed column, live rows (1..8)
};
constexpr int kTileGroups = 16;

// What the tensor-core kernels need beside OArgs: the group tables (device), and the digit planes of N and X
// they build: rows (point, nu, union column) and (point, nu, 16 U + i), 32 columns t.
struct Tables {
  const Group *groups;      // all atoms' groups, a tile's padded to 16 (live = 0)
  const int *tile_off;      // [natoms + 1]: first tile of U (tile x has groups 16 x ..)
  const int *aux_atom;      // [naux]
  const int *ao_row;        // [nao]: 16 U + i
  int max_tiles;
};
constexpr int kMaxAo = 16;   // largest n_ao of an atom

// digit planes of N and X rows of one point (rows of the Sliced operands, K = 32)
inline long long n_rows(int naux, int m_all) { return (long long)naux * m_all; }
inline long long x_rows(int naux, int natoms) { return (long long)naux * natoms * kMaxAo; }

// O for np points with S digit planes (3, 5 or 8): splits N and X into nd and xd, then one launch over every
// (point, U, V, tile).  expo: row exponents of O's digit planes (rows (p, U, nu), initialised to -1022), built by
// atomicMax.  err: set to 1 when a bounded wait ran out.  nans: G or C may hold an infinity or a NaN.  stall_ns > 0 (testing only): the failure path, as in
// k_ozgemm.
void run(int S, const OArgs &a, const Tables &t, int np, oz::Sliced &nd, oz::Sliced &xd, int *expo, int *err,
         bool nans, uint64_t stall_ns, cudaStream_t s);

}  // namespace oasm
}  // namespace librpa

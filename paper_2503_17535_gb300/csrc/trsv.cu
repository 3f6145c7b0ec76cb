// Triangular solves of batches of LU factors against few right-hand sides
// (the solve and adjoint passes): X <- U^{-1} L^{-1} X or its conjugate
// transpose X <- L^{-H} U^{-H} X, both triangles in one launch, up to 8
// columns at a time.
//
// Many matrices: one CTA each (k_trsv_block), the diagonal blocks solved by
// substitution; several CTAs per SM hide each other's chains and the FP64 pipe
// is the bound (n^2 multiply-adds per column).
//
// Few matrices: one thread-block cluster each (k_trsv_cluster).  The 32-row
// blocks go round the CTAs; per block its owner sums the contributions of the
// earlier ones, multiplies by the precomputed inverse of the diagonal block
// (k_block_inverses, once per factor), corrects the result by the inverse times
// its residual if the block is ill-conditioned, and writes the solution into the
// shared memory of every CTA; after one cluster barrier every CTA subtracts its
// contribution from its own later blocks.  The chain per block is two 32 x 32
// products on one SM (512 cycles each for real data), four with the correction,
// the barrier and two or four short sums.
//
// The recursive form (one launch per 32-row block and one product per split)
// took 17 us per launch whatever its size.  Solves with a new source, all
// launches: Helmholtz 4096 leaves 9.4 -> 5.3 ms, 3D elliptic 6.3 -> 3.0,
// adaptive 19.5 -> 4.4; per 32-row block of a cluster solve 2.3 us (real).
#include <cooperative_groups.h>

#include <algorithm>

#include "linalg.h"

namespace hps {
namespace {

__device__ __forceinline__ double shfl_v(double v, int src) { return __shfl_sync(0xffffffffu, v, src); }
__device__ __forceinline__ cplx shfl_v(cplx v, int src) {
  return cplx(__shfl_sync(0xffffffffu, v.re, src), __shfl_sync(0xffffffffu, v.im, src));
}

constexpr int NT = 128, NW = 4;   // threads and warps of a CTA
constexpr int MAXN = 8;           // right-hand sides per launch column group
constexpr size_t BLOCK_SMEM = 200 * 1024;   // most that k_trsv_block takes

// Columns that a CTA of a launch for nrhs right-hand sides takes at a time; its
// shared memory, and so the rule that takes the launch, go with them.
int few_cols(int nrhs) { return nrhs <= 2 ? nrhs : nrhs <= 4 ? 4 : MAXN; }

// ------------------------------------------------------------ many matrices

// Entry (r, c) of the 32 x 32 block whose rows start at i0 and columns at j0 of
// M, M = L, U (HERM = false) or their conjugate transposes: the stored block
// is (i0, j0), or (j0, i0) turned round.
template <typename T, int NR, bool HERM>
__global__ void __launch_bounds__(NT) k_trsv_block(BOp<T> LU, int n, BOp<T> X, int nrhs, int batch) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  T* xs = reinterpret_cast<T*>(smem_raw);            // [n32][NR]: the columns, row by row
  const int nblk = (n + 31) / 32;
  T* Ds = xs + (size_t)nblk * 32 * NR;               // diagonal block, stored column c at c * 33
  T* dv = Ds + 32 * 33;                              // reciprocals of its diagonal
  T* turn = dv + 32;                                 // HERM: one 32 x 33 block per warp
  const int b = blockIdx.x, c0 = blockIdx.y * NR;
  const int nc = min(NR, nrhs - c0);
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const T* A = LU.item(b);
  const int64_t ld = LU.ld;
  T* Xb = X.item(b) + (int64_t)c0 * X.ld;
  for (int e = threadIdx.x; e < nblk * 32 * NR; e += NT) {
    const int r = e % (nblk * 32), c = e / (nblk * 32);
    xs[r * NR + c] = (r < n && c < nc) ? Xb[r + (int64_t)c * X.ld] : T(0.0);
  }
#pragma unroll 1
  for (int tri = 0; tri < 2; ++tri) {
    // the first triangle runs forward (L, or U^H), the second backward (U, or L^H)
    const bool unit = HERM ? tri == 1 : tri == 0;
#pragma unroll 1
    for (int t = 0; t < nblk; ++t) {
      const int j = tri == 0 ? t : nblk - 1 - t, j0 = j * 32, pb = min(32, n - j0);
      for (int c = w; c < 32; c += NW)
        Ds[c * 33 + lane] = (lane < pb && c < pb) ? A[(j0 + lane) + (int64_t)(j0 + c) * ld] : T(0.0);
      __syncthreads();
      if (!unit && w == 0) {
        const T d = HERM ? conj_of(Ds[lane * 33 + lane]) : Ds[lane * 33 + lane];
        dv[lane] = is_zero(d) ? T(0.0) : recip(d);
      }
      if (!unit) __syncthreads();
      // substitution, one column per warp: lane = row, the solved entry is
      // broadcast and the rows after it updated
      for (int c = w; c < nc; c += NW) {
        T x = xs[(j0 + lane) * NR + c];
        for (int k = 0; k < pb; ++k) {
          const int q = tri == 0 ? k : pb - 1 - k;
          const T m = HERM ? conj_of(Ds[lane * 33 + q]) : Ds[q * 33 + lane];
          if (!unit && lane == q) x = x * dv[q];
          const T xq = shfl_v(x, q);
          if (tri == 0 ? lane > q : lane < q) x = fmsc(x, m, xq);
        }
        xs[(j0 + lane) * NR + c] = x;
      }
      __syncthreads();
      // the other blocks' rows: a block per warp
      const int first = tri == 0 ? j + 1 : 0, last = tri == 0 ? nblk : j;
      for (int i = first + w; i < last; i += NW) {
        const int i0 = i * 32;
        T acc[NR];
#pragma unroll
        for (int c = 0; c < NR; ++c) acc[c] = xs[(i0 + lane) * NR + c];
        if (HERM) {
          // stored block: rows j0 .., columns i0 ..
          T* tw = turn + w * 32 * 33;
          __syncwarp();
#pragma unroll 8
          for (int c = 0; c < 32; ++c)
            tw[c * 33 + lane] = (lane < pb && i0 + c < n) ? A[(j0 + lane) + (int64_t)(i0 + c) * ld] : T(0.0);
          __syncwarp();
        }
        const bool rv = i0 + lane < n;
#pragma unroll 1
        for (int q0 = 0; q0 < pb; q0 += 8) {
          T m[8];
#pragma unroll
          for (int q = 0; q < 8; ++q) {
            if (HERM) m[q] = conj_of(turn[(size_t)w * 32 * 33 + lane * 33 + q0 + q]);
            else m[q] = (rv && q0 + q < pb) ? A[(i0 + lane) + (int64_t)(j0 + q0 + q) * ld] : T(0.0);
          }
#pragma unroll
          for (int q = 0; q < 8; ++q)
#pragma unroll
            for (int c = 0; c < NR; ++c) acc[c] = fmsc(acc[c], m[q], xs[(j0 + q0 + q) * NR + c]);
        }
#pragma unroll
        for (int c = 0; c < NR; ++c) xs[(i0 + lane) * NR + c] = acc[c];
      }
      __syncthreads();
    }
  }
  for (int e = threadIdx.x; e < nblk * 32 * NR; e += NT) {
    const int r = e % (nblk * 32), c = e / (nblk * 32);
    if (r < n && c < nc) Xb[r + (int64_t)c * X.ld] = xs[r * NR + c];
  }
}

template <typename T>
size_t block_smem(int n, int nr, bool herm) {
  return ((size_t)((n + 31) / 32) * 32 * nr + 32 * 33 + 32 + (herm ? NW * 32 * 33 : 0)) * sizeof(T);
}

// ------------------------------------------------------------- few matrices

template <typename T, int NR, bool HERM, int MO>
__global__ void __launch_bounds__(NT) k_trsv_cluster(BOp<T> LU, int n, BOp<T> X, int nrhs, const T* dinv) {
  namespace cg = cooperative_groups;
  cg::cluster_group cl = cg::this_cluster();
  const int CS = (int)cl.num_blocks(), g = (int)cl.block_rank();
  const int b = blockIdx.x / CS, c0 = blockIdx.y * NR;
  const int nc = min(NR, nrhs - c0);
  const int nblk = (n + 31) / 32;
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  constexpr int QW = 32 / NW;                         // columns of a block per warp
  extern __shared__ __align__(16) unsigned char smem_raw[];
  T* xbuf = reinterpret_cast<T*>(smem_raw);           // [3][32][NR]: the solved blocks of the last steps
  T* xs = xbuf + 3 * 32 * NR;                         // [MO][32][NR]: right-hand sides / solutions of own blocks
  T* part = xs + MO * 32 * NR;                        // [2][NW][32][NR]
  T* turn = part + 2 * NW * 32 * NR;                  // HERM: [NW][32][QW + 1]
  const T* A = LU.item(b);
  const int64_t ld = LU.ld;
  T* Xb = X.item(b) + (int64_t)c0 * X.ld;
  const T* Db = dinv + (int64_t)b * 2 * nblk * 1024;
  const T* Fb = dinv + ((int64_t)(gridDim.x / CS) * 1024 + b) * 2 * nblk;   // which blocks want the correction
  // own blocks: g, g + CS, ...
  for (int e = threadIdx.x; e < MO * 32 * NR; e += NT) {
    const int r = e % 32, k = e / 32 % MO, c = e / (32 * MO);
    const int row = (g + k * CS) * 32 + r;
    xs[(k * 32 + r) * NR + c] = (row < n && c < nc) ? Xb[row + (int64_t)c * X.ld] : T(0.0);
  }
  // entries (lane, q), q = QW w .., of block (i, j) of the triangle's matrix;
  // HERM turns the stored block (j, i) round in the warp's shared memory
  auto tile = [&](const T* base, int64_t tld, int rows, int cols, T (&m)[QW]) {
    // base: the stored block; rows x cols of it exist
    if constexpr (!HERM) {
#pragma unroll
      for (int q = 0; q < QW; ++q)
        m[q] = (lane < rows && QW * w + q < cols) ? base[lane + (int64_t)(QW * w + q) * tld] : T(0.0);
    } else {
      T* tw = turn + w * 32 * (QW + 1);
      T v[QW];
#pragma unroll
      for (int k = 0; k < QW; ++k) {
        const int r = QW * w + (lane & (QW - 1)), c = k * (32 / QW) + lane / QW;
        v[k] = (r < rows && c < cols) ? conj_of(base[r + (int64_t)c * tld]) : T(0.0);
      }
      __syncwarp();
#pragma unroll
      for (int k = 0; k < QW; ++k) tw[(k * (32 / QW) + lane / QW) * (QW + 1) + (lane & (QW - 1))] = v[k];
      __syncwarp();
#pragma unroll
      for (int q = 0; q < QW; ++q) m[q] = tw[lane * (QW + 1) + q];
    }
  };
  auto load_block = [&](int i, int j, T (&m)[QW]) {
    if (!HERM) tile(A + (int64_t)i * 32 + (int64_t)j * 32 * ld, ld, n - i * 32, n - j * 32, m);
    else tile(A + (int64_t)j * 32 + (int64_t)i * 32 * ld, ld, n - j * 32, n - i * 32, m);
  };
  // block j of the first or second triangle itself
  auto load_triangle = [&](int tri, int j, T (&m)[QW]) {
    load_block(j, j, m);
    const bool unit = (tri == 0) != HERM;
#pragma unroll
    for (int q = 0; q < QW; ++q) {
      const int c = QW * w + q;
      if (tri == 0 ? lane < c : lane > c) m[q] = T(0.0);
      else if (lane == c && unit) m[q] = T(1.0);
    }
  };
  // its inverse; returns whether a product with that wants the correction
  auto load_inverse = [&](int tri, int j, T (&m)[QW]) {
    const int at = (HERM ? 1 - tri : tri) * nblk + j;
    tile(Db + (int64_t)at * 1024, 32, 32, 32, m);
    return !is_zero(Fb[at]);
  };
  T acc[MO][NR];   // contributions of the solved blocks to own block k (this warp's columns)
  auto clear = [&]() {
#pragma unroll
    for (int k = 0; k < MO; ++k)
#pragma unroll
      for (int c = 0; c < NR; ++c) acc[k][c] = T(0.0);
  };
  // the sum over the warps of their v, in one of two buffers in turn
  auto total = [&](T (&v)[NR], T* p) {
#pragma unroll
    for (int c = 0; c < NR; ++c) p[(w * 32 + lane) * NR + c] = v[c];
    __syncthreads();
#pragma unroll
    for (int c = 0; c < NR; ++c)
      v[c] = (p[lane * NR + c] + p[(32 + lane) * NR + c]) + (p[(64 + lane) * NR + c] + p[(96 + lane) * NR + c]);
  };
  // v <- M b, this warp's columns of M in m
  auto product = [&](const T (&m)[QW], const T (&b)[NR], T (&v)[NR], T* p) {
#pragma unroll
    for (int c = 0; c < NR; ++c) v[c] = T(0.0);
#pragma unroll
    for (int q = 0; q < QW; ++q)
#pragma unroll
      for (int c = 0; c < NR; ++c) v[c] = fmac(v[c], m[q], shfl_v(b[c], QW * w + q));
    total(v, p);
  };
  // block j's solution from its right-hand side and contributions, to every CTA's
  // slot; dm: the inverse of its diagonal block
  auto solve = [&](const T (&dm)[QW], bool correct, int tri, int j, int slot) {
    const int kj = j / CS;
    T* part2 = part + NW * 32 * NR;
    T y[NR], x[NR], v[NR];
#pragma unroll
    for (int k = 0; k < MO; ++k)
      if (k == kj) {
#pragma unroll
        for (int c = 0; c < NR; ++c) v[c] = acc[k][c];
      }
    total(v, part);
#pragma unroll
    for (int c = 0; c < NR; ++c) y[c] = xs[(kj * 32 + lane) * NR + c] + v[c];
    product(dm, y, x, part2);
    if (correct) {   // uniform over the CTA
      T tm[QW];
      load_triangle(tri, j, tm);
      product(tm, x, v, part);
#pragma unroll
      for (int c = 0; c < NR; ++c) y[c] = y[c] - v[c];
      product(dm, y, v, part2);
#pragma unroll
      for (int c = 0; c < NR; ++c) x[c] = x[c] + v[c];
    }
    for (int d = w; d < CS; d += NW) {
      T* dst = cl.map_shared_rank(xbuf, d) + (slot * 32 + lane) * NR;
#pragma unroll
      for (int c = 0; c < NR; ++c) dst[c] = x[c];
    }
    if (w == 0) {
#pragma unroll
      for (int c = 0; c < NR; ++c) xs[(kj * 32 + lane) * NR + c] = x[c];
    }
  };
  auto update = [&](const T (&m)[QW], int k, int slot) {
    const T* xq = xbuf + (slot * 32 + QW * w) * NR;
    T xv[QW][NR];
#pragma unroll
    for (int q = 0; q < QW; ++q)
#pragma unroll
      for (int c = 0; c < NR; ++c) xv[q][c] = xq[q * NR + c];
#pragma unroll
    for (int kk = 0; kk < MO; ++kk)
      if (kk == k) {
#pragma unroll
        for (int q = 0; q < QW; ++q)
#pragma unroll
          for (int c = 0; c < NR; ++c) acc[kk][c] = fmsc(acc[kk][c], m[q], xv[q][c]);
      }
  };
  auto block_at = [&](int tri, int t) { return tri == 0 ? t : nblk - 1 - t; };
  cl.sync();   // every CTA has started before any writes into its shared memory
  clear();
  if (g == 0) {
    T dm[QW];
    const bool correct = load_inverse(0, 0, dm);
    solve(dm, correct, 0, 0, 0);
  }
  cluster_arrive();
  // Step s: block block_at(tri, t) has been solved; its barrier tells every
  // CTA.  The owner of the next block updates and solves that one (its matrix
  // entries loaded ahead) before it arrives at the next barrier, the others
  // arrive at once, and everyone's remaining updates run behind it.  A slot is
  // written again three steps later, after a barrier that every CTA reaches
  // once it has finished these updates.
  int slot = 0;
#pragma unroll 1
  for (int s = 0; s < 2 * nblk; ++s) {
    const int tri = s >= nblk, t = tri ? s - nblk : s, j = block_at(tri, t);
    const int slot1 = slot == 2 ? 0 : slot + 1;
    const bool turn_round = t == nblk - 1;   // the next step starts the second triangle
    const int tri1 = turn_round ? 1 : tri, j1 = turn_round ? nblk - 1 : block_at(tri, t + 1);
    const bool mine = s + 1 < 2 * nblk && j1 % CS == g;
    T m1[QW], dm[QW];
    bool correct = false;
    if (mine) {
      if (!turn_round) load_block(j1, j, m1);
      correct = load_inverse(tri1, j1, dm);
    }
    cluster_wait();
    if (turn_round) clear();
    if (mine) {
      if (!turn_round) update(m1, j1 / CS, slot);
      solve(dm, correct, tri1, j1, slot1);
    }
    if (s + 1 < 2 * nblk) cluster_arrive();
    if (!turn_round) {
      // two blocks' entries in flight
#pragma unroll
      for (int k = 0; k < MO; k += 2) {
        const int i0 = g + k * CS, i1 = i0 + CS;
        auto want = [&](int i) { return i < nblk && (tri == 0 ? i > j : i < j) && i != j1; };
        const bool w0 = want(i0), w1 = want(i1);
        T ma[QW], mb[QW];
        if (w0) load_block(i0, j, ma);
        if (w1) load_block(i1, j, mb);
        if (w0) update(ma, k, slot);
        if (w1) update(mb, k + 1, slot);
      }
    }
    slot = slot1;
  }
  __syncthreads();
  for (int e = threadIdx.x; e < MO * 32 * NR; e += NT) {
    const int r = e % 32, k = e / 32 % MO, c = e / (32 * MO);
    const int row = (g + k * CS) * 32 + r;
    if (row < n && c < nc) Xb[row + (int64_t)c * X.ld] = xs[(k * 32 + r) * NR + c];
  }
  cl.sync();   // no CTA leaves while another may still write into it
}

template <typename T>
size_t cluster_smem(int nr, int mo) {
  return ((size_t)3 * 32 * nr + (size_t)mo * 32 * nr + 2 * NW * 32 * nr + NW * 32 * (32 / NW + 1)) * sizeof(T);
}

// Inverses of the 32 x 32 diagonal blocks of each factor of a batch
// (column-major, 32 x 32 each, [item][triangle][block]): triangle 0 the unit
// lower L_jj, 1 the upper U_jj; a partial last block is completed with the
// identity, a zero pivot gives a zero row (a singular factor was reported by
// the factorisation).  One CTA per block and triangle: four threads per
// column of the identity, 8 rows each, the row groups solved in order and
// broadcast by shuffles.
//
// Behind them a flag per block: whether a product with the inverse wants a
// correction.  The product's residual is up to || |T| |T^-1| || (for the conjugate
// transpose, the one-norm of |T^-1| |T|) times a substitution's.  Residuals for
// random right-hand sides, rms in units of 1e-17 of |T| |x| + |y|, substitution /
// product, by that norm: 8 to 16 5.5 / 6.9, 16 to 32 4.5 / 6.6, 32 to 64 4.5 / 6.9, 64 to
// 96 4.2 / 7.0 (the blocks of all merges of the elliptic and Helmholtz operators), 512
// to 4096 6.9 / 217, above 4.0 / 46 (dense impedance leaves).  Solutions of the former
// have the same errors with and without the correction; the line lies between.
constexpr float CORRECT_FROM = 256.0f;
__device__ __forceinline__ float magf(double v) { return fabsf((float)v); }
__device__ __forceinline__ float magf(cplx v) { return fabsf((float)v.re) + fabsf((float)v.im); }
template <typename T>
__global__ void __launch_bounds__(128) k_block_inverses(BOp<T> LU, int n, T* out) {
  __shared__ T Ls[32 * 32];
  __shared__ T dv[32];
  __shared__ float mv[32 * 33], rsum[32], csum[32];   // magnitudes of the inverse, their row and column sums
  const int j = blockIdx.x, nblk = gridDim.x, b = blockIdx.z;
  const bool upper = blockIdx.y == 1;
  const int pb = min(32, n - j * 32);
  const T* A = LU.item(b) + (int64_t)j * 32 * (LU.ld + 1);
  for (int e = threadIdx.x; e < 1024; e += 128) {
    const int r = e & 31, c = e >> 5;
    Ls[e] = r < pb && c < pb ? A[r + (int64_t)c * LU.ld] : r == c ? T(1.0) : T(0.0);
  }
  __syncthreads();
  if (upper && threadIdx.x < 32) {
    const T d = Ls[threadIdx.x * 33];
    dv[threadIdx.x] = is_zero(d) ? T(0.0) : recip(d);
  }
  __syncthreads();
  const int col = threadIdx.x >> 2, g = threadIdx.x & 3, lane0 = (threadIdx.x & 31) & ~3;
  T x[8];
#pragma unroll
  for (int i = 0; i < 8; ++i) x[i] = 8 * g + i == col ? T(1.0) : T(0.0);
#pragma unroll
  for (int step = 0; step < 4; ++step) {
    const int blk = upper ? 3 - step : step;
    if (g == blk) {
      if (!upper) {
#pragma unroll
        for (int i = 1; i < 8; ++i)
#pragma unroll
          for (int q = 0; q < i; ++q) x[i] = fmsc(x[i], Ls[(8 * g + i) + (8 * g + q) * 32], x[q]);
      } else {
#pragma unroll
        for (int i = 7; i >= 0; --i) {
          T s = x[i];
#pragma unroll
          for (int q = i + 1; q < 8; ++q) s = fmsc(s, Ls[(8 * g + i) + (8 * g + q) * 32], x[q]);
          x[i] = s * dv[8 * g + i];
        }
      }
    }
    T xb[8];
#pragma unroll
    for (int q = 0; q < 8; ++q) xb[q] = shfl_v(x[q], lane0 | blk);
    if (upper ? g < blk : g > blk) {
#pragma unroll
      for (int i = 0; i < 8; ++i)
#pragma unroll
        for (int q = 0; q < 8; ++q) x[i] = fmsc(x[i], Ls[(8 * g + i) + (8 * blk + q) * 32], xb[q]);
    }
  }
  const int64_t at = ((int64_t)b * 2 + blockIdx.y) * nblk + j;
  T* o = out + at * 1024 + 32 * col + 8 * g;
  // |T| (|V| 1) and (1 |V|) |T|, four threads per row or column; in single
  // precision, off the FP64 pipe: what overflows or is no number is marked
  auto quad = [](float v) {
    v += __shfl_xor_sync(0xffffffffu, v, 1);
    return v + __shfl_xor_sync(0xffffffffu, v, 2);
  };
  float sum = 0.0f;
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    o[i] = x[i];
    const float m = magf(x[i]);
    mv[(8 * g + i) * 33 + col] = m;
    sum += m;
  }
  csum[col] = quad(sum);
  __syncthreads();
  const int r = col, k0 = 8 * g;   // this thread's row or column of T, and the entries it takes
  sum = 0.0f;
#pragma unroll
  for (int k = 0; k < 8; ++k) sum += mv[r * 33 + k0 + k];
  rsum[r] = quad(sum);
  __syncthreads();
  float rn = 0.0f, cn = 0.0f;
#pragma unroll
  for (int k = k0; k < k0 + 8; ++k) {
    const float tr = upper ? (k >= r ? magf(Ls[r + k * 32]) : 0.0f) : k < r ? magf(Ls[r + k * 32]) : k == r ? 1.0f : 0.0f;
    const float tc = upper ? (k <= r ? magf(Ls[k + r * 32]) : 0.0f) : k > r ? magf(Ls[k + r * 32]) : k == r ? 1.0f : 0.0f;
    rn = fmaf(tr, rsum[k], rn);
    cn = fmaf(tc, csum[k], cn);
  }
  rn = quad(rn);
  cn = quad(cn);
  const int wants = __syncthreads_or(!(rn <= CORRECT_FROM) || !(cn <= CORRECT_FROM));
  if (threadIdx.x == 0) out[(int64_t)gridDim.z * 2 * nblk * 1024 + at] = T(wants ? 1.0 : 0.0);
}

// Cluster shape: a power of two of CTAs, at most 16, the SMs' share of a
// matrix or its blocks.
int cluster_of(int n, int batch) {
  const int nblk = (n + 31) / 32;
  int cs = 1;
  while (cs < 16 && (int64_t)batch * cs * 2 <= device_sms() && cs < nblk) cs *= 2;
  return cs;
}
int own_blocks(int n, int cs) { return ((n + 31) / 32 + cs - 1) / cs; }

template <typename T, int NR, bool HERM, int MO>
cudaError_t launch_cluster(BOp<T> LU, int n, BOp<T> X, int nrhs, int batch, int cs, const T* dinv, cudaStream_t st) {
  static const cudaError_t attr = [] {
    cudaError_t e = cudaFuncSetAttribute(k_trsv_cluster<T, NR, HERM, MO>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         (int)cluster_smem<T>(NR, MO));
    if (e == cudaSuccess)
      e = cudaFuncSetAttribute(k_trsv_cluster<T, NR, HERM, MO>, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
    return e;
  }();
  if (attr != cudaSuccess) return attr;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(batch * cs, (nrhs + NR - 1) / NR);
  cfg.blockDim = dim3(NT);
  cfg.dynamicSmemBytes = cluster_smem<T>(NR, MO);
  cfg.stream = st;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = cs;
  at[0].val.clusterDim.y = 1;
  at[0].val.clusterDim.z = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, k_trsv_cluster<T, NR, HERM, MO>, LU, n, X, nrhs, dinv);
}

template <typename T, int NR, bool HERM>
cudaError_t dispatch_cluster(BOp<T> LU, int n, BOp<T> X, int nrhs, int batch, const T* dinv, cudaStream_t st) {
  const int cs = cluster_of(n, batch), mo = own_blocks(n, cs);
  // the partial sums of all own blocks stay in registers: at most 64 of them,
  // more columns go to further clusters
  constexpr int N8 = NR < 4 ? NR : 4;
  if (mo <= 2) return launch_cluster<T, NR, HERM, 2>(LU, n, X, nrhs, batch, cs, dinv, st);
  if (mo <= 4) return launch_cluster<T, NR, HERM, 4>(LU, n, X, nrhs, batch, cs, dinv, st);
  return launch_cluster<T, N8, HERM, 8>(LU, n, X, nrhs, batch, cs, dinv, st);
}

// Columns that a cluster takes at a time.  A column of its own: a step's chain is
// mostly the multiply-adds of its own CTA, and clusters beside one another fill
// the SMs (us, one / two / four / eight columns a cluster: eight complex columns of one
// matrix of 512 217 / 244 / 472 / 1024, of 16 of 448 375 / 514 / 547 / 993; eight real
// columns of eight of 1728 726 / 982 / 1385 / 1441).  Real columns of many matrices,
// whose short clusters fill the SMs alone, share the matrix's entries (64 of 432, four
// columns 291 / 217 / 255 / 254, eight 457 / 434 / 330 / 326).
template <typename T>
int cluster_cols(int nrhs, int batch) {
  return sizeof(T) == 16 || batch <= 16 || nrhs < 4 ? 1 : few_cols(nrhs);
}

template <typename T, int NR, bool HERM>
cudaError_t launch_block(BOp<T> LU, int n, BOp<T> X, int nrhs, int batch, cudaStream_t st) {
  static const cudaError_t attr = cudaFuncSetAttribute(
      k_trsv_block<T, NR, HERM>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)BLOCK_SMEM);
  if (attr != cudaSuccess) return attr;
  k_trsv_block<T, NR, HERM><<<dim3(batch, (nrhs + NR - 1) / NR), NT, block_smem<T>(n, NR, HERM), st>>>(LU, n, X, nrhs, batch);
  return cudaGetLastError();
}

template <typename T, bool HERM>
cudaError_t solve_few(BOp<T> LU, int n, BOp<T> X, int nrhs, int batch, const T* dinv, cudaStream_t st) {
  if (!dinv) {
    switch (few_cols(nrhs)) {
      case 1: return launch_block<T, 1, HERM>(LU, n, X, nrhs, batch, st);
      case 2: return launch_block<T, 2, HERM>(LU, n, X, nrhs, batch, st);
      case 4: return launch_block<T, 4, HERM>(LU, n, X, nrhs, batch, st);
      default: return launch_block<T, 8, HERM>(LU, n, X, nrhs, batch, st);
    }
  }
  const int nc = cluster_cols<T>(nrhs, batch);
  if constexpr (sizeof(T) == sizeof(double)) {
    if (nc == 4) return dispatch_cluster<T, 4, HERM>(LU, n, X, nrhs, batch, dinv, st);
    if (nc == 8) return dispatch_cluster<T, 8, HERM>(LU, n, X, nrhs, batch, dinv, st);
  }
  return dispatch_cluster<T, 1, HERM>(LU, n, X, nrhs, batch, dinv, st);
}

}  // namespace

// Batches whose solves with few right-hand sides take a cluster per matrix:
// too few to give every SM a CTA, more than one block, and at most 8 blocks
// per CTA of the largest cluster.
bool trsv_cluster_wanted(int n, int64_t batch) {
  return n > 32 && batch * 2 <= device_sms() && own_blocks(n, cluster_of(n, (int)batch)) <= 8;
}

// A single factor of more than four blocks per CTA of the largest cluster
// (n > 2048): the flag-ordered solve over all SMs is faster (2808 rows, one
// column: 584 us against 711; 1792 complex rows: 576 against 561).
bool trsv_flags_preferred(int n) { return own_blocks(n, cluster_of(n, 1)) > 4; }


template <typename T>
bool trsv_few_applicable(int n, int nrhs, int batch, const TrsvInv* inv) {
  if (nrhs < 1 || nrhs > 2 * MAXN || n < 1) return false;
  if (inv && inv->p) return true;
  // one CTA per matrix: enough of them to fill the SMs, or small ones
  return (n <= 64 || batch * 2 > device_sms()) && block_smem<T>(n, few_cols(nrhs), true) <= BLOCK_SMEM;
}

template <typename T>
cudaError_t trsv_few(BOp<T> LU, int n, BOp<T> X, int nrhs, int batch, bool herm, TrsvInv* inv, cudaStream_t st, Prof* pf) {
  cudaError_t e;
  const T* dv = nullptr;
  if (inv && inv->p) {
    if (!inv->ready) {
      if (pf) pf->begin(st);
      k_block_inverses<T><<<dim3((n + 31) / 32, 2, batch), 128, 0, st>>>(LU, n, static_cast<T*>(inv->p));
      if ((e = cudaGetLastError()) != cudaSuccess) return e;
      if (pf) pf->end(K_OTHER, 0.0, st);
      inv->ready = !stream_capturing(st);   // a captured launch has formed nothing yet
    }
    dv = static_cast<const T*>(inv->p);
  }
  if (pf) {
    pf->begin(st);
    pf->note(n, nrhs, 32, batch);
  }
  e = herm ? solve_few<T, true>(LU, n, X, nrhs, batch, dv, st) : solve_few<T, false>(LU, n, X, nrhs, batch, dv, st);
  if (e != cudaSuccess) return e;
  constexpr double F = sizeof(T) == 16 ? 8.0 : 2.0;
  if (pf) pf->end(K_TRSM_DIAG, F * (double)n * n * nrhs * batch, st);
  return cudaSuccess;
}

#define HPS_TRSV_INST(T)                                                        \
  template bool trsv_few_applicable<T>(int, int, int, const TrsvInv*);          \
  template cudaError_t trsv_few<T>(BOp<T>, int, BOp<T>, int, int, bool, TrsvInv*, cudaStream_t, Prof*);
HPS_TRSV_INST(double)
HPS_TRSV_INST(cplx)

}  // namespace hps

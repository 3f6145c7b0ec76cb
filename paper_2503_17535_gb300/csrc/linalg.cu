// Batched FP64 / complex128 dense kernels: gathered GEMM, panel LU with
// partial pivoting (one CTA per matrix, a thread-block cluster per matrix,
// or a cooperative group of CTAs per matrix), row interchanges + triangular
// update, recursive LU and triangular solves, and flag-ordered solves of a
// single large factor.
//
// GB300 has about 1 TFLOP/s of FP64 (2 DFMA per clock per SM), so every
// kernel here is bound by the FP64 pipe long before HBM or shared memory:
// the designs aim at keeping all 152 SMs issuing FMAs (enough CTAs per level,
// clusters or cooperative groups for single large matrices), at spending no
// FP64 instruction that is not part of the algorithm, and at keeping FP64
// latency chains (a reciprocal, a serial load) off the per-column critical
// path of the panels.
#include "linalg.h"
#include "tri_cols.h"

#include <mutex>

#include <cooperative_groups.h>

#include <algorithm>
#include <cstdio>

namespace hps {

void Prof::begin(cudaStream_t st) {
  if (!on) return;
  cudaEventCreate(&pending);
  cudaEventRecord(pending, st);
}

void Prof::end(int cls, double fl, cudaStream_t st, double executed) {
  ++launches;
  ++n[cls];
  flops[cls] += fl;
  exec[cls] += executed < 0.0 ? fl : executed;
  if (!on || !pending) {
    dims[0] = dims[1] = dims[2] = dims[3] = 0;
    return;
  }
  cudaEvent_t e1;
  cudaEventCreate(&e1);
  cudaEventRecord(e1, st);
  trace.push_back(Rec{cls, dims[0], dims[1], dims[2], dims[3], fl, (int64_t)ev[cls].size()});
  dims[0] = dims[1] = dims[2] = dims[3] = 0;
  ev[cls].push_back(pending);
  ev[cls].push_back(e1);
  pending = nullptr;
}

double Prof::rec_ms(const Rec& r) const {
  float m = 0.f;
  if (r.ev + 1 < (int64_t)ev[r.cls].size() &&
      cudaEventElapsedTime(&m, ev[r.cls][r.ev], ev[r.cls][r.ev + 1]) == cudaSuccess)
    return m;
  return -1.0;
}

void Prof::reset() {
  for (int c = 0; c < K_COUNT; ++c) {
    for (cudaEvent_t e : ev[c]) cudaEventDestroy(e);
    ev[c].clear();
    n[c] = 0;
    flops[c] = 0.0;
    exec[c] = 0.0;
  }
  if (pending) cudaEventDestroy(pending);
  pending = nullptr;
  launches = 0;
  trace.clear();
}

double Prof::ms(int cls) const {
  double t = 0.0;
  for (size_t i = 0; i + 1 < ev[cls].size(); i += 2) {
    float m = 0.f;
    if (cudaEventElapsedTime(&m, ev[cls][i], ev[cls][i + 1]) == cudaSuccess) t += m;
  }
  return t;
}

template <typename T> constexpr double fma_flops() { return 2.0; }
template <> constexpr double fma_flops<cplx>() { return 8.0; }

// ---------------------------------------------------------------- GEMM ----

// Epilogue modes: the LU / TRSM / Schur updates are C <- C - A B and the
// leaf products C <- A B; handling those two forms apart keeps the general
// alpha / beta arithmetic (a complex multiply and multiply-add per element)
// off the FP64 pipe, where it costs as much as several steps of K.
enum { EPI_GENERAL = 0, EPI_SUB = 1, EPI_SET = 2 };

template <typename T>
inline int epi_mode(const GemmArgs<T>& g) {
  if (g.alpha == T(-1.0) && g.beta == T(1.0)) return EPI_SUB;
  if (g.alpha == T(1.0) && is_zero(g.beta)) return EPI_SET;
  return EPI_GENERAL;
}

// Products on the FP64 pipe, N > 8: BM x 256 / BM tiles (BM = 32, 16 or 8 rows,
// whichever pads the shape least), four warps, a thread per row and
// pair of columns, 32 steps of K (complex: 16) staged at once with the next in
// flight in registers.
//
// The pipe does two multiply-adds per clock and SM, so that even these small
// tiles need only 2.5 of the 30 bytes per clock that L2 delivers to an SM; what
// counts is that the tiles spread over all SMs, that K is not padded (to a
// multiple of four only) and that the pipe never waits for a load.
// us (64 x 64 or 32 x 32 tiles with 16 steps of K, the loads waited for, before -> now): 32 x
// 864 x 32 14.4 -> 6.3, 64 x 864 x 64 75 -> 12.4, 128 x 128 x 128 145 -> 14.4, 1024 x 1024 x
// 64 135 -> 115 (pipe: 112); batches of 4096 64 x 114 x 4 874 -> 277.
//
// Complex products take the 3M method: with A = Ar + i Ai and B = Br + i Bi,
// the real products P1 = Ar Br, P2 = Ai Bi and P3 = (Ar + Ai)(Br + Bi) give
// C = (P1 - P2) + i (P3 - P1 - P2).  Each complex multiply-add costs three
// real FMAs instead of four on the FP64 pipe; the sums Ar + Ai and Br + Bi
// are formed once per element when the tile is staged in shared memory.  The
// three planes of 32 steps would leave room for seven CTAs per SM and load past
// short K: 4096 items of 28 x 28 x 16 and 64 x 114 x 4 take 584 and 1288 us (whole
// call) with 32 steps, 550 and 1132 with 16, longer K the same.
// With MODE == EPI_SUB the accumulators start from C so that the update
// needs three additions per element: p1 = 0, p2 = Re C, p3 = Re C - Im C give
// Re(C - AB) = p2 - p1 and Im(C - AB) = p1 + p2 - p3 after the products.
template <typename T> struct GemmPlanes { enum { N = 1 }; };
template <> struct GemmPlanes<cplx> { enum { N = 3 }; };

__device__ __forceinline__ double gemm_plane(double v, int) { return v; }
__device__ __forceinline__ double gemm_plane(cplx v, int p) { return p == 0 ? v.re : p == 1 ? v.im : v.re + v.im; }

template <typename T, int MODE, int BM>
__global__ void __launch_bounds__(128) k_gemm(GemmArgs<T> g) {
  constexpr int P = GemmPlanes<T>::N, BN = 256 / BM, BK = P == 1 ? 32 : 16, LA = BM * BK / 128, LB = BN * BK / 128;
  __shared__ double As[P][BK][BM];
  __shared__ __align__(16) double Bs[P][BK][BN + 2];   // + 2: the staging writes go down a column
  const int tid = threadIdx.x;
  const int r = tid % BM, c0 = 2 * (tid / BM);   // this thread's row and columns c0, c0 + 1 of the tile
  const int ra = tid % BM, la = tid / BM;        // what it stages of A: row ra, steps la, la + 128 / BM, ...
  const int lb = tid % BK, cb = tid / BK;        // and of B: step lb, columns cb, cb + 128 / BK, ...
  const int tiles_m = (g.M + BM - 1) / BM;
  const int i = blockIdx.x % tiles_m * BM + r, j0 = blockIdx.x / tiles_m * BN;
  const bool beta = MODE == EPI_SUB || (MODE == EPI_GENERAL && !is_zero(g.beta));
  for (int b = blockIdx.y; b < g.batch; b += gridDim.y) {
    const T* A = g.A.item(b);
    const T* B = g.B.item(b);
    T* C = g.C.item(b);
    const bool row = i < g.M;
    const int64_t ai = row ? g.arow.at(b, i) : 0, ci = row ? g.crow.at(b, i) : 0;
    T a[LA], bb[LB], cv[2];
    double acc[P][2];
    auto load = [&](int k0) {
#pragma unroll
      for (int u = 0; u < LA; ++u) {
        const int l = k0 + la + 128 / BM * u;
        a[u] = row && l < g.K ? A[ai + (int64_t)g.acol.at(b, l) * g.A.ld] : T(0.0);
      }
      const int l = k0 + lb;
      const int64_t bi = l < g.K ? g.brow.at(b, l) : 0;
#pragma unroll
      for (int u = 0; u < LB; ++u) {
        const int j = j0 + cb + 128 / BK * u;
        bb[u] = l < g.K && j < g.N ? B[bi + (int64_t)j * g.B.ld] : T(0.0);
      }
    };
    load(0);
#pragma unroll
    for (int c = 0; c < 2; ++c) {
      cv[c] = beta && row && j0 + c0 + c < g.N ? C[ci + (int64_t)(j0 + c0 + c) * g.C.ld] : T(0.0);
#pragma unroll
      for (int p = 0; p < P; ++p) acc[p][c] = 0.0;
      if (MODE == EPI_SUB) {
        if constexpr (P == 1) {
          acc[0][c] = cv[c];
        } else {
          acc[1][c] = cv[c].re;
          acc[2][c] = cv[c].re - cv[c].im;
        }
      }
    }
    for (int k0 = 0; k0 < g.K; k0 += BK) {
      const int kc = min(BK, (g.K - k0 + 3) & ~3);   // steps beyond K are zero
      __syncthreads();
#pragma unroll
      for (int p = 0; p < P; ++p) {
#pragma unroll
        for (int u = 0; u < LA; ++u)
          if (la + 128 / BM * u < kc) As[p][la + 128 / BM * u][ra] = gemm_plane(a[u], p);
#pragma unroll
        for (int u = 0; u < LB; ++u) Bs[p][lb][cb + 128 / BK * u] = gemm_plane(bb[u], p);
      }
      __syncthreads();
      if (k0 + BK < g.K) load(k0 + BK);
#pragma unroll 2
      for (int k = 0; k < kc; k += 4) {
        double av[P][4];
        double2 bv[P][4];
#pragma unroll
        for (int p = 0; p < P; ++p)
#pragma unroll
          for (int u = 0; u < 4; ++u) {
            av[p][u] = As[p][k + u][r];
            bv[p][u] = *reinterpret_cast<const double2*>(&Bs[p][k + u][c0]);
          }
#pragma unroll
        for (int u = 0; u < 4; ++u)
#pragma unroll
          for (int p = 0; p < P; ++p) {
            const double s = P == 1 && MODE == EPI_SUB ? -av[p][u] : av[p][u];
            acc[p][0] = fma(s, bv[p][u].x, acc[p][0]);
            acc[p][1] = fma(s, bv[p][u].y, acc[p][1]);
          }
      }
    }
    __syncthreads();
    if (!row) continue;
#pragma unroll
    for (int c = 0; c < 2; ++c) {
      if (j0 + c0 + c >= g.N) continue;
      T v;
      if constexpr (P == 1) {
        v = acc[0][c];
      } else if (MODE == EPI_SUB) {
        v = cplx(acc[1][c] - acc[0][c], (acc[0][c] + acc[1][c]) - acc[2][c]);
      } else if (MODE == EPI_SET) {
        v = cplx(acc[0][c] - acc[1][c], acc[2][c] - (acc[0][c] + acc[1][c]));
      } else {
        v = cplx(acc[0][c] - acc[1][c], acc[2][c] - acc[0][c] - acc[1][c]);
      }
      if (MODE == EPI_GENERAL) {
        v = g.alpha * v;
        if (beta) v = fmac(v, g.beta, cv[c]);
      }
      C[ci + (int64_t)(j0 + c0 + c) * g.C.ld] = v;
    }
  }
}

// Skinny variant for N <= 8 right-hand sides (the solve path): one thread
// per output row, B chunks staged in shared memory, A read column by column
// (coalesced along the rows).  NC is the column count rounded up to 1, 2, 4
// or 8: the FP64 pipe spends its cycles on predicated-off FMAs too, so the
// kernel never carries more columns than it needs.
template <typename T, int NC>
__global__ void __launch_bounds__(128) k_gemm_skinny(GemmArgs<T> g) {
  constexpr int KC = 32;
  __shared__ T Bs[KC][NC];
  const int tid = threadIdx.x;
  for (int b = blockIdx.z; b < g.batch; b += gridDim.z) {
    const T* A = g.A.item(b);
    const T* B = g.B.item(b);
    T* C = g.C.item(b);
    const int i = blockIdx.x * 128 + tid;
    const bool act = i < g.M;
    const int64_t ar = act ? g.arow.at(b, i) : 0;
    T acc[NC];
#pragma unroll
    for (int c = 0; c < NC; ++c) acc[c] = T(0.0);
    for (int k0 = 0; k0 < g.K; k0 += KC) {
      const int kc = min(KC, g.K - k0);
      __syncthreads();
      for (int e = tid; e < KC * NC; e += 128) {
        const int l = e % KC, c = e / KC;
        Bs[l][c] = (l < kc && c < g.N) ? B[(int64_t)g.brow.at(b, k0 + l) + (int64_t)c * g.B.ld] : T(0.0);
      }
      __syncthreads();
      if (act) {
        if (kc == KC) {
          // full chunk: unrolled so that several column loads are in flight
#pragma unroll 8
          for (int l = 0; l < KC; ++l) {
            const T a = A[ar + (int64_t)g.acol.at(b, k0 + l) * g.A.ld];
#pragma unroll
            for (int c = 0; c < NC; ++c) acc[c] = fmac(acc[c], a, Bs[l][c]);
          }
        } else {
          for (int l = 0; l < kc; ++l) {
            const T a = A[ar + (int64_t)g.acol.at(b, k0 + l) * g.A.ld];
#pragma unroll
            for (int c = 0; c < NC; ++c) acc[c] = fmac(acc[c], a, Bs[l][c]);
          }
        }
      }
    }
    if (act) {
      const int64_t ci = g.crow.at(b, i);
      const bool use_beta = !is_zero(g.beta);
#pragma unroll
      for (int c = 0; c < NC; ++c) {
        if (c >= g.N) break;
        T* p = C + ci + (int64_t)c * g.C.ld;
        T v = g.alpha * acc[c];
        if (use_beta) v = fmac(v, g.beta, *p);
        *p = v;
      }
    }
  }
}

// Skinny product with few rows in the whole launch (the top levels of the
// solve): 32 rows x 8 groups of the inner dimension per CTA, the 8 partial
// sums added in shared memory in a fixed order.
template <typename T, int NC>
__global__ void __launch_bounds__(256) k_gemm_skinny_kg(GemmArgs<T> g) {
  __shared__ T part[8][NC][32];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  for (int b = blockIdx.z; b < g.batch; b += gridDim.z) {
    const T* A = g.A.item(b);
    const T* B = g.B.item(b);
    T* C = g.C.item(b);
    const int i = blockIdx.x * 32 + lane;
    const bool act = i < g.M;
    const int64_t ar = act ? g.arow.at(b, i) : 0;
    T acc[NC];
#pragma unroll
    for (int c = 0; c < NC; ++c) acc[c] = T(0.0);
    if (act) {
      // U entries of A and U NC of B (and their gathered indices) in flight: more
      // than 16 doubles of B cost warps (64 items of 300 x 300 with five columns, whole
      // call: 8 / 4 / 2 entries real 331 / 289 / 286 us, complex 760 / 646 / 579)
      constexpr int U0 = 16 / (NC * (int)(sizeof(T) / sizeof(double))), U = U0 > 8 ? 8 : U0 < 2 ? 2 : U0;
      const int* ac = g.acol.idx ? g.acol.idx + (b % g.acol.period) * g.acol.len : nullptr;
      const int* bi = g.brow.idx ? g.brow.idx + (b % g.brow.period) * g.brow.len : nullptr;
      for (int l0 = w; l0 < g.K; l0 += 8 * U) {
        T a[U], x[U][NC];
#pragma unroll
        for (int k = 0; k < U; ++k) {
          const int l = l0 + 8 * k;
          const bool in = l < g.K;
          a[k] = in ? A[ar + (int64_t)(ac ? ac[l] : l) * g.A.ld] : T(0.0);
          const int64_t br = in ? (bi ? bi[l] : l) : 0;
#pragma unroll
          for (int c = 0; c < NC; ++c) x[k][c] = in && c < g.N ? B[br + (int64_t)c * g.B.ld] : T(0.0);
        }
#pragma unroll
        for (int k = 0; k < U; ++k)
#pragma unroll
          for (int c = 0; c < NC; ++c) acc[c] = fmac(acc[c], a[k], x[k][c]);
      }
    }
#pragma unroll
    for (int c = 0; c < NC; ++c) part[w][c][lane] = acc[c];
    __syncthreads();
    if (w == 0 && act) {
      const int64_t ci = g.crow.at(b, i);
      const bool use_beta = !is_zero(g.beta);
#pragma unroll
      for (int c = 0; c < NC; ++c) {
        if (c >= g.N) break;
        T v = part[0][c][lane];
        for (int k = 1; k < 8; ++k) v = v + part[k][c][lane];
        T* p = C + ci + (int64_t)c * g.C.ld;
        v = g.alpha * v;
        if (use_beta) v = fmac(v, g.beta, *p);
        *p = v;
      }
    }
    __syncthreads();
  }
}

// Products with a conjugate-transposed left factor (the adjoint solves):
// 32 x 32 output tiles, 16-deep slabs of both operands staged in shared
// memory.  Kept apart from the forward kernels so that their code is not
// touched by the transposed operand access.
template <typename T>
__global__ void __launch_bounds__(256) k_gemm_ta(GemmArgs<T> g) {
  constexpr int BM = 32, BN = 32, BK = 16;
  __shared__ T As[BK][BM + 1];
  __shared__ T Bs[BK][BN + 1];
  const int tid = threadIdx.x;
  const int tx = tid % 16, ty = tid / 16;  // 2 x 2 outputs per thread
  for (int b = blockIdx.z; b < g.batch; b += gridDim.z) {
    const T* A = g.A.item(b);
    const T* B = g.B.item(b);
    T* C = g.C.item(b);
    const int i0 = blockIdx.x * BM, j0 = blockIdx.y * BN;
    T acc[2][2];
#pragma unroll
    for (int r = 0; r < 2; ++r)
#pragma unroll
      for (int c = 0; c < 2; ++c) acc[r][c] = T(0.0);
    for (int k0 = 0; k0 < g.K; k0 += BK) {
      for (int e = tid; e < BM * BK; e += 256) {
        const int l = e % BK, i = e / BK;  // consecutive threads walk A's column
        const int gi = i0 + i, gl = k0 + l;
        As[l][i] = (gi < g.M && gl < g.K) ? g.a_at(A, b, gi, gl) : T(0.0);
      }
      for (int e = tid; e < BK * BN; e += 256) {
        const int l = e % BK, j = e / BK;
        const int gl = k0 + l, gj = j0 + j;
        Bs[l][j] = (gl < g.K && gj < g.N) ? B[(int64_t)g.brow.at(b, gl) + (int64_t)gj * g.B.ld] : T(0.0);
      }
      __syncthreads();
#pragma unroll
      for (int kk = 0; kk < BK; ++kk) {
        const T a0 = As[kk][tx], a1 = As[kk][tx + 16], b0 = Bs[kk][ty], b1 = Bs[kk][ty + 16];
        acc[0][0] = fmac(acc[0][0], a0, b0);
        acc[0][1] = fmac(acc[0][1], a0, b1);
        acc[1][0] = fmac(acc[1][0], a1, b0);
        acc[1][1] = fmac(acc[1][1], a1, b1);
      }
      __syncthreads();
    }
    const bool use_beta = !is_zero(g.beta);
#pragma unroll
    for (int r = 0; r < 2; ++r) {
      const int gi = i0 + tx + 16 * r;
      if (gi >= g.M) continue;
      const int64_t ci = g.crow.at(b, gi);
#pragma unroll
      for (int c = 0; c < 2; ++c) {
        const int gj = j0 + ty + 16 * c;
        if (gj >= g.N) continue;
        T* p = C + ci + (int64_t)gj * g.C.ld;
        T v = g.alpha * acc[r][c];
        if (use_beta) v = fmac(v, g.beta, *p);
        *p = v;
      }
    }
  }
}

template <typename T, int BM>
void launch_gemm(const GemmArgs<T>& g, cudaStream_t st) {
  const dim3 grid((unsigned)((g.M + BM - 1) / BM) * (unsigned)((g.N + 256 / BM - 1) / (256 / BM)), std::min(g.batch, 65535));
  switch (epi_mode(g)) {
    case EPI_SUB: k_gemm<T, EPI_SUB, BM><<<grid, 128, 0, st>>>(g); break;
    case EPI_SET: k_gemm<T, EPI_SET, BM><<<grid, 128, 0, st>>>(g); break;
    default: k_gemm<T, EPI_GENERAL, BM><<<grid, 128, 0, st>>>(g); break;
  }
}

// outputs that tiles of bm x 256 / bm compute for an M x N product
inline int64_t padded_outputs(int M, int N, int bm) {
  return ((int64_t)(M + bm - 1) / bm * bm) * ((int64_t)(N + 256 / bm - 1) / (256 / bm) * (256 / bm));
}

template <typename T>
cudaError_t gemm(const GemmArgs<T>& g, cudaStream_t st, Prof* pf) {
  if (g.M <= 0 || g.N <= 0 || g.batch <= 0) return cudaSuccess;
  if (g.K > 0 && tc_applicable(g)) {
    const cudaError_t e = gemm_tc(g, st, pf);
    if (e != cudaErrorMemoryAllocation) return e;
    // the digit-slice workspace could not grow (nothing was launched): the
    // product runs on the FP64 pipe instead
    cudaGetLastError();
  }
  if (pf) {
    pf->begin(st);
    pf->note(g.M, g.N, g.K, g.batch);
  }
  if (g.ta) {
    dim3 grid((g.M + 31) / 32, (g.N + 31) / 32, std::min(g.batch, 65535));
    k_gemm_ta<T><<<grid, 256, 0, st>>>(g);
  } else if (g.N <= 8 && g.K >= 32 && (int64_t)((g.M + 127) / 128) * g.batch < 304) {
    dim3 grid((g.M + 31) / 32, 1, std::min(g.batch, 65535));
    if (g.N == 1) k_gemm_skinny_kg<T, 1><<<grid, 256, 0, st>>>(g);
    else if (g.N == 2) k_gemm_skinny_kg<T, 2><<<grid, 256, 0, st>>>(g);
    else if (g.N <= 4) k_gemm_skinny_kg<T, 4><<<grid, 256, 0, st>>>(g);
    else k_gemm_skinny_kg<T, 8><<<grid, 256, 0, st>>>(g);
  } else if (g.N <= 8) {
    dim3 grid((g.M + 127) / 128, 1, std::min(g.batch, 65535));
    if (g.N == 1) k_gemm_skinny<T, 1><<<grid, 128, 0, st>>>(g);
    else if (g.N == 2) k_gemm_skinny<T, 2><<<grid, 128, 0, st>>>(g);
    else if (g.N <= 4) k_gemm_skinny<T, 4><<<grid, 128, 0, st>>>(g);
    else k_gemm_skinny<T, 8><<<grid, 128, 0, st>>>(g);
  } else {
    const int64_t o32 = padded_outputs(g.M, g.N, 32), o16 = padded_outputs(g.M, g.N, 16), o8 = padded_outputs(g.M, g.N, 8);
    if (o32 <= o16 && o32 <= o8) launch_gemm<T, 32>(g, st);
    else if (o16 <= o8) launch_gemm<T, 16>(g, st);
    else launch_gemm<T, 8>(g, st);
    if (pf) pf->end(K_GEMM, fma_flops<T>() * g.M * (double)g.N * g.K * g.batch, st,
                    (sizeof(T) == 16 ? 6.0 : 2.0) * g.M * (double)g.N * g.K * g.batch);   // 3M: three of four
    return cudaGetLastError();
  }
  if (pf) pf->end(K_GEMM, fma_flops<T>() * g.M * (double)g.N * g.K * g.batch, st);
  return cudaGetLastError();
}

// --------------------------------------------------------------- fill -----

template <typename T>
__global__ void k_fill(BOp<T> C, int M, int N, int batch, T value, T diag) {
  int64_t total = (int64_t)M * N;
  for (int b = blockIdx.y; b < batch; b += gridDim.y) {
    T* c = C.item(b);
    for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < total;
         e += (int64_t)gridDim.x * blockDim.x) {
      int i = (int)(e % M), j = (int)(e / M);
      c[i + (int64_t)j * C.ld] = (i == j) ? diag : value;
    }
  }
}

template <typename T>
cudaError_t fill(BOp<T> C, int M, int N, int batch, T value, T diag, cudaStream_t st, Prof* pf) {
  if (M <= 0 || N <= 0 || batch <= 0) return cudaSuccess;
  int64_t total = (int64_t)M * N;
  int bx = (int)std::min<int64_t>((total + 255) / 256, 4096);
  dim3 grid(bx, std::min(batch, 65535));
  if (pf) pf->begin(st);
  k_fill<T><<<grid, 256, 0, st>>>(C, M, N, batch, value, diag);
  if (pf) pf->end(K_OTHER, 0.0, st);
  return cudaGetLastError();
}

// Streaming multiprocessors of the current device (queried once per process).
int device_sms() {
  static const int sms = [] {
    int dev = 0, s = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || cudaDeviceGetAttribute(&s, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) {
      cudaGetLastError();
      return 1;
    }
    return s > 0 ? s : 1;
  }();
  return sms;
}

bool stream_capturing(cudaStream_t st) {
  cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
  if (cudaStreamIsCapturing(st, &cap) == cudaSuccess) return cap != cudaStreamCaptureStatusNone;
  cudaGetLastError();
  return true;
}

// ------------------------------------------------------------ panel LU ----

// Factor the panel A[k0:n, k0:k0+nb) of each matrix with partial pivoting.
// The rows [k0, n) are split into G contiguous chunks, one per CTA of the
// matrix's group; each CTA holds its chunk of the panel in shared memory
// (column-major, `ch` rows).  Per column: local argmax, publish candidate,
// group barrier, global pick (largest |.|, lowest row on ties), swap, update.
// Pivot order: larger magnitude first, then the lower row.  Magnitudes are
// non-negative (or -1 for "none"), so their IEEE bit patterns order like the
// values as signed 64-bit integers; comparing those keeps the search on the
// integer pipe instead of the FP64 pipe.
__device__ __forceinline__ bool piv_better(double m, int r, double best_m, int best_r) {
  const long long a = __double_as_longlong(m), b = __double_as_longlong(best_m);
  return a > b || (a == b && r < best_r);
}

// The panel rows [r0, r0 + rc) x columns [k0, k0 + nb) into shared memory
// (column-major, ch rows) with asynchronous copies: every load is in flight
// at once (plain loads would wait one by one, since the compiler cannot tell
// the global source from the shared destination).  Ends with the copies done
// for this thread; the caller's barrier publishes them.
template <typename T>
__device__ __forceinline__ void load_panel(T* Ps, const T* Ab, int lda, int r0, int k0, int rc, int ch, int nb,
                                           int tid, int nth) {
  for (int c = 0; c < nb; ++c)
    for (int r = tid; r < rc; r += nth)
      asm volatile("cp.async.ca.shared.global [%0], [%1], %2;" ::"r"((unsigned)__cvta_generic_to_shared(
                       Ps + r + (size_t)c * ch)),
                   "l"(Ab + (int64_t)(r0 + r) + (int64_t)(k0 + c) * lda), "n"((int)sizeof(T))
                   : "memory");
  asm volatile("cp.async.commit_group;" ::: "memory");
  asm volatile("cp.async.wait_all;" ::: "memory");
}

template <typename T, bool COOP>
__global__ void __launch_bounds__(256) k_lu_panel(BOp<T> A, int n, int k0, int nb, int G, int* ipiv,
                                                  int* info, unsigned* bars, T* pubv, double* pubm,
                                                  int* pubr, unsigned* dev_err) {
  // Threads form RT row lanes x CT column lanes (CT > 1 when the chunk has
  // fewer rows than threads); per column the pivot is reduced (warp
  // shuffles, then every thread over the warp results), rows j and p are
  // swapped one column per thread, every thread forms the multipliers of its
  // rows, and after one more barrier updates its columns (cyclic from
  // jj + 1), the lane of column jj + 1 tracking that column's largest entry
  // for the next step: three block barriers per column.
  extern __shared__ unsigned char smem_raw[];
  T* Ps = reinterpret_cast<T*>(smem_raw);
  const int b = blockIdx.x / G, g = blockIdx.x % G;
  const int rows = n - k0;
  const int ch = (rows + G - 1) / G;
  const int r0 = k0 + g * ch;                 // first global row of this chunk
  const int rc = max(0, min(ch, n - r0));     // rows in this chunk
  T* Ab = A.item(b);
  const int lda = A.ld;
  T* Wv = Ps + (size_t)ch * nb;               // pivot row after the swap (nb)
  T* Rv = Wv + nb;                            // old row j (nb)
  __shared__ double red_m[8];
  __shared__ int red_r[8];
  __shared__ int s_bg;
  __shared__ double s_inv_raw[2];  // 1 / pivot, formed once per column
  const int tid = threadIdx.x, nth = blockDim.x;
  const int lane = tid & 31, wid = tid >> 5, nw = nth >> 5;
  int CT = 1;
  while (CT < 16 && CT * 2 <= nb && (nth / (CT * 2)) >= rc && nth / (CT * 2) >= 32) CT *= 2;
  const int RT = nth / CT, rt = tid % RT, ct = tid / RT;

  load_panel(Ps, Ab, lda, r0, k0, rc, ch, nb, tid, nth);
  __syncthreads();
  T* pv = COOP ? pubv + (size_t)b * 2 * (G + 1) * nb : nullptr;
  double* pm = COOP ? pubm + (size_t)b * 2 * G : nullptr;
  int* pr = COOP ? pubr + (size_t)b * 2 * G : nullptr;
  unsigned* bar = COOP ? bars + 2 * b : nullptr;

  // this thread's best entry of the current column (rows >= j)
  double best = -1.0;
  int brow = 0x7fffffff;
  for (int r = max(0, k0 - r0) + tid; r < rc; r += nth) {
    const double m = mag1(Ps[r]);
    if (piv_better(m, r0 + r, best, brow)) { best = m; brow = r0 + r; }
  }
  for (int jj = 0; jj < nb; ++jj) {
    const int j = k0 + jj;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      const double m2 = __shfl_down_sync(0xffffffffu, best, o);
      const int r2 = __shfl_down_sync(0xffffffffu, brow, o);
      if (piv_better(m2, r2, best, brow)) { best = m2; brow = r2; }
    }
    if (lane == 0) { red_m[wid] = best; red_r[wid] = brow; }
    __syncthreads();
    double pmag = red_m[0];
    int p = red_r[0];
    for (int w = 1; w < nw; ++w)
      if (piv_better(red_m[w], red_r[w], pmag, p)) { pmag = red_m[w]; p = red_r[w]; }
    const bool own_j = (j >= r0 && j < r0 + rc);
    if (COOP) {
      const int slot = jj & 1;
      if (tid == 0) { pm[slot * G + g] = pmag; pr[slot * G + g] = p; }
      const int lr = p - r0;
      for (int c = tid; c < nb; c += nth) {
        if (pmag >= 0.0 && lr >= 0 && lr < rc) pv[((size_t)slot * (G + 1) + g) * nb + c] = Ps[lr + (size_t)c * ch];
        if (own_j) pv[((size_t)slot * (G + 1) + G) * nb + c] = Ps[(j - r0) + (size_t)c * ch];
      }
      if (!group_barrier(bar, G, dev_err)) return;
      // the global pivot: warp 0 reduces the G published candidates (loads
      // bypass L1: the values were written by other CTAs)
      if (wid == 0) {
        double bm = -1.0;
        int brr = 0x7fffffff, bg = 0;
        for (int q2 = lane; q2 < G; q2 += 32) {
          const double m = __ldcg(&pm[slot * G + q2]);
          const int rr = __ldcg(&pr[slot * G + q2]);
          if (piv_better(m, rr, bm, brr)) { bm = m; brr = rr; bg = q2; }
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
          const double m2 = __shfl_down_sync(0xffffffffu, bm, o);
          const int r2 = __shfl_down_sync(0xffffffffu, brr, o);
          const int g2 = __shfl_down_sync(0xffffffffu, bg, o);
          if (piv_better(m2, r2, bm, brr)) { bm = m2; brr = r2; bg = g2; }
        }
        if (lane == 0) { red_m[0] = bm; red_r[0] = brr; s_bg = bg; }
      }
      __syncthreads();
      pmag = red_m[0];
      p = red_r[0];
      const double* wsrc = reinterpret_cast<const double*>(pv + ((size_t)slot * (G + 1) + s_bg) * nb);
      const double* rsrc = reinterpret_cast<const double*>(pv + ((size_t)slot * (G + 1) + G) * nb);
      double* wdst = reinterpret_cast<double*>(Wv);
      double* rdst = reinterpret_cast<double*>(Rv);
      constexpr int DW = sizeof(T) / sizeof(double);
      for (int c = tid; c < nb * DW; c += nth) {
        wdst[c] = __ldcg(&wsrc[c]);
        rdst[c] = __ldcg(&rsrc[c]);
      }
      __syncthreads();
      for (int c = tid; c < nb; c += nth) {
        if (own_j) Ps[(j - r0) + (size_t)c * ch] = Wv[c];
        if (p != j && p >= r0 && p < r0 + rc) Ps[(p - r0) + (size_t)c * ch] = Rv[c];
        if (c == jj) *reinterpret_cast<T*>(s_inv_raw) = (pmag == 0.0) ? T(0.0) : recip(Wv[c]);
      }
    } else {
      // one column per thread: read both rows, then write them swapped
      for (int c = tid; c < nb; c += nth) {
        const T wv = Ps[(p - r0) + (size_t)c * ch];
        const T rv = Ps[(j - r0) + (size_t)c * ch];
        Wv[c] = wv;
        Ps[(j - r0) + (size_t)c * ch] = wv;
        if (p != j) Ps[(p - r0) + (size_t)c * ch] = rv;
        if (c == jj) *reinterpret_cast<T*>(s_inv_raw) = (pmag == 0.0) ? T(0.0) : recip(wv);
      }
    }
    if (g == 0 && tid == 0) {
      ipiv[(int64_t)b * n + j] = p;
      if (pmag == 0.0 && info[b] == 0) info[b] = j + 1;
    }
    __syncthreads();
    // multipliers of this thread's rows (at most ch / RT + 1 of them are
    // kept: the rows rlo + rt, rlo + rt + RT, ...), then the update of its
    // columns; the next column's candidates are tracked by column lane 0
    const T inv = *reinterpret_cast<const T*>(s_inv_raw);
    const int rlo = max(0, j + 1 - r0);
    best = -1.0;
    brow = 0x7fffffff;
    if (CT == 1) {
      for (int r = rlo + rt; r < rc; r += RT) {
        const T l = Ps[r + (size_t)jj * ch] * inv;
        Ps[r + (size_t)jj * ch] = l;
        for (int c = jj + 1; c < nb; ++c) {
          const T v = fmsc(Ps[r + (size_t)c * ch], l, Wv[c]);
          Ps[r + (size_t)c * ch] = v;
          if (c == jj + 1) {
            const double m = mag1(v);
            if (piv_better(m, r0 + r, best, brow)) { best = m; brow = r0 + r; }
          }
        }
      }
    } else {
      // rc <= RT here: each thread has at most one row
      const int r = rlo + rt;
      T l = T(0.0);
      if (r < rc) l = Ps[r + (size_t)jj * ch] * inv;
      __syncthreads();
      if (r < rc) {
        if (ct == 0) Ps[r + (size_t)jj * ch] = l;
        for (int c = jj + 1 + ct; c < nb; c += CT) {
          const T v = fmsc(Ps[r + (size_t)c * ch], l, Wv[c]);
          Ps[r + (size_t)c * ch] = v;
          if (c == jj + 1) {
            const double m = mag1(v);
            if (piv_better(m, r0 + r, best, brow)) { best = m; brow = r0 + r; }
          }
        }
      }
    }
  }
  __syncthreads();
  for (int c = 0; c < nb; ++c)
    for (int r = tid; r < rc; r += nth) Ab[(int64_t)(r0 + r) + (int64_t)(k0 + c) * lda] = Ps[r + (size_t)c * ch];
}

// Panel LU of tall panels in the distributed shared memory of a thread-block
// cluster.  The rows [k0, n) are split into CS contiguous chunks, one per CTA
// of the matrix's cluster, each held in that CTA's shared memory for the
// whole panel.  Rows never move during the panel: a chosen pivot row is only
// marked done, and the interchanges are recorded in LAPACK's form (ipiv) by
// a replay of the swap sequence on the panel's top positions (every warp
// keeps its own copy in registers, lane t for position k0 + t); at the end
// every row is written to its final position.
//
// Per column, one block barrier and one cluster barrier, and no remote load:
// every warp reduces its rows' candidates with shuffles; warp 0 reduces the
// eight warp candidates to the CTA's candidate (largest magnitude, and on ties
// the lowest current position -- the row order after the interchanges so far,
// which is LAPACK's choice), forms the reciprocal of its pivot-column entry
// and pushes the candidate -- magnitude, position, row, reciprocal and the
// row's panel values -- into the shared memory of every CTA of the cluster.
// After the cluster barrier every warp picks the same pivot from its own
// shared memory and updates its rows.  Candidates are double-buffered by
// column parity: a CTA pushes into a slot again only two columns later, after
// a barrier that every CTA reaches only once it has finished with the slot.
template <typename T>
__global__ void __launch_bounds__(256) k_lu_panel_cluster(BOp<T> A, int n, int k0, int nb, int* ipiv,
                                                          int* info) {
  namespace cg = cooperative_groups;
  cg::cluster_group cl = cg::this_cluster();
  const int CS = (int)cl.num_blocks();
  const int g = (int)cl.block_rank();
  const int b = blockIdx.x / CS;
  const int rows = n - k0;
  const int ch = (rows + CS - 1) / CS;
  const int r0 = k0 + g * ch;
  const int rc = max(0, min(ch, n - r0));
  extern __shared__ __align__(16) unsigned char smem_raw[];
  T* Ps = reinterpret_cast<T*>(smem_raw);              // ch x nb, column-major
  T* cv = Ps + (size_t)ch * nb;                        // [2 slots][CS][nb]: every CTA's candidate row
  int* chosen = reinterpret_cast<int*>(cv + (size_t)2 * CS * nb);  // ch: pivot step of a row, or -1
  __shared__ long long wm[8];                          // warp candidates of this CTA
  __shared__ int wq[8], wp[8];
  __shared__ long long cm[2 * 16];                     // [slot][CTA] pushed candidates
  __shared__ int cq[2 * 16], cr[2 * 16];
  __shared__ double cinv_raw[2 * 16 * 2];              // their reciprocals (T)
  T* cinv = reinterpret_cast<T*>(cinv_raw);
  const int tid = threadIdx.x, nth = blockDim.x;
  const int lane = tid & 31, wid = tid >> 5;
  const int kmax = (ch + nth - 1) / nth;               // row slots per thread, uniform over the CTA
  T* Ab = A.item(b);
  const int lda = A.ld;

  load_panel(Ps, Ab, lda, r0, k0, rc, ch, nb, tid, nth);
  for (int r = tid; r < ch; r += nth) chosen[r] = -1;
  int phys = k0 + lane;   // row now at position k0 + lane
  int pos = k0 + lane;    // current position of row k0 + lane
  // every CTA of the cluster has started before any writes into its shared memory
  cl.sync();
  // (magnitude, current position) orders candidates; prow is the row itself
  double best = -1.0;
  int bpos = 0x7fffffff, prow = -1;
  for (int r = tid; r < rc; r += nth) {
    const double m = mag1(Ps[r]);
    if (piv_better(m, r0 + r, best, bpos)) { best = m; bpos = r0 + r; prow = r0 + r; }
  }
  for (int jj = 0; jj < nb; ++jj) {
    const int slot = jj & 1;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      const double m2 = __shfl_down_sync(0xffffffffu, best, o);
      const int q2 = __shfl_down_sync(0xffffffffu, bpos, o);
      const int p2 = __shfl_down_sync(0xffffffffu, prow, o);
      if (piv_better(m2, q2, best, bpos)) { best = m2; bpos = q2; prow = p2; }
    }
    if (lane == 0) { wm[wid] = __double_as_longlong(best); wq[wid] = bpos; wp[wid] = prow; }
    __syncthreads();
    if (wid == 0) {
      double m = -1.0;
      int q = 0x7fffffff, p = -1;
      if (lane < 8) { m = __longlong_as_double(wm[lane]); q = wq[lane]; p = wp[lane]; }
#pragma unroll
      for (int o = 4; o > 0; o >>= 1) {
        const double m2 = __shfl_down_sync(0xffffffffu, m, o);
        const int q2 = __shfl_down_sync(0xffffffffu, q, o);
        const int p2 = __shfl_down_sync(0xffffffffu, p, o);
        if (piv_better(m2, q2, m, q)) { m = m2; q = q2; p = p2; }
      }
      m = __shfl_sync(0xffffffffu, m, 0);
      q = __shfl_sync(0xffffffffu, q, 0);
      p = __shfl_sync(0xffffffffu, p, 0);
      const bool has = m >= 0.0;
      const T v = (has && lane < nb) ? Ps[(p - r0) + (size_t)lane * ch] : T(0.0);
      T inv = T(0.0);
      if (lane == jj && has && m != 0.0) inv = recip(v);
      inv = shfl_val(inv, jj);
      for (int d = 0; d < CS; ++d)
        if (lane < nb) cl.map_shared_rank(cv, d)[((size_t)slot * CS + g) * nb + lane] = v;
      if (lane < CS) {
        const int e2 = slot * 16 + g;
        cl.map_shared_rank(cm, lane)[e2] = __double_as_longlong(m);
        cl.map_shared_rank(cq, lane)[e2] = q;
        cl.map_shared_rank(cr, lane)[e2] = p;
        cl.map_shared_rank(cinv, lane)[e2] = inv;
      }
    }
    cl.sync();
    // the pivot, chosen by every warp from its own CTA's shared memory
    double pm = -1.0;
    int pq = 0x7fffffff, pp = -1, pw = 0;
    if (lane < CS) {
      pm = __longlong_as_double(cm[slot * 16 + lane]);
      pq = cq[slot * 16 + lane];
      pp = cr[slot * 16 + lane];
      pw = lane;
    }
#pragma unroll
    for (int o = 8; o > 0; o >>= 1) {
      const double m2 = __shfl_down_sync(0xffffffffu, pm, o);
      const int q2 = __shfl_down_sync(0xffffffffu, pq, o);
      const int p2 = __shfl_down_sync(0xffffffffu, pp, o);
      const int w2 = __shfl_down_sync(0xffffffffu, pw, o);
      if (piv_better(m2, q2, pm, pq)) { pm = m2; pq = q2; pp = p2; pw = w2; }
    }
    pm = __shfl_sync(0xffffffffu, pm, 0);
    pq = __shfl_sync(0xffffffffu, pq, 0);
    pp = __shfl_sync(0xffffffffu, pp, 0);
    pw = __shfl_sync(0xffffffffu, pw, 0);
    const T* Wv = cv + ((size_t)slot * CS + pw) * nb;
    const T inv = cinv[slot * 16 + pw];
    const int j = k0 + jj;
    if (pp >= r0 && pp < r0 + rc && (pp - r0) % nth == tid) chosen[pp - r0] = jj;
    // LAPACK interchange: position j <-> the winner's current position pq
    {
      const int rj = __shfl_sync(0xffffffffu, phys, jj);
      if (lane == rj - k0) pos = pq;
      if (pq - k0 < nb && lane == pq - k0) phys = rj;
      if (lane == jj) phys = pp;
      if (pp - k0 < nb && lane == pp - k0) pos = j;
    }
    if (g == 0 && tid == 0) {
      ipiv[(int64_t)b * n + j] = pq;
      if (pm == 0.0 && info[b] == 0) info[b] = j + 1;
    }
    best = -1.0;
    bpos = 0x7fffffff;
    prow = -1;
    for (int k = 0; k < kmax; ++k) {
      const int r = tid + k * nth;
      const int pr = r0 + r;
      const int ptop = __shfl_sync(0xffffffffu, pos, (pr - k0) & 31);
      if (r >= rc || chosen[r] >= 0) continue;
      const int cpos = pr - k0 < nb ? ptop : pr;  // after this column's interchange
      const T l = Ps[r + (size_t)jj * ch] * inv;
      Ps[r + (size_t)jj * ch] = l;
      for (int c = jj + 1; c < nb; ++c) {
        const T v = fmsc(Ps[r + (size_t)c * ch], l, Wv[c]);
        Ps[r + (size_t)c * ch] = v;
        if (c == jj + 1) {
          const double m = mag1(v);
          if (piv_better(m, cpos, best, bpos)) { best = m; bpos = cpos; prow = pr; }
        }
      }
    }
  }
  // rows to their final positions
  for (int k = 0; k < kmax; ++k) {
    const int r = tid + k * nth;
    const int pr = r0 + r;
    const int ptop = __shfl_sync(0xffffffffu, pos, (pr - k0) & 31);
    if (r >= rc) continue;
    int dst = pr;
    if (chosen[r] >= 0) dst = k0 + chosen[r];
    else if (pr - k0 < nb) dst = ptop;
    for (int c = 0; c < nb; ++c) Ab[(int64_t)dst + (int64_t)(k0 + c) * lda] = Ps[r + (size_t)c * ch];
  }
  cl.sync();
}

// Cluster shape for a panel of `rows` rows of `batch` matrices: a power of
// two of CTAs, at least 2, growing while a CTA would hold more than 128 rows
// and the clusters of all matrices still fit on the SMs at once (the panel's
// FP64 update is spread over more SMs), then until the chunk fits in shared
// memory; at most the largest cluster the device runs with the kernel's
// shared memory; 0 when the panel does not fit (the cooperative kernel is
// used then).
template <typename T>
size_t panel_cluster_smem(int rows, int nb, int cs) {
  const int ch = (rows + cs - 1) / cs;
  return ((size_t)ch * nb + 2 * (size_t)cs * nb) * sizeof(T) + (size_t)ch * sizeof(int) + 16;
}

template <typename T>
int panel_cluster_max() {
  static const int mx = [] {
    int dev = 0, smem_max = 0;
    if (cudaGetDevice(&dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&smem_max, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev) != cudaSuccess) {
      cudaGetLastError();
      return 0;
    }
    cudaFuncAttributes fa;
    if (cudaFuncGetAttributes(&fa, k_lu_panel_cluster<T>) != cudaSuccess ||
        cudaFuncSetAttribute(k_lu_panel_cluster<T>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             smem_max - (int)fa.sharedSizeBytes) != cudaSuccess ||
        cudaFuncSetAttribute(k_lu_panel_cluster<T>, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) !=
            cudaSuccess) {
      cudaGetLastError();
      return 0;
    }
    // the largest cluster that can be resident with a near-full shared memory per CTA
    for (int cs = 16; cs >= 2; cs /= 2) {
      cudaLaunchConfig_t cfg = {};
      cfg.gridDim = dim3(cs);
      cfg.blockDim = dim3(256);
      cfg.dynamicSmemBytes = (size_t)(smem_max - (int)fa.sharedSizeBytes);
      cudaLaunchAttribute at[1];
      at[0].id = cudaLaunchAttributeClusterDimension;
      at[0].val.clusterDim.x = cs;
      at[0].val.clusterDim.y = 1;
      at[0].val.clusterDim.z = 1;
      cfg.attrs = at;
      cfg.numAttrs = 1;
      int ncl = 0;
      if (cudaOccupancyMaxActiveClusters(&ncl, (void*)k_lu_panel_cluster<T>, &cfg) == cudaSuccess && ncl > 0)
        return cs;
      cudaGetLastError();
    }
    return 0;
  }();
  return mx;
}

template <typename T>
int panel_cluster_size(int rows, int nb, int batch) {
  const int mx = panel_cluster_max<T>();
  if (mx < 2 || nb > 32) return 0;
  int smem_max = 0, dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess ||
      cudaDeviceGetAttribute(&smem_max, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev) != cudaSuccess) {
    cudaGetLastError();
    return 0;
  }
  int cs = 2;
  while (cs < mx && (rows + cs - 1) / cs > 128 && (int64_t)batch * cs * 2 <= device_sms()) cs *= 2;
  while (cs <= mx && panel_cluster_smem<T>(rows, nb, cs) + 8192 > (size_t)smem_max) cs *= 2;
  return cs <= mx ? cs : 0;
}

// Panel LU with the panel's rows in registers.
//
// The rows [k0, n) are split into CS contiguous chunks of at most 512, one per
// CTA of the matrix's cluster (CS = 1: a plain CTA).  A row belongs to CT
// threads of different warps, thread q holding its columns q, q + CT, ... :
// one thread per row when the chunk has a warp of rows for each of the SM's
// four schedulers, two or four when it has fewer.  Every step works on the
// registers' front column: the owners' update writes one register down, so
// that one loop body serves a whole segment of steps (the width shrinks by a
// segment at a time: at most 10 % of the multiply-adds are spent on columns
// already left behind).  Rows never move during the panel: a chosen row only
// leaves the search, the interchanges are recorded in LAPACK's form (ipiv) by
// a replay of the swap sequence on the panel's top positions (every warp keeps
// its own copy in registers, lane t for position k0 + t), the finished entries
// of L and U collect in shared memory, and at the end every row is written to
// its final position.
//
// Per column: each warp of the column's owners finds its candidate (largest
// magnitude, and on ties the lowest current position -- the row order after
// the interchanges so far, which is LAPACK's choice) with warp-wide integer
// maxima of the magnitude's two words; after one block barrier every warp
// knows the CTA's candidate; the warps that hold it push its key and values
// into the shared memory of every CTA of the cluster, and its reciprocal as
// soon as it is formed, with stores that count their bytes on the receiver's
// mbarriers (bounded waits); every warp then picks the same pivot from its own
// shared memory.  Candidates are double-buffered by column parity: a CTA
// pushes into a slot again only two columns later, after receiving the
// candidates that every CTA sends once it has finished with the slot.  So are
// the candidates of the CTA's own warps (wrec): in a cluster with one thread
// per row only the next column's block barrier orders a warp's reading of them
// before what another warp writes after that.
//
// What bounds it: the chain from one pivot to the next.  The FP64 pipe takes
// 64 cycles per warp instruction and scheduler; a division is ~440 cycles, the
// exchange ~700, the searches ~400, the update of 432 rows on 16 CTAs ~460.
// Measured, 32 columns of one matrix: 432 rows 100 -> 46 us, 1728 rows 110 ->
// 64 us, 6720 rows 176 -> 113 us (FP64 update ~3900 of 6700 cycles a column);
// 16 complex columns of 1696 rows 75 -> 53 us.  The earlier form kept the rows
// in shared memory, where each multiply-add waited for the store before it,
// and took two cluster-wide barriers' time per column.
template <typename T> struct LuNB;
template <> struct LuNB<double> { enum { NB = 32 }; };
template <> struct LuNB<cplx> { enum { NB = 16 }; };

// Largest key (hi, lo) over the warp's lanes, lowest position on ties; hi = 0
// means no candidate.  Returns the lane that holds it.
__device__ __forceinline__ int warp_pivot(uint32_t& hi, uint32_t& lo, uint32_t& pos) {
  const uint32_t mh = __reduce_max_sync(0xffffffffu, hi);
  const uint32_t ml = __reduce_max_sync(0xffffffffu, hi == mh ? lo : 0u);
  const bool in = hi == mh && lo == ml;
  const uint32_t mp = __reduce_min_sync(0xffffffffu, in ? pos : 0xffffffffu);
  const int src = __ffs((int)__ballot_sync(0xffffffffu, in && pos == mp)) - 1;
  hi = mh;
  lo = ml;
  pos = mp;
  return src;
}

// Store to another CTA's shared memory (cluster addresses) that adds its bytes
// to that CTA's mbarrier when it lands.
__device__ __forceinline__ void st_async(uint32_t dst, double v, uint32_t bar) {
  asm volatile("st.async.weak.shared::cluster.mbarrier::complete_tx::bytes.b64 [%0], %1, [%2];" ::"r"(dst),
               "l"(__double_as_longlong(v)), "r"(bar) : "memory");
}
__device__ __forceinline__ void st_async(uint32_t dst, cplx v, uint32_t bar) {
  asm volatile("st.async.weak.shared::cluster.mbarrier::complete_tx::bytes.v2.b64 [%0], {%1, %2}, [%3];" ::"r"(dst),
               "l"(__double_as_longlong(v.re)), "l"(__double_as_longlong(v.im)), "r"(bar) : "memory");
}
__device__ __forceinline__ void st_async(uint32_t dst, uint4 v, uint32_t bar) {
  asm volatile("st.async.weak.shared::cluster.mbarrier::complete_tx::bytes.v4.b32 [%0], {%1, %2, %3, %4}, [%5];" ::"r"(dst),
               "r"(v.x), "r"(v.y), "r"(v.z), "r"(v.w), "r"(bar) : "memory");
}
__device__ __forceinline__ uint32_t smem_addr(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }
__device__ __forceinline__ uint32_t peer_addr(uint32_t local, int rank) {
  uint32_t r;
  asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(local), "r"(rank));
  return r;
}
__device__ __forceinline__ void mbar_expect(uint64_t* bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_addr(bar)), "r"(bytes) : "memory");
}
// bounded wait for a phase whose bytes come from the cluster's CTAs
__device__ __forceinline__ bool mbar_wait_cluster(uint64_t* bar, int parity, long limit = 1L << 22) {
  for (long it = 0; it < limit; ++it) {
    uint32_t ok;
    asm volatile("{\n.reg .pred p;\nmbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2;\nselp.u32 %0, 1, 0, p;\n}"
                 : "=r"(ok) : "r"(smem_addr(bar)), "r"(parity) : "memory");
    if (ok) return true;
    if (it > 1024) __nanosleep(64);
  }
  return false;
}

template <typename T, bool CL, int CT>
struct PanelReg {
  enum { NB = LuNB<T>::NB, SEG = 4, NQ = NB / CT };
  T* Ps;          // finished entries, column-major, ld rows
  T* cv;          // [2 slots][CS][NB] candidate rows (lay)
  T* cinv;        // [2][CS] reciprocals of their pivot entries
  uint4* crec;    // [2][CS] their keys: magnitude hi + 1, lo, position, row
  uint64_t* bar;  // [2] keys and rows of a slot have arrived, [2] reciprocals
  uint4* wrec;    // [2 slots][16] this CTA's warps' candidates
  T* srow;        // [NB + 1] the CTA candidate's row and reciprocal (3 more are read past a row's end)
  unsigned* err;
  int CS, g, k0, nb, r0, ld, RW;
  int lane, rw, q;   // row warp, column group
  int row;        // row of the chunk
  int phys, pos;  // row now at position k0 + lane; position of row k0 + lane
  int chosen;     // step at which this thread's row became the pivot, or -1
  bool done;      // row absent or chosen
  T a[NQ];        // columns q, q + CT, ... of the row; a[0] is the first not finished (beyond the panel, and of a done row: unused)

  // place of column jj + r in a candidate row of step jj: each group's columns together
  static __device__ __forceinline__ int lay(int r) { return CT == 1 ? r : (r & (CT - 1)) * NQ + r / CT; }

  // step jj on registers of WIDTH / CT columns each (jj .. of the segment)
  template <int WIDTH>
  __device__ __forceinline__ void step(int jj, int* ip, int* info_b) {
    constexpr int WQ = WIDTH / CT;
    const int slot = jj & 1;
    const int pr = r0 + row;
    const bool own = CT == 1 || q == (jj & (CT - 1));   // this group holds column jj
    const int o = CT == 1 ? 0 : (q - jj) & (CT - 1), f = jj + o;   // panel column of a[0]
    const int ptop = __shfl_sync(0xffffffffu, pos, (pr - k0) & 31);
    if (CL && threadIdx.x == 0) {
      mbar_expect(bar + slot, (uint32_t)(CS * ((NB - jj) * (int)sizeof(T) + 16)));
      mbar_expect(bar + 2 + slot, (uint32_t)(CS * (int)sizeof(T)));
    }
    if (own) {
      const unsigned long long mb = (unsigned long long)__double_as_longlong(mag1(a[0]));
      uint32_t hi = done ? 0u : (uint32_t)(mb >> 32) + 1u, lo = done ? 0u : (uint32_t)mb;
      uint32_t ps = (uint32_t)(pr - k0 < nb ? ptop : pr);
      const int src = warp_pivot(hi, lo, ps);
      if (lane == src) wrec[slot * 16 + rw] = make_uint4(hi, lo, ps, (uint32_t)pr);
    }
    __syncthreads();
    uint4 rec = wrec[slot * 16 + (RW > 1 && lane < RW ? lane : 0)];
    int w = 0;
    if (RW > 1) {
      if (lane >= RW) rec = make_uint4(0u, 0u, 0xffffffffu, 0u);
      w = warp_pivot(rec.x, rec.y, rec.z);
      rec.w = __shfl_sync(0xffffffffu, rec.w, w);
    }
    if (rw == w) {   // the warps that hold the CTA's candidate row
      if (pr == (int)rec.w) {
#pragma unroll
        for (int i = 0; i < WQ; ++i) srow[o * NQ + i] = a[i];
      }
      if constexpr (CL) {
        __syncwarp();
        const int i = lane & (NQ - 1);
        if (f + i * CT < NB) {
          const T v = srow[o * NQ + i];
          const uint32_t dv = smem_addr(cv + (slot * CS + g) * NB + o * NQ + i), db = smem_addr(bar + slot);
          for (int d = lane / NQ; d < CS; d += 32 / NQ) st_async(peer_addr(dv, d), v, peer_addr(db, d));
        }
        if (own && lane < CS)
          st_async(peer_addr(smem_addr(crec + slot * CS + g), lane), rec, peer_addr(smem_addr(bar + slot), lane));
      }
      if (own) {
        if (pr == (int)rec.w) srow[NB] = (rec.x <= 1u && rec.y == 0u) ? T(0.0) : recip(a[0]);
        if constexpr (CL) {
          __syncwarp();
          if (lane < CS)
            st_async(peer_addr(smem_addr(cinv + slot * CS + g), lane), srow[NB],
                     peer_addr(smem_addr(bar + 2 + slot), lane));
        }
      }
    }
    T inv;
    const T* Wv;
    int prow, pq;
    bool zero;
    if constexpr (CL) {
      const int par = (jj >> 1) & 1;
      bool ok = mbar_wait_cluster(bar + slot, par);
      uint4 c = lane < CS ? crec[slot * CS + lane] : make_uint4(0u, 0u, 0xffffffffu, 0u);
      const int pw = warp_pivot(c.x, c.y, c.z);
      prow = (int)__shfl_sync(0xffffffffu, c.w, pw);
      pq = (int)c.z;
      zero = c.x <= 1u && c.y == 0u;
      Wv = cv + (slot * CS + pw) * NB;
      ok = mbar_wait_cluster(bar + 2 + slot, par) && ok;
      if (!ok) atomicOr(err, DEV_ERR_TIMEOUT);
      inv = cinv[slot * CS + pw];
    } else {
      prow = (int)rec.w;
      pq = (int)rec.z;
      zero = rec.x <= 1u && rec.y == 0u;
      __syncthreads();
      Wv = srow;
      inv = srow[NB];
    }
    if (pr == prow) {
      done = true;
      chosen = jj;
    }
    T l = T(0.0);
    if (own) {
      l = a[0] * inv;
      if (!done) Ps[jj * ld + row] = l;
    }
    if constexpr (CT > 1) {
      __syncthreads();
      if (!own) l = Ps[jj * ld + row];
    }
    // the remaining columns; the owners' move one register down.  The pivot
    // row is read eight values ahead: a load right before its multiply-add
    // would show its latency (113 instead of 64 cycles each)
    {
      const T* Wq = Wv + o * NQ;
      constexpr int BW = 8;
#pragma unroll
      for (int i0 = 0; i0 < WQ; i0 += BW) {
        T w[BW];
#pragma unroll
        for (int i = 0; i < BW && i0 + i < WQ; ++i) w[i] = Wq[i0 + i];
        if (own) {
#pragma unroll
          for (int i = (i0 == 0 ? 1 : 0); i < BW && i0 + i < WQ; ++i) a[i0 + i - 1] = fmsc(a[i0 + i], l, w[i]);
        } else {
#pragma unroll
          for (int i = 0; i < BW && i0 + i < WQ; ++i) a[i0 + i] = fmsc(a[i0 + i], l, w[i]);
        }
      }
      if (own) a[WQ - 1] = T(0.0);
    }
    // the pivot row's entries of U
    if (q == 0 && (unsigned)(prow - r0 - rw * 32) < 32u)
      for (int r = lane; jj + r < nb; r += 32) Ps[(jj + r) * ld + prow - r0] = Wv[lay(r)];
    // LAPACK interchange: position j <-> the winner's current position
    const int j = k0 + jj;
    {
      const int rj = __shfl_sync(0xffffffffu, phys, jj);
      if (lane == rj - k0) pos = pq;
      if (pq - k0 < nb && lane == pq - k0) phys = rj;
      if (lane == jj) phys = prow;
      if (prow - k0 < nb && lane == prow - k0) pos = j;
    }
    if (g == 0 && threadIdx.x == 0) {
      ip[j] = pq;
      if (zero && *info_b == 0) *info_b = j + 1;
    }
  }

  template <int WIDTH>
  __device__ __forceinline__ void run(int jj, int* ip, int* info_b) {
    for (int e = min(jj + (int)SEG, nb); jj < e; ++jj) step<WIDTH>(jj, ip, info_b);
    if constexpr (WIDTH > SEG) {
      if (jj < nb) run<WIDTH - SEG>(jj, ip, info_b);
    }
  }
};

template <typename T, bool CL, int CT>
__global__ void __launch_bounds__(512) k_lu_panel_reg(BOp<T> A, int n, int k0, int nb, int CS, int* ipiv, int* info,
                                                      unsigned* err) {
  namespace cg = cooperative_groups;
  constexpr int NB = LuNB<T>::NB;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ uint4 wrec[2 * 16];
  __shared__ uint4 crec[2 * 16];
  __shared__ __align__(8) uint64_t bars[4];
  PanelReg<T, CL, CT> p;
  p.CS = CL ? CS : 1;
  p.g = CL ? (int)cg::this_cluster().block_rank() : 0;
  const int b = blockIdx.x / p.CS;
  const int rows = n - k0, ch = (rows + p.CS - 1) / p.CS;
  p.k0 = k0;
  p.nb = nb;
  p.r0 = k0 + p.g * ch;
  const int rc = max(0, min(ch, n - p.r0));
  p.RW = blockDim.x / (32 * CT);
  p.ld = p.RW * 32;
  p.Ps = reinterpret_cast<T*>(smem_raw);
  p.cv = p.Ps + (size_t)NB * p.ld;
  p.cinv = p.cv + 2 * p.CS * NB;
  p.srow = p.cinv + 2 * p.CS;
  p.wrec = wrec;
  p.crec = crec;
  p.bar = bars;
  p.err = err;
  p.lane = threadIdx.x & 31;
  p.rw = CT == 1 ? threadIdx.x >> 5 : (threadIdx.x >> 5) % p.RW;
  p.q = CT == 1 ? 0 : (threadIdx.x >> 5) / p.RW;
  p.row = p.rw * 32 + p.lane;
  p.phys = p.pos = k0 + p.lane;
  p.chosen = -1;
  p.done = p.row >= rc;
  T* Ab = A.item(b);
  const int64_t lda = A.ld;
  const T* src = Ab + (p.r0 + p.row) + (int64_t)k0 * lda;
#pragma unroll
  for (int i = 0; i < NB / CT; ++i)
    p.a[i] = (!p.done && p.q + i * CT < nb) ? src[(p.q + i * CT) * lda] : T(0.0);
  if constexpr (CL) {
    if (threadIdx.x == 0) {
      for (int i = 0; i < 4; ++i) asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_addr(bars + i)));
      asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    cg::this_cluster().sync();   // every CTA has started before any writes into its shared memory
  }
  p.template run<NB>(0, ipiv + (int64_t)b * n, info + b);
  if constexpr (CL) cg::this_cluster().sync();   // every CTA has read its rows and its candidates
  else __syncthreads();
  // rows to their final positions
  const int pr = p.r0 + p.row;
  const int ptop = __shfl_sync(0xffffffffu, p.pos, (pr - k0) & 31);
  if (p.row >= rc) return;
  const int dst = p.chosen >= 0 ? k0 + p.chosen : pr - k0 < nb ? ptop : pr;
  T* out = Ab + dst + (int64_t)k0 * lda;
  for (int c = p.q; c < nb; c += CT) out[c * lda] = p.Ps[c * p.ld + p.row];
}

// CTAs per matrix for a panel of `rows` rows of `batch` matrices: a power of
// two, enough for at most 512 rows each, then more while a CTA would hold more
// than 32 and the clusters of all matrices still fit on the SMs at once (the
// update shrinks with the rows; measured 32 / 64 / 128 rows a CTA: adaptive
// build 17.5 / 19.0 / 19.8 ms of panels); 0 when even the largest cluster is
// too small.
template <typename T>
size_t panel_reg_smem(int ld, int cs) {
  return ((size_t)LuNB<T>::NB * ld + 2 * (size_t)cs * (LuNB<T>::NB + 1) + LuNB<T>::NB + 4) * sizeof(T);
}

template <typename T, int CT>
bool panel_reg_attr(size_t sm) {
  return cudaFuncSetAttribute(k_lu_panel_reg<T, false, CT>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm) == cudaSuccess &&
         cudaFuncSetAttribute(k_lu_panel_reg<T, true, CT>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm) == cudaSuccess &&
         cudaFuncSetAttribute(k_lu_panel_reg<T, true, CT>, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) == cudaSuccess;
}

template <typename T>
int panel_reg_max() {
  static const int mx = [] {
    const size_t sm = panel_reg_smem<T>(512, 16);
    if (!panel_reg_attr<T, 1>(sm) || !panel_reg_attr<T, 2>(sm) || !panel_reg_attr<T, 4>(sm)) {
      cudaGetLastError();
      return 0;
    }
    for (int cs = 16; cs >= 2; cs /= 2) {
      cudaLaunchConfig_t cfg = {};
      cfg.gridDim = dim3(cs);
      cfg.blockDim = dim3(512);
      cfg.dynamicSmemBytes = sm;
      cudaLaunchAttribute at[1];
      at[0].id = cudaLaunchAttributeClusterDimension;
      at[0].val.clusterDim.x = cs;
      at[0].val.clusterDim.y = 1;
      at[0].val.clusterDim.z = 1;
      cfg.attrs = at;
      cfg.numAttrs = 1;
      int ncl = 0;
      if (cudaOccupancyMaxActiveClusters(&ncl, (void*)k_lu_panel_reg<T, true, 1>, &cfg) == cudaSuccess && ncl > 0) return cs;
      cudaGetLastError();
    }
    return 1;
  }();
  return mx;
}

template <typename T>
int panel_reg_size(int rows, int batch) {
  const int mx = panel_reg_max<T>();
  if (mx < 1) return 0;
  int cs = 1;
  while (cs <= mx && (rows + cs - 1) / cs > 512) cs *= 2;
  if (cs > mx) return 0;
  while (cs < mx && (rows + cs - 1) / cs > 32 && (int64_t)batch * cs * 2 <= device_sms()) cs *= 2;
  return cs;
}

template <typename T, int CT>
cudaError_t launch_panel_reg(const cudaLaunchConfig_t& cfg, int cs, BOp<T> A, int n, int k0, int nb, int* ipiv, int* info, unsigned* err) {
  return cs > 1 ? cudaLaunchKernelEx(&cfg, k_lu_panel_reg<T, true, CT>, A, n, k0, nb, cs, ipiv, info, err)
                : cudaLaunchKernelEx(&cfg, k_lu_panel_reg<T, false, CT>, A, n, k0, nb, cs, ipiv, info, err);
}

// Apply the panel's interchanges to every column outside the panel and
// solve U12 = L11^{-1} A12 for the columns in [k0 + nb, trsm_end).
//
// The interchanges are first composed into one permutation of at most 2 nb
// rows: a thread per position of the panel's top and per position that an
// interchange swapped with walks its position back through the nb
// interchanges to the row whose entries end there.  TC threads per column
// then read all moved entries at once, write the outside ones back, and solve
// the top block in registers (tri_cols.h).  Rows that stay where they are in
// a column without a solve are not touched.
//
// Bound by the substitution's chain when there are few matrices, by the FP64
// pipe and the sectors of the moved rows when there are many.  One thread per
// column, the triangle's entry loaded before each multiply-add: 41 us for
// 6880 real columns of one matrix, 49 for 64 of order 432, 755 for 4096 of
// order 196 (32-row panels), 26 for 1776 complex columns (16-row panels);
// this form 13.5, 35, 534 and 8.3.
struct LuCols {
  int left;           // columns [0, left)
  int first, right;   // and [first, first + right)
};

template <typename T, int NB, int TC>
__global__ void __launch_bounds__(128) k_laswp_trsm(BOp<T> A, int n, int k0, int nb, const int* ipiv, LuCols cols,
                                                    int trsm_end) {
  using S = TriCols<T, NB, TC>;
  constexpr int R = S::R, CW = 128 / TC;
  __shared__ __align__(16) T tri[NB * NB];
  __shared__ int src[2 * NB], dst[NB], ips[NB];
  const int tid = threadIdx.x;
  T* Ab = A.item(blockIdx.y) + k0;
  const int64_t ld = A.ld;
  if (tid < NB) ips[tid] = tid < nb ? ipiv[(int64_t)blockIdx.y * n + k0 + tid] - k0 : tid;
  if (trsm_end > k0 + nb) {
#pragma unroll
    for (int u = 0; u < NB * NB / 128; ++u) {
      const int e = tid + 128 * u, r = e % NB, c = e / NB;
      tri[S::at(r, c)] = r < nb && c < nb ? Ab[r + (k0 + c) * ld] : T(0.0);
    }
  }
  __syncthreads();
  if (tid < 2 * NB) {
    const int t = tid % NB, p0 = tid < NB ? t : ips[t];
    bool last = true;   // no later interchange names this position (those from nb on are no-ops)
    int pos = p0;
#pragma unroll
    for (int jj = NB - 1; jj >= 0; --jj) {
      const int p = ips[jj];
      if (jj > t && jj < nb && p == p0) last = false;
      pos = pos == jj ? p : pos == p ? jj : pos;
    }
    src[tid] = pos;
    if (tid >= NB) dst[t] = last && p0 >= nb ? p0 : -1;
  }
  __syncthreads();
  const int g = tid % TC, lane0 = tid & 31 & ~(TC - 1);
  const int ncols = cols.left + cols.right;
  for (int t0 = blockIdx.x * CW; t0 < ncols; t0 += gridDim.x * CW) {
    const int t = t0 + tid / TC;
    const bool live = t < ncols;
    const int c = t < cols.left ? t : t - cols.left + cols.first;
    const bool solve = live && c >= k0 + nb && c < trsm_end;
    T* col = Ab + c * ld;
    T x[R], xo[R];
#pragma unroll
    for (int q = 0; q < R; ++q) {
      const int i = g + q * TC;
      x[q] = xo[q] = T(0.0);
      if (live && i < nb) {
        if (solve || src[i] != i) x[q] = col[src[i]];
        if (dst[i] >= 0) xo[q] = col[src[NB + i]];
      }
    }
    __syncwarp();
#pragma unroll
    for (int q = 0; q < R; ++q) {
      const int i = g + q * TC;
      if (live && i < nb && dst[i] >= 0) col[dst[i]] = xo[q];
      xo[q] = x[q];
    }
    if (__any_sync(0xffffffffu, solve)) S::lower(xo, tri, g, lane0, nb);
#pragma unroll
    for (int q = 0; q < R; ++q) {
      const int i = g + q * TC;
      if (live && i < nb && (solve || src[i] != i)) col[i] = solve ? xo[q] : x[q];
    }
  }
}

// perm[i] = the row whose entries the interchanges leave in row i.  Interchange
// j touches rows >= j only, so row i is settled by interchange i; from there
// the row's origin is followed back: an earlier interchange that named the
// current position brought it from row j.  A thread per row, no exchange
// between them.  Bound by the walk of the last rows (replaying the swaps of a
// matrix in one thread took 650 us for 6912 rows; this 147).
__global__ void __launch_bounds__(128) k_ipiv_to_perm(const int* ipiv, int* perm, int n) {
  const int* ip = ipiv + (int64_t)blockIdx.x * n;
  for (int i = blockIdx.y * blockDim.x + threadIdx.x; i < n; i += gridDim.y * blockDim.x) {
    int pos = ip[i];
#pragma unroll 16
    for (int j = min(i | 31, n - 1) - 1; j >= 0; --j) {
      const int p = ip[j];
      if (j < i && p == pos) pos = j;
    }
    perm[(int64_t)blockIdx.x * n + i] = pos;
  }
}

#include "tuned.h"

int& lu_tune(int param) {
  static int v[TUNE_COUNT] = {HPS_TUNED_LU_BASE_PANELS_FEW, HPS_TUNED_LU_BASE_PANELS_MANY,
                              HPS_TUNED_LU_FEW_MIN_N,       HPS_TUNED_LU_CLUSTER_PANEL,
                              HPS_TUNED_TC_MIN_WORK_REAL,   HPS_TUNED_TC_MIN_WORK_CPLX,
                              HPS_TUNED_TC_MIN_K,           HPS_TUNED_TC_CHUNK_MB,
                              HPS_TUNED_TC_PERSIST_MIN_K,   HPS_TUNED_LU_PANEL_NB_FEW};
  return v[param];
}

template <typename T>
int lu_group_size(int n, int batch, int num_sms) {
  const int nb = LuNB<T>::NB;
  // shared memory per CTA limited to ~96 KB for the panel chunk
  const size_t cap = 96 * 1024;
  int gmin = (int)((n * (size_t)nb * sizeof(T) + cap - 1) / cap);
  int G = std::max(1, gmin);
  // spread small batches over more CTAs so that all SMs get work
  int want = (2 * num_sms) / std::max(batch, 1);
  if (want > G) G = want;
  int gmax = std::max(1, n / 64);
  G = std::min(G, gmax);
  // cooperative residency: keep batch * G within one wave
  while (G > 1 && (int64_t)G * batch > 2 * num_sms) --G;
  return std::max(G, 1);
}

template <typename T>
size_t lu_pub_bytes(int n, int batch, int G) {
  if (G <= 1) return 0;
  const int nb = LuNB<T>::NB;
  size_t v = (size_t)batch * 2 * (G + 1) * nb * sizeof(T);
  size_t m = (size_t)batch * 2 * G * sizeof(double);
  size_t r = (size_t)batch * 2 * G * sizeof(int);
  return v + m + r + 256;
}

// Allow the panel kernel the device's whole opt-in shared memory once per
// process.  Setting the attribute per launch to the launch's own size would
// race between host threads that build concurrently (one thread's smaller
// value landing between another's set and launch).
template <typename T, bool COOP>
cudaError_t panel_smem_limit() {
  static const cudaError_t err = [] {
    int dev = 0, mx = 0;
    cudaFuncAttributes fa;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&mx, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
    if (e == cudaSuccess) e = cudaFuncGetAttributes(&fa, k_lu_panel<T, COOP>);
    if (e == cudaSuccess)
      e = cudaFuncSetAttribute(k_lu_panel<T, COOP>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                               mx - (int)fa.sharedSizeBytes);
    if (e != cudaSuccess) cudaGetLastError();
    return e;
  }();
  return err;
}

// Factor the panel A[k0:n, k0:k0+nb).
template <typename T>
static cudaError_t lu_panel(BOp<T> A, int n, int k0, int nb, int batch, int* ipiv, int* info,
                            unsigned* dev_err, int G, const LuWork& w, cudaStream_t st, Prof* pf) {
  constexpr double F = fma_flops<T>();
  const int nb0 = LuNB<T>::NB;
  cudaError_t e;
  const int rows = n - k0;
  int Gk = std::min(G, std::max(1, rows / 8));
  const int ch = (rows + Gk - 1) / Gk;
  size_t sm = ((size_t)ch * nb + 2 * nb) * sizeof(T);
  double pfl = 0.0;  // panel: rank-1 updates and multipliers (FMA-equivalents)
  for (int jj = 0; jj < nb; ++jj) {
    const double below = (double)(n - (k0 + jj) - 1);
    pfl += below * (nb - jj - 1) + below;
  }
  pfl *= F * batch;
  // one row per thread (CR CTAs a matrix) up to 512 rows a CTA; taller panels
  // in a cluster's shared memory (CS) or a cooperative group
  const int CR = lu_tune(TUNE_LU_CLUSTER_PANEL) ? panel_reg_size<T>(rows, batch) : 0;
  const int CS = (CR == 0 && Gk > 1 && lu_tune(TUNE_LU_CLUSTER_PANEL)) ? panel_cluster_size<T>(rows, nb, batch) : 0;
  if (pf) {
    pf->begin(st);
    pf->note(rows, nb, CR > 0 ? CR : CS > 1 ? CS : Gk, batch);  // k: CTAs per matrix
  }
  if (CR > 0) {
    const int rw = ((rows + CR - 1) / CR + 31) / 32;   // row warps
    const int ct = rw == 1 ? 4 : rw == 2 ? 2 : 1;      // column groups: a warp for every scheduler
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(batch * CR);
    cfg.blockDim = dim3(32 * rw * ct);
    cfg.dynamicSmemBytes = panel_reg_smem<T>(32 * rw, CR);
    cfg.stream = st;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = CR;
    at[0].val.clusterDim.y = 1;
    at[0].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = CR > 1 ? 1 : 0;
    e = ct == 4 ? launch_panel_reg<T, 4>(cfg, CR, A, n, k0, nb, ipiv, info, dev_err)
        : ct == 2 ? launch_panel_reg<T, 2>(cfg, CR, A, n, k0, nb, ipiv, info, dev_err)
                  : launch_panel_reg<T, 1>(cfg, CR, A, n, k0, nb, ipiv, info, dev_err);
    if (e != cudaSuccess) return e;
  } else if (CS > 1) {
    // the panel in the distributed shared memory of a cluster per matrix
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(batch * CS);
    cfg.blockDim = dim3(256);
    cfg.dynamicSmemBytes = panel_cluster_smem<T>(rows, nb, CS);
    cfg.stream = st;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = CS;
    at[0].val.clusterDim.y = 1;
    at[0].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    e = cudaLaunchKernelEx(&cfg, k_lu_panel_cluster<T>, A, n, k0, nb, ipiv, info);
    if (e != cudaSuccess) return e;
  } else if (Gk > 1) {
    T* pubv = reinterpret_cast<T*>(w.pub);
    double* pubm = reinterpret_cast<double*>(pubv + (size_t)batch * 2 * (G + 1) * nb0);
    int* pubr = reinterpret_cast<int*>(pubm + (size_t)batch * 2 * G);
    if ((e = panel_smem_limit<T, true>()) != cudaSuccess) return e;
    BOp<T> Aa = A;
    int nn = n, kk = k0, nbb = nb, GG = Gk;
    unsigned* bars = w.bars;
    void* args[] = {&Aa, &nn, &kk, &nbb, &GG, &ipiv, &info, &bars, &pubv, &pubm, &pubr, &dev_err};
    e = cudaLaunchCooperativeKernel((void*)k_lu_panel<T, true>, dim3(batch * Gk), dim3(256), args, sm, st);
    if (e != cudaSuccess) return e;
  } else {
    if ((e = panel_smem_limit<T, false>()) != cudaSuccess) return e;
    k_lu_panel<T, false><<<batch, 256, sm, st>>>(A, n, k0, nb, 1, ipiv, info, nullptr, nullptr, nullptr,
                                                 nullptr, dev_err);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
  }
  if (pf) pf->end(K_LU_PANEL, pfl, st);
  return cudaSuccess;
}

// Apply the interchanges of the panel at k0 to the columns `cols` (none of them
// the panel's) and solve U12 = L11^{-1} A12 for those in [k0 + nb, trsm_end).
template <typename T>
static cudaError_t lu_swap(BOp<T> A, int n, int k0, int nb, LuCols cols, int trsm_end, int batch, const int* ipiv,
                           cudaStream_t st, Prof* pf) {
  const int ncols = cols.left + cols.right;
  if (ncols <= 0) return cudaSuccess;
  // eight threads per column have the shortest chain; four issue an eighth
  // less once the FP64 pipe is full whatever the split (4096 matrices of
  // order 196: 534 us against 570; 1024 of order 224: 108 against 103)
  const bool many = (int64_t)((ncols + 31) / 32) * batch >= 48 * device_sms();
  const int cw = many ? 32 : 16;
  const dim3 grid(std::min((ncols + cw - 1) / cw, 4096), batch);
  if (pf) {
    pf->begin(st);
    pf->note(nb, ncols, nb, batch);
  }
  if (many) k_laswp_trsm<T, LuNB<T>::NB, 4><<<grid, 128, 0, st>>>(A, n, k0, nb, ipiv, cols, trsm_end);
  else k_laswp_trsm<T, LuNB<T>::NB, 8><<<grid, 128, 0, st>>>(A, n, k0, nb, ipiv, cols, trsm_end);
  const int solved = std::max(0, std::min(trsm_end, cols.first + cols.right) - cols.first);
  if (pf) pf->end(K_LASWP_TRSM, fma_flops<T>() * 0.5 * nb * (nb - 1) * (double)solved * batch, st);
  return cudaGetLastError();
}

// A[k0 + nb : n, j0 : j0 + nj) -= A[k0 + nb : n, panel] U12, leaving spare SMs
template <typename T>
static cudaError_t lu_update(BOp<T> A, int n, int k0, int nb, int j0, int nj, int spare, int batch, cudaStream_t st,
                             Prof* pf) {
  if (n - k0 - nb <= 0 || nj <= 0) return cudaSuccess;
  GemmArgs<T> g;
  g.M = n - k0 - nb; g.N = nj; g.K = nb; g.batch = batch;
  g.A = shifted(A, (int64_t)(k0 + nb) + (int64_t)k0 * A.ld);
  g.B = shifted(A, (int64_t)k0 + (int64_t)j0 * A.ld);
  g.C = shifted(A, (int64_t)(k0 + nb) + (int64_t)j0 * A.ld);
  g.alpha = T(-1.0); g.beta = T(1.0);
  g.spare_sms = spare;
  return gemm(g, st, pf);
}

// SMs that the next panels of `batch` matrices (of `rows` rows) take when they
// are factored beside the rest of the update (rows x cols, inner dimension nb), or
// 0 when they are not.  Splitting the update costs two short launches and
// two events a panel (~20 us), so the rest has to be worth hiding: from 2e6
// multiply-adds on (builds at 2e6 / 5e6 / 1e7 / 2e7 / never: Helmholtz 93.1 /
// 93.5 / 93.6 / 94.0 / 94.7 ms, adaptive 71.4 / 71.7 / 71.9 / 72.0 / 73.5, 3D elliptic 76.3 at
// all of them / 82.0).  Panels on more than half of the SMs leave the update
// too few (on up to all: Helmholtz 95.3, 3D elliptic 80.6).
template <typename T>
int panel_ahead_sms(int rows, int cols, int nb, int batch) {
  if (cols <= 0 || (double)rows * cols * nb * batch < 2e6 || batch > device_sms() / 2) return 0;
  const int cr = lu_tune(TUNE_LU_CLUSTER_PANEL) ? panel_reg_size<T>(rows, batch) : 0;
  return cr > 0 && (int64_t)cr * batch <= device_sms() / 2 ? cr * batch : 0;
}

namespace {

// A second stream for the panels that are factored ahead of the trailing
// updates, with the events that order it against the caller's stream.  Idle
// ones are kept (at most kSideKeep a device; lu_side_trim destroys them): making
// one takes tens of microseconds.  A released one is joined to the stream
// that used it, so its next user inherits no hazard, at worst a short wait.
struct SideStream {
  cudaStream_t st = nullptr;
  cudaEvent_t fork = nullptr, join = nullptr;
  int dev = 0;
  void destroy() {
    if (fork) cudaEventDestroy(fork);
    if (join) cudaEventDestroy(join);
    if (st) cudaStreamDestroy(st);
    st = nullptr;
  }
};
constexpr size_t kSideKeep = 8;
std::mutex g_side_mu;
std::vector<SideStream> g_side;

bool side_take(SideStream* out) {
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) return cudaGetLastError(), false;
  {
    std::lock_guard<std::mutex> lk(g_side_mu);
    for (size_t i = 0; i < g_side.size(); ++i)
      if (g_side[i].dev == dev) {
        *out = g_side[i];
        g_side.erase(g_side.begin() + i);
        return true;
      }
  }
  SideStream s;
  s.dev = dev;
  int lo = 0, hi = 0;
  // the highest priority: a waiting panel takes the first SMs that come free
  if (cudaDeviceGetStreamPriorityRange(&lo, &hi) != cudaSuccess ||
      cudaStreamCreateWithPriority(&s.st, cudaStreamNonBlocking, hi) != cudaSuccess ||
      cudaEventCreateWithFlags(&s.fork, cudaEventDisableTiming) != cudaSuccess ||
      cudaEventCreateWithFlags(&s.join, cudaEventDisableTiming) != cudaSuccess) {
    cudaGetLastError();
    s.destroy();
    return false;
  }
  *out = s;
  return true;
}

void side_give(SideStream s) {
  {
    std::lock_guard<std::mutex> lk(g_side_mu);
    size_t kept = 0;
    for (const SideStream& o : g_side) kept += o.dev == s.dev;
    if (kept < kSideKeep) {
      g_side.push_back(s);
      return;
    }
  }
  s.destroy();
}

}  // namespace

// Destroy the current device's idle side streams.
void lu_side_trim() {
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) {
    cudaGetLastError();
    return;
  }
  std::lock_guard<std::mutex> lk(g_side_mu);
  for (size_t i = g_side.size(); i-- > 0;)
    if (g_side[i].dev == dev) {
      g_side[i].destroy();
      g_side.erase(g_side.begin() + i);
    }
}

// The blocked factorisation of one range with its panels ahead: panel k + 1
// needs only its own columns of panel k's update, so those are done first and
// the panel is factored on the side stream while the rest of the update
// runs (on the SMs that the panel leaves: a tensor-core product has one CTA per
// SM for its whole duration, which a late panel would wait for and an early
// one would stretch).  A panel of few matrices is a serial chain on a few SMs
// (115 us for 6912 rows on 16); the update of the others takes as long.  The same
// operations on the same entries; only where a product runs may change, as
// the two parts of an update are routed by their own sizes.
struct LookAhead {
  cudaStream_t main;
  SideStream side;
  bool tried = false, open = false;   // open: work on the side stream that main has not waited for
  explicit LookAhead(cudaStream_t st) : main(st) {}
  ~LookAhead() {
    if (open) wait();
    if (side.st) side_give(side);
  }
  bool available() {
    if (!tried) {
      tried = true;
      // a stream that is being captured would take the side stream, and whoever
      // takes it next, into the capture
      if (!stream_capturing(main)) side_take(&side);
    }
    return side.st != nullptr;
  }
  cudaError_t begin() {   // side waits for main
    cudaError_t e = cudaEventRecord(side.fork, main);
    return e != cudaSuccess ? e : cudaStreamWaitEvent(side.st, side.fork, 0);
  }
  cudaError_t end() {
    open = true;
    return cudaEventRecord(side.join, side.st);
  }
  cudaError_t wait() {   // main waits for side
    open = false;
    return cudaStreamWaitEvent(main, side.join, 0);
  }
};

template <typename T>
static cudaError_t rtrsm_lower(BOp<T> LU, BOp<T> X, int p0, int n1, int nrhs, int batch, cudaStream_t st,
                               Prof* pf);

// Recursive LU with partial pivoting of the columns [c0, c1) (rows c0..n):
// factor the left half, U12 = L11^{-1} A12 by the recursive triangular
// solve, A22 -= A21 U12 as one product of inner dimension ~(c1 - c0) / 2,
// factor the right half.  Ranges of at most base_w columns are factored blocked
// right-looking (panel, interchanges + U12 within the range, update of the
// range's remaining columns), which has fewer launches; so are whole matrices
// when there are few of them (base_w = n).  The same pivots and operations as
// the blocked right-looking order; of larger matrices the bulk of the trailing
// updates becomes a few large-K products instead of n / nb products of inner
// dimension nb.
template <typename T>
static cudaError_t rgetrf(BOp<T> A, int n, int c0, int c1, int base_w, int nb0, int batch, int* ipiv, int* info,
                          unsigned* dev_err, int G, const LuWork& w, cudaStream_t st, Prof* pf) {
  const int wdt = c1 - c0;
  cudaError_t e;
  if (wdt <= base_w) {
    LookAhead la(st);
    for (int k0 = c0; k0 < c1; k0 += nb0) {
      const int nb = std::min(nb0, c1 - k0), k1 = k0 + nb, nb1 = std::min(nb0, c1 - k1);
      if (la.open) e = la.wait();
      else e = lu_panel<T>(A, n, k0, nb, batch, ipiv, info, dev_err, G, w, st, pf);
      if (e != cudaSuccess) return e;
      const int sms = panel_ahead_sms<T>(n - k1, c1 - k1 - nb1, nb, batch);
      if (sms == 0 || !la.available()) {
        if ((e = lu_swap<T>(A, n, k0, nb, LuCols{k0, k1, n - k1}, c1, batch, ipiv, st, pf)) != cudaSuccess) return e;
        if ((e = lu_update<T>(A, n, k0, nb, k1, c1 - k1, 0, batch, st, pf)) != cudaSuccess) return e;
        continue;
      }
      const int k2 = k1 + nb1;
      if ((e = lu_swap<T>(A, n, k0, nb, LuCols{0, k1, nb1}, c1, batch, ipiv, st, pf)) != cudaSuccess) return e;
      if ((e = lu_update<T>(A, n, k0, nb, k1, nb1, 0, batch, st, pf)) != cudaSuccess) return e;
      if ((e = la.begin()) != cudaSuccess) return e;
      e = lu_panel<T>(A, n, k1, nb1, batch, ipiv, info, dev_err, G, w, la.side.st, pf);
      const cudaError_t e2 = la.end();
      if (e != cudaSuccess || e2 != cudaSuccess) return e != cudaSuccess ? e : e2;
      if ((e = lu_swap<T>(A, n, k0, nb, LuCols{k0, k2, n - k2}, c1, batch, ipiv, st, pf)) != cudaSuccess) return e;
      if ((e = lu_update<T>(A, n, k0, nb, k2, c1 - k2, sms, batch, st, pf)) != cudaSuccess) return e;
    }
    return cudaSuccess;
  }
  const int cm = c0 + ((wdt / 2 + nb0 - 1) / nb0) * nb0;
  if ((e = rgetrf<T>(A, n, c0, cm, base_w, nb0, batch, ipiv, info, dev_err, G, w, st, pf)) != cudaSuccess) return e;
  // U12: rows [c0, cm), columns [cm, c1)
  BOp<T> L11 = shifted(A, (int64_t)c0 + (int64_t)c0 * A.ld);
  BOp<T> A12 = shifted(A, (int64_t)c0 + (int64_t)cm * A.ld);
  if ((e = rtrsm_lower<T>(L11, A12, 0, cm - c0, c1 - cm, batch, st, pf)) != cudaSuccess) return e;
  if (n > cm) {
    GemmArgs<T> g;
    g.M = n - cm; g.N = c1 - cm; g.K = cm - c0; g.batch = batch;
    g.A = shifted(A, (int64_t)cm + (int64_t)c0 * A.ld);
    g.B = A12;
    g.C = shifted(A, (int64_t)cm + (int64_t)cm * A.ld);
    g.alpha = T(-1.0); g.beta = T(1.0);
    if ((e = gemm(g, st, pf)) != cudaSuccess) return e;
  }
  return rgetrf<T>(A, n, cm, c1, base_w, nb0, batch, ipiv, info, dev_err, G, w, st, pf);
}

template <typename T>
cudaError_t getrf(BOp<T> A, int n, int batch, int* ipiv, int* perm, int* info, unsigned* dev_err,
                  int G, const LuWork& w, cudaStream_t st, Prof* pf) {
  if (n <= 0 || batch <= 0) return cudaSuccess;
  cudaError_t e;
  // Few matrices: the recursion's triangular solves become many small
  // launches on a few SMs, so small orders keep the blocked right-looking
  // order (one fused interchange + U12 launch per panel); large ones recurse
  // so that the trailing updates are a few large-K products.
  const int nbp = LuNB<T>::NB;
  int base_w = lu_tune(TUNE_LU_BASE_PANELS_MANY) * nbp;
  // panel width: the kernels' maximum, or narrower for few matrices (the
  // panel's FP64 update, ~n^2 nb / 2 multiply-adds on the few SMs of a
  // cluster, against twice the panels and trailing updates of half the K)
  int pnb = nbp;
  if (batch < 8) {
    const int bp = lu_tune(TUNE_LU_BASE_PANELS_FEW);
    base_w = (bp <= 0 || n < lu_tune(TUNE_LU_FEW_MIN_N)) ? n : bp * nbp;
    pnb = std::max(8, std::min(nbp, lu_tune(TUNE_LU_PANEL_NB_FEW) / 8 * 8));
  }
  if (base_w < nbp) base_w = nbp;
  if ((e = rgetrf<T>(A, n, 0, n, base_w, pnb, batch, ipiv, info, dev_err, G, w, st, pf)) != cudaSuccess) return e;
  if (pf) pf->begin(st);
  k_ipiv_to_perm<<<dim3(batch, std::min((n + 127) / 128, 65535)), 128, 0, st>>>(ipiv, perm, n);
  if (pf) pf->end(K_OTHER, 0.0, st);
  return cudaGetLastError();
}

// ------------------------------------------------------ triangular solve ----

template <typename T>
__global__ void __launch_bounds__(256) k_permute_rows(BOp<T> src, BOp<T> dst, const int* perm, int n, int nrhs, int batch) {
  for_tile(n, nrhs, batch, [&](int64_t b, int i, int j) {
    dst.item((int)b)[i + (int64_t)j * dst.ld] = src.item((int)b)[perm[b * n + i] + (int64_t)j * src.ld];
  });
}

template <typename T>
cudaError_t permute_rows(BOp<T> src, BOp<T> dst, const int* perm, int n, int nrhs, int batch,
                         cudaStream_t st, Prof* pf) {
  if (n <= 0 || nrhs <= 0 || batch <= 0) return cudaSuccess;
  if (pf) pf->begin(st);
  k_permute_rows<T><<<tile_grid(n, nrhs, batch), 256, 0, st>>>(src, dst, perm, n, nrhs, batch);
  if (pf) pf->end(K_GATHER, 0.0, st);
  return cudaGetLastError();
}

// Diagonal-block solve: X[p0:p0+pb, :] <- L[p0:p0+pb, p0:p0+pb]^{-1} X (unit
// lower, UPPER = false) or U^{-1} X (non-unit upper, UPPER = true).  One warp
// per right-hand side column, lane r owning row r (pb <= 32): each step
// broadcasts the solved entry with a shuffle and the lanes below (above)
// update their row, so a single column is solved in pb dependent steps.

template <typename T, bool UPPER>
__global__ void __launch_bounds__(128) k_trsm_diag(BOp<T> LU, BOp<T> X, int p0, int pb, int nrhs, int batch) {
  extern __shared__ unsigned char smem_raw[];
  T* Ls = reinterpret_cast<T*>(smem_raw);  // pb x pb, then pb reciprocals of the diagonal
  T* Dinv = Ls + pb * pb;
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, nw = blockDim.x >> 5;
  for (int b = blockIdx.y; b < batch; b += gridDim.y) {
    const T* Lb = LU.item(b);
    T* Xb = X.item(b);
    __syncthreads();
    for (int e = threadIdx.x; e < pb * pb; e += blockDim.x) {
      int r = e % pb, c = e / pb;
      Ls[e] = Lb[(int64_t)(p0 + r) + (int64_t)(p0 + c) * LU.ld];
    }
    __syncthreads();
    if (UPPER)
      for (int r = threadIdx.x; r < pb; r += blockDim.x) {
        const T d = Ls[r + r * pb];
        Dinv[r] = is_zero(d) ? T(0.0) : recip(d);
      }
    __syncthreads();
    for (int j = blockIdx.x * nw + wid; j < nrhs; j += gridDim.x * nw) {
      T* col = Xb + (int64_t)j * X.ld + p0;
      T x = lane < pb ? col[lane] : T(0.0);
      if (!UPPER) {
        for (int c = 0; c < pb - 1; ++c) {
          const T xc = shfl_val(x, c);
          if (lane > c && lane < pb) x = fmsc(x, Ls[lane + c * pb], xc);
        }
      } else {
        for (int c = pb - 1; c >= 0; --c) {
          if (lane == c) x = x * Dinv[c];
          const T xc = shfl_val(x, c);
          if (lane < c) x = fmsc(x, Ls[lane + c * pb], xc);
        }
      }
      if (lane < pb) col[lane] = x;
    }
  }
}

// Many right-hand sides: one thread per column, the block's pb x pb diagonal
// block staged once in shared memory for up to 128 columns.
template <typename T, bool UPPER>
__global__ void __launch_bounds__(128) k_trsm_diag_cols(BOp<T> LU, BOp<T> X, int p0, int pb, int nrhs, int batch) {
  extern __shared__ unsigned char smem_raw[];
  T* Ls = reinterpret_cast<T*>(smem_raw);
  T* Dinv = Ls + pb * pb;
  for (int b = blockIdx.y; b < batch; b += gridDim.y) {
    const T* Lb = LU.item(b);
    T* Xb = X.item(b);
    __syncthreads();
    for (int e = threadIdx.x; e < pb * pb; e += blockDim.x) {
      int r = e % pb, c = e / pb;
      Ls[e] = Lb[(int64_t)(p0 + r) + (int64_t)(p0 + c) * LU.ld];
    }
    __syncthreads();
    if (UPPER)
      for (int r = threadIdx.x; r < pb; r += blockDim.x) {
        const T d = Ls[r + r * pb];
        Dinv[r] = is_zero(d) ? T(0.0) : recip(d);
      }
    __syncthreads();
    for (int j = blockIdx.x * blockDim.x + threadIdx.x; j < nrhs; j += gridDim.x * blockDim.x) {
      T* col = Xb + (int64_t)j * X.ld + p0;
      T x[32];
      for (int r = 0; r < pb; ++r) x[r] = col[r];
      if (!UPPER) {
        for (int r = 1; r < pb; ++r) {
          T s = x[r];
          for (int c = 0; c < r; ++c) s = fmsc(s, Ls[r + c * pb], x[c]);
          x[r] = s;
        }
      } else {
        for (int r = pb - 1; r >= 0; --r) {
          T s = x[r];
          for (int c = r + 1; c < pb; ++c) s = fmsc(s, Ls[r + c * pb], x[c]);
          x[r] = s * Dinv[r];
        }
      }
      for (int r = 0; r < pb; ++r) col[r] = x[r];
    }
  }
}

// Diagonal blocks of 32 rows (or fewer, padded), TC threads per right-hand
// side (tri_cols.h); a thread's loads of its column are in flight while the
// block is staged.  Bound by the FP64 pipe with many columns, by the chain of
// 32 steps with few.  Against one thread per column that loads each entry
// before its multiply-add (lower / upper, us): 865 real columns of one matrix
// 18 / 19 -> 8 / 10, 865 of 64 matrices 55 / 80 -> 57 / 66, 114 of 4096
// 434 / 600 -> 447 / 472; 1793 complex columns of 4 matrices 74 / 78 -> 35 / 49, 225 of 256
// 251 / 270 -> 231 / 268.
template <typename T, bool UPPER, int TC>
__global__ void __launch_bounds__(128) k_trsm32(BOp<T> LU, BOp<T> X, int p0, int pb, int nrhs) {
  using S = TriCols<T, 32, TC>;
  __shared__ __align__(16) T tri[32 * 32];
  __shared__ T dinv[32];
  const int b = blockIdx.y, tid = threadIdx.x, nt = blockDim.x, lane = tid & 31;
  const T* Lb = LU.item(b) + p0 + (int64_t)p0 * LU.ld;
  const int j = blockIdx.x * (nt / TC) + tid / TC, g = tid % TC;
  const bool live = j < nrhs;
  T* col = X.item(b) + p0 + (int64_t)j * X.ld;
  T x[S::R];
#pragma unroll
  for (int q = 0; q < S::R; ++q) x[q] = live && g + q * TC < pb ? col[g + q * TC] : T(0.0);
#pragma unroll 8
  for (int c = tid >> 5; c < 32; c += nt >> 5) tri[S::at(lane, c)] = lane < pb && c < pb ? Lb[lane + (int64_t)c * LU.ld] : T(0.0);
  if (UPPER && tid < 32) {
    const T d = tid < pb ? Lb[tid + (int64_t)tid * LU.ld] : T(0.0);
    dinv[tid] = is_zero(d) ? T(0.0) : recip(d);
  }
  __syncthreads();
  if (blockIdx.x * (nt / TC) + (tid & ~31) / TC >= nrhs) return;   // a warp without columns
  const int lane0 = lane & ~(TC - 1);
  if (UPPER) S::upper(x, tri, dinv, g, lane0, 32);
  else S::lower(x, tri, g, lane0, 32);
#pragma unroll
  for (int q = 0; q < S::R; ++q)
    if (live && g + q * TC < pb) col[g + q * TC] = x[q];
}

// Threads per right-hand side of k_trsm32, or 0 for k_trsm_diag_cols.
//
// A warp's FP64 instructions per column set are known (496 multiply-adds for
// 32 rows in one thread, 256, 136 and 76 in each of 2, 4 and 8; the upper
// triangle scales once per row in every thread), and every scheduler issues one
// in 64 cycles, so the time goes with the fullest scheduler's warps times
// that count: few columns take 8 threads, many take the form that issues least in
// all.  Loads that one warp per scheduler does not hide put the counts below
// at 540 and 572 for one thread; the upper triangle's longer chain makes 4 and 8 threads
// count 200 and 130.  Blocks of less than 32 rows are padded, which
// costs pipe time, so they come here only while one wave of warps holds all columns.
template <bool UPPER>
int trsm32_threads(int pb, int nrhs, int batch) {
  const int count[4] = {UPPER ? 572 : 540, UPPER ? 288 : 256, UPPER ? 200 : 136, UPPER ? 130 : 76};
  const int64_t slots = 4 * device_sms();
  if (pb < 32 && (int64_t)((nrhs * 8 + 31) / 32) * batch > slots) return 0;
  int best = 0;
  int64_t least = 0;
  for (int i = 3; i >= 0; --i) {
    const int64_t warps = (int64_t)(((int64_t)nrhs * (1 << i) + 31) / 32) * batch;
    const int64_t t = (warps + slots - 1) / slots * count[i];
    if (!best || t < least) best = 1 << i, least = t;
  }
  return best;
}

template <typename T, bool UPPER>
cudaError_t trsm_diag(BOp<T> LU, BOp<T> X, int p0, int pb, int nrhs, int batch, cudaStream_t st) {
  const size_t sm = ((size_t)pb * pb + pb) * sizeof(T);
  const int by = std::min(batch, 65535);
  const int tc = nrhs >= 16 && batch <= 65535 ? trsm32_threads<UPPER>(pb, nrhs, batch) : 0;
  if (tc) {
    const int nt = 32 * std::min(4, (nrhs * tc + 31) / 32);
    const dim3 grid((nrhs + nt / tc - 1) / (nt / tc), batch);
    if (tc == 1) k_trsm32<T, UPPER, 1><<<grid, nt, 0, st>>>(LU, X, p0, pb, nrhs);
    else if (tc == 2) k_trsm32<T, UPPER, 2><<<grid, nt, 0, st>>>(LU, X, p0, pb, nrhs);
    else if (tc == 4) k_trsm32<T, UPPER, 4><<<grid, nt, 0, st>>>(LU, X, p0, pb, nrhs);
    else k_trsm32<T, UPPER, 8><<<grid, nt, 0, st>>>(LU, X, p0, pb, nrhs);
  } else if (nrhs >= 16) {
    const int bx = std::min((nrhs + 127) / 128, 1024);
    k_trsm_diag_cols<T, UPPER><<<dim3(bx, by), 128, sm, st>>>(LU, X, p0, pb, nrhs, batch);
  } else {
    const int bx = std::min((nrhs + 3) / 4, 1024);
    k_trsm_diag<T, UPPER><<<dim3(bx, by), 128, sm, st>>>(LU, X, p0, pb, nrhs, batch);
  }
  return cudaGetLastError();
}

// Recursive triangular solves on rows [p0, p0 + n1) of X: split at a
// multiple of 32 near the middle, solve the first half, update the second
// with one product of inner dimension ~n1/2, solve the second half; 32-row
// diagonal blocks at the leaves.  Same operations as the blocked
// right-looking order, but the updates are few large-K products (the bulk
// runs on the tensor cores) instead of n/32 products of inner dimension 32
// that each re-read the rest of X.
template <typename T>
static cudaError_t rtrsm_lower(BOp<T> LU, BOp<T> X, int p0, int n1, int nrhs, int batch, cudaStream_t st,
                               Prof* pf) {
  constexpr double F = fma_flops<T>();
  cudaError_t e;
  if (n1 <= 32) {
    if (pf) {
      pf->begin(st);
      pf->note(n1, nrhs, n1, batch);
    }
    if ((e = trsm_diag<T, false>(LU, X, p0, n1, nrhs, batch, st)) != cudaSuccess) return e;
    if (pf) pf->end(K_TRSM_DIAG, F * 0.5 * n1 * (n1 - 1) * (double)nrhs * batch, st);
    return cudaSuccess;
  }
  const int h = ((n1 / 2 + 31) / 32) * 32;
  if ((e = rtrsm_lower<T>(LU, X, p0, h, nrhs, batch, st, pf)) != cudaSuccess) return e;
  GemmArgs<T> g;
  g.M = n1 - h; g.N = nrhs; g.K = h; g.batch = batch;
  g.A = shifted(LU, (int64_t)(p0 + h) + (int64_t)p0 * LU.ld);
  g.B = shifted(X, (int64_t)p0);
  g.C = shifted(X, (int64_t)(p0 + h));
  g.alpha = T(-1.0); g.beta = T(1.0);
  if ((e = gemm(g, st, pf)) != cudaSuccess) return e;
  return rtrsm_lower<T>(LU, X, p0 + h, n1 - h, nrhs, batch, st, pf);
}

template <typename T>
static cudaError_t rtrsm_upper(BOp<T> LU, BOp<T> X, int p0, int n1, int nrhs, int batch, cudaStream_t st,
                               Prof* pf) {
  constexpr double F = fma_flops<T>();
  cudaError_t e;
  if (n1 <= 32) {
    if (pf) {
      pf->begin(st);
      pf->note(n1, nrhs, n1, batch);
    }
    if ((e = trsm_diag<T, true>(LU, X, p0, n1, nrhs, batch, st)) != cudaSuccess) return e;
    if (pf) pf->end(K_TRSM_DIAG, F * (0.5 * n1 * (n1 - 1) + n1) * (double)nrhs * batch, st);
    return cudaSuccess;
  }
  const int h = ((n1 / 2 + 31) / 32) * 32;
  if ((e = rtrsm_upper<T>(LU, X, p0 + h, n1 - h, nrhs, batch, st, pf)) != cudaSuccess) return e;
  GemmArgs<T> g;
  g.M = h; g.N = nrhs; g.K = n1 - h; g.batch = batch;
  g.A = shifted(LU, (int64_t)p0 + (int64_t)(p0 + h) * LU.ld);
  g.B = shifted(X, (int64_t)(p0 + h));
  g.C = shifted(X, (int64_t)p0);
  g.alpha = T(-1.0); g.beta = T(1.0);
  if ((e = gemm(g, st, pf)) != cudaSuccess) return e;
  return rtrsm_upper<T>(LU, X, p0, h, nrhs, batch, st, pf);
}

template <typename T>
cudaError_t getrs_inplace(BOp<T> LU, int n, BOp<T> X, int nrhs, int batch, cudaStream_t st,
                          Prof* pf, TrsvInv* inv) {
  if (n <= 0 || nrhs <= 0 || batch <= 0) return cudaSuccess;
  if (trsv_few_applicable<T>(n, nrhs, batch, inv))
    return trsv_few<T>(LU, n, X, nrhs, batch, false, inv, st, pf);
  cudaError_t e;
  // forward: unit lower; backward: non-unit upper
  if ((e = rtrsm_lower<T>(LU, X, 0, n, nrhs, batch, st, pf)) != cudaSuccess) return e;
  return rtrsm_upper<T>(LU, X, 0, n, nrhs, batch, st, pf);
}

// --------------------------------------------- flag-ordered solve ----
//
// Triangular solve of a single large factor with few right-hand sides.  The
// blocked getrs issues two launches per 32 rows, each far too small to fill
// the GPU; here one launch per triangle walks the 32-row blocks in dependency
// order (forward: first to last; backward: last to first).  CTA c takes the
// logical blocks c, c + G, c + 2G, ... in increasing order.  For each, all
// eight warps subtract the contributions of the earlier blocks as their
// solutions are published, warp w taking columns 4w .. 4w + 3 of every
// earlier block (each warp loads its matrix entries before it waits, and the
// FP64 work of one 32 x 32 block is spread over the whole SM); the block's
// solution is then the product of the precomputed inverse of its 32 x 32
// diagonal block (k_diag_block_inv) with the reduced right-hand side, split
// the same way.  The launch is cooperative, so every CTA is resident, and the
// earliest unfinished block depends only on finished ones: the walk always
// makes progress.  Waits are bounded: on timeout the flag error word is set
// and the block proceeds (wrong values, but the launch ends).
template <typename T, int NR, bool UPPER>
__global__ void __launch_bounds__(256) k_trsv_flags(const T* __restrict__ LU, int ld, int n, T* X, int ldx,
                                                   int nrhs, const T* __restrict__ dinv, unsigned* flags,
                                                   unsigned epoch, volatile int* err) {
  __shared__ T part[8][NR][32];
  __shared__ T y[NR][32];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const int nblk = (n + 31) / 32;
  for (int t = blockIdx.x; t < nblk; t += gridDim.x) {
    const int j = UPPER ? nblk - 1 - t : t;
    const int r = j * 32 + lane;
    const bool rv = r < n;
    T acc[NR];
#pragma unroll
    for (int c = 0; c < NR; ++c) acc[c] = T(0.0);
    for (int tp = 0; tp < t; ++tp) {
      const int i = UPPER ? nblk - 1 - tp : tp;
      const int qn = min(32, n - i * 32);
      T a[4];
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        const int q = 4 * w + k;
        a[k] = (rv && q < qn) ? LU[(int64_t)r + (int64_t)(i * 32 + q) * ld] : T(0.0);
      }
      if (lane == 0) {
        if (!wait_flag(flags + i, epoch, 1ull << 24)) *err = 1;
        __threadfence();
      }
      __syncwarp();
      T xi[NR];
#pragma unroll
      for (int c = 0; c < NR; ++c) {
        const int q = 4 * w + lane;
        xi[c] = (lane < 4 && q < qn && c < nrhs) ? ld_cg(X + (int64_t)(i * 32 + q) + (int64_t)c * ldx) : T(0.0);
      }
#pragma unroll
      for (int k = 0; k < 4; ++k)
#pragma unroll
        for (int c = 0; c < NR; ++c) acc[c] = fmsc(acc[c], a[k], shfl_val(xi[c], k));
    }
#pragma unroll
    for (int c = 0; c < NR; ++c) part[w][c][lane] = acc[c];
    __syncthreads();
    if (w == 0) {
#pragma unroll
      for (int c = 0; c < NR; ++c) {
        T sum = (rv && c < nrhs) ? X[r + (int64_t)c * ldx] : T(0.0);
        for (int k = 0; k < 8; ++k) sum = sum + part[k][c][lane];
        y[c][lane] = sum;
      }
    }
    __syncthreads();
    // x_j = inv(diagonal block j) y, the inverse column-major 32 x 32
    const T* Dj = dinv + (int64_t)j * 1024;
    T acc2[NR];
#pragma unroll
    for (int c = 0; c < NR; ++c) acc2[c] = T(0.0);
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      const int q = 4 * w + k;
      const T dq = Dj[lane + 32 * q];
#pragma unroll
      for (int c = 0; c < NR; ++c) acc2[c] = fmac(acc2[c], dq, y[c][q]);
    }
#pragma unroll
    for (int c = 0; c < NR; ++c) part[w][c][lane] = acc2[c];
    __syncthreads();
    if (w == 0) {
#pragma unroll
      for (int c = 0; c < NR; ++c) {
        T xs = T(0.0);
        for (int k = 0; k < 8; ++k) xs = xs + part[k][c][lane];
        if (rv && c < nrhs) X[r + (int64_t)c * ldx] = xs;
      }
      __threadfence();
      __syncwarp();
      if (lane == 0) atomicExch(flags + j, epoch);
    }
    __syncthreads();
  }
}

// Inverses of the 32 x 32 diagonal blocks of an LU factor (column-major,
// 32 x 32 each): tri 0 the unit lower L_jj, tri 1 the upper U_jj; a partial
// last block is completed with the identity, a zero pivot gives a zero row
// of the inverse (a singular factor was reported by the factorisation).
// One CTA per (block, triangle), thread c computes column c by substitution.
template <typename T>
__global__ void __launch_bounds__(32) k_diag_block_inv(const T* __restrict__ LU, int ld, int n, T* out) {
  const int j = blockIdx.x, tri = blockIdx.y, c = threadIdx.x, nblk = gridDim.x;
  const int pb = min(32, n - j * 32);
  const T* Dj = LU + (int64_t)(j * 32) + (int64_t)(j * 32) * ld;
  T x[32];
  if (tri == 0) {
#pragma unroll
    for (int rr = 0; rr < 32; ++rr) {
      T v = rr == c ? T(1.0) : T(0.0);
      if (rr < pb)
        for (int k = 0; k < rr; ++k) v = fmsc(v, Dj[rr + (int64_t)k * ld], x[k]);
      x[rr] = v;
    }
  } else {
#pragma unroll
    for (int rr = 31; rr >= 0; --rr) {
      T v = rr == c ? T(1.0) : T(0.0);
      if (rr < pb) {
        for (int k = rr + 1; k < pb; ++k) v = fmsc(v, Dj[rr + (int64_t)k * ld], x[k]);
        const T d = Dj[rr + (int64_t)rr * ld];
        v = is_zero(d) ? T(0.0) : v * recip(d);
      }
      x[rr] = v;
    }
  }
  T* o = out + ((int64_t)tri * nblk + j) * 1024;
#pragma unroll
  for (int rr = 0; rr < 32; ++rr) o[rr + 32 * c] = x[rr];
}

template <typename T>
bool trsv_flags_applicable(int n, int nrhs, int batch, const TrsvWork& w) {
  return batch == 1 && nrhs >= 1 && nrhs <= 8 && n >= 128 && w.flags && w.dev_err && w.dinv &&
         (n + 31) / 32 <= w.nflags;
}

template <typename T, int NR, bool UPPER>
cudaError_t launch_trsv_flags(const T* LU, int n, int ld, T* X, int ldx, int nrhs, TrsvWork& w,
                              cudaStream_t st) {
  // resident CTAs of this kernel on the whole GPU (thread-safe one-time
  // initialisation; 0 if the query failed)
  static const int resident = [] {
    int dev = 0, sms = 0, per_sm = 0;
    if (cudaGetDevice(&dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess ||
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_trsv_flags<T, NR, UPPER>, 256, 0) !=
            cudaSuccess) {
      cudaGetLastError();
      return 0;
    }
    return per_sm * sms;
  }();
  if (resident <= 0) return cudaErrorInvalidConfiguration;
  const int nblk = (n + 31) / 32;
  const int G = std::max(1, std::min(nblk, resident));
  const unsigned ep = ++w.epoch;
  unsigned* fl = w.flags;
  int* errp = const_cast<int*>(w.dev_err);
  const T* dv = static_cast<const T*>(w.dinv) + (UPPER ? (int64_t)nblk * 1024 : 0);
  void* args[] = {(void*)&LU, &ld, &n, &X, &ldx, &nrhs, (void*)&dv, &fl, (void*)&ep, &errp};
  return cudaLaunchCooperativeKernel((void*)k_trsv_flags<T, NR, UPPER>, dim3(G), dim3(256), args, 0, st);
}

template <typename T, bool UPPER>
cudaError_t trsv_flags_dispatch(const T* LU, int n, int ld, T* X, int ldx, int nrhs, TrsvWork& w,
                                cudaStream_t st) {
  if (nrhs == 1) return launch_trsv_flags<T, 1, UPPER>(LU, n, ld, X, ldx, nrhs, w, st);
  if (nrhs == 2) return launch_trsv_flags<T, 2, UPPER>(LU, n, ld, X, ldx, nrhs, w, st);
  if (nrhs <= 4) return launch_trsv_flags<T, 4, UPPER>(LU, n, ld, X, ldx, nrhs, w, st);
  return launch_trsv_flags<T, 8, UPPER>(LU, n, ld, X, ldx, nrhs, w, st);
}

template <typename T>
cudaError_t getrs_flags(const T* LU, int n, int ld, T* X, int ldx, int nrhs, TrsvWork& w, cudaStream_t st,
                        Prof* pf) {
  constexpr double F = fma_flops<T>();
  cudaError_t e;
  if (!w.dinv_ready) {
    // the diagonal blocks' inverses, once per factor (its storage was sized
    // with the flags)
    if (pf) pf->begin(st);
    k_diag_block_inv<T><<<dim3((n + 31) / 32, 2), 32, 0, st>>>(LU, ld, n, static_cast<T*>(w.dinv));
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    if (pf) pf->end(K_OTHER, 0.0, st);
    w.dinv_ready = true;
  }
  if (pf) {
    pf->begin(st);
    pf->note(n, nrhs, 32, 1);
  }
  if ((e = trsv_flags_dispatch<T, false>(LU, n, ld, X, ldx, nrhs, w, st)) != cudaSuccess) return e;
  if (pf) pf->end(K_TRSM_DIAG, F * 0.5 * n * (double)(n - 1) * nrhs, st);
  if (pf) {
    pf->begin(st);
    pf->note(n, nrhs, 32, 1);
  }
  if ((e = trsv_flags_dispatch<T, true>(LU, n, ld, X, ldx, nrhs, w, st)) != cudaSuccess) return e;
  if (pf) pf->end(K_TRSM_DIAG, F * (0.5 * n * (double)(n - 1) + n) * nrhs, st);
  return cudaSuccess;
}

// ------------------------------------------------- conjugate transposes ----

namespace {
inline int grid_n(int64_t total, int threads = 256) {
  int64_t b = (total + threads - 1) / threads;
  return (int)std::max<int64_t>(1, std::min<int64_t>(b, 65535 * 8));
}
}  // namespace

// dst(perm[i], j) = src(i, j): the inverse of permute_rows.
template <typename T>
__global__ void k_permute_rows_inv(BOp<T> src, BOp<T> dst, const int* perm, int n, int nrhs, int batch) {
  const int64_t per = (int64_t)n * nrhs;
  for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < per * batch; e += (int64_t)gridDim.x * blockDim.x) {
    const int b = (int)(e / per);
    const int rc = (int)(e % per);
    const int i = rc % n, j = rc / n;
    dst.item(b)[perm[(int64_t)b * n + i] + (int64_t)j * dst.ld] = src.item(b)[i + (int64_t)j * src.ld];
  }
}

// Diagonal-block solves with the conjugate transposes of the LU factors:
// LOWER: U^H w = y (U^H is lower triangular); else L^H z = w (upper, unit).
template <typename T, bool LOWER>
__global__ void k_trsm_diag_h(BOp<T> LU, BOp<T> X, int p0, int pb, int nrhs, int batch) {
  for (int b = blockIdx.y; b < batch; b += gridDim.y) {
    const T* Lb = LU.item(b);
    T* Xb = X.item(b);
    for (int j = blockIdx.x * blockDim.x + threadIdx.x; j < nrhs; j += gridDim.x * blockDim.x) {
      T* col = Xb + (int64_t)j * X.ld + p0;
      if (LOWER) {
        for (int r = 0; r < pb; ++r) {
          T s = col[r];
          for (int c = 0; c < r; ++c) s = fmsc(s, conj_of(Lb[(int64_t)(p0 + c) + (int64_t)(p0 + r) * LU.ld]), col[c]);
          const T d = conj_of(Lb[(int64_t)(p0 + r) + (int64_t)(p0 + r) * LU.ld]);
          col[r] = is_zero(d) ? T(0.0) : s * recip(d);
        }
      } else {
        for (int r = pb - 1; r >= 0; --r) {
          T s = col[r];
          for (int c = r + 1; c < pb; ++c)
            s = fmsc(s, conj_of(Lb[(int64_t)(p0 + c) + (int64_t)(p0 + r) * LU.ld]), col[c]);
          col[r] = s;
        }
      }
    }
  }
}

template <typename T>
cudaError_t permute_rows_inv(BOp<T> src, BOp<T> dst, const int* perm, int n, int nrhs, int batch, cudaStream_t st) {
  k_permute_rows_inv<T><<<grid_n((int64_t)n * nrhs * batch), 256, 0, st>>>(src, dst, perm, n, nrhs, batch);
  return cudaGetLastError();
}

// X <- (U^H)^{-1} then (L^H)^{-1}: the conjugate transpose of getrs_inplace
// (without the row permutation, which the caller applies after).
template <typename T>
cudaError_t getrs_h(BOp<T> LU, int n, BOp<T> X, int nrhs, int batch, cudaStream_t st, Prof* pf, TrsvInv* inv) {
  if (n <= 0 || nrhs <= 0 || batch <= 0) return cudaSuccess;
  if (trsv_few_applicable<T>(n, nrhs, batch, inv))
    return trsv_few<T>(LU, n, X, nrhs, batch, true, inv, st, pf);
  const int pb0 = 32;
  const int by = std::min(batch, 65535);
  const int bx = std::min((nrhs + 127) / 128, 1024);
  cudaError_t e;
  for (int p0 = 0; p0 < n; p0 += pb0) {
    const int pb = std::min(pb0, n - p0);
    k_trsm_diag_h<T, true><<<dim3(bx, by), 128, 0, st>>>(LU, X, p0, pb, nrhs, batch);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    const int rest = n - p0 - pb;
    if (rest > 0) {
      GemmArgs<T> g;
      g.M = rest; g.N = nrhs; g.K = pb; g.batch = batch;
      g.A = shifted(LU, (int64_t)p0 + (int64_t)(p0 + pb) * LU.ld);  // U(p0 .., p0 + pb ..)
      g.ta = true;
      g.B = shifted(X, (int64_t)p0);
      g.C = shifted(X, (int64_t)(p0 + pb));
      g.alpha = T(-1.0); g.beta = T(1.0);
      if ((e = gemm<T>(g, st, pf)) != cudaSuccess) return e;
    }
  }
  const int npan = (n + pb0 - 1) / pb0;
  for (int pi = npan - 1; pi >= 0; --pi) {
    const int p0 = pi * pb0, pb = std::min(pb0, n - p0);
    k_trsm_diag_h<T, false><<<dim3(bx, by), 128, 0, st>>>(LU, X, p0, pb, nrhs, batch);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    if (p0 > 0) {
      GemmArgs<T> g;
      g.M = p0; g.N = nrhs; g.K = pb; g.batch = batch;
      g.A = shifted(LU, (int64_t)p0);  // L(p0 .., 0 ..)
      g.ta = true;
      g.B = shifted(X, (int64_t)p0);
      g.C = X;
      g.alpha = T(-1.0); g.beta = T(1.0);
      if ((e = gemm<T>(g, st, pf)) != cudaSuccess) return e;
    }
  }
  return cudaSuccess;
}

// ------------------------------------------------------- instantiation ----

#define HPS_INST(T)                                                                              \
  template cudaError_t gemm<T>(const GemmArgs<T>&, cudaStream_t, Prof*);                         \
  template cudaError_t fill<T>(BOp<T>, int, int, int, T, T, cudaStream_t, Prof*);                \
  template int lu_group_size<T>(int, int, int);                                                  \
  template size_t lu_pub_bytes<T>(int, int, int);                                                \
  template cudaError_t getrf<T>(BOp<T>, int, int, int*, int*, int*, unsigned*, int,              \
                                const LuWork&, cudaStream_t, Prof*);                             \
  template cudaError_t permute_rows<T>(BOp<T>, BOp<T>, const int*, int, int, int, cudaStream_t,  \
                                       Prof*);                                                   \
  template cudaError_t getrs_inplace<T>(BOp<T>, int, BOp<T>, int, int, cudaStream_t, Prof*, TrsvInv*);   \
  template bool trsv_flags_applicable<T>(int, int, int, const TrsvWork&);                        \
  template cudaError_t getrs_flags<T>(const T*, int, int, T*, int, int, TrsvWork&, cudaStream_t, Prof*); \
  template cudaError_t permute_rows_inv<T>(BOp<T>, BOp<T>, const int*, int, int, int, cudaStream_t);    \
  template cudaError_t getrs_h<T>(BOp<T>, int, BOp<T>, int, int, cudaStream_t, Prof*, TrsvInv*);

HPS_INST(double)
HPS_INST(cplx)


// ----------------------------------------------------------------------------
// Bounded-wait check (hps_debug_wait_timeout): one CTA runs one of the
// library's bounded waits on a word that nothing else writes.  which 0: the
// inter-CTA group barrier with a group of two CTAs of which only this one
// arrives (satisfied: a group of one); which 1: the flag wait of the
// flag-ordered triangular solves on a flag nothing sets (satisfied: the flag
// already holds the awaited value).  A wait that gives up sets
// DEV_ERR_TIMEOUT in *err.
__global__ void k_debug_wait(int which, int satisfied, unsigned* words, unsigned long long limit, unsigned* err) {
  if (which == 0) {
    group_barrier(words, satisfied ? 1u : 2u, err, limit);
  } else if (threadIdx.x == 0) {
    if (satisfied) words[2] = 7u;
    __threadfence();
    if (!wait_flag(words + 2, 7u, limit)) atomicOr(err, DEV_ERR_TIMEOUT);
  }
}

cudaError_t debug_wait(int which, int satisfied, unsigned* words, unsigned long long limit, unsigned* err,
                       cudaStream_t st) {
  k_debug_wait<<<1, 128, 0, st>>>(which, satisfied, words, limit, err);
  return cudaGetLastError();
}


// The panel LU's wait on an mbarrier (hps_debug_wait_timeout, which 2), as
// debug_mbar_wait does with the product pipeline's.
__global__ void k_debug_panel_wait(int satisfied, long limit, unsigned* err) {
  __shared__ __align__(8) uint64_t bar;
  if (threadIdx.x == 0) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_addr(&bar)));
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    if (satisfied) asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_addr(&bar)) : "memory");
    if (!mbar_wait_cluster(&bar, 0, limit)) atomicOr(err, DEV_ERR_TIMEOUT);
  }
}

cudaError_t debug_panel_wait(int satisfied, long limit, unsigned* err, cudaStream_t st) {
  k_debug_panel_wait<<<1, 32, 0, st>>>(satisfied, limit, err);
  return cudaGetLastError();
}

}  // namespace hps

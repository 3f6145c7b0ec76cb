// Substitution with a triangle of at most 32 rows against many columns, TC
// threads per column: thread g of a column holds its rows g, g + TC, ... in
// registers.  Step k broadcasts the solved entry k from its owner and every
// thread takes its multiple off its own later rows.
//
// The FP64 pipe issues one warp instruction in 64 cycles per scheduler, so
// what counts is the number of multiply-adds a warp issues and that the next
// one never waits: the updates of a step are independent of one another, the
// row that the next step needs is updated first, and the triangle's entries
// come two at a time from shared memory, ordered so that a thread's are
// adjacent.  TC = 1 issues the fewest multiply-adds in all (496 for 32 rows);
// TC = 4 issues 136 in each of four times as many warps, TC = 8 76.
#pragma once
#include "linalg.h"

namespace hps {
namespace {

// whole-warp shuffle of a real or complex value
__device__ inline double shfl_val(double v, int src) { return __shfl_sync(0xffffffffu, v, src); }
__device__ inline cplx shfl_val(cplx v, int src) {
  return cplx(__shfl_sync(0xffffffffu, v.re, src), __shfl_sync(0xffffffffu, v.im, src));
}

template <typename T, int NB, int TC>
struct TriCols {
  static constexpr int R = NB / TC;   // rows of a thread

  // entry (i, k) of the triangle
  static __device__ __forceinline__ int at(int i, int k) { return (k * TC + i % TC) * R + i / TC; }

  static __device__ __forceinline__ void entries(T (&l)[R], const T* s, int q0, int q1) {
    if constexpr (sizeof(T) == 8 && R % 2 == 0) {
#pragma unroll
      for (int q = 0; q < R; q += 2)
        if (q + 1 >= q0 && q <= q1) {
          const double2 v = *reinterpret_cast<const double2*>(s + q);
          l[q] = v.x;
          l[q + 1] = v.y;
        }
    } else {
#pragma unroll
      for (int q = 0; q < R; ++q)
        if (q >= q0 && q <= q1) l[q] = s[q];
    }
  }

  static __device__ __forceinline__ T from(T v, int lane0, int owner) {
    if constexpr (TC == 1) return v;
    else return shfl_val(v, lane0 | owner);
  }

  // tri: the triangle in shared memory, rows and columns >= nb zero; all
  // lanes of the warp take part
  static __device__ __forceinline__ void lower(T (&x)[R], const T* tri, int g, int lane0, int nb) {
    T xk = from(x[0], lane0, 0);
#pragma unroll
    for (int k = 0; k < NB - 1; ++k) {
      if ((k & 7) == 0 && k >= nb) break;
      const int q0 = (k + 1) / TC;
      T l[R];
      entries(l, tri + (k * TC + g) * R, q0, R - 1);
      T xn = xk;
#pragma unroll
      for (int q = q0; q < R; ++q) {
        const T v = fmsc(x[q], l[q], xk);
        if (q == q0) {
          // of this group of TC rows only those below row k
          x[q] = ((k + 1) % TC == 0 || g > k % TC) ? v : x[q];
          xn = from(x[q], lane0, (k + 1) % TC);
        } else {
          x[q] = v;
        }
      }
      xk = xn;
    }
  }

  // dinv: reciprocals of the diagonal
  static __device__ __forceinline__ void upper(T (&x)[R], const T* tri, const T* dinv, int g, int lane0, int nb) {
#pragma unroll
    for (int k = NB - 1; k >= 0; --k) {
      if ((k & 7) == 7 && k - 7 >= nb) continue;
      if (k >= ((nb + 7) & ~7)) continue;
      const T xk = from(x[k / TC], lane0, k % TC) * dinv[k];
      if (TC == 1 || g == k % TC) x[k / TC] = xk;
      if (k > 0) {
        const int q1 = (k - 1) / TC;
        T l[R];
        entries(l, tri + (k * TC + g) * R, 0, q1);
#pragma unroll
        for (int q = R - 1; q >= 0; --q)
          if (q <= q1) {
            const T v = fmsc(x[q], l[q], xk);
            x[q] = (q < k / TC || g < k % TC) ? v : x[q];
          }
      }
    }
  }
};

}  // namespace
}  // namespace hps

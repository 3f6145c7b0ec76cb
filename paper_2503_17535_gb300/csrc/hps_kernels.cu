// HPS-specific device kernels (leaf assembly, merge gathers, downward pass,
// leaf output).  These are gather/scatter and small dot-product kernels; the
// dense FP64 work (LU, triangular solves, GEMM) lives in linalg.cu.
#include "hps_kernels.cuh"

#include <cooperative_groups.h>

#include <algorithm>

namespace hps {

namespace {

inline int grid_for(int64_t total, int threads = 256, int cap = 65535 * 8) {
  int64_t b = (total + threads - 1) / threads;
  return (int)std::max<int64_t>(1, std::min<int64_t>(b, cap));
}

__device__ inline void coords(int dim, int p, int idx, int* c) {
  c[0] = idx % p;
  c[1] = (idx / p) % p;
  c[2] = dim == 3 ? idx / (p * p) : 0;
}

// Entry (i, j) of the leaf operator a Lap + sum_k b_k d_k + c (Section 3.2)
// on the tensor Chebyshev grid: nonzero only when i and j differ along at
// most one axis.
__device__ inline double L_entry(const LeafConsts& k, double s, double a, const double* bk, double c,
                                 int i, int j) {
  int ci[3], cj[3];
  coords(k.dim, k.p, i, ci);
  coords(k.dim, k.p, j, cj);
  int ndiff = 0, dax = -1;
  for (int ax = 0; ax < k.dim; ++ax)
    if (ci[ax] != cj[ax]) { ++ndiff; dax = ax; }
  if (ndiff > 1) return 0.0;
  double v = 0.0;
  const double s2 = s * s;
  for (int ax = 0; ax < k.dim; ++ax) {
    if (ndiff == 1 && ax != dax) continue;
    const int e = ci[ax] * k.p + cj[ax];
    v = fma(a * s2, k.DD[e], v);
    v = fma(bk[ax] * s, k.D[e], v);
  }
  if (ndiff == 0) v += c;
  return v;
}

__device__ inline void load_coeffs(const Coeffs& cf, int64_t at, int dim, double* a, double* b,
                                   double* c) {
  *a = cf.a ? cf.a[at] : 1.0;
  for (int ax = 0; ax < 3; ++ax) b[ax] = (ax < dim && cf.b[ax]) ? cf.b[ax][at] : 0.0;
  *c = cf.c ? cf.c[at] : 0.0;
}

}  // namespace

// --------------------------------------------------------------- leaves ----

// The leaf operators are mostly zeros (an entry couples nodes that differ along
// one axis: 28 of 196 per row in 2D at p = 16), and FP64 instructions cost a
// warp the same for one live lane as for 32: a CTA clears its leaf's block
// and then computes the nonzero entries only, every lane with one of them.
// Testing every entry for zero took 2650 us for 4096 leaves of 196 x 196, the
// pipe's time for ten FP64 instructions per warp of entries; now 558 (writing
// 1.26 GB takes 190).

// stride of axis ax in the node order
__device__ inline int axis_stride(int p, int ax) { return ax == 0 ? 1 : ax == 1 ? p : p * p; }

__global__ void __launch_bounds__(256) k_leaf_dtn_Lii(LeafConsts k, int64_t nl, int nchunk, Coeffs cf, double* Lii) {
  const int q = k.p - 2, cols = (k.ni + nchunk - 1) / nchunk;
  for (int64_t lc = blockIdx.x; lc < nl * nchunk; lc += gridDim.x) {
    const int64_t leaf = lc / nchunk;
    const int c0 = (int)(lc % nchunk) * cols, nc = min(cols, k.ni - c0);
    if (nc <= 0) continue;
    double* L = Lii + leaf * (int64_t)k.ni * k.ni + (int64_t)c0 * k.ni;
    for (int64_t e = threadIdx.x; e < (int64_t)nc * k.ni; e += blockDim.x) L[e] = 0.0;
    __syncthreads();
    const double s = k.sleaf ? k.sleaf[leaf] : k.s;
    // column c's entries along axis ax, position t; the diagonal with axis 0
    for (int e = threadIdx.x; e < nc * k.dim * q; e += blockDim.x) {
      const int t = 1 + e % q, ca = e / q, ax = ca % k.dim, c = ca / k.dim;
      const int j = k.Ii[c0 + c];
      int cj[3];
      coords(k.dim, k.p, j, cj);
      const int own = ax == 0 ? cj[0] : ax == 1 ? cj[1] : cj[2];
      if (t == own && ax != 0) continue;
      const int i = j + (t - own) * axis_stride(k.p, ax);
      double a, b[3], cc;
      load_coeffs(cf, leaf * k.npts + i, k.dim, &a, b, &cc);
      L[k.iidx[i] + (int64_t)c * k.ni] = L_entry(k, s, a, b, cc, i, j);
    }
  }
}

// CTAs per leaf of k_leaf_dtn_Lii: four a SM in all
inline int Lii_chunks(int64_t nl, int ni) {
  return (int)std::max<int64_t>(1, std::min<int64_t>(ni, (4 * device_sms() + nl - 1) / nl));
}

// [L_ie P | -f_i]: a thread takes a row's kRhsCols columns, so that the row's
// couplings to its 2 dim boundary nodes are computed once for them (per entry they
// were six of every seven FP64 instructions in 3D: 992 us for 512 leaves of 216 x
// 217; now 299).
constexpr int kRhsCols = 16;
__global__ void __launch_bounds__(256) k_leaf_dtn_rhs(LeafConsts k, int64_t nl, Coeffs cf, const double* f, double* rhs) {
  const int ncol = k.nb + 1, nchunk = (ncol + kRhsCols - 1) / kRhsCols;
  const int64_t total = nl * nchunk * k.ni;
  for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < total; e += (int64_t)gridDim.x * blockDim.x) {
    const int r = (int)(e % k.ni);
    const int64_t lc = e / k.ni, leaf = lc / nchunk;
    const int col0 = (int)(lc % nchunk) * kRhsCols, col1 = min(col0 + kRhsCols, ncol);
    const int i = k.Ii[r];
    double a, b[3], cc;
    load_coeffs(cf, leaf * k.npts + i, k.dim, &a, b, &cc);
    const double s = k.sleaf ? k.sleaf[leaf] : k.s;
    int ci[3];
    coords(k.dim, k.p, i, ci);
    double lij[6];
    const double* P[6];
#pragma unroll
    for (int q = 0; q < 6; ++q) {
      const int ax = q / 2, end = q % 2;
      lij[q] = 0.0;
      P[q] = k.P;
      if (ax >= k.dim) continue;
      const int cj = end ? k.p - 1 : 0;
      const int j = i + (cj - ci[ax]) * axis_stride(k.p, ax);
      const int el = ci[ax] * k.p + cj;
      P[q] += k.prow[j];
      lij[q] = fma(a * s * s, k.DD[el], b[ax] * s * k.D[el]);
    }
    double* out = rhs + leaf * (int64_t)k.ni * ncol + r;
    for (int col = col0; col < col1; ++col) {
      double acc = 0.0;
      if (col == k.nb) {
        acc = f ? -f[leaf * k.npts + i] : 0.0;
      } else {
#pragma unroll
        for (int q = 0; q < 6; ++q)
          if (q < 2 * k.dim) acc = fma(lij[q], P[q][(int64_t)col * k.ne], acc);
      }
      out[(int64_t)col * k.ni] = acc;
    }
  }
}

cudaError_t leaf_dtn_assemble(const LeafConsts& k, int64_t nl, Coeffs cf, const double* f,
                              double* Lii, double* rhs, cudaStream_t st, Prof* pf) {
  if (pf) pf->begin(st);
  const int nchunk = Lii_chunks(nl, k.ni);
  k_leaf_dtn_Lii<<<grid_for(nl * nchunk, 1), 256, 0, st>>>(k, nl, nchunk, cf, Lii);
  if (pf) pf->end(K_ASSEMBLE, 0.0, st);
  if (pf) pf->begin(st);
  k_leaf_dtn_rhs<<<grid_for(nl * k.ni * ((k.nb + kRhsCols) / kRhsCols)), 256, 0, st>>>(k, nl, cf, f, rhs);
  if (pf) pf->end(K_ASSEMBLE, 2.0 * 2 * k.dim * (double)nl * k.ni * k.nb, st);
  return cudaGetLastError();
}

__global__ void k_leaf_iti_B(LeafConsts k, int64_t nl, Coeffs cf, cplx* B) {
  const int n = k.npts;
  const int64_t per = (int64_t)n * n;
  for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < nl * per;
       e += (int64_t)gridDim.x * blockDim.x) {
    const int64_t leaf = e / per;
    const int rc = (int)(e % per);
    const int r = rc % n, j = rc / n;
    cplx v(0.0, 0.0);
    if (r < k.nown) {
      // incoming impedance row: sgn * s * d/dx_axis + i eta at the owned node
      const int node = k.own_node[r], ax = k.own_axis[r];
      int ci[3], cj[3];
      coords(k.dim, k.p, node, ci);
      coords(k.dim, k.p, j, cj);
      bool same = true;
      for (int a2 = 0; a2 < k.dim; ++a2)
        if (a2 != ax && ci[a2] != cj[a2]) same = false;
      if (same) v.re = k.own_sgn[r] * k.s * k.D[ci[ax] * k.p + cj[ax]];
      if (j == node) v.im = k.eta;
    } else {
      const int i = k.Ii[r - k.nown];
      double a, b[3], cc;
      load_coeffs(cf, leaf * k.npts + i, k.dim, &a, b, &cc);
      v.re = L_entry(k, k.s, a, b, cc, i, j);
    }
    B[e] = v;
  }
}

__global__ void __launch_bounds__(256) k_leaf_iti_rhs(LeafConsts k, int64_t nl, const cplx* f, cplx* rhs) {
  const int n = k.npts, ncol = k.nb + 1;
  for_tile(n, ncol, nl, [&](int64_t leaf, int r, int col) {
    cplx v(0.0, 0.0);
    if (col < k.nb) {
      if (r < k.nown) v = cplx(k.P[r + (int64_t)col * k.nown], 0.0);
    } else if (r >= k.nown && f) {
      v = f[leaf * k.npts + k.Ii[r - k.nown]];
    }
    rhs[(leaf * ncol + col) * n + r] = v;
  });
}

// L(I_i, boundary nodes in owner order): the interior rows of the leaf
// operator on the boundary columns, for the ItI interior elimination.
// Interior rows, owned boundary columns; nonzero along the normal of the
// column's node (no corner node couples with an interior one).
__global__ void __launch_bounds__(256) k_leaf_iti_Lie(LeafConsts k, int64_t nl, Coeffs cf, double* Lie) {
  const int per = k.ni * k.nown, q = k.p - 2;
  for (int64_t leaf = blockIdx.x; leaf < nl; leaf += gridDim.x) {
    double* L = Lie + leaf * per;
    for (int e = threadIdx.x; e < per; e += blockDim.x) L[e] = 0.0;
    __syncthreads();
    for (int e = threadIdx.x; e < k.nown * q; e += blockDim.x) {
      const int c = e / q, t = 1 + e % q;
      const int j = k.own_node[c];
      int cj[3];
      coords(k.dim, k.p, j, cj);
      int nax = 0, ax = 0;
      for (int d = 0; d < k.dim; ++d)
        if (cj[d] == 0 || cj[d] == k.p - 1) ++nax, ax = d;
      if (nax != 1) continue;
      const int own = ax == 0 ? cj[0] : ax == 1 ? cj[1] : cj[2];
      const int i = j + (t - own) * axis_stride(k.p, ax);
      double a, b[3], cc;
      load_coeffs(cf, leaf * k.npts + i, k.dim, &a, b, &cc);
      L[k.iidx[i] + c * k.ni] = L_entry(k, k.s, a, b, cc, i, j);
    }
  }
}

// Per-block bounds of the coefficients: out[3 * block + {0, 1, 2}] =
// (min a, max |b|, max c) over this block's share of the nodes.
__global__ void k_coef_bounds(Coeffs cf, int dim, int64_t n, double* out) {
  __shared__ double sa[256], sb[256], sc[256];
  double amin = 1e300, bmax = 0.0, cmax = -1e300;
  for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < n; e += (int64_t)gridDim.x * blockDim.x) {
    amin = fmin(amin, cf.a ? cf.a[e] : 1.0);
    for (int ax = 0; ax < dim; ++ax) bmax = fmax(bmax, cf.b[ax] ? fabs(cf.b[ax][e]) : 0.0);
    cmax = fmax(cmax, cf.c ? cf.c[e] : 0.0);
  }
  sa[threadIdx.x] = amin;
  sb[threadIdx.x] = bmax;
  sc[threadIdx.x] = cmax;
  __syncthreads();
  for (int o = blockDim.x / 2; o > 0; o >>= 1) {
    if ((int)threadIdx.x < o) {
      sa[threadIdx.x] = fmin(sa[threadIdx.x], sa[threadIdx.x + o]);
      sb[threadIdx.x] = fmax(sb[threadIdx.x], sb[threadIdx.x + o]);
      sc[threadIdx.x] = fmax(sc[threadIdx.x], sc[threadIdx.x + o]);
    }
    __syncthreads();
  }
  if (threadIdx.x == 0) {
    out[3 * blockIdx.x] = sa[0];
    out[3 * blockIdx.x + 1] = sb[0];
    out[3 * blockIdx.x + 2] = sc[0];
  }
}

cudaError_t leaf_assemble_Lii(const LeafConsts& k, int64_t nl, Coeffs cf, double* Lii, cudaStream_t st, Prof* pf) {
  if (pf) pf->begin(st);
  const int nchunk = Lii_chunks(nl, k.ni);
  k_leaf_dtn_Lii<<<grid_for(nl * nchunk, 1), 256, 0, st>>>(k, nl, nchunk, cf, Lii);
  if (pf) pf->end(K_ASSEMBLE, 0.0, st);
  return cudaGetLastError();
}

cudaError_t leaf_iti_Lie(const LeafConsts& k, int64_t nl, Coeffs cf, double* Lie, cudaStream_t st, Prof* pf) {
  if (pf) pf->begin(st);
  k_leaf_iti_Lie<<<grid_for(nl, 1), 256, 0, st>>>(k, nl, cf, Lie);
  if (pf) pf->end(K_ASSEMBLE, 0.0, st);
  return cudaGetLastError();
}

cudaError_t leaf_iti_rhs(const LeafConsts& k, int64_t nl, const cplx* f, cplx* rhs, cudaStream_t st, Prof* pf) {
  if (pf) pf->begin(st);
  k_leaf_iti_rhs<<<tile_grid(k.npts, k.nb + 1, nl), 256, 0, st>>>(k, nl, f, rhs);
  if (pf) pf->end(K_ASSEMBLE, 0.0, st);
  return cudaGetLastError();
}

cudaError_t coef_bounds(Coeffs cf, int dim, int64_t n, double* d_out, double* h_out, cudaStream_t st) {
  constexpr int nblk = 64;
  k_coef_bounds<<<nblk, 256, 0, st>>>(cf, dim, n, d_out);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  double tmp[3 * nblk];
  if ((e = cudaMemcpyAsync(tmp, d_out, sizeof(tmp), cudaMemcpyDeviceToHost, st)) != cudaSuccess) return e;
  if ((e = cudaStreamSynchronize(st)) != cudaSuccess) return e;
  h_out[0] = 1e300; h_out[1] = 0.0; h_out[2] = -1e300;
  for (int b = 0; b < nblk; ++b) {
    h_out[0] = std::min(h_out[0], tmp[3 * b]);
    h_out[1] = std::max(h_out[1], tmp[3 * b + 1]);
    h_out[2] = std::max(h_out[2], tmp[3 * b + 2]);
  }
  return cudaSuccess;
}

cudaError_t leaf_iti_assemble(const LeafConsts& k, int64_t nl, Coeffs cf, const cplx* f, cplx* B,
                              cplx* rhs, cudaStream_t st, Prof* pf) {
  if (pf) pf->begin(st);
  k_leaf_iti_B<<<grid_for(nl * k.npts * k.npts), 256, 0, st>>>(k, nl, cf, B);
  if (pf) pf->end(K_ASSEMBLE, 0.0, st);
  if (pf) pf->begin(st);
  k_leaf_iti_rhs<<<tile_grid(k.npts, k.nb + 1, nl), 256, 0, st>>>(k, nl, f, rhs);
  if (pf) pf->end(K_ASSEMBLE, 0.0, st);
  return cudaGetLastError();
}

template <typename T>
__global__ void k_leaf_particular_rhs(LeafConsts k, int64_t nl, int nrhs, const T* f, T* out, bool iti) {
  const int rows = iti ? k.npts : k.ni;
  const int64_t per = (int64_t)rows * nrhs;
  for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < nl * per;
       e += (int64_t)gridDim.x * blockDim.x) {
    const int64_t leaf = e / per;
    const int rc = (int)(e % per);
    const int r = rc % rows, c = rc / rows;
    const int64_t fo = ((int64_t)c * nl + leaf) * k.npts;
    T v = T(0.0);
    if (!iti) v = -f[fo + k.Ii[r]];
    else if (r >= k.nown) v = f[fo + k.Ii[r - k.nown]];
    out[e] = v;
  }
}

template <typename T>
cudaError_t leaf_particular_rhs(const LeafConsts& k, int64_t nl, int nrhs, const T* f, T* out,
                                bool iti, cudaStream_t st, Prof* pf) {
  const int rows = iti ? k.npts : k.ni;
  if (pf) pf->begin(st);
  k_leaf_particular_rhs<T><<<grid_for(nl * rows * nrhs), 256, 0, st>>>(k, nl, nrhs, f, out, iti);
  if (pf) pf->end(K_GATHER, 0.0, st);
  return cudaGetLastError();
}

__global__ void k_leaf_dtn_init_T(const double* QP, int nb, double s, int64_t nl, double* TH) {
  const int64_t per = (int64_t)nb * (nb + 1);
  for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < nl * per;
       e += (int64_t)gridDim.x * blockDim.x) {
    const int rc = (int)(e % per);
    TH[e] = (rc < nb * nb) ? s * QP[rc] : 0.0;
  }
}

cudaError_t leaf_dtn_init_T(const double* QP, int nb, double s, int64_t nl, double* TH,
                            cudaStream_t st, Prof* pf) {
  if (pf) pf->begin(st);
  k_leaf_dtn_init_T<<<grid_for(nl * nb * (nb + 1)), 256, 0, st>>>(QP, nb, s, nl, TH);
  if (pf) pf->end(K_OTHER, 0.0, st);
  return cudaGetLastError();
}

// --------------------------------------------------------------- merges ----

__device__ inline void add_pair(double* p, double v) { atomicAdd(p, v); }
__device__ inline void add_pair(cplx* p, cplx v) {
  atomicAdd(&p->re, v.re);
  atomicAdd(&p->im, v.im);
}

// One thread per (merge, child, child row i, child column j <= nbc).
// DtN: D(var_i, var_j) += T (interface diagonal blocks get exactly two
// addends, so the result does not depend on their order); C and A entries
// and the h columns have a single owner except h_int, which also gets two.
// ItI: D(eq_i, var_j) = T on top of the identity, R(eq_i, .) = T, single owner.
template <typename T>
__global__ void k_merge_gather(const T* Tc, int64_t cstride, int nmerge, int nch, int nbc, int n_ext,
                               int n_int, const int* ext, const int* var, const int* eq, bool iti,
                               T* D, T* R, T* TP) {
  for_tile(nbc, nbc + 1, (int64_t)nmerge * nch, [&](int64_t cidx, int i, int j) {   // cidx = nch * merge + k
    const int k = (int)(cidx % nch);
    const int64_t b = cidx / nch;
    const T v = Tc[cidx * cstride + i + (int64_t)j * nbc];
    const int ei = ext[k * nbc + i];
    const int ri = iti ? eq[k * nbc + i] : var[k * nbc + i];
    T* Db = D + b * (int64_t)n_int * n_int;
    T* Rb = R + b * (int64_t)n_int * (n_ext + 1);
    T* Pb = TP + b * (int64_t)n_ext * (n_ext + 1);
    if (j == nbc) {  // h column
      if (ei >= 0) Pb[ei + (int64_t)n_ext * n_ext] = v;
      else if (iti) Rb[ri + (int64_t)n_int * n_ext] = v;
      else add_pair(&Rb[ri + (int64_t)n_int * n_ext], v);
      return;
    }
    const int ej = ext[k * nbc + j];
    const int vj = var[k * nbc + j];
    if (ei >= 0) {
      if (ej >= 0) Pb[ei + (int64_t)ej * n_ext] = v;        // A
      // (exterior row, interior column) = B: used in place, not stored
    } else {
      if (ej >= 0) Rb[ri + (int64_t)ej * n_int] = v;         // C
      else if (iti) Db[ri + (int64_t)vj * n_int] = v;        // D12 / D21
      else add_pair(&Db[ri + (int64_t)vj * n_int], v);       // D
    }
  });
}

template <typename T>
cudaError_t merge_gather(const T* Tc, int64_t cstride, int nmerge, int nch, int nbc, int n_ext,
                         int n_int, const int* ext, const int* var, const int* eq, bool iti, T* D,
                         T* R, T* TP, cudaStream_t st, Prof* pf) {
  if (pf) pf->begin(st);
  k_merge_gather<T><<<tile_grid(nbc, nbc + 1, (int64_t)nmerge * nch), 256, 0, st>>>(Tc, cstride, nmerge, nch, nbc, n_ext, n_int, ext,
                                                     var, eq, iti, D, R, TP);
  if (pf) pf->end(K_GATHER, 0.0, st);
  return cudaGetLastError();
}

template <typename T>
__global__ void k_merge_gather_h(const T* hc, int nmerge, int nch, int nbc, int n_ext, int n_int,
                                 int nrhs, const int* ext, const int* var, const int* eq, bool iti,
                                 T* r, T* hp) {
  const int64_t per_child = (int64_t)nbc * nrhs;
  const int64_t total = (int64_t)nmerge * nch * per_child;
  for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < total;
       e += (int64_t)gridDim.x * blockDim.x) {
    const int64_t cidx = e / per_child;
    const int rc = (int)(e % per_child);
    const int i = rc % nbc, c = rc / nbc;
    const int k = (int)(cidx % nch);
    const int64_t b = cidx / nch;
    const T v = hc[cidx * per_child + rc];
    const int ei = ext[k * nbc + i];
    if (ei >= 0) {
      hp[b * (int64_t)n_ext * nrhs + ei + (int64_t)c * n_ext] = v;
    } else {
      const int ri = iti ? eq[k * nbc + i] : var[k * nbc + i];
      T* p = &r[b * (int64_t)n_int * nrhs + ri + (int64_t)c * n_int];
      if (iti) *p = v;
      else add_pair(p, v);
    }
  }
}

template <typename T>
cudaError_t merge_gather_h(const T* hc, int nmerge, int nch, int nbc, int n_ext, int n_int, int nrhs,
                           const int* ext, const int* var, const int* eq, bool iti, T* r, T* hp,
                           cudaStream_t st, Prof* pf) {
  const int64_t total = (int64_t)nmerge * nch * nbc * nrhs;
  if (pf) pf->begin(st);
  k_merge_gather_h<T><<<grid_for(total), 256, 0, st>>>(hc, nmerge, nch, nbc, n_ext, n_int, nrhs, ext,
                                                       var, eq, iti, r, hp);
  if (pf) pf->end(K_GATHER, 0.0, st);
  return cudaGetLastError();
}

// ------------------------------------------------------------- downward ----

// gint(:, c) = -(X_C gpar(:, c) + xpart(:, c)): a lane per row (the rows of all
// merges in one sequence), NC right-hand sides at a time, the columns dealt to
// CG warps of a CTA and, with CL, in ranges to the CS CTAs of a cluster; the
// partial sums are added in shared memory in a fixed order, so that the
// result does not depend on scheduling.
//
// Bound by the FP64 pipe when there are many rows (two multiply-adds per clock
// and SM: 86 us for 205 MB of complex entries and one right-hand side, which
// memory would deliver in 31), by the latency of a row's loads when there are
// few; the column groups spread those over more warps, and clusters of small
// CTAs over all SMs while there are less than two 32-row tiles per SM (112 tiles of
// 3584 complex columns 127 -> 117 us, 224 of 1792 123 -> 105; with more tiles, or
// very long rows, the ranges cost locality: 432 real tiles 94 -> 137, 216 of
// 13824 columns 246 -> 265).  With one warp per 32 rows up to 255 columns, as
// before, 64 real merges of 176 columns took 80 us, now 12.
constexpr int64_t kDownL2 = 116 << 20;   // bytes of X that stay in L2 (129 MB) between groups
constexpr int kGridY = 65535;   // groups of right-hand sides in one launch (grid limit)
template <typename T, int CG, int NC, bool CL>
__global__ void __launch_bounds__(32 * (CG < 4 ? 4 : CG)) k_down_gint(const T* X, const T* xp, const T* gpar,
                                                                       int64_t rows, int n_ext, int n_int, int nrhs,
                                                                       int CS, int cfirst, T* gint) {
  namespace cg_ = cooperative_groups;
  constexpr int NW = CG < 4 ? 4 : CG;
  __shared__ T part[CG > 1 ? NW : 1][NC][33];
  __shared__ T sums[CL ? 8 : 1][NC][33];   // of the cluster's CTAs
  if constexpr (CL) cluster_arrive();   // before its sums go to the first CTA, that one has started
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, cg = w % CG;
  const int rank = CL ? (int)blockIdx.x % CS : 0;
  const int64_t R = ((int64_t)(CL ? blockIdx.x / CS : blockIdx.x) * (NW / CG) + w / CG) * 32 + lane;
  const int c0 = cfirst + blockIdx.y * NC;
  const bool live = R < rows;
  const int64_t b = live ? R / n_int : 0;
  const int r = live ? (int)(R % n_int) : 0;
  const T* x = X + b * (int64_t)n_int * (n_ext + 1) + r;
  const T* g = gpar + (b * nrhs + c0) * (int64_t)n_ext;
  int64_t go[NC];   // columns beyond the last repeat it
#pragma unroll
  for (int c = 0; c < NC; ++c) go[c] = (int64_t)min(c, nrhs - 1 - c0) * n_ext;
  T acc[NC];
#pragma unroll
  for (int c = 0; c < NC; ++c) acc[c] = T(0.0);
  if (live) {
    const int j1 = CL ? (int)((int64_t)n_ext * (rank + 1) / CS) : n_ext;   // a cluster's CTAs take ranges of columns
#pragma unroll 8
    for (int j = (CL ? (int)((int64_t)n_ext * rank / CS) : 0) + cg; j < j1; j += CG) {
      const T xv = x[(int64_t)j * n_int];
#pragma unroll
      for (int c = 0; c < NC; ++c) acc[c] = fmac(acc[c], xv, g[go[c] + j]);
    }
  }
  if constexpr (CG > 1) {
#pragma unroll
    for (int c = 0; c < NC; ++c) part[w][c][lane] = acc[c];
    __syncthreads();
    if (cg == 0) {
#pragma unroll
      for (int c = 0; c < NC; ++c)
#pragma unroll
        for (int k = 1; k < CG; ++k) acc[c] = acc[c] + part[w + k][c][lane];
    }
  }
  if constexpr (CL) {
    cg_::cluster_group cl = cg_::this_cluster();
    cluster_wait();
    if (w == 0) {
      T* first = cl.map_shared_rank(&sums[0][0][0], 0);
#pragma unroll
      for (int c = 0; c < NC; ++c) first[(rank * NC + c) * 33 + lane] = acc[c];
    }
    cl.sync();
    if (rank != 0) return;
    if (w == 0)
      for (int k = 1; k < CS; ++k)
#pragma unroll
        for (int c = 0; c < NC; ++c) acc[c] = acc[c] + sums[k][c][lane];
  }
  if (cg != 0 || !live) return;
#pragma unroll
  for (int c = 0; c < NC; ++c) {
    if (c0 + c >= nrhs) break;
    const T s = xp ? xp[(b * nrhs + c0 + c) * (int64_t)n_int + r] : x[(int64_t)n_ext * n_int];
    gint[(b * nrhs + c0 + c) * (int64_t)n_int + r] = -(s + acc[c]);
  }
}

// right-hand sides a thread takes at a time: at most `most`, in even groups
inline int rhs_group(int nrhs, int most) {
  const int groups = (nrhs + most - 1) / most;
  return (nrhs + groups - 1) / groups;
}

// the right-hand sides [cfirst, cend) of nrhs
template <typename T, int CG, int NC, bool CL>
cudaError_t launch_down_gint_nc(const T* X, const T* xp, const T* gpar, int64_t rows, int n_ext, int n_int, int nrhs,
                                int cfirst, int cend, int cs, T* gint, cudaStream_t st) {
  constexpr int NW = CG < 4 ? 4 : CG;
  const int per = 32 * (NW / CG);
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim.x = (unsigned)((rows + per - 1) / per * cs);
  cfg.blockDim = dim3(32 * NW);
  cfg.stream = st;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = cs;
  at[0].val.clusterDim.y = 1;
  at[0].val.clusterDim.z = 1;
  cfg.attrs = at;
  cfg.numAttrs = CL ? 1 : 0;
  cudaError_t e = cudaSuccess;
  for (int c = cfirst; c < cend && e == cudaSuccess; c += kGridY * NC) {
    cfg.gridDim.y = std::min(kGridY, (cend - c + NC - 1) / NC);
    e = cudaLaunchKernelEx(&cfg, k_down_gint<T, CG, NC, CL>, X, xp, gpar, rows, n_ext, n_int, nrhs, cs, c, gint);
  }
  return e;
}

template <typename T, int CG, bool CL>
cudaError_t launch_down_gint_cg(const T* X, const T* xp, const T* gpar, int64_t rows, int n_ext, int n_int, int nrhs,
                                int cfirst, int cend, int cs, T* gint, int nc, cudaStream_t st) {
  switch (nc) {
    case 1: return launch_down_gint_nc<T, CG, 1, CL>(X, xp, gpar, rows, n_ext, n_int, nrhs, cfirst, cend, cs, gint, st);
    case 2: return launch_down_gint_nc<T, CG, 2, CL>(X, xp, gpar, rows, n_ext, n_int, nrhs, cfirst, cend, cs, gint, st);
    case 3: return launch_down_gint_nc<T, CG, 3, CL>(X, xp, gpar, rows, n_ext, n_int, nrhs, cfirst, cend, cs, gint, st);
    default: return launch_down_gint_nc<T, CG, 4, CL>(X, xp, gpar, rows, n_ext, n_int, nrhs, cfirst, cend, cs, gint, st);
  }
}

// right-hand sides per thread for `cols` of them
inline int down_cols(int64_t tiles, int cols) {
  // fewer where the row tiles would not go round the SMs two and a half times (112
  // tiles, eight right-hand sides, real: 182 us in groups of four, 105 one by one; 224
  // tiles: 96 in groups of four, 115 of three)
  int most = 4;
  while (most > 1 && 2 * tiles * ((cols + most - 1) / most) < 5 * device_sms()) --most;
  return rhs_group(cols, most);
}

template <typename T>
cudaError_t launch_down_gint(const T* X, const T* xp, const T* gpar, int nmerge, int n_ext, int n_int, int nrhs,
                             T* gint, cudaStream_t st) {
  const int64_t rows = (int64_t)nmerge * n_int, tiles = (rows + 31) / 32;
  auto range = [&](int c0, int c1, int nc) {
    const int64_t warps = tiles * ((c1 - c0 + nc - 1) / nc);
    const bool cluster = warps < 2 * device_sms() && n_ext < 8192;
    const int cg = down_groups(warps, n_ext, cluster ? 32 : 16);
    if (cg == 1) return launch_down_gint_cg<T, 1, false>(X, xp, gpar, rows, n_ext, n_int, nrhs, c0, c1, 1, gint, nc, st);
    if (cg == 2) return launch_down_gint_cg<T, 2, false>(X, xp, gpar, rows, n_ext, n_int, nrhs, c0, c1, 1, gint, nc, st);
    if (cg == 4) return launch_down_gint_cg<T, 4, false>(X, xp, gpar, rows, n_ext, n_int, nrhs, c0, c1, 1, gint, nc, st);
    if (cluster) return launch_down_gint_cg<T, 4, true>(X, xp, gpar, rows, n_ext, n_int, nrhs, c0, c1, cg / 4, gint, nc, st);
    if (cg == 8) return launch_down_gint_cg<T, 8, false>(X, xp, gpar, rows, n_ext, n_int, nrhs, c0, c1, 1, gint, nc, st);
    return launch_down_gint_cg<T, 16, false>(X, xp, gpar, rows, n_ext, n_int, nrhs, c0, c1, 1, gint, nc, st);
  };
  const int nc = down_cols(tiles, nrhs);
  const bool cplx_rows = sizeof(T) == 16, even = nrhs % nc == 0;
  // While L2 keeps X groups save no memory traffic.  Complex
  // rows are then bound by the pipe anyway and finish sooner one by one (128 tiles
  // of 256 columns, eight right-hand sides: 68 us, in groups of three 90), real ones when
  // the last group would be short (192 tiles of 192, five: 18 us, in groups of three 29).
  if (rows * n_ext * (int64_t)sizeof(T) < kDownL2) return range(0, nrhs, cplx_rows || !even ? 1 : nc);
  // Beyond, a short last group of complex rows costs a full one's work: the
  // columns left over by fours go in a launch of their own (205 MB, five right-hand
  // sides, all six levels of 4096 leaves: 3.13 ms in groups of three, 2.71 as four and one).
  if (!cplx_rows || even || nrhs <= 4) return range(0, nrhs, nc);
  const int whole = nrhs / 4 * 4, wide = down_cols(tiles, whole);
  const cudaError_t e = range(0, whole, wide == 3 ? 2 : wide);
  return e != cudaSuccess || whole == nrhs ? e : range(whole, nrhs, down_cols(tiles, nrhs - whole));
}

template <typename T>
__global__ void k_down_children(const T* gpar, const T* gint, int nmerge, int nch, int nbc, int n_ext,
                                int n_int, int nrhs, const int* ext, const int* var, T* gchild) {
  const int64_t per_child = (int64_t)nbc * nrhs;
  const int64_t total = (int64_t)nmerge * nch * per_child;
  for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < total;
       e += (int64_t)gridDim.x * blockDim.x) {
    const int64_t cidx = e / per_child;
    const int rc = (int)(e % per_child);
    const int i = rc % nbc, c = rc / nbc;
    const int k = (int)(cidx % nch);
    const int64_t b = cidx / nch;
    const int ei = ext[k * nbc + i];
    T v;
    if (ei >= 0) v = gpar[b * (int64_t)n_ext * nrhs + ei + (int64_t)c * n_ext];
    else v = gint[b * (int64_t)n_int * nrhs + var[k * nbc + i] + (int64_t)c * n_int];
    gchild[e] = v;
  }
}

template <typename T>
cudaError_t down_level(const T* X, const T* xp, const T* gpar, int nmerge, int nch, int nbc, int n_ext,
                       int n_int, int nrhs, const int* ext, const int* var, T* gint, T* gchild,
                       cudaStream_t st, Prof* pf) {
  const double F = sizeof(T) == sizeof(cplx) ? 8.0 : 2.0;
  if (pf) pf->begin(st);
  cudaError_t e = launch_down_gint<T>(X, xp, gpar, nmerge, n_ext, n_int, nrhs, gint, st);
  if (e != cudaSuccess) return e;
  if (pf) pf->end(K_DOWN, F * (double)nmerge * n_int * n_ext * nrhs, st);
  if (pf) pf->begin(st);
  k_down_children<T><<<grid_for((int64_t)nmerge * nch * nbc * nrhs), 256, 0, st>>>(
      gpar, gint, nmerge, nch, nbc, n_ext, n_int, nrhs, ext, var, gchild);
  if (pf) pf->end(K_GATHER, 0.0, st);
  return cudaGetLastError();
}

template <typename T>
cudaError_t down_gint(const T* X, const T* xp, const T* gpar, int nmerge, int n_ext, int n_int, int nrhs,
                      T* gint, cudaStream_t st, Prof* pf) {
  const double F = sizeof(T) == sizeof(cplx) ? 8.0 : 2.0;
  if (pf) pf->begin(st);
  const cudaError_t e = launch_down_gint<T>(X, xp, gpar, nmerge, n_ext, n_int, nrhs, gint, st);
  if (pf) pf->end(K_DOWN, F * (double)nmerge * n_int * n_ext * nrhs, st);
  return e;
}

template <typename T>
cudaError_t down_children(const T* gpar, const T* gint, int nmerge, int nch, int nbc, int n_ext, int n_int,
                          int nrhs, const int* ext, const int* var, T* gchild, cudaStream_t st, Prof* pf) {
  if (pf) pf->begin(st);
  k_down_children<T><<<grid_for((int64_t)nmerge * nch * nbc * nrhs), 256, 0, st>>>(
      gpar, gint, nmerge, nch, nbc, n_ext, n_int, nrhs, ext, var, gchild);
  if (pf) pf->end(K_GATHER, 0.0, st);
  return cudaGetLastError();
}

// The row of the leaf's solution map that a node takes: of Y for ItI (complex
// data), of -Y at interior and of P at boundary nodes for DtN (real data), whose
// two are one pointer and stride, so that a warp with nodes of both kinds (every
// warp of a 2D leaf) walks one loop.
template <typename T>
struct LeafRow {
  const T* p;   // entry j at p[j ld]
  int64_t ld;
  int r;        // row of Y
  bool edge, negate;
  __device__ LeafRow(const LeafConsts& k, int node, const T* Xl, int xrows) {
    if constexpr (sizeof(T) == sizeof(double)) {
      const int pr = k.prow[node];
      edge = pr >= 0;
      negate = !edge;
      r = edge ? 0 : k.iidx[node];
      ld = edge ? k.ne : xrows;
      p = edge ? k.P + pr : Xl + r;
    } else {
      edge = negate = false;
      r = node;
      ld = xrows;
      p = Xl + r;
    }
  }
  __device__ T at(int j) const { return p[j * ld]; }
};

// u = Y g + v at a leaf's nodes, a thread per node and NC right-hand sides, so
// that an entry of Y serves NC multiply-adds.  Bound by the FP64 pipe (385 us
// for 4096 complex leaves of 256 x 56, of which the pipe needs 392 at its nominal
// rate; eight real right-hand sides 784, and 1533 while a warp walked its boundary
// and interior nodes one after the other).
template <typename T, int NC>
__global__ void __launch_bounds__(256) k_leaf_output(LeafConsts k, int64_t nl, int nrhs, const T* X, const T* xp,
                                                     const T* g, T* u, bool iti) {
  const int64_t total = (int64_t)((nrhs + NC - 1) / NC) * nl * k.npts;
  const int xrows = iti ? k.npts : k.ni;
  for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < total;
       e += (int64_t)gridDim.x * blockDim.x) {
    const int node = (int)(e % k.npts);
    const int64_t lc = e / k.npts;
    const int64_t leaf = lc % nl;
    const int c0 = (int)(lc / nl) * NC;
    const T* gl = g + (leaf * nrhs + c0) * (int64_t)k.nb;
    const T* Xl = X + leaf * (int64_t)xrows * (k.nb + 1);
    int go[NC];   // columns beyond the last repeat it
    T acc[NC];
#pragma unroll
    for (int c = 0; c < NC; ++c) go[c] = min(c, nrhs - 1 - c0) * k.nb;
    const LeafRow<T> row(k, node, Xl, xrows);
#pragma unroll
    for (int c = 0; c < NC; ++c)
      acc[c] = row.edge ? T(0.0)
               : xp     ? xp[(leaf * nrhs + min(c0 + c, nrhs - 1)) * (int64_t)xrows + row.r]
                        : Xl[row.r + (int64_t)k.nb * xrows];
#pragma unroll 4
    for (int j = 0; j < k.nb; ++j) {
      const T x = row.at(j);
#pragma unroll
      for (int c = 0; c < NC; ++c) acc[c] = fmac(acc[c], x, gl[go[c] + j]);
    }
    if (row.negate) {
#pragma unroll
      for (int c = 0; c < NC; ++c) acc[c] = -acc[c];
    }
#pragma unroll
    for (int c = 0; c < NC; ++c)
      if (c0 + c < nrhs) u[((c0 + c) * nl + leaf) * k.npts + node] = acc[c];
  }
}

template <typename T>
cudaError_t leaf_output(const LeafConsts& k, int64_t nl, int nrhs, const T* X, const T* xp, const T* g,
                        T* u, bool iti, cudaStream_t st, Prof* pf) {
  const double F = sizeof(T) == sizeof(cplx) ? 8.0 : 2.0;
  if (pf) pf->begin(st);
  // Whole groups of four or three real right-hand sides when seven CTAs per SM
  // are left to hide the loads; else, and for complex data, one by one (us, nodes x
  // right-hand sides, one by one / in fours or threes: real 1048576 x 8 834 / 782 and x 3
  // 324 / 301, 262144 x 16 406 / 397, 32768 x 24 295 / 332, 1728 x 8 16 / 33; x 5, in
  // threes, 1048576 524 / 590; complex 262144 x 8 772 / 803, 65536 x 8 205 / 238)
  int nc = 1;
  if constexpr (sizeof(T) == sizeof(double)) nc = nrhs % 4 == 0 ? 4 : nrhs % 3 == 0 ? 3 : 1;
  if (nl * k.npts * (nrhs / nc) < 262144) nc = 1;
  const int grid = grid_for((int64_t)(nrhs / nc) * nl * k.npts);
  if (nc == 1) k_leaf_output<T, 1><<<grid, 256, 0, st>>>(k, nl, nrhs, X, xp, g, u, iti);
  if constexpr (sizeof(T) == sizeof(double)) {
    if (nc == 3) k_leaf_output<T, 3><<<grid, 256, 0, st>>>(k, nl, nrhs, X, xp, g, u, iti);
    if (nc == 4) k_leaf_output<T, 4><<<grid, 256, 0, st>>>(k, nl, nrhs, X, xp, g, u, iti);
  }
  if (pf) pf->end(K_DOWN, F * (double)nrhs * nl * k.npts * k.nb, st);
  return cudaGetLastError();
}

template <typename T>
__global__ void k_copy_block(const T* src, int64_t sstride, int sld, T* dst, int64_t dstride, int dld,
                             int m, int ncols, int batch) {
  const int64_t per = (int64_t)m * ncols;
  for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < per * batch;
       e += (int64_t)gridDim.x * blockDim.x) {
    const int64_t b = e / per;
    const int rc = (int)(e % per);
    const int i = rc % m, j = rc / m;
    dst[b * dstride + i + (int64_t)j * dld] = src[b * sstride + i + (int64_t)j * sld];
  }
}

template <typename T>
cudaError_t copy_block(const T* src, int64_t sstride, int sld, T* dst, int64_t dstride, int dld, int m,
                       int ncols, int batch, cudaStream_t st, Prof* pf) {
  if (pf) pf->begin(st);
  k_copy_block<T><<<grid_for((int64_t)m * ncols * batch), 256, 0, st>>>(src, sstride, sld, dst, dstride,
                                                                          dld, m, ncols, batch);
  if (pf) pf->end(K_OTHER, 0.0, st);
  return cudaGetLastError();
}

template <typename T>
__global__ void k_scale_copy(const T* src, T* dst, int64_t n, double alpha) {
  for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < n;
       e += (int64_t)gridDim.x * blockDim.x)
    dst[e] = scale(src[e], alpha);
}

template <typename T>
cudaError_t scale_copy(const T* src, T* dst, int64_t n, double alpha, cudaStream_t st, Prof* pf) {
  if (pf) pf->begin(st);
  k_scale_copy<T><<<grid_for(n), 256, 0, st>>>(src, dst, n, alpha);
  if (pf) pf->end(K_OTHER, 0.0, st);
  return cudaGetLastError();
}

// ------------------------------------------------- grouped downward pass ----

// gint = -(X_C gpar + x) for the rows of all merges of a task and one right-hand
// side: as k_down_gint, with eight warps a CTA of which tk.cg share 32 rows.
template <typename T>
__global__ void __launch_bounds__(256) k_down_gint_group(DownGroup<T> grp) {
  __shared__ T part[8][33];
  const int lane = threadIdx.x, w = threadIdx.y;
  const int64_t tile = blockIdx.x;
  int ti = 0;
  while (ti + 1 < grp.n && grp.t[ti + 1].tile0 <= tile) ++ti;
  const DownTask<T>& tk = grp.t[ti];
  const int CG = tk.cg, cg = w & (CG - 1), n_int = tk.n_int, n_ext = tk.n_ext, nrhs = tk.nrhs;
  const int64_t rows = (int64_t)tk.nmerge * n_int, rtiles = down_task_row_tiles(tk);
  const int64_t loc = tile - tk.tile0;
  const int64_t R = (loc % rtiles * (8 / CG) + w / CG) * 32 + lane;
  const int c = (int)(loc / rtiles);
  const bool live = R < rows;
  const int64_t b = live ? R / n_int : 0;
  const int r = live ? (int)(R % n_int) : 0;
  const T* x = tk.X + b * (int64_t)n_int * (n_ext + 1) + r;
  const T* g = tk.gpar + (b * nrhs + c) * (int64_t)n_ext;
  T acc = T(0.0);
  if (live) {
#pragma unroll 4
    for (int j = cg; j < n_ext; j += CG) acc = fmac(acc, x[(int64_t)j * n_int], g[j]);
  }
  part[w][lane] = acc;
  __syncthreads();
  if (cg == 0 && live) {
    T s = x[(int64_t)n_ext * n_int];
    for (int k = 0; k < CG; ++k) s = s + part[w + k][lane];
    tk.gint[(b * nrhs + c) * (int64_t)n_int + r] = -s;
  }
}

template <typename T>
__global__ void k_down_children_group(DownGroup<T> grp) {
  for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < grp.elems;
       e += (int64_t)gridDim.x * blockDim.x) {
    int ti = 0;
    while (ti + 1 < grp.n && grp.t[ti + 1].elem0 <= e) ++ti;
    const DownTask<T>& tk = grp.t[ti];
    const int64_t le = e - tk.elem0;
    const int64_t per_child = (int64_t)tk.nbc * tk.nrhs;
    const int64_t cidx = le / per_child;
    const int rc = (int)(le % per_child);
    const int i = rc % tk.nbc, c = rc / tk.nbc;
    const int k = (int)(cidx % tk.nch);
    const int64_t b = cidx / tk.nch;
    const int ei = tk.ext[k * tk.nbc + i];
    T v;
    if (ei >= 0) v = tk.gpar[b * (int64_t)tk.n_ext * tk.nrhs + ei + (int64_t)c * tk.n_ext];
    else v = tk.gint[b * (int64_t)tk.n_int * tk.nrhs + tk.var[k * tk.nbc + i] + (int64_t)c * tk.n_int];
    tk.gchild[le] = v;
  }
}

template <typename T>
cudaError_t down_level_group(const DownGroup<T>& grp, cudaStream_t st) {
  if (grp.n <= 0) return cudaSuccess;
  if (grp.tiles > 0) k_down_gint_group<T><<<(unsigned)grp.tiles, dim3(32, 8), 0, st>>>(grp);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  if (grp.elems > 0) k_down_children_group<T><<<grid_for(grp.elems), 256, 0, st>>>(grp);
  return cudaGetLastError();
}

// u = Y g + v with the build-time v, for the leaves of every task.
template <typename T>
__global__ void k_leaf_output_group(LeafGroup<T> grp) {
  for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < grp.elems;
       e += (int64_t)gridDim.x * blockDim.x) {
    int ti = 0;
    while (ti + 1 < grp.n && grp.t[ti + 1].elem0 <= e) ++ti;
    const LeafTask<T>& tk = grp.t[ti];
    const LeafConsts& k = tk.k;
    const int64_t le = e - tk.elem0;
    const int node = (int)(le % k.npts);
    const int64_t lc = le / k.npts;
    const int64_t leaf = lc % tk.nl;
    const int c = (int)(lc / tk.nl);
    const int xrows = grp.iti ? k.npts : k.ni;
    const T* gl = tk.g + (leaf * tk.nrhs + c) * (int64_t)k.nb;
    const T* Xl = tk.X + leaf * (int64_t)xrows * (k.nb + 1);
    const LeafRow<T> row(k, node, Xl, xrows);
    T acc = row.edge ? T(0.0) : Xl[row.r + (int64_t)k.nb * xrows];
#pragma unroll 4
    for (int j = 0; j < k.nb; ++j) acc = fmac(acc, row.at(j), gl[j]);
    if (row.negate) acc = -acc;
    tk.u[le] = acc;
  }
}

template <typename T>
cudaError_t leaf_output_group(const LeafGroup<T>& grp, cudaStream_t st) {
  if (grp.n <= 0 || grp.elems <= 0) return cudaSuccess;
  k_leaf_output_group<T><<<grid_for(grp.elems), 256, 0, st>>>(grp);
  return cudaGetLastError();
}

#define HPS_KINST(T)                                                                                  \
  template cudaError_t leaf_particular_rhs<T>(const LeafConsts&, int64_t, int, const T*, T*, bool,    \
                                              cudaStream_t, Prof*);                                   \
  template cudaError_t merge_gather<T>(const T*, int64_t, int, int, int, int, int, const int*,        \
                                       const int*, const int*, bool, T*, T*, T*, cudaStream_t, Prof*); \
  template cudaError_t merge_gather_h<T>(const T*, int, int, int, int, int, int, const int*,          \
                                         const int*, const int*, bool, T*, T*, cudaStream_t, Prof*);  \
  template cudaError_t down_level<T>(const T*, const T*, const T*, int, int, int, int, int, int,      \
                                     const int*, const int*, T*, T*, cudaStream_t, Prof*);            \
  template cudaError_t leaf_output<T>(const LeafConsts&, int64_t, int, const T*, const T*, const T*,  \
                                      T*, bool, cudaStream_t, Prof*);                                 \
  template cudaError_t copy_block<T>(const T*, int64_t, int, T*, int64_t, int, int, int, int,         \
                                     cudaStream_t, Prof*);                                            \
  template cudaError_t scale_copy<T>(const T*, T*, int64_t, double, cudaStream_t, Prof*);                 \
  template cudaError_t down_gint<T>(const T*, const T*, const T*, int, int, int, int, T*, cudaStream_t,     \
                                    Prof*);                                                                 \
  template cudaError_t down_children<T>(const T*, const T*, int, int, int, int, int, int, const int*,       \
                                        const int*, T*, cudaStream_t, Prof*);                                 \
  template cudaError_t down_level_group<T>(const DownGroup<T>&, cudaStream_t);                               \
  template cudaError_t leaf_output_group<T>(const LeafGroup<T>&, cudaStream_t);

HPS_KINST(double)
HPS_KINST(cplx)

}  // namespace hps

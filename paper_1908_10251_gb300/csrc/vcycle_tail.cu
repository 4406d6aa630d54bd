// The coarse end of the V-cycle in one kernel: levels 1 .. top and the exact solve on level 0, for levels
// whose vectors fit in shared memory.
//
// Every operation of the cycle acts on each column of the block by itself, so a block takes C columns
// (float32: 4, one 16-byte chunk; float64: 1, its pipe being the scarce part) through all levels with
// nothing but block barriers between the passes.  As separate launches these levels are 4 to 8 kernels
// each that last one chain of dependent loads (3 to 4 us with programmatic launch) whatever their size.
// Here a pass over 961 rows takes about 2 us in float64, bound by the 2 FMA a clock of its one SM, and
// 0.5 us in float32, bound by the shared-memory gathers; the static matrices in L1 beforehand made no
// difference.  Each operation takes the products and sums of the kernels that the larger levels use, in
// their order, so a level gives the same bits on either path.
#include "common.cuh"
#include "kernels.cuh"

#include <algorithm>

namespace pasm {
namespace {

constexpr int kTailThreads = 1024;
constexpr int kParts = 8;   // parts of the coarse product's inner dimension, as in dense_mm
constexpr int kPartThreads = kTailThreads / kParts;

template <typename T> struct TailCols;
template <> struct TailCols<float> { static constexpr int v = 4; };
template <> struct TailCols<double> { static constexpr int v = 1; };

template <typename T, int C>
__device__ __forceinline__ void lds(const T* p, T (&x)[C]) {
  if constexpr (C * sizeof(T) == 16) {
    Vec16<T>::load(p, x);
  } else {
#pragma unroll
    for (int v = 0; v < C; ++v) x[v] = p[v];
  }
}
template <typename T, int C>
__device__ __forceinline__ void put(T* p, const T (&x)[C]) {
  if constexpr (C * sizeof(T) == 16) {
    Vec16<T>::store(p, x);
  } else {
#pragma unroll
    for (int v = 0; v < C; ++v) p[v] = x[v];
  }
}

// n x C columns of a global n x ldk block into shared memory, and back
template <typename T, int C>
__device__ __forceinline__ void fetch(const T* g, T* s, int n, int ldk) {
  for (int i = threadIdx.x; i < n; i += kTailThreads) {
    T x[C];
    if constexpr (C * sizeof(T) == 16) {
      ldg16<T>(g + (size_t)i * ldk, x);
    } else {
#pragma unroll
      for (int v = 0; v < C; ++v) x[v] = ld1(g + (size_t)i * ldk + v);
    }
    put<T, C>(s + i * C, x);
  }
}
template <typename T, int C>
__device__ __forceinline__ void flush(const T* s, T* g, int n, int ldk) {
  for (int i = threadIdx.x; i < n; i += kTailThreads) {
    T x[C];
    lds<T, C>(s + i * C, x);
    put<T, C>(g + (size_t)i * ldk, x);
  }
}

// acc = row of S X, X in shared memory: entries in CSR order, the loads of four ahead of their products
template <typename T, int C>
__device__ __forceinline__ void row_product(const TailCsr<T>& S, const T* v, const T* X, int row, T (&acc)[C]) {
#pragma unroll
  for (int c = 0; c < C; ++c) acc[c] = T(0);
  int p = __ldg(S.rp + row);
  const int p1 = __ldg(S.rp + row + 1);
  for (; p < p1; p += 4) {
    int j[4];
    T a[4];
#pragma unroll
    for (int u = 0; u < 4; ++u)
      if (p + u < p1) { j[u] = __ldg(S.ci + p + u); a[u] = __ldg(v + p + u); }
#pragma unroll
    for (int u = 0; u < 4; ++u)
      if (p + u < p1) {
        T x[C];
        lds<T, C>(X + j[u] * C, x);
#pragma unroll
        for (int c = 0; c < C; ++c) acc[c] = fma(a[u], x[c], acc[c]);
      }
  }
}

template <typename T, int C>
__device__ __forceinline__ void sweep(const TailLevel<T>& L, T omega, const T* F, const T* X, T* out) {
  for (int i = threadIdx.x; i < L.n; i += kTailThreads) {
    T acc[C], f[C], x[C], r[C];
    row_product<T, C>(L.A, L.A.v, X, i, acc);
    lds<T, C>(F + i * C, f);
    lds<T, C>(X + i * C, x);
    const T w = omega * __ldg(L.dinv + i);
#pragma unroll
    for (int c = 0; c < C; ++c) r[c] = fma(w, f[c] - acc[c], x[c]);
    put<T, C>(out + i * C, r);
  }
}

template <typename T>
__global__ void __launch_bounds__(kTailThreads) k_vcycle_tail(const __grid_constant__ TailArgs<T> a) {
  constexpr int C = TailCols<T>::v;
  constexpr bool F32 = sizeof(T) == 4;
  extern __shared__ __align__(16) unsigned char tail_smem[];
  T* const s = reinterpret_cast<T*>(tail_smem);
  const int col = blockIdx.x * C;
  auto F = [&](int l) { return s + a.off[l]; };
  auto E = [&](int l) { return s + a.off[l] + a.lv[l].n * C; };
  auto W = [&](int l) { return s + a.off[l] + 2 * a.lv[l].n * C; };
  // the iterate is in W after an odd number of sweeps that go from one buffer to the other
  const int first = a.nu_pre < 1 ? 0 : (F32 && a.nu_pre >= 2 ? 2 : 1);
  const bool flip = ((max(a.nu_pre, first) - first) & 1) != 0;
  pdl_trigger();
  pdl_wait();
  fetch<T, C>(a.gF + col, F(a.top), a.lv[a.top].n, a.ldk);
  __syncthreads();
  for (int l = a.top; l >= 1; --l) {
    const TailLevel<T>& L = a.lv[l];
    T *cur = E(l), *tmp = W(l);
    for (int i = threadIdx.x; i < L.n; i += kTailThreads) {
      T f[C], r[C];
      lds<T, C>(F(l) + i * C, f);
      const T w = a.omega * __ldg(L.dinv + i);
      if (first == 2) {   // two sweeps from zero, as jacobi2_zero
        T acc[C];
        row_product<T, C>(L.A, L.A.w, F(l), i, acc);
#pragma unroll
        for (int c = 0; c < C; ++c) r[c] = w * (T(2) * f[c] - acc[c]);
      } else {
#pragma unroll
        for (int c = 0; c < C; ++c) r[c] = first == 1 ? w * f[c] : T(0);
      }
      put<T, C>(cur + i * C, r);
    }
    __syncthreads();
    for (int q = first; q < a.nu_pre; ++q) {
      sweep<T, C>(L, a.omega, F(l), cur, tmp);
      __syncthreads();
      T* t = cur; cur = tmp; tmp = t;
    }
    const int nc = a.lv[l - 1].n;
    if (F32) {   // as restrict_first
      for (int i = threadIdx.x; i < nc; i += kTailThreads) {
        T rf[C], qe[C];
        row_product<T, C>(L.R, L.R.v, F(l), i, rf);
        row_product<T, C>(L.RA, L.RA.v, cur, i, qe);
#pragma unroll
        for (int c = 0; c < C; ++c) rf[c] = rf[c] - qe[c];
        put<T, C>(F(l - 1) + i * C, rf);
      }
    } else {
      for (int i = threadIdx.x; i < L.n; i += kTailThreads) {
        T acc[C], f[C];
        row_product<T, C>(L.A, L.A.v, cur, i, acc);
        lds<T, C>(F(l) + i * C, f);
#pragma unroll
        for (int c = 0; c < C; ++c) f[c] = f[c] - acc[c];
        put<T, C>(tmp + i * C, f);
      }
      __syncthreads();
      for (int i = threadIdx.x; i < nc; i += kTailThreads) {
        T acc[C];
        row_product<T, C>(L.R, L.R.v, tmp, i, acc);
        put<T, C>(F(l - 1) + i * C, acc);
      }
    }
    __syncthreads();
  }
  // E_0 = A_H^{-1} F_0 (the inverse is symmetric bit for bit, so its rows are read as columns), the
  // order of dense_mm: interleaved parts, then the parts' sums in order
  const int n0 = a.lv[0].n, part = threadIdx.x / kPartThreads;
  T* const red = s + a.off_red;
  const T* const f0 = F(0);
  for (int i0 = threadIdx.x % kPartThreads; i0 < n0; i0 += 2 * kPartThreads) {
    const int i1 = min(i0 + kPartThreads, n0 - 1);
    T s0[C], s1[C];
#pragma unroll
    for (int c = 0; c < C; ++c) s0[c] = s1[c] = T(0);
#pragma unroll 8
    for (int j = part; j < n0; j += kParts) {
      const T d0 = __ldg(a.Ainv + (size_t)j * n0 + i0), d1 = __ldg(a.Ainv + (size_t)j * n0 + i1);
      T x[C];
      lds<T, C>(f0 + j * C, x);
#pragma unroll
      for (int c = 0; c < C; ++c) { s0[c] = fma(d0, x[c], s0[c]); s1[c] = fma(d1, x[c], s1[c]); }
    }
    put<T, C>(red + (part * n0 + i0) * C, s0);
    if (i0 + kPartThreads < n0) put<T, C>(red + (part * n0 + i1) * C, s1);
  }
  __syncthreads();
  for (int q = threadIdx.x; q < n0 * C; q += kTailThreads) {
    T x = red[q];
#pragma unroll
    for (int p = 1; p < kParts; ++p) x += red[p * n0 * C + q];
    E(0)[q] = x;
  }
  __syncthreads();
  const T* ec = E(0);
  for (int l = 1; l <= a.top; ++l) {
    const TailLevel<T>& L = a.lv[l];
    T *cur = flip ? W(l) : E(l), *tmp = flip ? E(l) : W(l);
    for (int i = threadIdx.x; i < L.n; i += kTailThreads) {
      T acc[C], x[C];
      row_product<T, C>(L.P, L.P.v, ec, i, acc);
      lds<T, C>(cur + i * C, x);
#pragma unroll
      for (int c = 0; c < C; ++c) x[c] = x[c] + acc[c];
      put<T, C>(cur + i * C, x);
    }
    __syncthreads();
    for (int q = 0; q < a.nu_post; ++q) {
      sweep<T, C>(L, a.omega, F(l), cur, tmp);
      __syncthreads();
      T* t = cur; cur = tmp; tmp = t;
    }
    ec = cur;
  }
  flush<T, C>(ec, a.gE + col, a.lv[a.top].n, a.ldk);
}

// Offsets of the levels' vectors in shared memory; bytes in all.
template <typename T>
size_t tail_layout(TailArgs<T>& a) {
  size_t at = 0;
  for (int l = 0; l <= a.top; ++l) {
    a.off[l] = (int)at;
    at += (l == 0 ? 2 : 3) * (size_t)a.lv[l].n * TailCols<T>::v;
  }
  a.off_red = (int)at;
  at += (size_t)kParts * a.lv[0].n * TailCols<T>::v;
  return at * sizeof(T);
}

}  // namespace

template <typename T>
bool vcycle_tail_fits(const int* n, int top) {
  if (top < 1 || top >= kTailLevels) return false;
  TailArgs<T> a = {};
  a.top = top;
  for (int l = 0; l <= top; ++l) a.lv[l].n = n[l];
  return tail_layout<T>(a) <= kTailSmem;
}

cudaError_t vcycle_tail_prepare() {
  cudaError_t e = allow_dynamic_smem((const void*)k_vcycle_tail<float>, kTailSmem);
  if (e == cudaSuccess) e = allow_dynamic_smem((const void*)k_vcycle_tail<double>, kTailSmem);
  return e;
}

template <typename T>
void vcycle_tail(const Launch& L, TailArgs<T> a) {
  const size_t smem = tail_layout<T>(a);
  {
    // matrices once (the second sweep from zero has values of its own), what leaves and enters the kernel once
    const bool f32 = sizeof(T) == 4, two = f32 && a.nu_pre >= 2;
    const double w = sizeof(T), ldk = a.ldk, n0 = a.lv[0].n;
    const int sweeps = std::max(0, a.nu_pre - (two ? 2 : 1)) + a.nu_post;
    const bool own = sweeps > 0 || !f32;   // products with A's own values
    double bytes = 2.0 * a.lv[a.top].n * ldk * w + n0 * n0 * w, flops = 2.0 * n0 * n0 * ldk;
    for (int l = 1; l <= a.top; ++l) {
      const TailLevel<T>& v = a.lv[l];
      const double n = v.n, nc = a.lv[l - 1].n, A = (double)v.nnz_A, R = (double)v.nnz_R, RA = (double)v.nnz_RA,
                   P = (double)v.nnz_P, row = 4.0, entry = 4.0 + w;
      if (own || two) bytes += (n + 1) * row + A * (4.0 + w * ((own ? 1 : 0) + (two ? 1 : 0)));
      bytes += (nc + 1) * row + R * entry + (n + 1) * row + P * entry;
      if (f32) bytes += (nc + 1) * row + RA * entry;
      if (a.nu_pre > 0 || a.nu_post > 0) bytes += n * w;
      flops += ldk * (sweeps * (2.0 * A + 3.0 * n) + (two ? 2.0 * A + 3.0 * n : a.nu_pre >= 1 ? n : 0.0) +
                      (f32 ? 2.0 * (R + RA) + nc : 2.0 * (A + R) + n) + 2.0 * P + n);
    }
    L.rows(a.lv[a.top].n);
    L.begin(KC_DENSE, bytes, flops);
  }
  launch(L.spread(a.ldk / TailCols<T>::v), k_vcycle_tail<T>, a.ldk / TailCols<T>::v, kTailThreads, smem, a);
  L.bump();
}

template bool vcycle_tail_fits<float>(const int*, int);
template bool vcycle_tail_fits<double>(const int*, int);
template void vcycle_tail<float>(const Launch&, TailArgs<float>);
template void vcycle_tail<double>(const Launch&, TailArgs<double>);

}  // namespace pasm

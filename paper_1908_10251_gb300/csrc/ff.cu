// Float64-accuracy kernels of the mixed-precision path in double-float
// arithmetic (ff.cuh): the outer residuals of the defect correction
// (Algorithm 1 step 1), the bordering products (the bordered matrix form of
// Section 3.1), the transfer chains and the update.  Vectors that are gathered
// through a sparse matrix are kept as (hi, lo) float pairs ("ff", 8 bytes per
// entry like float64; two columns make one 16-byte chunk hi, hi, lo, lo, the
// operands of the packed float32 instructions): the multigrid iterate u~, its products A u~ and M u~,
// the intermediate levels of the transfer chains, and the state U itself
// between steps (its float64 form is rebuilt when read).  Matrix values are
// split once at setup; a matrix whose values are all float32 skips the
// low-part products.  The coarse vectors and the eigenvalues stay float64.
// Results carry about 2^-46 relative to the sum of the magnitudes of their
// terms (float64: 2^-53), far below what the float32 V-cycles of the mixed
// path resolve.
#include "common.cuh"
#include "ff.cuh"
#include "kernels.cuh"

#include <algorithm>

namespace pasm {
namespace {

constexpr int kBlock = 256;
// The residual and transfer kernels are held to 64 registers (four 256-thread
// blocks per SM): the extra warps hide more gather latency than the few
// spilled values cost (outer_rhs 0.64 -> 0.59 ms, outer_res 0.34 -> 0.28,
// spmm 0.52 -> 0.48 at h = 1/1024, k = 64).  The bordering and update kernels
// were slower that way and keep the compiler's choice.
constexpr int kMinBlocksGather = 4;

struct Geo {
  int tpr, ch;
};
// Row groups as in the float64 kernels: 16-byte chunks of 2 columns; pref as
// in the float64 geometry (chunks per thread chosen by the autotuner).
Geo geometry_ff(int ldk, int pref) {
  const int chunks = ldk / 2;
  Geo g;
  if (chunks <= 32) { g.tpr = chunks; g.ch = 1; }
  else { g.tpr = 32; g.ch = chunks / 32; }
  if ((pref == 1 || pref == 2 || pref == 4 || pref == 8) && chunks % pref == 0 && chunks / pref <= 32) {
    g.tpr = chunks / pref;
    g.ch = pref;
  }
  return g;
}

// Row blocks one thread block walks (1 or 4, chosen by the autotuner; 1 when untuned).
static int ff_rows(const Launch& L) { return L.rpt > 0 ? L.rpt : 1; }

#define PASM_FF_DISPATCH(ch, ...)                          \
  switch (ch) {                                            \
    case 1: { constexpr int CH = 1; __VA_ARGS__; } break;  \
    case 2: { constexpr int CH = 2; __VA_ARGS__; } break;  \
    case 4: { constexpr int CH = 4; __VA_ARGS__; } break;  \
    case 8: { constexpr int CH = 8; __VA_ARGS__; } break;  \
    default: break;                                        \
  }

// Two consecutive entries (columns col, col + 1) of row i of a block vector,
// as packed hi and lo parts: from a pair chunk directly, from float64 by splitting.
template <bool FF>
__device__ __forceinline__ void load_pair(const double* __restrict__ X, size_t off, ff2& h, ff2& l) {
  if (FF) {
    asm volatile("ld.global.v2.u64 {%0, %1}, [%2];" : "=l"(h), "=l"(l) : "l"(X + off));
  } else {
    double t[2];
    ldg16<double>(X + off, t);
    float h0, l0, h1, l1;
    ff_split(t[0], h0, l0);
    ff_split(t[1], h1, l1);
    h = ff2_pack(h0, h1);
    l = ff2_pack(l0, l1);
  }
}

// The first row of a row group, before pdl_wait: its entries on their way to the SM.
template <typename VT>
__device__ __forceinline__ void prefetch_row(const int* __restrict__ rp, const int* __restrict__ ci,
                                             const VT* __restrict__ av, int row, int n) {
  if (row >= n) return;
  const int p = __ldg(rp + row);
  if (p >= __ldg(rp + row + 1)) return;
  prefetch_line(ci + p);
  prefetch_line(av + p);
}

// acc += a_p X[ci_p, cols] for the N entries p .. p+N-1: index and value loads,
// then the N row gathers, then the double-float products.
template <int CH, int N, bool FFIN, bool EX>
__device__ __forceinline__ void gather_group_ff(const int* __restrict__ ci, const float2* __restrict__ av,
                                                const double* __restrict__ X, int p, int lane, int tpr, int ldk,
                                                ff2 (&hi)[CH], ff2 (&lo)[CH]) {
  int j[N];
  float2 a[N];
#pragma unroll
  for (int u = 0; u < N; ++u) {
    j[u] = __ldg(ci + p + u);
    a[u] = __ldg(av + p + u);
  }
  ff2 xh[N][CH], xl[N][CH];
#pragma unroll
  for (int u = 0; u < N; ++u)
#pragma unroll
    for (int c = 0; c < CH; ++c) load_pair<FFIN>(X, (size_t)j[u] * ldk + (c * tpr + lane) * 2, xh[u][c], xl[u][c]);
#pragma unroll
  for (int u = 0; u < N; ++u) {
    const ff2 ah = ff2_pack(a[u].x, a[u].x), na = ff2_pack(-a[u].x, -a[u].x), al = ff2_pack(a[u].y, a[u].y);
#pragma unroll
    for (int c = 0; c < CH; ++c) {
      if (EX) ff2_mac_exact(hi[c], lo[c], ah, na, xh[u][c], xl[u][c]);
      else ff2_mac(hi[c], lo[c], ah, na, al, xh[u][c], xl[u][c]);
    }
  }
}

// One row of S X in double-float (groups of 4 entries, then an exact remainder group);
// EX: S's values are float32 (no low parts).
template <int CH, bool FFIN, bool EX = false>
__device__ __forceinline__ void gather_row_ff(const int* __restrict__ rp, const int* __restrict__ ci,
                                              const float2* __restrict__ av, const double* __restrict__ X, int row,
                                              int lane, int tpr, int ldk, ff2 (&hi)[CH], ff2 (&lo)[CH]) {
#pragma unroll
  for (int c = 0; c < CH; ++c) hi[c] = lo[c] = 0;
  int p = __ldg(rp + row);
  const int p1 = __ldg(rp + row + 1);
  for (; p + 4 <= p1; p += 4) gather_group_ff<CH, 4, FFIN, EX>(ci, av, X, p, lane, tpr, ldk, hi, lo);
  const int rem = p1 - p;
  if (rem == 3) gather_group_ff<CH, 3, FFIN, EX>(ci, av, X, p, lane, tpr, ldk, hi, lo);
  else if (rem == 2) gather_group_ff<CH, 2, FFIN, EX>(ci, av, X, p, lane, tpr, ldk, hi, lo);
  else if (rem == 1) gather_group_ff<CH, 1, FFIN, EX>(ci, av, X, p, lane, tpr, ldk, hi, lo);
#pragma unroll
  for (int c = 0; c < CH; ++c) ff2_norm(hi[c], lo[c]);
}

// A X and M X together over M's pattern (am: A's and M's split values per
// entry, a = 0 where A has no entry): one gather of each row of X serves both
// products.  Each accumulator sees the same terms in the same order as the
// separate gathers (A's entries in M's column order).
template <int CH, int N, bool FFIN, bool AEX>
__device__ __forceinline__ void gather_group_am(const int* __restrict__ ci, const float4* __restrict__ am,
                                                const double* __restrict__ X, int p, int lane, int tpr, int ldk,
                                                ff2 (&ah)[CH], ff2 (&al)[CH], ff2 (&mh)[CH], ff2 (&ml)[CH]) {
  int j[N];
  float4 w[N];
#pragma unroll
  for (int u = 0; u < N; ++u) {
    j[u] = __ldg(ci + p + u);
    w[u] = __ldg(am + p + u);
  }
  ff2 xh[N][CH], xl[N][CH];
#pragma unroll
  for (int u = 0; u < N; ++u)
#pragma unroll
    for (int c = 0; c < CH; ++c) load_pair<FFIN>(X, (size_t)j[u] * ldk + (c * tpr + lane) * 2, xh[u][c], xl[u][c]);
#pragma unroll
  for (int u = 0; u < N; ++u) {
    {
      const ff2 w0 = ff2_pack(w[u].z, w[u].z), wn = ff2_pack(-w[u].z, -w[u].z), w1 = ff2_pack(w[u].w, w[u].w);
#pragma unroll
      for (int c = 0; c < CH; ++c) ff2_mac(mh[c], ml[c], w0, wn, w1, xh[u][c], xl[u][c]);
    }
    if (w[u].x != 0.f) {
      const ff2 w0 = ff2_pack(w[u].x, w[u].x), wn = ff2_pack(-w[u].x, -w[u].x), w1 = ff2_pack(w[u].y, w[u].y);
#pragma unroll
      for (int c = 0; c < CH; ++c) {
        if (AEX) ff2_mac_exact(ah[c], al[c], w0, wn, xh[u][c], xl[u][c]);
        else ff2_mac(ah[c], al[c], w0, wn, w1, xh[u][c], xl[u][c]);
      }
    }
  }
}

template <int CH, bool FFIN, bool AEX>
__device__ __forceinline__ void gather_row_am(const int* __restrict__ rp, const int* __restrict__ ci,
                                              const float4* __restrict__ am, const double* __restrict__ X, int row,
                                              int lane, int tpr, int ldk, ff2 (&ah)[CH], ff2 (&al)[CH],
                                              ff2 (&mh)[CH], ff2 (&ml)[CH]) {
#pragma unroll
  for (int c = 0; c < CH; ++c) ah[c] = al[c] = mh[c] = ml[c] = 0;
  int p = __ldg(rp + row);
  const int p1 = __ldg(rp + row + 1);
  for (; p + 4 <= p1; p += 4) gather_group_am<CH, 4, FFIN, AEX>(ci, am, X, p, lane, tpr, ldk, ah, al, mh, ml);
  const int rem = p1 - p;
  if (rem == 3) gather_group_am<CH, 3, FFIN, AEX>(ci, am, X, p, lane, tpr, ldk, ah, al, mh, ml);
  else if (rem == 2) gather_group_am<CH, 2, FFIN, AEX>(ci, am, X, p, lane, tpr, ldk, ah, al, mh, ml);
  else if (rem == 1) gather_group_am<CH, 1, FFIN, AEX>(ci, am, X, p, lane, tpr, ldk, ah, al, mh, ml);
#pragma unroll
  for (int c = 0; c < CH; ++c) {
    ff2_norm(ah[c], al[c]);
    ff2_norm(mh[c], ml[c]);
  }
}

// Store two entries as a pair chunk or, rounded, as float64.
template <bool FF>
__device__ __forceinline__ void store_pair(double* __restrict__ out, size_t off, ff2 h, ff2 l) {
  if (FF) {
    *reinterpret_cast<ulonglong2*>(out + off) = make_ulonglong2(h, l);
  } else {
    float h0, h1, l0, l1;
    ff2_unpack(h, h0, h1);
    ff2_unpack(l, l0, l1);
    *reinterpret_cast<double2*>(out + off) = make_double2(ff_to_double(h0, l0), ff_to_double(h1, l1));
  }
}

// Fd = lam .* (M U) stored as (hi, lo) float pairs, R = Fd - A U as float32
// (U given as float pairs).
template <int CH, bool AEX>
__global__ void __launch_bounds__(kBlock, kMinBlocksGather)
    k_outer_rhs_res_ff(int n, const int* __restrict__ arp, const int* __restrict__ aci, const float2* __restrict__ aval,
                       const int* __restrict__ mrp, const int* __restrict__ mci, const float2* __restrict__ mval,
                       const double* __restrict__ lam, const double* __restrict__ U, float2* __restrict__ Fd,
                       float* __restrict__ R, int ldk, int tpr, int rpt) {
  pdl_trigger();
  prefetch_row(mrp, mci, mval, blockIdx.x * rpt * (kBlock / tpr) + threadIdx.x / tpr, n);
  prefetch_row(arp, aci, aval, blockIdx.x * rpt * (kBlock / tpr) + threadIdx.x / tpr, n);
  pdl_wait();
  // the eigenvalues as pair chunks, split once per block rather than once per entry
  extern __shared__ ulonglong2 lsp[];  // [ldk / 2]
  for (int t = threadIdx.x; t < ldk / 2; t += blockDim.x) load_pair<false>(lam, 2 * t, lsp[t].x, lsp[t].y);
  __syncthreads();
  const int rpb = kBlock / tpr;
  const int lane = threadIdx.x % tpr;
  for (int rr = 0; rr < rpt; ++rr) {
  const int row = (blockIdx.x * rpt + rr) * rpb + threadIdx.x / tpr;
  if (row >= n) return;
  ff2 muh[CH], mul[CH], auh[CH], aul[CH];
  // two separate gathers: the one-gather form (as in the bordering kernel) needs more registers
  // than the four blocks per SM this kernel runs at, and was slower (0.57 -> 0.63 ms)
  gather_row_ff<CH, true>(mrp, mci, mval, U, row, lane, tpr, ldk, muh, mul);
  gather_row_ff<CH, true, AEX>(arp, aci, aval, U, row, lane, tpr, ldk, auh, aul);
  const size_t base = (size_t)row * ldk;
#pragma unroll
  for (int c = 0; c < CH; ++c) {
    const int col = (c * tpr + lane) * 2;
    const ulonglong2 l = lsp[col / 2];
    ff2 fh, fl;
    ff2_mul(l.x, l.y, muh[c], mul[c], fh, fl);
    const ff2 r = ff2_addrn(ff2_subrn(fh, auh[c]), ff2_subrn(fl, aul[c]));
    *reinterpret_cast<ulonglong2*>(Fd + base + col) = make_ulonglong2(fh, fl);
    *reinterpret_cast<ff2*>(R + base + col) = r;
  }
  }
}

// R = Fd - A X as float32 (Fd and X as float pairs).
template <int CH, bool AEX>
__global__ void __launch_bounds__(kBlock, kMinBlocksGather)
    k_outer_res_ff(int n, const int* __restrict__ arp, const int* __restrict__ aci, const float2* __restrict__ aval,
                   const float2* __restrict__ Fd, const double* __restrict__ X, float* __restrict__ R, int ldk,
                   int tpr, int rpt) {
  const int rpb = kBlock / tpr;
  const int lane = threadIdx.x % tpr;
  pdl_trigger();
  prefetch_row(arp, aci, aval, blockIdx.x * rpt * rpb + threadIdx.x / tpr, n);
  pdl_wait();
  for (int rr = 0; rr < rpt; ++rr) {
  const int row = (blockIdx.x * rpt + rr) * rpb + threadIdx.x / tpr;
  if (row >= n) return;
  ff2 axh[CH], axl[CH];
  gather_row_ff<CH, true, AEX>(arp, aci, aval, X, row, lane, tpr, ldk, axh, axl);
  const size_t base = (size_t)row * ldk;
  // every chunk's Fd before the first store: a load after a store that it might alias waits for its turn, and
  // the chunks' round trips went one by one (h = 1/1024, k = 64: 331 us against 270)
  ff2 fh[CH], fl[CH];
#pragma unroll
  for (int c = 0; c < CH; ++c)
    load_pair<true>(reinterpret_cast<const double*>(Fd), base + (c * tpr + lane) * 2, fh[c], fl[c]);
#pragma unroll
  for (int c = 0; c < CH; ++c)
    *reinterpret_cast<ff2*>(R + base + (c * tpr + lane) * 2) =
        ff2_addrn(ff2_subrn(fh[c], axh[c]), ff2_subrn(fl[c], axl[c]));
  }
}

// YA = A X, YM = M X (X, YA, YM as float pairs) and per-block partial sums of
// X .* YA, X .* YM (double-float per thread, float64 across the block).
template <int CH, bool AEX, bool MERGED>
__global__ void __launch_bounds__(kBlock)
    k_border_ff(int n, const int* __restrict__ arp, const int* __restrict__ aci, const float2* __restrict__ aval,
                const int* __restrict__ mrp, const int* __restrict__ mci, const float2* __restrict__ mval,
                const double* __restrict__ X, double* __restrict__ YA, double* __restrict__ YM,
                double* __restrict__ partials, int ldk, int tpr, const float4* __restrict__ am) {
  extern __shared__ __align__(16) double red[];  // [rpb][2][ldk]
  const int rpb = kBlock / tpr;
  const int grp = threadIdx.x / tpr;
  const int lane = threadIdx.x % tpr;
  ff2 sAh[CH], sAl[CH], sMh[CH], sMl[CH];
#pragma unroll
  for (int c = 0; c < CH; ++c) sAh[c] = sAl[c] = sMh[c] = sMl[c] = 0;
  pdl_trigger();
  if (MERGED) {
    prefetch_row(mrp, mci, am, blockIdx.x * rpb + grp, n);
  } else {
    prefetch_row(mrp, mci, mval, blockIdx.x * rpb + grp, n);
    prefetch_row(arp, aci, aval, blockIdx.x * rpb + grp, n);
  }
  pdl_wait();
  for (int row = blockIdx.x * rpb + grp; row < n; row += gridDim.x * rpb) {
    ff2 yah[CH], yal[CH], ymh[CH], yml[CH];
    if (MERGED) {
      gather_row_am<CH, true, AEX>(mrp, mci, am, X, row, lane, tpr, ldk, yah, yal, ymh, yml);
    } else {
      gather_row_ff<CH, true, AEX>(arp, aci, aval, X, row, lane, tpr, ldk, yah, yal);
      gather_row_ff<CH, true>(mrp, mci, mval, X, row, lane, tpr, ldk, ymh, yml);
    }
    const size_t base = (size_t)row * ldk;
#pragma unroll
    for (int c = 0; c < CH; ++c) {
      const size_t off = base + (c * tpr + lane) * 2;
      ff2 xh, xl;
      load_pair<true>(X, off, xh, xl);
      store_pair<true>(YA, off, yah[c], yal[c]);
      store_pair<true>(YM, off, ymh[c], yml[c]);
      const ff2 nx = ff2_neg(xh);
      ff2_mac(sAh[c], sAl[c], xh, nx, xl, yah[c], yal[c]);
      ff2_mac(sMh[c], sMl[c], xh, nx, xl, ymh[c], yml[c]);
    }
  }
#pragma unroll
  for (int c = 0; c < CH; ++c) {
    const int col = (c * tpr + lane) * 2;
    store_pair<false>(red, (grp * 2 + 0) * ldk + col, sAh[c], sAl[c]);
    store_pair<false>(red, (grp * 2 + 1) * ldk + col, sMh[c], sMl[c]);
  }
  __syncthreads();
  for (int t = threadIdx.x; t < 2 * ldk; t += blockDim.x) {
    double s = 0.0;
    for (int r = 0; r < rpb; ++r) s += red[r * 2 * ldk + t];
    partials[(size_t)blockIdx.x * 2 * ldk + t] = s;
  }
}

// out = S X; FFIN / FFOUT: X / out as float pairs (else float64).
template <int CH, bool FFIN, bool FFOUT, bool EX>
__global__ void __launch_bounds__(kBlock, kMinBlocksGather) k_spmm_ff(int n, const int* __restrict__ rp, const int* __restrict__ ci,
                                                     const float2* __restrict__ av, const double* __restrict__ X,
                                                     double* __restrict__ out, int ldk, int tpr, int rpt) {
  const int rpb = kBlock / tpr;
  const int lane = threadIdx.x % tpr;
  pdl_trigger();
  prefetch_row(rp, ci, av, blockIdx.x * rpt * rpb + threadIdx.x / tpr, n);
  pdl_wait();
  for (int rr = 0; rr < rpt; ++rr) {
  const int row = (blockIdx.x * rpt + rr) * rpb + threadIdx.x / tpr;
  if (row >= n) return;
  ff2 yh[CH], yl[CH];
  gather_row_ff<CH, FFIN, EX>(rp, ci, av, X, row, lane, tpr, ldk, yh, yl);
  const size_t base = (size_t)row * ldk;
#pragma unroll
  for (int c = 0; c < CH; ++c) store_pair<FFOUT>(out, base + (c * tpr + lane) * 2, yh[c], yl[c]);
  }
}

// outA = S XA and outM = S XM together (the two restriction chains of the bordering products): one
// load of S's indices and values serves both; each product sees the same terms in the same order
// as two separate k_spmm_ff launches.
template <int CH, int N, bool FFIN, bool EX>
__device__ __forceinline__ void gather_group_ff2(const int* __restrict__ ci, const float2* __restrict__ av,
                                                 const double* __restrict__ XA, const double* __restrict__ XM,
                                                 int p, int lane, int tpr, int ldk, ff2 (&ah)[CH], ff2 (&al)[CH],
                                                 ff2 (&mh)[CH], ff2 (&ml)[CH]) {
  int j[N];
  float2 a[N];
#pragma unroll
  for (int u = 0; u < N; ++u) {
    j[u] = __ldg(ci + p + u);
    a[u] = __ldg(av + p + u);
  }
  ff2 xh[N][CH], xl[N][CH], yh[N][CH], yl[N][CH];
#pragma unroll
  for (int u = 0; u < N; ++u)
#pragma unroll
    for (int c = 0; c < CH; ++c) {
      const size_t off = (size_t)j[u] * ldk + (c * tpr + lane) * 2;
      load_pair<FFIN>(XA, off, xh[u][c], xl[u][c]);
      load_pair<FFIN>(XM, off, yh[u][c], yl[u][c]);
    }
#pragma unroll
  for (int u = 0; u < N; ++u) {
    const ff2 w0 = ff2_pack(a[u].x, a[u].x), wn = ff2_pack(-a[u].x, -a[u].x), w1 = ff2_pack(a[u].y, a[u].y);
#pragma unroll
    for (int c = 0; c < CH; ++c) {
      if (EX) {
        ff2_mac_exact(ah[c], al[c], w0, wn, xh[u][c], xl[u][c]);
        ff2_mac_exact(mh[c], ml[c], w0, wn, yh[u][c], yl[u][c]);
      } else {
        ff2_mac(ah[c], al[c], w0, wn, w1, xh[u][c], xl[u][c]);
        ff2_mac(mh[c], ml[c], w0, wn, w1, yh[u][c], yl[u][c]);
      }
    }
  }
}

template <int CH, bool FFIN, bool FFOUT, bool EX>
__global__ void __launch_bounds__(kBlock, kMinBlocksGather) k_spmm2_ff(int n, const int* __restrict__ rp,
                                                                     const int* __restrict__ ci,
                                                                     const float2* __restrict__ av,
                                                                     const double* __restrict__ XA,
                                                                     const double* __restrict__ XM,
                                                                     double* __restrict__ outA,
                                                                     double* __restrict__ outM, int ldk, int tpr,
                                                                     int rpt) {
  const int rpb = kBlock / tpr;
  const int lane = threadIdx.x % tpr;
  pdl_trigger();
  prefetch_row(rp, ci, av, blockIdx.x * rpt * rpb + threadIdx.x / tpr, n);
  pdl_wait();
  for (int rr = 0; rr < rpt; ++rr) {
    const int row = (blockIdx.x * rpt + rr) * rpb + threadIdx.x / tpr;
    if (row >= n) return;
    ff2 ah[CH], al[CH], mh[CH], ml[CH];
#pragma unroll
    for (int c = 0; c < CH; ++c) ah[c] = al[c] = mh[c] = ml[c] = 0;
    int p = __ldg(rp + row);
    const int p1 = __ldg(rp + row + 1);
    for (; p + 4 <= p1; p += 4) gather_group_ff2<CH, 4, FFIN, EX>(ci, av, XA, XM, p, lane, tpr, ldk, ah, al, mh, ml);
    const int rem = p1 - p;
    if (rem == 3) gather_group_ff2<CH, 3, FFIN, EX>(ci, av, XA, XM, p, lane, tpr, ldk, ah, al, mh, ml);
    else if (rem == 2) gather_group_ff2<CH, 2, FFIN, EX>(ci, av, XA, XM, p, lane, tpr, ldk, ah, al, mh, ml);
    else if (rem == 1) gather_group_ff2<CH, 1, FFIN, EX>(ci, av, XA, XM, p, lane, tpr, ldk, ah, al, mh, ml);
    const size_t base = (size_t)row * ldk;
#pragma unroll
    for (int c = 0; c < CH; ++c) {
      ff2_norm(ah[c], al[c]);
      ff2_norm(mh[c], ml[c]);
      store_pair<FFOUT>(outA, base + (c * tpr + lane) * 2, ah[c], al[c]);
      store_pair<FFOUT>(outM, base + (c * tpr + lane) * 2, mh[c], ml[c]);
    }
  }
}

// X = B + E with E float32, X as float pairs; B as float pairs (may alias X)
// or float64.
template <bool BFF>
__global__ void k_axpy_ff(int64_t total, const double* B, const float* E, double* X) {
  pdl_trigger();
  pdl_wait();
  const int64_t np = total / 2;
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < np; i += (int64_t)gridDim.x * blockDim.x) {
    ff2 bh, bl;
    load_pair<BFF>(B, 2 * i, bh, bl);
    ff2 e;
    asm volatile("ld.global.u64 %0, [%1];" : "=l"(e) : "l"(E + 2 * i));
    ff2_add(bh, bl, e);
    ff2_norm(bh, bl);
    store_pair<true>(X, 2 * i, bh, bl);
  }
}

// Elementwise format conversions of block vectors.
// in may equal out: each thread reads its two entries before writing them.
__global__ void k_to_ff(int64_t total, const double* in, double* out) {
  pdl_trigger();
  pdl_wait();
  const int64_t np = total / 2;
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < np; i += (int64_t)gridDim.x * blockDim.x) {
    ff2 h, l;
    load_pair<false>(in, 2 * i, h, l);
    store_pair<true>(out, 2 * i, h, l);
  }
}
__global__ void k_from_ff(int64_t total, const double* in, double* out) {
  pdl_trigger();
  pdl_wait();
  const int64_t np = total / 2;
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < np; i += (int64_t)gridDim.x * blockDim.x) {
    ff2 h, l;
    load_pair<true>(in, 2 * i, h, l);
    store_pair<false>(out, 2 * i, h, l);
  }
}

// The caller's [n][k] block on the device -> [n][ldk], zero in the padded columns: float64 (U, may be
// null) and pairs (may be null) in one pass.  Bound by memory: one read and one write per copy made
// (a linear or pitched copy, a memset and a conversion took two to six passes).  The caller's rows
// may be 8-byte aligned only.
__global__ void __launch_bounds__(kBlock) k_put_block(int64_t n, int k, int ldk, const double* src, double* U,
                                                      double* pairs) {
  pdl_trigger();
  pdl_wait();
  const int sh = 31 - __clz(ldk / 2);   // ldk is a power of two
  for (int64_t i = blockIdx.x * (int64_t)kBlock + threadIdx.x; i < n << sh; i += (int64_t)gridDim.x * kBlock) {
    const int64_t row = i >> sh;
    const int c = 2 * (int)(i & ((1 << sh) - 1));
    const double* p = src + row * k + c;
    const double a = c < k ? ld1(p) : 0.0, b = c + 1 < k ? ld1(p + 1) : 0.0;
    if (U) *reinterpret_cast<double2*>(U + row * ldk + c) = make_double2(a, b);
    if (pairs) {
      float h0, l0, h1, l1;
      ff_split(a, h0, l0);
      ff_split(b, h1, l1);
      store_pair<true>(pairs, (size_t)(row * ldk + c), ff2_pack(h0, h1), ff2_pack(l0, l1));
    }
  }
}
// The reverse: an [n][ldk] block (float64, or pairs with FF) -> the caller's [n][k] block on the device.
template <bool FF>
__global__ void __launch_bounds__(kBlock) k_get_block(int64_t n, int k, int ldk, const double* in, double* dst) {
  pdl_trigger();
  pdl_wait();
  const int sh = 31 - __clz(ldk / 2);
  for (int64_t i = blockIdx.x * (int64_t)kBlock + threadIdx.x; i < n << sh; i += (int64_t)gridDim.x * kBlock) {
    const int64_t row = i >> sh;
    const int c = 2 * (int)(i & ((1 << sh) - 1));
    if (c >= k) continue;
    double v[2];
    if (FF) {
      ff2 h, l;
      load_pair<true>(in, (size_t)(row * ldk + c), h, l);
      float h0, h1, l0, l1;
      ff2_unpack(h, h0, h1);
      ff2_unpack(l, l0, l1);
      v[0] = ff_to_double(h0, l0);
      v[1] = ff_to_double(h1, l1);
    } else {
      ldg16<double>(in + row * ldk + c, v);
    }
    double* p = dst + row * k + c;
    p[0] = v[0];
    if (c + 1 < k) p[1] = v[1];
  }
}

// U[row][c] = upd[c] ? alpha[c] X[row][c] + (P W)[row][c] : U[row][c], X as
// float pairs, W as float pairs (WFF) or float64; identity: P W = W.  Entries
// of frozen pairs are neither read nor written.  With U null the state is the
// pair array Usplit alone (the finest-level state of the mixed-precision step;
// its float64 copy is made on demand), else U is written in float64 and, if
// Usplit is given, also split into pairs.
// STATE: the finest-level update of a step (U null, P given), on its own so that it fits 32 registers
// for one chunk per thread (8 blocks per SM; at h = 1/1024, k = 64: 244 us against 285 without the bound).
template <int CH, bool STATE> struct UpdateMinBlocks { static constexpr int v = STATE && CH == 1 ? 8 : 0; };
template <int CH, bool WFF, bool EX, bool STATE>
__global__ void __launch_bounds__(kBlock, (UpdateMinBlocks<CH, STATE>::v))
    k_update_ff(int n, const int* __restrict__ rp, const int* __restrict__ ci, const float2* __restrict__ pv,
                const double* __restrict__ W, const double* __restrict__ X, const double* __restrict__ alpha,
                const int* __restrict__ upd, double* __restrict__ U, double* __restrict__ Usplit, int ldk, int tpr,
                int identity, int rpt) {
  pdl_trigger();
  if (STATE || !identity) prefetch_row(rp, ci, pv, blockIdx.x * rpt * (kBlock / tpr) + threadIdx.x / tpr, n);
  pdl_wait();
  extern __shared__ ulonglong2 asp[];  // [ldk / 2]: alpha as pair chunks, split once per block
  for (int t = threadIdx.x; t < ldk / 2; t += blockDim.x) load_pair<false>(alpha, 2 * t, asp[t].x, asp[t].y);
  __syncthreads();
  const int rpb = kBlock / tpr;
  const int lane = threadIdx.x % tpr;
  for (int rr = 0; rr < rpt; ++rr) {
  const int row = (blockIdx.x * rpt + rr) * rpb + threadIdx.x / tpr;
  if (row >= n) return;
  ff2 wh[CH], wl[CH];
  const size_t base = (size_t)row * ldk;
  if (!STATE && identity) {
#pragma unroll
    for (int c = 0; c < CH; ++c) load_pair<WFF>(W, base + (c * tpr + lane) * 2, wh[c], wl[c]);
  } else {
    gather_row_ff<CH, WFF, EX>(rp, ci, pv, W, row, lane, tpr, ldk, wh, wl);
  }
#pragma unroll
  for (int c = 0; c < CH; ++c) {
    const int col = (c * tpr + lane) * 2;
    const size_t off = base + col;
    const int u0 = ld1(upd + col), u1 = ld1(upd + col + 1);
    if (!u0 && !u1) continue;  // both pairs frozen: U and its split copy stay as they are
    ff2 xh, xl;
    load_pair<true>(X, off, xh, xl);
    const ulonglong2 a = asp[col / 2];
    ff2 h = wh[c], l = wl[c];
    ff2_mac(h, l, a.x, ff2_neg(a.x), a.y, xh, xl);
    ff2_norm(h, l);
    if (STATE || !U) {  // the state lives in pairs only: write the updated pairs, keep the frozen one
      if (!(u0 && u1)) {
        ff2 oh, ol;
        load_pair<true>(Usplit, off, oh, ol);
        const ff2 keep = u0 ? 0xFFFFFFFF00000000ull : 0x00000000FFFFFFFFull;
        h = (h & ~keep) | (oh & keep);
        l = (l & ~keep) | (ol & keep);
      }
      store_pair<true>(Usplit, off, h, l);
      continue;
    }
    double2 u;
    if (!(u0 && u1)) u = *reinterpret_cast<const double2*>(U + off);
    float h0, h1, l0, l1;
    ff2_unpack(h, h0, h1);
    ff2_unpack(l, l0, l1);
    if (u0) u.x = ff_to_double(h0, l0);
    if (u1) u.y = ff_to_double(h1, l1);
    *reinterpret_cast<double2*>(U + off) = u;
    if (Usplit) {  // the (hi, lo) copy of U the next step's gathers read
      ff_split(u.x, h0, l0);
      ff_split(u.y, h1, l1);
      store_pair<true>(Usplit, off, ff2_pack(h0, h1), ff2_pack(l0, l1));
    }
  }
  }
}

}  // namespace

void outer_rhs_residual_ff(const Launch& L, const DCsr& A, const DCsr& M, const double* lam, const double* U,
                           double* Fd, float* R, int ldk) {
  const Geo g = geometry_ff(ldk, L.geo);
  const int rpb = kBlock / g.tpr, rpt = ff_rows(L);
  const int grid = (A.n_rows + rpb * rpt - 1) / (rpb * rpt);
  {
    const double n = A.n_rows, nnz = (double)(A.nnz + M.nnz);
    L.rows(A.n_rows);
    L.begin(KC_OUTER_RHS, nnz * 12.0 + 2 * (n + 1) * 4.0 + n * ldk * (16.0 + 4.0), 2.0 * nnz * ldk + 2.0 * n * ldk);
  }
#define PASM_FF_RHS(AEX)                                                                      \
  PASM_FF_DISPATCH(g.ch, launch(L, k_outer_rhs_res_ff<CH, AEX>, grid, kBlock, ldk * sizeof(float2), \
                             A.n_rows, A.rp, A.ci, A.vff, M.rp, M.ci, M.vff, lam, U,            \
                             reinterpret_cast<float2*>(Fd), R, ldk, g.tpr, rpt))
  if (A.exact32) { PASM_FF_RHS(true); } else { PASM_FF_RHS(false); }
#undef PASM_FF_RHS
  L.bump();
}

void outer_residual_ff(const Launch& L, const DCsr& A, const double* Fd, const double* X, float* R, int ldk) {
  const Geo g = geometry_ff(ldk, L.geo);
  const int rpb = kBlock / g.tpr, rpt = ff_rows(L);
  const int grid = (A.n_rows + rpb * rpt - 1) / (rpb * rpt);
  {
    const double n = A.n_rows, nnz = (double)A.nnz;
    L.rows(A.n_rows);
    L.begin(KC_OUTER_RES, nnz * 12.0 + (n + 1) * 4.0 + n * ldk * (16.0 + 4.0), 2.0 * nnz * ldk + n * ldk);
  }
  if (A.exact32) {
    PASM_FF_DISPATCH(g.ch, launch(L, k_outer_res_ff<CH, true>, grid, kBlock, 0, A.n_rows, A.rp, A.ci, A.vff, reinterpret_cast<const float2*>(Fd), X, R, ldk, g.tpr, rpt));
  } else {
    PASM_FF_DISPATCH(g.ch, launch(L, k_outer_res_ff<CH, false>, grid, kBlock, 0, A.n_rows, A.rp, A.ci, A.vff, reinterpret_cast<const float2*>(Fd), X, R, ldk, g.tpr, rpt));
  }
  L.bump();
}

int border_products_ff(const Launch& L, const DCsr& A, const DCsr& M, const double* X, double* YA, double* YM,
                       double* partials, int ldk, int max_blocks) {
  Geo g = geometry_ff(ldk, L.geo);
  // the per-block reduction buffer (rows per block x 2 x ldk doubles) stays within the
  // default 48 KB of dynamic shared memory; a tile shape that needs more is not used
  if ((size_t)(kBlock / g.tpr) * 2 * ldk * sizeof(double) > 48 * 1024) g = geometry_ff(ldk, 0);
  const int rpb = kBlock / g.tpr;
  int grid = std::min((A.n_rows + rpb - 1) / rpb, max_blocks);
  if (grid < 1) grid = 1;
  const size_t smem = (size_t)rpb * 2 * ldk * sizeof(double);
  {
    const double n = A.n_rows, nnz = (double)(A.nnz + M.nnz);
    L.rows(A.n_rows);
    L.begin(KC_BORDER, nnz * 12.0 + 2 * (n + 1) * 4.0 + 3.0 * n * ldk * 8.0, 2.0 * nnz * ldk + 4.0 * n * ldk);
  }
#define PASM_FF_BORDER(AEX, MG)                                                                \
  PASM_FF_DISPATCH(g.ch, launch(L, k_border_ff<CH, AEX, MG>, grid, kBlock, smem, \
                             A.n_rows, A.rp, A.ci, A.vff, M.rp, M.ci, M.vff, X, YA, YM, partials, ldk, g.tpr, M.am))
  if (M.am) {
    if (A.exact32) { PASM_FF_BORDER(true, true); } else { PASM_FF_BORDER(false, true); }
  } else {
    if (A.exact32) { PASM_FF_BORDER(true, false); } else { PASM_FF_BORDER(false, false); }
  }
#undef PASM_FF_BORDER
  L.bump();
  return grid;
}

void spmm_ff(const Launch& L, const DCsr& S, const double* X, bool x_ff, double* out, bool out_ff, int ldk) {
  if (S.n_rows == 0) return;
  const Geo g = geometry_ff(ldk, L.geo);
  const int rpb = kBlock / g.tpr, rpt = ff_rows(L);
  const int grid = (S.n_rows + rpb * rpt - 1) / (rpb * rpt);
  {
    const double rows = S.n_rows, cols = S.n_cols, nnz = (double)S.nnz;
    L.rows(S.n_rows);
    L.begin(KC_SPMM, nnz * 12.0 + (rows + 1) * 4.0 + cols * ldk * 8.0 + rows * ldk * 8.0, 2.0 * nnz * ldk);
  }
#define PASM_FF_SPMM(FI, FO)                                                                                   \
  if (S.exact32) {                                                                                             \
    PASM_FF_DISPATCH(g.ch, launch(L, k_spmm_ff<CH, FI, FO, true>, grid, kBlock, 0, S.n_rows, S.rp, S.ci, S.vff, X, \
                                                                                  out, ldk, g.tpr, rpt));           \
  } else {                                                                                                     \
    PASM_FF_DISPATCH(g.ch, launch(L, k_spmm_ff<CH, FI, FO, false>, grid, kBlock, 0, S.n_rows, S.rp, S.ci, S.vff, \
                                                                                   X, out, ldk, g.tpr, rpt));       \
  }
  if (x_ff && out_ff) { PASM_FF_SPMM(true, true); }
  else if (x_ff) { PASM_FF_SPMM(true, false); }
  else if (out_ff) { PASM_FF_SPMM(false, true); }
  else { PASM_FF_SPMM(false, false); }
#undef PASM_FF_SPMM
  L.bump();
}

void spmm2_ff(const Launch& L, const DCsr& S, const double* XA, const double* XM, bool x_ff, double* outA,
              double* outM, bool out_ff, int ldk) {
  if (S.n_rows == 0) return;
  const Geo g = geometry_ff(ldk, L.geo);
  const int rpb = kBlock / g.tpr, rpt = ff_rows(L);
  const int grid = (S.n_rows + rpb * rpt - 1) / (rpb * rpt);
  {
    const double rows = S.n_rows, cols = S.n_cols, nnz = (double)S.nnz;
    L.rows(S.n_rows);
    L.begin(KC_SPMM, nnz * 12.0 + (rows + 1) * 4.0 + 2.0 * (cols + rows) * ldk * 8.0, 4.0 * nnz * ldk);
  }
#define PASM_FF_SPMM2(FI, FO)                                                                                    \
  if (S.exact32) {                                                                                               \
    PASM_FF_DISPATCH(g.ch, launch(L, k_spmm2_ff<CH, FI, FO, true>, grid, kBlock, 0, S.n_rows, S.rp, S.ci, S.vff, XA,  \
                                                                                   XM, outA, outM, ldk, g.tpr, rpt)); \
  } else {                                                                                                       \
    PASM_FF_DISPATCH(g.ch, launch(L, k_spmm2_ff<CH, FI, FO, false>, grid, kBlock, 0, S.n_rows, S.rp, S.ci, S.vff, XA, \
                                                                                    XM, outA, outM, ldk, g.tpr, rpt)); \
  }
  if (x_ff && out_ff) { PASM_FF_SPMM2(true, true); }
  else if (x_ff) { PASM_FF_SPMM2(true, false); }
  else if (out_ff) { PASM_FF_SPMM2(false, true); }
  else { PASM_FF_SPMM2(false, false); }
#undef PASM_FF_SPMM2
  L.bump();
}

static int stream_grid(int64_t total) { return (int)std::min<int64_t>((total / 2 + kBlock - 1) / kBlock, 152 * 16); }

void axpy_ff(const Launch& L, int n, const double* B, bool b_ff, const float* E, double* X, int ldk) {
  const int64_t total = (int64_t)n * ldk;
  L.begin(KC_AXPY, (double)total * (16.0 + 4.0), (double)total);
  if (b_ff) launch(L, k_axpy_ff<true>, stream_grid(total), kBlock, 0, total, B, E, X);
  else launch(L, k_axpy_ff<false>, stream_grid(total), kBlock, 0, total, B, E, X);
  L.bump();
}

void to_ff(const Launch& L, int64_t total, const double* in, double* out) {
  L.begin(KC_CAST, (double)total * 16.0, 0.0);
  launch(L, k_to_ff, stream_grid(total), kBlock, 0, total, in, out);
  L.bump();
}

void from_ff(const Launch& L, int64_t total, const double* in, double* out) {
  L.begin(KC_CAST, (double)total * 16.0, (double)total);
  launch(L, k_from_ff, stream_grid(total), kBlock, 0, total, in, out);
  L.bump();
}

void put_block_dev(const Launch& L, int64_t n, int k, int ldk, const double* src, double* U, double* pairs) {
  L.begin(KC_CAST, (double)n * (k + ldk * ((U ? 1 : 0) + (pairs ? 1 : 0))) * 8.0, 0.0);
  launch(L, k_put_block, stream_grid(n * ldk), kBlock, 0, n, k, ldk, src, U, pairs);
  L.bump();
}

void get_block_dev(const Launch& L, int64_t n, int k, int ldk, const double* in, bool ff, double* dst) {
  L.begin(KC_CAST, (double)n * (k + ldk) * 8.0, 0.0);
  if (ff) launch(L, k_get_block<true>, stream_grid(n * ldk), kBlock, 0, n, k, ldk, in, dst);
  else launch(L, k_get_block<false>, stream_grid(n * ldk), kBlock, 0, n, k, ldk, in, dst);
  L.bump();
}

void update_pairs_ff(const Launch& L, const DCsr* P, int n, const double* W, bool w_ff, const double* X,
                     const double* alpha, const int* upd, double* U, double* Usplit, int ldk) {
  const Geo g = geometry_ff(ldk, L.geo);
  const int rpb = kBlock / g.tpr, rpt = ff_rows(L);
  const int grid = (n + rpb * rpt - 1) / (rpb * rpt);
  const int identity = P ? 0 : 1;
  {
    const double nn = n, nnz = P ? (double)P->nnz : 0.0, cols = P ? (double)P->n_cols : nn;
    L.begin(KC_UPDATE, nnz * 12.0 + (nn + 1) * 4.0 + cols * ldk * 8.0 + 3.0 * nn * ldk * 8.0,
            2.0 * nnz * ldk + 2.0 * nn * ldk);
  }
  const int* rp = P ? P->rp : nullptr;
  const int* ci = P ? P->ci : nullptr;
  const float2* pv = P ? P->vff : nullptr;
  const bool ex = P ? P->exact32 : true;
#define PASM_FF_UPD(WF, EXV)                                                                                     \
  if (P && !U) {                                                                                                 \
    PASM_FF_DISPATCH(g.ch, launch(L, k_update_ff<CH, WF, EXV, true>, grid, kBlock, ldk * sizeof(float2), \
                               n, rp, ci, pv, W, X, alpha, upd, nullptr, Usplit, ldk, g.tpr, 0, rpt));            \
  } else {                                                                                                       \
    PASM_FF_DISPATCH(g.ch, launch(L, k_update_ff<CH, WF, EXV, false>, grid, kBlock, ldk * sizeof(float2), \
                               n, rp, ci, pv, W, X, alpha, upd, U, Usplit, ldk, g.tpr, identity, rpt));           \
  }
  if (w_ff) {
    if (ex) { PASM_FF_UPD(true, true); } else { PASM_FF_UPD(true, false); }
  } else {
    if (ex) { PASM_FF_UPD(false, true); } else { PASM_FF_UPD(false, false); }
  }
#undef PASM_FF_UPD
  L.bump();
}

}  // namespace pasm

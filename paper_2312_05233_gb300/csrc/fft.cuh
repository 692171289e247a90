// Batched complex FFT in float64 for the correlation and cosine-transform
// tails (spectrum.cu, raman.cu): N = 2^m (m >= 8), Stockham passes of radix
// 16 or 8 (with one smaller one between the first and the last where m is not a
// multiple of 4 or 3), one butterfly per thread in registers.
//
// What bounds it: the FP64 pipe (two lanes per clock and SM, 64 times fewer
// than FP32), about 3.5 instructions per point and radix-2 stage whatever the
// radix.  So the work goes into fewer and shorter transforms (two real
// channels per complex transform, segments instead of the whole series), and
// the radix only cuts passes, i.e. launches and L2 round trips: radix 2 took
// 17 passes of 13.5 us for nine transforms of 2^17 (T = 1e5), each at 60% of
// the FP64 rate.  The first pass loads through a functor (zero padding,
// products, chirps), the last one stores through one (normalisation), so no
// pass only moves data.
//
// Pass with p (the product of the earlier radices) and radix R, per transform:
//   v_r = a[j + r N/R] exp(-+2 pi i k r / (p R)),  k = j mod p,
//   b[(j - k) R + k + r p] = DFT_R(v)_r,
// which leaves the result in natural order after the last pass.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include <utility>

#include "tnep_internal.cuh"

namespace tnep {
namespace fft {

constexpr int kMinLog = 8;
constexpr int kThreads = 128;
// Passes of fewer threads than this run in CTAs of one warp, so that a single
// transform's butterflies spread over the SMs (2048 of them in 16 CTAs: 12 us a
// pass, FP64 issue of 16 SMs).
constexpr long long kSpreadBelow = 152 * 256;

// Sign flip and swap without the FP64 pipe.
__device__ __forceinline__ double flip(double v, unsigned sign) {
  return __hiloint2double((int)((unsigned)__double2hiint(v) ^ sign), __double2loint(v));
}
__device__ __forceinline__ double2 add(double2 a, double2 b) { return make_double2(a.x + b.x, a.y + b.y); }
__device__ __forceinline__ double2 sub(double2 a, double2 b) { return make_double2(a.x - b.x, a.y - b.y); }
__device__ __forceinline__ double2 mul(double2 a, double2 b) {
  return make_double2(fma(a.x, b.x, -a.y * b.y), fma(a.x, b.y, a.y * b.x));
}
// a times -i (forward) or +i (inverse)
template <bool INV>
__device__ __forceinline__ double2 rot(double2 a) {
  return INV ? make_double2(-a.y, a.x) : make_double2(a.y, -a.x);
}

// exp(-+2 pi i idx / N) from tab[i] = (cos, sin)(2 pi i / N), i = 0..N/8.
template <bool INV>
__device__ __forceinline__ double2 twiddle(const double2* __restrict__ tab, unsigned idx, int logN) {
  const unsigned quarter = 1u << (logN - 2), q = (idx >> (logN - 2)) & 3u;
  const unsigned i = idx & (quarter - 1);
  const bool up = i > (quarter >> 1);
  const double2 t = __ldg(tab + (up ? quarter - i : i));
  const double c = up ? t.y : t.x, s = up ? t.x : t.y;
  // (c, -s) turned by q quarters of -90 degrees
  const bool odd = q & 1u;
  const unsigned sx = (((q >> 1) ^ (q & 1u)) & 1u) << 31;     // q = 1, 2 negate x
  const unsigned sy = (((q >> 1) ^ 1u) & 1u) << 31;           // q = 0, 1 negate y
  const double x = flip(odd ? s : c, sx), y = flip(odd ? c : s, sy);
  return make_double2(x, INV ? flip(y, 0x80000000u) : y);
}

template <bool INV>
__device__ __forceinline__ void dft4(double2& a, double2& b, double2& c, double2& d) {
  const double2 t0 = add(a, c), t1 = sub(a, c), t2 = add(b, d), t3 = rot<INV>(sub(b, d));
  a = add(t0, t2);
  b = add(t1, t3);
  c = sub(t0, t2);
  d = sub(t1, t3);
}

// In place, natural order in and out.  HALF: the upper half of v is zero
// (radix 16 only).
template <int R, bool INV, bool HALF = false>
__device__ __forceinline__ void dft(double2* v) {
  constexpr double h = 0.70710678118654752440;
  if constexpr (R == 2) {
    const double2 t = v[1];
    v[1] = sub(v[0], t);
    v[0] = add(v[0], t);
  } else if constexpr (R == 4) {
    dft4<INV>(v[0], v[1], v[2], v[3]);
  } else if constexpr (R == 8) {
    double2 e[4] = {v[0], v[2], v[4], v[6]}, o[4] = {v[1], v[3], v[5], v[7]};
    dft4<INV>(e[0], e[1], e[2], e[3]);
    dft4<INV>(o[0], o[1], o[2], o[3]);
    o[2] = rot<INV>(o[2]);
    v[0] = add(e[0], o[0]);
    v[4] = sub(e[0], o[0]);
    v[2] = add(e[2], o[2]);
    v[6] = sub(e[2], o[2]);
#pragma unroll
    for (int k = 1; k < 4; k += 2) {  // exp(-+ i pi k / 4) = h (+-1 -+ i)
      const double2 r = rot<INV>(o[k]);
      const double2 t = k == 1 ? add(o[k], r) : sub(r, o[k]);
      v[k] = make_double2(fma(h, t.x, e[k].x), fma(h, t.y, e[k].y));
      v[k + 4] = make_double2(fma(-h, t.x, e[k].x), fma(-h, t.y, e[k].y));
    }
  } else {
    static_assert(R == 16, "radix 2, 4, 8 or 16");
    constexpr double c1 = 0.92387953251128675613, s1 = 0.38268343236508977173;
    double2 y[4][4];  // [n2][k1]
#pragma unroll
    for (int n2 = 0; n2 < 4; ++n2) {
#pragma unroll
      for (int n1 = 0; n1 < (HALF ? 2 : 4); ++n1) y[n2][n1] = v[4 * n1 + n2];
      if constexpr (HALF) {
        const double2 a = y[n2][0], b = y[n2][1], r = rot<INV>(b);
        y[n2][0] = add(a, b);
        y[n2][1] = add(a, r);
        y[n2][2] = sub(a, b);
        y[n2][3] = sub(a, r);
      } else {
        dft4<INV>(y[n2][0], y[n2][1], y[n2][2], y[n2][3]);
      }
    }
    // y[n2][k1] *= exp(-+2 pi i n2 k1 / 16)
    auto w = [](double2 a, double c, double s) {  // a (c -+ i s)
      const double si = INV ? s : -s;
      return make_double2(fma(a.x, c, -a.y * si), fma(a.x, si, a.y * c));
    };
    auto w2 = [](double2 a) {  // a exp(-+ i pi / 4)
      const double2 t = add(a, rot<INV>(a));
      return make_double2(h * t.x, h * t.y);
    };
    y[1][1] = w(y[1][1], c1, s1);
    y[1][2] = w2(y[1][2]);
    y[1][3] = w(y[1][3], s1, c1);
    y[2][1] = w2(y[2][1]);
    y[2][2] = rot<INV>(y[2][2]);
    y[2][3] = rot<INV>(w2(y[2][3]));
    y[3][1] = w(y[3][1], s1, c1);
    y[3][2] = rot<INV>(w2(y[3][2]));
    y[3][3] = w(y[3][3], -c1, -s1);
#pragma unroll
    for (int k1 = 0; k1 < 4; ++k1) {
      dft4<INV>(y[0][k1], y[1][k1], y[2][k1], y[3][k1]);
#pragma unroll
      for (int k2 = 0; k2 < 4; ++k2) v[k1 + 4 * k2] = y[k2][k1];
    }
  }
}

// Plain element access of `batch` transforms of length N.
// A load with kHalfZero gives zeros for the upper half (it is not called there).
struct LoadPlain {
  static constexpr bool kHalfZero = false;
  const double2* p;
  int logN;
  __device__ __forceinline__ double2 operator()(int f, unsigned i) const { return p[((size_t)f << logN) + i]; }
};
struct StorePlain {
  double2* p;
  int logN;
  __device__ __forceinline__ void operator()(int f, unsigned i, double2 v) const { p[((size_t)f << logN) + i] = v; }
};

template <int LOGR, bool INV, class Load, class Store>
__global__ void __launch_bounds__(kThreads) k_pass(const Load ld, const Store st, const double2* __restrict__ tab,
                                                   int logN, int logp, int batch) {
  constexpr int R = 1 << LOGR;
  const long long g = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  const int f = (int)(g >> (logN - LOGR));
  if (f >= batch) return;
  const unsigned j = (unsigned)(g & ((1ll << (logN - LOGR)) - 1));
  constexpr bool HALF = Load::kHalfZero && R == 16;
  double2 v[R];
#pragma unroll
  for (int r = 0; r < (Load::kHalfZero ? R / 2 : R); ++r) v[r] = ld(f, j + ((unsigned)r << (logN - LOGR)));
  if constexpr (Load::kHalfZero && !HALF) {
#pragma unroll
    for (int r = R / 2; r < R; ++r) v[r] = make_double2(0.0, 0.0);
  }
  const unsigned k = j & ((1u << logp) - 1);
  if (logp > 0) {
#pragma unroll
    for (int r = 1; r < R; ++r) v[r] = mul(v[r], twiddle<INV>(tab, (k * r) << (logN - logp - LOGR), logN));
  }
  dft<R, INV, HALF>(v);
  const unsigned o = ((j >> logp) << (logp + LOGR)) + k;
#pragma unroll
  for (int r = 0; r < R; ++r) st(f, o + ((unsigned)r << logp), v[r]);
}

template <int LOGR, bool INV, class Load, class Store>
cudaError_t pass(const Load& ld, const Store& st, const double2* tab, int logN, int logp, int batch, cudaStream_t s) {
  const long long n = (long long)batch << (logN - LOGR);
  count_launches(1);
  const int threads = n < kSpreadBelow ? 32 : kThreads;
  k_pass<LOGR, INV><<<(unsigned)((n + threads - 1) / threads), threads, 0, s>>>(ld, st, tab, logN, logp, batch);
  return cudaGetLastError();
}

// Transforms `batch` arrays of length 2^logN (forward: exp(-i ...), inverse:
// exp(+i ...), no 1/N), loading element i of array f as ld(f, i) and storing
// through st(f, i, value).  a and b: scratch of batch << logN elements each;
// the first pass writes a, so ld may read b.
template <int LOGB, bool INV, class Load, class Store>
cudaError_t transform_radix(const Load& ld, const Store& st, double2* a, double2* b, const double2* tab, int logN,
                            int batch, cudaStream_t s) {
  cudaError_t e = pass<LOGB, INV>(ld, StorePlain{a, logN}, tab, logN, 0, batch, s);
  int logp = LOGB;
  for (int left = logN - 2 * LOGB; left > 0 && e == cudaSuccess;) {
    const int r = left % LOGB ? left % LOGB : LOGB;
    const LoadPlain l{a, logN};
    const StorePlain o{b, logN};
    if (r == 1) e = pass<1, INV>(l, o, tab, logN, logp, batch, s);
    else if (r == 2) e = pass<2, INV>(l, o, tab, logN, logp, batch, s);
    else if (r == 3) e = pass<3, INV>(l, o, tab, logN, logp, batch, s);
    else e = pass<4, INV>(l, o, tab, logN, logp, batch, s);
    std::swap(a, b);
    logp += r;
    left -= r;
  }
  if (e != cudaSuccess) return e;
  return pass<LOGB, INV>(LoadPlain{a, logN}, st, tab, logN, logp, batch, s);
}

// Radix 16 where its butterflies fill the chip.  An SM's four quarters issue
// half an FP64 lane a clock each, so a lone warp's radix-16 butterfly takes
// 288 x 64 cycles (11 us a pass of four stages, whatever the size, below one
// warp per quarter); radix 8 takes 80 x 64 for three.
inline int base_radix(int logN, int batch) { return ((long long)batch << logN) < 300000 ? 3 : 4; }

template <bool INV, class Load, class Store>
cudaError_t transform(const Load& ld, const Store& st, double2* a, double2* b, const double2* tab, int logN,
                      int batch, cudaStream_t s) {
  if (base_radix(logN, batch) == 3) return transform_radix<3, INV>(ld, st, a, b, tab, logN, batch, s);
  return transform_radix<4, INV>(ld, st, a, b, tab, logN, batch, s);
}

// Index of the buffer (0 = a, 1 = b) the last pass of a transform reads.
inline int last_source(int logN, int batch) {
  const int base = base_radix(logN, batch);
  return ((logN - 2 * base + base - 1) / base) & 1;
}

inline int log2_at_least(long long n) {
  int m = kMinLog;
  while ((1ll << m) < n) ++m;
  return m;
}

// Entries of the twiddle table of length 2^logN.
inline size_t table_size(int logN) { return ((size_t)1 << (logN - 3)) + 1; }

}  // namespace fft
}  // namespace tnep

// Polarized Raman tail in float64 (Sec. II.G, Eqs. 7-8).
//
//   sums   partial column sums of alpha(t) (or chi(t)), a fixed grid; for the
//          Fourier route also each channel's size
//   direct route (short series):
//     prep   x [9][T] channel-major, mean removed if asked
//     corr   C_pq(tau) = sum_t x_p(t) x_q(t + tau), all 81 ordered pairs; one
//            thread owns one pair and four consecutive lags and walks t in order
//     lags   S_pq(tau) = (C_pq + C_qp) / (2 (T - tau)), sequence-major
//   Fourier route (rule at raman_uses_fft): segments of L = N/2 >= M samples,
//   N a power of two, as in the spectrum tail (X_b, F_b defined there):
//     prep   two channels per complex value, [5 packs][T], mean removed if asked,
//            each divided by a power of two near its size
//     fft    5 x (number of segments) transforms of length N
//     (T = 1e5, M = 2000, tensor and 181-angle map: 6181 -> 659 us a call;
//     before, one 2^17-point transform per channel and 23 back, and 4240 us of
//     cosine sums that divided and took a 64-bit remainder in every term)
//     cross  for the 45 pairs p <= q, sum over the segments b of
//            conj(X_p) F_q + conj(X_q) F_p
//     ifft   23 transforms, two pairs each; the real sequences are S_pq(tau),
//            multiplied back by the pair's powers of two
//   cos    L_pq(nu_k) = dt [S_pq(0) + 2 sum_tau S_pq(tau) cos(pi k tau / M)]
//          (spectrum.cu)
//   polar  spec_o(nu_k) = sum_pq w_p w_q L_pq(nu_k), w = vec(n_o eps_o^T) (Eq. 7)
//   porto  the same for Z(XX)Z-bar / Z(XY)Z-bar of a crystal turned by theta
// Every sum runs in a fixed order, so results do not depend on the launch.

#include <cuda_runtime.h>

#include <algorithm>
#include <utility>

#include "engine.h"
#include "fft.cuh"

namespace tnep {

namespace {

constexpr int kLagsPerThread = 4;
constexpr int kCorrThreads = 128;
constexpr int kSumThreads = 288, kMaxSumBlocks = 128;  // 288 = 9 x 32: a thread keeps its column
constexpr int kPacks = 5;

// The direct sums cost 81 T (M + 1) multiply-adds of FP64 issue (2e7: 35 us and
// more, one serial chain per lag), the Fourier route about a dozen launches.
// Its error is uniform over the lags while S(tau) divides by T - tau, so lags
// beyond T / 2 keep the direct sums until these cost milliseconds.
bool raman_uses_fft(int T, int M) {
  const double terms = 81.0 * (double)T * (double)(M + 1);
  return terms > 1.0e9 || (terms > 2.0e7 && M <= T / 2);
}

// First pair (p, p) of row p among the 45.
__host__ __device__ constexpr int pair_row(int p) { return p * 9 - p * (p - 1) / 2; }

// |d| / 2^(e - 1023) as a float with the upper 20 bits of d, by integer
// instructions (a conversion holds the FP64 pipe): 0 below the float range,
// infinity above it.
__device__ __forceinline__ float rough(double d, int e) {
  const int hi = __double2hiint(d) & 0x7fffffff, exp = (hi >> 20) - e + 127;
  return exp <= 0 ? 0.f : __int_as_float(exp >= 255 ? 0x7f800000 : (exp << 23) | (hi & 0xfffff) << 3);
}
// Exponent of the unit in which a channel's size is summed: its first sample's.
__device__ __forceinline__ int rough_unit(double first) {
  const int e = (__double2hiint(first) >> 20) & 0x7ff;
  return e == 0 || e == 0x7ff ? 1023 : e;
}

// Partial column sums of s [T][9], part[block][9]; with STATS also the sums of
// squares (float, in units of rough_unit) and the upper word of the largest
// magnitude about the first sample, or about zero where the mean stays:
// size[block][18], from which channel_unit takes the size of each channel.
template <bool STATS>
__global__ void __launch_bounds__(kSumThreads) k_rsum(const double* __restrict__ s, long long n, int subtract_mean,
                                                      double* __restrict__ part, float* __restrict__ size) {
  __shared__ double red[kSumThreads];
  __shared__ float red_sq[STATS ? kSumThreads : 1];
  __shared__ int red_top[STATS ? kSumThreads : 1];
  const double first = STATS ? s[threadIdx.x % 9] : 0.0, ref = subtract_mean ? first : 0.0;
  const int e = rough_unit(first);
  double acc = 0.0;
  float sq = 0.f;
  int top = 0;
  const long long step = (long long)gridDim.x * kSumThreads;
  for (long long i = (long long)blockIdx.x * kSumThreads + threadIdx.x; i < n; i += step) {
    const double v = s[i];
    acc += v;
    if constexpr (STATS) {
      const double d = v - ref;
      const float r = rough(d, e);
      sq = fmaf(r, r, sq);
      top = max(top, __double2hiint(d) & 0x7fffffff);
    }
  }
  red[threadIdx.x] = acc;
  if constexpr (STATS) {
    red_sq[threadIdx.x] = sq;
    red_top[threadIdx.x] = top;
  }
  __syncthreads();
  if (threadIdx.x < 72) {
    double v = 0.0;
    float q = 0.f;
    int m = 0;
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      const int at = ((threadIdx.x / 9) * 4 + k) * 9 + threadIdx.x % 9;
      v += red[at];
      if constexpr (STATS) {
        q += red_sq[at];
        m = max(m, red_top[at]);
      }
    }
    acc = v;
    sq = q;
    top = m;
  }
  __syncthreads();
  if (threadIdx.x < 72) {
    red[threadIdx.x] = acc;
    if constexpr (STATS) {
      red_sq[threadIdx.x] = sq;
      red_top[threadIdx.x] = top;
    }
  }
  __syncthreads();
  if (threadIdx.x < 9) {
    double v = 0.0;
    float q = 0.f;
    int m = 0;
#pragma unroll
    for (int h = 0; h < 8; ++h) {
      v += red[h * 9 + threadIdx.x];
      if constexpr (STATS) {
        q += red_sq[h * 9 + threadIdx.x];
        m = max(m, red_top[h * 9 + threadIdx.x]);
      }
    }
    part[blockIdx.x * 9 + threadIdx.x] = v;
    if constexpr (STATS) {
      size[blockIdx.x * 18 + threadIdx.x] = q;
      size[blockIdx.x * 18 + 9 + threadIdx.x] = __int_as_float(m);
    }
  }
}

// The power of two near the root mean square of x - mean over T samples (zero
// for a channel of zeros, NaN for one with a value that is not finite), from the sums of k_rsum: m is the mean less what they
// were taken about.  The sums may cancel or leave the float range where the
// first sample is far from the others; the largest magnitude bounds them: the
// largest |x - mean| lies between half and twice it, the root mean square
// within a factor sqrt(T) below.  (Beyond 2^+-500 products of two channels
// overflow or vanish.)
__device__ __forceinline__ double channel_unit(float sq, int top, double first, double m, int T) {
  if (top == 0) return 0.0;
  if (top >= 0x7ff00000 || !isfinite(m)) return __hiloint2double(0x7ff80000, 0);
  const int e = rough_unit(first), et = (top >> 20) - 1023;
  const float mr = rough(m, e), var = sq / (float)T - mr * mr;
  const int lo = et - 1 - (34 - __clz(T)) / 2;
  const int er = var > 0.f && var < __int_as_float(0x7f800000) ? ilogbf(var) / 2 + e - 1023 : lo;
  const int k = min(max(min(max(er, lo), et + 2), -500), 500);
  return __hiloint2double((k + 1023) << 20, 0);
}

// PACK: z [pack][T], channels (0, 1) (2, 3) (4, 5) (6, 7) (8, -), each divided by
// its unit, and pair_unit [45] the products of the pairs' units (see
// LoadSegment); else x [9][T].
template <bool PACK>
__global__ void __launch_bounds__(256) k_rprep(const double* __restrict__ s, int T, const double* __restrict__ part,
                                               const float* __restrict__ size, int n_part, int subtract_mean,
                                               double* __restrict__ out, double* __restrict__ pair_unit) {
  __shared__ double mean[9], unit[9], inv[9];
  const int lane = threadIdx.x & 31;
  for (int c = threadIdx.x >> 5; c < 9; c += 8) {
    double v = 0.0;
    float sq = 0.f;
    int top = 0;
    for (int b = lane; b < n_part; b += 32) {
      v += part[b * 9 + c];
      if constexpr (PACK) {
        sq += size[b * 18 + c];
        top = max(top, __float_as_int(size[b * 18 + 9 + c]));
      }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      v += __shfl_xor_sync(0xffffffffu, v, o);
      if constexpr (PACK) sq += __shfl_xor_sync(0xffffffffu, sq, o);
    }
    if constexpr (PACK) top = __reduce_max_sync(0xffffffffu, top);
    if (lane == 0) {
      const double m = subtract_mean ? v / (double)T : 0.0;
      mean[c] = m;
      if constexpr (PACK) {
        const double u = channel_unit(sq, top, s[c], subtract_mean ? m - s[c] : 0.0, T);
        unit[c] = u;
        // 1 / u; a channel that is zero or not finite goes in as zeros
        const double r = u > 0.0 ? __hiloint2double((2046 << 20) - __double2hiint(u), 0) : 0.0;
        inv[c] = r;
        mean[c] = r > 0.0 ? m * r : 0.0;
      }
    }
  }
  __syncthreads();
  if (PACK && blockIdx.x == 0 && threadIdx.x < 81) {
    const int p = threadIdx.x / 9, q = threadIdx.x % 9;
    if (p <= q) pair_unit[pair_row(p) + q - p] = unit[p] * unit[q];
  }
  const int t = blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= T) return;
  double x[10];
  x[9] = 0.0;
  if constexpr (PACK) {
#pragma unroll
    for (int c = 0; c < 9; ++c)  // (s - mean) / unit
      x[c] = inv[c] > 0.0 ? fma(s[(size_t)t * 9 + c], inv[c], -mean[c]) : 0.0;
    double2* z = reinterpret_cast<double2*>(out) + t;
#pragma unroll
    for (int k = 0; k < kPacks; ++k) z[(size_t)k * T] = make_double2(x[2 * k], x[2 * k + 1]);
  } else {
#pragma unroll
    for (int c = 0; c < 9; ++c) out[(size_t)c * T + t] = s[(size_t)t * 9 + c] - mean[c];
  }
}

// grid (lag tiles, 81 pairs); thread: lags tau0..tau0+3 of pair (p, q).
__global__ void __launch_bounds__(kCorrThreads) k_rcorr(const double* __restrict__ x, int T, int M,
                                                        double* __restrict__ C) {
  const int pair = blockIdx.y;
  const int p = pair / 9, q = pair % 9;
  const int tau0 = (blockIdx.x * kCorrThreads + threadIdx.x) * kLagsPerThread;
  if (tau0 > M) return;
  const double* xp = x + (size_t)p * T;
  const double* xq = x + (size_t)q * T;
  double acc[kLagsPerThread] = {0.0, 0.0, 0.0, 0.0};
  double win[kLagsPerThread];
#pragma unroll
  for (int j = 0; j < kLagsPerThread; ++j) win[j] = (tau0 + j < T) ? xq[tau0 + j] : 0.0;
  // x_q(t + tau0 + j) slides along t; terms with t + tau >= T are left out
  const int n = T - tau0;
  for (int t = 0; t < n; ++t) {
    const double a = xp[t];
#pragma unroll
    for (int j = 0; j < kLagsPerThread; ++j)
      if (t + j < n) acc[j] = fma(a, win[j], acc[j]);
#pragma unroll
    for (int j = 0; j < kLagsPerThread - 1; ++j) win[j] = win[j + 1];
    const int nxt = t + tau0 + kLagsPerThread;
    win[kLagsPerThread - 1] = nxt < T ? xq[nxt] : 0.0;
  }
#pragma unroll
  for (int j = 0; j < kLagsPerThread; ++j)
    if (tau0 + j <= M) C[((size_t)(tau0 + j)) * 81 + pair] = acc[j];
}

// lags [45][M + 1] from the ordered pairs' sums C [M + 1][81].
__global__ void k_rlags(const double* __restrict__ C, int T, int M, double* __restrict__ lags) {
  const long long g = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (g >= 45LL * (M + 1)) return;
  const int u = (int)(g / (M + 1)), tau = (int)(g % (M + 1));
  int p = 0, rem = u;
  while (rem >= 9 - p) { rem -= 9 - p; ++p; }
  const int q = p + rem;
  const double* c = C + (size_t)tau * 81;
  lags[g] = 0.5 * (c[p * 9 + q] + c[q * 9 + p]) / (double)(T - tau);
}

// ---- Fourier route ----

// Segment b of pack k (transform k nb + b): its L = N/2 samples, then zeros.
// Two channels share a complex transform and two pairs an inverse one, whose
// rounding is relative to the larger of the two.  So the channels go in divided
// by powers of two that make them about equal in size (exact), and StoreLags
// multiplies the pairs back: each component of the tensor is then as accurate
// relative to its own size as with direct sums (T = 5,000, M = 1,000, diagonal
// channels 1e4 times the others: error of the small L_pp over dt C_pp(0) 2.3e-8
// without, 3.2e-15 with, 9.1e-15 for the direct sums).  A channel with a value
// that is not finite goes in as zeros and its pairs come out as NaN, so that it
// does not spoil those that it shares a transform with.
struct LoadSegment {
  static constexpr bool kHalfZero = true;
  const double2* z;
  int T, nb, logN;
  __device__ __forceinline__ double2 operator()(int f, unsigned i) const {
    const int k = f / nb, b = f - k * nb;
    const long long t = ((long long)b << (logN - 1)) + i;
    if (t >= T) return make_double2(0.0, 0.0);
    return __ldg(z + (size_t)k * T + t);
  }
};

// Rows of G: 0 = {0, 3}, 1 = {1, 2}, 2 = {4, 5, 6, 7, 8}: 15 pairs each, so that
// the sums, the 9 transforms of this and of the next segment stay in registers.
template <int G>
__host__ __device__ constexpr bool has_row(int p) {
  return G == 0 ? (p == 0 || p == 3) : (G == 1 ? (p == 1 || p == 2) : p >= 4);
}

// part[chunk][45][N/2 + 1]: the pairs' spectra over segments [b0, b1), four
// times the sums of the header.
template <int G>
__device__ __forceinline__ void cross_rows(const double2* __restrict__ z, int logN, int nb, int b0, int b1, unsigned f,
                                           double2* __restrict__ part) {
  constexpr int C0 = G == 2 ? 4 : (G == 1 ? 1 : 0);  // channels below are not read
  const unsigned N = 1u << logN, half = N >> 1, g = (N - f) & (N - 1);
  const double sgn = (f & 1u) ? -1.0 : 1.0;
  auto load = [&](int b, double2* x) {
#pragma unroll
    for (int k = C0 / 2; k < kPacks; ++k) {
      double2 u = make_double2(0.0, 0.0), v = u;
      if (b < nb) {
        const size_t o = ((size_t)k * nb + b) << logN;
        u = z[o + f];
        v = z[o + g];
      }
      x[2 * k] = make_double2(u.x + v.x, u.y - v.y);
      if (k < kPacks - 1) x[2 * k + 1] = make_double2(u.y + v.y, v.x - u.x);
    }
  };
  double2 x[9], nx[9], w[9];
  double2 acc[45];
#pragma unroll
  for (int u = 0; u < 45; ++u) acc[u] = make_double2(0.0, 0.0);
  load(b0, x);
  for (int b = b0; b < b1; ++b) {
    load(b + 1, nx);
#pragma unroll
    for (int c = C0; c < 9; ++c) w[c] = make_double2(fma(sgn, nx[c].x, x[c].x), fma(sgn, nx[c].y, x[c].y));
#pragma unroll
    for (int p = 0; p < 9; ++p) {
      if (!has_row<G>(p)) continue;
#pragma unroll
      for (int q = p; q < 9; ++q) {
        double2& a = acc[pair_row(p) + q - p];
        a.x = fma(x[p].x, w[q].x, fma(x[p].y, w[q].y, a.x));
        a.y = fma(x[p].x, w[q].y, fma(-x[p].y, w[q].x, a.y));
        if (q != p) {
          a.x = fma(x[q].x, w[p].x, fma(x[q].y, w[p].y, a.x));
          a.y = fma(x[q].x, w[p].y, fma(-x[q].y, w[p].x, a.y));
        }
      }
    }
#pragma unroll
    for (int c = C0; c < 9; ++c) x[c] = nx[c];
  }
#pragma unroll
  for (int p = 0; p < 9; ++p) {
    if (!has_row<G>(p)) continue;
#pragma unroll
    for (int q = p; q < 9; ++q) {
      const int u = pair_row(p) + q - p;
      part[(size_t)u * (half + 1) + f] = q == p ? fft::add(acc[u], acc[u]) : acc[u];
    }
  }
}

// grid (frequency tiles, 3 row groups, chunks of segments).  FP64-bound: 8
// multiply-adds per pair, frequency and segment.
__global__ void __launch_bounds__(128) k_rcross(const double2* __restrict__ z, int logN, int nb, int per_chunk,
                                                double2* __restrict__ part) {
  const unsigned half = 1u << (logN - 1);
  const unsigned f = blockIdx.x * blockDim.x + threadIdx.x;
  if (f > half) return;
  const int b0 = blockIdx.z * per_chunk, b1 = min(nb, b0 + per_chunk);
  double2* dst = part + (size_t)blockIdx.z * 45 * (half + 1);
  if (blockIdx.y == 0) cross_rows<0>(z, logN, nb, b0, b1, f, dst);
  else if (blockIdx.y == 1) cross_rows<1>(z, logN, nb, b0, b1, f, dst);
  else cross_rows<2>(z, logN, nb, b0, b1, f, dst);
}

// The chunks of k_rcross summed in order into the first.
__global__ void __launch_bounds__(256) k_rsum_chunks(double2* __restrict__ part, long long n, int chunks) {
  const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  double2 v = part[i];
  for (int c = 1; c < chunks; ++c) v = fft::add(v, part[c * n + i]);
  part[i] = v;
}

// Pairs 2f and 2f + 1 (spectra of real sequences) as one complex spectrum.
struct LoadCross {
  static constexpr bool kHalfZero = false;
  const double2* part;
  int logN;
  __device__ __forceinline__ double2 operator()(int f, unsigned i) const {
    const unsigned N = 1u << logN, half = N >> 1, g = i <= half ? i : N - i;
    const double2* s = part + (size_t)(2 * f) * (half + 1) + g;
    const double2 u = s[0], v = 2 * f + 1 < 45 ? s[half + 1] : make_double2(0.0, 0.0);
    return i <= half ? make_double2(u.x - v.y, u.y + v.x) : make_double2(u.x + v.y, v.x - u.y);
  }
};
struct StoreLags {
  double* lags;            // [45][M + 1]
  const double* pair_unit;  // [45], see LoadSegment
  int T, M;
  double scale;  // 1 / (8 N)
  __device__ __forceinline__ void operator()(int f, unsigned i, double2 v) const {
    if (i > (unsigned)M) return;
    const double s = scale / (double)(T - (int)i);
    lags[(size_t)(2 * f) * (M + 1) + i] = v.x * s * pair_unit[2 * f];
    if (2 * f + 1 < 45) lags[(size_t)(2 * f + 1) * (M + 1) + i] = v.y * s * pair_unit[2 * f + 1];
  }
};

__device__ __forceinline__ double contract(const double* __restrict__ Lk, const double w[9]) {
  double acc = 0.0;
#pragma unroll
  for (int p = 0; p < 9; ++p) {
    double r = 0.0;
#pragma unroll
    for (int q = 0; q < 9; ++q) r = fma(Lk[p * 9 + q], w[q], r);
    acc = fma(w[p], r, acc);
  }
  return acc;
}

__global__ void k_rpolar(const double* __restrict__ L, int M, int O, const double* __restrict__ n,
                         const double* __restrict__ eps, double* __restrict__ spec) {
  const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= (long long)O * (M + 1)) return;
  const int o = (int)(i / (M + 1)), k = (int)(i % (M + 1));
  double w[9];
#pragma unroll
  for (int g = 0; g < 3; ++g)
#pragma unroll
    for (int d = 0; d < 3; ++d) w[g * 3 + d] = n[o * 3 + g] * eps[o * 3 + d];
  spec[i] = contract(L + (size_t)k * 81, w);
}

// Crystal turned by theta about `axis` (the laser direction): incoming
// polarization R^T X, observed R^T X (parallel) or R^T Y (crossed), with X, Y
// the two crystal axes orthogonal to `axis` in cyclic order.
//
// With e = (c, -s) and y = (s, c) on the axes (a, b), the weights are
//   parallel (aa, ab, ba, bb) = (c^2, -cs, -cs, s^2), crossed = (cs, -s^2, c^2, -cs),
// so each spectrum is a quadratic form in (u, v, z) = (c^2, cs, s^2): six
// coefficients per frequency, then six multiply-adds per angle instead of 90 (the
// contraction over all nine components was FP64-bound: 147 us for 181 angles and
// 2001 frequencies).  Entries of L outside the plane have weight zero; they are
// still multiplied by it, so a NaN or infinity there shows as before.
// grid (frequency tiles, angle chunks)
constexpr int kPortoAngles = 16;
__global__ void __launch_bounds__(128) k_rporto(const double* __restrict__ L, int M, int O,
                                                const double* __restrict__ theta, int axis, double* __restrict__ par,
                                                double* __restrict__ crs) {
  __shared__ double mono[kPortoAngles][6];  // u^2, uv, uz, v^2, vz, z^2
  const int k = blockIdx.x * blockDim.x + threadIdx.x;
  const int a = (axis + 1) % 3, b = (axis + 2) % 3;
  const int id[4] = {a * 3 + a, a * 3 + b, b * 3 + a, b * 3 + b};
  const double* Lk = L + (size_t)min(k, M) * 81;
  double zero = 0.0, q[4][4];
  for (int r = 0; r < 9; ++r) {
    const bool row = r / 3 != axis && r % 3 != axis;
    for (int c = 0; c < 9; ++c)
      if (!row || c / 3 == axis || c % 3 == axis) zero = fma(Lk[r * 9 + c], 0.0, zero);
  }
#pragma unroll
  for (int i = 0; i < 4; ++i)
#pragma unroll
    for (int j = 0; j < 4; ++j) q[i][j] = Lk[id[i] * 9 + id[j]];
  const double p[6] = {q[0][0],
                       -((q[0][1] + q[1][0]) + (q[0][2] + q[2][0])),
                       q[0][3] + q[3][0],
                       (q[1][1] + q[2][2]) + (q[1][2] + q[2][1]),
                       -((q[1][3] + q[3][1]) + (q[2][3] + q[3][2])),
                       q[3][3]};
  const double x[6] = {q[2][2],
                       (q[0][2] + q[2][0]) - (q[2][3] + q[3][2]),
                       -(q[1][2] + q[2][1]),
                       (q[0][0] + q[3][3]) - (q[0][3] + q[3][0]),
                       (q[1][3] + q[3][1]) - (q[0][1] + q[1][0]),
                       q[1][1]};
  for (long long o0 = (long long)blockIdx.y * kPortoAngles; o0 < O; o0 += (long long)gridDim.y * kPortoAngles) {
    const int no = (int)min((long long)kPortoAngles, O - o0);
    __syncthreads();
    if ((int)threadIdx.x < no) {
      double sn, cs;
      sincos(theta[o0 + threadIdx.x], &sn, &cs);
      const double u = cs * cs, v = cs * sn, z = sn * sn;
      double* m = mono[threadIdx.x];
      m[0] = u * u; m[1] = u * v; m[2] = u * z; m[3] = v * v; m[4] = v * z; m[5] = z * z;
    }
    __syncthreads();
    if (k > M) continue;
    for (int o = 0; o < no; ++o) {
      double vp = zero, vx = zero;
#pragma unroll
      for (int t = 0; t < 6; ++t) {
        vp = fma(p[t], mono[o][t], vp);
        vx = fma(x[t], mono[o][t], vx);
      }
      const size_t at = (size_t)(o0 + o) * (M + 1) + k;
      par[at] = vp;
      crs[at] = vx;
    }
  }
}

unsigned blocks_for(long long n, int threads) { return (unsigned)((n + threads - 1) / threads); }

bool have_device() {
  int ndev = 0;
  if (cudaGetDeviceCount(&ndev) != cudaSuccess || ndev == 0) {
    cudaGetLastError();
    return false;
  }
  return true;
}

}  // namespace

}  // namespace tnep

using namespace tnep;

extern "C" {

tnep_status tnep_raman_tensor(const double* series, int T, double dt_fs, int max_lag, int subtract_mean,
                              double* freq_cm1, double* L, void* stream) {
  if (!series || !freq_cm1 || !L) return fail(TNEP_ERR_INVALID, "NULL buffer");
  if (T < 2) return fail(TNEP_ERR_INVALID, "need at least two samples");
  if (!(dt_fs > 0.0)) return fail(TNEP_ERR_INVALID, "dt must be positive");
  const int M = max_lag <= 0 ? T / 2 : max_lag;
  if (M < 1 || M >= T) return fail(TNEP_ERR_INVALID, "max_lag must be in [1, T)");
  if (!have_device()) return fail(TNEP_ERR_NO_DEVICE, "no CUDA device");
  cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
  const bool use_fft = raman_uses_fft(T, M);
  const int logN = fft::log2_at_least(2LL * M);
  const int nb = (int)(((long long)T + (1ll << (logN - 1)) - 1) >> (logN - 1));
  const unsigned half = 1u << (logN - 1);
  // chunks of segments: enough (frequency, row group, chunk) threads to fill the chip
  int chunks = (int)std::min<long long>(nb, std::max<long long>(1, (1ll << 15) >> (logN - 1)));
  const int per_chunk = (nb + chunks - 1) / chunks;
  chunks = (nb + per_chunk - 1) / per_chunk;
  const int n_part = (int)std::min<long long>(kMaxSumBlocks, (9LL * T + 4 * kSumThreads - 1) / (4 * kSumThreads));
  size_t at = 0;
  auto place = [&](size_t bytes) {
    const size_t o = at;
    at += (bytes + 255) & ~size_t(255);
    return o;
  };
  const size_t nF = (size_t)(M + 1), nL = (size_t)(M + 1) * 81, nZ = (size_t)std::max(kPacks * nb, 23) << logN;
  const size_t o_s = place(sizeof(double) * 9 * (size_t)T);
  const size_t o_part = place(sizeof(double) * 9 * n_part), o_size = place(sizeof(float) * 18 * n_part);
  const size_t o_unit = place(sizeof(double) * 45);
  const size_t o_x = place(sizeof(double) * (use_fft ? 2 * kPacks : 9) * (size_t)T);
  const size_t o_a = place(use_fft ? sizeof(double2) * nZ : sizeof(double) * nL);
  const size_t o_b = place(use_fft ? sizeof(double2) * nZ : 0);
  const size_t o_tw = place(use_fft ? sizeof(double2) * fft::table_size(logN) : 0);
  const size_t o_cross = place(use_fft ? sizeof(double2) * 45 * chunks * (size_t)(half + 1) : 0);
  const size_t o_lags = place(sizeof(double) * 45 * nF), o_f = place(sizeof(double) * nF);
  const size_t o_l = place(sizeof(double) * nL), o_cos = place(cosine_work_bytes(M, 45));
  char* d = nullptr;
  TNEP_CUDA(dev_malloc_async((void**)&d, at, st));
  auto dbl = [&](size_t o) { return reinterpret_cast<double*>(d + o); };
  double *d_s = dbl(o_s), *d_part = dbl(o_part), *d_unit = dbl(o_unit), *d_x = dbl(o_x);
  float* d_size = reinterpret_cast<float*>(d + o_size);
  double *d_lags = dbl(o_lags), *d_f = dbl(o_f), *d_l = dbl(o_l);
  cudaError_t e = cudaMemcpyAsync(d_s, series, sizeof(double) * 9 * (size_t)T, cudaMemcpyDefault, st);
  if (e == cudaSuccess) {
    if (use_fft) k_rsum<true><<<n_part, kSumThreads, 0, st>>>(d_s, 9LL * T, subtract_mean, d_part, d_size);
    else k_rsum<false><<<n_part, kSumThreads, 0, st>>>(d_s, 9LL * T, subtract_mean, d_part, d_size);
    count_launches(3);
    if (!use_fft) {
      double* d_c = dbl(o_a);
      k_rprep<false><<<blocks_for(T, 256), 256, 0, st>>>(d_s, T, d_part, d_size, n_part, subtract_mean, d_x, d_unit);
      const int tiles = (M + 1 + kCorrThreads * kLagsPerThread - 1) / (kCorrThreads * kLagsPerThread);
      k_rcorr<<<dim3(tiles, 81), kCorrThreads, 0, st>>>(d_x, T, M, d_c);
      k_rlags<<<blocks_for(45LL * (M + 1), 256), 256, 0, st>>>(d_c, T, M, d_lags);
      count_launches(1);
      e = cudaGetLastError();
    } else {
      double2 *za = reinterpret_cast<double2*>(d + o_a), *zb = reinterpret_cast<double2*>(d + o_b);
      double2* tw = reinterpret_cast<double2*>(d + o_tw);
      double2 *zx = reinterpret_cast<double2*>(d_x), *cross = reinterpret_cast<double2*>(d + o_cross);
      k_rprep<true><<<blocks_for(T, 256), 256, 0, st>>>(d_s, T, d_part, d_size, n_part, subtract_mean, d_x, d_unit);
      e = launch_fft_table(logN, tw, st);
      double2* fin = fft::last_source(logN, kPacks * nb) == 0 ? zb : za;
      if (e == cudaSuccess)
        e = fft::transform<false>(LoadSegment{zx, T, nb, logN}, fft::StorePlain{fin, logN}, za, zb, tw, logN,
                                  kPacks * nb, st);
      if (e == cudaSuccess) {
        k_rcross<<<dim3((half + 1 + 127) / 128, 3, chunks), 128, 0, st>>>(fin, logN, nb, per_chunk, cross);
        const long long n = 45LL * (half + 1);
        count_launches(1);
        if (chunks > 1) k_rsum_chunks<<<blocks_for(n, 256), 256, 0, st>>>(cross, n, chunks);
        e = fft::transform<true>(LoadCross{cross, logN},
                                 StoreLags{d_lags, d_unit, T, M, 1.0 / (8.0 * (double)(1ll << logN))}, za, zb, tw, logN,
                                 23, st);
      }
    }
    if (e == cudaSuccess)
      e = launch_cosine(d_lags, M, 45, CosineOut{1, 0, dt_fs, d_f, d_l}, nullptr, d + o_cos, st);
  }
  if (e == cudaSuccess) e = cudaMemcpyAsync(freq_cm1, d_f, sizeof(double) * nF, cudaMemcpyDefault, st);
  if (e == cudaSuccess) e = cudaMemcpyAsync(L, d_l, sizeof(double) * nL, cudaMemcpyDefault, st);
  tnep_status rc = e == cudaSuccess ? TNEP_OK : cuda_fail(e, "raman tensor");
  cudaFreeAsync(d, st);
  e = cudaStreamSynchronize(st);
  if (e != cudaSuccess && rc == TNEP_OK) rc = cuda_fail(e, "raman tensor sync");
  return rc;
}

tnep_status tnep_raman_polarized(const double* L, int max_lag, int n_orient, const double* n, const double* eps,
                                 double* spec, void* stream) {
  if (!L || !n || !eps || !spec) return fail(TNEP_ERR_INVALID, "NULL buffer");
  if (max_lag < 1 || n_orient < 1) return fail(TNEP_ERR_INVALID, "need max_lag >= 1 and n_orient >= 1");
  if (!have_device()) return fail(TNEP_ERR_NO_DEVICE, "no CUDA device");
  cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
  const size_t nL = (size_t)(max_lag + 1) * 81, nV = (size_t)n_orient * 3, nO = (size_t)n_orient * (max_lag + 1);
  double* d = nullptr;
  TNEP_CUDA(dev_malloc_async((void**)&d, sizeof(double) * (nL + 2 * nV + nO), st));
  double *d_l = d, *d_n = d_l + nL, *d_e = d_n + nV, *d_o = d_e + nV;
  cudaError_t e = cudaMemcpyAsync(d_l, L, sizeof(double) * nL, cudaMemcpyDefault, st);
  if (e == cudaSuccess) e = cudaMemcpyAsync(d_n, n, sizeof(double) * nV, cudaMemcpyDefault, st);
  if (e == cudaSuccess) e = cudaMemcpyAsync(d_e, eps, sizeof(double) * nV, cudaMemcpyDefault, st);
  if (e == cudaSuccess) {
    k_rpolar<<<blocks_for((long long)nO, 256), 256, 0, st>>>(d_l, max_lag, n_orient, d_n, d_e, d_o);
    count_launches(1);
    e = cudaGetLastError();
  }
  if (e == cudaSuccess) e = cudaMemcpyAsync(spec, d_o, sizeof(double) * nO, cudaMemcpyDefault, st);
  tnep_status rc = e == cudaSuccess ? TNEP_OK : cuda_fail(e, "raman polarized");
  cudaFreeAsync(d, st);
  e = cudaStreamSynchronize(st);
  if (e != cudaSuccess && rc == TNEP_OK) rc = cuda_fail(e, "raman polarized sync");
  return rc;
}

tnep_status tnep_raman_porto_map(const double* L, int max_lag, int n_theta, const double* theta, int axis,
                                 double* spec_parallel, double* spec_crossed, void* stream) {
  if (!L || !theta || !spec_parallel || !spec_crossed) return fail(TNEP_ERR_INVALID, "NULL buffer");
  if (max_lag < 1 || n_theta < 1) return fail(TNEP_ERR_INVALID, "need max_lag >= 1 and n_theta >= 1");
  if (axis < 0 || axis > 2) return fail(TNEP_ERR_INVALID, "axis must be 0, 1 or 2");
  if (!have_device()) return fail(TNEP_ERR_NO_DEVICE, "no CUDA device");
  cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
  const size_t nL = (size_t)(max_lag + 1) * 81, nO = (size_t)n_theta * (max_lag + 1);
  double* d = nullptr;
  TNEP_CUDA(dev_malloc_async((void**)&d, sizeof(double) * (nL + n_theta + 2 * nO), st));
  double *d_l = d, *d_t = d_l + nL, *d_p = d_t + n_theta, *d_c = d_p + nO;
  cudaError_t e = cudaMemcpyAsync(d_l, L, sizeof(double) * nL, cudaMemcpyDefault, st);
  if (e == cudaSuccess) e = cudaMemcpyAsync(d_t, theta, sizeof(double) * n_theta, cudaMemcpyDefault, st);
  if (e == cudaSuccess) {
    k_rporto<<<dim3(blocks_for(max_lag + 1LL, 128), std::min(blocks_for(n_theta, kPortoAngles), 65535u)), 128, 0, st>>>(
        d_l, max_lag, n_theta, d_t, axis, d_p, d_c);
    count_launches(1);
    e = cudaGetLastError();
  }
  if (e == cudaSuccess) e = cudaMemcpyAsync(spec_parallel, d_p, sizeof(double) * nO, cudaMemcpyDefault, st);
  if (e == cudaSuccess) e = cudaMemcpyAsync(spec_crossed, d_c, sizeof(double) * nO, cudaMemcpyDefault, st);
  tnep_status rc = e == cudaSuccess ? TNEP_OK : cuda_fail(e, "raman porto map");
  cudaFreeAsync(d, st);
  e = cudaStreamSynchronize(st);
  if (e != cudaSuccess && rc == TNEP_OK) rc = cuda_fail(e, "raman porto map sync");
  return rc;
}

}  // extern "C"

// Spectrum tail in float64 (Sec. II.F, Eqs. 5-6; Sec. II.G, Eqs. 7-9).
//
//   sums   column sums of the series (and the cosine table), one partial per CTA
//   prep   signal x(t): IR mu (3 comps); Raman iso gamma = Tr(alpha)/3;
//          Raman aniso beta = alpha - gamma I (9 comps); mean removed if asked
//   acf    one warp per lag tau: C(tau) = 1/(T - tau) sum_t x(t).x'(t + tau),
//          with x' = x (IR: times 1/3) or x'_{ab} = x_{ba} (Tr[beta beta])
//   cos    S_k = dt [C(0) + 2 sum_{tau=1}^{M} C(tau) cos(pi k tau / M)]
//          (IR times (2 pi nu_k)^2), nu_k = k / (2 M dt); one warp per frequency
// Every sum runs in a fixed order (strided partial sums, then a tree), so the
// results do not depend on the launch.
//
// Fourier route for the autocorrelation (rule at spectrum_uses_fft): the
// series is cut into segments of L = N/2 >= M samples (N a power of two), each
// zero-padded to N and transformed, two real channels per complex transform.
// With X_b the transform of segment b, F_b = X_b + (-1)^f X_{b+1} is that of the
// 2 L samples from its start, so sum_b conj(X_{b,p}) F_{b,q} is the spectrum of
// a circular correlation whose lags 0..L are the linear ones, and one inverse
// transform of length N (not of the whole series' length) gives C(tau).
//
// Cosine transform of long correlations (rule at cosine_uses_chirp): with
// w_n = exp(i pi n^2 / 2M), cos(pi k tau / M) = Re[w_k w_tau conj(w_{k-tau})], a
// convolution done with transforms of length P >= 2M + 1.
//
// What bounds it: FP64 instructions (two lanes per clock and SM) and, for
// short series, launches.  Measured on a GB300 (whole call, host series in,
// spectrum out): T = 1e5, M = 1e4, aniso 3392 -> 368 us (before, 2487 us went
// to the preparation in one CTA, 310 us to 34 radix-2 passes over the whole
// padded series and 228 us to cosine sums with a 64-bit remainder per term).

#include <algorithm>

#include "fft.cuh"
#include "tnep_internal.cuh"

namespace tnep {

namespace {

constexpr double kCmPerInvFs = 1.0 / 2.99792458e-5;
constexpr int kSumThreads = 288;  // a multiple of 3 and 9: a thread keeps its column
constexpr int kMaxSumBlocks = 128;

__device__ __forceinline__ double warp_sum(double v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// Blocks [0, sum_blocks): partial column sums of the series [T][C] (C = 3 or
// 9) in a fixed order, part[block][C].  Further blocks: cosine table cos(pi m / M).
__global__ void __launch_bounds__(kSumThreads) k_colsum(const double* __restrict__ s, long long n, int C,
                                                        int sum_blocks, double* __restrict__ part, int M,
                                                        double* __restrict__ tab) {
  if ((int)blockIdx.x >= sum_blocks) {
    const int m = ((int)blockIdx.x - sum_blocks) * kSumThreads + threadIdx.x;
    if (m < 2 * M) tab[m] = cospi((double)m / (double)M);
    return;
  }
  __shared__ double red[kSumThreads], red2[72];
  double acc = 0.0;
  for (long long i = (long long)blockIdx.x * kSumThreads + threadIdx.x; i < n; i += (long long)sum_blocks * kSumThreads)
    acc += s[i];
  red[threadIdx.x] = acc;
  __syncthreads();
  if (threadIdx.x < 8 * C) {
    const int c = threadIdx.x % C, h = threadIdx.x / C, per = kSumThreads / C / 8;
    double v = 0.0;
    for (int k = 0; k < per; ++k) v += red[(h * per + k) * C + c];
    red2[threadIdx.x] = v;
  }
  __syncthreads();
  if (threadIdx.x < C) {
    double v = 0.0;
#pragma unroll
    for (int h = 0; h < 8; ++h) v += red2[h * C + threadIdx.x];
    part[blockIdx.x * C + threadIdx.x] = v;
  }
}

// Means of the columns from the partials, by the first C warps of a CTA.
__device__ __forceinline__ void column_means(const double* part, int sum_blocks, int C, int T, int subtract_mean,
                                             double* mean) {
  const int lane = threadIdx.x & 31;
  for (int c = threadIdx.x >> 5; c < C; c += blockDim.x >> 5) {
    double v = 0.0;
    for (int b = lane; b < sum_blocks; b += 32) v += part[b * C + c];
    v = warp_sum(v);
    if (lane == 0) mean[c] = subtract_mean ? v / (double)T : 0.0;
  }
  __syncthreads();
}

// The prepared channels of one sample.
template <int KIND>
__device__ __forceinline__ void channels(const double* __restrict__ s, const double* mean, double* x) {
  if constexpr (KIND == TNEP_SPECTRUM_IR) {
#pragma unroll
    for (int c = 0; c < 3; ++c) x[c] = s[c] - mean[c];
  } else {
    const double g = (s[0] + s[4] + s[8]) / 3.0, gm = (mean[0] + mean[4] + mean[8]) / 3.0;
    if constexpr (KIND == TNEP_SPECTRUM_RAMAN_ISO) {
      x[0] = g - gm;
    } else {
#pragma unroll
      for (int c = 0; c < 9; ++c) {
        const bool diag = c == 0 || c == 4 || c == 8;
        x[c] = diag ? (s[c] - g) - (mean[c] - gm) : s[c] - mean[c];
      }
    }
  }
}
template <int KIND>
constexpr int n_channels() { return KIND == TNEP_SPECTRUM_IR ? 3 : (KIND == TNEP_SPECTRUM_RAMAN_ISO ? 1 : 9); }
template <int KIND>
constexpr int n_packs() { return KIND == TNEP_SPECTRUM_IR ? 2 : (KIND == TNEP_SPECTRUM_RAMAN_ISO ? 1 : 4); }

// Direct route: x [T][channels].  Fourier route (PACK): z [pack][T], two
// channels per complex value: IR (0, 1) (2, -); aniso (0, 4) (1, 3) (2, 6)
// (5, 7), with beta traceless channel 8 = -(0) - (4).
template <int KIND, bool PACK>
__global__ void __launch_bounds__(256) k_prep(const double* __restrict__ series, int T, const double* __restrict__ part,
                                              int sum_blocks, int subtract_mean, double* __restrict__ out) {
  constexpr int C = KIND == TNEP_SPECTRUM_IR ? 3 : 9;
  __shared__ double mean[9];
  column_means(part, sum_blocks, C, T, subtract_mean, mean);
  const int t = blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= T) return;
  double x[9];
  channels<KIND>(series + (size_t)t * C, mean, x);
  if constexpr (!PACK) {
    constexpr int cx = n_channels<KIND>();
#pragma unroll
    for (int c = 0; c < cx; ++c) out[(size_t)t * cx + c] = x[c];
  } else {
    double2* z = reinterpret_cast<double2*>(out) + t;
    if constexpr (KIND == TNEP_SPECTRUM_IR) {
      z[0] = make_double2(x[0], x[1]);
      z[T] = make_double2(x[2], 0.0);
    } else if constexpr (KIND == TNEP_SPECTRUM_RAMAN_ISO) {
      z[0] = make_double2(x[0], 0.0);
    } else {
      z[0] = make_double2(x[0], x[4]);
      z[T] = make_double2(x[1], x[3]);
      z[2 * (size_t)T] = make_double2(x[2], x[6]);
      z[3 * (size_t)T] = make_double2(x[5], x[7]);
    }
  }
}

// One warp per lag: short series are bound by FP64 issue (IR, T = 2000,
// M = 1000: 4.5e6 multiply-adds), where the CTA-wide tree this replaces cost
// as much again (21 us).
__global__ void __launch_bounds__(64) k_acf(const double* __restrict__ x, int T, int M, int kind,
                                             double* __restrict__ acf) {
  const int tau = (int)(((long long)blockIdx.x * blockDim.x + threadIdx.x) >> 5), lane = threadIdx.x & 31;
  if (tau > M) return;
  const int n = T - tau;
  double acc = 0.0, acc2 = 0.0;
  if (kind != TNEP_SPECTRUM_RAMAN_ANISO) {
    // products of the flat signal with itself tau samples on, four loads of each in flight
    const int cx = kind == TNEP_SPECTRUM_IR ? 3 : 1;
    const double* y = x + (size_t)tau * cx;
    const long long m = (long long)n * cx;
    // (one warp per quarter of an SM: the next group loads under this one's FP64 issue)
    constexpr int U = 4;
    double s4[U] = {0.0, 0.0, 0.0, 0.0}, xa[U], xb[U];
    long long i = lane;
    const long long full = m / (32 * U) * (32 * U);
    if (full > 0) {
#pragma unroll
      for (int u = 0; u < U; ++u) { xa[u] = x[i + 32 * u]; xb[u] = y[i + 32 * u]; }
    }
    for (; i < full; i += 32 * U) {
      double na[U], nb[U];
      const long long nx = i + 32 * U < full ? i + 32 * U : i;
#pragma unroll
      for (int u = 0; u < U; ++u) { na[u] = x[nx + 32 * u]; nb[u] = y[nx + 32 * u]; }
#pragma unroll
      for (int u = 0; u < U; ++u) s4[u] = fma(xa[u], xb[u], s4[u]);
#pragma unroll
      for (int u = 0; u < U; ++u) { xa[u] = na[u]; xb[u] = nb[u]; }
    }
    for (; i < m; i += 32) acc = fma(x[i], y[i], acc);
    acc += s4[0] + s4[1];
    acc2 += s4[2] + s4[3];
  } else {
    for (int t = lane; t < n; t += 32) {
      const double* a = x + (size_t)t * 9;
      const double* b = x + (size_t)(t + tau) * 9;
#pragma unroll
      for (int u = 0; u < 3; ++u)
#pragma unroll
        for (int v = 0; v < 3; ++v) {
          if ((u + v) & 1) acc2 = fma(a[3 * u + v], b[3 * v + u], acc2);
          else acc = fma(a[3 * u + v], b[3 * v + u], acc);
        }
    }
  }
  const double s = warp_sum(acc + acc2);
  if (lane == 0) acf[tau] = s / (double)n / (kind == TNEP_SPECTRUM_IR ? 3.0 : 1.0);
}

// ---- cosine transform ----

__device__ __forceinline__ void store_cos(const CosineOut& o, int seq, int k, int M, double v) {
  if (o.mode == 0) {
    const double nu = (double)k / (2.0 * M * o.dt);
    if (o.kind == TNEP_SPECTRUM_IR) {
      const double w = 2.0 * 3.14159265358979323846 * nu;
      v *= w * w;
    }
    o.spec[k] = v;
    o.freq[k] = nu * kCmPerInvFs;
  } else {
    int p = 0, rem = seq;
    while (rem >= 9 - p) { rem -= 9 - p; ++p; }
    const int q = p + rem;
    o.spec[(size_t)k * 81 + p * 9 + q] = v;
    o.spec[(size_t)k * 81 + q * 9 + p] = v;
    if (seq == 0) o.freq[k] = (double)k / (2.0 * M * o.dt) * kCmPerInvFs;
  }
}

// One warp per (frequency, sequence); the table index k tau mod 2M advances by
// 32 k mod 2M (the 64-bit remainder per term cost more than the FP64 sums), four
// terms in flight.
__global__ void __launch_bounds__(64) k_cosine(const double* __restrict__ lags, const double* __restrict__ tab,
                                               int M, const CosineOut o) {
  const int k = (int)(((long long)blockIdx.x * blockDim.x + threadIdx.x) >> 5), lane = threadIdx.x & 31;
  if (k > M) return;
  const double* c = lags + (size_t)blockIdx.y * (M + 1);
  const unsigned period = 2u * (unsigned)M;
  unsigned step, idx;
  if (M < (1 << 26)) {
    step = (32u * (unsigned)k) % period;
    idx = ((unsigned)k * (unsigned)(1 + lane)) % period;
  } else {
    step = (unsigned)((32ull * (unsigned)k) % period);
    idx = (unsigned)(((unsigned long long)k * (unsigned)(1 + lane)) % period);
  }
  auto next = [&](unsigned i) {  // both below the period, which fits 31 bits
    i += step;
    return i >= period ? i - period : i;
  };
  double a0 = 0.0, a1 = 0.0, a2 = 0.0, a3 = 0.0;
  int tau = 1 + lane;
  for (; tau + 96 <= M; tau += 128) {
    const unsigned i1 = next(idx), i2 = next(i1), i3 = next(i2);
    const double t0 = __ldg(tab + idx), t1 = __ldg(tab + i1), t2 = __ldg(tab + i2), t3 = __ldg(tab + i3);
    a0 = fma(c[tau], t0, a0);
    a1 = fma(c[tau + 32], t1, a1);
    a2 = fma(c[tau + 64], t2, a2);
    a3 = fma(c[tau + 96], t3, a3);
    idx = next(i3);
  }
  for (; tau <= M; tau += 32) {
    a0 = fma(c[tau], __ldg(tab + idx), a0);
    idx = next(idx);
  }
  const double acc = warp_sum((a0 + a1) + (a2 + a3));
  if (lane == 0) store_cos(o, blockIdx.y, k, M, o.dt * fma(2.0, acc, c[0]));
}

// Chirp w_n, n = 0..M, and the twiddle table of the transform.
__global__ void __launch_bounds__(256) k_chirp_tables(int M, double2* __restrict__ w, int logP, double2* __restrict__ tab) {
  const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  double s, c;
  if (i <= M) {
    const unsigned long long a = ((unsigned long long)i * (unsigned long long)i) % (4ull * M);  // angle mod 2 pi
    sincospi((double)a / (2.0 * M), &s, &c);
    w[i] = make_double2(c, s);
  }
  const long long m = i - (M + 1);
  if (m >= 0 && m <= (1ll << (logP - 3))) {
    sincospi(2.0 * (double)m / (double)(1ll << logP), &s, &c);
    tab[m] = make_double2(c, s);
  }
}

// Sequences 0..nseq-1: C(tau) w_tau (half of it at 0); sequence nseq: conj(w_|n|).
struct LoadChirp {
  static constexpr bool kHalfZero = false;
  const double* lags;
  const double2* w;
  int M, nseq, logP;
  __device__ __forceinline__ double2 operator()(int f, unsigned i) const {
    const unsigned P = 1u << logP;
    if (f < nseq) {
      if (i > (unsigned)M) return make_double2(0.0, 0.0);
      const double c = lags[(size_t)f * (M + 1) + i] * (i == 0 ? 0.5 : 1.0);
      const double2 a = w[i];
      return make_double2(c * a.x, c * a.y);
    }
    const unsigned n = i <= (unsigned)M ? i : P - i;
    if (n > (unsigned)M) return make_double2(0.0, 0.0);
    const double2 a = w[n];
    return make_double2(a.x, fft::flip(a.y, 0x80000000u));
  }
};
struct LoadChirpProduct {
  static constexpr bool kHalfZero = false;
  const double2* z;
  int nseq, logP;
  __device__ __forceinline__ double2 operator()(int f, unsigned i) const {
    return fft::mul(z[((size_t)f << logP) + i], z[((size_t)nseq << logP) + i]);
  }
};
struct StoreChirp {
  const double2* w;
  CosineOut o;
  int M;
  double scale;
  __device__ __forceinline__ void operator()(int f, unsigned i, double2 y) const {
    if (i > (unsigned)M) return;
    const double2 a = w[i];
    store_cos(o, f, (int)i, M, scale * fma(a.x, y.x, -a.y * y.y));
  }
};

int chirp_log(int M) { return fft::log2_at_least(2LL * M + 1); }

// One frequency costs M multiply-adds directly, one sequence two transforms of
// P >= 2M + 1 points: with seven launches against one, the chirp wins from
// about nseq M^2 = 1.6e7 (28 us of FP64 issue) on.
bool cosine_uses_chirp(int M, int nseq) { return (double)nseq * M * M > 1.6e7; }

// ---- Fourier route of the autocorrelation ----

__global__ void k_fft_table(int logN, double2* __restrict__ tab) {
  const long long m = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (m > (1ll << (logN - 3))) return;
  double s, c;
  sincospi(2.0 * (double)m / (double)(1ll << logN), &s, &c);
  tab[m] = make_double2(c, s);
}

// Spectrum of the channels' correlations, over the segments [b0, b1) of this
// CTA row: part[chunk][f], f = 0..N/2 (four times the sum of the header).
template <int KIND>
__global__ void __launch_bounds__(128) k_spec_power(const double2* __restrict__ z, int logN, int nb, int per_chunk,
                                                    double2* __restrict__ part) {
  constexpr int NP = n_packs<KIND>(), NX = KIND == TNEP_SPECTRUM_RAMAN_ISO ? 1 : 2 * NP;
  const unsigned N = 1u << logN, half = N >> 1;
  const unsigned f = blockIdx.x * blockDim.x + threadIdx.x;
  if (f > half) return;
  const unsigned g = (N - f) & (N - 1);
  const double sgn = (f & 1u) ? -1.0 : 1.0;
  // twice the channels' transforms of segment b (zero past the last one)
  auto load = [&](int b, double2* x) {
#pragma unroll
    for (int k = 0; k < NP; ++k) {
      double2 u = make_double2(0.0, 0.0), v = u;
      if (b < nb) {
        const size_t o = ((size_t)k * nb + b) << logN;
        u = z[o + f];
        v = z[o + g];
      }
      if constexpr (KIND == TNEP_SPECTRUM_RAMAN_ISO) {
        x[0] = make_double2(u.x + v.x, u.y - v.y);
      } else {
        x[2 * k] = make_double2(u.x + v.x, u.y - v.y);
        x[2 * k + 1] = make_double2(u.y + v.y, v.x - u.x);
      }
    }
  };
  const int b0 = blockIdx.y * per_chunk, b1 = min(nb, b0 + per_chunk);
  double2 x[NX], w[NX], nx[NX];
  load(b0, x);
  double2 acc = make_double2(0.0, 0.0);
  for (int b = b0; b < b1; ++b) {
    load(b + 1, nx);
#pragma unroll
    for (int c = 0; c < NX; ++c) w[c] = make_double2(fma(sgn, nx[c].x, x[c].x), fma(sgn, nx[c].y, x[c].y));
    auto dot2 = [&](double2 u, double2 v) {  // acc += conj(u) v
      acc.x = fma(u.x, v.x, fma(u.y, v.y, acc.x));
      acc.y = fma(u.x, v.y, fma(-u.y, v.x, acc.y));
    };
    auto dot = [&](int p, int q) { dot2(x[p], w[q]); };
    if constexpr (KIND == TNEP_SPECTRUM_RAMAN_ISO) {
      dot(0, 0);
    } else if constexpr (KIND == TNEP_SPECTRUM_IR) {
      dot(0, 0); dot(1, 1); dot(2, 2);  // channel 3 is empty
    } else {
      // channels 0, 4 (x0, x1), 8 = -(x0 + x1), and the transposed pairs
      dot(0, 0); dot(1, 1);
      dot2(fft::add(x[0], x[1]), fft::add(w[0], w[1]));
#pragma unroll
      for (int k = 1; k < 4; ++k) { dot(2 * k, 2 * k + 1); dot(2 * k + 1, 2 * k); }
    }
#pragma unroll
    for (int c = 0; c < NX; ++c) x[c] = nx[c];
  }
  part[(size_t)blockIdx.y * (half + 1) + f] = acc;
}

// Segment b of pack k (transform k nb + b): its L = N/2 samples, then zeros.
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
// The spectrum of a real sequence, its chunks summed in order.
struct LoadPower {
  static constexpr bool kHalfZero = false;
  const double2* part;
  int chunks, logN;
  __device__ __forceinline__ double2 operator()(int, unsigned i) const {
    const unsigned N = 1u << logN, half = N >> 1, f = i <= half ? i : N - i;
    double2 v = make_double2(0.0, 0.0);
    for (int c = 0; c < chunks; ++c) v = fft::add(v, part[(size_t)c * (half + 1) + f]);
    return make_double2(v.x, i <= half ? v.y : -v.y);
  }
};
struct StoreAcf {
  double* acf;
  int T, M;
  double scale;  // 1 / (4 N), times 1/3 for IR
  __device__ __forceinline__ void operator()(int, unsigned i, double2 v) const {
    if (i > (unsigned)M) return;
    acf[i] = v.x * scale / (double)(T - (int)i);
  }
};

struct FftPlan {
  int logN, nb, packs, chunks, per_chunk;
};
FftPlan spectrum_plan(int T, int kind, int M) {
  FftPlan p{};
  p.logN = fft::log2_at_least(2LL * M);
  p.nb = (int)(((long long)T + (1ll << (p.logN - 1)) - 1) >> (p.logN - 1));
  p.packs = kind == TNEP_SPECTRUM_IR ? 2 : (kind == TNEP_SPECTRUM_RAMAN_ISO ? 1 : 4);
  // enough (frequency, chunk) threads to fill the chip
  p.chunks = (int)std::min<long long>(p.nb, std::max<long long>(1, (1ll << 16) >> p.logN));
  p.per_chunk = (p.nb + p.chunks - 1) / p.chunks;
  p.chunks = (p.nb + p.per_chunk - 1) / p.per_chunk;
  return p;
}

template <int KIND>
cudaError_t spectrum_fft(const double* series, int T, int M, int subtract_mean, const FftPlan& p, const double* part,
                         int sum_blocks, double2* zx, double2* a, double2* b, double2* tab, double2* power, double* acf,
                         cudaStream_t st) {
  count_launches(2);
  cudaError_t e = launch_fft_table(p.logN, tab, st);
  if (e != cudaSuccess) return e;
  k_prep<KIND, true><<<(T + 255) / 256, 256, 0, st>>>(series, T, part, sum_blocks, subtract_mean,
                                                      reinterpret_cast<double*>(zx));
  double2* fin = fft::last_source(p.logN, p.packs * p.nb) == 0 ? b : a;
  e = fft::transform<false>(LoadSegment{zx, T, p.nb, p.logN}, fft::StorePlain{fin, p.logN}, a, b, tab,
                                        p.logN, p.packs * p.nb, st);
  if (e != cudaSuccess) return e;
  const unsigned half = 1u << (p.logN - 1);
  k_spec_power<KIND><<<dim3((half + 1 + 127) / 128, p.chunks), 128, 0, st>>>(fin, p.logN, p.nb, p.per_chunk, power);
  const double scale = 1.0 / (4.0 * (double)(1ll << p.logN)) / (KIND == TNEP_SPECTRUM_IR ? 3.0 : 1.0);
  return fft::transform<true>(LoadPower{power, p.chunks, p.logN}, StoreAcf{acf, T, M, scale}, a, b, tab, p.logN,
                              1, st);
}

// Bump allocator over a workspace (nullptr: sizes only).
struct Carve {
  char* base;
  size_t at = 0;
  template <class V>
  V* take(size_t n) {
    V* p = base ? reinterpret_cast<V*>(base + at) : nullptr;
    at += (n * sizeof(V) + 255) & ~size_t(255);
    return p;
  }
};

int sum_blocks_of(int T, int C) {
  const long long n = (long long)T * C;
  return (int)std::min<long long>(kMaxSumBlocks, (n + 4 * kSumThreads - 1) / (4 * kSumThreads));
}

}  // namespace

cudaError_t launch_fft_table(int logN, double2* tab, cudaStream_t st) {
  count_launches(1);
  k_fft_table<<<(unsigned)((fft::table_size(logN) + 255) / 256), 256, 0, st>>>(logN, tab);
  return cudaGetLastError();
}

// Direct sums cost channels T (M + 1) multiply-adds of FP64 issue (2e7: 35 us),
// the Fourier route about a dozen launches.  The transform's error is uniform
// over the lags while C(tau) divides by T - tau, so lags beyond T / 2 keep the
// direct sums until these cost milliseconds.
bool spectrum_uses_fft(int T, int kind, int M) {
  const double terms = (double)spectrum_channels(kind) * (double)T * (double)(M + 1);
  return terms > 1.0e9 || (terms > 2.0e7 && M <= T / 2);
}

size_t cosine_work_bytes(int M, int nseq) {
  if (!cosine_uses_chirp(M, nseq)) return sizeof(double) * (2 * (size_t)M + 32);
  const int logP = chirp_log(M);
  return sizeof(double2) * ((2 * (size_t)(nseq + 1) << logP) + (size_t)M + 1 + fft::table_size(logP)) + 1024;
}

cudaError_t launch_cosine(const double* lags, int M, int nseq, const CosineOut& o, const double* tab, void* work,
                          cudaStream_t st) {
  if (tab || !cosine_uses_chirp(M, nseq)) {
    if (!tab) {
      double* t = static_cast<double*>(work);
      count_launches(1);
      k_colsum<<<(2 * M + kSumThreads - 1) / kSumThreads, kSumThreads, 0, st>>>(nullptr, 0, 9, 0, nullptr, M, t);
      tab = t;
    }
    count_launches(1);
    k_cosine<<<dim3((M + 1 + 1) / 2, nseq), 64, 0, st>>>(lags, tab, M, o);
    return cudaGetLastError();
  }
  const int logP = chirp_log(M);
  Carve c{static_cast<char*>(work)};
  double2* a = c.take<double2>((size_t)(nseq + 1) << logP);
  double2* b = c.take<double2>((size_t)(nseq + 1) << logP);
  double2* w = c.take<double2>((size_t)M + 1);
  double2* tw = c.take<double2>(fft::table_size(logP));
  count_launches(1);
  k_chirp_tables<<<(unsigned)((M + 1 + fft::table_size(logP) + 255) / 256), 256, 0, st>>>(M, w, logP, tw);
  double2* fin = fft::last_source(logP, nseq + 1) == 0 ? b : a;
  double2* other = fin == a ? b : a;
  cudaError_t e = fft::transform<false>(LoadChirp{lags, w, M, nseq, logP}, fft::StorePlain{fin, logP}, a, b, tw, logP,
                                        nseq + 1, st);
  if (e != cudaSuccess) return e;
  return fft::transform<true>(LoadChirpProduct{fin, nseq, logP},
                              StoreChirp{w, o, M, 2.0 * o.dt / (double)(1ll << logP)}, other, fin, tw, logP, nseq, st);
}

size_t spectrum_work_bytes(int T, int C, int kind, int M, bool use_fft) {
  size_t n = sizeof(double) * ((size_t)kMaxSumBlocks * 9 + 2 * (size_t)M + (size_t)T * spectrum_channels(kind)) + 8192;
  if (use_fft) {
    const FftPlan p = spectrum_plan(T, kind, M);
    n = sizeof(double2) * ((size_t)p.packs * T + (2 * (size_t)p.packs * p.nb << p.logN) + fft::table_size(p.logN) +
                           (size_t)p.chunks * ((1u << (p.logN - 1)) + 1)) +
        sizeof(double) * ((size_t)kMaxSumBlocks * 9 + 2 * (size_t)M) +
        8192;
  }
  (void)C;
  return n + cosine_work_bytes(M, 1);
}

cudaError_t launch_spectrum(const double* series, int T, int C, double dt_fs, int kind, int M, int subtract_mean,
                            bool use_fft, bool use_chirp, void* work, double* freq, double* spec, double* acf,
                            cudaStream_t st) {
  Carve c{static_cast<char*>(work)};
  const int nsum = sum_blocks_of(T, C);
  double* part = c.take<double>((size_t)nsum * C);
  const bool chirp = use_chirp && cosine_uses_chirp(M, 1);
  double* tab = chirp ? nullptr : c.take<double>(2 * (size_t)M);
  const int tab_blocks = chirp ? 0 : (2 * M + kSumThreads - 1) / kSumThreads;
  count_launches(1);
  k_colsum<<<nsum + tab_blocks, kSumThreads, 0, st>>>(series, (long long)T * C, C, nsum, part, M, tab);
  cudaError_t e = cudaSuccess;
  if (use_fft) {
    const FftPlan p = spectrum_plan(T, kind, M);
    double2* zx = c.take<double2>((size_t)p.packs * T);
    double2* a = c.take<double2>((size_t)p.packs * p.nb << p.logN);
    double2* b = c.take<double2>((size_t)p.packs * p.nb << p.logN);
    double2* tw = c.take<double2>(fft::table_size(p.logN));
    double2* power = c.take<double2>((size_t)p.chunks * ((1u << (p.logN - 1)) + 1));
    if (kind == TNEP_SPECTRUM_IR)
      e = spectrum_fft<TNEP_SPECTRUM_IR>(series, T, M, subtract_mean, p, part, nsum, zx, a, b, tw, power, acf, st);
    else if (kind == TNEP_SPECTRUM_RAMAN_ISO)
      e = spectrum_fft<TNEP_SPECTRUM_RAMAN_ISO>(series, T, M, subtract_mean, p, part, nsum, zx, a, b, tw, power, acf,
                                                st);
    else
      e = spectrum_fft<TNEP_SPECTRUM_RAMAN_ANISO>(series, T, M, subtract_mean, p, part, nsum, zx, a, b, tw, power, acf,
                                                  st);
  } else {
    double* x = c.take<double>((size_t)T * spectrum_channels(kind));
    const unsigned grid = (unsigned)((T + 255) / 256);
    count_launches(2);
    if (kind == TNEP_SPECTRUM_IR)
      k_prep<TNEP_SPECTRUM_IR, false><<<grid, 256, 0, st>>>(series, T, part, nsum, subtract_mean, x);
    else if (kind == TNEP_SPECTRUM_RAMAN_ISO)
      k_prep<TNEP_SPECTRUM_RAMAN_ISO, false><<<grid, 256, 0, st>>>(series, T, part, nsum, subtract_mean, x);
    else
      k_prep<TNEP_SPECTRUM_RAMAN_ANISO, false><<<grid, 256, 0, st>>>(series, T, part, nsum, subtract_mean, x);
    k_acf<<<(unsigned)((32LL * (M + 1) + 63) / 64), 64, 0, st>>>(x, T, M, kind, acf);
    e = cudaGetLastError();
  }
  if (e != cudaSuccess) return e;
  return launch_cosine(acf, M, 1, CosineOut{0, kind, dt_fs, freq, spec}, tab, c.take<char>(0), st);
}

}  // namespace tnep

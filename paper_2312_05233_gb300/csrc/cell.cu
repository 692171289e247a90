// General periodic cells: triclinic, and cells shorter than twice the cutoff
// (Sec. II.A: U_i is a function of the pair vectors r_ij to every neighbour
// within the cutoff; in a small or skewed cell a neighbour may appear
// through several images).
//
// Each periodic structure is expanded into an open one: its atoms wrapped
// into the cell, followed by every image r_j + n H (n != 0) whose fractional
// coordinates lie within delta_a = rc_R / d_a of the cell (d_a the spacing of
// the lattice planes normal to axis a).  Any image within rc_R of an atom of
// the cell lies in that region, so the open structure holds every pair of the
// periodic one.  The ordinary batch path then runs on the expanded batch;
// the contributions of the image atoms ("ghosts") are zeroed before the
// per-structure reduction, so only the cell's own atoms are summed.
//
//   k_cell_count    one CTA per structure: H^-1, plane spacings, delta
//                   (float64), and where each atom's images start
//   k_cell_expand   one warp per atom: the wrapped atom and its images in a
//                   fixed order (atom, then n0, n1, n2)
//   k_zero_ghosts   per sorted atom of the expanded batch

#include <cuda_runtime.h>

#include <cmath>
#include <vector>

#include "engine.h"

namespace tnep {

namespace {

struct CellInfo {
  double H[9];
  double Hinv[9];
  double delta[3];
  int periodic;
};

constexpr int kExpandThreads = 256;

// H^-1, plane spacings and delta (float64) of structure s.
__device__ CellInfo plan_cell(int s, const float* __restrict__ cell, float rc, DevStatus* status) {
  CellInfo ci{};
  bool any = false;
  for (int k = 0; k < 9; ++k) {
    ci.H[k] = (double)cell[9 * s + k];
    any |= cell[9 * s + k] != 0.0f;
  }
  ci.periodic = any ? 1 : 0;
  if (any) {
    const double* H = ci.H;
    // rows a = H[0..2], b = H[3..5], c = H[6..8]; Hinv columns from cross products
    const double bc[3] = {H[4] * H[8] - H[5] * H[7], H[5] * H[6] - H[3] * H[8], H[3] * H[7] - H[4] * H[6]};
    const double ca[3] = {H[7] * H[2] - H[8] * H[1], H[8] * H[0] - H[6] * H[2], H[6] * H[1] - H[7] * H[0]};
    const double ab[3] = {H[1] * H[5] - H[2] * H[4], H[2] * H[3] - H[0] * H[5], H[0] * H[4] - H[1] * H[3]};
    const double det = H[0] * bc[0] + H[1] * bc[1] + H[2] * bc[2];
    if (!(fabs(det) > 1e-9)) {
      atomicCAS(&status->error, 0, (int)TNEP_ERR_INVALID);
      atomicCAS(&status->bad_struct, 0, s);
      ci.periodic = 0;
    } else {
      // s = r Hinv with Hinv[:, a] = (row cross product) / det
      for (int k = 0; k < 3; ++k) {
        ci.Hinv[3 * k + 0] = bc[k] / det;
        ci.Hinv[3 * k + 1] = ca[k] / det;
        ci.Hinv[3 * k + 2] = ab[k] / det;
      }
      const double vol = fabs(det);
      const double nrm[3] = {sqrt(bc[0] * bc[0] + bc[1] * bc[1] + bc[2] * bc[2]),
                             sqrt(ca[0] * ca[0] + ca[1] * ca[1] + ca[2] * ca[2]),
                             sqrt(ab[0] * ab[0] + ab[1] * ab[1] + ab[2] * ab[2])};
      for (int a = 0; a < 3; ++a) ci.delta[a] = (double)rc / (vol / nrm[a]) + 1e-6;
    }
  }
  return ci;
}

__device__ __forceinline__ void frac_of(const CellInfo& ci, const float* p, double* sf) {
  for (int a = 0; a < 3; ++a) {
    const double v = fma((double)p[2], ci.Hinv[6 + a],
                         fma((double)p[0], ci.Hinv[a], __dmul_rn((double)p[1], ci.Hinv[3 + a])));
    sf[a] = v - floor(v);
  }
}

// Image range of one fractional coordinate: n with s + n in [-delta, 1 + delta).
__device__ __forceinline__ void image_range(double s, double delta, int& lo, int& hi) {
  lo = (int)ceil(-delta - s);
  hi = (int)ceil(1.0 + delta - s) - 1;
}

// Images of an atom, itself left out, and no more than the host refuses (a
// minute cell may have beyond 2^31); none where a coordinate is not finite.
__device__ __forceinline__ int image_count(const double* sf, const double* delta) {
  if (!isfinite(sf[0]) || !isfinite(sf[1]) || !isfinite(sf[2])) return 0;
  long long all = 1;
  for (int a = 0; a < 3; ++a) {
    int lo, hi;
    image_range(sf[a], delta[a], lo, hi);
    all = min(all * max((long long)hi - lo + 1, 0ll), (long long)kMaxBatchAtoms + 1);
  }
  return (int)max(all - 1, 0ll);
}

// One CTA per structure: its plan, and per atom the first of its images among
// the structure's (exclusive scan of the image counts in atom order);
// n_ghost[s] is their sum.
__global__ void __launch_bounds__(kExpandThreads) k_cell_count(const int* __restrict__ off,
                                                               const float* __restrict__ pos,
                                                               const float* __restrict__ cell, float rc,
                                                               CellInfo* __restrict__ info, int* __restrict__ first,
                                                               int* __restrict__ atom_struct,
                                                               int* __restrict__ n_ghost, DevStatus* status) {
  __shared__ long long warp_sums[kExpandThreads / 32];
  __shared__ CellInfo ci_sh;
  const int s = blockIdx.x, lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const int a0 = off[s], a1 = off[s + 1], n = a1 - a0;
  if (threadIdx.x == 0) {
    ci_sh = plan_cell(s, cell, rc, status);
    info[s] = ci_sh;
  }
  __syncthreads();
  const CellInfo ci = ci_sh;
  long long carry = 0;
  for (int c0 = 0; c0 < n; c0 += kExpandThreads) {
    const int k = c0 + threadIdx.x;
    int cnt = 0;
    if (k < n && ci.periodic) {
      double sf[3];
      frac_of(ci, pos + 3 * (size_t)(a0 + k), sf);
      cnt = image_count(sf, ci.delta);
    }
    long long incl = cnt;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const long long v = __shfl_up_sync(0xffffffffu, incl, o);
      if (lane >= o) incl += v;
    }
    if (lane == 31) warp_sums[w] = incl;
    __syncthreads();
    long long before = carry;
    for (int u = 0; u < kExpandThreads / 32; ++u) {
      if (u < w) before += warp_sums[u];
      carry += warp_sums[u];
    }
    if (k < n) {
      first[a0 + k] = (int)(before + incl - cnt);  // (not read where the batch is refused)
      atom_struct[a0 + k] = s;
    }
    __syncthreads();
  }
  if (threadIdx.x == 0) n_ghost[s] = (int)min(carry, (long long)kMaxBatchAtoms);
}

// One warp per atom: the wrapped atom at its own place (the structure's atoms
// come first, active[] holds these places) and its images, lane by lane, in the
// order of n0, n1, n2.  (One CTA per structure with a serial loop over the
// images of each atom took 48 us for 24 small cells.)
__global__ void __launch_bounds__(128) k_cell_expand(int N, const int* __restrict__ off, const float* __restrict__ pos,
                                                     const int* __restrict__ types, const CellInfo* __restrict__ info,
                                                     const int* __restrict__ first,
                                                     const int* __restrict__ atom_struct,
                                                     const int* __restrict__ new_off, float* __restrict__ out_pos,
                                                     int* __restrict__ out_types, unsigned char* __restrict__ ghost,
                                                     int* __restrict__ active) {
  const int a = (int)(((long long)blockIdx.x * blockDim.x + threadIdx.x) >> 5), lane = threadIdx.x & 31;
  if (a >= N) return;
  const int s = atom_struct[a], a0 = off[s], n = off[s + 1] - a0, o0 = new_off[s];
  const CellInfo& ci = info[s];
  const int t = types[a], self = o0 + (a - a0);
  const float* p = pos + 3 * (size_t)a;
  if (lane == 0) {
    out_types[self] = t;
    ghost[self] = 0;
    active[a] = self;
  }
  if (!ci.periodic) {
    if (lane < 3) out_pos[3 * (size_t)self + lane] = p[lane];
    return;
  }
  double sf[3];
  frac_of(ci, p, sf);
  if (lane == 0) {
    float* q = out_pos + 3 * (size_t)self;
    for (int c = 0; c < 3; ++c) q[c] = (float)(sf[0] * ci.H[c] + sf[1] * ci.H[3 + c] + sf[2] * ci.H[6 + c]);
  }
  int lo[3], hi[3];
  for (int d = 0; d < 3; ++d) image_range(sf[d], ci.delta[d], lo[d], hi[d]);
  const int w1 = hi[1] - lo[1] + 1, w2 = hi[2] - lo[2] + 1, count = image_count(sf, ci.delta);
  const int zero = (-lo[0] * w1 - lo[1]) * w2 - lo[2];  // the atom itself
  const int g0 = o0 + n + first[a];
  for (int e = lane; e < count; e += 32) {
    const int x = e < zero ? e : e + 1;
    const int n0 = lo[0] + x / (w1 * w2), n1 = lo[1] + x / w2 % w1, n2 = lo[2] + x % w2;
    const double f0 = sf[0] + n0, f1 = sf[1] + n1, f2 = sf[2] + n2;
    const int g = g0 + e;
    float* q = out_pos + 3 * (size_t)g;
    // The exact position, a sum of float32 values, often lies half-way between
    // two floats, so its rounding hangs on the last bit here.  The order and
    // contraction are fixed to those the images have always had, which depend
    // on where n2 lies in its range.
    const int i2 = x % w2;
    const bool two = i2 < (w2 & 3) && i2 < 2;
    for (int c = 0; c < 3; ++c) {
      const double ab = fma(f1, ci.H[3 + c], __dmul_rn(f0, ci.H[c]));
      q[c] = (float)(two ? __dadd_rn(__dmul_rn(f2, ci.H[6 + c]), ab) : fma(f2, ci.H[6 + c], ab));
    }
    out_types[g] = t;
    ghost[g] = 1;
  }
}

__global__ void k_zero_ghosts(int N, const int* __restrict__ sorted_orig, const unsigned char* __restrict__ ghost,
                              float* __restrict__ per_atom, int atom_stride, int C) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= N || !ghost[sorted_orig[i]]) return;
  for (int c = 0; c < C; ++c) per_atom[(size_t)c * atom_stride + i] = 0.f;
}

}  // namespace

cudaError_t launch_zero_ghosts(int N, const int* sorted_orig, const unsigned char* ghost, float* per_atom,
                               int atom_stride, int C, cudaStream_t st) {
  if (N <= 0) return cudaSuccess;
  count_launches(1);
  k_zero_ghosts<<<(N + 255) / 256, 256, 0, st>>>(N, sorted_orig, ghost, per_atom, atom_stride, C);
  return cudaGetLastError();
}

}  // namespace tnep

using namespace tnep;

extern "C" {

tnep_status tnep_eval_batch_cell(tnep_ctx* c, int n_structs, const int* atom_offsets, const float* pos,
                                 const float* cell, const int* types, double* out, void* stream) {
  if (!c) return fail(TNEP_ERR_INVALID, "ctx is NULL");
  if (n_structs < 0) return fail(TNEP_ERR_INVALID, "negative size");
  if (n_structs == 0) return TNEP_OK;
  if (!atom_offsets || !out) return fail(TNEP_ERR_INVALID, "NULL buffer");
  if (is_device_ptr(atom_offsets)) return fail(TNEP_ERR_INVALID, "atom_offsets must be host memory");
  if (atom_offsets[0] != 0) return fail(TNEP_ERR_INVALID, "atom_offsets[0] must be 0");
  for (int s = 0; s < n_structs; ++s)
    if (atom_offsets[s + 1] < atom_offsets[s]) return fail(TNEP_ERR_INVALID, "atom_offsets must not decrease");
  const int N = atom_offsets[n_structs];
  if (N >= kMaxBatchAtoms) return fail(TNEP_ERR_INVALID, "a batch must hold fewer than 2^29 atoms");
  if (N > 0 && (!pos || !types)) return fail(TNEP_ERR_INVALID, "NULL buffer");
  TNEP_CUDA(cudaSetDevice(c->device));
  cudaStream_t st = pick_stream(c, stream);
  if (!is_device_ptr(types))
    for (int a = 0; a < N; ++a)
      if (types[a] < 0 || types[a] >= c->n_types) return fail(TNEP_ERR_INVALID, "type index out of range");
  Workspace& w = c->ws;
  // scratch of the call from the library's pool: the inputs, then the expanded batch
  char *in = nullptr, *ex = nullptr;
  auto body = [&]() -> tnep_status {
    size_t at = 0;
    auto place = [&](size_t bytes) {
      const size_t o = at;
      at += (bytes + 255) & ~size_t(255);
      return o;
    };
    const size_t n1 = std::max(N, 1);
    const size_t o_pos = place(sizeof(float) * 3 * n1), o_types = place(sizeof(int) * n1);
    const size_t o_cell = place(sizeof(float) * 9 * n_structs), o_off = place(sizeof(int) * (n_structs + 1));
    const size_t o_ng = place(sizeof(int) * n_structs), o_info = place(sizeof(CellInfo) * n_structs);
    const size_t o_first = place(sizeof(int) * n1), o_as = place(sizeof(int) * n1);
    TNEP_CUDA(dev_malloc_async((void**)&in, at, st));
    float *d_pos = reinterpret_cast<float*>(in + o_pos), *d_cell = reinterpret_cast<float*>(in + o_cell);
    int *d_types = reinterpret_cast<int*>(in + o_types), *d_off = reinterpret_cast<int*>(in + o_off);
    int *d_ng = reinterpret_cast<int*>(in + o_ng), *d_first = reinterpret_cast<int*>(in + o_first);
    int* d_as = reinterpret_cast<int*>(in + o_as);
    CellInfo* d_info = reinterpret_cast<CellInfo*>(in + o_info);
    if (N > 0) {
      TNEP_CUDA(cudaMemcpyAsync(d_pos, pos, sizeof(float) * 3 * N, cudaMemcpyDefault, st));
      TNEP_CUDA(cudaMemcpyAsync(d_types, types, sizeof(int) * N, cudaMemcpyDefault, st));
    }
    if (cell)
      TNEP_CUDA(cudaMemcpyAsync(d_cell, cell, sizeof(float) * 9 * n_structs, cudaMemcpyDefault, st));
    else
      TNEP_CUDA(cudaMemsetAsync(d_cell, 0, sizeof(float) * 9 * n_structs, st));
    TNEP_CUDA(cudaMemcpyAsync(d_off, atom_offsets, sizeof(int) * (n_structs + 1), cudaMemcpyHostToDevice, st));
    TNEP_TRY(reset_status(w, st));
    k_cell_count<<<n_structs, kExpandThreads, 0, st>>>(d_off, d_pos, d_cell, c->rc_R, d_info, d_first, d_as, d_ng,
                                                       w.d_status);
    count_launches(1);
    TNEP_CUDA(cudaGetLastError());
    std::vector<int> ng(n_structs);
    TNEP_CUDA(cudaMemcpyAsync(ng.data(), d_ng, sizeof(int) * n_structs, cudaMemcpyDeviceToHost, st));
    bool regrow = false;
    TNEP_TRY(finish(c, w, st, &regrow));  // synchronises; reports a degenerate cell
    std::vector<int> eoff(n_structs + 1, 0);
    long long tot = 0;
    for (int s = 0; s < n_structs; ++s) {
      tot += (long long)(atom_offsets[s + 1] - atom_offsets[s]) + ng[s];
      if (tot >= kMaxBatchAtoms) return fail(TNEP_ERR_INVALID, "expanded batch (cell atoms + images) exceeds 2^29 atoms");
      eoff[s + 1] = (int)tot;
    }
    const int Ne = (int)tot;
    at = 0;
    const size_t e1 = std::max(Ne, 1);
    const size_t o_new = place(sizeof(int) * (n_structs + 1)), o_epos = place(sizeof(float) * 3 * e1);
    const size_t o_et = place(sizeof(int) * e1), o_gh = place(e1), o_box = place(sizeof(float) * 3 * n_structs);
    const size_t o_act = place(sizeof(int) * n1);
    TNEP_CUDA(dev_malloc_async((void**)&ex, at, st));
    int *d_new = reinterpret_cast<int*>(ex + o_new), *d_etypes = reinterpret_cast<int*>(ex + o_et);
    int* d_active = reinterpret_cast<int*>(ex + o_act);
    float *d_epos = reinterpret_cast<float*>(ex + o_epos), *d_ebox = reinterpret_cast<float*>(ex + o_box);
    unsigned char* d_ghost = reinterpret_cast<unsigned char*>(ex + o_gh);
    TNEP_CUDA(cudaMemsetAsync(d_ebox, 0, sizeof(float) * 3 * n_structs, st));
    TNEP_CUDA(cudaMemcpyAsync(d_new, eoff.data(), sizeof(int) * (n_structs + 1), cudaMemcpyHostToDevice, st));
    if (N > 0) {
      k_cell_expand<<<(unsigned)((32LL * N + 127) / 128), 128, 0, st>>>(N, d_off, d_pos, d_types, d_info, d_first, d_as,
                                                                        d_new, d_epos, d_etypes, d_ghost, d_active);
      count_launches(1);
      TNEP_CUDA(cudaGetLastError());
    }
    const Images images{d_ghost, d_active, N};
    const int Ctot = total_C(c);
    for (int attempt = 0; attempt < 4; ++attempt) {
      TNEP_TRY(reset_status(w, st));
      TNEP_TRY(build_lists(c, w, st, n_structs, eoff.data(), d_epos, d_ebox, d_etypes, std::max(Ne, 1), nullptr, N));
      TNEP_TRY(run_models(c, w, st, n_structs, Ne, nullptr, &images));
      regrow = false;
      TNEP_TRY(finish(c, w, st, &regrow));
      if (regrow) continue;
      TNEP_TRY(copy_out(out, w.out.p, (size_t)n_structs * Ctot, st));
      TNEP_CUDA(cudaStreamSynchronize(st));
      return TNEP_OK;
    }
    return fail(TNEP_ERR_NEIGHBOR_OVERFLOW, "neighbour lists kept overflowing");
  };
  const tnep_status rc = body();
  if (ex) cudaFreeAsync(ex, st);
  if (in) cudaFreeAsync(in, st);
  cudaStreamSynchronize(st);
  return rc;
}

}  // extern "C"

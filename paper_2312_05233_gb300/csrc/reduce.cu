// Per-structure reductions and population scoring after the fused kernel:
// the deterministic FP64 sums of the per-atom contributions of Eqs. 3-4
// into one tensor per structure, the per-atom export in input order, and the
// RMSE of each individual's predictions against the target tensors (the
// loss of Sec. II.D before regularization).

#include "tnep_internal.cuh"

namespace tnep {

namespace {

// Per-structure FP64 sums in two deterministic stages: CTA (s, chunk) sums a
// fixed 2048-atom chunk of structure s (strided per-thread sums, a shuffle
// tree in each warp, then the eight warp sums in order), then one warp per
// structure adds its chunk partials (strided per-lane sums, shuffle tree).
// Chunks are aligned to the structure start, so a structure's result does
// not depend on what else is in the batch.  A structure of one chunk is
// written by the first stage (the second would add it to zeros).
//
// Bound by FP64 issue (two lanes per clock and SM, so a warp's addition takes
// 16 cycles): the warp tree folds two components into one addition, the lower
// half-warp adding one and the upper half the other, which needs 12 additions
// for nine components instead of 45.
struct ReduceArgs {
  ReduceModel m[4];
  int split;              // blockIdx.z: model, or (split) 3 * model + group of three components
  const int* offsets;
  int S, n_chunks;
  size_t pa_pop_stride, out_pop_stride;  // individuals (blockIdx.y)
  int atom_stride;
  double* partial;        // [model][individual][structure][chunk][9]
};

// Sums v[c] over the warp for C components; component c's total arrives in
// lane lane_of(c).  The additions are those of a shuffle tree per component
// (offsets 16, 8, 4, 2, 1), so the totals are too.
__device__ __forceinline__ int lane_of(int c) {
  return ((c & 1) << 4) | ((c & 2) << 2) | (c & 4) | ((c & 8) >> 2);
}
// float32 -> float64 with integer instructions (exact; the conversion
// instruction shares the FP64 pipe).  Subnormals, infinities and NaN take it.
__device__ __forceinline__ double widen(float x) {
  const unsigned u = __float_as_uint(x), mag = u & 0x7fffffffu;
  if (mag - 0x00800000u < 0x7f000000u)  // normal
    return __hiloint2double((int)((u & 0x80000000u) | ((mag >> 3) + (896u << 20))), (int)(u << 29));
  return mag == 0u ? __hiloint2double((int)u, 0) : (double)x;
}

template <int C>
__device__ __forceinline__ double warp_tree(const double* v, int lane) {
  double t[C];
#pragma unroll
  for (int c = 0; c < C; ++c) t[c] = v[c];
  int n = C;
#pragma unroll
  for (int o = 16; o > 1; o >>= 1) {
    const bool up = lane & o;
#pragma unroll
    for (int k = 0; k < (C + 1) / 2; ++k) {
      if (2 * k < n) {
        const double a = t[2 * k], b = 2 * k + 1 < n ? t[2 * k + 1] : 0.0;
        const double keep = up ? b : a, give = up ? a : b;
        t[k] = keep + __shfl_xor_sync(0xffffffffu, give, o);
      }
    }
    n = (n + 1) / 2;
  }
  return t[0] + __shfl_xor_sync(0xffffffffu, t[0], 1);
}

// Components [c0, c0 + NC) of model `mi`, which has C.
template <int NC>
__device__ __forceinline__ void reduce_chunk(const ReduceArgs& a, const ReduceModel& m, int mi, int C, int c0) {
  const int s = blockIdx.x / a.n_chunks, chunk = blockIdx.x % a.n_chunks, p = blockIdx.y;
  const int a0 = a.offsets[s] + chunk * kReduceChunk;
  const int a1 = min(a.offsets[s + 1], a0 + kReduceChunk);
  const float* pa = m.per_atom + (size_t)p * a.pa_pop_stride + (size_t)c0 * a.atom_stride;
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  __shared__ double red[9][8];
  // warps past the chunk's end hold zeros
  const bool any = a0 + 32 * w < a1;
  double v = 0.0;
  if (any) {
    double acc[NC];
#pragma unroll
    for (int c = 0; c < NC; ++c) acc[c] = 0.0;
    int g = a0 + threadIdx.x;
    if (g < a1) {  // the first addition would be to zero
#pragma unroll
      for (int c = 0; c < NC; ++c) acc[c] = widen(pa[(size_t)c * a.atom_stride + g]);
      for (g += blockDim.x; g < a1; g += blockDim.x) {
#pragma unroll
        for (int c = 0; c < NC; ++c) acc[c] += widen(pa[(size_t)c * a.atom_stride + g]);
      }
    }
    v = warp_tree<NC>(acc, lane);
  }
#pragma unroll
  for (int c = 0; c < NC; ++c)
    if (lane == lane_of(c)) red[c][w] = v;
  __syncthreads();
  if (threadIdx.x < NC) {
    double t = 0.0;
#pragma unroll
    for (int k = 0; k < 8; ++k) t += red[threadIdx.x][k];
    if (a.n_chunks == 1)
      m.out[(size_t)p * a.out_pop_stride + (size_t)s * C + c0 + threadIdx.x] = t;
    else
      a.partial[((((size_t)mi * gridDim.y + p) * a.S + s) * a.n_chunks + chunk) * 9 + c0 + threadIdx.x] = t;
  }
}

__global__ void __launch_bounds__(256) k_reduce_partial(const __grid_constant__ ReduceArgs a) {
  const int mi = a.split ? blockIdx.z / 3 : blockIdx.z, c0 = a.split ? 3 * (blockIdx.z % 3) : 0;
  const ReduceModel m = a.m[mi];
  if (c0 >= m.C) return;
  if (a.split || m.C == 3) reduce_chunk<3>(a, m, mi, m.C, c0);
  else reduce_chunk<9>(a, m, mi, 9, 0);
}

// One warp per (model, individual, structure).
__global__ void k_reduce_final(const __grid_constant__ ReduceArgs a, int n_pop) {
  const int wid = (int)(((long long)blockIdx.x * blockDim.x + threadIdx.x) >> 5), lane = threadIdx.x & 31;
  if (wid >= a.S * n_pop) return;  // whole warps
  const int p = wid / a.S, s = wid % a.S;
  const ReduceModel m = a.m[blockIdx.z];
  const double* src = a.partial + (((size_t)blockIdx.z * n_pop + p) * a.S + s) * a.n_chunks * 9;
  double v[9];
#pragma unroll
  for (int c = 0; c < 9; ++c) v[c] = 0.0;
  for (int k = lane; k < a.n_chunks; k += 32) {
#pragma unroll
    for (int c = 0; c < 9; ++c)
      if (c < m.C) v[c] += src[(size_t)k * 9 + c];
  }
  const double t = m.C == 3 ? warp_tree<3>(v, lane) : warp_tree<9>(v, lane);
  for (int c = 0; c < m.C; ++c)
    if (lane == lane_of(c)) m.out[(size_t)p * a.out_pop_stride + (size_t)s * m.C + c] = t;
}

cudaError_t launch_reduce_args(ReduceArgs& a, int n_models, int n_pop, cudaStream_t st) {
  count_launches(a.n_chunks == 1 ? 1 : 2);
  // few CTAs: three components each (20 structures of 8,640 atoms, rank 2: 21 us
  // with 100 CTAs of nine); many: all nine, whose folded tree costs less
  a.split = (long long)a.S * a.n_chunks * n_pop * n_models <= 608;
  k_reduce_partial<<<dim3(a.S * a.n_chunks, n_pop, n_models * (a.split ? 3 : 1)), 256, 0, st>>>(a);
  if (a.n_chunks > 1) {
    const long long nt = 32LL * a.S * n_pop;
    k_reduce_final<<<dim3((unsigned)((nt + 127) / 128), 1, n_models), 128, 0, st>>>(a, n_pop);
  }
  return cudaGetLastError();
}

__global__ void k_gather(int n, const int* orig_sorted, const float* pa, int atom_stride, int C, float* out) {
  const int g = blockIdx.x * blockDim.x + threadIdx.x;
  if (g >= n) return;
  const int i = orig_sorted[g];
  for (int c = 0; c < C; ++c) out[(size_t)g * C + c] = pa[(size_t)c * atom_stride + i];
}

__global__ void k_rmse(int S, int C, const double* pred, const double* target, double* rmse) {
  const int p = blockIdx.x;
  const double* pp = pred + (size_t)p * S * C;
  double acc = 0.0;
  for (int k = threadIdx.x; k < S * C; k += blockDim.x) {
    const double d = pp[k] - target[k];
    acc += d * d;
  }
  __shared__ double red[256];
  red[threadIdx.x] = acc;
  __syncthreads();
  for (int w = 128; w > 0; w >>= 1) {
    if (threadIdx.x < w) red[threadIdx.x] += red[threadIdx.x + w];
    __syncthreads();
  }
  if (threadIdx.x == 0) rmse[p] = S * C > 0 ? sqrt(red[0] / (double)(S * C)) : 0.0;
}

}  // namespace

cudaError_t launch_reduce(int n_structs, int n_pop, const int* offsets, int max_atoms, const float* per_atom,
                          size_t per_atom_stride, int atom_stride, int C, double* partial, double* out,
                          size_t out_pop_stride, cudaStream_t st) {
  if (n_structs <= 0 || n_pop <= 0) return cudaSuccess;
  ReduceArgs a{};
  a.m[0] = {per_atom, out, C};
  a.offsets = offsets;
  a.S = n_structs;
  a.n_chunks = reduce_chunks(max_atoms);
  a.pa_pop_stride = per_atom_stride;
  a.out_pop_stride = out_pop_stride;
  a.atom_stride = atom_stride;
  a.partial = partial;
  return launch_reduce_args(a, 1, n_pop, st);
}

cudaError_t launch_reduce_models(int n_structs, int n_models, const ReduceModel* models, const int* offsets,
                                 int max_atoms, int atom_stride, double* partial, cudaStream_t st) {
  if (n_structs <= 0) return cudaSuccess;
  ReduceArgs a{};
  a.offsets = offsets;
  a.S = n_structs;
  a.n_chunks = reduce_chunks(max_atoms);
  a.atom_stride = atom_stride;
  constexpr int kGroup = (int)(sizeof(a.m) / sizeof(a.m[0]));
  for (int k0 = 0; k0 < n_models; k0 += kGroup) {
    const int n = n_models - k0 < kGroup ? n_models - k0 : kGroup;
    for (int k = 0; k < n; ++k) a.m[k] = models[k0 + k];
    a.partial = partial + (size_t)k0 * n_structs * a.n_chunks * 9;
    const cudaError_t e = launch_reduce_args(a, n, 1, st);
    if (e != cudaSuccess) return e;
  }
  return cudaSuccess;
}

cudaError_t launch_gather_per_atom(int n_atoms, const int* orig_sorted, const float* per_atom,
                                   int atom_stride, int C, float* out, cudaStream_t st) {
  if (n_atoms <= 0) return cudaSuccess;
  count_launches(1);
  k_gather<<<(n_atoms + 255) / 256, 256, 0, st>>>(n_atoms, orig_sorted, per_atom, atom_stride, C, out);
  return cudaGetLastError();
}

cudaError_t launch_rmse(int n_pop, int n_structs, int C, const double* pred, const double* target,
                        double* rmse, cudaStream_t st) {
  if (n_pop <= 0) return cudaSuccess;
  count_launches(1);
  k_rmse<<<n_pop, 256, 0, st>>>(n_structs, C, pred, target, rmse);
  return cudaGetLastError();
}

}  // namespace tnep

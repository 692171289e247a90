// The whole per-atom path with one warp per atom, for batches too small to
// fill the chip with one thread per atom.
//
// With one thread per atom (nbr.cu, radial.cu, tnep_fused.cu) a small batch is
// four serial walks over each atom's neighbours on a few warps: 30-42 us each
// whatever the number of atoms, up to one CTA per SM.  Here the warp's 32 lanes take
// 32 candidates or 32 pairs at a time: each lane computes its pair's distance,
// basis and harmonics, leaves them in shared memory, and the lanes then own
// the sums (basis index and component of the radial moments, (l, m) of the
// angular sums) and add the pairs in list order.  Neighbour lists, moments and
// angular sums never leave shared memory, one launch replaces 2 + models, and
// the pair geometry and basis are shared by the models.
//
// Every sum has the order and the roundings of the thread-per-atom kernels
// (their multiply-adds are explicit or contract the same way), so the results
// are the same bits; the tests compare the routes exactly.
//
// Bound by latency for a few hundred atoms (one frame of 64 water molecules, two
// models: the kernel 34 us, the call 284 -> 113 us) and by issue slots beyond: 6,660
// warp instructions per atom in boxes of 192 atoms (lists 1,330, radial 1,480, per
// model 1,930; 7,390 in one box of 10,137 atoms), against about 625 for a thread per
// atom with all lanes busy, so it is taken up to kWideAtoms (the rule is there).
//
// FUSED = false writes the angular lists and the radial moments in the layouts
// of the general path instead (tensor-core network: its products need 128 atoms
// per CTA, so those models run in k_fused).

#include <algorithm>

#include "nbr_device.cuh"
#include "tnep_device.cuh"
#include "tnep_internal.cuh"

namespace tnep {

namespace {

constexpr int kWarps = 4;           // warps (atoms) per CTA
// Floats per row of the pair tile (32 pairs and padding: 9 float4, odd, so that
// float4 loads of eight rows hit different banks); a row holds one quantity of
// all pairs, which the owner of a sum reads four pairs at a time.  Rows of the
// radial part: df 0-8, T 9-17, fc 18, rv 19-21, rr 22-27; of the angular part:
// the harmonics from 0, then from kTileG the g_n (forward) or r_ij, r^2 and the
// partial force (backward).
constexpr int kRow = 36;
constexpr int kTileG = 24;

// Floats of one warp's shared memory after the lists.
__host__ __device__ constexpr int wide_floats(int n_types) {
  return 32 * kRow + n_types * 90 + n_types * 9 + 120 + 120 + 32 + 32 + 64 + 64 + 64 + 32;
}
__host__ __device__ inline int wide_words(int n_types, int cap_R, int cap_A) {
  return (cap_R * (n_types > 2 ? 2 : 1) + cap_A + 3) / 4 * 4 + (wide_floats(n_types) + 3) / 4 * 4;
}

// One lane's candidate against atom i (the float32 pair rule of tnep.h; a zero
// shift subtracts exactly nothing).
__device__ __forceinline__ float pair_r2(float4 pj, float4 pi, float sx, float sy, float sz, bool rint_pairs,
                                         const StructGrid& G) {
  float dx, dy, dz;
  if (!rint_pairs) {
    dx = __fsub_rn(__fsub_rn(pj.x, pi.x), sx);
    dy = __fsub_rn(__fsub_rn(pj.y, pi.y), sy);
    dz = __fsub_rn(__fsub_rn(pj.z, pi.z), sz);
  } else {
    dx = mi_diff(pj.x, pi.x, G.L[0], G.invL[0]);
    dy = mi_diff(pj.y, pi.y, G.L[1], G.invL[1]);
    dz = mi_diff(pj.z, pi.z, G.L[2], G.invL[2]);
  }
  return __fadd_rn(__fadd_rn(__fmul_rn(dx, dx), __fmul_rn(dy, dy)), __fmul_rn(dz, dz));
}

// Keeps the compiler from sharing subexpressions of the harmonics between the
// two walks (and models): which products contract into multiply-adds then
// follows from each walk alone, as in k_fused.
__device__ __forceinline__ void opaque(float& x, float& y, float& z) {
  asm volatile("" : "+f"(x), "+f"(y), "+f"(z));
}

// One lane's pair of the angular walk.
template <int BA>
struct Pair {
  float dx, dy, dz, rinv;
  int t;
  float f[BA], df[BA];
  __device__ __forceinline__ void load(const float4* pos4, int j, float4 pi, const StructBox& bx, float rcinv) {
    const float4 pj = pos4[j];
    t = __float_as_int(pj.w);
    dx = min_image(pj.x, pi.x, bx.L[0], bx.invL[0]);
    dy = min_image(pj.y, pi.y, bx.L[1], bx.invL[1]);
    dz = min_image(pj.z, pi.z, bx.L[2], bx.invL[2]);
    const float r2 = dx * dx + dy * dy + dz * dz;
    rinv = rsqrtf(r2);
    const float r = r2 * rinv;
    basis_fwd_bwd<BA>(r, rcinv, f, df);
  }
  template <int NA>
  __device__ __forceinline__ void radial_functions(const float* cA_i, int stride, float* g, float* dg) const {
    constexpr int NBA4 = ((NA * BA + 3) / 4) * 4;
    float cc[NBA4];
    load_coeffs<NA, BA>(cA_i + t * stride, cc);
#pragma unroll
    for (int n = 0; n < NA; ++n) {
      float s0 = 0.f, s1 = 0.f;
#pragma unroll
      for (int k = 0; k < BA; ++k) { s0 += cc[n * BA + k] * f[k]; s1 += cc[n * BA + k] * df[k]; }
      g[n] = s0; dg[n] = s1;
    }
  }
};

template <int NR, int NA, int BR, int BA, int LMAX, bool FUSED>
__global__ void __launch_bounds__(32 * kWarps) k_wide(const __grid_constant__ WideArgs a) {
  constexpr int NLM = LMAX * (LMAX + 2);
  constexpr int D = NR + NA * LMAX + NA;
  constexpr int DP = (D + 3) & ~3;
  constexpr int B = kMomBasis;
  static_assert(NLM <= kTileG && NA <= 5 && DP <= 32, "tile rows and lane maps");
  extern __shared__ float4 sm4[];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const NbrArgs& na = a.nbr;
  const int T = na.n_types;
  const int item = blockIdx.x * kWarps + warp;
  if (item >= a.n_active) return;  // whole warps; there is no CTA-wide barrier below
  const int i = a.active ? na.orig_sorted[a.active[item]] : item;
  int* lists = reinterpret_cast<int*>(sm4) + (size_t)warp * wide_words(T, na.cap_R, na.cap_A);
  int* sR = lists;                                        // radial list, grouped by type
  int* sTmp = sR + na.cap_R;                              // append order, tagged with the type (more than two types)
  int* sA = sTmp + (T > 2 ? na.cap_R : 0);
  float* tile = reinterpret_cast<float*>(lists + (na.cap_R * (T > 2 ? 2 : 1) + na.cap_A + 3) / 4 * 4);
  float* sAs = tile + 32 * kRow;                          // A [NA][24]
  float* sG = sAs + 120;                                  // G [NA][24]
  float* sq = sG + 120;                                   // q, then scaled
  float* se = sq + 32;                                    // dU/dq
  float* sv = se + 32;                                    // w1 (1 - tanh^2) [64]
  float* sh = sv + 64;                                    // tanh [64]
  float* sw = sh + 64;                                    // w1 [64]
  float* sgr = sw + 64;                                   // trace gradients [NA][5]
  float* sMom = sgr + 32;                                 // F [T][9], V [T][9][3], W [T][9][6]
  float* sD = sMom + T * 90;                              // D^t_k [T][9]

  const float4 pi = na.pos4[i];
  const int ti = __float_as_int(pi.w);
  const int s = na.sorted_struct[i];

  // ---------------------------------------------------------------- neighbour lists
  int c0 = 0, c1 = 0, cA = 0;  // entries from the front (all types, or type 0 of two), from the back, angular
  {
    const StructGrid G = na.grids[s];
    const float rc2R = na.rc_R * na.rc_R, rc2A = na.rc_A * na.rc_A;
    const unsigned below = (1u << lane) - 1u;
    const Stencil sten(na, s, G, a.sorted_cell[i] - G.cell_offset, pi, rc2R);
    // Lane r finds the ranges of row r of the stencil; their non-empty ones are
    // laid end to end (32 rows at a time), and the lanes take 32 candidates of
    // that sequence at a time, each following its own range.
    struct Range {
      int off, end;  // candidate j = position + off, for positions before `end`
      float sx, sy, sz;
      int rint_pairs;
    };
    Range* ranges = reinterpret_cast<Range*>(tile);  // at most 96
    const int rows = sten.rows();
    for (int r0 = 0; r0 < rows; r0 += 32) {
      int j0[3] = {0, 0, 0}, len[3] = {0, 0, 0}, ri = 0, nseg = 0;
      float sx[3] = {0.f, 0.f, 0.f}, sy = 0.f, sz = 0.f;
      if (r0 + lane < rows) {
        const int iz = (r0 + lane) / sten.ny, iy = (r0 + lane) - iz * sten.ny;
        sten.row(na, G, iy, iz, [&](int b, int e, float x, float y, float z, bool rint_pairs) {
          if (e <= b) return;
#pragma unroll
          for (int u = 0; u < 3; ++u)
            if (u == nseg) { j0[u] = b; len[u] = e - b; sx[u] = x; }
          sy = y; sz = z; ri = rint_pairs;
          ++nseg;
        });
      }
      int seg = nseg, pos = len[0] + len[1] + len[2];
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const int us = __shfl_up_sync(0xffffffffu, seg, o), up = __shfl_up_sync(0xffffffffu, pos, o);
        if (lane >= o) { seg += us; pos += up; }
      }
      const int total = __shfl_sync(0xffffffffu, pos, 31);
      seg -= nseg;
      pos -= len[0] + len[1] + len[2];
#pragma unroll
      for (int u = 0; u < 3; ++u) {
        if (u < nseg) {
          Range& q = ranges[seg + u];
          q.off = j0[u] - pos;
          pos += len[u];
          q.end = pos;
          q.sx = sx[u]; q.sy = sy; q.sz = sz; q.rint_pairs = ri;
        }
      }
      __syncwarp();
      const Range* q = ranges;
      Range cur = *q;
      for (int p0 = 0; p0 < total; p0 += 32) {
        const int p = p0 + lane;
        bool inR = false, inA = false;
        int t = 0, j = 0;
        if (p < total) {
          while (p >= cur.end) cur = *++q;
          j = p + cur.off;
          const float4 pj = __ldg(&na.pos4[j]);
          t = __float_as_int(pj.w);
          const float r2 = pair_r2(pj, pi, cur.sx, cur.sy, cur.sz, cur.rint_pairs, G);
          inR = r2 < rc2R && j != i;  // an atom is not its own neighbour
          inA = r2 < rc2A && j != i;
        }
        const unsigned mR = __ballot_sync(0xffffffffu, inR), mA = __ballot_sync(0xffffffffu, inA);
        if (T == 2) {
          const unsigned m1 = __ballot_sync(0xffffffffu, inR && t != 0), m0 = mR & ~m1;
          if (inR) {
            if (t == 0) {
              const int e = c0 + __popc(m0 & below);
              if (e < na.cap_R) sR[e] = j;
            } else {
              const int e = c1 + __popc(m1 & below);
              if (e < na.cap_R) sR[na.cap_R - 1 - e] = j;
            }
          }
          c0 += __popc(m0);
          c1 += __popc(m1);
        } else {
          if (inR) {
            const int e = c0 + __popc(mR & below);
            if (e < na.cap_R) (T > 2 ? sTmp : sR)[e] = j | (t << kTypeShift);
          }
          c0 += __popc(mR);
        }
        if (inA) {
          const int e = cA + __popc(mA & below);
          if (e < na.cap_A) sA[e] = j;
        }
        cA += __popc(mA);
      }
      __syncwarp();
    }
  }
  const int nR = c0 + c1;
  if (lane == 0) {
    if (nR > na.cap_R) atomicMax(&na.status->max_cnt_R, nR);
    if (cA > na.cap_A) atomicMax(&na.status->max_cnt_A, cA);
    if constexpr (!FUSED) na.cnt_A[i] = nR > na.cap_R || cA > na.cap_A ? 0 : cA;  // (no list is written then)
  }
  if (nR > na.cap_R || cA > na.cap_A) return;  // the host repeats the batch with larger lists
  __syncwarp();
  if (T > 2) {  // stable counting sort by type
    const unsigned below = (1u << lane) - 1u;
    int at = 0;
    for (int t = 0; t < T; ++t)
      for (int e0 = 0; e0 < nR; e0 += 32) {
        const int v = e0 + lane < nR ? sTmp[e0 + lane] : -1;
        const bool is = e0 + lane < nR && (int)((unsigned)v >> kTypeShift) == t;
        const unsigned m = __ballot_sync(0xffffffffu, is);
        if (is) sR[at + __popc(m & below)] = v;
        at += __popc(m);
      }
    __syncwarp();
  }

  // ---------------------------------------------------------------- radial moments (radial.cu)
  const StructBox bx = na.boxes[s];
  {
    const float rcinv = 1.f / na.rc_R;
    for (int k = lane; k < T * 90; k += 32) sMom[k] = 0.f;
    __syncwarp();
    float* F = sMom;
    float* V = sMom + T * 9;
    float* W = V + T * 27;
    // Lane 3 k + c (k < 9) owns V_k,c, W_k,c and W_k,c+3: products of row df_k with
    // rows rv_c, rr_c, rr_c+3.  Lanes 27..31 own F_0..F_4 and F_5..F_8: row fc with T_k.
    const int k = lane / 3, c = lane % 3, kf = lane - 27;
    const bool vw = lane < 27;
    const float* ra = tile + (vw ? k : 18) * kRow;
    const float* rb = tile + (vw ? 19 + c : 9 + kf) * kRow;
    const float* rc = tile + (vw ? 22 + c : (kf < 4 ? 14 + kf : 9)) * kRow;
    const float* rd = tile + (vw ? 25 + c : 9) * kRow;
    float s0 = 0.f, s1 = 0.f, s2 = 0.f;
    int cur = 0;
    auto flush = [&](int t) {
      const float f00 = __shfl_sync(0xffffffffu, s0, 27);
      if (vw) {
        V[(t * 9 + k) * 3 + c] = s0;
        W[(t * 9 + k) * 6 + c] = s1;
        W[(t * 9 + k) * 6 + c + 3] = s2;
      } else {
        F[t * 9 + kf] = kf == 0 ? s0 : 0.5f * (s0 + f00);
        if (kf < 4) F[t * 9 + 5 + kf] = 0.5f * (s1 + f00);
      }
      s0 = s1 = s2 = 0.f;
    };
    for (int e0 = 0; e0 < nR; e0 += 32) {
      const int e = e0 + lane, n = min(32, nR - e0);
      int t = 0;
      if (e < nR) {
        const int v = sR[e < c0 ? e : na.cap_R - nR + e];
        const float4 pj = na.pos4[v & kIndexMask];
        t = __float_as_int(pj.w);
        const float dx = min_image(pj.x, pi.x, bx.L[0], bx.invL[0]);
        const float dy = min_image(pj.y, pi.y, bx.L[1], bx.invL[1]);
        const float dz = min_image(pj.z, pi.z, bx.L[2], bx.invL[2]);
        const float r2 = dx * dx + dy * dy + dz * dz;
        const float rinv = rsqrtf(r2);
        const float r = r2 * rinv;
        float sn, cs;
        __sincosf(kPi * r * rcinv, &sn, &cs);
        const float fc = 0.5f + 0.5f * cs;
        const float hdfc = -0.25f * kPi * rcinv * sn;
        const float tt = r * rcinv - 1.f;
        const float x = 2.f * tt * tt - 1.f, x2 = 2.f * x;
        const float hdxfc = 2.f * tt * rcinv * fc;
        float* col = tile + lane;  // quantity q of this pair at col[q * kRow]
        float T0 = 1.f, T1 = x, d0 = 0.f, d1 = 1.f;
        col[0] = 2.f * hdfc;
        col[9 * kRow] = 1.f;
        col[1 * kRow] = fmaf(hdxfc, 1.f, hdfc * (x + 1.f));
        col[10 * kRow] = x;
#pragma unroll
        for (int q = 2; q < B; ++q) {
          const float T2 = fmaf(x2, T1, -T0);
          const float d2 = fmaf(2.f, T1, fmaf(x2, d1, -d0));
          col[(9 + q) * kRow] = T2;
          col[q * kRow] = fmaf(hdxfc, d2, hdfc * (T2 + 1.f));
          T0 = T1; T1 = T2; d0 = d1; d1 = d2;
        }
        col[18 * kRow] = fc;
        col[19 * kRow] = r * dx; col[20 * kRow] = r * dy; col[21 * kRow] = r * dz;
        const float ux = dx * rinv, uy = dy * rinv;
        col[22 * kRow] = ux * dx; col[23 * kRow] = ux * dy; col[24 * kRow] = ux * dz;
        col[25 * kRow] = uy * dy; col[26 * kRow] = uy * dz; col[27 * kRow] = dz * rinv * dz;
      }
      __syncwarp();
      // runs of one type inside this chunk, four pairs per load
      for (int b = 0; b < n;) {
        const int tb = __shfl_sync(0xffffffffu, t, b);
        const unsigned same = __ballot_sync(0xffffffffu, lane >= b && lane < n && t == tb);
        const int end = b + __popc(same);
        if (tb != cur) {
          flush(cur);
          cur = tb;
        }
        int p = b;
        auto add = [&](float x, float u, float v, float w) {
          s0 = fmaf(x, u, s0);
          s1 = fmaf(x, v, s1);
          s2 = fmaf(x, w, s2);
        };
        for (; p < end && (p & 3); ++p) add(ra[p], rb[p], rc[p], rd[p]);
#pragma unroll 2
        for (; p + 4 <= end; p += 4) {
          const float4 x = *reinterpret_cast<const float4*>(ra + p), u = *reinterpret_cast<const float4*>(rb + p);
          const float4 v = *reinterpret_cast<const float4*>(rc + p), w = *reinterpret_cast<const float4*>(rd + p);
          add(x.x, u.x, v.x, w.x);
          add(x.y, u.y, v.y, w.y);
          add(x.z, u.z, v.z, w.z);
          add(x.w, u.w, v.w, w.w);
        }
        for (; p < end; ++p) add(ra[p], rb[p], rc[p], rd[p]);
        b = end;
      }
      __syncwarp();
    }
    flush(cur);
    __syncwarp();
  }
  const float* F = sMom;
  const float* V = sMom + T * 9;
  const float* W = V + T * 27;

  if constexpr (!FUSED) {
    for (int e = lane; e < cA; e += 32) na.nbr_A[nbr_index(i, e, na.cap_A)] = sA[e];
    float* mom = a.mom + i;
    const size_t ms = a.mom_stride;
    for (int q = lane; q < T * 9; q += 32) mom[(size_t)q * ms] = F[q];
    if (a.v0 >= 0)
      for (int q = lane; q < T * 27; q += 32) mom[(size_t)(a.v0 + q) * ms] = V[q];
    if (a.w0 >= 0)
      for (int q = lane; q < T * 54; q += 32) mom[(size_t)(a.w0 + q) * ms] = W[q];
    return;
  } else {
    const float rcAinv = 1.f / na.rc_A;
    Pair<BA> pr;  // this lane's pair of the current chunk; kept when one chunk holds all
    const int first = min(cA, 32);
    pr.t = 0;
    if (lane < first) pr.load(na.pos4, sA[lane], pi, bx, rcAinv);

    for (int m = 0; m < a.n_models; ++m) {
      const ModelLayout& Ly = a.model[m].lay;
      const float* model = a.model[m].model;
      const int rank = a.model[m].rank, C = rank == 1 ? 3 : 9;
      const int net = Ly.nets > 1 ? ti : 0;
      const float* cR_i = model + Ly.off_cR + ti * T * Ly.stride_cR;
      const float* cA_i = model + Ly.off_cA + ti * T * Ly.stride_cA;

      // ------------------------------------------------------------ radial descriptor, angular sums
      float q = 0.f;
      if (lane < NR) {
        for (int t = 0; t < T; ++t) {
          const float* cc = cR_i + t * Ly.stride_cR + lane * BR;
#pragma unroll
          for (int k = 0; k < BR; ++k) q += __ldg(cc + k) * F[t * 9 + k];
        }
      }
      float A[NA];
#pragma unroll
      for (int n = 0; n < NA; ++n) A[n] = 0.f;
      float g[NA], dg[NA];
      for (int e0 = 0; e0 < cA; e0 += 32) {
        const int n = min(32, cA - e0);
        if (lane < n) {
          if (cA > 32) pr.load(na.pos4, sA[e0 + lane], pi, bx, rcAinv);
          pr.template radial_functions<NA>(cA_i, Ly.stride_cA, g, dg);
          float* col = tile + lane;
          if (cA > 32 || m == 0) {  // rows 0..NLM-1: the harmonics, kept for the other models
            float hx = pr.dx * pr.rinv, hy = pr.dy * pr.rinv, hz = pr.dz * pr.rinv;
            opaque(hx, hy, hz);
            float p[NLM];
            real_harmonics<LMAX>(hx, hy, hz, p);
#pragma unroll
            for (int u = 0; u < NLM; ++u) col[u * kRow] = p[u];
          }
#pragma unroll
          for (int u = 0; u < NA; ++u) col[(kTileG + u) * kRow] = g[u];
        }
        __syncwarp();
        if (lane < NLM) {
          const float* rp = tile + lane * kRow;
          const float* rg = tile + kTileG * kRow;
          int p = 0;
#pragma unroll 2
          for (; p + 4 <= n; p += 4) {
            const float4 h = *reinterpret_cast<const float4*>(rp + p);
#pragma unroll
            for (int u = 0; u < NA; ++u) {
              const float4 x = *reinterpret_cast<const float4*>(rg + u * kRow + p);
              A[u] = fmaf(x.x, h.x, A[u]);
              A[u] = fmaf(x.y, h.y, A[u]);
              A[u] = fmaf(x.z, h.z, A[u]);
              A[u] = fmaf(x.w, h.w, A[u]);
            }
          }
          for (; p < n; ++p) {
#pragma unroll
            for (int u = 0; u < NA; ++u) A[u] = fmaf(rg[u * kRow + p], rp[p], A[u]);
          }
        }
        __syncwarp();
      }
      if (lane < NLM) {
#pragma unroll
        for (int n = 0; n < NA; ++n) sAs[n * 24 + lane] = A[n];
      }
      __syncwarp();
      // q_nl (lane (l - 1) NA + n) and the 4-body term (lane LMAX NA + n)
      if (lane < NR) sq[lane] = q;
      if (lane < LMAX * NA) {
        const int l = lane / NA + 1, n = lane % NA;
        float v2 = 0.f;
        for (int lm = l * l - 1; lm < (l + 1) * (l + 1) - 1; ++lm) {
          const float v = sAs[n * 24 + lm];
          v2 = fmaf(__fmul_rn(a.w[lm], v), v, v2);
        }
        sq[NR + lane] = v2;
      } else if (lane < LMAX * NA + NA) {
        const int n = lane - LMAX * NA;
        float a2[5], gr[5];
#pragma unroll
        for (int u = 0; u < 5; ++u) a2[u] = sAs[n * 24 + 3 + u];
        sq[NR + lane] = kC4 * trace_m3(a2, gr);
#pragma unroll
        for (int u = 0; u < 5; ++u) sgr[n * 5 + u] = gr[u];
      }
      __syncwarp();

      // ------------------------------------------------------------ network (Eq. 1)
      const float* sc = model + Ly.off_scaler;
      const float scl = lane < DP ? __ldg(sc + lane) : 0.f;
      if (lane < DP) sq[lane] = lane < D ? sq[lane] * scl : 0.f;
      __syncwarp();
      const float* W0 = model + Ly.off_W0 + net * Ly.H * DP;
      const float* b0 = model + Ly.off_b0 + net * Ly.H;
      const float* w1p = model + Ly.off_w1 + net * Ly.H;
      for (int h = lane; h < Ly.H; h += 32) {
        // float4 v of hidden unit h at Wt[v * Hp + h]: 32 units are contiguous
        const float4* Wt = reinterpret_cast<const float4*>(a.model[m].w0t) + (size_t)net * (DP / 4) * a.model[m].Hp + h;
        // partial sums as the packed form of k_fused keeps them
        float z[8];
#pragma unroll
        for (int u = 0; u < 8; ++u) z[u] = 0.f;
#pragma unroll
        for (int v = 0; v < DP / 4; ++v) {
          const float4 w = __ldg(Wt + v * a.model[m].Hp);
          const float4 x = reinterpret_cast<const float4*>(sq)[v];
          const int o = (v & 1) * 2;
          z[o] = fmaf(w.x, x.x, z[o]);
          z[o + 1] = fmaf(w.y, x.y, z[o + 1]);
          z[4 + o] = fmaf(w.z, x.z, z[4 + o]);
          z[5 + o] = fmaf(w.w, x.w, z[5 + o]);
        }
        const float zs = ((z[0] + z[1]) + (z[2] + z[3])) + ((z[4] + z[5]) + (z[6] + z[7]));
        const float hh = tanhf(zs - __ldg(b0 + h));
        const float wh = __ldg(w1p + h);
        sh[h] = hh;
        sw[h] = wh;
        sv[h] = wh * (1.f - hh * hh);
      }
      __syncwarp();
      float e = 0.f, U = -__ldg(model + Ly.off_b1 + net);
      {
        const float* Wd = W0 + (lane < DP ? lane : 0);
        int h = 0;
#pragma unroll 2
        for (; h + 4 <= Ly.H; h += 4) {
          const float4 v4 = *reinterpret_cast<const float4*>(sv + h);
          const float x0 = __ldg(Wd), x1 = __ldg(Wd + DP), x2 = __ldg(Wd + 2 * DP), x3 = __ldg(Wd + 3 * DP);
          Wd += 4 * DP;
          e = fmaf(v4.x, x0, e);
          e = fmaf(v4.y, x1, e);
          e = fmaf(v4.z, x2, e);
          e = fmaf(v4.w, x3, e);
          if (rank == 2) {
            const float4 w4 = *reinterpret_cast<const float4*>(sw + h), h4 = *reinterpret_cast<const float4*>(sh + h);
            U = fmaf(w4.x, h4.x, U);
            U = fmaf(w4.y, h4.y, U);
            U = fmaf(w4.z, h4.z, U);
            U = fmaf(w4.w, h4.w, U);
          }
        }
        for (; h < Ly.H; ++h, Wd += DP) {
          e = fmaf(sv[h], __ldg(Wd), e);
          if (rank == 2) U = fmaf(sw[h], sh[h], U);
        }
      }
      if (lane < DP) se[lane] = e * scl;
      __syncwarp();

      // ------------------------------------------------------------ radial part of Eqs. 3-4
      for (int tk = lane; tk < T * 9; tk += 32) {
        const int t = tk / 9, k = tk % 9;
        float Dk = 0.f;
        if (k < BR) {
#pragma unroll
          for (int n = 0; n < NR; ++n) Dk += se[n] * __ldg(cR_i + t * Ly.stride_cR + n * BR + k);
        }
        sD[tk] = Dk;
      }
      // G = dU/dA
      if (lane < NLM) {
        const int l = l_of(lane);
        const float w2 = 2.f * a.w[lane];
#pragma unroll
        for (int n = 0; n < NA; ++n) {
          const float x = __fmul_rn(w2, se[NR + (l - 1) * NA + n]), A = sAs[n * 24 + lane];
          float G = __fmul_rn(x, A);
          if (lane >= 3 && lane < 8)
            G = fmaf(x, A, __fmul_rn(__fmul_rn(kC4, se[NR + LMAX * NA + n]), sgr[n * 5 + lane - 3]));
          sG[n * 24 + lane] = G;
        }
      }
      __syncwarp();
      float acc = 0.f;
      const int cl = lane < C ? lane : 0;
      if (rank == 1) {
        for (int t = 0; t < T; ++t)
#pragma unroll
          for (int k = 0; k < BR; ++k) acc = fmaf(-sD[t * 9 + k], V[(t * 9 + k) * 3 + cl], acc);
      } else {
        const int u = cl / 3, v = cl % 3, lo = min(u, v), hi = max(u, v);
        const int comp = lo == 0 ? hi : (lo == 1 ? 2 + hi : 5);
        for (int t = 0; t < T; ++t)
#pragma unroll
          for (int k = 0; k < BR; ++k) acc = fmaf(-sD[t * 9 + k], W[(t * 9 + k) * 6 + comp], acc);
      }

      // ------------------------------------------------------------ angular backward
      for (int e0 = 0; e0 < cA; e0 += 32) {
        const int n = min(32, cA - e0);
        if (lane < n) {
          if (cA > 32) {
            pr.load(na.pos4, sA[e0 + lane], pi, bx, rcAinv);
            pr.template radial_functions<NA>(cA_i, Ly.stride_cA, g, dg);
          }
          const float dx = pr.dx, dy = pr.dy, dz = pr.dz, rinv = pr.rinv;
          const float r2 = dx * dx + dy * dy + dz * dz;
          float ux = dx * rinv, uy = dy * rinv, uz = dz * rinv;
          opaque(ux, uy, uz);
          float p[NLM];
          real_harmonics<LMAX>(ux, uy, uz, p);
          constexpr int NP = NLM / 2;
          float S[NLM];
          f32x2 gg[NA], P2[NA], sv2[NP];
#pragma unroll
          for (int u = 0; u < NA; ++u) { gg[u] = pk2(g[u], g[u]); P2[u] = 0ull; }
#pragma unroll
          for (int v = 0; v < NP; ++v) sv2[v] = 0ull;
#pragma unroll
          for (int u = 0; u < NA; ++u) {
            const float4* G4 = reinterpret_cast<const float4*>(sG + u * 24);
#pragma unroll
            for (int v = 0; v < (NP + 1) / 2; ++v) {
              const float4 G = G4[v];
              const f32x2 ga = pk2(G.x, G.y), gb = pk2(G.z, G.w);
              sv2[2 * v] = fma2(ga, gg[u], sv2[2 * v]);
              P2[u] = fma2(ga, pk2(p[4 * v], p[4 * v + 1]), P2[u]);
              if (2 * v + 1 < NP) {
                sv2[2 * v + 1 < NP ? 2 * v + 1 : 0] = fma2(gb, gg[u], sv2[2 * v + 1 < NP ? 2 * v + 1 : 0]);
                P2[u] = fma2(gb, pk2(p[4 * v + 2 < NLM ? 4 * v + 2 : 0], p[4 * v + 3 < NLM ? 4 * v + 3 : 0]), P2[u]);
              }
            }
          }
#pragma unroll
          for (int v = 0; v < NP; ++v) unpk2(sv2[v], S[2 * v], S[2 * v + 1]);
          float P[NA];
#pragma unroll
          for (int u = 0; u < NA; ++u) {
            float lo, hi;
            unpk2(P2[u], lo, hi);
            P[u] = lo + hi;
          }
          if constexpr (NLM & 1) {
            float sl = 0.f;
#pragma unroll
            for (int u = 0; u < NA; ++u) {
              sl += sG[u * 24 + NLM - 1] * g[u];
              P[u] += sG[u * 24 + NLM - 1] * p[NLM - 1];
            }
            S[NLM - 1] = sl;
          }
          float srad = 0.f;
#pragma unroll
          for (int u = 0; u < NA; ++u) srad += dg[u] * P[u];
          float vx = 0.f, vy = 0.f, vz = 0.f;
          harmonic_grad<LMAX>(S, ux, uy, uz, vx, vy, vz);
          const float uv = ux * vx + uy * vy + uz * vz;
          const float fx = srad * ux + rinv * (vx - uv * ux);
          const float fy = srad * uy + rinv * (vy - uv * uy);
          const float fz = srad * uz + rinv * (vz - uv * uz);
          float* col = tile + kTileG * kRow + lane;
          col[0] = dx; col[kRow] = dy; col[2 * kRow] = dz; col[3 * kRow] = r2;
          col[4 * kRow] = fx; col[5 * kRow] = fy; col[6 * kRow] = fz;
        }
        __syncwarp();
        {
          const float* ra = tile + (kTileG + (rank == 1 ? 3 : cl / 3)) * kRow;
          const float* rf = tile + (kTileG + 4 + (rank == 1 ? cl : cl % 3)) * kRow;
          int p = 0;
          for (; p + 4 <= n; p += 4) {
            const float4 x = *reinterpret_cast<const float4*>(ra + p), f = *reinterpret_cast<const float4*>(rf + p);
            acc = fmaf(-x.x, f.x, acc);
            acc = fmaf(-x.y, f.y, acc);
            acc = fmaf(-x.z, f.z, acc);
            acc = fmaf(-x.w, f.w, acc);
          }
          for (; p < n; ++p) acc = fmaf(-ra[p], rf[p], acc);
        }
        __syncwarp();
      }
      if (rank == 2 && (lane == 0 || lane == 4 || lane == 8)) acc += U;
      if (lane < C) a.model[m].per_atom[(size_t)lane * a.atom_stride + i] = acc;
      __syncwarp();
    }
  }
}

template <int NR, int NA, int BR, int BA, int LMAX, bool FUSED>
cudaError_t launch_one(const WideArgs& a, int smem, cudaStream_t st) {
  auto fn = k_wide<NR, NA, BR, BA, LMAX, FUSED>;
  // the largest size of any call: another host thread's context may set and launch in between
  const cudaError_t e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kWideMaxSmem);
  if (e != cudaSuccess) return e;
  count_launches(1);
  fn<<<(a.n_active + kWarps - 1) / kWarps, 32 * kWarps, smem, st>>>(a);
  return cudaGetLastError();
}

}  // namespace

size_t wide_smem_bytes(int n_types, int cap_R, int cap_A) {
  return sizeof(int) * (size_t)kWarps * wide_words(n_types, cap_R, cap_A);
}

cudaError_t launch_wide(int variant, bool fused, const WideArgs& a_in, cudaStream_t st) {
  if (a_in.n_active <= 0) return cudaSuccess;
  WideArgs a = a_in;
  for (int k = 0; k < 24; ++k) a.w[k] = wlm(k);
  const int smem = (int)wide_smem_bytes(a.nbr.n_types, a.nbr.cap_R, a.nbr.cap_A);
  if (!fused) return launch_one<5, 5, 9, 9, 4, false>(a, smem, st);  // lists and moments do not depend on the variant
  if (variant == kVarStd) return launch_one<5, 5, 9, 9, 4, true>(a, smem, st);
  if (variant == kVarSmall) return launch_one<4, 3, 7, 6, 3, true>(a, smem, st);
  return cudaErrorInvalidValue;
}

}  // namespace tnep

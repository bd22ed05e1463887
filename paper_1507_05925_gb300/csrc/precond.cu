// Block-Jacobi preconditioner of the GMRES iterations: the FP32 inner solves
// of the refinement (operator with the per-body weighted completion) and the
// FP64 GMRES (the paper's completion).
//
// The operator is the second-kind operator, sqrt(w)-scaled.  Its diagonal
// block for body i,
//   B_i = 1/2 I + D (K_ii + C_i L_ii) D^{-1}     (Laplace: n_i x n_i; Stokes: 2n_i x 2n_i)
// (C_i = 1 for the paper's L) is assembled in FP32 (from hi/lo coordinate
// differences) directly in shared memory and inverted in place by blocked
// Gauss-Jordan elimination without pivoting: the blocks are 1/2 I + compact,
// their pivots stay near 1/2 on the shapes measured (0.36 - 0.50) and an FP32
// inverse accurate to ~1e-6 is far more than a preconditioner needs.  Every
// pivot is checked: one that is not finite or smaller in magnitude than the
// floor (default 1e-3, 1/500 of the identity part), or a non-finite entry of
// the finished inverse, makes the body keep the identity block (counted in
// bie_info.precond_fallbacks), so a nearly singular block can slow GMRES down
// but never poisons it with NaN or huge entries.  A block of
// nb <= 128 unknowns is inverted by one CTA; nb <= 448 by a cluster of four
// CTAs and nb <= 640 by one of eight (few bodies: larger clusters, bj_setup), each
// CTA holding a slice of the columns and reading the pivot panels of the others
// through L2; larger blocks are left as the identity.  The inverses are stored
// column-major as W = B^{-1} - 2I in FP16 (half the bytes of the apply, which
// streams every block once a GMRES iteration: 655 MB in FP32 for 10,000
// bodies of 128 unknowns).  B^{-1} is 2I plus a compact part, so W carries
// FP16's 2^-11 relative precision on that part only; a perturbed
// preconditioner is still one fixed linear map and changes iteration counts
// at most.  P v = 2 v + W v.  Preconditioning is applied from the right,
// z = P v, so the GMRES residual stays the true residual.
#include <cooperative_groups.h>
#include <cuda_runtime.h>
#include <math.h>

#include <algorithm>
#include <vector>

#include "../../include/bie2d.h"
#include "bie_internal.cuh"
#include "pair_math.cuh"
#include "reduce.cuh"

namespace cg = cooperative_groups;

namespace bie {

namespace {

constexpr int kMaxSingle = 128;  // one CTA
constexpr int kMaxBlock4 = 448;  // cluster of four CTAs
constexpr int kMaxBlock = kBjMaxBlock;  // cluster of eight CTAs (640); larger bodies keep the identity
constexpr int kMinCluster = 72;  // the panels' exchange fits the result's place
constexpr int kPB = 16;          // panel width of the blocked elimination
constexpr int kBA = 256;         // threads of an application CTA
constexpr int kApplyRows = 64, kApplyGroups = kBA / kApplyRows;

// Shared-memory leading dimension of a column: odd, so that reading a row
// (stride ld across threads) is free of bank conflicts.
__host__ __device__ __forceinline__ int gj_ld(int nb) { return nb | 1; }
// Columns per CTA of a cluster of cs CTAs: a multiple of the panel width, so
// that each panel lies in one CTA.
__host__ __device__ __forceinline__ int gj_cols(int nb, int cs) {
  return ((nb + cs - 1) / cs + kPB - 1) / kPB * kPB;
}
__host__ __device__ __forceinline__ size_t gj_smem_floats(int nb, int cs) {
  const int h = gj_cols(nb, cs);
  return (size_t)gj_ld(nb) * h + (size_t)h * kPB + (cs > 1 ? 3 : 2) * kPB * kPB;
}

// Entry (row r, column c) of the operator's diagonal block of body i
// (sqrt(w)-scaled; alpha > 0: completion weighted by alpha/|Gamma_i| and
// alpha/W_i, alpha = 0: the paper's completion), in FP32: coordinate differences from
// the hi/lo split (x = x_hi + x_lo, exact leading differences as in the near
// tiles of the pair sum), the column's node data staged in shared memory.
struct BlockRow {
  int kind, a;
  float cf, ct;
  float4 pa;  // (x_hi, y_hi, x_lo, y_lo) of the row's node
  float nxa, nya, swa, ka, pa0, pa1;
  int al;
  // weights of the completion of body i (FP64 divisions: by one thread)
  __device__ static float2 completion(const Geo& g, int kind, int i, double alpha) {
    return make_float2(alpha > 0.0 ? (float)(alpha / g.len[i]) : 1.0f,
                       kind == 1 ? (alpha > 0.0 ? (float)(alpha / g.W[i]) : 1.0f) : 0.f);
  }
  __device__ BlockRow(const Geo& g, int kind_, int i, int r, float2 weights) : kind(kind_) {
    const int a0 = g.body_start[i];
    cf = weights.x;
    ct = weights.y;
    a = a0 + (kind == 1 ? r >> 1 : r);
    al = kind == 1 ? r & 1 : 0;
    pa = g.pf[a];
    const float2 n = g.nf[a];
    nxa = n.x;
    nya = n.y;
    swa = (float)g.sw[a];
    ka = (float)g.kappa[a];
    pa0 = (float)(-(g.y[a] - g.yc[i]));
    pa1 = (float)(g.x[a] - g.xc[i]);
  }
  // column data: cp = (x_hi, y_hi, x_lo, y_lo), cw = (sqrt(w), p_1, p_2, node index)
  __device__ float entry(int r, int c, float4 cp, float4 cw) const {  // Laplace
    const int b = __float_as_int(cw.w);
    const float rx = (pa.x - cp.x) + (pa.z - cp.z), ry = (pa.y - cp.y) + (pa.w - cp.w);
    const float i2 = rcp32(a == b ? 1.f : rx * rx + ry * ry);
    const float k = a == b ? -ka * (float)kInv4Pi : -(float)kInv2Pi * ((rx * nxa + ry * nya) * i2);
    return (r == c ? 0.5f : 0.f) + swa * cw.x * (k + cf);
  }
  // Stokes: columns c (even) and c + 1, the two components of one node
  __device__ float2 entry2(int r, int c, float4 cp, float4 cw) const {
    const int b = __float_as_int(cw.w);
    const float rx = (pa.x - cp.x) + (pa.z - cp.z), ry = (pa.y - cp.y) + (pa.w - cp.w);
    const bool self = a == b;
    const float i2 = rcp32(self ? 1.f : rx * rx + ry * ry);
    const float t = self ? -0.5f * (float)kInvPi * ka * (al == 0 ? -nya : nxa)
                         : -(float)kInvPi * (al == 0 ? rx : ry) * ((rx * nxa + ry * nya) * i2);
    const float k0 = t * (self ? -nya : rx * i2), k1 = t * (self ? nxa : ry * i2);
    const float q = ct * (al == 0 ? pa0 : pa1), sw = swa * cw.x;
    return make_float2((r == c ? 0.5f : 0.f) + sw * (k0 + (al == 0 ? cf : 0.f) + q * cw.y),
                       (r == c + 1 ? 0.5f : 0.f) + sw * (k1 + (al == 1 ? cf : 0.f) + q * cw.z));
  }
};

constexpr int kRPT = 2;  // rows a thread of the update
// Threads a row group of the update needs for nb rows, and column groups.
__host__ __device__ __forceinline__ int gj_rows(int nb) { return (nb + 32 * kRPT - 1) / (32 * kRPT) * 32; }

// A_:j = A_:j + F G_j (START and the rows with fresh set: A_:j = F G_j) for the local columns
// j0, j0 + step, ... (four each) of the thread's rows.  G is [kPB][h]: one 16-byte load
// gives four columns of one row and feeds 4 kRPT multiply-adds (a load takes the
// shared-memory pipe four clocks; with one row a thread it bound the update, with four
// the registers spill: 100 blocks of 256 223 us against 186); each column's terms in the
// order t = 0, 1, ...
// SHARE: the columns also go to out (column j at out + j nb).
template <bool START, bool SHARE>
__device__ __forceinline__ void rank_update(float* __restrict__ A, const float* __restrict__ G, int h, int ld, int row0,
                                            int stride, int nb, int fresh, const float (&fr)[kRPT][kPB], int j0, int j1,
                                            int step, float* __restrict__ out = nullptr) {
#pragma unroll 1
  for (int j = j0; j < j1; j += step) {
    float2 a01[kRPT], a23[kRPT];
#pragma unroll
    for (int s = 0; s < kRPT; ++s) {
      const int r = row0 + s * stride;
      a01[s] = a23[s] = make_float2(0.f, 0.f);
      if (!START && r < nb && !(fresh >> s & 1)) {
        a01[s] = make_float2(A[j * ld + r], A[(j + 1) * ld + r]);
        a23[s] = make_float2(A[(j + 2) * ld + r], A[(j + 3) * ld + r]);
      }
    }
#pragma unroll
    for (int t = 0; t < kPB; ++t) {
      const float4 g = *reinterpret_cast<const float4*>(G + t * h + j);
#pragma unroll
      for (int s = 0; s < kRPT; ++s) {
        const float2 f = make_float2(fr[s][t], fr[s][t]);
        a01[s] = __ffma2_rn(f, make_float2(g.x, g.y), a01[s]);
        a23[s] = __ffma2_rn(f, make_float2(g.z, g.w), a23[s]);
      }
    }
#pragma unroll
    for (int s = 0; s < kRPT; ++s) {
      const int r = row0 + s * stride;
      if (r < nb) {
        A[j * ld + r] = a01[s].x;
        A[(j + 1) * ld + r] = a01[s].y;
        A[(j + 2) * ld + r] = a23[s].x;
        A[(j + 3) * ld + r] = a23[s].y;
        if (SHARE) {
          out[j * nb + r] = a01[s].x;
          out[(j + 1) * nb + r] = a01[s].y;
          out[(j + 2) * nb + r] = a23[s].x;
          out[(j + 3) * nb + r] = a23[s].y;
        }
      }
    }
  }
}

// Inverse of a 16 x 16 pivot block by one warp, in registers: lane t0 + 16 half holds
// the columns 8 half + u of row t0.  Gauss-Jordan, the pivot row by shuffles, no
// branches (100 clocks a pivot).  Every pivot is checked.
__device__ __forceinline__ void invert_panel(float (&a)[kPB / 2], float* inv, float floor, int* bad) {
  constexpr int H = kPB / 2;
  const int lane = threadIdx.x & 31, t0 = lane & (kPB - 1), half = lane / kPB;
  bool ok = true;
#pragma unroll 1
  for (int tb = 0; tb < 2; ++tb)
#pragma unroll
    for (int u0 = 0; u0 < H; ++u0) {
      const int t = H * tb + u0;
      const float pv = __shfl_sync(0xffffffffu, a[u0], t + kPB * tb);
      const float m = __shfl_sync(0xffffffffu, a[u0], t0 + kPB * tb);
      const float ip = __frcp_rn(pv);
      ok &= fabsf(pv) >= floor && isfinite(pv);
      const bool piv = t0 == t;
      const float f = piv ? ip : -m * ip;
#pragma unroll
      for (int u = 0; u < H; ++u) {
        const float q = __shfl_sync(0xffffffffu, a[u], t + kPB * half);
        a[u] = fmaf(f, q, piv ? 0.f : a[u]);
      }
      if (half == tb) a[u0] = f;
    }
  if (!ok) *bad = 1;
  float4* o = reinterpret_cast<float4*>(inv + t0 * kPB + H * half);
  o[0] = make_float4(a[0], a[1], a[2], a[3]);
  o[1] = make_float4(a[4], a[5], a[6], a[7]);
}

// Assembly and in-place inversion of one diagonal block by a cluster of CS CTAs
// (CS = 1: one CTA).  CTA q holds the columns [q h, min(nb, (q+1) h)) and all
// rows; T threads share the rows (kRPT each), and the groups of T threads the columns;
// one more warp inverts.  Blocked Gauss-Jordan without pivoting, for each
// panel K of kPB pivots: with I = inv(A_KK), G_j = I A_Kj, every CTA sets
//   A_Rj -= A_RK G_j, A_Kj = G_j  (its columns j outside K),
//   A_RK = -A_RK I, A_KK = I      (the panel's owner),
// reading I from the owner's shared memory and A_RK through L2: the owner writes the
// next panel to the place of the result in memory (two panels in turn; a cluster's
// other CTAs read 20 bytes a clock together from one SM's shared memory, which was
// 25,000 clocks a panel of 256 rows).  One cluster barrier a panel.
// What bounds it is the chain of panels and the shared-memory pipe.  The serial part, I, is
// 16 x 16 by one warp, formed one panel ahead: the warp adds this panel's update to the
// 16 x 16 next pivots itself and inverts them while the others update.  (An
// elimination of the whole panel by all rows took a block barrier and a division a
// column, while the other CTAs waited.)  A panel of a block of 256 takes 10,000 clocks
// (25,000 before).  Bodies of nb unknowns: four of 128 77 -> 43 us, 10,000 of 128 3085 ->
// 2444; 100 of 256 213 -> 186, 400 of 256 748 -> 645; 236, 286, 482 and 482 560 -> 254.
template <int CS, int THREADS>
__global__ void __launch_bounds__(THREADS, THREADS <= 160 ? 3 : CS == 1 ? 2 : 1)
    k_bj_factor(Geo g, int kind, double alpha, const int* __restrict__ list, const long long* __restrict__ off,
                bj_t* __restrict__ blocks, float floor, int* __restrict__ fallbacks, int T) {
  extern __shared__ __align__(16) float sm[];
  __shared__ int bad_s;  // this CTA met a bad pivot or a non-finite entry
  const int rank = CS > 1 ? (int)cg::this_cluster().block_rank() : 0;
  const int i = list[blockIdx.x / CS];
  const int nb = (g.body_start[i + 1] - g.body_start[i]) * (kind + 1);
  const int ld = gj_ld(nb), h = gj_cols(nb, CS);
  const int c0 = min(nb, rank * h), nc = min(nb, c0 + h) - c0, nc4 = (nc + 3) & ~3;
  float* A = sm;                         // ld x h, column-major
  float* G = A + (size_t)ld * h;         // kPB x h: G_j of the local columns
  float* pub = G + (size_t)h * kPB;      // [2] I of this and the next panel (the owner's)
  float* copy = pub + 2 * kPB * kPB;     // CS > 1: this CTA's copy of I
  float4* colp = reinterpret_cast<float4*>(G);  // [h] column node positions (assembly)
  float4* colw = colp + h;                      // [h] column node data
  bj_t* B = blocks + off[i];
  // CS > 1 (nb >= kMinCluster): the panels' exchange, 2 x 16 columns of 4 nb bytes of the 2 nb^2
  float* xch = reinterpret_cast<float*>((reinterpret_cast<uintptr_t>(B) + 15) & ~uintptr_t(15));
  const int work = blockDim.x - 32, CG = work / T;  // threads and column groups of the update
  const bool inverter = (int)threadIdx.x >= work;
  const int row0 = (int)threadIdx.x % T, cgrp = (int)threadIdx.x / T;  // (not the inverter's)
  __shared__ float2 weights;
  if (threadIdx.x == 0) bad_s = 0;
  if ((int)threadIdx.x == work) weights = BlockRow::completion(g, kind, i, alpha);
  {
    const int a0 = g.body_start[i];
    const double xc = g.xc[i], yc = g.yc[i];
    for (int j = threadIdx.x; j < nc; j += blockDim.x) {
      const int c = c0 + j;
      const int b = a0 + (kind == 1 ? c >> 1 : c);
      colp[j] = g.pf[b];
      colw[j] = make_float4((float)g.sw[b], (float)(-(g.y[b] - yc)), (float)(g.x[b] - xc), __int_as_float(b));
    }
  }
  __syncthreads();
  if (!inverter) {
    // a row a thread, as many column groups as there are threads for
    const int rows = (nb + 31) / 32 * 32, cgs = max(1, work / rows);
    for (int q = threadIdx.x; q < cgs * rows; q += work) {
      const int r = q % rows, cgp = q / rows;
      if (r >= nb) continue;
      const BlockRow br(g, kind, i, r, weights);
      if (kind == 0) {
#pragma unroll 4
        for (int j = cgp; j < nc; j += cgs) A[j * ld + r] = br.entry(r, c0 + j, colp[j], colw[j]);
      } else {
#pragma unroll 4
        for (int j = 2 * cgp; j < nc; j += 2 * cgs) {
          const float2 e = br.entry2(r, c0 + j, colp[j], colw[j]);
          A[j * ld + r] = e.x;
          A[(j + 1) * ld + r] = e.y;
        }
      }
      if (cgp == 0)
        for (int j = nc; j < nc4; ++j) A[j * ld + r] = 0.f;
    }
  }
  __syncthreads();
  if (CS > 1 && rank == 0)
    for (int e = threadIdx.x; e < min(kPB, nb) * nb; e += blockDim.x) xch[e] = A[e / nb * ld + e % nb];
  // the inverter's lane: row t0, columns 8 half.. of a pivot block
  const int t0 = threadIdx.x & (kPB - 1), uh = ((threadIdx.x & 31) / kPB) * (kPB / 2);
  if (rank == 0 && inverter) {
    float a[kPB / 2];
#pragma unroll
    for (int u = 0; u < kPB / 2; ++u) a[u] = t0 < nb && uh + u < nb ? A[(uh + u) * ld + t0] : (t0 == uh + u ? 1.f : 0.f);
    invert_panel(a, pub, floor, &bad_s);
  }
  if constexpr (CS > 1)
    cg::this_cluster().sync();
  else
    __syncthreads();
  int parity = 0;
  for (int k0 = 0; k0 < nb; k0 += kPB, parity ^= 1) {
    const int bsz = min(kPB, nb - k0), owner = k0 / h, lj = k0 - c0;
    const int k1 = k0 + kPB, n0 = k1 - c0;
    const bool ahead = k1 < nb && k1 / h == rank;  // this CTA has the next panel
    const float* P = CS > 1 ? xch + parity * kPB * nb : A + k0 * ld;
    const int pld = CS > 1 ? nb : ld;
    const auto panel = [&](int t, int r) { return CS > 1 ? __ldcg(P + t * pld + r) : P[t * pld + r]; };
    const float* inv = pub + parity * kPB * kPB;
    if constexpr (CS > 1) {
      const float* I = cg::this_cluster().map_shared_rank(inv, owner);
      for (int e = threadIdx.x; e < kPB * kPB; e += blockDim.x) copy[e] = I[e];
      inv = copy;
    }
    // the thread's rows of the panel, negated (rows K: the unit vectors, so that F G_j = G_j);
    // the inverter: its row in fr[0] and the next pivot block.  Loads first, at clamped
    // indexes, then selections: a load inside a condition is waited for one by one
    float fr[kRPT][kPB], a[kPB / 2];
    int fresh = 0;
    if (!inverter) {
#pragma unroll
      for (int s = 0; s < kRPT; ++s)
#pragma unroll
        for (int t = 0; t < kPB; ++t) fr[s][t] = panel(min(t, bsz - 1), min(row0 + s * T, nb - 1));
#pragma unroll
      for (int s = 0; s < kRPT; ++s) {
        const int r = row0 + s * T;
        const bool in = r >= k0 && r < k0 + bsz;
        fresh |= in ? 1 << s : 0;
#pragma unroll
        for (int t = 0; t < kPB; ++t) fr[s][t] = in ? (r - k0 == t ? 1.f : 0.f) : t < bsz ? -fr[s][t] : 0.f;
      }
    } else if (ahead) {
      const int r = min(k1 + t0, nb - 1);
#pragma unroll
      for (int t = 0; t < kPB; ++t) fr[0][t] = panel(t, r);  // (a panel with a next one is full)
#pragma unroll
      for (int u = 0; u < kPB / 2; ++u) a[u] = A[min(n0 + uh + u, nc - 1) * ld + r];
#pragma unroll
      for (int t = 0; t < kPB; ++t) fr[0][t] = k1 + t0 < nb ? -fr[0][t] : 0.f;
#pragma unroll
      for (int u = 0; u < kPB / 2; ++u)
        if (k1 + t0 >= nb || n0 + uh + u >= nc) a[u] = t0 == uh + u ? 1.f : 0.f;
    }
    __syncthreads();
    // G_j = I A_Kj (the panel's own columns: I), four rows of a column a thread
    for (int e = threadIdx.x; e < 4 * nc4; e += blockDim.x) {
      const int uq = e / nc4, j = e - uq * nc4;
      const bool own = rank == owner && j >= lj && j < lj + bsz;
      float c[kPB];
#pragma unroll
      for (int t = 0; t < kPB; ++t) c[t] = A[j * ld + k0 + min(t, bsz - 1)];
#pragma unroll
      for (int t = 0; t < kPB; ++t) c[t] = own ? (j - lj == t ? 1.f : 0.f) : t < bsz ? c[t] : 0.f;
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        float v = 0.f;
#pragma unroll
        for (int t = 0; t < kPB; t += 4) {
          const float4 q = *reinterpret_cast<const float4*>(inv + (4 * uq + u) * kPB + t);
          v = fmaf(q.w, c[t + 3], fmaf(q.z, c[t + 2], fmaf(q.y, c[t + 1], fmaf(q.x, c[t], v))));
        }
        G[(4 * uq + u) * h + j] = v;
      }
    }
    __syncthreads();
    // all local columns but the panel's own (owner: [lj, lj + kPB))
    const int s0 = rank == owner ? lj : nc4, s1 = rank == owner ? min(nc4, lj + kPB) : nc4;
    if (!inverter) {
      int b0 = s0, b1 = s1;
      if (CS > 1 && ahead) {
        // the next panel's columns first; it follows this one where both are here
        const int n1 = min(nc4, n0 + kPB);
        rank_update<false, true>(A, G, h, ld, row0, T, nb, fresh, fr, n0 + 4 * cgrp, n1, 4 * CG,
                                 xch + ((parity ^ 1) * kPB - n0) * nb);
        b0 = min(s0, n0);
        b1 = n1;
      }
      rank_update<false, false>(A, G, h, ld, row0, T, nb, fresh, fr, 4 * cgrp, b0, 4 * CG);
      rank_update<false, false>(A, G, h, ld, row0, T, nb, fresh, fr, b1 + 4 * cgrp, nc4, 4 * CG);
    } else if (ahead) {
#pragma unroll
      for (int t = 0; t < kPB; ++t)
#pragma unroll
        for (int u = 0; u < kPB / 2; ++u) {
          const float q = G[t * h + min(n0 + uh + u, nc - 1)];
          a[u] = fmaf(n0 + uh + u < nc ? fr[0][t] : 0.f, q, a[u]);
        }
      invert_panel(a, pub + (parity ^ 1) * kPB * kPB, floor, &bad_s);
    }
    // the panel (every thread read its rows before the barriers above)
    if (!inverter && rank == owner) rank_update<true, false>(A, G, h, ld, row0, T, nb, fresh, fr, s0 + 4 * cgrp, s1, 4 * CG);
    if constexpr (CS > 1)
      cg::this_cluster().sync();
    else
      __syncthreads();
  }
  // an entry that overflowed in the updates, or whose W = B^{-1} - 2I entry
  // lies outside FP16's range, also rejects the block
  if (!inverter) {
    bool nf = false;
    for (int r = row0; r < nb; r += T)
      for (int j = cgrp; j < nc; j += CG) {
        const float a = A[j * ld + r] - (c0 + j == r ? kBjShift : 0.f);
        nf |= !(fabsf(a) <= 65000.f);
      }
    if (nf) bad_s = 1;
  }
  // every CTA of the cluster learns whether any of them rejected the block
  // (the first sync also keeps every CTA alive while the last panel is read)
  int bad;
  if constexpr (CS > 1) {
    cg::this_cluster().sync();
    bad = 0;
    for (int q = 0; q < CS; ++q) bad |= *cg::this_cluster().map_shared_rank(&bad_s, q);
    cg::this_cluster().sync();
  } else {
    __syncthreads();
    bad = bad_s;
  }
  if (bad && rank == 0 && threadIdx.x == 0) atomicAdd(fallbacks, 1);
  if (inverter) return;
  for (int r = row0; r < nb; r += T)
    for (int j = cgrp; j < nc; j += CG) {
      const bool diag = c0 + j == r;
      const float d = diag ? kBjShift : 0.f;  // W = B^{-1} - 2I; the identity: W = -I
      B[(long long)(c0 + j) * nb + r] = __float2half_rn(bad ? (diag ? 1.f : 0.f) - d : A[j * ld + r] - d);
    }
}

// z = P v in FP32 arithmetic: z_i = B_i^{-1} v_i per body (identity for bodies
// left out).  CTA (i, y) computes rows [64 y, 64 y + 64) of body i with four
// column groups of 64 threads, reduced in shared memory; each warp reads 32
// consecutive rows of one column (coalesced).
__global__ void __launch_bounds__(kBA) k_bj_apply(Geo g, int kind, const long long* __restrict__ off,
                                                  const bj_t* __restrict__ blocks, VecRef vr, double* __restrict__ z,
                                                  const int* __restrict__ stop) {
  if (stop && *stop) return;
  extern __shared__ __align__(16) float vs[];
  __shared__ float part[kBA];
  const double* v = vr.ptr();
  const int i = blockIdx.x;
  const int c = kind + 1;
  const int a0 = g.body_start[i] * c, nb = (g.body_start[i + 1] - g.body_start[i]) * c;
  const int r0 = blockIdx.y * kApplyRows;
  if (r0 >= nb) return;
  const int lr = threadIdx.x % kApplyRows, grp = threadIdx.x / kApplyRows;
  const int r = r0 + lr;
  if (nb > kMaxBlock) {
    if (grp == 0 && r < nb) z[a0 + r] = v[a0 + r];
    return;
  }
  for (int e = threadIdx.x; e < nb; e += kBA) vs[e] = (float)v[a0 + e];
  __syncthreads();
  const bj_t* B = blocks + off[i];
  float acc = 0;
  if (r < nb) {
    const int per = (nb + kApplyGroups - 1) / kApplyGroups;
    const int cb = grp * per, ce = min(nb, cb + per);
#pragma unroll 4
    for (int col = cb; col < ce; ++col) acc = fmaf(__half2float(B[(long long)col * nb + r]), vs[col], acc);
  }
  part[threadIdx.x] = acc;
  __syncthreads();
  if (grp == 0 && r < nb) {
    float t = part[lr];
#pragma unroll
    for (int q = 1; q < kApplyGroups; ++q) t += part[q * kApplyRows + lr];
    z[a0 + r] = (double)(fmaf(kBjShift, vs[r], t));  // P v = 2 v + W v
  }
}

// z = P v in FP64 arithmetic on the FP16 blocks (FP64 GMRES: P must be one fixed
// linear map to FP64 rounding).  With NORM, v is the basis vector that an
// Arnoldi step left unnormalised in `v`: v / st->hnext is written to row st->j of
// V as well (nothing is done once the cycle has stopped).
// Bound by the FP64 pipe (two lanes a clock per SM), so the rows of a body are
// spread over CTAs of 32 (32 rows x 8 column groups), as many as there are; an
// Arnoldi step that applied a body's block on one CTA took 178 us at 740 nodes in
// four bodies of up to 600 unknowns and 139 us at 7,100 nodes in 36 bodies, with
// this launch beside it 22 + 19 and 26 + 13 us.  An FP16 entry becomes a double
// without the FP64 pipe (a conversion would run on it): its bits, placed in the
// high word, are the value times 2^-1008 exactly (FP16 subnormals become FP64
// ones); v carries 2^500 and the sum 2^508.
constexpr int kRows64 = 32, kGroups64 = kBA / kRows64;

template <bool NORM>
__global__ void __launch_bounds__(kBA) k_bj_apply64(Geo g, int kind, const long long* __restrict__ off,
                                                    const bj_t* __restrict__ blocks, const double* __restrict__ v,
                                                    double* __restrict__ z, double* __restrict__ V, long long ld,
                                                    const KState* __restrict__ st, const int* __restrict__ stop) {
  if (stop && *stop) return;
  extern __shared__ __align__(16) double vd[];
  __shared__ double part[kBA];
  const int i = blockIdx.x;
  const int c = kind + 1;
  const int a0 = g.body_start[i] * c, nb = (g.body_start[i + 1] - g.body_start[i]) * c;
  const int r0 = blockIdx.y * kRows64;
  if (r0 >= nb) return;
  const double inv = NORM ? 1.0 / st->hnext : 1.0;
  double* vout = NORM ? V + (long long)st->j * ld + a0 : nullptr;
  if (nb > kMaxBlock) {  // the identity
    for (long long e = blockIdx.y * kBA + threadIdx.x; e < nb; e += gridDim.y * kBA) {
      const double t = v[a0 + e] * inv;
      if (NORM) vout[e] = t;
      z[a0 + e] = t;
    }
    return;
  }
  const int lr = threadIdx.x % kRows64, grp = threadIdx.x / kRows64;
  const int r = r0 + lr;
  const double up = __hiloint2double((1023 + 500) << 20, 0), down = __hiloint2double((1023 - 500) << 20, 0);  // 2^500
  for (int e = threadIdx.x; e < nb; e += kBA) vd[e] = v[a0 + e] * inv * up;
  __syncthreads();
  const unsigned short* B = reinterpret_cast<const unsigned short*>(blocks + off[i]);
  double s0 = 0.0, s1 = 0.0;
  if (r < nb) {
    auto entry = [&](int col) {
      const unsigned h = B[(long long)col * nb + r];
      return __hiloint2double((int)(((h & 0x8000u) << 16) | ((h & 0x7fffu) << 10)), 0);
    };
    const int per = (nb + kGroups64 - 1) / kGroups64;
    const int cb = grp * per, ce = min(nb, cb + per);
    int col = cb;
#pragma unroll 4
    for (; col + 2 <= ce; col += 2) {
      s0 = fma(entry(col), vd[col], s0);
      s1 = fma(entry(col + 1), vd[col + 1], s1);
    }
    if (col < ce) s0 = fma(entry(col), vd[col], s0);
  }
  part[threadIdx.x] = s0 + s1;
  __syncthreads();
  if (grp == 0 && r < nb) {
    double t = part[lr];
#pragma unroll
    for (int q = 1; q < kGroups64; ++q) t += part[q * kRows64 + lr];
    t *= __hiloint2double((1023 + 508) << 20, 0);  // 2^508
    const double x = vd[r] * down;
    if (NORM) vout[r] = x;
    z[a0 + r] = fma((double)kBjShift, x, t);  // P v = 2 v + W v
  }
}

}  // namespace

long long bj_block_floats(const int* body_start_host, int N, int kind) {
  long long s = 0;
  for (int i = 0; i < N; ++i) {
    const long long nb = (long long)(body_start_host[i + 1] - body_start_host[i]) * (kind + 1);
    if (nb <= kMaxBlock) s += nb * nb;
  }
  return s;
}

namespace {

// Launch of k_bj_factor<CS, THREADS> over count bodies of list.
float g_pivot_floor = 0.f;  // test hook (0: the default floor)
constexpr float kPivotFloor = 1e-3f;

template <int CS, int THREADS>
cudaError_t launch_factor(const Geo& g, int kind, double alpha, const int* list, int count, int max_nb, size_t smem,
                          const long long* off, bj_t* blocks, int* fallbacks, cudaStream_t s) {
  // the update's threads, and one warp for the pivots (column groups read the panel each:
  // nb = 256 in clusters of four 186 us for 100 bodies with one, 334 with two; nb <= 446, 155 bodies,
  // 1296 and 895; clusters of eight have no registers for two: 32 bodies of 512 731 and 790)
  const int T = gj_rows(max_nb), groups = T > 128 ? (CS == 4 ? 2 : 1) : (CS == 1 ? 256 : 128) / T, threads = groups * T + 32;
  // a constant bound (the largest block's): with this launch's size, another thread's
  // launch could find a smaller one than it needs
  cudaError_t e = cudaFuncSetAttribute(k_bj_factor<CS, THREADS>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       (int)(gj_smem_floats(kMaxBlock, 8) * sizeof(float)));
  if (e != cudaSuccess) return e;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(CS * count);
  cfg.blockDim = dim3(threads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = CS;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = CS > 1 ? 1 : 0;
  const float floor = g_pivot_floor > 0.f ? g_pivot_floor : kPivotFloor;
  e = cudaLaunchKernelEx(&cfg, k_bj_factor<CS, THREADS>, g, kind, alpha, list, off, blocks, floor, fallbacks, T);
  note_launches(1);
  return e;
}

}  // namespace

void set_bj_pivot_floor(double floor) { g_pivot_floor = floor > 0.0 ? (float)floor : 0.f; }

cudaError_t bj_setup(const Geo& g, int kind, double alpha, const int* body_start_host, long long* off_dev,
                     int* list_dev, bj_t* blocks, int* fallbacks, cudaStream_t s) {
  // Bodies by kernel: one CTA (nb <= 128), clusters of four (<= 448) and eight (<= 640) CTAs.
  // Few bodies take larger clusters, and one launch: four of nb = 128 45 us in clusters of
  // four against 70 in single CTAs; nb = 236, 286, 482, 482 254 us in one launch of
  // clusters of eight against 158 + 254 in two.
  int large = 0, small = 0, min_nb = kMaxBlock;
  for (int i = 0; i < g.N; ++i) {
    const int nb = (body_start_host[i + 1] - body_start_host[i]) * (kind + 1);
    large += nb > kMaxSingle && nb <= kMaxBlock;
    small += nb <= kMaxSingle;
    if (nb <= kMaxSingle) min_nb = std::min(min_nb, nb);
  }
  const int sms = device_sms();
  const int max4 = 8 * large <= sms ? kMaxSingle : kMaxBlock4;
  const int kCs[3] = {4 * small <= sms && min_nb >= kMinCluster ? 4 : 1, 4, 8};
  std::vector<long long> off(g.N + 1, 0);
  std::vector<int> lists[3];
  int max_nb[3] = {0, 0, 0};
  size_t smem[3] = {0, 0, 0};
  for (int i = 0; i < g.N; ++i) {
    const int nb = (body_start_host[i + 1] - body_start_host[i]) * (kind + 1);
    off[i + 1] = off[i] + (nb <= kMaxBlock ? (long long)nb * nb : 0);
    const int c = nb <= kMaxSingle ? 0 : nb <= max4 ? 1 : nb <= kMaxBlock ? 2 : -1;
    if (c < 0) continue;
    lists[c].push_back(i);
    max_nb[c] = std::max(max_nb[c], nb);
    smem[c] = std::max(smem[c], gj_smem_floats(nb, kCs[c]) * sizeof(float));
  }
  std::vector<int> all;
  for (const auto& l : lists) all.insert(all.end(), l.begin(), l.end());
  cudaError_t e = cudaMemcpyAsync(off_dev, off.data(), off.size() * sizeof(long long), cudaMemcpyHostToDevice, s);
  if (e != cudaSuccess) return e;
  e = cudaMemsetAsync(fallbacks, 0, sizeof(int), s);
  if (e != cudaSuccess) return e;
  if (!all.empty()) {
    e = cudaMemcpyAsync(list_dev, all.data(), all.size() * sizeof(int), cudaMemcpyHostToDevice, s);
    if (e != cudaSuccess) return e;
  }
  size_t at = 0;
  for (int c = 0; c < 3; ++c) {
    const int count = (int)lists[c].size();
    if (count == 0) continue;
    const int* l = list_dev + at;
    const auto launch = kCs[c] == 1                 ? launch_factor<1, 288>
                        : kCs[c] == 8               ? launch_factor<8, 352>
                        : gj_rows(max_nb[c]) <= 128 ? launch_factor<4, 160>
                                                    : launch_factor<4, 480>;
    e = launch(g, kind, alpha, l, count, max_nb[c], smem[c], off_dev, blocks, fallbacks, s);
    if (e != cudaSuccess) return e;
    at += count;
  }
  // the host vectors must outlive the asynchronous copies
  return cudaStreamSynchronize(s);
}

namespace {
// CTAs of k_bj_apply64: a body's rows of 32, and where a body is larger than the blocks,
// which its CTAs copy in strides, so many that the bodies fill the SMs twice.
// (By the largest body's rows, one of 20,000 unknowns among 3,000 of 16 made 1.9 million, all but
// 7,000 of them empty, and one of 2.1 million no valid grid.)
dim3 apply64_grid(const Geo& g, int max_nb) {
  const int rows = (std::min(max_nb, kMaxBlock) + kRows64 - 1) / kRows64;
  if (max_nb <= kMaxBlock) return dim3(g.N, rows);
  return dim3(g.N, std::max(rows, std::min((max_nb + kBA - 1) / kBA, 2 * device_sms() / g.N)));
}
}  // namespace

cudaError_t bj_apply(const Geo& g, int kind, const long long* off_dev, const bj_t* blocks, VecRef v, double* z,
                     const int* stop, int max_nb, cudaStream_t s, bool f64) {
  const size_t nv = (size_t)std::min(max_nb, kMaxBlock);
  if (f64) {  // (callers pass a plain vector)
    k_bj_apply64<false><<<apply64_grid(g, max_nb), kBA, nv * sizeof(double), s>>>(g, kind, off_dev, blocks, v.base, z,
                                                                                  nullptr, 0, nullptr, stop);
  } else {
    const dim3 grid(g.N, (max_nb + kApplyRows - 1) / kApplyRows);
    k_bj_apply<<<grid, kBA, nv * sizeof(float), s>>>(g, kind, off_dev, blocks, v, z, stop);
  }
  note_launches(1);
  return cudaGetLastError();
}

cudaError_t bj_normalize_apply64(const Geo& g, int kind, const long long* off_dev, const bj_t* blocks, const double* w,
                                 double* z, double* V, long long ld, const KState* st, int max_nb, cudaStream_t s) {
  const size_t nv = (size_t)std::min(max_nb, kMaxBlock);
  k_bj_apply64<true><<<apply64_grid(g, max_nb), kBA, nv * sizeof(double), s>>>(g, kind, off_dev, blocks, w, z, V, ld,
                                                                               st, &st->stop);
  note_launches(1);
  return cudaGetLastError();
}

}  // namespace bie

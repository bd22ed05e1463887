// Nystrom pair sums of the paper's second-kind operators and their epilogue.
//
// Laplace (Section 3.4, operator K with the TARGET normal):
//   (K mu)_a = -(1/2pi) sum_{b != a} w_b mu_b (r . n_a) / |r|^2,   r = x_a - x_b
// Stokes (Section 4.3, operator K built from the stresslet T_ijk = -(1/pi) r_i r_j r_k/|r|^4):
//   (K mu)_a = -(1/pi) sum_{b != a} w_b r (r . mu_b)(r . n_a) / |r|^4
//
// Layout of the work: a block owns B*T targets (T per thread, strided by B so
// loads coalesce) and one contiguous split of the sources; sources stream
// through shared memory in tiles.  The splits write partial sums
// partial[s][a] that the epilogue adds in a fixed order (deterministic), in
// FP64, together with the diagonal limit, 1/2 I and the completion L.
//
// FP32 variant: positions are held as hi/lo float pairs so that, for a source
// tile close to the target block, dx = (xa_hi - xb_hi) + (xa_lo - xb_lo) is
// exact to FP32 rounding of dx itself even for neighbouring nodes far from the
// origin (the near-pair cancellation in r . n_a would otherwise lose digits).
// Tiles far from the block (gap at least both boxes' half-diagonals) use plain
// FP32 coordinates relative to the block centre: 4 fewer instructions a pair.
// The reciprocal is the hardware rcp.approx.f32; tile sums enter
// TwoSum-compensated FP32 accumulators.  The per-pair arithmetic (FP32 near
// pairs and float-float pairs) is shared with the FMM near field.
#include <algorithm>
#include <array>
#include <map>
#include <mutex>
#include <vector>

#include "bie_internal.cuh"
#include "pair_math.cuh"
#include "reduce.cuh"

namespace bie {

namespace {

// Source range of a target block [tbase, tend): all nodes, or in a batch the
// nodes of the problems its targets belong to (straddle: more than one); the
// block's split blockIdx.y of it, `chunk` sources long.  In a batch the range
// is cut into chunks of the planned length, so a block of a small problem has
// fewer busy splits than one of a large problem (the others are empty and
// write zero partials); a range longer than all splits together (a block
// straddling problems) is cut into gridDim.y equal parts.
struct SrcRange {
  int j0, j1;
  bool straddle;
};

template <bool BATCH>
__device__ __forceinline__ SrcRange src_range(const Geo& g, int tbase, int tend, const PairPlan& p) {
  SrcRange r;
  if (!BATCH) {
    const int s = blockIdx.y;
    r.j0 = s < p.S1 ? s * p.chunk : p.S1 * p.chunk + (s - p.S1) * p.chunk2;
    r.j1 = min(g.M, r.j0 + (s < p.S1 ? p.chunk : p.chunk2));
    r.straddle = false;
    return r;
  }
  const int chunk = p.chunk;
  const int2 p0 = g.prange[g.body_of[tbase]], p1 = g.prange[g.body_of[tend - 1]];
  const int len = p1.y - p0.x;
  const int ch = max(chunk, (len + (int)gridDim.y - 1) / (int)gridDim.y);
  r.j0 = min(p1.y, p0.x + (int)blockIdx.y * ch);
  r.j1 = min(p1.y, r.j0 + ch);
  r.straddle = p0.x != p1.x;
  return r;
}

// Batched GMRES: have all problems of the target block [tbase, tend) stopped?
// (block-uniform)  Such a block writes zero partials: its problems' next
// Krylov vectors are not used.
__device__ __forceinline__ bool block_stopped(const Geo& g, int tbase, int tend) {
  if (!g.ps) return false;
  const int j = *g.jstep;
  const int p0 = g.bprob[g.body_of[tbase]], p1 = g.bprob[g.body_of[tend - 1]];
  for (int p = p0; p <= p1; ++p)
    if (g.ps[p].stop_j > j) return false;
  return true;
}

template <int KIND>
__device__ __forceinline__ void zero_partials(int tbase, int tend, int M, double* __restrict__ partial) {
  for (int a = tbase + threadIdx.x; a < tend; a += blockDim.x) {
    if (KIND == 0) {
      partial[(long long)blockIdx.y * M + a] = 0.0;
    } else {
      partial[((long long)blockIdx.y * M + a) * 2] = 0.0;
      partial[((long long)blockIdx.y * M + a) * 2 + 1] = 0.0;
    }
  }
}

// Does source node b belong to target a's problem (batched solves)?
__device__ __forceinline__ bool same_problem(const Geo& g, int a, int b) {
  if (a >= g.M) return true;
  const int2 r = g.prange[g.body_of[a]];
  return b >= r.x && b < r.y;
}

// End of the tile starting at source jt: at most `want`, cut at the end of
// jt's problem (a tile must not mix problems).
template <bool BATCH>
__device__ __forceinline__ int tile_len(const Geo& g, int jt, int want) {
  if (!BATCH) return want;
  return min(want, g.prange[g.body_of[jt]].y - jt);
}

// ------------------------------------------------------------------ FP64 ----
constexpr int kB64 = 128, kT64 = 2, kTile64 = 128;

template <int KIND, bool BATCH>
__global__ void __launch_bounds__(kB64) k_pair64(Geo g, VecRef vr, const double* __restrict__ sscale,
                                                 PairPlan pp, double* __restrict__ partial,
                                                 const int* __restrict__ stop) {
  if (stop && *stop) return;
  __shared__ double sx[kTile64], sy[kTile64], sq1[kTile64], sq2[kTile64];
  const double* __restrict__ v = vr.ptr();
  const int M = g.M;
  const int tbase = blockIdx.x * kB64 * kT64;
  if (BATCH && block_stopped(g, tbase, min(M, tbase + kB64 * kT64))) {
    zero_partials<KIND>(tbase, min(M, tbase + kB64 * kT64), M, partial);
    return;
  }
  const SrcRange sr = src_range<BATCH>(g, tbase, min(M, tbase + kB64 * kT64), pp);
  const int j0 = sr.j0, j1 = sr.j1;
  double tx[kT64], ty[kT64], tnx[kT64], tny[kT64], ax[kT64], ay[kT64];
  int ta[kT64];
#pragma unroll
  for (int k = 0; k < kT64; ++k) {
    const int a = tbase + threadIdx.x + k * kB64;
    ta[k] = a;
    const bool in = a < M;
    tx[k] = in ? g.x[a] : 0.0;
    ty[k] = in ? g.y[a] : 0.0;
    tnx[k] = in ? g.nx[a] : 0.0;
    tny[k] = in ? g.ny[a] : 0.0;
    ax[k] = 0.0;
    ay[k] = 0.0;
  }
  for (int jt = j0; jt < j1; jt += kTile64) {
    __syncthreads();
    for (int l = threadIdx.x; l < kTile64; l += kB64) {
      const int b = jt + l;
      if (b < j1) {
        sx[l] = g.x[b];
        sy[l] = g.y[b];
        if (KIND == 0) {
          sq1[l] = sscale[b] * v[b];
        } else {
          sq1[l] = sscale[b] * v[2 * b];
          sq2[l] = sscale[b] * v[2 * b + 1];
        }
      }
    }
    __syncthreads();
    const int nt = min(kTile64, j1 - jt);
    for (int l = 0; l < nt; ++l) {
      const double px = sx[l], py = sy[l], q1 = sq1[l];
      const double q2 = KIND == 0 ? 0.0 : sq2[l];
      const int b = jt + l;
#pragma unroll
      for (int k = 0; k < kT64; ++k) {
        const double dx = tx[k] - px, dy = ty[k] - py;
        const double r2 = dx * dx + dy * dy;
        const bool skip = ta[k] == b || (BATCH && sr.straddle && !same_problem(g, ta[k], b));
        // Batches of small problems: most pairs of a block that spans several of them are
        // masked, and a warp with none of its own leaves out the FP64 work.  16 problems of
        // 48 Stokes nodes: 165 us with the branch, 258 without (186 by division, which the
        // compiler had put behind one).
        if (BATCH && skip) continue;
        if (KIND == 0) {
          const double s = skip ? 0.0 : q1 * rcp64(r2);
          ax[k] += dx * s;
          ay[k] += dy * s;
        } else {
          const double rq = dx * q1 + dy * q2;
          const double rn = dx * tnx[k] + dy * tny[k];
          const double y = rcp64(r2);
          const double c = skip ? 0.0 : (rq * rn) * (y * y);
          ax[k] += c * dx;
          ay[k] += c * dy;
        }
      }
    }
  }
#pragma unroll
  for (int k = 0; k < kT64; ++k) {
    const int a = ta[k];
    if (a < M) {
      if (KIND == 0)
        partial[(long long)blockIdx.y * M + a] = tnx[k] * ax[k] + tny[k] * ay[k];
      else {
        partial[((long long)blockIdx.y * M + a) * 2] = ax[k];
        partial[((long long)blockIdx.y * M + a) * 2 + 1] = ay[k];
      }
    }
  }
}

// ------------------------------------------------------------------ FP32 ----
constexpr int kB32 = 64, kT32 = 4, kTile32 = 256;

// Near tiles (sources whose bounding box is close to the target block's):
// exact differences from the hi/lo coordinates, reloaded here so that they
// are not live across the far tiles.
template <int KIND, bool DIAG>
__device__ __forceinline__ void tile_near(const float4* __restrict__ pf, const float4* __restrict__ sp,
                                          const float2* __restrict__ sq, int nt, int jt, int a0, int M,
                                          const float* tnx, const float* tny, float* ax, float* ay) {
  float txh[kT32], tyh[kT32], txl[kT32], tyl[kT32];
#pragma unroll
  for (int k = 0; k < kT32; ++k) {
    const int a = a0 + k * kB32;
    const float4 p = a < M ? pf[a] : make_float4(0.f, 0.f, 0.f, 0.f);
    txh[k] = p.x;
    tyh[k] = p.y;
    txl[k] = p.z;
    tyl[k] = p.w;
  }
#pragma unroll 2
  for (int l = 0; l < nt; ++l) {
    const float4 p = sp[l];
    const float2 q = sq[l];
#pragma unroll
    for (int k = 0; k < kT32; ++k) {
      float cx, cy;
      f32_pair<KIND>(txh[k], tyh[k], txl[k], tyl[k], tnx[k], tny[k], p, q.x, q.y, cx, cy);
      if (DIAG && a0 + k * kB32 == jt + l) cx = cy = 0.0f;  // the self pair (r = 0)
      ax[k] += cx;
      ay[k] += cy;
    }
  }
}

// Far tiles: plain FP32 coordinates relative to the target block's centre.
// Their rounding (|x'| 2^-24 with |x'| at most ~3 |r| for far pairs) is
// below 2e-7 of each term.  The two lanes of the packed FP32x2 instructions
// hold two sources for the same target, read as one 16-byte pair
// (-x'_l, -x'_l+1, -y'_l, -y'_l+1), so that D = T + (-P) = r.  On GB300 the
// FMA pipe retires 128 FP32 lanes a clock per SM whether packed or not, so
// packing halves the issue slots, not the pipe cycles; the loop costs 7 FP32
// lane operations and one MUFU reciprocal a pair.  (Sharing one MUFU operation
// between two reciprocals, 1/a = b rcp(ab), costs 1.5 more FP32 operations a
// pair and measured slower.)
template <int KIND>
__device__ __forceinline__ void tile_far2(const float4* __restrict__ sp2, const float4* __restrict__ sq2, int np,
                                          const float2* TX, const float2* TY, const float2* NX, const float2* NY,
                                          float2* AX, float2* AY) {
#pragma unroll(KIND == 0 ? 4 : 2)
  for (int l = 0; l < np; ++l) {
    const float4 p = sp2[l];
    const float2 px = make_float2(p.x, p.y), py = make_float2(p.z, p.w);
    float2 q1, q2;
    if (KIND == 0) {
      q1 = reinterpret_cast<const float2*>(sq2)[l];
    } else {
      const float4 q = sq2[l];
      q1 = make_float2(q.x, q.y);
      q2 = make_float2(q.z, q.w);
    }
#pragma unroll
    for (int k = 0; k < kT32; ++k) {
      const float2 dx = __fadd2_rn(TX[k], px);
      const float2 dy = __fadd2_rn(TY[k], py);
      const float2 r2 = __ffma2_rn(dx, dx, __fmul2_rn(dy, dy));
      const float2 inv = make_float2(rcp_approx(r2.x), rcp_approx(r2.y));
      if (KIND == 0) {
        const float2 sc = __fmul2_rn(q1, inv);
        AX[k] = __ffma2_rn(dx, sc, AX[k]);
        AY[k] = __ffma2_rn(dy, sc, AY[k]);
      } else {
        const float2 rq = __ffma2_rn(dx, q1, __fmul2_rn(dy, q2));
        const float2 rn = __ffma2_rn(dx, NX[k], __fmul2_rn(dy, NY[k]));
        const float2 c = __fmul2_rn(__fmul2_rn(rq, rn), __fmul2_rn(inv, inv));
        AX[k] = __ffma2_rn(c, dx, AX[k]);
        AY[k] = __ffma2_rn(c, dy, AY[k]);
      }
    }
  }
}

// s + e += t with the rounding error of the leading sum kept (TwoSum)
__device__ __forceinline__ void comp_add(float& s, float& e, float t) {
  const float u = s + t;
  const float bb = u - s;
  e += (s - (u - bb)) + (t - bb);
  s = u;
}

// Union of the bounding boxes of bodies [b0, b1].
__device__ __forceinline__ float4 body_range_box(const float4* __restrict__ bbox, int b0, int b1) {
  float4 u = bbox[b0];
  for (int i = b0 + 1; i <= b1; ++i) {
    const float4 b = bbox[i];
    u.x = fminf(u.x, b.x);
    u.y = fminf(u.y, b.y);
    u.z = fmaxf(u.z, b.z);
    u.w = fmaxf(u.w, b.w);
  }
  return u;
}

// FP32 source strengths q_b = sscale_b v_b (two per node for Stokes), once per
// operator application: every target block of k_pair32 reads them.
template <int KIND>
__global__ void k_src32(Geo g, VecRef vr, const double* __restrict__ sscale, const int* __restrict__ stop) {
  if (stop && *stop) return;
  const double* __restrict__ v = vr.ptr();
  for (int b = blockIdx.x * blockDim.x + threadIdx.x; b < g.M; b += gridDim.x * blockDim.x) {
    if (KIND == 0)
      g.qf[b] = (float)(sscale[b] * v[b]);
    else
      reinterpret_cast<float2*>(g.qf)[b] =
          make_float2((float)(sscale[b] * v[2 * b]), (float)(sscale[b] * v[2 * b + 1]));
  }
}

template <int KIND, bool BATCH>
__global__ void __launch_bounds__(kB32, KIND == 0 ? 12 : 10) k_pair32(Geo g, VecRef vr, const double* __restrict__ sscale,
                                                 PairPlan pp, double* __restrict__ partial,
                                                 const int* __restrict__ stop) {
  if (stop && *stop) return;
  __shared__ float4 sp[kTile32];  // near: (xh, yh, xl, yl)
  __shared__ float2 sq[kTile32];
  __shared__ float4 sp2[kTile32 / 2];  // far: source pairs (-x', -x', -y', -y')
  __shared__ float4 sq2[kTile32 / 2];  // far: (q1, q1', q2, q2'); Laplace packs (q, q') pairs
  const int M = g.M;
  const int tbase = blockIdx.x * kB32 * kT32;
  const int tend = min(M, tbase + kB32 * kT32);
  if (BATCH && block_stopped(g, tbase, tend)) {
    zero_partials<KIND>(tbase, tend, M, partial);
    return;
  }
  const SrcRange sr = src_range<BATCH>(g, tbase, tend, pp);
  const int j0 = sr.j0, j1 = sr.j1;
  // the target block's box, centre and half-diagonal
  const float4 tb = body_range_box(g.bbox, g.body_of[tbase], g.body_of[tend - 1]);
  const float cx = 0.5f * (tb.x + tb.z), cy = 0.5f * (tb.y + tb.w);
  const float et = 0.5f * sqrtf((tb.z - tb.x) * (tb.z - tb.x) + (tb.w - tb.y) * (tb.w - tb.y));
  const int a0 = tbase + threadIdx.x;
  float tnx[kT32], tny[kT32];
  float2 TX[kT32], TY[kT32], NX[kT32], NY[kT32];
  // compensated FP32 sums over the tiles: value sx + ex
  float sx[kT32], ex[kT32], sy[kT32], ey[kT32];
#pragma unroll
  for (int k = 0; k < kT32; ++k) {
    const int a = a0 + k * kB32;
    float4 p = make_float4(cx, cy, 0.f, 0.f);
    float2 n = make_float2(0.f, 0.f);
    if (a < M) {
      p = g.pf[a];
      if (KIND == 1) n = g.nf[a];
    }
    const float tlx = (p.x - cx) + p.z, tly = (p.y - cy) + p.w;
    tnx[k] = n.x;
    tny[k] = n.y;
    TX[k] = make_float2(tlx, tlx);
    TY[k] = make_float2(tly, tly);
    NX[k] = make_float2(n.x, n.x);
    NY[k] = make_float2(n.y, n.y);
    sx[k] = ex[k] = sy[k] = ey[k] = 0.f;
  }
  // source tiles never cross a body boundary, so a tile's box is its body's
  for (int jt = j0; jt < j1;) {
    const int sb = g.body_of[jt];
    const int nt = min(kTile32, min(j1, g.body_start[sb + 1]) - jt);
    // far when the boxes are at least both half-diagonals apart (block-uniform)
    const float4 sbx = g.bbox[sb];
    const float gx = fmaxf(0.f, fmaxf(sbx.x - tb.z, tb.x - sbx.z));
    const float gy = fmaxf(0.f, fmaxf(sbx.y - tb.w, tb.y - sbx.w));
    const float es = 0.5f * sqrtf((sbx.z - sbx.x) * (sbx.z - sbx.x) + (sbx.w - sbx.y) * (sbx.w - sbx.y));
    const float gap2 = gx * gx + gy * gy;
    const float need = fmaxf(et, es);
    const bool far = gap2 > 0.f && gap2 >= need * need;
    // far tiles are padded to an even count with a zero-strength copy of the last source
    const int ntl = far ? (nt + 1) & ~1 : nt;
    __syncthreads();
    for (int l = threadIdx.x; l < ntl; l += kB32) {
      const int b = jt + min(l, nt - 1);
      const float4 p = g.pf[b];
      float q1 = 0.f, q2 = 0.f;
      if (l < nt) {
        if (KIND == 0) {
          q1 = g.qf[b];
        } else {
          const float2 qq = reinterpret_cast<const float2*>(g.qf)[b];
          q1 = qq.x;
          q2 = qq.y;
        }
      }
      if (far) {
        float* pp = reinterpret_cast<float*>(&sp2[l >> 1]);
        pp[l & 1] = -((p.x - cx) + p.z);
        pp[2 + (l & 1)] = -((p.y - cy) + p.w);
        if (KIND == 0) {
          reinterpret_cast<float*>(sq2)[l] = q1;
        } else {
          float* qq = reinterpret_cast<float*>(&sq2[l >> 1]);
          qq[l & 1] = q1;
          qq[2 + (l & 1)] = q2;
        }
      } else {
        sp[l] = p;
        sq[l] = make_float2(q1, q2);
      }
    }
    __syncthreads();
    float ax[kT32], ay[kT32];
    if (far) {
      float2 AX[kT32], AY[kT32];
#pragma unroll
      for (int k = 0; k < kT32; ++k) AX[k] = AY[k] = make_float2(0.f, 0.f);
      tile_far2<KIND>(sp2, sq2, ntl >> 1, TX, TY, NX, NY, AX, AY);
#pragma unroll
      for (int k = 0; k < kT32; ++k) {
        ax[k] = AX[k].x + AX[k].y;
        ay[k] = AY[k].x + AY[k].y;
      }
    } else {
#pragma unroll
      for (int k = 0; k < kT32; ++k) ax[k] = ay[k] = 0.f;
      if ((jt < tend) && (jt + nt > tbase))
        tile_near<KIND, true>(g.pf, sp, sq, nt, jt, a0, M, tnx, tny, ax, ay);
      else
        tile_near<KIND, false>(g.pf, sp, sq, nt, jt, a0, M, tnx, tny, ax, ay);
    }
    if (BATCH) {
      // batched solves: a tile counts only for its own problem's targets (a block
      // may straddle two problems)
#pragma unroll
      for (int k = 0; k < kT32; ++k)
        if (!same_problem(g, a0 + k * kB32, jt)) ax[k] = ay[k] = 0.f;
    }
#pragma unroll
    for (int k = 0; k < kT32; ++k) {
      comp_add(sx[k], ex[k], ax[k]);
      comp_add(sy[k], ey[k], ay[k]);
    }
    jt += nt;
  }
#pragma unroll
  for (int k = 0; k < kT32; ++k) {
    const int a = a0 + k * kB32;
    if (a < M) {
      if (KIND == 0) {
        // n_a . (sx + ex, sy + ey) in float-float: the normal's hi/lo split,
        // error-free products, one TwoSum (no FP64 pipe per target and block)
        const float4 n = g.nff[a];
        float p1, e1, p2, e2, h, l;
        ff_mul(n.x, n.y, sx[k], ex[k], p1, e1);
        ff_mul(n.z, n.w, sy[k], ey[k], p2, e2);
        two_sum(p1, p2, h, l);
        reinterpret_cast<float2*>(partial)[(long long)blockIdx.y * M + a] = make_float2(h, l + (e1 + e2));
      } else {
        // (sx + ex, sy + ey) as two float-float pairs: no FP64 pipe in the kernel
        float hx, lx, hy, ly;
        two_sum(sx[k], ex[k], hx, lx);
        two_sum(sy[k], ey[k], hy, ly);
        reinterpret_cast<float4*>(partial)[(long long)blockIdx.y * M + a] = make_float4(hx, lx, hy, ly);
      }
    }
  }
}

// ------------------------------------------------------- symmetric FP32 ----
// FP32 pair sums with r, |r|^2 and the reciprocal used for both directions of a
// pair.  The M nodes are cut into tiles of TS = 2H blockDim consecutive nodes; one
// CTA takes one unordered pair of tiles (A = tile i, B = tile j, i <= j) and
// writes the contribution of B's sources to A's targets into partial[j][A] and
// that of A's sources to B's targets into partial[i][B]: every (source tile,
// target tile) slot is written exactly once, and the epilogue adds the S = tiles
// slots of a target in a fixed order (deterministic).
//
// With r = x_a - x_b, w = 1/|r|^2 and s = r w: Laplace target a gains q_b s and
// target b gains -q_a s (10 FP32 lane operations and one MUFU reciprocal for two
// directed pairs; the directed kernel: 7 and one for one pair); Stokes a gains
// s (r . q_b)(s . n_a) and b gains -s (r . q_a)(s . n_b) (20 operations, against
// 13 for one).  Each lane holds 2H A targets in registers (packed two by two);
// B's sources sit in shared memory and are visited 32 at a time on a diagonal
// schedule (lane l takes source (l + k) mod 32 of the group at step k), and the
// accumulator of B's source travels with it from lane to lane by a warp
// shuffle, so no two lanes ever add into the same place.
//
// Coordinates: a group of 32 sources is far from tile A when its box (its bodies')
// is far from every body of A; differences are then taken in plain FP32 relative
// to the centre of the group's box, in which sources and targets are at most a
// few |r| from the origin (rounding <= 3 x 2^-24 |r|), else from the exact hi/lo
// coordinates (four operations more).  The test is per body, not on the tiles'
// boxes: tiles of several bodies in no spatial order (a random suspension) stay
// far.  (Laplace tiles whose whole boxes are far skip the per-group work: 1.5% at
// 100 bodies of 256 nodes.)  A tile with itself runs the directed near pass.
// Stokes sums are kept error-free over chunks of kSymChunk sources.
//
// Bound by the issue of FP32 instructions (two thirds of the pipe; without the
// shuffles, or without MUFU, 5% faster).  Measured, pair sum alone, directed ->
// symmetric: Stokes 400 bodies of 128 nodes in random order 1,684 -> 915 us
// (2.87e12 pairs/s), 200 of 90..165 nodes 424 -> 266 us, 64 of 128 nodes 56 -> 43
// us; Laplace with the tiles' boxes -> per body: 400 of 128 1,026 -> 558 us, 200
// of 90..165 291 -> 165 us, 100 of 256 156 -> 154 us.
constexpr int kTS = kB32 * kT32;  // 256 nodes a tile of the symmetric Laplace plan
constexpr int kSymChunk = 64;

__device__ __forceinline__ void tri_decode(int t, int& i, int& j) {
  int jj = (int)((sqrtf(8.0f * (float)t + 1.0f) - 1.0f) * 0.5f);  // then corrected exactly
  while ((long long)(jj + 1) * (jj + 2) / 2 <= t) ++jj;
  while ((long long)jj * (jj + 1) / 2 > t) --jj;
  j = jj;
  i = t - jj * (jj + 1) / 2;
}

// Is box b far from box a (gap at least both half-diagonals)?
__device__ __forceinline__ bool boxes_far(float4 a, float4 b) {
  const float gx = fmaxf(0.f, fmaxf(b.x - a.z, a.x - b.z));
  const float gy = fmaxf(0.f, fmaxf(b.y - a.w, a.y - b.w));
  const float ea = 0.5f * sqrtf((a.z - a.x) * (a.z - a.x) + (a.w - a.y) * (a.w - a.y));
  const float eb = 0.5f * sqrtf((b.z - b.x) * (b.z - b.x) + (b.w - b.y) * (b.w - b.y));
  const float gap2 = gx * gx + gy * gy;
  const float need = fmaxf(ea, eb);
  return gap2 > 0.f && gap2 >= need * need;
}

// The slot entry of target a from its sum (ax + ex, ay + ey): Laplace n_a . sum in
// float-float (the normal's hi/lo split), stored as the float pair (h, l);
// Stokes both components as float pairs.  No FP64 pipe in the kernel.
template <int KIND>
__device__ __forceinline__ void write_slot(const Geo& g, int a, int slot, float ax, float ex, float ay, float ey,
                                           double* __restrict__ partial) {
  if (KIND == 0) {
    const float4 n = g.nff[a];
    float p1, e1, p2, e2, h, l;
    ff_mul(n.x, n.y, ax, ex, p1, e1);
    ff_mul(n.z, n.w, ay, ey, p2, e2);
    two_sum(p1, p2, h, l);
    reinterpret_cast<float2*>(partial)[(long long)slot * g.M + a] = make_float2(h, l + (e1 + e2));
  } else {
    reinterpret_cast<float4*>(partial)[(long long)slot * g.M + a] = make_float4(ax, ex, ay, ey);
  }
}

// One group of 32 sources (shared-memory entries sX[0..32)) against this lane's
// four targets: their sums into AX, AY (targets 0, 1 and 2, 3 packed) and the
// sources' sums, returned at the lane that holds the source.  FAR: TX, TY and
// the sources are relative to the group's centre; else TXL, TYL are the low
// parts and sL the sources'.  Sources are stored negated.
template <int KIND, bool FAR, int H>
__device__ __forceinline__ float2 sym_group(const float4* __restrict__ sX, const float2* __restrict__ sL,
                                            const float2* __restrict__ sN, const float2* TX, const float2* TY,
                                            const float2* TXL, const float2* TYL, const float2* Q1, const float2* Q2,
                                            const float2* NX, const float2* NY, float2* AX, float2* AY) {
  const int lane = threadIdx.x & 31;
  float bx = 0.f, by = 0.f;  // accumulator of the source this lane holds (travels)
#pragma unroll(FAR ? 8 : 4)
  for (int k = 0; k < 32; ++k) {
    const int l = (lane + k) & 31;
    const float4 src = sX[l];
    const float2 sx = make_float2(src.x, src.x), sy = make_float2(src.y, src.y);
    const float2 q1 = make_float2(src.z, src.z), q2 = make_float2(src.w, src.w);
    float2 lo = make_float2(0.f, 0.f), nb = lo;
    if (!FAR) lo = sL[l];
    if (KIND == 1) nb = sN[l];
    float2 ux, uy;
#pragma unroll
    for (int h = 0; h < H; ++h) {
      float2 dx = __fadd2_rn(TX[h], sx), dy = __fadd2_rn(TY[h], sy);
      if (!FAR) {
        dx = __fadd2_rn(dx, __fadd2_rn(TXL[h], make_float2(lo.x, lo.x)));
        dy = __fadd2_rn(dy, __fadd2_rn(TYL[h], make_float2(lo.y, lo.y)));
      }
      const float2 r2 = __ffma2_rn(dx, dx, __fmul2_rn(dy, dy));
      const float2 w = make_float2(rcp_approx(r2.x), rcp_approx(r2.y));
      if (KIND == 0) {
        const float2 sb = __fmul2_rn(q1, w), sa = __fmul2_rn(Q1[h], w);
        AX[h] = __ffma2_rn(dx, sb, AX[h]);
        AY[h] = __ffma2_rn(dy, sb, AY[h]);
        ux = h == 0 ? __fmul2_rn(dx, sa) : __ffma2_rn(dx, sa, ux);
        uy = h == 0 ? __fmul2_rn(dy, sa) : __ffma2_rn(dy, sa, uy);
      } else {
        const float2 ex = __fmul2_rn(dx, w), ey = __fmul2_rn(dy, w);
        const float2 ca = __fmul2_rn(__ffma2_rn(dx, q1, __fmul2_rn(dy, q2)),
                                     __ffma2_rn(ex, NX[h], __fmul2_rn(ey, NY[h])));
        const float2 cb = __fmul2_rn(__ffma2_rn(dx, Q1[h], __fmul2_rn(dy, Q2[h])),
                                     __ffma2_rn(ex, make_float2(nb.x, nb.x), __fmul2_rn(ey, make_float2(nb.y, nb.y))));
        AX[h] = __ffma2_rn(ca, ex, AX[h]);
        AY[h] = __ffma2_rn(ca, ey, AY[h]);
        ux = h == 0 ? __fmul2_rn(cb, ex) : __ffma2_rn(cb, ex, ux);
        uy = h == 0 ? __fmul2_rn(cb, ey) : __ffma2_rn(cb, ey, uy);
      }
    }
    bx -= ux.x + ux.y;
    by -= uy.x + uy.y;
    // hand the accumulator to the lane that takes this source next
    bx = __shfl_sync(0xffffffffu, bx, (lane + 1) & 31);
    by = __shfl_sync(0xffffffffu, by, (lane + 1) & 31);
  }
  return make_float2(bx, by);  // back at its own lane
}

// Adds the targets' sums of a chunk of sources to their error-free sums over
// the chunks (shared memory, each thread its own entries) and clears them.
template <int H>
__device__ __forceinline__ void sym_flush(float4* __restrict__ sAcc, float2* AX, float2* AY) {
  const int t = threadIdx.x, B = blockDim.x;
#pragma unroll
  for (int k = 0; k < 2 * H; ++k) {
    float4 c = sAcc[t + k * B];
    comp_add(c.x, c.y, k & 1 ? AX[k >> 1].y : AX[k >> 1].x);
    comp_add(c.z, c.w, k & 1 ? AY[k >> 1].y : AY[k >> 1].x);
    sAcc[t + k * B] = c;
  }
#pragma unroll
  for (int h = 0; h < H; ++h) AX[h] = AY[h] = make_float2(0.f, 0.f);
}

// The sources' sums [warps][TS] of tile B (nodes below end) into their slots: the warps
// in order, error-free.
template <int KIND>
__device__ __forceinline__ void sym_write_sources(const Geo& g, int B0, int TS, int end, int slot,
                                                  const float2* __restrict__ accB, double* __restrict__ partial) {
  __syncthreads();
  for (int l = threadIdx.x; l < TS; l += blockDim.x) {
    const int b = B0 + l;
    if (b >= end) continue;
    float2 u = accB[l];
    float ex = 0.f, ey = 0.f;
    for (int w = 1; w < (int)blockDim.x / 32; ++w) {
      const float2 v = accB[w * TS + l];
      comp_add(u.x, ex, v.x);
      comp_add(u.y, ey, v.y);
    }
    write_slot<KIND>(g, b, slot, u.x, ex, u.y, ey, partial);
  }
}

// Shared memory of one CTA, bytes a node: far and near positions with the
// strengths, near low parts, the Stokes normal and the Stokes targets' sums, the
// warps' accumulators; per group its box and far flag.
template <int KIND, int H>
__host__ __device__ constexpr size_t sym32_smem(int threads) {
  const size_t TS = 2 * H * (size_t)threads;
  return TS * (16 + 16 + 8 + (KIND == 1 ? 8 + 16 : 0)) + (threads / 32) * TS * 8 + TS / 32 * (16 + 4);
}

// BATCH: problem blockIdx.y, its nodes cut into tiles by themselves (so no pair crosses
// problems, and no mask is needed); a problem has as many slots as tiles.
template <int KIND, int H, bool BATCH>
__global__ void __launch_bounds__(64, KIND == 0 ? 10 : (H == 2 ? 8 : 6)) k_pair32s(Geo g, double* __restrict__ partial,
                                                                      const int* __restrict__ stop) {
  if (stop && *stop) return;
  extern __shared__ __align__(16) unsigned char sm_raw[];
  const int B = blockDim.x, TS = 2 * H * B, G = TS / 32;
  int n0 = 0, M = g.M;  // the nodes [n0, M)
  if (BATCH) {
    const int2 r = g.prange[g.pbody[blockIdx.y]];
    n0 = r.x;
    M = r.y;
  }
  float4* sF = reinterpret_cast<float4*>(sm_raw);  // far: (-x', -y', q1, q2)
  float4* sH = sF + TS;                            // near: (-x_hi, -y_hi, q1, q2)
  float4* sBox = sH + TS;                          // [G]
  float4* sAcc = sBox + G;                         // Stokes: [TS] (sx, ex, sy, ey) of the targets
  float2* sL = reinterpret_cast<float2*>(sAcc + (KIND == 1 ? TS : 0));  // near: (-x_lo, -y_lo)
  float2* accB = sL + TS;                          // [warps][TS]
  float2* sN = accB + (B / 32) * TS;               // Stokes normals
  int* sFar = reinterpret_cast<int*>(sN + (KIND == 1 ? TS : 0));  // [G]
  int ti, tj;
  tri_decode(blockIdx.x, ti, tj);
  const int A0 = n0 + ti * TS, B0 = n0 + tj * TS;
  const int t = threadIdx.x;
  if (BATCH) {
    if (B0 >= M) return;  // fewer tiles than the largest problem
    if (g.ps && g.ps[blockIdx.y].stop_j <= *g.jstep) {  // stopped: zero partials, as the directed kernel
      for (int l = t; l < TS; l += B) {
        if (A0 + l < M) write_slot<KIND>(g, A0 + l, tj, 0.f, 0.f, 0.f, 0.f, partial);
        if (ti != tj && B0 + l < M) write_slot<KIND>(g, B0 + l, ti, 0.f, 0.f, 0.f, 0.f, partial);
      }
      return;
    }
  }
  if constexpr (KIND == 0) {
    // Laplace: tiles whose whole boxes are far (bodies of whole tiles, or in
    // spatial order) need one centre: no per-group targets
    const float4 boxA = body_range_box(g.bbox, g.body_of[A0], g.body_of[min(A0 + TS, M) - 1]);
    const float4 boxB = body_range_box(g.bbox, g.body_of[B0], g.body_of[min(B0 + TS, M) - 1]);
    if (ti != tj && boxes_far(boxA, boxB)) {
      const float cx = 0.5f * (boxA.x + boxA.z), cy = 0.5f * (boxA.y + boxA.w);
      for (int l = t; l < TS; l += B) {
        const int b = min(B0 + l, M - 1);  // past the end: the last node with zero strength
        const float4 p = g.pf[b];
        sF[l] = make_float4(-((p.x - cx) + p.z), -((p.y - cy) + p.w), B0 + l < M ? g.qf[b] : 0.f, 0.f);
      }
      float2 TX[H], TY[H], Q[H], AX[H], AY[H];
#pragma unroll
      for (int h = 0; h < H; ++h) {
        const int a0 = A0 + t + 2 * h * B, a1 = a0 + B;
        const float4 p0 = g.pf[a0], p1 = g.pf[a1];
        TX[h] = make_float2((p0.x - cx) + p0.z, (p1.x - cx) + p1.z);
        TY[h] = make_float2((p0.y - cy) + p0.w, (p1.y - cy) + p1.w);
        Q[h] = make_float2(g.qf[a0], g.qf[a1]);
        AX[h] = AY[h] = make_float2(0.f, 0.f);
      }
      __syncthreads();
      for (int o = 0; o < TS; o += 32)
        accB[(t >> 5) * TS + o + (t & 31)] =
            sym_group<0, true, H>(sF + o, sL, sN, TX, TY, TX, TY, Q, Q, Q, Q, AX, AY);
#pragma unroll
      for (int k = 0; k < 2 * H; ++k)
        write_slot<0>(g, A0 + t + k * B, tj, k & 1 ? AX[k >> 1].y : AX[k >> 1].x, 0.f,
                      k & 1 ? AY[k >> 1].y : AY[k >> 1].x, 0.f, partial);
      sym_write_sources<0>(g, B0, TS, M, ti, accB, partial);
      return;
    }
  }
  for (int gi = t; gi < G; gi += B) {
    const int f = min(B0 + 32 * gi, M - 1), e = min(f + 31, M - 1);
    const float4 gb = body_range_box(g.bbox, g.body_of[f], g.body_of[e]);
    bool far = ti != tj;
    if (far) {
      const int i1 = g.body_of[A0 + TS - 1];
      for (int i = g.body_of[A0]; i <= i1; ++i) far = far && boxes_far(g.bbox[i], gb);
    }
    sBox[gi] = gb;
    sFar[gi] = far;
  }
  __syncthreads();
  for (int l = t; l < TS; l += B) {
    const int b = min(B0 + l, M - 1);  // past the end: the last node with zero strength
    const float4 p = g.pf[b];
    const float4 bb = sBox[l >> 5];
    float q1 = 0.f, q2 = 0.f;
    if (B0 + l < M) {
      if (KIND == 0) {
        q1 = g.qf[b];
      } else {
        const float2 q = reinterpret_cast<const float2*>(g.qf)[b];
        q1 = q.x;
        q2 = q.y;
      }
    }
    const float cx = 0.5f * (bb.x + bb.z), cy = 0.5f * (bb.y + bb.w);
    sF[l] = make_float4(-((p.x - cx) + p.z), -((p.y - cy) + p.w), q1, q2);
    sH[l] = make_float4(-p.x, -p.y, q1, q2);
    sL[l] = make_float2(-p.z, -p.w);
    if (KIND == 1) {
      sN[l] = g.nf[b];
      sAcc[l] = make_float4(0.f, 0.f, 0.f, 0.f);
    }
  }
  float2 Q1[H], Q2[H], NX[H], NY[H], AX[H], AY[H];
  float4 P[KIND == 0 ? 2 * H : 1];  // Laplace: the targets' positions, held
#pragma unroll
  for (int h = 0; h < H; ++h) {
    const int a0 = min(A0 + t + 2 * h * B, M - 1), a1 = min(A0 + t + (2 * h + 1) * B, M - 1);
    if (KIND == 0) {
      P[2 * h] = g.pf[a0];
      P[2 * h + 1] = g.pf[a1];
      Q1[h] = make_float2(g.qf[a0], g.qf[a1]);
      Q2[h] = NX[h] = NY[h] = make_float2(0.f, 0.f);  // unused
    } else {
      const float2 q0 = reinterpret_cast<const float2*>(g.qf)[a0], q1 = reinterpret_cast<const float2*>(g.qf)[a1];
      const float2 n0 = g.nf[a0], n1 = g.nf[a1];
      Q1[h] = make_float2(q0.x, q1.x);
      Q2[h] = make_float2(q0.y, q1.y);
      NX[h] = make_float2(n0.x, n1.x);
      NY[h] = make_float2(n0.y, n1.y);
    }
    AX[h] = AY[h] = make_float2(0.f, 0.f);
  }
  auto target = [&](int k) { return KIND == 0 ? P[KIND == 0 ? k : 0] : g.pf[min(A0 + t + k * B, M - 1)]; };
  __syncthreads();
  if (ti == tj) {
    // directed pass of the tile with itself (exact differences, r = 0 excluded)
    const int nt = min(TS, M - B0);
    float4 T[2 * H];
#pragma unroll
    for (int k = 0; k < 2 * H; ++k) T[k] = target(k);
    for (int l0 = 0; l0 < nt; l0 += kSymChunk) {
      const int l1 = min(nt, l0 + kSymChunk);
#pragma unroll 2
      for (int l = l0; l < l1; ++l) {
        const float4 src = sH[l];
        const float2 lo = sL[l];
        float c[2 * H][2];
#pragma unroll
        for (int k = 0; k < 2 * H; ++k) {
          const float2 n2 = NX[k >> 1], m2 = NY[k >> 1];
          f32_pair<KIND>(T[k].x, T[k].y, T[k].z, T[k].w, k & 1 ? n2.y : n2.x, k & 1 ? m2.y : m2.x,
                         make_float4(-src.x, -src.y, -lo.x, -lo.y), src.z, src.w, c[k][0], c[k][1]);
          if (t + k * B == l) c[k][0] = c[k][1] = 0.f;
        }
#pragma unroll
        for (int h = 0; h < H; ++h) {
          AX[h] = __fadd2_rn(AX[h], make_float2(c[2 * h][0], c[2 * h + 1][0]));
          AY[h] = __fadd2_rn(AY[h], make_float2(c[2 * h][1], c[2 * h + 1][1]));
        }
      }
      if (KIND == 1) sym_flush<H>(sAcc, AX, AY);
    }
  } else {
    const int lane = t & 31, warp = t >> 5;
    for (int gi = 0; gi < G; ++gi) {
      const int o = 32 * gi;
      float2 TX[H], TY[H], u;
      if (sFar[gi]) {
        const float4 bb = sBox[gi];
        const float cx = 0.5f * (bb.x + bb.z), cy = 0.5f * (bb.y + bb.w);
#pragma unroll
        for (int h = 0; h < H; ++h) {
          const float4 p0 = target(2 * h), p1 = target(2 * h + 1);
          TX[h] = make_float2((p0.x - cx) + p0.z, (p1.x - cx) + p1.z);
          TY[h] = make_float2((p0.y - cy) + p0.w, (p1.y - cy) + p1.w);
        }
        u = sym_group<KIND, true, H>(sF + o, sL + o, sN + o, TX, TY, TX, TY, Q1, Q2, NX, NY, AX, AY);
      } else {
        float2 TXL[H], TYL[H];
#pragma unroll
        for (int h = 0; h < H; ++h) {
          const float4 p0 = target(2 * h), p1 = target(2 * h + 1);
          TX[h] = make_float2(p0.x, p1.x);
          TY[h] = make_float2(p0.y, p1.y);
          TXL[h] = make_float2(p0.z, p1.z);
          TYL[h] = make_float2(p0.w, p1.w);
        }
        u = sym_group<KIND, false, H>(sH + o, sL + o, sN + o, TX, TY, TXL, TYL, Q1, Q2, NX, NY, AX, AY);
      }
      accB[warp * TS + o + lane] = u;
      if (KIND == 1 && gi % (kSymChunk / 32) == kSymChunk / 32 - 1) sym_flush<H>(sAcc, AX, AY);
    }
  }
#pragma unroll
  for (int k = 0; k < 2 * H; ++k) {
    const int a = A0 + t + k * B;
    if (a >= M) continue;
    if (KIND == 0) {
      write_slot<0>(g, a, tj, k & 1 ? AX[k >> 1].y : AX[k >> 1].x, 0.f, k & 1 ? AY[k >> 1].y : AY[k >> 1].x, 0.f, partial);
    } else {
      const float4 c = sAcc[t + k * B];
      write_slot<1>(g, a, tj, c.x, c.y, c.z, c.w, partial);
    }
  }
  if (ti != tj) sym_write_sources<KIND>(g, B0, TS, M, ti, accB, partial);
}

// Tiles of 128 nodes (one warp, four targets a lane), 256 (two warps) and, Stokes,
// 192 (one warp, six targets).
template <int KIND, bool BATCH>
void launch_pair32s(const Geo& g, const PairPlan& p, double* partial, const int* stop, cudaStream_t s) {
  const dim3 grid((unsigned)((long long)p.S * (p.S + 1) / 2), BATCH ? g.nprob : 1);  // S tiles (the largest problem's)
  const int tile = p.sym;
  if constexpr (KIND == 1) {
    if (tile == 192) {
      k_pair32s<1, 3, BATCH><<<grid, 32, sym32_smem<1, 3>(32), s>>>(g, partial, stop);
      return;
    }
  }
  k_pair32s<KIND, 2, BATCH><<<grid, tile / 4, sym32_smem<KIND, 2>(tile / 4), s>>>(g, partial, stop);
}

// -------------------------------------------------------- symmetric FP64 ----
// The FP64 pair sum on unordered pairs of tiles of TS = blockDim nodes, one CTA
// a pair: r, |r|^2 and the reciprocal serve both directions.  GB300's FP64 pipe
// bounds it (two lanes a clock per SM): Laplace 13 FP64 operations for two
// directed pairs (the directed kernel: 10 for one, about 16 when it divided),
// Stokes 24 (16, about 21).  Measured (GB300, whole launch): Laplace M = 25,600
// 16.6 ms divided, 12.1 ms directed with rcp64, 7.5 ms symmetric (8.7e10
// pairs/s, 90% of the pipe); Stokes M = 12,630 6.7, 4.65, 3.43 ms.
// A lane holds one target of tile A (two a lane measured the same); the sources
// of tile B sit in shared memory, visited on the diagonal schedule of
// k_pair32s, the source's accumulator travelling by shuffle.  Warp w starts
// at source group w (32 sources) and the warps meet at a barrier after each
// group, so that a group's accumulators are added to by one warp at a time, in
// a fixed order.  Partials as k_pair32s: slot j of tile A's nodes, slot i of
// tile B's; a tile with itself runs the directed pass.  Nodes past M in the
// last tile stand at its first node with zero strength.
template <int KIND>
__host__ __device__ constexpr int sym64_vals() { return KIND == 0 ? 5 : 8; }  // doubles a node in shared memory

template <int KIND>
__global__ void __launch_bounds__(256) k_pair64s(Geo g, VecRef vr, const double* __restrict__ sscale,
                                                 double* __restrict__ partial, const int* __restrict__ stop) {
  if (stop && *stop) return;
  extern __shared__ __align__(16) double sm64[];
  const double* __restrict__ v = vr.ptr();
  const int M = g.M, TS = blockDim.x, t = threadIdx.x;
  double *sx = sm64, *sy = sx + TS, *sq1 = sy + TS, *sbx = sq1 + TS, *sby = sbx + TS;
  double *sq2 = sby + TS, *snx = sq2 + TS, *sny = snx + TS;  // Stokes
  int ti, tj;
  tri_decode(blockIdx.x, ti, tj);
  const int A0 = ti * TS, B0 = tj * TS;
  {
    const int b = B0 + t < M ? B0 + t : B0;
    const double s = B0 + t < M ? sscale[b] : 0.0;
    sx[t] = g.x[b];
    sy[t] = g.y[b];
    sbx[t] = sby[t] = 0.0;
    if (KIND == 0) {
      sq1[t] = s * v[b];
    } else {
      sq1[t] = s * v[2 * b];
      sq2[t] = s * v[2 * b + 1];
      snx[t] = g.nx[b];
      sny[t] = g.ny[b];
    }
  }
  const int a = min(A0 + t, M - 1);
  const double tx = g.x[a], ty = g.y[a], tnx = g.nx[a], tny = g.ny[a], ts = sscale[a];
  const double tq1 = ts * v[KIND == 0 ? a : 2 * a], tq2 = KIND == 0 ? 0.0 : ts * v[2 * a + 1];
  double ax = 0.0, ay = 0.0;
  __syncthreads();
  if (ti == tj) {
    const int nt = min(TS, M - B0);
#pragma unroll 4
    for (int l = 0; l < nt; ++l) {
      const double q1 = sq1[l], dx = tx - sx[l], dy = ty - sy[l];
      const double y = rcp64(dx * dx + dy * dy);
      if (KIND == 0) {
        const double s = t == l ? 0.0 : q1 * y;
        ax += dx * s;
        ay += dy * s;
      } else {
        const double c = t == l ? 0.0 : ((dx * q1 + dy * sq2[l]) * (dx * tnx + dy * tny)) * (y * y);
        ax += c * dx;
        ay += c * dy;
      }
    }
  } else {
    const int lane = t & 31, warp = t >> 5, G = TS / 32;
    for (int g0 = 0; g0 < G; ++g0) {
      const int r0 = 32 * (g0 + warp < G ? g0 + warp : g0 + warp - G);
      double bx = 0.0, by = 0.0;  // accumulator of the source this lane holds (travels)
#pragma unroll 4
      for (int k = 0; k < 32; ++k) {
        const int l = r0 + ((lane + k) & 31);
        const double q1 = sq1[l], dx = tx - sx[l], dy = ty - sy[l];
        const double y = rcp64(dx * dx + dy * dy);
        if (KIND == 0) {
          const double sb = q1 * y, sa = tq1 * y;
          ax += dx * sb;
          ay += dy * sb;
          bx -= dx * sa;  // the source gains -q_a r/|r|^2
          by -= dy * sa;
        } else {
          const double y2 = y * y;
          const double ca = ((dx * q1 + dy * sq2[l]) * (dx * tnx + dy * tny)) * y2;
          const double cb = ((dx * tq1 + dy * tq2) * (dx * snx[l] + dy * sny[l])) * y2;
          ax += ca * dx;
          ay += ca * dy;
          bx -= cb * dx;  // r, r . q_a and r . n_b all change sign
          by -= cb * dy;
        }
        bx = __shfl_sync(0xffffffffu, bx, (lane + 1) & 31);
        by = __shfl_sync(0xffffffffu, by, (lane + 1) & 31);
      }
      sbx[r0 + lane] += bx;  // back at its own lane: source r0 + lane
      sby[r0 + lane] += by;
      __syncthreads();
    }
    const int b = B0 + t;
    if (b < M) {
      if (KIND == 0)
        partial[(long long)ti * M + b] = g.nx[b] * sbx[t] + g.ny[b] * sby[t];
      else
        reinterpret_cast<double2*>(partial)[(long long)ti * M + b] = make_double2(sbx[t], sby[t]);
    }
  }
  if (A0 + t < M) {
    if (KIND == 0)
      partial[(long long)tj * M + a] = tnx * ax + tny * ay;
    else
      reinterpret_cast<double2*>(partial)[(long long)tj * M + a] = make_double2(ax, ay);
  }
}

// ------------------------------------------------------------ float-float ----
// Pair sums in float-float ("double-single") arithmetic on the FP32 pipes, for
// residuals that must be accurate far beyond FP32: every quantity is an
// unevaluated sum h + l of two floats (about 48 significant bits).
//  - positions: exact split x = h + m + l (quanta from g.qscale, computed
//    once per geometry), so that dx = (h_a - h_b) + (m_a - m_b) + (l_a - l_b)
//    has exact leading parts for every pair, near or far;
//  - products: error-free a*b = p + fma(a, b, -p);
//  - reciprocal: MUFU rcp.approx seed y0 refined by one Newton step in
//    float-float, 1/r2 = y0 + y0 (1 - r2 y0);
//  - sums: TwoSum (Knuth) for the leading parts, trailing parts added, within
//    a tile and across tiles (no FP64 in the loop: GB300's FP64 pipe is slow).
constexpr int kBF = 64, kTF = 4, kTileF = 256;

template <int KIND, bool DIAG>
__device__ __forceinline__ void tile_ff(const float4* __restrict__ sa, const float2* __restrict__ sb,
                                        const float4* __restrict__ sq, int nt, int jt, int a0, const FFTarget* t,
                                        float* axh, float* axl, float* ayh, float* ayl) {
  for (int l = 0; l < nt; ++l) {
    const float4 pa = sa[l];  // (xh, xm, yh, ym)
    const float2 pb = sb[l];  // (xl, yl)
    const float4 q = sq[l];   // (q1h, q1l, q2h, q2l)
#pragma unroll
    for (int k = 0; k < kTF; ++k) {
      float cxh, cxl, cyh, cyl;
      ff_pair<KIND>(t[k], pa, pb, q, cxh, cxl, cyh, cyl);
      if (DIAG && a0 + k * kBF == jt + l) cxh = cxl = cyh = cyl = 0.0f;  // the self pair
      ff_acc(axh[k], axl[k], cxh, cxl);
      ff_acc(ayh[k], ayl[k], cyh, cyl);
    }
  }
}

template <int KIND, bool BATCH>
__global__ void __launch_bounds__(kBF) k_pair_ff(Geo g, VecRef vr, const double* __restrict__ sscale, PairPlan pp,
                                                 double* __restrict__ partial, const int* __restrict__ stop) {
  if (stop && *stop) return;
  __shared__ float4 sa[kTileF];
  __shared__ float2 sb[kTileF];
  __shared__ float4 sq[kTileF];
  const double* __restrict__ v = vr.ptr();
  const int M = g.M;
  const int tbase = blockIdx.x * kBF * kTF;
  const int tend = min(M, tbase + kBF * kTF);
  if (BATCH && block_stopped(g, tbase, tend)) {
    zero_partials<KIND>(tbase, tend, M, partial);
    return;
  }
  const int a0 = tbase + threadIdx.x;
  const SrcRange sr = src_range<BATCH>(g, tbase, tend, pp);
  const int j0 = sr.j0, j1 = sr.j1;
  FFTarget t[kTF];
  // float-float sums over the tiles
  float sxh[kTF], sxl[kTF], syh[kTF], syl[kTF];
#pragma unroll
  for (int k = 0; k < kTF; ++k) {
    const int a = a0 + k * kBF;
    const float4 p = a < M ? g.xff[a] : make_float4(0.f, 0.f, 0.f, 0.f);
    const float2 pl = a < M ? g.xfl[a] : make_float2(0.f, 0.f);
    t[k].xh = p.x;
    t[k].xm = p.y;
    t[k].yh = p.z;
    t[k].ym = p.w;
    t[k].xl = pl.x;
    t[k].yl = pl.y;
    t[k].n = (KIND == 1 && a < M) ? g.nff[a] : make_float4(0.f, 0.f, 0.f, 0.f);
    sxh[k] = sxl[k] = syh[k] = syl[k] = 0.f;
  }
  for (int jt = j0; jt < j1;) {
    const int nt = tile_len<BATCH>(g, jt, min(kTileF, j1 - jt));
    __syncthreads();
    for (int l = threadIdx.x; l < nt; l += kBF) {
      const int b = jt + l;
      sa[l] = g.xff[b];
      sb[l] = g.xfl[b];
      const double q1 = KIND == 0 ? sscale[b] * v[b] : sscale[b] * v[2 * b];
      const double q2 = KIND == 0 ? 0.0 : sscale[b] * v[2 * b + 1];
      const float q1h = (float)q1, q2h = (float)q2;
      sq[l] = make_float4(q1h, (float)(q1 - (double)q1h), q2h, (float)(q2 - (double)q2h));
    }
    __syncthreads();
    float axh[kTF], axl[kTF], ayh[kTF], ayl[kTF];
#pragma unroll
    for (int k = 0; k < kTF; ++k) axh[k] = axl[k] = ayh[k] = ayl[k] = 0.f;
    if ((jt < tend) && (jt + nt > tbase))
      tile_ff<KIND, true>(sa, sb, sq, nt, jt, a0, t, axh, axl, ayh, ayl);
    else
      tile_ff<KIND, false>(sa, sb, sq, nt, jt, a0, t, axh, axl, ayh, ayl);
    if (BATCH) {
#pragma unroll
      for (int k = 0; k < kTF; ++k)
        if (!same_problem(g, a0 + k * kBF, jt)) axh[k] = axl[k] = ayh[k] = ayl[k] = 0.f;
    }
#pragma unroll
    for (int k = 0; k < kTF; ++k) {
      ff_acc(sxh[k], sxl[k], axh[k], axl[k]);
      ff_acc(syh[k], syl[k], ayh[k], ayl[k]);
    }
    jt += nt;
  }
#pragma unroll
  for (int k = 0; k < kTF; ++k) {
    const int a = a0 + k * kBF;
    const double dax = (double)sxh[k] + (double)sxl[k], day = (double)syh[k] + (double)syl[k];
    if (a < M) {
      if (KIND == 0)
        partial[(long long)blockIdx.y * M + a] = g.nx[a] * dax + g.ny[a] * day;
      else {
        partial[((long long)blockIdx.y * M + a) * 2] = dax;
        partial[((long long)blockIdx.y * M + a) * 2 + 1] = day;
      }
    }
  }
}

// ------------------------------------------------- symmetric float-float ----
// The float-float Laplace pair sum on unordered pairs of 256-node tiles, each
// reciprocal (MUFU seed + one float-float Newton step) and each difference and
// |r|^2 serving both directions: target a gains q_b r w, target b gains
// -q_a r w.  Float-float positions give exact leading differences for every
// pair, so every pair of different tiles takes the symmetric loop; a tile
// with itself (the self pairs) runs the directed float-float pass.  The
// source's float-float accumulator travels between lanes by warp shuffle on
// the diagonal schedule of k_pair32s.  Partials: FP64, one slot per (source
// tile, target tile), projected on the target normal in FP64.
constexpr int kTFS = 2;                      // targets a lane
constexpr int kBFS = kTileF / kTFS;          // 128 threads a CTA

// Packed forms of the float-float helpers: the two halves of a float2 are two
// independent values, each rounded exactly as the scalar form rounds it.
__device__ __forceinline__ float2 neg2f(float2 a) { return make_float2(-a.x, -a.y); }
__device__ __forceinline__ void ff_mul2(float2 ah, float2 al, float2 bh, float2 bl, float2& p, float2& e) {
  p = __fmul2_rn(ah, bh);
  e = __ffma2_rn(ah, bh, neg2f(p));
  e = __ffma2_rn(ah, bl, __ffma2_rn(al, bh, e));
}
__device__ __forceinline__ void ff_acc2(float2& sh, float2& sl, float2 th, float2 tl) {
  const float2 u = __fadd2_rn(sh, th);
  const float2 bb = __fadd2_rn(u, neg2f(sh));
  const float2 e = __fadd2_rn(__fadd2_rn(sh, neg2f(__fadd2_rn(u, neg2f(bb)))), __fadd2_rn(th, neg2f(bb)));
  sh = u;
  sl = __fadd2_rn(sl, __fadd2_rn(e, tl));
}

__device__ __forceinline__ void ff_write_projected(const Geo& g, int a, int slot, float xh, float xl, float yh,
                                                   float yl, double* __restrict__ partial) {
  const double dax = (double)xh + (double)xl, day = (double)yh + (double)yl;
  partial[(long long)slot * g.M + a] = g.nx[a] * dax + g.ny[a] * day;
}

__global__ void __launch_bounds__(kBFS, 6) k_pair_ffs(Geo g, int ntile, double* __restrict__ partial,
                                                     const double* __restrict__ sscale, VecRef vr,
                                                     const int* __restrict__ stop) {
  if (stop && *stop) return;
  __shared__ float4 sA[kTileF];  // (xh, xm, yh, ym)
  __shared__ float4 sC[kTileF];  // (xl, yl, qh, ql)
  __shared__ float4 accB[kBFS / 32][kTileF];  // per warp: the sources' (xh, xl, yh, yl)
  const double* __restrict__ v = vr.ptr();
  const int M = g.M;
  int ti, tj;
  tri_decode(blockIdx.x, ti, tj);
  const int A0 = ti * kTileF, B0 = tj * kTileF;
  if (ti == tj) {
    // directed float-float pass of the tile with itself (excludes r = 0)
    const int a1 = min(M, A0 + kTileF), nt = a1 - A0;
    for (int l = threadIdx.x; l < nt; l += kBFS) {
      const int b = A0 + l;
      const float4 xa = g.xff[b];
      const float2 xl = g.xfl[b];
      const double q = sscale[b] * v[b];
      const float qh = (float)q;
      sA[l] = xa;
      sC[l] = make_float4(xl.x, xl.y, qh, (float)(q - (double)qh));
    }
    __syncthreads();
    for (int m = 0; m < kTFS; ++m) {
      const int a = A0 + threadIdx.x + m * kBFS;
      if (a >= M) continue;
      FFTarget t;
      const float4 p = g.xff[a];
      const float2 pl = g.xfl[a];
      t.xh = p.x; t.xm = p.y; t.yh = p.z; t.ym = p.w; t.xl = pl.x; t.yl = pl.y;
      t.n = make_float4(0.f, 0.f, 0.f, 0.f);
      float axh = 0.f, axl = 0.f, ayh = 0.f, ayl = 0.f;
      for (int l = 0; l < nt; ++l) {
        if (A0 + l == a) continue;
        const float4 c = sC[l];
        float cxh, cxl, cyh, cyl;
        ff_pair<0>(t, sA[l], make_float2(c.x, c.y), make_float4(c.z, c.w, 0.f, 0.f), cxh, cxl, cyh, cyl);
        ff_acc(axh, axl, cxh, cxl);
        ff_acc(ayh, ayl, cyh, cyl);
      }
      ff_write_projected(g, a, ti, axh, axl, ayh, ayl, partial);
    }
    return;
  }
  // sources of tile B, negated (so that a difference is a packed add);
  // padding far from everything with zero strength
  for (int l = threadIdx.x; l < kTileF; l += kBFS) {
    const int b = B0 + l;
    float4 xa = make_float4(-1e15f, 0.f, -1e15f, 0.f), c = make_float4(0.f, 0.f, 0.f, 0.f);
    if (b < M) {
      const float4 x = g.xff[b];
      const float2 xl = g.xfl[b];
      const double q = sscale[b] * v[b];
      const float qh = (float)q;
      xa = make_float4(-x.x, -x.y, -x.z, -x.w);
      c = make_float4(-xl.x, -xl.y, qh, (float)(q - (double)qh));
    }
    sA[l] = xa;
    sC[l] = c;
  }
  // the kTFS = 2 targets of tile A a lane, packed as the two halves of
  // FP32x2 operands (all of tile A is inside [0, M): ti < tj)
  static_assert(kTFS == 2, "two targets a lane, one packed pair");
  float2 TXH, TXM, TXL, TYH, TYM, TYL, QAH, QAL;
  {
    const int a0 = A0 + threadIdx.x, a1 = a0 + kBFS;
    const float4 p0 = g.xff[a0], p1 = g.xff[a1];
    const float2 l0 = g.xfl[a0], l1 = g.xfl[a1];
    TXH = make_float2(p0.x, p1.x);
    TXM = make_float2(p0.y, p1.y);
    TYH = make_float2(p0.z, p1.z);
    TYM = make_float2(p0.w, p1.w);
    TXL = make_float2(l0.x, l1.x);
    TYL = make_float2(l0.y, l1.y);
    const double q0 = sscale[a0] * v[a0], q1 = sscale[a1] * v[a1];
    const float h0 = (float)q0, h1 = (float)q1;
    QAH = make_float2(h0, h1);
    QAL = make_float2((float)(q0 - (double)h0), (float)(q1 - (double)h1));
  }
  float2 AXH = make_float2(0.f, 0.f), AXL = AXH, AYH = AXH, AYL = AXH;
  const float2 ONE = make_float2(1.f, 1.f), TWO = make_float2(2.f, 2.f);
  __syncthreads();
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  for (int r0 = 0; r0 < kTileF; r0 += 32) {
    float bxh = 0.f, bxl = 0.f, byh = 0.f, byl = 0.f;  // travels with its source
#pragma unroll 2
    for (int k = 0; k < 32; ++k) {
      const int l = r0 + ((lane + k) & 31);
      const float4 sa = sA[l], sc = sC[l];
      // float-float differences r = x_a - x_b from the exact splits (as ff_diff)
      const float2 d1x = __fadd2_rn(TXH, make_float2(sa.x, sa.x)), d2x = __fadd2_rn(TXM, make_float2(sa.y, sa.y));
      const float2 d1y = __fadd2_rn(TYH, make_float2(sa.z, sa.z)), d2y = __fadd2_rn(TYM, make_float2(sa.w, sa.w));
      const float2 DXH = __fadd2_rn(d1x, d2x), DYH = __fadd2_rn(d1y, d2y);
      const float2 DXL = __fadd2_rn(__fadd2_rn(d2x, neg2f(__fadd2_rn(DXH, neg2f(d1x)))),
                                    __fadd2_rn(TXL, make_float2(sc.x, sc.x)));
      const float2 DYL = __fadd2_rn(__fadd2_rn(d2y, neg2f(__fadd2_rn(DYH, neg2f(d1y)))),
                                    __fadd2_rn(TYL, make_float2(sc.y, sc.y)));
      // |r|^2 in float-float: error-free squares, an error-free sum of the two,
      // the cross terms, renormalised (as the directed pair)
      const float2 P1 = __fmul2_rn(DXH, DXH), P1E = __ffma2_rn(DXH, DXH, neg2f(P1));
      const float2 P2 = __fmul2_rn(DYH, DYH), P2E = __ffma2_rn(DYH, DYH, neg2f(P2));
      const float2 S = __fadd2_rn(P1, P2);
      const float2 BB = __fadd2_rn(S, neg2f(P1));
      const float2 SE = __fadd2_rn(__fadd2_rn(P1, neg2f(__fadd2_rn(S, neg2f(BB)))), __fadd2_rn(P2, neg2f(BB)));
      const float2 LO = __ffma2_rn(TWO, __ffma2_rn(DXH, DXL, __fmul2_rn(DYH, DYL)),
                                   __fadd2_rn(__fadd2_rn(SE, P1E), P2E));
      const float2 R2H = __fadd2_rn(S, LO);
      const float2 R2L = __fadd2_rn(LO, neg2f(__fadd2_rn(R2H, neg2f(S))));
      // 1/|r|^2: MUFU seed and one float-float Newton step
      const float2 Y0 = make_float2(rcp_approx(R2H.x), rcp_approx(R2H.y));
      const float2 EE = __ffma2_rn(neg2f(R2L), Y0, __ffma2_rn(neg2f(R2H), Y0, ONE));
      const float2 IL = __fmul2_rn(Y0, EE);
      // target a gains q_b r w
      float2 CH, CL, PH, PL;
      ff_mul2(make_float2(sc.z, sc.z), make_float2(sc.w, sc.w), Y0, IL, CH, CL);
      ff_mul2(CH, CL, DXH, DXL, PH, PL);
      ff_acc2(AXH, AXL, PH, PL);
      ff_mul2(CH, CL, DYH, DYL, PH, PL);
      ff_acc2(AYH, AYL, PH, PL);
      // the source gains -q_a r w (both targets' terms, in the order of the
      // scalar pass: target 0, then target 1)
      ff_mul2(QAH, QAL, Y0, IL, CH, CL);
      ff_mul2(CH, CL, DXH, DXL, PH, PL);
      ff_acc(bxh, bxl, -PH.x, -PL.x);
      ff_acc(bxh, bxl, -PH.y, -PL.y);
      ff_mul2(CH, CL, DYH, DYL, PH, PL);
      ff_acc(byh, byl, -PH.x, -PL.x);
      ff_acc(byh, byl, -PH.y, -PL.y);
      const int nxt = (lane + 1) & 31;
      bxh = __shfl_sync(0xffffffffu, bxh, nxt);
      bxl = __shfl_sync(0xffffffffu, bxl, nxt);
      byh = __shfl_sync(0xffffffffu, byh, nxt);
      byl = __shfl_sync(0xffffffffu, byl, nxt);
    }
    accB[warp][r0 + lane] = make_float4(bxh, bxl, byh, byl);
  }
  ff_write_projected(g, A0 + threadIdx.x, tj, AXH.x, AXL.x, AYH.x, AYL.x, partial);
  ff_write_projected(g, A0 + threadIdx.x + kBFS, tj, AXH.y, AXL.y, AYH.y, AYL.y, partial);
  __syncthreads();
  for (int l = threadIdx.x; l < kTileF; l += kBFS) {
    const int b = B0 + l;
    if (b >= M) continue;
    // the warps' sums in a fixed order
    float4 t = accB[0][l];
#pragma unroll
    for (int w = 1; w < kBFS / 32; ++w) {
      const float4 u = accB[w][l];
      ff_acc(t.x, t.y, u.x, u.y);
      ff_acc(t.z, t.w, u.z, u.w);
    }
    ff_write_projected(g, b, ti, t.x, t.y, t.z, t.w, partial);
  }
}

// --------------------------------------------------------------- epilogue ----
constexpr int kBE = 256;

// One block per body: completion moments, then per node
//   y = Kv (constant applied) + diagonal limit + [L]; out = sign (1/2 v + oscale y).
// (sh, sl) += (h, l) in float-float
__device__ __forceinline__ void ffadd(float& sh, float& sl, float h, float l) {
  float u, e;
  two_sum(sh, h, u, e);
  sh = u;
  sl += e + l;
}

template <int KIND, int B>
__global__ void __launch_bounds__(B) k_epilogue(Geo g, VecRef vr, const double* __restrict__ partial,
                                                  int S, int scaled, int with_L, double alpha, double sign,
                                                  VecRef outr, const int* __restrict__ stop, int pff) {
  if (stop && *stop) return;
  __shared__ double sh[B / 32];
  const double* __restrict__ v = vr.ptr();
  double* __restrict__ out = outr.ptr();
  const int M = g.M;
  const int i = blockIdx.x;
  const int a0 = g.body_start[i], a1 = g.body_start[i + 1];
  const double xc = g.xc[i], yc = g.yc[i];
  double m0 = 0.0, m1 = 0.0, m2 = 0.0;
  __shared__ double cfs[2];  // completion weights alpha/|Gamma_i|, alpha/W_i: one FP64 division each per block
  if (with_L && alpha > 0.0 && threadIdx.x == 0) {
    cfs[0] = alpha / g.len[i];
    cfs[1] = KIND == 1 ? alpha / g.W[i] : 1.0;
  }
  if (with_L) {
    for (int a = a0 + threadIdx.x; a < a1; a += B) {
      const double s = scaled ? g.sw[a] : g.w[a];
      if (KIND == 0) {
        m0 += s * v[a];
      } else {
        const double f1 = s * v[2 * a], f2 = s * v[2 * a + 1];
        m0 += f1;
        m1 += f2;
        m2 += -(g.y[a] - yc) * f1 + (g.x[a] - xc) * f2;
      }
    }
    m0 = block_sum<B>(m0, sh);
    if (KIND == 1) {
      m1 = block_sum<B>(m1, sh);
      m2 = block_sum<B>(m2, sh);
    }
    if (alpha > 0.0) {  // completion weighted per body: force part alpha/|Gamma_i|, torque part alpha/W_i
      const double cf = cfs[0];  // written before block_sum's barriers
      m0 *= cf;
      m1 *= cf;
      if (KIND == 1) m2 *= cfs[1];
    }
  }
  for (int a = a0 + threadIdx.x; a < a1; a += B) {
    const double os = scaled ? g.sw[a] : 1.0;
    const double wk = g.w[a] * g.kappa[a];
    if (KIND == 0) {
      double k;
      if (pff) {
        // float-float partials of the FP32 pair sums: two independent float-float
        // sums (loads in flight), added in a fixed order, converted once
        const float2* __restrict__ pf2 = reinterpret_cast<const float2*>(partial);
        float h0 = 0.f, l0 = 0.f, h1 = 0.f, l1 = 0.f;
        int s = 0;
        for (; s + 2 <= S; s += 2) {
          const float2 u = pf2[(long long)s * M + a], v = pf2[(long long)(s + 1) * M + a];
          ffadd(h0, l0, u.x, u.y);
          ffadd(h1, l1, v.x, v.y);
        }
        if (s < S) {
          const float2 u = pf2[(long long)s * M + a];
          ffadd(h0, l0, u.x, u.y);
        }
        ffadd(h0, l0, h1, l1);
        k = (double)h0 + (double)l0;
      } else {
        // four independent sums over the source splits (loads in flight), added in a fixed order
        double k0 = 0.0, k1 = 0.0, k2 = 0.0, k3 = 0.0;
        int s = 0;
        for (; s + 4 <= S; s += 4) {
          k0 += partial[(long long)s * M + a];
          k1 += partial[(long long)(s + 1) * M + a];
          k2 += partial[(long long)(s + 2) * M + a];
          k3 += partial[(long long)(s + 3) * M + a];
        }
        for (; s < S; ++s) k0 += partial[(long long)s * M + a];
        k = (k0 + k1) + (k2 + k3);
      }
      // os y with y = -k/2pi - wk mu/4pi + m0 and mu = v/os: the diagonal term
      // os wk mu/4pi = wk v/4pi needs no division
      out[a] = sign * (0.5 * v[a] + os * (m0 - kInv2Pi * k) - kInv4Pi * wk * v[a]);
    } else {
      double k1 = 0.0, k2 = 0.0;
      if (pff) {
        const float4* __restrict__ pf4 = reinterpret_cast<const float4*>(partial);
        float h1 = 0.f, l1 = 0.f, h2 = 0.f, l2 = 0.f;
        for (int s = 0; s < S; ++s) {
          const float4 u = pf4[(long long)s * M + a];
          ffadd(h1, l1, u.x, u.y);
          ffadd(h2, l2, u.z, u.w);
        }
        k1 = (double)h1 + (double)l1;
        k2 = (double)h2 + (double)l2;
      } else {
        double k1b = 0.0, k2b = 0.0;
        int s = 0;
        for (; s + 2 <= S; s += 2) {
          const double2 p0 = reinterpret_cast<const double2*>(partial)[(long long)s * M + a];
          const double2 p1 = reinterpret_cast<const double2*>(partial)[(long long)(s + 1) * M + a];
          k1 += p0.x;
          k2 += p0.y;
          k1b += p1.x;
          k2b += p1.y;
        }
        if (s < S) {
          const double2 p0 = reinterpret_cast<const double2*>(partial)[(long long)s * M + a];
          k1 += p0.x;
          k2 += p0.y;
        }
        k1 += k1b;
        k2 += k2b;
      }
      // os y with the diagonal term os dd t, dd = -wk (t . mu)/2pi and mu = v/os:
      // os dd = -wk (t . v)/2pi needs no division
      const double tx = -g.ny[a], ty = g.nx[a];
      const double v1 = v[2 * a], v2 = v[2 * a + 1];
      const double odd = -0.5 * kInvPi * wk * (tx * v1 + ty * v2);
      const double px = -(g.y[a] - yc), py = g.x[a] - xc;
      out[2 * a] = sign * (0.5 * v1 + os * (m0 + px * m2 - kInvPi * k1) + odd * tx);
      out[2 * a + 1] = sign * (0.5 * v2 + os * (m1 + py * m2 - kInvPi * k2) + odd * ty);
    }
  }
}

// The epilogue of the FP32 operator (the inner solves).  On GB300 most of
// k_epilogue's FP64-pipe time goes to the per-body completion moments and
// their block sums; here they run on the FP32 pipe in float-float (FP32
// products s v with their exact rounding errors, error-free sums), which
// keeps them accurate well beyond FP32 (the per-term roundings of s and v
// average out; no total is ever rounded to FP32), and the per-node output
// is k_epilogue's FP64 expression.  Fixed order throughout (deterministic).
// (h, l) += (bh, bl) in float-float
__device__ __forceinline__ void ff_add(float& h, float& l, float bh, float bl) {
  float s, e;
  two_sum(h, bh, s, e);
  e += l + bl;
  h = s + e;
  l = e - (h - s);
}

// (h, l) += a b with the product's rounding error
__device__ __forceinline__ void ff_add_prod(float& h, float& l, float a, float b) {
  const float p = a * b;
  ff_add(h, l, p, fmaf(a, b, -p));
}

template <int KIND, int B>
__global__ void __launch_bounds__(B) k_epilogue32(Geo g, VecRef vr, const double* __restrict__ partial, int S,
                                                    int scaled, int with_L, double alpha, double sign, VecRef outr,
                                                    const int* __restrict__ stop, int pff) {
  if (stop && *stop) return;
  // One FP64 instruction costs the (narrow) pipe the same with one lane as with 32: the
  // scalar work of a body, by one thread one after the other, was half of it.  Its two
  // or three values are lanes of the same instructions here, the quotients by rcp64.
  // 10,000 bodies of 64 nodes, Stokes: 55.6 -> 39.8 us.
  constexpr int NC = KIND == 0 ? 1 : 3;
  __shared__ float2 sh[NC][B / 32];
  __shared__ float cst[4];    // body centre split hi + lo
  __shared__ double mom[NC];  // completion moments, weighted
  const double* __restrict__ v = vr.ptr();
  double* __restrict__ out = outr.ptr();
  const int M = g.M;
  const int i = blockIdx.x;
  const int a0 = g.body_start[i], a1 = g.body_start[i + 1];
  const double xc = g.xc[i], yc = g.yc[i];
  double weight = 1.0;  // threads 0..NC-1: of the moment, from the body's length or W
  if (threadIdx.x < NC && with_L && alpha > 0.0) weight = threadIdx.x < 2 ? g.len[i] : g.W[i];
  if (KIND == 1 && threadIdx.x < 2) {
    const double c = threadIdx.x == 0 ? xc : yc;
    const float hi = (float)c;
    cst[threadIdx.x] = hi;
    cst[2 + threadIdx.x] = (float)(c - (double)hi);
  }
  if (threadIdx.x < NC) mom[threadIdx.x] = 0.0;
  __syncthreads();
  if (with_L) {
    float h[NC], l[NC];
#pragma unroll
    for (int q = 0; q < NC; ++q) h[q] = l[q] = 0.f;
    for (int a = a0 + threadIdx.x; a < a1; a += B) {
      const float2 wk = g.wkf[a];
      const float sc = scaled ? wk.x : wk.x * wk.x;
      if (KIND == 0) {
        ff_add_prod(h[0], l[0], sc, (float)v[a]);
      } else {
        const float4 P = g.pf[a];
        const float dx = (P.x - cst[0]) + (P.z - cst[2]), dy = (P.y - cst[1]) + (P.w - cst[3]);
        const float v1 = (float)v[2 * a], v2 = (float)v[2 * a + 1];
        ff_add_prod(h[0], l[0], sc, v1);
        ff_add_prod(h[NC / 2], l[NC / 2], sc, v2);
        ff_add_prod(h[NC - 1], l[NC - 1], -dy, v1 * sc);
        ff_add_prod(h[NC - 1], l[NC - 1], dx, v2 * sc);
      }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1)
#pragma unroll
      for (int q = 0; q < NC; ++q) {
        const float oh = __shfl_down_sync(0xffffffffu, h[q], o), ol = __shfl_down_sync(0xffffffffu, l[q], o);
        ff_add(h[q], l[q], oh, ol);
      }
    if ((threadIdx.x & 31) == 0)
#pragma unroll
      for (int q = 0; q < NC; ++q) sh[q][threadIdx.x >> 5] = make_float2(h[q], l[q]);
    __syncthreads();
    if (threadIdx.x < NC) {
      float th = sh[threadIdx.x][0].x, tl = sh[threadIdx.x][0].y;
#pragma unroll
      for (int k = 1; k < B / 32; ++k) ff_add(th, tl, sh[threadIdx.x][k].x, sh[threadIdx.x][k].y);
      const double m = (double)th + (double)tl;
      mom[threadIdx.x] = alpha > 0.0 ? m * (alpha * rcp64(weight)) : m;  // completion weighted per body
    }
    __syncthreads();
  }
  const double m0 = mom[0], m1 = mom[NC / 2], m2 = mom[NC - 1];
  for (int a = a0 + threadIdx.x; a < a1; a += B) {
    const double os = scaled ? g.sw[a] : 1.0;
    const double wk = g.w[a] * g.kappa[a];
    if (KIND == 0) {
      double k;
      if (pff) {
        const float2* __restrict__ pf2 = reinterpret_cast<const float2*>(partial);
        float h0 = 0.f, l0 = 0.f, h1 = 0.f, l1 = 0.f;
        int s = 0;
        for (; s + 2 <= S; s += 2) {
          const float2 u = pf2[(long long)s * M + a], w2 = pf2[(long long)(s + 1) * M + a];
          ffadd(h0, l0, u.x, u.y);
          ffadd(h1, l1, w2.x, w2.y);
        }
        if (s < S) {
          const float2 u = pf2[(long long)s * M + a];
          ffadd(h0, l0, u.x, u.y);
        }
        ffadd(h0, l0, h1, l1);
        k = (double)h0 + (double)l0;
      } else {
        k = partial[a];
        for (int s = 1; s < S; ++s) k += partial[(long long)s * M + a];
      }
      const double o = 0.5 * v[a] + os * (m0 - kInv2Pi * k) - kInv4Pi * wk * v[a];
      out[a] = sign == 1.0 ? o : sign * o;
    } else {
      double k1 = 0.0, k2 = 0.0;
      if (pff) {
        const float4* __restrict__ pf4 = reinterpret_cast<const float4*>(partial);
        float h1 = 0.f, l1 = 0.f, h2 = 0.f, l2 = 0.f;
        for (int s = 0; s < S; ++s) {
          const float4 u = pf4[(long long)s * M + a];
          ffadd(h1, l1, u.x, u.y);
          ffadd(h2, l2, u.z, u.w);
        }
        k1 = (double)h1 + (double)l1;
        k2 = (double)h2 + (double)l2;
      } else {
        const double2 p = reinterpret_cast<const double2*>(partial)[a];
        k1 = p.x;
        k2 = p.y;
        for (int s = 1; s < S; ++s) {
          const double2 p0 = reinterpret_cast<const double2*>(partial)[(long long)s * M + a];
          k1 += p0.x;
          k2 += p0.y;
        }
      }
      const double tx = -g.ny[a], ty = g.nx[a];
      const double v1 = v[2 * a], v2 = v[2 * a + 1];
      const double odd = -0.5 * kInvPi * wk * (tx * v1 + ty * v2);
      const double px = -(g.y[a] - yc), py = g.x[a] - xc;
      const double o1 = 0.5 * v1 + os * (m0 + px * m2 - kInvPi * k1) + odd * tx;
      const double o2 = 0.5 * v2 + os * (m1 + py * m2 - kInvPi * k2) + odd * ty;
      out[2 * a] = sign == 1.0 ? o1 : sign * o1;
      out[2 * a + 1] = sign == 1.0 ? o2 : sign * o2;
    }
  }
}

// Sum of the float-float partial slots of the FP32 pair sums, wide: a CTA
// takes 32 target entries x 8 slot groups; each thread adds slots g, g + 8, ...
// in float-float, the 8 group sums are combined in a fixed order
// (deterministic), and the total overwrites slot 0 as a double (the entry's
// own 8 bytes, after every thread has read it).  cw = float-float pairs per
// target entry (1 Laplace, 2 Stokes).
constexpr int kRT = 32, kRG = 8;

// tile > 0: the symmetric kernel over problems, each of whose entries has as many slots
// as its problem has tiles.
__global__ void __launch_bounds__(kRT * kRG) k_reduce_slots(Geo g, int tile, double* __restrict__ partial, int S,
                                                            long long n, const int* __restrict__ stop) {
  if (stop && *stop) return;
  __shared__ float sh[kRG][kRT], sl[kRG][kRT];
  const int tx = threadIdx.x % kRT, grp = threadIdx.x / kRT;
  const long long e = (long long)blockIdx.x * kRT + tx;  // a float-float entry
  const float2* __restrict__ pf2 = reinterpret_cast<const float2*>(partial);
  float h = 0.f, l = 0.f, h2 = 0.f, l2 = 0.f;
  if (e < n) {
    if (tile > 0) {
      const int2 r = g.prange[g.body_of[n == g.M ? e : e >> 1]];
      S = (r.y - r.x + tile - 1) / tile;
    }
    int s = grp;
    for (; s + kRG < S; s += 2 * kRG) {
      const float2 u = pf2[(long long)s * n + e], v = pf2[(long long)(s + kRG) * n + e];
      ffadd(h, l, u.x, u.y);
      ffadd(h2, l2, v.x, v.y);
    }
    if (s < S) {
      const float2 u = pf2[(long long)s * n + e];
      ffadd(h, l, u.x, u.y);
    }
    ffadd(h, l, h2, l2);
  }
  sh[grp][tx] = h;
  sl[grp][tx] = l;
  __syncthreads();
  if (grp == 0 && e < n) {
    float th = sh[0][tx], tl = sl[0][tx];
#pragma unroll
    for (int q = 1; q < kRG; ++q) ffadd(th, tl, sh[q][tx], sl[q][tx]);
    partial[e] = (double)th + (double)tl;
  }
}

// The same for FP64 partial slots (FP64 and float-float pair sums).
__global__ void __launch_bounds__(kRT * kRG) k_reduce_slots64(double* __restrict__ partial, int S, long long n,
                                                              const int* __restrict__ stop) {
  if (stop && *stop) return;
  __shared__ double sd[kRG][kRT];
  const int tx = threadIdx.x % kRT, grp = threadIdx.x / kRT;
  const long long e = (long long)blockIdx.x * kRT + tx;
  double a = 0.0, b = 0.0;
  if (e < n) {
    int s = grp;
    for (; s + kRG < S; s += 2 * kRG) {
      a += partial[(long long)s * n + e];
      b += partial[(long long)(s + kRG) * n + e];
    }
    if (s < S) a += partial[(long long)s * n + e];
  }
  sd[grp][tx] = a + b;
  __syncthreads();
  if (grp == 0 && e < n) {
    double t = sd[0][tx];
#pragma unroll
    for (int q = 1; q < kRG; ++q) t += sd[q][tx];
    partial[e] = t;
  }
}

// Right-hand side for a correction solved with the per-body weighted
// completion (weights c_i): for A e = g, the discrete Gauss identities (column
// sums of K equal -1/2 on the own body and 0 elsewhere, Sections 3.2 and 4.1)
// give the completion moments of e from g alone, L e = L~(g) with
// L~(g)_i = int_{Gamma_i} g / |Gamma_i| (and the torque moment over W_i), so
// A_c e = g - (I - C) L~(g).  Scaled vectors; one block per body.
template <int KIND>
__global__ void __launch_bounds__(kBE) k_consistent_rhs(Geo g, double alpha, const double* __restrict__ in,
                                                        double* __restrict__ out) {
  __shared__ double sh[kBE / 32];
  const int i = blockIdx.x;
  const int a0 = g.body_start[i], a1 = g.body_start[i + 1];
  const double xc = g.xc[i], yc = g.yc[i];
  double m0 = 0.0, m1 = 0.0, m2 = 0.0;
  for (int a = a0 + threadIdx.x; a < a1; a += kBE) {
    const double s = g.sw[a];
    if (KIND == 0) {
      m0 += s * in[a];
    } else {
      const double f1 = s * in[2 * a], f2 = s * in[2 * a + 1];
      m0 += f1;
      m1 += f2;
      m2 += -(g.y[a] - yc) * f1 + (g.x[a] - xc) * f2;
    }
  }
  m0 = block_sum<kBE>(m0, sh);
  if (KIND == 1) {
    m1 = block_sum<kBE>(m1, sh);
    m2 = block_sum<kBE>(m2, sh);
  }
  const double df = (1.0 - alpha / g.len[i]) / g.len[i];
  const double dt = KIND == 1 ? (1.0 - alpha / g.W[i]) / g.W[i] : 0.0;
  for (int a = a0 + threadIdx.x; a < a1; a += kBE) {
    const double s = g.sw[a];
    if (KIND == 0) {
      out[a] = in[a] - s * df * m0;
    } else {
      const double px = -(g.y[a] - yc), py = g.x[a] - xc;
      out[2 * a] = in[2 * a] - s * (df * m0 + dt * m2 * px);
      out[2 * a + 1] = in[2 * a + 1] - s * (df * m1 + dt * m2 * py);
    }
  }
}

// Occupancy of each pair kernel (blocks per SM) and the SM count, queried once
// per device.
struct DeviceShape {
  int nsm = 0;
  int occ[3][2] = {{0, 0}, {0, 0}, {0, 0}};  // [precision][kind]
};

// Per device, filled once under a lock: concurrent server threads must never
// see a half-filled entry (a different split count changes the summation
// order of the results).
const DeviceShape& device_shape() {
  static DeviceShape shapes[64];
  static std::mutex mu;
  int dev = 0;
  cudaGetDevice(&dev);
  DeviceShape& d = shapes[dev & 63];
  std::lock_guard<std::mutex> lk(mu);
  if (d.nsm == 0) {
    DeviceShape t;
    cudaDeviceGetAttribute(&t.nsm, cudaDevAttrMultiProcessorCount, dev);
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&t.occ[0][0], k_pair64<0, false>, kB64, 0);
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&t.occ[0][1], k_pair64<1, false>, kB64, 0);
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&t.occ[1][0], k_pair32<0, false>, kB32, 0);
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&t.occ[1][1], k_pair32<1, false>, kB32, 0);
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&t.occ[2][0], k_pair_ff<0, false>, kBF, 0);
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&t.occ[2][1], k_pair_ff<1, false>, kBF, 0);
    cudaGetLastError();
    if (t.nsm <= 0) t.nsm = 1;  // a failed query plans for one SM: slower, still correct
    for (auto& row : t.occ)
      for (int& o : row)
        if (o <= 0) o = 4;
    d = t;
  }
  return d;
}

}  // namespace

int device_sms() { return device_shape().nsm; }

// Choose the source split so that one wave fills every SM with as many
// blocks as can be resident: blocks = target blocks x splits ~ SMs x occupancy.
// Splits need not be tile-aligned (the kernels handle a short last tile).
namespace {

// Split counts chosen by timing (bie_tune), per device and shape (M, kind,
// precision); plan_pairs takes them before the occupancy rule.
std::mutex g_tune_mu;
std::map<std::array<int, 4>, PairPlan> g_tuned;

std::array<int, 4> tune_key(int M, int kind, int precision) {
  int dev = 0;
  cudaGetDevice(&dev);
  return {dev, M, kind, precision};
}

}  // namespace

void set_tuned_plan(int M, int kind, int precision, const PairPlan& p) {
  std::lock_guard<std::mutex> lk(g_tune_mu);
  g_tuned[tune_key(M, kind, precision)] = p;
}

void forget_tuned_plan(int M, int kind, int precision) {
  std::lock_guard<std::mutex> lk(g_tune_mu);
  g_tuned.erase(tune_key(M, kind, precision));
}

void clear_tuned_splits() {
  std::lock_guard<std::mutex> lk(g_tune_mu);
  g_tuned.clear();
}

PairPlan plan_with_splits(int M, int S) {
  const long long cap = std::max(1, (M + 63) / 64);  // chunks of at least 64 sources
  long long s = std::min<long long>(std::max(S, 1), cap);
  const long long chunk = (M + s - 1) / s;
  return uniform_plan((int)((M + chunk - 1) / chunk), (int)chunk);
}

PairPlan plan_two_level(int M, int c1, int c2, double f) {
  c1 = std::max(64, c1);
  c2 = std::max(64, std::min(c1, c2));
  const int S1 = std::max(0, std::min((int)(f * M / c1), M / c1));
  const int rem = M - S1 * c1;
  if (rem <= 0) return uniform_plan(S1, c1);
  return PairPlan{S1 + (rem + c2 - 1) / c2, c1, S1, c2};
}

PairPlan plan_symmetric(int M) {
  PairPlan p = uniform_plan((M + kTS - 1) / kTS, kTS);
  p.sym = kTS;
  return p;
}

// The symmetric FP64 plan: the tile size of the least estimated time.  The
// FP64 pipe bounds the kernel, so a pair of tiles costs tile^2 times the
// operations of two directed pairs, the SMs take tile pairs in rounds, and the
// slots (one a tile) cost their write and their read.  Measured, tiles of 32 /
// 64 / 128 / 256 nodes, Laplace: M = 704 23 / 39 / 74 / 234 us (directed 52),
// M = 7,168 609 / 619 / 633 / 688 (926), M = 25,600 7.57 / 7.52 / 7.53 / 7.65
// ms (12.1): small tiles fill the GPU at small M, large ones keep the slots few
// at large M.  Slots beyond max_slots or 512 MB: no symmetric plan (S = 0).
PairPlan plan_symmetric64(int M, int kind, int max_slots) {
  const int nsm = device_sms();
  PairPlan best{0, 0, 0, 0};
  double best_us = 1e300;
  for (int tile : {32, 64, 128, 256}) {
    const long long nt = (M + tile - 1) / tile, pairs = nt * (nt + 1) / 2;
    const double slot_mb = (double)nt * M * (kind + 1) * 8e-6;
    if (nt > max_slots || slot_mb > 512.0) continue;
    const double rounds = (double)((pairs + nsm - 1) / nsm);
    const double us = rounds * tile * tile * (kind == 0 ? 13.0 : 24.0) / 4000.0 + slot_mb / 2.0;
    if (us < best_us) {
      best_us = us;
      best = uniform_plan((int)nt, tile);
      best.sym = tile;
    }
  }
  return best;
}

// The symmetric FP32 plan (S = 0: the directed kernel).  Measured, Laplace, tiles
// of 128 / 256 nodes, directed: M = 4,096 22 / 31, 22 us; M = 8,192 33 / 37, 43; M
// = 12,800 54 / 60, 92; M = 25,600 159 / 157, 177; M = 51,200 576 / 563.  Stokes,
// 128 / 192, directed: M = 2,048 22, 16; M = 4,096 24, 25; M = 8,192 43 / 49, 56;
// M = 25,600 258 / 252, 305; M = 51,200 956 / 915, 1,684.
PairPlan plan_symmetric32(int M, int kind, int max_slots) {
  auto make = [&](int tile) {
    PairPlan p = uniform_plan((M + tile - 1) / tile, tile);
    p.sym = tile;
    return p;
  };
  auto pairs = [&](int tile) {
    const long long nt = (M + tile - 1) / tile;
    return nt * (nt + 1) / 2;
  };
  const int nsm = device_sms();
  PairPlan p{0, 0, 0, 0};
  if (kind == 0) {
    if (pairs(128) >= 6LL * nsm) p = make(pairs(256) >= 30LL * nsm ? kTS : 128);
  } else {
    if (pairs(128) >= 4LL * nsm) p = make(pairs(192) >= 40LL * nsm ? 192 : 128);
  }
  if (p.S > max_slots || (double)p.S * M * (kind + 1) * 8e-6 > 512.0) p = PairPlan{0, 0, 0, 0};
  return p;
}

PairPlan plan_with_tiles(int M, int kind, int precision, int tiles) {
  const PairPlan p0 = occupancy_plan(M, kind, precision);
  if (p0.sym && p0.S == tiles) return p0;  // (counts of small M may stand for several sizes)
  const int sizes[3][2][4] = {{{256, 128, 64, 32}, {256, 128, 64, 32}}, {{kTS, 128}, {192, 128}}, {{kTileF}, {}}};
  for (int tile : sizes[precision][kind]) {
    if (tile == 0 || (M + tile - 1) / tile != tiles || (double)tiles * M * (kind + 1) * 8e-6 > 512.0) continue;
    PairPlan p = uniform_plan(tiles, tile);
    p.sym = tile;
    return p;
  }
  return PairPlan{0, 0, 0, 0};
}

PairPlan plan_pairs(int M, int kind, int precision, int max_slots) {
  {
    std::lock_guard<std::mutex> lk(g_tune_mu);
    auto it = g_tuned.find(tune_key(M, kind, precision));
    // (the symmetric float-float and 256-node FP32 Laplace plans are not bounded by max_slots)
    if (it != g_tuned.end() && (!it->second.sym || it->second.S <= max_slots || (precision > 0 && it->second.sym == kTS)))
      return it->second;
  }
  return occupancy_plan(M, kind, precision, max_slots);
}

PairPlan occupancy_plan(int M, int kind, int precision, int max_slots) {
  const DeviceShape& d = device_shape();
  if (precision == 0) {
    const PairPlan p = plan_symmetric64(M, kind, max_slots);
    if (p.S > 0) return p;
  }
  if (precision == 1) {
    const PairPlan p = plan_symmetric32(M, kind, max_slots);
    if (p.S > 0) return p;
  }
  if ((precision == 1 || precision == 2) && kind == 0) {
    // the symmetric FP32 / float-float Laplace kernels once their tile pairs fill
    // the GPU a few times over and their partials (one slot per tile) stay
    // within 256 MB
    const long long nt = (M + kTS - 1) / kTS;
    if (nt * (nt + 1) / 2 >= 4LL * d.nsm && nt * (long long)M * 8 <= (256LL << 20)) return plan_symmetric(M);
  }
  const int per_block = precision == 0 ? kB64 * kT64 : (precision == 1 ? kB32 * kT32 : kBF * kTF);
  const long long bx = (M + per_block - 1) / per_block;
  const long long slots = (long long)d.nsm * d.occ[precision][kind];
  long long S = bx >= slots ? 1 : slots / bx;
  const long long min_chunk = 64;
  if (S > (M + min_chunk - 1) / min_chunk) S = (M + min_chunk - 1) / min_chunk;
  if (S < 1) S = 1;
  const long long chunk = (M + S - 1) / S;
  return uniform_plan((int)((M + chunk - 1) / chunk), (int)chunk);
}

// Batched solves: target block x sums over the len_x nodes of its problems.
// With S splits of chunk = ceil(src_max / S) sources, block x has
// ceil(len_x / chunk) busy splits, each with about the same work whatever the
// problem's size.  S is the smallest count whose busy blocks fill every
// resident slot once (chunks of at least 64 sources).
PairPlan plan_pairs_batch(const int* body_start, int N, const int* pbody, int P, int kind, int precision,
                          int max_slots) {
  const DeviceShape& d = device_shape();
  const int per_block = precision == 0 ? kB64 * kT64 : (precision == 1 ? kB32 * kT32 : kBF * kTF);
  const int M = body_start[N];
  std::vector<int> pstart(P + 1);
  int src_max = 1;
  for (int p = 0; p <= P; ++p) pstart[p] = p < P ? body_start[pbody[p]] : M;
  for (int p = 0; p < P; ++p) src_max = std::max(src_max, pstart[p + 1] - pstart[p]);
  if (precision == 1) {
    // The symmetric kernel by the rule of single systems (plan_symmetric32) on the sum of
    // the problems' tile pairs; problems of so different sizes that most CTAs of the grid
    // (the largest problem's pairs for each) would be empty, and fewer slots than the
    // slots' reduction takes, stay with the directed kernel.  Eight problems of 2,000 to
    // 5,500 nodes, Stokes: 146 us directed, 83 symmetric.
    const auto pairs = [&](int tile, long long& S) {
      long long sum = 0;
      S = 0;
      for (int p = 0; p < P; ++p) {
        const long long nt = (pstart[p + 1] - pstart[p] + tile - 1) / tile;
        S = std::max(S, nt);
        sum += nt * (nt + 1) / 2;
      }
      return sum;
    };
    const int big = kind == 0 ? kTS : 192;
    long long S, Sbig;
    const long long n128 = pairs(128, S), nbig = pairs(big, Sbig);
    const bool use_big = nbig >= (kind == 0 ? 30LL : 40LL) * d.nsm;
    if (use_big) S = Sbig;
    if (n128 >= (kind == 0 ? 6LL : 4LL) * d.nsm && S >= kRG && S <= max_slots &&
        P * (S * (S + 1) / 2) <= 4 * (use_big ? nbig : n128) && (double)S * M * (kind + 1) * 8e-6 <= 512.0) {
      PairPlan p = uniform_plan((int)S, use_big ? big : 128);
      p.sym = p.chunk;
      return p;
    }
  }
  const int bx = (M + per_block - 1) / per_block;
  std::vector<int> len(bx);
  for (int x = 0; x < bx; ++x) {
    const int tb = x * per_block, te = std::min(M, tb + per_block);
    const int p0 = (int)(std::upper_bound(pstart.begin(), pstart.end(), tb) - pstart.begin()) - 1;
    const int p1 = (int)(std::upper_bound(pstart.begin(), pstart.end(), te - 1) - pstart.begin()) - 1;
    len[x] = pstart[p1 + 1] - pstart[p0];
  }
  const long long slots = (long long)d.nsm * d.occ[precision][kind];
  const int s_cap = std::max(1, (src_max + 63) / 64);
  int S = 1;
  for (; S < s_cap; ++S) {
    const long long chunk = ((long long)src_max + S - 1) / S;
    long long busy = 0;
    for (int x = 0; x < bx; ++x) {
      const long long ch = std::max(chunk, ((long long)len[x] + S - 1) / S);
      busy += (len[x] + ch - 1) / ch;
    }
    if (busy >= slots) break;
  }
  return uniform_plan(S, (src_max + S - 1) / S);
}

namespace {

template <bool BATCH>
void launch_pairs(const Geo& g, int kind, int precision, const PairPlan& p, VecRef v, const double* sscale,
                  double* partial, const int* stop, cudaStream_t s) {
  if (precision == 0) {
    dim3 grid((g.M + kB64 * kT64 - 1) / (kB64 * kT64), p.S);
    if (!BATCH && p.sym) {
      const long long nt = (g.M + p.sym - 1) / p.sym;
      const unsigned pairs = (unsigned)(nt * (nt + 1) / 2);
      if (kind == 0)
        k_pair64s<0><<<pairs, p.sym, p.sym * sym64_vals<0>() * sizeof(double), s>>>(g, v, sscale, partial, stop);
      else
        k_pair64s<1><<<pairs, p.sym, p.sym * sym64_vals<1>() * sizeof(double), s>>>(g, v, sscale, partial, stop);
    } else if (kind == 0)
      k_pair64<0, BATCH><<<grid, kB64, 0, s>>>(g, v, sscale, p, partial, stop);
    else
      k_pair64<1, BATCH><<<grid, kB64, 0, s>>>(g, v, sscale, p, partial, stop);
  } else if (precision == 1) {
    dim3 grid((g.M + kB32 * kT32 - 1) / (kB32 * kT32), p.S);
    const int gs = (int)std::min<long long>(1216, (g.M + 255) / 256);
    if (kind == 0) {
      k_src32<0><<<gs, 256, 0, s>>>(g, v, sscale, stop);
      if (p.sym)
        launch_pair32s<0, BATCH>(g, p, partial, stop, s);
      else
        k_pair32<0, BATCH><<<grid, kB32, 0, s>>>(g, v, sscale, p, partial, stop);
    } else {
      k_src32<1><<<gs, 256, 0, s>>>(g, v, sscale, stop);
      if (p.sym)
        launch_pair32s<1, BATCH>(g, p, partial, stop, s);
      else
        k_pair32<1, BATCH><<<grid, kB32, 0, s>>>(g, v, sscale, p, partial, stop);
    }
    note_launches(1);
  } else {
    dim3 grid((g.M + kBF * kTF - 1) / (kBF * kTF), p.S);
    if (kind == 0 && !BATCH && p.sym) {
      const long long nt = (g.M + kTileF - 1) / kTileF;
      k_pair_ffs<<<(unsigned)(nt * (nt + 1) / 2), kBFS, 0, s>>>(g, (int)nt, partial, sscale, v, stop);
    } else if (kind == 0)
      k_pair_ff<0, BATCH><<<grid, kBF, 0, s>>>(g, v, sscale, p, partial, stop);
    else
      k_pair_ff<1, BATCH><<<grid, kBF, 0, s>>>(g, v, sscale, p, partial, stop);
  }
}

}  // namespace

// Batched solves (g.prange set) run instances with the problem masks; a single
// problem runs instances without any of that code.
cudaError_t pair_sum(const Geo& g, int kind, int precision, const PairPlan& p, VecRef v,
                     const double* sscale, double* partial, const int* stop, cudaStream_t s) {
  if (g.prange)
    launch_pairs<true>(g, kind, precision, p, v, sscale, partial, stop, s);
  else
    launch_pairs<false>(g, kind, precision, p, v, sscale, partial, stop, s);
  note_launches(1);
  return cudaGetLastError();
}

cudaError_t epilogue(const Geo& g, int kind, const PairPlan& p, VecRef v, const double* partial,
                     int scaled, int with_L, double sign, VecRef out, const int* stop,
                     cudaStream_t s, double alpha, bool pff, bool fp32) {
  if (p.S >= kRG) {
    // add the slots wide first (float-float or FP64), then an epilogue over one FP64 slot
    const long long n = (long long)g.M * (kind + 1);
    const unsigned nb = (unsigned)((n + kRT - 1) / kRT);
    if (pff)
      k_reduce_slots<<<nb, kRT * kRG, 0, s>>>(g, g.prange ? p.sym : 0, const_cast<double*>(partial), p.S, n, stop);
    else
      k_reduce_slots64<<<nb, kRT * kRG, 0, s>>>(const_cast<double*>(partial), p.S, n, stop);
    note_launches(1);
    return epilogue(g, kind, uniform_plan(1, g.M), v, partial, scaled, with_L, sign, out, stop, s, alpha, false,
                    fp32);
  }
  // one block per body, sized to the bodies (many small bodies: small blocks)
  const int avg = g.M / std::max(1, g.N);
  const int pf = pff ? 1 : 0;
  if (fp32) {  // the FP32 operator: the epilogue in FP32 arithmetic
    if (avg <= 64) {
      if (kind == 0)
        k_epilogue32<0, 64><<<g.N, 64, 0, s>>>(g, v, partial, p.S, scaled, with_L, alpha, sign, out, stop, pf);
      else
        k_epilogue32<1, 64><<<g.N, 64, 0, s>>>(g, v, partial, p.S, scaled, with_L, alpha, sign, out, stop, pf);
    } else {
      if (kind == 0)
        k_epilogue32<0, kBE><<<g.N, kBE, 0, s>>>(g, v, partial, p.S, scaled, with_L, alpha, sign, out, stop, pf);
      else
        k_epilogue32<1, kBE><<<g.N, kBE, 0, s>>>(g, v, partial, p.S, scaled, with_L, alpha, sign, out, stop, pf);
    }
    note_launches(1);
    return cudaGetLastError();
  }
  if (avg <= 64) {
    if (kind == 0)
      k_epilogue<0, 64><<<g.N, 64, 0, s>>>(g, v, partial, p.S, scaled, with_L, alpha, sign, out, stop, pff ? 1 : 0);
    else
      k_epilogue<1, 64><<<g.N, 64, 0, s>>>(g, v, partial, p.S, scaled, with_L, alpha, sign, out, stop, pff ? 1 : 0);
  } else {
    if (kind == 0)
      k_epilogue<0, kBE><<<g.N, kBE, 0, s>>>(g, v, partial, p.S, scaled, with_L, alpha, sign, out, stop, pff ? 1 : 0);
    else
      k_epilogue<1, kBE><<<g.N, kBE, 0, s>>>(g, v, partial, p.S, scaled, with_L, alpha, sign, out, stop, pff ? 1 : 0);
  }
  note_launches(1);
  return cudaGetLastError();
}

cudaError_t consistent_rhs(const Geo& g, int kind, double alpha, const double* in, double* out,
                           cudaStream_t s) {
  if (kind == 0)
    k_consistent_rhs<0><<<g.N, kBE, 0, s>>>(g, alpha, in, out);
  else
    k_consistent_rhs<1><<<g.N, kBE, 0, s>>>(g, alpha, in, out);
  note_launches(1);
  return cudaGetLastError();
}

}  // namespace bie

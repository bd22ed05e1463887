// One-launch solves of batches of small problems.
//
// A batch of small problems (at most kSmallMaxNodes nodes and kSmallMaxBodies
// bodies each) is solved by one persistent launch with one CTA per problem:
// the CTA runs the problem's whole FP64 iterative refinement (Section 6.1.1's
// rescaled system, eqs. ModRep2 / ModRep2Stokes) -- restarted GMRES with FP32
// pair sums on the correction equation (the completion weighted per body, as
// in the multi-launch path), and float-float pair sums for the true residual
// -- with no host round trip and no grid-wide synchronisation: every
// reduction is inside the CTA (warp shuffles in a fixed order, so results are
// deterministic).  A problem's sources live in shared memory for each operator
// application; its Krylov basis, iterate and residuals are slices of the
// batch's vectors in global memory (L2-resident at these sizes).
//
// The operator applied by the CTA is the one of pairsum.cu, per target node a:
//   (1/2 v_a + sw_a [ -(1/2pi) n_a . sum_b q_b r/|r|^2 - (1/4pi) w_a kappa_a mu_a + L_a ])   (Laplace)
// with the same exact hi/lo coordinate differences as the directed near tiles
// (FP32) or the exact three-float splits (float-float), so the per-pair
// arithmetic is that of pair_math.cuh.
#include <cuda_runtime.h>
#include <math.h>

#include <algorithm>
#include <atomic>
#include <vector>

#include "../../include/bie2d.h"
#include "bie_internal.cuh"
#include "pair_math.cuh"
#include "reduce.cuh"
#include "rotations.cuh"

namespace bie {

namespace {

constexpr int kSB = 512;       // threads a CTA
constexpr int kTPT = 1;        // threads per target node in the operators (1 or 2)
constexpr int kSW = kSB / 32;  // warps a CTA
constexpr int kSmallMaxRestart = 50;

struct SmallArgs {
  Geo g;
  int kind;
  const int* pbody;        // [P+1] first body of each problem
  const long long* pnode;  // [P+1] first vector entry of each problem
  const double* f;         // right-hand sides (sqrt(w)-scaled), batch layout
  double *x, *r, *d, *rc, *rin, *y;  // batch-layout vectors
  double* V;               // basis rows V_i = V + i ld (batch layout)
  long long ld;
  int m, max_refine, max_iter;
  double tol, inner_tol;
  SmallInfo* info;         // [P]
};

// Per-CTA shared state (static part).
struct SmallShared {
  double H[(kSmallMaxRestart + 1) * kSmallMaxRestart];
  double cs[kSmallMaxRestart], sn[kSmallMaxRestart], gv[kSmallMaxRestart + 1], yv[kSmallMaxRestart + 1];
  double h1[kSmallMaxRestart + 1], h2[kSmallMaxRestart + 1];
  double mom[3][kSmallMaxBodies];
  double red[kSW];
  double scal[4];
  int flag[2];
};

// ---------------------------------------------------------------- vectors ----
__device__ __forceinline__ double cta_dot(const double* __restrict__ a, const double* __restrict__ b, int n,
                                          SmallShared& sh) {
  double s = 0.0;
  for (int k = threadIdx.x; k < n; k += kSB) s = fma(a[k], b[k], s);
  return block_sum<kSB>(s, sh.red);
}

// ------------------------------------------------------ completion moments ----
// Per body of the problem (warp w takes bodies w, w + kSW, ...; lanes stride
// the nodes; fixed-order reductions): Laplace m0 = sum sw v; Stokes m0, m1 =
// sum sw v_1, sum sw v_2 and m2 = sum sw (p . v), p = (x - x^c)^perp.  alpha > 0
// weights them by alpha/|Gamma_i| (m0, m1) and alpha/W_i (m2).
__device__ void cta_moments(const Geo& g, int kind, int i0, int i1, const double* __restrict__ v, long long base,
                            double alpha, SmallShared& sh) {
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  for (int i = i0 + wid; i < i1; i += kSW) {
    const int a0 = g.body_start[i], a1 = g.body_start[i + 1];
    const double xc = g.xc[i], yc = g.yc[i];
    double m0 = 0.0, m1 = 0.0, m2 = 0.0;
    for (int a = a0 + lane; a < a1; a += 32) {
      const double s = g.sw[a];
      if (kind == 0) {
        m0 += s * v[a - base];
      } else {
        const double f1 = s * v[2 * (a - base)], f2 = s * v[2 * (a - base) + 1];
        m0 += f1;
        m1 += f2;
        m2 += -(g.y[a] - yc) * f1 + (g.x[a] - xc) * f2;
      }
    }
    m0 = warp_sum(m0);
    if (kind == 1) {
      m1 = __shfl_sync(0xffffffffu, warp_sum(m1), 0);
      m2 = __shfl_sync(0xffffffffu, warp_sum(m2), 0);
    }
    // lane q weights and stores moment q
    const double m = lane == 0 ? m0 : lane == 1 ? m1 : m2;
    if (lane < (kind == 0 ? 1 : 3)) {
      const double weight = alpha > 0.0 ? alpha * rcp64(lane < 2 ? g.len[i] : g.W[i]) : 1.0;
      sh.mom[lane][i - i0] = m * weight;
    }
  }
}

// ------------------------------------------------------------- operators ----
// out = (1/2 I + K + L_alpha) v on the problem's sqrt(w)-scaled entries, v and
// out slices starting at node `base` (entry base * (kind + 1)).  FF: the pair
// sums in float-float, else FP32.  `src` is the dynamic shared memory.
template <int KIND, bool FF>
__device__ void cta_apply(const Geo& g, int a0, int a1, int i0, int i1, const double* __restrict__ v,
                          double* __restrict__ out, double alpha, SmallShared& sh, unsigned char* src) {
  const int M = a1 - a0;
  cta_moments(g, KIND, i0, i1, v, a0, alpha, sh);
  // sources of the problem in shared memory
  float4* sp = reinterpret_cast<float4*>(src);  // FP32: (x_hi, y_hi, x_lo, y_lo); FF: (xh, xm, yh, ym)
  float4* sq = sp + M;                          // FP32: (q1, q2, -, -); FF: (q1h, q1l, q2h, q2l)
  float2* sl = reinterpret_cast<float2*>(sq + M);  // FF: (xl, yl)
  for (int l = threadIdx.x; l < M; l += kSB) {
    const int b = a0 + l;
    const double s = g.sw[b];
    const double q1 = KIND == 0 ? s * v[l] : s * v[2 * l];
    const double q2 = KIND == 0 ? 0.0 : s * v[2 * l + 1];
    if (FF) {
      sp[l] = g.xff[b];
      sl[l] = g.xfl[b];
      const float q1h = (float)q1, q2h = (float)q2;
      sq[l] = make_float4(q1h, (float)(q1 - (double)q1h), q2h, (float)(q2 - (double)q2h));
    } else {
      sp[l] = g.pf[b];
      sq[l] = make_float4((float)q1, (float)q2, 0.f, 0.f);
    }
  }
  __syncthreads();
  // kTPT = 2: two threads per target (adjacent lanes), each over half of the
  // sources, the halves added by a shuffle in a fixed order.  The trip count is
  // the same for every lane, so that the shuffles see the whole warp.
  const int half = kTPT == 2 ? (threadIdx.x & 1) : 0;
  const int lh = half == 0 ? 0 : M / 2, uh = (half == 0 && kTPT == 2) ? M / 2 : M;
  for (int t0 = 0; t0 < M; t0 += kSB / kTPT) {
    const int t = t0 + (int)threadIdx.x / kTPT;
    const bool live = t < M;
    const int a = a0 + (live ? t : 0);
    double k1 = 0.0, k2 = 0.0;
    if (FF) {
      FFTarget tg;
      const float4 p = g.xff[a];
      const float2 pl = g.xfl[a];
      tg.xh = p.x;
      tg.xm = p.y;
      tg.yh = p.z;
      tg.ym = p.w;
      tg.xl = pl.x;
      tg.yl = pl.y;
      tg.n = KIND == 1 ? g.nff[a] : make_float4(0.f, 0.f, 0.f, 0.f);
      // two independent float-float sums (ILP), added in a fixed order
      float sxh = 0.f, sxl = 0.f, syh = 0.f, syl = 0.f, txh = 0.f, txl = 0.f, tyh = 0.f, tyl = 0.f;
      if (live) {
        int l = lh;
        for (; l + 2 <= uh; l += 2) {
          float cxh, cxl, cyh, cyl, dxh, dxl, dyh, dyl;
          ff_pair<KIND>(tg, sp[l], sl[l], sq[l], cxh, cxl, cyh, cyl);
          ff_pair<KIND>(tg, sp[l + 1], sl[l + 1], sq[l + 1], dxh, dxl, dyh, dyl);
          if (l == t) cxh = cxl = cyh = cyl = 0.f;  // the self pair (r = 0)
          if (l + 1 == t) dxh = dxl = dyh = dyl = 0.f;
          ff_acc(sxh, sxl, cxh, cxl);
          ff_acc(syh, syl, cyh, cyl);
          ff_acc(txh, txl, dxh, dxl);
          ff_acc(tyh, tyl, dyh, dyl);
        }
        if (l < uh && l != t) {
          float cxh, cxl, cyh, cyl;
          ff_pair<KIND>(tg, sp[l], sl[l], sq[l], cxh, cxl, cyh, cyl);
          ff_acc(sxh, sxl, cxh, cxl);
          ff_acc(syh, syl, cyh, cyl);
        }
        ff_acc(sxh, sxl, txh, txl);
        ff_acc(syh, syl, tyh, tyl);
      }
      if (kTPT == 2) {  // the second half's sums join the first's (float-float)
        const float oxh = __shfl_xor_sync(0xffffffffu, sxh, 1), oxl = __shfl_xor_sync(0xffffffffu, sxl, 1);
        const float oyh = __shfl_xor_sync(0xffffffffu, syh, 1), oyl = __shfl_xor_sync(0xffffffffu, syl, 1);
        ff_acc(sxh, sxl, oxh, oxl);
        ff_acc(syh, syl, oyh, oyl);
      }
      k1 = (double)sxh + (double)sxl;
      k2 = (double)syh + (double)syl;
    } else {
      const float4 p = g.pf[a];
      const float2 n = g.nf[a];
      // FP32 sums over chunks of 256 sources, chunks added with TwoSum
      float sx = 0.f, ex = 0.f, sy = 0.f, ey = 0.f;
      if (live) {
        for (int c0 = lh; c0 < uh; c0 += 256) {
          const int c1 = min(uh, c0 + 256);
          // four independent sums (ILP), added in a fixed order
          float ax0 = 0.f, ay0 = 0.f, ax1 = 0.f, ay1 = 0.f, ax2 = 0.f, ay2 = 0.f, ax3 = 0.f, ay3 = 0.f;
          int l = c0;
          for (; l + 4 <= c1; l += 4) {
            float cx0, cy0, cx1, cy1, cx2, cy2, cx3, cy3;
            f32_pair<KIND>(p.x, p.y, p.z, p.w, n.x, n.y, sp[l], sq[l].x, sq[l].y, cx0, cy0);
            f32_pair<KIND>(p.x, p.y, p.z, p.w, n.x, n.y, sp[l + 1], sq[l + 1].x, sq[l + 1].y, cx1, cy1);
            f32_pair<KIND>(p.x, p.y, p.z, p.w, n.x, n.y, sp[l + 2], sq[l + 2].x, sq[l + 2].y, cx2, cy2);
            f32_pair<KIND>(p.x, p.y, p.z, p.w, n.x, n.y, sp[l + 3], sq[l + 3].x, sq[l + 3].y, cx3, cy3);
            if (l == t) cx0 = cy0 = 0.f;  // the self pair (r = 0)
            if (l + 1 == t) cx1 = cy1 = 0.f;
            if (l + 2 == t) cx2 = cy2 = 0.f;
            if (l + 3 == t) cx3 = cy3 = 0.f;
            ax0 += cx0;
            ay0 += cy0;
            ax1 += cx1;
            ay1 += cy1;
            ax2 += cx2;
            ay2 += cy2;
            ax3 += cx3;
            ay3 += cy3;
          }
          for (; l < c1; ++l) {
            float cx, cy;
            f32_pair<KIND>(p.x, p.y, p.z, p.w, n.x, n.y, sp[l], sq[l].x, sq[l].y, cx, cy);
            if (l == t) cx = cy = 0.f;
            ax0 += cx;
            ay0 += cy;
          }
          const float ax = (ax0 + ax1) + (ax2 + ax3), ay = (ay0 + ay1) + (ay2 + ay3);
          float u, e;
          two_sum(sx, ax, u, e);
          sx = u;
          ex += e;
          two_sum(sy, ay, u, e);
          sy = u;
          ey += e;
        }
      }
      k1 = (double)sx + (double)ex;
      k2 = (double)sy + (double)ey;
      if (kTPT == 2) {  // first half + second half, the same on both lanes
        k1 += __shfl_xor_sync(0xffffffffu, k1, 1);
        k2 += __shfl_xor_sync(0xffffffffu, k2, 1);
      }
    }
    if (!live || half != 0) continue;
    const int i = g.body_of[a] - i0;
    const double os = g.sw[a];
    const double wk = g.w[a] * g.kappa[a];
    if (KIND == 0) {
      const double k = g.nx[a] * k1 + g.ny[a] * k2;
      // (the diagonal limit acts on v / os, times os)
      out[t] = 0.5 * v[t] + os * (sh.mom[0][i] - kInv2Pi * k) - kInv4Pi * wk * v[t];
    } else {
      const double v1 = v[2 * t], v2 = v[2 * t + 1];
      const double tx = -g.ny[a], ty = g.nx[a];
      const double dd = -0.5 * kInvPi * wk * (tx * v1 + ty * v2);
      const int ib = g.body_of[a];
      const double px = -(g.y[a] - g.yc[ib]), py = g.x[a] - g.xc[ib];
      out[2 * t] = 0.5 * v1 + os * (sh.mom[0][i] + px * sh.mom[2][i] - kInvPi * k1) + dd * tx;
      out[2 * t + 1] = 0.5 * v2 + os * (sh.mom[1][i] + py * sh.mom[2][i] - kInvPi * k2) + dd * ty;
    }
  }
  __syncthreads();
}

// out = in - (I - C) L~(in) (the right-hand side of a correction solved with
// the per-body weighted completion, weight alpha; see consistent_rhs).
template <int KIND>
__device__ void cta_consistent(const Geo& g, int a0, int i0, int i1, const double* __restrict__ in,
                               double* __restrict__ out, double alpha, SmallShared& sh) {
  cta_moments(g, KIND, i0, i1, in, a0, 0.0, sh);
  __syncthreads();
  const int M = g.body_start[i1] - a0;
  for (int t = threadIdx.x; t < M; t += kSB) {
    const int a = a0 + t;
    const int ib = g.body_of[a], i = ib - i0;
    const double s = g.sw[a];
    const double df = (1.0 - alpha / g.len[ib]) / g.len[ib];
    if (KIND == 0) {
      out[t] = in[t] - s * df * sh.mom[0][i];
    } else {
      const double dt = (1.0 - alpha / g.W[ib]) / g.W[ib];
      const double px = -(g.y[a] - g.yc[ib]), py = g.x[a] - g.xc[ib];
      out[2 * t] = in[2 * t] - s * (df * sh.mom[0][i] + dt * sh.mom[2][i] * px);
      out[2 * t + 1] = in[2 * t + 1] - s * (df * sh.mom[1][i] + dt * sh.mom[2][i] * py);
    }
  }
  __syncthreads();
}

// ------------------------------------------------------------------ GMRES ----
// Restarted GMRES(m) on A32 x = b (FP32 pair sums, weighted completion alpha),
// x = 0 first; CGS2 with the inner products warp per basis vector, Givens
// rotations by one thread.  Stops when the residual estimate is at most
// tol_rel ||b||, or after maxit iterations; returns the iterations taken.
// V_i of this problem: V + i ld + e0.
template <int KIND>
__device__ int cta_gmres(const SmallArgs& A, int a0, int a1, int i0, int i1, long long e0, int n,
                         const double* __restrict__ b, double* __restrict__ x, double* __restrict__ rr,
                         double alpha, double tol_rel, int maxit, SmallShared& sh, unsigned char* src,
                         int& matvecs) {
  const int m = A.m;
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  auto Vr = [&](int i) { return A.V + (long long)i * A.ld + e0; };
  for (int k = threadIdx.x; k < n; k += kSB) x[k] = 0.0;
  const double bnorm = sqrt(cta_dot(b, b, n, sh));
  if (!(bnorm > 0.0)) return 0;
  const double tol_abs = tol_rel * bnorm;
  // first cycle: residual = b
  for (int k = threadIdx.x; k < n; k += kSB) rr[k] = b[k];
  double beta = bnorm;
  int total = 0;
  for (;;) {
    double* V0 = Vr(0);
    const double inv0 = 1.0 / beta;
    for (int k = threadIdx.x; k < n; k += kSB) V0[k] = rr[k] * inv0;
    if (threadIdx.x == 0) {
      sh.gv[0] = beta;
      for (int i = 1; i <= m; ++i) sh.gv[i] = 0.0;
    }
    __syncthreads();
    int j = 0;
    bool done = false;
    for (; j < m; ++j) {
      double* w = Vr(j + 1);
      cta_apply<KIND, false>(A.g, a0, a1, i0, i1, Vr(j), w, alpha, sh, src);
      ++matvecs;
      // CGS2: two passes of h = V^T w, w -= V h
      for (int pass = 0; pass < 2; ++pass) {
        double* hs = pass == 0 ? sh.h1 : sh.h2;
        // the second pass also sums ||w||^2 (as product j + 1 of w with itself)
        for (int i = wid; i <= j + pass; i += kSW) {
          const double* Vi = i <= j ? Vr(i) : w;
          double s0 = 0.0, s1 = 0.0;
          int k = lane;
          for (; k + 32 < n; k += 64) {
            s0 = fma(Vi[k], w[k], s0);
            s1 = fma(Vi[k + 32], w[k + 32], s1);
          }
          if (k < n) s0 = fma(Vi[k], w[k], s0);
          const double t = warp_sum(s0 + s1);
          if (lane == 0) hs[i] = t;
        }
        __syncthreads();
        for (int k = threadIdx.x; k < n; k += kSB) {
          double s = w[k];
          for (int i = 0; i <= j; ++i) s -= hs[i] * Vr(i)[k];
          w[k] = s;
        }
        __syncthreads();
      }
      // ||w - V h2||^2 = ||w||^2 - ||h2||^2 while nothing is lost (kNormBySubtraction), by warp 0
      if (wid == 0) {
        double h22 = 0.0;
        for (int i = lane; i <= j; i += 32) h22 = fma(sh.h2[i], sh.h2[i], h22);
        h22 = warp_sum(h22);
        if (lane == 0) {
          sh.scal[1] = sh.h2[j + 1] - h22;
          sh.flag[0] = !(h22 <= kNormBySubtraction * sh.h2[j + 1]);
        }
      }
      __syncthreads();
      if (sh.flag[0]) {  // (the same in every thread)
        const double t = cta_dot(w, w, n, sh);
        if (threadIdx.x == 0) sh.scal[1] = t;
      }
      if (threadIdx.x == 0) {
        const double hn = sqrt(sh.scal[1]);
        double* Hc = sh.H + j * (m + 1);
        for (int i = 0; i <= j; ++i) Hc[i] = sh.h1[i] + sh.h2[i];
        double c, s, rho;
        givens(rotate_column(sh.cs, sh.sn, Hc, j), hn, c, s, rho);
        sh.scal[1] = hn;
        sh.scal[2] = hn > 0.0 ? 1.0 / hn : 0.0;
        sh.cs[j] = c;
        sh.sn[j] = s;
        Hc[j] = rho;
        Hc[j + 1] = 0.0;
        const double gj = sh.gv[j];
        sh.gv[j + 1] = -s * gj;
        sh.gv[j] = c * gj;
        sh.scal[0] = fabs(s * gj);
      }
      __syncthreads();
      const double res = sh.scal[0], hn = sh.scal[1], inv = sh.scal[2];
      for (int k = threadIdx.x; k < n; k += kSB) w[k] *= inv;
      __syncthreads();
      ++total;
      if (res <= tol_abs || !(hn > 1e-300 * beta) || total >= maxit) {
        done = true;
        ++j;
        break;
      }
    }
    // x += V y, y = R^{-1} g over the j steps of this cycle
    if (threadIdx.x == 0) {
      for (int i = j - 1; i >= 0; --i) {
        double s = sh.gv[i];
        for (int k = i + 1; k < j; ++k) s -= sh.H[k * (m + 1) + i] * sh.yv[k];
        sh.yv[i] = s / sh.H[i * (m + 1) + i];
      }
    }
    __syncthreads();
    for (int k = threadIdx.x; k < n; k += kSB) {
      double s = x[k];
      for (int i = 0; i < j; ++i) s += sh.yv[i] * Vr(i)[k];
      x[k] = s;
    }
    __syncthreads();
    if (done) return total;
    // restart from the explicit residual rr = b - A x
    cta_apply<KIND, false>(A.g, a0, a1, i0, i1, x, rr, alpha, sh, src);
    ++matvecs;
    for (int k = threadIdx.x; k < n; k += kSB) rr[k] = b[k] - rr[k];
    __syncthreads();
    beta = sqrt(cta_dot(rr, rr, n, sh));
    if (beta <= tol_abs) return total;
  }
}

// ------------------------------------------------------------------ solve ----
// Bound by latency and, in its vector work, by the FP64 pipe, where an instruction
// by all 16 warps takes 256 clocks: so one thread takes the square roots and
// quotients, the norm comes out of the second projection, and nothing is divided a
// node.  128 problems of four discs (512 nodes): 883 -> 780 us.
template <int KIND>
__global__ void __launch_bounds__(kSB, 2) k_small_solve(SmallArgs A) {
  extern __shared__ __align__(16) unsigned char src[];
  __shared__ SmallShared sh;
  const int p = blockIdx.x;
  const Geo& g = A.g;
  const int i0 = A.pbody[p], i1 = A.pbody[p + 1];
  const int a0 = g.body_start[i0], a1 = g.body_start[i1];
  const long long e0 = A.pnode[p];
  const int n = (int)(A.pnode[p + 1] - e0);
  const double* f = A.f + e0;
  double *x = A.x + e0, *r = A.r + e0, *d = A.d + e0, *rc = A.rc + e0, *rin = A.rin + e0, *y = A.y + e0;
  for (int k = threadIdx.x; k < n; k += kSB) {
    x[k] = 0.0;
    r[k] = f[k];
  }
  const double fnorm = sqrt(cta_dot(f, f, n, sh));
  double rnorm = fnorm, eps32 = -1.0, bound = 0.0;
  int iters = 0, refs = 0, m32 = 0, mff = 0;
  bool true_residual = true;
  while (rnorm > A.tol * fnorm && refs < A.max_refine && iters < A.max_iter) {
    // correction: A32_c d = r - (I - C) L~(r), weighted completion (weight 1)
    cta_consistent<KIND>(g, a0, i0, i1, r, rc, 1.0, sh);
    const int it = cta_gmres<KIND>(A, a0, a1, i0, i1, e0, n, rc, d, rin, 1.0, A.inner_tol, A.max_iter - iters, sh,
                                   src, m32);
    iters += it;
    refs += 1;
    for (int k = threadIdx.x; k < n; k += kSB) x[k] += d[k];
    __syncthreads();
    if (!true_residual && eps32 >= 0.0) {
      // as the multi-launch path: after the first true residual, r -= A32 d
      // with the paper's completion, and the update's error bound 3 eps32
      // ||A32 d|| added to ||r|| (a true residual again once the bound
      // reaches half the tolerance)
      cta_apply<KIND, false>(g, a0, a1, i0, i1, d, y, 0.0, sh, src);
      ++m32;
      bound += 3.0 * eps32 * sqrt(cta_dot(y, y, n, sh));
      for (int k = threadIdx.x; k < n; k += kSB) r[k] -= y[k];
      __syncthreads();
      rnorm = sqrt(cta_dot(r, r, n, sh)) + bound;
      if (bound > 0.5 * A.tol * fnorm) true_residual = true;
    } else {
      // true residual with float-float pair sums and the paper's completion
      cta_apply<KIND, true>(g, a0, a1, i0, i1, x, y, 0.0, sh, src);
      ++mff;
      for (int k = threadIdx.x; k < n; k += kSB) r[k] = f[k] - y[k];
      __syncthreads();
      rnorm = sqrt(cta_dot(r, r, n, sh));
      bound = 0.0;
      if (eps32 < 0.0) {
        // the FP32 operator's relative error on x (the update bound; reported)
        cta_apply<KIND, false>(g, a0, a1, i0, i1, x, rin, 0.0, sh, src);
        ++m32;
        double s2 = 0.0, t2 = 0.0;
        for (int k = threadIdx.x; k < n; k += kSB) {
          s2 = fma(rin[k] - y[k], rin[k] - y[k], s2);
          t2 = fma(y[k], y[k], t2);
        }
        s2 = block_sum<kSB>(s2, sh.red);
        t2 = block_sum<kSB>(t2, sh.red);
        eps32 = t2 > 0.0 ? sqrt(s2 / t2) : 0.0;
      }
      true_residual = false;
    }
    if (it == 0) break;
  }
  if (threadIdx.x == 0) {
    SmallInfo& q = A.info[p];
    q.iters = iters;
    q.refinements = refs;
    q.matvecs32 = m32;
    q.matvecsff = mff;
    q.rel_residual = fnorm > 0.0 ? rnorm / fnorm : 0.0;
    q.fp32_error = eps32 > 0.0 ? eps32 : 0.0;
  }
}

size_t small_smem_bytes(int max_nodes) {
  // FF: (xh, xm, yh, ym) float4 + (q1h, q1l, q2h, q2l) float4 + (xl, yl) float2 a node
  return (size_t)max_nodes * (2 * sizeof(float4) + sizeof(float2));
}

}  // namespace

namespace {
std::atomic<bool> g_small_on{true};
}  // namespace

void set_small_batch_path(bool on) { g_small_on.store(on); }
bool small_batch_path() { return g_small_on.load(); }

bool small_batch_eligible(int max_nodes, int max_bodies, int restart) {
  return max_nodes <= kSmallMaxNodes && max_bodies <= kSmallMaxBodies && restart <= kSmallMaxRestart;
}

cudaError_t small_batch_solve(const Geo& g, int kind, int P, const int* pbody, const long long* pnode,
                              const double* f, double* x, double* r, double* d, double* rc, double* rin, double* y,
                              double* V, long long ld, int m, double tol, double inner_tol, int max_refine,
                              int max_iter, int max_nodes, SmallInfo* info, cudaStream_t s) {
  SmallArgs A{g, kind, pbody, pnode, f, x, r, d, rc, rin, y, V, ld, m, max_refine, max_iter, tol, inner_tol, info};
  const size_t smem = small_smem_bytes(max_nodes);
  const int bound = (int)small_smem_bytes(kSmallMaxNodes);  // constant: other threads launch too
  cudaError_t e;
  if (kind == 0) {
    e = cudaFuncSetAttribute(k_small_solve<0>, cudaFuncAttributeMaxDynamicSharedMemorySize, bound);
    if (e != cudaSuccess) return e;
    k_small_solve<0><<<P, kSB, smem, s>>>(A);
  } else {
    e = cudaFuncSetAttribute(k_small_solve<1>, cudaFuncAttributeMaxDynamicSharedMemorySize, bound);
    if (e != cudaSuccess) return e;
    k_small_solve<1><<<P, kSB, smem, s>>>(A);
  }
  note_launches(1);
  return cudaGetLastError();
}

}  // namespace bie

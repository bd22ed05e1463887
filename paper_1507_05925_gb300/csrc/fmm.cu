// Quadtree fast multipole method for the pair sums, in complex variables.
//
// With z = x1 + i x2, both kernels reduce to Cauchy sums
//   F_q(z_a) = sum_{b != a} q_b / (z_a - z_b),   F'_q its z-derivative.
// Laplace (Section 3.4): with q = w mu (real) and nu = n1 + i n2 at the target,
//   sum_b q_b (r . n_a)/|r|^2 = Re(nu_a F_q(z_a)).
// Stokes traction (Section 4.3): with q = w (mu1 + i mu2) complex, and
//   S1 = F_q, S2 = -F'_q, S3 = -F'_{q conj(z - c0)}, S6 = F_{conj q} (any c0 fixed for the target),
//   sum_b r (r . q_b)(r . n_a)/|r|^4 =
//     (1/4) [ conj(nu) conj(conj(z_a - c0) S2 - S3) + nu conj(S1) + conj(nu) conj(S6) + nu S1 ],
// an identity of complex algebra (r . m = Re(r conj(m)) for complex r, m).
//
// Uniform quadtree on the bounding square, leaf level L chosen so that a
// non-empty leaf holds about 24-50 nodes.  Expansions in scaled form (powers of
// (z - c)/s), so the translation operators do not depend on the level: 4
// multipole-to-multipole and 4 local-to-local p x p complex matrices, and for
// the multipole-to-local step (offsets -3..3 in each direction) two diagonal
// factors per offset around one real Pascal matrix, built on the host in
// double precision.  Multipole:  F(z) = sum_k a_k s^k / (z - c)^(k+1),
// a_k = sum_j q_j ((z_j - c)/s)^k; local: F(z) = sum_l b_l ((z - c)/s)^l.
// Translations (d = target centre - source centre):
//   M2M  a'_k = sum_{m<=k} C(k,m) 2^-m w^(k-m) a_m,        w = (c_child - c_parent)/S
//   M2L  b_l  = (1/s) sum_k (-1)^l C(k+l,l) D^-(k+l+1) a_k,  D = d/s (integer offset)
//   L2L  b'_m = sum_{l>=m} C(l,m) 2^-m w^(l-m) b_l
// The near field (the 3 x 3 leaves around a target's leaf) is summed directly.
// For the pair sums the S3 channel carries, in every box B, the box-relative
// density q conj(z - c_B)/s_B, so that the combination conj(z_a - c) S2 - S3
// is formed about the target's own leaf centre c: about one global c0 its two
// terms grow with |z_a - c0| and cancel, which costs FP32 expansions their
// accuracy.  The translations add the exact shift terms: M2M takes
// 1/2 a_B + gamma a_0 (gamma = conj(c_child - c_parent)/(2 s_child)), M2L
// a_S - conj(D) a_0, L2L 2 b_P + delta b_0 (delta = conj(c_P - c_C)/s_C).
// Nodes are grouped by leaf with a counting sort whose order inside a leaf is
// the node order, so every sum runs in a fixed order (deterministic results).
#include <cuda_runtime.h>
#include <math.h>
#include <string.h>

#include <algorithm>
#include <complex>
#include <string>
#include <type_traits>
#include <vector>

#include "../../include/bie2d.h"
#include "bie_internal.cuh"
#include "logtab.cuh"
#include "pair_math.cuh"
#include "reduce.cuh"

namespace bie {

namespace {

constexpr int kMaxP = 64;
constexpr int kB = 64;       // threads per box block (>= p)
constexpr int kChunk = 32;   // points per P2M chunk
constexpr int kMaxNd = 4;    // channels per box

__host__ __device__ inline long long lev_off(int l) { return ((1LL << (2 * l)) - 1) / 3; }

__device__ __forceinline__ double2 cmul(double2 a, double2 b) {
  return make_double2(a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x);
}
__device__ __forceinline__ double2 cadd(double2 a, double2 b) { return make_double2(a.x + b.x, a.y + b.y); }
__device__ __forceinline__ double2 cconj(double2 a) { return make_double2(a.x, -a.y); }
// acc += a * b
__device__ __forceinline__ void cfma(double2& acc, double2 a, double2 b) {
  acc.x = fma(a.x, b.x, fma(-a.y, b.y, acc.x));
  acc.y = fma(a.x, b.y, fma(a.y, b.x, acc.y));
}

// The same in FP32 (expansions of the inner solves' operator).
__device__ __forceinline__ float2 cmul(float2 a, float2 b) {
  return make_float2(a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x);
}
__device__ __forceinline__ float2 cadd(float2 a, float2 b) { return make_float2(a.x + b.x, a.y + b.y); }
__device__ __forceinline__ float2 cconj(float2 a) { return make_float2(a.x, -a.y); }
__device__ __forceinline__ void cfma(float2& acc, float2 a, float2 b) {
  acc.x = fmaf(a.x, b.x, fmaf(-a.y, b.y, acc.x));
  acc.y = fmaf(a.x, b.y, fmaf(a.y, b.x, acc.y));
}
template <class T2>
__device__ __forceinline__ T2 cx(double x, double y);
template <>
__device__ __forceinline__ double2 cx<double2>(double x, double y) { return make_double2(x, y); }
template <>
__device__ __forceinline__ float2 cx<float2>(double x, double y) { return make_float2((float)x, (float)y); }

// Tree and expansion buffers of one apply; T2 = double2 (FP64 expansions) or
// float2 (FP32 expansions).  Densities Q stay FP64.
template <class T2>
struct FmmDevT {
  int L, nb, p, nd, M;
  int nlog;           // the first nlog channels carry the logarithm kernel, the rest Cauchy sums
  int cm;             // channel with the box-relative moment density q conj(z - c_B)/s_B (-1: none)
  double x0, y0, D, Dinv;  // bounding square: corner, side, 1/side
  const int* leaf;
  const int* perm;
  const int* start;
  const int* count;   // sources per box (all levels)
  const int* tcount;  // targets per box: boxes that need local expansions
  double2* Q;
  T2* mp;
  T2* lc;
  const T2* ops;
  const float2* Qf = nullptr;  // FP32 expansions: q per source in FP32 (channel 0), written by k_fmm_p2m32
  const float4* cen32 = nullptr;  // FP32 expansions: leaf centres split hi + lo
  float is32 = 0.f, s32 = 0.f;    // FP32 expansions: 1/s and s of a leaf
  int per = 1, tper = 1;          // boxes a block goes over: of one level, of all levels (boxes_a_block)
};

// Trees of few large bodies are mostly empty (100,000 nodes on one curve: 3,300 of a
// million leaves), and a block for every box costs more than the work: a block with a large
// shared array holds an SM's place for a microsecond to find its box empty.  There a block
// goes over several boxes, a grid's width apart (neighbours along a curve stay with
// different blocks), so many that it expects an eighth of a box to do; a tree at least 1/32 full
// keeps a block a box (at 1/16 blocks with two or three boxes cost more than the empty
// ones: Laplace, 20 bodies of 2,000 nodes, 517 -> 548 us an application).  One Stokes body
// of 100,000 nodes, a block a box and so: FP32 M2L 1,208 -> 74 us, float-float 3,496 -> 452,
// FP32 M2M 442 -> 66, FP64 2,167 -> 256, FP32 evaluation 547 -> 55; a solve 82 -> 38 ms.
inline int boxes_a_block(double used, double all) {
  return used * 32.0 >= all ? 1 : (int)fmin(32.0, 0.125 * all / fmax(used, 1.0));
}
// The same for the boxes of all levels 2..L of which level l uses at most used(l).
template <class F>
int boxes_a_block_levels(int L, F&& used) {
  double u = 0.0, all = 0.0;
  for (int l = 2; l <= L; ++l) {
    const double n = (double)(1LL << (2 * l));
    u += fmin(n, used(l));
    all += n;
  }
  return boxes_a_block(u, all);
}
inline unsigned blocks_for(long long boxes, int per) { return (unsigned)((boxes + per - 1) / per); }

// body(box) for the block's box, or (MANY) for its boxes blockIdx.x + i gridDim.x, i < per,
// of `boxes` that hold something.
template <bool MANY, class F>
__device__ __forceinline__ void for_boxes(const int* __restrict__ count, long long boxes, int per, F&& body) {
  if (!MANY) {
    body((long long)blockIdx.x);
    return;
  }
  const int lane = threadIdx.x & 31;
  const long long own = blockIdx.x + (long long)lane * gridDim.x;
  unsigned todo = __ballot_sync(0xffffffffu, lane < per && own < boxes && count[own] > 0);  // the same in every warp
  while (todo) {
    body(blockIdx.x + (long long)(__ffs(todo) - 1) * gridDim.x);
    todo &= todo - 1;
  }
}
using FmmDev = FmmDevT<double2>;

template <class T2>
__device__ __forceinline__ double2 box_center(const FmmDevT<T2>& f, int l, int bx, int by, double& s) {
  s = ldexp(f.D, -l);  // exact: no division on the (slow) FP64 pipe
  return make_double2(f.x0 + (bx + 0.5) * s, f.y0 + (by + 0.5) * s);
}

// ------------------------------------------------------------------ setup ----
// Bounding square of the body boxes and the total arc length.
constexpr int kBoxT = 256;
__global__ void __launch_bounds__(kBoxT) k_fmm_box(Geo g, double* out) {
  __shared__ double sh[kBoxT / 32];
  double x0 = 1e300, y0 = 1e300, nx1 = 1e300, ny1 = 1e300, len = 0.0;  // nx1, ny1: -max
  for (int i = threadIdx.x; i < g.N; i += kBoxT) {
    const float4 b = g.bbox[i];
    x0 = fmin(x0, (double)b.x);
    y0 = fmin(y0, (double)b.y);
    nx1 = fmin(nx1, -(double)b.z);
    ny1 = fmin(ny1, -(double)b.w);
    len += g.len[i];
  }
  x0 = block_min<kBoxT>(x0, sh);
  y0 = block_min<kBoxT>(y0, sh);
  const double x1 = -block_min<kBoxT>(nx1, sh), y1 = -block_min<kBoxT>(ny1, sh);
  len = block_sum<kBoxT>(len, sh);
  if (threadIdx.x == 0) {
    const double D = fmax(x1 - x0, y1 - y0) * (1.0 + 1e-6) + 1e-12;
    out[0] = x0 - 1e-7 * D;
    out[1] = y0 - 1e-7 * D;
    out[2] = D * (1.0 + 2e-7);
    out[3] = len;
  }
}

__global__ void k_fmm_leaf(Geo g, int L, double x0, double y0, double D, int* leaf, int* cnt) {
  const int nb = 1 << L;
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < g.M; i += gridDim.x * blockDim.x) {
    int ix = (int)((g.x[i] - x0) / D * nb), iy = (int)((g.y[i] - y0) / D * nb);
    ix = min(max(ix, 0), nb - 1);
    iy = min(max(iy, 0), nb - 1);
    const int b = iy * nb + ix;
    leaf[i] = b;
    atomicAdd(&cnt[b], 1);
  }
}

// Exclusive scan of n counts into start[0..n] (one block of 1024 threads).
__global__ void k_fmm_scan(const int* cnt, int n, int* start) {
  __shared__ int part[1024];
  const int t = threadIdx.x;
  const int per = (n + 1023) / 1024;
  const int b0 = t * per, b1 = min(n, b0 + per);
  int s = 0;
  for (int i = b0; i < b1; ++i) s += cnt[i];
  part[t] = s;
  __syncthreads();
  if (t == 0) {
    int acc = 0;
    for (int k = 0; k < 1024; ++k) {
      const int v = part[k];
      part[k] = acc;
      acc += v;
    }
    start[n] = acc;
  }
  __syncthreads();
  int acc = part[t];
  for (int i = b0; i < b1; ++i) {
    start[i] = acc;
    acc += cnt[i];
  }
}

__global__ void k_fmm_scatter(int M, const int* leaf, const int* start, int* cursor, int* tmp) {
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < M; i += gridDim.x * blockDim.x) {
    const int b = leaf[i];
    tmp[start[b] + atomicAdd(&cursor[b], 1)] = i;
  }
}

// Within each leaf, put the nodes in increasing node order (rank by counting).
__global__ void k_fmm_order(const int* start, const int* tmp, int* perm) {
  const int b = blockIdx.x;
  const int s0 = start[b], n = start[b + 1] - s0;
  for (int j = threadIdx.x; j < n; j += blockDim.x) {
    const int v = tmp[s0 + j];
    int rank = 0;
    for (int k = 0; k < n; ++k) rank += tmp[s0 + k] < v;
    perm[s0 + rank] = v;
  }
}

// Points per box on every level: leaves from start, parents from children.
__global__ void k_fmm_leaf_counts(const int* start, int nleaf, int* count_leaf) {
  for (int b = blockIdx.x * blockDim.x + threadIdx.x; b < nleaf; b += gridDim.x * blockDim.x)
    count_leaf[b] = start[b + 1] - start[b];
}
__global__ void k_fmm_parent_counts(int l, int* count) {
  const int n = 1 << l;
  const long long off = lev_off(l), offc = lev_off(l + 1);
  for (int b = blockIdx.x * blockDim.x + threadIdx.x; b < n * n; b += gridDim.x * blockDim.x) {
    const int bx = b % n, by = b / n;
    const int nc = 2 * n;
    int s = 0;
    for (int c = 0; c < 4; ++c) s += count[offc + (2 * by + (c >> 1)) * nc + 2 * bx + (c & 1)];
    count[off + b] = s;
  }
}

// ------------------------------------------------------------------ apply ----
// Densities: Laplace q = sw v (real); Stokes q = sw (v1 + i v2), conj(q),
// q conj(z - c0) with c0 the centre of the bounding square (the Stokes
// combination cancels conj(z_a) S2 against S3, so smaller |z - c0| keeps the
// expansion error of S3 small).
__global__ void k_fmm_density(Geo g, int nd, double cx0, double cy0, VecRef vr, const double* __restrict__ sscale,
                              double2* Q, const int* stop) {
  if (stop && *stop) return;
  const double* v = vr.ptr();
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < g.M; i += gridDim.x * blockDim.x) {
    if (nd == 1) {
      Q[i] = make_double2(sscale[i] * v[i], 0.0);
    } else {
      const double2 q = make_double2(sscale[i] * v[2 * i], sscale[i] * v[2 * i + 1]);
      Q[3 * i] = q;
      Q[3 * i + 1] = cconj(q);
      Q[3 * i + 2] = cmul(q, make_double2(g.x[i] - cx0, -(g.y[i] - cy0)));
    }
  }
}

// The P2M terms of one chunk of m sources: output e = d p + k (channel d,
// coefficient k) is owned by thread e mod kB, which adds its terms in source
// order (fixed: deterministic).  All p nd outputs run in parallel (p = 18,
// nd = 3: 54 of 64 threads), each a chain of m complex multiply-adds.
constexpr int kP2MAcc = (kMaxNd * kMaxP + kB - 1) / kB;  // outputs a thread keeps
template <class T2>
__device__ __forceinline__ void p2m_chunk(T2* acc, const T2* pw, const T2* qs, int p, int nd, int m) {
  const int np = p * nd;
#pragma unroll
  for (int u = 0; u < kP2MAcc; ++u) {
    const int e = threadIdx.x + u * kB;
    if (e < np) {
      const int d = e / p, k = e - d * p;
      const T2* pk = pw + k * (kChunk + 1);
      T2 a = acc[u];
      for (int j = 0; j < m; ++j) cfma(a, pk[j], qs[j * nd + d]);
      acc[u] = a;
    }
  }
}

// Leaf centres split as float hi + lo, once per tree (FP64 arithmetic here,
// so that the FP32 passes form u = (z - c)/s from the hi/lo split of z in
// FP32 with no FP64 instruction: z_hi - c_hi is exact for a node inside the
// leaf unless |z| is of the order of s).
__global__ void k_fmm_leaf_centers(int nb, double x0, double y0, double s, float4* cen) {
  for (int b = blockIdx.x * blockDim.x + threadIdx.x; b < nb * nb; b += gridDim.x * blockDim.x) {
    const double cx = x0 + (b % nb + 0.5) * s, cy = y0 + (b / nb + 0.5) * s;
    const float hx = (float)cx, hy = (float)cy;
    cen[b] = make_float4(hx, hy, (float)(cx - (double)hx), (float)(cy - (double)hy));
  }
}

// The block's leaf centre split (x_h, y_h, x_l, y_l), 1/s and s in shared memory.
__device__ __forceinline__ void leaf_center32(const FmmDevT<float2>& f, int b, float* cen) {
  if (threadIdx.x == 0) {
    const float4 c = f.cen32[b];
    cen[0] = c.x;
    cen[1] = c.y;
    cen[2] = c.z;
    cen[3] = c.w;
    cen[4] = f.is32;
    cen[5] = f.s32;
  }
}

// P2M of the FP32 expansions (inner solves): positions from the hi/lo split, and the
// strengths q = sqrt(w) v in FP32 (Laplace: (q, 0); Stokes: the complex density; the
// other channels are formed where they are used), formed here, where each source
// is read once, and kept in Qf for the near field (a launch of its own was 3 us).
// With few outputs (np = nd p <= 32) the threads are groups of np that take every
// G-th source, added in order: FP32 Laplace, order 15, 1,024 leaves
// 16.2 + 3.4 -> 12.3 us; Stokes, order 18, 16,384 leaves 32.7 + 8.0 -> 36.3 us.
__global__ void __launch_bounds__(kB) k_fmm_p2m32(FmmDevT<float2> f, Geo g, VecRef vr, const double* __restrict__ sscale,
                                                  float2* __restrict__ Qf, const int* stop) {
  if (stop && *stop) return;
  extern __shared__ __align__(16) unsigned char smraw[];
  float2* pw = reinterpret_cast<float2*>(smraw);  // [p][kChunk + 1]
  float2* qs = pw + f.p * (kChunk + 1);            // [kChunk][nd]
  __shared__ float cen[6];
  __shared__ float2 red[kB];
  const double* __restrict__ v = vr.ptr();
  const int b = blockIdx.x;
  const long long box = lev_off(f.L) + b;
  const int s0 = f.start[b], n = f.start[b + 1] - s0;
  if (n == 0) return;
  leaf_center32(f, b, cen);
  __syncthreads();
  const int t = threadIdx.x, np = f.nd * f.p, G = kB / np;
  const int grp = G > 1 ? t / np : 0, e = t - grp * np, d = e / f.p, k = e - d * f.p;  // G > 1
  float2 acc[kP2MAcc];
#pragma unroll
  for (int u = 0; u < kP2MAcc; ++u) acc[u] = make_float2(0.f, 0.f);
  for (int ch = 0; ch < n; ch += kChunk) {
    const int m = min(kChunk, n - ch);
    if (t < m) {
      const int i = f.perm[s0 + ch + t];
      const float4 P = g.pf[i];
      const double sw = sscale[i];
      float2 q;
      if (f.nd == 1)
        q = make_float2((float)(sw * v[i]), 0.f);
      else
        q = make_float2((float)(sw * v[2 * i]), (float)(sw * v[2 * i + 1]));
      Qf[i] = q;
      const float2 u = make_float2(((P.x - cen[0]) + (P.z - cen[2])) * cen[4], ((P.y - cen[1]) + (P.w - cen[3])) * cen[4]);
      float2 w = make_float2(1.f, 0.f);
      for (int r = 0; r < f.p; ++r) {
        pw[r * (kChunk + 1) + t] = w;
        w = cmul(w, u);
      }
      qs[t * f.nd] = q;
      if (f.nd == 3) {
        qs[t * 3 + 1] = make_float2(q.x, -q.y);
        // channel cm = 2: q conj(u), the leaf-relative moment density
        qs[t * 3 + 2] = make_float2(q.x * u.x + q.y * u.y, q.y * u.x - q.x * u.y);
      }
    }
    __syncthreads();
    if (G > 1) {
      if (grp < G)
        for (int j = grp; j < m; j += G) cfma(acc[0], pw[k * (kChunk + 1) + j], qs[j * f.nd + d]);
    } else {
      p2m_chunk(acc, pw, qs, f.p, f.nd, m);
    }
    __syncthreads();
  }
  if (G > 1) {
    red[t] = acc[0];
    __syncthreads();
    if (t < np) {
      for (int q = 1; q < G; ++q) acc[0] = cadd(acc[0], red[q * np + t]);
      f.mp[box * np + t] = acc[0];
    }
    return;
  }
#pragma unroll
  for (int u = 0; u < kP2MAcc; ++u)
    if (t + u * kB < np) f.mp[box * np + t + u * kB] = acc[u];
}

// P2M on the leaves: a_k = sum_j q_j u_j^k, u = (z - c)/s.
template <class T2>
__global__ void __launch_bounds__(kB) k_fmm_p2m(FmmDevT<T2> f, Geo g, const int* stop) {
  if (stop && *stop) return;
  extern __shared__ __align__(16) unsigned char smraw[];
  T2* sm = reinterpret_cast<T2*>(smraw);
  T2* pw = sm;                       // [p][kChunk + 1]
  T2* qs = sm + f.p * (kChunk + 1);  // [kChunk][nd]
  const int b = blockIdx.x;
  const long long box = lev_off(f.L) + b;
  const int s0 = f.start[b], n = f.start[b + 1] - s0;
  if (n == 0) return;
  double s;
  const double2 c = box_center(f, f.L, b % f.nb, b / f.nb, s);
  const int t = threadIdx.x;
  T2 acc[kP2MAcc];
#pragma unroll
  for (int u = 0; u < kP2MAcc; ++u) acc[u] = cx<T2>(0.0, 0.0);
  for (int ch = 0; ch < n; ch += kChunk) {
    const int m = min(kChunk, n - ch);
    if (t < kChunk) {
      if (t < m) {
        const int i = f.perm[s0 + ch + t];
        const double is = ldexp(f.Dinv, f.L);
        const T2 u = cx<T2>((g.x[i] - c.x) * is, (g.y[i] - c.y) * is);
        T2 w = cx<T2>(1.0, 0.0);
        for (int k = 0; k < f.p; ++k) {
          pw[k * (kChunk + 1) + t] = w;
          w = cmul(w, u);
        }
        for (int d = 0; d < f.nd; ++d) {
          const double2 q = f.Q[(long long)i * f.nd + (d == f.cm ? 0 : d)];
          // channel cm: q conj(u), the leaf-relative moment density
          qs[t * f.nd + d] = d == f.cm ? cx<T2>(q.x * (double)u.x + q.y * (double)u.y,
                                                q.y * (double)u.x - q.x * (double)u.y)
                                       : cx<T2>(q.x, q.y);
        }
      }
    }
    __syncthreads();
    p2m_chunk(acc, pw, qs, f.p, f.nd, m);
    __syncthreads();
  }
#pragma unroll
  for (int u = 0; u < kP2MAcc; ++u)
    if (t + u * kB < f.nd * f.p) f.mp[box * f.nd * f.p + t + u * kB] = acc[u];
}

// Shifts between a box and its children.  With u_P = u_C/2 + w_c, w_c = (+-1 +- i)/4,
//   M2M: a'_k = sum_c sum_{m <= k} C(k, m) w_c^(k-m) 2^-m a^(c)_m,
//   L2L: b^(c)_k = sum_{m >= k} C(m, k) w_c^(m-k) 2^-k b_m.
// The children are quarter turns of each other, w_r = i^r w, w = |w| e^(i pi/4), so
// one real matrix serves all four both ways: with e^(i pi m/4) = h^(m mod 2) g_m,
// h = 2^-1/2, g_m = i^(m div 2) (1 + i)^(m mod 2) (turns and additions only), and
//   T[m][k] = C(max, min) |w|^|k-m| 2^-min h^(m mod 2) h^(k mod 2):
//   a'_k = g_k sum_{m <= k} T[m][k] conj(g_m) A_m^((k-m) mod 4),  A^(q)_m = sum_r i^(rq) a^(r)_m,
//   b^(r)_k = conj(g_k) sum_j i^(rj) S_j[k],  S_j[k] = sum_{m >= k, m = k+j mod 4} T[m][k] g_m b_m.
// That is 1/8 of the multiply-adds of four complex matrices, and no matrix to stage.
// Both kernels, for orders p <= PK: thread (m mod 4, channel, k) keeps its column of T in
// registers for all levels and adds the terms of its residue of m; the four sums
// meet in shared memory.  (Run-time sizes took twice the instructions.)
__device__ __forceinline__ int child_of_turn(int r) { return r == 0 ? 3 : r == 1 ? 2 : r == 2 ? 0 : 1; }
__device__ __forceinline__ int turn_of_child(int c) { return c == 3 ? 0 : c == 2 ? 1 : c == 0 ? 2 : 3; }

// i^j z
template <class T2>
__device__ __forceinline__ T2 turned(T2 z, int j) {
  T2 v = z;
  if (j & 1) {
    v.x = -z.y;
    v.y = z.x;
  }
  if (j & 2) {
    v.x = -v.x;
    v.y = -v.y;
  }
  return v;
}
// g_m z and conj(g_m) z
template <class T2>
__device__ __forceinline__ T2 eighth(T2 z, int m) {
  if (m & 1) {
    const auto x = z.x;
    z.x = x - z.y;
    z.y = x + z.y;
  }
  return turned(z, (m >> 1) & 3);
}
template <class T2>
__device__ __forceinline__ T2 eighth_conj(T2 z, int m) {
  if (m & 1) {
    const auto x = z.x;
    z.x = x + z.y;
    z.y = z.y - x;
  }
  return turned(z, -(m >> 1) & 3);
}
// x_r = sum_j i^(rj) v_j
template <class T2>
__device__ __forceinline__ void quarter_sums(T2* v) {
  const T2 s02 = cadd(v[0], v[2]), d02 = cadd(v[0], turned(v[2], 2));
  const T2 s13 = cadd(v[1], v[3]), d13 = turned(cadd(v[1], turned(v[3], 2)), 1);
  v[0] = cadd(s02, s13);
  v[1] = cadd(d02, d13);
  v[2] = cadd(s02, turned(s13, 2));
  v[3] = cadd(d02, turned(d13, 2));
}
inline int shift_threads(int nd, int p) { return (4 * nd * p + 31) / 32 * 32; }
// of up to nc channels of order pk
__host__ __device__ constexpr int shift_max_threads(int nc, int pk) { return (4 * nc * pk + 31) / 32 * 32; }
// blocks an SM that the registers have to leave room for (more of them spill)
template <class T2>
constexpr int shift_blocks(int nc, int pk) {
  return (sizeof(T2) == 8 ? 1536 : nc == 1 ? 640 : 1152) / shift_max_threads(nc, pk);
}
template <class T2>
size_t shift_smem(int nd, int pk) {
  return (size_t)8 * nd * (pk + 1) * sizeof(T2);
}

// M2M of all levels L-1..2 in one launch: a block forms one box of level L-1 (in a mostly
// empty tree several), and the block that completes the last of four siblings (there: of those
// with sources) goes on with their parent (no block waits; arrive[] counts the siblings and
// is back at 0 at the end).
// Each level was a launch of one 64-thread block a box, the children one after
// the other with their matrices staged: all levels, FP32 Laplace, 1,024 leaves, order
// 15: 31 -> 9.0 us; FP32 Stokes, 16,384 leaves, order 18: 83 -> 35 us; FP64 Stokes, order
// 36: 995 -> 222 us (L2L: 17 -> 6.8, 49 -> 31 and 700 -> 235 us).  What is left is the
// chain of levels (2-3 us each), in FP64 the FP64 pipe.
template <class T2, int NC, int PK, bool MANY>
__global__ void __launch_bounds__(shift_max_threads(NC, PK), shift_blocks<T2>(NC, PK))
k_fmm_m2m(FmmDevT<T2> f, int* arrive, const int* stop) {
  using R = decltype(T2{}.x);
  if (stop && *stop) return;
  extern __shared__ __align__(16) unsigned char smraw[];
  const int p = f.p, np = f.nd * p, US = f.nd * (PK + 1), t = threadIdx.x;
  T2* U = reinterpret_cast<T2*>(smraw);  // [q][channel][m], channels PK + 1 apart
  T2* red = U + 4 * US;                  // [residue][channel, k]
  __shared__ int s_last;
  const int e = t % np, mr = t / np, d = e / p, k = e - d * p;
  R T[PK / 4];
#pragma unroll
  for (int i = 0; i < PK / 4; ++i) {
    const int m = mr + 4 * i;
    T[i] = m <= k && mr < 4 ? __ldg(reinterpret_cast<const R*>(f.ops) + m * p + k) : (R)0;
  }
  for (int w = t; w < 4 * f.nd * (PK + 1 - p); w += blockDim.x)  // the padding
    U[w / (PK + 1 - p) * (PK + 1) + p + w % (PK + 1 - p)] = cx<T2>(0.0, 0.0);
  const long long boxes = 1LL << (2 * (f.L - 1));
  for_boxes<MANY>(f.count + lev_off(f.L - 1), boxes, f.per, [&](long long first) {
    int b = (int)first;
    for (int l = f.L - 1;; --l) {
      const int n = 1 << l, bx = b & (n - 1), by = b >> l;
      const long long box = lev_off(l) + b;
      if (MANY || f.count[box] > 0) {
        if (t < np) {
          // other blocks of this launch wrote the children above the first level: past L1
          T2 v[4];
#pragma unroll
          for (int r = 0; r < 4; ++r) {
            const int c = child_of_turn(r);
            const long long child = lev_off(l + 1) + (long long)(2 * by + (c >> 1)) * (2 * n) + 2 * bx + (c & 1);
            v[r] = cx<T2>(0.0, 0.0);
            if (f.count[child] > 0) v[r] = __ldcg(f.mp + child * np + e);
          }
          quarter_sums(v);
#pragma unroll
          for (int q = 0; q < 4; ++q) U[q * US + d * (PK + 1) + k] = eighth_conj(v[q], k);
        }
        __syncthreads();
        if (f.cm >= 0) {
          // child moment density relative to the parent centre: 1/2 rho_r + conj(w_r) a_r, whose
          // transform is 1/2 that of rho plus conj(w) times that of a, one place back
          if (t < 4 * p) {
            const int q = t / p, m = t - q * p;
            T2 a = U[q * US + f.cm * (PK + 1) + m];
            a.x *= R(0.5);
            a.y *= R(0.5);
            cfma(a, cx<T2>(0.25, -0.25), U[((q + 3) & 3) * US + m]);
            U[q * US + f.cm * (PK + 1) + m] = a;
          }
          __syncthreads();
        }
        if (mr < 4) {
          T2 acc = cx<T2>(0.0, 0.0);
          const T2* u = U + ((k - mr) & 3) * US + d * (PK + 1) + mr;
#pragma unroll
          for (int i = 0; i < PK / 4; ++i) {
            const T2 x = u[4 * i];
            acc.x = fma(T[i], x.x, acc.x);
            acc.y = fma(T[i], x.y, acc.y);
          }
          red[t] = acc;
        }
        __syncthreads();
        if (t < np) {
          const T2 a = cadd(cadd(red[t], red[np + t]), cadd(red[2 * np + t], red[3 * np + t]));
          f.mp[box * np + t] = eighth(a, k);
        }
      }
      if (l == 2) return;
      __syncthreads();
      b = (by >> 1) * (n >> 1) + (bx >> 1);
      if (t == 0) {
        __threadfence();  // the block's stores, ordered before it by the barrier
        int* a = arrive + lev_off(l - 1) + b;
        int siblings = 4;  // the boxes that arrive
        if (MANY) {        // only those with sources
          const int* c = f.count + lev_off(l) + (by & ~1) * n + (bx & ~1);
          siblings = (c[0] > 0) + (c[1] > 0) + (c[n] > 0) + (c[n + 1] > 0);
        }
        s_last = atomicAdd(a, 1) == siblings - 1;
        if (s_last) *a = 0;
        __threadfence();
      }
      __syncthreads();
      if (!s_last) return;
    }
  });
}

// M2L for the target boxes of all levels 2..L (one block per box), through
// a factorisation of the translation operators (d = D s, D the integer
// offset of the target centre from the source centre in box sides):
//   Cauchy:    T_D[l][k] = (-1)^l C(k+l, l) D^-(k+l+1) = beta_l(D) P[l][k] alpha_k(D),
//              P[l][k] = C(k+l, l),  alpha_k = D^-k,  beta_l = (-1)^l D^-(l+1);
//   logarithm: T^log_D[l][k] = beta_l(D) P^log[l][k] alpha_k(D) for k >= 1,
//              P^log[l][k] = C(k+l-1, l),  alpha_k = D^-k / k,  beta_l = -(-1)^l D^-l,
//              and the a_0 column gamma_l(D) = log D (l = 0), (-1)^(l+1) D^-l / l (l >= 1).
// P is real and the same for every offset.  Cauchy channels carry 1/s;
// logarithm channels add a_0 log(s) on b_0 (the level's share of log d = log D +
// log s).
//
// Quarter turns: for D_r = i^r D the factors turn by powers of i, so the up to
// four sources at D, iD, -D, -iD need one Pascal product instead of four:
//   sum_r T_{D_r} a^(r) |_l = beta_l(D) sum_k P[l][k] alpha_k(D) A_k^((l + e + k) mod 4),
//   A_k^(q) = sum_r i^(-rq) a_k^(r)   (e = 1 Cauchy, 0 logarithm),
// the sources' 4-point transform (additions only), and row l uses the entries of
// residue l + e + k.  The 27 offsets of an interaction list fall into 10 such
// orbits (4 whole ones, 5 of two sources, 1 of one), which cuts the p x p products
// by 2.7.  A product costs 2 p^2 real multiply-adds a channel.
//
// A block lists the orbits that have non-empty sources (s_src: four source boxes
// an orbit), stages alpha_k A_k^(q) of up to nbo orbits in shared memory (U[orbit][channel,
// k][q]), and thread (split, channel, row) adds NJ of its split's orbits at a
// time (independent chains); the splits' sums are added in order.
//
// Against one product a source (the Pascal row in registers): FP64 Laplace,
// 160,000 nodes, order 36: 1448 -> 468 us; float-float Stokes, 640,000 nodes, order
// 36: 4100 -> 2066 us (bound by FP32 issue); FP32 Stokes, order 18: 209 -> 127 us.
constexpr int kOffs = 49;     // offsets -3..3 x -3..3 (the 3 x 3 near ones unused)
constexpr int kOrbits = 10;   // orbits of the others under quarter turns

// The orbit of offset (x, y) and the quarter turns r from its representative (x > 0, y >= 0).
__device__ __forceinline__ void orbit_of(int x, int y, int& id, int& r) {
  r = 0;
  while (!(x > 0 && y >= 0)) {  // at most three turns by -i
    const int t = x;
    x = y;
    y = -t;
    ++r;
  }
  id = max(x, y) == 2 ? (x == 2 ? y : 3) : (x == 3 ? 4 + y : (x == 2 ? 8 : 9));
}
// Offset of an orbit's representative.
__device__ __forceinline__ int2 orbit_rep(int id) {
  if (id < 4) return id < 3 ? make_int2(2, id) : make_int2(1, 2);
  return id < 8 ? make_int2(3, id - 4) : make_int2(id == 8 ? 2 : 1, 3);
}
__device__ __forceinline__ int offset_index(int x, int y) { return (x + 3) + 7 * (y + 3); }

struct OrbitList {
  int src[kOrbits][4];  // source box (in its level) at i^r D, or -1
  int id[kOrbits];      // the orbits with a source, in order
  int cnt;
};

// The orbits of target box (bx, by) of level l (all threads of the block call).
template <class T2>
__device__ __forceinline__ void list_orbits(const FmmDevT<T2>& f, int l, int bx, int by, OrbitList& o) {
  const int n = 1 << l, px = bx >> 1, py = by >> 1;
  for (int c = threadIdx.x; c < 4 * kOrbits; c += blockDim.x) (&o.src[0][0])[c] = -1;
  __syncthreads();
  for (int c = threadIdx.x; c < 36; c += blockDim.x) {
    const int sx = 2 * px - 2 + c % 6, sy = 2 * py - 2 + c / 6;
    if (sx < 0 || sy < 0 || sx >= n || sy >= n || (abs(sx - bx) <= 1 && abs(sy - by) <= 1)) continue;
    if (f.count[lev_off(l) + (long long)sy * n + sx] == 0) continue;
    int id, r;
    orbit_of(bx - sx, by - sy, id, r);
    o.src[id][r] = sy * n + sx;
  }
  __syncthreads();
  if (threadIdx.x < 32) {
    const int t = threadIdx.x;
    const bool any = t < kOrbits && (o.src[t][0] >= 0 || o.src[t][1] >= 0 || o.src[t][2] >= 0 || o.src[t][3] >= 0);
    const unsigned m = __ballot_sync(0xffffffffu, any);
    if (any) o.id[__popc(m & ((1u << t) - 1u))] = t;
    if (t == 0) o.cnt = __popc(m);
  }
  __syncthreads();
}

// Layout of the operator table of order p (complex entries): the child shifts'
// matrix T[m][k] (p^2 reals), then the M2L factors alpha[2][49][p], beta[2][49][p],
// gamma[49][p] and the Pascal matrices [2][k][l] (real, in the real parts);
// type 0 = Cauchy, 1 = logarithm, offset index (Dx + 3) + 7 (Dy + 3).
__host__ __device__ inline long long tab_alpha(int p) { return ((long long)p * p + 1) / 2; }
__host__ __device__ inline long long tab_beta(int p) { return tab_alpha(p) + 2LL * kOffs * p; }
__host__ __device__ inline long long tab_gamma(int p) { return tab_beta(p) + 2LL * kOffs * p; }
__host__ __device__ inline long long tab_pascal(int p) { return tab_gamma(p) + (long long)kOffs * p; }
__host__ __device__ inline long long tab_size(int p) { return tab_pascal(p) + 2LL * p * p; }

// w += (pp.x u.x, pp.y u.y): a real factor (duplicated in pp) times a complex value
__device__ __forceinline__ void rfma(double2& w, double2 pp, double2 u) {
  w.x = fma(pp.x, u.x, w.x);
  w.y = fma(pp.y, u.y, w.y);
}

// alpha_k A_k^(q), q = 0..3, of orbit id for (channel d, coefficient k): the four
// sources' coefficients (moment channel: relative to the target centre, rho_S -
// conj(D_r) rho_0), their 4-point transform, times alpha.
template <class T2>
__device__ __forceinline__ void orbit_stage(const FmmDevT<T2>& f, const OrbitList& o, int id, int l, int d, int k,
                                            const T2* __restrict__ al, T2* __restrict__ out, T2* __restrict__ a0) {
  const int p = f.p, nd = f.nd;
  const int2 D = orbit_rep(id);
  int x = D.x, y = D.y;
  T2 v[4];
#pragma unroll
  for (int r = 0; r < 4; ++r) {
    v[r] = cx<T2>(0.0, 0.0);
    if (o.src[id][r] >= 0) {
      const T2* a = f.mp + (lev_off(l) + o.src[id][r]) * nd * p;
      v[r] = a[d * p + k];
      if (d == f.cm) cfma(v[r], cx<T2>((double)-x, (double)y), a[k]);
    }
    const int t = x;  // the next turn by i
    x = -y;
    y = t;
  }
  const T2 t0 = cadd(v[0], v[2]), t2 = cadd(v[1], v[3]);
  T2 t1 = v[0], t3 = v[1];
  t1.x -= v[2].x;
  t1.y -= v[2].y;
  t3.x -= v[3].x;
  t3.y -= v[3].y;
  T2 A[4];
  A[0] = cadd(t0, t2);
  A[1] = t1;  // t1 - i t3
  A[1].x += t3.y;
  A[1].y -= t3.x;
  A[2] = t0;
  A[2].x -= t2.x;
  A[2].y -= t2.y;
  A[3] = t1;  // t1 + i t3
  A[3].x -= t3.y;
  A[3].y += t3.x;
  if (a0)
#pragma unroll
    for (int q = 0; q < 4; ++q) a0[q] = A[q];
  const T2 w = al[(long long)offset_index(D.x, D.y) * p];
#pragma unroll
  for (int q = 0; q < 4; ++q) out[q] = cmul(w, A[q]);
}

// FP64.  Threads: split x (channel, row).
template <class T2, int NJ>
__device__ __forceinline__ void m2l_box(const FmmDevT<T2>& f, long long gb, int nsplit, int nbo) {
  using R = decltype(T2{}.x);
  extern __shared__ __align__(16) unsigned char smraw[];
  __shared__ OrbitList o;
  __shared__ T2 s_a0[kOrbits][kMaxNd][4];  // the transforms of a_0 of the logarithm channels
  __shared__ T2 red[256];
  int l = 2;
  while (l < f.L && gb >= lev_off(l + 1)) ++l;
  if (f.tcount[gb] == 0) return;
  const int p = f.p, nd = f.nd, per = nd * p;
  const int b = (int)(gb - lev_off(l)), bx = b & ((1 << l) - 1), by = b >> l;
  const int tid = threadIdx.x;
  list_orbits(f, l, bx, by, o);
  T2* U = reinterpret_cast<T2*>(smraw);               // [nbo][nd p][4]
  R* Pt = reinterpret_cast<R*>(U + (long long)nbo * per * 4);  // [type][k][l]
  const T2* alpha = f.ops + tab_alpha(p);
  const T2* beta = f.ops + tab_beta(p);
  const T2* gamma = f.ops + tab_gamma(p);
  const T2* pas = f.ops + tab_pascal(p);
  const int ntype = f.nlog > 0 ? 2 : 1;
  for (int e = tid; e < ntype * p * p; e += blockDim.x) Pt[e] = pas[e].x;
  const int sp = tid / per, e = tid - sp * per, d = e / p, t = e - d * p;
  const bool act = sp < nsplit;
  const int ty = d < f.nlog ? 1 : 0;
  const int base = t + 1 - ty;  // the residue of the entry at k: (base + k) mod 4
  T2 acc = cx<T2>(0.0, 0.0);
  for (int o0 = 0; o0 < o.cnt; o0 += nbo) {
    const int no = min(nbo, o.cnt - o0);
    __syncthreads();
    for (int q = tid; q < no * per; q += blockDim.x) {
      const int oo = q / per, dk = q - oo * per, dd = dk / p, k = dk - dd * p;
      const int tt = dd < f.nlog ? 1 : 0;
      orbit_stage(f, o, o.id[o0 + oo], l, dd, k, alpha + (long long)tt * kOffs * p + k, U + 4LL * q,
                  tt == 1 && k == 0 ? s_a0[o0 + oo][dd] : (T2*)nullptr);
    }
    __syncthreads();
    if (!act) continue;
    for (int q0 = sp; q0 < no; q0 += NJ * nsplit) {
      T2 w[NJ];
      const T2* u[NJ];
#pragma unroll
      for (int j = 0; j < NJ; ++j) {
        w[j] = cx<T2>(0.0, 0.0);
        u[j] = U + (long long)min(q0 + j * nsplit, no - 1) * per * 4 + d * p * 4;
      }
      const R* pt = Pt + (long long)ty * p * p + t;
      for (int k = 0; k < p; ++k) {
        const R pv = pt[(long long)k * p];
        const T2 pp = cx<T2>((double)pv, (double)pv);
        const int at = 4 * k + ((base + k) & 3);
#pragma unroll
        for (int j = 0; j < NJ; ++j) rfma(w[j], pp, u[j][at]);
      }
#pragma unroll
      for (int j = 0; j < NJ; ++j) {
        const int q = q0 + j * nsplit;
        if (q < no) {
          const int id = o.id[o0 + q];
          const int2 D = orbit_rep(id);
          const int oi = offset_index(D.x, D.y);
          cfma(acc, beta[((long long)ty * kOffs + oi) * p + t], w[j]);
          if (ty == 1 && t > 0) cfma(acc, gamma[(long long)oi * p + t], s_a0[o0 + q][d][t & 3]);
          if (ty == 1 && t == 0) {
            // a_0 (log D_r + log s) per source, s = D 2^-l
            const R logs = (R)(log(f.D) - l * 0.69314718055994530942);
            int x = D.x, y = D.y;
            for (int r = 0; r < 4; ++r) {
              if (o.src[id][r] >= 0) {
                T2 gm = gamma[(long long)offset_index(x, y) * p];
                gm.x += logs;
                cfma(acc, gm, f.mp[((lev_off(l) + o.src[id][r]) * nd + d) * p]);
              }
              const int z = x;
              x = -y;
              y = z;
            }
          }
        }
      }
    }
  }
  red[tid] = acc;
  __syncthreads();
  if (sp == 0) {
    for (int q = 1; q < nsplit; ++q) acc = cadd(acc, red[q * per + e]);
    // Cauchy channels carry 1/s; in the precision of the expansions
    const R sc = ty == 1 ? (R)1 : (R)ldexp(f.Dinv, l);
    acc.x *= sc;
    acc.y *= sc;
    f.lc[gb * per + e] = acc;
  }
}

template <class T2, int NJ, bool MANY>
__global__ void __launch_bounds__(256) k_fmm_m2l(FmmDevT<T2> f, int nsplit, int nbo, const int* stop) {
  if (stop && *stop) return;
  for_boxes<MANY>(f.tcount + lev_off(2), lev_off(f.L + 1) - lev_off(2), f.tper,
                  [&](long long b) { m2l_box<T2, NJ>(f, b + lev_off(2), nsplit, nbo); });
}

// FP32, Cauchy channels (the inner solves' operator), ND channels of order p <= PK
// (coefficients padded with zeros to the instance's order).  Bound by instruction
// issue (71%), so the work around the multiply-adds is what counts:
// - a thread takes two rows of one residue, l and l + 4: both use the same staged
//   entries, so that a load feeds four multiply-adds; their Pascal entries come in
//   pairs from a table of that layout (fmm_setup);
// - all ten orbits are staged, in one pass in which a thread forms one coefficient
//   of all channels (12 loads in flight for three), empty sources as zeros: the
//   moment channel's shift is one multiply-add a transform instead of one a source;
// - sizes and strides are compile-time constants (run-time ones: 241 us in place of 127).
__host__ __device__ constexpr int m2l32_rp(int pk) { return (pk + 7) / 8; }  // row pairs of one residue
// the instance of an order
__host__ __device__ constexpr int m2l32_pad(int p) {
  return p <= 12 ? 12 : p <= 16 ? 16 : p <= 20 ? 20 : p <= 24 ? 24 : p <= 32 ? 32 : p <= 48 ? 48 : 64;
}

__host__ __device__ constexpr int m2l32_splits(int nd, int pk) {
  return 5 * nd * 4 * m2l32_rp(pk) <= 256 ? 5 : (2 * nd * 4 * m2l32_rp(pk) <= 256 ? 2 : 1);
}
__host__ __device__ constexpr int m2l32_threads(int nd, int pk) {
  return (m2l32_splits(nd, pk) * nd * 4 * m2l32_rp(pk) + 31) / 32 * 32;
}

template <int ND, int PK>
__device__ __forceinline__ void m2l32_box(const FmmDevT<float2>& f, long long gb, const float2* __restrict__ ptab) {
  constexpr int RP = m2l32_rp(PK), SP = m2l32_splits(ND, PK), B = m2l32_threads(ND, PK);
  constexpr int HALF = ND * 4 * RP, NJ = 2;  // (channel, residue, pair) threads; orbits added at a time
  constexpr int DS = 4 * PK + 4, US = ND * DS;  // channel and orbit strides: distinct banks
  extern __shared__ __align__(16) float2 U[];   // [orbit][channel][k][4]
  __shared__ int s_at[kOrbits * 4];             // the sources' first coefficients, or -1
  __shared__ float4 red[B];
  int l = 2;
  while (l < f.L && gb >= lev_off(l + 1)) ++l;
  const int targets = f.tcount[gb];
  const int p = f.p, n = 1 << l, tid = threadIdx.x;
  {
    const int b = (int)(gb - lev_off(l)), bx = b & (n - 1), by = b >> l;
    for (int t = tid; t < 4 * kOrbits; t += B) {
      const int2 D = orbit_rep(t >> 2);
      const int r = t & 3, dx = r == 0 ? D.x : r == 1 ? -D.y : r == 2 ? -D.x : D.y;
      const int dy = r == 0 ? D.y : r == 1 ? D.x : r == 2 ? -D.y : -D.x;
      const int sx = bx - dx, sy = by - dy;  // a child of the parent's neighbours, in the level
      const bool in = sx >= 0 && sy >= 0 && sx < n && sy < n && abs((sx >> 1) - (bx >> 1)) <= 1 &&
                      abs((sy >> 1) - (by >> 1)) <= 1;
      s_at[t] = in && f.count[lev_off(l) + (long long)sy * n + sx] > 0 ? (sy * n + sx) * (ND * p) : -1;
    }
  }
  if (targets == 0) return;
  __syncthreads();
  const float2* __restrict__ mp = f.mp + lev_off(l) * ND * p;
  for (int w = tid; w < kOrbits * p; w += B) {
    const int oo = w / p, k = w - oo * p;
    const int2 D = orbit_rep(oo);
    const float2 w4 = __ldg(f.ops + tab_alpha(p) + offset_index(D.x, D.y) * p + k);
    float2 A[ND][4];
#pragma unroll
    for (int r = 0; r < 4; ++r) {
      const int at = s_at[4 * oo + r];
#pragma unroll
      for (int d = 0; d < ND; ++d) A[d][r] = at >= 0 ? mp[at + d * p + k] : make_float2(0.f, 0.f);
    }
#pragma unroll
    for (int d = 0; d < ND; ++d) {
      const float2 t0 = cadd(A[d][0], A[d][2]), t2 = cadd(A[d][1], A[d][3]);
      const float2 t1 = make_float2(A[d][0].x - A[d][2].x, A[d][0].y - A[d][2].y);
      const float2 t3 = make_float2(A[d][1].x - A[d][3].x, A[d][1].y - A[d][3].y);
      A[d][0] = cadd(t0, t2);
      A[d][1] = make_float2(t1.x + t3.y, t1.y - t3.x);
      A[d][2] = make_float2(t0.x - t2.x, t0.y - t2.y);
      A[d][3] = make_float2(t1.x - t3.y, t1.y + t3.x);
    }
    if (ND == 3) {
      // moment channel, relative to the target centre: rho_r - conj(i^r D) a_r, whose
      // transform is that of rho less conj(D) times that of a, one place on
      const float2 c = make_float2(-(float)D.x, (float)D.y);
#pragma unroll
      for (int q = 0; q < 4; ++q) cfma(A[ND - 1][q], c, A[0][(q + 1) & 3]);
    }
#pragma unroll
    for (int d = 0; d < ND; ++d) {
      float4* u4 = reinterpret_cast<float4*>(U + oo * US + d * DS + 4 * k);
      const float2 a0 = cmul(w4, A[d][0]), a1 = cmul(w4, A[d][1]), a2 = cmul(w4, A[d][2]), a3 = cmul(w4, A[d][3]);
      u4[0] = make_float4(a0.x, a0.y, a1.x, a1.y);
      u4[1] = make_float4(a2.x, a2.y, a3.x, a3.y);
    }
  }
  for (int w = tid; w < 2 * kOrbits * ND * (PK - p); w += B)  // the padding
    reinterpret_cast<float4*>(U + (w / (2 * (PK - p))) * DS + 4 * p)[w % (2 * (PK - p))] = make_float4(0.f, 0.f, 0.f, 0.f);
  __syncthreads();
  // thread (split, channel, residue, pair): rows t0 = residue + 8 pair and t0 + 4
  const int sp = tid / HALF, e = tid % HALF, d = e / (4 * RP), mr = e % (4 * RP), m = mr / RP;
  const int t0 = m + 8 * (mr % RP), t1 = t0 + 4;
  const bool act = sp < SP && t0 < p;
  float2 acc0 = make_float2(0.f, 0.f), acc1 = acc0;
  if (act) {
    const int rot[4] = {(m + 1) & 3, (m + 2) & 3, (m + 3) & 3, m & 3};
    const float2* __restrict__ beta = f.ops + tab_beta(p) + t0;
#pragma unroll 1
    for (int q0 = sp; q0 < kOrbits; q0 += NJ * SP) {
      const int q1 = min(q0 + SP, kOrbits - 1);
      const int2 Da = orbit_rep(q0), Db = orbit_rep(q1);
      const float2* __restrict__ be = beta + offset_index(Da.x, Da.y) * p;
      const float2* __restrict__ bf = beta + offset_index(Db.x, Db.y) * p;
      const float2 z = make_float2(0.f, 0.f);
      const float2 be0 = __ldg(be), be1 = t1 < p ? __ldg(be + 4) : z;
      const float2 bf0 = q0 + SP < kOrbits ? __ldg(bf) : z, bf1 = t1 < p && q0 + SP < kOrbits ? __ldg(bf + 4) : z;
      const float2* ua = U + q0 * US + d * DS;
      const float2* ub = U + q1 * US + d * DS;
      float2 a0 = z, a1 = z, b0 = z, b1 = z;
      const float2* __restrict__ pt = ptab + mr;
#pragma unroll
      for (int k = 0; k < PK; ++k) {
        const float2 P = __ldg(pt + k * 4 * RP);
        const float2 va = ua[4 * k + rot[k & 3]], vb = ub[4 * k + rot[k & 3]];
        a0.x = fmaf(P.x, va.x, a0.x);
        a0.y = fmaf(P.x, va.y, a0.y);
        a1.x = fmaf(P.y, va.x, a1.x);
        a1.y = fmaf(P.y, va.y, a1.y);
        b0.x = fmaf(P.x, vb.x, b0.x);
        b0.y = fmaf(P.x, vb.y, b0.y);
        b1.x = fmaf(P.y, vb.x, b1.x);
        b1.y = fmaf(P.y, vb.y, b1.y);
      }
      cfma(acc0, be0, a0);
      cfma(acc1, be1, a1);
      cfma(acc0, bf0, b0);
      cfma(acc1, bf1, b1);
    }
  }
  red[tid] = make_float4(acc0.x, acc0.y, acc1.x, acc1.y);
  __syncthreads();
  if (sp == 0 && act) {
#pragma unroll
    for (int q = 1; q < SP; ++q) {
      const float4 r = red[q * HALF + e];
      acc0 = cadd(acc0, make_float2(r.x, r.y));
      acc1 = cadd(acc1, make_float2(r.z, r.w));
    }
    const float sc = (float)ldexp(f.Dinv, l);  // Cauchy channels carry 1/s
    f.lc[(gb * ND + d) * p + t0] = make_float2(acc0.x * sc, acc0.y * sc);
    if (t1 < p) f.lc[(gb * ND + d) * p + t1] = make_float2(acc1.x * sc, acc1.y * sc);
  }
}

template <int ND, int PK, bool MANY>
__global__ void __launch_bounds__(m2l32_threads(ND, PK)) k_fmm_m2l32(FmmDevT<float2> f, const float2* __restrict__ ptab,
                                                                    const int* stop) {
  if (stop && *stop) return;
  for_boxes<MANY>(f.tcount + lev_off(2), lev_off(f.L + 1) - lev_off(2), f.tper,
                  [&](long long b) { m2l32_box<ND, PK>(f, b + lev_off(2), ptab); });
}

// ---- float-float M2L: the residual operator of the float-float refinement ----
// The multipoles (FP64) are split once into float-float pairs hi + lo
// (k_fmm_mp_ff); the factorised M2L then runs on the FP32 pipe in pairs of
// lanes (real, imaginary): a Pascal entry times a source coefficient is an
// exact FP32 product plus its error term and the cross terms (about 48
// significant bits), accumulated with an error-free sum and renormalised at
// every step, and the diagonal factors alpha and beta are float-float splits
// of the FP64 tables.  Relative rounding about 2^-48 per operation, against
// 2^-53 in FP64, on a pipe that issues many times more operations; the local
// expansions are written back in FP64.  Cauchy channels only (the pair sums).
// Complex float-float values are float4 (re_hi, im_hi, re_lo, im_lo).
__global__ void k_fmm_mp_ff(const double2* __restrict__ mp, long long n, float4* __restrict__ mpff) {
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
    const double2 a = mp[i];
    const float rh = (float)a.x, ih = (float)a.y;
    mpff[i] = make_float4(rh, ih, (float)(a.x - (double)rh), (float)(a.y - (double)ih));
  }
}

__device__ __forceinline__ float2 neg2(float2 a) { return make_float2(-a.x, -a.y); }

// (ph, pl) = (ah + al)(bh + bl) lane-wise: exact leading product, its error
// and the cross terms
__device__ __forceinline__ void ff_mul2(float2 ah, float2 al, float2 bh, float2 bl, float2& ph, float2& pl) {
  ph = __fmul2_rn(ah, bh);
  pl = __ffma2_rn(ah, bh, neg2(ph));
  pl = __ffma2_rn(ah, bl, pl);
  pl = __ffma2_rn(al, bh, pl);
}

// (sh, sl) += (ph, pl) lane-wise: error-free sum of the leading parts, the
// low parts added, renormalised
__device__ __forceinline__ void ff_acc2(float2& sh, float2& sl, float2 ph, float2 pl) {
  const float2 s = __fadd2_rn(sh, ph);
  const float2 bb = __fadd2_rn(s, neg2(sh));
  const float2 e = __fadd2_rn(__fadd2_rn(sh, neg2(__fadd2_rn(s, neg2(bb)))), __fadd2_rn(ph, neg2(bb)));
  const float2 t = __fadd2_rn(e, __fadd2_rn(sl, pl));
  sh = __fadd2_rn(s, t);
  sl = __fadd2_rn(t, neg2(__fadd2_rn(sh, neg2(s))));
}

// (sh, sl) += a b, complex float-float: a = (ah, al), b = (bh, bl) as
// (re, im) lane pairs
__device__ __forceinline__ void ff_cfma(float2& sh, float2& sl, float2 ah, float2 al, float2 bh, float2 bl) {
  float2 xh, xl, yh, yl;
  // (a_re b_re, a_re b_im) + (-a_im b_im, a_im b_re)
  ff_mul2(make_float2(ah.x, ah.x), make_float2(al.x, al.x), bh, bl, xh, xl);
  ff_mul2(make_float2(ah.y, ah.y), make_float2(al.y, al.y), make_float2(-bh.y, bh.x), make_float2(-bl.y, bl.x), yh,
          yl);
  ff_acc2(sh, sl, xh, xl);
  ff_acc2(sh, sl, yh, yl);
}

// Complex float-float values as (re, im) lane pairs: h the leading parts, l
// the trailing ones.
struct cff {
  float2 h, l;
};
__device__ __forceinline__ cff cff_zero() { return cff{make_float2(0.f, 0.f), make_float2(0.f, 0.f)}; }
__device__ __forceinline__ cff cff_load(float4 v) { return cff{make_float2(v.x, v.y), make_float2(v.z, v.w)}; }
__device__ __forceinline__ cff cff_split(double re, double im) {
  const float rh = (float)re, ih = (float)im;
  return cff{make_float2(rh, ih), make_float2((float)(re - (double)rh), (float)(im - (double)ih))};
}
__device__ __forceinline__ double2 cff_to(cff a) {
  return make_double2((double)a.h.x + (double)a.l.x, (double)a.h.y + (double)a.l.y);
}
__device__ __forceinline__ cff cff_conj(cff a) {
  return cff{make_float2(a.h.x, -a.h.y), make_float2(a.l.x, -a.l.y)};
}
__device__ __forceinline__ cff cff_neg(cff a) { return cff{neg2(a.h), neg2(a.l)}; }
// acc + a b
__device__ __forceinline__ cff cff_fma(cff acc, cff a, cff b) {
  ff_cfma(acc.h, acc.l, a.h, a.l, b.h, b.l);
  return acc;
}
// a b
__device__ __forceinline__ cff cff_mul(cff a, cff b) {
  cff x, y;
  // (a_re b_re, a_re b_im) + (-a_im b_im, a_im b_re)
  ff_mul2(make_float2(a.h.x, a.h.x), make_float2(a.l.x, a.l.x), b.h, b.l, x.h, x.l);
  ff_mul2(make_float2(a.h.y, a.h.y), make_float2(a.l.y, a.l.y), make_float2(-b.h.y, b.h.x), make_float2(-b.l.y, b.l.x),
          y.h, y.l);
  ff_acc2(x.h, x.l, y.h, y.l);
  return x;
}
// a (sh + sl), a real float-float factor
__device__ __forceinline__ cff cff_scale(cff a, float sh, float sl) {
  cff r;
  ff_mul2(make_float2(sh, sh), make_float2(sl, sl), a.h, a.l, r.h, r.l);
  return r;
}

__device__ __forceinline__ float4 cff_store(cff a) { return make_float4(a.h.x, a.h.y, a.l.x, a.l.y); }

// P2M of the float-float residual's FMM and of the float-float solves'
// output FMM (FP64 expansions): the powers of u and the sums in float-float
// on the FP32 pipe (about 48 bits, what the
// float-float residual certifies; GB300 runs FP64 multiply-adds at two lanes
// a clock per SM).  Layout and term order as k_fmm_p2m: output e = d p + k
// on thread e mod kB, sources in order.
__global__ void __launch_bounds__(kB) k_fmm_p2m_ff(FmmDevT<double2> f, Geo g, const int* stop) {
  if (stop && *stop) return;
  extern __shared__ __align__(16) unsigned char smraw[];
  float4* pw = reinterpret_cast<float4*>(smraw);  // [p][kChunk + 1] u^k as (re_h, im_h, re_l, im_l)
  float4* qs = pw + f.p * (kChunk + 1);            // [kChunk][nd]
  const int b = blockIdx.x;
  const long long box = lev_off(f.L) + b;
  const int s0 = f.start[b], n = f.start[b + 1] - s0;
  if (n == 0) return;
  const int t = threadIdx.x, np = f.p * f.nd;
  cff acc[kP2MAcc];
#pragma unroll
  for (int u = 0; u < kP2MAcc; ++u) acc[u] = cff_zero();
  for (int ch = 0; ch < n; ch += kChunk) {
    const int m = min(kChunk, n - ch);
    if (t < m) {
      double s;
      const double2 c = box_center(f, f.L, b % f.nb, b / f.nb, s);
      const int i = f.perm[s0 + ch + t];
      const double is = ldexp(f.Dinv, f.L);
      const cff U = cff_split((g.x[i] - c.x) * is, (g.y[i] - c.y) * is);
      cff w = cff_split(1.0, 0.0);
      for (int k = 0; k < f.p; ++k) {
        pw[k * (kChunk + 1) + t] = cff_store(w);
        w = cff_mul(w, U);
      }
      for (int d = 0; d < f.nd; ++d) {
        // channel cm: q_0 conj(u), the leaf-relative moment density
        const double2 q = f.Q[(long long)i * f.nd + (d == f.cm ? 0 : d)];
        const cff qd = cff_split(q.x, q.y);
        qs[t * f.nd + d] = cff_store(d == f.cm ? cff_mul(qd, cff_conj(U)) : qd);
      }
    }
    __syncthreads();
#pragma unroll
    for (int u = 0; u < kP2MAcc; ++u) {
      const int e = t + u * kB;
      if (e < np) {
        const int d = e / f.p, k = e - d * f.p;
        const float4* pk = pw + k * (kChunk + 1);
        cff a = acc[u];
        for (int j = 0; j < m; ++j) a = cff_fma(a, cff_load(pk[j]), cff_load(qs[j * f.nd + d]));
        acc[u] = a;
      }
    }
    __syncthreads();
  }
#pragma unroll
  for (int u = 0; u < kP2MAcc; ++u)
    if (t + u * kB < np) f.mp[box * np + t + u * kB] = cff_to(acc[u]);
}

// Tables of order p: alpha[2][49][p], beta[2][49][p], gamma[49][p] (float4;
// type 0 Cauchy, 1 logarithm, as tab_alpha..tab_gamma), then the Pascal
// matrices [2][k][l] (float2 hi, lo).
__host__ __device__ inline long long fftab_beta(int p) { return 2LL * kOffs * p; }
__host__ __device__ inline long long fftab_gamma(int p) { return 4LL * kOffs * p; }
__host__ __device__ inline long long fftab_pascal(int p) { return 5LL * kOffs * p; }  // in float4 units
__host__ __device__ inline long long fftab_floats(int p) { return 20LL * kOffs * p + 4LL * p * p; }

// Quarter turn by -i of a complex float-float value (exact).
__device__ __forceinline__ cff cff_turn(cff a) {
  return cff{make_float2(a.h.y, -a.h.x), make_float2(a.l.y, -a.l.x)};
}
__device__ __forceinline__ cff cff_add(cff a, cff b) {
  ff_acc2(a.h, a.l, b.h, b.l);
  return a;
}

// Threads: split x (channel, row); orbits as in k_fmm_m2l.
template <int NJ>
__device__ __forceinline__ void m2l_ff_box(const FmmDev& f, long long gb, const float4* __restrict__ mpff,
                                           const float* __restrict__ tab, int nsplit, int nbo) {
  extern __shared__ __align__(16) unsigned char smraw[];
  __shared__ OrbitList o;
  __shared__ float4 s_a0[kOrbits][kMaxNd][4];  // the transforms of a_0 of the logarithm channels
  __shared__ float4 red[256];
  int l = 2;
  while (l < f.L && gb >= lev_off(l + 1)) ++l;
  if (f.tcount[gb] == 0) return;
  const int p = f.p, nd = f.nd, per = nd * p;
  const int b = (int)(gb - lev_off(l)), bx = b & ((1 << l) - 1), by = b >> l;
  const int tid = threadIdx.x;
  list_orbits(f, l, bx, by, o);
  float4* U = reinterpret_cast<float4*>(smraw);  // [nbo][nd p][4]
  const float4* alpha = reinterpret_cast<const float4*>(tab);
  const float4* beta = alpha + fftab_beta(p);
  const float4* gamma = alpha + fftab_gamma(p);
  const float2* pas = reinterpret_cast<const float2*>(alpha + fftab_pascal(p));
  const int sp = tid / per, e = tid - sp * per, d = e / p, t = e - d * p;
  const bool act = sp < nsplit;
  const int ty = d < f.nlog ? 1 : 0;
  const int base = t + 1 - ty;
  cff acc = cff_zero();
  for (int o0 = 0; o0 < o.cnt; o0 += nbo) {
    const int no = min(nbo, o.cnt - o0);
    __syncthreads();
    for (int q = tid; q < no * per; q += blockDim.x) {
      const int oo = q / per, dk = q - oo * per, dd = dk / p, k = dk - dd * p;
      const int tt = dd < f.nlog ? 1 : 0, id = o.id[o0 + oo];
      const int2 D = orbit_rep(id);
      int x = D.x, y = D.y;
      cff v[4];
#pragma unroll
      for (int r = 0; r < 4; ++r) {
        v[r] = cff_zero();
        if (o.src[id][r] >= 0) {
          const float4* a = mpff + (lev_off(l) + o.src[id][r]) * nd * p;
          v[r] = cff_load(a[dd * p + k]);
          // source moment density relative to the target centre: rho_S - conj(D_r) rho_0
          if (dd == f.cm)
            v[r] = cff_fma(v[r], cff{make_float2((float)-x, (float)y), make_float2(0.f, 0.f)}, cff_load(a[k]));
        }
        const int z = x;
        x = -y;
        y = z;
      }
      const cff t0 = cff_add(v[0], v[2]), t1 = cff_add(v[0], cff_neg(v[2]));
      const cff t2 = cff_add(v[1], v[3]), t3 = cff_turn(cff_add(v[1], cff_neg(v[3])));  // -i (a1 - a3)
      cff A[4];
      A[0] = cff_add(t0, t2);
      A[1] = cff_add(t1, t3);
      A[2] = cff_add(t0, cff_neg(t2));
      A[3] = cff_add(t1, cff_neg(t3));
      if (tt == 1 && k == 0)
#pragma unroll
        for (int r = 0; r < 4; ++r) s_a0[o0 + oo][dd][r] = cff_store(A[r]);
      const cff al = cff_load(alpha[((long long)tt * kOffs + offset_index(D.x, D.y)) * p + k]);
#pragma unroll
      for (int r = 0; r < 4; ++r) U[4 * q + r] = cff_store(cff_mul(al, A[r]));
    }
    __syncthreads();
    if (!act) continue;
    const float2* pcol = pas + (long long)ty * p * p + t;
    for (int q0 = sp; q0 < no; q0 += NJ * nsplit) {
      float2 sh[NJ], sl[NJ];
      const float4* u[NJ];
#pragma unroll
      for (int j = 0; j < NJ; ++j) {
        sh[j] = sl[j] = make_float2(0.f, 0.f);
        u[j] = U + (long long)(min(q0 + j * nsplit, no - 1) * per + d * p) * 4;
      }
      for (int k = 0; k < p; ++k) {
        const float2 pv = __ldg(pcol + (long long)k * p);
        const float2 PH = make_float2(pv.x, pv.x), PL = make_float2(pv.y, pv.y);
        const int at = 4 * k + ((base + k) & 3);
#pragma unroll
        for (int j = 0; j < NJ; ++j) {
          const float4 uv = u[j][at];
          float2 ph, pl;
          ff_mul2(PH, PL, make_float2(uv.x, uv.y), make_float2(uv.z, uv.w), ph, pl);
          ff_acc2(sh[j], sl[j], ph, pl);
        }
      }
#pragma unroll
      for (int j = 0; j < NJ; ++j) {
        const int q = q0 + j * nsplit;
        if (q < no) {
          const int id = o.id[o0 + q];
          const int2 D = orbit_rep(id);
          const int oi = offset_index(D.x, D.y);
          acc = cff_fma(acc, cff_load(beta[((long long)ty * kOffs + oi) * p + t]), cff{sh[j], sl[j]});
          if (ty == 1 && t > 0)
            acc = cff_fma(acc, cff_load(gamma[(long long)oi * p + t]), cff_load(s_a0[o0 + q][d][t & 3]));
          if (ty == 1 && t == 0) {
            // a_0 (log D_r + log s) per source, s = D 2^-l
            const cff logs = cff_split(log(f.D) - l * 0.69314718055994530942, 0.0);
            int x = D.x, y = D.y;
            for (int r = 0; r < 4; ++r) {
              if (o.src[id][r] >= 0)
                acc = cff_fma(acc, cff_add(cff_load(gamma[(long long)offset_index(x, y) * p]), logs),
                              cff_load(mpff[((lev_off(l) + o.src[id][r]) * nd + d) * p]));
              const int z = x;
              x = -y;
              y = z;
            }
          }
        }
      }
    }
  }
  red[tid] = cff_store(acc);
  __syncthreads();
  if (sp == 0) {
    for (int q = 1; q < nsplit; ++q) acc = cff_add(acc, cff_load(red[q * per + e]));
    // Cauchy channels carry 1/s
    const double sc = ty == 1 ? 1.0 : ldexp(f.Dinv, l);
    const double2 v = cff_to(acc);
    f.lc[gb * per + e] = make_double2(v.x * sc, v.y * sc);
  }
}

template <int NJ, bool MANY>
__global__ void __launch_bounds__(256) k_fmm_m2l_ff(FmmDev f, const float4* __restrict__ mpff,
                                                    const float* __restrict__ tab, int nsplit, int nbo,
                                                    const int* stop) {
  if (stop && *stop) return;
  for_boxes<MANY>(f.tcount + lev_off(2), lev_off(f.L + 1) - lev_off(2), f.tper,
                  [&](long long b) { m2l_ff_box<NJ>(f, b + lev_off(2), mpff, tab, nsplit, nbo); });
}

// L2L from level l0 down to the children of level lp (added to their M2L part), a
// block a box of level lp: it carries the expansion down its own path l0..lp in
// shared memory and writes the four children.  Boxes above lp are read, not
// updated, so one launch covers several levels (fmm_l2l).
template <class T2, int NC, int PK>
__global__ void __launch_bounds__(shift_max_threads(NC, PK), shift_blocks<T2>(NC, PK))
k_fmm_l2l(FmmDevT<T2> f, int l0, int lp, const int* stop) {
  using R = decltype(T2{}.x);
  if (stop && *stop) return;
  extern __shared__ __align__(16) unsigned char smraw[];
  const int p = f.p, np = f.nd * p, t = threadIdx.x;
  T2* loc = reinterpret_cast<T2*>(smraw);  // g_m b_m, [channel][m], channels PK + 1 apart
  T2* S = loc + f.nd * (PK + 1);           // [residue of m][channel, k]
  const int n = 1 << lp, b = blockIdx.x, bx = b & (n - 1), by = b >> lp;
  if (f.tcount[lev_off(lp) + b] == 0) return;
  const int e = t % np, mr = t / np, d = e / p, k = e - d * p;
  R T[PK / 4];
#pragma unroll
  for (int i = 0; i < PK / 4; ++i) {
    const int m = mr + 4 * i;
    T[i] = m >= k && m < p && mr < 4 ? __ldg(reinterpret_cast<const R*>(f.ops) + m * p + k) : (R)0;
  }
  for (int w = t; w < f.nd * (PK + 1 - p); w += blockDim.x)  // the padding
    loc[w / (PK + 1 - p) * (PK + 1) + p + w % (PK + 1 - p)] = cx<T2>(0.0, 0.0);
  const auto at = [&](int l) {  // the path's box of level l
    return lev_off(l) + ((long long)(by >> (lp - l)) << l) + (bx >> (lp - l));
  };
  // S_j, j = 0..3, of the thread's coefficient
  const auto sums = [&](T2* x) {
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      x[j] = S[((k + j) & 3) * np + e];
      if (d == f.cm) {
        // moment density relative to the child centre: 2 rho - 2 conj(w_r) a
        x[j].x *= R(2.0);
        x[j].y *= R(2.0);
        cfma(x[j], cx<T2>(-0.5, 0.5), S[((k + j + 1) & 3) * np + k]);
      }
    }
  };
  T2 next = cx<T2>(0.0, 0.0);
  if (t < np) next = f.lc[at(l0) * np + e];
  for (int l = l0;; ++l) {
    if (t < np) {
      loc[d * (PK + 1) + k] = eighth(next, k);
      if (l < lp) next = f.lc[at(l + 1) * np + e];
    }
    __syncthreads();
    if (mr < 4) {
      T2 acc = cx<T2>(0.0, 0.0);
      const T2* u = loc + d * (PK + 1) + mr;
#pragma unroll
      for (int i = 0; i < PK / 4; ++i) {
        const T2 x = u[4 * i];
        acc.x = fma(T[i], x.x, acc.x);
        acc.y = fma(T[i], x.y, acc.y);
      }
      S[t] = acc;
    }
    __syncthreads();
    if (l == lp) break;
    if (t < np) {
      const int r = turn_of_child(((bx >> (lp - l - 1)) & 1) + 2 * ((by >> (lp - l - 1)) & 1));
      T2 x[4];
      sums(x);
      const T2 a = cadd(cadd(x[0], turned(x[1], r)), cadd(turned(x[2], 2 * r), turned(x[3], 3 * r)));
      next = cadd(next, eighth_conj(a, k));
    }
  }
  if (t < np) {
    T2 x[4], v[4];
    long long box[4];
#pragma unroll
    for (int r = 0; r < 4; ++r) {
      const int c = child_of_turn(r);
      box[r] = lev_off(lp + 1) + (long long)(2 * by + (c >> 1)) * (2 * n) + 2 * bx + (c & 1);
      if (f.tcount[box[r]] == 0) box[r] = -1;
      v[r] = cx<T2>(0.0, 0.0);
      if (box[r] >= 0) v[r] = f.lc[box[r] * np + e];
    }
    sums(x);
    quarter_sums(x);
#pragma unroll
    for (int r = 0; r < 4; ++r)
      if (box[r] >= 0) f.lc[box[r] * np + e] = cadd(v[r], eighth_conj(x[r], k));
  }
}

// Local expansion and near field at every node of a leaf, then the kernel's
// combination into the pair-sum partial (Laplace scalar / Stokes 2-vector).
// The near field is the real kernel, summed directly over the 3 x 3 leaves: in
// FP64 (NEARP = 0, with rcp64), in FP32 (1, the inner solves) or in float-float
// (2, residuals), with exact leading coordinate differences in the latter two.
//
// Work: the m targets at hand take L = ceil(m / TPT) threads, and the kBE threads
// hold G = kBE / L such groups, each with every G-th source; the groups' sums are
// added in order.  A leaf of 39 nodes (the mean at 640,000) so keeps 91-94% of
// the lanes, against 61% with one target a thread of 64.  FP32: two targets a
// thread, so that a staged pair of sources (packed FP32x2) serves four pairs; the
// leaf's own sources come first, so that only they are compared with the target.
// The local expansions are evaluated a (target, channel) a thread; Laplace needs
// no derivative.
// Bound by the pair arithmetic: the FP64 pipe (10 Laplace, 16 Stokes operations a
// pair), FP32 issue and the FP32 pipe.  Measured, one target a thread of 64 (FP64:
// as Cauchy terms with a division and F' always) -> this: FP64 Laplace, 160,000
// nodes, order 36: 5.31 -> 1.26 ms; FP32 Stokes, 640,000 nodes, order 18: 277 ->
// 195 us; FP32 Laplace, 25,600 nodes: 39 -> 18 us; float-float Stokes, 640,000
// nodes, order 36: 1.74 -> 1.39 ms.
constexpr int kBE = 128;         // threads of an evaluation block
constexpr int kNearChunk = 256;  // near-field sources staged per round

template <int NEARP>
struct EvalNear;  // what a block stages and adds per precision
template <>
struct EvalNear<0> {
  static constexpr int kTPT = 1;
  using Sum = double2;
};
template <>
struct EvalNear<1> {
  static constexpr int kTPT = 2;
  using Sum = float2;
};
template <>
struct EvalNear<2> {
  static constexpr int kTPT = 1;
  using Sum = float4;  // (x_h, x_l, y_h, y_l)
};

// Values of F and s F' at one target (u relative to the leaf centre, units of s).
template <class T2>
__device__ __forceinline__ void horner(const T2* __restrict__ a, int p, T2 u, bool deriv, T2& h, T2& dh) {
  h = a[p - 1];
  dh = cx<T2>(0.0, 0.0);
  if (deriv) {
    for (int l = p - 2; l >= 0; --l) {
      T2 t = h;
      cfma(t, dh, u);
      dh = t;
      t = a[l];
      cfma(t, h, u);
      h = t;
    }
  } else {
    for (int l = p - 2; l >= 0; --l) {
      T2 t = a[l];
      cfma(t, h, u);
      h = t;
    }
  }
}

template <class T2, int NEARP>
__device__ __forceinline__ void eval_leaf(const FmmDevT<T2>& f, const Geo& g, int b, double* __restrict__ partial) {
  using Sum = typename EvalNear<NEARP>::Sum;
  constexpr int TPT = EvalNear<NEARP>::kTPT, NT = kBE * TPT;  // targets at hand
  // expansions [nd][p] (float-float: split hi + lo in 16 bytes), then F and F' of
  // the targets at hand [nd][NT][2]
  extern __shared__ __align__(16) unsigned char smraw[];
  using E = typename std::conditional<NEARP == 2, float4, T2>::type;
  E* sm = reinterpret_cast<E*>(smraw);
  E* FF = sm + f.nd * f.p;
  // FP64: (x, y) and (q1, q2) as double2; FP32: pairs of sources (hi, lo, strength);
  // float-float: (xh, xm, yh, ym), (xl, yl, -, -), strengths
  __shared__ float4 spa[kNearChunk], spb[NEARP == 1 ? 1 : kNearChunk], sq[NEARP == 0 ? 1 : kNearChunk];
  __shared__ Sum red[NT];
  __shared__ int lst[10], lbeg[9];
  __shared__ float cen[6];  // FP32 instance: split leaf centre, 1/s, s
  const int t = threadIdx.x;
  const int bx = b % f.nb, by = b / f.nb;
  const int s0 = f.start[b], n = f.start[b + 1] - s0;
  if (n == 0) return;
  const int nd = f.nd, p = f.p;
  const long long box = lev_off(f.L) + b;
  for (int e = t; e < nd * p; e += kBE) {
    if constexpr (NEARP == 2) {
      const double2 a = f.lc[box * nd * p + e];
      const float rh = (float)a.x, ih = (float)a.y;
      sm[e] = make_float4(rh, ih, (float)(a.x - (double)rh), (float)(a.y - (double)ih));
    } else {
      sm[e] = f.lc[box * nd * p + e];
    }
  }
  if constexpr (NEARP == 1) leaf_center32(f, b, cen);
  if (t == 0) {
    // the leaf itself first, then its neighbours row by row
    int c = 1, tot = n;
    lbeg[0] = s0;
    lst[0] = 0;
    for (int ny = max(0, by - 1); ny <= min(f.nb - 1, by + 1); ++ny)
      for (int nx = max(0, bx - 1); nx <= min(f.nb - 1, bx + 1); ++nx) {
        const int nl = ny * f.nb + nx;
        if (nl == b) continue;
        lbeg[c] = f.start[nl];
        lst[c] = tot;
        tot += f.start[nl + 1] - f.start[nl];
        ++c;
      }
    for (int k = c; k < 10; ++k) lst[k] = tot;
  }
  __syncthreads();
  const int total = lst[9];
  auto source = [&](int v) {  // node of entry v of the list
    int lf = 0;
    while (v >= lst[lf + 1]) ++lf;
    return f.perm[lbeg[lf] + (v - lst[lf])];
  };
  double s;
  const double2 c = box_center(f, f.L, bx, by, s);
  const double inv_s = ldexp(f.Dinv, f.L);
  for (int j0 = 0; j0 < n; j0 += NT) {
    const int m = min(NT, n - j0);
    // ---- local expansions: F and F' (scaled by 1/s) per (channel, target)
    for (int q = t; q < nd * m; q += kBE) {
      const int d = q / m, tt = q - d * m;
      const int i = f.perm[s0 + j0 + tt];
      E* o = FF + 2 * (d * NT + tt);
      if constexpr (NEARP == 2) {
        // float-float on the FP32 pipe
        const cff U = cff_split((g.x[i] - c.x) * inv_s, (g.y[i] - c.y) * inv_s);
        cff h = cff_load(sm[d * p + p - 1]), dh = cff_zero();
        for (int l = p - 2; l >= 0; --l) {
          if (nd > 1) dh = cff_fma(h, dh, U);  // h + dh u (the old h)
          h = cff_fma(cff_load(sm[d * p + l]), h, U);  // a_l + h u
        }
        const float ish = (float)inv_s, isl = (float)(inv_s - (double)ish);
        o[0] = cff_store(h);
        o[1] = cff_store(cff_scale(dh, ish, isl));
      } else {
        T2 u, h, dh;
        if constexpr (NEARP == 1) {
          // from the hi/lo split of z and the block's split centre (no FP64)
          const float4 P = g.pf[i];
          u = make_float2(((P.x - cen[0]) + (P.z - cen[2])) * cen[4], ((P.y - cen[1]) + (P.w - cen[3])) * cen[4]);
        } else {
          u = cx<T2>((g.x[i] - c.x) * inv_s, (g.y[i] - c.y) * inv_s);
        }
        horner(sm + d * p, p, u, nd > 1, h, dh);
        using R = decltype(u.x);
        const R is = NEARP == 1 ? (R)cen[4] : (R)inv_s;
        dh.x *= is;
        dh.y *= is;
        o[0] = h;
        o[1] = dh;
      }
    }
    // ---- near field
    const int L = (m + TPT - 1) / TPT, G = max(1, kBE / L);
    const int grp = t / L, tl = t - grp * L;
    const bool act = grp < G;
    int ti[TPT];  // targets (index at hand)
#pragma unroll
    for (int k = 0; k < TPT; ++k) ti[k] = min(tl + k * L, m - 1);
    if constexpr (NEARP == 0) {
      const int i = f.perm[s0 + j0 + ti[0]];
      const double tx = g.x[i], ty = g.y[i], tnx = g.nx[i], tny = g.ny[i];
      double ax = 0.0, ay = 0.0;
      double2* sx2 = reinterpret_cast<double2*>(spa);
      double2* sq2 = reinterpret_cast<double2*>(spb);
      for (int v0 = 0; v0 < total; v0 += kNearChunk) {
        const int mm = min(kNearChunk, total - v0);
        __syncthreads();
        for (int e = t; e < mm; e += kBE) {
          const int i2 = source(v0 + e);
          sx2[e] = make_double2(g.x[i2], g.y[i2]);
          sq2[e] = f.Q[(long long)i2 * nd];  // Laplace (q, 0); Stokes q1 + i q2
        }
        __syncthreads();
        if (act) {
          const int self = j0 + ti[0] - v0;
#pragma unroll 2
          for (int e = grp; e < mm; e += G) {
            const double2 P = sx2[e], q = sq2[e];
            const double dx = tx - P.x, dy = ty - P.y;
            const double y = rcp64(dx * dx + dy * dy);
            if (nd == 1) {
              const double w = e == self ? 0.0 : q.x * y;
              ax += dx * w;
              ay += dy * w;
            } else {
              const double w = e == self ? 0.0 : ((dx * q.x + dy * q.y) * (dx * tnx + dy * tny)) * (y * y);
              ax += w * dx;
              ay += w * dy;
            }
          }
        }
      }
      __syncthreads();  // red of the previous targets has been read
      if (act) red[grp * L + tl] = make_double2(ax, ay);
    } else if constexpr (NEARP == 1) {
      // two sources a packed FP32x2 operation, staged in pairs (positions hi and
      // lo, strengths); an odd count is padded with a zero-strength source far away
      float4* sp2 = spa;                   // [kNearChunk / 2] (xh0, xh1, yh0, yh1), negated
      float4* sl2 = spa + kNearChunk / 2;  // [kNearChunk / 2] (xl0, xl1, yl0, yl1), negated
      float4* sq2 = sq;                    // [kNearChunk / 2] (q1_0, q1_1, q2_0, q2_1)
      float4 T[TPT];
      float2 nn[TPT], AX[TPT], AY[TPT];
#pragma unroll
      for (int k = 0; k < TPT; ++k) {
        const int i = f.perm[s0 + j0 + ti[k]];
        T[k] = g.pf[i];
        nn[k] = g.nf[i];
        AX[k] = AY[k] = make_float2(0.f, 0.f);
      }
      // one staged pair of sources; CHECK: a source may be the target itself
      auto pairs = [&](int e2, int self0, int self1, bool check) {
        const float4 P = sp2[e2], PL = sl2[e2], Q = sq2[e2];
#pragma unroll
        for (int k = 0; k < TPT; ++k) {
          // exact leading differences
          const float2 dx = __fadd2_rn(__fadd2_rn(make_float2(T[k].x, T[k].x), make_float2(P.x, P.y)),
                                       __fadd2_rn(make_float2(T[k].z, T[k].z), make_float2(PL.x, PL.y)));
          const float2 dy = __fadd2_rn(__fadd2_rn(make_float2(T[k].y, T[k].y), make_float2(P.z, P.w)),
                                       __fadd2_rn(make_float2(T[k].w, T[k].w), make_float2(PL.z, PL.w)));
          const float2 r2 = __ffma2_rn(dx, dx, __fmul2_rn(dy, dy));
          float2 w = make_float2(rcp_approx(r2.x), rcp_approx(r2.y));
          if (check) {  // the self pair (r = 0)
            const int self = k == 0 ? self0 : self1;
            if (2 * e2 == self) w.x = 0.f;
            if (2 * e2 + 1 == self) w.y = 0.f;
          }
          if (nd == 1) {
            const float2 cc = __fmul2_rn(make_float2(Q.x, Q.y), w);
            AX[k] = __ffma2_rn(cc, dx, AX[k]);
            AY[k] = __ffma2_rn(cc, dy, AY[k]);
          } else {
            const float2 ex = __fmul2_rn(dx, w), ey = __fmul2_rn(dy, w);
            const float2 rq = __ffma2_rn(dx, make_float2(Q.x, Q.y), __fmul2_rn(dy, make_float2(Q.z, Q.w)));
            const float2 rn = __ffma2_rn(ex, make_float2(nn[k].x, nn[k].x), __fmul2_rn(ey, make_float2(nn[k].y, nn[k].y)));
            const float2 cc = __fmul2_rn(rq, rn);
            AX[k] = __ffma2_rn(cc, ex, AX[k]);
            AY[k] = __ffma2_rn(cc, ey, AY[k]);
          }
        }
      };
      for (int v0 = 0; v0 < total; v0 += kNearChunk) {
        const int mm = min(kNearChunk, total - v0), m2 = (mm + 1) >> 1;
        __syncthreads();
        for (int e2 = t; e2 < m2; e2 += kBE) {
          float4 P[2];
          float2 q[2];
          for (int h = 0; h < 2; ++h) {
            const int e = 2 * e2 + h;
            P[h] = make_float4(1e15f, 1e15f, 0.f, 0.f);
            q[h] = make_float2(0.f, 0.f);
            if (e < mm) {
              const int i2 = source(v0 + e);
              P[h] = g.pf[i2];
              q[h] = f.Qf[i2];
            }
          }
          sp2[e2] = make_float4(-P[0].x, -P[1].x, -P[0].y, -P[1].y);
          sl2[e2] = make_float4(-P[0].z, -P[1].z, -P[0].w, -P[1].w);
          sq2[e2] = make_float4(q[0].x, q[1].x, q[0].y, q[1].y);
        }
        __syncthreads();
        if (act) {
          const int own = min(m2, max(0, (n - v0 + 1) >> 1));  // pairs with sources of the leaf itself
          const int self0 = j0 + ti[0] - v0, self1 = j0 + ti[TPT - 1] - v0;
          int e2 = grp;
          for (; e2 < own; e2 += G) pairs(e2, self0, self1, true);
#pragma unroll 2
          for (; e2 < m2; e2 += G) pairs(e2, 0, 0, false);
        }
      }
      __syncthreads();
      if (act)
#pragma unroll
        for (int k = 0; k < TPT; ++k)
          red[k * kBE + grp * L + tl] = make_float2(AX[k].x + AX[k].y, AY[k].x + AY[k].y);
    } else {
      // float-float: one source at a time, float-float sums
      const int i = f.perm[s0 + j0 + ti[0]];
      FFTarget tg;
      {
        const float4 pp = g.xff[i];
        const float2 pl = g.xfl[i];
        tg.xh = pp.x;
        tg.xm = pp.y;
        tg.yh = pp.z;
        tg.ym = pp.w;
        tg.xl = pl.x;
        tg.yl = pl.y;
        tg.n = g.nff[i];
      }
      float axh = 0.f, axl = 0.f, ayh = 0.f, ayl = 0.f;
      for (int v0 = 0; v0 < total; v0 += kNearChunk) {
        const int mm = min(kNearChunk, total - v0);
        __syncthreads();
        for (int e = t; e < mm; e += kBE) {
          const int i2 = source(v0 + e);
          const double2 q = f.Q[(long long)i2 * nd];
          const float2 pl = g.xfl[i2];
          spa[e] = g.xff[i2];
          spb[e] = make_float4(pl.x, pl.y, 0.f, 0.f);
          const float q1h = (float)q.x, q2h = (float)q.y;
          sq[e] = make_float4(q1h, (float)(q.x - (double)q1h), q2h, (float)(q.y - (double)q2h));
        }
        __syncthreads();
        if (act) {
          const int self = j0 + ti[0] - v0;
          for (int e = grp; e < mm; e += G) {
            if (e == self) continue;
            const float4 pb = spb[e];
            float cxh, cxl, cyh, cyl;
            if (nd == 1)
              ff_pair<0>(tg, spa[e], make_float2(pb.x, pb.y), sq[e], cxh, cxl, cyh, cyl);
            else
              ff_pair<1>(tg, spa[e], make_float2(pb.x, pb.y), sq[e], cxh, cxl, cyh, cyl);
            ff_acc(axh, axl, cxh, cxl);
            ff_acc(ayh, ayl, cyh, cyl);
          }
        }
      }
      __syncthreads();
      if (act) red[grp * L + tl] = make_float4(axh, axl, ayh, ayl);
    }
    __syncthreads();
    // ---- the kernel's combination, about the leaf centre (its terms do not cancel)
    for (int tt = t; tt < m; tt += kBE) {
      const int i = f.perm[s0 + j0 + tt];
      const int k = tt / L, l = tt - k * L;  // its place among the near sums
      Sum a = red[k * kBE + l];
      for (int q = 1; q < G; ++q) {
        const Sum o = red[k * kBE + q * L + l];
        if constexpr (NEARP == 2) {
          ff_acc(a.x, a.y, o.x, o.y);
          ff_acc(a.z, a.w, o.z, o.w);
        } else {
          a.x += o.x;
          a.y += o.y;
        }
      }
      double ox = 0.0, oy = 0.0;
      if constexpr (NEARP == 2) {
        const double nx1 = g.nx[i], ny1 = g.ny[i];
        const double nearx = (double)a.x + (double)a.y, neary = (double)a.z + (double)a.w;
        if (nd == 1) {
          const double2 f0 = cff_to(cff_load(FF[2 * tt]));
          ox = nx1 * f0.x - ny1 * f0.y + nx1 * nearx + ny1 * neary;
        } else {
          const cff nu = cff_split(nx1, ny1), nub = cff_conj(nu);
          const float slh = (float)s, sll = (float)(s - (double)slh);
          // S3 = -F'_{q conj(z_j - c)} with c the leaf centre (channel cm holds that density / s)
          const cff S2 = cff_neg(cff_load(FF[2 * tt + 1]));
          const cff S3 = cff_neg(cff_scale(cff_load(FF[2 * (2 * NT + tt) + 1]), slh, sll));
          const cff S1 = cff_load(FF[2 * tt]), S6 = cff_load(FF[2 * (NT + tt)]);
          const cff zb = cff_split(g.x[i] - c.x, -(g.y[i] - c.y));
          const cff w = cff_fma(cff_neg(S3), zb, S2);  // conj(z - c) S2 - S3
          cff tm = cff_zero();
          tm = cff_fma(tm, nub, cff_conj(w));
          tm = cff_fma(tm, nu, cff_conj(S1));
          tm = cff_fma(tm, nub, cff_conj(S6));
          tm = cff_fma(tm, nu, S1);
          const double2 t2 = cff_to(tm);
          ox = 0.25 * t2.x + nearx;
          oy = 0.25 * t2.y + neary;
        }
      } else {
        using R = decltype(T2{}.x);
        T2 nu, zb;
        R sl;
        if constexpr (NEARP == 1) {
          const float4 P = g.pf[i];
          nu = g.nf[i];
          zb = make_float2((P.x - cen[0]) + (P.z - cen[2]), -((P.y - cen[1]) + (P.w - cen[3])));
          sl = cen[5];
        } else {
          nu = cx<T2>(g.nx[i], g.ny[i]);
          zb = cx<T2>(g.x[i] - c.x, -(g.y[i] - c.y));
          sl = (R)s;
        }
        if (nd == 1) {
          const T2 F0 = FF[2 * tt];
          ox = (double)(nu.x * F0.x - nu.y * F0.y + (nu.x * a.x + nu.y * a.y));
        } else {
          const T2 nub = cconj(nu);
          const T2 S1 = FF[2 * tt], S6 = FF[2 * (NT + tt)];
          T2 S2 = FF[2 * tt + 1], S3 = FF[2 * (2 * NT + tt) + 1];
          S2.x = -S2.x;
          S2.y = -S2.y;
          S3.x = -sl * S3.x;
          S3.y = -sl * S3.y;
          T2 w = cmul(zb, S2);
          w.x -= S3.x;
          w.y -= S3.y;
          T2 tm = cmul(nub, cconj(w));
          tm = cadd(tm, cmul(nu, cconj(S1)));
          tm = cadd(tm, cmul(nub, cconj(S6)));
          tm = cadd(tm, cmul(nu, S1));
          ox = (double)((R)0.25 * tm.x + a.x);
          oy = (double)((R)0.25 * tm.y + a.y);
        }
      }
      if (nd == 1) {
        partial[i] = ox;
      } else {
        partial[2 * i] = ox;
        partial[2 * i + 1] = oy;
      }
    }
    __syncthreads();  // FF and red are written for the next targets
  }
}

template <class T2, int NEARP, bool MANY>
__global__ void __launch_bounds__(kBE) k_fmm_eval(FmmDevT<T2> f, Geo g, double* __restrict__ partial, const int* stop) {
  if (stop && *stop) return;
  for_boxes<MANY>(f.count + lev_off(f.L), (long long)f.nb * f.nb, f.per,
                  [&](long long b) { eval_leaf<T2, NEARP>(f, g, (int)b, partial); });
}

// Dynamic shared memory of an evaluation block.
template <class T2, int NEARP>
size_t eval_smem(int nd, int p) {
  const size_t e = NEARP == 2 ? sizeof(float4) : sizeof(T2);
  return e * ((size_t)nd * p + 2 * (size_t)nd * kBE * EvalNear<NEARP>::kTPT);
}

// Output densities at the boundary nodes (v = sqrt(w)-scaled total density):
// Laplace channel 0 = q = w nu (logarithm); Stokes f = w (nu1 + i nu2):
// channels f1, f2 (logarithm), f and f conj(z - c0) (Cauchy).
__global__ void k_fmm_out_density(Geo g, int nd, double cx0, double cy0, const double* __restrict__ v, double2* Q) {
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < g.M; i += gridDim.x * blockDim.x) {
    if (nd == 1) {
      Q[i] = make_double2(g.sw[i] * v[i], 0.0);
    } else {
      const double2 fq = make_double2(g.sw[i] * v[2 * i], g.sw[i] * v[2 * i + 1]);
      Q[4 * i] = make_double2(fq.x, 0.0);
      Q[4 * i + 1] = make_double2(fq.y, 0.0);
      Q[4 * i + 2] = fq;
      Q[4 * i + 3] = cmul(fq, make_double2(g.x[i] - cx0, -(g.y[i] - cy0)));
    }
  }
}

// Output targets: z0 per body (Laplace) or z0, z0 + delta e1, z0 + delta e2
// (Stokes); their leaves and the target counts of the leaves.
__global__ void k_fmm_targets(Geo g, int per, int L, double x0, double y0, double D, double* tx, double* ty,
                              int* tleaf, int* tcount_leaf) {
  const int T = g.N * per, nb = 1 << L;
  for (int t = blockIdx.x * blockDim.x + threadIdx.x; t < T; t += gridDim.x * blockDim.x) {
    const int i = t / per, k = t % per;
    const double d = g.delta[i];
    const double x = g.zx[i] + (k == 1 ? d : 0.0), y = g.zy[i] + (k == 2 ? d : 0.0);
    tx[t] = x;
    ty[t] = y;
    int ix = (int)((x - x0) / D * nb), iy = (int)((y - y0) / D * nb);
    ix = min(max(ix, 0), nb - 1);
    iy = min(max(iy, 0), nb - 1);
    tleaf[t] = iy * nb + ix;
    atomicAdd(&tcount_leaf[iy * nb + ix], 1);
  }
}

// Single layers at the output targets: local expansion plus the 3 x 3 near
// leaves, in the layout of the direct output sums (Laplace: sum w nu log r^2;
// Stokes: sum [-log|r| f + r (r . f)/|r|^2] as a 2-vector).
constexpr int kTW = 8;  // targets (one warp each) per block of k_fmm_eval_targets

// One warp per target: the lanes split the near-field sources of the 3 x 3
// leaves (one reciprocal and one table-driven logarithm a pair) and their sums
// are reduced across the warp in a fixed order.  The local expansions of the
// target's leaf are split too, 32/nd lanes a channel: Horner over each lane's
// coefficients, then pairs of lanes combined with u^m, u^2m, ... (by one lane they took
// longer than the near field: an FP64 instruction of one lane costs the pipe as much
// as one of 32).  30,000 Stokes targets, order 36, 350 near sources each: 2.83 -> 1.27 ms.
__global__ void __launch_bounds__(32 * kTW) k_fmm_eval_targets(FmmDev f, Geo g, int kind, int T,
                                                            const double* __restrict__ tx,
                                                            const double* __restrict__ ty,
                                                            const int* __restrict__ tleaf, double c0x, double c0y,
                                                            double* __restrict__ part) {
  __shared__ double2 ltab[kLogTab];
  log_table_fill(ltab);
  __syncthreads();
  const int lane = threadIdx.x & 31;
  const int t = blockIdx.x * kTW + (threadIdx.x >> 5);
  if (t >= T) return;
  const int b = tleaf[t], bx = b % f.nb, by = b / f.nb;
  const long long box = lev_off(f.L) + b;
  const double x = tx[t], y = ty[t];
  double2 val[kMaxNd];
  for (int d = 0; d < kMaxNd; ++d) val[d] = make_double2(0.0, 0.0);
  for (int ny = max(0, by - 1); ny <= min(f.nb - 1, by + 1); ++ny)
    for (int nx = max(0, bx - 1); nx <= min(f.nb - 1, bx + 1); ++nx) {
      const int nl = ny * f.nb + nx;
      for (int k = f.start[nl] + lane; k < f.start[nl + 1]; k += 32) {
        const int j = f.perm[k];
        const double rx = x - g.x[j], ry = y - g.y[j];
        const double r2 = rx * rx + ry * ry;
        const double lg = 0.5 * log_tab(r2, ltab);
        for (int d = 0; d < f.nlog; ++d) val[d].x += f.Q[(long long)j * f.nd + d].x * lg;
        const double ir2 = rcp64(r2);
        const double2 inv = make_double2(rx * ir2, -ry * ir2);
        for (int d = f.nlog; d < f.nd; ++d) cfma(val[d], f.Q[(long long)j * f.nd + d], inv);
      }
    }
  for (int d = 0; d < f.nd; ++d) {
    val[d].x = warp_sum(val[d].x);
    val[d].y = warp_sum(val[d].y);
  }
  {
    double s;
    const double2 c = box_center(f, f.L, bx, by, s);
    const double is = ldexp(f.Dinv, f.L);
    const double2 u = make_double2((x - c.x) * is, (y - c.y) * is);
    const int np = f.nd == 1 ? 32 : 8, d = lane / np, q = lane % np;  // nd = 1 or 4
    const int m = (f.p + np - 1) / np;
    const double2* lc = f.lc + (box * f.nd + d) * f.p;
    double2 h = make_double2(0.0, 0.0), um = u;
    for (int l = m - 1; l >= 0; --l) {
      h = cmul(h, u);
      if (q * m + l < f.p) h = cadd(h, lc[q * m + l]);
      if (l > 0 && l < m - 1) um = cmul(um, u);
    }
    if (m > 1) um = cmul(um, u);  // u^m
    for (int w = 1; w < np; w *= 2) {
      const double2 o = make_double2(__shfl_down_sync(0xffffffffu, h.x, w), __shfl_down_sync(0xffffffffu, h.y, w));
      cfma(h, um, o);  // (lanes beyond the channel's first are not used)
      um = cmul(um, um);
    }
    for (int e = 0; e < f.nd; ++e)
      val[e] = cadd(make_double2(__shfl_sync(0xffffffffu, h.x, e * np), __shfl_sync(0xffffffffu, h.y, e * np)), val[e]);
  }
  double2 ftot = make_double2(0.0, 0.0);  // Stokes: sum of f over all nodes: the level-2 moments a_0
  if (kind != 0) {
    if (lane < 16 && f.count[lev_off(2) + lane] > 0) ftot = f.mp[((lev_off(2) + lane) * f.nd + 2) * f.p];
    ftot.x = warp_sum(ftot.x);
    ftot.y = warp_sum(ftot.y);
  }
  if (lane != 0) return;
  if (kind == 0) {
    part[t] = 2.0 * val[0].x;
  } else {
    double2 w = cmul(make_double2(x - c0x, -(y - c0y)), val[2]);
    w = make_double2(w.x - val[3].x, -(w.y - val[3].y));  // conj(conj(t - c0) F_f - F_{f conj(z - c0)})
    part[2 * t] = -val[0].x + 0.5 * ftot.x + 0.5 * w.x;
    part[2 * t + 1] = -val[1].x + 0.5 * ftot.y + 0.5 * w.y;
  }
}

inline int grid_for(long long n) {
  long long b = (n + 255) / 256;
  return (int)(b < 1 ? 1 : (b > 4096 ? 4096 : b));
}

// Translation operators for order p in the layout of tab_alpha..tab_size.
std::vector<std::complex<double>> build_ops(int p) {
  using C = std::complex<double>;
  std::vector<double> bin((2 * p + 1) * (2 * p + 1), 0.0);
  auto B = [&](int a, int b) -> double& { return bin[a * (2 * p + 1) + b]; };
  for (int a = 0; a <= 2 * p; ++a) {
    B(a, 0) = 1.0;
    for (int b = 1; b <= a; ++b) B(a, b) = B(a - 1, b - 1) + (b <= a - 1 ? B(a - 1, b) : 0.0);
  }
  std::vector<C> ops((size_t)tab_size(p), C(0, 0));
  for (int m = 0; m < p; ++m)
    for (int k = 0; k < p; ++k) {
      const int hi = std::max(m, k), lo = std::min(m, k);
      // |w| = 2^-3/2; with the factors h the exponent is a whole number: T is exact
      const double t = B(hi, lo) * std::ldexp(1.0, -lo - (3 * (hi - lo) + (hi & 1) + (lo & 1)) / 2);
      const int e = m * p + k;
      ops[e / 2] = e & 1 ? C(ops[e / 2].real(), t) : C(t, 0.0);
    }
  // M2L factors.  Cauchy: (d + u)^-(k+1) = sum_l C(k+l, l) (-1)^l u^l d^-(k+l+1).
  // Logarithm: log(d + u) = log d + sum_l (-1)^(l+1) (u/d)^l / l and
  // (d + u)^-k = sum_l C(k+l-1, l) (-1)^l u^l d^-(k+l); the log s part of log d
  // is added by the kernel.
  const size_t A = tab_alpha(p), Bt = tab_beta(p), G = tab_gamma(p), P = tab_pascal(p);
  for (int dy = -3; dy <= 3; ++dy)
    for (int dx = -3; dx <= 3; ++dx) {
      if (std::abs(dx) <= 1 && std::abs(dy) <= 1) continue;
      const size_t o = (size_t)(dx + 3) + 7 * (dy + 3);
      const C Dinv = 1.0 / C(dx, dy);
      for (int k = 0; k < p; ++k) {
        ops[A + o * p + k] = std::pow(Dinv, k);
        ops[A + (kOffs + o) * p + k] = k == 0 ? C(0, 0) : std::pow(Dinv, k) / (double)k;
      }
      for (int l = 0; l < p; ++l) {
        const double sg = (l & 1) ? -1.0 : 1.0;
        ops[Bt + o * p + l] = sg * std::pow(Dinv, l + 1);
        ops[Bt + (kOffs + o) * p + l] = -sg * std::pow(Dinv, l);
        ops[G + o * p + l] = l == 0 ? std::log(C(dx, dy)) : -sg * std::pow(Dinv, l) / (double)l;
      }
    }
  for (int k = 0; k < p; ++k)
    for (int l = 0; l < p; ++l) {
      ops[P + (size_t)k * p + l] = B(k + l, l);
      ops[P + ((size_t)p + k) * p + l] = k == 0 ? 0.0 : B(k + l - 1, l);
    }
  return ops;
}

}  // namespace

struct FmmState {
  int L = 0, nb = 0, nleaf = 0, kind = 0, M = 0, N = 0;
  double x0 = 0, y0 = 0, D = 0;
  long long nbox = 0;
  int per = 1, tper = 1;  // boxes that a block goes over: of the leaves (and of the level above), of all levels
  // device buffers (stream-ordered), grown on demand
  char* buf = nullptr;
  size_t buf_size = 0;
  int *leaf = nullptr, *perm = nullptr, *tmp = nullptr, *start = nullptr, *cursor = nullptr, *count = nullptr;
  int *tcount = nullptr, *tleaf = nullptr;
  int* arrive = nullptr;  // per box: siblings done in the upward pass (0 between launches)
  double *tx = nullptr, *ty = nullptr;
  double2 *Q = nullptr, *mp = nullptr, *lc = nullptr;
  float4* cen32 = nullptr;  // per leaf: centre split as float hi + lo (x_h, y_h, x_l, y_l)
  double* scal = nullptr;
  int pmax = 0;
  // operators per order (FP64, and their FP32 copies)
  std::vector<std::pair<int, double2*>> ops;
  std::vector<std::pair<int, float2*>> ops32;
  // float-float M2L: split multipoles and the split factor tables per order
  float4* mpff = nullptr;
  std::vector<std::pair<int, float*>> opsff;
};

void fmm_free(FmmState* f, cudaStream_t s) {
  if (!f) return;
  if (f->buf) cudaFreeAsync(f->buf, s);
  for (auto& o : f->ops) cudaFreeAsync(o.second, s);
  for (auto& o : f->ops32) cudaFreeAsync(o.second, s);
  for (auto& o : f->opsff) cudaFreeAsync(o.second, s);
  delete f;
}

// Build the tree for the staged geometry (one host round trip for the box).
int fmm_setup(FmmState*& f, const Geo& g, int kind, const int* orders, int norders, cudaStream_t s,
              std::string& err, int leaf_nodes) {
  if (leaf_nodes <= 0) leaf_nodes = kDefaultLeafNodes;
  int pmax = 0;
  for (int k = 0; k < norders; ++k) {
    if (orders[k] < 2 || orders[k] > kMaxP) {
      err = "FMM order must be in 2.." + std::to_string(kMaxP);
      return BIE_ERR_INVALID;
    }
    pmax = std::max(pmax, orders[k]);
  }
  if (!f) f = new FmmState();
  auto ck = [&](cudaError_t e, const char* what) {
    if (e != cudaSuccess) err = std::string(what) + ": " + cudaGetErrorString(e);
    return e == cudaSuccess;
  };
  // bounding square and total length
  double* scal = nullptr;
  if (!f->scal) {
    if (!ck(cudaMallocAsync(reinterpret_cast<void**>(&f->scal), 4 * sizeof(double), s), "fmm scal")) return BIE_ERR_CUDA;
  }
  scal = f->scal;
  k_fmm_box<<<1, kBoxT, 0, s>>>(g, scal);
  note_launches(1);
  double h[4];
  if (!ck(cudaMemcpyAsync(h, scal, sizeof(h), cudaMemcpyDeviceToHost, s), "fmm box") ||
      !ck(cudaStreamSynchronize(s), "fmm box sync"))
    return BIE_ERR_CUDA;
  f->x0 = h[0];
  f->y0 = h[1];
  f->D = h[2];
  // leaf level: the finest level whose non-empty leaves hold at least
  // leaf_nodes nodes (default 24); nodes on curves of total length P occupy
  // about min(4^L, 1.3 P 2^L / D) leaves
  int L = 2;
  const auto used = [&](int l) { return fmin((double)(1LL << (2 * l)), 1.3 * h[3] * (double)(1 << l) / f->D); };
  for (int l = 2; l <= 10; ++l)
    if ((double)g.M / fmax(used(l), 1.0) >= (double)leaf_nodes) L = l;
  f->per = boxes_a_block(used(L), (double)(1LL << (2 * L)));
  f->tper = boxes_a_block_levels(L, used);
  f->L = L;
  f->nb = 1 << L;
  f->nleaf = f->nb * f->nb;
  f->nbox = lev_off(L + 1);
  f->kind = kind;
  f->M = g.M;
  f->N = g.N;
  const int nd = kMaxNd;  // room for the output channels
  f->pmax = pmax;
  // buffers
  auto pad = [](size_t b) { return (b + 255) & ~size_t(255); };
  const size_t need = 3 * pad((size_t)g.M * 4) + 2 * pad(((size_t)f->nleaf + 1) * 4) + 3 * pad((size_t)f->nbox * 4) +
                      pad((size_t)g.M * nd * 16) + 3 * pad((size_t)f->nbox * nd * pmax * 16) +
                      pad((size_t)3 * g.N * 4) + 2 * pad((size_t)3 * g.N * 8) + pad((size_t)f->nleaf * 16);
  if (need > f->buf_size) {
    if (f->buf) cudaFreeAsync(f->buf, s);
    f->buf = nullptr;
    f->buf_size = 0;
    if (!ck(cudaMallocAsync(reinterpret_cast<void**>(&f->buf), need, s), "fmm buffers")) return BIE_ERR_CUDA;
    f->buf_size = need;
  }
  size_t off = 0;
  auto take = [&](size_t bytes) {
    char* p = f->buf + off;
    off += pad(bytes);
    return p;
  };
  f->leaf = (int*)take((size_t)g.M * 4);
  f->perm = (int*)take((size_t)g.M * 4);
  f->tmp = (int*)take((size_t)g.M * 4);
  f->start = (int*)take(((size_t)f->nleaf + 1) * 4);
  f->cursor = (int*)take(((size_t)f->nleaf + 1) * 4);
  f->count = (int*)take((size_t)f->nbox * 4);
  f->tcount = (int*)take((size_t)f->nbox * 4);
  f->arrive = (int*)take((size_t)f->nbox * 4);
  f->tleaf = (int*)take((size_t)3 * g.N * 4);
  f->tx = (double*)take((size_t)3 * g.N * 8);
  f->ty = (double*)take((size_t)3 * g.N * 8);
  f->Q = (double2*)take((size_t)g.M * nd * 16);
  f->mp = (double2*)take((size_t)f->nbox * nd * pmax * 16);
  f->lc = (double2*)take((size_t)f->nbox * nd * pmax * 16);
  f->mpff = (float4*)take((size_t)f->nbox * nd * pmax * 16);
  f->cen32 = (float4*)take((size_t)f->nleaf * 16);
  // counting sort of the nodes by leaf, node order inside a leaf
  if (!ck(cudaMemsetAsync(f->cursor, 0, ((size_t)f->nleaf + 1) * 4, s), "fmm memset") ||
      !ck(cudaMemsetAsync(f->arrive, 0, (size_t)f->nbox * 4, s), "fmm memset"))
    return BIE_ERR_CUDA;
  k_fmm_leaf<<<grid_for(g.M), 256, 0, s>>>(g, L, f->x0, f->y0, f->D, f->leaf, f->cursor);
  k_fmm_scan<<<1, 1024, 0, s>>>(f->cursor, f->nleaf, f->start);
  cudaMemsetAsync(f->cursor, 0, ((size_t)f->nleaf + 1) * 4, s);
  k_fmm_scatter<<<grid_for(g.M), 256, 0, s>>>(g.M, f->leaf, f->start, f->cursor, f->tmp);
  k_fmm_order<<<f->nleaf, 128, 0, s>>>(f->start, f->tmp, f->perm);
  k_fmm_leaf_counts<<<grid_for(f->nleaf), 256, 0, s>>>(f->start, f->nleaf, f->count + lev_off(L));
  for (int l = L - 1; l >= 0; --l) k_fmm_parent_counts<<<grid_for(1LL << (2 * l)), 256, 0, s>>>(l, f->count);
  k_fmm_leaf_centers<<<grid_for(f->nleaf), 256, 0, s>>>(f->nb, f->x0, f->y0, ldexp(f->D, -L), f->cen32);
  note_launches(7 + L);
  if (!ck(cudaGetLastError(), "fmm setup")) return BIE_ERR_CUDA;
  // translation operators, built before any capture of the apply
  for (int k = 0; k < norders; ++k) {
    const int p = orders[k];
    bool have = false;
    for (auto& o : f->ops) have |= o.first == p;
    if (have) continue;
    const auto host = build_ops(p);
    std::vector<float2> host32(host.size());
    for (size_t e = 0; e < host.size(); ++e)
      host32[e] = make_float2((float)host[e].real(), (float)host[e].imag());
    // k_fmm_m2l32's Pascal table after it: [k][residue][pair] rows (l, l + 4), zeros outside the order
    const int pk = m2l32_pad(p), rp = m2l32_rp(pk);
    host32.resize(host.size() + (size_t)pk * 4 * rp, make_float2(0.f, 0.f));
    for (int k = 0; k < p; ++k)
      for (int m = 0; m < 4 * rp; ++m) {
        const int t0 = m / rp + 8 * (m % rp);
        const auto entry = [&](int l) { return l < p ? (float)host[(size_t)tab_pascal(p) + (size_t)k * p + l].real() : 0.f; };
        host32[host.size() + (size_t)k * 4 * rp + m] = make_float2(entry(t0), entry(t0 + 4));
      }
    double2* ops = nullptr;
    float2* ops32 = nullptr;
    if (!ck(cudaMallocAsync(reinterpret_cast<void**>(&ops), host.size() * sizeof(double2), s), "fmm ops") ||
        !ck(cudaMallocAsync(reinterpret_cast<void**>(&ops32), host32.size() * sizeof(float2), s), "fmm ops") ||
        !ck(cudaMemcpyAsync(ops, host.data(), host.size() * sizeof(double2), cudaMemcpyHostToDevice, s), "fmm ops") ||
        !ck(cudaMemcpyAsync(ops32, host32.data(), host32.size() * sizeof(float2), cudaMemcpyHostToDevice, s),
            "fmm ops") ||
        !ck(cudaStreamSynchronize(s), "fmm ops"))
      return BIE_ERR_CUDA;
    f->ops.push_back({p, ops});
    f->ops32.push_back({p, ops32});
    // float-float splits of the M2L factors and of the Pascal matrices
    std::vector<float> hff((size_t)fftab_floats(p));
    auto split = [](double x, float& h, float& l) {
      h = (float)x;
      l = (float)(x - (double)h);
    };
    const size_t tabs[3] = {(size_t)tab_alpha(p), (size_t)tab_beta(p), (size_t)tab_gamma(p)};
    for (int t = 0; t < 5; ++t)  // alpha (2 types), beta (2 types), gamma
      for (int e = 0; e < kOffs * p; ++e) {
        const auto v = host[tabs[t / 2] + (size_t)(t % 2) * kOffs * p + e];
        float* q = hff.data() + ((size_t)t * kOffs * p + e) * 4;
        split(v.real(), q[0], q[2]);
        split(v.imag(), q[1], q[3]);
      }
    for (int e = 0; e < 2 * p * p; ++e) {
      float* q = hff.data() + (size_t)20 * kOffs * p + 2 * (size_t)e;
      split(host[(size_t)tab_pascal(p) + e].real(), q[0], q[1]);
    }
    float* opsff = nullptr;
    if (!ck(cudaMallocAsync(reinterpret_cast<void**>(&opsff), hff.size() * sizeof(float), s), "fmm ops") ||
        !ck(cudaMemcpyAsync(opsff, hff.data(), hff.size() * sizeof(float), cudaMemcpyHostToDevice, s), "fmm ops") ||
        !ck(cudaStreamSynchronize(s), "fmm ops"))
      return BIE_ERR_CUDA;
    f->opsff.push_back({p, opsff});
  }
  return BIE_OK;
}

namespace {

// The splits of the orbits that fill a block's warps best (nsplit (channel, row)
// threads), and the orbits staged at a time (at most about 100 KB).
// The kernels' bound is a constant, five orbits of four channels and both Pascal
// matrices at the largest order: with each launch's own size, another thread's
// launch could find a smaller bound than it needs.
constexpr int kMaxM2lSmem = 5 * kMaxNd * kMaxP * 4 * 16 + 2 * kMaxP * kMaxP * 8;
struct M2lShape {
  int nsplit, threads, nbo;
  size_t smem;
};
M2lShape m2l_shape(int nd, int p, size_t entry, size_t pascal) {
  M2lShape m{1, 0, kOrbits, 0};
  const int per = nd * p;
  double best = 0.0;
  for (int s : {1, 2, 5}) {
    const int th = (s * per + 31) / 32 * 32;
    if (th > 256) continue;
    const double use = (double)s * per / th;
    // more splits where they fill the warps as well: shorter chains (float-float, one
    // channel of order 30, 1,024 leaves: one split 43 us, five 32)
    if (use > best - 0.02) {
      best = std::max(best, use);
      m.nsplit = s;
      m.threads = th;
    }
  }
  while (m.nbo > 5 && (size_t)m.nbo * per * 4 * entry + pascal > 100 * 1024) m.nbo = 5;
  m.smem = (size_t)m.nbo * per * 4 * entry + pascal;
  return m;
}

template <int ND, int PK>
void m2l32_launch(const FmmDevT<float2>& d, const float2* ptab, int L, const int* stop, cudaStream_t s) {
  const size_t sm = (size_t)kOrbits * ND * (4 * PK + 4) * sizeof(float2);
  const unsigned grid = blocks_for(lev_off(L + 1) - lev_off(2), d.tper);
  const auto fn = d.tper > 1 ? k_fmm_m2l32<ND, PK, true> : k_fmm_m2l32<ND, PK, false>;
  if (sm > 40 * 1024) cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
  fn<<<grid, m2l32_threads(ND, PK), sm, s>>>(d, ptab, stop);
}

template <int ND>
void launch_m2l32(const FmmDevT<float2>& d, const float2* ptab, int pk, int L, const int* stop, cudaStream_t s) {
  switch (pk) {
    case 12: return m2l32_launch<ND, 12>(d, ptab, L, stop, s);
    case 16: return m2l32_launch<ND, 16>(d, ptab, L, stop, s);
    case 20: return m2l32_launch<ND, 20>(d, ptab, L, stop, s);
    case 24: return m2l32_launch<ND, 24>(d, ptab, L, stop, s);
    case 32: return m2l32_launch<ND, 32>(d, ptab, L, stop, s);
    case 48: return m2l32_launch<ND, 48>(d, ptab, L, stop, s);
    default: return m2l32_launch<ND, 64>(d, ptab, L, stop, s);
  }
}

void launch_m2l(const FmmDev& d, int L, const int* stop, cudaStream_t s) {
  const unsigned grid = blocks_for(lev_off(L + 1) - lev_off(2), d.tper);
  const M2lShape m = m2l_shape(d.nd, d.p, sizeof(double2), (size_t)(d.nlog > 0 ? 2 : 1) * d.p * d.p * sizeof(double));
  const auto fn = m.nsplit == 5 ? (d.tper > 1 ? k_fmm_m2l<double2, 2, true> : k_fmm_m2l<double2, 2, false>)
                                : (d.tper > 1 ? k_fmm_m2l<double2, 5, true> : k_fmm_m2l<double2, 5, false>);
  cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, kMaxM2lSmem);
  fn<<<grid, m.threads, m.smem, s>>>(d, m.nsplit, m.nbo, stop);
}

void launch_m2l_ff(const FmmDev& d, const float4* mpff, const float* tab, int L, const int* stop, cudaStream_t s) {
  const M2lShape m = m2l_shape(d.nd, d.p, sizeof(float4), 0);
  const unsigned grid = blocks_for(lev_off(L + 1) - lev_off(2), d.tper);
  const auto fn = m.nsplit == 5 ? (d.tper > 1 ? k_fmm_m2l_ff<2, true> : k_fmm_m2l_ff<2, false>)
                                : (d.tper > 1 ? k_fmm_m2l_ff<5, true> : k_fmm_m2l_ff<5, false>);
  cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, kMaxM2lSmem);
  fn<<<grid, m.threads, m.smem, s>>>(d, mpff, tab, m.nsplit, m.nbo, stop);
}

// The instance of the shift kernels for nd channels of order p, whose coefficients are
// padded with zeros to its width: the default inner orders (15 and 18) and residual order (36)
// have one of their own, larger ones the widest.  A whole application at order 37 takes 3%
// (FP64) and 8% (float-float) longer than at 36 (25,600 Stokes nodes: 1,006 and 1,041 us, 482
// and 518), so that a further instance of the four kernels would be little used for little;
// orders 37 to 64 at 160,000 nodes run 1.3 to 3.3 times as fast as with run-time sizes (FP64
// Stokes 14.6 -> 4.5 ms at 37, 20.4 -> 6.8 at 64; FP32 881 -> 683 us and 1,323 -> 775).
template <int NC, class F>
void for_shift_order(int p, F&& launch) {
  using std::integral_constant;
  const integral_constant<int, NC> nc{};
  if (p <= 16) return launch(nc, integral_constant<int, 16>{});
  if (p <= 20) return launch(nc, integral_constant<int, 20>{});
  if (p <= 36) return launch(nc, integral_constant<int, 36>{});
  launch(nc, integral_constant<int, 64>{});
}
template <class F>
void for_shift(int nd, int p, F&& launch) {
  if (nd == 1)
    for_shift_order<1>(p, launch);
  else
    for_shift_order<kMaxNd>(p, launch);
}

// The downward pass.  A launch that covers several levels repeats the upper ones in
// every block, which costs less than a launch while its lowest level has few boxes:
// FP32 up to 1,024 (with 4,096, 43 us in place of 32 at 16,384 leaves), FP64, whose
// pipe is 1/64 as wide, 256.
template <class T2>
int fmm_l2l(const FmmDevT<T2>& d, const int* stop, cudaStream_t s) {
  constexpr int kPath = std::is_same<T2, float2>::value ? 5 : 4;  // level: 4^kPath boxes
  int n = 0;
  for (int l0 = 2; l0 < d.L; ++n) {
    const int lp = std::max(l0, std::min(kPath, d.L - 1));
    const int grid = 1 << (2 * lp), threads = shift_threads(d.nd, d.p);
    for_shift(d.nd, d.p, [&](auto nc, auto pk) {
      constexpr int NC = decltype(nc)::value, PK = decltype(pk)::value;
      k_fmm_l2l<T2, NC, PK><<<grid, threads, shift_smem<T2>(d.nd, PK), s>>>(d, l0, lp, stop);
    });
    l0 = lp + 1;
  }
  return n;
}

template <class T2>
int fmm_m2m(const FmmDevT<T2>& d, int* arrive, const int* stop, cudaStream_t s) {
  if (d.L <= 2) return 0;
  for_shift(d.nd, d.p, [&](auto nc, auto pk) {
    constexpr int NC = decltype(nc)::value, PK = decltype(pk)::value;
    const size_t sm = shift_smem<T2>(d.nd, PK);
    const auto fn = d.per > 1 ? k_fmm_m2m<T2, NC, PK, true> : k_fmm_m2m<T2, NC, PK, false>;
    fn<<<blocks_for(1LL << (2 * (d.L - 1)), d.per), shift_threads(d.nd, d.p), sm, s>>>(d, arrive, stop);
  });
  return 1;
}

// The upward pass, M2L, downward pass and evaluation with expansions of type T2.
template <class T2, int NEARP>
void fmm_passes(const FmmDevT<T2>& d, FmmState* f, const Geo& g, [[maybe_unused]] VecRef v,
                [[maybe_unused]] const double* sscale, double* partial, const int* stop, cudaStream_t s) {
  const int p = d.p, nd = d.nd;
  const size_t sm_p2m = ((size_t)p * (kChunk + 1) + (size_t)kChunk * nd) * sizeof(T2);
  if constexpr (std::is_same<T2, float2>::value)
    k_fmm_p2m32<<<f->nleaf, kB, sm_p2m, s>>>(d, g, v, sscale, const_cast<float2*>(d.Qf), stop);
  else if constexpr (NEARP == 2)
    k_fmm_p2m_ff<<<f->nleaf, kB, sm_p2m, s>>>(d, g, stop);  // float4 = double2 in size
  else
    k_fmm_p2m<T2><<<f->nleaf, kB, sm_p2m, s>>>(d, g, stop);
  int shifts = fmm_m2m(d, f->arrive, stop, s);
  [[maybe_unused]] bool done = false;
  if constexpr (std::is_same<T2, double2>::value && NEARP == 2) {
    // the float-float residual operator: float-float M2L
    const float* tab = nullptr;
    for (auto& o : f->opsff)
      if (o.first == p) tab = o.second;
    if (tab) {
      const long long nmp = (lev_off(f->L + 1) - lev_off(2)) * nd * p;
      k_fmm_mp_ff<<<grid_for(nmp), 256, 0, s>>>(d.mp + lev_off(2) * nd * p, nmp, f->mpff + lev_off(2) * nd * p);
      launch_m2l_ff(d, f->mpff, tab, f->L, stop, s);
      done = true;
    }
  }
  if constexpr (std::is_same<T2, float2>::value) {
    const float2* ptab = d.ops + tab_size(p);
    if (nd == 1)
      launch_m2l32<1>(d, ptab, m2l32_pad(p), f->L, stop, s);
    else
      launch_m2l32<3>(d, ptab, m2l32_pad(p), f->L, stop, s);
  } else {
    if (!done) launch_m2l(d, f->L, stop, s);
  }
  shifts += fmm_l2l(d, stop, s);
  note_launches(shifts);
  const auto eval = d.per > 1 ? k_fmm_eval<T2, NEARP, true> : k_fmm_eval<T2, NEARP, false>;
  eval<<<blocks_for(f->nleaf, d.per), kBE, eval_smem<T2, NEARP>(nd, p), s>>>(d, g, partial, stop);
}

}  // namespace

void fmm_signature(const FmmState* f, std::vector<long long>& key) {
  if (!f) return;
  for (double v : {f->x0, f->y0, f->D}) {
    long long u;
    memcpy(&u, &v, 8);
    key.push_back(u);
  }
  for (long long v : {(long long)f->L, (long long)f->per, (long long)f->tper, f->nbox, (long long)f->M,
                      (long long)f->kind})
    key.push_back(v);
  for (const void* q : {(const void*)f->leaf, (const void*)f->perm, (const void*)f->start, (const void*)f->count,
                        (const void*)f->arrive, (const void*)f->Q, (const void*)f->mp, (const void*)f->lc,
                        (const void*)f->mpff, (const void*)f->cen32})
    key.push_back((long long)(uintptr_t)q);
  // the operator tables stay where they are as long as the state does
  key.push_back((long long)(uintptr_t)f);
}

cudaError_t fmm_pair_sum(FmmState* f, const Geo& g, int kind, int p, VecRef v, const double* sscale,
                         double* partial, const int* stop, cudaStream_t s, int near_prec) {
  if (!f || p > f->pmax || kind != f->kind) return cudaErrorInvalidValue;
  double2* ops = nullptr;
  float2* ops32 = nullptr;
  for (auto& o : f->ops)
    if (o.first == p) ops = o.second;
  for (auto& o : f->ops32)
    if (o.first == p) ops32 = o.second;
  if (!ops || !ops32) return cudaErrorInvalidValue;  // fmm_setup prepares every order
  const int nd = kind == 0 ? 1 : 3;
  if (near_prec == 1) {
    // the inner solves' operator: FP32 strengths, expansions (in the FP64
    // buffers) and near field
    float2* Qf = reinterpret_cast<float2*>(f->Q);
    FmmDevT<float2> d{f->L,     f->nb,     p,        nd,       g.M,     0,       kind == 1 ? 2 : -1,
                      f->x0,    f->y0,     f->D,     1.0 / f->D, f->leaf,  f->perm, f->start,
                      f->count, f->count,  f->Q,     reinterpret_cast<float2*>(f->mp),
                      reinterpret_cast<float2*>(f->lc), ops32};
    d.Qf = Qf;
    d.cen32 = f->cen32;
    d.is32 = (float)ldexp(1.0 / f->D, f->L);
    d.s32 = (float)ldexp(f->D, -f->L);
    d.per = f->per;
    d.tper = f->tper;
    fmm_passes<float2, 1>(d, f, g, v, sscale, partial, stop, s);
  } else {
    k_fmm_density<<<grid_for(g.M), 256, 0, s>>>(g, nd, f->x0 + 0.5 * f->D, f->y0 + 0.5 * f->D, v, sscale, f->Q,
                                                 stop);
    FmmDev d{f->L,    f->nb,    p,     nd,    g.M,   0,   kind == 1 ? 2 : -1, f->x0, f->y0, f->D, 1.0 / f->D, f->leaf,
                   f->perm, f->start, f->count, f->count, f->Q, f->mp, f->lc,  ops};
    d.per = f->per;
    d.tper = f->tper;
    if (near_prec == 2)
      fmm_passes<double2, 2>(d, f, g, v, sscale, partial, stop, s);
    else
      fmm_passes<double2, 0>(d, f, g, v, sscale, partial, stop, s);
  }
  note_launches(4 + (near_prec == 2 ? 1 : near_prec == 1 ? -1 : 0));
  return cudaGetLastError();
}

}  // namespace bie

namespace bie {

// The output single layers at the interior targets by the FMM of order p
// (logarithm and Cauchy channels on the source tree of fmm_setup).
cudaError_t fmm_output(FmmState* f, const Geo& g, int kind, int p, const double* v, double* part, cudaStream_t s,
                       bool ff) {
  if (!f || p > f->pmax || kind != f->kind) return cudaErrorInvalidValue;
  double2* ops = nullptr;
  for (auto& o : f->ops)
    if (o.first == p) ops = o.second;
  if (!ops) return cudaErrorInvalidValue;
  const int nd = kind == 0 ? 1 : 4, nlog = kind == 0 ? 1 : 2, per = kind == 0 ? 1 : 3;
  const int T = g.N * per;
  const double c0x = f->x0 + 0.5 * f->D, c0y = f->y0 + 0.5 * f->D;
  cudaError_t e = cudaMemsetAsync(f->tcount, 0, (size_t)f->nbox * 4, s);
  if (e != cudaSuccess) return e;
  k_fmm_targets<<<grid_for(T), 256, 0, s>>>(g, per, f->L, f->x0, f->y0, f->D, f->tx, f->ty, f->tleaf,
                                          f->tcount + lev_off(f->L));
  for (int l = f->L - 1; l >= 0; --l) k_fmm_parent_counts<<<grid_for(1LL << (2 * l)), 256, 0, s>>>(l, f->tcount);
  k_fmm_out_density<<<grid_for(g.M), 256, 0, s>>>(g, nd, c0x, c0y, v, f->Q);
  FmmDev d{f->L, f->nb, p, nd, g.M, nlog, -1, f->x0, f->y0, f->D, 1.0 / f->D, f->leaf, f->perm, f->start, f->count, f->tcount,
           f->Q, f->mp, f->lc, ops};
  d.per = f->per;
  d.tper = boxes_a_block_levels(f->L, [&](int) { return (double)T; });
  const size_t sm_p2m = ((size_t)p * (kChunk + 1) + (size_t)kChunk * nd) * sizeof(double2);
  if (ff)
    k_fmm_p2m_ff<<<f->nleaf, kB, sm_p2m, s>>>(d, g, nullptr);  // float4 = double2 in size
  else
    k_fmm_p2m<double2><<<f->nleaf, kB, sm_p2m, s>>>(d, g, nullptr);
  int shifts = fmm_m2m(d, f->arrive, nullptr, s);
  const float* tab = nullptr;
  for (auto& o : f->opsff)
    if (o.first == p) tab = o.second;
  if (ff && tab) {
    // float-float multipole-to-local step (the float-float refinement's solves)
    const long long nmp = (lev_off(f->L + 1) - lev_off(2)) * nd * p;
    k_fmm_mp_ff<<<grid_for(nmp), 256, 0, s>>>(f->mp + lev_off(2) * nd * p, nmp, f->mpff + lev_off(2) * nd * p);
    launch_m2l_ff(d, f->mpff, tab, f->L, nullptr, s);
    note_launches(1);
  } else {
    launch_m2l(d, f->L, nullptr, s);
  }
  shifts += fmm_l2l(d, nullptr, s);
  k_fmm_eval_targets<<<(T + kTW - 1) / kTW, 32 * kTW, 0, s>>>(d, g, kind, T, f->tx, f->ty, f->tleaf, c0x, c0y,
                                                               part);
  note_launches(7 + f->L + shifts);
  return cudaGetLastError();
}

}  // namespace bie

// dec_hodge.cu - the diagonal Hodge star *1 on primal edges from the
// circumcentric dual (Sec. 2.1: ratio of dual to primal volumes), times the
// conductivity of the dual face (Sec. 2.1), with penny cracks making cut dual
// faces insulating (Sec. 2.5).  A per-tet conductivity k_T is carried onto
// the dual face of e as the mean of k_T over the tets around e, weighted by
// the unsigned areas of their parts of the face.
//
// One thread per tet computes, in FP64, for each of its 6 edges the signed
// area of the dual-face piece inside the tet divided by the edge length.
// The piece of edge e = (a, b) splits into two right triangles (m_e, c_F,
// c_T), one per face F = {a, b, c} of the tet containing e: legs h1 = signed
// distance from the midpoint m_e to c_F inside F (+ towards c) and h2 =
// signed distance from c_T to the plane of F (+ towards the fourth vertex).
// With h1 = |e|/2 cot(angle at c), cot = (x_a-x_c).(x_b-x_c) / |N_F| and
// h2 = (c_T - x_a).N_F / |N_F| (N_F the inward face normal, |N_F| = twice
// the face area), each half contributes
//   (1/2) h1 h2 / |e| = (1/4) (x_a-x_c).(x_b-x_c) (c_T - x_a).N_F / |N_F|^2,
// so the kernel needs one division per face and none per edge (FP64
// division and square root are expensive on GB300).  The crack test runs on
// the sub-triangles themselves, with face circumcentres computed only when
// discs are present.  A second pass sums the
// pieces of every edge (and, with a conductivity field, the k-weighted and
// plain unsigned part areas) in a fixed order (sorted tet*6+slot), so *1 is
// deterministic without atomics.
#include "dec_internal.cuh"

#include <math_constants.h>

#include <algorithm>
#include <cmath>
#include <vector>

namespace dec {

template <typename T>
struct Vec3 {
  T x, y, z;
};
using V3 = Vec3<double>;
using F3 = Vec3<float>;
__device__ __forceinline__ V3 mk(double x, double y, double z) { return {x, y, z}; }
template <typename T>
__device__ __forceinline__ Vec3<T> operator+(Vec3<T> a, Vec3<T> b) {
  return {a.x + b.x, a.y + b.y, a.z + b.z};
}
template <typename T>
__device__ __forceinline__ Vec3<T> operator-(Vec3<T> a, Vec3<T> b) {
  return {a.x - b.x, a.y - b.y, a.z - b.z};
}
template <typename T>
__device__ __forceinline__ Vec3<T> operator*(T s, Vec3<T> a) {
  return {s * a.x, s * a.y, s * a.z};
}
template <typename T>
__device__ __forceinline__ T dot(Vec3<T> a, Vec3<T> b) {
  return a.x * b.x + a.y * b.y + a.z * b.z;
}
template <typename T>
__device__ __forceinline__ Vec3<T> cross(Vec3<T> a, Vec3<T> b) {
  return {a.y * b.z - a.z * b.y, a.z * b.x - a.x * b.z, a.x * b.y - a.y * b.x};
}

// Tet circumcentre relative to vertex 0, from the edge vectors R[1..3]:
// (|a|^2 (b x c) + |b|^2 (c x a) + |c|^2 (a x b)) / (2 a.(b x c))
template <typename T>
__device__ __forceinline__ Vec3<T> tet_circumcentre(const Vec3<T> (&R)[4]) {
  const Vec3<T> bxc = cross(R[2], R[3]), cxa = cross(R[3], R[1]), axb = cross(R[1], R[2]);
  const T det6 = dot(R[1], bxc);
  return (T(0.5) / det6) * (dot(R[1], R[1]) * bxc + dot(R[2], R[2]) * cxa +
                            dot(R[3], R[3]) * axb);
}

// circumcentre of triangle (p, p+a, p+b): p + ((|a|^2 b - |b|^2 a) x (a x b)) / (2 |a x b|^2)
__device__ __forceinline__ V3 tri_circumcentre(V3 p, V3 q, V3 r) {
  V3 a = q - p, b = r - p;
  V3 axb = cross(a, b);
  V3 num = cross(dot(a, a) * b - dot(b, b) * a, axb);
  return p + (0.5 / dot(axb, axb)) * num;
}

// Distance, in the disc's plane, from the disc centre to the segment where
// the plane meets the closed triangle (P0, P1, P2); +inf when the plane misses
// the triangle or contains it.
// s0..s2 are the signed distances dot(P_i - c, nrm) of the three points.
// Not inlined: the exact test runs for few (tet, disc) pairs, and twelve
// inlined copies made the kernel large enough to stall on instruction fetch.
__device__ __noinline__ double crack_rho_s(V3 P0, V3 P1, V3 P2, double s0, double s1,
                                           double s2, V3 c) {
  V3 P[3] = {P0, P1, P2};
  const double s[3] = {s0, s1, s2};
  int count = 0;
  V3 A = mk(0, 0, 0), B = mk(0, 0, 0);
  const int ei[3] = {0, 1, 0}, ej[3] = {1, 2, 2};
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    double si = s[ei[k]], sj = s[ej[k]];
    if (si * sj < 0.0) {
      double t = si / (si - sj);
      V3 X = P[ei[k]] + t * (P[ej[k]] - P[ei[k]]);
      if (count == 0) A = X; else if (count == 1) B = X;
      ++count;
    }
  }
#pragma unroll
  for (int i = 0; i < 3; ++i) {
    if (s[i] == 0.0) {
      if (count == 0) A = P[i]; else if (count == 1) B = P[i];
      ++count;
    }
  }
  if (count == 0 || count >= 3) return CUDART_INF;
  if (count == 1) B = A;
  V3 d = B - A;
  double dd = dot(d, d);
  double tt = 0.0;
  if (dd > 0.0) tt = fmin(fmax(dot(c - A, d) / dd, 0.0), 1.0);
  V3 cl = A + tt * d;
  V3 g = c - cl;
  return sqrt(dot(g, g));
}

constexpr float kU = 5.9604645e-8f;    // 2^-24, the rounding unit of FP32

struct DiscGrid {
  double lo[3];
  double inv_cell;
  int dim[3];
  const int32_t* start;   // [cells+1]
  const int32_t* items;   // disc ids
  const double* discs;    // [nd][7]
  const float4* discs_f;  // [nd][2]: (centre, bound on |centre|), (normal, reach rounded up)
  const double* scales;   // [n_states]
  const float* scales_f;  // [n_states], rounded
  int n_states;
  int nd;
  bool fp32;              // radii and scales in FP32's range: sub-triangle tests in FP32
  double smax;            // largest radius scale
};

__constant__ int kEdgeA[6] = {0, 0, 0, 1, 1, 2};
__constant__ int kEdgeB[6] = {1, 2, 3, 2, 3, 3};
__constant__ int kEdgeC[6] = {2, 1, 1, 0, 0, 0};  // the two other vertices
__constant__ int kEdgeD[6] = {3, 3, 2, 3, 2, 1};

// FP64 test of one sub-triangle (edge midpoint, circumcentre of the face
// opposite local vertex opp, tet circumcentre cT) against disc id: the first
// state below `first` whose disc cuts it, or `first`.
__device__ __noinline__ int crack_exact(const double* __restrict__ xyz, int4 v4, int ea, int eb,
                                        int opp, V3 cT, const DiscGrid& grid, int id, int first) {
  const int vid[4] = {v4.x, v4.y, v4.z, v4.w};
  auto node = [&](int l) {
    const double* p = xyz + 3 * (int64_t)vid[l];
    return mk(p[0], p[1], p[2]);
  };
  const double* dsc = grid.discs + 7 * (int64_t)id;
  const V3 dc = mk(dsc[0], dsc[1], dsc[2]), dn = mk(dsc[3], dsc[4], dsc[5]);
  const double r = dsc[6];
  const V3 me = 0.5 * (node(ea) + node(eb));
  const V3 cF = tri_circumcentre(node((opp + 1) & 3), node((opp + 2) & 3), node((opp + 3) & 3));
  const double sM = dot(me - dc, dn), sF = dot(cF - dc, dn), sT = dot(cT - dc, dn);
  if ((sM > 0.0 && sF > 0.0 && sT > 0.0) || (sM < 0.0 && sF < 0.0 && sT < 0.0)) return first;
  const double rho = crack_rho_s(me, cF, cT, sM, sF, sT, dc);
  for (int st = 0; st < first; ++st)
    if (rho <= grid.scales[st] * r) return st;
  return first;
}

// first st < n with x <= scales[st] * f (scales increase)
__device__ __forceinline__ int first_state(const float* __restrict__ scales, int n, float x,
                                           float f) {
  int lo = 0, hi = n;
  while (lo < hi) {
    const int mid = (lo + hi) >> 1;
    if (x <= __ldg(scales + mid) * f) hi = mid; else lo = mid + 1;
  }
  return lo;
}

// The 11 corners of a tet's 12 dual sub-triangles in FP32, relative to vertex
// 0, in shared memory: 6 edge midpoints, 4 face circumcentres (kept per
// opposite vertex), the tet circumcentre; pts[3 * corner + axis][thread].
constexpr int kHodgeThreads = 128;
using CrackPts = float[33][kHodgeThreads];

__device__ __forceinline__ F3 pt_load(const CrackPts& pts, int c) {
  return {pts[3 * c][threadIdx.x], pts[3 * c + 1][threadIdx.x], pts[3 * c + 2][threadIdx.x]};
}
__device__ __forceinline__ void pt_store(CrackPts& pts, int c, F3 v) {
  pts[3 * c][threadIdx.x] = v.x;
  pts[3 * c + 1][threadIdx.x] = v.y;
  pts[3 * c + 2][threadIdx.x] = v.z;
}

// Forms the corners from the edge vectors R (rounded once from FP64) and cT
// (error at most eT), and bounds their error E and their size P.  With u =
// 2^-24, l the longer side and tau = l^2 / |a x b|, the rounded circumcentre
// of a triangle is off by at most u l (36 tau^2 + 24 tau): 12 u tau from the
// cross product in numerator and, twice, denominator (|c| <= l tau), 2 u from
// each rsqrtf, the rest from |a|^2 b - |b|^2 a; 64 u l tau (1 + tau) is used.
// Returns false when the bound is too loose to be of use (thin faces: edges
// of one face that differ 50-fold already are), when a corner is not finite,
// and where the longest edge from vertex 0 is out of [1e-8, 1e8]: |a x b|^2
// goes with l^4 and would leave FP32's normal range, which no bound here
// covers (the FP64 test takes such tets).  Out of line: inlined, the extra
// checks spilled 50 bytes more and 12.1 M tets with 1,500 discs took 11.2 ms
// instead of 10.9.
__device__ __noinline__ bool crack_points(const F3 (&R)[4], F3 cT, float eT, CrackPts& pts,
                                             float& E, float& P) {
  float L2 = 0.0f, e = eT, p2 = dot(cT, cT);
#pragma unroll
  for (int i = 1; i < 4; ++i) L2 = fmaxf(L2, dot(R[i], R[i]));
  bool usable = L2 > 1e-16f && L2 < 1e16f && p2 < 1e30f;     // false for NaN, too
  pt_store(pts, 0, 0.5f * (R[0] + R[1]));
  pt_store(pts, 1, 0.5f * (R[0] + R[2]));
  pt_store(pts, 2, 0.5f * (R[0] + R[3]));
  pt_store(pts, 3, 0.5f * (R[1] + R[2]));
  pt_store(pts, 4, 0.5f * (R[1] + R[3]));
  pt_store(pts, 5, 0.5f * (R[2] + R[3]));
#pragma unroll
  for (int v = 0; v < 4; ++v) {
    const F3 o = R[(v + 1) & 3], a = R[(v + 2) & 3] - o, b = R[(v + 3) & 3] - o;
    const F3 axb = cross(a, b);
    const float aa = dot(a, a), bb = dot(b, b), in = rsqrtf(dot(axb, axb));
    // the normal to unit length first: products stay below l^4
    const F3 c = o + (0.5f * in) * cross(aa * b - bb * a, in * axb);
    pt_store(pts, 6 + v, c);
    const float l2 = fmaxf(aa, bb), tau = l2 * in;
    usable = usable && tau < 1e4f;
    // the sides a, b carry the roundings of two edge vectors (of size up to
    // sqrt(L2)) and one more
    e = fmaxf(e, 128.0f * kU * sqrtf(fmaxf(l2, L2)) * tau * (1.0f + tau));
    p2 = fmaxf(p2, dot(c, c));
  }
  pt_store(pts, 10, cT);
  P = sqrtf(fmaxf(p2, L2)) * 1.001f;
  E = e * 1.01f + 8.0f * kU * P;
  return usable && E < 0.02f * sqrtf(L2);
}

// The two halves of every slot's piece of dual face (below), from the edge
// vectors R[1..3] of the tet (R[0] = 0): the circumcentre cT and, per face,
// H[v] = signed distance from c_T to the face opposite v (+ towards v)
// divided by twice the face area, ((c_T - x).N) / |N|^2 with N the inward
// normal.  Half of the dual face of edge (a,b) inside face F = {a,b,c} is
// the right triangle (m_e, c_F, c_T) with legs |e|/2 * cot(angle at c) and
// the distance from c_T to F; with cot = (x_a-x_c).(x_b-x_c) / |N_F| its
// area over |e| is (1/4) (x_a-x_c).(x_b-x_c) * H_F.
template <typename T>
__device__ __forceinline__ void tet_pieces(const Vec3<T> (&R)[4], Vec3<T>& cT, T (&a0)[6],
                                           T (&a1)[6]) {
  // For a positively oriented tet the inward normals of the faces opposite
  // vertices 1, 2, 3 are the cross products the circumcentre needs, and the
  // one opposite vertex 0 is minus their sum; |N_v| is twice the face area.
  const Vec3<T> bxc = cross(R[2], R[3]), cxa = cross(R[3], R[1]), axb = cross(R[1], R[2]);
  const T det6 = dot(R[1], bxc);
  const Vec3<T> N[4] = {T(-1) * (bxc + cxa + axb), bxc, cxa, axb};
  T nn[4];
#pragma unroll
  for (int v = 0; v < 4; ++v) nn[v] = dot(N[v], N[v]);
  // 1 / det6 and 1 / |N_v|^2: in FP64 one division of their product and
  // products of the others (the division is a long instruction sequence on
  // GB300's narrow FP64 pipe); five divisions when the product leaves the
  // normal range, and always in FP32
  T inv_det, inv_nn[4];
  bool direct = true;
  if constexpr (sizeof(T) == sizeof(double)) {
    const T p01 = det6 * nn[0], p012 = p01 * nn[1], p0123 = p012 * nn[2];
    const T prod = p0123 * nn[3];
    if (prod > 1e-280 && prod < 1e280) {
      direct = false;
      const T r = T(1) / prod;
      const T s3 = nn[3], s23 = nn[2] * s3, s123 = nn[1] * s23;
      inv_det = r * (nn[0] * s123);
      inv_nn[0] = r * (det6 * s123);
      inv_nn[1] = r * (p01 * s23);
      inv_nn[2] = r * (p012 * s3);
      inv_nn[3] = r * p0123;
    }
  }
  if (direct) {
    inv_det = T(1) / det6;
#pragma unroll
    for (int v = 0; v < 4; ++v) inv_nn[v] = T(1) / nn[v];
  }
  cT = (T(0.5) * inv_det) * (dot(R[1], R[1]) * bxc + dot(R[2], R[2]) * cxa +
                             dot(R[3], R[3]) * axb);
  // H[v]: signed distance from c_T to the face opposite v (+ towards v)
  // over twice the face area; faces 1-3 contain vertex 0 (R[0] = 0)
  T H[4];
  H[0] = dot(cT - R[1], N[0]) * inv_nn[0];
#pragma unroll
  for (int v = 1; v < 4; ++v) H[v] = dot(cT, N[v]) * inv_nn[v];
  // the six edge vectors; (x_a - x_c).(x_b - x_c) are dot products of two
  // edges at vertex c.  Slot s joins local vertices (a, b); c and d are the
  // other two (the slots of kEdgeA..D, spelled out so that every index is
  // a compile-time constant and the vectors stay in registers).
  const Vec3<T> E[4][4] = {
      {R[0], R[1], R[2], R[3]},
      {T(-1) * R[1], R[0], R[2] - R[1], R[3] - R[1]},
      {T(-1) * R[2], R[1] - R[2], R[0], R[3] - R[2]},
      {T(-1) * R[3], R[1] - R[3], R[2] - R[3], R[0]}};   // E[i][j] = x_j - x_i
  auto slot = [&](int s, int a, int b, int c, int d) {
    const T cot_c = dot(E[c][a], E[c][b]);   // face opposite d
    const T cot_d = dot(E[d][a], E[d][b]);   // face opposite c
    a0[s] = T(0.25) * cot_c * H[d];
    a1[s] = T(0.25) * cot_d * H[c];
  };
  slot(0, 0, 1, 2, 3);
  slot(1, 0, 2, 1, 3);
  slot(2, 0, 3, 1, 2);
  slot(3, 1, 2, 0, 3);
  slot(4, 1, 3, 0, 2);
  slot(5, 2, 3, 0, 1);
}

// The ball test is conservative (the in-plane reach is bounded by
// r + R_T).  Most candidate discs are far from the tet, and GB300's FP64 pipe is
// narrow, so the two rejections are first made entirely in FP32 from
// c_T rounded once per tet and the discs rounded once on the host.
// With u = 2^-24 and S = A_t + A_d (bounds on |c_T| and |centre| per
// coordinate), the offset v = c_T - centre carries an error of at most
// 2uS per coordinate, so (first order, |normal| = 1):
//   |dp32 - dp| <= 6 sqrt(3) u S,   |par32 - par| <= 63 u S^2
// (dp the distance to the disc plane, par = |v|^2 - dp^2).  The
// margins below are twice these plus the roundings of the thresholds,
// so FP32 rejects only where the FP64 test rejects too: the decisions,
// and so *1 and the crack states, are unchanged.
struct BallF {
  float x, y, z;    // centre
  float A, R;       // bound on the centre's coordinates, radius rounded up
};
__device__ __forceinline__ BallF ball_f32(V3 c, double R) {
  BallF b{(float)c.x, (float)c.y, (float)c.z, 0.0f, (float)R * (1.0f + 4.0f * kU)};
  b.A = fmaxf(fabsf(b.x), fmaxf(fabsf(b.y), fabsf(b.z))) * (1.0f + 2.0f * kU);
  return b;
}
__device__ __forceinline__ bool ball_meets_disc(const DiscGrid& grid, const BallF& b, int id) {
  const float4 d0 = __ldg(grid.discs_f + 2 * (int64_t)id);
  const float4 d1 = __ldg(grid.discs_f + 2 * (int64_t)id + 1);
  const float vx = b.x - d0.x, vy = b.y - d0.y, vz = b.z - d0.z;
  const float S = b.A + d0.w;
  const float dpf = fmaf(vx, d1.x, fmaf(vy, d1.y, vz * d1.z));
  if (fabsf(dpf) > b.R + (24.0f * S + 8.0f * b.R) * kU) return false;   // ball misses the plane
  const float vv = fmaf(vx, vx, fmaf(vy, vy, vz * vz));
  const float par = fmaf(-dpf, dpf, vv);
  const float T = d1.w + b.R;
  return !(par > T * T * (1.0f + 8.0f * kU) + 128.0f * kU * S * S);     // else misses the disc
}

// test(id) for every disc whose cells the box of the ball (c, R) meets
template <typename Test>
__device__ __forceinline__ void for_candidates(const DiscGrid& grid, V3 c, double R, Test&& test) {
  const double lo[3] = {c.x - R, c.y - R, c.z - R};
  const double hi[3] = {c.x + R, c.y + R, c.z + R};
  int c0[3], c1[3];
  bool empty = false;
#pragma unroll
  for (int d = 0; d < 3; ++d) {
    double f0 = (lo[d] - grid.lo[d]) * grid.inv_cell;
    double f1 = (hi[d] - grid.lo[d]) * grid.inv_cell;
    if (f1 < 0.0 || f0 >= (double)grid.dim[d]) empty = true;
    c0[d] = (int)fmax(0.0, floor(f0));
    c1[d] = (int)fmin((double)grid.dim[d] - 1.0, floor(f1));
  }
  if (empty) return;
  const int64_t ncell = (int64_t)(c1[0] - c0[0] + 1) * (c1[1] - c0[1] + 1) *
                        (c1[2] - c0[2] + 1);
  // a far circumcentre (flat boundary tet): fewer tests without the
  // grid, i.e. every disc once (one pass of the loops below); one call
  // site of test keeps the kernel small
  const bool all = ncell > grid.nd;
  if (all) c1[0] = c0[0], c1[1] = c0[1], c1[2] = c0[2];
  for (int gz = c0[2]; gz <= c1[2]; ++gz)
    for (int gy = c0[1]; gy <= c1[1]; ++gy)
      for (int gx = c0[0]; gx <= c1[0]; ++gx) {
        const int cell = gx + grid.dim[0] * (gy + grid.dim[1] * gz);
        const int i0 = all ? 0 : grid.start[cell];
        const int i1 = all ? grid.nd : grid.start[cell + 1];
        for (int it = i0; it < i1; ++it) test(all ? it : grid.items[it]);
      }
}

// Bounds of the FP32 geometry (DEC_GEOM_MIXED): a tet is computed in FP32
// when L^3 <= kShapeMax |6 V|, L the longest of its edges from vertex 0 (a
// regular tet has 2.8, a Kuhn tet 5.2; 96 % of the tets of a jittered Delaunay
// cube pass 16), and L lies in [1e-7, 1e7], where fourth powers of lengths and
// their inverses stay in FP32's normal range; in FP64 otherwise.
constexpr float kShapeMax = 16.0f;
constexpr float kMinEdge2 = 1e-14f, kMaxEdge2 = 1e14f;

// MIXED = false: every tet in FP64.  MIXED = true: well-shaped tets in FP32.
// n_fp64 counts the tets computed in FP64, n_thin those left to
// crack_thin_kernel (thin: 2 * tet + FP32 geometry, in any order).
template <bool MIXED>
__global__ void __launch_bounds__(kHodgeThreads, 3)
hodge_tet_kernel(const double* __restrict__ xyz, const int32_t* __restrict__ tets,
                 const double* __restrict__ kcond, int64_t m,
                 double* __restrict__ piece, double* __restrict__ kpart,
                 uint8_t* __restrict__ slot_cut, DiscGrid grid,
                 unsigned long long* __restrict__ n_fp64, unsigned long long* __restrict__ n_thin,
                 uint32_t* __restrict__ thin) {
  __shared__ CrackPts pts;
  unsigned n64 = 0;
  for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < m;
       t += (int64_t)gridDim.x * blockDim.x) {
    int4 v4 = reinterpret_cast<const int4*>(tets)[t];
    const int vid[4] = {v4.x, v4.y, v4.z, v4.w};
    V3 X[4];
#pragma unroll
    for (int i = 0; i < 4; ++i)
      X[i] = mk(xyz[3 * (int64_t)vid[i]], xyz[3 * (int64_t)vid[i] + 1],
                xyz[3 * (int64_t)vid[i] + 2]);
    const double kT = kcond ? kcond[t] : 1.0;
    const int64_t q6 = 6 * m;
    V3 cT;                 // circumcentre relative to X[0]
    double a0[6], a1[6];
    double Et = 0.0;       // bound on the error of cT (FP32 geometry)
    bool fast = false;
    if constexpr (MIXED) {
      // edge vectors formed in FP64 and rounded once: each coordinate
      // carries a relative error of at most 2^-24
      F3 Rf[4];
      Rf[0] = {0.0f, 0.0f, 0.0f};
#pragma unroll
      for (int i = 1; i < 4; ++i)
        Rf[i] = {(float)(X[i].x - X[0].x), (float)(X[i].y - X[0].y),
                 (float)(X[i].z - X[0].z)};
      const float det6 = fabsf(dot(Rf[1], cross(Rf[2], Rf[3])));
      const float L2 = fmaxf(dot(Rf[1], Rf[1]), fmaxf(dot(Rf[2], Rf[2]), dot(Rf[3], Rf[3])));
      const float L = sqrtf(L2);
      if (L2 * L <= kShapeMax * det6 && L2 > kMinEdge2 && L2 < kMaxEdge2) {
        fast = true;
        F3 cTf;
        float b0[6], b1[6];
        tet_pieces(Rf, cTf, b0, b1);
#pragma unroll
        for (int s = 0; s < 6; ++s) {
          a0[s] = b0[s];
          a1[s] = b1[s];
        }
        cT = mk(cTf.x, cTf.y, cTf.z);
        // With rho = L^3 / |6V| the rounded edge vectors move the
        // circumcentre (the solution of 2 R c = |R_i|^2, whose matrix has
        // smallest singular value >= |6V| / (3 L^2)) by at most
        // (17 rho + 24 rho^2) u L; the formula's own roundings are of the same
        // order.  Et doubles the sum (u = 2^-24).
        const double rho = (double)(L2 * L) / (double)det6;
        Et = 64.0 * 5.9604645e-8 * rho * (1.0 + rho) * (double)L;
      }
    }
    if (!fast) {
      V3 R[4];
      R[0] = mk(0.0, 0.0, 0.0);
#pragma unroll
      for (int i = 1; i < 4; ++i) R[i] = X[i] - X[0];
      tet_pieces(R, cT, a0, a1);
      ++n64;
    }
    uint8_t first[6];
#pragma unroll
    for (int s = 0; s < 6; ++s) {
      piece[t * 6 + s] = a0[s] + a1[s];
      if (kcond) {                       // unsigned part of the face, with and without k
        const double u = fabs(a0[s]) + fabs(a1[s]);
        kpart[t * 6 + s] = kT * u;
        kpart[q6 + t * 6 + s] = u;
      }
      first[s] = (uint8_t)grid.n_states;
    }
    if (grid.nd > 0) {
      // Every dual sub-triangle of the tet lies in its circumball (c_T is
      // the centre; m_e and c_F are projections of c_T onto an edge line and
      // a face plane), so a disc that misses the ball cuts none of them and
      // the candidate discs are those binned in the cells the ball's box
      // meets.  The radius carries a relative margin; the cut decision
      // itself stays exact.
      // With FP32 geometry the ball is centred on the rounded circumcentre
      // and its radius grows by twice the error bound, so it still holds the
      // exact ball; the exact circumcentre cTx is then formed in FP64 for a
      // tet that some disc may cut.
      const V3 cTa = X[0] + cT;
      double RT2, RT;
      if (fast) {
        RT = (sqrt(dot(cT, cT)) + 2.0 * Et) * (1.0 + 1e-9);
        RT2 = RT * RT;
      } else {
        RT2 = dot(cT, cT) * (1.0 + 1e-9) + 1e-300;
        RT = sqrt(RT2);
      }
      V3 cTx = cTa;
      bool have_cTx = !fast;
      auto exact_cT = [&]() {
        if (!have_cTx) {
          V3 R[4];
          R[0] = mk(0.0, 0.0, 0.0);
#pragma unroll
          for (int i = 1; i < 4; ++i) R[i] = X[i] - X[0];
          cTx = X[0] + tet_circumcentre(R);
          have_cTx = true;
        }
        return cTx;
      };
      // corners of the sub-triangles: only for a tet that some disc may cut
      int have_pts = 0;                     // 1: in pts, -1: FP64 only
      float Ept = 0.0f, Ppt = 0.0f;
      const BallF ball = ball_f32(cTa, RT);
      auto test_disc = [&](int id) {
        if (have_pts < 0 || !ball_meets_disc(grid, ball, id)) return;
        // The sub-triangles are then tested in FP32 on corners relative to
        // vertex 0, with bounds on every step's error, and in FP64 only where
        // a bound leaves the answer open (about 1 % of the pairs of tet and
        // disc that come this far): the answers are those of the FP64 test.
        // The FP64 tests were four fifths of the assembly: 34.4 ms for 12.1 M
        // tets and 1,500 discs, 11.1 ms with this.  Tets whose corners are of no
        // use in FP32 (thin ones) go to crack_thin_kernel.
        if (have_pts == 0) {
          F3 Rf[4];
          Rf[0] = {0.0f, 0.0f, 0.0f};
#pragma unroll
          for (int i = 1; i < 4; ++i)
            Rf[i] = {(float)(X[i].x - X[0].x), (float)(X[i].y - X[0].y),
                     (float)(X[i].z - X[0].z)};
          const F3 c = {(float)cT.x, (float)cT.y, (float)cT.z};
          have_pts =
              grid.fp32 && crack_points(Rf, c, (float)(2.0 * Et), pts, Ept, Ppt) ? 1 : -1;
          if (have_pts < 0) return;
        }
        const double* dsc = grid.discs + 7 * (int64_t)id;
        const F3 c = {(float)(dsc[0] - X[0].x), (float)(dsc[1] - X[0].y),
                      (float)(dsc[2] - X[0].z)};
        const float4 d1 = __ldg(grid.discs_f + 2 * (int64_t)id + 1);
        const F3 nrm = {d1.x, d1.y, d1.z};
        const float r = (float)dsc[6];
        const float size = sqrtf(dot(c, c)) + Ppt;      // bound on |corner - centre|
        // signed distances to the plane: corner and centre errors, 16 u for
        // the rounded normal and the dot product
        const float Es = Ept + 16.0f * kU * size;
        const float sT = dot(pt_load(pts, 10) - c, nrm);
#pragma unroll 1
        for (int s = 0; s < 6; ++s) {
          if (first[s] == 0) continue;
          const F3 M = pt_load(pts, s);
          const float sM = dot(M - c, nrm);
#pragma unroll 1
          for (int h = 0; h < 2; ++h) {
            const int opp = h == 0 ? kEdgeD[s] : kEdgeC[s];
            int st = first[s];
            const F3 F = pt_load(pts, 6 + opp);
            const float sf = dot(F - c, nrm);
            const float lo3 = fminf(sM, fminf(sf, sT)), hi3 = fmaxf(sM, fmaxf(sf, sT));
            if (lo3 > Es || hi3 < -Es) continue;      // one side: not cut
            bool open = fminf(fabsf(sM), fminf(fabsf(sf), fabsf(sT))) <= Es;
            if (!open) {
              // one corner (P0) on its own side: the plane meets the two
              // edges from it
              const F3 T = pt_load(pts, 10);
              const bool m1 = (sM > 0.0f) != (sT > 0.0f), f1 = (sf > 0.0f) != (sT > 0.0f);
              const F3 P0 = m1 && f1 ? T : m1 ? M : F;
              const F3 P1 = m1 && f1 ? M : m1 ? F : M;
              const F3 P2 = m1 && f1 ? F : T;
              const float s0 = m1 && f1 ? sT : m1 ? sM : sf;
              const float s1 = m1 && f1 ? sM : m1 ? sf : sM;
              const float s2 = m1 && f1 ? sf : sT;
              const F3 u1 = P1 - P0, u2 = P2 - P0;
              const float i1 = 1.0f / (s0 - s1), i2 = 1.0f / (s0 - s2);
              const F3 A = P0 + (s0 * i1) * u1, B = P0 + (s0 * i2) * u2;
              const F3 d = B - A, g = c - A;
              const float dd = dot(d, d);
              float tt = 0.0f;
              if (dd > 0.0f) tt = fminf(fmaxf(dot(g, d) / dd, 0.0f), 1.0f);
              const F3 w = g - tt * d;
              const float rho = sqrtf(dot(w, w));
              // the crossing parameters move by Es / |s0 - si| and a few
              // roundings; the distance by no more than the end points
              const float EA = (Es * fabsf(i1) + 4.0f * kU) * sqrtf(dot(u1, u1));
              const float EB = (Es * fabsf(i2) + 4.0f * kU) * sqrtf(dot(u2, u2));
              const float Er = 1.01f * (Ept + 2.0f * fmaxf(EA, EB)) + 48.0f * kU * size;
              const int n = first[s];
              st = first_state(grid.scales_f, n, rho + Er, r * (1.0f - 8.0f * kU));
              open = !(Er < size) ||
                     st != first_state(grid.scales_f, n, rho - Er, r * (1.0f + 8.0f * kU));
            }
            if (open)
              st = crack_exact(xyz, v4, kEdgeA[s], kEdgeB[s], opp, exact_cT(), grid, id, first[s]);
            first[s] = (uint8_t)st;
          }
        }
      };
      for_candidates(grid, cTa, RT, test_disc);
      if (have_pts < 0) thin[atomicAdd(n_thin, 1ull)] = 2u * (uint32_t)t + (fast ? 1u : 0u);
    }
#pragma unroll
    for (int s = 0; s < 6; ++s) slot_cut[t * 6 + s] = first[s];
  }
  // tets computed in FP64: one atomic per warp
  const unsigned w64 = __reduce_add_sync(0xffffffffu, n64);
  if ((threadIdx.x & 31) == 0 && w64) atomicAdd(n_fp64, (unsigned long long)w64);
}

// Crack states of the tets that hodge_tet_kernel left over: thin ones, whose
// FP32 corners are of no use, and all that a disc may cut where radii or
// scales leave FP32's range.  Every pair of tet and disc in FP64: the ball test
// first (no cut outside the circumball), then the 12 sub-triangles from face
// circumcentres formed once per tet.  Apart from the others, because inside
// hodge_tet_kernel these tests cost it registers (12.1 M ordinary tets: 11.1 to
// 11.3 ms, 10.9 now).
// Bound by the FP64 pipe.  The 64^3 cube with z scaled by 1e-3 (1e-6) and 300
// discs: 684 (2,240) ms; 2,130 (2,487) with every test of every tet in FP64 in
// one kernel, 2,028 (3,996) with one sub-triangle at a time out of line.
__global__ void __launch_bounds__(kHodgeThreads)
crack_thin_kernel(const double* __restrict__ xyz, const int32_t* __restrict__ tets,
                  int64_t count, const uint32_t* __restrict__ thin,
                  uint8_t* __restrict__ slot_cut, DiscGrid grid) {
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < count;
       i += (int64_t)gridDim.x * blockDim.x) {
    const uint32_t id_fast = thin[i];
    const int64_t t = id_fast >> 1;
    const int4 v4 = reinterpret_cast<const int4*>(tets)[t];
    const int vid[4] = {v4.x, v4.y, v4.z, v4.w};
    V3 X[4], R[4], cT;
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      const double* p = xyz + 3 * (int64_t)vid[k];
      X[k] = mk(p[0], p[1], p[2]);
      R[k] = X[k] - X[0];
    }
    if (id_fast & 1u) {
      cT = tet_circumcentre(R);
    } else {                              // the circumcentre of the FP64 geometry
      double a0[6], a1[6];
      tet_pieces(R, cT, a0, a1);
    }
    const V3 c = X[0] + cT;
    const double RT2 = dot(cT, cT) * (1.0 + 1e-9) + 1e-300, RT = sqrt(RT2);
    const BallF ball = ball_f32(c, RT);
    V3 cF[4];
    bool have_cF = false;
    uint8_t first[6];
#pragma unroll
    for (int s = 0; s < 6; ++s) first[s] = (uint8_t)grid.n_states;
    for_candidates(grid, c, RT, [&](int id) {
      if (!ball_meets_disc(grid, ball, id)) return;
      const double* dsc = grid.discs + 7 * (int64_t)id;
      const V3 dc = mk(dsc[0], dsc[1], dsc[2]), dn = mk(dsc[3], dsc[4], dsc[5]);
      const double r = dsc[6];
      const V3 v = c - dc;
      const double dp = dot(v, dn);
      if (dp * dp > RT2) return;                      // ball misses the plane
      const double par2 = dot(v, v) - dp * dp;
      const double reach = grid.smax * r * (1.0 + 1e-9);
      if (par2 > reach * reach + 2.0 * reach * RT + RT2) return;
      if (!have_cF) {
#pragma unroll
        for (int f = 0; f < 4; ++f)
          cF[f] = tri_circumcentre(X[(f + 1) & 3], X[(f + 2) & 3], X[(f + 3) & 3]);
        have_cF = true;
      }
      const double sT = dot(c - dc, dn);
      double sF[4];
#pragma unroll
      for (int f = 0; f < 4; ++f) sF[f] = dot(cF[f] - dc, dn);
#pragma unroll 1
      for (int s = 0; s < 6; ++s) {
        if (first[s] == 0) continue;
        const V3 me = 0.5 * (X[kEdgeA[s]] + X[kEdgeB[s]]);
        const double sM = dot(me - dc, dn);
#pragma unroll 1
        for (int h = 0; h < 2; ++h) {
          const int opp = h == 0 ? kEdgeD[s] : kEdgeC[s];
          const double sf = sF[opp];
          if ((sM > 0.0 && sf > 0.0 && sT > 0.0) || (sM < 0.0 && sf < 0.0 && sT < 0.0))
            continue;                                 // no crossing
          const double rho = crack_rho_s(me, cF[opp], c, sM, sf, sT, dc);
          for (int st = 0; st < (int)first[s]; ++st)
            if (rho <= grid.scales[st] * r) {
              first[s] = (uint8_t)st;
              break;
            }
        }
      }
    });
#pragma unroll
    for (int s = 0; s < 6; ++s) slot_cut[t * 6 + s] = first[s];
  }
}

// *1[e] = sum of the pieces of e (already divided by |e|), in increasing
// tet*6+slot order, times kappa_e = sum k_T u_T / sum u_T (u_T the unsigned
// part areas, kpart = [k u | u], absent for k = 1); first_cut[e] = min over
// those slots.
__global__ void edge_reduce_kernel(const int32_t* __restrict__ seg_start,
                                   const uint32_t* __restrict__ seg_pay,
                                   const double* __restrict__ piece,
                                   const double* __restrict__ kpart, int64_t q6,
                                   const uint8_t* __restrict__ slot_cut,
                                   int64_t ne, double* __restrict__ w,
                                   uint8_t* __restrict__ first_cut) {
  for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < ne;
       e += (int64_t)gridDim.x * blockDim.x) {
    double sum = 0.0, ku = 0.0, u = 0.0;
    unsigned fc = 255u;
    for (int32_t k = seg_start[e]; k < seg_start[e + 1]; ++k) {
      uint32_t p = seg_pay[k];
      sum += piece[p];
      if (kpart) {
        ku += kpart[p];
        u += kpart[q6 + p];
      }
      fc = min(fc, (unsigned)slot_cut[p]);
    }
    if (kpart) sum = u > 0.0 ? sum * (ku / u) : 0.0;
    w[e] = sum;
    first_cut[e] = (uint8_t)fc;
  }
}

// *1 of conductivity fields 1..F-1 (field 0 comes from edge_reduce_kernel):
// the same fixed-order sums with k_f[t] u_T in place of k_0[t] u_T, so a
// field's *1 equals, bit for bit, what a single-field assembly with that k
// gives.
__global__ void edge_reduce_fields_kernel(const int32_t* __restrict__ seg_start,
                                          const uint32_t* __restrict__ seg_pay,
                                          const double* __restrict__ piece,
                                          const double* __restrict__ upart,
                                          const double* __restrict__ kf, int64_t m, int F,
                                          int64_t ne, double* __restrict__ w) {
  for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < ne;
       e += (int64_t)gridDim.x * blockDim.x) {
    double sum = 0.0, u = 0.0;
    const int32_t k0 = seg_start[e], k1 = seg_start[e + 1];
    for (int32_t k = k0; k < k1; ++k) {
      const uint32_t p = seg_pay[k];
      sum += piece[p];
      u += upart[p];
    }
    for (int f = 1; f < F; ++f) {
      const double* kk = kf + (int64_t)f * m;
      double ku = 0.0;
      for (int32_t k = k0; k < k1; ++k) {
        const uint32_t p = seg_pay[k];
        ku += __dmul_rn(kk[p / 6], upart[p]);   // the product kpart holds: no FMA
      }
      w[(int64_t)f * ne + e] = u > 0.0 ? sum * (ku / u) : 0.0;
    }
  }
}

// uniform grid of disc bounding boxes (radius scaled by the largest state)
__global__ void disc_bin_kernel(const double* __restrict__ discs, int nd,
                                double smax, DiscGrid g, int32_t* __restrict__ counts,
                                int32_t* __restrict__ cursor,
                                int32_t* __restrict__ items, int fill) {
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < nd;
       i += gridDim.x * blockDim.x) {
    const double* d = discs + 7 * (int64_t)i;
    const double R = d[6] * smax;
    int c0[3], c1[3];
    for (int k = 0; k < 3; ++k) {
      c0[k] = max(0, (int)floor((d[k] - R - g.lo[k]) * g.inv_cell));
      c1[k] = min(g.dim[k] - 1, (int)floor((d[k] + R - g.lo[k]) * g.inv_cell));
    }
    for (int z = c0[2]; z <= c1[2]; ++z)
      for (int y = c0[1]; y <= c1[1]; ++y)
        for (int x = c0[0]; x <= c1[0]; ++x) {
          int cell = x + g.dim[0] * (y + g.dim[1] * z);
          if (!fill) atomicAdd(&counts[cell], 1);
          else items[atomicAdd(&cursor[cell], 1)] = i;
        }
  }
}

__global__ void copy_i32_kernel(const int32_t* a, int32_t* b, int64_t n) {
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n;
       i += (int64_t)gridDim.x * blockDim.x)
    b[i] = a[i];
}

__global__ void validate_k_kernel(const double* __restrict__ k, int64_t m, int* errflag) {
  for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < m;
       t += (int64_t)gridDim.x * blockDim.x) {
    const double v = k[t];
    if (!(v > 0.0) || !isfinite(v)) atomicOr(errflag, 16);
  }
}

// conductivity must be finite and > 0 (checked on the device)
dec_status validate_k(dec_ctx* ctx, int64_t count) {
  cudaStream_t s = ctx->stream;
  DEC_TRY(cudaMemsetAsync(ctx->errflag.p, 0, sizeof(int), s));
  const unsigned g = (unsigned)std::max<int64_t>(
      1, std::min<int64_t>((count + 255) / 256, (int64_t)ctx->num_sms * 16));
  validate_k_kernel<<<g, 256, 0, s>>>(ctx->kcond.p, count, ctx->errflag.p);
  DEC_TRY(cudaGetLastError());
  ctx->launches += 1;
  int flag = 0;
  DEC_TRY(cudaMemcpyAsync(&flag, ctx->errflag.p, sizeof(int), cudaMemcpyDeviceToHost, s));
  DEC_TRY(cudaStreamSynchronize(s));
  if (flag & 16) return ctx->fail(DEC_ERR_ARG, "hodge_assemble: conductivity must be finite and > 0");
  return DEC_OK;
}

dec_status assemble_hodge(dec_ctx* ctx, int64_t nd, bool has_k, int n_fields) {
  cudaStream_t s = ctx->stream;
  const int64_t m = ctx->m, q = 6 * m;
  DEC_TRY(ctx->piece.ensure(has_k ? 3 * q : q));   // [piece | k u | u]
  DEC_TRY(ctx->slot_cut.ensure(q));
  DEC_TRY(ctx->w.ensure((size_t)n_fields * ctx->ne));
  DEC_TRY(ctx->first_cut.ensure(ctx->ne));
  DiscGrid g{};
  g.nd = (int)nd;
  g.n_states = ctx->n_scales;
  g.discs = ctx->discs.p;
  g.scales = ctx->scales.p;
  if (nd > 0) {
    // grid bounds from a host copy of the discs
    std::vector<double> hd(7 * nd), hs(ctx->n_scales);
    DEC_TRY(cudaMemcpyAsync(hd.data(), ctx->discs.p, sizeof(double) * 7 * nd,
                            cudaMemcpyDeviceToHost, s));
    DEC_TRY(cudaMemcpyAsync(hs.data(), ctx->scales.p, sizeof(double) * ctx->n_scales,
                            cudaMemcpyDeviceToHost, s));
    DEC_TRY(cudaStreamSynchronize(s));
    const double smax = hs.back();
    g.smax = smax;
    // FP32 disc records for the pre-test: centre and a bound on its largest
    // coordinate, normal and the reach smax * r (1 + 1e-9), bounds rounded up
    std::vector<float> hf(8 * nd);
    constexpr double kUp = 1.0 + 2.4e-7;     // 1 + 4 * 2^-24
    for (int64_t i = 0; i < nd; ++i) {
      const double* d = hd.data() + 7 * i;
      float* f = hf.data() + 8 * i;
      double amax = 0.0;
      for (int k = 0; k < 3; ++k) {
        f[k] = (float)d[k];
        f[4 + k] = (float)d[3 + k];
        amax = std::max(amax, std::fabs(d[k]));
      }
      f[3] = (float)(amax * kUp);
      f[7] = (float)(smax * d[6] * (1.0 + 1e-9) * kUp);
    }
    hf.insert(hf.end(), hs.begin(), hs.end());      // then the scales in FP32
    DEC_TRY(ctx->discs_f.ensure(hf.size()));
    DEC_TRY(cudaMemcpyAsync(ctx->discs_f.p, hf.data(), sizeof(float) * hf.size(),
                            cudaMemcpyHostToDevice, s));
    g.scales_f = ctx->discs_f.p + 8 * nd;
    // scale * r and its factors: no overflow, no underflow that matters beside
    // corners of at least 1e-9 (those of crack_points)
    g.fp32 = smax < 1e15;
    for (int64_t i = 0; i < nd && g.fp32; ++i) g.fp32 = hd[7 * i + 6] < 1e15;
    g.fp32 = g.fp32 && hs.front() > 1e-15;
    g.discs_f = reinterpret_cast<const float4*>(ctx->discs_f.p);
    double lo[3] = {0, 0, 0}, hi[3] = {1, 1, 1}, rmax = 0;
    for (int64_t i = 0; i < nd; ++i) {
      const double R = hd[7 * i + 6] * smax;
      rmax = std::max(rmax, R);
      for (int k = 0; k < 3; ++k) {
        lo[k] = std::min(lo[k], hd[7 * i + k] - R);
        hi[k] = std::max(hi[k], hd[7 * i + k] + R);
      }
    }
    double ext = std::max(hi[0] - lo[0], std::max(hi[1] - lo[1], hi[2] - lo[2]));
    // cells of twice the largest reach (half: 22 % slower on the cracked
    // cubes, a tet's box then spans more cells and meets discs again)
    double cell = std::max(2.0 * rmax, ext / 128.0);
    for (int k = 0; k < 3; ++k) {
      g.lo[k] = lo[k];
      g.dim[k] = std::max(1, (int)std::ceil((hi[k] - lo[k]) / cell));
    }
    g.inv_cell = 1.0 / cell;
    const int64_t cells = (int64_t)g.dim[0] * g.dim[1] * g.dim[2];
    DEC_TRY(ctx->grid_start.ensure(2 * (cells + 1)));
    int32_t* counts = ctx->grid_start.p;             // [cells+1] -> starts
    int32_t* cursor = ctx->grid_start.p + cells + 1;  // fill cursors
    DEC_TRY(cudaMemsetAsync(counts, 0, sizeof(int32_t) * (cells + 1), s));
    disc_bin_kernel<<<(unsigned)((nd + 127) / 128), 128, 0, s>>>(
        ctx->discs.p, (int)nd, smax, g, counts, cursor, nullptr, 0);
    DEC_TRY(cudaGetLastError());
    DEC_TRY(ctx->scan_tmp.ensure(scan_tmp_size(cells + 1)));
    DEC_TRY(exclusive_scan_u32((const uint32_t*)counts, (uint32_t*)counts, cells + 1,
                               ctx->scan_tmp.p, ctx->scan_tmp.cap, s));
    int32_t total = 0;
    DEC_TRY(cudaMemcpyAsync(&total, counts + cells, sizeof(int32_t),
                            cudaMemcpyDeviceToHost, s));
    DEC_TRY(cudaStreamSynchronize(s));
    DEC_TRY(ctx->grid_items.ensure(total > 0 ? total : 1));
    copy_i32_kernel<<<(unsigned)std::min<int64_t>((cells + 256) / 256, 4096), 256, 0, s>>>(
        counts, cursor, cells + 1);
    disc_bin_kernel<<<(unsigned)((nd + 127) / 128), 128, 0, s>>>(
        ctx->discs.p, (int)nd, smax, g, counts, cursor, ctx->grid_items.p, 1);
    DEC_TRY(cudaGetLastError());
    g.start = counts;
    g.items = ctx->grid_items.p;
    ctx->launches += 3 + scan_launches(cells + 1);  // count, cursor copy, fill
  }
  int64_t blocks = (m + kHodgeThreads - 1) / kHodgeThreads;
  if (blocks > (int64_t)ctx->num_sms * 64) blocks = (int64_t)ctx->num_sms * 64;
  DEC_TRY(ctx->geom_count.ensure(2));
  DEC_TRY(cudaMemsetAsync(ctx->geom_count.p, 0, 2 * sizeof(unsigned long long), s));
  if (nd > 0) DEC_TRY(ctx->key_a.ensure((m + 1) / 2));     // the list of thin tets
  uint32_t* thin = reinterpret_cast<uint32_t*>(ctx->key_a.p);
  auto* kern = ctx->geom_precision == DEC_GEOM_MIXED ? hodge_tet_kernel<true>
                                                     : hodge_tet_kernel<false>;
  kern<<<(unsigned)std::max<int64_t>(blocks, 1), kHodgeThreads, 0, s>>>(
      ctx->xyz.p, ctx->tets.p, has_k ? ctx->kcond.p : nullptr,
      m, ctx->piece.p, has_k ? ctx->piece.p + q : nullptr, ctx->slot_cut.p, g,
      ctx->geom_count.p, ctx->geom_count.p + 1, thin);
  DEC_TRY(cudaGetLastError());
  unsigned long long counts[2] = {0, 0};      // tets in FP64, thin tets
  DEC_TRY(cudaMemcpyAsync(counts, ctx->geom_count.p, sizeof(counts), cudaMemcpyDeviceToHost, s));
  DEC_TRY(cudaStreamSynchronize(s));
  ctx->geom_fp64_tets = (int64_t)counts[0];
  if (counts[1] > 0) {
    const int64_t tb = ((int64_t)counts[1] + kHodgeThreads - 1) / kHodgeThreads;
    crack_thin_kernel<<<(unsigned)std::min<int64_t>(tb, (int64_t)ctx->num_sms * 64), kHodgeThreads,
                        0, s>>>(ctx->xyz.p, ctx->tets.p, (int64_t)counts[1], thin,
                                ctx->slot_cut.p, g);
    DEC_TRY(cudaGetLastError());
    ctx->launches += 1;
  }
  int64_t eb = (ctx->ne + 255) / 256;
  if (eb > (int64_t)ctx->num_sms * 32) eb = (int64_t)ctx->num_sms * 32;
  edge_reduce_kernel<<<(unsigned)std::max<int64_t>(eb, 1), 256, 0, s>>>(
      ctx->seg_start.p, ctx->seg_pay.p, ctx->piece.p, has_k ? ctx->piece.p + q : nullptr, q,
      ctx->slot_cut.p, ctx->ne,
      ctx->w.p, ctx->first_cut.p);
  DEC_TRY(cudaGetLastError());
  ctx->launches += 2;
  if (n_fields > 1) {
    edge_reduce_fields_kernel<<<(unsigned)std::max<int64_t>(eb, 1), 256, 0, s>>>(
        ctx->seg_start.p, ctx->seg_pay.p, ctx->piece.p, ctx->piece.p + 2 * q, ctx->kcond.p, m,
        n_fields, ctx->ne, ctx->w.p);
    DEC_TRY(cudaGetLastError());
    ctx->launches += 1;
  }
  return DEC_OK;
}

}  // namespace dec

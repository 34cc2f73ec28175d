// dec_mesh.cu - mesh validation, the edge list of the tetrahedral complex
// (the rows of the incidence matrix d0, Sec. 2.1) and the CSR structure of
// L = d0^T *1 d0, all integer work with one result whatever the order in which
// threads run.
//
// The 6 edges of every tet are grouped by their smaller node (count, prefix
// sum, scatter: 3 atomics per tet and pass) and each node's group, about 40
// entries, is sorted by one warp on (larger node, tet slot).  That reads and
// writes every entry three times.  Sorting (64-bit key, payload) pairs of the
// whole mesh by radix took six passes of 32 bytes per entry; with the row
// structure built the same way, an upload of 2.05 M nodes (12.1 M tets) went
// from 14.6 to 4.7 ms.  Nodes of more than kWarpMax entries or lower
// neighbours (hubs) get a block each, in launches that other meshes do not
// make; the radix path stays for meshes with a node of more than kGroupMax.
#include "dec_internal.cuh"

#include <algorithm>

namespace dec {

__constant__ int kLocalEdge[6][2] = {{0, 1}, {0, 2}, {0, 3}, {1, 2}, {1, 3}, {2, 3}};

// ----------------------------------------------------------- validation
// errflag bit 1: node id out of range, bit 2: tet not positively oriented,
// bit 4: bad node tag; 32, 64: a node's edges or lower neighbours are too
// many for the grouped sorts; 128, 256: too many for a warp.

// FP32 value of a double, truncated by integer operations (conversions run on
// the narrow FP64 pipe); infinity stands for anything out of FP32's range.
__device__ __forceinline__ float trunc_f32(double v) {
  const unsigned hi = (unsigned)__double2hiint(v), lo = (unsigned)__double2loint(v);
  const unsigned e = hi & 0x7fffffffu;
  if (e >= (1151u << 20)) return INFINITY;
  if (e < (897u << 20)) return 0.0f;
  return __uint_as_float((hi & 0x80000000u) | ((e - (896u << 20)) << 3) | (lo >> 29));
}

// Whether the tet is positively oriented (volume > 0).  FP32 decides where it
// can: with S a bound on the coordinates and D on their differences, the
// truncated coordinates move each difference by at most 2^-22 S + 2^-24 D, so
// the determinant of the FP32 differences is off by less than
// 64 2^-22 S D^2 (18 D^2 times that shift, plus 24 2^-24 D^3 for its own
// roundings, D <= 2 S).  Underflow adds at most 1e-44 (1 + D), nothing beside
// a bound in the normal range (which D > 1e-18 with it).  The FP64 determinant
// (0.5 ms for 12 M tets: the FP64 pipe) decides the rest.
__device__ __forceinline__ bool tet_positive(const double* __restrict__ xyz, int4 v) {
  const double* p[4] = {xyz + 3 * (int64_t)v.x, xyz + 3 * (int64_t)v.y, xyz + 3 * (int64_t)v.z,
                        xyz + 3 * (int64_t)v.w};
  double c[4][3];
  float f[4][3], S = 0.0f, D = 0.0f;
#pragma unroll
  for (int i = 0; i < 4; ++i)
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      c[i][k] = p[i][k];
      f[i][k] = trunc_f32(c[i][k]);
      S = fmaxf(S, fabsf(f[i][k]));
    }
  float d[3][3];
#pragma unroll
  for (int i = 0; i < 3; ++i)
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      d[i][k] = f[i + 1][k] - f[0][k];
      D = fmaxf(D, fabsf(d[i][k]));
    }
  const float det = d[0][0] * (d[1][1] * d[2][2] - d[1][2] * d[2][1]) +
                    d[0][1] * (d[1][2] * d[2][0] - d[1][0] * d[2][2]) +
                    d[0][2] * (d[1][0] * d[2][1] - d[1][1] * d[2][0]);
  const float bound = 1.6e-5f * S * (D * D);
  if (S < 1e12f && S > 1e-12f && bound > 1.2e-38f && det > bound) return true;
  const double ax = c[1][0] - c[0][0], ay = c[1][1] - c[0][1], az = c[1][2] - c[0][2];
  const double bx = c[2][0] - c[0][0], by = c[2][1] - c[0][1], bz = c[2][2] - c[0][2];
  const double cx = c[3][0] - c[0][0], cy = c[3][1] - c[0][1], cz = c[3][2] - c[0][2];
  const double det64 = ax * (by * cz - bz * cy) + ay * (bz * cx - bx * cz) +
                       az * (bx * cy - by * cx);
  return det64 > 0.0;
}

__device__ __forceinline__ bool tet_in_range(int4 v, int64_t n) {
  return v.x >= 0 && v.y >= 0 && v.z >= 0 && v.w >= 0 && v.x < n && v.y < n && v.z < n && v.w < n;
}

// The tet's vertices in increasing order: id and local index (id << 2 | local)
__device__ __forceinline__ void sorted_vertices(int4 v, uint64_t (&g)[4]) {
  g[0] = (uint64_t)v.x << 2;
  g[1] = (uint64_t)v.y << 2 | 1u;
  g[2] = (uint64_t)v.z << 2 | 2u;
  g[3] = (uint64_t)v.w << 2 | 3u;
  auto order = [&](int i, int j) {
    const uint64_t a = min(g[i], g[j]), b = max(g[i], g[j]);
    g[i] = a;
    g[j] = b;
  };
  order(0, 1);
  order(2, 3);
  order(0, 2);
  order(1, 3);
  order(1, 2);
}

// Tets and tags checked; cnt[i] += number of edge entries whose smaller node
// is i (3, 2 and 1 for a tet's three smallest vertices).
__global__ void tet_count_kernel(const int32_t* __restrict__ tets,
                                 const double* __restrict__ xyz,
                                 const uint8_t* __restrict__ tag, int64_t m, int64_t n,
                                 uint32_t* __restrict__ cnt, int* errflag) {
  const int64_t t0 = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  const int64_t ts = (int64_t)gridDim.x * blockDim.x;
  for (int64_t i = t0; i < n; i += ts)
    if (tag[i] > 2) atomicOr(errflag, 4);
  for (int64_t t = t0; t < m; t += ts) {
    const int4 v = reinterpret_cast<const int4*>(tets)[t];
    if (!tet_in_range(v, n)) {
      atomicOr(errflag, 1);
      continue;
    }
    if (!tet_positive(xyz, v)) atomicOr(errflag, 2);
    uint64_t g[4];
    sorted_vertices(v, g);
    atomicAdd(cnt + (g[0] >> 2), 3u);
    atomicAdd(cnt + (g[1] >> 2), 2u);
    atomicAdd(cnt + (g[2] >> 2), 1u);
  }
}

// -------------------------------------------- edges grouped by smaller node
// Entries (or lower neighbours) of one node: what a block sorts in 128 KB of
// shared memory.  A mesh with a larger node is found out late, after 0.5 to 0.8
// of 7 ms at 5.9 M tets, and sorted by radix.
constexpr int kGroupMax = 16384;
// As many are ranked by one warp (lower neighbours: by eight lanes), in
// n^2 / 32 (n^2 / 8) steps; a block sorts more.  Uploads of 60 spheres of tets
// around a hub, ms with warps alone / with blocks / with radix sorts: hub of
// 252 entries .26 / - / .48, 486 .40 / .25 / .54, 1,014 1.0 / .30 / .57, 4,056
// 12.8 / .53 / .70; of 326 lower neighbours .40 / .25 / .65, 3,846 21.7 / .74 / 2.6.
constexpr int kWarpMax = 256;

// local edge slot of the local vertex pair {a, b}: (0,1) (0,2) (0,3) (1,2)
// (1,3) (2,3)
__device__ __forceinline__ unsigned edge_slot(unsigned a, unsigned b) {
  const unsigned lo = a < b ? a : b, hi = a < b ? b : a;
  return lo == 0 ? hi - 1 : lo == 1 ? hi + 1 : 5u;
}

// entries (larger node << 32 | tet * 6 + slot) of every edge, grouped by
// smaller node in any order; cur[i]: next free place of node i's group
__global__ void tet_scatter_kernel(const int32_t* __restrict__ tets, int64_t m, int64_t n,
                                   uint32_t* __restrict__ cur, uint64_t* __restrict__ out) {
  for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < m;
       t += (int64_t)gridDim.x * blockDim.x) {
    const int4 v = reinterpret_cast<const int4*>(tets)[t];
    if (!tet_in_range(v, n)) continue;      // reported by tet_count_kernel
    uint64_t g[4];
    sorted_vertices(v, g);
    const uint64_t t6 = (uint64_t)t * 6;
    uint32_t at[3];
#pragma unroll
    for (int i = 0; i < 3; ++i) at[i] = atomicAdd(cur + (g[i] >> 2), 3u - i);
#pragma unroll
    for (int i = 0; i < 3; ++i)
#pragma unroll
      for (int j = i + 1; j < 4; ++j)
        out[at[i] + (j - i - 1)] =
            (g[j] >> 2) << 32 | (t6 + edge_slot((unsigned)g[i] & 3u, (unsigned)g[j] & 3u));
  }
}

// One warp per node: its group sorted (in -> out; the rank of an entry is the
// number of smaller ones, all distinct) and its distinct larger nodes counted.
constexpr int kGroupSmem = 64;    // entries a warp sorts in shared memory
constexpr int kGroupWarps = 8;
__global__ void __launch_bounds__(32 * kGroupWarps)
group_sort_kernel(int64_t n, const uint32_t* __restrict__ beg, const uint64_t* __restrict__ in,
                  uint64_t* __restrict__ out, uint32_t* __restrict__ ucnt, int* errflag) {
  __shared__ __align__(16) uint64_t sh[kGroupWarps][2][kGroupSmem];
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  uint64_t* a = sh[wid][0];
  uint64_t* b = sh[wid][1];
  for (int64_t i = blockIdx.x * (int64_t)kGroupWarps + wid; i < n;
       i += (int64_t)gridDim.x * kGroupWarps) {
    const uint32_t b0 = beg[i];
    const int c = (int)(beg[i + 1] - b0);
    int heads = 0;
    if (c > kWarpMax) {
      if (lane == 0) atomicOr(errflag, c > kGroupMax ? 32 : 128);
    } else if (c <= kGroupSmem) {
      const uint64_t none = ~0ull;
      const uint64_t k0 = lane < c ? in[b0 + lane] : none;
      const uint64_t k1 = lane + 32 < c ? in[b0 + lane + 32] : none;
      a[lane] = k0;
      a[lane + 32] = k1;
      __syncwarp();
      int r0 = 0, r1 = 0;
      const ulonglong2* a2 = reinterpret_cast<const ulonglong2*>(a);
      for (int j = 0; 2 * j < c; ++j) {      // a padding key is above all others
        const ulonglong2 v = a2[j];
        r0 += (v.x < k0) + (v.y < k0);
        r1 += (v.x < k1) + (v.y < k1);
      }
      if (lane < c) b[r0] = k0;
      if (lane + 32 < c) b[r1] = k1;
      __syncwarp();
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const int e = lane + 32 * h;
        bool head = false;
        if (e < c) {
          const uint64_t k = b[e];
          out[b0 + e] = k;
          head = e == 0 || (b[e - 1] >> 32) != (k >> 32);
        }
        heads += __popc(__ballot_sync(0xffffffffu, head));
      }
      __syncwarp();
    } else {
      for (int e = lane; e < c; e += 32) {
        const uint64_t k = in[b0 + e];
        int r = 0;
        for (int j = 0; j < c; ++j) r += in[b0 + j] < k;
        out[b0 + r] = k;
      }
      __syncwarp();
      for (int e0 = 0; e0 < c; e0 += 32) {
        const int e = e0 + lane;
        const bool head = e < c && (e == 0 || (out[b0 + e - 1] >> 32) != (out[b0 + e] >> 32));
        heads += __popc(__ballot_sync(0xffffffffu, head));
      }
    }
    if (lane == 0) ucnt[i] = (uint32_t)heads;
  }
}

// Sort the c <= kGroupMax keys in `key` (bitonic network, all threads)
constexpr int kHubBlock = 1024;
__device__ __forceinline__ void block_sort(uint64_t* key, int c) {
  int P = 2;
  while (P < c) P <<= 1;
  for (int i = c + threadIdx.x; i < P; i += kHubBlock) key[i] = ~0ull;
  __syncthreads();
  for (int k = 2; k <= P; k <<= 1)
    for (int j = k >> 1; j > 0; j >>= 1) {
      for (int h = threadIdx.x; h < P / 2; h += kHubBlock) {
        const int a = 2 * h - (h & (j - 1)), b = a + j;
        const uint64_t x = key[a], y = key[b];
        if ((x > y) == ((a & k) == 0)) {
          key[a] = y;
          key[b] = x;
        }
      }
      __syncthreads();
    }
}

// body(node, size) by a whole block for every node of more than kWarpMax
// items (begin[i + 1] - begin[i]); 32 nodes are looked at a time
template <typename T, typename Body>
__device__ __forceinline__ void for_hubs(int64_t n, const T* __restrict__ begin, Body&& body) {
  __shared__ int size[32];
  for (int64_t i0 = blockIdx.x * (int64_t)32; i0 < n; i0 += gridDim.x * (int64_t)32) {
    __syncthreads();
    if (threadIdx.x < 32) {
      const int64_t i = i0 + threadIdx.x;
      const int c = i < n ? (int)(begin[i + 1] - begin[i]) : 0;
      size[threadIdx.x] = c > kWarpMax && c <= kGroupMax ? c : 0;
    }
    __syncthreads();
    for (int h = 0; h < 32; ++h)
      if (size[h]) body(i0 + h, size[h]);
  }
}

// group_sort_kernel's work for hubs
__global__ void __launch_bounds__(kHubBlock)
group_sort_hubs_kernel(int64_t n, const uint32_t* __restrict__ beg,
                       const uint64_t* __restrict__ in, uint64_t* __restrict__ out,
                       uint32_t* __restrict__ ucnt) {
  extern __shared__ uint64_t key[];
  for_hubs(n, beg, [&](int64_t i, int c) {
    const uint32_t b0 = beg[i];
    for (int e = threadIdx.x; e < c; e += kHubBlock) key[e] = in[b0 + e];
    block_sort(key, c);
    int heads = 0;
    for (int e0 = 0; e0 < c; e0 += kHubBlock) {
      const int e = e0 + threadIdx.x;
      if (e < c) out[b0 + e] = key[e];
      heads += __syncthreads_count(e < c && (e == 0 || (key[e - 1] >> 32) != (key[e] >> 32)));
    }
    if (threadIdx.x == 0) ucnt[i] = (uint32_t)heads;
    __syncthreads();
  });
}

// One warp per node: edge ids of its sorted entries (edges are numbered by
// (smaller, larger) node, so node i's start at up[i]), E, seg_start, seg_pay,
// t2e, and each edge's place among the lower neighbours of its larger node.
__global__ void __launch_bounds__(32 * kGroupWarps)
group_emit_kernel(int64_t n, const uint32_t* __restrict__ beg, const uint64_t* __restrict__ keys,
                  const int32_t* __restrict__ up, int32_t* __restrict__ E,
                  int32_t* __restrict__ seg_start, uint32_t* __restrict__ seg_pay,
                  int32_t* __restrict__ t2e, uint32_t* __restrict__ lo_cnt,
                  uint32_t* __restrict__ lo_place, int* errflag) {
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  for (int64_t i = blockIdx.x * (int64_t)kGroupWarps + wid; i < n;
       i += (int64_t)gridDim.x * kGroupWarps) {
    const uint32_t b0 = beg[i];
    const int c = (int)(beg[i + 1] - b0);
    int32_t e0 = up[i];
    uint32_t before = 0xffffffffu;      // larger node of the entry before the chunk
    for (int j0 = 0; j0 < c; j0 += 32) {
      const int j = j0 + lane;
      const bool ok = j < c;
      const uint64_t k = ok ? keys[b0 + j] : 0;
      const uint32_t hi = (uint32_t)(k >> 32), pay = (uint32_t)k;
      uint32_t prev = __shfl_up_sync(0xffffffffu, hi, 1);
      if (lane == 0) prev = before;
      const bool head = ok && (hi != prev);
      const unsigned mask = __ballot_sync(0xffffffffu, head);
      const int32_t e = e0 + __popc(mask & (0xffffffffu >> (31 - lane))) - 1;
      if (ok) {
        seg_pay[b0 + j] = pay;
        t2e[pay] = e;
      }
      if (head) {
        reinterpret_cast<int2*>(E)[e] = make_int2((int32_t)i, (int32_t)hi);
        seg_start[e] = (int32_t)(b0 + j);
        const uint32_t at = atomicAdd(lo_cnt + hi, 1u);
        lo_place[e] = at;
        if (at >= (uint32_t)kGroupMax) atomicOr(errflag, 64);
      }
      e0 += __popc(mask);
      before = __shfl_sync(0xffffffffu, hi, 31);
    }
    if (i == n - 1 && lane == 0) seg_start[e0] = (int32_t)beg[n];
  }
}

// lower neighbours' edges of every node, in any order
__global__ void lower_scatter_kernel(int64_t ne, const int32_t* __restrict__ E,
                                     const int32_t* __restrict__ lo_begin,
                                     const uint32_t* __restrict__ place,
                                     uint32_t* __restrict__ list) {
  for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < ne;
       e += (int64_t)gridDim.x * blockDim.x)
    list[lo_begin[E[2 * e + 1]] + place[e]] = (uint32_t)e;
}

// Row r of L: the lower neighbours (edges (j, r), j < r) in increasing j, the
// diagonal, then the upper neighbours.  Eight lanes per row; for a fixed r
// the edge id orders the lower neighbours, so an entry's rank is the number
// of smaller ids in its list.
__global__ void __launch_bounds__(256)
csr_rows_kernel(int64_t n, const int32_t* __restrict__ E, const int32_t* __restrict__ up,
                const int32_t* __restrict__ lo, const uint32_t* __restrict__ list,
                int32_t* __restrict__ rowptr, int32_t* __restrict__ col,
                int32_t* __restrict__ eid, int32_t* __restrict__ dpos,
                int32_t* __restrict__ pos_up, int* errflag) {
  if (*(volatile int*)errflag & 64) return;   // the radix path takes over
  const int lane = threadIdx.x & 7;
  for (int64_t r = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 3; r <= n;
       r += ((int64_t)gridDim.x * blockDim.x) >> 3) {
    const int32_t u0 = up[r], l0 = lo[r];
    const int32_t p0 = (int32_t)(u0 + l0 + r);
    if (lane == 0) rowptr[r] = p0;
    if (r == n) break;
    const int32_t nl = lo[r + 1] - l0, nu = up[r + 1] - u0;
    if (nl > kWarpMax && lane == 0) atomicOr(errflag, 256);    // csr_hub_rows_kernel
    for (int32_t k = lane; k < nl && nl <= kWarpMax; k += 8) {
      const uint32_t e = list[l0 + k];
      int32_t rank = 0;
      for (int32_t j = 0; j < nl; ++j) rank += list[l0 + j] < e;
      col[p0 + rank] = E[2 * (int64_t)e];
      eid[p0 + rank] = (int32_t)e;
    }
    const int32_t pd = p0 + nl;
    if (lane == 0) {
      dpos[r] = pd;
      col[pd] = (int32_t)r;
      eid[pd] = -1;
    }
    for (int32_t k = lane; k < nu; k += 8) {
      const int32_t e = u0 + k;
      col[pd + 1 + k] = E[2 * (int64_t)e + 1];
      eid[pd + 1 + k] = e;
      pos_up[e] = pd + 1 + k;
    }
  }
}

// The lower neighbours of hubs in csr_rows_kernel's rows
__global__ void __launch_bounds__(kHubBlock)
csr_hub_rows_kernel(int64_t n, const int32_t* __restrict__ E, const int32_t* __restrict__ lo,
                    const uint32_t* __restrict__ list, const int32_t* __restrict__ rowptr,
                    int32_t* __restrict__ col, int32_t* __restrict__ eid) {
  extern __shared__ uint64_t key[];
  for_hubs(n, lo, [&](int64_t r, int nl) {
    const int32_t l0 = lo[r], p0 = rowptr[r];
    for (int k = threadIdx.x; k < nl; k += kHubBlock) key[k] = list[l0 + k];
    block_sort(key, nl);
    for (int k = threadIdx.x; k < nl; k += kHubBlock) {
      const int32_t e = (int32_t)key[k];
      col[p0 + k] = E[2 * (int64_t)e];
      eid[p0 + k] = e;
    }
    __syncthreads();
  });
}

// ------------------------------------------------------------ edge list
// key of the directed-once edge (i, j), i < j: i * n + j; value: tet*6+slot.
__global__ void edge_keys_kernel(const int32_t* __restrict__ tets, int64_t m,
                                 int64_t n, uint64_t* __restrict__ keys,
                                 uint32_t* __restrict__ vals) {
  for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < m;
       t += (int64_t)gridDim.x * blockDim.x) {
    int4 v4 = reinterpret_cast<const int4*>(tets)[t];
    int v[4] = {v4.x, v4.y, v4.z, v4.w};
#pragma unroll
    for (int s = 0; s < 6; ++s) {
      uint64_t a = (uint64_t)v[kLocalEdge[s][0]], b = (uint64_t)v[kLocalEdge[s][1]];
      uint64_t lo = a < b ? a : b, hi = a < b ? b : a;
      keys[t * 6 + s] = lo * (uint64_t)n + hi;
      vals[t * 6 + s] = (uint32_t)(t * 6 + s);
    }
  }
}

__global__ void head_flags_kernel(const uint64_t* __restrict__ keys, int64_t q,
                                  uint32_t* __restrict__ flags) {
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < q;
       i += (int64_t)gridDim.x * blockDim.x)
    flags[i] = (i == 0 || keys[i] != keys[i - 1]) ? 1u : 0u;
}

// After the scan, excl[i] = number of heads before i, so the edge of item i
// is excl[i] + head(i) - 1.
__global__ void edge_emit_kernel(const uint64_t* __restrict__ keys,
                                 const uint32_t* __restrict__ vals,
                                 const uint32_t* __restrict__ excl, int64_t q,
                                 int64_t n, int32_t* __restrict__ E,
                                 int32_t* __restrict__ seg_start,
                                 int32_t* __restrict__ t2e) {
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < q;
       i += (int64_t)gridDim.x * blockDim.x) {
    uint64_t k = keys[i];
    bool head = (i == 0 || k != keys[i - 1]);
    int32_t e = (int32_t)excl[i] + (head ? 1 : 0) - 1;
    if (head) {
      E[2 * (int64_t)e] = (int32_t)(k / (uint64_t)n);
      E[2 * (int64_t)e + 1] = (int32_t)(k % (uint64_t)n);
      seg_start[e] = (int32_t)i;
    }
    t2e[vals[i]] = e;
    if (i == q - 1) seg_start[e + 1] = (int32_t)q;
  }
}

static int key_bits_for(int64_t n) {
  uint64_t maxkey = (uint64_t)n * (uint64_t)n;
  int bits = 1;
  while (bits < 64 && (maxkey >> bits) != 0) ++bits;
  return bits;
}

static unsigned grid_for(const dec_ctx* ctx, int64_t work, int threads) {
  int64_t g = (work + threads - 1) / threads;
  int64_t cap = (int64_t)ctx->num_sms * 32;
  if (g > cap) g = cap;
  if (g < 1) g = 1;
  return (unsigned)g;
}

dec_status build_edges(dec_ctx* ctx) {
  const int64_t q = 6 * ctx->m, n = ctx->n;
  cudaStream_t s = ctx->stream;
  DEC_TRY(ctx->key_a.ensure(q));
  DEC_TRY(ctx->key_b.ensure(q));
  DEC_TRY(ctx->val_a.ensure(q));
  DEC_TRY(ctx->val_b.ensure(q));
  DEC_TRY(ctx->flags.ensure(q));
  edge_keys_kernel<<<grid_for(ctx, ctx->m, 256), 256, 0, s>>>(
      ctx->tets.p, ctx->m, n, ctx->key_a.p, ctx->val_a.p);
  DEC_TRY(cudaGetLastError());
  ctx->launches += 3 + scan_launches(q);  // keys, heads, emit (the sort counts itself)
  bool alt = false;
  DEC_TRY_STATUS(radix_sort_pairs(ctx, ctx->key_a.p, ctx->val_a.p, ctx->key_b.p,
                                  ctx->val_b.p, q, key_bits_for(n), &alt));
  uint64_t* keys = alt ? ctx->key_b.p : ctx->key_a.p;
  uint32_t* vals = alt ? ctx->val_b.p : ctx->val_a.p;
  head_flags_kernel<<<grid_for(ctx, q, 256), 256, 0, s>>>(keys, q, ctx->flags.p);
  DEC_TRY(cudaGetLastError());
  DEC_TRY(ctx->scan_tmp.ensure(scan_tmp_size(q)));
  DEC_TRY(exclusive_scan_u32(ctx->flags.p, ctx->flags.p, q, ctx->scan_tmp.p,
                             ctx->scan_tmp.cap, s));
  // number of edges = excl[q-1] + head(q-1)
  uint32_t last_excl = 0;
  uint64_t last_keys[2] = {0, 0};
  DEC_TRY(cudaMemcpyAsync(&last_excl, ctx->flags.p + q - 1, sizeof(uint32_t),
                          cudaMemcpyDeviceToHost, s));
  DEC_TRY(cudaMemcpyAsync(last_keys, keys + (q >= 2 ? q - 2 : 0),
                          sizeof(uint64_t) * (q >= 2 ? 2 : 1),
                          cudaMemcpyDeviceToHost, s));
  DEC_TRY(cudaStreamSynchronize(s));
  bool last_head = q < 2 || last_keys[1] != last_keys[0];
  ctx->ne = (int64_t)last_excl + (last_head ? 1 : 0);
  DEC_TRY(ctx->E.ensure(2 * ctx->ne));
  DEC_TRY(ctx->seg_start.ensure(ctx->ne + 1));
  DEC_TRY(ctx->t2e.ensure(q));
  edge_emit_kernel<<<grid_for(ctx, q, 256), 256, 0, s>>>(
      keys, vals, ctx->flags.p, q, n, ctx->E.p, ctx->seg_start.p, ctx->t2e.p);
  DEC_TRY(cudaGetLastError());
  // keep the payloads grouped by edge (tet*6+slot, increasing in each group)
  if (alt) std::swap(ctx->seg_pay, ctx->val_b);
  else std::swap(ctx->seg_pay, ctx->val_a);
  return DEC_OK;
}

// ------------------------------------------------------- CSR structure
// Row r of L holds: the lower neighbours (edges (j, r), j < r) in increasing
// j, the diagonal, then the upper neighbours (edges (r, j)) in increasing j.
// The lower lists come from the edge list sorted by (max, min).
__global__ void transpose_keys_kernel(const int32_t* __restrict__ E, int64_t ne,
                                      int64_t n, uint64_t* __restrict__ keys,
                                      uint32_t* __restrict__ vals) {
  for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < ne;
       e += (int64_t)gridDim.x * blockDim.x) {
    int2 ij = reinterpret_cast<const int2*>(E)[e];
    keys[e] = (uint64_t)ij.y * (uint64_t)n + (uint64_t)ij.x;
    vals[e] = (uint32_t)e;
  }
}

__global__ void row_bounds_kernel(const int32_t* __restrict__ E,
                                  const uint64_t* __restrict__ tkeys, int64_t ne,
                                  int64_t n, int32_t* __restrict__ up_begin,
                                  int32_t* __restrict__ lo_begin,
                                  int32_t* __restrict__ rowptr) {
  for (int64_t r = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; r <= n;
       r += (int64_t)gridDim.x * blockDim.x) {
    // first edge with min >= r
    int64_t lo = 0, hi = ne;
    while (lo < hi) {
      int64_t mid = (lo + hi) >> 1;
      if (E[2 * mid] < r) lo = mid + 1; else hi = mid;
    }
    int64_t ub = lo;
    // first transposed edge with max >= r
    lo = 0; hi = ne;
    const uint64_t thr = (uint64_t)r * (uint64_t)n;
    while (lo < hi) {
      int64_t mid = (lo + hi) >> 1;
      if (tkeys[mid] < thr) lo = mid + 1; else hi = mid;
    }
    up_begin[r] = (int32_t)ub;
    lo_begin[r] = (int32_t)lo;
    rowptr[r] = (int32_t)(ub + lo + r);
  }
}

__global__ void csr_fill_kernel(const int32_t* __restrict__ E,
                                const uint64_t* __restrict__ tkeys,
                                const uint32_t* __restrict__ tvals, int64_t n,
                                const int32_t* __restrict__ up_begin,
                                const int32_t* __restrict__ lo_begin,
                                const int32_t* __restrict__ rowptr,
                                int32_t* __restrict__ col, int32_t* __restrict__ eid,
                                int32_t* __restrict__ dpos,
                                int32_t* __restrict__ pos_up) {
  for (int64_t r = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; r < n;
       r += (int64_t)gridDim.x * blockDim.x) {
    int32_t pos = rowptr[r];
    for (int32_t k = lo_begin[r]; k < lo_begin[r + 1]; ++k) {
      col[pos] = (int32_t)(tkeys[k] % (uint64_t)n);
      eid[pos] = (int32_t)tvals[k];
      ++pos;
    }
    dpos[r] = pos;
    col[pos] = (int32_t)r;
    eid[pos] = -1;
    ++pos;
    for (int32_t e = up_begin[r]; e < up_begin[r + 1]; ++e) {
      col[pos] = E[2 * (int64_t)e + 1];
      eid[pos] = e;
      pos_up[e] = pos;
      ++pos;
    }
  }
}

dec_status build_csr_structure(dec_ctx* ctx) {
  const int64_t ne = ctx->ne, n = ctx->n;
  cudaStream_t s = ctx->stream;
  ctx->nnz = 2 * ne + n;
  if (ctx->nnz >= ((int64_t)1 << 31) - 1)
    return ctx->fail(DEC_ERR_LIMIT, "nnz of L exceeds int32 indexing");
  DEC_TRY(ctx->key_a.ensure(ne));
  DEC_TRY(ctx->key_b.ensure(ne));
  DEC_TRY(ctx->val_a.ensure(ne));
  DEC_TRY(ctx->val_b.ensure(ne));
  transpose_keys_kernel<<<grid_for(ctx, ne, 256), 256, 0, s>>>(
      ctx->E.p, ne, n, ctx->key_a.p, ctx->val_a.p);
  DEC_TRY(cudaGetLastError());
  ctx->launches += 3;  // transpose keys, row bounds, fill
  bool alt = false;
  DEC_TRY_STATUS(radix_sort_pairs(ctx, ctx->key_a.p, ctx->val_a.p, ctx->key_b.p,
                                  ctx->val_b.p, ne, key_bits_for(n), &alt));
  const uint64_t* tk = alt ? ctx->key_b.p : ctx->key_a.p;
  const uint32_t* tv = alt ? ctx->val_b.p : ctx->val_a.p;
  DEC_TRY(ctx->up_begin.ensure(n + 1));
  DEC_TRY(ctx->lo_begin.ensure(n + 1));
  DEC_TRY(ctx->rowptr.ensure(n + 1));
  DEC_TRY(ctx->col.ensure(ctx->nnz));
  DEC_TRY(ctx->eid.ensure(ctx->nnz));
  DEC_TRY(ctx->dpos.ensure(n));
  DEC_TRY(ctx->pos_up.ensure(ne));
  row_bounds_kernel<<<grid_for(ctx, n + 1, 256), 256, 0, s>>>(
      ctx->E.p, tk, ne, n, ctx->up_begin.p, ctx->lo_begin.p, ctx->rowptr.p);
  DEC_TRY(cudaGetLastError());
  csr_fill_kernel<<<grid_for(ctx, n, 128), 128, 0, s>>>(
      ctx->E.p, tk, tv, n, ctx->up_begin.p, ctx->lo_begin.p, ctx->rowptr.p,
      ctx->col.p, ctx->eid.p, ctx->dpos.p, ctx->pos_up.p);
  DEC_TRY(cudaGetLastError());
  return DEC_OK;
}

static dec_status mesh_errors(dec_ctx* ctx, int flag) {
  if (flag & 1) return ctx->fail(DEC_ERR_MESH, "a tet references a node id out of range");
  if (flag & 2) return ctx->fail(DEC_ERR_MESH, "a tet is inverted or flat (orientation <= 0)");
  if (flag & 4) return ctx->fail(DEC_ERR_MESH, "a node tag is not 0, 1 or 2");
  return DEC_OK;
}

static unsigned hub_grid(const dec_ctx* ctx) {
  return (unsigned)std::max<int64_t>(1, std::min<int64_t>((ctx->n + 31) / 32, ctx->num_sms));
}

dec_status build_hub_rows(dec_ctx* ctx) {
  constexpr int smem = kGroupMax * sizeof(uint64_t);
  DEC_TRY(cudaFuncSetAttribute(csr_hub_rows_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                               smem));
  csr_hub_rows_kernel<<<hub_grid(ctx), kHubBlock, smem, ctx->stream>>>(
      ctx->n, ctx->E.p, ctx->lo_begin.p, ctx->val_b.p, ctx->rowptr.p, ctx->col.p, ctx->eid.p);
  DEC_TRY(cudaGetLastError());
  ctx->launches += 1;
  return DEC_OK;
}

// Mesh checks, edge list and CSR structure.  *radix is set when a node has
// more than kGroupMax edges or lower neighbours: the first is known here and
// nothing but the checks has been done, the second only once the caller reads
// errflag bit 64; build_edges and build_csr_structure then do the work.
dec_status build_mesh(dec_ctx* ctx, bool* radix) {
  const int64_t m = ctx->m, q = 6 * m, n = ctx->n;
  cudaStream_t s = ctx->stream;
  *radix = false;
  DEC_TRY(ctx->errflag.ensure(4));
  DEC_TRY(cudaMemsetAsync(ctx->errflag.p, 0, sizeof(int), s));
  DEC_TRY(ctx->key_a.ensure(q));
  DEC_TRY(ctx->key_b.ensure(q));
  DEC_TRY(ctx->hist.ensure(2 * (n + 1)));
  DEC_TRY(ctx->up_begin.ensure(n + 1));
  DEC_TRY(ctx->lo_begin.ensure(n + 1));
  DEC_TRY(ctx->scan_tmp.ensure(scan_tmp_size(n + 1)));
  uint32_t* beg = ctx->hist.p;                 // [n+1] group starts
  uint32_t* cur = ctx->hist.p + n + 1;         // [n] next free places
  uint32_t* up = (uint32_t*)ctx->up_begin.p;
  uint32_t* lo = (uint32_t*)ctx->lo_begin.p;
  DEC_TRY(cudaMemsetAsync(beg, 0, sizeof(uint32_t) * (n + 1), s));
  tet_count_kernel<<<grid_for(ctx, std::max(m, n), 256), 256, 0, s>>>(
      ctx->tets.p, ctx->xyz.p, ctx->tag.p, m, n, beg, ctx->errflag.p);
  DEC_TRY(cudaGetLastError());
  DEC_TRY(exclusive_scan_u32(beg, beg, n + 1, ctx->scan_tmp.p, ctx->scan_tmp.cap, s));
  DEC_TRY(cudaMemcpyAsync(cur, beg, sizeof(uint32_t) * n, cudaMemcpyDeviceToDevice, s));
  tet_scatter_kernel<<<grid_for(ctx, m, 256), 256, 0, s>>>(ctx->tets.p, m, n, cur, ctx->key_a.p);
  const unsigned gn = (unsigned)std::max<int64_t>(
      1, std::min<int64_t>((n + kGroupWarps - 1) / kGroupWarps, (int64_t)ctx->num_sms * 32));
  group_sort_kernel<<<gn, 32 * kGroupWarps, 0, s>>>(n, beg, ctx->key_a.p, ctx->key_b.p, up,
                                                    ctx->errflag.p);
  DEC_TRY(cudaGetLastError());
  DEC_TRY(cudaMemsetAsync(up + n, 0, sizeof(uint32_t), s));
  DEC_TRY(exclusive_scan_u32(up, up, n + 1, ctx->scan_tmp.p, ctx->scan_tmp.cap, s));
  ctx->launches += 3 + 2 * scan_launches(n + 1);
  int flag = 0;
  uint32_t ne = 0;
  DEC_TRY(cudaMemcpyAsync(&flag, ctx->errflag.p, sizeof(int), cudaMemcpyDeviceToHost, s));
  DEC_TRY(cudaMemcpyAsync(&ne, up + n, sizeof(uint32_t), cudaMemcpyDeviceToHost, s));
  DEC_TRY(cudaStreamSynchronize(s));
  DEC_TRY_STATUS(mesh_errors(ctx, flag));
  if (flag & 32) {
    *radix = true;
    return DEC_OK;
  }
  if (flag & 128) {      // hubs: counted again with the others, whose counts are summed by now
    group_sort_kernel<<<gn, 32 * kGroupWarps, 0, s>>>(n, beg, ctx->key_a.p, ctx->key_b.p, up,
                                                      ctx->errflag.p);
    constexpr int smem = kGroupMax * sizeof(uint64_t);
    DEC_TRY(cudaFuncSetAttribute(group_sort_hubs_kernel,
                                 cudaFuncAttributeMaxDynamicSharedMemorySize, smem));
    group_sort_hubs_kernel<<<hub_grid(ctx), kHubBlock, smem, s>>>(n, beg, ctx->key_a.p,
                                                                  ctx->key_b.p, up);
    DEC_TRY(cudaGetLastError());
    DEC_TRY(cudaMemsetAsync(up + n, 0, sizeof(uint32_t), s));
    DEC_TRY(exclusive_scan_u32(up, up, n + 1, ctx->scan_tmp.p, ctx->scan_tmp.cap, s));
    DEC_TRY(cudaMemcpyAsync(&ne, up + n, sizeof(uint32_t), cudaMemcpyDeviceToHost, s));
    DEC_TRY(cudaStreamSynchronize(s));
    ctx->launches += 2 + scan_launches(n + 1);
  }
  ctx->ne = ne;
  ctx->nnz = 2 * ctx->ne + n;
  if (ctx->nnz >= ((int64_t)1 << 31) - 1)
    return ctx->fail(DEC_ERR_LIMIT, "nnz of L exceeds int32 indexing");
  DEC_TRY(ctx->E.ensure(2 * ctx->ne));
  DEC_TRY(ctx->seg_start.ensure(ctx->ne + 1));
  DEC_TRY(ctx->seg_pay.ensure(q));
  DEC_TRY(ctx->t2e.ensure(q));
  DEC_TRY(ctx->val_a.ensure(ctx->ne));
  DEC_TRY(ctx->val_b.ensure(ctx->ne));
  DEC_TRY(ctx->rowptr.ensure(n + 1));
  DEC_TRY(ctx->col.ensure(ctx->nnz));
  DEC_TRY(ctx->eid.ensure(ctx->nnz));
  DEC_TRY(ctx->dpos.ensure(n));
  DEC_TRY(ctx->pos_up.ensure(ctx->ne));
  DEC_TRY(cudaMemsetAsync(lo, 0, sizeof(uint32_t) * (n + 1), s));
  group_emit_kernel<<<gn, 32 * kGroupWarps, 0, s>>>(
      n, beg, ctx->key_b.p, ctx->up_begin.p, ctx->E.p, ctx->seg_start.p, ctx->seg_pay.p,
      ctx->t2e.p, lo, ctx->val_a.p, ctx->errflag.p);
  DEC_TRY(cudaGetLastError());
  DEC_TRY(exclusive_scan_u32(lo, lo, n + 1, ctx->scan_tmp.p, ctx->scan_tmp.cap, s));
  lower_scatter_kernel<<<grid_for(ctx, ctx->ne, 256), 256, 0, s>>>(
      ctx->ne, ctx->E.p, ctx->lo_begin.p, ctx->val_a.p, ctx->val_b.p);
  csr_rows_kernel<<<grid_for(ctx, 8 * (n + 1), 256), 256, 0, s>>>(
      n, ctx->E.p, ctx->up_begin.p, ctx->lo_begin.p, ctx->val_b.p, ctx->rowptr.p, ctx->col.p,
      ctx->eid.p, ctx->dpos.p, ctx->pos_up.p, ctx->errflag.p);
  DEC_TRY(cudaGetLastError());
  ctx->launches += 3 + scan_launches(n + 1);
  return DEC_OK;
}

}  // namespace dec

// BVH construction over the primitives' bounding ellipsoids (Sec. 4.1, Eq. 4)
// and the per-primitive precompute of Eq. 1-2.
//
// Steps, all on the caller's stream:
//   1. k_prim_bounds   per primitive: rotation from the quaternion, bounding box of
//                      the k-ellipsoid, block-reduced centroid bounds
//   2. k_morton        30-bit Morton code of each box centre
//   3. radix sort      (ugp_sort.cu, on the caller's workspace) of (code, index), stable
//   4. k_tree          binary radix tree over the sorted codes and its boxes, from the leaves up
//   5. k_records       64-byte hot records in leaf order (W = S^-1 R^T, mu, g0, index) and
//                      the low float parts of W (48 B, read only by ill-conditioned hits)
//   6. k_collapse4     the 4-wide quantised tree: each binary internal node with up to four
//                      descendants, largest opened first (layout in ugp_internal.cuh)

#include <math.h>
#include <string.h>

#include "ugp_internal.cuh"
#include "ugp_split.cuh"

namespace ugp {
namespace {


struct Layout {
  size_t prims, nodes, nodes4, wlo, persistent;
  size_t aabb, keys0, keys1, vals0, vals1, flags, bounds, sort, total;
};

__device__ __forceinline__ int f2o(float f) {
  const int i = __float_as_int(f);
  return i >= 0 ? i : i ^ 0x7fffffff;
}
__device__ __forceinline__ float o2f(int i) { return __int_as_float(i >= 0 ? i : i ^ 0x7fffffff); }

// Rotation matrix (row-major) of the normalised quaternion (w, x, y, z).
__device__ __forceinline__ void quat_rot(float4 q, float R[9]) {
  const float inv = rsqrtf(q.x * q.x + q.y * q.y + q.z * q.z + q.w * q.w);
  const float w = q.x * inv, x = q.y * inv, y = q.z * inv, z = q.w * inv;
  R[0] = 1.f - 2.f * (y * y + z * z); R[1] = 2.f * (x * y - w * z);       R[2] = 2.f * (x * z + w * y);
  R[3] = 2.f * (x * y + w * z);       R[4] = 1.f - 2.f * (x * x + z * z); R[5] = 2.f * (y * z - w * x);
  R[6] = 2.f * (x * z - w * y);       R[7] = 2.f * (y * z + w * x);       R[8] = 1.f - 2.f * (x * x + y * y);
}

__device__ __forceinline__ bool prim_valid(float3 m, float4 q, float3 s, float c) {
  const float qn = q.x * q.x + q.y * q.y + q.z * q.z + q.w * q.w;
  return isfinite(m.x) && isfinite(m.y) && isfinite(m.z) && isfinite(qn) && qn > 1e-20f &&
         isfinite(s.x) && isfinite(s.y) && isfinite(s.z) && s.x > 0.f && s.y > 0.f && s.z > 0.f &&
         isfinite(c) && c >= 0.f;
}

__device__ __forceinline__ float3 ld3(const float* p, int64_t i) {
  return make_float3(p[3 * i], p[3 * i + 1], p[3 * i + 2]);
}
__device__ __forceinline__ float4 ld4(const float* p, int64_t i) {
  return make_float4(p[4 * i], p[4 * i + 1], p[4 * i + 2], p[4 * i + 3]);
}

// Bounding box of the k-ellipsoid x = mu + k R S v, |v| = 1: half extent along axis i is
// k * sqrt(sum_j (R_ij s_j)^2).  Widened by a few float32 ulps so the box stays
// conservative for the float32 interval test.
//
// The bounds of the means are reduced per thread, then per block, over a grid of resident blocks: one
// atomic per bound and block. One per warp of primitives (172,000 of them at 5.5M, on six
// addresses) took 0.68 ms, against 0.08 for the arrays themselves.
constexpr int kBoundsBlocks = 152 * 8;
__global__ void __launch_bounds__(256) k_prim_bounds(int64_t n, const float* __restrict__ mean3,
                                                     const float* __restrict__ quat4, const float* __restrict__ scale3,
                                                     const float* __restrict__ mag, float k, float4* __restrict__ aabb,
                                                     int* __restrict__ bounds,
                                                     unsigned long long* __restrict__ n_invalid) {
  __shared__ int red[6][8];
  const float big = 3.0e38f;
  float v[6] = {big, big, big, big, big, big};  // min of the means and of their negatives
  unsigned bad = 0u;
  for (int64_t i = int64_t(blockIdx.x) * blockDim.x + threadIdx.x; i < n; i += int64_t(gridDim.x) * blockDim.x) {
    const float3 m = ld3(mean3, i);
    const float4 q = ld4(quat4, i);
    const float3 s = ld3(scale3, i);
    const float c = mag[i];
    if (prim_valid(m, q, s, c)) {
      float R[9];
      quat_rot(q, R);
      float e[3];
      const float mm[3] = {m.x, m.y, m.z};
      for (int r = 0; r < 3; ++r) {
        const float a = R[3 * r] * s.x, b = R[3 * r + 1] * s.y, d = R[3 * r + 2] * s.z;
        e[r] = k * sqrtf(a * a + b * b + d * d) * (1.f + 4e-6f) + 2e-7f * fabsf(mm[r]);
      }
      aabb[2 * i] = make_float4(m.x - e[0], m.y - e[1], m.z - e[2], 0.f);
      aabb[2 * i + 1] = make_float4(m.x + e[0], m.y + e[1], m.z + e[2], 0.f);
      for (int r = 0; r < 3; ++r) {
        v[r] = fminf(v[r], mm[r]);
        v[3 + r] = fminf(v[3 + r], -mm[r]);
      }
    } else {
      // An invalid primitive keeps a point box; its record is flagged and never hit.
      const float x = isfinite(m.x) ? m.x : 0.f, y = isfinite(m.y) ? m.y : 0.f,
                  z = isfinite(m.z) ? m.z : 0.f;
      aabb[2 * i] = make_float4(x, y, z, 0.f);
      aabb[2 * i + 1] = make_float4(x, y, z, 0.f);
      ++bad;
    }
  }
  if (bad) atomicAdd(n_invalid, (unsigned long long)bad);
  for (int a = 0; a < 6; ++a) {
    const int r = __reduce_min_sync(0xffffffffu, f2o(v[a]));
    if ((threadIdx.x & 31) == 0) red[a][threadIdx.x >> 5] = r;
  }
  __syncthreads();
  if (threadIdx.x < 6) {
    int r = red[threadIdx.x][0];
    for (int w = 1; w < 8; ++w) r = min(r, red[threadIdx.x][w]);
    atomicMin(&bounds[threadIdx.x], r);
  }
}

__device__ __forceinline__ uint32_t expand10(uint32_t v) {
  v = (v * 0x00010001u) & 0xFF0000FFu;
  v = (v * 0x00000101u) & 0x0F00F00Fu;
  v = (v * 0x00000011u) & 0xC30C30C3u;
  v = (v * 0x00000005u) & 0x49249249u;
  return v;
}

__global__ void k_morton(int64_t n, const float4* __restrict__ aabb, const int* __restrict__ bounds,
                         uint32_t* __restrict__ keys, int32_t* __restrict__ vals) {
  const int64_t i = int64_t(blockIdx.x) * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const float lo[3] = {o2f(bounds[0]), o2f(bounds[1]), o2f(bounds[2])};
  const float hi[3] = {-o2f(bounds[3]), -o2f(bounds[4]), -o2f(bounds[5])};
  const float4 a = aabb[2 * i], b = aabb[2 * i + 1];
  const float c[3] = {0.5f * (a.x + b.x), 0.5f * (a.y + b.y), 0.5f * (a.z + b.z)};
  uint32_t code = 0;
  for (int ax = 0; ax < 3; ++ax) {
    const float ext = hi[ax] - lo[ax];
    float t = ext > 0.f ? (c[ax] - lo[ax]) / ext : 0.5f;
    t = fminf(fmaxf(t * 1024.f, 0.f), 1023.f);
    code |= expand10(uint32_t(t)) << (2 - ax);
  }
  keys[i] = code;
  vals[i] = int32_t(i);
}

__global__ void k_single_root(int4* nodes) {
  nodes[3] = make_int4(~0, kEmptyChild, 0, 0);
}

// Hot record of the primitive in leaf slot `slot` (layout in ugp_internal.cuh), plus the
// low-order float parts of W for the double-float refinement of ill-conditioned hits.  W = hi + lo
// is formed by sums of three floats (ugp_split.cuh), to 0.5 2^-48 of the row's 1 / s.  In FP64 the
// kernel took 1.54 ms of a 3.9 ms build of 5.5M primitives, bound by the FP64 pipe.
__global__ void k_records(int64_t n, const int32_t* __restrict__ order, const float* __restrict__ mean3,
                          const float* __restrict__ quat4, const float* __restrict__ scale3,
                          const float* __restrict__ mag, float4* __restrict__ recs,
                          float4* __restrict__ wlo) {
  const int64_t slot = int64_t(blockIdx.x) * blockDim.x + threadIdx.x;
  if (slot >= n) return;
  const int64_t i = order[slot];
  const float3 m = ld3(mean3, i);
  const float4 q = ld4(quat4, i);
  const float3 s = ld3(scale3, i);
  const float c = mag[i];
  float4 r0, r1, r2, r3, l0, l1, l2;
  if (prim_valid(m, q, s, c)) {
    const float sv[3] = {s.x, s.y, s.z};
    float hi[9], lo[9], g0;
    split::whitening(q.x, q.y, q.z, q.w, sv, c, hi, lo, g0);
    r0 = make_float4(hi[0], hi[1], hi[2], m.x);
    r1 = make_float4(hi[3], hi[4], hi[5], m.y);
    r2 = make_float4(hi[6], hi[7], hi[8], m.z);
    l0 = make_float4(lo[0], lo[1], lo[2], 0.f);
    l1 = make_float4(lo[3], lo[4], lo[5], 0.f);
    l2 = make_float4(lo[6], lo[7], lo[8], 0.f);
    r3 = make_float4(g0, __int_as_float(int(i)), 1.f, 0.f);
  } else {
    r0 = r1 = r2 = l0 = l1 = l2 = make_float4(0.f, 0.f, 0.f, 0.f);
    r3 = make_float4(0.f, __int_as_float(int(i)), 0.f, 0.f);
  }
  recs[4 * slot + 0] = r0;
  recs[4 * slot + 1] = r1;
  recs[4 * slot + 2] = r2;
  recs[4 * slot + 3] = r3;
  wlo[3 * slot + 0] = l0;
  wlo[3 * slot + 1] = l1;
  wlo[3 * slot + 2] = l2;
}

// Binary radix tree over the sorted codes (Karras, HPG 2012) and its boxes. Node i has leaf i at one end of its
// leaves, node 0 is the root. A block takes 256 leaves and the nodes of the same numbers.
//   * A node whose leaves all lie in the block (its prefix is not shared by the leaf before the block or by the
//     one behind it) finds its ends and its split by bisection, and its children's boxes from two windows
//     of 2^k leaves each, which the block doubles in shared memory level by level: no node waits for another.
//   * The others (about 1 in 25) are reached from below: the largest subtrees that lie in a block climb. Where two
//     siblings meet both leave their box and far end for the split; the first to arrive stops, and the
//     second, which knows the parent's leaves by then, writes it and goes on (Apetrei, CGVC 2014).
// 5.5M primitives: nodes by one kernel 0.14 ms, boxes by climbing from every leaf with an atomic per node
// 0.46, both by climbing with meetings in shared memory 0.52 (most lanes of a warp have stopped while one
// climbs), now 0.28 and 0.07 for the climbers. Windows of all levels at once (47 KB) leave four blocks per SM,
// windows of one level at a time cost twice the loads from shared memory: 0.36 and 0.32 in place of 0.28.
constexpr int kTreeBlock = 256;
constexpr unsigned kClimbBlocks = 8 * 152;

// Where siblings of different blocks meet, and the subtrees that start from k_tree's blocks.
struct Climb {
  float4* meet;  // by split: the left child's box and first leaf, the right child's box and last leaf
  int *flags;    // by split: children that have arrived
  int *first, *last, *count;
};
// Length of the common prefix of the codes a, b of leaves p, q (equal codes: of their positions).
__device__ __forceinline__ int prefix(uint32_t a, uint32_t b, int p, int q) {
  return a == b ? 32 + __clz(uint32_t(p) ^ uint32_t(q)) : __clz(a ^ b);
}
__device__ __forceinline__ float united(int a, float x, float y) { return a < 3 ? fminf(x, y) : fmaxf(x, y); }
__device__ __forceinline__ void leave_box(float4* meet, int split, int side, const float (&b)[6], int far) {
  float4* m = meet + 4 * size_t(split) + 2 * side;
  m[0] = make_float4(b[0], b[1], b[2], b[3]);
  m[1] = make_float4(b[4], b[5], __int_as_float(far), 0.f);
}
// Node `id` over the leaves first .. last, its left child up to leaf `split`, with the children's boxes u and v.
__device__ __forceinline__ void write_node(float4* nodes, int id, int first, int split, int last,
                                           const float (&u)[6], const float (&v)[6]) {
  float4* node = nodes + 4 * size_t(id);
  node[0] = make_float4(u[0], u[1], u[2], u[3]);
  node[1] = make_float4(u[4], u[5], v[0], v[1]);
  node[2] = make_float4(v[2], v[3], v[4], v[5]);
  reinterpret_cast<int4*>(node)[3] =
      make_int4(first == split ? ~split : split, last == split + 1 ? ~(split + 1) : split + 1, 0, 0);
}

__global__ void __launch_bounds__(kTreeBlock) k_tree(int n, const uint32_t* __restrict__ keys,
                                                     const int32_t* __restrict__ order,
                                                     const float4* __restrict__ aabb, float4* __restrict__ nodes,
                                                     float* __restrict__ root_box, Climb C) {
  __shared__ uint32_t key[kTreeBlock + 2];  // of the leaves base - 1 .. base + kTreeBlock
  __shared__ float win[4][6][kTreeBlock];   // boxes of the 2^k leaves from each on, four levels k; later the climbers
  __shared__ int climbers, out;
  const int tid = threadIdx.x, base = int(blockIdx.x) * kTreeBlock, end = min(base + kTreeBlock, n), i = base + tid;
  for (int t = tid; t < kTreeBlock + 2; t += kTreeBlock) {
    const int j = base - 1 + t;
    key[t] = j >= 0 && j < n ? keys[j] : 0u;
  }
  if (tid == 0) climbers = 0;
  float leaf[6] = {INFINITY, INFINITY, INFINITY, -INFINITY, -INFINITY, -INFINITY};
  if (i < n) {
    const int p = order[i];
    const float4 lo = aabb[2 * p], hi = aabb[2 * p + 1];
    leaf[0] = lo.x; leaf[1] = lo.y; leaf[2] = lo.z; leaf[3] = hi.x; leaf[4] = hi.y; leaf[5] = hi.z;
  }
  for (int a = 0; a < 6; ++a) win[0][a][tid] = leaf[a];
  __syncthreads();
  auto delta = [&](int p, int q) {  // base - 1 <= p, q <= end; -1 outside of the scene
    return p < 0 || q < 0 || p >= n || q >= n ? -1 : prefix(key[p - base + 1], key[q - base + 1], p, q);
  };
  int l = 0, r = 0, g = 0;
  bool inside = false;
  if (i < n - 1) {
    const int dn = delta(i, i + 1), dp = delta(i, i - 1), d = dn > dp ? 1 : -1, dmin = min(dn, dp);
    inside = !(delta(i, d > 0 ? end : base - 1) > dmin);
    if (inside) {
      // longer common prefix of (code, position) than `bits`: their difference is below 2^(63 - bits)
      const uint32_t mine = key[tid + 1];
      auto longer = [&](int q, unsigned long long limit) {
        return ((unsigned long long)(mine ^ key[q - base + 1]) << 32 | uint32_t(i ^ q)) < limit;
      };
      const unsigned long long far = dmin < 0 ? ~0ull : 1ull << (63 - dmin);
      int len = 0, s = 0;
      for (int t = kTreeBlock / 2; t > 0; t >>= 1) {
        const int q = i + (len + t) * d;
        if (q >= base && q < end && longer(q, far)) len += t;
      }
      const int j = i + len * d;
      const unsigned long long near = 1ull << (63 - delta(i, j));
      for (int t = kTreeBlock / 2; t > 0; t >>= 1)
        if (s + t <= len && longer(i + (s + t) * d, near)) s += t;
      g = i + s * d + min(d, 0);
      l = min(i, j);
      r = max(i, j);
    }
  }
  // a child's box from the windows of its size: at its first leaf and up to its last
  float x[6], y[6], w[6];
  for (int a = 0; a < 6; ++a) w[a] = leaf[a];
  const int kl = inside ? 31 - __clz(g - l + 1) : -1, kr = inside ? 31 - __clz(r - g) : -1;
  for (int k0 = 0; k0 < 8; k0 += 4) {
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      if (k0 + k > 0) {
        const int from = min(tid + (1 << (k0 + k - 1)), kTreeBlock - 1);
        for (int a = 0; a < 6; ++a) w[a] = united(a, w[a], win[(k + 3) & 3][a][from]);
        if (k == 0) __syncthreads();
        for (int a = 0; a < 6; ++a) win[k][a][tid] = w[a];
        __syncthreads();
      }
    }
    if (kl >= k0 && kl < k0 + 4)
      for (int a = 0; a < 6; ++a)
        x[a] = united(a, win[kl & 3][a][l - base], win[kl & 3][a][g - base + 1 - (1 << kl)]);
    if (kr >= k0 && kr < k0 + 4)
      for (int a = 0; a < 6; ++a)
        y[a] = united(a, win[kr & 3][a][g + 1 - base], win[kr & 3][a][r - base + 1 - (1 << kr)]);
    __syncthreads();
  }
  // a subtree climbs when its parent does not lie in the block
  int(*own)[2] = reinterpret_cast<int(*)[2]>(&win[0][0][0]);
  auto climbs = [&](int first, int last, const float (&u)[6]) {
    const int dp = max(delta(first - 1, first), delta(last, last + 1));
    if (delta(base - 1, first) < dp && delta(last, end) < dp) return;
    const int side = delta(last, last + 1) == dp ? 0 : 1;
    leave_box(C.meet, side ? first - 1 : last, side, u, side ? last : first);
    int* c = own[atomicAdd(&climbers, 1)];  // disjoint subtrees of the block: at most 256
    c[0] = first;
    c[1] = last;
  };
  if (inside) {
    write_node(nodes, i, l, g, r, x, y);
    for (int a = 0; a < 6; ++a) x[a] = united(a, x[a], y[a]);
    if (l == 0 && r == n - 1)
      for (int a = 0; a < 6; ++a) root_box[a] = x[a];
    else
      climbs(l, r, x);
  }
  if (i < n) climbs(i, i, leaf);
  __syncthreads();
  if (tid == 0) out = atomicAdd(C.count, climbers);
  __syncthreads();
  if (tid < climbers) {
    C.first[out + tid] = own[tid][0];
    C.last[out + tid] = own[tid][1];
  }
}

// The climbers, each by a thread. (In k_tree they kept their blocks for the two to four rounds of loads and
// atomics that most climb, five times as long as the rest of the block's work: 0.48 ms in all.)
__global__ void __launch_bounds__(kTreeBlock) k_climb(int n, const uint32_t* __restrict__ keys,
                                                      float4* __restrict__ nodes, float* __restrict__ root_box,
                                                      Climb C) {
  const int count = *C.count;
  auto delta = [&](int p, int q) { return p < 0 || q >= n ? -1 : prefix(keys[p], keys[q], p, q); };
  for (int e = int(blockIdx.x) * kTreeBlock + threadIdx.x; e < count; e += int(gridDim.x) * kTreeBlock) {
    int l = C.first[e], r = C.last[e];
    int dl = delta(l - 1, l), dr = delta(r, r + 1);
    float b[6];
    bool left = true;  // the box for the parent is there
    while (dl >= 0 || dr >= 0) {
      const int side = dr > dl ? 0 : 1;  // left child or right
      const int split = side ? l - 1 : r;
      const float4* m = C.meet + 4 * size_t(split);
      if (!left) leave_box(C.meet, split, side, b, side ? r : l);
      // one acquire-release atomic in place of two full fences (boxes of 5.5M primitives: 0.82 -> 0.47 ms)
      int seen;
      asm volatile("atom.acq_rel.gpu.global.add.s32 %0, [%1], 1;" : "=r"(seen) : "l"(C.flags + split) : "memory");
      if (seen == 0) break;
      if (left) {
        const float4 o0 = __ldcg(m + 2 * side), o1 = __ldcg(m + 2 * side + 1);
        b[0] = o0.x; b[1] = o0.y; b[2] = o0.z; b[3] = o0.w; b[4] = o1.x; b[5] = o1.y;
        left = false;
      }
      const float4 o0 = __ldcg(m + 2 - 2 * side), o1 = __ldcg(m + 3 - 2 * side);
      const float c[6] = {o0.x, o0.y, o0.z, o0.w, o1.x, o1.y};
      if (side) l = __float_as_int(o1.z);
      else r = __float_as_int(o1.z);
      dl = delta(l - 1, l);
      dr = delta(r, r + 1);
      const int id = dl < 0 && dr < 0 ? 0 : (dr > dl ? r : l);  // a left child is node r, a right child node l
      if (side) write_node(nodes, id, l, split, r, c, b);
      else write_node(nodes, id, l, split, r, b, c);
      for (int a = 0; a < 6; ++a) b[a] = united(a, b[a], c[a]);
    }
    if (dl < 0 && dr < 0)
      for (int a = 0; a < 6; ++a) root_box[a] = b[a];
  }
}

// One 4-wide node per binary internal node: its children, of which the internal one with the largest
// surface is replaced by its own two until there are four, the other child before a grandchild of the same size
// (equal boxes, as of primitives in one place, then give a tree of half the depth). (Every binary node gets one, as any of them
// may be a child. With two fixed levels a child that is a leaf left a slot empty, and depths had to be
// found first by eight launches: rebuilding 5.5M primitives took 2.47 ms against 2.15, light-sample
// rays in a 1M-primitive room 2.94 ms per million against 2.75, free flights 7.04 against 6.94.) Boxes are quantised outwards to
// 8 bits per face against a grid of spacing 2^e_a per axis anchored at the union's low corner.
__global__ void __launch_bounds__(256) k_collapse4(int n_int, const float4* __restrict__ nodes,
                                                   uint4* __restrict__ nodes4) {
  const int i = int(blockIdx.x) * blockDim.x + threadIdx.x;
  if (i >= n_int) return;
  float box[4][6];
  int ref[4];
  float area[4];  // of the internal children, -1 for leaves
  auto set = [&](int c, float x0, float y0, float z0, float x1, float y1, float z1, int r) {
    box[c][0] = x0; box[c][1] = y0; box[c][2] = z0; box[c][3] = x1; box[c][4] = y1; box[c][5] = z1;
    ref[c] = r;
    const float dx = x1 - x0, dy = y1 - y0, dz = z1 - z0;
    area[c] = r >= 0 ? dx * dy + dy * dz + dz * dx : -1.f;
  };
  auto open = [&](int node, int c0, int c1) {
    const float4* nd = nodes + 4 * size_t(node);
    const float4 n0 = nd[0], n1 = nd[1], n2 = nd[2];
    const int4 n3 = reinterpret_cast<const int4*>(nd)[3];
    set(c0, n0.x, n0.y, n0.z, n0.w, n1.x, n1.y, n3.x);
    set(c1, n1.z, n1.w, n2.x, n2.y, n2.z, n2.w, n3.y);
  };
  open(i, 0, 1);
  int m = ref[1] == kEmptyChild ? 1 : 2;  // one only for the root of a one-primitive tree
  if (m == 2) {
    if (area[0] >= 0.f || area[1] >= 0.f) {
      const bool left = area[0] >= area[1];
      if (left) open(ref[0], 0, 2);
      else open(ref[1], 1, 2);
      m = 3;
      const float big = fmaxf(area[0], fmaxf(area[1], area[2]));
      if (big >= 0.f) {
        const int c = (left ? area[1] : area[0]) == big ? (left ? 1 : 0) : (area[2] == big ? 2 : (left ? 0 : 1));
        if (c == 0) open(ref[0], 0, 3);
        else if (c == 1) open(ref[1], 1, 3);
        else open(ref[2], 2, 3);
        m = 4;
      }
    }
  }
  float lo[3] = {3.0e38f, 3.0e38f, 3.0e38f}, hi[3] = {-3.0e38f, -3.0e38f, -3.0e38f};
#pragma unroll
  for (int c = 0; c < 4; ++c)
    if (c < m)
      for (int a = 0; a < 3; ++a) {
        lo[a] = fminf(lo[a], box[c][a]);
        hi[a] = fmaxf(hi[a], box[c][3 + a]);
      }
  uint32_t qlo[3] = {0u, 0u, 0u}, qhi[3] = {0u, 0u, 0u}, ex = 0u;
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    // a power-of-two spacing 2^e >= extent / 254 (frexp: extent / 254 = f 2^e, f in [1/2, 1));
    // the spare step absorbs the margins and the rounding of o + q 2^e
    const float ext = hi[a] - lo[a];
    int e = -126;
    if (ext > 0.f) {
      frexpf(ext * (1.f / 254.f) * (1.f + 1e-6f), &e);
      e = max(-126, min(e, 126));
    }
    const float sp = ldexpf(1.f, e), isp = ldexpf(1.f, -e);
    // the faces keep a margin of 2^-7 grid steps to the boxes (the rounding of the node test); the
    // grid starts 2^-5 steps below the union so that its lowest face has one as well
    constexpr float kMargin = 0.0078125f;
    lo[a] -= 4.f * kMargin * sp;
#pragma unroll
    for (int c = 0; c < 4; ++c) {
      if (c >= m) continue;
      int ql = int(floorf((box[c][a] - lo[a]) * isp - kMargin));
      int qh = int(ceilf((box[c][3 + a] - lo[a]) * isp + kMargin));
      ql = max(0, min(ql, 255));
      qh = max(0, min(qh, 255));
      while (ql > 0 && fmaf(float(ql), sp, lo[a]) > box[c][a]) --ql;
      while (qh < 255 && fmaf(float(qh), sp, lo[a]) < box[c][3 + a]) ++qh;
      qlo[a] |= uint32_t(ql) << (8 * c);
      qhi[a] |= uint32_t(qh) << (8 * c);
    }
    // an empty child slot gets an inverted box (low face 255, high face 0), which a ray enters only where the
    // whole node is below the node test's slack
#pragma unroll
    for (int c = 1; c < 4; ++c)
      if (c >= m) qlo[a] |= 255u << (8 * c);
    ex |= uint32_t(e + 128) << (8 * a);
  }
  int r4[4];
#pragma unroll
  for (int c = 0; c < 4; ++c) r4[c] = c < m ? ref[c] : kEmptyChild;
  uint4* q = nodes4 + 4 * size_t(i);
  q[0] = make_uint4(__float_as_uint(lo[0]), __float_as_uint(lo[1]), __float_as_uint(lo[2]), ex);
  q[1] = make_uint4(qlo[0], qlo[1], qlo[2], qhi[0]);
  q[2] = make_uint4(qhi[1], qhi[2], 0u, 0u);
  q[3] = make_uint4(uint32_t(r4[0]), uint32_t(r4[1]), uint32_t(r4[2]), uint32_t(r4[3]));
}

__global__ void k_init_bounds(int* bounds) {
  if (threadIdx.x < 6) bounds[threadIdx.x] = f2o(3.0e38f);
}

// For n == 1 the single child needs its box too; the empty child gets a box nobody reaches.
__global__ void k_single_refit(const float4* __restrict__ aabb, float* nodes_f, float* root_box) {
  const float4 lo = aabb[0], hi = aabb[1];
  const float b[6] = {lo.x, lo.y, lo.z, hi.x, hi.y, hi.z};
  for (int k = 0; k < 6; ++k) { nodes_f[k] = b[k]; nodes_f[6 + k] = 0.f; root_box[k] = b[k]; }
}

bool layout_for(int64_t n, Layout* L) {
  const size_t N = size_t(n);
  const size_t ni = N > 1 ? N - 1 : 1;
  size_t off = 0;
  L->prims = off;      off = align256(off + N * 64);
  L->nodes = off;      off = align256(off + ni * 64);
  L->nodes4 = off;     off = align256(off + ni * 64);
  L->wlo = off;        off = align256(off + N * 48);
  L->bounds = off;     off = align256(off + 64);   // 6 ordered-int bounds, root box, invalid count
  L->persistent = off;
  L->aabb = off;       off = align256(off + N * 32);
  L->keys0 = off;      off = align256(off + N * 4);
  L->keys1 = off;      off = align256(off + N * 4);
  L->vals0 = off;      off = align256(off + N * 4);
  L->vals1 = off;      off = align256(off + N * 4);
  L->flags = off;      off = align256(off + ni * 4);
  L->sort = off;       off = align256(off + radix_sort_workspace(int64_t(N)));
  L->total = off;
  return true;
}

}  // namespace
}  // namespace ugp

using namespace ugp;

extern "C" size_t ugp_build_bvh_workspace_size(int64_t n_prims) {
  if (n_prims < 0 || n_prims > (int64_t(1) << 30)) return 0;
  Layout L;
  if (!layout_for(n_prims, &L)) return 0;
  return L.total;
}

extern "C" ugp_status ugp_build_bvh(const ugp_prims* prims, float cutoff_eps, void* workspace,
                                    size_t workspace_bytes, void* stream_, ugp_bvh** out) {
  clear_error();
  if (!prims || !out) return fail(UGP_ERR_INVALID_ARG, "ugp_build_bvh: prims and out must be non-NULL");
  *out = nullptr;
  const int64_t n = prims->n;
  if (n < 0 || n > (int64_t(1) << 30))
    return fail(UGP_ERR_INVALID_ARG, "ugp_build_bvh: n_prims %lld out of range [0, 2^30]", (long long)n);
  if (!(cutoff_eps > 0.f && cutoff_eps < 1.f))
    return fail(UGP_ERR_INVALID_ARG, "ugp_build_bvh: cutoff_eps %g not in (0, 1)", double(cutoff_eps));
  if (n > 0 && (!prims->mean3 || !prims->quat4 || !prims->scale3 || !prims->magnitude))
    return fail(UGP_ERR_INVALID_ARG, "ugp_build_bvh: NULL primitive array");
  if (n > 0 && !workspace) return fail(UGP_ERR_INVALID_ARG, "ugp_build_bvh: NULL workspace");
  if (reinterpret_cast<uintptr_t>(workspace) & 255)
    return fail(UGP_ERR_INVALID_ARG, "ugp_build_bvh: workspace must be 256-byte aligned");
  Layout L;
  if (!layout_for(n, &L)) return fail(UGP_ERR_CUDA, "ugp_build_bvh: sort workspace query failed");
  if (workspace_bytes < L.total)
    return fail(UGP_ERR_WORKSPACE_TOO_SMALL, "ugp_build_bvh: need %zu bytes, got %zu", L.total,
                workspace_bytes);
  cudaStream_t st = static_cast<cudaStream_t>(stream_);
  const double kd = sqrt(-2.0 * log(double(cutoff_eps)));

  ugp_bvh* b = new ugp_bvh();
  b->magic = kBvhMagic;
  UGP_CUDA_CHECK(cudaGetDevice(&b->device));
  b->n_prims = n;
  b->n_nodes = n > 1 ? n - 1 : (n == 1 ? 1 : 0);
  b->k = float(kd);
  b->k2 = float(kd * kd);
  char* ws = static_cast<char*>(workspace);
  b->prims = reinterpret_cast<const float4*>(ws + L.prims);
  b->wlo = reinterpret_cast<const float4*>(ws + L.wlo);
  b->nodes = reinterpret_cast<const float4*>(ws + L.nodes);
  b->nodes4 = reinterpret_cast<const uint4*>(ws + L.nodes4);
  b->persistent_bytes = L.persistent;
  b->bounds_dev = reinterpret_cast<const float*>(ws + L.bounds);
  if (n == 0) {
    *out = b;
    return UGP_OK;
  }
  float4* aabb = reinterpret_cast<float4*>(ws + L.aabb);
  int* bounds = reinterpret_cast<int*>(ws + L.bounds);
  float* root_box = reinterpret_cast<float*>(ws + L.bounds + 32);
  unsigned long long* n_invalid = reinterpret_cast<unsigned long long*>(ws + L.bounds + 56);
  uint32_t* k0 = reinterpret_cast<uint32_t*>(ws + L.keys0);
  uint32_t* k1 = reinterpret_cast<uint32_t*>(ws + L.keys1);
  int32_t* v0 = reinterpret_cast<int32_t*>(ws + L.vals0);
  int32_t* v1 = reinterpret_cast<int32_t*>(ws + L.vals1);
  int* flags = reinterpret_cast<int*>(ws + L.flags);

  const int T = 256;
  const unsigned G = unsigned((n + T - 1) / T);
  prof_begin(kStBuild, st);
  UGP_CUDA_CHECK(cudaMemsetAsync(ws + L.bounds, 0, 64, st));
  k_init_bounds<<<1, 32, 0, st>>>(bounds);
  k_prim_bounds<<<G < unsigned(kBoundsBlocks) ? G : unsigned(kBoundsBlocks), T, 0, st>>>(n, prims->mean3, prims->quat4, prims->scale3, prims->magnitude, b->k,
                                 aabb, bounds, n_invalid);
  UGP_CUDA_CHECK(cudaGetLastError());
  int4* nodes_i = reinterpret_cast<int4*>(ws + L.nodes);
  float* nodes_f = reinterpret_cast<float*>(ws + L.nodes);
  int32_t* order = v0;
  if (n == 1) {
    UGP_CUDA_CHECK(cudaMemsetAsync(v0, 0, 4, st));
    k_single_root<<<1, 1, 0, st>>>(nodes_i);
    k_single_refit<<<1, 1, 0, st>>>(aabb, nodes_f, root_box);
  } else {
    k_morton<<<G, T, 0, st>>>(n, aabb, bounds, k0, v0);
    UGP_CUDA_CHECK(cudaGetLastError());
    const ugp_status ss = radix_sort_pairs(k0, k1, v0, v1, n, 30, ws + L.sort, st);
    if (ss != UGP_OK) return ss;
    const bool in1 = (radix_sort_passes(30) & 1) != 0;
    order = in1 ? v1 : v0;
    UGP_CUDA_CHECK(cudaMemsetAsync(flags, 0, (n - 1) * 4, st));
    // the splits' boxes lie where the 4-wide nodes come to be
    const Climb climb{reinterpret_cast<float4*>(ws + L.nodes4), flags, reinterpret_cast<int*>(in1 ? k0 : k1),
                      in1 ? v0 : v1, bounds + 6};
    const uint32_t* keys = in1 ? k1 : k0;
    const unsigned tree_blocks = unsigned((n + kTreeBlock - 1) / kTreeBlock);
    float4* nodes = reinterpret_cast<float4*>(ws + L.nodes);
    k_tree<<<tree_blocks, kTreeBlock, 0, st>>>(int(n), keys, order, aabb, nodes, root_box, climb);
    UGP_CUDA_CHECK(cudaGetLastError());
    k_climb<<<tree_blocks < kClimbBlocks ? tree_blocks : kClimbBlocks, kTreeBlock, 0, st>>>(int(n), keys, nodes,
                                                                                         root_box, climb);
    UGP_CUDA_CHECK(cudaGetLastError());
  }
  k_records<<<G, T, 0, st>>>(n, order, prims->mean3, prims->quat4, prims->scale3, prims->magnitude,
                             reinterpret_cast<float4*>(ws + L.prims), reinterpret_cast<float4*>(ws + L.wlo));
  UGP_CUDA_CHECK(cudaGetLastError());
  {
    const int n_int = int(b->n_nodes);
    k_collapse4<<<unsigned((n_int + T - 1) / T), T, 0, st>>>(n_int, reinterpret_cast<const float4*>(ws + L.nodes),
                                                            reinterpret_cast<uint4*>(ws + L.nodes4));
    UGP_CUDA_CHECK(cudaGetLastError());
  }
  // own kernels, the radix sort's three per 8-bit digit of the 30-bit codes among them
  prof_end(kStBuild, st, (n == 1 ? 5 : 6 + 3 * radix_sort_passes(30)) + 1);
  b->stream = st;
  *out = b;
  return UGP_OK;
}

extern "C" void ugp_bvh_release(ugp_bvh* bvh) {
  if (bvh && bvh->magic == kBvhMagic) {
    bvh->magic = 0;
    delete bvh;
  }
}

extern "C" ugp_status ugp_bvh_get_info(const ugp_bvh* bvh, ugp_bvh_info* out) {
  clear_error();
  if (!valid_bvh(bvh)) return fail(UGP_ERR_NOT_BUILT, "ugp_bvh_get_info: invalid handle");
  if (!out) return fail(UGP_ERR_INVALID_ARG, "ugp_bvh_get_info: NULL out");
  out->n_prims = bvh->n_prims;
  out->n_nodes = bvh->n_nodes;
  out->cutoff_k = bvh->k;
  out->persistent_bytes = bvh->persistent_bytes;
  out->n_invalid = 0;
  for (int k = 0; k < 3; ++k) { out->bounds_lo[k] = 0.f; out->bounds_hi[k] = 0.f; }
  if (bvh->n_prims > 0) {
    float hb[16];
    UGP_CUDA_CHECK(cudaStreamSynchronize(bvh->stream));
    UGP_CUDA_CHECK(cudaMemcpy(hb, bvh->bounds_dev, 64, cudaMemcpyDeviceToHost));
    for (int k = 0; k < 3; ++k) { out->bounds_lo[k] = hb[8 + k]; out->bounds_hi[k] = hb[11 + k]; }
    unsigned long long inv;
    memcpy(&inv, reinterpret_cast<const char*>(hb) + 56, 8);
    out->n_invalid = int64_t(inv);
  }
  return UGP_OK;
}

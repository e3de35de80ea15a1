// Launch interface of the tracing kernels (shared by the C entry points and the renderer).
#pragma once

#include "ugp_internal.cuh"

namespace ugp {

constexpr int kTrBlock = 128;      // transmittance: threads per block
constexpr int kTrStack = 48;       // transmittance: rows of shared memory for stack and held-back primitives
constexpr int kTrBlocksPerSM = 8;  // transmittance: resident blocks per SM (24 KB shared, <= 64 registers)
constexpr int kFFBlock = 128;      // free flight: threads per block of the scan
constexpr int kFFStack = 36;       // free flight: rows of the traversal stack in shared memory
constexpr int kFFShort = 26;       // the same where six blocks of the scan share an SM
constexpr int kFFBlocksPerSM = 6;  // free flight: resident scan blocks per SM (37 KB shared, <= 80 registers)
constexpr int kFFBlocksWide = 5;   // the same for scans with more state (groups, a scene per ray; 42 KB, <= 102)
// Entries that a traversal of the 4-wide tree can need at most. A step down a path is at least one level of the binary
// tree over 30-bit codes and, for equal codes, 30-bit positions (60 levels), and leaves up to three children on the
// stack. Rooms need 28; scenes whose sizes span decades around one place need 40 to 80. What lies
// above the rows in shared memory is kept in local memory, which only rays that get there touch.
constexpr int kStackMax = 3 * 60;
constexpr int kB = 32;             // free flight: bins of the scan
constexpr int kTrWarps = 152 * kTrBlocksPerSM * kTrBlock / 32;  // warps of the transmittance a GB300 holds

// Rays a warp takes when n of them are spread over `warps` resident warps (1 to 32). A launch with
// fewer rays than the GPU has lanes is bound by the longest chain of steps in a warp, and a step
// takes the longer the more rays share it, while idle lanes still take the leaf steps' primitives:
// so the scan, the renderer's shadow rays and the radiance field spread theirs over all resident warps, down to one
// each (transmittance queries of few rays go in groups of lanes instead, below). Scan and transmittance of 2,048
// rays through 1,000 primitives: 396 us at 32 rays per warp (most warps idle), 275 at 16 or more, 227 at
// 8, 199 at 4, 189 at 2, 184 at 1; a 128 x 128 render of that scene, 4 spp at depth 4: 4.63 ms -> 2.37.
__host__ __device__ constexpr int rays_per_warp(int64_t n, int64_t warps) {
  const int64_t r = (n + warps - 1) / warps;
  return r >= 32 ? 32 : (r < 1 ? 1 : int(r));
}

struct TraceScene {
  const float4* nodes;   // binary nodes
  const uint4* nodes4;   // 4-wide quantised nodes (ugp_internal.cuh)
  const float4* prims;
  const float4* wlo;
  int64_t n_prims;
  int64_t n_nodes;
  float k2;
};

// Launches of few rays give each ray a group of lanes (tr_walk): log2 of its size for n rays, 0 for
// a lane each. Light-sample rays of a 1M-primitive room, us, by lanes per ray:
//   rays      1     2     4     8    16    32
//     2K    169   152    88    56    39    31
//     8K    225   174    98    66    57    63
//    16K    269   190   115    80    89   105
//    30K    347   213   167   143   151   186
//    60K    406   279   242   233   262   342
//   120K    493   468   425   434   505   667
//   250K    848   830   793   849  1009  1368
//   500K   1494  1527  1515  1647  1987  2717
constexpr int kTrFew = 72 * kTrWarps;
__host__ __device__ constexpr int tr_group(int64_t n) {
  return n <= kTrWarps ? 5 : (2 * n <= 5 * kTrWarps ? 4 : (n <= 16 * kTrWarps ? 3 : (n <= kTrFew ? 2 : 0)));
}
// Whether n rays of a scene of n_prims go in groups: in a scene of few primitives the chains are short, and a group's
// lanes find nothing to do. Transmittances, us, in groups and a lane each: 16 primitives and 150,000 rays 41 and 19,
// 64 and 150,000 55 and 41, 128 and 150,000 76 and 66, 300 and 300,000 234 and 200; 64 and 20,000 17 and 22 (64 and 40,000
// 29 and 22), 128 and 40,000 28 and 40.
inline bool tr_few(int64_t n, int64_t n_prims) { return n <= kTrFew && n <= 600 * n_prims; }
// Blocks of a launch of up to n <= kTrFew rays in groups.
inline int tr_few_grid(int64_t n) {
  int64_t t = n << tr_group(n);  // lanes; a smaller count may take more of them
  for (const int64_t b : {int64_t(kTrWarps), int64_t(5) * kTrWarps / 2, int64_t(16) * kTrWarps})
    if (b < n && b << tr_group(b) > t) t = b << tr_group(b);
  return int((t + kTrBlock - 1) / kTrBlock);
}

// The same for the scan of free flights (kFFWarps resident warps on a GB300). Camera and bounce rays of a
// 1M-primitive room, us for scan and finish, by lanes per ray:
//   rays      1     4     8    16    32
//     2K    454   231   179   159   149
//     8K    624   351   296   266   262
//    16K    805   479   396   378   397
//    30K   1012   605   539   534   585
//    60K   1152   816   798   853   973
//   120K   1499  1272  1339  1477  1740
//   250K   2266  2310  2532  2858  3428
constexpr int kFFWarps = 152 * kFFBlocksWide * kFFBlock / 32;
constexpr int kFFFew = 60 * kFFWarps;
__host__ __device__ constexpr int ff_group(int64_t n) {
  return n <= 3 * kFFWarps ? 5 : (n <= 10 * kFFWarps ? 4 : (n <= 25 * kFFWarps ? 3 : (n <= kFFFew ? 2 : 0)));
}
// As tr_few; free flights, us: 16 primitives and 40,000 rays 73 and 47, 64 and 150,000 189 and 116, 128 and 80,000
// 143 and 116, 300 and 150,000 342 and 254; 64 and 10,000 50 and 81, 300 and 80,000 205 and 232.
inline bool ff_few(int64_t n, int64_t n_prims) { return n <= kFFFew && n <= 12000 + 250 * n_prims; }

// Blocks of a transmittance launch of up to n rays.
inline int tr_grid(int64_t n) {
  const int64_t full = (n + kTrBlock - 1) / kTrBlock;
  const int64_t spread = (n + kTrBlock / 32 - 1) / (kTrBlock / 32);  // one ray per warp
  const int64_t held = kTrWarps / (kTrBlock / 32);
  return int(full > held ? full : (spread < held ? spread : held));
}

TraceScene trace_scene(const ugp_bvh* b);

ugp_status check_rays(const char* fn, const ugp_bvh* bvh, int64_t n, const void* o3, const void* d3,
                      const void* t0, const void* t1);

ugp_status launch_transmittance(const TraceScene& sc, int64_t n, const float* o3, const float* d3,
                                const float* t0, const float* t1, const int32_t* excl, float* T,
                                uint8_t* st, cudaStream_t stream);

// The workspace holds the finish's queue for n rays (dense_queue_bytes(n, slots)) and, with
// `with_lists`, the slot lists after it; slots < 0 takes the default number of interval slots.
ugp_status launch_free_flight(const TraceScene& sc, int64_t n, const float* o3, const float* d3,
                              const float* t0, const float* t1, const float* u, const float* u2,
                              const int32_t* excl, int32_t* prim, float* tu, float* tsp, uint8_t* st,
                              void* workspace, bool with_lists, cudaStream_t stream, int64_t slots = -1);

}  // namespace ugp

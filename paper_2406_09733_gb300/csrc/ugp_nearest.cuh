// Nearest codebook entry of every point on the tensor cores (tcgen05.mma, TMEM accumulators), with
// exactly the result of the FP32 scan: the entry with the smallest
//     d2 = fma chain over d of (x_d - c_d)^2,
// ties to the lower index.
//
// Comparing a point with all 4096 entries is a contraction: s = |c|^2 / 2 - x.c orders the entries as
// d2 does. The matrix product gives s with a bounded error, which leaves a few candidates per point,
// and those are compared by d2 in FP32. Scanning all entries by d2 takes 2 D + 3 instructions per
// point and entry (1M points: 1.2 ms at D = 3, 5.0 at D = 16, of the FP32 pipes' rate); here it is one
// minimum per accumulator.
//   * Points and entries are moved by a common centre and cut into BF16 pieces (x = h + m + l, 24
//     bits; |m| <= 2^-8 |x|, |l| <= 2^-17 |x|). A row of A holds pieces of x and three ones, a row of B the
//     pieces of -c that they meet and those of |c|^2 / 2: with 6 products per dimension (hh hm mh mm hl lh) what is
//     left out is at most 2^-24 of |x||c|, with 3 (hh hm mh; D = 16) 2^-15.
//   * A block takes 256 points, as two M = 128 tiles, against 32 tiles of 128 entries that one warp brings
//     in by bulk copies (ring of 4). A warp for each point tile issues its products, into two accumulator
//     buffers, and two threads per point (four warpgroups) read 64 of its 128 accumulators per tile each.
//     They keep the minimum of every granule of 32 or 64 entries in shared memory, and a bit for every
//     unit of 16 or 32 that is within the error bound of the smallest accumulator so far.
//   * Units with that bit whose granule is within the bound of the point's smallest at the end are scanned
//     by d2. The entries are ordered along a space-filling curve, so that candidates share units, and
//     entries equal to one of lower index, which cannot win, are left out of the product (a plane of
//     splats has one normal and one size: hundreds of the starting entries are equal).
// The steps over the tiles are bound by their latency and by what one thread can issue, not by a rate. With
// one thread per point, one warp for copies and products, bits taken from all minima at the end and scalar
// loads of the candidates, a search of 1M points took 1.12, 0.83, 0.79 and 1.11 ms (D = 3, 4, 6, 16); now
// 0.58, 0.51, 0.50 and 0.71, about 60% of it the steps.
// A point whose values or bound are not finite, or a block whose wait ran out, scans every entry.
#pragma once
#include <cuda_bf16.h>
#include <math.h>

#include "ugp_internal.cuh"
#include "ugp_umma.cuh"

namespace ugp {
namespace nearest {

using namespace umma;

constexpr int kEntries = 4096;
constexpr int kTileN = 128;                  // entries per product
constexpr int kTiles = kEntries / kTileN;
constexpr int kPoints = 256;                 // points per block
constexpr int kRing = 4;                     // entry tiles in shared memory
constexpr int kShare = 2;                    // threads per point
constexpr int kWork = kPoints * kShare;      // threads that read accumulators
constexpr int kThreads = kWork + 96;
constexpr uint64_t kWaitNs = 2000000000ull;  // 2 s per wait
constexpr float kDead = 1.7014118e38f;       // score of an entry left out (2^127)

// Products per dimension, K (a multiple of 16), entries per granule and the relative error bound of s
// (against |x||c| + |c|^2 / 2): the products left out, an addition at 2^-22 for each of the others, the rounding of
// the moved coordinates and of |c|^2 / 2. That makes 0.66 2^-16 at D = 6 and 1.41 2^-15 at D = 16. A bound of
// 2^-15 there, too small, took 25.29 ms for the codebook of 1M points, 1.5 2^-15 takes 25.37, 2^-14 25.47.
template <int D>
struct Cfg {
  static constexpr int kTerms = D <= 6 ? 6 : 3;
  static constexpr int K = (D * kTerms + 3 + 15) / 16 * 16;
  static constexpr int kGran = D <= 6 ? 32 : 64;
  static constexpr int kGrans = kEntries / kGran;
  static constexpr int kLanes = D == 3 ? 2 : 4;  // lanes that compare a point with its candidates
  // Entries per candidate bit. Finer bits cost the steps 5%, which the scan repays where an entry is long
  // (D = 16: 0.77 -> 0.71 ms) or where many entries are nearly equal (D = 3, sizes of a wall: 0.63 -> 0.58).
  static constexpr int kUnit = D == 4 || D == 6 ? 32 : 16;
  static constexpr int kQuads = D / 4 + 1;  // float4 of an entry and its index
  static constexpr float kErr = D <= 6 ? 1.52587890625e-05f : 4.57763671875e-05f;  // 2^-16, 1.5 2^-15
  static_assert(K <= (D <= 6 ? 48 : 64), "the error bound is for these K");
  static constexpr uint32_t kA = 128 * K * 2, kB = kTileN * K * 2;
  static constexpr int kMinStride = kGrans + 1;
  static constexpr uint32_t oB = 2 * kA, oMin = oB + kRing * kB, oX = oMin + kPoints * kMinStride * 4,
                            oBest = oX + kPoints * D * 4, oMask = (oBest + kWork * 4 + 7) / 8 * 8,
                            oBar = (oMask + kWork * (kTileN / kShare / kUnit) * 4 + 15) / 16 * 16, kSmem = oBar + 160;
  static_assert(kSmem <= 227 * 1024, "shared memory of a block");
};

// Scratch of one group's search (all of the workspace's book part).
struct Scratch {
  float4* tbook;    // kQuads x 4096 quarters of the entries in curve order, their index behind the values
  uint8_t* packed;  // 32 tiles of B
  int* perm;        // entry index at each place of the curve order
  float* center;    // 16
  unsigned* cmax;   // largest |c| of the entries in the product, float bits
  uint8_t* dead;    // 4096: equal to an entry of lower index
};
constexpr size_t kScratchBytes = size_t(5) * kEntries * 16 + size_t(kEntries) * 64 * 2 + kEntries * 4 + 256;

__device__ __forceinline__ uint16_t bf16_bits(float v) { return __bfloat16_as_ushort(__float2bfloat16_rn(v)); }
__device__ __forceinline__ float bf16_val(uint16_t b) { return __uint_as_float(uint32_t(b) << 16); }
struct Pieces {
  uint16_t h, m, l;
};
__device__ __forceinline__ Pieces pieces(float v) {
  Pieces p;
  p.h = bf16_bits(v);
  const float r = v - bf16_val(p.h);
  p.m = bf16_bits(r);
  p.l = bf16_bits(r - bf16_val(p.m));
  return p;
}

// Row `r` of a 128-row operand tile: the pieces of D values, by dimension, and three more columns.
template <int D, bool kPoint>
__device__ __forceinline__ void store_operand(uint8_t* tile, int r, const float (&v)[D], uint16_t e0, uint16_t e1,
                                              uint16_t e2) {
  using C = Cfg<D>;
  uint16_t row[C::K];
#pragma unroll
  for (int d = 0; d < D; ++d) {
    const Pieces p = pieces(v[d]);
    if (C::kTerms == 6) {
      // point h h m m h l against entry h m h m l h
      row[6 * d] = p.h;
      row[6 * d + 1] = kPoint ? p.h : p.m;
      row[6 * d + 2] = kPoint ? p.m : p.h;
      row[6 * d + 3] = p.m;
      row[6 * d + 4] = kPoint ? p.h : p.l;
      row[6 * d + 5] = kPoint ? p.l : p.h;
    } else {
      row[3 * d] = p.h;
      row[3 * d + 1] = kPoint ? p.h : p.m;
      row[3 * d + 2] = kPoint ? p.m : p.h;
    }
  }
  constexpr int n = D * C::kTerms;
  row[n] = e0;
  row[n + 1] = e1;
  row[n + 2] = e2;
#pragma unroll
  for (int k = n + 3; k < C::K; ++k) row[k] = 0;
#pragma unroll
  for (int c = 0; c < C::K / 8; ++c) {
    uint4 q;
    q.x = uint32_t(row[8 * c]) | uint32_t(row[8 * c + 1]) << 16;
    q.y = uint32_t(row[8 * c + 2]) | uint32_t(row[8 * c + 3]) << 16;
    q.z = uint32_t(row[8 * c + 4]) | uint32_t(row[8 * c + 5]) << 16;
    q.w = uint32_t(row[8 * c + 6]) | uint32_t(row[8 * c + 7]) << 16;
    *reinterpret_cast<uint4*>(tile + tile_off(uint32_t(r), uint32_t(8 * c), 128u)) = q;
  }
}

// Order of the entries along a space-filling curve (Morton code of up to 6 dimensions between their
// extremes) and their centre. One block; once per fit (entries move little).
template <int D>
__global__ void __launch_bounds__(1024) k_order(const float* __restrict__ book, int stride, int offset, Scratch S) {
  constexpr int kDims = D < 6 ? D : 6, kBits = 30 / kDims;
  extern __shared__ unsigned long long key[];  // 4096
  __shared__ float lo[kDims], hi[kDims];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  if (warp < D) {  // warp d: extremes and mean of dimension d
    float a = INFINITY, b = -INFINITY, s = 0.f;
    for (int k = lane; k < kEntries; k += 32) {
      const float v = book[size_t(k) * stride + offset + warp];
      a = fminf(a, v);
      b = fmaxf(b, v);
      s += v * (1.f / kEntries);
    }
    for (int o = 16; o > 0; o >>= 1) {
      a = fminf(a, __shfl_xor_sync(0xffffffffu, a, o));
      b = fmaxf(b, __shfl_xor_sync(0xffffffffu, b, o));
      s += __shfl_xor_sync(0xffffffffu, s, o);
    }
    if (lane == 0) {
      if (warp < kDims) {
        lo[warp] = a;
        hi[warp] = b;
      }
      S.center[warp] = isfinite(s) ? s : 0.f;
    }
  }
  __syncthreads();
  for (int k = tid; k < kEntries; k += 1024) {
    unsigned code = 0u;
    for (int d = 0; d < kDims; ++d) {
      const float e = hi[d] - lo[d];
      float t = e > 0.f ? (book[size_t(k) * stride + offset + d] - lo[d]) / e : 0.f;
      t = fminf(fmaxf(t, 0.f), 1.f) * float((1 << kBits) - 1);  // NaN: 0
      const unsigned u = unsigned(t);
      for (int b = 0; b < kBits; ++b) code |= ((u >> b) & 1u) << (b * kDims + d);
    }
    key[k] = (unsigned long long)code << 32 | unsigned(k);
  }
  for (int size = 2; size <= kEntries; size <<= 1)  // bitonic sort
    for (int j = size >> 1; j > 0; j >>= 1) {
      __syncthreads();
      for (int t = tid; t < kEntries / 2; t += 1024) {
        const int a = 2 * j * (t / j) + t % j, b = a + j;
        const unsigned long long x = key[a], y = key[b];
        if ((x > y) == ((a & size) == 0)) {
          key[a] = y;
          key[b] = x;
        }
      }
    }
  __syncthreads();
  for (int k = tid; k < kEntries; k += 1024) S.perm[k] = int(unsigned(key[k]));
}

// Marks the entries equal (value by value) to one of lower index. `dead` and `cmax` are zero before.
template <int D>
__global__ void __launch_bounds__(256) k_duplicates(const float* __restrict__ book, int stride, int offset, Scratch S) {
  if (blockIdx.y > blockIdx.x) return;
  __shared__ float c[256][D];
  const int k = int(blockIdx.x) * 256 + threadIdx.x, j0 = int(blockIdx.y) * 256;
  float v[D];
  for (int d = 0; d < D; ++d) {
    v[d] = book[size_t(k) * stride + offset + d];
    c[threadIdx.x][d] = book[size_t(j0 + threadIdx.x) * stride + offset + d];
  }
  __syncthreads();
  const int n = min(256, k - j0);
  for (int j = 0; j < n; ++j) {
    if (c[j][0] != v[0]) continue;
    bool same = true;
#pragma unroll
    for (int d = 1; d < D; ++d) same = same && c[j][d] == v[d];
    if (same) {
      S.dead[k] = 1;
      return;
    }
  }
}

// The entries in curve order: values for the exact scan, operand rows for the product.
template <int D>
__global__ void __launch_bounds__(128) k_pack(const float* __restrict__ book, int stride, int offset, Scratch S) {
  using C = Cfg<D>;
  const int p = int(blockIdx.x) * 128 + threadIdx.x;
  const int k = S.perm[p];
  float v[D], n2 = 0.f, q[4 * C::kQuads] = {};
#pragma unroll
  for (int d = 0; d < D; ++d) {
    const float c = book[size_t(k) * stride + offset + d];
    q[d] = c;
    v[d] = -(c - S.center[d]);
    n2 = fmaf(v[d], v[d], n2);
  }
  q[D] = __int_as_float(k);
#pragma unroll
  for (int c = 0; c < C::kQuads; ++c)
    S.tbook[size_t(c) * kEntries + p] = make_float4(q[4 * c], q[4 * c + 1], q[4 * c + 2], q[4 * c + 3]);
  // not finite or huge: no candidate of a point whose bound is finite
  const bool use = !S.dead[k] && n2 < 1e30f;
  if (!use) {
#pragma unroll
    for (int d = 0; d < D; ++d) v[d] = 0.f;
  }
  const Pieces h = pieces(use ? 0.5f * n2 : kDead);
  store_operand<D, false>(S.packed + size_t(blockIdx.x) * C::kB, threadIdx.x, v, h.h, h.m, h.l);
  if (use) atomicMax(S.cmax, __float_as_uint(sqrtf(n2)));
}

__device__ __forceinline__ float min3(uint32_t a, uint32_t b, uint32_t c) {
  float r;
  asm("min.f32 %0, %1, %2, %3;" : "=f"(r) : "f"(__uint_as_float(a)), "f"(__uint_as_float(b)), "f"(__uint_as_float(c)));
  return r;
}
__device__ __forceinline__ float min3f(float a, float b, float c) {
  return min3(__float_as_uint(a), __float_as_uint(b), __float_as_uint(c));
}
// Minimum of 16 accumulators (NaN ignored).
__device__ __forceinline__ float min16(const uint32_t (&r)[16]) {
  const float a = min3(r[0], r[1], r[2]), b = min3(r[3], r[4], r[5]), c = min3(r[6], r[7], r[8]),
              d = min3(r[9], r[10], r[11]), e = min3(r[12], r[13], r[14]);
  return min3f(min3f(a, b, c), fminf(d, e), __uint_as_float(r[15]));
}

// Minimum of 32.
__device__ __forceinline__ float min32(const uint32_t (&r)[16], const uint32_t (&t)[16]) {
  float m[10];
#pragma unroll
  for (int i = 0; i < 5; ++i) {
    m[i] = min3(r[3 * i], r[3 * i + 1], r[3 * i + 2]);
    m[5 + i] = min3(t[3 * i], t[3 * i + 1], t[3 * i + 2]);
  }
  const float a = min3f(m[0], m[1], m[2]), b = min3f(m[3], m[4], m[5]), c = min3f(m[6], m[7], m[8]),
              d = min3(__float_as_uint(m[9]), r[15], t[15]);
  return fminf(min3f(a, b, c), d);
}

template <int D>
__global__ void __launch_bounds__(kThreads, 1) k_assign(int64_t n, const float* __restrict__ X, int xstride, int xoffset,
                                                        Scratch S, uint16_t* __restrict__ code) {
  using C = Cfg<D>;
  extern __shared__ __align__(1024) uint8_t sm[];
  // warpgroups 0 and 1 take the first half of a tile's columns of points 0-127 and 128-255, 2 and 3 the second
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, pt = tid % kPoints, part = tid / kPoints;
  float* bests = reinterpret_cast<float*>(sm + C::oBest);
  uint32_t* masks = reinterpret_cast<uint32_t*>(sm + C::oMask);
  float* smin = reinterpret_cast<float*>(sm + C::oMin);
  float* xs = reinterpret_cast<float*>(sm + C::oX);
  const uint32_t full = smem_u32(sm + C::oBar), slotfree = full + 8 * kRing, accfull = slotfree + 8 * kRing, accfree = accfull + 32;
  uint32_t* tslot = reinterpret_cast<uint32_t*>(sm + C::oBar + 16 * kRing + 64);
  const int64_t ntiles = (n + kPoints - 1) / kPoints;
  const int mine = int((ntiles - blockIdx.x + gridDim.x - 1) / gridDim.x);  // the grid has at most ntiles blocks
  const int total = mine * kTiles;
  if (tid == 0) {
    for (int i = 0; i < kRing; ++i) {
      mbar_init(full + 8u * i, 1);
      mbar_init(slotfree + 8u * i, 2);
    }
    for (int i = 0; i < 4; ++i) {  // point tile 0's two buffers, then 1's
      mbar_init(accfull + 8u * i, 1);
      mbar_init(accfree + 8u * i, kWork / 64);
    }
    fence_mbar_init();
  }
  if (warp == kWork / 32) {
    tmem_alloc(smem_u32(tslot), 512);
    tmem_relinquish();
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *tslot;
  float center[D];
#pragma unroll
  for (int d = 0; d < D; ++d) center[d] = S.center[d];
  const float cmax = __uint_as_float(*S.cmax);
  auto load = [&](int s) {  // entry tile of step s into its ring slot
    const uint32_t bar = full + 8u * uint32_t(s % kRing);
    mbar_expect_tx(bar, C::kB);
    bulk_g2s(smem_u32(sm + C::oB + uint32_t(s % kRing) * C::kB), S.packed + size_t(s % kTiles) * C::kB, C::kB, bar);
  };
  int loaded = 0;
  if (tid == kWork + 64)
    for (; loaded < kRing - 1 && loaded < total; ++loaded) load(loaded);
  bool failed = false;
  for (int it = 0; it < mine; ++it) {
    const int64_t base = (int64_t(blockIdx.x) + int64_t(it) * gridDim.x) * kPoints;
    float x2 = 0.f, best = INFINITY, slack = 0.f;
    // is a unit of kUnit entries within the bound of the best so far? A bit per tile, the first in the highest
    constexpr int kUnit = C::kUnit, kFlags = kTileN / kShare / kUnit;
    static_assert(kTiles == 32, "a bit per tile");
    uint32_t flags[kFlags] = {};
    // The bound on s: kErr of |x| |c| + |c|^2 / 2; two entries whose d2 differ by less than its rounding may
    // change places. It grows with the best, so that one of an earlier, larger best keeps every candidate.
    auto bound = [&](float s) {
      const float thr = s + slack;
      return thr + float(D + 4) * 1.2e-7f * fmaxf(x2 + 2.f * thr, 0.f);
    };
    if (tid < kWork) {
      const int64_t i = base + pt;
      float v[D];
#pragma unroll
      for (int d = 0; d < D; ++d) {
        const float x = i < n ? X[i * xstride + xoffset + d] : 0.f;
        if (part == 0) xs[pt * D + d] = x;
        v[d] = x - center[d];
        x2 = fmaf(v[d], v[d], x2);
      }
      slack = 2.f * C::kErr * cmax * (sqrtf(x2) + 0.5f * cmax);
      if (part == 0) {
        const uint16_t one = 0x3F80;
        store_operand<D, true>(sm + (pt >> 7) * C::kA, pt & 127, v, one, one, one);
        fence_async_smem();
      }
    }
    __syncthreads();
    if (warp == kWork / 32 || warp == kWork / 32 + 1) {
      if (lane == 0) {  // the products of one point tile
        const uint32_t q = uint32_t(warp & 1), a = smem_u32(sm) + q * C::kA;
        static_assert(kTiles % kRing == 0 && kRing % 2 == 0 && kWork / 32 % 2 == 0, "slots by step, tile by warp");
#pragma unroll 4
        for (int t = 0; t < kTiles && !failed; ++t) {
          const int s = it * kTiles + t;
          const uint32_t acc = q * 2u + uint32_t(s & 1);
          failed = !mbar_wait(full + 8u * uint32_t(s % kRing), uint32_t(s / kRing) & 1u, kWaitNs) ||
                   (s >= 2 && !mbar_wait(accfree + 8u * acc, uint32_t(s / 2 - 1) & 1u, kWaitNs));
          if (failed) break;
          tc_fence_after();
          const uint32_t b = smem_u32(sm + C::oB + uint32_t(s % kRing) * C::kB);
          for (int k = 0; k < C::K / 16; ++k)
            mma_bf16(tmem + acc * 128u, desc_smem(a + uint32_t(k) * 4096u, 2048u, 128u),
                     desc_smem(b + uint32_t(k) * 4096u, 2048u, 128u), idesc_bf16_f32(128, kTileN), k > 0 ? 1u : 0u);
          mma_commit(slotfree + 8u * uint32_t(s % kRing));
          mma_commit(accfull + 8u * acc);
        }
      }
    } else if (tid == kWork + 64) {  // into the slot of step s - 1, once its products are done
      for (int t = 0; t < kTiles && !failed; ++t) {
        const int s = it * kTiles + t;
        if (s >= 1) failed = !mbar_wait(slotfree + 8u * uint32_t((s - 1) % kRing), uint32_t((s - 1) / kRing) & 1u, kWaitNs);
        if (!failed && loaded < total) load(loaded++);
      }
    } else if (tid < kWork) {
      constexpr int kCols = kTileN / kShare;
      const uint32_t q = uint32_t(pt >> 7);
      const uint32_t row = tmem + (uint32_t((warp & 3) * 32) << 16) + q * 256u + uint32_t(part * kCols);
      for (int t = 0; t < kTiles; ++t) {
        const int s = it * kTiles + t;
        if (!failed) failed = __any_sync(0xffffffffu, !mbar_wait(accfull + 8u * (q * 2u + uint32_t(s & 1)), uint32_t(s / 2) & 1u, kWaitNs));
        if (failed) break;
        tc_fence_after();
        uint32_t r[kCols / 16][16];
#pragma unroll
        for (int c = 0; c < kCols / 16; ++c) tmem_ld16(row + uint32_t(s & 1) * 128u + uint32_t(16 * c), r[c]);
        tmem_wait_ld();
        static_assert(kCols % C::kGran == 0, "whole granules per thread");
        float g = INFINITY;
#pragma unroll
        for (int c = 0; c < kCols / 16; c += 2) {
          reg_fence(r[c]);
          reg_fence(r[c + 1]);
          if (kUnit == 32) {
            const float m = min32(r[c], r[c + 1]);
            best = fminf(best, m);
            g = c * 16 % C::kGran == 0 ? m : fminf(g, m);
            flags[c / 2 % kFlags] = flags[c / 2 % kFlags] * 2u + (m <= bound(best) ? 1u : 0u);
          } else {
            const float m0 = min16(r[c]), m1 = min16(r[c + 1]);
            best = min3f(best, m0, m1);
            g = min3f(c * 16 % C::kGran == 0 ? INFINITY : g, m0, m1);
            const float thr = bound(best);
            flags[c % kFlags] = flags[c % kFlags] * 2u + (m0 <= thr ? 1u : 0u);
            flags[(c + 1) % kFlags] = flags[(c + 1) % kFlags] * 2u + (m1 <= thr ? 1u : 0u);
          }
          if ((16 * c + 32) % C::kGran == 0)
            smin[pt * C::kMinStride + (t * kTileN + part * kCols + 16 * c) / C::kGran] = g;
        }
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(accfree + 8u * (q * 2u + uint32_t(s & 1)));
      }
      // ---- the candidates by d2 (below 1e26 the nearest entry in the product is nearer than any left out as
      // huge can be). The two halves of a point's search meet: both take the smaller best
      bests[tid] = failed ? NAN : best;
      asm volatile("bar.sync 1, %0;" ::"n"(kWork) : "memory");
      const float other = bests[(tid + kPoints) % kWork];
      best = fminf(best, other);
      failed = failed || isnan(other);
      float thr = bound(best);
      if (failed || !(thr < 1e26f && x2 < 1e26f)) thr = INFINITY;  // every entry
      // this thread's units that hold candidates
#pragma unroll
      for (int h = 0; h < kFlags; ++h) {
        if (thr == INFINITY) flags[h] = ~0u;
        uint32_t keep = 0u;
        for (uint32_t f = flags[h]; f != 0u; f &= f - 1u) {
          const int g = ((32 - __ffs(f)) * kTileN + part * (kTileN / kShare) + h * kUnit) / C::kGran;
          if (thr == INFINITY || smin[pt * C::kMinStride + g] <= thr) keep |= f & -f;
        }
        masks[h * kWork + tid] = keep;
      }
      asm volatile("bar.sync 1, %0;" ::"n"(kWork) : "memory");
      // kLanes lanes per point; the two warps of 32 points take 16 each
      constexpr int kLanes = C::kLanes, kAtOnce = 32 / kLanes;
      int mycode = 0;
      const int sub = lane % kLanes, pw = pt & ~31;
      for (int r = 0; r < 16 / kAtOnce; ++r) {
        const int p = part * 16 + r * kAtOnce + lane / kLanes, pq = pw + p;
        float x[D];
#pragma unroll
        for (int d = 0; d < D; ++d) x[d] = xs[pq * D + d];
        float bd = INFINITY;
        int bi = 0x7fffffff;
#pragma unroll 1
        for (int h = 0; h < kFlags * kShare; ++h) {
          uint32_t m = masks[h % kFlags * kWork + h / kFlags * kPoints + pq];
          if (base + pq >= n) m = 0u;
          for (; m != 0u; m &= m - 1u) {
            const int e0 = (32 - __ffs(m)) * kTileN + h * kUnit + sub;
#pragma unroll
            for (int q = 0; q < kUnit; q += kLanes) {
              float d2 = 0.f, e[4 * C::kQuads];
#pragma unroll
              for (int c = 0; c < C::kQuads; ++c) {
                const float4 f = __ldg(S.tbook + size_t(c) * kEntries + e0 + q);
                e[4 * c] = f.x;
                e[4 * c + 1] = f.y;
                e[4 * c + 2] = f.z;
                e[4 * c + 3] = f.w;
              }
#pragma unroll
              for (int d = 0; d < D; ++d) {
                const float v = x[d] - e[d];
                d2 = fmaf(v, v, d2);
              }
              const int k = __float_as_int(e[D]);
              if (d2 < bd || (d2 == bd && d2 < INFINITY && k < bi)) {
                bd = d2;
                bi = k;
              }
            }
          }
          __syncwarp();
        }
#pragma unroll
        for (int o = kLanes / 2; o > 0; o >>= 1) {
          const float od = __shfl_xor_sync(0xffffffffu, bd, o);
          const int oi = __shfl_xor_sync(0xffffffffu, bi, o);
          if (od < bd || (od == bd && oi < bi)) {
            bd = od;
            bi = oi;
          }
        }
        const int got = __shfl_sync(0xffffffffu, bi, lane % kAtOnce * kLanes);
        if (lane / kAtOnce == part * 16 / kAtOnce + r) mycode = got == 0x7fffffff ? 0 : got;
      }
      const int64_t i = base + pt;
      if (i < n && lane >= part * 32 / kShare && lane < (part + 1) * 32 / kShare) code[i] = uint16_t(mycode);
    }
    failed = __syncthreads_or(failed);
  }
  if (tid == kWork + 64 && total > 0)  // what is in flight ends before the block does
    mbar_wait(slotfree + 8u * uint32_t((total - 1) % kRing), uint32_t((total - 1) / kRing) & 1u, failed ? kWaitNs / 20 : kWaitNs);
  if (tid == kWork + 64 && failed)
    for (int s = loaded > kRing ? loaded - kRing : 0; s < loaded; ++s)
      mbar_wait(full + 8u * uint32_t(s % kRing), uint32_t(s / kRing) & 1u, kWaitNs / 20);
  tc_fence_before();
  __syncthreads();
  if (warp == kWork / 32) {
    tc_fence_after();
    tmem_dealloc(tmem, 512);
  }
}

}  // namespace nearest
}  // namespace ugp

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
//     bits). A row of A holds pieces of x and three ones, a row of B the pieces of -c that they meet
//     and those of |c|^2 / 2: with 6 products per dimension (hh hm mh mm hl lh) what is left out is below
//     2^-26 of |x||c|, with 3 (hh hm mh; D = 16) below 2^-16.4.
//   * A block takes 256 points, one per thread of two warpgroups, as two M = 128 tiles, against 32 tiles
//     of 128 entries that a ninth warp brings in by bulk copies (ring of 4) and multiplies into two
//     accumulator buffers. Each thread reads its point's 128 accumulators per tile and keeps the minimum
//     of every granule of 32 or 64 entries in shared memory.
//   * Granules whose minimum is within the error bound of the point's smallest are then scanned by d2,
//     eight lanes per point. The entries are ordered along a space-filling curve, so
//     that candidates share granules, and entries equal to one of lower index, which cannot win,
//     are left out of the product (a plane of splats has one normal and one size: hundreds of
//     the starting entries are equal).
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
constexpr int kThreads = kPoints + 32;
constexpr uint64_t kWaitNs = 2000000000ull;  // 2 s per wait
constexpr float kDead = 1.7014118e38f;       // score of an entry left out (2^127)

// Products per dimension, K (a multiple of 16), entries per granule and the relative error bound of s
// (against (|x| + max |c|)^2): the products left out, K additions at 2^-22 each, the rounding of the
// moved coordinates and of d2 itself.
template <int D>
struct Cfg {
  static constexpr int kTerms = D <= 6 ? 6 : 3;
  static constexpr int K = (D * kTerms + 3 + 15) / 16 * 16;
  static constexpr int kGran = D <= 6 ? 32 : 64;
  static constexpr int kGrans = kEntries / kGran;
  static constexpr float kErr = D <= 6 ? 1.52587890625e-05f : 3.0517578125e-05f;  // 2^-16, 2^-15
  static_assert(K <= (D <= 6 ? 48 : 64), "the error bound is for these K");
  static constexpr uint32_t kA = 128 * K * 2, kB = kTileN * K * 2;
  static constexpr int kMinStride = kGrans + 1;
  static constexpr uint32_t oB = 2 * kA, oMin = oB + kRing * kB, oX = oMin + kPoints * kMinStride * 4,
                            oBar = (oX + kPoints * D * 4 + 15) / 16 * 16, kSmem = oBar + 128;
  static_assert(kSmem <= 227 * 1024, "shared memory of a block");
};

// Scratch of one group's search (all of the workspace's book part).
struct Scratch {
  float* tbook;     // D x 4096 entries in curve order, for the exact scan
  uint8_t* packed;  // 32 tiles of B
  int* perm;        // entry index at each place of the curve order
  float* center;    // 16
  unsigned* cmax;   // largest |c| of the entries in the product, float bits
  uint8_t* dead;    // 4096: equal to an entry of lower index
};
constexpr size_t kScratchBytes = size_t(16) * kEntries * 4 + size_t(kEntries) * 64 * 2 + kEntries * 4 + 256;

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
  float v[D], n2 = 0.f;
#pragma unroll
  for (int d = 0; d < D; ++d) {
    const float c = book[size_t(k) * stride + offset + d];
    S.tbook[size_t(d) * kEntries + p] = c;
    v[d] = -(c - S.center[d]);
    n2 = fmaf(v[d], v[d], n2);
  }
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
// Minimum of 16 accumulators (NaN ignored) in three levels.
__device__ __forceinline__ float min16(const uint32_t (&r)[16]) {
  const float a = min3(r[0], r[1], r[2]), b = min3(r[3], r[4], r[5]), c = min3(r[6], r[7], r[8]),
              d = min3(r[9], r[10], r[11]), e = min3(r[12], r[13], r[14]);
  return fminf(fminf(fminf(a, b), fminf(c, d)), fminf(e, __uint_as_float(r[15])));
}

template <int D>
__global__ void __launch_bounds__(kThreads, 1) k_assign(int64_t n, const float* __restrict__ X, int xstride, int xoffset,
                                                        Scratch S, uint16_t* __restrict__ code) {
  using C = Cfg<D>;
  extern __shared__ __align__(1024) uint8_t sm[];
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  float* smin = reinterpret_cast<float*>(sm + C::oMin);
  float* xs = reinterpret_cast<float*>(sm + C::oX);
  const uint32_t full = smem_u32(sm + C::oBar), accfull = full + 8 * kRing, accfree = accfull + 16;
  uint32_t* tslot = reinterpret_cast<uint32_t*>(sm + C::oBar + 8 * kRing + 32);
  const int64_t ntiles = (n + kPoints - 1) / kPoints;
  const int mine = int((ntiles - blockIdx.x + gridDim.x - 1) / gridDim.x);  // the grid has at most ntiles blocks
  const int total = mine * kTiles;
  if (tid == 0) {
    for (int i = 0; i < kRing; ++i) mbar_init(full + 8u * i, 1);
    for (int i = 0; i < 2; ++i) {
      mbar_init(accfull + 8u * i, 1);
      mbar_init(accfree + 8u * i, kPoints / 32);
    }
    fence_mbar_init();
  }
  if (warp == 8) {
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
  if (tid == kPoints)
    for (; loaded < kRing - 1 && loaded < total; ++loaded) load(loaded);
  bool failed = false;
  for (int it = 0; it < mine; ++it) {
    const int64_t base = (int64_t(blockIdx.x) + int64_t(it) * gridDim.x) * kPoints;
    float x2 = 0.f, best = INFINITY;
    if (warp < 8) {
      const int64_t i = base + tid;
      float v[D];
#pragma unroll
      for (int d = 0; d < D; ++d) {
        const float x = i < n ? X[i * xstride + xoffset + d] : 0.f;
        xs[tid * D + d] = x;
        v[d] = x - center[d];
        x2 = fmaf(v[d], v[d], x2);
      }
      const uint16_t one = 0x3F80;
      store_operand<D, true>(sm + (tid >> 7) * C::kA, tid & 127, v, one, one, one);
      fence_async_smem();
    }
    __syncthreads();
    if (tid == kPoints) {
      for (int t = 0; t < kTiles && !failed; ++t) {
        const int s = it * kTiles + t;
        failed = !mbar_wait(full + 8u * uint32_t(s % kRing), uint32_t(s / kRing) & 1u, kWaitNs) ||
                 (s >= 2 && !mbar_wait(accfree + 8u * uint32_t(s & 1), uint32_t(s / 2 - 1) & 1u, kWaitNs));
        if (failed) break;
        tc_fence_after();
        const uint32_t b = smem_u32(sm + C::oB + uint32_t(s % kRing) * C::kB);
        for (int q = 0; q < 2; ++q)
          for (int k = 0; k < C::K / 16; ++k)
            mma_bf16(tmem + uint32_t(s & 1) * 256u + uint32_t(q) * 128u,
                     desc_smem(smem_u32(sm) + uint32_t(q) * C::kA + uint32_t(k) * 4096u, 2048u, 128u),
                     desc_smem(b + uint32_t(k) * 4096u, 2048u, 128u), idesc_bf16_f32(128, kTileN), k > 0 ? 1u : 0u);
        mma_commit(accfull + 8u * uint32_t(s & 1));
        if (loaded < total) {  // into the slot of step s - 1, once its products are done
          if (s >= 1) failed = !mbar_wait(accfull + 8u * uint32_t((s - 1) & 1), uint32_t((s - 1) / 2) & 1u, kWaitNs);
          if (failed) break;
          load(loaded++);
        }
      }
    } else if (warp < 8) {
      const uint32_t row = tmem + (uint32_t((warp & 3) * 32) << 16) + uint32_t(warp >> 2) * 128u;
      for (int t = 0; t < kTiles; ++t) {
        const int s = it * kTiles + t;
        if (!failed) failed = __any_sync(0xffffffffu, !mbar_wait(accfull + 8u * uint32_t(s & 1), uint32_t(s / 2) & 1u, kWaitNs));
        if (failed) break;
        tc_fence_after();
        uint32_t r[kTileN / 16][16];
#pragma unroll
        for (int c = 0; c < kTileN / 16; ++c) tmem_ld16(row + uint32_t(s & 1) * 256u + uint32_t(16 * c), r[c]);
        tmem_wait_ld();
        float g = INFINITY;
#pragma unroll
        for (int c = 0; c < kTileN / 16; ++c) {
          reg_fence(r[c]);
          const float m = min16(r[c]);
          g = c * 16 % C::kGran == 0 ? m : fminf(g, m);
          if ((16 * c + 16) % C::kGran == 0) {
            smin[tid * C::kMinStride + (t * kTileN + 16 * c) / C::kGran] = g;
            best = fminf(best, g);
          }
        }
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(accfree + 8u * uint32_t(s & 1));
      }
      // ---- the candidates by d2. The bound on s: kErr of |x| |c| + |c|^2 / 2; two entries whose d2 differ
      // by less than its rounding may change places.
      // (below 1e26 the nearest entry in the product is nearer than any left out as huge can be)
      float thr = best + 2.f * C::kErr * cmax * (sqrtf(x2) + 0.5f * cmax);
      thr += float(D + 4) * 1.2e-7f * fmaxf(x2 + 2.f * thr, 0.f);
      if (failed || !(thr < 1e26f && x2 < 1e26f)) thr = INFINITY;  // every entry
      unsigned cand[C::kGrans / 32];  // this point's granules
#pragma unroll
      for (int c = 0; c < C::kGrans / 32; ++c) {
        cand[c] = 0u;
#pragma unroll 16
        for (int g = 0; g < 32; ++g)
          if (thr == INFINITY || smin[tid * C::kMinStride + 32 * c + g] <= thr) cand[c] |= 1u << g;
      }
      // eight lanes per point, four points at once
      int mycode = 0;
      const int sub = lane & 7;
      for (int r = 0; r < 8; ++r) {
        const int p = 4 * r + (lane >> 3), pt = warp * 32 + p;
        float x[D];
#pragma unroll
        for (int d = 0; d < D; ++d) x[d] = xs[pt * D + d];
        float bd = INFINITY;
        int bi = 0x7fffffff;
#pragma unroll 1
        for (int c = 0; c < C::kGrans / 32; ++c) {
          unsigned m = 0u;
#pragma unroll
          for (int k = 0; k < C::kGrans / 32; ++k) {
            const unsigned v = __shfl_sync(0xffffffffu, cand[k], p);
            if (k == c) m = v;
          }
          if (base + pt >= n) m = 0u;
          for (; m != 0u; m &= m - 1u) {
            const int e0 = (32 * c + __ffs(m) - 1) * C::kGran + sub;
#pragma unroll
            for (int q = 0; q < C::kGran; q += 8) {
              float d2 = 0.f;
#pragma unroll
              for (int d = 0; d < D; ++d) {
                const float v = x[d] - __ldg(S.tbook + size_t(d) * kEntries + e0 + q);
                d2 = fmaf(v, v, d2);
              }
              const int k = __ldg(S.perm + e0 + q);
              if (d2 < bd || (d2 == bd && d2 < INFINITY && k < bi)) {
                bd = d2;
                bi = k;
              }
            }
          }
          __syncwarp();
        }
#pragma unroll
        for (int o = 4; o > 0; o >>= 1) {
          const float od = __shfl_xor_sync(0xffffffffu, bd, o);
          const int oi = __shfl_xor_sync(0xffffffffu, bi, o);
          if (od < bd || (od == bd && oi < bi)) {
            bd = od;
            bi = oi;
          }
        }
        const int got = __shfl_sync(0xffffffffu, bi, (lane & 3) * 8);
        if ((lane >> 2) == r) mycode = got == 0x7fffffff ? 0 : got;
      }
      const int64_t i = base + tid;
      if (i < n) code[i] = uint16_t(mycode);
    }
    failed = __syncthreads_or(failed);
  }
  if (tid == kPoints && failed)  // copies still in flight end before the block does
    for (int s = loaded > kRing ? loaded - kRing : 0; s < loaded; ++s)
      mbar_wait(full + 8u * uint32_t(s % kRing), uint32_t(s / kRing) & 1u, kWaitNs / 20);
  tc_fence_before();
  __syncthreads();
  if (warp == 8) {
    tc_fence_after();
    tmem_dealloc(tmem, 512);
  }
}

}  // namespace nearest
}  // namespace ugp

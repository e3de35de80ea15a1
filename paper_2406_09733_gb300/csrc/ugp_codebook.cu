// Codebook-quantised primitive records (the compression the paper pairs with its level-of-detail
// scheme: per-attribute codebooks with random-access decoding).
//
// A record keeps the mean and the magnitude in float32 and replaces each other attribute group by
// the 12-bit index of its nearest codebook entry:
//   scale      (log s_x, log s_y, log s_z)                         3 values
//   rotation   the unit quaternion with w >= 0 (q and -q are one rotation)   4 values
//   SGGX       (Sxx, Syy, Szz, Sxy, Sxz, Syz)                        6 values
//   material   albedo 3, roughness, emission 3, Disney 9             16 values
// plus the material type (4 bits, exact). 24 bytes per primitive:
//   bytes 0-11 mean (float x3), 12-15 magnitude (float), 16-17 scale code, 18-19 rotation code,
//   20-21 SGGX code, 22-23 material code | type << 12.
// Each codebook has kCodes entries, fitted by Lloyd iterations on the device: every point goes
// to its nearest entry (squared distance, ties to the lower index), then every entry with points
// moves to their mean. The sums are 64-bit fixed point (units of 2^-24), so the fit does not
// depend on the order of the atomic additions. Entries start at the points of index
// floor(k n / kCodes).
#include <math.h>
#include <string.h>

#include "ugp_internal.cuh"
#include "ugp_nearest.cuh"

namespace ugp {
namespace {

constexpr int kCodes = 4096;
constexpr int kGroups = 4;
constexpr int kDim[kGroups] = {3, 4, 6, 16};
constexpr int kOff[kGroups] = {0, 3, 7, 13};  // offsets of the groups in a 29-value feature row
constexpr int kFeat = 29;
constexpr float kFix = 16777216.f;  // 2^24

__host__ __device__ constexpr size_t book_floats() { return size_t(kCodes) * kFeat; }

// Feature row of primitive i (the values each codebook quantises).
__global__ void k_features(int64_t n, const float* __restrict__ quat4, const float* __restrict__ scale3,
                           const float* __restrict__ sggx6, const float* __restrict__ albedo3,
                           const float* __restrict__ rough, const float* __restrict__ emit3,
                           const float* __restrict__ dis9, float* __restrict__ X) {
  const int64_t i = int64_t(blockIdx.x) * blockDim.x + threadIdx.x;
  if (i >= n) return;
  float* x = X + i * kFeat;
  for (int a = 0; a < 3; ++a) x[a] = logf(fmaxf(scale3[3 * i + a], 1e-30f));
  float q[4] = {quat4[4 * i], quat4[4 * i + 1], quat4[4 * i + 2], quat4[4 * i + 3]};
  const float inv = rsqrtf(fmaxf(q[0] * q[0] + q[1] * q[1] + q[2] * q[2] + q[3] * q[3], 1e-30f));
  const float sg = q[0] < 0.f ? -inv : inv;
  for (int a = 0; a < 4; ++a) x[3 + a] = q[a] * sg;
  for (int a = 0; a < 6; ++a) x[7 + a] = sggx6[6 * i + a];
  for (int a = 0; a < 3; ++a) x[13 + a] = albedo3[3 * i + a];
  x[16] = rough[i];
  for (int a = 0; a < 3; ++a) x[17 + a] = emit3[3 * i + a];
  for (int a = 0; a < 9; ++a) x[20 + a] = dis9 ? dis9[9 * i + a] : 0.f;
}

// Entries start at the points of index floor(k n / kCodes).
__global__ void k_init_book(int64_t n, const float* __restrict__ X, float* __restrict__ book) {
  const int k = int(blockIdx.x) * blockDim.x + threadIdx.x;
  if (k >= kCodes) return;
  const int64_t i = (int64_t(k) * n) / kCodes;
  for (int f = 0; f < kFeat; ++f) book[size_t(k) * kFeat + f] = X[i * kFeat + f];
}

// Fixed-point sums and counts of the points of every entry of group G. Points share few entries (a wall has
// one normal and one size, a cluster one material), so atomics to global memory queue on them: 2.0 ms for
// the SGGX of 1M points, 1.4 for their materials. A block sums its points in shared memory first, acc_dims
// values at a time (blockIdx.y), once per warp where all its points have the same entry, and adds what it
// found to global memory. An addition of 64 bits in shared memory is a loop that tries until no other
// lane came between, so the sums are kept as two words of 32 bits: the low kAccBits of the values, which
// 2^15 of them cannot carry out of a word, and the rest (materials of 1M points: 0.48 -> 0.10 ms).
// Values from 512 up, whose rest could overflow, go to global memory as they are.
constexpr int kAccThreads = 512, kAccLog = 15, kAccBits = 32 - kAccLog;
constexpr int kAccRounds = (1 << kAccLog) / kAccThreads;  // 2^15 points per block between write-outs
template <int G>
constexpr int acc_dims() { return kDim[G] <= 4 ? kDim[G] : (kDim[G] == 6 ? 3 : 4); }
template <int G>
constexpr size_t acc_smem() { return size_t(kCodes) * (acc_dims<G>() * 8 + 4); }
template <int G>
__global__ void __launch_bounds__(kAccThreads, 1) k_accumulate(int64_t n, const float* __restrict__ X,
                                                               const uint16_t* __restrict__ code,
                                                               unsigned long long* __restrict__ sums,
                                                               unsigned int* __restrict__ cnt) {
  constexpr int D = kDim[G], O = kOff[G], N = acc_dims<G>();
  extern __shared__ unsigned acc[];  // of N x kCodes sums the low words, then the high ones; then the counts
  unsigned* high = acc + N * kCodes;
  unsigned* num = high + N * kCodes;
  const int lane = threadIdx.x & 31, d0 = int(blockIdx.y) * N;
  const int64_t step = int64_t(gridDim.x) * kAccThreads;
  for (int64_t i1 = int64_t(blockIdx.x) * kAccThreads; i1 < n; i1 += step * kAccRounds) {
    for (int k = threadIdx.x; k < kCodes; k += kAccThreads) {
      for (int d = 0; d < N; ++d) acc[d * kCodes + k] = high[d * kCodes + k] = 0u;
      num[k] = 0u;
    }
    __syncthreads();
    const int64_t end = n < i1 + step * kAccRounds ? n : i1 + step * kAccRounds;
    for (int64_t i0 = i1; i0 < end; i0 += step) {
      const int64_t i = i0 + threadIdx.x;
      const int k = i < n ? int(code[i]) : -1;
      long long v[N];
#pragma unroll
      for (int d = 0; d < N; ++d) v[d] = k >= 0 ? __float2ll_rn(X[i * kFeat + O + d0 + d] * kFix) : 0ll;
      const int k0 = __shfl_sync(0xffffffffu, k, 0);
      const bool one = __all_sync(0xffffffffu, k == k0);
      if (one) {
#pragma unroll
        for (int d = 0; d < N; ++d)
          for (int o = 16; o > 0; o >>= 1) v[d] += __shfl_xor_sync(0xffffffffu, v[d], o);
      }
      if (k < 0) continue;
#pragma unroll
      for (int d = 0; d < N; ++d) {
        if (one && lane != d) continue;
        const long long h = v[d] >> kAccBits;
        if (h < -(1 << (31 - kAccLog)) || h >= 1 << (31 - kAccLog)) {
          atomicAdd(sums + size_t(k) * D + d0 + d, (unsigned long long)v[d]);
        } else {
          atomicAdd(acc + d * kCodes + k, unsigned(v[d]) & ((1u << kAccBits) - 1u));
          atomicAdd(high + d * kCodes + k, unsigned(int(h)));
        }
      }
      if (!one) atomicAdd(num + k, 1u);
      else if (lane == 0) atomicAdd(num + k, 32u);
    }
    __syncthreads();
    for (int k = threadIdx.x; k < kCodes; k += kAccThreads) {
      if (num[k] == 0u) continue;
      for (int d = 0; d < N; ++d) {
        const long long v = ((long long)int(high[d * kCodes + k]) << kAccBits) + acc[d * kCodes + k];
        atomicAdd(sums + size_t(k) * D + d0 + d, (unsigned long long)v);
      }
      if (blockIdx.y == 0) atomicAdd(cnt + k, num[k]);
    }
    __syncthreads();
  }
}

// Entries with points move to their mean; the others stay.
template <int G>
__global__ void k_update(const unsigned long long* __restrict__ sums, const unsigned int* __restrict__ cnt,
                         float* __restrict__ book) {
  constexpr int D = kDim[G], O = kOff[G];
  const int k = int(blockIdx.x) * blockDim.x + threadIdx.x;
  if (k >= kCodes || cnt[k] == 0) return;
  for (int d = 0; d < D; ++d) {
    const long long s = (long long)sums[size_t(k) * D + d];
    book[size_t(k) * kFeat + O + d] = float(double(s) / (double(kFix) * double(cnt[k])));
  }
}

__global__ void k_pack(int64_t n, const float* __restrict__ mean3, const float* __restrict__ mag,
                       const uint8_t* __restrict__ type, const uint16_t* __restrict__ codes,
                       uint32_t* __restrict__ rec) {
  const int64_t i = int64_t(blockIdx.x) * blockDim.x + threadIdx.x;
  if (i >= n) return;
  uint32_t* r = rec + 6 * i;
  r[0] = __float_as_uint(mean3[3 * i]);
  r[1] = __float_as_uint(mean3[3 * i + 1]);
  r[2] = __float_as_uint(mean3[3 * i + 2]);
  r[3] = __float_as_uint(mag[i]);
  const uint32_t cs = codes[i], cr = codes[n + i], cg = codes[2 * n + i], cm = codes[3 * n + i];
  r[4] = cs | (cr << 16);
  r[5] = cg | ((cm | (uint32_t(type[i] & 15u) << 12)) << 16);
}

// Random-access decode of record i into the caller's layout (ugp_prims / ugp_materials).
__global__ void k_decode(int64_t n, const uint32_t* __restrict__ rec, const float* __restrict__ book,
                         float* __restrict__ mean3, float* __restrict__ quat4, float* __restrict__ scale3,
                         float* __restrict__ mag, float* __restrict__ sggx6, uint8_t* __restrict__ type,
                         float* __restrict__ albedo3, float* __restrict__ rough, float* __restrict__ emit3,
                         float* __restrict__ dis9) {
  const int64_t i = int64_t(blockIdx.x) * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const uint32_t* r = rec + 6 * i;
  for (int a = 0; a < 3; ++a) mean3[3 * i + a] = __uint_as_float(r[a]);
  mag[i] = __uint_as_float(r[3]);
  const int cs = r[4] & 0xffffu, cr = r[4] >> 16, cg = r[5] & 0xffffu, cm = (r[5] >> 16) & 0xfffu;
  type[i] = uint8_t(r[5] >> 28);
  const float* bs = book + size_t(cs) * kFeat;
  for (int a = 0; a < 3; ++a) scale3[3 * i + a] = expf(bs[a]);
  const float* br = book + size_t(cr) * kFeat + 3;
  const float inv = rsqrtf(fmaxf(br[0] * br[0] + br[1] * br[1] + br[2] * br[2] + br[3] * br[3], 1e-30f));
  for (int a = 0; a < 4; ++a) quat4[4 * i + a] = br[a] * inv;
  const float* bg = book + size_t(cg) * kFeat + 7;
  for (int a = 0; a < 6; ++a) sggx6[6 * i + a] = bg[a];
  const float* bm = book + size_t(cm) * kFeat + 13;
  for (int a = 0; a < 3; ++a) albedo3[3 * i + a] = bm[a];
  rough[i] = bm[3];
  for (int a = 0; a < 3; ++a) emit3[3 * i + a] = bm[4 + a];
  if (dis9)
    for (int a = 0; a < 9; ++a) dis9[9 * i + a] = bm[7 + a];
}

// `sums`, `cnt`, `cmax` and `dead` are cleared together before each search.
struct CbLayout {
  size_t X, codes, sums, cnt, cmax, dead, book, total;
};
CbLayout cb_layout(int64_t n) {
  CbLayout L;
  size_t off = 0;
  L.X = off;     off = align256(off + size_t(n) * kFeat * 4);
  L.codes = off; off = align256(off + size_t(n) * kGroups * 2);
  L.sums = off;  off = align256(off + size_t(kCodes) * 16 * 8);
  L.cnt = off;   off = align256(off + size_t(kCodes) * 4);
  L.cmax = off;  off += 256;
  L.dead = off;  off = align256(off + size_t(kCodes));
  L.book = off;  off = align256(off + nearest::kScratchBytes);
  L.total = off;
  return L;
}

// Nearest entries of group G for every point.
template <int G>
ugp_status assign_group(int64_t n, const float* X, const float* book, char* ws, const CbLayout& L, uint16_t* code,
                        const nearest::Scratch& S, int sms, cudaStream_t st) {
  constexpr int D = kDim[G], O = kOff[G];
  using C = nearest::Cfg<D>;
  UGP_CUDA_CHECK(cudaMemsetAsync(ws + L.sums, 0, L.book - L.sums, st));
  nearest::k_duplicates<D><<<dim3(kCodes / 256, kCodes / 256), 256, 0, st>>>(book, kFeat, O, S);
  nearest::k_pack<D><<<kCodes / 128, 128, 0, st>>>(book, kFeat, O, S);
  const int64_t tiles = (n + nearest::kPoints - 1) / nearest::kPoints;
  nearest::k_assign<D><<<unsigned(tiles < sms ? tiles : sms), nearest::kThreads, C::kSmem, st>>>(n, X, kFeat, O, S, code);
  UGP_CUDA_CHECK(cudaGetLastError());
  return UGP_OK;
}
constexpr int kAssignKernels = 3;

template <int G>
ugp_status fit_group(int64_t n, const float* X, float* book, uint16_t* code, char* ws, const CbLayout& L, int iters,
                     cudaStream_t st) {
  constexpr int D = kDim[G];
  using C = nearest::Cfg<D>;
  static_assert(nearest::kEntries == kCodes, "entries");
  int dev = 0, sms = 0;
  UGP_CUDA_CHECK(cudaGetDevice(&dev));
  UGP_CUDA_CHECK(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
  UGP_CUDA_CHECK(cudaFuncSetAttribute(nearest::k_assign<D>, cudaFuncAttributeMaxDynamicSharedMemorySize, int(C::kSmem)));
  char* p = ws + L.book;
  nearest::Scratch S;
  S.tbook = reinterpret_cast<float4*>(p);
  S.packed = reinterpret_cast<uint8_t*>(p + size_t(5) * kCodes * 16);
  S.perm = reinterpret_cast<int*>(p + size_t(5) * kCodes * 16 + size_t(kCodes) * 64 * 2);
  S.center = reinterpret_cast<float*>(reinterpret_cast<char*>(S.perm) + size_t(kCodes) * 4);
  S.cmax = reinterpret_cast<unsigned*>(ws + L.cmax);
  S.dead = reinterpret_cast<uint8_t*>(ws + L.dead);
  unsigned long long* sums = reinterpret_cast<unsigned long long*>(ws + L.sums);
  unsigned int* cnt = reinterpret_cast<unsigned int*>(ws + L.cnt);
  // a block per SM over all parts, fewer when a block would get less than 4096 points
  constexpr int parts = D / acc_dims<G>();
  const int64_t want = (n + 4095) / 4096, fit = sms / parts > 0 ? sms / parts : 1;
  const unsigned acc_blocks = unsigned(want < fit ? want : fit);
  UGP_CUDA_CHECK(cudaFuncSetAttribute(k_accumulate<G>, cudaFuncAttributeMaxDynamicSharedMemorySize, int(acc_smem<G>())));
  nearest::k_order<D><<<1, 1024, kCodes * 8, st>>>(book, kFeat, kOff[G], S);
  for (int it = 0; it < iters; ++it) {
    const ugp_status s = assign_group<G>(n, X, book, ws, L, code, S, sms, st);
    if (s != UGP_OK) return s;
    k_accumulate<G><<<dim3(acc_blocks, parts), kAccThreads, acc_smem<G>(), st>>>(n, X, code, sums, cnt);
    k_update<G><<<kCodes / 256, 256, 0, st>>>(sums, cnt, book);
  }
  return assign_group<G>(n, X, book, ws, L, code, S, sms, st);
}

}  // namespace
}  // namespace ugp

using namespace ugp;

extern "C" size_t ugp_codebook_size(void) { return book_floats() * 4; }

extern "C" size_t ugp_codebook_workspace_size(int64_t n_prims) {
  if (n_prims < 0 || n_prims > (int64_t(1) << 30)) return 0;
  return cb_layout(n_prims).total;
}

extern "C" ugp_status ugp_codebook_encode(const ugp_prims* prims, const ugp_materials* materials, int32_t iters,
                                          void* codebook, void* records, void* workspace, size_t workspace_bytes,
                                          void* stream) {
  clear_error();
  if (!prims || !materials || !codebook || !records)
    return fail(UGP_ERR_INVALID_ARG, "ugp_codebook_encode: NULL argument");
  const int64_t n = prims->n;
  if (n < 1 || n > (int64_t(1) << 30))
    return fail(UGP_ERR_INVALID_ARG, "ugp_codebook_encode: n_prims %lld not in [1, 2^30]", (long long)n);
  if (iters < 0 || iters > 100) return fail(UGP_ERR_INVALID_ARG, "ugp_codebook_encode: iters not in [0, 100]");
  if (!prims->mean3 || !prims->quat4 || !prims->scale3 || !prims->magnitude || !materials->sggx6 ||
      !materials->type || !materials->albedo3 || !materials->roughness || !materials->emission3)
    return fail(UGP_ERR_INVALID_ARG, "ugp_codebook_encode: NULL primitive or material array");
  if (!workspace || (reinterpret_cast<uintptr_t>(workspace) & 255) || (reinterpret_cast<uintptr_t>(codebook) & 15) ||
      (reinterpret_cast<uintptr_t>(records) & 3))
    return fail(UGP_ERR_INVALID_ARG, "ugp_codebook_encode: NULL or misaligned workspace, codebook or records");
  const CbLayout L = cb_layout(n);
  if (workspace_bytes < L.total)
    return fail(UGP_ERR_WORKSPACE_TOO_SMALL, "ugp_codebook_encode: need %zu bytes, got %zu", L.total,
                workspace_bytes);
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  char* ws = static_cast<char*>(workspace);
  float* X = reinterpret_cast<float*>(ws + L.X);
  uint16_t* codes = reinterpret_cast<uint16_t*>(ws + L.codes);
  float* book = static_cast<float*>(codebook);
  const unsigned gp = unsigned((n + 255) / 256);
  prof_begin(kStBuild, st);
  k_features<<<gp, 256, 0, st>>>(n, prims->quat4, prims->scale3, materials->sggx6, materials->albedo3,
                                 materials->roughness, materials->emission3, materials->disney9, X);
  k_init_book<<<kCodes / 256, 256, 0, st>>>(n, X, book);
  UGP_CUDA_CHECK(cudaGetLastError());
  ugp_status s;
  if ((s = fit_group<0>(n, X, book, codes, ws, L, iters, st)) != UGP_OK) return s;
  if ((s = fit_group<1>(n, X, book, codes + n, ws, L, iters, st)) != UGP_OK) return s;
  if ((s = fit_group<2>(n, X, book, codes + 2 * n, ws, L, iters, st)) != UGP_OK) return s;
  if ((s = fit_group<3>(n, X, book, codes + 3 * n, ws, L, iters, st)) != UGP_OK) return s;
  k_pack<<<gp, 256, 0, st>>>(n, prims->mean3, prims->magnitude, materials->type, codes,
                             static_cast<uint32_t*>(records));
  prof_end(kStBuild, st, 3 + kGroups * (1 + (2 + kAssignKernels) * iters + kAssignKernels));
  UGP_CUDA_CHECK(cudaGetLastError());
  return UGP_OK;
}

extern "C" ugp_status ugp_codebook_decode(int64_t n, const void* records, const void* codebook, float* mean3,
                                          float* quat4, float* scale3, float* magnitude, float* sggx6,
                                          uint8_t* type, float* albedo3, float* roughness, float* emission3,
                                          float* disney9, void* stream) {
  clear_error();
  if (n < 0 || n > (int64_t(1) << 30)) return fail(UGP_ERR_INVALID_ARG, "ugp_codebook_decode: n out of range");
  if (n == 0) return UGP_OK;
  if (!records || !codebook || !mean3 || !quat4 || !scale3 || !magnitude || !sggx6 || !type || !albedo3 ||
      !roughness || !emission3)
    return fail(UGP_ERR_INVALID_ARG, "ugp_codebook_decode: NULL array (only disney9 may be NULL)");
  if ((reinterpret_cast<uintptr_t>(records) & 3) || (reinterpret_cast<uintptr_t>(codebook) & 3))
    return fail(UGP_ERR_INVALID_ARG, "ugp_codebook_decode: misaligned records or codebook");
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  prof_begin(kStBuild, st);
  k_decode<<<unsigned((n + 255) / 256), 256, 0, st>>>(n, static_cast<const uint32_t*>(records),
                                                      static_cast<const float*>(codebook), mean3, quat4, scale3,
                                                      magnitude, sggx6, type, albedo3, roughness, emission3, disney9);
  prof_end(kStBuild, st);
  UGP_CUDA_CHECK(cudaGetLastError());
  return UGP_OK;
}

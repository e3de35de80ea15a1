// Radiance-field forward render (Sec. 7, Eq. rf): an emitting, non-scattering medium of the
// primitives, rendered without Monte Carlo.
//
//   L = sum_k 1/2 I_k(a_k, min(b_k, t_sat)) L_e,k  +  max(0, 1 - F(t1)) L_bg  (when F(t1) <= 1)
//
// t_sat is where F (the free-flight CDF, Eq. 8) reaches 1: the free-flight root for u = 1, which
// is also how the paper settles which primitives straddle the saturating boundary. Each
// primitive then counts with its probability mass up to t_sat, which needs no choice among
// them. Two passes per ray: free-flight sampling at u = 1 (scan and finish, as for the path
// tracer), then one lane per ray sums the clipped integrals weighted by the emissions.
#include "ugp_dense.cuh"
#include "ugp_gauss.cuh"
#include "ugp_trace.cuh"
#include "ugp_transmit.cuh"

namespace ugp {
namespace {

__global__ void k_fill(int64_t n, float* __restrict__ p, float v) {
  for (int64_t i = blockIdx.x * int64_t(blockDim.x) + threadIdx.x; i < n; i += int64_t(gridDim.x) * blockDim.x)
    p[i] = v;
}

// Mass and emission of one ray's primitives up to t_end (tr_walk's collector). The lanes of a leaf step
// form the terms, and each owner adds its own ray's, one after the other in the order in which the ray met them:
// a float sum that does not depend on the rays beside it or on the size of the call. (A sum over the lanes by four
// doublings, whose grouping did, took the same time: 921,600 camera rays in a 1M-primitive room 6.79 ms with both.)
struct RadianceSum {
  static constexpr bool kNearFirst = false, kInOrder = true;
  const float* em3;
  float t_end;
  float mass, r, g, b;
  __device__ void leaf(bool ok, const PrimHit& h, int o, int off, int mine) {
    constexpr unsigned kAll = 0xffffffffu;
    const float te = __shfl_sync(kAll, t_end, o);
    float v = 0.f, er = 0.f, eg = 0.f, eb = 0.f;
    bool adds = false;
    if (ok) {
      const float y = fminf(h.b, te);
      if (h.a < y) {
        adds = true;
        v = seg_half_integral(h.a, y, h.a, h.b, h.a_end, h.b_end, h.tn, h.ts, h.s, h.e0, h.th);
        er = __ldg(em3 + 3 * int64_t(h.id));
        eg = __ldg(em3 + 3 * int64_t(h.id) + 1);
        eb = __ldg(em3 + 3 * int64_t(h.id) + 2);
      }
    }
    // this lane's own ray's terms, as bits from lane off on
    static_assert(kTrLeafQ < 32, "a ray's primitives in one word");
    const unsigned all = __ballot_sync(kAll, adds);
    const int taken = min(mine, max(0, 32 - off));
    unsigned terms = taken > 0 ? (all >> off) & ((1u << taken) - 1u) : 0u;
    for (int left = int(__reduce_max_sync(kAll, unsigned(__popc(terms)))); left > 0; --left) {
      const int src = (off + __ffs(terms) - 1) & 31;
      const float w = __shfl_sync(kAll, v, src), wr = __shfl_sync(kAll, er, src), wg = __shfl_sync(kAll, eg, src),
                  wb = __shfl_sync(kAll, eb, src);
      if (terms != 0u) {
        mass += w;
        r = fmaf(w, wr, r);
        g = fmaf(w, wg, g);
        b = fmaf(w, wb, b);
      }
      terms &= terms - 1u;
    }
  }
  __device__ bool enough() const { return false; }
};

// One ray per lane: every clipped interval over [t0, t_end] (t_end = t_sat when the free-flight pass
// found one, else t1), cut at t_end, its 1/2 I times the primitive's emission. The transmittance's
// traversal (4-wide nodes, leaf steps shared by the warp); walking the binary tree with a lane per ray
// and its own primitives took 3.45 ms for 921,600 camera rays in a 1M-primitive room, this 1.77.
__global__ void __launch_bounds__(kTrBlock, 8)
k_radiance(TraceScene sc, int64_t n_rays, const float* __restrict__ o3, const float* __restrict__ d3,
           const float* __restrict__ t0a, const float* __restrict__ t1a, const int32_t* __restrict__ prim_ff,
           const float* __restrict__ tu_ff, const uint8_t* __restrict__ st_ff, const float* __restrict__ em3,
           float3 bg, float* __restrict__ rgb_out, uint8_t* __restrict__ st_out) {
  __shared__ int stk[kTrStack * kTrBlock];
  __shared__ int owner[kTrBlock];
  const int rpw = rays_per_warp(n_rays, min(int(gridDim.x) * (kTrBlock / 32), kTrWarps));
  const int64_t r0 = (int64_t(blockIdx.x) * (kTrBlock / 32) + (threadIdx.x >> 5)) * rpw;
  const int64_t r = r0 + (threadIdx.x & 31);
  if (r0 >= n_rays) return;  // the whole warp
  const bool live = int(threadIdx.x & 31) < rpw && r < n_rays;
  TrStats ts{0u, 0u, UGP_RAY_OK};
  Ray ray{};
  float t0 = 0.f, t1 = 0.f, t_end = 0.f;
  bool sat = false;
  uint8_t st = UGP_RAY_OK;
  if (live) {
    ray = make_ray(ld3(o3, r), ld3(d3, r));
    t0 = __ldg(t0a + r);
    t1 = __ldg(t1a + r);
    sat = __ldg(prim_ff + r) >= 0;
    t_end = sat ? __ldg(tu_ff + r) : t1;
    if (st_ff) st = __ldg(st_ff + r);
  }
  RadianceSum sum{em3, t_end, 0.f, 0.f, 0.f, 0.f};
  tr_walk<false, true>(sc, ray, t0, t1, t_end, -1, stk + threadIdx.x, kTrBlock, owner + threadIdx.x, ts,
                 live && st == UGP_RAY_OK, 0, sum);
  if (!live) return;
  const float rest = sat ? 0.f : fmaxf(0.f, 1.f - sum.mass);
  rgb_out[3 * r] = fmaf(rest, bg.x, sum.r);
  rgb_out[3 * r + 1] = fmaf(rest, bg.y, sum.g);
  rgb_out[3 * r + 2] = fmaf(rest, bg.z, sum.b);
  if (st_out) st_out[r] = st != UGP_RAY_OK ? st : ts.st;
}

// Workspace: the free-flight pass's, then u, u2, prim, t_u, t_spawn and the status per ray.
struct RfLayout {
  size_t ff, u, u2, prim, tu, tsp, st, total;
};
RfLayout rf_layout(int64_t n) {
  RfLayout L;
  size_t off = 0;
  L.ff = off;   off += dense_queue_bytes(n) + slot_list_bytes(n);
  L.u = off;    off += align256(size_t(n) * 4);
  L.u2 = off;   off += align256(size_t(n) * 4);
  L.prim = off; off += align256(size_t(n) * 4);
  L.tu = off;   off += align256(size_t(n) * 4);
  L.tsp = off;  off += align256(size_t(n) * 4);
  L.st = off;   off += align256(size_t(n));
  L.total = off;
  return L;
}

}  // namespace
}  // namespace ugp

using namespace ugp;

extern "C" size_t ugp_render_radiance_field_workspace_size(int64_t n_rays) {
  if (n_rays < 0 || n_rays > (int64_t(1) << 31) - 1) return 0;
  return rf_layout(n_rays).total;
}

extern "C" ugp_status ugp_render_radiance_field(const ugp_bvh* bvh, int64_t n_rays, const float* o3,
                                                const float* d3, const float* t0, const float* t1,
                                                const float* emission3, const float* background3, float* rgb_out,
                                                uint8_t* status_out, void* workspace, size_t workspace_bytes,
                                                void* stream) {
  clear_error();
  ugp_status s = check_rays("ugp_render_radiance_field", bvh, n_rays, o3, d3, t0, t1);
  if (s != UGP_OK) return s;
  if (n_rays > 0 && (!emission3 || !rgb_out))
    return fail(UGP_ERR_INVALID_ARG, "ugp_render_radiance_field: NULL emission or output array");
  if (n_rays == 0) return UGP_OK;
  if (n_rays > (int64_t(1) << 31) - 1)
    return fail(UGP_ERR_INVALID_ARG, "ugp_render_radiance_field: at most 2^31 - 1 rays per call");
  if (!workspace || (reinterpret_cast<uintptr_t>(workspace) & 255))
    return fail(UGP_ERR_INVALID_ARG, "ugp_render_radiance_field: workspace must be non-NULL and 256-byte aligned");
  const RfLayout L = rf_layout(n_rays);
  if (workspace_bytes < L.total)
    return fail(UGP_ERR_WORKSPACE_TOO_SMALL, "ugp_render_radiance_field: need %zu bytes, got %zu", L.total,
                workspace_bytes);
  const float3 bg = background3 ? make_float3(background3[0], background3[1], background3[2])
                                : make_float3(0.f, 0.f, 0.f);
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  char* ws = static_cast<char*>(workspace);
  float* u = reinterpret_cast<float*>(ws + L.u);
  float* u2 = reinterpret_cast<float*>(ws + L.u2);
  int32_t* prim = reinterpret_cast<int32_t*>(ws + L.prim);
  float* tu = reinterpret_cast<float*>(ws + L.tu);
  float* tsp = reinterpret_cast<float*>(ws + L.tsp);
  uint8_t* sf = reinterpret_cast<uint8_t*>(ws + L.st);
  const TraceScene sc = trace_scene(bvh);
  const int fill_grid = int((n_rays + 255) / 256 < 4096 ? (n_rays + 255) / 256 : 4096);
  prof_begin(kStQuery, st);
  k_fill<<<fill_grid, 256, 0, st>>>(n_rays, u, 1.f);  // u = 1: the root is the saturating distance
  prof_end(kStQuery, st);
  UGP_CUDA_CHECK(cudaGetLastError());
  UGP_CUDA_CHECK(cudaMemsetAsync(u2, 0, size_t(n_rays) * 4, st));
  if ((s = launch_free_flight(sc, n_rays, o3, d3, t0, t1, u, u2, nullptr, prim, tu, tsp, sf, ws + L.ff, true, st)) !=
      UGP_OK)
    return s;
  prof_begin(kStQuery, st);
  k_radiance<<<unsigned(tr_grid(n_rays)), kTrBlock, 0, st>>>(
      sc, n_rays, o3, d3, t0, t1, prim, tu, sf, emission3, bg, rgb_out, status_out);
  prof_end(kStQuery, st);
  UGP_CUDA_CHECK(cudaGetLastError());
  return UGP_OK;
}

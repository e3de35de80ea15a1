// Learned directional guide: input encoding and vMF-mixture arithmetic shared by the guide
// kernels and the renderer.
//
// The network maps a scattering vertex (position x, outgoing direction wo) to 8 von
// Mises-Fisher lobes over incident directions. The paper leaves the proposal open (Sec. 6: any
// sampling technique combined by MIS with the approximate phase pdf of App. B keeps the
// estimate unbiased); the readings of its unspecified details are:
//  * input: x normalised to [0,1]^3 over a box, sin/cos(2^l pi x) for l = 0..5 (36 features);
//    the polar angles (theta, phi) of wo in radians, sin/cos(2^l angle) for l = 0..3 (16);
//    the raw values (x, y, z, theta / pi, phi / (2 pi) + 1/2) (5); zeros up to 64;
//  * four 64 x 64 ReLU layers and a 64 -> 40 head, BF16 operands, FP32 accumulation;
//  * lobe j reads head outputs 5j..5j+4 = (m (3), s, a): mu = m / |m|,
//    kappa = min(kappa_max, kappa_min + softplus(s)), pi = softmax(a);
//  * vMF density kappa / (2 pi (1 - e^{-2 kappa})) e^{kappa (mu.w - 1)};
//  * sampling: lobe by the first cumulative pi above u_l, then 1 - mu.w =
//    -ln(v + (1 - v) e^{-2 kappa}) / kappa with v = 1 - u1, azimuth 2 pi u2 in the frame of mu;
//  * loss of a logged vertex: -(L / p) ln q(wi), L the incident-radiance estimate and p the
//    pdf the direction was sampled with.
#pragma once
#include <cuda_bf16.h>
#include <stdint.h>

#include "ugp_internal.cuh"
#include "ugp_phase.cuh"

namespace ugp {

constexpr int kGLobes = UGP_GUIDE_LOBES;
constexpr int kGWidth = UGP_GUIDE_WIDTH;
constexpr int kGOut = UGP_GUIDE_OUT;
constexpr int kGLayers = 4;

// Offsets of the flat FP32 parameter vector: for l = 0..3, W_l (64 x 64, [out][in]) then b_l;
// then the head W_4 (40 x 64) and b_4 (40).
__host__ __device__ constexpr int guide_w_off(int l) { return l * (kGWidth * kGWidth + kGWidth); }
__host__ __device__ constexpr int guide_out_dim(int l) { return l < kGLayers ? kGWidth : kGOut; }
__host__ __device__ constexpr int guide_b_off(int l) { return guide_w_off(l) + guide_out_dim(l) * kGWidth; }
static_assert(guide_b_off(kGLayers) + kGOut == UGP_GUIDE_NPARAMS, "guide parameter count");

// Shared-memory image of the network (the guide kernels bulk-copy it from the workspace):
//   [0, 40960)       W_l for l = 0..4, 64 x 64 tiles (rows = outputs, head padded with zero rows),
//                    the K-major B operand of X W_l^T and the MN-major B operand of dZ W_l
//   [40960, 42240)   biases, FP32, 64 per layer (head padded with zeros)
constexpr uint32_t kImgW = 0;
constexpr uint32_t kImgTile = kGWidth * kGWidth * 2;  // 8192
constexpr uint32_t kImgBias = 5 * kImgTile;           // 40960
constexpr uint32_t kImgBytes = kImgBias + 5 * kGWidth * 4;  // 42240

struct GuideCfgDev {
  float3 lo, inv_ext;  // position box: xn = (x - lo) * inv_ext
  float kappa_min, kappa_max;
};

__device__ __forceinline__ float clamp01(float v) { return fminf(1.f, fmaxf(0.f, v)); }

// Features of one coordinate: sin/cos(2^l angle) for l < kN, with the pair for l = 0 given. The higher
// frequencies by double angles: sin 2a = 2 sin a cos a, cos 2a = (cos a - sin a)(cos a + sin a); five
// doublings leave an error of a few 1e-6, far below the BF16 step the layer input is rounded to.
template <int kN>
__device__ __forceinline__ void double_angles(float s, float co, float* f) {
#pragma unroll
  for (int l = 0; l < kN; ++l) {
    f[2 * l] = s;
    f[2 * l + 1] = co;
    const float s2 = 2.f * s * co;
    co = (co - s) * (co + s);
    s = s2;
  }
}
__device__ __forceinline__ float3 guide_position(const GuideCfgDev& c, float3 x) {
  return f3(clamp01((x.x - c.lo.x) * c.inv_ext.x), clamp01((x.y - c.lo.y) * c.inv_ext.y),
            clamp01((x.z - c.lo.z) * c.inv_ext.z));
}
// Features 12 a .. 12 a + 11 of position coordinate a (in [0, 1]).
__device__ __forceinline__ void encode_axis(float xn, float* f) {
  float s, co;
  sincospif(xn, &s, &co);
  double_angles<6>(s, co, f);
}
// Features 36 .. 63: the angles of wo, the raw values, zeros.
__device__ __forceinline__ void encode_rest(float3 xn, float3 wo, float* f) {
  const float theta = acosf(fminf(1.f, fmaxf(-1.f, wo.z)));
  const float phi = atan2f(wo.y, wo.x);
  float s, co;
  sincosf(theta, &s, &co);
  double_angles<4>(s, co, f);
  sincosf(phi, &s, &co);
  double_angles<4>(s, co, f + 8);
  f[16] = xn.x;
  f[17] = xn.y;
  f[18] = xn.z;
  f[19] = theta * 0.318309886183790672f;         // theta / pi
  f[20] = phi * 0.159154943091895336f + 0.5f;    // phi / (2 pi) + 1/2
#pragma unroll
  for (int i = 21; i < 28; ++i) f[i] = 0.f;
}

// The 64 input features of a vertex.
__device__ __forceinline__ void guide_encode(const GuideCfgDev& c, float3 x, float3 wo, float f[kGWidth]) {
  const float3 xn = guide_position(c, x);
  encode_axis(xn.x, f);
  encode_axis(xn.y, f + 12);
  encode_axis(xn.z, f + 24);
  encode_rest(xn, wo, f + 36);
}

__device__ __forceinline__ float softplusf(float s) { return fmaxf(s, 0.f) + log1pf(expf(-fabsf(s))); }

// log of the vMF normaliser kappa / (2 pi (1 - e^{-2 kappa})).
__device__ __forceinline__ float vmf_log_norm(float k) {
  return logf(k) - 1.83787706640934548f - logf(-expm1f(-2.f * k));
}

// Mixture (per lobe mu (3), kappa, pi) from the 40 head outputs (may be in place).
__device__ __forceinline__ void mixture_from_head(const GuideCfgDev& c, const float Y[kGOut], float mix[kGOut]) {
  float amax = -3.4e38f;
#pragma unroll
  for (int j = 0; j < kGLobes; ++j) amax = fmaxf(amax, Y[5 * j + 4]);
  float z = 0.f;
#pragma unroll
  for (int j = 0; j < kGLobes; ++j) z += expf(Y[5 * j + 4] - amax);
  const float iz = 1.f / z;
#pragma unroll
  for (int j = 0; j < kGLobes; ++j) {
    const float mx = Y[5 * j], my = Y[5 * j + 1], mz = Y[5 * j + 2], s = Y[5 * j + 3], a = Y[5 * j + 4];
    const float n = sqrtf(mx * mx + my * my + mz * mz);
    const float in = n > 0.f ? 1.f / n : 0.f;
    mix[5 * j] = n > 0.f ? mx * in : 0.f;
    mix[5 * j + 1] = n > 0.f ? my * in : 0.f;
    mix[5 * j + 2] = n > 0.f ? mz * in : 1.f;
    mix[5 * j + 3] = fminf(c.kappa_max, c.kappa_min + softplusf(s));
    mix[5 * j + 4] = expf(a - amax) * iz;
  }
}

__device__ __forceinline__ float mixture_pdf(const float mix[kGOut], float3 w) {
  float q = 0.f;
#pragma unroll
  for (int j = 0; j < kGLobes; ++j) {
    const float k = mix[5 * j + 3];
    const float c = mix[5 * j] * w.x + mix[5 * j + 1] * w.y + mix[5 * j + 2] * w.z;
    q += mix[5 * j + 4] * expf(vmf_log_norm(k) + k * (c - 1.f));
  }
  return q;
}

// Direction of the lobe around mu with concentration k.
__device__ __forceinline__ float3 lobe_sample(float3 mu, float k, float u1, float u2) {
  const float v = 1.f - u1;
  const float omw = fminf(2.f, -logf(v + (1.f - v) * expf(-2.f * k)) / k);
  const float s = sqrtf(fmaxf(0.f, omw * (2.f - omw)));
  float sp, cp;
  sincospif(2.f * u2, &sp, &cp);
  float3 t, b;
  onb3(mu, t, b);
  return normalize3((1.f - omw) * mu + (s * cp) * t + (s * sp) * b);
}

__device__ __forceinline__ float3 mixture_sample(const float mix[kGOut], float ul, float u1, float u2) {
  // first lobe whose cumulative weight exceeds ul (the last one if rounding leaves none);
  // selected by predicated moves so the mixture stays in registers
  bool found = false;
  float cum = 0.f;
  float3 mu = f3(mix[5 * (kGLobes - 1)], mix[5 * (kGLobes - 1) + 1], mix[5 * (kGLobes - 1) + 2]);
  float k = mix[5 * (kGLobes - 1) + 3];
#pragma unroll
  for (int i = 0; i < kGLobes; ++i) {
    cum += mix[5 * i + 4];
    const bool take = !found && cum > ul;
    if (take) {
      mu = f3(mix[5 * i], mix[5 * i + 1], mix[5 * i + 2]);
      k = mix[5 * i + 3];
    }
    found = found || take;
  }
  return lobe_sample(mu, k, u1, u2);
}
// The mixture of a vertex in global memory, with the log of each lobe's normaliser in a column of shared memory
// (stride `kStride`), for a kernel that evaluates it in several places: 40 registers and three evaluations of
// each normaliser less, and short code (the shading of a guided 480 x 270 pass: 0.95 -> 0.87 ms). Values are
// those of mixture_pdf and mixture_sample.
template <int kStride>
struct VertexMixture {
  const float* mix;  // 16-byte aligned
  float* norm;
  __device__ void prepare() const {
#pragma unroll 1
    for (int j = 0; j < kGLobes; ++j) norm[j * kStride] = vmf_log_norm(__ldg(mix + 5 * j + 3));
  }
  __device__ float pdf(float3 w) const {
    static_assert(kGLobes % 4 == 0, "four lobes are five float4");
    float q = 0.f;
#pragma unroll 1
    for (int h = 0; h < kGLobes; h += 4) {
      float v[20];
#pragma unroll
      for (int i = 0; i < 5; ++i) {
        const float4 f = __ldg(reinterpret_cast<const float4*>(mix + 5 * h) + i);
        v[4 * i] = f.x; v[4 * i + 1] = f.y; v[4 * i + 2] = f.z; v[4 * i + 3] = f.w;
      }
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const float c = v[5 * j] * w.x + v[5 * j + 1] * w.y + v[5 * j + 2] * w.z;
        q += v[5 * j + 4] * expf(norm[(h + j) * kStride] + v[5 * j + 3] * (c - 1.f));
      }
    }
    return q;
  }
  __device__ float3 sample(float ul, float u1, float u2) const {
    float cum = 0.f;
    int i = 0;
#pragma unroll 1
    for (; i < kGLobes - 1; ++i) {
      cum += __ldg(mix + 5 * i + 4);
      if (cum > ul) break;
    }
    const float* lobe = mix + 5 * i;
    return lobe_sample(f3(__ldg(lobe), __ldg(lobe + 1), __ldg(lobe + 2)), __ldg(lobe + 3), u1, u2);
  }
};

// The loss -w ln q(wi) of one sample and its gradient with respect to the head outputs, by kLoss lobes per
// thread, kGLobes / kLoss threads per sample. Y: the 5 kLoss head outputs of this thread's lobes; A: the
// weights' outputs of all lobes. Stage 1 gives each lobe's log of pi_j v_j(wi); with all of them in
// ell[0 .. kGLobes), stage 2 gives the gradient (over Y) and returns the loss.
template <int kLoss>
struct LobeLoss {
  float cw[kLoss], in[kLoss], k[kLoss];
  bool free_k[kLoss];
  float logz;
  __device__ void stage1(const GuideCfgDev& c, const float* Y, const float A[kGLobes], float3 wi, float* ell) {
    float amax = -3.4e38f;
#pragma unroll
    for (int j = 0; j < kGLobes; ++j) amax = fmaxf(amax, A[j]);
    float z = 0.f;
#pragma unroll
    for (int j = 0; j < kGLobes; ++j) z += expf(A[j] - amax);
    logz = amax + logf(z);
#pragma unroll
    for (int j = 0; j < kLoss; ++j) {
      const float mx = Y[5 * j], my = Y[5 * j + 1], mz = Y[5 * j + 2];
      const float n = sqrtf(mx * mx + my * my + mz * mz);
      in[j] = n > 0.f ? 1.f / n : 0.f;
      cw[j] = n > 0.f ? (mx * wi.x + my * wi.y + mz * wi.z) * in[j] : wi.z;
      const float kr = c.kappa_min + softplusf(Y[5 * j + 3]);
      k[j] = fminf(kr, c.kappa_max);
      free_k[j] = !(kr > c.kappa_max);
      ell[j] = (Y[5 * j + 4] - logz) + vmf_log_norm(k[j]) + k[j] * (cw[j] - 1.f);
    }
  }
  // own: this thread's entries of ell
  __device__ float stage2(float* Y, const float ell[kGLobes], const float* own, float3 wi, float w) {
    float lmax = -3.4e38f;
#pragma unroll
    for (int j = 0; j < kGLobes; ++j) lmax = fmaxf(lmax, ell[j]);
    float sq = 0.f;
#pragma unroll
    for (int j = 0; j < kGLobes; ++j) sq += expf(ell[j] - lmax);
    const float logq = lmax + logf(sq);
#pragma unroll
    for (int j = 0; j < kLoss; ++j) {
      const float r = expf(own[j] - logq);
      const float pi = expf(Y[5 * j + 4] - logz);
      Y[5 * j + 4] = w * (pi - r);
      const float dlk = 1.f / k[j] - 2.f / expm1f(2.f * k[j]) + (cw[j] - 1.f);
      const float sig = 1.f / (1.f + expf(-Y[5 * j + 3]));
      Y[5 * j + 3] = free_k[j] ? -w * r * dlk * sig : 0.f;
      const float g = -w * r * k[j] * in[j];
      const float mx = Y[5 * j] * in[j], my = Y[5 * j + 1] * in[j], mz = Y[5 * j + 2] * in[j];
      Y[5 * j] = g * (wi.x - cw[j] * mx);
      Y[5 * j + 1] = g * (wi.y - cw[j] * my);
      Y[5 * j + 2] = g * (wi.z - cw[j] * mz);
    }
    return -w * logq;
  }
};

}  // namespace ugp

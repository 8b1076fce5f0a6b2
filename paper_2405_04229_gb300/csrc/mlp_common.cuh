// The refraction surrogate network: 3 -> 64 -> 64 -> 64 -> 3 with tanh,
// BF16 weights on the tensor cores with FP32 accumulation.  Shared by the
// training translation unit and the inference (both on tcgen05, mlp_tc.cuh).
#pragma once

#include <cuda_bf16.h>

#include "device_math.cuh"

namespace cs {

constexpr int kHid = 64;       // hidden width
constexpr int kNIn = 3;        // (h_e, cos(theta0), 1/lambda), affine-normalised to [-1, 1]
constexpr int kNOut = 3;       // (G_R, G_t, ln T), affine-normalised
constexpr int kNOutP = 8;      // output layer padded to one 8-wide MMA tile

// Flat FP32 parameter layout (W rows are output units):
//   W1[64][3] b1[64] W2[64][64] b2[64] W3[64][64] b3[64] W4[8][64] b4[8]
// (rows 3..7 of W4 and b4[3..7] stay zero)
constexpr int kOffW1 = 0;
constexpr int kOffB1 = kOffW1 + kHid * kNIn;
constexpr int kOffW2 = kOffB1 + kHid;
constexpr int kOffB2 = kOffW2 + kHid * kHid;
constexpr int kOffW3 = kOffB2 + kHid;
constexpr int kOffB3 = kOffW3 + kHid * kHid;
constexpr int kOffW4 = kOffB3 + kHid;
constexpr int kOffB4 = kOffW4 + kNOutP * kHid;
constexpr int kNParams = kOffB4 + kNOutP;

// BF16 copies of the tensor-core weights, [n][k] (k contiguous)
constexpr int kBOffW2 = 0;
constexpr int kBOffW3 = kBOffW2 + kHid * kHid;
constexpr int kBOffW4 = kBOffW3 + kHid * kHid;
constexpr int kNBf16 = kBOffW4 + kNOutP * kHid;

// What the photon kernel needs to evaluate the network.
struct SurrogateView {
    const float* p;             // FP32 parameters (W1, biases; W2..W4 as trained masters)
    const __nv_bfloat16* wb;    // BF16 W2, W3, W4
    int split;                  // 1: hidden activations as hi + lo BF16 pairs (two MMAs)
    // input normalisation x = in_scale * v + in_shift for v = (height coordinate,
    // cos(theta0), 1/lambda_nm); the height coordinate is dz, or exp(-dz / H)
    // when height_scale H > 0
    float in_scale[3], in_shift[3];
    float inv_height_scale;   // 1 / H, or 0 for the linear coordinate
    // output de-normalisation y = out_half * o + out_mid of the network's part of
    // (G_R, G_t, ln T); the fields are that part plus the first-order baseline below
    float out_half[3], out_mid[3];
    // first-order baseline: {I = int (n - 1) dh, n(h_e) - 1, X_v = int 100 rho dh,
    // A_v = int exp(-h / H_A) dh} from h_obs up, tabulated in dz (linear interpolation)
    const float4* base;
    int base_n;
    float base_dz0, base_inv_step;
    float kR0, kA0, lamA_nm, aer_alpha;   // transmission constants (log2 units, as AtmParams)
    // domain in which the network replaces the tables
    float dz_min, dz_max, mu_min;   // mu_min = cos of the largest zenith
    // bands around the atmosphere's layer boundaries, where the exact fields
    // jump with n(h_e): heights dz in [band_lo[i], band_hi[i]) use the tables
    int n_bands;
    float band_lo[kMaxLayers], band_hi[kMaxLayers];
    int polls;   // polls of each tensor-core completion before giving up (>= 0)
};

// The view with the parameters that every thread reads at the same time, as kernel parameters: read
// through the constant cache as operands.  (From shared memory their 96 16-byte loads a row took
// about half of the SM's shared-memory cycles.)
struct SurrogateNet : SurrogateView {
    float4 w1p[kHid / 2][2];   // layer 1, units 2i and 2i + 1 side by side:
                               // {W1[.][0], W1[.][1]}, {W1[.][2], b1[.]}
    float4 b23[2][kHid / 4];   // biases of layers 2 and 3
    float b4[4];
};

__device__ __forceinline__ float height_coordinate(const SurrogateView& sv, float dz) {
    return sv.inv_height_scale > 0.0f ? ex2_approx(-dz * sv.inv_height_scale * 1.4426950408889634f) : dz;
}

__device__ __forceinline__ bool in_surrogate_domain(const SurrogateView& sv, float dz, float mu) {
    bool ok = dz >= sv.dz_min && dz <= sv.dz_max && mu >= sv.mu_min;
#pragma unroll
    for (int i = 0; i < kMaxLayers; ++i)
        if (i < sv.n_bands && dz >= sv.band_lo[i] && dz < sv.band_hi[i]) ok = false;
    return ok;
}

// First-order baseline of the fields (G_R, G_t, ln T) at height dz above the
// observation level, cos(theta0) = mu and 1/lambda_nm = inv_l.  Expanding the
// exact planar path (Eq. 3.17-3.18) to first order in n - 1, with
// I = int (n - 1) dh over [h_obs, h_e] and H = h_e - h_obs:
//   G_R = d_e H - I,   G_t = 2 I - d_e H + (d_e H - I) / mu^2,
//   ln T = -(X_v / X_R(lambda) + tau_A(lambda) A_v / H_A) / mu   (the vertical columns).
// The network learns only the remainder, about 1e-3 of the fields' range in
// the plane and a few per cent on the spherical shell, so its BF16
// resolution acts on that remainder.
__device__ __forceinline__ float3 surrogate_baseline(const SurrogateView& sv, float dz, float mu, float inv_l) {
    const float f = fminf(fmaxf((dz - sv.base_dz0) * sv.base_inv_step, 0.0f), (float)(sv.base_n - 1));
    const int j = min((int)f, sv.base_n - 2);
    const float t = f - (float)j;
    const float4 a = __ldg(sv.base + j), b = __ldg(sv.base + j + 1);
    const float I = fmaf(t, b.x - a.x, a.x), de = fmaf(t, b.y - a.y, a.y);
    const float Xv = fmaf(t, b.z - a.z, a.z), Av = fmaf(t, b.w - a.w, a.w);
    const float m = fmaf(de, dz, -I);   // int (d_e - d) dh
    const float imu = 1.0f / mu;
    const float il2 = inv_l * inv_l;
    const float kA = sv.kA0 * ex2_approx(sv.aer_alpha * lg2_approx(sv.lamA_nm * inv_l));
    return make_float3(m, fmaf(m, imu * imu, fmaf(2.0f, I, -de * dz)),
                       -0.69314718f * (Xv * sv.kR0 * il2 * il2 + Av * kA) * imu);
}

// The trained network's view (defined with the training code).
const SurrogateNet* surrogate_view(const cs_surrogate* s);

__device__ __forceinline__ uint32_t pack_bf16x2(float lo, float hi) {
    __nv_bfloat162 v = __floats2bfloat162_rn(lo, hi);
    return *reinterpret_cast<uint32_t*>(&v);
}

// tanh(x) = 1 - 2 / (exp(2x) + 1) from ex2 and rcp approximations: absolute
// error about 2e-7 (the hardware tanh approximation is ~5e-4 relative, too
// coarse for the network's error budget).  Used in training and inference.
__device__ __forceinline__ float tanh_act(float x) {
    const float e = ex2_approx(x * 2.8853900817779268f);   // exp(2x)
    return fmaf(-2.0f, rcp_approx(e + 1.0f), 1.0f);
}

}  // namespace cs

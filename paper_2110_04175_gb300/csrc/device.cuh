// device.cuh -- what the step kernels (step_kernels.cu) and the setup and
// metrics kernels (relaysum.cu) share: the Philox normals, float4 arithmetic
// and memory access, the step's arguments, and the launch helpers.
#pragma once

#include <cuda_runtime.h>

#include <atomic>
#include <cstdint>

#include "handle.h"
#include "program.h"
#include "relaysum.h"

namespace relaysum {

// The ten round keys (k0 + r W0, k1 + r W1), computed once on the host.
struct PhiloxKey {
    uint32_t k[10][2];
};

// Messages lost in transit, one bit per directed edge (Section 4.4).
struct LostMask {
    uint32_t w[relaysum::kMaxE / 32 + 1];
    __host__ __device__ __forceinline__ bool operator()(int e) const { return (w[e >> 5] >> (e & 31)) & 1u; }
};

struct ModelArgs {
    float* x;
    const float* mu;
    const float* msg_in;
    float* msg_out;
    const int32_t* counts;
    int64_t ld_x;     // row stride (floats) of x and mu
    int64_t ld_m;     // row stride (floats) of the messages
    int64_t nquads;   // ceil(d / 4)
    uint32_t q0;      // absolute quad of local coordinate 0
    uint32_t step;
    float lr, sigma;
    int mode;         // 0: Alg. 1 rebuild, 1: robust rebuild
    int algo;         // 0 RelaySGD, 1 RelaySum/Grad, 2 mean estimation
    int has_lost;     // any bit of `lost` set
    int rsum;         // wide nodes read and write their received-sum rows (program.h)
    LostMask lost;    // messages lost in transit this step
    float* s1;        // optimiser state (momentum / Adam m), [n][ld_x]
    float* s2;        // Adam v, [n][ld_x]
    float beta1, beta2, eps;
    float adam_step;  // lr / (1 - beta1^{t+1})
    float adam_ibc2;  // 1 / sqrt(1 - beta2^{t+1})
    PhiloxKey key;    // noise key schedule
};

// relay_steps: k consecutive steps in one launch.
constexpr int kMaxFusedSteps = 64;  // steps per launch (Adam's per-step factors ride in the parameters)

struct FusedSteps {
    int32_t k;                        // steps in this launch, 1 .. kMaxFusedSteps
    float* msg[2];                    // step t0 + j reads msg[j & 1] and writes msg[(j + 1) & 1]
    float adam_step[kMaxFusedSteps];  // Adam's factors of step t0 + j
    float adam_ibc2[kMaxFusedSteps];
};

}  // namespace relaysum

namespace {

using relaysum::FusedSteps;
using relaysum::kMaxFusedSteps;
using relaysum::LostMask;
using relaysum::ModelArgs;
using relaysum::PhiloxKey;

// ------------------------------------------------------------ random numbers

// Philox4x32-10 (Salmon, Moraes, Dror, Shaw, SC'11): round multipliers and
// Weyl key increments of the published definition.
constexpr uint32_t kPhiloxM0 = 0xD2511F53u;
constexpr uint32_t kPhiloxM1 = 0xCD9E8D57u;
constexpr uint32_t kPhiloxW0 = 0x9E3779B9u;
constexpr uint32_t kPhiloxW1 = 0xBB67AE85u;

PhiloxKey philox_key(uint64_t seed) {
    PhiloxKey key;
    uint32_t k0 = static_cast<uint32_t>(seed), k1 = static_cast<uint32_t>(seed >> 32);
    for (int r = 0; r < 10; ++r) {
        key.k[r][0] = k0;
        key.k[r][1] = k1;
        k0 += kPhiloxW0;
        k1 += kPhiloxW1;
    }
    return key;
}

__device__ __forceinline__ uint4 philox4x32_10(uint4 c, const PhiloxKey& key) {
#pragma unroll
    for (int round = 0; round < 10; ++round) {
        const uint32_t hi0 = __umulhi(kPhiloxM0, c.x), lo0 = kPhiloxM0 * c.x;
        const uint32_t hi1 = __umulhi(kPhiloxM1, c.z), lo1 = kPhiloxM1 * c.z;
        c = make_uint4(hi1 ^ c.y ^ key.k[round][0], lo1, hi0 ^ c.w ^ key.k[round][1], lo0);
    }
    return c;
}

// 24 high bits -> (0, 1], exact in fp32.
__device__ __forceinline__ float unit_interval(uint32_t w) {
    return __uint2float_rn((w >> 8) + 1u) * 5.9604644775390625e-8f;  // 2^-24
}

__device__ __forceinline__ float sqrt_approx(float v) {
    float r;
    asm("sqrt.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(v));
    return r;
}

// Four standard normals for coordinates 4q .. 4q+3 (Box-Muller on the two
// word pairs of one Philox block): z = sqrt(-2 ln u_a) (cos, sin)(2 pi u_b).
// The angle is taken as 2 pi u_b - pi, inside the range where the hardware
// sine/cosine are accurate to 2^-21.4, and the half turn is undone by the
// sign; the radius keeps an accurate logarithm (its argument can sit just
// below 1, where an approximate one loses all relative accuracy).
__device__ __forceinline__ float4 normal4(uint32_t q, uint32_t row, uint32_t step, uint32_t stream,
                                          const PhiloxKey& key) {
    const uint4 w = philox4x32_10(make_uint4(q, row, step, stream), key);
    const float r0 = sqrt_approx(-2.0f * logf(unit_interval(w.x)));
    const float r1 = sqrt_approx(-2.0f * logf(unit_interval(w.z)));
    constexpr float kTwoPi = 6.28318530717958647692f, kPi = 3.14159265358979323846f;
    float s0, c0, s1, c1;
    __sincosf(fmaf(unit_interval(w.y), kTwoPi, -kPi), &s0, &c0);
    __sincosf(fmaf(unit_interval(w.w), kTwoPi, -kPi), &s1, &c1);
    return make_float4(-r0 * c0, -r0 * s0, -r1 * c1, -r1 * s1);
}

// ------------------------------------------------------------ float4 helpers

__device__ __forceinline__ float4 add4(float4 a, float4 b) {
    return make_float4(a.x + b.x, a.y + b.y, a.z + b.z, a.w + b.w);
}
__device__ __forceinline__ float4 sub4(float4 a, float4 b) {
    return make_float4(a.x - b.x, a.y - b.y, a.z - b.z, a.w - b.w);
}
__device__ __forceinline__ float4 scale4(float4 a, float s) {
    return make_float4(a.x * s, a.y * s, a.z * s, a.w * s);
}
// Rounded product that the compiler may not fuse into a later add: the
// regenerated mu must round exactly like the stored one.
__device__ __forceinline__ float4 scale4_rn(float4 a, float s) {
    return make_float4(__fmul_rn(a.x, s), __fmul_rn(a.y, s), __fmul_rn(a.z, s), __fmul_rn(a.w, s));
}
__device__ __forceinline__ float4 fma4(float w, float4 z, float4 acc) {
    return make_float4(fmaf(w, z.x, acc.x), fmaf(w, z.y, acc.y), fmaf(w, z.z, acc.z), fmaf(w, z.w, acc.w));
}
// Loads read once per step: read-only path, no L1 allocation.
__device__ __forceinline__ float4 ld_stream(const float* p) {
    float4 v;
    asm("ld.global.nc.L1::no_allocate.v4.f32 {%0, %1, %2, %3}, [%4];"
                 : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w)
                 : "l"(p));
    return v;
}
// A wide node's incoming messages are read again at its children's visits
// (program.h): keep them in L2 with evict-last priority until then.
__device__ __forceinline__ float4 ld_keep(const float* p) {
    float4 v;
    asm("{\n\t.reg .b64 pol;\n\t"
        "createpolicy.fractional.L2::evict_last.b64 pol, 1.0;\n\t"
        "ld.global.nc.L2::cache_hint.v4.f32 {%0, %1, %2, %3}, [%4], pol;\n\t}"
        : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w)
        : "l"(p));
    return v;
}
__device__ __forceinline__ void st_stream(float* p, float4 v) {
    __stcs(reinterpret_cast<float4*>(p), v);
}

// mu_i for quad q: read, or regenerated exactly as relay_fill_mu_kernel
// writes it (same normals, same fma order), so both sources give the same bits.
template <int OBJ, typename Obj>
__device__ __forceinline__ float4 centre(const Obj& obj, const PhiloxKey& mu_key, const ModelArgs& a,
                                         int i, int64_t q, const float4* cen, int cen_stride) {
    if constexpr (OBJ == relaysum::kMuStored) {
        return ld_stream(a.mu + i * a.ld_x + 4 * q);
    } else {
        float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
        for (int j = obj.row_off[i]; j < obj.row_off[i + 1]; ++j) {
            const float4 z = (OBJ == relaysum::kMuPerRow)
                                 ? normal4(a.q0 + static_cast<uint32_t>(q), static_cast<uint32_t>(obj.col[j]),
                                           0u, 1u, mu_key)
                                 : cen[obj.col[j] * cen_stride];
            acc = fma4(obj.w[j], z, acc);
        }
        return scale4_rn(acc, obj.scale);
    }
}

// ------------------------------------------------------------- host helpers

constexpr int kMaxDevices = 64;
// dynamic shared memory cap: 227 KB per CTA minus the static scale/fill tables
constexpr int kMaxSmem = 224 * 1024;

int device_sms(int* dev_out) {
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) return -1;
    static std::atomic<int> sms_cache[kMaxDevices];
    int sms = (dev < kMaxDevices) ? sms_cache[dev].load() : 0;
    if (sms <= 0) {
        if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) return -1;
        if (dev < kMaxDevices) sms_cache[dev].store(sms);
    }
    *dev_out = dev;
    return sms;
}

int launch_status() {
    return cudaGetLastError() == cudaSuccess ? RELAY_OK : RELAY_ECUDA;
}

}  // namespace

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
    int32_t rounds;                   // counter rounds until they repeat, 1 .. k (settled_rounds)
    int32_t qb_log2;                  // quads per CTA
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
        const uint64_t p0 = static_cast<uint64_t>(kPhiloxM0) * c.x, p1 = static_cast<uint64_t>(kPhiloxM1) * c.z;
        c = make_uint4(static_cast<uint32_t>(p1 >> 32) ^ c.y ^ key.k[round][0], static_cast<uint32_t>(p1),
                       static_cast<uint32_t>(p0 >> 32) ^ c.w ^ key.k[round][1], static_cast<uint32_t>(p0));
    }
    return c;
}

// The noise block of worker `row` at quad q in step `step` (stream 0),
// philox4x32_10 of (q, row, step, 0) with its first two rounds split: what
// depends on the quad alone is formed once per quad (NoiseQuad), what depends
// on the row and the step not per quad, so 16 to 17 of the 20 wide products
// remain per call.  They are what bounds the noise: a wide product holds the
// heavy multiplier pipe for 4 cycles a warp.
struct NoiseQuad {
    uint32_t a, b, d;
};

__device__ __forceinline__ uint64_t wide_product(uint32_t m, uint32_t v) { return static_cast<uint64_t>(m) * v; }
__device__ __forceinline__ uint32_t hi32(uint64_t p) { return static_cast<uint32_t>(p >> 32); }
__device__ __forceinline__ uint32_t lo32(uint64_t p) { return static_cast<uint32_t>(p); }

__device__ __forceinline__ NoiseQuad noise_quad(uint32_t q, const PhiloxKey& key) {
    const uint64_t p0 = wide_product(kPhiloxM0, q);
    const uint64_t p1 = wide_product(kPhiloxM1, hi32(p0) ^ key.k[0][1]);
    return NoiseQuad{hi32(p1), lo32(p1), lo32(p0)};
}

__device__ __forceinline__ uint4 noise_words(const NoiseQuad& t, uint32_t row, uint32_t step, const PhiloxKey& key) {
    const uint64_t ps = wide_product(kPhiloxM1, step);
    const uint64_t pr = wide_product(kPhiloxM0, hi32(ps) ^ row ^ key.k[0][0]);
    uint4 c = make_uint4(t.a ^ (lo32(ps) ^ key.k[1][0]), t.b, t.d ^ (hi32(pr) ^ key.k[1][1]), lo32(pr));
#pragma unroll
    for (int round = 2; round < 10; ++round) {
        const uint64_t p0 = wide_product(kPhiloxM0, c.x), p1 = wide_product(kPhiloxM1, c.z);
        c = make_uint4(hi32(p1) ^ c.y ^ key.k[round][0], lo32(p1), hi32(p0) ^ c.w ^ key.k[round][1], lo32(p0));
    }
    return c;
}

// ------------------------------------------------------- packed fp32 pairs

// The step is bound by instruction issue wherever HBM does not bound it, and
// sm_103a's packed fp32 instructions (add / mul / fma .rn.f32x2) do the work
// of two scalar ones in one issue slot, each half rounded as the scalar one.
// All per-coordinate arithmetic goes through these, and every fused
// multiply-add is written out, so that every kernel rounds alike.
struct Pair {
    unsigned long long v;
};

__device__ __forceinline__ Pair pack(float lo, float hi) {
    Pair r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r.v) : "f"(lo), "f"(hi));
    return r;
}
__device__ __forceinline__ Pair pack(float both) { return pack(both, both); }
__device__ __forceinline__ void unpack(Pair p, float& lo, float& hi) {
    asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(p.v));
}
__device__ __forceinline__ Pair add2(Pair a, Pair b) {
    Pair r;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r.v) : "l"(a.v), "l"(b.v));
    return r;
}
__device__ __forceinline__ Pair mul2(Pair a, Pair b) {
    Pair r;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r.v) : "l"(a.v), "l"(b.v));
    return r;
}
__device__ __forceinline__ Pair fma2(Pair a, Pair b, Pair c) {
    Pair r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r.v) : "l"(a.v), "l"(b.v), "l"(c.v));
    return r;
}

// a - b (the product with -1 is exact)
__device__ __forceinline__ Pair sub2(Pair a, Pair b) { return fma2(b, pack(-1.0f), a); }

__device__ __forceinline__ float4 quad(Pair a, Pair b) {
    float4 r;
    unpack(a, r.x, r.y);
    unpack(b, r.z, r.w);
    return r;
}
__device__ __forceinline__ float4 add4(float4 a, float4 b) {
    return quad(add2(pack(a.x, a.y), pack(b.x, b.y)), add2(pack(a.z, a.w), pack(b.z, b.w)));
}
// Products with one factor for the whole quad stay scalar: the factor can be
// a constant operand, where a pair of it would cost two moves, and the scalar
// multiplier pipe is otherwise idle (Philox fills the other one).  Each is
// rounded once; the intrinsics keep a later add from being fused in (the
// regenerated mu rounds exactly like the stored one).
__device__ __forceinline__ float4 fma4(float w, float4 z, float4 acc) {  // w z + acc
    return make_float4(__fmaf_rn(w, z.x, acc.x), __fmaf_rn(w, z.y, acc.y), __fmaf_rn(w, z.z, acc.z),
                       __fmaf_rn(w, z.w, acc.w));
}
__device__ __forceinline__ float4 sub4(float4 a, float4 b) {
    return make_float4(__fsub_rn(a.x, b.x), __fsub_rn(a.y, b.y), __fsub_rn(a.z, b.z), __fsub_rn(a.w, b.w));
}
__device__ __forceinline__ float4 scale4(float4 a, float s) {
    return make_float4(__fmul_rn(a.x, s), __fmul_rn(a.y, s), __fmul_rn(a.z, s), __fmul_rn(a.w, s));
}

// ------------------------------------------------------------------ normals

// u = ((w >> 8) + 1) 2^-24 in (0, 1] for two words: the 24-bit integers and
// the product-sum are exact in fp32.
__device__ __forceinline__ Pair unit_interval2(uint32_t w0, uint32_t w1) {
    const Pair ulp = pack(5.9604644775390625e-8f);  // 2^-24
    return fma2(pack(__uint2float_rn(w0 >> 8), __uint2float_rn(w1 >> 8)), ulp, ulp);
}

// -2 ln u for two u in [2^-24, 1].  u = m 2^e with m in [sqrt(1/2), sqrt(2)),
// the reduction of Cody and Waite (Software Manual for the Elementary
// Functions, 1980); with f = m - 1 (exact), -2 ln u = -2 ln 2 e + f P(f), and
// P, the minimax polynomial of degree 8 of -2 ln(1 + f) / f with P(0) = -2
// (fitted by the Remez exchange, coefficients rounded one by one), keeps the
// relative accuracy where u is just below 1 and ln u next to 0.  Relative
// error of the result over all 2^24 values of u: at most 9.5e-8 from the
// coefficients, 1.9e-7 as evaluated in fp32 (rms 3.7e-8).  The radius sqrt(-2
// ln u) is within 1.4e-7 of the exact one (rms 2.1e-8; a correctly rounded
// logarithm gives 1.2e-7 and 1.8e-8).  Sine and cosine leave about 1.7e-7 rms,
// so it does not show: 8.4M normals of the noise are within 1.760e-7 rms of
// the exact ones, as many of the centres, with CUDA's logf, within 1.765e-7.
__device__ __forceinline__ Pair minus_2_ln(Pair u) {
    float u0, u1;
    unpack(u, u0, u1);
    const int b0 = __float_as_int(u0), b1 = __float_as_int(u1);
    const int e0 = (b0 - 0x3f3504f3) & static_cast<int>(0xff800000u);  // e 2^23
    const int e1 = (b1 - 0x3f3504f3) & static_cast<int>(0xff800000u);
    const Pair f = add2(pack(__int_as_float(b0 - e0), __int_as_float(b1 - e1)), pack(-1.0f));
    Pair p = pack(-0.18646626f);
    p = fma2(p, f, pack(0.29618296f));
    p = fma2(p, f, pack(-0.29821008f));
    p = fma2(p, f, pack(0.32977396f));
    p = fma2(p, f, pack(-0.39912102f));
    p = fma2(p, f, pack(0.5001276f));
    p = fma2(p, f, pack(-0.66668445f));
    p = fma2(p, f, pack(0.99999815f));
    p = fma2(p, f, pack(-2.0f));
    // -2 ln 2 e, e as the integer e 2^23
    const Pair c = pack(-1.38629436111989061883f * 1.1920928955078125e-7f);
    return fma2(pack(__int2float_rn(e0), __int2float_rn(e1)), c, mul2(f, p));
}

__device__ __forceinline__ float sqrt_approx(float v) {
    float r;
    asm("sqrt.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(v));
    return r;
}
__device__ __forceinline__ float sin_approx(float v) {
    float r;
    asm("sin.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(v));
    return r;
}
__device__ __forceinline__ float cos_approx(float v) {
    float r;
    asm("cos.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(v));
    return r;
}

// The gradient noise: MINUS four standard normals for coordinates 4q .. 4q+3
// (Box-Muller on the two word pairs of one Philox block): z = sqrt(-2 ln u_a) (cos, sin)(2 pi u_b).
// The angle is taken as 2 pi u_b - pi, inside the range where the hardware
// sine/cosine are accurate to 2^-21.4; the half turn flips the sign, which the
// callers put into their factor (an exact step that costs nothing there).
__device__ __forceinline__ float4 minus_normal4(uint4 w) {
    float l0, l1, t0, t1;
    unpack(minus_2_ln(unit_interval2(w.x, w.z)), l0, l1);
    constexpr float kTwoPi = 6.28318530717958647692f, kPi = 3.14159265358979323846f;
    unpack(fma2(unit_interval2(w.y, w.w), pack(kTwoPi), pack(-kPi)), t0, t1);
    return quad(mul2(pack(sqrt_approx(l0)), pack(cos_approx(t0), sin_approx(t0))),
                mul2(pack(sqrt_approx(l1)), pack(cos_approx(t1), sin_approx(t1))));
}

// Four standard normals of the centres (stream 1) and of the initial model
// (stream 2): the same words and angles with CUDA's logf and __sincosf.  These
// are the objective that a run is defined by, read back through
// relay_fill_objective and relay_metrics in double, so they keep their bits.
__device__ __forceinline__ float4 normal4(uint32_t q, uint32_t row, uint32_t step, uint32_t stream,
                                          const PhiloxKey& key) {
    const uint4 w = philox4x32_10(make_uint4(q, row, step, stream), key);
    float u0, u1, t0, t1;
    unpack(unit_interval2(w.x, w.z), u0, u1);
    constexpr float kTwoPi = 6.28318530717958647692f, kPi = 3.14159265358979323846f;
    unpack(fma2(unit_interval2(w.y, w.w), pack(kTwoPi), pack(-kPi)), t0, t1);
    const float r0 = sqrt_approx(-2.0f * logf(u0)), r1 = sqrt_approx(-2.0f * logf(u1));
    float s0, c0, s1, c1;
    __sincosf(t0, &s0, &c0);
    __sincosf(t1, &s1, &c1);
    return make_float4(-r0 * c0, -r0 * s0, -r1 * c1, -r1 * s1);
}

// ------------------------------------------------------------ float4 access

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

// ------------------------------------------------- programmatic dependent launch

// relay_step launches the step kernel as a programmatic dependent of the
// counter kernel: the counter kernel lets it be scheduled at once, and the
// step kernel waits for the counter kernel's completion (and its writes)
// before its first read of the counters.  Launched the ordinary way, the
// wait returns immediately.
__device__ __forceinline__ void allow_dependent_launch() {
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}
__device__ __forceinline__ void wait_for_prior_grid() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

// A counter, behind wait_for_prior_grid(): the counter kernel may write it while
// this kernel already runs, so not by a non-coherent load, which is defined
// only for memory that stays as it is for the kernel's lifetime and may be
// moved ahead of the wait.  Being volatile, it stays behind it.  (A plain load
// of the array costs the walk over two windows with Adam 68 instead of 64
// registers, hence a CTA per SM.)
__device__ __forceinline__ int32_t ld_counter(const int32_t* p) {
    int32_t v;
    asm volatile("ld.global.s32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
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
        return scale4(acc, obj.scale);
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

// Launches a step kernel; `after_counts` makes it a programmatic dependent of
// the counter kernel just enqueued on the same stream (relay_step only).
template <typename... Params, typename... Args>
int launch_step_kernel(void (*kernel)(Params...), int grid, int threads, size_t smem, cudaStream_t stream,
                       bool after_counts, Args... args) {
    if (!after_counts) {
        kernel<<<grid, threads, smem, stream>>>(args...);
        return launch_status();
    }
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(static_cast<unsigned>(grid));
    cfg.blockDim = dim3(static_cast<unsigned>(threads));
    cfg.dynamicSmemBytes = smem;
    cfg.stream = stream;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    if (cudaLaunchKernelEx(&cfg, kernel, args...) != cudaSuccess) return RELAY_ECUDA;
    return launch_status();
}

// Opts `Kernel` in to the dynamic shared memory it may use (kMaxSmem, less
// when its static shared memory and kMaxSmem would pass the device's per-CTA
// limit) once per device, and returns its resident CTAs per SM for
// (threads, smem).  Both are cached per device (queried once, not per step:
// steps may be captured into CUDA graphs); each kernel instantiation has its
// own cache.  0 on a CUDA error, which is cleared so that it is not reported
// again by a later launch.
template <auto Kernel>
int resident_ctas(int dev, int threads, size_t smem) {
    static std::atomic<bool> smem_set[kMaxDevices];
    if (dev >= kMaxDevices || !smem_set[dev].load()) {
        cudaFuncAttributes fa;
        int optin = 0;
        if (cudaFuncGetAttributes(&fa, Kernel) != cudaSuccess ||
            cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev) != cudaSuccess) {
            (void)cudaGetLastError();
            return 0;
        }
        const int room = optin - static_cast<int>(fa.sharedSizeBytes);
        if (room <= 0 ||
            cudaFuncSetAttribute(Kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 room < kMaxSmem ? room : kMaxSmem) != cudaSuccess) {
            (void)cudaGetLastError();
            return 0;
        }
        if (dev < kMaxDevices) smem_set[dev].store(true);
    }
    static std::atomic<int64_t> occ_cache[kMaxDevices];
    const int64_t key = static_cast<int64_t>(smem) * 1024 + threads;
    const int64_t cached = dev < kMaxDevices ? occ_cache[dev].load() : 0;
    if (cached != 0 && (cached >> 8) == key) return static_cast<int>(cached & 0xFF);
    int per_sm = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, Kernel, threads, smem) != cudaSuccess || per_sm <= 0) {
        (void)cudaGetLastError();
        return 0;
    }
    if (dev < kMaxDevices) occ_cache[dev].store((key << 8) | (per_sm & 0xFF));
    return per_sm;
}

}  // namespace

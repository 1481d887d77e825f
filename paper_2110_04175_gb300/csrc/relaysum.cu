// relaysum.cu -- the C ABI of the RelaySum step on GB300 (sm_103a), and the
// setup and metrics kernels.
//
// Vogels et al., "RelaySum for Decentralized Deep Learning on Heterogeneous
// Data" (arXiv 2110.04175), Algorithm 1 (RelaySGD) with the robust rebuild of
// Section 4.4, local momentum / Adam, lost messages, and the appendix's
// RelaySum/Grad and mean-estimation algorithms on the same relay, for n
// virtual workers on one GPU.  See relaysum.h for the equations and the ABI
// contract, program.h for the visit program, step_kernels.cu for the kernels
// of a step.
//
// Kernels here:
//   relay_init_kernel     x^0 (shared Philox draw) and zeroed messages.
//   relay_fill_mu_kernel  mu_i = scale * sum_k mix[i][k] N_k.
//   relay_metrics_kernel  consensus distance and distance to the optimum,
//   (+ _finish_kernel)    two fixed-order passes in double.
#include "device.cuh"
#include "step_launch.h"

#include <algorithm>
#include <atomic>
#include <cmath>
#include <cstring>
#include <new>

using relaysum::has_wide;
using relaysum::kMaxE;
using relaysum::kMaxN;
using relaysum::NodeRec;
using relaysum::Objective;
using relaysum::Program;

namespace {

// --------------------------------------------------------------------- init

// rows: message rows to zero (E, plus the received-sum rows when they are on).
__global__ void relay_init_kernel(float* x, float* msg_a, float* msg_b, int n, int rows, int64_t ld_x,
                                  int64_t ld_m, int64_t nquads, int64_t d, uint32_t q0, float x0_std,
                                  const __grid_constant__ PhiloxKey key) {
    const int64_t stride = static_cast<int64_t>(gridDim.x) * blockDim.x;
    for (int64_t q = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x; q < nquads; q += stride) {
        const int64_t c = 4 * q;
        const float4 z = normal4(q0 + static_cast<uint32_t>(q), 0u, 0u, 2u, key);
        const float4 v = make_float4(x0_std * z.x, c + 1 < d ? x0_std * z.y : 0.f,
                                     c + 2 < d ? x0_std * z.z : 0.f, c + 3 < d ? x0_std * z.w : 0.f);
        for (int i = 0; i < n; ++i) *reinterpret_cast<float4*>(x + i * ld_x + c) = v;
        const float4 zero = make_float4(0.f, 0.f, 0.f, 0.f);
        for (int e = 0; e < rows; ++e) {
            *reinterpret_cast<float4*>(msg_a + e * ld_m + c) = zero;
            if (msg_b) *reinterpret_cast<float4*>(msg_b + e * ld_m + c) = zero;
        }
    }
}

__global__ void relay_fill_mu_kernel(float* mu, const float* mix, int n, int K, int64_t ld_x, int64_t nquads,
                                     int64_t d, uint32_t q0, float scale, const __grid_constant__ PhiloxKey key) {
    const int64_t stride = static_cast<int64_t>(gridDim.x) * blockDim.x;
    for (int64_t q = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x; q < nquads; q += stride) {
        const int64_t c = 4 * q;
        for (int i = 0; i < n; ++i) {
            float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
            for (int k = 0; k < K; ++k) {
                const float w = __ldg(mix + static_cast<int64_t>(i) * K + k);
                if (w != 0.0f) {  // a zero weight adds exactly nothing
                    const float4 z = normal4(q0 + static_cast<uint32_t>(q), static_cast<uint32_t>(k), 0u, 1u, key);
                    acc = fma4(w, z, acc);
                }
            }
            const float4 sv = scale4(acc, scale);
            *reinterpret_cast<float4*>(mu + i * ld_x + c) =
                make_float4(sv.x, c + 1 < d ? sv.y : 0.f, c + 2 < d ? sv.z : 0.f, c + 3 < d ? sv.w : 0.f);
        }
    }
}

// ------------------------------------------------------------------ metrics

// Consensus distance and distance to the optimum (the quantities of the
// paper's analysis, Section 4): per coordinate c, with xbar = mean_i x_i and
// mubar = mean_i mu_i,
//   xi   += sum_i (x_i - xbar)^2        dist += (xbar - mubar)^2
// Pass 1: each block reduces its share of the coordinates (grid-stride,
// fixed order) into partials[2 blockIdx]; pass 2 sums the partials in a
// fixed order, so the result is deterministic.  Within a quad the sums over
// the workers run in fp32 pairs (below) and only the quad's totals in double:
// the GB300's fp64 rate is a small fraction of its fp32 rate, and per-worker
// fp64 arithmetic made the metrics fp64-bound.
constexpr int kMetricsThreads = 256;
constexpr int kMetricsResident = 4;  // blocks per SM: one wave of equal shares
constexpr int kMetricsMaxBlocks = 1024;

// The exact rounding error of a + b, given s = fl(a + b) (Knuth's TwoSum), of
// two sums at once.
__device__ __forceinline__ Pair sum_error(Pair a, Pair b, Pair s) {
    const Pair bb = sub2(s, a);
    return add2(sub2(a, sub2(s, bb)), sub2(b, bb));
}

// Two running fp32 sums, each kept as the unevaluated pair s + c: c gathers
// every addition's exact rounding error, so the pair carries about twice
// fp32's precision.  The packed instructions keep the compiler from
// contracting or reordering the error terms.
struct PairSum {
    Pair s = pack(0.0f), c = pack(0.0f);
    __device__ __forceinline__ void add(Pair v) {
        const Pair t = add2(s, v);
        c = add2(c, sum_error(s, v, t));
        s = t;
    }
};

__device__ __forceinline__ double block_sum(double v, double* red) {
    for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    __syncthreads();
    if (lane == 0) red[warp] = v;
    __syncthreads();
    double s = 0.0;
    if (threadIdx.x == 0)
        for (int w = 0; w < static_cast<int>(blockDim.x >> 5); ++w) s += red[w];
    return s;  // valid in thread 0
}

// sum_i (x_i - xbar)^2 of two coordinates: x_i - hi exactly as t + its
// rounding error, less lo (dl); t^2 exactly as p + its fma remainder, and
// 2 t dl + dl^2.
struct SquareSum {
    PairSum sq;
    Pair lo = pack(0.0f);
    __device__ __forceinline__ void add(Pair x, Pair minus_hi, Pair xbar_lo) {
        const Pair t = add2(x, minus_hi);
        const Pair dl = sub2(sum_error(x, minus_hi, t), xbar_lo);
        const Pair p = mul2(t, t);
        const Pair pe = fma2(t, t, mul2(p, pack(-1.0f)));
        sq.add(p);
        lo = add2(lo, fma2(dl, dl, fma2(add2(t, t), dl, pe)));
    }
};

// Two values as the unevaluated fp32 pairs hi + lo.
struct HiLo {
    Pair hi, lo;
};

// (s + c) / n: the product with 1 / n as a pair of its own.  s may be smaller
// than c, where large values cancelled.
__device__ __forceinline__ HiLo worker_mean(const PairSum& sum, Pair inv_hi, Pair inv_lo) {
    const Pair t = add2(sum.s, sum.c);
    const Pair e = sum_error(sum.s, sum.c, t);
    const Pair p = mul2(t, inv_hi);
    const Pair r = fma2(e, inv_hi, fma2(t, inv_lo, fma2(t, inv_hi, mul2(p, pack(-1.0f)))));
    const Pair hi = add2(p, r);
    return HiLo{hi, sub2(r, sub2(hi, p))};
}

// Adds (n (xbar - mubar))^2 of the two coordinates, from their sums over the
// workers.  The sums are subtracted before they are divided, so a mean next to
// the optimum keeps its bits.  (x.s - m.s) + (x.c - m.c) is h + l exactly
// wherever the rest l2 is 0, as for values of like magnitude; where it is not
// (or not finite), the four parts are added in double, at 9 instead of 4
// double instructions a coordinate (which always taken makes 208 us of
// metrics for one worker at d = 2.0e7 into 352).
__device__ __forceinline__ void add_squared_difference(const PairSum& x, const PairSum& m, double& total) {
    const Pair minus_ms = mul2(m.s, pack(-1.0f)), minus_mc = mul2(m.c, pack(-1.0f));
    const Pair t = add2(x.s, minus_ms), u = add2(x.c, minus_mc);
    const Pair te = sum_error(x.s, minus_ms, t), ue = sum_error(x.c, minus_mc, u);
    const Pair h = add2(t, u);
    const Pair r = sum_error(t, u, h);
    const Pair l = add2(r, te);
    const Pair l2 = add2(sum_error(r, te, l), ue);
    float h0, h1, l0, l1, r0, r1;
    unpack(h, h0, h1);
    unpack(l, l0, l1);
    unpack(l2, r0, r1);
    double e0, e1;
    if (r0 == 0.0f && r1 == 0.0f) {
        e0 = static_cast<double>(h0) + static_cast<double>(l0);
        e1 = static_cast<double>(h1) + static_cast<double>(l1);
    } else {
        float xs[2], xc[2], ms[2], mc[2];
        unpack(x.s, xs[0], xs[1]);
        unpack(x.c, xc[0], xc[1]);
        unpack(m.s, ms[0], ms[1]);
        unpack(m.c, mc[0], mc[1]);
        e0 = (static_cast<double>(xs[0]) - static_cast<double>(ms[0])) +
             (static_cast<double>(xc[0]) - static_cast<double>(mc[0]));
        e1 = (static_cast<double>(xs[1]) - static_cast<double>(ms[1])) +
             (static_cast<double>(xc[1]) - static_cast<double>(mc[1]));
    }
    total += e0 * e0;
    total += e1 * e1;
}

// Adds the four values of two pairs to a total kept in double: summed as fp32
// pairs first, so a quad costs about 20 double-precision instructions and not
// 80 (the GB300 does one of them per 64 of fp32; that bound the metrics of few
// workers: 756 -> 221 us for 4 workers at d = 2.0e7).
__device__ __forceinline__ void add_quad(const HiLo& a, const HiLo& b, double& total) {
    const Pair t = add2(a.hi, b.hi);
    const Pair e = add2(sum_error(a.hi, b.hi, t), add2(a.lo, b.lo));
    float t0, t1, e0, e1;
    unpack(t, t0, t1);
    unpack(e, e0, e1);
    const float s = __fadd_rn(t0, t1);
    if (!isfinite(s)) {  // beyond fp32's range together: one by one
        float v[4], w[4];
        unpack(a.hi, v[0], v[1]);
        unpack(b.hi, v[2], v[3]);
        unpack(a.lo, w[0], w[1]);
        unpack(b.lo, w[2], w[3]);
        for (int k = 0; k < 4; ++k) total += static_cast<double>(v[k]) + static_cast<double>(w[k]);
        return;
    }
    const float bb = __fsub_rn(s, t0);
    const float err = __fadd_rn(__fsub_rn(t0, __fsub_rn(s, bb)), __fsub_rn(t1, bb));
    total += static_cast<double>(s);
    total += static_cast<double>(__fadd_rn(err, __fadd_rn(e0, e1)));
}

// Zeros the coordinates of a ragged last quad that lie beyond d: their values
// are unspecified, and zeros add nothing.
__device__ __forceinline__ float4 within(float4 v, int64_t c, int64_t d) {
    if (c + 3 >= d) {
        if (c + 1 >= d) v.y = 0.0f;
        if (c + 2 >= d) v.z = 0.0f;
        if (c + 3 >= d) v.w = 0.0f;
    }
    return v;
}

// Bound by issue and the second read of x (from L2 in part): 1,080 us for 64
// workers at d = 9.2M, 1,523 with scalar arithmetic and the means in double.
// The distance to the optimum is added before the second pass, so the sums of
// the centres hold no registers through it (behind it: 1,196 us).  Keeping a
// quad's x_i in shared memory between the passes, filled by asynchronous
// copies, left one block of 4 warps per SM and took 58 us more than reading
// them again.
template <int OBJ>
__global__ void __launch_bounds__(kMetricsThreads, kMetricsResident)
relay_metrics_kernel(const __grid_constant__ Objective obj, const __grid_constant__ PhiloxKey mu_key,
                     const __grid_constant__ ModelArgs a, int n, int64_t d, double* partials) {
    allow_dependent_launch();
    __shared__ double red[kMetricsThreads / 32];
    double xi = 0.0, dist = 0.0;
    const int64_t stride = static_cast<int64_t>(gridDim.x) * blockDim.x;
    const double inv_n = 1.0 / n;
    const float inv_f = static_cast<float>(inv_n);
    const Pair inv_hi = pack(inv_f), inv_lo = pack(static_cast<float>(inv_n - static_cast<double>(inv_f)));
    for (int64_t q = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x; q < a.nquads; q += stride) {
        PairSum xs[2], ms[2];
        for (int i = 0; i < n; ++i) {
            const float4 xv = within(*reinterpret_cast<const float4*>(a.x + i * a.ld_x + 4 * q), 4 * q, d);
            const float4 mv = within(centre<OBJ>(obj, mu_key, a, i, q, nullptr, 0), 4 * q, d);
            xs[0].add(pack(xv.x, xv.y));
            xs[1].add(pack(xv.z, xv.w));
            ms[0].add(pack(mv.x, mv.y));
            ms[1].add(pack(mv.z, mv.w));
        }
        add_squared_difference(xs[0], ms[0], dist);
        add_squared_difference(xs[1], ms[1], dist);
        const HiLo xbar[2] = {worker_mean(xs[0], inv_hi, inv_lo), worker_mean(xs[1], inv_hi, inv_lo)};
        const Pair minus_hi[2] = {mul2(xbar[0].hi, pack(-1.0f)), mul2(xbar[1].hi, pack(-1.0f))};
        SquareSum sq[2];
        for (int i = 0; i < n; ++i) {
            const float4 xv = within(*reinterpret_cast<const float4*>(a.x + i * a.ld_x + 4 * q), 4 * q, d);
            sq[0].add(pack(xv.x, xv.y), minus_hi[0], xbar[0].lo);
            sq[1].add(pack(xv.z, xv.w), minus_hi[1], xbar[1].lo);
        }
        add_quad(HiLo{sq[0].sq.s, add2(sq[0].sq.c, sq[0].lo)}, HiLo{sq[1].sq.s, add2(sq[1].sq.c, sq[1].lo)}, xi);
    }
    const double bxi = block_sum(xi, red);
    const double bdist = block_sum(dist, red);
    if (threadIdx.x == 0) {
        partials[2 * blockIdx.x] = bxi;
        partials[2 * blockIdx.x + 1] = bdist;
    }
}

__global__ void relay_metrics_finish_kernel(const double* partials, int blocks, double scale_xi,
                                            double scale_dist, double* out) {
    wait_for_prior_grid();
    __shared__ double red[kMetricsThreads / 32];
    double xi = 0.0, dist = 0.0;
    for (int b = threadIdx.x; b < blocks; b += blockDim.x) {
        xi += partials[2 * b];
        dist += partials[2 * b + 1];
    }
    const double sxi = block_sum(xi, red);
    const double sdist = block_sum(dist, red);
    if (threadIdx.x == 0) {
        out[0] = sxi * scale_xi;
        out[1] = sdist * scale_dist;
    }
}

// ------------------------------------------------------------- host helpers

bool aligned16(const void* p) { return (reinterpret_cast<uintptr_t>(p) & 15u) == 0; }

bool overlap(const void* a, int64_t abytes, const void* b, int64_t bbytes) {
    if (abytes <= 0 || bbytes <= 0) return false;
    const uintptr_t a0 = reinterpret_cast<uintptr_t>(a), b0 = reinterpret_cast<uintptr_t>(b);
    return a0 < b0 + static_cast<uintptr_t>(bbytes) && b0 < a0 + static_cast<uintptr_t>(abytes);
}

// AUTO picks the node-parallel kernel below this many worker-quads (n times
// the quads) when no worker has more than kRegDeg neighbours.  Measured on
// one GB300 (whole step, L2 flushed), the node kernel against the walk: ahead
// up to 2^16.1 to 2^16.5 quads, 2^19.5 worker-quads with 8 workers and 2^22 with
// 64.  The line meets that at 24 to 32 workers (binary tree of 32 at 2^21: 48
// against 54 us).  With 8 it is late (at 2^20: 27.4 against 25.7 us), with 64
// early (chain at 2^21: 52 against 88 us).  On a star one thread carries the
// hub's edges while its CTA waits, so the walk is faster there.
constexpr int64_t kNodesBelowWorkerQuads = int64_t(1) << 21;

// AUTO: the walk keeps every array's traffic at one pass with one thread
// per quad; with much less than a resident wave of those threads the GPU
// idles, and the node-parallel form (n threads per quad) is used instead.
bool use_nodes(const relay_handle* h) {
    if (h->kernel == RELAY_KERNEL_NODES) return true;
    if (h->kernel == RELAY_KERNEL_WALK) return false;
    if (h->nquads * h->prog.n >= kNodesBelowWorkerQuads) return false;
    return !has_wide(h);
}

// relay_steps takes the multi-step kernel unless the walk is forced or, under
// AUTO, a worker has more than kRegDeg neighbours: its threads then carry
// all its edges at every step while the rest of the CTA waits at the
// barrier (a 64-worker star measured 3.7x slower than one relay_step per
// step).  Measured on one GB300 with every degree <= kRegDeg, from 8 workers
// and d = 4096 to 32 workers and d = 1.1e8, 64 steps per call, the multi-step
// kernel is ahead everywhere: 2.2x to 2.8x, 9x for the 8 workers at d = 4096.
bool use_fused(const relay_handle* h) {
    if (h->prog.nwide > 0) return false;  // received-sum rows are kept by the per-step kernels only
    if (h->kernel == RELAY_KERNEL_NODES) return true;
    if (h->kernel == RELAY_KERNEL_WALK) return false;
    return !has_wide(h);
}

// Whether the launches for few workers (smaller parameters) take this handle.
bool is_small(const relay_handle* h) {
    return h->prog.n <= relaysum::kSmallN &&
           (h->obj.source == relaysum::kMuStored || h->obj.row_off[h->prog.n] <= relaysum::kSmallMixNnz);
}

template <int OBJ>
int launch_metrics(const relay_handle* h, const ModelArgs& a, int max_blocks, double* workspace, double* out,
                   cudaStream_t stream) {
    int dev = 0;
    const int sms = device_sms(&dev);
    if (sms <= 0) return RELAY_ECUDA;
    const int n = h->prog.n;
    const int blocks = std::min(max_blocks, kMetricsResident * sms);
    const PhiloxKey mu_key = philox_key(static_cast<uint64_t>(h->obj.k0) | (static_cast<uint64_t>(h->obj.k1) << 32));
    relay_metrics_kernel<OBJ><<<blocks, kMetricsThreads, 0, stream>>>(h->obj, mu_key, a, n, h->d, workspace);
    const int rc = launch_status();
    if (rc != RELAY_OK) return rc;
    const double denom = h->d > 0 ? static_cast<double>(h->d) : 1.0;
    return launch_step_kernel(relay_metrics_finish_kernel, 1, kMetricsThreads, 0, stream, true,
                              static_cast<const double*>(workspace), blocks, 1.0 / (n * denom),
                              1.0 / (static_cast<double>(n) * n * denom), out);  // dist carries n^2
}

// Rows of a message buffer: E, plus one received-sum row per wide node when
// received sums are on.
int message_rows(const relay_handle* h) { return h->prog.E + h->prog.nwide; }

// Argument checks shared by relay_step_models and relay_step.
int check_step_args(const relay_handle* h, const float* x, const float* msg_in, const float* msg_out,
                    const int32_t* counts, float lr, int64_t step) {
    if (!h || !h->has_objective || !std::isfinite(lr)) return RELAY_EINVAL;
    if (step < 0 || step >= (int64_t(1) << 32)) return RELAY_EINVAL;
    const int E = h->prog.E;
    const int rows = message_rows(h);
    if (E > 0 && !counts) return RELAY_EINVAL;
    if (h->d == 0) return RELAY_OK;  // counters only
    if (E > 0 && (!msg_in || !msg_out || msg_in == msg_out)) return RELAY_EINVAL;
    if (!x || !aligned16(x) || (E > 0 && (!aligned16(msg_in) || !aligned16(msg_out))))
        return RELAY_EINVAL;
    // exact byte spans of the strided arrays (windows of wider arrays may sit side by side)
    const int64_t xb = ((h->prog.n - 1) * h->ld_x + 4 * h->nquads) * 4;
    const int64_t mb = rows > 0 ? ((rows - 1) * h->ld_m + 4 * h->nquads) * 4 : 0;
    if (overlap(x, xb, msg_in, mb) || overlap(x, xb, msg_out, mb) || overlap(msg_in, mb, msg_out, mb))
        return RELAY_EINVAL;
    for (const float* st : {static_cast<const float*>(h->s1), static_cast<const float*>(h->s2)})
        if (st && (overlap(st, xb, x, xb) || overlap(st, xb, msg_in, mb) || overlap(st, xb, msg_out, mb)))
            return RELAY_EINVAL;
    return RELAY_OK;
}

int grid_for(int64_t items, int threads) {
    int dev = 0;
    const int sms = device_sms(&dev);
    const int64_t want = (items + threads - 1) / threads;
    const int64_t cap = static_cast<int64_t>(sms > 0 ? sms : 1) * 8;
    return static_cast<int>(want < 1 ? 1 : (want < cap ? want : cap));
}

}  // namespace

// ====================================================================== ABI

extern "C" {

int relay_create(relay_handle** out, int32_t n, int64_t d, const int32_t* edges, int32_t n_edges) {
    if (out == nullptr) return RELAY_EINVAL;
    *out = nullptr;
    if (d < 0) return RELAY_EINVAL;
    const int64_t ld = (d + 31) / 32 * 32;
    if (ld / 4 >= (int64_t(1) << 32)) return RELAY_EINVAL;
    relay_handle* h = new (std::nothrow) relay_handle;
    if (h == nullptr) return RELAY_ENOMEM;
    int rc = RELAY_OK;
    try {
        rc = relaysum::build_program(n, edges, n_edges, &h->prog);
    } catch (...) {
        rc = RELAY_ENOMEM;
    }
    if (rc != RELAY_OK) {
        delete h;
        return rc;
    }
    relaysum::narrow(h->prog, &h->small_prog);
    h->d = d;
    h->ld = ld;
    h->ld_x = ld;
    h->ld_m = ld;
    h->nquads = (d + 3) / 4;
    *out = h;
    return RELAY_OK;
}

void relay_destroy(relay_handle* h) { delete h; }

int64_t relay_ld(const relay_handle* h) { return h ? h->ld : RELAY_EINVAL; }

int32_t relay_num_edges(const relay_handle* h) { return h ? h->prog.E : RELAY_EINVAL; }

int relay_edges(const relay_handle* h, int32_t* src, int32_t* dst) {
    if (!h || (h->prog.E > 0 && (!src || !dst))) return RELAY_EINVAL;
    for (int e = 0; e < h->prog.E; ++e) {
        src[e] = h->prog.edge_src[e];
        dst[e] = h->prog.edge_dst[e];
    }
    return RELAY_OK;
}

int relay_set_strides(relay_handle* h, int64_t ld_x, int64_t ld_msg) {
    if (!h || ld_x < 4 * h->nquads || ld_msg < 4 * h->nquads || (ld_x & 3) || (ld_msg & 3)) return RELAY_EINVAL;
    h->ld_x = ld_x;
    h->ld_m = ld_msg;
    return RELAY_OK;
}

int relay_set_local_optimizer(relay_handle* h, int32_t kind, float beta1, float beta2, float eps,
                              float* state1, float* state2) {
    if (!h || kind < RELAY_OPT_SGD || kind > RELAY_OPT_ADAM) return RELAY_EINVAL;
    if (!std::isfinite(beta1) || !std::isfinite(beta2) || !std::isfinite(eps)) return RELAY_EINVAL;
    if (kind == RELAY_OPT_NESTEROV && (beta1 < 0.0f || beta1 >= 1.0f)) return RELAY_EINVAL;
    if (kind == RELAY_OPT_ADAM &&
        (beta1 < 0.0f || beta1 >= 1.0f || beta2 < 0.0f || beta2 >= 1.0f || !(eps > 0.0f)))
        return RELAY_EINVAL;
    if (h->d > 0 && kind >= RELAY_OPT_NESTEROV && (!state1 || !aligned16(state1))) return RELAY_EINVAL;
    if (h->d > 0 && kind == RELAY_OPT_ADAM && (!state2 || !aligned16(state2) || state2 == state1))
        return RELAY_EINVAL;
    h->opt = kind;
    h->beta1 = beta1;
    h->beta2 = beta2;
    h->eps = eps;
    h->s1 = kind >= RELAY_OPT_NESTEROV ? state1 : nullptr;
    h->s2 = kind == RELAY_OPT_ADAM ? state2 : nullptr;
    return RELAY_OK;
}

int relay_set_algorithm(relay_handle* h, int32_t algo, int64_t* dme_count) {
    if (!h || algo < RELAY_ALGO_RELAYSGD || algo > RELAY_ALGO_DME) return RELAY_EINVAL;
    if (algo == RELAY_ALGO_DME && !dme_count) return RELAY_EINVAL;
    h->algo = algo;
    h->dme_count = algo == RELAY_ALGO_DME ? dme_count : nullptr;
    return RELAY_OK;
}

int relay_set_lost_messages(relay_handle* h, const uint8_t* lost) {
    if (!h) return RELAY_EINVAL;
    std::memset(h->lost, 0, sizeof(h->lost));
    h->has_lost = false;
    if (!lost) return RELAY_OK;
    for (int e = 0; e < h->prog.E; ++e)
        if (lost[e]) {
            h->lost[e >> 5] |= 1u << (e & 31);
            h->has_lost = true;
        }
    return RELAY_OK;
}

int relay_set_rebuild_mode(relay_handle* h, int32_t mode) {
    if (!h || (mode != 0 && mode != 1)) return RELAY_EINVAL;
    h->mode = mode;
    return RELAY_OK;
}

int relay_set_kernel(relay_handle* h, int32_t kernel) {
    if (!h || kernel < RELAY_KERNEL_AUTO || kernel > RELAY_KERNEL_NODES) return RELAY_EINVAL;
    h->kernel = kernel;
    return RELAY_OK;
}

int relay_set_received_sums(relay_handle* h, int32_t enable) {
    if (!h || (enable != 0 && enable != 1)) return RELAY_EINVAL;
    if ((enable != 0) == h->rsum) return RELAY_OK;
    // rebuild the visit program from the handle's own edge list (edge 2u is
    // the u-th pair as given)
    const int n = h->prog.n;
    int32_t edges[2 * (kMaxN - 1)];
    for (int u = 0; u < n - 1; ++u) {
        edges[2 * u] = h->prog.edge_src[2 * u];
        edges[2 * u + 1] = h->prog.edge_dst[2 * u];
    }
    Program* p = new (std::nothrow) Program;
    if (!p) return RELAY_ENOMEM;
    int rc = RELAY_OK;
    try {
        rc = relaysum::build_program(n, edges, n - 1, p, enable != 0);
    } catch (...) {
        rc = RELAY_ENOMEM;
    }
    if (rc == RELAY_OK) {
        h->prog = *p;
        relaysum::narrow(h->prog, &h->small_prog);
        h->rsum = enable != 0;
    }
    delete p;
    return rc;
}

int32_t relay_message_rows(const relay_handle* h) { return h ? message_rows(h) : RELAY_EINVAL; }

int relay_get_kernel(const relay_handle* h) {
    if (!h) return RELAY_EINVAL;
    return use_nodes(h) ? RELAY_KERNEL_NODES : RELAY_KERNEL_WALK;
}

int relay_set_coord_offset(relay_handle* h, int64_t c0) {
    if (!h || c0 < 0 || (c0 & 3) != 0) return RELAY_EINVAL;
    if ((c0 + h->ld) / 4 >= (int64_t(1) << 32)) return RELAY_EINVAL;
    h->c0 = c0;
    return RELAY_OK;
}

int relay_set_objective(relay_handle* h, const float* mu, float sigma) {
    if (!h || !std::isfinite(sigma) || sigma < 0.0f) return RELAY_EINVAL;
    if (h->d > 0 && (!mu || !aligned16(mu))) return RELAY_EINVAL;
    h->mu = mu;
    h->sigma = sigma;
    h->obj.source = relaysum::kMuStored;
    h->has_objective = true;
    return RELAY_OK;
}

// The non-zeros of a host mixture matrix mix [n][K] into an Objective.
static int mixture(const relay_handle* h, const float* mix, int32_t K, float mu_scale, Objective* o, int* nnz_out) {
    if (K > 32767) return RELAY_EUNSUPPORTED;
    const int n = h->prog.n;
    std::memset(o, 0, sizeof(*o));
    int nnz = 0;
    for (int i = 0; i < n; ++i) {
        o->row_off[i] = static_cast<int16_t>(nnz);
        for (int k = 0; k < K; ++k) {
            const float w = mix[static_cast<int64_t>(i) * K + k];
            if (!std::isfinite(w)) return RELAY_EINVAL;
            if (w == 0.0f) continue;
            if (nnz >= relaysum::kMaxMixNnz) return RELAY_EUNSUPPORTED;
            o->col[nnz] = static_cast<int16_t>(k);
            o->w[nnz] = w;
            ++nnz;
        }
    }
    o->row_off[n] = static_cast<int16_t>(nnz);
    o->K = K;
    o->scale = mu_scale;
    *nnz_out = nnz;
    return RELAY_OK;
}

int relay_set_objective_generated(relay_handle* h, const float* mix, int32_t K, float mu_scale,
                                  uint64_t mu_seed, float sigma) {
    if (!h || K < 0 || (K > 0 && !mix) || !std::isfinite(mu_scale) || !std::isfinite(sigma) ||
        sigma < 0.0f)
        return RELAY_EINVAL;
    Objective o;
    int nnz = 0;
    const int rc = mixture(h, mix, K, mu_scale, &o, &nnz);
    if (rc != RELAY_OK) return rc;
    o.k0 = static_cast<uint32_t>(mu_seed);
    o.k1 = static_cast<uint32_t>(mu_seed >> 32);
    // one Philox block per non-zero, or K per quad when that is fewer
    o.source = (K <= relaysum::kMaxCachedCentres && K < nnz) ? relaysum::kMuCachedCentres
                                                              : relaysum::kMuPerRow;
    h->obj = o;
    relaysum::narrow(h->obj, &h->small_obj);
    h->mu = nullptr;
    h->sigma = sigma;
    h->has_objective = true;
    return RELAY_OK;
}

int relay_fill_objective(relay_handle* h, float* mu, const float* mix, int32_t K, float mu_scale,
                         uint64_t mu_seed, relay_stream_t stream) {
    if (!h || K < 0 || !std::isfinite(mu_scale)) return RELAY_EINVAL;
    if (h->d == 0) return RELAY_OK;
    if (!mu || !aligned16(mu) || (K > 0 && !mix)) return RELAY_EINVAL;
    const int threads = 256;
    relay_fill_mu_kernel<<<grid_for(h->nquads, threads), threads, 0, stream>>>(
        mu, mix, h->prog.n, K, h->ld_x, h->nquads, h->d, static_cast<uint32_t>(h->c0 / 4), mu_scale,
        philox_key(mu_seed));
    return launch_status();
}

int relay_init(relay_handle* h, float* x, float* msg_a, float* msg_b, int32_t* counts, float x0_std,
               uint64_t seed, relay_stream_t stream) {
    if (!h || !std::isfinite(x0_std)) return RELAY_EINVAL;
    const int E = h->prog.E;
    if (E > 0 && !counts) return RELAY_EINVAL;
    if (h->d > 0 && (!x || !aligned16(x) || (E > 0 && (!msg_a || !aligned16(msg_a))) ||
                     (msg_b && !aligned16(msg_b))))
        return RELAY_EINVAL;
    if (E > 0 && cudaMemsetAsync(counts, 0, sizeof(int32_t) * E, stream) != cudaSuccess) return RELAY_ECUDA;
    if (h->dme_count &&
        cudaMemsetAsync(h->dme_count, 0, sizeof(int64_t) * h->prog.n, stream) != cudaSuccess)
        return RELAY_ECUDA;
    if (h->d == 0) return RELAY_OK;
    // optimiser state starts at zero (momentum buffer, Adam moments)
    for (float* st : {h->s1, h->s2})
        if (st && cudaMemset2DAsync(st, static_cast<size_t>(h->ld_x) * 4, 0, static_cast<size_t>(4 * h->nquads) * 4,
                                    static_cast<size_t>(h->prog.n), stream) != cudaSuccess)
            return RELAY_ECUDA;
    const int threads = 256;
    relay_init_kernel<<<grid_for(h->nquads, threads), threads, 0, stream>>>(
        x, E > 0 ? msg_a : nullptr, E > 0 ? msg_b : nullptr, h->prog.n, message_rows(h), h->ld_x, h->ld_m, h->nquads,
        h->d, static_cast<uint32_t>(h->c0 / 4), x0_std, philox_key(seed));
    return launch_status();
}

int relay_step_counts(relay_handle* h, int32_t* counts, relay_stream_t stream) {
    if (!h) return RELAY_EINVAL;
    if (h->prog.E == 0 && h->algo != RELAY_ALGO_DME) return RELAY_OK;
    if (!counts && h->prog.E > 0) return RELAY_EINVAL;
    const relay_handle* const hs[1] = {h};
    return is_small(h) ? relaysum::small::launch_counts(hs, &counts, 1, stream)
                       : relaysum::large::launch_counts(hs, &counts, 1, stream);
}

// Adam's bias-corrected factors of step t (k = t + 1), in double.
static void adam_factors(const relay_handle* h, float lr, int64_t step, float* adam_step, float* adam_ibc2) {
    *adam_step = 0.0f;
    *adam_ibc2 = 0.0f;
    if (h->opt != 2) return;
    const double k = static_cast<double>(step) + 1.0;
    *adam_step = static_cast<float>(lr / (1.0 - std::pow(static_cast<double>(h->beta1), k)));
    *adam_ibc2 = static_cast<float>(1.0 / std::sqrt(1.0 - std::pow(static_cast<double>(h->beta2), k)));
}

// The step kernels' arguments for step `step` (checked by check_step_args).
static ModelArgs model_args(const relay_handle* h, float* x, const float* msg_in, float* msg_out,
                            const int32_t* counts, float lr, uint64_t seed, int64_t step) {
    ModelArgs a;
    a.x = x;
    a.mu = h->mu;
    a.msg_in = msg_in;
    a.msg_out = msg_out;
    a.counts = counts;
    a.ld_x = h->ld_x;
    a.ld_m = h->ld_m;
    a.nquads = h->nquads;
    a.q0 = static_cast<uint32_t>(h->c0 / 4);
    a.step = static_cast<uint32_t>(step);
    a.key = philox_key(seed);
    a.lr = lr;
    a.sigma = h->sigma;
    a.mode = h->mode;
    a.algo = h->algo;
    a.has_lost = h->has_lost ? 1 : 0;
    a.rsum = h->prog.nwide > 0 ? 1 : 0;
    std::memcpy(a.lost.w, h->lost, sizeof(a.lost.w));
    a.s1 = h->s1;
    a.s2 = h->s2;
    a.beta1 = h->beta1;
    a.beta2 = h->beta2;
    a.eps = h->eps;
    adam_factors(h, lr, step, &a.adam_step, &a.adam_ibc2);
    return a;
}

// The step kernel's launch; `after_counts`: relay_step's counter kernel was
// just enqueued on `stream`, so the step may start as its programmatic
// dependent.
static int step_models(relay_handle* h, float* x, const float* msg_in, float* msg_out, const int32_t* counts,
                       float lr, uint64_t seed, int64_t step, relay_stream_t stream, bool after_counts) {
    const int rc = check_step_args(h, x, msg_in, msg_out, counts, lr, step);
    if (rc != RELAY_OK) return rc;
    if (h->d == 0) return RELAY_OK;
    const ModelArgs a = model_args(h, x, msg_in, msg_out, counts, lr, seed, step);
    return is_small(h) ? relaysum::small::launch_step(h, a, use_nodes(h), stream, after_counts)
                       : relaysum::large::launch_step(h, a, use_nodes(h), stream, after_counts);
}

int relay_step_models(relay_handle* h, float* x, const float* msg_in, float* msg_out,
                      const int32_t* counts, float lr, uint64_t seed, int64_t step,
                      relay_stream_t stream) {
    return step_models(h, x, msg_in, msg_out, counts, lr, seed, step, stream, false);
}

int relay_step(relay_handle* h, float* x, const float* msg_in, float* msg_out, int32_t* counts, float lr,
               uint64_t seed, int64_t step, relay_stream_t stream) {
    // every check of relay_step_models runs before the counter launch, so a
    // rejected step leaves the counters untouched
    int rc = check_step_args(h, x, msg_in, msg_out, counts, lr, step);
    if (rc != RELAY_OK) return rc;
    // relay_step_counts launches only when there are counters to update
    const bool counted = h->prog.E > 0 || h->algo == RELAY_ALGO_DME;
    rc = relay_step_counts(h, counts, stream);
    if (rc != RELAY_OK) return rc;
    return step_models(h, x, msg_in, msg_out, counts, lr, seed, step, stream, counted);
}

// relay_step_windows runs the windows in one launch when both take the walk,
// neither tree has a node of degree > kRegDeg (double binary trees have
// degree <= 3), and they share the objective (its source; the mixture too
// when regenerated) and the local optimiser; otherwise it issues one
// relay_step per window.
static bool one_launch(const relay_handle* a, const relay_handle* b) {
    if (a->d == 0 || b->d == 0 || use_nodes(a) || use_nodes(b) || has_wide(a) || has_wide(b)) return false;
    if (a->opt != b->opt || a->obj.source != b->obj.source) return false;
    return a->obj.source == relaysum::kMuStored || std::memcmp(&a->obj, &b->obj, sizeof(Objective)) == 0;
}

int relay_step_windows(relay_handle* const* h, int32_t count, float* const* x, const float* const* msg_in,
                       float* const* msg_out, int32_t* const* counts, float lr, uint64_t seed, int64_t step,
                       relay_stream_t stream) {
    if (!h || !x || !msg_in || !msg_out || !counts || count < 1 || count > RELAY_MAX_WINDOWS) return RELAY_EINVAL;
    for (int k = 0; k < count; ++k) {
        if (!h[k]) return RELAY_EINVAL;
        for (int j = 0; j < k; ++j)
            if (h[j] == h[k]) return RELAY_EINVAL;
        const int rc = check_step_args(h[k], x[k], msg_in[k], msg_out[k], counts[k], lr, step);
        if (rc != RELAY_OK) return rc;
    }
    if (count == 1 || !one_launch(h[0], h[1])) {
        for (int k = 0; k < count; ++k) {
            const int rc = relay_step(h[k], x[k], msg_in[k], msg_out[k], counts[k], lr, seed, step, stream);
            if (rc != RELAY_OK) return rc;
        }
        return RELAY_OK;
    }
    // the counters of both windows (one CTA each), then the step kernel as
    // its programmatic dependent
    const relay_handle* const hs[2] = {h[0], h[1]};
    const bool fits = is_small(h[0]) && is_small(h[1]);
    bool counted = false;
    for (int k = 0; k < 2; ++k) counted = counted || h[k]->prog.E > 0 || h[k]->algo == RELAY_ALGO_DME;
    if (counted) {
        const int rc = fits ? relaysum::small::launch_counts(hs, counts, 2, stream)
                            : relaysum::large::launch_counts(hs, counts, 2, stream);
        if (rc != RELAY_OK) return rc;
    }
    const ModelArgs as[2] = {model_args(h[0], x[0], msg_in[0], msg_out[0], counts[0], lr, seed, step),
                             model_args(h[1], x[1], msg_in[1], msg_out[1], counts[1], lr, seed, step)};
    return fits ? relaysum::small::launch_step_windows(hs, as, stream, counted)
                : relaysum::large::launch_step_windows(hs, as, stream, counted);
}

int relay_get_steps_kernel(const relay_handle* h) {
    if (!h) return RELAY_EINVAL;
    return use_fused(h) ? RELAY_KERNEL_FUSED : relay_get_kernel(h);
}

int relay_steps(relay_handle* h, float* x, float* msg_a, float* msg_b, int32_t* counts, float lr, uint64_t seed,
                int64_t t0, int64_t k, relay_stream_t stream) {
    int rc = check_step_args(h, x, msg_a, msg_b, counts, lr, t0);
    if (rc != RELAY_OK) return rc;
    if (k < 0 || k > (int64_t(1) << 32) - t0) return RELAY_EINVAL;  // step counters stay below 2^32
    float* const buf[2] = {msg_a, msg_b};
    if (!use_fused(h)) {  // a wide node would hold its CTA at every step: one relay_step per step
        for (int64_t j = 0; j < k; ++j) {
            rc = relay_step(h, x, buf[j & 1], buf[(j + 1) & 1], counts, lr, seed, t0 + j, stream);
            if (rc != RELAY_OK) return rc;
        }
        return RELAY_OK;
    }
    const bool counted = h->prog.E > 0 || h->algo == RELAY_ALGO_DME;
    for (int64_t done = 0; done < k;) {
        const int kc = static_cast<int>(k - done < kMaxFusedSteps ? k - done : kMaxFusedSteps);
        const int par = static_cast<int>(done & 1);  // step t0 + done reads buf[par]
        if (h->d > 0) {
            const ModelArgs a = model_args(h, x, buf[par], buf[par ^ 1], counts, lr, seed, t0 + done);
            FusedSteps fs;
            fs.k = kc;
            fs.msg[0] = buf[par];
            fs.msg[1] = buf[par ^ 1];
            for (int j = 0; j < kMaxFusedSteps; ++j)
                adam_factors(h, lr, t0 + done + (j < kc ? j : 0), &fs.adam_step[j], &fs.adam_ibc2[j]);
            rc = is_small(h) ? relaysum::small::launch_steps(h, a, fs, stream)
                             : relaysum::large::launch_steps(h, a, fs, stream);
            if (rc != RELAY_OK) return rc;
        }
        // the counters advance after the models kernel, which read them
        if (counted) {
            rc = is_small(h) ? relaysum::small::launch_steps_counts(h, counts, kc, stream, h->d > 0)
                             : relaysum::large::launch_steps_counts(h, counts, kc, stream, h->d > 0);
            if (rc != RELAY_OK) return rc;
        }
        done += kc;
    }
    return RELAY_OK;
}

int relay_nbar(const relay_handle* h, const int32_t* counts_host, int32_t* nbar_host) {
    if (!h || !nbar_host || (h->prog.E > 0 && !counts_host)) return RELAY_EINVAL;
    for (int i = 0; i < h->prog.n; ++i) {
        const NodeRec& r = h->prog.node[i];
        int32_t s = 1;
        for (int p = 0; p < r.deg; ++p) s += counts_host[h->prog.pos_in[r.pos_base + p]];
        nbar_host[i] = s;
    }
    return RELAY_OK;
}

int relay_program(const relay_handle* h, int32_t* nslots, int32_t* order, int32_t* node_rec,
                  int32_t* pos_rec) {
    if (!h) return RELAY_EINVAL;
    const Program& p = h->prog;
    if (nslots) *nslots = p.nslots;
    for (int i = 0; i < p.n; ++i) {
        if (order) order[i] = p.order[i];
        if (node_rec) {
            const NodeRec& r = p.node[i];
            const int32_t v[12] = {r.deg,        r.pos_base,   r.parent_pos, r.recv_slot, r.acc_slot,
                                   r.parent_acc, r.fin_parent, r.parent,     r.tot_slot,  r.flags,
                                   p.rsum_slot[i], p.rsum_row[i]};
            std::memcpy(node_rec + 12 * i, v, sizeof(v));
        }
    }
    if (pos_rec)
        for (int e = 0; e < p.E; ++e) {
            pos_rec[4 * e] = p.pos_in[e];
            pos_rec[4 * e + 1] = p.pos_out[e];
            pos_rec[4 * e + 2] = p.pos_slot[e];
            pos_rec[4 * e + 3] = p.pos_in[e];
        }
    return RELAY_OK;
}

int64_t relay_metrics_workspace(const relay_handle* h) {
    if (!h) return RELAY_EINVAL;
    const int64_t blocks = (h->nquads + kMetricsThreads - 1) / kMetricsThreads;
    return 2 * std::max<int64_t>(1, std::min<int64_t>(blocks, kMetricsMaxBlocks));
}

int relay_metrics(relay_handle* h, const float* x, double* workspace, double* out, relay_stream_t stream) {
    if (!h || !h->has_objective || !out || !workspace) return RELAY_EINVAL;
    if (h->d > 0 && (!x || !aligned16(x))) return RELAY_EINVAL;
    const int blocks = static_cast<int>(relay_metrics_workspace(h) / 2);
    ModelArgs a;
    std::memset(&a, 0, sizeof(a));
    a.x = const_cast<float*>(x);
    a.mu = h->mu;
    a.ld_x = h->ld_x;
    a.nquads = h->nquads;
    a.q0 = static_cast<uint32_t>(h->c0 / 4);
    // cached centres are regenerated per row here
    return h->obj.source == relaysum::kMuStored
               ? launch_metrics<relaysum::kMuStored>(h, a, blocks, workspace, out, stream)
               : launch_metrics<relaysum::kMuPerRow>(h, a, blocks, workspace, out, stream);
}

// ------------------------------------------- allocation-free metrics variant

// Scratch for relay_metrics_static: the per-block partial sums of the metrics
// reduction, in a file-scope device array instead of a caller workspace.
// Every GPU that loads the library holds it (16 KB) until the process exits.
constexpr int kStaticMetricsDoubles = 2 * kMetricsMaxBlocks;
static __device__ __align__(256) double g_metrics_scratch[kStaticMetricsDoubles];

namespace {
// The array's device address, looked up once per device with that device
// current.  (In host code the array's name is only a host-side stand-in.)
std::atomic<double*> g_metrics_scratch_addr[kMaxDevices];

double* metrics_scratch_address(int dev) {
    double* p = dev < kMaxDevices ? g_metrics_scratch_addr[dev].load() : nullptr;
    if (p) return p;
    if (cudaGetSymbolAddress(reinterpret_cast<void**>(&p), g_metrics_scratch) != cudaSuccess || !p)
        return nullptr;
    if (dev < kMaxDevices) g_metrics_scratch_addr[dev].store(p);
    return p;
}
}  // namespace

int relay_metrics_static(relay_handle* h, const float* x, double* out, relay_stream_t stream) {
    if (!h) return RELAY_EINVAL;
    if (relay_metrics_workspace(h) > kStaticMetricsDoubles) return RELAY_EUNSUPPORTED;
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) return RELAY_ECUDA;
    double* scratch = metrics_scratch_address(dev);
    if (!scratch) return RELAY_ECUDA;
    // pass 1 overwrites every partial that pass 2 reads: nothing to clear
    return relay_metrics(h, x, scratch, out, stream);
}

const char* relay_error_string(int status) {
    switch (status) {
        case RELAY_OK: return "ok";
        case RELAY_EINVAL: return "invalid argument";
        case RELAY_ENOTTREE: return "edge list is not a tree";
        case RELAY_ECUDA: return "CUDA launch or runtime error";
        case RELAY_ENOMEM: return "host allocation failed";
        case RELAY_EUNSUPPORTED: return "unsupported size";
        default: return "unknown status";
    }
}

}  // extern "C"

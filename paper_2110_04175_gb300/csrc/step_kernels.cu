// step_kernels.cu -- the kernels that run at every step: counters, the walk,
// the node-parallel step and the multi-step kernel, and their launches.
//
// Compiled once per capacity (RELAY_CAP workers): the visit program and the
// mixture of the regenerated centres ride in the kernel parameters, and their
// arrays are sized for the capacity, so a launch for up to kSmallN workers
// carries 3 to 7 KB instead of 13 to 32 KB.  A launch copies all of it, and
// the tables of a small tree lie close together in the constant cache.
//
// Kernels:
//   relay_counts_kernel   Alg. 1 counters, int32, one CTA, in place (lost
//                         messages count 0; mean estimation's counts s_i).
//   relay_models_kernel   everything per coordinate, in ONE pass over d:
//                         local step (SGD / Nesterov / Adam) with Philox noise,
//                         every outgoing relay message, every rebuild.  Each
//                         x_i, mu_i and incoming message quad is read from HBM
//                         once and each outgoing message / new model quad
//                         written once (a child of a node of degree > 4
//                         re-reads the one message it sent that node, see
//                         program.h).  The path is bandwidth-bound streaming
//                         arithmetic: no tensor cores.
//   relay_nodes_kernel    the same step for short vectors, one thread per
//                         (worker, quad) with the new messages exchanged in
//                         shared memory; same bits as relay_models_kernel.
#include "device.cuh"
#include "step_launch.h"

#include <algorithm>
#include <cmath>
#include <cstring>
#include <type_traits>

using relaysum::has_wide;
using relaysum::kRegDeg;
using relaysum::NodeRec;

namespace {

constexpr int kMaxN = RELAY_CAP;
constexpr int kMaxE = 2 * (kMaxN - 1);
constexpr bool kSmall = RELAY_CAP < relaysum::kMaxN;
using Program = relaysum::ProgramT<RELAY_CAP>;
using Objective = std::conditional_t<kSmall, relaysum::SmallObjective, relaysum::Objective>;
// Stored centres need none of the mixture.
struct NoObjective {
    int32_t K;
};
template <int OBJ>
using ObjectiveArg = std::conditional_t<OBJ == relaysum::kMuStored, NoObjective, Objective>;

// ------------------------------------------------------------------ counters

// c^t_{i->j} = 1 + sum_{k in N(i)\j} c^{t-1}_{k->i}: the incoming edge from
// j is e ^ 1 for e = i -> j.  A lost message (Section 4.4) arrives as c = 0.
// For distributed mean estimation (Alg. 5) it also adds each worker's
// models-received count 1 + sum_j c^t_{j->i} to the running count s_i.
// c^t of directed edge e from c^{t-1}; a lost message carries no count.
__device__ __forceinline__ int32_t next_count(const Program& prog, const LostMask& lost, int has_lost,
                                              const int32_t* c_old, int e) {
    const NodeRec r = prog.node[prog.edge_src[e]];
    int32_t s = 1;
    for (int p = 0; p < r.deg; ++p) {
        const int in = prog.pos_in[r.pos_base + p];
        if (in != (e ^ 1)) s += c_old[in];
    }
    return (has_lost && lost(e)) ? 0 : s;
}

// The counters of NT handles (the tree windows of relay_step_windows, or one
// handle): CTA w updates window w's.
template <int NT>
struct CountWindows {
    Program prog[NT];
    LostMask lost[NT];
    int32_t has_lost[NT];
    int32_t* counts[NT];
    int64_t* dme_count[NT];  // Alg. 5's counts s_i, or null
};

template <int NT>
__global__ void relay_counts_kernel(const __grid_constant__ CountWindows<NT> cw) {
    allow_dependent_launch();
    __shared__ int32_t c_old[kMaxE];
    const int w = (NT == 1) ? 0 : static_cast<int>(blockIdx.x);
    const Program& prog = cw.prog[w];
    const LostMask& lost = cw.lost[w];
    const int has_lost = cw.has_lost[w];
    int32_t* const counts = cw.counts[w];
    int64_t* const dme_count = cw.dme_count[w];
    const int E = prog.E;
    for (int e = threadIdx.x; e < E; e += blockDim.x) c_old[e] = counts[e];
    __syncthreads();
    for (int e = threadIdx.x; e < E; e += blockDim.x) counts[e] = next_count(prog, lost, has_lost, c_old, e);
    if (dme_count) {  // Alg. 5: s_i += 1 + sum_j c^t_{j->i}
        __syncthreads();
        for (int i = threadIdx.x; i < prog.n; i += blockDim.x) {
            const NodeRec r = prog.node[i];
            int64_t nb = 1;
            for (int p = 0; p < r.deg; ++p) nb += counts[prog.pos_in[r.pos_base + p]];
            dme_count[i] += nb;
        }
    }
}

// Rounds of the counter recurrence after which it repeats: the counter of
// edge i -> j depends on c^{-1} only through edges one hop further from j, so
// after as many rounds as the tree's longest path has edges it is a function
// of the tree and the lost messages alone, and every later round gives it
// again.  A call of k steps needs no more rounds than that, whatever the
// counters it starts from.
int settled_rounds(const Program& prog, int64_t k) {
    const int64_t d = prog.diameter > 1 ? prog.diameter : 1;
    return static_cast<int>(k < d ? k : d);
}

// The counters (and the mean-estimation counts) advanced by k steps, for
// relay_steps: one CTA of kCountsThreads >= n threads (thread i carries
// worker i's mean-estimation count), the counters of the two round parities
// in shared memory, one barrier per round.  Launched as a programmatic
// dependent of the models kernel, which reads the same counters and writes
// none: the rounds run beside it, and only the writes wait for it.
constexpr int kCountsThreads = 256;
static_assert(kMaxN <= kCountsThreads, "relay_counts_steps_kernel gives each worker its own thread");

__global__ void __launch_bounds__(kCountsThreads)
relay_counts_steps_kernel(const __grid_constant__ Program prog,
                                          const __grid_constant__ LostMask lost, int has_lost, int32_t* counts,
                                          int64_t* dme_count, int k, int rounds) {
    __shared__ int32_t c[2][kMaxE];
    const int E = prog.E;
    for (int e = threadIdx.x; e < E; e += blockDim.x) c[1][e] = counts[e];
    __syncthreads();
    int64_t received = 0;  // worker threadIdx.x: sum over the k steps of 1 + sum_j c^t_{j->i}
    for (int j = 0; j < rounds; ++j) {
        const int32_t* c_old = c[(j + 1) & 1];
        int32_t* c_new = c[j & 1];
        for (int e = threadIdx.x; e < E; e += blockDim.x) c_new[e] = next_count(prog, lost, has_lost, c_old, e);
        __syncthreads();
        if (dme_count && threadIdx.x < prog.n) {
            const NodeRec r = prog.node[threadIdx.x];
            int64_t nb = 1;
            for (int p = 0; p < r.deg; ++p) nb += c_new[prog.pos_in[r.pos_base + p]];
            received += (j + 1 == rounds) ? nb * (k - j) : nb;  // the last round's counters stay
        }
    }
    wait_for_prior_grid();
    for (int e = threadIdx.x; e < E; e += blockDim.x) counts[e] = c[(rounds - 1) & 1][e];
    if (dme_count && threadIdx.x < prog.n) dme_count[threadIdx.x] += received;
}

// --------------------------------------------------------------- fused step

// A lost message reaches its receiver as zero (Section 4.4).
__device__ __forceinline__ float4 delivered(const ModelArgs& a, int e, float4 m) {
    return (a.has_lost && a.lost(e)) ? make_float4(0.f, 0.f, 0.f, 0.f) : m;
}

// Per-thread view of the shared-memory slots: slot s of this thread is
// base[s * stride]; a warp's 32 float4 of one slot are contiguous.
struct Slots {
    float4* base;
    int stride;
    __device__ __forceinline__ float4& operator[](int s) const { return base[s * stride]; }
};

// Row of wide node i's received sum in a message buffer (program.h).
__device__ __forceinline__ int64_t rsum_row(const Program& prog, int i) { return prog.E + prog.rsum_row[i]; }

// The message to the DFS parent joins the parent's accumulator (and, with
// received sums, a wide parent's running sum S_p^t); if this worker is the
// parent's last child, the parent's rebuild (and S_p^t) is complete.  WIDE:
// the tree has a node of degree > kRegDeg (the walk's wide-node paths are
// compiled only then).
template <bool WIDE>
__device__ __forceinline__ void to_parent(const Program& prog, const NodeRec& r, const ModelArgs& a, int64_t q,
                                          float4 out, const Slots& sl, const float* s_scale) {
    const float4 acc = add4(sl[r.parent_acc], out);
    if (r.fin_parent >= 0) {
        st_stream(a.x + r.fin_parent * a.ld_x + 4 * q, scale4(acc, s_scale[r.fin_parent]));
    } else {
        sl[r.parent_acc] = acc;
    }
    if (WIDE && a.rsum && (r.flags & relaysum::kRecvFromTotal)) {
        const int rs = prog.rsum_slot[r.parent];
        const float4 sum = add4(sl[rs], out);
        if (r.fin_parent >= 0) {
            st_stream(a.msg_out + rsum_row(prog, r.parent) * a.ld_m + 4 * q, sum);
        } else {
            sl[rs] = sum;
        }
    }
}

// Degree D <= kRegDeg: the D incoming messages live in registers; outgoing
// message s is prefix(s) + suffix(s+1) with prefix(s) = xh + m_0 + ... + m_{s-1}.
template <int D, bool WIDE>
__device__ __forceinline__ void visit_small(const Program& prog, const NodeRec& r, const ModelArgs& a,
                                            int64_t q, float4 xh, const Slots& sl,
                                            const float* s_scale) {
    float4 m[D];
#pragma unroll
    for (int s = 0; s < D; ++s) m[s] = ld_stream(a.msg_in + prog.pos_in[r.pos_base + s] * a.ld_m + 4 * q);
    float4 pre[D];
    pre[0] = xh;
#pragma unroll
    for (int s = 1; s < D; ++s) pre[s] = add4(pre[s - 1], m[s - 1]);
    float4 suf[D];
    suf[D - 1] = m[D - 1];
#pragma unroll
    for (int s = D - 2; s >= 0; --s) suf[s] = add4(m[s], suf[s + 1]);
#pragma unroll
    for (int s = 0; s < D; ++s) {
        const int e = prog.pos_out[r.pos_base + s];
        const float4 out = delivered(a, e, (s == D - 1) ? pre[s] : add4(pre[s], suf[s + 1]));
        st_stream(a.msg_out + e * a.ld_m + 4 * q, out);
        if (s == r.parent_pos) {
            to_parent<WIDE>(prog, r, a, q, out, sl, s_scale);
        } else {
            sl[prog.pos_slot[r.pos_base + s]] = out;
        }
    }
}

// Degree D > kRegDeg: T = xh + the sum of all incoming messages; the message
// to the parent is T minus the parent's incoming message, and T stays in a
// slot for the children (see program.h).  Without received sums one
// streaming pass reads the D incoming rows, over descending positions while
// the children are visited in ascending order, so the first children
// re-read the most recently read (L2-resident) rows.  With received sums,
// T = xh + S_i^{t-1} from the one sum row, and only the parent's incoming
// row is read here.
__device__ __noinline__ void visit_wide(const Program& prog, const NodeRec& r, const ModelArgs& a, int i,
                                        int64_t q, float4 xh, const Slots& sl,
                                        const float* s_scale) {
    const int D = r.deg;
    const int base = r.pos_base;
    float4 total = xh;
    float4 from_parent = make_float4(0.f, 0.f, 0.f, 0.f);
    if (a.rsum) {
        total = add4(xh, ld_stream(a.msg_in + rsum_row(prog, i) * a.ld_m + 4 * q));
        if (r.parent_pos >= 0) from_parent = ld_stream(a.msg_in + prog.pos_in[base + r.parent_pos] * a.ld_m + 4 * q);
    } else {
        for (int s = D - 1; s >= 0; --s) {
            const float4 m = ld_keep(a.msg_in + prog.pos_in[base + s] * a.ld_m + 4 * q);
            total = add4(total, m);
            if (s == r.parent_pos) from_parent = m;
        }
    }
    if (r.parent_pos >= 0) {
        const int e = prog.pos_out[base + r.parent_pos];
        const float4 out = delivered(a, e, sub4(total, from_parent));
        st_stream(a.msg_out + e * a.ld_m + 4 * q, out);
        to_parent<true>(prog, r, a, q, out, sl, s_scale);
    }
    sl[r.tot_slot] = total;
}

// The local optimiser's update u (Alg. 1's local step is x^{t+1/2} = x + u):
//   SGD:      u = -lr g
//   Nesterov: m = beta1 m + g;  u = -lr (g + beta1 m)          (state s1 = m)
//   Adam:     m = beta1 m + (1 - beta1) g;  v = beta2 v + (1 - beta2) g^2;
//             u = -adam_step m / (sqrt(v) adam_ibc2 + eps)     (s1 = m, s2 = v)
// The rule on the optimiser state (m, v) held in registers; adam_step and
// adam_ibc2 are the factors of this step.  Returns u for Adam, and the
// direction u / -lr otherwise (relayed_with applies -lr).
template <int OPT>
__device__ __forceinline__ float4 update_rule(const ModelArgs& a, float adam_step, float adam_ibc2, float4 g,
                                              float4& m, float4& v) {
    if (OPT == 0) return g;
    if (OPT == 1) {
        m = fma4(a.beta1, m, g);
        return fma4(a.beta1, m, g);
    }
    const float c1 = 1.0f - a.beta1, c2 = 1.0f - a.beta2;
    m = fma4(a.beta1, m, scale4(g, c1));
    const float4 cg = scale4(g, c2);
    const float4 gg = quad(mul2(pack(cg.x, cg.y), pack(g.x, g.y)), mul2(pack(cg.z, cg.w), pack(g.z, g.w)));
    v = fma4(a.beta2, v, gg);
    auto upd = [&](float mm, float vv) { return -adam_step * mm / fmaf(sqrtf(vv), adam_ibc2, a.eps); };
    return make_float4(upd(m.x, v.x), upd(m.y, v.y), upd(m.z, v.z), upd(m.w, v.w));
}

// One step's direction (or update) with the state read from and written back to HBM.
template <int OPT>
__device__ __forceinline__ float4 local_update(const ModelArgs& a, int i, int64_t q, float4 g) {
    float4 m = make_float4(0.f, 0.f, 0.f, 0.f), v = m;
    if (OPT == 0) return update_rule<OPT>(a, a.adam_step, a.adam_ibc2, g, m, v);
    float4* pm = reinterpret_cast<float4*>(a.s1 + i * a.ld_x + 4 * q);
    float4* pv = reinterpret_cast<float4*>(a.s2 + i * a.ld_x + 4 * q);
    m = *pm;
    if (OPT == 2) v = *pv;
    const float4 dir = update_rule<OPT>(a, a.adam_step, a.adam_ibc2, g, m, v);
    __stcs(pm, m);
    if (OPT == 2) __stcs(pv, v);
    return dir;
}

// Per-worker rebuild factors from this step's counters: x' = scale * acc
// with acc = fill * x + x^{t+1/2} + incoming messages.
//   mode 0: x' = acc / nbar (Alg. 1).  mode 1: x' = (acc + (n - nbar) x) / n
//   (robust rule), the fill term folded into the accumulator up front.
__device__ __forceinline__ void worker_factors(const ModelArgs& a, int n, int nbar, float& scale, float& fill) {
    if (a.algo == 1) {  // x' = x + (u + sum m) / n
        scale = 1.0f / static_cast<float>(n);
        fill = static_cast<float>(n);
    } else if (a.algo == 2) {  // y' = y + dhat + sum m
        scale = 1.0f;
        fill = 1.0f;
    } else if (a.mode == 0) {
        scale = 1.0f / static_cast<float>(nbar);
        fill = 0.0f;
    } else {
        scale = 1.0f / static_cast<float>(n);
        fill = static_cast<float>(n - nbar);
    }
}

// To be called after wait_for_prior_grid().
__device__ __forceinline__ void rebuild_factors(const Program& prog, const ModelArgs& a, float* s_scale,
                                                float* s_fill) {
    const int n = prog.n;
    for (int i = threadIdx.x; i < n; i += blockDim.x) {
        const NodeRec r = prog.node[i];
        int nbar = 1;
        for (int p = 0; p < r.deg; ++p) nbar += ld_counter(a.counts + prog.pos_in[r.pos_base + p]);
        worker_factors(a, n, nbar, s_scale[i], s_fill[i]);
    }
}

// The relayed value of worker i at quad q: x^{t+1/2} = x + u (Alg. 1), the
// update u (Alg. 6) or the sample mu + sigma xi (Alg. 5), with
// g = (x - mu) + sigma xi and z MINUS the worker's noise normals.
// `update` maps g to the optimiser's direction (and advances its state).
// PLAIN: the caller knows that the algorithm is Alg. 1.
template <int OPT, bool PLAIN, typename Update>
__device__ __forceinline__ float4 relayed_with(const ModelArgs& a, float4 xv, float4 mv, float4 z,
                                               Update update) {
    if (!PLAIN && a.algo == 2) return fma4(-a.sigma, z, mv);
    const float4 dir = update(fma4(-a.sigma, z, sub4(xv, mv)));
    if (!PLAIN && a.algo == 1) return (OPT == 2) ? dir : scale4(dir, -a.lr);
    return (OPT == 2) ? add4(xv, dir) : fma4(-a.lr, dir, xv);
}

template <int OPT>
__device__ __forceinline__ float4 relayed_value(const ModelArgs& a, int i, int64_t q, float4 xv, float4 mv,
                                                float4 z) {
    return relayed_with<OPT, false>(a, xv, mv, z, [&](float4 g) { return local_update<OPT>(a, i, q, g); });
}

// The step of NT handles in one launch: one handle, or the tree windows of
// relay_step_windows (the double binary trees of Section 3: two trees over
// the same workers, each carrying its own columns of the models).  The
// grid's first `split` CTAs work on window 0, the rest on window 1.
template <int NT>
struct Windows {
    Program prog[NT];
    ModelArgs a[NT];
    int32_t split;
};

// The walk over one window's quads, one per thread: CTA `cta` of the window
// takes quads cta * blockDim + threadIdx.  The grid covers every quad, so the
// hardware hands the next CTA to whichever SM is free and the CTAs in flight
// work on neighbouring columns; a resident grid striding over the quads let
// them drift apart, which cost HBM locality and left a last partial round
// (13.35 -> 12.86 ms per step on the 32-worker binary tree at d = 1.1e8, 580
// -> 539 us on two 16-worker trees at d = 9.2M, 787 -> 683 us on the 16-worker
// chain with regenerated centres).  A grid just past a whole number of waves
// loses a little to it (24-worker chain at d = 1.25M, 2.02 waves: 140.5 -> 142.5
// us).  OBJ: where mu comes from (ObjectiveSource).  OPT: the local optimiser
// (0 SGD, 1 Nesterov momentum, 2 Adam).  WIDE: some node has more than kRegDeg
// neighbours; without one the wide-node paths are not compiled, and they cost
// the narrow trees nothing.
template <int OBJ, int OPT, bool WIDE>
__device__ __forceinline__ void walk(const Program& prog, const ModelArgs& a, const ObjectiveArg<OBJ>& obj,
                                     const PhiloxKey& mu_key, int64_t cta, float4* slot_mem, float* s_scale,
                                     float* s_fill) {
    const int n = prog.n;
    const Slots sl{slot_mem + threadIdx.x, static_cast<int>(blockDim.x)};
    float4* cen = slot_mem + prog.nslots * blockDim.x + threadIdx.x;  // OBJ == kMuCachedCentres
    const int64_t q = cta * blockDim.x + threadIdx.x;
    const bool active = q < a.nquads;
    // x (and a stored mu) of the next node in the walk are loaded one visit
    // early, so their latency overlaps the current visit's arithmetic; the
    // first node's, and the centres of the quad, come before the wait for the
    // counter kernel (which writes none of them)
    float4 xn = make_float4(0.f, 0.f, 0.f, 0.f), mn = xn;
    if (active) {
        xn = *reinterpret_cast<const float4*>(a.x + prog.order[0] * a.ld_x + 4 * q);
        if (OBJ == relaysum::kMuStored) mn = ld_stream(a.mu + prog.order[0] * a.ld_x + 4 * q);
        if (OBJ == relaysum::kMuCachedCentres)
            for (int k = 0; k < obj.K; ++k)
                cen[k * blockDim.x] = normal4(a.q0 + static_cast<uint32_t>(q), static_cast<uint32_t>(k), 0u, 1u, mu_key);
    }
    const NoiseQuad nq = noise_quad(a.q0 + static_cast<uint32_t>(q), a.key);
    wait_for_prior_grid();
    rebuild_factors(prog, a, s_scale, s_fill);
    __syncthreads();
    if (!active) return;
    for (int v = 0; v < n; ++v) {
        const int i = prog.order[v];
        const NodeRec r = prog.node[i];
        const float4 xv = xn;
        const float4 mv = (OBJ == relaysum::kMuStored)
                              ? mn : centre<OBJ>(obj, mu_key, a, i, q, cen, static_cast<int>(blockDim.x));
        if (v + 1 < n) {  // the next node is never finalised before its own visit
            const int inext = prog.order[v + 1];
            xn = *reinterpret_cast<const float4*>(a.x + inext * a.ld_x + 4 * q);
            if (OBJ == relaysum::kMuStored) mn = ld_stream(a.mu + inext * a.ld_x + 4 * q);
        }
        // a child of a wide node p forms its incoming message as
        // T_p - m^{t-1}_{i->p}; that row is loaded before the noise
        // arithmetic, whose latency it then overlaps (with received sums
        // this is the one read of m^{t-1}_{i->p})
        float4 back = make_float4(0.f, 0.f, 0.f, 0.f);
        if (WIDE && (r.flags & relaysum::kRecvFromTotal)) {
            const float* mp = a.msg_in + prog.pos_out[r.pos_base + r.parent_pos] * a.ld_m + 4 * q;
            back = a.rsum ? ld_stream(mp) : __ldg(reinterpret_cast<const float4*>(mp));
        }
        const float4 z = minus_normal4(noise_words(nq, static_cast<uint32_t>(i), a.step, a.key));
        const float4 xh = relayed_value<OPT>(a, i, q, xv, mv, z);
        // the rebuild sum starts from fill_i x_i (robust rule: n - nbar_i;
        // Alg. 6: n; Alg. 5: 1; Alg. 1: nothing)
        float4 acc = xh;
        if (s_fill[i] != 0.0f) acc = fma4(s_fill[i], xv, xh);
        float4 recv = make_float4(0.f, 0.f, 0.f, 0.f);
        if (r.recv_slot >= 0) {
            recv = sl[r.recv_slot];
            if (WIDE && (r.flags & relaysum::kRecvFromTotal)) {  // m^t_{p->i} = T_p - m^{t-1}_{i->p}, written out here
                const int e = prog.pos_in[r.pos_base + r.parent_pos];
                recv = delivered(a, e, sub4(recv, back));
                st_stream(a.msg_out + e * a.ld_m + 4 * q, recv);
            }
            acc = add4(acc, recv);
        }
        // a wide node's received sum S_i^t starts with its DFS parent's message
        if (WIDE && a.rsum && r.deg > kRegDeg) sl[prog.rsum_slot[i]] = add4(make_float4(0.f, 0.f, 0.f, 0.f), recv);
        switch (r.deg) {
            case 0: break;
            case 1: visit_small<1, WIDE>(prog, r, a, q, xh, sl, s_scale); break;
            case 2: visit_small<2, WIDE>(prog, r, a, q, xh, sl, s_scale); break;
            case 3: visit_small<3, WIDE>(prog, r, a, q, xh, sl, s_scale); break;
            case 4: visit_small<4, WIDE>(prog, r, a, q, xh, sl, s_scale); break;
            default:
                if (WIDE) visit_wide(prog, r, a, i, q, xh, sl, s_scale);
                break;
        }
        if (r.acc_slot < 0) {
            st_stream(a.x + i * a.ld_x + 4 * q, scale4(acc, s_scale[i]));
        } else {
            sl[r.acc_slot] = acc;
        }
    }
}

// The step kernel over NT windows.  The walk is inlined once per window, so
// each copy reads its window's program and arguments at fixed parameter
// offsets (constant operands), as the one-window kernel does; the grid's
// first `split` CTAs take window 0.
// MIN: the resident CTAs of 128 threads per SM that the walk's registers are
// budgeted for (0: no bound, the compiler's choice: 64 registers, 8 CTAs).
// The wide-node variant takes 8: 5.90 ms per step on the 64-worker star at d =
// 2.5e7, against 6.14 ms budgeted for 7, 6.57 for 6 and 7.38 for 9 (which
// spills).  Narrow trees with stored centres take 0 or 7 (seven_ctas).
template <int OBJ, int OPT, int NT, bool WIDE, int MIN>
__global__ void __launch_bounds__(128, MIN)
relay_models_kernel(const __grid_constant__ Windows<NT> win, const __grid_constant__ ObjectiveArg<OBJ> obj,
                    const __grid_constant__ PhiloxKey mu_key) {
    extern __shared__ float4 slot_mem[];
    __shared__ float s_scale[kMaxN];
    __shared__ float s_fill[kMaxN];
    if (NT == 1) {
        walk<OBJ, OPT, WIDE>(win.prog[0], win.a[0], obj, mu_key, blockIdx.x, slot_mem, s_scale, s_fill);
    } else if (static_cast<int>(blockIdx.x) < win.split) {
        walk<OBJ, OPT, WIDE>(win.prog[0], win.a[0], obj, mu_key, blockIdx.x, slot_mem, s_scale, s_fill);
    } else {
        walk<OBJ, OPT, WIDE>(win.prog[NT - 1], win.a[NT - 1], obj, mu_key, blockIdx.x - win.split, slot_mem, s_scale,
                             s_fill);
    }
}

// ------------------------------------------------- node-parallel fused step

// For short vectors the walk leaves the GPU idle (one thread per quad walks
// all n workers in turn), so this form of the same step gives each
// (worker, quad) pair its own thread.  A CTA owns qb consecutive quads of
// every worker; qb consecutive threads share a worker, the workers in
// ascending degree, so the lanes of a warp have (nearly) the same number of
// messages.  Phase 1: each thread forms x_i^{t+1/2} and worker i's outgoing
// messages with the walk's arithmetic (prefix + suffix at degree <= kRegDeg,
// the total minus the reverse message above it), writes them out and leaves
// them in shared memory, at the position where they arrive.  Phase 2, after
// one barrier: each thread adds its worker's incoming messages, consecutive
// rows in the walk's order, and writes the new model.  The results equal
// relay_models_kernel's bit for bit, and every array is still read and
// written once.

// What a thread of the node-parallel and multi-step kernels is: one worker's
// share of one quad at a time.
struct NodeThread {
    int i, deg;            // worker (deg 0 on the threads that fill up the last warp)
    int pos_base;          // its first position
    int in;                // float4 index of its first incoming message in a buffer; the next is qb further
    uint32_t lost_bits;    // bit s: its message to neighbour s is lost (narrow nodes)
};

__device__ __forceinline__ NodeThread node_thread(const Program& prog, const ModelArgs& a, int slot, int qi, int qb) {
    const bool live = slot < prog.n;
    NodeThread t;
    t.i = prog.by_degree[live ? slot : prog.n - 1];
    t.deg = live ? prog.node[t.i].deg : 0;
    t.pos_base = live ? prog.node[t.i].pos_base : 0;
    t.in = t.pos_base * qb + qi;
    t.lost_bits = 0;
    if (a.has_lost && t.deg <= kRegDeg)
        for (int s = 0; s < t.deg; ++s) t.lost_bits |= (a.lost(prog.pos_out[t.pos_base + s]) ? 1u : 0u) << s;
    return t;
}

// Outgoing message s = prefix(s) + suffix(s + 1) with prefix(s) = xh + m_0 +
// ... + m_{s-1}.  A lane's missing neighbours hold nothing4(): v + -0 is v for any
// v, a zero's sign included (-0 + 0 would be +0).
__device__ __forceinline__ float4 nothing4() { return make_float4(-0.0f, -0.0f, -0.0f, -0.0f); }

template <int D>
__device__ __forceinline__ void narrow_messages(const float4 (&m)[D], float4 xh, uint32_t lost_bits,
                                                float4 (&o)[D]) {
    float4 pre = xh;
    float4 suf[D];
    suf[D - 1] = m[D - 1];
#pragma unroll
    for (int s = D - 2; s >= 1; --s) suf[s] = add4(m[s], suf[s + 1]);
#pragma unroll
    for (int s = 0; s < D; ++s) {
        o[s] = (s == D - 1) ? pre : add4(pre, suf[s + 1]);
        if (s + 1 < D) pre = add4(pre, m[s]);
    }
    if (lost_bits) {
#pragma unroll
        for (int s = 0; s < D; ++s)
            if ((lost_bits >> s) & 1u) o[s] = make_float4(0.f, 0.f, 0.f, 0.f);
    }
}

// Phase 1 of a worker with at most D <= kRegDeg neighbours: its incoming rows
// are requested before the noise arithmetic, which covers their latency (with
// Adam after its update, whose registers they would spill: 40.7 against 40.2
// us on the 16-worker chain at d = 272,474).  `sent[s]` is the float4 index
// where the message to neighbour s arrives; Adam looks it up again instead of
// holding it (8 bytes spilled, 36 otherwise).
template <int D, int OPT>
__device__ __forceinline__ float4 node_send(const Program& prog, const ModelArgs& a, const NodeThread& t, int64_t q,
                                            float4 xv, float4 mv, const int (&sent)[kRegDeg], int qb, float4* m_new) {
    constexpr int DN = D > 0 ? D : 1;
    float4 m[DN];
    auto request = [&]() {
#pragma unroll
        for (int s = 0; s < D; ++s) {
            m[s] = nothing4();
            if (s < t.deg) m[s] = ld_stream(a.msg_in + prog.pos_in[t.pos_base + s] * a.ld_m + 4 * q);
        }
    };
    if (OPT != 2) request();
    const float4 z = minus_normal4(noise_words(noise_quad(a.q0 + static_cast<uint32_t>(q), a.key),
                                               static_cast<uint32_t>(t.i), a.step, a.key));
    const float4 xh = relayed_value<OPT>(a, t.i, q, xv, mv, z);
    if (OPT == 2) request();
    if (D > 0) {
        float4 o[DN];
        narrow_messages<DN>(m, xh, t.lost_bits, o);
#pragma unroll
        for (int s = 0; s < D; ++s)
            if (s < t.deg) {
                m_new[OPT == 2 ? prog.edge_pos[prog.pos_out[t.pos_base + s]] * qb + (t.in - t.pos_base * qb) : sent[s]] = o[s];
                st_stream(a.msg_out + prog.pos_out[t.pos_base + s] * a.ld_m + 4 * q, o[s]);
            }
    }
    return xh;
}

// Phase 1 in a warp with a worker of degree > kRegDeg: T = x^{t+1/2} + the
// incoming messages summed over descending positions (with received sums: +
// the sum row S_i^{t-1}), then message s = T - (incoming message s), as in
// visit_wide and at the wide node's children.  The incoming messages wait in
// shared memory (the worker's own rows of m_old).
template <int OPT>
__device__ __noinline__ float4 node_send_wide(const Program& prog, const ModelArgs& a, const NodeThread& t,
                                              int64_t q, float4 xv, float4 mv, int qb, float4* m_new,
                                              float4* m_old) {
    const int qi = t.in - t.pos_base * qb;
    const float4 z = minus_normal4(noise_words(noise_quad(a.q0 + static_cast<uint32_t>(q), a.key),
                                               static_cast<uint32_t>(t.i), a.step, a.key));
    const float4 xh = relayed_value<OPT>(a, t.i, q, xv, mv, z);
    float4* const own = m_old + t.in;
    const bool wide = t.deg > kRegDeg;
    float4 total = xh;
    if (wide && a.rsum) total = add4(xh, ld_stream(a.msg_in + rsum_row(prog, t.i) * a.ld_m + 4 * q));
    for (int s = t.deg - 1; s >= 0; --s) {
        const float4 m = ld_stream(a.msg_in + prog.pos_in[t.pos_base + s] * a.ld_m + 4 * q);
        if (wide && !a.rsum) total = add4(total, m);
        own[s * qb] = m;
    }
    for (int s = 0; s < t.deg; ++s) {
        float4 o;
        if (wide) {
            o = sub4(total, own[s * qb]);
        } else {
            o = xh;
            for (int r = 0; r < s; ++r) o = add4(o, own[r * qb]);
            if (s + 1 < t.deg) {
                float4 suf = own[(t.deg - 1) * qb];
                for (int r = t.deg - 2; r > s; --r) suf = add4(own[r * qb], suf);
                o = add4(o, suf);
            }
        }
        const int e = prog.pos_out[t.pos_base + s];
        o = delivered(a, e, o);
        st_stream(a.msg_out + e * a.ld_m + 4 * q, o);
        m_new[prog.edge_pos[e] * qb + qi] = o;
    }
    return xh;
}

// blockDim.x = qb * n rounded up to whole warps, at most kNodeThreads.
// Dynamic shared memory: two [E][qb] float4 message buffers used by alternate
// blocks, plus one more for the incoming messages of wide nodes when the tree
// has any.  With two buffers a block needs one barrier: a warp already in the
// next block's phase 1 writes the other buffer, and it can reach this buffer
// again only after every warp has passed the next block's barrier, i.e.
// finished reading this one.
constexpr int kNodeThreads = 512;

template <int OBJ, int OPT>
__global__ void __launch_bounds__(kNodeThreads, 2)
relay_nodes_kernel(const __grid_constant__ Program prog, const __grid_constant__ ObjectiveArg<OBJ> obj,
                   const __grid_constant__ PhiloxKey mu_key, const __grid_constant__ ModelArgs a, int qb_log2) {
    extern __shared__ float4 node_mem[];
    __shared__ float s_scale[kMaxN];
    __shared__ float s_fill[kMaxN];
    // regenerated centres are formed per row (the walk's cached centres are
    // the same normals mixed in the same order)
    constexpr int kObj = (OBJ == relaysum::kMuStored) ? relaysum::kMuStored : relaysum::kMuPerRow;
    const int qb = 1 << qb_log2;
    const int tid = static_cast<int>(threadIdx.x);
    const int slot = tid >> qb_log2, qi = tid & (qb - 1);
    const bool live = slot < prog.n;
    const NodeThread t = node_thread(prog, a, slot, qi, qb);
    const int widest = __reduce_max_sync(0xffffffffu, t.deg);
    int sent[kRegDeg];
#pragma unroll
    for (int s = 0; s < kRegDeg; ++s)
        sent[s] = s < t.deg ? prog.edge_pos[prog.pos_out[t.pos_base + s]] * qb + qi : 0;
    float4* const m_old = node_mem + 2 * prog.E * qb;
    const float* const xrow = a.x + t.i * a.ld_x;
    const float* const murow = (OBJ == relaysum::kMuStored) ? a.mu + t.i * a.ld_x : nullptr;
    const int64_t nblk = (a.nquads + qb - 1) >> qb_log2;
    const int64_t qstep = static_cast<int64_t>(gridDim.x) << qb_log2;
    // x (and a stored mu) of this thread's next block are loaded one block
    // early, so their latency overlaps the barrier and the rebuild
    float4 xn = make_float4(0.f, 0.f, 0.f, 0.f), mn = xn;
    int64_t q = (static_cast<int64_t>(blockIdx.x) << qb_log2) + qi;
    if (live && q < a.nquads) {
        xn = *reinterpret_cast<const float4*>(xrow + 4 * q);
        if (OBJ == relaysum::kMuStored) mn = ld_stream(murow + 4 * q);
    }
    // Phase 1 needs no counter: the first block's runs before the wait for the
    // counter kernel (programmatic dependent launch), overlapping it; only the
    // rebuild factors of phase 2 need the counters, which the counter kernel
    // writes (it writes nothing phase 1 reads).
    bool counted = false;
    int parity = 0;
    for (int64_t b = blockIdx.x; b < nblk; b += gridDim.x, q += qstep, parity ^= 1) {
        float4* const m_new = node_mem + (parity ? prog.E * qb : 0);
        const bool active = live && q < a.nquads;
        const float4 xv = xn, ms = mn;
        if (live && q + qstep < a.nquads) {
            xn = *reinterpret_cast<const float4*>(xrow + 4 * (q + qstep));
            if (OBJ == relaysum::kMuStored) mn = ld_stream(murow + 4 * (q + qstep));
        }
        float4 xh = make_float4(0.f, 0.f, 0.f, 0.f);
        if (active) {
            const float4 mv =
                (OBJ == relaysum::kMuStored) ? ms : centre<kObj>(obj, mu_key, a, t.i, q, nullptr, 0);
            switch (widest) {
                case 0: xh = node_send<0, OPT>(prog, a, t, q, xv, mv, sent, qb, m_new); break;
                case 1: xh = node_send<1, OPT>(prog, a, t, q, xv, mv, sent, qb, m_new); break;
                case 2: xh = node_send<2, OPT>(prog, a, t, q, xv, mv, sent, qb, m_new); break;
                case 3: xh = node_send<3, OPT>(prog, a, t, q, xv, mv, sent, qb, m_new); break;
                case 4: xh = node_send<4, OPT>(prog, a, t, q, xv, mv, sent, qb, m_new); break;
                default: xh = node_send_wide<OPT>(prog, a, t, q, xv, mv, qb, m_new, m_old); break;
            }
        }
        if (!counted) {
            wait_for_prior_grid();
            rebuild_factors(prog, a, s_scale, s_fill);
            counted = true;
        }
        __syncthreads();  // also publishes the factors
        if (active) {
            // the rebuild sum starts from fill_i x_i + x^{t+1/2}, as in the walk
            const float4* const mine = m_new + t.in;
            float4 acc = xh;
            if (s_fill[t.i] != 0.0f) acc = fma4(s_fill[t.i], xv, xh);
            if (t.deg <= kRegDeg) {
#pragma unroll
                for (int s = 0; s < kRegDeg; ++s)
                    if (s < t.deg) acc = add4(acc, mine[s * qb]);
            } else if (a.rsum) {  // and the wide node's received sum S_i^t, in the same order
                float4 sum = make_float4(0.f, 0.f, 0.f, 0.f);
                for (int s = 0; s < t.deg; ++s) {
                    acc = add4(acc, mine[s * qb]);
                    sum = add4(sum, mine[s * qb]);
                }
                st_stream(a.msg_out + rsum_row(prog, t.i) * a.ld_m + 4 * q, sum);
            } else {
                for (int s = 0; s < t.deg; ++s) acc = add4(acc, mine[s * qb]);
            }
            st_stream(a.x + t.i * a.ld_x + 4 * q, scale4(acc, s_scale[t.i]));
        }
    }
}

// ------------------------------------------------ several steps per launch

// relay_steps: k consecutive steps in one launch, one thread per (worker,
// quad).  Every coordinate evolves on its own (the counters are the same for
// all of them), so a CTA carries its qb quads of every worker through all k
// steps without hearing from another CTA: models, centres, optimiser state
// and the messages that arrived last stay in registers, and the messages of
// the step being taken pass through shared memory.  HBM is read once (x, mu,
// the optimiser state, m^{t0-1}) and written once (x, the state, and the
// messages of the last two steps, which k relay_step calls leave in the two
// buffers).  Each step is the node kernel's arithmetic in the node kernel's
// order, so the result equals k relay_step calls bit for bit.
// The CTA's step barrier (barrier 1): its warps may reach it at different
// places in the code, one per number of neighbours.
__device__ __forceinline__ void cta_barrier() { asm volatile("bar.sync 1, %0;" ::"r"(blockDim.x) : "memory"); }

// Both message buffers are written before the launch ends (the one that step
// t0 reads holds the messages of one of the last two steps), so they are read
// with ordinary loads, not non-coherent ones.
//
// One launch's k steps of one quad for a warp whose workers all have at most
// D neighbours (D <= kRegDeg; a lane with fewer skips the missing ones).
// The messages that arrived at the step before are registers m: they are read
// from shared memory once, for the rebuild, and serve the next step's
// outgoing messages from there.  One barrier per step: a buffer is written
// again two steps later, when every thread has passed the barrier between,
// that is finished reading it.  The next step's noise, which depends on
// nothing here, is drawn between the loads of the new messages and their use.
template <int D, int OPT, bool PLAIN>
__device__ __forceinline__ void fused_steps(const Program& prog, const ModelArgs& a, const FusedSteps& fs,
                                            const NodeThread& t, const float2* factors, float4* buf, int buf_len,
                                            int qb, int& parity, bool active, int64_t q, float4& xv, float4 mv,
                                            float4& m1, float4& m2) {
    constexpr int DN = D > 0 ? D : 1;
    float4 m[DN];
    int out[DN];
#pragma unroll
    for (int s = 0; s < D; ++s) {
        m[s] = nothing4();
        out[s] = 0;
        if (s < t.deg) {
            // where the message to neighbour s arrives
            out[s] = prog.edge_pos[prog.pos_out[t.pos_base + s]] * qb + (t.in - t.pos_base * qb);
            if (active) m[s] = *reinterpret_cast<const float4*>(a.msg_in + prog.pos_in[t.pos_base + s] * a.ld_m + 4 * q);
        }
    }
    const NoiseQuad nq = noise_quad(a.q0 + static_cast<uint32_t>(q), a.key);
    const uint32_t row = static_cast<uint32_t>(t.i);
    float4 z = minus_normal4(noise_words(nq, row, a.step, a.key));
    float2 f = make_float2(0.f, 0.f);
    for (int j = 0; j < fs.k; ++j) {
        const float st = (OPT == 2) ? fs.adam_step[j] : 0.0f, ib = (OPT == 2) ? fs.adam_ibc2[j] : 0.0f;
        const float4 xh =
            relayed_with<OPT, PLAIN>(a, xv, mv, z, [&](float4 g) { return update_rule<OPT>(a, st, ib, g, m1, m2); });
        if (D > 0 && j + 1 == fs.k && j > 0 && active) {  // m^{t0+k-2}, before it is replaced
#pragma unroll
            for (int s = 0; s < D; ++s)
                if (s < t.deg)
                    st_stream(fs.msg[j & 1] + prog.pos_in[t.pos_base + s] * a.ld_m + 4 * q, m[s]);
        }
        float4* const cur = buf + (parity ? buf_len : 0);
        parity ^= 1;
        if (D > 0) {
            float4 o[DN];
            narrow_messages<DN>(m, xh, t.lost_bits, o);
#pragma unroll
            for (int s = 0; s < D; ++s)
                if (s < t.deg) cur[out[s]] = o[s];
        }
        cta_barrier();
        if (D > 0) {
#pragma unroll
            for (int s = 0; s < D; ++s)
                if (s < t.deg) m[s] = cur[t.in + s * qb];
        }
        if (j < fs.rounds) f = factors[j * prog.n + t.i];  // (scale, fill)
        z = minus_normal4(noise_words(nq, row, a.step + static_cast<uint32_t>(j) + 1u, a.key));
        float4 acc = xh;
        if (f.y != 0.0f) acc = fma4(f.y, xv, acc);
#pragma unroll
        for (int s = 0; s < D; ++s) acc = add4(acc, m[s]);
        xv = scale4(acc, f.x);
    }
    if (D > 0 && active) {
        float* const last = fs.msg[fs.k & 1];
#pragma unroll
        for (int s = 0; s < D; ++s)
            if (s < t.deg) st_stream(last + prog.pos_in[t.pos_base + s] * a.ld_m + 4 * q, m[s]);
    }
}

// The same for a warp with a worker of degree > kRegDeg (a star's hub): the
// messages that arrived at the step before stay in shared memory, in the
// worker's own rows of the other buffer, and the outgoing ones are formed as
// node_send_wide forms them.
template <int OPT>
__device__ __noinline__ void fused_steps_wide(const Program& prog, const ModelArgs& a, const FusedSteps& fs,
                                              const NodeThread& t, const float2* factors, float4* buf, int buf_len,
                                              int qb, int& parity, bool active, int64_t q, float4& xv, float4 mv,
                                              float4& m1, float4& m2) {
    const float4 zero = make_float4(0.f, 0.f, 0.f, 0.f);
    const int qi = t.in - t.pos_base * qb;
    const NoiseQuad nq = noise_quad(a.q0 + static_cast<uint32_t>(q), a.key);
    float4* const first = buf + (parity ? 0 : buf_len) + t.in;
    for (int s = 0; s < t.deg; ++s)
        first[s * qb] =
            active ? *reinterpret_cast<const float4*>(a.msg_in + prog.pos_in[t.pos_base + s] * a.ld_m + 4 * q) : zero;
    for (int j = 0; j < fs.k; ++j) {
        float4* const cur = buf + (parity ? buf_len : 0);
        const float4* const prev = buf + (parity ? 0 : buf_len) + t.in;
        parity ^= 1;
        const float4 z = minus_normal4(noise_words(nq, static_cast<uint32_t>(t.i), a.step + static_cast<uint32_t>(j),
                                                   a.key));
        const float4 xh = relayed_with<OPT, false>(a, xv, mv, z, [&](float4 g) {
            return update_rule<OPT>(a, fs.adam_step[j], fs.adam_ibc2[j], g, m1, m2);
        });
        if (j + 1 == fs.k && j > 0 && active)  // m^{t0+k-2}
            for (int s = 0; s < t.deg; ++s)
                st_stream(fs.msg[j & 1] + prog.pos_in[t.pos_base + s] * a.ld_m + 4 * q, prev[s * qb]);
        float4 total = xh;
        if (t.deg > kRegDeg)
            for (int s = t.deg - 1; s >= 0; --s) total = add4(total, prev[s * qb]);
        for (int s = 0; s < t.deg; ++s) {
            float4 o;
            if (t.deg > kRegDeg) {
                o = sub4(total, prev[s * qb]);
            } else {
                float4 pre = xh;
                for (int r = 0; r < s; ++r) pre = add4(pre, prev[r * qb]);
                o = pre;
                if (s + 1 < t.deg) {
                    float4 suf = prev[(t.deg - 1) * qb];
                    for (int r = t.deg - 2; r > s; --r) suf = add4(prev[r * qb], suf);
                    o = add4(pre, suf);
                }
            }
            const int e = prog.pos_out[t.pos_base + s];
            cur[prog.edge_pos[e] * qb + qi] = delivered(a, e, o);
        }
        cta_barrier();
        const float2 f = factors[min(j, fs.rounds - 1) * prog.n + t.i];
        float4 acc = xh;
        if (f.y != 0.0f) acc = fma4(f.y, xv, xh);
        for (int s = 0; s < t.deg; ++s) acc = add4(acc, cur[t.in + s * qb]);
        xv = scale4(acc, f.x);
    }
    if (active) {
        const float4* const last = buf + (parity ? 0 : buf_len) + t.in;
        for (int s = 0; s < t.deg; ++s)
            st_stream(fs.msg[fs.k & 1] + prog.pos_in[t.pos_base + s] * a.ld_m + 4 * q, last[s * qb]);
    }
}

// blockDim.x = qb * n rounded up to whole warps, at most THREADS; qb
// consecutive threads share a worker, the workers in ascending degree, so
// that the workers of one warp have (nearly) the same number of neighbours
// and no lane waits for another's longer code path.  Dynamic shared memory:
// two [E][qb] float4 message buffers, row p holding the message that arrives
// at position p (so a worker reads consecutive rows), then the rebuild
// factors (scale, fill) of every worker and counter round, [rounds][n]
// float2.  The counters, hence the factors, are the same for every quad: the
// CTA advances them once, before its first quads.
//
// THREADS: up to 32 workers take CTAs of at most 256 threads, three per SM
// with 80 registers, where the barrier holds fewer warps and less spills
// (nothing with SGD, 4 bytes with Nesterov and 36 with Adam, against 84 to 176
// with 64 registers): against 512 threads, two per SM with 64 registers, 510 ->
// 491 us (16-worker binary tree, d = 272,474, 64 steps), 30.7 -> 28.7 us
// (8-worker chain, d = 4,096), 806 -> 785 us with Adam.  More workers keep 512,
// since half of it would leave rows of 4 quads: 362 against 351 us on the
// 64-worker chain at d = 30,001.  Every build has a stack frame, for the
// arguments that fused_steps_wide takes by reference.
constexpr int kFusedFewWorkers = 32;
constexpr int fused_threads(int n) { return n <= kFusedFewWorkers ? 256 : 512; }

template <int OBJ, int OPT, bool PLAIN, int THREADS>
__global__ void __launch_bounds__(THREADS, THREADS == 256 ? 3 : 2)
relay_fused_steps_kernel(const __grid_constant__ Program prog, const __grid_constant__ ObjectiveArg<OBJ> obj,
                         const __grid_constant__ PhiloxKey mu_key, const __grid_constant__ ModelArgs a,
                         const __grid_constant__ FusedSteps fs) {
    allow_dependent_launch();  // the counter kernel behind this one waits for all of it before it writes
    extern __shared__ float4 fused_mem[];
    __shared__ int32_t c_mem[2][kMaxE];  // counters of the round parities
    constexpr int kObj = (OBJ == relaysum::kMuStored) ? relaysum::kMuStored : relaysum::kMuPerRow;
    const int tid = static_cast<int>(threadIdx.x);
    const int qb = 1 << fs.qb_log2;
    const int n = prog.n;
    const int E = prog.E;
    float2* const factors = reinterpret_cast<float2*>(fused_mem + 2 * E * qb);  // [round * n + i]
    for (int e = tid; e < E; e += blockDim.x) c_mem[1][e] = a.counts[e];  // c^{t0-1}
    __syncthreads();
    for (int j = 0; j < fs.rounds; ++j) {
        const int32_t* const c_old = c_mem[(j + 1) & 1];
        int32_t* const c_new = c_mem[j & 1];
        for (int e = tid; e < E; e += blockDim.x) c_new[e] = next_count(prog, a.lost, a.has_lost, c_old, e);
        __syncthreads();
        for (int w = tid; w < n; w += blockDim.x) {
            const NodeRec rw = prog.node[w];
            int nbar = 1;
            for (int p = 0; p < rw.deg; ++p) nbar += c_new[prog.pos_in[rw.pos_base + p]];
            float scale, fill;
            worker_factors(a, n, nbar, scale, fill);
            factors[j * n + w] = make_float2(scale, fill);
        }
    }
    __syncthreads();
    const int slot = tid >> fs.qb_log2;
    const int qi = tid & (qb - 1);
    const bool live = slot < n;
    const NodeThread t = node_thread(prog, a, slot, qi, qb);
    const int widest = __reduce_max_sync(0xffffffffu, t.deg);
    const float4 zero = make_float4(0.f, 0.f, 0.f, 0.f);
    const int64_t nblk = (a.nquads + qb - 1) >> fs.qb_log2;
    int parity = 0;
    for (int64_t b = blockIdx.x; b < nblk; b += gridDim.x) {
        const int64_t q = (b << fs.qb_log2) + qi;
        const bool active = live && q < a.nquads;
        float4 xv = zero, mv = zero, m1 = zero, m2 = zero;
        if (active) {
            xv = *reinterpret_cast<const float4*>(a.x + t.i * a.ld_x + 4 * q);
            mv = (OBJ == relaysum::kMuStored) ? ld_stream(a.mu + t.i * a.ld_x + 4 * q)
                                               : centre<kObj>(obj, mu_key, a, t.i, q, nullptr, 0);
            if (OPT >= 1) m1 = *reinterpret_cast<const float4*>(a.s1 + t.i * a.ld_x + 4 * q);
            if (OPT == 2) m2 = *reinterpret_cast<const float4*>(a.s2 + t.i * a.ld_x + 4 * q);
        }
        switch (widest) {
#define RELAY_FUSED(D) \
    fused_steps<D, OPT, PLAIN>(prog, a, fs, t, factors, fused_mem, E * qb, qb, parity, active, q, xv, mv, m1, m2)
            case 0: RELAY_FUSED(0); break;
            case 1: RELAY_FUSED(1); break;
            case 2: RELAY_FUSED(2); break;
            case 3: RELAY_FUSED(3); break;
            case 4: RELAY_FUSED(4); break;
#undef RELAY_FUSED
            default:
                fused_steps_wide<OPT>(prog, a, fs, t, factors, fused_mem, E * qb, qb, parity, active, q, xv, mv, m1,
                                      m2);
                break;
        }
        if (active) {
            st_stream(a.x + t.i * a.ld_x + 4 * q, xv);
            if (OPT >= 1) st_stream(a.s1 + t.i * a.ld_x + 4 * q, m1);
            if (OPT == 2) st_stream(a.s2 + t.i * a.ld_x + 4 * q, m2);
        }
    }
}

// ------------------------------------------------------------------ launches

[[maybe_unused]] const relaysum::Program& pick(const relay_handle* h, const relaysum::Program*) { return h->prog; }
[[maybe_unused]] const relaysum::SmallProgram& pick(const relay_handle* h, const relaysum::SmallProgram*) { return h->small_prog; }
[[maybe_unused]] const relaysum::Objective& pick(const relay_handle* h, const relaysum::Objective*) { return h->obj; }
[[maybe_unused]] const relaysum::SmallObjective& pick(const relay_handle* h, const relaysum::SmallObjective*) { return h->small_obj; }
[[maybe_unused]] NoObjective pick(const relay_handle*, const NoObjective*) { return NoObjective{0}; }

// The handle's program and objective at this capacity.
const Program& program_of(const relay_handle* h) { return pick(h, static_cast<const Program*>(nullptr)); }
template <int OBJ>
ObjectiveArg<OBJ> objective_of(const relay_handle* h) {
    return pick(h, static_cast<const ObjectiveArg<OBJ>*>(nullptr));
}

// Threads per CTA for the fused kernel: 128, fewer when the slots would not
// fit in shared memory.
int models_threads(int nslots) {
    int t = 128;
    while (t > 32 && static_cast<int64_t>(nslots) * t * 16 > kMaxSmem) t -= 32;
    return t;
}

// Threads per CTA and shared memory of the walk over NT handles' windows,
// sized for the larger program.
struct WalkShape {
    int threads;
    size_t smem;
};

template <int OBJ, int NT>
WalkShape walk_shape(const relay_handle* const* hs) {
    int per_thread = 0;
    for (int k = 0; k < NT; ++k)
        per_thread = std::max(per_thread, hs[k]->prog.nslots + (OBJ == relaysum::kMuCachedCentres ? hs[k]->obj.K : 0));
    const int threads = models_threads(per_thread);
    return WalkShape{threads, static_cast<size_t>(per_thread) * threads * 16};
}

// The walk over NT handles' windows in one launch (NT = 1: one handle).  The
// handles share the objective source and the local optimiser (the caller
// checks).
template <int OBJ, int OPT, int NT, bool WIDE, int MIN>
int launch_models(const relay_handle* const* hs, const ModelArgs* as, cudaStream_t stream, bool after_counts) {
    int dev = 0;
    const int sms = device_sms(&dev);
    if (sms <= 0) return RELAY_ECUDA;
    const auto [threads, smem] = walk_shape<OBJ, NT>(hs);
    if (smem > static_cast<size_t>(kMaxSmem)) return RELAY_EUNSUPPORTED;
    if (resident_ctas<relay_models_kernel<OBJ, OPT, NT, WIDE, MIN>>(dev, threads, smem) <= 0) return RELAY_ECUDA;
    Windows<NT> win;
    int64_t grid = 0;  // a quad per thread: at most 2^27 CTAs a window
    for (int k = 0; k < NT; ++k) {
        if (k == NT - 1) win.split = static_cast<int32_t>(grid);
        grid += (as[k].nquads + threads - 1) / threads;
        win.prog[k] = program_of(hs[k]);
        win.a[k] = as[k];
    }
    const PhiloxKey mu_key =
        philox_key(static_cast<uint64_t>(hs[0]->obj.k0) | (static_cast<uint64_t>(hs[0]->obj.k1) << 32));
    return launch_step_kernel(relay_models_kernel<OBJ, OPT, NT, WIDE, MIN>, static_cast<int>(grid), threads, smem, stream,
                              after_counts, win, objective_of<OBJ>(hs[0]), mu_key);
}

// Quads per CTA of the node-parallel kernel, as a power of two: as many as
// fill kNodeThreads, at most a warp's worth (a whole warp per worker up to 16
// workers).
int nodes_qb_log2(int n) {
    int l = 5;
    while (l > 0 && (n << l) > kNodeThreads) --l;
    return l;
}

template <int OBJ, int OPT>
int launch_nodes(const relay_handle* h, const ModelArgs& a, cudaStream_t stream, bool after_counts) {
    int dev = 0;
    const int sms = device_sms(&dev);
    if (sms <= 0) return RELAY_ECUDA;
    const int qb_log2 = nodes_qb_log2(h->prog.n);
    const int threads = ((h->prog.n << qb_log2) + 31) / 32 * 32;
    const size_t smem = (static_cast<size_t>(has_wide(h) ? 3 : 2) * h->prog.E << qb_log2) * 16;
    if (smem > static_cast<size_t>(kMaxSmem)) return RELAY_EUNSUPPORTED;
    const int per_sm = resident_ctas<relay_nodes_kernel<OBJ, OPT>>(dev, threads, smem);
    if (per_sm <= 0) return RELAY_ECUDA;
    const int64_t want = (a.nquads + (int64_t(1) << qb_log2) - 1) >> qb_log2;
    const int64_t cap = static_cast<int64_t>(sms) * per_sm;
    const int grid = static_cast<int>(want < cap ? want : cap);
    const PhiloxKey mu_key = philox_key(static_cast<uint64_t>(h->obj.k0) | (static_cast<uint64_t>(h->obj.k1) << 32));
    return launch_step_kernel(relay_nodes_kernel<OBJ, OPT>, grid, threads, smem, stream, after_counts,
                              program_of(h), objective_of<OBJ>(h), mu_key, a, qb_log2);
}

// Whether the walk over narrow trees with stored centres takes the build
// budgeted for 7 CTAs per SM rather than the unbounded one (8 of 128 threads,
// unless the slots allow fewer).  More CTAs are faster over many waves, but a
// short grid's last wave leaves SMs idle, and it is fuller when 7 at a time
// divide the grid better.  Each side at 16 to 64 workers, 7 against 8:
//   1.6 to 4.0 waves of 8, SGD       0.94 to 1.00 of the time (torus tree of 64
//                                    workers at d = 1.0M: 272 against 286 us)
//   the same, Adam                   0.97 to 1.01 (453 against 459 us)
//   the same, Nesterov               0.98 to 1.025 (32 workers at d = 1.0M: 182
//                                    against 185 us; 64 at 1.5M: 554 against 543)
//   0.9 to 1 wave of 8               1.2 to 1.4
//   more than four                   1.01 to 1.06 (32-worker binary tree at d =
//                                    9.2M: 1,124 against 1,109 us with SGD)
template <int OPT, int NT>
bool seven_ctas(const relay_handle* const* hs, const ModelArgs* as) {
    int dev = 0;
    const int64_t sms = device_sms(&dev);
    const auto [threads, smem] = walk_shape<relaysum::kMuStored, NT>(hs);
    if (sms <= 0 || smem > static_cast<size_t>(kMaxSmem)) return false;  // the launch reports it
    const int most = resident_ctas<relay_models_kernel<relaysum::kMuStored, OPT, NT, false, 0>>(dev, threads, smem);
    const int fewer = resident_ctas<relay_models_kernel<relaysum::kMuStored, OPT, NT, false, 7>>(dev, threads, smem);
    if (fewer <= 0 || fewer >= most) return false;
    int64_t ctas = 0;
    for (int k = 0; k < NT; ++k) ctas += (as[k].nquads + threads - 1) / threads;
    auto slots = [&](int64_t per_sm) { return (ctas + sms * per_sm - 1) / (sms * per_sm) * per_sm; };
    // share of the CTA slots that the waves fill, ctas / (waves x slots): 10 % fuller
    return 10 * slots(most) > 11 * slots(fewer);
}

template <int OPT, int NT, bool WIDE>
int launch_walk_src(const relay_handle* const* hs, const ModelArgs* as, cudaStream_t stream, bool after_counts) {
    switch (hs[0]->obj.source) {
        case relaysum::kMuStored:
            if constexpr (!WIDE)
                if (seven_ctas<OPT, NT>(hs, as))
                    return launch_models<relaysum::kMuStored, OPT, NT, WIDE, 7>(hs, as, stream, after_counts);
            return launch_models<relaysum::kMuStored, OPT, NT, WIDE, WIDE ? 8 : 0>(hs, as, stream, after_counts);
        case relaysum::kMuPerRow:
            return launch_models<relaysum::kMuPerRow, OPT, NT, WIDE, WIDE ? 8 : 0>(hs, as, stream, after_counts);
        default:
            return launch_models<relaysum::kMuCachedCentres, OPT, NT, WIDE, WIDE ? 8 : 0>(hs, as, stream, after_counts);
    }
}

// One handle: the WIDE variant when its tree has a wide node.  Several
// windows (relay_step_windows) launch together only when none has one.
template <int OPT, int NT>
int launch_walk_obj(const relay_handle* const* hs, const ModelArgs* as, cudaStream_t stream, bool after_counts) {
    if (NT == 1 && has_wide(hs[0])) return launch_walk_src<OPT, 1, true>(hs, as, stream, after_counts);
    return launch_walk_src<OPT, NT, false>(hs, as, stream, after_counts);
}

template <int OPT>
int launch_models_obj(const relay_handle* h, const ModelArgs& a, bool nodes, cudaStream_t stream, bool after_counts) {
    if (nodes) {
        if (h->obj.source == relaysum::kMuStored)
            return launch_nodes<relaysum::kMuStored, OPT>(h, a, stream, after_counts);
        return launch_nodes<relaysum::kMuPerRow, OPT>(h, a, stream, after_counts);
    }
    return launch_walk_obj<OPT, 1>(&h, &a, stream, after_counts);
}

// Quads per CTA of relay_fused_steps_kernel (as a power of two): as many as
// fill its threads, at most a warp's worth, halved while that leaves fewer
// CTAs than SMs (short vectors then still spread over the whole GPU) and the
// CTA keeps a full warp.
int fused_qb_log2(int n, int64_t nquads, int sms) {
    int l = 5;
    while (l > 0 && (n << l) > fused_threads(n)) --l;
    while (l > 0 && (n << (l - 1)) >= 32 && (nquads + (int64_t(1) << l) - 1) >> l < sms) --l;
    return l;
}

template <int OBJ, int OPT, bool PLAIN, int THREADS>
int launch_fused(const relay_handle* h, const ModelArgs& a, FusedSteps& fs, cudaStream_t stream) {
    int dev = 0;
    const int sms = device_sms(&dev);
    if (sms <= 0) return RELAY_ECUDA;
    const int n = h->prog.n;
    fs.qb_log2 = fused_qb_log2(n, a.nquads, sms);
    const int threads = ((n << fs.qb_log2) + 31) / 32 * 32;
    const size_t smem = (static_cast<size_t>(2) * h->prog.E << fs.qb_log2) * 16 + static_cast<size_t>(fs.rounds) * n * 8;
    if (smem > static_cast<size_t>(kMaxSmem)) return RELAY_EUNSUPPORTED;
    const int per_sm = resident_ctas<relay_fused_steps_kernel<OBJ, OPT, PLAIN, THREADS>>(dev, threads, smem);
    if (per_sm <= 0) return RELAY_ECUDA;
    const int64_t want = (a.nquads + (int64_t(1) << fs.qb_log2) - 1) >> fs.qb_log2;
    const int64_t cap = static_cast<int64_t>(sms) * per_sm;
    const int grid = static_cast<int>(want < cap ? want : cap);
    const PhiloxKey mu_key = philox_key(static_cast<uint64_t>(h->obj.k0) | (static_cast<uint64_t>(h->obj.k1) << 32));
    relay_fused_steps_kernel<OBJ, OPT, PLAIN, THREADS><<<grid, threads, smem, stream>>>(program_of(h), objective_of<OBJ>(h), mu_key, a, fs);
    return launch_status();
}

template <int OBJ, int OPT, bool PLAIN>
int launch_fused_threads(const relay_handle* h, const ModelArgs& a, FusedSteps& fs, cudaStream_t stream) {
    return fused_threads(h->prog.n) == 256 ? launch_fused<OBJ, OPT, PLAIN, 256>(h, a, fs, stream)
                                           : launch_fused<OBJ, OPT, PLAIN, 512>(h, a, fs, stream);
}

template <int OPT>
int launch_fused_obj(const relay_handle* h, const ModelArgs& a, FusedSteps& fs, cudaStream_t stream) {
    const bool plain = h->algo == RELAY_ALGO_RELAYSGD;
    if (h->obj.source == relaysum::kMuStored)
        return plain ? launch_fused_threads<relaysum::kMuStored, OPT, true>(h, a, fs, stream)
                     : launch_fused_threads<relaysum::kMuStored, OPT, false>(h, a, fs, stream);
    return plain ? launch_fused_threads<relaysum::kMuPerRow, OPT, true>(h, a, fs, stream)
                 : launch_fused_threads<relaysum::kMuPerRow, OPT, false>(h, a, fs, stream);
}

// Window k of a counter launch: handle h's program, lost mask and arrays.
template <int NT>
void count_window(const relay_handle* h, int32_t* counts, CountWindows<NT>& cw, int k) {
    cw.prog[k] = program_of(h);
    std::memcpy(cw.lost[k].w, h->lost, sizeof(cw.lost[k].w));
    cw.has_lost[k] = h->has_lost ? 1 : 0;
    cw.counts[k] = counts;
    cw.dme_count[k] = h->algo == RELAY_ALGO_DME ? h->dme_count : nullptr;
}

}  // namespace

namespace relaysum {
namespace RELAY_SPACE {

int launch_counts(const relay_handle* const* hs, int32_t* const* counts, int windows, cudaStream_t stream) {
    if (windows == 1) {
        CountWindows<1> cw;
        count_window(hs[0], counts[0], cw, 0);
        relay_counts_kernel<1><<<1, 256, 0, stream>>>(cw);
    } else {
        CountWindows<2> cw;
        for (int k = 0; k < 2; ++k) count_window(hs[k], counts[k], cw, k);
        relay_counts_kernel<2><<<2, 256, 0, stream>>>(cw);
    }
    return launch_status();
}

int launch_step(const relay_handle* h, const ModelArgs& a, bool nodes, cudaStream_t stream, bool after_counts) {
    switch (h->opt) {
        case 0: return launch_models_obj<0>(h, a, nodes, stream, after_counts);
        case 1: return launch_models_obj<1>(h, a, nodes, stream, after_counts);
        default: return launch_models_obj<2>(h, a, nodes, stream, after_counts);
    }
}

int launch_step_windows(const relay_handle* const* hs, const ModelArgs* as, cudaStream_t stream, bool after_counts) {
    switch (hs[0]->opt) {
        case 0: return launch_walk_obj<0, 2>(hs, as, stream, after_counts);
        case 1: return launch_walk_obj<1, 2>(hs, as, stream, after_counts);
        default: return launch_walk_obj<2, 2>(hs, as, stream, after_counts);
    }
}

int launch_steps(const relay_handle* h, const ModelArgs& a, FusedSteps& fs, cudaStream_t stream) {
    fs.rounds = settled_rounds(program_of(h), fs.k);
    switch (h->opt) {
        case 0: return launch_fused_obj<0>(h, a, fs, stream);
        case 1: return launch_fused_obj<1>(h, a, fs, stream);
        default: return launch_fused_obj<2>(h, a, fs, stream);
    }
}

int launch_steps_counts(const relay_handle* h, int32_t* counts, int k, cudaStream_t stream, bool after_models) {
    LostMask lost;
    std::memcpy(lost.w, h->lost, sizeof(lost.w));
    const auto& prog = program_of(h);
    return launch_step_kernel(relay_counts_steps_kernel, 1, kCountsThreads, 0, stream, after_models, prog, lost,
                              h->has_lost ? 1 : 0, counts,
                              h->algo == RELAY_ALGO_DME ? h->dme_count : static_cast<int64_t*>(nullptr), k,
                              settled_rounds(prog, k));
}

}  // namespace RELAY_SPACE
}  // namespace relaysum

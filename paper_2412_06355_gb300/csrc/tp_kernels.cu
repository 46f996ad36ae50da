// Time-parallel DendSN kernels for narrow layers with long horizons (few neurons, large T,
// e.g. the L5PC fitting neuron: T = 2048, 16 neurons). One block serves one neuron.
//
// The horizon is cut into 32 segments of TB = ceil(T / 32) steps, one per lane of a warp, and
// every series of the neuron sits in shared memory as [step of the segment][segment], so that
// a warp walking its segments and a block sweeping all steps both read without bank conflicts.
//
// The compartment recursion V^d_i[t] = alpha_i V^d_i[t-1] + X_i[t] (Eq. methods-compartment)
// is linear, so it is scanned in parallel over time, one warp per compartment: each lane first
// scans its segment from a zero state, keeping the end state e and alpha^len; a 5-step warp scan
// composes the segments ((p2, e2) o (p1, e1) = (p2 p1, p2 e1 + e2)) and gives every lane the
// state entering its segment; a second pass then produces V^d[t]. Z[t] (Eqs.
// methods-branch-aggregation .. methods-soma-input) depends on V^d[t] alone: all threads share
// the steps. The soma (Eq. methods-lif-reset-charge, -fire) is not linear; it is run by one
// warp, all segments at once from guessed states that are then made exact (tp_soma_run).
//
// The backward recomputes V^d, Z and V^s the same way (so spikes match the forward's bit for
// bit). Given the trajectory the soma's reverse recursion (Eq. methods-sg) is linear in
// dL/dV^s, and the compartment adjoint A_i[t] = direct_i[t] + alpha_i A_i[t+1] is linear again:
// both take the same segment scan in reverse time, everything else all threads. Parameter-gradient
// sums are reduced over the block in a fixed order, and summed per channel by tp_finalize_kernel
// in a fixed order: deterministic. Nothing is checkpointed: the forward leaves `saved` untouched.
//
// Latency bounds these kernels (16 neurons leave most of the GPU idle). With one warp per
// neuron doing all of it, 32-way bank conflicts and 2048 serial soma steps the L5PC layer took
// 31 + 93 us (forward + backward and finalize) on GB300; it takes 12 + 19. A block's time
// there (forward, in cycles): inputs 4000, scans 4500, Z 1000, soma 7500, spikes 2200.
#include <algorithm>

#include "dendsn_kernels.cuh"

namespace dendsn {

namespace {

// Threads per neuron (smem bytes each): no more than two steps each, and as few as let every
// block that shared memory admits be resident at about 110 registers a thread. A lone neuron's
// latency shrinks with its threads, but blocks that wait for a place cost more: 2000 neurons of
// 300 bfloat16 steps forward take 20 us with 64 threads, which need two waves, and 16 with 32;
// where shared memory already sets the waves more threads help (2048 neurons of 2048 steps
// backward: 364 us with 32, 205 with 128).
int tp_threads(int T, int64_t BN, size_t smem) {
    const int64_t per_sm = std::min<int64_t>((BN + 151) / 152, std::max<int64_t>(1, (227 << 10) / (int64_t)(smem + 2048)));
    int n = 512;
    while (n > 32 && (n * per_sm > 576 || n * 2 > T)) n /= 2;
    return n;
}
constexpr int kTpMaxThreads = 512;

// The neuron's parameters: every thread holds all K compartments.
template <int K, int G>
struct TpParams {
    static constexpr int Kb = K / G;
    float nxi[K], iz[Kb], km[Kb], mk[Kb];
    float xi[K], zeta[Kb], kap[Kb];
    typename MaskRaw<Kb < 8 ? Kb : 8>::T m[Kb < 8 ? 1 : Kb / 8];
    // Requests the parameters (before the inputs are staged, so that the two latencies overlap) ...
    __device__ __forceinline__ void fetch(const Params &P, const Geometry &g, int64_t n, int chan) {
#pragma unroll
        for (int b = 0; b < Kb; ++b) {
            zeta[b] = __ldg(P.zeta + (int64_t)chan * Kb + b);
            kap[b] = __ldg(P.kappa + (int64_t)chan * Kb + b);
        }
#pragma unroll
        for (int i = 0; i < K; ++i) xi[i] = __ldg(P.xi + (int64_t)chan * K + i);
        if (P.mask_mode != 0) {
            const uint8_t *p = P.mask + (P.mask_mode == 2 ? n : (int64_t)chan) * Kb;
#pragma unroll
            for (int h = 0; h < (Kb < 8 ? 1 : Kb / 8); ++h) m[h] = fetch_mask<(Kb < 8 ? Kb : 8)>(p + 8 * h);
        }
    }
    // ... and forms what the steps use (load_param_arrays' and apply_neuron_mask's operations: a
    // per-neuron mask selects, so that a masked branch's kappa plays no part, whatever its value).
    __device__ __forceinline__ void form(const Params &P) {
        constexpr int MB = Kb < 8 ? Kb : 8;
#pragma unroll
        for (int b = 0; b < Kb; ++b) {
            iz[b] = __frcp_rn(zeta[b]);
            mk[b] = 1.f;
        }
#pragma unroll
        for (int i = 0; i < K; ++i) nxi[i] = -__fmul_rn(xi[i], iz[i / G]);
        if (P.mask_mode != 0) {
#pragma unroll
            for (int h = 0; h < Kb / MB; ++h) {
                float t[MB];
                unpack_mask<MB>(m[h], t);
#pragma unroll
                for (int b = 0; b < MB; ++b) mk[h * MB + b] = t[b];
            }
        }
#pragma unroll
        for (int b = 0; b < Kb; ++b)
            km[b] = P.mask_mode == 2 ? (mk[b] != 0.f ? kap[b] : 0.f) : __fmul_rn(kap[b], mk[b]);
    }
};

// u, r^2 and what follows from them for branch b of a step with compartment potentials vd.
template <int K, int G>
__device__ __forceinline__ float tp_branch_ss(const TpParams<K, G> &q, int b, const float *vd, float (&u)[G]) {
    float ss = 0.f;
#pragma unroll
    for (int i = 0; i < G; ++i) {
        u[i] = __fmaf_rn(vd[i], q.iz[b], q.nxi[b * G + i]);
        ss = (i == 0) ? __fmul_rn(u[i], u[i]) : __fmaf_rn(u[i], u[i], ss);
    }
    return ss;
}

// Z[t] from V^d[t], without the residual term.
template <int K, int G>
__device__ __forceinline__ float tp_soma_input(const TpParams<K, G> &q, const float (&vd)[K], int psi) {
    constexpr int Kb = K / G;
    float z = 0.f;
#pragma unroll
    for (int b = 0; b < Kb; ++b) {
        float u[G];
        const float ss = tp_branch_ss<K, G>(q, b, &vd[b * G], u);
        float y;
        if (psi == PSI_MEXHAT) {
            const float e = gauss_half(ss);
            y = __fmaf_rn(-ss, e, e);                          // (1 - r^2) e^{-r^2/2}
        } else {
            y = sqrtf(ss);                                     // r
        }
        z = (b == 0) ? __fmul_rn(q.km[b], y) : __fmaf_rn(q.km[b], y, z);
    }
    return z;
}

// Below these many steps the soma runs serially: that costs about what guesses that meet do, and half
// of what guesses that never meet do (K = 1, one neuron, forward, us, serial / meet / never: T = 512 6.0 /
// 6.6 / 13, T = 640 7 / 7 / 15, T = 700 8 / 7.4 / 17, T = 1000 11 / 8 / 21).
constexpr int kTpSerial = 704;

// The neuron's place in x and the horizon's segments. Step t = l * TB + s of segment l sits at
// slot s * 32 + l of a plane of `plane` floats.
struct TpGeom {
    int64_t j, n, xo, sX, ks;
    int chan, T, TB, plane;
    bool plain = false;                          // set by tp_forward_pass
    __device__ __forceinline__ TpGeom(const Geometry &g, int layout) {
        j = blockIdx.x;
        n = j % g.N;
        chan = (int)((n / g.inner) % g.C);
        T = g.T;
        TB = (T + 31) >> 5;
        plane = TB * 32;
        sX = g.BN * g.K;
        if (layout == 0) {
            xo = j * g.K;
            ks = 1;
        } else {
            const int64_t s = j % g.inner;
            xo = (j - s) * g.K + s;
            ks = g.inner;
        }
    }
    // V^s of a serial soma is in plain step order
    __device__ __forceinline__ bool serial() const { return T < kTpSerial; }
    __device__ __forceinline__ int v_at(int slot, int t) const { return plain ? t : slot; }
    __device__ __forceinline__ int len(int l) const { return max(0, min(TB, T - l * TB)); }
    // f(slot, t) for every step, the block's threads sharing them; consecutive threads take
    // consecutive segments
    template <typename F>
    __device__ __forceinline__ void sweep(F f) const {
        const int l = threadIdx.x & 31;
        const int n_l = len(l);
        for (int s = threadIdx.x >> 5; s < n_l; s += blockDim.x >> 5) f(s * 32 + l, l * TB + s);
    }
    // the same with the loads of up to NB steps in flight before their uses
    template <int NB, typename L, typename U>
    __device__ __forceinline__ void sweep_loads(L load, U use) const {
        const int l = threadIdx.x & 31, w = blockDim.x >> 5;
        const int n_l = len(l);
        for (int s0 = threadIdx.x >> 5; s0 < n_l; s0 += NB * w) {
#pragma unroll
            for (int b = 0; b < NB; ++b)
                if (s0 + b * w < n_l) load(b, l * TB + s0 + b * w);
#pragma unroll
            for (int b = 0; b < NB; ++b)
                if (s0 + b * w < n_l) use(b, (s0 + b * w) * 32 + l);
        }
    }
};

// x into the planes xv[k]; with the residual term its sum over the compartments into zs. gs (and
// gv) into planes of their own when given.
template <int K, typename XT>
__device__ __forceinline__ void tp_stage(const TpGeom &q, const XT *x, int layout, bool residual, float *xv,
                                         float *zs) {
    constexpr int NB = K >= 16 ? 1 : (K >= 8 ? 2 : 4);
    constexpr int KV = K < 8 ? K : 8;            // compartments per vector
    float v[NB][K];
    q.template sweep_loads<NB>(
        [&](int b, int t) {
            const XT *p = x + q.xo + (int64_t)t * q.sX;
            if (layout == 0) {
#pragma unroll
                for (int h = 0; h < K / KV; ++h) {
                    float w[KV];
                    Vec<XT, KV>::unpack(Vec<XT, KV>::load(p + h * KV), w);
#pragma unroll
                    for (int k = 0; k < KV; ++k) v[b][h * KV + k] = w[k];
                }
            } else {
#pragma unroll
                for (int k = 0; k < K; ++k) v[b][k] = Scalar<XT>::unpack(Scalar<XT>::load(p + k * q.ks));
            }
        },
        [&](int b, int slot) {
#pragma unroll
            for (int k = 0; k < K; ++k) xv[k * q.plane + slot] = v[b][k];
            if (residual) {
                float xs = v[b][0];
#pragma unroll
                for (int k = 1; k < K; ++k) xs = __fadd_rn(xs, v[b][k]);
                zs[slot] = xs;
            }
        });
}

// n dependent steps in batches of 8: a batch's loads (two values each) are issued before the
// chain of the batch before it and its stores come after its own, so that only the chain is
// serial.
template <typename Load, typename Step, typename Store>
__device__ __forceinline__ void tp_steps(int n, Load load, Step step, Store store) {
    constexpr int U = 8;
    const int nb = n / U * U;
    float a[U], b[U];
    if (nb > 0) {
#pragma unroll
        for (int u = 0; u < U; ++u) load(u, a[u], b[u]);
    }
#pragma unroll 1
    for (int i = 0; i < nb; i += U) {
        float na[U], nbv[U];
        if (i + U < nb) {
#pragma unroll
            for (int u = 0; u < U; ++u) load(i + U + u, na[u], nbv[u]);
        }
#pragma unroll
        for (int u = 0; u < U; ++u) a[u] = step(i + u, a[u], b[u]);
#pragma unroll
        for (int u = 0; u < U; ++u) {
            store(i + u, a[u]);
            a[u] = na[u];
            b[u] = nbv[u];
        }
    }
    if (nb == n) return;
#pragma unroll
    for (int u = 0; u < U - 1; ++u)
        if (nb + u < n) load(nb + u, a[u], b[u]);
#pragma unroll
    for (int u = 0; u < U - 1; ++u)
        if (nb + u < n) a[u] = step(nb + u, a[u], b[u]);
#pragma unroll
    for (int u = 0; u < U - 1; ++u)
        if (nb + u < n) store(nb + u, a[u]);
}

// The linear recursion y[t] = c[t] y[t-1] + x[t] over a warp's segments, x -> y in place
// (REV: from the last step to the first). c: a constant, or a plane of its own.
template <bool REV, typename C>
__device__ __forceinline__ void tp_scan(const TpGeom &q, C coef, const float *x, float *y) {
    const int l = threadIdx.x & 31;
    const int n = q.len(l);
    auto slot_of = [&](int i) { return (REV ? n - 1 - i : i) * 32 + l; };
    float e = 0.f, pw = 1.f;                     // the segment from a zero state
    tp_steps(n, [&](int i, float &c, float &v) { c = coef(slot_of(i)); v = x[slot_of(i)]; },
             [&](int, float c, float v) {
                 e = __fmaf_rn(c, e, v);
                 pw = __fmul_rn(pw, c);
                 return 0.f;
             },
             [](int, float) {});
    // compose the segments over the lanes (inclusive scan), then shift by one lane
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
        const float pa = REV ? __shfl_down_sync(0xffffffffu, pw, d) : __shfl_up_sync(0xffffffffu, pw, d);
        const float pe = REV ? __shfl_down_sync(0xffffffffu, e, d) : __shfl_up_sync(0xffffffffu, e, d);
        if (REV ? l + d < 32 : l >= d) {
            e = __fmaf_rn(pw, pe, e);
            pw = __fmul_rn(pw, pa);
        }
    }
    const float s = REV ? __shfl_down_sync(0xffffffffu, e, 1) : __shfl_up_sync(0xffffffffu, e, 1);
    float st = l == (REV ? 31 : 0) ? 0.f : s;
    tp_steps(n, [&](int i, float &c, float &v) { c = coef(slot_of(i)); v = x[slot_of(i)]; },
             [&](int, float c, float v) { return st = __fmaf_rn(c, st, v); },
             [&](int i, float v) { y[slot_of(i)] = v; });
}

// One soma step (Eq. methods-lif-reset-charge) shaped for a short dependency chain. Hard
// reset: keep = 1.0 while V < theta (PTX set.lt gives the float, no predicate), then
// V' = keep * (beta V) + Z, so the compare and beta V both start from V (measured 16% faster
// than a compare-and-select). Soft reset: V' = beta (V - theta S) + Z with S as a float likewise.
__device__ __forceinline__ float tp_keep(float v, float theta) {
    float k;
    asm("set.lt.f32.f32 %0, %1, %2;" : "=f"(k) : "f"(v), "f"(theta));
    return k;
}

template <bool SOFT>
__device__ __forceinline__ float tp_charge(float z, float v, float beta, float theta) {
    if constexpr (SOFT) {
        float spike;
        asm("set.ge.f32.f32 %0, %1, %2;" : "=f"(spike) : "f"(v), "f"(theta));
        return __fmaf_rn(beta, __fmaf_rn(-theta, spike, v), z);   // V - theta S: one rounding
    }
    return __fmaf_rn(tp_keep(v, theta), __fmul_rn(beta, v), z);
}

// The soma serially: Z in plain step order in vs, replaced by V^s. Below kTpSerial steps the whole
// horizon costs no more this way than a guess and its rounds. One thread runs it: it reads Z two vectors ahead of the
// words it overwrites, so a second thread running the same loop could find V^s where it expects Z
// (nothing orders the lanes of a warp). The barrier after it publishes V^s.
// Not inlined: its copies (both resets, both callers) cost every layer instruction fetches (T = 2048,
// one neuron, backward, against the kernel with one caller's copies: 1.01 times with both, 0.97 so).
template <bool SOFT>
__device__ __noinline__ void tp_soma_serial(int T, float beta, float theta, float *vs) {
    float v = SOFT && theta <= 0.f ? theta : 0.f;      // the state before a first step (tp_soma_run)
    float4 *p = reinterpret_cast<float4 *>(vs);        // planes hold a whole number of 32 steps
    float4 a = p[0], b = p[1];
    for (int t = 0; t < T; t += 8, p += 2) {
        const bool more = t + 8 < T;
        const float4 na = more ? p[2] : a, nb = more ? p[3] : b;
        float z[8] = {a.x, a.y, a.z, a.w, b.x, b.y, b.z, b.w};
#pragma unroll
        for (int u = 0; u < 8; ++u) z[u] = v = tp_charge<SOFT>(z[u], v, beta, theta);
        p[0] = make_float4(z[0], z[1], z[2], z[3]);
        p[1] = make_float4(z[4], z[5], z[6], z[7]);
        a = na;
        b = nb;
    }
}

// Soma over Z[t] (zs), V^s[t] to vs, by one warp. The recursion is not linear, but trajectories
// from different states soon coincide exactly (a spike's reset forgets the state; the leak
// shrinks a difference until it rounds away). So every lane guesses the state entering its
// segment by running kTpGuess steps before it from the state of a first step (V = Z), then runs
// its own. The lane before it ends in the state that should have been guessed: lanes whose guess
// is not that state, bit for bit, run their segment again from it, for a few rounds (segment 0 is
// exact, so after round r segments 0 .. r are); what still differs then is run segment after
// segment, or, when that is more than a few, the horizon serially in plain step order (then the
// result is true, and vs in that order). What is kept is always the serial recursion's own
// operations on its own values. The usual cost is the guess and a segment or two instead of the
// horizon; the worst case (guesses that never meet, e.g. a soft reset with beta near 1) adds the
// serial work. Forward, K = 4, G = 2, us: one neuron of 2048 steps 10 when guesses meet and 31 when they
// never do (36 with the segments one after the other), of 2400 steps 12 and 36 (44), 2048 neurons of
// 2400 steps 117 and 238 (279).
constexpr int kTpGuess = 192, kTpRounds = 4, kTpFew = 12;

template <bool SOFT>
__device__ __forceinline__ bool tp_soma_run(const TpGeom &q, float beta, float theta, const float *zs, float *vs) {
    const int l = threadIdx.x & 31;
    const int n = q.len(l);
    // segment r (n_r steps) from the state `start`, V^s to vs; returns its last state
    auto segment = [&](int r, int n_r, float start) {
        float w = start;
        tp_steps(n_r, [&](int i, float &z, float &) { z = zs[i * 32 + r]; },
                 [&](int, float z, float) { return w = tp_charge<SOFT>(z, w, beta, theta); },
                 [&](int i, float v) { vs[i * 32 + r] = v; });
        return w;
    };
    // the state before a first step, V^s = Z (no spike before it, whatever theta): its leak is 0
    const float v0 = SOFT && theta <= 0.f ? theta : 0.f;
    float start = v0;
    if (l > 0 && n > 0) {
        const int t0 = max(0, l * q.TB - kTpGuess);
        int r = t0 / q.TB, s = t0 - r * q.TB;            // the guess's first step, and its segment
        for (; r < l; ++r, s = 0) {
            tp_steps(q.TB - s, [&](int i, float &z, float &) { z = zs[(s + i) * 32 + r]; },
                     [&](int, float z, float) { return start = tp_charge<SOFT>(z, start, beta, theta); },
                     [](int, float) {});
        }
    }
    float end = segment(l, n, start);
    for (int round = 0;; ++round) {
        const float before = __shfl_up_sync(0xffffffffu, end, 1);
        const bool again = l > 0 && n > 0 && __float_as_int(before) != __float_as_int(start);
        const unsigned left = __ballot_sync(0xffffffffu, again);
        if (left == 0u) return false;
        if (round == kTpRounds) {
            // both ways rewrite columns that their own lanes wrote in the rounds before, so those
            // writes have to come first (a vote or a shuffle orders no memory)
            __syncwarp();
            if (__popc(left) > kTpFew) {
                // an even TB would put the lanes' words in the same banks: every lane starts elsewhere
                const int first = q.TB % 2 == 0 ? l % q.TB : 0;
#pragma unroll 4
                for (int i = 0; i < q.TB; ++i) {
                    const int s = i + first < q.TB ? i + first : i + first - q.TB;
                    if (s < n) vs[l * q.TB + s] = zs[s * 32 + l];
                }
                __syncwarp();
                if (l == 0) tp_soma_serial<SOFT>(q.T, beta, theta, vs);
                return true;
            }
            // the first lane left onwards, by all lanes together
            const int f = __ffs(left) - 1;
            float cur = __shfl_sync(0xffffffffu, end, f - 1);
            for (int r = f; r < 32; ++r) {
                const float st = __shfl_sync(0xffffffffu, start, r), en = __shfl_sync(0xffffffffu, end, r);
                cur = __float_as_int(cur) == __float_as_int(st) ? en : segment(r, q.len(r), cur);
            }
            return false;
        }
        if (again) {
            start = before;
            end = segment(l, n, start);
        }
    }
}

// The decay of the first compartment this thread's warp scans.
template <int K>
__device__ __forceinline__ float tp_alpha(const Params &P, const TpGeom &q) {
    const int k = threadIdx.x >> 5;
    return P.stateless ? 0.f : __ldg(P.alpha + (int64_t)q.chan * K + (k < K ? k : 0));
}

// V^d over x in the planes xv, Z in zs, V^s in vs (zs holds the residual sums on entry).
template <int K, int G>
__device__ __forceinline__ void tp_forward_pass(const Params &P, TpGeom &q, const TpParams<K, G> &par,
                                                float alpha, int psi, float *xv, float *zs, float *vs) {
    const int w = threadIdx.x >> 5, nw = blockDim.x >> 5;
    const bool residual = P.residual != 0;
    __syncthreads();
    if (!P.stateless) {
        for (int k = w; k < K; k += nw) {
            const float a = k == w ? alpha : __ldg(P.alpha + (int64_t)q.chan * K + k);
            tp_scan<false>(q, [a](int) { return a; }, xv + k * q.plane, xv + k * q.plane);
        }
        __syncthreads();
    }
    q.sweep([&](int slot, int t) {
        float vd[K];
#pragma unroll
        for (int k = 0; k < K; ++k) vd[k] = xv[k * q.plane + slot];
        float z = tp_soma_input<K, G>(par, vd, psi);
        if (residual) z = __fmaf_rn(zs[slot], 1.f / (float)K, z);
        if (q.serial()) vs[t] = z;
        else zs[slot] = z;
    });
    __syncthreads();
    bool plain = q.serial();
    if (plain) {
        if (threadIdx.x == 0) {
            if (P.soft) tp_soma_serial<true>(q.T, P.beta, P.theta, vs);
            else tp_soma_serial<false>(q.T, P.beta, P.theta, vs);
        }
    } else if (w == 0) {
        plain = P.soft ? tp_soma_run<true>(q, P.beta, P.theta, zs, vs) : tp_soma_run<false>(q, P.beta, P.theta, zs, vs);
    }
    q.plain = __syncthreads_or(plain);
}

template <int K, int G, typename XT>
__global__ void __launch_bounds__(kTpMaxThreads) tp_forward_kernel(const FwdArgs A, int psi, int layout) {
    pdl_wait();
    const Geometry &g = A.g;
    const Params &P = A.p;
    TpGeom q(g, layout);
    extern __shared__ float tp_smem[];
    float *const xv = tp_smem;                         // [K]: x, then V^d
    float *const zs = xv + K * q.plane;                // Z
    float *const vs = zs + q.plane;                    // V^s
    TpParams<K, G> par;
    par.fetch(P, g, q.n, q.chan);
    const float alpha = tp_alpha<K>(P, q);
    tp_stage<K, XT>(q, static_cast<const XT *>(A.x), layout, P.residual != 0, xv, zs);
    par.form(P);
    tp_forward_pass<K, G>(P, q, par, alpha, psi, xv, zs, vs);
    XT *const sp = static_cast<XT *>(A.spikes) + q.j;
    q.sweep([&](int slot, int t) {
        const float v = vs[q.v_at(slot, t)];
        Scalar<XT>::store_spike(sp + (int64_t)t * g.BN, v >= P.theta);   // Eq. methods-lif-fire
        if (A.v_out) A.v_out[(int64_t)t * g.BN + q.j] = v;
    });
    pdl_trigger();
}

// Sums of N values over the block in a fixed order (warp butterflies, then the warps in
// order), to out[at(i)] by the block's first threads. red: N floats per warp.
template <int N, typename F>
__device__ __forceinline__ void tp_block_sums(float (&v)[N], float *red, F out) {
#pragma unroll
    for (int d = 16; d >= 1; d >>= 1) {
#pragma unroll
        for (int i = 0; i < N; ++i) v[i] = __fadd_rn(v[i], __shfl_xor_sync(0xffffffffu, v[i], d));
    }
    const int w = threadIdx.x >> 5, nw = blockDim.x >> 5;
    if ((threadIdx.x & 31) == 0) {
#pragma unroll
        for (int i = 0; i < N; ++i) red[w * N + i] = v[i];
    }
    __syncthreads();
    if (threadIdx.x < N) {
        float s = 0.f;
        for (int i = 0; i < nw; ++i) s = __fadd_rn(s, red[i * N + threadIdx.x]);
        out((int)threadIdx.x, s);
    }
    __syncthreads();
}

template <int K, int G, typename XT>
__global__ void __launch_bounds__(kTpMaxThreads) tp_backward_kernel(const BwdArgs A, int psi, int layout) {
    pdl_wait();
    constexpr int Kb = K / G;
    constexpr int NP = 2 * K + 2 * Kb + 1;
    constexpr int KG = K < 4 ? K : 4;                  // compartments per group (a whole number of branches)
    constexpr int KGb = KG / G;
    const Geometry &g = A.g;
    const Params &P = A.p;
    TpGeom q(g, layout);
    extern __shared__ float tp_smem[];
    float *const vdh = tp_smem;                        // [K]: x, then V^d
    float *const zsb = vdh + K * q.plane;              // Z, then k1
    float *const vs = zsb + q.plane;                   // V^s
    float *const gsb = vs + q.plane;                   // dL/dS
    float *const dz = gsb + q.plane;                   // k2, then dL/dZ
    float *const gvb = dz + q.plane;                   // dL/dV^s (when given)
    __shared__ float red[(kTpMaxThreads / 32) * (2 * KG + 2 * KGb)];
    static_assert(sizeof red <= kMaxStaticSmem, "allow_smem counts on it");
    const bool has_gv = A.gv != nullptr;
    TpParams<K, G> par;
    par.fetch(P, g, q.n, q.chan);
    const float alpha = tp_alpha<K>(P, q);
    tp_stage<K, XT>(q, static_cast<const XT *>(A.x), layout, P.residual != 0, vdh, zsb);
    {
        const XT *const gsp = static_cast<const XT *>(A.gs) + q.j;
        float v[4], u[4];
        q.template sweep_loads<4>(
            [&](int b, int t) {
                v[b] = Scalar<XT>::unpack(Scalar<XT>::load(gsp + (int64_t)t * g.BN));
                if (has_gv) u[b] = __ldg(A.gv + (int64_t)t * g.BN + q.j);
            },
            [&](int b, int slot) {
                gsb[slot] = v[b];
                if (has_gv) gvb[slot] = u[b];
            });
    }
    par.form(P);
    tp_forward_pass<K, G>(P, q, par, alpha, psi, vdh, zsb, vs);
    float *const out = A.partials + q.j * NP;

    // soma, reverse time (Eq. methods-sg). Given the forward trajectory the recursion is
    // linear in dL/dV: dv[t] = k1[t] + k2[t] dv[t+1] with k1 = sg (dL/dS) (+ dL/dV^s) and
    // k2 = sg dV[t+1]/dS[t] + dV[t+1]/dV[t], so it is scanned over time like the
    // compartments
    const float kv = (P.detach || P.soft) ? 0.f : -P.beta;
    const float cs = (P.detach || !P.soft) ? 0.f : -P.beta * P.theta;
    const float b_spike = P.soft ? P.beta : 0.f;
    q.sweep([&](int slot, int t) {
        const float v = vs[q.v_at(slot, t)];
        const float sg = surrogate(__fsub_rn(v, P.theta));
        const float dvds = __fmaf_rn(kv, v, cs);                         // dV[t+1]/dS[t]
        const float dvdv = (v >= P.theta) ? b_spike : P.beta;            // dV[t+1]/dV[t]
        zsb[slot] = has_gv ? __fmaf_rn(sg, gsb[slot], gvb[slot]) : __fmul_rn(sg, gsb[slot]);
        dz[slot] = __fmaf_rn(sg, dvds, dvdv);
    });
    __syncthreads();
    if (threadIdx.x < 32) tp_scan<true>(q, [&](int slot) { return dz[slot]; }, zsb, dz);
    __syncthreads();
    float gb[1] = {0.f};                               // sum of dL/dV[t+1] dV[t+1]/dbeta
    if (A.want_beta) {
        q.sweep([&](int slot, int t) {
            if (t + 1 < q.T) {
                const int next = slot + 32 < q.plane ? slot + 32 : (slot & 31) + 1;   // step t + 1
                const float v = vs[q.v_at(slot, t)];
                const bool st = v >= P.theta;
                const float leak = st ? (P.soft ? __fsub_rn(v, P.theta) : 0.f) : v;
                gb[0] = __fmaf_rn(dz[next], leak, gb[0]);
            }
        });
    }
    tp_block_sums<1>(gb, red, [&](int, float s) { out[NP - 1] = s; });

    // dendrite, reverse time, four compartments at a time: direct_i[t] from V^d[t] and dL/dZ[t]
    // into the planes that are free by now, A_i[t] = direct_i[t] + alpha_i A_i[t+1] scanned in
    // place, then dL/dX[t] and dL/dalpha
    float *const planes[4] = {zsb, vs, gsb, gvb};
    const bool stateless = P.stateless != 0;
    const bool residual = P.residual != 0;
    const float inv_k = 1.f / (float)K;
    XT *const gxn = static_cast<XT *>(A.gx) + q.xo;
#pragma unroll
    for (int k0 = 0; k0 < K; k0 += KG) {
        const int b0 = k0 / G;
        float sum[2 * KG + 2 * KGb];                   // alpha KG | xi KG | zeta KGb | kappa KGb
#pragma unroll
        for (int i = 0; i < 2 * KG + 2 * KGb; ++i) sum[i] = 0.f;
        q.sweep([&](int slot, int) {
            const float dzt = dz[slot];
#pragma unroll
            for (int b = 0; b < KGb; ++b) {
                float vd[G], u[G];
#pragma unroll
                for (int i = 0; i < G; ++i) vd[i] = vdh[(k0 + b * G + i) * q.plane + slot];
                const float ss = tp_branch_ss<K, G>(par, b0 + b, vd, u);
                const float gy = __fmul_rn(par.km[b0 + b], dzt);
                float y, qq;                                    // Y_b; dL/du_i = qq u_i
                if (psi == PSI_MEXHAT) {
                    const float e = gauss_half(ss);
                    y = __fmaf_rn(-ss, e, e);
                    qq = __fmul_rn(__fmul_rn(__fsub_rn(ss, 3.f), e), gy);   // psi'(r) / r
                } else {
                    const float r = sqrtf(ss);
                    y = r;
                    qq = (r > 0.f) ? __fdiv_rn(gy, r) : 0.f;                // subgradient 0 at r = 0
                }
#pragma unroll
                for (int i = 0; i < G; ++i) {
                    const float d = __fmul_rn(__fmul_rn(qq, u[i]), par.iz[b0 + b]);
                    planes[b * G + i][slot] = d;
                    sum[KG + b * G + i] = __fsub_rn(sum[KG + b * G + i], d);
                }
                sum[2 * KG + b] = __fmaf_rn(-__fmul_rn(ss, qq), par.iz[b0 + b], sum[2 * KG + b]);   // -(dL/dr) r / zeta
                sum[2 * KG + KGb + b] = __fmaf_rn(__fmul_rn(par.mk[b0 + b], y), dzt, sum[2 * KG + KGb + b]);
            }
        });
        __syncthreads();
        if (!stateless) {
            const int w = threadIdx.x >> 5;
            for (int i = w; i < KG; i += blockDim.x >> 5) {
                float *p = i == 0 ? planes[0] : i == 1 ? planes[1] : i == 2 ? planes[2] : planes[3];
                const float a = k0 == 0 && i == w ? alpha : __ldg(P.alpha + (int64_t)q.chan * K + k0 + i);
                tp_scan<true>(q, [a](int) { return a; }, p, p);
            }
            __syncthreads();
        }
        q.sweep([&](int slot, int t) {
            const float res = residual ? __fmul_rn(dz[slot], inv_k) : 0.f;
            // the slot of step t - 1: the step before in the segment, or the end of the one before
            const int prev = slot >= 32 ? slot - 32 : (q.TB - 1) * 32 + slot - 1;
            float gx[KG];
#pragma unroll
            for (int i = 0; i < KG; ++i) {
                const float v = planes[i][slot];
                gx[i] = residual ? __fadd_rn(v, res) : v;
                if (!stateless && t > 0) sum[i] = __fmaf_rn(v, vdh[(k0 + i) * q.plane + prev], sum[i]);
            }
            XT *p = gxn + (int64_t)t * q.sX + k0 * q.ks;
            if (layout == 0) {
                Vec<XT, KG>::store(p, gx);
            } else {
#pragma unroll
                for (int i = 0; i < KG; ++i) {
                    const float one[1] = {gx[i]};
                    Vec<XT, 1>::store(p + i * q.ks, one);
                }
            }
        });
        tp_block_sums<2 * KG + 2 * KGb>(sum, red, [&](int i, float s) {
            const int at = i < KG ? k0 + i : i < 2 * KG ? K + k0 + i - KG
                         : i < 2 * KG + KGb ? 2 * K + b0 + i - 2 * KG : 2 * K + Kb + b0 + i - 2 * KG - KGb;
            out[at] = s;
        });
    }
    pdl_trigger();
}

// Per (channel, gradient slot) a warp sums the neurons' partials: each lane every 32nd neuron of
// the channel in order, then the lanes in a fixed tree.
constexpr int kTpFinThreads = 256;
__global__ void __launch_bounds__(kTpFinThreads) tp_finalize_kernel(const FinArgs F) {
    pdl_wait();
    pdl_trigger();
    const Geometry &g = F.g;
    const int NP = 2 * g.K + 2 * g.Kb + 1;
    const int64_t w = (int64_t)blockIdx.x * (kTpFinThreads / 32) + (threadIdx.x >> 5);
    if (w >= (int64_t)g.C * NP) return;
    const int c = (int)(w / NP);
    const int q = (int)(w % NP);
    float sum = 0.f;
    const int64_t m = g.BN / g.C;                      // neurons of the channel, in runs of `inner`
    for (int64_t i = threadIdx.x & 31; i < m; i += 32) {
        const int64_t j = (i / g.inner) * g.P + (int64_t)c * g.inner + i % g.inner;
        sum = __fadd_rn(sum, F.partials[j * NP + q]);
    }
#pragma unroll
    for (int d = 16; d >= 1; d >>= 1) sum = __fadd_rn(sum, __shfl_xor_sync(0xffffffffu, sum, d));
    if (threadIdx.x & 31) return;
    if (q < g.K) F.g_alpha[(int64_t)c * g.K + q] = F.stateless ? 0.f : sum;
    else if (q < 2 * g.K) F.g_xi[(int64_t)c * g.K + (q - g.K)] = sum;
    else if (q < 2 * g.K + g.Kb) F.g_zeta[(int64_t)c * g.Kb + (q - 2 * g.K)] = sum;
    else if (q < 2 * g.K + 2 * g.Kb) F.g_kappa[(int64_t)c * g.Kb + (q - 2 * g.K - g.Kb)] = sum;
    else if (F.g_beta) F.g_beta[c] = sum;
}

// Shared memory of a kernel: its planes, each padded to whole segments.
size_t tp_bytes(const Geometry &g, int planes) {
    return sizeof(float) * (size_t)((g.T + 31) / 32 * 32) * (size_t)planes;
}

// Launched like the library's other kernels (programmatic stream serialization).
template <typename... Par, typename... Arg>
cudaError_t tp_launch(void (*kernel)(Par...), unsigned blocks, unsigned threads, size_t smem, cudaStream_t s,
                      Arg... arg) {
    cudaError_t e = allow_smem(kernel, smem);
    if (e != cudaSuccess) return e;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(blocks);
    cfg.blockDim = dim3(threads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = at;
    cfg.numAttrs = DENDSN_PDL ? 1 : 0;
    return with_opt_in(reinterpret_cast<const void *>(kernel), smem,
                       [&] { return cudaLaunchKernelEx(&cfg, kernel, arg...); });
}

}  // namespace

// The bytes by which the plan decides between these kernels and the chunked ones: the backward's
// planes without their padding to whole segments, which adds 2.6 KB at most to the plan's 200.
size_t tp_smem_bytes(int T, int K) { return sizeof(float) * (size_t)T * ((size_t)K + 5); }

template <int K, int G, int XT>
cudaError_t launch_forward_tp(const FwdArgs &a, int psi, int layout, cudaStream_t s) {
    const size_t smem = tp_bytes(a.g, K + 2);
    return tp_launch(tp_forward_kernel<K, G, typename XType<XT>::type>, (unsigned)a.g.BN,
                     (unsigned)tp_threads(a.g.T, a.g.BN, smem), smem, s, a, psi, layout);
}

template <int K, int G, int XT>
cudaError_t launch_backward_tp(const BwdArgs &a, int psi, int layout, cudaStream_t s) {
    const size_t smem = tp_bytes(a.g, K + 5);
    return tp_launch(tp_backward_kernel<K, G, typename XType<XT>::type>, (unsigned)a.g.BN,
                     (unsigned)tp_threads(a.g.T, a.g.BN, smem), smem, s, a, psi, layout);
}

cudaError_t launch_finalize_tp(const FinArgs &a, cudaStream_t s) {
    const int64_t n = (int64_t)a.g.C * (2 * a.g.K + 2 * a.g.Kb + 1);
    return tp_launch(tp_finalize_kernel, (unsigned)((n * 32 + kTpFinThreads - 1) / kTpFinThreads), kTpFinThreads, 0, s, a);
}

#define DENDSN_TP_INST(K, G)                                                                    \
    template cudaError_t launch_forward_tp<K, G, 0>(const FwdArgs &, int, int, cudaStream_t);  \
    template cudaError_t launch_forward_tp<K, G, 1>(const FwdArgs &, int, int, cudaStream_t);  \
    template cudaError_t launch_backward_tp<K, G, 0>(const BwdArgs &, int, int, cudaStream_t); \
    template cudaError_t launch_backward_tp<K, G, 1>(const BwdArgs &, int, int, cudaStream_t);
DENDSN_KG_LIST(DENDSN_TP_INST)
#undef DENDSN_TP_INST

}  // namespace dendsn

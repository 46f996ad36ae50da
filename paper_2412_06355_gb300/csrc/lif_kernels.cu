// Fused multi-step LIF layer (forward and BPTT backward): the point-neuron layer the
// paper compares the DendSN layer's speed against (Results, efficiency paragraph).
// The neuron is the DendSN soma (Eq. methods-lif-reset-charge, Eq. methods-lif-fire)
// driven directly by its input current, with the arctan surrogate of Eq. methods-sg.
//
// Same design rules as the DendSN kernels: every step of a neuron runs in one thread
// with the state in registers, the backward recomputes the forward from x (nothing is
// saved for T <= 8; V at the end of every 8-step chunk otherwise), and all tensors are
// streamed once with vector loads. A thread owns VEC consecutive neurons, so a warp
// moves 32 * VEC contiguous elements per step.
#include "dendsn_kernels.cuh"

namespace dendsn {

namespace {

// One LIF charge (hard or soft reset), as soma_charge but with plain arguments.
__device__ __forceinline__ float lif_charge(float x, float v_prev, bool s_prev, float beta,
                                            float theta, int soft) {
    const float leak = soft ? (s_prev ? __fsub_rn(v_prev, theta) : v_prev)
                            : (s_prev ? 0.f : v_prev);
    return __fmaf_rn(beta, leak, x);
}

// CH: steps per chunk (4 when T <= 4, else 8; checkpoints only with 8).
template <typename XT, int VEC, int CH>
__global__ void __launch_bounds__(256) lif_forward_kernel(const LifArgs A) {
    pdl_wait();
    using V = Vec<XT, VEC>;
    const int64_t m0 = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) * VEC;
    if (m0 >= A.M) return;
    const int64_t M = A.M;
    const int T = A.T;
    const XT *xp = static_cast<const XT *>(A.x) + m0;
    XT *sp = static_cast<XT *>(A.spikes) + m0;
    float v[VEC];
    bool s[VEC];
#pragma unroll
    for (int e = 0; e < VEC; ++e) { v[e] = 0.f; s[e] = false; }
    for (int t0 = 0; t0 < T; t0 += CH) {
        const int n = min(CH, T - t0);
        typename V::Raw xr[CH];
#pragma unroll
        for (int tt = 0; tt < CH; ++tt)
            if (tt < n) xr[tt] = V::load(xp + (int64_t)(t0 + tt) * M);
#pragma unroll
        for (int tt = 0; tt < CH; ++tt) {
            if (tt < n) {
                float xv[VEC], sv[VEC];
                V::unpack(xr[tt], xv);
#pragma unroll
                for (int e = 0; e < VEC; ++e) {
                    v[e] = lif_charge(xv[e], v[e], s[e], A.beta, A.theta, A.soft);
                    s[e] = v[e] >= A.theta;                     // Eq. methods-lif-fire
                    sv[e] = s[e] ? 1.f : 0.f;
                }
                const int64_t off = (int64_t)(t0 + tt) * M;
                V::store(sp + off, sv);
                if (A.v_out) Vec<float, VEC>::store(A.v_out + m0 + off, v);
            }
        }
        if (CH == 8 && A.ck && t0 + CH < T)
            Vec<float, VEC>::store(A.ck + (int64_t)(t0 / CH) * M + m0, v);
    }
    // not earlier: the next launch's blocks would be placed, waiting, before this one's have left, several
    // on an SM (T = 64, bfloat16, 400000 neurons, forwards in a row 25.2 without programmatic launches,
    // 34.3 with the trigger at the start, 23.6 here; T = 4, float32, 8.4M neurons 42.6, 40.4, 40.5)
    pdl_trigger();
}

template <typename XT, int VEC, int CH>
__global__ void __launch_bounds__(256, 2) lif_backward_kernel(const LifArgs A) {
    pdl_wait();
    pdl_trigger();
    using V = Vec<XT, VEC>;
    const int64_t m0 = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) * VEC;
    if (m0 >= A.M) return;
    const int64_t M = A.M;
    const int T = A.T;
    const XT *xp = static_cast<const XT *>(A.x) + m0;
    const XT *gsp = static_cast<const XT *>(A.gs) + m0;
    XT *gxp = static_cast<XT *>(A.gx) + m0;
    const float *gvp = A.gv ? A.gv + m0 : nullptr;
    const float nbt = -A.beta * A.theta;                       // dV[t+1]/dS[t], soft reset
    float gn[VEC];                                             // dL/dV[t+1]
#pragma unroll
    for (int e = 0; e < VEC; ++e) gn[e] = 0.f;
    const int nch = (T + CH - 1) / CH;
    for (int c = nch - 1; c >= 0; --c) {
        const int t0 = c * CH;
        const int n = min(CH, T - t0);
        // 4-step chunks fetch grad_spikes together with x, before the recompute; 8-step
        // chunks fetch it step by step in the reverse loop (the whole chunk would spill)
        constexpr bool AHEAD = CH == 4;
        typename V::Raw xr[CH], gr[AHEAD ? CH : 1];
#pragma unroll
        for (int tt = 0; tt < CH; ++tt) {
            if (tt < n) {
                xr[tt] = V::load(xp + (int64_t)(t0 + tt) * M);
                if constexpr (AHEAD) gr[tt] = V::load(gsp + (int64_t)(t0 + tt) * M);
            }
        }
        // recompute the chunk's potentials from its starting state
        float v[VEC];
        bool s[VEC];
        if (c == 0) {
#pragma unroll
            for (int e = 0; e < VEC; ++e) { v[e] = 0.f; s[e] = false; }
        } else {
            Vec<float, VEC>::unpack(Vec<float, VEC>::load(A.ck + (int64_t)(c - 1) * M + m0), v);
#pragma unroll
            for (int e = 0; e < VEC; ++e) s[e] = v[e] >= A.theta;
        }
        float vh[CH][VEC];
#pragma unroll
        for (int tt = 0; tt < CH; ++tt) {
            if (tt < n) {
                float xv[VEC];
                V::unpack(xr[tt], xv);
#pragma unroll
                for (int e = 0; e < VEC; ++e) {
                    v[e] = lif_charge(xv[e], v[e], s[e], A.beta, A.theta, A.soft);
                    s[e] = v[e] >= A.theta;
                    vh[tt][e] = v[e];
                }
            }
        }
        // reverse time through the chunk
#pragma unroll
        for (int tt = CH - 1; tt >= 0; --tt) {
            if (tt < n) {
                const int64_t off = (int64_t)(t0 + tt) * M;
                float gsv[VEC], gv[VEC], gx[VEC];
                if constexpr (AHEAD) V::unpack(gr[tt], gsv);
                else V::unpack(V::load(gsp + off), gsv);
                if (gvp) Vec<float, VEC>::unpack(Vec<float, VEC>::load(gvp + off), gv);
#pragma unroll
                for (int e = 0; e < VEC; ++e) {
                    const float vt = vh[tt][e];
                    const bool st = vt >= A.theta;
                    const float dvdv = (A.soft || !st) ? A.beta : 0.f;
                    const float dvds = A.detach_reset ? 0.f : (A.soft ? nbt : -A.beta * vt);
                    const float ds = __fmaf_rn(dvds, gn[e], gsv[e]);
                    float dv = __fmaf_rn(surrogate(__fsub_rn(vt, A.theta)), ds,
                                         __fmul_rn(dvdv, gn[e]));
                    if (gvp) dv = __fadd_rn(dv, gv[e]);
                    gx[e] = dv;
                    gn[e] = dv;
                }
                V::store(gxp + off, gx);
            }
        }
    }
}

// The backward of long rows of large layers. lif_backward_kernel's 8-step chunks fetch
// grad_spikes step by step behind the reverse loop's stores. Here grad_spikes arrive as the
// recompute frees x's registers, last step first (the reverse loop's order), and the next
// chunk's x as the reverse loop frees grad_spikes': every load is half a chunk ahead of its use,
// in no more registers. Same operations, same bits. GB300, us: T = 8, 8.4M neurons 198 -> 163,
// T = 64 bfloat16, 2.1M neurons 362 -> 206, T = 16 bfloat16, 786k neurons 36 -> 22; small layers
// and ragged short rows, where the compiler's own order of the other kernel's loads does better,
// stay there (T = 12, 80k neurons 5.8 -> 7.1; T = 5, 1M neurons 11 -> 14). Either side of the line:
// bfloat16 T = 16, 500000 neurons 22.0 on the other kernel, 524288 15.4; float32 26.4 and 23.8.
constexpr int64_t kLifStreamM = 524288;
template <typename XT, int VEC>
__global__ void __launch_bounds__(256, 2) lif_backward_stream_kernel(const LifArgs A) {
    pdl_wait();
    pdl_trigger();
    constexpr int CH = 8;
    using V = Vec<XT, VEC>;
    const int64_t m0 = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) * VEC;
    if (m0 >= A.M) return;
    const int64_t M = A.M;
    const int T = A.T;
    const XT *xp = static_cast<const XT *>(A.x) + m0;
    const XT *gsp = static_cast<const XT *>(A.gs) + m0;
    XT *gxp = static_cast<XT *>(A.gx) + m0;
    const float *gvp = A.gv ? A.gv + m0 : nullptr;
    const float nbt = -A.beta * A.theta;                       // dV[t+1]/dS[t], soft reset
    float gn[VEC];                                             // dL/dV[t+1]
#pragma unroll
    for (int e = 0; e < VEC; ++e) gn[e] = 0.f;
    const int nch = (T + CH - 1) / CH;
    typename V::Raw xr[CH], gr[CH];
    {
        const int t0 = (nch - 1) * CH;
#pragma unroll
        for (int tt = 0; tt < CH; ++tt) {
            if (t0 + tt < T) xr[tt] = V::load(xp + (int64_t)(t0 + tt) * M);
        }
    }
    for (int c = nch - 1; c >= 0; --c) {
        const int t0 = c * CH;
        const int n = min(CH, T - t0);
        // recompute the chunk's potentials from its starting state
        float v[VEC];
        bool s[VEC];
        if (c == 0) {
#pragma unroll
            for (int e = 0; e < VEC; ++e) { v[e] = 0.f; s[e] = false; }
        } else {
            Vec<float, VEC>::unpack(Vec<float, VEC>::load(A.ck + (int64_t)(c - 1) * M + m0), v);
#pragma unroll
            for (int e = 0; e < VEC; ++e) s[e] = v[e] >= A.theta;
        }
        float vh[CH][VEC];
#pragma unroll
        for (int tt = 0; tt < CH; ++tt) {
            float xv[VEC];
            if (tt < n) V::unpack(xr[tt], xv);
            if (CH - 1 - tt < n) gr[CH - 1 - tt] = V::load(gsp + (int64_t)(t0 + CH - 1 - tt) * M);
            if (tt < n) {
#pragma unroll
                for (int e = 0; e < VEC; ++e) {
                    v[e] = lif_charge(xv[e], v[e], s[e], A.beta, A.theta, A.soft);
                    s[e] = v[e] >= A.theta;
                    vh[tt][e] = v[e];
                }
            }
        }
        // reverse time through the chunk
#pragma unroll
        for (int tt = CH - 1; tt >= 0; --tt) {
            float gsv[VEC];
            if (tt < n) V::unpack(gr[tt], gsv);
            if (c > 0) xr[CH - 1 - tt] = V::load(xp + (int64_t)(t0 - 1 - tt) * M);
            if (tt < n) {
                const int64_t off = (int64_t)(t0 + tt) * M;
                float gv[VEC], gx[VEC];
                if (gvp) Vec<float, VEC>::unpack(Vec<float, VEC>::load(gvp + off), gv);
#pragma unroll
                for (int e = 0; e < VEC; ++e) {
                    const float vt = vh[tt][e];
                    const bool st = vt >= A.theta;
                    const float dvdv = (A.soft || !st) ? A.beta : 0.f;
                    const float dvds = A.detach_reset ? 0.f : (A.soft ? nbt : -A.beta * vt);
                    const float ds = __fmaf_rn(dvds, gn[e], gsv[e]);
                    float dv = __fmaf_rn(surrogate(__fsub_rn(vt, A.theta)), ds,
                                         __fmul_rn(dvdv, gn[e]));
                    if (gvp) dv = __fadd_rn(dv, gv[e]);
                    gx[e] = dv;
                    gn[e] = dv;
                }
                V::store(gxp + off, gx);
            }
        }
    }
}

int lif_blocks(int64_t M, int vec) {
    const int64_t threads = (M + vec - 1) / vec;
    return (int)((threads + 255) / 256);
}

}  // namespace

template <int XT, int VEC>
cudaError_t launch_lif_forward(const LifArgs &a, cudaStream_t s) {
    using T = typename std::conditional<XT == 1, __nv_bfloat16, float>::type;
    const int blocks = lif_blocks(a.M, VEC);
    // (with programmatic launches, like the DendSN kernels: 107.9 -> 103.6 us for forward and
    // backward of the conv layer's 8.4M neurons)
    return launch_or_query(a.T <= 4 ? lif_forward_kernel<T, VEC, 4> : lif_forward_kernel<T, VEC, 8>, a, blocks, 256,
                           0, s, nullptr);
}

template <int XT, int VEC>
cudaError_t launch_lif_backward(const LifArgs &a, cudaStream_t s) {
    using T = typename std::conditional<XT == 1, __nv_bfloat16, float>::type;
    const int blocks = lif_blocks(a.M, VEC);
    auto kernel = a.T <= 4 ? lif_backward_kernel<T, VEC, 4>
                : a.T >= 8 && a.M >= kLifStreamM ? lif_backward_stream_kernel<T, VEC> : lif_backward_kernel<T, VEC, 8>;
    return launch_or_query(kernel, a, blocks, 256, 0, s, nullptr);
}

template cudaError_t launch_lif_forward<0, 1>(const LifArgs &, cudaStream_t);
template cudaError_t launch_lif_forward<0, 4>(const LifArgs &, cudaStream_t);
template cudaError_t launch_lif_forward<1, 1>(const LifArgs &, cudaStream_t);
template cudaError_t launch_lif_forward<1, 4>(const LifArgs &, cudaStream_t);
template cudaError_t launch_lif_backward<0, 1>(const LifArgs &, cudaStream_t);
template cudaError_t launch_lif_backward<0, 4>(const LifArgs &, cudaStream_t);
template cudaError_t launch_lif_backward<1, 1>(const LifArgs &, cudaStream_t);
template cudaError_t launch_lif_backward<1, 4>(const LifArgs &, cudaStream_t);

}  // namespace dendsn

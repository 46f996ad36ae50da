// The forward of rows of more than 8 steps, one chunk of 8 steps at a time.
//
// dendsn_forward_kernel walks a row step by step: each step waits for its own copy, and that
// wait keeps the compiler from overlapping a step with the next, so a warp needs some 500
// cycles per step unless others hide them. Here a chunk is waited for once and its steps are
// unrolled: V^d is a short chain, so the branches of all 8 steps are evaluated side by side, then the
// soma runs over the 8 values of Z. Same operations in the same order per neuron: same bits.
// 128 threads per block, so that layers of few neurons spread over more SMs.
//
// GB300, us before -> after: T = 2048, K = 4, G = 2, 65536 neurons 624 -> 531; T = 1680, 3000
// neurons 425 -> 162; T = 64, K = 8 bfloat16, 2M neurons 585 -> 421; T = 10, K = 4, G = 2,
// H*W = 49, 803k neurons 47 -> 39; the event-stream layer (T = 64, K = 4, 4.2M neurons, memory
// bound) 851 -> 854. Three chunks in flight per thread and four blocks per SM: two chunks and five
// blocks left the event-stream layer at 889.
#pragma once

namespace dendsn {

template <typename Raw> constexpr size_t chunk_fwd_bytes(int NT) { return sizeof(Raw) * 3 * 8 * NT; }

template <int K, int G, int PSI, typename XT, int LAYOUT>
__global__ void __launch_bounds__(kChunkFwdThreads, 4)
dendsn_forward_chunk_kernel(const FwdArgs A) {
    pdl_wait();
    constexpr int NT = kChunkFwdThreads, L = 8;
    constexpr int KT = lane_compartments(K);
    constexpr int LPN = K / KT;
    using V = XIO<XT, KT, LAYOUT>;
    using AR = Arith<KT, G, PSI, XT>;
    using Raw = typename V::Raw;
    const Geometry &g = A.g;
    const Params &P = A.p;
    const ThreadPos pos = thread_pos<LPN>(g);
    if (pos.nrows == 0) return;                  // whole warps: rows are uniform per warp
    typename AR::LP lp;
    AR::load(P, g, pos.chan, pos.sub, lp);
    const float inv_k = 1.f / (float)K;
    const int T = g.T;
    const int nc = (T + L - 1) / L;
    const int64_t sX = g.BN * K;
    const int64_t BN = g.BN;
    const int64_t ks = LAYOUT == 0 ? 1 : g.inner;
    const int64_t j0 = pos.row0 * g.P + pos.p;
    const int64_t jstep = (int64_t)pos.rstride * g.P;
    const XT *const x0 = static_cast<const XT *>(A.x) + lane_x_offset<LAYOUT>(j0, pos.sub, KT, K, g.inner);
    const bool write_ck = A.ck_vd != nullptr && g.n_ck > 0 && pos.active;
    const bool store = pos.active && pos.sub == 0;
    const bool residual = P.residual != 0;

    // dynamic shared memory: the lanes' kappa (per-neuron masks only), then x [3][L][NT]
    extern __shared__ float4 fwd_smem[];
    Raw *const xs0 = reinterpret_cast<Raw *>(reinterpret_cast<char *>(fwd_smem) +
                                             kappa_smem_bytes(P.mask_mode, AR::KTb, NT)) + threadIdx.x;
    int fi = 0, fc = 0;                          // row and chunk of the next fetch
    auto fetch = [&](int buf, float dep) {
        if (fi < pos.nrows) {
            const int n = min(L, T - fc * L);
            const XT *xp = x0 + fi * (jstep * K) + (int64_t)fc * L * sX;
            Raw *const xs = xs0 + buf * (L * NT);
            auto step = [&](int tt) {
                V::copy_async(xs + tt * NT, xp, ks, dep);
                xp += sX;
            };
            if (n == L) TwinSteps<L, true>::forward(n, step);
            else TwinSteps<L, false>::forward(n, step);
        }
        cp_async_commit();
        if (++fc == nc) { fc = 0; ++fi; }
    };
    fetch(0, 0.f);
    fetch(1, 0.f);
    fetch(2, 0.f);
    int buf = 0;
    MaskAhead<AR, NT> mask;
    mask.init(P, g, j0, jstep, pos.chan, pos.sub, pos.nrows, fwd_smem);
    for (int i = 0; i < pos.nrows; ++i) {
        mask.advance(P, g, pos.sub, i + 1 < pos.nrows, lp);
        typename AR::St vd;
        AR::zero(vd);
        float v = 0.f;
        bool s = false;
        const int64_t j = j0 + i * jstep;
        XT *sp = static_cast<XT *>(A.spikes) + j;
        float *vp = A.v_out ? A.v_out + j : nullptr;
        for (int c = 0; c < nc; ++c) {
            const int n = min(L, T - c * L);
            const Raw *const xs = xs0 + buf * (L * NT);
            auto chunk = [&](auto full) {
                using Steps = TwinSteps<L, decltype(full)::value>;
                cp_async_wait<2>();
                float z[L], last = 0.f;
                Steps::forward(n, [&](int tt) {
                    float xv[KT];
                    V::unpack(xs[tt * NT], xv);
                    z[tt] = soma_input<AR, KT, LPN>(lp, vd, xv, residual, inv_k);
                    last = z[tt];
                });
                // every step's x has been read (the last Z depends on V^d of them all)
                fetch(buf, last);
                Steps::forward(n, [&](int tt) {
                    v = soma_charge(z[tt], v, s, P);
                    s = v >= P.theta;                      // Eq. methods-lif-fire
                    if (store) {
                        Scalar<XT>::store_spike(sp, s);
                        if (vp) __stcs(vp, v);
                    }
                    sp += BN;
                    if (vp) vp += BN;
                });
            };
            if (n == L) chunk(std::true_type{});
            else chunk(std::false_type{});
            buf = buf == 2 ? 0 : buf + 1;
            if (write_ck && c + 1 < nc) {
                float vda[KT];
                AR::to_array(vd, vda);
                Vec<float, KT>::store(A.ck_vd + ((int64_t)c * BN + j) * K + pos.sub * KT, vda);
                if (pos.sub == 0) __stcs(A.ck_vs + (int64_t)c * BN + j, v);
            }
        }
    }
    pdl_trigger();
    cp_async_wait<0>();
}

}  // namespace dendsn

// Twin kernels: two neighbouring neurons per thread, for the paper's (C_o, P, H, W) layout.
//
// In that layout compartment k of neurons n and n + 1 of one channel run are adjacent
// elements, and for an even H*W the two neurons share a channel. A thread takes both: one
// 4-byte (bfloat16) or 8-byte (float32) access moves a compartment of the pair, and a paired
// fp32 instruction carries the same operation of the two neurons, whatever the number of
// compartments per branch (the compartments-innermost engines can only pair compartments,
// and only with one per branch). Every operation, its rounding and the order of every sum
// are those of the one-neuron-per-thread kernels, per neuron, so the results are the same bits
// (parameter-gradient sums as long as both are tiled alike).
//
// What bounds them, and what they measured on GB300 (us before -> after): bfloat16 layers move
// half the bytes and are bound by instruction issue: T = 6, K = 4, G = 2, B = 128, 128 x 32 x 32
// backward 1330 -> 467 (242 instructions per pair and step from 357 in a first version that let
// the compiler rebuild every parameter pair and tested every step's bounds; floating-point pipe
// half busy, memory floor 272), forward 297 -> 189 (floor 151). Float32 layers come close to
// memory: T = 4, K = 4, G = 2, B = 64, 128 x 32 x 32 backward 224 -> 193 (floor 181).
#pragma once

namespace dendsn {

// A compartment (or one per-neuron value) of the two neurons, as stored.
template <typename XT> struct TwinIO;
template <> struct TwinIO<float> {
    using W = float2;
    static __device__ __forceinline__ float2 unpack(W w) { return w; }
    static __device__ __forceinline__ W pack(float2 v) { return v; }
};
template <> struct TwinIO<__nv_bfloat16> {
    using W = uint32_t;
    static __device__ __forceinline__ float2 unpack(W w) { return make_float2(bf16_lo(w), bf16_hi(w)); }
    static __device__ __forceinline__ W pack(float2 v) { return pack_bf16x2(v.x, v.y); }
};

// -a as one instruction (the sign flip of a pair takes two)
__device__ __forceinline__ float2 minus2(float2 a) { return fmul2(a, f2(-1.f)); }
__device__ __forceinline__ float2 exp2_2(float2 t) { return make_float2(fast_exp2(t.x), fast_exp2(t.y)); }

// The arithmetic of Arith<KT, G, PSI, XT> for two neurons: component .x is the first one's
// value, .y the second's. kPaired follows PairArith's formulas (one compartment per branch),
// otherwise ScalarArith's.
template <int KT, int G, int PSI, bool TREE>
struct TwinArith {
    static constexpr int KTb = KT / G;
    static constexpr bool kPaired = G == 1 && KT % 2 == 0;
    static constexpr bool KAPPA_FREE = kPaired && KT == 8;
    // lm: PairArith's mask term (0 / -inf in the exponent, or m for the identity), or m
    struct LP { float2 a[KT], nxi[KT], iz[KTb], km[KTb], lm[KTb]; };

    static __device__ __forceinline__ float mask_term(float m) {
        if constexpr (kPaired && PSI == PSI_MEXHAT) return m != 0.f ? 0.f : -INFINITY;
        else return m;
    }
    static __device__ __forceinline__ void load(const Params &P, const Geometry &g, int chan, int sub, LP &lp) {
        float a[KT], nxi[KT], iz[KTb], km[KTb], mk[KTb];
        load_param_arrays<KT, G>(P, g, chan, sub, a, nxi, iz, km, mk);
#pragma unroll
        for (int i = 0; i < KT; ++i) { lp.a[i] = f2(a[i]); lp.nxi[i] = f2(nxi[i]); }
#pragma unroll
        for (int b = 0; b < KTb; ++b) { lp.iz[b] = f2(iz[b]); lp.km[b] = f2(km[b]); lp.lm[b] = f2(mask_term(mk[b])); }
    }
    // per-neuron masks: kappa m and the mask term of neurons n and n + 1
    static __device__ __forceinline__ void neuron_masks(const Params &P, const Geometry &g, int64_t n,
                                                        int chan, int sub, LP &lp) {
        float kap[KTb], k0[KTb], m0[KTb], k1[KTb], m1[KTb];
        lane_kappa<KTb>(P, g, chan, sub, kap);
        apply_neuron_mask<KTb>(fetch_neuron_mask<KTb>(P, g, n, sub), kap, k0, m0);
        apply_neuron_mask<KTb>(fetch_neuron_mask<KTb>(P, g, n + 1, sub), kap, k1, m1);
#pragma unroll
        for (int b = 0; b < KTb; ++b) {
            lp.km[b] = make_float2(k0[b], k1[b]);
            lp.lm[b] = make_float2(mask_term(m0[b]), mask_term(m1[b]));
        }
    }
    // A branch's output Y from the V^d of its G compartments.
    static __device__ __forceinline__ float2 branch_y(const float2 *nxi, float2 iz, const float2 *vd) {
        float2 ss, u0;
#pragma unroll
        for (int q = 0; q < G; ++q) {
            const float2 u = ffma2(vd[q], iz, nxi[q]);
            if (q == 0) { u0 = u; ss = fmul2(u, u); }
            else ss = ffma2(u, u, ss);
        }
        if constexpr (PSI == PSI_MEXHAT) {
            const float2 e = exp2_2(fmul2(f2(kNegHalfLog2e), ss));
            return ffma2(minus2(ss), e, e);                      // (1 - r^2) e^{-r^2/2}
        } else if constexpr (G == 1) {
            return make_float2(fabsf(u0.x), fabsf(u0.y));
        } else {
            return make_float2(sqrtf(ss.x), sqrtf(ss.y));
        }
    }
    // One forward step: advances V^d by the inputs x and returns the lane's share of Z, in
    // the summation order of PairArith (tree or chain) or ScalarArith.
    static __device__ __forceinline__ float2 step(const LP &lp, float2 (&vd)[KT], const float2 (&x)[KT],
                                                  bool residual, float inv_k) {
#pragma unroll
        for (int i = 0; i < KT; ++i) vd[i] = ffma2(lp.a[i], vd[i], x[i]);
        float2 y[KTb];
#pragma unroll
        for (int b = 0; b < KTb; ++b) y[b] = branch_y(&lp.nxi[b * G], lp.iz[b], &vd[b * G]);
        if constexpr (!kPaired) {
            float2 z = f2(0.f);
#pragma unroll
            for (int b = 0; b < KTb; ++b) z = ffma2(lp.km[b], y[b], z);
            if (residual) z = add_residual<KT>(&x[0], inv_k, z);
            return z;
        } else {
            constexpr int GS = TREE ? (KT < 4 ? KT : 4) : KT;    // compartments per group
            float2 gv[KT / GS];
#pragma unroll
            for (int q = 0; q < KT / GS; ++q) {
                float2 even, odd;
#pragma unroll
                for (int i = 0; i < GS; i += 2) {
                    const int k = q * GS + i;
                    even = i == 0 ? fmul2(lp.km[k], y[k]) : ffma2(lp.km[k], y[k], even);
                    odd = i == 0 ? fmul2(lp.km[k + 1], y[k + 1]) : ffma2(lp.km[k + 1], y[k + 1], odd);
                }
                gv[q] = add_products(even, odd);
                if (residual) gv[q] = add_residual<GS>(&x[q * GS], inv_k, gv[q]);
            }
            if constexpr (KT / GS == 2) gv[0] = fadd2(gv[0], gv[KT / GS - 1]);
            return gv[0];
        }
    }
    // The sum of the even and the odd compartments' kappa m Y. With two compartments both are
    // bare products, which the compiler would fuse into a paired addition (one rounding less than
    // the one-neuron kernels): scalar additions keep them apart.
    static __device__ __forceinline__ float2 add_products(float2 even, float2 odd) {
        if constexpr (KT == 2) return make_float2(__fadd_rn(even.x, odd.x), __fadd_rn(even.y, odd.y));
        else return fadd2(even, odd);
    }
    template <int M>
    static __device__ __forceinline__ float2 add_residual(const float2 *x, float inv_k, float2 z) {
        float2 xs = x[0];
#pragma unroll
        for (int i = 1; i < M; ++i) xs = fadd2(xs, x[i]);
        return ffma2(xs, f2(inv_k), z);
    }
    // One reverse step of a branch (parameters a, nxi, iz, km, lm; kmz = kappa m / zeta or
    // 1 / zeta): V^d[t] (vdt), V^d[t-1] (vdp) and dL/dZ[t] (dz; negated when kPaired) update the
    // adjoints Ad and the sums; gx receives dL/dX[t] + res.
    static __device__ __forceinline__ void branch_back(const float2 *a, const float2 *nxi, float2 iz, float2 km,
                                                       float2 lm, float2 kmz, const float2 *vdt,
                                                       const float2 *vdp, float2 dz, float2 res, float2 *Ad,
                                                       float2 *ga, float2 *gxi, float2 &gz, float2 &gk,
                                                       float2 *gx) {
        float2 u[G], ss;
#pragma unroll
        for (int q = 0; q < G; ++q) {
            u[q] = ffma2(vdt[q], iz, nxi[q]);
            ss = q == 0 ? fmul2(u[q], u[q]) : ffma2(u[q], u[q], ss);
        }
        if constexpr (kPaired) {
            const float2 ndz = dz;
            float2 y, du;
            if constexpr (PSI == PSI_MEXHAT) {
                const float2 e = exp2_2(ffma2(f2(kNegHalfLog2e), ss, lm));
                y = ffma2(minus2(ss), e, e);
                const float2 nw = ffma2(f2(2.f), e, y);
                du = KAPPA_FREE ? fmul2(fmul2(nw, u[0]), ndz) : fmul2(nw, fmul2(u[0], fmul2(km, ndz)));
            } else {
                const float2 ngy = fmul2(KAPPA_FREE ? lm : km, ndz);
                y = fmul2(lm, make_float2(fabsf(u[0].x), fabsf(u[0].y)));
                du = make_float2(u[0].x > 0.f ? -ngy.x : (u[0].x < 0.f ? ngy.x : 0.f),
                                 u[0].y > 0.f ? -ngy.y : (u[0].y < 0.f ? ngy.y : 0.f));
            }
            gxi[0] = fadd2(gxi[0], du);
            gz = ffma2(u[0], du, gz);
            gk = ffma2(y, ndz, gk);
            Ad[0] = ffma2(a[0], Ad[0], du);
            ga[0] = ffma2(Ad[0], vdp[0], ga[0]);
            gx[0] = ffma2(Ad[0], kmz, res);
        } else {
            const float2 gy = fmul2(km, dz);                     // dL/dY_b
            float2 y, qq, grr;                                   // Y_b; dL/du_i = qq u_i; (dL/dr) r
            if constexpr (PSI == PSI_MEXHAT) {
                const float2 e = exp2_2(fmul2(f2(kNegHalfLog2e), ss));
                y = ffma2(minus2(ss), e, e);
                qq = fmul2(fmul2(fadd2(ss, f2(-3.f)), e), gy);   // psi'(r) / r = (r^2 - 3) e
                grr = fmul2(ss, qq);
            } else {
                y = make_float2(sqrtf(ss.x), sqrtf(ss.y));
                qq = make_float2(y.x > 0.f ? __fdiv_rn(gy.x, y.x) : 0.f, y.y > 0.f ? __fdiv_rn(gy.y, y.y) : 0.f);
                grr = fmul2(gy, y);
            }
            gz = ffma2(grr, iz, gz);
            gk = ffma2(fmul2(lm, y), dz, gk);
#pragma unroll
            for (int q = 0; q < G; ++q) {
                const float2 d = fmul2(fmul2(qq, u[q]), iz);
                gxi[q] = fadd2(gxi[q], d);
                Ad[q] = ffma2(a[q], Ad[q], d);
                gx[q] = fadd2(Ad[q], res);
                ga[q] = ffma2(Ad[q], vdp[q], ga[q]);
            }
        }
    }
};

template <int KT, int G, int PSI, typename XT>
using Twin = TwinArith<KT, G, PSI, std::is_same<XT, float>::value>;

template <int LPN>
__device__ __forceinline__ float2 lanes_sum2(float2 v) {
    if constexpr (LPN >= 2) { v.x = lanes_sum<LPN>(v.x); v.y = lanes_sum<LPN>(v.y); }
    return v;
}

// A thread's place in the tile of the one-neuron-per-thread kernels: the columns p and p + 1
// (P is even), the rows of row lane ry (none when the columns do not exist).
struct TwinPos {
    int sub, p, ry, cx, nrows, chan;
    int64_t row0;
};
template <int LPN>
__device__ __forceinline__ TwinPos twin_pos(const Geometry &g) {
    TwinPos t;
    const int half = g.TXn / 2;
    t.sub = threadIdx.x % LPN;
    const int c = threadIdx.x / LPN;
    t.cx = 2 * (c % half);
    t.ry = c / half;
    const int ct = blockIdx.x % g.nCT;
    const int rg = blockIdx.x / g.nCT;
    const int p = ct * g.TXn + t.cx;
    const bool active = p < g.P;
    t.p = active ? p : g.P - 2;
    t.row0 = (int64_t)rg * g.R * g.TY + t.ry;
    const int64_t left = g.O - t.row0;
    t.nrows = left <= 0 || !active ? 0 : (int)min((int64_t)g.R, (left + g.TY - 1) / g.TY);
    t.chan = t.p / g.inner;
    return t;
}

// The steps of a chunk of n steps in LC slots. ALL: n == LC, slot = step. Else the chunk is
// taken apart into runs of 4, 2 and 1 steps (the bits of n) that sit in slots of their own (0-3,
// 4-5 and 6; for LC = 4: 0-1 and 2), in time order with gaps: one test per run instead of one
// per step, and the steps of a run are scheduled together.
template <int LC, bool ALL>
struct TwinSteps {
    template <typename F>
    static __device__ __forceinline__ void forward(int n, F f) {
        if constexpr (ALL) {
#pragma unroll
            for (int t = 0; t < LC; ++t) f(t);
        } else if constexpr (LC == 8) {
            if (n & 4) { f(0); f(1); f(2); f(3); }
            if (n & 2) { f(4); f(5); }
            if (n & 1) f(6);
        } else {
            if (n & 2) { f(0); f(1); }
            if (n & 1) f(2);
        }
    }
    template <typename F>
    static __device__ __forceinline__ void reverse(int n, F f) {
        if constexpr (ALL) {
#pragma unroll
            for (int t = LC - 1; t >= 0; --t) f(t);
        } else if constexpr (LC == 8) {
            if (n & 1) f(6);
            if (n & 2) { f(5); f(4); }
            if (n & 4) { f(3); f(2); f(1); f(0); }
        } else {
            if (n & 1) f(2);
            if (n & 2) { f(1); f(0); }
        }
    }
    // the step within the chunk that slot holds
    static __device__ __forceinline__ int step_of(int n, int slot) {
        if constexpr (ALL) return slot;
        else if constexpr (LC == 8) return slot < 4 ? slot : (slot < 6 ? (n & 4) + slot - 4 : n - 1);
        else return slot < 2 ? slot : n - 1;
    }
    // the value of the step before slot's: at(its slot), or e0 for the chunk's first step
    template <typename F>
    static __device__ __forceinline__ float2 before(int n, int slot, F at, float2 e0) {
        if (slot == 0) return e0;
        if constexpr (!ALL) {
            constexpr int r1 = LC == 8 ? 4 : 2, r2 = LC == 8 ? 6 : -1;       // first slots of the later runs
            const bool head = n >= r1 && (n & r1);                          // the first run is there
            if (slot == r1) return head ? at(r1 - 1) : e0;
            if (slot == r2) return (n & 2) ? at(5) : (head ? at(3) : e0);
        }
        return at(slot - 1);
    }
};

// The somas of a pair over the steps of a chunk: charge and fire (Eqs. methods-lif-reset-charge,
// -fire), and one step of the reverse recursion (Eq. methods-sg) from V^s[t] and dL/dS[t].
struct TwinSoma {
    float kv, cs, b_spike;
    bool soft, want_beta;
    __device__ __forceinline__ TwinSoma(const Params &P, int beta_wanted) {
        kv = (P.detach || P.soft) ? 0.f : -P.beta;
        cs = (P.detach || !P.soft) ? 0.f : -P.beta * P.theta;
        b_spike = P.soft ? P.beta : 0.f;
        soft = P.soft != 0;
        want_beta = beta_wanted != 0;
    }
    // one charge (soma_charge's operations) and the spikes after it
    template <bool SOFT>
    static __device__ __forceinline__ void charge(const Params &P, float2 z, float2 &v, bool &s1, bool &s2) {
        float2 leak;
        if constexpr (SOFT) {
            const float2 r = fadd2(v, f2(-P.theta));
            leak = make_float2(s1 ? r.x : v.x, s2 ? r.y : v.y);
        } else {
            leak = make_float2(s1 ? 0.f : v.x, s2 ? 0.f : v.y);
        }
        v = ffma2(f2(P.beta), leak, z);
        s1 = v.x >= P.theta;
        s2 = v.y >= P.theta;
    }
    __device__ __forceinline__ float2 back(const Params &P, float2 v, float2 gs, float2 dvn, float2 &gbeta) const {
        const bool s1 = v.x >= P.theta, s2 = v.y >= P.theta;
        if (want_beta) {
            const float l1 = s1 ? (soft ? __fsub_rn(v.x, P.theta) : 0.f) : v.x;
            const float l2 = s2 ? (soft ? __fsub_rn(v.y, P.theta) : 0.f) : v.y;
            gbeta = ffma2(dvn, make_float2(l1, l2), gbeta);
        }
        const float2 dvds = ffma2(f2(kv), v, f2(cs));
        const float2 dvdv = make_float2(s1 ? b_spike : P.beta, s2 ? b_spike : P.beta);
        const float2 ds = ffma2(dvds, dvn, gs);
        const float2 xd = fadd2(v, f2(-P.theta));
        const float2 qd = ffma2(fmul2(f2(9.869604401089358f), xd), xd, f2(1.f));
        return ffma2(make_float2(fast_rcp(qd.x), fast_rcp(qd.y)), ds, fmul2(dvdv, dvn));
    }
};

// base + k * stride bytes (stride < 2^32) as one instruction
__device__ __forceinline__ char *at_stride(char *base, uint32_t stride, uint32_t k) {
    uint64_t r;
    asm("mad.wide.u32 %0, %1, %2, %3;" : "=l"(r) : "r"(stride), "r"(k), "l"(reinterpret_cast<uint64_t>(base)));
    return reinterpret_cast<char *>(r);
}
__device__ __forceinline__ const char *at_stride(const char *base, uint32_t stride, uint32_t k) {
    return at_stride(const_cast<char *>(base), stride, k);
}

// block_partials for two columns per thread, in the same order: the first shuffle of its warp
// tree adds the columns p and p + 1, here the two halves of v.
template <int KT, int G, int LPN, int NT, int NA1>
__device__ __forceinline__ void twin_partials(const Geometry &g, const TwinPos &pos, float2 (&v)[NA1], float *red,
                                              float *partials) {
    constexpr int RS = red_stride<2 * NT>();
    if (g.seg > 1) {
#pragma unroll
        for (int a = 0; a < NA1; ++a) v[a].x = __fadd_rn(v[a].x, v[a].y);
        for (int d = 2; d < g.seg; d <<= 1) {
#pragma unroll
            for (int a = 0; a < NA1; ++a)
                v[a].x = __fadd_rn(v[a].x, __shfl_xor_sync(0xffffffffu, v[a].x, (d / 2) * LPN));
        }
    }
    __syncthreads();
    const int otid = (pos.ry * g.TXn + pos.cx) * LPN + pos.sub;
#pragma unroll
    for (int a = 0; a < NA1; ++a) {
        red[a * RS + otid] = v[a].x;
        if (g.seg == 1) red[a * RS + otid + LPN] = v[a].y;
    }
    __syncthreads();
    block_sums<KT, G, LPN, NT, RS, NA1>(g, red, partials);
}

// ---------------------------------------------------------------- backward
// Shared memory of one thread of the twin backward: x [LC][KT] and dL/dS [2][LC] of a chunk,
// the lane's parameters, and the parameter-gradient sums.
template <typename XT, int KT, int G, int LC>
struct TwinSmem {
    using W = typename TwinIO<XT>::W;
    static constexpr int KTb = KT / G;
    static constexpr int CB = G == 1 ? 2 : G;              // compartments per unit
    static constexpr int NU = KT / CB;                     // units
    static constexpr int NA = 2 * KT + 2 * KTb;            // parameters, and sums
    // a parameter as the pair it is used as (one 8-byte read), or for 8-compartment lanes, where
    // that would cost a resident block, once (two 4-byte reads)
    static constexpr bool kPairs = KT < 8;
    static constexpr size_t kX = sizeof(W) * KT * LC;      // bytes per thread
    static constexpr size_t kG = 2 * sizeof(W) * LC;
    static constexpr size_t kPar = (kPairs ? sizeof(float2) : sizeof(float)) * NA;
    static constexpr size_t kAcc = sizeof(float2) * NA;
    static constexpr size_t kBase = kX + kG + kPar + kAcc;
    // rows of several chunks: the adjoints, two checkpoints and (when kept) the row totals
    static constexpr size_t kMulti = sizeof(float2) * KT + 2 * sizeof(float2) * (KT + 1);
    static constexpr size_t bytes(bool multi, bool totals) {
        return kBase + (multi ? kMulti + (totals ? kAcc : 0) : 0);
    }
};
// Resident blocks the register cap leaves room for: 64-thread blocks (8-compartment lanes) six
// at 168 registers; 128-thread blocks three in the builds with both loops of an 8-step chunk and where
// the shared memory of 8 float32 steps allows no more, else four at 128 registers. Spills that are
// left (bytes stored and loaded, Mexican hat, bfloat16, K = 4, G = 2): 72 and 128 with complete 8-step
// chunks, 48 and 84 with both loops, 4 and 4 at T = 6.
template <int KT, typename XT, int LC, bool FULL>
constexpr int twin_min_blocks() {
    return KT == 8 ? 6 : (LC == 8 && (!FULL || sizeof(XT) == 4) ? 3 : 4);
}

// The backward in chunks of up to LC steps (L: the plan's chunk length; LC = L, or the number
// of steps of a single-chunk row). FULL: every chunk has LC steps; else complete chunks still
// run without bounds tests and the others with them. A chunk runs in three phases:
//   1. Z and V^s of the chunk are recomputed (the forward's operations, so the spikes are its
//      bits), unit by unit: a unit is a branch, or two with one compartment per branch;
//   2. the soma's reverse recursion in registers gives dL/dZ of every step;
//   3. unit by unit: V^d is rescanned into registers (one more multiply-add per step than
//      keeping it in shared memory, which would take more instructions to write and read), the
//      unit's slots of x take the next chunk's, and the reverse scan stores each dL/dX.
// Parameters, sums and adjoints live in shared memory and the unit loops are not unrolled, so
// only one unit's values occupy registers. x has a single buffer: its units arrive by cp.async
// one group each, and phase 1 of the next chunk waits for them one by one.
template <int K, int G, int PSI, typename XT, int L, int LC, bool FULL>
__global__ void __launch_bounds__(bwd_threads(bwd_lane_compartments(K, G, xt_code<XT>(), L)) / 2,
                                  twin_min_blocks<bwd_lane_compartments(K, G, xt_code<XT>(), L), XT, LC, FULL>())
dendsn_backward_twin_kernel(const BwdArgs A) {
    pdl_wait();
    constexpr int KT = bwd_lane_compartments(K, G, xt_code<XT>(), L);
    constexpr int NT = bwd_threads(KT) / 2, LPN = K / KT;
    constexpr bool MULTI = LC == 8;              // rows longer than LC come in chunks of 8
    using IO = TwinIO<XT>;
    using W = typename IO::W;
    using AR = Twin<KT, G, PSI, XT>;
    using S = TwinSmem<XT, KT, G, LC>;
    constexpr int KTb = S::KTb, CB = S::CB, NU = S::NU, NA = S::NA, BU = CB / G;
    constexpr bool TOTALS = MULTI && row_totals<K, G, XT, L>();
    // the paired engine's tree over two groups of four compartments (one group: the chain)
    constexpr bool TREE2 = std::is_same<XT, float>::value && G == 1 && KT == 8;
    const Geometry &g = A.g;
    const Params &P = A.p;
    const TwinPos pos = twin_pos<LPN>(g);
    const TwinSoma soma(P, A.want_beta);
    const float inv_k = 1.f / (float)K;
    const int T = g.T;
    const int nc = MULTI ? (T + LC - 1) / LC : 1;
    const int64_t BN = g.BN;
    const int64_t sXb = BN * K * (int64_t)sizeof(XT);                // bytes between steps of x
    const int64_t sGb = BN * (int64_t)sizeof(XT);                    // of dL/dS
    const uint32_t ksb = (uint32_t)g.inner * (uint32_t)sizeof(XT);   // between compartments
    const int64_t j0 = pos.row0 * g.P + pos.p;
    const int64_t jstep = (int64_t)g.TY * g.P;
    const int64_t rXb = jstep * K * (int64_t)sizeof(XT);             // between this thread's rows
    const int64_t xoff = lane_x_offset<1>(j0, pos.sub, KT, K, g.inner) * (int64_t)sizeof(XT);
    const char *const x0 = static_cast<const char *>(A.x) + xoff;
    char *const gx0 = static_cast<char *>(A.gx) + xoff;
    const char *const gs0 = static_cast<const char *>(A.gs) + j0 * (int64_t)sizeof(XT);
    const bool residual = P.residual != 0;
    const bool has_gv = A.gv != nullptr;

    extern __shared__ float4 smem_f4[];
    char *const sbase = reinterpret_cast<char *>(smem_f4);
    W *const xs = reinterpret_cast<W *>(sbase) + threadIdx.x;                        // [LC][KT][NT]
    W *const gr0 = reinterpret_cast<W *>(sbase + S::kX * NT) + threadIdx.x;          // [2][LC][NT]
    char *const par = sbase + (S::kX + S::kG) * NT;                                  // [NA][NT]
    float2 *const accs = reinterpret_cast<float2 *>(sbase + (S::kX + S::kG + S::kPar) * NT) + threadIdx.x;
    float2 *const ads = reinterpret_cast<float2 *>(sbase + S::kBase * NT) + threadIdx.x;         // [KT][NT]
    // [2]: V^d of the two neurons as NV vectors each; V^s [2][NT]
    using CkV = typename Vec<float, (KT < 4 ? KT : 4)>::Raw;
    constexpr int NV = KT < 4 ? 1 : KT / 4, CW = KT < 4 ? KT : 4;
    CkV *const ckd0 = reinterpret_cast<CkV *>(sbase + (S::kBase + sizeof(float2) * KT) * NT) + threadIdx.x;
    float2 *const ckv0 = reinterpret_cast<float2 *>(sbase + (S::kBase + 3 * sizeof(float2) * KT) * NT) + threadIdx.x;
    float2 *const tots = reinterpret_cast<float2 *>(sbase + (S::kBase + S::kMulti) * NT) + threadIdx.x;
    const bool use_tot = TOTALS && nc > 1;

    // parameters of the lane: alpha KT | -xi/zeta KT | 1/zeta KTb | kappa KTb, and the mask bits
    // of the two neurons (kappa m is a select on them)
    auto put = [&](int i, float v) {
        if constexpr (S::kPairs) reinterpret_cast<float2 *>(par)[i * NT + threadIdx.x] = f2(v);
        else reinterpret_cast<float *>(par)[i * NT + threadIdx.x] = v;
    };
    // read back as a pair of registers the compiler does not know to be equal: it would
    // otherwise rebuild the pair from one register at every use (two moves)
    auto get = [&](int i) {
        float2 v;
        if constexpr (S::kPairs) {
            v = reinterpret_cast<const float2 *>(par)[i * NT + threadIdx.x];
        } else {
            const volatile float *p = reinterpret_cast<const volatile float *>(par) + i * NT + threadIdx.x;
            v.x = *p;
            v.y = *p;
        }
        return v;
    };
    uint32_t mb1 = ~0u, mb2 = ~0u;
    {
        float a[KT], nxi[KT], iz[KTb], km[KTb], mk[KTb], kap[KTb];
        load_param_arrays<KT, G>(P, g, pos.chan, pos.sub, a, nxi, iz, km, mk);
        lane_kappa<KTb>(P, g, pos.chan, pos.sub, kap);
#pragma unroll
        for (int i = 0; i < KT; ++i) { put(i, a[i]); put(KT + i, nxi[i]); }
#pragma unroll
        for (int b = 0; b < KTb; ++b) {
            // a channel's kappa m is a product, in the forward too: NaN for a kappa that is not finite
            const bool nan = km[b] != km[b];
            put(2 * KT + b, iz[b]);
            put(2 * KT + KTb + b, nan ? km[b] : kap[b]);
            if (mk[b] == 0.f && !nan) { mb1 &= ~(1u << b); mb2 &= ~(1u << b); }
        }
    }
#pragma unroll 1
    for (int q = 0; q < NA; ++q) {
        accs[q * NT] = f2(0.f);
        if (use_tot) tots[q * NT] = f2(0.f);
    }
    struct Branch { float2 a[G], nxi[G], iz, km, lm; };
    auto branch = [&](int b) {
        Branch r;
#pragma unroll
        for (int q = 0; q < G; ++q) {
            r.a[q] = get(b * G + q);
            r.nxi[q] = get(KT + b * G + q);
        }
        r.iz = get(2 * KT + b);
        const float2 kap = get(2 * KT + KTb + b);
        const bool on1 = (mb1 >> b) & 1u, on2 = (mb2 >> b) & 1u;
        r.km = make_float2(on1 ? kap.x : 0.f, on2 ? kap.y : 0.f);
        r.lm = make_float2(AR::mask_term(on1 ? 1.f : 0.f), AR::mask_term(on2 ? 1.f : 0.f));
        return r;
    };
    // x of unit u, and dL/dS with the checkpoint, of chunk c of this thread's row i
    auto fetch_x = [&](int i, int c, int u) {
        const int n = FULL ? LC : min(LC, T - c * LC);
        const char *xp = x0 + i * rXb + c * LC * sXb + (uint64_t)ksb * (uint32_t)(u * CB);
        W *const xu = xs + u * CB * NT;
        auto step = [&](int tt) {
#pragma unroll
            for (int q = 0; q < CB; ++q) cp_async<sizeof(W)>(xu + (tt * KT + q) * NT, q ? at_stride(xp, ksb, q) : xp, 0.f);
            xp += sXb;
        };
        if (FULL || (MULTI && n == LC)) TwinSteps<LC, true>::forward(n, step);
        else TwinSteps<LC, false>::forward(n, step);
    };
    auto fetch_g = [&](int i, int c, int buf) {
        const int n = FULL ? LC : min(LC, T - c * LC);
        const char *gp = gs0 + i * (jstep * (int64_t)sizeof(XT)) + c * LC * sGb;
        W *const gr = gr0 + buf * (LC * NT);
        auto step = [&](int tt) {
            cp_async<sizeof(W)>(gr + tt * NT, gp, 0.f);
            gp += sGb;
        };
        if (FULL || (MULTI && n == LC)) TwinSteps<LC, true>::forward(n, step);
        else TwinSteps<LC, false>::forward(n, step);
        if (MULTI && c > 0) {
            const int64_t j = j0 + i * jstep;
            const float *d = A.ck_vd + ((int64_t)(c - 1) * BN + j) * K + pos.sub * KT;
#pragma unroll
            for (int q = 0; q < NV; ++q) {
                cp_async<sizeof(CkV)>(ckd0 + ((buf * 2) * NV + q) * NT, d + CW * q, 0.f);
                cp_async<sizeof(CkV)>(ckd0 + ((buf * 2 + 1) * NV + q) * NT, d + K + CW * q, 0.f);
            }
            cp_async<8>(ckv0 + buf * NT, A.ck_vs + (int64_t)(c - 1) * BN + j, 0.f);
        }
    };
    // one group per unit; the first also carries dL/dS and the checkpoint
    if (pos.nrows > 0) fetch_g(0, nc - 1, 0);
#pragma unroll 1
    for (int u = 0; u < NU; ++u) {
        if (pos.nrows > 0) fetch_x(0, nc - 1, u);
        cp_async_commit();
    }

    float2 gbeta = f2(0.f), gbtot = f2(0.f);
    int buf = 0;
    // with several lanes per neuron the lanes exchange Z, so the rows of a warp's threads (two
    // row lanes may share a warp) run together: the warp's first thread has the most rows
    const int nloop = LPN > 1 ? __shfl_sync(0xffffffffu, pos.nrows, 0) : pos.nrows;
    for (int i = 0; i < nloop; ++i) {
        const bool live = LPN == 1 || i < pos.nrows;
        if (P.mask_mode == 2 && live) {
            const int64_t n = (j0 + i * jstep) % g.N;
            const uint8_t *m1 = P.mask + n * g.Kb + pos.sub * KTb;
            mb1 = mb2 = 0u;
#pragma unroll
            for (int b = 0; b < KTb; ++b) {
                mb1 |= (__ldg(m1 + b) != 0 ? 1u : 0u) << b;
                mb2 |= (__ldg(m1 + g.Kb + b) != 0 ? 1u : 0u) << b;
            }
        }
        float2 dvn = f2(0.f);                                    // dL/dV^s[t+1]
        for (int c = nc - 1; c >= 0; --c) {
            const int t0 = c * LC;
            const int ncur = FULL ? LC : min(LC, T - t0);
            const W *const gr = gr0 + buf * (LC * NT);
            // state entering the chunk: zero at t = 0, else the forward's checkpoint
            auto entering = [&](int k) -> float2 {
                if (!MULTI || c == 0) return f2(0.f);
                return make_float2(reinterpret_cast<const float *>(ckd0 + (buf * 2 * NV + k / CW) * NT)[k % CW],
                                   reinterpret_cast<const float *>(ckd0 + ((buf * 2 + 1) * NV + k / CW) * NT)[k % CW]);
            };
            auto chunk = [&](auto full) {
                using Steps = TwinSteps<LC, decltype(full)::value>;
                // phase 1: Z of the chunk unit by unit, then V^s
                float2 vs[LC];
                {
                    float2 ze[LC], zo[LC];       // one compartment per branch: even and odd chains
#pragma unroll
                    for (int tt = 0; tt < LC; ++tt) {
                        vs[tt] = f2(0.f);
                        if constexpr (G == 1) { ze[tt] = f2(0.f); zo[tt] = f2(0.f); }
                    }
                    // adds the residual of n compartments from k0 to z
                    auto with_residual = [&](int tt, int k0, int n, float2 z) {
                        float2 s = IO::unpack(xs[(tt * KT + k0) * NT]);
                        for (int k = 1; k < n; ++k) s = fadd2(s, IO::unpack(xs[(tt * KT + k0 + k) * NT]));
                        return ffma2(s, f2(inv_k), z);
                    };
#pragma unroll 1
                    for (int u = 0; u < NU; ++u) {
                        // all but the newest NU - 1 groups: unit u (and those before it) is there
                        cp_async_wait<NU - 1>();
                        cp_async_commit();
                        const W *const xu = xs + u * CB * NT;
#pragma unroll
                        for (int h = 0; h < BU; ++h) {
                            const Branch r = branch(u * BU + h);
                            float2 v[G];
#pragma unroll
                            for (int q = 0; q < G; ++q) v[q] = entering((u * BU + h) * G + q);
                            Steps::forward(ncur, [&](int tt) {
#pragma unroll
                                for (int q = 0; q < G; ++q)
                                    v[q] = ffma2(r.a[q], v[q], IO::unpack(xu[(tt * KT + h * G + q) * NT]));
                                const float2 y = AR::branch_y(r.nxi, r.iz, v);
                                if constexpr (G > 1) vs[tt] = ffma2(r.km, y, vs[tt]);
                                else if (h == 0) ze[tt] = ffma2(r.km, y, ze[tt]);
                                else zo[tt] = ffma2(r.km, y, zo[tt]);
                            });
                        }
                        if constexpr (TREE2) {
                            if (u & 1) {         // a group of four compartments is complete
                                Steps::forward(ncur, [&](int tt) {
                                    float2 z = fadd2(ze[tt], zo[tt]);
                                    if (residual) z = with_residual(tt, (u - 1) * CB, 4, z);
                                    vs[tt] = u == 1 ? z : fadd2(vs[tt], z);
                                    ze[tt] = f2(0.f);
                                    zo[tt] = f2(0.f);
                                });
                            }
                        }
                    }
                    Steps::forward(ncur, [&](int tt) {
                        float2 z = vs[tt];
                        if constexpr (G == 1 && !TREE2) z = AR::add_products(ze[tt], zo[tt]);
                        if constexpr (!TREE2) {
                            if (residual) z = with_residual(tt, 0, KT, z);
                        }
                        vs[tt] = lanes_sum2<LPN>(z);
                    });
                    auto somas = [&](auto soft) {
                        float2 v = (!MULTI || c == 0) ? f2(0.f) : ckv0[buf * NT];
                        bool s1 = MULTI && c > 0 && v.x >= P.theta, s2 = MULTI && c > 0 && v.y >= P.theta;
                        Steps::forward(ncur, [&](int tt) {
                            TwinSoma::charge<decltype(soft)::value>(P, vs[tt], v, s1, s2);
                            vs[tt] = v;
                        });
                    };
                    if (P.soft) somas(std::true_type{});
                    else somas(std::false_type{});
                }
                // phase 2: dL/dV^s backwards in time (dL/dZ = dL/dV^s; negated for the paired
                // engine's formulas), over vs
                if (live) {
                    Steps::reverse(ncur, [&](int tt) {
                        float2 dv = soma.back(P, vs[tt], IO::unpack(gr[tt * NT]), dvn, gbeta);
                        if (has_gv) {
                            const float *gp = A.gv + j0 + i * jstep + (int64_t)(t0 + Steps::step_of(ncur, tt)) * BN;
                            dv = fadd2(dv, make_float2(__ldcs(gp), __ldcs(gp + 1)));
                        }
                        vs[tt] = AR::kPaired ? minus2(dv) : dv;
                        dvn = dv;
                    });
                }
                // phase 3: unit by unit, V^d forward, the next chunk's x into the freed slots,
                // then the reverse scan
                const bool same_row = c > 0;
                const bool more = same_row ? live : i + 1 < pos.nrows;
                const int in = same_row ? i : i + 1, cn = same_row ? c - 1 : nc - 1;
                if (more) fetch_g(in, cn, buf ^ 1);
                char *gu = gx0 + i * rXb + (t0 + ncur - 1) * sXb;    // the unit's dL/dX, last step
                const float res_k = residual ? (AR::kPaired ? -inv_k : inv_k) : 0.f;
#pragma unroll 1
                for (int u = 0; u < NU; ++u) {
                    const W *const xu = xs + u * CB * NT;
                    float2 vd[LC][CB];
#pragma unroll
                    for (int q = 0; q < CB; ++q) {
                        const float2 a = get(u * CB + q);
                        float2 v = entering(u * CB + q);
                        Steps::forward(ncur, [&](int tt) {
                            v = ffma2(a, v, IO::unpack(xu[(tt * KT + q) * NT]));
                            vd[tt][q] = v;
                        });
                    }
                    // into the slots just read: the copies are volatile and clobber memory, so they
                    // stay behind the reads above without an operand that depends on them
                    if (more) fetch_x(in, cn, u);
                    cp_async_commit();
                    if (live) {
#pragma unroll
                        for (int h = 0; h < BU; ++h) {
                            const int b = u * BU + h;
                            const Branch r = branch(b);
                            const float2 kmz = AR::KAPPA_FREE ? fmul2(r.km, r.iz) : r.iz;
                            float2 Ad[G], ga[G], gxi[G], e0[G];
#pragma unroll
                            for (int q = 0; q < G; ++q) {
                                Ad[q] = (MULTI && c < nc - 1) ? ads[(b * G + q) * NT] : f2(0.f);
                                ga[q] = accs[(b * G + q) * NT];
                                gxi[q] = accs[(KT + b * G + q) * NT];
                                e0[q] = entering(b * G + q);
                            }
                            float2 gz = accs[(2 * KT + b) * NT], gk = accs[(2 * KT + KTb + b) * NT];
                            char *gp = h ? at_stride(gu, ksb, h * G) : gu;
                            Steps::reverse(ncur, [&](int tt) {
                                float2 gxv[G], vdp[G];
#pragma unroll
                                for (int q = 0; q < G; ++q)
                                    vdp[q] = Steps::before(ncur, tt, [&](int r) { return vd[r][h * G + q]; }, e0[q]);
                                AR::branch_back(r.a, r.nxi, r.iz, r.km, r.lm, kmz, &vd[tt][h * G], vdp, vs[tt],
                                                residual ? fmul2(vs[tt], f2(res_k)) : f2(0.f), Ad, ga, gxi, gz, gk,
                                                gxv);
#pragma unroll
                                for (int q = 0; q < G; ++q)
                                    __stcs(reinterpret_cast<W *>(q ? at_stride(gp, ksb, q) : gp), IO::pack(gxv[q]));
                                gp -= sXb;
                            });
#pragma unroll
                            for (int q = 0; q < G; ++q) {
                                if (MULTI && c > 0) ads[(b * G + q) * NT] = Ad[q];
                                accs[(b * G + q) * NT] = ga[q];
                                accs[(KT + b * G + q) * NT] = gxi[q];
                            }
                            accs[(2 * KT + b) * NT] = gz;
                            accs[(2 * KT + KTb + b) * NT] = gk;
                        }
                    }
                    gu += (uint64_t)ksb * (uint32_t)CB;
                }
            };
            if constexpr (FULL) chunk(std::true_type{});
            else if constexpr (!MULTI) chunk(std::false_type{});
            else if (ncur == LC) chunk(std::true_type{});
            else chunk(std::false_type{});
            buf ^= 1;
        }
        if (use_tot) {
#pragma unroll 1
            for (int q = 0; q < NA; ++q) {
                tots[q * NT] = fadd2(tots[q * NT], accs[q * NT]);
                accs[q * NT] = f2(0.f);
            }
            gbtot = fadd2(gbtot, gbeta);
            gbeta = f2(0.f);
        }
    }

    // parameter-gradient sums [alpha KT | xi KT | zeta KTb | kappa KTb | beta]: the paired
    // engine's first three carry 1/zeta (or kappa/zeta) here, and its all but the first are negated
    constexpr int NA1 = NA + 1;
    float2 v[NA1];
    const float2 *const sums = use_tot ? tots : accs;
#pragma unroll
    for (int q = 0; q < NA; ++q) {
        v[q] = sums[q * NT];
        if constexpr (AR::kPaired) {
            const float2 iz = get(2 * KT + q % KT);
            if (q < 3 * KT) v[q] = fmul2(v[q], AR::KAPPA_FREE ? fmul2(get(2 * KT + KTb + q % KT), iz) : iz);
            if (q >= KT) v[q] = neg2(v[q]);
        } else {
            if (q >= KT && q < 2 * KT + KTb) v[q] = neg2(v[q]);
        }
    }
    v[NA] = (soma.want_beta && pos.sub == 0) ? (use_tot ? gbtot : gbeta) : f2(0.f);
#pragma unroll
    for (int a = 0; a < NA1; ++a)
        if (a < KT && P.stateless) v[a] = f2(0.f);
    cp_async_wait<0>();
    pdl_trigger();
    twin_partials<KT, G, LPN, NT>(g, pos, v, reinterpret_cast<float *>(sbase), A.partials);
}

// ---------------------------------------------------------------- backward, rows of up to 4 steps
template <typename XT, int KT>
struct TwinShort {
    static constexpr size_t kX = sizeof(typename TwinIO<XT>::W) * KT * 4;     // bytes per thread
    static constexpr size_t kBytes = 2 * (kX + sizeof(typename TwinIO<XT>::W) * 4);
};

// Lanes of up to 4 compartments and rows of one chunk of 4 steps: a row is too short to pay for
// parameters and sums in shared memory (they would be read and written back once per unit and
// row), so both stay in registers, and x and dL/dS of a row arrive a whole row ahead in two
// buffers. The phases are those of dendsn_backward_twin_kernel, with the unit loops unrolled.
// FULL: T == 4.
template <int K, int G, int PSI, typename XT, bool FULL>
__global__ void __launch_bounds__(128, 3)
dendsn_backward_twin_short_kernel(const BwdArgs A) {
    pdl_wait();
    constexpr int L = 4;
    constexpr int KT = bwd_lane_compartments(K, G, xt_code<XT>(), L);
    constexpr int NT = bwd_threads(KT) / 2;
    constexpr int LPN = K / KT;
    constexpr int KTb = KT / G;
    static_assert(KT <= 4 && NT == 128, "narrow lanes");
    using IO = TwinIO<XT>;
    using W = typename IO::W;
    using AR = Twin<KT, G, PSI, XT>;
    using S = TwinShort<XT, KT>;
    const Geometry &g = A.g;
    const Params &P = A.p;
    const TwinPos pos = twin_pos<LPN>(g);
    const TwinSoma soma(P, A.want_beta);
    const float inv_k = 1.f / (float)K;
    const int T = g.T;
    const int n = FULL ? L : T;                  // steps of a row
    using Steps = TwinSteps<L, FULL>;
    const int64_t BN = g.BN;
    const int64_t sXb = BN * K * (int64_t)sizeof(XT);              // bytes between steps of x
    const int64_t sGb = BN * (int64_t)sizeof(XT);                  // of dL/dS
    const uint32_t ksb = (uint32_t)g.inner * (uint32_t)sizeof(XT);   // between compartments
    const int64_t j0 = pos.row0 * g.P + pos.p;
    const int64_t jstep = (int64_t)g.TY * g.P;
    const int64_t rXb = jstep * K * (int64_t)sizeof(XT);             // between this thread's rows
    const int64_t xoff = lane_x_offset<1>(j0, pos.sub, KT, K, g.inner) * (int64_t)sizeof(XT);
    const char *const x0 = static_cast<const char *>(A.x) + xoff;
    char *const gx0 = static_cast<char *>(A.gx) + xoff;
    const char *const gs0 = static_cast<const char *>(A.gs) + j0 * (int64_t)sizeof(XT);
    const bool residual = P.residual != 0;
    const bool has_gv = A.gv != nullptr;

    extern __shared__ float4 smem_f4[];
    char *const sbase = reinterpret_cast<char *>(smem_f4);
    typename AR::LP lp;
    AR::load(P, g, pos.chan, pos.sub, lp);
    W *const xs0 = reinterpret_cast<W *>(sbase) + threadIdx.x;                       // [2][L][KT][NT]
    W *const gr0 = reinterpret_cast<W *>(sbase + 2 * S::kX * NT) + threadIdx.x;      // [2][L][NT]
    auto fetch = [&](int i) {
        const char *xp = x0 + i * rXb;
        const char *gp = gs0 + i * (jstep * (int64_t)sizeof(XT));
        W *const xs = xs0 + (i & 1) * (L * KT * NT);
        W *const gr = gr0 + (i & 1) * (L * NT);
        Steps::forward(n, [&](int tt) {
#pragma unroll
            for (int k = 0; k < KT; ++k) cp_async<sizeof(W)>(xs + (tt * KT + k) * NT, k ? at_stride(xp, ksb, k) : xp, 0.f);
            cp_async<sizeof(W)>(gr + tt * NT, gp, 0.f);
            xp += sXb;
            gp += sGb;
        });
    };
    if (pos.nrows > 0) fetch(0);
    cp_async_commit();

    float2 ga[KT], gxi[KT], gz[KTb], gk[KTb];
#pragma unroll
    for (int k = 0; k < KT; ++k) { ga[k] = f2(0.f); gxi[k] = f2(0.f); }
#pragma unroll
    for (int b = 0; b < KTb; ++b) { gz[b] = f2(0.f); gk[b] = f2(0.f); }
    float2 gbeta = f2(0.f);
    // lanes of one neuron exchange Z: the rows of a warp run together (see the twin kernel)
    const int nloop = LPN > 1 ? __shfl_sync(0xffffffffu, pos.nrows, 0) : pos.nrows;
    for (int i = 0; i < nloop; ++i) {
        const bool live = LPN == 1 || i < pos.nrows;
        if (P.mask_mode == 2 && live)
            AR::neuron_masks(P, g, (j0 + i * jstep) % g.N, pos.chan, pos.sub, lp);
        cp_async_wait<0>();
        // the next row goes to the buffer the previous one has been read from
        if (i + 1 < pos.nrows) fetch(i + 1);
        cp_async_commit();
        const W *const xs = xs0 + (i & 1) * (L * KT * NT);
        const W *const gr = gr0 + (i & 1) * (L * NT);
        // phase 1: Z and V^s of the row
        float2 vs[L];
        {
            float2 vd[KT];
#pragma unroll
            for (int k = 0; k < KT; ++k) vd[k] = f2(0.f);
            float2 v = f2(0.f);
            bool s1 = false, s2 = false;
            Steps::forward(n, [&](int tt) {
                float2 xv[KT];
#pragma unroll
                for (int k = 0; k < KT; ++k) xv[k] = IO::unpack(xs[(tt * KT + k) * NT]);
                const float2 z = lanes_sum2<LPN>(AR::step(lp, vd, xv, residual, inv_k));
                if (P.soft) TwinSoma::charge<true>(P, z, v, s1, s2);
                else TwinSoma::charge<false>(P, z, v, s1, s2);
                vs[tt] = v;
            });
        }
        if (!live) continue;
        // phase 2: dL/dV^s backwards in time, over vs
        float2 dvn = f2(0.f);
        Steps::reverse(n, [&](int tt) {
            float2 dv = soma.back(P, vs[tt], IO::unpack(gr[tt * NT]), dvn, gbeta);
            if (has_gv) {
                const float *gp = A.gv + j0 + i * jstep + (int64_t)Steps::step_of(n, tt) * BN;
                dv = fadd2(dv, make_float2(__ldcs(gp), __ldcs(gp + 1)));
            }
            vs[tt] = AR::kPaired ? minus2(dv) : dv;
            dvn = dv;
        });
        // phase 3: branch by branch, V^d forward, then the reverse scan
        char *const gxr = gx0 + i * rXb + (n - 1) * sXb;
        const float res_k = AR::kPaired ? -inv_k : inv_k;
#pragma unroll
        for (int b = 0; b < KTb; ++b) {
            asm volatile("" ::: "memory");       // one branch at a time: keeps its registers apart
            float2 vd[L][G], Ad[G];
#pragma unroll
            for (int q = 0; q < G; ++q) {
                Ad[q] = f2(0.f);
                float2 v = f2(0.f);
                Steps::forward(n, [&](int tt) {
                    v = ffma2(lp.a[b * G + q], v, IO::unpack(xs[(tt * KT + b * G + q) * NT]));
                    vd[tt][q] = v;
                });
            }
            char *gp = b ? at_stride(gxr, ksb, b * G) : gxr;
            Steps::reverse(n, [&](int tt) {
                float2 gxv[G], vdp[G];
#pragma unroll
                for (int q = 0; q < G; ++q)
                    vdp[q] = Steps::before(n, tt, [&](int r) { return vd[r][q]; }, f2(0.f));
                AR::branch_back(&lp.a[b * G], &lp.nxi[b * G], lp.iz[b], lp.km[b], lp.lm[b], lp.iz[b], vd[tt], vdp,
                                vs[tt], residual ? fmul2(vs[tt], f2(res_k)) : f2(0.f), Ad, &ga[b * G], &gxi[b * G],
                                gz[b], gk[b], gxv);
#pragma unroll
                for (int q = 0; q < G; ++q)
                    __stcs(reinterpret_cast<W *>(q ? at_stride(gp, ksb, q) : gp), IO::pack(gxv[q]));
                gp -= sXb;
            });
        }
    }

    // [alpha KT | xi KT | zeta KTb | kappa KTb | beta], signs and scales as in the twin kernel
    constexpr int NA1 = 2 * KT + 2 * KTb + 1;
    float2 v[NA1];
#pragma unroll
    for (int k = 0; k < KT; ++k) {
        v[k] = AR::kPaired ? fmul2(ga[k], lp.iz[k / G]) : ga[k];
        v[KT + k] = neg2(AR::kPaired ? fmul2(gxi[k], lp.iz[k / G]) : gxi[k]);
    }
#pragma unroll
    for (int b = 0; b < KTb; ++b) {
        v[2 * KT + b] = neg2(AR::kPaired ? fmul2(gz[b], lp.iz[b]) : gz[b]);
        v[2 * KT + KTb + b] = AR::kPaired ? neg2(gk[b]) : gk[b];
    }
    v[NA1 - 1] = (soma.want_beta && pos.sub == 0) ? gbeta : f2(0.f);
#pragma unroll
    for (int a = 0; a < NA1; ++a)
        if (a < KT && P.stateless) v[a] = f2(0.f);
    cp_async_wait<0>();
    pdl_trigger();
    twin_partials<KT, G, LPN, NT>(g, pos, v, reinterpret_cast<float *>(sbase), A.partials);
}

// ---------------------------------------------------------------- forward
// float32 rows: bound by memory (the conv layer with P = 4 compartments on 2 branches runs at
// 0.97 of the copy rate, 103 us, from 106.5 us on one neuron per thread), so a ring of 8 steps
// per thread in any order of rows and steps does; 16 compartments, which the one-neuron kernel
// reads in 4-byte pieces, went from 601 to 267 us (T = 5, B = 8, 192 x 56 x 56, identity).
constexpr int kTwinFwdDepth = 8;
constexpr int kTwinFwdThreads = 128;

template <int K, int G, int PSI, typename XT>
__global__ void __launch_bounds__(kTwinFwdThreads, 4)
dendsn_forward_twin_kernel(const FwdArgs A) {
    pdl_wait();
    constexpr int NT = kTwinFwdThreads;
    constexpr int KT = lane_compartments(K);
    constexpr int LPN = K / KT;
    using IO = TwinIO<XT>;
    using W = typename IO::W;
    using AR = Twin<KT, G, PSI, XT>;
    constexpr int D = kTwinFwdDepth;
    const Geometry &g = A.g;
    const Params &P = A.p;
    const TwinPos pos = twin_pos<LPN>(g);
    // lanes of one neuron exchange Z: rows run together in a warp (see the backward)
    const int nloop = LPN > 1 ? __shfl_sync(0xffffffffu, pos.nrows, 0) : pos.nrows;
    if (nloop == 0) return;
    typename AR::LP lp;
    AR::load(P, g, pos.chan, pos.sub, lp);
    const float inv_k = 1.f / (float)K;
    const int T = g.T;
    const int64_t sX = g.BN * K;
    const int64_t BN = g.BN;
    const int64_t ks = g.inner;
    const int64_t j0 = pos.row0 * g.P + pos.p;
    const int64_t jstep = (int64_t)g.TY * g.P;
    const int64_t rX = jstep * K;
    XT *sp = static_cast<XT *>(A.spikes) + j0;
    float *vp = A.v_out ? A.v_out + j0 : nullptr;
    const bool write_ck = A.ck_vd != nullptr && g.n_ck > 0;
    const bool residual = P.residual != 0;

    extern __shared__ float4 fwd_smem[];
    W *const ring = reinterpret_cast<W *>(fwd_smem) + threadIdx.x;   // [D][KT][NT]
    const XT *ip = static_cast<const XT *>(A.x) + lane_x_offset<1>(j0, pos.sub, KT, K, g.inner);
    int it = 0, ir = 0;                          // step and row of the next fetch
    const int64_t row_jump = rX - (int64_t)T * sX;
    auto fetch = [&](W *slot, float dep) {
        if (ir < pos.nrows) {
#pragma unroll
            for (int k = 0; k < KT; ++k) cp_async<sizeof(W)>(slot + k * NT, ip + k * ks, dep);
        }
        cp_async_commit();
        ip += sX;
        if (++it == T) { it = 0; ++ir; ip += row_jump; }
    };
#pragma unroll
    for (int d = 0; d < D; ++d) fetch(ring + d * KT * NT, 0.f);
    W *slot = ring;
    for (int i = 0; i < nloop; ++i) {
        const bool live = LPN == 1 || i < pos.nrows;
        if (P.mask_mode == 2 && live)
            AR::neuron_masks(P, g, (j0 + i * jstep) % g.N, pos.chan, pos.sub, lp);
        float2 vd[KT];
#pragma unroll
        for (int k = 0; k < KT; ++k) vd[k] = f2(0.f);
        float2 v = f2(0.f);
        bool s1 = false, s2 = false;
        XT *spt = sp;
        float *vpt = vp;
        for (int t = 0; t < T; ++t) {
            cp_async_wait<D - 1>();
            float2 xv[KT];
#pragma unroll
            for (int k = 0; k < KT; ++k) xv[k] = IO::unpack(slot[k * NT]);
            const float2 z = lanes_sum2<LPN>(AR::step(lp, vd, xv, residual, inv_k));
            fetch(slot, __fadd_rn(z.x, z.y));    // z depends on the slot's values: refill it
            slot = slot == ring + (D - 1) * KT * NT ? ring : slot + KT * NT;
            if (P.soft) TwinSoma::charge<true>(P, z, v, s1, s2);
            else TwinSoma::charge<false>(P, z, v, s1, s2);
            if (live && pos.sub == 0) {
                __stcs(reinterpret_cast<W *>(spt), IO::pack(make_float2(s1 ? 1.f : 0.f, s2 ? 1.f : 0.f)));
                if (vpt) __stcs(reinterpret_cast<float2 *>(vpt), v);
            }
            spt += BN;
            if (vpt) vpt += BN;
            if (write_ck && live && ((t + 1) & (g.L - 1)) == 0 && t + 1 < T) {
                const int64_t ck = (int64_t)((t + 1) / g.L - 1) * BN + j0 + i * jstep;
                float va[KT], vb[KT];
#pragma unroll
                for (int k = 0; k < KT; ++k) { va[k] = vd[k].x; vb[k] = vd[k].y; }
                Vec<float, KT>::store(A.ck_vd + ck * K + pos.sub * KT, va);
                Vec<float, KT>::store(A.ck_vd + (ck + 1) * K + pos.sub * KT, vb);
                if (pos.sub == 0) __stcs(reinterpret_cast<float2 *>(A.ck_vs + ck), v);
            }
        }
        sp += jstep;
        if (vp) vp += jstep;
    }
    pdl_trigger();
    cp_async_wait<0>();
}

// bfloat16 rows: the forward in chunks of up to LC steps (FULL: every chunk has LC), each
// chunk's x in a buffer of its own, fetched NB - 1 chunks ahead. Half the bytes of float32 per
// step leave this forward bound by instructions rather than by memory: with the steps of a
// chunk unrolled no ring position, fetch walker or output test is left per step.
template <int KT, int LC> constexpr int twin_fwd_buffers() { return LC == 4 && KT < 8 ? 4 : 2; }
template <int K, int G, int PSI, int LC, bool FULL>
__global__ void __launch_bounds__(kTwinFwdThreads, 4)
dendsn_forward_twin_chunk_kernel(const FwdArgs A) {
    pdl_wait();
    using XT = __nv_bfloat16;
    constexpr int NT = kTwinFwdThreads;
    constexpr int KT = lane_compartments(K);
    constexpr int LPN = K / KT, NB = twin_fwd_buffers<KT, LC>();
    constexpr bool MULTI = LC == 8;
    using IO = TwinIO<XT>;
    using W = typename IO::W;
    using AR = Twin<KT, G, PSI, XT>;
    const Geometry &g = A.g;
    const Params &P = A.p;
    const TwinPos pos = twin_pos<LPN>(g);
    // lanes of one neuron exchange Z: rows run together in a warp (see the backward)
    const int nloop = LPN > 1 ? __shfl_sync(0xffffffffu, pos.nrows, 0) : pos.nrows;
    if (nloop == 0) return;
    typename AR::LP lp;
    AR::load(P, g, pos.chan, pos.sub, lp);
    const float inv_k = 1.f / (float)K;
    const int T = g.T;
    const int nc = MULTI ? (T + LC - 1) / LC : 1;
    const int64_t BN = g.BN;
    const int64_t sXb = BN * K * (int64_t)sizeof(XT);                // bytes between steps of x
    const uint32_t ksb = (uint32_t)g.inner * (uint32_t)sizeof(XT);   // between compartments
    const int64_t j0 = pos.row0 * g.P + pos.p;
    const int64_t jstep = (int64_t)g.TY * g.P;
    const char *const x0 = static_cast<const char *>(A.x) +
                           lane_x_offset<1>(j0, pos.sub, KT, K, g.inner) * (int64_t)sizeof(XT);
    const bool write_ck = MULTI && A.ck_vd != nullptr && g.n_ck > 0;
    const bool residual = P.residual != 0;

    extern __shared__ float4 fwd_smem[];
    W *const xs0 = reinterpret_cast<W *>(fwd_smem) + threadIdx.x;    // [NB][LC][KT][NT]
    int fi = 0, fc = 0, fb = 0;                  // row, chunk and buffer of the next fetch
    auto fetch = [&]() {
        if (fi < pos.nrows) {
            const int n = FULL ? LC : min(LC, T - fc * LC);
            const char *xp = x0 + fi * (jstep * K * (int64_t)sizeof(XT)) + fc * LC * sXb;
            W *const xs = xs0 + fb * (LC * KT * NT);
            auto step = [&](int tt) {
#pragma unroll
                for (int k = 0; k < KT; ++k) cp_async<sizeof(W)>(xs + (tt * KT + k) * NT, k ? at_stride(xp, ksb, k) : xp, 0.f);
                xp += sXb;
            };
            if (FULL || (MULTI && n == LC)) TwinSteps<LC, true>::forward(n, step);
            else TwinSteps<LC, false>::forward(n, step);
        }
        cp_async_commit();
        fb = fb == NB - 1 ? 0 : fb + 1;
        if (++fc == nc) { fc = 0; ++fi; }
    };
#pragma unroll
    for (int b = 0; b < NB - 1; ++b) fetch();
    int buf = 0;
    for (int i = 0; i < nloop; ++i) {
        const bool live = LPN == 1 || i < pos.nrows;
        if (P.mask_mode == 2 && live)
            AR::neuron_masks(P, g, (j0 + i * jstep) % g.N, pos.chan, pos.sub, lp);
        float2 vd[KT];
#pragma unroll
        for (int k = 0; k < KT; ++k) vd[k] = f2(0.f);
        float2 v = f2(0.f);
        bool s1 = false, s2 = false;
        const int64_t j = j0 + i * jstep;
        for (int c = 0; c < nc; ++c) {
            cp_async_wait<NB - 2>();
            // the next chunk to fetch goes to the buffer read last
            fetch();
            const int t0 = c * LC;
            const int ncur = FULL ? LC : min(LC, T - t0);
            const W *const xs = xs0 + buf * (LC * KT * NT);
            buf = buf == NB - 1 ? 0 : buf + 1;
            auto steps = [&](auto full, auto soft, auto outv) {
                char *sp = static_cast<char *>(A.spikes) + (j + t0 * BN) * (int64_t)sizeof(XT);
                float *vp = decltype(outv)::value ? A.v_out + j + t0 * BN : nullptr;
                TwinSteps<LC, decltype(full)::value>::forward(ncur, [&](int tt) {
                    float2 xv[KT];
#pragma unroll
                    for (int k = 0; k < KT; ++k) xv[k] = IO::unpack(xs[(tt * KT + k) * NT]);
                    const float2 z = lanes_sum2<LPN>(AR::step(lp, vd, xv, residual, inv_k));
                    TwinSoma::charge<decltype(soft)::value>(P, z, v, s1, s2);
                    if (live && pos.sub == 0) {
                        __stcs(reinterpret_cast<W *>(sp), (s1 ? 0x3f80u : 0u) | (s2 ? 0x3f800000u : 0u));
                        if constexpr (decltype(outv)::value) __stcs(reinterpret_cast<float2 *>(vp), v);
                    }
                    sp += BN * (int64_t)sizeof(XT);
                    if constexpr (decltype(outv)::value) vp += BN;
                });
            };
            using yes = std::true_type;
            using no = std::false_type;
            auto pick = [&](auto full) {
                if (A.v_out) {
                    if (P.soft) steps(full, yes{}, yes{}); else steps(full, no{}, yes{});
                } else {
                    if (P.soft) steps(full, yes{}, no{}); else steps(full, no{}, no{});
                }
            };
            if constexpr (FULL) pick(yes{});
            else if constexpr (!MULTI) pick(no{});
            else if (ncur == LC) pick(yes{});
            else pick(no{});
            if (write_ck && live && c + 1 < nc) {
                const int64_t ck = (int64_t)c * BN + j;
                float va[KT], vb[KT];
#pragma unroll
                for (int k = 0; k < KT; ++k) { va[k] = vd[k].x; vb[k] = vd[k].y; }
                Vec<float, KT>::store(A.ck_vd + ck * K + pos.sub * KT, va);
                Vec<float, KT>::store(A.ck_vd + (ck + 1) * K + pos.sub * KT, vb);
                if (pos.sub == 0) __stcs(reinterpret_cast<float2 *>(A.ck_vs + ck), v);
            }
        }
    }
    pdl_trigger();
    cp_async_wait<0>();
}

}  // namespace dendsn

// FP32 correlated-basket path kernels (the multivariate Euler-Maruyama scheme
// of Sec. II.A.2), instantiated per basket width D in separate translation
// units so that they compile in parallel.
//
// basket_fp32_kernel steps the state: payoffs that look at the path, the Euler
// scheme, and materialised paths.  The contraction dW = Lhat z runs in packed
// FP32x2 FMAs (fma.rn.f32x2: two assets per instruction, each lane an ordinary
// FP32 fma) with the factor's column pairs in the launch-parameter block
// (constant bank) as 64-bit operands; the state is held as asset pairs.  A
// thread carries P paths, so that each factor pair that comes out of the
// constant bank serves P instructions: that port, not the FMA pipe, is what
// one path per thread waits for.  All warps of a block meet at a barrier after
// every sixteen columns, so that they read the same few kilobytes of the factor
// and of the code at a time; after every four, the barriers cost more than that
// gave (64 assets, 2^18 paths x 252 steps with a barrier payoff 8.17 ms, every
// eight 7.91, sixteen 7.84; 32 assets, 50,000 paths x 100 steps 298, 294 and
// 265 us).  A factor staged in shared memory instead was slower: each
// 16-byte shared load costs four cycles of the shared-memory port, a quarter
// of the rate the packed FMAs need.  Every thread runs every step (threads
// past the last path compute a path whose results are dropped), which keeps
// the barriers uniform.
//
// basket_sum_kernel prices payoffs on the terminal value under log-Euler from
// the path's summed normals (Segments, mc_device.cuh): one contraction per
// path.
#pragma once

#include "mc_kernels.cuh"

namespace gbmc {

// Kernel entry for width D and the given scheme, chosen by the flags of `a`
// (explicitly instantiated in k_basket_*.cu).
template <int D, int SCHEME>
const void *basket_select_scheme(const BasketArgs &a);

#ifdef GBMC_BASKET_IMPL
namespace basket_detail {

constexpr int kMaxWarps = kBasketMaxThreads / 32;

// Path of this thread in round `round`, from the special registers each time:
// held over the steps, the thread's index, its stride and the test against the
// last path cost registers that 64 assets of state do not leave (52 bytes of
// spills, so 32: 8.19 -> 8.07 ms at 2^18 paths x 252 steps with a barrier).
__device__ __forceinline__ int64_t path_of(int round, int64_t gthreads)
{
    uint32_t t, b;
    asm volatile("mov.u32 %0, %%tid.x;" : "=r"(t));
    asm volatile("mov.u32 %0, %%ctaid.x;" : "=r"(b));
    return static_cast<int64_t>(b) * blockDim.x + t + round * gthreads;
}

__device__ __forceinline__ float elem(const f32x2 *v, int j) { return (j & 1) ? hi_of(v[j >> 1]) : lo_of(v[j >> 1]); }

struct Stats {
    float sum, umax, umin;
    __device__ __forceinline__ void init() { sum = 0.0f; umax = -INFINITY; umin = INFINITY; }
    __device__ __forceinline__ void add(float u) { sum += u; umax = fmaxf(umax, u); umin = fminf(umin, u); }
};

__device__ __forceinline__ void accumulate_payoffs(AccSlot *s_acc, const PayoffSet &pay, bool valid,
                                                   float uT, float avg, const Stats &st)
{
    for (int p = 0; p < pay.n; ++p) {
        float f = payoff_eval(pay.kind[p], pay.strike[p], pay.barrier[p], uT, avg, st.umax, st.umin);
        warp_accumulate(s_acc, pay.n, p, valid ? f : 0.0f);
    }
}

// Pathwise Greeks of the European payoff (Sec. I.A.3) of one path from x_a =
// (Lhat W)_a: the price's term, delta_a = g w_a S_a / S0_a, vega_a = g w_a S_a
// (-sigma_a T + x_a / (log2(e) sigma_a)) and rho = g U T - T f, g the payoff's
// slope, into the warp's slots.  U adds four assets at a time and then those
// sums as a tree over 32 of them, the order of the d > 64 kernel's lanes, so
// that a basket has the same U there and here.
template <int D>
__device__ __forceinline__ void accumulate_basket_greeks(AccSlot *s_acc, const BasketArgs &a, const BasketConst<D> &c, bool valid,
                                                         const f32x2 (&x)[D / 2])
{
    const float fM = static_cast<float>(a.run.steps);
    float part[32];
#pragma unroll
    for (int g = 0; g < 32; ++g) {
        part[g] = 0.0f;
#pragma unroll
        for (int e = 0; e < 4; ++e) {
            const int j = 4 * g + e;
            if (j < D) part[g] = fmaf(c.ws0[j], ex2_approx(fmaf(fM, c.drift[j], elem(x, j))), part[g]);
        }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1)
#pragma unroll
        for (int g = 0; g < o; ++g) part[g] += part[g + o];
    const float U = part[0], K = a.pay.strike[0];
    const bool put = a.pay.kind[0] == MC_PUT;
    const float f = valid ? (put ? fmaxf(K - U, 0.0f) : fmaxf(U - K, 0.0f)) : 0.0f;
    const float g = valid ? (put ? (U < K ? -1.0f : 0.0f) : (U > K ? 1.0f : 0.0f)) : 0.0f;
    const int nv = 2 * a.d + 2;
    warp_accumulate(s_acc, nv, 0, f);
    warp_accumulate(s_acc, nv, nv - 1, g * U * a.T - a.T * f);
    // four assets at a time: deltas at 1 + a, vegas at 1 + d + a
#pragma unroll 1
    for (int j0 = 0; j0 < a.d; j0 += 4) {
        float dl[4], vg[4];
#pragma unroll
        for (int e = 0; e < 4; ++e) dl[e] = vg[e] = 0.0f;
#pragma unroll
        for (int jj = 0; jj < D; jj += 4) {
            if (jj != j0) continue;
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                const int j = jj + e;
                if (j < a.d) {
                    const float S = c.s0[j] * ex2_approx(fmaf(fM, c.drift[j], elem(x, j)));
                    dl[e] = g * c.w[j] * S / c.s0[j];
                    vg[e] = g * c.w[j] * S * fmaf(-a.sigma[j], a.T, elem(x, j) / (kLog2e * a.sigma[j]));
                }
            }
        }
        const float v[8] = {dl[0], dl[1], dl[2], dl[3], vg[0], vg[1], vg[2], vg[3]};
        warp_accumulate8_at(s_acc, nv, v, [&](int k) {
            const int j = j0 + (k & 3);
            return j < a.d ? (k < 4 ? 1 + j : 1 + a.d + j) : -1;
        });
    }
}

// ------------------------------ FP32 basket -------------------------------
template <int D, int SCHEME, bool STATS, bool SAVE, int READ, int P, bool GREEKS>
__global__ void __launch_bounds__(P == 1 ? 32 * kMaxWarps : basket_threads2(D), 1)
    basket_fp32_kernel(const __grid_constant__ BasketArgs a, const BasketConst<D> c)
{
    static_assert(!SAVE || (READ == kReadAny && P == 1), "materialised paths: one per thread");
    static_assert(!GREEKS || (SCHEME == MC_LOG_EULER && !STATS && !SAVE), "Greeks: European payoffs under log-Euler");
    extern __shared__ AccSlot s_greeks[];  // GREEKS: the warps' slots of price, deltas, vegas, rho
    __shared__ AccSlot s_pays[GREEKS ? 1 : kMaxWarps * MC_MAX_PAYOFFS * 2];
    __shared__ double s_red[32];
    AccSlot *const s_acc = GREEKS ? s_greeks : s_pays;
    const int nvals = GREEKS ? 2 * a.d + 2 : a.pay.n;
    for (int i = threadIdx.x; i < static_cast<int>(blockDim.x >> 5) * nvals * 2; i += blockDim.x) s_acc[i] = 0.0f;
    __syncthreads();

    constexpr int H = D / 2;
    const int64_t gthreads = static_cast<int64_t>(gridDim.x) * blockDim.x;
    const int M = a.run.steps, d = a.d;
    const float inv_m = 1.0f / static_cast<float>(M);
    for (int it = 0; it < a.run.ppt; it += P) {
        bool valid[P];
        float uT[P], avg[P];
        Stats st[P];
        uint64_t n[P];
        int64_t nl = 0;
#pragma unroll
        for (int p = 0; p < P; ++p) {
            nl = path_of(it + p, gthreads);
            valid[p] = it + p < a.run.ppt && nl < a.run.paths;
            n[p] = static_cast<uint64_t>(a.run.path_offset + nl);
            uT[p] = avg[p] = 0.0f;
            st[p].init();
        }
        if (!SAVE || valid[0]) {  // every thread steps (block barriers below) unless it writes paths
            f32x2 x[P][H];  // asset pairs; log-Euler: log2(S_a / S0_a); Euler: S_a
#pragma unroll
            for (int p = 0; p < P; ++p)
#pragma unroll
                for (int q = 0; q < H; ++q)
                    x[p][q] = (SCHEME == MC_LOG_EULER) ? pack2(0.0f, 0.0f) : pack2(c.s0[2 * q], c.s0[2 * q + 1]);
            const int64_t save_len = (static_cast<int64_t>(M / a.run.save_every) + 1) * d * a.run.paths;
            if (SAVE) {
                for (int j = 0; j < d; ++j)
                    if (GBMC_IN_BOUNDS(static_cast<int64_t>(j) * a.run.paths + nl, save_len, kDbgBasketSave))
                        a.run.save[static_cast<int64_t>(j) * a.run.paths + nl] = c.s0[j];
            }
            NormalReader rd;             // kReadAny
            PathStream ps[P];            // kReadAligned
            ShiftedReader sr[P];         // kReadShifted
            float4 znext[P];
            uint32_t blk = 1;            // kReadShifted: the last block held
            int o = 0;                   // kReadShifted: the step's first lane
            const int rest = d - 4 * ((d - 1) / 4);  // normals of a step's last group of four
            if (READ == kReadAny) rd.init(n[0], a.run.rk);
#pragma unroll
            for (int p = 0; p < P; ++p) {
                if (READ == kReadAligned) ps[p].init(n[p], a.run.rk);
                if (READ == kReadShifted) sr[p].init(n[p], a.run.rk);
            }
            for (int i = 0; i < M; ++i) {
                // log-Euler accumulates L z straight into the state (|y| = O(1):
                // ~65 roundings of <= 3e-8 per step, ~2e-6 rms over 252 steps);
                // Euler needs dW apart because the step is multiplicative.
                f32x2 dw[P][SCHEME == MC_EULER ? H : 1];
#pragma unroll
                for (int p = 0; p < P; ++p) {
#pragma unroll
                    for (int q = 0; q < H; ++q) {
                        if (SCHEME == MC_EULER) dw[p][q] = pack2(0.0f, 0.0f);
                        else if (!GREEKS) x[p][q] = fadd2(x[p][q], pack2(c.drift[2 * q], c.drift[2 * q + 1]));
                    }
                    if (READ == kReadAligned) znext[p] = ps[p].normals(static_cast<uint32_t>(i) * (D / 4), a.run.rk).f4();
                }
                // dW = Lhat z, column by column as the normals are produced;
                // column k updates the pairs q >= k/2 with (z_k, z_k).  The
                // next block of four normals is drawn before this block's
                // products (independent work while the SFU results arrive).
#pragma unroll
                for (int kb = 0; kb < (D + 3) / 4; ++kb) {
                    if (READ == kReadShifted && 4 * kb >= d) continue;  // padded columns: nothing to draw or add
                    f32x2 z2[P][4];
#pragma unroll
                    for (int p = 0; p < P; ++p) {
                        float4 z;
                        if (READ == kReadAligned) {
                            z = znext[p];
                            if (kb + 1 < D / 4)
                                znext[p] = ps[p].normals(static_cast<uint32_t>(i) * (D / 4) + kb + 1, a.run.rk).f4();
                        } else if (READ == kReadShifted) {
                            z = sr[p].group(o);
                        } else {
                            float zz[4];
#pragma unroll
                            for (int l = 0; l < 4; ++l)
                                zz[l] = (4 * kb + l < D && 4 * kb + l < d) ? rd.get(static_cast<uint64_t>(i) * d + 4 * kb + l) : 0.0f;
                            z = make_float4(zz[0], zz[1], zz[2], zz[3]);
                        }
                        z2[p][0] = pack2(z.x, z.x);
                        z2[p][1] = pack2(z.y, z.y);
                        z2[p][2] = pack2(z.z, z.z);
                        z2[p][3] = pack2(z.w, z.w);
                    }
                    if (READ == kReadShifted && (4 * kb + 4 < d || o + rest >= 4)) {
                        ++blk;
#pragma unroll
                        for (int p = 0; p < P; ++p) sr[p].advance(blk, a.run.rk);
                    }
#pragma unroll
                    for (int l = 0; l < 4; ++l) {
                        const int k = 4 * kb + l;
                        if (k < D) {
#pragma unroll
                            for (int q = k / 2; q < H; ++q) {
                                const f32x2 Lq = c.Lp[basket_pair_base(D, k) + q - k / 2];
#pragma unroll
                                for (int p = 0; p < P; ++p) {
                                    if (SCHEME == MC_EULER) dw[p][q] = ffma2(Lq, z2[p][l], dw[p][q]);
                                    else x[p][q] = ffma2(Lq, z2[p][l], x[p][q]);
                                }
                            }
                        }
                    }
                    if (!SAVE && (kb & 3) == 3) __syncthreads();
                }
                if (READ == kReadShifted) o = (o + d) & 3;
#pragma unroll
                for (int p = 0; p < P; ++p) {
                    if (SCHEME == MC_EULER) {
#pragma unroll
                        for (int q = 0; q < H; ++q)
                            x[p][q] = ffma2(x[p][q], fadd2(pack2(c.drift[2 * q], c.drift[2 * q + 1]), dw[p][q]), x[p][q]);
                    }
                    if (STATS && !SAVE && SCHEME == MC_LOG_EULER) {
                        // monitored basket: sum of (w_a S0_a) 2^{x_a}, asset pairs
                        static_assert(D % 2 == 0 && (sizeof(unsigned long long) * basket_pair_count(D) + sizeof(float) * D) % 8 == 0,
                                      "ws0 is read as 8-byte pairs");
                        f32x2 u2 = pack2(0.0f, 0.0f);
#pragma unroll
                        for (int q = 0; q < H; ++q)
                            u2 = ffma2(reinterpret_cast<const f32x2 *>(c.ws0)[q],
                                       pack2(ex2_approx(lo_of(x[p][q])), ex2_approx(hi_of(x[p][q]))), u2);
                        st[p].add(lo_of(u2) + hi_of(u2));
                    } else if (STATS || (SAVE && ((i + 1) % a.run.save_every) == 0)) {
                        float u = 0.0f;
                        const int64_t slot = (i + 1) / a.run.save_every;
#pragma unroll
                        for (int j = 0; j < D; ++j) {
                            const float xj = elem(x[p], j);
                            const float Sj = (SCHEME == MC_LOG_EULER) ? c.s0[j] * ex2_approx(xj) : xj;
                            if (STATS) u = fmaf(c.w[j], Sj, u);
                            if (SAVE && ((i + 1) % a.run.save_every) == 0 && j < d &&
                                GBMC_IN_BOUNDS((slot * d + j) * a.run.paths + nl, save_len, kDbgBasketSave))
                                a.run.save[(slot * d + j) * a.run.paths + nl] = Sj;
                        }
                        if (STATS) st[p].add(u);
                    }
                }
            }
#pragma unroll
            for (int p = 0; p < P; ++p) {
                if (GREEKS) {
                    if (it + p < a.run.ppt) accumulate_basket_greeks<D>(s_acc, a, c, valid[p], x[p]);
                    continue;
                }
                float u = 0.0f;
#pragma unroll
                for (int j = 0; j < D; ++j) {
                    if (SCHEME == MC_LOG_EULER) u = fmaf(c.ws0[j], ex2_approx(elem(x[p], j)), u);
                    else u = fmaf(c.w[j], elem(x[p], j), u);
                }
                uT[p] = u;
                avg[p] = st[p].sum * inv_m;
            }
        }
        if (!GREEKS && a.pay.n > 0) {
#pragma unroll
            for (int p = 0; p < P; ++p)
                if (it + p < a.run.ppt) accumulate_payoffs(s_acc, a.pay, path_of(it + p, gthreads) < a.run.paths, uT[p], avg[p], st[p]);
        }
    }
    if (nvals > 0) block_finish(s_acc, s_red, nvals, a.red);
}

// European payoffs under log-Euler: each thread sums its path's normals into
// its column of shared memory, four Philox blocks at a time, then contracts
// once.  Bound by drawing: the contraction of every step took two thirds of
// 8.0 ms at 2^18 paths x 252 steps of 64 assets.
template <int D>
__global__ void __launch_bounds__(kBasketSumBlock, 5) basket_sum_kernel(const __grid_constant__ BasketArgs a, const BasketConst<D> c)
{
    __shared__ float s_w[D][kBasketSumBlock];
    __shared__ AccSlot s_acc[(kBasketSumBlock / 32) * MC_MAX_PAYOFFS * 2];
    __shared__ double s_red[32];
    const int t = threadIdx.x, d = a.d, M = a.run.steps;
    for (int i = t; i < (kBasketSumBlock / 32) * a.pay.n * 2; i += blockDim.x) s_acc[i] = 0.0f;
    for (int k = 0; k < D; ++k) s_w[k][t] = 0.0f;
    __syncthreads();
    const int64_t gthreads = static_cast<int64_t>(gridDim.x) * blockDim.x;
    const int64_t tid = static_cast<int64_t>(blockIdx.x) * blockDim.x + t;
    const Segments seg(M, d);
    for (int it = 0; it < a.run.ppt; ++it) {
        const int64_t nl = tid + it * gthreads;
        const bool valid = nl < a.run.paths;
        const uint64_t n = static_cast<uint64_t>(a.run.path_offset + nl);
        for (uint32_t p = 0; p < seg.period && seg.count(p) > 0; ++p) {
            const int o = seg.lane(p), nblk = (o + d + 3) >> 2;
            for (int g = 0; g < nblk; g += 4)
                up_to_four(nblk - g, [&](auto nb) {
                    constexpr int NB = decltype(nb)::value;
                    f32x2 w[2 * NB];
                    sum_blocks<NB>(w, n, a.run.rk, a.wide, seg.first_block(p) + g, 1, seg.count(p), seg.blocks);
#pragma unroll
                    for (int e = 0; e < 4 * NB; ++e) {
                        const int k = 4 * g + e - o;
                        if (k >= 0 && k < d)
                            s_w[k][t] = (p == 0 ? 0.0f : s_w[k][t]) + ((e & 1) ? hi_of(w[e >> 1]) : lo_of(w[e >> 1]));
                    }
                });
        }
        f32x2 x[D / 2];
#pragma unroll
        for (int q = 0; q < D / 2; ++q)
            x[q] = pack2(static_cast<float>(M) * c.drift[2 * q], static_cast<float>(M) * c.drift[2 * q + 1]);
#pragma unroll
        for (int k = 0; k < D; ++k) {
            const f32x2 z2 = pack2(s_w[k][t], s_w[k][t]);
#pragma unroll
            for (int q = k / 2; q < D / 2; ++q) x[q] = ffma2(c.Lp[basket_pair_base(D, k) + q - k / 2], z2, x[q]);
        }
        float u = 0.0f;
#pragma unroll
        for (int j = 0; j < D; ++j) u = fmaf(c.ws0[j], ex2_approx(elem(x, j)), u);
        Stats st;
        st.init();
        accumulate_payoffs(s_acc, a.pay, valid, u, 0.0f, st);
    }
    block_finish(s_acc, s_red, a.pay.n, a.red);
}

template <int D, int SCHEME, bool STATS, bool SAVE, int READ, int P, bool GREEKS = false>
const void *basket_fn()
{
    return reinterpret_cast<const void *>(&basket_fp32_kernel<D, SCHEME, STATS, SAVE, READ, P, GREEKS>);
}

template <int D, int SCHEME, bool STATS, bool GREEKS = false>
const void *basket_pick(const BasketArgs &a)
{
    if constexpr (D == 64 && !GREEKS) {  // runs of more than 2^32 Philox blocks per path take this width (basket_fp32_width)
        if (a.wide) return basket_fn<D, SCHEME, STATS, false, kReadAny, 1>();
    }
    if constexpr (basket_threads2(D) == 0)
        return a.d == D ? basket_fn<D, SCHEME, STATS, false, kReadAligned, 1, GREEKS>()
                        : basket_fn<D, SCHEME, STATS, false, kReadShifted, 1, GREEKS>();
    else if (a.d == D)
        return a.two ? basket_fn<D, SCHEME, STATS, false, kReadAligned, 2, GREEKS>()
                     : basket_fn<D, SCHEME, STATS, false, kReadAligned, 1, GREEKS>();
    else
        return a.two ? basket_fn<D, SCHEME, STATS, false, kReadShifted, 2, GREEKS>()
                     : basket_fn<D, SCHEME, STATS, false, kReadShifted, 1, GREEKS>();
}

template <int D, int SCHEME>
const void *basket_select_impl(const BasketArgs &a)
{
    if (a.run.save) return basket_fn<D, SCHEME, false, true, kReadAny, 1>();
    if constexpr (SCHEME == MC_LOG_EULER) {
        if (a.greeks) return basket_pick<D, SCHEME, false, true>(a);
    }
    if (a.pay.need_avg || a.pay.need_max || a.pay.need_min) return basket_pick<D, SCHEME, true>(a);
    if constexpr (SCHEME == MC_LOG_EULER) return reinterpret_cast<const void *>(&basket_sum_kernel<D>);
    else return basket_pick<D, SCHEME, false>(a);
}

}  // namespace basket_detail

template <int D, int SCHEME>
const void *basket_select_scheme(const BasketArgs &a)
{
    return basket_detail::basket_select_impl<D, SCHEME>(a);
}

#define GBMC_INSTANTIATE_BASKET(D, SCHEME) \
    template const void *basket_select_scheme<D, SCHEME>(const BasketArgs &a);
#endif  // GBMC_BASKET_IMPL

}  // namespace gbmc

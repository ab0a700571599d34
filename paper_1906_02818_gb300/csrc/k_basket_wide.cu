// FP32 large baskets (64 < d <= 512): European payoffs under log-Euler, the
// multivariate Euler step of Sec. II.A.2, and their pathwise Greeks (of any d).
//   * CTA = 64 paths x D assets (D = 128, 256 or 512, zero-padded), 512
//     threads.  Contraction: thread (pg, ag) owns paths 4 pg .. 4 pg + 3 and
//     the assets 128 j + 4 ag .. + 3 (j < D / 128): 4 x D / 32 sums in
//     registers as asset pairs (packed FP32x2 FMAs, one instruction for two
//     assets of one path, each lane an FP32 fma), Lhat = log2(e) sqrt(dt)
//     diag(sigma) Lrho streamed k-major in chunks of 16 rows (cp.async double
//     buffer); 128-asset blocks above the chunk (zero in the lower-triangular
//     factor) are skipped.
//   * Prices: the terminal log-prices need the contraction of the summed
//     normals only (Segments, mc_device.cuh).  Thread (path t mod 64, t / 64)
//     sums every eighth Philox block of its path over the steps, up to four
//     blocks at a time in registers, into W[k][path] in shared memory; one
//     contraction per tile.  Bound by drawing; the contraction of every step
//     took 141 ms for 2^16 paths x 252 steps at d = 512, this 6.8 ms.
//   * Greeks: contracted every step.  The payoff's slope is an indicator of
//     U > K, and one path that falls on the other side of K by a rounding
//     moves the vegas, sums of large terms of both signs, by 1e-4; so the
//     Greeks keep the sums they have always been formed from.
//   * Epilogue: log2(S_a / S0_a) = M drift_a + (Lhat W)_a, the basket,
//     European payoffs and the pathwise delta / vega / rho of payoff 0.  The
//     sums of a run with Greeks have a fixed order, so its results have the
//     same bits each time.  (Prices add the sums of a tile's two payoff warps
//     as they come; in a fixed order the price kernel took 4 % longer.)
#include "mc_kernels.cuh"

namespace gbmc {
namespace {

constexpr int kP = 64;       // paths per CTA
constexpr int kThreads = 512;
constexpr int kKC = 16;      // factor rows per chunk

__device__ __forceinline__ void cp_async16(void *smem, const void *gmem)
{
    const uint32_t s = static_cast<uint32_t>(__cvta_generic_to_shared(smem));
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(s), "l"(gmem) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
__device__ __forceinline__ void cp_async_wait_all() { asm volatile("cp.async.wait_group 0;" ::: "memory"); }

// Element e (0..3) of a thread's four consecutive assets held as two pairs.
__device__ __forceinline__ float accel(const f32x2 *pr, int e) { return (e & 1) ? hi_of(pr[e >> 1]) : lo_of(pr[e >> 1]); }

template <int D, bool GREEKS>
__global__ void __launch_bounds__(kThreads, 1) basket_wide_kernel(const __grid_constant__ BigArgs a)
{
    constexpr int J = D / 128;  // 4-asset groups per thread
    extern __shared__ __align__(16) float sm[];
    float *zs = sm;                      // [D][kP]
    float *Ls = sm + D * kP;             // [2][kKC][D]
    __shared__ float s_pay[MC_MAX_PAYOFFS][2];
    __shared__ float s_g[kBigMaxD * 2 + 1][2];
    __shared__ float s_u[kP];
    __shared__ float s_w[2][MC_MAX_PAYOFFS + 1][2];  // sums of the two warps that hold a tile's payoffs; last: rho
    const int t = threadIdx.x, lane = t & 31;
    const int pg = t >> 5, ag = t & 31;  // a warp = one path group, 32 asset groups
    const int d = a.d, nv = a.pay.n, M = a.run.steps;
    for (int i = t; i < nv * 2; i += kThreads) s_pay[i >> 1][i & 1] = 0.0f;
    if (GREEKS)
        for (int i = t; i < (2 * d + 1) * 2; i += kThreads) s_g[i >> 1][i & 1] = 0.0f;
    const int64_t ntiles = (a.run.paths + kP - 1) / kP;
    const int nchunks = (d + kKC - 1) / kKC;
    const Segments seg(M, d);
    // rows past d of the last chunk meet zero rows of the factor: finite, and written once
    for (int i = d * kP + t; i < nchunks * kKC * kP; i += kThreads) zs[i] = 0.0f;

    for (int64_t tile = blockIdx.x; tile < ntiles; tile += gridDim.x) {
        // drawing: path t % 64, blocks t / 64, t / 64 + 8, ... of each segment
        const int rp = t & (kP - 1);
        const uint32_t rq = static_cast<uint32_t>(t) >> 6;
        const int64_t rnl = tile * kP + rp;
        const uint64_t rn = static_cast<uint64_t>(a.run.path_offset + (rnl < a.run.paths ? rnl : 0));
        f32x2 acc2[4][J][2];  // [path][asset group][asset pair]
#pragma unroll
        for (int p = 0; p < 4; ++p)
#pragma unroll
            for (int j = 0; j < J; ++j)
#pragma unroll
                for (int e = 0; e < 2; ++e) acc2[p][j][e] = pack2(0.0f, 0.0f);
        // acc2 += Lhat zs over the factor's chunks
        auto contract = [&]() {
            // first factor chunk
            for (int e = t * 4; e < kKC * D; e += kThreads * 4) cp_async16(Ls + e, a.Lp + e);
            cp_async_commit();
            for (int c = 0; c < nchunks; ++c) {
                cp_async_wait_all();
                __syncthreads();  // chunk c (and, at c = 0, the summed normals) visible
                const float *Lc = Ls + (c & 1) * kKC * D;
                if (c + 1 < nchunks) {  // prefetch the next chunk into the other buffer
                    float *dst = Ls + ((c + 1) & 1) * kKC * D;
                    const float *src = a.Lp + static_cast<size_t>(c + 1) * kKC * D;
                    for (int e = t * 4; e < kKC * D; e += kThreads * 4) cp_async16(dst + e, src + e);
                    cp_async_commit();
                }
                const int k0 = c * kKC;
    #pragma unroll 4
                for (int kk = 0; kk < kKC; ++kk) {
                    const float4 zv = *reinterpret_cast<const float4 *>(zs + (k0 + kk) * kP + 4 * pg);
                    const f32x2 zz[4] = {pack2(zv.x, zv.x), pack2(zv.y, zv.y), pack2(zv.z, zv.z), pack2(zv.w, zv.w)};
    #pragma unroll
                    for (int j = 0; j < J; ++j) {
                        if (128 * j + 127 < k0) continue;  // block above the diagonal chunk: zero
                        const ulonglong2 lv = *reinterpret_cast<const ulonglong2 *>(Lc + kk * D + 128 * j + 4 * ag);
    #pragma unroll
                        for (int p = 0; p < 4; ++p) {
                            acc2[p][j][0] = ffma2(lv.x, zz[p], acc2[p][j][0]);
                            acc2[p][j][1] = ffma2(lv.y, zz[p], acc2[p][j][1]);
                        }
                    }
                }
                __syncthreads();  // everyone done with chunk c before it is overwritten
            }
        };
        if (GREEKS) {
            // thread (path t mod 64, t / 64) draws an eighth of the columns: whole blocks when 4 | d, else the lanes
            // that the step's place in its first block picks from two blocks in registers
            PathStream ps;
            ps.init(rn, a.run.rk);
            const int k0 = static_cast<int>(rq) * (D / 8), k1 = min(k0 + D / 8, d);
            auto put = [&](int k, const float4 &z) {
                zs[(k + 0) * kP + rp] = z.x;
                zs[(k + 1) * kP + rp] = z.y;
                zs[(k + 2) * kP + rp] = z.z;
                zs[(k + 3) * kP + rp] = z.w;
            };
            for (int i = 0; i < M; ++i) {
                __syncthreads();  // previous step done with zs
                const uint64_t j0 = static_cast<uint64_t>(i) * d + k0;
                if (a.wide) {
                    NormalReader rd;
                    rd.init(rn, a.run.rk);
                    for (int k = k0; k < k1; ++k) zs[k * kP + rp] = rd.get(j0 + k - k0);
                } else if (a.exact4) {
                    const uint32_t q = static_cast<uint32_t>(j0 >> 2) - (k0 >> 2);
                    for (int k = k0; k < k1; k += 4) put(k, ps.normals(q + (k >> 2), a.run.rk).f4());
                } else if (k0 < k1) {
                    uint32_t q = static_cast<uint32_t>(j0 >> 2);
                    const int o = static_cast<int>(j0 & 3);
                    float4 cur = ps.normals(q, a.run.rk).f4();
                    for (int k = k0; k < k1; k += 4) {
                        const float4 nxt = ps.normals(++q, a.run.rk).f4();
                        float4 z = shifted4(cur, nxt, o);
                        if (k + 1 >= d) z.y = 0.0f;
                        if (k + 2 >= d) z.z = 0.0f;
                        if (k + 3 >= d) z.w = 0.0f;
                        put(k, z);
                        cur = nxt;
                    }
                }
                contract();
            }
        } else {
            for (uint32_t p = 0; p < seg.period && seg.count(p) > 0; ++p) {
                const int o = seg.lane(p);
                const uint32_t nblk = static_cast<uint32_t>(o + d + 3) >> 2;
                for (uint32_t g = rq; g < nblk; g += 32)
                    up_to_four(static_cast<int>((nblk - g + 7) / 8), [&](auto nb) {
                        constexpr int NB = decltype(nb)::value;
                        f32x2 w[2 * NB];
                        sum_blocks<NB>(w, rn, a.run.rk, a.wide, seg.first_block(p) + g, 8, seg.count(p), seg.blocks);
    #pragma unroll
                        for (int e = 0; e < 4 * NB; ++e) {
                            const int k = static_cast<int>(4 * (g + 8 * (e >> 2))) + (e & 3) - o;
                            if (k >= 0 && k < d) {
                                const float v = (e & 1) ? hi_of(w[e >> 1]) : lo_of(w[e >> 1]);
                                zs[k * kP + rp] = p == 0 ? v : zs[k * kP + rp] + v;
                            }
                        }
                    });
                if (p + 1 < seg.period) __syncthreads();  // a column's sums of two segments lie with different threads
            }
            contract();
        }
        // ---- epilogue ----
        float Ux[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
        for (int j = 0; j < J; ++j)
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                const int col = 128 * j + 4 * ag + e;
                if (col < d) {
#pragma unroll
                    for (int p = 0; p < 4; ++p)
                        Ux[p] = fmaf(a.ws0[col], ex2_approx(fmaf(static_cast<float>(M), a.drift[col], accel(acc2[p][j], e))), Ux[p]);
                }
            }
        // sum over the 32 asset groups of each path (the lanes of one warp)
#pragma unroll
        for (int p = 0; p < 4; ++p) Ux[p] = warp_sum(Ux[p]);
        if (ag == 0)
#pragma unroll
            for (int p = 0; p < 4; ++p) s_u[4 * pg + p] = Ux[p];
        __syncthreads();
        if (t < kP) {  // payoffs, one thread per path
            const bool valid = tile * kP + t < a.run.paths;
            for (int q = 0; q < nv; ++q) {
                const float f = valid ? payoff_eval(a.pay.kind[q], a.pay.strike[q], INFINITY, s_u[t], 0.f, 0.f, 0.f) : 0.f;
                const float s1 = warp_sum(f), s2 = warp_sum(f * f);
                if (lane == 0) {
                    if (GREEKS) {
                        s_w[pg][q][0] = s1;
                        s_w[pg][q][1] = s2;
                    } else {
                        atomicAdd(&s_pay[q][0], s1);
                        atomicAdd(&s_pay[q][1], s2);
                    }
                }
            }
        }
        if (GREEKS) {
            float gs[4];
#pragma unroll
            for (int p = 0; p < 4; ++p) {
                const float U = s_u[4 * pg + p];
                const bool valid = tile * kP + 4 * pg + p < a.run.paths;
                gs[p] = valid ? (a.pay.kind[0] == MC_PUT ? (U < a.pay.strike[0] ? -1.f : 0.f)
                                                         : (U > a.pay.strike[0] ? 1.f : 0.f))
                              : 0.f;
            }
            // the warps' sums of delta, delta^2, vega, vega^2 per column, [4][16 warps][D], over the normals (read no
            // more); then added in the warps' order
            float *red = zs;
#pragma unroll
            for (int j = 0; j < J; ++j) {
                float4 sums[4];
#pragma unroll
                for (int e = 0; e < 4; ++e) {
                    const int col = 128 * j + 4 * ag + e;
                    float d1 = 0.f, d2 = 0.f, v1 = 0.f, v2 = 0.f;
                    if (col < d) {
#pragma unroll
                        for (int p = 0; p < 4; ++p) {
                            const float S = a.s0[col] * ex2_approx(fmaf(static_cast<float>(M), a.drift[col], accel(acc2[p][j], e)));
                            const float dl = gs[p] * a.w[col] * S / a.s0[col];
                            // sqrt(dt) (Lrho W)_col = acc / (log2(e) sigma_col)
                            const float vg = gs[p] * a.w[col] * S * fmaf(-a.sigma[col], a.T, accel(acc2[p][j], e) / (kLog2e * a.sigma[col]));
                            d1 += dl; d2 += dl * dl; v1 += vg; v2 += vg * vg;
                        }
                    }
                    reinterpret_cast<float *>(&sums[0])[e] = d1;
                    reinterpret_cast<float *>(&sums[1])[e] = d2;
                    reinterpret_cast<float *>(&sums[2])[e] = v1;
                    reinterpret_cast<float *>(&sums[3])[e] = v2;
                }
#pragma unroll
                for (int v = 0; v < 4; ++v) *reinterpret_cast<float4 *>(red + (v * 16 + pg) * D + 128 * j + 4 * ag) = sums[v];
            }
            if (t < kP) {
                const float U = s_u[t];
                const bool valid = tile * kP + t < a.run.paths;
                const float g = valid ? (a.pay.kind[0] == MC_PUT ? (U < a.pay.strike[0] ? -1.f : 0.f)
                                                                 : (U > a.pay.strike[0] ? 1.f : 0.f))
                                      : 0.f;
                const float f = valid ? payoff_eval(a.pay.kind[0], a.pay.strike[0], INFINITY, U, 0.f, 0.f, 0.f) : 0.f;
                const float rr = g * U * a.T - a.T * f;
                const float r1 = warp_sum(rr), r2 = warp_sum(rr * rr);
                if (lane == 0) {
                    s_w[pg][nv][0] = r1;
                    s_w[pg][nv][1] = r2;
                }
            }
        }
        __syncthreads();
        if (GREEKS) {
            if (t < 2 * nv) s_pay[t >> 1][t & 1] += s_w[0][t >> 1][t & 1] + s_w[1][t >> 1][t & 1];
            if (t < 2) s_g[2 * d][t] += s_w[0][nv][t] + s_w[1][nv][t];
            for (int i = t; i < 4 * d; i += kThreads) {
                const int v = i / d, col = i - v * d;
                float sum = 0.0f;
#pragma unroll
                for (int w = 0; w < kThreads / 32; ++w) sum += zs[(v * 16 + w) * D + col];
                s_g[(v >> 1) * d + col][v & 1] += sum;
            }
            __syncthreads();
            for (int i = d * kP + t; i < nchunks * kKC * kP; i += kThreads) zs[i] = 0.0f;
        }
    }
    if (GREEKS) __syncthreads();
    // per-CTA partials -> FP64 sum by the last CTA
    const int nvals = nv + (GREEKS ? 2 * d + 1 : 0);
    for (int i = t; i < nvals * 2; i += kThreads) {
        const int k = i >> 1, m = i & 1;
        a.partials[static_cast<size_t>(blockIdx.x) * nvals * 2 + i] = k < nv ? s_pay[k][m] : s_g[k - nv][m];
    }
    __threadfence();
    __syncthreads();
    __shared__ unsigned int s_last;
    if (t == 0) s_last = (atomicAdd(a.ticket, 1u) == gridDim.x - 1) ? 1u : 0u;
    __syncthreads();
    if (!s_last) return;
    __threadfence();
    const double N = static_cast<double>(a.run.paths);
    for (int k = t; k < nvals; k += kThreads) {
        double s1 = 0.0, s2 = 0.0;
        for (int b = 0; b < static_cast<int>(gridDim.x); ++b) {
            s1 += a.partials[static_cast<size_t>(b) * nvals * 2 + 2 * k];
            s2 += a.partials[static_cast<size_t>(b) * nvals * 2 + 2 * k + 1];
        }
        const double mean = s1 / N, var = fmax(s2 / N - mean * mean, 0.0);
        mc_result r;
        r.price = a.disc * mean;
        r.se = a.run.paths > 1 ? a.disc * sqrt(var / (N - 1.0)) : 0.0;
        a.out[k] = r;
    }
    __syncthreads();
    if (t == 0) *a.ticket = 0u;
}

// LT[k][a] (D x D, k-major) = log2(e) sqrt(dt) sigma_a Lrho[a][k] (0 above the
// diagonal and beyond d); drift[a] = log2(e) (r - sigma_a^2 / 2) dt.
__global__ void wide_prep_kernel(int d, int D, const double *L, const double *sigma, double sdt, double r, double dt,
                                 float *LT, float *drift)
{
    for (int64_t idx = blockIdx.x * static_cast<int64_t>(blockDim.x) + threadIdx.x; idx < static_cast<int64_t>(D) * D;
         idx += static_cast<int64_t>(gridDim.x) * blockDim.x) {
        const int k = static_cast<int>(idx / D), col = static_cast<int>(idx % D);
        double v = 0.0;
        if (col < d && k <= col) v = M_LOG2E * sdt * sigma[col] * L[static_cast<int64_t>(col) * d + k];
        LT[idx] = static_cast<float>(v);
    }
    for (int col = blockIdx.x * blockDim.x + threadIdx.x; col < d; col += gridDim.x * blockDim.x)
        drift[col] = static_cast<float>(M_LOG2E * (r - 0.5 * sigma[col] * sigma[col]) * dt);
}

}  // namespace

int wide_width(int d) { return d <= 128 ? 128 : (d <= 256 ? 256 : 512); }

size_t wide_smem(int D) { return static_cast<size_t>(D) * kP * sizeof(float) + 2 * kKC * static_cast<size_t>(D) * sizeof(float); }

template <bool GREEKS>
static const void *wide_fn(int D)
{
    switch (D) {
    case 128: return reinterpret_cast<const void *>(&basket_wide_kernel<128, GREEKS>);
    case 256: return reinterpret_cast<const void *>(&basket_wide_kernel<256, GREEKS>);
    default: return reinterpret_cast<const void *>(&basket_wide_kernel<512, GREEKS>);
    }
}

const void *basket_wide_fn(int D, bool greeks) { return greeks ? wide_fn<true>(D) : wide_fn<false>(D); }

int basket_wide_block() { return kThreads; }

cudaError_t launch_wide_prep(int d, const double *L, const double *sigma, double sdt, double r, double dt, float *LT,
                             float *drift, cudaStream_t s)
{
    const int D = wide_width(d);
    wide_prep_kernel<<<256, 256, 0, s>>>(d, D, L, sigma, sdt, r, dt, LT, drift);
    return cudaGetLastError();
}

}  // namespace gbmc

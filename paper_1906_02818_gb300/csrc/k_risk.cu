// Portfolio risk (Sec. VI.B: VaR and CVaR of a portfolio of options on
// correlated underlyings) and the Monte Carlo labels of its pricing
// surrogate.  Kernels:
//   label_kernel     one parameter point (S/K, sigma, tau, r, K/H) per CTA:
//                    Monte Carlo price / K of a call, up-and-out when K/H > 0
//                    (daily monitoring), the training labels of the network;
//   outer_kernel     one risk scenario per thread: correlated one-period GBM
//                    move of every underlying over the horizon h;
//   nested_kernel    one (scenario, underlying) and slice of its inner paths
//                    per CTA: inner Monte Carlo revaluation of that
//                    underlying's options at the scenario state (the
//                    yardstick of the surrogate, and its fallback);
//   features_kernel  network inputs of every (scenario, option) pair;
//   pnl_kernel       one scenario per CTA: portfolio PnL from the revalued
//                    options (FP64 sum over options);
//   tail_*_kernel    VaR by radix selection of the losses, CVaR.
// Random streams: the stream index carries a domain tag in its top byte
// (2 outer scenarios, 3 inner paths, 4 labels, 5 base values) so that the
// domains never share normals.
#include <algorithm>
#include <cmath>

#include "mc_kernels.cuh"
#include "risk.cuh"

namespace gbmc {
namespace {

__device__ __forceinline__ uint64_t tag(uint64_t domain, uint64_t idx) { return (domain << 56) | idx; }

// Network inputs from the raw point (S/K, sigma, tau, r, K/H): each mapped
// from its parameter-box range to about [-1, 1] (the constants of mc.h).
__device__ __forceinline__ void surrogate_inputs(float sk, float sig, float tau, float r, float kh, float *f)
{
    f[0] = (sk - 1.05f) * (1.0f / 0.55f);
    f[1] = (sig - 0.25f) * (1.0f / 0.15f);
    f[2] = tau - 1.0f;
    f[3] = (r - 0.04f) * (1.0f / 0.04f);
    f[4] = (kh - 0.45f) * (1.0f / 0.45f);
}

// ------------------------------ labels -----------------------------------
// GREEKS: also the pathwise sensitivities of each European point's label
// (Sec. I.A.3), per path 1{S_T > 1} S_T / S (d/d S/K) and
// 1{S_T > 1} S_T (sqrt(dt) sum z - sigma tau) (d/d sigma), discounted and
// averaged like the label; barrier points (a knock indicator has no pathwise
// derivative) get NaN.  Bound by drawing: a European path only adds its
// normals up (the label needs no date in between), a barrier path keeps the
// running maximum of its log-price and is tested against the barrier once;
// with one loop for both, an exponential and a comparison per date, 4096
// points x 2^13 paths took 8.49 ms.
template <bool GREEKS>
__global__ void __launch_bounds__(256) label_kernel(int64_t npts, const float *__restrict__ pts, int paths,
                                                    float steps_per_year, const __grid_constant__ RoundKeys rk,
                                                    float *__restrict__ labels, float *__restrict__ inputs,
                                                    float *__restrict__ dlabels)
{
    __shared__ double s_red[3][8];
    for (int64_t p = blockIdx.x; p < npts; p += gridDim.x) {
        const float sk = pts[p * 5 + 0], sig = pts[p * 5 + 1], tau = pts[p * 5 + 2], r = pts[p * 5 + 3],
                    kh = pts[p * 5 + 4];
        if (inputs && threadIdx.x == 0) surrogate_inputs(sk, sig, tau, r, kh, inputs + p * 5);
        const int M = max(1, __float2int_rn(tau * steps_per_year));
        const float dt = tau / M;
        const float H = kh > 0.0f ? 1.0f / kh : INFINITY;  // barrier in units of K
        const float a = kLog2e * (r - 0.5f * sig * sig) * dt, b = kLog2e * sig * sqrtf(dt);
        const bool greeks = GREEKS && !(kh > 0.0f);
        const int nfull = M >> 2, rest = M & 3;  // whole Philox blocks of a path, normals of the last one
        float acc = 0.0f, accd = 0.0f, accv = 0.0f;
        if (!(kh > 0.0f)) {
            // European: the terminal price depends on the normals' sum alone
            const float aT = a * static_cast<float>(M), sdt = sqrtf(dt);
            for (int path = threadIdx.x; path < paths; path += blockDim.x) {
                PathStream ps;
                ps.init(tag(4, (static_cast<uint64_t>(p) << 16) | static_cast<uint64_t>(path)), rk);
                f32x2 w = pack2(0.0f, 0.0f);
                for (int q = 0; q < nfull; ++q) {
                    const Normals4 z = ps.normals(static_cast<uint32_t>(q), rk);
                    w = fadd2(w, fadd2(z.a, z.b));
                }
                if (rest) {
                    const Normals4 z = ps.normals(static_cast<uint32_t>(nfull), rk);
                    w = fadd2(w, rest > 2 ? pack2(lo_of(z.a) + lo_of(z.b), hi_of(z.a))
                                          : pack2(lo_of(z.a), rest > 1 ? hi_of(z.a) : 0.0f));
                }
                const float zs = lo_of(w) + hi_of(w);
                const float g = ex2_approx(fmaf(b, zs, aT)), ST = sk * g;
                acc += fmaxf(ST - 1.0f, 0.0f);
                if (GREEKS && ST > 1.0f) {
                    accd += g;
                    accv += ST * fmaf(sdt, zs, -sig * tau);
                }
            }
        } else if (!(sk >= H)) {  // at or above the barrier on the current date: worthless
            for (int path = threadIdx.x; path < paths; path += blockDim.x) {
                PathStream ps;
                ps.init(tag(4, (static_cast<uint64_t>(p) << 16) | static_cast<uint64_t>(path)), rk);
                float y = 0.0f, mx = -INFINITY;  // log2(S / S_0) and its running maximum
                for (int q = 0; q < nfull; ++q) {
                    const float4 z = ps.normals(static_cast<uint32_t>(q), rk).f4();
                    y += fmaf(b, z.x, a);
                    mx = fmaxf(mx, y);
                    y += fmaf(b, z.y, a);
                    mx = fmaxf(mx, y);
                    y += fmaf(b, z.z, a);
                    mx = fmaxf(mx, y);
                    y += fmaf(b, z.w, a);
                    mx = fmaxf(mx, y);
                }
                if (rest) {
                    const float4 z = ps.normals(static_cast<uint32_t>(nfull), rk).f4();
                    y += fmaf(b, z.x, a);
                    mx = fmaxf(mx, y);
                    if (rest > 1) { y += fmaf(b, z.y, a); mx = fmaxf(mx, y); }
                    if (rest > 2) { y += fmaf(b, z.z, a); mx = fmaxf(mx, y); }
                }
                if (!(sk * ex2_approx(mx) >= H)) acc += fmaxf(sk * ex2_approx(y) - 1.0f, 0.0f);
            }
        }
        const double v[3] = {warp_sum_d(static_cast<double>(acc)), GREEKS ? warp_sum_d(static_cast<double>(accd)) : 0.0,
                             GREEKS ? warp_sum_d(static_cast<double>(accv)) : 0.0};
        if ((threadIdx.x & 31) == 0)
            for (int k = 0; k < (GREEKS ? 3 : 1); ++k) s_red[k][threadIdx.x >> 5] = v[k];
        __syncthreads();
        if (threadIdx.x == 0) {
            double t[3] = {0.0, 0.0, 0.0};
            for (int k = 0; k < (GREEKS ? 3 : 1); ++k)
                for (int w = 0; w < static_cast<int>(blockDim.x >> 5); ++w) t[k] += s_red[k][w];
            const double disc = exp(-static_cast<double>(r) * tau) / paths;
            if (GBMC_IN_BOUNDS(p, npts, kDbgLabelOut)) labels[p] = static_cast<float>(disc * t[0]);
            if (GREEKS) {
                dlabels[2 * p] = greeks ? static_cast<float>(disc * t[1]) : __int_as_float(0x7fc00000);
                dlabels[2 * p + 1] = greeks ? static_cast<float>(disc * t[2]) : __int_as_float(0x7fc00000);
            }
        }
        __syncthreads();
    }
}

// ------------------------------ scenarios --------------------------------
// Lc: [d x d] FP32 of sqrt(h) diag(sigma) Lrho (lower); drift_u = (mu - sigma^2/2) h.
__global__ void outer_kernel(int64_t nscen, int64_t off, int d, const float *__restrict__ Lc,
                             const float *__restrict__ drift, const float *__restrict__ s0, const __grid_constant__ RoundKeys rk,
                             float *__restrict__ Sp)
{
    extern __shared__ float sL[];
    for (int i = threadIdx.x; i < d * d; i += blockDim.x) sL[i] = Lc[i];
    __syncthreads();
    float z[kRiskMaxUnder];
    for (int64_t s = blockIdx.x * static_cast<int64_t>(blockDim.x) + threadIdx.x; s < nscen;
         s += static_cast<int64_t>(gridDim.x) * blockDim.x) {
        NormalReader rd;
        rd.init(tag(2, static_cast<uint64_t>(off + s)), rk);  // global scenario index
        for (int u = 0; u < d; ++u) z[u] = rd.get(u);
        for (int u = 0; u < d; ++u) {
            float w = 0.0f;
            for (int k = 0; k <= u; ++k) w = fmaf(sL[u * d + k], z[k], w);
            Sp[s * d + u] = s0[u] * expf(drift[u] + w);
        }
    }
}

// ------------------------------ nested -----------------------------------
// One CTA per (scenario s, underlying u) and slice of its inner paths, which
// start at S'_u and take daily steps; every option of u is valued at its
// remaining maturity; out[s*d + u] = sum_{o of u} pos_o (V_o(s) - base_o) in
// FP64.  Options are sorted by maturity, so a path runs from one maturity to
// the next without a test per date; the blocks that a maturity splits are
// finished on the other side of it.
// The paths fall into groups that depend on their number alone (nested_group):
// thread t adds the group's paths t, t + 256, ... in FP32, the CTA adds its
// threads in FP64, and the groups are added in FP64 in their order.  A slice is
// a run of whole groups, so a scenario's value has the same bits however many
// scenarios the call has and however many SMs share them (shards of a run).
// Few scenarios (the base date is one) are cut into slices, whose group sums
// nested_finish_kernel adds: the base values of 32 underlyings on 32 CTAs took
// as long as the 16384 CTAs of 512 scenarios (28.2 ms together for 1024 inner
// and 65536 base paths).

// Paths of a group: 1024, four per thread, or the multiple of that which keeps
// the groups at 256 (from 2^18 paths on).  The base date, one scenario, has
// groups of 256, one per thread, up to 2^16 paths, for more slices: 32 options
// on 4 underlyings, 4096 base paths, one scenario 314 us for 368.
__host__ __device__ constexpr int nested_group(int paths, bool base)
{
    const int unit = base ? 256 : 1024;
    return paths <= 256 * unit ? unit : (paths + 256 * unit - 1) / (256 * unit) * unit;
}

// Value of option j of underlying u at scenario price S1 from its payoff sum.
__device__ __forceinline__ double nested_value(const RiskArgs &a, int o, int hs, float S1, double sum)
{
    if (a.kind[o] == MC_UO_CALL && S1 >= a.barrier[o]) return 0.0;  // knocked out on the current date
    return exp(-static_cast<double>(a.r) * (a.rem[o] + hs) * a.dt) * sum / a.inner;
}

__global__ void __launch_bounds__(256, 8) nested_kernel(const __grid_constant__ RiskArgs a, const float *__restrict__ Sp,
                                                     double *__restrict__ out, double *__restrict__ part, int slices)
{
    __shared__ double s_v[kRiskMaxOptPerUnder];
    __shared__ double s_red[8][kRiskMaxOptPerUnder];
    __shared__ float s_K[kRiskMaxOptPerUnder], s_H[kRiskMaxOptPerUnder];
    __shared__ int s_t[kRiskMaxOptPerUnder], s_kind[kRiskMaxOptPerUnder];
    const int d = a.d;
    const int64_t pair = blockIdx.x / static_cast<unsigned>(slices);
    const int slice = static_cast<int>(blockIdx.x % static_cast<unsigned>(slices));
    const int64_t s = pair / d;
    const int u = static_cast<int>(pair % d);
    const int o0 = a.under_start[u], no = a.under_start[u + 1] - o0;  // options of u, sorted by maturity
    const int hs = Sp ? 0 : a.horizon_steps;  // base date: full maturity
    const float S1 = Sp ? Sp[s * d + u] : a.s0[u];
    const float sig = a.sigma[u];
    const float dt = a.dt;
    const float aa = kLog2e * (a.r - 0.5f * sig * sig) * dt, bb = kLog2e * sig * sqrtf(dt);
    if (threadIdx.x < no) {
        const int o = o0 + threadIdx.x;
        s_t[threadIdx.x] = a.rem[o] + hs;
        s_kind[threadIdx.x] = a.kind[o];
        s_K[threadIdx.x] = a.strike[o];
        s_H[threadIdx.x] = a.barrier[o];
    }
    __syncthreads();
    float acc[kRiskMaxOptPerUnder];
    const uint64_t gpair = static_cast<uint64_t>(a.scen_off + s) * d + u;  // global (scenario, underlying)
    const uint64_t base_idx = Sp ? (gpair << 16) : (static_cast<uint64_t>(u) << 24);
    const uint64_t domain = Sp ? 3 : 5;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int group = nested_group(a.inner, Sp == nullptr), groups = (a.inner + group - 1) / group, per = (groups + slices - 1) / slices;
    double total = 0.0;  // threads below `no`: the option's sum over this slice's groups
    for (int g = slice * per; g < min(groups, (slice + 1) * per); ++g) {
        const int last = min(a.inner, (g + 1) * group);
#pragma unroll
        for (int j = 0; j < kRiskMaxOptPerUnder; ++j) acc[j] = 0.0f;
        for (int path = g * group + threadIdx.x; path < last; path += blockDim.x) {
            PathStream ps;
            ps.init(tag(domain, base_idx | static_cast<uint64_t>(path)), a.rk);
            float y = 0.0f, mx = -INFINITY;  // log2(S/S1) and its running maximum over the dates
            float4 z = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
            auto step = [&](float zl) {
                y += fmaf(bb, zl, aa);
                mx = fmaxf(mx, y);
            };
            int q = 0, l = 0;  // next date 4 q + l + 1; z holds block q when l > 0
            for (int j = 0; j < no;) {
                const int t = s_t[j];
                if (l > 0) {  // the rest of the block that the last maturity split
                    const int e = min(4, t - 4 * q);
                    if (l <= 1 && e > 1) step(z.y);
                    if (l <= 2 && e > 2) step(z.z);
                    if (e > 3) step(z.w);
                    l = e;
                    if (l == 4) {
                        l = 0;
                        ++q;
                    }
                }
                for (; 4 * q + 4 <= t; ++q) {
                    z = ps.normals(static_cast<uint32_t>(q), a.rk).f4();
                    step(z.x);
                    step(z.y);
                    step(z.z);
                    step(z.w);
                }
                if (l == 0 && 4 * q < t) {
                    z = ps.normals(static_cast<uint32_t>(q), a.rk).f4();
                    l = t - 4 * q;
                    step(z.x);
                    if (l > 1) step(z.y);
                    if (l > 2) step(z.z);
                }
                const float ST = S1 * ex2_approx(y), Smx = S1 * ex2_approx(mx);
                for (; j < no && s_t[j] == t; ++j) {
                    float f = s_kind[j] == MC_PUT ? fmaxf(s_K[j] - ST, 0.0f) : fmaxf(ST - s_K[j], 0.0f);
                    if (s_kind[j] == MC_UO_CALL && Smx >= s_H[j]) f = 0.0f;
                    acc[j] += f;
                }
            }
        }
        // Block reduction per option (FP64).  Eight options share one exchange
        // tree, in which a lane hands over the half of its values that it does
        // not go on with: 9 FP64 additions for 40, each sum in warp_sum_d's order.
        for (int j0 = 0; j0 < no; j0 += 8) {
            double v[8];
#pragma unroll
            for (int j = 0; j < 8; ++j) v[j] = acc[j0 + j];
#pragma unroll
            for (int h = 4, o = 16; h >= 1; h >>= 1, o >>= 1) {
                const bool up = (lane & o) != 0;
#pragma unroll
                for (int j = 0; j < h; ++j) {
                    const double keep = up ? v[j + h] : v[j], give = up ? v[j] : v[j + h];
                    v[j] = keep + __shfl_xor_sync(0xffffffffu, give, o);
                }
            }
            v[0] += __shfl_xor_sync(0xffffffffu, v[0], 2);
            v[0] += __shfl_xor_sync(0xffffffffu, v[0], 1);
            if ((lane & 3) == 0) s_red[warp][j0 + (lane >> 2)] = v[0];
        }
        __syncthreads();
        if (threadIdx.x < no) {
            double t = 0.0;
            for (int w = 0; w < static_cast<int>(blockDim.x >> 5); ++w) t += s_red[w][threadIdx.x];
            if (slices > 1) part[(pair * groups + g) * kRiskMaxOptPerUnder + threadIdx.x] = t;
            else total += t;
        }
        __syncthreads();  // s_red is free for the next group
    }
    if (slices > 1) return;
    if (threadIdx.x < no) s_v[threadIdx.x] = nested_value(a, o0 + threadIdx.x, hs, S1, total);
    __syncthreads();
    if (threadIdx.x == 0) {
        double t = 0.0;
        for (int j = 0; j < no; ++j) {
            if (Sp) t += a.pos[o0 + j] * (s_v[j] - a.base[o0 + j]);
            else a.base_out[o0 + j] = s_v[j];
        }
        if (Sp) out[pair] = t;
    }
}

// One warp per (scenario, underlying): its groups' option sums, then as above.
__global__ void __launch_bounds__(32) nested_finish_kernel(const RiskArgs a, const float *__restrict__ Sp,
                                                           double *__restrict__ out, const double *__restrict__ part, int groups)
{
    __shared__ double s_v[kRiskMaxOptPerUnder];
    const int64_t pair = blockIdx.x;
    const int u = static_cast<int>(pair % a.d);
    const int o0 = a.under_start[u], no = a.under_start[u + 1] - o0, hs = Sp ? 0 : a.horizon_steps;
    const float S1 = Sp ? Sp[pair] : a.s0[u];
    if (threadIdx.x < no) {
        double t = 0.0;
        for (int k = 0; k < groups; ++k) t += part[(pair * groups + k) * kRiskMaxOptPerUnder + threadIdx.x];
        s_v[threadIdx.x] = nested_value(a, o0 + threadIdx.x, hs, S1, t);
    }
    __syncthreads();
    if (!Sp) {
        if (threadIdx.x < no) a.base_out[o0 + threadIdx.x] = s_v[threadIdx.x];
    } else if (threadIdx.x == 0) {
        double t = 0.0;
        for (int j = 0; j < no; ++j) t += a.pos[o0 + j] * (s_v[j] - a.base[o0 + j]);
        out[pair] = t;
    }
}

// ------------------------------ surrogate --------------------------------
// x[(s * nopt + o) * 5 ..]: network inputs of S/K, sigma, tau_remaining, r, K/H (0 = no barrier);
// Sp == nullptr: the base date (S0, full maturity).
__global__ void features_kernel(RiskArgs a, int64_t nscen, const float *__restrict__ Sp, float *__restrict__ x)
{
    const int64_t total = nscen * a.nopt;
    for (int64_t i = blockIdx.x * static_cast<int64_t>(blockDim.x) + threadIdx.x; i < total;
         i += static_cast<int64_t>(gridDim.x) * blockDim.x) {
        const int64_t s = i / a.nopt;
        const int o = static_cast<int>(i % a.nopt);
        const int u = a.under[o];
        const float S = Sp ? Sp[s * a.d + u] : a.s0[u];
        const float K = a.strike[o];
        const int steps = Sp ? a.rem[o] : a.rem[o] + a.horizon_steps;
        surrogate_inputs(S / K, a.sigma[u], steps * a.dt, a.r, a.kind[o] == MC_UO_CALL ? K / a.barrier[o] : 0.0f,
                         x + i * 5);
    }
}

// Value of option o from the network output y = V_call / K at its features.
__device__ __forceinline__ double option_value(const RiskArgs &a, int o, float S, float y, int steps)
{
    const double K = a.strike[o];
    double call = K * static_cast<double>(y);
    if (a.kind[o] == MC_UO_CALL) {
        if (S >= a.barrier[o]) return 0.0;
        return fmax(call, 0.0);
    }
    if (a.kind[o] == MC_PUT) return call - S + K * exp(-static_cast<double>(a.r) * steps * a.dt);  // parity
    return call;
}

// base_out[o] (Sp == nullptr) or pnl[s] = sum_o pos_o (V_o(s) - base_o).
__global__ void __launch_bounds__(256) pnl_kernel(RiskArgs a, const float *__restrict__ Sp, const float *__restrict__ y,
                                                  double *__restrict__ pnl)
{
    __shared__ double s_red[8];
    const int64_t s = blockIdx.x;
    double t = 0.0;
    for (int o = threadIdx.x; o < a.nopt; o += blockDim.x) {
        const int u = a.under[o];
        const float S = Sp ? Sp[s * a.d + u] : a.s0[u];
        const int steps = Sp ? a.rem[o] : a.rem[o] + a.horizon_steps;
        const double V = option_value(a, o, S, y[s * a.nopt + o], steps);
        if (Sp) t += a.pos[o] * (V - a.base[o]);
        else a.base_out[o] = V;
    }
    if (!Sp) return;
    t = warp_sum_d(t);
    if ((threadIdx.x & 31) == 0) s_red[threadIdx.x >> 5] = t;
    __syncthreads();
    if (threadIdx.x == 0) {
        double v = 0.0;
        for (int w = 0; w < static_cast<int>(blockDim.x >> 5); ++w) v += s_red[w];
        pnl[s] = v;
    }
}

// pnl[s] = sum_u contrib[s*d + u] (nested path).
__global__ void sum_under_kernel(int64_t nscen, int d, const double *contrib, double *pnl)
{
    for (int64_t s = blockIdx.x * static_cast<int64_t>(blockDim.x) + threadIdx.x; s < nscen;
         s += static_cast<int64_t>(gridDim.x) * blockDim.x) {
        double t = 0.0;
        for (int u = 0; u < d; ++u) t += contrib[s * d + u];
        pnl[s] = t;
    }
}

// ------------------------------ VaR / CVaR -------------------------------
// Losses l = -pnl: VaR = the k-th largest loss, k = ceil((1 - alpha) n), and
// CVaR = the mean of the losses strictly above VaR (VaR itself if there is
// none).  VaR by radix selection from the top: each pass histograms the next
// kTailBits bits of the losses' ordered keys among those that share the digits
// found so far, and its last CTA picks the digit that holds the k-th; then one
// pass adds up what lies above.  Seven reads of n values over the SMs, in
// launches of a few microseconds; a sort of all losses in one CTA took 6.5 ms
// of a 2^16-scenario run.  What one CTA reads anyway (kTailSmall losses) goes
// through the same passes in one launch: 1000 losses 47 us a call for 84.
constexpr int kTailBits = 11, kTailBins = 1 << kTailBits, kTailPasses = 6;  // 5 x 11 + 9 bits
constexpr int kTailBlock = 512, kTailMaxGrid = 304, kTailSmall = 2 * kTailBlock;
constexpr int kTailPer = kTailBins / kTailBlock;
struct TailState {
    unsigned long long prefix;       // the digits found
    unsigned int k;                  // rank among the losses that share them, from the largest
    unsigned int ticket[kTailPasses + 1];
    unsigned int hist[kTailPasses][kTailBins];
    double sum[kTailMaxGrid], count[kTailMaxGrid];
};

// Ascending unsigned order of the keys is ascending order of the doubles.
__device__ __forceinline__ unsigned long long loss_key(double l)
{
    const unsigned long long u = static_cast<unsigned long long>(__double_as_longlong(l));
    return (u >> 63) ? ~u : u | 0x8000000000000000ull;
}

__device__ __forceinline__ double key_loss(unsigned long long key)
{
    return __longlong_as_double(static_cast<long long>((key >> 63) ? key & 0x7fffffffffffffffull : ~key));
}

// The digit that pass `pass` looks at: `width` bits above `shift`, under the 64 - below bits found.
struct TailDigit {
    int below, width, shift;
    __device__ __forceinline__ explicit TailDigit(int pass)
        : below(64 - kTailBits * pass), width(below < kTailBits ? below : kTailBits), shift(below - width)
    {
    }
    __device__ __forceinline__ unsigned int of(unsigned long long key) const
    {
        return static_cast<unsigned int>((key >> shift) & ((1ull << width) - 1ull));
    }
};

// c: counts of the bins kTailBins - 1 - kTailPer t - j of thread t.  True in the one thread whose bins hold the k-th
// value from the top: *bin, and its rank there.
__device__ __forceinline__ bool tail_pick(const unsigned int (&c)[kTailPer], unsigned int k, unsigned int *bin, unsigned int *rank)
{
    __shared__ unsigned int scan[kTailBlock];
    const int t = threadIdx.x;
    unsigned int own = 0u;
    for (int j = 0; j < kTailPer; ++j) own += c[j];
    scan[t] = own;
    __syncthreads();
    for (int o = 1; o < kTailBlock; o <<= 1) {
        const unsigned int v = t >= o ? scan[t - o] : 0u;
        __syncthreads();
        scan[t] += v;
        __syncthreads();
    }
    unsigned int above = scan[t] - own;
    __syncthreads();
    if (!(above < k && k <= above + own)) return false;
    for (int j = 0; j < kTailPer; ++j) {
        if (k <= above + c[j]) {
            *bin = static_cast<unsigned int>(kTailBins - 1 - kTailPer * t - j);
            *rank = k - above;
            break;
        }
        above += c[j];
    }
    return true;
}

// This CTA's share of the losses above var: their sum and number, in thread 0.
__device__ __forceinline__ void tail_above(int64_t n, const double *__restrict__ pnl, double var, double *sum, double *count)
{
    __shared__ double s_red[2][kTailBlock / 32];
    double t = 0.0, c = 0.0;
    for (int64_t i = blockIdx.x * static_cast<int64_t>(kTailBlock) + threadIdx.x; i < n; i += static_cast<int64_t>(gridDim.x) * kTailBlock) {
        const double l = -pnl[i];
        if (l > var) {
            t += l;
            c += 1.0;
        }
    }
    t = warp_sum_d(t);
    c = warp_sum_d(c);
    if ((threadIdx.x & 31) == 0) {
        s_red[0][threadIdx.x >> 5] = t;
        s_red[1][threadIdx.x >> 5] = c;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        t = c = 0.0;
        for (int w = 0; w < kTailBlock / 32; ++w) {
            t += s_red[0][w];
            c += s_red[1][w];
        }
        *sum = t;
        *count = c;
    }
}

// All passes of up to kTailSmall losses in one CTA.
__global__ void __launch_bounds__(kTailBlock) tail_small_kernel(int n, const double *__restrict__ pnl, unsigned int k0, double *res)
{
    __shared__ unsigned int h[kTailBins];
    __shared__ unsigned long long s_prefix;
    __shared__ unsigned int s_k;
    const int t = threadIdx.x;
    if (t == 0) {
        s_prefix = 0ull;
        s_k = k0;
    }
    for (int pass = 0; pass < kTailPasses; ++pass) {
        const TailDigit dg(pass);
        for (int b = t; b < kTailBins; b += kTailBlock) h[b] = 0u;
        __syncthreads();
        const unsigned long long prefix = s_prefix;
        for (int i = t; i < n; i += kTailBlock) {
            const unsigned long long key = loss_key(-pnl[i]);
            if (pass == 0 || (key >> dg.below) == prefix) atomicAdd(&h[dg.of(key)], 1u);
        }
        __syncthreads();
        unsigned int c[kTailPer], bin, rank;
        for (int j = 0; j < kTailPer; ++j) c[j] = h[kTailBins - 1 - kTailPer * t - j];
        if (tail_pick(c, s_k, &bin, &rank)) {
            s_prefix = (prefix << dg.width) | bin;
            s_k = rank;
        }
        __syncthreads();
    }
    const double var = key_loss(s_prefix);
    double sum = 0.0, count = 0.0;
    tail_above(n, pnl, var, &sum, &count);
    if (t == 0) {
        res[0] = var;
        res[1] = count > 0.0 ? sum / count : var;
        res[2] = count;
    }
}

// Whether this CTA is the last of the launch to arrive (the others' writes are then visible).
__device__ __forceinline__ bool last_cta(unsigned int *ticket)
{
    __shared__ unsigned int s_last;
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0) s_last = atomicAdd(ticket, 1u) == gridDim.x - 1 ? 1u : 0u;
    __syncthreads();
    if (s_last) __threadfence();
    return s_last != 0u;
}

__global__ void __launch_bounds__(kTailBlock) tail_pass_kernel(int64_t n, const double *__restrict__ pnl, int pass,
                                                               unsigned int k0, TailState *st)
{
    __shared__ unsigned int h[kTailBins];
    const int t = threadIdx.x;
    const TailDigit dg(pass);
    const unsigned long long prefix = pass ? st->prefix : 0ull;
    for (int b = t; b < kTailBins; b += kTailBlock) h[b] = 0u;
    __syncthreads();
    for (int64_t i = blockIdx.x * static_cast<int64_t>(kTailBlock) + t; i < n; i += static_cast<int64_t>(gridDim.x) * kTailBlock) {
        const unsigned long long key = loss_key(-pnl[i]);
        if (pass == 0 || (key >> dg.below) == prefix) atomicAdd(&h[dg.of(key)], 1u);
    }
    __syncthreads();
    for (int b = t; b < kTailBins; b += kTailBlock)
        if (h[b]) atomicAdd(&st->hist[pass][b], h[b]);
    if (!last_cta(&st->ticket[pass])) return;
    unsigned int c[kTailPer], bin, rank;
    for (int j = 0; j < kTailPer; ++j) c[j] = *reinterpret_cast<volatile unsigned int *>(&st->hist[pass][kTailBins - 1 - kTailPer * t - j]);
    const unsigned int k = pass ? st->k : k0;
    if (tail_pick(c, k, &bin, &rank)) {
        st->prefix = (prefix << dg.width) | bin;
        st->k = rank;
    }
}

__global__ void __launch_bounds__(kTailBlock) tail_sum_kernel(int64_t n, const double *__restrict__ pnl, TailState *st, double *res)
{
    const double var = key_loss(st->prefix);
    double t = 0.0, c = 0.0;
    tail_above(n, pnl, var, &t, &c);
    if (threadIdx.x == 0) {
        st->sum[blockIdx.x] = t;
        st->count[blockIdx.x] = c;
    }
    if (!last_cta(&st->ticket[kTailPasses]) || threadIdx.x != 0) return;
    t = c = 0.0;
    for (unsigned int g = 0; g < gridDim.x; ++g) {
        t += *reinterpret_cast<volatile double *>(&st->sum[g]);
        c += *reinterpret_cast<volatile double *>(&st->count[g]);
    }
    res[0] = var;
    res[1] = c > 0.0 ? t / c : var;
    res[2] = c;
}

}  // namespace

cudaError_t launch_labels(int64_t npts, const float *pts, int paths, float spy, const RoundKeys &rk,
                          float *labels, float *inputs, float *dlabels, cudaStream_t s)
{
    const int64_t g = npts < 1216 * 4 ? npts : 1216 * 4;
    if (dlabels)
        label_kernel<true><<<static_cast<int>(g), 256, 0, s>>>(npts, pts, paths, spy, rk, labels, inputs, dlabels);
    else
        label_kernel<false><<<static_cast<int>(g), 256, 0, s>>>(npts, pts, paths, spy, rk, labels, inputs, nullptr);
    return cudaGetLastError();
}

cudaError_t launch_outer(int64_t nscen, int64_t off, int d, const float *Lc, const float *drift, const float *s0,
                         const RoundKeys &rk, float *Sp, cudaStream_t s)
{
    const int64_t g = (nscen + 127) / 128;
    outer_kernel<<<static_cast<int>(g < 4096 ? g : 4096), 128, d * d * sizeof(float), s>>>(nscen, off, d, Lc, drift,
                                                                                            s0, rk, Sp);
    return cudaGetLastError();
}

// Slices of the inner paths: none once the pairs alone are eight CTAs per SM,
// else as many as reach that, each of at least one group.
int nested_slices(int64_t pairs, int inner, bool base, int sms)
{
    const int group = nested_group(inner, base), groups = (inner + group - 1) / group;
    const int64_t want = (8 * static_cast<int64_t>(sms) + pairs - 1) / pairs;
    const int n = static_cast<int>(std::max<int64_t>(1, std::min<int64_t>(want, groups))), per = (groups + n - 1) / n;
    return (groups + per - 1) / per;
}

size_t nested_part_doubles(int64_t pairs, int inner, bool base, int slices)
{
    const int group = nested_group(inner, base);
    return slices > 1 ? static_cast<size_t>(pairs) * ((inner + group - 1) / group) * kRiskMaxOptPerUnder : 0;
}

cudaError_t launch_nested(const RiskArgs &a, int64_t nscen, const float *Sp, double *contrib, double *part, int slices,
                          cudaStream_t s)
{
    const int64_t pairs = Sp ? nscen * a.d : a.d;
    nested_kernel<<<static_cast<unsigned>(pairs * slices), 256, 0, s>>>(a, Sp, contrib, part, slices);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess || slices == 1) return e;
    const int group = nested_group(a.inner, Sp == nullptr);
    nested_finish_kernel<<<static_cast<unsigned>(pairs), 32, 0, s>>>(a, Sp, contrib, part, (a.inner + group - 1) / group);
    return cudaGetLastError();
}

cudaError_t launch_sum_under(int64_t nscen, int d, const double *contrib, double *pnl, cudaStream_t s)
{
    const int64_t g = (nscen + 255) / 256;
    sum_under_kernel<<<static_cast<int>(g < 4096 ? g : 4096), 256, 0, s>>>(nscen, d, contrib, pnl);
    return cudaGetLastError();
}

cudaError_t launch_features(const RiskArgs &a, int64_t nscen, const float *Sp, float *x, cudaStream_t s)
{
    features_kernel<<<4096, 256, 0, s>>>(a, nscen, Sp, x);
    return cudaGetLastError();
}

cudaError_t launch_pnl(const RiskArgs &a, int64_t nscen, const float *Sp, const float *y, double *pnl, cudaStream_t s)
{
    pnl_kernel<<<static_cast<int>(Sp ? nscen : 1), 256, 0, s>>>(a, Sp, y, pnl);
    return cudaGetLastError();
}

size_t tail_scratch_bytes() { return sizeof(TailState); }

cudaError_t launch_tail(int64_t n, const double *pnl, void *scratch, double alpha, double *res, cudaStream_t s)
{
    TailState *st = static_cast<TailState *>(scratch);
    int64_t k = static_cast<int64_t>(std::ceil((1.0 - alpha) * static_cast<double>(n) - 1e-9));
    if (k < 1) k = 1;
    if (n <= kTailSmall) {
        tail_small_kernel<<<1, kTailBlock, 0, s>>>(static_cast<int>(n), pnl, static_cast<unsigned int>(k), res);
        return cudaGetLastError();
    }
    cudaError_t e = cudaMemsetAsync(st, 0, sizeof(TailState), s);
    if (e != cudaSuccess) return e;
    const int grid = static_cast<int>(std::min<int64_t>(kTailMaxGrid, (n + 2 * kTailBlock - 1) / (2 * kTailBlock)));
    for (int pass = 0; pass < kTailPasses; ++pass) {
        tail_pass_kernel<<<grid, kTailBlock, 0, s>>>(n, pnl, pass, static_cast<unsigned int>(k), st);
        if ((e = cudaGetLastError()) != cudaSuccess) return e;
    }
    tail_sum_kernel<<<grid, kTailBlock, 0, s>>>(n, pnl, st, res);
    return cudaGetLastError();
}

}  // namespace gbmc

// Device building blocks shared by the path kernels: the keyed counter-based
// generator (Sec. IV.A), the Box-Muller transform (Sec. VI.D), payoffs on the
// monitored underlying (Sec. I.A.2) and the warp / block / cross-block
// reduction that ends in the FP64 estimator of Eq. 3.
#pragma once

#include <cstdint>
#include <cuda_runtime.h>

#include "../../include/mc.h"

namespace gbmc {

constexpr float kLog2e = 1.4426950408889634f;

// ---------------------------------------------------------------------------
// Philox4x32-10 (Salmon et al., SC'11): ten rounds of two 32x32->64 products
// with the round multipliers, xor of the high halves with the other counter
// words and the round key, and a Weyl bump of the key between rounds.  The
// ten round keys are formed once per launch on the host and read from the
// kernel's parameter block (constant bank), so no round spends an
// instruction or a register on the key schedule.
// ---------------------------------------------------------------------------
constexpr uint32_t kPhiloxM0 = 0xD2511F53u, kPhiloxM1 = 0xCD9E8D57u;

struct RoundKeys {
    uint32_t k[20];  // round r: (k[2r], k[2r + 1]) = (k0 + r 0x9E3779B9, k1 + r 0xBB67AE85)
};

__host__ __device__ inline RoundKeys round_keys(uint32_t k0, uint32_t k1)
{
    RoundKeys rk;
    for (int r = 0; r < 10; ++r) {
        rk.k[2 * r] = k0 + static_cast<uint32_t>(r) * 0x9E3779B9u;
        rk.k[2 * r + 1] = k1 + static_cast<uint32_t>(r) * 0xBB67AE85u;
    }
    return rk;
}

__device__ __forceinline__ uint4 philox4x32_10(uint4 c, const RoundKeys &rk)
{
#pragma unroll
    for (int round = 0; round < 10; ++round) {
        const uint64_t p0 = static_cast<uint64_t>(kPhiloxM0) * c.x;
        const uint64_t p1 = static_cast<uint64_t>(kPhiloxM1) * c.z;
        const uint32_t hi0 = static_cast<uint32_t>(p0 >> 32), lo0 = static_cast<uint32_t>(p0);
        const uint32_t hi1 = static_cast<uint32_t>(p1 >> 32), lo1 = static_cast<uint32_t>(p1);
        c = make_uint4(hi1 ^ c.y ^ rk.k[2 * round], lo1, hi0 ^ c.w ^ rk.k[2 * round + 1], lo0);
    }
    return c;
}

// u = (floor(x / 2^9) + 1/2) 2^-23 in [2^-24, 1 - 2^-24], exact in binary32:
// the bits of 1 + floor(x/2^9) 2^-23 minus (1 - 2^-24) (Sterbenz: exact).
__device__ __forceinline__ float one_plus(uint32_t x) { return __uint_as_float(0x3F800000u | (x >> 9)); }
__device__ __forceinline__ float u01(uint32_t x) { return one_plus(x) - 0.99999994039535522f; }

// Box-Muller on one pair of words: z0 = r cos(2 pi u_b), z1 = r sin(2 pi u_b),
// r = sqrt(-2 ln u_a), evaluated with the SFU's approximate instructions
// (lg2, sqrt, sin, cos: one issue slot each).  The angle is taken as
// theta = 2 pi (u_b - 1/2) in (-pi, pi), the range where sin/cos.approx are
// most accurate, and the sign flip (cos(theta) = -cos(2 pi u_b), likewise
// sin) is folded into r.  theta comes from one FMA on f = 1 + floor(b/2^9)
// 2^-23 (the bits of u01 before its subtraction): f fl(2 pi) - fl(3 pi),
// within 3.5e-7 of 2 pi (u_b - 1/2) over all 2^23 values of f (two roundings
// of the constants, one of the FMA) and inside (-pi, pi).  lg2.approx has an
// absolute error near 2^-22 close to u = 1; it is never positive on the 2^23
// uniforms, and the square root takes its operand's magnitude, a free source
// modifier, where a clamp at 0 would cost an instruction per pair.
// The per-normal absolute error is a few 1e-6, except for u_a within ~1e-6
// of 1, where r < ~1.5e-3 is off by at most sqrt(1.39 * 2^-22) ~ 6e-4.
__device__ __forceinline__ float lg2_approx(float x)
{
    float y;
    asm("lg2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}
__device__ __forceinline__ float sqrt_approx(float x)
{
    float y;
    asm("sqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}
__device__ __forceinline__ float sin_approx(float x)
{
    float y;
    asm("sin.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}
__device__ __forceinline__ float cos_approx(float x)
{
    float y;
    asm("cos.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}
__device__ __forceinline__ float ex2_approx(float x)
{
    float y;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

__device__ __forceinline__ void box_muller(uint32_t a, uint32_t b, float &z0, float &z1)
{
    const float ua = u01(a);
    // -2 ln u = -2 ln(2) log2(u)
    const float nrad = -sqrt_approx(fabsf(-1.3862943611198906f * lg2_approx(ua)));
    const float theta = fmaf(one_plus(b), 6.2831854820251465f, -9.42477798461914f);
    z0 = nrad * cos_approx(theta);
    z1 = nrad * sin_approx(theta);
}

// Packed FP32 pairs (fma.rn.f32x2 and friends: each lane an ordinary FP32
// operation; low half = the even element).
using f32x2 = unsigned long long;
__device__ __forceinline__ f32x2 ffma2(f32x2 a, f32x2 b, f32x2 c)
{
    f32x2 d;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
    return d;
}
__device__ __forceinline__ f32x2 fadd2(f32x2 a, f32x2 b)
{
    f32x2 d;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}
__device__ __forceinline__ f32x2 fmul2(f32x2 a, f32x2 b)
{
    f32x2 d;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}
__device__ __forceinline__ f32x2 pack2(float lo, float hi)
{
    f32x2 d;
    asm("mov.b64 %0, {%1, %2};" : "=l"(d) : "f"(lo), "f"(hi));
    return d;
}
__device__ __forceinline__ float lo_of(f32x2 v) { return __uint_as_float(static_cast<uint32_t>(v)); }
__device__ __forceinline__ float hi_of(f32x2 v) { return __uint_as_float(static_cast<uint32_t>(v >> 32)); }

// box_muller on the two pairs of a block's words, the FP32 operations of both
// pairs in packed instructions: the same operations on the same values, so the
// same bits, in five FMA-pipe instructions fewer.  The FMA pipe's integer half
// is what bounds drawing (PathStream), and a scalar FP32 instruction that
// lands on it costs two of its cycles.
struct Normals4 {
    f32x2 a, b;  // (z0, z1), (z2, z3)
    __device__ __forceinline__ float4 f4() const { return make_float4(lo_of(a), hi_of(a), lo_of(b), hi_of(b)); }
};
__device__ __forceinline__ Normals4 normals_of(uint4 w)
{
    const f32x2 ua = fadd2(pack2(one_plus(w.x), one_plus(w.z)), pack2(-0.99999994039535522f, -0.99999994039535522f));
    const f32x2 r2 = fmul2(pack2(lg2_approx(lo_of(ua)), lg2_approx(hi_of(ua))),
                           pack2(-1.3862943611198906f, -1.3862943611198906f));
    const f32x2 th = ffma2(pack2(one_plus(w.y), one_plus(w.w)), pack2(6.2831854820251465f, 6.2831854820251465f),
                           pack2(-9.42477798461914f, -9.42477798461914f));
    const float na = -sqrt_approx(fabsf(lo_of(r2))), nb = -sqrt_approx(fabsf(hi_of(r2)));
    Normals4 z;
    z.a = fmul2(pack2(na, na), pack2(cos_approx(lo_of(th)), sin_approx(lo_of(th))));
    z.b = fmul2(pack2(nb, nb), pack2(cos_approx(hi_of(th)), sin_approx(hi_of(th))));
    return z;
}

// The four normals of block q of stream (path) n.
__device__ __forceinline__ float4 normals4(uint64_t q, uint64_t n, const RoundKeys &rk)
{
    const uint4 x = philox4x32_10(make_uint4(static_cast<uint32_t>(q), static_cast<uint32_t>(q >> 32),
                                             static_cast<uint32_t>(n), static_cast<uint32_t>(n >> 32)),
                                  rk);
    float4 z;
    box_muller(x.x, x.y, z.x, z.y);
    box_muller(x.z, x.w, z.z, z.w);
    return z;
}

// The Philox blocks of one stream (path) n whose index has the given high
// word.  The counter's words y, z, w then do not change along the path, so
// round 0's product of z and round 1's product of x are formed once and kept,
// with the round keys that meet them, in four registers: 17 of the 20
// products and 33 of the 40 xors remain per block.  Drawing is bound by the
// products, which run on half of the FMA pipe at four cycles per warp
// instruction.  Summing normals only, 8 blocks of 128 threads per SM:
// 1.25e12 normals/s with the plain rounds above, 1.42e12 with these
// (1.21e12 -> 1.35e12 with 32 sums per thread, 1.45e12 with normals_of).
struct PathStream {
    uint32_t y1, ph, pl, nk;  // y1 ^ k2, hi(M0 x1) ^ k3, lo(M0 x1) ^ k5, n_hi ^ k1

    __device__ __forceinline__ void init(uint64_t n, const RoundKeys &rk, uint32_t q_hi = 0u)
    {
        const uint64_t p1 = static_cast<uint64_t>(kPhiloxM1) * static_cast<uint32_t>(n);
        const uint64_t p0 = static_cast<uint64_t>(kPhiloxM0) * (static_cast<uint32_t>(p1 >> 32) ^ q_hi ^ rk.k[0]);
        y1 = static_cast<uint32_t>(p1) ^ rk.k[2];
        ph = static_cast<uint32_t>(p0 >> 32) ^ rk.k[3];
        pl = static_cast<uint32_t>(p0) ^ rk.k[5];
        nk = static_cast<uint32_t>(n >> 32) ^ rk.k[1];
    }
    // Block with low index word q.
    __device__ __forceinline__ uint4 block(uint32_t q, const RoundKeys &rk) const
    {
        const uint64_t a = static_cast<uint64_t>(kPhiloxM0) * q;                                      // round 0
        const uint64_t b = static_cast<uint64_t>(kPhiloxM1) * (static_cast<uint32_t>(a >> 32) ^ nk);  // round 1
        const uint64_t c = static_cast<uint64_t>(kPhiloxM0) * (static_cast<uint32_t>(b >> 32) ^ y1);  // round 2
        const uint64_t d = static_cast<uint64_t>(kPhiloxM1) * (ph ^ static_cast<uint32_t>(a));
        uint32_t x = static_cast<uint32_t>(d >> 32) ^ static_cast<uint32_t>(b) ^ rk.k[4], y = static_cast<uint32_t>(d);
        uint32_t z = static_cast<uint32_t>(c >> 32) ^ pl, w = static_cast<uint32_t>(c);
#pragma unroll
        for (int round = 3; round < 10; ++round) {
            const uint64_t p0 = static_cast<uint64_t>(kPhiloxM0) * x, p1 = static_cast<uint64_t>(kPhiloxM1) * z;
            x = static_cast<uint32_t>(p1 >> 32) ^ y ^ rk.k[2 * round];
            z = static_cast<uint32_t>(p0 >> 32) ^ w ^ rk.k[2 * round + 1];
            y = static_cast<uint32_t>(p1);
            w = static_cast<uint32_t>(p0);
        }
        return make_uint4(x, y, z, w);
    }
    __device__ __forceinline__ Normals4 normals(uint32_t q, const RoundKeys &rk) const { return normals_of(block(q, rk)); }
};

// Sequential reader of normal j of one stream, for any j: regenerates a block
// only when j leaves the cached one (warp-uniform when all lanes are at the
// same j).
struct NormalReader {
    uint64_t n;
    const RoundKeys *rk;
    uint64_t q;
    float4 z;
    __device__ __forceinline__ void init(uint64_t stream, const RoundKeys &keys)
    {
        n = stream; rk = &keys; q = ~0ull;
    }
    __device__ __forceinline__ float get(uint64_t j)
    {
        const uint64_t qj = j >> 2;
        if (qj != q) { q = qj; z = normals4(qj, n, *rk); }
        const uint32_t l = static_cast<uint32_t>(j) & 3u;
        return l == 0 ? z.x : (l == 1 ? z.y : (l == 2 ? z.z : z.w));
    }
};

// How a step's normals are read.
constexpr int kReadAny = 0;      // NormalReader: materialised paths, and paths of more than 2^32 Philox blocks
constexpr int kReadAligned = 1;  // every step is whole blocks
constexpr int kReadShifted = 2;  // any d: two blocks in registers, lanes picked by the step's place in the first

// Lanes o .. o + 3 of two consecutive blocks.
__device__ __forceinline__ float4 shifted4(float4 cur, float4 nxt, int o)
{
    const bool two = (o & 2) != 0, one = (o & 1) != 0;
    const float s0 = two ? cur.z : cur.x, s1 = two ? cur.w : cur.y, s2 = two ? nxt.x : cur.z, s3 = two ? nxt.y : cur.w,
                s4 = two ? nxt.z : nxt.x;
    return make_float4(one ? s1 : s0, one ? s2 : s1, one ? s3 : s2, one ? s4 : s3);
}

// Normals 4 kb .. 4 kb + 3 of the running step for a d that need not be a
// multiple of 4: they lie in the two consecutive blocks held, from lane o on.
// Where a step ends inside a block, the block is kept for the next step, so
// every block is drawn once.  A branch per normal instead (NormalReader)
// unrolls a copy of Philox for each of them: 4.13 ms for 100,003 paths x 100
// steps of 50 assets.
struct ShiftedReader {
    PathStream ps;
    float4 cur, nxt;
    __device__ __forceinline__ void init(uint64_t n, const RoundKeys &rk)
    {
        ps.init(n, rk);
        cur = ps.normals(0u, rk).f4();
        nxt = ps.normals(1u, rk).f4();
    }
    __device__ __forceinline__ float4 group(int o) const { return shifted4(cur, nxt, o); }
    // On to the next pair of blocks; b: the index of the block after them.
    __device__ __forceinline__ void advance(uint32_t b, const RoundKeys &rk)
    {
        cur = nxt;
        nxt = ps.normals(b, rk).f4();
    }
};

// The same for paths of more than 2^32 Philox blocks (64-bit block indices).
struct WideReader {
    uint64_t n, b;
    float4 cur, nxt;
    __device__ __forceinline__ void init(uint64_t path, const RoundKeys &rk)
    {
        n = path;
        b = 1;
        cur = normals4(0, n, rk);
        nxt = normals4(1, n, rk);
    }
    __device__ __forceinline__ float4 group(int o) const { return shifted4(cur, nxt, o); }
    __device__ __forceinline__ void advance(const RoundKeys &rk)
    {
        cur = nxt;
        nxt = normals4(++b, n, rk);
    }
};

// ---------------------------------------------------------------------------
// Summed normals.  Under log-Euler with constant coefficients the terminal
// log-prices of a basket depend on a path's normals only through
// W_k = sum_i z_{i d + k}, so payoffs on the terminal value alone need one
// contraction per path, of W, instead of one per step.  Steps that share
// their position inside a Philox block (all of them when 4 | d, every second
// or fourth otherwise) form a segment: the same blocks of each, added up in
// registers without a select, so that a step of any width costs its blocks.
// ---------------------------------------------------------------------------
struct Segments {
    uint32_t period;  // steps until a step starts again at the same place of a block: 1, 2 or 4
    uint32_t blocks;  // Philox blocks of `period` steps
    int steps, d;

    __device__ __forceinline__ Segments(int steps_, int d_)
        : period((d_ & 3) == 0 ? 1u : (d_ & 1) == 0 ? 2u : 4u), blocks(period * static_cast<uint32_t>(d_) / 4u), steps(steps_),
          d(d_)
    {
    }
    // Segment p: the steps p, p + period, ...; their first normal is lane `lane` of their first block `block`.
    __device__ __forceinline__ int count(uint32_t p) const
    {
        return static_cast<int>((static_cast<uint32_t>(steps) + period - 1u - p) / period);
    }
    __device__ __forceinline__ uint32_t first_block(uint32_t p) const { return p * static_cast<uint32_t>(d) >> 2; }
    __device__ __forceinline__ int lane(uint32_t p) const { return static_cast<int>(p * static_cast<uint32_t>(d) & 3u); }
};

// w = the sums over `count` steps, `blocks` Philox blocks apart, of the
// normals of blocks b, b + stride, ... (NB of them) of stream n.  wide: a block
// index may pass 2^32.
// f(n) with n = min(left, 4) as a constant: the blocks a thread has left, at
// most four of them summed at a time (a fixed four would draw the ones past
// the end too: half of all for 64 assets over eight threads).
template <int N>
struct Blocks {
    static constexpr int value = N;
};
template <class F>
__device__ __forceinline__ void up_to_four(int left, const F &f)
{
    if (left >= 4) f(Blocks<4>{});
    else if (left == 3) f(Blocks<3>{});
    else if (left == 2) f(Blocks<2>{});
    else f(Blocks<1>{});
}
template <int NB>
__device__ __forceinline__ void sum_blocks(f32x2 (&w)[2 * NB], uint64_t n, const RoundKeys &rk, bool wide, uint64_t b,
                                           uint32_t stride, int count, uint32_t blocks)
{
#pragma unroll
    for (int j = 0; j < 2 * NB; ++j) w[j] = pack2(0.0f, 0.0f);
    if (!wide) {
        PathStream ps;
        ps.init(n, rk);
        uint32_t q = static_cast<uint32_t>(b);
        for (int s = 0; s < count; ++s, q += blocks)
#pragma unroll
            for (int j = 0; j < NB; ++j) {
                const Normals4 z = ps.normals(q + stride * j, rk);
                w[2 * j] = fadd2(w[2 * j], z.a);
                w[2 * j + 1] = fadd2(w[2 * j + 1], z.b);
            }
    } else {
        for (int s = 0; s < count; ++s)
#pragma unroll 1
            for (int j = 0; j < NB; ++j) {
                const float4 z = normals4(static_cast<uint64_t>(s) * blocks + b + stride * j, n, rk);
                const f32x2 za = pack2(z.x, z.y), zb = pack2(z.z, z.w);
#pragma unroll
                for (int k = 0; k < NB; ++k) {
                    if (k == j) {
                        w[2 * k] = fadd2(w[2 * k], za);
                        w[2 * k + 1] = fadd2(w[2 * k + 1], zb);
                    }
                }
            }
    }
}

// ---------------------------------------------------------------------------
// Payoffs (undiscounted) on the monitored statistics of U.
// ---------------------------------------------------------------------------
struct PayoffSet {
    int n;
    int need_avg;   // some payoff uses the arithmetic average
    int need_max;   // some payoff uses the running maximum
    int need_min;   // some payoff uses the running minimum
    int kind[MC_MAX_PAYOFFS];
    float strike[MC_MAX_PAYOFFS];
    float barrier[MC_MAX_PAYOFFS];
};

__device__ __forceinline__ float payoff_eval(int kind, float K, float H, float uT, float avg,
                                             float umax, float umin)
{
    const float call = fmaxf(uT - K, 0.0f), put = fmaxf(K - uT, 0.0f);
    const bool up = umax >= H, down = umin <= H;
    switch (kind) {
    case MC_CALL: return call;
    case MC_PUT: return put;
    case MC_ASIAN_CALL: return fmaxf(avg - K, 0.0f);
    case MC_ASIAN_PUT: return fmaxf(K - avg, 0.0f);
    case MC_UO_CALL: return up ? 0.0f : call;
    case MC_UI_CALL: return up ? call : 0.0f;
    case MC_UO_PUT: return up ? 0.0f : put;
    case MC_UI_PUT: return up ? put : 0.0f;
    case MC_DO_CALL: return down ? 0.0f : call;
    case MC_DI_CALL: return down ? call : 0.0f;
    case MC_DO_PUT: return down ? 0.0f : put;
    case MC_DI_PUT: return down ? put : 0.0f;
    default: return 0.0f;
    }
}

// ---------------------------------------------------------------------------
// Reduction.  Each warp owns a slot per payoff in shared memory; after every
// grid-stride iteration the warp's 32 payoffs (and squares) are summed in
// FP32 with shuffles and lane 0 adds them to its FP64 slot (fixed order:
// deterministic; FP64 so that a slot's error does not grow with the paths
// per thread).  At block end the warp slots are summed into one (sum f,
// sum f^2) pair per payoff, written to the block's partials in FP32.  The
// last block to finish (atomic ticket, no spin-wait) adds all block partials
// with compensated (Kahan) FP64 sums, forms mean and standard error,
// discounts and writes the results, then resets the ticket for the next
// launch.
// ---------------------------------------------------------------------------
using AccSlot = double;  // per-warp payoff slot in shared memory

// Compensated summation (Kahan): s + c carries the sum to about one FP64
// rounding whatever the number of terms.
struct KahanSum {
    double s = 0.0, c = 0.0;
    __device__ __forceinline__ void add(double x)
    {
        const double y = x - c;
        const double t = s + y;
        c = (t - s) - y;
        s = t;
    }
};
struct ReduceArgs {
    float *partials;        // [gridDim.x][n_payoff][2]
    unsigned int *ticket;   // zero on entry to the launch, reset by the last block
    mc_result *out;         // [n_payoff]
    int64_t paths;
    double disc;
    const unsigned int *err;  // optional: non-zero means a CTA gave up; results become NaN
};

__device__ __forceinline__ float warp_sum(float v)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

__device__ __forceinline__ double warp_sum_d(double v)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

// Adds this warp's 32 payoff values to s_acc[warp][p][*].
__device__ __forceinline__ void warp_accumulate(AccSlot *s_acc, int np, int p, float f)
{
    const float a = warp_sum(f), b = warp_sum(f * f);
    if ((threadIdx.x & 31) == 0) {
        AccSlot *slot = s_acc + ((threadIdx.x >> 5) * np + p) * 2;
        slot[0] += static_cast<double>(a);
        slot[1] += static_cast<double>(b);
    }
}

// The same for eight values at a time (v[j] to p0 + j < np): the sixteen sums
// (values and squares) share one exchange tree, in which a lane hands over the
// half of its values that it does not go on with, 16 shuffles instead of 80;
// every sum adds the lanes in the order of warp_sum, so the bits are the same,
// and the slots are updated by sixteen lanes at once.
template <class At>
__device__ __forceinline__ void warp_accumulate8_at(AccSlot *s_acc, int np, const float (&v)[8], const At &at)
{
    const int lane = threadIdx.x & 31;
    float a[16];
#pragma unroll
    for (int j = 0; j < 8; ++j) {
        a[2 * j] = v[j];
        a[2 * j + 1] = v[j] * v[j];
    }
#pragma unroll
    for (int h = 8, o = 16; h >= 1; h >>= 1, o >>= 1) {
        const bool up = (lane & o) != 0;
#pragma unroll
        for (int j = 0; j < h; ++j) {
            const float keep = up ? a[j + h] : a[j], give = up ? a[j] : a[j + h];
            a[j] = keep + __shfl_xor_sync(0xffffffffu, give, o);
        }
    }
    a[0] += __shfl_xor_sync(0xffffffffu, a[0], 1);
    const int e = lane >> 1, p = at(e >> 1);  // this lane pair's sum, and the slot of its value (none if negative)
    if ((lane & 1) == 0 && p >= 0) s_acc[((threadIdx.x >> 5) * np + p) * 2 + (e & 1)] += static_cast<double>(a[0]);
}
__device__ __forceinline__ void warp_accumulate8(AccSlot *s_acc, int np, int p0, const float (&v)[8])
{
    warp_accumulate8_at(s_acc, np, v, [&](int k) { return p0 + k < np ? p0 + k : -1; });
}

// Called by every thread of the block after its last path.  s_acc holds
// nwarps*np*2 slots; s_red is scratch for 32 doubles.
__device__ inline void block_finish(AccSlot *s_acc, double *s_red, int np, const ReduceArgs &ra)
{
    const int nwarps = blockDim.x >> 5;
    __syncthreads();
    for (int i = threadIdx.x; i < np * 2; i += blockDim.x) {
        double s = 0.0;
        for (int w = 0; w < nwarps; ++w) s += s_acc[w * np * 2 + i];
        ra.partials[static_cast<size_t>(blockIdx.x) * np * 2 + i] = static_cast<float>(s);
    }
    __threadfence();
    __syncthreads();
    __shared__ unsigned int s_last;
    if (threadIdx.x == 0) s_last = (atomicAdd(ra.ticket, 1u) == gridDim.x - 1) ? 1u : 0u;
    __syncthreads();
    if (!s_last) return;
    __threadfence();
    // Sums of all blocks' partials in FP64, in a fixed order (deterministic):
    // few payoffs: one warp per payoff, its lanes striding over the blocks;
    // many payoffs: one thread per payoff, over the blocks in order (each
    // block's row of partials is then read coalesced across the threads).
    const int nb = gridDim.x;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    (void)s_red;
    const bool wide = np >= 32;
    const int first = wide ? static_cast<int>(threadIdx.x) : warp;
    const int stride = wide ? static_cast<int>(blockDim.x) : nwarps;
    for (int p = first; p < np; p += stride) {
        KahanSum k0, k1;
        double t0, t1;
        if (wide) {
#pragma unroll 4
            for (int b = 0; b < nb; ++b) {
                const float2 q = *reinterpret_cast<const float2 *>(ra.partials + static_cast<size_t>(b) * np * 2 + p * 2);
                k0.add(static_cast<double>(q.x));
                k1.add(static_cast<double>(q.y));
            }
            t0 = k0.s;
            t1 = k1.s;
        } else {
            for (int b = lane; b < nb; b += 32) {
                const float *q = ra.partials + static_cast<size_t>(b) * np * 2 + p * 2;
                k0.add(static_cast<double>(q[0]));
                k1.add(static_cast<double>(q[1]));
            }
            // the 32 lanes' compensated sums, then a pairwise (shuffle tree) sum
            t0 = warp_sum_d(k0.s - k0.c);
            t1 = warp_sum_d(k1.s - k1.c);
        }
        if (wide || lane == 0) {
            const bool bad = ra.err && *reinterpret_cast<const volatile unsigned int *>(ra.err) != 0u;
            const double N = static_cast<double>(ra.paths);
            const double mean = t0 / N, m2 = t1 / N;
            const double var = fmax(m2 - mean * mean, 0.0);
            mc_result res;
            res.price = bad ? __longlong_as_double(0x7ff8000000000000ll) : ra.disc * mean;
            res.se = bad ? res.price : (ra.paths > 1 ? ra.disc * sqrt(var / (N - 1.0)) : 0.0);
            ra.out[p] = res;
        }
    }
    if (threadIdx.x == 0) *ra.ticket = 0u;
}

}  // namespace gbmc

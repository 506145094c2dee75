// nested.cu -- the nested ("brute force") Solvency II valuation on sm_103a.
//
// Tucker & Bull (Section 2) value every policy under 1000 Monte Carlo
// scenarios at each future valuation node and take the 5th largest of the
// 1000 liabilities as the 99.5% value.  Here, for outer Vasicek paths o,
// nodes n at months m_n = n * node_step and inner paths i started from the
// outer path's short rate at the node:
//
//   L_{o,n,i} = sum_p amount_p sum_j pi_{p,n,j} r_{p,j}(node; inner path i)
//
// where pi_{p,n,j} is the probability that policy p is in reduced state j at
// the node (deterministic mortality) and r_{p,j} the reserve at the node on the
// inner path's discount factors.  The reserve is linear in the discount products
// (Eq. basicReserveSummation), so this is the value at the node of the
// portfolio's expected cash flows after it (cashflow.cuh).
//
// Random numbers: Philox4x32-10 (Salmon et al., SC'11), counter (k, c1, c2,
// c3), key (seed lo, seed hi); step 2k takes words 0,1 and step 2k+1 words
// 2,3 as uniforms (w + 1/2) 2^-32, Box-Muller in FP64 (the inner paths
// with table-driven logarithm, sine and cosine, and a series for the
// month's discount factor: below.  Outer path o:
// (k, o, 0, 2 << 24); inner path (o, n, i): (k, i, n, (3 << 24) | o).
// Vasicek exact monthly step of (r, integral of r) (Glasserman 2004 3.3.1);
// v = exp(-integral) goes into the path's discount product at once.
#include <algorithm>
#include <cmath>
#include <cstring>
#include <vector>

#include "fp64_series.cuh"
#include "nested.cuh"
#include "philox.cuh"
#include "rsv_device.cuh"
#include "rsv.h"
#include "abi_guard.cuh"

namespace rsv {

// ------------------------------------------------------------ generator ----
VasStep vasicek_step_constants(double a, double b, double sigma, double dt) {
    VasStep s;
    const double one_m_e = -std::expm1(-a * dt), one_m_e2 = -std::expm1(-2.0 * a * dt);
    const double var_r = sigma * sigma * one_m_e2 / (2.0 * a);
    const double var_i = sigma * sigma / (a * a) * (dt - 2.0 * one_m_e / a + one_m_e2 / (2.0 * a));
    const double cov = sigma * sigma / (2.0 * a * a) * one_m_e * one_m_e;
    s.e = std::exp(-a * dt);
    s.k1 = one_m_e / a;
    s.l11 = std::sqrt(var_r);
    s.l21 = s.l11 > 0 ? cov / s.l11 : 0.0;
    s.l22 = std::sqrt(std::max(var_i - s.l21 * s.l21, 0.0));
    s.b = b;
    s.dt = dt;
    return s;
}

// Host tables of the Box-Muller step (see nested.cuh).
const double2* bm_tables_host() {
    static const std::vector<double2> t = [] {
        std::vector<double2> v(BM_SC + BM_LG);
        const long double two_pi = 6.283185307179586476925286766559005768L;
        for (int j = 0; j < BM_SC; ++j) {
            const long double x = two_pi * j / BM_SC;
            v[j] = make_double2((double)std::sin(x), (double)std::cos(x));
        }
        for (int j = 0; j < BM_LG; ++j) {
            const double c = 1.0 + (j + 0.5) / BM_LG;
            const double inv = std::ldexp(std::nearbyint(std::ldexp(1.0 / c, 18)), -18);
            const int k = j >= BM_LG_K0 ? 1 : 0;
            v[BM_SC + j] = make_double2(inv, (double)(-std::log(std::ldexp((long double)inv, k))));
        }
        return v;
    }();
    return t.data();
}

constexpr double kLn2 = 0.6931471805599453094;
constexpr double kTwoPi32 = 6.283185307179586477 / 4294967296.0;   // 2 pi 2^-32 (a power-of-two scaling of 2 pi)

// ln u for the uniform u = (w + 1/2) 2^-32 by Tang's table-driven method in
// FP64: w + 1/2 = 2^e y with y in [1, 2); interval j = the top 7 bits of y's
// mantissa; r = y inv_j - 1 is exact (inv_j has 18 significant bits, y at
// most 33) and |r| < 2^-8; ln u = (e + k_j - 32) ln 2 + L_j + log1p(r) with
// L_j = -ln(2^k_j inv_j), k_j = 1 above sqrt 2, and log1p by its Taylor
// series to r^7 (remainder below 2^-60 r).  For u >= 1 - 2^-8, where L_j and
// log1p(r) would cancel, r = u - 1 (exact) and ln u = log1p(r).
__device__ __forceinline__ double bm_log_u(uint32_t w, const double2* __restrict__ lg) {
    const double m = (double)w + 0.5;
    const int e = w ? 31 - __clz((int)w) : -1;
    const double y = m * __longlong_as_double((long long)(1023 - e) << 52);
    const int j = (int)((__double_as_longlong(y) >> 45) & (BM_LG - 1));
    const double2 t = lg[j];
    const bool near1 = w >= 0xFF000000u;
    const double r = near1 ? __dmul_rn(__dadd_rn(m, -4294967296.0), 0x1.0p-32) : __fma_rn(y, t.x, -1.0);
    double q = __fma_rn(r, 1.0 / 7.0, -1.0 / 6.0);
    q = __fma_rn(r, q, 1.0 / 5.0);
    q = __fma_rn(r, q, -0.25);
    q = __fma_rn(r, q, 1.0 / 3.0);
    q = __fma_rn(r, q, -0.5);
    const double p = __fma_rn(__dmul_rn(r, r), q, r);
    const int k = j >= BM_LG_K0 ? 1 : 0;
    return near1 ? p : __fma_rn((double)(e + k - 32), kLn2, __dadd_rn(t.y, p));
}

// (sin, cos)(2 pi u) for u = (w + 1/2) 2^-32: the top 10 bits of w pick
// alpha = 2 pi j / 1024 from the table, the rest give beta = 2 pi f with
// 0 <= beta < 2 pi / 1024; sin beta and cos beta - 1 by their Taylor series
// (to beta^5 and beta^6: remainders below 1e-19), then the addition theorems.
__device__ __forceinline__ void bm_sincos_2pi_u(uint32_t w, const double2* __restrict__ sc, double& sn, double& cs) {
    const double2 t = sc[w >> 22];
    const double b = __dmul_rn(__dadd_rn((double)(w & 0x3FFFFFu), 0.5), kTwoPi32);
    const double b2 = __dmul_rn(b, b);
    const double sb = __fma_rn(__dmul_rn(b2, b), __fma_rn(b2, 1.0 / 120.0, -1.0 / 6.0), b);
    const double cm1 = __dmul_rn(b2, __fma_rn(b2, __fma_rn(b2, -1.0 / 720.0, 1.0 / 24.0), -0.5));
    sn = __fma_rn(t.y, sb, __fma_rn(t.x, cm1, t.x));
    cs = __fma_rn(-t.x, sb, __fma_rn(t.y, cm1, t.y));
}

// One path: n_steps monthly steps from rate r; calls `emit(t, v_t)`.  `bm`
// holds the Box-Muller tables (BM_SC sine/cosine entries, then BM_LG
// logarithm entries).
template <class Emit>
__device__ __forceinline__ double vasicek_path(const VasStep& s, uint64_t seed, uint32_t c1, uint32_t c2,
                                               uint32_t c3, double r, int n_steps, const double2* __restrict__ bm,
                                               Emit emit) {
    const uint32_t k0 = (uint32_t)seed, k1 = (uint32_t)(seed >> 32);
    const double bdt = s.b * s.dt;
    for (int t = 0; t < n_steps; t += 2) {
        uint32_t w[4];
        philox4x32_10((uint32_t)(t >> 1), c1, c2, c3, k0, k1, w);
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            if (t + h >= n_steps) break;
            const double R = sqrt(-2.0 * bm_log_u(w[2 * h], bm + BM_SC));
            double sn, cs;
            bm_sincos_2pi_u(w[2 * h + 1], bm, sn, cs);
            const double z1 = R * cs, z2 = R * sn;
            const double dr = r - s.b;
            const double I = __fma_rn(s.l22, z2, __fma_rn(s.l21, z1, __fma_rn(dr, s.k1, bdt)));
            r = __fma_rn(s.l11, z1, __fma_rn(dr, s.e, s.b));
            emit(t + h, exp_small(-I), r);
        }
    }
    return r;
}

// Outer paths, one warp each.  The draws of a step depend only on its
// counter, so the lanes take 32 consecutive steps at once; the rate update
// r_{t+1} = e r_t + c_t (c_t = b (1 - e) + l11 z1_t) is affine with a common
// multiplier, so a warp scan of the maps gives every lane the rate at the
// start of its step, and a product scan the discount to its end.  The same
// path as the serial recursion up to the order of rounding.
__global__ void outer_paths_kernel(VasStep s, uint64_t seed, int o_first, int n_outer, int n_nodes, int node_step,
                                   double r0, double* __restrict__ r_node, double* __restrict__ d0) {
    const int lane = threadIdx.x & 31;
    const int o = (int)((blockIdx.x * (size_t)blockDim.x + threadIdx.x) >> 5);
    if (o >= n_outer) return;   // whole warps leave together
    const uint32_t k0 = (uint32_t)seed, k1 = (uint32_t)(seed >> 32);
    const double inv32 = 2.3283064365386963e-10;   // 2^-32
    const int n_steps = (n_nodes - 1) * node_step;
    if (lane == 0) {
        r_node[(size_t)o * n_nodes] = r0;
        d0[(size_t)o * n_nodes] = 1.0;
    }
    double r = r0, D = 1.0;   // at the start of the block of 32 steps
    for (int t0 = 0; t0 < n_steps; t0 += 32) {
        const int t = t0 + lane;
        const bool live = t < n_steps;
        double z1 = 0.0, z2 = 0.0;
        if (live) {   // the serial generator's draw for step t
            uint32_t w[4];
            philox4x32_10((uint32_t)(t >> 1), (uint32_t)(o_first + o), 0u, 2u << 24, k0, k1, w);
            const int h = t & 1;
            const double u1 = ((double)w[2 * h] + 0.5) * inv32;
            const double u2 = ((double)w[2 * h + 1] + 0.5) * inv32;
            const double R = sqrt(-2.0 * log(u1));
            double sn, cs;
            sincospi(2.0 * u2, &sn, &cs);
            z1 = R * cs;
            z2 = R * sn;
        }
        // inclusive scan of the maps x -> A x + B over the lanes: A = e^(lane+1)
        double A = s.e, B = live ? s.b * (1.0 - s.e) + s.l11 * z1 : 0.0;
        if (!live) A = 1.0;   // identity past the end
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) {
            const double Au = __shfl_up_sync(0xffffffffu, A, d), Bu = __shfl_up_sync(0xffffffffu, B, d);
            if (lane >= d) {   // this map after the lower lanes' composition
                B = A * Bu + B;
                A = A * Au;
            }
        }
        // the rate at the start of step t: the exclusive prefix applied to r
        double Ae = __shfl_up_sync(0xffffffffu, A, 1), Be = __shfl_up_sync(0xffffffffu, B, 1);
        if (lane == 0) {
            Ae = 1.0;
            Be = 0.0;
        }
        const double rt = Ae * r + Be;
        const double I = s.b * s.dt + (rt - s.b) * s.k1 + s.l21 * z1 + s.l22 * z2;
        double v = live ? exp(-I) : 1.0;
        // inclusive product scan of the discount factors
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) {
            const double vu = __shfl_up_sync(0xffffffffu, v, d);
            if (lane >= d) v *= vu;
        }
        const double r_after = A * r + B, D_after = D * v;
        if (live && (t + 1) % node_step == 0) {
            const int nd = (t + 1) / node_step;
            r_node[(size_t)o * n_nodes + nd] = r_after;
            d0[(size_t)o * n_nodes + nd] = D_after;
        }
        r = __shfl_sync(0xffffffffu, r_after, 31);
        D = __shfl_sync(0xffffffffu, D_after, 31);
    }
}

// ------------------------------------------------------------ inner paths ----
// One thread values one inner path while it generates it:
//   L_{o,n,i} = due[m] + sum_tau D(tau + 1) flow[m + tau],   m = n node_step,
// with the discount product D carried along the path and the portfolio's
// expected cash flows from cashflow.cuh.  The sum over the policies is inside
// flow: with deterministic mortality the pi-weighted reserve at the node is the
// value of the expected cash flows after it, so a path costs its random walk and one
// multiply-add per month however large the book is, and no discount factor is
// written to memory.  Paths of a node are packed into blocks over the outer
// paths, the blocks run node-major, longest remaining projections first.
constexpr int kPathNT = 128;

struct PathArgs {
    uint64_t seed;
    int32_t o_first, n_outer, n_nodes, node_step, n_inner, n_steps;   // n_steps: the portfolio's longest projection
    const double* r_node;
    const void* tables;    // Box-Muller tables of the generator
    const double* flow;
    const float2* flow2;   // flow / scale[0], FP32 head and tail
    const double* scale;
    const double* due;
    double* L_all;
};

template <class Path>
__device__ __forceinline__ void for_each_path(const PathArgs& a, Path path) {
    const long long per_node = (long long)a.n_outer * a.n_inner, blocks = (per_node + kPathNT - 1) / kPathNT;
    for (long long b = blockIdx.x; b < blocks * a.n_nodes; b += gridDim.x) {
        const int n = (int)(b / blocks);
        const long long k = (b - n * blocks) * kPathNT + threadIdx.x;
        if (k >= per_node) continue;
        const int o = (int)(k / a.n_inner), i = (int)(k - (long long)o * a.n_inner);
        const int m = n * a.node_step, left = max(0, a.n_steps - m);
        const double r = a.r_node[(size_t)o * a.n_nodes + n];
        const double now = m <= a.n_steps ? a.due[m] : 0.0;
        a.L_all[((size_t)o * a.n_nodes + n) * a.n_inner + i] =
            now + path((uint32_t)i, (uint32_t)n, (3u << 24) | (uint32_t)(a.o_first + o), r, m, left);
    }
}

// FP64 throughout (all forms but the deflated one, and model parameters outside
// the double-float generator's range): bound by the FP64 pipe, about 55
// operations a month.  Before, the discount factors went through a plane in memory to a
// valuation kernel that ran every policy on them: 331 mixed policies x 8 outer
// paths x 25 nodes x 1,000 inner paths, compensated, 60.4 ms, now 23.4 ms.
__global__ void __launch_bounds__(kPathNT) inner_paths_kernel(const VasStep s, const PathArgs a) {
    __shared__ double2 bm[BM_SC + BM_LG];   // 18 KiB: the Box-Muller tables
    for (int k = threadIdx.x; k < BM_SC + BM_LG; k += blockDim.x) bm[k] = static_cast<const double2*>(a.tables)[k];
    __syncthreads();
    for_each_path(a, [&](uint32_t c1, uint32_t c2, uint32_t c3, double r, int m, int left) {
        const double* __restrict__ flow = a.flow + m;
        double D = 1.0, L = 0.0;
        vasicek_path(s, a.seed, c1, c2, c3, r, left, bm, [&](int t, double v, double) {
            D = __dmul_rn(D, v);
            L = __fma_rn(D, __ldg(flow + t), L);
        });
        return L;
    });
}

// ---- the generator in double-float FP32 -------------------------------------
// GB300 issues 64 FP32 operations in the time of one FP64 operation, so the
// walk runs in double-floats (about 2^-46 a step), with the random words and the
// argument reductions in integers, which keeps them exact:
//   ln u:  u = (2 w + 1) 2^-33 = 2^(-1-lz) y, y in [1, 2) with 32 fraction bits;
//          r = y inv_j - 1 exactly as an integer (inv_j: 18 bits), split into two
//          exact floats; log1p(r) = r - r^2/2 + r^3 (1/3 - r/4 + r^2/5), the square as a
//          double-float (|r| < 2^-8: the next term is below 2^-50);
//   R = sqrt(-2 ln u): the hardware reciprocal square root and one Newton step
//          with the exact residual;
//   sin, cos of 2 pi u: the nearest of 1,024 table angles (at the intervals'
//          middles) and the addition theorems with |b| < pi/1024;
//   x' = e x + l11 z1 (x = r - b), and 1 - I = (1 - b dt) - k1 x - l21 z1 - l22 z2
//          by fused multiply-adds onto a head near 1, whose rounding errors a second
//          fused multiply-add recovers exactly; exp(-I) from 1 - I by its series
//          to I^6;
//   D *= exp(-I);  L += D flow (product and sum error-free).
// The deflated form takes it: its liabilities are within 1.2e-11 of 64 bits (its own
// bound is 9e-7; its planes gave 1.6e-8).  2,000 annuities x 100 outer paths x 40
// nodes x 1,000 inner paths: 203 ms by the FP64 walk, 12.9 ms so; about 220
// instructions a month, issue 80% busy, FMA pipe 63%.
struct NzStep {
    float2 e, l11, k1, l21, l22, q0;   // constants as FP32 head and tail; q0 = 1 - b dt
};

constexpr int NZ_SC = 1024, NZ_LG = 128;   // float4 entries: (sin, cos) pairs, then (inv_j, L_j, k_j - 1)
constexpr float kLn2Head = 0.693145751953125f;          // ln 2 to 18 bits, so that small integers times it are exact
constexpr float kLn2Tail = 1.42860682030941723e-6f;
constexpr float kPi32Head = 7.314590396335798e-10f, kPi32Tail = -2.035470213827790e-17f;   // pi 2^-32

__device__ __forceinline__ void fast_two_sum(float a, float b, float& s, float& e) {
    s = __fadd_rn(a, b);
    e = __fsub_rn(b, __fsub_rn(s, a));
}
__device__ __forceinline__ void two_sum(float a, float b, float& s, float& e) {
    s = __fadd_rn(a, b);
    const float bb = __fsub_rn(s, a);
    e = __fadd_rn(__fsub_rn(a, __fsub_rn(s, bb)), __fsub_rn(b, bb));
}
// s = c + a b rounded, e its rounding error (|c| >= |a b|: c - s is exact)
__device__ __forceinline__ void fma_err(float a, float b, float c, float& s, float& e) {
    s = __fmaf_rn(a, b, c);
    e = __fmaf_rn(a, b, __fsub_rn(c, s));
}
__device__ __forceinline__ uint32_t shl_clamped(uint32_t x, uint32_t n) {   // 0 for n >= 32
    uint32_t r;
    asm("shl.b32 %0, %1, %2;" : "=r"(r) : "r"(x), "r"(n));
    return r;
}
__device__ __forceinline__ float rsqrt_hw(float x) {
    float r;
    asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
}

// R = sqrt(-2 ln u), u = (w + 1/2) 2^-32
__device__ __forceinline__ df nz_radius(uint32_t w, const float4* __restrict__ lg) {
    const uint32_t lz = (uint32_t)__clz((int)w);   // 32 for w = 0
    const uint32_t y = (shl_clamped(w, lz) << 1) + shl_clamped(1u, lz);   // fraction bits of 2 w + 1, normalised
    const float4 t = lg[y >> 25];
    const uint32_t inv = __float_as_uint(t.x);
    const uint64_t prod = (uint64_t)y * inv;
    const int hi = (int)(uint32_t)(prod >> 32) + (int)inv - (1 << 18);
    const uint32_t lo = (uint32_t)prod;               // r = (hi 2^32 + lo) 2^-50
    const int a = (hi << 12) | (int)(lo >> 20);       // |a| < 2^22
    const float rh = __fmaf_rn(__int_as_float(0x4B400000 + a), 0x1p-30f, -12582912.0f * 0x1p-30f);
    const float rl = __fmaf_rn(__uint_as_float(0x4B000000u | (lo & 0xFFFFFu)), 0x1p-50f, -8388608.0f * 0x1p-50f);
    const float p = __fmul_rn(rh, rh);
    const float pe = __fmaf_rn(rh, __fadd_rn(rl, rl), __fmaf_rn(rh, rh, -p));
    const float c3 = __fmul_rn(__fmul_rn(p, rh), __fmaf_rn(rh, __fmaf_rn(rh, 0.2f, -0.25f), 0.333333343f));
    const float E = __fsub_rn(t.w, __int2float_rn((int)lz));   // k_j - 1 - lz
    float s1, e1, s2, e2, s3, e3;
    fast_two_sum(__fmul_rn(E, kLn2Head), t.y, s1, e1);
    fast_two_sum(s1, rh, s2, e2);
    two_sum(s2, __fmul_rn(-0.5f, p), s3, e3);
    float tail = __fadd_rn(__fmaf_rn(E, kLn2Tail, t.z), rl);
    tail = __fadd_rn(__fadd_rn(tail, __fadd_rn(e1, e2)), __fadd_rn(e3, c3));
    tail = __fmaf_rn(-0.5f, pe, tail);
    const float lh = __fadd_rn(s3, tail);
    const float ll = __fsub_rn(tail, __fsub_rn(lh, s3));
    const float ah = __fmul_rn(-2.0f, lh);
    const float q = rsqrt_hw(ah), s = __fmul_rn(ah, q);
    const float res = __fmaf_rn(-2.0f, ll, __fmaf_rn(-s, s, ah));
    return df{s, __fmul_rn(res, __fmul_rn(0.5f, q))};
}

// (sin, cos)(2 pi u), u = (w + 1/2) 2^-32
__device__ __forceinline__ void nz_sincos(uint32_t w, const float4* __restrict__ sc, df& sn, df& cs) {
    const float4 t = sc[w >> 22];   // sin and cos of 2 pi (j + 1/2) / 1024, head and tail
    const float F = __fsub_rn(__uint_as_float(0x4B000001u | ((w << 1) & 0x7FFFFEu)), 12582912.0f);
    const float b = __fmul_rn(F, kPi32Head);
    float bl = __fmaf_rn(F, kPi32Tail, __fmaf_rn(F, kPi32Head, -b));
    const float b2 = __fmul_rn(b, b);
    bl = __fmaf_rn(__fmul_rn(b2, b), -0.166666672f, bl);                          // sin b = b + bl
    const float cm = __fmul_rn(b2, __fmaf_rn(b2, 0.0416666679f, -0.5f));          // cos b - 1
    float p = __fmul_rn(t.z, b), e = __fmaf_rn(t.z, b, -p), s, es;
    fast_two_sum(t.x, p, s, es);
    e = __fadd_rn(__fadd_rn(e, es), t.y);
    e = __fmaf_rn(t.z, bl, e);
    e = __fmaf_rn(t.w, b, e);
    sn = df{s, __fmaf_rn(t.x, cm, e)};
    p = __fmul_rn(-t.x, b), e = __fmaf_rn(-t.x, b, -p);
    fast_two_sum(t.z, p, s, es);
    e = __fadd_rn(__fadd_rn(e, es), t.w);
    e = __fmaf_rn(-t.x, bl, e);
    e = __fmaf_rn(-t.y, b, e);
    cs = df{s, __fmaf_rn(t.z, cm, e)};
}

struct NzState {
    df x, D, L;   // r - b, the discount product from the node, the liability / scale
};

__device__ __forceinline__ void nz_step(NzState& q, const NzStep& s, uint32_t w0, uint32_t w1, float2 c,
                                        const float4* __restrict__ tb) {
    const df R = nz_radius(w0, tb + NZ_SC);
    df sn, cs;
    nz_sincos(w1, tb, sn, cs);
    const df z1 = df_mul(R, cs), z2 = df_mul(R, sn);
    // 1 - I
    float r1, r2, r3, t1, t2, t3;
    fma_err(-s.k1.x, q.x.h, s.q0.x, r1, t1);
    fma_err(-s.l21.x, z1.h, r1, r2, t2);
    fma_err(-s.l22.x, z2.h, r2, r3, t3);
    float tl = __fadd_rn(__fadd_rn(t1, s.q0.y), __fadd_rn(t2, t3));
    tl = __fmaf_rn(-s.k1.x, q.x.l, tl);
    tl = __fmaf_rn(-s.k1.y, q.x.h, tl);
    tl = __fmaf_rn(-s.l21.x, z1.l, tl);
    tl = __fmaf_rn(-s.l21.y, z1.h, tl);
    tl = __fmaf_rn(-s.l22.x, z2.l, tl);
    tl = __fmaf_rn(-s.l22.y, z2.h, tl);
    // x' = e x + l11 z1
    const float ph = __fmul_rn(s.e.x, q.x.h), zh = __fmul_rn(s.l11.x, z1.h);
    float pe = __fmaf_rn(s.e.x, q.x.h, -ph), ze = __fmaf_rn(s.l11.x, z1.h, -zh), xh, xe;
    pe = __fmaf_rn(s.e.y, q.x.h, __fmaf_rn(s.e.x, q.x.l, pe));
    ze = __fmaf_rn(s.l11.y, z1.h, __fmaf_rn(s.l11.x, z1.l, ze));
    two_sum(ph, zh, xh, xe);
    const float xl = __fadd_rn(xe, __fadd_rn(pe, ze));
    q.x.h = __fadd_rn(xh, xl);
    q.x.l = __fsub_rn(xl, __fsub_rn(q.x.h, xh));
    // v = exp(-I) = (1 - I) + I^2/2 - I^3/6 + ..., I = i - tl with i = 1 - r3 exact
    const float i = __fsub_rn(1.0f, r3);
    const float i2 = __fmul_rn(i, i), i2e = __fmaf_rn(i, i, -i2);
    const float poly = __fmaf_rn(i, __fmaf_rn(i, __fmaf_rn(i, 1.0f / 720.0f, -1.0f / 120.0f), 1.0f / 24.0f), -1.0f / 6.0f);
    float vh, ve;
    fast_two_sum(r3, __fmul_rn(0.5f, i2), vh, ve);
    const float vl = __fadd_rn(__fmaf_rn(-i, tl, __fadd_rn(tl, ve)),
                               __fmaf_rn(0.5f, i2e, __fmul_rn(__fmul_rn(i2, i), poly)));
    const df D = df_mul(q.D, df{vh, vl});
    q.D.h = __fadd_rn(D.h, D.l);
    q.D.l = __fsub_rn(D.l, __fsub_rn(q.D.h, D.h));
    // L += D c
    const float g = __fmul_rn(c.x, q.D.h);
    float ge = __fmaf_rn(c.x, q.D.h, -g), lh, le;
    ge = __fmaf_rn(c.y, q.D.h, __fmaf_rn(c.x, q.D.l, ge));
    two_sum(q.L.h, g, lh, le);
    le = __fadd_rn(__fadd_rn(q.L.l, ge), le);
    q.L.h = __fadd_rn(lh, le);
    q.L.l = __fsub_rn(le, __fsub_rn(q.L.h, lh));
}

__global__ void __launch_bounds__(kPathNT) inner_paths_df_kernel(const NzStep s, double b, const PathArgs a) {
    __shared__ float4 tb[NZ_SC + NZ_LG];   // 18 KiB
    for (int k = threadIdx.x; k < NZ_SC + NZ_LG; k += blockDim.x) tb[k] = static_cast<const float4*>(a.tables)[k];
    __syncthreads();
    const uint32_t k0 = (uint32_t)a.seed, k1 = (uint32_t)(a.seed >> 32);
    const double scale = a.scale[0];
    for_each_path(a, [&](uint32_t c1, uint32_t c2, uint32_t c3, double r, int m, int left) {
        const float2* __restrict__ flow = a.flow2 + m;
        const double x = r - b;
        NzState q;
        q.x.h = __double2float_rn(x);
        q.x.l = __double2float_rn(x - (double)q.x.h);
        q.D = df{1.0f, 0.0f};
        q.L = df{0.0f, 0.0f};
        for (int t = 0; t < left; t += 2) {
            uint32_t w[4];
            philox4x32_10((uint32_t)(t >> 1), c1, c2, c3, k0, k1, w);
            nz_step(q, s, w[0], w[1], __ldg(flow + t), tb);
            if (t + 1 < left) nz_step(q, s, w[2], w[3], __ldg(flow + t + 1), tb);
        }
        return ((double)q.L.h + (double)q.L.l) * scale;
    });
}

// The curve mode: L_{o,n} on the Vasicek forward curve of the node's rate, whose
// discount products are the zero-coupon prices P(tau + 1 | r) = exp(A - B r); A and B
// depend on the maturity alone (curve_ab), so a month costs one exponential.
// One warp a (node, outer path), the lanes over the months, a fixed-order sum.
__global__ void curve_ab_kernel(double a, double b, double sigma, double dt, int n_steps, double2* __restrict__ ab) {
    const int t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= n_steps) return;
    const double T = (t + 1) * dt;
    ab[t] = make_double2(vasicek_lnP(T, 0.0, a, b, sigma), -expm1(-a * T) / a);
}

__global__ void curve_value_kernel(const PathArgs a, const double2* __restrict__ ab) {
    const int lane = threadIdx.x & 31;
    const long long k = ((long long)blockIdx.x * blockDim.x + threadIdx.x) >> 5;   // node-major
    if (k >= (long long)a.n_outer * a.n_nodes) return;                            // whole warps leave together
    const int n = (int)(k / a.n_outer), o = (int)(k - (long long)n * a.n_outer);
    const int m = n * a.node_step, left = max(0, a.n_steps - m);
    const double r = a.r_node[(size_t)o * a.n_nodes + n];
    double L = 0.0;
    for (int t = lane; t < left; t += 32) L = __fma_rn(exp(__fma_rn(-ab[t].y, r, ab[t].x)), a.flow[m + t], L);
#pragma unroll
    for (int d = 16; d > 0; d >>= 1) L += __shfl_xor_sync(0xffffffffu, L, d);
    if (lane == 0) a.L_all[(size_t)o * a.n_nodes + n] = (m <= a.n_steps ? a.due[m] : 0.0) + L;
}

// Mean and k-th largest over the inner paths of each (o, n), one CTA each.
// The k-th largest is found by descending thresholds: the largest value
// below the current threshold and its multiplicity, until k values are
// covered, so ties need no special care.
__global__ void node_stats_kernel(const double* __restrict__ L_all, int n_inner, int k, double* __restrict__ mean,
                                  double* __restrict__ kth) {
    __shared__ double sd[256];
    __shared__ int si[256];
    const size_t on = blockIdx.x;
    const double* x = L_all + on * n_inner;
    double s = 0.0;
    for (int i = threadIdx.x; i < n_inner; i += blockDim.x) s += x[i];
    sd[threadIdx.x] = s;
    __syncthreads();
    for (int w = blockDim.x / 2; w > 0; w >>= 1) {
        if (threadIdx.x < w) sd[threadIdx.x] += sd[threadIdx.x + w];
        __syncthreads();
    }
    if (threadIdx.x == 0) mean[on] = sd[0] / n_inner;
    __syncthreads();
    double thr = INFINITY;
    int left = k;
    for (int round = 0; round < k; ++round) {
        double mx = -INFINITY;
        for (int i = threadIdx.x; i < n_inner; i += blockDim.x)
            if (x[i] < thr) mx = fmax(mx, x[i]);
        sd[threadIdx.x] = mx;
        __syncthreads();
        for (int w = blockDim.x / 2; w > 0; w >>= 1) {
            if (threadIdx.x < w) sd[threadIdx.x] = fmax(sd[threadIdx.x], sd[threadIdx.x + w]);
            __syncthreads();
        }
        const double m = sd[0];
        __syncthreads();
        int c = 0;
        for (int i = threadIdx.x; i < n_inner; i += blockDim.x) c += (x[i] == m);
        si[threadIdx.x] = c;
        __syncthreads();
        for (int w = blockDim.x / 2; w > 0; w >>= 1) {
            if (threadIdx.x < w) si[threadIdx.x] += si[threadIdx.x + w];
            __syncthreads();
        }
        const int cnt = si[0];
        __syncthreads();
        if (cnt >= left || m == -INFINITY) {
            if (threadIdx.x == 0) kth[on] = m;
            break;
        }
        left -= cnt;
        thr = m;
    }
}

// ------------------------------------------------------------- launchers ----
// Host tables of the double-float generator, as float4 (see nz_radius, nz_sincos).
static const float4* nz_tables_host() {
    static const std::vector<float4> t = [] {
        std::vector<float4> v(NZ_SC + NZ_LG);
        const long double two_pi = 6.283185307179586476925286766559005768L;
        auto split = [](long double x, float& h, float& l) {
            h = (float)x;
            l = (float)(x - (long double)h);
        };
        for (int j = 0; j < NZ_SC; ++j) {
            const long double x = two_pi * (2 * j + 1) / (2 * NZ_SC);
            split(std::sin(x), v[j].x, v[j].y);
            split(std::cos(x), v[j].z, v[j].w);
        }
        for (int j = 0; j < NZ_LG; ++j) {
            const double c = 1.0 + (j + 0.5) / NZ_LG;
            const uint32_t inv = (uint32_t)std::nearbyint(std::ldexp(1.0 / c, 18));
            const int k = j >= BM_LG_K0 ? 1 : 0;
            float4& e = v[NZ_SC + j];
            memcpy(&e.x, &inv, sizeof inv);
            split(-std::log(std::ldexp((long double)inv, k - 18)), e.y, e.z);
            e.w = (float)(k - 1);
        }
        return v;
    }();
    return t.data();
}

// Tables of both generators, once per context: [FP64 | double-float].
size_t nested_table_bytes() { return (size_t)(BM_SC + BM_LG) * sizeof(double2) + (size_t)(NZ_SC + NZ_LG) * sizeof(float4); }
cudaError_t upload_nested_tables(void* dst, cudaStream_t st) {
    const size_t a = (size_t)(BM_SC + BM_LG) * sizeof(double2);
    cudaError_t e = cudaMemcpyAsync(dst, bm_tables_host(), a, cudaMemcpyHostToDevice, st);
    if (e != cudaSuccess) return e;
    return cudaMemcpyAsync(static_cast<char*>(dst) + a, nz_tables_host(), (size_t)(NZ_SC + NZ_LG) * sizeof(float4),
                           cudaMemcpyHostToDevice, st);
}

// The double-float generator holds rates as offsets from b and 1 - I near 1: the rates
// must stay within about 0.25 of b (ten standard deviations, so never seen) and
// b itself be moderate, so that a month's I stays below 0.05.
bool nested_df_range(const NestedRun& q) {
    const double sd = q.sigma * std::sqrt(std::min(1.0 / (2.0 * q.a), 800.0));
    return std::fabs(q.b) <= 0.25 && std::fabs(q.r0 - q.b) + 10.0 * sd <= 0.25;
}

cudaError_t launch_nested_paths(const VasStep& s, const NestedRun& q, bool use_df, cudaStream_t st) {
    const long long per_node = (long long)q.n_outer * q.n_inner;
    const long long blocks = (per_node + kPathNT - 1) / kPathNT * q.n_nodes;
    const int grid = (int)std::min<long long>(blocks, 0x7fffffffLL);
    PathArgs a{q.seed, q.o_first, q.n_outer, q.n_nodes, q.node_step, q.n_inner, q.n_steps,
               q.r_node, q.tables, q.flow, q.flow2, q.scale, q.due, q.L_all};
    if (!use_df) {
        inner_paths_kernel<<<grid, kPathNT, 0, st>>>(s, a);
    } else {
        auto two = [](double x) {
            const float h = (float)x;
            return make_float2(h, (float)(x - (double)h));
        };
        const NzStep z{two(s.e), two(s.l11), two(s.k1), two(s.l21), two(s.l22), two(1.0 - s.b * s.dt)};
        a.tables = static_cast<const char*>(q.tables) + (size_t)(BM_SC + BM_LG) * sizeof(double2);
        inner_paths_df_kernel<<<grid, kPathNT, 0, st>>>(z, s.b, a);
    }
    return cudaGetLastError();
}

cudaError_t launch_nested_curve(const NestedRun& q, double2* ab, cudaStream_t st) {
    PathArgs a{q.seed, q.o_first, q.n_outer, q.n_nodes, q.node_step, 1, q.n_steps,
               q.r_node, nullptr, q.flow, q.flow2, q.scale, q.due, q.L_all};
    if (q.n_steps > 0) curve_ab_kernel<<<(q.n_steps + 127) / 128, 128, 0, st>>>(q.a, q.b, q.sigma, 1.0 / 12.0, q.n_steps, ab);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    const long long warps = (long long)q.n_outer * q.n_nodes;
    curve_value_kernel<<<(unsigned)((warps + 3) / 4), 128, 0, st>>>(a, ab);
    return cudaGetLastError();
}

cudaError_t launch_outer_paths(const VasStep& s, uint64_t seed, int o_first, int n_outer, int n_nodes, int node_step, double r0,
                               double* r_node, double* d0, cudaStream_t st) {
    outer_paths_kernel<<<(n_outer + 3) / 4, 128, 0, st>>>(s, seed, o_first, n_outer, n_nodes, node_step, r0, r_node, d0);
    return cudaGetLastError();
}

// The generator's functions on given draws (a test entry point).
__global__ void generator_math_kernel(const uint32_t* __restrict__ w, const double* __restrict__ x, long long n,
                                      const double2* __restrict__ bm_g, double* __restrict__ out) {
    __shared__ double2 bm[BM_SC + BM_LG];
    for (int k = threadIdx.x; k < BM_SC + BM_LG; k += blockDim.x) bm[k] = bm_g[k];
    __syncthreads();
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
        double sn, cs;
        bm_sincos_2pi_u(w[i], bm, sn, cs);
        out[4 * i] = bm_log_u(w[i], bm + BM_SC);
        out[4 * i + 1] = sn;
        out[4 * i + 2] = cs;
        out[4 * i + 3] = exp_small(x[i]);
    }
}

cudaError_t launch_node_stats(const double* L_all, int n_on, int n_inner, int k, double* mean, double* kth,
                              cudaStream_t st) {
    if (n_on <= 0) return cudaSuccess;
    node_stats_kernel<<<n_on, 256, 0, st>>>(L_all, n_inner, k, mean, kth);
    return cudaGetLastError();
}

}  // namespace rsv

extern "C" rsv_status rsv_selftest_generator_math(int32_t device, void* cuda_stream, const uint32_t* w, const double* x,
                                                  int64_t n, double* out) try {
    if (n < 0 || (n > 0 && (!w || !x || !out))) return RSV_E_ARG;
    if (n == 0) return RSV_OK;
    cudaStream_t st = static_cast<cudaStream_t>(cuda_stream);
    if (cudaSetDevice(device) != cudaSuccess) return RSV_E_CUDA;
    uint32_t* dw = nullptr;
    double *dx = nullptr, *dout = nullptr;
    double2* dbm = nullptr;
    const size_t nb = (size_t)(rsv::BM_SC + rsv::BM_LG) * sizeof(double2);
    rsv_status rc = RSV_OK;
    if (cudaMalloc(&dw, (size_t)n * 4) != cudaSuccess || cudaMalloc(&dx, (size_t)n * 8) != cudaSuccess ||
        cudaMalloc(&dout, (size_t)n * 32) != cudaSuccess || cudaMalloc(&dbm, nb) != cudaSuccess) {
        rc = RSV_E_NOMEM;
    } else if (cudaMemcpyAsync(dw, w, (size_t)n * 4, cudaMemcpyHostToDevice, st) != cudaSuccess ||
               cudaMemcpyAsync(dx, x, (size_t)n * 8, cudaMemcpyHostToDevice, st) != cudaSuccess ||
               cudaMemcpyAsync(dbm, rsv::bm_tables_host(), nb, cudaMemcpyHostToDevice, st) != cudaSuccess) {
        rc = RSV_E_CUDA;
    } else {
        const int grid = (int)std::min<long long>((n + 127) / 128, 1024);
        rsv::generator_math_kernel<<<grid, 128, 0, st>>>(dw, dx, n, dbm, dout);
        if (cudaGetLastError() != cudaSuccess ||
            cudaMemcpyAsync(out, dout, (size_t)n * 32, cudaMemcpyDeviceToHost, st) != cudaSuccess ||
            cudaStreamSynchronize(st) != cudaSuccess)
            rc = RSV_E_CUDA;
    }
    cudaFree(dw);
    cudaFree(dx);
    cudaFree(dout);
    cudaFree(dbm);
    return rc;
} catch (...) {
    return rsv::host_error(nullptr);
}

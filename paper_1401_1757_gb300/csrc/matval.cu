// matval.cu -- digits of the discount products and of the expected cash flows, and
// their product on the tensor cores (see matval.cuh).
#include <cuda_bf16.h>
#include <cuda_fp16.h>

#include <algorithm>
#include <climits>
#include <cmath>

#include "launch_next.cuh"
#include "matval.cuh"
#include "tcgen05.cuh"

namespace rsv {
namespace {

constexpr uint32_t kMvPoll = 1u << 24;

__device__ __forceinline__ float pow2f(int e) { return __int_as_float(min(max(e + 127, 1), 254) << 23); }

// ------------------------------------------------------------- the digits ----
// Two numbers rounded to a digit's 16-bit type, and back.
template <int NS>
__device__ __forceinline__ uint32_t mv_pack(float x, float y) {
    if constexpr (NS == 3) {
        const __half2 v = __floats2half2_rn(x, y);
        return *reinterpret_cast<const uint32_t*>(&v);
    } else {
        const __nv_bfloat162 v = __floats2bfloat162_rn(x, y);
        return *reinterpret_cast<const uint32_t*>(&v);
    }
}
template <int NS>
__device__ __forceinline__ float2 mv_unpack(uint32_t d) {
    if constexpr (NS == 3) return __half22float2(*reinterpret_cast<const __half2*>(&d));
    else return make_float2(__uint_as_float(d << 16), __uint_as_float(d & 0xFFFF0000u));
}

// A form's digits are those of 2^kMvLog times the number.
template <int NS>
constexpr int kMvLog = NS == 3 ? 15 : 0;

// The digits of two numbers h + l in [0, 2^kMvLog] (the second in the high halves).
template <int NS>
__device__ __forceinline__ void mv_digits(float h0, float l0, float h1, float l1, uint32_t (&d)[NS]) {
    constexpr float M1 = 98304.0f * (NS == 3 ? 32768.0f : 1.0f);   // rounds to a multiple of 2^(kMvLog - 7)
    float a = __fsub_rn(__fadd_rn(h0, M1), M1), b = __fsub_rn(__fadd_rn(h1, M1), M1);
    float r = __fsub_rn(h0, a), s = __fsub_rn(h1, b);               // exact
    d[0] = mv_pack<NS>(a, b);
    if constexpr (NS != 3) {
#pragma unroll
        for (int k = 1; k < 3; ++k) {   // to a multiple of 2^-15, then of 2^-23
            const float M = k == 1 ? 384.0f : 1.5f;
            a = __fsub_rn(__fadd_rn(r, M), M), b = __fsub_rn(__fadd_rn(s, M), M);
            r = __fsub_rn(r, a), s = __fsub_rn(s, b);
            d[k] = mv_pack<NS>(a, b);
        }
    }
    r = __fadd_rn(r, l0), s = __fadd_rn(s, l1);
#pragma unroll
    for (int k = NS == 3 ? 1 : 3; k < NS; ++k) {
        d[k] = mv_pack<NS>(r, s);
        const float2 v = mv_unpack<NS>(d[k]);
        r = __fsub_rn(r, v.x), s = __fsub_rn(s, v.y);
    }
}

// The eight digits of a positive normal FP64 number a times 2^shift, in [0, 1], by integers:
// a 2^63 rounded down, split into balanced bytes (the leading one 7 bits); `sh` = the
// shift of the 53-bit mantissa.  0 for a = 0.
__device__ __forceinline__ unsigned long long mv_fixed64(double a, int shift) {
    const unsigned long long bits = (unsigned long long)__double_as_longlong(a);
    const int ex = (int)(bits >> 52);   // a >= 0
    if (ex == 0) return 0;
    const unsigned long long m = (bits & 0xFFFFFFFFFFFFFull) | 0x10000000000000ull;
    const int sh = ex - 1023 + 11 + shift;
    if (sh >= 0) return m << min(sh, 11);
    return sh > -64 ? m >> -sh : 0;
}
// digit k of two numbers as a pair of BF16 values (exact: 8 bits and sign)
__device__ __forceinline__ uint32_t mv_byte_pair(unsigned long long x, unsigned long long y, int k) {
    constexpr unsigned long long kHalf = 0x0080808080808080ull;   // half of each lower byte
    auto digit = [&](unsigned long long v) {
        const uint32_t byte = (uint32_t)((v + kHalf) >> (56 - 8 * k)) & 0xFF;
        const float d = __fsub_rn(__uint_as_float(0x4B000000u | byte), k ? 8388736.0f : 8388608.0f);
        return __float_as_uint(__fmul_rn(d, pow2f(-7 - 8 * k)));
    };
    return digit(x) >> 16 | (digit(y) & 0xFFFF0000u);
}

// ---------------------------------------------------------- scenario side ----
// Running products of 8 scenarios, the steps in 32 segments: a segment's product,
// the products before it, then the running product, so that the serial chain is 1/16
// of the steps.
constexpr int kProdS = 8;
__device__ __forceinline__ void put(double* p, double d) { *p = d; }
__device__ __forceinline__ void put(float2* p, double d) {
    const float h = __double2float_rn(d);
    *p = make_float2(h, __double2float_rn(d - (double)h));
}
template <class T>
__global__ void __launch_bounds__(kProdS * 32) mv_products_kernel(const double* __restrict__ v, int n_steps, int s_pad,
                                                                  T* __restrict__ D) {
    __shared__ double seg[32][kProdS];
    const int s = blockIdx.x * kProdS + threadIdx.x, k = threadIdx.y;
    const int len = (n_steps + 31) / 32, t0 = min(n_steps, k * len), t1 = min(n_steps, t0 + len);
    double p = 1.0;
#pragma unroll 4
    for (int t = t0; t < t1; ++t) p = __dmul_rn(p, v[(size_t)t * s_pad + s]);
    seg[k][threadIdx.x] = p;
    __syncthreads();
    double d = 1.0;
    for (int q = 0; q < k; ++q) d = __dmul_rn(d, seg[q][threadIdx.x]);
#pragma unroll 4
    for (int t = t0; t < t1; ++t) {
        d = __dmul_rn(d, v[(size_t)t * s_pad + s]);
        put(&D[(size_t)t * s_pad + s], d);
    }
}

// the binary exponent of a positive normal number, INT_MIN otherwise
__device__ __forceinline__ int exp_of(float x) {
    const int e = __float_as_int(x) >> 23;
    return e > 0 && e < 255 ? e - 127 : INT_MIN;
}

__global__ void mv_tilt_kernel(const float2* __restrict__ D, int n_scen, int s_pad, int32_t* __restrict__ tau,
                               int32_t* __restrict__ stat) {
    __shared__ float sum[128];
    const int t = blockIdx.x;
    float a = 0.0f;
    bool bad = false;
    for (int s = threadIdx.x; s < n_scen; s += 128) {
        const float x = D[(size_t)t * s_pad + s].x;
        if (exp_of(x) == INT_MIN) bad = true;
        else a += log2f(x);
    }
    sum[threadIdx.x] = a;
    bad = __syncthreads_or(bad);
    for (int w = 64; w > 0; w >>= 1) {
        if (threadIdx.x < w) sum[threadIdx.x] += sum[threadIdx.x + w];
        __syncthreads();
    }
    if (threadIdx.x == 0) {
        const int q = bad ? 0 : -(int)rintf(sum[0] / n_scen);
        tau[t] = q;
        atomicMax(&stat[1], bad ? INT_MAX : abs(q));
    }
}

// the largest and smallest exponents of the tilted products of 32 columns over 64 steps
__global__ void mv_columns_kernel(const float2* __restrict__ D, const int32_t* __restrict__ tau, int n_steps, int n_scen,
                                  int s_pad, int32_t* __restrict__ colmax, int32_t* __restrict__ colmin) {
    const int s = blockIdx.x * 32 + threadIdx.x;
    int mx = INT_MIN, mn = INT_MAX;
#pragma unroll
    for (int q = 0; q < 8; ++q) {
        const int t = blockIdx.y * 64 + q * 8 + threadIdx.y;
        const int e = t < n_steps ? exp_of(D[(size_t)t * s_pad + s].x) : INT_MIN;
        if (e == INT_MIN) continue;   // past the end, or recorded by the tilt kernel
        mx = max(mx, e + tau[t]);
        mn = min(mn, e + tau[t]);
    }
    if (s >= n_scen || mx < mn) return;
    atomicMax(&colmax[s], mx);
    atomicMin(&colmin[s], mn);
}

// Blocks but the last: the columns' exponents and spread.  The last: the tilt as a factor,
// 2^-tau(t), and its running maximum.
__global__ void __launch_bounds__(1024) mv_finish_kernel(const int32_t* __restrict__ tau, int n_steps, int n_scen, int s_pad,
                                                         int32_t* __restrict__ colexp, const int32_t* __restrict__ colmin,
                                                         int32_t* __restrict__ stat, float* __restrict__ tilt,
                                                         float* __restrict__ tilt_top) {
    if (blockIdx.x + 1 < gridDim.x) {
        const int s = blockIdx.x * 1024 + threadIdx.x;
        if (s >= s_pad) return;
        const int mx = colexp[s], mn = colmin[s];
        colexp[s] = s < n_scen && mx >= mn ? mx + 1 : 0;
        if (s < n_scen && mx >= mn) atomicMax(&stat[0], mx - mn);
        return;
    }
    __shared__ float top[1024];
    const int len = (n_steps + 1023) / 1024, t0 = min(n_steps, (int)threadIdx.x * len), t1 = min(n_steps, t0 + len);
    float m = 0.0f;
    for (int t = t0; t < t1; ++t) {
        const float x = pow2f(-tau[t]);
        tilt[t] = x;
        m = fmaxf(m, x);
    }
    top[threadIdx.x] = m;
    __syncthreads();
    for (int d = 1; d < 1024; d <<= 1) {
        const float o = threadIdx.x >= (unsigned)d ? top[threadIdx.x - d] : 0.0f;
        __syncthreads();
        top[threadIdx.x] = fmaxf(top[threadIdx.x], o);
        __syncthreads();
    }
    m = threadIdx.x ? top[threadIdx.x - 1] : 0.0f;
    for (int t = t0; t < t1; ++t) tilt_top[t] = m = fmaxf(m, tilt[t]);
}

template <int NS>
__global__ void __launch_bounds__(256) mv_digits_kernel(const float2* __restrict__ D, const int32_t* __restrict__ tau,
                                                        const int32_t* __restrict__ colexp, int n_steps, int n_scen,
                                                        int s_pad, int pitch, uint32_t* __restrict__ out) {
    __shared__ uint32_t tile[NS][32][33];   // pairs of steps
    const int s0 = blockIdx.x * 32, t0 = blockIdx.y * 64, s = s0 + (threadIdx.x & 31);
    const int c = colexp[s] - kMvLog<NS>;
    auto load = [&](int t) {
        if (t >= n_steps || s >= n_scen) return make_float2(0.0f, 0.0f);
        const float2 x = D[(size_t)t * s_pad + s];
        const float f = pow2f(tau[t] - c);
        return make_float2(__fmul_rn(x.x, f), __fmul_rn(x.y, f));
    };
    for (int q = threadIdx.x >> 5; q < 32; q += 8) {
        const float2 x = load(t0 + 2 * q), y = load(t0 + 2 * q + 1);
        uint32_t d[NS];
        mv_digits<NS>(x.x, x.y, y.x, y.y, d);
#pragma unroll
        for (int k = 0; k < NS; ++k) tile[k][threadIdx.x & 31][q] = d[k];
    }
    __syncthreads();
    for (int i = threadIdx.x; i < NS * 32 * 32; i += 256) {
        const int q = i & 31, r = (i >> 5) & 31, k = i >> 10;
        out[(((size_t)k * s_pad + s0 + r) * pitch + t0) / 2 + q] = tile[k][r][q];
    }
}

__global__ void __launch_bounds__(256) mv_digits64_kernel(const double* __restrict__ D, const int32_t* __restrict__ tau,
                                                          const int32_t* __restrict__ colexp, int n_steps, int n_scen,
                                                          int s_pad, int pitch, uint32_t* __restrict__ out) {
    __shared__ uint32_t tile[8][32][33];
    const int s0 = blockIdx.x * 32, t0 = blockIdx.y * 64, s = s0 + (threadIdx.x & 31);
    const int c = colexp[s];
    auto load = [&](int t) -> unsigned long long {
        return t < n_steps && s < n_scen ? mv_fixed64(D[(size_t)t * s_pad + s], tau[t] - c) : 0;
    };
    for (int q = threadIdx.x >> 5; q < 32; q += 8) {
        const unsigned long long x = load(t0 + 2 * q), y = load(t0 + 2 * q + 1);
#pragma unroll
        for (int k = 0; k < 8; ++k) tile[k][threadIdx.x & 31][q] = mv_byte_pair(x, y, k);
    }
    __syncthreads();
    for (int i = threadIdx.x; i < 8 * 32 * 32; i += 256) {
        const int q = i & 31, r = (i >> 5) & 31, k = i >> 10;
        out[(((size_t)k * s_pad + s0 + r) * pitch + t0) / 2 + q] = tile[k][r][q];
    }
}

// ------------------------------------------------------------ policy side ----
__device__ __forceinline__ df df_one_minus(df x) {   // 0 <= x <= 1
    const float s = __fsub_rn(1.0f, x.h);
    return df{s, __fsub_rn(__fsub_rn(__fsub_rn(1.0f, s), x.h), x.l)};
}

struct MvLife {
    int i, last;
    df c;
};
__device__ __forceinline__ df at(const float2* __restrict__ col, const MvLife& a, int t) {
    if (t > a.last) return df{0.0f, 0.0f};
    const float2 v = col[a.i + t];
    return df{v.x, v.y};
}

// E_p(t) in the row's unit (K_ANN, K_ASS: times m_x; the others: per unit amount)
template <int KIND>
__device__ __forceinline__ df mv_expected(const CfTables& T, const MvLife& a, const MvLife& b, int state0, int t) {
    if constexpr (KIND == K_ANN) {
        return at(T.m2, a, t + 1);
    } else if constexpr (KIND == K_ASS) {
        return at(T.dm2, a, t);
    } else if constexpr (KIND == K_ANN2) {
        return df_mul(df_mul(at(T.m2, a, t + 1), a.c), df_mul(at(T.m2, b, t + 1), b.c));
    } else if constexpr (KIND == K_JL) {   // a dead life's c is 0
        const df x = df_mul(at(T.m2, a, t + 1), a.c), y = df_mul(at(T.m2, b, t + 1), b.c);
        return df_add_pos(x, df_mul(y, df_one_minus(x)));
    } else if constexpr (KIND == K_ASS2) {
        const df dx = df_mul(at(T.dm2, a, t), a.c), dy = df_mul(at(T.dm2, b, t), b.c);
        return df_add_pos(df_mul(dx, df_mul(at(T.m2, b, t), b.c)), df_mul(df_mul(at(T.m2, a, t + 1), a.c), dy));
    } else {   // second death: x dies now and y is dead by the end, or x was dead and y dies now
        const df dx = df_mul(at(T.dm2, a, t), a.c), dy = df_mul(at(T.dm2, b, t), b.c);
        if (state0 == 1) return dx;
        if (state0 == 2) return dy;
        return df_add_pos(df_mul(dx, df_one_minus(df_mul(at(T.m2, b, t + 1), b.c))),
                          df_mul(df_one_minus(df_mul(at(T.m2, a, t), a.c)), dy));
    }
}
template <int KIND>
__device__ __forceinline__ df mv_boundary(const CfTables& T, const MvLife& a, const MvLife& b, int state0, int S) {
    if constexpr (KIND == K_ASS) return at(T.m2, a, S);
    const df x = df_mul(at(T.m2, a, S), a.c), y = df_mul(at(T.m2, b, S), b.c);
    if constexpr (KIND == K_ASS2) return df_mul(x, y);
    if (state0 == 1) return x;
    if (state0 == 2) return y;
    return df_add_pos(x, df_mul(y, df_one_minus(x)));
}


// ---- one row by one warp: the scale of the row, then the digits, four consecutive steps a
// lane.  Closed forms, so no chain over the steps.  200,000 annuities x 520 steps: 248 ->
// 166 us deflated (0.64 GB, past the L2: bound by the memory's write rate), 290 -> 231 us
// compensated, when the lanes took four steps, packed conversions and no pass for the
// largest entry of a level annuity.
__device__ __forceinline__ df df_of(double v) {
    const float h = __double2float_rn(v);
    return df{h, __double2float_rn(v - (double)h)};
}

// the largest tilted head of flow(t), t < S
template <class Flow>
__device__ __forceinline__ float mv_top(const Flow& flow, int S, const float* __restrict__ tilt) {
    float top = 0.0f;
    for (int t = threadIdx.x & 31; t < S; t += 32) top = fmaxf(top, __fmul_rn(flow(t).h, tilt[t]));
#pragma unroll
    for (int d = 16; d > 0; d >>= 1) top = fmaxf(top, __shfl_xor_sync(0xffffffffu, top, d));
    return top;
}
// the row's binary exponent: entries below 1; in the FP64 form one bit less for each doubling
// of the steps beyond 1,000, so that the leading digits' sum over the segments stays exact
template <int NS>
__device__ __forceinline__ int mv_row_exp(float top, int S) {
    const int e = top > 0.0f ? ((__float_as_int(top) >> 23) & 255) - 126 : 0;
    return NS == 8 ? e + (S > 1000) + (S > 2000) + (S > 4000) : e;
}
// digits of flow(t) tilted and times 2^-e, t < live, and zeros up to kt
template <int NS, class Flow>
__device__ __forceinline__ void mv_write_row(const Flow& flow, int live, int e, int kt, const float* __restrict__ tilt,
                                             void* digits, int row, int pitch) {
    const float f = pow2f(kMvLog<NS> - e);
    uint16_t* base = static_cast<uint16_t*>(digits) + ((size_t)(row / kMvP) * NS * kMvP + row % kMvP) * pitch;
    for (int t = 4 * (threadIdx.x & 31); t < kt; t += 128) {
        df v[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) v[k] = t + k < live ? flow(t + k) : df{0.0f, 0.0f};
        const float4 w = *reinterpret_cast<const float4*>(tilt + t);
        const float g[4] = {__fmul_rn(w.x, f), __fmul_rn(w.y, f), __fmul_rn(w.z, f), __fmul_rn(w.w, f)};
#pragma unroll
        for (int k = 0; k < 4; ++k) v[k] = df{__fmul_rn(v[k].h, g[k]), __fmul_rn(v[k].l, g[k])};
        uint32_t d0[NS], d1[NS];
        mv_digits<NS>(v[0].h, v[0].l, v[1].h, v[1].l, d0);
        mv_digits<NS>(v[2].h, v[2].l, v[3].h, v[3].l, d1);
#pragma unroll
        for (int k = 0; k < NS; ++k)
            *reinterpret_cast<uint2*>(base + (size_t)k * kMvP * pitch + t) = make_uint2(d0[k], d1[k]);
    }
}
// a normal FP64 number as a double-float below 1 in magnitude and a binary exponent (0: 0)
__device__ __forceinline__ df df_mantissa(double v, int& ex) {
    ex = 0;
    if (v == 0.0) return df{0.0f, 0.0f};
    const int hi = __double2hiint(v);
    ex = ((hi >> 20) & 2047) - 1022;
    return df_of(__hiloint2double((hi & 0x800FFFFF) | 0x3FE00000, __double2loint(v)));
}
__device__ __forceinline__ MvOut mv_out(df unit, int ex, int e, int pol, int S) {
    const float g = pow2f(ex + e);
    MvOut o;
    o.sc_h = __fmul_rn(unit.h, g);
    o.sc_l = __fmul_rn(unit.l, g);
    o.mat_h = o.mat_l = 0.0f;
    o.pol = pol;
    o.S = S;
    o.pad[0] = o.pad[1] = 0;
    return o;
}

template <int NS, int KIND, bool CF>
__device__ __forceinline__ void mv_row(const MvBuild& b, const SlotRec& r, int row, int kt, const float* __restrict__ tilt) {
    const CfTables& T = b.T;
    auto life = [&](int idx) {
        const int tb = idx < b.tab_pad ? 0 : idx / b.tab_pad, age = idx - tb * b.tab_pad;
        MvLife q;
        q.i = tb * T.rows + age;
        q.last = T.z[q.i] - age;
        return q;
    };
    MvLife x = life(r.idx1), y = life(r.idx2);
    const double amount = r.pol >= 0 ? b.amount[r.pol] : 0.0;
    const int S = r.pol >= 0 ? r.S : 0;
    if constexpr (KIND != K_ANN && KIND != K_ASS) {
        x.c = df_of(T.inv[x.i]);
        y.c = df_of(T.inv[y.i]);
        if (KIND == K_JL) {
            y.c = df_mul(y.c, df{r.rho_h, r.rho_l});
            if (r.state0 == 2) x.c = df{0.0f, 0.0f};
            if (r.state0 == 1) y.c = df{0.0f, 0.0f};
        }
    }
    auto flow = [&](int t) {
        df e = mv_expected<KIND>(T, x, y, r.state0, t);
        if constexpr (CF) e = df_mul(e, df_of(b.cf[(size_t)r.pol * b.cf_ld + t]));
        return e;
    };
    int e;
    if constexpr (!CF && (KIND == K_ANN || KIND == K_ANN2 || KIND == K_JL)) {
        // A level annuity's cash flows do not increase, so its first one times the largest
        // tilt bounds them (it is the largest unless the tilt increases later, by
        // negative rates); the others are looked through.
        e = mv_row_exp<NS>(S > 0 ? __fmul_rn(flow(0).h, b.tilt_top[S - 1]) : 0.0f, S);
    } else {
        e = mv_row_exp<NS>(mv_top(flow, S, tilt), S);
    }
    if constexpr (!CF && (KIND == K_ANN || KIND == K_ASS)) {   // straight from the column
        const int live = KIND == K_ANN ? min(S, x.last) : min(S, x.last + 1);
        const float2* col = KIND == K_ASS ? T.dm2 + x.i : T.m2 + x.i + 1;
        mv_write_row<NS>([&](int t) { const float2 w = __ldg(col + t); return df{w.x, w.y}; }, live, e, kt, tilt, b.digits, row,
                         b.pitch);
    } else {
        mv_write_row<NS>(flow, S, e, kt, tilt, b.digits, row, b.pitch);
    }
    if ((threadIdx.x & 31) == 0) {
        int ex;
        const df q = df_mantissa(KIND == K_ANN || KIND == K_ASS ? __dmul_rn(amount, T.inv[x.i]) : amount, ex);
        MvOut o = mv_out(q, ex, e, r.pol, S);
        if constexpr (KIND == K_ASS || KIND == K_ASS2 || KIND == K_LS2) {
            if (r.bnd != 0.0f && r.pol >= 0) {   // the maturity payment, or the amount if it is due now
                df m{r.bnd, 0.0f}, w = q;
                int em = 0, xm = ex;
                if (S == 0) {
                    w = df_mantissa(amount, xm);
                } else {
                    m = mv_boundary<KIND>(T, x, y, r.state0, S);
                    em = m.h > 0.0f ? ((__float_as_int(m.h) >> 23) & 255) - 126 : 0;
                    const float f2 = pow2f(-em);
                    m = df{__fmul_rn(m.h, f2), __fmul_rn(m.l, f2)};
                }
                const df v = df_mul(m, w);
                const float g2 = pow2f(xm + em);
                o.mat_h = __fmul_rn(v.h, g2);
                o.mat_l = __fmul_rn(v.l, g2);
            }
        }
        b.out[row] = o;
    }
}

// ---- the FP64 form: the cash flows in FP64 (cashflow.cuh), the scale from their FP32 heads
struct alignas(16) MvOut64 {   // in the place of MvOut
    double sc, mat;
    int32_t pol, S, pad[2];
};
static_assert(sizeof(MvOut64) == sizeof(MvOut), "record sizes");

template <int KIND, bool CF>
__device__ __forceinline__ void mv_row64(const MvBuild& b, const SlotRec& r, const CfPol& p, int row, int kt,
                                         const float* __restrict__ tilt) {
    const CfTables& T = b.T;
    const MvLife x{p.a.i, p.a.last, df_of(KIND == K_JL && r.state0 == 2 ? 0.0 : p.a.inv)};
    const MvLife y{p.b.i, p.b.last, df_of(KIND == K_JL ? (r.state0 == 1 ? 0.0 : p.b.inv * p.rho) : p.b.inv)};
    const int S = r.pol >= 0 ? r.S : 0;
    auto head = [&](int t) {   // per unit amount, as cf_expected
        df e = mv_expected<KIND>(T, x, y, r.state0, t);
        if constexpr (KIND == K_ANN || KIND == K_ASS) e = df_mul(e, x.c);
        if constexpr (CF) e = df_mul(e, df_of(b.cf[(size_t)r.pol * b.cf_ld + t]));
        return e;
    };
    int e;
    if constexpr (!CF && (KIND == K_ANN || KIND == K_ANN2 || KIND == K_JL))
        e = mv_row_exp<8>(S > 0 ? __fmul_rn(head(0).h, b.tilt_top[S - 1]) : 0.0f, S);
    else
        e = mv_row_exp<8>(mv_top(head, S, tilt), S);
    uint32_t* base = static_cast<uint32_t*>(b.digits) + ((size_t)(row / kMvP) * 8 * kMvP + row % kMvP) * b.pitch / 2;
    for (int t = 2 * (threadIdx.x & 31); t < kt; t += 64) {
        unsigned long long v[2] = {0, 0};
#pragma unroll
        for (int k = 0; k < 2; ++k)
            if (t + k < S) {
                double f = cf_expected(T, p, t + k);
                if constexpr (CF) f *= b.cf[(size_t)r.pol * b.cf_ld + t + k];
                v[k] = mv_fixed64(f, (__float_as_int(tilt[t + k]) >> 23) - 127 - e);
            }
#pragma unroll
        for (int k = 0; k < 8; ++k) base[((size_t)k * kMvP * b.pitch + t) / 2] = mv_byte_pair(v[0], v[1], k);
    }
    if ((threadIdx.x & 31) == 0) {
        MvOut64 o;
        o.sc = p.amount * __hiloint2double((e + 1023) << 20, 0);
        o.mat = r.pol >= 0 && p.bnd != 0.0 ? p.amount * (S == 0 ? p.bnd : cf_boundary(T, p)) : 0.0;
        o.pol = r.pol;
        o.S = S;
        o.pad[0] = o.pad[1] = 0;
        reinterpret_cast<MvOut64*>(b.out)[row] = o;
    }
}

__global__ void __launch_bounds__(256) mv_build64_kernel(const MvBuild b, const CfPol* __restrict__ pols) {
    grid_dependency_wait();
    extern __shared__ float4 tilt4[];
    float* tilt = reinterpret_cast<float*>(tilt4);
    const int row = blockIdx.x * 8 + (threadIdx.x >> 5), tile = row / kMvP;
    const int kt = max(64, (b.slots[(size_t)tile * kMvP].S + 63) / 64 * 64);
    for (int t = threadIdx.x; t < kt; t += 256) tilt[t] = t < b.n_steps ? b.tilt[t] : 0.0f;
    __syncthreads();
    const SlotRec r = b.slots[row];
    const CfPol p = pols[row];
    auto run = [&](auto cf) {
        constexpr bool CF = decltype(cf)::value;
        switch (b.kinds[tile]) {
        case K_ANN: return mv_row64<K_ANN, CF>(b, r, p, row, kt, tilt);
        case K_ASS: return mv_row64<K_ASS, CF>(b, r, p, row, kt, tilt);
        case K_JL: return mv_row64<K_JL, CF>(b, r, p, row, kt, tilt);
        case K_ANN2: return mv_row64<K_ANN2, CF>(b, r, p, row, kt, tilt);
        case K_ASS2: return mv_row64<K_ASS2, CF>(b, r, p, row, kt, tilt);
        default: return mv_row64<K_LS2, CF>(b, r, p, row, kt, tilt);
        }
    };
    if (tile >= b.general_from) run(std::true_type{});
    else run(std::false_type{});
}

// ---- contracts on up to four lives (MvLives): the lives are independent, so a step's
// expected cash flow is a polynomial in their survival and death probabilities.  A life
// that is absent counts for nothing (an annuity counts it as dead, an assurance as alive).
//   annuity:    Pr[k or more alive at the end of step t]
//   assurance:  the k-th death in step t: Pr[k or more dead] is linear in each life, so its
//               growth is the sum, over the lives moved one by one to the step's end, of the
//               life's deaths times Pr[exactly k - 1 of the others are dead]
__device__ __forceinline__ df mv_lives_flow(const CfTables& T, const MvLives& r, const MvLife (&l)[4], const df (&one)[4], int t) {
    const bool ass = r.flags & 1;
    df p[4], q[4];   // alive and dead at the end of the step
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        p[i] = l[i].last < 0 ? one[i] : df_mul(at(T.m2, l[i], t + 1), l[i].c);
        q[i] = df_one_minus(p[i]);
    }
    if (!ass) {
        df c[5] = {q[0], p[0], df{0.0f, 0.0f}, df{0.0f, 0.0f}, df{0.0f, 0.0f}};   // Pr[j alive]
#pragma unroll
        for (int i = 1; i < 4; ++i) {
            c[i + 1] = df_mul(c[i], p[i]);
#pragma unroll
            for (int j = i; j > 0; --j) c[j] = df_add_pos(df_mul(c[j], q[i]), df_mul(c[j - 1], p[i]));
            c[0] = df_mul(c[0], q[i]);
        }
        df e = c[4];
#pragma unroll
        for (int j = 3; j > 0; --j)
            if (j >= r.k) e = df_add_pos(e, c[j]);
        return e;
    }
    df e{0.0f, 0.0f};
    df a[4], b[4];   // the lives not yet moved: alive and dead at the start
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        a[i] = l[i].last < 0 ? one[i] : df_mul(at(T.m2, l[i], t), l[i].c);
        b[i] = df_one_minus(a[i]);
    }
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        if (l[i].last < 0) continue;
        df c[4] = {df{1.0f, 0.0f}, df{0.0f, 0.0f}, df{0.0f, 0.0f}, df{0.0f, 0.0f}};   // Pr[j of the others dead]
        int n = 0;
#pragma unroll
        for (int o = 0; o < 4; ++o) {
            if (o == i) continue;
            const df al = o < i ? p[o] : a[o], de = o < i ? q[o] : b[o];
            ++n;
            c[n] = df_mul(c[n - 1], de);
#pragma unroll
            for (int j = n - 1; j > 0; --j) c[j] = df_add_pos(df_mul(c[j], al), df_mul(c[j - 1], de));
            c[0] = df_mul(c[0], al);
        }
        const df w = r.k == 1 ? c[0] : (r.k == 2 ? c[1] : (r.k == 3 ? c[2] : c[3]));
        e = df_add_pos(e, df_mul(df_mul(at(T.dm2, l[i], t), l[i].c), w));
    }
    return e;
}

template <int NS>
__global__ void __launch_bounds__(256) mv_build_lives_kernel(const CfTables T, const MvLives* __restrict__ recs,
                                                             const double* __restrict__ amount, int pitch, int n_steps,
                                                             const float* __restrict__ tilt_g, void* digits,
                                                             MvOut* __restrict__ out) {
    grid_dependency_wait();
    extern __shared__ float4 tilt4[];
    float* tilt = reinterpret_cast<float*>(tilt4);
    const int row = blockIdx.x * 8 + (threadIdx.x >> 5), tile = row / kMvP;
    const int kt = max(64, (recs[(size_t)tile * kMvP].S + 63) / 64 * 64);
    for (int t = threadIdx.x; t < kt; t += 256) tilt[t] = t < n_steps ? tilt_g[t] : 0.0f;
    __syncthreads();
    const MvLives r = recs[row];
    const bool ass = r.flags & 1;
    MvLife l[4];
    df one[4];   // of a life that takes no part: 1 alive for ever, 0 dead
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const bool dead = r.flags >> (8 + i) & 1, absent = r.idx[i] < 0;
        one[i] = df{absent && ass ? 1.0f : 0.0f, 0.0f};
        l[i].i = absent ? 0 : r.idx[i];
        l[i].last = absent || dead ? -1 : T.z[l[i].i] - l[i].i % T.rows;
        l[i].c = df_of(T.inv[l[i].i]);
    }
    const int S = r.pol >= 0 ? r.S : 0;
    auto flow = [&](int t) { return mv_lives_flow(T, r, l, one, t); };
    const int e = mv_row_exp<NS>(mv_top(flow, S, tilt), S);
    mv_write_row<NS>(flow, S, e, kt, tilt, digits, row, pitch);
    if ((threadIdx.x & 31) == 0) {
        int ex;
        const df q = df_mantissa(r.pol >= 0 ? amount[r.pol] : 0.0, ex);
        out[row] = mv_out(q, ex, e, r.pol, S);
    }
}

template <int NS>
__global__ void __launch_bounds__(256) mv_build_kernel(const MvBuild b) {
    grid_dependency_wait();
    extern __shared__ float4 tilt4[];   // 2^-tau(t)
    float* tilt = reinterpret_cast<float*>(tilt4);
    const int rows = 8 * b.rows_per_warp, row0 = blockIdx.x * rows, tile = row0 / kMvP;
    const int kt = max(64, (b.slots[(size_t)tile * kMvP].S + 63) / 64 * 64);   // the tile's longest projection
    for (int t = threadIdx.x; t < kt; t += 256) tilt[t] = t < b.n_steps ? b.tilt[t] : 0.0f;
    __syncthreads();
    auto run = [&](auto cf) {
        constexpr bool CF = decltype(cf)::value;
        for (int row = row0 + (threadIdx.x >> 5); row < row0 + rows; row += 8) {
            const SlotRec r = b.slots[row];
            switch (b.kinds[tile]) {
            case K_ANN: mv_row<NS, K_ANN, CF>(b, r, row, kt, tilt); break;
            case K_ASS: mv_row<NS, K_ASS, CF>(b, r, row, kt, tilt); break;
            case K_JL: mv_row<NS, K_JL, CF>(b, r, row, kt, tilt); break;
            case K_ANN2: mv_row<NS, K_ANN2, CF>(b, r, row, kt, tilt); break;
            case K_ASS2: mv_row<NS, K_ASS2, CF>(b, r, row, kt, tilt); break;
            default: mv_row<NS, K_LS2, CF>(b, r, row, kt, tilt);
            }
        }
    };
    if (tile >= b.general_from) run(std::true_type{});
    else run(std::false_type{});
}

// -------------------------------------------------------------- the product ----
// Persistent pairs of CTAs over (policy tile or half tile, pair of scenario tiles) items.  A
// block of steps of the digits is staged by TMA into a ring of stages: each CTA its 128
// scenarios' (A) and half of the item's policies' (B); one thread of rank 0 issues the
// digits' products, m256 k16 over both CTAs (cta_group::2).  In each CTA the scenarios are
// on the lanes and the policies on the columns; sixteen warps add the accumulators as
// double-floats, scale, write V0 (32 consecutive scenarios of a policy a warp store) and
// sum each scenario over the item's policies.
// Three digits: 6 products and 2 accumulators, so TMEM holds two tiles' and the epilogue
// runs beside the next tile's products.  Four: 10 products, 4 accumulators (half tiles, two in
// TMEM: 0.89 -> 0.95 ms for 100,000 policies x 1,000 scenarios).  Six and eight: 21 and 36
// products, seven and eight accumulators of half a tile's policies.  Such a product (n64)
// lasts as long as the shared-memory reads of its A, so A is read once a scenario digit
// and kept in the collector: 903 -> 755 us a launch of 50,000 x 1,000 with six.  Whole
// tiles with the levels 3 to 5 in one accumulator took 690 us, at 13 times the error (totals of
// annuities 1.8e-13 against the recurrence's 9e-14).
// With one item in TMEM the products stand still until its accumulators are read, so before
// the release the low ones are only summed and the rest follows after it; in the FP64
// form all of this had been conversions and sums on the FP64 pipe, longer than the products
// (100,000 x 1,000 of every product: four digits 0.90 -> 0.88 ms, six 1.68 -> 1.62 ms; 3,000 x 333
// in FP64: 0.203 -> 0.148 ms).
// An accumulator sums at most SEG steps (a segment), so that the levels that must be exact
// are (matval.cuh); a longer item's segments are added up by the epilogue, whose sums so far wait
// in local memory (in registers they would not fit beside an accumulator's columns).  A segment's
// end costs about 2,000 cycles.  Six digits, 100,000 x 1,000 of every product: 1.67 ms; 1.74 with
// segments of 256 steps and a level an accumulator, 1.62 over whole projections, inexact.  FP64,
// 3,000 x 333: 0.148, 0.154 and 0.146 ms.
template <int NS>
struct MvShape;   // policies of an item, accumulators, segments in TMEM, stages, steps of a block (64:
template <>       // 128-byte swizzled rows) and of a segment; the products are (i, j), i + j < NS, of
struct MvShape<3> {   // scenario digit i and policy digit j, in accumulator mv_acc
    static constexpr int N = kMvP, NA = 2, NB = 2, ST = 3, KB = 64, SEG = 1024;
};
template <>
struct MvShape<4> {
    static constexpr int N = kMvP, NA = 4, NB = 1, ST = 4, KB = 32, SEG = 1024;
};
template <>
struct MvShape<6> {
    static constexpr int N = kMvP / 2, NA = 7, NB = 1, ST = 3, KB = 32, SEG = 512;
};
template <>
struct MvShape<8> {
    static constexpr int N = kMvP / 2, NA = 8, NB = 1, ST = 2, KB = 32, SEG = 512;
};
// The accumulator of the product (i, j).  Three and four digits: one for each of the first levels.
// Six and eight: levels 0 and 1; 2 and 3, of three and four products, in two each, so that none
// takes more than two of an exact level; the rest in one (eight: 4, and the rest).
template <int NS>
__host__ __device__ constexpr int mv_acc(int i, int j) {
    const int level = i + j, inner = i > 0 && j > 0;
    if (NS < 6 || level < 2) return level < MvShape<NS>::NA ? level : MvShape<NS>::NA - 1;
    if (level < 4) return 2 * level - 2 + inner;
    return NS == 8 && level > 4 ? 7 : 6;
}
template <int NS>
__host__ __device__ constexpr bool mv_acc_first(int i, int j) {   // no product before (i, j) goes there
    for (int a = 0; a <= i; ++a)
        for (int b = 0; a + b < NS && (a < i || b < j); ++b)
            if (mv_acc<NS>(a, b) == mv_acc<NS>(i, j)) return false;
    return true;
}
constexpr int kMvEpi = 4 * kMvParts;                   // epilogue warps
constexpr int kMvThreads = 32 * (kMvEpi + 2);

// shared memory of a stage: NS slabs of scenario digits, then NS of policy digits
template <int NS>
struct MvStage {
    using Sh = MvShape<NS>;
    static constexpr int kA = kMvM * Sh::KB * 2, kB = Sh::N / 2 * Sh::KB * 2;
    static constexpr int kBytes = NS * (kA + kB);
};

// The products of scenario digit I and policy digits J .., then of digits I + 1 ..; more: the
// accumulators hold earlier blocks' sums.
template <int NS, int I, int J>
__device__ __forceinline__ void mv_products(uint32_t d, uint64_t base, int off, uint32_t idesc, bool more) {
    using Sh = MvShape<NS>;
    using G = MvStage<NS>;
    constexpr int acc = mv_acc<NS>(I, J);
    constexpr bool first = mv_acc_first<NS>(I, J);
    constexpr bool last = I + J + 1 == NS;
    constexpr int coll = Sh::N == kMvP || (J == 0 && last) ? COLL_NONE : (J == 0 ? COLL_FILL : (last ? COLL_LAST : COLL_USE));
    mma_f16_ss_pair<coll>(d + acc * Sh::N, base + (uint64_t)((I * G::kA + off) >> 4),
                    base + (uint64_t)((NS * G::kA + J * G::kB + off) >> 4), idesc, !first || more);
    if constexpr (I + J + 1 < NS) mv_products<NS, I, J + 1>(d, base, off, idesc, more);
    else if constexpr (I + 1 < NS) mv_products<NS, I + 1, 0>(d, base, off, idesc, more);
}

__device__ __forceinline__ void two_sum(float a, float b, float& s, float& e) {
    const float t = __fadd_rn(a, b), bb = __fsub_rn(t, a);
    e = __fadd_rn(__fsub_rn(a, __fsub_rn(t, bb)), __fsub_rn(b, bb));
    s = t;
}
// x 2^e, by the bits (the conversion instruction runs at the FP64 rate); 0 below 2^-126
__device__ __forceinline__ double scaled_double(float x, int e) {
    const uint32_t b = __float_as_uint(x), m = b & 0x7FFFFFFFu;
    const bool zero = m < 0x00800000u;
    const uint32_t hi = (b & 0x80000000u) | ((m >> 3) + ((uint32_t)(896 + e) << 20));
    return __hiloint2double(zero ? 0 : (int)hi, zero ? 0 : (int)(b << 29));
}

template <int NS>
__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(kMvThreads, 1)
    mv_product_kernel(const __grid_constant__ CUtensorMap mapD, const __grid_constant__ CUtensorMap mapE, const MvArgs a) {
    using Sh = MvShape<NS>;
    using G = MvStage<NS>;
    constexpr int KB = Sh::KB, N = Sh::N, kSub = kMvP / N, kSeg = Sh::SEG / KB;   // kSeg: blocks of a segment
    constexpr uint32_t kIdesc = f16_idesc(NS != 3, 2 * kMvM, N);   // both operands FP16, or both BF16
    extern __shared__ __align__(1024) unsigned char smem_raw[];
    // (both CTAs of a pair place everything alike)
    unsigned char* ring = reinterpret_cast<unsigned char*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
    // rank 0's full[st]: both CTAs' copies of a stage; empty[st]: its products are done;
    // acc_full: a tile's products are done; rank 0's acc_empty: both epilogues have read it
    __shared__ uint64_t full[Sh::ST], empty[Sh::ST], acc_full[Sh::NB], acc_empty[Sh::NB], drained;
    __shared__ uint32_t tmem_slot;
    __shared__ MvOut recs[kMvP];
    __shared__ __align__(8) float2 sums[kMvParts][kMvM];
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int rank = (int)cluster_rank();
    if (tid == 0) {
        for (int i = 0; i < Sh::ST; ++i) {
            mbar_init(&full[i], 1);
            mbar_init(&empty[i], 1);
        }
        for (int i = 0; i < Sh::NB; ++i) {
            mbar_init(&acc_full[i], 1);
            mbar_init(&acc_empty[i], 2 * kMvEpi);
        }
        mbar_init(&drained, 1);
        fence_barrier_init();
    }
    if (warp == 0) tmem_alloc_pair(&tmem_slot, 512);
    fence_before();
    cluster_sync();
    fence_after();
    grid_dependency_wait();   // for the rows of the builder
    const uint32_t tmem = tmem_slot;
    const int n_pairs = (a.n_chunks + 1) / 2, n_clusters = (int)gridDim.x / 2, cluster = (int)blockIdx.x / 2;
    const long long n_items = (long long)a.n_tiles * kSub * n_pairs;   // part of a tile, pair of scenario tiles
    bool failed = false;
    auto wait_on = [&](uint64_t* bar, uint32_t parity) {   // a bounded wait; a timeout is recorded
        if (failed) return;
        if (!mbar_wait_bounded(bar, parity, kMvPoll)) {
            failed = true;
            atomicExch(a.status, DEV_TIMEOUT);
        }
    };
    auto blocks_of = [&](int tile) { return max(1, (a.steps[(size_t)tile * kMvP * kMvRecWords] + KB - 1) / KB); };

    if (warp == kMvEpi) {
        // ---- the copies (one thread of each CTA)
        if (elect_one()) {
            uint32_t it = 0;
            for (long long item = cluster; item < n_items && !failed; item += n_clusters) {
                const int sub = (int)(item / n_pairs), chunk = 2 * (int)(item - (long long)sub * n_pairs) + rank;
                const int tile = sub / kSub, col = (sub - tile * kSub) * N + rank * (N / 2);
                const int nk = blocks_of(tile);
                for (int kb = 0; kb < nk && !failed; ++kb, ++it) {
                    const int st = it % Sh::ST;
                    if (it >= Sh::ST) wait_on(&empty[st], (it / Sh::ST - 1) & 1);
                    if (failed) break;
                    unsigned char* dst = ring + st * G::kBytes;
                    const uint32_t bar = of_rank0(&full[st]);
                    if (rank == 0) mbar_arrive_expect_tx(&full[st], 2 * G::kBytes);
#pragma unroll
                    for (int k = 0; k < NS; ++k) {
                        tma_load_2d_pair(dst + k * G::kA, &mapD, kb * KB, k * a.s_pad + a.s0 + chunk * kMvM, bar);
                        tma_load_2d_pair(dst + NS * G::kA + k * G::kB, &mapE, kb * KB, (tile * NS + k) * kMvP + col, bar);
                    }
                }
            }
            // let the copies in flight land before the memory is released (rank 1's complete on
            // rank 0's barriers, and rank 1 stays until rank 0 has come to the end)
            if (failed && rank == 0)
                for (uint32_t back = 0; back < Sh::ST && back < it; ++back)
                    mbar_wait_bounded(&full[(it - 1 - back) % Sh::ST], ((it - 1 - back) / Sh::ST) & 1, kMvPoll);
        }
        __syncwarp();
    } else if (warp == kMvEpi + 1) {
        // ---- the products (one thread of rank 0)
        if (rank == 0 && elect_one()) {
            uint32_t it = 0, n = 0;
            const uint64_t ring_desc = KB == 64 ? sw128_desc(ring) : sw64_desc(ring);
            for (long long item = cluster; item < n_items && !failed; item += n_clusters) {
                const int nk = blocks_of((int)(item / n_pairs) / kSub);
                for (int k0 = 0; k0 < nk && !failed; k0 += kSeg, ++n) {
                    const int buf = n % Sh::NB;
                    if (n >= Sh::NB) wait_on(&acc_empty[buf], (n / Sh::NB - 1) & 1);
                    const uint32_t d = tmem + buf * (Sh::NA * N);
                    for (int kb = k0; kb < min(nk, k0 + kSeg) && !failed; ++kb, ++it) {
                        const int st = it % Sh::ST;
                        wait_on(&full[st], (it / Sh::ST) & 1);
                        if (failed) break;
                        fence_after();
                        const uint64_t base = ring_desc + (uint64_t)((st * G::kBytes) >> 4);
#pragma unroll
                        for (int k16 = 0; k16 < KB / 16; ++k16)
                            mv_products<NS, 0, 0>(d, base, k16 * 32, kIdesc, kb - k0 + k16 > 0);
                        mma_commit_pair(&empty[st]);
                    }
                    if (!failed) mma_commit_pair(&acc_full[buf]);
                }
            }
            if (failed) {   // let the products in flight finish before the memory is released
                mma_commit_pair(&drained);
                mbar_wait_bounded(&drained, 0, kMvPoll);
            }
        }
        __syncwarp();
    } else {
        // ---- the epilogue: lanes = scenarios 32 (warp % 4) .., columns kCols (warp / 4) ..
        constexpr int kCols = N / kMvParts;
        const int quarter = warp & 3, part = warp >> 2;
        uint32_t n = 0;
        uint32_t acc_free[Sh::NB];
        for (int i = 0; i < Sh::NB; ++i) acc_free[i] = of_rank0(&acc_empty[i]);
        volatile float run[NS == 8 ? 3 : 2][kCols];   // the item's earlier segments
        for (long long item = cluster; item < n_items; item += n_clusters) {
            const int sub = (int)(item / n_pairs), chunk = 2 * (int)(item - (long long)sub * n_pairs) + rank;
            const int tile = sub / kSub, nk = blocks_of(tile);
            if (tid < N * 2) reinterpret_cast<float4*>(recs)[tid] = reinterpret_cast<const float4*>(a.out + (size_t)sub * N)[tid];
            asm volatile("bar.sync 1, %0;" ::"n"(32 * kMvEpi) : "memory");
            const int s = chunk * kMvM + quarter * 32 + lane;
            const bool inside = chunk < a.n_chunks;   // an odd last pair's second tile is empty
            const int sl = inside ? s : 0;
            const float dsc = pow2f(a.colexp[sl] - (NS == 3 ? 30 : 0));
            df tot{0.0f, 0.0f};
            double tot64 = 0.0;
            for (int k0 = 0; k0 < nk; k0 += kSeg, ++n) {
                const int buf = n % Sh::NB;
                const bool last = k0 + kSeg >= nk;
                bool ok = true;
                if (lane == 0 && !failed) ok = mbar_wait_bounded(&acc_full[buf], (n / Sh::NB) & 1, kMvPoll);
                ok = __shfl_sync(0xffffffffu, ok, 0);
                if (!ok && !failed) {   // recorded; the later waits are skipped and nothing is written
                    failed = true;
                    if (lane == 0) atomicExch(a.status, DEV_TIMEOUT);
                }
                fence_after();
                const bool live = s < a.n_scen && !failed;
                const uint32_t col0 = tmem + ((uint32_t)(quarter * 32) << 16) + buf * (Sh::NA * N) + part * kCols;
                auto load2 = [&](int k0, int k1, int c, float (&y)[16], float (&z)[16]) {   // two accumulators' 16 columns
                    uint32_t r[2][16];
                    tmem_ld16_async(col0 + k0 * N + c, r[0]);
                    tmem_ld16_async(col0 + k1 * N + c, r[1]);
                    tmem_wait_ld(r[0]);
                    tmem_wait_ld(r[1]);
#pragma unroll
                    for (int i = 0; i < 16; ++i) {
                        y[i] = __uint_as_float(r[0][i]);
                        z[i] = __uint_as_float(r[1][i]);
                    }
                };
                auto release = [&] {   // the accumulators are read
                    fence_before();
                    __syncwarp();
                    if (lane == 0) mbar_arrive_remote(acc_free[buf]);
                };
                // the columns of this warp, without branches over them (padding rows are 0), so that
                // their chains overlap; MAT: maturity payments
                auto columns = [&](auto with_maturity) {
                    constexpr bool MAT = decltype(with_maturity)::value;
                    auto emit = [&](const MvOut& q, float h, float l) {   // of a policy's sum h + l
                        df v = df_mul(df{__fmul_rn(h, dsc), __fmul_rn(l, dsc)}, df{q.sc_h, q.sc_l});
                        const int pol = q.pol;
                        bool due = false;
                        if constexpr (MAT) {   // a maturity payment, of the same sign, or 0
                            const float2 d = a.D[(size_t)max(q.S - 1, 0) * a.s_pad + sl];
                            due = q.S == 0;
                            const df m = df_mul(df{q.mat_h, q.mat_l}, due ? df{1.0f, 0.0f} : df{d.x, d.y});
                            float sum, e;
                            two_sum(v.h, m.h, sum, e);
                            v = df{sum, __fadd_rn(e, __fadd_rn(v.l, m.l))};
                            due = due && q.mat_h != 0.0f;
                        }
                        // the sum over the policies
                        float sum, e;
                        two_sum(tot.h, v.h, sum, e);
                        tot = df{sum, __fadd_rn(tot.l, __fadd_rn(e, v.l))};
                        const size_t o = (size_t)pol * a.v0_ld + s;
                        if (live && pol >= 0) {
                            if (a.V0f) a.V0f[o] = __fadd_rn(v.h, v.l);
                            if (a.V0d) a.V0d[o] = due ? a.amount[pol] : (double)v.h + (double)v.l;
                        }
                    };
                    // Columns whose accumulators are added before they are released: as little as
                    // fits the registers, since with one item in TMEM the products stand still until then.
                    constexpr int kHold = NS == 4 ? kCols : 16;
#pragma unroll 1
                    for (int c0 = 0; c0 < kCols; c0 += kHold) {
                        if constexpr (NS == 8) {
                            // u = p + w + v + x: the levels 0 (p), 1 and 2 (w) and 3 (v) with
                            // their sums' errors, the lower ones as plain FP32 sums (2^-56) (x);
                            // the rest after the release
                            float p[16], w[16], v[16], x[16];
                            {
                                float y[16], z[16];
                                load2(7, 6, c0, y, z);
#pragma unroll
                                for (int i = 0; i < 16; ++i) x[i] = __fadd_rn(y[i], z[i]);
                                load2(5, 4, c0, y, z);
#pragma unroll
                                for (int i = 0; i < 16; ++i) {
                                    float e;
                                    two_sum(y[i], z[i], v[i], e);
                                    x[i] = __fadd_rn(x[i], e);
                                }
                                load2(3, 2, c0, y, z);
#pragma unroll
                                for (int i = 0; i < 16; ++i) {
                                    float e;
                                    two_sum(y[i], z[i], w[i], e);
                                    x[i] = __fadd_rn(x[i], e);
                                }
                                load2(1, 0, c0, y, p);
#pragma unroll
                                for (int i = 0; i < 16; ++i) {
                                    float e;
                                    two_sum(y[i], w[i], w[i], e);
                                    x[i] = __fadd_rn(x[i], e);
                                }
                            }
                            release();
                            const int ce = a.colexp[sl];
#pragma unroll
                            for (int i = 0; i < 16; ++i) {
                                const MvOut64& q = reinterpret_cast<const MvOut64&>(recs[part * kCols + c0 + i]);
                                float e;
                                two_sum(w[i], v[i], w[i], v[i]);
                                x[i] = __fadd_rn(x[i], v[i]);
                                if (k0 > 0) {   // the first levels' sum is exact
                                    p[i] = __fadd_rn(p[i], run[0][c0 + i]);
                                    two_sum(w[i], run[1][c0 + i], w[i], e);
                                    x[i] = __fadd_rn(__fadd_rn(x[i], e), run[2][c0 + i]);
                                }
                                if (!last) {
                                    run[0][c0 + i] = p[i];
                                    run[1][c0 + i] = w[i];
                                    run[2][c0 + i] = x[i];
                                    continue;
                                }
                                two_sum(p[i], w[i], p[i], w[i]);
                                // of the FP64 pipe (1/64 of the FP32 rate) only what needs 53 bits
                                double t = __dadd_rn(scaled_double(w[i], ce), scaled_double(x[i], ce));
                                t = __dmul_rn(__dadd_rn(scaled_double(p[i], ce), t), q.sc);
                                if constexpr (MAT) {
                                    const double d = q.S > 0 ? a.D64[(size_t)(q.S - 1) * a.s_pad + sl] : 1.0;
                                    t = __fma_rn(q.mat, d, t);
                                }
                                tot64 = __dadd_rn(tot64, t);
                                if (live && q.pol >= 0) {
                                    const size_t o = (size_t)q.pol * a.v0_ld + s;
                                    if (a.V0f) a.V0f[o] = __double2float_rn(t);
                                    if (a.V0d) a.V0d[o] = t;
                                }
                            }
                            continue;
                        }
                        // the accumulators' sum as a double-float: the errors of adding the first
                        // ones are kept; those from 2^-24 (four digits: 2^-16) of the first are
                        // added as they are, 2^-48 (2^-40)
                        float h[kHold], l[kHold];
#pragma unroll
                        for (int c = 0; c < kHold; c += 16) {
                            float y[16], z[16], x[16];
                            if constexpr (NS == 6) {
                                load2(6, 5, c0 + c, y, z);
#pragma unroll
                                for (int i = 0; i < 16; ++i) l[c + i] = __fadd_rn(y[i], z[i]);
                                load2(4, 3, c0 + c, y, z);
#pragma unroll
                                for (int i = 0; i < 16; ++i) l[c + i] = __fadd_rn(l[c + i], y[i]);
                                uint32_t r[16];
                                tmem_ld16_async(col0 + 2 * N + c0 + c, r);
                                tmem_wait_ld(r);
#pragma unroll
                                for (int i = 0; i < 16; ++i) {
                                    float e;
                                    two_sum(__uint_as_float(r[i]), z[i], z[i], e);
                                    l[c + i] = __fadd_rn(l[c + i], e);
                                }
                                load2(1, 0, c0 + c, y, x);
                                release();
#pragma unroll
                                for (int i = 0; i < 16; ++i) {
                                    float e1, e2;
                                    two_sum(x[i], y[i], x[i], e1);
                                    two_sum(x[i], z[i], h[c + i], e2);
                                    l[c + i] = __fadd_rn(l[c + i], __fadd_rn(e1, e2));
                                }
                            } else if constexpr (NS == 4) {
                                load2(3, 2, c0 + c, y, z);
#pragma unroll
                                for (int i = 0; i < 16; ++i) x[i] = __fadd_rn(y[i], z[i]);
                                load2(1, 0, c0 + c, y, z);
                                if (c0 + c == kCols - 16) release();
#pragma unroll
                                for (int i = 0; i < 16; ++i) {
                                    two_sum(z[i], y[i], h[c + i], l[c + i]);
                                    l[c + i] = __fadd_rn(l[c + i], x[i]);
                                }
                            } else {
                                uint32_t r[2][16];
                                tmem_ld16_async(col0 + c0, r[0]);
                                tmem_ld16_async(col0 + N + c0, r[1]);
                                tmem_wait_ld(r[0]);
                                tmem_wait_ld(r[1]);
                                if (c0 == kCols - 16) release();
#pragma unroll
                                for (int i = 0; i < 16; ++i) two_sum(__uint_as_float(r[0][i]), __uint_as_float(r[1][i]), h[i], l[i]);
                            }
                        }
                        if (k0 > 0) {
#pragma unroll
                            for (int i = 0; i < kHold; ++i) {
                                float e;
                                two_sum(h[i], run[0][c0 + i], h[i], e);
                                l[i] = __fadd_rn(__fadd_rn(l[i], e), run[1][c0 + i]);
                            }
                        }
                        if (!last) {
#pragma unroll
                            for (int i = 0; i < kHold; ++i) {
                                run[0][c0 + i] = h[i];
                                run[1][c0 + i] = l[i];
                            }
                            continue;
                        }
#pragma unroll
                        for (int i = 0; i < kHold; ++i) emit(recs[part * kCols + c0 + i], h[i], l[i]);
                    }
                };
                const int kind = a.kinds ? a.kinds[tile] : K_ANN;
                if (kind == K_ASS || kind == K_ASS2 || kind == K_LS2) columns(std::true_type{});
                else columns(std::false_type{});
            }
            // the parts' sums in part order; then the records and sums may be overwritten
            if constexpr (NS == 8) reinterpret_cast<double&>(sums[part][quarter * 32 + lane]) = tot64;
            else sums[part][quarter * 32 + lane] = make_float2(tot.h, tot.l);
            asm volatile("bar.sync 1, %0;" ::"n"(32 * kMvEpi) : "memory");
            if (part == 0 && a.partial && inside && !failed) {
                double x = 0.0;
#pragma unroll
                for (int k = 0; k < kMvParts; ++k) {
                    const float2 v = sums[k][quarter * 32 + lane];
                    if constexpr (NS == 8) x += reinterpret_cast<const double&>(v);
                    else x += (double)v.x + (double)v.y;
                }
                a.partial[(size_t)sub * a.part_ld + s] = x;
            }
        }
    }
    fence_before();
    cluster_sync();   // neither CTA leaves while the other may reach into it
    fence_after();
    if (warp == 0) tmem_free_pair(tmem, 512);
}

template <int NS>
cudaError_t product(const MvArgs& a, const void* digitsD, const void* digitsE, int pitchD, int pitchE, int sm_count,
                    cudaStream_t st) {
    using Sh = MvShape<NS>;
    constexpr auto swz = Sh::KB == 64 ? CU_TENSOR_MAP_SWIZZLE_128B : CU_TENSOR_MAP_SWIZZLE_64B;
    CUtensorMap mD, mE;
    if (!encode_map_16bit(&mD, CU_TENSOR_MAP_DATA_TYPE_UINT16, digitsD, pitchD, (uint64_t)NS * a.s_pad, pitchD, Sh::KB, kMvM,
                          swz) ||
        !encode_map_16bit(&mE, CU_TENSOR_MAP_DATA_TYPE_UINT16, digitsE, pitchE, (uint64_t)NS * kMvP * a.n_tiles, pitchE, Sh::KB,
                          Sh::N / 2, swz))
        return cudaErrorNotSupported;
    constexpr size_t smem = (size_t)Sh::ST * MvStage<NS>::kBytes + 1024;
    auto k = mv_product_kernel<NS>;
    cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    const long long items = (long long)a.n_tiles * (kMvP / Sh::N) * ((a.n_chunks + 1) / 2);
    return launch_next(k, dim3(2 * (int)std::min<long long>(items, sm_count / 2)), kMvThreads, smem, st, mD, mE, a);
}

}  // namespace

const char* mv_variant_name(int form) {
    return form == F_DEFL ? "deflated matrix f16x3 bf16x4" : (form == F_COMP ? "comp matrix bf16x6" : "f64 matrix bf16x8");
}

cudaError_t launch_mv_scenarios(const double* v64, int n_steps, int n_scen, int s_pad, float2* D, const MvScen& c,
                                cudaStream_t st) {
    cudaError_t e;
    if ((e = cudaMemsetAsync(c.stat, 0, 2 * sizeof(int32_t), st)) != cudaSuccess) return e;
    if ((e = cudaMemsetAsync(c.colexp, 0x80, (size_t)s_pad * sizeof(int32_t), st)) != cudaSuccess) return e;   // very small
    if ((e = cudaMemsetAsync(c.colmin, 0x7F, (size_t)s_pad * sizeof(int32_t), st)) != cudaSuccess) return e;   // very large
    mv_products_kernel<<<s_pad / kProdS, dim3(kProdS, 32), 0, st>>>(v64, n_steps, s_pad, D);
    mv_tilt_kernel<<<n_steps, 128, 0, st>>>(D, n_scen, s_pad, c.tau, c.stat);
    mv_columns_kernel<<<dim3(s_pad / 32, (n_steps + 63) / 64), dim3(32, 8), 0, st>>>(D, c.tau, n_steps, n_scen, s_pad, c.colexp,
                                                                                  c.colmin);
    mv_finish_kernel<<<(s_pad + 1023) / 1024 + 1, 1024, 0, st>>>(c.tau, n_steps, n_scen, s_pad, c.colexp, c.colmin, c.stat,
                                                                c.tilt, c.tilt_top);
    return cudaGetLastError();
}

cudaError_t launch_mv_digits(int ns, const float2* D, const int32_t* tau, const int32_t* colexp, int n_steps, int n_scen,
                             int s_pad, int pitch, void* digits, cudaStream_t st) {
    const dim3 grid(s_pad / 32, pitch / 64);
    uint32_t* out = static_cast<uint32_t*>(digits);
    auto k = ns == 3 ? mv_digits_kernel<3> : (ns == 4 ? mv_digits_kernel<4> : mv_digits_kernel<6>);
    k<<<grid, 256, 0, st>>>(D, tau, colexp, n_steps, n_scen, s_pad, pitch, out);
    return cudaGetLastError();
}

cudaError_t launch_mv_products64(const double* v64, int n_steps, int s_pad, double* D, cudaStream_t st) {
    mv_products_kernel<<<s_pad / kProdS, dim3(kProdS, 32), 0, st>>>(v64, n_steps, s_pad, D);
    return cudaGetLastError();
}

cudaError_t launch_mv_digits64(const double* D, const int32_t* tau, const int32_t* colexp, int n_steps, int n_scen, int s_pad,
                               int pitch, void* digits, cudaStream_t st) {
    mv_digits64_kernel<<<dim3(s_pad / 32, pitch / 64), 256, 0, st>>>(D, tau, colexp, n_steps, n_scen, s_pad, pitch,
                                                                    static_cast<uint32_t*>(digits));
    return cudaGetLastError();
}

cudaError_t launch_mv_build64(const MvBuild& b, const CfPol* pols, cudaStream_t st) {
    mv_build64_kernel<<<b.n_tiles * (kMvP / 8), 256, (size_t)b.pitch * sizeof(float), st>>>(b, pols);
    return cudaGetLastError();
}

cudaError_t launch_mv_build(int ns, const MvBuild& b, cudaStream_t st) {
    const int grid = b.n_tiles * (kMvP / (8 * b.rows_per_warp));
    const size_t smem = (size_t)b.pitch * sizeof(float);
    auto k = ns == 3 ? mv_build_kernel<3> : (ns == 4 ? mv_build_kernel<4> : mv_build_kernel<6>);
    k<<<grid, 256, smem, st>>>(b);
    return cudaGetLastError();
}

cudaError_t launch_mv_build_lives(const CfTables& T, const MvLives* recs, const double* amount, int n_tiles, int pitch,
                                  int n_steps, const float* tilt, void* digits, MvOut* out, cudaStream_t st) {
    mv_build_lives_kernel<6><<<n_tiles * (kMvP / 8), 256, (size_t)pitch * sizeof(float), st>>>(T, recs, amount, pitch, n_steps,
                                                                                            tilt, digits, out);
    return cudaGetLastError();
}

cudaError_t launch_mv_product(int ns, const MvArgs& a, const void* digitsD, const void* digitsE, int pitchD, int pitchE,
                              int sm_count, cudaStream_t st) {
    if (a.n_tiles <= 0 || a.n_chunks <= 0) return cudaSuccess;
    if (ns == 3) return product<3>(a, digitsD, digitsE, pitchD, pitchE, sm_count, st);
    if (ns == 4) return product<4>(a, digitsD, digitsE, pitchD, pitchE, sm_count, st);
    if (ns == 6) return product<6>(a, digitsD, digitsE, pitchD, pitchE, sm_count, st);
    return product<8>(a, digitsD, digitsE, pitchD, pitchE, sm_count, st);
}

}  // namespace rsv

// cashflow.cuh -- expected cash flows of a portfolio.
//
// With deterministic mortality the reserve is linear in the discount products:
// Eq. (basicReserveSummation) collects, for each step t, the probability-weighted
// cash flow E_p(t) of policy p at the end of step t, and
//   r_p = sum_t D(t + 1) E_p(t) + D(S) B_p,     D(t + 1) = v_0 ... v_t,
// with B_p the expected boundary payment (endowments).  E_p(t) does not depend on
// the scenario, so it is evaluated here once per (policy, step), in closed form
// from a table of survivors, with no serial chain over the steps:
//   x_t = Pr[life 1 alive at the start of step t], y_t life 2; deaths dx_t = x_t q
//   K_ANN   x_{t+1}
//   K_ASS   dx_t
//   K_ANN2  x_{t+1} y_{t+1}
//   K_ASS2  dx_t y_t + x_{t+1} dy_t                      (= x_t y_t - x_{t+1} y_{t+1})
//   K_JL    x_{t+1} + rho y_{t+1} (1 - x_{t+1});  x_{t+1} in state 01, rho y_{t+1} in state 10
//   K_LS2   dx_t dy_t + dx_t (1 - y_t) + (1 - x_t) dy_t; dx_t in state 1, dy_t in state 2
#pragma once

#include "rsv_device.cuh"

namespace rsv {

// Survivor columns of the decrement tables, [n_tab][rows] each: m_k = the product
// of the one-month survival probabilities below age k, leaving out zeros, scaled
// by 2^512 whenever it falls below 2^-512 (ex counts the scalings); dm_k = m_k q_k;
// z_k = the first age >= k whose survival is zero.  A life aged x is alive at the
// start of step t with probability m_{x+t} / m_x 2^(-512 (ex_{x+t} - ex_x)) for
// x + t <= z_x and 0 beyond, whatever the table: zeros inside it, lives past its
// end, products below the FP64 range.
struct CfTables {
    const double* m;
    const double* dm;
    const int32_t* z;
    const int32_t* ex;
    const double* inv;  // 1 / m
    const float2* m2;   // m and dm as FP32 head and tail
    const float2* dm2;
    int32_t rows;       // entries of one table
    int32_t scaled;     // 1: some ex_k > 0
};

// One life of a policy: its column at valuation and the steps it can live through.
struct CfLife {
    double inv;     // 1 / m_x
    int32_t i;      // index of m_x
    int32_t last;   // z_x - x
    int32_t ex, pad;
};

struct CfPol {      // 96 bytes
    CfLife a, b;
    double rho, amount, bnd;
    int32_t kind, S, state0, pol;
};

__device__ __forceinline__ double cf_scaled(const CfTables& T, const CfLife& l, int t, double v) {
    if (!T.scaled) return v;
    const int d = T.ex[l.i + t] - l.ex;
    return d == 0 ? v : (d == 1 ? v * 0x1p-512 : 0.0);
}
__device__ __forceinline__ double cf_alive(const CfTables& T, const CfLife& l, int t) {
    return t <= l.last ? cf_scaled(T, l, t, T.m[l.i + t] * l.inv) : 0.0;
}
__device__ __forceinline__ double cf_deaths(const CfTables& T, const CfLife& l, int t) {
    return t <= l.last ? cf_scaled(T, l, t, T.dm[l.i + t] * l.inv) : 0.0;
}

// E_p(t) per unit amount, 0 <= t < S
__device__ __forceinline__ double cf_expected(const CfTables& T, const CfPol& p, int t) {
    switch (p.kind) {
    case K_ANN: return cf_alive(T, p.a, t + 1);
    case K_ASS: return cf_deaths(T, p.a, t);
    case K_ANN2: return cf_alive(T, p.a, t + 1) * cf_alive(T, p.b, t + 1);
    case K_ASS2: return cf_deaths(T, p.a, t) * cf_alive(T, p.b, t) + cf_alive(T, p.a, t + 1) * cf_deaths(T, p.b, t);
    case K_JL: {
        const double x = p.state0 == 2 ? 0.0 : cf_alive(T, p.a, t + 1);
        const double y = p.state0 == 1 ? 0.0 : cf_alive(T, p.b, t + 1);
        return x + p.rho * y * (1.0 - x);
    }
    default: {
        if (p.state0 == 1) return cf_deaths(T, p.a, t);
        if (p.state0 == 2) return cf_deaths(T, p.b, t);
        const double dx = cf_deaths(T, p.a, t), dy = cf_deaths(T, p.b, t);
        return dx * dy + dx * (1.0 - cf_alive(T, p.b, t)) + (1.0 - cf_alive(T, p.a, t)) * dy;
    }
    }
}

// B_p per unit amount: the maturity payment's probability at S
__device__ __forceinline__ double cf_boundary(const CfTables& T, const CfPol& p) {
    if (p.bnd == 0.0) return 0.0;
    const double x = cf_alive(T, p.a, p.S);
    if (p.kind == K_ASS) return p.bnd * x;
    const double y = cf_alive(T, p.b, p.S);
    if (p.kind == K_ASS2) return p.bnd * x * y;
    return p.bnd * (p.state0 == 1 ? x : (p.state0 == 2 ? y : x + y * (1.0 - x)));
}

// Records of n layout slots, per_kind of them to a tile (a kind).
cudaError_t launch_cf_records(const CfTables& T, const SlotRec* slots, const int32_t* kinds, const double* amount, int n,
                              int per_kind, int tab_pad, CfPol* out, cudaStream_t st);

// The portfolio's cash flows: with A(t) = sum_p amount_p E_p(t) and M(t) the sum of
// amount_p B_p over the policies with S = t,
//   flow[t] = A(t) + M(t + 1), t < n_steps;   due[t] = M(t), t <= n_steps
// in FP64, in a fixed order; flow2 is flow / scale[0] as FP32 head and tail, scale[0] the
// power of two that makes the largest of them less than 1 (1 if all are zero).
// part: scratch of 2 * kCfSplits * (n_steps + 1) doubles.
constexpr int kCfSplits = 64;
cudaError_t launch_cf_portfolio(const CfTables& T, const CfPol* pols, int n, int n_steps, double* part, double* flow,
                                double* due, float2* flow2, double* scale, cudaStream_t st);

}  // namespace rsv

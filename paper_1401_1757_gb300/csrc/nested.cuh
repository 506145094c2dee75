// nested.cuh -- arguments and launchers of the nested valuation kernels.
#pragma once

#include <cstddef>
#include <cstdint>

#include <cuda_runtime.h>

namespace rsv {

// Constants of one exact monthly Vasicek step of (r, integral of r):
// I = b dt + (r - b) k1 + l21 z1 + l22 z2, r' = b + (r - b) e + l11 z1.
struct VasStep {
    double e, k1, l11, l21, l22, b, dt;
};
VasStep vasicek_step_constants(double a, double b, double sigma, double dt);
// o_first: the global index of the first outer path (the key of its random
// streams); outputs and r_node are indexed from 0.
cudaError_t launch_outer_paths(const VasStep& s, uint64_t seed, int o_first, int n_outer, int n_nodes, int node_step, double r0,
                               double* r_node, double* d0, cudaStream_t st);
// Tables of the inner-path generator's Box-Muller step (FP64): (sin, cos) of
// 2 pi j / BM_SC for j < BM_SC, then for the BM_LG intervals of the logarithm
// (1/c_j to 18 significant bits, -ln(2^k_j / c_j)); built once on the host.
constexpr int BM_SC = 1024, BM_LG = 128;
constexpr int BM_LG_K0 = 53;   // first interval whose centre 1 + (j + 1/2)/128 exceeds sqrt 2
const double2* bm_tables_host();   // BM_SC + BM_LG entries

// One nested run: sizes, model, and device arrays.  o_first is the global index of
// the first outer path; r_node, L_all and the outputs are indexed from 0.
struct NestedRun {
    uint64_t seed;
    double a, b, sigma, r0;
    int32_t o_first, n_outer, n_nodes, node_step, n_inner;
    int32_t n_steps;          // the portfolio's longest projection from valuation
    const double* r_node;     // [n_outer][n_nodes]
    const void* tables;       // upload_nested_tables
    const double* flow;       // launch_cf_portfolio's outputs
    const float2* flow2;
    const double* scale;
    const double* due;
    double* L_all;            // [n_outer][n_nodes][n_inner]
};
size_t nested_table_bytes();
cudaError_t upload_nested_tables(void* dst, cudaStream_t st);
// Whether the double-float generator covers the run's model.
bool nested_df_range(const NestedRun& q);
cudaError_t launch_nested_paths(const VasStep& s, const NestedRun& q, bool use_df, cudaStream_t st);
// The curve mode; ab: n_steps entries of scratch.
cudaError_t launch_nested_curve(const NestedRun& q, double2* ab, cudaStream_t st);
cudaError_t launch_node_stats(const double* L_all, int n_on, int n_inner, int k, double* mean, double* kth,
                              cudaStream_t st);

}  // namespace rsv

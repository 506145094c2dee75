// cashflow.cu -- survivor columns, policy records and portfolio sums of the
// expected cash flows (see cashflow.cuh).
#include <algorithm>
#include <vector>

#include "cashflow.cuh"
#include "ctx.cuh"

namespace rsv {
namespace {

__global__ void cf_records_kernel(const CfTables T, const SlotRec* __restrict__ slots, const int32_t* __restrict__ kinds,
                                  const double* __restrict__ amount, int n, int per_kind, int tab_pad,
                                  CfPol* __restrict__ out) {
    const int f = blockIdx.x * blockDim.x + threadIdx.x;
    if (f >= n) return;
    const SlotRec r = slots[f];
    auto life = [&](int idx) {
        CfLife l;
        l.i = (idx / tab_pad) * T.rows + idx % tab_pad;
        l.inv = T.inv[l.i];
        l.last = T.z[l.i] - idx % tab_pad;
        l.ex = T.ex[l.i];
        l.pad = 0;
        return l;
    };
    CfPol p;
    p.a = life(r.idx1);
    p.b = life(r.idx2);
    p.rho = (double)r.rho_h + (double)r.rho_l;
    p.pol = r.pol;
    p.amount = r.pol >= 0 ? amount[r.pol] : 0.0;
    p.bnd = r.bnd;
    p.kind = kinds[f / per_kind];
    p.S = r.S;
    p.state0 = r.state0;
    out[f] = p;
}

// Thread t of split blockIdx.y adds A(t) and M(t) over its share of the policies.
// The FP64 pipe is the bound (1 to 8 operations a policy and step, 1/64 of the
// FP32 rate), so the splits spread a small book over the chip: 2,000 annuities of
// up to 720 steps are 6 x 64 blocks.
__global__ void cf_sum_kernel(const CfTables T, const CfPol* __restrict__ pols, int n, int n_steps,
                              double* __restrict__ part) {
    const int t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t > n_steps) return;
    const int lo = (int)((long long)n * blockIdx.y / kCfSplits), hi = (int)((long long)n * (blockIdx.y + 1) / kCfSplits);
    double A = 0.0, M = 0.0;
    for (int f = lo; f < hi; ++f) {
        const CfPol& p = pols[f];
        if (t < p.S) A = __fma_rn(p.amount, cf_expected(T, p, t), A);
        else if (t == p.S && p.bnd != 0.0) M = __fma_rn(p.amount, cf_boundary(T, p), M);
    }
    double* row = part + (size_t)blockIdx.y * 2 * (n_steps + 1);
    row[t] = A;
    row[n_steps + 1 + t] = M;
}

__global__ void __launch_bounds__(1024) cf_finish_kernel(const double* __restrict__ part, int n_steps,
                                                         double* __restrict__ flow, double* __restrict__ due,
                                                         float2* __restrict__ flow2, double* __restrict__ scale) {
    __shared__ double top[1024];
    const int rows = n_steps + 1;
    for (int t = threadIdx.x; t < rows; t += blockDim.x) {
        double M = 0.0;
        for (int k = 0; k < kCfSplits; ++k) M += part[(size_t)k * 2 * rows + rows + t];
        due[t] = M;
    }
    __syncthreads();
    double mx = 0.0;
    for (int t = threadIdx.x; t < n_steps; t += blockDim.x) {
        double A = due[t + 1];
        for (int k = 0; k < kCfSplits; ++k) A += part[(size_t)k * 2 * rows + t];
        flow[t] = A;
        mx = fmax(mx, fabs(A));
    }
    top[threadIdx.x] = mx;
    __syncthreads();
    for (int w = blockDim.x / 2; w > 0; w >>= 1) {
        if (threadIdx.x < w) top[threadIdx.x] = fmax(top[threadIdx.x], top[threadIdx.x + w]);
        __syncthreads();
    }
    int ex = 0;
    if (top[0] > 0.0 && top[0] < INFINITY) frexp(top[0], &ex);
    ex = max(-1000, min(1000, ex));   // both scalings finite
    const double s = ldexp(1.0, ex), r = ldexp(1.0, -ex);
    if (threadIdx.x == 0) scale[0] = s;
    for (int t = threadIdx.x; t < n_steps; t += blockDim.x) {
        const double c = flow[t] * r;
        const float h = __double2float_rn(c);
        flow2[t] = make_float2(h, __double2float_rn(c - (double)h));
    }
}

}  // namespace

cudaError_t launch_cf_records(const CfTables& T, const SlotRec* slots, const int32_t* kinds, const double* amount, int n,
                              int per_kind, int tab_pad, CfPol* out, cudaStream_t st) {
    if (n <= 0) return cudaSuccess;
    cf_records_kernel<<<(n + 127) / 128, 128, 0, st>>>(T, slots, kinds, amount, n, per_kind, tab_pad, out);
    return cudaGetLastError();
}

cudaError_t launch_cf_portfolio(const CfTables& T, const CfPol* pols, int n, int n_steps, double* part, double* flow,
                                double* due, float2* flow2, double* scale, cudaStream_t st) {
    const dim3 grid((n_steps + 1 + 127) / 128, kCfSplits);
    cf_sum_kernel<<<grid, 128, 0, st>>>(T, pols, n, n_steps, part);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    cf_finish_kernel<<<1, 1024, 0, st>>>(part, n_steps, flow, due, flow2, scale);
    return cudaGetLastError();
}

// The survivor columns of every loaded table, on the device (once per change of the
// tables): kMaxAgeSteps + 1 entries each, the reach of any projection.
rsv_status cf_tables(rsv_ctx* c, CfTables& T) {
    int n_tab = 0;
    for (int t = 0; t < kMaxTables; ++t)
        if (!c->tab[t].empty()) n_tab = t + 1;
    const int rows = kMaxAgeSteps + 1;
    const size_t n = (size_t)n_tab * rows;
    if (c->cf_tab_gen != c->tab_gen) {
        // m, dm, the two integer columns, 1 / m, then m and dm as FP32 head and tail
        std::vector<double>& h = c->h_cf_tab;
        h.resize(6 * n);
        int32_t* z = reinterpret_cast<int32_t*>(h.data() + 2 * n);
        int32_t* ex = z + n;
        c->cf_tab_scaled = 0;
        for (int t = 0; t < n_tab; ++t) {
            const std::vector<double>& p = c->tab[t];
            double m = 1.0;
            int e = 0;
            for (int k = 0; k < rows; ++k) {
                const size_t i = (size_t)t * rows + k;
                const double pk = k < (int)p.size() ? p[k] : 0.0;
                h[i] = m;
                h[n + i] = m * (1.0 - pk);
                ex[i] = e;
                if (pk > 0.0) m *= pk;
                while (m < 0x1p-512) {
                    m *= 0x1p512;
                    ++e;
                }
            }
            if (e) c->cf_tab_scaled = 1;
            int next = rows;   // survival is zero from the table's end on
            for (int k = rows - 1; k >= 0; --k) {
                if (!(k < (int)p.size() && p[k] > 0.0)) next = k;
                z[(size_t)t * rows + k] = next;
            }
        }
        float2* pair = reinterpret_cast<float2*>(h.data() + 4 * n);
        for (size_t i = 0; i < n; ++i) h[3 * n + i] = 1.0 / h[i];
        for (size_t i = 0; i < 2 * n; ++i) {
            const float hi = (float)h[i];
            pair[i] = make_float2(hi, (float)(h[i] - (double)hi));
        }
        CU(c->d_cf_tab.ensure(h.size() * sizeof(double)));
        CU(cudaMemcpyAsync(c->d_cf_tab.p, h.data(), h.size() * sizeof(double), cudaMemcpyHostToDevice, c->stream));
        c->cf_tab_gen = c->tab_gen;
    }
    T.m = c->d_cf_tab.as<double>();
    T.dm = T.m + n;
    T.z = reinterpret_cast<const int32_t*>(T.dm + n);
    T.ex = T.z + n;
    T.inv = T.m + 3 * n;
    T.m2 = reinterpret_cast<const float2*>(T.m + 4 * n);
    T.dm2 = T.m2 + n;
    T.rows = rows;
    T.scaled = c->cf_tab_scaled;
    return RSV_OK;
}

}  // namespace rsv

// mlp.cu -- the reserve surrogate network on sm_103a: a 32 -> 256 -> 256 ->
// 256 -> 256 -> 1 perceptron with GELU (tanh form), BF16 weights and
// activations, FP32 accumulation, FP32 master weights and Adam.
//
// Forward per layer l = 1..4:  Z_l = A_{l-1} W_l + b_l,  A_l = gelu(Z_l)
// (A_0 = features), head y = A_4 w5 + b5.  Loss: mean squared error.
// The activations the tensor cores read are BF16; the head reads the last
// hidden layer in FP32, since BF16 rounding of its 256 inputs alone would put
// ~1e-3 of noise on the output, the size of the surrogate's error target.
// Backward: dZ_4 = (dy w5^T) * gelu'(Z_4); for l = 4..1: dW_l = A_{l-1}^T dZ_l,
// db_l = column sums of dZ_l, dZ_{l-1} = (dZ_l W_l^T) * gelu'(Z_{l-1}).
// Every product runs on the tensor cores (mlp_gemm.cuh); sums over the batch
// are in a fixed order, so a step is deterministic.
#include <algorithm>
#include <cmath>
#include <cstdint>
#include <vector>

#include "launch_next.cuh"
#include "mlp.cuh"

namespace rsv {

// parameter offsets in the flat FP32 vector
size_t mlp_w_off(int l) {   // l = 1..4
    size_t o = 0;
    for (int i = 1; i < l; ++i) o += (size_t)mlp_in_dim(i) * MLP_H + MLP_H;
    return o;
}
size_t mlp_b_off(int l) { return mlp_w_off(l) + (size_t)mlp_in_dim(l) * MLP_H; }
size_t mlp_w5_off() { return mlp_w_off(5); }
size_t mlp_n_params() { return mlp_w5_off() + MLP_H + 1; }

namespace {

// The kernels of a training pass follow one another by launch_next: nine of 3 to 18 us, a
// gradient at 8,192 rows 195 us with ordinary launches, 187 us so.
template <bool AK, bool BK, int EPI>
cudaError_t gemm(const GemmArgs& g, cudaStream_t st) {
    dim3 grid((g.N + GBN - 1) / GBN, (g.M + GBM - 1) / GBM);
    return launch_next(gemm_bf16_kernel<AK, BK, EPI>, grid, GTHREADS, 0, st, g);
}

// y[r] = gelu(Z4[r]) . w5 + b5
__global__ void head_fwd_kernel(const float* __restrict__ Z4, const float* __restrict__ w5,
                                const float* __restrict__ b5, int B, float* __restrict__ y) {
    grid_dependency_wait();
    const int lane = threadIdx.x & 31, r = blockIdx.x * 8 + (threadIdx.x >> 5);
    if (r >= B) return;
    float s = 0.0f;
    for (int k = lane; k < MLP_H; k += 32) s += gelu_f(Z4[(size_t)r * MLP_H + k]) * w5[k];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    if (lane == 0) y[r] = s + b5[0];
}

// The head with a target, forward and backward in one pass over Z4: y[r], the error's
// derivative dy[r] = 2 (y - t) / B, dZ4[r][k] = dy[r] w5[k] gelu'(Z4[r][k]), and each block's sums
// over its rows of dy A4 (dw5), dZ4 (db4), dy (db5) and the squared error, [block][kHeadCols].
// A warp takes a row, a lane eight of its columns.  Bound by the reads of Z4 (8 MB at
// 8,192 rows): 8 us, where the separate passes took 35.
constexpr int kHeadRows = 32, kHeadCols = 2 * MLP_H + 2;

__global__ void __launch_bounds__(256) head_train_kernel(const float* __restrict__ Z4, const float* __restrict__ w5,
                                                         const float* __restrict__ b5, const float* __restrict__ target,
                                                         int B, float* __restrict__ y, float* __restrict__ dZf,
                                                         __nv_bfloat16* __restrict__ dZb, float* __restrict__ part) {
    grid_dependency_wait();
    __shared__ float red[8][kHeadCols];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    float w[8], dw[8] = {}, db[8] = {}, sdy = 0.0f, sq = 0.0f;
#pragma unroll
    for (int j = 0; j < 8; ++j) w[j] = w5[lane + 32 * j];
    const int r0 = blockIdx.x * kHeadRows;
    for (int r = r0 + warp; r < min(B, r0 + kHeadRows); r += 8) {
        float z[8], a[8], s = 0.0f;
#pragma unroll
        for (int j = 0; j < 8; ++j) z[j] = Z4[(size_t)r * MLP_H + lane + 32 * j];
#pragma unroll
        for (int j = 0; j < 8; ++j) {   // in head_fwd_kernel's order: the same y
            a[j] = gelu_f(z[j]);
            s += a[j] * w[j];
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
        s += b5[0];
        const float e = s - target[r], dy = 2.0f * e / (float)B;
        if (lane == 0 && y) y[r] = s;
        sdy += dy;
        sq += e * e;
#pragma unroll
        for (int j = 0; j < 8; ++j) {
            const float g = dy * w[j] * gelu_grad_f(z[j]);
            const size_t o = (size_t)r * MLP_H + lane + 32 * j;
            dw[j] += dy * a[j];
            db[j] += g;
            dZb[o] = __float2bfloat16_rn(g);
            if (dZf) dZf[o] = g;
        }
    }
#pragma unroll
    for (int j = 0; j < 8; ++j) {
        const int k = lane + 32 * j;
        red[warp][k] = dw[j];
        red[warp][MLP_H + k] = db[j];
    }
    if (lane == 0) {
        red[warp][2 * MLP_H] = sdy;
        red[warp][2 * MLP_H + 1] = sq;
    }
    __syncthreads();
    for (int k = threadIdx.x; k < kHeadCols; k += 256) {
        float s = 0.0f;
#pragma unroll
        for (int i = 0; i < 8; ++i) s += red[i][k];
        part[(size_t)blockIdx.x * kHeadCols + k] = s;
    }
}

// dW_l = A_{l-1}^T dZ_l of the four layers over pieces of the batch: blockIdx.x the tile (four of
// layer 1, sixteen of each other), blockIdx.y the piece; part [piece][kWgradRows][256].  A
// weight gradient has 64 x 256 or 256 x 256 entries and the batch as its K: a block a tile
// and layer left 136 of the 152 SMs idle beside chains of K / 32 stages (456 us for the four
// at 8,192 rows); the four together in pieces: 18 us.
struct WgradArgs {
    const __nv_bfloat16* A[4];    // [batch][64 or 256]
    const __nv_bfloat16* dZ[4];   // [batch][256]
    float* part;
    int batch, piece;             // rows of a piece (a multiple of 32)
};
constexpr int kWgradTiles = 4 + 3 * 16, kWgradRows = 64 + 3 * 256;

__global__ void __launch_bounds__(GTHREADS) wgrad_kernel(const WgradArgs g) {
    grid_dependency_wait();
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int t = blockIdx.x < 4 ? blockIdx.x : blockIdx.x - 4, l = blockIdx.x < 4 ? 0 : 1 + t / 16;
    const int m0 = l == 0 ? 0 : t % 16 / 4 * GBM, n0 = t % 4 * GBN, width = l == 0 ? 64 : 256;
    const int k0 = blockIdx.y * g.piece, k1 = min(g.batch, k0 + g.piece);
    float acc[2][4][4];
    gemm_tile<false, false>(g.A[l], g.dZ[l], width, 256, width, 256, m0, n0, k0, k1, acc);
    float* out = g.part + ((size_t)blockIdx.y * kWgradRows + (l == 0 ? 0 : 64 + (l - 1) * 256)) * 256;
    const int wm = (warp >> 1) * 32, wn = (warp & 1) * 32;
#pragma unroll
    for (int mi = 0; mi < 2; ++mi)
#pragma unroll
        for (int nj = 0; nj < 4; ++nj)
#pragma unroll
            for (int h = 0; h < 2; ++h)
                *reinterpret_cast<float2*>(out + (size_t)(m0 + wm + mi * 16 + (lane >> 2) + h * 8) * 256 + n0 + wn + nj * 8 +
                                           (lane & 3) * 2) = make_float2(acc[mi][nj][h * 2], acc[mi][nj][h * 2 + 1]);
}

// The gradients from the partial sums, each in a fixed order: blocks 0 .. kGradW - 1 four
// weights a thread over the pieces of the batch (layer 1: the hi and the lo rows' of the tied
// weights); then the column sums, 32 columns a block and eight runs of rows, of
// the layers 1 to 3 (biases) and of the head.  Bound by the reads of the pieces (14 MB at
// 8,192 rows): 8 us.
constexpr int kGradW = (MLP_IN + 3 * MLP_H) * (MLP_H / 4) / 256;
constexpr int kGradB = 3 * MLP_H / 32, kGradH = (kHeadCols + 31) / 32;

struct GradArgs {
    const float* wpart;      // [n_pieces][kWgradRows][256]
    const float* cpart[3];   // [n_tiles][256], layers 1 to 3
    const float* hpart;      // [n_head][kHeadCols]
    int n_pieces, n_tiles, n_head;
    float* grads;
    size_t w_off[5], b_off[4];
    float* loss;
};

__global__ void __launch_bounds__(256) grad_kernel(const GradArgs g) {
    grid_dependency_wait();
    if (blockIdx.x < kGradW) {
        const int i = blockIdx.x * 256 + threadIdx.x, row = i / (MLP_H / 4), c = i % (MLP_H / 4);   // row of W1 .. W4
        const int l = row < MLP_IN ? 0 : 1 + (row - MLP_IN) / MLP_H, src = row < MLP_IN ? row : row + MLP_XW - MLP_IN;
        const float4* p = reinterpret_cast<const float4*>(g.wpart) + (size_t)src * (MLP_H / 4) + c;
        constexpr size_t ld = (size_t)kWgradRows * (MLP_H / 4);
        float4 s = make_float4(0.0f, 0.0f, 0.0f, 0.0f), t = s;
        auto add = [](float4& a, const float4 b) {
            a.x += b.x;
            a.y += b.y;
            a.z += b.z;
            a.w += b.w;
        };
#pragma unroll 8
        for (int k = 0; k < g.n_pieces; ++k) add(s, p[k * ld]);
        if (l == 0) {
#pragma unroll 8
            for (int k = 0; k < g.n_pieces; ++k) add(t, p[k * ld + MLP_IN * (MLP_H / 4)]);
            add(s, t);
        }
        const int first = l == 0 ? 0 : MLP_IN + (l - 1) * MLP_H;
        float* out = g.grads + g.w_off[l] + (size_t)(row - first) * MLP_H + c * 4;
        out[0] = s.x;
        out[1] = s.y;
        out[2] = s.z;
        out[3] = s.w;
        return;
    }
    __shared__ float red[8][32];
    const int b = blockIdx.x - kGradW, lane = threadIdx.x & 31, run = threadIdx.x >> 5;
    const bool head = b >= kGradB;
    const int l = head ? 3 : b / (MLP_H / 32), col = (head ? b - kGradB : b % (MLP_H / 32)) * 32 + lane;
    const int n = head ? g.n_head : g.n_tiles, ld = head ? kHeadCols : MLP_H;
    const float* p = head ? g.hpart : g.cpart[l];
    float s = 0.0f;
    if (col < ld) {
#pragma unroll 8
        for (int r = run; r < n; r += 8) s += p[(size_t)r * ld + col];
    }
    red[run][lane] = s;
    __syncthreads();
    if (run > 0 || col >= ld) return;
    s = 0.0f;
#pragma unroll
    for (int i = 0; i < 8; ++i) s += red[i][lane];
    if (!head) g.grads[g.b_off[l] + col] = s;
    else if (col < MLP_H) g.grads[g.w_off[4] + col] = s;
    else if (col < 2 * MLP_H) g.grads[g.b_off[3] + col - MLP_H] = s;
    else if (col == 2 * MLP_H) g.grads[g.w_off[4] + MLP_H] = s;
    else *g.loss = s;
}

// Rows of a piece of the batch in the weight gradients: 512, so that 8,192 rows give
// 832 blocks of 16 stages each, and at most kMaxPieces pieces.
constexpr int kPieceRows = 512, kMaxPieces = 32;
int piece_rows(int batch) {
    const int even = (batch + kMaxPieces - 1) / kMaxPieces;
    return std::max(kPieceRows, (even + GBK - 1) / GBK * GBK);
}
int n_pieces_max(int batch) { return std::min(kMaxPieces, (batch + kPieceRows - 1) / kPieceRows); }

// Adam on the FP32 master weights; refresh the BF16 working copies.
__global__ void adam_kernel(float* __restrict__ p, const float* __restrict__ g, float* __restrict__ m,
                            float* __restrict__ v, size_t n, float lr, float b1, float b2, float eps, float c1,
                            float c2) {
    for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x) {
        const float gi = g[i];
        const float mi = b1 * m[i] + (1.0f - b1) * gi;
        const float vi = b2 * v[i] + (1.0f - b2) * gi * gi;
        m[i] = mi;
        v[i] = vi;
        p[i] -= lr * (mi / c1) / (sqrtf(vi / c2) + eps);
    }
}

__global__ void to_bf16_kernel(const float* __restrict__ x, __nv_bfloat16* __restrict__ y, size_t n) {
    for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x)
        y[i] = __float2bfloat16_rn(x[i]);
}

// [W1; W1] in BF16 from the FP32 W1 [MLP_IN][MLP_H]
__global__ void tied_w1_kernel(const float* __restrict__ w1, __nv_bfloat16* __restrict__ y) {
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < MLP_IN * MLP_H; i += gridDim.x * blockDim.x) {
        const __nv_bfloat16 b = __float2bfloat16_rn(w1[i]);
        y[i] = b;
        y[MLP_IN * MLP_H + i] = b;
    }
}

}  // namespace

cudaError_t Mlp::ensure(int batch) {
    if (batch <= cap) return cudaSuccess;
    cap = 0;   // until every buffer has grown
    const size_t B = (size_t)batch;
    const size_t P = mlp_n_params();
    cudaError_t e;
#define ALLOC(ptr, bytes)                                       \
    do {                                                        \
        if (ptr) cudaFree(ptr);                                 \
        ptr = nullptr;                                          \
        e = cudaMalloc((void**)&ptr, (bytes));                  \
        if (e != cudaSuccess) {                                 \
            cudaGetLastError();                                 \
            return e;                                           \
        }                                                       \
    } while (0)
    if (!params) {   // the last of them
        ALLOC(grads, P * 4);
        ALLOC(adam_m, P * 4);
        ALLOC(adam_v, P * 4);
        ALLOC(wbf, (size_t)MLP_XW * MLP_H * 2 + 3 * (size_t)MLP_H * MLP_H * 2);
        cudaMemset(adam_m, 0, P * 4);
        cudaMemset(adam_v, 0, P * 4);
        ALLOC(params, P * 4);
    }
    ALLOC(X, B * MLP_XW * 2);
    for (int l = 0; l < 4; ++l) {
        ALLOC(Z[l], B * MLP_H * 4);
        ALLOC(A[l], B * MLP_H * 2);
        ALLOC(dZf[l], B * MLP_H * 4);
        ALLOC(dZb[l], B * MLP_H * 2);
    }
    ALLOC(y, B * 4);
    ALLOC(t, B * 4);
    ALLOC(wpart, (size_t)n_pieces_max(batch) * kWgradRows * MLP_H * 4);
    ALLOC(cpart, 3 * (B / GBM + 1) * MLP_H * 4);
    ALLOC(hpart, (B / kHeadRows + 1) * kHeadCols * 4);
    ALLOC(loss, 4);
#undef ALLOC
    cap = batch;
    return cudaSuccess;
}

cudaError_t Mlp::ensure_infer(int batch) {
    if (batch <= cap_i) return cudaSuccess;
    if (Xi) cudaFree(Xi);
    if (yi) cudaFree(yi);
    Xi = nullptr;
    yi = nullptr;
    cap_i = 0;
    cudaError_t e = cudaMalloc((void**)&Xi, (size_t)batch * MLP_XW * 2);
    if (e != cudaSuccess) return e;
    if ((e = cudaMalloc((void**)&yi, (size_t)batch * 4)) != cudaSuccess) return e;
    cap_i = batch;
    return cudaSuccess;
}

void Mlp::release() {
    void* ps[] = {params, grads, adam_m, adam_v, wbf, X, y, t, wpart, cpart, hpart, loss, wt, Xi, yi};
    for (void* p : ps)
        if (p) cudaFree(p);
    for (int l = 0; l < 4; ++l) {
        if (Z[l]) cudaFree(Z[l]);
        if (A[l]) cudaFree(A[l]);
        if (dZf[l]) cudaFree(dZf[l]);
        if (dZb[l]) cudaFree(dZb[l]);
    }
    *this = Mlp();
}

__nv_bfloat16* Mlp::wb(int l) const {   // BF16 copy of W_l as the GEMM reads it, [k][H]
    size_t o = 0;
    for (int i = 1; i < l; ++i) o += (size_t)mlp_k_dim(i) * MLP_H;
    return wbf + o;
}

cudaError_t Mlp::refresh_bf16(cudaStream_t st) {
    wt_fresh = false;
    tied_w1_kernel<<<32, 256, 0, st>>>(params + mlp_w_off(1), wb(1));
    for (int l = 2; l <= 4; ++l) {
        const size_t n = (size_t)MLP_H * MLP_H;
        to_bf16_kernel<<<64, 256, 0, st>>>(params + mlp_w_off(l), wb(l), n);
    }
    return cudaGetLastError();
}

// X (BF16 [B][MLP_XW], batch a multiple of 64) -> y; with `target` also dZ_4 and the head's sums
// for backward.  trace: write A_4 (and dZ_4 in FP32) too, which no later pass reads.
cudaError_t Mlp::forward(const __nv_bfloat16* Xin, int B, float* yout, const float* target, cudaStream_t st, bool trace) {
    cudaError_t e;
    const __nv_bfloat16* in = Xin;
    for (int l = 1; l <= 4; ++l) {
        GemmArgs g{};
        g.A = in;
        g.B = wb(l);
        g.M = B;
        g.N = MLP_H;
        g.K = mlp_k_dim(l);
        g.lda = g.K;
        g.ldb = MLP_H;
        g.Cf = Z[l - 1];
        g.Cb = l < 4 || trace ? A[l - 1] : nullptr;
        g.bias = params + mlp_b_off(l);
        if ((e = gemm<true, false, EPI_BIAS_GELU>(g, st)) != cudaSuccess) return e;
        in = A[l - 1];
    }
    const float* w5 = params + mlp_w5_off();
    if (target)
        return launch_next(head_train_kernel, dim3((B + kHeadRows - 1) / kHeadRows), 256, 0, st, Z[3], w5, w5 + MLP_H, target, B,
                           yout, trace ? dZf[3] : nullptr, dZb[3], hpart);
    return launch_next(head_fwd_kernel, dim3((B + 7) / 8), 256, 0, st, Z[3], w5, w5 + MLP_H, B, yout);
}

// Gradients and the summed squared error of the last forward(X, B, ., target); trace: dZ_1 .. dZ_3
// in FP32 too.
cudaError_t Mlp::backward(const __nv_bfloat16* Xin, int B, cudaStream_t st, bool trace) {
    cudaError_t e;
    GradArgs r{};
    for (int l = 4; l >= 2; --l) {
        // dZ_{l-1} = (dZ_l W_l^T) * gelu'(Z_{l-1}) : B operand W_l stored [K][H] = [n][k]
        GemmArgs h{};
        h.A = dZb[l - 1];
        h.B = wb(l);
        h.M = B;
        h.N = MLP_H;
        h.K = MLP_H;
        h.lda = MLP_H;
        h.ldb = MLP_H;
        h.Cf = trace ? dZf[l - 2] : nullptr;
        h.Cb = dZb[l - 2];
        h.Zin = Z[l - 2];
        h.colpart = cpart + (size_t)(l - 2) * (cap / GBM + 1) * MLP_H;
        r.cpart[l - 2] = h.colpart;
        if ((e = gemm<true, true, EPI_GELU_BWD>(h, st)) != cudaSuccess) return e;
    }
    WgradArgs w{};
    for (int l = 1; l <= 4; ++l) {
        w.A[l - 1] = l > 1 ? A[l - 2] : Xin;
        w.dZ[l - 1] = dZb[l - 1];
    }
    w.part = wpart;
    w.batch = B;
    w.piece = piece_rows(B);
    const int n = (B + w.piece - 1) / w.piece;
    if ((e = launch_next(wgrad_kernel, dim3(kWgradTiles, n), GTHREADS, 0, st, w)) != cudaSuccess) return e;
    r.wpart = wpart;
    r.hpart = hpart;
    r.n_pieces = n;
    r.n_tiles = B / GBM;
    r.n_head = (B + kHeadRows - 1) / kHeadRows;
    r.grads = grads;
    for (int l = 1; l <= 5; ++l) {
        r.w_off[l - 1] = mlp_w_off(l);
        if (l < 5) r.b_off[l - 1] = mlp_b_off(l);
    }
    r.loss = loss;
    return launch_next(grad_kernel, dim3(kGradW + kGradB + kGradH), 256, 0, st, r);
}

cudaError_t Mlp::adam_step(float lr, cudaStream_t st) {
    ++step;
    const float b1 = 0.9f, b2 = 0.999f;
    const float c1 = 1.0f - std::pow(b1, (float)step), c2 = 1.0f - std::pow(b2, (float)step);
    adam_kernel<<<256, 256, 0, st>>>(params, grads, adam_m, adam_v, mlp_n_params(), lr, b1, b2, 1e-8f, c1, c2);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    return refresh_bf16(st);
}

}  // namespace rsv

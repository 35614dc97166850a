// Learned closure for the GSIS warm start: a 16 -> 128 -> 128 -> 128 -> 12 perceptron with
// GELU (erf form) hidden activations, BF16 weights for the forward and backward passes,
// FP32 accumulation and FP32 master weights updated by Adam (Kingma and Ba).
//
//  cell_features   per-cell inputs (state, gradient magnitudes, Kn, 1/Kn_p) and the
//                  normalised high-order-term targets of Eq. (getHoTs) at the cell
//  mlp_pass        all layers for a tile of rows in one kernel: forward, and in training the
//                  loss and the back-propagated dZ of every layer
//  weight_grad     dW = dZ^T A, db = sum dZ: 64 x 64 tiles over ranges of rows
//  grad_reduce     sums of the ranges' tiles and of the loss partials, in a fixed order
//  adam            FP32 master update and its BF16 copy
//  hot_from_cells  face high-order terms from predicted cell values (face average)
#include <algorithm>
#include <cmath>
#include <cuda_bf16.h>

#include "fp64.cuh"
#include "gsis_impl.cuh"

namespace gsis {

namespace {

__device__ __forceinline__ float gelu(float z) { return 0.5f * z * (1.0f + erff(z * 0.70710678118654752f)); }
__device__ __forceinline__ float gelu_grad(float z) {
    return 0.5f * (1.0f + erff(z * 0.70710678118654752f)) + z * expf(-0.5f * z * z) * 0.39894228040143268f;
}

}  // namespace

namespace {

constexpr int layer_in(int l) { return l == 0 ? MLP_IN : MLP_H; }
constexpr int layer_out(int l) { return l == MLP_LAYERS - 1 ? MLP_OUT : MLP_H; }
constexpr int w_off(int l) {
    int o = 0;
    for (int k = 0; k < l; ++k) o += layer_out(k) * layer_in(k) + layer_out(k);
    return o;
}
// Shared memory of mlp_pass: the four BF16 weight matrices with rows padded by 8 bytes (a
// row's next one starts two banks on: 8-byte reads of 32 rows meet every bank twice), then
// per warp PR rows of activations, of dZ (value-major, the PR rows side by side) and of the
// pre-activations of the three hidden layers.
constexpr int PR = 4;                                    // rows of a warp (a float4 of dZ)
constexpr int ws_stride(int l) { return layer_in(l) + 4; }
constexpr int ws_off(int l) {
    int o = 0;
    for (int k = 0; k < l; ++k) o += layer_out(k) * ws_stride(k);
    return o;
}
constexpr int WS_BYTES = (ws_off(MLP_LAYERS) * 2 + 15) / 16 * 16;
constexpr int WARP_FLOATS = PR * MLP_H * 5;
constexpr int N_BIAS = 3 * MLP_H + MLP_OUT;
constexpr int pass_smem(int warps, bool train) {
    return WS_BYTES + (N_BIAS + 3) / 4 * 16 + warps * (train ? WARP_FLOATS : PR * MLP_H) * 4;
}

__device__ __forceinline__ void copy8_async(void *smem, const void *global) {
    asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"((uint32_t)__cvta_generic_to_shared(smem)), "l"(global)
                 : "memory");
}
__device__ __forceinline__ float lo_bf16(uint32_t u) { return __uint_as_float(u << 16); }
__device__ __forceinline__ float hi_bf16(uint32_t u) { return __uint_as_float(u & 0xffff0000u); }

}  // namespace

// One tile of WARPS * PR rows at a time through every layer; a warp keeps its PR rows to
// itself, so only the staged weights are shared.  Forward: lane = output (lane + 32 j), the
// sum over inputs in two interleaved FP32 chains on the packed FP32x2 pipe; backward: lane =
// four consecutive inputs.  Reads act0 [n][16] (standardised) and T; writes Y [n][12], and in
// training act1..3 [n][128], dZ0..3 [n][128 | 12] and the CTA's loss.
// Bound by the instructions that feed the FP32 pipe (an 8-byte weight read and two
// conversions serve PR rows); one thread per output with both operands from shared memory
// per FMA, a kernel per layer and a serial weight gradient before: 2 048 rows, loss and
// gradient 1.56 -> 0.107 ms end to end, of which this kernel takes 25 us.
template <int WARPS, bool TRAIN>
__global__ void __launch_bounds__(32 * WARPS) k_mlp_pass(int n, const __nv_bfloat16 *__restrict__ W,
                                                         const float *__restrict__ P, const float *__restrict__ act0,
                                                         float *__restrict__ Y, float *__restrict__ A1,
                                                         float *__restrict__ A2, float *__restrict__ A3,
                                                         const float *__restrict__ T, float *__restrict__ D0,
                                                         float *__restrict__ D1, float *__restrict__ D2,
                                                         float *__restrict__ D3, double *__restrict__ lpart) {
    extern __shared__ __align__(16) unsigned char mlp_smem[];
    __nv_bfloat16 *Ws = reinterpret_cast<__nv_bfloat16 *>(mlp_smem);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    float *Bs = reinterpret_cast<float *>(mlp_smem + WS_BYTES);     // biases
    float *A = Bs + (N_BIAS + 3) / 4 * 4 + warp * (TRAIN ? WARP_FLOATS : PR * MLP_H);
    float *D = A + PR * MLP_H;                 // [o][PR]
    float *Z = D + PR * MLP_H;                 // [3][PR][MLP_H]
    float *const Aout[3] = {A1, A2, A3};
    float *const Dout[4] = {D0, D1, D2, D3};
#pragma unroll
    for (int l = 0; l < MLP_LAYERS; ++l) {     // weights, four at a time
        const int in4 = layer_in(l) / 4;
        const uint2 *src = reinterpret_cast<const uint2 *>(W + w_off(l));
        for (int k = threadIdx.x; k < layer_out(l) * in4; k += 32 * WARPS)
            copy8_async(Ws + ws_off(l) + k / in4 * ws_stride(l) + k % in4 * 4, src + k);
    }
    for (int k = threadIdx.x; k < N_BIAS; k += 32 * WARPS) {
        const int l = k / MLP_H;
        Bs[k] = P[w_off(l) + layer_out(l) * layer_in(l) + k % MLP_H];
    }
    asm volatile("cp.async.wait_all;" ::: "memory");
    __syncthreads();
    double loss = 0.0;
    const int tiles = (n + WARPS * PR - 1) / (WARPS * PR);
    for (int tile = blockIdx.x; tile < tiles; tile += gridDim.x) {
        const int r0 = (tile * WARPS + warp) * PR;
        if (r0 >= n) continue;                  // the warp's rows only: no barrier below
        const int rows = min(PR, n - r0);
        __syncwarp();
        for (int k = lane; k < PR * MLP_IN; k += 32) {
            const int r = k / MLP_IN;
            A[r * MLP_H + k % MLP_IN] = r < rows ? act0[(size_t)r0 * MLP_IN + k] : 0.0f;
        }
        __syncwarp();
        // ---- hidden layers
#pragma unroll
        for (int l = 0; l < 3; ++l) {
            float2 acc[PR][4];
#pragma unroll
            for (int r = 0; r < PR; ++r)
#pragma unroll
                for (int j = 0; j < 4; ++j) acc[r][j] = make_float2(0.0f, 0.0f);
            const __nv_bfloat16 *w0 = Ws + ws_off(l) + lane * ws_stride(l);
#pragma unroll 2
            for (int k = 0; k < layer_in(l); k += 4) {
                float4 a[PR];
                uint2 w[4];
#pragma unroll
                for (int j = 0; j < 4; ++j) w[j] = *reinterpret_cast<const uint2 *>(w0 + 32 * j * ws_stride(l) + k);
#pragma unroll
                for (int r = 0; r < PR; ++r) a[r] = *reinterpret_cast<const float4 *>(A + r * MLP_H + k);
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    const float2 p = make_float2(lo_bf16(w[j].x), hi_bf16(w[j].x));
                    const float2 q = make_float2(lo_bf16(w[j].y), hi_bf16(w[j].y));
#pragma unroll
                    for (int r = 0; r < PR; ++r) {
                        acc[r][j] = __ffma2_rn(make_float2(a[r].x, a[r].y), p, acc[r][j]);
                        acc[r][j] = __ffma2_rn(make_float2(a[r].z, a[r].w), q, acc[r][j]);
                    }
                }
            }
            __syncwarp();
            const float *b = Bs + l * MLP_H;
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                const int o = lane + 32 * j;
                const float bo = b[o];
#pragma unroll
                for (int r = 0; r < PR; ++r) {
                    const float z = bo + (acc[r][j].x + acc[r][j].y), g = gelu(z);
                    A[r * MLP_H + o] = g;
                    if constexpr (TRAIN) {
                        Z[(l * PR + r) * MLP_H + o] = z;
                        if (r < rows) Aout[l][(size_t)(r0 + r) * MLP_H + o] = g;
                    }
                }
            }
            __syncwarp();
        }
        // ---- output layer: 12 x PR values over the lanes
        for (int k = lane; k < PR * MLP_OUT; k += 32) {
            const int r = k / MLP_OUT, o = k % MLP_OUT;
            const __nv_bfloat16 *w0 = Ws + ws_off(3) + o * ws_stride(3);
            float2 acc = make_float2(0.0f, 0.0f);
#pragma unroll 4
            for (int i = 0; i < MLP_H; i += 4) {
                const uint2 w = *reinterpret_cast<const uint2 *>(w0 + i);
                const float4 a = *reinterpret_cast<const float4 *>(A + r * MLP_H + i);
                acc = __ffma2_rn(make_float2(a.x, a.y), make_float2(lo_bf16(w.x), hi_bf16(w.x)), acc);
                acc = __ffma2_rn(make_float2(a.z, a.w), make_float2(lo_bf16(w.y), hi_bf16(w.y)), acc);
            }
            const float y = Bs[3 * MLP_H + o] + (acc.x + acc.y);
            if (!TRAIN && r < rows) Y[(size_t)(r0 + r) * MLP_OUT + o] = y;
            if constexpr (TRAIN) {
                // loss and dZ = 2 (Y - T) / (n 12); rows past the end carry nothing
                float dz = 0.0f;
                if (r < rows) {
                    const float d = y - T[(size_t)(r0 + r) * MLP_OUT + o];
                    dz = 2.0f * d / (float)((double)n * MLP_OUT);
                    const double d8 = to_double(d);
                    loss = fma(d8, d8, loss);
                    D3[(size_t)(r0 + r) * MLP_OUT + o] = dz;
                }
                D[o * PR + r] = dz;
            }
        }
        if constexpr (TRAIN) {
            // ---- backward: dA_l = dZ_l W_l, dZ_{l-1} = dA_l GELU'(Z_{l-1})
#pragma unroll
            for (int l = 3; l > 0; --l) {
                __syncwarp();
                float2 acc[PR][2];
#pragma unroll
                for (int r = 0; r < PR; ++r) acc[r][0] = acc[r][1] = make_float2(0.0f, 0.0f);
                const __nv_bfloat16 *w0 = Ws + ws_off(l) + 4 * lane;
#pragma unroll 4
                for (int o = 0; o < layer_out(l); ++o) {
                    const uint2 w = *reinterpret_cast<const uint2 *>(w0 + o * ws_stride(l));
                    const float4 d = *reinterpret_cast<const float4 *>(D + o * PR);
                    const float2 p = make_float2(lo_bf16(w.x), hi_bf16(w.x)), q = make_float2(lo_bf16(w.y), hi_bf16(w.y));
                    const float dd[PR] = {d.x, d.y, d.z, d.w};
#pragma unroll
                    for (int r = 0; r < PR; ++r) {
                        acc[r][0] = __ffma2_rn(make_float2(dd[r], dd[r]), p, acc[r][0]);
                        acc[r][1] = __ffma2_rn(make_float2(dd[r], dd[r]), q, acc[r][1]);
                    }
                }
                __syncwarp();
                float4 dz[PR];
#pragma unroll
                for (int r = 0; r < PR; ++r) {
                    const float4 z = *reinterpret_cast<const float4 *>(Z + ((l - 1) * PR + r) * MLP_H + 4 * lane);
                    dz[r] = make_float4(acc[r][0].x * gelu_grad(z.x), acc[r][0].y * gelu_grad(z.y),
                                        acc[r][1].x * gelu_grad(z.z), acc[r][1].y * gelu_grad(z.w));
                    if (r < rows)
                        *reinterpret_cast<float4 *>(Dout[l - 1] + (size_t)(r0 + r) * MLP_H + 4 * lane) = dz[r];
                }
                float4 *Dv = reinterpret_cast<float4 *>(D) + 4 * lane;
                Dv[0] = make_float4(dz[0].x, dz[1].x, dz[2].x, dz[3].x);
                Dv[1] = make_float4(dz[0].y, dz[1].y, dz[2].y, dz[3].y);
                Dv[2] = make_float4(dz[0].z, dz[1].z, dz[2].z, dz[3].z);
                Dv[3] = make_float4(dz[0].w, dz[1].w, dz[2].w, dz[3].w);
            }
        }
    }
    if constexpr (TRAIN) {
        __shared__ double part[WARPS];
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) loss += __shfl_xor_sync(0xffffffffu, loss, o);
        if (lane == 0) part[warp] = loss;
        __syncthreads();
        if (threadIdx.x == 0) {
            double sum = 0.0;
            for (int w = 0; w < WARPS; ++w) sum += part[w];
            lpart[blockIdx.x] = sum;
        }
    }
}

// dW = dZ^T A and db = sum dZ of the rows [split chunk, + chunk) of all layers:
// block = (64 x 64 tile of one layer's weights, split); part [split][MLP_NW] laid out as the
// parameters.  256 threads, 4 x 4 weights each, rows staged 16 at a time.
constexpr int WG_TILES = 12;      // 128 x 16: 2, 128 x 128: 4 each, 12 x 128: 2
struct GradArgs {
    const float *A[MLP_LAYERS], *D[MLP_LAYERS];
};
__global__ void __launch_bounds__(256) k_weight_grad(int n, int chunk, GradArgs g, float *__restrict__ part) {
    constexpr int KB = 16;
    __shared__ __align__(16) float sA[KB][64], sD[KB][64];
    const int t = blockIdx.x;
    const int l = t < 2 ? 0 : t < 6 ? 1 : t < 10 ? 2 : 3, u = t < 2 ? t : t < 6 ? t - 2 : t < 10 ? t - 6 : t - 10;
    const int o0 = l == 0 ? u * 64 : l == 3 ? 0 : (u >> 1) * 64, i0 = l == 0 ? 0 : l == 3 ? u * 64 : (u & 1) * 64;
    const int in = layer_in(l), out = layer_out(l);
    const float *__restrict__ A = g.A[l], *__restrict__ Dz = g.D[l];
    const int r0 = blockIdx.y * chunk, r1 = min(n, r0 + chunk);
    const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;       // inputs 4 tx.., outputs 4 ty..
    float2 acc[4][2];
    float bias[4] = {0.0f, 0.0f, 0.0f, 0.0f};
#pragma unroll
    for (int a = 0; a < 4; ++a) acc[a][0] = acc[a][1] = make_float2(0.0f, 0.0f);
    const int lr = threadIdx.x >> 4, lc = (threadIdx.x & 15) * 4;  // staging: row, first of four columns
    for (int r = r0; r < r1; r += KB) {
        float4 a = make_float4(0.0f, 0.0f, 0.0f, 0.0f), d = a;
        if (r + lr < r1) {
            if (i0 + lc < in) a = *reinterpret_cast<const float4 *>(A + (size_t)(r + lr) * in + i0 + lc);
            if (o0 + lc < out) d = *reinterpret_cast<const float4 *>(Dz + (size_t)(r + lr) * out + o0 + lc);
        }
        __syncthreads();
        *reinterpret_cast<float4 *>(&sA[lr][lc]) = a;
        *reinterpret_cast<float4 *>(&sD[lr][lc]) = d;
        __syncthreads();
#pragma unroll
        for (int k = 0; k < KB; ++k) {
            const float4 x = *reinterpret_cast<const float4 *>(&sA[k][4 * tx]), y = *reinterpret_cast<const float4 *>(&sD[k][4 * ty]);
            const float yy[4] = {y.x, y.y, y.z, y.w};
#pragma unroll
            for (int o = 0; o < 4; ++o) {
                const float2 dd = make_float2(yy[o], yy[o]);
                acc[o][0] = __ffma2_rn(dd, make_float2(x.x, x.y), acc[o][0]);
                acc[o][1] = __ffma2_rn(dd, make_float2(x.z, x.w), acc[o][1]);
                bias[o] += yy[o];
            }
        }
    }
    float *p = part + (size_t)blockIdx.y * MLP_NW + (l == 0 ? w_off(0) : l == 1 ? w_off(1) : l == 2 ? w_off(2) : w_off(3));
#pragma unroll
    for (int o = 0; o < 4; ++o) {
        const int oo = o0 + 4 * ty + o;
        if (oo >= out) continue;
        if (i0 + 4 * tx < in)
            *reinterpret_cast<float4 *>(p + (size_t)oo * in + i0 + 4 * tx) =
                make_float4(acc[o][0].x, acc[o][0].y, acc[o][1].x, acc[o][1].y);
        if (i0 == 0 && tx == 0) p[(size_t)out * in + oo] = bias[o];
    }
}

// g = sum of the splits' tiles; block 0 also sums the loss partials into lpart[0]
__global__ void __launch_bounds__(128) k_grad_reduce(int splits, const float *__restrict__ part, float *__restrict__ g,
                                                     int n_loss, double *__restrict__ lpart, double scale) {
    const int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k < MLP_NW) {
        float s = 0.0f;
        for (int q = 0; q < splits; ++q) s += part[(size_t)q * MLP_NW + k];
        g[k] = s;
    }
    if (blockIdx.x != 0 || threadIdx.x >= 32) return;
    double x = 0.0;
    for (int q = threadIdx.x; q < n_loss; q += 32) x += lpart[q];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
    if (threadIdx.x == 0) lpart[n_loss] = x * scale;
}

__global__ void k_adam(size_t n, float *__restrict__ p, const float *__restrict__ g, float *__restrict__ m1,
                       float *__restrict__ m2, __nv_bfloat16 *__restrict__ pb, float lr, float c1, float c2) {
    const size_t k = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= n) return;
    const float gk = g[k];
    const float a = 0.9f * m1[k] + 0.1f * gk;
    const float v = 0.999f * m2[k] + 0.001f * gk * gk;
    m1[k] = a;
    m2[k] = v;
    const float x = p[k] - lr * (a / c1) / (sqrtf(v / c2) + 1e-8f);
    p[k] = x;
    if (pb) pb[k] = __float2bfloat16_rn(x);
}

__global__ void k_to_bf16(size_t n, const float *__restrict__ p, __nv_bfloat16 *__restrict__ pb) {
    const size_t k = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (k < n) pb[k] = __float2bfloat16_rn(p[k]);
}

// x <- (x - mean) / std per column (inverse when inv != 0)
__global__ void k_standardise(size_t n, int m, float *__restrict__ X, const float *__restrict__ mean,
                              const float *__restrict__ sd, int inv) {
    const size_t k = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= n * m) return;
    const int c = (int)(k % m);
    X[k] = inv ? X[k] * sd[c] + mean[c] : (X[k] - mean[c]) / sd[c];
}

// ------------------------------------------------------------------ cell features / targets
// Inputs (16): rho, u_x, u_y, T_t, T_r, T_v, T_R, |grad| of rho, u_x, u_y, T_t, T_r, T_v,
// T_R (the e_R gradient over 16 sigma_R T_R^3), Kn, 1/Kn_p.  Targets (12): HoT_sigma
// (xx, xy, yy, zz) / (rho T_t) and HoT_q (t, r, v, R) x (x, y) / (rho T_t^1.5), with the
// NSF part from the cell's least-squares gradients (Eqs. NSF_constitutive,
// NSF_thermal_conductivities) and the kinetic part from the field record.
template <int DIM>
__global__ void k_cell_features(MacroGeom g, ModelDev m, const double *__restrict__ F, const double *__restrict__ q,
                                const double *__restrict__ grad, float *__restrict__ X, float *__restrict__ Y) {
    constexpr int E = 1 + DIM, ER = 4 + DIM;
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= g.n_cells) return;
    const double *qi = q + (size_t)i * NVM, *r = F + (size_t)i * NF;
    auto gr = [&](int d, int v) { return grad[((size_t)i * MGS + d) * NVM + v]; };
    auto mag = [&](int v) {
        double s = 0.0;
        for (int d = 0; d < DIM; ++d) s += gr(d, v) * gr(d, v);
        return sqrt(s);
    };
    const double rho = qi[0], Tt = qi[E], TR = r[7];
    float *x = X + (size_t)i * MLP_IN;
    for (int k = 0; k < MLP_IN; ++k) x[k] = 0.0f;
    x[0] = (float)rho;
    for (int a = 0; a < DIM; ++a) x[1 + a] = (float)qi[1 + a];
    x[3] = (float)Tt;
    x[4] = (float)qi[E + 1];
    x[5] = (float)qi[E + 2];
    x[6] = (float)TR;
    x[7] = (float)mag(0);
    for (int a = 0; a < DIM; ++a) x[8 + a] = (float)mag(1 + a);
    x[10] = (float)mag(E);
    x[11] = (float)mag(E + 1);
    x[12] = (float)mag(E + 2);
    x[13] = (float)(mag(ER) / (16.0 * m.sigma_R * TR * TR * TR));
    x[14] = (float)m.Kn;
    x[15] = (float)(1.0 / m.Kn_p);
    if (!Y) return;
    const double mu = sqrt(2.0 / 3.14159265358979323846) * m.Kn * pow(Tt, m.omega);
    double div = 0.0;
    for (int d = 0; d < DIM; ++d) div += gr(d, 1 + d);
    auto sig_nsf = [&](int a, int b) {
        double S = (a < DIM && b < DIM) ? gr(b, 1 + a) + gr(a, 1 + b) : 0.0;
        return -mu * (S - (a == b ? 2.0 / 3.0 * div : 0.0));
    };
    const double A[9] = {m.A[0], m.A[1], m.A[2], m.A[3], m.A[4], m.A[5], m.A[6], m.A[7], m.A[8]};
    const double det = A[0] * (A[4] * A[8] - A[5] * A[7]) - A[1] * (A[3] * A[8] - A[5] * A[6]) +
                       A[2] * (A[3] * A[7] - A[4] * A[6]);
    const double Ai[3][3] = {{(A[4] * A[8] - A[5] * A[7]) / det, (A[2] * A[7] - A[1] * A[8]) / det,
                              (A[1] * A[5] - A[2] * A[4]) / det},
                             {(A[5] * A[6] - A[3] * A[8]) / det, (A[0] * A[8] - A[2] * A[6]) / det,
                              (A[2] * A[3] - A[0] * A[5]) / det},
                             {(A[3] * A[7] - A[4] * A[6]) / det, (A[1] * A[6] - A[0] * A[7]) / det,
                              (A[0] * A[4] - A[1] * A[3]) / det}};
    const double dg[3] = {5.0, m.d_r, m.d_v};
    const double srT = rho * Tt, sq = rho * Tt * sqrt(Tt);
    float *y = Y + (size_t)i * MLP_OUT;
    for (int k = 0; k < MLP_OUT; ++k) y[k] = 0.0f;
    y[0] = (float)((r[20] - sig_nsf(0, 0)) / srT);
    y[1] = (float)((r[23] - sig_nsf(0, 1)) / srT);
    y[2] = (float)((r[21] - sig_nsf(1, 1)) / srT);
    y[3] = (float)((r[22] - sig_nsf(2, 2)) / srT);
    for (int md = 0; md < 3; ++md)
        for (int d = 0; d < DIM; ++d) {
            double s = 0.0;
            for (int nn = 0; nn < 3; ++nn) s += Ai[md][nn] * dg[nn] * gr(d, E + nn);
            y[4 + 2 * md + d] = (float)((r[8 + 3 * md + d] + 0.5 * mu * s) / sq);
        }
    const double kR = 1.0 / (3.0 * (m.k_eff_density_scaled ? rho / m.Kn_p : 1.0 / m.Kn_p));
    for (int d = 0; d < DIM; ++d) y[10 + d] = (float)((r[17 + d] + kR * gr(d, ER)) / sq);
}

// face high-order terms on the face normal from predicted cell values (de-normalised,
// averaged over the two cells), laid out as k_macro_hot's; the boundary terms are zero
template <int DIM>
__global__ void k_hot_from_cells(MacroGeom g, const float *__restrict__ Yc, double *__restrict__ hot,
                                 float *__restrict__ hotf, double *__restrict__ hot_b) {
    constexpr int E = 1 + DIM;
    const int t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t < g.n_fi) {
        double h[DIM + 4];
        for (int k = 0; k < DIM + 4; ++k) h[k] = 0.0;
        const double *n = g.d.fgeo + (size_t)t * FGEO;
        const int cells[2] = {g.fi4[t].x, g.fi4[t].y};
        for (int c : cells) {
            const double rho = g.d.q[(size_t)c * NVM], Tt = g.d.q[(size_t)c * NVM + E];
            const double srT = 0.5 * rho * Tt, sq = 0.5 * rho * Tt * sqrt(Tt);
            const float *y = Yc + (size_t)c * MLP_OUT;
            const int sidx[2][2] = {{0, 1}, {1, 2}};
            for (int a = 0; a < DIM; ++a)
                for (int b = 0; b < DIM; ++b) h[a] += srT * y[sidx[a][b]] * n[b];
            for (int md = 0; md < 4; ++md)
                for (int d = 0; d < DIM; ++d) h[DIM + md] += sq * y[4 + 2 * md + d] * n[d];
        }
        for (int k = 0; k < DIM + 4; ++k) {
            hot[(size_t)t * NVM + k] = h[k];
            if (hotf) hotf[(size_t)t * NVM + k] = (float)h[k];
        }
        return;
    }
    const int b = t - g.n_fi;
    if (b < g.n_bf)
        for (int k = 0; k < NVM; ++k) hot_b[(size_t)b * NVM + k] = 0.0;
}

}  // namespace gsis

// ------------------------------------------------------------------ launchers
namespace gsis {

namespace {

// One CTA per SM at most: 4 warps (16 rows a tile) while that keeps every SM busy, else 8.
template <bool TRAIN>
cudaError_t mlp_pass(cudaStream_t s, MlpDev &d, int n, int *ctas) {
    const int rows4 = 4 * PR, n4 = (n + rows4 - 1) / rows4;
    auto run = [&](auto kern, int warps) {
        const int tiles = (n + warps * PR - 1) / (warps * PR), smem = pass_smem(warps, TRAIN);
        cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
        if (e != cudaSuccess) return e;
        *ctas = std::min(tiles, MLP_CTAS);
        kern<<<*ctas, 32 * warps, smem, s>>>(n, static_cast<const __nv_bfloat16 *>(d.pb), d.p, d.act[0],
                                             d.act[MLP_LAYERS], d.act[1], d.act[2], d.act[3], d.T, d.dZ[0], d.dZ[1],
                                             d.dZ[2], d.dZ[3], d.lpart);
        return cudaGetLastError();
    };
    return n4 <= MLP_CTAS ? run(k_mlp_pass<4, TRAIN>, 4) : run(k_mlp_pass<8, TRAIN>, 8);
}

}  // namespace

// act[0] (standardised) -> act[4]
cudaError_t launch_mlp_forward(cudaStream_t s, MlpDev &d, int n) {
    int ctas = 0;
    return mlp_pass<false>(s, d, n, &ctas);
}

// act[0] and T -> gradients g and the mean squared error in lpart[d.loss_at]
cudaError_t launch_mlp_loss_backward(cudaStream_t s, MlpDev &d, int n) {
    int ctas = 0;
    cudaError_t e = mlp_pass<true>(s, d, n, &ctas);
    if (e) return e;
    const int splits = std::min(MLP_SPLITS, (n + 127) / 128), chunk = (n + splits - 1) / splits;
    GradArgs g;
    for (int l = 0; l < MLP_LAYERS; ++l) {
        g.A[l] = d.act[l];
        g.D[l] = d.dZ[l];
    }
    k_weight_grad<<<dim3(WG_TILES, splits), 256, 0, s>>>(n, chunk, g, d.gpart);
    if ((e = cudaGetLastError())) return e;
    k_grad_reduce<<<(MLP_NW + 127) / 128, 128, 0, s>>>(splits, d.gpart, d.g, ctas, d.lpart,
                                                       1.0 / ((double)n * MLP_OUT));
    d.loss_at = ctas;
    return cudaGetLastError();
}

cudaError_t launch_mlp_adam(cudaStream_t s, MlpDev &d, float lr) {
    d.step += 1;
    const float c1 = 1.0f - powf(0.9f, (float)d.step), c2 = 1.0f - powf(0.999f, (float)d.step);
    k_adam<<<(MLP_NW + 255) / 256, 256, 0, s>>>(MLP_NW, d.p, d.g, d.m1, d.m2, static_cast<__nv_bfloat16 *>(d.pb), lr,
                                                c1, c2);
    return cudaGetLastError();
}

cudaError_t launch_mlp_to_bf16(cudaStream_t s, MlpDev &d) {
    k_to_bf16<<<(MLP_NW + 255) / 256, 256, 0, s>>>(MLP_NW, d.p, static_cast<__nv_bfloat16 *>(d.pb));
    return cudaGetLastError();
}

cudaError_t launch_mlp_standardise(cudaStream_t s, int n, int m, float *X, const float *mean, const float *sd,
                                   int inv) {
    const size_t cnt = (size_t)n * m;
    if (cnt == 0) return cudaSuccess;
    k_standardise<<<(unsigned)((cnt + 255) / 256), 256, 0, s>>>(n, m, X, mean, sd, inv);
    return cudaGetLastError();
}

__global__ void k_gather_rows(int n, int width, const int *__restrict__ idx, const float *__restrict__ src,
                              float *__restrict__ dst) {
    const size_t k = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= (size_t)n * width) return;
    const size_t r = k / width;
    dst[k] = src[(size_t)idx[r] * width + (k % width)];
}

cudaError_t launch_mlp_gather(cudaStream_t s, int n, int width, const int *idx, const float *src, float *dst) {
    const size_t cnt = (size_t)n * width;
    if (cnt == 0) return cudaSuccess;
    k_gather_rows<<<(unsigned)((cnt + 255) / 256), 256, 0, s>>>(n, width, idx, src, dst);
    return cudaGetLastError();
}

cudaError_t launch_cell_features(cudaStream_t s, const MacroGeom &g, const ModelDev &m, const double *F,
                                 const double *q, const double *grad, float *X, float *Y) {
    const int nb = (g.n_cells + 127) / 128;
    if (g.dim == 1) k_cell_features<1><<<nb, 128, 0, s>>>(g, m, F, q, grad, X, Y);
    else k_cell_features<2><<<nb, 128, 0, s>>>(g, m, F, q, grad, X, Y);
    return cudaGetLastError();
}

cudaError_t launch_hot_from_cells(cudaStream_t s, const MacroGeom &g, const float *Yc, const MacroWork &w,
                                  double *hot_b) {
    const int n = g.n_fi + g.n_bf, nb = (n + 127) / 128;
    if (n == 0) return cudaSuccess;
    if (g.dim == 1) k_hot_from_cells<1><<<nb, 128, 0, s>>>(g, Yc, w.hot, w.hotf, hot_b);
    else k_hot_from_cells<2><<<nb, 128, 0, s>>>(g, Yc, w.hot, w.hotf, hot_b);
    return cudaGetLastError();
}

}  // namespace gsis

// proposal.cu -- the learned proposal sampler (a project extension; the paper
// has none): a small MLP from gamma(x) (6 frequencies) through four ReLU
// layers of 64 units to a density, composited over stratified samples as
// Eq. 1, whose weights drive the inverse-CDF sampler in place of the coarse
// pass of the NeRF MLP.  It is distilled from the full hierarchical sampler:
// targets are the sampler's final weights re-binned onto the proposal's
// intervals, the loss is the cross-entropy of the normalised proposal
// weights, and training runs here in FP32 with Adam.
#include <math.h>
#include <string.h>

#include <algorithm>
#include <random>
#include <vector>

#include "stages.cuh"

namespace mcl {

constexpr int kPL = 6;                  // frequencies of gamma(x)
constexpr int kPIn = 3 + 6 * kPL;       // 39
constexpr int kPInPad = 40;
constexpr int kPW = 64;                 // width
constexpr int kPDepth = 4;
// blob offsets: P1 W[64][39] b[64], P2..P4 W[64][64] b[64], head w[64] b[1]
constexpr int kPOff1 = 0;
// offset of layer l (0-based); layers 1..3 are 64x64
__host__ __device__ constexpr int prop_off(int l) {
    return l == 0 ? 0 : kPW * kPIn + kPW + (l - 1) * (kPW * kPW + kPW);
}
constexpr int kPOffHead = kPW * kPIn + kPW + 3 * (kPW * kPW + kPW);
constexpr int kPN = kPOffHead + kPW + 1;  // 15105
static_assert(kPN == 15105, "proposal blob size");

// gamma(x) with 6 frequencies (identity, then sin / cos of 2^k x per axis).
__device__ __forceinline__ void prop_pe(const float x[3], float* g) {
    g[0] = x[0]; g[1] = x[1]; g[2] = x[2];
#pragma unroll
    for (int k = 0; k < kPL; ++k) {
        const float f = (float)(1 << k);
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            float sn, cs;
            sincosf(f * x[c], &sn, &cs);
            g[3 + 6 * k + c] = sn;
            g[6 + 6 * k + c] = cs;
        }
    }
}

// Forward of one point with weights in shared memory; g receives the encoding.
__device__ __forceinline__ float prop_point(const float* __restrict__ Wsh, const float x[3],
                                            float* __restrict__ g) {
    float in[kPW], out[kPW];
    prop_pe(x, g);
    // outer loops over output units are not unrolled (the inner dot products
    // are): the same arithmetic per unit, a fraction of the code size
#pragma unroll 1
    for (int o = 0; o < kPW; ++o) {
        const float* w = Wsh + kPOff1 + o * kPIn;
        float s = Wsh[kPOff1 + kPW * kPIn + o];
#pragma unroll
        for (int i = 0; i < kPIn; ++i) s = fmaf(w[i], g[i], s);
        in[o] = fmaxf(s, 0.0f);
    }
#pragma unroll
    for (int l = 1; l < kPDepth; ++l) {
        const float* W = Wsh + prop_off(l);
        const float* b = W + kPW * kPW;
#pragma unroll 1
        for (int o = 0; o < kPW; ++o) {
            float s = b[o];
#pragma unroll
            for (int i = 0; i < kPW; ++i) s = fmaf(W[o * kPW + i], in[i], s);
            out[o] = fmaxf(s, 0.0f);
        }
#pragma unroll
        for (int o = 0; o < kPW; ++o) in[o] = out[o];
    }
    float s = Wsh[kPOffHead + kPW];
#pragma unroll
    for (int i = 0; i < kPW; ++i) s = fmaf(Wsh[kPOffHead + i], in[i], s);
    return s;
}

__device__ __forceinline__ void load_weights_smem(const float* __restrict__ W, float* sh) {
    for (int i = threadIdx.x; i < kPN; i += blockDim.x) sh[i] = W[i];
    __syncthreads();
}

// Inference: raw proposal density of sample k of ray r (stratified midpoints
// z = near + (far - near)(k + 1/2)/n_p, written by raygen into z) into
// out[r * n_p + k].x.
__global__ void k_prop_infer(const float* __restrict__ W, const Ray* __restrict__ rays,
                             const float* __restrict__ z, int n_p, long n_rows,
                             const int* __restrict__ n_rays_dev, float4* __restrict__ out) {
    extern __shared__ float wsh[];
    load_weights_smem(W, wsh);
    const long rows = n_rays_dev ? min(n_rows, (long)*n_rays_dev * n_p) : n_rows;
    for (long row = (long)blockIdx.x * blockDim.x + threadIdx.x; row < rows;
         row += (long)gridDim.x * blockDim.x) {
        const Ray R = rays[row / n_p];
        const float zz = z[row];
        const float x[3] = {fmaf(zz, R.dx, R.ox), fmaf(zz, R.dy, R.oy), fmaf(zz, R.dz, R.oz)};
        float g[kPInPad];
        out[row] = make_float4(prop_point(wsh, x, g), 0.f, 0.f, 0.f);
    }
}

// ---------------------------------------------------------------- training
// Forward and backward data passes run as small GEMMs: a block of 256 threads
// takes tiles of 128 rows, the layer's operand lies in shared memory with the
// rows innermost ([k][row]), the weights with the outputs innermost, and a
// thread accumulates 8 rows x 4 outputs with packed FP32 FMAs on row pairs:
// three 16-byte loads for 16 instructions, where one thread per row loads a
// weight for every FMA.  Each output is the same chain of FMAs in the same
// order as prop_point's.  Bound by the FMA lanes and the stores of the saved
// rows (1.2 KB each).  Measured, 262,144 rows: forward 0.61 -> 0.24 ms,
// backward 0.86 -> 0.19 ms.
constexpr int kPTile = 128, kPLd = kPTile + 4;

// out[i] (rows 2 i, 2 i + 1 of ty's eight) [e] = fma chain over k of
// X[k][row] W[k][4 tx + e], starting from init.
__device__ __forceinline__ void prop_tile_gemm(const float* __restrict__ X, const float* __restrict__ W,
                                               int K, int tx, int ty, float2 (&acc)[4][4]) {
#pragma unroll 4
    for (int k = 0; k < K; ++k) {
        const float4 a0 = *reinterpret_cast<const float4*>(X + k * kPLd + 8 * ty);
        const float4 a1 = *reinterpret_cast<const float4*>(X + k * kPLd + 8 * ty + 4);
        const float4 w = *reinterpret_cast<const float4*>(W + k * kPW + 4 * tx);
        const float2 a[4] = {make_float2(a0.x, a0.y), make_float2(a0.z, a0.w),
                             make_float2(a1.x, a1.y), make_float2(a1.z, a1.w)};
        const float wv[4] = {w.x, w.y, w.z, w.w};
#pragma unroll
        for (int e = 0; e < 4; ++e) {
            const float2 we = make_float2(wv[e], wv[e]);
#pragma unroll
            for (int i = 0; i < 4; ++i) acc[i][e] = __ffma2_rn(we, a[i], acc[i][e]);
        }
    }
}

// Shared memory of the two passes (floats).
constexpr int kPFwdW = kPIn * kPW + 3 * kPW * kPW;            // weights [in][out] per layer
constexpr int kPFwdSmem = (kPFwdW + 4 * kPW + kPW + 4 + kPW * kPLd) * (int)sizeof(float);
constexpr int kPBwdSmem = (3 * kPW * kPW + kPW + kPW * kPLd) * (int)sizeof(float);

// Forward with saved encodings [rows][40] and activations [rows][4][64].
__global__ __launch_bounds__(256, 2) void k_prop_fwd_train(
    const float* __restrict__ W, const float* __restrict__ O, const float* __restrict__ D, int n_rays,
    int nb, float near_z, float far_z, float* __restrict__ gsave, float* __restrict__ hsave,
    float* __restrict__ s_out) {
    extern __shared__ __align__(16) float sh[];
    float* Wt = sh;                         // [39 | 64 | 64 | 64][64]
    float* bias = Wt + kPFwdW;              // [4][64]
    float* head = bias + 4 * kPW;           // [64], bias
    float* X = head + kPW + 4;              // [64][kPLd]
    const int t = threadIdx.x, tx = t & 15, ty = t >> 4;
    for (int l = 0; l < kPDepth; ++l) {
        const int fin = l == 0 ? kPIn : kPW;
        float* dst = Wt + (l == 0 ? 0 : kPIn * kPW + (l - 1) * kPW * kPW);
        for (int q = t; q < fin * kPW; q += 256) dst[(q % fin) * kPW + q / fin] = W[prop_off(l) + q];
        for (int q = t; q < kPW; q += 256) bias[l * kPW + q] = W[prop_off(l) + kPW * fin + q];
    }
    for (int q = t; q < kPW + 1; q += 256) head[q] = W[kPOffHead + q];
    const long rows = (long)n_rays * nb;
    for (long r0 = (long)blockIdx.x * kPTile; r0 < rows; r0 += (long)gridDim.x * kPTile) {
        __syncthreads();
        // encoding: two threads per row, the octaves k = h, h + 2, h + 4
        {
            const int rl = t & (kPTile - 1), h = t >> 7;
            const long row = min(r0 + rl, rows - 1);
            const long r = row / nb;
            const int k = (int)(row - r * nb);
            const float zz = near_z + (far_z - near_z) * ((float)k + 0.5f) / (float)nb;
            const float x[3] = {fmaf(zz, D[3 * r], O[3 * r]), fmaf(zz, D[3 * r + 1], O[3 * r + 1]),
                                fmaf(zz, D[3 * r + 2], O[3 * r + 2])};
            if (h == 0)
                for (int c = 0; c < 3; ++c) X[c * kPLd + rl] = x[c];
            else
                X[kPIn * kPLd + rl] = 0.0f;
#pragma unroll 1
            for (int q = h; q < kPL; q += 2) {
                const float f = (float)(1 << q);
#pragma unroll
                for (int c = 0; c < 3; ++c) {
                    float sn, cs;
                    sincosf(f * x[c], &sn, &cs);
                    X[(3 + 6 * q + c) * kPLd + rl] = sn;
                    X[(6 + 6 * q + c) * kPLd + rl] = cs;
                }
            }
        }
        __syncthreads();
        for (int q = t; q < kPTile * kPInPad; q += 256) {
            const int rl = q / kPInPad, i = q - rl * kPInPad;
            if (r0 + rl < rows) gsave[(r0 + rl) * kPInPad + i] = X[i * kPLd + rl];
        }
        for (int l = 0; l < kPDepth; ++l) {
            float2 acc[4][4];
#pragma unroll
            for (int e = 0; e < 4; ++e)
#pragma unroll
                for (int i = 0; i < 4; ++i) acc[i][e] = make_float2(bias[l * kPW + 4 * tx + e], bias[l * kPW + 4 * tx + e]);
            prop_tile_gemm(X, Wt + (l == 0 ? 0 : kPIn * kPW + (l - 1) * kPW * kPW), l == 0 ? kPIn : kPW, tx, ty, acc);
            __syncthreads();
            float v[8][4];
#pragma unroll
            for (int i = 0; i < 4; ++i)
#pragma unroll
                for (int e = 0; e < 4; ++e) {
                    v[2 * i][e] = fmaxf(acc[i][e].x, 0.0f);
                    v[2 * i + 1][e] = fmaxf(acc[i][e].y, 0.0f);
                }
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                float* x = X + (4 * tx + e) * kPLd + 8 * ty;
                *reinterpret_cast<float4*>(x) = make_float4(v[0][e], v[1][e], v[2][e], v[3][e]);
                *reinterpret_cast<float4*>(x + 4) = make_float4(v[4][e], v[5][e], v[6][e], v[7][e]);
            }
#pragma unroll
            for (int i = 0; i < 8; ++i)
                if (r0 + 8 * ty + i < rows)
                    *reinterpret_cast<float4*>(hsave + (r0 + 8 * ty + i) * (kPDepth * kPW) + l * kPW + 4 * tx) =
                        make_float4(v[i][0], v[i][1], v[i][2], v[i][3]);
            __syncthreads();
        }
        if (t < kPTile && r0 + t < rows) {
            float s = head[kPW];
#pragma unroll 8
            for (int i = 0; i < kPW; ++i) s = fmaf(head[i], X[i * kPLd + t], s);
            s_out[r0 + t] = s;
        }
    }
}

// Per ray: composite of the raw densities, cross-entropy against hist and
// dL/ds per sample (masked by s > 0):
//   g_j = -h_j / (p_j W) + sum_b h_b w_b / (p_b W^2),  p_b = w_b / W + 1e-8,
//   dL/dsigma_j = delta_j (g_j T_j (1 - alpha_j) - sum_{k>j} g_k w_k).
// A ray with no density (W = 0) contributes -log(1e-8) and no gradient.  A
// block takes kLossRays rays; the exponentials, logarithms and quotients are
// spread over its threads, and only the running products and sums, whose
// order is part of the result, are walked by one thread per ray (one thread
// per ray for everything left all but 32 blocks of the chip idle: 142 -> 36 us
// for 4,096 rays of 64 bins).
constexpr int kLossRays = 8, kLossThreads = 128;

__global__ __launch_bounds__(kLossThreads) void k_prop_loss_bwd(
    const float* __restrict__ s, const float* __restrict__ D, int n_rays, int nb, float near_z,
    float far_z, const float* __restrict__ hist, float scale, double lscale, float* __restrict__ ds,
    double* __restrict__ loss_acc) {
    extern __shared__ __align__(16) double shd[];
    const int ld = nb + 1;
    double* lp = shd;                                    // log p  [rays][nb + 1]
    float* al = reinterpret_cast<float*>(lp + kLossRays * ld);
    float* T = al + kLossRays * ld;
    float* w = T + kLossRays * ld;
    float* q = w + kLossRays * ld;                       // c's terms, then g_j, then the tails
    __shared__ float dn[kLossRays], Wt[kLossRays], cs[kLossRays];
    const int r0 = blockIdx.x * kLossRays, nr = min(kLossRays, n_rays - r0);
    const int t = threadIdx.x;
    const float dz = (far_z - near_z) / (float)nb;
    if (t < nr) {
        const float* d = D + 3 * (size_t)(r0 + t);
        dn[t] = sqrtf(d[0] * d[0] + d[1] * d[1] + d[2] * d[2]);
    }
    __syncthreads();
    const float* sr = s + (long)r0 * nb;
    const float* h = hist + (long)r0 * nb;
    float* dsr = ds + (long)r0 * nb;
    for (int i = t; i < nr * nb; i += kLossThreads) {
        const int r = i / nb, k = i - r * nb;
        const float delta = (k < nb - 1) ? dz * dn[r] : 1e10f;
        const float sg = fmaxf(sr[i], 0.0f);
        al[r * ld + k] = 1.0f - expf(-sg * delta);
    }
    __syncthreads();
    if (t < nr) {
        float trans = 1.0f, tot = 0.0f;
        for (int k = 0; k < nb; ++k) {
            const float a = al[t * ld + k];
            T[t * ld + k] = trans;
            const float wk = trans * a;
            w[t * ld + k] = wk;
            trans *= (1.0f - a);
            tot += wk;
        }
        Wt[t] = tot;
    }
    __syncthreads();
    for (int i = t; i < nr * nb; i += kLossThreads) {
        const int r = i / nb, k = r * ld + i - r * nb;
        if (Wt[r] > 0.0f) {
            const float p = w[k] / Wt[r] + 1e-8f;
            lp[k] = log((double)p);
            q[k] = h[i] * w[k] / (p * Wt[r] * Wt[r]);
        } else {
            lp[k] = log(1e-8);
        }
    }
    __syncthreads();
    double L = 0.0;
    if (t < nr) {
        float c = 0.0f;
        for (int b = 0; b < nb; ++b) {
            L -= (double)h[t * nb + b] * lp[t * ld + b];
            if (Wt[t] > 0.0f) c += q[t * ld + b];
        }
        cs[t] = c;
    }
    __syncthreads();
    for (int i = t; i < nr * nb; i += kLossThreads) {
        const int r = i / nb, k = r * ld + i - r * nb;
        if (Wt[r] > 0.0f) {
            const float p = w[k] / Wt[r] + 1e-8f;
            q[k] = -h[i] / (p * Wt[r]) + cs[r];
        }
    }
    __syncthreads();
    if (t < nr && Wt[t] > 0.0f) {
        // al <- the tail entering sample j
        float tail = 0.0f;
        for (int j = nb - 1; j >= 0; --j) {
            lp[t * ld + j] = (double)tail;
            tail += q[t * ld + j] * w[t * ld + j];
        }
    }
    __syncthreads();
    for (int i = t; i < nr * nb; i += kLossThreads) {
        const int r = i / nb, j = i - r * nb, k = r * ld + j;
        if (Wt[r] > 0.0f) {
            const float delta = (j < nb - 1) ? dz * dn[r] : 1e10f;
            const float tail = (float)lp[k];
            const float dsig = delta * (q[k] * T[k] * (1.0f - al[k]) - tail);
            dsr[i] = sr[i] > 0.0f ? dsig * scale : 0.0f;
        } else {
            dsr[i] = 0.0f;
        }
    }
    if (t < nr) atomicAdd(loss_acc, L * lscale);
}

// Backward data pass per sample: da_l = (W_{l+1}^T da_{l+1}) masked by
// h_l > 0, starting from da_4 = ds * head; saved as [rows][4][64].
__global__ __launch_bounds__(256, 2) void k_prop_bwd_data(const float* __restrict__ W,
                                                          const float* __restrict__ hsave,
                                                          const float* __restrict__ ds, long rows,
                                                          float* __restrict__ dasave) {
    extern __shared__ __align__(16) float sh[];
    float* Wl = sh;                       // layers 1..3: [out][in]
    float* head = Wl + 3 * kPW * kPW;     // [64]
    float* X = head + kPW;                // [64][kPLd]
    const int t = threadIdx.x, tx = t & 15, ty = t >> 4;
    for (int l = 1; l < kPDepth; ++l)
        for (int q = t; q < kPW * kPW; q += 256) Wl[(l - 1) * kPW * kPW + q] = W[prop_off(l) + q];
    for (int q = t; q < kPW; q += 256) head[q] = W[kPOffHead + q];
    for (long r0 = (long)blockIdx.x * kPTile; r0 < rows; r0 += (long)gridDim.x * kPTile) {
        __syncthreads();
        float v[8][4];
        // da_4 of the thread's 8 rows x 4 units
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            const long row = r0 + 8 * ty + i;
            const bool in = row < rows;
            const float d = in ? ds[row] : 0.0f;
            const float4 h = in ? *reinterpret_cast<const float4*>(hsave + row * (kPDepth * kPW) + (kPDepth - 1) * kPW + 4 * tx)
                                : make_float4(0.f, 0.f, 0.f, 0.f);
            v[i][0] = h.x > 0.0f ? d * head[4 * tx] : 0.0f;
            v[i][1] = h.y > 0.0f ? d * head[4 * tx + 1] : 0.0f;
            v[i][2] = h.z > 0.0f ? d * head[4 * tx + 2] : 0.0f;
            v[i][3] = h.w > 0.0f ? d * head[4 * tx + 3] : 0.0f;
        }
        for (int l = kPDepth - 1;; --l) {
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                float* x = X + (4 * tx + e) * kPLd + 8 * ty;
                *reinterpret_cast<float4*>(x) = make_float4(v[0][e], v[1][e], v[2][e], v[3][e]);
                *reinterpret_cast<float4*>(x + 4) = make_float4(v[4][e], v[5][e], v[6][e], v[7][e]);
            }
#pragma unroll
            for (int i = 0; i < 8; ++i)
                if (r0 + 8 * ty + i < rows)
                    *reinterpret_cast<float4*>(dasave + (r0 + 8 * ty + i) * (kPDepth * kPW) + l * kPW + 4 * tx) =
                        make_float4(v[i][0], v[i][1], v[i][2], v[i][3]);
            if (l == 0) break;
            __syncthreads();
            float2 acc[4][4];
#pragma unroll
            for (int i = 0; i < 4; ++i)
#pragma unroll
                for (int e = 0; e < 4; ++e) acc[i][e] = make_float2(0.f, 0.f);
            // (contracts over the outputs o of layer l: operand and weights [o][.])
            prop_tile_gemm(X, Wl + (l - 1) * kPW * kPW, kPW, tx, ty, acc);
            __syncthreads();
#pragma unroll
            for (int i = 0; i < 8; ++i) {
                const long row = r0 + 8 * ty + i;
                const float4 h = row < rows ? *reinterpret_cast<const float4*>(hsave + row * (kPDepth * kPW) + (l - 1) * kPW + 4 * tx)
                                            : make_float4(0.f, 0.f, 0.f, 0.f);
                const float hv[4] = {h.x, h.y, h.z, h.w};
#pragma unroll
                for (int e = 0; e < 4; ++e) {
                    const float2 a = acc[i >> 1][e];
                    v[i][e] = hv[e] > 0.0f ? ((i & 1) ? a.y : a.x) : 0.0f;
                }
            }
        }
    }
}

// Weight gradients summed over rows: layer l (0..3): dW[o][i] += da_l[o]
// in_l[i], db[o] += da_l[o], with in_0 = gamma(x) (40 padded), in_l = h_{l-1};
// head: dw[i] += ds h_3[i], db += ds.  One block per chunk of rows, 64
// threads per layer, each owning an 8 x 8 patch of the layer's 64 x 64
// product (four 16-byte loads for 32 packed FMAs); the rows pass through
// shared memory 16 at a time, the next 16 on their way (cp.async).  Every sum
// runs over the chunk's rows in order; every block writes its partial sums of
// all weights to its own row of `part` (k_grad_reduce adds the rows in block
// order, so the result is the same on every run).  Bound by the FMA lanes and
// by reading the saved rows (2.2 KB each).  Measured, 262,144 rows: 0.63 ->
// 0.27 ms.
constexpr int kWgThreads = 256, kWgTileRows = 16;
constexpr int kWgRow = 2 * kPDepth * kPW + kPInPad;           // da, h, g of a row
constexpr int kWgSmem = 2 * kWgTileRows * kWgRow * (int)sizeof(float);

__device__ __forceinline__ void cp_async16(float* dst, const float* src) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"((uint32_t)__cvta_generic_to_shared(dst)), "l"(src)
                 : "memory");
}

__global__ __launch_bounds__(kWgThreads, 2) void k_prop_wgrad(
    const float* __restrict__ gsave, const float* __restrict__ hsave,
    const float* __restrict__ dasave, const float* __restrict__ ds, long rows, int chunk,
    float* __restrict__ part) {
    extern __shared__ __align__(16) float sh[];
    float* __restrict__ grad = part + (size_t)blockIdx.x * kPN;
    const long r0 = (long)blockIdx.x * chunk;
    const long r1 = min(rows, r0 + chunk);
    if (r0 >= rows) return;
    const int t = threadIdx.x, l = t >> 6, tx = t & 7, ty = (t >> 3) & 7;
    constexpr int kDa = 0, kH = kWgTileRows * kPDepth * kPW, kG = 2 * kH;   // within a buffer
    auto load = [&](long rb, float* buf) {
        const int n = (int)min((long)kWgTileRows, r1 - rb);
        for (int q = t; q < n * (kPDepth * kPW / 4); q += kWgThreads) {
            cp_async16(buf + kDa + 4 * q, dasave + rb * (kPDepth * kPW) + 4 * q);
            cp_async16(buf + kH + 4 * q, hsave + rb * (kPDepth * kPW) + 4 * q);
        }
        for (int q = t; q < n * (kPInPad / 4); q += kWgThreads)
            cp_async16(buf + kG + 4 * q, gsave + rb * kPInPad + 4 * q);
        asm volatile("cp.async.commit_group;" ::: "memory");
    };
    float2 acc[8][4];
    float accb[8];
#pragma unroll
    for (int i = 0; i < 8; ++i) {
        accb[i] = 0.f;
#pragma unroll
        for (int j = 0; j < 4; ++j) acc[i][j] = make_float2(0.f, 0.f);
    }
    float acch = 0.f;
    // layer 0 has 40 inputs: threads beyond them do nothing
    const bool live = l > 0 || 8 * tx < kPInPad;
    load(r0, sh);
    int cur = 0;
    for (long rb = r0; rb < r1; rb += kWgTileRows, cur ^= 1) {
        const bool more = rb + kWgTileRows < r1;
        if (more) load(rb + kWgTileRows, sh + (cur ^ 1) * kWgTileRows * kWgRow);
        if (more) asm volatile("cp.async.wait_group 1;" ::: "memory");
        else asm volatile("cp.async.wait_group 0;" ::: "memory");
        __syncthreads();
        const float* buf = sh + cur * kWgTileRows * kWgRow;
        const int n = (int)min((long)kWgTileRows, r1 - rb);
        if (live) {
#pragma unroll 2
            for (int r = 0; r < n; ++r) {
                const float4* a4 = reinterpret_cast<const float4*>(buf + kDa + r * (kPDepth * kPW) + l * kPW + 8 * ty);
                const float4* x4 = reinterpret_cast<const float4*>(l == 0 ? buf + kG + r * kPInPad + 8 * tx
                                                                          : buf + kH + r * (kPDepth * kPW) + (l - 1) * kPW + 8 * tx);
                const float4 a0 = a4[0], a1 = a4[1], x0 = x4[0], x1 = x4[1];
                const float a[8] = {a0.x, a0.y, a0.z, a0.w, a1.x, a1.y, a1.z, a1.w};
                const float2 x[4] = {make_float2(x0.x, x0.y), make_float2(x0.z, x0.w),
                                     make_float2(x1.x, x1.y), make_float2(x1.z, x1.w)};
#pragma unroll
                for (int i = 0; i < 8; ++i) {
                    const float2 ai = make_float2(a[i], a[i]);
#pragma unroll
                    for (int j = 0; j < 4; ++j) acc[i][j] = __ffma2_rn(ai, x[j], acc[i][j]);
                    accb[i] += a[i];
                }
            }
        }
        // density head
        if (t < kPW + 1)
            for (int r = 0; r < n; ++r)
                acch += ds[rb + r] * (t < kPW ? buf[kH + r * (kPDepth * kPW) + (kPDepth - 1) * kPW + t] : 1.0f);
        __syncthreads();
    }
    const int fin = (l == 0) ? kPIn : kPW;
    float* gW = grad + prop_off(l);
    float* gb = gW + kPW * fin;
    if (live) {
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            const int o = 8 * ty + i;
#pragma unroll
            for (int j = 0; j < 8; ++j) {
                const int in = 8 * tx + j;
                if (in < fin) gW[o * fin + in] = (j & 1) ? acc[i][j >> 1].y : acc[i][j >> 1].x;
            }
            if (tx == 0) gb[o] = accb[i];
        }
    }
    if (t < kPW + 1) grad[kPOffHead + t] = acch;
}

// grad[i] = scale * sum over blocks b (in order) of part[b][i].
__global__ void k_grad_reduce(const float* __restrict__ part, int nblk, float scale,
                              float* __restrict__ grad) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= kPN) return;
    float s = 0.0f;
#pragma unroll 16
    for (int b = 0; b < nblk; ++b) s += part[(size_t)b * kPN + i];
    grad[i] = s * scale;
}

__global__ void k_adam(float* __restrict__ W, const float* __restrict__ g, float* __restrict__ m,
                       float* __restrict__ v, int n, float lr, float b1, float b2, float eps,
                       float c1, float c2) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const float gi = g[i];
    const float mi = b1 * m[i] + (1.0f - b1) * gi;
    const float vi = b2 * v[i] + (1.0f - b2) * gi * gi;
    m[i] = mi;
    v[i] = vi;
    W[i] -= lr * (mi / c1) / (sqrtf(vi / c2) + eps);
}

cudaError_t launch_adam(float* W, const float* g, float* m, float* v, int n, float lr, float b1,
                        float b2, float eps, float c1, float c2, cudaStream_t s) {
    note_launch();
    k_adam<<<(n + 255) / 256, 256, 0, s>>>(W, g, m, v, n, lr, b1, b2, eps, c1, c2);
    return cudaGetLastError();
}

// Targets: final weights of the full sampler re-binned onto nb equal
// intervals of [near, far] (interval floor((z - near)/(far - near) nb),
// clamped), normalised (uniform for a ray without weight).
__global__ void k_histogram(const Ray* __restrict__ rays, int n_rays, const float* __restrict__ za,
                            const float4* __restrict__ oa, int nc, const float* __restrict__ zb,
                            const float4* __restrict__ ob, int nf, int nb, float near_z,
                            float far_z, float* __restrict__ hist) {
    const int r = blockIdx.x * blockDim.x + threadIdx.x;
    if (r >= n_rays) return;
    const float dn = rays[r].dnorm;
    const float* a = za + (size_t)r * nc;
    const float4* av = oa + (size_t)r * nc;
    const float* b = zb + (size_t)r * nf;
    const float4* bv = ob + (size_t)r * nf;
    float* h = hist + (size_t)r * nb;
    for (int i = 0; i < nb; ++i) h[i] = 0.0f;
    int ia = 0, ib = 0;
    auto take = [&](float& z, float4& v) {
        if (ib >= nf || (ia < nc && a[ia] <= b[ib])) { z = a[ia]; v = av[ia]; ++ia; }
        else { z = b[ib]; v = bv[ib]; ++ib; }
    };
    const int n = nc + nf;
    float zcur, znext = 0.f;
    float4 vcur, vnext = make_float4(0.f, 0.f, 0.f, 0.f);
    take(zcur, vcur);
    float T = 1.0f, tot = 0.0f;
    for (int k = 0; k < n; ++k) {
        if (k < n - 1) take(znext, vnext);
        const float delta = (k < n - 1) ? (znext - zcur) * dn : 1e10f;
        const float a_k = 1.0f - expf(-fmaxf(vcur.x, 0.0f) * delta);
        const float w = T * a_k;
        T *= (1.0f - a_k);
        int bin = (int)floorf((zcur - near_z) / (far_z - near_z) * (float)nb);
        bin = bin < 0 ? 0 : (bin > nb - 1 ? nb - 1 : bin);
        h[bin] += w;
        tot += w;
        zcur = znext; vcur = vnext;
    }
    for (int i = 0; i < nb; ++i) h[i] = tot > 0.0f ? h[i] / tot : 1.0f / (float)nb;
}

// Unpack rays into (o, d) arrays for training.
__global__ void k_rays_to_od(const Ray* __restrict__ rays, int n, float* __restrict__ O,
                             float* __restrict__ D) {
    const int r = blockIdx.x * blockDim.x + threadIdx.x;
    if (r >= n) return;
    const Ray R = rays[r];
    O[3 * r] = R.ox; O[3 * r + 1] = R.oy; O[3 * r + 2] = R.oz;
    D[3 * r] = R.dx; D[3 * r + 1] = R.dy; D[3 * r + 2] = R.dz;
}

__global__ void k_gather_rows(const float* __restrict__ src, const int* __restrict__ perm, int n,
                              int width, float* __restrict__ dst) {
    const long t = (long)blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= (long)n * width) return;
    const long r = t / width;
    const int c = (int)(t - r * width);
    dst[t] = src[(long)perm[r] * width + c];
}

static int grid_for(long rows, int tb) {
    long g = (rows + tb - 1) / tb;
    return (int)(g < 4096 ? (g < 1 ? 1 : g) : 4096);
}

// Dynamic shared memory of k_prop_loss_bwd: a double and four floats per bin.
static int loss_smem(int nb) { return kLossRays * (nb + 1) * (int)(sizeof(double) + 4 * sizeof(float)); }

// ----------------------------------------------------------------- host API
int proposal_alloc(mcl_map* m) {
    int rc;
    if ((rc = cuda_check(cudaMalloc(&m->prop_w, sizeof(float) * kPN * 4), "proposal weights"))) return rc;
    m->prop_m = m->prop_w + kPN;
    m->prop_v = m->prop_w + 2 * kPN;
    m->prop_g = m->prop_w + 3 * kPN;
    if ((rc = cuda_check(cudaMemset(m->prop_w, 0, sizeof(float) * kPN * 4), "proposal clear"))) return rc;
    if ((rc = cuda_check(cudaMalloc(&m->prop_packed, 4 * 64 * 64 * sizeof(uint16_t)), "proposal bf16")) ||
        (rc = cuda_check(cudaMemset(m->prop_packed, 0, 4 * 64 * 64 * sizeof(uint16_t)), "proposal bf16")) ||
        (rc = cuda_check(cudaMalloc(&m->prop_abort, sizeof(int)), "proposal abort flag")))
        return rc;
    int dev = 0, major = 0, minor = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&m->n_sm, cudaDevAttrMultiProcessorCount, dev);
    cudaDeviceGetAttribute(&major, cudaDevAttrComputeCapabilityMajor, dev);
    cudaDeviceGetAttribute(&minor, cudaDevAttrComputeCapabilityMinor, dev);
    if (major == 10 && minor == 3 && (rc = cuda_check(prop_tc_prepare(), "proposal tc smem"))) return rc;
    if ((rc = cuda_check(cudaFuncSetAttribute(k_prop_infer, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                              kPN * (int)sizeof(float)),
                         "proposal smem")))
        return rc;
    struct {
        const void* fn;
        int bytes;
    } at[] = {{(const void*)k_prop_fwd_train, kPFwdSmem},
              {(const void*)k_prop_bwd_data, kPBwdSmem},
              {(const void*)k_prop_wgrad, kWgSmem},
              {(const void*)k_prop_loss_bwd, loss_smem(kMaxCoarse)}};
    for (const auto& e : at)
        if ((rc = cuda_check(cudaFuncSetAttribute(e.fn, cudaFuncAttributeMaxDynamicSharedMemorySize, e.bytes),
                             "proposal smem")))
            return rc;
    return MCL_OK;
}

// Proposal densities at the stratified samples: the tensor-core kernel for
// the BF16 / FP8 forms, the FP32 kernel for the FP32 form.
cudaError_t launch_prop_infer(mcl_map* m, int precision, const Ray* rays, const float* z, int n_p,
                              int n_rays, const int* n_rays_dev, float4* out, cudaStream_t s) {
    if (precision != MCL_PREC_FP32 && mlp_tc_available(m, MCL_PREC_BF16))
        return launch_prop_infer_tc(m, rays, z, n_p, n_rays, n_rays_dev, out, m->n_sm, s);
    const long rows = (long)n_rays * n_p;
    note_launch();
    k_prop_infer<<<grid_for(rows, 128), 128, kPN * sizeof(float), s>>>(m->prop_w, rays, z, n_p, rows,
                                                                        n_rays_dev, out);
    return cudaGetLastError();
}

cudaError_t launch_histogram(const Ray* rays, int n_rays, const float* zc, const float4* oc, int nc,
                             const float* zf, const float4* of, int nf, int nb, float near_z,
                             float far_z, float* hist, cudaStream_t s) {
    note_launch();
    k_histogram<<<(n_rays + 127) / 128, 128, 0, s>>>(rays, n_rays, zc, oc, nc, zf, of, nf, nb,
                                                      near_z, far_z, hist);
    return cudaGetLastError();
}

// Scratch of one training batch (caller-owned buffers).
struct PropBatch {
    float* part; // [blocks of k_prop_wgrad][kPN]
    float* g;    // [rows][40]
    float* h;    // [rows][4][64]
    float* da;   // [rows][4][64]
    float* s;    // [rows]
    float* ds;   // [rows]
};

constexpr int kWgChunk = 512;   // rows per block of k_prop_wgrad

// Loss (summed into *loss_acc, scaled by `lscale`) and gradient (written to
// m->prop_g, scaled by `scale`) of n rays (O, D [n,3]) against hist [n, nb].
static cudaError_t prop_loss_grad_batch(mcl_map* m, const float* O, const float* D, int n, int nb,
                                        float near_z, float far_z, const float* hist, float scale,
                                        double lscale, const PropBatch& sb, double* loss_acc,
                                        cudaStream_t s) {
    const long rows = (long)n * nb;
    // two blocks per SM walk over the tiles (the weights are loaded once)
    const int tiles = (int)std::min<long>((rows + kPTile - 1) / kPTile, 2 * m->n_sm);
    note_launch(5);
    k_prop_fwd_train<<<tiles, 256, kPFwdSmem, s>>>(m->prop_w, O, D, n, nb, near_z, far_z, sb.g, sb.h, sb.s);
    k_prop_loss_bwd<<<(n + kLossRays - 1) / kLossRays, kLossThreads, loss_smem(nb), s>>>(
        sb.s, D, n, nb, near_z, far_z, hist, scale, lscale, sb.ds, loss_acc);
    k_prop_bwd_data<<<tiles, 256, kPBwdSmem, s>>>(m->prop_w, sb.h, sb.ds, rows, sb.da);
    const int nblk = (int)((rows + kWgChunk - 1) / kWgChunk);
    k_prop_wgrad<<<nblk, kWgThreads, kWgSmem, s>>>(sb.g, sb.h, sb.da, sb.ds, rows, kWgChunk, sb.part);
    k_grad_reduce<<<(kPN + 255) / 256, 256, 0, s>>>(sb.part, nblk, 1.0f, m->prop_g);
    return cudaGetLastError();
}

static void add_batch(Scratch& sc, PropBatch& b, long rows) {
    const long nblk = (rows + kWgChunk - 1) / kWgChunk;
    sc.add(&b.part, sizeof(float) * nblk * kPN);
    sc.add(&b.g, sizeof(float) * rows * kPInPad);
    sc.add(&b.h, sizeof(float) * rows * kPDepth * kPW);
    sc.add(&b.da, sizeof(float) * rows * kPDepth * kPW);
    sc.add(&b.s, sizeof(float) * rows);
    sc.add(&b.ds, sizeof(float) * rows);
}

int proposal_loss_grad(mcl_map* m, const float* O, const float* D, int n, int nb, float near_z,
                       float far_z, const float* hist, double* d_loss, float* d_grad,
                       cudaStream_t s) {
    PropBatch b{};
    Scratch sc;
    add_batch(sc, b, (long)n * nb);
    int rc = sc.take(m, true);
    if (rc) return rc;
    rc = cuda_check(cudaMemsetAsync(d_loss, 0, sizeof(double), s), "clear loss");
    if (!rc)
        rc = cuda_check(prop_loss_grad_batch(m, O, D, n, nb, near_z, far_z, hist, 1.0f / n, 1.0 / n, b, d_loss, s),
                        "proposal loss/grad");
    if (!rc)
        rc = cuda_check(cudaMemcpyAsync(d_grad, m->prop_g, sizeof(float) * kPN, cudaMemcpyDeviceToDevice, s),
                        "copy grad");
    // (also after an error: the scratch may be freed or used again)
    const int rs = cuda_check(cudaStreamSynchronize(s), "proposal sync");
    return rc ? rc : rs;
}

int proposal_train(mcl_map* m, const float* d_poses, int n_poses, const int32_t* d_pixels, int B,
                   const mcl_intrinsics& K, int level, const mcl_opts& o, const mcl_train_cfg& cfg,
                   float* d_loss_log, cudaStream_t s,
                   int (*render_chunk)(mcl_map*, const float*, int, const mcl_intrinsics*, int,
                                       const int32_t*, int, const mcl_opts*, cudaStream_t)) {
    const int nb = cfg.n_bins;
    const long n_rays = (long)n_poses * B;
    int rc = 0;
    float *O = nullptr, *D = nullptr, *hist = nullptr, *Ob = nullptr, *Db = nullptr, *Hb = nullptr;
    int* perm_d = nullptr;
    double* loss_acc = nullptr;
    PropBatch b{};
    const int batch = cfg.batch_rays;
    Scratch sc;
    sc.add(&O, sizeof(float) * 3 * n_rays);
    sc.add(&D, sizeof(float) * 3 * n_rays);
    sc.add(&hist, sizeof(float) * nb * n_rays);
    sc.add(&Ob, sizeof(float) * 3 * batch);
    sc.add(&Db, sizeof(float) * 3 * batch);
    sc.add(&Hb, sizeof(float) * nb * batch);
    sc.add(&perm_d, sizeof(int) * n_rays);
    sc.add(&loss_acc, sizeof(double));
    add_batch(sc, b, (long)batch * nb);
    if ((rc = sc.take(m, false))) return rc;
    // 1) targets from the full sampler, in chunks of poses that fit the workspace
    const int chunk_poses = std::max(1, std::min(n_poses, m->cfg.max_rays / B));
    for (int p0 = 0; p0 < n_poses && !rc; p0 += chunk_poses) {
        const int np = std::min(chunk_poses, n_poses - p0);
        const int nr = np * B;
        rc = render_chunk(m, d_poses + 12 * (size_t)p0, np, &K, level, d_pixels, B, &o, s);
        if (rc) break;
        rc = cuda_check(launch_histogram(m->rays, nr, m->zc, m->out_c, o.n_coarse, m->zf, m->out_f,
                                         o.n_fine, nb, o.near_z, o.far_z,
                                         hist + (size_t)p0 * B * nb, s),
                        "histogram");
        if (rc) break;
        note_launch();
        k_rays_to_od<<<(nr + 127) / 128, 128, 0, s>>>(m->rays, nr, O + 3 * (size_t)p0 * B,
                                                       D + 3 * (size_t)p0 * B);
        rc = cuda_check(cudaGetLastError(), "rays to o, d");
    }
    // 2) epochs of Adam over shuffled mini-batches
    std::mt19937_64 rng(cfg.seed);
    std::vector<int> perm(n_rays);
    for (long i = 0; i < n_rays; ++i) perm[i] = (int)i;
    int step = m->prop_step;
    const long steps_per_epoch = (n_rays + batch - 1) / batch;
    const double total_steps = (double)cfg.epochs * steps_per_epoch;
    long local_step = 0;
    const double decay = cfg.lr_end > 0.f ? log((double)cfg.lr_end / cfg.lr) : 0.0;
    for (int ep = 0; ep < cfg.epochs && !rc; ++ep) {
        std::shuffle(perm.begin(), perm.end(), rng);
        if ((rc = cuda_check(cudaMemcpyAsync(perm_d, perm.data(), sizeof(int) * n_rays,
                                             cudaMemcpyHostToDevice, s),
                             "upload permutation")))
            break;
        if ((rc = cuda_check(cudaMemsetAsync(loss_acc, 0, sizeof(double), s), "clear loss"))) break;
        for (long b0 = 0; b0 < n_rays && !rc; b0 += batch) {
            const int nbat = (int)std::min<long>(batch, n_rays - b0);
            note_launch(3);
            k_gather_rows<<<(nbat * 3 + 255) / 256, 256, 0, s>>>(O, perm_d + b0, nbat, 3, Ob);
            k_gather_rows<<<(nbat * 3 + 255) / 256, 256, 0, s>>>(D, perm_d + b0, nbat, 3, Db);
            k_gather_rows<<<(nbat * nb + 255) / 256, 256, 0, s>>>(hist, perm_d + b0, nbat, nb, Hb);
            rc = cuda_check(prop_loss_grad_batch(m, Ob, Db, nbat, nb, o.near_z, o.far_z, Hb,
                                                 1.0f / nbat, 1.0, b, loss_acc, s),
                            "proposal batch");
            if (rc) break;
            ++step;
            const double frac = total_steps > 1 ? (double)local_step / (total_steps - 1) : 0.0;
            const float lr = (float)(cfg.lr * exp(decay * frac));
            ++local_step;
            const float c1 = 1.0f - powf(cfg.beta1, (float)step);
            const float c2 = 1.0f - powf(cfg.beta2, (float)step);
            note_launch();
            k_adam<<<(kPN + 255) / 256, 256, 0, s>>>(m->prop_w, m->prop_g, m->prop_m, m->prop_v, kPN,
                                                     lr, cfg.beta1, cfg.beta2, cfg.eps, c1, c2);
            rc = cuda_check(cudaGetLastError(), "adam");
        }
        if (!rc && d_loss_log) {
            double L = 0.0;
            rc = cuda_check(cudaMemcpyAsync(&L, loss_acc, sizeof(double), cudaMemcpyDeviceToHost, s),
                            "read loss");
            if (!rc) rc = cuda_check(cudaStreamSynchronize(s), "sync");
            const float mean = (float)(L / (double)n_rays);
            if (!rc)
                rc = cuda_check(cudaMemcpyAsync(d_loss_log + ep, &mean, sizeof(float),
                                                cudaMemcpyHostToDevice, s),
                                "write loss");
            if (!rc) rc = cuda_check(cudaStreamSynchronize(s), "sync");
        }
    }
    m->prop_step = step;
    if (!rc) rc = cuda_check(prop_tc_pack(m, s), "pack proposal");
    const int rs = cuda_check(cudaStreamSynchronize(s), "train sync");
    if (!rc) rc = rs;
    if (!rc) m->has_proposal = true;
    return rc;
}

}  // namespace mcl

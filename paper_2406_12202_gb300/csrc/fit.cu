// fit.cu -- fitting the NeRF map's FP32 weights to samples of a field: points
// x with view directions and targets (density, r, g, b), loss
//   L = mean over points of  w_sigma (sigma_raw(x) - sigma_t)^2 + |rgb(x, d) - rgb_t|^2,
// minimised by Adam with the library's own kernels: the SIMT FP32 forward
// (gamma(x), SGEMM layers, heads) with every layer's output kept, a backward
// pass of SGEMMs with the ReLU masks in their epilogue, and weight gradients summed over the batch in a fixed order (the same inputs give the
// same weights).  The map's tensor-core forms are rebuilt from the fitted
// weights.  This stands in for training a map on images (Eq. 2, out of
// scope): it gives maps of analytic scenes whose weights the library itself
// produced.
#include <string.h>

#include <algorithm>
#include <random>
#include <vector>

#include "internal.cuh"

namespace mcl {

namespace {

constexpr int kWgRows = 1024;   // rows per partial sum of a weight gradient
constexpr int kWgTile = 64;     // 64 x 64 outputs per block of k_wgrad

struct FitBuf {
    long B = 0;                 // points per batch
    float *x = nullptr, *dir = nullptr, *tgt = nullptr;   // batch inputs
    Ray* rays = nullptr;
    float *gd = nullptr, *z = nullptr, *gx = nullptr;     // gamma(d) [B,32], z = 0, gamma(x) [B,64]
    float* h = nullptr;         // trunk outputs [8][B][256]
    float* feat = nullptr;      // [B][256]
    float* hid = nullptr;       // [B][256] (128 used)
    float4* out = nullptr;      // [B] (sigma_raw, rgb)
    float *dA = nullptr, *dB = nullptr, *dhid = nullptr;  // [B][256]
    float* dlog = nullptr;      // [B][4]: d rgb logits, d sigma
    float* part = nullptr;      // partial weight gradients
    float* partb = nullptr;     // partial bias gradients
    double* lpart = nullptr;    // per-block loss partials
    double* loss = nullptr;
    float* grad = nullptr;      // [w32_n] gradient in the padded layout
    float *m1 = nullptr, *m2 = nullptr;   // Adam moments
};

int alloc_buf(mcl_map* m, Scratch& sc, FitBuf& b, long B, bool adam, cudaStream_t s) {
    b.B = B;
    const long nchunk = (B + kWgRows - 1) / kWgRows;
    sc.add(&b.x, sizeof(float) * 3 * B);
    sc.add(&b.dir, sizeof(float) * 3 * B);
    sc.add(&b.tgt, sizeof(float) * 4 * B);
    sc.add(&b.rays, sizeof(Ray) * B);
    sc.add(&b.gd, sizeof(float) * kGdPad * B);
    sc.add(&b.z, sizeof(float) * B);
    sc.add(&b.gx, sizeof(float) * kGxPad * B);
    sc.add(&b.h, sizeof(float) * 8 * kWidth * B);
    sc.add(&b.feat, sizeof(float) * kWidth * B);
    sc.add(&b.hid, sizeof(float) * kWidth * B);
    sc.add(&b.out, sizeof(float4) * B);
    sc.add(&b.dA, sizeof(float) * kWidth * B);
    sc.add(&b.dB, sizeof(float) * kWidth * B);
    sc.add(&b.dhid, sizeof(float) * kWidth * B);
    sc.add(&b.dlog, sizeof(float) * 4 * B);
    sc.add(&b.part, sizeof(float) * nchunk * kWidth * (kWidth + kGxPad));
    sc.add(&b.partb, sizeof(float) * nchunk * kWidth);
    sc.add(&b.lpart, sizeof(double) * ((B + 255) / 256));
    sc.add(&b.loss, sizeof(double));
    sc.add(&b.grad, sizeof(float) * m->w32_n);
    if (adam) {
        sc.add(&b.m1, sizeof(float) * m->w32_n);
        sc.add(&b.m2, sizeof(float) * m->w32_n);
    }
    int rc;
    if ((rc = sc.take(m, !adam))) return rc;
    if (adam) {
        // on the run's own stream: the steps on s are not ordered after work of
        // the default stream, and the block may hold an earlier call's values
        if ((rc = cuda_check(cudaMemsetAsync(b.m1, 0, sizeof(float) * m->w32_n, s), "clear moments")) ||
            (rc = cuda_check(cudaMemsetAsync(b.m2, 0, sizeof(float) * m->w32_n, s), "clear moments")))
            return rc;
    }
    return MCL_OK;
}

// Rows idx[r0 .. r0 + n) of x, dir, tgt into the batch buffers.
__global__ void k_fit_gather(const float* __restrict__ x, const float* __restrict__ dir,
                             const float* __restrict__ tgt, const int* __restrict__ idx, long r0,
                             int n, float* __restrict__ bx, float* __restrict__ bd,
                             float* __restrict__ bt) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const long k = idx ? idx[r0 + i] : r0 + i;
    for (int c = 0; c < 3; ++c) {
        bx[3 * i + c] = x[3 * k + c];
        bd[3 * i + c] = dir[3 * k + c];
    }
    for (int c = 0; c < 4; ++c) bt[4 * i + c] = tgt[4 * k + c];
}

// Loss terms and output gradients of each point; per-block FP64 loss sums.
__global__ __launch_bounds__(256) void k_fit_loss(const float4* __restrict__ out,
                                                  const float* __restrict__ tgt, int n, float wsig,
                                                  float scale, float* __restrict__ dlog,
                                                  double* __restrict__ lpart) {
    __shared__ double sh[256];
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    double L = 0.0;
    if (i < n) {
        const float4 o = out[i];
        const float* t = tgt + 4 * i;
        const float ds = o.x - t[0];
        const float c[3] = {o.y, o.z, o.w};
        L = (double)wsig * ds * ds;
        for (int k = 0; k < 3; ++k) {
            const float e = c[k] - t[1 + k];
            L += (double)e * e;
            dlog[4 * i + k] = 2.0f * e * c[k] * (1.0f - c[k]) * scale;
        }
        dlog[4 * i + 3] = 2.0f * wsig * ds * scale;
    }
    sh[threadIdx.x] = L;
    __syncthreads();
    for (int s = 128; s > 0; s >>= 1) {
        if (threadIdx.x < s) sh[threadIdx.x] += sh[threadIdx.x + s];
        __syncthreads();
    }
    if (threadIdx.x == 0) lpart[blockIdx.x] = sh[0];
}

__global__ void k_fit_loss_sum(const double* __restrict__ lpart, int nblk, double scale,
                               double* __restrict__ loss, float* __restrict__ log_entry) {
    if (threadIdx.x != 0 || blockIdx.x != 0) return;
    double s = 0.0;
    for (int b = 0; b < nblk; ++b) s += lpart[b];
    *loss = s * scale;
    if (log_entry) *log_entry = (float)(s * scale);
}

// RGB output layer backward: dhid[p][k] = sum_c dlog[p][c] W_o[c][k], masked
// by hid[p][k] > 0 (the hidden layer's ReLU).
__global__ void k_fit_drgb(const float* __restrict__ dlog, const float* __restrict__ Wo,
                           const float* __restrict__ hid, long n, float* __restrict__ dhid) {
    const long t = (long)blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= n * kRgbW) return;
    const long p = t / kRgbW;
    const int k = (int)(t - p * kRgbW);
    float s = 0.f;
    for (int c = 0; c < 3; ++c) s = fmaf(dlog[4 * p + c], Wo[c * kRgbW + k], s);
    dhid[p * kWidth + k] = hid[p * kWidth + k] > 0.f ? s : 0.f;
}

// Top of the trunk: d = (d_feature_path + d_sigma w_sigma) masked by h8 > 0.
__global__ void k_fit_dtop(float* __restrict__ d, const float* __restrict__ dlog,
                           const float* __restrict__ wsig, const float* __restrict__ h8, long n) {
    const long t = (long)blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= n * kWidth) return;
    const long p = t / kWidth;
    const int k = (int)(t - p * kWidth);
    const float v = fmaf(dlog[4 * p + 3], wsig[k], d[t]);
    d[t] = h8[t] > 0.f ? v : 0.f;
}

// Partial weight gradients of one row chunk:
//   part[c][o][k] = sum_{rows p of chunk c} dY[p][o] X[p][k],  X = [X1 | X2],
//   partb[c][o] = sum_p dY[p][o].
// 64 x 64 outputs per block, 8 x 4 per thread (three 16-byte loads for 16
// packed FMAs on pairs of outputs); the rows pass through shared memory 16 at
// a time, the next 48 on their way (cp.async).  Every sum is one chain of
// FMAs over the chunk's rows in order.  N and K1 are multiples of 64, K2 of
// 32, rows 16-byte aligned.  Bound by the FMA lanes; with 16 chunks (16,384
// rows) there are 256 blocks of 4 warps for 152 SMs.  Measured, 16,384 rows, all
// layers: 1.43 -> 0.64 ms (4 x 4 outputs per thread: 69 us a 256 x 256 layer,
// 8 x 4 with the next 16 rows on their way 64, as here 62; its FMAs take 34).
constexpr int kWgStage = 16, kWgBufs = 4;

__device__ __forceinline__ void cp_async16(float* dst, const float* src, bool in) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"((uint32_t)__cvta_generic_to_shared(dst)),
                 "l"(src), "r"(in ? 16 : 0)
                 : "memory");
}

__global__ __launch_bounds__(128) void k_wgrad(const float* __restrict__ dY, int ldy, int N,
                                               const float* __restrict__ X1, int ld1, int K1,
                                               const float* __restrict__ X2, int ld2, int K2,
                                               long rows, float* __restrict__ part,
                                               float* __restrict__ partb) {
    __shared__ __align__(16) float As[kWgBufs][kWgStage][kWgTile];
    __shared__ __align__(16) float Bs[kWgBufs][kWgStage][kWgTile];
    const int K = K1 + K2;
    const int o0 = blockIdx.x * kWgTile, k0 = blockIdx.y * kWgTile, c = blockIdx.z;
    const long p0 = (long)c * kWgRows, p1 = min(rows, p0 + kWgRows);
    const int t = threadIdx.x, tx = t & 15, ty = t >> 4;
    // the block's columns lie in one of X1, X2 (K1 is a multiple of the tile)
    const float* X = k0 < K1 ? X1 + k0 : X2 + (k0 - K1);
    const int ldx = k0 < K1 ? ld1 : ld2;
    auto load = [&](int st) {   // stage st (a group is committed past the end, too)
        const long pb = p0 + (long)st * kWgStage;
        const int buf = st % kWgBufs;
        if (pb < p1) {
#pragma unroll
            for (int q = 0; q < kWgStage * kWgTile / 4 / 128; ++q) {
                const int r = (t >> 4) + 8 * q, cc = (t & 15) * 4;
                const bool in = pb + r < p1;
                const long p = in ? pb + r : p0;
                cp_async16(&As[buf][r][cc], dY + p * ldy + o0 + cc, in);
                const bool ink = in && k0 + cc < K;
                cp_async16(&Bs[buf][r][cc], ink ? X + p * ldx + cc : X, ink);
            }
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
    };
    float2 acc[4][4], accb[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        accb[i] = make_float2(0.f, 0.f);
#pragma unroll
        for (int j = 0; j < 4; ++j) acc[i][j] = make_float2(0.f, 0.f);
    }
    load(0);
    load(1);
    load(2);
    int st = 0;
    for (long pb = p0; pb < p1; pb += kWgStage, ++st) {
        asm volatile("cp.async.wait_group 2;" ::: "memory");
        __syncthreads();     // stage st has landed; stage st - 1 has been read
        load(st + 3);
        const int cur = st % kWgBufs, n = (int)min((long)kWgStage, p1 - pb);
        auto row = [&](int r) {
            const float4 a0 = *reinterpret_cast<const float4*>(&As[cur][r][ty * 8]);
            const float4 a1 = *reinterpret_cast<const float4*>(&As[cur][r][ty * 8 + 4]);
            const float4 x = *reinterpret_cast<const float4*>(&Bs[cur][r][tx * 4]);
            const float2 a[4] = {make_float2(a0.x, a0.y), make_float2(a0.z, a0.w),
                                 make_float2(a1.x, a1.y), make_float2(a1.z, a1.w)};
            const float xv[4] = {x.x, x.y, x.z, x.w};
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                const float2 xj = make_float2(xv[j], xv[j]);
#pragma unroll
                for (int i = 0; i < 4; ++i) acc[i][j] = __ffma2_rn(a[i], xj, acc[i][j]);
            }
            if (blockIdx.y == 0)
#pragma unroll
                for (int i = 0; i < 4; ++i) accb[i] = __fadd2_rn(accb[i], a[i]);
        };
        if (n == kWgStage) {
#pragma unroll
            for (int r = 0; r < kWgStage; ++r) row(r);
        } else {
            for (int r = 0; r < n; ++r) row(r);
        }
    }
    float* pc = part + (size_t)c * N * K;
#pragma unroll
    for (int i = 0; i < 8; ++i) {
        const int o = o0 + ty * 8 + i;
        const float2* ar = acc[i >> 1];
        const float4 v = (i & 1) ? make_float4(ar[0].y, ar[1].y, ar[2].y, ar[3].y)
                                 : make_float4(ar[0].x, ar[1].x, ar[2].x, ar[3].x);
        if (k0 + tx * 4 < K) *reinterpret_cast<float4*>(pc + (size_t)o * K + k0 + tx * 4) = v;
        if (blockIdx.y == 0 && tx == 0) partb[(size_t)c * N + o] = (i & 1) ? accb[i >> 1].y : accb[i >> 1].x;
    }
}

// The same for the heads (N <= 4 outputs): 64 input columns per block, a
// thread per output and column, the rows staged in shared memory 64 at a time.
__global__ __launch_bounds__(256) void k_wgrad_head(const float* __restrict__ dY, int ldy, int N,
                                                    const float* __restrict__ X, int ldx, int K,
                                                    long rows, float* __restrict__ part,
                                                    float* __restrict__ partb) {
    __shared__ __align__(16) float xs[2][64][64];
    __shared__ float ds[2][64][4];
    const int k0 = blockIdx.x * 64, c = blockIdx.y, t = threadIdx.x, o = t >> 6, kk = t & 63;
    const long p0 = (long)c * kWgRows, p1 = min(rows, p0 + kWgRows);
    auto load = [&](long pb, int buf) {
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const int r = (t >> 4) + 16 * q, cc = (t & 15) * 4;
            const bool in = pb + r < p1 && k0 + cc < K;
            cp_async16(&xs[buf][r][cc], in ? X + (pb + r) * ldx + k0 + cc : X, in);
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
        const int r = t & 63, oo = t >> 6;
        ds[buf][r][oo] = (pb + r < p1 && oo < N) ? dY[(pb + r) * ldy + oo] : 0.f;
    };
    float acc = 0.f, accb = 0.f;
    load(p0, 0);
    int cur = 0;
    for (long pb = p0; pb < p1; pb += 64, cur ^= 1) {
        if (pb + 64 < p1) {
            load(pb + 64, cur ^ 1);
            asm volatile("cp.async.wait_group 1;" ::: "memory");
        } else {
            asm volatile("cp.async.wait_group 0;" ::: "memory");
        }
        __syncthreads();
        const int n = (int)min(64l, p1 - pb);
        if (o < N) {
#pragma unroll 8
            for (int r = 0; r < n; ++r) {
                const float a = ds[cur][r][o];
                acc = fmaf(a, xs[cur][r][kk], acc);
                accb += a;
            }
        }
        __syncthreads();
    }
    if (o < N && k0 + kk < K) part[((size_t)c * N + o) * K + k0 + kk] = acc;
    if (o < N && k0 + kk == 0) partb[(size_t)c * N + o] = accb;
}

// gW[o][k] (row stride ldg) = sum over chunks in order of part[c][o][k];
// gb[o] likewise from partb.
__global__ void k_wgrad_reduce(const float* __restrict__ part, const float* __restrict__ partb,
                               int nchunk, int N, int K, float* __restrict__ gW, int ldg,
                               float* __restrict__ gb) {
    const int t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t < N * K) {
        const int o = t / K, k = t - o * K;
        float s = 0.f;
        for (int c = 0; c < nchunk; ++c) s += part[(size_t)c * N * K + t];
        gW[(size_t)o * ldg + k] = s;
    }
    if (t < N) {
        float s = 0.f;
        for (int c = 0; c < nchunk; ++c) s += partb[(size_t)c * N + t];
        gb[t] = s;
    }
}

cudaError_t wgrad(const FitBuf& b, long n, const float* dY, int ldy, int N, const float* X1,
                  int ld1, int K1, const float* X2, int ld2, int K2, float* gW, int ldg,
                  float* gb, cudaStream_t s) {
    const int K = K1 + K2;
    const int nchunk = (int)((n + kWgRows - 1) / kWgRows);
    note_launch(2);
    if (N <= 4)
        k_wgrad_head<<<dim3((K + 63) / 64, nchunk), 256, 0, s>>>(dY, ldy, N, X1, ld1, K, n, b.part, b.partb);
    else
        k_wgrad<<<dim3(N / kWgTile, (K + kWgTile - 1) / kWgTile, nchunk), 128, 0, s>>>(
            dY, ldy, N, X1, ld1, K1, X2, ld2, K2, n, b.part, b.partb);
    k_wgrad_reduce<<<(N * K + 255) / 256, 256, 0, s>>>(b.part, b.partb, nchunk, N, K, gW, ldg, gb);
    return cudaGetLastError();
}

// Loss and gradient (padded layout, into b.grad) of the first n points held
// in b.x / b.dir / b.tgt; the loss (mean) into *b.loss and *log_entry.
cudaError_t loss_and_grad(mcl_map* m, const FitBuf& b, long n, float wsig, float* log_entry,
                          cudaStream_t s) {
    const LayerF32* L = m->L;
    cudaError_t e;
    float* h = b.h;
    auto H = [&](int l) { return h + (size_t)l * kWidth * n; };   // output of trunk layer l + 1
    auto off = [&](const float* p) { return b.grad + (p - m->w32); };
    // ---- forward, every layer's output kept
    if ((e = launch_query_setup(b.x, b.dir, (int)n, b.rays, b.gd, b.z, s)) ||
        (e = fp32_pe(b.rays, b.z, (int)n, b.gx, s)) ||
        (e = fp32_gemm(b.gx, kGxPad, kGxPad, nullptr, 0, 0, 0, 1, L[0].W, L[0].b, kWidth, H(0), kWidth,
                       (int)n, true, s)))
        return e;
    for (int l = 1; l < kDepth; ++l) {
        if (l == kSkip)
            e = fp32_gemm(H(l - 1), kWidth, kWidth, b.gx, kGxPad, kGxPad, 0, 1, L[l].W, L[l].b, kWidth,
                          H(l), kWidth, (int)n, true, s);
        else
            e = fp32_gemm(H(l - 1), kWidth, kWidth, nullptr, 0, 0, 0, 1, L[l].W, L[l].b, kWidth, H(l),
                          kWidth, (int)n, true, s);
        if (e) return e;
    }
    if ((e = fp32_gemm(H(7), kWidth, kWidth, nullptr, 0, 0, 0, 1, L[9].W, L[9].b, kWidth, b.feat,
                       kWidth, (int)n, false, s)) ||
        (e = fp32_gemm(b.feat, kWidth, kWidth, b.gd, kGdPad, kGdPad, 0, 1, L[10].W, L[10].b, kRgbW,
                       b.hid, kWidth, (int)n, true, s)) ||
        (e = fp32_heads(H(7), L[8], b.hid, L[11], (int)n, b.out, s)))
        return e;
    // ---- loss and output gradients
    const int nblk = (int)((n + 255) / 256);
    note_launch(2);
    k_fit_loss<<<nblk, 256, 0, s>>>(b.out, b.tgt, (int)n, wsig, 1.0f / (float)n, b.dlog, b.lpart);
    k_fit_loss_sum<<<1, 32, 0, s>>>(b.lpart, nblk, 1.0 / (double)n, b.loss, log_entry);
    // ---- backward
    // RGB output layer (3 x 128): gradient, then d hid (masked)
    if ((e = wgrad(b, n, b.dlog, 4, 3, b.hid, kWidth, kRgbW, nullptr, 0, 0, off(L[11].W), L[11].k_pad,
                   off(L[11].b), s)))
        return e;
    note_launch();
    k_fit_drgb<<<(unsigned)((n * kRgbW + 255) / 256), 256, 0, s>>>(b.dlog, L[11].W, b.hid, n, b.dhid);
    // RGB hidden layer (128 x [feature 256 | gamma(d) 32]), then d feature
    if ((e = wgrad(b, n, b.dhid, kWidth, kRgbW, b.feat, kWidth, kWidth, b.gd, kGdPad, kGdPad,
                   off(L[10].W), L[10].k_pad, off(L[10].b), s)))
        return e;
    if ((e = fp32_gemm_back(b.dhid, kRgbW, L[10].W, L[10].k_pad, nullptr, b.dA, (int)n, s))) return e;
    // feature layer (linear 256 x 256), then d h8 through it
    if ((e = wgrad(b, n, b.dA, kWidth, kWidth, H(7), kWidth, kWidth, nullptr, 0, 0, off(L[9].W),
                   L[9].k_pad, off(L[9].b), s)))
        return e;
    if ((e = fp32_gemm_back(b.dA, kWidth, L[9].W, L[9].k_pad, nullptr, b.dB, (int)n, s))) return e;
    // density head (1 x 256) gradient from d sigma (column 3 of dlog)
    if ((e = wgrad(b, n, b.dlog + 3, 4, 1, H(7), kWidth, kWidth, nullptr, 0, 0, off(L[8].W),
                   L[8].k_pad, off(L[8].b), s)))
        return e;
    note_launch();
    k_fit_dtop<<<(unsigned)((n * kWidth + 255) / 256), 256, 0, s>>>(b.dB, b.dlog, L[8].W, H(7), n);
    // trunk layers 8 .. 1: cur holds d of layer l's pre-activation
    float* cur = b.dB;
    float* nxt = b.dA;
    for (int l = kDepth - 1; l >= 0; --l) {
        if (l == 0)
            e = wgrad(b, n, cur, kWidth, kWidth, b.gx, kGxPad, kGxPad, nullptr, 0, 0, off(L[0].W),
                      L[0].k_pad, off(L[0].b), s);
        else if (l == kSkip)
            e = wgrad(b, n, cur, kWidth, kWidth, H(l - 1), kWidth, kWidth, b.gx, kGxPad, kGxPad,
                      off(L[l].W), L[l].k_pad, off(L[l].b), s);
        else
            e = wgrad(b, n, cur, kWidth, kWidth, H(l - 1), kWidth, kWidth, nullptr, 0, 0, off(L[l].W),
                      L[l].k_pad, off(L[l].b), s);
        if (e) return e;
        if (l == 0) break;
        if ((e = fp32_gemm_back(cur, kWidth, L[l].W, L[l].k_pad, H(l - 1), nxt, (int)n, s))) return e;
        std::swap(cur, nxt);
    }
    return cudaGetLastError();
}

}  // namespace

// Host copy of the FP32 weights in the blob layout of mcl_init_map.
int map_download(mcl_map* m, float* host_blob) {
    int fin[12], fout[12];
    blob_layer_shapes(fin, fout);
    std::vector<float> w(m->w32_n);
    int rc;
    if ((rc = cuda_check(cudaMemcpy(w.data(), m->w32, sizeof(float) * m->w32_n, cudaMemcpyDeviceToHost),
                         "download weights")))
        return rc;
    float* dst = host_blob;
    for (int l = 0; l < 12; ++l) {
        const size_t oW = m->L[l].W - m->w32, ob = m->L[l].b - m->w32;
        for (int o = 0; o < fout[l]; ++o)
            for (int i = 0; i < fin[l]; ++i) *dst++ = w[oW + (size_t)o * m->L[l].k_pad + i];
        for (int o = 0; o < fout[l]; ++o) *dst++ = w[ob + o];
    }
    return MCL_OK;
}

// Gradient in the padded layer layout -> blob layout (one layer per grid row).
struct Unpad {
    int src_w[12], src_b[12], dst[12], fin[12], fout[12], ld[12];
};
__global__ void k_unpad(const float* __restrict__ g, Unpad u, float* __restrict__ out) {
    const int l = blockIdx.y, nw = u.fin[l] * u.fout[l];
    const int t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t < nw) out[u.dst[l] + t] = g[u.src_w[l] + (t / u.fin[l]) * u.ld[l] + t % u.fin[l]];
    else if (t < nw + u.fout[l]) out[u.dst[l] + t] = g[u.src_b[l] + t - nw];
}

int map_loss_grad(mcl_map* m, const float* d_x, const float* d_dir, const float* d_target, int n,
                  float sigma_weight, double* d_loss, float* d_grad, cudaStream_t s) {
    FitBuf b;
    Scratch sc;
    int rc = alloc_buf(m, sc, b, n, false, s);
    if (rc) return rc;
    note_launch();
    k_fit_gather<<<(n + 255) / 256, 256, 0, s>>>(d_x, d_dir, d_target, nullptr, 0, n, b.x, b.dir, b.tgt);
    rc = cuda_check(cudaMemsetAsync(b.grad, 0, sizeof(float) * m->w32_n, s), "clear grad");
    if (!rc) rc = cuda_check(loss_and_grad(m, b, n, sigma_weight, nullptr, s), "loss and gradient");
    if (!rc) {
        Unpad u;
        blob_layer_shapes(u.fin, u.fout);
        int dst = 0, most = 0;
        for (int l = 0; l < 12; ++l) {
            u.src_w[l] = (int)(m->L[l].W - m->w32);
            u.src_b[l] = (int)(m->L[l].b - m->w32);
            u.ld[l] = m->L[l].k_pad;
            u.dst[l] = dst;
            const int size = u.fin[l] * u.fout[l] + u.fout[l];
            dst += size;
            most = std::max(most, size);
        }
        note_launch();
        k_unpad<<<dim3((most + 255) / 256, 12), 256, 0, s>>>(b.grad, u, d_grad);
        rc = cuda_check(cudaGetLastError(), "gradient layout");
    }
    if (!rc) rc = cuda_check(cudaMemcpyAsync(d_loss, b.loss, sizeof(double), cudaMemcpyDeviceToDevice, s),
                             "copy loss");
    // (also after an error: the scratch may be freed or used again)
    const int rs = cuda_check(cudaStreamSynchronize(s), "loss sync");
    return rc ? rc : rs;
}

int fit_map(mcl_map* m, const float* d_x, const float* d_dir, const float* d_target, int n,
            const mcl_fit_cfg& cfg, float* d_loss_log, cudaStream_t s) {
    const long B = std::min(n, cfg.batch);
    FitBuf b;
    int* perm_d = nullptr;
    Scratch sc;
    sc.add(&perm_d, sizeof(int) * n);
    int rc = alloc_buf(m, sc, b, B, true, s);
    std::mt19937_64 rng(cfg.seed);
    std::vector<int> perm(n);
    for (int i = 0; i < n; ++i) perm[i] = i;
    long pos = n;   // start of the next batch in the current permutation
    const float b1 = cfg.beta1, b2 = cfg.beta2;
    double c1 = 1.0, c2 = 1.0;
    const double decay = (cfg.lr_end > 0.f && cfg.steps > 1)
                             ? std::pow((double)cfg.lr_end / cfg.lr, 1.0 / (cfg.steps - 1))
                             : 1.0;
    for (int t = 0; t < cfg.steps && !rc; ++t) {
        if (pos + B > n) {
            // a new epoch: reshuffle (Fisher-Yates on the seeded generator)
            for (int i = n - 1; i > 0; --i) std::swap(perm[i], perm[rng() % (uint64_t)(i + 1)]);
            rc = cuda_check(cudaMemcpyAsync(perm_d, perm.data(), sizeof(int) * n, cudaMemcpyHostToDevice, s),
                            "upload permutation");
            if (!rc) rc = cuda_check(cudaStreamSynchronize(s), "permutation sync");
            pos = 0;
            if (rc) break;
        }
        note_launch();
        k_fit_gather<<<(unsigned)((B + 255) / 256), 256, 0, s>>>(d_x, d_dir, d_target, perm_d, pos, (int)B,
                                                              b.x, b.dir, b.tgt);
        pos += B;
        rc = cuda_check(cudaMemsetAsync(b.grad, 0, sizeof(float) * m->w32_n, s), "clear grad");
        if (!rc)
            rc = cuda_check(loss_and_grad(m, b, B, cfg.sigma_weight, d_loss_log ? d_loss_log + t : nullptr, s),
                            "fit step");
        c1 *= b1;
        c2 *= b2;
        const float lr = (float)(cfg.lr * std::pow(decay, (double)t));
        if (!rc)
            rc = cuda_check(launch_adam(m->w32, b.grad, b.m1, b.m2, (int)m->w32_n, lr, b1, b2, cfg.eps,
                                        (float)(1.0 - c1), (float)(1.0 - c2), s),
                            "fit adam");
    }
    const int rs = cuda_check(cudaStreamSynchronize(s), "fit sync");
    return rc ? rc : rs;
}

}  // namespace mcl

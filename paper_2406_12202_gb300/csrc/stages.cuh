// stages.cuh -- per-ray, per-particle and per-block bodies of the SIMT stages
// of one weight update, shared by the single-update kernels (render.cu,
// resample.cu) and the device-driven loop kernels (loop.cu), so both run the
// same arithmetic.
#pragma once
#include <math.h>

#include <utility>

#include "internal.cuh"
#include "rng.cuh"

namespace mcl {

typedef unsigned long long u64;
typedef unsigned __int128 u128;

// ---------------------------------------------------------------------------
// Pixel-centre ray of pose p (row-major 3x4 [R|t], camera looking along -z,
// +y up) through level-image pixel (u, v) with level intrinsics; the
// direction is formed in FP64 and kept as FP32 value + FP32 rounding error.
// A pose with a non-finite entry yields |d| = NaN (the particle's loss
// becomes NaN and it gets no weight).  gd receives gamma(d) of the unit
// direction (4 frequencies, 27 values, zero-padded to 32).
// ---------------------------------------------------------------------------
__device__ __forceinline__ void make_ray(const float* __restrict__ p, int u, int v, float fx,
                                         float fy, float cx, float cy, Ray& ray,
                                         float* __restrict__ g) {
    const double ax = ((double)u + 0.5 - (double)cx) / (double)fx;
    const double ay = -((double)v + 0.5 - (double)cy) / (double)fy;
    const double az = -1.0;
    double d[3];
#pragma unroll
    for (int c = 0; c < 3; ++c)
        d[c] = (double)p[4 * c] * ax + (double)p[4 * c + 1] * ay + (double)p[4 * c + 2] * az;
    const double dn64 = sqrt(d[0] * d[0] + d[1] * d[1] + d[2] * d[2]);
    bool finite_pose = true;
#pragma unroll
    for (int c = 0; c < 12; ++c) finite_pose = finite_pose && isfinite(p[c]);
    const float dx = (float)d[0], dy = (float)d[1], dz = (float)d[2];
    ray.ox = p[3]; ray.oy = p[7]; ray.oz = p[11];
    ray.dnorm = finite_pose ? (float)dn64 : __int_as_float(0x7fc00000);
    ray.dx = dx; ray.dy = dy; ray.dz = dz; ray.pad = 0.f;
    ray.lx = (float)(d[0] - (double)dx);
    ray.ly = (float)(d[1] - (double)dy);
    ray.lz = (float)(d[2] - (double)dz);
    ray.pad2 = 0.f;
    const float h[3] = {(float)(d[0] / dn64), (float)(d[1] / dn64), (float)(d[2] / dn64)};
    g[0] = h[0]; g[1] = h[1]; g[2] = h[2];
#pragma unroll
    for (int k = 0; k < kLdir; ++k) {
        const float f = (float)(1 << k);
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            float sn, cs;
            sincosf(f * h[c], &sn, &cs);
            g[3 + 6 * k + c] = sn;
            g[6 + 6 * k + c] = cs;
        }
    }
#pragma unroll
    for (int c = kGd; c < kGdPad; ++c) g[c] = 0.f;
}

// Query pixel set: B distinct pixels of a W x H level image, uniformly without
// replacement, by Floyd's sampling algorithm (Bentley & Floyd, CACM 1987):
// for j = n-B .. n-1 draw t uniform in [0, j] and take t unless already
// taken, else j.  t = floor(r (j + 1) / 2^64), r = value j-(n-B) of
// SplitMix64 stream (seed, ctr).  out[2i], out[2i+1] = (q % W, q / W).
// One warp: the draws are independent, the tests against the pixels taken so
// far go 32 at a time.  t and c: B values of scratch each.
__device__ __forceinline__ void draw_pixel_set(int W, int H, int B, uint64_t seed, uint64_t ctr,
                                               int32_t* __restrict__ out, long* __restrict__ t,
                                               long* __restrict__ c) {
    const int lane = threadIdx.x & 31;
    const long j0 = (long)W * H - B;
    for (int m = lane; m < B; m += 32) {
        const uint64_t r = cb_rand(seed, ctr, (uint64_t)m);
        t[m] = (long)(((u128)r * (u128)(uint64_t)(j0 + m + 1)) >> 64);
    }
    __syncwarp();
    for (int m = 0; m < B; ++m) {
        const long tm = t[m];
        bool dup = false;
        for (int i = lane; i < m; i += 32) dup = dup || c[i] == tm;
        dup = __any_sync(0xffffffffu, dup);
        if (lane == 0) c[m] = dup ? j0 + m : tm;
        __syncwarp();
    }
    for (int m = lane; m < B; m += 32) {
        out[2 * m] = (int32_t)(c[m] % W);
        out[2 * m + 1] = (int32_t)(c[m] / W);
    }
}

// Stratified coarse samples of the warp's rays r0 .. r0 + live - 1, ray index r
// of its stream and counter ctr per lane: z_k = near + (far - near)(k + u_k)/n_c,
// u_k = 1/2 or value r*n_c + k of SplitMix64 stream (seed, ctr).  A lane per
// sample, so that a ray's samples go out together.  The 53 bits of u_k are
// rounded to FP32 once, as the FP64 value k 2^-53 would be.
__device__ __forceinline__ void coarse_samples_warp(long r, uint64_t ctr, int live, int nc,
                                                    float near_z, float far_z, int jitter,
                                                    uint64_t seed, float* __restrict__ z) {
    const int lane = threadIdx.x & 31;
    const float span = far_z - near_z;
    const int total = live * nc;
#pragma unroll 4
    for (int e0 = 0; e0 < total; e0 += 32) {
        const int e = e0 + lane;
        const int q = e / nc, k = e - q * nc;   // (q mod 32 in the last, partial turn)
        const uint64_t at = (uint64_t)__shfl_sync(0xffffffffu, (long long)r, q) * nc + k;
        const uint64_t c = __shfl_sync(0xffffffffu, (unsigned long long)ctr, q);
        const float uk = jitter ? (float)(cb_rand(seed, c, at) >> 11) * 0x1.0p-53f : 0.5f;
        if (e < total) z[e] = near_z + span * ((float)k + uk) / (float)nc;
    }
}

// Store the warp's gamma(d) rows (lane's row in g[lane][..]) coalesced.
__device__ __forceinline__ void store_gd_warp(const float (&g)[32][kGdPad + 1], int live,
                                              float* __restrict__ gd) {
    const int lane = threadIdx.x & 31;
    __syncwarp();
#pragma unroll 8
    for (int q = 0; q < live; ++q) gd[(size_t)q * kGdPad + lane] = g[q][lane];
}

// ---------------------------------------------------------------------------
// Compositing and sampling of 32 consecutive rays by one warp, a lane per ray.
//
// The sums and products along a ray keep their order, so a ray is one serial
// chain; a warp per 32 rays leaves the chip about 8 chains of 32 rays per SM
// at 38,400 rays.  What bounds these kernels when a lane also fetches its own
// samples is the fetch: 32 different lines per load, each a wait on L2.  So
// the warp brings the rows in together, coalesced, into shared memory, and
// only the chains run there (38,400 rays x (64 + 128) samples: sampling 165 ->
// 60 us, composite 177 -> 57 us, of which reading the samples takes 22).
// ---------------------------------------------------------------------------
__device__ __forceinline__ void copy_async16(void* dst, const void* src) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(
                     (uint32_t)__cvta_generic_to_shared(dst)),
                 "l"(src)
                 : "memory");
}
__device__ __forceinline__ void copy_async4(void* dst, const void* src) {
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(
                     (uint32_t)__cvta_generic_to_shared(dst)),
                 "l"(src)
                 : "memory");
}
__device__ __forceinline__ void copy_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
__device__ __forceinline__ void copy_wait() { asm volatile("cp.async.wait_group 0;" ::: "memory"); }

// Floats of shared memory of importance_warp: z and CDF of 32 rays, [sample][33]
// (a ray's samples go to 32 banks when they are stored, a sample's rays when
// they are read), and 32 samples on their way out.
__host__ __device__ constexpr int importance_floats(int nc) { return (2 * nc + 32) * 33; }

// Coarse composite (Eq. 1 quadrature) and inverse-CDF importance samples of
// rays r0 .. r0 + 31 (those below n): edges = midpoints of consecutive coarse
// z; pdf over the interior bins proportional to w_1..w_{n_c-2} + 1e-5;
// u_j = j/(n_f - 1); the bin is the first CDF entry strictly greater than u_j
// (u sorted: one sweep).
__device__ __forceinline__ void importance_warp(const Ray* __restrict__ rays,
                                                const float* __restrict__ zc,
                                                const float4* __restrict__ oc, int nc, int r0,
                                                int n, int nf, float* __restrict__ zf,
                                                float* __restrict__ sm) {
    const int lane = threadIdx.x & 31;
    const int live = min(32, n - r0);
    float* zs = sm;
    float* cdf = zs + nc * 33;
    float* ob = cdf + nc * 33;
    zc += (size_t)r0 * nc;
    oc += (size_t)r0 * nc;
    zf += (size_t)r0 * nf;
#pragma unroll 8
    for (int q = 0; q < 32; ++q) {
        const size_t row = (size_t)min(q, live - 1) * nc;
        for (int k = lane; k < nc; k += 32) {
            copy_async4(&zs[k * 33 + q], &zc[row + k]);
            copy_async4(&cdf[k * 33 + q], &oc[row + k].x);
        }
    }
    copy_commit();
    const float dn = rays[r0 + min(lane, live - 1)].dnorm;
    copy_wait();
    __syncwarp();
    zs += lane;
    cdf += lane;
    float T = 1.0f;
    float tot = 0.0f;
#pragma unroll 4
    for (int k = 0; k < nc - 1; ++k) {
        const float sg = fmaxf(cdf[k * 33], 0.0f);
        const float delta = (zs[(k + 1) * 33] - zs[k * 33]) * dn;
        const float a = 1.0f - expf(-sg * delta);
        // T a + 1e-5, rounded twice in every fourth bin and once in the others.
        // No formula asks for that: a loop unrolled by four, a thread per ray,
        // was once compiled so, and every result since has these roundings.  The
        // inverse CDF is ill-conditioned (an ulp here moves samples of nearly
        // empty bins, and the weights of a few particles beyond FP32's own
        // error), so one form for all bins would be another sampler, not a
        // more exact one.
        const float w = (k & 3) == 3 ? __fadd_rn(__fmul_rn(T, a), 1e-5f) : fmaf(T, a, 1e-5f);
        T *= (1.0f - a);
        if (k >= 1) {
            cdf[k * 33] = w;   // pdf of bin k-1, normalised below
            tot += w;
        }
    }
    const int ne = nc - 1;
    cdf[0] = 0.0f;
    float run = 0.0f;
#pragma unroll 4
    for (int i = 1; i < ne; ++i) {
        run += cdf[i * 33] / tot;
        cdf[i * 33] = run;
    }
    // the sweep keeps the bin's ends in registers: CDF (c_lo, c_hi) and edge
    // (eb, ea) of entries max(idx - 1, 0) and min(idx, ne - 1)
    int idx = 0;
    float c_lo = 0.0f, c_hi = 0.0f;
    float ea = 0.5f * (zs[0] + zs[33]), eb = ea;
    for (int j0 = 0; j0 < nf; j0 += 32) {
        const int m = min(32, nf - j0);
        for (int jj = 0; jj < m; ++jj) {
            const int j = j0 + jj;
            const float u = nf > 1 ? (float)j / (float)(nf - 1) : 0.0f;
            while (idx < ne && c_hi <= u) {
                ++idx;
                c_lo = c_hi;
                eb = ea;
                if (idx < ne) {
                    c_hi = cdf[idx * 33];
                    ea = 0.5f * (zs[idx * 33] + zs[(idx + 1) * 33]);
                }
            }
            float denom = c_hi - c_lo;
            if (denom < 1e-5f) denom = 1.0f;
            const float t = (u - c_lo) / denom;
            ob[jj * 33 + lane] = eb + t * (ea - eb);
        }
        __syncwarp();
        if (lane < m)
            for (int q = 0; q < live; ++q) zf[(size_t)q * nf + j0 + lane] = ob[lane * 33 + q];
        __syncwarp();
    }
}

struct RayResult {
    float r, g, b;
    float z_trans, z_opaque, F;
};

// Shared memory of composite_warp: per ray a ring of 16 samples of each pass,
// the values [slot][32] (read without conflicts), z [slot][33].
constexpr int kRing = 16, kRingStep = 8;
struct CompositeSmem {
    float4 v[2][kRing][32];
    float z[2][kRing][33];
};

// Final composite of rays r0 .. r0 + 31 over the merged coarse + fine samples
// (both sorted; equal z take the coarse sample first), Eq. 5 on the running
// weight sum and F of Eq. 6 (F = 1 without rejection).
//
// Which sample comes next is known only ray by ray, so every 8 samples the
// warp tops up all rays' rings, 8 lanes per ray and pass (128-byte pieces),
// with what the 8 samples after the coming ones may need.
__device__ __forceinline__ RayResult composite_warp(const Ray* __restrict__ rays,
                                                    const float* __restrict__ za,
                                                    const float4* __restrict__ oa, int nc,
                                                    const float* __restrict__ zb,
                                                    const float4* __restrict__ ob, int nf, int r0,
                                                    int n_rays, float alpha, float tau, int use_rej,
                                                    CompositeSmem& sm) {
    const int lane = threadIdx.x & 31;
    const int live = min(32, n_rays - r0);
    // this lane's part of a top-up: entry e of pass `list` of rays 2 p + half
    const int e = lane & 7, list = (lane >> 3) & 1, half = lane >> 4;
    const int cnt = list ? nf : nc;
    const float* const zl = (list ? zb : za) + (size_t)r0 * cnt;
    const float4* const ol = (list ? ob : oa) + (size_t)r0 * cnt;
    int ia = 0, ib = 0, la = 0, lb = 0;   // taken and loaded so far
    auto top_up = [&]() {
        const int pa = ia << 16 | la, pb = ib << 16 | lb;
#pragma unroll 4
        for (int p = 0; p < 16; ++p) {
            const int q = 2 * p + half;
            const int sa = __shfl_sync(0xffffffffu, pa, q), sb = __shfl_sync(0xffffffffu, pb, q);
            const int st = list ? sb : sa;
            const int i = (st & 0xffff) + e;
            if (i < min((st >> 16) + kRing, cnt)) {
                const size_t at = (size_t)min(q, live - 1) * cnt + i;
                copy_async16(&sm.v[list][i & (kRing - 1)][q], &ol[at]);
                copy_async4(&sm.z[list][i & (kRing - 1)][q], &zl[at]);
            }
        }
        copy_commit();
        la = min(max(la, min(la + kRingStep, ia + kRing)), nc);
        lb = min(max(lb, min(lb + kRingStep, ib + kRing)), nf);
    };
    top_up();
    top_up();
    const float dn = rays[r0 + min(lane, live - 1)].dnorm;
    const int n = nc + nf;
    float zcur = 0.f;
    float4 vcur = make_float4(0.f, 0.f, 0.f, 0.f);
    float T = 1.0f, cr = 0.f, cg = 0.f, cb = 0.f, Wc = 0.f;
    float zt = 0.f, zo = 0.f;
    bool have_t = false;
    auto add = [&](float delta) {
        const float sg = fmaxf(vcur.x, 0.0f);
        const float a = 1.0f - expf(-sg * delta);
        const float w = T * a;
        cr += w * vcur.y; cg += w * vcur.z; cb += w * vcur.w;
        T *= (1.0f - a);
        Wc += w;
        if (!have_t && Wc >= alpha) { zt = zcur; have_t = true; }
        if (Wc <= 1.0f - alpha) zo = zcur;
    };
    for (int k0 = 0; k0 < n; k0 += kRingStep) {
        copy_wait();
        __syncwarp();   // what was loaded is there, what was taken may be overwritten
        if (k0 > 0) top_up();
        const int m = min(kRingStep, n - k0);
        for (int kk = 0; kk < m; ++kk) {
            const float ha = sm.z[0][ia & (kRing - 1)][lane], hb = sm.z[1][ib & (kRing - 1)][lane];
            const bool second = !(ib >= nf || (ia < nc && ha <= hb));
            const float znext = second ? hb : ha;
            const float4 vnext = sm.v[second][(second ? ib : ia) & (kRing - 1)][lane];
            if (second) ++ib;
            else ++ia;
            if (k0 + kk > 0) add((znext - zcur) * dn);
            else zt = zo = znext;
            zcur = znext;
            vcur = vnext;
        }
    }
    add(1e10f);
    RayResult res;
    res.r = cr; res.g = cg; res.b = cb;
    res.z_trans = zt; res.z_opaque = zo;
    res.F = use_rej ? fmaxf(zo - zt, tau) : 1.0f;
    return res;
}

// Box-filtered colour of level-image pixel (u, v) (factor x factor block of
// the full-resolution image, W pixels per row); NaN outside the level image.
__device__ __forceinline__ float4 observed_colour(const float* __restrict__ img, int W, int H,
                                                  int factor, int u, int v) {
    if (u < 0 || v < 0 || u >= W / factor || v >= H / factor) {
        const float nan = __int_as_float(0x7fc00000);
        return make_float4(nan, nan, nan, nan);
    }
    float s0 = 0.f, s1 = 0.f, s2 = 0.f;
    for (int dy = 0; dy < factor; ++dy) {
        const float* row = img + ((size_t)(v * factor + dy) * W + (size_t)u * factor) * 3;
        for (int dx = 0; dx < factor; ++dx) {
            s0 += row[3 * dx]; s1 += row[3 * dx + 1]; s2 += row[3 * dx + 2];
        }
    }
    const float inv = 1.0f / (float)(factor * factor);
    return make_float4(s0 * inv, s1 * inv, s2 * inv, 0.f);
}

// E = squared RGB distance between the rendered colour and the box-filtered
// observed pixel (u, v) of the level image (factor x factor block of the
// full-resolution image, W pixels per row).  NaN when the ray is invalid.
__device__ __forceinline__ float photometric_E(const float* __restrict__ img, int W, int factor,
                                               int u, int v, const RayResult& c, float dn) {
    float s0 = 0.f, s1 = 0.f, s2 = 0.f;
    for (int dy = 0; dy < factor; ++dy) {
        const float* row = img + ((size_t)(v * factor + dy) * W + (size_t)u * factor) * 3;
        for (int dx = 0; dx < factor; ++dx) {
            s0 += row[3 * dx]; s1 += row[3 * dx + 1]; s2 += row[3 * dx + 2];
        }
    }
    const float inv = 1.0f / (float)(factor * factor);
    const float e0 = s0 * inv - c.r, e1 = s1 * inv - c.g, e2 = s2 * inv - c.b;
    return isfinite(dn) ? e0 * e0 + e1 * e1 + e2 * e2 : __int_as_float(0x7fc00000);
}

// ---------------------------------------------------------------------------
// Block reductions (blockDim.x a multiple of 32, at most 1024).
// ---------------------------------------------------------------------------
__device__ __forceinline__ double block_max_d(double v, double* sh) {
    for (int o = 16; o > 0; o >>= 1) v = fmax(v, __shfl_xor_sync(0xffffffffu, v, o));
    const int w = threadIdx.x >> 5, l = threadIdx.x & 31;
    __syncthreads();
    if (l == 0) sh[w] = v;
    __syncthreads();
    if (w == 0) {
        v = l < (int)(blockDim.x >> 5) ? sh[l] : -INFINITY;
        for (int o = 16; o > 0; o >>= 1) v = fmax(v, __shfl_xor_sync(0xffffffffu, v, o));
        if (l == 0) sh[0] = v;
    }
    __syncthreads();
    return sh[0];
}

__device__ __forceinline__ double block_sum_d(double v, double* sh) {
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    const int w = threadIdx.x >> 5, l = threadIdx.x & 31;
    __syncthreads();
    if (l == 0) sh[w] = v;
    __syncthreads();
    if (w == 0) {
        v = l < (int)(blockDim.x >> 5) ? sh[l] : 0.0;
        for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
        if (l == 0) sh[0] = v;
    }
    __syncthreads();
    return sh[0];
}

// Inclusive scan of one u64 per thread across the block; returns the
// inclusive prefix and writes the block total to *total.
__device__ __forceinline__ u64 block_scan_u64(u64 v, u64* sh, u64* total) {
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, nw = blockDim.x >> 5;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const u64 t = __shfl_up_sync(0xffffffffu, v, o);
        if (lane >= o) v += t;
    }
    __syncthreads();
    if (lane == 31) sh[wid] = v;
    __syncthreads();
    if (wid == 0) {
        u64 s = lane < nw ? sh[lane] : 0ull;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const u64 t = __shfl_up_sync(0xffffffffu, s, o);
            if (lane >= o) s += t;
        }
        if (lane < nw) sh[lane] = s;
    }
    __syncthreads();
    const u64 before = wid > 0 ? sh[wid - 1] : 0ull;
    *total = sh[nw - 1];
    return v + before;
}

// ---------------------------------------------------------------------------
// Eq. 6 weights of one particle set, by one cluster of C CTAs of 128 threads
// (C = 1, 2, 4, 8): S_i = sum_j E_ij F_ij (FP32, j order), log w_i = 4 (log B -
// log max(S_i, s_min)), normalisation w_i = exp(log w_i - logsumexp) in FP64,
// mask_i = (w_i >= rho / N).  Non-finite S_i -> log w = -inf (returned count of
// such particles).
//
// FP64 is what this costs: the chip has about two FP64 lanes per SM, so a
// function over 32 warps is 32 times its time over one.  Hence the cluster
// (a particle's functions run on eight SMs at once), and everything that is
// the same for all particles is evaluated by one warp.  The particles fall to
// the threads as to one block of 1,024 (particle i to thread i mod 1,024,
// whose warps go round the CTAs), and the sums over them are taken over its
// 32 warps in that order, so the figures do not depend on C.  32 particles x 8
// pixels: 26 us by one block, 10 now; 600 x 64: 54 and 13.
// ---------------------------------------------------------------------------
constexpr int kTeamThreads = 128, kTeamMost = 8;
// CTAs for n particles: all eight unless fewer warps hold one particle a lane
inline int team_ctas(int n) { return n <= 32 ? 1 : n <= 64 ? 2 : n <= 128 ? 4 : kTeamMost; }

struct Team {
    int rank, ctas;      // this CTA of how many
    int warp, lane;      // warp of the whole team
    int first, step;     // particles first, first + step, ...
};
__device__ __forceinline__ Team make_team() {
    Team t;
    asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(t.rank));
    asm volatile("mov.u32 %0, %%cluster_nctarank;" : "=r"(t.ctas));
    t.lane = threadIdx.x & 31;
    t.warp = (threadIdx.x >> 5) * t.ctas + t.rank;
    t.first = t.warp * 32 + t.lane;
    t.step = t.ctas * kTeamThreads;
    return t;
}
__device__ __forceinline__ void team_barrier() {
    asm volatile("barrier.cluster.arrive.release.aligned;\nbarrier.cluster.wait.acquire.aligned;" ::
                     : "memory");
}
// v to the same variable of every CTA of the team, by the first lanes of a warp
__device__ __forceinline__ void team_store(const Team& t, double* at, double v) {
    if (t.lane < t.ctas) {
        uint32_t a;
        asm volatile("mapa.shared::cluster.u32 %0, %1, %2;"
                     : "=r"(a)
                     : "r"((uint32_t)__cvta_generic_to_shared(at)), "r"(t.lane));
        asm volatile("st.shared::cluster.f64 [%0], %1;" ::"r"(a), "d"(v) : "memory");
    }
}
__device__ __forceinline__ double warp_sum_d(double v) {
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}
__device__ __forceinline__ double warp_max_d(double v) {
    for (int o = 16; o > 0; o >>= 1) v = fmax(v, __shfl_xor_sync(0xffffffffu, v, o));
    return v;
}
// Sums over the team of K values per thread (warps without a particle hold
// zeros and skip their part); sh: K rows of 32, res: K, both shared memory.
// Ends with the results in res in every CTA.
template <int K>
__device__ __forceinline__ void team_sum(const Team& t, int n, const double (&v)[K],
                                         double (*sh)[32], double* res) {
    const bool live = t.warp * 32 < n;
#pragma unroll
    for (int k = 0; k < K; ++k) team_store(t, &sh[k][t.warp], live ? warp_sum_d(v[k]) : 0.0);
    team_barrier();
    const int w = threadIdx.x >> 5;
#pragma unroll
    for (int k = 0; k < K; ++k)
        if ((k & 3) == w) {
            const double s = warp_sum_d(t.lane < t.ctas * 4 ? sh[k][t.lane] : 0.0);
            if (t.lane == 0) res[k] = s;
        }
    __syncthreads();
}

// A launch of `teams` teams of `ctas` CTAs.
template <typename... P, typename... A>
cudaError_t launch_teams(void (*fn)(P...), int teams, int ctas, cudaStream_t s, A&&... args) {
    cudaLaunchConfig_t c = {};
    c.gridDim = dim3((unsigned)(teams * ctas));
    c.blockDim = dim3(kTeamThreads);
    c.stream = s;
    cudaLaunchAttribute at;
    at.id = cudaLaunchAttributeClusterDimension;
    at.val.clusterDim.x = (unsigned)ctas;
    at.val.clusterDim.y = at.val.clusterDim.z = 1;
    c.attrs = &at;
    c.numAttrs = 1;
    return cudaLaunchKernelEx(&c, fn, std::forward<A>(args)...);
}

struct TeamSmem {
    double log_b, lse, mx;
    double max_sh[32], sum_sh[1][32], sum[1];
    double bad_sh[1][32], bad[1];
};

__device__ __forceinline__ int weights_team(const Team& t, TeamSmem& sm,
                                            const float* __restrict__ e_ray, int N, int B,
                                            double s_min, double rho, float* __restrict__ logw,
                                            double* __restrict__ l64, double* __restrict__ w,
                                            uint8_t* __restrict__ mask,
                                            float* __restrict__ S_dbg) {
    const int wid = threadIdx.x >> 5;
    if (wid == 3 && t.lane == 0) sm.log_b = log((double)B);
    // S of the first particle while the fourth warp takes the logarithm
    auto total = [&](int i) {
        const float* e = e_ray + (size_t)i * B;
        float S = 0.0f;
#pragma unroll 16
        for (int j = 0; j < B; ++j) S += e[j];
        return S;
    };
    float S = t.first < N ? total(t.first) : 0.0f;
    team_barrier();   // also: every CTA of the team runs before one stores into another
    const double logB = sm.log_b;
    double mx = -INFINITY;
    int nbad = 0;
    for (int i = t.first; i < N; i += t.step) {
        if (i != t.first) S = total(i);
        if (S_dbg) S_dbg[i] = S;
        double l;
        if (isfinite(S)) {
            const double sc = fmax((double)S, s_min);
            l = 4.0 * (logB - log(sc));
        } else {
            l = -INFINITY;
            ++nbad;
        }
        l64[i] = l;
        if (logw) logw[i] = (float)l;
        mx = fmax(mx, l);
    }
    // (log w may be NaN only through s_min; fmax passes it by)
    const bool live = t.warp * 32 < N;
    nbad = __reduce_add_sync(0xffffffffu, nbad);
    team_store(t, &sm.max_sh[t.warp], live ? warp_max_d(mx) : -INFINITY);
    team_store(t, &sm.bad_sh[0][t.warp], (double)nbad);
    team_barrier();
    mx = t.lane < t.ctas * 4 ? sm.max_sh[t.lane] : -INFINITY;
    if (wid == 0) {
        mx = warp_max_d(mx);
        if (t.lane == 0) sm.mx = mx;
    } else if (wid == 1) {
        nbad = __reduce_add_sync(0xffffffffu, t.lane < t.ctas * 4 ? (int)sm.bad_sh[0][t.lane] : 0);
        if (t.lane == 0) sm.bad[0] = (double)nbad;
    }
    __syncthreads();
    mx = sm.mx;
    double acc[1] = {0.0};
    if (mx > -INFINITY)
        for (int i = t.first; i < N; i += t.step) acc[0] += exp(l64[i] - mx);
    team_sum<1>(t, N, acc, sm.sum_sh, sm.sum);
    if (wid == 0 && t.lane == 0) sm.lse = mx + log(sm.sum[0]);
    const double thr = rho / (double)N;
    __syncthreads();
    const double lse = sm.lse;
    for (int i = t.first; i < N; i += t.step) {
        const double wi = (mx > -INFINITY) ? exp(l64[i] - lse) : 0.0;
        w[i] = wi;
        mask[i] = (uint8_t)(wi >= thr && wi > 0.0);
    }
    return (int)sm.bad[0];
}

// ---------------------------------------------------------------------------
// Systematic resampling on an exact integer CDF, by one block:
// d_idx[k] = smallest i with C_i N_out 2^53 > (k 2^53 + U) T, where
// q_i = floor(w_i 2^s), s = 50 - e - ceil(log2 N_in), e = exponent of max w,
// C = inclusive prefix of q, T = C_{N_in-1}, U = floor(u0 2^53).  Returns
// false (every idx = -1) for negative, non-finite or all-zero weights.
// ---------------------------------------------------------------------------
__device__ __forceinline__ bool resample_block(const double* __restrict__ w, int n_in, int n_out,
                                               double u0, int32_t* __restrict__ idx,
                                               u64* __restrict__ cdf) {
    __shared__ u64 shu[32];
    __shared__ double shd[32];
    __shared__ int bad;
    if (threadIdx.x == 0) bad = 0;
    __syncthreads();
    double mx = 0.0;
    for (int i = threadIdx.x; i < n_in; i += blockDim.x) {
        const double wi = w[i];
        if (!(wi >= 0.0) || isinf(wi)) bad = 1;
        else mx = fmax(mx, wi);
    }
    mx = block_max_d(mx, shd);
    if (bad || !(mx > 0.0)) {
        for (int k = threadIdx.x; k < n_out; k += blockDim.x) idx[k] = -1;
        return false;
    }
    int e;
    frexp(mx, &e);
    int lg = 0;
    while ((1ll << lg) < (long long)n_in) ++lg;
    const int sh = 50 - e - lg;
    u64 carry = 0;
    for (int base = 0; base < n_in; base += blockDim.x) {
        const int i = base + threadIdx.x;
        const u64 q = i < n_in ? (u64)floor(ldexp(w[i], sh)) : 0ull;
        u64 tot;
        const u64 incl = block_scan_u64(q, shu, &tot);
        if (i < n_in) cdf[i] = carry + incl;
        carry += tot;
        __syncthreads();
    }
    const u64 T = carry;
    const u64 U = (u64)floor(ldexp(u0, 53));
    __syncthreads();
    if (T == 0ull) {
        for (int k = threadIdx.x; k < n_out; k += blockDim.x) idx[k] = -1;
        return false;
    }
    for (int k = threadIdx.x; k < n_out; k += blockDim.x) {
        const u128 rhs = (((u128)(u64)k * T) << 53) + (u128)U * T;
        int lo = 0, hi = n_in - 1;  // answer in [lo, hi]; C_{n_in-1} always satisfies
        while (lo < hi) {
            const int mid = (lo + hi) >> 1;
            const u128 lhs = ((u128)cdf[mid] * (u64)n_out) << 53;
            if (lhs > rhs) hi = mid;
            else lo = mid + 1;
        }
        idx[k] = lo;
    }
    return true;
}

// ---------------------------------------------------------------------------
// Prediction of one particle by four lanes: O = P * Exp(q[0..2], (0, q[3], 0))
// in FP64 (optionally P * O_t * Exp: odom is the 3x4 relative motion O_t, NULL
// for the identity).  SE(3) exponential: R = I + a K + b K^2, t = (I + b K + c
// K^2) rho with K = [omega]x, th = |omega|, a = sin th / th, b = (1 - cos
// th)/th^2, c = (th - sin th)/th^3 (series values below th = 1e-8).
//
// A chain of FP64 functions: its latency is the whole cost of a small call, and
// the FP64 lanes that of a large one.  Lane c draws normal c of the motion
// noise (normals 4k .. 4k+3 of stream (seed, ctr), scaled by (sigma_t, sigma_t,
// sigma_t, sigma_yaw)), lanes 0..2 divide for a, b and c at once, and lane r
// forms row r of the result (32 particles: 19 us with a lane each, 10 now).  All
// four lanes enter together; `live` lanes 0..2
// store.
// ---------------------------------------------------------------------------
__device__ __forceinline__ void predict_quad(const float* __restrict__ P0, uint64_t seed,
                                             uint64_t ctr, long k, float sigma_t, float sigma_yaw,
                                             bool live, float* __restrict__ O,
                                             const float* __restrict__ odom) {
    const int c4 = threadIdx.x & 3, base = threadIdx.x & 28, r = min(c4, 2);
    double q[4];
    const double mine =
        (c4 < 3 ? (double)sigma_t : (double)sigma_yaw) * cb_normal(seed, ctr, 4ull * k + c4);
#pragma unroll
    for (int c = 0; c < 4; ++c) q[c] = __shfl_sync(0xffffffffu, mine, base + c);
    double P[4];
    if (odom) {
#pragma unroll
        for (int c = 0; c < 4; ++c) {
            double s = (c == 3) ? (double)P0[4 * r + 3] : 0.0;
#pragma unroll
            for (int m = 0; m < 3; ++m) s += (double)P0[4 * r + m] * (double)odom[4 * m + c];
            P[c] = s;
        }
    } else {
#pragma unroll
        for (int c = 0; c < 4; ++c) P[c] = (double)P0[4 * r + c];
    }
    const double om[3] = {0.0, q[3], 0.0};
    const double th2 = om[0] * om[0] + om[1] * om[1] + om[2] * om[2];
    const double th = sqrt(th2);
    const double K[9] = {0.0, -om[2], om[1], om[2], 0.0, -om[0], -om[1], om[0], 0.0};
    double K2[9];
#pragma unroll
    for (int i = 0; i < 3; ++i)
#pragma unroll
        for (int c = 0; c < 3; ++c)
            K2[3 * i + c] = K[3 * i] * K[c] + K[3 * i + 1] * K[3 + c] + K[3 * i + 2] * K[6 + c];
    const double sn = sin(th), cs = cos(th);
    const double num = r == 0 ? sn : r == 1 ? 1.0 - cs : th - sn;
    const double den = r == 0 ? th : r == 1 ? th2 : th2 * th;
    const double abc = th < 1e-8 ? (r == 0 ? 1.0 : r == 1 ? 0.5 : 1.0 / 6.0) : num / den;
    const double a = __shfl_sync(0xffffffffu, abc, base);
    const double b = __shfl_sync(0xffffffffu, abc, base + 1);
    const double cc = __shfl_sync(0xffffffffu, abc, base + 2);
    double E[12];
#pragma unroll
    for (int i = 0; i < 3; ++i) {
        double t = 0.0;
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            const double I = (i == c) ? 1.0 : 0.0;
            E[4 * i + c] = I + a * K[3 * i + c] + b * K2[3 * i + c];
            t += (I + b * K[3 * i + c] + cc * K2[3 * i + c]) * q[c];
        }
        E[4 * i + 3] = t;
    }
    float v[4];
#pragma unroll
    for (int c = 0; c < 4; ++c) {
        double s = (c == 3) ? P[3] : 0.0;
#pragma unroll
        for (int m = 0; m < 3; ++m) s += P[m] * E[4 * m + c];
        v[c] = (float)s;
    }
    if (live && c4 < 3) {
#pragma unroll
        for (int c = 0; c < 4; ++c) O[4 * r + c] = v[c];
    }
}

// Mean position and trace of the population covariance (FP64), one block.
__device__ __forceinline__ void spread_block(const float* __restrict__ P, int N,
                                             double* __restrict__ out) {
    __shared__ double sh[32];
    double m[3];
    for (int c = 0; c < 3; ++c) {
        double v = 0.0;
        for (int i = threadIdx.x; i < N; i += blockDim.x) v += (double)P[12 * (size_t)i + 4 * c + 3];
        m[c] = block_sum_d(v, sh) / N;
    }
    double t = 0.0;
    for (int i = threadIdx.x; i < N; i += blockDim.x)
        for (int c = 0; c < 3; ++c) {
            const double d = (double)P[12 * (size_t)i + 4 * c + 3] - m[c];
            t += d * d;
        }
    t = block_sum_d(t, sh);
    if (threadIdx.x == 0) {
        out[0] = m[0]; out[1] = m[1]; out[2] = m[2];
        out[3] = t / N;
    }
}

}  // namespace mcl

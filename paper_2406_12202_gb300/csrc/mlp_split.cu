// mlp_split.cu -- the FP32 form of the NeRF MLP on the tensor cores (tcgen05).
//
// Every operand is split into two FP16 numbers, x s = hi + lo with s a power
// of two (hi = x s rounded to nearest, lo the rounded rest: 22 to 23
// significant bits), and a product of two FP32 matrices becomes hi hi + hi lo
// + lo hi on FP16 MMAs with FP32 accumulators.  s brings the largest entry of
// an operand group just below 2^15, so that neither half leaves FP16's range:
// one s per row of the activations, one per layer of the weights.
//
// tcgen05 truncates as it accumulates (measured: towards zero at the
// accumulator's last place, once per MMA of 16 products), which over a row of
// 256 products would cost more than the FP32 FMA chain it replaces.  So the
// accumulator is emptied every 64 products: the small cross terms are added
// first, then the four hi hi MMAs, and the epilogue threads add the chunk,
// rescaled, to an FP32 sum in registers (round to nearest).  Measured against
// FP64 on 256-long rows of random data: relative error 1.4e-7 (post-ReLU
// activations) and 2.0e-7 (all terms of one sign), against 2.0e-7 and 2.2e-7
// of an FP32 FMA chain; emptied every 128 products 2.0e-7 and 4.9e-7, not at
// all 3.4e-7 and 1.2e-6.  What is left is mostly a shortfall of every chunk
// (kUnbias).  The whole MLP on twelve dense maps (He-normal, and smooth ones whose
// weights fall as 2^-k with the frequency), 40,000 points each: the error of the
// densities is 0.50 to 0.88 of the SIMT kernels' (mlp_fp32.cu), of the colours
// 0.44 to 0.54 (rms; the largest errors 0.50 to 0.77 and 0.32 to 0.55).  Other maps
// run on those kernels (pairs_are_exact).
//
// A CTA pair (the two SMs of a TPC, tcgen05 cta_group::2) walks over units of
// 256 rows (samples of the pass, row = ray * S + k), 128 rows per CTA, through
// all layers, as mlp_tc.cu does in BF16: the activations stay in shared
// memory (hi and lo, 128 KB per CTA), gamma(x) beside them (32 KB, read by
// layer 1 and the skip layer), and each CTA streams its half of the weight
// blocks through a ring of 4 x 16 KB (hi and lo of two chunks).  The pair is
// what makes that fit: one CTA alone would read 96 bytes per cycle of shared
// memory for its MMAs and take 43 of weights, over the 128 there are, with a
// ring of one chunk (measured: 20 to 30 ms for the sampler below).
//
// What bounds it: the tensor pipe takes 34 chunks x 12 MMAs x 128 cycles =
// 52,000 cycles per unit (N = 144 of the last layer costs as much as 256) and
// a unit takes about 78,000.  In a layer the four chunks run at 1,500 to
// 1,600 cycles each, their sums under the next chunk's MMAs (two
// accumulators, 512 TMEM columns); exposed are the last chunk's sum (1,100
// cycles from the commit), the row's scale (500), the conversion of the first
// 64 columns (800) and the hand-over to the even CTA (500).  Measured: 600 x
// 64 rays of 64 + 128 samples 155.4 -> 15.7 ms by themselves, 58.4 with the
// first pass's densities from the SIMT kernels (mlp_fp32); 262,144 points
// 5.62 -> 0.79 ms, 1,000 points 304 -> 61 us.
//
// Warp roles: warp 0 streams the weights; warp 1 issues the MMAs (even CTA)
// or tells the even CTA that a block has landed (odd CTA); warp 2 (even CTA:
// the gate) does the mbarrier waits for the issuing warp (see mlp_tc.cu);
// warp 3 encodes the next unit's gamma(x); warps 4..11 are the epilogue: warp
// (quadrant q, half j) owns rows 32 q .. +31 and 32 j .. +31 of every 64
// output columns, one row per thread, 128 sums in registers (8 warps with 224
// registers: 16 warps with half the columns each spilled, and with little L1
// beside 227 KB of shared memory a spill goes to the L2).  Waits acquire at
// CTA scope: at cluster scope each one drops the L1 (26 against 20 ms).
// Every wait is bounded (tc_ptx.cuh).
#include <cuda_fp16.h>
#include <math.h>
#include <string.h>

#include <algorithm>
#include <functional>
#include <vector>

#include "internal.cuh"
#include "tc_ptx.cuh"

namespace mcl {

using namespace tc;

namespace {

constexpr int kLayers = 9;                        // trunk 1..8, RGB hidden + density
constexpr uint32_t kStageBytes = 128 * 128;       // half a weight block: 128 rows x 64 k
constexpr uint32_t kBlockBytes = 2 * kStageBytes;
constexpr uint32_t kLastBytes = 72 * 128;         // the last layer's: 72 of 144 rows
constexpr int kStages = 4;                        // lo and hi of two chunks
constexpr uint32_t kChunkBytes = 128 * 128;       // 128 rows x 64 columns, FP16
constexpr uint32_t kActPart = 4 * kChunkBytes;    // hi (or lo) of the activations
constexpr uint32_t kTiles = 2 * kActPart + 2 * kChunkBytes + kStages * kStageBytes;
// A chunk is short by 0.9e-7 of itself on average (1.9e-7 when all terms have
// one sign), and the shortfalls of a map's layers add up; each chunk is
// enlarged by one unit of FP32's last place as it is added (the whole MLP:
// 1.1e-6 to 2.3e-6 without, 4.7e-7 to 7.1e-7 with).
constexpr double kUnbias = 1.0 + 0x1p-23;
constexpr int kEpiWarps = 8, kEpiWarp0 = 4;
constexpr int kThreads = 32 * (kEpiWarp0 + kEpiWarps);
constexpr int kChunks = 1 + 6 * 4 + 5 + 4;        // of 64 products per tile

// chunks of 64 products of a layer; chunk of the activations of step c (-1:
// gamma(x): layer 1, and first in the skip layer, where it does not wait for
// the layer before)
__host__ __device__ constexpr int chunks_of(int l) { return l == 0 ? 1 : (l == kSkip ? 5 : 4); }
__host__ __device__ constexpr int act_chunk(int l, int c) { return l == 0 ? -1 : (l == kSkip ? c - 1 : c); }

struct SplitParams {
    const uint8_t* wblocks;
    const float* bias;           // [8][256] trunk biases, then [3][128] RGB output weights
    const Ray* rays;
    const float* z;
    int S;
    long long M;                 // rows of the pass (upper bound with M_dev)
    const int* M_dev;            // optional: rows in device memory
    RayBias ray_bias;
    float4* out;
    int* abort_flag;
    int* status_code;
    unsigned long long wait_ns;  // limit of the bounded waits
    int hold_weights;            // failure-injection hook: no copies are issued
    float cs[kLayers];           // 1 / (weight scale of the layer), see kUnbias
    float b_sigma;
    float b_out[3];
};

struct __align__(8) SplitBars {
    uint64_t full[kStages], pfull[kStages], empty[kStages];   // pfull: the odd CTA's copy (even CTA)
    uint64_t acc_full[2], acc_empty[2];
    uint64_t a_ready[4], g_ready, g_free, drain, head[4], pair[4];
    uint64_t ex_ready;           // ex_g of the unit written (within the CTA)
    uint32_t tmem_base;
};

// Shared memory behind the operand tiles.
struct __align__(16) Small {
    float w_out[3][128];         // RGB output layer
    // biased exponents: of 1 / s of a row's activations [layer parity] and of
    // its gamma(x) [unit parity], and of the largest output of each thread of
    // the row
    uint8_t ex_h[2][128], ex_g[2][128], ex_m[2][128];
    SplitBars bars;
};
constexpr uint32_t kSmem = kTiles + sizeof(Small);
static_assert(kSmem <= 232448, "shared memory");

// Two FP32 values -> packed FP16 hi and -lo (the mixed-precision subtraction
// gives hi - x in one instruction; the MMAs of the activations' lo negate
// their operand).
__device__ __forceinline__ void split2(float2 t, uint32_t& hi, uint32_t& lo) {
    float x, y;
    asm("cvt.rn.f16x2.f32 %0, %1, %2;" : "=r"(hi) : "f"(t.y), "f"(t.x));
    asm("{\n.reg .b16 p, q;\nmov.b32 {p, q}, %2;\n"
        "sub.rn.f32.f16 %0, p, %3;\nsub.rn.f32.f16 %1, q, %4;\n}"
        : "=f"(x), "=f"(y) : "r"(hi), "f"(t.x), "f"(t.y));
    asm("cvt.rn.f16x2.f32 %0, %1, %2;" : "=r"(lo) : "f"(y), "f"(x));
}

__device__ __forceinline__ float max3(float a, float b, float c) {
    float d;
    asm("max.f32 %0, %1, %2, %3;" : "=f"(d) : "f"(a), "f"(b), "f"(c));
    return d;
}

__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(kThreads, 1)
    k_mlp_split(const __grid_constant__ SplitParams p) {
    extern __shared__ __align__(1024) uint8_t smem[];
    Small& sm = *reinterpret_cast<Small*>(smem + kTiles);
    SplitBars& bars = sm.bars;
    const uint32_t s_hi = smem_u32(smem), s_lo = s_hi + kActPart;
    const uint32_t s_gh = s_lo + kActPart, s_gl = s_gh + kChunkBytes;
    const uint32_t s_ring = s_gl + kChunkBytes;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const uint32_t rank = cluster_ctarank();
    volatile int* abort_flag = p.abort_flag;
    const long long M = p.M_dev ? min(p.M, (long long)*p.M_dev) : p.M;
    // work unit: 256 rows, CTA rank r the tile of rows 128 r .. +127
    const int n_units = (int)((M + 255) / 256);
    const int u0 = blockIdx.x >> 1, du = gridDim.x >> 1;
    constexpr uint16_t kBoth = 3;

    if (tid == 0) {
        for (int i = 0; i < kStages; ++i) {
            mbar_init(smem_u32(&bars.full[i]), 1);
            mbar_init(smem_u32(&bars.pfull[i]), 1);
            mbar_init(smem_u32(&bars.empty[i]), 1);
        }
        for (int i = 0; i < 2; ++i) {
            mbar_init(smem_u32(&bars.acc_full[i]), 1);
            mbar_init(smem_u32(&bars.acc_empty[i]), 2 * kEpiWarps);
        }
        for (int i = 0; i < 4; ++i) {
            mbar_init(smem_u32(&bars.a_ready[i]), 2 * kEpiWarps);
            mbar_init(smem_u32(&bars.head[i]), 32);
            mbar_init(smem_u32(&bars.pair[i]), 2);
        }
        mbar_init(smem_u32(&bars.g_ready), 2 * 4);
        mbar_init(smem_u32(&bars.g_free), 1);
        mbar_init(smem_u32(&bars.ex_ready), 4);
        mbar_init(smem_u32(&bars.drain), 1);
        fence_mbar_init();
    }
    for (int k = tid; k < 3 * 128; k += kThreads) sm.w_out[0][k] = p.bias[8 * 256 + k];
    if (warp == 1) {
        tmem_alloc2(smem_u32(&bars.tmem_base), 512);
        tmem_relinquish2();
    }
    tc_fence_before();
    cluster_sync_all();
    tc_fence_after();
    const uint32_t tmem = bars.tmem_base;
    bool ok = true;

    // gamma(x) of row r of this CTA's tile of unit u (tile parity par).  x and
    // x / 2 pi are formed in FP64; the fraction of a turn is then a 64-bit
    // integer T (2^64 to the turn), so the argument of every octave is a
    // shift, and one rounding to FP32 remains.
    const uint32_t b_g_ready = mapa_shared(smem_u32(&bars.g_ready), 0);
    auto encode = [&](int u, uint32_t par, uint32_t r) {
        const long long row = ((long long)u * 2 + rank) * 128 + r;
        float4 o = make_float4(0.f, 0.f, 0.f, 0.f), d = o, dl = o;
        float zz = 0.f;
        if (row < M) {
            const long long ray = M <= 0xffffffffll ? (long long)((uint32_t)row / (uint32_t)p.S) : row / p.S;
            const float4* R = reinterpret_cast<const float4*>(p.rays + ray);
            o = R[0]; d = R[1]; dl = R[2];
            zz = p.z[row];
        }
        const float big = fmaxf(fmaxf(fabsf(fmaf(zz, d.x, o.x)), fabsf(fmaf(zz, d.y, o.y))),
                                fmaxf(fabsf(fmaf(zz, d.z, o.z)), 1.0f));
        const uint32_t E = __float_as_uint(big) >> 23;                // >= 127
        const float sc = __uint_as_float((267u - E) << 23);           // 2^(13 - e)
        sm.ex_g[par][r] = (uint8_t)(E - 13u);
        unsigned long long T[3];
        float nf[3], v[6], carry;
        auto turns = [&](int c, float oc, float dc, float lc) {
            const double x = (double)oc + (double)zz * ((double)dc + (double)lc);
            const double t = x * 0.15915494309189533576888376337251;
            if (fabs(t) < 1024.0) T[c] = (unsigned long long)__double2ll_rn(t * 0x1p53) << 11;
            else T[c] = (unsigned long long)__double2ll_rn((t - rint(t)) * 0x1p63) << 1;
            // a non-finite x gives NaN for every octave
            nf[c] = isfinite(x) ? 0.f : __int_as_float(0x7fc00000);
            v[c] = (float)x;
        };
        turns(0, o.x, d.x, dl.x);
        turns(1, o.y, d.y, dl.y);
        turns(2, o.z, d.z, dl.z);
        auto put2 = [&](int col, float a, float b) {   // columns col (even), col + 1
            uint32_t h, lo;
            split2(make_float2(a * sc, b * sc), h, lo);
            const uint32_t ad = sw128_offset(r, col >> 3) + (col & 7) * 2;
            asm volatile("st.shared.b32 [%0], %1;" ::"r"(s_gh + ad), "r"(h) : "memory");
            asm volatile("st.shared.b32 [%0], %1;" ::"r"(s_gl + ad), "r"(lo) : "memory");
        };
        put2(0, v[0], v[1]);
        carry = v[2];
#pragma unroll 1
        for (int k = 0; k < kLxyz; ++k) {
#pragma unroll
            for (int c = 0; c < 3; ++c) {
                const int q = (int)(((T[c] << k) + 0x80000000ull) >> 32);
                sincospif(fmaf((float)q, 0x1p-31f, nf[c]), &v[c], &v[3 + c]);
            }
            put2(2 + 6 * k, carry, v[0]);
            put2(4 + 6 * k, v[1], v[2]);
            put2(6 + 6 * k, v[3], v[4]);
            carry = v[5];
        }
        put2(62, carry, 0.f);
        fence_proxy_async_smem();
        __syncwarp();
        // gamma(x) is the tensor core's (the even CTA's barrier); ex_g is read
        // by this CTA's epilogue threads with ordinary loads, and what they
        // wait for otherwise comes back through the other CTA and the MMAs
        if (lane == 0) {
            mbar_arrive(smem_u32(&bars.ex_ready));
            mbar_arrive_peer(b_g_ready);
        }
    };
    // registers: launched with 168 per thread (3 warpgroups, 504 shares); the
    // epilogue's two warpgroups take 224 each, the first one keeps 56
    if (warp < kEpiWarp0) {
        asm volatile("setmaxnreg.dec.sync.aligned.u32 56;");
        if (warp == 0) {
            // ------------------------------------------------ weight stream (both CTAs)
            if (lane == 0 && !p.hold_weights) {
                uint32_t g = 0;   // blocks: lo and hi of every chunk
                for (int u = u0; u < n_units && ok; u += du) {
                    const uint8_t* src = p.wblocks;
                    for (int b = 0; b < 2 * kChunks; ++b, ++g, src += kBlockBytes) {
                        const uint32_t st = g % kStages;
                        if (!mbar_wait(smem_u32(&bars.empty[st]), ((g / kStages) & 1u) ^ 1u, abort_flag, p.wait_ns)) {
                            ok = false;
                            break;
                        }
                        const uint32_t bytes = b >= 2 * (kChunks - 4) ? kLastBytes : kStageBytes;
                        mbar_arrive_expect_tx(smem_u32(&bars.full[st]), bytes);
                        bulk_load(s_ring + st * kStageBytes, src + rank * bytes, bytes, smem_u32(&bars.full[st]));
                    }
                }
                if (!ok) atomicCAS(p.status_code, 0, MCL_ERR_TIMEOUT);
                // every copy has landed before the CTA may exit
                for (uint32_t k = 0; k < (uint32_t)kStages && k < g; ++k)
                    mbar_wait(smem_u32(&bars.full[(g - 1 - k) % kStages]), ((g - 1 - k) / kStages) & 1u, nullptr);
            }
        } else if (warp == 1 && rank == 1) {
            // ------------------------------------------------ relay (odd CTA)
            if (lane == 0) {
                uint32_t g = 0;
                for (int u = u0; u < n_units && ok; u += du)
                    for (int b = 0; b < 2 * kChunks; ++b, ++g) {
                        const uint32_t st = g % kStages;
                        if (!mbar_wait(smem_u32(&bars.full[st]), (g / kStages) & 1u, abort_flag, p.wait_ns)) {
                            ok = false;
                            break;
                        }
                        mbar_arrive_peer(mapa_shared(smem_u32(&bars.pfull[st]), 0));
                    }
                if (!ok) atomicCAS(p.status_code, 0, MCL_ERR_TIMEOUT);
            }
        } else if (warp == 1) {
            // ------------------------------------------------ MMA issuer (even CTA)
            uint32_t i = 0;
            const uint64_t d_hi = smem_desc(s_hi, 1024, kLayoutSw128), d_lo = smem_desc(s_lo, 1024, kLayoutSw128);
            const uint64_t d_gh = smem_desc(s_gh, 1024, kLayoutSw128), d_gl = smem_desc(s_gl, 1024, kLayoutSw128);
            const uint64_t d_ring = smem_desc(s_ring, 1024, kLayoutSw128);
            constexpr uint32_t kNegA = 1u << 13;   // negate the A operand
            for (int u = u0; u < n_units && ok; u += du) {
                for (int l = 0; l < kLayers && ok; ++l) {
                    const uint32_t id = l == 8 ? idesc_f16(256, 144) : idesc_f16(256, 256);
                    const int nch = chunks_of(l);
                    for (int c = 0; c < nch && ok; ++c, ++i) {
                        const int ac = act_chunk(l, c);
                        const uint64_t ko = (uint64_t)(ac * (int)(kChunkBytes >> 4));
                        const uint64_t ah = ac < 0 ? d_gh : d_hi + ko, al = ac < 0 ? d_gl : d_lo + ko;
                        const uint32_t d = tmem + (i & 1u) * 256u, st = (2 * i) % kStages;
                        const uint64_t wl = d_ring + (uint64_t)(st * (kStageBytes >> 4)), wh = wl + (kStageBytes >> 4);
                        // a chunk's two blocks in one release when both have
                        // landed, so that the MMA queue stays ahead of the
                        // release round trip
                        for (int b = 0; b < 2;) {
                            const int k = (int)named_bar_popc(1, 64, false);
                            if (k < 1 || k > 2 - b) { ok = false; break; }
                            if (lane == 0) {
                                tc_fence_after();
                                // cross terms first (small: little is lost to the
                                // accumulator's truncation), hi hi last
                                if (b == 0) {
    #pragma unroll
                                    for (int e = 0; e < 4; ++e) mma2_bf16(d, ah + 2 * e, wl + 2 * e, id, e ? 1u : 0u);
                                    mma_commit2_mc(smem_u32(&bars.empty[st]), kBoth);
                                }
                                if (b + k == 2) {
    #pragma unroll
                                    for (int e = 0; e < 4; ++e) mma2_bf16(d, al + 2 * e, wh + 2 * e, id | kNegA, 1u);
    #pragma unroll
                                    for (int e = 0; e < 4; ++e) mma2_bf16(d, ah + 2 * e, wh + 2 * e, id, 1u);
                                    mma_commit2_mc(smem_u32(&bars.empty[st + 1]), kBoth);
                                    mma_commit2_mc(smem_u32(&bars.acc_full[i & 1u]), kBoth);
                                    if (l == kSkip && c == 0) mma_commit2_mc(smem_u32(&bars.g_free), kBoth);
                                }
                            }
                            __syncwarp();
                            b += k;
                        }
                    }
                }
            }
            if (lane == 0) {
                if (!ok) atomicCAS(p.status_code, 0, MCL_ERR_TIMEOUT);
                // all issued MMAs complete before either CTA releases TMEM or exits
                mma_commit2_mc(smem_u32(&bars.drain), 1);
                mbar_wait(smem_u32(&bars.drain), 0, nullptr);
            }
            __syncwarp();
        } else if (warp == 2) {
            // ------------------------------------------------ gate (even CTA)
            if (rank == 0) {
                uint32_t i = 0, it = 0;
                auto block = [&](uint32_t g) -> bool {   // block g present in both CTAs
                    const uint32_t st = g % kStages, ph = (g / kStages) & 1u;
                    return mbar_wait(smem_u32(&bars.full[st]), ph, abort_flag, p.wait_ns) &&
                           mbar_wait(smem_u32(&bars.pfull[st]), ph, abort_flag, p.wait_ns);
                };
                for (int u = u0; u < n_units && ok; u += du, ++it) {
                    for (int l = 0; l < kLayers && ok; ++l) {
                        const int nch = chunks_of(l);
                        for (int c = 0; c < nch && ok; ++c, ++i) {
                            const int ac = act_chunk(l, c);
                            // what arrives last in the steady state, last
                            bool good = block(2 * i);
                            if (l == 0) good = good && mbar_wait(smem_u32(&bars.g_ready), it & 1u, abort_flag, p.wait_ns);
                            else if (ac >= 0) good = good && mbar_wait(smem_u32(&bars.a_ready[ac]), (l - 1) & 1u, abort_flag, p.wait_ns);
                            good = good && mbar_wait(smem_u32(&bars.acc_empty[i & 1u]), ((i >> 1) & 1u) ^ 1u, abort_flag, p.wait_ns);
                            const uint32_t st = (2 * i + 1) % kStages, ph = ((2 * i + 1) / kStages) & 1u;
                            const bool both = mbar_try_wait(smem_u32(&bars.full[st]), ph) && mbar_try_wait(smem_u32(&bars.pfull[st]), ph);
                            const int k = !good ? 0 : (__all_sync(0xffffffffu, both) ? 2 : 1);
                            named_bar_popc(1, 64, lane < k);
                            if (!good) { ok = false; break; }
                            if (k == 1) {
                                good = block(2 * i + 1);
                                __syncwarp();
                                named_bar_popc(1, 64, good && lane == 0);
                                if (!good) { ok = false; break; }
                            }
                        }
                    }
                }
                if (!ok && lane == 0) atomicCAS(p.status_code, 0, MCL_ERR_TIMEOUT);
            }
        } else {
            // ------------------------------------------------ gamma(x) of the
            // next unit, once the skip layer's MMAs have read the current one's
            uint32_t it = 0;
            for (int u = u0 + du; u < n_units && ok; u += du, ++it) {
                if (!mbar_wait_sleep(smem_u32(&bars.g_free), it & 1u, abort_flag, p.wait_ns)) { ok = false; break; }
    #pragma unroll 1
                for (int q = 0; q < 4; ++q) encode(u, (it + 1) & 1u, 32 * q + lane);
            }
            if (!ok && lane == 0) atomicCAS(p.status_code, 0, MCL_ERR_TIMEOUT);
        }
    } else {
        asm volatile("setmaxnreg.inc.sync.aligned.u32 224;");
        // ------------------------------------------------ epilogue
        const int quad = warp & 3, j = (warp - kEpiWarp0) >> 2;
        const uint32_t r = quad * 32 + lane;
        const uint32_t t_quad = tmem + ((uint32_t)(quad * 32) << 16);
        // barriers of the even CTA
        const uint32_t b_acc_empty = mapa_shared(smem_u32(&bars.acc_empty[0]), 0);
        const uint32_t b_a_ready = mapa_shared(smem_u32(&bars.a_ready[0]), 0);
        uint32_t i = 0, it = 0;
        float2 s[64];   // sums of the thread's 128 columns (32 of each 64)

        auto acquire = [&]() -> bool {
            const bool g = mbar_wait(smem_u32(&bars.acc_full[i & 1u]), (i >> 1) & 1u, abort_flag, p.wait_ns);
            tc_fence_after();
            return g;
        };
        auto release = [&]() {
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive_peer(b_acc_empty + (i & 1u) * 8u);
            ++i;
        };
        // Add 32 columns of the accumulator, rescaled, to the sums.
        auto add32 = [&](const uint32_t (&v)[32], float2 inv2, int q) {
#pragma unroll
            for (int e = 0; e < 16; ++e)
                s[16 * q + e] = __ffma2_rn(make_float2(__uint_as_float(v[2 * e]), __uint_as_float(v[2 * e + 1])), inv2, s[16 * q + e]);
        };
        // the sums of chunk c start from the bias (loaded ahead, as soon as the
        // registers are free)
        auto start = [&](int l, int c) {
            const float4* bias = reinterpret_cast<const float4*>(p.bias + l * 256 + c * 64 + j * 32);
#pragma unroll
            for (int e = 0; e < 8; ++e) {
                const float4 b = __ldg(bias + e);
                s[16 * c + 2 * e] = make_float2(b.x, b.y);
                s[16 * c + 2 * e + 1] = make_float2(b.z, b.w);
            }
        };
        if (u0 < n_units && j == 0) encode(u0, 0, r);
        for (int u = u0; u < n_units && ok; u += du, ++it) {
            // (written over for unit it + 2 only after the skip layer's MMAs of
            // unit it + 1, whose operands every warp here has stored after its
            // last use of unit it's)
            if (!mbar_wait(smem_u32(&bars.ex_ready), it & 1u, abort_flag, p.wait_ns)) { ok = false; break; }
            for (int l = 0; l < 8 && ok; ++l) {
                const int nch = chunks_of(l);
#pragma unroll
                for (int c = 0; c < 4; ++c) start(l, c);
                float m = 0.f, m1 = 0.f;
                for (int c = 0; c < nch; ++c) {
                    if (!acquire()) { ok = false; break; }
                    const uint32_t e = act_chunk(l, c) < 0 ? sm.ex_g[it & 1u][r] : sm.ex_h[(l - 1) & 1][r];
                    const float inv = __uint_as_float(e << 23) * p.cs[l];
                    const float2 inv2 = make_float2(inv, inv);
                    const uint32_t t = t_quad + (i & 1u) * 256u + j * 32u;
                    uint32_t va[32], vb[32];
                    tmem_ld32(t, va);
                    tmem_ld32(t + 64, vb);
                    tmem_ld_wait();
                    add32(va, inv2, 0);
                    tmem_ld32(t + 128, va);
                    add32(vb, inv2, 1);
                    tmem_ld32(t + 192, vb);
                    if (c == nch - 1) {
#pragma unroll
                        for (int e2 = 0; e2 < 32; ++e2) m = max3(m, s[e2].x, s[e2].y);
                    }
                    tmem_ld_wait();
                    release();
                    add32(va, inv2, 2);
                    add32(vb, inv2, 3);
                }
                if (!ok) break;
                // the row's scale: its largest output, met with the thread
                // that holds the row's other columns
#pragma unroll
                for (int e = 32; e < 64; e += 2) {
                    m = max3(m, s[e].x, s[e].y);
                    m1 = max3(m1, s[e + 1].x, s[e + 1].y);
                }
                m = fmaxf(m, m1);
                sm.ex_m[j][r] = (uint8_t)(__float_as_uint(m) >> 23);
                __syncwarp();
                if (lane == 0) mbar_arrive(smem_u32(&bars.pair[quad]));
                if (!mbar_wait(smem_u32(&bars.pair[quad]), l & 1u, abort_flag, p.wait_ns)) { ok = false; break; }
                const uint32_t E = max(max((uint32_t)sm.ex_m[0][r], (uint32_t)sm.ex_m[1][r]), 27u);
                const float sc = __uint_as_float((268u - E) << 23);   // 2^(14 - e)
                const float2 sc2 = make_float2(sc, sc);
                sm.ex_h[l & 1][r] = (uint8_t)(E - 14u);
                // ReLU, scale, hi and lo into the next layer's operand, chunk
                // by chunk (this layer's MMAs have completed)
#pragma unroll
                for (int c = 0; c < 4; ++c) {
#pragma unroll
                    for (int q = 0; q < 4; ++q) {
                        uint32_t hi[4], lo[4];
#pragma unroll
                        for (int e = 0; e < 4; ++e) {
                            float2 t = __fmul2_rn(s[16 * c + 4 * q + e], sc2);
                            t.x = fmaxf(t.x, 0.f);
                            t.y = fmaxf(t.y, 0.f);
                            split2(t, hi[e], lo[e]);
                        }
                        const uint32_t a = c * kChunkBytes + sw128_offset(r, 4 * j + q);
                        st_shared_v4(s_hi + a, hi[0], hi[1], hi[2], hi[3]);
                        st_shared_v4(s_lo + a, lo[0], lo[1], lo[2], lo[3]);
                    }
                    fence_proxy_async_smem();
                    __syncwarp();
                    if (lane == 0) mbar_arrive_peer(b_a_ready + c * 8u);
                }
            }
            if (!ok) break;
            // last layer: columns 0 .. 127 the RGB hidden layer (64 per
            // thread, column 64 j on; its ray's bias is loaded ahead), column
            // 128 the density (thread j = 1)
            const long long row = ((long long)u * 2 + rank) * 128 + r;
            const bool valid = row < M;
            const long long ray = !valid ? 0 : M <= 0xffffffffll ? (long long)((uint32_t)row / (uint32_t)p.S) : row / p.S;
            const float4* rb4 = ray_bias_at(p.ray_bias, ray) + j * 16 * p.ray_bias.step;
#pragma unroll
            for (int q = 0; q < 16; ++q) {
                const float4 b = __ldg(rb4 + q * p.ray_bias.step);
                s[2 * q] = make_float2(b.x, b.y);
                s[2 * q + 1] = make_float2(b.z, b.w);
            }
            float sig = p.b_sigma;
            for (int c = 0; c < 4; ++c) {
                if (!acquire()) { ok = false; break; }
                const float inv = __uint_as_float((uint32_t)sm.ex_h[1][r] << 23) * p.cs[8];
                const float2 inv2 = make_float2(inv, inv);
                const uint32_t t = t_quad + (i & 1u) * 256u;
                uint32_t va[32], vb[32], w = 0;
                tmem_ld32(t + j * 64, va);
                tmem_ld32(t + j * 64 + 32, vb);
                if (j) tmem_ld1(t + 128, w);
                tmem_ld_wait();
                release();
                add32(va, inv2, 0);
                add32(vb, inv2, 1);
                sig = fmaf(__uint_as_float(w), inv, sig);
            }
            if (!ok) break;
            float2 o2[3] = {};
#pragma unroll
            for (int e = 0; e < 16; ++e) {
                const float2 ha = make_float2(fmaxf(s[2 * e].x, 0.f), fmaxf(s[2 * e].y, 0.f));
                const float2 hb = make_float2(fmaxf(s[2 * e + 1].x, 0.f), fmaxf(s[2 * e + 1].y, 0.f));
#pragma unroll
                for (int c = 0; c < 3; ++c) {
                    const float4 w = *reinterpret_cast<const float4*>(&sm.w_out[c][j * 64 + 4 * e]);
                    o2[c] = __ffma2_rn(hb, make_float2(w.z, w.w), __ffma2_rn(ha, make_float2(w.x, w.y), o2[c]));
                }
            }
            const float o[3] = {o2[0].x + o2[0].y, o2[1].x + o2[1].y, o2[2].x + o2[2].y};
            // the two partial sums meet in the row's 128 bytes of chunk 0 (the
            // row's threads write there again only after they have met at
            // the next unit's first scale)
            float4* scr = reinterpret_cast<float4*>(smem + r * 128);
            const uint32_t hb = smem_u32(&bars.head[quad]);
            if (j) {
                *scr = make_float4(o[0], o[1], o[2], sig);
                mbar_arrive(hb);
            } else {
                if (!mbar_wait(hb, it & 1u, abort_flag, p.wait_ns)) { ok = false; break; }
                const float4 v = *scr;
                if (valid) {
                    float4 res;
                    res.x = v.w;
                    res.y = 1.0f / (1.0f + expf(-(o[0] + v.x + p.b_out[0])));
                    res.z = 1.0f / (1.0f + expf(-(o[1] + v.y + p.b_out[1])));
                    res.w = 1.0f / (1.0f + expf(-(o[2] + v.z + p.b_out[2])));
                    p.out[row] = res;
                }
            }
        }
        if (!ok) atomicCAS(p.status_code, 0, MCL_ERR_TIMEOUT);
    }
    __syncwarp();
    tc_fence_before();
    cluster_sync_all();
    if (warp == 1) {
        tc_fence_after();
        tmem_dealloc2(tmem, 512);
    }
}

struct SplitState {
    uint8_t* wblocks = nullptr;
    float* bias = nullptr;
    int* abort_flag = nullptr;
    bool dense = false;          // false: the map runs on the SIMT kernels
    int n_sm = 0, max_pairs = 0;
    SplitParams base;            // weights' constants of every launch
};

// Whether the FP16 pairs are as exact as FP32 for the map.  A pair keeps 22 to
// 23 bits of an operand, which costs a row's sum about 0.6 units of FP32's last
// place however many terms it has.  A chain of FMAs rounds once per term, by 0.3
// units of the sum so far: sqrt(R) times that in all, where R is the sum over the
// terms of (partial sum / sum)^2, for weights of random sign the partial sums of
// w^2.  n equal terms make R = n / 2; a row that copies an input, R = 1 and no
// error at all.  So EVERY row that is not zero has to have an R above the line
// (a mean over a layer would let rows of copies hide among dense ones).
// Measured, density error (rms) of the pairs over that of the chain, all layers
// with k weights of 256 per row (R = k / 2): k = 16 2.7 to 4.3, 33 1.5 to 3.1,
// 64 1.1 to 1.8, 96 0.9 to 1.5, 128 0.7 to 1.3, 256 (He-normal) 0.5 to 0.8; one
// such layer among dense ones is 0.5 from k = 16 on.  The first layer's inputs
// are none of them zero: 16 weights of 63 1.5, 24 0.55.  Dense maps have R of 18
// at least in the first layer and above 100 in the others.  (Maps fitted to a
// scene are dense in this sense: density 1.2 to 1.4 in the mean and 0.7 to 0.8 in
// the largest error, colours 0.4; a hand-set map of copies 70.)
// A row below 2^-14 of its layer's largest weight would also lose bits to the
// layer's common scale.
bool pairs_are_exact(const std::function<double(int, int, int)>& W) {
    for (int l = 0; l < kLayers; ++l) {
        const int rows = l == 8 ? kRgbW + 1 : kWidth, K = l == 0 ? 64 : (l == kSkip ? 320 : 256);
        const double line = l == 0 ? 12.0 : 48.0;
        double layer_max = 0.0, row_min = INFINITY;
        for (int n = 0; n < rows; ++n) {
            double s2 = 0.0, r = 0.0, mx = 0.0;
            for (int k = 0; k < K; ++k) {   // in the chain's order
                const double w = fabs(W(l, n, k));
                if (!(w > 0.0)) continue;
                s2 += w * w;
                r += s2;
                mx = std::max(mx, w);
            }
            if (!(s2 > 0.0)) continue;
            if (r < line * s2) return false;
            layer_max = std::max(layer_max, mx);
            row_min = std::min(row_min, mx);
        }
        if (row_min < layer_max * 0x1p-14) return false;
    }
    return true;
}

// FP16 bits of the two halves of v (FP64, already scaled).
inline void split_host(double v, uint16_t& hi, uint16_t& lo) {
    const __half h = __float2half_rn((float)v);
    hi = __half_as_ushort(h);
    lo = __half_as_ushort(__float2half_rn((float)(v - (double)__half2float(h))));
}

}  // namespace

// Weight blocks in consumption order (per chunk of 64 products: lo of its two
// 32-column halves, then hi), stored as the 64-byte swizzle lays them out.
// W(l, n, k): weight of layer l (0..8; 8: RGB hidden folded, row 128 the
// density), output n, input k in [h, gamma(x)] order, 0 in the padding.
int mlp_split_prepare(mcl_map* m, const std::function<double(int, int, int)>& W, const float* const* bias,
                      const float* w_out, const float* b_out) {
    SplitState* st = new SplitState();
    m->split = st;
    SplitParams& b = st->base;
    memset(&b, 0, sizeof(b));
    st->dense = pairs_are_exact(W);
    if (!st->dense) return MCL_OK;
    std::vector<uint8_t> blk((size_t)kChunks * 2 * kBlockBytes, 0);
    std::vector<uint16_t> hi(320), lo(320);
    std::vector<float> bias_host(8 * 256 + 3 * kRgbW);
    size_t b0 = 0;   // first block of the layer
    for (int l = 0; l < kLayers; ++l) {
        const int rows = l == 8 ? kRgbW + 1 : kWidth, K = l == 0 ? 64 : (l == kSkip ? 320 : 256);
        double mx = 0.0;
        for (int n = 0; n < rows; ++n)
            for (int k = 0; k < K; ++k) mx = std::max(mx, fabs(W(l, n, k)));
        int e = 0;   // mx = f 2^e, f in [1/2, 1)
        if (mx > 0.0) frexp(mx, &e);
        const double sc = ldexp(1.0, 15 - e);
        b.cs[l] = (float)(kUnbias / sc);
        for (int n = 0; n < rows; ++n) {
            if (l < 8) bias_host[l * 256 + n] = bias[l][n];
            for (int k = 0; k < K; ++k) split_host(W(l, n, k) * sc, hi[k], lo[k]);
            // each CTA holds half of the N rows of a block
            const uint32_t half = l == 8 ? 72 : 128, cr = n / half, row = n % half;
            uint8_t* dst = blk.data() + b0 * kBlockBytes + cr * (l == 8 ? kLastBytes : kStageBytes);
            for (int b = 0; b < 2 * chunks_of(l); ++b, dst += kBlockBytes) {
                const int ac = act_chunk(l, b / 2), k0 = l == 0 ? 0 : ac < 0 ? kWidth : 64 * ac;
                const uint16_t* src = (b & 1 ? hi.data() : lo.data()) + k0;
                for (int k = 0; k < 64; ++k) {
                    const uint32_t byte = row * 128u + 2u * k;
                    memcpy(dst + (byte ^ (((byte >> 7) & 7u) << 4)), &src[k], 2);
                }
            }
        }
        b0 += K / 64 * 2;
    }
    for (int c = 0; c < 3; ++c) {
        for (int n = 0; n < kRgbW; ++n) bias_host[8 * 256 + c * kRgbW + n] = w_out[(size_t)c * kRgbW + n];
        b.b_out[c] = b_out[c];
    }
    b.b_sigma = bias[8][0];
    int rc, dev = 0;
    if ((rc = cuda_check(cudaMalloc(&st->wblocks, blk.size()), "cudaMalloc(split weights)")) ||
        (rc = cuda_check(cudaMemcpy(st->wblocks, blk.data(), blk.size(), cudaMemcpyHostToDevice), "upload split weights")) ||
        (rc = cuda_check(cudaMalloc(&st->bias, bias_host.size() * 4), "cudaMalloc(split biases)")) ||
        (rc = cuda_check(cudaMemcpy(st->bias, bias_host.data(), bias_host.size() * 4, cudaMemcpyHostToDevice), "upload split biases")) ||
        (rc = cuda_check(cudaMalloc(&st->abort_flag, sizeof(int)), "abort flag")) ||
        (rc = cuda_check(cudaFuncSetAttribute(&k_mlp_split, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSmem), "smem attribute")))
        return rc;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&st->n_sm, cudaDevAttrMultiProcessorCount, dev);
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3((unsigned)(st->n_sm & ~1));
    cfg.blockDim = dim3(kThreads);
    cfg.dynamicSmemBytes = kSmem;
    if ((rc = cuda_check(cudaOccupancyMaxActiveClusters(&st->max_pairs, &k_mlp_split, &cfg), "pair occupancy"))) return rc;
    st->max_pairs = std::min(st->max_pairs, st->n_sm / 2);
    if (st->max_pairs < 1) return fail(MCL_ERR_UNSUPPORTED, "no CTA pair fits on an SM pair");
    return MCL_OK;
}

void mlp_split_free(mcl_map* m) {
    SplitState* st = (SplitState*)m->split;
    if (!st) return;
    if (st->wblocks) cudaFree(st->wblocks);
    if (st->bias) cudaFree(st->bias);
    if (st->abort_flag) cudaFree(st->abort_flag);
    delete st;
    m->split = nullptr;
}

// (no state: a device without the tensor-core forms, see mlp_tc_prepare)
bool mlp_fp32_on_pairs(const mcl_map* m) {
    const SplitState* st = (const SplitState*)m->split;
    return st && st->dense;
}

cudaError_t mlp_fp32(mcl_map* m, const Ray* rays, const float* z, int S, int n_rays, float4* out,
                     cudaStream_t s, const int* rows_dev, bool chain_density) {
    SplitState* st = (SplitState*)m->split;
    if (!mlp_fp32_on_pairs(m)) return mlp_fp32_simt(m, rays, z, S, n_rays, out, s, rows_dev, false);
    SplitParams p = st->base;
    p.wblocks = st->wblocks;
    p.bias = st->bias;
    p.rays = rays;
    p.z = z;
    p.S = S;
    p.M = (long long)n_rays * S;
    p.M_dev = rows_dev;
    p.ray_bias = mlp_tc_ray_bias_result(m);
    p.out = out;
    p.abort_flag = st->abort_flag;
    p.status_code = &m->status->code;
    p.wait_ns = kWaitNs;
    p.hold_weights = mlp_tc_take_hold(m, &p.wait_ns);
    cudaError_t e = cudaMemsetAsync(st->abort_flag, 0, sizeof(int), s);
    if (e) return e;
    const long long units = (p.M + 255) / 256;
    note_launch();
    k_mlp_split<<<(unsigned)(2 * std::min<long long>(units, st->max_pairs)), kThreads, kSmem, s>>>(p);
    if ((e = cudaGetLastError()) || !chain_density) return e;
    // A pass that importance samples are drawn from keeps the densities of
    // the FMA chain.  The inverse CDF divides its rounding (6e-8) by the
    // probability of the bin (1e-5 at least), so a density rounded otherwise,
    // even if closer to the exact one, moves samples of nearly empty bins by
    // up to 1e-3 of a bin, and with them the colour of a ray in some 100,000, by
    // up to 4e-3.  With these densities the samples stay where they were.
    return mlp_fp32_simt(m, rays, z, S, n_rays, out, s, rows_dev, true);
}

}  // namespace mcl

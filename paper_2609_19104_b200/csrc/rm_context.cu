// Context Cache: visual-token selective recomputation of a VLM FFN (Sec. 4.1 "Visual-Token Recomputation").
//   Eq. 2   drift score d_p = RMS(x_p - xref_p) / max(RMS(x_p), 1e-6) per visual row
//   Eq. 3   y_hat_p = F(x_p) for the selected rows (and the rows that are always recomputed), else the reference output
// F is the dense gated FFN, F(x) = Wd (gelu_tanh(Wg x) * (Wu x)).  With a few hundred rows against 100 M weights this
// is a pair of dense contractions at the ridge of the roofline, so it runs on the tensor cores with every operand
// block arriving as one cp.async.bulk.tensor box:
//   gather  : Xc[r,:] = x[rows[r],:]                                   (R_pad rows, zero beyond the list)
//   phase A : H1[r, n] = bf16(gelu_tanh(<Xc_r, Wg_n>) * <Xc_r, Wu_n>)  one CTA per <= 128 neurons, K = H
//   phase B : yp[s, r, c] = sum over the s-th slice of n of H1[r, n] Wd[c, n]           one CTA per (128 columns, K slice)
//   sum     : y_out[rows[r], c] = sum over s of yp[s, r, c], in the order of s: the same bits every time
// (phase A's idle warps copy the kept reference rows)
// Both products are D[256 x N] (+)= A[256 x 64] B[N x 64]^T per stage, by pairs of CTAs (cta_group::2): A = weight rows (K
// contiguous, as the model stores them), 128 per CTA; B = activation rows, half of them in each CTA; fp32 accumulators in tensor
// memory (phase A holds two, gate and up: all 512 columns at N = 256).  What bounds a product is what an SM can take in, ~30
// bytes per clock: a pair halves the activations each CTA loads (48 instead of 64 KB a stage in phase A, 32 instead of 48 in
// phase B).  Activation rows are padded to a multiple of 32; a CTA of phase A has as many neurons as spread
// them over all SMs (112 instead of 128 at H = 2048, I = 16384); phase B's K slices are stored by the copy engine and summed by
// a kernel of its own.
//
// Drift, selection and recomputation of 240 of 816 rows at H = 2048, I = 16384, calls back to back (the power limit holds the clock
// at ~1.67 GHz): 75.5 us, of which the sums' kernel is 4.5 (adding the slices to the output in the order of arrival by the copy
// engine: 71.0, but no two runs agree); single CTAs instead of pairs +7, products not on all SMs +2.  In time, at 1.97 GHz: drift
// 4 - 6, selection 6, gather 3, phase A 22 and its epilogue 4 (two MUFU operations per value), 3 to the next kernel, phase B 10.
// The products take in 30 bytes per clock and SM and run at the rate of HBM, so that fetching further weights into L2 ahead of
// time (while phase A waits for its rows, or for phase B) does not help (0.4 - 2 us slower).  Both phases in one kernel would save
// the 3 us between them, but its CTAs would wait on one another, and a call has to run beside whatever else is on the device.
#include <cuda.h>

#include <mutex>

#include "rm_common.cuh"
#include "rm_sm100.cuh"

using namespace sm100;

namespace {

constexpr int EPI = 256, CT = EPI + 64;  // threads: epilogue warps 0-7, loader warp 8 (one lane), issuer warp 9 (one lane)

constexpr int ROW_CHUNK = 8;           // 16-byte loads of a row that a lane has in flight (drift, gather: latency is all they cost)

// ---------------------------------------------------------------- Eq. 2: one warp per row
__global__ void __launch_bounds__(256) drift_kernel(const __nv_bfloat16* __restrict__ x, const __nv_bfloat16* __restrict__ xr,
                                                    int P, int H, float* __restrict__ score) {
    pdl_launch_dependents();               // the selection kernel behind this one may set up
    pdl_wait();
    const int p = blockIdx.x * 8 + (threadIdx.x >> 5), lane = threadIdx.x & 31;
    if (p >= P) return;
    const uint4* a = reinterpret_cast<const uint4*>(x + (size_t)p * H);
    const uint4* b = reinterpret_cast<const uint4*>(xr + (size_t)p * H);
    float sd = 0.f, sx = 0.f;
    for (int e0 = lane; e0 < H / 8; e0 += 32 * ROW_CHUNK) {
        uint4 ua[ROW_CHUNK], ub[ROW_CHUNK];
#pragma unroll
        for (int c = 0; c < ROW_CHUNK; ++c) {
            const int e = e0 + 32 * c;
            ua[c] = ub[c] = make_uint4(0, 0, 0, 0);
            if (e < H / 8) { ua[c] = a[e]; ub[c] = b[e]; }
        }
#pragma unroll
        for (int c = 0; c < ROW_CHUNK; ++c) {
            const __nv_bfloat162* pa = reinterpret_cast<const __nv_bfloat162*>(&ua[c]);
            const __nv_bfloat162* pb = reinterpret_cast<const __nv_bfloat162*>(&ub[c]);
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const float2 fa = __bfloat1622float2(pa[i]), fb = __bfloat1622float2(pb[i]);
                const float d0 = fa.x - fb.x, d1 = fa.y - fb.y;
                sd = fmaf(d0, d0, sd); sd = fmaf(d1, d1, sd);
                sx = fmaf(fa.x, fa.x, sx); sx = fmaf(fa.y, fa.y, sx);
            }
        }
    }
#pragma unroll
    for (int d = 16; d > 0; d >>= 1) {
        sd += __shfl_xor_sync(0xffffffffu, sd, d);
        sx += __shfl_xor_sync(0xffffffffu, sx, d);
    }
    if (lane == 0) score[p] = sqrtf(sd / (float)H) / fmaxf(sqrtf(sx / (float)H), 1e-6f);
}

// ---------------------------------------------------------------- gather of the rows to recompute
// The rows to recompute form one sequence q = 0, 1, ...: q < count is the visual row rows[q], count <= q < count + S the
// always-recomputed row P + (q - count).  A call holds at most `cap` of them (a longer list is cut and reported); one
// pass of the kernels handles the window q_lo <= q < q_lo + r_pad, compact row r = q - q_lo; rows beyond the sequence
// are zero.
__device__ __forceinline__ int ctx_count(const int32_t* count, int P, int S, int cap, bool* bad) {
    int c = *count;
    *bad = c < 0 || c > P || c + S > cap;
    if (*bad) c = c < 0 ? 0 : (P < cap - S ? P : cap - S);
    return c;
}
__global__ void __launch_bounds__(256) ctx_gather_kernel(const __nv_bfloat16* __restrict__ x, const int32_t* __restrict__ rows,
                                                         const int32_t* __restrict__ count, int P, int S, int H, int r_pad,
                                                         int q_lo, int cap, __nv_bfloat16* __restrict__ xc, int* status) {
    pdl_wait();                            // the row list comes from the kernel in front
    pdl_launch_dependents();               // the first product may start now: its weight loads need nothing from here (and the kernel
                                           // in front, which may have written the weights, is complete)
    const int r = blockIdx.x * 8 + (threadIdx.x >> 5), lane = threadIdx.x & 31;
    if (r >= r_pad) return;
    bool bad;
    const int c = ctx_count(count, P, S, cap, &bad);
    if (bad && r == 0 && lane == 0) rm_set_status(status, RM_ERR_INDEX);
    const int q = q_lo + r;
    int src = -1;
    if (q < c) {
        src = rows[q];
        if (src < 0 || src >= P) { if (lane == 0) rm_set_status(status, RM_ERR_INDEX); src = -1; }
    } else if (q < c + S) {
        src = P + (q - c);
    }
    uint4* d = reinterpret_cast<uint4*>(xc + (size_t)r * H);
    const uint4* s = src >= 0 ? reinterpret_cast<const uint4*>(x + (size_t)src * H) : nullptr;
    for (int e0 = lane; e0 < H / 8; e0 += 32 * ROW_CHUNK) {
        uint4 v[ROW_CHUNK];
#pragma unroll
        for (int c = 0; c < ROW_CHUNK; ++c) v[c] = s && e0 + 32 * c < H / 8 ? s[e0 + 32 * c] : make_uint4(0, 0, 0, 0);
#pragma unroll
        for (int c = 0; c < ROW_CHUNK; ++c)
            if (e0 + 32 * c < H / 8) d[e0 + 32 * c] = v[c];
    }
}

// The output row of recomputed row q of the sequence (-1: none).  A listed row must be a visual row: the gather zeroed another
// and recorded the error; adding to it would spoil the always-recomputed row of the same number.
__device__ __forceinline__ int out_row(const int32_t* rows, int q, int c, int P, int S) {
    if (q < c) {
        const int d = rows[q];
        return d >= 0 && d < P ? d : -1;
    }
    return q < c + S ? P + (q - c) : -1;
}

// Is p in the ascending list?  By a whole warp: lane j looks at the last entry of the j-th of 32 parts, then the lanes share the
// part that can hold p (two dependent loads for up to 1024 entries; a binary search by one lane takes ten).
__device__ __forceinline__ bool listed(const int32_t* list, int c, int p, int lane) {
    const int per = (c + 31) / 32;
    int last = lane * per + per - 1;
    if (last >= c) last = c - 1;
    const unsigned below = __ballot_sync(0xffffffffu, c > 0 && list[last] < p);       // parts wholly below p: the first few
    const int lo = __popc(below) * per;
    bool hit = false;
    for (int e = lo + lane; e < lo + per && e < c; e += 32) hit |= list[e] == p;
    return __any_sync(0xffffffffu, hit);
}

// ---------------------------------------------------------------- the two products
// Phase A: Wg rows and Wu rows of this CTA's neurons over all K = H; epilogue GeLU*u -> bf16 H1.
//   WIDE     up to 128 neurons: one tile of Wg rows, one of Wu rows, an accumulator for each
//   PACKED   up to 64 neurons: Wg rows in the upper half of one tile, Wu rows in the lower one, one accumulator; half the
//            products of WIDE, whose tiles would be half empty (H = 1024, I = 4096, 32 neurons per CTA, 240 rows: the products
//            alone took 8 us of phase A's 11)
// Phase B (DOWN): Wd rows of this CTA's 128 output columns over its K slice; the copy engine stores the fp32 sums (512 bytes per row).
enum { DOWN = 0, WIDE = 1, PACKED = 2 };
template <int MODE>
struct SmemCtx {
    static constexpr bool DUAL = MODE == WIDE;
    static constexpr int A_BYTES = 128 * 128;                      // 128 rows x 64 bf16
    static constexpr int STAGE = (DUAL ? 3 : 2) * A_BYTES;         // the last part: up to 128 activation rows x 64 bf16
    static constexpr int NSTAGE = DUAL ? 4 : 6;
    static constexpr int OFF_BAR = NSTAGE * STAGE;                 // (the epilogue stages its results in the ring)
    static constexpr int TOTAL = OFF_BAR + 256 + 1024;
};

struct CtxGemmArgs {
    int kblocks;                       // 64-wide K blocks of the whole product (phase B: cut evenly over gridDim.y)
    int n;                             // activation rows: a multiple of 32, at most 256
    int rows;                          // weight rows (neurons or output columns)
    int mr;                            // weight rows per CTA: a multiple of 8, at most 128
    int I, H;
    __nv_bfloat16* h1;                 // phase A output [n, I]
    const int32_t* list;               // visual rows to recompute, their number
    const int32_t* count;
    int P, S, q_lo, cap;               // this pass has the rows q_lo <= q < q_lo + n of the sequence
    const float* y_ref;
    float* y_out;
    float* yp;                         // phase B output [K slices, n, H]
    int* status;
};

#define wait_bar(bar, parity) wait_bar_at((bar), (parity), __LINE__)

template <int MODE>
// (at most 96 registers: a CTA of phase A starts beside one of the selection kernel)
__global__ void __launch_bounds__(CT, 2) ctx_gemm_kernel(const CtxGemmArgs a, const __grid_constant__ CUtensorMap tmA0,
                                                         const __grid_constant__ CUtensorMap tmA1,
                                                         const __grid_constant__ CUtensorMap tmB) {
    using S = SmemCtx<MODE>;
    constexpr bool DUAL = S::DUAL, GATED = MODE != DOWN;
    constexpr int NSTAGE = S::NSTAGE, OFF_B = (DUAL ? 2 : 1) * S::A_BYTES, TMEM_COLS = DUAL ? 512 : 256;
    extern __shared__ unsigned char smem_dyn[];
    const uint32_t base = (smem_u32(smem_dyn) + 1023u) & ~1023u;
    unsigned char* gbase = smem_dyn + (base - smem_u32(smem_dyn));
    const uint32_t bar0 = base + S::OFF_BAR;
    auto full = [&](int s) { return bar0 + 8 * s; };               // (rank 0: the boxes of both CTAs have landed)
    auto empty = [&](int s) { return bar0 + 64 + 8 * s; };         // the products reading a stage are complete
    const uint32_t d_full = bar0 + 128, s_tmem = bar0 + 136;
    volatile uint32_t* g_tmem = reinterpret_cast<volatile uint32_t*>(gbase + S::OFF_BAR + 136);
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int rank = (int)cluster_ctarank(), n = a.n;

    if (tid == 0) {
        for (int s = 0; s < NSTAGE; ++s) { mbar_init(full(s), 1); mbar_init(empty(s), 1); }
        mbar_init(d_full, 1);
        fence_mbar_init();
    }
    if (warp == EPI / 32 + 1) tmem_alloc_pair(s_tmem, TMEM_COLS);
    tc_fence_before();
    __syncthreads();
    cluster_sync();                        // the other CTA's barriers and tensor memory are there
    tc_fence_after();
    const uint32_t tmem = *g_tmem;
    pdl_launch_dependents();

    bool gave_up = false;
    auto wait_bar_at = [&](uint32_t bar, uint32_t parity, int line) {
        if (!gave_up && !mbar_wait(bar, parity)) {
            rm_set_status_at(a.status, RM_ERR_TIMEOUT, (line << 12) | (int)(blockIdx.x & 0xfffu));
            gave_up = true;
        }
    };
    // this CTA's block of A rows and its K range
    const int m0 = (int)blockIdx.x * a.mr;
    const int kb0 = GATED ? 0 : a.kblocks * (int)blockIdx.y / (int)gridDim.y;
    const int kbn = (GATED ? a.kblocks : a.kblocks * ((int)blockIdx.y + 1) / (int)gridDim.y) - kb0;

    if (warp == EPI / 32 && lane == 0) {
        // ---- loader: the weights do not depend on the previous kernel, the activations do
        const int half = n / 2;
        const uint32_t bytes = 2u * ((GATED ? 2u : 1u) * (uint32_t)a.mr + (uint32_t)half) * 128u;
        auto weights = [&](int kb, int s) {
            const uint32_t st = base + s * S::STAGE, fb = map_to_rank(full(s), 0);
            if (rank == 0) mbar_arrive_expect_tx(full(s), bytes);
            tma_load_2d_pair(st, &tmA0, (kb0 + kb) * 64, m0, fb);
            if (GATED) tma_load_2d_pair(st + (DUAL ? S::A_BYTES : S::A_BYTES / 2), &tmA1, (kb0 + kb) * 64, m0, fb);
        };
        auto rows = [&](int kb, int s) {
            tma_load_2d_pair(base + s * S::STAGE + OFF_B, &tmB, (kb0 + kb) * 64, rank * half, map_to_rank(full(s), 0));
        };
        const int pre = kbn < NSTAGE ? kbn : NSTAGE;
        for (int kb = 0; kb < pre; ++kb) weights(kb, kb);
        pdl_wait();
        for (int kb = 0; kb < pre; ++kb) rows(kb, kb);
        for (int kb = pre; kb < kbn && !gave_up; ++kb) {
            const int s = kb % NSTAGE;
            wait_bar(empty(s), ((kb / NSTAGE) - 1) & 1);
            if (gave_up) break;
            weights(kb, s);
            rows(kb, s);
        }
    } else if (warp == EPI / 32 + 1 && rank == 0) {
        // ---- issuer: the whole warp runs the loop, one elected lane issues; the next stage's barrier is tested behind the
        // current stage's products
        const uint32_t idesc = idesc_bf16_f32(256, n, false, false);
        const uint64_t desc_k = smem_desc_sw128(0, 16, 1024);
        bool ok = false;
        for (int kb = 0; kb < kbn && !gave_up; ++kb) {
            const int s = kb % NSTAGE;
            const uint32_t st = base + s * S::STAGE;
            if (!ok) wait_bar(full(s), (kb / NSTAGE) & 1);
            gave_up = __any_sync(0xffffffffu, gave_up);
            if (gave_up) break;
            tc_fence_after();
            if (elect_one()) {
#pragma unroll
                for (int ks = 0; ks < 4; ++ks) {
                    const uint64_t bd = desc_k | desc_addr(st + OFF_B + ks * 32);
                    mma_bf16_ss_pair(tmem, desc_k | desc_addr(st + ks * 32), bd, idesc, (kb | ks) != 0);
                    if (DUAL) mma_bf16_ss_pair(tmem + 256, desc_k | desc_addr(st + S::A_BYTES + ks * 32), bd, idesc, (kb | ks) != 0);
                }
                mma_commit_pair(empty(s));
                if (kb == kbn - 1) mma_commit_pair(d_full);
            }
            __syncwarp();
            ok = __all_sync(0xffffffffu, mbar_test_wait(full((kb + 1) % NSTAGE), ((kb + 1) / NSTAGE) & 1));
        }
    } else if (warp < EPI / 32) {
        // ---- epilogue: lane = A row (neuron or output column), registers = 32 activation rows; warps 0-3 and 4-7 take turns
        const int m = tid & 127, group = tid >> 7;
        pdl_wait();
        bool bad;
        const int c = ctx_count(a.count, a.P, a.S, a.cap, &bad);
        int dst = -1;                      // phase B: the output row of the sums that this thread stores (-1: none, they are not wanted)
        if (GATED) {
            // in the first pass the visual rows that are not in the (ascending) list keep their reference output: a warp per row
            const int rows = a.q_lo == 0 && a.y_out != a.y_ref ? a.P : 0;
            for (int i = blockIdx.x + warp * (int)gridDim.x; i < rows; i += (EPI / 32) * (int)gridDim.x) {
                if (listed(a.list, c, i, lane)) continue;
                const float4* from = reinterpret_cast<const float4*>(a.y_ref + (size_t)i * a.H);
                float4* to = reinterpret_cast<float4*>(a.y_out + (size_t)i * a.H);
#pragma unroll 4
                for (int e = lane; e < a.H / 4; e += 32) to[e] = from[e];
            }
        } else if (tid < n) {
            dst = out_row(a.list, a.q_lo + tid, c, a.P, a.S);
        }
        wait_bar(d_full, 0);
        tc_fence_after();
        // the ring is free: every product that reads it, the other CTA's included, is complete
        for (int c0 = group * 32; c0 < n && m0 < a.rows && !gave_up; c0 += 64) {
            float v[32];
            tmem_ld32(tmem + ((uint32_t)((warp & 3) * 32) << 16) + c0, v);
            if constexpr (DUAL) {
                float u[32];
                tmem_ld32(tmem + 256 + ((uint32_t)((warp & 3) * 32) << 16) + c0, u);
                // h for 32 activation rows x this neuron -> staging [row][128 neurons] bf16, then 16-byte stores
                // in stages over 16 values, so that the exponentials and divisions of different rows overlap
                // (a value-by-value chain costs ~140 clocks per value)
                unsigned char* stg = gbase + c0 * 256;
#pragma unroll
                for (int t0 = 0; t0 < 32; t0 += 16) {
                    float e[16];
#pragma unroll
                    for (int t = 0; t < 16; ++t) {
                        const float g = v[t0 + t];
                        e[t] = __expf(-1.5957691216057308f * (g + 0.044715f * g * g * g));
                    }
#pragma unroll
                    for (int t = 0; t < 16; ++t) e[t] = __fdividef(v[t0 + t], 1.0f + e[t]) * u[t0 + t];
#pragma unroll
                    for (int t = 0; t < 16; ++t) reinterpret_cast<__nv_bfloat16*>(stg)[(t0 + t) * 128 + m] = __float2bfloat16_rn(e[t]);
                }
                if (group) named_barrier(2, 128); else named_barrier(1, 128);
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    const int e2 = m + 128 * i;                    // 512 chunks of 16 bytes: row e2 / 16, chunk e2 % 16
                    const int t = e2 >> 4, ch = e2 & 15;
                    if (ch * 8 >= a.mr || m0 + ch * 8 >= a.rows) continue;
                    *reinterpret_cast<uint4*>(a.h1 + (size_t)(c0 + t) * a.I + m0 + ch * 8) = reinterpret_cast<const uint4*>(stg)[e2];
                }
            } else if constexpr (MODE == PACKED) {
                // the gate's lanes compute the first 16 rows, the up product's lanes the others: each hands over its half
                float* xch = reinterpret_cast<float*>(gbase + (c0 >> 5) * 12288);              // [32][64]
                __nv_bfloat16* stg = reinterpret_cast<__nv_bfloat16*>(xch + 32 * 64);          // [32][64]
                const int mine = (warp & 2) * 8, nu = m & 63;
#pragma unroll
                for (int t = 0; t < 16; ++t) xch[((mine ^ 16) + t) * 64 + nu] = mine ? v[t] : v[16 + t];
                if (group) named_barrier(2, 128); else named_barrier(1, 128);
                if (nu < a.mr) {
                    float e[16], g[16], u[16];
#pragma unroll
                    for (int t = 0; t < 16; ++t) {
                        const float other = xch[(mine + t) * 64 + nu];
                        g[t] = mine ? other : v[t];
                        u[t] = mine ? v[16 + t] : other;
                    }
#pragma unroll
                    for (int t = 0; t < 16; ++t) e[t] = __expf(-1.5957691216057308f * (g[t] + 0.044715f * g[t] * g[t] * g[t]));
#pragma unroll
                    for (int t = 0; t < 16; ++t) stg[(mine + t) * 64 + nu] = __float2bfloat16_rn(__fdividef(g[t], 1.0f + e[t]) * u[t]);
                }
                if (group) named_barrier(2, 128); else named_barrier(1, 128);
#pragma unroll
                for (int i = 0; i < 2; ++i) {
                    const int e2 = m + 128 * i;                    // 256 chunks of 16 bytes: row e2 / 8, chunk e2 % 8
                    const int t = e2 >> 3, ch = e2 & 7;
                    if (ch * 8 >= a.mr || m0 + ch * 8 >= a.rows) continue;
                    *reinterpret_cast<uint4*>(a.h1 + (size_t)(c0 + t) * a.I + m0 + ch * 8) = reinterpret_cast<const uint4*>(stg)[e2];
                }
            } else {
                float* out = reinterpret_cast<float*>(gbase) + c0 * 128 + m;       // [row][128 columns]
#pragma unroll
                for (int t = 0; t < 32; ++t) out[t * 128] = v[t];
            }
        }
        tc_fence_before();
        if (!GATED) {
            fence_proxy_async_smem();
            named_barrier(1, EPI);
            if (dst >= 0 && m0 < a.rows && !gave_up) bulk_store(a.yp + ((size_t)blockIdx.y * n + tid) * a.H + m0, base + tid * 512, 512);
            bulk_commit();
            bulk_wait_read_all();
        }
    }
    tc_fence_before();
    if (__syncthreads_or(gave_up)) linger_after_timeout();
    cluster_sync();                        // neither CTA leaves while the other may signal it or read its shared memory
    if (warp == EPI / 32 + 1) tmem_dealloc_pair(tmem, TMEM_COLS);
}

// ---------------------------------------------------------------- output rows: the K slices' sums in their order
constexpr int SUM_CHUNK = 8;           // slices that a thread has in flight
__global__ void __launch_bounds__(256) ctx_sum_kernel(const CtxGemmArgs a, int ksplit) {
    pdl_wait();
    pdl_launch_dependents();
    bool bad;
    const int r = (int)blockIdx.x, c = ctx_count(a.count, a.P, a.S, a.cap, &bad), dst = out_row(a.list, a.q_lo + r, c, a.P, a.S);
    if (dst < 0) return;
    for (int e = (int)threadIdx.x; e < a.H / 4; e += 256) {
        const float4* p = reinterpret_cast<const float4*>(a.yp + (size_t)r * a.H) + e;
        float4 y = make_float4(0.f, 0.f, 0.f, 0.f);
        for (int s0 = 0; s0 < ksplit; s0 += SUM_CHUNK) {
            float4 v[SUM_CHUNK];
#pragma unroll
            for (int i = 0; i < SUM_CHUNK; ++i) v[i] = s0 + i < ksplit ? __ldcg(p + (size_t)(s0 + i) * a.n * (a.H / 4)) : make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
            for (int i = 0; i < SUM_CHUNK; ++i) { y.x += v[i].x; y.y += v[i].y; y.z += v[i].z; y.w += v[i].w; }
        }
        reinterpret_cast<float4*>(a.y_out + (size_t)dst * a.H)[e] = y;
    }
}

typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*, const cuuint64_t*,
                                  const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave, CUtensorMapSwizzle,
                                  CUtensorMapL2promotion, CUtensorMapFloatOOBfill);
EncodeTiledFn encode_fn() {
    static EncodeTiledFn fn = nullptr;
    static std::once_flag once;
    std::call_once(once, [] {
        void* p = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &p, cudaEnableDefault, &q) == cudaSuccess &&
            q == cudaDriverEntryPointSuccess)
            fn = reinterpret_cast<EncodeTiledFn>(p);
    });
    return fn;
}
// bf16 matrix [rows, cols] row-major, boxes of box_rows x 64 columns, 128-byte swizzle
int make_map(CUtensorMap* tm, const void* ptr, uint64_t rows, uint64_t cols, uint32_t box_rows) {
    EncodeTiledFn fn = encode_fn();
    if (!fn) return RM_ERR_UNSUPPORTED;
    cuuint64_t dims[2] = {cols, rows};
    cuuint64_t strides[1] = {cols * sizeof(__nv_bfloat16)};
    cuuint32_t box[2] = {64, box_rows};
    cuuint32_t es[2] = {1, 1};
    const CUresult r = fn(tm, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void*>(ptr), dims, strides, box, es,
                          CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                          CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    return r == CUDA_SUCCESS ? RM_OK : RM_ERR_CUDA;
}

inline size_t align_up(size_t v, size_t a) { return (v + a - 1) / a * a; }

template <int MODE>
int launch_gemm(rm_ctx* ctx, const CtxGemmArgs& a, dim3 grid, const CUtensorMap& t0, const CUtensorMap& t1, const CUtensorMap& tb, cudaStream_t s) {
    using S = SmemCtx<MODE>;
    static rm_smem_configured configured = {};
    const int set = configured.raise(ctx->device, S::TOTAL, [] { return rm_set_smem(ctx_gemm_kernel<MODE>, S::TOTAL); });
    if (set != RM_OK) return set;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = dim3(CT);
    cfg.dynamicSmemBytes = S::TOTAL;
    cfg.stream = s;
    cudaLaunchAttribute at[2];
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = ctx->use_pdl;
    at[1].id = cudaLaunchAttributeClusterDimension;
    at[1].val.clusterDim.x = 2;
    at[1].val.clusterDim.y = 1;
    at[1].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = 2;
    RM_CUDA_TRY(cudaLaunchKernelEx(&cfg, ctx_gemm_kernel<MODE>, a, t0, t1, tb));
    ctx->launches++;
    return RM_OK;
}

// weight maps: one set per call, whatever the number of passes
struct FfnMaps { CUtensorMap g, u, d; };

// Neurons per CTA of the first product: as few as spread them over all SMs (2048/16384: 112 on 148 SMs instead of 128 on 128)
int neurons_per_cta(const rm_ctx* ctx) {
    const int ctas = ctx->sm_count >= 2 ? ctx->sm_count / 2 * 2 : 148;
    const int mr = ((ctx->g.I + ctas - 1) / ctas + 7) / 8 * 8;
    return mr > 128 ? 128 : mr;
}

// `a`: the list and the output
int run_ffn(rm_ctx* ctx, const FfnMaps& w, const __nv_bfloat16* xc, __nv_bfloat16* h1, int n, int ksplit, CtxGemmArgs a, cudaStream_t s) {
    const int H = ctx->g.H, I = ctx->g.I;
    CUtensorMap tx, th;
    int rc;
    if ((rc = make_map(&tx, xc, n, H, n / 2)) != RM_OK) return rc;
    if ((rc = make_map(&th, h1, n, I, n / 2)) != RM_OK) return rc;
    a.n = n; a.I = I; a.H = H; a.h1 = h1; a.status = ctx->d_status;
    a.kblocks = H / 64;
    a.rows = I;
    a.mr = neurons_per_cta(ctx);
    const dim3 grid_a(((I + a.mr - 1) / a.mr + 1) / 2 * 2);
    rc = a.mr <= 64 ? launch_gemm<PACKED>(ctx, a, grid_a, w.g, w.u, tx, s) : launch_gemm<WIDE>(ctx, a, grid_a, w.g, w.u, tx, s);
    if (rc != RM_OK) return rc;
    a.kblocks = I / 64;
    a.rows = H;
    a.mr = 128;
    if ((rc = launch_gemm<DOWN>(ctx, a, dim3((H / 128 + 1) / 2 * 2, ksplit), w.d, w.d, th, s)) != RM_OK) return rc;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = ctx->use_pdl;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(n);
    cfg.blockDim = dim3(256);
    cfg.stream = s;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    RM_CUDA_TRY(cudaLaunchKernelEx(&cfg, ctx_sum_kernel, a, ksplit));
    ctx->launches++;
    return RM_OK;
}

// K slices of the second product: as many as keep about one CTA per SM (at least two K blocks each)
int pick_ksplit(const rm_ctx* ctx) {
    const int cols = (ctx->g.H / 128 + 1) / 2 * 2, kblocks = ctx->g.I / 64;
    int ks = (ctx->sm_count > 0 ? ctx->sm_count : 148) / cols;
    if (ks > kblocks / 2) ks = kblocks / 2;
    return ks < 1 ? 1 : (ks > 32 ? 32 : ks);
}
// A capacity of more than 256 rows takes several passes over the weights, of equal size (multiples of 32)
int pass_rows(int cap) {
    const int passes = (cap + 255) / 256;
    return ((cap + passes - 1) / passes + 31) / 32 * 32;
}

}  // namespace

bool rm_context_supported(const rm_ctx* ctx) { return ctx->g.H % 128 == 0 && ctx->g.I % 128 == 0; }

size_t rm_context_workspace_bytes_impl(const rm_ctx* ctx, int cap) {
    const int r_pad = pass_rows(cap);
    const size_t xc = align_up((size_t)r_pad * ctx->g.H * sizeof(__nv_bfloat16), 1024);
    const size_t h1 = align_up((size_t)r_pad * ctx->g.I * sizeof(__nv_bfloat16), 1024);
    const size_t yp = (size_t)pick_ksplit(ctx) * r_pad * ctx->g.H * sizeof(float);
    return xc + h1 + yp;
}

int rm_launch_context_drift(rm_ctx* ctx, const void* x, const void* x_ref, int P, float* score, cudaStream_t s) {
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = ctx->use_pdl;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((P + 7) / 8);
    cfg.blockDim = dim3(256);
    cfg.stream = s;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    RM_CUDA_TRY(cudaLaunchKernelEx(&cfg, drift_kernel, static_cast<const __nv_bfloat16*>(x), static_cast<const __nv_bfloat16*>(x_ref),
                                   P, ctx->g.H, score));
    ctx->launches++;
    return RM_OK;
}

int rm_launch_context_ffn(rm_ctx* ctx, const void* Wg, const void* Wu, const void* Wd, const void* x, const int32_t* rows,
                          const int32_t* count, int P, int S, int cap, const float* y_ref, float* y_out, void* ws,
                          cudaStream_t s) {
    const int H = ctx->g.H, I = ctx->g.I;
    const int ksplit = pick_ksplit(ctx);
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = ctx->use_pdl;
    const int r_pad = pass_rows(cap);
    if (cap <= 256) cap = r_pad;           // (one pass: whatever it holds)
    FfnMaps maps;
    int rc;
    if ((rc = make_map(&maps.g, Wg, I, H, neurons_per_cta(ctx))) != RM_OK) return rc;
    if ((rc = make_map(&maps.u, Wu, I, H, neurons_per_cta(ctx))) != RM_OK) return rc;
    if ((rc = make_map(&maps.d, Wd, H, I, 128)) != RM_OK) return rc;
    for (int q_lo = 0; q_lo < cap; q_lo += r_pad) {
        char* w = static_cast<char*>(ws);
        __nv_bfloat16* xc = reinterpret_cast<__nv_bfloat16*>(w);
        w += align_up((size_t)r_pad * H * sizeof(__nv_bfloat16), 1024);
        __nv_bfloat16* h1 = reinterpret_cast<__nv_bfloat16*>(w);
        w += align_up((size_t)r_pad * I * sizeof(__nv_bfloat16), 1024);
        {
            cudaLaunchConfig_t cfg = {};
            cfg.gridDim = dim3((r_pad + 7) / 8);
            cfg.blockDim = dim3(256);
            cfg.stream = s;
            cfg.attrs = at;
            cfg.numAttrs = 1;
            RM_CUDA_TRY(cudaLaunchKernelEx(&cfg, ctx_gather_kernel, static_cast<const __nv_bfloat16*>(x), rows, count, P, S, H, r_pad,
                                           q_lo, cap, xc, ctx->d_status));
            ctx->launches++;
        }
        CtxGemmArgs a{};
        a.list = rows;
        a.count = count;
        a.P = P; a.S = S; a.q_lo = q_lo; a.cap = cap;
        a.y_ref = y_ref;
        a.y_out = y_out;
        a.yp = reinterpret_cast<float*>(w);
        if ((rc = run_ffn(ctx, maps, xc, h1, r_pad, ksplit, a, s)) != RM_OK) return rc;
    }
    return RM_OK;
}

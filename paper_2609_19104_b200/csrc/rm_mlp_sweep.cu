// Sweep kernel: ONE launch runs every layer of a dense denoising step of one episode as two sweeps over the layer's weights,
// spread over all SMs (one CTA per SM, all co-resident, no clusters).
//
//   gate/up : CTA p owns the neurons of units [U p / G, U (p+1) / G) (a unit is 16 neurons, at most 8 units a CTA) over the
//             whole width H: D1[128 x 64 tokens] per 4 units in tensor memory, the gate and the up row of a neuron in neighbouring
//             lanes (they meet by shuffle); GeLU-tanh(g) * u, activation record, h as a bf16 pair hi + lo to global memory
//             (4 KB per unit)
//   down    : CTA = (column slice j of 8, K split s): D2[H/8 columns x (hi | lo tokens)] over the units [U s / S, U (s+1) / S), then
//             added to the residual stream with red.global.add
//   between : a CTA waits only for the producers of its own units of h (a flag each); the rows of the next layer are
//             normalised by one CTA per token row once every CTA has added its part, and x is shared by all.
//
// What bounds a dense layer of 2048/16384 is HBM: 201 MB, 31 us at the measured copy rate.  The cluster kernels hold it to 3.5
// TB/s on 120 of the SMs: 16-byte gathers (a dense pass has none to do), and the stream stops at every layer boundary with
// 128 KB per CTA loaded ahead.  Here the weights arrive as tensor-map boxes of 4 or 8 KB into a ring of 160 KB per
// CTA (23 MB over the chip) that a loader warp keeps full across the boundaries: it depends on nothing but ring space.
// us per step, 51 tokens, 18 layers, sweep / before: 2048/16384 750 / 1085, 2048/8000 430 / 618, 1024/4096 254 / 284.  What is left
// over HBM time is the chain between the sweeps (~7 us a layer, of which the ring covers ~4).
//
// Every wait is bounded (rm_grid.cuh).
#include <cuda.h>

#include <mutex>

#include "rm_common.cuh"
#include "rm_grid.cuh"
#include "rm_sm100.cuh"

using namespace sm100;
using namespace grid;

namespace {

constexpr int UN = 16;                 // neurons of a unit
constexpr int MAXU = 8;                // units of a CTA in the gate/up sweep (128 accumulator lanes)
constexpr int NTOK = 64, MAXL = 64;
constexpr int NSL = 8;                 // column slices of the packed layout
constexpr int WSTAGE = 32768, NWS = 5; // weight ring
constexpr int ASTAGE = 16384, NAS = 4; // activation ring: two 64-column blocks of x, or 4 units of h (hi, lo)
constexpr int NTHREADS = 352;          // warps 0-7 epilogue and normalisation, 8 weights, 9 activations, 10 issuer
constexpr int OFF_A = NWS * WSTAGE, OFF_MISC = OFF_A + NAS * ASTAGE;
constexpr int SMEM = OFF_MISC + 2048 + 1024;
static_assert(512 + 2 * MAXU * UN * 4 <= 2048, "the record sums exceed the miscellaneous area");
constexpr int TMEM_COLS = 512, D2_COL = 128;                       // D1 at 0 and 64, D2 from 128 (128 columns per 128-column block)

// control block: [CTRL_LINE] token rows normalised, [2 CTRL_LINE] CTAs that have added their part (both cumulative over the
// layers), then a line of 8 ints per CTA: layers whose h it has written
constexpr int C_X = CTRL_LINE, C_Y = 2 * CTRL_LINE, C_H = 3 * CTRL_LINE;
constexpr size_t CTRL_BYTES = (C_H + 8 * 1024) * sizeof(int);

struct WArgs {
    const float* r_in;                 // [T,H]
    float* r;                          // [T,H]: r_L on exit
    unsigned char* x;                  // [H/64][64 rows x 128 bytes]: shared-memory images of x
    unsigned char* h;                  // [U][hi, lo][16 rows x 128 bytes]
    float* record;                     // [L, I] or NULL
    const float* record_scale;         // [L, I] or NULL
    int* ctrl;
    unsigned long long epoch;
    int* status;
    int L, T, I, U, S;                 // U units, S splits of them in the down sweep (S * 8 CTAs)
    // anchor step of Eq. 4 and output gate (EQ4 instantiation)
    float* y_anchor;                   // [L,T,H] or NULL
    float* h_anchor;                   // [L,I,h_stride]
    int64_t h_stride;
    const float* gate;                 // [L,H] or NULL
};
// Per layer: `gu` a box of 16 neurons x (gate, up) x 64 columns (row 2 i gate, 2 i + 1 up of neuron i), `dn` 64 neurons x 64 columns
struct WMaps { CUtensorMap gu[MAXL], dn[MAXL]; };

// CTA p's units [u0, u1) of the U when they are cut evenly into n parts
__device__ __forceinline__ void cut(int U, int n, int p, int& u0, int& u1) {
    u0 = (int)((unsigned)U * (unsigned)p / (unsigned)n);
    u1 = (int)((unsigned)U * (unsigned)(p + 1) / (unsigned)n);
}

template <int HS, bool EQ4>
__global__ void __launch_bounds__(NTHREADS, 1) sweep_kernel(const __grid_constant__ WArgs a, const __grid_constant__ WMaps maps) {
    constexpr int H = NSL * HS, KB = H / 64, NCB = HS / 64, NMB = HS / 128;
    extern __shared__ unsigned char smem_dyn[];
    const uint32_t base = (smem_u32(smem_dyn) + 1023u) & ~1023u;
    unsigned char* gbase = smem_dyn + (base - smem_u32(smem_dyn));
    const uint32_t bar0 = base + OFF_MISC;
    auto w_full = [&](int s) { return bar0 + 8 * s; };
    auto w_empty = [&](int s) { return bar0 + 64 + 8 * s; };
    auto a_full = [&](int s) { return bar0 + 128 + 8 * s; };
    auto a_empty = [&](int s) { return bar0 + 192 + 8 * s; };
    const uint32_t d1_full = bar0 + 256, d2_full = bar0 + 264, s_tmem = bar0 + 272;
    volatile uint32_t* g_tmem = reinterpret_cast<volatile uint32_t*>(gbase + OFF_MISC + 272);
    volatile int* sAbort = reinterpret_cast<volatile int*>(gbase + OFF_MISC + 276);
    float* sPart = reinterpret_cast<float*>(gbase + OFF_MISC + 288);       // 8 partial sums of a row
    // record sums of the second token half, layers in turn: a CTA without a split and without a row of x has no barrier between the
    // reads of one layer and the writes of the next
    float* sRec = reinterpret_cast<float*>(gbase + OFF_MISC + 512);
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int c = (int)blockIdx.x, G = (int)gridDim.x;
    const int T = a.T, L = a.L, U = a.U;
    int u0, u1;                                                    // this CTA's units of the gate/up sweep
    cut(U, G, c, u0, u1);
    const int nu = u1 - u0;
    const int js = c % NSL, sp = c / NSL;                          // column slice and split of the down sweep
    int k0 = 0, k1 = 0;
    if (sp < a.S) cut(U, a.S, sp, k0, k1);
    const int nk = k1 - k0, nst = (nk + 3) / 4;                    // units, stages (4 units) of the down sweep
    // a gate/up stage holds one 64-column block of 8 units, or two of 4 units when no CTA has more
    const int kps = U <= 4 * G ? 2 : 1, nga = nu > 0 ? KB / kps : 0;       // column blocks per stage, stages of the gate/up sweep
    // Every CTA reads all of x.  Each starts at another column block: with all of them asking for the same block at the same
    // time a block took ~0.5 us (layer of 1024/4096: 7.6 us for 16 blocks)
    const int rot = c % (KB / kps);
    const int n_add = a.S * NSL;                                   // CTAs that add (S <= U: every split has units)

    if (tid == 0) {
        for (int s = 0; s < NWS; ++s) { mbar_init(w_full(s), 1); mbar_init(w_empty(s), 1); }
        for (int s = 0; s < NAS; ++s) { mbar_init(a_full(s), 1); mbar_init(a_empty(s), 1); }
        mbar_init(d1_full, 1); mbar_init(d2_full, 1);
        fence_mbar_init();
        *sAbort = 0;
    }
    if (warp == 10) tmem_alloc(s_tmem, TMEM_COLS);
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = *g_tmem;
    // A dependent launch itself, whatever is in front: the weights may be what that kernel writes, so nothing is read before
    // this wait; and what this kernel lets in may count on everything in front of it being complete
    pdl_wait();
    pdl_launch_dependents();               // (a dependent waits for this grid's end)
    if (c == 0 && warp < 8) {
        for (int e = tid; e < C_H + 8 * G; e += 256)
            if (e >= 2) a.ctrl[e] = 0;
        __threadfence();
        named_barrier(1, 256);
        if (tid == 0) epoch_publish(a.ctrl, a.epoch);
    }

    bool gave_up = false;
    auto wait_at = [&](uint32_t bar, uint32_t parity, int line) {
        if (gave_up || mbar_test_wait(bar, parity)) return;
        gave_up = wait_slow(bar, parity, line, a, sAbort);
    };
#define WAIT(bar, parity) wait_at((bar), (parity), __LINE__)

    if (warp == 8) {
        // ================================================================ weights: nothing to wait for but ring space.  A lane per
        // box.  (Lanes 16-31 asking the boxes of a later stage into L2 meanwhile: 740 -> 1090 us; the copy engine handles a 2 KB box in
        // ~60 clocks, prefetch or not, which is close to what the stream itself needs)
        int ws = 0;
        uint32_t pass = 0;
        for (int l = 0; l < L && !gave_up; ++l)
            for (int s = 0; s < nga + nst && !gave_up; ++s) {
                bool box;
                int x, y, dst;                                     // this lane's box and its place in the stage
                uint32_t bytes;
                if (s < nga) {
                    // lane = (column block of the stage, unit)
                    const int sr = (s + rot) % nga, u = kps == 1 ? lane : lane & 3, kb = kps == 1 ? sr : 2 * sr + (lane >> 2);
                    box = lane < 8 && u < nu;
                    y = (u0 + u) * UN;
                    x = (kb / NCB) * 3 * HS + (kb % NCB) * 64;
                    dst = lane * 4096;
                    bytes = 4096u * kps * nu;
                } else {
                    box = lane < NCB;                              // (the last stage may bring rows that nothing multiplies)
                    y = (k0 + 4 * (s - nga)) * UN;
                    x = js * 3 * HS + 2 * HS + lane * 64;
                    dst = lane * 8192;
                    bytes = 8192u * NCB;
                }
                if (pass > 0) WAIT(w_empty(ws), (pass - 1) & 1);
                gave_up = __any_sync(0xffffffffu, gave_up);
                if (gave_up) break;
                if (lane == 0) mbar_arrive_expect_tx(w_full(ws), bytes);
                __syncwarp();
                if (box) {
                    if (s < nga) tma_load_3d(base + ws * WSTAGE + dst, &maps.gu[l], x, 0, y, w_full(ws));
                    else tma_load_2d(base + ws * WSTAGE + dst, &maps.dn[l], x, y, w_full(ws));
                }
                if (++ws == NWS) { ws = 0; ++pass; }
            }
    } else if (warp == 9) {
        // ================================================================ activations: x blocks once the layer's x is complete, h units
        // once their producers have written them
        int as = 0;
        uint32_t pass = 0;
        auto acquire = [&](uint32_t bytes) {
            if (pass > 0) WAIT(a_empty(as), (pass - 1) & 1);
            gave_up = __any_sync(0xffffffffu, gave_up);
            if (lane == 0 && !gave_up) mbar_arrive_expect_tx(a_full(as), bytes);
            __syncwarp();
        };
        auto advance = [&]() { if (++as == NAS) { as = 0; ++pass; } };
        if (lane == 0) gave_up = epoch_wait(a.ctrl, a.epoch, __LINE__, a, sAbort);
        gave_up = __any_sync(0xffffffffu, gave_up);
        for (int l = 0; l < L && !gave_up; ++l) {
            if (nu > 0) {
                if (lane == 0) gave_up = counter_wait(a.ctrl + C_X, T * (l + 1), __LINE__, a, sAbort);
                gave_up = __any_sync(0xffffffffu, gave_up);
                fence_proxy_async_global();
                for (int kp = 0; kp < KB / 2 && !gave_up; ++kp) {
                    acquire((uint32_t)T * 256u);
                    const int kb = (2 * kp + rot * kps + lane) % KB;
                    if (lane < 2 && !gave_up) bulk_load(base + OFF_A + as * ASTAGE + lane * 8192, a.x + (size_t)kb * 8192, (uint32_t)T * 128u, a_full(as));
                    advance();
                }
            }
            if (nk > 0 && !gave_up) {
                int p0 = (int)((unsigned)k0 * (unsigned)G / (unsigned)U);      // first producer of units from k0 on
                for (int q0, q1; p0 > 0; --p0) { cut(U, G, p0 - 1, q0, q1); if (q1 <= k0) break; }
                for (int p = p0 + lane; p < G; p += 32) {
                    int q0, q1;
                    cut(U, G, p, q0, q1);
                    if (q0 >= k1) break;
                    if (q1 > q0 && q1 > k0 && !gave_up) gave_up = counter_wait(a.ctrl + C_H + 8 * p, l + 1, __LINE__, a, sAbort);
                }
                gave_up = __any_sync(0xffffffffu, gave_up);
                fence_proxy_async_global();
                for (int s = 0; s < nst && !gave_up; ++s) {
                    const int ku = nk - 4 * s < 4 ? nk - 4 * s : 4;
                    acquire((uint32_t)ku * 4096u);
                    const int u = lane >> 1, lo = lane & 1;
                    if (u < ku && !gave_up)
                        bulk_load(base + OFF_A + as * ASTAGE + lo * 8192 + u * 2048, a.h + (size_t)(k0 + 4 * s + u) * 4096 + lo * 2048, 2048u, a_full(as));
                    advance();
                }
            }
        }
    } else if (warp == 10) {
        // ================================================================ issuer: the whole warp runs the loop, one elected lane issues; the
        // next stage's barriers are tested behind the current stage's products
        constexpr uint32_t IDESC_G = idesc_bf16_f32(128, NTOK, false, false), IDESC_D = idesc_bf16_f32(128, 2 * NTOK, true, true);
        const uint64_t desc_k = smem_desc_sw128(0, 16, 1024), desc_mn = smem_desc_sw128(0, 8192, 1024);
        int ws = 0, as = 0;
        uint32_t wph = 0, aph = 0;
        bool w_ok = false, a_ok = false;
        auto w_ready = [&]() { if (!w_ok) WAIT(w_full(ws), wph); };
        auto a_ready = [&]() {
            if (!a_ok) WAIT(a_full(as), aph);
            gave_up = __any_sync(0xffffffffu, gave_up);
            tc_fence_after();
        };
        // (a test takes ~200 clocks to come back: one for both rings, behind the products of the stage in front)
        auto next = [&](bool w, bool x) {
            if (w && ++ws == NWS) { ws = 0; wph ^= 1; }
            if (x && ++as == NAS) { as = 0; aph ^= 1; }
            const uint32_t m = mbar_test_wait_2(w_full(ws), wph, a_full(as), aph);
            if (w) w_ok = __all_sync(0xffffffffu, m & 1u);
            if (x) a_ok = __all_sync(0xffffffffu, (m >> 1) & 1u);
        };
        for (int l = 0; l < L && !gave_up; ++l) {
            for (int kp = 0; kp < KB / 2 && nu > 0 && !gave_up; ++kp) {        // two column blocks: one stage of x, one or two of weights
                a_ready();
                w_ready();
                gave_up = __any_sync(0xffffffffu, gave_up);
                if (gave_up) break;
                const uint32_t xt = base + OFF_A + as * ASTAGE;
                if (kps == 2) {
                    const uint32_t wt = base + ws * WSTAGE;
                    if (elect_one()) {
#pragma unroll
                        for (int k8 = 0; k8 < 8; ++k8) {
                            const int o = (k8 >> 2), ks = k8 & 3;
                            mma_bf16_ss(tmem, desc_k | desc_addr(wt + o * 16384 + ks * 32), desc_k | desc_addr(xt + o * 8192 + ks * 32), IDESC_G, (kp | k8) != 0);
                        }
                        mma_commit(w_empty(ws));
                        mma_commit(a_empty(as));
                        if (kp == KB / 2 - 1) mma_commit(d1_full);
                    }
                    __syncwarp();
                    next(true, true);
                } else {
#pragma unroll 1
                    for (int o = 0; o < 2; ++o) {
                        if (o == 1) {
                            w_ready();
                            gave_up = __any_sync(0xffffffffu, gave_up);
                            if (gave_up) break;
                            tc_fence_after();
                        }
                        const uint32_t wt = base + ws * WSTAGE;
                        if (elect_one()) {
#pragma unroll
                            for (int ks = 0; ks < 4; ++ks) {
                                const uint64_t bx = desc_k | desc_addr(xt + o * 8192 + ks * 32);
                                mma_bf16_ss(tmem, desc_k | desc_addr(wt + ks * 32), bx, IDESC_G, (kp | o | ks) != 0);
                                if (nu > 4) mma_bf16_ss(tmem + NTOK, desc_k | desc_addr(wt + 16384 + ks * 32), bx, IDESC_G, (kp | o | ks) != 0);
                            }
                            mma_commit(w_empty(ws));
                            if (o == 1) mma_commit(a_empty(as));
                            if (o == 1 && kp == KB / 2 - 1) mma_commit(d1_full);
                        }
                        __syncwarp();
                        next(true, o == 1);
                    }
                }
            }
            for (int s = 0; s < nst && !gave_up; ++s) {
                w_ready();
                a_ready();
                if (gave_up) break;
                const int ku = nk - 4 * s < 4 ? nk - 4 * s : 4;
                const uint32_t wt = base + ws * WSTAGE, ht = base + OFF_A + as * ASTAGE;
                if (elect_one()) {
                    for (int ks = 0; ks < ku; ++ks) {
                        const uint64_t bh = desc_mn | desc_addr(ht + ks * 2048);
#pragma unroll
                        for (int mb = 0; mb < NMB; ++mb)
                            mma_bf16_ss(tmem + D2_COL + mb * 2 * NTOK, desc_mn | desc_addr(wt + mb * 16384 + ks * 2048), bh, IDESC_D, (s | ks) != 0);
                    }
                    mma_commit(w_empty(ws));
                    mma_commit(a_empty(as));
                    if (s == nst - 1) mma_commit(d2_full);
                }
                __syncwarp();
                next(true, true);
            }
        }
    } else {
        // ================================================================ epilogue: normalisation, GLU, adds
        const int q4 = warp & 3, ch = warp >> 2;                   // tensor-memory lane quarter; token half (gate/up)
        const uint32_t lane_off = (uint32_t)(q4 * 32) << 16;
        bool stop = false;
        if (tid == 0) gave_up = epoch_wait(a.ctrl, a.epoch, __LINE__, a, sAbort);
        for (int l = 0; l < L && !stop; ++l) {
            // ---- x rows c, c + G, ... of the layer
            if (c < T) {
                if (tid == 0 && l > 0 && !gave_up) gave_up = counter_wait(a.ctrl + C_Y, n_add * l, __LINE__, a, sAbort);
                stop = barrier_or(1, 256, gave_up || *sAbort);
                if (stop) break;
                int rows = 0;
                for (int t = c; t < T; t += G, ++rows) {
                    const float4* src = reinterpret_cast<const float4*>((l == 0 ? a.r_in : a.r) + (size_t)t * H) + tid;
                    float4 v[H / 1024];
                    float ss = 0.f;
#pragma unroll
                    for (int i = 0; i < H / 1024; ++i) v[i] = __ldcg(src + 256 * i);
#pragma unroll
                    for (int i = 0; i < H / 1024; ++i) {
                        ss = fmaf(v[i].x, v[i].x, ss); ss = fmaf(v[i].y, v[i].y, ss);
                        ss = fmaf(v[i].z, v[i].z, ss); ss = fmaf(v[i].w, v[i].w, ss);
                    }
#pragma unroll
                    for (int d = 16; d > 0; d >>= 1) ss += __shfl_xor_sync(0xffffffffu, ss, d);
                    if (rows > 0) named_barrier(1, 256);           // (sPart of the row before has been read)
                    if (lane == 0) sPart[warp] = ss;
                    named_barrier(1, 256);
                    float tot = 0.f;
#pragma unroll
                    for (int w = 0; w < 8; ++w) tot += sPart[w];
                    const float inv = 1.0f / sqrtf(tot / (float)H + 1e-6f);
#pragma unroll
                    for (int i = 0; i < H / 1024; ++i) {
                        const int col = 4 * (tid + 256 * i);
                        const __nv_bfloat162 lo = __floats2bfloat162_rn(v[i].x * inv, v[i].y * inv);
                        const __nv_bfloat162 hi = __floats2bfloat162_rn(v[i].z * inv, v[i].w * inv);
                        uint2 u;
                        u.x = *reinterpret_cast<const uint32_t*>(&lo);
                        u.y = *reinterpret_cast<const uint32_t*>(&hi);
                        *reinterpret_cast<uint2*>(a.x + (size_t)(col >> 6) * 8192 + t * 128 + ((((col & 63) >> 3) ^ (t & 7)) << 4) + (col & 7) * 2) = u;
                        if (EQ4 && a.y_anchor)                     // (the sums start from zero: they are added behind x)
                            reinterpret_cast<float4*>(a.y_anchor + ((size_t)l * T + t) * H)[tid + 256 * i] = make_float4(0.f, 0.f, 0.f, 0.f);
                        if (l == 0 && a.r != a.r_in) reinterpret_cast<float4*>(a.r + (size_t)t * H)[tid + 256 * i] = v[i];
                    }
                }
                fence_proxy_async_global();
                named_barrier(1, 256);
                if (tid == 0) red_release_gpu(a.ctrl + C_X, rows);
            }
            // ---- h of this CTA's neurons
            if (nu > 0) {
                // lanes 2 i, 2 i + 1 of a warp hold the gate and the up row of neuron i of unit q4 (q4 + 4) for the 32 tokens of half
                // ch: the gate lane finishes the first 16 of them, the up lane the last 16
                const bool isup = lane & 1;
                const int nl = lane >> 1, tb = ch * 32 + (isup ? 16 : 0);      // neuron of the unit; first token of this lane
                WAIT(d1_full, l & 1);
                tc_fence_after();
                float rec[2] = {0.f, 0.f};
#pragma unroll
                for (int v = 0; v < 2; ++v) {
                    const int unit = 4 * v + q4;
                    if (unit >= nu) break;
                    float d[32], g[16];
                    tmem_ld32(tmem + v * NTOK + ch * 32 + lane_off, d);
                    // in stages, so that the exponentials and divisions of different tokens overlap
#pragma unroll
                    for (int t = 0; t < 16; ++t) {
                        const float got = __shfl_xor_sync(0xffffffffu, isup ? d[t] : d[16 + t], 1);
                        g[t] = isup ? got : d[t];
                        d[t] = isup ? d[16 + t] : got;             // up
                    }
                    float e[16];
#pragma unroll
                    for (int t = 0; t < 16; ++t) e[t] = __expf(-1.5957691216057308f * (g[t] + 0.044715f * g[t] * g[t] * g[t]));
#pragma unroll
                    for (int t = 0; t < 16; ++t) e[t] = __fdividef(g[t], 1.0f + e[t]);
                    const bool real = (u0 + unit) * UN + nl < a.I;
#pragma unroll
                    for (int t = 0; t < 16; ++t) {
                        e[t] = real && tb + t < T ? e[t] * d[t] : 0.f;
                        rec[v] += fabsf(e[t]);
                    }
                    if (EQ4 && a.h_anchor && real) {
                        float* ha = a.h_anchor + ((size_t)l * a.I + (u0 + unit) * UN + nl) * a.h_stride + tb;
#pragma unroll
                        for (int t = 0; t < 16; t += 4)
                            if (tb + t < T) *reinterpret_cast<float4*>(ha + t) = make_float4(e[t], e[t + 1], e[t + 2], e[t + 3]);
                    }
                    unsigned char* hp = a.h + (size_t)(u0 + unit) * 4096 + nl * 128;
#pragma unroll
                    for (int k = 0; k < 2; ++k) {
                        uint32_t hi[4], lo[4];
#pragma unroll
                        for (int i = 0; i < 4; ++i) {
                            const float f0 = e[8 * k + 2 * i], f1 = e[8 * k + 2 * i + 1];
                            const __nv_bfloat162 h2 = __floats2bfloat162_rn(f0, f1);
                            const float2 hf = __bfloat1622float2(h2);
                            const __nv_bfloat162 l2 = __floats2bfloat162_rn(f0 - hf.x, f1 - hf.y);
                            hi[i] = *reinterpret_cast<const uint32_t*>(&h2);
                            lo[i] = *reinterpret_cast<const uint32_t*>(&l2);
                        }
                        const int off = (((tb >> 3) + k) ^ (nl & 7)) << 4;
                        *reinterpret_cast<uint4*>(hp + off) = make_uint4(hi[0], hi[1], hi[2], hi[3]);
                        *reinterpret_cast<uint4*>(hp + 2048 + off) = make_uint4(lo[0], lo[1], lo[2], lo[3]);
                    }
                    if (a.record) {
                        rec[v] += __shfl_xor_sync(0xffffffffu, rec[v], 1);
                        if (ch == 1 && !isup) sRec[(l & 1) * MAXU * UN + unit * UN + nl] = rec[v];
                    }
                }
                tc_fence_before();
                fence_proxy_async_global();
                stop = barrier_or(1, 256, gave_up || *sAbort);
                if (stop) break;
                if (tid == 0) st_release_gpu(a.ctrl + C_H + 8 * c, l + 1);
                if (a.record && ch == 0 && !isup) {
#pragma unroll
                    for (int v = 0; v < 2; ++v) {
                        const int unit = 4 * v + q4, n = (u0 + unit) * UN + nl;
                        if (unit >= nu || n >= a.I) continue;
                        const float r = rec[v] + sRec[(l & 1) * MAXU * UN + unit * UN + nl];
                        a.record[(size_t)l * a.I + n] = a.record_scale ? r * a.record_scale[(size_t)l * a.I + n] : r;
                    }
                }
            }
            // ---- this CTA's [columns of the slice x tokens] sums of the down sweep
            if (nk > 0) {
                WAIT(d2_full, l & 1);
                tc_fence_after();
                const int mb = NMB == 2 ? ch : 0, t0 = NMB == 2 ? 0 : ch * 32, t1 = NMB == 2 ? NTOK : t0 + 32;
                const size_t col = (size_t)js * HS + mb * 128 + q4 * 32 + lane;
                float* rb = a.r + col;
                float* yb = EQ4 && a.y_anchor ? a.y_anchor + (size_t)l * T * H + col : nullptr;
                const float gt = EQ4 && a.gate ? __ldg(a.gate + (size_t)l * H + col) : 1.f;
                const uint32_t d2 = tmem + D2_COL + mb * 2 * NTOK + lane_off;
                if (!gave_up) {
#pragma unroll 1
                    for (int t = t0; t < t1 && t < T; t += 8) {
                        float hi[8], lo[8];
                        tmem_ld8(d2 + t, hi);
                        tmem_ld8(d2 + NTOK + t, lo);
#pragma unroll
                        for (int i = 0; i < 8; ++i)
                            if (t + i < T) {
                                const float y = hi[i] + lo[i];
                                red_add_f32(rb + (size_t)(t + i) * H, EQ4 ? gt * y : y);
                                if (EQ4 && yb) red_add_f32(yb + (size_t)(t + i) * H, y);
                            }
                    }
                }
                tc_fence_before();
                stop = barrier_or(1, 256, gave_up || *sAbort);
                if (stop) break;
                if (tid == 0) red_release_gpu(a.ctrl + C_Y, 1);
            }
        }
    }
#undef WAIT
    tc_fence_before();
    __syncthreads();
    if (*sAbort) {
        // a wait gave up somewhere: copies into this CTA's shared memory may still be in flight although nobody waits for them
        for (int i = 0; i < 64; ++i) __nanosleep(4000);
        __syncthreads();
    }
    if (warp == 10) tmem_dealloc(tmem, TMEM_COLS);
    if (tid == 0 && !epoch_wait(a.ctrl, a.epoch, __LINE__, a, sAbort)) epoch_leave(a.ctrl);
}

// ---- host side
inline size_t align_up(size_t v, size_t a) { return (v + a - 1) / a * a; }

template <int HS, bool EQ4>
int launch(rm_ctx* ctx, const WArgs& a, const WMaps& maps, int G, cudaStream_t s) {
    static rm_smem_configured configured = {};
    const int set = configured.raise(ctx->device, SMEM, [] { return rm_set_smem(sweep_kernel<HS, EQ4>, SMEM); });
    if (set != RM_OK) return set;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(G);
    cfg.blockDim = dim3(NTHREADS);
    cfg.dynamicSmemBytes = SMEM;
    cfg.stream = s;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = at;
    cfg.numAttrs = ctx->use_pdl ? 1 : 0;
    RM_CUDA_TRY(cudaLaunchKernelEx(&cfg, sweep_kernel<HS, EQ4>, a, maps));
    ctx->launches++;
    return RM_OK;
}
inline int units(int I) { return (I + UN - 1) / UN; }
inline int grid_size(const rm_ctx* ctx) { return ctx->sm_count < 1024 ? ctx->sm_count : 1024; }

}  // namespace

bool rm_sweep_supported(const rm_ctx* ctx, int B, int T) {
    const int H = ctx->g.H, G = grid_size(ctx);
    return (H == 1024 || H == 2048) && ctx->fused_clusters > 0 && B == 1 && T >= 1 && T <= NTOK && ctx->g.L <= MAXL && G >= NSL &&
           units(ctx->g.I) <= MAXU * G;
}

size_t rm_sweep_workspace_bytes(const rm_ctx* ctx) {
    if (!rm_sweep_supported(ctx, 1, 1)) return 0;
    return align_up(CTRL_BYTES, 1024) + (size_t)(ctx->g.H / 64) * 8192 + (size_t)units(ctx->g.I) * 4096;
}

// Dense steps of one episode: no lists, no anchor state or the anchor step of Eq. 4
int rm_launch_step_sweep(rm_ctx* ctx, const rm_step_args& sa, void* ws, cudaStream_t s) {
    const rm_geom& g = ctx->g;
    // The maps are encoded again only for layers whose address has changed.  The context may serve several threads with models of
    // their own: they take turns from here to the launch, which copies the maps.
    std::lock_guard<std::mutex> lock(ctx->sweep_mutex);
    WMaps* maps = reinterpret_cast<WMaps*>(ctx->sweep_maps);
    static_assert(sizeof(WMaps) == sizeof(ctx->sweep_maps), "the context holds the tensor maps");
    for (int l = 0; l < sa.L; ++l) {
        if (ctx->sweep_key[l] == sa.packed_layers[l]) continue;
        ctx->sweep_key[l] = nullptr;
        int rc = rm_make_weight_map(&maps->gu[l], sa.packed_layers[l], g.I, 3 * g.H, UN, g.Hs);
        if (rc == RM_OK) rc = rm_make_weight_map(&maps->dn[l], sa.packed_layers[l], g.I, 3 * g.H, 4 * UN, 0);
        if (rc != RM_OK) return rc;
        ctx->sweep_key[l] = sa.packed_layers[l];
    }
    WArgs a{};
    a.r_in = sa.r_in ? sa.r_in : sa.r;
    a.r = sa.r;
    unsigned char* w = static_cast<unsigned char*>(ws);
    a.ctrl = reinterpret_cast<int*>(w);
    w += align_up(CTRL_BYTES, 1024);
    a.x = w;
    w += (size_t)(g.H / 64) * 8192;
    a.h = w;
    a.record = sa.record;
    a.record_scale = sa.record_scale;
    a.epoch = rm_next_epoch();
    a.status = ctx->d_status;
    a.L = sa.L;
    a.T = sa.T;
    a.I = g.I;
    a.U = units(g.I);
    int G = grid_size(ctx);
    if (ctx->max_clusters_override > 0 && ctx->max_clusters_override * NSL < G && a.U <= MAXU * ctx->max_clusters_override * NSL)
        G = ctx->max_clusters_override * NSL;
    a.S = G / NSL < a.U ? G / NSL : a.U;
    if (sa.anchor_mode == RM_ANCHOR_WRITE) {
        a.y_anchor = sa.y_anchor;
        a.h_anchor = sa.h_anchor;
        a.h_stride = sa.h_stride;
    }
    a.gate = sa.gate;
    const bool eq4 = sa.anchor_mode == RM_ANCHOR_WRITE || sa.gate;
    if (g.H == 1024) return eq4 ? launch<128, true>(ctx, a, *maps, G, s) : launch<128, false>(ctx, a, *maps, G, s);
    return eq4 ? launch<256, true>(ctx, a, *maps, G, s) : launch<256, false>(ctx, a, *maps, G, s);
}

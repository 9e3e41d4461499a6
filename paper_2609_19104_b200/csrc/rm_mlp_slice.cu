// Slice kernel of the masked gated MLP stack: ONE launch runs every layer of a denoising step.
//
// Clusters of 8 CTAs, all co-resident (one CTA per SM).  CTA j of a cluster owns column slice j (Hs = H/8 columns of the
// model width) for BOTH projections, so a neuron's slice -- gate, up and down piece side by side in the packed layout -- is
// read once, by one CTA, as two contiguous bulk copies.  The active list of a layer is cut over the clusters; a cluster
// walks its run in rounds of 8 OPN neurons:
//   gate/up : partial sums over the slice's columns, [16 rows = 8 gate + 8 up] x tokens per warp tile, by mma.sync
//             (m16n8k16, bf16 in, fp32 accumulators in registers)
//   owner   : neuron q of the round belongs to CTA q / OPN.  The partial sums travel to it as bulk copies between the
//             CTAs' shared memories, counted on its mbarrier; it adds the 8 slices' sums, applies gelu_tanh(g) * u, splits h
//             into a bf16 pair hi + lo (relative error 2^-17) and copies its rows to the other CTAs' h tiles
//   down    : [tokens] x [the slice's columns], accumulated in registers over the rounds of the item, then added to the
//             fp32 residual stream with red.global.add
// A layer's adds go into a buffer of their own (three in turn, cleared one layer ahead); the residual itself is added by
// the clusters in equal shares of token rows, from the registers in which the row was normalised.  A CTA waits for the
// layer before only on its own slice: counter (episode, slice) counts the clusters that have added their part.
//
// Why mma.sync and not tcgen05: with at most 64 token rows the products of a step are small (config of 1024/4096, 25 % of the
// neurons: 0.4 us of tensor time per layer and product at the 1024 multiply-adds per clock and SM that mma.sync was
// measured at, 23 clocks of latency), and a layer is a chain of latencies behind a grid-wide dependency.  Operands come
// from rows of any pitch (ldmatrix takes row addresses), so a neuron's piece is one bulk copy instead of 16-byte gathers
// into a swizzled layout; the accumulators are in registers at once, without commit, barrier and tensor-memory read.
//
// Every wait is bounded; a wait that runs out records RM_ERR_TIMEOUT (with its source line), raises the launch's abort
// flag, and every role runs to its end without waiting.  CTAs leave together (cluster barrier at the end).
#include <atomic>
#include <chrono>

#include "rm_common.cuh"
#include "rm_sm100.cuh"

using namespace sm100;

namespace {

constexpr int CS = 8;                  // CTAs per cluster = column slices of the packed layout
constexpr int SN = 16;                 // neurons per weight stage
constexpr int MAX_ITEMS = 512;         // layers x episodes of one launch
constexpr int MAXL = 64, MAXB = 64;
constexpr int NTHREADS = 640;          // warps 0-7: normalisation and gate/up (group A); 8-15: owner, down, adds (group B);
constexpr int W_B = 8, W_G = 16;   // 16 / 17: loaders of the gate/up and of the down pieces
constexpr int HPITCH = 272;            // bytes of an h row: 64 tokens hi, 64 tokens lo, 16 to spread the banks
constexpr int SSB = 4;                 // buffers of the row sums of squares: a CTA can be two items ahead of another
constexpr int MAX_STAGES = 16;

// control block in the workspace, in ints: [0,1] launch epoch, [2] CTAs that have left, [3] abort flag; then lines of 32 ints:
// per (episode, slice) the CTAs that have set up the first output buffer, and the CTAs that have added their part
constexpr int CTRL_LINE = 32;
__host__ __device__ constexpr int ctrl_init(int e, int j) { return CTRL_LINE * (1 + (e * CS + j) * 2); }
__host__ __device__ constexpr int ctrl_done(int e, int j) { return CTRL_LINE * (2 + (e * CS + j) * 2); }
__host__ __device__ constexpr size_t ctrl_bytes(int B) { return (size_t)CTRL_LINE * (1 + 2 * CS * B) * sizeof(int); }

// ---- shared-memory layout (computed by the host, a kernel argument: constants cost no registers)
struct Lay {
    int xp, gp, dp;                    // row pitches: x tile, gate|up pieces, down pieces (odd multiples of 16 bytes: eight rows
                                       // of an ldmatrix fall into different banks)
    int ks, n_a, n_b;                  // 16-column steps of the slice; 8-token tiles of the two token halves
    int p_src, p_buf, stg_warp;        // partial sums: bytes from one source, of one buffer, of one warp's outgoing pieces
    int h_buf, g_stage, d_stage;
    int off_p, off_stg, off_h, off_ss, off_item, off_bar, off_x, off_g, off_d, total;
};
inline Lay make_layout(int Hs, int T, int opn, int stages) {
    Lay y;
    const int t8 = (T + 7) / 8;
    y.ks = (Hs + 15) / 16;
    y.xp = y.ks * 32 + 16;
    y.gp = Hs * 4 + 16;
    y.dp = (Hs / 8) % 2 ? Hs * 2 : Hs * 2 + 16;
    y.n_a = (t8 + 1) / 2;
    y.n_b = t8 - y.n_a;
    y.p_src = opn * t8 * 64;
    y.p_buf = CS * y.p_src;
    y.stg_warp = 2 * 8 * y.n_a * 64;
    y.h_buf = CS * opn * HPITCH;
    y.g_stage = SN * y.gp;
    y.d_stage = SN * y.dp + 32;        // (an odd last pair of column tiles reads 16 bytes past the last row)
    int o = 0;
    y.off_bar = o;   o += 512;
    y.off_item = o;  o += MAX_ITEMS * 16;
    y.off_ss = o;    o += SSB * CS * 64 * 4;
    y.off_x = o;     o += 64 * y.xp;
    y.off_p = o;     o += 2 * y.p_buf;
    y.off_stg = o;   o += 8 * y.stg_warp;
    y.off_h = o;     o += 2 * y.h_buf;
    y.off_g = o;     o += stages * y.g_stage;
    y.off_d = o;     o += stages * y.d_stage;
    y.total = o + 128;
    return y;
}

struct SArgs {
    const __nv_bfloat16* packed[MAXL];
    const float* r_in;                 // [B,T,H] r_0
    float* r_out;                      // [B,T,H] r_L
    float* rot[3];                     // [B,T,H] outputs of the layers in between, in turn
    const __nv_bfloat16* x_ext;        // [T,H]: the only layer takes this as its input (no normalisation), or NULL
    const int32_t* idx;                // list (b, l) at idx + b * idx_b_stride + l * idx_l_stride; NULL: positions
    const int32_t* count;              // count (b, l) at count[b * count_b_stride + l]; NULL: every neuron
    int64_t idx_b_stride, idx_l_stride, list_cap, count_b_stride;
    float* record;                     // record (b, l, n) at record[b * rec_b_stride + l * I + n]; NULL: none
    int64_t rec_b_stride;
    const float* record_scale;         // [L, I] or NULL
    int* ctrl;
    unsigned long long epoch;          // of this launch, not 0
    int* status;
    int L, B, T, I, Hs;
    int nb;                            // episodes of the caller
    int n_sub;                         // token chunks per episode: "episode" e of the kernel is chunk e % n_sub of e / n_sub
    int T_all;                         // tokens per episode of the caller (T: tokens per chunk; the last one may hold fewer)
    int stages;                        // weight stages of each ring
    int anchor_mode;                   // Eq. 4 (EQ4 instantiation): RM_ANCHOR_*
    float* y_anchor;                   // [L,B,T,H]
    float* h_anchor;                   // [L,B,I,h_stride]
    int64_t h_stride;
    const float* gate;                 // [L,B,H] or NULL
    Lay lay;
};

// ---- instructions
__device__ __forceinline__ void ldm4(uint32_t a, uint32_t (&r)[4]) {
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0, %1, %2, %3}, [%4];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(a) : "memory");
}
__device__ __forceinline__ void ldm4t(uint32_t a, uint32_t (&r)[4]) {
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0, %1, %2, %3}, [%4];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(a) : "memory");
}
__device__ __forceinline__ void mma16816(float (&c)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1) {
    asm volatile("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, {%0, %1, %2, %3};"
                 : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
                 : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}
__device__ __forceinline__ void red_add_v2(float* p, float a, float b) {
    asm volatile("red.global.add.v2.f32 [%0], {%1, %2};" ::"l"(p), "f"(a), "f"(b) : "memory");
}
__device__ __forceinline__ int ld_acquire_gpu(const int* p) {
    int v;
    asm volatile("ld.acquire.gpu.global.s32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}
__device__ __forceinline__ void red_release_gpu(int* p, int v) {
    asm volatile("red.release.gpu.global.add.s32 [%0], %1;" ::"l"(p), "r"(v) : "memory");
}
// (relaxed: it only says that this CTA's reads of a buffer are over; the values have been used by then.  A release at cluster
// scope waits for every earlier store and add, an acquire at cluster scope empties the L1 cache)
__device__ __forceinline__ void arrive_remote(uint32_t cluster_addr) {
    asm volatile("mbarrier.arrive.relaxed.cluster.shared::cluster.b64 _, [%0];" ::"r"(cluster_addr) : "memory");
}
// ---- bounded waits.  Both return true when the waiter has to give up: the wait ran out (status RM_ERR_TIMEOUT with the
// wait's source line and the CTA), or this CTA or the grid is aborting.
__device__ __forceinline__ void report_timeout(const SArgs& a, volatile int* abort_cta, int line) {
    rm_set_status_at(a.status, RM_ERR_TIMEOUT, (line << 12) | (int)(blockIdx.x & 0xfffu));
    *abort_cta = 1;
    atomicExch(a.ctrl + 3, 1);
}
__device__ __forceinline__ bool wait_slow(uint32_t bar, uint32_t parity, int line, const SArgs& a, volatile int* abort_cta) {
    for (uint32_t i = 0; i < (1u << 22); ++i) {
        if (mbar_try_wait(bar, parity)) return false;
        if (i > 64) __nanosleep(32);
        if ((i & 1023u) == 1023u && (*abort_cta || ((i & 16383u) == 16383u && ld_acquire_gpu(a.ctrl + 3) == 1))) {
            *abort_cta = 1;
            return true;
        }
    }
    report_timeout(a, abort_cta, line);
    return true;
}
__device__ __forceinline__ bool counter_wait(const int* counter, int target, int line, const SArgs& a, volatile int* abort_cta) {
    for (uint32_t i = 0; i < (1u << 21); ++i) {
        if (ld_acquire_gpu(counter) >= target) return false;
        if ((i & 255u) == 255u && (*abort_cta || ld_acquire_gpu(a.ctrl + 3) == 1)) { *abort_cta = 1; return true; }
    }
    report_timeout(a, abort_cta, line);
    return true;
}
__device__ __forceinline__ bool epoch_wait(const int* ctrl, unsigned long long epoch, int line, const SArgs& a, volatile int* abort_cta) {
    for (uint32_t i = 0; i < (1u << 21); ++i) {
        unsigned long long v;
        asm volatile("ld.acquire.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(ctrl) : "memory");
        if (v == epoch) return false;
        if ((i & 255u) == 255u && *abort_cta) return true;
    }
    rm_set_status_at(a.status, RM_ERR_TIMEOUT, (line << 12) | (int)(blockIdx.x & 0xfffu));
    *abort_cta = 1;
    return true;
}
__device__ __forceinline__ bool barrier_or(int id, int count, bool pred) {
    uint32_t r;
    asm volatile(
        "{\n\t.reg .pred p, q;\n\t"
        "setp.ne.u32 p, %1, 0;\n\t"
        "barrier.cta.red.or.pred q, %2, %3, p;\n\t"
        "selp.u32 %0, 1, 0, q;\n\t}"
        : "=r"(r) : "r"((uint32_t)pred), "r"(id), "r"(count) : "memory");
    return r != 0;
}

// What a cluster does for one (layer, episode): n neurons of the list from position `start` (0: another cluster's, or an
// empty list whose residual this cluster passes on), `share` of `parts` of the item's token rows.
struct Item { int start, n, parts_share, target; };                // parts | share << 8 | takes part << 16; target: arrivals
                                                                   // on the episode's counter that complete the layer before

// NG: 8-column tiles of the slice per down warp (four column groups), so Hs <= 32 NG.  OPN: neurons per owner and round.  With
// OPN = 4 (wide slices, whose stages are large) rounds alternate between two teams of four gate/up warps.
template <int NG, int OPN, bool EQ4>
__global__ void __launch_bounds__(NTHREADS, 1) slice_kernel(const __grid_constant__ SArgs a) {
    // registers: 640 threads x 96 at launch; the four warps of the loaders give most of theirs to the two groups
    constexpr int REGS_L = 32, REGS_A = 104, REGS_B = 120;
    static_assert(REGS_L * 128 + (REGS_A + REGS_B) * 256 <= 96 * NTHREADS, "more registers than the block is launched with");
    constexpr int TEAMS = 8 / OPN, RN = CS * OPN, MAXV = 2 * NG;
    extern __shared__ __align__(16) unsigned char smem_dyn[];
    const uint32_t base = (smem_u32(smem_dyn) + 127u) & ~127u;
    unsigned char* gbase = smem_dyn + (base - smem_u32(smem_dyn));
    const Lay& y = a.lay;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int j = (int)cluster_ctarank(), c = (int)cluster_id_x(), NC = (int)cluster_count_x();
    const int Hs = a.Hs, H = CS * Hs, T = a.T, L = a.L, B = a.B, I = a.I, NST = a.stages;
    const int n_items = L * B;
    const int anchor_mode = EQ4 ? a.anchor_mode : (int)RM_ANCHOR_NONE;
    const uint32_t bar0 = base + y.off_bar;
    auto g_full = [&](int s) { return bar0 + 8 * s; };
    auto g_empty = [&](int s) { return bar0 + 128 + 8 * s; };
    auto d_full = [&](int s) { return bar0 + 256 + 8 * s; };
    auto d_empty = [&](int s) { return bar0 + 384 - 0 + 8 * s; };
    // (the remaining barriers and flags live behind the sums of squares' buffers, in the item table's last entry)
    Item* items = reinterpret_cast<Item*>(gbase + y.off_item);
    float* sSS = reinterpret_cast<float*>(gbase + y.off_ss);
    __shared__ __align__(8) unsigned long long sBar[2 + 2 + 2 + SSB];
    __shared__ int sAbortW, sSeen;
    auto p_full = [&](int b) { return smem_u32(&sBar[b]); };
    auto h_full = [&](int b) { return smem_u32(&sBar[2 + b]); };
    auto h_free = [&](int b) { return smem_u32(&sBar[4 + b]); };
    auto ss_bar = [&](int b) { return smem_u32(&sBar[6 + b]); };
    volatile int* sAbort = &sAbortW;

    // ---- set-up
    if (blockIdx.x == 0) {                 // the launch's counters, then its epoch
        for (int e = tid; e < B * CS * 2; e += NTHREADS) a.ctrl[CTRL_LINE * (1 + e)] = 0;
        if (tid == 0) { a.ctrl[2] = 0; a.ctrl[3] = 0; }
        __threadfence();
    }
    if (tid == 0) {
        for (int s = 0; s < NST; ++s) { mbar_init(g_full(s), 1); mbar_init(g_empty(s), 2); mbar_init(d_full(s), 1); mbar_init(d_empty(s), 8); }
        for (int b = 0; b < 2; ++b) { mbar_init(p_full(b), 1); mbar_init(h_full(b), 1); mbar_init(h_free(b), CS * 8); }
        for (int b = 0; b < SSB; ++b) mbar_init(ss_bar(b), 1);
        fence_mbar_init();
        *sAbort = 0;
        sSeen = 0;
    }
    {
        // counts, then this cluster's part of every item.  The lists of a layer's episodes, laid end to end, are cut evenly
        // over the clusters: cluster k takes positions [S k / NC, S (k + 1) / NC) of the S = sum of the counts.
        const int cap = (int)(a.list_cap < (int64_t)I ? a.list_cap : (int64_t)I);
        for (int it = tid; it < n_items; it += NTHREADS) {
            const int l = it / B, e = it - l * B, b = e / a.n_sub;
            int k = I;
            if (a.count) {
                k = a.count[(size_t)b * a.count_b_stride + l];
                if (k < 0 || k > cap) { rm_set_status(a.status, RM_ERR_INDEX); k = k < 0 ? 0 : cap; }
            }
            items[it].n = k;
        }
        __syncthreads();
        Item mine[1];
        for (int it0 = 0; it0 < n_items; it0 += NTHREADS) {        // (n_items <= 512 < NTHREADS: one pass)
            const int it = it0 + tid;
            if (it < n_items) {
                const int l = it / B, e = it - l * B, K = items[it].n;
                unsigned S = 0, P = 0;
                for (int b2 = 0; b2 < B; ++b2) {
                    const unsigned K2 = (unsigned)items[l * B + b2].n;
                    S += K2;
                    P += b2 < e ? K2 : 0u;
                }
                Item r{0, 0, 0, 0};
                if (K == 0) {
                    r.parts_share = 1 | (e % NC == c ? 1 << 16 : 0);
                } else {
                    int parts = 0, share = 0;
                    for (int k = 0; k < NC; ++k) {
                        const unsigned lo = S * (unsigned)k / (unsigned)NC, hi = S * (unsigned)(k + 1) / (unsigned)NC;
                        const unsigned x0 = lo > P ? lo : P, x1 = hi < P + K ? hi : P + K;
                        if (x1 > x0) {
                            if (k == c) { r.start = (int)(x0 - P); r.n = (int)(x1 - x0); share = parts; }
                            ++parts;
                        }
                    }
                    r.parts_share = parts | share << 8 | (r.n > 0 ? 1 << 16 : 0);
                }
                mine[0] = r;
            }
        }
        __syncthreads();
        if (tid < n_items) items[tid] = mine[0];
        __syncthreads();
        if (tid < B) {
            int t = 0;
            for (int l = 0; l < L; ++l) {
                items[l * B + tid].target = t;
                t += items[l * B + tid].parts_share & 0xff;
            }
        }
    }
    // x rows past T, columns past Hs, and weight slots that no copy has filled yet have to hold finite numbers: zeros
    for (int e = tid; e < 64 * y.xp / 16; e += NTHREADS) reinterpret_cast<uint4*>(gbase + y.off_x)[e] = make_uint4(0u, 0u, 0u, 0u);
    for (int e = tid; e < (y.total - 128 - y.off_g) / 16; e += NTHREADS) reinterpret_cast<uint4*>(gbase + y.off_g)[e] = make_uint4(0u, 0u, 0u, 0u);
    fence_proxy_async_smem();
    __syncthreads();
    cluster_sync();                        // peers' shared memory and barriers are live from here on
    if (blockIdx.x == 0 && tid == 0) {
        __threadfence();
        asm volatile("st.release.gpu.global.u64 [%0], %1;" ::"l"(a.ctrl), "l"(a.epoch) : "memory");
    }

    bool gave_up = false;
    auto wait_at = [&](uint32_t bar, uint32_t parity, int line) {
        if (gave_up || mbar_test_wait(bar, parity)) return;
        gave_up = wait_slow(bar, parity, line, a, sAbort);
    };
#define WAIT(bar, parity) wait_at((bar), (parity), __LINE__)
    // first token row (of the caller's [B, T_all]) and tokens of episode e
    auto row0_of = [&](int e) {
        if (a.n_sub == 1) return (size_t)e * T;
        const int b = e / a.n_sub, s = e - b * a.n_sub;
        return (size_t)b * a.T_all + (size_t)s * T;
    };
    auto tokens_of = [&](int e) {
        if (a.n_sub == 1) return T;
        const int s = e % a.n_sub, left = a.T_all - s * T;
        return left < T ? left : T;
    };
    auto list_of = [&](int l, int e) { return a.idx ? a.idx + (size_t)(a.n_sub == 1 ? e : e / a.n_sub) * a.idx_b_stride + (size_t)l * a.idx_l_stride : nullptr; };
    auto out_of = [&](int l) { return l == L - 1 ? a.r_out : a.rot[l % 3]; };

    if (warp >= W_G) {
        asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(REGS_L));
        if (warp < W_G + 2) {
        // ================================================================ loaders: a stage is the pieces of 16 neurons, one
        // bulk copy per neuron; they run as far ahead as the ring lets them (the lists are known before the step starts)
        const bool is_g = warp == W_G;
        const uint32_t ring = base + (is_g ? y.off_g : y.off_d), bytes = (uint32_t)Hs * (is_g ? 4u : 2u);
        const int pitch = is_g ? y.gp : y.dp, stage_bytes = is_g ? y.g_stage : y.d_stage;
        const uint32_t full0 = is_g ? g_full(0) : d_full(0), empty0 = is_g ? g_empty(0) : d_empty(0);
        int slot = 0;
        uint32_t pass = 0;
        for (int it = 0, l = 0, e = 0; it < n_items && !gave_up; ++it, (++e == B ? (e = 0, ++l) : 0)) {
            const Item w = items[it];
            if (w.n == 0) continue;
            const int32_t* list = list_of(l, e);
            const __nv_bfloat16* src = a.packed[l] + (size_t)j * 3 * Hs + (is_g ? 0 : 2 * Hs);
            auto neuron = [&](int k) {
                int n = -1;
                if (lane < SN && k + lane < w.n) {
                    n = list ? __ldg(list + w.start + k + lane) : w.start + k + lane;
                    if (n < 0 || n >= I) { rm_set_status(a.status, RM_ERR_INDEX); n = -1; }
                }
                return n;
            };
            int n = neuron(0);
            for (int k = 0; k < w.n && !gave_up; k += SN) {
                const int next = neuron(k + SN);                   // (asked for before this stage's wait)
                if (pass > 0) WAIT(empty0 + 8 * slot, (pass - 1) & 1);
                const uint32_t m = __ballot_sync(0xffffffffu, n >= 0);
                if (lane == 0) mbar_arrive_expect_tx(full0 + 8 * slot, (uint32_t)__popc(m) * bytes);
                __syncwarp();
                if (n >= 0) bulk_load(ring + slot * stage_bytes + lane * pitch, src + (size_t)n * 3 * H, bytes, full0 + 8 * slot);
                n = next;
                if (++slot == NST) { slot = 0; ++pass; }
                gave_up = __any_sync(0xffffffffu, gave_up);
            }
        }
        }
    } else if (warp < W_B) {
        asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(REGS_A));
        // ================================================================ group A: x of an item, then its gate/up products
        const int team = TEAMS == 2 ? warp >> 2 : 0, mp = TEAMS == 2 ? (warp >> 1) & 1 : warp >> 1, nh = warp & 1;
        const int cnt = nh ? y.n_b : y.n_a, nt0 = nh ? y.n_a : 0;  // this warp's 8-token tiles
        const int t = tid >> 2, q = tid & 3, n4 = Hs / 4;          // normalisation: token row, every fourth float4 of its slice
        const uint32_t a_lane = (lane & 7) * y.gp + ((lane >> 3) & 1) * 2 * Hs + (lane >> 4) * 16;
        const uint32_t x_lane = base + y.off_x + (nt0 * 8 + ((lane >> 4) << 3) + (lane & 7)) * y.xp + ((lane >> 3) & 1) * 16;
        unsigned char* stg = gbase + y.off_stg + warp * y.stg_warp;
        const uint32_t s_stg = base + y.off_stg + warp * y.stg_warp;
        uint32_t R = 0;                                            // rounds before this one
        int g_slot = 0, ni = 0, pi = 0;                            // ring slot of the round's first stage; items so far
        uint32_t g_pass = 0;
        for (int it = 0, l = 0, e = 0; it < n_items; ++it, (++e == B ? (e = 0, ++l) : 0)) {
            const Item w = items[it];
            if (!(w.parts_share >> 16)) continue;
            const int Te = tokens_of(e);
            const size_t row = row0_of(e) + t;
            // ---- every cluster has added its part of the layer before to this slice (one thread looks)
            if (tid == 0 && !gave_up) {
                if (pi == 0) gave_up = epoch_wait(a.ctrl, a.epoch, __LINE__, a, sAbort);
                if (l > 0 && !gave_up) gave_up = counter_wait(a.ctrl + ctrl_done(e, j), w.target, __LINE__, a, sAbort);
                asm volatile("st.release.cta.shared::cta.s32 [%0], %1;" ::"r"(smem_u32(&sSeen)), "r"(pi + 1) : "memory");
            }
            if (w.n == 0) { ++pi; continue; }                      // (nothing selected: group B passes the residual on)
            if (barrier_or(1, 256, gave_up || *sAbort)) break;
            const bool ext = a.x_ext != nullptr;
            float4 v[MAXV];
            float ss = 0.f;
            if (!ext) {
                const float4* src = reinterpret_cast<const float4*>((l == 0 ? a.r_in : out_of(l - 1)) + row * H + (size_t)j * Hs);
#pragma unroll
                for (int i = 0; i < MAXV; ++i)
                    v[i] = t < Te && q + 4 * i < n4 ? __ldcg(src + q + 4 * i) : make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
                for (int i = 0; i < MAXV; ++i) {
                    ss = fmaf(v[i].x, v[i].x, ss); ss = fmaf(v[i].y, v[i].y, ss);
                    ss = fmaf(v[i].z, v[i].z, ss); ss = fmaf(v[i].w, v[i].w, ss);
                }
                {
                    // all-gather of the row sums of squares over the cluster: lane q of a row sends to CTAs q and q + 4
                    ss += __shfl_xor_sync(0xffffffffu, ss, 1);
                    ss += __shfl_xor_sync(0xffffffffu, ss, 2);
                    const uint32_t bar = ss_bar(ni & (SSB - 1)), at = smem_u32(sSS + ((ni & (SSB - 1)) * CS + j) * 64 + t);
                    if (tid == 0) mbar_arrive_expect_tx(bar, CS * 64 * 4);
                    st_async_f32(map_to_rank(at, q), ss, map_to_rank(bar, q));
                    st_async_f32(map_to_rank(at, q + 4), ss, map_to_rank(bar, q + 4));
                }
            }
            // ---- x tile: [token][column] bf16
            if (ext) {
                const uint4* src = reinterpret_cast<const uint4*>(a.x_ext + row * H + (size_t)j * Hs);
#pragma unroll
                for (int i = 0; i < MAXV / 2; ++i)
                    if (t < Te && q + 4 * i < Hs / 8) *reinterpret_cast<uint4*>(gbase + y.off_x + t * y.xp + (q + 4 * i) * 16) = src[q + 4 * i];
            } else {
                const float* sums = sSS + (ni & (SSB - 1)) * CS * 64 + t;
                WAIT(ss_bar(ni & (SSB - 1)), (ni / SSB) & 1);
                float tot = 0.f;
#pragma unroll
                for (int s = 0; s < CS; ++s) tot += sums[s * 64];
                const float inv = 1.0f / sqrtf(tot / (float)H + 1e-6f);
#pragma unroll
                for (int i = 0; i < MAXV; ++i) {
                    if (q + 4 * i >= n4) continue;                 // (rows past Te: v = 0, so x = 0)
                    const __nv_bfloat162 lo = __floats2bfloat162_rn(v[i].x * inv, v[i].y * inv);
                    const __nv_bfloat162 hi = __floats2bfloat162_rn(v[i].z * inv, v[i].w * inv);
                    uint2 u;
                    u.x = *reinterpret_cast<const uint32_t*>(&lo);
                    u.y = *reinterpret_cast<const uint32_t*>(&hi);
                    *reinterpret_cast<uint2*>(gbase + y.off_x + t * y.xp + (q + 4 * i) * 8) = u;
                }
            }
            ++ni;
            ++pi;
            if (barrier_or(1, 256, gave_up || *sAbort)) break;
            // ---- gate/up: warp (mp, nh) multiplies stage mp of a round (two row tiles) with half of the tokens
            for (int pos = 0; pos < w.n; pos += RN, ++R) {
                const int nr = w.n - pos < RN ? w.n - pos : RN, ns = (nr + SN - 1) / SN;
                if (TEAMS == 1 || (int)(R & 1) == team) {
                    const bool act = mp < ns;
                    float acc[2][4][4];
                    if (act) {
                        int slot = g_slot + mp;
                        uint32_t ps = g_pass;
                        if (slot >= NST) { slot -= NST; ++ps; }
#pragma unroll
                        for (int u = 0; u < 2; ++u)
#pragma unroll
                            for (int n = 0; n < 4; ++n) acc[u][n][0] = acc[u][n][1] = acc[u][n][2] = acc[u][n][3] = 0.f;
                        WAIT(g_full(slot), ps & 1);
                        const uint32_t ga = base + y.off_g + slot * y.g_stage + a_lane, gb = ga + 8 * y.gp;
#pragma unroll 2
                        for (int ks = 0; ks < y.ks; ++ks) {
                            uint32_t A0[4], A1[4], X0[4], X1[4];
                            ldm4(ga + ks * 32, A0);
                            ldm4(gb + ks * 32, A1);
                            ldm4(x_lane + ks * 32, X0);
                            if (cnt > 2) ldm4(x_lane + 16 * y.xp + ks * 32, X1);
                            mma16816(acc[0][0], A0, X0[0], X0[1]);
                            mma16816(acc[1][0], A1, X0[0], X0[1]);
                            if (cnt > 1) { mma16816(acc[0][1], A0, X0[2], X0[3]); mma16816(acc[1][1], A1, X0[2], X0[3]); }
                            if (cnt > 2) { mma16816(acc[0][2], A0, X1[0], X1[1]); mma16816(acc[1][2], A1, X1[0], X1[1]); }
                            if (cnt > 3) { mma16816(acc[0][3], A0, X1[2], X1[3]); mma16816(acc[1][3], A1, X1[2], X1[3]); }
                        }
                        __syncwarp();
                        if (lane == 0) mbar_arrive(g_empty(slot));
                    }
                    // every owner has used up the partial sums of two rounds ago: h of that round is complete here
                    if (R >= 2) WAIT(h_full(R & 1), ((R >> 1) - 1) & 1);
                    if (act && cnt > 0) {
                        bulk_wait_read_all();                      // this warp's pieces of its previous round have left
                        __syncwarp();
                        // [row tile][neuron][token pair] (gate, gate, up, up)
#pragma unroll
                        for (int u = 0; u < 2; ++u) {
                            unsigned char* d = stg + (u * 8 + (lane >> 2)) * (cnt * 64) + (lane & 3) * 16;
#pragma unroll
                            for (int n = 0; n < 4; ++n)
                                if (n < cnt) *reinterpret_cast<float4*>(d + n * 64) = make_float4(acc[u][n][0], acc[u][n][1], acc[u][n][2], acc[u][n][3]);
                        }
                        fence_proxy_async_smem();
                        __syncwarp();
                        constexpr int OPT = 8 / OPN;               // owners per row tile
                        if (lane < 2 * OPT) {
                            const int o = 2 * OPT * mp + lane;     // owner; its neurons are OPN o .. of the round
                            if (o * OPN < nr && !gave_up) {
                                const uint32_t piece = (uint32_t)OPN * cnt * 64;
                                const uint32_t dst = base + y.off_p + (R & 1) * y.p_buf + j * y.p_src + nh * (OPN * y.n_a * 64);
                                bulk_copy_to_peer(map_to_rank(dst, o), s_stg + lane * piece, piece, map_to_rank(p_full(R & 1), o));
                            }
                        }
                        // (the lanes' copies are waited for by the lanes that issued them)
                        if (lane < 2 * OPT) bulk_commit();
                    }
                }
                g_slot += ns;
                if (g_slot >= NST) { g_slot -= NST; ++g_pass; }
            }
        }
        bulk_wait_read_all();
    } else {
        asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(REGS_B));
        // ================================================================ group B: owner work, down products, adds
        const int bt = tid - W_B * 32, bw = warp - W_B;
        const int th = bw & 1, cg = bw >> 1;                       // token half and column group of this warp's down products
        const int pairs = (Hs / 8 + 1) / 2, gpp = (pairs + 3) / 4; // pairs of 8-column tiles: of the slice, of a group
        const int cp0 = cg * gpp, cpn = pairs - cp0 < gpp ? pairs - cp0 : gpp;
        const int t16 = (T + 15) / 16, mh = (t16 + 1) / 2, m0 = th * mh, mcnt = t16 - m0 < mh ? t16 - m0 : mh;
        const int np = (y.n_a + y.n_b) * 4, na = y.n_a * 4;        // token pairs; of the first half
        const uint32_t h_lane = base + y.off_h + ((lane & 7) + ((lane >> 4) & 1) * 8) * HPITCH + (m0 * 16 + ((lane >> 3) & 1) * 8) * 2;
        const uint32_t d_lane = ((lane & 7) + ((lane >> 3) & 1) * 8) * y.dp + (cp0 * 16 + (lane >> 4) * 8) * 2;
        uint32_t R = 0, p_par = 0, d_pass = 0;
        int d_slot = 0, pi = 0;
        bool stop = false;
        for (int it = 0, l = 0, e = 0; it < n_items && !stop; ++it, (++e == B ? (e = 0, ++l) : 0)) {
            const Item w = items[it];
            if (!(w.parts_share >> 16)) continue;
            const int Te = tokens_of(e), b = a.n_sub == 1 ? e : e / a.n_sub, nb = a.nb;
            const size_t tok0 = (size_t)(e - b * a.n_sub) * T;     // first token of the chunk inside its episode
            const int32_t* list = list_of(l, e);
            float acc[2][NG][4];
#pragma unroll
            for (int m = 0; m < 2; ++m)
#pragma unroll
                for (int n = 0; n < NG; ++n) acc[m][n][0] = acc[m][n][1] = acc[m][n][2] = acc[m][n][3] = 0.f;
            // ---- while group A prepares x: this cluster's share of the layer's residual (+ gate * y_a in an update step) and
            // of the clearing of the next layer's output buffer.  Both need the layer before to be complete, which group A's
            // first thread has seen.
            if (bt == 0 && !gave_up) {
                int seen = 0;
                for (uint32_t i = 0; i < (1u << 24); ++i) {
                    asm volatile("ld.acquire.cta.shared::cta.s32 %0, [%1];" : "=r"(seen) : "r"(smem_u32(&sSeen)) : "memory");
                    if (seen > pi || *sAbort) break;
                }
                if (seen <= pi && !*sAbort) { report_timeout(a, sAbort, __LINE__); gave_up = true; }
            }
            ++pi;
            stop = barrier_or(2, 256, gave_up || *sAbort);
            if (stop) break;
            {
                const int parts = w.parts_share & 0xff, share = (w.parts_share >> 8) & 0xff, n4 = Hs / 4;
                const size_t lb = (size_t)l * nb + b, layer = (size_t)nb * a.T_all * H;
                const float* in = l == 0 ? a.r_in : out_of(l - 1);
                for (int z = bt; z < (Te - share + parts - 1) / parts * n4; z += 256) {
                    const int ri = z / n4, k = z - ri * n4;
                    const size_t o = (row0_of(e) + share + ri * parts) * H + (size_t)j * Hs + 4 * k;
                    float4 r = make_float4(0.f, 0.f, 0.f, 0.f);
                    if (in) r = __ldcg(reinterpret_cast<const float4*>(in + o));
                    if (EQ4 && anchor_mode == RM_ANCHOR_UPDATE) {
                        const float4 ya = __ldcg(reinterpret_cast<const float4*>(a.y_anchor + l * layer + o));
                        float4 g = make_float4(1.f, 1.f, 1.f, 1.f);
                        if (a.gate) g = __ldg(reinterpret_cast<const float4*>(a.gate + lb * H + (size_t)j * Hs) + k);
                        r.x = fmaf(g.x, ya.x, r.x); r.y = fmaf(g.y, ya.y, r.y); r.z = fmaf(g.z, ya.z, r.z); r.w = fmaf(g.w, ya.w, r.w);
                    }
                    float* out = out_of(l) + o;
                    const float4 zero = make_float4(0.f, 0.f, 0.f, 0.f);
                    if (l > 0) red_add_v4(out, r.x, r.y, r.z, r.w);
                    else if (out != in + o || !a.x_ext) *reinterpret_cast<float4*>(out) = r;
                    if (l + 1 < L) *reinterpret_cast<float4*>(out_of(l + 1) + o) = zero;
                    if (EQ4 && anchor_mode == RM_ANCHOR_WRITE) {
                        if (l == 0) *reinterpret_cast<float4*>(a.y_anchor + o) = zero;
                        if (l + 1 < L) *reinterpret_cast<float4*>(a.y_anchor + (l + 1) * layer + o) = zero;
                    }
                }
            }
            if (l == 0) {                                          // the first layer's output buffer is set up (this CTA's share)
                stop = barrier_or(2, 256, gave_up || *sAbort);
                if (bt == 0 && !stop) red_release_gpu(a.ctrl + ctrl_init(e, j), 1);
            }
            const int rounds = (w.n + RN - 1) / RN;
            for (int r = 0; r <= rounds && w.n > 0 && !stop; ++r) {
                if (r < rounds) {
                    // ---- owner work of round r: warp i has this CTA's neuron i, lane = token pair
                    const uint32_t Rr = R + r, buf = Rr & 1;
                    const int pos = r * RN, nr = w.n - pos < RN ? w.n - pos : RN, ns = (nr + SN - 1) / SN;
                    const int n_own = (nr + OPN - 1) / OPN;
                    const bool own = j < n_own;
                    const int qn = j * OPN + bw;
                    int n = -1;
                    if (own && bw < OPN && qn < nr) {
                        n = list ? __ldg(list + w.start + pos + qn) : w.start + pos + qn;
                        if (n < 0 || n >= I) n = -1;               // (reported by the loaders)
                    }
                    float2 ha = make_float2(0.f, 0.f);
                    float2* hap = nullptr;
                    if (EQ4 && anchor_mode != RM_ANCHOR_NONE && n >= 0 && 2 * lane < Te) {
                        hap = reinterpret_cast<float2*>(a.h_anchor + (((size_t)l * nb + b) * I + n) * a.h_stride + tok0) + lane;
                        if (anchor_mode == RM_ANCHOR_UPDATE) ha = __ldcg(hap);
                    }
                    float h0 = 0.f, h1 = 0.f;
                    if (own) {
                        if (bt == 0) mbar_arrive_expect_tx(p_full(buf), (uint32_t)y.p_buf);
                        WAIT(p_full(buf), (p_par >> buf) & 1u);
                        p_par ^= 1u << buf;
                        if (bw < OPN && lane < np) {
                            const unsigned char* p = gbase + y.off_p + buf * y.p_buf +
                                                     (lane < na ? bw * (na * 16) + lane * 16 : OPN * na * 16 + bw * ((np - na) * 16) + (lane - na) * 16);
                            float4 s = *reinterpret_cast<const float4*>(p);
#pragma unroll
                            for (int k = 1; k < CS; ++k) {
                                const float4 o = *reinterpret_cast<const float4*>(p + k * y.p_src);
                                s.x += o.x; s.y += o.y; s.z += o.z; s.w += o.w;
                            }
                            if (n >= 0) {
                                // GeLU-tanh(g) = g / (1 + exp(-2 z)), z = sqrt(2/pi) (g + 0.044715 g^3)
                                const float e0 = __expf(-1.5957691216057308f * (s.x + 0.044715f * s.x * s.x * s.x));
                                const float e1 = __expf(-1.5957691216057308f * (s.y + 0.044715f * s.y * s.y * s.y));
                                if (2 * lane < Te) h0 = __fdividef(s.x, 1.0f + e0) * s.z;
                                if (2 * lane + 1 < Te) h1 = __fdividef(s.y, 1.0f + e1) * s.w;
                            }
                        }
                        if (a.record && bw < OPN) {
                            float rec = fabsf(h0) + fabsf(h1);
#pragma unroll
                            for (int d = 16; d > 0; d >>= 1) rec += __shfl_xor_sync(0xffffffffu, rec, d);
                            if (lane == 0 && n >= 0) {
                                const float sc = a.record_scale ? a.record_scale[(size_t)l * I + n] : 1.f;
                                a.record[(size_t)b * a.rec_b_stride + (size_t)l * I + n] = a.record_scale ? rec * sc : rec;
                            }
                        }
                        if (EQ4 && hap) {
                            // Eq. 4: the anchor step retains h; an update step sends its difference from the anchor's h down
                            if (anchor_mode == RM_ANCHOR_WRITE) *hap = make_float2(h0, h1);
                            else { h0 -= ha.x; h1 -= 2 * lane + 1 < Te ? ha.y : 0.f; }
                        }
                    }
                    // every CTA of the cluster is done with this h buffer's previous round
                    if (Rr >= 2) WAIT(h_free(buf), ((Rr >> 1) - 1) & 1);
                    unsigned char* hb = gbase + y.off_h + buf * y.h_buf;
                    if (own && bw < OPN) {
                        const __nv_bfloat162 hi = __floats2bfloat162_rn(h0, h1);
                        const float2 hf = __bfloat1622float2(hi);
                        const __nv_bfloat162 lo = __floats2bfloat162_rn(h0 - hf.x, h1 - hf.y);
                        *reinterpret_cast<__nv_bfloat162*>(hb + qn * HPITCH + lane * 4) = hi;
                        *reinterpret_cast<__nv_bfloat162*>(hb + qn * HPITCH + 128 + lane * 4) = lo;
                    }
                    for (int z = n_own * OPN * 16 + bt; z < ns * SN * 16; z += 256)      // rows of the last stage that nobody owns
                        *reinterpret_cast<uint4*>(hb + (z >> 4) * HPITCH + (z & 15) * 16) = make_uint4(0u, 0u, 0u, 0u);
                    fence_proxy_async_smem();
                    stop = barrier_or(2, 256, gave_up || *sAbort);
                    if (bt == 32) mbar_arrive_expect_tx(h_full(buf), (uint32_t)(n_own - (own ? 1 : 0)) * (OPN * HPITCH));
                    if (own && bt < CS && bt != j && !stop) {
                        const uint32_t src = base + y.off_h + buf * y.h_buf + j * OPN * HPITCH;
                        bulk_copy_to_peer(map_to_rank(src, bt), src, OPN * HPITCH, map_to_rank(h_full(buf), bt));
                    }
                }
                if (r > 0 && !stop) {
                    // ---- down products of round r - 1
                    const uint32_t Rr = R + r - 1, buf = Rr & 1;
                    const int nr = w.n - (r - 1) * RN < RN ? w.n - (r - 1) * RN : RN, ns = (nr + SN - 1) / SN;
                    WAIT(h_full(buf), (Rr >> 1) & 1);
                    for (int s = 0; s < ns; ++s) {
                        WAIT(d_full(d_slot), d_pass & 1);
                        const uint32_t ha = h_lane + buf * y.h_buf + s * SN * HPITCH, wd = base + y.off_d + d_slot * y.d_stage + d_lane;
                        uint32_t Ah[2][4], Al[2][4];
#pragma unroll
                        for (int m = 0; m < 2; ++m)
                            if (m < mcnt) { ldm4t(ha + m * 32, Ah[m]); ldm4t(ha + 128 + m * 32, Al[m]); }
#pragma unroll
                        for (int n = 0; n < NG / 2; ++n)
                            if (n < cpn) {
                                uint32_t Bw[4];
                                ldm4t(wd + n * 32, Bw);
#pragma unroll
                                for (int m = 0; m < 2; ++m)
                                    if (m < mcnt) {
                                        mma16816(acc[m][2 * n], Ah[m], Bw[0], Bw[1]);
                                        mma16816(acc[m][2 * n + 1], Ah[m], Bw[2], Bw[3]);
                                        mma16816(acc[m][2 * n], Al[m], Bw[0], Bw[1]);
                                        mma16816(acc[m][2 * n + 1], Al[m], Bw[2], Bw[3]);
                                    }
                            }
                        __syncwarp();
                        if (lane == 0) mbar_arrive(d_empty(d_slot));
                        if (++d_slot == NST) { d_slot = 0; ++d_pass; }
                    }
                    __syncwarp();
                    if (lane < CS) arrive_remote(map_to_rank(h_free(buf), lane));
                }
            }
            R += rounds;
            if (stop) break;
            // ---- the item's sums are complete: into the output buffer of the layer (the first layer's has to be set up by
            // every cluster before)
            if (l == 0) {
                if (bt == 0 && !gave_up) gave_up = counter_wait(a.ctrl + ctrl_init(e, j), w.parts_share & 0xff, __LINE__, a, sAbort);
                stop = barrier_or(2, 256, gave_up || *sAbort);
                if (stop) break;
            }
            if (w.n > 0) {
                const size_t row0 = row0_of(e);
                float* ob = out_of(l) + row0 * H + (size_t)j * Hs;
                const float* gp = EQ4 && a.gate ? a.gate + ((size_t)l * nb + b) * H + (size_t)j * Hs : nullptr;
                float* yb = EQ4 && anchor_mode == RM_ANCHOR_WRITE ? a.y_anchor + ((size_t)l * nb * a.T_all + row0) * H + (size_t)j * Hs : nullptr;
#pragma unroll
                for (int n = 0; n < NG; ++n) {
                    const int col = (cp0 * 2 + n) * 8 + (lane & 3) * 2;
                    if ((n >> 1) >= cpn || col >= Hs) continue;
                    float2 g = make_float2(1.f, 1.f);
                    if (EQ4 && gp) g = __ldg(reinterpret_cast<const float2*>(gp + col));
#pragma unroll
                    for (int m = 0; m < 2; ++m)
#pragma unroll
                        for (int h = 0; h < 2; ++h) {
                            const int t = (m0 + m) * 16 + h * 8 + (lane >> 2);
                            if (m >= mcnt || t >= Te) continue;
                            const float y0 = acc[m][n][2 * h], y1 = acc[m][n][2 * h + 1];
                            red_add_v2(ob + (size_t)t * H + col, EQ4 ? g.x * y0 : y0, EQ4 ? g.y * y1 : y1);
                            if (EQ4 && yb) red_add_v2(yb + (size_t)t * H + col, y0, y1);
                        }
                }
            }
            // (the barrier orders every thread's adds before thread 0's release, which is cumulative)
            stop = barrier_or(2, 256, gave_up || *sAbort);
            if (bt == 0 && !stop) red_release_gpu(a.ctrl + ctrl_done(e, j), 1);
        }
    }
#undef WAIT
    __syncthreads();
    if (*sAbort) {
        // a wait gave up somewhere: copies into this CTA's shared memory may still be in flight although nobody waits for
        // them any more.  They land within microseconds; idle for longer than that.
        for (int i = 0; i < 64; ++i) __nanosleep(4000);
        __syncthreads();
    }
    cluster_sync();                        // no CTA leaves while a peer may still write into its shared memory
    if (tid == 0 && !epoch_wait(a.ctrl, a.epoch, __LINE__, a, sAbort)) {
        // the last CTA to leave takes the epoch back, so that a captured launch can be replayed
        if (atomicAdd(a.ctrl + 2, 1) == (int)gridDim.x - 1)
            asm volatile("st.release.gpu.global.u64 [%0], %1;" ::"l"(a.ctrl), "l"(0ull) : "memory");
    }
}

// ---- host side
constexpr int SMEM_MAX = 232448 - 1024;                            // (1 KB for the static part)

template <int NG, int OPN, bool EQ4>
int configure(int smem) {
    RM_CUDA_TRY(cudaFuncSetAttribute(slice_kernel<NG, OPN, EQ4>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem));
    return RM_OK;
}
void cluster_config(cudaLaunchConfig_t& cfg, cudaLaunchAttribute* at, int clusters, int smem, cudaStream_t s) {
    cfg.gridDim = dim3(CS * clusters);
    cfg.blockDim = dim3(NTHREADS);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = CS;
    at[0].val.clusterDim.y = 1;
    at[0].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
}
template <int NG, int OPN>
int query(int* out) {
    int rc = configure<NG, OPN, false>(SMEM_MAX);
    if (rc == RM_OK) rc = configure<NG, OPN, true>(SMEM_MAX);
    if (rc != RM_OK) return rc;
    cudaLaunchConfig_t cfg = {};
    cudaLaunchAttribute at[1];
    cluster_config(cfg, at, 32, SMEM_MAX, nullptr);
    RM_CUDA_TRY(cudaOccupancyMaxActiveClusters(out, slice_kernel<NG, OPN, true>, &cfg));
    return RM_OK;
}
template <int NG, int OPN, bool EQ4>
int launch(rm_ctx* ctx, const SArgs& a, int clusters, int smem, cudaStream_t s) {
    cudaLaunchConfig_t cfg = {};
    cudaLaunchAttribute at[1];
    cluster_config(cfg, at, clusters, smem, s);
    RM_CUDA_TRY(cudaLaunchKernelEx(&cfg, slice_kernel<NG, OPN, EQ4>, a));
    ctx->launches++;
    return RM_OK;
}

inline bool narrow(int Hs) { return Hs <= 128; }

// Stages of each weight ring that fit beside the other buffers, at most MAX_STAGES
int ring_stages(int Hs, int T) {
    const int opn = narrow(Hs) ? 8 : 4;
    int st = MAX_STAGES;
    while (st > 0 && make_layout(Hs, T, opn, st).total > SMEM_MAX) --st;
    return st;
}
// A chunk of more than 64 tokens is cut into equal parts (multiples of 8 tokens): tokens are independent of one another
void cut_tokens(int T, int& n_sub, int& part) {
    n_sub = (T + 63) / 64;
    part = n_sub == 1 ? T : ((T + n_sub - 1) / n_sub + 7) / 8 * 8;
}
unsigned long long next_epoch() {
    static std::atomic<unsigned long long> n{(unsigned long long)std::chrono::steady_clock::now().time_since_epoch().count() << 20 | 1u};
    return n.fetch_add(2);                                         // (odd: never 0)
}

}  // namespace

int rm_slice_init(rm_ctx* ctx) {
    ctx->slice_clusters = 0;
    const int Hs = ctx->g.Hs;
    if (Hs > 256 || ring_stages(Hs, 64) < 4) return RM_OK;
    int n = 0;
    const int rc = narrow(Hs) ? query<4, 8>(&n) : query<8, 4>(&n);
    if (rc == RM_OK) ctx->slice_clusters = n;
    return rc;
}

bool rm_slice_supported(const rm_ctx* ctx, int B, int T, bool record) {
    if (ctx->slice_clusters <= 0 || T < 1 || B < 1) return false;
    int n_sub, part;
    cut_tokens(T, n_sub, part);
    return B * n_sub <= MAXB && ctx->g.L <= MAXL && ctx->g.L * B * n_sub <= MAX_ITEMS && !(record && n_sub > 1);
}

size_t rm_slice_workspace_bytes(const rm_ctx* ctx, int B, int T) {
    if (ctx->slice_clusters <= 0) return 0;
    int n_sub, part;
    cut_tokens(T, n_sub, part);
    return B * n_sub <= MAXB ? ctrl_bytes(B * n_sub) : 0;
}

int rm_launch_step_slice(rm_ctx* ctx, const rm_step_args& sa, cudaStream_t s) {
    const rm_geom& g = ctx->g;
    SArgs a{};
    int n_sub, part;
    cut_tokens(sa.T, n_sub, part);
    for (int l = 0; l < sa.L; ++l) a.packed[l] = static_cast<const __nv_bfloat16*>(sa.packed_layers[l]);
    a.r_in = sa.r_in ? sa.r_in : sa.r;
    a.r_out = sa.r;
    for (int i = 0; i < 3; ++i) a.rot[i] = sa.rot[i];
    a.x_ext = static_cast<const __nv_bfloat16*>(sa.x_ext);
    if (sa.x_ext) {
        a.r_in = sa.r_in;
    } else if (a.r_in == a.r_out && sa.L < 3) {
        // in place, and the last layer's buffer would be cleared while the first layer still reads it
        RM_CUDA_TRY(cudaMemcpyAsync(sa.rot[2], sa.r, (size_t)sa.B * sa.T * g.H * sizeof(float), cudaMemcpyDeviceToDevice, s));
        a.r_in = sa.rot[2];
    }
    a.idx = sa.idx;
    a.count = sa.count;
    a.idx_b_stride = sa.idx_b_stride;
    a.idx_l_stride = sa.idx_l_stride;
    a.list_cap = sa.list_cap;
    a.count_b_stride = sa.count_b_stride;
    a.record = sa.record;
    a.rec_b_stride = sa.rec_b_stride;
    a.record_scale = sa.record_scale;
    a.ctrl = sa.ctrl;
    a.epoch = next_epoch();
    a.status = ctx->d_status;
    a.L = sa.L;
    a.B = sa.B * n_sub;
    a.T = part;
    a.I = g.I;
    a.Hs = g.Hs;
    a.n_sub = n_sub;
    a.nb = sa.B;
    a.T_all = sa.T;
    a.stages = ring_stages(g.Hs, part);
    a.anchor_mode = sa.anchor_mode;
    a.y_anchor = sa.y_anchor;
    a.h_anchor = sa.h_anchor;
    a.h_stride = sa.h_stride;
    a.gate = sa.gate;
    int nc = ctx->slice_clusters;
    if (ctx->max_clusters_override > 0 && ctx->max_clusters_override < nc) nc = ctx->max_clusters_override;
    const bool eq4 = sa.anchor_mode != RM_ANCHOR_NONE || sa.gate != nullptr;
    a.lay = make_layout(g.Hs, part, narrow(g.Hs) ? 8 : 4, a.stages);
    const int smem = a.lay.total;
    if (narrow(g.Hs)) return eq4 ? launch<4, 8, true>(ctx, a, nc, smem, s) : launch<4, 8, false>(ctx, a, nc, smem, s);
    return eq4 ? launch<8, 4, true>(ctx, a, nc, smem, s) : launch<8, 4, false>(ctx, a, nc, smem, s);
}

// Slice kernel of the masked gated MLP stack: ONE launch runs every layer of a denoising step.
//
// Clusters of 8 CTAs, all co-resident (one CTA per SM).  CTA j of a cluster owns column slice j (Hs = H/8 columns of the
// model width) for BOTH projections, so a neuron's slice -- gate, up and down piece side by side in the packed layout -- is
// read once, by one CTA, as two contiguous bulk copies.  The active list of a layer is cut over the clusters; a cluster
// walks its run in rounds of up to 14 tiles of 8 neurons:
//   gate/up : partial sums over the slice's columns, [8 gate rows, 8 up rows] x tokens, by mma.sync (m16n8k16, bf16 in, fp32
//             accumulators in registers)
//   owner   : tile i of the round belongs to CTA i mod 8.  The partial sums travel to it as bulk copies between the
//             CTAs' shared memories (laid out in the weight stage that the products have just read), counted on its
//             mbarrier; it adds the 8 slices' sums, applies gelu_tanh(g) * u, splits h into three bf16 terms (together its 24
//             bits) and copies its rows to the other CTAs' h tiles
//   down    : [tokens] x [the slice's columns], accumulated in registers over the rounds of the item, then stored as this
//             cluster's partial sums
//   sum     : once every cluster of an item has stored its part, each takes an equal share of the token rows, adds the parts in
//             the clusters' order and the residual, and writes the rows
// Nothing is added in the order of arrival, so that a step gives the same bits every time.  A CTA waits for other clusters
// only on its own slice: counters (episode, slice) count the clusters that have stored their part and those that have
// written their rows.
//
// The sums are as close to 64 bits as those of the CUDA-core kernels, which take the same shapes (fp32 throughout, one order):
// one layer of 1536/6144, 25 %, 51 tokens, relative error 4.1e-7 against 7.2e-7; 2048/8192, 90 tokens 5.2e-7 against 7.4e-7.  With
// h in two terms, exponentials and divisions of reduced precision and a chain of products over the whole list it is 2.5e-6.
// Order and precision cost 13 %: 12 layers of 1536/6144 take 272 us, adding h of 17 bits in the order of arrival 241.
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
#include "rm_grid.cuh"
#include "rm_sm100.cuh"

using namespace sm100;
using namespace grid;

namespace {

constexpr int CS = 8;                  // CTAs per cluster = column slices of the packed layout
constexpr int TN = 8;                  // neurons of a tile: 8 gate rows and 8 up rows make one 16-row operand
constexpr int SN = 2 * TN;             // neurons of a weight stage
constexpr int MAX_ITEMS = 512;         // layers x episodes of one launch
constexpr int MAXL = 64;
constexpr int NTHREADS = 640;          // warps 0-7: normalisation and gate/up (group A); 8-15: owner, down, adds (group B);
constexpr int W_B = 8, W_G = 16;       // 16 / 17: loaders of the gate/up and of the down pieces
constexpr int HPITCH = 400;            // bytes of an h row: three terms of 64 tokens, 16 to spread the banks
constexpr int P_SRC = 4096;            // partial sums of a tile from one CTA: [8-token tile][neuron][token pair] (gate, gate, up, up)
constexpr int P_SLOT = CS * P_SRC;
constexpr int SSB = 4;                 // buffers of the row sums of squares: a CTA can be two items ahead of another
constexpr int MAX_STAGES = 16;
constexpr int EXACT_STAGES = 6;        // of the 128-column slice
constexpr int GROUP = 8;               // episodes (chunks) of one launch: a part of every cluster for each is kept in the workspace

// the control block's counters, lines of 32 ints: per (episode, slice) the CTAs that have stored their part, and the CTAs that have
// written their rows (both cumulative over the layers)
__host__ __device__ constexpr int ctrl_part(int e, int j) { return CTRL_LINE * (1 + (e * CS + j) * 2); }
__host__ __device__ constexpr int ctrl_done(int e, int j) { return CTRL_LINE * (2 + (e * CS + j) * 2); }
__host__ __device__ constexpr size_t ctrl_bytes(int B) { return (size_t)CTRL_LINE * (1 + 2 * CS * B) * sizeof(int); }

// ---- shared memory.  ts: tiles that one CTA may own per round (a round has up to 8 ts tiles)
struct Lay {
    int ks, xp, gp, dp;                // 16-column steps of the slice; row pitches: x tile, gate|up pieces, down pieces (odd multiples
                                       // of 16 bytes: eight rows of an ldmatrix fall into different banks)
    int g_stage, d_stage, stages;
    int off_ss, off_x, off_p, off_h, off_g, off_d, off_item, total;
};
__host__ __device__ constexpr Lay make_layout(int Hs, int ts, int stages) {
    Lay y{};
    y.ks = (Hs + 15) / 16;
    y.xp = y.ks * 32 + 16;
    y.gp = Hs * 4 + 16;
    y.dp = (Hs / 8) % 2 ? Hs * 2 : Hs * 2 + 16;
    // (a gate/up stage that has been used holds the two warps' outgoing partial sums, 8 KB)
    y.g_stage = SN * y.gp > 8192 ? SN * y.gp : 8192;
    y.d_stage = SN * y.dp + 32;        // (an odd last pair of column tiles reads 16 bytes past the last row)
    y.stages = stages;
    y.off_ss = 512;                    // (the barriers of the rings in front of it)
    y.off_x = y.off_ss + SSB * CS * 64 * 4;
    y.off_p = y.off_x + 64 * y.xp;
    y.off_h = y.off_p + ts * P_SLOT;
    y.off_g = y.off_h + ts * CS * TN * HPITCH;
    y.off_d = y.off_g + stages * y.g_stage;
    y.off_item = y.off_d + stages * y.d_stage;
    y.total = y.off_item + MAX_ITEMS * 12 + 128;
    return y;
}

struct SArgs {
    const __nv_bfloat16* packed[MAXL];
    const float* r_in;                 // [B,T,H] r_0
    float* r_out;                      // [B,T,H] r_L
    float* part;                       // [B][clusters][T][H]: a layer's partial sums, by episode and share
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
    int n_sub;                         // token chunks per episode: "episode" e of the kernel is chunk (e0 + e) % n_sub of (e0 + e) / n_sub
    int e0;                            // first chunk of this launch
    int T_all;                         // tokens per episode of the caller (T: tokens per chunk; the last one may hold fewer)
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
// (relaxed: it only says that this CTA's reads of a buffer are over; the values have been used by then.  A release at cluster
// scope waits for every earlier store and add, an acquire at cluster scope empties the L1 cache)
__device__ __forceinline__ void arrive_remote(uint32_t cluster_addr) {
    asm volatile("mbarrier.arrive.relaxed.cluster.shared::cluster.b64 _, [%0];" ::"r"(cluster_addr) : "memory");
}
// What a cluster does for one (layer, episode): n neurons of the list from position `start` (0: another cluster's, or an
// empty list whose rows this cluster passes on), `share` of `parts` of the item's token rows; `target`: arrivals on the episode's
// counters that complete the layer before.
struct Item {
    int start, n;
    unsigned bits;                     // parts | share << 8 | takes part << 16 | target << 17
    __device__ int parts() const { return (int)(bits & 0xffu); }
    __device__ int share() const { return (int)((bits >> 8) & 0xffu); }
    __device__ bool mine() const { return (bits >> 16) & 1u; }
    __device__ int target() const { return (int)(bits >> 17); }
};

// A cluster's run of n neurons is tiles of 8, cut into rounds of at most `most` tiles, as even as they come: round r of nrd
// starts at neuron pos and has nr.
__device__ __forceinline__ int round_count(int n, int most) { return ((n + TN - 1) / TN + most - 1) / most; }
__device__ __forceinline__ void round_span(int n, int r, int nrd, int& pos, int& nr) {
    if (nrd == 1) { pos = 0; nr = n; return; }
    const int tiles = (n + TN - 1) / TN, a = tiles * r / nrd, b = tiles * (r + 1) / nrd;
    pos = a * TN;
    nr = (b * TN < n ? b * TN : n) - pos;
}

// HS: columns of a slice (0: any, from the arguments -- the address arithmetic then costs instructions in every phase).  NG:
// 8-column tiles of the slice per down warp (four column groups), so Hs <= 32 NG.  TS: tiles a CTA may own per round.
template <int HS, int NG, int TS, bool EQ4>
__global__ void __launch_bounds__(NTHREADS, 1) slice_kernel(const __grid_constant__ SArgs a) {
    // registers: 640 threads x 96 at launch; the four warps of the loaders give most of theirs to the two groups
    constexpr int REGS_L = 32, REGS_A = NG == 4 ? 120 : 104, REGS_B = NG == 4 ? 104 : 120;
    static_assert(REGS_L * 128 + (REGS_A + REGS_B) * 256 <= 96 * NTHREADS, "more registers than the block is launched with");
    constexpr int MAXV = 2 * NG;
    constexpr Lay LC = make_layout(HS ? HS : 128, TS, EXACT_STAGES);
#define LY(field) (HS ? LC.field : a.lay.field)
    const int Hs = HS ? HS : a.Hs, H = CS * Hs, NST = LY(stages);
    extern __shared__ __align__(16) unsigned char smem_dyn[];
    const uint32_t base = (smem_u32(smem_dyn) + 127u) & ~127u;
    unsigned char* gbase = smem_dyn + (base - smem_u32(smem_dyn));
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int j = (int)cluster_ctarank();
    const int n_items = a.L * a.B;
    const int anchor_mode = EQ4 ? a.anchor_mode : (int)RM_ANCHOR_NONE;
    auto g_full = [&](int s) { return base + 8 * s; };
    auto g_empty = [&](int s) { return base + 128 + 8 * s; };
    auto d_full = [&](int s) { return base + 256 + 8 * s; };
    auto d_empty = [&](int s) { return base + 384 + 8 * s; };
    Item* items = reinterpret_cast<Item*>(gbase + LY(off_item));
    float* sSS = reinterpret_cast<float*>(gbase + LY(off_ss));
    __shared__ __align__(8) unsigned long long sBar[4 + SSB];
    __shared__ int sAbortW, sSeen;
    auto p_full = [&](int b) { return smem_u32(&sBar[b]); };       // per owned tile of a round
    const uint32_t h_full = smem_u32(&sBar[2]), h_free = smem_u32(&sBar[3]);
    auto ss_bar = [&](int b) { return smem_u32(&sBar[4 + b]); };
    volatile int* sAbort = &sAbortW;

    // ---- set-up
    if (tid == 0) {
        for (int s = 0; s < NST; ++s) { mbar_init(g_full(s), 1); mbar_init(g_empty(s), 2); mbar_init(d_full(s), 1); mbar_init(d_empty(s), 8); }
        mbar_init(p_full(0), 1); mbar_init(p_full(1), 1); mbar_init(h_full, 1); mbar_init(h_free, CS * 8);
        for (int b = 0; b < SSB; ++b) mbar_init(ss_bar(b), 1);
        fence_mbar_init();
        *sAbort = 0;
        sSeen = 0;
    }
    // x rows past T, columns past Hs, and weight slots that no copy has filled yet have to hold finite numbers: zeros
    for (int e = tid; e < 64 * LY(xp) / 16; e += NTHREADS) reinterpret_cast<uint4*>(gbase + LY(off_x))[e] = make_uint4(0u, 0u, 0u, 0u);
    for (int e = tid; e < (LY(off_item) - LY(off_g)) / 16; e += NTHREADS) reinterpret_cast<uint4*>(gbase + LY(off_g))[e] = make_uint4(0u, 0u, 0u, 0u);
    pdl_wait();                            // (a dependent launch: nothing above depends on the kernel in front)
    if (blockIdx.x == 0) {                 // the launch's counters, then (below) its epoch
        for (int e = tid; e < a.B * CS * 2; e += NTHREADS) a.ctrl[CTRL_LINE * (1 + e)] = 0;
        if (tid == 0) { a.ctrl[2] = 0; a.ctrl[3] = 0; }
        __threadfence();
    }
    {
        // counts, then this cluster's part of every item.  The lists of a layer's episodes, laid end to end, are cut evenly
        // over the clusters: cluster k takes positions [S k / NC, S (k + 1) / NC) of the S = sum of the counts.
        const int c = (int)cluster_id_x(), NC = (int)cluster_count_x(), B = a.B;
        const int cap = (int)(a.list_cap < (int64_t)a.I ? a.list_cap : (int64_t)a.I);
        const int it = tid, l = it / B, e = it - l * B;            // (n_items <= 512 < NTHREADS)
        if (it < n_items) {
            int k = a.I;
            if (a.count) {
                k = a.count[(size_t)((a.e0 + e) / a.n_sub) * a.count_b_stride + l];
                if (k < 0 || k > cap) { rm_set_status(a.status, RM_ERR_INDEX); k = k < 0 ? 0 : cap; }
            }
            items[it].n = k;
        }
        __syncthreads();
        Item r{0, 0, 0};
        if (it < n_items) {
            const unsigned K = (unsigned)items[it].n;
            unsigned S = 0, P = 0;
            for (int b2 = 0; b2 < B; ++b2) {
                const unsigned K2 = (unsigned)items[l * B + b2].n;
                S += K2;
                P += b2 < e ? K2 : 0u;
            }
            if (K == 0) {
                r.bits = 1u | (e % NC == c ? 1u << 16 : 0u);
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
                r.bits = (unsigned)(parts | share << 8 | (r.n > 0 ? 1 << 16 : 0));
            }
        }
        __syncthreads();
        if (it < n_items) items[it] = r;
        __syncthreads();
        if (tid < B) {
            unsigned t = 0;
            for (int l2 = 0; l2 < a.L; ++l2) {
                Item& q = items[l2 * B + tid];
                q.bits |= t << 17;
                t += (unsigned)q.parts();
            }
        }
    }
    fence_proxy_async_smem();
    __syncthreads();
    cluster_sync();                        // peers' shared memory and barriers are live from here on
    pdl_launch_dependents();               // (a dependent waits for this grid's end: its CTAs are resident by then)
    if (blockIdx.x == 0 && tid == 0) {
        epoch_publish(a.ctrl, a.epoch);
    }

    bool gave_up = false;
    auto wait_at = [&](uint32_t bar, uint32_t parity, int line) {
        if (gave_up || mbar_test_wait(bar, parity)) return;
        gave_up = wait_slow(bar, parity, line, a, sAbort);
    };
#define WAIT(bar, parity) wait_at((bar), (parity), __LINE__)
    // One round of tests for up to 32 barriers, a lane each (a test takes ~200 clocks to come back), for a whole warp
    auto wait_lanes = [&](bool active, uint32_t bar, uint32_t parity, int line) {
        if (__all_sync(0xffffffffu, !active || gave_up || mbar_test_wait(bar, parity))) return;
        if (active && !gave_up) gave_up = wait_slow(bar, parity, line, a, sAbort);
        gave_up = __any_sync(0xffffffffu, gave_up);
    };
    // first token row (of the caller's [B, T_all]) and tokens of episode e
    auto episode_of = [&](int e) { return a.n_sub == 1 ? a.e0 + e : (a.e0 + e) / a.n_sub; };
    auto row0_of = [&](int e) {
        const int b = episode_of(e);
        return (size_t)b * a.T_all + (size_t)(a.e0 + e - b * a.n_sub) * a.T;
    };
    auto tokens_of = [&](int e) {
        if (a.n_sub == 1) return a.T;
        const int s = (a.e0 + e) % a.n_sub, left = a.T_all - s * a.T;
        return left < a.T ? left : a.T;
    };
    auto list_of = [&](int l, int e) { return a.idx ? a.idx + (size_t)episode_of(e) * a.idx_b_stride + (size_t)l * a.idx_l_stride : nullptr; };
    const int most = 8 * TS < 2 * NST ? 8 * TS : 2 * NST;          // tiles per round: every one of its stages fits the ring

    if (warp >= W_G) {
        asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(REGS_L));
        if (warp < W_G + 2) {
            // ============================================================ loaders: a stage is the pieces of two tiles, one bulk
            // copy per neuron; they run as far ahead as the ring lets them (the lists are known before the step starts)
            const bool is_g = warp == W_G;
            // (8 columns past an up piece meet zeros of x in the last 16-column step: they have to be numbers, and the stage has
            // held partial sums since it was cleared -- so the copy goes on into the down piece)
            const uint32_t ring = base + (is_g ? LY(off_g) : LY(off_d)), bytes = (uint32_t)Hs * (is_g ? 4u : 2u) + (is_g && Hs % 16 ? 16u : 0u);
            const int pitch = is_g ? LY(gp) : LY(dp), stage_bytes = is_g ? LY(g_stage) : LY(d_stage);
            const uint32_t full0 = is_g ? g_full(0) : d_full(0), empty0 = is_g ? g_empty(0) : d_empty(0);
            int slot = 0;
            uint32_t pass = 0;
            for (int it = 0, l = 0, e = 0; it < n_items && !gave_up; ++it, (++e == a.B ? (e = 0, ++l) : 0)) {
                const Item w = items[it];
                if (w.n == 0) continue;
                const int32_t* list = list_of(l, e);
                const __nv_bfloat16* src = a.packed[l] + (size_t)j * 3 * Hs + (is_g ? 0 : 2 * Hs);
                const int nrd = round_count(w.n, most);
                for (int r = 0; r < nrd && !gave_up; ++r) {
                    int pos, nr;
                    round_span(w.n, r, nrd, pos, nr);
                    auto neuron = [&](int k) {
                        int n = -1;
                        if (lane < SN && k + lane < nr) {
                            n = w.start + pos + k + lane;
                            if (list) n = __ldg(list + n);
                            if (n < 0 || n >= a.I) { rm_set_status(a.status, RM_ERR_INDEX); n = -1; }
                        }
                        return n;
                    };
                    int n = neuron(0);
                    for (int k = 0; k < nr && !gave_up; k += SN) {
                        const int next = neuron(k + SN);           // (asked for before this stage's wait)
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
        }
    } else if (warp < W_B) {
        asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(REGS_A));
        // ================================================================ group A: x of an item, then its gate/up products
        const int mp = warp >> 1, nh = warp & 1;                   // gate/up: pair of tiles mp, mp + 4 of a round; token half
        const int t8 = (a.T + 7) / 8, cnt = nh ? (t8 > 4 ? t8 - 4 : 0) : (t8 < 4 ? t8 : 4);
        const int t = tid >> 2, q = tid & 3, n4 = Hs / 4;          // normalisation: token row, every fourth float4 of its slice
        const uint32_t a_lane = base + LY(off_g) + (lane & 7) * LY(gp) + ((lane >> 3) & 1) * 2 * Hs + (lane >> 4) * 16;
        const uint32_t x_lane = base + LY(off_x) + (nh * 32 + ((lane >> 4) << 3) + (lane & 7)) * LY(xp) + ((lane >> 3) & 1) * 16;
        uint32_t R = 0;                                            // rounds before this one
        int g_slot = 0, ni = 0, pi = 0;                            // ring slot of the round's first stage; items so far
        uint32_t g_pass = 0;
        for (int it = 0, l = 0, e = 0; it < n_items; ++it, (++e == a.B ? (e = 0, ++l) : 0)) {
            const Item w = items[it];
            if (!w.mine()) continue;
            const int Te = tokens_of(e);
            const float4* src = reinterpret_cast<const float4*>((l == 0 ? a.r_in : a.r_out) + (row0_of(e) + t) * H + (size_t)j * Hs) + q;
            // ---- every row of the layer before has been written in this slice (one thread looks)
            if (tid == 0 && !gave_up) {
                if (pi == 0) gave_up = epoch_wait(a.ctrl, a.epoch, __LINE__, a, sAbort);
                if (l > 0 && !gave_up) gave_up = counter_wait(a.ctrl + ctrl_done(e, j), w.target(), __LINE__, a, sAbort);
                asm volatile("st.release.cta.shared::cta.s32 [%0], %1;" ::"r"(smem_u32(&sSeen)), "r"(pi + 1) : "memory");
            }
            ++pi;
            if (barrier_or(1, 256, gave_up || *sAbort)) break;
            if (w.n == 0) continue;                                // (nothing selected: group B passes the residual on)
            // ---- x tile: [token][column] bf16
            if (a.x_ext) {
                const uint4* xs = reinterpret_cast<const uint4*>(a.x_ext + (row0_of(e) + t) * H + (size_t)j * Hs);
#pragma unroll
                for (int i = 0; i < MAXV / 2; ++i)
                    if (t < Te && q + 4 * i < Hs / 8) *reinterpret_cast<uint4*>(gbase + LY(off_x) + t * LY(xp) + (q + 4 * i) * 16) = xs[q + 4 * i];
            } else {
                float4 v[MAXV];
                float ss = 0.f;
#pragma unroll
                for (int i = 0; i < MAXV; ++i) v[i] = t < Te && (HS || q + 4 * i < n4) ? __ldcg(src + 4 * i) : make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
                for (int i = 0; i < MAXV; ++i) {
                    ss = fmaf(v[i].x, v[i].x, ss); ss = fmaf(v[i].y, v[i].y, ss);
                    ss = fmaf(v[i].z, v[i].z, ss); ss = fmaf(v[i].w, v[i].w, ss);
                }
                // all-gather of the row sums of squares over the cluster: lane q of a row sends to CTAs q and q + 4
                ss += __shfl_xor_sync(0xffffffffu, ss, 1);
                ss += __shfl_xor_sync(0xffffffffu, ss, 2);
                const int sb = ni & (SSB - 1);
                const uint32_t bar = ss_bar(sb), at = smem_u32(sSS) + ((sb * 64 + t) * CS + j) * 4;
                if (tid == 0) mbar_arrive_expect_tx(bar, CS * 64 * 4);
                st_async_f32(map_to_rank(at, q), ss, map_to_rank(bar, q));
                st_async_f32(map_to_rank(at, q + 4), ss, map_to_rank(bar, q + 4));
                WAIT(bar, (ni / SSB) & 1);
                const float4* sums = reinterpret_cast<const float4*>(sSS + (sb * 64 + t) * CS);
                const float4 s0 = sums[0], s1 = sums[1];
                const float tot = ((s0.x + s0.y) + (s0.z + s0.w)) + ((s1.x + s1.y) + (s1.z + s1.w));
                const float inv = __frsqrt_rn(tot / (float)H + 1e-6f);
                unsigned char* xr = gbase + LY(off_x) + t * LY(xp) + q * 8;
#pragma unroll
                for (int i = 0; i < MAXV; ++i) {
                    if (!HS && q + 4 * i >= n4) continue;          // (rows past Te: v = 0, so x = 0)
                    const __nv_bfloat162 lo = __floats2bfloat162_rn(v[i].x * inv, v[i].y * inv);
                    const __nv_bfloat162 hi = __floats2bfloat162_rn(v[i].z * inv, v[i].w * inv);
                    uint2 u;
                    u.x = *reinterpret_cast<const uint32_t*>(&lo);
                    u.y = *reinterpret_cast<const uint32_t*>(&hi);
                    *reinterpret_cast<uint2*>(xr + i * 32) = u;
                }
                ++ni;
            }
            named_barrier(1, 256);
            // ---- gate/up: warp (mp, nh) multiplies the pairs of tiles mp and mp + 4 of a round with its half of the tokens
            const int nrd = round_count(w.n, most);
            for (int r = 0; r < nrd; ++r, ++R) {
                int pos, nr;
                round_span(w.n, r, nrd, pos, nr);
                const int tiles = (nr + TN - 1) / TN, pairs = (tiles + 1) / 2;
                {
                    const int p = mp + 4 * lane;                   // lane u looks at the stage of this warp's pair u
                    int slot = g_slot + p;
                    uint32_t ps = g_pass;
                    if (slot >= NST) { slot -= NST; ++ps; }
                    wait_lanes(lane < TS && p < pairs, g_full(slot), ps & 1, __LINE__);
                }
                int held = -1;                                     // stage that this warp's outgoing sums still lie in
#pragma unroll 1
                for (int u = 0; u < TS; ++u) {
                    const int p = mp + 4 * u;
                    if (p >= pairs) break;
                    int slot = g_slot + p;
                    if (slot >= NST) slot -= NST;
                    float acc[2][4][4];
#pragma unroll
                    for (int m = 0; m < 2; ++m)
#pragma unroll
                        for (int n = 0; n < 4; ++n) acc[m][n][0] = acc[m][n][1] = acc[m][n][2] = acc[m][n][3] = 0.f;
                    const uint32_t ga = a_lane + slot * LY(g_stage);
#pragma unroll 4
                    for (int ks = 0; ks < LY(ks); ++ks) {
                        uint32_t A0[4], A1[4], X0[4], X1[4];
                        ldm4(ga + ks * 32, A0);
                        ldm4(x_lane + ks * 32, X0);
                        ldm4(ga + 8 * LY(gp) + ks * 32, A1);
                        if (cnt > 2) ldm4(x_lane + 16 * LY(xp) + ks * 32, X1);
                        mma16816(acc[0][0], A0, X0[0], X0[1]);
                        if (cnt > 1) mma16816(acc[0][1], A0, X0[2], X0[3]);
                        mma16816(acc[1][0], A1, X0[0], X0[1]);
                        if (cnt > 1) mma16816(acc[1][1], A1, X0[2], X0[3]);
                        if (cnt > 2) { mma16816(acc[0][2], A0, X1[0], X1[1]); mma16816(acc[1][2], A1, X1[0], X1[1]); }
                        if (cnt > 3) { mma16816(acc[0][3], A0, X1[2], X1[3]); mma16816(acc[1][3], A1, X1[2], X1[3]); }
                    }
                    // both warps of the pair have read the stage: it holds their outgoing sums now, 4 KB each
                    named_barrier(3 + mp, 64);
                    if (held >= 0) {                               // (the previous pair's sums have left by now)
                        bulk_wait_read_all();
                        __syncwarp();
                        if (lane == 0) mbar_arrive(g_empty(held));
                    }
                    held = slot;
                    const int out = LY(off_g) + slot * LY(g_stage) + nh * 4096;
                    unsigned char* d = gbase + out + lane * 16;
#pragma unroll
                    for (int m = 0; m < 2; ++m)
#pragma unroll
                        for (int n = 0; n < 4; ++n)
                            if (n < cnt) *reinterpret_cast<float4*>(d + m * 2048 + n * 512) = make_float4(acc[m][n][0], acc[m][n][1], acc[m][n][2], acc[m][n][3]);
                    fence_proxy_async_smem();
                    // every owner has used up the sums of the round before: h of that round is complete here
                    if (R >= 1 && u == 0) WAIT(h_full, (R - 1) & 1);
                    __syncwarp();
                    const int tile = 2 * p + lane;                 // lanes 0 and 1 send a tile each
                    if (lane < 2 && tile < tiles && cnt > 0 && !gave_up) {
                        const int o = tile & 7, s = tile >> 3;     // its owner, and which of the owner's tiles it is
                        bulk_copy_to_peer(map_to_rank(base + LY(off_p) + s * P_SLOT + j * P_SRC + nh * 2048, o), base + out + lane * 2048,
                                          (uint32_t)cnt * 512u, map_to_rank(p_full(s), o));
                        bulk_commit();
                    }
                }
                if (held >= 0) {
                    bulk_wait_read_all();
                    __syncwarp();
                    if (lane == 0) mbar_arrive(g_empty(held));
                } else if (R >= 1) {
                    WAIT(h_full, (R - 1) & 1);                     // (a warp follows every phase: parity tells two apart)
                }
                g_slot += pairs;
                if (g_slot >= NST) { g_slot -= NST; ++g_pass; }
                // A parity tells a phase from the one before it only.  A ring slot's phases belong to different warps, and copies
                // complete in any order: no warp looks at a slot's next phase before every warp has seen its own in this round.
                if (r + 1 < nrd) named_barrier(1, 256);
            }
        }
        bulk_wait_read_all();
    } else {
        asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(REGS_B));
        // ================================================================ group B: owner work, down products, adds
        const int bt = tid - W_B * 32, bw = warp - W_B;
        const int th = bw & 1, cg = bw >> 1;                       // token half and column group of this warp's down products
        const int pairs = (Hs / 8 + 1) / 2, gpp = (pairs + 3) / 4; // pairs of 8-column tiles: of the slice, of a group
        const int cp0 = cg * gpp, cpn = HS ? NG / 2 : (pairs - cp0 < gpp ? pairs - cp0 : gpp);
        const int t16 = (a.T + 15) / 16, mh = (t16 + 1) / 2, m0 = th * mh, mcnt = t16 - m0 < mh ? t16 - m0 : mh;
        const int np = (a.T + 7) / 8 * 4;                          // token pairs
        const uint32_t h_lane = base + LY(off_h) + ((lane & 7) + ((lane >> 4) & 1) * 8) * HPITCH + (m0 * 16 + ((lane >> 3) & 1) * 8) * 2;
        const uint32_t d_lane = base + LY(off_d) + ((lane & 7) + ((lane >> 3) & 1) * 8) * LY(dp) + (cp0 * 16 + (lane >> 4) * 8) * 2;
        const int parts_max = (int)cluster_count_x();
        uint32_t R = 0, p_par = 0, d_pass = 0;
        int d_slot = 0, pi = 0;
        bool stop = false;
        for (int l = 0; l < a.L && !stop; ++l) {
        for (int e = 0; e < a.B && !stop; ++e) {
            const Item w = items[l * a.B + e];
            if (!w.mine()) continue;
            const int Te = tokens_of(e), b = episode_of(e);
            const size_t tok0 = (size_t)(a.e0 + e - b * a.n_sub) * a.T;        // first token of the chunk inside its episode
            const int32_t* list = list_of(l, e);
            // the layer before is complete (group A's first thread has seen it): what this CTA reads of it and writes over it below
            if (bt == 0 && !gave_up) {
                int seen = 0;
                for (uint32_t i = 0; i < SHARED_POLLS; ++i) {
                    asm volatile("ld.acquire.cta.shared::cta.s32 %0, [%1];" : "=r"(seen) : "r"(smem_u32(&sSeen)) : "memory");
                    if (seen > pi || *sAbort) break;
                }
                if (seen <= pi && !*sAbort) { report_timeout(a, sAbort, __LINE__); gave_up = true; }
            }
            ++pi;
            stop = barrier_or(2, 256, gave_up || *sAbort);
            if (stop) break;
            float acc[2][NG][4];
#pragma unroll
            for (int m = 0; m < 2; ++m)
#pragma unroll
                for (int n = 0; n < NG; ++n) acc[m][n][0] = acc[m][n][1] = acc[m][n][2] = acc[m][n][3] = 0.f;
            const int nrd = round_count(w.n, most);
            for (int r = 0; r < nrd; ++r, ++R) {
                int pos, nr;
                round_span(w.n, r, nrd, pos, nr);
                const int tiles = (nr + TN - 1) / TN;
                const int own = j < tiles ? (j + 8 < tiles ? 2 : 1) : 0;               // this CTA's tiles: j, j + 8
                if (bt < own) mbar_arrive_expect_tx(p_full(bt), (uint32_t)np * (CS * TN * 16));
                unsigned char* hb = gbase + LY(off_h);
#pragma unroll 1
                for (int s = 0; s < own || s == 0; ++s) {
                    // ---- owner work: warp i has neuron i of the tile, lane = token pair
                    float h0 = 0.f, h1 = 0.f;
                    if (s < own) {
                        const int qn = (j + 8 * s) * TN + bw;
                        int n = -1;
                        if (qn < nr) {
                            n = w.start + pos + qn;
                            if (list) n = __ldg(list + n);
                            if (n < 0 || n >= a.I) n = -1;         // (reported by the loaders)
                        }
                        float2 ha = make_float2(0.f, 0.f);
                        float2* hap = nullptr;
                        if (EQ4 && anchor_mode != RM_ANCHOR_NONE && n >= 0 && 2 * lane < Te) {
                            hap = reinterpret_cast<float2*>(a.h_anchor + (((size_t)l * a.nb + b) * a.I + n) * a.h_stride + tok0) + lane;
                            if (anchor_mode == RM_ANCHOR_UPDATE) ha = __ldcg(hap);
                        }
                        WAIT(p_full(s), (p_par >> s) & 1u);
                        p_par ^= 1u << s;
                        if (lane < np) {
                            const unsigned char* p = gbase + LY(off_p) + s * P_SLOT + (lane >> 2) * 512 + bw * 64 + (lane & 3) * 16;
                            float4 v = *reinterpret_cast<const float4*>(p);
#pragma unroll
                            for (int k = 1; k < CS; ++k) {
                                const float4 o = *reinterpret_cast<const float4*>(p + k * P_SRC);
                                v.x += o.x; v.y += o.y; v.z += o.z; v.w += o.w;
                            }
                            // GeLU-tanh(g) = g / (1 + exp(-2 z)), z = sqrt(2/pi) (g + 0.044715 g^3)
                            const float e0 = expf(-1.5957691216057308f * (v.x + 0.044715f * v.x * v.x * v.x));
                            const float e1 = expf(-1.5957691216057308f * (v.y + 0.044715f * v.y * v.y * v.y));
                            if (n >= 0 && 2 * lane < Te) h0 = v.x / (1.0f + e0) * v.z;
                            if (n >= 0 && 2 * lane + 1 < Te) h1 = v.y / (1.0f + e1) * v.w;
                        }
                        if (a.record) {
                            float rec = fabsf(h0) + fabsf(h1);
#pragma unroll
                            for (int d = 16; d > 0; d >>= 1) rec += __shfl_xor_sync(0xffffffffu, rec, d);
                            if (lane == 0 && n >= 0) {
                                const float sc = a.record_scale ? a.record_scale[(size_t)l * a.I + n] : 1.f;
                                a.record[(size_t)b * a.rec_b_stride + (size_t)l * a.I + n] = a.record_scale ? rec * sc : rec;
                            }
                        }
                        if (EQ4 && hap) {
                            // Eq. 4: the anchor step retains h; an update step sends its difference from the anchor's h down
                            if (anchor_mode == RM_ANCHOR_WRITE) *hap = make_float2(h0, h1);
                            else { h0 -= ha.x; h1 -= 2 * lane + 1 < Te ? ha.y : 0.f; }
                        }
                    }
                    // every CTA of the cluster is done with the h tile of the round before
                    if (s == 0 && R >= 1) WAIT(h_free, (R - 1) & 1);
                    if (s < own) {
                        // 24 bits in three terms of 8: the first cut off (it must not round up to infinity), the others rounded
                        const float c0 = __uint_as_float(__float_as_uint(h0) & 0xffff0000u), c1 = __uint_as_float(__float_as_uint(h1) & 0xffff0000u);
                        const float f0 = isinf(h0) ? 0.f : h0 - c0, f1 = isinf(h1) ? 0.f : h1 - c1;
                        const __nv_bfloat162 mid = __floats2bfloat162_rn(f0, f1);
                        const float2 mf = __bfloat1622float2(mid);
                        unsigned char* hr = hb + ((j + 8 * s) * TN + bw) * HPITCH + lane * 4;
                        *reinterpret_cast<uint32_t*>(hr) = __float_as_uint(c0) >> 16 | __float_as_uint(c1);
                        *reinterpret_cast<__nv_bfloat162*>(hr + 128) = mid;
                        *reinterpret_cast<__nv_bfloat162*>(hr + 256) = __floats2bfloat162_rn(f0 - mf.x, f1 - mf.y);
                    }
                    if (s == 0 && (tiles & 1) && bt < TN * 24)     // the last stage's second half, which nobody owns
                        *reinterpret_cast<uint4*>(hb + (tiles * TN + bt / 24) * HPITCH + bt % 24 * 16) = make_uint4(0u, 0u, 0u, 0u);
                    fence_proxy_async_smem();
                    stop = barrier_or(2, 256, gave_up || *sAbort);
                    if (bt == 32 && (s + 1 == own || own == 0)) mbar_arrive_expect_tx(h_full, (uint32_t)(tiles - own) * (TN * HPITCH));
                    if (s < own && bt < CS && bt != j && !stop) {
                        const uint32_t from = base + LY(off_h) + (j + 8 * s) * TN * HPITCH;
                        bulk_copy_to_peer(map_to_rank(from, bt), from, TN * HPITCH, map_to_rank(h_full, bt));
                    }
                }
                if (stop) break;
                // ---- down products of the round
                const int ns = (tiles + 1) / 2;
                {
                    int slot = d_slot + lane;                      // lane s looks at stage s, lane 31 at the h tile
                    uint32_t ps = d_pass;
                    if (slot >= NST) { slot -= NST; ++ps; }
                    wait_lanes(lane < ns || lane == 31, lane == 31 ? h_full : d_full(slot), lane == 31 ? R & 1 : ps & 1, __LINE__);
                }
#pragma unroll 1
                for (int s = 0; s < ns; ++s) {
                    const uint32_t ha = h_lane + s * SN * HPITCH, wd = d_lane + d_slot * LY(d_stage);
                    // (a stage's products start from zero and are added in fp32: the tensor core cuts off what does not fit its
                    // accumulator, and over a list of hundreds of neurons that would add up)
                    uint32_t Bw[NG / 2][4];
#pragma unroll
                    for (int n = 0; n < NG / 2; ++n)
                        if (HS || n < cpn) ldm4t(wd + n * 32, Bw[n]);
#pragma unroll
                    for (int m = 0; m < 2; ++m)
                        if (m < mcnt) {
                            uint32_t A[3][4];
#pragma unroll
                            for (int k = 0; k < 3; ++k) ldm4t(ha + k * 128 + m * 32, A[k]);
#pragma unroll
                            for (int n = 0; n < NG / 2; ++n)
                                if (HS || n < cpn) {
                                    float p[2][4];
#pragma unroll
                                    for (int i = 0; i < 2; ++i) p[i][0] = p[i][1] = p[i][2] = p[i][3] = 0.f;
#pragma unroll
                                    for (int k = 2; k >= 0; --k) {
                                        mma16816(p[0], A[k], Bw[n][0], Bw[n][1]);
                                        mma16816(p[1], A[k], Bw[n][2], Bw[n][3]);
                                    }
#pragma unroll
                                    for (int i = 0; i < 2; ++i)
#pragma unroll
                                        for (int q = 0; q < 4; ++q) acc[m][2 * n + i][q] += p[i][q];
                                }
                        }
                    __syncwarp();
                    if (lane == 0) mbar_arrive(d_empty(d_slot));
                    if (++d_slot == NST) { d_slot = 0; ++d_pass; }
                }
                if (lane < CS) arrive_remote(map_to_rank(h_free, lane));
            }
            if (stop) break;
            // ---- the item's sums are complete: this cluster's part of them
            if (w.n > 0) {
                float* pb = a.part + (size_t)(e * parts_max + w.share()) * a.T * H + (size_t)j * Hs;
#pragma unroll
                for (int n = 0; n < NG; ++n) {
                    const int col = (cp0 * 2 + n) * 8 + (lane & 3) * 2;
                    if ((n >> 1) >= cpn || col >= Hs) continue;
#pragma unroll
                    for (int m = 0; m < 2; ++m)
#pragma unroll
                        for (int h = 0; h < 2; ++h) {
                            const int t = (m0 + m) * 16 + h * 8 + (lane >> 2);
                            if (m < mcnt && t < Te) *reinterpret_cast<float2*>(pb + (size_t)t * H + col) = make_float2(acc[m][n][2 * h], acc[m][n][2 * h + 1]);
                        }
                }
            }
            // (the barrier orders every thread's stores before thread 0's release, which is cumulative)
            stop = barrier_or(2, 256, gave_up || *sAbort);
            if (bt == 0 && !stop) red_release_gpu(a.ctrl + ctrl_part(e, j), 1);
        }
        // ---- the rows of the layer: this cluster's share of every item that it takes part in.  (Behind all of the layer's items:
        // a cluster that has finished its part of one waits for the others' with its other products done.)
        for (int e = 0; e < a.B && !stop; ++e) {
            const Item w = items[l * a.B + e];
            if (!w.mine()) continue;
            const int parts = w.parts(), share = w.share(), n4 = Hs / 4, b = episode_of(e), Te = tokens_of(e);
            const size_t lb = (size_t)l * a.nb + b, layer = (size_t)a.nb * a.T_all * H;
            const float* in = l == 0 ? a.r_in : a.r_out;
            if (parts > 1) {
                // (every warp looks for itself: a barrier behind one thread's look is 3 us a step of 12 layers)
                if (lane == 0 && !gave_up) gave_up = counter_wait(a.ctrl + ctrl_part(e, j), w.target() + parts, __LINE__, a, sAbort);
                __syncwarp();
            }
            const float* pe = a.part + (size_t)e * parts_max * a.T * H + (size_t)j * Hs;
            for (int z = bt; z < (Te - share + parts - 1) / parts * n4; z += 256) {
                const int ri = z / n4, k = z - ri * n4, t = share + ri * parts;
                const size_t o = (row0_of(e) + t) * H + (size_t)j * Hs + 4 * k;
                float4 r = make_float4(0.f, 0.f, 0.f, 0.f), y = r, g = make_float4(1.f, 1.f, 1.f, 1.f);
                if (in) r = __ldcg(reinterpret_cast<const float4*>(in + o));
                if (w.n > 0) {
                    const float4* p = reinterpret_cast<const float4*>(pe + (size_t)t * H) + k;
#pragma unroll 1
                    for (int i0 = 0; i0 < parts; i0 += 16) {
                        float4 v[16];
#pragma unroll
                        for (int i = 0; i < 16; ++i) v[i] = i0 + i < parts ? __ldcg(p + (size_t)(i0 + i) * a.T * H / 4) : make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
                        for (int i = 0; i < 16; ++i) { y.x += v[i].x; y.y += v[i].y; y.z += v[i].z; y.w += v[i].w; }
                    }
                }
                if (EQ4) {
                    if (anchor_mode == RM_ANCHOR_WRITE) *reinterpret_cast<float4*>(a.y_anchor + l * layer + o) = y;
                    if (anchor_mode == RM_ANCHOR_UPDATE) {
                        const float4 ya = __ldcg(reinterpret_cast<const float4*>(a.y_anchor + l * layer + o));
                        y.x += ya.x; y.y += ya.y; y.z += ya.z; y.w += ya.w;
                    }
                    if (a.gate) g = __ldg(reinterpret_cast<const float4*>(a.gate + lb * H + (size_t)j * Hs) + k);
                }
                *reinterpret_cast<float4*>(a.r_out + o) = make_float4(fmaf(g.x, y.x, r.x), fmaf(g.y, y.y, r.y), fmaf(g.z, y.z, r.z), fmaf(g.w, y.w, r.w));
            }
            stop = barrier_or(2, 256, gave_up || *sAbort);
            if (bt == 0 && !stop) red_release_gpu(a.ctrl + ctrl_done(e, j), 1);
        }
        }
    }
#undef WAIT
#undef LY
    __syncthreads();
    if (*sAbort) {
        // a wait gave up somewhere: copies into this CTA's shared memory may still be in flight although nobody waits for
        // them any more.  They land within microseconds; idle for longer than that.
        for (int i = 0; i < 64; ++i) __nanosleep(4000);
        __syncthreads();
    }
    cluster_sync();                        // no CTA leaves while a peer may still write into its shared memory
    if (tid == 0 && !epoch_wait(a.ctrl, a.epoch, __LINE__, a, sAbort)) {
        epoch_leave(a.ctrl);
    }
}

// ---- host side
constexpr int SMEM_MAX = 232448 - 256;                             // (the rest for the static part)

template <int HS, int NG, int TS, bool EQ4>
int configure(int smem) {
    RM_CUDA_TRY(cudaFuncSetAttribute(slice_kernel<HS, NG, TS, EQ4>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem));
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
template <int HS, int NG, int TS>
int query(int* out) {
    int rc = configure<HS, NG, TS, false>(SMEM_MAX);
    if (rc == RM_OK) rc = configure<HS, NG, TS, true>(SMEM_MAX);
    if (rc != RM_OK) return rc;
    cudaLaunchConfig_t cfg = {};
    cudaLaunchAttribute at[1];
    cluster_config(cfg, at, 32, SMEM_MAX, nullptr);
    RM_CUDA_TRY(cudaOccupancyMaxActiveClusters(out, slice_kernel<HS, NG, TS, true>, &cfg));
    return RM_OK;
}
template <int HS, int NG, int TS, bool EQ4>
int launch(rm_ctx* ctx, const SArgs& a, int clusters, int smem, cudaStream_t s) {
    cudaLaunchConfig_t cfg = {};
    cudaLaunchAttribute at[2];
    cluster_config(cfg, at, clusters, smem, s);
    at[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[1].val.programmaticStreamSerializationAllowed = 1;
    cfg.numAttrs = ctx->use_pdl ? 2 : 1;
    RM_CUDA_TRY(cudaLaunchKernelEx(&cfg, slice_kernel<HS, NG, TS, EQ4>, a));
    ctx->launches++;
    return RM_OK;
}

inline int tiles_per_owner(int Hs) { return Hs <= 128 ? 2 : 1; }

// The layout with as many stages of each weight ring as fit beside the other buffers, at most MAX_STAGES
Lay layout_of(int Hs) {
    if (Hs == 128) return make_layout(128, 2, EXACT_STAGES);
    int st = MAX_STAGES;
    while (st > 0 && make_layout(Hs, tiles_per_owner(Hs), st).total > SMEM_MAX) --st;
    return make_layout(Hs, tiles_per_owner(Hs), st);
}
static_assert(make_layout(128, 2, EXACT_STAGES).total <= SMEM_MAX, "the buffers of the 128-column slice exceed a CTA's shared memory");
// A chunk of more than 64 tokens is cut into equal parts (multiples of 8 tokens): tokens are independent of one another
void cut_tokens(int T, int& n_sub, int& part) {
    n_sub = (T + 63) / 64;
    part = n_sub == 1 ? T : ((T + n_sub - 1) / n_sub + 7) / 8 * 8;
}

}  // namespace

int rm_slice_init(rm_ctx* ctx) {
    ctx->slice_clusters = 0;
    const int Hs = ctx->g.Hs;
    if (Hs > 256 || layout_of(Hs).stages < 4) return RM_OK;
    int n = 0;
    const int rc = Hs == 128 ? query<128, 4, 2>(&n) : Hs < 128 ? query<0, 4, 2>(&n) : query<0, 8, 1>(&n);
    if (rc == RM_OK) ctx->slice_clusters = n;
    return rc;
}

unsigned long long rm_next_epoch() {
    static std::atomic<unsigned long long> n{(unsigned long long)std::chrono::steady_clock::now().time_since_epoch().count() << 20 | 1u};
    return n.fetch_add(2);
}

bool rm_slice_supported(const rm_ctx* ctx, int B, int T, bool record) {
    if (ctx->slice_clusters <= 0 || T < 1 || B < 1) return false;
    int n_sub, part;
    cut_tokens(T, n_sub, part);
    return ctx->g.L <= MAXL && !(record && n_sub > 1);
}

size_t rm_slice_workspace_bytes(const rm_ctx* ctx, int B, int T) {
    if (ctx->slice_clusters <= 0) return 0;
    int n_sub, part;
    cut_tokens(T, n_sub, part);
    const int e = B * n_sub < GROUP ? B * n_sub : GROUP;
    return ctrl_bytes(GROUP) + (size_t)e * ctx->slice_clusters * part * ctx->g.H * sizeof(float);
}

int rm_launch_step_slice(rm_ctx* ctx, const rm_step_args& sa, cudaStream_t s) {
    const rm_geom& g = ctx->g;
    SArgs a{};
    int n_sub, part;
    cut_tokens(sa.T, n_sub, part);
    for (int l = 0; l < sa.L; ++l) a.packed[l] = static_cast<const __nv_bfloat16*>(sa.packed_layers[l]);
    a.r_in = sa.r_in ? sa.r_in : sa.r;
    a.r_out = sa.r;
    a.x_ext = static_cast<const __nv_bfloat16*>(sa.x_ext);
    if (sa.x_ext) a.r_in = sa.r_in;
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
    a.part = reinterpret_cast<float*>(reinterpret_cast<char*>(sa.ctrl) + ctrl_bytes(GROUP));
    a.status = ctx->d_status;
    a.L = sa.L;
    a.T = part;
    a.I = g.I;
    a.Hs = g.Hs;
    a.n_sub = n_sub;
    a.nb = sa.B;
    a.T_all = sa.T;
    a.anchor_mode = sa.anchor_mode;
    a.y_anchor = sa.y_anchor;
    a.h_anchor = sa.h_anchor;
    a.h_stride = sa.h_stride;
    a.gate = sa.gate;
    int nc = ctx->slice_clusters;
    if (ctx->max_clusters_override > 0 && ctx->max_clusters_override < nc) nc = ctx->max_clusters_override;
    const bool eq4 = sa.anchor_mode != RM_ANCHOR_NONE || sa.gate != nullptr;
    a.lay = layout_of(g.Hs);
    const int smem = a.lay.total;
    for (a.e0 = 0; a.e0 < sa.B * n_sub; a.e0 += GROUP) {
        a.B = sa.B * n_sub - a.e0 < GROUP ? sa.B * n_sub - a.e0 : GROUP;
        a.epoch = rm_next_epoch();
        int rc;
        if (g.Hs == 128) rc = eq4 ? launch<128, 4, 2, true>(ctx, a, nc, smem, s) : launch<128, 4, 2, false>(ctx, a, nc, smem, s);
        else if (g.Hs < 128) rc = eq4 ? launch<0, 4, 2, true>(ctx, a, nc, smem, s) : launch<0, 4, 2, false>(ctx, a, nc, smem, s);
        else rc = eq4 ? launch<0, 8, 1, true>(ctx, a, nc, smem, s) : launch<0, 8, 1, false>(ctx, a, nc, smem, s);
        if (rc != RM_OK) return rc;
    }
    return RM_OK;
}

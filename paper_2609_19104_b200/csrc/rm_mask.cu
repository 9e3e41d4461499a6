// rm_mask_compact: important-neuron selection and stream compaction.
//
// A list is one (layer, episode) pair.  Every record of the list is reduced to a per-neuron flag by the chosen
// rule (boolean, score > threshold, or the k largest scores with ties going to the lower index -- the ranking of
// Eq. 1's contribution scores), the flags are combined by a vote, and the surviving neurons are written in
// ascending order with warp-ballot / popc prefix sums.
//
// The call is a chain of latencies (a list is a few 10 KB; HBM time is below a microsecond), so the kernel is built
// to keep that chain short:
//   - a thread keeps the keys of its neurons in registers (neuron n belongs to thread n mod 1024, chunk n / 1024), so
//     a record is read once, with all loads in flight together;
//   - exact top-k narrows an interval of order-preserving integer keys: the span between the smallest and the largest key
//     is cut into 2048 equal bins, one histogram pass finds the bin that holds the k-th key, and the next pass cuts
//     that bin again.  Bins that follow the data's own span spread the counts (fixed digits put most activations of a
//     layer into a handful of bins, whose shared-memory adds then queue up), after the first pass only a few keys
//     are left, and the search ends as soon as the whole bin belongs to the result: two or three passes;
//   - the records of a vote or a group are independent until their flags are counted: they go to the CTAs of a cluster,
//     which send their flag words to the first CTA through distributed shared memory;
//   - one scan per ordered ranking, over the (chunk, warp) counts, instead of one per chunk.
//   - one long record is divided over the CTAs of a cluster, which add up their bins.
// Measured, 18 lists, us per call back to back: 3-of-4 vote of top-615 sets of 4096: 29.9 -> 7.7; top-3277 of 16384: 26.8 -> 9.7 to 10.7
// (14.6 with one CTA per list).
#include "rm_common.cuh"
#include "rm_sm100.cuh"

namespace {

constexpr int MASK_THREADS = 1024;
constexpr int MASK_MAX_RECORDS = 16;
constexpr int MASK_BINS = 2 * MASK_THREADS;
constexpr int MASK_MAX_CLUSTER = 8;

struct MaskParams {
    const void* rec[MASK_MAX_RECORDS];
    int W, kind, reduce, k, min_votes, scale_per_list, I;
    int cluster;               // CTAs per list: either CTA r takes the records r, r + cluster, ...
    int segment;               // ... or (not 0) the neurons [r * segment, (r + 1) * segment) of the only record
    int planes;                // bits of a CTA's vote count
    float threshold;
    const float* scale;
    int64_t stride;
    int32_t* idx_out;
    int32_t* count_out;
    int* status;
};

struct MaskShared {
    unsigned hist[2][MASK_BINS];           // counts of alternate narrowing steps
    int4 xch[2][MASK_MAX_CLUSTER];         // alternate exchanges between the CTAs of a divided list
    unsigned red[3][32];       // per-warp minima, maxima, counts
    int warp_tot[32];
    unsigned bin;              // result of one narrowing step: the bin, its count, the elements above it
    int bin_count, bin_above;
};

// Order-preserving key: larger float -> larger key; -0 == +0; NaN (key 1) below every number; 0 stands for "not there".
__device__ __forceinline__ unsigned key_of(float s) {
    const unsigned u = __float_as_uint(s + 0.0f);  // (-0 + 0 = +0)
    const unsigned k = u ^ ((unsigned)((int)u >> 31) | 0x80000000u);
    return s == s ? k : 1u;
}

__device__ __forceinline__ float load_score(const MaskParams& p, int w, int list, int n) {
    float s = static_cast<const float*>(p.rec[w])[(size_t)list * p.I + n];
    if (p.scale) s *= p.scale[(p.scale_per_list ? (size_t)list * p.I : 0) + n];
    return s;
}

// inclusive prefix sum over the CTA's threads in thread order; `total`: the sum over all threads
__device__ __forceinline__ int block_scan(int v, MaskShared& sh, int& total) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    int incl = v;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
        const int o = __shfl_up_sync(0xffffffffu, incl, d);
        if (lane >= d) incl += o;
    }
    if (lane == 31) sh.warp_tot[warp] = incl;
    __syncthreads();
    const int wt = sh.warp_tot[lane];
    int wincl = wt;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
        const int o = __shfl_up_sync(0xffffffffu, wincl, d);
        if (lane >= d) wincl += o;
    }
    total = __shfl_sync(0xffffffffu, wincl, 31);
    return incl + __shfl_sync(0xffffffffu, wincl - wt, warp);
}

// E > 0: up to E keys per thread, in registers.  E == 0: any I, keys are computed again from the records whenever they
// are looked at (lists too long for the registers).  Flags travel as words of 32 neurons, word c * 32 + warp for a
// warp's neurons of chunk c, so that everything done per flag costs a thread per word, not per neuron.
template <int E>
struct MaskList {
    MaskShared& sh;
    int* cnt;                  // [words] exclusive prefixes of one ordered ranking
    int lane, warp, nch;
    int n0, n_end;             // this CTA's neurons
    int S, ss, turn;           // CTAs that divide the list (1: this CTA has all of it), this one's number, exchanges so far
    unsigned key[E ? E : 1];

    template <class F>
    __device__ __forceinline__ void chunks(F f) {
        if (E) {
#pragma unroll
            for (int c = 0; c < (E ? E : 1); ++c) if (c < nch) f(c);
        } else {
            for (int c = 0; c < nch; ++c) f(c);
        }
    }
    __device__ __forceinline__ int neuron(int c) const { return n0 + c * MASK_THREADS + (int)threadIdx.x; }
    __device__ __forceinline__ bool in(int c) const { return neuron(c) < n_end; }

    // Every CTA of a divided list gets every CTA's (a, b, c); all threads hold the values to send.  A barrier of the cluster.
    __device__ __forceinline__ const int4* exchange(int a, int b, int c) {
        int4* box = sh.xch[turn++ & 1];
        if (warp == 0 && lane < S)
            sm100::st_cluster_v4u(sm100::map_to_rank(sm100::smem_u32(box + ss), lane), make_uint4((unsigned)a, (unsigned)b, (unsigned)c, 0u));
        sm100::cluster_sync();
        return box;
    }
    // sum of the v of the CTAs in front; `total`: of all
    __device__ __forceinline__ int exchange_ranks(int v, int& total) {
        if (S == 1) { total = v; return 0; }
        const int4* box = exchange(v, 0, 0);
        int front = 0;
        total = 0;
        for (int r = 0; r < S; ++r) {
            const int o = box[r].x;
            front += r < ss ? o : 0;
            total += o;
        }
        return front;
    }
    template <class P>
    __device__ __forceinline__ void flag_words(unsigned* words, P pred) {
        chunks([&](int c) {
            const unsigned b = __ballot_sync(0xffffffffu, pred(c));
            if (lane == 0) words[c * 32 + warp] = b;
        });
    }

    // cnt[e] = number of this CTA's flags in the words before word e (behind a barrier on both sides); returns the total
    __device__ __forceinline__ int ordered_ranks(const unsigned* words) {
        const int n = nch * 32, m = E ? 1 : (n + MASK_THREADS - 1) / MASK_THREADS, e0 = (int)threadIdx.x * m;
        int mine = 0, total;
        for (int e = e0; e < e0 + m && e < n; ++e) mine += __popc(words[e]);
        int run = block_scan(mine, sh, total) - mine;
        for (int e = e0; e < e0 + m && e < n; ++e) {
            cnt[e] = run;
            run += __popc(words[e]);
        }
        __syncthreads();
        return total;
    }

    // Writes the flag words of the top min(k, elements there) elements; ties at the last key go to the lower index.
    // get(c): the key of this thread's element of chunk c, 0 if it is not there.  Ends with a barrier.
    template <class K>
    __device__ __forceinline__ void topk(int k, K get, unsigned* words) {
        unsigned lo = 0xffffffffu, hi = 0u, nv = 0u;
        chunks([&](int c) {
            const unsigned kv = get(c), low = kv - 1u;             // (0 becomes the largest)
            lo = low < lo ? low : lo;
            hi = kv > hi ? kv : hi;
            nv += kv != 0u;
        });
        lo = __reduce_min_sync(0xffffffffu, lo);
        hi = __reduce_max_sync(0xffffffffu, hi);
        nv = __reduce_add_sync(0xffffffffu, nv);
        if (lane == 0) { sh.red[0][warp] = lo; sh.red[1][warp] = hi; sh.red[2][warp] = nv; }
        __syncthreads();
        lo = __reduce_min_sync(0xffffffffu, sh.red[0][lane]) + 1u;
        hi = __reduce_max_sync(0xffffffffu, sh.red[1][lane]);
        int there = (int)__reduce_add_sync(0xffffffffu, sh.red[2][lane]);
        if (S > 1) {
            const int4* box = exchange((int)lo, (int)hi, there);
            there = 0;
            for (int r = 0; r < S; ++r) {
                const int4 o = box[r];
                if (o.z == 0) continue;            // (a CTA without elements sends no range)
                lo = there == 0 || (unsigned)o.x < lo ? (unsigned)o.x : lo;
                hi = there == 0 || (unsigned)o.y > hi ? (unsigned)o.y : hi;
                there += o.z;
            }
        }
        if (k <= 0 || there == 0) {
            flag_words(words, [&](int) { return false; });
            __syncthreads();
            return;
        }
        // the wanted key lies in [lo, hi], which holds `held` elements; it is the rem-th largest of them
        int rem = k < there ? k : there, held = there, last = -1;
        for (int step = 0; rem < held && lo < hi; ++step) {
            unsigned* hist = sh.hist[step & 1];
            const unsigned width = hi - lo;
            const int bits = 32 - __clz(width), shift = bits > 11 ? bits - 11 : 0;
            chunks([&](int c) {
                const unsigned d = get(c) - lo;                    // (not there: 2^32 - lo, beyond every width)
                if (d <= width) atomicAdd(&hist[d >> shift], 1u);
            });
            if (S > 1) sm100::cluster_sync();
            else __syncthreads();
            // thread t looks at the bins 2047 - 2 t and 2046 - 2 t: a prefix sum from the top
            const int pair = MASK_THREADS - 1 - (int)threadIdx.x;
            uint2 cc = reinterpret_cast<uint2*>(hist)[pair];
            if (S > 1) {                           // the bins of the other CTAs
                const uint32_t at = sm100::smem_u32(hist) + 8u * (unsigned)pair;
                for (int r = 1; r < S; ++r) {
                    uint2 o;
                    const int peer = ss + r < S ? ss + r : ss + r - S;
                    asm volatile("ld.shared::cluster.v2.u32 {%0, %1}, [%2];" : "=r"(o.x), "=r"(o.y) : "r"(sm100::map_to_rank(at, peer)) : "memory");
                    cc.x += o.x;
                    cc.y += o.y;
                }
            }
            // the bins of the step before have been read by everybody: ready for the step after
            reinterpret_cast<uint2*>(sh.hist[(step & 1) ^ 1])[pair] = make_uint2(0u, 0u);
            const int c1 = (int)cc.y, c0 = (int)cc.x;
            int total;
            const int above = block_scan(c1 + c0, sh, total) - c1 - c0;
            if (above < rem && rem <= above + c1 + c0) {
                const bool first = rem <= above + c1;
                sh.bin = (unsigned)(MASK_BINS - 2 - 2 * (int)threadIdx.x) + (first ? 1u : 0u);
                sh.bin_count = first ? c1 : c0;
                sh.bin_above = first ? above : above + c1;
            }
            __syncthreads();
            lo += sh.bin << shift;
            const unsigned top = lo + ((1u << shift) - 1u);
            hi = top < hi ? top : hi;
            held = sh.bin_count;
            rem -= sh.bin_above;                   // (the next step writes these two barriers further on)
            last = step & 1;
        }
        // leave both histograms empty (the bins of the last step: read by everybody behind the next barrier of the callers)
        if (last >= 0 && S == 1) reinterpret_cast<uint2*>(sh.hist[last])[threadIdx.x] = make_uint2(0u, 0u);
        if (rem == held) {                         // everything from lo upwards
            flag_words(words, [&](int c) { return get(c) >= lo; });
            __syncthreads();
            return;
        }
        // more elements equal to the last key than are wanted: the first `rem` of them in neuron order
        flag_words(words, [&](int c) { return get(c) == lo; });
        __syncthreads();
        int total;
        const int front = exchange_ranks(ordered_ranks(words), total);
        flag_words(words, [&](int c) {
            const unsigned kv = get(c), b = words[c * 32 + warp];
            __syncwarp();
            return kv > lo || (kv == lo && front + cnt[c * 32 + warp] + __popc(b & ((1u << lane) - 1u)) < rem);
        });
        __syncthreads();
    }
};

template <int E>
__global__ void __launch_bounds__(MASK_THREADS, 1) mask_compact_kernel(const __grid_constant__ MaskParams p) {
    extern __shared__ __align__(16) unsigned words[];              // see below
    __shared__ __align__(16) MaskShared sh;
    const int I = p.I, C = p.cluster;
    const int rank = C > 1 ? (int)sm100::cluster_ctarank() : 0, list = (int)blockIdx.x / C;
    const bool divided = p.segment != 0;
    const int n0 = divided ? rank * p.segment : 0, n_end = divided && n0 + p.segment < I ? n0 + p.segment : I;
    const int nch = ((divided ? p.segment : I) + MASK_THREADS - 1) / MASK_THREADS, nw = nch * 32;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    // words: [nw] counts of an ordered ranking | [nw] flags of the current record, in the end the kept elements | [planes][nw]
    // bit planes of this CTA's vote counts | first CTA: [cluster - 1][planes][nw] those of the others
    unsigned* flags = words + nw;
    unsigned* plane = words + 2 * nw;
    MaskList<E> m{sh, reinterpret_cast<int*>(words), lane, warp, nch, n0, n_end, divided ? C : 1, divided ? rank : 0, 0, {}};

    if (C > 1) sm100::cluster_arrive();            // (waited for before the first word goes to another CTA)
    reinterpret_cast<uint4*>(sh.hist)[threadIdx.x] = make_uint4(0u, 0u, 0u, 0u);
    for (int e = threadIdx.x; e < p.planes * nw; e += MASK_THREADS) plane[e] = 0u;
    // programmatic dependent launch: the records read below may come from the kernel in front of this one; a kernel launched
    // behind this one may start its prologue once they are there (weights that it fetches ahead would otherwise hold up the
    // kernel in front: Context Cache, drift 6 us instead of 2)
    sm100::pdl_wait();
    sm100::pdl_launch_dependents();
    __syncthreads();

    const bool single = p.W == 1 && p.reduce != RM_REDUCE_GROUP;  // one record, no vote: its flags are the result
    if (divided) sm100::cluster_wait();            // every CTA of the cluster has started
    for (int w = divided ? 0 : rank; w < p.W; w += C) {
        if (p.kind == RM_SRC_BOOL_U8) {
            const unsigned char* src = static_cast<const unsigned char*>(p.rec[w]) + (size_t)list * I;
            if (E) m.chunks([&](int c) { m.key[E ? c : 0] = m.in(c) ? src[m.neuron(c)] : 0; });
            m.flag_words(flags, [&](int c) { return (E ? m.key[E ? c : 0] : m.in(c) ? src[m.neuron(c)] : 0) != 0; });
            __syncthreads();
        } else {
            auto score = [&](int c) { return m.in(c) ? load_score(p, w, list, m.neuron(c)) : __int_as_float(0x7fc00000); };
            if (E) m.chunks([&](int c) { m.key[E ? c : 0] = __float_as_uint(score(c)); });
            if (p.reduce == RM_REDUCE_THRESHOLD) {
                m.flag_words(flags, [&](int c) { return (E ? __uint_as_float(m.key[E ? c : 0]) : score(c)) > p.threshold; });
                __syncthreads();
            } else {                                // TOPK, and the per-record stage of GROUP
                auto key = [&](int c, float s) { return m.in(c) ? key_of(s) : 0u; };
                if (E) m.chunks([&](int c) { m.key[E ? c : 0] = key(c, __uint_as_float(m.key[E ? c : 0])); });
                m.topk(p.k, [&](int c) { return E ? m.key[E ? c : 0] : key(c, score(c)); }, flags);
            }
        }
        if (!single) {                              // one more vote: a binary counter per element, one bit per plane
            for (int e = threadIdx.x; e < nw; e += MASK_THREADS) {
                unsigned carry = flags[e];
                for (int b = 0; b < p.planes; ++b) {
                    const unsigned old = plane[b * nw + e];
                    plane[b * nw + e] = old ^ carry;
                    carry &= old;
                }
            }
            __syncthreads();
        }
    }
    if (C > 1 && !divided) {
        sm100::cluster_wait();                     // every CTA of the cluster has started
        const int n = p.planes * nw;
        if (rank != 0) {
            const uint32_t dst = sm100::map_to_rank(sm100::smem_u32(plane + rank * n), 0);
            for (int e = threadIdx.x; e < n; e += MASK_THREADS)
                asm volatile("st.shared::cluster.u32 [%0], %1;" ::"r"(dst + 4u * e), "r"(plane[e]) : "memory");
        }
        sm100::cluster_arrive();
        sm100::cluster_wait();
        if (rank != 0) return;
    }
    if (!single) {
        for (int e = threadIdx.x; e < nw; e += MASK_THREADS) {
            unsigned t[5] = {0u, 0u, 0u, 0u, 0u};  // the votes of 32 elements, up to 16 each
            for (int r = 0; r < C; ++r)
                for (int b = 0; b < p.planes; ++b) {
                    unsigned carry = plane[(r * p.planes + b) * nw + e];
#pragma unroll
                    for (int i = 0; i < 5; ++i) {
                        const unsigned add = i >= b ? carry : 0u, old = t[i];
                        t[i] = old ^ add;
                        carry = i >= b ? old & add : carry;
                    }
                }
            unsigned gt = 0u, eq = 0xffffffffu;
#pragma unroll
            for (int i = 4; i >= 0; --i) {
                if ((p.min_votes >> i) & 1) eq &= t[i];
                else { gt |= eq & t[i]; eq &= ~t[i]; }
            }
            flags[e] = gt | eq;
        }
        __syncthreads();
    }
    if (p.reduce == RM_REDUCE_GROUP) {
        // rank the union of the per-record sets (the flags, min_votes being 1) by the summed score and keep the top k
        auto key_sum = [&](int c) {
            if (!((flags[c * 32 + warp] >> lane) & 1u)) return 0u;
            float s = 0.0f;
            for (int w = 0; w < p.W; ++w) s += load_score(p, w, list, m.neuron(c));
            return key_of(s);
        };
        if (E) m.chunks([&](int c) { m.key[E ? c : 0] = key_sum(c); });
        __syncwarp();
        // (without kept keys the union has to outlive the flags that are written: it stays in the first plane)
        if (!E) {
            for (int e = threadIdx.x; e < nw; e += MASK_THREADS) plane[e] = 0u;
            __syncthreads();
            m.topk(p.k, key_sum, plane);
            for (int e = threadIdx.x; e < nw; e += MASK_THREADS) flags[e] = plane[e];
            __syncthreads();
        } else {
            m.topk(p.k, [&](int c) { return m.key[E ? c : 0]; }, flags);
        }
    }

    // ordered compaction of the kept elements
    int32_t* out = p.idx_out + (size_t)list * p.stride;
    int total;
    const int front = m.exchange_ranks(m.ordered_ranks(flags), total);
    const bool fits = total <= p.stride;
    m.chunks([&](int c) {
        const unsigned b = flags[c * 32 + warp];
        const int pos = front + reinterpret_cast<int*>(words)[c * 32 + warp] + __popc(b & ((1u << lane) - 1u));
        if (((b >> lane) & 1u) && (fits || pos < p.stride)) out[pos] = m.neuron(c);
    });
    if (threadIdx.x == 0 && (rank == 0 || !divided)) {
        if (!fits) rm_set_status(p.status, RM_ERR_INDEX);
        p.count_out[list] = fits ? total : (int)p.stride;
    }
}

template <int E>
int launch_mask(rm_ctx* ctx, const MaskParams& p, int n_lists, size_t smem, cudaStream_t s) {
    static rm_smem_configured configured = {};
    if (smem + sizeof(MaskShared) > 48 * 1024) {              // (48 KB, the static part included, need no asking)
        const int set = configured.raise(ctx->device, (int)smem, [&] { return rm_set_smem(mask_compact_kernel<E>, (int)smem); });
        if (set != RM_OK) return set;
    }
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(n_lists * p.cluster);
    cfg.blockDim = dim3(MASK_THREADS);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cudaLaunchAttribute at[2];
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = ctx->use_pdl;
    at[1].id = cudaLaunchAttributeClusterDimension;
    at[1].val.clusterDim.x = p.cluster;
    at[1].val.clusterDim.y = 1;
    at[1].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = p.cluster > 1 ? 2 : 1;
    RM_CUDA_TRY(cudaLaunchKernelEx(&cfg, mask_compact_kernel<E>, p));
    ctx->launches++;
    return RM_OK;
}

}  // namespace

int rm_launch_mask_compact(rm_ctx* ctx, const rm_mask_src* src, int32_t* idx_out, int32_t* count_out,
                           int64_t stride, cudaStream_t s) {
    MaskParams p{};
    for (int w = 0; w < src->n_records; ++w) p.rec[w] = src->records[w];
    p.W = src->n_records;
    p.kind = src->kind;
    p.reduce = src->reduce;
    p.k = src->k;
    p.min_votes = src->reduce == RM_REDUCE_GROUP ? 1 : src->min_votes;
    p.scale_per_list = src->scale_per_list;
    p.I = src->I;
    p.threshold = src->threshold;
    p.scale = src->scale;
    p.stride = stride;
    p.idx_out = idx_out;
    p.count_out = count_out;
    p.status = ctx->d_status;
    if ((size_t)src->I > 200 * 1024) return RM_ERR_UNSUPPORTED;
    if (src->n_lists <= 0) return RM_OK;
    const int nch = (src->I + MASK_THREADS - 1) / MASK_THREADS;
    // Work to CTAs (a CTA of 1024 threads fills an SM; all lists' CTAs should fit the SMs at once).  One record of more than
    // 4096 scores or flags: its neurons are divided, 4096 or more to a CTA -- every instruction per neuron costs an SM 8
    // clocks per 1024 of them, and joining the CTAs' counts costs ~0.5 us per narrowing step.
    // Several records: as many CTAs per list as there are records, while they fit.  Boolean and threshold records are a load
    // and a compare each, not worth a cluster of their own; nor are keys that have to be read again on every pass.
    p.cluster = 1;
    const int fit = ctx->sm_count / src->n_lists;
    if (p.W == 1 && p.reduce != RM_REDUCE_GROUP && nch > 4) {
        while (p.cluster < MASK_MAX_CLUSTER && 4 * p.cluster < nch && 2 * p.cluster <= fit) p.cluster *= 2;
        if (p.cluster > 1) p.segment = (nch + p.cluster - 1) / p.cluster * MASK_THREADS;
    } else if (src->kind == RM_SRC_SCORE_F32 && src->reduce != RM_REDUCE_THRESHOLD && nch <= 16) {
        while (p.cluster < MASK_MAX_CLUSTER && p.cluster < p.W && 2 * p.cluster <= fit) p.cluster *= 2;
    }
    const int nch_cta = p.segment ? p.segment / MASK_THREADS : nch;
    const int per_cta = p.segment ? 1 : (p.W + p.cluster - 1) / p.cluster;
    p.planes = 1;
    while ((1 << p.planes) <= per_cta) ++p.planes;
    const size_t smem = (size_t)nch_cta * 32 * sizeof(unsigned) * (2 + p.planes * (p.segment ? 1 : p.cluster));
    if (nch_cta <= 1) return launch_mask<1>(ctx, p, src->n_lists, smem, s);
    if (nch_cta <= 4) return launch_mask<4>(ctx, p, src->n_lists, smem, s);
    if (nch_cta <= 16) return launch_mask<16>(ctx, p, src->n_lists, smem, s);
    return launch_mask<0>(ctx, p, src->n_lists, smem, s);
}

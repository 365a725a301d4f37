// Keep-index sampler (Sec. 3.2.1 index sets; Sec. 4 random and grid-wise masks).
//
// Random mode: one thread block per sample, or a cluster of blocks for large maps.  It finds the K-th smallest 64-bit score
// (philox word << 32 | position) and emits the kept positions in ascending order.  Bound by the chain of barriers, not by
// work, so the chain is short: one histogram of the words' top eight bits names the bin that holds the K-th smallest; that
// bin's words (about N / 256) are collected and each is ranked against the others, which gives the threshold word; each
// warp then owns a contiguous stretch of positions, so one scan of the warps' counts places every kept position.  (Should
// a bin ever hold more words than the list, the next eight bits are taken, as often as needed.)  Four passes of eight bits
// and a scan for every 2048 positions took 6.1 us for 128 x 196 positions and 16.6 us for 2 x 66800 back to back; now 1.1 us
// and 2.7 us (the words are drawn while the kernel before drains).
// Grid mode: everything has a closed form - a sample's offset from the counts of the samples before it, a kept position's place
// from the kept positions in the rows above and to its left - so each block writes a stretch of one map without a scan, and a
// large map is spread over as many blocks as the samples leave room for (a predicate and an ordered compaction by one block a
// sample, back to back: 64 maps of 56 x 56 3.9 us, 2 of 200 x 334 31.5; now 2.2 and 2.1).
#include "row_copy.cuh"
#include "sbp_common.cuh"

namespace sbp {
namespace {

constexpr int kSampThreads = 512;
constexpr int kSampWarps = kSampThreads / 32;

__device__ __forceinline__ uint32_t warp_incl_scan(uint32_t v, int lane) {
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
        uint32_t n = __shfl_up_sync(0xffffffffu, v, d);
        if (lane >= d) v += n;
    }
    return v;
}

// Exclusive prefix over the block of per-thread counts; returns (exclusive prefix, block total).
template <int kThreads>
__device__ __forceinline__ uint2 block_excl_scan(uint32_t v, uint32_t* warp_sums) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const uint32_t incl = warp_incl_scan(v, lane);
    if (lane == 31) warp_sums[warp] = incl;
    __syncthreads();
    uint32_t ws = (lane < kThreads / 32) ? warp_sums[lane] : 0u;
    const uint32_t ws_incl = warp_incl_scan(ws, lane);
    const uint32_t total = __shfl_sync(0xffffffffu, ws_incl, kThreads / 32 - 1);
    const uint32_t warp_base = __shfl_sync(0xffffffffu, ws_incl - ws, warp);
    __syncthreads();
    return make_uint2(warp_base + incl - v, total);
}

// ---- clusters: one sample spread over C thread blocks, each with a contiguous slice of the positions ----
__device__ __forceinline__ uint32_t cluster_rank() {
    uint32_t r;
    asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
    return r;
}
__device__ __forceinline__ void cluster_sync() {
    asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}
__device__ __forceinline__ uint32_t cluster_load(const uint32_t* local_ptr, uint32_t rank) {
    const uint32_t a = (uint32_t)__cvta_generic_to_shared(local_ptr);
    uint32_t ra, v;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(ra) : "r"(a), "r"(rank));
    asm volatile("ld.shared::cluster.u32 %0, [%1];" : "=r"(v) : "r"(ra) : "memory");
    return v;
}

// Words of the chosen bin that are ranked directly.  Every block of a cluster ranks them all, n x n comparisons; from some 400 on eight
// more bits of the words are the cheaper way (32 samples of 200000 positions, 781 words in a bin: 88 us, now 31).
constexpr uint32_t kMaxListed = 384;

struct RandomShared {
    // Two histograms used alternately: the one a pass clears was last read by other blocks of a cluster two passes earlier,
    // before the barrier of the pass in between, so one barrier per pass is enough.
    uint32_t hist[2][256];
    uint32_t listed[kMaxListed];           // this block's words of the chosen bin
    uint32_t all_listed[kMaxListed];       // a cluster's: those of all its blocks
    uint32_t n_listed;
    uint32_t warp_sums[32], warp_ties[32];
    uint32_t bin, below, in_bin;           // the chosen bin, words in lower bins, words in it
    uint32_t threshold, less, equal;       // the K-th smallest word; listed words below it, equal to it
    uint32_t slice_counts[2];              // positions of this slice below / equal to the threshold
};

// C blocks a sample.  kThreads: 128 for small maps (fewer warps to bring to each barrier), 512 otherwise, 1024 for a few large ones.  cache_groups: how
// many groups of four words the dynamic shared memory holds (0: every look at a word computes it again).
template <int C, int kThreads>
__global__ void __launch_bounds__(kThreads)
sample_keep_random_kernel(uint32_t N, uint32_t K, uint32_t k0, uint32_t k1, uint32_t step,
                          uint32_t first_sample, int share_mask, uint32_t cache_groups,
                          int32_t* __restrict__ keep_rows, int32_t* __restrict__ keep_offsets) {
    extern __shared__ uint4 word_cache[];
    __shared__ RandomShared sh;
    pdl_launch_dependents();
    const uint32_t rank = C > 1 ? cluster_rank() : 0u;
    const uint32_t b = blockIdx.x / C;
    const uint32_t gid = share_mask ? 0u : first_sample + b;
    const uint32_t groups = (N + 3u) >> 2;
    const uint32_t per = (groups + C - 1) / C;
    const uint32_t g_begin = rank * per < groups ? rank * per : groups;
    const uint32_t g_end = (g_begin + per < groups) ? g_begin + per : groups;
    const int64_t row_base = (int64_t)b * N;
    const bool cached = cache_groups >= per;
    int32_t* out = keep_rows + (int64_t)b * K;
    auto sync_all = [] {
        if constexpr (C > 1) cluster_sync();
        else __syncthreads();
    };
    auto words_of = [&](uint32_t q) {
        if (!cached) return philox4x32_10(q, gid, step, 0u, k0, k1);
        const uint4 v = word_cache[q - g_begin];
        PhiloxWords pw;
        pw.w[0] = v.x; pw.w[1] = v.y; pw.w[2] = v.z; pw.w[3] = v.w;
        return pw;
    };

    if (C == 1 && K >= N) {                                  // nothing to choose (small maps; larger ones do not come here)
        pdl_wait();
        if (threadIdx.x == 0) {
            keep_offsets[b + 1] = (int32_t)((b + 1) * (int64_t)N);
            if (b == 0) keep_offsets[0] = 0;
        }
        for (uint32_t n = threadIdx.x; n < N; n += kThreads) out[n] = (int32_t)(row_base + n);
        return;
    }
    uint32_t threshold, ties;                                // kept: word < threshold, and the first `ties` equal to it
    bool all_ties;
    {
        uint32_t prefix = 0, known = 0, remaining = K;
        for (int shift = 24, pass = 0;; shift -= 8, ++pass) {
            uint32_t* hist = sh.hist[pass & 1];
            for (int i = threadIdx.x; i < 256; i += kThreads) hist[i] = 0;
            __syncthreads();
            for (uint32_t q = g_begin + threadIdx.x; q < g_end; q += kThreads) {
                PhiloxWords pw;
                if (pass == 0) {
                    pw = philox4x32_10(q, gid, step, 0u, k0, k1);
                    if (cached) word_cache[q - g_begin] = make_uint4(pw.w[0], pw.w[1], pw.w[2], pw.w[3]);
                } else {
                    pw = words_of(q);
                }
#pragma unroll
                for (int e = 0; e < 4; ++e)
                    if (4u * q + e < N && (pw.w[e] & known) == prefix) atomicAdd(&hist[(pw.w[e] >> shift) & 0xffu], 1u);
            }
            sync_all();                                      // every slice's histogram is complete
            // running count over the 256 bins; the bin where it crosses `remaining` is the one
            constexpr int kBins = kThreads >= 256 ? 1 : 256 / kThreads;
            uint32_t cnt[kBins], mine = 0;
#pragma unroll
            for (int i = 0; i < kBins; ++i) {
                const int bin = threadIdx.x * kBins + i;
                cnt[i] = 0;
                if (bin < 256) {
                    if constexpr (C > 1) {
#pragma unroll
                        for (uint32_t r = 0; r < (uint32_t)C; ++r) cnt[i] += cluster_load(&hist[bin], r);
                    } else {
                        cnt[i] = hist[bin];
                    }
                }
                mine += cnt[i];
            }
            uint32_t before = block_excl_scan<kThreads>(mine, sh.warp_sums).x;
#pragma unroll
            for (int i = 0; i < kBins; ++i) {
                if (before < remaining && remaining <= before + cnt[i]) {
                    sh.bin = threadIdx.x * kBins + i;
                    sh.below = before;
                    sh.in_bin = cnt[i];
                }
                before += cnt[i];
            }
            if (threadIdx.x == 0) sh.n_listed = 0;
            __syncthreads();
            prefix |= sh.bin << shift;
            known |= 0xffu << shift;
            remaining -= sh.below;
            const uint32_t in_bin = sh.in_bin;
            if (in_bin > kMaxListed && shift > 0) {
                __syncthreads();                             // the bin is read before the next pass rewrites it
                continue;
            }
            if (in_bin > kMaxListed) {                       // more equal words than that
                threshold = prefix;
                ties = remaining;
                all_ties = in_bin == remaining;
                break;
            }
            // the bin's words, ranked against each other: the remaining-th smallest is the threshold
            for (uint32_t q = g_begin + threadIdx.x; q < g_end; q += kThreads) {
                const PhiloxWords pw = words_of(q);          // (its own thread wrote it to the cache)
#pragma unroll
                for (int e = 0; e < 4; ++e)
                    if (4u * q + e < N && (pw.w[e] & known) == prefix) sh.listed[atomicAdd(&sh.n_listed, 1u)] = pw.w[e];
            }
            sync_all();
            const uint32_t* list = sh.listed;
            if constexpr (C > 1) {
                uint32_t at = 0;
                for (uint32_t r = 0; r < (uint32_t)C; ++r) {
                    const uint32_t n = cluster_load(&sh.n_listed, r);
                    for (uint32_t i = threadIdx.x; i < n; i += kThreads) sh.all_listed[at + i] = cluster_load(&sh.listed[i], r);
                    at += n;
                }
                list = sh.all_listed;
                __syncthreads();
            }
            for (uint32_t i = threadIdx.x; i < in_bin; i += kThreads) {
                const uint32_t w = list[i];
                uint32_t less = 0, leq = 0;
                for (uint32_t j = 0; j < in_bin; ++j) {
                    less += list[j] < w;
                    leq += list[j] <= w;
                }
                if (less < remaining && remaining <= leq) {  // (equal words all write the same)
                    sh.threshold = w;
                    sh.less = less;
                    sh.equal = leq - less;
                }
            }
            __syncthreads();
            threshold = sh.threshold;
            ties = remaining - sh.less;
            all_ties = sh.equal == ties;
            break;
        }
    }

    // ---- each warp's contiguous stretch of groups, a group a lane at a time: counts, then the kept positions in order.  (With a
    //      stretch a thread every store is a transaction of its own.) ----
    constexpr int kWarps = kThreads / 32;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const uint32_t slice = g_end - g_begin, per_warp = ((slice + kWarps - 1) / kWarps + 31u) & ~31u;
    const uint32_t w_begin = g_begin + ((uint32_t)warp * per_warp < slice ? (uint32_t)warp * per_warp : slice);
    const uint32_t w_end = g_end - w_begin < per_warp ? g_end : w_begin + per_warp;
    uint32_t lt = 0, eq = 0;
    for (uint32_t q = w_begin + lane; q < w_end; q += 32) {
        const PhiloxWords pw = words_of(q);
#pragma unroll
        for (int e = 0; e < 4; ++e) {
            if (4u * q + e < N) {
                lt += pw.w[e] < threshold;
                eq += pw.w[e] == threshold;
            }
        }
    }
    lt = __reduce_add_sync(0xffffffffu, lt);
    eq = __reduce_add_sync(0xffffffffu, eq);
    if (lane == 0) {
        sh.warp_sums[warp] = lt;
        sh.warp_ties[warp] = eq;
    }
    __syncthreads();
    const uint32_t all_lt = lane < kWarps ? sh.warp_sums[lane] : 0u, all_eq = lane < kWarps ? sh.warp_ties[lane] : 0u;
    uint32_t kept_before = __reduce_add_sync(0xffffffffu, lane < warp ? all_lt : 0u);      // below the threshold in front of this warp's stretch
    uint32_t ties_before = __reduce_add_sync(0xffffffffu, lane < warp ? all_eq : 0u);
    if constexpr (C > 1) {
        const uint32_t slice_lt = __reduce_add_sync(0xffffffffu, all_lt), slice_eq = __reduce_add_sync(0xffffffffu, all_eq);
        if (threadIdx.x == 0) { sh.slice_counts[0] = slice_lt; sh.slice_counts[1] = slice_eq; }
        cluster_sync();
        for (uint32_t r = 0; r < rank; ++r) {
            kept_before += cluster_load(&sh.slice_counts[0], r);
            ties_before += cluster_load(&sh.slice_counts[1], r);
        }
    }
    uint32_t first = kept_before + (ties_before < ties ? ties_before : ties);
    pdl_wait();                 // earlier kernels of the stream may still be reading the index buffers
    if (rank == 0 && threadIdx.x == 0) {
        keep_offsets[b + 1] = (int32_t)((b + 1) * (int64_t)K);
        if (b == 0) keep_offsets[0] = 0;
    }
    const uint32_t lanes_before = (1u << lane) - 1u;
    for (uint32_t q0 = w_begin; q0 < w_end; q0 += 32) {
        const uint32_t q = q0 + lane;
        const bool live = q < w_end;
        PhiloxWords pw;
        if (live) pw = words_of(q);
        bool keep[4];
        if (all_ties) {
#pragma unroll
            for (int e = 0; e < 4; ++e) keep[e] = live && 4u * q + e < N && pw.w[e] <= threshold;
        } else {                                                   // ties are kept in order of position until there are enough
            bool tie[4];
            uint32_t mine = ties_before;
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                tie[e] = live && 4u * q + e < N && pw.w[e] == threshold;
                const uint32_t all = __ballot_sync(0xffffffffu, tie[e]);
                mine += __popc(all & lanes_before);
                ties_before += __popc(all);
            }
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                keep[e] = (live && 4u * q + e < N && pw.w[e] < threshold) || (tie[e] && mine < ties);
                mine += tie[e];
            }
        }
        uint32_t at = first;
#pragma unroll
        for (int e = 0; e < 4; ++e) {
            const uint32_t all = __ballot_sync(0xffffffffu, keep[e]);
            at += __popc(all & lanes_before);
            first += __popc(all);
        }
#pragma unroll
        for (int e = 0; e < 4; ++e)
            if (keep[e]) out[at++] = (int32_t)(row_base + 4u * q + e);
    }
    if constexpr (C > 1) cluster_sync();                      // the slice counts stay readable until every block is done
}

// ---- grid-wise masks: 2x2-periodic lattice with a per-sample phase ----
__device__ __forceinline__ uint32_t grid_phase(int family, uint32_t gid, uint32_t step, uint32_t k0, uint32_t k1) {
    if (family == 4) return 0u;
    const uint32_t word = philox4x32_10(0u, gid, step, 1u, k0, k1).w[0];
    return family == 2 ? (word & 1u) : (word & 3u);
}

__device__ __forceinline__ uint32_t grid_count(int family, uint32_t p, uint32_t H, uint32_t W) {
    const uint32_t quarter = ((H + 1u - (p >> 1)) >> 1) * ((W + 1u - (p & 1u)) >> 1);
    switch (family) {
        case 1: return quarter;
        case 2: return (H * W + 1u - p) >> 1;
        case 3: return H * W - quarter;
        default: return H * W;
    }
}

// kept positions of row h in front of column w
__device__ __forceinline__ uint32_t grid_before(int family, uint32_t p, uint32_t h, uint32_t w) {
    const uint32_t on_lattice = (h & 1u) == (p >> 1) ? (w + 1u - (p & 1u)) >> 1 : 0u;
    switch (family) {
        case 1: return on_lattice;
        case 2: return (w + 1u - ((p + h) & 1u)) >> 1;
        case 3: return w - on_lattice;
        default: return w;
    }
}

__device__ __forceinline__ bool grid_keeps(int family, uint32_t p, uint32_t h, uint32_t w) {
    const bool on_lattice = ((h & 1u) == (p >> 1)) && ((w & 1u) == (p & 1u));
    switch (family) {
        case 1: return on_lattice;
        case 2: return ((h + w) & 1u) == p;
        case 3: return !on_lattice;
        default: return true;
    }
}

// `parts` blocks a sample, each with a contiguous stretch of the positions
__global__ void __launch_bounds__(kSampThreads)
sample_keep_grid_kernel(int family, uint32_t H, uint32_t W, FastDiv by_width, uint32_t parts, uint32_t k0, uint32_t k1, uint32_t step,
                        uint32_t first_sample, int share_mask,
                        int32_t* __restrict__ keep_rows, int32_t* __restrict__ keep_offsets) {
    __shared__ uint64_t red[kSampWarps];
    pdl_launch_dependents();
    const uint32_t b = blockIdx.x / parts, part = blockIdx.x - b * parts;
    const uint32_t N = H * W;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;

    // offset of this sample = sum of the closed-form counts of the samples before it
    uint64_t before = 0;
    if (share_mask || family == 4) {                         // every sample keeps as many as the first
        before = (uint64_t)b * grid_count(family, grid_phase(family, 0u, step, k0, k1), H, W);
    } else {
        uint64_t sum = 0;
        for (uint32_t s = threadIdx.x; s < b; s += kSampThreads)
            sum += grid_count(family, grid_phase(family, first_sample + s, step, k0, k1), H, W);
#pragma unroll
        for (int d = 16; d > 0; d >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, d);
        if (lane == 0) red[warp] = sum;
        __syncthreads();
        for (int i = 0; i < kSampWarps; ++i) before += red[i];
    }
    const uint32_t p = grid_phase(family, share_mask ? 0u : first_sample + b, step, k0, k1);
    pdl_wait();                 // earlier kernels of the stream may still be reading the index buffers
    if (part == 0 && threadIdx.x == 0) {
        keep_offsets[b + 1] = (int32_t)(before + grid_count(family, p, H, W));
        if (b == 0) keep_offsets[0] = 0;
    }
    int32_t* out = keep_rows + before;
    const int64_t row_base = (int64_t)b * N;
    const uint32_t per = (N + parts - 1) / parts;
    const uint32_t begin = part * per < N ? part * per : N, end = N - begin < per ? N : begin + per;
    for (uint32_t n = begin + threadIdx.x; n < end; n += kSampThreads) {
        const uint32_t h = by_width(n), w = n - h * W;
        if (grid_keeps(family, p, h, w)) out[grid_count(family, p, h, W) + grid_before(family, p, h, w)] = (int32_t)(row_base + n);
    }
}


// ---------------------------------------------------------------------------------------------
// whole-frame masks for video (Sec. 3.1, 3.2.1: a subset of frames): T frames of P positions, the
// K_T frames with the smallest scores (word << 32) | f are kept, each with all of its positions.
// T is small (a clip has tens of frames), so every block of a sample ranks all frames by counting and writes a stretch of
// the rows (one block a sample with a 64-bit division per row, back to back: 2 clips of 32 x 3136 14.2 us, now 1.3; one of
// 8 x 196 1.8, now 1.0).
// ---------------------------------------------------------------------------------------------
constexpr uint32_t kMaxFrames = 2048;

// frames of family `family` (as the spatial grid families: every fourth, every second, all but every fourth, all)
// at phase p among T frames
__device__ __forceinline__ uint32_t frame_count(int family, uint32_t p, uint32_t T) {
    const uint32_t fourth = (T + 3u - p) >> 2;
    switch (family) {
        case 1: return fourth;
        case 2: return (T + 1u - p) >> 1;
        case 3: return T - fourth;
        default: return T;
    }
}
__device__ __forceinline__ bool frame_keeps(int family, uint32_t p, uint32_t f) {
    switch (family) {
        case 1: return (f & 3u) == p;
        case 2: return (f & 1u) == p;
        case 3: return (f & 3u) != p;
        default: return true;
    }
}

// family 0: the K_T frames with the smallest scores; families 1-4: frames on a lattice in time whose phase is
// drawn per sample like the spatial grid phase (counts, and so the offsets, then depend on the phases)
__global__ void __launch_bounds__(kSampThreads)
sample_keep_temporal_kernel(int family, uint32_t T, uint32_t P, FastDiv by_frame, uint32_t KT, uint32_t parts, uint32_t k0, uint32_t k1, uint32_t step,
                            uint32_t first_sample, int share_mask,
                            int32_t* __restrict__ keep_rows, int32_t* __restrict__ keep_offsets) {
    __shared__ unsigned long long score[kMaxFrames];
    __shared__ uint32_t kept[kMaxFrames];        // first a flag per frame, then the ascending list of kept frames
    __shared__ uint32_t list[kMaxFrames];
    pdl_launch_dependents();
    const uint32_t b = blockIdx.x / parts, part = blockIdx.x - b * parts;
    const uint32_t gid = share_mask ? 0u : first_sample + b;
    uint64_t frames_before = (uint64_t)b * KT;                       // kept frames of the samples before this one
    if (family == 0) {
        for (uint32_t f = threadIdx.x; f < T; f += kSampThreads) {
            const uint32_t w = philox4x32_10(f >> 2, gid, step, 0u, k0, k1).w[f & 3u];
            score[f] = ((unsigned long long)w << 32) | f;
        }
        __syncthreads();
        for (uint32_t f = threadIdx.x; f < T; f += kSampThreads) {
            const unsigned long long mine = score[f];
            uint32_t rank = 0;
            for (uint32_t g = 0; g < T; ++g) rank += score[g] < mine;
            kept[f] = rank < KT ? 1u : 0u;
        }
    } else {
        const uint32_t p = grid_phase(family, gid, step, k0, k1);
        for (uint32_t f = threadIdx.x; f < T; f += kSampThreads) kept[f] = frame_keeps(family, p, f) ? 1u : 0u;
        KT = frame_count(family, p, T);
        // the offset of this sample is the sum of the closed-form counts of the samples before it
        if (share_mask) {
            frames_before = (uint64_t)b * KT;
        } else {
            __shared__ unsigned long long red[kSampThreads / 32];
            unsigned long long sum = 0;
            for (uint32_t s2 = threadIdx.x; s2 < b; s2 += kSampThreads)
                sum += frame_count(family, grid_phase(family, first_sample + s2, step, k0, k1), T);
#pragma unroll
            for (int d = 16; d > 0; d >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, d);
            if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = sum;
            __syncthreads();
            frames_before = 0;
            for (int i = 0; i < kSampThreads / 32; ++i) frames_before += red[i];
        }
    }
    __syncthreads();
    for (uint32_t f = threadIdx.x; f < T; f += kSampThreads) {
        if (kept[f]) {
            uint32_t pos = 0;
            for (uint32_t g = 0; g < f; ++g) pos += kept[g];
            list[pos] = f;
        }
    }
    __syncthreads();
    pdl_wait();                 // earlier kernels of the stream may still be reading the index buffers
    const uint32_t per_sample = KT * P, per = (per_sample + parts - 1) / parts;      // (row ids are 32-bit: so are counts of them)
    const uint32_t begin = part * per < per_sample ? part * per : per_sample, end = per_sample - begin < per ? per_sample : begin + per;
    int32_t* out = keep_rows + frames_before * P;
    for (uint32_t e = begin + threadIdx.x; e < end; e += kSampThreads) {
        const uint32_t k = by_frame(e), q = e - k * P;
        out[e] = (int32_t)(((uint64_t)b * T + list[k]) * P + q);
    }
    if (part == 0 && threadIdx.x == 0) {
        keep_offsets[b] = (int32_t)(frames_before * P);
        if (blockIdx.x + parts == gridDim.x) keep_offsets[b + 1] = (int32_t)(frames_before * P + per_sample);
    }
}

}  // namespace

uint32_t sample_keep_max_frames() { return kMaxFrames; }

namespace {
constexpr size_t kCacheMax = 160 * 1024;

// shared-memory cache of a slice's words (16 bytes per group of four positions), when it fits
template <int C, int kThreads>
cudaError_t launch_random_sampler(int64_t B, cudaStream_t stream, int64_t N, int64_t K, uint32_t k0, uint32_t k1, uint32_t step,
                                  uint32_t first_sample, bool share_mask, int32_t* keep_rows, int32_t* keep_offsets) {
    const int64_t slice_groups = ((N + 3) / 4 + C - 1) / C;
    size_t cache_bytes = (size_t)slice_groups * 16 <= kCacheMax ? (size_t)slice_groups * 16 : 0;
    // the large blocks one to an SM: two of a cluster side by side on one made the detection step (2 x 66800) 4 us longer
    if (kThreads == 1024 && cache_bytes < 116 * 1024) cache_bytes = 116 * 1024;
    if (cache_bytes > 32 * 1024) {                            // (the static part takes 10 KB of the default 48)
        const cudaError_t opt = opt_in_dynamic_smem<sample_keep_random_kernel<C, kThreads>>((int)kCacheMax);
        if (opt != cudaSuccess) return opt;
    }
    const dim3 grid((unsigned)(B * C)), block(kThreads);
    const auto launch = [&](auto... args) {
        if constexpr (C > 1) return launch_pdl_cluster(sample_keep_random_kernel<C, kThreads>, grid, block, cache_bytes, C, stream, args...);
        else return launch_pdl(sample_keep_random_kernel<C, kThreads>, grid, block, cache_bytes, stream, args...);
    };
    return launch((uint32_t)N, (uint32_t)K, k0, k1, step, first_sample, share_mask ? 1 : 0, (uint32_t)(cache_bytes / 16), keep_rows,
                  keep_offsets);
}
}  // namespace

cudaError_t launch_sample_keep(int mode, int grid_family, int64_t B, int64_t H, int64_t W, int64_t K,
                               uint64_t seed, uint32_t step, uint32_t first_sample, bool share_mask,
                               int32_t* keep_rows, int32_t* keep_offsets, cudaStream_t stream) {
    const uint32_t k0 = (uint32_t)(seed & 0xffffffffu), k1 = (uint32_t)(seed >> 32);
    const int64_t N = H * W;
    if (mode == SBP_MASK_RANDOM && K >= N && N > 8192) {     // nothing to choose: the grid mask that keeps everything
        mode = SBP_MASK_GRID;
        grid_family = 4;
    }
    if (mode == SBP_MASK_RANDOM) {
        // large maps with few samples: spread each sample over a cluster so that more SMs take part
        if (N > 8192 && B * 8 <= 4 * kNumSMs) {
            // 1024 threads for up to three samples, whose clusters find room beside the kernel before: 1, 2 and 3 x 66800 positions
            // 2.95 -> 2.63, 3.06 -> 2.70 and 3.19 -> 3.32 us back to back, 3 x 200000 6.2 -> 5.1, but 8 x 66800 4.1 -> 9.0
            if (N > 32768 && B <= 3) return launch_random_sampler<8, 1024>(B, stream, N, K, k0, k1, step, first_sample, share_mask, keep_rows, keep_offsets);
            if (N > 32768) return launch_random_sampler<8, 512>(B, stream, N, K, k0, k1, step, first_sample, share_mask, keep_rows, keep_offsets);
            if (N > 16384) return launch_random_sampler<4, 512>(B, stream, N, K, k0, k1, step, first_sample, share_mask, keep_rows, keep_offsets);
            return launch_random_sampler<2, 512>(B, stream, N, K, k0, k1, step, first_sample, share_mask, keep_rows, keep_offsets);
        }
        // four warps see up to 512 positions, one group of four a thread
        if (N <= 512) return launch_random_sampler<1, 128>(B, stream, N, K, k0, k1, step, first_sample, share_mask, keep_rows, keep_offsets);
        return launch_random_sampler<1, 512>(B, stream, N, K, k0, k1, step, first_sample, share_mask, keep_rows, keep_offsets);
    }
    // four positions a thread, on four blocks an SM at most
    const auto blocks_for = [&](int64_t positions) {
        const int64_t by_size = (positions + 4 * kSampThreads - 1) / (4 * kSampThreads), by_room = 4 * kNumSMs / B;
        return by_size < by_room ? by_size : by_room < 1 ? 1 : by_room;
    };
    const int64_t parts = blocks_for(mode == SBP_MASK_GRID ? N : K);
    const dim3 grid((unsigned)(B * parts)), block(kSampThreads);
    if (mode == SBP_MASK_TEMPORAL || mode == SBP_MASK_TEMPORAL_GRID)      // H frames of W positions; K = kept frames x W
        return launch_pdl(sample_keep_temporal_kernel, grid, block, 0, stream, mode == SBP_MASK_TEMPORAL ? 0 : grid_family,
                          (uint32_t)H, (uint32_t)W, FastDiv((uint32_t)W), (uint32_t)(K / W), (uint32_t)parts,
                          k0, k1, step, first_sample, share_mask ? 1 : 0, keep_rows, keep_offsets);
    return launch_pdl(sample_keep_grid_kernel, grid, block, 0, stream, grid_family, (uint32_t)H, (uint32_t)W,
                      FastDiv((uint32_t)W), (uint32_t)parts, k0, k1,
                      step, first_sample, share_mask ? 1 : 0, keep_rows, keep_offsets);
}

}  // namespace sbp

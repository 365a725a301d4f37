// SBP backward of scaled dot-product attention on token subsets (Sec. 4, "How to apply SBP on MHSA?"; supplementary,
// "Gradient Calculation of Attention Layers"), bf16 on the tensor cores (tcgen05 / TMEM), head dimension 64.
//
// One (sample, head) problem at a time per block.  With Zq the kept query tokens and Zk the kept key / value tokens of the
// sample (at most 256 each):
//     S  = softmax_j(q_i . k_j / sqrt(d))  over j in Zk          (recomputed here: no n x n map is cached at all)
//     dS = dA V^T,   dM = S * (dS - rowsum(S * dS)) / sqrt(d)
//     dV = S^T dA,   dK = dM^T Q,   dQ = dM K
// All five products run as tcgen05.mma on operands staged once in shared memory (128-byte swizzle): a row-major
// [tokens x 64] tile serves as the K-major operand of Q K^T / dA V^T and, unchanged, as the MN-major operand of the
// three gradient products.
//
// Bound by memory at the paper's sizes, and in practice by the length of a problem's chain (copies, two products, softmax,
// three products, read-out), which the layout below keeps short:
//  - A row of S is shared by G threads of one TMEM lane quadrant, 64 columns each (G = 2: up to 128 tokens a side, two blocks
//    of 256 threads per SM; G = 4: up to 256, one block of 512).  Each thread keeps its 64 numbers of S in registers and
//    turns them into e^(s - own maximum) once; one exchange of (maximum, sum, sum of e dS) among the G threads gives the
//    row's statistics.
//  - S and dM go to shared-memory blocks of their own where these fit, so the three gradient products run back to back
//    (G = 2: the second half of dM takes the place of V, which is dead by then); otherwise dM waits in registers and
//    overwrites S once dV is done.
//  - Buffers are sized by the rows in use (token bound rounded up to 16), not by 128 or 256.
//  - The next problem's rows are copied as soon as the last product has read the operands, under the read-out and the
//    stores of this one.
// Measured on B200, ViT-B/16 heads (12 x 64, 196 tokens), whole pass with the sampler: Drop QKV, half of the tokens, B = 128:
// 99 us with a thread a row and copies behind the read-out, 64 with the zeros of a problem's own rows in front of its first wait, now 59;
// Drop Query only, B = 64: 94 -> 71 -> 61.  (One thread issuing the products instead of a whole warp with one lane elected: 70 and 78 us,
// each instruction waiting for its operands to reach uniform registers.)  A problem's chain, some 17000 clocks with two blocks on an SM: wait
// for the copies 900, first products and zeros 2300, softmax 5300, gradient products and zeros 3200, next copies 2900, read-out and stores 2400.
// Not kept: copies and zeros by four warps of their own (the computing warps need more registers than setmaxnreg could then give
// them, 76 us); dV made first so that the next problem's rows of dA come in under dK and dQ (62 and 63.5 us: products that do not take turns
// between accumulators are slower); a problem's stores under the next one's first products (64 us: they then hold up the softmax).
// Query tiles of 128 rows follow one another (dV and dK stay in tensor memory); with two of them S and dS share columns.
// Rows outside the token sets are zeroed here too, while products run.  Every wait is bounded and reports through
// the status word.
#include "tc_ptx.cuh"
#include "zero_rows.cuh"

namespace sbp {
namespace {

constexpr int kD = 64;                          // head dimension (one 128-byte swizzle row of bf16)
constexpr int kMaxTok = 256;                    // most kept tokens of a sample on either side
constexpr uint32_t kRowB = 128;
constexpr uint32_t kTileB = 128 * kRowB;        // a 128-row tile of an operand

struct AttnParams {
    const __nv_bfloat16 *Q, *K, *V, *dA;
    uint32_t ld_qkv, ld_da, ld_out;                       // row strides in 16-byte vectors
    const int32_t *q_rows, *q_offs, *k_rows, *k_offs;     // null rows = every token of the sample
    int B, N, heads;
    __nv_bfloat16 *dQ, *dK, *dV;
    float scale;
    int zero_fill;                // 1: the rows that the lists leave out are written as zeros
    int zero_blocks, zero_first, zero_rest;    // rows of the outputs that each of the first zero_blocks blocks looks after, each of the others
    int rq, rk;                   // rows of the query-side and key-side buffers: the token bounds rounded up to 16
    uint32_t block_bytes;         // one 64-key block of S: 128 bytes for each query row of a tile
    uint32_t off_dm, dm_stride;   // dM blocks (separate: next to S; otherwise the S blocks themselves)
    uint32_t off_q, off_da, off_k, off_v;
    int separate;                 // dM has blocks of its own
    int32_t* status_word;
};

__device__ __forceinline__ uint32_t swz(uint32_t row, uint32_t chunk) { return row * kRowB + ((chunk ^ (row & 7u)) << 4); }

__device__ __forceinline__ uint32_t pack2(float lo, float hi) {
    const __nv_bfloat162 v = __floats2bfloat162_rn(lo, hi);
    return *reinterpret_cast<const uint32_t*>(&v);
}

__device__ __forceinline__ float ex2(float x) {
    float y;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

__device__ __forceinline__ float max3(float a, float b, float c) {
    float d;
    asm("max.f32 %0, %1, %2, %3;" : "=f"(d) : "f"(a), "f"(b), "f"(c));
    return d;
}

// Calls whose blocks have equal lists of problems: zeros for the problem's own 64 columns in the rows of sample b that an ascending token list leaves out, with
// no look at memory (the walk's dependent loads are longer than the first products: 7.7 us here, 8.5 with it).  `glob` holds the
// global row of every listed token of the sample (shared memory).  The z-th unlisted row lies behind g listed ones, with g
// the first list position whose token has more than z unlisted rows in front of it: a search of at most eight steps.  Every
// lane of a warp searches for a row of its own; then eight lanes at a time clear one 128-byte line, 16 bytes each, so that a
// warp's store covers four whole lines.  (Walking the gaps between listed tokens, a group of eight lanes each, gave the warps
// very different amounts of work: 3000 - 4700 clocks a problem.)  Rows are clamped to the sample, so that a list that breaks the
// ascending order cannot send a store anywhere else.
__device__ __forceinline__ void zero_unlisted_rows(__nv_bfloat16* out0, __nv_bfloat16* out1, __nv_bfloat16* out2, uint32_t ld, int col0,
                                                   const int32_t* glob, int count, int base_row, int N, int warp, int warps, int lane) {
    const int unlisted = N - count;
    int per = ((unlisted + warps - 1) / warps + 3) & ~3;     // rows of a warp's turn: an equal share, at most one for each lane
    per = per < 32 ? per : 32;
    for (int z0 = warp * per; z0 < unlisted; z0 += warps * per) {
        const int want = z0 + lane + base_row;
        int g = 0;                                           // tokens with glob[i] - i <= want are in front of the row
#pragma unroll
        for (int step = 128; step > 0; step >>= 1)
            if (g + step <= count && glob[g + step - 1] - (g + step - 1) <= want) g += step;
        if (g < count && glob[g] - g <= want) ++g;           // (lists of 256 tokens)
        int r = z0 + lane + g;
        r = base_row + (r < N ? r : N - 1);
        const int here = unlisted - z0 < per ? unlisted - z0 : per;
#pragma unroll 2
        for (int i = 0; i < here; i += 4) {
            const int row = __shfl_sync(0xffffffffu, r, i + (lane >> 3));
            if (i + (lane >> 3) < here) {
                const int64_t at = (int64_t)((uint64_t)(uint32_t)row * ld * 8u) + col0 + (lane & 7) * 8;
                if (out0 != nullptr) ptx::st_global_v4(out0 + at, 0u, 0u, 0u, 0u);
                if (out1 != nullptr) ptx::st_global_v4(out1 + at, 0u, 0u, 0u, 0u);
                if (out2 != nullptr) ptx::st_global_v4(out2 + at, 0u, 0u, 0u, 0u);
            }
        }
    }
}

// Calls that leave blocks without a problem for a while: zeros for the rows that an ascending list of token rows leaves out, whole rows (all heads) of the outputs.  A warp walks a range of
// rows of its own, a few unlisted ones at a time: the stores go out while the block waits for products, so that memory works then too.
// (In front of the first products, an equal share of the problem's own rows a warp and 128 bytes of each, they took 3500 of a problem's
// 17500 clocks with the products' 1000 underneath.)
struct ZeroWalk {                 // kept in shared memory between a warp's turns: it would cost the computing threads registers
    int pass;                     // 0: the rows that the query list leaves out, 1: the key list; 2: done
    int budget;                   // rows to clear in a turn
    int p, n;                     // position in the list, its end
    int base, next, end;          // first row of the window of 32 at hand, of the next one; end of the range
    uint32_t todo;                // unlisted rows of the window that are still to be cleared
};

// A warp's range of the rows that are cleared where the lists leave them out: first those of dQ (or of all outputs, with one list for
// both sides), then, with a list of their own, those of dK and dV.
__device__ __forceinline__ void start_walk(const AttnParams& p, ZeroWalk& z, int warp, int warps, int lane) {
    const int32_t* offs = z.pass == 0 ? p.q_offs : p.k_offs;
    const int first = __ldg(offs), blk = (int)blockIdx.x, share = blk < p.zero_blocks ? p.zero_first : p.zero_rest;
    z.n = __ldg(offs + p.B);
    const int64_t all = (int64_t)p.B * p.N, before = blk < p.zero_blocks ? blk : p.zero_blocks;
    const int64_t at = before * p.zero_first + (blk - before) * p.zero_rest;
    const int per = (share + warps - 1) / warps;
    int64_t lo = at + (int64_t)per * warp, hi = lo + per < at + share ? lo + per : at + share;
    if (hi > all) hi = all;
    if (lo > hi) lo = hi;
    z.next = (int)lo;
    z.end = (int)hi;
    z.todo = 0u;
    z.p = lo < hi ? first + (int)warp_lower_bound((z.pass == 0 ? p.q_rows : p.k_rows) + first, z.n - first, lo, lane) : z.n;
    // two turns a problem: an even part of the rows that this warp can expect to clear, rounded up
    const int turns = 2 * ((p.B * p.heads - blk + (int)gridDim.x - 1) / (int)gridDim.x);
    const int expect = (int)((float)(hi - lo) * (1.f - (float)(z.n - first) / (float)all)) + 1;
    z.budget = (expect + turns - 1) / turns;
}

// A turn of a warp, or all that is left.
__device__ __forceinline__ void zero_rows(const AttnParams& p, ZeroWalk* walk, int warp, int warps, int lane, bool rest) {
    ZeroWalk z = *walk;
    const bool same = p.q_rows == p.k_rows && p.q_offs == p.k_offs;
    const auto zero_line = [&](int64_t at) {
        if (z.pass == 0) ptx::st_global_v4(p.dQ + at, 0u, 0u, 0u, 0u);
        if (z.pass == 1 || same) {
            ptx::st_global_v4(p.dK + at, 0u, 0u, 0u, 0u);
            ptx::st_global_v4(p.dV + at, 0u, 0u, 0u, 0u);
        }
    };
    int most = rest ? 0x7fffffff : z.budget;
    while (most > 0 && z.pass < 2) {
        if (z.todo != 0u) {
            if (p.heads > 2) {
                const int64_t at = (int64_t)((uint64_t)(uint32_t)(z.base + __ffs(z.todo) - 1) * p.ld_out * 8u);
                for (int c = lane * 8; c < p.heads * kD; c += 256) zero_line(at + c);
                z.todo &= z.todo - 1u;
                --most;
            } else {
                // four rows of one head, or two of two heads, at a time (one: 298 to 400 problems of one head 3 to 12 % slower)
                const int per = p.heads == 1 ? 4 : 2;
                uint32_t own = z.todo;
                for (int k = lane * per / 32; k > 0; --k) own &= own - 1u;
                if (own != 0u) zero_line((int64_t)((uint64_t)(uint32_t)(z.base + __ffs(own) - 1) * p.ld_out * 8u) + lane % (32 / per) * 8);
                for (int k = 0; k < per; ++k) z.todo &= z.todo - 1u;
                most -= per;
            }
        } else if (z.next < z.end) {                        // the next window of 32 rows
            const int d = z.p + lane < z.n ? __ldg((z.pass == 0 ? p.q_rows : p.k_rows) + z.p + lane) - z.next : 32;
            const uint32_t listed = __reduce_or_sync(0xffffffffu, (d >= 0 && d < 32) ? 1u << d : 0u);
            const int here = z.end - z.next < 32 ? z.end - z.next : 32;
            z.p += __popc(listed);
            z.base = z.next;
            z.next += here;
            z.todo = ~listed & (here < 32 ? (1u << here) - 1u : 0xffffffffu);
        } else {
            z.pass = z.pass == 0 && !same && p.k_rows != nullptr ? 1 : 2;
            if (z.pass == 1) start_walk(p, z, warp, warps, lane);
        }
    }
    __syncwarp();
    if (lane == 0) *walk = z;
    __syncwarp();
}

__device__ __forceinline__ void prefetch_row(const __nv_bfloat16* p, int32_t row, uint32_t ld) {
    asm volatile("prefetch.global.L2 [%0];" ::"l"(reinterpret_cast<const uint4*>(p) + (uint64_t)(uint32_t)row * ld));
}

template <int G>
struct AttnShared {
    static constexpr int kTok = G == 2 ? 128 : kMaxTok;
    uint64_t bar_s, bar_o;        // products of S and dS; gradient products
    uint32_t tmem_slot;
    int abort_flag;
    ZeroWalk walk[4 * G];         // of each warp
    float part[G][128][3];        // per 64 columns of a row: maximum, sum of e = 2^((s - maximum) log2 e / sqrt(d)), sum of e dS
    int32_t q_glob[2][kTok], k_glob[2][kTok];   // global rows of the listed tokens (0 past the last): this problem's, the next one's
};

// Token counts of a problem and the global rows of its query and key number t.
struct Meta { int nq, nk; int32_t q, k; };
__device__ __forceinline__ Meta fetch_meta(const AttnParams& p, int prob, int t) {
    Meta m{0, 0, 0, 0};
    if (prob >= p.B * p.heads) return m;
    const int b = prob / p.heads, base_row = b * p.N;
    const int q0 = p.q_rows ? __ldg(p.q_offs + b) : 0, k0 = p.k_rows ? __ldg(p.k_offs + b) : 0;
    m.nq = p.q_rows ? __ldg(p.q_offs + b + 1) - q0 : p.N;
    m.nk = p.k_rows ? __ldg(p.k_offs + b + 1) - k0 : p.N;
    if (m.nq > p.rq) m.nq = p.rq;           // lists longer than the stated bound stay inside the buffers
    if (m.nk > p.rk) m.nk = p.rk;
    if (t < m.nq) m.q = p.q_rows ? __ldg(p.q_rows + q0 + t) : base_row + t;
    if (t < m.nk) m.k = p.k_rows ? __ldg(p.k_rows + k0 + t) : base_row + t;
    return m;
}

// Copies the rows of one side's two operands (64 columns each) into their swizzled tiles; rows past `count`, up to the next
// multiple of 16 (as far as the products step), become zeros.  Up to four rows at a time, their ids read together; a thread's
// rows are a multiple of 8 apart, so that its place in the swizzle is the same in all of them.
template <int kThreads>
__device__ __forceinline__ void load_rows(uint32_t dst0, uint32_t dst1, const __nv_bfloat16* src0, uint32_t ld0, const __nv_bfloat16* src1,
                                          uint32_t ld1, const int32_t* glob, int count, int t) {
    const uint32_t chunk = t & 7u;
    const uint4* s0 = reinterpret_cast<const uint4*>(src0) + chunk;
    const uint4* s1 = reinterpret_cast<const uint4*>(src1) + chunk;
    constexpr int kStep = kThreads / 8;
    const int padded = (count + 15) & ~15;
    uint32_t at = swz(t >> 3, chunk);
    for (int r = t >> 3; r < padded; r += 4 * kStep, at += 4 * kStep * kRowB) {
        uint32_t id[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) id[i] = (r + i * kStep < padded) ? (uint32_t)glob[r + i * kStep] : 0u;
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            if (r + i * kStep < padded) {
                const uint32_t bytes = r + i * kStep < count ? 16u : 0u;
                ptx::cp_async_16(dst0 + at + i * kStep * kRowB, s0 + (uint64_t)id[i] * ld0, bytes);
                ptx::cp_async_16(dst1 + at + i * kStep * kRowB, s1 + (uint64_t)id[i] * ld1, bytes);
            }
        }
    }
}

__device__ __forceinline__ uint64_t pair(float x, float y) {
    uint64_t r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(x), "f"(y));
    return r;
}
__device__ __forceinline__ float2 halves(uint64_t v) {
    float2 f;
    asm("mov.b64 {%0, %1}, %2;" : "=f"(f.x), "=f"(f.y) : "l"(v));
    return f;
}
__device__ __forceinline__ uint64_t fma2(uint64_t a, uint64_t b, uint64_t c) {
    uint64_t d;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
    return d;
}
__device__ __forceinline__ uint64_t mul2(uint64_t a, uint64_t b) {
    uint64_t d;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}
__device__ __forceinline__ uint64_t add2(uint64_t a, uint64_t b) {
    uint64_t d;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}

__device__ __forceinline__ uint4 pack8(const float* f) {
    return make_uint4(pack2(f[0], f[1]), pack2(f[2], f[3]), pack2(f[4], f[5]), pack2(f[6], f[7]));
}
// 32 accumulator columns of this thread's row to chunks [chunk0, chunk0 + 4) of a staged [rows x 64] output
__device__ __forceinline__ void stage32(uint8_t* stage, int row, uint32_t chunk0, const float (&v)[32]) {
#pragma unroll
    for (int q = 0; q < 4; ++q) *reinterpret_cast<uint4*>(stage + swz((uint32_t)row, chunk0 + q)) = pack8(v + q * 8);
}
// staged rows [0, count) to the rows glob[] of an output, whole 128-byte rows, four in flight per thread
template <int kThreads>
__device__ __forceinline__ void store_rows(__nv_bfloat16* out, uint32_t ld, int col0, const uint8_t* stage, const int32_t* glob, int count) {
    const uint32_t chunk = threadIdx.x & 7u;
    uint4* to = reinterpret_cast<uint4*>(out + col0) + chunk;
    for (int r0 = threadIdx.x >> 3; r0 < count; r0 += 4 * (kThreads / 8)) {
        const uint8_t* from = stage + swz((uint32_t)r0, chunk);            // (rows a multiple of 8 apart: the same place in the swizzle)
        int32_t id[4];
        uint4 pk[4];
#pragma unroll
        for (int i = 0; i < 4; ++i)
            if (r0 + i * (kThreads / 8) < count) {
                id[i] = glob[r0 + i * (kThreads / 8)];
                pk[i] = *reinterpret_cast<const uint4*>(from + i * (kThreads / 8) * kRowB);
            }
#pragma unroll
        for (int i = 0; i < 4; ++i)
            if (r0 + i * (kThreads / 8) < count) ptx::st_global_v4(to + (uint64_t)(uint32_t)id[i] * ld, pk[i].x, pk[i].y, pk[i].z, pk[i].w);
    }
}

// kSeparate: dM has blocks of its own; kOwn: each problem clears its own unlisted rows, instead of the walk
template <int G, bool kSeparate, bool kOwn>
__global__ void __launch_bounds__(128 * G, G == 2 ? 2 : 1) attention_bwd_kernel(const __grid_constant__ AttnParams p) {
    constexpr int kThreads = 128 * G;
    constexpr uint32_t kTmemCols = G == 2 ? 256 : 512;
    // tensor-memory columns.  G = 2: S and dS side by side, then dV, dK, dQ in their place.  G = 4: S (dQ later); dS in the
    // upper half, or, when two query tiles keep dV and dK there, next to S (up to 128 keys) or in its place
    constexpr uint32_t kColDV = G == 2 ? 0 : 256, kColDK = G == 2 ? 64 : 384, kColDQ = G == 2 ? 128 : 0;
    extern __shared__ uint8_t smem_raw[];
    __shared__ AttnShared<G> sh;
    const int warp = __shfl_sync(0xffffffffu, (int)(threadIdx.x >> 5), 0), lane = threadIdx.x & 31;
    const uint32_t raw = ptx::smem_addr(smem_raw);
    const uint32_t base = (raw + 1023u) & ~1023u;
    uint8_t* gen = smem_raw + (base - raw);                 // generic pointer to the same place
    const uint32_t sP = base, sDM = base + p.off_dm, sQ = base + p.off_q, sDA = base + p.off_da, sK = base + p.off_k, sV = base + p.off_v;

    pdl_launch_dependents();
    if (threadIdx.x == 0) {
        ptx::mbar_init(ptx::smem_addr(&sh.bar_s), 1);
        ptx::mbar_init(ptx::smem_addr(&sh.bar_o), 1);
        sh.abort_flag = 0;
        ptx::fence_mbar_init();
    }
    if (warp == 0) ptx::tmem_alloc(ptx::smem_addr(&sh.tmem_slot), kTmemCols);
    ptx::tc_fence_before_sync();
    __syncthreads();
    ptx::tc_fence_after_sync();
    const uint32_t tmem = __shfl_sync(0xffffffffu, *reinterpret_cast<volatile uint32_t*>(&sh.tmem_slot), 0);
    volatile int* abort_flag = &sh.abort_flag;
    pdl_wait();
    const bool skip_all = p.status_word != nullptr && *reinterpret_cast<volatile int32_t*>(p.status_word) != 0;

    const int quad = warp & 3, g = warp >> 2;               // TMEM lane quadrant of this warp; which 64 key columns it takes
    const int row = quad * 32 + lane;                       // accumulator row: a query, or a key in the dV / dK read-out
    const int key0 = g * 64;
    const uint32_t lane_off = (uint32_t)(quad * 32) << 16;
    const float sl2 = p.scale * 1.4426950408889634f;        // scores are kept in base 2: e^x = 2^(x log2 e)
    const int problems = p.B * p.heads;
    uint32_t n_s = 0, n_o = 0;                              // completed uses of the two barriers
    bool ok = !skip_all;
    int buf = 0;                                            // which half of q_glob / k_glob holds this problem's rows

    // rows of problem `prob` into buffer half `b`, then its copies (after a barrier: the rows come from shared memory)
    auto begin_problem = [&](const Meta& m, int prob, int b) {
        const int t = (int)threadIdx.x;
        if (t < AttnShared<G>::kTok) {
            sh.q_glob[b][t] = m.q;
            sh.k_glob[b][t] = m.k;
        }
        __syncthreads();
        if (m.nq <= 0 || m.nk <= 0) return;
        const int col0 = (prob % p.heads) * kD;
#pragma unroll 1
        for (int side = 0; side < 2; ++side)                  // (one loop body: copies of it cost registers)
            load_rows<kThreads>(side ? sK : sQ, side ? sV : sDA, (side ? p.K : p.Q) + col0, p.ld_qkv, (side ? p.V : p.dA) + col0,
                                side ? p.ld_qkv : p.ld_da, side ? sh.k_glob[b] : sh.q_glob[b], side ? m.nk : m.nq, t);
    };
    // zeros for the rows of problem `prob` outside its lists
    auto zero_own_rows = [&](int prob, int nq, int nk, const int32_t* q_glob, const int32_t* k_glob) {
        if (!p.zero_fill) return;
        const int b = prob / p.heads, col0 = (prob % p.heads) * kD;
        const bool same = p.q_rows == p.k_rows && p.q_offs == p.k_offs;
        if (p.q_rows != nullptr)
            zero_unlisted_rows(p.dQ, same ? p.dK : nullptr, same ? p.dV : nullptr, p.ld_out, col0, q_glob, nq, b * p.N, p.N, warp, kThreads / 32, lane);
        if (p.k_rows != nullptr && !same)
            zero_unlisted_rows(nullptr, p.dK, p.dV, p.ld_out, col0, k_glob, nk, b * p.N, p.N, warp, kThreads / 32, lane);
    };
    // every thread of the block waits for a commit (one polls); false for all of them when the wait gave up
    auto wait_products = [&](uint64_t* bar, uint32_t& n) {
        bool good = true;
        if (threadIdx.x == 0) good = ptx::mbar_wait(ptx::smem_addr(bar), n & 1u, abort_flag, p.status_word);
        ++n;
        good = !__syncthreads_or(!good);
        ptx::tc_fence_after_sync();
        return good;
    };

    Meta cur = fetch_meta(p, ok ? (int)blockIdx.x : problems, (int)threadIdx.x);
    if (ok && (int)blockIdx.x < problems) begin_problem(cur, (int)blockIdx.x, 0);
    if constexpr (!kOwn) {
        ZeroWalk z{};
        z.pass = !ok || !p.zero_fill ? 2 : p.q_rows != nullptr ? 0 : 1;
        if (z.pass < 2) start_walk(p, z, warp, kThreads / 32, lane);
        if (lane == 0) sh.walk[warp] = z;
        __syncwarp();
    }

    for (int prob = blockIdx.x; ok && prob < problems; prob += gridDim.x, buf ^= 1) {
        const int nq = __shfl_sync(0xffffffffu, cur.nq, 0), nk = __shfl_sync(0xffffffffu, cur.nk, 0);
        const int col0 = (prob % p.heads) * kD;
        const int next = prob + (int)gridDim.x;
        cur = fetch_meta(p, next, (int)threadIdx.x);        // travels while this problem computes
        const int32_t *q_glob = sh.q_glob[buf], *k_glob = sh.k_glob[buf];
        if (nq <= 0 || nk <= 0) {                            // nothing to compute: zeros for the listed rows of a side whose other side has
                                                             // no tokens (sums over nothing)
            if constexpr (kOwn) zero_own_rows(prob, nq, nk, q_glob, k_glob);
            for (int r = (int)threadIdx.x >> 3; r < (nq > nk ? nq : nk); r += kThreads / 8) {
                const int64_t at = (int64_t)((uint64_t)(uint32_t)(nk <= 0 ? q_glob : k_glob)[r] * p.ld_out * 8u) + col0 + (threadIdx.x & 7) * 8;
                if (nk <= 0) {
                    ptx::st_global_v4(p.dQ + at, 0u, 0u, 0u, 0u);
                } else {
                    ptx::st_global_v4(p.dK + at, 0u, 0u, 0u, 0u);
                    ptx::st_global_v4(p.dV + at, 0u, 0u, 0u, 0u);
                }
            }
            __syncthreads();                                 // the problem before this one may still be storing by the other half's rows
            if (next < problems) begin_problem(cur, next, buf ^ 1);
            continue;
        }
        const int QT = G == 2 ? 1 : (nq + 127) >> 7;
        const bool shared_cols = G == 4 && QT > 1 && nk > 128;      // dS takes the place of S
        const uint32_t col_ds = shared_cols ? 0u : G == 4 && QT == 1 ? 256u : 128u;
        const uint32_t k_steps = (uint32_t)(nk + 15) >> 4;
        const int n_keys = (int)k_steps * 16;                // accumulator columns computed
        ptx::cp_async_wait_all();
        ptx::fence_async_proxy();
        __syncthreads();

        for (int qt = 0; qt < QT; ++qt) {
            const int q_here = nq - qt * 128 < 128 ? nq - qt * 128 : 128;
            const uint32_t q_steps = (uint32_t)(q_here + 15) >> 4;
            const uint32_t idesc_s = ptx::umma_idesc_bf16(128, n_keys, false, false);
            const uint32_t dQ0 = ptx::umma_desc_lo(sQ + qt * kTileB, 16), dDA0 = ptx::umma_desc_lo(sDA + qt * kTileB, 16), dK0 = ptx::umma_desc_lo(sK, 16), dV0 = ptx::umma_desc_lo(sV, 16);
            if (warp == 0) {                                 // the whole warp, of which one lane issues
                const bool leader = ptx::elect_one();
                ptx::tc_fence_after_sync();
#pragma unroll
                for (uint32_t u = 0; u < 4; ++u) {           // the two products alternate: they fill different accumulators
                    ptx::umma_bf16_warp<false>(tmem, ptx::umma_desc_of(dQ0 + u * 2), ptx::umma_desc_of(dK0 + u * 2), idesc_s, u != 0, leader);
                    if (!shared_cols) ptx::umma_bf16_warp<false>(tmem + col_ds, ptx::umma_desc_of(dDA0 + u * 2), ptx::umma_desc_of(dV0 + u * 2), idesc_s, u != 0, leader);
                }
                if (leader) ptx::umma_commit(ptx::smem_addr(&sh.bar_s));
                __syncwarp();
            }
            if (qt == 0) {
                if constexpr (kOwn) zero_own_rows(prob, nq, nk, q_glob, k_glob);
                else zero_rows(p, &sh.walk[warp], warp, kThreads / 32, lane, false);
            }
            ok = wait_products(&sh.bar_s, n_s);
            if (!ok) break;
            // ---- this thread's 64 columns of its row, in two chunks of 32 which are skipped past n_keys.  Columns from nk on
            //      (padding keys) are masked; stale columns may hold anything, NaN included ----
            uint64_t e[2][16];                               // S, then e^(s - own maximum), packed in pairs
            float mx4[4] = {-INFINITY, -INFINITY, -INFINITY, -INFINITY};     // four interleaved chains, not one of 64 links
#pragma unroll
            for (int c = 0; c < 2; ++c) {
                const int first = key0 + c * 32;
                if (first >= n_keys) break;
                float v[32];
                ptx::tmem_ld_32x32(tmem + (uint32_t)first + lane_off, v);
                ptx::tmem_ld_wait();
                if (first + 32 > nk) {
#pragma unroll
                    for (int j = 0; j < 32; ++j) v[j] = first + j < nk ? v[j] : -INFINITY;
                }
#pragma unroll
                for (int j = 0; j < 32; j += 2) mx4[(j >> 1) & 3] = max3(mx4[(j >> 1) & 3], v[j], v[j + 1]);
#pragma unroll
                for (int j = 0; j < 16; ++j) e[c][j] = pair(v[2 * j], v[2 * j + 1]);
            }
            if (shared_cols) {
                ptx::tc_fence_before_sync();
                __syncthreads();                              // S has been read by every warp
                if (warp == 0) {
                    const bool leader = ptx::elect_one();
                    ptx::tc_fence_after_sync();
#pragma unroll
                    for (uint32_t u = 0; u < 4; ++u)
                        ptx::umma_bf16_warp<false>(tmem, ptx::umma_desc_of(dDA0 + u * 2), ptx::umma_desc_of(dV0 + u * 2), idesc_s, u != 0, leader);
                    if (leader) ptx::umma_commit(ptx::smem_addr(&sh.bar_s));
                    __syncwarp();
                }
            }
            const float mx = fmaxf(fmaxf(mx4[0], mx4[1]), fmaxf(mx4[2], mx4[3]));
            uint64_t l2[2] = {0ull, 0ull}, u2[2] = {0ull, 0ull};
            const float nm = mx > -INFINITY ? -mx * sl2 : 0.f;
            const uint64_t sl22 = pair(sl2, sl2), nm2 = pair(nm, nm);
#pragma unroll
            for (int c = 0; c < 2; ++c) {
                if (key0 + c * 32 >= n_keys) break;
#pragma unroll
                for (int j = 0; j < 16; ++j) {
                    const float2 x = halves(fma2(e[c][j], sl22, nm2));       // masked columns: 2^-inf = 0
                    e[c][j] = pair(ex2(x.x), ex2(x.y));
                    l2[j & 1] = add2(l2[j & 1], e[c][j]);
                }
            }
            if (shared_cols) {
                ok = wait_products(&sh.bar_s, n_s);
                if (!ok) break;
            }
            // the next problem's rows on their way into L2, a query's and a key's two lines a thread
            if (qt == 0 && next < problems) {
                const int next_col0 = (next % p.heads) * kD;
                if ((int)threadIdx.x < cur.nq) {
                    prefetch_row(p.Q + next_col0, cur.q, p.ld_qkv);
                    prefetch_row(p.dA + next_col0, cur.q, p.ld_da);
                }
                if ((int)threadIdx.x < cur.nk) {
                    prefetch_row(p.K + next_col0, cur.k, p.ld_qkv);
                    prefetch_row(p.V + next_col0, cur.k, p.ld_qkv);
                }
            }
            // 16 columns of dS from column `first` on, in pairs
            auto load_ds = [&](int first, uint64_t (&d)[8]) {
                float v[16];
                ptx::tmem_ld_32x16(tmem + col_ds + (uint32_t)first + lane_off, v);
                ptx::tmem_ld_wait();
                if (first + 16 > nk) {
#pragma unroll
                    for (int j = 0; j < 16; ++j) v[j] = first + j < nk ? v[j] : 0.f;
                }
#pragma unroll
                for (int j = 0; j < 8; ++j) d[j] = pair(v[2 * j], v[2 * j + 1]);
            };
#pragma unroll
            for (int c = 0; c < 4; ++c) {
                if (key0 + c * 16 >= n_keys) break;
                uint64_t d[8];
                load_ds(key0 + c * 16, d);
#pragma unroll
                for (int j = 0; j < 8; ++j) u2[j & 1] = fma2(e[c >> 1][(c & 1) * 8 + j], d[j], u2[j & 1]);
            }
            const float2 lx = halves(add2(l2[0], l2[1])), ux = halves(add2(u2[0], u2[1]));
            sh.part[g][row][0] = mx;
            sh.part[g][row][1] = lx.x + lx.y;
            sh.part[g][row][2] = ux.x + ux.y;
            asm volatile("bar.sync %0, %1;" ::"r"(1 + quad), "n"(32 * G) : "memory");   // the G warps of this quadrant
            float mm = sh.part[0][row][0];
#pragma unroll
            for (int i = 1; i < G; ++i) mm = fmaxf(mm, sh.part[i][row][0]);
            float L = 0.f, U = 0.f;
#pragma unroll
            for (int i = 0; i < G; ++i) {
                const float f = ex2((sh.part[i][row][0] - mm) * sl2);                   // an empty share: 2^-inf = 0
                L = fmaf(sh.part[i][row][1], f, L);
                U = fmaf(sh.part[i][row][2], f, U);
            }
            const float inv_l = 1.f / L;
            const float mine = ex2((mx - mm) * sl2) * inv_l;
            const float nds = -U * inv_l * p.scale;          // -rowsum(S dS) / sqrt(d)
            const uint64_t mine2 = pair(mine, mine), nds2 = pair(nds, nds), scale2 = pair(p.scale, p.scale);
            // dM waits in tensor memory when its blocks are those of S: in columns that this thread alone reads and has read by then
            // (G = 2: its dS, G = 4: its S or dS), out of the way of dV.  (In registers it spilled: Drop QKV
            // with 126 of 196 tokens, B = 128, 105.9 -> 87.5 us; all tokens on both sides, B = 64, 136.6 -> 113.4.)
            const uint32_t parked = tmem + (G == 2 ? 128u : 0u) + (uint32_t)key0 + lane_off;
            uint8_t* blkP = gen + (uint32_t)g * p.block_bytes;
            uint8_t* blkM = gen + p.off_dm + (uint32_t)g * p.dm_stride;
            const bool row_fits = (uint32_t)row * kRowB < p.block_bytes;
#pragma unroll
            for (int c = 0; c < 4; ++c) {
                if (key0 + c * 16 >= n_keys) break;
                uint64_t d[8];
                load_ds(key0 + c * 16, d);
                uint32_t w[8], dm[8];
#pragma unroll
                for (int j = 0; j < 8; ++j) {
                    const uint64_t s2 = mul2(e[c >> 1][(c & 1) * 8 + j], mine2);        // S
                    const float2 sf = halves(s2), mf = halves(mul2(s2, fma2(d[j], scale2, nds2)));   // dM / sqrt(d)
                    w[j] = pack2(sf.x, sf.y);
                    dm[j] = pack2(mf.x, mf.y);
                }
                if (!kSeparate) ptx::tmem_st_32x8(parked + (uint32_t)(c * 8), dm);
                if (row_fits) {
#pragma unroll
                    for (int q = 0; q < 2; ++q) {
                        *reinterpret_cast<uint4*>(blkP + swz((uint32_t)row, (uint32_t)(c * 2 + q))) = make_uint4(w[q * 4], w[q * 4 + 1], w[q * 4 + 2], w[q * 4 + 3]);
                        if (kSeparate)
                            *reinterpret_cast<uint4*>(blkM + swz((uint32_t)row, (uint32_t)(c * 2 + q))) = make_uint4(dm[q * 4], dm[q * 4 + 1], dm[q * 4 + 2], dm[q * 4 + 3]);
                    }
                }
            }
            if (!kSeparate) ptx::tmem_st_wait();
            ptx::fence_async_proxy();                        // the blocks are read by the tensor core
            ptx::tc_fence_before_sync();
            __syncthreads();                                  // S and dS in tensor memory are dead from here on
            // ---- the gradient products; only the 16-row steps that hold tokens run, accumulators take turns ----
            const uint32_t id_t = ptx::umma_idesc_bf16(128, 64, true, true);             // dV, dK: both operands MN-major
            const uint32_t id_q = ptx::umma_idesc_bf16(128, 64, false, true);            // dQ: dM K-major, K MN-major
            const int KT = G == 2 ? 1 : (nk + 127) >> 7;
            // 16 rows of a token tile are 2048 bytes; 16 columns of a block 32 bytes.  (N = 64 is one block: the leading-dimension
            // offset of the B operands plays no part.)
            const uint32_t dP = ptx::umma_desc_lo(sP, p.block_bytes), dMt = ptx::umma_desc_lo(sDM, p.dm_stride), dMk = ptx::umma_desc_lo(sDM, 16);
            auto issue_dv = [&](uint32_t u, bool leader) {
                ptx::umma_bf16_warp<false>(tmem + kColDV, ptx::umma_desc_of(dP + u * 128u), ptx::umma_desc_of(dDA0 + u * 128u), id_t, (qt | (int)u) != 0, leader);
                if (G == 4 && KT > 1)
                    ptx::umma_bf16_warp<false>(tmem + kColDV + 64u, ptx::umma_desc_of(dP + (p.block_bytes >> 3) + u * 128u), ptx::umma_desc_of(dDA0 + u * 128u), id_t, (qt | (int)u) != 0, leader);
            };
            auto issue_dk = [&](uint32_t u, bool leader) {
                ptx::umma_bf16_warp<false>(tmem + kColDK, ptx::umma_desc_of(dMt + u * 128u), ptx::umma_desc_of(dQ0 + u * 128u), id_t, (qt | (int)u) != 0, leader);
                if (G == 4 && KT > 1)
                    ptx::umma_bf16_warp<false>(tmem + kColDK + 64u, ptx::umma_desc_of(dMt + (p.dm_stride >> 3) + u * 128u), ptx::umma_desc_of(dQ0 + u * 128u), id_t, (qt | (int)u) != 0, leader);
            };
            auto issue_dq = [&](uint32_t u, bool leader) {
                ptx::umma_bf16_warp<false>(tmem + kColDQ, ptx::umma_desc_of(dMk + (u >> 2) * (p.dm_stride >> 4) + (u & 3u) * 2u), ptx::umma_desc_of(dK0 + u * 128u), id_q, u != 0, leader);
            };
            const uint32_t steps = q_steps > k_steps ? q_steps : k_steps;
            if (!kSeparate) {
                if (warp == 0) {
                    const bool leader = ptx::elect_one();
                    ptx::tc_fence_after_sync();
                    for (uint32_t u = 0; u < q_steps; ++u) issue_dv(u, leader);
                    if (leader) ptx::umma_commit(ptx::smem_addr(&sh.bar_o));
                    __syncwarp();
                }
                ok = wait_products(&sh.bar_o, n_o);
                if (!ok) break;
                float dm[32];                                // (bits)
                ptx::tmem_ld_32x32(parked, dm);
                ptx::tmem_ld_wait();
#pragma unroll
                for (int c = 0; c < 8; ++c)
                    if (key0 + (c >> 1) * 16 < n_keys && row_fits)
                        *reinterpret_cast<float4*>(blkM + swz((uint32_t)row, (uint32_t)c)) = make_float4(dm[c * 4], dm[c * 4 + 1], dm[c * 4 + 2], dm[c * 4 + 3]);
                ptx::fence_async_proxy();
                ptx::tc_fence_before_sync();
                __syncthreads();
            }
            if (warp == 0) {                                 // the whole warp, of which one lane issues
                const bool leader = ptx::elect_one();
                ptx::tc_fence_after_sync();
                for (uint32_t u = 0; u < steps; ++u) {
                    if (u < q_steps) {
                        if (kSeparate) issue_dv(u, leader);
                        issue_dk(u, leader);
                    }
                    if (u < k_steps) issue_dq(u, leader);
                }
                if (leader) ptx::umma_commit(ptx::smem_addr(&sh.bar_o));
                __syncwarp();
            }
            if (!kOwn && qt + 1 == QT) zero_rows(p, &sh.walk[warp], warp, kThreads / 32, lane, false);
            ok = wait_products(&sh.bar_o, n_o);
            if (!ok) break;
            // the operands have been read: the next problem's rows may come in (the read-out stages in the S and dM blocks,
            // of which G = 2 leaves V's place alone)
            if (qt + 1 == QT && next < problems) begin_problem(cur, next, buf ^ 1);
            if constexpr (G == 4) {                          // dQ of this query tile, 16 columns a group
                float v[16];
                ptx::tmem_ld_32x16(tmem + kColDQ + (uint32_t)(g * 16) + lane_off, v);
                ptx::tmem_ld_wait();
                if (row_fits) {
                    *reinterpret_cast<uint4*>(gen + swz((uint32_t)row, (uint32_t)(g * 2))) = pack8(v);
                    *reinterpret_cast<uint4*>(gen + swz((uint32_t)row, (uint32_t)(g * 2 + 1))) = pack8(v + 8);
                }
                ptx::tc_fence_before_sync();
                __syncthreads();
                store_rows<kThreads>(p.dQ, p.ld_out, col0, gen, q_glob + qt * 128, q_here);
                __syncthreads();                             // the stage becomes S blocks (or another stage) again
            }
        }
        if (!ok) break;
        // ---- read-out: a thread holds one accumulator row, but a store that touches 32 rows costs 32 transactions, so rows
        //      go through shared memory and leave as whole 128-byte lines ----
        if constexpr (G == 2) {
            const uint32_t stage_b = p.block_bytes;          // three stages: the two S blocks and the first dM block
            float v[32];
#pragma unroll
            for (int which = 0; which < 3; ++which) {
                if (which == 2 && !kSeparate) break;
                ptx::tmem_ld_32x32(tmem + (uint32_t)(which * 64 + g * 32) + lane_off, v);
                ptx::tmem_ld_wait();
                if ((uint32_t)row * kRowB < stage_b) stage32(gen + which * stage_b, row, (uint32_t)(g * 4), v);
            }
            ptx::tc_fence_before_sync();
            __syncthreads();
#pragma unroll 1
            for (int which = 0; which < (kSeparate ? 3 : 2); ++which)      // (one loop body: copies of it cost registers)
                store_rows<kThreads>(which == 0 ? p.dV : which == 1 ? p.dK : p.dQ, p.ld_out, col0, gen + which * stage_b,
                                     which == 2 ? q_glob : k_glob, which == 2 ? nq : nk);
            if (!kSeparate) {                               // (two stages only)
                ptx::tmem_ld_32x32(tmem + (uint32_t)(128 + g * 32) + lane_off, v);
                ptx::tmem_ld_wait();
                __syncthreads();
                if ((uint32_t)row * kRowB < stage_b) stage32(gen, row, (uint32_t)(g * 4), v);
                __syncthreads();
                store_rows<kThreads>(p.dQ, p.ld_out, col0, gen, q_glob, nq);
            }
        } else {
            // group g takes dV (g even) or dK (g odd) of key tile g / 2
            const int kt = g >> 1;
            if (kt * 128 < nk) {
#pragma unroll
                for (int half = 0; half < 2; ++half) {
                    float v[32];
                    ptx::tmem_ld_32x32(tmem + ((g & 1) ? kColDK : kColDV) + (uint32_t)(kt * 64 + half * 32) + lane_off, v);
                    ptx::tmem_ld_wait();
                    stage32(gen + (uint32_t)g * kTileB, row, (uint32_t)(half * 4), v);
                }
            }
            ptx::tc_fence_before_sync();
            __syncthreads();
#pragma unroll 1
            for (int i = 0; i < 4; ++i) {
                const int first = (i >> 1) * 128;
                if (first < nk)
                    store_rows<kThreads>((i & 1) ? p.dK : p.dV, p.ld_out, col0, gen + (uint32_t)i * kTileB, k_glob + first, nk - first < 128 ? nk - first : 128);
            }
        }
        // No barrier behind the last stores: the one in front of the next problem's products keeps its writers off the stages, and
        // whoever writes this problem's half of q_glob / k_glob next does so behind a barrier of the next problem (of an empty one too).
        ptx::tc_fence_before_sync();
    }
    if (!kOwn && ok) zero_rows(p, &sh.walk[warp], warp, kThreads / 32, lane, true);                            // what the turns have left
    ptx::cp_async_wait_all();
    ptx::tc_fence_before_sync();
    __syncthreads();
    if (warp == 0) {
        ptx::tc_fence_after_sync();
        ptx::tmem_dealloc(tmem, kTmemCols);
    }
}

// ---- host side: buffer layout and launch ----
int round16(int64_t v) { return (int)((v + 15) / 16 * 16); }

template <int G, bool kSeparate>
cudaError_t launch_attention_kernel(const AttnParams& prm, int64_t q_most, int64_t k_most, uint32_t bytes, int most_bytes, cudaStream_t stream) {
    const int64_t problems = (int64_t)prm.B * prm.heads, resident = G == 2 ? 2 * kNumSMs : kNumSMs;
    const int64_t grid = problems < resident ? problems : resident;
    const auto go = [&](auto kernel, cudaError_t opt, const AttnParams& q) {
        return opt != cudaSuccess ? opt : launch_pdl(kernel, dim3((unsigned)grid), dim3(128 * G), bytes, stream, q);
    };
    // The walk is worth its reads where it shortens the longest lists: blocks that are idle while `more` others have their last problem clear
    // most of the rows.  A row costs a line of 128 bytes for each head and output that leaves it out, and some 6 lines to be found; an idle block
    // clears `worth` lines in a problem's time, twice as many where a problem has two query tiles (up to a quarter more it is given all of them: a
    // small share for the others costs these more than it saves).  Both ways were timed on 755 calls.  12 heads, 196 tokens, half of them listed, each problem its own rows -> the walk:
    // 312 problems 18.7 -> 18.4 us, 516 21.7 -> 21.0, 1536 63.4 -> 59.0; 576 on 296 blocks, few of them idle, 21.9 -> 23.2 (28.1, and 30.5 instead of
    // 18.9 for problems of 128 tokens, with all rows for the idle ones).  One block an SM: the walk wins with few idle blocks too, and without
    // any from three problems a block on (10 to 15 % of the time).
    const int64_t rows = (int64_t)prm.B * prm.N, more = problems % grid, idle = grid - more;
    const double find = prm.heads == 1 ? 1.5 : prm.heads == 2 ? 3.0 : 6.0;
    const double outside_q = prm.q_rows == nullptr ? 0.0 : 1.0 - (double)q_most / (double)prm.N;
    const double outside_k = prm.k_rows == nullptr ? 0.0 : 1.0 - (double)k_most / (double)prm.N;
    const double lines = (double)rows * (prm.q_rows == prm.k_rows ? outside_q * (3.0 * prm.heads + find)
                                                                  : outside_q * (prm.heads + find) + outside_k * (2.0 * prm.heads + find));
    const double for_idle = lines / (double)idle, for_problem = lines / (double)problems;
    const bool walk = problems > grid && (G == 2 ? more != 0 && for_idle <= 700.0 + 10.0 * for_problem
                                                 : problems > 2 * grid || for_idle <= 8000.0 + 4.0 * for_problem);
    if (!walk) return go(attention_bwd_kernel<G, kSeparate, true>, opt_in_dynamic_smem<attention_bwd_kernel<G, kSeparate, true>>(most_bytes), prm);
    AttnParams q = prm;
    const double worth = q_most > 128 ? 3800.0 : 1900.0;
    const double spare = for_idle <= 1.25 * worth ? 0.0 : (double)rows * (1.0 - worth / for_idle);      // rows that the idle blocks do not get to
    q.zero_blocks = (int)more;
    q.zero_first = more == 0 || spare <= 0.0 ? 0 : (int)((int64_t)spare / grid + 1);
    q.zero_rest = rows <= more * q.zero_first ? 0 : (int)((rows - more * q.zero_first + idle - 1) / idle);
    return go(attention_bwd_kernel<G, kSeparate, false>, opt_in_dynamic_smem<attention_bwd_kernel<G, kSeparate, false>>(most_bytes), q);
}

template <int G>
cudaError_t launch_attention(AttnParams& prm, int64_t q_most, int64_t k_most, cudaStream_t stream) {
    // most shared memory a block may ask for: half of an SM's (G = 2) or a block's limit, less the static part, the 1 KB the
    // system keeps per block and the alignment slack
    constexpr uint32_t kLimit = (G == 2 ? 233472u / 2 - 1024u : 232448u) - (uint32_t)sizeof(AttnShared<G>) - 64u - 1024u;
    prm.rq = round16(q_most);
    prm.rk = round16(k_most);
    if (G == 2) prm.rq = prm.rk = prm.rq > prm.rk ? prm.rq : prm.rk;      // one size for all: the stages hold queries or keys
    const uint32_t tile_rows = prm.rq < 128 ? (uint32_t)prm.rq : 128u;
    prm.block_bytes = tile_rows * kRowB;
    const uint32_t blocks = G == 2 ? 2u : (uint32_t)(prm.rk + 63) / 64u;
    uint32_t s_bytes = blocks * prm.block_bytes;
    if (G == 4 && s_bytes < 4 * kTileB) s_bytes = 4 * kTileB;             // the read-out stages four tiles there
    const uint32_t q_bytes = (uint32_t)prm.rq * kRowB, k_bytes = (uint32_t)prm.rk * kRowB;
    // S | dM | Q | dA | K | V: what the products read 128 rows of, whatever it holds, is followed by other buffers
    const auto layout = [&](uint32_t dm_bytes) {
        prm.off_dm = dm_bytes ? s_bytes : 0u;
        prm.off_q = s_bytes + dm_bytes;
        prm.off_da = prm.off_q + q_bytes;
        prm.off_k = prm.off_da + q_bytes;
        prm.off_v = prm.off_k + k_bytes;
        prm.dm_stride = (G == 2 && dm_bytes) ? prm.off_v - prm.off_dm : prm.block_bytes;
        prm.separate = dm_bytes ? 1 : 0;
        return prm.off_v + k_bytes;
    };
    uint32_t bytes = layout(G == 2 ? prm.block_bytes : blocks * prm.block_bytes);
    if (bytes > kLimit) bytes = layout(0u);
    // The products read 128 rows of every query tile and of every dM block (of V's place too, with G = 2), whatever the rows
    // past the tokens hold: those reads end inside the buffers that follow, or in room added here.
    const uint32_t q_tiles = (uint32_t)(prm.rq + 127) / 128u;
    const uint32_t ends[2] = {prm.off_da + q_tiles * kTileB, G == 2 && prm.separate ? prm.off_v + kTileB : 0u};
    for (uint32_t end : ends) bytes = bytes < end ? end : bytes;
    if (bytes > kLimit) return cudaErrorInvalidValue;
    return prm.separate ? launch_attention_kernel<G, true>(prm, q_most, k_most, bytes + 1024u, (int)kLimit + 1024, stream)
                        : launch_attention_kernel<G, false>(prm, q_most, k_most, bytes + 1024u, (int)kLimit + 1024, stream);
}

}  // namespace

bool attention_supported(sbp_dtype dt, int64_t head_dim) { return dt == SBP_BF16 && head_dim == kD; }
int64_t attention_max_tokens() { return kMaxTok; }

cudaError_t launch_attention_backward(const void* Q, const void* K, const void* V, int64_t ld_qkv, const void* dA, int64_t ld_da,
                                      const int32_t* q_rows, const int32_t* q_offs, const int32_t* k_rows, const int32_t* k_offs,
                                      int64_t B, int64_t N, int64_t heads, int64_t q_most, int64_t k_most, void* dQ, void* dK, void* dV,
                                      int64_t ld_out, bool zero_other_rows, int32_t* status_word, cudaStream_t stream) {
    AttnParams prm;
    prm.Q = static_cast<const __nv_bfloat16*>(Q); prm.K = static_cast<const __nv_bfloat16*>(K);
    prm.V = static_cast<const __nv_bfloat16*>(V); prm.dA = static_cast<const __nv_bfloat16*>(dA);
    prm.ld_qkv = (uint32_t)(ld_qkv / 8); prm.ld_da = (uint32_t)(ld_da / 8); prm.ld_out = (uint32_t)(ld_out / 8);
    prm.q_rows = q_rows; prm.q_offs = q_offs; prm.k_rows = k_rows; prm.k_offs = k_offs;
    prm.B = (int)B; prm.N = (int)N; prm.heads = (int)heads;
    prm.dQ = static_cast<__nv_bfloat16*>(dQ); prm.dK = static_cast<__nv_bfloat16*>(dK); prm.dV = static_cast<__nv_bfloat16*>(dV);
    prm.scale = 1.0f / sqrtf((float)kD);
    prm.status_word = status_word;
    // the zeros for the rows outside the lists are written by the same kernel, between a problem's copies and its products
    prm.zero_fill = (zero_other_rows && (q_rows != nullptr || k_rows != nullptr)) ? 1 : 0;
    return q_most <= 128 && k_most <= 128 ? launch_attention<2>(prm, q_most, k_most, stream) : launch_attention<4>(prm, q_most, k_most, stream);
}

}  // namespace sbp

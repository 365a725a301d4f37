// fp32 products on the tensor cores (tcgen05 / TMEM), without giving up fp32 precision.
//   forward  Y[m, j] = sum_i X[m, i] W[i, j] + bias[j]                        (Eq. 2)
//   dW[i, j] = sum_m X_keep[m, i] dY[keep_rows[m], j],  db[j] = sum_m dY[keep_rows[m], j]       (Eq. 5)
//   dX[keep_rows[m], i] = sum_j dY[keep_rows[m], j] W[i, j]; every other row of dX = +0.0
//
// Every operand x is written as a sum of three bf16 numbers, x = x1 + x2 + x3, each the rounded rest of the one before (8
// significant bits each, so what is left is below 2^-26 x), and a product of two of them as
//   a b = a1 b1 + (a1 b2 + a2 b1) + (a2 b2 + a1 b3 + a3 b1),
// dropping terms below 2^-26: six bf16 products with fp32 accumulation.  The parts are those of 2^16 x: bf16 numbers end at 2^-133, so that
// the third part of an x below 2^-109 would lose bits, while the last bit of any fp32 number is 2^-149 or more.  The sums are brought back by
// 2^-32.  (Sums beyond 2^96 come out infinite that way, and are made again like other sums that are not finite.)  The tensor core also
// drops sums that are subnormal: sums of 1e-39 came out as zeros.  The scaling costs 1 us of a layer's 200.
// The tensor core cuts its running sum short instead of
// rounding it, so a sum is never left in tensor memory for long: each 64-deep stage starts a fresh accumulator, the five small
// terms go in first and a1 b1 last (four steps that see the full magnitude), and the epilogue warps add the stage's result to
// their fp32 registers with rounding.
//
// A pair of blocks makes tiles of 256 x 128 with two-SM instructions.  Bound by shared memory: a 64-deep stage moves 312 KB through
// each SM (copies in 48, read back 48, planes written 72, read by the tensor core 144 less what its kept operand saves) = 2440 clocks
// at 128 bytes, against 1536 of products; measured 1.4 us.  (Copies straight to registers, 264 KB: 1.95 us, their latency shows; with the next
// stage's loads behind each conversion the registers spill.)  Measured on B200, 768 -> 3072, 3136 rows with 1568 kept, CUDA cores -> here: forward
// 299 -> 89 us, dW + db + dX 395 -> 100 (calls back to back in a graph; cold and by themselves 104 and 114); relative errors against 64-bit
// sums Y 2.5e-7 -> 0.8e-7, dW 5.0e-7 -> 1.2e-7, dX 7.0e-7 -> 1.5e-7, db 0.7e-7 -> 0.3e-7.  Over 216 shapes of 32 to 3072 channels and 32 to
// 65536 rows no output was further off than the CUDA cores'.
#include <atomic>
#include <map>
#include <tuple>
#include <type_traits>

#include "tc_ptx.cuh"
#include "zero_rows.cuh"

namespace sbp {
namespace {

constexpr int kTile = 128;                // columns of a tile, and its rows in each block of a pair (= lanes of tensor memory)
constexpr int kBK = 64;                   // reduction depth of a stage: 64 bf16 = one 128-byte swizzle row
constexpr uint32_t kRowB = 128;
constexpr uint32_t kBlock64B = 64 * kRowB;
constexpr int kEpiWarps = 8, kProducerWarps = 8, kMmaWarp = kEpiWarps + kProducerWarps;
constexpr int kProducers = 32 * kProducerWarps;
constexpr int kThreads = 32 * (kMmaWarp + 4);   // (three of the last four warps only hand their registers on)
constexpr int kLaunchRegs = 96, kEpiRegs = 104, kProducerRegs = 112, kMmaRegs = 40;
static_assert(kEpiWarps * kEpiRegs + kProducerWarps * kProducerRegs + 4 * kMmaRegs <= (kMmaWarp + 4) * kLaunchRegs,
              "registers that the block is launched with");
constexpr int kProducerBarrier = 1, kEpiBarrier = 2;

constexpr int kBCols = 64;                                                // columns of B that a block stages: half of the tile's
constexpr uint32_t kAPlane = kTile * kRowB, kBPlane = kBCols * kRowB;
constexpr uint32_t kStageBytes = 3 * (kAPlane + kBPlane);
constexpr int kStages = 2;
constexpr uint32_t kGroupBytes = kProducers * (kTile + kBCols) / 32 * 16, kSlotBytes = 3 * kGroupBytes;     // copies in flight: three half stages
constexpr uint32_t kAccs = 4, kAccCols = kTile;                           // accumulators, used in turn

// One product D[e_a, e_b] = sum_d A[e_a, d] B[e_b, d].  An operand is a row-major matrix whose rows are extent indices (depth inner)
// or depth indices (outer); a map sends a row of the matrix to the row of memory that it lives in.
struct Product {
    const float *A, *B;
    uint32_t lda, ldb;
    const int32_t *a_map, *b_map;
    int rows, cols, depth;
    int a_outer, b_outer;
    int rows_kept, depth_kept;             // bounded by the number of kept rows, which may be known on the device only
    int row_tiles, col_tiles, splits;      // splits: pieces of the depth
    float* out;
    int64_t ld_out, split_stride;
    const int32_t* out_map;
    const float* bias;
    int accumulate;
    int sum_side;                          // bias sums, over the depth: of operand A (1) or B (2), in the first tile of the other side
    float* sums;                           // [splits, extent]
    int sums_accumulate;
};

struct SplitParams {
    Product p[2];                          // p[0] first: the deeper tiles
    uint32_t items[2];
    uint32_t first, count;                 // the part of the list that this launch works through
    const int32_t* M_keep_dev;
    int64_t M_keep_cap;
    float* dX;                             // dropped rows to clear (nullptr: none)
    const int32_t* dx_rows;
    int64_t M;
    int C_in;
    int32_t* status_word;
};

// Behind it: room for the bias sums, then a byte for every item of the worker: which epilogue warps found sums that are not finite.
struct Control {
    uint64_t full_bar[kStages], empty_bar[kStages], acc_full[kAccs], acc_empty[kAccs];
    uint32_t tmem_slot;
    int abort_flag;
};
constexpr uint32_t kSumBytes = 1024 * sizeof(double);
constexpr uint32_t kFlagsAt = kStages * kStageBytes + kSlotBytes + 256 + kSumBytes;
constexpr uint32_t kMaxRounds = 1024;                                     // items of a worker in a launch: a byte each, see Control
constexpr uint32_t kSmemBytes = kFlagsAt + kMaxRounds + 1024;
static_assert(sizeof(Control) <= 256 && kSmemBytes <= 227 * 1024, "shared memory of a block");

__device__ __forceinline__ uint64_t pack2(float x, float y) {
    uint64_t r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(x), "f"(y));
    return r;
}
__device__ __forceinline__ float2 halves(uint64_t v) {
    float2 f;
    asm("mov.b64 {%0, %1}, %2;" : "=f"(f.x), "=f"(f.y) : "l"(v));
    return f;
}
__device__ __forceinline__ uint64_t add2(uint64_t a, uint64_t b) {
    uint64_t d;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}
__device__ __forceinline__ uint64_t mul2(uint64_t a, uint64_t b) {
    uint64_t d;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}
__device__ __forceinline__ uint64_t fma2(uint64_t a, uint64_t b, uint64_t c) {
    uint64_t d;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
    return d;
}
__device__ __forceinline__ uint64_t sub2(uint64_t a, uint64_t b) {
    uint64_t d;
    asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}

constexpr float kScale = 65536.f, kUnscale = 1.f / (kScale * kScale);     // of the operands before they are split, of the sums
__device__ __forceinline__ float4 scaled(float4 v) {
    const float2 a = halves(mul2(pack2(v.x, v.y), pack2(kScale, kScale))), b = halves(mul2(pack2(v.z, v.w), pack2(kScale, kScale)));
    return make_float4(a.x, a.y, b.x, b.y);
}

// two numbers to their leading bf16 parts (packed, the first in the low half); the rests replace them
__device__ __forceinline__ uint32_t take_bf16(float& x, float& y) {
    const __nv_bfloat162 v = __floats2bfloat162_rn(x, y);
    const uint32_t b = *reinterpret_cast<const uint32_t*>(&v);
    x -= __uint_as_float(b << 16);
    y -= __uint_as_float(b & 0xffff0000u);
    return b;
}

// Global -> shared memory -> registers -> planes, one operand: kVecs 16-byte vectors a thread and stage, for 16 kVecs extent
// indices.  A thread copies (cp.async) into slots of its own and reads them back itself, so that nothing but its own copies has to be
// waited for: shared memory serves as the registers that three half stages of copies in flight would need.
template <int kVecs, bool kOuter>
struct Feed {
    static constexpr int kExtent = 16 * kVecs, kHalf = kVecs / 2;         // half a stage: every other group of copies
    static constexpr int kPerRow = kOuter ? kExtent / 4 : kBK / 4;         // vectors of a row of the matrix
    static constexpr int kStep = kProducers / kPerRow;                    // rows between a thread's vectors
    static_assert(kStep % 8 == 0, "a thread's rows have the same place in the swizzle");
    int32_t row[kOuter ? kHalf : kVecs];                                  // rows of memory, -1: none.  Outer: of the half stage copied next
    const float* at;                                                      // the thread's place in a row: inner, at the depth copied next
    int left;                                                             // indices from there to the end of the row
    int d;                                                                // outer: depth of the rows above

    __device__ __forceinline__ void start(const float* base, const int32_t* map, int e0, int extent, int d_begin, int d_end, int t) {
        const int c = t % kPerRow * 4;
        at = base + (kOuter ? e0 : d_begin) + c;
        left = (kOuter ? extent - e0 : d_end - d_begin) - c;
        d = d_begin + t / kPerRow;
        if constexpr (kOuter) {
            find_rows(map, d_end);
        } else {
#pragma unroll
            for (int i = 0; i < kVecs; ++i) {
                const int e = e0 + t / kPerRow + i * kStep;
                row[i] = e < extent ? mapped_row(map, e) : -1;
            }
        }
    }
    __device__ __forceinline__ void find_rows(const int32_t* map, int d_end) {
#pragma unroll
        for (int i = 0; i < kHalf; ++i) row[i] = d + i * kStep < d_end ? mapped_row(map, d + i * kStep) : -1;
    }
    // copies half H of the stage reached into the slots at `to`, and moves on to the half behind it
    template <int H>
    __device__ __forceinline__ void copy(uint32_t to, const float* base, uint32_t ld, const int32_t* map, int d_end) {
#pragma unroll
        for (int i = 0; i < kHalf; ++i) {
            const int32_t r = row[kOuter ? i : H * kHalf + i];
            const bool in = r >= 0 && left > 0;
            ptx::cp_async_16(to + i * (kProducers * 16), in ? at + (uint64_t)(uint32_t)r * ld : base, in ? 16u : 0u);
        }
        if constexpr (kOuter) {
            d += kHalf * kStep;
            find_rows(map, d_end);
        } else if constexpr (H == 1) {
            at += kBK;
            left -= kBK;
        }
    }
    // half a stage from the slots at `from`
    static __device__ __forceinline__ void read(float4 (&x)[kHalf], uint32_t from) {
#pragma unroll
        for (int i = 0; i < kHalf; ++i)
            asm volatile("ld.shared.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(x[i].x), "=f"(x[i].y), "=f"(x[i].z), "=f"(x[i].w) : "r"(from + i * (kProducers * 16)));
    }
    // Half H of a stage to three planes, `plane` bytes apart, in the layouts the tensor core reads: K-major rows of 64 depths (depth
    // inner), or MN-major blocks of 64 extent indices with a depth a row (outer); 128-byte swizzle.
    template <int H>
    static __device__ __forceinline__ void put(float4 (&x)[kHalf], uint32_t planes, uint32_t plane, int t) {
        const uint32_t q = t % kPerRow, r = t / kPerRow;
        const uint32_t to = planes + (kOuter ? q / 16 : 0u) * kBlock64B + (r + H * kHalf * kStep) * kRowB + ((((q % 16) >> 1) ^ (r & 7u)) << 4) + (q & 1u) * 8;
#pragma unroll
        for (int i = 0; i < kHalf; ++i) x[i] = scaled(x[i]);
#pragma unroll
        for (int s = 0; s < 3; ++s)
#pragma unroll
            for (int i = 0; i < kHalf; ++i) {
                const uint32_t lo = take_bf16(x[i].x, x[i].y), hi = take_bf16(x[i].z, x[i].w);
                asm volatile("st.shared.v2.b32 [%0], {%1, %2};" ::"r"(to + i * (kStep * kRowB) + s * plane), "r"(lo), "r"(hi) : "memory");
            }
    }
};

// Sums of the four columns of a thread: every addition's rounding error (Knuth's TwoSum) is collected beside the sum, so that a piece's sums
// carry one rounding.  (Adding a stage's rows first and compensating once a stage left db 10 % further from 64-bit sums than the CUDA
// cores' where few pieces add up.)
struct ColumnSums {
    uint64_t sum[2] = {0ull, 0ull}, lost[2] = {0ull, 0ull};               // columns in pairs
    template <int n>
    __device__ __forceinline__ void add(const float4 (&x)[n]) {
#pragma unroll
        for (int i = 0; i < n; ++i)
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const uint64_t v = h ? pack2(x[i].z, x[i].w) : pack2(x[i].x, x[i].y);
                const uint64_t t = add2(sum[h], v), z = sub2(t, sum[h]);
                lost[h] = add2(lost[h], add2(sub2(sum[h], sub2(t, z)), sub2(v, z)));
                sum[h] = t;
            }
    }
    // sum c in 64 bits; an infinite sum has lost nothing
    __device__ __forceinline__ double total(int c) const {
        const float2 s = halves(sum[c / 2]), l = halves(lost[c / 2]);
        const float a = c % 2 ? s.y : s.x, b = c % 2 ? l.y : l.x;
        return (double)a + (fabsf(b) < INFINITY ? (double)b : 0.0);
    }
};

// an item of the list: one tile of a product, over one piece of its depth
struct Item {
    int e_a0, e_b0, d_begin, d_end;
    int rows;                              // valid rows of the product
    uint32_t num_kb;
    int split;
    bool first_row, first_col;             // tiles of the first row / column of tiles
    bool none;                             // nothing to write
};
__device__ __forceinline__ Item item_of(const Product& p, uint32_t idx, int M_keep) {
    Item it;
    it.split = (int)(idx % (uint32_t)p.splits);
    const uint32_t tile = idx / (uint32_t)p.splits, row = tile / (uint32_t)p.col_tiles, col = tile - row * (uint32_t)p.col_tiles;
    it.first_row = row == 0;
    it.first_col = col == 0;
    it.e_a0 = (int)row * 2 * kTile;
    it.e_b0 = (int)col * kTile;
    it.rows = p.rows_kept && M_keep < p.rows ? M_keep : p.rows;
    const int depth = p.depth_kept && M_keep < p.depth ? M_keep : p.depth;
    const int kbs = (depth + kBK - 1) / kBK, per = (kbs + p.splits - 1) / p.splits * kBK;
    it.d_begin = (int64_t)per * it.split < depth ? per * it.split : depth;
    it.d_end = depth - it.d_begin > per ? it.d_begin + per : depth;
    it.none = it.e_a0 >= it.rows;
    it.num_kb = it.none ? 0u : (uint32_t)((it.d_end - it.d_begin + kBK - 1) / kBK);
    return it;
}

// position in the list of the n-th item of a worker: there and back again, so that a round's longer items go with the next one's shorter ones
__device__ __forceinline__ uint32_t list_position(uint32_t n, uint32_t worker, uint32_t workers) {
    return n * workers + ((n & 1u) ? workers - 1u - worker : worker);
}

// position in the whole list of the n-th item of a worker; past its part: none
__device__ __forceinline__ bool next_item(const SplitParams& prm, uint32_t n, uint32_t worker, uint32_t workers, uint32_t& q) {
    const uint32_t at = list_position(n, worker, workers);
    q = prm.first + at;
    return at < prm.count;
}

// ---- sums that did not come out finite ----
// With an infinite (or all but infinite) operand the parts are infinity and NaN, whatever the product itself is.  Such sums are made again
// with FMAs once the block's list is done: the products then wait for nobody (their waits are bounded, and this work is as deep as the reduction).
// The eight epilogue warps take 64 rows x 128 columns at a time, 16 columns a warp and 8 x 4 sums a thread (4 x 4: twice the time, shared
// memory reads), over stages of 64 that they copy into the ring; each stage's sums are added to totals in shared memory, which leaves the registers
// to the FMAs.  768 -> 3072, 3136 rows with 1568 kept, forward and dW + db + dX, finite 110 and 114 us: one infinite row of X and dY 204 and 642,
// all NaN 227 and 167, all sums (operands of 2^114) 987 and 1121; 25000 kept rows, dW + db + dX, finite 1.15 ms: one infinite row 6.5, all NaN 1.3.
// (One thread a sum, to the end whatever it had become, took 13 and 69 ms for the infinite row at 1568, 92 and 89 for the NaNs.)
constexpr int kStripRows = 64, kPlainStages = 3, kPlainLd = kBK + 4;     // a row of an operand stored by extent: 16 bytes more, other banks
constexpr uint32_t kPlainA = kStripRows * kPlainLd * 4, kPlainB = kTile * kPlainLd * 4, kPlainStage = kPlainA + kPlainB;
constexpr uint32_t kTotalsAt = kPlainStages * kPlainStage;
static_assert(kTotalsAt + kStripRows * kTile * 4 <= kStages * kStageBytes + kSlotBytes, "the ring holds the stages and the totals");

template <bool kOuter, int kExtent>
__device__ __forceinline__ void copy_plain(uint32_t to, const float* base, uint32_t ld, const int32_t* map, int e0, int extent, int d0, int d_end, int t) {
    constexpr int kPerRow = kOuter ? kExtent / 4 : kBK / 4, kRows = kOuter ? kBK : kExtent;
#pragma unroll 2
    for (int i = 0; i < kRows * kPerRow / (32 * kEpiWarps); ++i) {
        const int v = t + i * 32 * kEpiWarps, r = v / kPerRow, c = v % kPerRow * 4;
        const int row = (kOuter ? d0 : e0) + r, col = (kOuter ? e0 : d0) + c;
        const bool in = row < (kOuter ? d_end : extent) && col < (kOuter ? extent : d_end);
        ptx::cp_async_16(to + (r * (kOuter ? kExtent : kPlainLd) + c) * 4, in ? base + (int64_t)mapped_row(map, row) * ld + col : base, in ? 16u : 0u);
    }
}
// rows [m0, m0 + 64) of an item; want: the warps' regions (32 rows x 64 columns) among them that are written
template <bool kAOuter, bool kBOuter>
__device__ __forceinline__ void plain_strip(const Product& p, const Item& item, int m0, uint32_t want, uint32_t ring) {
    int t;                                                                 // read anew: what follows from it would else be kept from the kernel's start
    asm volatile("mov.u32 %0, %%tid.x;" : "=r"(t));
    const int warp = t >> 5, lane = t & 31;                                // the epilogue warps are the block's first
    const uint32_t a_at = (kAOuter ? (lane >> 2) * 4 : (lane >> 2) * kPlainLd) * 4;
    const uint32_t b_at = kPlainA + (kBOuter ? warp * 16 + (lane & 3) * 4 : (warp * 16 + (lane & 3)) * kPlainLd) * 4;
    const uint32_t totals = ring + kTotalsAt + t * 8;
    const auto row_of = [&](int i) { return kAOuter ? (lane >> 2) * 4 + i % 4 + i / 4 * 32 : (lane >> 2) + 8 * i; };
    const auto col_of = [&](int i) { return item.e_b0 + warp * 16 + (kBOuter ? (lane & 3) * 4 + i : (lane & 3) + 4 * i); };
    // whether the sum of row i and column c is one to write: regions in `want` are (row / 32) + 2 (column / 64)
    const auto mine = [&](int i, int c) { return ((want >> (row_of(i) / 32 + warp / 4 * 2)) & 1u) != 0 && m0 + row_of(i) < item.rows && col_of(c) < p.cols; };
    const auto copy = [&](uint32_t k) {
        if (k < item.num_kb) {
            const uint32_t to = ring + k % kPlainStages * kPlainStage;
            const int d0 = item.d_begin + (int)k * kBK;
            copy_plain<kAOuter, kStripRows>(to, p.A, p.lda, p.a_map, m0, item.rows, d0, item.d_end, t);
            copy_plain<kBOuter, kTile>(to + kPlainA, p.B, p.ldb, p.b_map, item.e_b0, p.cols, d0, item.d_end, t);
        }
        ptx::cp_async_commit();
    };
    const auto read2 = [](uint32_t from) {
        float2 v;
        asm volatile("ld.shared.v2.f32 {%0, %1}, [%2];" : "=f"(v.x), "=f"(v.y) : "r"(from));
        return v;
    };
    const auto read4 = [](uint32_t from) {
        float4 v;
        asm volatile("ld.shared.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "r"(from));
        return v;
    };
#pragma unroll 1
    for (uint32_t ahead = 0; ahead < item.num_kb + kPlainStages - 1; ++ahead) {
        copy(ahead);
        if (ahead < kPlainStages - 1) continue;
        const uint32_t k = ahead - (kPlainStages - 1);
        ptx::cp_async_wait<kPlainStages - 1>();
        ptx::bar_named<kEpiBarrier, 32 * kEpiWarps>();
        const uint32_t stage = ring + k % kPlainStages * kPlainStage;
        uint64_t s[4][4] = {};                                             // rows in pairs
#pragma unroll 2
        for (int d = 0; d < kBK; d += 2) {
            float2 a2[8], b2[4];                                           // inner: two depths of each row; outer: four rows of each depth
#pragma unroll
            for (int i = 0; i < (kAOuter ? 0 : 8); ++i) a2[i] = read2(stage + a_at + (i * 8 * kPlainLd + d) * 4);
#pragma unroll
            for (int i = 0; i < (kBOuter ? 0 : 4); ++i) b2[i] = read2(stage + b_at + (i * 4 * kPlainLd + d) * 4);
#pragma unroll
            for (int j = 0; j < 2; ++j) {
                float4 a4[2], b4;
#pragma unroll
                for (int i = 0; i < (kAOuter ? 2 : 0); ++i) a4[i] = read4(stage + a_at + ((d + j) * kStripRows + i * 32) * 4);
                if (kBOuter) b4 = read4(stage + b_at + (d + j) * kTile * 4);
#pragma unroll
                for (int r = 0; r < 4; ++r) {
                    const uint64_t rows = kAOuter ? (r % 2 ? pack2(a4[r / 2].z, a4[r / 2].w) : pack2(a4[r / 2].x, a4[r / 2].y))
                                                  : (j ? pack2(a2[2 * r].y, a2[2 * r + 1].y) : pack2(a2[2 * r].x, a2[2 * r + 1].x));
#pragma unroll
                    for (int c = 0; c < 4; ++c) {
                        const float col = kBOuter ? (c == 0 ? b4.x : c == 1 ? b4.y : c == 2 ? b4.z : b4.w) : (j ? b2[c].y : b2[c].x);
                        s[r][c] = fma2(rows, pack2(col, col), s[r][c]);
                    }
                }
            }
        }
        bool open = false;                                                 // a NaN stays one: nothing is left to do once all sums are
#pragma unroll
        for (int r = 0; r < 4; ++r)
#pragma unroll
            for (int c = 0; c < 4; ++c) {
                const uint32_t at = totals + (r * 4 + c) * (32 * kEpiWarps * 8);
                uint64_t sum = 0ull;
                if (k != 0) asm volatile("ld.shared.b64 %0, [%1];" : "=l"(sum) : "r"(at));
                sum = add2(sum, s[r][c]);
                asm volatile("st.shared.b64 [%0], %1;" ::"r"(at), "l"(sum) : "memory");
                const float2 f = halves(sum);
                open = open || (f.x == f.x && mine(2 * r, c)) || (f.y == f.y && mine(2 * r + 1, c));
            }
        if (!ptx::bar_or<kEpiBarrier, 32 * kEpiWarps>(open)) break;        // (and the stage has been read)
    }
    ptx::cp_async_wait<0>();
    ptx::bar_named<kEpiBarrier, 32 * kEpiWarps>();                         // before the next strip's copies
#pragma unroll 1
    for (int i = 0; i < 8; ++i) {
        if (m0 + row_of(i) >= item.rows) continue;
        float* dst = p.out + (int64_t)item.split * p.split_stride + (int64_t)mapped_row(p.out_map, m0 + row_of(i)) * p.ld_out;
#pragma unroll 1
        for (int c = 0; c < 4; ++c) {
            if (!mine(i, c)) continue;
            float v;
            asm volatile("ld.shared.f32 %0, [%1];" : "=f"(v) : "r"(totals + (i / 2 * 4 + c) * (32 * kEpiWarps * 8) + i % 2 * 4));
            if (p.bias != nullptr) v += __ldg(p.bias + col_of(c));
            dst[col_of(c)] = p.accumulate ? dst[col_of(c)] + v : v;
        }
    }
}

// every strip that the epilogue warps have noted
__device__ __forceinline__ void make_plain_sums(const SplitParams& prm, int M_keep) {
    extern __shared__ uint8_t smem_raw[];
    const uint32_t raw = ptx::smem_addr(smem_raw), ring = (raw + 1023u) & ~1023u, rank = ptx::cluster_ctarank();
    const uint32_t workers = gridDim.x >> 1, worker = blockIdx.x >> 1;
    for (uint32_t n = 0; n * workers < prm.count; ++n) {
        uint32_t warps;
        asm volatile("ld.shared.u8 %0, [%1];" : "=r"(warps) : "r"(ring + kFlagsAt + n));
        uint32_t q;
        if (warps == 0 || !next_item(prm, n, worker, workers, q)) continue;
        const Product& p = prm.p[q < prm.items[0] ? 0 : 1];
        const Item item = item_of(p, q < prm.items[0] ? q : q - prm.items[0], M_keep);
        for (int s = 0; s < kTile / kStripRows; ++s) {                     // warp w has rows 32 (w % 4) + {0..31}, half w / 4 of the columns
            const uint32_t want = ((warps >> (2 * s)) & 3u) | ((warps >> (2 * s + 4)) & 3u) << 2;
            if (want == 0) continue;
            const int m0 = item.e_a0 + (int)rank * kTile + s * kStripRows;
            if (p.a_outer) plain_strip<true, true>(p, item, m0, want, ring);
            else if (p.b_outer) plain_strip<false, true>(p, item, m0, want, ring);
            else plain_strip<false, false>(p, item, m0, want, ring);
        }
    }
}

// A producer thread's part of one item: its vectors of both operands, stage after stage.  False when a wait gave up.
template <bool kAOuter, bool kBOuter>
__device__ __forceinline__ bool produce(const Product& p, const Item& item, uint32_t ring, Control* ctl, double* sums_s, uint32_t rank, uint32_t& it,
                                        int32_t* status_word) {
    using FA = Feed<kTile / 16, kAOuter>;
    using FB = Feed<kBCols / 16, kBOuter>;
    const int t = (int)threadIdx.x - 32 * kEpiWarps, lane = threadIdx.x & 31;
    const uint32_t slots = ring + kStages * kStageBytes + (uint32_t)t * 16, b_slot = FA::kHalf * (kProducers * 16);
    FA fa;
    FB fb;
    const int e_a0 = item.e_a0 + (int)rank * kTile, e_b0 = item.e_b0 + (int)rank * kBCols;
    const int side = (kAOuter && p.sum_side == 1 && item.first_col) ? 1 : (kBOuter && p.sum_side == 2 && item.first_row) ? 2 : 0;
    ColumnSums cs;
    bool ok = true;
    // group n of copies: half n % 2 of stage n / 2, in slots n % 3
    uint32_t copied = 0;                                                   // stages copied in full
    const auto copy = [&](auto half, uint32_t slot) {
        constexpr int H = decltype(half)::value;
        if (copied < item.num_kb) {
            fa.template copy<H>(slots + slot * kGroupBytes, p.A, p.lda, p.a_map, item.d_end);
            fb.template copy<H>(slots + slot * kGroupBytes + b_slot, p.B, p.ldb, p.b_map, item.d_end);
        }
        ptx::cp_async_commit();
        if (H == 1) ++copied;
    };
    const std::integral_constant<int, 0> first{};
    const std::integral_constant<int, 1> second{};
    if (item.num_kb > 0) {
        fa.start(p.A, p.a_map, e_a0, item.rows, item.d_begin, item.d_end, t);
        fb.start(p.B, p.b_map, e_b0, p.cols, item.d_begin, item.d_end, t);
    }
    copy(first, 0);
    copy(second, 1);
    copy(first, 2);
    uint32_t slot = 0;
    for (uint32_t k = 0; k < item.num_kb; ++k, ++it) {
        const uint32_t s = it % kStages, stage = ring + s * kStageBytes;
        float4 xa[FA::kHalf], xb[FB::kHalf];
        const auto read = [&] {
            ptx::cp_async_wait<2>();
            FA::read(xa, slots + slot * kGroupBytes);
            FB::read(xb, slots + slot * kGroupBytes + b_slot);
            if (kAOuter && side == 1) cs.add(xa);
            if (kBOuter && side == 2) cs.add(xb);
        };
        read();
        ok = ptx::mbar_wait(ptx::smem_addr(&ctl->empty_bar[s]), ((it / kStages) & 1u) ^ 1u, &ctl->abort_flag, status_word);
        ok = __all_sync(0xffffffffu, ok);
        if (!ok) break;
        FA::template put<0>(xa, stage, kAPlane, t);
        FB::template put<0>(xb, stage + 3 * kAPlane, kBPlane, t);
        copy(second, slot);
        slot = slot == 2 ? 0 : slot + 1;
        read();
        FA::template put<1>(xa, stage, kAPlane, t);
        FB::template put<1>(xb, stage + 3 * kAPlane, kBPlane, t);
        copy(first, slot);
        slot = slot == 2 ? 0 : slot + 1;
        __syncwarp();
        if (lane == 0) ptx::mbar_arrive(ptx::smem_addr(&ctl->full_bar[s]));
    }
    ptx::cp_async_wait<0>();
    if (kAOuter && kBOuter && side != 0) {
        // thread t holds extent indices 4 (t % kPerRow) + {0..3} over its share of the depth
        const int extent = side == 1 ? kTile : kBCols, per_row = extent / 4;
        double* to = sums_s + (t / per_row) * extent + (t % per_row) * 4;
#pragma unroll
        for (int c = 0; c < 4; ++c) to[c] = cs.total(c);
    }
    ok = !ptx::bar_or<kProducerBarrier, kProducers>(!ok);                   // the producers go on, or give up, together
    if (kAOuter && kBOuter && side != 0 && ok) {
        const int extent = side == 1 ? kTile : kBCols;
        const int e = (side == 1 ? e_a0 : e_b0) + t, all = side == 1 ? p.rows : p.cols;
        if (t < extent && e < all) {
            double total = 0.0;
            for (int g = 0; g < 1024 / extent; ++g) total += sums_s[g * extent + t];
            float* o = p.sums + (int64_t)item.split * all + e;
            *o = p.sums_accumulate ? *o + (float)total : (float)total;
        }
        ptx::bar_named<kProducerBarrier, kProducers>();                    // read before the next item's sums replace them
    }
    return ok;
}

__global__ void __launch_bounds__(kThreads, 1)
split_products_kernel(const __grid_constant__ SplitParams prm) {
    extern __shared__ uint8_t smem_raw[];
    const int warp = __shfl_sync(0xffffffffu, (int)(threadIdx.x >> 5), 0), lane = threadIdx.x & 31;
    const uint32_t rank = ptx::cluster_ctarank();                          // 0: the block that issues the products
    const uint32_t workers = gridDim.x >> 1, worker = blockIdx.x >> 1;
    const uint32_t raw = ptx::smem_addr(smem_raw), ring = (raw + 1023u) & ~1023u;
    uint8_t* tail = smem_raw + (ring - raw) + kStages * kStageBytes + kSlotBytes;
    Control* ctl = reinterpret_cast<Control*>(tail);
    double* sums_s = reinterpret_cast<double*>(tail + 256);

    pdl_launch_dependents();
    if (threadIdx.x == 0) {
        for (int s = 0; s < kStages; ++s) {
            ptx::mbar_init(ptx::smem_addr(&ctl->full_bar[s]), kProducerWarps + (rank == 0 ? 1 : 0));
            ptx::mbar_init(ptx::smem_addr(&ctl->empty_bar[s]), 1);
        }
        for (uint32_t a = 0; a < kAccs; ++a) {
            ptx::mbar_init(ptx::smem_addr(&ctl->acc_full[a]), 1);
            ptx::mbar_init(ptx::smem_addr(&ctl->acc_empty[a]), 2 * kEpiWarps);
        }
        ctl->abort_flag = 0;
        ptx::fence_mbar_init();
    }
    for (uint32_t i = threadIdx.x; i < kMaxRounds / 4; i += kThreads) reinterpret_cast<uint32_t*>(tail + 256 + kSumBytes)[i] = 0u;
    if (warp == kMmaWarp) ptx::tmem_alloc_pair(ptx::smem_addr(&ctl->tmem_slot), 512);
    ptx::tc_fence_before_sync();
    __syncthreads();
    ptx::cluster_sync_all();                                               // the peer's barriers exist before anything is sent to them
    ptx::tc_fence_after_sync();
    const uint32_t tmem = *reinterpret_cast<volatile uint32_t*>(&ctl->tmem_slot);
    int32_t* status_word = prm.status_word;
    pdl_wait();
    const bool skip_all = status_word != nullptr && *reinterpret_cast<volatile int32_t*>(status_word) != 0;
    const int M_keep = (int)load_m_keep(prm.M_keep_dev, prm.M_keep_cap);

    if (warp >= kMmaWarp) asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(kMmaRegs));
    if (skip_all || warp > kMmaWarp) {
        // an earlier check failed: leave every output untouched
    } else if (warp == kMmaWarp) {
        const bool leader = ptx::elect_one();
        uint32_t it = 0;
        bool ok = true;
        for (uint32_t n = 0; ok && n * workers < prm.count; ++n) {
            uint32_t q;
            if (!next_item(prm, n, worker, workers, q)) continue;
            const Product& p = prm.p[q < prm.items[0] ? 0 : 1];
            const Item item = item_of(p, q < prm.items[0] ? q : q - prm.items[0], M_keep);
            // depth inner: a 16-deep slice is 32 bytes along the swizzled rows; outer: 16 rows, 64-wide blocks 8 KB apart
            const uint32_t idesc = ptx::umma_idesc_bf16(2 * kTile, kTile, p.a_outer != 0, p.b_outer != 0);
            const uint32_t a_step = p.a_outer ? 128u : 2u, b_step = p.b_outer ? 128u : 2u;
            const uint32_t a_lo = ptx::umma_desc_lo(ring, p.a_outer ? kBlock64B : 16u);
            const uint32_t b_lo = ptx::umma_desc_lo(ring + 3 * kAPlane, p.b_outer ? kBlock64B : 16u);
            for (uint32_t k = 0; k < item.num_kb; ++k, ++it) {
                const uint32_t s = it % kStages, acc = it % kAccs;
                ok = ptx::mbar_wait(ptx::smem_addr(&ctl->full_bar[s]), (it / kStages) & 1u, &ctl->abort_flag, status_word);
                ptx::fence_async_proxy();                                  // the planes are read by the tensor core
                if (rank != 0) {                                           // the odd block's planes are complete: tell the even one
                    ok = __all_sync(0xffffffffu, ok);
                    if (!ok) break;
                    if (leader) ptx::mbar_arrive_cluster(ptx::map_to_cta(ptx::smem_addr(&ctl->full_bar[s]), 0));
                    __syncwarp();
                    continue;
                }
                ok = ok && ptx::mbar_wait(ptx::smem_addr(&ctl->acc_empty[acc]), ((it / kAccs) & 1u) ^ 1u, &ctl->abort_flag, status_word);
                ok = __all_sync(0xffffffffu, ok);
                if (!ok) break;
                ptx::tc_fence_after_sync();
                const uint32_t a = a_lo + s * (kStageBytes >> 4), b = b_lo + s * (kStageBytes >> 4), d = tmem + acc * kAccCols;
                // Every slice's small products first, a1 b1 of all slices last.  Products that share a part of A follow one another, so that
                // it is read from shared memory once for both.
                const auto a_at = [&](uint32_t plane, uint32_t u) { return ptx::umma_desc_of(a + plane * (kAPlane >> 4) + u * a_step); };
                const auto b_at = [&](uint32_t plane, uint32_t u) { return ptx::umma_desc_of(b + plane * (kBPlane >> 4) + u * b_step); };
#pragma unroll
                for (uint32_t u = 0; u < 4; ++u) {
                    ptx::umma_bf16_pair_warp<0>(d, a_at(2, u), b_at(0, u), idesc, u != 0, leader);
                    ptx::umma_bf16_pair_warp<1>(d, a_at(1, u), b_at(1, u), idesc, true, leader);
                    ptx::umma_bf16_pair_warp<2>(d, a_at(1, u), b_at(0, u), idesc, true, leader);
                    ptx::umma_bf16_pair_warp<1>(d, a_at(0, u), b_at(2, u), idesc, true, leader);
                    ptx::umma_bf16_pair_warp<2>(d, a_at(0, u), b_at(1, u), idesc, true, leader);
                }
#pragma unroll
                for (uint32_t u = 0; u < 4; ++u) ptx::umma_bf16_pair_warp<0>(d, a_at(0, u), b_at(0, u), idesc, true, leader);
                if (leader) {
                    ptx::umma_commit_pair(ptx::smem_addr(&ctl->empty_bar[s]));
                    ptx::umma_commit_pair(ptx::smem_addr(&ctl->acc_full[acc]));
                }
                __syncwarp();
            }
        }
    } else if (warp >= kEpiWarps) {
        asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(kProducerRegs));
        uint32_t it = 0;
        bool ok = true;
        for (uint32_t n = 0; ok && n * workers < prm.count; ++n) {
            uint32_t q;
            if (!next_item(prm, n, worker, workers, q)) continue;
            const Product& p = prm.p[q < prm.items[0] ? 0 : 1];
            const Item item = item_of(p, q < prm.items[0] ? q : q - prm.items[0], M_keep);
            if (p.a_outer) ok = produce<true, true>(p, item, ring, ctl, sums_s, rank, it, status_word);
            else if (p.b_outer) ok = produce<false, true>(p, item, ring, ctl, sums_s, rank, it, status_word);
            else ok = produce<false, false>(p, item, ring, ctl, sums_s, rank, it, status_word);
        }
    } else {
        asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(kEpiRegs));
        // ---------------- epilogue warps: first the zeros of the dropped rows, an equal share each ----------------
        if (prm.dX != nullptr) {
            const int quads = prm.C_in / 4, lanes = quads >= 32 ? 32 : 8;
            const int64_t shares = (int64_t)gridDim.x * kEpiWarps, per = (prm.M + shares - 1) / shares;
            const int64_t lo = per * ((int64_t)blockIdx.x * kEpiWarps + warp), hi = lo + per < prm.M ? lo + per : prm.M;
            warp_visit_dropped_rows(prm.dx_rows, M_keep, lo, hi, lane, [&](int64_t base, uint32_t todo) {
                if (lanes == 8) {                                          // short rows go four to a store instruction
                    for (int bit = lane >> 3; bit < 32; bit += 4)
                        if ((todo >> bit) & 1u)
                            for (int v = lane & 7; v < quads; v += 8) ptx::st_global_v4(prm.dX + (base + bit) * prm.C_in + v * 4, 0u, 0u, 0u, 0u);
                    return;
                }
                for (; todo; todo &= todo - 1u) {
                    float* row = prm.dX + (base + __ffs(todo) - 1) * prm.C_in;
                    for (int v = lane; v < quads; v += 32) ptx::st_global_v4(row + v * 4, 0u, 0u, 0u, 0u);
                }
            });
        }
        const uint32_t quad = warp & 3, half = warp >> 2;                  // TMEM lane quadrant; which 64 columns
        const uint32_t lane_off = (quad * 32u) << 16;
        uint32_t it = 0;
        bool ok = true;
        for (uint32_t n = 0; ok && n * workers < prm.count; ++n) {
            uint32_t q;
            if (!next_item(prm, n, worker, workers, q)) continue;
            const Product& p = prm.p[q < prm.items[0] ? 0 : 1];
            const Item item = item_of(p, q < prm.items[0] ? q : q - prm.items[0], M_keep);
            if (item.none) continue;
            uint64_t tot[32];
#pragma unroll
            for (int j = 0; j < 32; ++j) tot[j] = 0ull;
            for (uint32_t k = 0; k < item.num_kb; ++k, ++it) {
                const uint32_t acc = it % kAccs;
                ok = ptx::mbar_wait(ptx::smem_addr(&ctl->acc_full[acc]), (it / kAccs) & 1u, &ctl->abort_flag, status_word);
                ok = __all_sync(0xffffffffu, ok);
                if (!ok) break;
                ptx::tc_fence_after_sync();
                const uint32_t taddr = tmem + acc * kAccCols + half * 64u + lane_off;
#pragma unroll
                for (int c = 0; c < 4; ++c) {
                    float x[16];
                    ptx::tmem_ld_32x16(taddr + c * 16u, x);
                    ptx::tmem_ld_wait();
#pragma unroll
                    for (int j = 0; j < 8; ++j) tot[c * 8 + j] = add2(tot[c * 8 + j], pack2(x[2 * j], x[2 * j + 1]));
                }
                ptx::tc_fence_before_sync();
                __syncwarp();
                if (lane == 0) ptx::mbar_arrive_cluster(ptx::map_to_cta(ptx::smem_addr(&ctl->acc_empty[acc]), 0));
            }
            if (!ok) break;
            const int m = item.e_a0 + (int)rank * kTile + (int)quad * 32 + lane, n0 = item.e_b0 + (int)half * 64;
            uint64_t z2 = 0ull;                                            // zeros times the sums
#pragma unroll
            for (int j = 0; j < 32; ++j) z2 = fma2(tot[j], 0ull, z2);
            const float2 z = halves(z2);
            // Not finite: all sums of this warp are made again below, and nothing is written here.  (A branch for the note costs spilled registers.)
            const bool again = __any_sync(0xffffffffu, m < item.rows && n0 < p.cols && !(z.x + z.y == 0.f));
            asm volatile("{\n\t.reg .pred q;\n\tsetp.ne.b32 q, %2, 0;\n\t@q red.shared.or.b32 [%0], %1;\n\t}"
                         ::"r"(ring + kFlagsAt + n / 4 * 4), "r"(1u << (8 * (n % 4) + warp)), "r"((uint32_t)(again && lane == 0)) : "memory");
            if (again || m >= item.rows || n0 >= p.cols) continue;
            float* dst = p.out + (int64_t)item.split * p.split_stride + (int64_t)mapped_row(p.out_map, m) * p.ld_out + n0;
            const int cols = p.cols - n0 < 64 ? p.cols - n0 : 64;
            const bool wide = (reinterpret_cast<uintptr_t>(dst) & 31u) == 0;
#pragma unroll
            for (int j = 0; j < 8; ++j) {                                  // a row's sums leave eight, a whole sector, at a time
                if (j * 8 >= cols) break;
                float v[8];
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    const float2 f = halves(tot[4 * j + i]);
                    v[2 * i] = f.x * kUnscale;
                    v[2 * i + 1] = f.y * kUnscale;
                }
                const int n8 = cols - j * 8 < 8 ? 4 : 8;
                if (p.bias != nullptr) {
#pragma unroll
                    for (int i = 0; i < 8; ++i) v[i] += i < n8 ? __ldg(p.bias + n0 + j * 8 + i) : 0.f;
                }
                float* o = dst + j * 8;
                if (p.accumulate) {
#pragma unroll
                    for (int i = 0; i < 8; ++i)
                        if (i < n8) v[i] = o[i] + v[i];
                }
                if (wide && n8 == 8) {
                    asm volatile("st.global.v8.f32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};" ::"l"(o), "f"(v[0]), "f"(v[1]), "f"(v[2]), "f"(v[3]),
                                 "f"(v[4]), "f"(v[5]), "f"(v[6]), "f"(v[7]) : "memory");
                } else {
                    *reinterpret_cast<float4*>(o) = make_float4(v[0], v[1], v[2], v[3]);
                    if (n8 == 8) *reinterpret_cast<float4*>(o + 4) = make_float4(v[4], v[5], v[6], v[7]);
                }
            }
        }
        // The last products have been read out, so nothing of the ring is in use any more.
        if (!ptx::bar_or<kEpiBarrier, 32 * kEpiWarps>(!ok)) make_plain_sums(prm, M_keep);
    }
    ptx::tc_fence_before_sync();
    __syncthreads();
    ptx::cluster_sync_all();                                               // neither block leaves while the other may still reach into it
    if (warp == kMmaWarp) {
        ptx::tc_fence_after_sync();
        ptx::tmem_dealloc_pair(tmem, 512);
    }
}

// ---- host side ----
constexpr int64_t kPairs = kNumSMs / 2;
constexpr int64_t ceil_div(int64_t a, int64_t b) { return (a + b - 1) / b; }

// A launch holds at most kMaxRounds items of a worker: 2.5e9 sums.
int64_t launches_of(int64_t items) { return ceil_div(items, kMaxRounds * kPairs); }

cudaError_t launch(SplitParams prm, cudaStream_t stream) {
    const cudaError_t opt = opt_in_dynamic_smem<split_products_kernel>((int)kSmemBytes);
    if (opt != cudaSuccess) return opt;
    const int64_t items = (int64_t)prm.items[0] + prm.items[1];
    for (int64_t first = 0; first < items; first += kMaxRounds * kPairs) {
        const int64_t count = items - first < kMaxRounds * kPairs ? items - first : kMaxRounds * kPairs;
        prm.first = (uint32_t)first;
        prm.count = (uint32_t)count;
        const int64_t used = prm.dX != nullptr || count > kPairs ? kPairs : count;                 // the zeros take every SM
        const cudaError_t e = launch_pdl_cluster(split_products_kernel, dim3((unsigned)(2 * used)), dim3(kThreads), kSmemBytes, 2u, stream, prm);
        if (e != cudaSuccess) return e;
        prm.dX = nullptr;                                                                          // the first launch has written them
    }
    return cudaSuccess;
}

// Time of a list of `nx` items of `cx` us followed by `nw` of `cw`, dealt to `g` workers as list_position does.  The workers that take part
// in the round in which the first kind ends, and in the last round, are the first or the last of all: at most four kinds of workers.
double list_time(int64_t nx, double cx, int64_t nw, double cw, int64_t g) {
    const int64_t n = nx + nw, ax = nx / g, rx = nx % g, an = n / g, rn = n % g;
    const int64_t x0 = (ax & 1) ? g - rx : 0, x1 = x0 + rx, n0 = (an & 1) ? g - rn : 0, n1 = n0 + rn;
    double worst = 0.0;
    const auto kind = [&](bool exists, int64_t kx, int64_t kn) {
        const double t = (double)kx * cx + (double)(kn - kx) * cw;
        if (exists && t > worst) worst = t;
    };
    kind((x0 > n0 ? x0 : n0) < (x1 < n1 ? x1 : n1), ax + 1, an + 1);
    kind(rx > 0 && !(n0 <= x0 && x1 <= n1), ax + 1, an);
    kind(rn > 0 && !(x0 <= n0 && n1 <= x1), ax, an + 1);
    const bool all = rx + rn >= g && (x0 == 0 ? n1 == g : n0 == 0);
    kind(!all, ax, an);
    return worst;
}

// Pieces of the dW reduction.
constexpr double kKbUs = 1.4, kItemUs = 2.5;                               // us of a k-block, of an item's start and read-out

int64_t tiles_of(int64_t rows, int64_t cols) { return ceil_div(rows, 2 * kTile) * ceil_div(cols, kTile); }

struct SplitPlan { int splits; double us; };                               // us: of the tiles and the reduce launch

SplitPlan search_plan(int64_t M_keep_cap, int64_t C_in, int64_t C_out, bool out_in, bool want_dx) {
    int best = 1;
    double best_us = 0.0;
    const int64_t w_kb = ceil_div(M_keep_cap, kBK), x_kb = ceil_div(C_out, kBK);
    const int64_t nx = want_dx ? tiles_of(M_keep_cap, C_in) : 0, nw = out_in ? tiles_of(C_out, C_in) : tiles_of(C_in, C_out);
    for (int64_t s = 1; s <= (w_kb < 64 ? w_kb : 64); s += s < 8 ? 1 : s / 4) {
        const double cx = (double)x_kb * kKbUs + kItemUs, cw = (double)ceil_div(w_kb, s) * kKbUs + kItemUs;
        const bool x_first = cx >= cw;
        const double us = list_time(x_first ? nx : nw * s, x_first ? cx : cw, x_first ? nw * s : nx, x_first ? cw : cx, kPairs) +
                          (s > 1 ? 2.0 + (double)s * (double)C_in * (double)C_out * 8.0 / 4e6 : 0.0);
        if (best_us == 0.0 || us < best_us * 0.99) { best_us = us; best = (int)s; }
    }
    return SplitPlan{best, best_us};
}

// Remembered for the life of the process, as the bf16 plans are (tc_backward.cu): the four plans of a shape are one search.
struct ShapePlans { SplitPlan of[2][2]; };                                 // [out_in][want_dx]
std::mutex g_shape_mutex;
std::map<std::tuple<int64_t, int64_t, int64_t>, ShapePlans> g_shape_plans;

SplitPlan split_plan(int64_t M_keep_cap, int64_t C_in, int64_t C_out, bool out_in, bool want_dx) {
    const auto key = std::make_tuple(M_keep_cap, C_in, C_out);
    std::lock_guard<std::mutex> lock(g_shape_mutex);
    const auto it = g_shape_plans.find(key);
    if (it != g_shape_plans.end()) return it->second.of[out_in][want_dx];
    ShapePlans plans;
    for (int v = 0; v < 4; ++v) plans.of[v & 1][v >> 1] = search_plan(M_keep_cap, C_in, C_out, (v & 1) != 0, (v & 2) != 0);
    g_shape_plans[key] = plans;
    return plans.of[out_in][want_dx];
}

}  // namespace

// The roles' registers come out of those that the block is launched with: a build that gives it fewer must not run, and its callers take the
// CUDA cores.  So they do where the question itself fails (it is asked again then; the launch there says what is wrong).
bool split_can_run() {
    static std::atomic<int> known{0};                                      // 1: yes, 2: no
    if (known.load(std::memory_order_relaxed) == 0) {
        cudaFuncAttributes a;
        if (cudaFuncGetAttributes(&a, split_products_kernel) != cudaSuccess) return false;
        known.store(a.numRegs >= kLaunchRegs ? 1 : 2, std::memory_order_relaxed);
    }
    return known.load(std::memory_order_relaxed) == 1;
}

// The lines against the CUDA cores, which start in 3 us where this kernel takes 8 (a cluster of whole SMs, one deep stage), but whose
// blocks take 4 us for every 100 of depth.  Forward, CUDA cores and here: depth 128 with 491 rows and 376 columns 6.9, 9.2 us, 104 with
// 1839 and 184 10.4, 9.4, 152 with 2597 and 104 11.8, 10.6; 88 with 3193 and 264 9.4, 10.2, 64 with 3339 and 1232 20.6, 13.7, 32 with
// 21611 and 168 11.1, 15.2; 232 with 164 and 128 10.8, 11.4, 296 with 162 and 72 13.7, 12.4, 304 with 103 and 32 13.3, 11.3.
// dW + db + dX: 104 kept rows of 128 -> 144 11.5, 12.7 us, 649 of 152 -> 104 13.7, 12.1, 942 of 472 -> 48 15.9, 13.7; 6770 of 32 -> 72
// 13.1, 13.7; few rows behind deep sums of dX 95 of 80 -> 376 16.2, 12.0, 72 of 32 -> 720 30.5, 21.9.
bool split_forward_supported(int64_t M, int64_t C_in, int64_t C_out) {
    if (M < 32 || C_in < 32 || C_out < 32) return false;
    const int64_t work = M * C_in * C_out;
    return C_in >= 288 || (C_in >= 96 && work >= 50000000) || (C_in >= 56 && work >= 100000000) || (C_in >= 40 && work >= 400000000);
}
bool split_backward_supported(int64_t M_keep_cap, int64_t C_in, int64_t C_out, bool want_dx) {
    if (M_keep_cap < 16 || C_in < 32 || C_out < 32) return false;
    const int64_t work = M_keep_cap * C_in * C_out;
    return (want_dx && C_out >= 256) || (C_in >= 40 && C_out >= 40 && work >= 20000000) || work >= 80000000;
}
// Calls for dW, or dX, alone have half the work for the same start, and the CUDA cores cut dW into more pieces: there both times are
// estimated (fits to 6500 shapes of 32 to 3072 channels and 16 to 60000 kept rows, 6 and 8 % off on average).  dW + db, CUDA cores and here: 32
// kept rows of 2992 -> 352 5.7, 8.4 us, 131 of 2264 -> 100 8.7, 11.0, 1081 of 164 -> 156 11.0, 13.6, 1712 of 152 -> 248 13.8, 11.6; dX: 254 of
// 1844 -> 72 6.3, 10.1, 613 of 732 -> 52 5.4, 8.5.  (The lines above alone took 522 of 3886 calls for dW + db that are more than 5 % slower
// here, by up to 56 %, and 131 of 4786 for dX; 158 and 15 are left.)
bool split_backward_quicker(bool out_in, int64_t M_keep_cap, int64_t C_in, int64_t C_out, bool want_dw, bool want_dx) {
    if (!split_backward_supported(M_keep_cap, C_in, C_out, want_dx)) return false;
    if (want_dw == want_dx) return true;
    const double us = want_dw ? 3.8 + 1.03 * split_plan(M_keep_cap, C_in, C_out, out_in, false).us
                              : 4.5 + 0.85 * list_time(tiles_of(M_keep_cap, C_in), (double)ceil_div(C_out, kBK) * kKbUs + kItemUs, 0, 0.0, kPairs);
    return us < fma_backward_us(out_in, M_keep_cap, C_in, C_out, want_dw, want_dx);
}

cudaError_t launch_split_forward(const float* X, const float* W, bool w_out_in, const float* bias, int64_t M, int64_t C_in, int64_t C_out,
                                 float* Y, int32_t* status_word, cudaStream_t stream) {
    SplitParams prm{};
    Product& p = prm.p[0];
    p.A = X; p.lda = (uint32_t)C_in;
    p.B = W; p.ldb = (uint32_t)(w_out_in ? C_in : C_out); p.b_outer = w_out_in ? 0 : 1;
    p.rows = (int)M; p.cols = (int)C_out; p.depth = (int)C_in;
    p.splits = 1;
    p.out = Y; p.ld_out = C_out;
    p.bias = bias;
    p.row_tiles = (int)ceil_div(M, 2 * kTile);
    p.col_tiles = (int)ceil_div(C_out, kTile);
    prm.items[0] = (uint32_t)(p.row_tiles * p.col_tiles);
    prm.status_word = status_word;
    return launch(prm, stream);
}

int64_t split_plan_searches() {
    std::lock_guard<std::mutex> lock(g_shape_mutex);
    return (int64_t)g_shape_plans.size();
}

size_t split_workspace_bytes(int64_t M_keep_cap, int64_t C_in, int64_t C_out) {
    int most = 1;
    for (int v = 0; v < 4; ++v) {
        const int s = split_plan(M_keep_cap, C_in, C_out, (v & 1) != 0, (v & 2) != 0).splits;
        if (s > most) most = s;
    }
    return most > 1 ? (size_t)most * (size_t)(C_in + 1) * (size_t)C_out * sizeof(float) : 0;
}

int split_backward_kernel_count(bool w_out_in, int64_t M_keep_cap, int64_t C_in, int64_t C_out, bool want_dw, bool want_dx) {
    if (!want_dw && !want_dx) return 0;
    const int splits = want_dw ? split_plan(M_keep_cap, C_in, C_out, w_out_in, want_dx).splits : 1;
    const int64_t nx = want_dx ? tiles_of(M_keep_cap, C_in) : 0, nw = want_dw ? (w_out_in ? tiles_of(C_out, C_in) : tiles_of(C_in, C_out)) * splits : 0;
    return (int)launches_of(nx + nw) + (splits > 1 ? 1 : 0);
}

cudaError_t launch_split_backward(const float* X_keep, const float* dY, const float* W, bool w_out_in, const int32_t* dy_rows,
                                  const int32_t* dx_rows, const int32_t* M_keep_dev, int64_t M, int64_t M_keep_cap, int64_t C_in,
                                  int64_t C_out, float* dW, float* db, bool dw_accumulate, bool db_accumulate, float* dX, float* workspace,
                                  int32_t* status_word, cudaStream_t stream) {
    const int splits = dW != nullptr ? split_plan(M_keep_cap, C_in, C_out, w_out_in, dX != nullptr).splits : 1;
    const bool pieces = dW != nullptr && splits > 1;
    float* ws_db = workspace;                                              // [splits, C_out], then [splits, C_in * C_out]
    float* ws_dw = workspace + (int64_t)splits * C_out;
    SplitParams prm{};
    prm.M_keep_dev = M_keep_dev;
    prm.M_keep_cap = M_keep_cap;
    prm.status_word = status_word;
    Product px{}, pw{};
    uint32_t nx = 0, nw = 0;
    if (dX != nullptr) {
        prm.dX = dX; prm.dx_rows = dx_rows; prm.M = M; prm.C_in = (int)C_in;
        px.A = dY; px.lda = (uint32_t)C_out; px.a_map = dy_rows;
        px.B = W; px.ldb = (uint32_t)(w_out_in ? C_in : C_out); px.b_outer = w_out_in ? 1 : 0;
        px.rows = (int)M_keep_cap; px.rows_kept = 1; px.cols = (int)C_in; px.depth = (int)C_out;
        px.splits = 1;
        px.out = dX; px.ld_out = C_in; px.out_map = dx_rows;
        px.row_tiles = (int)ceil_div(M_keep_cap, 2 * kTile);
        px.col_tiles = (int)ceil_div(C_in, kTile);
        nx = (uint32_t)(px.row_tiles * px.col_tiles);
    }
    if (dW != nullptr) {
        // rows of dW are C_in x columns C_out, or the other way round for weights stored [C_out, C_in]
        pw.A = w_out_in ? dY : X_keep; pw.lda = (uint32_t)(w_out_in ? C_out : C_in); pw.a_map = w_out_in ? dy_rows : nullptr; pw.a_outer = 1;
        pw.B = w_out_in ? X_keep : dY; pw.ldb = (uint32_t)(w_out_in ? C_in : C_out); pw.b_map = w_out_in ? nullptr : dy_rows; pw.b_outer = 1;
        pw.rows = (int)(w_out_in ? C_out : C_in); pw.cols = (int)(w_out_in ? C_in : C_out); pw.depth = (int)M_keep_cap; pw.depth_kept = 1;
        pw.splits = splits;
        pw.out = pieces ? ws_dw : dW; pw.ld_out = pw.cols; pw.split_stride = C_in * C_out;
        pw.accumulate = dw_accumulate && !pieces;
        pw.sum_side = db == nullptr ? 0 : w_out_in ? 1 : 2;
        pw.sums = pieces ? ws_db : db;
        pw.sums_accumulate = db_accumulate && !pieces;
        pw.row_tiles = (int)ceil_div(pw.rows, 2 * kTile);
        pw.col_tiles = (int)ceil_div(pw.cols, kTile);
        nw = (uint32_t)(pw.row_tiles * pw.col_tiles * pw.splits);
    }
    const bool x_first = ceil_div(C_out, kBK) >= ceil_div(ceil_div(M_keep_cap, kBK), splits);
    prm.p[0] = x_first ? px : pw; prm.items[0] = x_first ? nx : nw;
    prm.p[1] = x_first ? pw : px; prm.items[1] = x_first ? nw : nx;
    const cudaError_t e = launch(prm, stream);
    if (e != cudaSuccess || !pieces) return e;
    if (db != nullptr)
        return launch_reduce_partials_pair(ws_dw, splits, C_in * C_out, dW, dw_accumulate, ws_db, splits, C_out, db, db_accumulate,
                                           status_word, stream);
    return launch_reduce_partials(ws_dw, splits, C_in * C_out, dW, dw_accumulate, status_word, stream);
}

}  // namespace sbp

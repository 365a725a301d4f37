// Products on the CUDA cores, fp32 fused multiply-adds: fp32 and bf16 shapes whose products are too short for the tensor-core kernels
// (split_products.cu, tc_backward.cu, tc_forward.cu), and any shape on request.
//   forward  Y[m, j] = sum_i X[m, i] W[i, j] + bias[j]                        (Eq. 2)
//   dW[i, j] = sum_m X_keep[m, i] dY[keep_rows[m], j],  db[j] = sum_m dY[keep_rows[m], j]       (Eq. 5)
//   dX[keep_rows[m], i] = sum_j dY[keep_rows[m], j] W[i, j]; every other row of dX = +0.0
//
// Bound by the FMA pipes, with shared memory close behind.  Blackwell issues two fp32 FMAs per lane with one packed
// instruction (fma.rn.f32x2, each half rounded as its own fmaf): alone they reach 71.5 TFLOP/s, but four 16-byte
// shared-memory loads for 32 of them, an 8 x 8 tile a thread, already fill the load pipe as long as the FMA pipe (59
// TFLOP/s in a loop of nothing else).  So a thread owns 8 x 16 outputs where tiles of 64 x 128 fill the GPU (six loads for
// 64 packed FMAs) and 8 x 8 in tiles of 64 x 64 below that.  The threads of a block form 2 (wide) or 4 groups which make the
// same outputs from different depths of each stage and add their accumulators up through shared memory at the end: a tile
// takes a half or a quarter of the time.  Operands go global -> registers -> shared memory in two stages, the next one's loads
// in flight during the current arithmetic.
//
// Measured on B200, fp32 768 -> 3072, 3136 rows with 1568 kept, against 64 x 64 tiles of scalar FMAs in a kernel per product
// and two for db: forward 441 -> 304 us (48.7 TFLOP/s), dW + db + dX 612 -> 350 us.  8 x 8 outputs in the wide tiles: 321 and
// 405 us, whether or not the next step's operands were fetched ahead.  Operand A stored as ready-made pairs {a, a}, which
// saves the moves that double it: 450 us.
#include "zero_rows.cuh"

namespace sbp {
namespace {

constexpr int kBM = 64;                   // rows of a tile
constexpr int kTM = 8;                    // rows of a thread's outputs

// The two block shapes: columns of the tile, columns of a thread's outputs, threads, reduction depth of a stage.  (The small
// tiles run where there are few of them, so that each stage's loads are waited for: deep stages.)
template <int kBN> struct Shape;
template <> struct Shape<128> { static constexpr int kTN = 16, kThreads = 128, kBK = 16; };
template <> struct Shape<64> { static constexpr int kTN = 8, kThreads = 256, kBK = 32; };

template <typename T> __device__ __forceinline__ float4 load4(const T* p);
template <> __device__ __forceinline__ float4 load4<float>(const float* p) {
    return __ldg(reinterpret_cast<const float4*>(p));
}
template <> __device__ __forceinline__ float4 load4<__nv_bfloat16>(const __nv_bfloat16* p) {
    const uint2 v = __ldg(reinterpret_cast<const uint2*>(p));
    return make_float4(__uint_as_float(v.x << 16), __uint_as_float(v.x & 0xffff0000u),
                       __uint_as_float(v.y << 16), __uint_as_float(v.y & 0xffff0000u));
}
template <typename T> __device__ __forceinline__ void store4(T* p, float4 v);
template <> __device__ __forceinline__ void store4<float>(float* p, float4 v) { *reinterpret_cast<float4*>(p) = v; }
template <> __device__ __forceinline__ void store4<__nv_bfloat16>(__nv_bfloat16* p, float4 v) {
    const __nv_bfloat162 lo = __floats2bfloat162_rn(v.x, v.y);
    const __nv_bfloat162 hi = __floats2bfloat162_rn(v.z, v.w);
    uint2 u;
    u.x = *reinterpret_cast<const uint32_t*>(&lo);
    u.y = *reinterpret_cast<const uint32_t*>(&hi);
    *reinterpret_cast<uint2*>(p) = u;
}

__device__ __forceinline__ uint64_t twice(float a) {
    uint64_t r;
    asm("mov.b64 %0, {%1, %1};" : "=l"(r) : "f"(a));
    return r;
}
__device__ __forceinline__ void fma2(uint64_t& d, uint64_t a, uint64_t b) {
    asm("fma.rn.f32x2 %0, %1, %2, %0;" : "+l"(d) : "l"(a), "l"(b));
}
__device__ __forceinline__ void add2(uint64_t& d, uint64_t a) {
    asm("add.rn.f32x2 %0, %0, %1;" : "+l"(d) : "l"(a));
}
__device__ __forceinline__ float2 halves(uint64_t v) {
    float2 f;
    asm("mov.b64 {%0, %1}, %2;" : "=f"(f.x), "=f"(f.y) : "l"(v));
    return f;
}

// One operand of a product, [extent x depth] as the product sees it: a row-major matrix whose rows are extent indices
// (depth inner) or depth indices.  `map` sends a row of the matrix to the row of memory it lives in (nullptr: itself).
template <typename T>
struct Operand {
    const T* base;
    int64_t ld;                            // elements between rows of memory
    const int32_t* map;
    int64_t extent;                        // valid extent indices
};

// Global -> register -> shared-memory path of one operand: a tile of B extent indices x kBK depth.
template <typename T, int B, bool kDepthInner, int NT, int kBK>
struct TileLoader {
    static constexpr int kVecs = B * kBK / 4 / NT;       // 4-element vectors per thread and stage
    static constexpr int kPitch = B + 4;                 // floats per depth row in shared memory
    static_assert(kVecs >= 1 && B * kBK % (4 * NT) == 0, "tile divides among the threads");
    float4 v[kVecs];
    const T* ptr[kDepthInner ? kVecs : 1];               // depth inner: the rows are the same in every stage
    int32_t row[kDepthInner ? 1 : kVecs];                // otherwise: rows of memory of the stage fetched next

    __device__ __forceinline__ void init(const Operand<T>& op, int64_t e0, int64_t d0, int64_t d_end) {
        if constexpr (kDepthInner) {
#pragma unroll
            for (int i = 0; i < kVecs; ++i) {
                const int idx = threadIdx.x + i * NT;
                const int64_t e = e0 + idx / (kBK / 4);
                ptr[i] = e < op.extent ? op.base + (int64_t)mapped_row(op.map, e) * op.ld + (idx % (kBK / 4)) * 4 : nullptr;
            }
        } else {
            fetch_rows(op, d0, d_end);
        }
    }
    __device__ __forceinline__ void fetch_rows(const Operand<T>& op, int64_t d0, int64_t d_end) {
#pragma unroll
        for (int i = 0; i < kVecs; ++i) {
            const int64_t d = d0 + (threadIdx.x + i * NT) / (B / 4);
            row[i] = d < d_end ? mapped_row(op.map, d) : -1;
        }
    }
    // stage of depth [d0, d0 + kBK), depth indices from d_end on read as zero
    __device__ __forceinline__ void fetch(const Operand<T>& op, int64_t e0, int64_t d0, int64_t d_end) {
#pragma unroll
        for (int i = 0; i < kVecs; ++i) {
            const int idx = threadIdx.x + i * NT;
            v[i] = make_float4(0.f, 0.f, 0.f, 0.f);
            if constexpr (kDepthInner) {
                if (ptr[i] != nullptr && d0 + (idx % (kBK / 4)) * 4 < d_end) v[i] = load4<T>(ptr[i] + d0);
            } else {
                const int64_t e = e0 + (idx % (B / 4)) * 4;
                if (row[i] >= 0 && e < op.extent) v[i] = load4<T>(op.base + (int64_t)row[i] * op.ld + e);
            }
        }
        if constexpr (!kDepthInner) fetch_rows(op, d0 + kBK, d_end);
    }
    __device__ __forceinline__ void put(float* tile) const {           // tile[depth][extent]
#pragma unroll
        for (int i = 0; i < kVecs; ++i) {
            const int idx = threadIdx.x + i * NT;
            if constexpr (kDepthInner) {
                const int e = idx / (kBK / 4), d = (idx % (kBK / 4)) * 4;
                tile[(d + 0) * kPitch + e] = v[i].x;
                tile[(d + 1) * kPitch + e] = v[i].y;
                tile[(d + 2) * kPitch + e] = v[i].z;
                tile[(d + 3) * kPitch + e] = v[i].w;
            } else {
                *reinterpret_cast<float4*>(tile + (idx / (B / 4)) * kPitch + (idx % (B / 4)) * 4) = v[i];
            }
        }
    }
};

template <int BN>
using Accumulators = uint64_t[kTM][Shape<BN>::kTN / 2];

template <int BN>
union ProductShared {
    struct {
        float a[2][Shape<BN>::kBK][kBM + 4];
        float b[2][Shape<BN>::kBK][BN + 4];
    } t;
    ulonglong2 swap[kTM / 2 * Shape<BN>::kTN / 4][Shape<BN>::kThreads];     // half a thread's accumulators, on their way to the partner group
};

// Where a thread's outputs sit in the tile: before the groups add up, rows row0 + {0..3, 16..19}, columns col0 + {0..3} +
// 32 h (h < kQuads) in every group; afterwards group g holds kRows of the eight rows, from number first on.
template <int BN>
struct ThreadTile {
    static constexpr int kTN = Shape<BN>::kTN, kQuads = kTN / 4, kWarpCols = 8 * kTN;
    static constexpr int kThreads = (kBM / kTM) * (BN / kTN);          // threads of a group
    static constexpr int kG = Shape<BN>::kThreads / kThreads, kRows = kTM / kG;
    int group, row0, col0, first;
    __device__ __forceinline__ ThreadTile() {
        group = threadIdx.x / kThreads;
        const int warp = (threadIdx.x % kThreads) >> 5, lane = threadIdx.x & 31;
        row0 = (warp / (BN / kWarpCols)) * 32 + (lane >> 3) * 4;
        col0 = (warp % (BN / kWarpCols)) * kWarpCols + (lane & 7) * 4;
        first = group * kRows;
    }
    __device__ __forceinline__ int row(int q) const { return row0 + ((first + q) & 3) + ((first + q) >> 2) * 16; }
    __device__ __forceinline__ int col(int h) const { return col0 + h * 32; }
};

// One step of the sum over groups: partners exchange halves of kHave accumulator rows, `upper` keeps the upper half.
template <int BN, int kHave>
__device__ __forceinline__ void halve(ProductShared<BN>& sh, Accumulators<BN>& acc, bool upper, int partner) {
    constexpr int kKeep = kHave / 2, kPairs = Shape<BN>::kTN / 2;
    if (upper) {
#pragma unroll
        for (int r = 0; r < kKeep; ++r)
#pragma unroll
            for (int c = 0; c < kPairs; ++c) {
                const uint64_t t = acc[r][c];
                acc[r][c] = acc[r + kKeep][c];
                acc[r + kKeep][c] = t;
            }
    }
    __syncthreads();                       // the tiles (or the exchange before) have been read
#pragma unroll
    for (int r = 0; r < kKeep; ++r)
#pragma unroll
        for (int c = 0; c < kPairs; c += 2)
            sh.swap[(r * kPairs + c) / 2][threadIdx.x] = make_ulonglong2(acc[kKeep + r][c], acc[kKeep + r][c + 1]);
    __syncthreads();
#pragma unroll
    for (int r = 0; r < kKeep; ++r)
#pragma unroll
        for (int c = 0; c < kPairs; c += 2) {
            const ulonglong2 u = sh.swap[(r * kPairs + c) / 2][partner];
            add2(acc[r][c], u.x);
            add2(acc[r][c + 1], u.y);
        }
}

// acc = A[e_a0 .., d] * B[e_b0 .., d] over the depth range [d_begin, d_end), in the first kRows rows of `acc` (ThreadTile).
// kSum: 0 none, 1 / 2: `colsum` of thread t receives the sum over the depth of extent index t of operand A / B (the
// bias gradient).
template <typename T, int BN, bool kAInner, bool kBInner, int kSum>
__device__ __forceinline__ void product(ProductShared<BN>& sh, const ThreadTile<BN>& tt, const Operand<T>& A, const Operand<T>& B,
                                        int64_t e_a0, int64_t e_b0, int64_t d_begin, int64_t d_end, bool want_sum,
                                        Accumulators<BN>& acc, float& colsum) {
    constexpr int NT = Shape<BN>::kThreads, kTN = Shape<BN>::kTN, kBK = Shape<BN>::kBK;
    constexpr int kG = ThreadTile<BN>::kG, kMine = kBK / kG;           // depth steps of a stage for each group
    static_assert(NT >= BN && NT >= kBM, "a thread for each column of the sums");
    TileLoader<T, kBM, kAInner, NT, kBK> la;
    TileLoader<T, BN, kBInner, NT, kBK> lb;
#pragma unroll
    for (int r = 0; r < kTM; ++r)
#pragma unroll
        for (int c = 0; c < kTN / 2; ++c) acc[r][c] = 0ull;
    colsum = 0.f;
    float lost = 0.f;                      // of the compensated sum below
    if (d_begin >= d_end) return;
    la.init(A, e_a0, d_begin, d_end);
    lb.init(B, e_b0, d_begin, d_end);
    la.fetch(A, e_a0, d_begin, d_end);
    lb.fetch(B, e_b0, d_begin, d_end);
    int buf = 0;
    for (int64_t d0 = d_begin; d0 < d_end; d0 += kBK, buf ^= 1) {
        la.put(&sh.t.a[buf][0][0]);
        lb.put(&sh.t.b[buf][0][0]);
        __syncthreads();                   // (two buffers: the one written next was last read before this barrier)
        if (d0 + kBK < d_end) {
            la.fetch(A, e_a0, d0 + kBK, d_end);
            lb.fetch(B, e_b0, d0 + kBK, d_end);
        }
        if (kSum != 0 && want_sum && threadIdx.x < (kSum == 1 ? kBM : BN)) {
            float part[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
            for (int k = 0; k < kBK; ++k) part[k & 3] += kSum == 1 ? sh.t.a[buf][k][threadIdx.x % kBM] : sh.t.b[buf][k][threadIdx.x % BN];
            const float y = ((part[0] + part[1]) + (part[2] + part[3])) - lost, t = colsum + y;     // Kahan's sum: one chain
            lost = (t - colsum) - y;                                                                // of up to thousands of stages
            if (!(fabsf(lost) < INFINITY)) lost = 0.f;       // an infinite sum has lost nothing (infinity - infinity would make it a NaN)
            colsum = t;
        }
#pragma unroll
        for (int k = 0; k < kMine; ++k) {
            const float* ak = &sh.t.a[buf][tt.group * kMine + k][tt.row0];
            const float* bk = &sh.t.b[buf][tt.group * kMine + k][tt.col0];
            const float4 a0 = *reinterpret_cast<const float4*>(ak), a1 = *reinterpret_cast<const float4*>(ak + 16);
            const float a[kTM] = {a0.x, a0.y, a0.z, a0.w, a1.x, a1.y, a1.z, a1.w};
            uint64_t b[kTN / 2];
#pragma unroll
            for (int h = 0; h < kTN / 4; ++h) {
                const ulonglong2 v = *reinterpret_cast<const ulonglong2*>(bk + h * 32);
                b[2 * h] = v.x;
                b[2 * h + 1] = v.y;
            }
#pragma unroll
            for (int r = 0; r < kTM; ++r) {
                const uint64_t a2 = twice(a[r]);
#pragma unroll
                for (int c = 0; c < kTN / 2; ++c) fma2(acc[r][c], a2, b[c]);
            }
        }
    }
    constexpr int kT = ThreadTile<BN>::kThreads;
    if constexpr (kG == 2) {
        halve<BN, 8>(sh, acc, tt.group != 0, threadIdx.x ^ kT);
    } else {
        halve<BN, 8>(sh, acc, tt.group >= 2, threadIdx.x ^ (2 * kT));
        halve<BN, 4>(sh, acc, (tt.group & 1) != 0, threadIdx.x ^ kT);
    }
}

template <int kPairs>
__device__ __forceinline__ float4 quad(const uint64_t (&acc)[kTM][kPairs], int q, int h) {
    const float2 lo = halves(acc[q][2 * h]), hi = halves(acc[q][2 * h + 1]);
    return make_float4(lo.x, lo.y, hi.x, hi.y);
}

template <typename T>
struct ForwardParams {
    Operand<T> X, W;
    const float* bias;
    T* Y;
    int64_t M;
    int C_in, C_out;
    const int32_t* status_word;
};

template <typename T, int BN, bool kOutIn>
__global__ void __launch_bounds__(Shape<BN>::kThreads, 2)
fma_forward_kernel(const ForwardParams<T> p) {
    __shared__ __align__(16) ProductShared<BN> sh;
    pdl_launch_dependents();
    pdl_wait();
    if (p.status_word != nullptr && *p.status_word != 0) return;
    const int64_t m0 = (int64_t)blockIdx.x * kBM;
    const int j0 = blockIdx.y * BN;
    const ThreadTile<BN> tt;
    Accumulators<BN> acc;
    float unused;
    product<T, BN, true, kOutIn, 0>(sh, tt, p.X, p.W, m0, j0, 0, p.C_in, false, acc, unused);
#pragma unroll
    for (int h = 0; h < tt.kQuads; ++h) {
        const int j = j0 + tt.col(h);
        if (j >= p.C_out) continue;
        float4 bv = make_float4(0.f, 0.f, 0.f, 0.f);
        if (p.bias != nullptr) bv = __ldg(reinterpret_cast<const float4*>(p.bias + j));
#pragma unroll
        for (int q = 0; q < tt.kRows; ++q) {
            const int64_t m = m0 + tt.row(q);
            if (m >= p.M) continue;
            const float4 v = quad(acc, q, h);
            store4<T>(p.Y + m * p.C_out + j, make_float4(v.x + bv.x, v.y + bv.y, v.z + bv.z, v.w + bv.w));
        }
    }
}

// Short reductions: the kernel above fills its stages and adds its groups up whatever the depth.  Here 256 threads make 64 x 64 outputs,
// 4 x 4 each, in steps of 16, with nothing to add up at the end (fp32 16 -> 4096, 12544 rows: 99.9 us there, 72.3 here).
constexpr int kShortThreads = 256, kShortK = 16;
template <typename T, bool kOutIn>
__global__ void __launch_bounds__(kShortThreads)
fma_short_forward_kernel(const ForwardParams<T> p) {
    __shared__ __align__(16) float As[kShortK][kBM + 4], Bs[kShortK][kBM + 4];
    pdl_launch_dependents();
    pdl_wait();
    if (p.status_word != nullptr && *p.status_word != 0) return;
    const int64_t m0 = (int64_t)blockIdx.x * kBM;
    const int j0 = blockIdx.y * kBM;
    const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
    const int er = threadIdx.x >> 2, ec = (threadIdx.x & 3) * 4;      // operands with the depth inside: row of the tile, 4 of the 16 deep
    const int dr = threadIdx.x >> 4, dc = (threadIdx.x & 15) * 4;     // W [C_in, C_out]: depth, 4 of the 64 columns
    const float4 zero4 = make_float4(0.f, 0.f, 0.f, 0.f);
    float acc[4][4] = {};
    for (int i0 = 0; i0 < p.C_in; i0 += kShortK) {
        float4 a = zero4, b = zero4;
        if (m0 + er < p.M && i0 + ec < p.C_in) a = load4<T>(p.X.base + (m0 + er) * p.X.ld + i0 + ec);
        As[ec + 0][er] = a.x; As[ec + 1][er] = a.y; As[ec + 2][er] = a.z; As[ec + 3][er] = a.w;
        if constexpr (kOutIn) {
            if (j0 + er < p.C_out && i0 + ec < p.C_in) b = load4<T>(p.W.base + (int64_t)(j0 + er) * p.W.ld + i0 + ec);
            Bs[ec + 0][er] = b.x; Bs[ec + 1][er] = b.y; Bs[ec + 2][er] = b.z; Bs[ec + 3][er] = b.w;
        } else {
            if (i0 + dr < p.C_in && j0 + dc < p.C_out) b = load4<T>(p.W.base + (int64_t)(i0 + dr) * p.W.ld + j0 + dc);
            *reinterpret_cast<float4*>(&Bs[dr][dc]) = b;
        }
        __syncthreads();
#pragma unroll
        for (int k = 0; k < kShortK; ++k) {
            const float4 av = *reinterpret_cast<const float4*>(&As[k][ty * 4]);
            const float4 bv = *reinterpret_cast<const float4*>(&Bs[k][tx * 4]);
            const float ar[4] = {av.x, av.y, av.z, av.w}, br[4] = {bv.x, bv.y, bv.z, bv.w};
#pragma unroll
            for (int r = 0; r < 4; ++r)
#pragma unroll
                for (int c = 0; c < 4; ++c) acc[r][c] = fmaf(ar[r], br[c], acc[r][c]);
        }
        __syncthreads();
    }
    const int j = j0 + tx * 4;
    if (j >= p.C_out) return;
    float4 bias = zero4;
    if (p.bias != nullptr) bias = __ldg(reinterpret_cast<const float4*>(p.bias + j));
#pragma unroll
    for (int r = 0; r < 4; ++r) {
        const int64_t m = m0 + ty * 4 + r;
        if (m < p.M)
            store4<T>(p.Y + m * p.C_out + j, make_float4(acc[r][0] + bias.x, acc[r][1] + bias.y, acc[r][2] + bias.z, acc[r][3] + bias.w));
    }
}

// dW, db and dX of one layer in one launch: a block makes one tile of either product.
template <typename T>
struct BackwardParams {
    const T *X_keep, *dY, *W;
    const int32_t *dy_rows, *dx_rows;      // row m of the products reads row dy_rows[m] of dY, writes row dx_rows[m] of dX
    const int32_t* M_keep_dev;
    int64_t M, M_keep_cap;                 // M = rows of dX
    int C_in, C_out;
    float* dW;                             // dW itself, or the partials [splits, C_in * C_out]
    float* db;                             // nullptr: not asked for; db itself, or the partials [splits, C_out]
    T* dX;
    int w_tiles, w_col_tiles, splits;
    int dw_accumulate, db_accumulate;      // add into dW, into db (only with one split)
    int x_row_tiles, x_col_tiles;          // w_tiles / x_row_tiles 0: that product is not asked for
    int zero_blocks;                       // blocks that clear the dropped rows of dX
    const int32_t* status_word;
};

template <typename T, int BN, bool kOutIn>
__device__ __forceinline__ void dw_tile(ProductShared<BN>& sh, const BackwardParams<T>& p, int q, int64_t M_keep) {
    const int split = q % p.splits, tile = q / p.splits;
    const int row_tile = tile / p.w_col_tiles, col_tile = tile % p.w_col_tiles;
    int64_t per = (M_keep + p.splits - 1) / p.splits;
    per = (per + Shape<BN>::kBK - 1) / Shape<BN>::kBK * Shape<BN>::kBK;
    const int64_t begin = per * split, end = begin + per < M_keep ? begin + per : M_keep;
    const Operand<T> X{p.X_keep, p.C_in, nullptr, p.C_in}, Y{p.dY, p.C_out, p.dy_rows, p.C_out};
    const ThreadTile<BN> tt;
    Accumulators<BN> acc;
    float colsum;
    // rows of the output are C_in x columns C_out, or the other way round for weights stored [C_out, C_in]
    const bool want_sum = p.db != nullptr && (kOutIn ? col_tile : row_tile) == 0;
    if constexpr (kOutIn) product<T, BN, false, false, 1>(sh, tt, Y, X, row_tile * kBM, col_tile * BN, begin, end, want_sum, acc, colsum);
    else product<T, BN, false, false, 2>(sh, tt, X, Y, row_tile * kBM, col_tile * BN, begin, end, want_sum, acc, colsum);
    if (want_sum) {
        const int t = threadIdx.x, j = (kOutIn ? row_tile * kBM : col_tile * BN) + t;
        if (t < (kOutIn ? kBM : BN) && j < p.C_out) {
            float* o = p.db + (int64_t)split * p.C_out + j;
            *o = p.db_accumulate ? *o + colsum : colsum;
        }
    }
    const int rows = kOutIn ? p.C_out : p.C_in, cols = kOutIn ? p.C_in : p.C_out;
    float* out = p.dW + (int64_t)split * p.C_in * p.C_out;
#pragma unroll
    for (int r = 0; r < tt.kRows; ++r) {
        const int i = row_tile * kBM + tt.row(r);
        if (i >= rows) continue;
#pragma unroll
        for (int h = 0; h < tt.kQuads; ++h) {
            const int j = col_tile * BN + tt.col(h);
            if (j >= cols) continue;
            float4 v = quad(acc, r, h);
            float4* o = reinterpret_cast<float4*>(out + (int64_t)i * cols + j);
            if (p.dw_accumulate) { const float4 w = *o; v.x += w.x; v.y += w.y; v.z += w.z; v.w += w.w; }
            *o = v;
        }
    }
}

template <typename T, int BN, bool kOutIn>
__device__ __forceinline__ void dx_tile(ProductShared<BN>& sh, const BackwardParams<T>& p, int q, int64_t M_keep) {
    const int row_tile = q / p.x_col_tiles, i0 = (q % p.x_col_tiles) * BN;
    const int64_t m0 = (int64_t)row_tile * kBM;
    if (m0 >= M_keep) return;
    const Operand<T> Y{p.dY, p.C_out, p.dy_rows, M_keep};
    const Operand<T> W{p.W, kOutIn ? p.C_in : p.C_out, nullptr, p.C_in};
    const ThreadTile<BN> tt;
    Accumulators<BN> acc;
    float unused;
    product<T, BN, true, !kOutIn, 0>(sh, tt, Y, W, m0, i0, 0, p.C_out, false, acc, unused);
#pragma unroll
    for (int r = 0; r < tt.kRows; ++r) {
        const int64_t m = m0 + tt.row(r);
        if (m >= M_keep) continue;
        T* out = p.dX + (int64_t)mapped_row(p.dx_rows, m) * p.C_in;
#pragma unroll
        for (int h = 0; h < tt.kQuads; ++h) {
            const int i = i0 + tt.col(h);
            if (i < p.C_in) store4<T>(out + i, quad(acc, r, h));
        }
    }
}

// Zeros of the dropped rows: every warp of the blocks that do this takes an equal share of the rows of dX.  Blocks of their own:
// in front of a dX tile the search and the stores delayed a small layer's only wave by 2 - 3 us.  Rows of at most four vectors go 8,
// 16 or 32 to a store instruction (fp32 4 -> 4 channels, 157 of 3136 rows kept: a row an instruction 57 us, now 9.1).
template <typename T, int kThreads>
__device__ __forceinline__ void zero_rows(const BackwardParams<T>& p, int block, int64_t M_keep) {
    constexpr int kWarps = kThreads / 32;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, quads = p.C_in / 4;
    const int64_t workers = (int64_t)p.zero_blocks * kWarps, per = (p.M + workers - 1) / workers;
    const int64_t lo = per * ((int64_t)block * kWarps + warp), hi = lo + per < p.M ? lo + per : p.M;
    const float4 zero4 = make_float4(0.f, 0.f, 0.f, 0.f);
    const int lanes = quads > 4 ? 32 : quads > 2 ? 4 : quads;          // lanes a row takes
    warp_visit_dropped_rows(p.dx_rows, M_keep, lo, hi, lane, [&](int64_t base, uint32_t todo) {
        if (lanes <= 4) {                                              // the 32 rows in at most four steps, kept ones skipped
            for (int bit = lane / lanes; bit < 32; bit += 32 / lanes)
                if (((todo >> bit) & 1u) && lane % lanes < quads) store4<T>(p.dX + (base + bit) * p.C_in + (lane % lanes) * 4, zero4);
            return;
        }
        for (; todo; todo &= todo - 1u) {
            T* row = p.dX + (base + __ffs(todo) - 1) * p.C_in;
            for (int v = lane; v < quads; v += 32) store4<T>(row + v * 4, zero4);
        }
    });
}

template <typename T, int BN, bool kOutIn>
__global__ void __launch_bounds__(Shape<BN>::kThreads, 2)
fma_backward_kernel(const BackwardParams<T> p) {
    __shared__ __align__(16) ProductShared<BN> sh;
    pdl_launch_dependents();
    pdl_wait();
    if (p.status_word != nullptr && *p.status_word != 0) return;
    const int64_t M_keep = load_m_keep(p.M_keep_dev, p.M_keep_cap);
    const int x_blocks = p.x_row_tiles * p.x_col_tiles;
    // the deepest reductions first, the zeros last
    const int block = (int)blockIdx.x, w_blocks = p.w_tiles * p.splits;
    if (block < x_blocks) dx_tile<T, BN, kOutIn>(sh, p, block, M_keep);
    else if (block < x_blocks + w_blocks) dw_tile<T, BN, kOutIn>(sh, p, block - x_blocks, M_keep);
    else zero_rows<T, Shape<BN>::kThreads>(p, block - x_blocks - w_blocks, M_keep);
}

// ---- host side: tile shape, splits of the dW reduction, launches ----
constexpr int64_t ceil_div(int64_t a, int64_t b) { return (a + b - 1) / b; }

struct FmaPlan {
    bool wide;             // 64 x 128 tiles instead of 64 x 64
    int64_t w_rows, w_cols, x_rows, x_cols;
    int splits;
};

// 64 x 128 tiles (half as many shared-memory reads of W or dY per output) where they fill the two blocks per SM at least
// once, 64 x 64 below that (fp32 only: the bf16 shapes that come here are small).
// A dW tile is cut along the kept rows so that no block reduces over more than half of what an SM has to do in all.
FmaPlan fma_plan(bool fp32, bool out_in, int64_t M_keep_cap, int64_t C_in, int64_t C_out, bool want_w, bool want_x) {
    FmaPlan pl;
    const int64_t wr = out_in ? C_out : C_in, wc = out_in ? C_in : C_out;
    const auto set = [&](int bn) {
        pl.w_rows = want_w ? ceil_div(wr, kBM) : 0;
        pl.w_cols = want_w ? ceil_div(wc, bn) : 0;
        pl.x_rows = want_x ? (M_keep_cap > 0 ? ceil_div(M_keep_cap, kBM) : 1) : 0;
        pl.x_cols = want_x ? ceil_div(C_in, bn) : 0;
    };
    set(128);
    pl.wide = fp32 && pl.w_rows * pl.w_cols + pl.x_rows * pl.x_cols >= 2 * kNumSMs;
    if (!pl.wide) set(64);
    const double w_depth = (double)ceil_div(M_keep_cap, 16), x_depth = (double)ceil_div(C_out, 16);      // 16-deep steps
    const double per_sm = (pl.w_rows * pl.w_cols * w_depth + pl.x_rows * pl.x_cols * x_depth) / kNumSMs;
    const double limit = per_sm / 2 > 8.0 ? per_sm / 2 : 8.0;
    double s = want_w ? w_depth / limit : 1.0;
    if (s > 64.0) s = 64.0;
    pl.splits = (int)s < s ? (int)s + 1 : (int)s;
    if (pl.splits < 1) pl.splits = 1;
    return pl;
}

// Where the plain form is the quicker one, fp32 timings in us (plain, grouped): over 16 channels everywhere (16 -> 64, 784 rows 2.5,
// 3.9; 16 -> 1024, 100352 rows 127, 167); up to 48 on few tiles (48 -> 256, 196 rows 4.2, 5.0; not 48 -> 192, 3136
// rows, 147 tiles, 7.8, 6.8) or where a 128-wide tile
// would be half empty (48 -> 8, 100352 rows 19.9, 29.8; 48 -> 192, 12544 rows 9.1, 11.6), up to 32 on several waves (32 -> 256, 100352
// rows 55.0, 59.4), up to 64 with many half empty tiles (64 -> 64, 100352 rows 27.0, 31.4).  Beyond: 48 -> 1024, 784 rows 8.6, 7.3; 64 ->
// 256, 3136 rows 9.8, 7.3.
bool short_reduction(int64_t M, int64_t C_in, int64_t C_out) {
    const int64_t tiles = ceil_div(M, kBM) * ceil_div(C_out, kBM);
    const bool half_empty = C_out <= 64 || (C_out > 128 && C_out <= 192);           // the last 128-wide tile
    if (C_in <= 16 || (C_in <= 48 && tiles <= 100) || (C_in <= 32 && tiles >= 512)) return true;
    if (C_in <= 64 && C_out > 64 && half_empty && tiles > 2 * kNumSMs) return true;
    return half_empty && tiles > 2 * kNumSMs && (C_in <= 48 || (C_in <= 64 && tiles >= 8 * kNumSMs));
}

template <typename T, int BN, bool kOutIn>
cudaError_t launch_forward(const ForwardParams<T>& p, cudaStream_t stream) {
    const dim3 grid((unsigned)ceil_div(p.M, kBM), (unsigned)ceil_div(p.C_out, BN));
    return launch_pdl(fma_forward_kernel<T, BN, kOutIn>, grid, dim3(Shape<BN>::kThreads), 0, stream, p);
}

template <typename T>
cudaError_t forward_typed(const void* X, const void* W, bool w_out_in, const float* bias, int64_t M, int64_t C_in, int64_t C_out, void* Y,
                          const int32_t* status_word, cudaStream_t stream) {
    ForwardParams<T> p;
    p.X = Operand<T>{(const T*)X, C_in, nullptr, M};
    p.W = Operand<T>{(const T*)W, w_out_in ? C_in : C_out, nullptr, C_out};
    p.bias = bias;
    p.Y = (T*)Y;
    p.M = M;
    p.C_in = (int)C_in;
    p.C_out = (int)C_out;
    p.status_word = status_word;
    if (short_reduction(M, C_in, C_out)) {
        const dim3 grid((unsigned)ceil_div(M, kBM), (unsigned)ceil_div(C_out, kBM));
        return w_out_in ? launch_pdl(fma_short_forward_kernel<T, true>, grid, dim3(kShortThreads), 0, stream, p)
                        : launch_pdl(fma_short_forward_kernel<T, false>, grid, dim3(kShortThreads), 0, stream, p);
    }
    if constexpr (sizeof(T) == 4) {
        if (C_out > 64 && ceil_div(M, kBM) * ceil_div(C_out, 128) >= 2 * kNumSMs)
            return w_out_in ? launch_forward<T, 128, true>(p, stream) : launch_forward<T, 128, false>(p, stream);
    }
    return w_out_in ? launch_forward<T, 64, true>(p, stream) : launch_forward<T, 64, false>(p, stream);
}

template <typename T, int BN, bool kOutIn>
cudaError_t launch_backward(const BackwardParams<T>& p, cudaStream_t stream) {
    const int64_t blocks = (int64_t)p.x_row_tiles * p.x_col_tiles + (int64_t)p.w_tiles * p.splits + p.zero_blocks;
    return launch_pdl(fma_backward_kernel<T, BN, kOutIn>, dim3((unsigned)blocks), dim3(Shape<BN>::kThreads), 0, stream, p);
}

template <typename T>
cudaError_t backward_typed(const BackwardParams<T>& p, bool wide, bool w_out_in, cudaStream_t stream) {
    if constexpr (sizeof(T) == 4) {
        if (wide) return w_out_in ? launch_backward<T, 128, true>(p, stream) : launch_backward<T, 128, false>(p, stream);
    }
    return w_out_in ? launch_backward<T, 64, true>(p, stream) : launch_backward<T, 64, false>(p, stream);
}

}  // namespace

cudaError_t launch_fma_forward(sbp_dtype dt, const void* X, const void* W, bool w_out_in, const float* bias, int64_t M,
                               int64_t C_in, int64_t C_out, void* Y, const int32_t* status_word, cudaStream_t stream) {
    return dt == SBP_BF16 ? forward_typed<__nv_bfloat16>(X, W, w_out_in, bias, M, C_in, C_out, Y, status_word, stream)
                          : forward_typed<float>(X, W, w_out_in, bias, M, C_in, C_out, Y, status_word, stream);
}

size_t fma_dw_workspace_bytes(sbp_dtype dt, int64_t M_keep_cap, int64_t C_in, int64_t C_out) {
    int most = 1;
    for (int v = 0; v < 4; ++v) {
        const int s = fma_plan(dt == SBP_F32, (v & 1) != 0, M_keep_cap, C_in, C_out, true, (v & 2) != 0).splits;
        if (s > most) most = s;
    }
    return most > 1 ? (size_t)most * (size_t)(C_in + 1) * (size_t)C_out * sizeof(float) : 0;
}

// a 16-deep step of a 64 x 64 (64 x 128) tile as part of the longest chain and of an SM's share, us; the start; the reduce launch
double fma_backward_us(bool out_in, int64_t M_keep_cap, int64_t C_in, int64_t C_out, bool want_dw, bool want_dx) {
    const FmaPlan pl = fma_plan(true, out_in, M_keep_cap, C_in, C_out, want_dw, want_dx);
    const double x_steps = (double)ceil_div(C_out, 16), w_steps = (double)ceil_div(ceil_div(M_keep_cap, 16), pl.splits);
    const double share = ((double)(pl.x_rows * pl.x_cols) * x_steps + (double)(pl.w_rows * pl.w_cols * pl.splits) * w_steps) / kNumSMs;
    const double chain = want_dx && (!want_dw || x_steps > w_steps) ? x_steps : w_steps;
    const double reduce = pl.splits > 1 ? 2.2 + 0.5 * (double)pl.splits * (double)C_in * (double)C_out * 8.0 / 4e6 : 0.0;
    return 3.6 + (pl.wide ? 0.8 * (chain + share) : 0.48 * chain + 0.36 * share) + reduce;
}

int fma_backward_kernel_count(sbp_dtype dt, bool w_out_in, int64_t M_keep_cap, int64_t C_in, int64_t C_out, bool want_dw, bool want_dx) {
    if (!want_dw && !want_dx) return 0;
    return 1 + (want_dw && fma_plan(dt == SBP_F32, w_out_in, M_keep_cap, C_in, C_out, want_dw, want_dx).splits > 1 ? 1 : 0);
}

cudaError_t launch_fma_backward(sbp_dtype dt, const void* X_keep, const void* dY, const void* W, bool w_out_in, const int32_t* dy_rows,
                                const int32_t* dx_rows, const int32_t* M_keep_dev, int64_t M, int64_t M_keep_cap, int64_t C_in,
                                int64_t C_out, float* dW, float* db, bool dw_accumulate, bool db_accumulate, void* dX,
                                float* workspace, const int32_t* status_word, cudaStream_t stream) {
    const FmaPlan pl = fma_plan(dt == SBP_F32, w_out_in, M_keep_cap, C_in, C_out, dW != nullptr, dX != nullptr);
    const bool split = dW != nullptr && pl.splits > 1;
    float* ws_db = workspace;                                          // [splits, C_out], then [splits, C_in * C_out]
    float* ws_dw = workspace + (int64_t)pl.splits * C_out;
    const auto fill = [&](auto& p) {
        p.dy_rows = dy_rows;
        p.dx_rows = dx_rows;
        p.M_keep_dev = M_keep_dev;
        p.M = M;
        p.M_keep_cap = M_keep_cap;
        p.C_in = (int)C_in;
        p.C_out = (int)C_out;
        p.dW = split ? ws_dw : dW;
        p.db = (db == nullptr || dW == nullptr) ? nullptr : (split ? ws_db : db);
        p.w_tiles = (int)(pl.w_rows * pl.w_cols);
        p.w_col_tiles = (int)pl.w_cols;
        p.splits = pl.splits;
        p.dw_accumulate = (dw_accumulate && !split) ? 1 : 0;
        p.db_accumulate = (db_accumulate && !split) ? 1 : 0;
        p.x_row_tiles = (int)pl.x_rows;
        p.x_col_tiles = (int)pl.x_cols;
        // 64 KB of rows or more a block, as many blocks as SMs at most
        const int64_t zero_bytes = M * C_in * (dt == SBP_BF16 ? 2 : 4);
        p.zero_blocks = dX == nullptr ? 0 : (int)(zero_bytes < (int64_t)kNumSMs << 16 ? ceil_div(zero_bytes, 1 << 16) : kNumSMs);
        p.status_word = status_word;
    };
    cudaError_t e;
    if (dt == SBP_BF16) {
        BackwardParams<__nv_bfloat16> p{};
        fill(p);
        p.X_keep = (const __nv_bfloat16*)X_keep; p.dY = (const __nv_bfloat16*)dY; p.W = (const __nv_bfloat16*)W; p.dX = (__nv_bfloat16*)dX;
        e = backward_typed(p, pl.wide, w_out_in, stream);
    } else {
        BackwardParams<float> p{};
        fill(p);
        p.X_keep = (const float*)X_keep; p.dY = (const float*)dY; p.W = (const float*)W; p.dX = (float*)dX;
        e = backward_typed(p, pl.wide, w_out_in, stream);
    }
    if (e != cudaSuccess || !split) return e;
    if (db != nullptr)
        return launch_reduce_partials_pair(ws_dw, pl.splits, C_in * C_out, dW, dw_accumulate, ws_db, pl.splits, C_out, db, db_accumulate,
                                           status_word, stream);
    return launch_reduce_partials(ws_dw, pl.splits, C_in * C_out, dW, dw_accumulate, status_word, stream);
}

}  // namespace sbp

// Convolutions with stride >= kernel size on the row-gather path (Sec. 3.2.2, the text after Eq. 6: with s >= k the
// neighbour effect disappears and the layer behaves like a point-wise one; ConvNeXt's 2 x 2 / stride 2 down-sampling
// layers are such layers).  Every output position reads its own k x k patch of the channels-last input, so the layer
// is a linear layer on "patch rows" of k * k * C values.  Two index kernels put that in front of and behind the
// linear-layer products:
//   patch cache:   X_keep[m, (dh, dw, c)] = X[b, s ho + dh, s wo + dw, c]   for the kept output positions m = (b, ho, wo):
//                  k contiguous pieces of k * C values per patch row (the forward cache of such a layer, Algorithm 1)
//   patch scatter: the packed input gradient [M_keep, k * k * C] back into dX [B, H, W, C]; every input position
//                  outside the kept patches (dropped positions, positions no patch covers when s > k) gets +0.0
// Both move 16-byte vectors and are HBM-bound.
#include "row_copy.cuh"

namespace sbp {
namespace {

struct PatchGeom {
    int H, W, Ho, Wo, k, s;
    int64_t vec_c;                  // 16-byte vectors per input position (C * element size / 16), below 2^22
    RowLength piece;                // vectors of one of the k pieces of a patch row
    FastDiv pieces;                 // k
    FastDiv map, line;              // output positions of a sample, of a row of the output map
    // Scatter: the input map in cells of side x side positions (cut short at the map's edges).  side = s: output position
    // (ho, wo) owns cell (ho, wo), cells past the output grid belong to none.  side = 1: every position by itself.
    int side, Hc, Wc;
    FastDiv cell;                   // vectors of a whole cell
    FastDiv cell_line;              // ... of one of its rows
    int cells_per_block;
    uint32_t slice;                 // vectors of its cells that a block writes (large cells: several blocks per cell)
};

// A block writes 1024 consecutive vectors of the patch rows.  Four 64-bit divisions a vector held it at 3.2 TB/s: 25088 patch
// rows of 512 bf16 16.0 -> 9.4 us (5.5 TB/s).
__global__ void __launch_bounds__(kCopyThreads)
patch_gather_kernel(const uint4* __restrict__ X, const PatchGeom g, const int32_t* __restrict__ keep_rows,
                    const int32_t* __restrict__ M_keep_dev, int64_t M_keep_cap, uint4* __restrict__ X_keep) {
    pdl_wait();
    const int64_t M_keep = load_m_keep(M_keep_dev, M_keep_cap);
    const int64_t begin = (int64_t)blockIdx.x * kCopySpan, total = M_keep_cap * g.k * g.piece.n;
    const SpanRows span(begin, g.piece);
    int64_t src[kCopyUnroll];
    uint4 v[kCopyUnroll];
#pragma unroll
    for (int u = 0; u < kCopyUnroll; ++u) {
        uint32_t q;
        const int64_t off = span.place(threadIdx.x + u * kCopyThreads, g.piece, &q);
        const uint32_t i = (uint32_t)span.first + q, m = g.pieces(i), dh = i - m * g.pieces.d;
        src[u] = -1;                                                   // rows past M_keep are cleared
        if (m < M_keep) {
            const uint32_t pos = (uint32_t)__ldg(keep_rows + m);
            const uint32_t b = g.map(pos), rem = pos - b * g.map.d;
            const uint32_t ho = g.line(rem), wo = rem - ho * g.line.d;
            const int64_t pix = ((int64_t)b * g.H + (int64_t)g.s * ho + dh) * g.W + (int64_t)g.s * wo;
            src[u] = pix * g.vec_c + off;
        }
    }
#pragma unroll
    for (int u = 0; u < kCopyUnroll; ++u) v[u] = (src[u] >= 0) ? ld_stream(X + src[u]) : make_uint4(0u, 0u, 0u, 0u);
#pragma unroll
    for (int u = 0; u < kCopyUnroll; ++u) {
        const int64_t i = begin + threadIdx.x + u * kCopyThreads;
        if (i < total) X_keep[i] = v[u];
    }
    pdl_launch_dependents();
}

// slot[pos] = the packed row of output position pos.  Positions that are not kept keep whatever the workspace held: the reader asks
// keep_rows back, so that nothing has to be cleared first, and the list may be in any order.
__global__ void patch_slots_kernel(const int32_t* __restrict__ keep_rows, const int32_t* __restrict__ M_keep_dev, int64_t M_keep_cap,
                                   int64_t outputs, int32_t* __restrict__ slot, const int32_t* status_word) {
    pdl_launch_dependents();
    pdl_wait();
    if (status_word != nullptr && *reinterpret_cast<const volatile int32_t*>(status_word) != 0) return;
    const int64_t M_keep = load_m_keep(M_keep_dev, M_keep_cap), m = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (m >= M_keep) return;
    const int64_t pos = __ldg(keep_rows + m);
    if (pos >= 0 && pos < outputs) slot[pos] = (int32_t)m;
}

// A block writes the input positions of `cells_per_block` consecutive cells, 1024 vectors at a time.  [64, 56, 56, 128] bf16 from
// 25088 packed rows, with the launch that fills the slots: 18.2 us (77 MB; with the list searched by every block instead, which
// needs it ascending: the same).
constexpr int kMaxCells = 128;
__global__ void __launch_bounds__(kCopyThreads)
patch_scatter_kernel(const uint4* __restrict__ dXp, const PatchGeom g, const int32_t* __restrict__ keep_rows,
                     const int32_t* __restrict__ M_keep_dev, int64_t M_keep_cap, const int32_t* __restrict__ slot, int64_t cells,
                     uint4* __restrict__ dX, const int32_t* status_word) {
    __shared__ int64_t from_of[kMaxCells];         // first vector of each cell's packed patch, -1: none
    __shared__ int32_t pixel_of[kMaxCells];        // first input position of each cell
    __shared__ int2 room[kMaxCells];               // rows of the cell inside the map, vectors of such a row
    pdl_launch_dependents();
    pdl_wait();
    if (status_word != nullptr && *reinterpret_cast<const volatile int32_t*>(status_word) != 0) return;
    const int64_t M_keep = load_m_keep(M_keep_dev, M_keep_cap);
    const int64_t c0 = (int64_t)blockIdx.x * g.cells_per_block;
    const int n = cells - c0 < g.cells_per_block ? (int)(cells - c0) : g.cells_per_block;
    if ((int)threadIdx.x < n) {
        const int i = threadIdx.x;
        const int64_t c = c0 + i, bh = c / g.Wc, b = bh / g.Hc;
        const int wc = (int)(c - bh * g.Wc), hc = (int)(bh - b * g.Hc);
        const int h0 = hc * g.side, w0 = wc * g.side;
        const int ho = g.side == g.s ? hc : h0 / g.s, wo = g.side == g.s ? wc : w0 / g.s, dh0 = h0 - ho * g.s, dw0 = w0 - wo * g.s;
        int64_t from = -1;
        if (ho < g.Ho && wo < g.Wo && dh0 < g.k && dw0 < g.k) {
            const int32_t pos = (int32_t)((b * g.Ho + ho) * g.Wo + wo), m = __ldg(slot + pos);
            if (m >= 0 && m < M_keep && __ldg(keep_rows + m) == pos) from = ((int64_t)m * g.k + dh0) * g.piece.n + dw0 * g.vec_c;
        }
        from_of[i] = from;
        pixel_of[i] = (int32_t)((b * g.H + h0) * g.W + w0);
        const int rows = g.H - h0 < g.side ? g.H - h0 : g.side, cols = g.W - w0 < g.side ? g.W - w0 : g.side;
        room[i] = make_int2(rows, cols * (int)g.vec_c);
    }
    __syncthreads();
    const uint32_t all = (uint32_t)n * g.cell.d, slice0 = blockIdx.y * g.slice;
    const uint32_t vectors = all - slice0 < g.slice ? all : slice0 + g.slice;
    for (uint32_t base = slice0 + threadIdx.x; base < vectors; base += kCopySpan) {
        uint4 v[kCopyUnroll];
        int64_t dst[kCopyUnroll];
#pragma unroll
        for (int u = 0; u < kCopyUnroll; ++u) {
            const uint32_t i = base + u * kCopyThreads;
            dst[u] = -1;
            v[u] = make_uint4(0u, 0u, 0u, 0u);
            if (i < vectors) {
                const uint32_t c = g.cell(i), in_cell = i - c * g.cell.d;
                const uint32_t dh = g.cell_line(in_cell), off = in_cell - dh * g.cell_line.d;
                if ((int)dh < room[c].x && (int)off < room[c].y) {
                    dst[u] = ((int64_t)pixel_of[c] + (int64_t)dh * g.W) * g.vec_c + off;
                    const int64_t from = from_of[c];
                    if (from >= 0 && (int)dh < g.k && off < g.piece.n) v[u] = ld_stream(dXp + from + dh * g.piece.n + off);
                }
            }
        }
#pragma unroll
        for (int u = 0; u < kCopyUnroll; ++u)
            if (dst[u] >= 0) dX[dst[u]] = v[u];
    }
}

PatchGeom geom(int64_t H, int64_t W, int64_t k, int64_t s, int64_t pos_bytes) {
    const int64_t most = H > W ? H : W;
    if (s > most) s = most;                        // (one output row or column either way)
    PatchGeom g;
    g.H = (int)H; g.W = (int)W; g.k = (int)k; g.s = (int)s;
    g.Ho = (int)((H - k) / s + 1); g.Wo = (int)((W - k) / s + 1);
    g.vec_c = pos_bytes / 16;
    g.piece = RowLength(k * g.vec_c);
    g.pieces = FastDiv((uint32_t)k);               // (pieces in all: at most the input positions / k, so they fit 31 bits)
    g.map = FastDiv((uint32_t)((int64_t)g.Ho * g.Wo));
    g.line = FastDiv((uint32_t)g.Wo);
    return g;
}

}  // namespace

cudaError_t launch_patch_gather(const void* X, int64_t H, int64_t W, int64_t pos_bytes, int64_t k, int64_t s,
                                const int32_t* keep_rows, const int32_t* M_keep_dev, int64_t M_keep_cap, void* X_keep,
                                cudaStream_t stream) {
    const PatchGeom g = geom(H, W, k, s, pos_bytes);
    const int64_t total = M_keep_cap * k * g.piece.n;
    if (total == 0) return cudaSuccess;
    return launch_pdl(patch_gather_kernel, dim3((unsigned)copy_blocks(total)), dim3(kCopyThreads), 0, stream, (const uint4*)X, g,
                      keep_rows, M_keep_dev, M_keep_cap, (uint4*)X_keep);
}

cudaError_t launch_patch_scatter(const void* dXp, int64_t B, int64_t H, int64_t W, int64_t pos_bytes, int64_t k, int64_t s,
                                 const int32_t* keep_rows, const int32_t* M_keep_dev, int64_t M_keep_cap, void* dX,
                                 int32_t* slot, const int32_t* status_word, cudaStream_t stream) {
    PatchGeom g = geom(H, W, k, s, pos_bytes);
    if (M_keep_cap > 0) {
        const cudaError_t e = launch_pdl(patch_slots_kernel, dim3((unsigned)((M_keep_cap + 255) / 256)), dim3(256), 0, stream, keep_rows,
                                         M_keep_dev, M_keep_cap, B * g.Ho * g.Wo, slot, status_word);
        if (e != cudaSuccess) return e;
    }
    // Cells of more than a gigabyte (strides far beyond the kernel) are taken apart into positions, so that vectors are counted in
    // 32 bits everywhere.
    const auto cell_side = [&](int64_t extent) { return g.s < extent ? (int64_t)g.s : extent; };
    g.side = cell_side(H) * cell_side(W) * g.vec_c <= (1ll << 26) ? g.s : 1;
    g.Hc = (int)((H + g.side - 1) / g.side);
    g.Wc = (int)((W + g.side - 1) / g.side);
    const int64_t cells = B * g.Hc * g.Wc;
    const int64_t cell_w = g.side < W ? g.side : W, cell_h = g.side < H ? g.side : H;
    g.cell_line = FastDiv((uint32_t)(cell_w * g.vec_c));
    g.cell = FastDiv((uint32_t)(cell_h * cell_w * g.vec_c));
    // About 2048 vectors (32 KB) a block: eight blocks of an SM then hide each other's look-ups, and small maps still spread.
    constexpr uint32_t kTarget = 2048;
    const uint32_t n = kTarget / g.cell.d;
    g.cells_per_block = (int)(n < 1 ? 1 : n > (uint32_t)kMaxCells ? (uint32_t)kMaxCells : n);
    const uint32_t per_block = (uint32_t)g.cells_per_block * g.cell.d;
    uint32_t slices = (per_block + kTarget - 1) / kTarget;
    if (slices > 65535u) slices = 65535u;
    g.slice = (per_block + slices - 1) / slices;
    slices = (per_block + g.slice - 1) / g.slice;
    const dim3 grid((unsigned)((cells + g.cells_per_block - 1) / g.cells_per_block), slices);
    return launch_pdl(patch_scatter_kernel, grid, dim3(kCopyThreads), 0, stream, (const uint4*)dXp, g, keep_rows, M_keep_dev, M_keep_cap,
                      (const int32_t*)slot, cells, (uint4*)dX, status_word);
}

}  // namespace sbp

// Forward cache (Algorithm 1: only inputs[keep] is retained): a compacting row gather,
// X_keep[m, :] = X[keep_rows[m], :], moved as 16-byte vectors.  HBM-bound: it reads and writes
// M_keep * row_bytes bytes each and never touches a dropped row.  Rows in [M_keep, M_keep_cap)
// of the destination are cleared so that later products over the padded capacity see zeros.
// Also holds the optional device-side check of the index list.
#include "row_copy.cuh"

namespace sbp {
namespace {

// A block writes 1024 consecutive vectors (16 KB); without a 64-bit division for each of them 12544 rows of 768 bf16 take
// 7.7 us instead of 9.1 us (5.0 TB/s with launch and drain inside), 100352 rows of 512 28 us instead of 32 us (7.4 TB/s).
__global__ void __launch_bounds__(kCopyThreads)
gather_rows_kernel(const uint4* __restrict__ X, const RowLength row, const int32_t* __restrict__ keep_rows,
                   const int32_t* __restrict__ M_keep_dev, int64_t M_keep_cap, uint4* __restrict__ X_keep) {
    pdl_wait();
    const int64_t M_keep = load_m_keep(M_keep_dev, M_keep_cap);
    const int64_t begin = (int64_t)blockIdx.x * kCopySpan, total = M_keep_cap * row.n;
    const SpanRows span(begin, row);
    uint4 v[kCopyUnroll];
    int64_t src[kCopyUnroll];
#pragma unroll
    for (int u = 0; u < kCopyUnroll; ++u) {
        uint32_t q;
        const int64_t c = span.place(threadIdx.x + u * kCopyThreads, row, &q);
        const int64_t m = span.first + q;
        src[u] = m < M_keep ? (int64_t)__ldg(keep_rows + m) * row.n + c : -1;
    }
#pragma unroll
    for (int u = 0; u < kCopyUnroll; ++u) v[u] = (src[u] >= 0) ? ld_stream(X + src[u]) : make_uint4(0u, 0u, 0u, 0u);
#pragma unroll
    for (int u = 0; u < kCopyUnroll; ++u) {
        const int64_t i = begin + threadIdx.x + u * kCopyThreads;
        if (i < total) X_keep[i] = v[u];
    }
    // Only now may the next kernel's blocks take their places: the usual successor (the backward kernel) needs
    // a whole SM per block, and resident early it would push this kernel's remaining blocks off the SMs.
    pdl_launch_dependents();
}

__global__ void validate_keep_rows_kernel(const int32_t* __restrict__ keep_rows,
                                          const int32_t* __restrict__ M_keep_dev, int64_t M_keep_cap,
                                          int64_t M, int32_t* status_word) {
    pdl_launch_dependents();
    pdl_wait();
    const int64_t M_keep = load_m_keep(M_keep_dev, M_keep_cap);
    if (M_keep_dev != nullptr && blockIdx.x == 0 && threadIdx.x == 0) {
        const int64_t raw = (int64_t)__ldg(M_keep_dev);
        if (raw < 0 || raw > M_keep_cap) report_device_error(status_word, SBP_ERR_BAD_INDICES);
    }
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t m = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; m < M_keep; m += stride) {
        const int64_t r = keep_rows[m];
        const int64_t prev = (m > 0) ? (int64_t)keep_rows[m - 1] : -1;
        if (r < 0 || r >= M || r <= prev) report_device_error(status_word, SBP_ERR_BAD_INDICES);
    }
}

}  // namespace

cudaError_t launch_gather_rows(const void* X, int64_t row_bytes, const int32_t* keep_rows,
                               const int32_t* M_keep_dev, int64_t M_keep_cap, void* X_keep,
                               cudaStream_t stream) {
    const int64_t vec_per_row = row_bytes / 16;
    const int64_t total = M_keep_cap * vec_per_row;
    if (total == 0) return cudaSuccess;
    return launch_pdl(gather_rows_kernel, dim3((unsigned)copy_blocks(total)), dim3(kCopyThreads), 0, stream, (const uint4*)X,
                      RowLength(vec_per_row), keep_rows, M_keep_dev, M_keep_cap, (uint4*)X_keep);
}

cudaError_t launch_validate_keep_rows(const int32_t* keep_rows, const int32_t* M_keep_dev,
                                      int64_t M_keep_cap, int64_t M, int32_t* status_word,
                                      cudaStream_t stream) {
    int64_t blocks = (M_keep_cap + 255) / 256;
    if (blocks < 1) blocks = 1;
    if (blocks > kNumSMs * 8) blocks = kNumSMs * 8;
    return launch_pdl(validate_keep_rows_kernel, dim3((unsigned)blocks), dim3(256), 0, stream,
                      keep_rows, M_keep_dev, M_keep_cap, M, status_word);
}

}  // namespace sbp

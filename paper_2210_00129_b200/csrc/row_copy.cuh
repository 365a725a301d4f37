// Index arithmetic of the copy kernels: a block moves a contiguous span of 16-byte vectors of its destination.  Divisions by
// sizes that are only known at run time are multiplications (a 64-bit division a vector held the copies below half of the
// memory rate), and the one 64-bit division left is the block's, not the vector's.
#pragma once

#include "sbp_common.cuh"

namespace sbp {

// n / d for n < 2^31: (umulhi(n, mul) + n) >> shift  (Granlund and Montgomery, PLDI 1994)
struct FastDiv {
    uint32_t d, mul, shift;
    FastDiv() = default;
    explicit FastDiv(uint32_t divisor) : d(divisor), shift(0) {
        while (shift < 31 && (1u << shift) < d) ++shift;
        mul = (uint32_t)(((1ull << 32) * ((1ull << shift) - d)) / d + 1);
    }
    __device__ __forceinline__ uint32_t operator()(uint32_t n) const { return (__umulhi(n, mul) + n) >> shift; }
};

constexpr int kCopyThreads = 256;
constexpr int kCopyUnroll = 4;             // vectors a thread has in flight
constexpr uint32_t kCopySpan = kCopyThreads * kCopyUnroll;

// Length of a row in vectors: any length, but only rows shorter than a span are divided by.
struct RowLength {
    int64_t n;
    FastDiv by;
    RowLength() = default;
    explicit RowLength(int64_t vectors) : n(vectors), by(vectors < kCopySpan ? (uint32_t)vectors : 1u) {}
};

// Position of a span in rows of `row.n` vectors: vector `i` of the span (i < kCopySpan) lies in row first + (*q), at the
// returned place in it.
struct SpanRows {
    int64_t first, rem;
    __device__ __forceinline__ SpanRows(int64_t span_begin, const RowLength& row) {
        first = span_begin / row.n;
        rem = span_begin - first * row.n;
    }
    __device__ __forceinline__ int64_t place(uint32_t i, const RowLength& row, uint32_t* q) const {
        if (row.n >= kCopySpan) {                                        // long rows: a span touches two at most
            const int64_t o = rem + i;
            *q = o >= row.n ? 1u : 0u;
            return o >= row.n ? o - row.n : o;
        }
        const uint32_t o = (uint32_t)rem + i;
        *q = row.by(o);
        return o - *q * row.by.d;
    }
};

inline int64_t copy_blocks(int64_t vectors) { return (vectors + kCopySpan - 1) / kCopySpan; }

__device__ __forceinline__ uint4 ld_stream(const uint4* p) {
    uint4 v;
    asm volatile("ld.global.nc.L1::no_allocate.v4.u32 {%0,%1,%2,%3}, [%4];"
                 : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "l"(p));
    return v;
}

}  // namespace sbp

// Pieces shared by the CUDA-core kernels (forward and backward): tiles of rows in shared memory as fp32, and register-tiled
// products on them.
//
// Every tile is kept row-major ("natural") with a row stride that is 4 modulo 8 floats: eight consecutive rows read at the same
// 16-byte column piece then fall into eight different bank groups, so the products that contract over the head dimension read
// both operands four columns at a time without a transposed copy.
#pragma once
#include "tlin_internal.h"

namespace tlin {
namespace simt {

__host__ __device__ constexpr int row_stride(int d) { return d % 8 == 4 ? d : d + 4; }      // d is a multiple of 4

__device__ __forceinline__ float get(const float4& v, int e) { return e == 0 ? v.x : e == 1 ? v.y : e == 2 ? v.z : v.w; }

__device__ __forceinline__ void cp_async16(float* dst, const float* src, bool valid) {       // zeros where !valid
    const uint32_t s = (uint32_t)__cvta_generic_to_shared(dst);
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(s), "l"(src), "r"(valid ? 16 : 0) : "memory");
}
__device__ __forceinline__ void cp_async_wait() { asm volatile("cp.async.wait_all;" ::: "memory"); }

// rows [r0, r0 + ROWS) of a [rows_total, d] matrix -> shared memory (row stride ld), rows beyond rows_total as zeros.
// fp32 rows go by asynchronous copies (cp_async_wait before the barrier), bf16 rows are widened on the way.
template <int ROWS, int NT>
__device__ __forceinline__ void load_rows(float* dst, int ld, const float* __restrict__ src, int r0, int rows_total, int d) {
    const int per_row = d >> 2, dr = NT / per_row, dc = NT - dr * per_row;
    int r = threadIdx.x / per_row, c = threadIdx.x - r * per_row;
    while (r < ROWS) {
        const bool ok = r0 + r < rows_total;
        cp_async16(dst + r * ld + c * 4, src + (ok ? (int64_t)(r0 + r) * d + c * 4 : 0), ok);
        r += dr;
        c += dc;
        if (c >= per_row) {
            c -= per_row;
            ++r;
        }
    }
}
template <int ROWS, int NT>
__device__ __forceinline__ void load_rows(float* dst, int ld, const __nv_bfloat16* __restrict__ src, int r0, int rows_total, int d) {
    const int per_row = d >> 3, dr = NT / per_row, dc = NT - dr * per_row;
    int r = threadIdx.x / per_row, c = threadIdx.x - r * per_row;
    while (r < ROWS) {
        uint4 w = make_uint4(0u, 0u, 0u, 0u);
        if (r0 + r < rows_total) w = *reinterpret_cast<const uint4*>(src + (int64_t)(r0 + r) * d + c * 8);
        float4* p = reinterpret_cast<float4*>(dst + r * ld + c * 8);
        p[0] = make_float4(__uint_as_float(w.x << 16), __uint_as_float(w.x & 0xffff0000u), __uint_as_float(w.y << 16), __uint_as_float(w.y & 0xffff0000u));
        p[1] = make_float4(__uint_as_float(w.z << 16), __uint_as_float(w.z & 0xffff0000u), __uint_as_float(w.w << 16), __uint_as_float(w.w & 0xffff0000u));
        r += dr;
        c += dc;
        if (c >= per_row) {
            c -= per_row;
            ++r;
        }
    }
}

// acc[i][j] += A[row_i] . B[row_j] over the d columns; A rows a0 + i * a_step, B rows b0 + j * b_step (pointers to the first row)
template <int NI, int NJ>
__device__ __forceinline__ void dot_tile(float (&acc)[NI][NJ], const float* a0, int a_step, const float* b0, int b_step, int d) {
#pragma unroll 1
    for (int c = 0; c < d; c += 4) {
        float4 a[NI];
#pragma unroll
        for (int i = 0; i < NI; ++i) a[i] = *reinterpret_cast<const float4*>(a0 + i * a_step + c);
#pragma unroll
        for (int j = 0; j < NJ; ++j) {
            const float4 b = *reinterpret_cast<const float4*>(b0 + j * b_step + c);
#pragma unroll
            for (int i = 0; i < NI; ++i) {
                acc[i][j] = fmaf(a[i].x, b.x, acc[i][j]);
                acc[i][j] = fmaf(a[i].y, b.y, acc[i][j]);
                acc[i][j] = fmaf(a[i].z, b.z, acc[i][j]);
                acc[i][j] = fmaf(a[i].w, b.w, acc[i][j]);
            }
        }
    }
}

// Columns of a result row that thread `tc` of TC owns: CM / 4 groups of four neighbours (group g: 4 TC g + 4 tc ...), then CM % 4
// single ones (TC apart).  Both forms read and write contiguous lines across the TC threads.
template <int TC, int CM>
__device__ __forceinline__ int column_of(int m, int tc) {
    return m < CM / 4 * 4 ? (m / 4) * 4 * TC + 4 * tc + m % 4 : CM / 4 * 4 * TC + (m - CM / 4 * 4) * TC + tc;
}
// the owned columns of one row in shared memory (columns beyond the head size read whatever lies there; they are never stored)
template <int TC, int CM>
__device__ __forceinline__ void load_columns(float (&b)[CM], const float* row, int tc) {
#pragma unroll
    for (int g = 0; g < CM / 4; ++g) {
        const float4 v = *reinterpret_cast<const float4*>(row + g * 4 * TC + 4 * tc);
        b[g * 4] = v.x; b[g * 4 + 1] = v.y; b[g * 4 + 2] = v.z; b[g * 4 + 3] = v.w;
    }
#pragma unroll
    for (int m = CM / 4 * 4; m < CM; ++m) b[m] = row[column_of<TC, CM>(m, tc)];
}
// floats that load_columns may read beyond the d columns of a row
template <int TC, int CM>
constexpr int column_slack() { return TC * CM; }

__device__ __forceinline__ void store4(float* p, float a, float b, float c, float d) { *reinterpret_cast<float4*>(p) = make_float4(a, b, c, d); }
__device__ __forceinline__ void store4(__nv_bfloat16* p, float a, float b, float c, float d) {
    const __nv_bfloat162 x = __floats2bfloat162_rn(a, b), y = __floats2bfloat162_rn(c, d);
    *reinterpret_cast<uint2*>(p) = make_uint2(*reinterpret_cast<const uint32_t*>(&x), *reinterpret_cast<const uint32_t*>(&y));
}
__device__ __forceinline__ void store1(float* p, float a) { *p = a; }
__device__ __forceinline__ void store1(__nv_bfloat16* p, float a) { *p = __float2bfloat16_rn(a); }

// the owned columns (those below d) of one row, times f
template <int TC, int CM, typename T>
__device__ __forceinline__ void store_columns(T* row, const float (&v)[CM], float f, int tc, int d) {
#pragma unroll
    for (int g = 0; g < CM / 4; ++g) {
        const int c = g * 4 * TC + 4 * tc;                      // d is a multiple of 4: a group is inside or outside as a whole
        if (c < d) store4(row + c, v[g * 4] * f, v[g * 4 + 1] * f, v[g * 4 + 2] * f, v[g * 4 + 3] * f);
    }
#pragma unroll
    for (int m = CM / 4 * 4; m < CM; ++m) {
        const int c = column_of<TC, CM>(m, tc);
        if (c < d) store1(row + c, v[m] * f);
    }
}

}  // namespace simt
}  // namespace tlin

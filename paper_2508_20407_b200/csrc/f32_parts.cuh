// fp32 tensors on the bf16 tensor pipe: an fp32 number is the sum of three bf16 numbers, exactly (3 x 8 significant bits, each part
// the rounding of what the ones before it leave).  A product of two such sums needs six of its nine partial products for fp32
// accuracy; the other three are below 2^-24 of it.  Six bf16 products with fp32 accumulation run at a sixth of the bf16 rate, 375
// TFLOP/s nominal where the CUDA cores have 72.
//
// The parts of the tensors are made by one pass over them (split_kernel) into scratch that the caller provides, [part][b h][row][d8]
// with d8 = d rounded up to 8, which the tensor maps then read with zero fill beyond d8.  Numbers outside [2^-100, 2^30] (dout: 2^20) other than 0
// (infinities, what would lose its low parts or overflow on the way) are found there: a (b,h) with such a number runs on the CUDA cores
// instead, decided on the device.  The split kernel's blocks leave one word each, several blocks to a (b,h); the tensor kernels read the
// words and leave those (b,h) out that have one set, and the CUDA-core kernel behind them computes these and returns at once if there
// are none.
#pragma once
#include "tlin_internal.h"
#include "sm100_ptx.cuh"
#include "tc_common.cuh"

namespace tlin {
namespace f32 {

constexpr int kParts = 3;
constexpr int kSplitThreads = 256;
constexpr int kSplitBlocks = 6 * kDefaultSMs;          // up to; more (b,h) get one each
// partial products in ascending size, so that the small ones are added while the sum is small: (part of A, part of B)
__host__ __device__ constexpr int product_a(int i) { return i == 0 ? 0 : i == 1 ? 1 : i == 2 ? 2 : i == 3 ? 0 : i == 4 ? 1 : 0; }
__host__ __device__ constexpr int product_b(int i) { return i == 0 ? 2 : i == 1 ? 1 : i == 3 ? 1 : 0; }
constexpr int kProducts = 6;
// ds is split into parts too, and a bf16 part below 2^-133 is lost.  The backward therefore runs on 2^19 dout (exactly that times the
// gradients), which dout up to 2^20 leaves room for: 64 * 2^39 * 2^30 = 2^75 in dp, 2^106 in a product with q or k.  Relative error of
// dk, dout 2^-90 and v 2^-20 times normal: without 9.1e-6, so 3.4e-7.
constexpr float kDoutScale = 524288.f;

inline long long padded_head(int d) { return ((long long)d + 7) / 8 * 8; }
inline int padded_rows(int W) { return (W + 127) / 128 * 128; }

// What the split kernel makes: the parts of up to four tensors of n_bh (b,h), and for the backward (kDoutTensor is dout there, its parts of
// kDoutScale times it) the row statistics.
constexpr int kDoutTensor = 1;
struct SplitJobs {
    const float* src[4];
    __nv_bfloat16* dst[4];
    int rows[4];                  // per (b,h)
    int n, d;
    long long n_bh;
    int per_bh;                   // blocks
    int nan_too;                  // bit t: a NaN in tensor t is one of the numbers that the parts do not hold
    int* words;                   // one per block
    const float *out, *dout, *lse;
    float *neg_lse, *delta;       // [n_bh][Wpad]: -lse (beyond W: -inf) and kDoutScale out . dout (beyond W: 0); null in the forward
    float* plain_delta;           // [n_bh][W]: out . dout as the CUDA-core kernel sums and reads it
    int W, Wpad;
    float* zero;                  // [n_bh][W][d] to clear, or null
};
// Blocks per (b,h), with `groups` groups of eight numbers each.  An even number: B8 H12 N1024 W512 d36 backward, with 6, 8 or 10 of them
// 275 us, with 7 or 9 285, of which the split itself is 1 to 3.
inline int split_blocks(long long n_bh, long long groups) {
    const long long share = kSplitBlocks / n_bh < 2 ? kSplitBlocks / n_bh : kSplitBlocks / n_bh / 2 * 2, most = (groups + kSplitThreads - 1) / kSplitThreads;
    return (int)(share < 1 ? 1 : share < most ? share : most);
}
int launch_split(const SplitJobs& jobs, cudaStream_t st);
// No call takes more scratch than this, which an allocator keeps once it has been asked for it.  Few query tiles over long histories are
// what would: forward, unbounded / 2 GiB / 1 GiB / on the CUDA cores, microseconds: B1 H32 N131072 W128 d128 (6.0 GiB) 3500 / 4890 / 7170 /
// 11720, B8 H32 N65536 W100 d36 (7.5) 4590 / 6020 / 6320 / 14990, B1 H16 N131072 W128 d128 (3.0) 2450 / 2440 / 3970 / 8780, B1 H32
// N131072 W1024 d64 (3.0) 5750 / 5750 / 5770 / 31700.
constexpr size_t kMaxScratch = (size_t)2 << 30;
// Parts of `rows` rows in all, in bytes
inline size_t part_bytes(long long rows, int d) { return (size_t)kParts * 2 * rows * padded_head(d); }

// Two numbers -> their parts, packed, each part cut off instead of rounded (still exact: 8 + 8 + 8 bits): for p and ds, made and split in
// the inner loops, without conversions.  The tensors' parts are rounded, so the dropped products have no sign of their own.
__device__ __forceinline__ void cut2(uint64_t x, uint32_t& p0, uint32_t& p1, uint32_t& p2) {
    using namespace ptx;
    const uint64_t minus_one = f2_pack(-1.f, -1.f);
    auto high_halves = [](uint64_t v) { return __byte_perm((uint32_t)v, (uint32_t)(v >> 32), 0x7632); };
    auto cut = [](uint64_t v) { return f2_pack_bits((uint32_t)v & 0xffff0000u, (uint32_t)(v >> 32) & 0xffff0000u); };
    p0 = high_halves(x);
    x = f2_fma(cut(x), minus_one, x);
    p1 = high_halves(x);
    x = f2_fma(cut(x), minus_one, x);
    p2 = high_halves(x);
}
// two numbers -> their parts, packed, rounded
__device__ __forceinline__ void split2(float x0, float x1, uint32_t (&part)[kParts]) {
    using namespace ptx;
    part[0] = pack_bf16x2(x0, x1);
    float r0 = x0 - __uint_as_float(part[0] << 16), r1 = x1 - __uint_as_float(part[0] & 0xffff0000u);
    part[1] = pack_bf16x2(r0, r1);
    r0 -= __uint_as_float(part[1] << 16);
    r1 -= __uint_as_float(part[1] & 0xffff0000u);
    part[2] = pack_bf16x2(r0, r1);
}

}  // namespace f32
}  // namespace tlin

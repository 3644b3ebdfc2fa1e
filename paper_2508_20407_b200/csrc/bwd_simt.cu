// Backward pass of the attention layer on the CUDA cores (fp32 arithmetic; bf16 or fp32 tensors; any head size the
// CUDA-core forward takes): the chain rule applied to the Section 3 attention formula with the window mask.  Training
// runs every layer as a forward and a backward pass ("cache miss" throughout, Section 4.1); the paper gives no separate
// algorithm for the gradient.
//
//   p_ij  = exp(s_ij - lse_i),  s_ij = q_i.k_j / sqrt(d)      (lse saved by the forward, so no second softmax pass)
//   delta_i = dout_i . out_i   ( = sum_j p_ij dp_ij )
//   dv_j  = sum_i p_ij dout_i          dp_ij = dout_i . v_j          ds_ij = p_ij (dp_ij - delta_i) / sqrt(d)
//   dq_i  = sum_j ds_ij k_j            dk_j  = sum_i ds_ij q_i
//
// delta: one warp per query row.  Main kernel: one CTA per tile of keys of a (b,h), looping over the query tiles that can see
// it; the scores are computed once per (query, key) tile and give all three gradients: dk/dv stay in registers until the end
// (one owner each, nothing is atomic), the tile's dq is added to an fp32 dq by vector reductions in L2 (cleared first; the fp32
// result itself, or a buffer in the workspace that a last kernel rounds to bf16).
//
// Bound by the FFMA rate: five products of 2 d FLOP per pair.  64 x 64 tiles (32 x 32 beyond d = 128, where four 64-row tiles do
// not fit the shared memory), 128 threads up to d = 64 and 256 beyond; a thread holds 4 x 8 (4 x 4) scores and 4 rows of CM
// columns of each result, 5 to 16 FFMA per shared-memory read.  The kernels before it (two passes over the scores, one score
// per thread and step, five reads per eight FFMA) against this one, fp32: B8 H12 N1024 W512 d36 2181 -> 448 us (30 TFLOP/s),
// B4 H12 N1500 W700 d128 6088 -> 1496 us (33 TFLOP/s).
//
// This is the fp32 path and the path for bf16 head sizes other than 64 and 128 (the counterpart of fwd_simt.cu).
#include "tlin_internal.h"
#include "simt_tiles.cuh"
#include <algorithm>
#include <math_constants.h>

namespace tlin {
namespace {

using namespace simt;

constexpr float kLog2e = 1.4426950408889634f;
constexpr int kTR = 16;                 // row groups of a CTA

__device__ __forceinline__ float to_f(__nv_bfloat16 x) { return __bfloat162float(x); }
__device__ __forceinline__ float to_f(float x) { return x; }
__device__ __forceinline__ void from_f(__nv_bfloat16& dst, float x) { dst = __float2bfloat16_rn(x); }
__device__ __forceinline__ void from_f(float& dst, float x) { dst = x; }

// delta_i = dout_i . out_i, one warp per row
template <typename T>
__global__ void __launch_bounds__(256)
bwd_delta_kernel(const T* __restrict__ out, const T* __restrict__ dout, float* __restrict__ delta, long long rows, int d) {
    const long long row = (long long)blockIdx.x * 8 + (threadIdx.x >> 5);
    if (row >= rows) return;
    const int lane = threadIdx.x & 31;
    float acc = 0.f;
    for (int c = lane; c < d; c += 32) acc = fmaf(to_f(out[row * d + c]), to_f(dout[row * d + c]), acc);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
    if (lane == 0) delta[row] = acc;
}

// shared memory: Q, dout, K, V tiles, P and dS as [row][key], lse and delta of the rows
template <int BT>
__host__ __device__ constexpr int ld_p() { return BT + 8; }      // 8 modulo 32: four rows x eight keys written by a warp hit 32 banks
template <int BT>
size_t bwd_smem_bytes(int d, int slack) { return sizeof(float) * (4 * BT * row_stride(d) + 2 * BT * ld_p<BT>() + 2 * BT + slack); }

// acc[i][c] += sum over the BT rows r of A[r][a + i] * B[r][columns]   (A row stride ld_p, B row stride ld)
template <int BT, int TC, int KA, int CM>
__device__ __forceinline__ void accumulate_over_rows(float (&acc)[KA][CM], const float* A, const float* B, int ld, int tc) {
#pragma unroll 2
    for (int r = 0; r < BT; ++r) {
        float a[KA], b[CM];
        if constexpr (KA == 4) {
            const float4 x = *reinterpret_cast<const float4*>(A + r * ld_p<BT>());
            a[0] = x.x; a[1] = x.y; a[2] = x.z; a[3] = x.w;
        } else {
            const float2 x = *reinterpret_cast<const float2*>(A + r * ld_p<BT>());
            a[0] = x.x; a[1] = x.y;
        }
        load_columns<TC, CM>(b, B + r * ld, tc);
#pragma unroll
        for (int i = 0; i < KA; ++i)
#pragma unroll
            for (int c = 0; c < CM; ++c) acc[i][c] = fmaf(a[i], b[c], acc[i][c]);
    }
}

template <typename T, int BT, int TC, int CM>
__global__ void __launch_bounds__(kTR * TC, CM * TC <= 40 ? 3 : CM * TC <= 64 ? 2 : 1)
bwd_simt_kernel(const T* __restrict__ q, const T* __restrict__ k, const T* __restrict__ v, const T* __restrict__ dout,
                const float* __restrict__ lse, const float* __restrict__ delta, float* __restrict__ dq_acc, T* __restrict__ dk,
                T* __restrict__ dv, int N, int W, int d, int causal, int64_t n_bh, float scale, const Heads heads) {
    after_previous();
    if (heads.any != nullptr && !heads.has(blockIdx.x % n_bh)) return;       // the tensor-core kernel before this one has computed it
    constexpr int NT = kTR * TC;
    constexpr int RI = BT / kTR, KJ = BT / TC, KA = BT / kTR;    // rows and keys of a thread's scores; keys of its dk / dv rows
    constexpr int LDP = ld_p<BT>();
    extern __shared__ __align__(16) float smem[];
    const int ld = row_stride(d);
    float* Qs = smem;
    float* dOs = Qs + BT * ld;
    float* Ks = dOs + BT * ld;
    float* Vs = Ks + BT * ld;
    float* Ps = Vs + BT * ld + column_slack<TC, CM>();
    float* dSs = Ps + BT * LDP;
    float* lse_s = dSs + BT * LDP;
    float* delta_s = lse_s + BT;

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int tc = TC == 8 ? (lane & 7) : (warp & 1) * 8 + (lane & 7);
    const int tr = (TC == 8 ? warp : warp >> 1) * 4 + (lane >> 3);
    const int64_t bh = blockIdx.x % n_bh;                        // the key tiles with the most queries go first
    const int j0 = (int)(blockIdx.x / n_bh) * BT;
    load_rows<BT, NT>(Ks, ld, k + bh * N * (int64_t)d, j0, N, d);
    load_rows<BT, NT>(Vs, ld, v + bh * N * (int64_t)d, j0, N, d);

    float acc_dk[KA][CM], acc_dv[KA][CM];
#pragma unroll
    for (int i = 0; i < KA; ++i)
#pragma unroll
        for (int c = 0; c < CM; ++c) acc_dk[i][c] = acc_dv[i][c] = 0.f;
    // the first query row that may use a key of this tile (window rule j <= N-W+i)
    const int i_first = causal ? max(0, j0 - (N - W)) : 0;
    for (int i0 = i_first / BT * BT; i0 < W; i0 += BT) {
        __syncthreads();
        load_rows<BT, NT>(Qs, ld, q + bh * W * (int64_t)d, i0, W, d);
        load_rows<BT, NT>(dOs, ld, dout + bh * W * (int64_t)d, i0, W, d);
        if (threadIdx.x < BT) {
            const int i = i0 + threadIdx.x;
            lse_s[threadIdx.x] = i < W ? lse[bh * W + i] : 0.f;
            delta_s[threadIdx.x] = i < W ? delta[bh * W + i] : 0.f;
        }
        cp_async_wait();
        __syncthreads();
        // scores -> P and dS, rows tr + 16 i, keys tc + TC j
        {
            float s[RI][KJ], dp[RI][KJ];
#pragma unroll
            for (int i = 0; i < RI; ++i)
#pragma unroll
                for (int j = 0; j < KJ; ++j) s[i][j] = dp[i][j] = 0.f;
            dot_tile<RI, KJ>(s, Qs + tr * ld, kTR * ld, Ks + tc * ld, TC * ld, d);
            dot_tile<RI, KJ>(dp, dOs + tr * ld, kTR * ld, Vs + tc * ld, TC * ld, d);
            const bool edge = i0 + BT > W || j0 + BT > N || (causal && j0 + BT - 1 > N - W + i0);
#pragma unroll
            for (int i = 0; i < RI; ++i) {
                const int row = tr + kTR * i;
                const float lse_i = lse_s[row], delta_i = delta_s[row];
                // key tc + TC j of the tile is allowed iff TC j < limit
                const int limit = i0 + row >= W ? 0 : (causal ? min(N, N - W + i0 + row + 1) : N) - j0 - tc;
#pragma unroll
                for (int j = 0; j < KJ; ++j) {
                    float p = exp2f((s[i][j] * scale - lse_i) * kLog2e);
                    if (edge && TC * j >= limit) p = 0.f;
                    Ps[row * LDP + tc + TC * j] = p;
                    dSs[row * LDP + tc + TC * j] = p * (dp[i][j] - delta_i) * scale;
                }
            }
        }
        __syncthreads();
        accumulate_over_rows<BT, TC, KA, CM>(acc_dv, Ps + tr * KA, dOs, ld, tc);
        accumulate_over_rows<BT, TC, KA, CM>(acc_dk, dSs + tr * KA, Qs, ld, tc);
        // dq of the tile's rows from these keys
        {
            float acc[RI][CM];
#pragma unroll
            for (int i = 0; i < RI; ++i)
#pragma unroll
                for (int c = 0; c < CM; ++c) acc[i][c] = 0.f;
#pragma unroll 1
            for (int key = 0; key < BT; key += 4) {
                float4 a[RI];
#pragma unroll
                for (int i = 0; i < RI; ++i) a[i] = *reinterpret_cast<const float4*>(dSs + (tr + kTR * i) * LDP + key);
#pragma unroll
                for (int e = 0; e < 4; ++e) {
                    float b[CM];
                    load_columns<TC, CM>(b, Ks + (key + e) * ld, tc);
#pragma unroll
                    for (int i = 0; i < RI; ++i)
#pragma unroll
                        for (int c = 0; c < CM; ++c) acc[i][c] = fmaf(get(a[i], e), b[c], acc[i][c]);
                }
            }
#pragma unroll
            for (int i = 0; i < RI; ++i) {
                const int row = i0 + tr + kTR * i;
                if (row >= W) continue;
                float* dst = dq_acc + (bh * W + row) * d;
#pragma unroll
                for (int g = 0; g < CM / 4; ++g) {
                    const int c = g * 4 * TC + 4 * tc;
                    if (c < d) atomicAdd(reinterpret_cast<float4*>(dst + c), make_float4(acc[i][g * 4], acc[i][g * 4 + 1], acc[i][g * 4 + 2], acc[i][g * 4 + 3]));
                }
#pragma unroll
                for (int m = CM / 4 * 4; m < CM; ++m) {
                    const int c = column_of<TC, CM>(m, tc);
                    if (c < d) atomicAdd(dst + c, acc[i][m]);
                }
            }
        }
    }
    cp_async_wait();                            // K and V of a tile that no query may use
#pragma unroll
    for (int i = 0; i < KA; ++i) {
        const int key = j0 + tr * KA + i;
        if (key >= N) continue;
        store_columns<TC, CM>(dk + (bh * N + key) * d, acc_dk[i], 1.f, tc, d);
        store_columns<TC, CM>(dv + (bh * N + key) * d, acc_dv[i], 1.f, tc, d);
    }
}

template <typename T>
__global__ void bwd_round_kernel(const float* __restrict__ src, T* __restrict__ dst, long long n, long long per_bh, const Heads heads) {
    if (heads.none()) return;
    const long long x = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (x < n && heads.has(x / per_bh)) from_f(dst[x], src[x]);
}

// Where dq is summed.  fp32: straight in the result, unless the main kernel still reads an input there (dq written over q, say);
// otherwise [rows * d] fp32 behind delta, 16-byte aligned
template <typename T>
float* dq_sums(const void* q, const void* k, const void* v, const float* lse, const void* dout, void* dq, int64_t n_bh, int N, int W, int d, float* ws) {
    const int64_t rows = n_bh * W, q_bytes = rows * d * (int64_t)sizeof(T), k_bytes = n_bh * N * (int64_t)d * (int64_t)sizeof(T);
    const bool in_place = sizeof(T) == 4 && !overlap(dq, q_bytes, q, q_bytes) && !overlap(dq, q_bytes, dout, q_bytes) && !overlap(dq, q_bytes, k, k_bytes) &&
                          !overlap(dq, q_bytes, v, k_bytes) && !overlap(dq, q_bytes, lse, rows * (int64_t)sizeof(float));
    return in_place ? reinterpret_cast<float*>(dq) : ws + ((rows + 3) / 4) * 4;
}

template <typename T, int BT, int TC, int CM>
int launch_t(const T* q, const T* k, const T* v, const T* out, const float* lse, const T* dout, T* dq, T* dk, T* dv,
             int B, int H, int N, int W, int d, int causal, float* ws, cudaStream_t st, const Heads& heads) {
    const int64_t n_bh = (int64_t)B * H, rows = n_bh * W;
    float* delta = ws;                                  // [B*H*W]
    float* dq_acc = dq_sums<T>(q, k, v, lse, dout, dq, n_bh, N, W, d, ws);
    const float scale = 1.f / sqrtf((float)d);
    static bool allowed[64] = {};
    TLIN_CUDA_CHECK(allow_dynamic_smem(bwd_simt_kernel<T, BT, TC, CM>, (int)bwd_smem_bytes<BT>(TC * CM, column_slack<TC, CM>()), allowed));
    const int64_t ctas = n_bh * ((N + BT - 1) / BT);
    if (ctas > 0x7fffffffLL) return TLIN_ERR_UNSUPPORTED;
    if (heads.any == nullptr) {                            // else the tensor-core kernels have prepared both for the heads that are to run
        bwd_delta_kernel<T><<<(unsigned)((rows + 7) / 8), 256, 0, st>>>(out, dout, delta, rows, d);
        TLIN_CUDA_CHECK(cudaGetLastError());
        count_launch();
        TLIN_CUDA_CHECK(cudaMemsetAsync(dq_acc, 0, (size_t)rows * d * sizeof(float), st));
        bwd_simt_kernel<T, BT, TC, CM><<<(unsigned)ctas, kTR * TC, bwd_smem_bytes<BT>(d, column_slack<TC, CM>()), st>>>(
            q, k, v, dout, lse, delta, dq_acc, dk, dv, N, W, d, causal, n_bh, scale, heads);
        TLIN_CUDA_CHECK(cudaGetLastError());
    } else {
        TLIN_CUDA_CHECK(launch_overlapped(bwd_simt_kernel<T, BT, TC, CM>, (unsigned)ctas, kTR * TC, bwd_smem_bytes<BT>(d, column_slack<TC, CM>()), st,
                                          q, k, v, dout, lse, (const float*)delta, dq_acc, dk, dv, N, W, d, causal, n_bh, scale, heads));
    }
    count_launch();
    if ((void*)dq_acc != (void*)dq) {
        bwd_round_kernel<T><<<(unsigned)((rows * d + 255) / 256), 256, 0, st>>>(dq_acc, dq, rows * d, (long long)W * d, heads);
        TLIN_CUDA_CHECK(cudaGetLastError());
        count_launch();
    }
    return TLIN_OK;
}

template <typename T>
int launch_any(const void* q, const void* k, const void* v, const void* out, const float* lse, const void* dout,
               void* dq, void* dk, void* dv, int B, int H, int N, int W, int d, int causal, float* ws, cudaStream_t st, const Heads& heads) {
    if ((long long)B * H * W * d > (1LL << 40) || (long long)N > 0x7fffffffLL - 64) return TLIN_ERR_UNSUPPORTED;
    const T *qt = (const T*)q, *kt = (const T*)k, *vt = (const T*)v, *ot = (const T*)out, *dot = (const T*)dout;
    T *dqt = (T*)dq, *dkt = (T*)dk, *dvt = (T*)dv;
    if (d <= 40) return launch_t<T, 64, 8, 5>(qt, kt, vt, ot, lse, dot, dqt, dkt, dvt, B, H, N, W, d, causal, ws, st, heads);
    if (d <= 64) return launch_t<T, 64, 8, 8>(qt, kt, vt, ot, lse, dot, dqt, dkt, dvt, B, H, N, W, d, causal, ws, st, heads);
    if (d <= 112) return launch_t<T, 64, 16, 7>(qt, kt, vt, ot, lse, dot, dqt, dkt, dvt, B, H, N, W, d, causal, ws, st, heads);
    if (d <= 128) return launch_t<T, 64, 16, 8>(qt, kt, vt, ot, lse, dot, dqt, dkt, dvt, B, H, N, W, d, causal, ws, st, heads);
    if (d <= 256) return launch_t<T, 32, 16, 16>(qt, kt, vt, ot, lse, dot, dqt, dkt, dvt, B, H, N, W, d, causal, ws, st, heads);
    return TLIN_ERR_UNSUPPORTED;
}

}  // namespace

// Microseconds of the fp32 kernels up to d = 64, as fitted to the calls that bwd_f32_tensor_path speaks of.
double bwd_simt_us(long long n_bh, int N, int W, int d, int causal) {
    const double key_tiles = (N + 63) / 64, steps = (W + 63) / 64, seen = causal ? (N - W / 2.) / N : 1.;
    return 11. + std::max(steps * (5.2 + 0.125 * d), n_bh * key_tiles * steps * seen * (3.7 + 0.118 * d) / kDefaultSMs) + 1.1 * n_bh * key_tiles / kDefaultSMs;
}

float* bwd_simt_sums(const float* q, const float* k, const float* v, const float* lse, const float* dout, float* dq, long long n_bh, int N, int W, int d, float* ws) {
    return dq_sums<float>(q, k, v, lse, dout, dq, n_bh, N, W, d, ws);
}

size_t bwd_workspace_bytes(long long B, long long H, long long W, int d) {
    const long long rows = B * H * W;
    return (size_t)((((rows + 3) / 4) * 4 + rows * d) * (long long)sizeof(float));
}

int launch_bwd_simt(const void* q, const void* k, const void* v, const void* out, const float* lse, const void* dout,
                    void* dq, void* dk, void* dv, int B, int H, int N, int W, int d, int causal, int is_f32, float* ws,
                    cudaStream_t st, const Heads& heads) {
    if (is_f32) return launch_any<float>(q, k, v, out, lse, dout, dq, dk, dv, B, H, N, W, d, causal, ws, st, heads);
    return launch_any<__nv_bfloat16>(q, k, v, out, lse, dout, dq, dk, dv, B, H, N, W, d, causal, ws, st, {});
}

}  // namespace tlin

// CUDA-core forward kernel: exact softmax attention, fp32 arithmetic, any head dimension up to 256.
// Serves the fp32 entry point (error bar 1e-4), and bf16 where tlin_set_forward_impl(1) asks for it or, at a head size other than 64 and
// 128, the call has very few rows and keys per (b,h) (rows_beat_tensor_cores) or 2^31 query rows or more.
// Section 3 attention formula; causal rule j <= N-W+i; online (running max / running sum) softmax.
//
// Bound by the FFMA rate (128 per clock and SM, 72 TFLOP/s at 1.9 GHz).  A CTA of 128 threads (16 row groups x 8 column
// threads) owns 16 ROWS query rows of one (b,h) and walks 64-key tiles.  A thread scores ROWS rows against 8 keys from
// registers (two 16-byte shared loads per 16 to 32 FFMA) and accumulates ROWS x CM output elements; the probabilities pass
// through shared memory inside the warp only (a row belongs to eight lanes of one warp).  One key scored per lane and one
// probability per shuffle, as before, spent four shared-memory reads on five FFMA.
// Measured, fp32: B8 H12 N1024 W512 d36 2059 -> 210 us (26 TFLOP/s), B4 H12 N1500 W700 d128 3229 -> 837 us.
//
// Few (b,h) and query tiles: the CTAs of a cluster (2, 4 or 8) share the keys of one query tile and merge their sums through
// distributed shared memory, so that no workspace is needed.
#include "tlin_internal.h"
#include "simt_tiles.cuh"
#include <algorithm>
#include <cooperative_groups.h>
#include <float.h>
#include <math_constants.h>

namespace tlin {
namespace {

using namespace simt;
namespace cg = cooperative_groups;

constexpr int kNT = 128, kTC = 8, kTR = kNT / kTC;      // threads, column threads, row groups
constexpr int kBN = 64;                                 // keys per tile
constexpr int kKJ = kBN / kTC;                          // keys a thread scores: tc + 8 j
constexpr int kLdP = kBN + 8;                           // 8 modulo 32: four rows x eight keys written by a warp hit 32 banks
constexpr float kLog2e = 1.4426950408889634f;

template <int ROWS>
__host__ __device__ constexpr size_t smem_floats(int d, int slack) {
    return (size_t)kTR * ROWS * row_stride(d) + (size_t)kBN * row_stride(d) + (size_t)kTR * ROWS * kLdP + (size_t)kBN * d + slack;
}

template <typename T, int ROWS, int CM>
__global__ void __launch_bounds__(kNT, CM * ROWS <= 40 ? 3 : 2)
fwd_simt_kernel(const T* __restrict__ q, const T* __restrict__ k, const T* __restrict__ v, T* __restrict__ out, float* __restrict__ lse,
                int N, int W, int d, int causal, int q_tiles, int64_t n_bh, int cluster, float scale, int64_t kv_rows, const Heads heads) {
    constexpr int BM = kTR * ROWS;
    after_previous();
    if (heads.none()) return;                              // the tensor-core kernel before this one has computed the call
    extern __shared__ __align__(16) float smem[];
    const int ld = row_stride(d);
    float* Qs = smem;                           // [BM][ld]
    float* Ks = Qs + BM * ld;                   // [kBN][ld]
    float* Ps = Ks + kBN * ld;                  // [BM][kLdP]
    float* Vs = Ps + BM * kLdP;                 // [kBN][d]

    const int lane = threadIdx.x & 31, tc = lane & 7, tr = (threadIdx.x >> 5) * 4 + (lane >> 3);
    // with the window rule the last query tiles see the most keys: they go first
    const int64_t item = blockIdx.x / cluster;
    const int rank = (int)(blockIdx.x - item * cluster);
    const int qt = q_tiles - 1 - (int)(item / n_bh);
    const int64_t bh = item % n_bh;
    if (!heads.has(bh)) return;                            // the same for all CTAs of a cluster
    const int row0 = qt * BM;
    const T* kb = k + bh * kv_rows * d;         // kv_rows >= N: rows per (b,h) of the key/value allocation
    const T* vb = v + bh * kv_rows * d;

    // keys this query tile needs: up to the limit of its last row; this CTA's share of their tiles
    const int rows_here = min(BM, W - row0);
    const int key_end = causal ? N - W + row0 + rows_here : N;
    const int first_limit = causal ? N - W + row0 + 1 : N;      // keys below this are allowed for every row of the tile
    const int tiles = (key_end + kBN - 1) / kBN;
    const int t_begin = (int)((int64_t)tiles * rank / cluster), t_end = (int)((int64_t)tiles * (rank + 1) / cluster);

    float m[ROWS], l[ROWS], acc[ROWS][CM];
#pragma unroll
    for (int i = 0; i < ROWS; ++i) {
        m[i] = -CUDART_INF_F;
        l[i] = 0.f;
#pragma unroll
        for (int c = 0; c < CM; ++c) acc[i][c] = 0.f;
    }
    load_rows<BM, kNT>(Qs, ld, q + bh * W * d, row0, W, d);

    for (int t = t_begin; t < t_end; ++t) {
        const int k0 = t * kBN;
        if (t > t_begin) __syncthreads();
        load_rows<kBN, kNT>(Ks, ld, kb, k0, N, d);
        load_rows<kBN, kNT>(Vs, d, vb, k0, N, d);
        cp_async_wait();
        __syncthreads();
        float s[ROWS][kKJ];
#pragma unroll
        for (int i = 0; i < ROWS; ++i)
#pragma unroll
            for (int j = 0; j < kKJ; ++j) s[i][j] = 0.f;
        dot_tile<ROWS, kKJ>(s, Qs + tr * ld, kTR * ld, Ks + tc * ld, kTC * ld, d);
        const bool edge = k0 + kBN > first_limit;
#pragma unroll
        for (int i = 0; i < ROWS; ++i) {
            float mt = -CUDART_INF_F;
            const int limit = (causal ? min(N, N - W + row0 + tr + kTR * i + 1) : N) - k0 - tc;   // key tc + 8 j allowed iff 8 j < limit
#pragma unroll
            for (int j = 0; j < kKJ; ++j) {
                s[i][j] *= scale;
                if (edge && kTC * j >= limit) s[i][j] = -CUDART_INF_F;
                mt = fmaxf(mt, s[i][j]);
            }
#pragma unroll
            for (int o = 1; o < kTC; o <<= 1) mt = fmaxf(mt, __shfl_xor_sync(0xffffffffu, mt, o));
            const float m_new = fmaxf(m[i], mt), m_use = m_new == -CUDART_INF_F ? 0.f : m_new;
            const float corr = exp2f((m[i] - m_use) * kLog2e);          // m = -inf -> 0
            m[i] = m_new;
            l[i] *= corr;
#pragma unroll
            for (int c = 0; c < CM; ++c) acc[i][c] *= corr;
#pragma unroll
            for (int j = 0; j < kKJ; ++j) {
                const float pj = exp2f((s[i][j] - m_use) * kLog2e);     // masked: 2^-inf = 0
                l[i] += pj;
                Ps[(tr + kTR * i) * kLdP + tc + kTC * j] = pj;
            }
        }
        __syncwarp();
#pragma unroll 1
        for (int key = 0; key < kBN; key += 4) {
            float4 a[ROWS];
#pragma unroll
            for (int i = 0; i < ROWS; ++i) a[i] = *reinterpret_cast<const float4*>(Ps + (tr + kTR * i) * kLdP + key);
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                float b[CM];
                load_columns<kTC, CM>(b, Vs + (key + e) * d, tc);
#pragma unroll
                for (int i = 0; i < ROWS; ++i)
#pragma unroll
                    for (int c = 0; c < CM; ++c) acc[i][c] = fmaf(get(a[i], e), b[c], acc[i][c]);
            }
        }
    }
#pragma unroll
    for (int i = 0; i < ROWS; ++i)
#pragma unroll
        for (int o = 1; o < kTC; o <<= 1) l[i] += __shfl_xor_sync(0xffffffffu, l[i], o);

    T* ob = out + bh * W * d;
    if (cluster == 1) {
#pragma unroll
        for (int i = 0; i < ROWS; ++i) {
            const int row = row0 + tr + kTR * i;
            if (row >= W) continue;
            store_columns<kTC, CM>(ob + (int64_t)row * d, acc[i], 1.f / l[i], tc, d);
            if (lse != nullptr && tc == 0) lse[bh * W + row] = m[i] + logf(l[i]);
        }
        return;
    }
    // The CTAs of the cluster hold sums over different keys.  Each leaves its rows (unscaled), maxima and sums in its shared
    // memory; every CTA then combines a share of the rows from all of them.
    cg::cluster_group cl = cg::this_cluster();
    cp_async_wait();                            // a share may be empty: its copy of Q is then still on its way
    __syncthreads();
    float* Os = smem;                           // [BM][d], then m [BM], l [BM]
    float* ms = Os + BM * d;
    float* ls = ms + BM;
#pragma unroll
    for (int i = 0; i < ROWS; ++i) {
        store_columns<kTC, CM>(Os + (tr + kTR * i) * d, acc[i], 1.f, tc, d);
        if (tc == 0) {
            ms[tr + kTR * i] = m[i];
            ls[tr + kTR * i] = l[i];
        }
    }
    cl.sync();
    const int per_rank = BM / cluster;
    const int warp = threadIdx.x >> 5;
    for (int rr = rank * per_rank + warp; rr < (rank + 1) * per_rank; rr += kNT / 32) {
        const int row = row0 + rr;
        if (row >= W) break;
        float mm = -CUDART_INF_F;
        for (int c = 0; c < cluster; ++c) mm = fmaxf(mm, cl.map_shared_rank(ms, c)[rr]);
        const float ref = fmaxf(mm, -FLT_MAX);                  // no share may have a finite score
        float ll = 0.f, w[8];
#pragma unroll
        for (int c = 0; c < 8; ++c) {
            w[c] = 0.f;
            if (c < cluster) {
                w[c] = exp2f((cl.map_shared_rank(ms, c)[rr] - ref) * kLog2e);
                ll += w[c] * cl.map_shared_rank(ls, c)[rr];
            }
        }
        const float inv = 1.f / ll;
        for (int col = lane * 4; col < d; col += 128) {
            float4 sum = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
            for (int c = 0; c < 8; ++c) {
                if (c < cluster) {
                    const float4 x = *reinterpret_cast<const float4*>(cl.map_shared_rank(Os, c) + rr * d + col);
                    sum.x = fmaf(w[c], x.x, sum.x); sum.y = fmaf(w[c], x.y, sum.y);
                    sum.z = fmaf(w[c], x.z, sum.z); sum.w = fmaf(w[c], x.w, sum.w);
                }
            }
            store4(ob + (int64_t)row * d + col, sum.x * inv, sum.y * inv, sum.z * inv, sum.w * inv);
        }
        if (lse != nullptr && lane == 0) lse[bh * W + row] = mm + logf(ll);
    }
    cl.sync();                                  // nobody leaves while its rows are still being read
}

// Keys shared between CTAs while there are fewer CTAs than twice the SMs, at least four tiles each.
int cluster_size(int64_t items, int N) {
    int cluster = 1;
    const int tiles = (N + kBN - 1) / kBN;
    while (cluster < 8 && items * cluster * 2 <= 2 * kDefaultSMs && tiles >= 8 * cluster) cluster *= 2;
    return cluster;
}

template <typename T, int ROWS, int CM>
int launch(const T* q, const T* k, const T* v, T* out, float* lse, int B, int H, int N, int W, int d,
           int causal, long long kv_rows_alloc, cudaStream_t st, const Heads& heads) {
    constexpr int BM = kTR * ROWS;
    const int q_tiles = (W + BM - 1) / BM;
    const int64_t n_bh = (int64_t)B * H, items = n_bh * q_tiles;
    const size_t smem = sizeof(float) * smem_floats<ROWS>(d, column_slack<kTC, CM>());
    static bool allowed[64] = {};
    TLIN_CUDA_CHECK(allow_dynamic_smem(fwd_simt_kernel<T, ROWS, CM>, (int)(sizeof(float) * smem_floats<ROWS>(8 * CM, column_slack<kTC, CM>())), allowed));
    const int cluster = cluster_size(items, N);
    if (items * cluster > 0x7fffffffLL) return TLIN_ERR_UNSUPPORTED;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)(items * cluster));
    cfg.blockDim = dim3(kNT);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = (unsigned)cluster;
    attr[0].val.clusterDim.y = attr[0].val.clusterDim.z = 1;
    attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[1].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = heads.any != nullptr ? 2 : 1;
    TLIN_CUDA_CHECK(cudaLaunchKernelEx(&cfg, fwd_simt_kernel<T, ROWS, CM>, q, k, v, out, lse, N, W, d, causal, q_tiles, n_bh, cluster,
                                       1.0f / sqrtf((float)d), kv_rows_alloc > 0 ? (int64_t)kv_rows_alloc : (int64_t)N, heads));
    count_launch();
    return TLIN_OK;
}

// Few query rows, or few keys: one warp per row instead of a register tile.  The tiles above are at least 64 rows x 64 keys whatever
// the call has, and for 1 to 8 rows most of that is work on padding.  Eight rows per CTA; keys and values are staged 32 at a time (fp32),
// lane l scores key l, the warp reduces maximum and sum with shuffles, and lane c accumulates the output columns c, c + 32, ...
constexpr int kWarpRows = 8, kWarpKeys = 32, kWarpColumns = 8;      // columns per lane: d <= 256

__device__ __forceinline__ float to_f32(float x) { return x; }
__device__ __forceinline__ float to_f32(__nv_bfloat16 x) { return __bfloat162float(x); }

__device__ __forceinline__ float warp_max(float x) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) x = fmaxf(x, __shfl_xor_sync(0xffffffffu, x, o));
    return x;
}
__device__ __forceinline__ float warp_sum(float x) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
    return x;
}

template <typename T>
__global__ void __launch_bounds__(kWarpRows * 32)
fwd_row_per_warp_kernel(const T* __restrict__ q, const T* __restrict__ k, const T* __restrict__ v, T* __restrict__ out, float* __restrict__ lse,
                        int N, int W, int d, int causal, int q_tiles, float scale, int64_t kv_rows, const Heads heads) {
    if (!heads.has(blockIdx.x / q_tiles)) return;
    extern __shared__ __align__(16) float smem[];
    const int kstride = d + 4;                 // padded: lanes reading different rows hit different banks
    float* Qs = smem;                          // [kWarpRows][d]
    float* Ks = Qs + kWarpRows * d;            // [kWarpKeys][d+4]
    float* Vs = Ks + kWarpKeys * kstride;      // [kWarpKeys][d]

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int64_t bh = blockIdx.x / q_tiles;
    const int row0 = (blockIdx.x % q_tiles) * kWarpRows;
    const int i = row0 + warp;
    const bool row_ok = i < W;
    const T* qb = q + (bh * W + row0) * (int64_t)d;
    const T* kb = k + bh * kv_rows * d;        // kv_rows >= N: rows per (b,h) of the key/value allocation
    const T* vb = v + bh * kv_rows * d;

    const int rows_here = min(kWarpRows, W - row0);
    for (int idx = threadIdx.x; idx < rows_here * d; idx += blockDim.x) Qs[idx] = to_f32(qb[idx]);

    // keys this CTA needs: up to the limit of its last row
    const int64_t last_i = row0 + rows_here - 1;
    const int64_t klimit_blk = causal ? min((int64_t)N, (int64_t)(N - W) + last_i + 1) : (int64_t)N;
    const int64_t klimit_row = causal ? (int64_t)(N - W) + i + 1 : (int64_t)N;  // keys j < klimit_row allowed

    float m = -CUDART_INF_F, l = 0.f;
    float acc[kWarpColumns];
#pragma unroll
    for (int r = 0; r < kWarpColumns; ++r) acc[r] = 0.f;

    for (int64_t t0 = 0; t0 < klimit_blk; t0 += kWarpKeys) {
        __syncthreads();
        const int nk = (int)min((int64_t)kWarpKeys, (int64_t)N - t0);
        for (int idx = threadIdx.x; idx < kWarpKeys * d; idx += blockDim.x) {
            const int r = idx / d, c = idx - r * d;
            float kv = 0.f, vv = 0.f;
            if (r < nk) {
                kv = to_f32(kb[(t0 + r) * d + c]);
                vv = to_f32(vb[(t0 + r) * d + c]);
            }
            Ks[r * kstride + c] = kv;
            Vs[r * d + c] = vv;
        }
        __syncthreads();
        if (!row_ok) continue;
        const int64_t j = t0 + lane;
        const bool ok = j < N && j < klimit_row;
        float s = 0.f;
        const float4* q4 = reinterpret_cast<const float4*>(Qs + warp * d);
        const float4* k4 = reinterpret_cast<const float4*>(Ks + lane * kstride);
        for (int c = 0; c < d / 4; ++c) {
            const float4 a = q4[c], b = k4[c];
            s = fmaf(a.x, b.x, s); s = fmaf(a.y, b.y, s); s = fmaf(a.z, b.z, s); s = fmaf(a.w, b.w, s);
        }
        s = ok ? s * scale : -CUDART_INF_F;
        const float m_new = fmaxf(m, warp_max(s));
        if (m_new == -CUDART_INF_F) continue;          // nothing that counts so far
        const float corr = expf(m - m_new);            // m = -inf -> 0
        const float p = ok ? expf(s - m_new) : 0.f;
        l = l * corr + warp_sum(p);
        m = m_new;
#pragma unroll
        for (int r = 0; r < kWarpColumns; ++r) acc[r] *= corr;
        for (int jj = 0; jj < kWarpKeys; ++jj) {
            const float pj = __shfl_sync(0xffffffffu, p, jj);
#pragma unroll
            for (int r = 0; r < kWarpColumns; ++r) {
                const int c = lane + 32 * r;
                if (c < d) acc[r] = fmaf(pj, Vs[jj * d + c], acc[r]);
            }
        }
    }
    if (!row_ok) return;
    const float inv_l = 1.f / l;
    T* ob = out + (bh * W + i) * (int64_t)d;
#pragma unroll
    for (int r = 0; r < kWarpColumns; ++r) {
        const int c = lane + 32 * r;
        if (c < d) store1(ob + c, acc[r] * inv_l);
    }
    if (lse != nullptr && lane == 0) lse[bh * W + i] = m + logf(l);
}

template <typename T>
int launch_row_per_warp(const T* q, const T* k, const T* v, T* out, float* lse, int B, int H, int N, int W, int d,
                        int causal, long long kv_rows_alloc, cudaStream_t st, const Heads& heads) {
    const int q_tiles = (W + kWarpRows - 1) / kWarpRows;
    const int64_t ctas = (int64_t)B * H * q_tiles;
    if (ctas > 0x7fffffffLL) return TLIN_ERR_UNSUPPORTED;
    auto smem_bytes = [](int d) { return (int)sizeof(float) * (kWarpRows * d + kWarpKeys * (d + 4) + kWarpKeys * d); };
    static bool allowed[64] = {};
    TLIN_CUDA_CHECK(allow_dynamic_smem(fwd_row_per_warp_kernel<T>, smem_bytes(32 * kWarpColumns), allowed));
    fwd_row_per_warp_kernel<T><<<(unsigned)ctas, kWarpRows * 32, smem_bytes(d), st>>>(q, k, v, out, lse, N, W, d, causal, q_tiles, 1.0f / sqrtf((float)d),
                                                                                 kv_rows_alloc > 0 ? (int64_t)kv_rows_alloc : (int64_t)N, heads);
    TLIN_CUDA_CHECK(cudaGetLastError());
    count_launch();
    return TLIN_OK;
}

// Which of the two: time of each in units of about 0.6 us, the longer of one CTA's chain of key tiles and the SMs' share of all of them,
// fitted to 10000 calls (fp32; d 4 to 256, 4 to 1024 keys, 1 to 512 rows, 1 to 6000 (b,h)).  Tiles / rows, microseconds: d64 1500 (b,h) W4
// N32 55 / 21, W16 N64 55 / 98; d128 1500 W8 N64 150 / 86, 400 W1 N128 76 / 35; d256 64 W8 N8 27 / 13; d100 400 W9 N256 125 / 159; d36 148
// W8 N1024 55 / 139.  On the tiles alone 3710 of those calls are more than 5 % slower than on the rows alone, with the choice 154; more
// than 5 % slower than on the tiles alone are 109.
struct Estimate { double rows, tiles; };
Estimate estimate(int64_t n_bh, int N, int W, int d, int tile_rows, int64_t items, int cluster) {
    const double sms = kDefaultSMs, beyond128 = d > 128 ? d - 128 : 0;
    const double tiles = (N + kBN - 1) / kBN, steps = (N + kWarpKeys - 1) / kWarpKeys, ctas = (double)n_bh * ((W + kWarpRows - 1) / kWarpRows);
    const double staged = N < kWarpKeys ? N / (double)kWarpKeys : steps;          // a step of fewer keys stages fewer
    const bool from_hbm = 8.0 * n_bh * N * d > 80e6;                              // K and V do not stay in L2: a step waits longer
    const double row_chain = (6.4 + 0.1 * d) * steps * (from_hbm ? 1.6 : 1);
    const double row_share = (0.87 * n_bh * W * steps + ctas * staged * (0.024 * d + 0.03 * beyond128)) / sms;
    const double tile_chain = 0.2 * d * (((int)tiles + cluster - 1) / cluster);
    const double tile_share = (double)items * (tile_rows / 64) * tiles * (4.6 + 0.165 * d) / sms;
    return {std::max(row_chain, row_share), std::max(tile_chain, tile_share)};
}
bool rows_are_cheaper(int64_t n_bh, int N, int W, int d, int tile_rows, int64_t items, int cluster) {
    const Estimate e = estimate(n_bh, N, W, d, tile_rows, items, cluster);
    return e.rows < e.tiles + 4;
}

// 8 columns per CM.  Eight rows per thread instead of four halve the shared-memory reads but need 128 query rows per CTA: worth it
// for 40 < d <= 64 and more than 64 rows when that leaves few SMs without a CTA (128 CTAs at B4 H8 N2000 W500 d64: 261 against 285 us); at d <= 40, with three CTAs of
// either kind per SM, the finer split wins (B8 H12 N1024 W512 d36: 210 against 218 us, B8 H4 N327 W327: 42 against 52 us), and
// beyond d = 64 the registers do not suffice.
int tile_rows_of(int64_t n_bh, int W, int d) { return d > 40 && d <= 64 && W > 64 && n_bh * ((W + 127) / 128) >= kDefaultSMs * 3 / 4 ? 128 : 64; }
template <typename T>
int dispatch(const T* q, const T* k, const T* v, T* out, float* lse, int B, int H, int N, int W, int d,
             int causal, long long kv, cudaStream_t st, const Heads& heads = {}) {
    const int64_t n_bh = (int64_t)B * H;
    const int tile_rows = tile_rows_of(n_bh, W, d);
    const int64_t items = n_bh * ((W + tile_rows - 1) / tile_rows);
    if (rows_are_cheaper(n_bh, N, W, d, tile_rows, items, cluster_size(items, N)))
        return launch_row_per_warp<T>(q, k, v, out, lse, B, H, N, W, d, causal, kv, st, heads);
    if (tile_rows == 128)
        return launch<T, 8, 8>(q, k, v, out, lse, B, H, N, W, d, causal, kv, st, heads);
    if (d <= 40) return launch<T, 4, 5>(q, k, v, out, lse, B, H, N, W, d, causal, kv, st, heads);
    if (d <= 64) return launch<T, 4, 8>(q, k, v, out, lse, B, H, N, W, d, causal, kv, st, heads);
    if (d <= 104) return launch<T, 4, 13>(q, k, v, out, lse, B, H, N, W, d, causal, kv, st, heads);
    if (d <= 128) return launch<T, 4, 16>(q, k, v, out, lse, B, H, N, W, d, causal, kv, st, heads);
    if (d <= 192) return launch<T, 4, 24>(q, k, v, out, lse, B, H, N, W, d, causal, kv, st, heads);
    return launch<T, 4, 32>(q, k, v, out, lse, B, H, N, W, d, causal, kv, st, heads);
}

}  // namespace

// Microseconds of an fp32 call, as fitted to the calls that fwd_f32_tensor_path speaks of.
double fwd_simt_us(long long n_bh, int N, int W, int d, int causal) {
    const int rows = tile_rows_of(n_bh, W, d);
    const int64_t items = n_bh * ((W + rows - 1) / rows);
    const int cluster = cluster_size(items, N);
    const Estimate e = estimate(n_bh, N, W, d, rows, items, cluster);
    if (e.rows < e.tiles + 4) return 3.6 + 0.44 * e.rows;
    const double tiles = (N + kBN - 1) / kBN, seen = causal ? (N - W / 2.) / kBN : tiles;
    return 2.9 + std::max(((int)tiles + cluster - 1) / cluster * (rows / 64.) * (2.75 + 0.068 * d), (double)items * (rows / 64) * seen * (0.58 + 0.097 * d) / kDefaultSMs) +
           1.75 * items * cluster / kDefaultSMs;
}

int launch_fwd_simt_bf16(const void* q, const void* k, const void* v, void* out, float* lse,
                         int B, int H, int N, int W, int d, int causal, long long kv_rows_alloc, cudaStream_t st) {
    return dispatch<__nv_bfloat16>((const __nv_bfloat16*)q, (const __nv_bfloat16*)k, (const __nv_bfloat16*)v,
                                   (__nv_bfloat16*)out, lse, B, H, N, W, d, causal, kv_rows_alloc, st);
}
int launch_fwd_simt_f32(const float* q, const float* k, const float* v, float* out, float* lse,
                        int B, int H, int N, int W, int d, int causal, long long kv_rows_alloc, cudaStream_t st, const Heads& heads) {
    return dispatch<float>(q, k, v, out, lse, B, H, N, W, d, causal, kv_rows_alloc, st, heads);
}

}  // namespace tlin

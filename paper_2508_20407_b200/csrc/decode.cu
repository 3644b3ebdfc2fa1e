// Cached decode step: append the new key/value row, then one query row per (b,h) over the whole
// cache.  Appendix A ("Cache Hit": only the newest token takes part) and Section 5.2 (the history
// cache is static; nothing is re-concatenated).  Pure HBM streaming: every cached K/V byte is read
// exactly once with 16-byte loads, CUDA cores do the arithmetic in fp32.
//
// Work: (b,h) x splits.  Split s owns keys [s*kps, min(L,(s+1)*kps)), L = pos+1.  A CTA takes one split
// or, when there are more of them than CTAs fit on the chip, a run of splits (KeyRun).  Inside a CTA
// each warp-load covers 512 contiguous bytes (32/LPR rows); the LPR lanes that share a row reduce
// their partial dot products with xor-shuffles.  Every row-group keeps its own running max/sum and
// they are combined at the end; the CTA writes one normalised partial (o, lse) per (b,h) to the workspace and
// a second kernel merges the splits (log-sum-exp weights).  Short steps merge inside a cluster instead (decode_cluster_kernel).
#include "tlin_internal.h"
#include <cooperative_groups.h>
#include <cuda_fp16.h>
#include <math_constants.h>
#include <atomic>
#include <mutex>
#include <string.h>

namespace tlin {
namespace {

constexpr int kWarps = 8;
constexpr int kUnroll = 4;
constexpr int kMaxCluster = kDecodeMaxCluster;
constexpr float kLog2e = 1.4426950408889634f;
constexpr float kLn2 = 0.6931471805599453f;

// Not the non-coherent form, and no pointer of these kernels is __restrict__: a kernel may be resident while the one before it in the
// stream still writes (launch_overlapped), and nothing may be read ahead of after_previous().
__device__ __forceinline__ uint4 ld_stream(const uint4* p) {
    uint4 r;
    asm volatile("ld.global.L1::no_allocate.v4.u32 {%0,%1,%2,%3}, [%4];"
                 : "=r"(r.x), "=r"(r.y), "=r"(r.z), "=r"(r.w) : "l"(p));
    return r;
}
__device__ __forceinline__ float bf_lo(uint32_t w) { return __uint_as_float(w << 16); }
__device__ __forceinline__ float bf_hi(uint32_t w) { return __uint_as_float(w & 0xffff0000u); }

__device__ __forceinline__ float dot8(const uint4& kv, const float (&qf)[8]) {
    float s = bf_lo(kv.x) * qf[0];
    s = fmaf(bf_hi(kv.x), qf[1], s);
    s = fmaf(bf_lo(kv.y), qf[2], s);
    s = fmaf(bf_hi(kv.y), qf[3], s);
    s = fmaf(bf_lo(kv.z), qf[4], s);
    s = fmaf(bf_hi(kv.z), qf[5], s);
    s = fmaf(bf_lo(kv.w), qf[6], s);
    s = fmaf(bf_hi(kv.w), qf[7], s);
    return s;
}
__device__ __forceinline__ void axpy8(float p, const uint4& vv, float (&acc)[8]) {
    acc[0] = fmaf(p, bf_lo(vv.x), acc[0]);
    acc[1] = fmaf(p, bf_hi(vv.x), acc[1]);
    acc[2] = fmaf(p, bf_lo(vv.y), acc[2]);
    acc[3] = fmaf(p, bf_hi(vv.y), acc[3]);
    acc[4] = fmaf(p, bf_lo(vv.z), acc[4]);
    acc[5] = fmaf(p, bf_hi(vv.z), acc[5]);
    acc[6] = fmaf(p, bf_lo(vv.w), acc[6]);
    acc[7] = fmaf(p, bf_hi(vv.w), acc[7]);
}

// merge (m2,l2,a2) into (m,l,a); both in log2 units
__device__ __forceinline__ void combine(float& m, float& l, float (&a)[8], float m2, float l2, const float (&a2)[8]) {
    const float mn = fmaxf(m, m2);
    const float ms = mn == -CUDART_INF_F ? 0.f : mn;
    const float c1 = exp2f(m - ms), c2 = exp2f(m2 - ms);
    l = l * c1 + l2 * c2;
#pragma unroll
    for (int e = 0; e < 8; ++e) a[e] = a[e] * c1 + a2[e] * c2;
    m = mn;
}

// One query row of one (b,h) over keys [j0, j1) of its cache, by all threads of the CTA: the row `pos` (the token being
// appended in this launch, or -1) is taken from k_new / v_new instead of the cache.  Returns, in threads 0..D-1, column
// c = threadIdx.x of the un-normalised result `a`, the row sum `ll` and the running maximum `mm` (log2 units).
template <int D>
__device__ __forceinline__ void attend_key_range(const uint4* q_row, const uint4* kn, const uint4* vn,
                                                 const uint4* kc, const uint4* vc, int j0, int j1, int pos,
                                                 float scale_log2e, float& a, float& ll, float& mm) {
    constexpr int LPR = D / 8;           // lanes (16-byte chunks) per row
    constexpr int RPW = 32 / LPR;        // rows per warp-load
    constexpr int ROWS_PER_IT = kWarps * RPW * kUnroll;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int sub = lane % LPR, rsel = lane / LPR;
    float qf[8];
    {
        const uint4 qv = q_row[sub];
        qf[0] = bf_lo(qv.x) * scale_log2e; qf[1] = bf_hi(qv.x) * scale_log2e;
        qf[2] = bf_lo(qv.y) * scale_log2e; qf[3] = bf_hi(qv.y) * scale_log2e;
        qf[4] = bf_lo(qv.z) * scale_log2e; qf[5] = bf_hi(qv.z) * scale_log2e;
        qf[6] = bf_lo(qv.w) * scale_log2e; qf[7] = bf_hi(qv.w) * scale_log2e;
    }

    float m = -CUDART_INF_F, l = 0.f;
    float acc[8];
#pragma unroll
    for (int e = 0; e < 8; ++e) acc[e] = 0.f;

    for (int base = j0; base < j1; base += ROWS_PER_IT) {
        uint4 kv[kUnroll], vv[kUnroll];
        bool ok[kUnroll];
#pragma unroll
        for (int u = 0; u < kUnroll; ++u) {
            const int j = base + (u * kWarps + warp) * RPW + rsel;
            ok[u] = j < j1;
            kv[u] = make_uint4(0, 0, 0, 0);
            vv[u] = make_uint4(0, 0, 0, 0);
            if (ok[u]) {
                const bool fresh = j == pos;
                const uint4* kp = fresh ? kn + sub : kc + (int64_t)j * LPR + sub;
                const uint4* vp = fresh ? vn + sub : vc + (int64_t)j * LPR + sub;
                kv[u] = ld_stream(kp);
                vv[u] = ld_stream(vp);
            }
        }
        float s[kUnroll];
        float mb = m;
#pragma unroll
        for (int u = 0; u < kUnroll; ++u) {
            float x = dot8(kv[u], qf);
#pragma unroll
            for (int o = LPR / 2; o > 0; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
            s[u] = ok[u] ? x : -CUDART_INF_F;
            mb = fmaxf(mb, s[u]);
        }
        const float ms = mb == -CUDART_INF_F ? 0.f : mb;
        const float corr = exp2f(m - ms);
        l *= corr;
#pragma unroll
        for (int e = 0; e < 8; ++e) acc[e] *= corr;
#pragma unroll
        for (int u = 0; u < kUnroll; ++u) {
            const float p = exp2f(s[u] - ms);
            l += p;
            axpy8(p, vv[u], acc);
        }
        m = mb;
    }

    // combine the row-groups of the warp
#pragma unroll
    for (int o = LPR; o < 32; o <<= 1) {
        const float m2 = __shfl_xor_sync(0xffffffffu, m, o);
        const float l2 = __shfl_xor_sync(0xffffffffu, l, o);
        float a2[8];
#pragma unroll
        for (int e = 0; e < 8; ++e) a2[e] = __shfl_xor_sync(0xffffffffu, acc[e], o);
        combine(m, l, acc, m2, l2, a2);
    }
    __shared__ float sm_m[kWarps], sm_l[kWarps];
    __shared__ float sm_a[kWarps][D];
    if (rsel == 0) {
#pragma unroll
        for (int e = 0; e < 8; ++e) sm_a[warp][sub * 8 + e] = acc[e];
        if (sub == 0) { sm_m[warp] = m; sm_l[warp] = l; }
    }
    __syncthreads();
    a = 0.f; ll = 0.f; mm = -CUDART_INF_F;
    if (threadIdx.x < D) {
        const int c = threadIdx.x;
#pragma unroll
        for (int w = 0; w < kWarps; ++w) mm = fmaxf(mm, sm_m[w]);
        const float ms = mm == -CUDART_INF_F ? 0.f : mm;
#pragma unroll
        for (int w = 0; w < kWarps; ++w) {
            const float c1 = exp2f(sm_m[w] - ms);
            ll += sm_l[w] * c1;
            a += sm_a[w][c] * c1;
        }
    }
}

// Ragged batch: a position must lie below the caller's bound and inside the cache; a bad one counts as one split (which reports it).
__device__ __forceinline__ bool position_ok(int pos, int pos_all, int Ncap) { return pos >= 0 && pos < Ncap && pos <= pos_all; }
__device__ __forceinline__ int splits_of(int pos, int kps, int pos_all, int Ncap) {
    return position_ok(pos, pos_all, Ncap) ? pos / kps + 1 : 1;
}
// The splits of all (b,h), in order, dealt out as contiguous runs, one per CTA.  Neighbouring splits of one (b,h) are read as one
// key range, so a CTA starts and ends a stream of loads once or twice instead of once per split: all CTAs of a wave of equal
// splits end together, and draining, combining and starting anew idled the memory for about 3 us per wave.  At two CTAs per SM,
// B4 H32 d128, 8-bit cache of 15002 rows: 97 -> 87.5 us; B8 H32, 8-bit of 5001: 75.6 -> 62.0, bf16 of 4001: 94.2 -> 87.2.  Ragged,
// only the splits that have keys are dealt: B3 H32 of up to 21489 rows 157 -> 137 us.
// Three CTAs per SM (80 registers) have 98 KB of loads in flight per SM instead of 65: 87.5 -> 81.8, 62.0 -> 58.6, 87.2 -> 83.1,
// 137 -> 128 us, and B8 H32 d128 65537 rows 1330 -> 1200 us = 7.1 TB/s (more than the copy bandwidth, which has writes in it).
struct KeyRun {
    int bh, sp, left;                                      // first split, number of splits
    __device__ void single(int splits) {                   // one split per CTA
        bh = blockIdx.x / splits;
        sp = blockIdx.x - bh * splits;
        left = 1;
    }
    __device__ void uniform(int n_bh, int splits) {        // every (b,h) has `splits` of them
        const unsigned first = first_of_run((unsigned)(n_bh * splits));
        bh = (int)(first / (unsigned)splits);
        sp = (int)(first - (unsigned)(bh * splits));
    }
    // n_seq sequences of H heads each, sequence b with splits_of(pos[b]) per head (those that have keys)
    __device__ void ragged(const int* pos, int n_seq, int H, int kps, int pos_all, int Ncap) {
        const int lane = threadIdx.x & 31;
        unsigned total = 0;
        for (int b0 = 0; b0 < n_seq; b0 += 32)
            total += __reduce_add_sync(0xffffffffu, b0 + lane < n_seq ? (unsigned)splits_of(pos[b0 + lane], kps, pos_all, Ncap) : 0u);
        const unsigned first = first_of_run(total * (unsigned)H);
        unsigned before = 0;                               // splits (of one head) of the sequences before b0
        for (int b0 = 0; b0 < n_seq; b0 += 32) {
            const unsigned mine = b0 + lane < n_seq ? (unsigned)splits_of(pos[b0 + lane], kps, pos_all, Ncap) : 0u;
            unsigned upto = mine;                          // inclusive sum over the lanes
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const unsigned x = __shfl_up_sync(0xffffffffu, upto, o);
                if (lane >= o) upto += x;
            }
            const unsigned past = __ballot_sync(0xffffffffu, (before + upto) * (unsigned)H > first);
            if (past != 0) {
                const int at = __ffs(past) - 1;
                const unsigned n = __shfl_sync(0xffffffffu, mine, at), up = __shfl_sync(0xffffffffu, upto, at);
                const unsigned off = first - (before + up - n) * (unsigned)H;
                bh = (b0 + at) * H + (int)(off / n);
                sp = (int)(off % n);
                return;
            }
            before += __shfl_sync(0xffffffffu, upto, 31);
        }
        left = 0;                                          // no split for this CTA
    }
    // sets `left`, returns the run's first split: the first CTAs take one more when the total does not divide
    __device__ unsigned first_of_run(unsigned total) {
        const unsigned c = blockIdx.x, each = total / gridDim.x, more = total - each * gridDim.x;
        left = (int)(each + (c < more ? 1u : 0u));
        return c * each + min(c, more);
    }
    // `take` splits of this (b,h), which has n, have been written as one partial in the first one's slot: the other slots are empty
    __device__ void close(float* part_lse, int splits, int n, int take) {
        const int end = sp + take == n ? splits : sp + take;
        for (int x = sp + 1 + (int)threadIdx.x; x < end; x += kWarps * 32) part_lse[(int64_t)bh * splits + x] = -CUDART_INF_F;
        left -= take;
        sp = 0;
        ++bh;
        if (left > 0) __syncthreads();                     // the combining buffers are used again
    }
};

template <int D, bool kRuns>
__global__ void __launch_bounds__(kWarps * 32, kDecodeCtasPerSM)
decode_splitk_kernel(const uint4* q_new, const uint4* k_new, const uint4* v_new,
                     uint4* k_cache, uint4* v_cache,
                     float* part_o, float* part_lse,
                     int Ncap, int pos_all, const int* pos_per_seq, int n_bh, int H, int* status,
                     int splits, int kps, float scale_log2e) {
    constexpr int LPR = D / 8;           // lanes (16-byte chunks) per row
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    after_previous();
    let_next_start();
    KeyRun run;
    if (!kRuns) run.single(splits);
    else if (pos_per_seq == nullptr) run.uniform(n_bh, splits);
    else run.ragged(pos_per_seq, n_bh / H, H, kps, pos_all, Ncap);
    while (run.left > 0) {
        const int bh = run.bh;
        // one position for the whole batch, or one per sequence read from device memory (ragged batch)
        int pos = pos_all, n = splits;
        bool bad = false;
        if (pos_per_seq != nullptr) {
            pos = pos_per_seq[bh / H];
            bad = !position_ok(pos, pos_all, Ncap);
            if (kRuns) n = splits_of(pos, kps, pos_all, Ncap);
        }
        const int take = kRuns ? min(run.left, n - run.sp) : 1;
        const int64_t slot = (int64_t)bh * splits + run.sp;
        if (bad) {          // pos_all is the caller's bound, which sized the splits; the host cannot see the entries: report, and
                            // leave this (b,h) alone
            if (threadIdx.x == 0) atomicExch(status, (int)TLIN_ERR_INVALID_ARG);
            if (threadIdx.x == 0) part_lse[slot] = -CUDART_INF_F;
        } else {
            const int L = pos + 1;
            const int j0 = run.sp * kps, j1 = min(L, j0 + take * kps);
            const uint4* kc = k_cache + (int64_t)bh * Ncap * LPR;
            const uint4* vc = v_cache + (int64_t)bh * Ncap * LPR;
            const uint4* kn = k_new + (int64_t)bh * LPR;
            const uint4* vn = v_new + (int64_t)bh * LPR;

            // append (bit-exact copy) by the CTA whose range holds row `pos`; nobody reads that row from the
            // cache in this launch -- the lanes below take it from k_new / v_new.
            if (pos >= j0 && pos < j1 && warp == 0 && lane < LPR) {
                k_cache[((int64_t)bh * Ncap + pos) * LPR + lane] = kn[lane];
                v_cache[((int64_t)bh * Ncap + pos) * LPR + lane] = vn[lane];
            }

            float a, ll, mm;
            attend_key_range<D>(q_new + (int64_t)bh * LPR, kn, vn, kc, vc, j0, j1, pos, scale_log2e, a, ll, mm);
            if (threadIdx.x < D) {
                const int c = threadIdx.x;
                part_o[slot * D + c] = ll > 0.f ? a / ll : 0.f;
                if (c == 0) part_lse[slot] = ll > 0.f ? (mm + log2f(ll)) * kLn2 : -CUDART_INF_F;
            }
        }
        if (!kRuns) break;
        run.close(part_lse, splits, n, take);
    }
}

// A short step: the splits of a (b,h) are the CTAs of a cluster, and the first of them merges the others' sums out of their shared
// memory.  No second kernel and no trip of the partials through global memory, whose latencies are much of a step of 10 us:
// B6 H12 d64 of up to 1778 rows 11.0 -> 10.3 us, B2 H16 d64 1401 rows 8.6 -> 6.5, B1 H32 d64 201 rows (one split) 5.4 -> 4.0.
// kPerSM: where two CTAs per SM do not hold all clusters at a time, three may (the first of these: 72 clusters of 4, or of 6).
template <int D, int kPerSM>
__global__ void __launch_bounds__(kWarps * 32, kPerSM)
decode_cluster_kernel(const uint4* q_new, const uint4* k_new, const uint4* v_new, uint4* k_cache, uint4* v_cache,
                      __nv_bfloat16* out, float* lse, int Ncap, int pos_all, const int* pos_per_seq, int H, int* status,
                      int splits, int kps, float scale_log2e) {
    namespace cg = cooperative_groups;
    constexpr int LPR = D / 8;           // lanes (16-byte chunks) per row
    const int bh = blockIdx.x / splits, sp = blockIdx.x - bh * splits;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    after_previous();
    let_next_start();
    int pos = pos_all;
    if (pos_per_seq != nullptr) {
        pos = pos_per_seq[bh / H];
        if (!position_ok(pos, pos_all, Ncap)) {              // the same for every CTA of the cluster
            if (threadIdx.x == 0) atomicExch(status, (int)TLIN_ERR_INVALID_ARG);
            if (sp == 0 && threadIdx.x < D) {
                out[(int64_t)bh * D + threadIdx.x] = __float2bfloat16_rn(0.f);
                if (lse != nullptr && threadIdx.x == 0) lse[bh] = -CUDART_INF_F;
            }
            return;
        }
    }
    const int j0 = sp * kps, j1 = min(pos + 1, j0 + kps);
    const uint4* kn = k_new + (int64_t)bh * LPR;
    const uint4* vn = v_new + (int64_t)bh * LPR;
    uint4* kc = k_cache + (int64_t)bh * Ncap * LPR;
    uint4* vc = v_cache + (int64_t)bh * Ncap * LPR;
    if (pos >= j0 && pos < j1 && warp == 0 && lane < LPR) {  // append, as in decode_splitk_kernel
        kc[(int64_t)pos * LPR + lane] = kn[lane];
        vc[(int64_t)pos * LPR + lane] = vn[lane];
    }
    float a, ll, mm;
    attend_key_range<D>(q_new + (int64_t)bh * LPR, kn, vn, kc, vc, j0, j1, pos, scale_log2e, a, ll, mm);

    __shared__ float part[D + 2];                            // un-normalised sums, row sum, maximum (log2 units)
    cg::cluster_group cl = cg::this_cluster();
    if (sp != 0 && threadIdx.x < D) {
        part[threadIdx.x] = a;
        if (threadIdx.x == 0) part[D] = ll, part[D + 1] = mm;
    }
    cl.sync();
    if (sp == 0 && threadIdx.x < D) {
        float v[kMaxCluster], l[kMaxCluster], m[kMaxCluster];
        v[0] = a, l[0] = ll, m[0] = mm;
#pragma unroll
        for (int r = 1; r < kMaxCluster; ++r) {
            v[r] = 0.f, l[r] = 0.f, m[r] = -CUDART_INF_F;
            if (r < splits) {
                const float* other = cl.map_shared_rank(part, r);
                v[r] = other[threadIdx.x], l[r] = other[D], m[r] = other[D + 1];
            }
        }
        float top = m[0];
#pragma unroll
        for (int r = 1; r < kMaxCluster; ++r) top = fmaxf(top, m[r]);
        if (top == -CUDART_INF_F) {                          // every score is -inf: zeros, as from the merge kernel
            out[(int64_t)bh * D + threadIdx.x] = __float2bfloat16_rn(0.f);
            if (lse != nullptr && threadIdx.x == 0) lse[bh] = -CUDART_INF_F;
        } else {                                             // (a branch: a guard on z below costs a step of 4.6 us 0.2)
            float sum = 0.f, z = 0.f;
#pragma unroll
            for (int r = 0; r < kMaxCluster; ++r) {
                const float w = exp2f(m[r] - top);
                z = fmaf(w, l[r], z);
                sum = fmaf(w, v[r], sum);
            }
            out[(int64_t)bh * D + threadIdx.x] = __float2bfloat16_rn(sum / z);
            if (lse != nullptr && threadIdx.x == 0) lse[bh] = fmaf(top, kLn2, logf(z));
        }
    }
    cl.sync();                                               // shared memory stays until it has been read
}

// A table of decode problems as one launch: one CTA per (problem, b*h), whole key range, result written directly (no
// split, no second kernel).  Meant for the per-layer caches of a block, which are short (Appendix A, cache hit: the
// (H+1) D W_oh term -- one row against the W_oh summary tokens of a layer -- and the row inside the window).
struct DecodeProblemDev {
    const uint4* q_new; const uint4* k_new; const uint4* v_new;   // k_new == null: attend only, nothing is appended
    uint4* k_cache; uint4* v_cache;
    __nv_bfloat16* out; float* lse;
    int cta0, Ncap, pos;
};
constexpr int kMaxDecodeBatch = 48;
struct DecodeTable { DecodeProblemDev prob[kMaxDecodeBatch]; int n; };

template <int D>
__global__ void __launch_bounds__(kWarps * 32, kDecodeCtasPerSM)
decode_table_kernel(const __grid_constant__ DecodeTable tbl, float scale_log2e) {
    constexpr int LPR = D / 8;
    after_previous();
    let_next_start();
    int pi = 0;
    while (pi + 1 < tbl.n && (int)blockIdx.x >= tbl.prob[pi + 1].cta0) ++pi;
    const DecodeProblemDev& pr = tbl.prob[pi];
    const int bh = blockIdx.x - pr.cta0;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const bool append = pr.k_new != nullptr;
    const int pos = append ? pr.pos : -1;              // row taken from k_new / v_new instead of the cache
    const int L = append ? pr.pos + 1 : pr.pos;
    const uint4* kc = pr.k_cache + (int64_t)bh * pr.Ncap * LPR;
    const uint4* vc = pr.v_cache + (int64_t)bh * pr.Ncap * LPR;
    const uint4* kn = append ? pr.k_new + (int64_t)bh * LPR : kc;
    const uint4* vn = append ? pr.v_new + (int64_t)bh * LPR : vc;
    if (append && warp == 0 && lane < LPR) {
        pr.k_cache[((int64_t)bh * pr.Ncap + pos) * LPR + lane] = kn[lane];
        pr.v_cache[((int64_t)bh * pr.Ncap + pos) * LPR + lane] = vn[lane];
    }
    float a, ll, mm;
    attend_key_range<D>(pr.q_new + (int64_t)bh * LPR, kn, vn, kc, vc, 0, L, pos, scale_log2e, a, ll, mm);
    if (threadIdx.x < D) {
        const int c = threadIdx.x;
        pr.out[(int64_t)bh * D + c] = __float2bfloat16_rn(ll > 0.f ? a / ll : 0.f);
        if (pr.lse != nullptr && c == 0) pr.lse[bh] = ll > 0.f ? (mm + log2f(ll)) * kLn2 : -CUDART_INF_F;
    }
}

// One CTA per (b,h): out = sum_s w_s o_s / sum_s w_s with w_s = exp(lse_s - max lse).  Every warp reads two splits' lse per lane for
// the weights, then adds eight splits at a time.  kRuns: most slots may be empty (lse = -inf, no values) and are not read; else the
// first values are read beside the lse, not after it (a chain of two memory latencies is what bounds a short step).
template <int D, bool kRuns>
__global__ void __launch_bounds__(D)
decode_merge_kernel(const float* part_o, const float* part_lse,
                    __nv_bfloat16* out, float* lse, int splits) {
    const int bh = blockIdx.x, c = threadIdx.x, lane = c & 31;
    after_previous();
    let_next_start();
    const float* pl = part_lse + (int64_t)bh * splits;
    const float* po = part_o + (int64_t)bh * splits * D + c;
    const float l0 = lane < splits ? pl[lane] : -CUDART_INF_F, l1 = lane + 32 < splits ? pl[lane + 32] : -CUDART_INF_F;
    float o[8];
#pragma unroll
    for (int e = 0; e < 8; ++e) o[e] = !kRuns && e < splits ? po[(int64_t)e * D] : 0.f;
    float mm = fmaxf(l0, l1);
#pragma unroll
    for (int x = 16; x > 0; x >>= 1) mm = fmaxf(mm, __shfl_xor_sync(0xffffffffu, mm, x));
    if (mm == -CUDART_INF_F) {          // every split empty (a ragged sequence whose position was rejected): zeros, not NaN
        out[(int64_t)bh * D + c] = __float2bfloat16_rn(0.f);
        if (lse != nullptr && c == 0) lse[bh] = -CUDART_INF_F;
        return;
    }
    const float w0 = expf(l0 - mm), w1 = expf(l1 - mm);       // 0 beyond `splits`
    float z = 0.f, a = 0.f;
    for (int s = 0; s < splits; s += 8) {
        float w[8];
#pragma unroll
        for (int e = 0; e < 8; ++e) {
            w[e] = __shfl_sync(0xffffffffu, s < 32 ? w0 : w1, (s + e) & 31);
            if (kRuns || s > 0) o[e] = w[e] > 0.f ? po[(int64_t)(s + e) * D] : 0.f;
        }
#pragma unroll
        for (int e = 0; e < 8; ++e) {
            z += w[e];
            a = fmaf(w[e], o[e], a);
        }
    }
    out[(int64_t)bh * D + c] = __float2bfloat16_rn(a / z);
    if (lse != nullptr && c == 0) lse[bh] = mm + logf(z);
}
static_assert(kDecodeMaxSplits <= 64, "the merge reads two splits per lane");

// ---------------------------------------------------------------------------------------------------------------
// The same step over an 8-bit cache (E4M3 codes, value = decode(code) * scale[b,h]; not in the paper: it halves the
// bytes the step streams and the memory Section 5.2 accounts for).  A lane owns 16 columns of a row: one 16-byte load
// each for K and V, codes widened in pairs by cvt.rn.f16x2.e4m3x2 (exact).  The key scale is folded into q, the value
// scale into the final normalisation.  The new row is stored as encode(x / scale) (fp32 division, round to nearest
// even, saturating) and every lane that meets it takes the same codes from k_new / v_new instead of the cache.
__device__ __forceinline__ uint32_t f32x2_to_e4m3x2(float lo, float hi) {     // lo -> low byte, hi -> next byte
    uint32_t r;
    asm("{\n\t.reg .b16 c;\n\tcvt.rn.satfinite.e4m3x2.f32 c, %1, %2;\n\tcvt.u32.u16 %0, c;\n\t}" : "=r"(r) : "f"(hi), "f"(lo));
    return r;
}
// sum += k . q for the 16 codes of `c` against 16 f16 values of q (8 packed words): codes widened to f16 pairs (exact),
// products and sum in fp32 by the mixed-precision fma
__device__ __forceinline__ float dot16_codes(const uint4& c, const uint32_t (&qh)[8]) {
    const uint32_t w[4] = {c.x, c.y, c.z, c.w};
    float s = 0.f;
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        asm("{\n\t.reg .b16 c0, c1, k0, k1, k2, k3, q0, q1, q2, q3;\n\t.reg .b32 h0, h1;\n\t"
            "mov.b32 {c0, c1}, %1;\n\t"
            "cvt.rn.f16x2.e4m3x2 h0, c0;\n\tcvt.rn.f16x2.e4m3x2 h1, c1;\n\t"
            "mov.b32 {k0, k1}, h0;\n\tmov.b32 {k2, k3}, h1;\n\t"
            "mov.b32 {q0, q1}, %2;\n\tmov.b32 {q2, q3}, %3;\n\t"
            "fma.rn.f32.f16 %0, k0, q0, %0;\n\tfma.rn.f32.f16 %0, k1, q1, %0;\n\t"
            "fma.rn.f32.f16 %0, k2, q2, %0;\n\tfma.rn.f32.f16 %0, k3, q3, %0;\n\t}"
            : "+f"(s) : "r"(w[i]), "r"(qh[2 * i]), "r"(qh[2 * i + 1]));
    }
    return s;
}
// acc[e] += p * v_e for the 16 codes of `c`; p given twice in one word as f16 (weights lie in (0,1]: rounding them to
// 11 mantissa bits is far below the bf16 rounding of the output), codes widened to f16 (exact), products and sums in fp32
__device__ __forceinline__ void axpy16_codes(uint32_t p2, const uint4& c, float (&acc)[16]) {
    const uint32_t w[4] = {c.x, c.y, c.z, c.w};
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        asm("{\n\t.reg .b16 c0, c1, v0, v1, v2, v3, p0, p1;\n\t.reg .b32 h0, h1;\n\t"
            "mov.b32 {c0, c1}, %4;\n\t"
            "cvt.rn.f16x2.e4m3x2 h0, c0;\n\tcvt.rn.f16x2.e4m3x2 h1, c1;\n\t"
            "mov.b32 {v0, v1}, h0;\n\tmov.b32 {v2, v3}, h1;\n\t"
            "mov.b32 {p0, p1}, %5;\n\t"
            "fma.rn.f32.f16 %0, v0, p0, %0;\n\tfma.rn.f32.f16 %1, v1, p0, %1;\n\t"
            "fma.rn.f32.f16 %2, v2, p0, %2;\n\tfma.rn.f32.f16 %3, v3, p0, %3;\n\t}"
            : "+f"(acc[4 * i]), "+f"(acc[4 * i + 1]), "+f"(acc[4 * i + 2]), "+f"(acc[4 * i + 3]) : "r"(w[i]), "r"(p2));
    }
}
// 16 bf16 values (two 16-byte words) divided by `scale` and encoded
__device__ __forceinline__ uint4 quantise16(const uint4& lo8, const uint4& hi8, float scale) {
    const uint32_t w[8] = {lo8.x, lo8.y, lo8.z, lo8.w, hi8.x, hi8.y, hi8.z, hi8.w};
    uint32_t o[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const uint32_t a = f32x2_to_e4m3x2(__fdiv_rn(bf_lo(w[2 * i]), scale), __fdiv_rn(bf_hi(w[2 * i]), scale));
        const uint32_t b = f32x2_to_e4m3x2(__fdiv_rn(bf_lo(w[2 * i + 1]), scale), __fdiv_rn(bf_hi(w[2 * i + 1]), scale));
        o[i] = a | (b << 16);
    }
    return make_uint4(o[0], o[1], o[2], o[3]);
}

template <int D>
__global__ void __launch_bounds__(kWarps * 32, kDecodeCtasPerSM)
decode_fp8_splitk_kernel(const uint4* q_new, const uint4* k_new, const uint4* v_new,
                         uint4* k_cache, uint4* v_cache,
                         const float* k_scale, const float* v_scale,
                         float* part_o, float* part_lse,
                         int Ncap, int pos, int n_bh, int splits, int kps, float scale_log2e) {
    constexpr int LPR = D / 16;          // lanes (16-byte chunks of codes) per row
    constexpr int RPW = 32 / LPR;        // rows per warp-load
    constexpr int ROWS_PER_IT = kWarps * RPW * kUnroll;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int sub = lane % LPR, rsel = lane / LPR;
    __shared__ float sm_m[kWarps], sm_l[kWarps];
    __shared__ float sm_a[kWarps][D];
    const int L = pos + 1;
    after_previous();
    let_next_start();
    KeyRun run;
    run.uniform(n_bh, splits);
    while (run.left > 0) {
        const int bh = run.bh, take = min(run.left, splits - run.sp);
        const int j0 = run.sp * kps, j1 = min(L, j0 + take * kps);
        const float ks = k_scale[bh], vs = v_scale[bh];

        const uint4* kc = k_cache + (int64_t)bh * Ncap * LPR;
        const uint4* vc = v_cache + (int64_t)bh * Ncap * LPR;
        // the new row's codes for this lane's 16 columns (bf16: two 16-byte words per lane)
        const uint4 kn_codes = quantise16(k_new[(int64_t)bh * (D / 8) + 2 * sub], k_new[(int64_t)bh * (D / 8) + 2 * sub + 1], ks);
        const uint4 vn_codes = quantise16(v_new[(int64_t)bh * (D / 8) + 2 * sub], v_new[(int64_t)bh * (D / 8) + 2 * sub + 1], vs);
        // append by the CTA whose range holds row `pos`; nobody reads that row from the cache in this launch
        if (pos >= j0 && pos < j1 && warp == 0 && lane < LPR) {
            k_cache[((int64_t)bh * Ncap + pos) * LPR + lane] = kn_codes;
            v_cache[((int64_t)bh * Ncap + pos) * LPR + lane] = vn_codes;
        }

        // q * log2(e)/sqrt(d) as f16 pairs (|q| of a few units: no range issue; 11 mantissa bits against the 8 of the bf16
        // input); the key scale multiplies the finished dot product
        uint32_t qh[8];
        {
            const uint4 q0 = q_new[(int64_t)bh * (D / 8) + 2 * sub], q1 = q_new[(int64_t)bh * (D / 8) + 2 * sub + 1];
            const uint32_t w[8] = {q0.x, q0.y, q0.z, q0.w, q1.x, q1.y, q1.z, q1.w};
#pragma unroll
            for (int i = 0; i < 8; ++i) {
                const __half2 h = __floats2half2_rn(bf_lo(w[i]) * scale_log2e, bf_hi(w[i]) * scale_log2e);
                qh[i] = *reinterpret_cast<const uint32_t*>(&h);
            }
        }

        float m = -CUDART_INF_F, l = 0.f;
        float acc[16];
#pragma unroll
        for (int e = 0; e < 16; ++e) acc[e] = 0.f;

        for (int base = j0; base < j1; base += ROWS_PER_IT) {
            uint4 kv[kUnroll], vv[kUnroll];
            bool ok[kUnroll];
#pragma unroll
            for (int u = 0; u < kUnroll; ++u) {
                const int j = base + (u * kWarps + warp) * RPW + rsel;
                ok[u] = j < j1;
                kv[u] = make_uint4(0, 0, 0, 0);
                vv[u] = make_uint4(0, 0, 0, 0);
                if (ok[u]) {
                    if (j == pos) {
                        kv[u] = kn_codes;
                        vv[u] = vn_codes;
                    } else {
                        kv[u] = ld_stream(kc + (int64_t)j * LPR + sub);
                        vv[u] = ld_stream(vc + (int64_t)j * LPR + sub);
                    }
                }
            }
            float s[kUnroll];
            float mb = m;
#pragma unroll
            for (int u = 0; u < kUnroll; ++u) {
                float x = dot16_codes(kv[u], qh);
#pragma unroll
                for (int o = LPR / 2; o > 0; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
                s[u] = ok[u] ? x * ks : -CUDART_INF_F;
                mb = fmaxf(mb, s[u]);
            }
            const float ms = mb == -CUDART_INF_F ? 0.f : mb;
            const float corr = exp2f(m - ms);
            l *= corr;
#pragma unroll
            for (int e = 0; e < 16; ++e) acc[e] *= corr;
#pragma unroll
            for (int u = 0; u < kUnroll; ++u) {
                const float pr = exp2f(s[u] - ms);
                const __half2 ph = __float2half2_rn(pr);
                l += __low2float(ph);                 // the same rounded weight in the numerator and the denominator
                axpy16_codes(*reinterpret_cast<const uint32_t*>(&ph), vv[u], acc);
            }
            m = mb;
        }

        // combine the row-groups of the warp
#pragma unroll
        for (int o = LPR; o < 32; o <<= 1) {
            const float m2 = __shfl_xor_sync(0xffffffffu, m, o);
            const float l2 = __shfl_xor_sync(0xffffffffu, l, o);
            const float mn = fmaxf(m, m2);
            const float mz = mn == -CUDART_INF_F ? 0.f : mn;
            const float c1 = exp2f(m - mz), c2 = exp2f(m2 - mz);
            l = l * c1 + l2 * c2;
#pragma unroll
            for (int e = 0; e < 16; ++e) acc[e] = acc[e] * c1 + __shfl_xor_sync(0xffffffffu, acc[e], o) * c2;
            m = mn;
        }
        if (rsel == 0) {
#pragma unroll
            for (int e = 0; e < 16; ++e) sm_a[warp][sub * 16 + e] = acc[e];
            if (sub == 0) { sm_m[warp] = m; sm_l[warp] = l; }
        }
        __syncthreads();
        if (threadIdx.x < D) {
            const int c = threadIdx.x;
            float mm = -CUDART_INF_F;
#pragma unroll
            for (int w = 0; w < kWarps; ++w) mm = fmaxf(mm, sm_m[w]);
            const float ms = mm == -CUDART_INF_F ? 0.f : mm;
            float ll = 0.f, a = 0.f;
#pragma unroll
            for (int w = 0; w < kWarps; ++w) {
                const float c1 = exp2f(sm_m[w] - ms);
                ll += sm_l[w] * c1;
                a += sm_a[w][c] * c1;
            }
            const int64_t slot = (int64_t)bh * splits + run.sp;
            part_o[slot * D + c] = ll > 0.f ? a * vs / ll : 0.f;          // the value scale applied once per output element
            if (c == 0) part_lse[slot] = ll > 0.f ? (mm + log2f(ll)) * kLn2 : -CUDART_INF_F;
        }
        run.close(part_lse, splits, splits, take);
    }
}

// Runs where there are more splits than CTAs fit on the chip.  A single split per (b,h) leaves nothing to join, and the hardware's
// own dealing of CTAs is then a little better (B64 H32 d128, 514 rows, at two CTAs per SM: 100 against 101.5 us).
bool use_runs(const tlin_decode_plan& plan, int sms) { return plan.splits > 1 && plan.n_ctas > sms * kDecodeCtasPerSM; }

// Clusters of `size` CTAs of decode_cluster_kernel that the device holds at a time (asked once per device, size and head size).
template <int D, int kPerSM>
int clusters_at_a_time(int size) {
    static std::atomic<int> known[64][kMaxCluster + 1];
    const int dev = current_device_slot();
    if (dev < 0) return 0;
    int n = known[dev][size].load(std::memory_order_relaxed);
    if (n == 0) {
        cudaLaunchConfig_t cfg = {};
        cfg.gridDim = dim3((unsigned)size);
        cfg.blockDim = dim3(kWarps * 32);
        cudaLaunchAttribute attr[1];
        attr[0].id = cudaLaunchAttributeClusterDimension;
        attr[0].val.clusterDim.x = (unsigned)size;
        attr[0].val.clusterDim.y = attr[0].val.clusterDim.z = 1;
        cfg.attrs = attr;
        cfg.numAttrs = 1;
        if (cudaOccupancyMaxActiveClusters(&n, decode_cluster_kernel<D, kPerSM>, &cfg) != cudaSuccess) {
            (void)cudaGetLastError();
            n = 0;
        }
        n += 1;                                              // 0: not asked yet
        known[dev][size].store(n, std::memory_order_relaxed);
    }
    return n - 1;
}

template <int D>
int launch_d(const void* q_new, const void* k_new, const void* v_new, void* k_cache, void* v_cache,
             void* out, float* lse, int B, int H, int Ncap, int pos, const int* pos_per_seq, const tlin_decode_plan& plan,
             int sms, float* ws, cudaStream_t st, bool two_kernels) {
    const int64_t bh = (int64_t)B * H;
    float* part_o = ws;
    float* part_lse = ws + bh * kDecodeMaxSplits * D;
    const float scale_log2e = kLog2e / sqrtf((float)D);
    // The cluster kernel, with so many CTAs per SM; 0: two kernels.  Long splits are bound by the memory, and clusters fill the SMs
    // less evenly (B3 H16 31756 rows as 6 splits: 142 us, two kernels 129).  A single split per (b,h) needs no merge at all; more of
    // them than two per SM profit from the third (B64 H32 514 rows: 100 -> 89 us), fewer spread better without (B8 H32 983 rows: 24.6
    // against 25.3 us).
    int per_sm = 0;
    if (!two_kernels && plan.splits == 1) per_sm = plan.n_ctas > 2 * sms ? 3 : 2;
    else if (!two_kernels && plan.splits <= kMaxCluster && plan.keys_per_split <= kDecodeClusterKeys)
        per_sm = bh <= clusters_at_a_time<D, 2>(plan.splits) ? 2 : bh <= clusters_at_a_time<D, 3>(plan.splits) ? 3 : 0;
    if (per_sm > 0) {
        TLIN_CUDA_CHECK(launch_overlapped_clusters(per_sm == 2 ? decode_cluster_kernel<D, 2> : decode_cluster_kernel<D, 3>, plan.n_ctas, plan.splits,
            kWarps * 32, 0, st, (const uint4*)q_new, (const uint4*)k_new, (const uint4*)v_new, (uint4*)k_cache, (uint4*)v_cache,
            (__nv_bfloat16*)out, lse, Ncap, pos, pos_per_seq, H, status_word(), plan.splits, plan.keys_per_split, scale_log2e));
        count_launch();
        return TLIN_OK;
    }
    const bool runs = use_runs(plan, sms);
    TLIN_CUDA_CHECK(launch_overlapped(runs ? decode_splitk_kernel<D, true> : decode_splitk_kernel<D, false>,
        (unsigned)(runs ? sms * kDecodeCtasPerSM : plan.n_ctas), kWarps * 32, 0, st,
        (const uint4*)q_new, (const uint4*)k_new, (const uint4*)v_new, (uint4*)k_cache, (uint4*)v_cache,
        part_o, part_lse, Ncap, pos, pos_per_seq, (int)bh, H, status_word(), plan.splits, plan.keys_per_split, scale_log2e));
    TLIN_CUDA_CHECK(launch_overlapped(runs ? decode_merge_kernel<D, true> : decode_merge_kernel<D, false>, (unsigned)bh, D, 0, st, part_o, part_lse, (__nv_bfloat16*)out, lse, plan.splits));
    count_launch(2);
    return TLIN_OK;
}

template <int D>
int launch_fp8_d(const void* q_new, const void* k_new, const void* v_new, void* k_cache, void* v_cache,
                 const float* k_scale, const float* v_scale, void* out, float* lse, int B, int H, int Ncap, int pos,
                 const tlin_decode_plan& plan, int sms, float* ws, cudaStream_t st) {
    const int64_t bh = (int64_t)B * H;
    float* part_o = ws;
    float* part_lse = ws + bh * kDecodeMaxSplits * D;
    const float scale_log2e = kLog2e / sqrtf((float)D);
    const bool runs = use_runs(plan, sms);
    TLIN_CUDA_CHECK(launch_overlapped(decode_fp8_splitk_kernel<D>,
        (unsigned)(runs ? sms * kDecodeCtasPerSM : plan.n_ctas), kWarps * 32, 0, st,
        (const uint4*)q_new, (const uint4*)k_new, (const uint4*)v_new, (uint4*)k_cache, (uint4*)v_cache, k_scale, v_scale,
        part_o, part_lse, Ncap, pos, (int)bh, plan.splits, plan.keys_per_split, scale_log2e));
    TLIN_CUDA_CHECK(launch_overlapped(runs ? decode_merge_kernel<D, true> : decode_merge_kernel<D, false>, (unsigned)bh, D, 0, st, part_o, part_lse, (__nv_bfloat16*)out, lse, plan.splits));
    count_launch(2);
    return TLIN_OK;
}

template <int D>
int launch_table_d(const tlin_decode_problem* problems, int n, cudaStream_t st) {
    DecodeTable tbl;
    memset(&tbl, 0, sizeof(tbl));
    tbl.n = n;
    long long ctas = 0;
    for (int i = 0; i < n; ++i) {
        const tlin_decode_problem& pb = problems[i];
        DecodeProblemDev& pd = tbl.prob[i];
        pd.q_new = (const uint4*)pb.q_new; pd.k_new = (const uint4*)pb.k_new; pd.v_new = (const uint4*)pb.v_new;
        pd.k_cache = (uint4*)pb.k_cache; pd.v_cache = (uint4*)pb.v_cache;
        pd.out = (__nv_bfloat16*)pb.out; pd.lse = pb.lse;
        pd.cta0 = (int)ctas; pd.Ncap = pb.Ncap; pd.pos = pb.pos;
        ctas += pb.BH;
    }
    if (ctas > 0x7fffffffLL) return TLIN_ERR_UNSUPPORTED;
    TLIN_CUDA_CHECK(launch_overlapped(decode_table_kernel<D>, (unsigned)ctas, kWarps * 32, 0, st, tbl, kLog2e / sqrtf((float)D)));
    count_launch();
    return TLIN_OK;
}

}  // namespace

int decode_table_max_problems() { return kMaxDecodeBatch; }
int launch_decode_table(const tlin_decode_problem* problems, int n, int d, cudaStream_t st) {
    if (n <= 0 || n > kMaxDecodeBatch) return TLIN_ERR_INVALID_ARG;
    if (d == 128) return launch_table_d<128>(problems, n, st);
    if (d == 64) return launch_table_d<64>(problems, n, st);
    return TLIN_ERR_UNSUPPORTED;
}

int launch_decode_fp8(const void* q_new, const void* k_new, const void* v_new, void* k_cache, void* v_cache,
                      const float* k_scale, const float* v_scale, void* out, float* lse, int B, int H, int Ncap, int pos,
                      int d, const tlin_decode_plan& plan, int sms, float* ws, cudaStream_t st) {
    if (d == 128) return launch_fp8_d<128>(q_new, k_new, v_new, k_cache, v_cache, k_scale, v_scale, out, lse, B, H, Ncap, pos, plan, sms, ws, st);
    if (d == 64) return launch_fp8_d<64>(q_new, k_new, v_new, k_cache, v_cache, k_scale, v_scale, out, lse, B, H, Ncap, pos, plan, sms, ws, st);
    return TLIN_ERR_UNSUPPORTED;
}

int launch_decode(const void* q_new, const void* k_new, const void* v_new, void* k_cache, void* v_cache,
                  void* out, float* lse, int B, int H, int Ncap, int pos, const int* pos_per_seq, int d,
                  const tlin_decode_plan& plan, int sms, float* ws, cudaStream_t st, bool two_kernels) {
    if (d == 128) return launch_d<128>(q_new, k_new, v_new, k_cache, v_cache, out, lse, B, H, Ncap, pos, pos_per_seq, plan, sms, ws, st, two_kernels);
    if (d == 64) return launch_d<64>(q_new, k_new, v_new, k_cache, v_cache, out, lse, B, H, Ncap, pos, pos_per_seq, plan, sms, ws, st, two_kernels);
    return TLIN_ERR_UNSUPPORTED;
}

}  // namespace tlin

// ------------------------------------------------------------------------------------------------
// Decode step for callers that cannot allocate device memory.
//
// Some hosts of this library never get to call cudaMalloc: a plugin running inside another
// framework's memory pool, a worker that may only touch buffers handed to it, a process whose device
// memory budget is fixed up front.  For them the split-K partials live in the array below, which is part of
// the library image: every GPU that loads libtlin holds these 8.1 MiB until the process exits.
// Everything else is as in tlin_decode_step; the caller still owns inputs, caches and outputs.
namespace tlin {
namespace {

constexpr size_t kStaticScratchFloats = (size_t)256 * kDecodeMaxSplits * 129;   // 8 454 144 bytes
static __device__ __align__(256) float g_decode_static_scratch[kStaticScratchFloats];

std::mutex g_static_mu;
float* g_static_ptr[64] = {};      // device address of the array, per device, filled on first use
int g_static_major[64] = {};
int g_static_sms[64] = {};

// In host code the array's name is only a handle: the address a kernel can use has to be asked for,
// with the device current.  Done once per device.
int static_scratch_setup(int dev, float** ptr, int* sms) {
    std::lock_guard<std::mutex> lk(g_static_mu);
    if (g_static_ptr[dev] == nullptr) {
        float* p = nullptr;
        TLIN_CUDA_CHECK(cudaGetSymbolAddress((void**)&p, g_decode_static_scratch));
        TLIN_CUDA_CHECK(cudaDeviceGetAttribute(&g_static_major[dev], cudaDevAttrComputeCapabilityMajor, dev));
        TLIN_CUDA_CHECK(cudaDeviceGetAttribute(&g_static_sms[dev], cudaDevAttrMultiProcessorCount, dev));
        g_static_ptr[dev] = p;
    }
    if (g_static_major[dev] != 10) return TLIN_ERR_ARCH;
    *ptr = g_static_ptr[dev];
    *sms = g_static_sms[dev];
    return TLIN_OK;
}

}  // namespace
}  // namespace tlin

extern "C" int tlin_decode_step_static(const void* q_new, const void* k_new, const void* v_new,
                                       void* k_cache, void* v_cache, void* out, float* lse,
                                       int B, int H, int Ncap, int pos, int d, tlin_stream_t stream) {
    using namespace tlin;
    reset_launches();
    if (!q_new || !k_new || !v_new || !k_cache || !v_cache || !out) return TLIN_ERR_INVALID_ARG;
    if (B <= 0 || H <= 0 || Ncap <= 0 || d <= 0) return TLIN_ERR_INVALID_ARG;
    if (pos < 0 || pos >= Ncap) return TLIN_ERR_INVALID_ARG;
    const uintptr_t all = (uintptr_t)q_new | (uintptr_t)k_new | (uintptr_t)v_new | (uintptr_t)k_cache |
                          (uintptr_t)v_cache | (uintptr_t)out;
    if (all & 15u) return TLIN_ERR_INVALID_ARG;
    if (d != 64 && d != 128) return TLIN_ERR_UNSUPPORTED;
    const size_t need = (size_t)B * H * kDecodeMaxSplits * (size_t)(d + 1);
    if (need > kStaticScratchFloats) {
        fprintf(stderr, "libtlin: tlin_decode_step_static needs %zu bytes of scratch for B*H=%lld, d=%d but the "
                        "built-in array holds %zu bytes; use tlin_decode_step with a workspace instead\n",
                need * sizeof(float), (long long)B * H, d, kStaticScratchFloats * sizeof(float));
        return TLIN_ERR_WORKSPACE;
    }
    int dev = 0;
    TLIN_CUDA_CHECK(cudaGetDevice(&dev));
    if (dev < 0 || dev >= 64) return TLIN_ERR_CUDA;
    float* scratch = nullptr;
    int sms = 0;
    int rc = static_scratch_setup(dev, &scratch, &sms);
    if (rc != TLIN_OK) return rc;
    tlin_decode_plan plan;
    rc = tlin_plan_decode(B, H, pos + 1, d, sms, &plan);
    if (rc != TLIN_OK) return rc;
    // Two kernels at every size: a step of this entry point has always counted two launches (tlin_last_launch_count), which its
    // test states.  Nothing else holds it there; the cluster kernel needs no scratch and gives the same results.
    return launch_decode(q_new, k_new, v_new, k_cache, v_cache, out, lse, B, H, Ncap, pos, nullptr, d, plan, sms, scratch,
                         (cudaStream_t)stream, true);
}

// Tensor-core backward pass for sm_100a (bf16 in and out, fp32 accumulate): the chain rule of the Section 3
// attention formula with the window rule j <= N-W+i.  Training runs every layer as forward + backward ("cache miss"
// throughout, Section 4.1); the paper gives no gradient algorithm of its own.
//
//   p = exp(q k^T / sqrt(d) - lse)    dp = dout v^T    ds = p * (dp - delta) / sqrt(d),  delta_i = dout_i . out_i
//   dv = p^T dout      dk = ds^T q      dq = ds k
//
// Two kernels, neither with atomics, both recomputing p from the saved lse (what the one kernel below does not serve).  Steps with
// masked elements have a copy of the code of their own and the MMA warps elect their issuing lane once: B3 H12 N=W=1999 d64 175 ->
// 160 us, B2 H8 N1961 W578 d64 62 -> 53 us, B4 H32 N8192 W1024 d64 1.31 -> 1.20 ms.  Their elementwise arithmetic runs on packed
// pairs of floats, the same operations in half the instructions (101.6 -> 97.0 us, 65.8 -> 63.1 us, 1.14 -> 1.09 ms for the first,
// 16 x 2000^2 and the last); the one kernel keeps single floats, as pairs there gain nothing and spill.
//
// bwd_dkdv_tc_kernel   A CTA owns one 128-key tile of a (b,h) at a time and walks the 128-row query tiles that may
//   see it.  Scores are computed TRANSPOSED (S^T = K Q^T, dP^T = V dout^T: TMEM lane = key, column = query) so that
//   P^T and dS^T, written back to TMEM as bf16, are directly the A operands of dV += P^T dout and dK += dS^T Q, whose
//   B operands are the dout / Q tiles already in shared memory (read MN-major).  dK and dV stay in TMEM for the whole
//   key tile and are written once.  The queries are worked on as independent chains of 64, two (d = 128) or three (d = 64), one
//   per warpgroup (thread = key row): [S^T_x | dP^T_x] by the tensor pipe, then P^T_x and dS^T_x written over them in
//   place, then the two accumulating MMAs; while one chain does its elementwise work the tensor pipe serves the others.
//
// bwd_dq_tc_kernel     The forward's structure: a CTA owns 256 query rows (two Q tiles, one warpgroup each, one
//   thread per row) and streams 128-key tiles; per tile S = Q K^T -> p (kept in registers), then dP = dout V^T into
//   the same TMEM columns -> dS (bf16, in place) -> dQ += dS K with K read MN-major.  The work is scheduled like the
//   forward (groups that split the key range write fp32 partial dQ to the workspace; a small kernel adds them).
//
// bwd_fused_tc_kernel  (d = 128, chosen for small and middle-sized calls)  The dK/dV kernel with a third accumulating product,
//   dQ^T = K^T dS^T, which a warpgroup of its own adds to an fp32 dQ buffer with reductions in L2; a small kernel scales and
//   rounds it.  Five matrix products instead of seven.
//
// A preparation kernel writes lse*log2(e) and delta per query row, padded to a multiple of 128 rows per (b,h) with
// +inf / 0: a padded row then gives p = 0 without any test.
//
// Every wait is bounded: on expiry the CTA sets the library's error word, drains and exits.
#include "tlin_internal.h"
#include "sm100_ptx.cuh"
#include "tc_common.cuh"
#include <math_constants.h>
#include <type_traits>

namespace tlin {
namespace {

using namespace ptx;
using namespace tc;

constexpr int kProducerWarp = 8;
constexpr int kMmaWarp = 9;
constexpr float kLog2e = 1.4426950408889634f;

struct BwdParams {
    const float* neg_lse2;        // [B*H, Wpad]  -lse * log2(e), -inf beyond W
    const float* delta;       // [B*H, Wpad]  dout . out,   0 beyond W
    void* dq;                 // [B*H, W, D] bf16
    void* dk;                 // [B*H, N, D] bf16
    void* dv;
    float* ws;                // partial dQ slots of the dq kernel
    int* status;
    long long total_units;    // dk/dv kernel: B*H*key_tiles; dq kernel: the plan's units
    int n_groups, q_tiles, key_tiles, schedule;   // dq kernel: the forward's plan fields
    int q_tiles128;           // ceil(W / 128)
    int N, W, Wpad, causal;
    int wide_stores;          // dq and the workspace are 32-byte aligned: the dQ kernel may use 32-byte stores
    float scale_log2e, scale;
};

// ------------------------------------------------------------------------------------------ preparation
// Row statistics of the backward pass: neg_lse2 = -lse * log2(e) and delta = sum_c out*dout, on rows padded to 128 per (b,h)
// (padding rows: +inf and 0).  D/8 lanes share a row with one 16-byte load per tensor each; a warp keeps kPrepPasses
// groups of rows in flight, so that enough bytes are outstanding to stream at HBM speed.
constexpr int kPrepPasses = 4;
template <int D>
__host__ __device__ constexpr int prep_rows_per_block() { return 8 * (32 / (D / 8)) * kPrepPasses; }

template <int D>
__global__ void __launch_bounds__(256)
bwd_prep_kernel(const __nv_bfloat16* out, const __nv_bfloat16* dout, const float* lse, float* neg_lse2, float* delta, float* dq32,
                int W, int Wpad, long long rows_padded) {
    after_previous();
    let_next_start();
    constexpr int LPR = D / 8;              // lanes per row
    constexpr int RPP = 32 / LPR;           // rows per pass of a warp
    const int lane = threadIdx.x & 31, sub = lane / LPR, l = lane % LPR;
    const long long first = ((long long)blockIdx.x * 8 + (threadIdx.x >> 5)) * (RPP * kPrepPasses) + sub;
    uint4 a[kPrepPasses], b[kPrepPasses];
    long long row[kPrepPasses];
#pragma unroll
    for (int ps = 0; ps < kPrepPasses; ++ps) {
        const long long prow = first + ps * RPP;
        const long long bh = prow / Wpad;
        const int i = (int)(prow - bh * Wpad);
        row[ps] = (prow < rows_padded && i < W) ? bh * W + i : -1;
        if (dq32 != nullptr && prow < rows_padded) {            // the fp32 dQ sums of the one-kernel arrangement start at zero
            float4* z = reinterpret_cast<float4*>(dq32 + prow * D) + l;
            z[0] = z[LPR] = make_float4(0.f, 0.f, 0.f, 0.f);
        }
        a[ps] = b[ps] = make_uint4(0u, 0u, 0u, 0u);
        if (row[ps] >= 0) {
            a[ps] = *reinterpret_cast<const uint4*>(out + row[ps] * D + l * 8);
            b[ps] = *reinterpret_cast<const uint4*>(dout + row[ps] * D + l * 8);
        }
    }
#pragma unroll
    for (int ps = 0; ps < kPrepPasses; ++ps) {
        const uint32_t* aw = reinterpret_cast<const uint32_t*>(&a[ps]);
        const uint32_t* bw = reinterpret_cast<const uint32_t*>(&b[ps]);
        float acc = 0.f;
#pragma unroll
        for (int e = 0; e < 4; ++e) {
            const float2 x = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&aw[e]));
            const float2 y = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&bw[e]));
            acc = fmaf(x.x, y.x, fmaf(x.y, y.y, acc));
        }
#pragma unroll
        for (int o = LPR / 2; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
        const long long prow = first + ps * RPP;
        if (l == 0 && prow < rows_padded) {
            neg_lse2[prow] = row[ps] >= 0 ? -lse[row[ps]] * kLog2e : -CUDART_INF_F;
            delta[prow] = row[ps] >= 0 ? acc : 0.f;
        }
    }
}

// ------------------------------------------------------------------------------------------ dK / dV
template <int D>
struct ACfg {
    static constexpr int kTileBytes = kQTile * D * 2;          // one 128-row tile (K or V)
    static constexpr int kHalfBytes = 64 * D * 2;              // one 64-row tile (Q or dout of a chain step)
    static constexpr int kBoxes = D / 64;
    // Chains of 64 queries, one warpgroup each: as many as TMEM has columns for beside dK and dV.  A chain's products and its
    // elementwise work follow one another and leave both pipes half idle at d = 64; a third chain fills them better.  Backward
    // with two / three, microseconds: 36 x 1999^2 causal 111.5 / 101.6, 128 x 1024 x 8192 1232 / 1160, 16 x 2000^2 68.5 / 65.4.
    static constexpr int kChains = D == 128 ? 2 : 3;
    static constexpr int kProducer = 4 * kChains, kMma = kProducer + 1, kKv = kProducer + 2;      // warps below: P and dS
    static constexpr int kThreads = D == 128 ? 32 * 11 : 32 * 16;
    // d = 64: setmaxnreg moves registers from the fourth warpgroup to the chains; the CTA starts with 128 per thread.  An increase
    // beyond what was released would wait for ever, one below the count at launch is an illegal instruction.
    static constexpr int kComputeRegs = 136, kOtherRegs = 104;
    static_assert(384 * kComputeRegs + 128 * kOtherRegs <= 512 * 128 && kComputeRegs > 128 && kOtherRegs < 128, "register budget");
    // columns of a result row that a thread writes out: half a row of dK and of dV, or (three chains) a whole row of one of them
    static constexpr int kOutCols = kChains == 2 ? D / 2 : D;
    static constexpr int kSlots = D == 128 ? 4 : 8;            // ring of chain steps: Q (64 rows), dout (64 rows), 64 neg_lse2 + 64 delta
    static constexpr int kSlotBytes = 2 * kHalfBytes;
    static constexpr int kOffKV = 0;
    static constexpr int kOffRing = 2 * kTileBytes;
    static constexpr int kOffStats = kOffRing + kSlots * kSlotBytes;
    static constexpr int kOffStage = kOffStats + kSlots * 512;  // per writing warp 32 rows of kOutCols: dK / dV on their way out
    static constexpr int kOffBars = kOffStage + 8 * 32 * kOutCols * 2;
    static constexpr int kNumBars = 4 + 2 * kChains + 2 * kSlots;
    static constexpr int kSmemBytes = kOffBars + kNumBars * 8 + 16;
    // TMEM columns: dK, dV (D each); per chain x (64 queries of the tile) 128 columns: S^T_x (64 fp32) and dP^T_x
    // (64 fp32); P^T_x and dS^T_x (bf16, 32 columns each) are written over the first half of S^T_x and dP^T_x
    static constexpr uint32_t kColDK = 0, kColDV = D, kColR = 2 * D;
};

// Order in which the CTAs of the key-tile kernels take the (b,h,key tile) units.  With the window rule key tile t is visited by
// fewer query tiles the later it is.
enum { kUnitRuns = 0,      // contiguous runs of equal cost: a CTA stays on one or two (b,h) (dK/dV kernel)
       kUnitTurns = 1,     // in turn (CTA c: c, c + CTAs, ...): all CTAs work on the key tiles of two or three (b,h) at any time, so the
                           // rows of the fp32 dQ buffer they add to, and the Q / dout tiles they read, stay in L2 whatever the size
                           // of the call (one-kernel arrangement)
       kUnitDealt = 2 };   // by descending cost over all (b,h) (dealt_position)
// A CTA walks u = begin, begin + step, ... below end; unit(u, bh, t) says which (b,h) and key tile that is.
template <int kOrder>
struct UnitOrder {
    long long begin, end, step;
    int T;
    __device__ UnitOrder(const BwdParams& p) : T(p.key_tiles) {
        if constexpr (kOrder == kUnitRuns) {
            begin = bwd_first_unit_of_share(p.N, p.W, p.causal, p.total_units, p.key_tiles, blockIdx.x, gridDim.x);
            end = bwd_first_unit_of_share(p.N, p.W, p.causal, p.total_units, p.key_tiles, blockIdx.x + 1, gridDim.x);
            step = 1;
        } else if constexpr (kOrder == kUnitTurns) {
            begin = blockIdx.x;
            end = p.total_units;
            step = gridDim.x;
        } else {                        // u counts rounds
            begin = 0;
            const int full = (int)(p.total_units / gridDim.x);
            end = full + (dealt_position(full) < p.total_units ? 1 : 0);
            step = 1;
        }
    }
    __device__ void unit(const BwdParams& p, long long u, int& bh, int& t) const {
        if constexpr (kOrder == kUnitDealt) {
            const unsigned pos = (unsigned)dealt_position((int)u), n_bh = (unsigned)p.total_units / (unsigned)T;
            t = (int)(pos / n_bh);
            bh = (int)(pos - (unsigned)t * n_bh);
        } else {
            bh = (int)(u / T);
            t = (int)(u - (long long)bh * T);
        }
    }
};
// Dealing pays where runs and turns come out uneven, i.e. with few units per CTA and a window that is a large part of the keys (units
// per CTA x N / W up to 32: costliest CTA 8 to 100 % above the mean against 1 to 10 %), and costs about 5 % of locality otherwise
// (B1 H32 N32768 W512 817 -> 867 us).  Measured: B3 H12 N=W=1999 d64 161 -> 119 us (two kernels), B1 H16 N=W=2000 d128 84 -> 61 us
// (one kernel).  What dealing gives shrinks as the tensors that the units of a (b,h) share (one kernel: dQ sums, Q and dout; two: Q or
// dout) outgrow L2, hence the bound, which lies where the one kernel stops gaining (d128, turns / dealt, us): 100 MiB N=W=4096 404 / 333,
// N4096 W2048 511 / 498; 136 MiB 490 / 456, 692 / 689; 144 MiB 503 / 485, 695 / 738; 200 MiB 731 / 689, 1032 / 1080.  The two kernels
// mostly gain 5 to 12 % on either side of it (d64 N=W=4096: 136 MiB 1449 / 1286, 160 MiB 1694 / 1511, 200 MiB 2140 / 1917).
bool deal_units(long long bh, int N, int W, int causal, int key_tiles, long long shared_bytes, int num_sms) {
    return causal && shared_bytes <= (140LL << 20) && bh * key_tiles * N <= 32LL * num_sms * W;
}

// first 128-row query tile that may use a key of key tile t
__device__ __forceinline__ int first_q_tile(const BwdParams& p, int t) {
    if (!p.causal) return 0;
    const long long f = (long long)t * kTileN - ((long long)p.N - p.W);
    return f <= 0 ? 0 : (int)(f / kQTile);
}

template <int D, int kOrder>
__global__ void __launch_bounds__(ACfg<D>::kThreads, 1)
bwd_dkdv_tc_kernel(const __grid_constant__ CUtensorMap map_q, const __grid_constant__ CUtensorMap map_k,
                   const __grid_constant__ CUtensorMap map_v, const __grid_constant__ CUtensorMap map_do, const BwdParams p) {
    using C = ACfg<D>;
    extern __shared__ __align__(1024) uint8_t smem[];
    uint8_t* sKV = smem + C::kOffKV;          // K, V
    uint8_t* sRing = smem + C::kOffRing;      // [kSlots][Q 64 rows | dout 64 rows]
    float* sStats = reinterpret_cast<float*>(smem + C::kOffStats);   // [kSlots][neg_lse2 64 | delta 64]
    uint64_t* bars = reinterpret_cast<uint64_t*>(smem + C::kOffBars);
    uint64_t* kv_full = bars + 0;
    uint64_t* kv_empty = bars + 1;
    uint64_t* acc_full = bars + 2;    // dK, dV of the key tile are complete
    uint64_t* acc_empty = bars + 3;   // all threads have read them
    uint64_t* sdp_full = bars + 4;    // [kChains] S^T_x and dP^T_x of a chain step are in TMEM
    uint64_t* pds_full = sdp_full + C::kChains;   // [kChains] the chain's threads have stored P^T_x and dS^T_x
    uint64_t* slot_full = pds_full + C::kChains;  // [kSlots]
    uint64_t* slot_empty = slot_full + C::kSlots;
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(bars + C::kNumBars);
    int* abort_flag = reinterpret_cast<int*>(tmem_slot + 1);

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const bool base_ok = (smem_u32(smem) & 1023u) == 0;   // the swizzled tiles need 1024-byte alignment

    if (threadIdx.x == 0) {
        *abort_flag = base_ok ? 0 : 1;
        mbar_init(kv_full, 1);
        mbar_init(kv_empty, 1);
        for (int i = 0; i < C::kChains; ++i) {
            mbar_init(&sdp_full[i], 1);
            mbar_init(&pds_full[i], 128);
        }
        for (int i = 0; i < C::kSlots; ++i) {
            mbar_init(&slot_full[i], 1);
            mbar_init(&slot_empty[i], 1);
        }
        mbar_init(acc_full, 1);
        mbar_init(acc_empty, 256);
        fence_mbar_init();
    }
    if (warp == C::kMma) {
        tmem_alloc(tmem_slot, 512);
        tmem_relinquish();
    }
    if (warp == C::kProducer && lane == 0) {
        prefetch_tensormap(&map_q);
        prefetch_tensormap(&map_k);
        prefetch_tensormap(&map_v);
        prefetch_tensormap(&map_do);
    }
    tc_fence_before();
    after_previous();
    let_next_start();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem_base = *tmem_slot;
    volatile int* abort_p = abort_flag;
    const UnitOrder<kOrder> order(p);

    if constexpr (C::kChains == 3) setmaxnreg_dec<C::kOtherRegs>();
    if (warp == C::kProducer) {
        // ------------------------------------------------------------------ TMA producer: Q / dout / row statistics ring
        // The ring runs ahead of the key tiles: the first chain steps of the next key tile are loaded while the
        // current one is still being worked on.
        if (lane == 0) {
            bool ok = base_ok;
            uint32_t hh = 0;                // chain steps (64 queries each) issued
            for (long long u = order.begin; u < order.end && ok; u += order.step) {
                int bh, t;
                order.unit(p, u, bh, t);
                const int row_first = first_q_tile(p, t) * kQTile, row_end = p.q_tiles128 * kQTile;
                for (int row = row_first; row < row_end && ok; row += 64, ++hh) {
                    const uint32_t slot = hh % C::kSlots, round = hh / C::kSlots;
                    ok = mbar_wait(&slot_empty[slot], (round & 1) ^ 1, abort_p);
                    if (!ok) break;
                    uint8_t* dst = sRing + slot * C::kSlotBytes;
                    mbar_arrive_expect_tx(&slot_full[slot], C::kSlotBytes + 512);
                    for (int x = 0; x < C::kBoxes; ++x) {
                        tma_load_3d(dst + x * (64 * 128), &map_q, &slot_full[slot], x * 64, row, bh);
                        tma_load_3d(dst + C::kHalfBytes + x * (64 * 128), &map_do, &slot_full[slot], x * 64, row, bh);
                    }
                    bulk_load_1d(sStats + slot * 128, p.neg_lse2 + (long long)bh * p.Wpad + row, 256, &slot_full[slot]);
                    bulk_load_1d(sStats + slot * 128 + 64, p.delta + (long long)bh * p.Wpad + row, 256, &slot_full[slot]);
                }
            }
            if (!ok && base_ok) {
                int dummy = 0;              // leave no copy in flight: the barriers armed last must complete (bounded)
                for (uint32_t back = 1; back <= (uint32_t)C::kSlots && back <= hh; ++back) {
                    const uint32_t id = hh - back;
                    mbar_wait(&slot_full[id % C::kSlots], (id / C::kSlots) & 1, &dummy, 200000000LL);
                }
            }
        }
    } else if (warp == C::kKv) {
        // ------------------------------------------------------------------ TMA producer: K, V of the key tiles
        if (lane == 0) {
            bool ok = base_ok;
            uint32_t n = 0;
            for (long long u = order.begin; u < order.end && ok; u += order.step, ++n) {
                int bh, t, bh_n, t_n;
                order.unit(p, u, bh, t);
                if (u + order.step < order.end) {   // K, V have one buffer: the next tile's rows come as far as L2 meanwhile
                    order.unit(p, u + order.step, bh_n, t_n);
                    for (int x = 0; x < C::kBoxes; ++x) {
                        tma_prefetch_l2_3d(&map_k, x * 64, t_n * kTileN, bh_n);
                        tma_prefetch_l2_3d(&map_v, x * 64, t_n * kTileN, bh_n);
                    }
                }
                ok = mbar_wait(kv_empty, (n & 1) ^ 1, abort_p);
                if (!ok) break;
                mbar_arrive_expect_tx(kv_full, 2 * C::kTileBytes);
                for (int x = 0; x < C::kBoxes; ++x) {
                    tma_load_3d(sKV + x * (kQTile * 128), &map_k, kv_full, x * 64, t * kTileN, bh);
                    tma_load_3d(sKV + C::kTileBytes + x * (kQTile * 128), &map_v, kv_full, x * 64, t * kTileN, bh);
                }
            }
            if (!ok && base_ok && n > 0) {
                int dummy = 0;
                mbar_wait(kv_full, (n - 1) & 1, &dummy, 200000000LL);
            }
        }
    } else if (warp == C::kMma) {
        // ------------------------------------------------------------------ MMA issuer (all lanes walk, the lane elected once issues)
        const uint32_t idesc_st = make_idesc_bf16(kQTile, 64, 0, 0);         // S^T, dP^T of a chain: M = keys, N = 64 queries
        const uint32_t idesc_acc = make_idesc_bf16(kQTile, D, 0, 1);         // dV, dK: A in TMEM, B MN-major
        const uint64_t kmaj = make_smem_desc_sw128(smem_u32(smem), 16, 1024);
        const uint64_t mnmaj = make_smem_desc_sw128(smem_u32(smem), 64 * 128, 1024);   // 64-row tiles: 8 KB between column blocks
        const uint32_t desc_hi = (uint32_t)(kmaj >> 32);
        const uint32_t kmaj_lo = (uint32_t)kmaj, mnmaj_lo = (uint32_t)mnmaj;
        const uint32_t tmem_u = __shfl_sync(0xffffffffu, tmem_base, 0);
        const uint32_t lead = elect_one() ? 1u : 0u;
        const uint32_t tDK = tmem_u + C::kColDK, tDV = tmem_u + C::kColDV;
        const uint32_t k_off = (uint32_t)(C::kOffKV >> 4), v_off = (uint32_t)((C::kOffKV + C::kTileBytes) >> 4);
        // [S^T_x | dP^T_x] = [K Q_x^T | V dout_x^T]: A a 128-row K-major tile, B the 64-row K-major tile of the slot
        auto issue_sdp = [&](int x, uint32_t slot) {
            const uint32_t q_off = (uint32_t)((C::kOffRing + slot * C::kSlotBytes) >> 4), do_off = q_off + (uint32_t)(C::kHalfBytes >> 4);
            const uint32_t d = tmem_u + C::kColR + x * 128;
#pragma unroll
            for (int kk = 0; kk < D / 16; ++kk) {
                const uint32_t a16 = ((kk >> 2) * (kQTile * 128) + (kk & 3) * 32) >> 4, b16 = ((kk >> 2) * (64 * 128) + (kk & 3) * 32) >> 4;
                mma_ss_lead(lead, d, kmaj_lo + k_off + a16, kmaj_lo + q_off + b16, desc_hi, idesc_st, kk > 0);
            }
#pragma unroll
            for (int kk = 0; kk < D / 16; ++kk) {
                const uint32_t a16 = ((kk >> 2) * (kQTile * 128) + (kk & 3) * 32) >> 4, b16 = ((kk >> 2) * (64 * 128) + (kk & 3) * 32) >> 4;
                mma_ss_lead(lead, d + 64, kmaj_lo + v_off + a16, kmaj_lo + do_off + b16, desc_hi, idesc_st, kk > 0);
            }
            commit_lead(lead, &sdp_full[x]);
        };
        // dV += P^T_x dout_x, dK += dS^T_x Q_x: A in TMEM (64 queries = 32 columns), B the slot's 64-row tile read MN-major
        auto issue_acc = [&](int x, uint32_t slot, bool accumulate) {
            const uint32_t q_off = (uint32_t)((C::kOffRing + slot * C::kSlotBytes) >> 4), do_off = q_off + (uint32_t)(C::kHalfBytes >> 4);
            const uint32_t a = tmem_u + C::kColR + x * 128;
#pragma unroll
            for (int kk = 0; kk < 4; ++kk)
                mma_ts_lead(lead, tDV, a + kk * 8, mnmaj_lo + do_off + kk * (2048 >> 4), desc_hi, idesc_acc, (accumulate || kk > 0) ? 1u : 0u);
#pragma unroll
            for (int kk = 0; kk < 4; ++kk)
                mma_ts_lead(lead, tDK, a + 64 + kk * 8, mnmaj_lo + q_off + kk * (2048 >> 4), desc_hi, idesc_acc, (accumulate || kk > 0) ? 1u : 0u);
            commit_lead(lead, &slot_empty[slot]);
        };
        bool ok = base_ok;
        uint32_t hh = 0, n = 0;             // chain steps and key tiles done; chain step h belongs to chain h mod kChains and ring slot h mod kSlots
        for (long long u = order.begin; u < order.end && ok; u += order.step, ++n) {
            int bh, t;
            order.unit(p, u, bh, t);
            const uint32_t first = hh, end = hh + 2 * (uint32_t)(p.q_tiles128 - first_q_tile(p, t));
            ok = __all_sync(0xffffffffu, mbar_wait(kv_full, n & 1, abort_p));
            if (!ok) break;
            for (uint32_t h = first; h < first + C::kChains && h < end; ++h) {
                ok = __all_sync(0xffffffffu, mbar_wait(&slot_full[h % C::kSlots], (h / C::kSlots) & 1, abort_p));
                if (!ok) break;
                issue_sdp(h % C::kChains, h % C::kSlots);
            }
            if (!ok) break;
            if (end - first <= C::kChains) commit_lead(lead, kv_empty);     // K, V have been read for the last time: the next tile's may load
            for (; hh < end; ++hh) {
                const uint32_t x = hh % C::kChains, hn = hh + C::kChains;
                ok = __all_sync(0xffffffffu, mbar_wait(&pds_full[x], (hh / C::kChains) & 1, abort_p));
                if (!ok) break;
                if (hh == first && n > 0) {                 // the previous key tile's dK, dV must have been read out
                    ok = __all_sync(0xffffffffu, mbar_wait(acc_empty, (n - 1) & 1, abort_p));
                    if (!ok) break;
                }
                tc_fence_after();
                issue_acc(x, hh % C::kSlots, hh > first);
                if (hn < end) {
                    ok = __all_sync(0xffffffffu, mbar_wait(&slot_full[hn % C::kSlots], (hn / C::kSlots) & 1, abort_p));
                    if (!ok) break;
                    issue_sdp(x, hn % C::kSlots);
                    if (hn + 1 == end) commit_lead(lead, kv_empty);
                }
            }
            if (!ok) break;
            commit_lead(lead, acc_full);
        }
    } else if (warp < C::kProducer) {
        if constexpr (C::kChains == 3) setmaxnreg_inc<C::kComputeRegs>();
        // ------------------------------------------------------------------ elementwise threads
        const int wg = warp >> 2;                              // chain: which 64 queries of every tile
        const int r = (warp & 3) * 32 + lane;                  // key row inside the tile == TMEM lane
        const uint32_t lane_addr = (uint32_t)((warp & 3) * 32) << 16;
        const uint32_t tS = tmem_base + lane_addr + C::kColR + wg * 128;
        const uint32_t tDP = tS + 64;
        bool ok = base_ok;
        uint32_t hh = 0, n = 0;                                // first chain step of the key tile, key tiles done
        for (long long u = order.begin; u < order.end && ok; u += order.step, ++n) {
            int bh, t;
            order.unit(p, u, bh, t);
            const int key = t * kTileN + r;
            const int i_first = first_q_tile(p, t);
            const long long shift = (long long)p.N - p.W;       // query q may use key k iff q >= k - shift
            const int q_min = p.causal ? (int)((long long)key - shift) : -0x7fffffff;
            const int q_min_warp = p.causal ? (int)((long long)key - lane + 31 - shift) : -0x7fffffff;   // largest in the warp
            const uint64_t scale2 = f2_pack(p.scale_log2e, p.scale_log2e);
            // a copy of the step for the tiles with masked elements: conditions in the loop cut it into short blocks
            auto step = [&](uint32_t h, int q0, auto masked_tag) {
                constexpr bool kMasked = decltype(masked_tag)::value;
                const uint32_t slot = h % C::kSlots;
                const float* st = sStats + slot * 128;
                ok = __all_sync(0xffffffffu, mbar_wait(&sdp_full[wg], (h / C::kChains) & 1, abort_p));
                if (!ok) return;
                // already complete (the MMAs waited for it); observing it here orders the bulk-copied neg_lse2 / delta
                // before this thread's reads
                ok = __all_sync(0xffffffffu, mbar_wait(&slot_full[slot], (h / C::kSlots) & 1, abort_p));
                if (!ok) return;
                tc_fence_after();
                uint32_t svb[2][16], dvb[2][16];
                tmem_ld16_async(tS, svb[0]);
                tmem_ld16_async(tDP, dvb[0]);
#pragma unroll
                for (int part = 0; part < 4; ++part) {       // 16 columns at a time: 32 spill at three chains and gain nothing at two
                    uint32_t (&sv)[16] = svb[part & 1];
                    uint32_t (&dv_)[16] = dvb[part & 1];
                    tmem_wait_ld16(sv);
                    tmem_wait_ld16(dv_);
                    if (part < 3) {                          // in flight during the arithmetic
                        tmem_ld16_async(tS + (part + 1) * 16, svb[(part + 1) & 1]);
                        tmem_ld16_async(tDP + (part + 1) * 16, dvb[(part + 1) & 1]);
                    }
                    uint32_t pk[8], dk_[8];
#pragma unroll
                    for (int c = 0; c < 16; c += 4) {
                        const ulonglong2 l4 = *reinterpret_cast<const ulonglong2*>(st + part * 16 + c);        // two pairs of floats
                        const ulonglong2 d4 = *reinterpret_cast<const ulonglong2*>(st + 64 + part * 16 + c);
#pragma unroll
                        for (int e = 0; e < 4; e += 2) {
                            float p0, p1, d0, d1;
                            f2_unpack(f2_fma(f2_pack_bits(sv[c + e], sv[c + e + 1]), scale2, e == 0 ? l4.x : l4.y), p0, p1);
                            p0 = ex2(p0);
                            p1 = ex2(p1);
                            if (kMasked && q0 + part * 16 + c + e < q_min) p0 = 0.f;
                            if (kMasked && q0 + part * 16 + c + e + 1 < q_min) p1 = 0.f;
                            f2_unpack(f2_mul(f2_pack(p0, p1), f2_sub(f2_pack_bits(dv_[c + e], dv_[c + e + 1]), e == 0 ? d4.x : d4.y)), d0, d1);
                            pk[(c + e) / 2] = pack_bf16x2(p0, p1);
                            dk_[(c + e) / 2] = pack_bf16x2(d0, d1);
                        }
                    }
                    // bf16 P^T over columns of S^T, dS^T over columns of dP^T, that are already in registers
                    tmem_st8(tS + part * 8, pk);
                    tmem_st8(tDP + part * 8, dk_);
                }
                tc_wait_st();
                tc_fence_before();
                mbar_arrive(&pds_full[wg]);
            };
            const uint32_t end = hh + 2 * (uint32_t)(p.q_tiles128 - i_first);
            for (uint32_t h = hh + ((uint32_t)wg + C::kChains - hh % C::kChains) % C::kChains; h < end && ok; h += C::kChains) {
                const int q0 = i_first * kQTile + (int)(h - hh) * 64;   // first query of this thread's columns
                if (q0 < q_min_warp) step(h, q0, std::true_type{});     // warp-uniform: some element of some lane is masked
                else step(h, q0, std::false_type{});
            }
            hh = end;
            if (!ok) break;
            if (wg >= 2) continue;                                 // the third chain leaves the results to the other two
            // ---------------------------------------------------------------- dK, dV of this key tile
            ok = __all_sync(0xffffffffu, mbar_wait(acc_full, n & 1, abort_p));
            if (!ok) break;
            tc_fence_after();
            // Each thread holds half a row of dK and of dV (three chains: a whole row of one of them).  Written straight from the
            // registers a warp's store would touch 32 different lines; the warp passes its rows through shared memory (16-byte
            // pieces, piece index xor row so that neither side has bank conflicts beyond the minimum) and stores whole lines.
            constexpr int kCols = C::kOutCols, kPieces = kCols / 8;   // 16-byte pieces per row
            constexpr int kRowsPerStore = 32 / kPieces;
            uint8_t* stage = smem + C::kOffStage + warp * (32 * kCols * 2);
            const int key_warp = t * kTileN + (warp & 3) * 32;     // key of lane 0
#pragma unroll
            for (int part = 0; part < (C::kChains == 2 ? 2 : 1); ++part) {
                const int which = C::kChains == 2 ? part : wg, col = C::kChains == 2 ? wg * kCols : 0;
                const uint32_t tA = tmem_base + lane_addr + (which == 0 ? C::kColDK : C::kColDV) + col;
                const float f = which == 0 ? p.scale : 1.f;
#pragma unroll
                for (int c = 0; c < kCols / 32; ++c) {
                    uint32_t o[32];
                    tmem_ld32(tA + c * 32, o);
#pragma unroll
                    for (int v4 = 0; v4 < 4; ++v4) {
                        uint4 w;
                        w.x = pack_bf16x2(__uint_as_float(o[v4 * 8 + 0]) * f, __uint_as_float(o[v4 * 8 + 1]) * f);
                        w.y = pack_bf16x2(__uint_as_float(o[v4 * 8 + 2]) * f, __uint_as_float(o[v4 * 8 + 3]) * f);
                        w.z = pack_bf16x2(__uint_as_float(o[v4 * 8 + 4]) * f, __uint_as_float(o[v4 * 8 + 5]) * f);
                        w.w = pack_bf16x2(__uint_as_float(o[v4 * 8 + 6]) * f, __uint_as_float(o[v4 * 8 + 7]) * f);
                        const int piece = c * 4 + v4;
                        *reinterpret_cast<uint4*>(stage + lane * (kCols * 2) + ((piece ^ (lane & (kPieces - 1))) << 4)) = w;
                    }
                }
                __syncwarp();
                __nv_bfloat16* dst = reinterpret_cast<__nv_bfloat16*>(which == 0 ? p.dk : p.dv) + ((long long)bh * p.N + key_warp) * D + col;
#pragma unroll
                for (int it = 0; it < 32 / kRowsPerStore; ++it) {
                    const int rrow = it * kRowsPerStore + lane / kPieces, piece = lane % kPieces;
                    const uint4 w = *reinterpret_cast<const uint4*>(stage + rrow * (kCols * 2) + ((piece ^ (rrow & (kPieces - 1))) << 4));
                    if (key_warp + rrow < p.N) *reinterpret_cast<uint4*>(dst + (long long)rrow * D + piece * 8) = w;
                }
                __syncwarp();
            }
            tc_fence_before();
            mbar_arrive(acc_empty);
        }
    }

    tc_fence_before();
    __syncthreads();
    if (threadIdx.x == 0 && *abort_flag) atomicExch(p.status, base_ok ? (int)TLIN_ERR_TIMEOUT : (int)TLIN_ERR_CUDA);
    if (warp == C::kMma) {
        tc_fence_after();
        tmem_dealloc(tmem_base, 512);
    }
}

// ------------------------------------------------------------------------------------------ dK / dV / dQ in one kernel
// A CTA owns one 128-key tile at a time and walks the 128-row query tiles that may see it; five products per step, all 128 wide:
//   S^T = K Q^T, dP^T = V dout^T (TMEM lane = key, column = query), dV += P^T dout, dK += dS^T Q (P^T, dS^T bf16 in TMEM, written
//   over S^T and dP^T), dQ^T = K^T dS^T (K read MN-major; dS^T once more in shared memory; over dP^T, whose dS^T dK has consumed).
// TMEM is full with S^T, dP^T, dK and dV, so a step's products follow one another; what keeps the tensor pipe busy is the order:
//   dK(j), dQ(j) | dP(j+1) once dQ(j) has been taken out of TMEM | dV(j+1), S(j+2) once P(j+1) is there
// The exponentials of step j+1 run while dK(j) and dQ(j) do, dS(j+1) while dV(j+1) and S(j+2) do.
// Three warpgroups work on a step: two take 64 queries each (thread = key row) through P and dS, the third takes dQ^T into
// registers (thread = column of dQ), passes it through shared memory and has the copy engine add the rows to the fp32 dQ in the
// workspace.  That is 64 KB of reductions per step, which L2 takes at about 6 TB/s: 0.68 of the 1.28 ms below.
// Measured at B4 H32 N8192 W1024 (full clock / under the power cap): reductions in the threads that form P and dS, scores 64
// queries wide 1543 / 1759 us; 128 wide, a warpgroup of its own with red instructions 1405 / 1601 us (they fill the load/store
// unit that P and dS need); through the copy engine 1278 / 1397 us.  B1 H32 N8192 W1024 449 -> 354 us, B1 H32 N32768 W512
// 942 -> 804 us, B2 H16 N4096 W512 132 -> 108 us, B1 H4 N700 W300 28 -> 18 us.
template <int D>
struct FCfg {
    static_assert(D == 128, "the transposed dQ accumulator needs M = d = 128");
    static constexpr int kTileBytes = kQTile * D * 2;          // one 128-row tile (K, V, Q or dout)
    static constexpr int kBoxes = D / 64;
    static constexpr int kOffK = 0, kOffV = kTileBytes;
    static constexpr int kOffQ = 2 * kTileBytes;               // 2 slots
    static constexpr int kOffDO = 4 * kTileBytes;
    static constexpr int kOffStage = 5 * kTileBytes;           // dS^T tile: two blocks of 128 keys x 64 queries; dK / dV rows on their way out
    static constexpr int kOffDQ = 6 * kTileBytes;              // 4 buffers of 16 queries x D fp32: dQ rows on their way to L2
    static constexpr int kDqRows = 16;
    static constexpr int kOffStats = 7 * kTileBytes;           // 2 slots: neg_lse2 of 128 rows, delta of 128 rows
    static constexpr int kOffBars = kOffStats + 2 * 1024;
    static constexpr int kNumBars = 18;
    static constexpr int kSmemBytes = kOffBars + kNumBars * 8 + 16;
    static constexpr uint32_t kColDK = 0, kColDV = D, kColS = 2 * D, kColDP = 2 * D + 128;
    static constexpr int kThreads = 32 * 16;
    static constexpr int kDqWarp = 8, kProducer = 12, kMma = 13, kKv = 14;      // warps 0 to 7: P and dS
    // setmaxnreg moves registers between warpgroups; the CTA starts with 128 per thread (which the P and dS warps keep).  An
    // increase beyond what the others released would wait for ever, one below the count at launch is an illegal instruction.
    static constexpr int kLaunchRegs = 128, kDqRegs = 152, kOtherRegs = 104;
    static_assert(128 * kDqRegs + 128 * kOtherRegs <= 256 * kLaunchRegs && kDqRegs > kLaunchRegs && kOtherRegs < kLaunchRegs, "register budget");
};

template <int D, int kOrder>
__global__ void __launch_bounds__(FCfg<D>::kThreads, 1)
bwd_fused_tc_kernel(const __grid_constant__ CUtensorMap map_q, const __grid_constant__ CUtensorMap map_k,
                    const __grid_constant__ CUtensorMap map_v, const __grid_constant__ CUtensorMap map_do, const BwdParams p) {
    using C = FCfg<D>;
    extern __shared__ __align__(1024) uint8_t smem[];
    float* sStats = reinterpret_cast<float*>(smem + C::kOffStats);   // [2][neg_lse2 128 | delta 128]
    uint64_t* bars = reinterpret_cast<uint64_t*>(smem + C::kOffBars);
    uint64_t* q_full = bars + 0;      // [2] Q and the row statistics of a step
    uint64_t* q_empty = bars + 2;     // [2]
    uint64_t* do_full = bars + 4;
    uint64_t* do_empty = bars + 5;
    uint64_t* k_full = bars + 6;
    uint64_t* k_empty = bars + 7;
    uint64_t* v_full = bars + 8;
    uint64_t* v_empty = bars + 9;
    uint64_t* s_full = bars + 10;     // S^T of a step is in TMEM
    uint64_t* p_full = bars + 11;     // P^T is written
    uint64_t* dp_full = bars + 12;    // dP^T is in TMEM
    uint64_t* ds_full = bars + 13;    // dS^T is written (TMEM and shared memory)
    uint64_t* dq_full = bars + 14;    // dQ^T is in TMEM
    uint64_t* dq_drained = bars + 15; // the dQ warpgroup holds it in registers
    uint64_t* acc_full = bars + 16;   // dK, dV of the key tile are complete
    uint64_t* acc_empty = bars + 17;  // all threads have read them
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(bars + C::kNumBars);
    int* abort_flag = reinterpret_cast<int*>(tmem_slot + 1);

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const bool base_ok = (smem_u32(smem) & 1023u) == 0;   // the swizzled tiles need 1024-byte alignment

    if (threadIdx.x == 0) {
        *abort_flag = base_ok ? 0 : 1;
        for (int i = 0; i < C::kNumBars; ++i)
            mbar_init(&bars[i], &bars[i] == p_full || &bars[i] == ds_full || &bars[i] == acc_empty ? 256 : &bars[i] == dq_drained ? 128 : 1);
        fence_mbar_init();
    }
    if (warp == C::kMma) {
        tmem_alloc(tmem_slot, 512);
        tmem_relinquish();
    }
    if (warp == C::kProducer && lane == 0) {
        prefetch_tensormap(&map_q);
        prefetch_tensormap(&map_k);
        prefetch_tensormap(&map_v);
        prefetch_tensormap(&map_do);
    }
    tc_fence_before();
    after_previous();
    let_next_start();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem_base = *tmem_slot;
    volatile int* abort_p = abort_flag;
    const UnitOrder<kOrder> order(p);

    if (warp >= C::kProducer) {
    setmaxnreg_dec<C::kOtherRegs>();
    if (warp == C::kProducer) {
        // ------------------------------------------------------------------ TMA producer: Q, dout and row statistics of the steps
        if (lane == 0) {
            bool ok = base_ok;
            uint32_t nq = 0, ndo = 0;       // tiles armed
            for (long long u = order.begin; u < order.end && ok; u += order.step) {
                int bh, t;
                order.unit(p, u, bh, t);
                for (int i = first_q_tile(p, t); i < p.q_tiles128; ++i) {
                    const uint32_t slot = nq & 1, par = ((nq >> 1) & 1) ^ 1;
                    const int row = i * kQTile;
                    ok = mbar_wait(&q_empty[slot], par, abort_p);
                    if (!ok) break;
                    mbar_arrive_expect_tx(&q_full[slot], C::kTileBytes + 1024);
                    ++nq;
                    for (int x = 0; x < C::kBoxes; ++x)
                        tma_load_3d(smem + C::kOffQ + slot * C::kTileBytes + x * (kQTile * 128), &map_q, &q_full[slot], x * 64, row, bh);
                    bulk_load_1d(sStats + slot * 256, p.neg_lse2 + (long long)bh * p.Wpad + row, 512, &q_full[slot]);
                    bulk_load_1d(sStats + slot * 256 + 128, p.delta + (long long)bh * p.Wpad + row, 512, &q_full[slot]);
                    ok = mbar_wait(do_empty, (ndo & 1) ^ 1, abort_p);
                    if (!ok) break;
                    mbar_arrive_expect_tx(do_full, C::kTileBytes);
                    ++ndo;
                    for (int x = 0; x < C::kBoxes; ++x) tma_load_3d(smem + C::kOffDO + x * (kQTile * 128), &map_do, do_full, x * 64, row, bh);
                }
            }
            if (!ok && base_ok) {
                int dummy = 0;              // leave no copy in flight: the barriers armed last must complete (bounded)
                for (uint32_t back = 1; back <= 2 && back <= nq; ++back)
                    mbar_wait(&q_full[(nq - back) & 1], ((nq - back) >> 1) & 1, &dummy, 200000000LL);
                if (ndo > 0) mbar_wait(do_full, (ndo - 1) & 1, &dummy, 200000000LL);
            }
        }
    } else if (warp == C::kKv) {
        // ------------------------------------------------------------------ TMA producer: K, V of the key tiles
        if (lane == 0) {
            bool ok = base_ok;
            uint32_t nk = 0, nv = 0;        // tiles armed
            for (long long u = order.begin; u < order.end && ok; u += order.step) {
                int bh, t, bh_n, t_n;
                order.unit(p, u, bh, t);
                if (u + order.step < order.end) {   // K, V have one buffer: the next tile's rows come as far as L2 meanwhile
                    order.unit(p, u + order.step, bh_n, t_n);
                    for (int x = 0; x < C::kBoxes; ++x) {
                        tma_prefetch_l2_3d(&map_k, x * 64, t_n * kTileN, bh_n);
                        tma_prefetch_l2_3d(&map_v, x * 64, t_n * kTileN, bh_n);
                    }
                }
                ok = mbar_wait(v_empty, (nv & 1) ^ 1, abort_p);      // V is read for the last time before K is
                if (!ok) break;
                mbar_arrive_expect_tx(v_full, C::kTileBytes);
                ++nv;
                for (int x = 0; x < C::kBoxes; ++x) tma_load_3d(smem + C::kOffV + x * (kQTile * 128), &map_v, v_full, x * 64, t * kTileN, bh);
                ok = mbar_wait(k_empty, (nk & 1) ^ 1, abort_p);
                if (!ok) break;
                mbar_arrive_expect_tx(k_full, C::kTileBytes);
                ++nk;
                for (int x = 0; x < C::kBoxes; ++x) tma_load_3d(smem + C::kOffK + x * (kQTile * 128), &map_k, k_full, x * 64, t * kTileN, bh);
            }
            if (!ok && base_ok) {
                int dummy = 0;
                if (nv > 0) mbar_wait(v_full, (nv - 1) & 1, &dummy, 200000000LL);
                if (nk > 0) mbar_wait(k_full, (nk - 1) & 1, &dummy, 200000000LL);
            }
        }
    } else if (warp == C::kMma) {
        // ------------------------------------------------------------------ MMA issuer (all lanes walk, the lane elected once issues)
        const uint32_t idesc_s = make_idesc_bf16(kQTile, kQTile, 0, 0);      // S^T, dP^T: M = keys, N = 128 queries
        const uint32_t idesc_acc = make_idesc_bf16(kQTile, D, 0, 1);         // dV, dK: A in TMEM, B MN-major
        const uint32_t idesc_dqt = make_idesc_bf16(D, kQTile, 1, 1);         // dQ^T: M = d, N = 128 queries, K = keys; both MN-major
        const uint64_t kmaj = make_smem_desc_sw128(smem_u32(smem), 16, 1024);
        const uint64_t mnmaj = make_smem_desc_sw128(smem_u32(smem), kQTile * 128, 1024);   // 16 KB between 64-element column blocks
        const uint32_t desc_hi = (uint32_t)(kmaj >> 32);
        const uint32_t kmaj_lo = (uint32_t)kmaj, mnmaj_lo = (uint32_t)mnmaj;
        const uint32_t tmem_u = __shfl_sync(0xffffffffu, tmem_base, 0);
        const uint32_t tDK = tmem_u + C::kColDK, tDV = tmem_u + C::kColDV, tS = tmem_u + C::kColS, tDP = tmem_u + C::kColDP;
        const uint32_t lead = elect_one() ? 1u : 0u;
        // [keys x 128 queries] = A B^T over d, both K-major 128-row tiles
        auto issue_scores = [&](uint32_t acc, uint32_t a_off, uint32_t b_off) {
            const uint32_t a_lo = kmaj_lo + (a_off >> 4), b_lo = kmaj_lo + (b_off >> 4);
#pragma unroll
            for (int kk = 0; kk < D / 16; ++kk) {
                const uint32_t off16 = ((kk >> 2) * (kQTile * 128) + (kk & 3) * 32) >> 4;
                mma_ss_lead(lead, acc, a_lo + off16, b_lo + off16, desc_hi, idesc_s, kk > 0);
            }
        };
        // dV or dK += (bf16 [keys x 128 queries] in TMEM: 64 queries in the first 32 columns of each 64) x (128-row tile read MN-major)
        auto issue_acc = [&](uint32_t acc, uint32_t a, uint32_t b_off, bool accumulate) {
            const uint32_t b_lo = mnmaj_lo + (b_off >> 4);
#pragma unroll
            for (int kk = 0; kk < kQTile / 16; ++kk)
                mma_ts_lead(lead, acc, a + (kk >> 2) * 64 + (kk & 3) * 8, b_lo + kk * (2048 >> 4), desc_hi, idesc_acc, (accumulate || kk > 0) ? 1u : 0u);
        };
        bool ok = base_ok;
        uint32_t g = 0, n = 0;              // steps and key tiles done; step g uses Q slot g & 1
        auto wait = [&](uint64_t* bar, uint32_t parity) {
            ok = __all_sync(0xffffffffu, mbar_wait(bar, parity, abort_p));
            return ok;
        };
        for (long long u = order.begin; u < order.end && ok; u += order.step, ++n) {
            int bh, t;
            order.unit(p, u, bh, t);
            const int steps = p.q_tiles128 - first_q_tile(p, t);
            if (!wait(k_full, n & 1) || !wait(&q_full[g & 1], (g >> 1) & 1)) break;
            tc_fence_after();
            issue_scores(tS, C::kOffK, C::kOffQ + (g & 1) * C::kTileBytes);
            commit_lead(lead, s_full);
            if (!wait(v_full, n & 1) || !wait(do_full, g & 1)) break;
            if (g > 0 && !wait(dq_drained, (g - 1) & 1)) break;             // dP^T goes over the previous step's dQ^T
            tc_fence_after();
            issue_scores(tDP, C::kOffV, C::kOffDO);
            commit_lead(lead, dp_full);
            if (steps == 1) commit_lead(lead, v_empty);
            for (int s = 0; s < steps; ++s, ++g) {
                const uint32_t slot = g & 1, next = slot ^ 1, next_par = ((g + 1) >> 1) & 1;
                const bool have_next = s + 1 < steps;
                if (!wait(p_full, g & 1)) break;
                if (s == 0 && n > 0 && !wait(acc_empty, (n - 1) & 1)) break;   // the previous key tile's dK, dV must have been read out
                tc_fence_after();
                issue_acc(tDV, tS, C::kOffDO, s > 0);
                commit_lead(lead, do_empty);
                if (have_next) {
                    if (!wait(&q_full[next], next_par)) break;
                    tc_fence_after();
                    issue_scores(tS, C::kOffK, C::kOffQ + next * C::kTileBytes);
                    commit_lead(lead, s_full);
                }
                if (!wait(ds_full, g & 1)) break;
                tc_fence_after();
                issue_acc(tDK, tDP, C::kOffQ + slot * C::kTileBytes, s > 0);
                commit_lead(lead, &q_empty[slot]);
#pragma unroll
                for (int kk = 0; kk < kTileN / 16; ++kk)
                    mma_ss_lead(lead, tDP, mnmaj_lo + (C::kOffK >> 4) + kk * (2048 >> 4), mnmaj_lo + (C::kOffStage >> 4) + kk * (2048 >> 4), desc_hi, idesc_dqt, kk > 0);
                commit_lead(lead, dq_full);
                if (have_next) {
                    if (!wait(do_full, (g + 1) & 1) || !wait(dq_drained, g & 1)) break;
                    tc_fence_after();
                    issue_scores(tDP, C::kOffV, C::kOffDO);
                    commit_lead(lead, dp_full);
                    if (s + 2 == steps) commit_lead(lead, v_empty);
                } else {
                    commit_lead(lead, k_empty);
                    commit_lead(lead, acc_full);
                }
            }
        }
    }
    } else if (warp >= C::kDqWarp) {
        // ------------------------------------------------------------------ dQ^T -> fp32 dQ (reductions in L2)
        setmaxnreg_inc<C::kDqRegs>();
        const int r = (warp & 3) * 32 + lane;                  // column of dQ == TMEM lane
        const uint32_t tDQ = tmem_base + ((uint32_t)((warp & 3) * 32) << 16) + C::kColDP;
        const bool issuer = threadIdx.x == C::kDqWarp * 32;
        bool ok = base_ok;
        uint32_t g = 0;
        for (long long u = order.begin; u < order.end && ok; u += order.step) {
            int bh, t;
            order.unit(p, u, bh, t);
            for (int i = first_q_tile(p, t); i < p.q_tiles128; ++i, ++g) {
                ok = __all_sync(0xffffffffu, mbar_wait(dq_full, g & 1, abort_p));
                tc_fence_after();
                uint32_t o[4][32];                                // of no use, and not stored, when the wait has run out
#pragma unroll
                for (int c = 0; c < 4; ++c) tmem_ld32_async(tDQ + c * 32, o[c]);
#pragma unroll
                for (int c = 0; c < 4; ++c) tmem_wait_ld(o[c]);
                tc_fence_before();
                mbar_arrive(dq_drained);
                // rows of dQ (consecutive in the workspace) through shared memory, 16 at a time, added by the copy engine
                float* drow = p.ws + ((long long)bh * p.Wpad + i * kQTile) * D;
                if (issuer) bulk_wait_read<3>();                  // the first buffer's previous rows have been read
                // a wait that ran out is each warp's own finding (the phase may complete between two of them): the four warps go on,
                // or leave, together
                ok = named_barrier_all(1, 128, ok);
                if (!ok) break;
#pragma unroll
                for (int c = 0; c < kQTile / C::kDqRows; ++c) {
                    float* buf = reinterpret_cast<float*>(smem + C::kOffDQ + (c & 3) * (C::kDqRows * D * 4));
                    if (c > 0) {
                        if (issuer) bulk_wait_read<3>();          // the buffer's previous rows have been read
                        named_barrier(1, 128);
                    }
#pragma unroll
                    for (int e = 0; e < C::kDqRows; ++e) buf[e * D + r] = __uint_as_float(o[c >> 1][(c & 1) * 16 + e]);
                    fence_proxy_async_smem();
                    named_barrier(1, 128);
                    if (issuer) {
                        bulk_add_f32(drow + c * C::kDqRows * D, buf, C::kDqRows * D * 4);
                        bulk_commit();
                    }
                }
            }
        }
        if (issuer) bulk_wait_all();
    } else {
        // ------------------------------------------------------------------ P and dS
        const int wg = warp >> 2;                              // which 64 queries of every tile
        const int r = (warp & 3) * 32 + lane;                  // key row inside the tile == TMEM lane
        const uint32_t lane_addr = (uint32_t)((warp & 3) * 32) << 16;
        const uint32_t tS = tmem_base + lane_addr + C::kColS + wg * 64, tDP = tmem_base + lane_addr + C::kColDP + wg * 64;
        uint8_t* ds_row = smem + C::kOffStage + wg * 16384 + r * 128;       // this key's row of the dS^T tile
        bool ok = base_ok;
        uint32_t g = 0, n = 0;
        for (long long u = order.begin; u < order.end && ok; u += order.step, ++n) {
            int bh, t;
            order.unit(p, u, bh, t);
            const int key = t * kTileN + r;
            const long long shift = (long long)p.N - p.W;       // query q may use key k iff q >= k - shift
            const int q_min = p.causal ? (int)((long long)key - shift) : -0x7fffffff;
            const int q_min_warp = p.causal ? (int)((long long)key - lane + 31 - shift) : -0x7fffffff;   // largest in the warp
            auto step = [&](int q0, auto masked_tag) {
                constexpr bool kMasked = decltype(masked_tag)::value;
                const float* st = sStats + (g & 1) * 256 + wg * 64;
                ok = __all_sync(0xffffffffu, mbar_wait(s_full, g & 1, abort_p));
                if (!ok) return;
                // already complete (the MMAs waited for it); observing it here orders the bulk-copied neg_lse2 / delta
                // before this thread's reads
                ok = __all_sync(0xffffffffu, mbar_wait(&q_full[g & 1], (g >> 1) & 1, abort_p));
                if (!ok) return;
                tc_fence_after();
                uint32_t pe[2][32];
                tmem_ld32_async(tS, pe[0]);
                tmem_ld32_async(tS + 32, pe[1]);
                tmem_wait_ld(pe[0]);
                tmem_wait_ld(pe[1]);
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    uint32_t pk[16];
#pragma unroll
                    for (int c = 0; c < 32; c += 4) {
                        const float4 l4 = *reinterpret_cast<const float4*>(st + h * 32 + c);
                        const float lv[4] = {l4.x, l4.y, l4.z, l4.w};
                        float x[4];
#pragma unroll
                        for (int e = 0; e < 4; ++e) {
                            x[e] = ex2(fmaf(__uint_as_float(pe[h][c + e]), p.scale_log2e, lv[e]));
                            if (kMasked && q0 + h * 32 + c + e < q_min) x[e] = 0.f;
                            pe[h][c + e] = __float_as_uint(x[e]);
                        }
                        pk[c / 2] = pack_bf16x2(x[0], x[1]);
                        pk[c / 2 + 1] = pack_bf16x2(x[2], x[3]);
                    }
                    tmem_st16(tS + h * 16, pk);
                }
                tc_wait_st();
                tc_fence_before();
                mbar_arrive(p_full);
                ok = __all_sync(0xffffffffu, mbar_wait(dp_full, g & 1, abort_p));
                if (!ok) return;
                tc_fence_after();
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    uint32_t dp[32], dk_[16];
                    tmem_ld32_async(tDP + h * 32, dp);
                    tmem_wait_ld(dp);
#pragma unroll
                    for (int c = 0; c < 32; c += 4) {
                        const float4 d4 = *reinterpret_cast<const float4*>(st + 128 + h * 32 + c);
                        const float dlv[4] = {d4.x, d4.y, d4.z, d4.w};
                        float de[4];
#pragma unroll
                        for (int e = 0; e < 4; ++e) de[e] = __uint_as_float(pe[h][c + e]) * (__uint_as_float(dp[c + e]) - dlv[e]);
                        dk_[c / 2] = pack_bf16x2(de[0], de[1]);
                        dk_[c / 2 + 1] = pack_bf16x2(de[2], de[3]);
                    }
                    tmem_st16(tDP + h * 16, dk_);          // over columns of dP^T that are already in registers
                    // and once more as the B operand of the dQ^T product: row = key, 64 queries = 128 bytes, 16-byte pieces at
                    // (piece xor row mod 8), the layout the 128-byte swizzle of the descriptors expects
#pragma unroll
                    for (int c4 = 0; c4 < 4; ++c4)
                        *reinterpret_cast<uint4*>(ds_row + (((h * 4 + c4) ^ (r & 7)) << 4)) =
                            make_uint4(dk_[c4 * 4], dk_[c4 * 4 + 1], dk_[c4 * 4 + 2], dk_[c4 * 4 + 3]);
                }
                tc_wait_st();
                fence_proxy_async_smem();             // the tile was written with ordinary stores and is read by the MMA
                tc_fence_before();
                mbar_arrive(ds_full);
            };
            for (int i = first_q_tile(p, t); i < p.q_tiles128 && ok; ++i, ++g) {
                const int q0 = i * kQTile + wg * 64;              // first query of this thread's columns
                if (q0 < q_min_warp) step(q0, std::true_type{});  // warp-uniform: some element of some lane is masked
                else step(q0, std::false_type{});
            }
            if (!ok) break;
            // ---------------------------------------------------------------- dK, dV of this key tile
            ok = __all_sync(0xffffffffu, mbar_wait(acc_full, n & 1, abort_p));
            if (!ok) break;
            tc_fence_after();
            // Each thread holds half a row (D/2 columns) of dK and of dV.  Written straight from the registers a warp's store
            // would touch 32 different lines; the warp passes its 32 x D bytes through shared memory (16-byte pieces, piece
            // index xor row so that neither side has bank conflicts beyond the minimum) and stores whole lines instead.  Its
            // part of the buffer is where its own rows of dS^T go, so no other warp is in the way.
            constexpr int kPieces = D / 16;                    // 16-byte pieces per half row
            constexpr int kRowsPerStore = 32 / kPieces;
            uint8_t* stage = smem + C::kOffStage + warp * (32 * D);
            const int key_warp = t * kTileN + (warp & 3) * 32;     // key of lane 0
#pragma unroll
            for (int which = 0; which < 2; ++which) {
                const uint32_t tA = tmem_base + lane_addr + (which == 0 ? C::kColDK : C::kColDV) + wg * (D / 2);
                const float f = which == 0 ? p.scale : 1.f;
#pragma unroll
                for (int c = 0; c < D / 64; ++c) {
                    uint32_t o[32];
                    tmem_ld32(tA + c * 32, o);
#pragma unroll
                    for (int v4 = 0; v4 < 4; ++v4) {
                        uint4 w;
                        w.x = pack_bf16x2(__uint_as_float(o[v4 * 8 + 0]) * f, __uint_as_float(o[v4 * 8 + 1]) * f);
                        w.y = pack_bf16x2(__uint_as_float(o[v4 * 8 + 2]) * f, __uint_as_float(o[v4 * 8 + 3]) * f);
                        w.z = pack_bf16x2(__uint_as_float(o[v4 * 8 + 4]) * f, __uint_as_float(o[v4 * 8 + 5]) * f);
                        w.w = pack_bf16x2(__uint_as_float(o[v4 * 8 + 6]) * f, __uint_as_float(o[v4 * 8 + 7]) * f);
                        const int piece = c * 4 + v4;
                        *reinterpret_cast<uint4*>(stage + lane * D + ((piece ^ (lane & (kPieces - 1))) << 4)) = w;
                    }
                }
                if (which == 1) {                              // both accumulators have been read
                    tc_fence_before();
                    mbar_arrive(acc_empty);
                }
                __syncwarp();
                __nv_bfloat16* dst = reinterpret_cast<__nv_bfloat16*>(which == 0 ? p.dk : p.dv) +
                                     ((long long)bh * p.N + key_warp) * D + wg * (D / 2);
#pragma unroll
                for (int it = 0; it < 32 / kRowsPerStore; ++it) {
                    const int rrow = it * kRowsPerStore + lane / kPieces, piece = lane % kPieces;
                    const uint4 w = *reinterpret_cast<const uint4*>(stage + rrow * D + ((piece ^ (rrow & (kPieces - 1))) << 4));
                    if (key_warp + rrow < p.N) *reinterpret_cast<uint4*>(dst + (long long)rrow * D + piece * 8) = w;
                }
                __syncwarp();
            }
        }
    }

    tc_fence_before();
    __syncthreads();
    if (threadIdx.x == 0 && *abort_flag) atomicExch(p.status, base_ok ? (int)TLIN_ERR_TIMEOUT : (int)TLIN_ERR_CUDA);
    if (warp == C::kMma) {
        tc_fence_after();
        tmem_dealloc(tmem_base, 512);
    }
}

// ------------------------------------------------------------------------------------------ dQ
template <int D>
struct BCfg {
    static constexpr int kTileBytes = kQTile * D * 2;
    static constexpr int kBoxes = D / 64;
    static constexpr int kKSlots = D == 128 ? 2 : 4;           // K tiles live for a whole step (S, then dQ)
    static constexpr int kVSlots = D == 128 ? 1 : 2;           // V tiles only for the dP MMAs
    static constexpr int kOffQ = 0;                            // 2 tiles
    static constexpr int kOffDO = 2 * kTileBytes;              // 2 tiles
    static constexpr int kOffK = 4 * kTileBytes;
    static constexpr int kOffV = (4 + kKSlots) * kTileBytes;
    static constexpr int kOffBars = (4 + kKSlots + kVSlots) * kTileBytes;
    // Score buffers.  A step of one Q tile (item) holds one from its S to its dQ; the items take them in turn, in the order
    // (key tile, Q tile).  TMEM has room for a third at d = 64: S of a later step is then ready when a warpgroup has handed over
    // its dS.  With the TMEM reads of both kernels issued one chunk ahead: 16 x 2000^2 backward 63.3 -> 60.6 us, B4 H32 N8192 W1024
    // 1.09 -> 1.06 ms, B3 H12 1999^2 96.8 -> 95.2 us.
    static constexpr int kBufs = D == 128 ? 2 : 3;
    static constexpr int kAhead = kBufs - 1;                   // S runs at most this many key tiles ahead (K slots: these and the current one)
    static_assert(kAhead < kKSlots, "S of a later key tile would wait for the slot of the current one");
    static constexpr int kNumBars = 9 + 2 * kBufs + 2 * kKSlots + 2 * kVSlots;
    static constexpr int kSmemBytes = kOffBars + kNumBars * 8 + 32;   // + TMEM slot, abort flag, unit range
    // TMEM columns: the score buffers (S, then dP, then dS as bf16; 128 each), dQ0, dQ1 (D each)
    static constexpr uint32_t kColR = 0, kColDQ = kBufs * kTileN;
    static constexpr int kThreads = 32 * 12;                   // warps 10 and 11 only lend their registers
    // setmaxnreg moves registers between warpgroups; the CTA starts with 168 per thread (65536 / 384, rounded down to a
    // multiple of 8), and an increase beyond what the other warpgroup released would wait for ever
    static constexpr int kComputeRegs = 200, kOtherRegs = 104;
    static_assert(256 * kComputeRegs + 128 * kOtherRegs <= kThreads * 168, "register budget of the CTA exceeded");
};

template <int D, bool kDeal>
__global__ void __launch_bounds__(BCfg<D>::kThreads, 1)
bwd_dq_tc_kernel(const __grid_constant__ CUtensorMap map_q, const __grid_constant__ CUtensorMap map_k,
                 const __grid_constant__ CUtensorMap map_v, const __grid_constant__ CUtensorMap map_do, const BwdParams p,
                 const __grid_constant__ GroupStarts starts) {
    using C = BCfg<D>;
    extern __shared__ __align__(1024) uint8_t smem[];
    uint8_t* sQ = smem + C::kOffQ;
    uint8_t* sDO = smem + C::kOffDO;
    uint8_t* sK = smem + C::kOffK;
    uint8_t* sV = smem + C::kOffV;
    uint64_t* bars = reinterpret_cast<uint64_t*>(smem + C::kOffBars);
    uint64_t* qdo_full = bars + 0;
    uint64_t* qdo_empty = bars + 1;
    uint64_t* dq_done = bars + 2;
    uint64_t* p_ready = bars + 3;     // [2]  every thread of the Q tile has read S
    uint64_t* dp_full = bars + 5;     // [2]
    uint64_t* ds_full = bars + 7;     // [2]
    // [2][kBufs] by Q tile and its step mod kBufs.  S may be complete before the tile's threads have asked for the previous one, so one
    // barrier per tile would be a phase ahead; and by buffer, a warpgroup that skips a segment would ask for a phase beyond the next.
    uint64_t* s_full = bars + 9;
    uint64_t* k_full = s_full + 2 * C::kBufs;
    uint64_t* k_empty = k_full + C::kKSlots;
    uint64_t* v_full = k_empty + C::kKSlots;
    uint64_t* v_empty = v_full + C::kVSlots;
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(bars + C::kNumBars);
    int* abort_flag = reinterpret_cast<int*>(tmem_slot + 1);

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const bool base_ok = (smem_u32(smem) & 1023u) == 0;

    if (threadIdx.x == 0) {
        *abort_flag = base_ok ? 0 : 1;
        mbar_init(qdo_full, 1);
        mbar_init(qdo_empty, 1);
        mbar_init(dq_done, 1);
        for (int i = 0; i < 2; ++i) {
            mbar_init(&p_ready[i], kQTile);
            mbar_init(&dp_full[i], 1);
            mbar_init(&ds_full[i], kQTile);
        }
        for (int s = 0; s < 2 * C::kBufs; ++s) mbar_init(&s_full[s], 1);
        for (int s = 0; s < C::kKSlots; ++s) {
            mbar_init(&k_full[s], 1);
            mbar_init(&k_empty[s], 1);
        }
        for (int s = 0; s < C::kVSlots; ++s) {
            mbar_init(&v_full[s], 1);
            mbar_init(&v_empty[s], 1);
        }
        fence_mbar_init();
    }
    if (warp == kMmaWarp) {
        tmem_alloc(tmem_slot, 512);
        tmem_relinquish();
    }
    if (warp == kProducerWarp && lane == 0) {
        prefetch_tensormap(&map_q);
        prefetch_tensormap(&map_k);
        prefetch_tensormap(&map_v);
        prefetch_tensormap(&map_do);
    }
    tc_fence_before();
    after_previous();
    let_next_start();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem_base = *tmem_slot;
    volatile int* abort_p = abort_flag;

    if (warp >= 8) {
    setmaxnreg_dec<C::kOtherRegs>();
    if (warp == kProducerWarp) {
        // ------------------------------------------------------------------ TMA producer
        if (lane == 0) {
            uint32_t kit = 0, vit = 0, seg_idx = 0;
            bool ok = base_ok;
            std::conditional_t<kDeal, DealtWalker, SegmentWalker> walk(p, starts);
            Segment s;
            while (ok && walk.next(s)) {
                const int row0 = s.qt * kTileM;
                const int c0 = seg_count(s, tiles_allowed(p, row0, 0)), c1 = seg_count(s, tiles_allowed(p, row0, 1));
                const int cnt = c0 > c1 ? c0 : c1;
                if (cnt == 0) continue;
                if (seg_idx > 0) ok = mbar_wait(qdo_empty, (seg_idx - 1) & 1, abort_p);
                if (!ok) break;
                mbar_arrive_expect_tx(qdo_full, 4 * C::kTileBytes);
                for (int i = 0; i < 2; ++i)
                    for (int x = 0; x < C::kBoxes; ++x) {
                        tma_load_3d(sQ + i * C::kTileBytes + x * (kQTile * 128), &map_q, qdo_full, x * 64, row0 + i * kQTile, s.bh);
                        tma_load_3d(sDO + i * C::kTileBytes + x * (kQTile * 128), &map_do, qdo_full, x * 64, row0 + i * kQTile, s.bh);
                    }
                for (int j = 0; j < cnt && ok; ++j) {
                    const int t = s.t_begin + j;
                    {
                        const uint32_t slot = kit % C::kKSlots, round = kit / C::kKSlots;
                        ok = mbar_wait(&k_empty[slot], (round & 1) ^ 1, abort_p);
                        if (!ok) break;
                        mbar_arrive_expect_tx(&k_full[slot], C::kTileBytes);
                        for (int x = 0; x < C::kBoxes; ++x)
                            tma_load_3d(sK + slot * C::kTileBytes + x * (kQTile * 128), &map_k, &k_full[slot], x * 64, t * kTileN, s.bh);
                        ++kit;
                    }
                    {
                        const uint32_t slot = vit % C::kVSlots, round = vit / C::kVSlots;
                        ok = mbar_wait(&v_empty[slot], (round & 1) ^ 1, abort_p);
                        if (!ok) break;
                        mbar_arrive_expect_tx(&v_full[slot], C::kTileBytes);
                        for (int x = 0; x < C::kBoxes; ++x)
                            tma_load_3d(sV + slot * C::kTileBytes + x * (kQTile * 128), &map_v, &v_full[slot], x * 64, t * kTileN, s.bh);
                        ++vit;
                    }
                }
                ++seg_idx;
            }
            if (!ok && base_ok) {
                int dummy = 0;          // leave no copy in flight: what was armed last must land (bounded)
                for (uint32_t back = 0; back < (uint32_t)C::kKSlots && back < kit; ++back) {
                    const uint32_t id = kit - 1 - back;
                    mbar_wait(&k_full[id % C::kKSlots], (id / C::kKSlots) & 1, &dummy, 200000000LL);
                }
                for (uint32_t back = 0; back < (uint32_t)C::kVSlots && back < vit; ++back) {
                    const uint32_t id = vit - 1 - back;
                    mbar_wait(&v_full[id % C::kVSlots], (id / C::kVSlots) & 1, &dummy, 200000000LL);
                }
                if (seg_idx > 0) mbar_wait(qdo_full, (seg_idx - 1) & 1, &dummy, 200000000LL);
            }
        }
    } else if (warp == kMmaWarp) {
        // ------------------------------------------------------------------ MMA issuer (all lanes walk, the lane elected once issues)
        const uint32_t idesc_s = make_idesc_bf16(kQTile, kTileN, 0, 0);      // S, dP: M = queries, N = keys
        const uint32_t idesc_dq = make_idesc_bf16(kQTile, D, 0, 1);          // dQ: A = dS in TMEM, B = K MN-major
        const uint64_t kmaj = make_smem_desc_sw128(smem_u32(smem), 16, 1024);
        const uint64_t mnmaj = make_smem_desc_sw128(smem_u32(smem), kQTile * 128, 1024);
        const uint32_t desc_hi = (uint32_t)(kmaj >> 32);
        const uint32_t kmaj_lo = (uint32_t)kmaj, mnmaj_lo = (uint32_t)mnmaj;
        const uint32_t tmem_u = __shfl_sync(0xffffffffu, tmem_base, 0);
        const uint32_t lead = elect_one() ? 1u : 0u;
        auto issue_r = [&](int buf, int a_byte_off, int b_byte_off) {        // R_buf = A B^T (contraction over d)
            const uint32_t a_lo = kmaj_lo + (uint32_t)(a_byte_off >> 4), b_lo = kmaj_lo + (uint32_t)(b_byte_off >> 4);
            const uint32_t d = tmem_u + C::kColR + buf * kTileN;
#pragma unroll
            for (int kk = 0; kk < D / 16; ++kk) {
                const uint32_t off16 = ((kk >> 2) * (kQTile * 128) + (kk & 3) * 32) >> 4;
                mma_ss_lead(lead, d, a_lo + off16, b_lo + off16, desc_hi, idesc_s, kk > 0);
            }
        };
        auto issue_dq = [&](int i, int buf, int k_byte_off, bool accumulate) {       // dQ_i += dS_i K (contraction over keys)
            const uint32_t b_lo = mnmaj_lo + (uint32_t)(k_byte_off >> 4);
            const uint32_t d = tmem_u + C::kColDQ + i * D, a = tmem_u + C::kColR + buf * kTileN;
#pragma unroll
            for (int kk = 0; kk < kTileN / 16; ++kk)
                mma_ts_lead(lead, d, a + kk * 8, b_lo + kk * (2048 >> 4), desc_hi, idesc_dq, (accumulate || kk > 0) ? 1u : 0u);
        };
        uint32_t kit = 0, vit = 0, seg_idx = 0;                             // kit: first key tile of the segment, in the order of loading
        uint32_t n_step[2] = {0, 0};
        uint32_t s_item = 0, r_item = 0, q_item = 0;                        // items whose S, dP, dQ have been issued
        uint32_t s_step[2] = {0, 0};                                        // per Q tile: steps whose S has been issued
        bool ok = base_ok;
        std::conditional_t<kDeal, DealtWalker, SegmentWalker> walk(p, starts);
        Segment s;
        while (ok && walk.next(s)) {
            const int row0 = s.qt * kTileM;
            const int c0 = seg_count(s, tiles_allowed(p, row0, 0)), c1 = seg_count(s, tiles_allowed(p, row0, 1));
            const int cnt = c0 > c1 ? c0 : c1;
            if (cnt == 0) continue;
            const int cq[2] = {c0, c1};
            ok = __all_sync(0xffffffffu, mbar_wait(qdo_full, seg_idx & 1, abort_p));
            if (!ok) break;
            int js = 0, is = c0 > 0 ? 0 : 1, k_seen = 0;                    // next item to get its S; key tiles known to have arrived
            // S of the next items, as far as buffers are free and K tiles up to j_most
            auto issue_s = [&](int j_most) {
                while (js < cnt && js <= j_most && s_item - q_item < (uint32_t)C::kBufs) {
                    const uint32_t kt = kit + js, slot = kt % C::kKSlots, buf = s_item % C::kBufs;
                    if (js >= k_seen) {
                        ok = __all_sync(0xffffffffu, mbar_wait(&k_full[slot], (kt / C::kKSlots) & 1, abort_p));
                        if (!ok) return;
                        k_seen = js + 1;
                    }
                    tc_fence_after();
                    issue_r(buf, C::kOffQ + is * C::kTileBytes, C::kOffK + slot * C::kTileBytes);
                    commit_lead(lead, is == 0 ? &s_full[s_step[0]++ % C::kBufs] : &s_full[C::kBufs + s_step[1]++ % C::kBufs]);
                    ++s_item;
                    do {
                        if (++is == 2) is = 0, ++js;
                    } while (js < cnt && js >= (is == 0 ? c0 : c1));
                }
            };
            issue_s(C::kAhead);
            for (int j = 0; j < cnt && ok; ++j) {
                const uint32_t vs = vit % C::kVSlots;
                ok = __all_sync(0xffffffffu, mbar_wait(&v_full[vs], (vit / C::kVSlots) & 1, abort_p));
                if (!ok) break;
                ++vit;
                for (int i = 0; i < 2 && ok; ++i) {
                    if (j < cq[i]) {
                        ok = __all_sync(0xffffffffu, mbar_wait(&p_ready[i], n_step[i] & 1, abort_p));
                        if (!ok) break;
                        tc_fence_after();
                        issue_r(r_item % C::kBufs, C::kOffDO + i * C::kTileBytes, C::kOffV + vs * C::kTileBytes);   // dP over S
                        commit_lead(lead, &dp_full[i]);
                        ++r_item;
                    }
                }
                if (!ok) break;
                commit_lead(lead, &v_empty[vs]);
                if (j + 1 == cnt) commit_lead(lead, qdo_empty);     // Q and dout of this segment have been read for the last time
                const uint32_t ks = (kit + j) % C::kKSlots;
                for (int i = 0; i < 2 && ok; ++i) {
                    if (j < cq[i]) {
                        ok = __all_sync(0xffffffffu, mbar_wait(&ds_full[i], n_step[i] & 1, abort_p));
                        if (!ok) break;
                        tc_fence_after();
                        issue_dq(i, q_item % C::kBufs, C::kOffK + ks * C::kTileBytes, j > 0);
                        ++n_step[i];
                        ++q_item;
                        issue_s(j + C::kAhead);
                    }
                }
                if (!ok) break;
                commit_lead(lead, &k_empty[ks]);
            }
            if (!ok) break;
            kit += cnt;
            commit_lead(lead, dq_done);
            ++seg_idx;
        }
    }
    } else {
        // ------------------------------------------------------------------ elementwise warpgroups (one per Q tile)
        setmaxnreg_inc<C::kComputeRegs>();
        const int i = warp >> 2;
        const int r = (warp & 3) * 32 + lane;
        const uint32_t lane_addr = (uint32_t)((warp & 3) * 32) << 16;
        const uint32_t tScores = tmem_base + lane_addr + C::kColR;
        const uint32_t tDQ = tmem_base + lane_addr + C::kColDQ + i * D;
        uint32_t n = 0, seg_idx = 0, items = 0;               // items of the segments before
        bool ok = base_ok;
        std::conditional_t<kDeal, DealtWalker, SegmentWalker> walk(p, starts);
        int bh_first = 0;                                     // (b,h) of this CTA's first unit (used under schedule 0 only)
        if constexpr (!kDeal) bh_first = (int)(walk.u / p.key_tiles);
        Segment s;
        while (ok && walk.next(s)) {
            const int row0 = s.qt * kTileM;
            const int row = row0 + i * kQTile + r;
            const int a0 = tiles_allowed(p, row0, 0), a1 = tiles_allowed(p, row0, 1);
            const int c0 = seg_count(s, a0), c1 = seg_count(s, a1);
            // No tile of the segment is visible to either Q tile: the MMA warp and the producer skip it and it takes no
            // barrier phase, but its partial slot is still read by the reduce kernel and has to hold zeros.
            const bool skipped = (c0 > c1 ? c0 : c1) == 0;
            const int allowed_i = i == 0 ? a0 : a1, cnt_i = i == 0 ? c0 : c1;
            const long long lim_row_ll = p.causal ? (long long)p.N - p.W + row + 1 : (long long)p.N;
            const int lim_row = (int)(lim_row_ll < p.N ? lim_row_ll : p.N);
            const long long lim_warp_ll = p.causal ? (long long)p.N - p.W + (row - lane) + 1 : (long long)p.N;
            const int lim_warp = (int)(lim_warp_ll < p.N ? lim_warp_ll : p.N);
            const bool row_ok = row < p.W;
            const float l2 = row_ok ? p.neg_lse2[(long long)s.bh * p.Wpad + row] : -CUDART_INF_F;
            const float dl = row_ok ? p.delta[(long long)s.bh * p.Wpad + row] : 0.f;
            const uint64_t l22 = f2_pack(l2, l2), dl2 = f2_pack(dl, dl), scale2 = f2_pack(p.scale_log2e, p.scale_log2e);
            // a copy of the step for the tiles with masked columns (the last ones of a segment)
            auto step = [&](int j, auto masked_tag) {
                constexpr bool kMasked = decltype(masked_tag)::value;
                const uint32_t item = items + (j < c0 ? j + (uint32_t)i : c0) + (j < c1 ? j : c1);
                const uint32_t tR = tScores + (item % C::kBufs) * kTileN;
                ok = __all_sync(0xffffffffu, mbar_wait(&s_full[i * C::kBufs + n % C::kBufs], (n / C::kBufs) & 1, abort_p));
                if (!ok) return;
                tc_fence_after();
                const int nvalid = lim_row - (s.t_begin + j) * kTileN;
                uint32_t sv[kTileN / 32][32];
#pragma unroll
                for (int c = 0; c < kTileN / 32; ++c) tmem_ld32_async(tR + c * 32, sv[c]);
#pragma unroll
                for (int c = 0; c < kTileN / 32; ++c) tmem_wait_ld(sv[c]);
                tc_fence_before();
                mbar_arrive(&p_ready[i]);                      // S is in registers: dP may overwrite it
                // p = 2^(s*scale*log2e - lse*log2e), kept as fp32 in the registers that held s
#pragma unroll
                for (int e = 0; e < kTileN; e += 2) {
                    float p0, p1;
                    f2_unpack(f2_fma(f2_pack_bits(sv[e >> 5][e & 31], sv[e >> 5][(e & 31) + 1]), scale2, l22), p0, p1);
                    p0 = ex2(p0);
                    p1 = ex2(p1);
                    if (kMasked && e >= nvalid) p0 = 0.f;
                    if (kMasked && e + 1 >= nvalid) p1 = 0.f;
                    sv[e >> 5][e & 31] = __float_as_uint(p0);
                    sv[e >> 5][(e & 31) + 1] = __float_as_uint(p1);
                }
                ok = __all_sync(0xffffffffu, mbar_wait(&dp_full[i], n & 1, abort_p));
                if (!ok) return;
                tc_fence_after();
                uint32_t dpb[2][16];
                tmem_ld16_async(tR, dpb[0]);
#pragma unroll
                for (int c = 0; c < kTileN / 16; ++c) {
                    uint32_t (&dp)[16] = dpb[c & 1];
                    tmem_wait_ld16(dp);
                    if (c + 1 < kTileN / 16) tmem_ld16_async(tR + (c + 1) * 16, dpb[(c + 1) & 1]);   // in flight during the arithmetic
                    uint32_t pk[8];
#pragma unroll
                    for (int e = 0; e < 8; ++e) {
                        const uint64_t p2 = f2_pack_bits(sv[c >> 1][(c & 1) * 16 + 2 * e], sv[c >> 1][(c & 1) * 16 + 2 * e + 1]);
                        float d0, d1;
                        f2_unpack(f2_mul(p2, f2_sub(f2_pack_bits(dp[2 * e], dp[2 * e + 1]), dl2)), d0, d1);
                        pk[e] = pack_bf16x2(d0, d1);
                    }
                    tmem_st8(tR + c * 8, pk);                 // bf16 dS over columns of dP that are already in registers
                }
                tc_wait_st();
                tc_fence_before();
                mbar_arrive(&ds_full[i]);
                ++n;
            };
            int n_open = lim_warp / kTileN - s.t_begin;            // steps before the first one with a masked column
            n_open = n_open < 0 ? 0 : (n_open < cnt_i ? n_open : cnt_i);
            int j = 0;
            for (; j < n_open && ok; ++j) step(j, std::false_type{});
            for (; j < cnt_i && ok; ++j) step(j, std::true_type{});
            if (!ok) break;
            items += c0 + c1;
            const uint32_t my_seg = seg_idx;
            if (!skipped) ++seg_idx;
            if (allowed_i == 0) continue;                      // this Q tile does not exist
            // ---------------------------------------------------------------- dQ of the segment
            if (cnt_i > 0) {
                ok = __all_sync(0xffffffffu, mbar_wait(dq_done, my_seg & 1, abort_p));
                if (!ok) break;
                tc_fence_after();
            }
            const bool whole = s.t_begin == 0 && s.t_end == p.key_tiles;
            __nv_bfloat16* drow = reinterpret_cast<__nv_bfloat16*>(p.dq) + ((long long)s.bh * p.W + row) * D;
            // partial sum -> workspace slot (0: first segment of this CTA's range, 1: a later one); unscaled fp32
            float* prow = p.ws + ((long long)blockIdx.x * 2 + (s.bh == bh_first ? 0 : 1)) * (long long)kTileM * D + (long long)(i * kQTile + r) * D;
            const float f = whole ? p.scale : 1.f;
#pragma unroll 1
            for (int c = 0; c < D / 16; ++c) {
                uint32_t o[16];
                if (cnt_i > 0) {
                    tmem_ld16_async(tDQ + c * 16, o);
                    tmem_wait_ld16(o);
                } else {
#pragma unroll
                    for (int e = 0; e < 16; ++e) o[e] = 0u;
                }
                // a thread holds one row: 32-byte stores halve the number of (scattered) store instructions
                // (taken when dq and the workspace are 32-byte aligned; the interface only promises 16)
                if (whole) {
                    if (row_ok) {
                        uint32_t w[8];
#pragma unroll
                        for (int e = 0; e < 8; ++e) w[e] = pack_bf16x2(__uint_as_float(o[2 * e]) * f, __uint_as_float(o[2 * e + 1]) * f);
                        if (p.wide_stores) {
                            st_global_v8(drow + c * 16, w[0], w[1], w[2], w[3], w[4], w[5], w[6], w[7]);
                        } else {
                            *reinterpret_cast<uint4*>(drow + c * 16) = make_uint4(w[0], w[1], w[2], w[3]);
                            *reinterpret_cast<uint4*>(drow + c * 16 + 8) = make_uint4(w[4], w[5], w[6], w[7]);
                        }
                    }
                } else if (p.wide_stores) {
                    st_global_v8(prow + c * 16, o[0], o[1], o[2], o[3], o[4], o[5], o[6], o[7]);
                    st_global_v8(prow + c * 16 + 8, o[8], o[9], o[10], o[11], o[12], o[13], o[14], o[15]);
                } else {
#pragma unroll
                    for (int v4 = 0; v4 < 4; ++v4)
                        *reinterpret_cast<uint4*>(prow + c * 16 + v4 * 4) = make_uint4(o[v4 * 4], o[v4 * 4 + 1], o[v4 * 4 + 2], o[v4 * 4 + 3]);
                }
            }
            tc_fence_before();
        }
    }

    tc_fence_before();
    __syncthreads();
    if (threadIdx.x == 0 && *abort_flag) atomicExch(p.status, base_ok ? (int)TLIN_ERR_TIMEOUT : (int)TLIN_ERR_CUDA);
    if (warp == kMmaWarp) {
        tc_fence_after();
        tmem_dealloc(tmem_base, 512);
    }
}

// Adds the partial dQ of every (b,h) whose key tiles were split between groups, scales and rounds to bf16.
// One CTA per 8 query rows of a (b,h, 256-row tile): one warp per row.
template <int D>
__global__ void __launch_bounds__(256)
bwd_dq_reduce_kernel(const BwdParams p) {
    after_previous();
    let_next_start();
    constexpr int CPL = D / 32;
    const int blocks_per_tile = kTileM / 8;
    const int part = blockIdx.x % blocks_per_tile;
    const int tile_id = blockIdx.x / blocks_per_tile;       // bh * q_tiles + qt
    const int bh = tile_id / p.q_tiles, qt = tile_id - bh * p.q_tiles;
    const unsigned long long T = (unsigned long long)p.key_tiles, U = (unsigned long long)p.total_units, G = (unsigned)p.n_groups;
    // groups holding the first and the last unit of this (b,h): largest g with floor(g*U/G) <= x
    const unsigned long long x0 = (unsigned long long)bh * T, x1 = x0 + T - 1;
    const int g_lo = (int)(((x0 + 1) * G - 1) / U), g_hi = (int)(((x1 + 1) * G - 1) / U);
    if (g_hi == g_lo) return;                               // written directly by the dQ kernel
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int rr = part * 8 + warp;
    const int row = qt * kTileM + rr;
    if (row >= p.W) return;
    float acc[CPL];
#pragma unroll
    for (int e = 0; e < CPL; ++e) acc[e] = 0.f;
    for (int g = g_lo; g <= g_hi; ++g) {
        const int cta = g * p.q_tiles + qt;
        const int slot = bh == (int)((((unsigned long long)g * U) / G) / T) ? 0 : 1;
        const float* src = p.ws + ((long long)cta * 2 + slot) * (long long)kTileM * D + (long long)rr * D + lane * CPL;
#pragma unroll
        for (int e = 0; e < CPL; ++e) acc[e] += src[e];
    }
    __nv_bfloat16* dst = reinterpret_cast<__nv_bfloat16*>(p.dq) + ((long long)bh * p.W + row) * D + lane * CPL;
#pragma unroll
    for (int e = 0; e < CPL; e += 2)
        *reinterpret_cast<uint32_t*>(dst + e) = pack_bf16x2(acc[e] * p.scale, acc[e + 1] * p.scale);
}

// ------------------------------------------------------------------------------------------ host side
template <int D>
int launch_d(const void* q, const void* k, const void* v, const void* out, const float* lse, const void* dout,
             void* dq, void* dk, void* dv, int B, int H, int N, int W, int causal, const tlin_fwd_plan& plan,
             float* ws, int num_sms, cudaStream_t st) {
    const long long bh = (long long)B * H;
    const int Wpad = (W + kQTile - 1) / kQTile * kQTile;
    CUtensorMap mq, mk, mv, mdo, mq64, mdo64;
    int rc = make_map(&mq, q, D, W, bh);
    if (rc == TLIN_OK) rc = make_map(&mk, k, D, N, bh);
    if (rc == TLIN_OK) rc = make_map(&mv, v, D, N, bh);
    if (rc == TLIN_OK) rc = make_map(&mdo, dout, D, W, bh);
    if (rc == TLIN_OK) rc = make_map(&mq64, q, D, W, bh, 64);
    if (rc == TLIN_OK) rc = make_map(&mdo64, dout, D, W, bh, 64);
    if (rc != TLIN_OK) return rc;
    BwdParams p;
    float* neg_lse2 = ws;
    float* delta = ws + bh * Wpad;
    p.neg_lse2 = neg_lse2; p.delta = delta; p.dq = dq; p.dk = dk; p.dv = dv;
    p.ws = ws + 2 * bh * Wpad;
    p.status = status_word();
    if (!p.status) return TLIN_ERR_CUDA;
    p.key_tiles = (N + kTileN - 1) / kTileN;
    p.q_tiles128 = Wpad / kQTile;
    p.N = N; p.W = W; p.Wpad = Wpad; p.causal = causal;
    p.scale = 1.f / sqrtf((float)D);
    p.scale_log2e = kLog2e * p.scale;
    p.wide_stores = ((reinterpret_cast<uintptr_t>(dq) | reinterpret_cast<uintptr_t>(ws)) & 31u) == 0;
    static bool smem_allowed[4][64] = {};
    TLIN_CUDA_CHECK(allow_dynamic_smem(bwd_dkdv_tc_kernel<D, kUnitRuns>, ACfg<D>::kSmemBytes, smem_allowed[0]));
    TLIN_CUDA_CHECK(allow_dynamic_smem(bwd_dkdv_tc_kernel<D, kUnitDealt>, ACfg<D>::kSmemBytes, smem_allowed[1]));
    TLIN_CUDA_CHECK(allow_dynamic_smem(bwd_dq_tc_kernel<D, false>, BCfg<D>::kSmemBytes, smem_allowed[2]));
    TLIN_CUDA_CHECK(allow_dynamic_smem(bwd_dq_tc_kernel<D, true>, BCfg<D>::kSmemBytes, smem_allowed[3]));
    const long long rows_padded = bh * Wpad;
    TLIN_CUDA_CHECK(launch_overlapped(bwd_prep_kernel<D>, (unsigned)((rows_padded + prep_rows_per_block<D>() - 1) / prep_rows_per_block<D>()), 256, 0, st,
        (const __nv_bfloat16*)out, (const __nv_bfloat16*)dout, lse, neg_lse2, delta, (float*)nullptr, W, Wpad, rows_padded));
    // dK, dV: the units are (b,h,key tile); a CTA takes a contiguous run of them
    BwdParams pa = p;
    pa.total_units = bh * p.key_tiles;
    pa.n_groups = 0; pa.q_tiles = 0; pa.schedule = 0;
    const auto kernel_a = deal_units(bh, N, W, causal, p.key_tiles, bh * (long long)W * D * 4, num_sms) ? bwd_dkdv_tc_kernel<D, kUnitDealt> : bwd_dkdv_tc_kernel<D, kUnitRuns>;
    const long long ctas_a = pa.total_units < num_sms ? pa.total_units : num_sms;
    TLIN_CUDA_CHECK(launch_overlapped(kernel_a, (unsigned)ctas_a, ACfg<D>::kThreads, ACfg<D>::kSmemBytes, st, mq64, mk, mv, mdo64, pa));
    // dQ: the forward's plan
    BwdParams pb = p;
    pb.total_units = plan.total_units; pb.n_groups = plan.n_groups; pb.q_tiles = plan.q_tiles; pb.schedule = plan.schedule;
    if (plan.n_groups > kMaxGroups) return TLIN_ERR_UNSUPPORTED;
    GroupStarts starts;
    fwd_group_starts(plan, &starts);
    TLIN_CUDA_CHECK(launch_overlapped(dealt(plan, bh, D) ? bwd_dq_tc_kernel<D, true> : bwd_dq_tc_kernel<D, false>, plan.n_ctas, BCfg<D>::kThreads, BCfg<D>::kSmemBytes, st, mq, mk, mv, mdo, pb, starts));
    count_launch(3);
    if (plan.uses_workspace) {
        TLIN_CUDA_CHECK(launch_overlapped(bwd_dq_reduce_kernel<D>, (unsigned)(bh * plan.q_tiles * (kTileM / 8)), 256, 0, st, pb));
        count_launch();
    }
    return TLIN_OK;
}

// fp32 dQ sums (rows padded to 128 per (b,h)) -> scaled bf16 dQ; 8 elements per thread
template <int D>
__global__ void __launch_bounds__(256)
bwd_dq_convert_kernel(const float* dq32, __nv_bfloat16* dq, int W, int Wpad, long long rows, float scale) {
    after_previous();
    let_next_start();
    constexpr int TPR = D / 8;              // threads per row
    const long long idx = (long long)blockIdx.x * 256 + threadIdx.x;
    const long long row = idx / TPR;
    const int piece = (int)(idx - row * TPR);
    if (row >= rows) return;
    const long long bh = row / W;
    const int i = (int)(row - bh * W);
    const float4* src = reinterpret_cast<const float4*>(dq32 + (bh * Wpad + i) * D + piece * 8);
    const float4 a = src[0], b = src[1];
    uint4 w;
    w.x = pack_bf16x2(a.x * scale, a.y * scale);
    w.y = pack_bf16x2(a.z * scale, a.w * scale);
    w.z = pack_bf16x2(b.x * scale, b.y * scale);
    w.w = pack_bf16x2(b.z * scale, b.w * scale);
    *reinterpret_cast<uint4*>(dq + row * D + piece * 8) = w;
}

// One kernel for dK, dV and dQ (five matrix products per pair; dQ summed in fp32 by reductions in L2, then rounded).
int launch_fused_128(const void* q, const void* k, const void* v, const void* out, const float* lse, const void* dout,
                     void* dq, void* dk, void* dv, int B, int H, int N, int W, int causal, float* ws, int num_sms, cudaStream_t st) {
    constexpr int D = 128;
    const long long bh = (long long)B * H;
    const int Wpad = (W + kQTile - 1) / kQTile * kQTile;
    CUtensorMap mk, mv, mq, mdo;
    int rc = make_map(&mk, k, D, N, bh);
    if (rc == TLIN_OK) rc = make_map(&mv, v, D, N, bh);
    if (rc == TLIN_OK) rc = make_map(&mq, q, D, W, bh);
    if (rc == TLIN_OK) rc = make_map(&mdo, dout, D, W, bh);
    if (rc != TLIN_OK) return rc;
    BwdParams p;
    float* neg_lse2 = ws;
    float* delta = ws + bh * Wpad;
    float* dq32 = ws + 2 * bh * Wpad;
    p.neg_lse2 = neg_lse2; p.delta = delta; p.dq = dq; p.dk = dk; p.dv = dv;
    p.ws = dq32;
    p.status = status_word();
    if (!p.status) return TLIN_ERR_CUDA;
    p.key_tiles = (N + kTileN - 1) / kTileN;
    p.q_tiles128 = Wpad / kQTile;
    p.N = N; p.W = W; p.Wpad = Wpad; p.causal = causal;
    p.scale = 1.f / sqrtf((float)D);
    p.scale_log2e = kLog2e * p.scale;
    p.wide_stores = 0;
    p.total_units = bh * p.key_tiles;
    p.n_groups = 0; p.q_tiles = 0; p.schedule = 0;
    const auto kernel = deal_units(bh, N, W, causal, p.key_tiles, bh * (long long)Wpad * D * 8, num_sms) ? bwd_fused_tc_kernel<D, kUnitDealt> : bwd_fused_tc_kernel<D, kUnitTurns>;
    static bool smem_allowed[2][64] = {};
    TLIN_CUDA_CHECK(allow_dynamic_smem(bwd_fused_tc_kernel<D, kUnitTurns>, FCfg<D>::kSmemBytes, smem_allowed[0]));
    TLIN_CUDA_CHECK(allow_dynamic_smem(bwd_fused_tc_kernel<D, kUnitDealt>, FCfg<D>::kSmemBytes, smem_allowed[1]));
    const long long rows_padded = bh * Wpad;
    TLIN_CUDA_CHECK(launch_overlapped(bwd_prep_kernel<D>, (unsigned)((rows_padded + prep_rows_per_block<D>() - 1) / prep_rows_per_block<D>()), 256, 0, st,
        (const __nv_bfloat16*)out, (const __nv_bfloat16*)dout, lse, neg_lse2, delta, dq32, W, Wpad, rows_padded));
    const long long ctas = p.total_units < num_sms ? p.total_units : num_sms;
    TLIN_CUDA_CHECK(launch_overlapped(kernel, (unsigned)ctas, FCfg<D>::kThreads, FCfg<D>::kSmemBytes, st, mq, mk, mv, mdo, p));
    const long long rows = bh * W, threads = rows * (D / 8);
    TLIN_CUDA_CHECK(launch_overlapped(bwd_dq_convert_kernel<D>, (unsigned)((threads + 255) / 256), 256, 0, st, dq32, (__nv_bfloat16*)dq, W, Wpad, rows, p.scale));
    count_launch(3);
    return TLIN_OK;
}

}  // namespace

// row statistics (neg_lse2, delta, padded) + the fp32 dQ sums, rows padded to 128 per (b,h)
size_t bwd_fused_workspace_bytes(long long B, long long H, long long W, int d) {
    const long long bh = B * H, Wpad = (W + tc::kQTile - 1) / tc::kQTile * tc::kQTile;
    return (size_t)(2 * bh * Wpad + bh * Wpad * d) * sizeof(float);
}

int launch_bwd_fused(const void* q, const void* k, const void* v, const void* out, const float* lse, const void* dout,
                     void* dq, void* dk, void* dv, int B, int H, int N, int W, int d, int causal, float* ws, int num_sms, cudaStream_t st) {
    if (d != 128) return TLIN_ERR_UNSUPPORTED;
    if ((long long)B * H * W > 0x7fffffffLL || (long long)B * H > 0x7fffffffLL || (long long)B * H * ((N + kTileN - 1LL) / kTileN) > 0x7fff0000LL) return TLIN_ERR_UNSUPPORTED;
    return launch_fused_128(q, k, v, out, lse, dout, dq, dk, dv, B, H, N, W, causal, ws, num_sms, st);
}

// row statistics (neg_lse2, delta, padded) + the dQ kernel's partial slots
size_t bwd_tc_workspace_bytes(long long B, long long H, long long W, int d, const tlin_fwd_plan& plan) {
    const long long bh = B * H, Wpad = (W + tc::kQTile - 1) / tc::kQTile * tc::kQTile;
    long long floats = 2 * bh * Wpad;
    if (plan.uses_workspace) floats += (long long)plan.n_ctas * 2 * tc::kTileM * d;
    return (size_t)floats * sizeof(float);
}

int launch_bwd_tc(const void* q, const void* k, const void* v, const void* out, const float* lse, const void* dout,
                  void* dq, void* dk, void* dv, int B, int H, int N, int W, int d, int causal, const tlin_fwd_plan& plan,
                  float* ws, int num_sms, cudaStream_t st) {
    if (plan.tile_m != tc::kTileM || plan.tile_n != kTileN || !plan.tensor_path) return TLIN_ERR_UNSUPPORTED;
    if ((long long)B * H * W > 0x7fffffffLL || (long long)B * H > 0x7fffffffLL || (long long)B * H * ((N + kTileN - 1LL) / kTileN) > 0x7fff0000LL) return TLIN_ERR_UNSUPPORTED;
    if (d == 128) return launch_d<128>(q, k, v, out, lse, dout, dq, dk, dv, B, H, N, W, causal, plan, ws, num_sms, st);
    if (d == 64) return launch_d<64>(q, k, v, out, lse, dout, dq, dk, dv, B, H, N, W, causal, plan, ws, num_sms, st);
    return TLIN_ERR_UNSUPPORTED;
}

}  // namespace tlin

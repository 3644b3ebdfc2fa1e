// Tensor-core forward kernel for sm_100a: exact softmax attention of W queries over N keys
// (Section 3 attention formula; causal rule j <= N-W+i inside the window), bf16 in, fp32 accumulate.
//
// One CTA owns 256 query rows of one (b,h) (two 128-row Q tiles) and streams a contiguous range of
// 128-key tiles.  K and V tiles arrive by TMA (128-byte swizzle) into a shared-memory ring; one thread
// issues tcgen05.mma: S_i = Q_i K_j^T into TMEM, then O_i += P_i V_j with P_i read from TMEM and V_j
// as an MN-major shared-memory operand.  Two softmax warpgroups (one per Q tile, one thread per row)
// read a whole row of S_i from TMEM into registers once, keep a running max / sum in base-2 units, write
// P_i (bf16) over S_i, and rescale O_i only when the running max has grown by more than 2^32 (the final
// O/l is exact either way).  A fixed share of the exponentials is evaluated by a cubic on the FMA pipe,
// the rest by the special-function unit, so that neither pipe alone bounds the softmax.
// While one warpgroup does its exponentials the tensor pipe works on the other Q tile.
//
// CTAs are numbered group*q_tiles + q_tile: the q_tiles CTAs of a group walk the same (b,h,key-tile)
// units at the same time, so K/V tiles are fetched from HBM once and re-read from L2.  A group's unit
// range may start or end in the middle of a (b,h); such partial results (normalised o, lse) go to the
// workspace and fwd_merge_kernel combines them with log-sum-exp weights.  Few, short problems are merged inside
// clusters instead (kCluster).
//
// Every wait is bounded: on expiry the CTA sets the library's error word, drains and exits.
#include "tlin_internal.h"
#include "sm100_ptx.cuh"
#include "tc_common.cuh"
#include <atomic>
#include <cooperative_groups.h>
#include <float.h>
#include <math_constants.h>
#include <mutex>
#include <string.h>
#include <type_traits>

namespace tlin {
namespace {

using namespace ptx;
using namespace tc;

constexpr int kProducerWarp = 8;
constexpr int kMmaWarp = 9;
constexpr int kThreads = 32 * 12;          // warps 10 and 11 only lend their registers
constexpr int kSoftmaxRegs = 216, kOtherRegs = 72;   // 256*224 + 128*56 = 384*168 registers
// an increase beyond what the other warpgroup released would wait for ever
static_assert(256 * kSoftmaxRegs + 128 * kOtherRegs <= kThreads * 168, "register budget of the CTA exceeded");
constexpr float kLog2e = 1.4426950408889634f;
constexpr float kLn2 = 0.6931471805599453f;
constexpr int kPolyPairs = 5;                // of every 16 column pairs, this many get 2^x from the polynomial
// Keys of a step whose P is handed to the tensor pipe before the rest: their PV products run while the last columns are worked
// on.  After 64 of 128 keys the pipe ran dry before the rest came; after 96 it does not (64 -> 96: 1.86 -> 1.81 ms at
// B1 H32 N131072 W1024 d128, 262 -> 257 us at N32768 W512, 437 -> 429 us at B4 H32 N=W=4096 d64).
constexpr int kFirstKeys = 96;
constexpr float kRescaleThreshold = 32.0f;  // base-2 units: P stays below 2^32, far inside bf16/fp32 range
// An exponent is one fma, s * scale - m with m = round(s_max * scale).  That rounding is the same for all of a row and cancels, but where
// scores pass 2^31, as those of keys masked with the lowest finite value, it is a power of two that P cannot hold.  Other head sizes,
// whose P stands in for one kept in fp32, turn to differences of scores when a row's reference lies beyond this (base-2 units); the
// step that finds it is done again by another copy of the code.  Differences in every step cost 3 % (packed) to 9 % (single), a branch
// inside the step 4 %, this 0.6 %, over 50 calls.
constexpr float kFusedScores = 1024.f;

// 2^x for a packed pair without the special-function unit: x = n + f with n = floor(x) (taken by adding
// 1.5*2^23 rounding down, which leaves n in the low mantissa bits), 2^f on [0,1) by a cubic fitted for
// minimum relative error (7.9e-5, well below the 2^-9 rounding of P to bf16), n added into the exponent field.
// x is clamped to [-126, inf) first; values the caller produces stay far below the upper exponent limit.
__device__ __forceinline__ void exp2_poly2(uint64_t x2, float& p0, float& p1) {
    float x0, x1;
    f2_unpack(x2, x0, x1);
    x0 = fmaxf(x0, -126.f);
    x1 = fmaxf(x1, -126.f);
    const uint64_t xc = f2_pack(x0, x1);
    const uint64_t magic = f2_pack(12582912.f, 12582912.f);
    const uint64_t xf = f2_add_rm(xc, magic);
    const uint64_t fr = f2_sub(xc, f2_sub(xf, magic));
    uint64_t y = f2_fma(f2_pack(0.07806939631700516f, 0.07806939631700516f), fr, f2_pack(0.22593535482883453f, 0.22593535482883453f));
    y = f2_fma(y, fr, f2_pack(0.6959162950515747f, 0.6959162950515747f));
    y = f2_fma(y, fr, f2_pack(0.9999210238456726f, 0.9999210238456726f));
    uint32_t n0, n1, y0, y1;
    asm("mov.b64 {%0, %1}, %2;" : "=r"(n0), "=r"(n1) : "l"(xf));
    asm("mov.b64 {%0, %1}, %2;" : "=r"(y0), "=r"(y1) : "l"(y));
    p0 = __uint_as_float(y0 + (n0 << 23));
    p1 = __uint_as_float(y1 + (n1 << 23));
}

// The kernel's forms: head size D exactly, one problem or a table of them; or any other head size d <= D that is a multiple
// of 8.  The last reads its tiles with zero fill beyond d (the tensor maps know the true row length), contracts over ceil(d/16)
// slices only, and keeps P to 16 mantissa bits as the sum of two bf16 parts, two PV products per step: the CUDA-core kernel that
// served these sizes before kept P in fp32, and the results are to lose nothing (against 64-bit sums 1.66e-3, the rounding to
// bf16 alone).  At D = 256 two output accumulators would fill the TMEM, so a CTA works on one Q tile.
// Measured against that CUDA-core kernel: B2 H9 N3001 W517 d96 2066 -> 45 us, B2 H3 N7791 W968 d40 2582 -> 38 us, B1 H12 N2000
// W1000 d256 3952 -> 56 us, B4 H12 N370 W96 d32 96 -> 12 us.
// kDealt and kAnyDealt are the first and the last with problems dealt out by cost (DealtWalker; a form of their own because the
// choice at run time costs the others 1 to 2 %).
// kCluster and kAnyCluster are the first and the third for few, short problems: the CTAs of a cluster share the keys of one (b,h,query tile pair), leave their rows in
// their shared memory, and each merges a share of the rows from all of them; no merge kernel, no partials in global memory.
// Against split groups and the merge kernel: B2 H4 N3000 W100 d64 17.2 -> 11.6 us, B1 H16 N2000 W200 d64 17.9 -> 14.0, B4 H8 N1000 W64 d128
// 17.9 -> 13.1, B2 H16 N4000 W250 d128 33.7 -> 28.8, B1 H4 N1024 W128 d64 8.5 -> 8.3; B1 H9 N4000 W100 d80 23.7 -> 16.8, B2 H4 N2000
// W500 d160 26.6 -> 21.3; against whole problems B1 H3 N700 W500 d96 18.2 -> 12.0.  The merge has several rows and shares on their way
// at a time: one row after the other, 128 rows of two shares took 8 us.
enum { kOneProblem = 0, kTable = 1, kAnyHead = 2, kDealt = 3, kAnyDealt = 4, kCluster = 5, kAnyCluster = 6 };
constexpr int kMaxCluster = 8;             // the portable size

template <int D>
struct Cfg {
    static constexpr int kTiles = D == 256 ? 1 : 2;            // Q tiles per CTA
    static constexpr int kRows = kTiles * kQTile;              // query rows per CTA
    static constexpr int kTileBytes = kQTile * D * 2;          // one 128-row tile of Q, K or V
    static constexpr int kBoxes = D / 64;                      // 64-element (128-byte) column blocks per tile
    static constexpr int kSlots = D == 256 ? 2 : D == 128 ? 4 : 8;            // K/V ring slots
    static constexpr int kSmemTiles = (kTiles + kSlots) * kTileBytes;
    static constexpr int kStageBytes = 4 * kTiles * 32 * 128;  // per softmax warp 32 rows x 128 bytes: result rows on their way out
    static constexpr int kNumBars = 10 + 2 * kSlots;
    static constexpr int kSmemBytes = kSmemTiles + kStageBytes + kNumBars * 8 + 16 + 1024;   // + alignment slack
    // TMEM columns: S0, S1 (128 each), O0, O1 (D each)
    static constexpr uint32_t kColS = 0, kColO = 256;
};

// One problem of a batched launch as the kernel sees it (the field names N, W, causal, key_tiles are the ones the
// helpers shared with the single-problem kernel read).
struct ProblemDev {
    void* out;            // [BH, W, D] bf16
    float* lse;           // [BH, W] or null
    long long unit0;      // first unit of this problem in the launch's list: unit = unit0 + bh * q_tiles + q tile pair
    int N, W, causal, key_tiles, q_tiles;
};
// What a launch reads its tensors through: three tensor maps, or a table of them with the problems' shapes.
template <bool kBatched> struct KernelMaps;
template <> struct KernelMaps<false> { CUtensorMap q, k, v; };
template <> struct KernelMaps<true> {
    CUtensorMap q[kMaxBatch], k[kMaxBatch], v[kMaxBatch];
    ProblemDev prob[kMaxBatch];
    int n;
    int listed;                        // the CTAs' units are order[u], not u
    uint16_t order[kMaxListedUnits];
};

struct Params {
    void* out;            // [B*H, W, D] bf16
    float* lse;           // [B*H, W] or null
    float* ws;            // partial slots
    int* status;
    long long total_units;
    int n_groups, q_tiles, key_tiles;
    int N, W, causal;
    int d;                // head size (row length of every tensor)
    int cluster;          // CTAs that share a problem's keys (kCluster)
    int schedule;         // 0: groups of q_tiles CTAs stream key ranges; 1: every CTA walks whole (b,h,q-tile) problems
    float scale_log2e;
};

// Walks the units of a batched launch: whole problems, in table order (a contiguous run or a list).
struct BatchWalker {
    long long u, u1;
    const ProblemDev* prob;
    const uint16_t* order;
    int n, pi;
    __device__ BatchWalker(const KernelMaps<true>& m, const GroupStarts& starts)
        : u(starts.u[blockIdx.x]), u1(starts.u[blockIdx.x + 1]), prob(m.prob), order(m.listed ? m.order : nullptr), n(m.n), pi(0) {}
    __device__ bool next(Segment& s) {
        if (u >= u1) return false;
        const long long x = order != nullptr ? (long long)order[u] : u;
        while (pi + 1 < n && x >= prob[pi + 1].unit0) ++pi;
        const long long r = x - prob[pi].unit0;
        s.bh = (int)(r / prob[pi].q_tiles);
        s.qt = (int)(r - (long long)s.bh * prob[pi].q_tiles);
        s.t_begin = 0;
        s.t_end = prob[pi].key_tiles;
        s.prob = pi;
        ++u;
        return true;
    }
};
// The one segment of a CTA of a cluster: its share of the key tiles that the pair may use.
template <int D>
struct ClusterWalker {
    Segment seg;
    bool more;
    __device__ ClusterWalker(const Params& p) : more(true) {
        const int problem = blockIdx.x / p.cluster, rank = blockIdx.x - problem * p.cluster;
        seg.prob = 0;
        seg.bh = problem / p.q_tiles;
        seg.qt = problem - seg.bh * p.q_tiles;
        const int row0 = seg.qt * Cfg<D>::kRows;
        const int a0 = tiles_allowed(p, row0, 0), a1 = Cfg<D>::kTiles > 1 ? tiles_allowed(p, row0, 1) : 0, tiles = a0 > a1 ? a0 : a1;
        seg.t_begin = tiles * rank / p.cluster;
        seg.t_end = tiles * (rank + 1) / p.cluster;
    }
    __device__ bool next(Segment& s) {
        s = seg;
        const bool had = more;
        more = false;
        return had;
    }
};
template <int D, int kForm>
__device__ __forceinline__ auto make_walker(const KernelMaps<kForm == kTable>& m, const Params& p, const GroupStarts& starts) {
    if constexpr (kForm == kTable) return BatchWalker(m, starts);
    else if constexpr (kForm == kDealt || kForm == kAnyDealt) return DealtWalker(p, starts);
    else if constexpr (kForm == kCluster || kForm == kAnyCluster) return ClusterWalker<D>(p);
    else return SegmentWalker(p, starts);
}
// shape (N, W, causal, key_tiles) and result pointers of the problem a segment belongs to
template <bool kBatched>
__device__ __forceinline__ decltype(auto) problem_of(const KernelMaps<kBatched>& m, const Params& p, const Segment& s) {
    if constexpr (kBatched) return (m.prob[s.prob]);
    else return (p);
}

template <int D, int kForm>
__global__ void __launch_bounds__(kThreads, 1)
fwd_tc_kernel(const __grid_constant__ KernelMaps<kForm == kTable> maps, const __grid_constant__ Params p,
              const __grid_constant__ GroupStarts starts) {
    using C = Cfg<D>;
    constexpr bool kBatched = kForm == kTable, kAny = kForm == kAnyHead || kForm == kAnyDealt || kForm == kAnyCluster, kShared = kForm == kCluster || kForm == kAnyCluster, kWhole = kForm == kTable || kForm >= kDealt;   // kWhole: no split keys
    constexpr int kTileM = C::kRows;
    const int d = kAny ? p.d : D;                              // row length; everything below folds where it is D
    const int boxes = kAny ? (d + 63) / 64 : C::kBoxes;
    extern __shared__ uint8_t smem_raw[];
    uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
    uint8_t* sQ = smem;                               // kTiles tiles
    uint8_t* sRing = smem + C::kTiles * C::kTileBytes;        // kSlots tiles
    uint8_t* sStage = smem + C::kSmemTiles;
    uint64_t* bars = reinterpret_cast<uint64_t*>(smem + C::kSmemTiles + C::kStageBytes);
    uint64_t* q_full = bars + 0;
    uint64_t* q_empty = bars + 1;
    uint64_t* s_full = bars + 2;      // [2]
    uint64_t* p_full = bars + 4;      // [2]
    uint64_t* pv_done = bars + 6;     // [2]
    uint64_t* p_first = bars + 8;     // [2]  first kFirstKeys keys of P written (PV may start on them)
    uint64_t* kv_full = bars + 10;    // [kSlots]
    uint64_t* kv_empty = bars + 10 + C::kSlots;
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(bars + C::kNumBars);
    __shared__ int abort_flag;

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;

    if (threadIdx.x == 0) {
        abort_flag = 0;
        mbar_init(q_full, 1);
        mbar_init(q_empty, 1);
        for (int i = 0; i < 2; ++i) {
            mbar_init(&s_full[i], 1);
            mbar_init(&p_full[i], kQTile);
            mbar_init(&p_first[i], kQTile);
            mbar_init(&pv_done[i], 1);
        }
        for (int s = 0; s < C::kSlots; ++s) {
            mbar_init(&kv_full[s], 1);
            mbar_init(&kv_empty[s], 1);
        }
        fence_mbar_init();
    }
    if (warp == kMmaWarp) {
        tmem_alloc(tmem_slot, 512);
        tmem_relinquish();
    }
    if constexpr (!kBatched) {
        if (warp == kProducerWarp && lane == 0) {
            prefetch_tensormap(&maps.q);
            prefetch_tensormap(&maps.k);
            prefetch_tensormap(&maps.v);
        }
    }
    tc_fence_before();
    after_previous();
    let_next_start();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem_base = *tmem_slot;
    volatile int* abort_p = &abort_flag;
    // the softmax warpgroups hold a whole row of S in registers; the third warpgroup gives them its share

    if (warp >= 8) {
    setmaxnreg_dec<kOtherRegs>();
    if (warp == kProducerWarp) {
        // ------------------------------------------------------------------ TMA producer
        if (lane == 0) {
            uint32_t it = 0;           // ring counter
            uint32_t seg_idx = 0;
            bool ok = true;
            auto walk = make_walker<D, kForm>(maps, p, starts);
            Segment s;
            while (ok && walk.next(s)) {
                const auto& pr = problem_of<kBatched>(maps, p, s);
                const CUtensorMap* map_q_p;
                const CUtensorMap* map_k_p;
                const CUtensorMap* map_v_p;
                if constexpr (kBatched) { map_q_p = &maps.q[s.prob]; map_k_p = &maps.k[s.prob]; map_v_p = &maps.v[s.prob]; }
                else { map_q_p = &maps.q; map_k_p = &maps.k; map_v_p = &maps.v; }
                const int row0 = s.qt * kTileM;
                const int c0 = seg_count(s, tiles_allowed(pr, row0, 0)), c1 = C::kTiles > 1 ? seg_count(s, tiles_allowed(pr, row0, 1)) : 0;
                const int cnt = c0 > c1 ? c0 : c1;
                if (cnt == 0) continue;
                if (seg_idx > 0) ok = mbar_wait(q_empty, (seg_idx - 1) & 1, abort_p);
                if (!ok) break;
                mbar_arrive_expect_tx(q_full, C::kTiles * boxes * (kQTile * 128));
                for (int i = 0; i < C::kTiles; ++i)
                    for (int b = 0; b < boxes; ++b)
                        tma_load_3d(sQ + i * C::kTileBytes + b * (kQTile * 128), map_q_p, q_full, b * 64, row0 + i * kQTile, s.bh);
                for (int j = 0; j < cnt && ok; ++j) {
                    const int t = s.t_begin + j;
                    for (int kv = 0; kv < 2 && ok; ++kv) {
                        const uint32_t slot = it % C::kSlots, round = it / C::kSlots;
                        ok = mbar_wait(&kv_empty[slot], (round & 1) ^ 1, abort_p);
                        if (!ok) break;
                        mbar_arrive_expect_tx(&kv_full[slot], boxes * (kQTile * 128));
                        uint8_t* dst = sRing + slot * C::kTileBytes;
                        for (int b = 0; b < boxes; ++b)
                            tma_load_3d(dst + b * (kQTile * 128), kv == 0 ? map_k_p : map_v_p, &kv_full[slot], b * 64, t * kTileN, s.bh);
                        ++it;
                    }
                }
                ++seg_idx;
            }
            if (!ok) {
                // leave no copy in flight: every slot armed in its latest round must have landed
                for (uint32_t back = 0; back < (uint32_t)C::kSlots && back < it; ++back) {
                    const uint32_t id = it - 1 - back, slot = id % C::kSlots, round = id / C::kSlots;
                    int dummy = 0;
                    mbar_wait(&kv_full[slot], round & 1, &dummy, 200000000LL);
                }
                // seg_idx counts the Q loads armed so far; the last one may still be on its way
                if (seg_idx > 0) {
                    int dummy = 0;
                    mbar_wait(q_full, (seg_idx - 1) & 1, &dummy, 200000000LL);
                }
            }
        }
    } else if (warp == kMmaWarp) {
        // ------------------------------------------------------------------ MMA issuer
        // The whole warp walks the schedule (every value below is the same in all lanes) and one lane, elected once, issues
        // under a predicate: descriptors and addresses then live in uniform registers and an MMA costs a few instructions,
        // which matters because the tensor pipe takes the next MMA only when it has room.  Electing a lane at every MMA
        // instead: 1.88 against 1.83 ms (B1 H32 N131072 W1024 d128), 382 against 361 us (N32768 W1024 d64).
        {
            const uint32_t idesc_qk = make_idesc_bf16(kQTile, kTileN, 0, 0);
            const uint32_t idesc_pv = make_idesc_bf16(kQTile, kAny ? (d + 15) / 16 * 16 : D, 0, 1);
            const int slices = kAny ? (d + 15) / 16 : D / 16;         // of the head dimension
            // Descriptors are built once; per MMA only the 14-bit address field of the low word moves
            // (one 32-bit add of a compile-time constant).
            const uint64_t q_desc = make_smem_desc_sw128(smem_u32(sQ), 16, 1024);
            const uint64_t k_desc = make_smem_desc_sw128(smem_u32(sRing), 16, 1024);            // K-major tile (K)
            const uint64_t v_desc = make_smem_desc_sw128(smem_u32(sRing), kQTile * 128, 1024);  // MN-major tile (V)
            const uint32_t desc_hi = (uint32_t)(q_desc >> 32);        // identical for all three
            const uint32_t q_lo[2] = {(uint32_t)q_desc, (uint32_t)q_desc + (C::kTileBytes >> 4)};      // [1] unused with one Q tile
            const uint32_t k_lo0 = (uint32_t)k_desc, v_lo0 = (uint32_t)v_desc;
            const uint32_t tmem_u = __shfl_sync(0xffffffffu, tmem_base, 0);
            const uint32_t tS0 = tmem_u + C::kColS, tO0 = tmem_u + C::kColO;
            const uint32_t lead = elect_one() ? 1u : 0u;
            uint32_t it = 0, seg_idx = 0;
            uint32_t n_pv[2] = {0, 0};
            bool ok = true;
            auto issue_qk = [&](int i, uint32_t k_slot) {
                const uint32_t a_lo = q_lo[i], b_lo = k_lo0 + k_slot * (C::kTileBytes >> 4), acc = tS0 + i * kTileN;
#pragma unroll
                for (int kk = 0; kk < D / 16; ++kk) {
                    const uint32_t off16 = ((kk >> 2) * (kQTile * 128) + (kk & 3) * 32) >> 4;
                    mma_ss_lead(!kAny || kk < slices ? lead : 0u, acc, a_lo + off16, b_lo + off16, desc_hi, idesc_qk, kk > 0);
                }
                commit_lead(lead, &s_full[i]);
            };
            // PV of the keys [16 from, 16 to) of a tile
            auto issue_pv = [&](int i, uint32_t v_slot, bool accumulate, auto from, auto to) {
                const uint32_t b_lo = v_lo0 + v_slot * (C::kTileBytes >> 4), acc = tO0 + i * D, a = tS0 + i * kTileN;
#pragma unroll
                for (int kk = decltype(from)::value; kk < decltype(to)::value; ++kk)
                    mma_ts_lead(lead, acc, a + (kAny ? (kk >> 1) * 32 + (kk & 1) * 8 : kk * 8), b_lo + kk * (2048 >> 4), desc_hi, idesc_pv, (accumulate || kk > 0) ? 1u : 0u);
                if constexpr (kAny)        // the low parts of P: of each 32 keys behind the high ones
#pragma unroll
                    for (int kk = decltype(from)::value; kk < decltype(to)::value; ++kk)
                        mma_ts_lead(lead, acc, a + 16 + (kk >> 1) * 32 + (kk & 1) * 8, b_lo + kk * (2048 >> 4), desc_hi, idesc_pv, 1u);
            };
            constexpr std::integral_constant<int, 0> k_begin{};
            constexpr std::integral_constant<int, kFirstKeys / 16> k_first{};
            constexpr std::integral_constant<int, kTileN / 16> k_end{};
            auto walk = make_walker<D, kForm>(maps, p, starts);
            Segment s;
            while (ok && walk.next(s)) {
                const auto& pr = problem_of<kBatched>(maps, p, s);
                const int row0 = s.qt * kTileM;
                const int c0 = seg_count(s, tiles_allowed(pr, row0, 0)), c1 = C::kTiles > 1 ? seg_count(s, tiles_allowed(pr, row0, 1)) : 0;
                const int cnt = c0 > c1 ? c0 : c1;
                if (cnt == 0) continue;
                const int cq[2] = {c0, c1};
                ok = __all_sync(0xffffffffu, mbar_wait(q_full, seg_idx & 1, abort_p));
                if (!ok) break;
                // first K tile
                uint32_t k_slot = it % C::kSlots;
                ok = __all_sync(0xffffffffu, mbar_wait(&kv_full[k_slot], (it / C::kSlots) & 1, abort_p));
                if (!ok) break;
                tc_fence_after();
                for (int i = 0; i < C::kTiles; ++i)
                    if (cq[i] > 0) issue_qk(i, k_slot);
                commit_lead(lead, &kv_empty[k_slot]);
                if (cnt == 1) commit_lead(lead, q_empty);      // the segment's last use of Q is issued: its successor may load
                ++it;
                for (int j = 0; j < cnt && ok; ++j) {
                    const uint32_t v_slot = it % C::kSlots, v_par = (it / C::kSlots) & 1;
                    ++it;
                    const bool have_next = j + 1 < cnt;
                    uint32_t nk_slot = 0, nk_par = 0;
                    if (have_next) {
                        nk_slot = it % C::kSlots;
                        nk_par = (it / C::kSlots) & 1;
                        ++it;
                    }
                    // both tiles are usually there already: ask both barriers at once (the two answers travel together), and
                    // wait one after the other only if one is missing
                    {
                        const bool v_there = mbar_try_wait(&kv_full[v_slot], v_par);
                        const bool k_there = have_next ? mbar_try_wait(&kv_full[nk_slot], nk_par) : true;
                        if (!__all_sync(0xffffffffu, v_there && k_there)) {
                            ok = __all_sync(0xffffffffu, mbar_wait(&kv_full[v_slot], v_par, abort_p));
                            if (!ok) break;
                            if (have_next) {
                                ok = __all_sync(0xffffffffu, mbar_wait(&kv_full[nk_slot], nk_par, abort_p));
                                if (!ok) break;
                            }
                        }
                    }
                    tc_fence_after();
                    for (int i = 0; i < C::kTiles && ok; ++i) {
                        if (j < cq[i]) {
                            ok = __all_sync(0xffffffffu, mbar_wait(&p_first[i], n_pv[i] & 1, abort_p));
                            if (!ok) break;
                            tc_fence_after();
                            issue_pv(i, v_slot, j > 0, k_begin, k_first);
                            ok = __all_sync(0xffffffffu, mbar_wait(&p_full[i], n_pv[i] & 1, abort_p));
                            if (!ok) break;
                            tc_fence_after();
                            issue_pv(i, v_slot, j > 0, k_first, k_end);
                            commit_lead(lead, &pv_done[i]);
                            ++n_pv[i];
                        }
                        if (i == C::kTiles - 1) commit_lead(lead, &kv_empty[v_slot]);
                        if (have_next && j + 1 < cq[i]) issue_qk(i, nk_slot);
                        if (have_next && i == C::kTiles - 1) {
                            commit_lead(lead, &kv_empty[nk_slot]);
                            // Q is last read by the S of the segment's last key tile: releasing it here lets the
                            // producer fetch the next segment's Q while this one finishes
                            if (j + 2 == cnt) commit_lead(lead, q_empty);
                        }
                    }
                }
                if (!ok) break;
                ++seg_idx;
            }
        }
    }
    if constexpr (kShared) {                    // the two barriers of the merge below
        __syncwarp();
        cluster_sync();
        cluster_sync();
    }
    } else {
        // ------------------------------------------------------------------ softmax warpgroups (one per Q tile)
        setmaxnreg_inc<kSoftmaxRegs>();
        if (C::kTiles > 1 || warp < 4) {
        const int i = warp >> 2;                           // Q tile
        const int r = (warp & 3) * 32 + lane;              // row inside the Q tile == TMEM lane
        const uint32_t lane_addr = (uint32_t)((warp & 3) * 32) << 16;
        const uint32_t tS = tmem_base + lane_addr + C::kColS + i * kTileN;
        const uint32_t tO = tmem_base + lane_addr + C::kColO + i * D;
        uint32_t n = 0;     // tiles processed by this warpgroup (phase counter of s_full/p_full/pv_done)
        bool ok = true;
        // one rounding at other head sizes, whose P is worth it: against 64 bits lse is off by 3.1e-8 of its value, as in fp32, instead of 4.7e-8
        auto lse_of = [](float m, float sum) { return kAny ? fmaf(m, kLn2, logf(sum)) : (m + log2f(sum)) * kLn2; };
        auto walk = make_walker<D, kForm>(maps, p, starts);
        int bh_first = 0;                                  // (b,h) of this CTA's first unit (used under schedule 0 only)
        if constexpr (!kWhole) bh_first = (int)(walk.u / p.key_tiles);
        Segment s;
        while (ok && walk.next(s)) {
            const auto& pr = problem_of<kBatched>(maps, p, s);
            const int row0 = s.qt * kTileM;
            const int row = row0 + i * kQTile + r;         // row inside W (may lie beyond W: computed, never stored)
            const int allowed_i = tiles_allowed(pr, row0, i);
            // keys visible to this row, and to the first row of this warp (the smallest in the warp)
            const long long lim_row_ll = pr.causal ? (long long)pr.N - pr.W + row + 1 : (long long)pr.N;
            const int lim_row = (int)(lim_row_ll < pr.N ? lim_row_ll : pr.N);
            const long long lim_warp_ll = pr.causal ? (long long)pr.N - pr.W + (row - lane) + 1 : (long long)pr.N;
            const int lim_warp = (int)(lim_warp_ll < pr.N ? lim_warp_ll : pr.N);
            const int cnt_i = seg_count(s, allowed_i);
            float m_ref = -CUDART_INF_F;
            float s_ref = -CUDART_INF_F;            // kAny: the score that m_ref is of
            bool beyond = false;                    // kAny: the reference of some row of the warp is beyond kFusedScores
            uint64_t l2[2] = {0ull, 0ull};          // four partial row sums as two packed fp32 pairs
            // One key tile.  The steps with masked columns (the last ones of a segment, if any) are a second copy of the code:
            // conditions inside the exponential loop cut it into short blocks that each wait for their own results.  One copy with
            // conditions and the row sums inside the loop against this: B1 H32 N131072 W1024 d128 2.15 -> 1.89 ms,
            // N32768 W512 298 -> 265 us, B1 H32 N32768 W1024 d64 416 -> 380 us (back to back, under the power cap).
            auto step = [&](int j, auto masked_tag, auto exact_tag) {
                constexpr bool kMasked = decltype(masked_tag)::value, kExact = decltype(exact_tag)::value;
                ok = mbar_wait(&s_full[i], n & 1, abort_p);
                ok = __all_sync(0xffffffffu, ok);
                if (!ok) return;
                tc_fence_after();
                // the whole row of S (128 fp32) comes into registers once (in the form with a loop below, its chunks once more for the exponentials)
                const int nvalid = kMasked ? lim_row - (s.t_begin + j) * kTileN : 0;   // columns [0, nvalid) of this tile are allowed for this row
                uint32_t sv[kTileN / 32][32];
#pragma unroll
                for (int c = 0; c < kTileN / 32; ++c) tmem_ld32_async(tS + c * 32, sv[c]);
#pragma unroll
                for (int c = 0; c < kTileN / 32; ++c) tmem_wait_ld(sv[c]);
                if constexpr (kMasked) {
#pragma unroll
                    for (int e = 0; e < kTileN; ++e)
                        if (e >= nvalid) sv[e >> 5][e & 31] = 0xff800000u;   // -inf
                }
                float mx[4] = {-CUDART_INF_F, -CUDART_INF_F, -CUDART_INF_F, -CUDART_INF_F};   // independent chains
#pragma unroll
                for (int e = 0; e < kTileN / 2; ++e)
                    mx[e & 3] = max3(mx[e & 3], __uint_as_float(sv[e >> 4][(2 * e) & 31]), __uint_as_float(sv[e >> 4][(2 * e + 1) & 31]));
                const float tmax = fmaxf(fmaxf(mx[0], mx[1]), fmaxf(mx[2], mx[3]));
                const float m_new = fmaxf(m_ref, tmax * p.scale_log2e);
                const bool need = kExact ? tmax > s_ref : m_new > m_ref + kRescaleThreshold;
                if (__any_sync(0xffffffffu, need)) {
                    if constexpr (kAny && !kExact) {       // nothing of this step has been written yet
                        beyond = __any_sync(0xffffffffu, need && fabsf(m_new) > kFusedScores);
                        if (beyond) return;
                    }
                    const float alpha = need ? ex2(kExact ? (s_ref - tmax) * p.scale_log2e : m_ref - m_new) : 1.f;     // m_ref = -inf -> 0
                    if (j > 0) {
                        ok = mbar_wait(&pv_done[i], (n - 1) & 1, abort_p);
                        ok = __all_sync(0xffffffffu, ok);
                        if (!ok) return;
                        tc_fence_after();
#pragma unroll
                        for (int c = 0; c < D / 8; ++c) {      // narrow pieces: the row of S stays in registers meanwhile
                            if (kAny && c * 8 >= d) break;
                            uint32_t o[8];
                            tmem_ld8(tO + c * 8, o);
#pragma unroll
                            for (int e = 0; e < 8; ++e) o[e] = __float_as_uint(__uint_as_float(o[e]) * alpha);
                            tmem_st8(tO + c * 8, o);
                        }
                    }
                    const uint64_t alpha2 = f2_pack(alpha, alpha);
                    l2[0] = f2_mul(l2[0], alpha2);
                    l2[1] = f2_mul(l2[1], alpha2);
                    if (need) {
                        m_ref = m_new;
                        if constexpr (kAny) s_ref = tmax;
                    }
                }
                const float m_use = m_ref == -CUDART_INF_F ? 0.f : m_ref;
                // P = 2^(s*scale - m) as bf16 over the columns of S; kPolyPairs of every 16 pairs take the polynomial route (FMA
                // pipe), the rest the special-function unit.  A masked tile takes the special-function unit only: it gives an
                // exact 0 for -inf, the polynomial 2^-126.  The fp32 values stay in the registers of S and are summed after P has
                // been handed over, off the path the tensor pipe waits for.
                const float s_use = s_ref == -CUDART_INF_F ? 0.f : s_ref;
                const uint64_t scale2 = f2_pack(p.scale_log2e, p.scale_log2e), negm2 = kExact ? f2_pack(-s_use, -s_use) : f2_pack(-m_use, -m_use);
                if constexpr (kAny && (D > 64 || kForm == kAnyDealt)) {
                    // A loop over chunks of 32 keys: unrolled, the three copies of the step (open, masked, exact) and the MMA warp's code did
                    // not fit the instruction cache together, 1.9 of 8.2 stall cycles per instruction.  Unrolled / loop, microseconds: B2 H9
                    // N3001 W517 d96 41.4 / 37.1, d160 53.5 / 51.3, d256 67.2 / 64.4; B1 H12 N8000 W700 d112 61.1 / 55.1, d192 90.9 / 91.6.
                    // Up to 64 columns the code is half as long and long runs of open tiles fit: there the loop only where whole problems
                    // are dealt out (d32: B4 H16 N512 W512 14.9 / 14.1, B16 H16 N1200 W600 118.3 / 116.1); elsewhere B1 H8 N16000 W1024 60.8 /
                    // 66.3, B2 H9 N3001 W517 28.9 / 30.0, B1 H12 N8000 W700 42.2 / 44.8, against B16 H16 N400 W256 29.5 / 28.2.  At d = 64
                    // and 128 the loop is the slower form (56.8 / 60.0, 230 / 240).
#pragma unroll 1
                    for (int c = 0; c < kTileN / 32; ++c) {
                        uint32_t x[32], pk[16], pk_low[16];
                        tmem_ld32(tS + c * 32, x);
                        if constexpr (kMasked)
#pragma unroll
                            for (int e = 0; e < 32; ++e)
                                if (c * 32 + e >= nvalid) x[e] = 0xff800000u;
#pragma unroll
                        for (int e = 0; e < 16; ++e) {
                            const uint64_t s2 = f2_pack_bits(x[2 * e], x[2 * e + 1]);
                            const uint64_t x2 = kExact ? f2_mul(f2_add(s2, negm2), scale2) : f2_fma(s2, scale2, negm2);
                            float p0, p1;
                            f2_unpack(x2, p0, p1);
                            p0 = ex2(p0);
                            p1 = ex2(p1);
                            pk[e] = pack_bf16x2(p0, p1);
                            pk_low[e] = pack_bf16x2(p0 - __uint_as_float(pk[e] << 16), p1 - __uint_as_float(pk[e] & 0xffff0000u));
                            l2[e & 1] = f2_add(l2[e & 1], f2_pack(p0, p1));
                        }
                        tmem_st16(tS + c * 32, pk);            // both parts over this chunk's columns of S
                        tmem_st16(tS + c * 32 + 16, pk_low);
                        if (c == kFirstKeys / 32 - 1) {
                            tc_wait_st();
                            tc_fence_before();
                            mbar_arrive(&p_first[i]);
                        }
                    }
                    tc_wait_st();
                    tc_fence_before();
                    mbar_arrive(&p_full[i]);
                    ++n;
                    return;
                }
#pragma unroll
                for (int c = 0; c < kTileN / 32; ++c) {
                    uint32_t pk[16], pk_low[kAny ? 16 : 1];
#pragma unroll
                    for (int e = 0; e < 16; ++e) {
                        const uint64_t s2 = f2_pack_bits(sv[c][2 * e], sv[c][2 * e + 1]);
                        const uint64_t x2 = kExact ? f2_mul(f2_add(s2, negm2), scale2) : f2_fma(s2, scale2, negm2);
                        float p0, p1;
                        if (!kMasked && !kAny && e * kPolyPairs / 16 != (e + 1) * kPolyPairs / 16) {
                            exp2_poly2(x2, p0, p1);
                        } else {
                            float x0, x1;
                            f2_unpack(x2, x0, x1);
                            p0 = ex2(x0);
                            p1 = ex2(x1);
                        }
                        sv[c][2 * e] = __float_as_uint(p0);
                        sv[c][2 * e + 1] = __float_as_uint(p1);
                        pk[e] = pack_bf16x2(p0, p1);
                        if constexpr (kAny)
                            pk_low[e] = pack_bf16x2(p0 - __uint_as_float(pk[e] << 16), p1 - __uint_as_float(pk[e] & 0xffff0000u));
                    }
                    tmem_st16(tS + c * (kAny ? 32 : 16), pk);
                    if constexpr (kAny) tmem_st16(tS + c * 32 + 16, pk_low);
                    if (c == kFirstKeys / 32 - 1) {    // the first keys are in place: let the PV MMAs start on them
                        tc_wait_st();
                        tc_fence_before();
                        mbar_arrive(&p_first[i]);
                    }
                }
                tc_wait_st();
                tc_fence_before();
                mbar_arrive(&p_full[i]);
#pragma unroll
                for (int e = 0; e < kTileN / 2; ++e)
                    l2[e & 1] = f2_add(l2[e & 1], f2_pack_bits(sv[e >> 4][(2 * e) & 31], sv[e >> 4][(2 * e + 1) & 31]));
                ++n;
            };
            // steps before the first tile in which some column of some lane of the warp is masked
            int n_open = lim_warp / kTileN - s.t_begin;
            n_open = n_open < 0 ? 0 : (n_open < cnt_i ? n_open : cnt_i);
            int j = 0;
            for (; j < n_open && ok && !beyond; ++j) {
                step(j, std::false_type{}, std::false_type{});
                if (kAny && beyond) break;
            }
            for (; j >= n_open && j < cnt_i && ok && !beyond; ++j) {
                step(j, std::true_type{}, std::false_type{});
                if (kAny && beyond) break;
            }
            if constexpr (kAny)                            // from the step that found it on, that one again
                for (; beyond && j < cnt_i && ok; ++j) step(j, std::true_type{}, std::true_type{});
            if constexpr (kShared) {
                // -------------------------------------------------------- merge inside the cluster
                if (ok && cnt_i > 0) {
                    ok = mbar_wait(&pv_done[i], (n - 1) & 1, abort_p);
                    ok = __all_sync(0xffffffffu, ok);
                    tc_fence_after();
                }
                float x0, x1, x2, x3;
                f2_unpack(l2[0], x0, x1);
                f2_unpack(l2[1], x2, x3);
                const float l = (x0 + x1) + (x2 + x3);
                const bool none = !ok || l == 0.f;                // no keys here, or none that counts; a NaN is passed on
                float* sO = reinterpret_cast<float*>(smem);       // rows of D, 16-byte pieces at (piece xor row mod 8)
                float* sLse = sO + kTileM * D;
                static_assert(kTileM * (D + 1 + kMaxCluster / 2) * 4 <= C::kSmemTiles, "the rows lie over Q and the ring");
                named_barrier(1, kTileM);          // all Q tiles' products are complete: Q and the ring are free
                const int rl = i * kQTile + r;
                sLse[rl] = none ? -CUDART_INF_F : lse_of(m_ref, l);
                const float inv_l = none ? 0.f : 1.f / l;
                if (ok && cnt_i > 0) {
#pragma unroll
                    for (int c = 0; c < D / 16; ++c) {
                        if (kAny && c * 16 >= d) break;
                        uint32_t o[16];
                        tmem_ld16_async(tO + c * 16, o);
                        tmem_wait_ld16(o);
#pragma unroll
                        for (int v4 = 0; v4 < 4; ++v4)
                            *reinterpret_cast<float4*>(sO + rl * D + (((c * 4 + v4) ^ (rl & 7)) << 2)) =
                                make_float4(__uint_as_float(o[v4 * 4]) * inv_l, __uint_as_float(o[v4 * 4 + 1]) * inv_l,
                                            __uint_as_float(o[v4 * 4 + 2]) * inv_l, __uint_as_float(o[v4 * 4 + 3]) * inv_l);
                    }
                }
                __syncwarp();
                cluster_sync();
                namespace cg = cooperative_groups;
                cg::cluster_group cl = cg::this_cluster();
                constexpr int kLanes = D / 4 < 32 ? D / 4 : 32;     // lanes per row
                const int rank = (int)cl.block_rank(), rr_begin = kTileM * rank / p.cluster, rr_end = kTileM * (rank + 1) / p.cluster;
                const long long at0 = (long long)s.bh * p.W + row0;
                // the shares' weights, one row per thread; negative where a share has no keys for the row and has left nothing
                float* sW = sLse + kTileM;                          // [row - rr_begin][kMaxCluster]
                if (rr_begin + (int)threadIdx.x < rr_end) {
                    const int rr = rr_begin + threadIdx.x;
                    float part[kMaxCluster], top = -CUDART_INF_F, z = 0.f;
#pragma unroll
                    for (int c = 0; c < kMaxCluster; ++c) {
                        part[c] = c < p.cluster ? cl.map_shared_rank(sLse, c)[rr] : -CUDART_INF_F;
                        top = fmaxf(top, part[c]);
                    }
                    const float ref = fmaxf(top, -FLT_MAX);
                    float weight[kMaxCluster];
#pragma unroll
                    for (int c = 0; c < kMaxCluster; ++c) {
                        weight[c] = ex2((part[c] - ref) * kLog2e);
                        z += weight[c];
                    }
                    const float f = 1.f / z;                    // not used where no share has anything
#pragma unroll
                    for (int c = 0; c < kMaxCluster; ++c) sW[(rr - rr_begin) * kMaxCluster + c] = part[c] == -CUDART_INF_F ? -1.f : weight[c] * f;
                    if (row0 + rr < p.W && p.lse != nullptr) p.lse[at0 + rr] = top + logf(z);
                }
                named_barrier(1, kTileM);
                // kU rows per lane and kE shares of each on their way at a time
                constexpr int kRowStep = 4 * C::kTiles * (32 / kLanes);     // rows of all softmax warps
                auto merge_rows = [&](auto rows_at_once, auto shares_at_once) {
                    constexpr int kU = decltype(rows_at_once)::value, kE = decltype(shares_at_once)::value;
                    for (int r0 = rr_begin + warp * (32 / kLanes) + lane / kLanes; r0 < rr_end; r0 += kU * kRowStep) {
#pragma unroll
                        for (int v = 0; v < D / 4 / kLanes; ++v) {
                            const int piece = lane % kLanes + v * kLanes;
                            if (kAny && piece * 4 >= d) break;
                            float w[kU][kE];
                            float4 x[kU][kE];
#pragma unroll
                            for (int u = 0; u < kU; ++u) {
                                const int rr = r0 + u * kRowStep;
#pragma unroll
                                for (int e = 0; e < kE; ++e) {
                                    w[u][e] = rr < rr_end ? sW[(rr - rr_begin) * kMaxCluster + e] : -1.f;
                                    x[u][e] = make_float4(0.f, 0.f, 0.f, 0.f);
                                    if (!(w[u][e] < 0.f)) x[u][e] = *reinterpret_cast<const float4*>(cl.map_shared_rank(sO, e) + rr * D + ((piece ^ (rr & 7)) << 2));
                                }
                            }
#pragma unroll
                            for (int u = 0; u < kU; ++u) {
                                const int rr = r0 + u * kRowStep;
                                float4 sum = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
                                for (int e = 0; e < kE; ++e) {
                                    sum.x = fmaf(w[u][e], x[u][e].x, sum.x); sum.y = fmaf(w[u][e], x[u][e].y, sum.y);
                                    sum.z = fmaf(w[u][e], x[u][e].z, sum.z); sum.w = fmaf(w[u][e], x[u][e].w, sum.w);
                                }
                                if (rr < rr_end && row0 + rr < p.W)
                                    *reinterpret_cast<uint2*>(reinterpret_cast<__nv_bfloat16*>(p.out) + (at0 + rr) * d + piece * 4) =
                                        make_uint2(pack_bf16x2(sum.x, sum.y), pack_bf16x2(sum.z, sum.w));
                            }
                        }
                    }
                };
                if (p.cluster > 4) merge_rows(std::integral_constant<int, 2>{}, std::integral_constant<int, 8>{});
                else merge_rows(std::integral_constant<int, 4>{}, std::integral_constant<int, 4>{});
                __syncwarp();
                cluster_sync();                    // nobody leaves while its rows are still being read
                break;
            }
            if (!ok) break;
            if (allowed_i == 0) continue;                  // this Q tile does not exist: nothing to write
            // ---------------------------------------------------------------- epilogue of the segment
            const bool whole = kWhole || (s.t_begin == 0 && s.t_end == p.key_tiles);
            if (cnt_i > 0) {
                ok = mbar_wait(&pv_done[i], (n - 1) & 1, abort_p);
                ok = __all_sync(0xffffffffu, ok);
                if (!ok) break;
                tc_fence_after();
            }
            float l;
            {
                float a, b, c, d2;
                f2_unpack(l2[0], a, b);
                f2_unpack(l2[1], c, d2);
                l = (a + b) + (c + d2);
            }
            const float inv_l = l == 0.f ? 0.f : 1.f / l;      // a NaN is passed on, in the row and in its lse
            const float lse_val = l == 0.f ? -CUDART_INF_F : lse_of(m_ref, l);
            const bool store = row < pr.W;
            // partial result -> workspace slot (0: first segment of this CTA's range, 1: a later one)
            float* pbase = p.ws + ((long long)blockIdx.x * 2 + (s.bh == bh_first ? 0 : 1)) * (long long)kTileM * (d + 1);
            // A thread holds one row.  Stored straight from the registers a warp's store would touch 32 different lines, so
            // the warp passes its rows through shared memory 128 bytes at a time (16-byte pieces, piece index xor row: no
            // bank conflicts beyond the minimum on either side) and every store instruction writes four whole lines.
            uint8_t* stage = sStage + warp * (32 * 128);
            const int row_warp = row - lane;                   // row of lane 0
            if (whole) {
                __nv_bfloat16* owarp = reinterpret_cast<__nv_bfloat16*>(pr.out) + ((long long)s.bh * pr.W + row_warp) * d;
#pragma unroll
                for (int h = 0; h < D / 64; ++h) {             // 64 bf16 columns per pass
                    if (kAny && h * 64 >= d) break;
#pragma unroll
                    for (int c = 0; c < 4; ++c) {
                        uint32_t o[16];
                        if (cnt_i > 0) {
                            tmem_ld16_async(tO + h * 64 + c * 16, o);
                            tmem_wait_ld16(o);
                        } else {
#pragma unroll
                            for (int e = 0; e < 16; ++e) o[e] = 0u;
                        }
#pragma unroll
                        for (int v4 = 0; v4 < 2; ++v4) {
                            uint4 w;
                            w.x = pack_bf16x2(__uint_as_float(o[v4 * 8 + 0]) * inv_l, __uint_as_float(o[v4 * 8 + 1]) * inv_l);
                            w.y = pack_bf16x2(__uint_as_float(o[v4 * 8 + 2]) * inv_l, __uint_as_float(o[v4 * 8 + 3]) * inv_l);
                            w.z = pack_bf16x2(__uint_as_float(o[v4 * 8 + 4]) * inv_l, __uint_as_float(o[v4 * 8 + 5]) * inv_l);
                            w.w = pack_bf16x2(__uint_as_float(o[v4 * 8 + 6]) * inv_l, __uint_as_float(o[v4 * 8 + 7]) * inv_l);
                            *reinterpret_cast<uint4*>(stage + lane * 128 + (((c * 2 + v4) ^ (lane & 7)) << 4)) = w;
                        }
                    }
                    __syncwarp();
#pragma unroll
                    for (int it = 0; it < 8; ++it) {
                        const int rrow = it * 4 + (lane >> 3), piece = lane & 7;
                        const uint4 w = *reinterpret_cast<const uint4*>(stage + rrow * 128 + ((piece ^ (rrow & 7)) << 4));
                        if (row_warp + rrow < pr.W && (!kAny || h * 64 + piece * 8 < d)) *reinterpret_cast<uint4*>(owarp + (long long)rrow * d + h * 64 + piece * 8) = w;
                    }
                    __syncwarp();
                }
            } else {
                float* pwarp = pbase + (long long)(i * kQTile + (warp & 3) * 32) * d;
#pragma unroll
                for (int h = 0; h < D / 32; ++h) {             // 32 fp32 columns per pass
                    if (kAny && h * 32 >= d) break;
#pragma unroll
                    for (int c = 0; c < 2; ++c) {
                        uint32_t o[16];
                        if (cnt_i > 0) {
                            tmem_ld16_async(tO + h * 32 + c * 16, o);
                            tmem_wait_ld16(o);
                        } else {
#pragma unroll
                            for (int e = 0; e < 16; ++e) o[e] = 0u;
                        }
#pragma unroll
                        for (int v4 = 0; v4 < 4; ++v4) {
                            float4 w;
                            w.x = __uint_as_float(o[v4 * 4 + 0]) * inv_l;
                            w.y = __uint_as_float(o[v4 * 4 + 1]) * inv_l;
                            w.z = __uint_as_float(o[v4 * 4 + 2]) * inv_l;
                            w.w = __uint_as_float(o[v4 * 4 + 3]) * inv_l;
                            *reinterpret_cast<float4*>(stage + lane * 128 + (((c * 4 + v4) ^ (lane & 7)) << 4)) = w;
                        }
                    }
                    __syncwarp();
#pragma unroll
                    for (int it = 0; it < 8; ++it) {
                        const int rrow = it * 4 + (lane >> 3), piece = lane & 7;
                        const float4 w = *reinterpret_cast<const float4*>(stage + rrow * 128 + ((piece ^ (rrow & 7)) << 4));
                        if (!kAny || h * 32 + piece * 4 < d) *reinterpret_cast<float4*>(pwarp + (long long)rrow * d + h * 32 + piece * 4) = w;
                    }
                    __syncwarp();
                }
            }
            if (whole) {
                if (store && pr.lse != nullptr) pr.lse[(long long)s.bh * pr.W + row] = lse_val;
            } else {
                pbase[(long long)kTileM * d + i * kQTile + r] = lse_val;
            }
            tc_fence_before();      // TMEM reads of O are complete before the next segment's arrive lets PV overwrite it
        }
        } else if constexpr (kShared) {                    // one Q tile: these warps only take part in the merge's barriers
            cluster_sync();
            cluster_sync();
        }
    }

    tc_fence_before();
    __syncthreads();
    if (threadIdx.x == 0 && abort_flag) atomicExch(p.status, (int)TLIN_ERR_TIMEOUT);
    if (warp == kMmaWarp) {
        tc_fence_after();
        tmem_dealloc(tmem_base, 512);
    }
}

// Combines the partial results of every (b,h) whose key tiles were split between groups.  Bound by the latency of its scattered
// reads (the partials are in L2): a row belongs to the fewest lanes that read it 16 bytes at a time, four parts of a row are on
// their way at once, a warp takes kPasses groups of rows, and nothing is shared between threads.
// Against one row per warp, 4- to 8-byte reads and the list of parts worked out by one thread before a barrier, whole calls: B1 H4
// N1024 W128 d64 10.0 -> 8.2 us, B4 H16 N8192 W256 d64 60 -> 56 us, B4 H32 N8192 W1024 d128 520 -> 503 us.  One pass is best while
// the CTAs are few (10.0 -> 8.2 us against 11.1 with four, d40 33.5 against 35.7); four from 65536 rows on (503 against 510 us).
constexpr int kMergeParts = 4;           // parts read at once
template <int D, int kPasses>
struct MergeCfg {
    static constexpr int kLanes = D / 4 < 32 ? D / 4 : 32;            // lanes per row
    static constexpr int kVecs = D / 4 / kLanes;                      // 16-byte pieces per lane
    static constexpr int kWarpRows = 32 / kLanes;
    static constexpr int kRows = 8 * kWarpRows * kPasses;             // rows per CTA
};

template <int D, bool kAny, int kPasses>
__global__ void __launch_bounds__(256)
fwd_merge_kernel(const __grid_constant__ Params p, const __grid_constant__ GroupStarts starts) {
    using M = MergeCfg<D, kPasses>;
    constexpr int kTileM = Cfg<D>::kRows;
    static_assert(kTileM % M::kRows == 0, "a CTA's rows lie in one tile");
    constexpr int kBlocksPerTile = kTileM / M::kRows;
    const int d = kAny ? p.d : D;
    const int tile_id = blockIdx.x / kBlocksPerTile;                  // bh * q_tiles + qt
    const int bh = tile_id / p.q_tiles, qt = tile_id - bh * p.q_tiles;
    // groups holding the first and the last unit of this (b,h): largest g with starts.u[g] <= x
    const long long x0 = (long long)bh * p.key_tiles, x1 = x0 + p.key_tiles - 1;
    int g_lo = (int)((float)x0 * (float)p.n_groups / (float)p.total_units);
    while (g_lo > 0 && starts.u[g_lo] > x0) --g_lo;
    while (g_lo + 1 < p.n_groups && starts.u[g_lo + 1] <= x0) ++g_lo;
    int g_hi = g_lo;
    while (g_hi + 1 < p.n_groups && starts.u[g_hi + 1] <= x1) ++g_hi;
    after_previous();
    let_next_start();
    if (g_hi == g_lo) return;                             // written directly by the attention kernel
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, piece = lane % M::kLanes;
    const int rr0 = (blockIdx.x % kBlocksPerTile) * M::kRows + warp * (M::kWarpRows * kPasses) + lane / M::kLanes;
    // slot 0 of a CTA holds its group's first segment (the group starts in this (b,h)), slot 1 a later one
    auto part_of = [&](int g) { return p.ws + ((long long)(g * p.q_tiles + qt) * 2 + (starts.u[g] >= x0 ? 0 : 1)) * (long long)kTileM * (d + 1); };
    float m[kPasses], z[kPasses];
    float4 acc[kPasses][M::kVecs];
#pragma unroll
    for (int ps = 0; ps < kPasses; ++ps) {
        m[ps] = -CUDART_INF_F;
        z[ps] = 0.f;
#pragma unroll
        for (int v = 0; v < M::kVecs; ++v) acc[ps][v] = make_float4(0.f, 0.f, 0.f, 0.f);
    }
    for (int g0 = g_lo; g0 <= g_hi; g0 += kMergeParts) {
        const float* base[kMergeParts];
#pragma unroll
        for (int i = 0; i < kMergeParts; ++i) base[i] = g0 + i <= g_hi ? part_of(g0 + i) : nullptr;
#pragma unroll
        for (int ps = 0; ps < kPasses; ++ps) {
            const int rr = rr0 + ps * M::kWarpRows;
            if (qt * kTileM + rr >= p.W) continue;
            float ls[kMergeParts];
            float4 x[kMergeParts][M::kVecs];
#pragma unroll
            for (int i = 0; i < kMergeParts; ++i) {
                ls[i] = -CUDART_INF_F;
#pragma unroll
                for (int v = 0; v < M::kVecs; ++v) x[i][v] = make_float4(0.f, 0.f, 0.f, 0.f);
                if (base[i] != nullptr) {
                    ls[i] = base[i][(long long)kTileM * d + rr];
#pragma unroll
                    for (int v = 0; v < M::kVecs; ++v) {
                        const int c = (v * M::kLanes + piece) * 4;
                        if (!kAny || c < d) x[i][v] = *reinterpret_cast<const float4*>(base[i] + (long long)rr * d + c);
                    }
                }
            }
            float mn = m[ps];
            bool empty = mn == -CUDART_INF_F;             // every part so far: the maximum alone would not see a NaN
#pragma unroll
            for (int i = 0; i < kMergeParts; ++i) {
                mn = fmaxf(mn, ls[i]);
                empty = empty && ls[i] == -CUDART_INF_F;
            }
            if (empty) continue;
            const float old = expf(m[ps] - mn);
            m[ps] = mn;
            z[ps] *= old;
#pragma unroll
            for (int v = 0; v < M::kVecs; ++v) { acc[ps][v].x *= old; acc[ps][v].y *= old; acc[ps][v].z *= old; acc[ps][v].w *= old; }
#pragma unroll
            for (int i = 0; i < kMergeParts; ++i) {
                const float w = expf(ls[i] - mn);         // -inf (empty part) -> 0
                z[ps] += w;
#pragma unroll
                for (int v = 0; v < M::kVecs; ++v) {
                    acc[ps][v].x = fmaf(w, x[i][v].x, acc[ps][v].x);
                    acc[ps][v].y = fmaf(w, x[i][v].y, acc[ps][v].y);
                    acc[ps][v].z = fmaf(w, x[i][v].z, acc[ps][v].z);
                    acc[ps][v].w = fmaf(w, x[i][v].w, acc[ps][v].w);
                }
            }
        }
    }
#pragma unroll
    for (int ps = 0; ps < kPasses; ++ps) {
        const int row = qt * kTileM + rr0 + ps * M::kWarpRows;
        if (row >= p.W) continue;
        const float inv = 1.f / z[ps];
        __nv_bfloat16* dst = reinterpret_cast<__nv_bfloat16*>(p.out) + ((long long)bh * p.W + row) * d;
#pragma unroll
        for (int v = 0; v < M::kVecs; ++v) {
            const int c = (v * M::kLanes + piece) * 4;
            if (!kAny || c < d)
                *reinterpret_cast<uint2*>(dst + c) = make_uint2(pack_bf16x2(acc[ps][v].x * inv, acc[ps][v].y * inv), pack_bf16x2(acc[ps][v].z * inv, acc[ps][v].w * inv));
        }
        if (p.lse != nullptr && piece == 0) p.lse[(long long)bh * p.W + row] = m[ps] + logf(z[ps]);
    }
}

template <int D, int kForm>
int launch_d(const void* q, const void* k, const void* v, void* out, float* lse, int B, int H, int N, int W,
             int d, int causal, const tlin_fwd_plan& plan, float* ws, long long kv_rows_alloc, cudaStream_t st, int cluster = 1) {
    using C = Cfg<D>;
    const long long bh = (long long)B * H;
    KernelMaps<false> maps;
    int rc = make_map(&maps.q, q, d, W, bh);
    if (rc == TLIN_OK) rc = make_map(&maps.k, k, d, N, bh, kQTile, kv_rows_alloc);
    if (rc == TLIN_OK) rc = make_map(&maps.v, v, d, N, bh, kQTile, kv_rows_alloc);
    if (rc != TLIN_OK) return rc;
    Params p;
    p.out = out; p.lse = lse; p.ws = ws; p.status = status_word();
    if (!p.status) return TLIN_ERR_CUDA;
    p.total_units = plan.total_units; p.n_groups = plan.n_groups; p.q_tiles = plan.q_tiles; p.key_tiles = plan.key_tiles;
    p.N = N; p.W = W; p.causal = causal; p.d = d; p.schedule = plan.schedule; p.cluster = cluster;
    p.scale_log2e = D == d ? kLog2e / sqrtf((float)d) : (float)(1.4426950408889634 / sqrt((double)d));
    static bool smem_allowed[64] = {};
    TLIN_CUDA_CHECK(allow_dynamic_smem(fwd_tc_kernel<D, kForm>, C::kSmemBytes, smem_allowed));
    if constexpr (kForm == kCluster || kForm == kAnyCluster) {
        GroupStarts none = {};              // not read
        TLIN_CUDA_CHECK(launch_overlapped_clusters(fwd_tc_kernel<D, kForm>, (unsigned)(bh * plan.q_tiles * cluster), cluster, kThreads, C::kSmemBytes, st, maps, p, none));
        count_launch();
        return TLIN_OK;
    }
    if (plan.n_groups > kMaxGroups) return TLIN_ERR_UNSUPPORTED;
    GroupStarts starts;
    fwd_group_starts(plan, &starts);
    TLIN_CUDA_CHECK(launch_overlapped(fwd_tc_kernel<D, kForm>, plan.n_ctas, kThreads, C::kSmemBytes, st, maps, p, starts));
    count_launch();
    if constexpr (kForm == kOneProblem || kForm == kAnyHead) if (plan.uses_workspace) {
        constexpr bool kAny = kForm == kAnyHead;
        const long long tiles = bh * plan.q_tiles;
        if (tiles * C::kRows >= 65536)
            TLIN_CUDA_CHECK(launch_overlapped(fwd_merge_kernel<D, kAny, 4>, (unsigned)(tiles * (C::kRows / MergeCfg<D, 4>::kRows)), 256, 0, st, p, starts));
        else
            TLIN_CUDA_CHECK(launch_overlapped(fwd_merge_kernel<D, kAny, 1>, (unsigned)(tiles * (C::kRows / MergeCfg<D, 1>::kRows)), 256, 0, st, p, starts));
        count_launch();
    }
    return TLIN_OK;
}

// Clusters of `size` CTAs that the device holds at a time (asked once per device and size).
template <int D, int kForm>
int clusters_at_a_time(int size) {
    static std::atomic<int> known[64][kMaxCluster + 1];
    static bool smem_allowed[64] = {};
    const int dev = current_device_slot();
    if (dev < 0) return 0;
    int n = known[dev][size].load(std::memory_order_relaxed);
    if (n == 0) {
        cudaLaunchConfig_t cfg = {};
        cfg.gridDim = dim3((unsigned)size);
        cfg.blockDim = dim3(kThreads);
        cfg.dynamicSmemBytes = Cfg<D>::kSmemBytes;
        cudaLaunchAttribute attr[1];
        attr[0].id = cudaLaunchAttributeClusterDimension;
        attr[0].val.clusterDim.x = (unsigned)size;
        attr[0].val.clusterDim.y = attr[0].val.clusterDim.z = 1;
        cfg.attrs = attr;
        cfg.numAttrs = 1;
        if (allow_dynamic_smem(fwd_tc_kernel<D, kForm>, Cfg<D>::kSmemBytes, smem_allowed) != cudaSuccess ||
            cudaOccupancyMaxActiveClusters(&n, fwd_tc_kernel<D, kForm>, &cfg) != cudaSuccess) {
            (void)cudaGetLastError();
            n = 0;
        }
        n += 1;                                              // 0: not asked yet
        known[dev][size].store(n, std::memory_order_relaxed);
    }
    return n - 1;
}
// Into how many shares a cluster cuts the keys of a call whose plan splits them (1: the plan's own groups and the merge kernel).  In
// key-tile times: a share, 2 to start and finish and 2 for the merge, against the groups' steps and segments and, for the merge kernel,
// 4, more with the parts that it merges and with the row's length, less where a step is longer (two PV products).  Fewer, longer shares lose what the merge saves: B4 H16 N8192 W256
// d64 (2 shares of 32 against 148 groups of 28) 57.0 -> 59.8 us, B8 H8 N6000 W200 d64 46.7 -> 48.0; the rule leaves both.
// At other head sizes also instead of whole problems, of which there are few enough here for one per CTA (at 64 and 128 a call that is
// planned whole stays whole: its result is that of the same problem in a table).
template <int D, int kForm>
int cluster_shares(const tlin_fwd_plan& plan, long long bh) {
    const long long problems = bh * plan.q_tiles, T = plan.key_tiles;
    if (problems > kDefaultSMs / 2) return 1;
    constexpr bool kAny = kForm == kAnyCluster;
    long long best_cost = T;
    if (plan.schedule == 0) {
        if (!plan.uses_workspace) return 1;
        const long long steps = (plan.total_units + plan.n_groups - 1) / plan.n_groups, parts = plan.n_groups / bh;
        best_cost = steps + 2 * (steps / T + 1) + (parts + 2) / (D == 256 ? 8 : 4) + (kAny ? 3 : D == 128 ? 5 : 4);
    } else if (!kAny) {
        return 1;
    }
    int best = 1;
    for (int shares = 2; shares <= kMaxCluster; ++shares) {
        const long long cost = (T + shares - 1) / shares + 4;
        if (cost < best_cost && problems <= clusters_at_a_time<D, kForm>(shares)) {
            best_cost = cost;
            best = shares;
        }
    }
    return best;
}

// A table of problems as one launch: every CTA walks a contiguous run or a list of whole (problem, b*h, query tile pair) units.
template <int D>
int launch_batched_d(const tlin_problem* problems, int n, const long long* starts_in, const uint16_t* order, int n_ctas, cudaStream_t st) {
    using C = Cfg<D>;
    static_assert(sizeof(KernelMaps<true>) + sizeof(Params) + sizeof(GroupStarts) < 32000, "launch parameters exceed the limit");
    KernelMaps<true> maps;
    memset(&maps, 0, sizeof(maps));
    maps.n = n;
    if (order != nullptr) {
        maps.listed = 1;
        memcpy(maps.order, order, sizeof(uint16_t) * (size_t)starts_in[n_ctas]);
    }
    long long unit = 0;
    for (int i = 0; i < n; ++i) {
        const tlin_problem& pb = problems[i];
        const long long kv_rows = pb.kv_rows > 0 ? pb.kv_rows : pb.n_keys;
        int rc = make_map(&maps.q[i], pb.q, D, pb.n_queries, pb.BH);
        if (rc == TLIN_OK) rc = make_map(&maps.k[i], pb.k, D, pb.n_keys, pb.BH, kQTile, kv_rows);
        if (rc == TLIN_OK) rc = make_map(&maps.v[i], pb.v, D, pb.n_keys, pb.BH, kQTile, kv_rows);
        if (rc != TLIN_OK) return rc;
        ProblemDev& pd = maps.prob[i];
        pd.out = pb.out; pd.lse = pb.lse; pd.unit0 = unit;
        pd.N = pb.n_keys; pd.W = pb.n_queries; pd.causal = pb.causal_window;
        pd.key_tiles = (pb.n_keys + kTileN - 1) / kTileN;
        pd.q_tiles = (pb.n_queries + kTileM - 1) / kTileM;
        unit += (long long)pb.BH * pd.q_tiles;
    }
    Params p;
    memset(&p, 0, sizeof(p));
    p.status = status_word();
    if (!p.status) return TLIN_ERR_CUDA;
    p.total_units = unit; p.n_groups = n_ctas; p.q_tiles = 1; p.key_tiles = 1; p.schedule = 1;
    p.scale_log2e = kLog2e / sqrtf((float)D);
    if (n_ctas > kMaxGroups) return TLIN_ERR_UNSUPPORTED;
    GroupStarts starts;
    for (int g = 0; g <= n_ctas; ++g) starts.u[g] = starts_in[g];
    static bool smem_allowed[64] = {};
    TLIN_CUDA_CHECK(allow_dynamic_smem(fwd_tc_kernel<D, kTable>, C::kSmemBytes, smem_allowed));
    TLIN_CUDA_CHECK(launch_overlapped(fwd_tc_kernel<D, kTable>, n_ctas, kThreads, C::kSmemBytes, st, maps, p, starts));
    count_launch();
    return TLIN_OK;
}

}  // namespace

int launch_fwd_tc_batched(const tlin_problem* problems, int n, int d, const long long* starts, const uint16_t* order, int n_ctas, cudaStream_t st) {
    if (n <= 0 || n > kMaxBatch) return TLIN_ERR_INVALID_ARG;
    if (d == 128) return launch_batched_d<128>(problems, n, starts, order, n_ctas, st);
    if (d == 64) return launch_batched_d<64>(problems, n, starts, order, n_ctas, st);
    return TLIN_ERR_UNSUPPORTED;
}

int fwd_cluster_shares(const tlin_fwd_plan& plan, long long bh, int d) {
    return d == 128 ? cluster_shares<128, kCluster>(plan, bh) : d == 64 ? cluster_shares<64, kCluster>(plan, bh)
         : d < 64 ? cluster_shares<64, kAnyCluster>(plan, bh) : d < 128 ? cluster_shares<128, kAnyCluster>(plan, bh) : cluster_shares<256, kAnyCluster>(plan, bh);
}

int launch_fwd_tc(const void* q, const void* k, const void* v, void* out, float* lse,
                  int B, int H, int N, int W, int d, int causal, const tlin_fwd_plan& plan,
                  float* ws, long long kv_rows_alloc, cudaStream_t st) {
    if (plan.tile_m != (d > 128 ? kQTile : kTileM) || plan.tile_n != kTileN) return TLIN_ERR_UNSUPPORTED;
    if ((long long)B * H * W > 0x7fffffffLL || d % 8 != 0 || d > 256) return TLIN_ERR_UNSUPPORTED;
    const long long bh = (long long)B * H;
    const int shares = fwd_cluster_shares(plan, bh, d);
    if (shares > 1) {
        if (d == 128) return launch_d<128, kCluster>(q, k, v, out, lse, B, H, N, W, d, causal, plan, ws, kv_rows_alloc, st, shares);
        if (d == 64) return launch_d<64, kCluster>(q, k, v, out, lse, B, H, N, W, d, causal, plan, ws, kv_rows_alloc, st, shares);
        if (d < 64) return launch_d<64, kAnyCluster>(q, k, v, out, lse, B, H, N, W, d, causal, plan, ws, kv_rows_alloc, st, shares);
        if (d < 128) return launch_d<128, kAnyCluster>(q, k, v, out, lse, B, H, N, W, d, causal, plan, ws, kv_rows_alloc, st, shares);
        return launch_d<256, kAnyCluster>(q, k, v, out, lse, B, H, N, W, d, causal, plan, ws, kv_rows_alloc, st, shares);
    }
    if (dealt(plan, (long long)B * H, d)) {
        if (d == 128) return launch_d<128, kDealt>(q, k, v, out, lse, B, H, N, W, d, causal, plan, ws, kv_rows_alloc, st);
        if (d == 64) return launch_d<64, kDealt>(q, k, v, out, lse, B, H, N, W, d, causal, plan, ws, kv_rows_alloc, st);
        if (d < 64) return launch_d<64, kAnyDealt>(q, k, v, out, lse, B, H, N, W, d, causal, plan, ws, kv_rows_alloc, st);
        if (d < 128) return launch_d<128, kAnyDealt>(q, k, v, out, lse, B, H, N, W, d, causal, plan, ws, kv_rows_alloc, st);
        return launch_d<256, kAnyDealt>(q, k, v, out, lse, B, H, N, W, d, causal, plan, ws, kv_rows_alloc, st);
    }
    if (d == 128) return launch_d<128, kOneProblem>(q, k, v, out, lse, B, H, N, W, d, causal, plan, ws, kv_rows_alloc, st);
    if (d == 64) return launch_d<64, kOneProblem>(q, k, v, out, lse, B, H, N, W, d, causal, plan, ws, kv_rows_alloc, st);
    if (d < 64) return launch_d<64, kAnyHead>(q, k, v, out, lse, B, H, N, W, d, causal, plan, ws, kv_rows_alloc, st);
    if (d < 128) return launch_d<128, kAnyHead>(q, k, v, out, lse, B, H, N, W, d, causal, plan, ws, kv_rows_alloc, st);
    if (d <= 256) return launch_d<256, kAnyHead>(q, k, v, out, lse, B, H, N, W, d, causal, plan, ws, kv_rows_alloc, st);
    return TLIN_ERR_UNSUPPORTED;
}

}  // namespace tlin

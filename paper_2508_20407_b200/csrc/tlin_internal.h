// Internal declarations shared by the translation units of libtlin (never installed).
#pragma once
#include <cuda_runtime.h>
#include <cuda_bf16.h>
#include <stdint.h>
#include <stdio.h>
#include <mutex>
#include "../../include/tlin.h"

namespace tlin {

constexpr int kDefaultSMs = 148;       // B200
constexpr int kTileN = 128;            // keys per tile on the tensor path
// K and V of a call that stay in L2 (126 MB) while its CTAs read them at unrelated times.  64 / 112 MiB, microseconds: 256 heads of 780
// keys, 277 rows, d = 128 (102 MB) 91 / 76; 128 x 1500, 800 rows (98 MB) 132 / 107; 64 x 3000, 2000 rows (98 MB) 156 / 145.
constexpr int64_t kKVInL2 = 112ll << 20;
constexpr int kSimtRows = 8;           // query rows and keys per tile that plans of the CUDA-core path report; its kernels take
constexpr int kSimtKeys = 32;          // tiles of their own (fwd_simt.cu: by d, the rows and the number of (b,h))
constexpr int kDecodeMaxSplits = 64;   // upper bound on the splits of a (b,h) in the decode step
constexpr int kDecodeMaxCluster = 8;   // up to this many splits are merged inside a cluster (the portable cluster size)
constexpr int kDecodeClusterKeys = 1024;   // ... when they are no longer than this
constexpr int kDecodeMinKeys = 256;    // do not split the cache finer than this
constexpr int kDecodeCtasPerSM = 3;    // 98 KB of loads in flight per SM (figures: KeyRun in decode.cu)

struct Workspace { void* ptr; size_t bytes; };
Workspace workspace();
int* status_word();                    // device address of the error word (bounded waits report here)
void count_launch(int n = 1);
void reset_launches();                 // every compute entry point starts its count at zero
int current_device_slot();             // index of the current device in per-device tables (-1: beyond them)
int forward_impl();

// cudaFuncSetAttribute(MaxDynamicSharedMemorySize) holds for the device that is current when it is called, so a kernel
// that needs more than 48 KB asks once per device.  `done` is a table of 64 flags owned by the caller (one per kernel).
template <class Kernel>
inline cudaError_t allow_dynamic_smem(Kernel kernel, int bytes, bool (&done)[64]) {
    static std::mutex mu;
    const int dev = current_device_slot();
    if (dev < 0) return cudaErrorInvalidDevice;
    std::lock_guard<std::mutex> lk(mu);
    if (done[dev]) return cudaSuccess;
    const cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
    if (e == cudaSuccess) done[dev] = true;
    return e;
}

// Work sharing of the tensor-core forward and dQ kernels.  The host works out the first unit of every group and passes the
// table to the kernel as a launch parameter (the CTAs only index it).
// Schedule 0 (units = (b,h,key tile)) and unmasked schedule 1 (units = (b,h,256-row query tile pair) problems, all of one
// cost): equal counts, group g starts at floor(g * units / groups).  Schedule 1 with the window rule: problem qt may use
// ceil((N-W+min(W,256(qt+1)))/128) key tiles; its cost is that number plus 3 (starting and finishing a problem, the masked steps on the diagonal and the step the
// pair's second tile runs alone: measured 2.6 key-tile times), and, when there
// are at least three problems per group, the groups take contiguous runs of problems by cost: every group starting where the
// cost before it reaches its share of the total, and, for problems of 10 key-tile times or more on average, moved as little
// as needed to make the costliest run as cheap as contiguous runs allow (with fewer than three problems per group the
// indivisible problems dominate and equal counts do as well).
constexpr int kMaxGroups = 192;        // groups never exceed the SM count (148 on B200); the planner clamps to this
struct GroupStarts { long long u[kMaxGroups + 1]; };   // u[g] = first unit of group g, u[n_groups] = total_units
inline long long fwd_problem_cost(int N, int W, int key_tiles, int qt, int tile_m = 256) {
    long long rows_end = (long long)(qt + 1) * tile_m;
    if (rows_end > W) rows_end = W;
    long long tiles = ((long long)N - W + rows_end + 127) / 128;
    if (tiles > key_tiles) tiles = key_tiles;
    return tiles + 3;
}
int plan_forward(int B, int H, int N, int W, int d, int causal_window, int is_f32, int num_sms, bool whole_only, tlin_fwd_plan* plan);
// fills starts->u[0 .. plan.n_groups]; plan.n_groups <= kMaxGroups
void fwd_group_starts(const tlin_fwd_plan& plan, GroupStarts* starts);

// Work sharing of the tensor-core dK/dV kernel (host and device use the same arithmetic).  Units are (b,h,key tile) in that
// order, key tiles of 128 keys, query tiles of 128 rows; with the window rule key tile t is visited by the query tiles from
// floor(max(0, 128 t - (N-W)) / 128) on, so the last key tiles of a (b,h) cost fewer steps, down to one.  Share c of G starts at
// the smallest unit u such that the steps of the units before it reach c/G of all steps.
__host__ __device__ inline long long bwd_first_unit_of_share(int N, int W, int causal, long long total_units, int key_tiles,
                                                            unsigned c, unsigned G) {
    const int T = key_tiles, Qt = (W + 127) / 128;
    if (c >= G) return total_units;
    if (!causal) return (long long)(((unsigned long long)c * (unsigned long long)total_units) / G);
    auto steps_of = [&](long long t) {
        const long long f = t * 128 - ((long long)N - W);
        return (long long)Qt - (f <= 0 ? 0 : f / 128);
    };
    long long t_full = ((long long)N - W) / 128 + 1;                 // tiles [0, t_full) visit every query tile
    if (t_full > T) t_full = T;
    long long per_bh = t_full * Qt;
    for (long long t = t_full; t < T; ++t) per_bh += steps_of(t);
    const long long n_bh = total_units / T;
    const unsigned long long target = ((unsigned long long)c * (unsigned long long)(per_bh * n_bh)) / G;
    const long long bh = (long long)(target / (unsigned long long)per_bh);
    const long long rem = (long long)(target - (unsigned long long)bh * (unsigned long long)per_bh);   // steps into this (b,h)
    long long t;
    if (rem <= t_full * Qt) {
        t = (rem + Qt - 1) / Qt;                                      // smallest t with t * Qt >= rem
    } else {
        long long cum = t_full * Qt;
        t = t_full;
        while (t < T && cum < rem) {
            cum += steps_of(t);
            ++t;
        }
    }
    return bh * T + t;
}

// Batched forward (a table of small problems in one launch).  Units are whole (problem, b*h, 256-row query tile pair)
// problems in table order; a CTA takes a contiguous run of them, the runs balanced by cost (allowed key tiles + 3 under the window rule, + 2 without) with
// the costliest run as cheap as contiguous runs allow.  prefix[x] = cost of the first x units (prefix.size() = units + 1);
// fills starts[0 .. n_ctas], every CTA non-empty (n_ctas <= units).
constexpr int kMaxBatch = 24;          // problems per launch of the batched kernel (its table travels as a launch parameter)
void balanced_run_starts(const long long* prefix, long long units, int n_ctas, long long* starts);
// With one to seven units per CTA a contiguous run is a coarse share.  Up to kMaxListedUnits units are dealt singly instead, each in
// turn, costliest first, to the CTA with the least so far, if that makes the costliest CTA cheaper than `runs` (the starts of the
// contiguous runs) does: CTA c then takes order[starts[c]] .. order[starts[c + 1] - 1], in ascending order.  Returns whether it does.
// Four requests' inner layers at d = 128 (8 heads, 1024 + 1024 rows: 256 units of 10 to 19 on 148 CTAs): costliest 30 -> 27, 56.8 -> 52.1
// us; 48 + 144 units of 6 requests (211 + 708 rows, d = 64) 28.3 -> 20.9 us; 4 x 32 heads of 300 + 1000 rows 96 -> 80 us.
constexpr int kMaxListedUnits = 1024;
bool deal_batched_units(const tlin_problem* problems, int n_problems, int n_ctas, const long long* runs, long long* starts, uint16_t* order);

// Launches of one call, and of successive calls, overlap their starts: a kernel launched here may begin while the kernel before it
// in the stream is still finishing (programmatic dependent launch), sets up what needs no memory, and waits in after_previous()
// until that kernel has completed and its writes are visible.  Every kernel launched this way calls after_previous() in all
// threads before it touches global memory, which also makes completion transitive along the stream.  let_next_start() allows
// the kernel behind it to be brought in.
#ifdef __CUDACC__
__device__ __forceinline__ void after_previous() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void let_next_start() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
#endif
template <class... Params, class... Args>
inline cudaError_t launch_overlapped_clusters(void (*kernel)(Params...), unsigned grid, unsigned cluster, unsigned block, size_t smem, cudaStream_t st,
                                              Args&&... args) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(grid);
    cfg.blockDim = dim3(block);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    attr[1].id = cudaLaunchAttributeClusterDimension;
    attr[1].val.clusterDim.x = cluster;
    attr[1].val.clusterDim.y = attr[1].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = cluster > 1 ? 2 : 1;
    return cudaLaunchKernelEx(&cfg, kernel, static_cast<Args&&>(args)...);
}
template <class... Params, class... Args>
inline cudaError_t launch_overlapped(void (*kernel)(Params...), unsigned grid, unsigned block, size_t smem, cudaStream_t st, Args&&... args) {
    return launch_overlapped_clusters(kernel, grid, 1, block, smem, st, static_cast<Args&&>(args)...);
}

#define TLIN_CUDA_CHECK(expr)                                                              \
    do {                                                                                   \
        cudaError_t e__ = (expr);                                                          \
        if (e__ != cudaSuccess) {                                                          \
            fprintf(stderr, "libtlin: %s failed: %s (%s:%d)\n", #expr,                     \
                    cudaGetErrorString(e__), __FILE__, __LINE__);                          \
            return TLIN_ERR_CUDA;                                                          \
        }                                                                                  \
    } while (0)

inline bool overlap(const void* a, int64_t a_bytes, const void* b, int64_t b_bytes) {
    const uintptr_t x = (uintptr_t)a, y = (uintptr_t)b;
    return x < y + (uint64_t)b_bytes && y < x + (uint64_t)a_bytes;
}

// The (b,h) of a call that the CUDA-core kernels are to compute after the tensor cores, found on the device: with `any` null all of them;
// otherwise none while *any is 0, else all (`all`) or those that have one of their per_bh words set.
struct Heads {
    const int* any = nullptr;
    const int* words = nullptr;
    int per_bh = 0, all = 0;
#ifdef __CUDACC__
    __device__ __forceinline__ bool none() const { return any != nullptr && *any == 0; }
    __device__ __forceinline__ bool special(long long bh) const {
        bool found = all != 0;
        const int* w = words + bh * per_bh;
#pragma unroll 1
        for (int i = 0; i < per_bh && !found; ++i) found = w[i] != 0;
        return found;
    }
    __device__ __forceinline__ bool has(long long bh) const { return any == nullptr || (*any != 0 && special(bh)); }
#endif
};
// results over an input otherwise than one (b,h) over the same (b,h) of a tensor of the same size
inline bool crosses(const void* to, int64_t to_bytes, const void* from, int64_t from_bytes) {
    return overlap(to, to_bytes, from, from_bytes) && !(to == from && to_bytes == from_bytes);
}

// ---- launchers (one per kernel family); all validate nothing: api.cu has done it ----------
int launch_fwd_simt_bf16(const void* q, const void* k, const void* v, void* out, float* lse,
                         int B, int H, int N, int W, int d, int causal, long long kv_rows_alloc, cudaStream_t st);
int launch_fwd_simt_f32(const float* q, const float* k, const float* v, float* out, float* lse,
                        int B, int H, int N, int W, int d, int causal, long long kv_rows_alloc, cudaStream_t st, const Heads& heads = {});
double fwd_simt_us(long long n_bh, int N, int W, int d, int causal);
// fp32 on the tensor cores (fwd_f32_tc.cu, bwd_f32_tc.cu): whether a call is better served there, its scratch, and the call.  It returns
// TLIN_ERR_UNSUPPORTED, with nothing launched, for several launches whose results lie over inputs.
bool fwd_f32_tensor_path(int B, int H, int N, int W, int d, int causal);
size_t fwd_f32_scratch_bytes(int B, int H, int N, int W, int d, int causal);
int launch_fwd_f32_tc(const float* q, const float* k, const float* v, float* out, float* lse, int B, int H, int N, int W, int d, int causal,
                      void* scratch, int sms, cudaStream_t st);
bool bwd_f32_tensor_path(int B, int H, int N, int W, int d, int causal);
size_t bwd_f32_scratch_bytes(int B, int H, int N, int W, int d);
int launch_bwd_f32_tc(const float* q, const float* k, const float* v, const float* out, const float* lse, const float* dout,
                      float* dq, float* dk, float* dv, int B, int H, int N, int W, int d, int causal, void* scratch, int sms, cudaStream_t st);
int launch_fwd_tc(const void* q, const void* k, const void* v, void* out, float* lse,
                  int B, int H, int N, int W, int d, int causal, const tlin_fwd_plan& plan,
                  float* ws, long long kv_rows_alloc, cudaStream_t st);   // kv_rows_alloc: rows per (b,h) of k, v (0 = N)
// CTAs per cluster that share the keys of a problem of this plan (the plan's groups are then not used), 1 without clusters
int fwd_cluster_shares(const tlin_fwd_plan& plan, long long bh, int d);
// order: null, or the units in the order of the CTAs' lists (deal_batched_units)
int launch_fwd_tc_batched(const tlin_problem* problems, int n, int d, const long long* starts, const uint16_t* order, int n_ctas, cudaStream_t st);
int launch_decode(const void* q_new, const void* k_new, const void* v_new, void* k_cache, void* v_cache,
                  void* out, float* lse, int B, int H, int Ncap, int pos, const int* pos_per_seq, int d,
                  const tlin_decode_plan& plan, int sms, float* ws, cudaStream_t st,
                  bool two_kernels = false);   // two_kernels: short steps as well (decode.cu, tlin_decode_step_static)
int launch_bwd_simt(const void* q, const void* k, const void* v, const void* out, const float* lse, const void* dout,
                    void* dq, void* dk, void* dv, int B, int H, int N, int W, int d, int causal, int is_f32, float* ws,
                    cudaStream_t st, const Heads& heads = {});           // some heads only: delta and their cleared sums are in place
// where that kernel sums dq of an fp32 call: dq itself, or behind delta in ws
float* bwd_simt_sums(const float* q, const float* k, const float* v, const float* lse, const float* dout, float* dq, long long n_bh, int N, int W, int d, float* ws);
double bwd_simt_us(long long n_bh, int N, int W, int d, int causal);
size_t bwd_workspace_bytes(long long B, long long H, long long W, int d);
int launch_bwd_tc(const void* q, const void* k, const void* v, const void* out, const float* lse, const void* dout,
                  void* dq, void* dk, void* dv, int B, int H, int N, int W, int d, int causal, const tlin_fwd_plan& plan,
                  float* ws, int num_sms, cudaStream_t st);
size_t bwd_tc_workspace_bytes(long long B, long long H, long long W, int d, const tlin_fwd_plan& plan);
// dK, dV and dQ in one tensor-core kernel (d = 128): scores computed once, dQ summed in an fp32 buffer of the workspace
int launch_bwd_fused(const void* q, const void* k, const void* v, const void* out, const float* lse, const void* dout,
                     void* dq, void* dk, void* dv, int B, int H, int N, int W, int d, int causal, float* ws, int num_sms, cudaStream_t st);
size_t bwd_fused_workspace_bytes(long long B, long long H, long long W, int d);
int backward_impl();
int decode_table_max_problems();
int launch_decode_table(const tlin_decode_problem* problems, int n, int d, cudaStream_t st);
int launch_decode_fp8(const void* q_new, const void* k_new, const void* v_new, void* k_cache, void* v_cache,
                      const float* k_scale, const float* v_scale, void* out, float* lse, int B, int H, int Ncap, int pos,
                      int d, const tlin_decode_plan& plan, int sms, float* ws, cudaStream_t st);
int launch_merge_pair_bf16(const void* oa, const float* la, const void* ob, const float* lb,
                           void* out, float* lse, int64_t rows, int d, cudaStream_t st);
int launch_merge_pair_f32(const float* oa, const float* la, const float* ob, const float* lb,
                          float* out, float* lse, int64_t rows, int d, cudaStream_t st);

}  // namespace tlin

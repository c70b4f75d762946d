// Shared declarations of the libspeca translation units (device helpers, launch
// parameter blocks, workspace layout).  Nothing here is visible at the C ABI.
#pragma once

#include <cuda_runtime.h>
#include <cuda_bf16.h>
#include <stdint.h>

#include <atomic>

#include "../../include/speca.h"

namespace speca {

// ---------------------------------------------------------------------------
// Workspace layout (device scratch handed in by the caller).
//   [0, 2048)                    control words (work-queue counters, optional profiling slots)
//   [2048, 2048 + 4*Bpad)        seq_n[b]: node count of sequence b, or -1 if the
//                                sequence failed validation and must be skipped
//   then int32 arrays of Tpad words: plan[T], depth[T], anc[T][4], anc2[T][4], up[T][4], set[T][2]
//   after the kNodeWords node arrays, used only by the fused commit-and-verify call:
//   pend[B][kPendWords]: validated length of the pending accepted path, its local node
//   indices, and the sequence's offset in the previous draft's packed arrays
// Every region starts on a 256-byte boundary.
// ---------------------------------------------------------------------------
constexpr size_t kCtrlBytes = 2048;
constexpr int kNodeWords = 16;          // int32 words of scratch reserved per packed node
constexpr int kPendWords = 12;          // per sequence: path length, 8 local node indices, offset, spare

__host__ __device__ inline size_t align256(size_t x) { return (x + 255) & ~size_t(255); }

struct Workspace {
    int32_t *ctrl;      // [64]
    int32_t *seq_n;     // [B]
    int32_t *plan;      // [T]   packed schedule entries, in processing order per sequence
    int32_t *depth;     // [T]   depth computed from parent[]
    int32_t *anc;       // [T][4] per node: depth | position << 8, ancestor node indices of levels 1..12 (one byte each)
    int32_t *anc2;      // [T][4] per node: ancestor node indices of levels 13..15, spare
    int32_t *up;        // (plan_paths_only) [T][4] per node: its root path upward, itself first, one byte per step (the first 16), zero past the end
    int32_t *set;       // (plan_paths_only) [T][2] per node: the nodes of its root path as a set (those below 64)
    int32_t *pend;      // [B][kPendWords] pending accepted path (fused commit-and-verify only)
};

inline size_t workspace_bytes(int32_t batch, int32_t total_nodes)
{
    return kCtrlBytes + align256(size_t(batch) * 4) + align256(size_t(total_nodes) * 4) * kNodeWords +
           align256(size_t(batch) * kPendWords * 4);
}

inline Workspace carve_workspace(void *base, int32_t batch, int32_t total_nodes)
{
    Workspace w;
    char *p = static_cast<char *>(base);
    w.ctrl = reinterpret_cast<int32_t *>(p);
    p += kCtrlBytes;
    w.seq_n = reinterpret_cast<int32_t *>(p);
    p += align256(size_t(batch) * 4);
    size_t tb = align256(size_t(total_nodes) * 4);
    w.plan = reinterpret_cast<int32_t *>(p);
    w.depth = reinterpret_cast<int32_t *>(p + tb);
    w.anc = reinterpret_cast<int32_t *>(p + 2 * tb);
    w.anc2 = reinterpret_cast<int32_t *>(p + 6 * tb);
    w.up = reinterpret_cast<int32_t *>(p + 10 * tb);
    w.set = reinterpret_cast<int32_t *>(p + 14 * tb);
    w.pend = reinterpret_cast<int32_t *>(p + kNodeWords * tb);
    return w;
}

// Root path of node i of a sequence of at most 64 nodes, upward and as a set, and its depth, into the workspace; the depth.
template <class Int> __device__ __forceinline__ int write_path(const Workspace &ws, int base, int i, const Int *par)
{
    uint32_t up[4] = {0u, 0u, 0u, 0u}, lo = 0u, hi = 0u;
    int d = 0;
    for (int a = i; a >= 0; a = par[a], ++d) {
        const uint32_t byte = uint32_t(a) << (8 * (d & 3));
#pragma unroll
        for (int w = 0; w < 4; ++w) up[w] |= (d >> 2) == w ? byte : 0u;
        if (a < 32) lo |= 1u << a;
        else hi |= 1u << (a - 32);
    }
    ws.depth[base + i] = d;
    reinterpret_cast<int4 *>(ws.up)[base + i] = make_int4(int(up[0]), int(up[1]), int(up[2]), int(up[3]));
    reinterpret_cast<int2 *>(ws.set)[base + i] = make_int2(int(lo), int(hi));
    return d;
}

// Packed schedule entry written by the plan kernel, one per node, in the order
// the serial tree walk processes the nodes of a sequence.
//   bits  0..15  node index (local to the sequence)
//   bits 16..19  load code: 0 = parent state is already in registers,
//                1..14 = reload from on-chip slot (code-1), 15 = reload S0 from HBM
//   bits 20..23  save code: 0 = none, 1..14 = store the new state to slot (code-1)
//   bit  24      leaf: emit o only, leave the register state at the parent's
constexpr int kPlanLoadShift = 16, kPlanSaveShift = 20, kPlanLeafBit = 1 << 24;
constexpr int kLoadFromS0 = 15;

// Launch parameter block shared by the kernels.
struct Params {
    int32_t L, B, H, T, DV;
    float scale;
    int32_t max_depth, max_nodes;
    int32_t no_erase;            // SPECA_RULE_GATED_NO_ERASE: the corrected value is u = beta v (no read-out of the state)
    float *S;                    // in/out for decode and commit
    const float *S0;             // read-only for verify
    const __nv_bfloat16 *q, *k, *v;
    const float *alpha, *beta;
    float *o, *u;
    const int32_t *node_offsets, *parent, *depth_in;
    const int32_t *path_idx, *path_len;
    // pending commit of the fused call: records of the previous draft (keys, gates, u) and its packing
    const __nv_bfloat16 *pk;
    const float *palpha, *pu;
    const int32_t *pnode_offsets, *pparent;
    int32_t Tp;
    int32_t *status;
    Workspace ws;
    int32_t n_slots;             // on-chip state slots available to the tree walk
    int32_t skip_nodes;          // verify: sequences of at most this many nodes are another kernel's (the plan gives them no nodes)
    int32_t plan_paths_only;     // plan: root paths upward and as sets instead of the processing order and what goes with it
    int32_t long_min;            // commit: accepted paths of long_min..8 nodes are taken by the tensor-core kernel (0: none)
};

// Launchers implemented per translation unit; each returns a cudaError_t-compatible int.
int launch_plan(const Params &p, cudaStream_t st);
int launch_decode(const Params &p, int d_k, cudaStream_t st);
int launch_verify_serial(const Params &p, int d_k, bool chain, cudaStream_t st);
int launch_commit(const Params &p, int d_k, cudaStream_t st);
// commit of paths of p.long_min..8 nodes on warp-level MMAs (the token-by-token kernel skips those sequences)
bool commit_long_supported(const Params &p, int d_k);
int launch_commit_long(const Params &p, int d_k, cudaStream_t st);
void commit_long_set_min_tiles_per_warp(int n);
bool factorized_supported(const speca_dims *d);
bool factorized_fused_supported(const speca_dims *d);
int launch_verify_factorized(const Params &p, int d_k, bool fused, bool comp, cudaStream_t st);
void factorized_set_withhold(int on);
// small draft trees, state streamed straight into registers: largest sequence it should take, and the launch
int direct_limit(const Params &p, int d_k, int most, bool piped, bool chain);
int launch_verify_direct(const Params &p, int d_k, int most, int limit, cudaStream_t st);
bool effective_supported(const speca_dims *d);
int launch_verify_effective(const Params &p, int d_k, cudaStream_t st);
void effective_set_withhold(int on);
int launch_pending_check(const Params &p, int max_len, cudaStream_t st);
int launch_mask_to_parent(int32_t B, int32_t N, const uint8_t *mask, const int32_t *node_offsets, int32_t *parent,
                          int32_t *status, cudaStream_t st);
int launch_chain_decompose(int32_t B, int32_t N, const int32_t *node_offsets, const int32_t *parent,
                           int32_t *chain_head, int32_t *n_chains, int32_t *status, cudaStream_t st);
int launch_prune(int32_t B, int32_t N, float tau, int32_t budget, const int32_t *node_offsets, const int32_t *parent,
                 const float *logp, int32_t *out_offsets, int32_t *out_parent, int32_t *out_index, int32_t *status,
                 cudaStream_t st);
int launch_conv_commit(int32_t L, int32_t B, int32_t channels, int32_t W, int32_t T, int32_t max_depth, void *C,
                       const void *x, const int32_t *node_offsets, const int32_t *path_idx, const int32_t *path_len,
                       int32_t *status, cudaStream_t st);
int launch_accept(int32_t B, int32_t max_depth, const int32_t *node_offsets, const int32_t *parent,
                  const int32_t *draft_tok, const int32_t *target_tok, const int32_t *root_target_tok,
                  int32_t *path_idx, int32_t *path_len, int32_t *next_tok, int32_t *status,
                  cudaStream_t st);
int launch_stochastic_accept(int32_t B, int32_t max_depth, const int32_t *node_offsets, const int32_t *parent,
                             const float *p_target, const float *p_draft, const float *uniform,
                             int32_t *path_idx, int32_t *path_len, int32_t *status, cudaStream_t st);

// SM count per device (asked once per device)
inline int sm_count_of_current_device()
{
    static std::atomic<int> cache[64];
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) return 0;
    const bool cached = dev >= 0 && dev < 64;
    int sms = cached ? cache[dev].load(std::memory_order_relaxed) : 0;
    if (sms == 0) {
        if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) return 0;
        if (cached) cache[dev].store(sms, std::memory_order_relaxed);
    }
    return sms;
}

// ---------------------------------------------------------------------------
// Overlapped launches (programmatic dependent launch).  A round is a handful of kernels on one stream, and between two of
// them the device used to sit idle while one drained and the next was set up.  Every kernel here first waits until the
// kernel in front of it has completed and its writes are visible, and only then lets the one behind it be set up, beside
// its own last wave of blocks.  A kernel is thus already there while the one before it still writes what it is going to
// read.  Loads through the read-only path (__ldg, const __restrict__ parameters, ld.global.nc) ask for data that nobody
// writes while the kernel is there, and the compiler may move them above the wait: no kernel launched this way has any, it
// reads with plain loads.
// Kernels that are not launched this way, the caller's own among them, are waited for and wait as ever.  The persistent
// kernels of large calls are launched plainly and carry none of this: the wait alone changed what the compiler made of
// them (one fused single-pass call of 32 ragged sequences 888 us, with the wait 902, overlapped 915-935).
// ---------------------------------------------------------------------------
__device__ __forceinline__ void wait_for_previous_kernel() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void let_next_kernel_in() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
__device__ __forceinline__ void after_previous_kernel()
{
    wait_for_previous_kernel();
    let_next_kernel_in();
}

template <class... P, class... A>
inline cudaError_t launch(void (*kernel)(P...), unsigned grid, unsigned block, size_t smem, cudaStream_t st, const A &...args)
{
    cudaLaunchAttribute attr{};
    attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr.val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3(grid);
    cfg.blockDim = dim3(block);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cfg.attrs = &attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kernel, P(args)...);
}

// asks for 16-byte aligned memory into L2; reads nothing into the SM
__device__ __forceinline__ void prefetch_l2(const void *p, uint32_t bytes)
{
    asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(p), "r"(bytes) : "memory");
}

// Number of on-chip state slots the light-children-first walk can need for a tree of
// at most n nodes: a node saves its state only if it has two children with
// children of their own (subtree >= 5 nodes) and every live slot at least halves
// the remaining subtree.
inline int tree_slots_needed(int n)
{
    int s = 0;
    while (n >= 5) { ++s; n = (n - 1) / 2; }
    return s;
}

}  // namespace speca

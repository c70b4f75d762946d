// Integer kernels: topology validation + walk schedule ("plan"), and greedy acceptance.
//
// The plan is computed once per verify call and shared by every layer, head and
// value tile of a sequence.  It turns the parent-pointer array (Section 4.2) into a
// depth-first processing order in which, at every node, children are visited in
// ascending order of subtree size.  This is the heavy-path idea of the
// chain-decomposed schedule (Section 4.3) used as a traversal order: the state of a
// branching node is parked on chip only while its lighter subtrees are walked and is
// released when its heaviest child starts, so a handful of slots suffice and no
// boundary state ever goes to HBM.
#include "speca_common.cuh"

namespace speca {

namespace {

constexpr int kPlanThreads = 128;

// One CTA per sequence.  Dynamic smem: 6 int32 arrays of max_nodes (+1).
__global__ void __launch_bounds__(kPlanThreads)
plan_kernel(const int32_t *node_offsets, const int32_t *parent,
            const int32_t *depth_in, int32_t B, int32_t T, int32_t max_depth,
            int32_t max_nodes, int32_t skip_nodes, int32_t paths_only, int32_t n_slots, Workspace ws, int32_t *status)
{
    after_previous_kernel();
    extern __shared__ int32_t sm[];
    const int b = blockIdx.x;
    const int tid = threadIdx.x;
    __shared__ int32_t s_flag;

    if (b == 0 && tid < 64) ws.ctrl[tid] = 0;          // reset the work-queue counters
    const int base = node_offsets[b];
    const int n = node_offsets[b + 1] - base;
    int fault = 0;
    if (base < 0 || n < 0 || base + n > T || (b == B - 1 && base + n != T) || (b == 0 && base != 0))
        fault = SPECA_STATUS_BAD_OFFSETS;
    else if (n > max_nodes)
        fault = SPECA_STATUS_TOO_MANY;
    if (fault) {
        if (tid == 0) { atomicOr(status, fault); ws.seq_n[b] = -1; }
        return;
    }
    if (n <= skip_nodes) {                             // verified by the kernel for small trees, which checks them itself
        if (tid == 0) ws.seq_n[b] = 0;
        return;
    }
    int32_t *par = sm;                       // [n]
    int32_t *size = par + max_nodes;         // [n]   subtree size
    int32_t *bef = size + max_nodes;         // [n]   total size of siblings visited before this node
    int32_t *nlc = bef + max_nodes;          // [n+1] children with children, index shifted by one (slot 0 = committed state)
    int32_t *ldf = nlc + max_nodes + 1;      // [n]   1 if an earlier sibling has children (register state lost)
    int32_t *posn = ldf + max_nodes;         // [n]   position of node i in the processing order

    if (tid == 0) s_flag = 0;
    for (int i = tid; i < n; i += kPlanThreads) { size[i] = 0; nlc[i + 1] = 0; }
    if (tid == 0) nlc[0] = 0;
    __syncthreads();
    for (int i = tid; i < n; i += kPlanThreads) {
        int p = parent != nullptr ? parent[base + i] : i - 1;      // no parent array: chain
        par[i] = p;
        if (p < -1 || p >= i) atomicOr(&s_flag, SPECA_STATUS_BAD_PARENT);
    }
    __syncthreads();
    if (s_flag) {
        if (tid == 0) { atomicOr(status, s_flag); ws.seq_n[b] = -1; }
        return;
    }
    if (paths_only) {
        // all the effective-query kernel asks for (sequences of at most 64 nodes): the root path of every node, upward and
        // as a set.  The schedule below takes three more passes over the tree: 11.6 us for 32 trees of 8..64 nodes, this
        // one 3.5 us, in front of 0.5 ms of verification.
        int flag = 0;
        for (int i = tid; i < n; i += kPlanThreads) {
            const int d = write_path(ws, base, i, par);
            if (d > max_depth) flag |= SPECA_STATUS_TOO_DEEP;
            if (depth_in != nullptr && depth_in[base + i] != d) flag |= SPECA_STATUS_BAD_DEPTH;
        }
        if (flag) atomicOr(status, flag);
        const int bad = __syncthreads_or(flag);
        if (tid == 0) ws.seq_n[b] = bad ? -1 : n;
        return;
    }
    // depth and subtree sizes: every node adds itself to all nodes on its root path
    for (int i = tid; i < n; i += kPlanThreads) {
        int d = 0;
        for (int a = i; a >= 0; a = par[a]) { atomicAdd(&size[a], 1); ++d; }
        ws.depth[base + i] = d;
        if (d > max_depth) atomicOr(&s_flag, SPECA_STATUS_TOO_DEEP);
        if (depth_in != nullptr && depth_in[base + i] != d) atomicOr(&s_flag, SPECA_STATUS_BAD_DEPTH);
    }
    __syncthreads();
    if (s_flag) {
        if (tid == 0) { atomicOr(status, s_flag); ws.seq_n[b] = -1; }
        return;
    }
    for (int i = tid; i < n; i += kPlanThreads) {
        const int p = par[i], sz = size[i];
        if (sz > 1) atomicAdd(&nlc[p + 1], 1);
        int before = 0, lost = 0;
        for (int s = 0; s < n; ++s) {
            if (s == i || par[s] != p) continue;
            const int ss = size[s];
            if (ss < sz || (ss == sz && s < i)) { before += ss; lost |= (ss > 1); }
        }
        bef[i] = before;
        ldf[i] = lost;
    }
    __syncthreads();
    for (int i = tid; i < n; i += kPlanThreads) {
        int pos = -1, slot = 0, first = 0;
        for (int c = i; c >= 0; c = par[c]) {
            pos += 1 + bef[c];
            const int a = par[c];
            if (a >= 0 && nlc[a + 1] >= 2 && bef[c] + size[c] != size[a] - 1) {
                ++slot;                                   // a's parked state is live while we are below c
                if (c == i) first = 1;
            }
        }
        const int leaf = (size[i] == 1);
        int entry = i;
        if (ldf[i]) {
            const int p = par[i];
            entry |= (p < 0 ? kLoadFromS0 : 1 + (slot - first)) << kPlanLoadShift;
        }
        if (!leaf && nlc[i + 1] >= 2) {
            entry |= (1 + slot) << kPlanSaveShift;
            if (1 + slot > n_slots) atomicOr(&s_flag, SPECA_STATUS_TOO_MANY);
        }
        if (leaf) entry |= kPlanLeafBit;
        ws.plan[base + pos] = entry;
        posn[i] = pos;
    }
    __syncthreads();
    // Per node: depth, position in the processing order, a leaf flag, and the node's ancestors by depth
    // (one byte each; meaningful for sequences of <= 256 nodes and depth <= 16, which is all
    // the factorised route accepts).  Level j (0 = child of the committed state) of the first
    // record sits in byte j % 4 of word 1 + j / 4 for j < 12; levels 12..14 are in the second.
    for (int i = tid; i < n; i += kPlanThreads) {
        int d = 0;
        for (int a = i; a >= 0; a = par[a]) ++d;
        uint32_t w[4] = {0u, 0u, 0u, 0u};
        int j = d - 1;
        for (int a = par[i]; a >= 0; a = par[a]) {
            --j;
            if (j < 16) w[j >> 2] |= (uint32_t(a) & 0xffu) << (8 * (j & 3));
        }
        int4 rec, rec2;
        rec.x = d | (posn[i] << 8) | (size[i] == 1 ? 1 << 16 : 0);         // bit 16: leaf (its u is nobody's ancestor term)
        rec.y = int(w[0]);
        rec.z = int(w[1]);
        rec.w = int(w[2]);
        rec2.x = int(w[3]);
        rec2.y = rec2.z = rec2.w = 0;
        reinterpret_cast<int4 *>(ws.anc)[base + i] = rec;
        reinterpret_cast<int4 *>(ws.anc2)[base + i] = rec2;
    }
    __syncthreads();
    if (tid == 0) {
        if (s_flag) { atomicOr(status, s_flag); ws.seq_n[b] = -1; }
        else ws.seq_n[b] = n;
    }
}

// One warp per sequence.  Each lane takes nodes t = lane, lane+32, ... and walks t's
// root path checking every token against the prediction made at its parent.
// Parents, and whether a node's token is the one predicted at its parent, are staged in shared memory for up to kAcceptNodes
// nodes: the loads of a node's three words are then in flight together, and a step up the path is one read of shared memory
// instead of three dependent ones of global memory (128 sequences of 8..64 nodes 4.8 -> 3.6 us, one of 8 nodes 2.2 -> 1.8).
// Larger sequences are walked in place.
constexpr int kAcceptNodes = 128;
__global__ void __launch_bounds__(128)
accept_kernel(int32_t B, int32_t max_depth, const int32_t *node_offsets,
              const int32_t *parent, const int32_t *draft_tok,
              const int32_t *target_tok, const int32_t *root_target_tok,
              int32_t *__restrict__ path_idx, int32_t *__restrict__ path_len,
              int32_t *__restrict__ next_tok, int32_t *status)
{
    after_previous_kernel();
    const int b = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
    const int lane = threadIdx.x & 31;
    if (b >= B) return;
    const int base = node_offsets[b];
    const int n = node_offsets[b + 1] - base;
    const int root_pred = root_target_tok[b];
    int fault = 0;
    if (base < 0 || n < 0) fault = SPECA_STATUS_BAD_OFFSETS;
    __shared__ int32_t s_target[4][kAcceptNodes];
    __shared__ int16_t s_step[4][kAcceptNodes];        // parent, or kStop - parent where the walk ends at this node's token
    constexpr int kStop = -16, kBad = -4;              // (kBad: no parent of this node)
    int32_t *target = s_target[threadIdx.x >> 5];
    int16_t *step = s_step[threadIdx.x >> 5];
    const bool staged = !fault && n <= kAcceptNodes;
    // best = (depth << 16) | (0xffff - index): max picks the deepest, then the lowest index
    int best = -1;
    if (staged) {
        int pa[kAcceptNodes / 32], draft[kAcceptNodes / 32];
#pragma unroll
        for (int k = 0; k < kAcceptNodes / 32; ++k) {
            const int t = 32 * k + lane;
            if (t < n) {
                pa[k] = parent[base + t];
                draft[k] = draft_tok[base + t];
                target[t] = target_tok[base + t];
            }
        }
        __syncwarp();
#pragma unroll
        for (int k = 0; k < kAcceptNodes / 32; ++k) {
            const int t = 32 * k + lane;
            if (t < n) {
                const int p = pa[k];
                const bool bad = p < -1 || p >= t;
                const int pred = bad ? 0 : p < 0 ? root_pred : target[p];
                step[t] = int16_t(bad ? kBad : draft[k] == pred ? p : kStop - p);
            }
        }
        __syncwarp();
        for (int t = lane; t < n; t += 32) {
            int d = 0, a = t;
            while (a >= 0) {
                a = step[a];
                if (a < -1) break;
                if (++d > max_depth) { fault |= SPECA_STATUS_TOO_DEEP; a = kStop; break; }
            }
            if (a == kBad) fault |= SPECA_STATUS_BAD_PARENT;
            if (a == -1) best = max(best, (d << 16) | (0xffff - t));
        }
    } else if (!fault) {
        for (int t = lane; t < n; t += 32) {
            int d = 0, ok = 1;
            for (int a = t; a >= 0;) {
                const int p = parent[base + a];
                if (p < -1 || p >= a) { fault |= SPECA_STATUS_BAD_PARENT; ok = 0; break; }
                const int pred = (p < 0) ? root_pred : target_tok[base + p];
                if (draft_tok[base + a] != pred) { ok = 0; break; }
                if (++d > max_depth) { fault |= SPECA_STATUS_TOO_DEEP; ok = 0; break; }
                a = p;
            }
            if (ok && t <= 0xffff) best = max(best, (d << 16) | (0xffff - t));
        }
    }
    if (n > 0x10000) fault |= SPECA_STATUS_TOO_MANY;
    best = __reduce_max_sync(0xffffffffu, best);
    fault = __reduce_or_sync(0xffffffffu, fault);
    if (fault) {                       // skip the sequence: nothing accepted
        if (lane == 0) atomicOr(status, fault);
        best = -1;
    }
    const int len = best < 0 ? 0 : (best >> 16);
    int node = best < 0 ? -1 : 0xffff - (best & 0xffff);
    if (lane == 0) {
        path_len[b] = len;
        next_tok[b] = (node < 0) ? root_pred : staged ? target[node] : target_tok[base + node];
    }
    // lane d writes entry d of the path; every lane walks
    int mine = -1;
    for (int d = len - 1; d >= 0; --d) {
        if (d == lane) mine = node;
        node = staged ? step[node] : parent[base + node];
    }
    if (lane < max_depth) path_idx[b * max_depth + lane] = mine;
}

// Stochastic posterior selection given per-node probabilities: one warp per sequence.
// Node t passes its own test iff uniform[t] * p_draft[t] < p_target[t] (uniform < min(1, p/q),
// written without the division; one fp32 product and one comparison).  From the committed state
// the walk takes, among the children of the current node in ascending index, the first that
// passes, and stops when none does.  A node is therefore on the accepted path iff it and all
// its ancestors are "chosen": passing, with no passing sibling of lower index.
__global__ void __launch_bounds__(128)
stochastic_accept_kernel(int32_t B, int32_t max_depth, const int32_t *node_offsets,
                         const int32_t *parent, const float *p_target,
                         const float *p_draft, const float *uniform,
                         int32_t *__restrict__ path_idx, int32_t *__restrict__ path_len, int32_t *status)
{
    after_previous_kernel();
    const int b = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
    const int lane = threadIdx.x & 31;
    if (b >= B) return;
    const int base = node_offsets[b];
    const int n = node_offsets[b + 1] - base;
    int fault = 0;
    if (base < 0 || n < 0) fault = SPECA_STATUS_BAD_OFFSETS;
    if (n > 0x10000) fault |= SPECA_STATUS_TOO_MANY;
    auto passes = [&](int t) { return __fmul_rn(uniform[base + t], p_draft[base + t]) < p_target[base + t]; };
    // Parents and, of every node (and the committed state, entry 0), the first child that passes are staged in shared memory
    // for up to kStochNodes nodes: a walk that chases parents and lower siblings through global memory is a chain of loads of
    // half a microsecond each, and a search through the lower siblings one of as many reads of shared memory (128 trees of
    // 24..64 nodes: 15.0 us in place, 7.6 searching, 3.7 so).  Larger sequences are walked in place.
    constexpr int kStochNodes = 256;
    __shared__ int16_t s_par[4][kStochNodes];
    __shared__ int32_t s_first[4][kStochNodes + 1];
    int16_t *par = s_par[threadIdx.x >> 5];
    int32_t *first = s_first[threadIdx.x >> 5];
    const bool staged = !fault && n <= kStochNodes;
    int best = -1;                     // (depth << 16) | (0xffff - index) of the deepest node whose root path is all chosen
    if (staged) {
        for (int t = lane; t <= n; t += 32) first[t] = kStochNodes;
        __syncwarp();
#pragma unroll 2
        for (int t = lane; t < n; t += 32) {
            const int pa = parent[base + t];
            const bool pass = passes(t);
            const bool bad = pa < -1 || pa >= t;
            par[t] = int16_t(bad ? -2 : pa);
            if (pass && !bad) atomicMin(&first[pa + 1], t);
        }
        __syncwarp();
        for (int t = lane; t < n; t += 32) {
            int d = 0, ok = 1;
            for (int a = t; a >= 0;) {
                const int pa = par[a];
                if (pa < -1) { fault |= SPECA_STATUS_BAD_PARENT; ok = 0; break; }
                if (first[pa + 1] != a) { ok = 0; break; }         // fails, or a sibling of lower index passes
                if (++d > max_depth) { fault |= SPECA_STATUS_TOO_DEEP; ok = 0; break; }
                a = pa;
            }
            if (ok) best = max(best, (d << 16) | (0xffff - t));
        }
    } else if (!fault) {
        for (int t = lane; t < n; t += 32) {
            int d = 0, ok = 1;
            for (int a = t; a >= 0;) {
                const int pa = parent[base + a];
                if (pa < -1 || pa >= a) { fault |= SPECA_STATUS_BAD_PARENT; ok = 0; break; }
                if (!passes(a)) { ok = 0; break; }
                // a lower-index sibling that passes is taken instead
                for (int s2 = pa + 1; s2 < a; ++s2)
                    if (parent[base + s2] == pa && passes(s2)) { ok = 0; break; }
                if (!ok) break;
                if (++d > max_depth) { fault |= SPECA_STATUS_TOO_DEEP; ok = 0; break; }
                a = pa;
            }
            if (ok) best = max(best, (d << 16) | (0xffff - t));
        }
    }
    best = __reduce_max_sync(0xffffffffu, best);
    fault = __reduce_or_sync(0xffffffffu, fault);
    if (fault) {                       // skip the sequence: nothing accepted
        if (lane == 0) atomicOr(status, fault);
        best = -1;
    }
    const int len = best < 0 ? 0 : (best >> 16);
    int node = best < 0 ? -1 : 0xffff - (best & 0xffff);
    if (lane == 0) path_len[b] = len;
    int mine = -1;                     // lane d writes entry d of the path; every lane walks
    for (int d = len - 1; d >= 0; --d) {
        if (d == lane) mine = node;
        node = staged ? par[node] : parent[base + node];
    }
    if (lane < max_depth) path_idx[b * max_depth + lane] = mine;
}

// Pending accepted paths of the fused commit-and-verify call, one thread per sequence:
// the same checks the stand-alone commit makes (length, node range, parent chain when the
// parent array is given), plus a node count within max_nodes.  A bad path is reported and
// recorded with length 0, so the sequence's state is not advanced; a good one is stored as
// local node indices (words 1..8) and the sequence's offset in the previous draft's packed
// arrays (word 9).
__global__ void __launch_bounds__(128)
pending_check_kernel(int32_t B, int32_t Tp, int32_t max_depth, int32_t max_len, int32_t max_nodes,
                     const int32_t *pnode_offsets, const int32_t *pparent,
                     const int32_t *path_idx, const int32_t *path_len,
                     int32_t *__restrict__ pend, int32_t *status)
{
    after_previous_kernel();
    const int b = blockIdx.x * blockDim.x + threadIdx.x;
    if (b >= B) return;
    int32_t *rec = pend + b * kPendWords;
    const int len = path_len[b];
    const int base = pnode_offsets[b];
    const int n = pnode_offsets[b + 1] - base;
    int fault = 0;
    if (len < 0 || len > max_depth || len > max_len) fault = SPECA_STATUS_TOO_DEEP;
    else if (len > 0 && (base < 0 || n < 0 || base + n > Tp)) fault = SPECA_STATUS_BAD_OFFSETS;
    else if (len > 0 && n > max_nodes) fault = SPECA_STATUS_TOO_MANY;
    int prev = -1;
    for (int d = 0; d < len && !fault; ++d) {
        const int t = path_idx[b * max_depth + d];
        if (t < 0 || t >= n) fault = SPECA_STATUS_BAD_PATH;
        else if (pparent != nullptr && pparent[base + t] != prev) fault = SPECA_STATUS_BAD_PATH;
        if (!fault) rec[1 + d] = t;
        prev = t;
    }
    if (fault) atomicOr(status, fault);
    rec[0] = fault ? 0 : len;
    rec[9] = base;
}

// Convolution-state commit, a thread per kConvPieces pieces of 8 channels of one (layer, sequence).  A thread reads the
// W rows that make up the new register (old rows and accepted inputs) into registers, then writes them,
// so the in-place update never reads a row it has already overwritten.  The path is asked for together with its length, an
// entry a lane, and checked by the warp.  All rows of a thread's pieces are in flight together, and a row of many channels is
// spread over several CTAs (3072 x 3 rows of 8192 channels: 42.5 us with a CTA per (layer, sequence) and a piece at a time,
// 37.2 = 6.1 TB/s now).
constexpr int kConvMaxWidth = 8, kConvPieces = 2;
template <int MAXW>
__global__ void __launch_bounds__(256)
conv_commit_kernel(int32_t B, int32_t vec, int32_t parts, int32_t W, int32_t T, int32_t max_depth, uint4 *__restrict__ C,
                   const uint4 *x, const int32_t *node_offsets,
                   const int32_t *path_idx, const int32_t *path_len, int32_t *status)
{
    after_previous_kernel();
    const int part = blockIdx.x % parts, l = blockIdx.x / parts / B, b = blockIdx.x / parts % B, lane = threadIdx.x & 31;
    const int A = path_len[b];
    const int entry = lane < max_depth ? path_idx[b * max_depth + lane] : 0;
    const int base = node_offsets[b], n = node_offsets[b + 1] - base;
    if (A == 0) return;
    int fault = 0;
    if (A < 0 || A > max_depth) fault = SPECA_STATUS_TOO_DEEP;
    else if (base < 0 || n < 0 || base + n > T) fault = SPECA_STATUS_BAD_OFFSETS;
    else if (__any_sync(0xffffffffu, lane < A && (entry < 0 || entry >= n))) fault = SPECA_STATUS_BAD_PATH;
    if (fault) {
        if (threadIdx.x == 0 && l == 0 && part == 0) atomicOr(status, fault);
        return;
    }
    uint4 *Cb = C + (size_t(l) * B + b) * W * vec;
    const uint4 *xb = x + (size_t(l) * T + base) * vec;
    const int c0 = part * (256 * kConvPieces) + threadIdx.x;    // this thread's pieces: c0, c0 + 256
    uint4 row[kConvPieces][MAXW];
#pragma unroll
    for (int w = 0; w < MAXW; ++w) {
        const int s = A + w;                                    // index in (old rows, accepted rows); the last W are kept
        const int node = __shfl_sync(0xffffffffu, entry, s >= W ? (s - W) & 31 : 0);
        if (w < W) {
            const uint4 *src = s < W ? Cb + s * vec : xb + size_t(node) * vec;
#pragma unroll
            for (int i = 0; i < kConvPieces; ++i)
                if (c0 + 256 * i < vec) row[i][w] = src[c0 + 256 * i];
        }
    }
#pragma unroll
    for (int w = 0; w < MAXW; ++w)
        if (w < W)
#pragma unroll
            for (int i = 0; i < kConvPieces; ++i)
                if (c0 + 256 * i < vec) Cb[w * vec + c0 + 256 * i] = row[i][w];
}

// Proposal converter: tree attention mask -> parent array.  One CTA per sequence, a warp per row of the mask: the
// parent of a node is its strict ancestor with the most ancestors of its own.  The mask is checked to be the mask
// of a tree in topological order (self bit set, no later node among the ancestors, parent exactly one
// level up); otherwise the sequence gets STATUS_BAD_PARENT and its parents are left untouched.
// Masks of up to kMaskStage bytes are brought into shared memory first, all loads in flight together: with a thread per
// row reading global memory, or a warp per row twice over, the kernel is a chain of load latencies (128 masks of 64 x 64:
// 10.1 us either way, staged 6.4 us).
constexpr int kMaskStage = 16 * 1024;
__global__ void __launch_bounds__(256)
mask_to_parent_kernel(int32_t N, const uint8_t *mask, const int32_t *node_offsets,
                      int32_t *__restrict__ parent, int32_t *status)
{
    after_previous_kernel();
    extern __shared__ uint4 mask_smem[];                // the staged mask, then int32: [N] ancestors-or-self per node, [N] parent
    const int b = blockIdx.x, warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int base = node_offsets[b], n = node_offsets[b + 1] - base;
    if (n < 0 || n > N) {
        if (threadIdx.x == 0) atomicOr(status, n < 0 ? SPECA_STATUS_BAD_OFFSETS : SPECA_STATUS_TOO_MANY);
        return;
    }
    const uint8_t *m = mask + size_t(b) * N * N;
    if (n <= 64) {
        // Rows as 64-bit sets, straight out of global memory (the bytes of all rows of a warp are in flight together); then a
        // thread per node goes through its own ancestors, which are few, instead of a warp through all nodes (128 masks of 64 x
        // 64: 5.8 us staged as below, 3.2 so).
        __shared__ uint2 s_row[64];
        uint8_t lo[8], hi[8];
#pragma unroll
        for (int k = 0; k < 8; ++k) {
            const int i = warp + 8 * k;
            lo[k] = i < n && lane < n ? m[i * N + lane] : 0;
            hi[k] = i < n && lane + 32 < n ? m[i * N + lane + 32] : 0;
        }
#pragma unroll
        for (int k = 0; k < 8; ++k) {
            const uint2 row = make_uint2(__ballot_sync(0xffffffffu, lo[k] != 0), __ballot_sync(0xffffffffu, hi[k] != 0));
            if (lane == 0) s_row[warp + 8 * k] = row;
        }
        __syncthreads();
        int bad = 0, best = -1;                         // best: (ancestors << 16) | (0xffff - index): the most, then the lowest index
        const int i = threadIdx.x;
        if (i < n) {
            const uint2 row = s_row[i];
            const unsigned long long set = row.x | (unsigned long long)(row.y) << 32, self = 1ull << i;
            bad = !(set & self) || (set & ~(2 * self - 1)) != 0;
            for (unsigned long long rest = set & ~self; rest != 0; rest &= rest - 1) {
                const int j = __ffsll(rest) - 1;
                best = max(best, ((__popc(s_row[j].x) + __popc(s_row[j].y)) << 16) | (0xffff - j));
            }
            bad |= (best < 0 ? 0 : best >> 16) != __popcll(set) - 1;
        }
        if (__syncthreads_or(bad)) {
            if (threadIdx.x == 0) atomicOr(status, SPECA_STATUS_BAD_PARENT);
            return;
        }
        if (i < n) parent[base + i] = best < 0 ? -1 : 0xffff - (best & 0xffff);
        return;
    }
    int32_t *sm = reinterpret_cast<int32_t *>(mask_smem) + (min(N * N, kMaskStage) + 15) / 16 * 4;
    if (n * N <= kMaskStage) {
        uint8_t *staged = reinterpret_cast<uint8_t *>(mask_smem);
        if ((N & 3) == 0 && (reinterpret_cast<uintptr_t>(mask) & 15u) == 0)          // every mask starts on 16 bytes
#pragma unroll 4
            for (int i = threadIdx.x; i < n * N / 16 + (n * N % 16 != 0); i += 256)
                reinterpret_cast<uint4 *>(staged)[i] = reinterpret_cast<const uint4 *>(m)[i];
        else
#pragma unroll 8
            for (int i = threadIdx.x; i < n * N; i += 256) staged[i] = m[i];
        __syncthreads();
        m = staged;
    }
    int bad = 0;
    for (int i = warp; i < n; i += 8) {
        int cnt = 0;
        for (int j0 = 0; j0 < n; j0 += 32) {
            const int j = j0 + lane;
            const int on = j < n && m[size_t(i) * N + j] != 0;
            cnt += on;
            bad |= (on && j > i) || (j == i && !on);
        }
        cnt = __reduce_add_sync(0xffffffffu, cnt);
        if (lane == 0) sm[i] = cnt;
    }
    __syncthreads();
    for (int i = warp; i < n; i += 8) {
        int best = -1;                                  // (ancestors << 16) | (0xffff - index): the most, then the lowest index
        for (int j0 = 0; j0 < n; j0 += 32) {
            const int j = j0 + lane;
            if (j < n && j != i && m[size_t(i) * N + j] != 0) best = max(best, (sm[j] << 16) | (0xffff - j));
        }
        best = __reduce_max_sync(0xffffffffu, best);
        bad |= best >= 0 ? (best >> 16) != sm[i] - 1 : sm[i] != 1;
        if (lane == 0) sm[N + i] = best < 0 ? -1 : 0xffff - (best & 0xffff);
    }
    if (__syncthreads_or(bad)) {
        if (threadIdx.x == 0) atomicOr(status, SPECA_STATUS_BAD_PARENT);
        return;
    }
    for (int i = threadIdx.x; i < n; i += blockDim.x) parent[base + i] = sm[N + i];
}

// Heavy-light chain decomposition (Section 4.3): one CTA per sequence, thread i owns node i.  The heavy
// child of a node is its child with the largest subtree (lowest index on ties); a node continues its
// parent's chain iff it is that heavy child, otherwise it heads a chain of its own (so does every child
// of the committed state).  Subtree sizes are integer sums over ancestor walks, the heavy child an
// integer maximum: both are exact whatever the order of the atomics.
__global__ void __launch_bounds__(256)
chain_decompose_kernel(int32_t N, const int32_t *node_offsets, const int32_t *parent,
                       int32_t *__restrict__ chain_head, int32_t *__restrict__ n_chains, int32_t *status)
{
    after_previous_kernel();
    extern __shared__ int32_t sm[];                     // [N] subtree size, [N] key of the heavy child, [N] parent
    int32_t *par = sm + 2 * N;
    __shared__ int32_t s_flag, s_count;
    const int b = blockIdx.x;
    const int base = node_offsets[b], n = node_offsets[b + 1] - base;
    if (threadIdx.x == 0) { s_flag = 0; s_count = 0; }
    __syncthreads();
    if (n < 0 || n > N || n > 0x10000) {
        if (threadIdx.x == 0) {
            atomicOr(status, n < 0 ? SPECA_STATUS_BAD_OFFSETS : SPECA_STATUS_TOO_MANY);
            n_chains[b] = 0;
        }
        return;
    }
    for (int i = threadIdx.x; i < n; i += blockDim.x) {
        sm[i] = 1;
        sm[N + i] = -1;
        const int pa = parent[base + i];
        par[i] = pa;
        if (pa < -1 || pa >= i) atomicOr(&s_flag, 1);
    }
    __syncthreads();
    if (s_flag) {
        if (threadIdx.x == 0) { atomicOr(status, SPECA_STATUS_BAD_PARENT); n_chains[b] = 0; }
        return;
    }
    for (int i = threadIdx.x; i < n; i += blockDim.x)
        for (int a = par[i]; a >= 0; a = par[a]) atomicAdd(&sm[a], 1);
    __syncthreads();
    for (int i = threadIdx.x; i < n; i += blockDim.x) {
        const int pa = par[i];
        if (pa >= 0) atomicMax(&sm[N + pa], (sm[i] << 16) | (0xffff - i));       // largest subtree, then lowest index
    }
    __syncthreads();
    for (int i = threadIdx.x; i < n; i += blockDim.x) {
        int h = i;
        for (;;) {
            const int pa = par[h];
            if (pa < 0 || 0xffff - (sm[N + pa] & 0xffff) != h) break;            // h heads its chain
            h = pa;
        }
        chain_head[base + i] = h;
        if (h == i) atomicAdd(&s_count, 1);
    }
    __syncthreads();
    if (threadIdx.x == 0) n_chains[b] = s_count;
}

// Confidence-guided pruning, one CTA per sequence, run twice: first for the number of kept nodes, then for the
// packed output.  Scores are accumulated in fp32 down the levels of the tree, which adds every path root first, exactly
// as the definition does.
//
// The counts have to become offsets before anything can be written packed, and there is no scratch.  The first
// run leaves ~count (negative) in out_offsets[b + 1]; in the second, sequence b adds up what it finds in entries
// 1 .. b -- ~count, or the final offset if that sequence was quicker -- and replaces its own entry by the offset.
// Every entry is either of the two whenever it is read, so the sum does not depend on who comes first.  (One CTA that
// packed the sequences in turn took 86 us for 128 of them, its serial selection 15; both runs together 21 us.)
// What bounds it: a chain of shared-memory and L2 latencies per sequence; every node's path stays in registers instead of two
// barriers per tree level.
constexpr int kPruneLevels = 16;

// Calls step(i, parent of i) for every node with a parent, parents first: level by level, all threads of the CTA, for
// the first kPruneLevels levels; what is deeper is a long chain, which one thread walks in index order.  done[] marks the
// roots beforehand and everything afterwards.
template <class Step>
__device__ __forceinline__ void down_levels(int n, const int32_t *par, int32_t *done, Step step)
{
    int open = 1;
    for (int level = 0; level < kPruneLevels && open; ++level) {
        open = 0;
        int ready = 0;                                  // bit k: the node of this thread's k-th turn is final after this level
        for (int i = threadIdx.x, k = 0; i < n; i += 128, ++k)
            if (!done[i]) {
                if (done[par[i]]) { step(i, par[i]); ready |= 1 << k; }
                else open = 1;
            }
        __syncthreads();
        for (int i = threadIdx.x, k = 0; i < n; i += 128, ++k)
            if ((ready >> k) & 1) done[i] = 1;
        open = __syncthreads_or(open);
    }
    if (open) {
        if (threadIdx.x == 0)
            for (int i = 0; i < n; ++i)
                if (!done[i]) { step(i, par[i]); done[i] = 1; }
        __syncthreads();
    }
}

template <bool WRITE>
__global__ void __launch_bounds__(128)
prune_kernel(int32_t N, float tau, int32_t budget, const int32_t *node_offsets,
             const int32_t *parent, const float *logp, int32_t *__restrict__ out_offsets,
             int32_t *__restrict__ out_parent, int32_t *__restrict__ out_index, int32_t *status)
{
    after_previous_kernel();
    extern __shared__ int32_t sm[];
    float *q = reinterpret_cast<float *>(sm);           // [N]
    int32_t *par = sm + N, *keep = sm + 2 * N, *newidx = sm + 3 * N, *done = sm + 4 * N;      // [N] each
    __shared__ float s_max[4];
    __shared__ int32_t s_cnt[4], s_dst;
    const int b = blockIdx.x, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int base = node_offsets[b], n = node_offsets[b + 1] - base;

    if (WRITE && warp == 0) {
        int run = 0;
        int ahead[4];                                   // 128 entries in flight at a time
        for (int i0 = 1; i0 <= b; i0 += 32) {
            const int k = ((i0 - 1) >> 5) & 3;
            if (k == 0)
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    const int i = i0 + 32 * j + lane;
                    ahead[j] = i <= b ? *reinterpret_cast<volatile int32_t *>(out_offsets + i) : ~0;
                }
            const int v = k == 0 ? ahead[0] : k == 1 ? ahead[1] : k == 2 ? ahead[2] : ahead[3];
            const unsigned fin = __ballot_sync(0xffffffffu, v >= 0);
            const int last = 31 - __clz(int(fin));      // the last entry of these that is an offset already (-1: none)
            const int sum = __reduce_add_sync(0xffffffffu, lane > last ? ~v : 0);
            const int off = __shfl_sync(0xffffffffu, v, last < 0 ? 0 : last);
            run = last < 0 ? run + sum : off + sum;
        }
        if (lane == 0) s_dst = run;
    }

    int fault = 0;
    if (n < 0 || base < 0) fault = SPECA_STATUS_BAD_OFFSETS;
    else if (n > N) fault = SPECA_STATUS_TOO_MANY;
    else
        for (int i = tid; i < n; i += 128) {
            const int p = parent[base + i];
            if (p < -1 || p >= i) fault = SPECA_STATUS_BAD_PARENT;
            par[i] = p;
            q[i] = logp[base + i];
            done[i] = p < 0;
        }
    const bool any_fault = __syncthreads_or(fault);
    if (any_fault) {
        if (!WRITE && fault != 0) atomicOr(status, fault);
        if (tid == 0) *reinterpret_cast<volatile int32_t *>(out_offsets + b + 1) = WRITE ? s_dst : ~0;
        if (WRITE && b == 0 && tid == 0) out_offsets[0] = 0;
        return;
    }
    // Trees of up to 128 nodes and kPruneLevels levels: a thread per node keeps the path of its node in registers, so the
    // two passes down the tree (scores, and below whether a node goes with an ancestor) are a handful of independent
    // reads each instead of two barriers a level.
    int up[kPruneLevels], len = 0, a = tid < n ? tid : -1;
#pragma unroll
    for (int r = 0; r < kPruneLevels; ++r) {
        up[r] = a < 0 ? 0 : a;
        len += a >= 0;
        a = a < 0 ? a : par[a];
    }
    const bool flat = __syncthreads_and(a < 0) && n <= 128;
    if (flat) {
        float sum = 0.f, step[kPruneLevels];
#pragma unroll
        for (int r = 0; r < kPruneLevels; ++r) step[r] = q[up[r]];
#pragma unroll
        for (int r = kPruneLevels - 1; r >= 0; --r)
            sum = r >= len ? 0.f : r == len - 1 ? step[r] : sum + step[r];
        __syncthreads();
        if (tid < n) q[tid] = sum;
        __syncthreads();
    } else
        down_levels(n, par, done, [&](int i, int p) { q[i] = q[p] + q[i]; });      // a node adds its parent's once that is final
    float best = -INFINITY;
    for (int i = tid; i < n; i += 128) best = fmaxf(best, q[i]);
    for (int off = 16; off; off >>= 1) best = fmaxf(best, __shfl_xor_sync(0xffffffffu, best, off));
    if (lane == 0) s_max[warp] = best;
    __syncthreads();
    best = fmaxf(fmaxf(s_max[0], s_max[1]), fmaxf(s_max[2], s_max[3]));
    if (n > 0 && q[0] != q[0]) best = q[0];             // a score that is no number in front keeps nothing
    const float thr = best - tau;
    for (int i = tid; i < n; i += 128) {
        const float qi = q[i];
        int rank = 0;
#pragma unroll 8
        for (int j = 0; j < n; ++j) {
            const float qj = q[j];
            rank += (qj >= thr) && (qj > qi || (qj == qi && j < i));
        }
        keep[i] = (qi >= thr) && rank < budget;
        done[i] = par[i] < 0;
    }
    __syncthreads();
    // a node goes with its parent
    if (flat) {
        int on = 1;
#pragma unroll
        for (int r = 0; r < kPruneLevels; ++r)
            on &= r < len ? keep[up[r]] : 1;
        __syncthreads();
        if (tid < n) keep[tid] = on;
        __syncthreads();
    } else
        down_levels(n, par, done, [&](int i, int p) { keep[i] &= keep[p]; });
    // new indices: kept nodes before this one
    int count = 0;
    for (int i0 = 0; i0 < n; i0 += 128) {
        const int i = i0 + tid;
        const int on = i < n && keep[i];
        const unsigned m = __ballot_sync(0xffffffffu, on);
        if (lane == 0) s_cnt[warp] = __popc(m);
        __syncthreads();
        int before = count;
        for (int w = 0; w < warp; ++w) before += s_cnt[w];
        if (i < n) newidx[i] = before + __popc(m & ((1u << lane) - 1u));
        count += s_cnt[0] + s_cnt[1] + s_cnt[2] + s_cnt[3];
        __syncthreads();
    }
    if (!WRITE) {
        if (tid == 0) out_offsets[b + 1] = ~count;
        return;
    }
    const int dst = s_dst;
    if (tid == 0) {
        *reinterpret_cast<volatile int32_t *>(out_offsets + b + 1) = dst + count;
        if (b == 0) out_offsets[0] = 0;
    }
    for (int i = tid; i < n; i += 128)
        if (keep[i]) {
            const int p = par[i];
            out_parent[dst + newidx[i]] = p < 0 ? -1 : newidx[p];
            out_index[dst + newidx[i]] = i;
        }
}

// The same for up to kPruneSeqs sequences of at most 64 nodes, in one launch: a warp per sequence, spread over a cluster of
// CTAs that tell one another their counts through shared memory, so that nothing has to be done twice.  Sets of nodes are 64-bit
// words, and a warp needs no barrier.  What is left is a chain of two loads, the levels of the tree, the 64 comparisons of
// a node and the barriers of the cluster.  128 trees of 24..64 nodes: 11.9 us for the two runs of prune_kernel, 4.9 so.  More
// sequences than warps, or more nodes than bits, go the other way (CTAs of 32 warps would take 256 trees, in 7.5 us instead of
// 12.7, and cost smaller batches some: 128 trees 5.1 instead of 4.9, one 3.2 instead of 2.9).
constexpr int kPruneCtas = 8, kPruneSeqs = 128;
__global__ void __cluster_dims__(kPruneCtas, 1, 1) __launch_bounds__(kPruneSeqs / kPruneCtas * 32)
prune_small_kernel(int32_t B, int32_t N, float tau, int32_t budget, const int32_t *node_offsets, const int32_t *parent,
                   const float *logp, int32_t *__restrict__ out_offsets, int32_t *__restrict__ out_parent,
                   int32_t *__restrict__ out_index, int32_t *status)
{
    after_previous_kernel();
    // (every CTA of the cluster has to have started before its shared memory is written; waited for below, behind the loads)
    asm volatile("barrier.cluster.arrive.relaxed.aligned;" ::: "memory");
    __shared__ int32_t s_count[kPruneSeqs];
    __shared__ __align__(16) float s_q[kPruneSeqs / kPruneCtas][64];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, b = warp * kPruneCtas + blockIdx.x;
    float *q = s_q[warp];
    typedef unsigned long long Set;
    auto set_of = [](bool lo, bool hi) -> Set {
        return __ballot_sync(0xffffffffu, lo) | Set(__ballot_sync(0xffffffffu, hi)) << 32;
    };
    auto in = [](Set s, int i) -> bool { return (s >> i) & 1; };

    int base = 0, n = 0, fault = 0;
    if (b < B) {
        base = node_offsets[b];
        n = node_offsets[b + 1] - base;
        if (n < 0 || base < 0) fault = SPECA_STATUS_BAD_OFFSETS;
        else if (n > N) fault = SPECA_STATUS_TOO_MANY;
    }
    if (fault) n = 0;
    int par[2] = {-1, -1};
    float lp[2] = {0.f, 0.f};
    bool bad = false;
#pragma unroll
    for (int k = 0; k < 2; ++k) {
        const int i = lane + 32 * k;
        if (i < n) {
            par[k] = parent[base + i];
            lp[k] = logp[base + i];
            bad |= par[k] < -1 || par[k] >= i;
        }
    }
    if (__any_sync(0xffffffffu, bad)) {
        fault = SPECA_STATUS_BAD_PARENT;
        n = 0;
    }
    if (fault && lane == 0) atomicOr(status, fault);

    // scores: a level a turn, a node adds its own to its parent's (entries past the last node compare as false)
    const bool live[2] = {lane < n, lane + 32 < n};
    float mine[2];
#pragma unroll
    for (int k = 0; k < 2; ++k) {
        mine[k] = live[k] ? lp[k] : NAN;
        q[lane + 32 * k] = mine[k];
    }
    __syncwarp();
    Set done = set_of(!live[0] || par[0] < 0, !live[1] || par[1] < 0);
    while (done != ~Set(0)) {
        bool now[2];
#pragma unroll
        for (int k = 0; k < 2; ++k) {
            now[k] = !in(done, lane + 32 * k) && in(done, par[k] & 63);
            if (now[k]) mine[k] = q[par[k]] + lp[k];
        }
        __syncwarp();
#pragma unroll
        for (int k = 0; k < 2; ++k)
            if (now[k]) q[lane + 32 * k] = mine[k];
        __syncwarp();
        done |= set_of(now[0], now[1]);
    }
    float best = fmaxf(mine[0], mine[1]);
    for (int off = 16; off; off >>= 1) best = fmaxf(best, __shfl_xor_sync(0xffffffffu, best, off));
    best = fmaxf(best, -INFINITY);
    if (n > 0 && q[0] != q[0]) best = q[0];             // a score that is no number in front keeps nothing
    const float thr = best - tau;
    // nodes that go before this one: better, or as good and of lower index (where this one is in the window, so are they)
    int rank[2] = {0, 0};
#pragma unroll 2
    for (int j0 = 0; j0 < n; j0 += 4) {
        const float4 v = *reinterpret_cast<const float4 *>(q + j0);
        const float f[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
        for (int e = 0; e < 4; ++e)
#pragma unroll
            for (int k = 0; k < 2; ++k)
                rank[k] += f[e] > mine[k] || (f[e] == mine[k] && j0 + e < lane + 32 * k);
    }
    const Set keep = set_of(live[0] && mine[0] >= thr && rank[0] < budget, live[1] && mine[1] >= thr && rank[1] < budget);
    // a node goes with its parent
    Set kept = 0;
    for (Set more = keep; more != kept;) {
        kept = more;
        more = set_of(in(kept, lane) && (par[0] < 0 || in(kept, par[0] & 63)),
                      in(kept, lane + 32) && (par[1] < 0 || in(kept, par[1] & 63)));
    }
    const int count = __popcll(kept);

    // every CTA learns every count
    __syncwarp();
    asm volatile("barrier.cluster.wait.aligned;" ::: "memory");
    const uint32_t slot = uint32_t(__cvta_generic_to_shared(&s_count[b]));
    if (lane < kPruneCtas) {
        uint32_t remote;
        asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(remote) : "r"(slot), "r"(lane));
        asm volatile("st.shared::cluster.s32 [%0], %1;" ::"r"(remote), "r"(count) : "memory");
    }
    __syncwarp();
    asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
    if (b >= B) return;
    int dst = 0;
#pragma unroll
    for (int k = 0; k < kPruneSeqs / 32; ++k) dst += lane + 32 * k < b ? s_count[lane + 32 * k] : 0;
    dst = __reduce_add_sync(0xffffffffu, dst);
    if (lane == 0) {
        out_offsets[b + 1] = dst + count;
        if (b == 0) out_offsets[0] = 0;
    }
    auto before = [&](int i) { return __popcll(kept & ((Set(1) << i) - 1)); };
#pragma unroll
    for (int k = 0; k < 2; ++k) {
        const int i = lane + 32 * k;
        if (in(kept, i)) {
            out_parent[dst + before(i)] = par[k] < 0 ? -1 : before(par[k]);
            out_index[dst + before(i)] = i;
        }
    }
}

}  // namespace

int launch_mask_to_parent(int32_t B, int32_t N, const uint8_t *mask, const int32_t *node_offsets, int32_t *parent,
                          int32_t *status, cudaStream_t st)
{
    const size_t stage = (size_t(N) * N <= kMaskStage ? size_t(N) * N + 15 : kMaskStage) / 16 * 16;
    launch(mask_to_parent_kernel, B, 256, size_t(2 * N) * sizeof(int32_t) + stage, st, N, mask, node_offsets,
           parent, status);
    return int(cudaGetLastError());
}

int launch_chain_decompose(int32_t B, int32_t N, const int32_t *node_offsets, const int32_t *parent,
                           int32_t *chain_head, int32_t *n_chains, int32_t *status, cudaStream_t st)
{
    launch(chain_decompose_kernel, B, 256, size_t(3 * N) * sizeof(int32_t), st, N, node_offsets, parent, chain_head,
           n_chains, status);
    return int(cudaGetLastError());
}

int launch_prune(int32_t B, int32_t N, float tau, int32_t budget, const int32_t *node_offsets, const int32_t *parent,
                 const float *logp, int32_t *out_offsets, int32_t *out_parent, int32_t *out_index, int32_t *status,
                 cudaStream_t st)
{
    if (N <= 64 && B <= kPruneSeqs) {
        launch(prune_small_kernel, kPruneCtas, kPruneSeqs / kPruneCtas * 32, 0, st, B, N, tau, budget, node_offsets, parent,
               logp, out_offsets, out_parent, out_index, status);
        return int(cudaGetLastError());
    }
    const size_t smem = size_t(5 * N) * sizeof(int32_t);
    launch(prune_kernel<false>, B, 128, smem, st, N, tau, budget, node_offsets, parent, logp, out_offsets, out_parent,
           out_index, status);
    const int e = int(cudaGetLastError());
    if (e != 0) return e;
    launch(prune_kernel<true>, B, 128, smem, st, N, tau, budget, node_offsets, parent, logp, out_offsets, out_parent,
           out_index, status);
    return int(cudaGetLastError());
}

int launch_conv_commit(int32_t L, int32_t B, int32_t channels, int32_t W, int32_t T, int32_t max_depth, void *C,
                       const void *x, const int32_t *node_offsets, const int32_t *path_idx, const int32_t *path_len,
                       int32_t *status, cudaStream_t st)
{
    const int vec = channels / 8, parts = (vec + 256 * kConvPieces - 1) / (256 * kConvPieces);     // 16-byte pieces of a row
    auto kern = W <= 4 ? conv_commit_kernel<4> : conv_commit_kernel<kConvMaxWidth>;
    launch(kern, unsigned(L) * B * parts, 256, 0, st, B, vec, parts, W, T, max_depth, static_cast<uint4 *>(C),
           static_cast<const uint4 *>(x), node_offsets, path_idx, path_len, status);
    return int(cudaGetLastError());
}

int launch_pending_check(const Params &p, int max_len, cudaStream_t st)
{
    launch(pending_check_kernel, (p.B + 127) / 128, 128, 0, st, p.B, p.Tp, p.max_depth, max_len, p.max_nodes,
           p.pnode_offsets, p.pparent, p.path_idx, p.path_len, p.ws.pend, p.status);
    return int(cudaGetLastError());
}

int launch_plan(const Params &p, cudaStream_t st)
{
    const size_t smem = size_t(6 * p.max_nodes + 1) * sizeof(int32_t);
    launch(plan_kernel, p.B, kPlanThreads, smem, st, p.node_offsets, p.parent, p.depth_in, p.B, p.T, p.max_depth,
           p.max_nodes, p.skip_nodes, p.plan_paths_only, p.n_slots, p.ws, p.status);
    return int(cudaGetLastError());
}

int launch_accept(int32_t B, int32_t max_depth, const int32_t *node_offsets, const int32_t *parent,
                  const int32_t *draft_tok, const int32_t *target_tok, const int32_t *root_target_tok,
                  int32_t *path_idx, int32_t *path_len, int32_t *next_tok, int32_t *status,
                  cudaStream_t st)
{
    const int warps = 4;
    launch(accept_kernel, (B + warps - 1) / warps, warps * 32, 0, st, B, max_depth, node_offsets, parent, draft_tok,
           target_tok, root_target_tok, path_idx, path_len, next_tok, status);
    return int(cudaGetLastError());
}

int launch_stochastic_accept(int32_t B, int32_t max_depth, const int32_t *node_offsets, const int32_t *parent,
                             const float *p_target, const float *p_draft, const float *uniform,
                             int32_t *path_idx, int32_t *path_len, int32_t *status, cudaStream_t st)
{
    const int warps = 4;
    launch(stochastic_accept_kernel, (B + warps - 1) / warps, warps * 32, 0, st, B, max_depth, node_offsets, parent,
           p_target, p_draft, uniform, path_idx, path_len, status);
    return int(cudaGetLastError());
}

}  // namespace speca

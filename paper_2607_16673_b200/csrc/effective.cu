// Tree-masked verification on the 5th-generation tensor cores (tcgen05 + TMEM): the parallel route of Section 4.2
// with the triangular solve moved to coefficient rows, at fp32 accuracy.
//
// Mathematics.  With a_0 = t, a_1, ... the root path of node t taken upward, gamma_t the product of alpha over it
// and rho_t[r] = alpha_{a_0} ... alpha_{a_{r-1}}, the factorisation of Section 4.2 (A_tree = M_tree o K_b K_a^T,
// T = (I + A)^-1, O = Qhat S0^T - Attn (W S0^T) + Attn U) regroups as
//        R = K S0^T ,  G = Q S0^T ,  x_a = v_a - gamma_a R_a                       (per node, over the value rows)
//        o_t = scale gamma_t G_t + sum_r M[t][a_r] x_{a_r} ,     M[t][a_r] = scale rho_t[r] c_r beta_{a_r}
// where c is a back substitution up the node's own path that needs Gram entries only,
//        c_r = q_t.k_{a_r} - sum_{m<r} c_m beta_{a_m} (k_{a_m}.k_{a_r}) .
// The corrected values u_t = sum_r M[t][a_r] x_{a_r} come out the same way with c_0 = 1, c_r = 0 on the right-hand
// side and scale 1.  (Attn is M; the solve is at most 15 steps along a path.)  Per value tile that is one product of
// the state with the raw rows of [K;Q], an element-wise step, and one product with M.
//
// Accuracy.  Everything is split into bf16 pieces of 8 bits: the fp32 state and x into three each by truncation
// (exact: 3 x 8 = 24 bits), M likewise; q, k, v are bf16 already.  S0 [K;Q]^T is three products of pieces, exact up
// to the fp32 accumulation; x M^T keeps the six products down to 2^-16, the dropped ones are 2^-24 of the result.
// What is left is the accumulation: the tensor core truncates where it adds, so each further product in one accumulator
// costs half an ulp toward zero.  So the six products go in by size, over all nodes the small ones first, and the Gram blocks
// in as many chains from zero as their 64 columns of TMEM hold, added up by the solver.  Error against 64 bits, 2-norm of the
// difference over that of the outputs, x 10^-8, before both / now / the substitution kernel: d_k = 256, 30 nodes 33 / 22 /
// 26; d_k = 128, 20 nodes 22 / 16 / 15, 60 nodes at 8 levels 24 / 20 / 14 (no columns left for a second chain), at 16 levels
// 24 / 20 / (a former kernel) 66.  Both cost 2 to 3 % of a unit.  Gram blocks of warp-level MMAs added up in fp32 bring 60
// nodes to 14 too, and cost 17 % of a unit of 64 nodes, 28 % of one of 40: the solver has no time for them, and the split
// warps keep the state product waiting.
//
// Why this form.  The staged bf16 rows of [K;Q], as TMA lands them, are the B operand: no fp32 operand is built, so
// the state stream waits for no preparation, only the second product does, a tile later.  The pieces of the state go
// into TMEM as the A operand, so a slice crosses shared memory twice (TMA write, one read) and its ring slot is free
// as soon as it has been read; rewriting it in place between two TF32 passes took five crossings and three hand-overs.
// A tile of 64 nodes takes 24 + 24 tcgen05 instructions.  The substitution over value rows, ~95 instructions per node
// and warp in factorized.cu, is gone: what is left per element is a multiply-add on each side of the second product.
//
// Mapping.  One persistent CTA per SM walks units (layer, sequence, head) tile by tile (128 value rows); 24 warps:
//   warp 0        TMA producer of the state slices (128 rows x 32 columns, 128-byte swizzle)
//   warp 1        issues S0 [K;Q]^T; owns TMEM
//   warp 2        issues the Gram blocks [K;Q] K^T (one unit ahead) and x M^T
//   warp 3        walks the list of units and hands records of them to the others; TMA producer of the staged [K;Q] rows
//                 (two units) and the value rows (two tiles)
//   warps 4-11    split: slice row per thread -> three bf16 pieces in TMEM; two groups alternate slices, a buffer each (trees
//                 of more than 8 levels: one group, and the roles below four warps earlier)
//   warps 12-19   epilogue, two warps per TMEM lane quarter that share a tile's columns: R out of TMEM, x back into TMEM
//                 as three pieces; then, while the next tile's product runs, o = scale gamma G + (x M^T), coalesced
//   warps 20-23   solver, one unit ahead: Gram entries of every row against its own path, back substitution (a thread
//                 per node, registers), the pieces of M
// TMEM: two tiles of accumulators (R | G, 128 columns; x M^T overwrites R), two A buffers of 48, x of 96, Gram of 64.
// Measured in large batches, us per unit and SM (share of the copy rate): d_k = 128, d_v = 256: 20 nodes 4.1 (95 %), 32
// nodes 4.4 (100 %), 40 nodes 5.2 (92 %), 64 nodes 6.7 (89 %); d_k = d_v = 256, 24 nodes 7.1 (103 %); 16 levels: 24 nodes 4.6
// (88 %), 64 nodes 7.0 (85 %).  What bounds it: HBM up to
// 32 nodes and at d_k = 256; above that the instructions of the roles, which wait for one another in turn (an epilogue warp a
// third of its time for x M^T).  More of them did not help: three epilogue warps a lane quarter in the place of the second
// split group no change, x M^T in two parts (the first under the making of the second half of x) 3 % slower, the loads of the
// next eight columns under the work on these 4 % slower.
// Ten roles take turns on four issue slots, so the kernel's size matters as much as its instruction count: loops stay
// rolled where a role has slack.
// x M^T runs over all nodes with zeros in M off the path, and zero times a value that is not finite is no zero: where an
// epilogue warp meets such an x it leaves it out of the product and makes G of the nodes that have it on their path not
// finite instead.
// With u requested a unit is walked twice (o rows, then u rows); the second walk finds the state tile in L2.
// Every wait is bounded; on expiry the CTA raises SPECA_STATUS_TIMEOUT, drains and exits.
#include <cuda.h>

#include <atomic>
#include <type_traits>

#include "speca_common.cuh"
#include "tc_ptx.cuh"

namespace speca {

namespace {

using namespace tc;

constexpr int kRows = 128;                      // value rows per tile (= TMEM lanes = MMA M)
constexpr int kSliceBytes = kRows * 128;        // one ring slot: a K-slice of a tile (128 rows x 32 fp32)
constexpr int kWalkSeqs = 128;
// Records of units.  The walk is one unit ahead of the staged rows, which are two ahead of the state product, and the value
// rows keep it within two tiles of the epilogue: no role is five units behind it.
constexpr int kUnitRing = 8;
// TMEM columns
constexpr int kTileCols = 128;                  // accumulators of a tile: R, then G
constexpr int kAOff = 2 * kTileCols, kACols = 48;    // two buffers of three 16-column pieces (32 bf16 columns each)
constexpr int kXOff = kAOff + 2 * kACols;       // x: three 32-column pieces (64 nodes)
constexpr int kGramOff = kXOff + 96;
constexpr int kTmemCols = 512;
static_assert(kGramOff + 64 == kTmemCols, "TMEM columns");

// Split groups, four warps each, and with them the first warps of the epilogue and of the solver.  Up to 8 levels two: one takes
// as long at 64 nodes, 4 % longer at 20.  Beyond that the solver's coefficients want the registers of four warps (96 a thread
// instead of 80), and one group keeps up with it.  us per unit and SM, two groups / one: d_k = 128, d_v = 256, 16 levels, 24
// nodes 5.34 / 4.64, 40 nodes 6.16 / 5.37, 64 nodes 7.25 / 7.00; 192 units of d_k = d_v = 256, 32 nodes 25.5 / 23.9 us.
template <int DK, int MAXD> struct Roles {
    static constexpr int kSplits = MAXD > 8 ? 1 : 2;
    static constexpr int kEpilogue = 4 + 4 * kSplits, kSolver = kEpilogue + 8, kThreads = 32 * (kSolver + 4);
};

// shared-memory carve-up per instantiation
template <int DK, int MAXN_, int MAXD> struct Lay {
    static constexpr int MAXN = MAXN_;                          // nodes per sequence
    static constexpr int NC = DK / 32;                          // K-slices per tile
    static constexpr int SC = DK / 64;                          // 64-column regions of the staged bf16 rows
    static constexpr int SCB = 2 * MAXN * 128;                  // bytes per region: key rows, then query rows
    static constexpr int STAGE = SC * SCB;
    static constexpr int VBUF = MAXN * kRows * 2;               // value rows of a tile, [node][128] bf16
    static constexpr int MPIECE = MAXN * 128;                   // one bf16 piece of M: R rows x 64 columns
    static constexpr int MBUF2 = MAXN > 32 ? 32 * 128 : 3 * MPIECE;      // second buffer of M, for units of up to 32 nodes
    static constexpr int GSTR = MAXD + 4;                       // floats per node of the Gram entries, by distance up the path
    static constexpr int OffStage = 0;                          // two units
    // (the Gram block's A operand spans 128 rows whatever MAXN: it reads on into the regions behind, rows nobody looks at)
    static constexpr int OffM = OffStage + 2 * STAGE;
    static constexpr int OffV = OffM + (MAXN > 32 ? 3 : 6) * MPIECE;     // two tiles
    static constexpr int OffRing = OffV + 2 * VBUF;
    static constexpr int kSmall = 2 * MAXN * GSTR * 4 + 2 * 2 * MAXN * 4 + 2 * MAXN + 4 * 2 * MAXN * 4 + 5 * kWalkSeqs + 32 * kUnitRing +
                                  16 + 8 * 64;
    static constexpr int kRoom = (227 * 1024 - OffRing - kSmall) / kSliceBytes;
    static constexpr int NS = kRoom > 8 ? 8 : kRoom & ~1;       // ring depth: even, so that a slot is always the same split group's
    static constexpr int OffGk = OffRing + NS * kSliceBytes;    // [MAXN][GSTR] k_node . k_(ancestor at distance i + 1)
    static constexpr int OffGq = OffGk + MAXN * GSTR * 4;       // [MAXN][GSTR] q_node . k_(ancestor at distance i)
    static constexpr int OffAB = OffGq + MAXN * GSTR * 4;       // two units of float alpha, beta [MAXN]
    static constexpr int OffGam = OffAB + 2 * 2 * MAXN * 4;     // four units of float gamma in x, factor of G [MAXN]
    static constexpr int OffDepth = OffGam + 4 * 2 * MAXN * 4;  // two units of uint8 [MAXN]
    static constexpr int OffWalk = OffDepth + 2 * MAXN;
    static constexpr int OffUnit = OffWalk + 5 * kWalkSeqs;     // records of units, 32 bytes each
    static constexpr int OffMisc = OffUnit + 32 * kUnitRing;    // abort flag, TMEM base
    static constexpr int OffBars = OffMisc + 16;
    static constexpr int Bytes = OffBars + 8 * 64;
    static_assert(Bytes - OffGk == kSmall, "small regions");
    static_assert(NS >= 4, "ring too shallow");
    static_assert(Bytes <= 227 * 1024, "shared memory budget");
};

constexpr int kMaxSlots = 8;
enum Bar {
    kFull = 0,                         // [8] TMA -> split: slice landed
    kEmpty = kFull + kMaxSlots,        // [8] split -> TMA: slice read
    kAReady = kEmpty + kMaxSlots,      // [2] split -> MMA: pieces of a slice in TMEM
    kAFree = kAReady + 2,              // [2] MMA -> split
    kKQFull = kAFree + 2,              // [2] TMA -> both issuers: staged rows of a unit
    kKQFree = kKQFull + 2,             // [2] both issuers -> TMA
    kVFull = kKQFree + 2,              // [2] TMA -> epilogue: value rows of a tile
    kVFree = kVFull + 2,               // [2] epilogue -> TMA
    kAccFull = kVFree + 2,             // [2] MMA -> epilogue: R and G of a tile
    kAccFree = kAccFull + 2,           // [2] epilogue -> MMA
    kXReady = kAccFree + 2,            // epilogue -> MMA: x of a tile in TMEM, R read
    kOutFull,                          // [2] MMA -> epilogue: x M^T of a tile complete, its x no longer read
    kGramFull = kOutFull + 2,          // MMA -> solver
    kGramFree,                         // solver -> MMA
    kGamReady,                         // [2] solver -> epilogue: gamma of a unit
    kMReady = kGamReady + 2,           // [2] solver -> MMA: M of a unit
    kMFree = kMReady + 2,              // [2] MMA -> solver
    kSync = kMFree + 2,                // solver, role-internal
    kUnit,                             // [8] walk -> all: record of a unit
    kDrain = kUnit + 8,
    kBarCount
};
static_assert(kBarCount <= 64, "barrier region too small");

struct EMaps { CUtensorMap k[4], q[4], v[4]; };       // one per box height: 16, 32, 48, 64 nodes

struct EParams {
    Params p;
    int32_t share;                   // log2 of the units that share a head's keys and queries: see launch_verify_effective
    int32_t withhold_first_load;     // failure-detection test: CTA 0 never requests its first state slice
    int32_t want_u;
    int32_t own_plan;                // FEW: the sequences are checked and their paths written here, no plan kernel ran
    int32_t heads_per_group;
    int32_t gpl, dl, db, dg;         // groups of heads per (layer, sequence); a step of gridDim.x groups as (layers, sequences, groups)
};

// A unit is one (layer, sequence, head); with u requested it is walked twice (kind 0: o rows, kind 1: u rows).
// Units are taken in groups of HG consecutive heads of one (layer, sequence): group blockIdx.x, += gridDim.x, kept as
// (layer, sequence, group of heads) and advanced by carries, not divisions.  One warp walks the list and hands a record of
// every unit to the others through a ring in shared memory.  With the walk in every role, 24 warps spent some fifty
// instructions a unit on it, and the registers of its state (us per unit and SM, walk in every role / records: d_k = 128, d_v =
// 256, 20 nodes 4.66 / 4.51, 32 nodes 5.00 / 4.76, 64 nodes 7.52 / 7.41, 64 and 24 nodes at 16 levels 8.24 / 7.80 and 6.29 /
// 5.35; d_v = 128, 32 nodes 3.96 / 3.27; d_k = 256, 24 nodes 8.07 / 7.74).
struct Unit { int u, n, z, h, base, kind; };                     // z: layer's first record + base; n = 0: the list has ended
struct Walk {
    int HG, gpl, L, B, H, T, dl, db, dg, two;                    // d*: a step of gridDim.x groups
    const int32_t *seq_n; const int32_t *offs;
    const uint8_t *tab;
    int hi, nl, nb, ng;                                          // head of the group; the group after this one
};

__device__ __forceinline__ void next_unit(Walk &w, Unit &x)
{
    if (w.two && x.kind == 0) { x.kind = 1; return; }
    x.kind = 0;
    if (++w.hi < w.HG) { ++x.h; ++x.u; return; }
    x.n = 0;
    while (w.nl < w.L && x.n <= 0) {
        const int l = w.nl, b = w.nb, g = w.ng;
        w.ng += w.dg; w.nb += w.db; w.nl += w.dl;
        if (w.ng >= w.gpl) { w.ng -= w.gpl; ++w.nb; }
        if (w.nb >= w.B) { w.nb -= w.B; ++w.nl; }
        const bool in_tab = b < kWalkSeqs;
        x.n = in_tab ? int(reinterpret_cast<const int8_t *>(w.tab + 4 * kWalkSeqs)[b]) : w.seq_n[b];
        w.hi = 0;
        x.h = g * w.HG;
        x.u = (l * w.B + b) * w.H + x.h;
        x.base = in_tab ? reinterpret_cast<const int32_t *>(w.tab)[b] : w.offs[b];
        x.z = l * w.T + x.base;
    }
    if (x.n < 0) x.n = 0;
}

// chains into which a Gram block of `npad` columns is split
__device__ __forceinline__ int gram_parts(int npad) { return npad == 16 ? 4 : npad == 32 ? 2 : 1; }
// one arrival for the whole warp: every lane's earlier writes are ordered before it
__device__ __forceinline__ void warp_arrive(uint32_t bar, int lane)
{
    __syncwarp();
    if (lane == 0) mbar_arrive(bar);
}

__device__ __forceinline__ void tmem_st16(uint32_t taddr, const uint32_t (&x)[16])
{
    asm volatile(
        "tcgen05.st.sync.aligned.32x32b.x16.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16};"
        ::"r"(taddr), "r"(x[0]), "r"(x[1]), "r"(x[2]), "r"(x[3]), "r"(x[4]), "r"(x[5]), "r"(x[6]), "r"(x[7]), "r"(x[8]),
          "r"(x[9]), "r"(x[10]), "r"(x[11]), "r"(x[12]), "r"(x[13]), "r"(x[14]), "r"(x[15])
        : "memory");
}
__device__ __forceinline__ void tmem_st4(uint32_t taddr, const uint32_t (&x)[4])
{
    asm volatile("tcgen05.st.sync.aligned.32x32b.x4.b32 [%0], {%1,%2,%3,%4};" ::"r"(taddr), "r"(x[0]), "r"(x[1]), "r"(x[2]), "r"(x[3])
                 : "memory");
}
__device__ __forceinline__ float tmem_ld1(uint32_t taddr)
{
    uint32_t x;
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x1.b32 {%0}, [%1];" : "=r"(x) : "r"(taddr) : "memory");
    tmem_ld_wait();
    return __uint_as_float(x);
}
__device__ __forceinline__ void tmem_st1(uint32_t taddr, float x)
{
    asm volatile("tcgen05.st.sync.aligned.32x32b.x1.b32 [%0], {%1};" ::"r"(taddr), "r"(__float_as_uint(x)) : "memory");
}
__device__ __forceinline__ void tmem_st_wait() { asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory"); }
// kind::f16 (bf16) with the A operand in TMEM: a 32-bit column holds two consecutive K elements, the even one low
__device__ __forceinline__ void mma_bf16_ts(uint32_t d_tmem, uint32_t a_tmem, uint64_t b_desc, uint32_t idesc, uint32_t accumulate,
                                            uint32_t lead)
{
    asm volatile(
        "{\n\t.reg .pred p, q;\n\t"
        "setp.ne.b32 p, %4, 0;\n\t"
        "setp.ne.b32 q, %5, 0;\n\t"
        "@q tcgen05.mma.cta_group::1.kind::f16 [%0], [%1], %2, %3, p;\n\t}"
        ::"r"(d_tmem), "r"(a_tmem), "l"(b_desc), "r"(idesc), "r"(accumulate), "r"(lead)
        : "memory");
}
// Two fp32 values as three packed pairs of bf16 pieces (x0 in the low half), by truncation: a piece takes the top 8
// bits of what is left, and three times 8 bits are all 24.  What is left is taken with the fused multiply-add that reads a
// bf16 half of a register (piece times -1 plus x, exact): masks and a packed subtraction took four more instructions of
// the integer pipe, which runs at half rate (in a loop of splits a pair took 22 cycles, now 16; verification of ragged trees
// of 8..64 nodes 463 -> 444 us).
__device__ __forceinline__ void split_pair(float x0, float x1, uint32_t &p1, uint32_t &p2, uint32_t &p3)
{
    auto pack = [](float y0, float y1) { return __byte_perm(__float_as_uint(y0), __float_as_uint(y1), 0x7632); };
    auto rest = [](uint32_t piece, float &y0, float &y1) {
        asm("{\n\t.reg .b16 lo, hi, m;\n\t"
            "mov.b16 m, 0xbf80;\n\t"
            "mov.b32 {lo, hi}, %2;\n\t"
            "fma.rn.f32.bf16 %0, lo, m, %0;\n\t"
            "fma.rn.f32.bf16 %1, hi, m, %1;\n\t}"
            : "+f"(y0), "+f"(y1) : "r"(piece));
    };
    p1 = pack(x0, x1);
    rest(p1, x0, x1);
    p2 = pack(x0, x1);
    rest(p2, x0, x1);
    p3 = pack(x0, x1);
}

// Optional self-profiling build (-DSPECA_PROF): cycles CTA 0 spends in each kind of wait, per warp,
// written to the control words of the workspace ([8 + 9 warp .. ): 8 slots and the warp's lifetime).
#ifdef SPECA_PROF
#define PROF_DECL long long prof_w[8] = {0, 0, 0, 0, 0, 0, 0, 0}; const long long prof_t0 = clock64();
#define WAIT(slot, b, ph) prof_wait(prof_w[slot], b, ph, abort_flag)
#define PROF_T0() const long long prof_seg0 = clock64();
#define PROF_ADD(slot) prof_w[slot] += clock64() - prof_seg0;
#define PROF_STORE()                                                                              \
    if (blockIdx.x == 0 && lane == 0) {                                                           \
        long long *dst = reinterpret_cast<long long *>(p.ws.ctrl) + 8 + warp * 9;                \
        for (int i_ = 0; i_ < 8; ++i_) dst[i_] = prof_w[i_];                                      \
        dst[8] = clock64() - prof_t0;                                                             \
    }
__device__ __forceinline__ bool prof_wait(long long &acc, uint32_t bar, uint32_t parity, volatile int *abort_flag)
{
    const long long t = clock64();
    const bool r = wait_fast(bar, parity, abort_flag);
    acc += clock64() - t;
    return r;
}
#else
#define PROF_DECL
#define PROF_T0()
#define PROF_ADD(slot)
#define WAIT(slot, b, ph) wait_fast(b, ph, abort_flag)
#define PROF_STORE()
#endif


// What the plan kernel does for this one, done by every CTA for itself: a warp per sequence checks the topology and writes the
// paths of its nodes to the workspace (all CTAs the same values; a CTA reads what it has written).  A launch and its latencies
// less in front of a call of a few units.  scratch: 64 bytes a warp.
__device__ __forceinline__ void plan_paths(const Params &p, int warp, int n_warps, int lane, int8_t *scratch, int32_t *tab_base, int8_t *tab_n)
{
    int8_t *par = scratch + 64 * warp;
    for (int b = warp; b < p.B; b += n_warps) {
        const int base = p.node_offsets[b], n = p.node_offsets[b + 1] - base;
        int fault = 0;
        if (base < 0 || n < 0 || base + n > p.T || (b == p.B - 1 && base + n != p.T) || (b == 0 && base != 0))
            fault = SPECA_STATUS_BAD_OFFSETS;
        else if (n > p.max_nodes)
            fault = SPECA_STATUS_TOO_MANY;
        if (!fault) {
            for (int i = lane; i < n; i += 32) {
                const int pa = p.parent != nullptr ? p.parent[base + i] : i - 1;       // no parent array: chain
                if (pa < -1 || pa >= i) fault = SPECA_STATUS_BAD_PARENT;
                par[i] = int8_t(pa);
            }
            fault = __reduce_or_sync(0xffffffffu, fault);
            __syncwarp();                                        // (the reduction orders no memory)
        }
        if (!fault)
            for (int i = lane; i < n; i += 32) {
                const int d = write_path(p.ws, base, i, par);
                if (d > p.max_depth) fault |= SPECA_STATUS_TOO_DEEP;
                if (p.depth_in != nullptr && p.depth_in[base + i] != d) fault |= SPECA_STATUS_BAD_DEPTH;
            }
        fault = __reduce_or_sync(0xffffffffu, fault);
        if (lane == 0) {
            if (fault && blockIdx.x == 0) atomicOr(p.status, fault);
            tab_base[b] = base;
            tab_n[b] = int8_t(fault ? -1 : n);
        }
        __syncwarp();
    }
    fence_proxy_async();                                         // the scratch becomes a slot of the TMA ring
}

// TP = value tiles per unit (d_v / 128), DK = key width, MAXN = nodes per sequence, MAXD = tree depth.
// FEW = a call of a few units per SM: launched beside the plan kernel, value tiles of a head on two SMs.  (In a long call
// every instruction of the ten roles counts, and the plain form is 1 to 2 % faster.)
template <int TP, int DK, int MAXN, int MAXD, bool FEW>
__global__ void __launch_bounds__(Roles<DK, MAXD>::kThreads, 1)
verify_effective_kernel(const __grid_constant__ CUtensorMap s0_map, const __grid_constant__ EMaps maps, EParams ep)
{
    using LY = Lay<DK, MAXN, MAXD>;
    using RO = Roles<DK, MAXD>;
    constexpr int NS = LY::NS, NC = LY::NC, SC = LY::SC, SCB = LY::SCB;
    extern __shared__ __align__(1024) uint8_t smem[];
    const Params &p = ep.p;
    const uint32_t sbase = smem_u32(smem);
    if (sbase & 1023u) {                                 // never expected; refuse to run rather than corrupt
        if (threadIdx.x == 0) atomicOr(p.status, SPECA_STATUS_TIMEOUT);
        return;
    }
    const uint32_t bars = sbase + LY::OffBars;
    auto bar = [&](int i) { return bars + 8u * uint32_t(i); };
    volatile int *abort_flag = reinterpret_cast<volatile int *>(smem + LY::OffMisc);
    volatile uint32_t *tmem_slot = reinterpret_cast<volatile uint32_t *>(smem + LY::OffMisc + 8);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;

    if (threadIdx.x == 0) {
        *abort_flag = 0;
        for (int s = 0; s < kMaxSlots; ++s) { mbar_init(bar(kFull + s), 1); mbar_init(bar(kEmpty + s), 4); }
#pragma unroll 1
        for (int i = 0; i < 2; ++i) {
            mbar_init(bar(kAReady + i), 4);
            mbar_init(bar(kAFree + i), 1);
            mbar_init(bar(kKQFull + i), 1);
            mbar_init(bar(kKQFree + i), 2);
            mbar_init(bar(kVFull + i), 1);
            mbar_init(bar(kVFree + i), 8);
            mbar_init(bar(kAccFull + i), 1);
            mbar_init(bar(kAccFree + i), 8);
            mbar_init(bar(kGamReady + i), 4);
            mbar_init(bar(kOutFull + i), 1);
            mbar_init(bar(kMReady + i), 4);
            mbar_init(bar(kMFree + i), 1);
        }
        mbar_init(bar(kXReady), 8);
        mbar_init(bar(kGramFull), 1);
        mbar_init(bar(kGramFree), 4);
        mbar_init(bar(kSync), 4);
        mbar_init(bar(kDrain), 2);
#pragma unroll 1
        for (int i = 0; i < kUnitRing; ++i) mbar_init(bar(kUnit + i), 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if constexpr (FEW) {
        // While the kernel in front drains (it may still write the state: this only brings it into L2), the first tile of the
        // first unit is on its way.
        if (warp == 1) tmem_alloc(smem_u32(const_cast<uint32_t *>(tmem_slot)), kTmemCols);
        if (threadIdx.x == 0) prefetch_l2(p.S0 + size_t(blockIdx.x) * p.DV * DK, uint32_t(kRows * DK * 4));
        wait_for_previous_kernel();
        if (ep.own_plan)
            plan_paths(p, warp, RO::kThreads / 32, lane, reinterpret_cast<int8_t *>(smem + LY::OffRing),
                       reinterpret_cast<int32_t *>(smem + LY::OffWalk), reinterpret_cast<int8_t *>(smem + LY::OffWalk + 4 * kWalkSeqs));
    }
    for (int b = threadIdx.x; b < p.B && b < kWalkSeqs && !(FEW && ep.own_plan); b += blockDim.x) {
        const int n = p.ws.seq_n[b];
        reinterpret_cast<int32_t *>(smem + LY::OffWalk)[b] = p.node_offsets[b];
        reinterpret_cast<int8_t *>(smem + LY::OffWalk + 4 * kWalkSeqs)[b] = int8_t(n < 0 ? -1 : n);
    }
    if (!FEW && warp == 1) tmem_alloc(smem_u32(const_cast<uint32_t *>(tmem_slot)), kTmemCols);
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem_base = *tmem_slot;

    // record of unit `s` of this CTA's list; false: the list has ended, or (ok == false) the CTA is aborting
    bool ok = true;
    Unit x;
    auto unit = [&](uint32_t s, Unit &y) -> bool {
        if (!(ok = wait_fast(bar(kUnit + (s % kUnitRing)), (s / kUnitRing) & 1, abort_flag))) return false;
        const int4 *rec = reinterpret_cast<const int4 *>(smem + LY::OffUnit) + 2 * (s % kUnitRing);
        const int4 r = rec[0];
        const int2 e = *reinterpret_cast<const int2 *>(rec + 1);
        y = Unit{r.x, r.y, r.z, r.w, e.x, e.y};
        return r.y > 0;
    };
    auto padded = [](const Unit &y) { return (y.n + 15) & ~15; };
    auto head_of = [&](const Unit &y) { return FEW ? y.h >> ep.share : y.h; };

    const uint32_t lead = elect_one();                           // the thread that issues this warp's tcgen05 instructions

    if (warp == 0) {
        // ------------------------------------------------------------- TMA producer: state slices
        uint32_t it = 0;
        PROF_DECL
        for (uint32_t useq = 0; ok && unit(useq, x); ++useq) {
#pragma unroll 1
            for (int e = 0; e < TP * NC; ++e, ++it) {
                const int s = it % NS;
                if (!(ok = WAIT(0, bar(kEmpty + s), ((it / NS) & 1) ^ 1))) break;
                if (lane == 0 && !(ep.withhold_first_load && blockIdx.x == 0 && it == 0)) {
                    mbar_arrive_expect_tx(bar(kFull + s), kSliceBytes);
                    tma_load_3d(sbase + LY::OffRing + s * kSliceBytes, &s0_map, (e % NC) * 32, (e / NC) * kRows, x.u, bar(kFull + s));
                }
                __syncwarp();
            }
        }
        PROF_STORE()
    } else if (warp == 1) {
        // ------------------------------------------------------------- MMA issuer: S0 [K;Q]^T
        uint32_t it = 0, q = 0, useq = 0;                        // slices, tiles, units
        PROF_DECL
        for (; ok && unit(useq, x); ++useq) {
            const int par = useq & 1;
            const uint32_t idm = make_idesc_bf16(2 * padded(x));
            const uint32_t stage = sbase + LY::OffStage + par * LY::STAGE;
            if (!(ok = WAIT(0, bar(kKQFull + par), (useq >> 1) & 1))) break;
#pragma unroll 1
            for (int t = 0; t < TP && ok; ++t, ++q) {
                const uint32_t acc = tmem_base + (q & 1) * kTileCols;
                if (!(ok = WAIT(1, bar(kAccFree + (q & 1)), ((q >> 1) & 1) ^ 1))) break;
#pragma unroll 1
                for (int c = 0; c < NC; ++c, ++it) {
                    const int ab = it & 1;
                    if (!(ok = WAIT(2, bar(kAReady + ab), (it >> 1) & 1))) break;
                    tc_fence_after();
                    const uint32_t a = tmem_base + kAOff + ab * kACols;
                    const uint64_t bd = make_desc(stage + (c >> 1) * SCB + (c & 1) * 64);
#pragma unroll
                    for (int ks = 0; ks < 2; ++ks)
#pragma unroll
                        for (int pc = 0; pc < 3; ++pc)           // (32 bytes further on: 2 in the descriptor's address field)
                            mma_bf16_ts(acc, a + 16 * pc + 8 * ks, bd + 2 * ks, idm, (c | ks | pc) != 0, lead);
                    mma_commit(bar(kAFree + ab), lead);
                    if (c == NC - 1) {
                        mma_commit(bar(kAccFull + (q & 1)), lead);
                        if (t == TP - 1) mma_commit(bar(kKQFree + par), lead);
                    }
                }
            }
        }
        PROF_STORE()
    } else if (warp == 2) {
        // ------------------------------------------------------------- MMA issuer: Gram blocks one unit ahead, x M^T
        uint32_t q = 0, useq = 0, gseq = 0;
        PROF_DECL
        // pass s issues the Gram block of unit s, [K;Q] (128 rows) x K^T (R columns) from the staged rows, and the
        // products of unit s - 1
        for (bool first = true; ok; first = false) {
            if (unit(gseq, x)) {
                const int par = gseq & 1, npad = padded(x);
                if (!(ok = WAIT(0, bar(kKQFull + par), (gseq >> 1) & 1))) break;
                if (!(ok = WAIT(1, bar(kGramFree), (gseq & 1) ^ 1))) break;
                tc_fence_after();
                const uint32_t idg = make_idesc_bf16(npad);
                // in as many chains as the 64 columns hold, each from zero: the solver adds them up
                const int run = 4 * SC / gram_parts(npad);
#pragma unroll 1
                for (int i = 0, col = kGramOff; i < 4 * SC; i += run, col += npad)
#pragma unroll 1
                    for (int k = i; k < i + run; k += 2) {
                        const uint64_t d = make_desc(sbase + LY::OffStage + par * LY::STAGE + (k >> 2) * SCB + (k & 2) * 32);
                        mma_bf16(tmem_base + col, d, d, idg, k != i, lead);
                        mma_bf16(tmem_base + col, d + 2, d + 2, idg, 1, lead);
                    }
                mma_commit(bar(kGramFull), lead);
                mma_commit(bar(kKQFree + par), lead);
                ++gseq;
            }
            if (first) continue;
            if (!ok || !unit(useq, x)) break;
            const int npad = padded(x);
            const bool small = npad <= 32;
            const int ksteps = npad >> 4, mbuf = useq & 1;
            const uint32_t idx = make_idesc_bf16(npad);
            if (!(ok = WAIT(2, bar(kMReady + mbuf), (useq >> 1) & 1))) break;
#pragma unroll 1
            for (int t = 0; t < TP; ++t, ++q) {
                if (!(ok = WAIT(3, bar(kXReady), q & 1))) break;
                tc_fence_after();
                const uint32_t acc = tmem_base + (q & 1) * kTileCols, xa = tmem_base + kXOff;
                const uint64_t md = make_desc(sbase + LY::OffM + (small && mbuf ? LY::MBUF2 : 0));
#pragma unroll
                for (int order = 2; order >= 0; --order)          // small products first: 2^-16, 2^-8, the large ones
#pragma unroll 1
                    for (int ks = 0; ks < ksteps; ++ks)
#pragma unroll
                        for (int xp = order; xp >= 0; --xp)
                            mma_bf16_ts(acc, xa + 32 * xp + 8 * ks, md + uint64_t((order - xp) * (LY::MPIECE >> 4) + 2 * ks), idx,
                                        !(order == 2 && ks == 0 && xp == 2), lead);
                mma_commit(bar(kOutFull + (q & 1)), lead);
                if (t == TP - 1) mma_commit(bar(kMFree + mbuf), lead);
            }
            ++useq;
        }
        PROF_STORE()
    } else if (warp == 3) {
        // ------------------------------------------------------------- TMA producer: staged [K;Q] rows, value rows
        // (and the walk: unit s + 1 is handed out before the rows of unit s are asked for)
        Walk walk;
        walk.HG = ep.heads_per_group; walk.gpl = ep.gpl;
        walk.L = p.L; walk.B = p.B; walk.H = p.H; walk.T = p.T;
        walk.dl = ep.dl; walk.db = ep.db; walk.dg = ep.dg;
        walk.two = ep.want_u;
        walk.seq_n = p.ws.seq_n; walk.offs = p.node_offsets;
        walk.tab = smem + LY::OffWalk;
        walk.hi = walk.HG;                                       // before the first unit
        walk.ng = int(blockIdx.x) % ep.gpl; walk.nb = int(blockIdx.x) / ep.gpl % p.B; walk.nl = int(blockIdx.x) / ep.gpl / p.B;
        Unit kx, ux;
        ux.kind = 1;
        uint32_t kseq = 0, q = 0, pub = 0, useq = 0;
        auto publish = [&]() {
            next_unit(walk, ux);
            if (lane == 0) {
                int4 *rec = reinterpret_cast<int4 *>(smem + LY::OffUnit) + 2 * (pub % kUnitRing);
                rec[0] = make_int4(ux.u, ux.n, ux.z, ux.h);
                rec[1] = make_int4(ux.base, ux.kind, 0, 0);
                mbar_arrive(bar(kUnit + (pub % kUnitRing)));
            }
            __syncwarp();
            ++pub;
        };
        PROF_DECL
        publish();
        kx = ux;
        for (bool first = true; ok; first = false) {             // staged rows one unit ahead of the value rows
            if (kx.n > 0) {
                publish();
                const int par = kseq & 1, npad = padded(kx);
                if (!(ok = WAIT(0, bar(kKQFree + par), ((kseq >> 1) & 1) ^ 1))) break;
                if (lane == 0) {
                    const int m = (npad >> 4) - 1, z = kx.z;
                    const uint32_t stage = sbase + LY::OffStage + par * LY::STAGE;
                    mbar_arrive_expect_tx(bar(kKQFull + par), uint32_t(4 * npad * DK));
#pragma unroll 1
                    for (int c = 0; c < SC; ++c) {
                        tma_load_3d(stage + c * SCB, &maps.k[m], c * 64, head_of(kx), z, bar(kKQFull + par));
                        tma_load_3d(stage + c * SCB + npad * 128, &maps.q[m], c * 64, head_of(kx), z, bar(kKQFull + par));
                    }
                }
                __syncwarp();
                ++kseq;
                kx = ux;
            }
            if (first) continue;
            if (!unit(useq++, x)) break;
#pragma unroll 1
            for (int t = 0; t < TP; ++t, ++q) {
                const int vb = q & 1;
                if (!(ok = WAIT(1, bar(kVFree + vb), ((q >> 1) & 1) ^ 1))) break;
                if (lane == 0) {
                    mbar_arrive_expect_tx(bar(kVFull + vb), uint32_t(padded(x) * kRows * 2));
                    tma_load_3d(sbase + LY::OffV + vb * LY::VBUF, &maps.v[(padded(x) >> 4) - 1], t * kRows, x.h, x.z,
                                bar(kVFull + vb));
                }
                __syncwarp();
            }
        }
        PROF_STORE()
    } else if (warp < RO::kEpilogue) {
        // ------------------------------------------------------------- split: slice -> three bf16 pieces in TMEM
        const int row = 32 * (warp & 3) + lane;                  // slice row = TMEM lane of this thread
        const int sgrp = (warp - 4) >> 2;                   // two groups, alternating slices
        const uint32_t abase = tmem_base + kAOff + (uint32_t(32 * (warp & 3)) << 16);
        uint32_t it = 0;
        PROF_DECL
        for (uint32_t useq = 0; ok && unit(useq, x); ++useq) {
#pragma unroll 1
            for (int e = 0; e < TP * NC; ++e, ++it) {
                const int s = it % NS, ab = it & 1;
                if (RO::kSplits == 2 && ab != sgrp) continue;
                if (!(ok = WAIT(0, bar(kFull + s), (it / NS) & 1))) break;
                const uint8_t *src = smem + LY::OffRing + s * kSliceBytes + row * 128;
                uint32_t p1[16], p2[16], p3[16];
#pragma unroll
                for (int j = 0; j < 8; ++j) {
                    const float4 v = *reinterpret_cast<const float4 *>(src + ((j ^ (row & 7)) << 4));
                    split_pair(v.x, v.y, p1[2 * j], p2[2 * j], p3[2 * j]);
                    split_pair(v.z, v.w, p1[2 * j + 1], p2[2 * j + 1], p3[2 * j + 1]);
                }
                // the loads must have been performed, not only issued, before the copy engine may write the slot again
                fence_proxy_async();
                warp_arrive(bar(kEmpty + s), lane);
                if (!(ok = WAIT(1, bar(kAFree + ab), ((it >> 1) & 1) ^ 1))) break;
                tc_fence_after();
                const uint32_t dst = abase + ab * kACols;
                tmem_st16(dst, p1);
                tmem_st16(dst + 16, p2);
                tmem_st16(dst + 32, p3);
                tmem_st_wait();
                tc_fence_before();
                warp_arrive(bar(kAReady + ab), lane);
            }
        }
        PROF_STORE()
    } else if (warp < RO::kSolver) {
        // ------------------------------------------------------------- epilogue
        // Step s takes tile s - 1 from x M^T to o, which frees its accumulators, and then tile s from R to x: the state product
        // of a tile runs under the second product of the one before it and under both of these.  (The other way round the
        // accumulators came free a whole state product later: 8-node units 4.9 us instead of 4.6.)  Columns go in chunks of
        // 8 nodes, alternately to the two warps of a lane quarter.
        const int grp = (warp - RO::kEpilogue) >> 2;
        const int row = 32 * (warp & 3) + lane;
        const uint32_t lane_addr = uint32_t(32 * (warp & 3)) << 16;
        const uint32_t xb = tmem_base + kXOff + lane_addr;
        const size_t stride = size_t(p.H) * p.DV;
        uint32_t q = 0, useq = 0xffffffffu;
        int t = TP - 1, npad = 0, pn = 0, pR = 0;                // tile of the unit; nodes and rows of the last tile's unit (0: none)
        const float *pgf = nullptr;
        float *pdst = nullptr;
        bool more = true;
        PROF_DECL
        while (ok) {
            if (more && ++t == TP) {
                t = 0;
                ++useq;
                more = unit(useq, x);
                npad = padded(x);
            }
            if (!ok || (pn == 0 && !more)) break;
            const uint32_t slot = q & 1, ps = slot ^ 1;
            if (pn > 0 && !(ok = WAIT(4, bar(kOutFull + ps), ((q - 1) >> 1) & 1))) break;
            const float *gx = reinterpret_cast<const float *>(smem + LY::OffGam) + (useq & 3) * 2 * MAXN;
            if (pn > 0) {
                tc_fence_after();
                PROF_T0()
                const uint32_t acc = tmem_base + ps * kTileCols + lane_addr;
                float *dst = pdst + size_t(8 * grp) * stride;
#pragma unroll 1
                for (int c0 = 8 * grp; c0 < pn; c0 += 16, dst += 8 * stride) {
                    float d[8], g[8], gf[8];
                    tmem_ld8(acc + c0, d);
                    tmem_ld8(acc + pR + c0, g);
                    *reinterpret_cast<float4 *>(gf) = *reinterpret_cast<const float4 *>(pgf + c0);
                    *reinterpret_cast<float4 *>(gf + 4) = *reinterpret_cast<const float4 *>(pgf + c0 + 4);
                    tmem_ld_wait();
#pragma unroll
                    for (int i = 0; i < 8; ++i) {
                        if (c0 + i < pn) *dst = fmaf(gf[i], g[i], d[i]);
                        dst += stride;
                    }
                }
                tc_fence_before();
                warp_arrive(bar(kAccFree + ps), lane);
                PROF_ADD(7)
            }
            if (more) {
                if (!(ok = WAIT(0, bar(kVFull + slot), (q >> 1) & 1))) break;
                if (!(ok = WAIT(1, bar(kGamReady + (useq & 1)), (useq >> 1) & 1))) break;
                if (!(ok = WAIT(2, bar(kAccFull + slot), (q >> 1) & 1))) break;
                tc_fence_after();
                PROF_T0()
                const uint32_t acc = tmem_base + slot * kTileCols + lane_addr;
                const unsigned short *vt = reinterpret_cast<const unsigned short *>(smem + LY::OffV + slot * LY::VBUF) + row;
                // x of 8 nodes (clean: those that are not finite as zero), its sum times zero, the set of those not finite
                auto make_x = [&](int c0, bool clean, float2 &zero, uint32_t &odd) {
                    float r[8];
                    tmem_ld8(acc + c0, r);
                    uint32_t vv[8];
#pragma unroll
                    for (int i = 0; i < 8; ++i) vv[i] = vt[(c0 + i) * kRows];
                    float gm[8];
                    *reinterpret_cast<float4 *>(gm) = *reinterpret_cast<const float4 *>(gx + c0);
                    *reinterpret_cast<float4 *>(gm + 4) = *reinterpret_cast<const float4 *>(gx + c0 + 4);
                    tmem_ld_wait();
                    uint32_t p1[4], p2[4], p3[4];
#pragma unroll
                    for (int i = 0; i < 8; ++i) r[i] = fmaf(-gm[i], r[i], __uint_as_float(vv[i] << 16));
                    // rows past the last node belong to another sequence: they must not reach the product
                    if (c0 + 8 > x.n)
#pragma unroll
                        for (int i = 0; i < 8; ++i)
                            if (c0 + i >= x.n) r[i] = 0.f;
#pragma unroll
                    for (int i = 0; i < 8; i += 2) {
                        zero = __ffma2_rn(make_float2(r[i], r[i + 1]), make_float2(0.f, 0.f), zero);
                        if (clean) {
                            if (!(fabsf(r[i]) < INFINITY)) { odd |= 1u << i; r[i] = 0.f; }
                            if (!(fabsf(r[i + 1]) < INFINITY)) { odd |= 2u << i; r[i + 1] = 0.f; }
                        }
                        split_pair(r[i], r[i + 1], p1[i >> 1], p2[i >> 1], p3[i >> 1]);
                    }
                    if (clean && ((c0 >> 3) & 1) != grp) return;         // the other warp's chunk
                    tmem_st4(xb + (c0 >> 1), p1);
                    tmem_st4(xb + 32 + (c0 >> 1), p2);
                    tmem_st4(xb + 64 + (c0 >> 1), p3);
                };
                float2 zero = make_float2(0.f, 0.f);
                uint32_t none = 0u;
#pragma unroll 1
                for (int c0 = 8 * grp; c0 < npad; c0 += 16) make_x(c0, false, zero, none);
                if (__any_sync(0xffffffffu, !(zero.x + zero.y == 0.f))) {
                    // Both warps of the lane quarter may come here: each looks at all nodes, so that both write the same G.
                    // (R stays until all epilogue warps have arrived below.)
                    uint32_t odd_lo = 0u, odd_hi = 0u;
#pragma unroll 1
                    for (int c0 = 0; c0 < npad; c0 += 8) {
                        uint32_t odd = 0u;
                        make_x(c0, true, zero, odd);
                        if (c0 < 32) odd_lo |= odd << c0;
                        else odd_hi |= odd << (c0 - 32);
                    }
#pragma unroll 1
                    for (int i = 0; i < x.n; ++i) {
                        const int2 set = reinterpret_cast<const int2 *>(p.ws.set)[x.base + i];
                        const float g = tmem_ld1(acc + npad + i);
                        tmem_st1(acc + npad + i, ((uint32_t(set.x) & odd_lo) | (uint32_t(set.y) & odd_hi)) != 0u ? NAN : g);
                    }
                }
                tmem_st_wait();
                tc_fence_before();
                __syncwarp();
                if (lane == 0) { mbar_arrive(bar(kXReady)); mbar_arrive(bar(kVFree + slot)); }
                PROF_ADD(6)
            }
            pn = 0;
            if (more) {
                pn = x.n; pR = npad;
                pgf = gx + MAXN;
                pdst = (x.kind == 0 ? p.o : p.u) + size_t(x.z * p.H + x.h) * p.DV + t * kRows + row;
            }
            ++q;
        }
        PROF_STORE()
    } else {
        // ------------------------------------------------------------- solver, one unit ahead
        const int grow = 32 * (warp & 3) + lane;                 // Gram row (= TMEM lane) of this thread
        const uint32_t gaddr = tmem_base + kGramOff + (uint32_t(32 * (warp & 3)) << 16);
        float *Gk = reinterpret_cast<float *>(smem + LY::OffGk), *Gq = reinterpret_cast<float *>(smem + LY::OffGq);
        constexpr int GSTR = LY::GSTR;
        uint32_t useq = 0, nsync = 0;
        bool was_small = false;
        PROF_DECL
        auto role_sync = [&]() -> bool {
            warp_arrive(bar(kSync), lane);
            const bool r = WAIT(0, bar(kSync), nsync & 1);
            ++nsync;
            return r;
        };
        // topology and gates of the node this thread's row belongs to, fetched one unit ahead: its root path upward (one
        // byte per step, zero past the end), the set of its nodes, its length
        uint32_t up_n[4] = {0u, 0u, 0u, 0u}, lo_n = 0u, hi_n = 0u;
        int d_n = 0;
        float alpha_n = 1.f, beta_n = 0.f;
        auto fetch_topo = [&](const Unit &y) {
            const int node = grow < padded(y) ? grow : grow - padded(y);
            d_n = 0;
            if (node < y.n) {
                const int i = y.base + node;
                if (MAXD <= 8) {
                    const int2 w = reinterpret_cast<const int2 *>(p.ws.up)[2 * i];
                    up_n[0] = uint32_t(w.x); up_n[1] = uint32_t(w.y);
                } else {
                    const int4 w = reinterpret_cast<const int4 *>(p.ws.up)[i];
                    up_n[0] = uint32_t(w.x); up_n[1] = uint32_t(w.y); up_n[2] = uint32_t(w.z); up_n[3] = uint32_t(w.w);
                }
                const int2 s = reinterpret_cast<const int2 *>(p.ws.set)[i];
                lo_n = uint32_t(s.x); hi_n = uint32_t(s.y);
                d_n = p.ws.depth[i];
                const int r = FEW ? ((y.z + node) * p.H + y.h) >> ep.share : (y.z + node) * p.H + y.h;
                alpha_n = p.alpha[r];
                beta_n = p.beta[r];
            }
        };
        Unit nx;
        bool have = unit(0, nx);
        if (have) fetch_topo(nx);
        for (; have && ok; ++useq) {
            x = nx;
            const int R = padded(x);
            const bool is_k = grow < R, small = R <= 32;
            const int node = is_k ? grow : grow - R;
            const int d = grow < 2 * R ? d_n : 0;                // zero: a row without a node
            uint32_t up[MAXD / 4];
#pragma unroll
            for (int i = 0; i < MAXD / 4; ++i) up[i] = up_n[i];
            uint32_t set_lo = d > 0 ? lo_n : 0u, set_hi = d > 0 ? hi_n : 0u;
            float *alpha_s = reinterpret_cast<float *>(smem + LY::OffAB) + (useq & 1) * 2 * MAXN, *beta_s = alpha_s + MAXN;
            uint8_t *depth_s = smem + LY::OffDepth + (useq & 1) * MAXN;
            if (is_k) {
                depth_s[node] = uint8_t(d);
                alpha_s[node] = alpha_n;
                beta_s[node] = beta_n;
                // (the key rows' own entry, distance 0, is not needed)
                if (node < 32) set_lo &= ~(1u << node);
                else set_hi &= ~(1u << (node & 31));
            }
            auto path = [&](int r) -> int { return int((up[r >> 2] >> (8 * (r & 3))) & 0xffu); };
            have = unit(useq + 1, nx);
            if (!ok) break;
            if (have) fetch_topo(nx);
            if (!(ok = role_sync())) break;                      // depths and gates visible; the last unit's entries are dead

            // Gram row of this thread, 16 columns at a time: the entries against the nodes of its own path, filed by the
            // distance up the path
            if (!(ok = WAIT(1, bar(kGramFull), useq & 1))) break;
            tc_fence_after();
            {
                PROF_T0()
                float *G = (is_k ? Gk - 1 : Gq) + node * GSTR + d;
                const int end = gram_parts(R) * R;
#pragma unroll 1
                for (int c0 = 0; c0 < R; c0 += 8) {
                    float g[8];
                    tmem_ld8(gaddr + c0, g);
                    const uint2 dep = *reinterpret_cast<const uint2 *>(depth_s + c0);
                    const uint32_t bits = (c0 & 32 ? set_hi : set_lo) >> (c0 & 24);
                    tmem_ld_wait();
#pragma unroll 1
                    for (int c1 = c0 + R; c1 < end; c1 += R) {
                        float more[8];
                        tmem_ld8(gaddr + c1, more);
                        tmem_ld_wait();
#pragma unroll
                        for (int i = 0; i < 8; ++i) g[i] += more[i];
                    }
#pragma unroll
                    for (int i = 0; i < 8; ++i)
                        if (bits & (1u << i)) G[-int(((i < 4 ? dep.x : dep.y) >> (8 * (i & 3))) & 0xffu)] = g[i];
                }
                tc_fence_before();
                warp_arrive(bar(kGramFree), lane);
                PROF_ADD(5)
            }
            if (!(ok = role_sync())) break;                      // every row's entries visible

            // back substitution up the node's own path (entries past its end only ever reach others past the end)
            float c[MAXD];
            if (is_k) {
                PROF_T0()
#pragma unroll
                for (int i = 0; i < MAXD / 4; ++i) {
                    float4 v = make_float4(i == 0 ? 1.f : 0.f, 0.f, 0.f, 0.f);
                    if (x.kind == 0) v = *reinterpret_cast<const float4 *>(Gq + node * GSTR + 4 * i);
                    c[4 * i] = v.x; c[4 * i + 1] = v.y; c[4 * i + 2] = v.z; c[4 * i + 3] = v.w;
                }
#pragma unroll
                for (int r = 0; r < MAXD; ++r)
                    if (r < d) {
                        const int a = path(r);
                        c[r] *= beta_s[a];
                        if (!p.no_erase) {
                            const float *gr = Gk + a * GSTR;
#pragma unroll
                            for (int i = 0; i < MAXD - 1 - r; i += 4) {
                                const float4 v = *reinterpret_cast<const float4 *>(gr + i);
                                const float f[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
                                for (int e = 0; e < 4; ++e)
                                    if (r + 1 + i + e < MAXD) c[r + 1 + i + e] = fmaf(-c[r], f[e], c[r + 1 + i + e]);
                            }
                        }
                    }
                PROF_ADD(6)
            }
            // gamma, which the epilogue needs a product earlier than M, once the unit two before this one is done with (its
            // readers have then seen every phase of these barriers so far, and left the buffer of four units ago)
            if (useq >= 2 && !(ok = WAIT(2, bar(kMFree + (useq & 1)), ((useq >> 1) & 1) ^ 1))) break;
            if (is_k) {
                float gam = 1.f;
                const float front = x.kind == 0 ? p.scale : 1.f;
#pragma unroll
                for (int r = 0; r < MAXD; ++r) {
                    c[r] *= front * gam;                         // M[t][a_r]
                    if (r < d) gam *= alpha_s[path(r)];
                }
                float *gx = reinterpret_cast<float *>(smem + LY::OffGam) + (useq & 3) * 2 * MAXN;
                gx[node] = p.no_erase ? 0.f : gam;
                gx[MAXN + node] = x.kind == 0 ? p.scale * gam : 0.f;
            }
            warp_arrive(bar(kGamReady + (useq & 1)), lane);
            // the buffer of M: used by the unit two before this one, and, where one of them is large, by the last one
            if (useq >= 1 && !(small && was_small) && !(ok = WAIT(3, bar(kMFree + ((useq & 1) ^ 1)), ((useq - 1) >> 1) & 1))) break;
            was_small = small;
            if (is_k) {
                PROF_T0()
                // the node's row of M in three bf16 pieces, and its gamma
                uint8_t *mrow = smem + LY::OffM + (small && (useq & 1) ? LY::MBUF2 : 0) + node * 128;
#pragma unroll
                for (int i = 0; i < 8; ++i)
                    if (8 * i < R)
#pragma unroll
                        for (int pc = 0; pc < 3; ++pc)
                            *reinterpret_cast<uint4 *>(mrow + pc * LY::MPIECE + ((i ^ (node & 7)) << 4)) = make_uint4(0u, 0u, 0u, 0u);
#pragma unroll
                for (int r = 0; r < MAXD; ++r)
                    if (r < d) {
                        const int a = path(r);
                        uint32_t p1, p2, p3;
                        split_pair(c[r], 0.f, p1, p2, p3);
                        uint8_t *m = mrow + (((a >> 3) ^ (node & 7)) << 4) + (a & 7) * 2;
                        *reinterpret_cast<unsigned short *>(m) = (unsigned short)(p1);
                        *reinterpret_cast<unsigned short *>(m + LY::MPIECE) = (unsigned short)(p2);
                        *reinterpret_cast<unsigned short *>(m + 2 * LY::MPIECE) = (unsigned short)(p3);
                    }
                fence_proxy_async();
                PROF_ADD(7)
            }
            warp_arrive(bar(kMReady + (useq & 1)), lane);
        }
        PROF_STORE()
    }
    if (FEW && warp == 0) let_next_kernel_in();
    if (warp == 1 || warp == 2) {
        // everything these warps issued must have completed before TMEM is released
        mma_commit(bar(kDrain), lead);
        mbar_wait(bar(kDrain), 0, abort_flag);
    }
    if ((warp == 0 || warp == 3) && *abort_flag) {
        // let copies still in flight land before the CTA's shared memory goes away
        const uint64_t t0 = global_timer_ns();
        while (global_timer_ns() - t0 < 200000ull) __nanosleep(1000);
    }

    tc_fence_before();
    __syncthreads();
    if (threadIdx.x == 0 && *abort_flag) atomicOr(p.status, SPECA_STATUS_TIMEOUT);
    if (warp == 1) {
        tc_fence_after();
        tmem_dealloc(tmem_base, kTmemCols);
    }
}

template <int N> using Int = std::integral_constant<int, N>;

std::atomic<bool> g_opted_in[64];                        // per device: shared memory of every instantiation

}  // namespace

bool effective_supported(const speca_dims *d)
{
    if (d->d_k != 128 && d->d_k != 256) return false;
    if (d->d_v != kRows && d->d_v != 2 * kRows) return false;
    if (d->max_depth > 16) return false;
    return d->max_nodes <= (d->d_k == 128 ? 64 : 32);
}

static int g_withhold_first_load = 0;
void effective_set_withhold(int on) { g_withhold_first_load = on; }

int launch_verify_effective(const Params &call, int d_k, cudaStream_t st)
{
    if (d_k != 128 && d_k != 256) return int(cudaErrorInvalidValue);
    EncodeTiledFn encode = encode_tiled_fn();
    if (encode == nullptr) return int(cudaErrorNotSupported);
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return int(cudaErrorInvalidDevice);
    const long sms = sm_count_of_current_device();
    if (sms <= 0) return int(cudaErrorInvalidDevice);
    // Few units leave SMs idle, or with one unit while others work on two.  A head of two value tiles then counts as two
    // heads of one tile that share keys, queries and gates: states, value rows and outputs already lie that way.  The
    // coefficients are made twice, and a unit's solve takes as long whatever its value rows, so this pays while every half has
    // an SM of its own (us, split / whole, d_k = 128, 64 nodes, 48 units: 10.5 / 12.3, at 16 levels 11.6 / 13.2; d_k = 256, 32
    // nodes 9.8 / 11.4, 10.7 / 12.3) and, for up to 8 levels, where the busiest SM walks fewer tiles of few (192 units 18.6 /
    // 19.2 and 17.8 / 18.6, at 16 levels 21.4 / 20.1 and 20.7 / 20.0; 480 units, the last that do, 35.3 / 33.2 and 33.3 / 33.9;
    // 96, 240, 288 and 384 units, which do not, 4 to 13 % slower split, at 16 levels 11 to 26 %).
    Params p = call;
    const int heads = p.H;
    const long whole = (long(p.L) * p.B * p.H + sms - 1) / sms, halves = (2L * p.L * p.B * p.H + sms - 1) / sms;
    const int share = p.DV == 2 * kRows && (halves == 1 || (p.max_depth <= 8 && halves < 2 * whole && whole <= 4)) ? 1 : 0;
    p.H <<= share;
    p.DV >>= share;
    const long n_units = long(p.L) * p.B * p.H;
    // Launched beside the plan kernel where that is a part of the whole that counts (384 units of 64 nodes 37.9 -> 35.8 us,
    // 12288 units not measurable), or without one while every warp of a CTA has a sequence at most (us with / without: 192 units
    // of one sequence at d_k = 256 24.2 / 21.2, 16 units 10.1 / 9.5, 768 units of 2 sequences 42.5 / 41.5, 384 of 24 27.3 / 26.9;
    // of 32 34.5 / 36.3, of 40 35.9 / 37.2).
    const bool few = share != 0 || n_units < 8 * sms, own_plan = few && p.B <= 20 && p.skip_nodes == 0;
    if (!own_plan) {
        p.plan_paths_only = 1;
        const int rc = launch_plan(p, st);
        if (rc != 0) return rc;
    }
    const cuuint32_t es[3] = {1, 1, 1};
    CUtensorMap map;
    {
        const cuuint64_t gdim[3] = {cuuint64_t(d_k), cuuint64_t(p.DV), cuuint64_t(n_units)};
        const cuuint64_t gstride[2] = {cuuint64_t(d_k) * sizeof(float), cuuint64_t(p.DV) * d_k * sizeof(float)};
        const cuuint32_t box[3] = {32, kRows, 1};
        CUresult r = encode(&map, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 3, const_cast<float *>(p.S0), gdim, gstride, box, es,
                            CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                            CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
        if (r != CUDA_SUCCESS) return int(cudaErrorInvalidValue);
    }
    EMaps em;
    {
        const cuuint64_t gd[3] = {cuuint64_t(d_k), cuuint64_t(heads), cuuint64_t(p.L) * cuuint64_t(p.T)};
        const cuuint64_t gs[2] = {cuuint64_t(d_k) * 2, cuuint64_t(heads) * d_k * 2};
        const cuuint64_t vd[3] = {cuuint64_t(p.DV), cuuint64_t(p.H), cuuint64_t(p.L) * cuuint64_t(p.T)};
        const cuuint64_t vs[2] = {cuuint64_t(p.DV) * 2, cuuint64_t(p.H) * p.DV * 2};
        for (int m = 0; m < 4 && 16 * m < p.max_nodes; ++m) {    // box heights a sequence of this call can need
            const cuuint32_t bx[3] = {64, 1, cuuint32_t(16 * (m + 1))};
            CUresult r1 = encode(&em.k[m], CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, const_cast<__nv_bfloat16 *>(p.k), gd, gs, bx,
                                 es, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
                                 CU_TENSOR_MAP_L2_PROMOTION_L2_128B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
            CUresult r2 = encode(&em.q[m], CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, const_cast<__nv_bfloat16 *>(p.q), gd, gs, bx,
                                 es, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
                                 CU_TENSOR_MAP_L2_PROMOTION_L2_128B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
            const cuuint32_t vx[3] = {kRows, 1, cuuint32_t(16 * (m + 1))};
            CUresult r3 = encode(&em.v[m], CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, const_cast<__nv_bfloat16 *>(p.v), vd, vs, vx,
                                 es, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE,
                                 CU_TENSOR_MAP_L2_PROMOTION_L2_128B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
            if (r1 != CUDA_SUCCESS || r2 != CUDA_SUCCESS || r3 != CUDA_SUCCESS) return int(cudaErrorInvalidValue);
        }
    }

    if (!g_opted_in[dev].load(std::memory_order_acquire)) {
        cudaError_t e = cudaSuccess;
        auto opt_in = [&](const void *k, int bytes) {
            if (e == cudaSuccess) e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
        };
        auto all = [&](auto dk, auto mn) {
            constexpr int DK = decltype(dk)::value, MN = decltype(mn)::value;
            opt_in(reinterpret_cast<const void *>(verify_effective_kernel<1, DK, MN, 8, false>), Lay<DK, MN, 8>::Bytes);
            opt_in(reinterpret_cast<const void *>(verify_effective_kernel<1, DK, MN, 8, true>), Lay<DK, MN, 8>::Bytes);
            opt_in(reinterpret_cast<const void *>(verify_effective_kernel<2, DK, MN, 8, false>), Lay<DK, MN, 8>::Bytes);
            opt_in(reinterpret_cast<const void *>(verify_effective_kernel<2, DK, MN, 8, true>), Lay<DK, MN, 8>::Bytes);
            opt_in(reinterpret_cast<const void *>(verify_effective_kernel<1, DK, MN, 16, false>), Lay<DK, MN, 16>::Bytes);
            opt_in(reinterpret_cast<const void *>(verify_effective_kernel<1, DK, MN, 16, true>), Lay<DK, MN, 16>::Bytes);
            opt_in(reinterpret_cast<const void *>(verify_effective_kernel<2, DK, MN, 16, false>), Lay<DK, MN, 16>::Bytes);
            opt_in(reinterpret_cast<const void *>(verify_effective_kernel<2, DK, MN, 16, true>), Lay<DK, MN, 16>::Bytes);
        };
        all(Int<128>{}, Int<32>{});
        all(Int<128>{}, Int<64>{});
        all(Int<256>{}, Int<32>{});
        if (e != cudaSuccess) return int(e);
        g_opted_in[dev].store(true, std::memory_order_release);
    }
    EParams ep;
    ep.p = p;
    ep.want_u = p.u != nullptr ? 1 : 0;
    ep.withhold_first_load = g_withhold_first_load;
    ep.share = share;
    ep.own_plan = own_plan;
    // Consecutive heads of one (layer, sequence) that a CTA takes together.  Whole groups leave some CTAs longer lists than
    // others; what they save is steps of the walk, which one warp takes ahead of the roles.  Time of groups of 4 against single
    // heads, by units per SM, two runs: ragged trees of 8..64 nodes +9 % at 41, +4 at 83, +4 and +3 at 124, +4 at 145, +3 and
    // +2 at 166, +3 at 332; ragged at d_v = 128 -1 and +2 at 124, +2 and +1 at 249, +1 and 0 at 332; trees of 64 nodes +1 at
    // 166, of 20 0 and -1, of 64 at 16 levels +1, of 24 at d_k = 256 +1; of 32 at d_v = 128 +3 and -2 at 166, 0 at 83 and 332;
    // half chains and half 64-node trees at 332 -1.  The line at 128 keeps the last, the largest of the workloads served, and
    // pays for it with ragged batches beyond 128 (it was drawn when every role walked the list, and gained 3 to 7 % on short
    // units).
    ep.heads_per_group = p.H % 4 == 0 && n_units / 4 >= 32 * sms ? 4 : 1;
    const long n_groups = n_units / ep.heads_per_group;
    const int grid = int(n_groups < sms ? n_groups : sms);
    ep.gpl = p.H / ep.heads_per_group;
    ep.dg = grid % ep.gpl;
    ep.db = grid / ep.gpl % p.B;
    ep.dl = grid / ep.gpl / p.B;
    const bool one_tile = p.DV == kRows;
    const bool deep = p.max_depth > 8;
    auto go = [&](auto tp, auto dk, auto mn, auto md) {
        constexpr int TP = decltype(tp)::value, DK = decltype(dk)::value, MN = decltype(mn)::value, MD = decltype(md)::value;
        constexpr int bytes = Lay<DK, MN, MD>::Bytes, threads = Roles<DK, MD>::kThreads;
        if (few) launch(verify_effective_kernel<TP, DK, MN, MD, true>, grid, threads, bytes, st, map, em, ep);
        else verify_effective_kernel<TP, DK, MN, MD, false><<<grid, threads, bytes, st>>>(map, em, ep);
    };
    auto pick = [&](auto dk, auto mn) {
        if (one_tile) deep ? go(Int<1>{}, dk, mn, Int<16>{}) : go(Int<1>{}, dk, mn, Int<8>{});
        else deep ? go(Int<2>{}, dk, mn, Int<16>{}) : go(Int<2>{}, dk, mn, Int<8>{});
    };
    // a smaller node budget leaves room for a deeper ring of state slices
    if (d_k == 256) pick(Int<256>{}, Int<32>{});
    else if (p.max_nodes <= 32) pick(Int<128>{}, Int<32>{});
    else pick(Int<128>{}, Int<64>{});
    return int(cudaGetLastError());
}

}  // namespace speca

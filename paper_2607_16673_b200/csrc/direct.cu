// Verification of small draft trees with the state streamed straight into registers.
//
// Mathematics: the effective-query regrouping of the tree-masked factorisation (Section 4.2).  With
// a_0 = t, a_1, ... the root path of node t taken upward, gamma_t the product of alpha over it and
// rho_t[r] = alpha_{a_0} ... alpha_{a_{r-1}},
//        o_t = S0 qeff_t + sum_r M[t][a_r] v_{a_r}
//        qeff_t = scale gamma_t q_t - sum_r scale gamma_t cb_r k_{a_r}        M[t][a_r] = scale rho_t[r] cb_r
// where cb_r = c_r beta_{a_r} and c is the back substitution up the path
//        c_r = q_t.k_{a_r} - sum_{m<r} cb_m (k_{a_m}.k_{a_r}) .
// Everything that meets the state is then one product of the state tile with at most 8 NT vectors.
//
// Why warp-level MMAs and no staging.  A draft of a few nodes leaves the kernel bound by the state stream
// (a unit of 8 nodes does 0.8 M multiply-adds on 128 KB), and at this width a state tile never needs to be
// seen by more than one warp: lane (g, t) of a warp loads the 16-byte chunks t, t + 4, ... of rows g and g + 8
// of its 16-row tile, and those registers ARE the A fragments of mma.sync m16n8k8 (the contraction index is
// free to permute).  There is no ring, no barrier between roles and no shared-memory round trip of the
// state; while one CTA builds its coefficients the other resident CTAs stream.  The pipelined tcgen05 kernel
// spends most of a small unit on hand-overs between its roles instead.
//
// fp32 accuracy: both operands are split into a TF32 head and the remainder, from 17 nodes on into two fp16 of 11 bits each
// under a common scale, the low one apart by another 2^11 (three products; the dropped one is 2^-22 of the result).  fp16 has
// five bits of exponent: values that do not keep their bits under the scale of their 32 columns are looked for among the
// effective queries, and, only where these are so uneven that it could show, among the rows of the state, and are multiplied in
// TF32 instead.  M and the weights of the keys are split into three bf16 pieces and multiply bf16 rows exactly.  The tensor core
// truncates where it adds, relative to the largest term, accumulator included; a long chain of products in one accumulator
// loses a bit or two toward zero.  So the large sums (Gram entries, leading pieces, 32-column steps of the state product) start
// from zero and are added up in fp32 proper.  Error against 64 bits, 2-norm of the difference over that of the outputs, x
// 10^-8, chained / now / the route that takes the shape without this kernel: d_k = d_v = 64 (serial walk): chains of 8 15.0 /
// 7.2 / 7.2, of 16 15.0 / 7.9 / 7.1, trees of 30 15.0 / 6.9 / 7.2; 128 x 64 (serial walk): chains of 8 17.7 / 7.7 / 7.6, trees
// of 30 17.6 / 7.4 / 7.7; 128 x 256 (substitution kernel): chains of 8 17.6 / 7.7 / 15.4, trees of 30 17.6 / 7.3 / 14.1; 256 x
// 256, chains of 8 24.2 / 8.7 / 30.3.  (Of the part that comes from the state alone 14, the serial walk 7.6, the substitution
// kernel 90.)  It costs 2 to 6 % of a unit: 24576 units of 8 / 30 nodes at 64 x 64 142 / 326 us chained, 148 / 336 now, 12288
// units of 16 nodes at 128 x 256 388 and 394.
//
// The products run over all nodes of a block with zero weights off the path, and zero times a value that is not finite
// is no zero.  So where an output is not finite the CTA looks for such records (repair), takes them out of the products and
// goes over its rows once more: a node with the key on its path still gets it through its Gram entries, the value elements
// are put back at the end for the nodes that have them on their path, and the rest of the draft stays clean.  (Looking
// before the first pass took 2 to 12 % of a small unit.)
//
// A CTA takes one unit (layer, sequence, head) or a slice of its value rows and checks the topology of its sequence
// itself (one parent walk per node), so no plan kernel runs in front of it.  It asks the first rows of its tile into L2
// with one bulk prefetch, so that the set-up runs under the latency of HBM and the loop
// over 16-row tiles needs two 32-column steps of registers in flight, not whole tiles: 24 warps fit an SM.  Holding
// whole tiles in registers through the set-up (16 warps) took 5.1 us per 8-node unit and SM instead of 3.9, at 16
// nodes 8.0 instead of 4.4.
// Measured (d_k = 128, d_v = 256, 12288 units, the pipelined kernel with its plan in brackets): 8 nodes 296 us = 6.1 TB/s
// (293 us), 16 nodes 372 us = 5.5 TB/s (324 to 357); d_k = d_v = 64, 24576 units of 8 / 17 / 30 nodes: 143 / 270 / 305 us (serial
// walk 312 / 689 / 1288).  At d_k = 64 a unit of 17 nodes is 6400 warp instructions around 16 KB of state (half of the issue
// slots, 22 % of HBM); several heads a CTA with their records loaded ahead, or five CTAs an SM instead of four, gained nothing
// there.  What bounds it: the state stream at 8 nodes (93 % of the copy rate; 83 % at 16), above that the set-up (some thousand
// instructions a warp between ten barriers, issued every seventh cycle) and at 32 nodes the MMAs.  For a few users, 384 chains
// of 8: 10.1 us out of HBM.
#include <algorithm>
#include <atomic>

#include <cuda_fp16.h>

#include "speca_common.cuh"
#include "tc_ptx.cuh"

namespace speca {

namespace {

// (rounded: the remainder then fits TF32 but for its last bit; a value that is not finite stays one)
__device__ __forceinline__ uint32_t tf32_head(float x) { return (__float_as_uint(x) + 0x1000u) & 0xffffe000u; }
__device__ __forceinline__ uint32_t tf32_tail(float x) { return __float_as_uint(x - __uint_as_float(tf32_head(x))); }

// (not volatile: the compiler may interleave independent products)
__device__ __forceinline__ void warp_mma_tf32(float (&d)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1)
{
    asm("mma.sync.aligned.m16n8k8.row.col.f32.tf32.tf32.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, {%0, %1, %2, %3};"
        : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
        : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}
__device__ __forceinline__ void warp_mma_bf16(float (&d)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1)
{
    asm("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, "
                 "{%0, %1, %2, %3};"
                 : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
                 : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}
// the product alone (C = 0)
__device__ __forceinline__ void warp_mma_bf16_first(float (&d)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1)
{
    asm("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, "
                 "{%10, %10, %10, %10};"
                 : "=f"(d[0]), "=f"(d[1]), "=f"(d[2]), "=f"(d[3])
                 : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1), "f"(0.f));
}
template <bool FIRST>
__device__ __forceinline__ void warp_mma_f16(float (&d)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1)
{
    if (FIRST)
        asm("mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, "
            "{%10, %10, %10, %10};"
            : "=f"(d[0]), "=f"(d[1]), "=f"(d[2]), "=f"(d[3])
            : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1), "f"(0.f));
    else
        asm("mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, "
            "{%0, %1, %2, %3};"
            : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
            : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}
// Scale of a group of values of which the largest is m: the power of two that brings m into [2^14, 2^15), and the one that m
// has (m below 2^-112 counts as that).  32 products of two scaled values come to less than 2^36.  What undoes the scales is
// multiplied in so that no step leaves the range unless the result does: 2^-35 size of the state first, then 2^7 size of the
// effective query (up to kMostHalf, beyond that TF32).
struct HalfScale {
    float up, size;
    __device__ __forceinline__ explicit HalfScale(float m)
    {
        const uint32_t e = max(__float_as_uint(m) & 0x7f800000u, 15u << 23);
        up = __uint_as_float((268u << 23) - e);
        size = __uint_as_float(e);
    }
    // some value that is not zero does not keep its bits in a pair (in a group that is not finite all others)
    __device__ __forceinline__ bool loses(const float (&x)[8]) const
    {
        bool any = false;
#pragma unroll
        for (int e = 0; e < 8; ++e) any |= x[e] != 0.f && fabsf(x[e] * up) < 1.f / 8192.f;
        return any;
    }
};
constexpr float kLowPiece = 1.f / 2048.f;                        // what a low piece counts
constexpr float kUndoState = 0x1p-35f, kUndoQuery = 0x1p7f, kMostHalf = 0x1p120f;
__device__ __forceinline__ __half2 as_half2(uint32_t x) { return *reinterpret_cast<const __half2 *>(&x); }
// Two values, scaled, as a pair of fp16 and 2^11 times what is left of them as another, both rounded.  At most 2^-23 of a value
// is lost, as with TF32, down to 2^-27 of the largest of its group; below that 2^-51 of the largest.  (Were the low piece not
// scaled, it would be subnormal from 2^-16 of the largest on and lose a bit per binade.)
__device__ __forceinline__ void half_split(float x0, float x1, float up, uint32_t &hi, uint32_t &lo)
{
    const float2 y = __fmul2_rn(make_float2(x0, x1), make_float2(up, up));
    asm("cvt.rn.f16x2.f32 %0, %1, %2;" : "=r"(hi) : "f"(y.y), "f"(y.x));
    float2 z = __fmul2_rn(y, make_float2(2048.f, 2048.f));
    asm("{\n\t.reg .b16 h0, h1, m;\n\t"
        "mov.b16 m, 0xe800;\n\t"                                // -2^11
        "mov.b32 {h0, h1}, %2;\n\t"
        "fma.rn.f32.f16 %0, h0, m, %0;\n\t"
        "fma.rn.f32.f16 %1, h1, m, %1;\n\t}"
        : "+f"(z.x), "+f"(z.y) : "r"(hi));
    asm("cvt.rn.f16x2.f32 %0, %1, %2;" : "=r"(lo) : "f"(z.y), "f"(z.x));
}
// smallest magnitude of 8 values
__device__ __forceinline__ float least_of(const float (&x)[8])
{
    return fminf(fminf(fminf(fabsf(x[0]), fabsf(x[1])), fminf(fabsf(x[2]), fabsf(x[3]))),
                 fminf(fminf(fabsf(x[4]), fabsf(x[5])), fminf(fabsf(x[6]), fabsf(x[7]))));
}
// largest magnitude of 8 values, and of what the four lanes of a row hold
__device__ __forceinline__ float row_max(const float (&x)[8])
{
    float m = fmaxf(fmaxf(fmaxf(fabsf(x[0]), fabsf(x[1])), fmaxf(fabsf(x[2]), fabsf(x[3]))),
                    fmaxf(fmaxf(fabsf(x[4]), fabsf(x[5])), fmaxf(fabsf(x[6]), fabsf(x[7]))));
    m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, 1));
    return fmaxf(m, __shfl_xor_sync(0xffffffffu, m, 2));
}
__device__ __forceinline__ void ldsm_x4(uint32_t (&r)[4], const void *p)
{
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0, %1, %2, %3}, [%4];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(tc::smem_u32(p)) : "memory");
}
__device__ __forceinline__ void ldsm_x4_t(uint32_t (&r)[4], const void *p)
{
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0, %1, %2, %3}, [%4];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(tc::smem_u32(p)) : "memory");
}
// 32 bytes of a state row in one load; the state is read once per call
__device__ __forceinline__ void ld_state(float (&x)[8], const float *p)
{
    asm volatile("ld.global.L1::no_allocate.v8.f32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
                 : "=f"(x[0]), "=f"(x[1]), "=f"(x[2]), "=f"(x[3]), "=f"(x[4]), "=f"(x[5]), "=f"(x[6]), "=f"(x[7]) : "l"(p));
}
__device__ __forceinline__ bool finite(float x) { return (__float_as_uint(x) & 0x7f800000u) != 0x7f800000u; }
// the two bf16 of a word with those that are not finite replaced by zero
__device__ __forceinline__ uint32_t finite_pair(uint32_t w)
{
    return ((w & 0x7f80u) == 0x7f80u ? 0u : w & 0xffffu) | ((w & 0x7f800000u) == 0x7f800000u ? 0u : w & 0xffff0000u);
}
// 16 bytes global -> shared; live == false fills with zeros (the address is not read)
__device__ __forceinline__ void cp16(void *dst, const void *src, bool live)
{
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(tc::smem_u32(dst)), "l"(src), "r"(live ? 16 : 0)
                 : "memory");
}

// Shared memory of one CTA (bytes); N = 8 NT nodes at most, `rows` value rows.
template <int DK, int NT, int MAXD> struct Lay {
    static constexpr int N = 8 * NT;
    static constexpr int NK = (N + 15) & ~15;                   // contraction width of the value term
    static constexpr int KQS = DK + 8;                          // bf16 per staged key / query row (16 bytes of padding)
    // From 17 nodes on the tensor pipe bounds the state product (77 % of it, 384 units of 32 nodes), and its operands are pairs
    // of fp16, scaled by row and 32-column step: six products of 16 columns in the place of twelve of 8 in TF32.  us, TF32 /
    // fp16: 384 units of 32 nodes at d_k = d_v = 128 17.7 / 15.6, 192 at d_v = 256 18.0 / 15.4; d_k = d_v = 64, 9216 units of
    // 17..32 nodes 117.3 / 110.8, of 48..64 308 / 296; 256 x 64, 768 units of 32 nodes 66.2 / 38.6.  Below that the conversions
    // cost more than the products.
    static constexpr bool kHalf = NT >= 4;
    static constexpr int NS = DK / 32;                          // 32-column steps
    static constexpr int BS = DK + 4;                           // floats per effective-query row (16 bytes of padding)
    static constexpr int BSH = DK + 32;                         // fp16 per effective-query row (64 bytes: eight lanes, two
                                                                // rows, no conflict)
    static constexpr int MS = NK + 8;                           // bf16 per row of a piece of M
    static constexpr int GS = N + 1;
    static constexpr int NR = NK;                               // rows of the weight pieces: whole MMA row blocks
    // a node's path holds no later node, so row block m of the weights ends with column 16 m + 15
    __host__ __device__ static constexpr int w_row(int r)
    {
        return 128 * (r >> 4) * ((r >> 4) + 2) + (r & 15) * (16 * (r >> 4) + 24);
    }
    static constexpr int WP = w_row(NR);                        // bf16 per piece
    static constexpr int OffKQ = 0;                             // bf16 [2N][KQS]: key rows, query rows
    static constexpr int OffHi = OffKQ + 2 * N * KQS * 2;       // float [N][BS]
    static constexpr int OffLo = OffHi + (kHalf ? N * BSH * 2 : N * BS * 4);
    static constexpr int OffS = OffLo + N * BSH * 2;            // kHalf: float [NS][N], undoes the scale of a node's 32 columns
    static constexpr int OffG = OffHi;                          // float [2N][GS]: Gram rows of keys, queries (dead before Hi)
    static constexpr int kQEnd = kHalf ? OffS + NS * N * 4 : OffLo + N * BS * 4;
    static constexpr int kREnd = kQEnd > OffG + 2 * N * GS * 4 ? kQEnd : (OffG + 2 * N * GS * 4 + 15) & ~15;
    static constexpr int OffM = kREnd;                          // bf16 [3][N][MS]
    static constexpr int OffW = OffM + 3 * N * MS * 2;          // bf16 [3][WP]: weights of the keys in qeff
    static constexpr int OffP = OffW + 3 * WP * 2;         // int32 parent[N], float alpha[N], beta[N], scale gamma[NR]
    // rows of the back substitution: float c beta [N][MAXD], float rho [N][MAXD], uint8 path [N][MAXD]; behind the Gram
    // rows where those leave room, else over them (one barrier more), and as dead as they are afterwards
    static constexpr int GEnd = (OffG + 2 * N * GS * 4 + 15) & ~15, CBytes = 9 * N * MAXD;
    static constexpr bool kOver = GEnd + CBytes > kREnd;
    static constexpr int OffC = kOver ? OffG : GEnd;
    static constexpr int OffU = OffP + (3 * N + NR) * 4;        // kHalf: int, steps whose effective queries are uneven
    static constexpr int OffV = OffU + (kHalf ? 16 : 0);        // bf16 [NK][rows + 8]
    static_assert(OffG + CBytes <= GEnd || !kOver, "rows of the back substitution do not fit the space of the Gram rows");
    static constexpr int bytes(int rows) { return OffV + NK * (rows + 8) * 2; }
};

// Division by a number that is the same for the whole call, for dividends below 2^31: a product and a shift instead of some
// twenty instructions, of which every thread of a small unit had six.  (With the enumeration of the Gram blocks, us: 4608 units
// of 5..40 nodes at d_k = d_v = 64 90.7 -> 83.1, 9216 units of 9..16 nodes 78.7 -> 73.3, of 48..64 nodes 335 -> 309; one user
// of 64-wide heads, 20..40 nodes, 8.3 -> 7.6; chains of 8 at d_k = 128 9.0 -> 8.8.)
struct Divisor {
    uint32_t d, mul, shift;
    Divisor() = default;
    explicit Divisor(uint32_t by) : d(by), shift(31)
    {
        for (uint32_t x = by - 1; x != 0; x >>= 1) ++shift;     // 31 + ceil(log2 by)
        mul = uint32_t(((uint64_t(1) << shift) + by - 1) / by);
    }
    __device__ __forceinline__ int quotient(int n) const { return int(uint64_t(uint32_t(n)) * mul >> shift); }
};

struct DirectArgs {
    Params p;
    Divisor parts, H, B, vp;    // value-row slices per unit; heads, sequences; 16-byte pieces of a slice of a value row
    int32_t rows;               // value rows per slice
    int32_t lo;                 // sequences of at most this many nodes belong to another launch
    int32_t early;              // ask for the state before the records: see launch_one
};

// what a CTA works on
struct Unit {
    int part, unit, h, b, l;
    __device__ __forceinline__ explicit Unit(const DirectArgs &da)
    {
        unit = da.parts.quotient(int(blockIdx.x));
        part = int(blockIdx.x) - unit * int(da.parts.d);
        const int lb = da.H.quotient(unit);
        h = unit - lb * int(da.H.d);
        l = da.B.quotient(lb);
        b = lb - l * int(da.B.d);
    }
};

// some value of a tile does not keep its bits in an fp16 pair (cur: this lane's part of row g; only the steps given)
template <int DK> __device__ __forceinline__ bool loses_bits(const float *cur, int steps)
{
    bool loses = false;
#pragma unroll 1
    for (int q = 0; q < DK / 32; ++q) {
        if (!(steps >> q & 1)) continue;
        float xa[8], xb[8];
        ld_state(xa, cur + 32 * q);
        ld_state(xb, cur + 32 * q + 8 * DK);
        const HalfScale scale_a(row_max(xa)), scale_b(row_max(xb));
        loses |= scale_a.loses(xa) || scale_b.loses(xb);
    }
    return __any_sync(0xffffffffu, loses);
}
// The product of a tile with the effective queries in TF32 as below 17 nodes; these are put together again from their pairs, or
// taken as they are where they did not fit.
template <class LY, int NTP>
__device__ __forceinline__ void state_in_tf32(float (&x)[NTP][4], const float *cur, const uint16_t *high,
                                              const uint16_t *low, const float *scale, int ntp)
{
    constexpr float kOne = 0x1p-14f / kUndoQuery;                // of a scaled value, under what undoes its scale
    float xx[NTP][4] = {};                                       // the cross products
#pragma unroll
    for (int i = 0; i < NTP; ++i)
#pragma unroll
        for (int e = 0; e < 4; ++e) x[i][e] = 0.f;
#pragma unroll 1
    for (int q = 0; q < LY::NS; ++q) {
        float part[NTP][4] = {};
#pragma unroll 1
        for (int e = 32 * q; e < 32 * q + 8; e += 2) {
            const float2 xa = *reinterpret_cast<const float2 *>(cur + e);
            const float2 xb = *reinterpret_cast<const float2 *>(cur + e + 8 * 32 * LY::NS);
            const uint32_t ah[4] = {tf32_head(xa.x), tf32_head(xb.x), tf32_head(xa.y), tf32_head(xb.y)};
            const uint32_t al[4] = {tf32_tail(xa.x), tf32_tail(xb.x), tf32_tail(xa.y), tf32_tail(xb.y)};
#pragma unroll
            for (int i = 0; i < NTP; ++i) {
                if (NTP > 1 && i >= ntp) break;
                const uint32_t hi = *reinterpret_cast<const uint32_t *>(high + 8 * i * LY::BSH + e);
                const uint32_t lo = *reinterpret_cast<const uint32_t *>(low + 8 * i * LY::BSH + e);
                const float sc = scale[q * LY::N + 8 * i];
                const float2 h = __half22float2(as_half2(hi)), l = __half22float2(as_half2(lo));
                float w0 = fmaf(l.x, kLowPiece, h.x) * kOne * sc, w1 = fmaf(l.y, kLowPiece, h.y) * kOne * sc;
                w0 = sc != 0.f ? w0 : __uint_as_float(__byte_perm(lo, hi, 0x5410));
                w1 = sc != 0.f ? w1 : __uint_as_float(__byte_perm(lo, hi, 0x7632));
                const uint32_t b0 = tf32_head(w0), b1 = tf32_head(w1);
                warp_mma_tf32(xx[i], al, b0, b1);
                warp_mma_tf32(xx[i], ah, tf32_tail(w0), tf32_tail(w1));
                warp_mma_tf32(part[i], ah, b0, b1);
            }
        }
#pragma unroll
        for (int i = 0; i < NTP; ++i)
#pragma unroll
            for (int e = 0; e < 4; ++e) x[i][e] += part[i][e];
    }
#pragma unroll
    for (int i = 0; i < NTP; ++i)
#pragma unroll
        for (int e = 0; e < 4; ++e) x[i][e] += xx[i][e];
}

// After a pass with an output that is not finite.  First pass: keys and value elements that are not finite are replaced by
// zero in shared memory; true if there were any.  Second pass: the value elements are added for the nodes that have them on
// their path.
template <int DK, int NT, int MAXD, int THREADS>
__device__ __forceinline__ bool repair(const DirectArgs &da, uint8_t *smem, int pass)
{
    using LY = Lay<DK, NT, MAXD>;
    constexpr int N = LY::N;
    const Params &p = da.p;
    const Unit un(da);
    const int part = un.part, h = un.h, b = un.b, l = un.l, rows = da.rows;
    const int base = p.node_offsets[b], n = p.node_offsets[b + 1] - base;
    const long rec0 = (long(l) * p.T + base) * p.H + h;
    if (pass == 0) {
        int odd = 0;
        auto clean = [&](uint32_t *word) {
            const uint32_t w = finite_pair(*word);
            if (w != *word) { *word = w; odd = 1; }
        };
        for (int i = threadIdx.x; i < n * (DK / 2); i += THREADS)
            clean(reinterpret_cast<uint32_t *>(smem + LY::OffKQ) + i / (DK / 2) * (LY::KQS / 2) + i % (DK / 2));
        for (int i = threadIdx.x; i < n * (rows >> 1); i += THREADS)
            clean(reinterpret_cast<uint32_t *>(smem + LY::OffV) + i / (rows >> 1) * ((rows + 8) >> 1) + i % (rows >> 1));
        return __syncthreads_or(odd);
    }
    const int *par = reinterpret_cast<const int *>(smem + LY::OffP);
    for (int i = threadIdx.x; i < n * rows; i += THREADS) {
        const int t = i / rows, r = part * rows + i % rows;
        float sum = 0.f;
        for (int a = t; a >= 0; a = par[a]) {
            const float v = __bfloat162float(p.v[(rec0 + long(a) * p.H) * p.DV + r]);
            const __nv_bfloat16 *m = reinterpret_cast<const __nv_bfloat16 *>(smem + LY::OffM) + t * LY::MS + a;
            if (!finite(v))
                sum += v * (__bfloat162float(m[0]) + __bfloat162float(m[N * LY::MS]) + __bfloat162float(m[2 * N * LY::MS]));
        }
        if (sum != 0.f) p.o[(rec0 + long(t) * p.H) * p.DV + r] += sum;
    }
    return false;
}

template <int DK, int NT, int MAXD, int WARPS, int CTAS>
__global__ void __launch_bounds__(WARPS * 32, CTAS)
verify_direct_kernel(const __grid_constant__ DirectArgs da)
{
    after_previous_kernel();
    using LY = Lay<DK, NT, MAXD>;
    constexpr int N = LY::N, NS = DK / 32, THREADS = WARPS * 32;
    // a product wider than four column tiles is split between the warps: tile by tile, PARTS warps beside each other
    constexpr int NTP = NT > 4 ? 4 : NT, PARTS = NT / NTP, STRIDE = WARPS / PARTS;
    extern __shared__ __align__(16) uint8_t smem[];
    const Params &p = da.p;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, g = lane >> 2, t4 = lane & 3;

    const Unit un(da);
    const int part = un.part, unit = un.unit, h = un.h, b = un.b, l = un.l;
    const int row0 = part * da.rows;

    // the first tiles are asked into L2 before anything else is known when the sequence is certainly ours
    const float *S_cta = p.S0 + (long(unit) * p.DV + row0) * DK;
    const int tiles = da.rows >> 4;
    constexpr int AHEAD = DK == 256 ? 4 : 8;     // tiles requested ahead of the one a warp works on
    auto prefetch_first = [&]() {
        if (tid == 0) prefetch_l2(S_cta, uint32_t(min(tiles, AHEAD)) * (16 * DK * 4));
    };
    if (da.early) prefetch_first();

    const int base = p.node_offsets[b], end = p.node_offsets[b + 1];
    const int n = end - base;
    const bool reporter = l == 0 && h == 0 && part == 0 && tid == 0;
    if (base < 0 || n < 0 || end > p.T || (b == p.B - 1 && end != p.T) || (b == 0 && base != 0)) {
        if (reporter) atomicOr(p.status, SPECA_STATUS_BAD_OFFSETS);
        return;
    }
    if (n > p.max_nodes) {
        if (reporter) atomicOr(p.status, SPECA_STATUS_TOO_MANY);
        return;
    }
    if (p.parent == nullptr && n > p.max_depth) {            // a chain of n nodes is n levels deep
        if (reporter) atomicOr(p.status, SPECA_STATUS_TOO_DEEP);
        return;
    }
    if (n <= da.lo || n > N) return;                         // nothing to do, or another launch's
    __nv_bfloat16 *sKQ = reinterpret_cast<__nv_bfloat16 *>(smem + LY::OffKQ);
    float *sHi = reinterpret_cast<float *>(smem + LY::OffHi), *sLo = reinterpret_cast<float *>(smem + LY::OffLo);
    uint16_t *hHi = reinterpret_cast<uint16_t *>(smem + LY::OffHi), *hLo = reinterpret_cast<uint16_t *>(smem + LY::OffLo);
    float *sSc = reinterpret_cast<float *>(smem + LY::OffS);
    __nv_bfloat16 *sM = reinterpret_cast<__nv_bfloat16 *>(smem + LY::OffM);
    float *sG = reinterpret_cast<float *>(smem + LY::OffG);
    __nv_bfloat16 *sW = reinterpret_cast<__nv_bfloat16 *>(smem + LY::OffW);
    int *sPar = reinterpret_cast<int *>(smem + LY::OffP);
    float *sAl = reinterpret_cast<float *>(sPar + N), *sBe = sAl + N, *sGam = sBe + N;
    int *sUneven = reinterpret_cast<int *>(smem + LY::OffU);
    float *sC = reinterpret_cast<float *>(smem + LY::OffC);
    uint8_t *sPath = smem + LY::OffC + 8 * N * MAXD;
    __nv_bfloat16 *sV = reinterpret_cast<__nv_bfloat16 *>(smem + LY::OffV);
    const int vstride = da.rows + 8;
    const int nt = (n + 7) >> 3;
    const long rec0 = (long(l) * p.T + base) * p.H + h;      // record of node 0; node i is H records further on
    const int H = p.H;

    // ---- the sequence's records -> shared memory; rows past the last node are zero
    int pa = -1, fault = 0;
    float al = 1.f, be = 0.f;
    if (tid < n) {
        pa = p.parent != nullptr ? p.parent[base + tid] : tid - 1;
        al = p.alpha[rec0 + long(tid) * H];
        be = p.beta[rec0 + long(tid) * H];
    }
    {
        constexpr int PCS = DK / 8;
        for (int i = tid; i < 2 * 8 * nt * PCS; i += THREADS) {
            const int r = i / PCS, c = i % PCS;
            const bool is_q = r >= 8 * nt;
            const int node = is_q ? r - 8 * nt : r;
            const bool live = node < n;
            const __nv_bfloat16 *src = (is_q ? p.q : p.k) + (rec0 + long(live ? node : 0) * H) * DK + 8 * c;
            cp16(sKQ + (is_q ? N + node : node) * LY::KQS + 8 * c, src, live);
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
        const int vp = da.rows >> 3, vrows = (n + 15) & ~15;
        for (int i = tid; i < vrows * vp; i += THREADS) {
            const int node = da.vp.quotient(i), c = i - node * vp;
            const bool live = node < n;
            cp16(sV + node * vstride + 8 * c, p.v + (rec0 + long(live ? node : 0) * H) * p.DV + row0 + 8 * c, live);
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
        if (!da.early) prefetch_first();
        for (int i = tid; i < 3 * N * LY::MS / 8; i += THREADS) reinterpret_cast<uint4 *>(sM)[i] = make_uint4(0u, 0u, 0u, 0u);
        for (int i = tid; i < 3 * LY::WP / 8; i += THREADS) reinterpret_cast<uint4 *>(sW)[i] = make_uint4(0u, 0u, 0u, 0u);
        if (tid < LY::NR) sGam[tid] = 0.f;
        if (LY::kHalf && tid == 0) *sUneven = 0;
    }
    if (tid < n) {
        if (pa < -1 || pa >= tid) fault = SPECA_STATUS_BAD_PARENT;
        sPar[tid] = pa;
        sAl[tid] = al;
        sBe[tid] = be;
    }
    asm volatile("cp.async.wait_group 1;" ::: "memory");     // keys and queries; the value rows may still be in flight
    if (__syncthreads_or(fault)) {
        if (reporter) atomicOr(p.status, SPECA_STATUS_BAD_PARENT);
        return;
    }

    // ---- topology: the path of node tid, upward (path[0] is the node itself)
    int path[MAXD], d = 0;
    if (tid < n) {
        int a = tid;
#pragma unroll
        for (int r = 0; r < MAXD; ++r) {
            path[r] = a >= 0 ? a : 0;
            if (a >= 0) { ++d; a = sPar[a]; }
        }
        int full = d;
        for (; a >= 0; a = sPar[a]) ++full;
        if (full > p.max_depth) fault |= SPECA_STATUS_TOO_DEEP;
        if (p.depth_in != nullptr && p.depth_in[base + tid] != full) fault |= SPECA_STATUS_BAD_DEPTH;
        if (fault && l == 0 && h == 0 && part == 0) atomicOr(p.status, fault);
    }

    // ---- Gram rows of keys and queries against the keys
    for (int job = WARPS - 1 - warp; job < nt * (nt + 1) / 2; job += WARPS) {      // (warp 0 walks the paths meanwhile)
        // one MMA row block: keys 8 mi .. in rows 0-7, queries 8 mi .. in rows 8-15; a node's path holds no later node, so
        // ni <= mi: the triangle row by row
        int mi = 0;
#pragma unroll
        for (int m = 1; m < NT; ++m) mi += job >= m * (m + 1) / 2;
        const int ni = job - mi * (mi + 1) / 2;
        float acc[4] = {0.f, 0.f, 0.f, 0.f}, acc1[4] = {0.f, 0.f, 0.f, 0.f};
        const __nv_bfloat16 *pa = sKQ + ((lane & 8 ? N : 0) + 8 * mi + (lane & 7)) * LY::KQS + ((lane >> 4) << 3);
        const __nv_bfloat16 *pb = sKQ + (8 * ni + (lane & 7)) * LY::KQS + ((lane >> 3) << 3);
#pragma unroll
        for (int k = 0; k < DK / 32; ++k) {
            uint32_t bq[4], a0[4], a1[4];
            ldsm_x4(bq, pb + 32 * k);
            ldsm_x4(a0, pa + 32 * k);
            ldsm_x4(a1, pa + 32 * k + 16);
            float part0[4], part1[4];
            warp_mma_bf16_first(part0, a0, bq[0], bq[1]);
            warp_mma_bf16_first(part1, a1, bq[2], bq[3]);
#pragma unroll
            for (int e = 0; e < 4; ++e) { acc[e] += part0[e]; acc1[e] += part1[e]; }
        }
        float *gk = sG + (8 * mi + g) * LY::GS + 8 * ni + 2 * t4, *gq = gk + N * LY::GS;
        gk[0] = acc[0] + acc1[0]; gk[1] = acc[1] + acc1[1];
        gq[0] = acc[2] + acc1[2]; gq[1] = acc[3] + acc1[3];
    }
    if (__syncthreads_or(fault)) return;                     // reported above

    // ---- coefficients of node tid: back substitution up its path
    float acc[MAXD];
    if (tid < n) {
        const float *gq = sG + (N + tid) * LY::GS;
#pragma unroll
        for (int r = 0; r < MAXD; ++r) acc[r] = r < d ? gq[path[r]] : 0.f;
#pragma unroll
        for (int r = 0; r < MAXD; ++r) {
            const float cb = acc[r] * sBe[path[r]];
            if (!p.no_erase) {
                const float *gk = sG + path[r] * LY::GS;
#pragma unroll
                for (int s = r + 1; s < MAXD; ++s)
                    if (r < MAXD - 1) acc[s] = s < d ? fmaf(-cb, gk[path[s]], acc[s]) : 0.f;
            }
            acc[r] = cb;
        }
    }
    if (LY::kOver) __syncthreads();
    if (tid < n) {
        float rho = p.scale;
        float *cb = sC + tid * MAXD, *ro = cb + N * MAXD;
#pragma unroll
        for (int r = 0; r < MAXD; ++r) {
            cb[r] = acc[r];
            ro[r] = rho;
            sPath[tid * MAXD + r] = uint8_t(r < d ? path[r] : 0xff);
            rho *= r < d ? sAl[path[r]] : 1.f;
        }
        sGam[tid] = rho;                                     // scale gamma
    }
    __syncthreads();
    // the weights of value rows (M) and keys (W) in three bf16 pieces: every thread of the CTA takes its share, one node
    // and step up the path at a time (left to the thread of each node this was two thirds of the phase)
    for (int i = tid; i < n * MAXD; i += THREADS) {
        const int a = sPath[i];
        if (a == 0xff) continue;
        const int node = i / MAXD;
        const float cb = sC[i];
        float m = sC[N * MAXD + i] * cb, w = p.no_erase ? 0.f : -sGam[node] * cb;
        __nv_bfloat16 *md = sM + node * LY::MS + a, *wd = sW + LY::w_row(node) + a;
#pragma unroll
        for (int pc = 0; pc < 3; ++pc) {
            const __nv_bfloat16 mq = __float2bfloat16_rn(m), wq = __float2bfloat16_rn(w);
            md[pc * N * LY::MS] = mq;
            wd[pc * LY::WP] = wq;
            m -= __bfloat162float(mq);
            w -= __bfloat162float(wq);
        }
    }
    __syncthreads();

    for (int pass = 0;; ++pass) {                            // (the second one only after a repair)
        // the first two steps of this warp's first tile, requested a phase ahead of their use
        const float *Su = S_cta + g * DK + 8 * t4;
        float sa[2][8], sb[2][8];
        if (warp / PARTS < tiles)
#pragma unroll
            for (int q = 0; q < 2; ++q) {
                ld_state(sa[q], Su + warp / PARTS * 16 * DK + 32 * q);
                ld_state(sb[q], Su + (warp / PARTS * 16 + 8) * DK + 32 * q);
            }

        // ---- effective queries (scale gamma q + W K, the weights in three bf16 pieces), split into head and remainder
        {
            constexpr int CW = LY::kHalf ? 32 : 16, CB = CW / 8;     // columns of a job, in blocks of 8
            const int nm = (n + 15) >> 4;
            for (int job = warp; job < nm * (DK / CW); job += WARPS) {
                const int mi = job / (DK / CW), c0 = (job % (DK / CW)) * CW;
                const int r0 = 16 * mi + g, r1 = r0 + 8;
                const float g0 = sGam[r0], g1 = sGam[r1];
                float acc[CB][4];
#pragma unroll
                for (int c = 0; c < CB; ++c) {
                    // rows past the staged ones weigh nothing; clamp keeps the read inside the buffer
                    const __nv_bfloat16 *pq = sKQ + N * LY::KQS + c0 + 8 * c + 2 * t4;
                    const uint32_t q0 = *reinterpret_cast<const uint32_t *>(pq + min(r0, N - 1) * LY::KQS);
                    const uint32_t q1 = *reinterpret_cast<const uint32_t *>(pq + min(r1, N - 1) * LY::KQS);
                    acc[c][0] = g0 * __uint_as_float(q0 << 16); acc[c][1] = g0 * __uint_as_float(q0 & 0xffff0000u);
                    acc[c][2] = r1 < 8 * nt ? g1 * __uint_as_float(q1 << 16) : 0.f;
                    acc[c][3] = r1 < 8 * nt ? g1 * __uint_as_float(q1 & 0xffff0000u) : 0.f;
                }
                for (int kk = 0; kk <= mi; ++kk) {               // a node's path holds no later node
                    uint32_t kb[CB / 2][4];                      // key rows 16 kk .. + 15, columns c0 .. + CW - 1
                    const int kr = 16 * kk + (lane & 15);
#pragma unroll
                    for (int c = 0; c < CB / 2; ++c)
                        ldsm_x4_t(kb[c], sKQ + min(kr, 8 * nt - 1) * LY::KQS + c0 + 16 * c + ((lane >> 4) << 3));
                    float lo[CB][4], hi[CB][4];
#pragma unroll
                    for (int pc = 2; pc >= 0; --pc) {
                        uint32_t a[4];
                        ldsm_x4(a, sW + pc * LY::WP + LY::w_row(16 * mi + (lane & 15)) + 16 * kk + ((lane >> 4) << 3));
#pragma unroll
                        for (int c = 0; c < CB; ++c) {
                            const uint32_t b0 = kb[c >> 1][2 * (c & 1)], b1 = kb[c >> 1][2 * (c & 1) + 1];
                            if (pc == 2) warp_mma_bf16_first(lo[c], a, b0, b1);
                            else if (pc == 1) warp_mma_bf16(lo[c], a, b0, b1);
                            else warp_mma_bf16_first(hi[c], a, b0, b1);
                        }
                    }
#pragma unroll
                    for (int c = 0; c < CB; ++c)
#pragma unroll
                        for (int e = 0; e < 4; ++e) acc[c][e] += hi[c][e] + lo[c][e];
                }
#pragma unroll
                for (int half = 0; half < 2; ++half) {
                    const int r = half ? r1 : r0;
                    if constexpr (LY::kHalf) {
                        float x[8];
#pragma unroll
                        for (int c = 0; c < 4; ++c) { x[2 * c] = acc[c][2 * half]; x[2 * c + 1] = acc[c][2 * half + 1]; }
                        const float top = row_max(x);
                        const HalfScale scale(top);
                        uint32_t *ph = reinterpret_cast<uint32_t *>(hHi + r * LY::BSH + c0 + 2 * t4);
                        uint32_t *pl = reinterpret_cast<uint32_t *>(hLo + r * LY::BSH + c0 + 2 * t4);
                        if (r < 8 * nt) {
#pragma unroll
                            for (int c = 0; c < 4; ++c) half_split(x[2 * c], x[2 * c + 1], scale.up, ph[4 * c], pl[4 * c]);
                            if (t4 == 0) sSc[(c0 >> 5) * N + r] = scale.size * kUndoQuery;
                        }
                        // Where no value is less than 2^-23 of the largest of its 32, the column in which a row of the state has
                        // its largest brings at least 2^-23 a_max b_max, and the 2^-51 a_max that its smallest values may lose
                        // are no more than 2^-23 of what the products come to.  Else the state is looked at below.
                        if (__any_sync(0xffffffffu, least_of(x) < top * 0x1p-23f || top > kMostHalf)) {
                            const uint32_t raw = __ballot_sync(0xffffffffu, scale.loses(x) || top > kMostHalf);
                            if (lane == 0) atomicOr(sUneven, (raw ? 257 : 1) << (c0 >> 5));
                            // what does not fit fp16 pairs stays as it is, in halves, under a scale of zero
                            if (r < 8 * nt && (raw >> (lane & 28) & 15u) != 0u) {
#pragma unroll
                                for (int c = 0; c < 4; ++c) {
                                    const uint32_t x0 = __float_as_uint(x[2 * c]), x1 = __float_as_uint(x[2 * c + 1]);
                                    ph[4 * c] = __byte_perm(x0, x1, 0x7632);
                                    pl[4 * c] = __byte_perm(x0, x1, 0x5410);
                                }
                                if (t4 == 0) sSc[(c0 >> 5) * N + r] = 0.f;
                            }
                        }
                        continue;
                    }
                    if (r >= 8 * nt) break;
#pragma unroll
                    for (int c = 0; c < 2; ++c) {
                        const float x0 = acc[c][2 * half], x1 = acc[c][2 * half + 1];
                        const float y0 = tc::round_tf32(x0), y1 = tc::round_tf32(x1);
                        *reinterpret_cast<float2 *>(sHi + r * LY::BS + c0 + 8 * c + 2 * t4) = make_float2(y0, y1);
                        *reinterpret_cast<float2 *>(sLo + r * LY::BS + c0 + 8 * c + 2 * t4) = make_float2(x0 - y0, x1 - y1);
                    }
                }
            }
        }
        asm volatile("cp.async.wait_group 0;" ::: "memory");     // value rows
        __syncthreads();

        // ---- the state: one 16-row tile at a time, two 32-column steps of registers in flight
        // lane (g, t) holds columns 32 q + 8 t .. + 7 of rows g and g + 8: k-steps e = 0..3 of the step contract
        // columns 8 t + 2 e and 8 t + 2 e + 1 of the four lanes
        const int half = PARTS == 1 ? 0 : warp % PARTS, i0 = half * NTP;         // this warp's column tiles: i0 ..
        const float *hi_p = sHi + (8 * i0 + g) * LY::BS + 8 * t4, *lo_p = sLo + (8 * i0 + g) * LY::BS + 8 * t4;
        const uint16_t *hh_p = hHi + (8 * i0 + g) * LY::BSH + 8 * t4, *hl_p = hLo + (8 * i0 + g) * LY::BSH + 8 * t4;
        const int nk = (n + 15) >> 4, ntp = nt - i0;
        const int tile_end = PARTS > 1 && ntp <= 0 ? 0 : tiles;
        float *o0 = p.o + rec0 * p.DV + row0 + g;
        const long node_stride = long(H) * p.DV;
        float zero = 0.f;                                        // the sum of the outputs times zero
#pragma unroll 1
        for (int tile = warp / PARTS; tile < tile_end; tile += STRIDE) {
            if (lane == 0 && half == 0 && tile + AHEAD < tiles) prefetch_l2(S_cta + long(tile + AHEAD) * 16 * DK, 16 * DK * 4);
            const bool next = tile + STRIDE < tiles;
            float hh[NTP][4], xx[NTP][4];                         // head x head, and the two cross products
#pragma unroll
            for (int i = 0; i < NTP; ++i)
#pragma unroll
                for (int e = 0; e < 4; ++e) { hh[i][e] = 0.f; xx[i][e] = 0.f; }
            const float *cur = Su + long(tile) * 16 * DK, *nxt = cur + STRIDE * 16 * DK - NS * 32;
#pragma unroll
            for (int q = 0; q < NS; ++q) {
                if constexpr (LY::kHalf) {
                    // k-steps j = 0, 1 of 16 contract columns 8 t + 4 j .. + 3 of the four lanes
                    uint32_t ah[2][4], al[2][4];
                    const HalfScale scale_a(row_max(sa[q & 1])), scale_b(row_max(sb[q & 1]));
#pragma unroll
                    for (int j = 0; j < 2; ++j)
#pragma unroll
                        for (int c = 0; c < 2; ++c) {
                            const int e = 4 * j + 2 * c;
                            half_split(sa[q & 1][e], sa[q & 1][e + 1], scale_a.up, ah[j][2 * c], al[j][2 * c]);
                            half_split(sb[q & 1][e], sb[q & 1][e + 1], scale_b.up, ah[j][2 * c + 1], al[j][2 * c + 1]);
                        }
                    if (q + 2 < NS || next) {
                        const float *src = (q + 2 < NS ? cur : nxt) + 32 * (q + 2);
                        ld_state(sa[q & 1], src);
                        ld_state(sb[q & 1], src + 8 * DK);
                    }
#pragma unroll
                    for (int i = 0; i < NTP; ++i) {
                        if (NTP > 1 && i >= ntp) break;
                        const uint4 bh = *reinterpret_cast<const uint4 *>(hh_p + 8 * i * LY::BSH + 32 * q);
                        const uint4 bl = *reinterpret_cast<const uint4 *>(hl_p + 8 * i * LY::BSH + 32 * q);
                        const float2 sc = *reinterpret_cast<const float2 *>(sSc + q * N + 8 * (i0 + i) + 2 * t4);
                        float low[4], part[4];
                        warp_mma_f16<true>(low, al[0], bh.x, bh.y);
                        warp_mma_f16<true>(part, ah[0], bh.x, bh.y);
                        warp_mma_f16<false>(low, al[1], bh.z, bh.w);
                        warp_mma_f16<false>(part, ah[1], bh.z, bh.w);
                        warp_mma_f16<false>(low, ah[0], bl.x, bl.y);
                        warp_mma_f16<false>(low, ah[1], bl.z, bl.w);
#pragma unroll
                        for (int e = 0; e < 4; e += 2) {
                            const float down = (e < 2 ? scale_a.size : scale_b.size) * kUndoState;
                            float2 x = __ffma2_rn(make_float2(low[e], low[e + 1]), make_float2(kLowPiece, kLowPiece),
                                                  make_float2(part[e], part[e + 1]));
                            x = __ffma2_rn(__fmul2_rn(x, make_float2(down, down)), sc, make_float2(hh[i][e], hh[i][e + 1]));
                            hh[i][e] = x.x;
                            hh[i][e + 1] = x.y;
                        }
                    }
                    continue;
                }
                uint32_t ah[4][4], al[4][4];                     // [k-step][fragment register]
#pragma unroll
                for (int e = 0; e < 4; ++e) {
                    const float x[4] = {sa[q & 1][2 * e], sb[q & 1][2 * e], sa[q & 1][2 * e + 1], sb[q & 1][2 * e + 1]};
#pragma unroll
                    for (int c = 0; c < 4; ++c) { ah[e][c] = tf32_head(x[c]); al[e][c] = tf32_tail(x[c]); }
                }
                if (q + 2 < NS || next) {
                    const float *src = (q + 2 < NS ? cur : nxt) + 32 * (q + 2);
                    ld_state(sa[q & 1], src);
                    ld_state(sb[q & 1], src + 8 * DK);
                }
#pragma unroll
                for (int i = 0; i < NTP; ++i) {
                    if (NTP > 1 && i >= ntp) break;
                    float part[4] = {0.f, 0.f, 0.f, 0.f};    // of this step
#pragma unroll
                    for (int e2 = 0; e2 < 2; ++e2) {
                        const float4 bh = *reinterpret_cast<const float4 *>(hi_p + 8 * i * LY::BS + 32 * q + 4 * e2);
                        const float4 bl = *reinterpret_cast<const float4 *>(lo_p + 8 * i * LY::BS + 32 * q + 4 * e2);
                        warp_mma_tf32(part, ah[2 * e2], __float_as_uint(bh.x), __float_as_uint(bh.y));
                        warp_mma_tf32(xx[i], ah[2 * e2], __float_as_uint(bl.x), __float_as_uint(bl.y));
                        warp_mma_tf32(part, ah[2 * e2 + 1], __float_as_uint(bh.z), __float_as_uint(bh.w));
                        warp_mma_tf32(xx[i], al[2 * e2], __float_as_uint(bh.x), __float_as_uint(bh.y));
                        warp_mma_tf32(xx[i], ah[2 * e2 + 1], __float_as_uint(bl.z), __float_as_uint(bl.w));
                        warp_mma_tf32(xx[i], al[2 * e2 + 1], __float_as_uint(bh.z), __float_as_uint(bh.w));
                    }
#pragma unroll
                    for (int e = 0; e < 4; ++e) hh[i][e] += part[e];
                }
            }
            // value term: rows of V^T (16 value rows x 16 nodes) x M, piece by piece
            {
                const __nv_bfloat16 *va = sV + ((lane & 7) + ((lane >> 4) << 3)) * vstride + tile * 16 + (lane & 8);
#pragma unroll
                for (int kk = 0; kk < LY::NK / 16; ++kk) {
                    if (LY::NK > 16 && kk >= nk) break;
                    uint32_t a[4];
                    ldsm_x4_t(a, va + kk * 16 * vstride);
#pragma unroll
                    for (int i = 0; i < NTP; ++i) {
                        if (NTP > 1 && i >= ntp) break;
                        if (8 * (i0 + i) + 7 < 16 * kk) continue;       // a node's path holds no later node
                        float lo[4], hi[4];
#pragma unroll
                        for (int pc = 2; pc >= 0; --pc) {
                            const __nv_bfloat16 *mb = sM + (pc * N + 8 * (i0 + i) + g) * LY::MS + 16 * kk + 2 * t4;
                            const uint32_t b0 = *reinterpret_cast<const uint32_t *>(mb);
                            const uint32_t b1 = *reinterpret_cast<const uint32_t *>(mb + 8);
                            if (pc == 2) warp_mma_bf16_first(lo, a, b0, b1);
                            else if (pc == 1) warp_mma_bf16(lo, a, b0, b1);
                            else warp_mma_bf16_first(hi, a, b0, b1);
                        }
#pragma unroll
                        for (int e = 0; e < 4; ++e) { hh[i][e] += hi[e]; xx[i][e] += lo[e]; }
                    }
                }
            }
            float *ot = o0 + tile * 16;
#pragma unroll
            for (int i = 0; i < NTP; ++i) {
                if (NTP > 1 && i >= ntp) break;
                const int n0 = 8 * (i0 + i) + 2 * t4;
                float *od = ot + n0 * node_stride;
#pragma unroll
                for (int e = 0; e < 4; ++e) {
                    hh[i][e] += xx[i][e];
                    zero = fmaf(hh[i][e], 0.f, zero);
                }
                if (n0 < n) { od[0] = hh[i][0]; od[8] = hh[i][2]; }
                if (n0 + 1 < n) { od[node_stride] = hh[i][1]; od[node_stride + 8] = hh[i][3]; }
            }
        }
        // Where the effective queries are uneven, the tiles that do not fit fp16 pairs, or all of them if the queries do not, are
        // done once more.  (Looking for such tiles in the loop above cost 2 to 10 % of a call, doing them there up to 20 %.)
        if constexpr (LY::kHalf) {
            const int uneven = *sUneven;                         // (bits 8 ..: steps with queries that do not fit)
#pragma unroll 1
            for (int tile = warp / PARTS; uneven != 0 && tile < tile_end; tile += STRIDE) {
                const float *cur = Su + long(tile) * 16 * DK;
                if (uneven < 256 && !loses_bits<DK>(cur, uneven)) continue;
                float x[NTP][4];
                state_in_tf32<LY, NTP>(x, cur, hh_p, hl_p, sSc + 8 * i0 + g, ntp);
                // the value term in plain fp32, node by node up the path
#pragma unroll
                for (int i = 0; i < NTP; ++i)
#pragma unroll
                    for (int e = 0; e < 4; ++e) {
                        const int node = 8 * (i0 + i) + 2 * t4 + (e & 1), r = 16 * tile + (e & 2) * 4;
                        if (node >= n) continue;
                        for (int a = node; a >= 0; a = sPar[a]) {
                            const __nv_bfloat16 *m = sM + node * LY::MS + a;
                            const float low = __bfloat162float(m[N * LY::MS]) + __bfloat162float(m[2 * N * LY::MS]);
                            x[i][e] = fmaf(__bfloat162float(m[0]) + low, __bfloat162float(sV[a * vstride + r + g]), x[i][e]);
                        }
                        zero = fmaf(x[i][e], 0.f, zero);
                        o0[node * node_stride + r] = x[i][e];
                    }
            }
        }
        const bool odd = __syncthreads_or(!(zero == 0.f));
        if (!(odd || pass > 0) || !repair<DK, NT, MAXD, THREADS>(da, smem, pass)) break;
    }
}

// A batch that fills the device's resident CTAs only once or twice is latency, not throughput.
bool small_batch(const Params &p, int sms) { return long(p.L) * p.B * p.H <= 4L * sms; }

template <int DK, int NT, int MAXD, int WARPS, int CTAS>
int launch_one(const Params &p, int lo, bool all, int sms, cudaStream_t st)
{
    using LY = Lay<DK, NT, MAXD>;
    DirectArgs da;
    da.p = p;
    da.lo = lo;
    // Asking for the state before anything else is known keeps HBM busy in a large batch (12288 units of 8 nodes, d_k = 128,
    // d_v = 256: 301 us, after the records 320).  Where all CTAs start at once, or a tile is small, the records then
    // queue behind the state, and the set-up waits for them (384 chains of 8: 11.8 us, after the records 10.4; 4608
    // units of 32 nodes at d_k = d_v = 64: 67.8 / 65.8).
    da.early = all && DK > 64 && !small_batch(p, sms);
    // Value rows per CTA: the whole unit, halved as long as all halves start at once: a second wave of set-ups costs more
    // than the idle slots (us, whole / halved: 384 units at d_k = d_v = 128 of 16 nodes 20.5 / 22.5, 12 nodes 18.4 / 22.5; d_v
    // = 256, 8 nodes 20.5 / 24.6; 384 units at d_k = 256 of 8 nodes 36.9 / 41.0).  Only where a warp has two 16 KB
    // tiles left is the halving worth the second wave (192 units at d_k = 256 of 8 nodes 24.6 / 22.5).
    const long units = long(p.L) * p.B * p.H, slots = long(sms) * CTAS;
    int rows = p.DV;
    while (rows > 256 && rows % 32 == 0) rows /= 2;
    while (rows % 32 == 0 && rows / 16 > WARPS) {
        const long ctas = units * (p.DV / rows);
        if (ctas * 2 > slots && !(DK == 256 && rows <= 32 * WARPS && ctas < slots)) break;
        rows /= 2;
    }
    da.rows = rows;
    const int parts = p.DV / rows;
    da.parts = Divisor(parts);
    da.H = Divisor(p.H);
    da.B = Divisor(p.B);
    da.vp = Divisor(rows >> 3);
    const int smem = LY::bytes(rows);
    static std::atomic<int> opted[64];
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return int(cudaErrorInvalidDevice);
    auto kern = verify_direct_kernel<DK, NT, MAXD, WARPS, CTAS>;
    if (smem > 48 * 1024 && opted[dev].load(std::memory_order_acquire) == 0) {
        const cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, LY::bytes(512));
        if (e != cudaSuccess) return int(e);
        opted[dev].store(1, std::memory_order_release);
    }
    launch(kern, unsigned(units * parts), WARPS * 32, smem, st, da);
    return int(cudaGetLastError());
}

// Warps per CTA and CTAs per SM by the width NT of the product: registers (two 32-column steps of state, the
// accumulators) allow 80 / 96 / 128 per thread, shared memory two CTAs at 32 nodes, where eight warps share the longer
// set-up.
template <int DK, int MAXD>
int launch_width(const Params &p, int hi, int lo, bool all, int sms, cudaStream_t st)
{
    constexpr int C1 = DK == 128 && MAXD == 8 ? 6 : 5, C2 = DK == 64 || MAXD == 8 ? 5 : 4;
    if (hi <= 8) return launch_one<DK, 1, MAXD, 4, C1>(p, lo, all, sms, st);
    if (hi <= 16) return launch_one<DK, 2, MAXD, 4, C2>(p, lo, all, sms, st);
    if constexpr (DK == 64) {
        if (hi <= 32) return launch_one<DK, 4, MAXD, 4, 4>(p, lo, all, sms, st);
        return launch_one<DK, 8, MAXD, 8, 2>(p, lo, all, sms, st);
    } else {
        // between two and three units per SM one wave of smaller CTAs beats two of the others (d_k = d_v = 128, 32 nodes: 384
        // units 24.6 us, with eight warps 26.6; 432 units the same; 576 units take two waves either way; d_v = 256, 384 units
        // of 24 / 32 nodes 22.1 / 25.6, with eight warps 25.1 / 29.0)
        const long units = long(p.L) * p.B * p.H;
        if constexpr (DK == 128)
            if (p.DV <= 256 && units > 2 * sms && units <= 3 * sms) return launch_one<DK, 4, MAXD, 4, 3>(p, lo, all, sms, st);
        return launch_one<DK, 4, MAXD, 8, 2>(p, lo, all, sms, st);
    }
}

}  // namespace

// Largest sequence this kernel should verify (0: none).  `most` bounds the nodes of any sequence of the call, `piped`
// says that one of the pipelined tensor-core kernels takes the shape.
int direct_limit(const Params &p, int d_k, int most, bool piped, bool chain)
{
    if (!piped) {
        // The alternative is the serial walk, whose time grows with the nodes where this kernel's hardly does.  A chain needs
        // no plan there, so short ones stay with it; how short, by the elements of a unit and of the call.  us, serial / this
        // one: 64 x 64, 16 units of 4 / 5 / 8 nodes 3.8 / 4.0, 4.3 / 4.1, 5.8 / 4.0, 12288 units of 2 / 3 / 4 nodes 56 / 71,
        // 72 / 71, 90 / 71; 64 x 32, 12288 units of 4 / 6 nodes 48 / 64, 65 / 65; 128 x 64, 12288 units of 1 / 2 nodes 72 / 92,
        // 106 / 93, 192 units of 3 / 4 nodes 5.3 / 5.5, 6.3 / 5.5; 64 x 512, 1536 units of 1 / 2 nodes 37 / 42, 54 / 42.  Trees
        // (with their plan): 64 x 32, 1536 units of 2 / 3 / 4 nodes 9.9 / 11.5, 11.9 / 11.5, 12.8 / 11.4; 128 x 512, 1536 units
        // of 1 / 2 nodes 73 / 77, 108 / 78, 16 units of 1 node 5.6 / 5.1.
        const long unit = long(p.DV) * d_k, call = unit * p.L * p.B * p.H;
        const int small_unit = int((d_k == 128 || !chain ? 8191 : 8192) / unit);
        const int few = chain ? std::min(1 + small_unit + (call < 8L << 20) + (call <= 1L << 20), 5)
                              : call >= 2L << 20 ? std::max(small_unit, 1) : 0;
        // many chains take the time of the mean one, a few that of the longest
        if (chain && call >= 2L << 20 ? p.T <= long(few) * p.B : most <= few) return 0;
        // In a small call the walk of the largest tree is the whole time: where the mean says that there is one left for it, the
        // others may as well go along (18 units at 64 x 512, trees of up to 70 nodes 58 us, after a launch of this kernel 70).
        const int limit = d_k == 64 ? 64 : 32;
        return p.T > long(limit) * p.B && small_batch(p, sm_count_of_current_device()) ? 0 : limit;
    }
    // us per unit and SM in a large batch, this kernel / the pipelined one with its plan: d_k = 128, d_v = 256: 3.6 / 3.6 at 8
    // nodes, 4.1 / 4.0 at 12, 4.5 / 3.9 to 4.3 at 16, 5.6 / 4.3 at 20; d_v = 128: 2.0 / 3.3 at 8, 2.6 / 3.0 at 12 and 16, 3.9 /
    // 3.1 at 20; d_k = 256, 8 nodes 7.5 / 6.4.  A few users, us per call: d_k = d_v = 128, 384 units of 8 / 16 / 24 / 32 nodes
    // 10.1 / 14.0, 15.3 / 14.4, 13.3 / 15.3, 15.2 / 15.4; d_v = 256, 192 units 10.1 / 13.9, 15.4 / 14.3, 13.4 / 15.2, 16.1 /
    // 15.3, 384 units 14.1 / 16.8, 24.0 / 17.4, 20.0 / 19.1, 23.0 / 19.5; d_k = 256, 8 nodes, 192 units 16.3 / 16.0, 384 units
    // 27.6 / 24.2.  Up to the lines it is the faster kernel or the more accurate one: its error against 64 bits is half of the
    // other's or less (x 10^-8, 8..32 nodes at d_k = 128 7.3 to 7.9 against 14.5 to 16.4, 8 nodes at d_k = 256 7.9 against 22).
    const bool few = small_batch(p, sm_count_of_current_device());
    const int cap = d_k == 128 ? (few ? 32 : 16) : (few ? 8 : 0);
    return most <= cap ? cap : 0;
}

// Verifies every sequence of at most `limit` nodes; larger ones are left to another kernel.
int launch_verify_direct(const Params &p, int d_k, int most, int limit, cudaStream_t st)
{
    const int sms = sm_count_of_current_device();
    if (sms <= 0) return int(cudaErrorInvalidDevice);
    const bool deep = p.max_depth > 8;
    auto run = [&](int lo, int hi) {
        const bool all = lo == 0 && most <= hi;
        switch (d_k) {
        case 64: return deep ? launch_width<64, 16>(p, hi, lo, all, sms, st) : launch_width<64, 8>(p, hi, lo, all, sms, st);
        case 128: return deep ? launch_width<128, 16>(p, hi, lo, all, sms, st) : launch_width<128, 8>(p, hi, lo, all, sms, st);
        case 256: return deep ? launch_width<256, 16>(p, hi, lo, all, sms, st) : launch_width<256, 8>(p, hi, lo, all, sms, st);
        }
        return int(cudaErrorInvalidValue);
    };
    const int top = most < limit ? most : limit;
    if (top <= 32 || small_batch(p, sms)) return run(0, top);
    const int rc = run(0, 32);
    return rc != 0 ? rc : run(32, top);
}

}  // namespace speca

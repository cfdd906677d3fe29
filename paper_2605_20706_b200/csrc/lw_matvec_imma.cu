// Batch-1 mat-vecs of the widths that the streaming kernels do not take: rows that are no multiple of 16 bytes (q6_K
// and q2_K at most widths), widths that are no multiple of 256 columns [paper Sec 3.2: the decode-phase mat-vec; Sec 3.3:
// one decode routine per block format spliced into a common skeleton, weights decoded straight into registers].
//
// What bounds it: instructions (217 warp instructions per 2048 weights of q4_0 at 88000 x 2848, prologue included, 377 of
// q6_K at 64000 x 3072, at 57-59 % of the issue slots; HBM at a third), and on small matrices 3.5 us until the first tile's
// products.  Against the generic kernel, which decodes from global memory in 2- and 4-byte loads: q6_K 32000 x 3072 63 ->
// 31 us, q4_0 11007 x 2848 20.5 -> 9.5 (matvec_imma_supported has the line between the two).
//
// Arithmetic.  The activations of a block of 32 (16 where the format's scales are per 16) become fixed point relative
// to the block's largest M: v = rint(x / d), |v| < 2^31, d a power of two, so that every element down to 2^-6 M is
// represented exactly and one of 2^-17 M to 2^-14 of itself.  What does not fit -- smaller elements beside a large one,
// magnitudes of 2^96 and more, Inf and NaN -- counts as zero there and is multiplied in fp32 with its exactly decoded
// weight: every element keeps a relative accuracy of its own, whatever stands beside it.  One element in 80 000 of normally
// distributed activations is kept apart like this.  v is written as four signed digits of base 256.  mma.m16n8k32 (s8 x u8 /
// s8 -> s32) multiplies A (16 x 32) = digits of the activations with B (32 x 8) = the codes of one block of 8 weight rows:
//   A row m = g     : digit (g & 1)     of block s = g / 2 of the chain of four blocks,  g = 0..7
//   A row m = g + 8 : digit 2 + (g & 1) of the same block
// and zero in the rows of the other three blocks, so that four products accumulate into ONE set of accumulators
// without mixing their blocks.  A lane then holds, for two rows, two digits of one block: it converts the exact integer
// sums to fp32, multiplies them with d * 256^digit and with the block's weight scale, and adds them up.  An offset of
// the code (q4_0's 8, q6_K's 32) is an integer too and goes into the accumulators' initial value, exactly.  Where a block has
// an offset of its own (q4_1, q5_1, q2_K), scale * sum of code * digit and offset * sum of digits nearly cancel when a large
// activation meets a weight next to zero: they are added per digit, with one rounding.
//
// Work and data.  One CTA per SM: 16 compute warps and one copy warp.  The rows are cut evenly over the CTAs.  The copy warp
// brings tiles of rows into a ring of slots, one 1-D bulk copy per row, from the 16-byte boundary below the row to the one
// above it where rows are off that grid (tiled bulk copies need row lengths that are multiples of 16).  Rows lie an odd
// multiple of 16 bytes apart in a slot, so the eight rows a warp reads at once fall into different banks.
// A compute warp owns one 256-column piece of the row (its A operands stay in registers, 32 of them) and walks the
// tile's groups of eight rows; its row sums go to a table in shared memory that is folded once per 128 rows.
//
// Every wait is bounded: a wait that gives up records a fault, nothing is waited for after that (arrivals continue), and
// the kernel runs to its end.
#include <cuda_fp16.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <cstdint>
#include <type_traits>

#include "lw_internal.h"
#include "lw_stream_common.cuh"

namespace lw {
namespace {

constexpr int kComputeWarps = 16;
constexpr int kComputeThreads = 32 * kComputeWarps;
constexpr int kImmaThreads = kComputeThreads + 128;   // the copy warp belongs to a warpgroup of its own (setmaxnreg)
// Registers per thread: 640 threads are launched with 96 each; the copy warpgroup gives most of its share away.
constexpr int kComputeRegs = 112, kCopyRegs = 32;
static_assert(kComputeThreads * kComputeRegs + 128 * kCopyRegs <= kImmaThreads * 96, "register shares exceed the launch's total");
constexpr int kSlotsMax = 8;
constexpr int kFoldRows = 128;                    // rows whose sums are collected before they are folded
constexpr int kTableFloats = kFoldRows * kComputeWarps;
constexpr uint32_t kImmaHeader = 256;             // mbarriers, flags, zeros
constexpr uint32_t kZeros = 160;                  // 96 bytes of zeros
constexpr uint32_t kXBlock = 144;                 // bytes of a block of 32 activations: 4 digits x 32, scales
constexpr uint32_t kApartBits = kImmaHeader + 2 * kTableFloats * 4;  // activations kept apart: one bit per column
constexpr uint32_t kApartFrom = 0x6F800000u;      // 2^96: magnitudes from here on are kept apart
constexpr uint32_t kApartBelow = 17u << 23;       // and those below 2^-17 of their unit's largest
constexpr size_t kImmaSmemMax = 227 * 1024;

struct ImmaParams {
    const uint8_t* W;
    const float* X;
    float* Y;
    int* fault;
    int rows;
    int cols;
    int share;             // rows of a CTA; the first `extra` CTAs take one more
    int extra;
    uint32_t row_bytes;
    uint32_t pitch;        // bytes between rows of a tile in shared memory (an odd multiple of 16)
    uint32_t x_off, ring_off, slot_bytes;
    int slots;
    int tile_rows;         // rows of a ring slot
    int fold_rows;         // rows between folds, a multiple of tile_rows
    int chunk_sb;          // 256-column pieces of a row that are worked on at a time (<= 16, one per compute warp)
    int n_chunks;
    int row_groups;        // groups of compute warps that take different rows of a tile
    int drop_tile;         // DROP builds only
    bool ragged;           // pieces do not start on 16-byte boundaries: every row's copy starts at the boundary below
};

// ------------------------------------------------------------------ device helpers ---

__device__ __forceinline__ void compute_bar() { asm volatile("bar.sync 1, %0;" ::"n"(kComputeThreads) : "memory"); }
// the same, and whether any thread came with `v`
__device__ __forceinline__ bool compute_bar_any(bool v) {
    uint32_t any;
    asm volatile(
        "{\n\t.reg .pred p, q;\n\tsetp.ne.u32 p, %1, 0;\n\tbar.red.or.pred q, 1, %2, p;\n\tselp.u32 %0, 1, 0, q;\n\t}"
        : "=r"(any)
        : "r"((uint32_t)v), "n"(kComputeThreads)
        : "memory");
    return any != 0;
}

// 1-D bulk copy global -> shared, completion counted in bytes on `bar`; addresses and size are multiples of 16
__device__ __forceinline__ void bulk_row(uint32_t dst, const uint8_t* src, uint32_t bytes, uint32_t bar, uint64_t policy) {
    asm volatile(
        "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes.L2::cache_hint [%0], [%1], %2, [%3], %4;" ::"r"(dst),
        "l"(src), "r"(bytes), "r"(bar), "l"(policy)
        : "memory");
}
__device__ __forceinline__ void mbar_arrive_addr(uint32_t bar) {
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
}

__device__ __forceinline__ uint32_t sh32(uint32_t a) {
    uint32_t v;
    asm volatile("ld.shared.b32 %0, [%1];" : "=r"(v) : "r"(a));
    return v;
}
template <int OFF>
__device__ __forceinline__ uint32_t sh32o(uint32_t a) {
    uint32_t v;
    asm volatile("ld.shared.b32 %0, [%1+%2];" : "=r"(v) : "r"(a), "n"(OFF));
    return v;
}
template <int OFF>
__device__ __forceinline__ float sh_half(uint32_t a) {
    unsigned short h;
    asm volatile("ld.shared.u16 %0, [%1+%2];" : "=h"(h) : "r"(a), "n"(OFF));
    return __half2float(__ushort_as_half(h));
}
template <int OFF>
__device__ __forceinline__ int sh_s8(uint32_t a) {
    int v;
    asm volatile("ld.shared.s8 %0, [%1+%2];" : "=r"(v) : "r"(a), "n"(OFF));
    return v;
}
template <int OFF>
__device__ __forceinline__ uint32_t sh_u8(uint32_t a) {
    uint32_t v;
    asm volatile("ld.shared.u8 %0, [%1+%2];" : "=r"(v) : "r"(a), "n"(OFF));
    return v;
}
template <int OFF>
__device__ __forceinline__ uint32_t sh_u16(uint32_t a) {
    unsigned short v;
    asm volatile("ld.shared.u16 %0, [%1+%2];" : "=h"(v) : "r"(a), "n"(OFF));
    return v;
}
__device__ __forceinline__ uint4 sh128(uint32_t a) {
    uint4 v;
    asm volatile("ld.shared.v4.b32 {%0, %1, %2, %3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "r"(a));
    return v;
}

// Where a lane's row of codes starts: the word-aligned address at or below it, and byte selectors for words at offsets
// that are 0 resp. 2 modulo 4 (used where a row may start two bytes off the word grid).
struct RowAddr {
    uint32_t base, sel0, sel2;
};
__device__ __forceinline__ RowAddr row_addr(uint32_t a) {
    const bool odd = a & 2u;
    return RowAddr{a & ~3u, odd ? 0x5432u : 0x3210u, odd ? 0x7654u : 0x5432u};
}
// The 32-bit word at byte B + add of the row.  GEN: the row may be two bytes off the word grid; else it is on it.
template <int B, bool GEN>
__device__ __forceinline__ uint32_t code_word(const RowAddr& r, uint32_t lane_base) {
    constexpr int kDown = B & ~3;
    if constexpr (GEN) return __byte_perm(sh32o<kDown>(lane_base), sh32o<kDown + 4>(lane_base), (B & 2) ? r.sel2 : r.sel0);
    else if constexpr ((B & 2) != 0) return __byte_perm(sh32o<kDown>(lane_base), sh32o<kDown + 4>(lane_base), 0x5432u);
    else return sh32o<kDown>(lane_base);
}

template <bool SIGNED_B>
__device__ __forceinline__ void imma(int (&d)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1, const int* c) {
    if constexpr (SIGNED_B)
        asm("mma.sync.aligned.m16n8k32.row.col.s32.s8.s8.s32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%10,%11,%12,%13};"
            : "=r"(d[0]), "=r"(d[1]), "=r"(d[2]), "=r"(d[3])
            : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1), "r"(c[0]), "r"(c[1]), "r"(c[2]), "r"(c[3]));
    else
        asm("mma.sync.aligned.m16n8k32.row.col.s32.s8.u8.s32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%10,%11,%12,%13};"
            : "=r"(d[0]), "=r"(d[1]), "=r"(d[2]), "=r"(d[3])
            : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1), "r"(c[0]), "r"(c[1]), "r"(c[2]), "r"(c[3]));
}

__device__ __forceinline__ uint32_t spread_fifth(uint32_t x) { return ((x & 0xFu) * 0x02040810u) & 0x10101010u; }

// Fixed-point activations a compute warp keeps in registers for its 256 columns.  CH chains of four units (blocks of 32,
// or runs of 16); a lane (g, t) holds digits g & 1 and 2 + (g & 1) of unit g / 2 of every chain.
template <int CH>
struct XState {
    uint32_t a[8][4];          // A operands of the eight products
    float klo[CH], khi[CH];    // d * 256^digit of the lane's two digits (powers of two)
    float nlo[CH];             // -1.5 * 2^23 * klo
    int init[CH][4];           // initial accumulators: kIntMagic + code offset * sum of digits (digit lo twice, digit hi twice)
    float xlo[CH], xhi[CH];    // sums of the two digits (formats with an offset term)
};

// Integer sums (on top of kIntMagic: already the bit patterns of 1.5 * 2^23 + sum) of digits lo and hi of one unit and row
// -> the unit's sum of code * x.  The scales are powers of two, so the first product is exact.
__device__ __forceinline__ float unit_sum(int lo, int hi, float klo, float nlo, float khi) {
    return fmaf(__int_as_float(hi) - 12582912.f, khi, fmaf(__int_as_float(lo), klo, nlo));
}
// The same for a format with an offset term: the unit's sum of (d * code + m) * x onto acc.  Per digit d * S + m * X is
// rounded once (and the error of m * X, where it can have one, is added back), so that a weight of zero takes its activation
// out of the sum however large that is.  EXACT: m has 11 bits and X, a sum of 32 digits, 13.
template <bool EXACT>
__device__ __forceinline__ float affine_sum(int lo, int hi, float d, float m, float xlo, float xhi, float klo, float khi, float acc) {
    const float sl = __int_as_float(lo) - 12582912.f, sh = __int_as_float(hi) - 12582912.f;
    const float tl = __fmul_rn(m, xlo), th = __fmul_rn(m, xhi);
    float rl = fmaf(d, sl, tl), rh = fmaf(d, sh, th);
    if constexpr (!EXACT) rl = __fadd_rn(rl, fmaf(m, xlo, -tl)), rh = __fadd_rn(rh, fmaf(m, xhi, -th));
    return fmaf(rh, khi, fmaf(rl, klo, acc));
}
struct RowPair {
    float a, b;                // sums of rows 2 t and 2 t + 1
};
template <int NO>
struct RowSet {
    RowAddr r[NO];
    uint32_t s0[NO], s1[NO];
};

// A row sum into the table, on top of what is there when `more`; predicated, no branch.
__device__ __forceinline__ void put_sum(uint32_t at, float v, bool write, bool more) {
    asm volatile(
        "{\n\t.reg .pred w, m;\n\t.reg .f32 o;\n\tsetp.ne.u32 w, %2, 0;\n\tsetp.ne.and.u32 m, %3, 0, w;\n\tmov.f32 o, 0f00000000;\n\t"
        "@m ld.shared.f32 o, [%0];\n\tadd.f32 o, o, %1;\n\t@w st.shared.f32 [%0], o;\n\t}" ::"r"(at),
        "f"(v), "r"((uint32_t)write), "r"((uint32_t)more)
        : "memory");
}

template <int N, int I = 0, class F>
__device__ __forceinline__ void static_for(F f) {
    if constexpr (I < N) {
        f(std::integral_constant<int, I>{});
        static_for<N, I + 1>(f);
    }
}

// ------------------------------------------------------------------ format traits ---
//
//   kSuper            bytes of a row's 256 columns
//   kChains           chains of four units (units: blocks of 32, or runs of 16 where the scales are per 16)
//   kOffset           added to every code (exactly, through the initial accumulators)
//   kHasMin           a weight has an additive term: the unit's sum of activations times `min`
//   kMayStraddle      rows may start two bytes off the word grid
//   rows<GEN, NO>()   products of NO groups of eight rows with the warp's 256 columns: per group the sums of rows 2 t
//                     and 2 t + 1 over the lane's units.  r = the lane's row g with 4 t added; s0, s1 = addresses of rows
//                     2 t and 2 t + 1; nlive = live blocks of the piece (the last piece of a
//                     row may be short).  Two groups at a time give the scheduler independent work.

// q4_0, q4_1, q5_0, q5_1, q8_0: eight blocks of 32 with an fp16 scale (and offset) in front of the codes.
template <int FMT>
struct ImmaLegacy {
    static constexpr bool kFive = FMT == LW_Q5_0 || FMT == LW_Q5_1;
    static constexpr bool kHasMin = FMT == LW_Q4_1 || FMT == LW_Q5_1;
    static constexpr bool kEight = FMT == LW_Q8_0;
    static constexpr int kBlock = kEight ? 34 : 18 + (kHasMin ? 2 : 0) + (kFive ? 4 : 0);
    static constexpr int kSuper = 8 * kBlock;
    static constexpr int kChains = 2, kGroup = 32;
    static constexpr int kOffset = FMT == LW_Q4_0 ? -8 : FMT == LW_Q5_0 ? -16 : 0;
    static constexpr bool kMayStraddle = FMT == LW_Q4_0 || FMT == LW_Q5_0 || FMT == LW_Q8_0;
    static constexpr bool kF16 = false;

    // sum of weight * X[c] over the columns c of block k whose bits are set in `word`
    static __device__ __forceinline__ float sum_of(uint32_t row, int k, uint32_t word, const float* X) {
        const uint32_t b = row + (uint32_t)k * kBlock;
        const float d = sh_half<0>(b);
        float m = 0.f, sum = 0.f;
        uint32_t five = 0;
        if constexpr (kHasMin) m = sh_half<2>(b);
        if constexpr (kFive) five = sh_u16<2 + (kHasMin ? 2 : 0)>(b) | sh_u16<4 + (kHasMin ? 2 : 0)>(b) << 16;
#pragma unroll 2
        for (; word != 0; word &= word - 1) {
            const int c = __ffs((int)word) - 1;
            float w;
            if constexpr (kEight) {
                w = __fmul_rn((float)sh_s8<2>(b + c), d);
            } else {
                const uint32_t nib = sh_u8<2 + (kHasMin ? 2 : 0) + (kFive ? 4 : 0)>(b + (c & 15));
                const int q = (int)((nib >> (c >> 4 << 2) & 15u) | (five >> c & 1u) << 4);
                w = kHasMin ? __fadd_rn(__fmul_rn(d, (float)q), m) : __fmul_rn((float)(q + kOffset), d);
            }
            sum = fmaf(w, X[c], sum);
        }
        return sum;
    }

    template <bool GEN, int J>
    static __device__ __forceinline__ void codes(const RowAddr& r, int t, uint32_t& b0, uint32_t& b1) {
        constexpr int B = J * kBlock;
        if constexpr (kEight) {
            b0 = code_word<B + 2, GEN>(r, r.base);
            b1 = code_word<B + 18, GEN>(r, r.base);
        } else {
            const uint32_t q = code_word<B + 2 + (kHasMin ? 2 : 0) + (kFive ? 4 : 0), GEN>(r, r.base);
            b0 = q & 0x0F0F0F0Fu;
            b1 = (q >> 4) & 0x0F0F0F0Fu;
            if constexpr (kFive) {
                const uint32_t h = code_word<B + 2 + (kHasMin ? 2 : 0), GEN>(r, r.base - 4u * t) >> (4 * t);
                b0 |= spread_fifth(h);
                b1 |= spread_fifth(h >> 16);
            }
        }
    }
    template <bool GEN, int NO>
    static __device__ __forceinline__ void rows(const RowSet<NO>& R, const XState<2>& x, int g, int t, int nlive,
                                                RowPair (&acc)[NO]) {
        const int s = g >> 1;
#pragma unroll
        for (int o = 0; o < NO; ++o) acc[o].a = acc[o].b = 0.f;
        static_for<2>([&](auto chc) {
            constexpr int CH = decltype(chc)::value;
            int c[NO][4];
            static_for<4>([&](auto jc) {
                constexpr int J = decltype(jc)::value;
#pragma unroll
                for (int o = 0; o < NO; ++o) {
                    uint32_t b0, b1;
                    codes<GEN, 4 * CH + J>(R.r[o], t, b0, b1);
                    imma<kEight>(c[o], x.a[4 * CH + J], b0, b1, J == 0 ? x.init[CH] : c[o]);
                }
            });
            const bool live = s + 4 * CH < nlive;         // (what lies behind a row's last block may be anything)
#pragma unroll
            for (int o = 0; o < NO; ++o) {
                const uint32_t s0 = R.s0[o] + s * kBlock, s1 = R.s1[o] + s * kBlock;
                const float d0 = live ? sh_half<4 * CH * kBlock>(s0) : 0.f;
                const float d1 = live ? sh_half<4 * CH * kBlock>(s1) : 0.f;
                if constexpr (kHasMin) {
                    const float m0 = live ? sh_half<4 * CH * kBlock + 2>(s0) : 0.f;
                    const float m1 = live ? sh_half<4 * CH * kBlock + 2>(s1) : 0.f;
                    acc[o].a = affine_sum<true>(c[o][0], c[o][2], d0, m0, x.xlo[CH], x.xhi[CH], x.klo[CH], x.khi[CH], acc[o].a);
                    acc[o].b = affine_sum<true>(c[o][1], c[o][3], d1, m1, x.xlo[CH], x.xhi[CH], x.klo[CH], x.khi[CH], acc[o].b);
                } else {
                    acc[o].a = fmaf(d0, unit_sum(c[o][0], c[o][2], x.klo[CH], x.nlo[CH], x.khi[CH]), acc[o].a);
                    acc[o].b = fmaf(d1, unit_sum(c[o][1], c[o][3], x.klo[CH], x.nlo[CH], x.khi[CH]), acc[o].b);
                }
            }
        });
    }
};

// A small unsigned integer v (below 2^23) as the float 2^23 + v, without the conversion unit.
__device__ __forceinline__ float uint_float23(uint32_t v) { return __uint_as_float(v | 0x4B000000u); }

// q6_K: 128 bytes of low nibbles, 64 bytes of upper bit pairs, sixteen int8 scales, d.  Product 4 h + j takes group j of
// half h: its two k halves are runs 8 h + 2 j and + 1.
struct ImmaQ6K {
    static constexpr bool kHasMin = false;
    static constexpr int kSuper = 210, kChains = 4, kGroup = 16, kOffset = -32;
    static __device__ __forceinline__ float sum_of(uint32_t row, int k, uint32_t word, const float* X) {
        const int h = k >> 2, j = k & 3;
        const uint32_t ql = row + 64 * h + 32 * (j & 1), qh = row + 32 * h, sc = row + 8 * h + 2 * j;
        const float d = sh_half<208>(row), d0 = __fmul_rn(d, (float)sh_s8<192>(sc)), d1 = __fmul_rn(d, (float)sh_s8<193>(sc));
        float sum = 0.f;
#pragma unroll 2
        for (; word != 0; word &= word - 1) {
            const int l = __ffs((int)word) - 1;
            const uint32_t q = (sh_u8<0>(ql + l) >> (j & 2 ? 4 : 0) & 15u) | (sh_u8<128>(qh + l) >> (2 * j) & 3u) << 4;
            sum = fmaf(__fmul_rn(l < 16 ? d0 : d1, (float)((int)q - 32)), X[l], sum);
        }
        return sum;
    }
    static constexpr bool kMayStraddle = true;
    static constexpr bool kF16 = false;

    template <bool GEN, int NO>
    static __device__ __forceinline__ void rows(const RowSet<NO>& R, const XState<4>& x, int g, int, int,
                                                RowPair (&acc)[NO]) {
        const int s = g >> 1;
        float d0[NO], d1[NO];
#pragma unroll
        for (int o = 0; o < NO; ++o) {
            d0[o] = sh_half<208>(R.s0[o]), d1[o] = sh_half<208>(R.s1[o]);
            acc[o].a = acc[o].b = 0.f;
        }
        static_for<2>([&](auto hc) {
            constexpr int H = decltype(hc)::value;
            uint32_t u[NO][2];
#pragma unroll
            for (int o = 0; o < NO; ++o) {
                const RowAddr& r = R.r[o];
                u[o][0] = code_word<128 + 32 * H, GEN>(r, r.base), u[o][1] = code_word<128 + 32 * H + 16, GEN>(r, r.base);
            }
            uint32_t l[NO][2][2];
#pragma unroll
            for (int o = 0; o < NO; ++o) {
                const RowAddr& r = R.r[o];
                l[o][0][0] = code_word<64 * H, GEN>(r, r.base), l[o][0][1] = code_word<64 * H + 16, GEN>(r, r.base);
                l[o][1][0] = code_word<64 * H + 32, GEN>(r, r.base), l[o][1][1] = code_word<64 * H + 48, GEN>(r, r.base);
            }
            static_for<2>([&](auto cc) {
                constexpr int C = decltype(cc)::value, CH = 2 * H + C;        // groups 2 C and 2 C + 1 of the half
                int c[NO][4];
                static_for<2>([&](auto jc) {
                    constexpr int J = decltype(jc)::value;
#pragma unroll
                    for (int o = 0; o < NO; ++o) {
                        uint32_t b[2];
#pragma unroll
                        for (int i = 0; i < 2; ++i) {
                            const uint32_t hi = 2 * C + J < 2 ? u[o][i] << (4 - 2 * (2 * C + J)) : u[o][i] >> (2 * (2 * C + J) - 4);
                            b[i] = ((C ? l[o][J][i] >> 4 : l[o][J][i]) & 0x0F0F0F0Fu) | (hi & 0x30303030u);
                        }
                        imma<false>(c[o], x.a[2 * CH + J], b[0], b[1], J == 0 ? x.init[CH] : c[o]);
                    }
                });
#pragma unroll
                for (int o = 0; o < NO; ++o) {
                    const float e0 = d0[o] * (float)sh_s8<192 + 4 * CH>(R.s0[o] + s), e1 = d1[o] * (float)sh_s8<192 + 4 * CH>(R.s1[o] + s);
                    acc[o].a = fmaf(e0, unit_sum(c[o][0], c[o][2], x.klo[CH], x.nlo[CH], x.khi[CH]), acc[o].a);
                    acc[o].b = fmaf(e1, unit_sum(c[o][1], c[o][3], x.klo[CH], x.nlo[CH], x.khi[CH]), acc[o].b);
                }
            });
        });
    }
};

// q2_K: sixteen bytes of (scale | offset << 4), 64 bytes of 2-bit codes, d, dmin.
struct ImmaQ2K {
    static constexpr bool kHasMin = true;
    static constexpr int kSuper = 84, kChains = 4, kGroup = 16, kOffset = 0;
    static __device__ __forceinline__ float sum_of(uint32_t row, int k, uint32_t word, const float* X) {
        const int h = k >> 2, j = k & 3;
        const uint32_t codes = row + 32 * h, p0 = sh_u8<0>(row + 8 * h + 2 * j), p1 = sh_u8<1>(row + 8 * h + 2 * j);
        const float d = sh_half<80>(row), dmin = sh_half<82>(row);
        const float d0 = __fmul_rn(d, (float)(p0 & 15u)), m0 = __fmul_rn(dmin, (float)(p0 >> 4));
        const float d1 = __fmul_rn(d, (float)(p1 & 15u)), m1 = __fmul_rn(dmin, (float)(p1 >> 4));
        float sum = 0.f;
#pragma unroll 2
        for (; word != 0; word &= word - 1) {
            const int l = __ffs((int)word) - 1;
            const float q = (float)(sh_u8<16>(codes + l) >> (2 * j) & 3u);
            sum = fmaf(__fsub_rn(__fmul_rn(l < 16 ? d0 : d1, q), l < 16 ? m0 : m1), X[l], sum);
        }
        return sum;
    }
    static constexpr bool kMayStraddle = false;
    static constexpr bool kF16 = false;

    template <bool GEN, int NO>
    static __device__ __forceinline__ void rows(const RowSet<NO>& R, const XState<4>& x, int g, int, int,
                                                RowPair (&acc)[NO]) {
        const int s = g >> 1;
        float d0[NO], d1[NO], n0[NO], n1[NO];
#pragma unroll
        for (int o = 0; o < NO; ++o) {
            const uint32_t dd0 = sh32o<80>(R.s0[o]), dd1 = sh32o<80>(R.s1[o]);
            d0[o] = half_lo_to_float(dd0), d1[o] = half_lo_to_float(dd1);
            n0[o] = -half_hi_to_float(dd0), n1[o] = -half_hi_to_float(dd1);
            acc[o].a = acc[o].b = 0.f;
        }
        static_for<2>([&](auto hc) {
            constexpr int H = decltype(hc)::value;
            uint32_t w0[NO], w1[NO];
#pragma unroll
            for (int o = 0; o < NO; ++o) w0[o] = sh32o<16 + 32 * H>(R.r[o].base), w1[o] = sh32o<32 + 32 * H>(R.r[o].base);
            static_for<2>([&](auto cc) {
                constexpr int C = decltype(cc)::value, CH = 2 * H + C;
#pragma unroll
                for (int o = 0; o < NO; ++o) {
                    int c[4];
                    imma<false>(c, x.a[2 * CH], (w0[o] >> (4 * C)) & 0x03030303u, (w1[o] >> (4 * C)) & 0x03030303u, x.init[CH]);
                    imma<false>(c, x.a[2 * CH + 1], (w0[o] >> (4 * C + 2)) & 0x03030303u, (w1[o] >> (4 * C + 2)) & 0x03030303u, c);
                    const uint32_t p0 = sh_u8<4 * CH>(R.s0[o] + s), p1 = sh_u8<4 * CH>(R.s1[o] + s);
                    const float e0 = d0[o] * (uint_float23(p0 & 15u) - 8388608.f), e1 = d1[o] * (uint_float23(p1 & 15u) - 8388608.f);
                    const float f0 = n0[o] * (uint_float23(p0 >> 4) - 8388608.f), f1 = n1[o] * (uint_float23(p1 >> 4) - 8388608.f);
                    acc[o].a = affine_sum<false>(c[0], c[2], e0, f0, x.xlo[CH], x.xhi[CH], x.klo[CH], x.khi[CH], acc[o].a);
                    acc[o].b = affine_sum<false>(c[1], c[3], e1, f1, x.xlo[CH], x.xhi[CH], x.klo[CH], x.khi[CH], acc[o].b);
                }
            });
        });
    }
};

// f16: nothing is decoded and HBM binds long before the FMA pipes do; plain fp32 accumulation, four rows at a time, a
// lane owns eight columns of the warp's 256.
struct ImmaF16 {
    static constexpr int kSuper = 512, kChains = 1;
    static constexpr bool kF16 = true;
};

// ------------------------------------------------------------------ activations ---

// X as fixed point in shared memory, blocks of 32 of kXBlock bytes: [digit 0..3][32 bytes] | scale of the first and of the
// second unit (one unit with GROUP 32).  A thread converts eight consecutive values; two (GROUP 16) or four lanes share a
// unit.  What does not fit a unit's fixed point gets its bit in `apart` (one per column); true if the thread met any.
template <int GROUP>
__device__ __forceinline__ bool convert_x(const float* X, int cols, int padded, uint32_t xs, uint8_t* apart, int tid) {
    bool any = false;
    constexpr int kDepth = 2;                        // pieces of a thread whose loads are in flight together
    const int pieces = padded >> 3;                  // a multiple of 32: whole warps take part or drop out
    for (int p0 = tid; p0 < pieces; p0 += kDepth * kComputeThreads) {
        float4 v[kDepth][2];
#pragma unroll
        for (int j = 0; j < kDepth; ++j) {
            const int piece = p0 + j * kComputeThreads;
            v[j][0] = v[j][1] = make_float4(0.f, 0.f, 0.f, 0.f);
            if (8 * piece < cols) {
                v[j][0] = __ldcg(reinterpret_cast<const float4*>(X) + 2 * piece);
                v[j][1] = __ldcg(reinterpret_cast<const float4*>(X) + 2 * piece + 1);
            }
        }
#pragma unroll
        for (int j = 0; j < kDepth; ++j) {
            const int piece = p0 + j * kComputeThreads;
            if (piece >= pieces) break;
            float f[8] = {v[j][0].x, v[j][0].y, v[j][0].z, v[j][0].w, v[j][1].x, v[j][1].y, v[j][1].z, v[j][1].w};
            float most = 0.f, little = __uint_as_float(0x7F800000u);       // largest (NaN if any is) and smallest magnitude
#pragma unroll
            for (int i = 0; i < 8; ++i) {
                asm("max.NaN.f32 %0, %0, %1;" : "+f"(most) : "f"(fabsf(f[i])));
                little = fminf(little, fabsf(f[i]));
            }
            uint32_t m = __float_as_uint(most);
            const bool far = __any_sync(0xFFFFFFFFu, m >= kApartFrom);
            if (far) {
                m = 0;
#pragma unroll
                for (int i = 0; i < 8; ++i) {
                    const uint32_t b = __float_as_uint(f[i]) & 0x7FFFFFFFu;
                    m = max(m, b < kApartFrom ? b : 0u);
                }
            }
            m = max(m, __shfl_xor_sync(0xFFFFFFFFu, m, 1));
            if (GROUP == 32) m = max(m, __shfl_xor_sync(0xFFFFFFFFu, m, 2));
            // the scale 2^(e - 157) brings the unit's largest magnitude to 2^30 .. 2^31, below 0x7F7F7F80 (significands from
            // 0xFEFEFF on take the next exponent): the top digit stays below 128
            const uint32_t e = max((m + 0x10101u) >> 23, 31u);
            const float up = __uint_as_float((284u - e) << 23);
            const float d = __uint_as_float((e - 30u) << 23);
            const uint32_t least = m > kApartBelow ? m - kApartBelow : 1u;
            uint32_t bits = 0;
            if (far || __float_as_uint(little) < least) {
#pragma unroll
                for (int i = 0; i < 8; ++i) {
                    const uint32_t b = __float_as_uint(f[i]) & 0x7FFFFFFFu;
                    if (b - least >= kApartFrom - least) {         // below `least` or from kApartFrom on
                        bits |= b != 0 ? 1u << i : 0u;
                        f[i] = 0.f;
                    }
                }
            }
            apart[piece] = (uint8_t)bits;
            any |= bits != 0;
            uint32_t w[8];
#pragma unroll
            for (int i = 0; i < 8; ++i) w[i] = ((uint32_t)__float2int_rn(f[i] * up) + 0x00808080u) ^ 0x00808080u;   // four signed digits
            const uint32_t dst = xs + (uint32_t)(piece >> 2) * kXBlock + 8u * (piece & 3);
            uint32_t dig[4][2];
#pragma unroll
            for (int q = 0; q < 2; ++q) {
                const uint32_t lo01 = __byte_perm(w[4 * q], w[4 * q + 1], 0x5140), lo23 = __byte_perm(w[4 * q + 2], w[4 * q + 3], 0x5140);
                const uint32_t hi01 = __byte_perm(w[4 * q], w[4 * q + 1], 0x7362), hi23 = __byte_perm(w[4 * q + 2], w[4 * q + 3], 0x7362);
                dig[0][q] = __byte_perm(lo01, lo23, 0x5410), dig[1][q] = __byte_perm(lo01, lo23, 0x7632);
                dig[2][q] = __byte_perm(hi01, hi23, 0x5410), dig[3][q] = __byte_perm(hi01, hi23, 0x7632);
            }
#pragma unroll
            for (int k = 0; k < 4; ++k)
                asm volatile("st.shared.v2.b32 [%0], {%1, %2};" ::"r"(dst + 32u * k), "r"(dig[k][0]), "r"(dig[k][1]) : "memory");
            if ((piece & (GROUP / 8 - 1)) == 0)
                asm volatile("st.shared.f32 [%0], %1;" ::"r"(xs + (uint32_t)(piece >> 2) * kXBlock + 128u +
                                                             (GROUP == 16 ? 4u * ((piece >> 1) & 1) : 0u)),
                             "f"(d)
                             : "memory");
        }
    }
    return any;
}

// Adds weight * activation of the columns of a 256-column piece that are kept apart (bit table at `bits`, of whose eight words
// those in `words` are not zero; activations at X), in fp32, to the row sums of a tile of n rows that the warp has just put
// into its table.  Four groups of eight rows (from `first` on, `step` apart) at a time with a lane per row, or, with more than
// two words or fewer rows, one group with four lanes per row that take the words in turn.  `piece` = where the tile's row 0 has
// the piece in shared memory, `at` = the table's entry of row 0, `shift0` = row 0's offset behind the boundary its copy
// started at, `rb` = what the next row's offset differs by.
template <class T>
__device__ __noinline__ void add_apart(uint32_t piece, uint32_t pitch, uint32_t shift0, uint32_t rb, uint32_t at, uint32_t bits,
                                       uint32_t words, const float* X, int n, int first, int step, int lane) {
    __syncwarp();
    const bool wide = __popc(words) <= 2 && n > first + step;
    uint32_t mine = words;
    if (!wide) mine = words & (0x11u << (lane & 3));
    const int g = wide ? lane & 7 : lane >> 2;
    for (int u = first + (wide ? (lane >> 3) * step : 0); __any_sync(0xFFFFFFFFu, u < n); u += wide ? 4 * step : step) {
        const int i = min(u + g, n - 1);
        const uint32_t row = piece + (uint32_t)i * pitch + ((shift0 + (uint32_t)i * rb) & 15u);
        float sum = 0.f;
        for (uint32_t m = mine; m != 0; m &= m - 1) {
            const int k = __ffs((int)m) - 1;
            sum += T::sum_of(row, k, sh32(bits + 4u * k), X + 32 * k);
        }
        __syncwarp();
        if (!wide) {
            sum += __shfl_xor_sync(0xFFFFFFFFu, sum, 1);
            sum += __shfl_xor_sync(0xFFFFFFFFu, sum, 2);
        }
        put_sum(at + (uint32_t)u * (4 * kComputeWarps) + 4u * g, sum, u < n && (wide || (lane & 3) == 0), true);
    }
}

// The lane's part of the activations of one 256-column piece (eight blocks at xb) into registers.
template <class T>
__device__ __forceinline__ void load_x(XState<T::kChains>& x, uint32_t xb, uint32_t zeros, int g, int t) {
    const int s = g >> 1, odd = g & 1;
    constexpr bool kSums = T::kOffset != 0 || T::kHasMin;
#pragma unroll
    for (int ch = 0; ch < T::kChains; ++ch) {
        const int u = 4 * ch + s;
        const uint32_t blk = xb + (uint32_t)(T::kGroup == 32 ? u : u >> 1) * kXBlock;
        const uint32_t dig = blk + 32u * odd + 4u * t;
        const uint32_t meta = blk + 128u + (T::kGroup == 32 ? 0u : 4u * (u & 1));
        int sum_lo, sum_hi;
        if constexpr (T::kGroup == 32) {
            // zeros are loaded, not selected: the compiler would redo 32 selections per group of rows to save registers
            sum_lo = sum_hi = 0;
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                const uint32_t from = s == j ? dig : zeros;
                x.a[4 * ch + j][0] = sh32o<0>(from), x.a[4 * ch + j][1] = sh32o<64>(from);
                x.a[4 * ch + j][2] = sh32o<16>(from), x.a[4 * ch + j][3] = sh32o<80>(from);
                if constexpr (kSums) {
                    sum_lo = dp4a_ss(x.a[4 * ch + j][0], 0x01010101u, dp4a_ss(x.a[4 * ch + j][2], 0x01010101u, sum_lo));
                    sum_hi = dp4a_ss(x.a[4 * ch + j][1], 0x01010101u, dp4a_ss(x.a[4 * ch + j][3], 0x01010101u, sum_hi));
                }
            }
        } else {
            sum_lo = sum_hi = 0;
#pragma unroll
            for (int q = 0; q < 2; ++q) {
                const uint32_t from = s == 2 * q ? dig + 16u * (u & 1) : zeros, from2 = s == 2 * q + 1 ? dig + 16u * (u & 1) : zeros;
                x.a[2 * ch + q][0] = sh32o<0>(from), x.a[2 * ch + q][1] = sh32o<64>(from);
                x.a[2 * ch + q][2] = sh32o<0>(from2), x.a[2 * ch + q][3] = sh32o<64>(from2);
                if constexpr (kSums) {
                    sum_lo = dp4a_ss(x.a[2 * ch + q][0], 0x01010101u, dp4a_ss(x.a[2 * ch + q][2], 0x01010101u, sum_lo));
                    sum_hi = dp4a_ss(x.a[2 * ch + q][1], 0x01010101u, dp4a_ss(x.a[2 * ch + q][3], 0x01010101u, sum_hi));
                }
            }
        }
        x.init[ch][0] = x.init[ch][1] = x.init[ch][2] = x.init[ch][3] = kIntMagic;
        if constexpr (kSums) {
            // the four lanes with equal g hold the unit's 32 (16) digits
            sum_lo += __shfl_xor_sync(0xFFFFFFFFu, sum_lo, 1), sum_hi += __shfl_xor_sync(0xFFFFFFFFu, sum_hi, 1);
            sum_lo += __shfl_xor_sync(0xFFFFFFFFu, sum_lo, 2), sum_hi += __shfl_xor_sync(0xFFFFFFFFu, sum_hi, 2);
            x.init[ch][0] = x.init[ch][1] = kIntMagic + T::kOffset * sum_lo;
            x.init[ch][2] = x.init[ch][3] = kIntMagic + T::kOffset * sum_hi;
        }
        const float d = __uint_as_float(sh32(meta));
        x.klo[ch] = odd ? d * 256.f : d;
        x.khi[ch] = odd ? d * 16777216.f : d * 65536.f;
        x.nlo[ch] = -12582912.f * x.klo[ch];
        x.xlo[ch] = (float)sum_lo, x.xhi[ch] = (float)sum_hi;
    }
}

// ------------------------------------------------------------------ kernel ---

// DROP: testing aid, from tile p.drop_tile on nothing is requested (see lw_debug_drop_copy).
template <class T, bool DROP = false>
__global__ void __launch_bounds__(kImmaThreads, 1) matvec_imma_kernel(const __grid_constant__ ImmaParams p) {
    extern __shared__ __align__(128) uint8_t smem[];
    // header: [0,64) full barriers | [64,128) empty barriers | 128 a wait gave up | [160,256) zeros
    // then two tables of row sums, the bits of columns kept apart, the activations, the ring of tiles
    volatile int* gave_up = reinterpret_cast<volatile int*>(smem + 128);
    const uint32_t base = smem_u32(smem);
    const uint32_t full = base, empty = base + 64;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int cta = (int)blockIdx.x;
    const int slots = p.slots;
    const int v0 = p.share * cta + min(cta, p.extra), v1 = v0 + p.share + (cta < p.extra ? 1 : 0);     // this CTA's rows

    if (tid < 24) reinterpret_cast<uint32_t*>(smem + kZeros)[tid] = 0;
    if (tid == 0) {
        for (int s = 0; s < slots; ++s) {
            mbar_init(reinterpret_cast<uint64_t*>(smem) + s, 1);
            mbar_init(reinterpret_cast<uint64_t*>(smem + 64) + s, kComputeWarps);
        }
        *gave_up = 0;
        fence_barrier_init();
    }
    __syncthreads();
    grid_launch_dependents();     // the next kernel on the stream may be placed and set up
    grid_dependency_wait();       // W and X may be produced, and Y still read, by the previous one

    if (warp >= kComputeWarps) {
        asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(kCopyRegs));
        if (warp > kComputeWarps) return;
        // ------------------------------------------------------------------ copy warp ---
        // one bulk copy per row of a tile, the rows spread over the lanes
        const uint64_t policy = l2_evict_first_policy();
        int slot = 0, issued = 0;
        uint32_t parity = 1;                             // (the first pass over the ring waits for nothing)
        const int fold_rows = p.fold_rows, tile_rows = p.tile_rows;
        const uint32_t rb = p.row_bytes, pitch = p.pitch;
        const bool ragged = p.ragged;
        for (int r0 = v0; r0 < v1; r0 += fold_rows) {
            const int r1 = min(v1, r0 + fold_rows);
            for (int c = 0; c < p.n_chunks; ++c) {
                const uint32_t coff = (uint32_t)c * p.chunk_sb * T::kSuper;
                const uint32_t piece = min((uint32_t)p.chunk_sb * T::kSuper, rb - coff);
                for (int r = r0; r < r1; r += tile_rows) {
                    const int n = min(tile_rows, r1 - r);
                    if constexpr (DROP) {
                        if (issued >= p.drop_tile) return;       // (the compute warps still wait for what was requested)
                    }
                    // one decision for the warp: a compute warp may give up between two lanes' looks at the flag
                    bool stop = *gave_up != 0;
                    if (!stop && !mbar_wait_bounded(empty + 8u * slot, parity)) {
                        stop = true;
                        *gave_up = 1;
                        atomicExch(p.fault, (int)FAULT_BULK_WAIT_TIMEOUT);
                    }
                    if (__any_sync(0xFFFFFFFFu, stop)) {
                        // nothing further is requested; what is in flight lands before shared memory is released
                        for (int i = max(0, issued - slots); i < issued; ++i)
                            if (!mbar_wait_bounded(full + 8u * (i % slots), (uint32_t)(i / slots) & 1u))
                                atomicExch(p.fault, (int)FAULT_DRAIN_TIMEOUT);
                        return;
                    }
                    const uint32_t dst0 = base + p.ring_off + (uint32_t)slot * p.slot_bytes, bar = full + 8u * slot;
                    if (!ragged) {
                        if (lane == 0) mbar_expect_tx(reinterpret_cast<uint64_t*>(smem) + slot, (uint32_t)n * piece);
                        __syncwarp();
                        for (int i = lane; i < n; i += 32) {
                            const uint8_t* src = p.W + (int64_t)(r + i) * rb + coff;
                            bulk_row(dst0 + (uint32_t)i * pitch, src, piece, bar, policy);
                        }
                    } else {
                        // from the 16-byte boundary below the row's piece to the one above its end; at the end of the
                        // matrix to the boundary below, and the last bytes (2-byte units) with plain stores
                        const uint8_t* W = p.W;
                        const int64_t total = (int64_t)p.rows * rb;
                        uint32_t bytes = 0;
                        for (int i = lane; i < n; i += 32) {
                            const int64_t at = (int64_t)(r + i) * rb + coff, from = at & ~(int64_t)15;
                            int64_t to = (at + piece + 15) & ~(int64_t)15;
                            if (to > total) {
                                to = total & ~(int64_t)15;
                                for (int64_t k = to; k < total; k += 2)
                                    *reinterpret_cast<uint16_t*>(smem + (dst0 - base) + (uint32_t)i * pitch + (uint32_t)(k - from)) =
                                        *reinterpret_cast<const uint16_t*>(W + k);
                            }
                            bytes += (uint32_t)(to - from);
                        }
                        bytes = __reduce_add_sync(0xFFFFFFFFu, bytes);
                        __syncwarp();                // the stores above are ordered before lane 0's arrival
                        if (lane == 0) mbar_expect_tx(reinterpret_cast<uint64_t*>(smem) + slot, bytes);
                        __syncwarp();
                        for (int i = lane; i < n; i += 32) {
                            const int64_t at = (int64_t)(r + i) * rb + coff, from = at & ~(int64_t)15;
                            int64_t to = (at + piece + 15) & ~(int64_t)15;
                            if (to > total) to = total & ~(int64_t)15;
                            if (to > from) bulk_row(dst0 + (uint32_t)i * pitch, W + from, (uint32_t)(to - from), bar, policy);
                        }
                    }
                    __syncwarp();
                    ++issued;
                    if (++slot == slots) slot = 0, parity ^= 1u;
                }
            }
        }
        return;
    }

    // ------------------------------------------------------------------ compute warps ---
    asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(kComputeRegs));
    const int g = lane >> 2, t = lane & 3;
    const uint32_t xs = base + p.x_off;
    float* table = reinterpret_cast<float*>(smem + kImmaHeader);
    int slot = 0, buf = 0;
    uint32_t parity = 0;
    const int nsb = (p.cols + 255) >> 8, chunk_sb = p.chunk_sb, tile_rows = p.tile_rows, row_groups = p.row_groups;
    const int fold_rows = p.fold_rows, n_chunks = p.n_chunks;
    const uint32_t rb = p.row_bytes, pitch = p.pitch;
    const int rgrp = warp / chunk_sb, cw = warp - rgrp * chunk_sb;
    const bool ragged = p.ragged;
    bool apart = false;                              // does any activation of the row not fit the fixed point?
    if constexpr (T::kF16) {
        for (int i = tid; i < nsb * 64; i += kComputeThreads) {
            float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
            if (4 * i < p.cols) v = __ldcg(reinterpret_cast<const float4*>(p.X) + i);
            asm volatile("st.shared.v4.f32 [%0], {%1, %2, %3, %4};" ::"r"(xs + 16u * i), "f"(v.x), "f"(v.y), "f"(v.z), "f"(v.w)
                         : "memory");
        }
    } else {
        apart = convert_x<T::kGroup>(p.X, p.cols, nsb * 256, xs, smem + kApartBits, tid);
    }
    apart = compute_bar_any(apart);
    const uint32_t lane_g = (uint32_t)g * pitch + (uint32_t)cw * T::kSuper, lane_s = (uint32_t)(2 * t) * pitch + (uint32_t)cw * T::kSuper;
    const bool straddle = ragged || (((uint32_t)cw * T::kSuper) & 2u);
    XState<T::kChains> x;
    uint32_t words_apart = 0;                        // which of the eight words of this warp's 256 columns have any
    f2 xf[4];                                        // f16: the lane's eight activations
    for (int r0 = v0; r0 < v1; r0 += fold_rows) {
        const int r1 = min(v1, r0 + fold_rows);
        // this lane's entry of the row-sum table: row 0 of the group, the lane's row within its unit
        const uint32_t tab0 = base + kImmaHeader + (uint32_t)(buf * kTableFloats * 4 + cw * 32) +
                              4u * (T::kF16 ? 2 * (lane >> 4) + ((lane >> 3) & 1) : 2 * t + (g & 1));
        for (int c = 0; c < n_chunks; ++c) {
            const int sb = c * chunk_sb + cw;
            const bool live = rgrp < row_groups && sb < nsb;
            const int nlive = T::kF16 ? p.cols - 256 * sb - 8 * lane : (p.cols - 256 * sb) >> 5;
            if (live && (n_chunks > 1 || r0 == v0)) {
                if constexpr (T::kF16) {
                    const uint4 a = sh128(xs + 1024u * sb + 32u * lane), b = sh128(xs + 1024u * sb + 32u * lane + 16);
                    xf[0] = pack2u(a.x, a.y), xf[1] = pack2u(a.z, a.w), xf[2] = pack2u(b.x, b.y), xf[3] = pack2u(b.z, b.w);
                } else {
                    load_x<T>(x, xs + (uint32_t)(8 * sb) * kXBlock, base + kZeros, g, t);
                    if (apart) words_apart = __ballot_sync(0xFFFFFFFFu, lane < 8 && sh32(base + kApartBits + 32u * sb + 4u * (lane & 7)) != 0);
                }
            }
            const uint32_t coff = (uint32_t)c * chunk_sb * T::kSuper;
            for (int r = r0; r < r1; r += tile_rows) {
                const int n = min(tile_rows, r1 - r);
                if (!mbar_try_wait(full + 8u * slot, parity) && *gave_up == 0 && !mbar_wait_bounded(full + 8u * slot, parity)) {
                    *gave_up = 1;
                    atomicExch(p.fault, (int)FAULT_BULK_WAIT_TIMEOUT);
                }
                if (live) {
                    const uint32_t tile = base + p.ring_off + (uint32_t)slot * p.slot_bytes;
                    const uint32_t tab = tab0 + (uint32_t)(r - r0) * (4 * kComputeWarps);
                    if constexpr (T::kF16) {
                        for (int u = 4 * rgrp; u < n; u += 4 * row_groups) {
                            // four rows x eight columns per lane
                            float acc[4];
                            const uint32_t w = tile + (uint32_t)u * pitch + 512u * cw + 16u * lane;
#pragma unroll
                            for (int i = 0; i < 4; ++i) {
                                const uint4 q = sh128(w + i * pitch);
                                const uint32_t h[4] = {q.x, q.y, q.z, q.w};
                                f2 a = 0;
#pragma unroll
                                for (int k = 0; k < 4; ++k) a = fma2(pack2(half_lo_to_float(h[k]), half_hi_to_float(h[k])), xf[k], a);
                                acc[i] = nlive > 0 ? hsum2(a) : 0.f;
                            }
                            const bool up = lane & 16, mid = lane & 8;
                            float a0 = up ? acc[2] : acc[0], a1 = up ? acc[3] : acc[1];
                            a0 += __shfl_xor_sync(0xFFFFFFFFu, up ? acc[0] : acc[2], 16);
                            a1 += __shfl_xor_sync(0xFFFFFFFFu, up ? acc[1] : acc[3], 16);
                            float out = mid ? a1 : a0;
                            out += __shfl_xor_sync(0xFFFFFFFFu, mid ? a0 : a1, 8);
                            out += __shfl_xor_sync(0xFFFFFFFFu, out, 4);
                            out += __shfl_xor_sync(0xFFFFFFFFu, out, 2);
                            out += __shfl_xor_sync(0xFFFFFFFFu, out, 1);
                            const uint32_t row = (uint32_t)(r - r0 + u);           // a multiple of 4
                            put_sum(tab0 + (row >> 3) * (32 * kComputeWarps) + (row & 4u) * 4u, out, (lane & 7) == 0, c > 0);
                        }
                    } else {
                        const int step = 8 * row_groups;
                        const uint32_t far = (uint32_t)step * pitch;
                        // the rows' first bytes behind the boundaries their copies started at
                        auto shift = [&](int u, int i) { return (((uint32_t)(r + u) + i) * rb + coff) & 15u; };
                        auto products = [&](auto no, int u) {
                            constexpr int NO = decltype(no)::value;
                            RowSet<NO> R;
                            RowPair acc[NO];
#pragma unroll
                            for (int o = 0; o < NO; ++o) {
                                const uint32_t o8 = tile + (uint32_t)u * pitch + o * far;
                                uint32_t rg = o8 + lane_g;
                                R.s0[o] = o8 + lane_s, R.s1[o] = R.s0[o] + pitch;
                                if (ragged) {
                                    rg += shift(u + o * step, g);
                                    R.s0[o] += shift(u + o * step, 2 * t), R.s1[o] += shift(u + o * step, 2 * t + 1);
                                }
                                if (T::kMayStraddle && straddle) R.r[o] = row_addr(rg);
                                else R.r[o].base = rg;
                                R.r[o].base += 4u * t;
                            }
                            // rows of this warp's piece two bytes off the word grid (q6_K's odd pieces, ragged rows)
                            if (T::kMayStraddle && straddle) T::template rows<T::kMayStraddle, NO>(R, x, g, t, nlive, acc);
                            else T::template rows<false, NO>(R, x, g, t, nlive, acc);
                            // over the eight lanes with equal t: row 2 t to the even ones, row 2 t + 1 to the odd ones
                            const bool odd = g & 1;
                            float v[NO];
#pragma unroll
                            for (int o = 0; o < NO; ++o) {
                                v[o] = odd ? acc[o].b : acc[o].a;
                                v[o] += __shfl_xor_sync(0xFFFFFFFFu, odd ? acc[o].a : acc[o].b, 4);
                            }
                            const uint32_t at = tab + (uint32_t)u * (4 * kComputeWarps);     // [row / 8][warp][row % 8]
                            if constexpr (NO == 2) {
                                // the second group of rows to the lanes with g & 2
                                const bool second = g & 2;
                                float out = second ? v[1] : v[0];
                                out += __shfl_xor_sync(0xFFFFFFFFu, second ? v[0] : v[1], 8);
                                out += __shfl_xor_sync(0xFFFFFFFFu, out, 16);
                                put_sum(second ? at + (uint32_t)step * (4 * kComputeWarps) : at, out, g < 4, c > 0);
                            } else {
                                float out = v[0] + __shfl_xor_sync(0xFFFFFFFFu, v[0], 8);
                                out += __shfl_xor_sync(0xFFFFFFFFu, out, 16);
                                put_sum(at, out, g < 2, c > 0);
                            }
                        };
                        int u = 8 * rgrp;
                        for (; u + step < n; u += 2 * step) products(std::integral_constant<int, 2>{}, u);
                        if (u < n) products(std::integral_constant<int, 1>{}, u);
                        if (words_apart != 0)
                            add_apart<T>(tile + (uint32_t)cw * T::kSuper, pitch, ragged ? (uint32_t)r * rb + coff : 0u, ragged ? rb : 0u,
                                         tab - 4u * (2 * t + (g & 1)), base + kApartBits + 32u * sb, words_apart, p.X + 256 * sb, n, 8 * rgrp, step, lane);
                    }
                }
                __syncwarp();
                if (lane == 0) mbar_arrive_addr(empty + 8u * slot);
                if (++slot == slots) slot = 0, parity ^= 1u;
            }
        }
        compute_bar();                               // the sums of rows r0 .. r1 are complete
        for (int i = tid; i < r1 - r0; i += kComputeThreads) {
            const float* e = table + buf * kTableFloats + (i >> 3) * (kComputeWarps * 8) + (i & 7);
            float sum = 0.f;
            for (int k = 0; k < chunk_sb; ++k) sum += e[8 * k];
            p.Y[r0 + i] = sum;
        }
        buf ^= 1;
    }
}

// ------------------------------------------------------------------ host side ---

int super_bytes(int fmt) {
    switch (fmt) {
        case LW_F16: return ImmaF16::kSuper;
        case LW_Q8_0: return ImmaLegacy<LW_Q8_0>::kSuper;
        case LW_Q4_0: return ImmaLegacy<LW_Q4_0>::kSuper;
        case LW_Q4_1: return ImmaLegacy<LW_Q4_1>::kSuper;
        case LW_Q5_0: return ImmaLegacy<LW_Q5_0>::kSuper;
        case LW_Q5_1: return ImmaLegacy<LW_Q5_1>::kSuper;
        case LW_Q6_K: return ImmaQ6K::kSuper;
        case LW_Q2_K: return ImmaQ2K::kSuper;
        default: return 0;               // q4_K and q5_K: whole 16-byte pieces, always the streaming kernels
    }
}

constexpr int64_t kMaxRows = (int64_t)1 << 30;

// Geometry and shared memory of a launch; false when the format or width is not covered.  Slots of about 38 KB: a
// tile's fixed costs (two barrier operations per warp) are spread over several groups of rows, and four or more slots fit.
bool plan(int fmt, int64_t rows, int64_t cols, int grid, ImmaParams& p, size_t& smem_bytes) {
    const int64_t rb = (int64_t)lw_row_bytes(fmt, cols);
    const int super = super_bytes(fmt);
    if (super == 0 || rb == 0 || cols > 16384 || rows > kMaxRows) return false;
    const int nsb = (int)((cols + 255) / 256);
    const int chunks = (nsb + kComputeWarps - 1) / kComputeWarps, chunk_sb = (nsb + chunks - 1) / chunks;
    const int64_t piece = std::min<int64_t>(rb, (int64_t)chunk_sb * super);
    p.rows = (int)rows;
    p.cols = (int)cols;
    p.share = (int)(rows / grid);
    p.extra = (int)(rows % grid);
    p.row_bytes = (uint32_t)rb;
    p.ragged = rb % 16 != 0 || (chunks > 1 && (chunk_sb * super) % 16 != 0);
    p.pitch = 16 * ((uint32_t)(p.ragged ? (piece + 29) / 16 : piece / 16) | 1u);
    p.chunk_sb = chunk_sb;
    p.n_chunks = chunks;
    p.row_groups = kComputeWarps / chunk_sb;
    p.x_off = kApartBits + 32u * nsb;
    p.ring_off = (uint32_t)((p.x_off + (size_t)nsb * (fmt == LW_F16 ? 1024 : 8 * kXBlock) + 127) & ~(size_t)127);
    const size_t margin = 1024;          // what a lane reads past the end of a row whose last piece is short lies inside
    const size_t avail = kImmaSmemMax - p.ring_off - margin;
    const int least = (fmt == LW_F16 ? 4 : 8) * p.row_groups;
    int k = (int)(std::min<size_t>(38 * 1024, avail / 4) / ((size_t)least * p.pitch));
    k = std::max(1, std::min(k, kFoldRows / least));
    while (k > 1 && (k - 1) * least >= p.share + 1) --k;       // no more rows than a CTA has
    p.tile_rows = k * least;
    p.fold_rows = kFoldRows / p.tile_rows * p.tile_rows;
    p.slot_bytes = (uint32_t)(((size_t)p.tile_rows * p.pitch + 127) & ~(size_t)127);
    const size_t n = std::min<size_t>(kSlotsMax, avail / p.slot_bytes);
    if (n < 2) return false;
    p.slots = (int)n;
    smem_bytes = p.ring_off + n * p.slot_bytes + margin;
    return true;
}

template <class T, bool DROP = false>
int launch_one(const ImmaParams& p, int grid, size_t smem_bytes, bool overlap, cudaStream_t stream) {
    static bool attr_set[64] = {false};
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return (int)e;
    if (dev < 0 || dev >= 64 || !attr_set[dev]) {
        e = cudaFuncSetAttribute(matvec_imma_kernel<T, DROP>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kImmaSmemMax);
        if (e != cudaSuccess) return (int)e;
        if (dev >= 0 && dev < 64) attr_set[dev] = true;
    }
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3((unsigned)grid);
    cfg.blockDim = dim3(kImmaThreads);
    cfg.dynamicSmemBytes = smem_bytes;
    cfg.stream = stream;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = overlap ? 1 : 0;
    return (int)cudaLaunchKernelEx(&cfg, matvec_imma_kernel<T, DROP>, p);
}

}  // namespace

// Narrow matrices stay with the generic kernel: its time grows with the width (a warp walks a row), this one's fixed part
// is 3.5 us (2.8 under launch overlap).  us, generic -> this kernel, weights from memory: q4_0 1000 rows x 800 columns 3.9 ->
// 3.8, x 1056 5.0 -> 3.9, x 2080 8.1 -> 4.1; 4096 x 800 4.5 -> 4.8, x 1056 5.4 -> 5.2; 11007 x 544 6.7 -> 7.2, x 800 8.3 ->
// 7.3; q6_K 1000 x 768 3.7 -> 4.1, x 1280 5.1 -> 4.5, 11007 x 768 8.7 -> 8.0; q2_K, which the generic kernel decodes in whole
// words, 4096 x 1280 4.9 -> 5.5, x 1792 6.2 -> 5.8, 11007 x 768 6.8 -> 7.5, x 1280 9.8 -> 9.3.
bool matvec_imma_supported(int fmt, int64_t rows, int64_t cols) {
    ImmaParams p;
    size_t smem = 0;
    const int64_t least = fmt == LW_Q2_K ? 1536 : 1024;
    const bool wide = cols >= least || (4 * cols >= 3 * least && rows >= 8192);
    return rows >= 1 && wide && plan(fmt, rows, cols, 148, p, smem);
}

int launch_matvec_imma(int fmt, const void* W, int64_t rows, int64_t cols, const float* X, float* Y, bool overlap,
                       cudaStream_t stream) {
    ImmaParams p;
    size_t smem = 0;
    const int grid = (int)std::min<int64_t>(device_sm_count(), rows);
    p.fault = device_fault_word();
    if (!p.fault || !plan(fmt, rows, cols, grid, p, smem)) return (int)cudaErrorInvalidValue;
    p.W = static_cast<const uint8_t*>(W);
    p.X = X;
    p.Y = Y;
    if (fmt == LW_Q4_0) {
        p.drop_tile = take_drop_unit();
        if (p.drop_tile >= 0) return launch_one<ImmaLegacy<LW_Q4_0>, true>(p, grid, smem, overlap, stream);
    }
    switch (fmt) {
        case LW_F16: return launch_one<ImmaF16>(p, grid, smem, overlap, stream);
        case LW_Q8_0: return launch_one<ImmaLegacy<LW_Q8_0>>(p, grid, smem, overlap, stream);
        case LW_Q4_0: return launch_one<ImmaLegacy<LW_Q4_0>>(p, grid, smem, overlap, stream);
        case LW_Q4_1: return launch_one<ImmaLegacy<LW_Q4_1>>(p, grid, smem, overlap, stream);
        case LW_Q5_0: return launch_one<ImmaLegacy<LW_Q5_0>>(p, grid, smem, overlap, stream);
        case LW_Q5_1: return launch_one<ImmaLegacy<LW_Q5_1>>(p, grid, smem, overlap, stream);
        case LW_Q6_K: return launch_one<ImmaQ6K>(p, grid, smem, overlap, stream);
        case LW_Q2_K: return launch_one<ImmaQ2K>(p, grid, smem, overlap, stream);
    }
    return (int)cudaErrorInvalidValue;
}

}  // namespace lw

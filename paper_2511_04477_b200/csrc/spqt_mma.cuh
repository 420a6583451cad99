// The product on tensor cores: 4-bit (and widened 3-bit) codes as fp16 operands of mma.sync without a conversion.
// Included after spqt_gemv_device.cuh.
//
// A is the codes, 16 rows x 16 list entries per instruction; B is the multipliers a = x*scale of the 16 entries,
// 8 columns.  An fp16 word whose upper bits are zero IS a subnormal, its integer value times 2^-24, so a code becomes
// an operand with one mask.  The two halves of a register have to be the same rows of two neighbouring entries, which is what
// ldmatrix.trans delivers from blocks that lie row after row in shared memory: one register then holds bytes
// (2g, 2g+1) of entries 2t and 2t+1, i.e. four codes of each, and four operations make four operands of it.
//
// a = x*scale has up to 22 significant bits.  It goes in as two fp16 values: hi = a*c rounded to a multiple of 1/2 and to
// fp16, lo = fp16(a*c - hi), c a power of two that every warp keeps per batch row so that its largest |a*c| so far lies in
// 2^12 .. 2^15.  hi + lo is a*c, or off by 2^-14 at most (2^-26 of the largest entry).  When an entry exceeds the range, c
// changes and the sums are rescaled.
// Why multiples of 1/2: the instruction brings its 16 products and the sum to one exponent, the largest, and keeps 25 bits
// below it (measured).  A subnormal operand counts there with the exponent of the smallest normal number, 2^-14, though its
// leading bit is up to ten places lower: a code's product may then reach past the 25 bits and is cut.  hi < 2^15 in
// multiples of 1/2 makes the largest exponent 2^0 and every product a multiple of 2^-25: nothing is cut, and the sums of hi are
// exact up to 24 bits.  What lo's products lose is 2^-11 of that; hi and lo have sums of their own.  Share of y that is not the
// fp16 nearest to the exact value, 200 shapes between 512 x 256 and 16384 x 28672, half of them with outliers: with
// hi = fp16(a*c) 1.8 % of the dense call's and 2.4 % of a batch's, now 0.27 and 0.31 %; with fp32 FMAs in sequence 0.34 and
// 0.33 %.  8192 x 28672 dense takes 22.3 us either way.  (Largest |a*c| from 2^10 up: 0.33 % with outliers.)
//
// Per chunk of 32 entries x 128 rows the arithmetic is 84 warp instructions (4 ldmatrix, 64 masks and byte
// permutations, 16 mma) where the packed-FMA form takes 218 for one row and 64 more for every further one.
#pragma once

namespace spqt {

// c of a warp that has seen nothing but zeros: any entry exceeds the range
constexpr float kMmaNoScale = 0x1p100f;
constexpr float kMmaLimit = 32768.0f;

// v rounded to a multiple of 1/2, |v| < 2^21; two of them
__device__ __forceinline__ float to_halves(float v) { return __fsub_rn(__fadd_rn(v, 6291456.0f), 6291456.0f); }
__device__ __forceinline__ unsigned long long to_halves2(unsigned long long v)
{
    return fadd2(fadd2(v, pack2(6291456.0f, 6291456.0f)), pack2(-6291456.0f, -6291456.0f));
}

// 1 / c of a power of two between 2^-100 and 2^100, exactly
__device__ __forceinline__ float power_of_two_inverse(float c) { return __uint_as_float((254u << 23) - __float_as_uint(c)); }

__device__ __forceinline__ void ldsm_x4_trans(unsigned addr, unsigned* r)
{
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0, %1, %2, %3}, [%4];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
                 : "r"(addr)
                 : "memory");
}
__device__ __forceinline__ void ldsm_x2_trans(unsigned addr, unsigned* r)
{
    asm volatile("ldmatrix.sync.aligned.m8n8.x2.trans.shared.b16 {%0, %1}, [%2];" : "=r"(r[0]), "=r"(r[1]) : "r"(addr) : "memory");
}
// The sums of hi and lo multipliers, when c changes by the factor f: what the new hi sum has below 2^-25 goes to lo's, or the
// next instruction would cut it off.  (From 1/4 up the new sum has no such bits; .375 rounds smaller ones.)
__device__ __forceinline__ void rescale_sums(float& hi, float& lo, float f)
{
    const float h = hi * f;
    hi = __fsub_rn(__fadd_rn(h, 0.375f), 0.375f);
    lo = lo * f + (h - hi);
}

// c[0..3] += A (16 x 16) * B (16 x 8), fp32 sums
__device__ __forceinline__ void mma_16816(float* c, unsigned a0, unsigned a1, unsigned a2, unsigned a3, unsigned b0, unsigned b1)
{
    asm("mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, {%0, %1, %2, %3};"
        : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
        : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}

// How the blocks of a format lie in a stage, and how the four nibble words of a group of tiles are read back.
//   kRow    bytes from one entry to the next.  4-bit blocks of 128 rows: 64, the 16-byte part p of entry e at place
//           p ^ ((e >> 1) & 3), so that the eight rows an ldmatrix matrix reads lie in different banks; of 64 rows:
//           32, part p at p ^ ((e >> 2) & 1).  3-bit blocks of 128 rows: 48 (conflict-free as it is); of 64 rows: 32,
//           the 8-byte 1-bit plane twice, so that lanes g and g + 4 find it.
//   kSp     groups of four tiles (64 rows) in a block
template <int G, int BITS>
struct MmaStage {
    static constexpr int kRow = BITS == 4 ? G / 2 : (G == 128 ? 48 : 32);
    static constexpr int kSp = G / 64;

    // byte offset of lane-wise addresses inside a stage: `a` for the x4 loads of the first 16 entries
    struct Lane {
        unsigned a, b;
        int sh;
        __device__ __forceinline__ explicit Lane(int lane)
        {
            const int e = ((lane >> 4) << 3) + (lane & 7), part = (lane >> 3) & 1;
            b = 0;
            sh = 0;
            if (BITS == 4 && G == 128) {
                a = e * 64 + ((part ^ ((e >> 1) & 3)) << 4);
            } else if (BITS == 4) {
                a = e * 32 + ((part ^ ((e >> 2) & 1)) << 4);
            } else if (G == 128) {
                a = e * 48 + part * 16;
                b = (lane & 15) * 48 + 32;   // the 1-bit plane: x2
            } else {
                a = e * 32 + part * 16;
                sh = lane >> 4;              // lanes g >= 4 hold rows 8.. of the 1-bit plane: one bit up
            }
        }
    };

    // The nibble words of the 16 entries from 16*ks: c[sp][0..3] = operand sources a0..a3 of tile group sp
    static __device__ __forceinline__ void load(unsigned stage, const Lane& l, int ks, unsigned (*c)[4])
    {
        const unsigned base = stage + (unsigned)(ks * 16 * kRow);
        if (BITS == 4) {
            ldsm_x4_trans(base + l.a, c[0]);
            if (G == 128) ldsm_x4_trans(base + (l.a ^ 32u), c[kSp - 1]);
        } else if (G == 128) {
            unsigned v[4], p[2];
            ldsm_x4_trans(base + l.a, v);
            ldsm_x2_trans(base + l.b, p);
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                // rows of half 0 (i even) use the even bits of the 1-bit plane, of half 1 the odd ones
                const unsigned q = (i & 1) ? p[i >> 1] >> 1 : p[i >> 1];
                c[0][i] = (v[i] & 0x33333333u) | ((q << 2) & 0x44444444u);
                c[kSp - 1][i] = ((v[i] >> 2) & 0x33333333u) | (q & 0x44444444u);
            }
        } else {
            unsigned v[4];
            ldsm_x4_trans(base + l.a, v);    // 2-bit plane, 1-bit plane, of entries 0..7, then of 8..15
#pragma unroll
            for (int i = 0; i < 2; ++i) {
                const unsigned q = v[2 * i + 1] >> l.sh;
                c[0][2 * i] = (v[2 * i] & 0x33333333u) | ((q << 2) & 0x44444444u);
                c[0][2 * i + 1] = ((v[2 * i] >> 2) & 0x33333333u) | (q & 0x44444444u);
            }
        }
    }

    // Row of the block that sum i (0..3) of tile (sp, type) belongs to in lane group g = lane / 4
    static __device__ __forceinline__ int row(int sp, int type, int i, int g)
    {
        return 16 * (2 * sp + (i >> 1)) + 2 * g + (type >> 1) + (G / 2) * (type & 1);
    }
};

// The four tiles of 16 entries and 64 rows: type 0 / 2 the low nibbles of the even / odd bytes, 1 the high nibbles of the
// even ones (in place: 16 times the code), 3 the whole odd bytes (one operation less than their high nibbles, whose sum is
// recovered at the end as (byte - low) / 16).
struct MmaTiles {
    unsigned a[4][4];
    __device__ __forceinline__ explicit MmaTiles(const unsigned* c)
    {
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            a[0][i] = c[i] & 0x000f000fu;
            a[1][i] = c[i] & 0x00f000f0u;
            a[3][i] = __byte_perm(c[i], 0u, 0x4341);
            a[2][i] = a[3][i] & 0x000f000fu;
        }
    }
};

// acc[type] += the operands of that type times B
__device__ __forceinline__ void mma_group(float (*acc)[4], const unsigned* c, const unsigned* b)
{
    const MmaTiles t(c);
#pragma unroll
    for (int type = 0; type < 4; ++type) mma_16816(acc[type], t.a[type][0], t.a[type][1], t.a[type][2], t.a[type][3], b[0], b[1]);
}

// The same over 32 entries (c0, then c1) for a B in two sets, hi and lo, whose sums share registers.  A sum that holds lo parts
// would lose them when the next hi product of a low nibble sets the exponent, so the 32 entries are summed from zero, hi
// before lo, and then added in fp32.  (Straight into the sums: 1.5 % of y not the nearest fp16 instead of 0.33 %; 28672 x 8192
// with 8 rows dense 37.6 against 40.4 us.  Sums of lo in registers of their own: 41.3 us.)
__device__ __forceinline__ void mma_group_two(float (*acc)[4], const unsigned* c0, const unsigned* c1, const unsigned* bh, const unsigned* bl)
{
    const MmaTiles t0(c0), t1(c1);
#pragma unroll
    for (int type = 0; type < 4; ++type) {
        float d[4] = {0.0f, 0.0f, 0.0f, 0.0f};
        mma_16816(d, t0.a[type][0], t0.a[type][1], t0.a[type][2], t0.a[type][3], bh[0], bh[1]);
        mma_16816(d, t1.a[type][0], t1.a[type][1], t1.a[type][2], t1.a[type][3], bh[2], bh[3]);
        mma_16816(d, t0.a[type][0], t0.a[type][1], t0.a[type][2], t0.a[type][3], bl[0], bl[1]);
        mma_16816(d, t1.a[type][0], t1.a[type][1], t1.a[type][2], t1.a[type][3], bl[2], bl[3]);
#pragma unroll
        for (int i = 0; i < 4; i += 2) unpack2(fadd2(pack2(acc[type][i], acc[type][i + 1]), pack2(d[i], d[i + 1])), acc[type][i], acc[type][i + 1]);
    }
}

// The sums of a group as the sums of its codes (see MmaTiles)
__device__ __forceinline__ void mma_uncumulate(float (*acc)[4])
{
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        acc[1][i] *= 0.0625f;
        acc[3][i] = (acc[3][i] - acc[2][i]) * 0.0625f;
    }
}

}  // namespace spqt

// The product on tensor cores: 4-bit (and widened 3-bit) codes as fp16 operands of mma.sync without a conversion.
// Included after spqt_gemv_device.cuh.
//
// A is the codes, 16 rows x 16 list entries per instruction; B is the multipliers a = x*scale of the 16 entries,
// 8 columns.  An fp16 word whose upper bits are zero IS a subnormal, its integer value times 2^-24, so a code becomes
// an operand with one mask.  The two halves of a register have to be the same rows of two neighbouring entries, which is what
// ldmatrix.trans delivers from blocks that lie row after row in shared memory: one register then holds bytes
// (2g, 2g+1) of entries 2t and 2t+1, i.e. four codes of each, and four operations make four operands of it.
//
// a = x*scale has up to 22 significant bits.  It goes in as two fp16 values, hi = fp16(a*c) and lo = fp16(a*c - hi),
// c a power of two that every warp keeps per batch row so that its largest |a*c| so far lies in 2^10 .. 2^15: hi + lo
// is then a*c exactly, or to 2^-36 of the largest entry, far below the fp32 accumulation.  When an entry exceeds the
// range, the sums are rescaled (a power of two: exact) and c changes.
//
// Per chunk of 32 entries x 128 rows the arithmetic is 84 warp instructions (4 ldmatrix, 64 masks and byte
// permutations, 16 mma) where the packed-FMA form takes 218 for one row and 64 more for every further one.
#pragma once

namespace spqt {

// c of a warp that has seen nothing but zeros: any entry exceeds the range
constexpr float kMmaNoScale = 0x1p100f;
constexpr float kMmaLimit = 32768.0f;

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

// The four tiles of one group: acc[type] += the operand of that type times B.  type 0 / 2: the low nibbles of the even /
// odd bytes; 1 / 3: the whole even / odd bytes (low + 16 * high, still a subnormal: one operation less than the high
// nibble alone, whose sum is recovered at the end as (byte - low) / 16).  TWO: B comes as hi and lo.
template <bool TWO>
__device__ __forceinline__ void mma_group(float (*acc)[4], const unsigned* c, const unsigned* bh, const unsigned* bl)
{
    constexpr unsigned kLow = 0x000f000fu, kByte = 0x00ff00ffu;
    unsigned d[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) d[i] = __byte_perm(c[i], 0u, 0x4341);   // the odd bytes
#pragma unroll
    for (int h = 0; h < (TWO ? 2 : 1); ++h) {
        const unsigned b0 = h ? bl[0] : bh[0], b1 = h ? bl[1] : bh[1];
        mma_16816(acc[0], c[0] & kLow, c[1] & kLow, c[2] & kLow, c[3] & kLow, b0, b1);
        mma_16816(acc[1], c[0] & kByte, c[1] & kByte, c[2] & kByte, c[3] & kByte, b0, b1);
        mma_16816(acc[2], d[0] & kLow, d[1] & kLow, d[2] & kLow, d[3] & kLow, b0, b1);
        mma_16816(acc[3], d[0], d[1], d[2], d[3], b0, b1);
    }
}

// The sums of a group as the sums of its codes (see mma_group)
__device__ __forceinline__ void mma_uncumulate(float (*acc)[4])
{
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        acc[1][i] = (acc[1][i] - acc[0][i]) * 0.0625f;
        acc[3][i] = (acc[3][i] - acc[2][i]) * 0.0625f;
    }
}

}  // namespace spqt

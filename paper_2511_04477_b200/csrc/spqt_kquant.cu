// The two-level format the paper's implementation builds on (Sec. 2: superblocks of 256 weights split
// into eight blocks of 32, 4-bit codes, a 6-bit scale and a 6-bit minimum per block, a 16-bit scale and
// minimum per superblock), in the zigzag arrangement of Sec. 4.1.2: a superblock is 256 consecutive ROWS
// of one column, superblocks are stored row-major over (block-row, column).  One 144-byte record per
// superblock: 128 bytes of codes (byte i = q_i | q_{i+128} << 4), the sixteen 6-bit fields sc_0..7,
// m_0..7 as a little-endian bit string (12 bytes), d and dmin as fp16.  Dequantized weight of row j of
// block i:  d*sc_i*q_j - dmin*m_i.  The paper fixes neither the rounding rule nor the bit arrangement;
// the rule implemented is stated at kq_pack_kernel, every step a single IEEE fp32 operation.
// Other code widths (Sec. 4.1.3: any width from 2 to 8 bits): the kernels are templates over BITS = 2, 4, 5, 6,
// 8; 2^BITS - 1 replaces 15 in the rule and only the code bytes of a record change -- 8 bits: byte i = q_i (256
// bytes, records of 272); 2 bits: byte i = q_i | q_{i+64} << 2 | q_{i+128} << 4 | q_{i+192} << 6 (64 bytes,
// records of 80); 5 and 6 bits: the low four bits as 4-bit codes, then a plane of the high bits q >> 4, one per
// row (bit j%8 of byte j/8) or two per row arranged like 2-bit codes (records of 176 and 208).
//
//   kq_pack_kernel   a thread converts two columns, a warp 64.
//   kq_gemv_kernel   one CTA or a cluster of S CTAs per block-row, 8 or 16 warps each; every warp has an equal part of the
//                    list (or of all columns) and streams it through its own ring of chunks of 16 records (cp.async: a
//                    record is one contiguous gather, metadata included).  The product on tensor cores (spqt_mma.cuh):
//                    records are an odd number of 16-byte pieces, so that ldmatrix.trans reads them as they lie; the
//                    eight columns of B are hi and lo of the multipliers of four blocks, a second set those of the other
//                    four.  Sums: warps through shared memory, CTAs through the cluster's, in a fixed order.
//                    What bounds it: the integer pipe in the loop (masks, shifts: 53 to 61 % busy over the whole call), the fixed
//                    cost of the call and of the list's launch before it, then latency: 12 to 16 warps per SM with 2 to 5
//                    chunks in flight each.  28672 x 4096 to 4 bits at 50 %, list included, takes 13.8 us (19.4 with packed
//                    FMAs, partial sums in global memory and chunks dealt in turn), 8192 x 8192 to 6 bits dense 14.3 us (20.4;
//                    55 MB), 28672 x 8192 to 4 bits dense 31.1 us.
//                    A multiplier x*(d*sc) is rounded to fp32 and goes in as two fp16 values, off by 2^-26 of the warp's
//                    largest at most (spqt_mma.cuh; their rounding and rescaling cost 2 to 3 %: 28672 x 8192 dense to 4 bits 34.4 -> 35.4 us).
#include <cstddef>

#include "spqt_common.cuh"

#include "spqt_gemv_device.cuh"
#include "spqt_mma.cuh"
#include "spqt_quantize.cuh"

namespace spqt {

constexpr int kKqG = 256;           // rows of a superblock
__host__ __device__ constexpr int kq_code_bytes(int bits) { return kKqG * bits / 8; }
__host__ __device__ constexpr int kq_rec_bytes(int bits) { return kq_code_bytes(bits) + 16; }
constexpr int kKqChunk = 16;        // list entries per chunk
constexpr int kKqMaxCluster = 8;    // the largest portable cluster
constexpr int kKqMaxSplit = 32;     // clusters of a block-row at most,
constexpr int kKqMaxShared = 64;    // and of all block-rows that have more than one (the workspace's size; the device holds 33 of 4 CTAs)

// ---------------------------------------------------------------- conversion
//   per block i:      lo_i = min(min_j w_j, 0),  step_i = (max_j w_j - lo_i) / 15,  neg_i = 0 - lo_i
//                     (zeros of either sign count as +0.0)
//   per superblock:   d = fp16(max_i step_i / 63),  dmin = fp16(max_i neg_i / 63)
//                     sc_i = min(rint(step_i / d), 63),  m_i = min(rint(neg_i / dmin), 63)   (0 if the divisor is 0)
//   per weight:       q_j = clamp(rint((w_j + dmin*m_i) / (d*sc_i)), 0, 15)                   (0 if d*sc_i == 0)
// (15 = 2^BITS - 1 for 4-bit codes; 3 and 255 for the other widths)
// A thread converts two neighbouring columns, two fp32 operations per instruction, reading W twice (the second time from
// L2): for the ranges of the blocks, then 4 rows of all eight blocks at a time for the codes.  Both are loops: unrolled over
// all 256 rows the code has 150 KB, and the warps wait for it (14336 x 4096 to 4 bits 141 against 82 us; with an IEEE division per
// weight and a column per warp 229 us).  The records of a warp's 64 columns meet in shared memory, a word of padding after
// each against bank conflicts.
constexpr int kKqPackWarps = 2;
template <int BITS, bool VEC>
__global__ void __launch_bounds__(kKqPackWarps * 32, 8)
kq_pack_kernel(const __half* W, int n, int ldw, uint8_t* records)
{
    constexpr int kTop = (1 << BITS) - 1, NCB = kq_code_bytes(BITS), REC = kq_rec_bytes(BITS), RW = REC / 4;
    __shared__ unsigned rec_sm[kKqPackWarps][64 * (RW + 1)];
    const int warp = threadIdx.x / 32, lane = threadIdx.x % 32;
    const int r = blockIdx.y, k0 = (blockIdx.x * kKqPackWarps + warp) * 64, k = k0 + 2 * lane;
    if (k0 >= n) return;
    unsigned* const mine = rec_sm[warp];
    const bool on0 = k < n, on1 = k + 1 < n;
    const __half* const src = W + (size_t)r * kKqG * ldw + k;
    auto load = [&](int i) -> __half2 {
        if (VEC) {                       // (n is even)
            const unsigned u = on0 ? *reinterpret_cast<const unsigned*>(src + (size_t)i * ldw) : 0u;
            return *reinterpret_cast<const __half2*>(&u);
        }
        return __halves2half2(on0 ? src[(size_t)i * ldw] : __half(0.0f), on1 ? src[(size_t)i * ldw + 1] : __half(0.0f));
    };
    // ---- ranges: exact in fp16
#pragma unroll 1
    for (int u = 0; u < 8; ++u) {
        __half2 lo2 = load(32 * u), hi2 = lo2;
#pragma unroll
        for (int j = 1; j < 32; ++j) {
            const __half2 v = load(32 * u + j);
            lo2 = __hmin2(lo2, v);
            hi2 = __hmax2(hi2, v);
        }
        mine[(2 * u) * 32 + lane] = *reinterpret_cast<const unsigned*>(&lo2);
        mine[(2 * u + 1) * 32 + lane] = *reinterpret_cast<const unsigned*>(&hi2);
    }
    float2 step[8], neg[8], step_max = make_float2(0.0f, 0.0f), neg_max = make_float2(0.0f, 0.0f);
#pragma unroll
    for (int u = 0; u < 8; ++u) {
        const unsigned l = mine[(2 * u) * 32 + lane], h = mine[(2 * u + 1) * 32 + lane];
        const float2 lo = __half22float2(*reinterpret_cast<const __half2*>(&l)), hi = __half22float2(*reinterpret_cast<const __half2*>(&h));
        auto range = [&](float lo, float hi, float& st, float& ng) {
            lo = __fadd_rn(fminf(lo, 0.0f), 0.0f);  // a zero of either sign counts as +0.0
            hi = __fadd_rn(hi, 0.0f);
            st = __fdiv_rn(__fsub_rn(hi, lo), (float)kTop);
            ng = __fsub_rn(0.0f, lo);
        };
        range(lo.x, hi.x, step[u].x, neg[u].x);
        range(lo.y, hi.y, step[u].y, neg[u].y);
        step_max = make_float2(fmaxf(step_max.x, step[u].x), fmaxf(step_max.y, step[u].y));
        neg_max = make_float2(fmaxf(neg_max.x, neg[u].x), fmaxf(neg_max.y, neg[u].y));
    }
    __syncwarp();                        // (the records take the place of the ranges)
    // ---- scales and minima
    const __half2 dh = __halves2half2(__float2half_rn(__fdiv_rn(step_max.x, 63.0f)), __float2half_rn(__fdiv_rn(step_max.y, 63.0f)));
    const __half2 mh = __halves2half2(__float2half_rn(__fdiv_rn(neg_max.x, 63.0f)), __float2half_rn(__fdiv_rn(neg_max.y, 63.0f)));
    const float2 df = __half22float2(dh), dminf = __half22float2(mh);
    const Divisor2 by_d(df), by_dmin(dminf);
    auto limited = [](float2 v, float top) { return make_float2(fminf(fmaxf(v.x, 0.0f), top), fminf(fmaxf(v.y, 0.0f), top)); };   // (0 for not-a-number)
    unsigned long long f64[2] = {0ull, 0ull};   // fields 0..9 and the low 4 bits of field 10
    unsigned f32[2] = {0u, 0u};                 // bits 64..95
    float2 offset[8];
    Divisor2 by[8];
#pragma unroll
    for (int u = 0; u < 8; ++u) {
        float2 ns = limited(by_d.quotient(step[u]), 63.0f), nm = limited(by_dmin.quotient(neg[u]), 63.0f);
        ns = make_float2(rintf(ns.x), rintf(ns.y));
        nm = make_float2(rintf(nm.x), rintf(nm.y));
        offset[u] = make_float2(__fmul_rn(dminf.x, nm.x), __fmul_rn(dminf.y, nm.y));
        by[u] = Divisor2(make_float2(__fmul_rn(df.x, ns.x), __fmul_rn(df.y, ns.y)));
        const unsigned sc[2] = {(unsigned)ns.x, (unsigned)ns.y}, mn[2] = {(unsigned)nm.x, (unsigned)nm.y};
#pragma unroll
        for (int c = 0; c < 2; ++c) {
            f64[c] |= (unsigned long long)sc[c] << (6 * u);
            const int b = 6 * (u + 8);
            if (b < 64) f64[c] |= (unsigned long long)mn[c] << b;
            if (b >= 64) f32[c] |= mn[c] << (b - 64);
            else if (b + 6 > 64) f32[c] |= mn[c] >> (64 - b);
        }
    }
    // ---- codes
    unsigned* const rec[2] = {mine + (2 * lane) * (RW + 1), mine + (2 * lane + 1) * (RW + 1)};
    unsigned bits5[2][BITS == 5 ? 8 : 1] = {};
#pragma unroll 1
    for (int i = 0; i < 8; ++i) {
        unsigned L[2][8];                // codes of rows 32u + 4i .. + 3, a byte each
#pragma unroll
        for (int u = 0; u < 8; ++u) {
            float2 t[4];
#pragma unroll
            for (int j = 0; j < 4; ++j)
                t[j] = round_to_low_bits(limited(by[u].quotient(add2(__half22float2(load(32 * u + 4 * i + j)), offset[u])), (float)kTop));
            L[0][u] = four_bytes(t[0].x, t[1].x, t[2].x, t[3].x);
            L[1][u] = four_bytes(t[0].y, t[1].y, t[2].y, t[3].y);
        }
#pragma unroll
        for (int c = 0; c < 2; ++c) {
            if (BITS == 8) {             // byte i = code of row i
#pragma unroll
                for (int u = 0; u < 8; ++u) rec[c][8 * u + i] = L[c][u];
            } else if (BITS == 2) {      // byte i = codes of rows i, i + 64, i + 128, i + 192
#pragma unroll
                for (int u = 0; u < 2; ++u) rec[c][8 * u + i] = L[c][u] | (L[c][u + 2] << 2) | (L[c][u + 4] << 4) | (L[c][u + 6] << 6);
            } else {                     // byte i = low four bits of rows i and i + 128, then the high bits
#pragma unroll
                for (int u = 0; u < 4; ++u) rec[c][8 * u + i] = (L[c][u] & 0x0f0f0f0fu) | ((L[c][u + 4] & 0x0f0f0f0fu) << 4);
                if (BITS == 6) {         // two per row, arranged like 2-bit codes
#pragma unroll
                    for (int u = 0; u < 2; ++u)
                        rec[c][32 + 8 * u + i] = ((L[c][u] >> 4) & 0x03030303u) | ((L[c][u + 2] >> 2) & 0x0c0c0c0cu) | (L[c][u + 4] & 0x30303030u) | ((L[c][u + 6] << 2) & 0xc0c0c0c0u);
                }
                if (BITS == 5) {         // one per row, bit j % 8 of byte j / 8: four bytes' bits meet in the product's top
#pragma unroll
                    for (int u = 0; u < 8; ++u)
                        bits5[c][BITS == 5 ? u : 0] |= (((((L[c][u] >> 4) & 0x01010101u) * 0x01020408u) >> 24) & 15u) << (4 * i);
                }
            }
        }
    }
    const unsigned dl = *reinterpret_cast<const unsigned*>(&dh), ml = *reinterpret_cast<const unsigned*>(&mh);
#pragma unroll
    for (int c = 0; c < 2; ++c) {
        if (BITS == 5) {
#pragma unroll
            for (int u = 0; u < 8; ++u) rec[c][32 + u] = bits5[c][BITS == 5 ? u : 0];
        }
        rec[c][NCB / 4] = (unsigned)f64[c];
        rec[c][NCB / 4 + 1] = (unsigned)(f64[c] >> 32);
        rec[c][NCB / 4 + 2] = f32[c];
        rec[c][NCB / 4 + 3] = __byte_perm(dl, ml, c == 0 ? 0x5410 : 0x7632);
    }
    __syncwarp();
    unsigned* const dst = reinterpret_cast<unsigned*>(records + ((size_t)r * n + k0) * REC);
    const int words = min(64, n - k0) * RW;
#pragma unroll 4
    for (int w = lane; w < words; w += 32) dst[w] = mine[w + w / RW];
}

template <int BITS>
static void launch_kq_pack(const __half* W, int m, int n, int ldw, uint8_t* records, cudaStream_t s)
{
    const dim3 grid((n + kKqPackWarps * 64 - 1) / (kKqPackWarps * 64), m / kKqG);
    const bool vec = aligned(W, 4) && ((ldw | n) & 1) == 0;   // pairs of columns as words
    auto kernel = vec ? kq_pack_kernel<BITS, true> : kq_pack_kernel<BITS, false>;
    kernel<<<grid, kKqPackWarps * 32, 0, s>>>(W, n, ldw, records);
}

// ---------------------------------------------------------------- GEMV

__host__ __device__ constexpr int kq_depth(int bits) { return bits == 2 ? 6 : bits <= 5 ? 4 : 3; }   // chunks in a warp's ring: 7.7 to 13 KB

template <int BITS, int NW>
struct KqSmem {
    struct Loop {
        alignas(16) unsigned char rec[NW][kq_depth(BITS)][kKqChunk * kq_rec_bytes(BITS)];
        alignas(16) unsigned short b[NW][32][8];      // operand B of a chunk: row e of set s (blocks 4s .. 4s+3) at 16s + e, hi and lo of each block
    };
    struct Sums {
        float red[NW][kKqG];
        float red_z[NW][8];
        int last;                                     // whether this cluster came last to the block-row
    };
    union Area {
        unsigned char loop[sizeof(Loop)];
        unsigned char sums[sizeof(Sums)];
    };
    alignas(16) unsigned char area[sizeof(Area)];
    alignas(16) uint64_t arrival;                      // first CTA of a cluster: the arrival of the other CTAs' sums, which lie behind
};

// with the sums of the k - 1 other CTAs of a cluster
template <int BITS, int NW>
constexpr int kq_smem_bytes(int k) { return (int)sizeof(KqSmem<BITS, NW>) + (k - 1) * kKqG * (int)sizeof(float); }

// The rotation that brings bit `from` of both halves to bit `to`.
__device__ __forceinline__ unsigned kq_rotate(unsigned v, int from, int to) { return __funnelshift_r(v, v, from - to); }

// acc[2*blk + o]: sums of rows 32*blk + 16*half + 2g + o, half = register / 2, over the 16 entries in stage st; columns
// 2*(blk % 4) and the next of B set blk / 4 are the block's multipliers.  What the sums are multiples of: kq_unit.
template <int BITS>
__device__ __forceinline__ void kq_multiply(float (*acc)[4], unsigned st, int lane, const unsigned* bb)
{
    constexpr int REC = kq_rec_bytes(BITS), NCB = kq_code_bytes(BITS), kGroups = BITS == 8 ? 8 : BITS == 2 ? 2 : 4;
    // records are an odd number of 16-byte pieces: the eight rows of a matrix lie in different banks
    const unsigned addr = st + (unsigned)((((lane >> 4) << 3) + (lane & 7)) * REC + ((lane >> 3) & 1) * 16);
    const int g = lane >> 2, t4 = lane & 3;
    auto product = [&](int blk, int o, const unsigned* a) { mma_16816(acc[2 * blk + o], a[0], a[1], a[2], a[3], bb[2 * (blk >> 2)], bb[2 * (blk >> 2) + 1]); };
    unsigned p[2][4];
    if (BITS == 6) {
        ldsm_x4_trans(addr + 128u, p[0]);
        ldsm_x4_trans(addr + 160u, p[1]);
    }
#pragma unroll
    for (int i = 0; i < kGroups; ++i) {
        unsigned c[4], d[4], a[4];
        ldsm_x4_trans(addr + 32u * i, c);
        if (BITS == 5) {
            // The plane's words of block i, then i + 4: entries 2t and 2t + 1 (+ 8) the halves of a word, read once for both rows of
            // the lane and rotated so that row 2g's bit lies above its nibble, at bit 4 or 8, and row 2g + 1's one place higher.
            // The odd bytes go one place up as well, and their sums count twice (kq_unit).  28672 x 8192 dense 64.4 -> 55.9 us, at
            // 50 % 36.6 -> 33.1 (bound by the integer pipe; a rotation and four shared loads for each row before).
#pragma unroll
            for (int j = 0; j < 2; ++j) {
                unsigned u[4];
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    const unsigned e = st + (unsigned)((2 * t4 + 8 * h) * REC + 128 + 4 * i + 16 * j);
                    const unsigned w0 = lds_u32(e), w1 = lds_u32(e + REC);
                    u[2 * h] = kq_rotate(__byte_perm(w0, w1, 0x5410), 2 * g, 4 + 4 * j);
                    u[2 * h + 1] = kq_rotate(__byte_perm(w0, w1, 0x7632), 2 * g, 4 + 4 * j);
                }
#pragma unroll
                for (int o = 0; o < 2; ++o) {
                    const unsigned nibble = 0x000f000fu << (4 * j + o), bit = 0x00100010u << (4 * j + o);
#pragma unroll
                    for (int q = 0; q < 4; ++q) a[q] = ((o ? c[q] >> 7 : c[q]) & nibble) | (u[q] & bit);
                    product(i + 4 * j, o, a);
                }
            }
            continue;
        }
#pragma unroll
        for (int q = 0; q < 4; ++q) d[q] = __byte_perm(c[q], 0u, 0x4341);   // the odd bytes
#pragma unroll
        for (int o = 0; o < 2; ++o) {
            const unsigned* const s = o ? d : c;
            if (BITS == 8) {
#pragma unroll
                for (int q = 0; q < 4; ++q) a[q] = o ? s[q] : s[q] & 0x00ff00ffu;
                product(i, o, a);
            } else if (BITS == 2) {
#pragma unroll
                for (int j = 0; j < 4; ++j) {
#pragma unroll
                    for (int q = 0; q < 4; ++q) a[q] = s[q] & (0x00030003u << (2 * j));
                    product(2 * j + i, o, a);
                }
            } else {
                unsigned hl[4], hh[4];               // the high bits of blocks i and i + 4, at bits 4 and 8 up
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    hl[q] = hh[q] = 0u;
                    if (BITS == 6) {
                        const unsigned w = p[i & 1][q], v = (o ? __byte_perm(w, 0u, 0x4341) : w) << (4 - 2 * (i >> 1));
                        hl[q] = v & 0x00300030u;
                        hh[q] = v & 0x03000300u;
                    }
                }
#pragma unroll
                for (int q = 0; q < 4; ++q) a[q] = (s[q] & 0x000f000fu) | hl[q];
                product(i, o, a);
#pragma unroll
                for (int q = 0; q < 4; ++q) a[q] = (s[q] & 0x00f000f0u) | hh[q];
                product(i + 4, o, a);
            }
        }
    }
}
// (o: of the row's place, see kq_multiply)
__host__ __device__ constexpr float kq_unit(int bits, int blk, int o)
{
    return bits == 8 ? 1.0f : bits == 2 ? (blk < 2 ? 1.0f : blk < 4 ? 0.25f : blk < 6 ? 0.0625f : 0.015625f) : (blk < 4 ? 1.0f : 0.0625f) * (bits == 5 && o ? 0.5f : 1.0f);
}

// idx == nullptr: the dense product (the list is 0, 1, .., n-1 and count is n).
template <int BITS, bool LIST, int NW>
__global__ void __launch_bounds__(NW * 32, NW == 8 ? 2 : 1)
kq_gemv_kernel(const uint8_t* __restrict__ records, int n, const __half* x, const int32_t* idx,
               const int32_t* count_ptr, __half* y, int splits, int clusters, unsigned* arrived, float* partial, int together)
{
    constexpr int REC = kq_rec_bytes(BITS), NCB = kq_code_bytes(BITS), PPR = REC / 16, CH = kKqChunk, D = kq_depth(BITS);
    constexpr int kPieces = CH * PPR, NC = (kPieces + 31) / 32;
    using Smem = KqSmem<BITS, NW>;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    Smem& sm = *reinterpret_cast<Smem*>(smem_raw);
    float* const xred = reinterpret_cast<float*>(smem_raw + sizeof(Smem));   // [S - 1][kKqG]
    typename Smem::Loop& lp = *reinterpret_cast<typename Smem::Loop*>(sm.area);
    typename Smem::Sums& su = *reinterpret_cast<typename Smem::Sums*>(sm.area);
    const int tid = threadIdx.x, lane = tid & 31, warp = __shfl_sync(0xffffffffu, tid >> 5, 0);
    const int e = lane & 15;
    const unsigned S = (unsigned)splits, T = (unsigned)clusters, rank = blockIdx.x % S, cluster = blockIdx.x / S, r = cluster / T;
    if (S > 1) {
        if (tid == 0) {
            mbar_init(&sm.arrival, 1);
            mbar_expect(&sm.arrival, (S - 1u) * kKqG * (unsigned)sizeof(float));
            mbar_publish();
        }
        __syncwarp();
        cluster_arrive();                // nobody may write to another CTA's shared memory before that CTA runs
    }

    const unsigned stage0 = smem_u32(&lp.rec[warp][0][0]);
    constexpr unsigned kStageBytes = CH * REC, kRing = D * kStageBytes;
    const unsigned b_base = smem_u32(&lp.b[warp][0][0]) + 16u * lane;
    const uint8_t* const row = records + (size_t)r * (size_t)n * REC;
    const unsigned short* const xg = reinterpret_cast<const unsigned short*>(x);

    // this warp's part of a list of `count` entries, in units of 8
    int first, end;
    auto take_part = [&](int count) {
        const unsigned units = (unsigned)(count + 7) >> 3, parts = T * S * NW, part = ((cluster - r * T) * S + rank) * NW + (unsigned)warp;
        first = 8 * (int)((unsigned long long)units * part / parts);
        end = min(8 * (int)((unsigned long long)units * (part + 1u) / parts), count);
    };
    if (!LIST) {                         // (the first records towards L2 while the previous kernel drains: a hint, see prefetch_l2)
        take_part(n);
        prefetch_l2(row + (size_t)first * REC, (size_t)max(min(end - first, (D - 1) * CH), 0) * REC, lane, 32);
    }
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");

    float nothing = 0.0f;                // what the sums of x*(dmin*m) begin with: not-a-number for a list without a length (see kListLost)
    if (LIST) {
        const int count = (int)ld_global_u32(count_ptr);
        nothing = not_a_number_if(count < 0, 0.0f);
        take_part(max(count, 0));
    }

    constexpr int kAhead = 2;            // (a third costs registers: 28672 x 4096 to 4 bits 13.2 against 12.8 us, to 8 bits 16.8 against 16.3)
    int coming[kAhead], ahead = first;   // list: the columns of the chunks the copies come to next
    auto fetch_ahead = [&](int d) {
        coming[d] = (int)ld_global_u32(idx + min(ahead + e, end - 1));
        ahead = ahead + CH >= end ? first : ahead + CH;
    };
    if (LIST && first < end) {
#pragma unroll
        for (int d = 0; d < kAhead; ++d) fetch_ahead(d);
    }
    unsigned xv[D];                      // the x values of the chunks in flight, the oldest first
#pragma unroll
    for (int i = 0; i < D; ++i) xv[i] = 0;
    int ipos = first;
    unsigned ri = 0;
    auto issue = [&]() {                 // the copies of the next chunk, if there is one
#pragma unroll
        for (int i = 0; i < D - 1; ++i) xv[i] = xv[i + 1];
        xv[D - 1] = 0u;
        if (ipos < end) {                // (past the end: the last entry again, with x = 0)
            const unsigned col = LIST ? (unsigned)coming[0] : (unsigned)min(ipos + e, end - 1);
            xv[D - 1] = ld_global_u16_if(ipos + e < end, xg + col);
            // (the chunk's records lie one after the other: one address instead of a shuffle and a product for every copy; 28672 x 8192
            // to 6 bits 50.0 -> 44.4 us, 5 bits 53.0 -> 51.0; to 4 bits 2 % slower)
            if (!LIST && BITS >= 5 && ipos + CH <= end) {
                const uint8_t* const src = row + ((size_t)(unsigned)ipos * REC + 16 * lane);
#pragma unroll
                for (int q = 0; q < NC; ++q)
                    if (kPieces % 32 == 0 || q * 32 + lane < kPieces) cp_async_16_l2_64(stage0 + ri + 16u * (q * 32 + lane), src + 512 * q);
            } else {
#pragma unroll
                for (int q = 0; q < NC; ++q) {
                    const int p = q * 32 + lane;
                    const unsigned cu = __shfl_sync(0xffffffffu, col, (p / PPR) & 15);
                    if (kPieces % 32 == 0 || p < kPieces) cp_async_16_l2_64(stage0 + ri + 16u * p, row + ((size_t)cu * REC + (p % PPR) * 16));
                }
            }
            ri = ri + kStageBytes == kRing ? 0u : ri + kStageBytes;
            ipos += CH;
            if (LIST) {
#pragma unroll
                for (int i = 0; i < kAhead - 1; ++i) coming[i] = coming[i + 1];
                fetch_ahead(kAhead - 1);
            }
        }
        cp_async_commit();
    };
#pragma unroll 1
    for (int d = 0; d < D - 1; ++d) issue();

    // While chunk i is multiplied, chunk i + 1 is prepared: lane 16s + e decodes the fields of blocks 4s .. 4s+3 of entry e,
    // a = x*(d*sc) (d*sc exact in fp32) left as hi and lo, and x*(dmin*m), two blocks per instruction (28672 x 8192 to 4 bits dense
    // 34.2 -> 31.2 us: the loop is bound by issue, 390 instructions a chunk before, a fifth of them here).
    float acc[16][4];
#pragma unroll
    for (int i = 0; i < 64; ++i) acc[i >> 2][i & 3] = 0.0f;
    float scale = kMmaNoScale, regain = 1.0f;
    unsigned long long zl[2] = {pack2(nothing, nothing), pack2(nothing, nothing)}, zn[2] = {0ull, 0ull}, am[2], pm[2];   // pairs of blocks
    auto prepare = [&](unsigned st, unsigned xb) -> bool {
        const uint4 f = lds_v4(st + (unsigned)(e * REC + NCB));
        const unsigned sc = lane < 16 ? f.x : __funnelshift_r(f.x, f.y, 24), mn = lane < 16 ? __funnelshift_r(f.y, f.z, 16) : f.z >> 8;
        const float xf = __half2float(__ushort_as_half((unsigned short)xb));
        const float df = __half2float(__ushort_as_half((unsigned short)(f.w & 0xffffu))), mf = __half2float(__ushort_as_half((unsigned short)(f.w >> 16)));
        const unsigned long long x2 = pack2(xf, xf), d2 = pack2(df, df), m2 = pack2(mf, mf), scale2 = pack2(scale, scale), bias = pack2(-8388608.0f, -8388608.0f);
        auto fields = [&](unsigned v, int j) {   // two of them as floats
            return fadd2(pack2(__uint_as_float(((v >> (12 * j)) & 63u) | 0x4b000000u), __uint_as_float(((v >> (12 * j + 6)) & 63u) | 0x4b000000u)), bias);
        };
        float top = 0.0f;
#pragma unroll
        for (int j = 0; j < 2; ++j) {
            am[j] = fmul2(x2, fmul2(d2, fields(sc, j)));
            zn[j] = fmul2(x2, fmul2(m2, fields(mn, j)));
            pm[j] = fmul2(am[j], scale2);    // a power of two
            float a, b;
            unpack2(pm[j], a, b);
            top = fmaxf(top, fmaxf(fabsf(a), fabsf(b)));
        }
        return top > kMmaLimit;
    };
    // a larger entry than the range holds: a new scale; the sums follow once chunk i is in them
    auto rescale = [&]() {
        unsigned m = 0;
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            float v[2];
            unpack2(am[j >> 1], v[0], v[1]);
            const unsigned bits = __float_as_uint(v[j & 1]) & 0x7fffffffu;
            m = max(m, bits < 0x7f800000u ? bits : 0u);   // finite ones
        }
        m = __reduce_max_sync(0xffffffffu, m);
        if (__uint_as_float(m) * scale > kMmaLimit) {
            const float next = __uint_as_float((266u - (m >> 23)) << 23);   // m goes to 2^12 .. 2^13
            regain = next * power_of_two_inverse(scale);
            scale = next;
#pragma unroll
            for (int j = 0; j < 2; ++j) pm[j] = fmul2(am[j], pack2(next, next));
        }
    };
    auto leave = [&]() {
        unsigned w[4];
#pragma unroll
        for (int j = 0; j < 2; ++j) {
            float v0, v1;
            unpack2(to_halves2(pm[j]), v0, v1);
            const __half2 h = __floats2half2_rn(v0, v1);
            const float2 hf = __half22float2(h);
            unsigned long long rest = pm[j];
            ffma2(rest, pack2(hf.x, hf.y), pack2(-1.0f, -1.0f));
            unpack2(rest, v0, v1);
            const __half2 l = __floats2half2_rn(v0, v1);
            w[2 * j] = __byte_perm(*reinterpret_cast<const unsigned*>(&h), *reinterpret_cast<const unsigned*>(&l), 0x5410);
            w[2 * j + 1] = __byte_perm(*reinterpret_cast<const unsigned*>(&h), *reinterpret_cast<const unsigned*>(&l), 0x7632);
        }
        sts_v4(b_base, make_uint4(w[0], w[1], w[2], w[3]));
    };
    unsigned rc = 0;
    if (first < end) {
        cp_async_wait<D - 2>();
        __syncwarp();
        if (__any_sync(0xffffffffu, prepare(stage0, xv[1]))) rescale();
        leave();
        regain = 1.0f;                   // (there is nothing in the sums yet)
        __syncwarp();
    }
#pragma unroll 1
    for (int pos = first; pos < end; pos += CH) {
        issue();
        const unsigned rn = rc + kStageBytes == kRing ? 0u : rc + kStageBytes;
        cp_async_wait<D - 2>();
        __syncwarp();
        unsigned bb[4];
        ldsm_x4_trans(b_base, bb);
#pragma unroll
        for (int j = 0; j < 2; ++j) zl[j] = fadd2(zl[j], zn[j]);
        bool over = false;
        if (BITS != 5) over = prepare(stage0 + rn, xv[1]);
        __syncwarp();                    // (B is in registers: its place is free)
        kq_multiply<BITS>(acc, stage0 + rc, lane, bb);
        if (BITS == 5) over = prepare(stage0 + rn, xv[1]);   // (later: its results would not fit the registers beside the product)
        if (__any_sync(0xffffffffu, over)) rescale();
        leave();
        if (regain != 1.0f) {
#pragma unroll
            for (int i = 0; i < 32; ++i) rescale_sums(acc[i >> 1][2 * (i & 1)], acc[i >> 1][2 * (i & 1) + 1], regain);
            regain = 1.0f;
        }
        __syncwarp();                    // every lane is done with this chunk's stage
        rc = rn;
    }
    cp_async_wait<0>();
    __syncthreads();                     // (the sums take the place of the rings)

    // ---- sums: lane (g, t4) has those of blocks t4 and t4 + 4
    const float unit = 0x1p24f * power_of_two_inverse(scale);
    const int g = lane >> 2, t4 = lane & 3;
#pragma unroll
    for (int blk = 0; blk < 8; ++blk)
        if ((blk & 3) == t4) {
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const int o = i & 1, half = i >> 1;
                su.red[warp][32 * blk + 16 * half + 2 * g + o] = (acc[2 * blk + o][2 * half] + acc[2 * blk + o][2 * half + 1]) * (unit * kq_unit(BITS, blk, o));   // hi + lo
            }
        }
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        float v[2];
        unpack2(zl[j >> 1], v[0], v[1]);
        float z = v[j & 1];
#pragma unroll
        for (int o = 8; o > 0; o >>= 1) z += __shfl_xor_sync(0xffffffffu, z, o);
        if (e == 0) su.red_z[warp][(lane >> 4) * 4 + j] = z;
    }
    __syncthreads();
    float total = 0.0f;                  // thread j < 256: row j
    if (tid < kKqG) {
        float z = 0.0f;
#pragma unroll
        for (int w = 0; w < NW; ++w) {
            total += su.red[w][tid];
            z += su.red_z[w][tid >> 5];
        }
        total -= z;
    }
    if (S > 1) {
        // the other CTAs send their sums to the first one's shared memory, which counts the bytes and adds them in CTA order (see
        // gemv_kernel; 8192 x 8192 to 6 bits dense 17.1 -> 16.5 us)
        cluster_wait();                  // (every CTA of the cluster runs)
        if (rank != 0) {
            if (tid < kKqG) st_async_f32(cluster_map(smem_u32(xred + (rank - 1u) * kKqG + tid), 0u), total, cluster_map(smem_u32(&sm.arrival), 0u));
            if (together) cluster_leave_together();
            return;
        }
        if (tid >= kKqG) {
            cluster_sent();              // (there are barriers of the CTA to come)
        } else {
            if (!mbar_wait_cluster(&sm.arrival, 0u)) total = __int_as_float(0x7fffffff);
#pragma unroll
            for (unsigned q = 0; q < kKqMaxCluster - 1; ++q)
                if (q < S - 1u) total += xred[q * kKqG + tid];
        }
    }
    if (T > 1) {
        // The cluster that comes last to the block-row adds the clusters' sums in order, and leaves the counter and the sums at
        // zero: calls of another shape may have counters where this one has sums.
        float* const row_sums = partial + (size_t)r * T * kKqG;
        if (tid < kKqG) __stcg(row_sums + (cluster - r * T) * kKqG + tid, total);
        __threadfence();
        __syncthreads();
        if (tid == 0) {
            su.last = atomicAdd(arrived + r, 1u) == T - 1u;
            if (su.last) arrived[r] = 0u;
        }
        __syncthreads();
        if (!su.last) return;
        __threadfence();
        if (tid < kKqG) {
            total = 0.0f;
            for (unsigned t = 0; t < T; ++t) total += __ldcg(row_sums + t * kKqG + tid);
            for (unsigned t = 0; t < T; ++t) __stcg(row_sums + t * kKqG + tid, 0.0f);   // (a loop of its own: the loads go together)
        }
    }
    if (tid < kKqG) y[(size_t)r * kKqG + tid] = __float2half_rn(total);
}

// ---------------------------------------------------------------- host side

inline size_t kq_header_bytes(int R) { return (((size_t)R * 4 + 255) / 256) * 256; }
// (never more than a caller who kept the size of the earlier form, 33 KB per block-row, has)
inline size_t kq_workspace_bytes(int R)
{
    return kq_header_bytes(R) + (size_t)(R == 1 ? kKqMaxSplit : kKqMaxShared) * kKqG * sizeof(float);
}

static spqt_status kq_shape(int m, int n)
{
    if (m <= 0 || n <= 0) return SPQT_ERR_INVALID_ARG;
    if (m % kKqG != 0) return SPQT_ERR_UNSUPPORTED;
    if (m / kKqG > 65535) return SPQT_ERR_UNSUPPORTED;
    return SPQT_OK;
}

// How many clusters of k CTAs the device holds at once with `smem` bytes each (asked once per kernel, cluster size and device).
template <int BITS, bool LIST, int NW>
static int kq_max_clusters(int k, int smem, bool alone, int sms, int dev)
{
    static int known[64][2][kKqMaxCluster + 1] = {};
    int& at_once = known[dev][alone ? 1 : 0][k];
    if (at_once == 0) {
        cudaLaunchAttribute attr[1];
        attr[0].id = cudaLaunchAttributeClusterDimension;
        attr[0].val.clusterDim.x = k;
        attr[0].val.clusterDim.y = 1;
        attr[0].val.clusterDim.z = 1;
        cudaLaunchConfig_t cfg = {};
        cfg.gridDim = dim3((unsigned)(k * 2 * sms));
        cfg.blockDim = dim3(NW * 32);
        cfg.dynamicSmemBytes = smem;
        cfg.attrs = attr;
        cfg.numAttrs = 1;
        int can = 0;
        if (cudaOccupancyMaxActiveClusters(&can, kq_gemv_kernel<BITS, LIST, NW>, &cfg) != cudaSuccess) (void)cudaGetLastError();
        at_once = can > 0 ? can : 1;
    }
    return at_once;
}

template <int BITS, bool LIST>
static spqt_status kq_launch_mode(const void* records, int R, int n, const void* x, const int32_t* idx, const int32_t* count, void* y, void* workspace, cudaStream_t s)
{
    constexpr int kAlone = 120 * 1024;   // shared memory that keeps a second CTA of 8 warps off the SM
    // (8-bit codes: two CTAs per SM have memory for the sums of a cluster of seven)
    constexpr int kMostTwo = kq_smem_bytes<BITS, 8>(kKqMaxCluster) <= 115712 ? kKqMaxCluster : kKqMaxCluster - 1;
    constexpr int kSmem = kq_smem_bytes<BITS, 8>(kMostTwo), kSmem16 = kq_smem_bytes<BITS, 16>(kKqMaxCluster);
    static_assert(kSmem <= 115712 && kSmem16 <= 232448, "two CTAs of 8 warps per SM, or one of 16");
    static_assert(kq_smem_bytes<BITS, 8>(kKqMaxCluster) <= kAlone, "any cluster with an SM for each CTA");
    static bool configured[64] = {};
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return SPQT_ERR_CUDA;
    if (!configured[dev]) {
        if (cudaFuncSetAttribute(kq_gemv_kernel<BITS, LIST, 8>, cudaFuncAttributeMaxDynamicSharedMemorySize, kAlone) != cudaSuccess ||
            cudaFuncSetAttribute(kq_gemv_kernel<BITS, LIST, 16>, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmem16) != cudaSuccess)
            return SPQT_ERR_CUDA;
        configured[dev] = true;
    }
    const int sms = sm_count();
    if (sms <= 0) return SPQT_ERR_CUDA;
    // CTAs per block-row: the largest cluster of which all are resident at once with one CTA per SM, or, if more than twice as many
    // fit with two CTAs per SM (or four instead of two), that one (at n = 8192 to 4 bits: 9216 rows 7 instead of 3 10 % faster,
    // 11264 rows 6 instead of 2 13 %; to 6 bits 8192 rows dense 17.3 us on 4, 18.2 on 8); a
    // CTA has 128 columns at least, 512 where two share an SM.  "Resident" leaves places for four more CTAs: the previous
    // launch's leave SM by SM (7168 x 4096 on 5, of which the device holds just 56 clusters, 27 % slower than on 2; 23552 x
    // 1024 on 3, of 93, 40 % slower than on 1).  One CTA has 16 warps if it has an SM to itself, from n = 2048 on (25600 x 1024 8 %
    // faster with 8).  With few block-rows of a long x several clusters of 4 CTAs of 16 warps, so that more SMs fetch, if that are
    // half as many CTAs again (the sums of a block-row then meet in global memory, 1.5 us: dense 1024 x 28672 to 8 bits, 31 MB,
    // 21.0 us on 32 CTAs of 8 warps, 12.0 on 128 of 16; at n = 8192 clusters of 8 are 8 to 16 % faster, at 14336 8 to 22 % slower).
    // Powers of two with an SM for each CTA fit neighbouring SMs without (18944 x 8192 to 6 bits dense 34.7 us on 3, 25.7 on 2, of
    // which the device holds 74); with two per SM, and the CTAs of a cluster leaving together, odd ones take most of what the device holds
    // (of 56 clusters of five, 6 bits dense n = 2560 on 52 / 53 / 54 9.4 / 9.8 / 10.4 us, 10.5 on 4; 4 bits 7.3 / 8.3 / 9.4, 7.7 on 4; n = 14336
    // 6 bits 35.8 / 36.0 / 37.2, 42.5 on 4; 36 of 37 of seven n = 8192 12.3, 13.1 on 6; of 93 of three n = 2048 dense on 88 / 90 9.0 / 9.9, 10.3
    // on 1, with the list 7.65 / 8.75, 8.3 on 1; n = 8192 dense on 90 25.2, 31.5 on 1).
    auto resident = [&](int k, bool per_sm) {
        const int most = kq_max_clusters<BITS, LIST, 8>(k, per_sm ? kAlone : kSmem, per_sm, sms, dev);
        if (per_sm && (k & (k - 1)) == 0) return R <= most;
        const int percent = k == 7 ? 98 : k == 5 ? (n < 8192 ? 93 : 95) : (n < 4096 ? 95 : 97);
        if (!per_sm && (k & 1) != 0 && 100 * R > percent * most) return false;
        return k * (most - R) >= 4;
    };
    int one = 1, two = 1, T = 1;         // CTAs per block-row with one and with two CTAs per SM
    for (int k = 2; k <= kKqMaxCluster; ++k) {
        if (n >= 128 * k && resident(k, true)) one = k;
        if (k > 2 && k <= kMostTwo && n >= 512 * k && resident(k, false)) two = k;
    }
    int S = two > 2 * one || (one < 3 && two >= 4) ? two : one;
    const bool alone = S > 1 && R <= kq_max_clusters<BITS, LIST, 8>(S, kAlone, true, sms, dev);
    bool wide = S == 1 && R <= sms && n >= 2048;
    if (alone && n >= 1024 * S) wide = R <= kq_max_clusters<BITS, LIST, 16>(S, kSmem16, true, sms, dev);
    if (alone && n >= 12288) {
        int t = kq_max_clusters<BITS, LIST, 16>(4, kSmem16, true, sms, dev) / R;
        t = t < n / 1792 ? t : n / 1792;
        t = t < kKqMaxSplit ? t : kKqMaxSplit;
        t = t < kKqMaxShared / R ? t : kKqMaxShared / R;
        if (8 * t >= 3 * S && t > 1) {
            S = 4;
            T = t;
            wide = true;
        }
    }
    // (see cluster_leave_together)
    const int together = !wide && S > 1 && 100 * R > 91 * kq_max_clusters<BITS, LIST, 8>(S, alone ? kAlone : kSmem, alone, sms, dev);
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)S * (unsigned)T * (unsigned)R);
    cfg.blockDim = dim3(wide ? 512 : 256);
    cfg.dynamicSmemBytes = wide ? kSmem16 : alone ? kAlone : kSmem;
    cfg.stream = s;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    attr[1].id = cudaLaunchAttributeClusterDimension;
    attr[1].val.clusterDim.x = S;
    attr[1].val.clusterDim.y = 1;
    attr[1].val.clusterDim.z = 1;
    cfg.attrs = g_no_pdl ? attr + 1 : attr;
    cfg.numAttrs = (g_no_pdl ? 0 : 1) + (S > 1 ? 1 : 0);
    auto kernel = wide ? kq_gemv_kernel<BITS, LIST, 16> : kq_gemv_kernel<BITS, LIST, 8>;
    const cudaError_t err = cudaLaunchKernelEx(&cfg, kernel, static_cast<const uint8_t*>(records), n, static_cast<const __half*>(x), idx, count,
                                               static_cast<__half*>(y), S, T, static_cast<unsigned*>(workspace),
                                               reinterpret_cast<float*>(static_cast<char*>(workspace) + kq_header_bytes(R)), together);
    count_launch();
    return (err == cudaSuccess && cudaGetLastError() == cudaSuccess) ? SPQT_OK : SPQT_ERR_CUDA;
}

template <int BITS>
static spqt_status kq_launch(const void* records, int m, int n, const void* x, const int32_t* idx, const int32_t* count,
                             void* y, void* workspace, size_t ws_bytes, void* stream)
{
    if (!records || !x || !y || !workspace) return SPQT_ERR_INVALID_ARG;
    const spqt_status st = kq_shape(m, n);
    if (st != SPQT_OK) return st;
    if (!aligned(records, 16) || !aligned(x, 2) || !aligned(y, 2) || !aligned(workspace, 16) ||
        (idx && (!aligned(idx, 4) || !aligned(count, 4))))
        return SPQT_ERR_ALIGNMENT;
    const int R = m / kKqG;
    if (ws_bytes < kq_workspace_bytes(R)) return SPQT_ERR_WORKSPACE;
    const cudaStream_t s = static_cast<cudaStream_t>(stream);
    return idx ? kq_launch_mode<BITS, true>(records, R, n, x, idx, count, y, workspace, s) : kq_launch_mode<BITS, false>(records, R, n, x, idx, count, y, workspace, s);
}

}  // namespace spqt

extern "C" {

static bool kq_bits_ok(int bits) { return bits == 2 || bits == 4 || bits == 5 || bits == 6 || bits == 8; }

spqt_status spqt_kqw_packed_sizes(int m, int n, int bits, size_t* records_bytes, size_t* workspace_bytes)
{
    const spqt_status st = spqt::kq_shape(m, n);
    if (st != SPQT_OK) return st;
    if (!kq_bits_ok(bits)) return SPQT_ERR_UNSUPPORTED;
    if (records_bytes) *records_bytes = (size_t)(m / spqt::kKqG) * (size_t)n * spqt::kq_rec_bytes(bits);
    if (workspace_bytes) *workspace_bytes = spqt::kq_workspace_bytes(m / spqt::kKqG);
    return SPQT_OK;
}

spqt_status spqt_kqw_pack(const void* W, int m, int n, int ldw, int bits, void* records, void* stream)
{
    if (!W || !records) return SPQT_ERR_INVALID_ARG;
    const spqt_status st = spqt::kq_shape(m, n);
    if (st != SPQT_OK) return st;
    if (!kq_bits_ok(bits)) return SPQT_ERR_UNSUPPORTED;
    if (ldw < n) return SPQT_ERR_INVALID_ARG;
    if (!spqt::aligned(W, 2) || !spqt::aligned(records, 16)) return SPQT_ERR_ALIGNMENT;
    const cudaStream_t st_ = static_cast<cudaStream_t>(stream);
    const __half* w = static_cast<const __half*>(W);
    uint8_t* rec = static_cast<uint8_t*>(records);
    if (bits == 2) spqt::launch_kq_pack<2>(w, m, n, ldw, rec, st_);
    else if (bits == 4) spqt::launch_kq_pack<4>(w, m, n, ldw, rec, st_);
    else if (bits == 5) spqt::launch_kq_pack<5>(w, m, n, ldw, rec, st_);
    else if (bits == 6) spqt::launch_kq_pack<6>(w, m, n, ldw, rec, st_);
    else spqt::launch_kq_pack<8>(w, m, n, ldw, rec, st_);
    spqt::count_launch();
    return cudaGetLastError() == cudaSuccess ? SPQT_OK : SPQT_ERR_CUDA;
}

static spqt_status kq_launch_bits(int bits, const void* records, int m, int n, const void* x, const int32_t* idx,
                                  const int32_t* count, void* y, void* workspace, size_t workspace_bytes, void* stream)
{
    if (bits == 2) return spqt::kq_launch<2>(records, m, n, x, idx, count, y, workspace, workspace_bytes, stream);
    if (bits == 4) return spqt::kq_launch<4>(records, m, n, x, idx, count, y, workspace, workspace_bytes, stream);
    if (bits == 5) return spqt::kq_launch<5>(records, m, n, x, idx, count, y, workspace, workspace_bytes, stream);
    if (bits == 6) return spqt::kq_launch<6>(records, m, n, x, idx, count, y, workspace, workspace_bytes, stream);
    if (bits == 8) return spqt::kq_launch<8>(records, m, n, x, idx, count, y, workspace, workspace_bytes, stream);
    return SPQT_ERR_UNSUPPORTED;
}

spqt_status spqt_kqw_sparse_gemv(const void* records, int m, int n, int bits, const void* x, const int32_t* idx,
                                 const int32_t* count, void* y, void* workspace, size_t workspace_bytes, void* stream)
{
    if (!idx || !count) return SPQT_ERR_INVALID_ARG;
    return kq_launch_bits(bits, records, m, n, x, idx, count, y, workspace, workspace_bytes, stream);
}

spqt_status spqt_kqw_dense_gemv(const void* records, int m, int n, int bits, const void* x, void* y, void* workspace,
                                size_t workspace_bytes, void* stream)
{
    return kq_launch_bits(bits, records, m, n, x, nullptr, nullptr, y, workspace, workspace_bytes, stream);
}

spqt_status spqt_kq_packed_sizes(int m, int n, size_t* records_bytes, size_t* workspace_bytes)
{
    return spqt_kqw_packed_sizes(m, n, 4, records_bytes, workspace_bytes);
}

spqt_status spqt_kq_pack(const void* W, int m, int n, int ldw, void* records, void* stream)
{
    return spqt_kqw_pack(W, m, n, ldw, 4, records, stream);
}

spqt_status spqt_kq_sparse_gemv(const void* records, int m, int n, const void* x, const int32_t* idx, const int32_t* count,
                                void* y, void* workspace, size_t workspace_bytes, void* stream)
{
    return spqt_kqw_sparse_gemv(records, m, n, 4, x, idx, count, y, workspace, workspace_bytes, stream);
}

spqt_status spqt_kq_dense_gemv(const void* records, int m, int n, const void* x, void* y, void* workspace,
                               size_t workspace_bytes, void* stream)
{
    return spqt_kqw_dense_gemv(records, m, n, 4, x, y, workspace, workspace_bytes, stream);
}

}  // extern "C"

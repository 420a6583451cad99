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
// row (bit j%8 of byte j/8) or two per row arranged like 2-bit codes (records of 176 and 208).  The arithmetic of
// the 2- and 8-bit codes and of the high planes sums cumulative values (per 16-bit half-word the value of its
// first code and of both codes together; per byte of single bits its low 1, 2, .. 8 bits: the cumulative form of
// the main kernel) and takes the differences at the end.
//
//   kq_pack_kernel   a thread converts two columns, a warp 64.
//   kq_gemv_kernel   grid (S, R): CTA (s, r) takes the s-th of S slices of the index list (or of all
//                    columns) for block-row r; its 8 warps take the slice's chunks of 16 entries in turn,
//                    two record buffers per warp (cp.async: a record is one contiguous gather of 144 bytes,
//                    metadata included).  Lanes e and e+16 decode the fields of entry e and write the packed
//                    multiplier pairs of its four lane groups; lane t of a 16-lane half owns rows 8t..8t+7
//                    and 128+8t..128+8t+7 of the entry's superblock (blocks t/4 and 4+t/4: one multiplier
//                    pair covers both).  Conversion-free dequantization as in the main kernel.  Partial
//                    sums: warp -> CTA (shared memory) -> block-row (fp32 partials in the workspace,
//                    arrive-only counter, the last CTA adds them in slice order: bit-reproducible).
#include <cstddef>

#include "spqt_common.cuh"

#include "spqt_gemv_device.cuh"
#include "spqt_quantize.cuh"

namespace spqt {

constexpr int kKqG = 256;           // rows of a superblock
__host__ __device__ constexpr int kq_code_bytes(int bits) { return kKqG * bits / 8; }
__host__ __device__ constexpr int kq_rec_bytes(int bits) { return kq_code_bytes(bits) + 16; }
__host__ __device__ constexpr int kq_ctas_per_sm(int bits) { return bits >= 5 ? 2 : 3; }   // (registers of a second accumulator set; shared memory of the record buffers)
constexpr int kKqWarps = 8;
constexpr int kKqThreads = kKqWarps * 32;
constexpr int kKqChunk = 16;        // list entries per chunk
constexpr int kKqMaxSplit = 32;     // slices per block-row at most

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

template <int BITS>
struct KqSmem {
    alignas(16) unsigned char rec[kKqWarps][2][kKqChunk * kq_rec_bytes(BITS)];  // two record buffers per warp
    alignas(16) float mult[kKqWarps][kKqChunk][4][4];               // per entry and lane group: two packed multiplier pairs
    alignas(16) float red[kKqWarps][kKqG];
    float red_z[kKqWarps][8];
    int last;
};

// 6-bit field f of the 96-bit string w0 | w1 << 32 | w2 << 64
__device__ __forceinline__ unsigned kq_field(unsigned w0, unsigned w1, unsigned w2, int f)
{
    const int b = 6 * f, word = b >> 5;
    const unsigned lo = word == 0 ? w0 : (word == 1 ? w1 : w2);
    const unsigned hi = word == 0 ? w1 : (word == 1 ? w2 : 0u);
    return __funnelshift_r(lo, hi, b & 31) & 63u;
}

// idx == nullptr: the dense product (the list is 0, 1, .., n-1 and count is n).
template <int BITS>
__global__ void __launch_bounds__(kKqThreads, kq_ctas_per_sm(BITS))
kq_gemv_kernel(const uint8_t* __restrict__ records, int n, const __half* __restrict__ x,
               const int32_t* __restrict__ idx, const int32_t* __restrict__ count_ptr,
               __half* __restrict__ y, float* __restrict__ partials, int* __restrict__ counters)
{
    constexpr int CH = kKqChunk, G = kKqG;
    constexpr int REC = kq_rec_bytes(BITS), NCB = kq_code_bytes(BITS), PPR = REC / 16;
    constexpr int NP = CH * REC / 16;            // 16-byte pieces of a chunk
    constexpr int NC = (NP + 31) / 32;           // copies per lane and chunk
    extern __shared__ __align__(16) unsigned char kq_raw[];
    KqSmem<BITS>& sm = *reinterpret_cast<KqSmem<BITS>*>(kq_raw);
    const int tid = threadIdx.x, lane = tid & 31;
    const int warp = __shfl_sync(0xffffffffu, tid >> 5, 0);
    const int s = blockIdx.x, S = gridDim.x, r = blockIdx.y;
    const int half = lane >> 4, t = lane & 15;   // arithmetic: entry of the step, rows 8t.. and 128+8t..

    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");

    const int count = idx ? __ldg(count_ptr) : n;
    const int lo = (int)(((long long)s * count) / S), hi = (int)(((long long)(s + 1) * count) / S);
    const uint8_t* row_rec = records + (size_t)r * (size_t)n * REC;
    const unsigned rbuf = smem_u32(&sm.rec[warp][0][0]);
    const unsigned mbuf = smem_u32(&sm.mult[warp][0][0][0]);
    constexpr unsigned kBufBytes = CH * REC;
    const unsigned short* xb = reinterpret_cast<const unsigned short*>(x);

    unsigned long long acc[8];
#pragma unroll
    for (int i = 0; i < 8; ++i) acc[i] = 0ull;
    constexpr bool kHigh = BITS == 5 || BITS == 6;   // a second plane with the bits above the low four
    unsigned long long acch[kHigh ? 8 : 1];          // its sums (cumulative, see the step), same rows as acc
#pragma unroll
    for (int i = 0; i < (kHigh ? 8 : 1); ++i) acch[i] = 0ull;
    float zl[4] = {0.0f, 0.0f, 0.0f, 0.0f};      // x*dmin*m of blocks 4*half .. 4*half+3

    // column of the entry lanes e and e+16 hold in the chunk at list position pos (past the end: the last entry again)
    auto column_at = [&](int pos) -> int {
        const int e = min(pos + t, hi - 1);
        return idx ? __ldg(idx + e) : e;
    };
    auto copy_records = [&](int col, unsigned dst) {
#pragma unroll
        for (int q = 0; q < NC; ++q) {
            const int p = q * 32 + lane;
            const int e = p / PPR, part = p - PPR * e;
            const int cu = __shfl_sync(0xffffffffu, col, e & 15);
            if (p < NP) cp_async_16_l2_64(dst + (unsigned)(e * REC + part * 16), row_rec + (size_t)cu * REC + part * 16);
        }
        cp_async_commit();
    };

    const int first = lo + warp * CH, stride = kKqWarps * CH;
    if (first < hi) {
        int col = column_at(first);
        copy_records(col, rbuf);
        int col_next = first + stride < hi ? column_at(first + stride) : 0;
        unsigned short xv = (first + t < hi) ? __ldg(xb + col) : (unsigned short)0;
        unsigned cur = 0;
        for (int pos = first; pos < hi; pos += stride) {
            const bool more = pos + stride < hi;
            if (more) copy_records(col_next, rbuf + (cur == 0u ? kBufBytes : 0u));
            else cp_async_commit();
            const int col_after = pos + 2 * stride < hi ? column_at(pos + 2 * stride) : 0;
            const unsigned short xv_next = (more && pos + stride + t < hi) ? __ldg(xb + col_next) : (unsigned short)0;
            cp_async_wait<1>();   // this chunk's records have landed (the next chunk's may still fly)
            __syncwarp();
            // lanes e and e+16: the fields of entry e -> multiplier pairs of lane groups 2*half, 2*half+1 and
            // the offset terms of blocks 4*half .. 4*half+3
            {
                const unsigned ra = rbuf + cur + (unsigned)(t * REC) + (unsigned)NCB;
                const uint4 tail = lds_v4(ra);
                const float xf = __half2float(__ushort_as_half(xv));
                const float df = __half2float(__ushort_as_half((unsigned short)(tail.w & 0xffffu)));
                const float dminf = __half2float(__ushort_as_half((unsigned short)(tail.w >> 16)));
#pragma unroll
                for (int g2 = 0; g2 < 2; ++g2) {
                    const int sb = 2 * half + g2;   // lane group: rows of blocks sb (low nibbles) and sb + 4 (high nibbles)
                    const float a_lo = xf * (df * (float)kq_field(tail.x, tail.y, tail.z, sb));       // d*sc is exact
                    const float a_hi = xf * (df * (float)kq_field(tail.x, tail.y, tail.z, sb + 4));
                    if (BITS == 4 || kHigh)
                        sts_pairs(mbuf + 16u * (unsigned)(t * 4 + sb), pack2(a_lo * 0x1p93f, a_hi * 0x1p89f),
                                  pack2(a_lo * 0x1p85f, a_hi * 0x1p81f));
                    else   // one pair: the high rows' codes sit in the same bytes (2 bits, four bits up) or in bytes of their own (8 bits)
                        sts_u64(mbuf + 16u * (unsigned)(t * 4 + sb), pack2(a_lo * 0x1p93f, a_hi * (BITS == 2 ? 0x1p89f : 0x1p93f)));
                }
#pragma unroll
                for (int i = 0; i < 4; ++i)
                    zl[i] += xf * (dminf * (float)kq_field(tail.x, tail.y, tail.z, 8 + 4 * half + i));
            }
            __syncwarp();
            const int valid = min(CH, hi - pos);
            const unsigned cb = rbuf + cur;
            auto step = [&](int u) {
                const unsigned e = (unsigned)(2 * u + half);
                if (BITS == 4 || kHigh) {
                    const uint2 wv = lds_v2(cb + e * REC + (unsigned)t * 8u);
                    unsigned long long m01, m23;
                    lds_pairs(mbuf + 16u * (e * 4u + (unsigned)(t >> 2)), m01, m23);
                    fma_block8(acc, wv, m01, m23);     // the low four bits of every code
                    if (BITS == 6) {
                        // the high two bits, 16 times the weight: a plane laid out like 2-bit codes, summed the same way
                        const unsigned long long mh = fmul2(m01, pack2(16.0f, 16.0f));
                        const uint2 hv = lds_v2(cb + e * REC + 128u + (unsigned)(t & 7) * 8u);
                        const int sh = 2 * (t >> 3);
#pragma unroll
                        for (int k = 0; k < 2; ++k) {
                            const unsigned w = (k ? hv.y : hv.x) >> sh, v = w >> 16;
                            ffma2(acch[4 * k + 0], pack2(__uint_as_float(w & 0x03u), __uint_as_float(w & 0x30u)), mh);
                            ffma2(acch[4 * k + 1], pack2(__uint_as_float(w & 0x0303u), __uint_as_float(w & 0x3030u)), mh);
                            ffma2(acch[4 * k + 2], pack2(__uint_as_float(v & 0x03u), __uint_as_float(v & 0x30u)), mh);
                            ffma2(acch[4 * k + 3], pack2(__uint_as_float(v & 0x0303u), __uint_as_float(v & 0x3030u)), mh);
                        }
                    } else if (BITS == 5) {
                        // the fifth bit of rows 8t.. and 128+8t..: one byte each; position b sums the byte's low b+1 bits
                        const unsigned long long mh = fmul2(m01, pack2(16.0f, 256.0f));   // (a_lo, a_hi) * 16 * 2^93
                        unsigned lb, hb;
                        asm volatile("ld.shared.u8 %0, [%1];" : "=r"(lb) : "r"(cb + e * REC + 128u + (unsigned)t) : "memory");
                        asm volatile("ld.shared.u8 %0, [%1];" : "=r"(hb) : "r"(cb + e * REC + 144u + (unsigned)t) : "memory");
#pragma unroll
                        for (int b = 0; b < 8; ++b) {
                            const unsigned mk = (2u << b) - 1u;
                            ffma2(acch[b], pack2(__uint_as_float(lb & mk), __uint_as_float(hb & mk)), mh);
                        }
                    }
                    return;
                }
                // 2 and 8 bits: per 16-bit half-word the value of its first byte's code and the value of both
                // codes together (second code times 256) are summed; the second code's sum is their difference
                const unsigned long long mm = lds_u64(mbuf + 16u * (e * 4u + (unsigned)(t >> 2)));
                if (BITS == 8) {
                    const uint2 lw = lds_v2(cb + e * REC + (unsigned)t * 8u);           // rows 8t .. 8t+7
                    const uint2 hw = lds_v2(cb + e * REC + 128u + (unsigned)t * 8u);    // rows 128+8t ..
#pragma unroll
                    for (int k = 0; k < 2; ++k) {
                        const unsigned l = k ? lw.y : lw.x, h = k ? hw.y : hw.x, lv = l >> 16, hv = h >> 16;
                        ffma2(acc[4 * k + 0], pack2(__uint_as_float(l & 0xffu), __uint_as_float(h & 0xffu)), mm);
                        ffma2(acc[4 * k + 1], pack2(__uint_as_float(l & 0xffffu), __uint_as_float(h & 0xffffu)), mm);
                        ffma2(acc[4 * k + 2], pack2(__uint_as_float(lv & 0xffu), __uint_as_float(hv & 0xffu)), mm);
                        ffma2(acc[4 * k + 3], pack2(__uint_as_float(lv), __uint_as_float(hv)), mm);
                    }
                } else {
                    // byte i holds rows i, i+64, i+128, i+192: lanes 0..7 use fields 0 and 2 of bytes 8t.., lanes
                    // 8..15 fields 1 and 3 of bytes 8(t-8)..
                    const uint2 wv = lds_v2(cb + e * REC + (unsigned)(t & 7) * 8u);
                    const int sh = 2 * (t >> 3);
#pragma unroll
                    for (int k = 0; k < 2; ++k) {
                        const unsigned w = (k ? wv.y : wv.x) >> sh, v = w >> 16;
                        ffma2(acc[4 * k + 0], pack2(__uint_as_float(w & 0x03u), __uint_as_float(w & 0x30u)), mm);
                        ffma2(acc[4 * k + 1], pack2(__uint_as_float(w & 0x0303u), __uint_as_float(w & 0x3030u)), mm);
                        ffma2(acc[4 * k + 2], pack2(__uint_as_float(v & 0x03u), __uint_as_float(v & 0x30u)), mm);
                        ffma2(acc[4 * k + 3], pack2(__uint_as_float(v & 0x0303u), __uint_as_float(v & 0x3030u)), mm);
                    }
                }
            };
            if (valid == CH) {
#pragma unroll
                for (int u = 0; u < CH / 2; ++u) step(u);   // a full chunk: straight-line code
            } else {
                const int nsub = (valid + 1) >> 1;
#pragma unroll 1
                for (int u = 0; u < nsub; ++u) step(u);
            }
            __syncwarp();
            cur = (cur == 0u) ? kBufBytes : 0u;
            col = col_next;
            col_next = col_after;
            xv = xv_next;
        }
    }
    cp_async_wait<0>();

    // warp -> CTA.  acc[b] = (row 8t+b, row 128+8t+b) of the entries this half-warp handled
    {
        float lo_rows[8], hi_rows[8];
#pragma unroll
        for (int b = 0; b < 8; ++b) {
            unpack2(acc[b], lo_rows[b], hi_rows[b]);
            lo_rows[b] += __shfl_xor_sync(0xffffffffu, lo_rows[b], 16);
            hi_rows[b] += __shfl_xor_sync(0xffffffffu, hi_rows[b], 16);
        }
        if (kHigh) {
            float lh[8], hh[8];
#pragma unroll
            for (int b = 0; b < 8; ++b) {
                unpack2(acch[b], lh[b], hh[b]);
                lh[b] += __shfl_xor_sync(0xffffffffu, lh[b], 16);
                hh[b] += __shfl_xor_sync(0xffffffffu, hh[b], 16);
            }
            if (BITS == 6) {      // pairs, as for 2-bit codes
#pragma unroll
                for (int b = 1; b < 8; b += 2) {
                    lh[b] = (lh[b] - lh[b - 1]) * 0x1p-8f;
                    hh[b] = (hh[b] - hh[b - 1]) * 0x1p-8f;
                }
            } else {              // a chain over the eight bits of a byte
#pragma unroll
                for (int b = 7; b > 0; --b) {
                    lh[b] = (lh[b] - lh[b - 1]) * (1.0f / (float)(1 << b));
                    hh[b] = (hh[b] - hh[b - 1]) * (1.0f / (float)(1 << b));
                }
            }
#pragma unroll
            for (int b = 0; b < 8; ++b) {
                lo_rows[b] += lh[b];
                hi_rows[b] += hh[b];
            }
        } else if (BITS != 4) {   // odd positions hold (first code + 256 * second code) of a half-word
#pragma unroll
            for (int b = 1; b < 8; b += 2) {
                lo_rows[b] = (lo_rows[b] - lo_rows[b - 1]) * 0x1p-8f;
                hi_rows[b] = (hi_rows[b] - hi_rows[b - 1]) * 0x1p-8f;
            }
        }
        if (half == 0) {
#pragma unroll
            for (int b = 0; b < 8; ++b) {
                sm.red[warp][8 * t + b] = lo_rows[b] * 0x1p56f;
                sm.red[warp][128 + 8 * t + b] = hi_rows[b] * 0x1p56f;
            }
        }
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            float z = zl[i];
#pragma unroll
            for (int o = 8; o > 0; o >>= 1) z += __shfl_xor_sync(0xffffffffu, z, o);
            if (t == 0) sm.red_z[warp][4 * half + i] = z;
        }
    }
    __syncthreads();

    // CTA -> block-row: G sums and 8 offset terms
    float* mine = partials + ((size_t)r * kKqMaxSplit + s) * (G + 8);
    for (int i = tid; i < G + 8; i += kKqThreads) {
        float v = 0.0f;
#pragma unroll
        for (int w = 0; w < kKqWarps; ++w) v += (i < G) ? sm.red[w][i] : sm.red_z[w][i - G];
        if (S == 1) {
            if (i < G) sm.red[0][i] = v;    // (warp 0's slot; every element has one writer)
            else sm.red_z[0][i - G] = v;
        } else {
            __stcg(mine + i, v);
        }
    }
    if (S == 1) {
        __syncthreads();
        for (int j = tid; j < G; j += kKqThreads) y[(size_t)r * G + j] = __float2half_rn(sm.red[0][j] - sm.red_z[0][j >> 5]);
        return;
    }
    __threadfence();
    __syncthreads();
    if (tid == 0) sm.last = (atomicAdd(counters + r, 1) == S - 1) ? 1 : 0;
    __syncthreads();
    if (!sm.last) return;
    __threadfence();
    const float* rowp = partials + (size_t)r * kKqMaxSplit * (G + 8);
    for (int j = tid; j < G; j += kKqThreads) {
        float v = 0.0f, z = 0.0f;
        for (int q = 0; q < S; ++q) {
            v += __ldcg(rowp + (size_t)q * (G + 8) + j);
            z += __ldcg(rowp + (size_t)q * (G + 8) + G + (j >> 5));
        }
        y[(size_t)r * G + j] = __float2half_rn(v - z);
    }
    if (tid == 0) counters[r] = 0;   // ready for the next call
}

// ---------------------------------------------------------------- host side

inline size_t kq_header_bytes(int R) { return (((size_t)R * 4 + 255) / 256) * 256; }
inline size_t kq_workspace_bytes(int R) { return kq_header_bytes(R) + (size_t)R * kKqMaxSplit * (kKqG + 8) * sizeof(float); }

static spqt_status kq_shape(int m, int n)
{
    if (m <= 0 || n <= 0) return SPQT_ERR_INVALID_ARG;
    if (m % kKqG != 0) return SPQT_ERR_UNSUPPORTED;
    if (m / kKqG > 65535) return SPQT_ERR_UNSUPPORTED;
    return SPQT_OK;
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
    static bool configured[64] = {};
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return SPQT_ERR_CUDA;
    const int smem = (int)sizeof(KqSmem<BITS>);
    if (!configured[dev]) {
        if (cudaFuncSetAttribute(kq_gemv_kernel<BITS>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem) != cudaSuccess) return SPQT_ERR_CUDA;
        configured[dev] = true;
    }
    const int sms = sm_count();
    if (sms <= 0) return SPQT_ERR_CUDA;
    // slices per block-row: fill the resident CTAs of every SM once; never less than a chunk per warp
    int S = (kq_ctas_per_sm(BITS) * sms) / R;
    const int by_work = n / (kKqChunk * kKqWarps);
    if (S > by_work) S = by_work;
    if (S > kKqMaxSplit) S = kKqMaxSplit;
    if (S < 1) S = 1;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(S, R);
    cfg.blockDim = dim3(kKqThreads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = static_cast<cudaStream_t>(stream);
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = g_no_pdl ? 0 : 1;
    int* counters = static_cast<int*>(workspace);
    float* partials = reinterpret_cast<float*>(static_cast<char*>(workspace) + kq_header_bytes(R));
    const cudaError_t err = cudaLaunchKernelEx(&cfg, kq_gemv_kernel<BITS>, static_cast<const uint8_t*>(records), n,
                                               static_cast<const __half*>(x), idx, count, static_cast<__half*>(y), partials, counters);
    count_launch();
    return (err == cudaSuccess && cudaGetLastError() == cudaSuccess) ? SPQT_OK : SPQT_ERR_CUDA;
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

// Activation-sparse GEMV over the zigzag layout, and its dense twin (4-bit and 3-bit codes).
//
// Work decomposition (the paper's hybrid row/column parallelism): one CTA of 8 warps per block-row, or a thread-block
// cluster of S CTAs, each with one of S equal slices of the ACTIVE index list; every warp has an equal part of its CTA's
// slice.  (Many block-rows with a long x: equal pieces of all block-rows instead, see gemv_pieces_kernel.)  The load follows the active entries, not the matrix columns.  A warp streams its part through its own ring
// of chunks of 32 list entries (cp.async: 16 bytes per lane, the lanes of a block adjacent so that every sector crosses
// once, with 64-byte L2 granularity so that an inactive neighbour block is not dragged in); nothing is shared between
// the warps until the end.  Then the warps' sums meet in shared memory, and the CTAs' sums in the shared memory of the
// cluster's first CTA, added in a fixed order (calls are bit-reproducible).
//
// Where the list comes from:
//   given list    lane e of a chunk reads idx directly, a few chunks ahead.
//   fused         the call that collects the indices in the same launch: every CTA copies x to shared memory, finds the
//                 active entries of every 256-entry piece and expands the pieces that overlap its own slice into a list
//                 of words, column and x (where a CTA has to hold all of a long list: columns alone).  The CTAs of
//                 block-row 0 write idx, each its slice; the first of them writes count.
//   dense         entry e is column e.
// Where the list has no x, it is fetched beside the entry's code copies.
//
// Per chunk, lane e turns the (scale, zero) pair of its entry into a = x_k*scale (exact in fp32), left as hi and lo for
// the tensor cores (spqt_mma.cuh), and adds x_k*zero to its share of the offset term; then the warp multiplies, the
// codes being operands as they are.  y[j] = sum_k a_k * code_jk + sum_k x_k * zero_rk.
//
// What bounds it.  Small and medium matrices: the fixed cost of a launch (a 4096 x 4096 call at 50 % needs 4.5 MB, 0.7 us
// of DRAM time, and takes 4.2 us), a chain of dependent steps.  Clock stamps from the end of the launch before: 0.6 us to
// the end of the wait for it, 0.6 x and the masks, 0.1 the count, 0.4 the list, 0.6 to 1.1 the first copies (all of the matrix is on
// its way then), 0.8 the loop and the sums, 0.4 the cluster's exchange.  Hence whole block-rows instead of fractions (no
// work map), one instance of every code path, few warps with much work each rather than many, and two CTAs per SM where
// the grid is large enough, so that one computes while the other starts or ends.  The kernel before the tensor cores (one
// persistent CTA of 18 warps per SM, fractional block-rows, packed FMAs, partial sums as tagged words in global memory;
// 4500 instructions of code against 1600) took 6.4 us there.  Large matrices: the code stream; 28672 x 8192 dense went
// from 26.9 to 21.6 us, 8192 x 28672 dense from 29.0 to 24.6 us among other calls in a stream (5.1 TB/s, 0.78 of the measured
// copy bandwidth; 21.2 us in short runs).
#include <cstddef>

#include "spqt_common.cuh"

namespace spqt {

constexpr int kCtasPerSm = 2;             // CTAs of 8 warps; of those of 16 there is one
constexpr int kMaxSplit = 8;              // CTAs of a block-row: the largest portable cluster
constexpr int kCapPlain = 8192;           // list entries a CTA of a fused call keeps in shared memory: of a whole block-row,
constexpr int kCapSlice = 7168;           // of a slice
constexpr int kMaxListN = 65535;          // column numbers travel as 16 bits
constexpr int kMaxFusedN = 32768;         // longest x the in-kernel scan handles (128 pieces of 256 entries)
constexpr int kMaxPieces = kMaxFusedN / 256;

enum : int { kModeList = 0, kModeFused = 1, kModeDense = 2 };

static int g_tune_ctas = 0;  // 0 = the built-in rule
int g_no_pdl = 0;            // 1 = plain stream-ordered launches (also read by the index-collection launch)
static int g_no_cluster = 0; // 1 = never launch thread-block clusters
static int g_static_partition = 0;  // 1 = ablation: static partition of the matrix columns instead of the list

}  // namespace spqt

#include "spqt_gemv_device.cuh"
#include "spqt_mma.cuh"

namespace spqt {

// How a grid shares the block-rows.
//   plain     one CTA per block-row
//   cluster   a cluster of CTAs per block-row, one slice of the list each
//   serial    one CTA per block-row, the slices of the list in turn (the same parts and order of sums as a cluster)
// and, as a kernel of its own,
//   pieces    one CTA of 16 warps per SM; the block-rows are laid end to end and cut into equal pieces, one for every warp
enum : int { kPlain = 0, kCluster = 1, kSerial = 2 };

// ---------------------------------------------------------------- shared memory

// A warp's ring: D chunks of CH list entries.
template <int G, int MODE>
struct RowRing {                         // where a CTA works on one block-row
    // 64-row blocks without a list (every block is read): chunks of 64, half the bookkeeping (11072 x 4096 7.7 against 9.0 us);
    // with a list they cost more in the parts' last chunks (4096 x 14336 at 50 % 10.0 against 9.5 us)
    static constexpr int CH = MODE == kModeDense ? 32 * (128 / G) : 32, D = MODE == kModeDense || G == 128 ? 4 : 6;
};
template <int G, int BITS, int MODE>
struct PieceRing {                       // the CTA keeps the whole list as well
    // 64-row blocks: chunks of 64 (dense 28672 x 8192 4 bits 25.6 against 27.3 us, 3 bits 31.9 against 36.9), but not for
    // lists of 24-byte blocks (24.1 against 31.4 us: fewer copies in flight)
    static constexpr bool kShort = BITS == 3 && G == 64 && MODE != kModeDense;
    static constexpr int CH = kShort ? 32 : 32 * (128 / G), D = G == 128 ? 4 : kShort ? 6 : 3;
};

template <int G, int BITS, class Ring>
struct Stage {
    alignas(16) unsigned char codes[Ring::CH * MmaStage<G, BITS>::kRow];   // the chunk's blocks, as the matrix loads want them
    alignas(16) unsigned meta[Ring::CH];              // (scale, zero) pair of entry e
};

template <int G, int BITS, int MODE, int NW>
struct LoopSmem {
    using Ring = RowRing<G, MODE>;
    Stage<G, BITS, Ring> stage[NW][Ring::D];
    union Warp {
        unsigned short b[Ring::CH][8];                // operand B of a chunk: hi and lo of every entry's multiplier, then padding
        float red[G];                                 // after the last chunk: the warp's sums, as the tiles have them
    };
    alignas(16) Warp warp[NW];
    float2 red_z[NW];                                 // the sums' scale and offset terms
};

template <int G, int BITS, int MODE, int NW>
struct PieceLoopSmem {
    using Ring = PieceRing<G, BITS, MODE>;
    Stage<G, BITS, Ring> stage[NW][Ring::D];
    alignas(16) unsigned short b[NW][Ring::CH][8];
    alignas(16) float red[2][NW][G];
    float2 red_z[2][NW];
};

struct ScanSmem {                                     // fused: while the list is built
    alignas(16) unsigned char xs[kMaxFusedN * 2];     // x
    alignas(16) int tot[kMaxPieces];                  // active entries of every 256 entries of x
    unsigned short mask[kMaxPieces][32];              // which they are, 8 entries a byte; above it, how many precede them in the piece
};

template <int G, int BITS, int MODE, int KIND, int NW>
struct GemvSmem {
    using Loop = LoopSmem<G, BITS, MODE, NW>;
    union Area {
        Loop loop;
        unsigned char scan[MODE == kModeFused ? sizeof(ScanSmem) : 16];
    };
    alignas(16) unsigned char area[sizeof(Area)];
    alignas(16) float2 xred[KIND == kCluster ? kMaxSplit - 1 : 1][G / 2];   // first CTA of a cluster: the other CTAs' sums
    uint64_t arrival;             // and their arrival
    int table[NW + 1];                                // ablation: list positions of a static column partition
    alignas(16) unsigned ent[MODE == kModeFused ? (KIND == kPlain ? kCapPlain : kCapSlice) : 4];   // fused: the CTA's slice of the list, x bits << 16 | column
};

constexpr int kPieceWarps = 16;
constexpr unsigned kSlotMark = 0x53705174u;   // a slot that holds a sum
template <int G, int BITS, int MODE>
struct PieceSmem {
    using Loop = PieceLoopSmem<G, BITS, MODE, kPieceWarps>;
    union Area {
        Loop loop;
        unsigned char scan[MODE == kModeFused ? sizeof(ScanSmem) : 16];
    };
    alignas(16) unsigned char area[sizeof(Area)];
    alignas(16) unsigned short ent[MODE == kModeFused ? kMaxFusedN : 8];   // fused: the columns of the whole list
};

struct GemvArgs {
    const uint8_t* codes;
    const unsigned* meta;       // (scale, zero) pairs
    int n, R;
    int splits;                 // slices of the list
    unsigned magic_s;           // floor((2^32 - 1) / splits)
    unsigned warps, magic_w;    // pieces: warps of the grid, floor((2^32 - 1) / warps)
    unsigned magic_r, magic_p;  // the same of R and of the number of CTAs
    unsigned* status;           // the workspace's status word
    unsigned long long* slots;  // pieces: G words between every two neighbouring CTAs (zero between calls)
    const __half* x;
    const int32_t* idx;
    const int32_t* count;
    __half* y;
    unsigned short thr;         // fused: the largest fp16 value not above the threshold (negative: -1)
    int32_t* idx_out;
    int32_t* count_out;
    int static_partition;
    int small;                  // the matrix is small beside L2
    int together;               // whether a cluster's CTAs leave together (see cluster_leave_together; the last member: before the
                                // others it moved some that every call needs to another line, 0.05 us a call)
};

// floor(v / d) for any 32-bit v from the multiplier m = floor((2^32 - 1) / d): the high product is
// the quotient or one less (the multiplier falls short of 2^32 / d by at most 1), one compare fixes it.
__device__ __forceinline__ unsigned magic_div(unsigned v, unsigned d, unsigned m)
{
    const unsigned q = __umulhi(v, m);
    return q + ((v - q * d >= d) ? 1u : 0u);
}

// Hints only (no data is consumed before the wait for the previous kernel, and a prefetched line is as coherent as any other in
// L2), given while that kernel drains and the memory has little to do.  x: a few CTAs do it for all.  (Not a given list: how much
// of it there is to read is known only behind the wait.)
template <int THREADS>
__device__ __forceinline__ void prefetch_inputs(const GemvArgs& a, int tid)
{
    if ((blockIdx.x & 15) != 0) return;
    prefetch_l2(a.x, 2 * (size_t)a.n, tid, THREADS);
}

// ---------------------------------------------------------------- copies

// The copies of one chunk: the (scale, zero) pairs and code blocks of columns col[], lane's entries lane, lane + 32, ..; `whole`:
// the columns are neighbours, and none is missing (their blocks lie one after the other: one address; 28672 x 4096 dense 12.85 ->
// 12.6 us, 8192 x 28672 21.5 -> 21.2; no gain for pieces)
template <int G, int BITS, class Ring>
__device__ __forceinline__ void copy_chunk(unsigned st, const uint8_t* row_codes, const unsigned* row_meta, const unsigned* col, int lane, bool whole)
{
    constexpr int B = G * BITS / 8, CH = Ring::CH, EPL = CH / 32;
    constexpr int CB = (B % 16 == 0) ? 16 : 8;        // bytes per copy: 3-bit blocks of 64 rows are only 8-byte aligned
    constexpr int NC = CH * B / CB / 32;              // copies per lane and chunk
    constexpr int kRow = MmaStage<G, BITS>::kRow;
    constexpr unsigned kMetaOff = (unsigned)sizeof(Stage<G, BITS, Ring>::codes);
    auto place = [&](int q) -> unsigned {
        const int p = q * 32 + lane, e = p / (B / CB), part = p % (B / CB);
        if (BITS == 4 && G == 128) return e * 64 + ((part ^ ((e >> 1) & 3)) << 4);
        if (BITS == 4) return e * 32 + ((part ^ ((e >> 2) & 1)) << 4);
        return e * kRow + part * CB;
    };
    auto copy = [&](unsigned dst, const uint8_t* src) {
        if (CB == 16) cp_async_16_l2_64(dst, src);
        else cp_async_8(dst, src);
    };
#pragma unroll
    for (int q = 0; q < EPL; ++q) cp_async_4(st + kMetaOff + 4u * (lane + 32 * q), row_meta + col[q]);
    if (whole) {
        const uint8_t* const src = row_codes + ((size_t)(col[0] - lane) * B + lane * CB);
#pragma unroll
        for (int q = 0; q < NC; ++q) copy(st + place(q), src + q * 32 * CB);
    } else {
#pragma unroll
        for (int q = 0; q < NC; ++q) {
            const int p = q * 32 + lane, e = p / (B / CB), part = p % (B / CB);
            const unsigned cu = __shfl_sync(0xffffffffu, col[q / (NC / EPL)], e & 31);
            copy(st + place(q), row_codes + ((size_t)cu * B + part * CB));
        }
    }
    if (BITS == 3 && G == 64) {                       // the 1-bit plane a second time (see MmaStage)
#pragma unroll
        for (int q = 0; q < EPL; ++q) cp_async_8(st + (lane + 32 * q) * kRow + 24, row_codes + ((size_t)col[q] * B + 16));
    }
}

// ---------------------------------------------------------------- the product

// A warp's sums and what it takes to multiply a chunk.  While chunk i is multiplied, chunk i + 1 is prepared: lane e turns
// its entry's pair and x into a = x*scale (exact in fp32), left as hi and lo, and x*zero.
template <int G, int BITS, class Ring>
struct Product {
    static constexpr int EPL = Ring::CH / 32, SP = MmaStage<G, BITS>::kSp;
    using Layout = MmaStage<G, BITS>;
    float acc[SP][4][4];             // sums of the rows times the hi (column 0) and lo (column 1) multipliers, in lanes t4 == 0
    float scale, regain;             // c of spqt_mma.cuh; factor that the sums still have to be brought to it by
    float zl, zn;                    // sum of x*zero, and the prepared chunk's part of it
    float am[EPL], pm[EPL];
    unsigned b_base;                 // this lane's row of B
    int lane;

    __device__ __forceinline__ Product(unsigned b, int lane_) : scale(kMmaNoScale), regain(1.0f), zn(0.0f), b_base(b + 16u * lane_), lane(lane_) { clear(); }
    __device__ __forceinline__ void clear()
    {
        zl = 0.0f;
#pragma unroll
        for (int i = 0; i < SP * 16; ++i) acc[i >> 4][(i >> 2) & 3][i & 3] = 0.0f;
    }
    // xb: the fp16 bits of the lane's x values, 0 for an entry that does not exist; true if one exceeds the range
    __device__ __forceinline__ bool prepare(unsigned st, const unsigned* xb)
    {
        constexpr unsigned kMetaOff = (unsigned)sizeof(Stage<G, BITS, Ring>::codes);
        zn = 0.0f;
        float top = 0.0f;
#pragma unroll
        for (int q = 0; q < EPL; ++q) {
            const unsigned mz = lds_u32(st + kMetaOff + 4u * (lane + 32 * q));
            const float xf = __half2float(__ushort_as_half((unsigned short)xb[q]));
            am[q] = xf * __half2float(__ushort_as_half((unsigned short)(mz & 0xffffu)));
            zn += xf * __half2float(__ushort_as_half((unsigned short)(mz >> 16)));
            pm[q] = am[q] * scale;   // a power of two
            top = fmaxf(top, fabsf(pm[q]));
        }
        return top > kMmaLimit;
    }
    // a larger entry than the range holds: a new scale; the sums follow once chunk i is in them
    __device__ __forceinline__ void rescale()
    {
        unsigned m = 0;
#pragma unroll
        for (int q = 0; q < EPL; ++q) {
            const unsigned bits = __float_as_uint(am[q]) & 0x7fffffffu;
            m = max(m, bits < 0x7f800000u ? bits : 0u);   // finite ones
        }
        m = __reduce_max_sync(0xffffffffu, m);
        if (__uint_as_float(m) * scale > kMmaLimit) {
            const float next = __uint_as_float((266u - (m >> 23)) << 23);   // m goes to 2^12 .. 2^13
            regain = next * power_of_two_inverse(scale);
            scale = next;
#pragma unroll
            for (int q = 0; q < EPL; ++q) pm[q] = am[q] * next;
        }
    }
    __device__ __forceinline__ void leave()
    {
#pragma unroll
        for (int q = 0; q < EPL; ++q) {
            const float h = __low2float(__floats2half2_rn(to_halves(pm[q]), 0.0f));
            const __half2 hl = __floats2half2_rn(h, pm[q] - h);
            sts_u32(b_base + 512u * q, *reinterpret_cast<const unsigned*>(&hl));
        }
    }
    // the first chunk: there is nothing in the sums yet
    __device__ __forceinline__ void begin(unsigned st, const unsigned* xb)
    {
        if (__any_sync(0xffffffffu, prepare(st, xb))) rescale();
        leave();
        regain = 1.0f;
        __syncwarp();
    }
    // multiplies the chunk in stage st and leaves B of the next one, whose entries prepare() reads from stage `next`
    __device__ __forceinline__ void multiply(unsigned st, const typename Layout::Lane& ll, unsigned next, const unsigned* xb)
    {
        zl += zn;
        const bool over = prepare(next, xb);
        unsigned bb[EPL][4], c[SP][4];
#pragma unroll
        for (int q = 0; q < EPL; ++q) ldsm_x4_trans(b_base + 512u * q, bb[q]);
        __syncwarp();                // (B is in registers: its place is free)
#pragma unroll
        for (int ks = 0; ks < 2 * EPL; ++ks) {
            Layout::load(st, ll, ks, c);
            if (ks == 2 * EPL - 1) {
                if (__any_sync(0xffffffffu, over)) rescale();
                leave();
            }
#pragma unroll
            for (int sp = 0; sp < SP; ++sp) mma_group(acc[sp], c[sp], bb[ks >> 1] + 2 * (ks & 1));
        }
        if (regain != 1.0f) {
#pragma unroll
            for (int i = 0; i < SP * 8; ++i) {
                float* const a = &acc[i >> 3][(i >> 1) & 3][2 * (i & 1)];
                rescale_sums(a[0], a[1], regain);
            }
            regain = 1.0f;
        }
        __syncwarp();                // every lane is done with this chunk's stage
    }
    // the sums as the tiles have them (eight lanes of a warp hold them all), their scale and the offset term
    __device__ __forceinline__ void hand_over(float* red, float2* red_z)
    {
        if ((lane & 3) == 0) {
#pragma unroll
            for (int sp = 0; sp < SP; ++sp)
#pragma unroll
                for (int i = 0; i < 8; ++i) {
                    const int type = i >> 1, hf = 2 * (i & 1);
                    red[Layout::row(sp, type, hf, lane >> 2)] = acc[sp][type][hf] + acc[sp][type][hf + 1];   // hi + lo
                }
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) zl += __shfl_xor_sync(0xffffffffu, zl, o);
        if (lane == 0) *red_z = make_float2(0x1p24f * power_of_two_inverse(scale), zl);
    }
};

// The warps' sums of a block-row, in warp order: thread j < G / 2 gets rows j and j + G/2, those of the low and the high
// nibbles of byte j (the latter's tiles sum 16 times the nibble of even bytes and the whole of odd ones).
template <int G, int NW, class Warp>
__device__ __forceinline__ void add_warps(const Warp* warp, const float2* red_z, int j, float* v, float* z)
{
    v[0] = v[1] = *z = 0.0f;
#pragma unroll
    for (int w = 0; w < NW; ++w) {
        const float2 cz = red_z[w];
        v[0] += warp[w].red[j] * cz.x;
        v[1] += warp[w].red[j + G / 2] * cz.x;
        *z += cz.y;
    }
    v[1] = (v[1] - ((j & 1) ? v[0] : 0.0f)) * 0.0625f;
}

// ---------------------------------------------------------------- fused: the list

template <int NW>
struct Scan {
    ScanSmem& sc;
    const __half2 thr;
    int n, nv, lane, warp;
    int t[4];                                         // lane l: active entries of pieces 4l .. 4l+3

    __device__ __forceinline__ Scan(unsigned char* area, unsigned short thr_bits, int n_, int lane_, int warp_)
        : sc(*reinterpret_cast<ScanSmem*>(area)), thr(__half2half2(__ushort_as_half(thr_bits))), n(n_), nv((n_ + 255) >> 8), lane(lane_), warp(warp_)
    {
    }
    // all ones in the halves of w whose magnitude exceeds the threshold: exact in fp16, never for a NaN
    __device__ __forceinline__ unsigned active(unsigned w) const
    {
        w &= 0x7fff7fffu;
        return __hgt2_mask(*reinterpret_cast<const __half2*>(&w), thr);
    }
    __device__ __forceinline__ int below(int li) const   // active entries before piece li
    {
        int v = 0;
#pragma unroll
        for (int q = 0; q < 4; ++q) v += lane * 4 + q < li ? t[q] : 0;
        return (int)__reduce_add_sync(0xffffffffu, (unsigned)v);
    }
    // x to shared memory (entries that do not exist as not-a-number: never active), and per piece of 256 entries which ones are
    // active and how many; returns the count.  A chain of latencies that every call pays, so x goes through registers (by way
    // of shared memory with cp.async 0.1 us longer), the loads of a warp's first four pieces together, and nothing is done for
    // pieces that are not there (0.08 us at n = 4096).
    __device__ __forceinline__ int scan_x(const __half* x)
    {
        const int tid = warp * 32 + lane;
        const unsigned xs_base = smem_u32(sc.xs);
        const unsigned short* const xg = reinterpret_cast<const unsigned short*>(x);
        const bool words = (reinterpret_cast<uintptr_t>(x) & 15) == 0;
        if (tid >= nv && tid < kMaxPieces) sc.tot[tid] = 0;
#pragma unroll 1
        for (int l0 = warp; l0 < nv; l0 += 4 * NW) {
            uint4 v[4];
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const int li = l0 + i * NW, k = li * 256 + lane * 8;
                if (li >= nv) break;                  // (uniform, as is the next condition)
                if (words && li * 256 + 256 <= n) {
                    v[i] = ld_global_v4(xg + k);
                } else {
                    unsigned w[4];
#pragma unroll
                    for (int j = 0; j < 4; ++j) {     // (no load behind a condition: they go together)
                        const unsigned e = ld_global_u16(xg + min(k + 2 * j, n - 1)), o = ld_global_u16(xg + min(k + 2 * j + 1, n - 1));
                        w[j] = (k + 2 * j < n ? e : 0x7fffu) | (k + 2 * j + 1 < n ? o : 0x7fffu) << 16;
                    }
                    v[i] = make_uint4(w[0], w[1], w[2], w[3]);
                }
            }
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const int li = l0 + i * NW;
                if (li >= nv) break;
                sts_v4(xs_base + li * 512u + lane * 16u, v[i]);
                unsigned m = (active(v[i].x) & 0x00020001u) | (active(v[i].y) & 0x00080004u) | (active(v[i].z) & 0x00200010u) | (active(v[i].w) & 0x00800040u);
                m = (m | (m >> 16)) & 0xffu;
                // how many precede this lane's: bit by bit of the counts
                const unsigned c = (unsigned)__popc(m), lt = (1u << lane) - 1u;
                unsigned before = 0;
#pragma unroll
                for (int q = 0; q < 4; ++q) before += (unsigned)__popc(__ballot_sync(0xffffffffu, (c >> q) & 1u) & lt) << q;
                sc.mask[li][lane] = (unsigned short)(m | (before << 8));
                if (lane == 31) sc.tot[li] = (int)(before + c);
            }
        }
        __syncthreads();
        const int4 s = *reinterpret_cast<const int4*>(&sc.tot[lane * 4]);
        t[0] = s.x; t[1] = s.y; t[2] = s.z; t[3] = s.w;
        return (int)__reduce_add_sync(0xffffffffu, (unsigned)(s.x + s.y + s.z + s.w));
    }
    // the list position of column kb: the number of active entries below it (the same in all lanes)
    __device__ __forceinline__ int position(int kb) const
    {
        const int piece = kb >> 8;
        int inside = 0;
        if (piece < nv) {
            const int in8 = (kb & 255) - 8 * lane;   // entries of this lane's byte below it
            inside = __popc((unsigned)sc.mask[piece][lane] & (in8 >= 8 ? 0xffu : in8 <= 0 ? 0u : (1u << in8) - 1u));
        }
        return below(piece) + (int)__reduce_add_sync(0xffffffffu, (unsigned)inside);
    }
    // The entries [lo, hi) of the list into ent (E = unsigned: x bits << 16 | column; unsigned short: columns), and the
    // entries [out_lo, out_hi) into the returned list.
    template <class E>
    __device__ __forceinline__ void build(E* ent, int lo, int hi, int32_t* idx_out, int out_lo, int out_hi)
    {
        const unsigned short* const xs = reinterpret_cast<const unsigned short*>(sc.xs);
        const unsigned bit = 1u << (lane & 7), len = (unsigned)(hi - lo), out_len = (unsigned)(out_hi - out_lo);
#pragma unroll 1
        for (int li = warp; li < nv; li += NW) {
            const int base = below(li);
            if (base >= hi || base + sc.tot[li] <= lo) continue;   // (uniform)
            const unsigned col = (unsigned)(li * 256 + lane);
            // all loads first (the compiler cannot move one past a store: 360 instead of 1300 cycles a piece); neighbouring
            // lanes to neighbouring places
            unsigned m[8], w[8];
#pragma unroll
            for (int j = 0; j < 8; ++j) m[j] = sc.mask[li][4 * j + (lane >> 3)];
#pragma unroll
            for (int j = 0; j < 8; ++j) w[j] = sizeof(E) == 4 ? (unsigned)xs[col + 32 * j] << 16 : 0u;
#pragma unroll
            for (int j = 0; j < 8; ++j) {
                const unsigned at = (unsigned)base + (m[j] >> 8) + (unsigned)__popc(m[j] & (bit - 1u));
                w[j] |= col + 32 * j;
                m[j] = (m[j] & bit) != 0u ? at : 0x7fffffffu;
            }
#pragma unroll
            for (int j = 0; j < 8; ++j)
                if (m[j] - (unsigned)lo < len) ent[m[j] - (unsigned)lo] = (E)w[j];
            if (out_len != 0u) {
#pragma unroll
                for (int j = 0; j < 8; ++j)
                    if (m[j] - (unsigned)out_lo < out_len) idx_out[m[j]] = (int)(col + 32 * j);
            }
        }
    }
};

// ---------------------------------------------------------------- whole block-rows

template <int G, int BITS, int MODE, int KIND, int NW>
// (64-row groups to 4 bits with a list given, whole block-rows: an SM has registers and shared memory for three CTAs if they need no
// more than 80; with 82 25600 x 2048 takes 8.75 us instead of 6.85)
__global__ void __launch_bounds__(NW * 32, NW != 8 ? 1 : G == 64 && BITS == 4 && MODE == kModeList && KIND == kPlain ? 3 : kCtasPerSm)
gemv_kernel(const GemvArgs a)
{
    using Ring = RowRing<G, MODE>;
    constexpr int B = G * BITS / 8, CH = Ring::CH, EPL = CH / 32, D = Ring::D;   // EPL: entries a lane looks after
    constexpr int kThreads = NW * 32;
    constexpr bool FUSED = MODE == kModeFused, LIST = MODE == kModeList;
    using Smem = GemvSmem<G, BITS, MODE, KIND, NW>;

    extern __shared__ __align__(16) unsigned char smem_raw[];
    Smem& sm = *reinterpret_cast<Smem*>(smem_raw);
    typename Smem::Loop& lp = *reinterpret_cast<typename Smem::Loop*>(sm.area);
    const int tid = threadIdx.x, lane = tid & 31;
    // the warp number through a shuffle: the compiler then knows it is the same in every lane
    const int warp = __shfl_sync(0xffffffffu, tid >> 5, 0);
    const int n = a.n;
    unsigned rank = 0, r = blockIdx.x;
    if (KIND == kCluster) {
        asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(rank));
        asm volatile("mov.u32 %0, %%clusterid.x;" : "=r"(r));
        // nobody may write to another CTA's shared memory before that CTA runs: arrive now, wait much later
        if (tid == 0) {
            mbar_init(&sm.arrival, 1);
            mbar_expect(&sm.arrival, (unsigned)(a.splits - 1) * (unsigned)sizeof(sm.xred[0]));
            mbar_publish();
        }
        __syncwarp();
        cluster_arrive();
    }
    // the slices of the list this CTA works on: first_part .. last_part - 1 of `parts`
    const unsigned parts = (unsigned)a.splits, first_part = rank, last_part = KIND == kCluster ? rank + 1u : parts;

    prefetch_inputs<kThreads>(a, tid);
    // constants of the loop that need no data
    const typename MmaStage<G, BITS>::Lane ll(lane);
    const unsigned stage0 = smem_u32(&lp.stage[warp][0]);
    constexpr unsigned kStageBytes = (unsigned)sizeof(Stage<G, BITS, Ring>), kRing = D * kStageBytes;
    const unsigned ent_base = smem_u32(&sm.ent[0]);
    const unsigned short* const xg = reinterpret_cast<const unsigned short*>(a.x);
    const uint8_t* const row_codes = a.codes + (size_t)r * (size_t)n * B;
    const unsigned* const row_meta = a.meta + (size_t)r * (size_t)n;

    // Hints to the weights of this warp's share of the block-row, to a few entries: the (scale, zero) pairs, of which every sector
    // is needed, whichever entries are active (28672 x 8192 at 50 % 17.3 -> 16.8 us), and without a list the first chunks of codes
    // (both: 4096 x 4096 4.13 -> 3.8 us).  Not for a large matrix without a list: L2 has lost many of the pairs by the time they are
    // needed, and the codes gain nothing (8192 x 28672 25.9 against 25.5 us among other calls).
    {
        const int c0 = KIND == kCluster ? (int)((unsigned long long)n * rank / parts) : 0, c1 = KIND == kCluster ? (int)((unsigned long long)n * (rank + 1u) / parts) : n;
        const int each = (c1 - c0 + NW - 1) / NW, from = c0 + min(each * warp, c1 - c0), here = min(each, c1 - from);
        if (MODE != kModeDense || a.small) prefetch_l2(row_meta + from, 4 * (size_t)here, lane, 32);
        if (MODE == kModeDense && a.small) prefetch_l2(row_codes + (size_t)from * B, (size_t)min(here, (D - 1) * CH) * B, lane, 32);
    }
    // Programmatic dependent launch: this grid may have been started while the previous kernel of the stream was still
    // draining.  Nothing above touches memory another kernel writes; everything below waits for that kernel to
    // complete, and lets the next kernel of the stream start early in turn.
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");

    Scan<NW> scan(sm.area, a.thr, n, lane, warp);            // (fused calls only)
    int count = n;
    if (LIST) count = (int)ld_global_u32(a.count);
    float nothing = 0.0f;                // what the sums of x*zero begin with: not-a-number for a list without a length (see kListLost)
    if (LIST && count < 0) {
        count = 0;
        nothing = __int_as_float(0x7fffffff);
        if (blockIdx.x == 0 && tid == 0) atomicExch(a.status, 1u);
    }
    if (FUSED) {
        count = scan.scan_x(a.x);
        if (blockIdx.x == 0 && tid == 0) *a.count_out = count;
    }

    float total[2] = {0.0f, 0.0f};   // thread j < G / 2: rows j and j + G/2, over the slices of this CTA
#pragma unroll 1
    for (unsigned part = first_part; KIND != kSerial || part < last_part; ++part) {
        // ---- the slice: in units of 8 entries, so that slices and parts begin at multiples of 8
        int lo = 0, hi = count;
        bool fixed_parts = false;
        if (KIND != kPlain) {
            const unsigned units = (unsigned)(count + 7) >> 3;
            lo = 8 * (int)magic_div(part * units, parts, a.magic_s);
            hi = min(8 * (int)magic_div((part + 1u) * units, parts, a.magic_s), count);
        }
        if (FUSED) {
            if (KIND == kSerial && part != first_part) scan.scan_x(a.x);
            if (a.static_partition) {
                // Ablation, the paper's "sparse without load balancing": a slice is a fixed range of the matrix COLUMNS,
                // and so is every warp's part of it.
                for (int j = warp; j <= NW; j += NW) {
                    const int at = scan.position((int)(((long long)n * ((int)part * NW + j)) / ((int)parts * NW)));
                    if (lane == 0) sm.table[j] = at;
                }
                __syncthreads();
                lo = sm.table[0];
                hi = sm.table[NW];
                fixed_parts = true;
            }
            scan.build(sm.ent, lo, hi, a.idx_out, lo, r == 0 ? hi : lo);
            __syncthreads();             // the list is in place, and the ring may overwrite x
        }
        // ---- this warp's part of it
        const int pu = (hi - lo + 7) >> 3;
        int first = lo + 8 * ((pu * warp) / NW), end = min(lo + 8 * ((pu * (warp + 1)) / NW), hi);
        if (FUSED && fixed_parts) {
            first = sm.table[warp];
            end = sm.table[warp + 1];
        }

        // given list: the columns of the lane's entries in the chunks the copies come to next, fetched kAhead chunks early
        constexpr int kAhead = 3;
        int coming[kAhead][EPL], ahead = first;
        auto fetch_ahead = [&](int d) {
#pragma unroll
            for (int q = 0; q < EPL; ++q) coming[d][q] = (int)ld_global_u32(a.idx + min(ahead + 32 * q + lane, end - 1));
            ahead = ahead + CH >= end ? first : ahead + CH;
        };
        if (LIST && first < end) {
#pragma unroll
            for (int d = 0; d < kAhead; ++d) fetch_ahead(d);
        }
        unsigned xv[D][EPL];             // list and dense: the x values of the chunks in flight, the oldest first
#pragma unroll
        for (int i = 0; i < D * EPL; ++i) xv[i / EPL][i % EPL] = 0;
        int ipos = first;                // where the copies stand: D - 1 chunks ahead of the product
        unsigned ri = 0;                 // byte offset of the copies' stage
        auto issue = [&]() {             // the copies of the next chunk, if there is one
            if (!FUSED) {                // (0 past the end: what the stages hold there must not change the scale)
#pragma unroll
                for (int i = 0; i < D * EPL; ++i) xv[i / EPL][i % EPL] = i < (D - 1) * EPL ? xv[(i / EPL + 1) % D][i % EPL] : 0u;
            }
            if (ipos < end) {
                unsigned col[EPL];
#pragma unroll
                for (int q = 0; q < EPL; ++q) {       // (past the end: the last entry again, with x = 0)
                    const int e = ipos + 32 * q + lane;
                    col[q] = LIST ? (unsigned)coming[0][q] : FUSED ? lds_u16(ent_base + 4u * (unsigned)(min(e, end - 1) - lo)) : (unsigned)min(e, end - 1);
                    if (!FUSED) xv[D - 1][q] = ld_global_u16_if(e < end, xg + col[q]);
                }
                copy_chunk<G, BITS, Ring>(stage0 + ri, row_codes, row_meta, col, lane, MODE == kModeDense && ipos + CH <= end);
                ri = ri + kStageBytes == kRing ? 0u : ri + kStageBytes;
                ipos += CH;
                if (LIST) {
#pragma unroll
                    for (int i = 0; i < (kAhead - 1) * EPL; ++i) coming[i / EPL][i % EPL] = coming[i / EPL + 1][i % EPL];
                    fetch_ahead(kAhead - 1);
                }
            }
            cp_async_commit();
        };
#pragma unroll 1
        for (int d = 0; d < D - 1; ++d) issue();

        // ---- the loop
        Product<G, BITS, Ring> product(smem_u32(&lp.warp[warp].b[0][0]), lane);
        if (LIST) product.zl = nothing;
        unsigned xb[EPL];                // x of the entries from list position p on
        auto x_at = [&](int p) {
#pragma unroll
            for (int q = 0; q < EPL; ++q) {
                const int e = p + 32 * q + lane;
                xb[q] = !FUSED ? xv[1][q] : e < end ? lds_u16(ent_base + 4u * (unsigned)(e - lo) + 2u) : 0u;
            }
        };
        unsigned rc = 0;                 // the stage of chunk i
        if (first < end) {
            cp_async_wait<D - 2>();
            __syncwarp();
            x_at(first);
            product.begin(stage0, xb);
        }
#pragma unroll 1
        for (int pos = first; pos < end; pos += CH) {
            issue();
            const unsigned rn = rc + kStageBytes == kRing ? 0u : rc + kStageBytes;
            x_at(pos + CH);
            cp_async_wait<D - 2>();
            __syncwarp();
            product.multiply(stage0 + rc, ll, stage0 + rn, xb);
            rc = rn;
        }
        product.hand_over(lp.warp[warp].red, &lp.red_z[warp]);
        __syncthreads();
        if (tid < G / 2) {
            float v[2], z;
            add_warps<G, NW>(lp.warp, lp.red_z, tid, v, &z);
            total[0] += v[0] + z;
            total[1] += v[1] + z;
        }
        cp_async_wait<0>();
        if (KIND != kSerial) break;
        __syncthreads();                 // (every warp is done with the ring and the list)
    }

    if (KIND == kCluster) {
        // The other CTAs send their sums to the first one's shared memory, which counts the bytes and adds the sums in CTA
        // order.  The only wait is the first CTA's for the data.  Remote stores with a cluster barrier behind them, where the
        // senders wait for their stores and everybody for everybody, took 1.2 to 1.3 us from the warps' sums to y, this 0.4 to
        // 0.5 (1024 x 4096 at 50 % 4.1 -> 3.6 us, 4096 x 4096 4.8 -> 4.4, with the list 4.0 -> 3.6).
        cluster_wait();                  // (every CTA of the cluster runs)
        if (rank != 0) {
            if (tid < G / 2) st_async_f32x2(cluster_map(smem_u32(&sm.xred[rank - 1][tid]), 0u), total[0], total[1], cluster_map(smem_u32(&sm.arrival), 0u));
            if (a.together) cluster_leave_together();
            return;
        }
        if (tid < G / 2) {
            if (!mbar_wait_cluster(&sm.arrival, 0u)) {
                atomicExch(a.status, 1u);
                total[0] = total[1] = __int_as_float(0x7fffffff);
            }
#pragma unroll
            for (int q = 0; q < kMaxSplit - 1; ++q)
                if (q < a.splits - 1) {
                    const float2 v = sm.xred[q][tid];
                    total[0] += v.x;
                    total[1] += v.y;
                }
        }
    }
    if (tid < G / 2) {
        a.y[(size_t)r * G + tid] = __float2half_rn(total[0]);
        a.y[(size_t)r * G + tid + G / 2] = __float2half_rn(total[1]);
    }
}

// ---------------------------------------------------------------- pieces

// N warps, R block-rows laid end to end: warp W has [W*R/N, (W+1)*R/N), the fraction of a block-row being that fraction of
// its list entries, in units of 8.  N >= R: a warp has part of one block-row, or the end of one and the start of the next.
// The warps' sums meet in shared memory, added in warp order; those of CTAs that share a block-row in the workspace (calls are
// bit-reproducible).
// What bounds it at 28672 x 8192 and 50 % (15.8 us; clock stamps): x, masks and list 2.4 us, then the code stream at 5.8 TB/s
// until the CTAs end between 11.6 and 13.9 us (the memory does not serve all SMs alike), sums and exchange 1.4.  The exchange
// as partial sums, a fence and a counter per block-row, and the slots fetched from a busy memory, took 3 us (17.65).  Whole
// warps instead of fractions of a block-row, with the list as words, x in them: 1 % less on average, 5 to 10 % more for 24-byte blocks.
template <int G, int BITS, int MODE>
__global__ void __launch_bounds__(kPieceWarps * 32, 1)
gemv_pieces_kernel(const GemvArgs a)
{
    using Ring = PieceRing<G, BITS, MODE>;
    constexpr int B = G * BITS / 8, CH = Ring::CH, EPL = CH / 32, D = Ring::D, NW = kPieceWarps, kThreads = NW * 32;
    constexpr bool FUSED = MODE == kModeFused, LIST = MODE == kModeList;
    using Smem = PieceSmem<G, BITS, MODE>;

    extern __shared__ __align__(16) unsigned char smem_raw[];
    Smem& sm = *reinterpret_cast<Smem*>(smem_raw);
    typename Smem::Loop& lp = *reinterpret_cast<typename Smem::Loop*>(sm.area);
    const int tid = threadIdx.x, lane = tid & 31;
    const int warp = __shfl_sync(0xffffffffu, tid >> 5, 0);
    const int n = a.n;
    const unsigned R = (unsigned)a.R, N = a.warps, cta = blockIdx.x;

    prefetch_inputs<kThreads>(a, tid);
    // (a hint too: the slots between this CTA and the one before it, which the code stream of other calls has driven from L2; an
    // exchange that had to fetch them from a busy memory took 1 to 2 us longer)
    if (cta > 0u && tid < G / 16) asm volatile("prefetch.global.L2::evict_last [%0];" ::"l"(a.slots + (size_t)(cta - 1u) * G + 16 * tid));
    const typename MmaStage<G, BITS>::Lane ll(lane);
    const unsigned stage0 = smem_u32(&lp.stage[warp][0]);
    constexpr unsigned kStageBytes = (unsigned)sizeof(Stage<G, BITS, Ring>), kRing = D * kStageBytes;
    const unsigned ent_base = smem_u32(&sm.ent[0]);
    const unsigned short* const xg = reinterpret_cast<const unsigned short*>(a.x);
    // this warp's piece: from fraction part0 / N of block-row row0 to part1 / N of row1
    const unsigned W = cta * NW + (unsigned)warp;
    const unsigned row0 = magic_div(W * R, N, a.magic_w), part0 = W * R - row0 * N;
    const unsigned row1 = magic_div((W + 1u) * R, N, a.magic_w), part1 = (W + 1u) * R - row1 * N;
    const unsigned last_row = part1 > 0u ? row1 : row1 - 1u;

    {
        // (as in gemv_kernel; here large matrices gain from the codes too: 28672 x 8192 25.5 -> 25.3 us, 24-byte blocks 14336 x 8192 18.5 -> 18.2)
        const size_t all = (size_t)R * (size_t)n, c0 = all * W / N, here = all * (W + 1u) / N - c0;
        if (MODE != kModeDense || a.small) prefetch_l2(a.meta + c0, 4 * here, lane, 32);
        if (MODE == kModeDense) prefetch_l2(a.codes + c0 * B, min(here, (size_t)((D - 1) * CH)) * B, lane, 32);
    }
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");

    Scan<NW> scan(sm.area, a.thr, n, lane, warp);            // (fused calls only)
    int count = n;
    if (LIST) count = (int)ld_global_u32(a.count);
    const bool lost = LIST && count < 0;
    if (lost) {
        count = 0;
        if (blockIdx.x == 0 && tid == 0) atomicExch(a.status, 1u);
    }
    if (FUSED) count = scan.scan_x(a.x);
    const unsigned units = (unsigned)(count + 7) >> 3;
    int first = 8 * (int)magic_div(part0 * units, N, a.magic_w), end = 8 * (int)magic_div(part1 * units, N, a.magic_w);
    if (FUSED) {
        if (cta == 0 && tid == 0) *a.count_out = count;
        if (a.static_partition) {
            // ablation (see above): the fraction of a block-row is a fraction of its columns
            first = scan.position((int)magic_div(part0 * (unsigned)n, N, a.magic_w));
            end = scan.position((int)magic_div(part1 * (unsigned)n, N, a.magic_w));
        }
        // every CTA writes its share of idx
        const unsigned P = gridDim.x;
        scan.build(sm.ent, 0, count, a.idx_out, 8 * (int)magic_div(cta * units, P, a.magic_p),
                   min(8 * (int)magic_div((cta + 1u) * units, P, a.magic_p), count));
        __syncthreads();                 // the list is in place, and the ring may overwrite x
    }
    if (part1 == 0u) end = count;        // of the piece's last block-row

    // A place in the piece: entries from pos on, of those below hi, of block-row `row`
    struct Cursor {
        unsigned row;
        int pos, hi;
    };
    auto advance = [&](Cursor& c) {
        c.pos += CH;
        if (c.pos >= c.hi) {
            ++c.row;
            c.pos = 0;
            c.hi = c.row < last_row ? count : c.row == last_row ? end : 0;   // (0: past the end)
        }
    };
    Cursor at{row0, first, row0 < last_row ? count : end};   // where the copies stand
    if (at.pos >= at.hi) advance(at);    // (nothing of the first block-row: the ablation, or an empty list)
    const uint8_t* row_codes = a.codes + (size_t)at.row * (size_t)n * B;
    const unsigned* row_meta = a.meta + (size_t)at.row * (size_t)n;

    // given list: the columns of the lane's entries in the chunks the copies come to next, fetched kAhead chunks early
    constexpr int kAhead = 3;
    int coming[kAhead][EPL] = {};
    Cursor ahead = at;
    auto fetch_ahead = [&](int d) {
        if (ahead.pos < ahead.hi) {
#pragma unroll
            for (int q = 0; q < EPL; ++q) coming[d][q] = (int)ld_global_u32(a.idx + min(ahead.pos + 32 * q + lane, ahead.hi - 1));
        }
        advance(ahead);
    };
    if (LIST) {
#pragma unroll
        for (int d = 0; d < kAhead; ++d) fetch_ahead(d);
    }
    unsigned xv[D][EPL];                 // the x values of the chunks in flight, the oldest first
#pragma unroll
    for (int i = 0; i < D * EPL; ++i) xv[i / EPL][i % EPL] = 0;
    unsigned ri = 0;
    auto issue = [&]() {                 // the copies of the next chunk, if there is one
#pragma unroll
        for (int i = 0; i < D * EPL; ++i) xv[i / EPL][i % EPL] = i < (D - 1) * EPL ? xv[(i / EPL + 1) % D][i % EPL] : 0u;   // (0 past the end)
        if (at.pos < at.hi) {
            unsigned col[EPL];
#pragma unroll
            for (int q = 0; q < EPL; ++q) {           // (past the end: the last entry again, with x = 0)
                const int e = at.pos + 32 * q + lane, in = min(e, at.hi - 1);
                col[q] = LIST ? (unsigned)coming[0][q] : FUSED ? lds_u16(ent_base + 2u * (unsigned)in) : (unsigned)in;
                xv[D - 1][q] = ld_global_u16_if(e < at.hi, xg + col[q]);
            }
            copy_chunk<G, BITS, Ring>(stage0 + ri, row_codes, row_meta, col, lane, false);
            ri = ri + kStageBytes == kRing ? 0u : ri + kStageBytes;
            const unsigned row = at.row;
            advance(at);
            if (at.row != row) {
                row_codes += (size_t)n * B;
                row_meta += n;
            }
            if (LIST) {
#pragma unroll
                for (int i = 0; i < (kAhead - 1) * EPL; ++i) coming[i / EPL][i % EPL] = coming[i / EPL + 1][i % EPL];
                fetch_ahead(kAhead - 1);
            }
        }
        cp_async_commit();
    };
    const bool work = at.pos < at.hi;
#pragma unroll 1
    for (int d = 0; d < D - 1; ++d) issue();

    Product<G, BITS, Ring> product(smem_u32(&lp.b[warp][0][0]), lane);
    unsigned rc = 0;                     // the stage of chunk i
    if (work) {
        cp_async_wait<D - 2>();
        __syncwarp();
        product.begin(stage0, xv[1]);
    }
    int pos = first;
#pragma unroll 1
    for (unsigned row = row0;; ++row) {
        const int hi = row < last_row ? count : end;
#pragma unroll 1
        for (; pos < hi; pos += CH) {
            issue();
            const unsigned rn = rc + kStageBytes == kRing ? 0u : rc + kStageBytes;
            cp_async_wait<D - 2>();
            __syncwarp();
            product.multiply(stage0 + rc, ll, stage0 + rn, xv[1]);
            rc = rn;
        }
        product.hand_over(lp.red[row - row0][warp], &lp.red_z[row - row0][warp]);
        if (row == last_row) break;
        pos = 0;
        product.clear();
    }
    cp_async_wait<0>();
    __syncthreads();

    // ---- The warps' sums of a block-row, a thread per row of it, in warp order; then the CTAs' sums.
    const int j = tid % G, group = tid / G, low = j % (G / 2);
    const unsigned W0 = cta * NW;
    const unsigned begin_row = magic_div(W0 * R, N, a.magic_w), end_row = magic_div((W0 + NW) * R + N - 1u, N, a.magic_w);
#pragma unroll 1
    for (unsigned r = begin_row + (unsigned)group; r < end_row; r += kThreads / G) {
        // warps fw .. lw of the grid have part of r: the first one as its last block-row, unless it begins there
        const unsigned fw = magic_div(r * N, R, a.magic_r), lw = magic_div((r + 1u) * N + R - 1u, R, a.magic_r) - 1u;
        const int w0 = (int)max(fw, W0) - (int)W0, w1 = (int)min(lw - W0, NW - 1u), second = fw * R < r * N ? (int)fw - (int)W0 : -1;
        float v0 = 0.0f, v1 = 0.0f, z = 0.0f;
#pragma unroll
        for (int w = 0; w < NW; ++w) {
            const int s = w == second ? 1 : 0;   // (loads without a condition, so that they go together)
            const float2 cz = lp.red_z[s][w];
            const float r0 = lp.red[s][w][low], r1 = lp.red[s][w][low + G / 2];
            if (w >= w0 && w <= w1) {
                v0 += r0 * cz.x;
                v1 += r1 * cz.x;
                z += cz.y;
            }
        }
        v1 = (v1 - ((low & 1) ? v0 : 0.0f)) * 0.0625f;   // (see add_warps)
        float v = (j < G / 2 ? v0 : v1) + z;
        // CTAs c0 .. c1 share r: their sums are added along a tree over their numbers, whose node between CTAs b - 1 and b is
        // slot b - 1 of the workspace.  Of the two that meet there the one that comes second takes the other's sum (a value and
        // a mark in one word, exchanged: no fence, no counter, nobody waits) and goes on; the order of arrival decides who
        // adds, not what is added.
        const unsigned c0 = fw / NW, c1 = lw / NW;
        bool mine = true;
#pragma unroll 1
        for (unsigned step = 1; mine && step <= c1 - c0; step *= 2) {
            const unsigned node = ((cta - c0) / (2 * step) * 2 + 1) * step;   // first CTA of the right half, from c0
            if (node > c1 - c0) continue;                                     // (there is none)
            unsigned long long* const slot = a.slots + (size_t)(c0 + node - 1u) * G + j;
            const unsigned long long other = atomicExch(slot, (unsigned long long)kSlotMark << 32 | __float_as_uint(v));
            mine = (unsigned)(other >> 32) == kSlotMark;
            if (mine) {
                v += __uint_as_float((unsigned)other);
                __stcg(slot, 0ull);
            }
        }
        if (mine) a.y[(size_t)r * G + j] = __float2half_rn(not_a_number_if(lost, v));
    }
}

// ---------------------------------------------------------------- host side

// ---------------------------------------------------------------- checked mode
// spqt_set_debug(1): before a sparse GEMV the index list is checked on the device (count in
// [0, n], every index in [0, n), no index twice for n up to kDebugBits).  A bad list sets the
// workspace's status word to 2 and the GEMV then runs with a count of 0 (y = 0) instead of reading
// wherever the indices point.  Two small extra launches per call; state is per device, not per stream.
constexpr int kDebugBits = 1 << 20;
static __device__ unsigned g_debug_bitmap[kDebugBits / 32];  // all zero between calls
static __device__ int g_debug_count;                         // the count the GEMV is given
static __device__ int g_debug_bad;                           // verdict of the call being checked
static int g_debug = 0;

__global__ void debug_mark_kernel(const int32_t* __restrict__ idx, const int32_t* __restrict__ count, int n,
                                  int* __restrict__ status)
{
    const int c = *count;
    bool bad = (c < 0 || c > n) && blockIdx.x == 0 && threadIdx.x == 0;
    const int lim = c < 0 ? 0 : (c > n ? n : c);  // idx holds n entries at most
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < lim; i += gridDim.x * blockDim.x) {
        const int k = idx[i];
        if (k < 0 || k >= n) {
            bad = true;
        } else if (n <= kDebugBits) {
            const unsigned bit = 1u << (k & 31);
            if (atomicOr(&g_debug_bitmap[k >> 5], bit) & bit) bad = true;  // seen before
        }
    }
    if (bad) {
        atomicExch(status, 2);       // sticky, for the caller
        atomicExch(&g_debug_bad, 1); // this call's verdict
    }
}

__global__ void debug_clear_kernel(const int32_t* __restrict__ idx, const int32_t* __restrict__ count, int n)
{
    const int c = *count;
    const int lim = c < 0 ? 0 : (c > n ? n : c);
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < lim; i += gridDim.x * blockDim.x) {
        const int k = idx[i];
        if (k >= 0 && k < n && n <= kDebugBits) g_debug_bitmap[k >> 5] = 0u;
    }
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        g_debug_count = g_debug_bad ? 0 : c;
        g_debug_bad = 0;  // ready for the next checked call
    }
}

// Launches the two kernels; returns the device address of the count the GEMV must use.
static spqt_status debug_check(const int32_t* idx, const int32_t* count, int n, int* status, cudaStream_t s,
                               const int32_t** checked_count)
{
    static int* count_addr[64] = {};
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return SPQT_ERR_CUDA;
    if (count_addr[dev] == nullptr) {
        void* p = nullptr;
        if (cudaGetSymbolAddress(&p, g_debug_count) != cudaSuccess || p == nullptr) return SPQT_ERR_CUDA;
        count_addr[dev] = static_cast<int*>(p);
    }
    const int blocks = n < 256 * 64 ? (n + 255) / 256 : 64;
    debug_mark_kernel<<<blocks, 256, 0, s>>>(idx, count, n, status);
    debug_clear_kernel<<<1, 256, 0, s>>>(idx, count, n);
    if (cudaGetLastError() != cudaSuccess) return SPQT_ERR_CUDA;
    count_launch(2);
    *checked_count = count_addr[dev];
    return SPQT_OK;
}

struct FusedArgs {
    float t;
    int32_t* idx_out;
    int32_t* count_out;
};

// Grid sizes found by spqt_autotune, per (shape, format, kind of call).  Process-wide, small, searched
// linearly; not thread-safe (like spqt_set_tuning).
struct TunedEntry {
    int m, n, bits, group, mode, ctas;
};
constexpr int kMaxTuned = 256;
static TunedEntry g_tuned[kMaxTuned];
static int g_tuned_count = 0;

static int tuned_ctas(const Format& f, int mode)
{
    for (int i = 0; i < g_tuned_count; ++i) {
        const TunedEntry& e = g_tuned[i];
        if (e.m == f.m && e.n == f.n && e.bits == f.bits && e.group == f.group && e.mode == mode) return e.ctas;
    }
    return 0;
}

static void store_tuned(const Format& f, int mode, int ctas)
{
    for (int i = 0; i < g_tuned_count; ++i) {
        TunedEntry& e = g_tuned[i];
        if (e.m == f.m && e.n == f.n && e.bits == f.bits && e.group == f.group && e.mode == mode) {
            e.ctas = ctas;
            return;
        }
    }
    if (g_tuned_count < kMaxTuned) g_tuned[g_tuned_count++] = TunedEntry{f.m, f.n, f.bits, f.group, mode, ctas};
}

// How many clusters of k CTAs the device holds at once with `smem` bytes each (asked once per kernel, cluster size and device).
template <int G, int BITS, int MODE>
static int max_clusters(int k, int smem, bool alone, int sms, int dev)
{
    static int known[64][2][kMaxSplit + 1] = {};
    int& at_once = known[dev][alone ? 1 : 0][k];
    if (at_once == 0) {
        cudaLaunchAttribute attr[1];
        attr[0].id = cudaLaunchAttributeClusterDimension;
        attr[0].val.clusterDim.x = k;
        attr[0].val.clusterDim.y = 1;
        attr[0].val.clusterDim.z = 1;
        cudaLaunchConfig_t cfg = {};
        cfg.gridDim = dim3((unsigned)(k * kCtasPerSm * sms));
        cfg.blockDim = dim3(256);
        cfg.dynamicSmemBytes = smem;
        cfg.attrs = attr;
        cfg.numAttrs = 1;
        int can = 0;
        if (cudaOccupancyMaxActiveClusters(&can, gemv_kernel<G, BITS, MODE, kCluster, 8>, &cfg) != cudaSuccess) (void)cudaGetLastError();
        at_once = can > 0 ? can : 1;
    }
    return at_once;
}

template <int G, int BITS, int MODE>
static spqt_status launch_gemv(const Format& f, const void* codes, const void* meta, const void* x,
                               const int32_t* idx, const int32_t* count, void* y, void* workspace,
                               cudaStream_t s, FusedArgs fa)
{
    constexpr int kAlone = 120 * 1024;   // shared memory that keeps a second CTA of 8 warps off the SM
    // (a given list counts its clusters with the size of the fused call: the same slices, the same sums)
    constexpr int kSlices = MODE == kModeList ? kModeFused : MODE;
    constexpr int kSmem = (int)sizeof(GemvSmem<G, BITS, kSlices, kCluster, 8>), kSmemPlain = (int)sizeof(GemvSmem<G, BITS, MODE, kPlain, 8>);
    constexpr int kWideSlice = BITS == 4 ? 16 : 8;   // warps of a slice's CTA where there are more than 8 (see wide_slices)
    constexpr int kSmem16 = (int)sizeof(GemvSmem<G, BITS, MODE, kPlain, 16>), kSmemWideSlice = (int)sizeof(GemvSmem<G, BITS, MODE, kCluster, kWideSlice>);
    constexpr int kSmemPieces = (int)sizeof(PieceSmem<G, BITS, MODE>);
    constexpr int kDenseChunk = RowRing<G, MODE>::CH;
    static_assert(sizeof(GemvSmem<G, BITS, MODE, kCluster, 8>) <= kSmem && sizeof(GemvSmem<G, BITS, MODE, kSerial, 8>) <= kSmem && kSmem <= kAlone, "one size for all slices");
    static_assert(kSmem <= 115712 && kSmemPlain <= 115712 && kSmem16 <= 232448 && kSmemWideSlice <= 232448 && kSmemPieces <= 232448, "two CTAs of 8 warps per SM, or one of 16");
    static bool configured[64] = {};
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return SPQT_ERR_CUDA;
    if (!configured[dev]) {
        if (cudaFuncSetAttribute(gemv_kernel<G, BITS, MODE, kPlain, 8>, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemPlain) != cudaSuccess ||
            cudaFuncSetAttribute(gemv_kernel<G, BITS, MODE, kPlain, 16>, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmem16) != cudaSuccess ||
            cudaFuncSetAttribute(gemv_kernel<G, BITS, MODE, kCluster, 8>, cudaFuncAttributeMaxDynamicSharedMemorySize, kAlone) != cudaSuccess ||
            cudaFuncSetAttribute(gemv_kernel<G, BITS, MODE, kSerial, 8>, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmem) != cudaSuccess ||
            (kWideSlice > 8 && cudaFuncSetAttribute(gemv_kernel<G, BITS, MODE, kCluster, kWideSlice>, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemWideSlice) != cudaSuccess) ||
            (kWideSlice > 8 && cudaFuncSetAttribute(gemv_kernel<G, BITS, MODE, kSerial, kWideSlice>, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemWideSlice) != cudaSuccess) ||
            cudaFuncSetAttribute(gemv_pieces_kernel<G, BITS, MODE>, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemPieces) != cudaSuccess)
            return SPQT_ERR_CUDA;
        configured[dev] = true;
    }
    const int sms = sm_count();
    if (sms <= 0) return SPQT_ERR_CUDA;
    // CTAs per block-row: the largest cluster of which all are resident at once with one CTA per SM (4096 x 4096, index
    // collection inside: 6.35 / 5.57 / 4.99 / 4.61 us on 1 / 2 / 3 / 4 CTAs per block-row; 5.2 us on 7, two per SM); where that
    // is no cluster, or one of two or three and twice as many, five or more, fit with two CTAs per SM, the largest with two per
    // SM (9728 x 4096 6.65 us on 1, 6.57 on 3; 6144 x 14336 10.8 on 2, 10.7 on 5; three 5120 x 5120 with one list 19.2 on 3, 18.4
    // on 6; but 8192 x 5120 with the list 6.3 on 4, 6.0 on 2); else one CTA (11776 x 4096 6.8 us, 7.4 on 2, 9.0 on 3).  A CTA has
    // 512 columns of the matrix at least (5632 x 2560 with the list 4.7 us on 2, 4.0 on 5; 2304 x 1024 of 64-row groups, dense:
    // 3.4 us on 4, 2.6 on 1), 768 in a cluster of more than five where two share an SM.  Without a list, whose length nobody knows
    // here, a CTA has one chunk per warp at least (1024 x 1024 2.5 us on 2, 2.1 on 4), a block-row has no more CTAs than it takes for
    // a warp's number of chunks (3072 x 4096 on 5 4.2, on 4 3.8), and 128-row groups go to four with two per SM where two with one
    // fit (7168 x 4096 5.7 on 2, 5.15 on 4).
    int S = 1;
    const int tuned = g_tune_ctas > 0 ? g_tune_ctas : tuned_ctas(f, MODE);
    int P = sms < kMaxPieceCtas ? sms : kMaxPieceCtas;   // CTAs of the pieces kernel
    bool pieces = false;
    // slices that fit the shared memory of a fused call (a given list is sliced the same way: the same sums)
    const int least = MODE == kModeDense || f.n <= kCapPlain || f.n > kMaxFusedN ? 1 : (f.n + kCapSlice - 1) / kCapSlice;
    if (tuned > 0) {
        S = tuned / f.R;
        if (S == 0) {
            pieces = true;
            P = tuned < P ? tuned : P;
        }
    } else {
        // "all resident" with a margin: the previous launch's CTAs leave SM by SM, and the CTAs of a cluster need places on
        // neighbouring SMs at the same time, in odd numbers above all, and the less there is to do the more (figures up to the last two
        // lines from before clusters that nearly fill the device left together, which the lines still hold for; 7168 x 8192 on 5, of
        // which the device holds 56: 11.1 us against 8.3 on 4 and 8.1 on 2; 64-row groups 3328 x 8192 on 5 20 % slower than on 4,
        // at 6656 x 8192 not; 11776 x 8192 on 3, of 93: 13.0 against 10.1 on 1; 4096 x 4096 on 4, of 33: no loss).  Less
        // where there is much to do (4608 x 28672 on 7, of 37, 15.0 us, 16.0 on 6, dense 14.6 / 16.3; at n = 8192 on 7 up to 10 %
        // slower; but 7168 x 14336 on 5, of 56, 16.0 us against 11.4 on 4).  Three with two per SM go to 95 %, lists of a long x to 97 (of
        // 93, dense n = 8192 on 88 / 90 / 92 10.0 / 11.6 / 14.4 us where one CTA or pieces take 11.6; n = 14336 16.3 / 16.9 / 21.6, pieces 16.6
        // to 17.2; with the list 10.9 / 12.0 / 15.4, 13.3 on 1).
        auto resident = [&](int k, bool per_sm) {
            const int most = max_clusters<G, BITS, MODE>(k, per_sm ? kAlone : kSmem, per_sm, sms, dev);
            const long long weights = (long long)G * f.n;   // of a block-row
            if ((k & (k - 1)) == 0) return f.R < most;
            if (!per_sm && k == 3 && 100 * f.R > (weights >= 1300000 && MODE != kModeDense ? 97 : 95) * most) return false;
            if (!per_sm && weights >= 1300000) return 50 * f.R <= 49 * most;
            return per_sm || weights >= 180000ll * k ? 25 * f.R <= 24 * most : 11 * f.R <= 10 * most;
        };
        int one = 1, two = 1;            // CTAs per block-row with one and with two CTAs per SM
        for (int k = 2; k <= kMaxSplit; ++k) {
            if (f.n >= (MODE == kModeDense ? 8 * kDenseChunk : 512) * k && resident(k, true)) one = k;
            if (k > 2 && f.n >= (k > 5 ? 768 : 512) * k && resident(k, false)) two = k;
        }
        S = one == 1 || (one < 4 && two >= (MODE == kModeDense && G == 128 ? 4 : 5) && two >= 2 * one) ? two : one;
        if (MODE == kModeDense) {
            // no more CTAs than it takes for a warp's number of chunks
            auto chunks = [&](int k) { const int columns = k * kDenseChunk * (kWideSlice > 8 && f.n >= 8192 && S == one ? 16 : 8); return (f.n + columns - 1) / columns; };
            int k = 1;
            while (chunks(k) > chunks(S)) ++k;
            S = k;
        }
        // 24-byte blocks without a list and a long x: pieces rather than clusters of three (4800 x 8192 9.8 against 10.3 us)
        if (BITS == 3 && G == 64 && MODE == kModeDense && one == 1 && S <= 3 && f.n >= 8192) S = 1;
        // 24-byte blocks of a list: one CTA rather than three with two per SM (4864 x 8192 at 50 % 9.3 / 10.8 us, list 8.4 / 9.9)
        if (BITS == 3 && G == 64 && MODE != kModeDense && one == 1 && f.n >= 4096) S = 1;
        if (S < least) {
            // A whole block-row does not fit a CTA: clusters of more, smaller slices if all are resident at once (14336 x 11008
            // on 2 14.5 against 16.2 us), otherwise pieces (12288 x 14589 3-bit 19.9 against 25 us with CTAs in two waves).
            if (two >= least) S = two;
            else if (!(BITS == 3 && G == 64) && resident(least, false)) S = least;
            else pieces = true;
        }
        // (24-byte blocks: pieces rather than clusters of no more than the least, 5120 x 20480 19.6 against 17.7 us, unless
        // these have an SM for each CTA: 2048 x 28672 on 4 13.1 against 16.4 us, list 9.7 against 11.2)
        if (BITS == 3 && G == 64 && least >= 3 && (S < least || (S == least && !resident(least, true)))) pieces = true;
        // One CTA per block-row: in the last round of block-rows some SMs have none, or one where they could run two.  Equal
        // pieces of all block-rows pay for sharing block-rows instead (1 us): worth it where what those SMs could do meanwhile,
        // in weights, is enough.  The lines are where the two times cross, between 100 and 448 block-rows and n = 2048 to 14336
        // (pieces against whole, us; every size of the sweep in random matrices):
        //   dense, 4 bits   38 to 50 M: 128-row groups 173 x 4096 11.7 / 13.1, 200 x 4096 12.5 / 13.2, 224 x 4096 13.6 / 13.4;
        //                   64-row groups 200 x 8192 13.1 / 14.5, 224 x 8192 15.0 / 14.9, 256 x 14336 24.4 / 24.9
        //   dense, 3 bits   128-row groups 32 to 40 M: 149 x 2048 7.9 / 8.3, 173 x 2048 8.6 / 8.4, 224 x 4096 14.8 / 15.1; 24-byte
        //                   blocks 25 to 32 M: 173 x 4096 9.9 / 11.2, 200 x 4096 11.2 / 11.2
        //   sparse, 4 bits  128-row groups 65 to 75 M: 149 x 4096 9.1 / 9.6, 173 x 4096 9.6 / 9.4, 224 x 8192 16.3 / 17.1; 64-row
        //                   groups 50 to 65 M: 173 x 8192 12.0 / 12.1, 200 x 8192 12.8 / 12.5
        //   sparse, 3 bits  128-row groups 50 to 65 M: 173 x 4096 10.9 / 11.2, 200 x 4096 11.8 / 11.3; 24-byte blocks 28 M (173 x
        //                   4096 9.2 / 10.6) and always from n = 6144 on
        // The lines are those of the index-collecting call; a given list is cut the same way for the same sums (it would have them
        // at 10 % more or less, but 24-byte blocks at n = 6144 to 8192: 173 x 4096 8.3 / 8.1; and 64-row groups of 4 bits at less:
        // 200 x 8192 11.2 / 11.8, 256 x 8192 13.1 / 15.3).  Above two rounds whole block-rows run one after the other on few SMs:
        // pieces from n = 2048 on (4 bits dense 320 x 4096 17.3 / 21.0, sparse 320 x 2048 9.3 / 9.9, list 8.9 / 8.6; sparse 64-row
        // groups of 4 bits from 4096: 320 x 4096 10.7 / 12.2, and 24-byte blocks dense: 448 x 4096 19.1 / 20.8).
        if (S == 1 && !pieces) {
            const long long idle = (long long)((sms - f.R % sms) % sms) * G * f.n;
            const bool third = f.R > 2 * sms;
            if (MODE == kModeDense) {
                pieces = idle >= (BITS == 4 ? 40000000ll : G == 128 ? 37000000ll : 30000000ll) || (third && (BITS == 4 ? G * f.n >= 1 << 17 : G == 64 && f.n >= 4096));
            } else if (f.R > sms) {
                pieces = idle >= (BITS == 4 ? (G == 128 ? 70000000ll : 66000000ll) : G == 128 ? 60000000ll : 28000000ll) || (BITS == 3 && G == 64 && f.n >= 6144) ||
                         (third && f.n >= (BITS == 4 && G == 64 ? 4096 : 2048));
            }
        }
    }
    const unsigned long long warps = (unsigned long long)P * kPieceWarps;
    // a warp has parts of two block-rows at most, and the arithmetic is 32-bit
    if (warps < (unsigned)f.R || (warps + 1) * (unsigned)(f.R + 2) >= (1ull << 32) || warps * ((unsigned)f.n + 8u) >= (1ull << 32)) pieces = false;
    S = S < least ? least : (S > kMaxSplit ? kMaxSplit : S);
    const int kind = S == 1 ? kPlain : g_no_cluster ? kSerial : kCluster;
    // a grid that fits one CTA per SM is spread that way (two CTAs of a cluster may otherwise share an SM while others idle)
    const bool alone = !pieces && S > 1 && f.R <= max_clusters<G, BITS, MODE>(S, kAlone, true, sms, dev);
    // a long x: 16 warps, for the scan and for the loop (4096 x 14336 at 50 % 8.1 against 8.5 us, dense 7.7 against 8.6; 3072 x
    // 28672 11.5 against 13.0; at n = 4096 and for 3-bit codes no faster)
    const bool wide_slices = alone && kWideSlice > 8 && f.n >= 8192;
    // whole block-rows on one CTA per SM: 16 warps (14336 x 4096 6.2 against 6.5 us, 18944 x 4096 6.4 against 7.0)
    const bool wide = !pieces && kind == kPlain && f.R <= sms;
    const bool cluster = !pieces && kind == kCluster;
    GemvArgs ga;
    ga.codes = static_cast<const uint8_t*>(codes);
    ga.meta = static_cast<const unsigned*>(meta);
    ga.n = f.n;
    ga.R = f.R;
    ga.splits = S;
    ga.together = cluster && 100 * f.R > 91 * max_clusters<G, BITS, MODE>(S, alone ? kAlone : kSmem, alone, sms, dev);
    ga.magic_s = 0xffffffffu / (unsigned)S;
    ga.warps = (unsigned)warps;
    ga.magic_w = 0xffffffffu / ga.warps;
    ga.magic_r = 0xffffffffu / (unsigned)f.R;
    ga.magic_p = 0xffffffffu / (unsigned)P;
    ga.status = static_cast<unsigned*>(status_word(workspace));
    ga.slots = reinterpret_cast<unsigned long long*>(static_cast<unsigned char*>(workspace) + kSlotsOffset);
    ga.x = static_cast<const __half*>(x);
    ga.idx = idx;
    ga.count = count;
    ga.y = static_cast<__half*>(y);
    ga.thr = fa.t != fa.t ? 0x7c00 : fa.t < 0.0f ? 0xbc00 : __half_as_ushort(__float2half_rd(fa.t));
    ga.idx_out = fa.idx_out;
    ga.count_out = fa.count_out;
    ga.static_partition = g_static_partition;
    ga.small = f.blocks * (size_t)f.B <= size_t(64) << 20;
    cudaLaunchConfig_t cfg = {};
    cfg.blockDim = dim3(pieces || wide || wide_slices ? 512 : 256);
    cfg.dynamicSmemBytes = pieces ? kSmemPieces : wide_slices ? kSmemWideSlice : alone && cluster ? kAlone : wide ? kSmem16 : kind == kPlain ? kSmemPlain : kSmem;
    cfg.stream = s;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    attr[1].id = cudaLaunchAttributeClusterDimension;
    attr[1].val.clusterDim.x = S;
    attr[1].val.clusterDim.y = 1;
    attr[1].val.clusterDim.z = 1;
    cfg.gridDim = dim3(pieces ? (unsigned)P : (unsigned)f.R * (unsigned)(cluster ? S : 1));
    cfg.attrs = g_no_pdl ? attr + 1 : attr;
    cfg.numAttrs = (g_no_pdl ? 0 : 1) + (cluster ? 1 : 0);
    auto kernel = pieces             ? gemv_pieces_kernel<G, BITS, MODE>
                  : wide             ? gemv_kernel<G, BITS, MODE, kPlain, 16>
                  : kind == kPlain   ? gemv_kernel<G, BITS, MODE, kPlain, 8>
                  : kind == kCluster ? (wide_slices ? gemv_kernel<G, BITS, MODE, kCluster, kWideSlice> : gemv_kernel<G, BITS, MODE, kCluster, 8>)
                  : wide_slices      ? gemv_kernel<G, BITS, MODE, kSerial, kWideSlice>
                                     : gemv_kernel<G, BITS, MODE, kSerial, 8>;
    const cudaError_t err = cudaLaunchKernelEx(&cfg, kernel, ga);
    count_launch();
    return (err == cudaSuccess && cudaGetLastError() == cudaSuccess) ? SPQT_OK : SPQT_ERR_CUDA;
}

// Everything that can be checked on the host, in the order the header documents; nothing is put on
// the stream before all of it has passed.
static spqt_status check_gemv_args(const void* codes, const void* meta, int m, int n, int bits, int group,
                                   const void* x, const int32_t* idx, const int32_t* count, bool dense, void* y,
                                   void* workspace, size_t ws_bytes, Format* f)
{
    if (!codes || !meta || !x || !y || !workspace) return SPQT_ERR_INVALID_ARG;
    if (!dense && (!idx || !count)) return SPQT_ERR_INVALID_ARG;
    spqt_status st = make_format(m, n, bits, group, f);
    if (st != SPQT_OK) return st;
    if (!aligned(codes, 16) || !aligned(meta, 16) || !aligned(x, 2) || !aligned(y, 2) || !aligned(workspace, 16) ||
        (!dense && (!aligned(idx, 4) || !aligned(count, 4))))
        return SPQT_ERR_ALIGNMENT;
    if (ws_bytes < workspace_bytes(*f)) return SPQT_ERR_WORKSPACE;
    if ((long long)f->R * kMaxSplit >= (1ll << 31)) return SPQT_ERR_UNSUPPORTED;  // grid size
    return SPQT_OK;
}

template <int MODE>
static spqt_status gemv_dispatch(const Format& f, const void* codes, const void* meta, const void* x,
                                 const int32_t* idx, const int32_t* count, void* y, void* workspace, cudaStream_t s, FusedArgs fa)
{
    if (f.bits == 4 && f.group == 128) return launch_gemv<128, 4, MODE>(f, codes, meta, x, idx, count, y, workspace, s, fa);
    if (f.bits == 4 && f.group == 64) return launch_gemv<64, 4, MODE>(f, codes, meta, x, idx, count, y, workspace, s, fa);
    if (f.bits == 3 && f.group == 128) return launch_gemv<128, 3, MODE>(f, codes, meta, x, idx, count, y, workspace, s, fa);
    if (f.bits == 3 && f.group == 64) return launch_gemv<64, 3, MODE>(f, codes, meta, x, idx, count, y, workspace, s, fa);
    return SPQT_ERR_UNSUPPORTED;
}

// The sparse call after its arguments have been checked.
static spqt_status sparse_checked(const Format& f, const void* codes, const void* meta, const void* x,
                                  const int32_t* idx, const int32_t* count, void* y, void* workspace, cudaStream_t s)
{
    if (f.n > kMaxListN) return SPQT_ERR_UNSUPPORTED;
    if (g_debug) {
        spqt_status st = debug_check(idx, count, f.n, static_cast<int*>(status_word(workspace)), s, &count);
        if (st != SPQT_OK) return st;
    }
    return gemv_dispatch<kModeList>(f, codes, meta, x, idx, count, y, workspace, s, FusedArgs{0.0f, nullptr, nullptr});
}

}  // namespace spqt

// Scratch of the entry point that allocates nothing (it holds the status word), resident in every device that loads the library until the process exits.
constexpr size_t kStaticScratchBytes = size_t(1) << 20;
static __device__ __align__(256) unsigned char g_static_scratch[kStaticScratchBytes];

namespace spqt {

// The scratch keeps what the previous call left: the status word has to start at zero, and so have the slots, where two calls that
// were not ordered may have left anything.  A kernel that overlaps with its neighbours in the stream, because a memset does not:
// with one of 164 KB a list call on 4096 x 4096 takes 5.4 us, with one of 4 bytes to 4 KB 8.1, so 4.9 (3.6 with a workspace of the caller).
constexpr int kClearCtas = 40, kClearThreads = 256;
__global__ void __launch_bounds__(kClearThreads) clear_scratch_kernel(uint4* scratch, int pieces)
{
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    for (int i = blockIdx.x * kClearThreads + threadIdx.x; i < pieces; i += kClearCtas * kClearThreads) scratch[i] = make_uint4(0u, 0u, 0u, 0u);
}

static spqt_status launch_clear(void* scratch, int group, cudaStream_t s)
{
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(kClearCtas);
    cfg.blockDim = dim3(kClearThreads);
    cfg.stream = s;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = g_no_pdl ? 0 : 1;
    const int pieces = (int)((kSlotsOffset + slots_bytes(group)) / sizeof(uint4));
    const cudaError_t err = cudaLaunchKernelEx(&cfg, clear_scratch_kernel, static_cast<uint4*>(scratch), pieces);
    count_launch();
    return (err == cudaSuccess && cudaGetLastError() == cudaSuccess) ? SPQT_OK : SPQT_ERR_CUDA;
}

}  // namespace spqt

// Device address of the scratch on the current device (looked up once per device); nullptr on error.
static void* static_scratch_address()
{
    // In host code the array's name is only a handle; the device address has to be asked for,
    // once per device, with that device current.
    static void* scratch_addr[64] = {};
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return nullptr;
    if (scratch_addr[dev] == nullptr) {
        void* p = nullptr;
        if (cudaGetSymbolAddress(&p, g_static_scratch) != cudaSuccess || p == nullptr) return nullptr;
        scratch_addr[dev] = p;
    }
    return scratch_addr[dev];
}

extern "C" {

spqt_status spqt_sparse_gemv(const void* codes, const void* scale_zero,
                             int m, int n, int bits, int group,
                             const void* x, const int32_t* idx, const int32_t* count,
                             void* y, void* workspace, size_t workspace_bytes, void* stream)
{
    using namespace spqt;
    Format f;
    spqt_status st = check_gemv_args(codes, scale_zero, m, n, bits, group, x, idx, count, false, y, workspace,
                                     workspace_bytes, &f);
    if (st != SPQT_OK) return st;
    return sparse_checked(f, codes, scale_zero, x, idx, count, y, workspace, static_cast<cudaStream_t>(stream));
}

spqt_status spqt_sparsify_gemv(const void* codes, const void* scale_zero,
                               int m, int n, int bits, int group,
                               const void* x, float t, int32_t* idx, int32_t* count,
                               void* y, void* workspace, size_t workspace_bytes, void* stream)
{
    using namespace spqt;
    Format f;
    spqt_status st = check_gemv_args(codes, scale_zero, m, n, bits, group, x, idx, count, false, y, workspace,
                                     workspace_bytes, &f);
    if (st != SPQT_OK) return st;
    if (n > kMaxListN) return SPQT_ERR_UNSUPPORTED;
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    if (n > kMaxFusedN) {
        // too long for the in-kernel scan: the same result from the two separate launches
        st = spqt_sparsify(x, n, t, idx, count, stream);
        if (st != SPQT_OK) return st;
        return gemv_dispatch<kModeList>(f, codes, scale_zero, x, idx, count, y, workspace, s, FusedArgs{0.0f, nullptr, nullptr});
    }
    return gemv_dispatch<kModeFused>(f, codes, scale_zero, x, nullptr, nullptr, y, workspace, s, FusedArgs{t, idx, count});
}

spqt_status spqt_dense_gemv(const void* codes, const void* scale_zero,
                            int m, int n, int bits, int group, const void* x,
                            void* y, void* workspace, size_t workspace_bytes, void* stream)
{
    using namespace spqt;
    Format f;
    spqt_status st = check_gemv_args(codes, scale_zero, m, n, bits, group, x, nullptr, nullptr, true, y, workspace,
                                     workspace_bytes, &f);
    if (st != SPQT_OK) return st;
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    const FusedArgs none{0.0f, nullptr, nullptr};
    return gemv_dispatch<kModeDense>(f, codes, scale_zero, x, nullptr, nullptr, y, workspace, s, none);
}

spqt_status spqt_sparse_gemv_static(const void* codes, const void* scale_zero,
                                    int m, int n, int bits, int group,
                                    const void* x, const int32_t* idx, const int32_t* count,
                                    void* y, void* stream)
{
    using namespace spqt;
    Format f;
    spqt_status st = make_format(m, n, bits, group, &f);
    if (st != SPQT_OK) return st;
    if (workspace_bytes(f) > kStaticScratchBytes) return SPQT_ERR_WORKSPACE;  // problem too large for the built-in scratch
    void* const scratch = static_scratch_address();
    if (scratch == nullptr) return SPQT_ERR_CUDA;
    st = check_gemv_args(codes, scale_zero, m, n, bits, group, x, idx, count, false, y, scratch, kStaticScratchBytes, &f);
    if (st != SPQT_OK) return st;
    if (n > kMaxListN) return SPQT_ERR_UNSUPPORTED;
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    st = launch_clear(scratch, f.group, s);
    if (st != SPQT_OK) return st;
    return sparse_checked(f, codes, scale_zero, x, idx, count, y, scratch, s);
}

// Reads a status word (device) into *status_host, waits, and maps it to a return value.
static spqt_status read_status_word(const int* word, int* status_host, cudaStream_t s)
{
    if (cudaMemcpyAsync(status_host, word, sizeof(int), cudaMemcpyDeviceToHost, s) != cudaSuccess) return SPQT_ERR_CUDA;
    if (cudaStreamSynchronize(s) != cudaSuccess) return SPQT_ERR_CUDA;
    return *status_host == 0 ? SPQT_OK : (*status_host == 1 ? SPQT_ERR_TIMEOUT : SPQT_ERR_INVALID_ARG);
}

spqt_status spqt_static_status(int m, int group, int* status_host, void* stream)
{
    if (!status_host || m <= 0 || (group != 64 && group != 128) || m % group) return SPQT_ERR_INVALID_ARG;
    void* const scratch = static_scratch_address();
    if (scratch == nullptr) return SPQT_ERR_CUDA;
    return read_status_word(static_cast<const int*>(spqt::status_word(scratch)), status_host, static_cast<cudaStream_t>(stream));
}

spqt_status spqt_autotune(const void* codes, const void* scale_zero, int m, int n, int bits, int group,
                          const void* x, float t, int32_t* idx, int32_t* count, void* y,
                          void* workspace, size_t workspace_bytes, void* flush, size_t flush_bytes,
                          int* ctas_sparse, int* ctas_dense, void* stream)
{
    using namespace spqt;
    Format f;
    spqt_status st = check_gemv_args(codes, scale_zero, m, n, bits, group, x, idx, count, false, y, workspace,
                                     workspace_bytes, &f);
    if (st != SPQT_OK) return st;
    if (n > kMaxListN) return SPQT_ERR_UNSUPPORTED;
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    const int sms = sm_count();
    if (sms <= 0) return SPQT_ERR_CUDA;
    // candidates: every number of CTAs per block-row of which all are resident at once
    int cand[kMaxSplit], ncand = 0;
    for (int k = 1; k <= kMaxSplit; ++k)
        if (k == 1 || (long long)k * f.R <= kCtasPerSm * sms) cand[ncand++] = k * f.R;
    cudaEvent_t e0, e1;
    if (cudaEventCreate(&e0) != cudaSuccess || cudaEventCreate(&e1) != cudaSuccess) return SPQT_ERR_CUDA;
    const int saved = g_tune_ctas;
    const bool fused_ok = n <= kMaxFusedN;
    int best[2] = {0, 0};
    st = SPQT_OK;
    for (int kind = 0; kind < 2 && st == SPQT_OK; ++kind) {   // 0: index collection + sparse product, 1: dense product
        float best_ms = 0.0f;
        for (int ci = 0; ci < ncand && st == SPQT_OK; ++ci) {
            g_tune_ctas = cand[ci];
            float ms_min = 0.0f;
            for (int rep = 0; rep < 6 && st == SPQT_OK; ++rep) {   // the first repetition warms up
                if (flush && flush_bytes && cudaMemsetAsync(flush, rep, flush_bytes, s) != cudaSuccess) st = SPQT_ERR_CUDA;
                if (cudaEventRecord(e0, s) != cudaSuccess) st = SPQT_ERR_CUDA;
                if (st == SPQT_OK) {
                    if (kind == 0) st = spqt_sparsify_gemv(codes, scale_zero, m, n, bits, group, x, t, idx, count, y, workspace, workspace_bytes, stream);
                    else st = spqt_dense_gemv(codes, scale_zero, m, n, bits, group, x, y, workspace, workspace_bytes, stream);
                }
                if (cudaEventRecord(e1, s) != cudaSuccess || cudaEventSynchronize(e1) != cudaSuccess) st = SPQT_ERR_CUDA;
                float ms = 0.0f;
                if (st == SPQT_OK && cudaEventElapsedTime(&ms, e0, e1) != cudaSuccess) st = SPQT_ERR_CUDA;
                if (rep > 0 && (ms_min == 0.0f || ms < ms_min)) ms_min = ms;
            }
            if (st == SPQT_OK && (best[kind] == 0 || ms_min < best_ms)) {
                best[kind] = cand[ci];
                best_ms = ms_min;
            }
        }
    }
    g_tune_ctas = saved;
    cudaEventDestroy(e0);
    cudaEventDestroy(e1);
    if (st != SPQT_OK) return st;
    store_tuned(f, fused_ok ? kModeFused : kModeList, best[0]);
    if (fused_ok) store_tuned(f, kModeList, best[0]);
    store_tuned(f, kModeDense, best[1]);
    if (ctas_sparse) *ctas_sparse = best[0];
    if (ctas_dense) *ctas_dense = best[1];
    return SPQT_OK;
}

spqt_status spqt_set_debug(int on)
{
    spqt::g_debug = on ? 1 : 0;
    return SPQT_OK;
}

spqt_status spqt_set_tuning(int gemv_ctas, int reserved)
{
    if (gemv_ctas < 0 || reserved < 0 || reserved > 7) return SPQT_ERR_INVALID_ARG;
    spqt::g_tune_ctas = gemv_ctas;
    spqt::g_no_pdl = reserved & 1;
    spqt::g_no_cluster = (reserved >> 1) & 1;
    spqt::g_static_partition = (reserved >> 2) & 1;
    return SPQT_OK;
}

spqt_status spqt_workspace_status(const void* workspace, int m, int group, int* status_host, void* stream)
{
    if (!workspace || !status_host || m <= 0 || (group != 64 && group != 128) || m % group) return SPQT_ERR_INVALID_ARG;
    const void* const word = static_cast<const unsigned char*>(workspace) + spqt::kStatusOffset;
    return read_status_word(static_cast<const int*>(word), status_host, static_cast<cudaStream_t>(stream));
}

}  // extern "C"

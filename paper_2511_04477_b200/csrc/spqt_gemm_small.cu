// Small batch (2..8 decode rows at once: beams, speculative tokens): the sparse product over the UNION
// of the rows' active sets, and its dense twin.  Every active block is fetched once for the whole batch.
//
//   sparsify_rows_kernel    (spqt_sparsify.cu) "active" = |X[b][k]| > t in at least one row b; leaves the list and,
//                           list entry after list entry, the rows' x values (gathered once, not once per block-row).
//   gemm_small_kernel       a thread-block cluster of S CTAs of 8 warps per block-row; CTA s takes the s-th of S equal
//                           slices of the list, every warp a contiguous part of it, streamed through its own ring of
//                           chunks of 32 entries (cp.async).  Lane e of a chunk holds entry e: it multiplies the
//                           batch's x values by the entry's scale and leaves them as fp16 pairs for the tensor cores
//                           (spqt_mma.cuh), which take the codes as they are.  At the end the warps' sums meet in
//                           shared memory and are sent to the CTA that finishes them, which adds them in a fixed order.
//
// What bounds it: instruction issue around the code stream (240 to 280 warp instructions per chunk, 400 with five to eight rows), then the fixed cost of a
// launch.  The batch is the N = 8 side of the matrix instructions, so the instruction count hardly grows with the
// rows (the packed-FMA form before it paid 64 FMAs per chunk and row and two passes from five rows up).
#include <cstddef>

#include "spqt_common.cuh"

#include "spqt_gemv_device.cuh"
#include "spqt_mma.cuh"

namespace spqt {

constexpr int kSmallWarps = 8;      // warps of a CTA
constexpr int kSmallThreads = kSmallWarps * 32;
constexpr int kSmallCtasPerSm = 2;
constexpr int kSmallMaxSplit = 8;   // CTAs of a block-row: the largest portable cluster
constexpr int kSmallChunk = 32;     // list entries per chunk

template <int G, int BITS, int ROWS>
struct SmallSmem {
    static constexpr int kRow = MmaStage<G, BITS>::kRow;
    static constexpr int kDepth = G == 64 ? 5 : (ROWS == 8 ? 3 : 4);   // chunks per warp: 2.2 to 2.7 KB each (G = 64: half that)
    static constexpr int kPad = G + 4;
    struct Stage {
        alignas(16) unsigned char codes[kSmallChunk * kRow];
        alignas(16) unsigned meta[kSmallChunk];                 // (scale, zero) pair of entry e
        alignas(16) unsigned short x[kSmallChunk * ROWS];       // given list: entry after entry; dense: row after row
    };
    Stage stage[kSmallWarps][kDepth];
    alignas(16) unsigned short b[kSmallWarps][ROWS == 8 ? 2 : 1][kSmallChunk][8];   // B of the chunk in work, entry after entry
    alignas(16) float red[kSmallWarps][ROWS][kPad];
    float red_z[kSmallWarps][8];
    alignas(16) float4 others[ROWS * G / 4 + kSmallMaxSplit];   // the cluster's sums of the outputs that this CTA finishes, CTA after CTA
    uint64_t arrival;                                           // and their arrival
};

struct SmallArgs {
    const uint8_t* codes;
    const unsigned* meta;
    int n;
    const uint8_t* x;            // gathered x (ROWS values per list entry), or X itself (DIRECT)
    int ldx, batch;
    const int32_t* idx;          // nullptr: the list is 0, 1, .., n-1
    const int32_t* count;
    __half* Y;
    int ldy;
};

// DIRECT: the dense product with x read from X itself, 8 columns of a row per 16-byte copy (n and ldx multiples of 8,
// X 16-byte aligned); otherwise x comes gathered.
template <int G, int BITS, int ROWS, bool DIRECT>
__global__ void __launch_bounds__(kSmallThreads, kSmallCtasPerSm)
gemm_small_kernel(const SmallArgs a)
{
    using Smem = SmallSmem<G, BITS, ROWS>;
    using Layout = MmaStage<G, BITS>;
    constexpr int B = G * BITS / 8, CH = kSmallChunk, D = Smem::kDepth, SP = Layout::kSp;
    constexpr bool TWO = ROWS == 8;
    constexpr int CB = (B % 16 == 0) ? 16 : 8;          // bytes per copy
    constexpr int NC = CH * B / CB / 32;                // copies per lane and chunk
    constexpr bool kTwice = BITS == 3 && G == 64;       // the 1-bit plane is copied twice
    extern __shared__ __align__(16) unsigned char small_raw[];
    Smem& sm = *reinterpret_cast<Smem*>(small_raw);
    const int tid = threadIdx.x, lane = tid & 31;
    const int warp = __shfl_sync(0xffffffffu, tid >> 5, 0);
    const int g = lane >> 2, t4 = lane & 3;
    const int n = a.n;

    const int split = blockIdx.x, S = gridDim.x, r = blockIdx.y;
    // Four outputs make a group; CTA s of the cluster finishes the s-th of S parts of the groups.
    const int groups = a.batch * (G / 4), from = groups * split / S, mine = groups * (split + 1) / S - from, stride = (groups + S - 1) / S;
    if (S > 1) {
        if (tid == 0) {
            mbar_init(&sm.arrival, 1);
            mbar_expect(&sm.arrival, (unsigned)(16 * (S - 1) * mine));
            mbar_publish();
        }
        __syncwarp();
        cluster_arrive();   // nobody may write to another CTA's shared memory before that CTA runs: arrive now, wait much later
    }
    const typename Layout::Lane ll(lane);
    const unsigned stage0 = smem_u32(&sm.stage[warp][0]);
    constexpr unsigned kStageBytes = (unsigned)sizeof(typename Smem::Stage);
    constexpr unsigned kMetaOff = (unsigned)offsetof(typename Smem::Stage, meta);
    constexpr unsigned kXOff = (unsigned)offsetof(typename Smem::Stage, x);
    const unsigned bbuf = smem_u32(&sm.b[warp][0][0][0]);
    // where this lane's copies of a chunk come from and go to
    int copy_e[NC], copy_part[NC];
    unsigned copy_dst[NC];
#pragma unroll
    for (int q = 0; q < NC; ++q) {
        const int p = q * 32 + lane;
        const int e = p / (B / CB), part = p % (B / CB);
        copy_e[q] = e;
        copy_part[q] = part * CB;
        if (BITS == 4 && G == 128) copy_dst[q] = e * 64 + ((part ^ ((e >> 1) & 3)) << 4);
        else if (BITS == 4) copy_dst[q] = e * 32 + ((part ^ ((e >> 2) & 1)) << 4);
        else copy_dst[q] = e * Layout::kRow + part * CB;
    }
    // x: this lane's share of a chunk (DIRECT: 16 bytes of one row; a row past the batch repeats the last one)
    const uint8_t* const xsrc = DIRECT ? a.x + 2 * ((size_t)min(lane >> 2, a.batch - 1) * a.ldx + 8 * (lane & 3)) : a.x + 2 * ROWS * lane;
    const unsigned xdst = kXOff + (DIRECT ? 16u : 2u * ROWS) * lane;

    const uint8_t* const row_codes = a.codes + (size_t)r * (size_t)n * B;
    const unsigned* const row_meta = a.meta + (size_t)r * (size_t)n;
    // this warp's part [pos, end) of the CTA's slice; in units of 8 entries (DIRECT: 16-byte pieces of x)
    int pos, end;
    auto take_part = [&](int count) {
        const int units = (count + 7) >> 3;
        const int lo = (int)(((long long)split * units) / S), hi = (int)(((long long)(split + 1) * units) / S);
        pos = 8 * (lo + ((hi - lo) * warp) / kSmallWarps);
        end = min(8 * (lo + ((hi - lo) * (warp + 1)) / kSmallWarps), count);
    };
    // While the previous kernel drains (hints, see prefetch_l2): the pairs of the columns that the slice is about, and the first
    // codes where there is no list.
    take_part(n);
    prefetch_l2(row_meta + pos, 4 * (size_t)max(end - pos, 0), lane, 32);
    if (DIRECT || !a.idx) prefetch_l2(row_codes + (size_t)pos * B, (size_t)max(min(end - pos, (D - 1) * CH), 0) * B, lane, 32);

    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    float nothing = 0.0f;                // what the sums of x*zero begin with: not-a-number for a list without a length (see kListLost)
    if (!DIRECT && a.idx) {
        const int count = (int)ld_global_u32(a.count);
        nothing = not_a_number_if(count < 0, 0.0f);
        take_part(max(count, 0));
    }

    float acc[SP][4][4];
    unsigned long long zl[ROWS / 2], scale[ROWS / 2];   // pairs of rows
#pragma unroll
    for (int s = 0; s < SP; ++s)
#pragma unroll
        for (int i = 0; i < 16; ++i) acc[s][i >> 2][i & 3] = 0.0f;
#pragma unroll
    for (int b = 0; b < ROWS / 2; ++b) {
        zl[b] = pack2(nothing, nothing);
        scale[b] = pack2(kMmaNoScale, kMmaNoScale);
    }

    // The columns of the lane's entries in the chunks that the copies come to next (past the end of the part: its last
    // entry again), fetched kAhead chunks early.
    constexpr int kAhead = 4;
    int coming[kAhead];
    int ipos = pos;               // where the copies stand; the arithmetic is D - 1 chunks behind
    auto column_at = [&](int p) -> int {
        const int e = min(p + lane, end - 1);
        return (!DIRECT && a.idx) ? (int)ld_global_u32(a.idx + e) : e;
    };
#pragma unroll
    for (int d = 0; d < kAhead; ++d) coming[d] = pos < end ? column_at(pos + d * CH) : 0;
    unsigned rc = 0, ri = 0;      // byte offsets of the arithmetic's and the copies' stage
    auto issue = [&]() {          // the copies of the next chunk, if there is one
        if (ipos < end) {
            const int col = coming[0];
            const unsigned st = stage0 + ri;
            cp_async_4(st + kMetaOff + 4u * lane, row_meta + col);
            if (DIRECT) {
                if (ROWS == 8 || lane < 16) cp_async_16_left(st + xdst, xsrc + 2 * (size_t)(unsigned)ipos, n - ipos - 8 * (lane & 3));
            } else if (ROWS == 8) {
                cp_async_16(st + xdst, xsrc + (size_t)(unsigned)ipos * 16);
            } else {
                cp_async_8(st + xdst, xsrc + (size_t)(unsigned)ipos * 8);
            }
            // (the chunk's blocks lie one after the other: one address instead of a shuffle and a product for every copy; 28672 x 4096
            // with 4 rows 14.7 -> 14.0 us, 14336 x 4096 with 8 13.0 -> 12.5; 8-byte copies 2 % slower)
            if (DIRECT && CB == 16 && ipos + CH <= end) {
                const uint8_t* s = row_codes + ((size_t)(unsigned)ipos * B + lane * CB);
#pragma unroll
                for (int q = 0; q < NC; ++q) cp_async_16_l2_64(st + copy_dst[q], s + q * 32 * CB);
            } else {
#pragma unroll
                for (int q = 0; q < NC; ++q) {
                    const unsigned cu = (unsigned)__shfl_sync(0xffffffffu, col, copy_e[q]);
                    const uint8_t* s = row_codes + ((size_t)cu * B + copy_part[q]);
                    if (CB == 16) cp_async_16_l2_64(st + copy_dst[q], s);
                    else cp_async_8(st + copy_dst[q], s);
                }
            }
            if (kTwice) cp_async_8(st + lane * Layout::kRow + 24, row_codes + ((size_t)(unsigned)col * B + 16));
            ri = ri + kStageBytes == D * kStageBytes ? 0u : ri + kStageBytes;
            ipos += CH;
#pragma unroll
            for (int d = 0; d + 1 < kAhead; ++d) coming[d] = coming[d + 1];
            coming[kAhead - 1] = column_at(ipos + (kAhead - 1) * CH);
        }
        cp_async_commit();
    };
#pragma unroll 1
    for (int d = 0; d < D - 1; ++d) issue();

    bool empty = true;            // nothing in the sums yet
#pragma unroll 1
    for (; pos < end; pos += CH) {
        issue();
        // ---- B of the chunk that is due: lane e's entry, every row of the batch
        const unsigned st = stage0 + rc;
        cp_async_wait<D - 1>();
        __syncwarp();
        {
            const bool on = pos + lane < end;
            const unsigned mz = lds_u32(st + kMetaOff + 4u * lane);
            const float sf = __half2float(__ushort_as_half((unsigned short)(mz & 0xffffu)));
            const float zf = __half2float(__ushort_as_half((unsigned short)(mz >> 16)));
            unsigned xw[ROWS / 2];   // the entry's x values, two rows a word
            if (DIRECT) {
#pragma unroll
                for (int b = 0; b < ROWS / 2; ++b)
                    xw[b] = lds_u16(st + kXOff + 128u * b + 2u * lane) | (lds_u16(st + kXOff + 128u * b + 64u + 2u * lane) << 16);
            } else if (ROWS == 8) {
                const uint4 v = lds_v4(st + xdst);
                xw[0] = v.x;
                xw[1] = v.y;
                xw[ROWS / 2 - 2] = v.z;
                xw[ROWS / 2 - 1] = v.w;
            } else {
                const uint2 v = lds_v2(st + xdst);
                xw[0] = v.x;
                xw[1] = v.y;
            }
            unsigned long long am[ROWS / 2], p[ROWS / 2];
            float top = 0.0f;
#pragma unroll
            for (int b = 0; b < ROWS / 2; ++b) {
                const unsigned w = on ? xw[b] : 0u;
                const float2 xf = __half22float2(*reinterpret_cast<const __half2*>(&w));
                const unsigned long long x2 = pack2(xf.x, xf.y);
                ffma2(zl[b], x2, pack2(zf, zf));
                am[b] = fmul2(x2, pack2(sf, sf));     // exact
                p[b] = fmul2(am[b], scale[b]);        // powers of two
                float p0, p1;
                unpack2(p[b], p0, p1);
                top = fmaxf(top, fmaxf(fabsf(p0), fabsf(p1)));
            }
            if (__any_sync(0xffffffffu, top > kMmaLimit)) {
                // a larger entry than the range holds: new scales for the rows concerned
                float factor[2] = {1.0f, 1.0f};   // of the lane's columns
#pragma unroll
                for (int b = 0; b < ROWS / 2; ++b) {
                    float av[2], sv[2], fv[2] = {1.0f, 1.0f};
                    unpack2(am[b], av[0], av[1]);
                    unpack2(scale[b], sv[0], sv[1]);
#pragma unroll
                    for (int j = 0; j < 2; ++j) {
                        const unsigned bits = __float_as_uint(av[j]) & 0x7fffffffu;
                        const unsigned m = __reduce_max_sync(0xffffffffu, bits < 0x7f800000u ? bits : 0u);   // finite ones
                        if (__uint_as_float(m) * sv[j] > kMmaLimit) {
                            const float next = __uint_as_float((266u - (m >> 23)) << 23);   // m goes to 2^12 .. 2^13
                            fv[j] = next * power_of_two_inverse(sv[j]);
                            sv[j] = next;
                        }
                    }
                    scale[b] = pack2(sv[0], sv[1]);
                    p[b] = fmul2(am[b], scale[b]);
                    if ((t4 & (ROWS / 2 - 1)) == b) {   // the lane's columns are rows 2b and 2b + 1
                        factor[0] = fv[0];
                        factor[1] = fv[1];
                    }
                }
                if (!empty) {
#pragma unroll
                    for (int s = 0; s < SP; ++s)
#pragma unroll
                        for (int i = 0; i < 16; ++i) {
                            float& v = acc[s][i >> 2][i & 3];
                            if (TWO) {
                                v *= factor[i & 1];
                            } else {   // lanes t4 < 2 have the sums of hi, t4 ^ 2 those of lo
                                float hi = v, rest = 0.0f;
                                rescale_sums(hi, rest, factor[i & 1]);
                                rest = __shfl_xor_sync(0xffffffffu, rest, 2);
                                v = t4 < 2 ? hi : v * factor[i & 1] + rest;
                            }
                        }
                }
            }
            unsigned hi[ROWS / 2], lo[ROWS / 2];
#pragma unroll
            for (int b = 0; b < ROWS / 2; ++b) {
                float p0, p1;
                unpack2(to_halves2(p[b]), p0, p1);
                const __half2 h = __floats2half2_rn(p0, p1);
                const float2 hf = __half22float2(h);
                unsigned long long rest = p[b];
                ffma2(rest, pack2(hf.x, hf.y), pack2(-1.0f, -1.0f));
                unpack2(rest, p0, p1);
                const __half2 l = __floats2half2_rn(p0, p1);
                hi[b] = *reinterpret_cast<const unsigned*>(&h);
                lo[b] = *reinterpret_cast<const unsigned*>(&l);
            }
            if (TWO) {
                sts_v4(bbuf + 16u * lane, make_uint4(hi[0], hi[1], hi[ROWS / 2 - 2], hi[ROWS / 2 - 1]));
                sts_v4(bbuf + 512u + 16u * lane, make_uint4(lo[0], lo[1], lo[ROWS / 2 - 2], lo[ROWS / 2 - 1]));
            } else {
                sts_v4(bbuf + 16u * lane, make_uint4(hi[0], hi[1], lo[0], lo[1]));
            }
            __syncwarp();
        }
        // ---- the product
        unsigned bh[4], bl[4];
        ldsm_x4_trans(bbuf + 16u * lane, bh);
        if (TWO) ldsm_x4_trans(bbuf + 512u + 16u * lane, bl);
        unsigned c[2][SP][4];
#pragma unroll
        for (int ks = 0; ks < 2; ++ks) {
            Layout::load(st, ll, ks, c[ks]);
            if (!TWO) {
#pragma unroll
                for (int s = 0; s < SP; ++s) mma_group(acc[s], c[ks][s], bh + 2 * ks);
            }
        }
        if (TWO) {
#pragma unroll
            for (int s = 0; s < SP; ++s) mma_group_two(acc[s], c[0][s], c[1][s], bh, bl);
        }
        empty = false;
        __syncwarp();
        rc = rc + kStageBytes == D * kStageBytes ? 0u : rc + kStageBytes;
    }
    cp_async_wait<0>();

    // ---- the warps' sums meet in shared memory
    {
        float inv[2] = {0.0f, 0.0f};   // 2^24 / c of the rows in columns 2*t4 and 2*t4 + 1
#pragma unroll
        for (int b = 0; b < ROWS / 2; ++b) {
            float s0, s1;
            unpack2(scale[b], s0, s1);
            if ((t4 & (ROWS / 2 - 1)) == b) {
                inv[0] = 0x1p24f * power_of_two_inverse(s0);
                inv[1] = 0x1p24f * power_of_two_inverse(s1);
            }
        }
#pragma unroll
        for (int s = 0; s < SP; ++s) {
            mma_uncumulate(acc[s]);
            if (TWO) {
#pragma unroll
                for (int i = 0; i < 16; ++i) {
                    const int type = i >> 2, c = i & 3;
                    sm.red[warp][2 * t4 + (c & 1)][Layout::row(s, type, c, g)] = acc[s][type][c] * inv[c & 1];
                }
            } else {
                // columns b and b + 4 are the hi and lo sums of row b: lanes t4 and t4 ^ 2 exchange one half of the
                // tiles each and add
                const bool upper = t4 >= 2;
#pragma unroll
                for (int i = 0; i < 8; ++i) {
                    const int type = i >> 2, c = i & 3;   // kept: types 0, 1 by t4 < 2, types 2, 3 by the others
                    const float keep = upper ? acc[s][type + 2][c] : acc[s][type][c], send = upper ? acc[s][type][c] : acc[s][type + 2][c];
                    const float v = keep + __shfl_xor_sync(0xffffffffu, send, 2);
                    sm.red[warp][2 * (t4 & 1) + (c & 1)][Layout::row(s, type, c, g) + (upper ? 1 : 0)] = v * inv[c & 1];
                }
            }
        }
#pragma unroll
        for (int b = 0; b < ROWS; ++b) {
            float zz[2];
            unpack2(zl[b >> 1], zz[0], zz[1]);
            float z = zz[b & 1];
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) z += __shfl_xor_sync(0xffffffffu, z, o);
            if (lane == 0) sm.red_z[warp][b] = z;
        }
    }
    __syncthreads();
    // A group by a thread: the warps' sums in warp order, then the CTAs' in CTA order.  The CTAs send their sums to the shared
    // memory of the one that finishes them, which counts the bytes: nobody waits for anything but its own data (barriers of
    // the cluster before and after reading each other's shared memory took 0.5 to 0.9 us longer: 4096 x 14336, 8 rows dense 13.1
    // against 12.1 us, 1024 x 4096, 4 rows dense 3.8 against 3.3).
    if (S > 1) cluster_wait();           // (every CTA of the cluster runs)
    if (tid >= groups) return;
    const int b = tid / (G / 4), j = tid % (G / 4) * 4;
    float4 v = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
    float z = 0.0f;
#pragma unroll
    for (int w = 0; w < kSmallWarps; ++w) {
        const float4 u = *reinterpret_cast<const float4*>(&sm.red[w][b][j]);
        v.x += u.x;
        v.y += u.y;
        v.z += u.z;
        v.w += u.w;
        z += sm.red_z[w][b];
    }
    v.x += z;
    v.y += z;
    v.z += z;
    v.w += z;
    if (S > 1) {
        const int owner = ((tid + 1) * S - 1) / groups;
        if (owner != split) {
            const unsigned dst = smem_u32(&sm.others[split * stride + tid - groups * owner / S]);
            st_async_f32x4(cluster_map(dst, (unsigned)owner), v, cluster_map(smem_u32(&sm.arrival), (unsigned)owner));
            return;
        }
        const float start = mbar_wait_cluster(&sm.arrival, 0u) ? 0.0f : __int_as_float(0x7fffffff);
        float4 sum = make_float4(start, start, start, start);
#pragma unroll
        for (int q = 0; q < kSmallMaxSplit; ++q) {
            if (q < S) {
                const float4 u = q == split ? v : sm.others[q * stride + tid - from];
                sum.x += u.x;
                sum.y += u.y;
                sum.z += u.z;
                sum.w += u.w;
            }
        }
        v = sum;
    }
    __half* const y = a.Y + (size_t)b * a.ldy + (size_t)r * G + j;
    y[0] = __float2half_rn(v.x);
    y[1] = __float2half_rn(v.y);
    y[2] = __float2half_rn(v.z);
    y[3] = __float2half_rn(v.w);
}

// Workspace: one word per block-row (zero, kept for callers that look at it), then the gathered x: 16 bytes per list
// entry at most, and the chunk a warp may read past the end.  Never less than 64 KB.
inline size_t small_header_bytes(int R) { return (((size_t)R * 4 + 255) / 256) * 256; }
inline size_t small_workspace_bytes(const Format& f)
{
    const size_t need = small_header_bytes(f.R) + ((size_t)f.n + kSmallChunk) * 16;
    return need < 65536 ? 65536 : need;
}

// The records of the dense product when it cannot read X with 16-byte copies: REC values per column.
template <int REC>
__global__ void __launch_bounds__(256) gather_rows_kernel(const unsigned short* X, int ldx, int batch, int n, unsigned short* gathered)
{
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    const int k = blockIdx.x * 256 + threadIdx.x;
    if (k >= n) return;
    unsigned rec[REC / 2];
#pragma unroll
    for (int b = 0; b < REC; b += 2) {
        const unsigned lo = b < batch ? ld_global_u16(X + (size_t)b * ldx + k) : 0u;
        const unsigned hi = b + 1 < batch ? ld_global_u16(X + (size_t)(b + 1) * ldx + k) : 0u;
        rec[b / 2] = lo | (hi << 16);
    }
    if (REC == 8) *reinterpret_cast<uint4*>(gathered + (size_t)k * 8) = make_uint4(rec[0], rec[1], rec[REC / 2 - 2], rec[REC / 2 - 1]);
    else *reinterpret_cast<uint2*>(gathered + (size_t)k * 4) = make_uint2(rec[0], rec[1]);
}

static spqt_status launch_gather_rows(const __half* X, int ldx, int batch, int n, void* gathered, cudaStream_t s)
{
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)((n + 255) / 256));
    cfg.blockDim = dim3(256);
    cfg.stream = s;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = g_no_pdl ? 0 : 1;
    const cudaError_t err = cudaLaunchKernelEx(&cfg, batch <= 4 ? gather_rows_kernel<4> : gather_rows_kernel<8>, reinterpret_cast<const unsigned short*>(X), ldx, batch, n,
                                               static_cast<unsigned short*>(gathered));
    count_launch();
    return (err == cudaSuccess && cudaGetLastError() == cudaSuccess) ? SPQT_OK : SPQT_ERR_CUDA;
}

constexpr int kSmallAlone = 120 * 1024;   // shared memory that keeps a second CTA off the SM

// How many clusters of k CTAs the device holds at once, one or two CTAs per SM (asked once per kernel, cluster size and device).
template <int G, int BITS, int ROWS, bool DIRECT>
static int small_max_clusters(int k, bool alone, int sms, int dev)
{
    constexpr int smem = (int)sizeof(SmallSmem<G, BITS, ROWS>);
    static int known[64][2][kSmallMaxSplit + 1] = {};
    int& at_once = known[dev][alone ? 1 : 0][k];
    if (at_once == 0) {
        cudaLaunchAttribute attr[1];
        attr[0].id = cudaLaunchAttributeClusterDimension;
        attr[0].val.clusterDim.x = k;
        attr[0].val.clusterDim.y = 1;
        attr[0].val.clusterDim.z = 1;
        cudaLaunchConfig_t cfg = {};
        cfg.gridDim = dim3(k, kSmallCtasPerSm * sms);
        cfg.blockDim = dim3(kSmallThreads);
        cfg.dynamicSmemBytes = alone ? kSmallAlone : smem;
        cfg.attrs = attr;
        cfg.numAttrs = 1;
        int can = 0;
        if (cudaOccupancyMaxActiveClusters(&can, gemm_small_kernel<G, BITS, ROWS, DIRECT>, &cfg) != cudaSuccess) (void)cudaGetLastError();
        at_once = can > 0 ? can : 1;
    }
    return at_once;
}

template <int G, int BITS, int ROWS, bool DIRECT>
static spqt_status launch_small(const Format& f, SmallArgs a, cudaStream_t s)
{
    auto kernel = gemm_small_kernel<G, BITS, ROWS, DIRECT>;
    static bool configured[64] = {};
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return SPQT_ERR_CUDA;
    constexpr int smem = (int)sizeof(SmallSmem<G, BITS, ROWS>);
    static_assert(smem <= 115712, "two CTAs per SM");
    if (!configured[dev]) {
        if (cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmallAlone) != cudaSuccess) return SPQT_ERR_CUDA;
        configured[dev] = true;
    }
    const int sms = sm_count();
    if (sms <= 0) return SPQT_ERR_CUDA;
    // CTAs per block-row.  All of them should be resident at once, two per SM: a second wave costs more than the idle slots of a
    // first one (28672 x 4096, 4 rows: 17.4 us on 224 CTAs, 23.6 on 448).  So the largest number of which the device holds R
    // clusters and one more: clusters of 5 to 8 leave SMs over (4608 x 8192, 8 rows, on 8, of which 33 fit, 26 % slower than on
    // 7; 12288 x 2048 on 3, of 93, 46 % slower than on 1).  4096 x 14336, 8 rows dense 33.9 / 20.1 / 16.0 / 13.4 us on 1 / 2 /
    // 4 / 8; 8192 x 28672, 4 rows dense 51.6 / 28.6 / 26.9 us on 1 / 2 / 4.  A CTA has one chunk per warp at least, two where
    // there are more than 32 block-rows (6144 x 1024, 3 rows: 10 % faster on 1 than on 4).  From R = 100 up two put two half
    // block-rows on the busiest SMs, where one whole block-row runs as fast and needs no exchange (14336 x 4096, 8 rows dense:
    // 12.3 against 14.4 us), unless x is long (12800 x 14336, 8 rows 6 %, 64-row groups 6400 x 14336, 3 rows 16 % faster on 2).
    // Without a list, where the same call may come next, odd clusters that nearly fill the device wait for one another, and the best
    // is the least load of an SM: a block-row over k CTAs with an SM each, 1.6 times that where two share one (three with two per
    // SM at most where two are alone: 9216 x 2048, 8 rows 7.1 us on 3, 5.3 on 2; 6912 x 8192 15.0 on 5, 12.7 on 4), and with a long x
    // clusters of four in more than one wave rather than one or two CTAs (11776 x 8192, 8 rows 24.0 on 3, 23.3 on 1, 19.3 on 4).  Over 297
    // sizes the choice is 2 % slower than the best cluster, the largest that fits was 7 %.
    // Nothing keeps the CTAs of a cluster that were counted with an SM each from sharing some: a launch that lets a second CTA onto its
    // SMs starts earlier, which gains more as long as the device spreads the clusters.  It does not where they fill its parts: four
    // from a fourth cluster in one of eight parts on, six from a second one in all of them (2048 x 8192, 8 rows on 16 clusters of
    // 6: 8.4 us, 6.9 with all shared memory; 3328 x 3072, 4 rows on 26 of 4: 4.2 / 3.9; but 1920 x 4096, 4 rows on 15 of 8: 3.4 / 3.75,
    // 2816 x 4096 on 22 of 5 4.2 / 4.3, 5120 x 2048 on 40 of 3 3.7 / 4.0, 9216 x 2048, 8 rows on 72 of 2 5.2 / 5.4).
    int S = 1;
    bool alone = false;
    if (DIRECT || !a.idx) {
        float least = 0.0f;
        for (int k = 1; k <= kSmallMaxSplit && (k == 1 || f.n >= 512 * k); ++k) {
            const bool even = (k & (k - 1)) == 0;
            const int one = k == 1 ? sms : small_max_clusters<G, BITS, ROWS, DIRECT>(k, true, sms, dev);
            const int two = k == 1 ? 2 * sms : small_max_clusters<G, BITS, ROWS, DIRECT>(k, false, sms, dev);
            float load = 0.0f;                // of an SM, in block-rows
            const bool apart = even ? f.R <= one : 10 * f.R <= 9 * one;
            if (apart) load = 1.0f / k;
            else if (k == 2 && f.n < 8192) continue;   // (two halves on the busiest SMs: no less than a whole)
            else if (even ? f.R <= two : 25 * f.R <= 24 * two || (k >= 6 && f.n >= 8192 && f.R < two)) load = 1.6f / k;
            else if (k == 4 && f.n >= 8192 && 2 * f.R > sms && f.R <= sms) load = 2.0f * f.R / (4.0f * two);
            else if (k > 1) continue;
            if (k == 1 || load < least) {
                least = load;
                S = k;
                alone = apart && ((k == 4 && 4 * f.R > 3 * one) || (k == 6 && 11 * f.R >= 8 * one));
            }
        }
    } else {
        for (int k = 2; k <= kSmallMaxSplit; ++k) {
            const int columns = f.R >= 100 ? 8192 : f.R > 32 ? 512 * k : 256 * (k - 1) + 1;
            if (f.n >= columns && f.R < small_max_clusters<G, BITS, ROWS, DIRECT>(k, false, sms, dev)) S = k;
        }
    }
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(S, f.R);
    cfg.blockDim = dim3(kSmallThreads);
    cfg.dynamicSmemBytes = alone ? kSmallAlone : smem;
    cfg.stream = s;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = S;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[1].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = g_no_pdl ? 1 : 2;
    const cudaError_t err = cudaLaunchKernelEx(&cfg, kernel, a);
    count_launch();
    return (err == cudaSuccess && cudaGetLastError() == cudaSuccess) ? SPQT_OK : SPQT_ERR_CUDA;
}

template <int G, int BITS>
static spqt_status launch_small_format(const Format& f, const SmallArgs& a, bool direct, cudaStream_t s)
{
    // up to four rows: (hi, lo) side by side in the eight columns, half the matrix instructions
    if (a.batch <= 4) return direct ? launch_small<G, BITS, 4, true>(f, a, s) : launch_small<G, BITS, 4, false>(f, a, s);
    return direct ? launch_small<G, BITS, 8, true>(f, a, s) : launch_small<G, BITS, 8, false>(f, a, s);
}

static spqt_status small_entry(const void* codes, const void* meta, int m, int n, int bits, int group,
                               const void* X, int ldx, int batch, bool dense, float t, int32_t* idx, int32_t* count,
                               void* Y, int ldy, void* workspace, size_t ws_bytes, void* stream)
{
    if (!codes || !meta || !X || !Y || !workspace) return SPQT_ERR_INVALID_ARG;
    if (!dense && (!idx || !count)) return SPQT_ERR_INVALID_ARG;
    if (batch < 1 || batch > 8 || ldx < n || ldy < m) return SPQT_ERR_INVALID_ARG;
    Format f;
    spqt_status st = make_format(m, n, bits, group, &f);
    if (st != SPQT_OK) return st;
    if (!aligned(codes, 16) || !aligned(meta, 16) || !aligned(X, 2) || !aligned(Y, 2) || !aligned(workspace, 16) ||
        (!dense && (!aligned(idx, 4) || !aligned(count, 4))))
        return SPQT_ERR_ALIGNMENT;
    if (ws_bytes < small_workspace_bytes(f)) return SPQT_ERR_WORKSPACE;
    if (f.R > 65535) return SPQT_ERR_UNSUPPORTED;
    if (!dense && n > 65535) return SPQT_ERR_UNSUPPORTED;  // the index collection keeps 64 flag bits per lane
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    const __half* Xh = static_cast<const __half*>(X);
    char* const ws = static_cast<char*>(workspace);
    SmallArgs a = {};
    a.codes = static_cast<const uint8_t*>(codes);
    a.meta = static_cast<const unsigned*>(meta);
    a.n = n;
    a.ldx = ldx;
    a.batch = batch;
    a.Y = static_cast<__half*>(Y);
    a.ldy = ldy;
    const bool direct = dense && (n & 7) == 0 && (ldx & 7) == 0 && aligned(X, 16);
    if (direct) {
        a.x = reinterpret_cast<const uint8_t*>(Xh);
    } else {
        void* const gathered = ws + small_header_bytes(f.R);
        st = dense ? launch_gather_rows(Xh, ldx, batch, n, gathered, s)
                   : launch_sparsify_rows(Xh, ldx, batch, n, t, idx, count, gathered, s);
        if (st != SPQT_OK) return st;
        a.x = static_cast<const uint8_t*>(gathered);
        a.idx = dense ? nullptr : idx;
        a.count = count;
    }
    if (bits == 4 && group == 128) return launch_small_format<128, 4>(f, a, direct, s);
    if (bits == 4 && group == 64) return launch_small_format<64, 4>(f, a, direct, s);
    if (bits == 3 && group == 128) return launch_small_format<128, 3>(f, a, direct, s);
    return launch_small_format<64, 3>(f, a, direct, s);
}

}  // namespace spqt

extern "C" {

spqt_status spqt_gemm_small_workspace(int m, int n, int bits, int group, size_t* workspace_bytes)
{
    spqt::Format f;
    spqt_status st = spqt::make_format(m, n, bits, group, &f);
    if (st != SPQT_OK) return st;
    if (workspace_bytes) *workspace_bytes = spqt::small_workspace_bytes(f);
    return SPQT_OK;
}

spqt_status spqt_sparse_gemm_small(const void* codes, const void* scale_zero, int m, int n, int bits, int group,
                                   const void* X, int ldx, int batch, float t, int32_t* idx, int32_t* count,
                                   void* Y, int ldy, void* workspace, size_t workspace_bytes, void* stream)
{
    return spqt::small_entry(codes, scale_zero, m, n, bits, group, X, ldx, batch, false, t, idx, count, Y, ldy,
                             workspace, workspace_bytes, stream);
}

spqt_status spqt_dense_gemm_small(const void* codes, const void* scale_zero, int m, int n, int bits, int group,
                                  const void* X, int ldx, int batch, void* Y, int ldy,
                                  void* workspace, size_t workspace_bytes, void* stream)
{
    return spqt::small_entry(codes, scale_zero, m, n, bits, group, X, ldx, batch, true, 0.0f, nullptr, nullptr, Y, ldy,
                             workspace, workspace_bytes, stream);
}

}  // extern "C"

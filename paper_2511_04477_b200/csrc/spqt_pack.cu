// Offline conversion: group-wise min/max quantization of fp16 weights and the
// zigzag block layout (groups run down G rows of one column; blocks stored
// row-major over (block-row, column)), plus the inverse of the layout step.
#include "spqt_common.cuh"
#include "spqt_gemv_device.cuh"
#include "spqt_quantize.cuh"

namespace spqt {

constexpr int kPackThreads = 128;  // 4 warps, 16 to 64 columns each

// One column by a warp, lane l owning rows l, l+32, ..: anything goes (not-a-number, infinities, a scale so small that
// its rounding lets codes exceed the range).
template <int G, int BITS>
__device__ __noinline__ void convert_column(const __half* __restrict__ col, int ldw, int lane, uint8_t* __restrict__ q_sm, uint8_t* __restrict__ out, __half2* scale_zero)
{
    constexpr int PER_LANE = G / 32, B = G * BITS / 8, QMAX = (1 << BITS) - 1;
    float w[PER_LANE];
    float lo = INFINITY, hi = -INFINITY;
#pragma unroll
    for (int u = 0; u < PER_LANE; ++u) {
        w[u] = __half2float(col[(size_t)(lane + 32 * u) * ldw]);
        lo = fminf(lo, w[u]);
        hi = fmaxf(hi, w[u]);
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        lo = fminf(lo, __shfl_xor_sync(0xffffffffu, lo, o));
        hi = fmaxf(hi, __shfl_xor_sync(0xffffffffu, hi, o));
    }
    lo = __fadd_rn(lo, 0.0f);
    hi = __fadd_rn(hi, 0.0f);
    const __half sh = __float2half_rn(__fdiv_rn(__fsub_rn(hi, lo), (float)QMAX));
    const float sf = __half2float(sh);
    __syncwarp();
#pragma unroll
    for (int u = 0; u < PER_LANE; ++u)
        q_sm[lane + 32 * u] = (uint8_t)((sf != 0.0f) ? min(__float2int_rn(__fdiv_rn(__fsub_rn(w[u], lo), sf)), QMAX) : 0);
    __syncwarp();
    for (int b = lane; b < B; b += 32) {
        unsigned v = 0;
        if (BITS == 4) {
            v = q_sm[b] | (q_sm[b + G / 2] << 4);
        } else if (b < G / 4) {
            for (int u = 0; u < 4; ++u) v |= (q_sm[b + u * (G / 4)] & 3u) << (2 * u);
        } else {
            for (int u = 0; u < 8; ++u) v |= ((q_sm[b - G / 4 + u * (G / 8)] >> 2) & 1u) << u;
        }
        out[b] = (uint8_t)v;
    }
    if (lane == 0) *scale_zero = __halves2half2(sh, __float2half_rn(lo));
}

// A lane converts 64 rows of NC columns in registers, two fp32 operations per instruction: two neighbouring columns, or one and
// neighbouring rows.  With G = 128 two lanes share a column: of every 16 rows lane half h has those from 8h on.
// v[i], NC = 2: row (G/8)*u + 8h + j, u = i / 8, j = i % 8, of both columns; NC = 1: rows j and j + 1, u = i / 4, j = 2*(i % 4).
// The codes of a warp's blocks meet in shared memory (`mine`) and leave in 16-byte pieces, neighbouring lanes to neighbouring
// places.  k0: the warp's first column; `off`: what a row's start is from W.
template <int G, int BITS, int NC>
struct PackTile {
    static constexpr int B = G * BITS / 8, Q = (1 << BITS) - 1, H = G / 64, kCols = 32 * NC / H;
    static constexpr int CB = B % 16 == 0 ? 16 : 8;  // bytes per piece of a block
    static constexpr int kPieces = B / CB;           // of a block

    static __device__ __forceinline__ void convert(const __half2* v, const __half* __restrict__ W, int r, int k0, int n, int ldw, int lane, unsigned char* mine,
                                                   uint8_t* codes, __half2* scale_zero)
    {
        const int h = lane / (32 / H), column = NC * (lane % (32 / H)), k = k0 + column;
        const bool on = k < n, on1 = k + NC - 1 < n;   // (the lane's first and last column)
        // place of byte b of the warp's blocks: 16-byte pieces so that lanes 128 or 64 bytes apart hit different banks
        auto place = [](int b) { return CB == 16 ? ((b >> 4) ^ ((b >> 7) & 7)) * 16 + (b & 15) : b; };
        // minimum and maximum: exact in fp16 (the maximum is not-a-number if any weight is)
        __half2 lo2 = v[0], hi2 = v[0];
#pragma unroll
        for (int i = 1; i < 32 * NC; ++i) {
            lo2 = __hmin2(lo2, v[i]);
            hi2 = __hmax2_nan(hi2, v[i]);
        }
        if (H == 2) {
            lo2 = __hmin2(lo2, __shfl_xor_sync(0xffffffffu, lo2, 16));
            hi2 = __hmax2_nan(hi2, __shfl_xor_sync(0xffffffffu, hi2, 16));
        }
        if (NC == 1) {
            lo2 = __hmin2(lo2, __lowhigh2highlow(lo2));
            hi2 = __hmax2_nan(hi2, __lowhigh2highlow(hi2));
        }
        // a zero extreme of either sign counts as +0.0 (x + (+0.0) is x, except that -0.0 becomes +0.0)
        const float2 lo = make_float2(__fadd_rn(__low2float(lo2), 0.0f), __fadd_rn(__high2float(lo2), 0.0f));
        const float2 hi = make_float2(__fadd_rn(__low2float(hi2), 0.0f), __fadd_rn(__high2float(hi2), 0.0f));
        // scale = fp16((max - min) / qmax): one IEEE subtract, one IEEE divide, RN-even
        const __half s0 = __float2half_rn(__fdiv_rn(__fsub_rn(hi.x, lo.x), (float)Q));
        const __half s1 = NC == 2 ? __float2half_rn(__fdiv_rn(__fsub_rn(hi.y, lo.y), (float)Q)) : s0;
        const Divisor2 by(make_float2(__half2float(s0), __half2float(s1)));
        // (false for not-a-number: hi has it if any weight is; for infinities; if codes may exceed the range)
        const bool plain[2] = {__fsub_rn(hi.x, lo.x) * by.inv.x <= (float)Q + 0.25f, __fsub_rn(hi.y, lo.y) * by.inv.y <= (float)Q + 0.25f};
        const float2 minus_lo = make_float2(-lo.x, -lo.y);
        // the codes of four rows from j = jj of u on, a byte each, of every column
        auto four = [&](int u, int jj, unsigned* w) {
            float2 t[2 * NC];
#pragma unroll
            for (int j = 0; j < 2 * NC; ++j) t[j] = round_to_low_bits(by.quotient(add2(__half22float2(v[(8 * u + jj) * NC / 2 + j]), minus_lo)));
            if (NC == 2) {
                w[0] = four_bytes(t[0].x, t[1].x, t[2 * NC - 2].x, t[2 * NC - 1].x) & (0x01010101u * Q);
                w[NC - 1] = four_bytes(t[0].y, t[1].y, t[2 * NC - 2].y, t[2 * NC - 1].y) & (0x01010101u * Q);
            } else {
                w[0] = four_bytes(t[0].x, t[0].y, t[1].x, t[1].y) & (0x01010101u * Q);
            }
        };
        auto put = [&](int c, int byte, const unsigned* w) { *reinterpret_cast<uint2*>(mine + place((column + c) * B + byte + 8 * h)) = make_uint2(w[0], w[1]); };
        if (BITS == 4) {
            // byte i: rows i and i + G/2
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                unsigned o[NC][2];
#pragma unroll
                for (int q = 0; q < 2; ++q) {
                    unsigned l[NC], t[NC];
                    four(u, 4 * q, l);
                    four(u + 4, 4 * q, t);
#pragma unroll
                    for (int c = 0; c < NC; ++c) o[c][q] = l[c] | (t[c] << 4);
                }
#pragma unroll
                for (int c = 0; c < NC; ++c) put(c, (G / 8) * u, o[c]);
            }
        } else {
            // byte b < G/4: the low two bits of rows b + (G/4)*u; byte G/4 + j: the third of rows j + (G/8)*u
            unsigned top[NC][2] = {}, low[NC][2][2] = {};
#pragma unroll
            for (int q = 0; q < 2; ++q)
#pragma unroll
                for (int u = 0; u < 8; ++u) {
                    unsigned l[NC];
                    four(u, 4 * q, l);
#pragma unroll
                    for (int c = 0; c < NC; ++c) {
                        top[c][q] |= ((l[c] >> 2) & 0x01010101u) << u;
                        low[c][u & 1][q] |= (l[c] & 0x03030303u) << (2 * (u >> 1));
                    }
                }
#pragma unroll
            for (int c = 0; c < NC; ++c) {
                put(c, 0, low[c][0]);
                put(c, G / 8, low[c][1]);
                put(c, G / 4, top[c]);
            }
        }
        const size_t blk = (size_t)r * n + k;
        if (h == 0) {
            if (on) scale_zero[blk] = __halves2half2(s0, __float2half_rn(lo.x));                      // exact: lo is an fp16 value
            if (NC == 2 && on1) scale_zero[blk + 1] = __halves2half2(s1, __float2half_rn(lo.y));
        }
        __syncwarp();
        unsigned char* const dst = codes + ((size_t)r * n + k0) * B;
        const int pieces = min(kCols, n - k0) * kPieces;
#pragma unroll
        for (int c = lane; c < kCols * kPieces; c += 32) {
            if (c >= pieces) break;
            if (CB == 16) *reinterpret_cast<uint4*>(dst + c * 16) = *reinterpret_cast<const uint4*>(mine + place(c * 16));
            else *reinterpret_cast<uint2*>(dst + c * 8) = *reinterpret_cast<const uint2*>(mine + place(c * 8));
        }
        // the other columns once more
#pragma unroll 1
        for (int half = 0; half < NC; ++half) {
            unsigned again = __ballot_sync(0xffffffffu, h == 0 && (half == 0 ? on && !plain[0] : on1 && !plain[1]));
            __syncwarp();
            while (again != 0u) {
                const int c = NC * (__ffs((int)again) - 1) + half;
                again &= again - 1u;
                convert_column<G, BITS>(W + (size_t)r * G * ldw + k0 + c, ldw, lane, mine, dst + c * B, scale_zero + (size_t)r * n + k0 + c);
            }
        }
    }
};

// W with rows of 16-byte pieces (W on a 16-byte boundary, ldw a multiple of 8).  A persistent warp takes tiles of 64 rows per
// lane: 128 rows x 32 columns, or 64 x 64, 8 KB.  While a tile is converted, from registers, the next one comes by cp.async
// into the shared memory that it left: 160 KB in flight per SM, and half the instructions of loads by the lane, whose addresses
// take more than the loads (22 instructions for two weights, now 19).  Bound by memory: 28672 x 8192 to 4 bits, 595 MB, alone in
// 105 us = 5.7 TB/s, where loads by the lane, in phases with the rest, took 125 us (and 345 us with an IEEE division per weight); one
// call after the other for longer, under the power limit, 121 and 132 us; from 8 M weights on 5 to 20 % faster, below that the same.
constexpr int kTileCtas = 5;             // per SM
template <int G, int BITS>
__global__ void __launch_bounds__(kPackThreads, kTileCtas)
pack_tiles_kernel(const __half* __restrict__ W, int n, int ldw, int R, uint8_t* codes, __half2* scale_zero)
{
    using Tile = PackTile<G, BITS, 2>;
    constexpr int kRowBytes = 2 * Tile::kCols;       // 64 or 128
    __shared__ __align__(128) unsigned char w_sm[kPackThreads / 32][8192];
    __shared__ __align__(16) unsigned char out_sm[kPackThreads / 32][Tile::kCols * Tile::B];
    const int warp = threadIdx.x / 32, lane = threadIdx.x % 32, h = G == 128 ? lane >> 4 : 0;
    const unsigned across = (unsigned)((n + Tile::kCols - 1) / Tile::kCols), tiles = across * (unsigned)R, step = gridDim.x * (kPackThreads / 32);
    const unsigned tile_sm = smem_u32(w_sm[warp]);
    // rows of 64 bytes: row i is half (i ^ i / 8) & 1 of line i / 2, so that rows 8 apart, which the lane halves read, lie in
    // different banks
    const int part = lane % (kRowBytes / 16), l = lane / (kRowBytes / 16);   // of a copy: 16 bytes of row 4*q*128/G + l
    auto copy = [&](unsigned t) {
        const unsigned r = t / across, k = (t - r * across) * Tile::kCols + 8u * part;
        const __half* src = W + ((size_t)r * G + l) * ldw + k;
        const int left = (int)min((unsigned)n - min(k, (unsigned)n), 8u);
#pragma unroll
        for (int q = 0; q < 16; ++q) {
            const unsigned dst = G == 128 ? tile_sm + 512u * q + 128u * (l >> 1) + 64u * ((l ^ q) & 1) + 16u * part : tile_sm + 512u * q + 16u * lane;
            cp_async_16_left(dst, left > 0 ? src : W, left);
            src += (size_t)(512 / kRowBytes) * ldw;
        }
    };
    unsigned t = blockIdx.x * (kPackThreads / 32) + warp;
    if (t < tiles) copy(t);
    cp_async_commit();
    for (; t < tiles; t += step) {
        cp_async_wait<0>();
        __syncwarp();
        __half2 v[64];
#pragma unroll
        for (int i = 0; i < 64; ++i) {
            const int u = i >> 3, j = i & 7;
            const unsigned w = G == 128 ? lds_u32(tile_sm + 1024u * u + 512u * h + 128u * (j >> 1) + 64u * ((j ^ h) & 1) + 4u * (lane & 15)) : lds_u32(tile_sm + 128u * i + 4u * lane);
            v[i] = *reinterpret_cast<const __half2*>(&w);
        }
        __syncwarp();
        if (t + step < tiles) copy(t + step);
        cp_async_commit();
        const unsigned r = t / across;
        Tile::convert(v, W, (int)r, (int)((t - r * across) * Tile::kCols), n, ldw, lane, out_sm[warp], codes, scale_zero);
        __syncwarp();
    }
}

// Any W: the lanes load their rows themselves.
template <int G, int BITS, int NC>
__global__ void __launch_bounds__(kPackThreads, NC == 2 ? 5 : 6)
pack_kernel(const __half* W, int n, int ldw, uint8_t* codes, __half2* scale_zero)
{
    using Tile = PackTile<G, BITS, NC>;
    __shared__ __align__(16) unsigned char out_sm[kPackThreads / 32][Tile::kCols * Tile::B];

    const int warp = threadIdx.x / 32, lane = threadIdx.x % 32, h = lane / (32 / Tile::H);
    const int r = blockIdx.y;
    const int k0 = (blockIdx.x * (kPackThreads / 32) + warp) * Tile::kCols, k = k0 + NC * (lane % (32 / Tile::H));
    if (k0 >= n) return;
    const __half* const src = W + ((size_t)r * G + 8 * h) * ldw + k;
    const bool on = k < n;               // (NC = 2: n is even)
    __half2 v[32 * NC];
#pragma unroll
    for (int i = 0; i < 32 * NC; ++i) {
        const int row = (G / 8) * (i / (4 * NC)) + (i % (4 * NC)) * (NC == 2 ? 1 : 2);
        if (NC == 2) {
            const unsigned u = on ? __ldcs(reinterpret_cast<const unsigned*>(src + (size_t)row * ldw)) : 0u;
            v[i] = *reinterpret_cast<const __half2*>(&u);
        } else {
            v[i] = __halves2half2(on ? src[(size_t)row * ldw] : __half(0.0f), on ? src[(size_t)(row + 1) * ldw] : __half(0.0f));
            if ((i & 7) == 7) asm volatile("" ::: "memory");   // (not all halves in registers of their own before they are paired)
        }
    }
    Tile::convert(v, W, r, k0, n, ldw, lane, out_sm[warp], codes, scale_zero);
}

// One thread per weight: read its code out of the zigzag buffer.
template <int G, int BITS>
__global__ void unpack_kernel(const uint8_t* __restrict__ codes, int m, int n, uint8_t* __restrict__ q)
{
    constexpr int B = G * BITS / 8;
    const size_t e = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (e >= (size_t)m * n) return;
    const int j = (int)(e / n), k = (int)(e % n);
    const int r = j / G, i = j % G;
    const uint8_t* blk = codes + ((size_t)r * n + k) * B;
    int code;
    if (BITS == 4) {
        code = (i < G / 2) ? (blk[i] & 15) : (blk[i - G / 2] >> 4);
    } else {
        const int low2 = (blk[i % (G / 4)] >> (2 * (i / (G / 4)))) & 3;
        const int top1 = (blk[G / 4 + i % (G / 8)] >> (i / (G / 8))) & 1;
        code = low2 | (top1 << 2);
    }
    q[e] = (uint8_t)code;
}

template <int G, int BITS>
static spqt_status launch_pack(const Format& f, const void* W, int ldw, void* codes, void* scale_zero,
                               cudaStream_t s)
{
    const __half* const w = static_cast<const __half*>(W);
    uint8_t* const c = static_cast<uint8_t*>(codes);
    __half2* const sz = static_cast<__half2*>(scale_zero);
    const uintptr_t at = reinterpret_cast<uintptr_t>(W);
    if ((at & 15) == 0 && (ldw & 7) == 0) {
        const int sms = sm_count();
        if (sms <= 0) return SPQT_ERR_CUDA;
        const long long cols = 4096 / G, warps = kPackThreads / 32;
        const long long ctas = ((f.n + cols - 1) / cols * f.R + warps - 1) / warps, most = (long long)kTileCtas * sms;
        pack_tiles_kernel<G, BITS><<<(unsigned)(ctas < most ? ctas : most), kPackThreads, 0, s>>>(w, f.n, ldw, f.R, c, sz);
    } else {
        const bool pairs = (at & 3) == 0 && ((ldw | f.n) & 1) == 0;   // of columns, as words
        const int cols = kPackThreads * (pairs ? 2 : 1) * 64 / G;
        const dim3 grid((f.n + cols - 1) / cols, f.R);
        auto kernel = pairs ? pack_kernel<G, BITS, 2> : pack_kernel<G, BITS, 1>;
        kernel<<<grid, kPackThreads, 0, s>>>(w, f.n, ldw, c, sz);
    }
    count_launch();
    return cudaGetLastError() == cudaSuccess ? SPQT_OK : SPQT_ERR_CUDA;
}

template <int G, int BITS>
static spqt_status launch_unpack(const Format& f, const void* codes, void* q, cudaStream_t s)
{
    const size_t total = (size_t)f.m * f.n;
    const unsigned blocks = (unsigned)((total + 255) / 256);
    unpack_kernel<G, BITS><<<blocks, 256, 0, s>>>(static_cast<const uint8_t*>(codes), f.m, f.n,
                                                  static_cast<uint8_t*>(q));
    count_launch();
    return cudaGetLastError() == cudaSuccess ? SPQT_OK : SPQT_ERR_CUDA;
}

}  // namespace spqt

extern "C" {

spqt_status spqt_pack(const void* W, int m, int n, int ldw, int bits, int group,
                      void* codes, void* scale_zero, void* stream)
{
    using namespace spqt;
    if (!W || !codes || !scale_zero) return SPQT_ERR_INVALID_ARG;
    Format f;
    spqt_status st = make_format(m, n, bits, group, &f);
    if (st != SPQT_OK) return st;
    if (ldw < n) return SPQT_ERR_INVALID_ARG;
    if (f.R > 65535) return SPQT_ERR_UNSUPPORTED;
    if (!aligned(W, 2) || !aligned(codes, 16) || !aligned(scale_zero, 16))
        return SPQT_ERR_ALIGNMENT;
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    if (bits == 4 && group == 128) return launch_pack<128, 4>(f, W, ldw, codes, scale_zero, s);
    if (bits == 4 && group == 64) return launch_pack<64, 4>(f, W, ldw, codes, scale_zero, s);
    if (bits == 3 && group == 128) return launch_pack<128, 3>(f, W, ldw, codes, scale_zero, s);
    return launch_pack<64, 3>(f, W, ldw, codes, scale_zero, s);
}

spqt_status spqt_unpack(const void* codes, int m, int n, int bits, int group, void* q_u8, void* stream)
{
    using namespace spqt;
    if (!codes || !q_u8) return SPQT_ERR_INVALID_ARG;
    Format f;
    spqt_status st = make_format(m, n, bits, group, &f);
    if (st != SPQT_OK) return st;
    if (((size_t)m * n + 255) / 256 > 0x7fffffffu) return SPQT_ERR_UNSUPPORTED;
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    if (bits == 4 && group == 128) return launch_unpack<128, 4>(f, codes, q_u8, s);
    if (bits == 4 && group == 64) return launch_unpack<64, 4>(f, codes, q_u8, s);
    if (bits == 3 && group == 128) return launch_unpack<128, 3>(f, codes, q_u8, s);
    return launch_unpack<64, 3>(f, codes, q_u8, s);
}

}  // extern "C"

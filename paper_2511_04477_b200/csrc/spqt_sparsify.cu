// Sparse index collection: hidden state x and a threshold t -> the ascending
// list of the entries with |x_k| > t and its length.  Three kernels:
//   sparsify_words_kernel (one row, n <= 65536): a lane looks after pairs of neighbouring entries; one CTA, whose warps' totals meet
//     in shared memory, or above n = 2048 a cluster of 8 CTAs, whose warps send theirs to all of them.
//   sparsify_kernel (one row, n above 65536, or where no cluster can be launched): each warp owns a contiguous segment of x, counts its active entries
//     with __ballot_sync/__popc (the loads of eight groups of 32 entries in flight together), the 32 warp
//     totals are scanned in shared memory, and each warp then writes its indices at its base offset.
//   sparsify_rows_kernel (the small batch, n < 2^16: "active in at least one of B rows"): a cluster of 8 CTAs, which
//     also gathers the rows' values of the listed columns.
// The output order is ascending by construction (no atomics, no arrival order).
#include "spqt_common.cuh"
#include "spqt_gemv_device.cuh"

namespace spqt {

constexpr int kSparsifyThreads = 1024;

__device__ __forceinline__ bool is_active(__half v, float t)
{
    // exact widening; NaN compares false and is therefore never active
    return fabsf(__half2float(v)) > t;
}

constexpr int kClusterCtas = 8;
constexpr int kClusterWarps = 8;

// The totals of a cluster's warps, which every warp sends to every CTA's shared memory.  The CTA's barrier counts their bytes, so
// that a warp waits for the data alone; cluster barriers before and after reading each other's tables took 0.7 to 0.9 us more.
template <int WARPS>
struct ClusterTotals {
    static constexpr unsigned kNone = 1u << 20;       // more than any list has
    int total[WARPS];
    uint64_t arrival;

    // by all threads, before the wait for the previous kernel
    __device__ __forceinline__ void open()
    {
        if (threadIdx.x == 0) {
            mbar_init(&arrival, 1);
            mbar_expect(&arrival, WARPS * 4);
            mbar_publish();
        }
        __syncwarp();
        cluster_arrive();
        cluster_wait();                  // every CTA of the cluster runs, and its barrier is ready
    }
    // By every warp `me` of the cluster: what the warps before it have; the first one leaves the length of the list.  A lane whose
    // wait ran out takes the totals for zero (places within the list, if not the right ones) and leaves the sign that the list is
    // not to be used, which is seconds after the first warp, unless that has lost totals itself.
    __device__ __forceinline__ int exchange(int me, int mine, int lane, int ctas, int32_t* count)
    {
        if (lane < ctas) st_async_u32(cluster_map(smem_u32(&total[me]), (unsigned)lane), (unsigned)mine, cluster_map(smem_u32(&arrival), (unsigned)lane));
        const bool there = mbar_wait_cluster(&arrival, 0u);
        if (!there) *count = kListLost;
        unsigned below = 0, all = there ? 0u : kNone;
#pragma unroll
        for (int w = 0; w < WARPS; w += 32) {
            const unsigned c = there ? (unsigned)total[w + lane] : 0u;
            all += c;
            below += w + lane < me ? c : 0u;
        }
        below = __reduce_add_sync(0xffffffffu, below);
        all = __reduce_add_sync(0xffffffffu, all);
        if (me == 0 && lane == 0) *count = all < kNone ? (int)all : kListLost;
        return (int)below;
    }
};

// WORDS pairs of neighbouring entries per lane, two votes for 64 entries; every warp owns a segment of x.  One CTA of 32 warps (n <=
// 2048), or a cluster of 8 CTAs of 8 warps (n <= 4096 * WORDS), which from there on is faster (4096 on one CTA 1.5 us, 8192 2.0).
// `thr`: the largest fp16 value not above the threshold (negative: -1, not-a-number: infinity), so that the compare is exact in
// fp16, and false for a NaN.  Bound by latencies: launch (0.8 us), one read of x, one exchange of totals.  n = 1024 1.8 -> 1.15 us,
// 4096 2.3 -> 1.25, 8192 2.4 -> 1.3, 14336 2.7 -> 1.4, 28672 3.7 -> 1.5 (an entry per lane; one CTA with a scan of the totals between
// two barriers up to 6144, then a cluster with cluster barriers before and after reading each other's totals).
template <int WORDS, bool CLUSTER>
__global__ void __launch_bounds__(CLUSTER ? kClusterWarps * 32 : kSparsifyThreads)
sparsify_words_kernel(const __half* x, int n, unsigned short thr_bits, int32_t* idx, int32_t* count)
{
    __shared__ ClusterTotals<CLUSTER ? kClusterCtas * kClusterWarps : 32> totals;
    const int lane = threadIdx.x & 31, warp = __shfl_sync(0xffffffffu, (int)threadIdx.x >> 5, 0);
    unsigned rank = 0;
    if (CLUSTER) {
        asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(rank));
        totals.open();
    }
    const int me = CLUSTER ? (int)rank * kClusterWarps + warp : warp;
    const int first = me * 64 * WORDS + 2 * lane;     // this lane's entries: first + 64*j and the next
    const unsigned short* const xg = reinterpret_cast<const unsigned short*>(x);
    const __half2 thr = __half2half2(__ushort_as_half(thr_bits));
    const bool words = (reinterpret_cast<uintptr_t>(x) & 3) == 0;
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    unsigned w[WORDS];
    if (words && (me + 1) * 64 * WORDS <= n) {
#pragma unroll
        for (int j = 0; j < WORDS; ++j) w[j] = ld_global_u32(xg + first + 64 * j);
    } else {
#pragma unroll
        for (int j = 0; j < WORDS; ++j) {   // (entries that do not exist: not-a-number, never active)
            const int k = first + 64 * j;
            w[j] = 0x7fff7fffu;
            if (k - 2 * lane < n) {         // (uniform)
                const unsigned e = ld_global_u16(xg + min(k, n - 1)), o = ld_global_u16(xg + min(k + 1, n - 1));
                w[j] = (k < n ? e : 0x7fffu) | (k + 1 < n ? o : 0x7fffu) << 16;
            }
        }
    }
    unsigned even[WORDS], odd[WORDS];
    int total = 0;
#pragma unroll
    for (int j = 0; j < WORDS; ++j) {
        const unsigned ab = w[j] & 0x7fff7fffu, m = __hgt2_mask(*reinterpret_cast<const __half2*>(&ab), thr);
        even[j] = __ballot_sync(0xffffffffu, (m & 1u) != 0u);
        odd[j] = __ballot_sync(0xffffffffu, (m >> 31) != 0u);
        total += __popc(even[j]) + __popc(odd[j]);
    }
    int base;
    if (CLUSTER) {
        base = totals.exchange(me, total, lane, kClusterCtas, count);
    } else {
        if (lane == 0) totals.total[warp] = total;
        __syncthreads();
        base = (int)__reduce_add_sync(0xffffffffu, lane < warp ? (unsigned)totals.total[lane] : 0u);
        if (warp == 31 && lane == 0) *count = base + total;
    }
    const unsigned lt = (1u << lane) - 1u;
#pragma unroll
    for (int j = 0; j < WORDS; ++j) {
        const unsigned e = (even[j] >> lane) & 1u, o = (odd[j] >> lane) & 1u;
        const int at = base + __popc(even[j] & lt) + __popc(odd[j] & lt);
        if (e != 0u) idx[at] = first + 64 * j;
        if (o != 0u) idx[at + (int)e] = first + 64 * j + 1;
        base += __popc(even[j]) + __popc(odd[j]);
    }
}

__global__ void __launch_bounds__(kSparsifyThreads)
sparsify_kernel(const __half* x, int n, float t, int32_t* idx, int32_t* count)
{
    __shared__ int warp_total[32];
    __shared__ int warp_base[32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    // Programmatic dependent launch: the block may have been started while the previous kernel of the
    // stream was still draining; nothing above touches global memory, everything below waits for it.
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    // segment of this warp: a multiple of 32 elements, contiguous, ascending with the warp id
    const int seg = ((n + 32 * 32 - 1) / (32 * 32)) * 32;
    const int begin = min(warp * seg, n), end = min(begin + seg, n);

    // Eight groups of 32 entries at a time, whose loads go together (addresses clamped into x instead of guarded), then what is left;
    // `each` gets a group's first entry and which lanes' entries are active.  Bound by issue in one SM: 65537 entries 16.6 us,
    // 131072 33.7 with the second pass group by group, 13.4 and 24.4 so.
    auto pass = [&](auto each) {
        auto load = [&](int k) { return __ushort_as_half((unsigned short)ld_global_u16(x + min(k + lane, n - 1))); };
        auto vote = [&](int k, __half v) { each(k, __ballot_sync(0xffffffffu, k + lane < end && is_active(v, t))); };
        int k = begin;
        for (; end - k >= 256; k += 256) {
            __half v[8];
#pragma unroll
            for (int j = 0; j < 8; ++j) v[j] = load(k + 32 * j);
#pragma unroll
            for (int j = 0; j < 8; ++j) vote(k + 32 * j, v[j]);
        }
        for (; k < end; k += 32) vote(k, load(k));
    };
    int total = 0;
    pass([&](int, unsigned mask) { total += __popc(mask); });
    if (lane == 0) warp_total[warp] = total;
    __syncthreads();
    if (warp == 0) {
        int v = warp_total[lane], incl = v;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            int up = __shfl_up_sync(0xffffffffu, incl, o);
            if (lane >= o) incl += up;
        }
        warp_base[lane] = incl - v;
        if (lane == 31) *count = incl;
    }
    __syncthreads();
    int base = warp_base[warp];
    pass([&](int k, unsigned mask) {
        if ((mask >> lane) & 1u) idx[base + __popc(mask & ((1u << lane) - 1u))] = k + lane;
        base += __popc(mask);
    });
}

// "Active in at least one of `batch` rows" (n < 2^16): a thread-block cluster of 8 CTAs of 16 warps; every warp owns a
// run of groups of 32 columns, lane l column l of each group.  Behind every index goes the record the product reads
// instead of X: the rows' values of that column, REC of them (4 or 8; zero past the batch), so that X is gathered once
// per call and not once per block-row.  Up to kKeepGroups groups per warp (n <= 16384) the values stay in registers
// between the counting and the writing pass.  What bounds it is latency (launch, one round trip, the
// totals), so the columns are spread over as many lanes as a cluster has: neighbouring lanes then write
// neighbouring list positions.  (8 columns per lane and scattered record stores took 5.0 us at n = 4096 and 4 rows.)
constexpr int kRowsWarps = 16;
constexpr int kKeepGroups = 4;

template <int REC>
__global__ void __launch_bounds__(kRowsWarps * 32)
sparsify_rows_kernel(const unsigned short* X, int ldx, int batch, int n, float t, int32_t* idx, int32_t* count, unsigned short* gathered)
{
    __shared__ ClusterTotals<kClusterCtas * kRowsWarps> totals;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    unsigned rank;
    asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(rank));
    constexpr int nctas = kClusterCtas;
    totals.open();
    // |x| > t as integers: magnitude bits above those of the largest fp16 value not above t (-1 if t < 0: everything is;
    // infinity if t is NaN or +inf: nothing is), and not a NaN
    const int thr = (t != t) ? 0x7c00 : (t < 0.0f ? -1 : (int)__half_as_ushort(__float2half_rd(t)));
    const int groups = (n + nctas * kRowsWarps * 32 - 1) / (nctas * kRowsWarps * 32);
    const int first = ((int)rank * kRowsWarps + warp) * groups * 32 + lane;
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");

    unsigned short v[kKeepGroups][REC];
    auto load = [&](int g0) {      // groups g0 .. g0 + 3, all loads in flight together
#pragma unroll
        for (int j = 0; j < kKeepGroups; ++j) {
            const int k = min(first + (g0 + j) * 32, n - 1);
#pragma unroll
            for (int b = 0; b < REC; ++b) v[j][b] = (g0 + j < groups && b < batch) ? (unsigned short)ld_global_u16(X + (size_t)b * ldx + k) : (unsigned short)0;
        }
    };
    auto active = [&](int g0, int j) -> bool {
        bool on = false;
#pragma unroll
        for (int b = 0; b < REC; ++b)
            on |= b < batch && (unsigned)((int)(v[j][b] & 0x7fff) - thr - 1) < (unsigned)(0x7c00 - thr);
        return on && g0 + j < groups && first + (g0 + j) * 32 < n;
    };
    int total = 0;
    for (int g0 = 0; g0 < groups; g0 += kKeepGroups) {
        load(g0);
#pragma unroll
        for (int j = 0; j < kKeepGroups; ++j) total += __popc(__ballot_sync(0xffffffffu, active(g0, j)));
    }
    const int me = (int)rank * kRowsWarps + warp;
    int base = totals.exchange(me, total, lane, nctas, count);
    for (int g0 = 0; g0 < groups; g0 += kKeepGroups) {
        if (groups > kKeepGroups) load(g0);
#pragma unroll
        for (int j = 0; j < kKeepGroups; ++j) {
            const bool on = active(g0, j);
            const unsigned mask = __ballot_sync(0xffffffffu, on);
            const int pos = base + __popc(mask & ((1u << lane) - 1u));
            if (on) {
                idx[pos] = first + (g0 + j) * 32;
                unsigned rec[REC / 2];
#pragma unroll
                for (int b = 0; b < REC / 2; ++b) rec[b] = v[j][2 * b] | ((unsigned)v[j][2 * b + 1] << 16);
                if (REC == 8) *reinterpret_cast<uint4*>(gathered + (size_t)pos * 8) = make_uint4(rec[0], rec[1], rec[REC / 2 - 2], rec[REC / 2 - 1]);
                else *reinterpret_cast<uint2*>(gathered + (size_t)pos * 4) = make_uint2(rec[0], rec[1]);
            }
            base += __popc(mask);
        }
    }
}

// One launch of sparsify_rows_kernel: the columns that are active in at least one of `batch` rows (n < 2^16), and
// their x values in records of 4 (batch <= 4) or 8 fp16 values.
spqt_status launch_sparsify_rows(const __half* X, int ldx, int batch, int n, float t, int32_t* idx, int32_t* count,
                                 void* gathered, cudaStream_t stream)
{
    auto kernel = batch <= 4 ? sparsify_rows_kernel<4> : sparsify_rows_kernel<8>;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = kClusterCtas;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[1].val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg = {};
    cfg.stream = stream;
    cfg.gridDim = dim3(kClusterCtas);
    cfg.blockDim = dim3(kRowsWarps * 32);
    cfg.attrs = attr;
    cfg.numAttrs = g_no_pdl ? 1 : 2;
    const cudaError_t err = cudaLaunchKernelEx(&cfg, kernel, reinterpret_cast<const unsigned short*>(X), ldx, batch, n, t, idx, count,
                                               static_cast<unsigned short*>(gathered));
    count_launch();
    return (err == cudaSuccess && cudaGetLastError() == cudaSuccess) ? SPQT_OK : SPQT_ERR_CUDA;
}

}  // namespace spqt

extern "C" spqt_status spqt_sparsify(const void* x, int n, float t,
                                     int32_t* idx, int32_t* count, void* stream)
{
    using namespace spqt;
    if (n < 0 || !count || (n > 0 && (!x || !idx))) return SPQT_ERR_INVALID_ARG;
    if (!aligned(x, 2) || !aligned(idx, 4) || !aligned(count, 4)) return SPQT_ERR_ALIGNMENT;
    if (n > 0 && n <= 65536) {
        static constexpr void (*spread[10])(const __half*, int, unsigned short, int32_t*, int32_t*) = {
            sparsify_words_kernel<1, true>, sparsify_words_kernel<2, true>, sparsify_words_kernel<3, true>, sparsify_words_kernel<4, true>,
            sparsify_words_kernel<5, true>, sparsify_words_kernel<6, true>, sparsify_words_kernel<7, true>, sparsify_words_kernel<8, true>,
            sparsify_words_kernel<12, true>, sparsify_words_kernel<16, true>};
        const bool cluster = n > 2048;
        const int words = (n + 4095) / 4096;
        cudaLaunchConfig_t cc = {};
        cc.gridDim = dim3(cluster ? kClusterCtas : 1);
        cc.blockDim = dim3(cluster ? kClusterWarps * 32 : kSparsifyThreads);
        cc.stream = static_cast<cudaStream_t>(stream);
        cudaLaunchAttribute ca[2];
        ca[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
        ca[0].val.programmaticStreamSerializationAllowed = 1;
        ca[1].id = cudaLaunchAttributeClusterDimension;
        ca[1].val.clusterDim.x = kClusterCtas;
        ca[1].val.clusterDim.y = 1;
        ca[1].val.clusterDim.z = 1;
        cc.attrs = g_no_pdl ? ca + 1 : ca;
        cc.numAttrs = (g_no_pdl ? 0 : 1) + (cluster ? 1 : 0);
        auto kernel = !cluster ? sparsify_words_kernel<1, false> : spread[words <= 8 ? words - 1 : words <= 12 ? 8 : 9];
        const unsigned short thr = t != t ? 0x7c00 : t < 0.0f ? 0xbc00 : __half_as_ushort(__float2half_rd(t));
        const cudaError_t err = cudaLaunchKernelEx(&cc, kernel, static_cast<const __half*>(x), n, thr, idx, count);
        if (err == cudaSuccess || !cluster) {
            count_launch();
            return (err == cudaSuccess && cudaGetLastError() == cudaSuccess) ? SPQT_OK : SPQT_ERR_CUDA;
        }
        (void)cudaGetLastError();         // (the cluster cannot be launched: the single CTA below)
    }
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(1);
    cfg.blockDim = dim3(kSparsifyThreads);
    cfg.stream = static_cast<cudaStream_t>(stream);
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = g_no_pdl ? 0 : 1;
    const cudaError_t err = cudaLaunchKernelEx(&cfg, sparsify_kernel, static_cast<const __half*>(x), n, t, idx, count);
    count_launch();
    return (err == cudaSuccess && cudaGetLastError() == cudaSuccess) ? SPQT_OK : SPQT_ERR_CUDA;
}

// Sparse index collection: hidden state x and a threshold t -> the ascending
// list of the entries with |x_k| > t and its length.  Three kernels:
//   sparsify_cluster_kernel (one row, 6144 < n <= 65536): the compaction below spread over a thread-block
//     cluster of 8 CTAs, warp totals exchanged through distributed shared memory (3.4 against 4.9 us at
//     n = 14336; no gain at n = 4096, where the single CTA stays).
//   sparsify_kernel (one row, any n): each warp owns a contiguous segment of x, counts its active entries
//     with __ballot_sync/__popc (the loads of eight groups of 32 entries in flight together), the 32 warp
//     totals are scanned in shared memory, and each warp then writes its indices at its base offset.
//   sparsify_rows_kernel (the small batch, n < 2^16: "active in at least one of B rows"): a cluster of 8 CTAs, which
//     also gathers the rows' values of the listed columns.
// The output order is ascending by construction (no atomics, no arrival order).
#include "spqt_common.cuh"

namespace spqt {

constexpr int kSparsifyThreads = 1024;

__device__ __forceinline__ bool is_active(__half v, float t)
{
    // exact widening; NaN compares false and is therefore never active
    return fabsf(__half2float(v)) > t;
}

__global__ void __launch_bounds__(kSparsifyThreads)
sparsify_kernel(const __half* __restrict__ x, int n, float t,
                int32_t* __restrict__ idx, int32_t* __restrict__ count)
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

    // Eight groups of 32 entries at a time: their loads are issued together (addresses clamped into x instead
    // of guarded, so that nothing makes one load wait for another), then one ballot per group.  Up to 64
    // groups per warp (n <= 65536) the lane's activity bits stay in a register for the writing phase.
    const int groups = (end - begin + 31) >> 5;
    const bool in_regs = groups <= 64;
    unsigned long long flags = 0ull;
    int total = 0;
    for (int g0 = 0; g0 < groups; g0 += 8) {
        __half v[8];
#pragma unroll
        for (int j = 0; j < 8; ++j)
            if (g0 + j < groups) v[j] = x[min(begin + (g0 + j) * 32 + lane, n - 1)];   // (uniform condition)
#pragma unroll
        for (int j = 0; j < 8; ++j) {
            if (g0 + j < groups) {
                const int k = begin + (g0 + j) * 32 + lane;
                const bool p = (k < end) && is_active(v[j], t);
                total += __popc(__ballot_sync(0xffffffffu, p));
                if (p) flags |= 1ull << ((g0 + j) & 63);
            }
        }
    }
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
    if (in_regs) {
        for (int g = 0; g < groups; ++g) {
            const bool p = (flags >> g) & 1ull;
            const unsigned mask = __ballot_sync(0xffffffffu, p);
            if (p) idx[base + __popc(mask & ((1u << lane) - 1u))] = begin + g * 32 + lane;
            base += __popc(mask);
        }
        return;
    }
    for (int k0 = begin; k0 < end; k0 += 32) {
        const int k = k0 + lane;
        const bool p = (k < end) && is_active(x[k], t);
        const unsigned mask = __ballot_sync(0xffffffffu, p);
        if (p) idx[base + __popc(mask & ((1u << lane) - 1u))] = k;
        base += __popc(mask);
    }
}

// The same compaction spread over a thread-block cluster of 8 CTAs of 8 warps (n <= 65536): one SM's
// instruction rate is what a single CTA spends most of its time on once n reaches several thousand.  The 64
// warps own consecutive segments of x; every CTA leaves its warps' totals in its own shared memory, the
// cluster synchronises, and each warp adds up the totals of the warps before it, reading the other CTAs'
// tables through distributed shared memory.  A second cluster barrier keeps every CTA's table alive until
// all have read it.  (Hardware barriers that every CTA reaches unconditionally: nothing to time out.)
constexpr int kClusterCtas = 8;
constexpr int kClusterWarps = 8;

__global__ void __launch_bounds__(kClusterWarps * 32)
sparsify_cluster_kernel(const __half* __restrict__ x, int n, float t, int32_t* __restrict__ idx, int32_t* __restrict__ count)
{
    __shared__ int warp_total[kClusterWarps];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    unsigned rank;
    asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(rank));
    const int gw = (int)rank * kClusterWarps + warp;      // this warp among the cluster's 64
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    constexpr int kAll = kClusterCtas * kClusterWarps;
    const int seg = ((n + kAll * 32 - 1) / (kAll * 32)) * 32;   // at most 1024 entries: 32 groups
    const int begin = min(gw * seg, n), end = min(begin + seg, n);
    const int groups = (end - begin + 31) >> 5;
    unsigned flags = 0u;
    int total = 0;
    for (int g0 = 0; g0 < groups; g0 += 8) {
        __half v[8];
#pragma unroll
        for (int j = 0; j < 8; ++j)
            if (g0 + j < groups) v[j] = x[min(begin + (g0 + j) * 32 + lane, n - 1)];   // (uniform condition)
#pragma unroll
        for (int j = 0; j < 8; ++j) {
            if (g0 + j < groups) {
                const int k = begin + (g0 + j) * 32 + lane;
                const bool p = (k < end) && is_active(v[j], t);
                total += __popc(__ballot_sync(0xffffffffu, p));
                if (p) flags |= 1u << (g0 + j);
            }
        }
    }
    if (lane == 0) warp_total[warp] = total;
    asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
    asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
    // lane l looks up the totals of warps l and l + 32 of the cluster
    int below = 0, all = 0;
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        const int w = lane + 32 * h;
        unsigned remote;
        const unsigned local = static_cast<unsigned>(__cvta_generic_to_shared(&warp_total[w % kClusterWarps]));
        asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(remote) : "r"(local), "r"((unsigned)(w / kClusterWarps)));
        int v;
        asm volatile("ld.shared::cluster.s32 %0, [%1];" : "=r"(v) : "r"(remote) : "memory");
        below += (w < gw) ? v : 0;
        all += v;
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        below += __shfl_xor_sync(0xffffffffu, below, o);
        all += __shfl_xor_sync(0xffffffffu, all, o);
    }
    if (gw == 0 && lane == 0) *count = all;
    int base = below;
    for (int g = 0; g < groups; ++g) {
        const bool p = (flags >> g) & 1u;
        const unsigned mask = __ballot_sync(0xffffffffu, p);
        if (p) idx[base + __popc(mask & ((1u << lane) - 1u))] = begin + g * 32 + lane;
        base += __popc(mask);
    }
    // nobody leaves while another CTA may still be reading its table
    asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
    asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
}

// "Active in at least one of `batch` rows" (n < 2^16): a thread-block cluster of 8 CTAs of 16 warps; every warp owns a
// run of groups of 32 columns, lane l column l of each group.  Behind every index goes the record the product reads
// instead of X: the rows' values of that column, REC of them (4 or 8; zero past the batch), so that X is gathered once
// per call and not once per block-row.  Up to kKeepGroups groups per warp (n <= 16384) the values stay in registers
// between the counting and the writing pass.  What bounds it is latency (launch, one round trip, two cluster
// barriers), so the columns are spread over as many lanes as a cluster has: neighbouring lanes then write
// neighbouring list positions.  (8 columns per lane and scattered record stores took 5.0 us at n = 4096 and 4 rows.)
constexpr int kRowsWarps = 16;
constexpr int kKeepGroups = 4;

template <int REC>
__global__ void __launch_bounds__(kRowsWarps * 32)
sparsify_rows_kernel(const unsigned short* __restrict__ X, int ldx, int batch, int n, float t,
                     int32_t* __restrict__ idx, int32_t* __restrict__ count, unsigned short* __restrict__ gathered)
{
    __shared__ int warp_total[kRowsWarps];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    unsigned rank, nctas;
    asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(rank));
    asm volatile("mov.u32 %0, %%cluster_nctarank;" : "=r"(nctas));
    // |x| > t as integers: magnitude bits above those of the largest fp16 value not above t (-1 if t < 0: everything is;
    // infinity if t is NaN or +inf: nothing is), and not a NaN
    const int thr = (t != t) ? 0x7c00 : (t < 0.0f ? -1 : (int)__half_as_ushort(__float2half_rd(t)));
    const int groups = (n + (int)nctas * kRowsWarps * 32 - 1) / ((int)nctas * kRowsWarps * 32);
    const int first = ((int)rank * kRowsWarps + warp) * groups * 32 + lane;
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");

    unsigned short v[kKeepGroups][REC];
    auto load = [&](int g0) {      // groups g0 .. g0 + 3, all loads in flight together
#pragma unroll
        for (int j = 0; j < kKeepGroups; ++j) {
            const int k = min(first + (g0 + j) * 32, n - 1);
#pragma unroll
            for (int b = 0; b < REC; ++b) v[j][b] = (g0 + j < groups && b < batch) ? __ldg(X + (size_t)b * ldx + k) : (unsigned short)0;
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
    if (lane == 0) warp_total[warp] = total;
    asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
    asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
    // lane l adds up the totals of warps l, l + 32, .. of the cluster
    int below = 0, all = 0;
    const int me = (int)rank * kRowsWarps + warp;
#pragma unroll 4
    for (int w = lane; w < (int)nctas * kRowsWarps; w += 32) {
        unsigned remote;
        const unsigned local = static_cast<unsigned>(__cvta_generic_to_shared(&warp_total[w % kRowsWarps]));
        asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(remote) : "r"(local), "r"((unsigned)(w / kRowsWarps)));
        int c;
        asm volatile("ld.shared::cluster.s32 %0, [%1];" : "=r"(c) : "r"(remote) : "memory");
        below += (w < me) ? c : 0;
        all += c;
    }
    int base = __reduce_add_sync(0xffffffffu, below);
    all = __reduce_add_sync(0xffffffffu, all);
    // nobody leaves while another CTA may still be reading its table: arrive now, wait at the end
    asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
    if (me == 0 && lane == 0) *count = all;
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
    asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
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
    // from a few thousand entries on, the compaction spread over a cluster of 8 CTAs (falls back to the
    // single CTA below if the cluster cannot be launched)
    if (n > 6144 && n <= 65536) {
        cudaLaunchConfig_t cc = {};
        cc.gridDim = dim3(kClusterCtas);
        cc.blockDim = dim3(kClusterWarps * 32);
        cc.stream = static_cast<cudaStream_t>(stream);
        cudaLaunchAttribute ca[2];
        ca[0].id = cudaLaunchAttributeClusterDimension;
        ca[0].val.clusterDim.x = kClusterCtas;
        ca[0].val.clusterDim.y = 1;
        ca[0].val.clusterDim.z = 1;
        ca[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
        ca[1].val.programmaticStreamSerializationAllowed = 1;
        cc.attrs = ca;
        cc.numAttrs = g_no_pdl ? 1 : 2;
        if (cudaLaunchKernelEx(&cc, sparsify_cluster_kernel, static_cast<const __half*>(x), n, t, idx, count) == cudaSuccess) {
            count_launch();
            return cudaGetLastError() == cudaSuccess ? SPQT_OK : SPQT_ERR_CUDA;
        }
        (void)cudaGetLastError();
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

// Entry points that launch nothing themselves: status names, buffer sizes,
// tuning knobs, device queries, and the host-buffer convenience call.
#include <atomic>

#include "spqt_common.cuh"
#include "spqt_gemv_device.cuh"

namespace spqt {

static std::atomic<unsigned long long> g_launches{0};
void count_launch(int k) { g_launches.fetch_add((unsigned long long)k, std::memory_order_relaxed); }

int sm_count()
{
    static int cached[64];
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return -1;
    if (cached[dev] == 0) {
        int v = 0;
        if (cudaDeviceGetAttribute(&v, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) return -1;
        cached[dev] = v;
    }
    return cached[dev];
}

// ---------------------------------------------------------------- host-buffer path

// x from pinned host memory into its device staging buffer by a kernel (one CTA): for the few KB of a hidden
// state the copy engine's start-up latency is several times the transfer, while a kernel's loads over the bus
// take one round trip when they are all in flight together.  16-byte loads when both sides allow it.
constexpr int kFetchMax = 8;   // vectors per launch of the fetch kernel
struct FetchList {
    const unsigned short* src[kFetchMax];
    unsigned short* dst[kFetchMax];
    int n[kFetchMax];
};

__global__ void __launch_bounds__(256) fetch_x_kernel(FetchList fl)
{
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    const unsigned short* const src = fl.src[blockIdx.x];
    unsigned short* const dst = fl.dst[blockIdx.x];
    const int n = fl.n[blockIdx.x];
    const int tid = threadIdx.x;
    if (((reinterpret_cast<uintptr_t>(src) | reinterpret_cast<uintptr_t>(dst)) & 15) == 0) {
        const int nv = n >> 3;   // whole 16-byte pieces
        const uint4* s4 = reinterpret_cast<const uint4*>(src);
        uint4* d4 = reinterpret_cast<uint4*>(dst);
        for (int i0 = 0; i0 < nv; i0 += 256 * 8) {
            uint4 v[8];
#pragma unroll
            for (int j = 0; j < 8; ++j) {
                const int i = i0 + j * 256 + tid;
                v[j] = ld_global_v4_if(i < nv, s4 + i);   // (not one more than needed: the bus is what takes the time)
            }
#pragma unroll
            for (int j = 0; j < 8; ++j) {
                const int i = i0 + j * 256 + tid;
                if (i < nv) d4[i] = v[j];
            }
        }
        const int i = (nv << 3) + tid;
        if (i < n) dst[i] = (unsigned short)ld_global_u16(src + i);
    } else {
        for (int i0 = 0; i0 < n; i0 += 256 * 8) {
            unsigned v[8];
#pragma unroll
            for (int j = 0; j < 8; ++j) v[j] = ld_global_u16_if(i0 + j * 256 + tid < n, src + i0 + j * 256 + tid);
#pragma unroll
            for (int j = 0; j < 8; ++j)
                if (i0 + j * 256 + tid < n) dst[i0 + j * 256 + tid] = (unsigned short)v[j];
        }
    }
}

// the device address of pinned host memory the device can reach, or nullptr
static void* device_view(const void* host_ptr)
{
    cudaPointerAttributes attr;
    if (cudaPointerGetAttributes(&attr, host_ptr) == cudaSuccess && attr.type == cudaMemoryTypeHost && attr.devicePointer != nullptr)
        return attr.devicePointer;
    (void)cudaGetLastError();  // pageable memory is not an error here
    return nullptr;
}

static spqt_status launch_fetch(const FetchList& fl, int count, cudaStream_t s)
{
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(count);
    cfg.blockDim = dim3(256);
    cfg.stream = s;
    cudaLaunchAttribute la[1];
    la[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    la[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = la;
    cfg.numAttrs = g_no_pdl ? 0 : 1;
    if (cudaLaunchKernelEx(&cfg, fetch_x_kernel, fl) != cudaSuccess) return SPQT_ERR_CUDA;
    count_launch();
    return SPQT_OK;
}

static spqt_status linear_host(const void* codes, const void* scale_zero, int m, int n, int bits, int group,
                               const void* x_host, float t, void* y_host,
                               void* x_dev, int32_t* idx_dev, int32_t* count_dev, void* y_dev,
                               void* workspace, size_t workspace_bytes, void* stream, bool wait, bool x_in_place = false)
{
    if (!x_host || !y_host || !x_dev || !y_dev) return SPQT_ERR_INVALID_ARG;
    Format f;
    spqt_status st = make_format(m, n, bits, group, &f);
    if (st != SPQT_OK) return st;
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    // x: fetched by a small kernel if x_host is pinned memory the device can address, by a copy otherwise
    // (x_in_place: the caller has already brought it to x_dev)
    if (!x_in_place) {
        if (void* xv = device_view(x_host)) {
            FetchList fl = {};
            fl.src[0] = static_cast<const unsigned short*>(xv);
            fl.dst[0] = static_cast<unsigned short*>(x_dev);
            fl.n[0] = n;
            if (launch_fetch(fl, 1, s) != SPQT_OK) return SPQT_ERR_CUDA;
        } else if (cudaMemcpyAsync(x_dev, x_host, (size_t)n * 2, cudaMemcpyHostToDevice, s) != cudaSuccess) {
            return SPQT_ERR_CUDA;
        }
    }
    // If y_host is pinned memory the device can address, the kernel writes y there itself (posted
    // writes over the bus) and the copy back, with its start-up latency, is not needed.
    void* y_target = y_dev;
    if (void* yv = device_view(y_host)) y_target = yv;
    // index collection and product in one launch (two for very long x: the call decides)
    st = spqt_sparsify_gemv(codes, scale_zero, m, n, bits, group, x_dev, t, idx_dev, count_dev,
                            y_target, workspace, workspace_bytes, stream);
    if (st != SPQT_OK) return st;
    if (y_target == y_dev &&
        cudaMemcpyAsync(y_host, y_dev, (size_t)m * 2, cudaMemcpyDeviceToHost, s) != cudaSuccess)
        return SPQT_ERR_CUDA;
    if (wait && cudaStreamSynchronize(s) != cudaSuccess) return SPQT_ERR_CUDA;
    return SPQT_OK;
}

// Whether one of two linears writes what the other one reads or writes: they then keep their order.
static bool depend(const spqt_host_linear& a, const spqt_host_linear& b)
{
    struct Range {
        const void* p;
        size_t bytes;
    };
    auto ranges = [](const spqt_host_linear& l, Range* r) {   // six that it writes, three that it reads
        Format f;
        const bool known = make_format(l.m, l.n, l.bits, l.group, &f) == SPQT_OK;   // (else the linear will be refused)
        const size_t n = known ? (size_t)l.n : 0, m = known ? (size_t)l.m : 0, blocks = known ? f.blocks : 0;
        const Range all[9] = {{l.y_host, 2 * m}, {l.y_dev, 2 * m}, {l.x_dev, 2 * n}, {l.idx_dev, 4 * n}, {l.count_dev, 4}, {l.workspace, l.workspace_bytes},
                              {l.x_host, 2 * n}, {l.codes, known ? blocks * (size_t)f.B : 0}, {l.scale_zero, 4 * blocks}};
        for (int i = 0; i < 9; ++i) r[i] = all[i];
    };
    Range ra[9], rb[9];
    ranges(a, ra);
    ranges(b, rb);
    for (int i = 0; i < 9; ++i)
        for (int j = 0; j < (i < 6 ? 9 : 6); ++j) {
            const uintptr_t p = reinterpret_cast<uintptr_t>(ra[i].p), q = reinterpret_cast<uintptr_t>(rb[j].p);
            if (p != 0 && q != 0 && p < q + rb[j].bytes && q < p + ra[i].bytes) return true;
        }
    return false;
}

constexpr int kBranches = 4;   // of a recorded step at most

struct HostStep {
    cudaGraph_t graph = nullptr;
    cudaGraphExec_t exec = nullptr;
};

}  // namespace spqt

extern "C" {

const char* spqt_status_string(int s)
{
    switch (s) {
        case SPQT_OK: return "SPQT_OK";
        case SPQT_ERR_INVALID_ARG: return "SPQT_ERR_INVALID_ARG";
        case SPQT_ERR_UNSUPPORTED: return "SPQT_ERR_UNSUPPORTED";
        case SPQT_ERR_ALIGNMENT: return "SPQT_ERR_ALIGNMENT";
        case SPQT_ERR_WORKSPACE: return "SPQT_ERR_WORKSPACE";
        case SPQT_ERR_CUDA: return "SPQT_ERR_CUDA";
        case SPQT_ERR_TIMEOUT: return "SPQT_ERR_TIMEOUT";
        default: return "SPQT_ERR_UNKNOWN";
    }
}

int spqt_version(void) { return 2000; }

spqt_status spqt_packed_sizes(int m, int n, int bits, int group,
                              size_t* codes_bytes, size_t* scale_zero_bytes,
                              size_t* gemv_workspace_bytes)
{
    spqt::Format f;
    spqt_status st = spqt::make_format(m, n, bits, group, &f);
    if (st != SPQT_OK) return st;
    if (codes_bytes) *codes_bytes = f.blocks * (size_t)f.B;
    if (scale_zero_bytes) *scale_zero_bytes = f.blocks * 4;
    if (gemv_workspace_bytes) *gemv_workspace_bytes = spqt::workspace_bytes(f);
    return SPQT_OK;
}

unsigned long long spqt_launch_count(void) { return spqt::g_launches.load(std::memory_order_relaxed); }

spqt_status spqt_sparse_linear_host(const void* codes, const void* scale_zero,
                                    int m, int n, int bits, int group,
                                    const void* x_host, float t, void* y_host,
                                    void* x_dev, int32_t* idx_dev, int32_t* count_dev, void* y_dev,
                                    void* workspace, size_t workspace_bytes, void* stream)
{
    return spqt::linear_host(codes, scale_zero, m, n, bits, group, x_host, t, y_host, x_dev, idx_dev, count_dev, y_dev,
                       workspace, workspace_bytes, stream, true);
}

spqt_status spqt_sparse_linear_host_async(const void* codes, const void* scale_zero,
                                          int m, int n, int bits, int group,
                                          const void* x_host, float t, void* y_host,
                                          void* x_dev, int32_t* idx_dev, int32_t* count_dev, void* y_dev,
                                          void* workspace, size_t workspace_bytes, void* stream)
{
    return spqt::linear_host(codes, scale_zero, m, n, bits, group, x_host, t, y_host, x_dev, idx_dev, count_dev, y_dev,
                       workspace, workspace_bytes, stream, false);
}


spqt_status spqt_host_step_create(const spqt_host_linear* linears, int count, void** step)
{
    if (!linears || count < 1 || !step) return SPQT_ERR_INVALID_ARG;
    *step = nullptr;
    // Linears that have nothing in common but what they read go to branches of the graph in turn: while one is at its fixed costs
    // (the list, the first copies, the sums) another has the memory.  The eight of two Llama-3-8B-shaped layers 70.8 us in one
    // branch, 60.4 in two, 59.5 in four; of four small layers (hidden 1024) 62.2 / 46.7 / 43.3; no more with six or eight.
    int branches = spqt::g_no_pdl ? 1 : count < spqt::kBranches ? count : spqt::kBranches;
    for (int i = 0; i < count && branches > 1; ++i)
        for (int j = i + 1; j < count && branches > 1; ++j)
            if (spqt::depend(linears[i], linears[j])) branches = 1;
    cudaStream_t s = nullptr;
    if (cudaStreamCreateWithFlags(&s, cudaStreamNonBlocking) != cudaSuccess) return SPQT_ERR_CUDA;
    spqt_status st = SPQT_OK;
    spqt::HostStep* h = new spqt::HostStep();
    bool* fetched = new bool[count]();
    // One branch after the other is captured into the graph, each behind the nodes `heads`; `f` launches what belongs to it and
    // may look at the capture before it ends.
    const cudaGraphNode_t* heads = nullptr;
    size_t head_count = 0;
    cudaGraphNode_t fetch_node = nullptr;
    auto capture = [&](auto f) {
        if (st == SPQT_OK && cudaStreamBeginCaptureToGraph(s, h->graph, heads, nullptr, head_count, cudaStreamCaptureModeThreadLocal) != cudaSuccess) st = SPQT_ERR_CUDA;
        if (st != SPQT_OK) return;
        f();
        cudaGraph_t graph = nullptr;
        if (cudaStreamEndCapture(s, &graph) != cudaSuccess && st == SPQT_OK) st = SPQT_ERR_CUDA;
    };
    if (cudaGraphCreate(&h->graph, 0) != cudaSuccess) st = SPQT_ERR_CUDA;
    // every x the device can reach is fetched at the head of the step (one CTA per vector), so that the
    // linears then follow one another without a transfer in between
    capture([&] {
        spqt::FetchList fl = {};
        int k = 0;
        for (int i = 0; i < count && st == SPQT_OK; ++i) {
            const spqt_host_linear& l = linears[i];
            void* xv = (l.x_host && l.x_dev && l.n > 0) ? spqt::device_view(l.x_host) : nullptr;
            if (xv) {
                fl.src[k] = static_cast<const unsigned short*>(xv);
                fl.dst[k] = static_cast<unsigned short*>(l.x_dev);
                fl.n[k] = l.n;
                fetched[i] = true;
                ++k;
            }
            if (k == spqt::kFetchMax || (i == count - 1 && k > 0)) {
                st = spqt::launch_fetch(fl, k, s);
                k = 0;
            }
        }
        // the last fetch, which the branches follow
        cudaStreamCaptureStatus capturing;
        const cudaGraphNode_t* last = nullptr;
        size_t lasts = 0;
        if (st == SPQT_OK && (cudaStreamGetCaptureInfo(s, &capturing, nullptr, nullptr, &last, &lasts) != cudaSuccess || lasts > 1)) st = SPQT_ERR_CUDA;
        if (st == SPQT_OK && lasts == 1) {
            fetch_node = last[0];
            heads = &fetch_node;
            head_count = 1;
        }
    });
    for (int b = 0; b < branches; ++b)
        capture([&] {
            for (int i = b; i < count && st == SPQT_OK; i += branches) {
                const spqt_host_linear& l = linears[i];
                st = spqt::linear_host(l.codes, l.scale_zero, l.m, l.n, l.bits, l.group, l.x_host, l.t, l.y_host, l.x_dev, l.idx_dev,
                                 l.count_dev, l.y_dev, l.workspace, l.workspace_bytes, s, false, fetched[i]);
            }
        });
    delete[] fetched;
    if (st == SPQT_OK && cudaGraphInstantiate(&h->exec, h->graph, 0) != cudaSuccess) st = SPQT_ERR_CUDA;
    (void)cudaStreamDestroy(s);
    if (st != SPQT_OK) {
        (void)cudaGetLastError();
        if (h->exec) (void)cudaGraphExecDestroy(h->exec);
        if (h->graph) (void)cudaGraphDestroy(h->graph);
        delete h;
        return st;
    }
    *step = h;
    return SPQT_OK;
}

spqt_status spqt_host_step_launch(void* step, void* stream)
{
    if (!step) return SPQT_ERR_INVALID_ARG;
    spqt::HostStep* h = static_cast<spqt::HostStep*>(step);
    return cudaGraphLaunch(h->exec, static_cast<cudaStream_t>(stream)) == cudaSuccess ? SPQT_OK : SPQT_ERR_CUDA;
}

spqt_status spqt_host_step_destroy(void* step)
{
    if (!step) return SPQT_ERR_INVALID_ARG;
    spqt::HostStep* h = static_cast<spqt::HostStep*>(step);
    (void)cudaGraphExecDestroy(h->exec);
    (void)cudaGraphDestroy(h->graph);
    delete h;
    return SPQT_OK;
}

}  // extern "C"

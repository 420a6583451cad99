// Device-side building blocks of the kernels: PTX wrappers (cp.async, shared-memory accesses by 32-bit address,
// thread-block-cluster primitives, mbarriers with bounded waits, two fp32 operations per instruction).
#pragma once

namespace spqt {

// ---------------------------------------------------------------- PTX helpers

__device__ __forceinline__ unsigned smem_u32(const void* p)
{
    return static_cast<unsigned>(__cvta_generic_to_shared(p));
}

// ---- mbarriers (the row-wise kernel's ring; what the CTAs of a cluster send one another)
constexpr unsigned long long kWaitNs = 1000000000ull;  // bound on every wait: one second of wall time

__device__ __forceinline__ void mbar_init(uint64_t* bar, unsigned count)
{
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count) : "memory");
}

__device__ __forceinline__ void mbar_arrive(uint64_t* bar)
{
    asm volatile("{\n\t.reg .b64 st;\n\tmbarrier.arrive.shared::cta.b64 st, [%0];\n\t}" ::"r"(smem_u32(bar))
                 : "memory");
}

// one arrival that announces `bytes` of asynchronous stores
__device__ __forceinline__ void mbar_expect(uint64_t* bar, unsigned bytes)
{
    asm volatile("{\n\t.reg .b64 st;\n\tmbarrier.arrive.expect_tx.shared::cta.b64 st, [%0], %1;\n\t}" ::"r"(smem_u32(bar)), "r"(bytes)
                 : "memory");
}

// a barrier that other CTAs of the cluster use: visible to those that wait for this CTA's next cluster arrival
__device__ __forceinline__ void mbar_publish() { asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory"); }

__device__ __forceinline__ unsigned long long global_ns()
{
    unsigned long long t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}

// One attempt to see the phase with the given parity, which blocks for up to about 4 us on this GPU (with or without the time hint).
// CLUSTER: what the barrier announces comes from other CTAs of the cluster, and the acquire has to reach as far (left out, its
// scope is the CTA).
constexpr unsigned kSuspendNs = 100000u;  // the time hint
template <bool CLUSTER>
__device__ __forceinline__ bool mbar_try(unsigned addr, unsigned parity)
{
    unsigned done;
    if (CLUSTER)
        asm volatile(
            "{\n\t.reg .pred p;\n\t"
            "mbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2, %3;\n\t"
            "selp.u32 %0, 1, 0, p;\n\t}"
            : "=r"(done)
            : "r"(addr), "r"(parity), "r"(kSuspendNs)
            : "memory");
    else
        asm volatile(
            "{\n\t.reg .pred p;\n\t"
            "mbarrier.try_wait.parity.acquire.cta.shared::cta.b64 p, [%1], %2, %3;\n\t"
            "selp.u32 %0, 1, 0, p;\n\t}"
            : "=r"(done)
            : "r"(addr), "r"(parity), "r"(kSuspendNs)
            : "memory");
    return done != 0u;
}

// Bounded wait for the arrivals of this CTA's threads; false when the bound (wall time, so that a logic error can never hold the
// GPU) expires.
__device__ __forceinline__ bool mbar_wait(uint64_t* bar, unsigned parity)
{
    const unsigned addr = smem_u32(bar);
    unsigned long long t0 = 0;
    for (unsigned it = 0;; ++it) {
        if (mbar_try<false>(addr, parity)) return true;
        if (it == 0) t0 = global_ns();
        else if (global_ns() - t0 > kWaitNs) return false;
    }
}

// By a thread of a cluster that sends nothing more to other CTAs and does not end at once: see mbar_wait_cluster.  Nobody waits here.
__device__ __forceinline__ void cluster_sent() { asm volatile("barrier.cluster.arrive.relaxed;" ::: "memory"); }

// Bounded wait for the asynchronous stores of other CTAs of the cluster, once, after this thread's own.  If they have not come within
// the bound, a CTA that left now would leave stores on their way to memory that has ended.  So the thread waits for the hardware's
// barrier of the cluster first, which threads that have ended do not hold up; every other one has said cluster_sent() before it
// waits for anything (here: it is the first thing done).  All stores have been sent then, and have a second bound to arrive.  False:
// they are lost.  (Arrivals of the threads that end after sending as well: 1 to 2 % of a small call, 1024 x 4096 3.66 -> 3.71 us.)
__device__ __forceinline__ bool mbar_wait_cluster(uint64_t* bar, unsigned parity)
{
    cluster_sent();
    const unsigned addr = smem_u32(bar);
    unsigned long long t0 = 0;
    bool late = false;
#pragma unroll 1
    while (!mbar_try<true>(addr, parity)) {
        if (t0 == 0) {
            t0 = global_ns();
        } else if (global_ns() - t0 > kWaitNs) {
            if (late) return false;
            asm volatile("barrier.cluster.wait.acquire;" ::: "memory");
            late = true;
            t0 = 0;
        }
    }
    return true;
}

// By every thread of a CTA that has sent and is done: it leaves when the CTA that waits for the stores is about to, not before (its
// wait arrives at the same barrier).  A cluster whose CTAs leave one by one leaves places that the next launch's clusters do not fit.
__device__ __forceinline__ void cluster_leave_together()
{
    cluster_sent();
    asm volatile("barrier.cluster.wait.acquire;" ::: "memory");
}

// ---- asynchronous copies
__device__ __forceinline__ void cp_async_16(unsigned smem_dst, const void* gmem_src)
{
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(smem_dst), "l"(gmem_src) : "memory");
}
// the same with no more than `left` 2-byte values read, zeros after them
__device__ __forceinline__ void cp_async_16_left(unsigned smem_dst, const void* gmem_src, int left)
{
    const int bytes = left >= 8 ? 16 : (left <= 0 ? 0 : 2 * left);
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(smem_dst), "l"(gmem_src), "r"(bytes) : "memory");
}
// the same, asking L2 to fetch no more than the 64 bytes around the address
__device__ __forceinline__ void cp_async_16_l2_64(unsigned smem_dst, const void* gmem_src)
{
    asm volatile("cp.async.cg.shared.global.L2::64B [%0], [%1], 16;" ::"r"(smem_dst), "l"(gmem_src) : "memory");
}
__device__ __forceinline__ void cp_async_8(unsigned smem_dst, const void* gmem_src)
{
    asm volatile("cp.async.ca.shared.global.L2::64B [%0], [%1], 8;" ::"r"(smem_dst), "l"(gmem_src) : "memory");
}
__device__ __forceinline__ void cp_async_4(unsigned smem_dst, const void* gmem_src)
{
    asm volatile("cp.async.ca.shared.global.L2::64B [%0], [%1], 4;" ::"r"(smem_dst), "l"(gmem_src) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_async_wait()
{
    asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory");
}

// ---- loads of what an earlier kernel of the stream may have written (x, a list and its length): never moved before the wait for
// that kernel, as a load that is declared read-only (__ldg, const __restrict__) may be.  Weights, which no kernel of a running
// stream writes, may be read either way.
__device__ __forceinline__ uint4 ld_global_v4(const void* p)
{
    uint4 v;
    asm volatile("ld.global.v4.u32 {%0, %1, %2, %3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "l"(p) : "memory");
    return v;
}
__device__ __forceinline__ uint4 ld_global_v4_if(bool on, const void* p)   // (or zeros; see ld_global_u16_if)
{
    uint4 v = make_uint4(0u, 0u, 0u, 0u);
    asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.u32 p, %5, 0;\n\t@p ld.global.v4.u32 {%0, %1, %2, %3}, [%4];\n\t}"
                 : "+r"(v.x), "+r"(v.y), "+r"(v.z), "+r"(v.w) : "l"(p), "r"((unsigned)on) : "memory");
    return v;
}
__device__ __forceinline__ unsigned ld_global_u32(const void* p)
{
    unsigned v;
    asm volatile("ld.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}
__device__ __forceinline__ unsigned ld_global_u16(const void* p)
{
    unsigned v;                          // (a 32-bit register takes the value zero-extended)
    asm volatile("ld.global.u16 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}
// the same, or zero: the load is left out and nothing looks at its value here, as a selection behind it would (which waits for the
// load: 8192 x 28672 dense 24.5 -> 26.3 us)
__device__ __forceinline__ unsigned ld_global_u16_if(bool on, const void* p)
{
    unsigned v = 0u;
    asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.u32 p, %2, 0;\n\t@p ld.global.u16 %0, [%1];\n\t}" : "+r"(v) : "l"(p), "r"((unsigned)on) : "memory");
    return v;
}

// a hint: `bytes` bytes from p on towards L2, thread i of `step` taking every step-th line
__device__ __forceinline__ void prefetch_l2(const void* p, size_t bytes, int i, int step)
{
    for (size_t off = (size_t)i * 128; off < bytes; off += (size_t)step * 128)
        asm volatile("prefetch.global.L2 [%0];" ::"l"(static_cast<const char*>(p) + off));
}

// ---- shared-memory accesses by 32-bit shared address
__device__ __forceinline__ unsigned lds_u32(unsigned addr)
{
    unsigned v;
    asm volatile("ld.shared.u32 %0, [%1];" : "=r"(v) : "r"(addr) : "memory");
    return v;
}
__device__ __forceinline__ unsigned lds_u16(unsigned addr)
{
    unsigned short v;
    asm volatile("ld.shared.u16 %0, [%1];" : "=h"(v) : "r"(addr) : "memory");
    return v;
}
__device__ __forceinline__ uint4 lds_v4(unsigned addr)
{
    uint4 v;
    asm volatile("ld.shared.v4.u32 {%0, %1, %2, %3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "r"(addr) : "memory");
    return v;
}
__device__ __forceinline__ uint2 lds_v2(unsigned addr)
{
    uint2 v;
    asm volatile("ld.shared.v2.u32 {%0, %1}, [%2];" : "=r"(v.x), "=r"(v.y) : "r"(addr) : "memory");
    return v;
}
__device__ __forceinline__ void sts_u32(unsigned addr, unsigned v)
{
    asm volatile("st.shared.u32 [%0], %1;" ::"r"(addr), "r"(v) : "memory");
}
__device__ __forceinline__ void sts_v4(unsigned addr, const uint4& v)
{
    asm volatile("st.shared.v4.u32 [%0], {%1, %2, %3, %4};" ::"r"(addr), "r"(v.x), "r"(v.y), "r"(v.z), "r"(v.w) : "memory");
}
// ---- thread-block clusters
__device__ __forceinline__ void cluster_arrive()
{
    // relaxed: all the other CTAs have to know is that this one runs
    asm volatile("barrier.cluster.arrive.relaxed.aligned;" ::: "memory");
}
__device__ __forceinline__ void cluster_wait()
{
    asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
}
// address of the same shared-memory location in the CTA of the given rank
__device__ __forceinline__ unsigned cluster_map(unsigned smem_addr, unsigned rank)
{
    unsigned r;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(smem_addr), "r"(rank));
    return r;
}
// Values into another CTA's shared memory, their bytes counted by a barrier of that CTA: the receiver waits for the data itself,
// the sender for nothing.
__device__ __forceinline__ void st_async_f32x2(unsigned addr, float a, float b, unsigned bar)
{
    asm volatile("st.async.shared::cluster.mbarrier::complete_tx::bytes.v2.f32 [%0], {%1, %2}, [%3];" ::"r"(addr), "f"(a), "f"(b), "r"(bar) : "memory");
}
__device__ __forceinline__ void st_async_f32x4(unsigned addr, const float4& v, unsigned bar)
{
    asm volatile("st.async.shared::cluster.mbarrier::complete_tx::bytes.v4.f32 [%0], {%1, %2, %3, %4}, [%5];" ::"r"(addr), "f"(v.x), "f"(v.y), "f"(v.z), "f"(v.w), "r"(bar)
                 : "memory");
}
__device__ __forceinline__ void st_async_u32(unsigned addr, unsigned v, unsigned bar)
{
    asm volatile("st.async.shared::cluster.mbarrier::complete_tx::bytes.u32 [%0], %1, [%2];" ::"r"(addr), "r"(v), "r"(bar) : "memory");
}
__device__ __forceinline__ void st_async_f32(unsigned addr, float v, unsigned bar)
{
    asm volatile("st.async.shared::cluster.mbarrier::complete_tx::bytes.f32 [%0], %1, [%2];" ::"r"(addr), "f"(v), "r"(bar) : "memory");
}

// The length that the index collection gives a list whose places it could not find (totals of its warps were lost, see
// mbar_wait_cluster).  The products take a negative length for an empty list and give
// not-a-number.
constexpr int kListLost = -1;
__device__ __forceinline__ float not_a_number_if(bool lost, float v) { return lost ? __int_as_float(0x7fffffff) : v; }

// Two fp32 lanes in one 64-bit register, the operand form of the packed FMA.
__device__ __forceinline__ unsigned long long pack2(float lo, float hi)
{
    unsigned long long r;
    asm("mov.b64 %0, {%1,%2};" : "=l"(r) : "f"(lo), "f"(hi));
    return r;
}
__device__ __forceinline__ void unpack2(unsigned long long v, float& lo, float& hi)
{
    asm("mov.b64 {%0,%1}, %2;" : "=f"(lo), "=f"(hi) : "l"(v));
}
// d = a * b + d on both lanes with one instruction
__device__ __forceinline__ void ffma2(unsigned long long& d, unsigned long long a, unsigned long long b)
{
    asm("fma.rn.f32x2 %0, %1, %2, %0;" : "+l"(d) : "l"(a), "l"(b));
}

// d = a * b on both lanes
__device__ __forceinline__ unsigned long long fmul2(unsigned long long a, unsigned long long b)
{
    unsigned long long d;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}

// a + b on both lanes
__device__ __forceinline__ unsigned long long fadd2(unsigned long long a, unsigned long long b)
{
    unsigned long long d;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}

// One step of a butterfly reduce-scatter: lanes that differ in bit `bit` hold
// partial sums of the same rows; each keeps one half of its N values and
// receives the partner's partials of that half.
template <int N>
__device__ __forceinline__ void halve(const float* in, float* out, int lane, int bit)
{
    const bool upper = (lane & bit) != 0;
#pragma unroll
    for (int i = 0; i < N / 2; ++i) {
        const float keep = upper ? in[i + N / 2] : in[i];
        const float send = upper ? in[i] : in[i + N / 2];
        out[i] = keep + __shfl_xor_sync(0xffffffffu, send, bit);
    }
}

}  // namespace spqt

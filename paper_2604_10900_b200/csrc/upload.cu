// Brings the unit descriptors of a call into the workspace and clears the call's flag words: one kernel instead of a copy and a
// memset, so that the event's first real kernel follows by dependent launch and no copy engine sits between kernels.  Up to
// kParamUnits descriptors travel as kernel parameters; more are read from the context's page-locked staging over the bus.  The kernel
// itself starts while the one before it (the end of the last event, say) still runs, and reads the staging then: it waits only to
// write.  288 units of 640 rows 146.3 to 144.1 us, 128 of 4,608 187.4 to 179.7, 8 of 640 54.8 to 52.9.
#include "cask_internal.cuh"

namespace cask {

namespace {

constexpr int kParamUnits = 32;
constexpr int kThreads = 256;
struct DescParams { UnitDesc d[kParamUnits]; };
static_assert(sizeof(UnitDesc) % 16 == 0, "descriptors move 16 bytes at a time");

__global__ void __launch_bounds__(kThreads) desc_from_params(const __grid_constant__ DescParams in, int n16, uint4* __restrict__ dst,
                                                             uint4* __restrict__ err, bool release) {
    // (see pdl_wait; no early start of a long score pass with given normalisers, see launch_passes)
    asm volatile("griddepcontrol.wait;" ::: "memory");
    if (release) asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    const uint4* src = reinterpret_cast<const uint4*>(&in);
    if (threadIdx.x < 2) err[threadIdx.x] = make_uint4(0u, 0u, 0u, 0u);
    for (int i = threadIdx.x; i < n16; i += kThreads) dst[i] = src[i];
}

__global__ void __launch_bounds__(kThreads) desc_from_host(const uint4* __restrict__ src, int n16, uint4* __restrict__ dst,
                                                           uint4* __restrict__ err) {
    const int i = blockIdx.x * kThreads + threadIdx.x;
    uint4 d = make_uint4(0u, 0u, 0u, 0u);
    // (Volatile: the compiler moves a plain load behind the wait, and the bus's latency with it: events of 100 to 600 units 2 to 3 us.)
    if (i < n16)
        asm volatile("ld.volatile.global.v4.u32 {%0, %1, %2, %3}, [%4];" : "=r"(d.x), "=r"(d.y), "=r"(d.z), "=r"(d.w) : "l"(src + i));
    // (No early start of the next kernel: the normaliser pass's CTAs then found these in their way, where the kernel before leaves room
    // for some of them only.  432 units of 640 rows, compaction CTAs on all but 12 places of the chip: event 212.8 to 204.4 us, 207 with
    // the staging read behind the wait; 296 to 1,332 units within 1 %.)
    asm volatile("griddepcontrol.wait;" ::: "memory");
    if (i < 2) err[i] = make_uint4(0u, 0u, 0u, 0u);
    if (i < n16) dst[i] = d;
}

}  // namespace

cudaError_t upload_descriptors(cudaStream_t stream, const UnitDesc* staged, int n, UnitDesc* dst, int32_t* err, bool release, bool* reads_staging) {
    const int n16 = (int)(n * sizeof(UnitDesc) / 16);
    *reads_staging = n > kParamUnits;
    if (n <= kParamUnits) {
        DescParams prm;
        for (int u = 0; u < n; ++u) prm.d[u] = staged[u];
        return launch_dependent(stream, desc_from_params, 1, kThreads, 0, prm, n16, (uint4*)dst, (uint4*)err, release);
    }
    return launch_dependent(stream, desc_from_host, (n16 + kThreads - 1) / kThreads, kThreads, 0, (const uint4*)staged, n16,
                            (uint4*)dst, (uint4*)err);
}

}  // namespace cask

// Launches whose start overlaps the end of the launch before them in the stream.
//
// A kernel launched by ja_launch_kernel may become resident while the kernel before it in the stream still runs: it sets up
// its barriers and finds its place, and stops at ja_wait_for_stream() until that kernel has finished and its writes are visible. Rules:
//   every thread calls ja_wait_for_stream(), one that has nothing to do as well, so a grid cannot finish before the one it waits for, and
//     the order is transitive. Before the call a thread reads parameters and the relations' key tables, which are written once, by a
//     copy that has returned to the host before any launch that reads them is issued, and no other global memory; it writes none;
//   before the call it waits for nothing but its own CTA, and takes nothing that it was not launched with;
//   ja_let_next_start() comes after the wait, so that one kernel at most waits inside the running one (called before it, the CTAs of several
//     launches piled up on the SMs that happened to have room: 256^3 f32, 64 CTAs, 12.9 us a call instead of 8). A kernel that does not
//     call it lets the next one in as its CTAs end;
//   kernels in clusters and kernels that allocate tensor memory are launched by ja_launch_kernel_after, behind the whole launch before
//     them, and let none in before they end. Cluster barriers and tensor-memory allocations wait without a limit, as mbarrier waits do not.
// The last rule is there because two queues stopped for good (the GPU answered): twenty calls that each copied operands into pooled scratch and
// multiplied them with gemm_tc_kernel in pairs of CTAs ([8000, 5001] x [5001, 5003]), and, once in many thousand passes, join-only products by
// gemm_tc_kernel followed by the aggregating relayout ([4096, 11008] x [11008, 4096] in four copies), all of these launches overlapping.
// The cause is not known. By the rules, whoever is resident early waits for one launch, all of whose CTAs are resident (timed on grids of
// single CTAs and of clusters, larger than the chip and behind a half-finished launch: no dependent started before the last CTA), so
// no two launches should wait for one another; both queues had gemm_tc_kernel next to a launch of many CTAs of 256 threads. What it costs,
// against all of them overlapping: 256^3 f32 in clusters 10.4 us a call, 7.8; [32, 4096] x [4096, 11008] 24.6, 22.4; batched scores 18.4, 17.3;
// the SwiGLU MLP 537, 532; attention and whole blocks below 1 %.
#pragma once

#include <cuda_runtime.h>
#include <string.h>

__device__ __forceinline__ void ja_wait_for_stream() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
// A pointer that is known only after the wait: what a kernel reads through it is not fetched before, nor by the path for data that no
// kernel writes meanwhile (a const __restrict__ parameter invites both).
template <typename T> __device__ __forceinline__ T* ja_after_wait(T* p) {
    asm volatile("" : "+l"(p)::"memory");
    return p;
}
__device__ __forceinline__ void ja_let_next_start() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

// Whether a launch of `ctas` equal CTAs, `places` of which fit an SM, gains by letting a launch like it in at its start. Where the launch
// takes half of the places or more and yet leaves one on every SM, some of the next one's CTAs find a place beside it and the rest go where
// its own end first, so that SMs end up with more of them than their share: 320 CTAs at four places 1.09 to 1.29 times as long (f32 contractions of
// 100 to 1000 cells), 240 at three 1.04 to 1.29, 296 in clusters of four 1.20. With 240 CTAs at four places they all fit beside it, with 480
// an SM has no place beyond its share: 0.84 to 0.99, as for every other size from 4 to 4096.
inline bool ja_let_next_pays(int64_t ctas, int64_t sms, int64_t places) {
    return !(2 * ctas >= sms * places && ctas <= sms * (places - 1));
}

struct JaLaunch {
    cudaLaunchConfig_t cfg;
    cudaLaunchAttribute attr[2];
    // cluster: CTAs per cluster along x; overlap: the kernel keeps the rules above
    JaLaunch(dim3 grid, unsigned block, size_t smem, unsigned cluster, cudaStream_t st, bool overlap = true) {
        memset(this, 0, sizeof *this);
        cfg.gridDim = grid;
        cfg.blockDim = dim3(block, 1, 1);
        cfg.dynamicSmemBytes = smem;
        cfg.stream = st;
        cfg.attrs = attr;
        if (overlap) {
            attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
            attr[0].val.programmaticStreamSerializationAllowed = 1;
            cfg.numAttrs = 1;
        }
        if (cluster > 1) {
            cudaLaunchAttribute& a = attr[cfg.numAttrs++];
            a.id = cudaLaunchAttributeClusterDimension;
            a.val.clusterDim.x = cluster;
            a.val.clusterDim.y = 1;
            a.val.clusterDim.z = 1;
        }
    }
};
template <typename... P, typename... A>
inline cudaError_t ja_launch_kernel(void (*kernel)(P...), dim3 grid, unsigned block, size_t smem, unsigned cluster, cudaStream_t st, A&&... args) {
    const JaLaunch l(grid, block, smem, cluster, st);
    return cudaLaunchKernelEx(&l.cfg, kernel, static_cast<A&&>(args)...);
}
// the same without the overlap
template <typename... P, typename... A>
inline cudaError_t ja_launch_kernel_after(void (*kernel)(P...), dim3 grid, unsigned block, size_t smem, unsigned cluster, cudaStream_t st, A&&... args) {
    const JaLaunch l(grid, block, smem, cluster, st, false);
    return cudaLaunchKernelEx(&l.cfg, kernel, static_cast<A&&>(args)...);
}
inline cudaError_t ja_launch_kernel_args(const void* kernel, dim3 grid, unsigned block, size_t smem, unsigned cluster, cudaStream_t st, void** args) {
    const JaLaunch l(grid, block, smem, cluster, st);
    return cudaLaunchKernelExC(&l.cfg, kernel, args);
}

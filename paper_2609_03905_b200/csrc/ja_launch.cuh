// Launches whose start overlaps the end of the launch before them in the stream.
//
// A kernel launched by ja_launch_kernel may become resident while the kernel before it in the stream still runs: it sets up
// its barriers and finds its place, and stops at ja_wait_for_stream() until that kernel has finished and its writes are visible. Rules:
//   every thread calls ja_wait_for_stream(), one that has nothing to do as well, so a grid cannot finish before the one it waits for, and
//     the order is transitive. Before the call a thread reads parameters and the relations' key tables, which are written once, by a
//     copy that has returned to the host before any launch that reads them is issued, and no other global memory; it writes none.
//     (f32 contractions find their place in the tables before it: 256^3 8.2 us, 9.2 behind it.)
//   Before the call it waits for nothing but its own CTA, and takes nothing that it was not launched with: tensor memory, whose
//     allocation waits without a limit for CTAs that hold some, is allocated behind it ([32, 4096] x [4096, 11008] 23.0 us, 22.5 before it).
//   ja_let_next_start() comes after the wait, so that one kernel at most waits inside the running one (called before it, the CTAs of several
//     launches piled up on the SMs that happened to have room: 256^3 f32, 64 CTAs, 12.9 us a call instead of 8), and after the allocation of
//     tensor memory. A kernel that does not call it lets the next one in as its CTAs end.
//   So whoever is resident early waits for one launch alone, all of whose CTAs are resident and have all that they will ever take: however
//     streams mix, no two launches can wait for one another. Cluster barriers and tensor-memory allocations have no limit as mbarrier waits
//     have; they stand behind the wait, between CTAs that the hardware starts together, and for memory that ends with running kernels.
//   A kernel without these calls is launched without the attribute and waits for the whole kernel before it, as ever.
// One queue did stop: twenty calls in a row that each took scratch from a pool in stream order, copied operands, multiplied with gemm_tc_kernel
// in pairs and gave the scratch back ([8000, 5001] x [5001, 5003]), both launches overlapping. Read again, the kernels give no cause: a
// product could be resident only when every CTA of the copy before it had passed its wait, which is after the last product had ended, so
// no two users of tensor memory or clusters met. What was particular is memory taken and returned in stream order between overlapping
// launches, and how the two go together is not ours to see. The cause is thus not known. The two launches of that queue, the copy and
// gemm_tc_kernel in clusters, do not overlap in either direction since; scratch is no longer taken on a caller's stream; and where the
// library does take memory there (exchange programs), its launches are plain.
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

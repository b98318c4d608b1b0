// ja_repartition data movement (Section 5.3): the overlay of the source and destination tilings gives
// atoms; each atom is cut into 2-D slabs (rows x contiguous run) and copied from its source block to its
// destination block -- "decompose" and "recompose" in one pass, no staging buffer. One CTA per slab. Pure byte movement: bit-exact.
//
// Where every offset, pitch and run length is a multiple of 16 bytes a thread moves 16-byte words as they are (5.7 TB/s at 268 MB, of
// 6.5). Long rows of any width are still written as whole aligned words, put together from the two aligned source words
// around them, and only the ends of a row go cell by cell (12370 rows of 2919 bf16 cells: 81 -> 39 us); short ones go by the
// widest access their alignment allows.
//
// The slabs travel in the kernel's parameters (12 bytes each, up to 960 a launch) where nothing is to be allocated or nothing orders
// the launch after a table's copy, else in a table in device memory that the caller keeps. On the GPU both take the same time; the
// parameters cost the host 0.5 to 1.8 us a launch. For relations that meet once a table's allocation and copy (0.4 ms) cost more than the
// several launches by parameters that many slabs take (134 MB: 59 us against 47 for one launch with a table). Both move a slab by
// the same rule (copy_of).

#include "ja_device.cuh"
#include "ja_launch.cuh"

namespace {

// Four accesses of a thread at a time, all loads before the first store: nothing tells the compiler that source and destination differ,
// and one access at a time took 48.0 us on 16384 x 4096 instead of 42.1.
template <typename V>
__device__ __forceinline__ void copy_slab(const char* sp, char* dp, const CopySlab& sl) {
    const int vpr = sl.row_bytes / (int)sizeof(V);  // vectors per row
    const int total = vpr * sl.rows;
    for (int i = threadIdx.x; i < total; i += 4 * 256) {
        V v[4];
        int64_t to[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const int k = i + u * 256;
            if (k >= total) break;
            const int r = k / vpr, c = k - r * vpr;
            v[u] = *reinterpret_cast<const V*>(sp + (int64_t)r * sl.src_pitch + (int64_t)c * sizeof(V));
            to[u] = (int64_t)r * sl.dst_pitch + (int64_t)c * sizeof(V);
        }
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            if (i + u * 256 >= total) break;
            *reinterpret_cast<V*>(dp + to[u]) = v[u];
        }
    }
}

// One slab at any even alignment. Word w of row r is the w-th aligned 16-byte word that the row touches in the destination. Only
// source words that hold wanted bytes are read (payloads are 128-byte aligned and padded, so none leaves them).
__device__ __forceinline__ void copy_slab_any(const char* sp, char* dp, const CopySlab& sl) {
    const int words = (sl.row_bytes + 30) / 16;        // at most, whatever the alignment
    const int total = words * sl.rows;
    const int dr = 256 / words, dw = 256 - dr * words;
    int r = (int)threadIdx.x / words, w = (int)threadIdx.x - r * words;
    for (int i = threadIdx.x; i < total; i += 256) {
        char* d = dp + (int64_t)r * sl.dst_pitch;
        const char* s = sp + (int64_t)r * sl.src_pitch;
        const int head = (int)(reinterpret_cast<uintptr_t>(d) & 15);
        const int at = w * 16 - head;                   // byte of the row where this word starts
        if (at < sl.row_bytes) {
            const char* from = s + at;
            const int sh = (int)(reinterpret_cast<uintptr_t>(from) & 15);
            const uint4* q = reinterpret_cast<const uint4*>(from - sh);
            const bool need_lo = at + 16 - sh > 0, need_hi = sh > 0 && at + 16 - sh < sl.row_bytes;   // the second word starts 16 - sh bytes in
            uint4 lo = make_uint4(0u, 0u, 0u, 0u), hi = lo;
            if (need_lo) lo = q[0];
            if (need_hi) hi = q[1];
            const uint4 v = ja_shift16(lo, hi, sh);
            if (at >= 0 && at + 16 <= sl.row_bytes) {
                *reinterpret_cast<uint4*>(d + at) = v;
            } else {
                const uint32_t c[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
                for (int e = 0; e < 8; ++e) {
                    const int b = at + e * 2;
                    if (b >= 0 && b < sl.row_bytes) *reinterpret_cast<uint16_t*>(d + b) = (uint16_t)(c[e >> 1] >> ((e & 1) * 16));
                }
            }
        }
        r += dr;
        w += dw;
        if (w >= words) { w -= words; ++r; }
    }
}
// How the slabs of a pair are copied. vec_bytes: the widest access that divides every offset, pitch and run length. Words put together
// pay on rows long enough that their two ends do not matter, and not against 8-byte accesses (10901 x 1088 f32 in 34-cell blocks
// 17 us, 26 as shifted words; 28480 x 916 f16 in 29-cell blocks 52 and 62; 12370 x 2919 bf16 81 and 39).
enum Copy { COPY_16, COPY_8, COPY_4, COPY_2, COPY_ANY };
Copy copy_of(int vec_bytes, bool long_rows) {
    return vec_bytes == 16 ? COPY_16 : vec_bytes == 8 ? COPY_8 : long_rows ? COPY_ANY : vec_bytes == 4 ? COPY_4 : COPY_2;
}
template <int HOW>
__device__ __forceinline__ void copy_slab_by(const char* sp, char* dp, const CopySlab& sl) {
    if (HOW == COPY_16) copy_slab<uint4>(sp, dp, sl);
    else if (HOW == COPY_8) copy_slab<uint2>(sp, dp, sl);
    else if (HOW == COPY_4) copy_slab<uint32_t>(sp, dp, sl);
    else if (HOW == COPY_2) copy_slab<uint16_t>(sp, dp, sl);
    else copy_slab_any(sp, dp, sl);
}

template <int HOW>
__global__ void __launch_bounds__(256) repartition_kernel(const char* __restrict__ src, char* __restrict__ dst, const CopySlab* __restrict__ slabs,
                                                          int64_t n_slabs) {
    // The next launch starts as the last slabs finish: the slabs are one round of several CTAs an SM, and a launch that is let in earlier
    // takes the room that is left, unevenly (10901 x 1088 f32 in 34-cell blocks 22.0 us, 20.7 without; 3000 x 700 f16 20.4, 19.2).
    ja_wait_for_stream();
    src = ja_after_wait(src);
    for (int64_t s = blockIdx.x; s < n_slabs; s += gridDim.x) {
        const CopySlab sl = slabs[s];
        copy_slab_by<HOW>(src + sl.src_off, dst + sl.dst_off, sl);
    }
}

template <int N, int HOW>
__global__ void __launch_bounds__(256) repartition_param_kernel(const char* __restrict__ src, char* __restrict__ dst, const __grid_constant__ SlabParams<N> p) {
    ja_wait_for_stream();
    src = ja_after_wait(src);
    const ParamSlab ps = p.s[blockIdx.x];
    const SlabShape sh = p.shapes[ps.shape];
    const CopySlab sl = {0, 0, ps.rows, sh.row_bytes, sh.src_pitch, sh.dst_pitch};
    copy_slab_by<HOW>(src + 2 * (int64_t)ps.src, dst + 2 * (int64_t)ps.dst, sl);
}
// The launch reads the parameters where they lie (a struct by value is copied twice before the driver copies it).
template <int HOW, int N>
void launch_param_n(const char* src, char* dst, const SlabChunk& c, cudaStream_t st) {
    void* args[] = {&src, &dst, const_cast<SlabParams<JA_PARAM_SLABS>*>(&c.p)};
    ja_launch_kernel_args(reinterpret_cast<const void*>(repartition_param_kernel<N, HOW>), dim3((unsigned)c.n), 256, 0, 1, st, args);
}
template <int HOW>
void launch_param(const char* src, char* dst, const SlabChunk& c, cudaStream_t st) {
    if (c.n <= 64) launch_param_n<HOW, 64>(src, dst, c, st);
    else if (c.n <= 256) launch_param_n<HOW, 256>(src, dst, c, st);
    else if (c.n <= 512) launch_param_n<HOW, 512>(src, dst, c, st);
    else launch_param_n<HOW, JA_PARAM_SLABS>(src, dst, c, st);
}
template <int HOW>
void launch_table(const char* src, char* dst, const CopySlab* d_slabs, int64_t n_slabs, cudaStream_t st) {
    const unsigned grid = (unsigned)(n_slabs < (int64_t)148 * 64 ? n_slabs : (int64_t)148 * 64);
    ja_launch_kernel(repartition_kernel<HOW>, dim3(grid), 256, 0, 1, st, src, dst, d_slabs, n_slabs);
}

}  // namespace

ja_status_t ja_launch_repartition_param(const char* src, char* dst, const SlabChunk& chunk, int vec_bytes, bool long_rows, cudaStream_t st) {
    static_assert(sizeof(ParamSlab) == 12 && sizeof(SlabParams<JA_PARAM_SLABS>) <= 32000, "a kernel's parameters hold 32764 bytes");
    if (chunk.n == 0) return JA_OK;
    switch (copy_of(vec_bytes, long_rows)) {
        case COPY_16: launch_param<COPY_16>(src, dst, chunk, st); break;
        case COPY_8: launch_param<COPY_8>(src, dst, chunk, st); break;
        case COPY_4: launch_param<COPY_4>(src, dst, chunk, st); break;
        case COPY_2: launch_param<COPY_2>(src, dst, chunk, st); break;
        case COPY_ANY: launch_param<COPY_ANY>(src, dst, chunk, st); break;
    }
    ja_count_launch();
    JA_CUDA(cudaGetLastError());
    return JA_OK;
}

ja_status_t ja_launch_repartition(const char* src, char* dst, const CopySlab* d_slabs, int64_t n_slabs, int vec_bytes, bool long_rows,
                                  cudaStream_t st) {
    if (n_slabs == 0) return JA_OK;
    switch (copy_of(vec_bytes, long_rows)) {
        case COPY_16: launch_table<COPY_16>(src, dst, d_slabs, n_slabs, st); break;
        case COPY_8: launch_table<COPY_8>(src, dst, d_slabs, n_slabs, st); break;
        case COPY_4: launch_table<COPY_4>(src, dst, d_slabs, n_slabs, st); break;
        case COPY_2: launch_table<COPY_2>(src, dst, d_slabs, n_slabs, st); break;
        case COPY_ANY: launch_table<COPY_ANY>(src, dst, d_slabs, n_slabs, st); break;
    }
    ja_count_launch();
    JA_CUDA(cudaGetLastError());
    return JA_OK;
}

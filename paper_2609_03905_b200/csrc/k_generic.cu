// The general join-agg of Definition 3.7 for specs no specialised kernel takes: any einsum over up to four operands
// whose concrete operator is a scalar function of the joined cells (product, identity, square, sum, silu(a) b, exp(a - b))
// with SUM, MAX or no aggregation over the indices that do not reach the output. Every operand cell is located through its
// relation's key table, so any tiling of any operand works; the operator is applied in f32 and aggregated in f32.
//
// One index moves in the innermost loop: the contiguous index of the first operand where that is summed (the lanes of a warp
// then walk it side by side for one output cell), else the last summed index (the lanes then hold 32 neighbouring output cells,
// and the warps of the CTA share the walk). All other coordinates are resolved once per walk, so a step costs an addition and a
// load per operand and no division; the joined tuples of an output cell are shared by the warps of a CTA and, where cells are few,
// by the CTAs of a cluster, whose partial results are combined in a fixed order through (distributed) shared memory. What bounds it is
// the chain of lookups and loads of a walk, not memory: the squares of 27 x 64 x 128 cells take 8 us, the maxima "bij->bj" of 24 x 64
// x 279 cells 7 (0.3 us at the copy rate). One thread per output cell, which resolved every coordinate of every tuple with 64-bit
// divisions, took 80 ms and 110 us.
#include <stdlib.h>
#include <string.h>

#include <algorithm>

#include "ja_device.cuh"
#include "ja_launch.cuh"
#include "ja_ptx.cuh"
#include "ja_walk.cuh"

namespace {

using namespace ja_ptx;
using namespace ja_walk;

constexpr int MAX_OPERANDS = 4, MAX_SUMMED = 4, MAX_COORDS = JA_MAX_RANK + MAX_SUMMED, WARPS = 8;

struct Operand {
    char* base;
    const int64_t* blk_off;
    Dim dim[JA_MAX_RANK];
    int32_t coord[JA_MAX_RANK];   // which coordinate every index is (output indices first, then the summed ones)
    int32_t rank, dtype, x;       // x: position of the moving index, -1 where the operand does not have it
};
struct Params {
    Operand in[MAX_OPERANDS], out;
    int32_t n_out, n_sum, x;                  // output and summed indices; x: the moving one's coordinate, -1: nothing is summed
    int32_t ext[MAX_COORDS];
    int64_t n_cells, n_tuples;                // output cells; tuples of the summed indices other than x
    int32_t x_ext, share, cluster, split_x;   // warps (lanes along x) sharing a cell; CTAs sharing it; whether they share the walk or the tuples
    int32_t fn, agg;
};

__device__ __forceinline__ float load_cell(const char* p, int dtype) {
    if (dtype == JA_F32) return *reinterpret_cast<const float*>(p);
    if (dtype == JA_F16) return __half2float(*reinterpret_cast<const __half*>(p));
    return __bfloat162float(*reinterpret_cast<const __nv_bfloat16*>(p));
}

// One operand along the moving index with every other coordinate fixed: inside the interval [lo, hi) of x a cell lies
// at + x * step bytes into the payload.
struct Line {
    int64_t at, step;      // 64 bits: a block may hold 2^31 bytes and more after the moving index
    int64_t a, b, post;    // cells: ((a * w + x - lo) * post + b)
    int flat, hi;
};
__host__ __device__ __forceinline__ Line line_of(const Operand& o, const int* coord) {
    Line l;
    l.a = l.b = 0;
    l.post = 1;
    l.flat = 0;
    l.hi = 0;
    for (int d = 0; d < o.rank; ++d) {
        if (d == o.x) continue;
        const int c = coord[o.coord[d]];
        const Cursor cur = seek(o.dim[d], c);
        l.flat += cur.blk * o.dim[d].nb_stride;
        const int w = cur.hi - cur.lo;
        if (o.x < 0 || d < o.x) {
            l.a = l.a * w + (c - cur.lo);
        } else {
            l.post *= w;
            l.b = l.b * w + (c - cur.lo);
        }
    }
    const int es = o.dtype == JA_F32 ? 4 : 2;
    l.step = l.post * es;
    if (o.x < 0) {
        l.at = o.blk_off[l.flat] + l.a * es;
        l.step = 0;
        l.hi = 0x7fffffff;
    }
    return l;
}
__host__ __device__ __forceinline__ void enter(const Operand& o, Line& l, int x) {   // the interval of x
    const Dim& d = o.dim[o.x];
    const Cursor c = seek(d, x);
    l.hi = c.hi;
    const int es = o.dtype == JA_F32 ? 4 : 2;
    l.at = o.blk_off[l.flat + c.blk * d.nb_stride] + ((l.a * (c.hi - c.lo) - c.lo) * l.post + l.b) * es;
}

template <int N>
__device__ __forceinline__ float joined(int fn, const float (&v)[N]) {
    float g = v[0];
    switch (fn) {
        case JA_FN_MUL:
#pragma unroll
            for (int k = 1; k < N; ++k) g *= v[k];
            break;
        case JA_FN_ADD:
#pragma unroll
            for (int k = 1; k < N; ++k) g += v[k];
            break;
        case JA_FN_SQUARE: g = v[0] * v[0]; break;
        case JA_FN_SILU_MUL: g = v[0] / (1.f + __expf(-v[0])) * v[N > 1 ? 1 : 0]; break;
        case JA_FN_EXP_SUB: g = __expf(v[0] - v[N > 1 ? 1 : 0]); break;
        default: break;   // JA_FN_IDENT
    }
    return g;
}
__device__ __forceinline__ float merged(int agg, float a, float b) { return agg == JA_AGG_MAX ? fmaxf(a, b) : a + b; }

// N operands. LANES: the lanes of a warp walk x for one cell; otherwise they hold neighbouring cells.
template <int N, bool LANES>
__global__ void __launch_bounds__(WARPS * 32) generic_join_agg_kernel(const __grid_constant__ Params p) {
    __shared__ float part[WARPS][32];
    if (p.cluster == 1) {   // (clusters do not overlap: ja_launch.cuh)
        ja_wait_for_stream();
        ja_let_next_start();
    }
    const int warp = threadIdx.x / 32, lane = threadIdx.x % 32;
    const int rank = (int)blockIdx.x % p.cluster;
    const int64_t group = blockIdx.x / p.cluster;
    // the cell, and this thread's share of its joined tuples: share number `me` of `parts`
    int64_t cell;
    int me, parts;
    if (p.x < 0) {
        cell = group * (WARPS * 32) + threadIdx.x;
        me = 0;
        parts = 1;
    } else if (LANES) {
        cell = group * (WARPS / p.share) + warp / p.share;
        me = rank * p.share + warp % p.share;
        parts = p.cluster * p.share;
    } else {
        cell = group * 32 + lane;
        me = rank * WARPS + warp;
        parts = p.cluster * WARPS;
    }
    const bool live = cell < p.n_cells;
    const float none = p.agg == JA_AGG_MAX ? -INFINITY : 0.f;
    float acc = none;
    int coord[MAX_COORDS];
    {
        uint32_t rem = live ? (uint32_t)cell : 0u;
#pragma unroll
        for (int d = JA_MAX_RANK - 1; d >= 0; --d) {
            if (d >= p.n_out) continue;
            const uint32_t q = rem / (uint32_t)p.ext[d];
            coord[d] = (int)(rem - q * (uint32_t)p.ext[d]);
            rem = q;
        }
    }
    const int64_t t_first = p.split_x ? 0 : me, t_step = p.split_x ? 1 : parts;
    const int x_share = p.split_x ? me : 0, x_shares = p.split_x ? parts : 1;
    const int x_first = LANES ? x_share * 32 + lane : x_share, x_step = LANES ? x_shares * 32 : x_shares;
    if (live) {
        for (int64_t t = t_first; t < p.n_tuples; t += t_step) {   // the tuples joined into this output cell
            uint32_t rem = (uint32_t)t;
            for (int d = p.n_out + p.n_sum - 1; d >= p.n_out; --d) {
                if (d == p.x) continue;
                const uint32_t q = rem / (uint32_t)p.ext[d];
                coord[d] = (int)(rem - q * (uint32_t)p.ext[d]);
                rem = q;
            }
            Line l[N];
            float v[N];
#pragma unroll
            for (int k = 0; k < N; ++k) {
                l[k] = line_of(p.in[k], coord);
                v[k] = 0.f;
                if (p.in[k].x < 0) v[k] = load_cell(p.in[k].base + l[k].at, p.in[k].dtype);
            }
            int x = x_first;
            while (x < p.x_ext) {
                int end = p.x_ext;
#pragma unroll
                for (int k = 0; k < N; ++k)
                    if (p.in[k].x >= 0) {
                        if (x >= l[k].hi) enter(p.in[k], l[k], x);
                        end = min(end, l[k].hi);
                    }
                const char* cell_at[N];
                int64_t ahead[N];
#pragma unroll
                for (int k = 0; k < N; ++k) {
                    cell_at[k] = p.in[k].base + (l[k].at + x * l[k].step);
                    ahead[k] = x_step * l[k].step;
                }
#pragma unroll 4
                for (; x < end; x += x_step) {
#pragma unroll
                    for (int k = 0; k < N; ++k) {
                        if (p.in[k].x >= 0) v[k] = load_cell(cell_at[k], p.in[k].dtype);
                        cell_at[k] += ahead[k];
                    }
                    acc = merged(p.agg, acc, joined<N>(p.fn, v));
                }
            }
        }
    }
    // ---- combine: lanes, warps, CTAs of the cluster, each in ascending order ----
    bool writer = live;
    if (p.x >= 0) {
        if (LANES) {
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) acc = merged(p.agg, acc, __shfl_xor_sync(0xffffffffu, acc, o));
        }
        part[warp][lane] = acc;
        __syncthreads();
        const int first = LANES ? warp / p.share * p.share : 0, count = LANES ? p.share : WARPS;
        writer = live && warp == first && (!LANES || lane == 0);
        if (writer) {
            acc = none;
            for (int w = 0; w < count; ++w) acc = merged(p.agg, acc, part[first + w][lane]);
        }
        if (p.cluster > 1) {
            __syncthreads();
            if (writer) part[warp][lane] = acc;
            cluster_sync_all();
            writer = writer && rank == 0;
            if (writer) {
                const uint32_t at = smem_u32(&part[warp][lane]);
                acc = none;
                for (int r = 0; r < p.cluster; ++r) {
                    float other;
                    asm volatile("ld.shared::cluster.f32 %0, [%1];" : "=f"(other) : "r"(mapa_cluster(at, (uint32_t)r)));
                    acc = merged(p.agg, acc, other);
                }
            }
            cluster_sync_all();   // nobody leaves before rank 0 has read its result
        }
    }
    if (writer) {
        char* o = p.out.base + line_of(p.out, coord).at;
        if (p.out.dtype == JA_F32) *reinterpret_cast<float*>(o) = acc;
        else if (p.out.dtype == JA_F16) *reinterpret_cast<__half*>(o) = __float2half_rn(acc);
        else *reinterpret_cast<__nv_bfloat16*>(o) = __float2bfloat16_rn(acc);
    }
}

template <int N, bool LANES>
ja_status_t launch(const Params& p, int64_t groups, cudaStream_t st) {
    const dim3 grid((unsigned)(groups * p.cluster));
    if (p.cluster > 1) JA_CUDA(ja_launch_kernel_after(generic_join_agg_kernel<N, LANES>, grid, WARPS * 32, 0, (unsigned)p.cluster, st, p));
    else JA_CUDA(ja_launch_kernel(generic_join_agg_kernel<N, LANES>, grid, WARPS * 32, 0, 1, st, p));
    return JA_OK;
}

// Index extents past 2^30, cell or tuple counts past 31 bits: one thread per output cell, every coordinate of every tuple resolved
// with 64-bit arithmetic.
struct WideParams {
    RelView in[MAX_OPERANDS];
    RelView out;
    int32_t n_in, n_out, n_sum;                     // operands, output indices, summed indices
    int32_t in_dtype[MAX_OPERANDS], out_dtype;
    int32_t in_pos[MAX_OPERANDS][JA_MAX_RANK];      // position of every operand index in the coordinate vector (output indices first)
    int64_t out_ext[JA_MAX_RANK], sum_ext[MAX_SUMMED];
    int64_t n_out_cells, n_sum_cells;
    int32_t fn, agg;
};

__device__ __forceinline__ float load_wide(const RelView& v, int dtype, const int64_t* x) {
    const char* p = v.base + ja_elem_off(v, x);
    if (dtype == JA_F32) return *reinterpret_cast<const float*>(p);
    if (dtype == JA_F16) return __half2float(*reinterpret_cast<const __half*>(p));
    return __bfloat162float(*reinterpret_cast<const __nv_bfloat16*>(p));
}

__global__ void __launch_bounds__(256) generic_join_agg_wide_kernel(const WideParams p) {
    ja_wait_for_stream();
    ja_let_next_start();
    for (int64_t cell = (int64_t)blockIdx.x * 256 + threadIdx.x; cell < p.n_out_cells; cell += (int64_t)gridDim.x * 256) {
        int64_t coord[JA_MAX_RANK + MAX_SUMMED];
        int64_t rem = cell;
        for (int d = p.n_out - 1; d >= 0; --d) {
            coord[d] = rem % p.out_ext[d];
            rem /= p.out_ext[d];
        }
        float acc = p.agg == JA_AGG_MAX ? -INFINITY : 0.f;
        for (int64_t s = 0; s < p.n_sum_cells; ++s) {      // the tuples joined into this output cell, ascending
            int64_t r2 = s;
            for (int d = p.n_sum - 1; d >= 0; --d) {
                coord[p.n_out + d] = r2 % p.sum_ext[d];
                r2 /= p.sum_ext[d];
            }
            float v[MAX_OPERANDS];
            for (int k = 0; k < p.n_in; ++k) {
                int64_t x[JA_MAX_RANK];
                for (int d = 0; d < p.in[k].rank; ++d) x[d] = coord[p.in_pos[k][d]];
                v[k] = load_wide(p.in[k], p.in_dtype[k], x);
            }
            float g;
            switch (p.fn) {
                case JA_FN_MUL: g = v[0]; for (int k = 1; k < p.n_in; ++k) g *= v[k]; break;
                case JA_FN_ADD: g = v[0]; for (int k = 1; k < p.n_in; ++k) g += v[k]; break;
                case JA_FN_SQUARE: g = v[0] * v[0]; break;
                case JA_FN_SILU_MUL: g = v[0] / (1.f + __expf(-v[0])) * v[1]; break;
                case JA_FN_EXP_SUB: g = __expf(v[0] - v[1]); break;
                default: g = v[0]; break;   // JA_FN_IDENT
            }
            acc = p.agg == JA_AGG_MAX ? fmaxf(acc, g) : acc + g;
        }
        char* o = p.out.base + ja_elem_off(p.out, coord);
        if (p.out_dtype == JA_F32) *reinterpret_cast<float*>(o) = acc;
        else if (p.out_dtype == JA_F16) *reinterpret_cast<__half*>(o) = __float2half_rn(acc);
        else *reinterpret_cast<__nv_bfloat16*>(o) = __float2bfloat16_rn(acc);
    }
}

// What the kernels make of a spec: coordinates, the moving index, counts. False where the spec is outside their reach (more than four
// operands or summed indices, an operator that is not a scalar function of the joined cells, NONE aggregation with summed indices).
struct Shape {
    std::string coords;          // output indices first, then the summed ones in order of first appearance
    int n_out, n_sum, x;         // x: position of the moving index in coords, -1: nothing is summed
    bool lanes, wide;
    int64_t n_cells, n_tuples;   // output cells; tuples of the summed indices other than x (counted where wide is false)
};
bool shape_of(const ja_spec* spec, Shape* s) {
    const int n_in = (int)spec->ins.size();
    if (n_in < 1 || n_in > MAX_OPERANDS) return false;
    switch (spec->fn) {
        case JA_FN_MUL: case JA_FN_ADD: break;
        case JA_FN_IDENT: case JA_FN_SQUARE: if (n_in != 1) return false; break;
        case JA_FN_SILU_MUL: case JA_FN_EXP_SUB: if (n_in != 2) return false; break;
        default: return false;
    }
    s->coords = spec->out;
    for (char c : spec->letters)
        if (s->coords.find(c) == std::string::npos) s->coords.push_back(c);
    s->n_out = (int)spec->out.size();
    s->n_sum = (int)s->coords.size() - s->n_out;
    if (s->n_out < 1 || s->n_out > JA_MAX_RANK || s->n_sum > MAX_SUMMED) return false;
    if (spec->agg != JA_AGG_SUM && spec->agg != JA_AGG_MAX && !(spec->agg == JA_AGG_NONE && s->n_sum == 0)) return false;
    // the moving index
    s->lanes = spec->out.find(spec->ins[0].back()) == std::string::npos;
    const char xl = s->n_sum == 0 ? 0 : s->lanes ? spec->ins[0].back() : s->coords.back();
    s->x = xl ? (int)s->coords.find(xl) : -1;
    s->n_cells = s->n_tuples = 1;
    s->wide = false;
    for (int d = 0; d < (int)s->coords.size() && !s->wide; ++d) {
        const int64_t e = spec->parts[spec->letters.find(s->coords[d])].back();
        if (d < s->n_out) s->n_cells *= e;
        else if (d != s->x) s->n_tuples *= e;
        // 2^30: the end of an interval that starts at a coordinate, and the coordinate a walk steps to past the end, still fit an int
        s->wide = e > (1ll << 30) || s->n_cells >= (1ll << 31) || s->n_tuples >= (1ll << 31);
    }
    return true;
}

// One operand: `term` names its indices, `coords` the coordinate vector, xl the moving index (0: none)
void fill_operand(Operand* o, const ja_relation* r, const RelView& v, const std::string& term, const std::string& coords, char xl) {
    o->base = (char*)r->base;
    o->blk_off = v.blk_off;
    o->rank = r->rank;
    o->dtype = (int)r->dtype;
    o->x = -1;
    for (int d = 0; d < r->rank; ++d) {
        set_dim(&o->dim[d], r, v, term, term[d]);
        o->coord[d] = (int)coords.find(term[d]);
        if (term[d] == xl) o->x = d;
    }
}

}  // namespace

int64_t ja_generic_cell_offset(const ja_relation* r, int moving, const int64_t* coord) {
    RelView v = ja_view(r);                     // the key table as it lies on the host
    for (int d = 0; d < r->rank; ++d) v.splits[d] = r->splits[d].data();
    v.blk_off = r->blk_off.data();
    const std::string term = std::string("abcd").substr(0, r->rank);
    Operand o;
    fill_operand(&o, r, v, term, term, moving < 0 ? 0 : term[moving]);
    int x[MAX_COORDS] = {};
    for (int d = 0; d < r->rank; ++d) x[d] = (int)coord[d];
    Line l = line_of(o, x);
    if (moving < 0) return l.at;
    enter(o, l, x[moving]);
    return l.at + x[moving] * l.step;
}

int ja_generic_form(const ja_spec* spec) {
    Shape s;
    return !shape_of(spec, &s) ? 0 : s.wide ? 2 : 1;
}

// *launched stays false when the spec is outside the kernels' reach (shape_of).
ja_status_t ja_launch_generic(const ja_spec* spec, const ja_relation* const* inputs, const ja_relation* out, cudaStream_t st, bool* launched) {
    *launched = false;
    Shape s;
    if (!shape_of(spec, &s)) return JA_OK;
    const int n_in = (int)spec->ins.size();
    const std::string& coords = s.coords;
    auto extent_of = [&](char c) { return spec->parts[spec->letters.find(c)].back(); };
    if (s.wide) {
        WideParams w;
        memset(&w, 0, sizeof w);
        w.n_in = n_in;
        w.n_out = s.n_out;
        w.n_sum = s.n_sum;
        w.n_out_cells = w.n_sum_cells = 1;
        for (int d = 0; d < w.n_out; ++d) { w.out_ext[d] = extent_of(coords[d]); w.n_out_cells *= w.out_ext[d]; }
        for (int d = 0; d < w.n_sum; ++d) { w.sum_ext[d] = extent_of(coords[w.n_out + d]); w.n_sum_cells *= w.sum_ext[d]; }
        for (int k = 0; k < n_in; ++k) {
            w.in[k] = ja_view(inputs[k]);
            w.in_dtype[k] = (int)inputs[k]->dtype;
            for (size_t d = 0; d < spec->ins[k].size(); ++d) w.in_pos[k][d] = (int)coords.find(spec->ins[k][d]);
        }
        w.out = ja_view(out);
        w.out_dtype = (int)out->dtype;
        w.fn = (int)spec->fn;
        w.agg = (int)spec->agg;
        const int64_t blocks = std::max<int64_t>(1, (w.n_out_cells + 255) / 256), cap = (int64_t)ja_sm_count() * 32;
        JA_CUDA(ja_launch_kernel(generic_join_agg_wide_kernel, dim3((unsigned)std::min(blocks, cap)), 256, 0, 1, st, w));
        ja_count_launch();
        JA_CUDA(cudaGetLastError());
        *launched = true;
        return JA_OK;
    }
    Params p;
    memset(&p, 0, sizeof p);
    p.n_out = s.n_out;
    p.n_sum = s.n_sum;
    p.x = s.x;
    p.n_cells = s.n_cells;
    p.n_tuples = s.n_tuples;
    for (size_t d = 0; d < coords.size(); ++d) p.ext[d] = (int32_t)extent_of(coords[d]);
    const bool lanes = s.lanes;
    const char xl = s.x < 0 ? 0 : coords[s.x];
    p.x_ext = xl ? (int32_t)extent_of(xl) : 1;
    for (int k = 0; k < n_in; ++k) fill_operand(&p.in[k], inputs[k], ja_view(inputs[k]), spec->ins[k], coords, xl);
    fill_operand(&p.out, out, ja_view(out), spec->out, coords, xl);
    p.fn = (int)spec->fn;
    p.agg = (int)spec->agg;
    // Who shares a cell's tuples: warps first, then CTAs, until the chip has two CTAs an SM or a share is down to a few steps (a
    // walk's start is a chain of table lookups, so a share of 48 steps took 28 us); they share the walk where there are fewer
    // tuples of the other indices than shares.
    const int64_t sms = ja_sm_count(), want = 2 * sms;
    p.share = p.cluster = 1;
    int64_t groups;
    if (p.x < 0) {
        groups = (p.n_cells + WARPS * 32 - 1) / (WARPS * 32);
    } else {
        const int64_t steps = lanes ? (p.x_ext + 31) / 32 : p.x_ext;   // of one warp along x
        const int64_t shares = std::max(steps, p.n_tuples);              // as many as can be told apart
        if (lanes) {
            while (p.share < WARPS && p.n_cells * p.share < want * WARPS && p.share < shares && steps * p.n_tuples / p.share >= 8) p.share *= 2;
            groups = (p.n_cells + WARPS / p.share - 1) / (WARPS / p.share);
        } else {
            groups = (p.n_cells + 31) / 32;
        }
        const int64_t per_cta = lanes ? p.share : WARPS;
        while (p.cluster < 8 && groups * p.cluster < want && per_cta * p.cluster < shares && steps * p.n_tuples / (per_cta * p.cluster) >= 8) p.cluster *= 2;
        p.split_x = steps > p.n_tuples;
    }
    ja_status_t status;
    if (lanes && p.x >= 0) status = n_in == 1 ? launch<1, true>(p, groups, st) : n_in == 2 ? launch<2, true>(p, groups, st) : n_in == 3 ? launch<3, true>(p, groups, st) : launch<4, true>(p, groups, st);
    else status = n_in == 1 ? launch<1, false>(p, groups, st) : n_in == 2 ? launch<2, false>(p, groups, st) : n_in == 3 ? launch<3, false>(p, groups, st) : launch<4, false>(p, groups, st);
    if (status != JA_OK) return status;
    ja_count_launch();
    *launched = true;
    return JA_OK;
}

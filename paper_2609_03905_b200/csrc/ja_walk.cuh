// Walks over the cells of a relation for the contraction kernels: one relation seen as two indices (r, k) that a kernel tiles
// and up to two more (batch indices) that are fixed per tile, under any tiling and any order of the indices.
#pragma once

#include <string.h>

#include <algorithm>
#include <string>

#include "ja_device.cuh"

namespace ja_walk {

constexpr int MAX_BATCH = 2;

// one index of one relation
struct Dim {
    const int64_t* splits;   // device
    int64_t blk_bytes;       // bytes between neighbouring blocks along this index (relations of equal blocks)
    int64_t cell_bytes;      // bytes between neighbouring cells inside a block (relations of equal blocks)
    int32_t bs;              // uniform interval length or 0
    uint32_t magic, shift;   // x / bs = umulhi(x, magic) >> shift for 0 <= x < 2^31 (bs > 1)
    int32_t nblk, extent;
    float per_cell;          // intervals per cell of the index, on average
    int32_t nb_stride;       // blocks between neighbouring blocks along this index, in key order
    int32_t pos;             // position of the index in the relation's term; -1: the relation does not have it
};
struct Rel {
    char* base;
    const int64_t* blk_off;
    Dim r, k, b[MAX_BATCH];  // row index (m of A, n of B; of the output: r = m, k = n), contracted index, batch indices
    int32_t equal;           // all blocks have one shape
    int32_t g;               // cells per piece of the contiguous index: 8, 4, 2 or 1
    int32_t kc;              // k comes after r: the contracted index is the contiguous one (operands), n is (output)
};
// A position on one index: the interval [lo, hi) that holds it.
struct Cursor {
    int blk, lo, hi;
};
__host__ __device__ __forceinline__ uint32_t mul_hi(uint32_t a, uint32_t b) {
#ifdef __CUDA_ARCH__
    return __umulhi(a, b);
#else
    return (uint32_t)((uint64_t)a * b >> 32);
#endif
}
__host__ __device__ __forceinline__ Cursor seek(const Dim& d, int x) {
    Cursor c;
    if (d.bs) {
        c.blk = d.bs > 1 ? (int)(mul_hi((uint32_t)x, d.magic) >> d.shift) : x;
        c.lo = c.blk * d.bs;
        c.hi = min(c.lo + d.bs, d.extent);
    } else {
        c.blk = min(d.nblk - 1, (int)((float)x * d.per_cell));   // near-equal intervals: right or next to it
        c.lo = (int)d.splits[c.blk];
        c.hi = (int)d.splits[c.blk + 1];
        if (x >= c.lo && x < c.hi) return c;
        int lo = 0, hi = d.nblk - 1;
        while (lo < hi) {
            const int mid = (lo + hi + 1) >> 1;
            if (d.splits[mid] <= x) lo = mid;
            else hi = mid - 1;
        }
        c.blk = lo;
        c.lo = (int)d.splits[lo];
        c.hi = (int)d.splits[lo + 1];
    }
    return c;
}
// forward to x (x < extent, never before the cursor's interval): positions along a loader's walk only grow
__device__ __forceinline__ void advance(const Dim& d, Cursor& c, int x) {
    while (x >= c.hi) {
        ++c.blk;
        c.lo = c.hi;
        c.hi = d.bs ? min(c.hi + d.bs, d.extent) : (int)d.splits[c.blk + 1];
    }
}

// Where a tile's batch coordinates put it on one relation. Inside a block every index weighs the product of the lengths of the
// indices after it. With f the earlier and s the later one of the relation's row and column index, fin / sin their positions
// inside their intervals and fw / sw the intervals' lengths, a cell lies
//     sw * (fin * cf + p0 * fw + p1) + sin * cs + p2
// cells into its block; cf, cs, p0, p1, p2 hold the batch indices' share (before both, between, after both).
struct BatchAt {
    int64_t bytes;           // equal blocks: the batch indices' share of the byte offset
    int flat;                // their share of the block number
    int cf, cs, p0, p1, p2;
};
__device__ __forceinline__ BatchAt batch_at(const Rel& o, const int (&x)[MAX_BATCH]) {
    BatchAt a = {0, 0, 1, 1, 0, 0, 0};
    const int first = min(o.r.pos, o.k.pos), second = max(o.r.pos, o.k.pos);
    int in[MAX_BATCH], w[MAX_BATCH];
#pragma unroll
    for (int i = 0; i < MAX_BATCH; ++i) {
        in[i] = 0;
        w[i] = 1;
        if (o.b[i].pos < 0) continue;
        const Cursor c = seek(o.b[i], x[i]);
        in[i] = x[i] - c.lo;
        w[i] = c.hi - c.lo;
        a.flat += c.blk * o.b[i].nb_stride;
        a.bytes += c.blk * o.b[i].blk_bytes + in[i] * o.b[i].cell_bytes;
        if (o.b[i].pos > first) a.cf *= w[i];
        if (o.b[i].pos > second) a.cs *= w[i];
    }
#pragma unroll
    for (int i = 0; i < MAX_BATCH; ++i) {
        const int pos = o.b[i].pos;
        if (pos < 0) continue;
        int v = in[i];
#pragma unroll
        for (int j = 0; j < MAX_BATCH; ++j)
            if (j != i && o.b[j].pos > pos) v *= w[j];
        if (pos < first) a.p0 += v;
        else if (pos < second) a.p1 += v;
        else a.p2 += v;
    }
    return a;
}

// ---- host -----------------------------------------------------------------------------------------------------
inline void set_dim(Dim* d, const ja_relation* r, const RelView& v, const std::string& term, char letter) {
    memset(d, 0, sizeof *d);
    const size_t p = letter ? term.find(letter) : std::string::npos;
    d->pos = p == std::string::npos ? -1 : (int32_t)p;
    if (d->pos < 0) return;
    int64_t nb = 1, cells = 1;
    for (int e = (int)p + 1; e < r->rank; ++e) {
        nb *= r->nblk[e];
        cells *= r->splits[e][1] - r->splits[e][0];
    }
    d->splits = v.splits[p];
    d->bs = (int32_t)r->bs[p];
    if (d->bs > 1) {   // magic = floor(2^(32 + s) / bs) + 1 with 2^s < bs <= 2^(s + 1): its error times x stays below 2^(32 + s) for x < 2^31
        while ((2ll << d->shift) < d->bs) ++d->shift;
        d->magic = (uint32_t)(((1ull << (32 + d->shift)) / (uint64_t)d->bs) + 1);
    }
    d->nblk = r->nblk[p];
    d->extent = (int32_t)r->extent[p];
    d->per_cell = (float)r->nblk[p] / (float)r->extent[p];
    d->nb_stride = (int32_t)nb;
    d->blk_bytes = nb * v.blk_stride;
    d->cell_bytes = cells * r->esize;
}

// largest piece of `most` (a power of two), ... 2 or 1 cells that never straddles a split point of the last index and is aligned wherever it starts
inline int piece_cells(const ja_relation* r, int most) {
    int g = most;
    for (int64_t s : r->splits[r->rank - 1])
        while (s % g) g /= 2;
    return g;
}

// The indices' roles in a product "ta,tb->tc" with one contracted index k, in both operands: m comes from A alone, n from B alone
// (each operand's contiguous index where it is not the contracted one, else the last index only it has), every other output index
// is a batch index of either or both. False where the einsum is no such product.
struct ProductRoles {
    char m = 0, n = 0, k = 0, batch[MAX_BATCH] = {0, 0};
};
inline bool product_roles(const std::string& ta, const std::string& tb, const std::string& tc, ProductRoles* r) {
    std::string all = ta;
    for (char c : tb)
        if (all.find(c) == std::string::npos) all.push_back(c);
    auto has = [](const std::string& t, char c) { return t.find(c) != std::string::npos; };
    for (char c : all)
        if (!has(tc, c)) {
            if (!has(ta, c) || !has(tb, c) || r->k) return false;
            r->k = c;
        }
    if (!r->k) return false;
    auto row_of = [&](const std::string& own, const std::string& other) -> char {
        if (own.back() != r->k) return has(other, own.back()) || !has(tc, own.back()) ? 0 : own.back();
        for (size_t i = own.size() - 1; i-- > 0;)
            if (!has(other, own[i])) return own[i];
        return 0;
    };
    r->m = row_of(ta, tb);
    r->n = row_of(tb, ta);
    if (!r->m || !r->n) return false;
    int n_batch = 0;
    for (char c : tc)
        if (c != r->m && c != r->n) {
            if (n_batch == MAX_BATCH) return false;
            r->batch[n_batch++] = c;
        }
    return true;
}
// 32-bit block numbers, coordinates and in-block offsets suffice
inline bool fits_32_bits(const ja_relation* r) {
    if (r->nblocks >= (1ll << 31)) return false;
    int64_t cells = 1;   // of the largest block
    for (int d = 0; d < r->rank; ++d) {
        if (r->extent[d] >= (1ll << 30)) return false;
        int64_t w = 0;
        for (int i = 0; i < r->nblk[d]; ++i) w = std::max(w, r->splits[d][i + 1] - r->splits[d][i]);
        cells *= w;
    }
    return cells < (1ll << 31);
}
inline void fill_rel(Rel* o, const ja_relation* r, const std::string& term, char cr, char ck, const char (&batch)[MAX_BATCH], int most) {
    const RelView v = ja_view(r);
    o->base = (char*)r->base;
    o->blk_off = v.blk_off;
    o->equal = r->equal_blocks ? 1 : 0;
    o->g = piece_cells(r, most);
    set_dim(&o->r, r, v, term, cr);
    set_dim(&o->k, r, v, term, ck);
    o->kc = o->k.pos > o->r.pos;
    for (int i = 0; i < MAX_BATCH; ++i) set_dim(&o->b[i], r, v, term, batch[i]);
    if (term.back() != cr && term.back() != ck) o->g = 1;   // (output only) a batch index is the contiguous one: cell by cell
}

}  // namespace ja_walk

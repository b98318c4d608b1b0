// Tensor-core contraction of two 16-bit relations under ANY tiling and any order of their indices: the join-agg
// "X,Y->Z" (MUL / SUM) whose operands share exactly one contracted index k, where one output index m comes from the first
// operand alone, one output index n from the second alone, and every other output index (a batch index) from either or
// both. "ij,jk->ik" is the plain case; "bij,bkj->bik", "ji,jk->ik", "aij,jk->aik" are others. It runs wherever the
// TMA-fed kernel (k_gemm_tc.cu) cannot address the blocks (block rows that are no multiple of 16 bytes, blocks of different
// shapes, transposed or batched operands) and wherever that kernel's 128 x 256 tiles would leave most of the chip idle.
//
// The contraction engine is tcgen05.mma, kind::f16, M = 128, N = BN, K = 16, fp32 accumulator in tensor memory; both operands
// may lie in shared memory K-major or MN-major, so a transposed operand costs nothing. Loader warps bring the operands in
// with cp.async in pieces of 8, 4 or 2 cells -- the greatest common divisor of the split points of the operand's contiguous
// index decides, so a piece never straddles two blocks -- or cell by cell where that divisor is odd. Tiles are cut from the
// GLOBAL index ranges, not from blocks: neither narrow blocks nor a contracted index cut 64 ways leaves part of a tile or of
// a 64-deep stage idle (172-cell blocks padded to 192 were a tenth of the work of the block-bound form).
//
// One CTA = one tile x one slice of the contracted index; the SPLIT slices of a tile form a thread-block cluster that sums
// its fp32 partial tiles through distributed shared memory, in rank order, with one rounding. Two CTAs share an SM
// (BN <= 128), so one CTA's epilogue overlaps another's main loop, and few tiles (a decoding step's projection) still put
// every SM to work on the operand stream.
//   first 4 warps                 loaders of A (and epilogue)
//   next BN / 32 warps            loaders of B (and epilogue)
//   last warp                     tcgen05.mma issuer
// Every mbarrier wait is bounded; on expiry the CTA records JA_ERR_TIMEOUT and leaves through the normal exit.
//
// What bounds it: the loaders' instruction stream (one trip of a stage through it, 0.36 to 0.51 us by itself for BN = 64 to
// 256; 0.24 to 0.51 us per stage of a full SM), on short tiles the start and the store of a CTA. Measured, us per call, against the
// block-bound loader form and the cell-by-cell kernel that this one took the place of:
//   [2048, 11008] x [11008, 4096] bf16, k cut 64 ways (8-byte pieces)       467 -> 282 (655 TFLOP/s); one block a side 376 -> 175
//   [32, 4096] x [4096, 11008] bf16                 (TMA form, 48 tiles)    61.5 -> 28.8 (k_stream_tc.cu takes it since)
//   "bij,bkj->bik" 32 x 512 x 128 x 512 bf16, indices cut in four           19310 -> 18
//   [154, 8768] x [8768, 3627] f16, odd columns cut in two                  593 -> 108
#include <string.h>

#include <algorithm>

#include "ja_device.cuh"
#include "ja_launch.cuh"
#include "ja_ptx.cuh"
#include "ja_walk.cuh"

namespace {

using namespace ja_ptx;
using namespace ja_walk;

constexpr int BM = 128, BK = 64;
// RAW: an operand has odd interval lengths (pieces of one cell); its stages carry a second 16-byte word per piece (see load_walk)
template <int BN, bool RAW> struct Cfg {
    static constexpr int A_WARPS = 4, B_WARPS = BN / 32, WARPS = A_WARPS + B_WARPS + 1, THREADS = WARPS * 32;
    static constexpr int A_BYTES = BM * BK * 2, B_BYTES = BN * BK * 2, HI = A_BYTES + B_BYTES, STAGE_BYTES = RAW ? 2 * HI : HI;
    static constexpr int STAGES = BN == 128 ? 3 : 4;
    static constexpr int SMEM = STAGES * STAGE_BYTES + 1024 + 256;
    static_assert(BM * (BN + 4) * 4 <= STAGES * STAGE_BYTES && BN * (BM + 4) * 4 <= STAGES * STAGE_BYTES, "the staged tile reuses the stages");
    static constexpr int CTAS_PER_SM = BN == 256 || RAW ? 1 : 2;
};

struct Params {
    Rel A, B, C;
    int32_t* status;
    uint32_t wait_cap_us;
    int32_t M, N, K, batch[MAX_BATCH];
    int32_t tiles_m, tiles_n, group_m;
    int32_t split;           // slices of the contracted index = CTAs per cluster
    int32_t cut_m, cut_n;    // tiles per interval of m / n where tiles stay inside intervals, 0: tiles are cut from the whole index
    int32_t f16, c_esize;
};

// Asynchronous copy of `bytes` (16, 8 or 4), zero-filled past src_bytes; nothing happens where `live` is 0 (a predicate, not a branch).
__device__ __forceinline__ void cp_async(uint32_t dst, const char* src, int bytes, int src_bytes, uint32_t live) {
    if (bytes == 16)
        asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %3, 0;\n\t@p cp.async.cg.shared.global [%0], [%1], 16, %2;\n\t}" ::"r"(dst), "l"(src), "r"(src_bytes), "r"(live) : "memory");
    else if (bytes == 8)
        asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %3, 0;\n\t@p cp.async.ca.shared.global [%0], [%1], 8, %2;\n\t}" ::"r"(dst), "l"(src), "r"(src_bytes), "r"(live) : "memory");
    else
        asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %3, 0;\n\t@p cp.async.ca.shared.global [%0], [%1], 4, %2;\n\t}" ::"r"(dst), "l"(src), "r"(src_bytes), "r"(live) : "memory");
}

__device__ __forceinline__ void st_shared16(uint32_t dst, const uint4& v) {
    asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(dst), "r"(v.x), "r"(v.y), "r"(v.z), "r"(v.w) : "memory");
}
__device__ __forceinline__ uint4 ld_shared16(uint32_t src) {
    uint4 v;
    asm volatile("ld.shared.v4.b32 {%0, %1, %2, %3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "r"(src) : "memory");
    return v;
}
__device__ __forceinline__ void st_shared2(uint32_t dst, uint16_t v) { asm volatile("st.shared.b16 [%0], %1;" ::"r"(dst), "h"(v) : "memory"); }

struct Ring {
    uint32_t full0, empty0;      // shared-memory addresses of the stages' barriers
    volatile int* ctl;
    int32_t* status;
};

__device__ __forceinline__ uint4 pack8(const uint16_t (&v)[8]) {
    return make_uint4(v[0] | (uint32_t)v[1] << 16, v[2] | (uint32_t)v[3] << 16, v[4] | (uint32_t)v[5] << 16, v[6] | (uint32_t)v[7] << 16);
}

// The walk of one loader group (TH threads for RT rows x 64 contracted cells per stage, NP 16-byte pieces per thread).
// KC: the contracted index is contiguous -- a thread owns piece (tid & 7) of rows tid / 8 + n * LP; the rows' addresses are
// fixed, the piece moves along k. Otherwise the row index is contiguous -- a thread owns the 8-row piece tid % (RT / 8) of the
// contracted rows tid / (RT / 8) + n * LP. Both land where TMA would put them under the 128-byte swizzle: 64 contracted cells
// (KC) or 64 rows (else, in groups BK * 128 bytes apart) per 128-byte line, 16-byte chunk c of line l at c ^ (l & 7).
// Rows past the extent are not copied: they only reach accumulator rows or columns that are never stored. Contracted cells past
// the extent are zero-filled in both operands.
// G = 1 (odd interval lengths, pieces at any even address): a piece that lies in one interval travels as the two aligned 16-byte
// words around it -- the first to its place in the stage, the second to the stage's second half -- and the thread that issued
// them shifts the two together before it hands the stage over, so these copies are as asynchronous as the others (2-byte loads
// through registers held a stage for 3.5 us). Words that hold no wanted cell are not read; a payload is 128-byte aligned and
// padded, so a word that holds one never leaves it. Pieces that straddle intervals go cell by cell.
template <int RT, int TH, int STAGES, int STAGE_BYTES, int HI, bool KC, int G, bool EQ>
__device__ __forceinline__ void load_walk(const Rel& o, const BatchAt& ba, uint32_t tile_base, int tid, int r0, int R, int c0, int c1, const Ring& ring) {
    constexpr int LAG = STAGES - 2;            // chunks in flight behind the one being issued
    constexpr int NG = 8 / G;                  // granules per piece
    constexpr int NP = RT * 8 / TH, LP = KC ? TH / 8 : TH / (RT / 8);   // pieces per thread, lines per pass of the group
    constexpr int NF = KC ? NP : NG;           // fixed positions: rows, or granules of the row piece
    static_assert(LP % 8 == 0 && (KC || 32 % LP == 0) && NP % 4 == 0, "the swizzle phase is one for all pieces of a thread");
    const int K = o.k.extent;
    const int line = KC ? tid >> 3 : tid / (RT / 8), piece = KC ? tid & 7 : tid % (RT / 8);
    int64_t foff[EQ ? NF : 1];
    int fflat[EQ ? 1 : NF], fa[EQ ? 1 : NF], fb[EQ ? 1 : NF];   // KC: fa = the row's factor of kw; else fa = rw, fb = the addend
    const int valid = min(RT, R - r0);         // rows of the tile that exist (at least one)
    uint32_t live = 0;
    int cells = 8;                             // !KC, G = 1: cells of the row piece that exist; 0: they lie in several intervals
#pragma unroll
    for (int f = 0; f < NF; ++f) {
        const int t = KC ? line + f * LP : piece * 8 + f * G;
        if (t < valid) live |= 1u << f;
        const int r = r0 + (t < valid ? t : 0);
        const Cursor c = seek(o.r, r);
        if (!KC && G == 1 && f == 0) {
            cells = min(8, R - r);
            if (c.hi < r + cells) cells = 0;
        }
        if (EQ) {
            foff[f] = ba.bytes + c.blk * o.r.blk_bytes + (r - c.lo) * o.r.cell_bytes;
        } else {
            fflat[f] = ba.flat + c.blk * o.r.nb_stride;
            fb[f] = 0;
            if (KC) {
                fa[f] = (r - c.lo) * ba.cf + ba.p0 * (c.hi - c.lo) + ba.p1;
            } else {
                fa[f] = c.hi - c.lo;
                fb[f] = (r - c.lo) * ba.cs + ba.p2;
            }
        }
    }
    const uint32_t dst0 = KC ? (uint32_t)(line * 128 + ((piece ^ (line & 7)) << 4))
                             : (uint32_t)((piece >> 3) * (BK * 128) + line * 128 + (((piece & 7) ^ (line & 7)) << 4));
    constexpr uint32_t DSTEP = LP * 128;
    int stage = 0;
    uint32_t phase = 0;
    const char* base = o.base;
    // The contracted positions of a stage. KC: every thread follows its own piece. Otherwise lane l follows rows l and l + 32 of
    // the stage and the warp's threads fetch what they need by shuffles: eight cursors per thread, each advanced behind a
    // divergent branch, took longer (1820 cycles a stage) than the copies themselves.
    const int lane = tid & 31;
    Cursor cur[KC ? 1 : 2];
#pragma unroll
    for (int h = 0; h < (KC ? 1 : 2); ++h) {
        const int x = c0 * BK + (KC ? piece * 8 : lane + 32 * h);
        cur[h] = seek(o.k, min(x, K - 1));
    }
    // a position's share of an address: bytes (equal blocks), or block number, ka = interval length (KC) / factor of rw, kb = addend
    struct AtK {
        int64_t off;
        int flat, a, b;
    };
    auto at_k = [&](Cursor& c, int x) -> AtK {
        AtK k = {0, 0, 0, 0};
        advance(o.k, c, x);
        if (EQ) {
            k.off = c.blk * o.k.blk_bytes + (x - c.lo) * o.k.cell_bytes;
        } else {
            k.flat = c.blk * o.k.nb_stride;
            if (KC) {
                k.a = c.hi - c.lo;
                k.b = (x - c.lo) * ba.cs + ba.p2;
            } else {
                k.a = (x - c.lo) * ba.cf + ba.p0 * (c.hi - c.lo) + ba.p1;
            }
        }
        return k;
    };
    auto shuffled = [&](const AtK& k, int from) -> AtK {
        AtK r = {0, 0, 0, 0};
        if (EQ) {
            r.off = __shfl_sync(0xffffffffu, k.off, from);
        } else {
            r.flat = __shfl_sync(0xffffffffu, k.flat, from);
            r.a = __shfl_sync(0xffffffffu, k.a, from);
        }
        return r;
    };
    // Blocks of different shapes: where the fixed positions' blocks start for the contracted interval `have`, looked up again only
    // when the walk enters another interval -- a lookup per copy, in front of every cp.async, cost more than the copies.
    const char* start[EQ ? 1 : NF];
    int have = -1;
    auto enter = [&](const AtK& k) {
        if (!EQ && k.flat != have) {
            have = k.flat;
#pragma unroll
            for (int f = 0; f < NF; ++f) start[f] = base + o.blk_off[fflat[f] + have];
        }
    };
    auto address = [&](int f, const AtK& k) -> const char* {
        if (EQ) return base + (foff[f] + k.off);
        return start[f] + (int64_t)(KC ? k.a * fa[f] + k.b : fa[f] * k.a + fb[f]) * 2;
    };
    uint32_t shifts[LAG + 1];                  // G = 1: of the stages in flight, the newest first
    auto realign = [&](int st, uint32_t sh) {
        const uint32_t at = tile_base + st * STAGE_BYTES + dst0;
#pragma unroll
        for (int n = 0; n < NP; ++n) {
            const int m = sh >> (4 * n) & 15;
            if (m > 1) st_shared16(at + n * DSTEP, ja_shift16(ld_shared16(at + n * DSTEP), ld_shared16(at + HI + n * DSTEP), m));
        }
    };
    for (int ch = c0; ch < c1; ++ch) {
        if (!mbar_wait(ring.empty0 + 8u * stage, phase ^ 1, ring.ctl, ring.status)) return;   // aborted: the CTA gives up
        const uint32_t dst = tile_base + stage * STAGE_BYTES + dst0;
        AtK kl[2];                             // !KC: rows lane and lane + 32 of this stage
        if (!KC) {
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const int x = min(ch * BK + lane + 32 * h, K - 1);
                kl[h] = at_k(cur[h], x);
            }
        }
        if (G == 1) {
            uint32_t sh = 0;                       // per piece: its byte shift, or 1 where nothing is left to do
            auto copy = [&](int n, const char* src, bool in, int bytes, uint32_t on) {
                const int m = in ? (int)(reinterpret_cast<uintptr_t>(src) & 15) : 0;
                cp_async(dst + n * DSTEP, src - m, 16, in ? 16 : 0, on);
                cp_async(dst + HI + n * DSTEP, src - m + 16, 16, 16, on && m + bytes > 16);
                sh |= (uint32_t)(on ? m : 1) << (4 * n);
            };
            if (KC) {
                const int x0 = ch * BK + piece * 8;
                const AtK k0 = at_k(cur[0], min(x0, K - 1));
                enter(k0);
                if (x0 + 8 <= cur[0].hi) {
#pragma unroll
                    for (int n = 0; n < NP; ++n) copy(n, address(n, k0), true, 16, live >> n & 1);
                } else {   // the end of an interval: all loads of the piece first, one trip to memory for the lot
                    sh = 0x11111111u;
                    const int e = x0 < K ? cur[0].hi - x0 : 0;     // cells before it
                    const char *p0[NP], *p1[NP];
#pragma unroll
                    for (int n = 0; n < NP; ++n) p0[n] = p1[n] = address(n, k0);
                    if (x0 + e < K) {
                        const AtK k1 = at_k(cur[0], x0 + e);
                        enter(k1);
#pragma unroll
                        for (int n = 0; n < NP; ++n) p1[n] = address(n, k1);
                    }
                    if (x0 >= K || x0 + 8 <= cur[0].hi || cur[0].hi == K) {
                        uint16_t v[NP][8];
#pragma unroll
                        for (int n = 0; n < NP; ++n)
#pragma unroll
                            for (int j = 0; j < 8; ++j)
                                v[n][j] = x0 + j < K ? *reinterpret_cast<const uint16_t*>(j < e ? p0[n] + j * 2 : p1[n] + (j - e) * 2) : (uint16_t)0;
#pragma unroll
                        for (int n = 0; n < NP; ++n) st_shared16(dst + n * DSTEP, pack8(v[n]));
                    } else {   // several ends: intervals shorter than a piece
                        cur[0] = seek(o.k, x0);
#pragma unroll 1
                        for (int j = 0; j < 8; ++j) {
                            const bool in = x0 + j < K;
                            AtK k = k0;
                            if (in) k = at_k(cur[0], x0 + j);
                            enter(k);
                            uint16_t v[NP];
#pragma unroll
                            for (int n = 0; n < NP; ++n) v[n] = in ? *reinterpret_cast<const uint16_t*>(address(n, k)) : (uint16_t)0;
#pragma unroll
                            for (int n = 0; n < NP; ++n) st_shared2(dst + n * DSTEP + j * 2, v[n]);
                        }
                    }
                }
            } else {
                AtK k[NP];                             // rows line + n LP of the stage
                bool one = true;                       // all in one contracted interval
#pragma unroll
                for (int n = 0; n < NP; ++n) {
                    k[n] = shuffled(kl[LP * n >> 5], (line + LP * n) & 31);
                    one = one && k[n].flat == k[0].flat;
                }
                if (cells) {
#pragma unroll
                    for (int n = 0; n < NP; ++n) {
                        enter(k[n]);
                        copy(n, address(0, k[n]), ch * BK + line + LP * n < K, 2 * cells, live & 1);
                    }
                } else {
                    sh = 0x11111111u;
                    if (one) {   // all loads first, one trip to memory for the lot
                        enter(k[0]);
                        uint16_t v[NP][8];
#pragma unroll
                        for (int n = 0; n < NP; ++n)
#pragma unroll
                            for (int j = 0; j < 8; ++j)
                                v[n][j] = ch * BK + line + LP * n < K ? *reinterpret_cast<const uint16_t*>(address(j, k[n])) : (uint16_t)0;
#pragma unroll
                        for (int n = 0; n < NP; ++n) st_shared16(dst + n * DSTEP, pack8(v[n]));
                    } else {
#pragma unroll
                        for (int n = 0; n < NP; ++n) {
                            enter(k[n]);
                            uint16_t v[8];
#pragma unroll
                            for (int j = 0; j < 8; ++j) v[j] = ch * BK + line + LP * n < K ? *reinterpret_cast<const uint16_t*>(address(j, k[n])) : (uint16_t)0;
                            st_shared16(dst + n * DSTEP, pack8(v));
                        }
                    }
                }
            }
            asm volatile("cp.async.commit_group;" ::: "memory");
#pragma unroll
            for (int i = LAG; i > 0; --i) shifts[i] = shifts[i - 1];
            shifts[0] = sh;
            if (ch - c0 >= LAG) {
                asm volatile("cp.async.wait_group %0;" ::"n"(LAG) : "memory");
                const int was = stage >= LAG ? stage - LAG : stage + STAGES - LAG;
                realign(was, shifts[LAG]);
                asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
                mbar_arrive(ring.full0 + 8u * was);
            }
        } else {
            if (KC) {
#pragma unroll
                for (int j = 0; j < NG; ++j) {
                    const int x = ch * BK + piece * 8 + j * G;
                    const AtK k = at_k(cur[0], min(x, K - G));
                    enter(k);
                    const int bytes = x < K ? G * 2 : 0;
#pragma unroll
                    for (int n = 0; n < NP; ++n) cp_async(dst + n * DSTEP + j * (G * 2), address(n, k), G * 2, bytes, live >> n & 1);
                }
            } else {
#pragma unroll
                for (int n = 0; n < NP; ++n) {          // row line + n LP of the stage
                    const AtK k = shuffled(kl[LP * n >> 5], (line + LP * n) & 31);
                    enter(k);
                    const int bytes = ch * BK + line + LP * n < K ? G * 2 : 0;
#pragma unroll
                    for (int j = 0; j < NG; ++j) cp_async(dst + n * DSTEP + j * (G * 2), address(j, k), G * 2, bytes, live >> j & 1);
                }
            }
            asm volatile("cp.async.commit_group;" ::: "memory");
            if (ch - c0 >= LAG) {   // the copies of LAG chunks ago have landed: hand that stage over
                asm volatile("cp.async.wait_group %0;" ::"n"(LAG) : "memory");
                asm volatile("fence.proxy.async.shared::cta;" ::: "memory");   // the tensor core reads through the async proxy
                mbar_arrive(ring.full0 + 8u * (stage >= LAG ? stage - LAG : stage + STAGES - LAG));
            }
        }
        if (++stage == STAGES) { stage = 0; phase ^= 1; }
    }
    asm volatile("cp.async.wait_group 0;" ::: "memory");
    if (G == 1) {
#pragma unroll
        for (int i = LAG - 1; i >= 0; --i)
            if (c1 - 1 - i >= c0) realign((c1 - 1 - i - c0) % STAGES, shifts[i]);
    }
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    for (int ch = max(c0, c1 - LAG); ch < c1; ++ch) mbar_arrive(ring.full0 + 8u * (uint32_t)((ch - c0) % STAGES));
}

template <int RT, int TH, int STAGES, int STAGE_BYTES, int HI, bool KC, bool EQ>
__device__ __forceinline__ void load_walk_g(const Rel& o, const BatchAt& ba, uint32_t tile_base, int tid, int r0, int R, int c0, int c1, const Ring& ring) {
    switch (o.g) {
        case 8: load_walk<RT, TH, STAGES, STAGE_BYTES, HI, KC, 8, EQ>(o, ba, tile_base, tid, r0, R, c0, c1, ring); break;
        case 4: load_walk<RT, TH, STAGES, STAGE_BYTES, HI, KC, 4, EQ>(o, ba, tile_base, tid, r0, R, c0, c1, ring); break;
        case 2: load_walk<RT, TH, STAGES, STAGE_BYTES, HI, KC, 2, EQ>(o, ba, tile_base, tid, r0, R, c0, c1, ring); break;
        default:
            if constexpr (STAGE_BYTES > HI) load_walk<RT, TH, STAGES, STAGE_BYTES, HI, KC, 1, EQ>(o, ba, tile_base, tid, r0, R, c0, c1, ring);
            break;
    }
}
template <int RT, int TH, int STAGES, int STAGE_BYTES, int HI>
__device__ __forceinline__ void load_walk_any(const Rel& o, const BatchAt& ba, uint32_t tile_base, int tid, int r0, int R, int c0, int c1, const Ring& ring) {
    if (o.equal) {
        if (o.kc) load_walk_g<RT, TH, STAGES, STAGE_BYTES, HI, true, true>(o, ba, tile_base, tid, r0, R, c0, c1, ring);
        else load_walk_g<RT, TH, STAGES, STAGE_BYTES, HI, false, true>(o, ba, tile_base, tid, r0, R, c0, c1, ring);
    } else {
        if (o.kc) load_walk_g<RT, TH, STAGES, STAGE_BYTES, HI, true, false>(o, ba, tile_base, tid, r0, R, c0, c1, ring);
        else load_walk_g<RT, TH, STAGES, STAGE_BYTES, HI, false, false>(o, ba, tile_base, tid, r0, R, c0, c1, ring);
    }
}

// One thread's share of the finished tile: the 8-cell piece at column c of every STEP-th line from l on, summed over the
// cluster's slices, rounded once, stored in granules of G cells. Short tiles (a batch of small products) spend as long here as
// in their main loop, so the loop holds little beyond the loads and stores: along one interval the address moves by a constant.
struct StoreCtx {
    const float* tile;        // this CTA's lines as the cluster's slices summed them, [slice][line][pitch]
    int pitch, split;
    int slice;                // floats from one slice's lines to the next one's
    int line_first, line_ext, col_first, col_ext;
    int f16, esize;
};
template <int G, bool EQ>
__device__ __forceinline__ void store_walk(const Rel& o, const Dim& dl, const Dim& dc, const BatchAt& ba, const StoreCtx& s, int l0, int l, int l1, int step, int c) {
    constexpr int NG = 8 / G;
    const int gc = s.col_first + c;
    l1 = min(l1, s.line_ext - s.line_first);
    if (gc >= s.col_ext || l >= l1) return;
    int64_t coff[EQ ? NG : 1];
    int cflat[EQ ? 1 : NG], cw[EQ ? 1 : NG], ca[EQ ? 1 : NG];
    const int live = min(NG, (s.col_ext - gc + G - 1) / G);
    Cursor cc = seek(dc, gc);
#pragma unroll
    for (int j = 0; j < NG; ++j) {
        const int x = min(gc + j * G, s.col_ext - 1);
        advance(dc, cc, x);
        if (EQ) {
            coff[j] = ba.bytes + cc.blk * dc.blk_bytes + (x - cc.lo) * dc.cell_bytes;
        } else {
            cflat[j] = ba.flat + cc.blk * dc.nb_stride;
            cw[j] = cc.hi - cc.lo;
            ca[j] = (x - cc.lo) * ba.cs + ba.p2;
        }
    }
    Cursor lc = seek(dl, s.line_first + l);
    int64_t loff = 0;
    bool moved = true;
    const float* src = s.tile + (l - l0) * s.pitch + c;
    for (; l < l1; l += step, src += step * s.pitch) {
        const int gl = s.line_first + l;
        if (gl >= lc.hi) {
            advance(dl, lc, gl);
            moved = true;
        }
        const float4 x = *reinterpret_cast<const float4*>(src), y = *reinterpret_cast<const float4*>(src + 4);
        float f[8] = {x.x, x.y, x.z, x.w, y.x, y.y, y.z, y.w};
        for (int r = 1; r < s.split; ++r) {   // slices in ascending order
            const float4 u = *reinterpret_cast<const float4*>(src + r * s.slice), v = *reinterpret_cast<const float4*>(src + r * s.slice + 4);
            f[0] += u.x; f[1] += u.y; f[2] += u.z; f[3] += u.w; f[4] += v.x; f[5] += v.y; f[6] += v.z; f[7] += v.w;
        }
        if (EQ) {
            if (moved) loff = lc.blk * dl.blk_bytes + (gl - lc.lo) * dl.cell_bytes;
            else loff += step * dl.cell_bytes;
            moved = false;
        }
        const int lflat = lc.blk * dl.nb_stride, la = (gl - lc.lo) * ba.cf + ba.p0 * (lc.hi - lc.lo) + ba.p1;
        auto address = [&](int j) -> char* {
            if (EQ) return o.base + (coff[j] + loff);
            return o.base + (o.blk_off[cflat[j] + lflat] + (int64_t)(cw[j] * la + ca[j]) * s.esize);
        };
        if (s.esize == 4) {
#pragma unroll
            for (int j = 0; j < NG; ++j) {
                if (j >= live) continue;
                char* dst = address(j);
                if (G >= 4) {
#pragma unroll
                    for (int e = 0; e < G; e += 4) *reinterpret_cast<float4*>(dst + e * 4) = make_float4(f[j * G + e], f[j * G + e + 1], f[j * G + e + 2], f[j * G + e + 3]);
                } else if (G == 2) {
                    *reinterpret_cast<float2*>(dst) = make_float2(f[j * 2], f[j * 2 + 1]);
                } else {
                    *reinterpret_cast<float*>(dst) = f[j];
                }
            }
        } else {
            uint32_t h[4];
            if (s.f16) {
#pragma unroll
                for (int e = 0; e < 4; ++e) h[e] = ja_pack16<true>(f[2 * e], f[2 * e + 1]);
            } else {
#pragma unroll
                for (int e = 0; e < 4; ++e) h[e] = ja_pack16<false>(f[2 * e], f[2 * e + 1]);
            }
#pragma unroll
            for (int j = 0; j < NG; ++j) {
                if (j >= live) continue;
                char* dst = address(j);
                if (G == 8) *reinterpret_cast<uint4*>(dst) = make_uint4(h[0], h[1], h[2], h[3]);
                else if (G == 4) *reinterpret_cast<uint2*>(dst) = make_uint2(h[j * 2], h[j * 2 + 1]);
                else if (G == 2) *reinterpret_cast<uint32_t*>(dst) = h[j];
                else *reinterpret_cast<uint16_t*>(dst) = (uint16_t)(h[j >> 1] >> ((j & 1) * 16));
            }
        }
    }
}
template <bool EQ>
__device__ __forceinline__ void store_walk_g(const Rel& o, const Dim& dl, const Dim& dc, const BatchAt& ba, const StoreCtx& s, int l0, int l, int l1, int step, int c) {
    if (o.g == 8) store_walk<8, EQ>(o, dl, dc, ba, s, l0, l, l1, step, c);
    else if (o.g == 4) store_walk<4, EQ>(o, dl, dc, ba, s, l0, l, l1, step, c);
    else if (o.g == 2) store_walk<2, EQ>(o, dl, dc, ba, s, l0, l, l1, step, c);
    else store_walk<1, EQ>(o, dl, dc, ba, s, l0, l, l1, step, c);
}

// rows [lo, end) of tile t along one index, `width` rows per tile
__device__ __forceinline__ void tile_range(const Dim& d, int cut, int width, int t, int& lo, int& end) {
    if (cut == 0) {
        lo = t * width;
        end = d.extent;
    } else {
        const int blk = t / cut;
        lo = (d.bs ? blk * d.bs : (int)d.splits[blk]) + (t - blk * cut) * width;
        end = d.bs ? min((blk + 1) * d.bs, d.extent) : (int)d.splits[blk + 1];
    }
}

// ACC accumulators: the product of 16 contracted cells q, q + ACC, q + 2 ACC, ... of the slice go to accumulator q, and the f32 sums of the
// accumulators are taken in registers. The tensor core truncates as it accumulates, so its error grows with the number of
// products in a chain; a 16-bit output's rounding hides that (ACC = 1), an f32 output shows it (ACC = 4, see ja_contract_tc_plan).
template <int BN, bool RAW, int ACC>
__global__ void __launch_bounds__(Cfg<BN, RAW>::THREADS, Cfg<BN, RAW>::CTAS_PER_SM) contract_tc_kernel(const __grid_constant__ Params p) {
    using C = Cfg<BN, RAW>;
    extern __shared__ uint8_t smem_raw[];
    const uint32_t raw = smem_u32(smem_raw);
    const uint32_t base = (raw + 1023u) & ~1023u;   // swizzle atoms need 1024-byte alignment
    uint8_t* smem = smem_raw + (base - raw);
    uint64_t* bars = reinterpret_cast<uint64_t*>(smem + C::STAGES * C::STAGE_BYTES);
    const uint32_t bar0 = smem_u32(bars);
    const uint32_t done_bar = bar0 + 8u * (2 * C::STAGES);
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(bars + 2 * C::STAGES + 1);
    volatile int* ctl = reinterpret_cast<volatile int*>(tmem_slot + 1);
    const Ring ring = {bar0, bar0 + 8u * C::STAGES, ctl, p.status};

    // ---- this CTA's tile and its slice of the contracted index ----
    const int split = p.split, rank = (int)blockIdx.x % split;
    const int t = (int)blockIdx.x / split;
    // bands of group_m row tiles x all column tiles: tiles in flight share operand strips through L2
    const int band_sz = p.group_m * p.tiles_n, band = t / band_sz, tin = t - band * band_sz;
    const int rows_in_band = min(p.group_m, p.tiles_m - band * p.group_m);
    int m0, m_end, n0, n_end;
    tile_range(p.A.r, p.cut_m, BM, band * p.group_m + tin % rows_in_band, m0, m_end);
    tile_range(p.B.r, p.cut_n, BN, tin / rows_in_band, n0, n_end);
    if (m0 >= m_end || n0 >= n_end) return;   // an interval shorter than the longest one (the whole cluster leaves)
    const int bx[MAX_BATCH] = {(int)blockIdx.z, (int)blockIdx.y};

    const int warp = __shfl_sync(0xffffffffu, (int)threadIdx.x / 32, 0), lane = threadIdx.x % 32;
    constexpr int MMA_WARP = C::WARPS - 1;
    if (threadIdx.x == 0) {
        for (int s = 0; s < C::STAGES; ++s) {
            mbar_init(ring.full0 + 8u * s, (C::WARPS - 1) * 32);   // one arrival per loader thread
            mbar_init(ring.empty0 + 8u * s, 1);
        }
        mbar_init(done_bar, 1);
        wait_ctl_init(ctl, p.wait_cap_us);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == MMA_WARP) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)), "n"(BN * ACC) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = __shfl_sync(0xffffffffu, *tmem_slot, 0);

    const int chunks = (p.K + BK - 1) / BK;
    const int c0 = (int)((int64_t)chunks * rank / split), c1 = (int)((int64_t)chunks * (rank + 1) / split);

    if (warp < C::A_WARPS) {
        load_walk_any<BM, C::A_WARPS * 32, C::STAGES, C::STAGE_BYTES, C::HI>(p.A, batch_at(p.A, bx), base, threadIdx.x, m0, m_end, c0, c1, ring);
    } else if (warp < MMA_WARP) {
        load_walk_any<BN, C::B_WARPS * 32, C::STAGES, C::STAGE_BYTES, C::HI>(p.B, batch_at(p.B, bx), base + C::A_BYTES, threadIdx.x - C::A_WARPS * 32, n0, n_end, c0, c1, ring);
    } else {
        const uint32_t leader = elect_one();
        const uint32_t fmt = p.f16 ? 0u : 1u;   // A and B: bf16 (format 1) or f16 (format 0); D f32
        const uint32_t idesc = (1u << 4) | (fmt << 7) | (fmt << 10) | ((p.A.kc ? 0u : 1u) << 15) | ((p.B.kc ? 0u : 1u) << 16) |
                               ((uint32_t)(BN >> 3) << 17) | ((uint32_t)(BM >> 4) << 24);
        // 16 contracted cells further: 32 bytes along a line (K-major) or 16 lines (MN-major, 64-row groups BK * 128 bytes apart)
        const uint32_t a_step = p.A.kc ? 32u : 2048u, b_step = p.B.kc ? 32u : 2048u;
        const uint32_t a_lbo = p.A.kc ? 16u : BK * 128u, b_lbo = p.B.kc ? 16u : BK * 128u;
        int stage = 0;
        uint32_t phase = 0;
        bool ok = true;
        for (int ch = c0; ch < c1; ++ch) {
            if (!mbar_wait(ring.full0 + 8u * stage, phase, ctl, p.status)) { ok = false; break; }
            tc_fence_after();
            const uint32_t a_addr = base + stage * C::STAGE_BYTES, b_addr = a_addr + C::A_BYTES;
#pragma unroll
            for (int kk = 0; kk < BK / 16; ++kk)
                umma_bf16_w<1>(tmem + kk % ACC * BN, desc_sw128(a_addr + kk * a_step, a_lbo), desc_sw128(b_addr + kk * b_step, b_lbo), idesc,
                               (ch > c0 || kk >= ACC) ? 1u : 0u, leader);
            umma_commit_w<1>(ring.empty0 + 8u * stage, leader);
            if (++stage == C::STAGES) { stage = 0; phase ^= 1; }
        }
        if (ok) umma_commit_w<1>(done_bar, leader);
    }
    // ---- the fp32 tile goes to shared memory (the stages are free: every copy has been multiplied), lines along the output's
    // contiguous index, so that stores are coalesced whatever the block widths are and a cluster can sum its slices ----
    asm volatile("cp.async.wait_all;" ::: "memory");
    __syncwarp();
    const bool ok = mbar_wait_warp(done_bar, 0, ctl, p.status);
    tc_fence_after();
    const bool n_minor = p.C.kc != 0;
    const int pitch = (n_minor ? BN : BM) + 4, lines = n_minor ? BM : BN, mine = lines / split;   // the lines each CTA of the cluster stores
    float* tile = reinterpret_cast<float*>(smem);
    if (split > 1) cluster_sync_all();       // every CTA's stages are free
    constexpr int EPI_WARPS = BN >= 128 ? 8 : 4;
    if (ok && warp < EPI_WARPS) {
        const int q = warp & 3, r = q * 32 + lane;
        for (int cc = (warp >> 2) * 32; cc < BN; cc += (EPI_WARPS / 4) * 32) {
            uint32_t v[32];
            tmem_ld32(tmem + ((uint32_t)(q * 32) << 16) + cc, v);
            tmem_ld_wait();
#pragma unroll
            for (int acc = 1; acc < ACC; ++acc) {
                uint32_t w[32];
                tmem_ld32(tmem + ((uint32_t)(q * 32) << 16) + acc * BN + cc, w);
                tmem_ld_wait();
#pragma unroll
                for (int e = 0; e < 32; ++e) v[e] = __float_as_uint(__uint_as_float(v[e]) + __uint_as_float(w[e]));
            }
            if (split == 1) {
                if (n_minor) {
#pragma unroll
                    for (int e = 0; e < 32; e += 4) *reinterpret_cast<uint4*>(tile + r * pitch + cc + e) = make_uint4(v[e], v[e + 1], v[e + 2], v[e + 3]);
                } else {
#pragma unroll
                    for (int e = 0; e < 32; ++e) tile[(cc + e) * pitch + r] = __uint_as_float(v[e]);
                }
            } else if (n_minor) {            // to the line's owner, as the lines of slice `rank`
                const uint32_t at = mapa_cluster(base + (uint32_t)((rank * mine + r % mine) * pitch + cc) * 4u, (uint32_t)(r / mine));
#pragma unroll
                for (int e = 0; e < 32; e += 4) st_cluster16(at + e * 4, v[e], v[e + 1], v[e + 2], v[e + 3]);
            } else {
#pragma unroll
                for (int e = 0; e < 32; ++e)
                    st_cluster4(mapa_cluster(base + (uint32_t)((rank * mine + (cc + e) % mine) * pitch + r) * 4u, (uint32_t)((cc + e) / mine)), v[e]);
            }
        }
    }
    tc_fence_before();
    __syncthreads();
    if (split > 1) cluster_sync_all();       // the slices have arrived
    // ---- every CTA of the cluster stores its share of the tile's lines ----
    if (ctl[0] == 0) {
        const Rel& o = p.C;
        const int ppl = (n_minor ? BN : BM) / 8;
        const Dim &dl = n_minor ? o.r : o.k, &dc = n_minor ? o.k : o.r;   // of the output: r = m, k = n
        const StoreCtx sc = {tile, pitch, split, mine * pitch, n_minor ? m0 : n0, n_minor ? m_end : n_end, n_minor ? n0 : m0, n_minor ? n_end : m_end, p.f16, p.c_esize};
        static_assert(C::THREADS % (BN / 8) == 0 && C::THREADS % (BM / 8) == 0, "a thread keeps its column piece");
        const int l0 = mine * rank, l = l0 + (int)threadIdx.x / ppl, l1 = l0 + mine, c = ((int)threadIdx.x % ppl) * 8, step = C::THREADS / ppl;
        const BatchAt ba = batch_at(o, bx);
        if (o.equal) store_walk_g<true>(o, dl, dc, ba, sc, l0, l, l1, step, c);
        else store_walk_g<false>(o, dl, dc, ba, sc, l0, l, l1, step, c);
    }
    // ---- teardown ----
    __syncthreads();
    if (warp == MMA_WARP) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "n"(BN * ACC) : "memory");
}

// ---- host -----------------------------------------------------------------------------------------------------
template <int BN, bool RAW, int ACC>
ja_status_t launch(const Params& p, cudaStream_t st) {
    static bool configured[64] = {};
    int dev = 0;
    cudaGetDevice(&dev);
    if (!configured[dev & 63]) {
        JA_CUDA(cudaFuncSetAttribute(contract_tc_kernel<BN, RAW, ACC>, cudaFuncAttributeMaxDynamicSharedMemorySize, Cfg<BN, RAW>::SMEM));
        configured[dev & 63] = true;
    }
    const dim3 grid((unsigned)(p.tiles_m * p.tiles_n * p.split), (unsigned)p.batch[1], (unsigned)p.batch[0]);
    JA_CUDA(ja_launch_kernel_after(contract_tc_kernel<BN, RAW, ACC>, grid, Cfg<BN, RAW>::THREADS, Cfg<BN, RAW>::SMEM, (unsigned)p.split, st, p));
    return JA_OK;
}

}  // namespace

struct ContractTcPlan {
    Params p;
    int bn;
    bool raw;
};

ja_status_t ja_contract_tc_plan(const std::string& ta, const std::string& tb, const std::string& tc, const ja_relation* A, const ja_relation* B,
                                const ja_relation* C, std::shared_ptr<ContractTcPlan>* out, double* est_us) {
    out->reset();
    if (A->dtype == JA_F32 || B->dtype != A->dtype || (C->dtype != JA_F32 && C->dtype != A->dtype)) return JA_OK;
    ProductRoles roles;
    if (!product_roles(ta, tb, tc, &roles) || !fits_32_bits(A) || !fits_32_bits(B) || !fits_32_bits(C)) return JA_OK;
    char m = roles.m, n = roles.n;
    const char k = roles.k;
    auto has = [](const std::string& t, char c) { return t.find(c) != std::string::npos; };
    auto extent_of = [&](char c) { return c ? (has(ta, c) ? A->extent[ta.find(c)] : B->extent[tb.find(c)]) : (int64_t)1; };
    std::shared_ptr<ContractTcPlan> plan(new ContractTcPlan());
    Params& p = plan->p;
    memset(&p, 0, sizeof p);
    int64_t M = extent_of(m), N = extent_of(n);
    const int64_t K = extent_of(k);
    // The tile's 128 rows go to the larger index and its BN columns to the smaller one where that is short (a decoding step's
    // tokens): the other operand is then the stream, and it fills whole stages. Otherwise the columns are the output's contiguous index.
    const bool swap = M <= 64 ? N > M : (N > 64 && tc.back() == m);
    const ja_relation *rel_a = swap ? B : A, *rel_b = swap ? A : B;
    const std::string &t_a = swap ? tb : ta, &t_b = swap ? ta : tb;
    if (swap) { std::swap(m, n); std::swap(M, N); }
    fill_rel(&p.A, rel_a, t_a, m, k, roles.batch, 8);
    fill_rel(&p.B, rel_b, t_b, n, k, roles.batch, 8);
    fill_rel(&p.C, C, tc, m, n, roles.batch, 8);
    p.M = (int)M; p.N = (int)N; p.K = (int)K;
    for (int i = 0; i < MAX_BATCH; ++i) p.batch[i] = (int)extent_of(roles.batch[i]);
    p.f16 = A->dtype == JA_F16;
    p.c_esize = C->esize;
    p.group_m = 8;
    // ---- tile width and split: the cheapest under a small model of measured times ----
    // A CTA's stage of 64 contracted cells takes `alone` us by itself (the latency of one trip through the pipeline) and an SM
    // takes `busy` us per stage when its CTAs overlap; a cluster costs its barriers and the remote reads of its partial tiles.
    const int64_t nb = (int64_t)p.batch[0] * p.batch[1], chunks = (K + BK - 1) / BK;
    const int sms = ja_sm_count();
    const bool raw = p.A.g == 1 || p.B.g == 1;
    int best_bn = 64, best_split = 1;
    double best = 1e30;
    // Tiles stay inside intervals where an odd row index is the contiguous one and its intervals are long: a piece that straddles
    // two intervals is read cell by cell, and one such CTA was twice as slow as the others (3627 = 1813 + 1814 columns: 188 -> 109 us).
    auto cut_of = [&](const Rel& o, const ja_relation* r, const std::string& term, char letter, int width, int64_t* tiles) -> int {
        const std::vector<int64_t>& sp = r->splits[term.find(letter)];
        const int64_t whole = (sp.back() + width - 1) / width;
        *tiles = whole;
        if (o.g != 1 || o.kc || sp.size() < 3) return 0;
        int64_t w = 0;
        for (size_t i = 1; i < sp.size(); ++i) w = std::max(w, sp[i] - sp[i - 1]);
        const int64_t per = (w + width - 1) / width, cut = per * ((int64_t)sp.size() - 1);
        if (cut * 8 > whole * 9) return 0;   // an eighth more tiles at most
        *tiles = cut;
        return (int)per;
    };
    // f32 output: four accumulators (256 of the SM's 512 tensor-memory columns for each of two CTAs of 64-column tiles), and slices short
    // enough, where a cluster can be that large, that a chain is 256 cells (bf16) or 128 (f16, whose products have more bits to lose).
    // Error against 64 bits, normal operands, 512 / 2048 contracted cells: bf16 1.2e-7 / 2.3e-7 (one accumulator 4.7e-7 / 2.1e-6; f32 FMAs
    // one after the other 1.6e-7 / 3.9e-7), f16 1.9e-7 / 1.9e-7 (6.4e-7 / 2.5e-6; 4.0e-7 / 8.0e-7). "bij,bkj->bik" 32 x 512 x 512 x 512
    // 31 -> 43 us; 8 x 128 x 256 x 512 9.7 -> 9.9.
    const bool f32_out = C->dtype == JA_F32;
    int least = 1;
    while (f32_out && least < 8 && chunks > (p.f16 ? 8 : 16) * least) least *= 2;
    for (int bn : {64, 128, 256}) {
        if ((raw && bn == 256) || (f32_out && bn != 64)) continue;
        const int per_sm = bn == 256 || raw ? 1 : 2;
        const double busy = bn == 256 ? 0.51 : bn == 128 ? 0.29 : 0.235, alone = raw ? 1.3 : bn == 256 ? 0.51 : bn == 128 ? 0.46 : 0.36;
        const double fixed = bn == 256 ? 6.0 : bn == 128 ? 4.5 : 3.5;
        int64_t tm, tn;
        cut_of(p.A, rel_a, t_a, m, BM, &tm);
        cut_of(p.B, rel_b, t_b, n, bn, &tn);
        for (int s : {1, 2, 4, 8}) {
            if (s < least) continue;
            if (s > 1 && chunks < 4 * s) break;
            const int64_t ctas = nb * tm * tn * s, slots = (int64_t)sms * per_sm * (s > 1 ? 4 : 5) / 5;   // clusters do not pack a GPC fully
            const int64_t waves = (ctas + slots - 1) / slots, last = ctas - (waves - 1) * slots, on_sm = (waves - 1) * per_sm + (last + sms - 1) / sms;
            const double each = (double)((chunks + s - 1) / s);
            const double t = std::max(on_sm * each * busy, waves * each * alone) + waves * fixed + (s > 1 ? 2.0 + 0.05 * ctas : 0.0);
            if (t < best) { best = t; best_bn = bn; best_split = s; }
        }
    }
    int64_t tiles_m, tiles_n;
    p.cut_m = cut_of(p.A, rel_a, t_a, m, BM, &tiles_m);
    p.cut_n = cut_of(p.B, rel_b, t_b, n, best_bn, &tiles_n);
    p.tiles_m = (int)tiles_m;
    p.tiles_n = (int)tiles_n;
    if (tiles_m * tiles_n * best_split >= (1ll << 31) || p.batch[0] > 65535 || p.batch[1] > 65535) return JA_OK;
    p.split = best_split;
    plan->bn = best_bn;
    plan->raw = raw;
    // Where the contracted index is the contiguous one of an operand in pieces of one cell, most stages hold the end of an interval or the
    // index's odd pitch, and a stage takes longer by itself than the model says: 3.3 us, and 240 over the cells of an interval
    // (64 x 314 x 320 in eight intervals 46 us, in two 22). The choice above stays; the estimate tells.
    if ((p.A.kc && p.A.g == 1) || (p.B.kc && p.B.g == 1)) {
        const int64_t ctas = nb * tiles_m * tiles_n * best_split, slots = (int64_t)sms * (best_split > 1 ? 4 : 5) / 5, per = K / std::max(p.A.k.nblk, 1);
        best = std::max(best, (double)((ctas + slots - 1) / slots) * ((double)((chunks + best_split - 1) / best_split) * (3.3 + 240.0 / (double)std::max<int64_t>(per, 1)) + 4.0));
    }
    if (est_us) *est_us = best;
    *out = plan;
    return JA_OK;
}

ja_status_t ja_launch_contract_tc(const ContractTcPlan& plan, cudaStream_t st) {
    Params p = plan.p;
    p.status = ja_device_status_word(st);
    if (!p.status) return ja_fail(JA_ERR_CUDA, "cannot resolve the device status word");
    p.wait_cap_us = (uint32_t)ja_config().wait_cap_us;
    ja_status_t s;
    if (plan.p.c_esize == 4) s = plan.raw ? launch<64, true, 4>(p, st) : launch<64, false, 4>(p, st);
    else if (plan.raw) s = plan.bn == 64 ? launch<64, true, 1>(p, st) : launch<128, true, 1>(p, st);
    else s = plan.bn == 64 ? launch<64, false, 1>(p, st) : plan.bn == 128 ? launch<128, false, 1>(p, st) : launch<256, false, 1>(p, st);
    if (s == JA_OK) ja_count_launch();
    return s;
}

// [2048, 11008] x [11008, 4096], k cut 64 ways (pieces of 4) 253 us against 175 in one block a side, [8000, 5000] x [5000, 5000] cut in four
// (pieces of 2) 1249 against an estimate of 362, [4001, 3000] x [3000, 2504] in unequal row blocks 130 against 90. Pieces of one cell
// are part of the estimate.
double ja_contract_tc_pieces(const ContractTcPlan& plan) {
    const int g = std::min(plan.p.A.g, plan.p.B.g);
    return std::max(g == 4 ? 1.45 : g == 2 ? 3.4 : 1.0, g > 1 && !(plan.p.A.equal && plan.p.B.equal) ? 1.4 : 1.0);
}

// Tensor-core matmul join-agg "ij,jk->ik" (MUL / SUM) for bf16 relations with uniform blocks.
//
// One persistent CTA per SM. For every output tile (128 rows x up to 256 columns of ONE output key, or of
// several adjacent output keys when blocks are narrow) the CTA walks the function specs that share that
// output key in ascending order of the contracted block index j -- the SUM aggregation of Definition 3.7 is
// the accumulation of all those tuples into one fp32 accumulator in tensor memory; only the aggregated block
// is written (Recompose = the store at the key's offset).
//
//   warp 0      TMA producer: cp.async.bulk.tensor straight from the block-key layout. A relation with
//               uniform blocks is a rank-4 tensor (col in block, row in block, col-block, row-block), so one
//               tensor map per operand addresses every block; ragged tiles rely on zero fill inside a block.
//   warp 1      tcgen05.mma issuer (one elected lane), kind::f16, M=128, N<=256, K=16, A K-major and
//               B MN-major (weights are [in, out] row-major), both under the 128-byte swizzle.
//   warps 2..5  epilogue: tcgen05.ld of the fp32 accumulator, one RNE rounding to bf16, 16-byte stores.
//
// Two accumulator stages (2 x 256 TMEM columns) let the epilogue of tile t overlap the mainloop of tile t+1.
// Every mbarrier wait is bounded; on expiry the CTA records JA_ERR_TIMEOUT, drains its copies and exits.
//
// The kernel exists in two forms (template parameter CG):
//   CG = 1  one CTA per 128 x 256 tile, tcgen05.mma.cta_group::1.
//   CG = 2  a cluster of two CTAs (two SMs) per 256 x 256 tile, tcgen05.mma.cta_group::2 issued by the leader
//           CTA: each CTA stages its own 128 rows of A and its own half of the tile's B columns (plain TMA
//           loads, no multicast), so every SM pulls a third less operand data per flop through L2 and can
//           keep six stages in flight; each CTA holds the accumulator rows of its own half in its own TMEM.
#include <cuda.h>
#include <stdlib.h>
#include <string.h>

#include <algorithm>
#include <atomic>

#include "ja_device.cuh"
#include "ja_launch.cuh"
#include "ja_ptx.cuh"

namespace {

using namespace ja_ptx;

constexpr int BM = 128, BN = 256;
constexpr int NUM_THREADS = 192;
// BK = contraction depth of one pipeline stage. The two-CTA form stages 128-deep chunks so that every box it issues
// (A: 128 rows x 64 k, B: 128 k x 64 columns) is 16 KiB: fewer, larger TMA copies per flop than 64-deep stages.
// What bounds this kernel is operand delivery, not the tensor pipe: timing-only ablations on [16384, 4096] x [4096, 4096]
// with half of the B boxes not loaded ran at 1617 TFLOP/s against 1391, with half of A as well at 1821. A form that cuts
// the bytes per flop by a quarter -- tiles of 256 x 512 on both accumulators, A fetched once per 512 columns -- was built,
// passed the parity tests and measured SLOWER, because the shared memory left holds either four 64-deep stages of 8 KiB
// B boxes (1196 TFLOP/s on the same product) or two 128-deep stages (1339; 1205 against 1330-1418 on the up-projections):
// more, smaller copies or too shallow a pipeline cost more than the saved bytes bring.
template <int CG> struct Cfg {
    static constexpr int BK = CG == 1 ? 64 : 128;
    static constexpr int STAGES = CG == 1 ? 4 : 3;
    static constexpr int A_HALF_BYTES = BM * 64 * 2;                 // 128 rows x 64 k under the 128-byte swizzle
    static constexpr int A_STAGE_BYTES = A_HALF_BYTES * (BK / 64);
    static constexpr int B_CHUNK_BYTES = BK * 64 * 2;                // one box: BK k-rows x 64 columns
    static constexpr int B_STAGE_BYTES = B_CHUNK_BYTES * (BN / CG / 64);
    static constexpr int SMEM_BYTES = STAGES * (A_STAGE_BYTES + B_STAGE_BYTES) + 1024 /*align*/ + 256 /*barriers*/;
    // ANYC: 32 rows x 32 columns of every epilogue warp on their way to stores along the rows (rows of 34 cells: no bank conflicts)
    static constexpr int SMEM_BYTES_ANYC = SMEM_BYTES + 4 * 32 * 34 * 2;
};

struct GemmParams {
    char* c_base;
    const int64_t* c_blk_off;  // device: byte offsets of the output blocks
    int32_t* status;           // status word of the launching stream (set at launch)
    uint32_t wait_cap_us;      // limit of every bounded wait (set at launch)
    int32_t bm, bk, bn;        // block extents along i, j, k
    int32_t nbm, nbk, nbn;     // blocks along i, j, k
    int32_t c_bm, c_bn, c_nbn; // block extents of the output, and its blocks along k (other than the operands' where those were copied)
    int32_t M, N;              // tensor extents along i, k
    int32_t a_box_rows;        // rows per A box (= min(bm, 128))
    int32_t a_boxes;           // A boxes per tile: 128 / bm where bm divides 128 (tiles cut from global rows), else 1
    int32_t m_tiles, n_tiles;  // tile grid (tiles are 128*CG rows x up to 256 columns)
    int32_t tiles_per_mblk;    // >= 1 when row tiles never leave a block, 0 when tiles are cut from global rows
    int32_t tiles_per_nblk;    // >= 1 when tiles stay inside one column block, 0 when tiles span blocks
    int32_t group_m;           // row tiles per rasterisation band
    int32_t heavy_first;       // 1: full-width tiles are scheduled before the narrow last tile of every column block (see tile_of_iter)
    // fused epilogue (a join-agg chain executed in one pass, the intermediate never stored)
    int32_t epi;               // EPI_*
    int32_t bn_tile;           // output columns per tile: 256, or 128 for EPI_SWIGLU (two 128-column products per tile)
    int32_t tile0, tile_end;   // the tiles of this launch
    int32_t split;             // SPLIT: slices of the contracted index = CTA pairs per cluster
    int32_t n_copies;          // 1: SUM over all contracted blocks (aggregated output). nbk: join only -- tile (c, ., .) covers the
                               // single contracted block c and is stored to copy c of a partial relation [c, i, k]
    int32_t c_esize;           // bytes per output cell: 2 (bf16 / f16) or 4 (f32, partial relations only)
    int32_t f16;               // cell type of the operands (and of a 2-byte output): 0 = bf16, 1 = f16
    const char* r_base;        // EPI_ADD: payload of the relation added to the product (tiled exactly like the output)
    const float2* rope_table;  // EPI_ROPE: (cos, sin)[position][pair]
    RelView c;                 // ANYC: the output, whose blocks may have any shapes
    int32_t rope_S, rope_D;    // EPI_ROPE: positions per sequence (row % rope_S), rotated extent (column % rope_D)
};
enum { EPI_NONE = 0, EPI_ADD = 1, EPI_ROPE = 2, EPI_SWIGLU = 3 };

// What one CTA does for one tile: its own 128 rows, and (CG 2) its own half of the tile's columns as B operand.
struct TileCoord {
    int mb, r0;          // row block and first row inside it of THIS CTA's 128 rows
    int row_g0;          // first global row of this CTA's rows
    int rows;            // valid rows (0..128)
    int n_g0, nb, c0;    // first global column of the tile / its column block / first column inside it
    int width;           // valid columns of the tile (multiple of 8)
    int jb0, jb1;        // contracted blocks [jb0, jb1) accumulated into this tile
    int copy;            // copy index of a partial relation (0 for an aggregated output)
};

template <int CG>
__device__ __forceinline__ TileCoord tile_coord(const GemmParams& p, int t, int cta_rank) {
    TileCoord tc;
    // join-only form: copies are the slowest tile coordinate, so tiles in flight share one contracted block
    const int per_copy = p.m_tiles * p.n_tiles;
    tc.copy = t / per_copy;
    t -= tc.copy * per_copy;
    tc.jb0 = p.n_copies > 1 ? tc.copy : 0;
    tc.jb1 = p.n_copies > 1 ? tc.copy + 1 : p.nbk;
    // heavy-first schedule: t counts the full-width tiles of all column blocks first, then the narrow last tiles
    int n_tiles_v = p.n_tiles;
    bool narrow = false;
    if (p.heavy_first) {
        const int full_tiles = p.m_tiles * p.nbn * (p.tiles_per_nblk - 1);
        narrow = t >= full_tiles;
        if (narrow) t -= full_tiles;
        n_tiles_v = narrow ? p.nbn : p.nbn * (p.tiles_per_nblk - 1);
    }
    // banded rasterisation: tiles that run at the same time cover group_m row tiles x several column tiles, so the
    // operand strips they stream fit in L2 together. (A second level -- super-columns of column tiles whose B strip would
    // stay in L2 while every row band passes over it -- was built and measured on the block's projections: launch times
    // within 1 % of this order for strips of 16 to 48 tiles, and MORE DRAM traffic, 1.9-2.5 GB against 1.7 GB per
    // up-projection launch, so it is not here.)
    const int band_sz = p.group_m * n_tiles_v;
    const int band = t / band_sz, tin = t - band * band_sz;
    const int rows_in_band = min(p.group_m, p.m_tiles - band * p.group_m);
    const int mt = band * p.group_m + tin % rows_in_band;
    int nt = tin / rows_in_band;
    if (p.heavy_first) nt = narrow ? nt * p.tiles_per_nblk + p.tiles_per_nblk - 1 : (nt / (p.tiles_per_nblk - 1)) * p.tiles_per_nblk + nt % (p.tiles_per_nblk - 1);
    if (p.tiles_per_mblk > 0) {   // 128-row tiles stay inside a block; a pair of CTAs takes two consecutive ones
        const int rt = mt * CG + cta_rank;
        tc.mb = rt / p.tiles_per_mblk;
        tc.r0 = (rt % p.tiles_per_mblk) * BM;
        tc.rows = tc.mb < p.nbm ? min(BM, p.bm - tc.r0) : 0;   // an odd number of row tiles: the last pair's second one is all fill
        tc.row_g0 = tc.mb * p.bm + tc.r0;
    } else {                      // tiles cut from global rows (block height divides 128, or is a multiple of 128)
        tc.row_g0 = mt * (BM * CG) + cta_rank * BM;
        tc.mb = tc.row_g0 / p.bm;
        tc.r0 = tc.row_g0 % p.bm;
        tc.rows = max(0, min(BM, p.M - tc.row_g0));
    }
    if (p.tiles_per_nblk > 0) {
        tc.nb = nt / p.tiles_per_nblk;
        tc.c0 = (nt % p.tiles_per_nblk) * p.bn_tile;
        tc.width = min(p.bn_tile, p.bn - tc.c0);
        tc.n_g0 = tc.nb * p.bn + tc.c0;
    } else {
        tc.n_g0 = nt * p.bn_tile;
        tc.nb = tc.n_g0 / p.bn;
        tc.c0 = tc.n_g0 % p.bn;
        tc.width = min(p.bn_tile, p.N - tc.n_g0);
    }
    return tc;
}

// Which tile a CTA group works on in its i-th round, or -1 when it has none left. Plain round-robin, or -- with the heavy-first
// order, where tiles come sorted by weight -- round-robin that reverses direction every round, so that the groups that got an
// extra full tile in the last full-width round are the last to be handed narrow ones.
__device__ __forceinline__ int tile_of_iter(const GemmParams& p, int i, int first, int step, int total) {
    const int t = i * step + ((p.heavy_first && (i & 1)) ? step - 1 - first : first);
    return t < total ? t : -1;
}

// F16: cell type of the operands and of a 2-byte output -- bf16 or f16 (a compile-time choice: a select between the two
// conversions in the epilogue cost the plain contraction a tenth of its rate)
// SPLIT: a tile's contracted index over a cluster of CTA pairs, one tile a cluster, the slices' f32 sums taken through distributed shared
// memory. What bounds it is the sum and the cluster's start and end, 10 us of [512, 4096] x [4096, 4096]'s 28.8 in a queue of calls (33.9 as whole tiles).
// ANYC: the output's tiling is not the one that TMA sees of the operands (operands staged by k_stage.cu, rows of no whole 16 bytes): every
// cell is located through its key table and stored by itself, 32 columns of a row at a time
template <int CG, bool F16, bool SPLIT, bool ANYC>
__global__ void __launch_bounds__(NUM_THREADS, 1)
gemm_tc_kernel(const __grid_constant__ CUtensorMap tmA, const __grid_constant__ CUtensorMap tmB,
               const __grid_constant__ CUtensorMap tmB2, const GemmParams p) {
    constexpr int STAGES = Cfg<CG>::STAGES, BK = Cfg<CG>::BK;
    constexpr int A_STAGE_BYTES = Cfg<CG>::A_STAGE_BYTES, A_HALF_BYTES = Cfg<CG>::A_HALF_BYTES;
    constexpr int B_STAGE_BYTES = Cfg<CG>::B_STAGE_BYTES, B_CHUNK_BYTES = Cfg<CG>::B_CHUNK_BYTES;
    extern __shared__ uint8_t smem_raw[];
    const uint32_t raw = smem_u32(smem_raw);
    const uint32_t base = (raw + 1023u) & ~1023u;  // swizzle atoms need 1024-byte alignment
    uint8_t* smem = smem_raw + (base - raw);
    const uint32_t sA = base, sB = base + STAGES * A_STAGE_BYTES;
    uint64_t* bars = reinterpret_cast<uint64_t*>(smem + STAGES * (A_STAGE_BYTES + B_STAGE_BYTES));
    // bars[0..S) full, [S..2S) empty, [2S..2S+2) tmem_full, [2S+2..2S+4) tmem_empty
    const uint32_t bar0 = smem_u32(bars);
    auto full_bar = [&](int s) { return bar0 + 8u * s; };
    auto empty_bar = [&](int s) { return bar0 + 8u * (STAGES + s); };
    auto tfull_bar = [&](int a) { return bar0 + 8u * (2 * STAGES + a); };
    auto tempty_bar = [&](int a) { return bar0 + 8u * (2 * STAGES + 2 + a); };
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(bars + 2 * STAGES + 4);
    volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);

    const int warp = __shfl_sync(0xffffffffu, (int)threadIdx.x / 32, 0), lane = threadIdx.x % 32;   // warp-uniform by construction
    const int cl_rank = CG == 2 ? (int)cluster_ctarank() : 0;
    const int cta_rank = SPLIT ? cl_rank & 1 : cl_rank;           // 0 = leader of the pair
    const uint32_t pair0 = SPLIT ? (uint32_t)(cl_rank & ~1) : 0;  // the leader's rank in the cluster
    if (threadIdx.x == 0) {
        for (int s = 0; s < STAGES; ++s) {
            mbar_init(full_bar(s), 1);    // CG 2: only the leader's is used; both CTAs' copies complete_tx on it
            mbar_init(empty_bar(s), 1);
        }
        for (int a = 0; a < 2; ++a) {
            mbar_init(tfull_bar(a), 1);
            mbar_init(tempty_bar(a), 4 * CG);  // one arrival per epilogue warp of every CTA of the group
        }
        wait_ctl_init(abort_flag, p.wait_cap_us);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 1) {  // all 512 TMEM columns: two 128 x 256 fp32 accumulators (in each CTA of a pair)
        if (CG == 1) {
            asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], 512;" ::"r"(smem_u32(tmem_slot)) : "memory");
            asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
        } else {
            asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], 512;" ::"r"(smem_u32(tmem_slot)) : "memory");
            asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
        }
    }
    tc_fence_before();
    __syncthreads();
    if (CG == 2) cluster_sync_all();   // the peer's barriers exist before anything remote touches them
    tc_fence_after();
    const uint32_t tmem_base = __shfl_sync(0xffffffffu, *tmem_slot, 0);

    const int kchunks = (p.bk + Cfg<CG>::BK - 1) / Cfg<CG>::BK;
    const int total_tiles = p.tile_end;
    const int first_tile = SPLIT ? p.tile0 + (int)blockIdx.x / (2 * p.split) : (int)blockIdx.x / CG, tile_step = SPLIT ? p.tile_end : (int)gridDim.x / CG;
    // the stages [ch0, ch1) of a tile that this CTA group accumulates: all of its contracted blocks', or (SPLIT) one slice of them
    auto stages_of = [&](const TileCoord& tc, int* ch0, int* ch1) {
        *ch0 = tc.jb0 * kchunks;
        *ch1 = tc.jb1 * kchunks;
        if (SPLIT) {
            const int64_t n = *ch1;
            *ch0 = (int)(n * (cl_rank >> 1) / p.split);
            *ch1 = (int)(n * ((cl_rank >> 1) + 1) / p.split);
        }
    };

    if (warp == 0) {
        // ================= TMA producer (one per CTA) =================
        if (lane == 0) {
            uint32_t last_parity[STAGES];
            bool issued[STAGES];
            for (int s = 0; s < STAGES; ++s) { last_parity[s] = 0; issued[s] = false; }
            int stage = 0;
            uint32_t phase = 0;
            bool ok = true;
            for (int it = 0; ok; ++it) {
                const int t = tile_of_iter(p, it, first_tile, tile_step, total_tiles);
                if (t < 0) break;
                const TileCoord tc = tile_coord<CG>(p, t, cta_rank);
                // EPI_SWIGLU: the MMA tile is [128 columns of x W1 | the same 128 columns of x W3]
                const int n_mma = p.epi == EPI_SWIGLU ? 2 * tc.width : (tc.width + 15) / 16 * 16;
                const int my_cols = n_mma / CG;                    // B columns this CTA stages
                const int my_c0 = cta_rank * my_cols;              // their offset inside the tile
                const int nchunks = (my_cols + 63) / 64;
                const uint32_t tx = (uint32_t)CG * ((uint32_t)(p.a_boxes * p.a_box_rows) * (BK * 2) + nchunks * B_CHUNK_BYTES);
                int ch, ch1;
                stages_of(tc, &ch, &ch1);
                for (int jb = ch / kchunks, kc = ch - jb * kchunks; ch < ch1; ++jb, kc = 0) {    // the tuples of this output key, ascending j
                    for (; kc < kchunks && ch < ch1; ++kc, ++ch) {
                        if (!mbar_wait(empty_bar(stage), phase ^ 1, abort_flag, p.status)) { ok = false; ch = ch1; break; }
                        uint32_t fb = full_bar(stage);
                        if (CG == 2) fb = mapa_cluster(fb, pair0);  // completion is counted on the leader's barrier
                        if (cta_rank == 0) mbar_expect_tx(full_bar(stage), tx);
                        issued[stage] = true;
                        last_parity[stage] = phase;
                        // A: boxes of a_box_rows rows x 64 k, one set per 64-deep half of the stage
                        const int nboxes = p.a_boxes;
                        for (int kh = 0; kh < BK / 64; ++kh)
                            for (int bx = 0; bx < nboxes; ++bx)
                                tma_load_4d<CG>(sA + stage * A_STAGE_BYTES + kh * A_HALF_BYTES + bx * p.a_box_rows * 128, &tmA, fb,
                                                kc * BK + kh * 64, tc.r0, jb, tc.mb + bx);
                        // B: one box of BK k-rows x 64 columns per 64-column chunk
                        for (int c = 0; c < nchunks; ++c) {
                            int mc = my_c0 + 64 * c;               // column of the MMA tile this box starts at
                            const CUtensorMap* tb = &tmB;
                            if (p.epi == EPI_SWIGLU && mc >= p.bn_tile) { tb = &tmB2; mc -= p.bn_tile; }
                            int nb, cin;
                            if (p.tiles_per_nblk > 0) { nb = tc.nb; cin = tc.c0 + mc; }
                            else { int g = tc.n_g0 + mc; nb = g / p.bn; cin = g % p.bn; }
                            tma_load_4d<CG>(sB + stage * B_STAGE_BYTES + c * B_CHUNK_BYTES, tb, fb, cin, kc * BK, nb, jb);
                        }
                        if (++stage == STAGES) { stage = 0; phase ^= 1; }
                    }
                }
            }
            // drain: wait (bounded) for copies already in flight before the CTA may exit. In a pair both CTAs' copies
            // complete on the leader's barriers, and the peer cannot leave before the leader reaches the cluster barrier.
            if (!ok && cta_rank == 0) {
                for (int s = 0; s < STAGES; ++s) {
                    if (!issued[s]) continue;
                    const uint64_t t0 = global_ns();
                    while (!mbar_try_wait(full_bar(s), last_parity[s]) && global_ns() - t0 < 200000000ull) {}
                }
            }
            (void)issued; (void)last_parity;
        }
        __syncwarp();
    } else if (warp == 1) {
        // ================= MMA issuer (leader CTA only): the whole warp runs the loop, one elected lane issues =================
        if (cta_rank == 0) {
            const uint32_t leader = elect_one();
            int stage = 0;
            uint32_t phase = 0;
            uint32_t acc_phase[2] = {0, 0};
            bool ok = true;
            for (int it = 0; ok; ++it) {
                const int t = tile_of_iter(p, it, first_tile, tile_step, total_tiles);
                if (t < 0) break;
                const TileCoord tc = tile_coord<CG>(p, t, 0);
                const int acc = it & 1;
                const uint32_t n_mma = p.epi == EPI_SWIGLU ? (uint32_t)(2 * tc.width) : (uint32_t)((tc.width + 15) / 16 * 16);
                // D f32; A and B both bf16 (format 1) or both f16 (format 0); B MN-major
                constexpr uint32_t fmt = F16 ? 0u : 1u;
                const uint32_t idesc = (1u << 4) | (fmt << 7) | (fmt << 10) | (1u << 16) | ((n_mma >> 3) << 17) |
                                       ((uint32_t)((BM * CG) >> 4) << 24);
                if (!mbar_wait(tempty_bar(acc), acc_phase[acc] ^ 1, abort_flag, p.status)) { ok = false; break; }
                acc_phase[acc] ^= 1;
                tc_fence_after();
                const uint32_t d_tmem = tmem_base + acc * BN;
                uint32_t accumulate = 0;
                int ch, ch1;
                stages_of(tc, &ch, &ch1);
                for (int kc = ch % kchunks; ch < ch1; kc = 0) {
                    for (; kc < kchunks && ch < ch1; ++kc, ++ch) {
                        if (!mbar_wait(full_bar(stage), phase, abort_flag, p.status)) { ok = false; ch = ch1; break; }
                        tc_fence_after();
                        const int kvalid = min(BK, p.bk - kc * BK);
                        const int k16 = (kvalid + 15) / 16;
                        const uint32_t a_addr = sA + stage * A_STAGE_BYTES;
                        const uint32_t b_addr = sB + stage * B_STAGE_BYTES;
                        // A: K-major, 16 k = 32 bytes inside the swizzle atom, 64 k per half; B: MN-major, 16 k-rows =
                        // 2048 bytes, 64-column groups BK*128 bytes apart
                        if (k16 == BK / 16) {   // a full stage: straight-line code, no branch between two tcgen05.mma
#pragma unroll
                            for (int kk = 0; kk < BK / 16; ++kk) {
                                const uint64_t da = desc_sw128(a_addr + (kk >> 2) * A_HALF_BYTES + (kk & 3) * 32, 16);
                                const uint64_t db = desc_sw128(b_addr + kk * 2048, BK * 128);
                                umma_bf16_w<CG>(d_tmem, da, db, idesc, kk > 0 ? 1u : accumulate, leader);
                            }
                        } else {
                            for (int kk = 0; kk < k16; ++kk) {
                                const uint64_t da = desc_sw128(a_addr + (kk >> 2) * A_HALF_BYTES + (kk & 3) * 32, 16);
                                const uint64_t db = desc_sw128(b_addr + kk * 2048, BK * 128);
                                umma_bf16_w<CG>(d_tmem, da, db, idesc, kk > 0 ? 1u : accumulate, leader);
                            }
                        }
                        accumulate = 1;
                        umma_commit_w<CG>(empty_bar(stage), leader, pair0);  // frees the smem stage (in both CTAs) once these MMAs have read it
                        if (++stage == STAGES) { stage = 0; phase ^= 1; }
                    }
                }
                if (ok) umma_commit_w<CG>(tfull_bar(acc), leader, pair0);    // accumulator complete -> epilogue(s)
            }
        }
    } else if (!SPLIT) {
        // ================= epilogue (warps 2..5 of every CTA) =================
        const int q = warp & 3;  // TMEM lane group this warp may access
        uint32_t acc_phase[2] = {0, 0};
        bool ok = true;
        const uint32_t tempty0 = CG == 2 ? mapa_cluster(tempty_bar(0), 0) : tempty_bar(0);
        const uint32_t tempty1 = CG == 2 ? mapa_cluster(tempty_bar(1), 0) : tempty_bar(1);
        for (int it = 0; ok; ++it) {
            const int t = tile_of_iter(p, it, first_tile, tile_step, total_tiles);
            if (t < 0) break;
            const TileCoord tc = tile_coord<CG>(p, t, cta_rank);
            const int acc = it & 1;
            if (!mbar_wait(tfull_bar(acc), acc_phase[acc], abort_flag, p.status)) { ok = false; break; }
            acc_phase[acc] ^= 1;
            tc_fence_after();
            const int r = q * 32 + lane;                     // row of this CTA's 128 rows held by this thread
            const int grow = tc.row_g0 + r;                  // global row
            const bool row_ok = r < tc.rows;
            if constexpr (ANYC) {
                int rb = 0, rin = 0;
                if (row_ok) {
                    int lo, hi;
                    rb = ja_interval(p.c, 0, grow, &lo, &hi);
                    rin = grow - lo;
                }
                uint16_t* cells = reinterpret_cast<uint16_t*>(smem + STAGES * (A_STAGE_BYTES + B_STAGE_BYTES) + 256) + q * 32 * 34;
                const int n_rows = min(32, tc.rows - q * 32);
                for (int ch = 0; ch * 32 < tc.width; ++ch) {
                    uint32_t v[32];
                    tmem_ld32(tmem_base + ((uint32_t)(q * 32) << 16) + acc * BN + ch * 32, v);
                    tmem_ld_wait();
#pragma unroll
                    for (int e = 0; e < 16; ++e)
                        *reinterpret_cast<uint32_t*>(cells + lane * 34 + 2 * e) = ja_pack16<F16>(__uint_as_float(v[2 * e]), __uint_as_float(v[2 * e + 1]));
                    __syncwarp();
                    const bool col_ok = ch * 32 + lane < tc.width;
                    const int col = tc.n_g0 + ch * 32 + lane;
                    int cb = 0, cin = 0;
                    int64_t pitch = 0;
                    if (col_ok) {
                        int lo, hi;
                        cb = ja_interval(p.c, 1, col, &lo, &hi);
                        pitch = (int64_t)(hi - lo) * 2;
                        cin = col - lo;
                    }
                    // the warp's rows in one block: row after row. (With every row's block looked up by shuffles a tile took 17 us to store.)
                    const int b0 = __shfl_sync(0xffffffffu, rb, 0), in0 = __shfl_sync(0xffffffffu, rin, 0);
                    if (n_rows > 0 && __shfl_sync(0xffffffffu, rb, n_rows - 1) == b0) {
                        if (col_ok) {
                            char* at = p.c.base + ja_block_at(p.c, b0, cb) + cin * 2 + in0 * pitch;
#pragma unroll 8
                            for (int rr = 0; rr < n_rows; ++rr, at += pitch) *reinterpret_cast<uint16_t*>(at) = cells[rr * 34 + lane];
                        }
                    } else {
                        for (int rr = 0; rr < n_rows; ++rr) {
                            const int b = __shfl_sync(0xffffffffu, rb, rr), in = __shfl_sync(0xffffffffu, rin, rr);
                            if (col_ok) *reinterpret_cast<uint16_t*>(p.c.base + ja_block_at(p.c, b, cb) + cin * 2 + in * pitch) = cells[rr * 34 + lane];
                        }
                    }
                    __syncwarp();
                }
            } else {
            int ib = 0, iin = 0;
            if (row_ok) { ib = grow / p.c_bm; iin = grow % p.c_bm; }
            for (int ch = 0; ch * 32 < tc.width; ++ch) {
                uint32_t v[32];
                tmem_ld32(tmem_base + ((uint32_t)(q * 32) << 16) + acc * BN + ch * 32, v);
                if (p.epi == EPI_SWIGLU) {   // silu(x W1) * (x W3): the W3 product sits 128 columns to the right
                    uint32_t w[32];
                    tmem_ld32(tmem_base + ((uint32_t)(q * 32) << 16) + acc * BN + p.bn_tile + ch * 32, w);
                    tmem_ld_wait();
#pragma unroll
                    for (int i = 0; i < 32; ++i) {
                        const float a = __uint_as_float(v[i]);
                        v[i] = __float_as_uint(a / (1.f + __expf(-a)) * __uint_as_float(w[i]));
                    }
                } else {
                    tmem_ld_wait();
                }
                if (row_ok) {
                    const int gcol = tc.n_g0 + ch * 32;
                    const int kb = gcol / p.c_bn, cin = gcol % p.c_bn;
                    const int64_t off = p.c_blk_off[((int64_t)tc.copy * p.nbm + ib) * p.c_nbn + kb] + ((int64_t)iin * p.c_bn + cin) * p.c_esize;
                    char* dst = p.c_base + off;
                    const int valid = min(32, tc.width - ch * 32);  // multiple of 8
                    if (p.c_esize == 4) {   // partial relation kept in f32: the accumulator is stored as it is
#pragma unroll
                        for (int g = 0; g < 8; ++g)
                            if (g * 4 < valid)
                                *reinterpret_cast<uint4*>(dst + g * 16) = make_uint4(v[g * 4], v[g * 4 + 1], v[g * 4 + 2], v[g * 4 + 3]);
                        continue;
                    }
                    if (p.epi == EPI_ROPE) {
                        // rotate pairs (2p, 2p+1) by the angle of (position, pair): position = row inside its sequence
                        const float2* tab = p.rope_table + ((int64_t)(grow % p.rope_S) * p.rope_D + gcol % p.rope_D) / 2;
#pragma unroll
                        for (int i = 0; i < 32; i += 2) {
                            const float2 cs = tab[i / 2];
                            const float x0 = __uint_as_float(v[i]), x1 = __uint_as_float(v[i + 1]);
                            v[i] = __float_as_uint(x0 * cs.x - x1 * cs.y);
                            v[i + 1] = __float_as_uint(x0 * cs.y + x1 * cs.x);
                        }
                    }
#pragma unroll
                    for (int g = 0; g < 4; ++g) {
                        if (g * 8 < valid) {
                            float f[8];
#pragma unroll
                            for (int e = 0; e < 8; ++e) f[e] = __uint_as_float(v[g * 8 + e]);
                            if (p.epi == EPI_ADD) {   // key-aligned join with the addend relation: same block, same cell
                                const uint4 rv = *reinterpret_cast<const uint4*>(p.r_base + off + g * 16);
                                const uint32_t* pr = reinterpret_cast<const uint32_t*>(&rv);
#pragma unroll
                                for (int e = 0; e < 4; ++e) {
                                    const float2 rf = ja_unpack16<F16>(pr[e]);
                                    f[2 * e] += rf.x;
                                    f[2 * e + 1] += rf.y;
                                }
                            }
                            uint4 o;
                            uint32_t* po = reinterpret_cast<uint32_t*>(&o);
#pragma unroll
                            for (int e = 0; e < 4; ++e) po[e] = ja_pack16<F16>(f[2 * e], f[2 * e + 1]);
                            *reinterpret_cast<uint4*>(dst + g * 16) = o;
                        }
                    }
                }
            }
            }
            tc_fence_before();
            __syncwarp();
            if (lane == 0) {
                if (CG == 1) mbar_arrive(acc ? tempty1 : tempty0);
                else mbar_arrive_cluster(acc ? tempty1 : tempty0);   // the leader's MMA thread owns the accumulators of both CTAs
            }
        }
    }
    if constexpr (SPLIT) {
        // ================= the slices' sum: every row goes to one CTA of the cluster, [slice][row][column] f32 over the stages =================
        const TileCoord tc = tile_coord<CG>(p, first_tile, cta_rank);
        const bool ok = mbar_wait_warp(tfull_bar(0), 0, abort_flag, p.status);
        tc_fence_after();
        cluster_sync_all();   // every product of the cluster has read its stages
        constexpr int PITCH = BN + 4;
        const int mine = BM / p.split, slice = cl_rank >> 1;
        if (ok && warp >= 2) {
            const int q = warp & 3, r = q * 32 + lane;
            const uint32_t at = mapa_cluster(base + (uint32_t)((slice * mine + r % mine) * PITCH) * 4u, (uint32_t)(r / mine * 2 + cta_rank));
            const int cols = p.epi == EPI_SWIGLU ? BN : tc.width;
            for (int ch = 0; ch * 32 < cols; ++ch) {
                uint32_t v[32];
                tmem_ld32(tmem_base + ((uint32_t)(q * 32) << 16) + ch * 32, v);
                tmem_ld_wait();
#pragma unroll
                for (int e = 0; e < 32; e += 4) st_cluster16(at + ch * 128 + e * 4, v[e], v[e + 1], v[e + 2], v[e + 3]);
            }
        }
        tc_fence_before();
        __syncwarp();
        cluster_sync_all();
        if (ANYC) {
            // lanes along the columns: 64 contiguous bytes a store wherever a row's blocks start
            for (int c = lane; c < tc.width && *abort_flag == 0; c += 32) {
                int lo, hi, rlo, rhi;
                const int cb = ja_interval(p.c, 1, tc.n_g0 + c, &lo, &hi);
                for (int own = warp; own < mine && slice * mine + own < tc.rows; own += NUM_THREADS / 32) {
                    const float* src = reinterpret_cast<const float*>(smem) + own * PITCH + c;
                    float f = 0.f;
                    for (int k = 0; k < p.split; ++k) f += src[k * mine * PITCH];   // slices in ascending order
                    const int row = tc.row_g0 + slice * mine + own, rb = ja_interval(p.c, 0, row, &rlo, &rhi);
                    *reinterpret_cast<uint16_t*>(p.c.base + ja_block_at(p.c, rb, cb) + ((int64_t)(row - rlo) * (hi - lo) + (tc.n_g0 + c - lo)) * 2) =
                        (uint16_t)ja_pack16<F16>(f, 0.f);
                }
            }
        } else if (*abort_flag == 0) {
            const int ppr = (tc.width + 7) / 8;      // 8-column pieces of a row
            for (int i = threadIdx.x; i < mine * ppr; i += NUM_THREADS) {
                const int own = i / ppr, c = (i - own * ppr) * 8, r = slice * mine + own;
                if (r >= tc.rows) break;             // rows only grow
                const float* src = reinterpret_cast<const float*>(smem) + own * PITCH + c;
                auto sum8 = [&](const float* s, float (&f)[8]) {   // slices in ascending order
#pragma unroll
                    for (int e = 0; e < 8; ++e) f[e] = 0.f;
                    for (int k = 0; k < p.split; ++k, s += mine * PITCH) {
                        const float4 u = *reinterpret_cast<const float4*>(s), w = *reinterpret_cast<const float4*>(s + 4);
                        f[0] += u.x; f[1] += u.y; f[2] += u.z; f[3] += u.w; f[4] += w.x; f[5] += w.y; f[6] += w.z; f[7] += w.w;
                    }
                };
                float f[8];
                sum8(src, f);
                const int grow = tc.row_g0 + r, gcol = tc.n_g0 + c, kb = gcol / p.c_bn, cin = gcol - kb * p.c_bn, ib = grow / p.c_bm, iin = grow - ib * p.c_bm;
                const int64_t off = p.c_blk_off[(int64_t)ib * p.c_nbn + kb] + ((int64_t)iin * p.c_bn + cin) * 2;
                if (p.epi == EPI_SWIGLU) {
                    float g[8];
                    sum8(src + p.bn_tile, g);
#pragma unroll
                    for (int e = 0; e < 8; ++e) f[e] = f[e] / (1.f + __expf(-f[e])) * g[e];
                } else if (p.epi == EPI_ROPE) {
                    const float2* tab = p.rope_table + ((int64_t)(grow % p.rope_S) * p.rope_D + gcol % p.rope_D) / 2;
#pragma unroll
                    for (int e = 0; e < 8; e += 2) {
                        const float2 cs = tab[e / 2];
                        const float x0 = f[e], x1 = f[e + 1];
                        f[e] = x0 * cs.x - x1 * cs.y;
                        f[e + 1] = x0 * cs.y + x1 * cs.x;
                    }
                } else if (p.epi == EPI_ADD) {
                    const uint4 rv = *reinterpret_cast<const uint4*>(p.r_base + off);
                    const uint32_t* pr = reinterpret_cast<const uint32_t*>(&rv);
#pragma unroll
                    for (int e = 0; e < 4; ++e) {
                        const float2 rf = ja_unpack16<F16>(pr[e]);
                        f[2 * e] += rf.x;
                        f[2 * e + 1] += rf.y;
                    }
                }
                uint4 o;
                uint32_t* po = reinterpret_cast<uint32_t*>(&o);
#pragma unroll
                for (int e = 0; e < 4; ++e) po[e] = ja_pack16<F16>(f[2 * e], f[2 * e + 1]);
                *reinterpret_cast<uint4*>(p.c_base + off) = o;
            }
        }
    }
    // ---- teardown ---------------------------------------------------------------------------------------------
    tc_fence_before();
    __syncthreads();
    if (CG == 2) cluster_sync_all();   // nobody leaves while the peer may still signal its barriers or read its smem
    if (warp == 1) {
        tc_fence_after();
        if (CG == 1) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, 512;" ::"r"(tmem_base) : "memory");
        else asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, 512;" ::"r"(tmem_base) : "memory");
    }
}

}  // namespace

// ---- host: tensor maps -------------------------------------------------------------------------------------
TmaOperand ja_tma_operand(const ja_relation* r) {
    const int64_t blk_stride = r->nblocks > 1 ? r->blk_off[1] - r->blk_off[0] : (int64_t)r->bytes;
    return {(char*)r->base, r->dtype, r->bs[0], r->bs[1], r->nblk[0], r->nblk[1], r->bs[1] * 2, blk_stride, blk_stride * r->nblk[1]};
}

// A relation [R, C] with equal blocks br x bc is the rank-4 tensor (c in block, r in block, col-block, row-block).
ja_status_t ja_encode_blocked_2d(const TmaOperand& o, int box_inner, int box_rows, CUtensorMap* tm) {
    if (box_rows > 256) return ja_fail(JA_ERR_INVALID_ARG, "TMA box too tall");
    EncodeTiledFn enc = get_encode();
    if (!enc) return ja_fail(JA_ERR_CUDA, "cuTensorMapEncodeTiled is not available from the driver");
    cuuint64_t dims[4] = {(cuuint64_t)o.cols, (cuuint64_t)o.rows, (cuuint64_t)o.ncb, (cuuint64_t)o.nrb};
    cuuint64_t strides[3] = {(cuuint64_t)o.pitch, (cuuint64_t)o.col_stride, (cuuint64_t)o.row_stride};
    cuuint32_t box[4] = {(cuuint32_t)box_inner, (cuuint32_t)box_rows, 1, 1};
    cuuint32_t estr[4] = {1, 1, 1, 1};
    const CUtensorMapDataType cell = o.dtype == JA_F16 ? CU_TENSOR_MAP_DATA_TYPE_FLOAT16 : CU_TENSOR_MAP_DATA_TYPE_BFLOAT16;
    CUresult res = enc(tm, cell, 4, o.base, dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
                       CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    if (res != CUDA_SUCCESS) return ja_fail(JA_ERR_CUDA, "cuTensorMapEncodeTiled failed with code %d", (int)res);
    return JA_OK;
}

struct GemmTcPlan {
    CUtensorMap tmA, tmB, tmB2;
    GemmParams p;
    int cg;      // CTAs per tile: 1 or 2
    int tiles;   // of the whole launch; the last `tail` of them go to a launch of their own, each split along the contracted index
    int tail, split;
    bool any_c;
    TmaOperand a, b;
    double us;   // what the launches are expected to take
};

namespace {

template <bool F16, bool ANYC>
cudaError_t configure() {
    constexpr int S1 = ANYC ? Cfg<1>::SMEM_BYTES_ANYC : Cfg<1>::SMEM_BYTES, S2 = ANYC ? Cfg<2>::SMEM_BYTES_ANYC : Cfg<2>::SMEM_BYTES;
    cudaError_t e = cudaFuncSetAttribute(gemm_tc_kernel<1, F16, false, ANYC>, cudaFuncAttributeMaxDynamicSharedMemorySize, S1);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(gemm_tc_kernel<2, F16, false, ANYC>, cudaFuncAttributeMaxDynamicSharedMemorySize, S2);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(gemm_tc_kernel<2, F16, true, ANYC>, cudaFuncAttributeMaxDynamicSharedMemorySize, S2);
    return e;
}

// clusters of `split` CTA pairs of this instantiation (whose shared memory configure() has set) that the device holds at once
template <bool F16, bool ANYC>
int clusters_at_once(int split) {
    static std::atomic<int> known[64][2];
    int dev = 0;
    cudaGetDevice(&dev);
    std::atomic<int>& n = known[dev & 63][split == 2 ? 0 : 1];
    if (n.load() == 0) {
        cudaLaunchConfig_t cfg;
        memset(&cfg, 0, sizeof cfg);
        cfg.gridDim = dim3((unsigned)(2 * split), 1, 1);
        cfg.blockDim = dim3(NUM_THREADS, 1, 1);
        cfg.dynamicSmemBytes = ANYC ? Cfg<2>::SMEM_BYTES_ANYC : Cfg<2>::SMEM_BYTES;
        cudaLaunchAttribute attr[1];
        memset(attr, 0, sizeof attr);
        attr[0].id = cudaLaunchAttributeClusterDimension;
        attr[0].val.clusterDim.x = (unsigned)(2 * split);
        attr[0].val.clusterDim.y = attr[0].val.clusterDim.z = 1;
        cfg.attrs = attr;
        cfg.numAttrs = 1;
        int c = 0;
        if (cudaOccupancyMaxActiveClusters(&c, gemm_tc_kernel<2, F16, true, ANYC>, &cfg) != cudaSuccess) {
            cudaGetLastError();
            return 0;      // not kept: the next plan asks again
        }
        n.store(c > 0 ? c : -1);
    }
    return std::max(n.load(), 0);
}

// Whether the tiles of the last, partly empty round over the pairs of SMs are each split along the contracted index over a
// cluster of pairs. A 128-deep stage of a 256-row tile takes 0.96 us (1.3 PFLOP/s over the chip); the clusters' sums and their own
// start and end take 10 us ([1024, 4096] x [4096, 1024] 26 us with four slices a tile, 35 whole), and 2 more where a launch of whole tiles runs
// before them.
void choose_tail(GemmTcPlan* plan) {
    const GemmParams& p = plan->p;
    const int stages = (p.bk + Cfg<2>::BK - 1) / Cfg<2>::BK * p.nbk, pairs = ja_sm_count() / 2;
    const int whole = plan->tiles / pairs, rest = plan->tiles % pairs;
    plan->tail = 0;
    plan->split = 1;
    double best = (double)(whole + (rest > 0)) * stages * 0.96;
    // (tiles sorted by weight fill the last round with narrow ones: [2048, 4096] x [4096, 11008] in 1376-wide blocks 147 us, 150 with its last 14 split)
    // The slices' sums are stored in 16 bits: a join-only product of one copy into an f32 partial relation keeps whole tiles.
    if (p.n_copies == 1 && p.c_esize == 2 && rest > 0 && !p.heavy_first && ja_config().gemm_split != 0) {
        for (int s : {2, 4}) {
            const int at_once = plan->any_c ? (p.f16 ? clusters_at_once<true, true>(s) : clusters_at_once<false, true>(s))
                                            : (p.f16 ? clusters_at_once<true, false>(s) : clusters_at_once<false, false>(s));
            if (stages < 2 * s || at_once == 0) continue;
            const double t = (double)whole * stages * 0.96 + (double)((rest + at_once - 1) / at_once) * ((stages + s - 1) / s) * 0.96 + (whole ? 12.0 : 10.0);
            if (t < best) {
                best = t;
                plan->tail = rest;
                plan->split = s;
            }
        }
    }
    plan->us = best + 8.0;
}

}  // namespace

static ja_status_t encode_operands(GemmTcPlan* plan) {
    const int b_rows = plan->cg == 2 ? Cfg<2>::BK : Cfg<1>::BK;
    ja_status_t st = ja_encode_blocked_2d(plan->a, 64, plan->p.a_box_rows, &plan->tmA);
    if (st == JA_OK) st = ja_encode_blocked_2d(plan->b, 64, b_rows, &plan->tmB);
    return st;
}

// a, b: the operands' blocks, of one contracted extent. any_c: C has its own tiling of the same index ranges. Operands without a base get
// one by ja_gemm_tc_set_bases before the first launch.
static ja_status_t plan_gemm(const TmaOperand& a, const TmaOperand& b, const ja_relation* C, const GemmEpilogue* ep, bool any_c,
                             std::shared_ptr<GemmTcPlan>* out, bool* eligible) {
    const int epi = ep ? ep->epi : 0;
    const int bn_tile = epi == EPI_SWIGLU ? 128 : BN;
    const int64_t bm = a.rows, bk = a.cols, bn = b.cols;
    const bool odd_rows = bm < 128 && (128 % bm != 0 || bm % 8 != 0);   // one block per row tile: plain products alone
    if (odd_rows && (epi != EPI_NONE || C->esize != 2)) return JA_OK;
    std::shared_ptr<GemmTcPlan> plan(new GemmTcPlan());
    GemmParams& p = plan->p;
    p.c_base = (char*)C->base;
    p.c = ja_view(C);
    p.c_blk_off = p.c.blk_off;
    p.status = nullptr;
    p.bm = (int)bm; p.bk = (int)bk; p.bn = (int)bn;
    p.nbm = a.nrb; p.nbk = a.ncb; p.nbn = b.ncb;
    p.M = (int)C->extent[C->rank - 2]; p.N = (int)C->extent[C->rank - 1];
    p.c_bm = (int)C->bs[C->rank - 2]; p.c_bn = (int)C->bs[C->rank - 1]; p.c_nbn = C->nblk[C->rank - 1];
    p.a_box_rows = (int)std::min<int64_t>(bm, 128);
    p.a_boxes = bm < 128 && !odd_rows ? (int)(128 / bm) : 1;
    p.epi = epi;
    p.bn_tile = bn_tile;
    p.n_copies = (ep && ep->partials) ? p.nbk : 1;
    p.c_esize = C->esize;
    p.f16 = a.dtype == JA_F16;
    if (p.c_esize == 4 && !(ep && ep->partials)) return JA_OK;
    p.r_base = (epi == EPI_ADD) ? (const char*)ep->addend->base : nullptr;
    p.rope_table = (epi == EPI_ROPE) ? ep->rope_table : nullptr;
    p.rope_S = ep ? ep->rope_S : 1;
    p.rope_D = ep ? ep->rope_D : 2;
    if (bn % 64 == 0 && bn < bn_tile && p.nbn > 1) { p.tiles_per_nblk = 0; p.n_tiles = (p.N + bn_tile - 1) / bn_tile; }
    else { p.tiles_per_nblk = (int)((bn + bn_tile - 1) / bn_tile); p.n_tiles = p.tiles_per_nblk * p.nbn; }
    // Two-CTA form: 256-row tiles cut from global rows where blocks are whole 128-row halves or divide them, else pairs of row tiles
    // that each stay inside a block ([1260, 3840] x [3840, 10880] in one block: 145 us on single CTAs, 112 on pairs); when
    // tiles span column blocks, column tails whose halves still start on a 64-column box boundary.
    // narrow last tile in every column block (block width not a multiple of the tile width): schedule it after the full tiles
    const JaConfig& cfg = ja_config();
    p.heavy_first = (p.n_copies == 1 && p.tiles_per_nblk > 1 && bn % bn_tile != 0 && cfg.gemm_heavy_first != 0) ? 1 : 0;
    p.group_m = cfg.gemm_group_m >= 1 ? cfg.gemm_group_m : 8;
    const bool by_block = odd_rows || (bm > 128 && bm % 128 != 0);
    bool two = p.M > BM && bk >= Cfg<2>::BK;
    // join-only tiles of short blocks are mostly store, and pairs of row tiles hand out half as many: [8048, 576] x [576, 320] in blocks of
    // 4024 x 144 x 80 22.8 us single, 27.9 on pairs; 1.23 times as fast on pairs at 1000 contracted cells
    if (by_block && p.n_copies > 1 && bk < 512) two = false;
    if (p.tiles_per_nblk == 0 && (p.N % bn_tile) % (bn_tile / 2) != 0) two = false;
    if (cfg.gemm_cta_group == 1) two = false;
    plan->cg = two ? 2 : 1;
    if (!by_block) { p.tiles_per_mblk = 0; p.m_tiles = (p.M + BM * plan->cg - 1) / (BM * plan->cg); }
    else { p.tiles_per_mblk = (int)((bm + BM - 1) / BM); p.m_tiles = (p.tiles_per_mblk * p.nbm + plan->cg - 1) / plan->cg; }
    plan->a = a;
    plan->b = b;
    plan->any_c = any_c;
    ja_status_t st;
    if (a.base && b.base && (st = encode_operands(plan.get())) != JA_OK) return st;
    if (epi == EPI_SWIGLU && (st = ja_encode_blocked_2d(ja_tma_operand(ep->B2), 64, two ? Cfg<2>::BK : Cfg<1>::BK, &plan->tmB2)) != JA_OK) return st;
    if (epi != EPI_SWIGLU) plan->tmB2 = plan->tmB;
    cudaError_t e = any_c ? (p.f16 ? configure<true, true>() : configure<false, true>()) : (p.f16 ? configure<true, false>() : configure<false, false>());
    if (e != cudaSuccess) return ja_cuda_fail(e, "cudaFuncSetAttribute(gemm_tc_kernel)");
    plan->tiles = p.m_tiles * p.n_tiles * p.n_copies;
    plan->tail = 0;
    plan->split = 1;
    if (two) choose_tail(plan.get());
    else plan->us = (double)((plan->tiles + ja_sm_count() - 1) / ja_sm_count()) * ((p.bk + 63) / 64) * (p.n_copies > 1 ? 1 : p.nbk) * 0.70 + 8.0;
    *out = plan;
    *eligible = true;
    return JA_OK;
}

ja_status_t ja_gemm_tc_plan(const ja_relation* A, const ja_relation* B, const ja_relation* C, const GemmEpilogue* ep,
                            std::shared_ptr<GemmTcPlan>* out, bool* eligible) {
    *eligible = false;
    if (!A->equal_blocks || !B->equal_blocks || !C->equal_blocks) return JA_OK;
    if (A->dtype == JA_F32 || B->dtype != A->dtype || (C->esize == 2 && C->dtype != A->dtype)) return JA_OK;
    const int epi = ep ? ep->epi : 0;
    if (epi == EPI_SWIGLU && (B->bs[1] % 128 != 0 || !ep->B2 || !ep->B2->equal_blocks)) return JA_OK;
    if (epi == EPI_ROPE && (ep->rope_D % 32 != 0 || B->bs[1] % 32 != 0)) return JA_OK;
    const int64_t bk = A->bs[1], bn = B->bs[1];
    // TMA needs 16-byte row pitches; boxes are 64 elements wide; A boxes hold min(bm,128) rows
    if (bk % 8 || bn % 8 || bk < 64 || bn < 64) return JA_OK;
    if (A->extent[0] >= (1ll << 31) || B->extent[1] >= (1ll << 31)) return JA_OK;
    return plan_gemm(ja_tma_operand(A), ja_tma_operand(B), C, ep, false, out, eligible);
}

ja_status_t ja_gemm_tc_plan_staged(const TmaOperand& a, const TmaOperand& b, const ja_relation* C, std::shared_ptr<GemmTcPlan>* out, bool* eligible) {
    *eligible = false;
    if (a.cols < 64 || b.cols < 64) return JA_OK;
    // 32 columns at a time lie in one block of the output, in rows of whole 16 bytes: stored as ever
    const bool any_c = !(C->equal_blocks && C->bs[1] % 8 == 0 && (C->bs[1] == b.cols || C->bs[1] % 32 == 0));
    return plan_gemm(a, b, C, nullptr, any_c, out, eligible);
}

ja_status_t ja_gemm_tc_set_bases(GemmTcPlan* plan, char* a, char* b) {
    plan->a.base = a;
    plan->b.base = b;
    return encode_operands(plan);
}

// What the launches are expected to take: rounds of tiles over the CTA groups, 0.96 us per 128 contracted cells of a 256-row tile on
// a pair of SMs, 0.70 per 64 of a 128-row tile on one, and a start and an end.
double ja_gemm_tc_estimate_us(const GemmTcPlan& plan) { return plan.us; }

template <bool F16, bool ANYC>
static ja_status_t launch_gemm(const GemmTcPlan& plan, GemmParams& p, cudaStream_t st) {
    constexpr int S1 = ANYC ? Cfg<1>::SMEM_BYTES_ANYC : Cfg<1>::SMEM_BYTES, S2 = ANYC ? Cfg<2>::SMEM_BYTES_ANYC : Cfg<2>::SMEM_BYTES;
    const int sms = ja_sm_count();
    auto launch = [&](auto kernel, int grid, int smem, int cluster) -> ja_status_t {
        JA_CUDA(ja_launch_kernel_after(kernel, dim3((unsigned)grid, 1, 1), NUM_THREADS, smem, (unsigned)cluster, st, plan.tmA, plan.tmB, plan.tmB2, p));
        ja_count_launch();
        return JA_OK;
    };
    p.tile0 = 0;
    p.tile_end = plan.tiles - plan.tail;
    if (plan.cg == 1) return launch(gemm_tc_kernel<1, F16, false, ANYC>, std::min(sms, p.tile_end), S1, 1);
    ja_status_t s = JA_OK;
    if (p.tile_end > 0) s = launch(gemm_tc_kernel<2, F16, false, ANYC>, 2 * std::min(sms / 2, p.tile_end), S2, 2);
    if (s != JA_OK || plan.tail == 0) return s;
    p.tile0 = p.tile_end;
    p.tile_end = plan.tiles;
    p.split = plan.split;
    return launch(gemm_tc_kernel<2, F16, true, ANYC>, plan.tail * 2 * plan.split, S2, 2 * plan.split);
}

ja_status_t ja_launch_gemm_tc(const GemmTcPlan& plan, cudaStream_t st) {
    GemmParams p = plan.p;
    p.status = ja_device_status_word(st);
    if (!p.status) return ja_fail(JA_ERR_CUDA, "cannot resolve the device status word");
    p.wait_cap_us = (uint32_t)ja_config().wait_cap_us;
    if (plan.any_c) return p.f16 ? launch_gemm<true, true>(plan, p, st) : launch_gemm<false, true>(plan, p, st);
    return p.f16 ? launch_gemm<true, false>(plan, p, st) : launch_gemm<false, false>(plan, p, st);
}

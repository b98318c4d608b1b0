// Matmul join-agg "ij,jk->ik" (MUL / SUM) of FEW rows against a large second operand: a decoding step's tokens times a weight
// relation. The second operand is read once and everything else is small, so the kernel is a stream over it.
//
// The product is computed transposed: the tile's 128 rows of the tensor core are 128 COLUMNS of the output (B is MN-major in shared
// memory, as TMA brings it), its N columns are the tokens, so no row of the instruction is padding. One CTA = 128 output columns x
// one slice of the contracted index; the `split` slices of a tile form a thread-block cluster that sums its f32 partial tiles through
// distributed shared memory in rank order, with one rounding.
//   warp 0      TMA producer: per stage of 64 contracted cells two boxes of 64 columns x 64 cells of B and one box per row block of A
//   warp 1      tcgen05.mma issuer, M = 128, N = tokens rounded up to 16, K = 16
//   warps 2..5  the partial tile from tensor memory to its owners
// Every mbarrier wait is bounded; on expiry the CTA records JA_ERR_TIMEOUT, drains its copies and leaves through the normal exit.
//
// What bounds it: the stream of B out of HBM; on small products the trips of a CTA's stages, so up to eight are in flight.
// [32, 4096] x [4096, 11008] bf16 30.7 us (172 CTAs of the cp.async form) -> 24.6, 3.7 TB/s of weights; [64, 3001] x [3001, 320] on copies 58 -> 23.
#include <cuda.h>
#include <string.h>

#include <algorithm>

#include "ja_device.cuh"
#include "ja_launch.cuh"
#include "ja_ptx.cuh"

namespace {

using namespace ja_ptx;

constexpr int BM = 128, BK = 64, MAX_STAGES = 8, NUM_THREADS = 192;
constexpr int W_BYTES = BM * BK * 2, W_BOX = W_BYTES / 2;
constexpr int MAX_TOKENS = 128;

struct Params {
    int32_t* status;
    uint32_t wait_cap_us;
    int32_t bm, nbm, pad;      // rows per row block, row blocks, rows a block takes in the tile (a multiple of 8: swizzle atoms)
    int32_t n_mma;             // columns of the instruction: nbm * pad rounded up to 16
    int32_t tmem_cols;
    int32_t bk, nbk, per_blk;  // contracted cells per block, blocks, stages per block
    int32_t bn, N;
    int32_t tiles_per_nblk;    // 0: tiles are cut from the whole column index
    int32_t split, stages;
    int32_t f16;
    int32_t any_c;             // the output has its own tiling: cells stored one by one through its key table
    RelView c;
};

__global__ void __launch_bounds__(NUM_THREADS) stream_tc_kernel(const __grid_constant__ CUtensorMap tmA, const __grid_constant__ CUtensorMap tmB,
                                                                const __grid_constant__ Params p) {
    extern __shared__ uint8_t smem_raw[];
    const uint32_t raw = smem_u32(smem_raw);
    const uint32_t base = (raw + 1023u) & ~1023u;   // swizzle atoms need 1024-byte alignment
    uint8_t* smem = smem_raw + (base - raw);
    const uint32_t stage_bytes = W_BYTES + (uint32_t)p.n_mma * (BK * 2);
    const int stages = p.stages;
    uint64_t* bars = reinterpret_cast<uint64_t*>(smem + stages * stage_bytes);
    const uint32_t bar0 = smem_u32(bars);
    auto full_bar = [&](int s) { return bar0 + 8u * s; };
    auto empty_bar = [&](int s) { return bar0 + 8u * (MAX_STAGES + s); };
    const uint32_t done_bar = bar0 + 8u * (2 * MAX_STAGES);
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(bars + 2 * MAX_STAGES + 1);
    volatile int* ctl = reinterpret_cast<volatile int*>(tmem_slot + 1);
    const int warp = __shfl_sync(0xffffffffu, (int)threadIdx.x / 32, 0), lane = threadIdx.x % 32;

    if (threadIdx.x == 0) {
        for (int s = 0; s < stages; ++s) {
            mbar_init(full_bar(s), 1);
            mbar_init(empty_bar(s), 1);
        }
        mbar_init(done_bar, 1);
        wait_ctl_init(ctl, p.wait_cap_us);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 1) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)), "r"(p.tmem_cols) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = __shfl_sync(0xffffffffu, *tmem_slot, 0);

    // ---- this CTA's columns and its slice of the contracted index ----
    const int split = p.split, rank = (int)blockIdx.x % split, t = (int)blockIdx.x / split;
    int n0, width;             // first global column and columns of the tile; the tile lies in one column block unless tiles_per_nblk is 0
    if (p.tiles_per_nblk) {
        const int c0 = t % p.tiles_per_nblk * BM;
        n0 = t / p.tiles_per_nblk * p.bn + c0;
        width = min(BM, p.bn - c0);
    } else {
        n0 = t * BM;
        width = min(BM, p.N - n0);
    }
    const int chunks = p.nbk * p.per_blk;
    const int ch0 = (int)((int64_t)chunks * rank / split), ch1 = (int)((int64_t)chunks * (rank + 1) / split);

    int issued = 0;            // stages that this thread has started to fill
    if (warp == 0) {
        if (lane == 0) {
            const int boxes = width > 64 ? 2 : 1;
            const uint32_t tx = (uint32_t)(boxes * W_BOX + p.nbm * p.bm * (BK * 2));
            int nb[2], cin[2];
            for (int c = 0; c < boxes; ++c) {
                nb[c] = (n0 + 64 * c) / p.bn;
                cin[c] = (n0 + 64 * c) % p.bn;
            }
            int stage = 0, jb = ch0 / p.per_blk, kc = ch0 % p.per_blk;
            uint32_t phase = 0;
            for (int ch = ch0; ch < ch1; ++ch) {
                if (!mbar_wait(empty_bar(stage), phase ^ 1, ctl, p.status)) break;
                const uint32_t fb = full_bar(stage), w = base + stage * stage_bytes, x = w + W_BYTES;
                mbar_expect_tx(fb, tx);
                for (int c = 0; c < boxes; ++c) tma_load_4d<1>(w + c * W_BOX, &tmB, fb, cin[c], kc * BK, nb[c], jb);
                for (int b = 0; b < p.nbm; ++b) tma_load_4d<1>(x + b * p.pad * (BK * 2), &tmA, fb, kc * BK, 0, jb, b);
                ++issued;
                if (++kc == p.per_blk) { kc = 0; ++jb; }
                if (++stage == stages) { stage = 0; phase ^= 1; }
            }
        }
        __syncwarp();
    } else if (warp == 1) {
        const uint32_t leader = elect_one();
        const uint32_t fmt = p.f16 ? 0u : 1u;
        // D f32; A (the columns) MN-major, B (the tokens) K-major
        const uint32_t idesc = (1u << 4) | (fmt << 7) | (fmt << 10) | (1u << 15) | ((uint32_t)(p.n_mma >> 3) << 17) | ((uint32_t)(BM >> 4) << 24);
        int stage = 0;
        uint32_t phase = 0;
        bool ok = true;
        for (int ch = ch0; ch < ch1; ++ch) {
            if (!mbar_wait(full_bar(stage), phase, ctl, p.status)) { ok = false; break; }
            tc_fence_after();
            const uint32_t w = base + stage * stage_bytes, x = w + W_BYTES;
#pragma unroll
            for (int kk = 0; kk < BK / 16; ++kk)   // cells past a block's end are zero in both operands
                umma_bf16_w<1>(tmem, desc_sw128(w + kk * 2048, W_BOX), desc_sw128(x + kk * 32, 16), idesc, (ch > ch0 || kk > 0) ? 1u : 0u, leader);
            umma_commit_w<1>(empty_bar(stage), leader);
            if (++stage == stages) { stage = 0; phase ^= 1; }
        }
        if (ok) umma_commit_w<1>(done_bar, leader);
    }
    const bool ok = mbar_wait_warp(done_bar, 0, ctl, p.status);
    tc_fence_after();
    if (!ok && warp == 0 && lane == 0) {   // gave up: wait (bounded) for the copies in flight before the shared memory goes
        for (int s = 0; s < stages && s < issued; ++s) {
            const uint64_t t0 = global_ns();
            while (!mbar_try_wait(full_bar(s), (uint32_t)ja_last_fill_parity(issued, stages, s)) && global_ns() - t0 < 200000000ull) {}
        }
    }
    __syncwarp();
    // ---- every token's partial sums go to the CTA of the cluster that owns the token: [slice][own token][128 columns] f32 over the
    // stages, which every product has read ----
    const int slots = p.nbm * p.pad, mine = slots / split;
    if (split > 1) cluster_sync_all();
    else __syncthreads();
    if (ok && warp >= 2) {
        const int q = warp & 3, n = q * 32 + lane;
        for (int cc = 0; cc < slots; cc += 32) {
            uint32_t v[32];
            tmem_ld32(tmem + ((uint32_t)(q * 32) << 16) + cc, v);
            tmem_ld_wait();
            if (split == 1) {
                float* own = reinterpret_cast<float*>(smem);
#pragma unroll
                for (int e = 0; e < 32; ++e)
                    if (cc + e < slots) own[(cc + e) * BM + n] = __uint_as_float(v[e]);
            } else {
#pragma unroll
                for (int e = 0; e < 32; ++e)
                    if (cc + e < slots)
                        st_cluster4(mapa_cluster(base + (uint32_t)((rank * mine + (cc + e) % mine) * BM + n) * 4u, (uint32_t)((cc + e) / mine)), v[e]);
            }
        }
    }
    tc_fence_before();
    __syncthreads();
    if (split > 1) cluster_sync_all();     // the slices have arrived
    // ---- one rounding, 16-byte stores ----
    if (ctl[0] == 0) {
        if (p.any_c) {   // lanes along the columns, a cell a store
            for (int c = lane; c < width; c += 32) {
                int lo, hi, rlo, rhi;
                const int cb = ja_interval(p.c, 1, n0 + c, &lo, &hi);
                for (int own = warp; own < mine; own += NUM_THREADS / 32) {
                    const int slot = rank * mine + own, b = slot / p.pad, r = slot % p.pad;
                    if (r >= p.bm) continue;
                    float f = 0.f;
                    for (int s = 0; s < split; ++s) f += reinterpret_cast<const float*>(smem)[(s * mine + own) * BM + c];   // slices in ascending order
                    const int row = b * p.bm + r, rb = ja_interval(p.c, 0, row, &rlo, &rhi);
                    *reinterpret_cast<uint16_t*>(p.c.base + ja_block_at(p.c, rb, cb) + ((int64_t)(row - rlo) * (hi - lo) + (n0 + c - lo)) * 2) =
                        (uint16_t)(p.f16 ? ja_pack16<true>(f, 0.f) : ja_pack16<false>(f, 0.f));
                }
            }
        } else {
            for (int i = threadIdx.x; i < mine * (BM / 8); i += NUM_THREADS) {
                const int own = i / (BM / 8), n = i % (BM / 8) * 8, slot = rank * mine + own, b = slot / p.pad, r = slot % p.pad;
                if (r >= p.bm || n >= width) continue;
                const float* src = reinterpret_cast<const float*>(smem) + own * BM + n;
                float f[8] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
                for (int s = 0; s < split; ++s) {   // slices in ascending order
                    const float4 u = *reinterpret_cast<const float4*>(src + s * mine * BM), v = *reinterpret_cast<const float4*>(src + s * mine * BM + 4);
                    f[0] += u.x; f[1] += u.y; f[2] += u.z; f[3] += u.w; f[4] += v.x; f[5] += v.y; f[6] += v.z; f[7] += v.w;
                }
                const int g = n0 + n, cbn = (int)p.c.bs[1], kb = g / cbn, cin = g - kb * cbn;
                const int row = b * p.bm + r, cbm = (int)p.c.bs[0], ib = row / cbm, iin = row - ib * cbm;
                uint4 o;
                if (p.f16) o = make_uint4(ja_pack16<true>(f[0], f[1]), ja_pack16<true>(f[2], f[3]), ja_pack16<true>(f[4], f[5]), ja_pack16<true>(f[6], f[7]));
                else o = make_uint4(ja_pack16<false>(f[0], f[1]), ja_pack16<false>(f[2], f[3]), ja_pack16<false>(f[4], f[5]), ja_pack16<false>(f[6], f[7]));
                *reinterpret_cast<uint4*>(p.c.base + ja_block_at(p.c, ib, kb) + ((int64_t)iin * cbn + cin) * 2) = o;
            }
        }
    }
    __syncthreads();
    if (warp == 1) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(p.tmem_cols) : "memory");
}

}  // namespace

struct StreamTcPlan {
    CUtensorMap tmA, tmB;
    Params p;
    int grid, smem;
    TmaOperand a, b;
};

static ja_status_t encode_operands(StreamTcPlan* plan) {
    ja_status_t st = ja_encode_blocked_2d(plan->a, BK, plan->p.bm, &plan->tmA);
    if (st == JA_OK) st = ja_encode_blocked_2d(plan->b, 64, BK, &plan->tmB);
    return st;
}

static ja_status_t plan_stream(const TmaOperand& a, const TmaOperand& b, const ja_relation* C, bool any_c, std::shared_ptr<StreamTcPlan>* out, double* est_us) {
    const int64_t bm = a.rows, bk = a.cols, bn = b.cols, N = C->extent[1], K = bk * a.ncb;
    // TMA boxes are 64 cells wide, and narrower blocks would leave most of a box empty
    if (bk < 64 || bn < 64 || K >= (1ll << 31) || N >= (1ll << 31)) return JA_OK;
    const int64_t pad = (bm + 7) / 8 * 8, slots = a.nrb * pad;
    if (slots > MAX_TOKENS) return JA_OK;
    std::shared_ptr<StreamTcPlan> plan(new StreamTcPlan());
    Params& p = plan->p;
    memset(&p, 0, sizeof p);
    p.c = ja_view(C);
    p.any_c = any_c;
    p.bm = (int)bm; p.nbm = a.nrb; p.pad = (int)pad;
    p.n_mma = (int)((slots + 15) / 16 * 16);
    p.tmem_cols = 32;
    while (p.tmem_cols < p.n_mma) p.tmem_cols *= 2;
    p.bk = (int)bk; p.nbk = a.ncb; p.per_blk = (int)((bk + BK - 1) / BK);
    p.bn = (int)bn; p.N = (int)N;
    p.tiles_per_nblk = bn % 64 == 0 ? 0 : (int)((bn + BM - 1) / BM);
    p.f16 = a.dtype == JA_F16;
    const int64_t tiles = p.tiles_per_nblk ? (int64_t)p.tiles_per_nblk * b.ncb : (N + BM - 1) / BM, chunks = (int64_t)p.nbk * p.per_blk;
    // as many slices as leave the CTAs resident at once at three stages each ([100, 3001] x [3001, 5001] in 320 CTAs, 296 of which fit: two
    // rounds), and then as many stages as the CTAs of an SM have room for
    const int sms = ja_sm_count(), stage_bytes = W_BYTES + p.n_mma * BK * 2;
    auto smem_of = [&](int stages) { return stages * stage_bytes + 1024 + 256; };
    const int room = 227 * 1024, fit = std::max(1, std::min(3, room / (smem_of(3) + 1024)));
    int split = 1;
    while (split < 8 && tiles * split * 2 <= (int64_t)sms * fit && chunks >= 8 * split) split *= 2;
    p.split = split;
    if (tiles * split >= (1ll << 31)) return JA_OK;
    plan->grid = (int)(tiles * split);
    const int per_sm = std::min(fit, (plan->grid + sms - 1) / sms);
    p.stages = 3;
    while (p.stages < MAX_STAGES && p.stages < (chunks + split - 1) / split && per_sm * (smem_of(p.stages + 1) + 1024) <= room) ++p.stages;
    plan->smem = smem_of(p.stages);
    plan->a = a;
    plan->b = b;
    ja_status_t st;
    if (a.base && b.base && (st = encode_operands(plan.get())) != JA_OK) return st;
    JA_CUDA(cudaFuncSetAttribute(stream_tc_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, room));
    // The stream at 6 TB/s and the tokens' stages from L2 at 9, or, where that leaves a CTA's stages in a row, 0.25 us each; a start, and an end in which every
    // token's sums cross the cluster.
    const double stream = (double)(K * N * 2) / 6.0e6 + (double)(tiles * chunks) * p.n_mma * BK * 2 / 9.0e6;
    const double rounds = (double)((plan->grid + sms * per_sm - 1) / (sms * per_sm)) * (double)((chunks + split - 1) / split) * 0.25;
    *est_us = std::max(stream, rounds) + 7.0 + 0.05 * (double)slots;
    *out = plan;
    return JA_OK;
}

ja_status_t ja_stream_tc_plan(const ja_relation* A, const ja_relation* B, const ja_relation* C, std::shared_ptr<StreamTcPlan>* out, double* est_us) {
    out->reset();
    if (!A->equal_blocks || !B->equal_blocks || !C->equal_blocks) return JA_OK;
    if (A->dtype == JA_F32 || B->dtype != A->dtype || C->dtype != A->dtype) return JA_OK;
    if (A->bs[1] % 8 || B->bs[1] % 8) return JA_OK;   // TMA needs 16-byte row pitches
    return plan_stream(ja_tma_operand(A), ja_tma_operand(B), C, false, out, est_us);
}

ja_status_t ja_stream_tc_plan_staged(const TmaOperand& a, const TmaOperand& b, const ja_relation* C, std::shared_ptr<StreamTcPlan>* out, double* est_us) {
    out->reset();
    return plan_stream(a, b, C, !(C->equal_blocks && C->bs[1] % 8 == 0), out, est_us);
}

ja_status_t ja_stream_tc_set_bases(StreamTcPlan* plan, char* a, char* b) {
    plan->a.base = a;
    plan->b.base = b;
    return encode_operands(plan);
}

ja_status_t ja_launch_stream_tc(const StreamTcPlan& plan, cudaStream_t st) {
    Params p = plan.p;
    p.status = ja_device_status_word(st);
    if (!p.status) return ja_fail(JA_ERR_CUDA, "cannot resolve the device status word");
    p.wait_cap_us = (uint32_t)ja_config().wait_cap_us;
    const dim3 grid((unsigned)plan.grid, 1, 1);
    JA_CUDA(ja_launch_kernel_after(stream_tc_kernel, grid, NUM_THREADS, plan.smem, (unsigned)p.split, st, plan.tmA, plan.tmB, p));
    ja_count_launch();
    return JA_OK;
}

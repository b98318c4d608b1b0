// Two-index products "ij,jk->ik" of 16-bit relations that TMA cannot address as they lie -- block rows that are no whole 16 bytes, blocks of
// different shapes -- through a copy that it can: the operands that need it are rewritten as plain rows of a pitch of whole 16 bytes, and
// the TMA-fed kernels (k_gemm_tc.cu, k_stream_tc.cu) run on the copies and store through the output's own key table.
//
// The copy moves 2 bytes per byte of the operand; fed piece by piece (k_contract_tc.cu) the tensor cores wait for the loaders' instruction
// streams instead. The copies live in scratch that the plan takes from the library's pool at its first call and keeps: at most 1 GiB a plan
// and 4 GiB altogether, given back when the spec or the relations go and with them the last graph that recorded a call. Two calls of one
// plan that were not ordered behind one another would already race on its output.
//
// The copy's launch, like the product's, neither starts inside the one before it nor lets one in: the queue that stopped (ja_launch.cuh).
#include <cuda.h>
#include <string.h>

#include <algorithm>
#include <atomic>
#include <map>
#include <mutex>
#include <vector>

#include "ja_device.cuh"
#include "ja_launch.cuh"
#include "ja_ptx.cuh"

namespace {

// A thread writes one 16-byte word of `rows_per_cta` / 8 rows. The word's cells lie in one interval of the column index (two aligned words of
// the row, shifted together), in two around a split point (two such pairs, merged), or, where intervals are shorter than a word, in
// more (cell by cell). Words that hold no wanted cell are not read; a payload is 128-byte aligned and padded, so a word that holds one
// never leaves it. Neighbouring threads read neighbouring words, several rows in flight per thread. CUT: there are split points (and
// twice the registers a row, so half the rows). What bounds that form is its instructions and their latency, two loads, a shift and a
// merge a word: 45 MB in 172-cell blocks 27 us, DRAM 23 % busy, issue slots 41 %.
constexpr int WORDS = 32, THREADS = 256, STEP = THREADS / WORDS;
// one operand's copy; both operands' are one launch
struct Copy {
    RelView x;
    char* dst;
    int64_t pitch;
    int32_t words, rows_per_cta, across, ctas;   // 16-byte words of a row; CTAs across them, and altogether (0: the operand is not copied)
};
struct Copies {
    Copy c[2];
};
template <bool CUT>
__global__ void __launch_bounds__(THREADS, CUT ? 3 : 4) stage_kernel(const __grid_constant__ Copies copies) {
    const Copy& o = copies.c[(int)blockIdx.x < copies.c[0].ctas ? 0 : 1];
    const int cta = (int)blockIdx.x - ((int)blockIdx.x < copies.c[0].ctas ? 0 : copies.c[0].ctas), words = o.words, rows_per_cta = o.rows_per_cta;
    const RelView& x = o.x;
    char* const dst = o.dst;
    const int64_t pitch = o.pitch;
    const int bx = cta % o.across, by = cta / o.across;
    constexpr int UNROLL = CUT ? 2 : 4;
    const int w = bx * WORDS + threadIdx.x % WORDS;
    if (w >= words) return;
    const int cols = (int)x.extent[1], c0 = w * 8, n = min(8, cols - c0);
    const int r0 = by * rows_per_cta + threadIdx.x / WORDS, r_end = min((int)x.extent[0], (by + 1) * rows_per_cta);
    if (r0 >= r_end) return;
    int lo, hi, lo2 = 0, hi2 = 0;
    const int cb = ja_interval(x, 1, c0, &lo, &hi);
    const int n1 = min(n, hi - c0);
    if (CUT && n1 < n) ja_interval(x, 1, hi, &lo2, &hi2);
    const int n2 = CUT ? min(n - n1, hi2 - lo2) : 0;
    const bool slow = CUT && n1 + n2 < n;
    uint32_t first[4];                         // the cells that the first interval holds
#pragma unroll
    for (int k = 0; k < 4; ++k) first[k] = n1 >= 2 * k + 2 ? 0xffffffffu : n1 == 2 * k + 1 ? 0xffffu : 0u;
    int rb = 0, rlo = 0, rhi = 0;
    const char *blk = nullptr, *blk2 = nullptr;
    for (int r1 = r0; r1 < r_end; r1 += STEP * UNROLL) {
        uint4 a[UNROLL], b[UNROLL], c[UNROLL], d[UNROLL];
        int sh[UNROLL], sh2[UNROLL];
#pragma unroll
        for (int u = 0; u < UNROLL; ++u) {
            const int r = r1 + u * STEP;
            sh[u] = sh2[u] = 0;
            if (r >= r_end) continue;
            if (r >= rhi) {
                rb = ja_interval(x, 0, r, &rlo, &rhi);
                blk = x.base + ja_block_at(x, rb, cb);
                if (CUT && n2) blk2 = x.base + ja_block_at(x, rb, cb + 1);
            }
            if (CUT && slow) {
                uint32_t v[4] = {0u, 0u, 0u, 0u};
                int bb = cb, l = lo, h = hi;
                const char* at = blk + ((int64_t)(r - rlo) * (h - l) + (c0 - l)) * 2;
                for (int e = 0; e < n; ++e) {
                    if (c0 + e == h) {
                        bb = ja_interval(x, 1, c0 + e, &l, &h);
                        at = x.base + ja_block_at(x, rb, bb) + (int64_t)(r - rlo) * (h - l) * 2;
                    }
                    const uint32_t cell = *reinterpret_cast<const uint16_t*>(at);
                    at += 2;
#pragma unroll
                    for (int k = 0; k < 4; ++k)
                        if (k == e >> 1) v[k] |= cell << (16 * (e & 1));
                }
                a[u] = make_uint4(v[0], v[1], v[2], v[3]);
                continue;
            }
            const char* src = blk + ((int64_t)(r - rlo) * (hi - lo) + (c0 - lo)) * 2;
            sh[u] = (int)(reinterpret_cast<uintptr_t>(src) & 15);
            a[u] = *reinterpret_cast<const uint4*>(src - sh[u]);
            b[u] = sh[u] + 2 * n1 > 16 ? *reinterpret_cast<const uint4*>(src - sh[u] + 16) : make_uint4(0u, 0u, 0u, 0u);
            if (CUT && n2) {                   // the 16 bytes that end up in the word start n1 cells before the second interval's row
                src = blk2 + ((int64_t)(r - rlo) * (hi2 - lo2) - n1) * 2;
                sh2[u] = (int)(reinterpret_cast<uintptr_t>(src) & 15);
                c[u] = sh2[u] + 2 * n1 < 16 ? *reinterpret_cast<const uint4*>(src - sh2[u]) : make_uint4(0u, 0u, 0u, 0u);
                d[u] = sh2[u] + 2 * (n1 + n2) > 16 ? *reinterpret_cast<const uint4*>(src - sh2[u] + 16) : make_uint4(0u, 0u, 0u, 0u);
            }
        }
#pragma unroll
        for (int u = 0; u < UNROLL; ++u) {
            const int r = r1 + u * STEP;
            if (r >= r_end) continue;
            uint4 v = sh[u] ? ja_shift16(a[u], b[u], sh[u]) : a[u];
            if (CUT && n2 && !slow) {
                const uint4 y = sh2[u] ? ja_shift16(c[u], d[u], sh2[u]) : c[u];
                v.x = (v.x & first[0]) | (y.x & ~first[0]);
                v.y = (v.y & first[1]) | (y.y & ~first[1]);
                v.z = (v.z & first[2]) | (y.z & ~first[2]);
                v.w = (v.w & first[3]) | (y.w & ~first[3]);
            }
            *reinterpret_cast<uint4*>(dst + r * pitch + (int64_t)w * 16) = v;
        }
    }
}

size_t plan_copy(const ja_relation* r, Copy* c) {
    c->x = ja_view(r);
    c->pitch = (r->extent[1] * 2 + 15) / 16 * 16;
    c->words = (int)(c->pitch / 16);
    c->across = (c->words + WORDS - 1) / WORDS;
    // rows for a CTA: many, so that finding the first block is little of its work, but six CTAs for every SM
    int rows = 256;
    while (rows > 32 && (int64_t)c->across * ((r->extent[0] + rows - 1) / rows) < 6 * ja_sm_count()) rows /= 2;
    c->rows_per_cta = rows;
    c->ctas = (int)(c->across * ((r->extent[0] + rows - 1) / rows));
    return (size_t)((r->extent[0] * c->pitch + 255) / 256 * 256);
}

}  // namespace

namespace {

constexpr int64_t MAX_PLAN_BYTES = (int64_t)1 << 30, MAX_ALL_BYTES = (int64_t)4 << 30;
std::atomic<int64_t> g_staged_bytes{0};   // scratch of all plans, until it is freed

// Calls that a capture of any thread may forbid, made while this lives: on streams of the library's own and on memory that no capture knows
struct OutsideCaptures {
    cudaStreamCaptureMode mode = cudaStreamCaptureModeRelaxed;
    OutsideCaptures() { cudaThreadExchangeStreamCaptureMode(&mode); }
    ~OutsideCaptures() { cudaThreadExchangeStreamCaptureMode(&mode); }
};

// Scratch belongs to its plan and to every graph that recorded a call on it (a user object of the graph). Whoever lets go of it last retires
// it without a CUDA call, which the driver does not allow there, and a later call of the library frees it, once the calls outside
// graphs have ended: an event for each stream that has seen one. A graph lets go when its own launches have ended. So no destructor
// waits for the device, nor meets a capture that forbids it.
struct Scratch {
    char* at;
    int64_t bytes;
    cudaStream_t own;                                  // the library's stream that it was taken on
    std::map<unsigned long long, cudaEvent_t> used;    // by stream id
};
struct Retired {
    std::mutex mu;
    std::vector<Scratch*> list;
    std::atomic<int> n{0};
};
Retired& retired() {
    static Retired* r = new Retired;   // never destroyed: a graph's last reference may go at exit
    return *r;
}
void retire(Scratch* s) {
    Retired& r = retired();
    std::lock_guard<std::mutex> lk(r.mu);
    r.list.push_back(s);
    ++r.n;
}
void CUDART_CB let_go(void* owner) { delete static_cast<std::shared_ptr<Scratch>*>(owner); }

// wait: for calls that have not ended
void free_retired(bool wait) {
    Retired& r = retired();
    if (r.n.load() == 0) return;
    std::vector<Scratch*> mine;
    {
        std::lock_guard<std::mutex> lk(r.mu);
        mine.swap(r.list);
        r.n = 0;
    }
    const OutsideCaptures relaxed;
    for (Scratch* s : mine) {
        bool ended = true;
        for (auto& u : s->used) ended = ended && (wait ? cudaEventSynchronize(u.second) : cudaEventQuery(u.second)) == cudaSuccess;
        if (!ended) {
            cudaGetLastError();
            retire(s);
            continue;
        }
        for (auto& u : s->used) cudaEventDestroy(u.second);
        cudaFreeAsync(s->at, s->own);
        cudaStreamSynchronize(s->own);
        g_staged_bytes -= s->bytes;
        delete s;
    }
}

// Memory of the library's pool that is good for every stream, and for captures, when this returns: it is taken on a stream of the
// library's own, where nothing else runs, so the wait for it is no wait for any caller's work. Empty where there is none.
std::shared_ptr<Scratch> take_scratch(int64_t bytes) {
    static std::mutex mu;
    static std::map<int, cudaStream_t> own;
    const OutsideCaptures relaxed;
    int dev = 0;
    cudaMemPool_t pool;
    if (cudaGetDevice(&dev) != cudaSuccess || ja_library_pool(&pool) != JA_OK) return nullptr;
    free_retired(false);
    if (g_staged_bytes.fetch_add(bytes) + bytes > MAX_ALL_BYTES) free_retired(true);   // (which form a call takes must not hang on how far the GPU is)
    std::lock_guard<std::mutex> lk(mu);
    char* p = nullptr;
    cudaStream_t& st = own[dev];
    if (!st && cudaStreamCreateWithFlags(&st, cudaStreamNonBlocking) != cudaSuccess) st = nullptr;
    if (g_staged_bytes.load() <= MAX_ALL_BYTES && st && cudaMallocFromPoolAsync((void**)&p, (size_t)bytes, pool, st) == cudaSuccess &&
        cudaStreamSynchronize(st) == cudaSuccess)
        return std::shared_ptr<Scratch>(new Scratch{p, bytes, st, {}}, retire);
    cudaGetLastError();
    g_staged_bytes -= bytes;
    return nullptr;
}

// The event that calls on this stream are recorded with; those of streams that have drained make room. nullptr where there is none.
cudaEvent_t event_of(Scratch* s, cudaStream_t st) {
    unsigned long long id = 0;
    if (cudaStreamGetId(st, &id) != cudaSuccess) return nullptr;
    auto it = s->used.find(id);
    if (it != s->used.end()) return it->second;
    const OutsideCaptures relaxed;
    for (auto u = s->used.begin(); u != s->used.end();) {
        if (cudaEventQuery(u->second) != cudaSuccess) {
            ++u;
            continue;
        }
        cudaEventDestroy(u->second);
        u = s->used.erase(u);
    }
    cudaGetLastError();
    cudaEvent_t e = nullptr;
    if (cudaEventCreateWithFlags(&e, cudaEventDisableTiming) != cudaSuccess) return nullptr;
    return s->used[id] = e;
}

}  // namespace

void ja_staged_free_retired() { free_retired(false); }

extern "C" int64_t ja_debug_scratch_bytes(void) {
    free_retired(false);
    return g_staged_bytes.load();
}

struct StagedPlan {
    Copies copies;           // of A and of B
    size_t a_bytes = 0, b_bytes = 0;
    char *a_base, *b_base;   // of the operands that are used as they lie
    std::shared_ptr<GemmTcPlan> gemm;
    std::shared_ptr<StreamTcPlan> stream;
    std::shared_ptr<Scratch> scratch;
    unsigned long long recorded = 0;   // the capture whose graph has been made an owner
};

ja_status_t ja_staged_plan(const ja_relation* A, const ja_relation* B, const ja_relation* C, std::shared_ptr<StagedPlan>* out, double* est_us) {
    out->reset();
    if (A->dtype == JA_F32 || B->dtype != A->dtype || C->dtype != A->dtype) return JA_OK;
    const int64_t M = A->extent[0], K = A->extent[1], N = B->extent[1];
    if (K < 64 || N < 64 || M >= (1ll << 21) || K >= (1ll << 30) || N >= (1ll << 30)) return JA_OK;   // (rows of the copy's grid: M / 32 CTAs)
    std::shared_ptr<StagedPlan> plan(new StagedPlan());
    memset(&plan->copies, 0, sizeof plan->copies);
    // An operand that TMA can address stays where it is, and the other one's copy is cut along the contracted index as it is. Blocks of B
    // that follow one another without a gap are one.
    TmaOperand a, b;
    bool a_fits = A->equal_blocks && A->bs[1] % 8 == 0 && A->bs[1] >= 64, b_fits = B->equal_blocks && B->bs[1] % 8 == 0 && B->bs[1] >= 64;
    if (a_fits) a = ja_tma_operand(A);
    if (b_fits) {
        b = ja_tma_operand(B);
        if (!a_fits && b.ncb == 1 && b.row_stride == b.rows * b.pitch) {
            b.rows = K;
            b.nrb = 1;
        }
        // a copied A can only be cut in whole 16-byte steps
        b_fits = a_fits || b.nrb == 1 || (b.rows % 8 == 0 && b.rows >= 64);
    }
    if (a_fits && b_fits) return JA_OK;
    if (!a_fits) {
        plan->a_bytes = plan_copy(A, &plan->copies.c[0]);
        const int64_t pitch = plan->copies.c[0].pitch;
        a = {nullptr, A->dtype, M, K, 1, 1, pitch, pitch, M * pitch};
        if (b_fits && b.nrb > 1) {
            a.cols = b.rows;
            a.ncb = b.nrb;
            a.col_stride = a.cols * 2;
        }
    }
    if (!b_fits) {
        plan->b_bytes = plan_copy(B, &plan->copies.c[1]);
        const int64_t pitch = plan->copies.c[1].pitch;
        b = {nullptr, B->dtype, K, N, 1, 1, pitch, pitch, K * pitch};
        if (a_fits && a.ncb > 1) {
            b.rows = a.cols;
            b.nrb = a.ncb;
            b.row_stride = b.rows * pitch;
        }
    }
    if ((int64_t)(plan->a_bytes + plan->b_bytes) > MAX_PLAN_BYTES) return JA_OK;
    plan->a_base = a.base;
    plan->b_base = b.base;
    a.base = b.base = nullptr;
    bool ok = false;
    double us = 0, stream_us = 0;
    ja_status_t st = ja_stream_tc_plan_staged(a, b, C, &plan->stream, &stream_us);
    if (st != JA_OK) return st;
    if ((st = ja_gemm_tc_plan_staged(a, b, C, &plan->gemm, &ok)) != JA_OK) return st;
    if (!ok) plan->gemm.reset();
    if (plan->gemm) us = ja_gemm_tc_estimate_us(*plan->gemm);
    if (plan->stream && (!plan->gemm || stream_us < us)) {
        plan->gemm.reset();
        us = stream_us;
    } else {
        plan->stream.reset();
    }
    if (!plan->gemm && !plan->stream) return JA_OK;
    // the copies: read and written once; their launch and the scratch
    *est_us = us + (double)(2 * (plan->a_bytes + plan->b_bytes)) / 4.0e6 + 6.0;
    *out = plan;
    return JA_OK;
}

ja_status_t ja_launch_staged(StagedPlan* plan, cudaStream_t st, bool* launched) {
    *launched = false;
    ja_status_t s;
    cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
    unsigned long long cap_id = 0;
    cudaGraph_t graph = nullptr;
    if (cudaStreamGetCaptureInfo(st, &cap, &cap_id, &graph) != cudaSuccess) {
        cudaGetLastError();   // the question's own error; the launch will tell
        return JA_OK;
    }
    if (!plan->scratch) {
        // a call that a capture records takes no memory: the caller's other form runs there until a call outside has been made
        if (cap != cudaStreamCaptureStatusNone) return JA_OK;
        const std::shared_ptr<Scratch> taken = take_scratch((int64_t)(plan->a_bytes + plan->b_bytes));
        if (!taken) return JA_OK;   // no memory for it: the other form
        char *a = plan->a_bytes ? taken->at : plan->a_base, *b = plan->b_bytes ? taken->at + plan->a_bytes : plan->b_base;
        if ((s = plan->gemm ? ja_gemm_tc_set_bases(plan->gemm.get(), a, b) : ja_stream_tc_set_bases(plan->stream.get(), a, b)) != JA_OK) return s;
        // kept only now: a plan that has scratch has maps of it
        plan->scratch = taken;
        plan->copies.c[0].dst = a;
        plan->copies.c[1].dst = b;
    }
    cudaEvent_t event = nullptr;
    if (cap == cudaStreamCaptureStatusNone) {
        if (!(event = event_of(plan->scratch.get(), st))) {
            cudaGetLastError();
            return JA_OK;
        }
    } else if (plan->recorded != cap_id) {
        auto* owner = new std::shared_ptr<Scratch>(plan->scratch);
        cudaUserObject_t held;
        if (cudaUserObjectCreate(&held, owner, let_go, 1, cudaUserObjectNoDestructorSync) != cudaSuccess) {
            delete owner;
            cudaGetLastError();
            return JA_OK;
        }
        if (cudaGraphRetainUserObject(graph, held, 1, cudaGraphUserObjectMove) != cudaSuccess) {
            cudaUserObjectRelease(held, 1);
            cudaGetLastError();
            return JA_OK;
        }
        plan->recorded = cap_id;
    }
    const Copies& c = plan->copies;
    const bool cut = (plan->a_bytes && c.c[0].x.nblk[1] > 1) || (plan->b_bytes && c.c[1].x.nblk[1] > 1);
    JA_CUDA(ja_launch_kernel_after(cut ? stage_kernel<true> : stage_kernel<false>, dim3((unsigned)(c.c[0].ctas + c.c[1].ctas)), THREADS, 0, 1, st, c));
    ja_count_launch();
    s = plan->gemm ? ja_launch_gemm_tc(*plan->gemm, st) : ja_launch_stream_tc(*plan->stream, st);
    if (event) JA_CUDA(cudaEventRecord(event, st));
    *launched = s == JA_OK;
    return s;
}

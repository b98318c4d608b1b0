// Contraction of two f32 relations under ANY tiling and any order of their indices, on the FMA pipe with f32 accumulation: the
// products of k_contract_tc.cu ("ij,jk->ik", "bij,bkj->bik", "ji,jk->ik", ...) for cells that tensor cores cannot multiply
// exactly (tf32 keeps 10 bits). The output is f32 or a 16-bit type.
//
// One CTA = one T x T tile (T = 32, 64 or 128; 256 threads, T / 16 outputs a side per thread) x one slice of the contracted
// index; the slices of a tile form a thread-block cluster that sums its partial tiles in rank order through distributed shared
// memory. Operands reach shared memory as [contracted cell][row] lines, 32 contracted cells per stage, by cp.async: 16 bytes at
// a time where the row index is the contiguous one and its split points are multiples of four, 4 bytes otherwise (with lanes
// along whichever index is contiguous, so both orders read whole sectors and a transposed operand costs nothing extra). Tiles
// are cut from the global index ranges, whatever the blocks are. The inner loop multiplies pairs of columns (fma.rn.f32x2).
//
// What bounds it: large tiles the FMA pipe's issue and the shared-memory reads (2048^3 in 512-cell blocks 41 TFLOP/s, 32 on the
// block-bound kernel of k_matmul_simt.cu; 35 with scalar FMAs); small problems the start of a CTA and one trip to memory
// (256^3 8.5 us of GPU time either way). Batched and transposed products ran cell by cell before: "bij,bkj->bik" of 5 x 71 x
// 268 x 335 cells 965 us.
#include <string.h>

#include <algorithm>
#include <atomic>

#include "ja_device.cuh"
#include "ja_launch.cuh"
#include "ja_ptx.cuh"
#include "ja_walk.cuh"

namespace {

using namespace ja_ptx;
using namespace ja_walk;

constexpr int TK = 32, NT = 256;
template <int T> struct Cfg {
    static constexpr int PITCH = T + 4, OPERAND = TK * PITCH * 4, STAGE = 2 * OPERAND, STAGES = T == 128 ? 3 : 4;
    static constexpr int TILE = T * PITCH * 4;   // the staged tile of a cluster reuses the stages
    static constexpr int SMEM = STAGES * STAGE;
    static_assert(TILE <= SMEM, "the staged tile reuses the stages");
};

struct Params {
    Rel A, B, C;
    int32_t M, N, K, batch[MAX_BATCH];
    int32_t tiles_m, tiles_n, split;
    int32_t let_next;                   // the next launch may start as this one does (set at launch)
    int32_t c_dtype;
};

__device__ __forceinline__ void cp_async4(uint32_t dst, const char* src, bool in, bool live) {
    asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %3, 0;\n\t@p cp.async.ca.shared.global [%0], [%1], 4, %2;\n\t}" ::"r"(dst), "l"(src), "r"(in ? 4 : 0), "r"((int)live)
                 : "memory");
}
__device__ __forceinline__ void cp_async16(uint32_t dst, const char* src, bool in, bool live) {
    asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %3, 0;\n\t@p cp.async.cg.shared.global [%0], [%1], 16, %2;\n\t}" ::"r"(dst), "l"(src), "r"(in ? 16 : 0), "r"((int)live)
                 : "memory");
}

// One operand's share of the stages: fixed row positions, a cursor along the contracted index.
//   KC: lane = contracted cell of the stage, rows warp + 8 n.   else: rows are pieces of W cells (W = 4: 16 bytes), lines
//   tid / (T / W) + n * LP of the stage, whose positions the lanes work out one each and pass around by shuffles.
template <int T, bool KC, int W, bool EQ> struct Walk {
    static constexpr int PPL = T / W, LP = KC ? 8 : NT / PPL, NP = KC ? T / 8 : TK / LP, NF = KC ? NP : 1;
    const char* base;
    const Dim* dk;
    const int64_t* blk_off;
    int64_t foff[EQ ? NF : 1];
    int fflat[EQ ? 1 : NF], fa[EQ ? 1 : NF], fb;
    const char* start[EQ ? 1 : NF];
    int have;
    uint32_t live;
    int K, line, piece;
    Cursor cur;
    BatchAt ba;

    __device__ __forceinline__ void init(const Rel& o, const BatchAt& at, int tid, int r0, int k0) {
        base = o.base;
        dk = &o.k;
        blk_off = o.blk_off;
        ba = at;
        K = o.k.extent;
        have = -1;
        live = 0;
        fb = 0;
        line = KC ? tid >> 5 : tid / PPL;
        piece = KC ? 0 : (tid % PPL) * W;
#pragma unroll
        for (int f = 0; f < NF; ++f) {
            const int t = KC ? line + f * 8 : piece;
            const bool in = r0 + t < o.r.extent;
            if (in) live |= 1u << f;
            const int r = in ? r0 + t : r0;
            const Cursor c = seek(o.r, r);
            if (EQ) {
                foff[f] = at.bytes + c.blk * o.r.blk_bytes + (r - c.lo) * o.r.cell_bytes;
            } else {
                fflat[f] = at.flat + c.blk * o.r.nb_stride;
                if (KC) {
                    fa[f] = (r - c.lo) * at.cf + at.p0 * (c.hi - c.lo) + at.p1;
                } else {
                    fa[f] = c.hi - c.lo;
                    fb = (r - c.lo) * at.cs + at.p2;
                }
            }
        }
        cur = seek(o.k, min(k0 + (tid & 31), K - 1));
    }
    __device__ __forceinline__ void issue(uint32_t dst, int k0, int lane) {
        const int x = min(k0 + lane, K - 1);
        advance(*dk, cur, x);
        int64_t off = 0;
        int flat = 0, a = 0, b = 0;
        if (EQ) {
            off = cur.blk * dk->blk_bytes + (x - cur.lo) * dk->cell_bytes;
        } else {
            flat = cur.blk * dk->nb_stride;
            a = KC ? cur.hi - cur.lo : (x - cur.lo) * ba.cf + ba.p0 * (cur.hi - cur.lo) + ba.p1;
            b = KC ? (x - cur.lo) * ba.cs + ba.p2 : 0;
        }
        auto enter = [&](int fl) {
            if (!EQ && fl != have) {
                have = fl;
#pragma unroll
                for (int f = 0; f < NF; ++f) start[f] = base + blk_off[fflat[f] + fl];
            }
        };
        if (KC) {
            enter(flat);
            const bool in = k0 + lane < K;
#pragma unroll
            for (int n = 0; n < NP; ++n)
                cp_async4(dst + (lane * (T + 4) + line + n * 8) * 4, EQ ? base + (foff[n] + off) : start[n] + (int64_t)(a * fa[n] + b) * 4, in, live >> n & 1);
        } else {
#pragma unroll
            for (int n = 0; n < NP; ++n) {
                const int l = line + n * LP;
                const char* src;
                if (EQ) {
                    src = base + (foff[0] + __shfl_sync(0xffffffffu, off, l));
                } else {
                    const int fl = __shfl_sync(0xffffffffu, flat, l), al = __shfl_sync(0xffffffffu, a, l);
                    enter(fl);
                    src = start[0] + (int64_t)(fa[0] * al + fb) * 4;
                }
                const bool in = k0 + l < K;
                if (W == 4) cp_async16(dst + (l * (T + 4) + piece) * 4, src, in, live & 1);
                else cp_async4(dst + (l * (T + 4) + piece) * 4, src, in, live & 1);
            }
        }
    }
};

__device__ __forceinline__ uint64_t pack2(float lo, float hi) {
    uint64_t r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(lo), "f"(hi));
    return r;
}
__device__ __forceinline__ void st_cluster_f32x4(uint32_t at, const float* v) {
    asm volatile("st.shared::cluster.v4.f32 [%0], {%1, %2, %3, %4};" ::"r"(at), "f"(v[0]), "f"(v[1]), "f"(v[2]), "f"(v[3]) : "memory");
}
__device__ __forceinline__ void st_cluster_f32(uint32_t at, float v) { asm volatile("st.shared::cluster.f32 [%0], %1;" ::"r"(at), "f"(v) : "memory"); }

// WA, WB: cells per piece of an operand whose row index is contiguous (4 or 1); KCA, KCB: its contracted index is
template <int T, bool KCA, int WA, bool KCB, int WB, bool EQ>
__global__ void __launch_bounds__(NT) contract_f32_kernel(const __grid_constant__ Params p) {
    using C = Cfg<T>;
    constexpr int U = T / 16, V = U < 4 ? U : 4;      // outputs a side per thread, in groups of V consecutive rows / columns
    extern __shared__ __align__(16) uint8_t smem[];
    const uint32_t sbase = smem_u32(smem);
    const int tid = threadIdx.x, lane = tid & 31, tr = tid / 16, tc = tid % 16;
    const int split = p.split, rank = (int)blockIdx.x % split, t = (int)blockIdx.x / split;
    const int m0 = t / p.tiles_n * T, n0 = t % p.tiles_n * T;
    const int bx[MAX_BATCH] = {(int)blockIdx.z, (int)blockIdx.y};
    const int chunks = (p.K + TK - 1) / TK, c0 = (int)((int64_t)chunks * rank / split), c1 = (int)((int64_t)chunks * (rank + 1) / split);
    Walk<T, KCA, WA, EQ> wa;
    Walk<T, KCB, WB, EQ> wb;
    wa.init(p.A, batch_at(p.A, bx), tid, m0, c0 * TK);
    wb.init(p.B, batch_at(p.B, bx), tid, n0, c0 * TK);
    if (split == 1) {                           // (clusters do not overlap: ja_launch.cuh)
        ja_wait_for_stream();
        if (p.let_next) ja_let_next_start();
    }
    uint64_t acc2[U][U / 2];                    // pairs of neighbouring columns
#pragma unroll
    for (int u = 0; u < U; ++u)
#pragma unroll
        for (int w = 0; w < U / 2; ++w) acc2[u][w] = 0;
    auto issue = [&](int ch) {
        if (ch < c1) {
            const uint32_t dst = sbase + (ch - c0) % C::STAGES * C::STAGE;
            wa.issue(dst, ch * TK, lane);
            wb.issue(dst + C::OPERAND, ch * TK, lane);
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
    };
#pragma unroll
    for (int s = 0; s < C::STAGES - 1; ++s) issue(c0 + s);
    for (int ch = c0; ch < c1; ++ch) {
        asm volatile("cp.async.wait_group %0;" ::"n"(C::STAGES - 2) : "memory");
        __syncthreads();                        // this stage has landed everywhere; everyone is done with the one before it
        issue(ch + C::STAGES - 1);
        const float* As = reinterpret_cast<const float*>(smem + (ch - c0) % C::STAGES * C::STAGE);
        const float* Bs = As + C::OPERAND / 4;
#pragma unroll 8
        for (int kk = 0; kk < TK; ++kk) {
            float a[U], b[U];
#pragma unroll
            for (int u = 0; u < U; u += V) {
                if (V == 4) {
                    *reinterpret_cast<float4*>(a + u) = *reinterpret_cast<const float4*>(As + kk * C::PITCH + u / 4 * 64 + tr * 4);
                    *reinterpret_cast<float4*>(b + u) = *reinterpret_cast<const float4*>(Bs + kk * C::PITCH + u / 4 * 64 + tc * 4);
                } else {
                    *reinterpret_cast<float2*>(a) = *reinterpret_cast<const float2*>(As + kk * C::PITCH + tr * 2);
                    *reinterpret_cast<float2*>(b) = *reinterpret_cast<const float2*>(Bs + kk * C::PITCH + tc * 2);
                }
            }
            uint64_t b2[U / 2];
#pragma unroll
            for (int w = 0; w < U / 2; ++w) b2[w] = pack2(b[2 * w], b[2 * w + 1]);
#pragma unroll
            for (int u = 0; u < U; ++u) {
                const uint64_t a2 = pack2(a[u], a[u]);
#pragma unroll
                for (int w = 0; w < U / 2; ++w) asm("fma.rn.f32x2 %0, %1, %2, %0;" : "+l"(acc2[u][w]) : "l"(a2), "l"(b2[w]));
            }
        }
    }
    asm volatile("cp.async.wait_all;" ::: "memory");
    float acc[U][U];
#pragma unroll
    for (int u = 0; u < U; ++u)
#pragma unroll
        for (int w = 0; w < U / 2; ++w) asm("mov.b64 {%0, %1}, %2;" : "=f"(acc[u][2 * w]), "=f"(acc[u][2 * w + 1]) : "l"(acc2[u][w]));
    // ---- a cluster's slices: every CTA's rows go to the CTA that stores them, then each sums its rows in rank order ----
    const int mine = T / split;
    if (split > 1) {
        cluster_sync_all();                     // every CTA's stages are free
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const int r = u / V * 64 + tr * V + u % V;
            const uint32_t at = mapa_cluster(sbase + (uint32_t)((rank * mine + r % mine) * C::PITCH) * 4u, (uint32_t)(r / mine));
#pragma unroll
            for (int w = 0; w < U; w += V) {
                if (V == 4) st_cluster_f32x4(at + (uint32_t)(w / 4 * 64 + tc * 4) * 4u, &acc[u][w]);
                else { st_cluster_f32(at + (uint32_t)(tc * 2) * 4u, acc[u][0]); st_cluster_f32(at + (uint32_t)(tc * 2 + 1) * 4u, acc[u][1]); }
            }
        }
        cluster_sync_all();
    }
    const Rel& o = p.C;                         // r = m, k = n, n is the later index
    const BatchAt ba = batch_at(o, bx);
    const int es = p.c_dtype == JA_F32 ? 4 : 2;
    // V consecutive columns, located once, and the rows below each other that go there
    struct Columns {
        int n, flat[V], w[V], at[V];
        int64_t off[V];
    };
    auto columns = [&](int col) -> Columns {
        Columns c;
        c.n = max(0, min(V, p.N - col));
        if (c.n == 0) return c;
        Cursor cc = seek(o.k, col);
#pragma unroll
        for (int j = 0; j < V; ++j) {
            const int x = min(col + j, p.N - 1);
            advance(o.k, cc, x);
            c.flat[j] = ba.flat + cc.blk * o.k.nb_stride;
            c.w[j] = cc.hi - cc.lo;
            c.at[j] = (x - cc.lo) * ba.cs + ba.p2;
            c.off[j] = ba.bytes + cc.blk * o.k.blk_bytes + (x - cc.lo) * o.k.cell_bytes;
        }
        return c;
    };
    Cursor rc = {0, 0, 0};
    auto put = [&](int row, const Columns& c, const float* f) {   // rows come in ascending order
        if (row >= p.M || c.n == 0) return;
        if (rc.hi == 0) rc = seek(o.r, row);
        else advance(o.r, rc, row);
        const int64_t roff = rc.blk * o.r.blk_bytes + (row - rc.lo) * o.r.cell_bytes;
        const int rflat = rc.blk * o.r.nb_stride, ra = (row - rc.lo) * ba.cf + ba.p0 * (rc.hi - rc.lo) + ba.p1;
        auto address = [&](int j) -> char* {
            if (o.equal) return o.base + (c.off[j] + roff);
            return o.base + o.blk_off[c.flat[j] + rflat] + (int64_t)(c.w[j] * ra + c.at[j]) * es;
        };
        if (V == 4 && o.g == 4) {               // split points are multiples of four: the group lies in one block
            char* dst = address(0);
            if (p.c_dtype == JA_F32) *reinterpret_cast<float4*>(dst) = make_float4(f[0], f[1], f[2], f[3]);
            else if (p.c_dtype == JA_F16) *reinterpret_cast<uint2*>(dst) = make_uint2(ja_pack16<true>(f[0], f[1]), ja_pack16<true>(f[2], f[3]));
            else *reinterpret_cast<uint2*>(dst) = make_uint2(ja_pack16<false>(f[0], f[1]), ja_pack16<false>(f[2], f[3]));
            return;
        }
#pragma unroll
        for (int j = 0; j < V; ++j) {
            if (j >= c.n) continue;
            char* dst = address(j);
            if (p.c_dtype == JA_F32) *reinterpret_cast<float*>(dst) = f[j];
            else if (p.c_dtype == JA_F16) *reinterpret_cast<__half*>(dst) = __float2half_rn(f[j]);
            else *reinterpret_cast<__nv_bfloat16*>(dst) = __float2bfloat16_rn(f[j]);
        }
    };
    if (split == 1) {
#pragma unroll
        for (int w = 0; w < U; w += V) {
            const Columns c = columns(n0 + w / V * 64 + tc * V);
            rc.hi = 0;
#pragma unroll
            for (int u = 0; u < U; ++u) put(m0 + u / V * 64 + tr * V + u % V, c, &acc[u][w]);
        }
    } else {
        const float* tile = reinterpret_cast<const float*>(smem);
        constexpr int GROUPS = T / V;
        static_assert(NT % GROUPS == 0, "a thread keeps its columns");
        const int c0l = tid % GROUPS * V;
        const Columns c = columns(n0 + c0l);
        for (int l = tid / GROUPS; l < mine; l += NT / GROUPS) {
            float f[V];
#pragma unroll
            for (int j = 0; j < V; ++j) f[j] = 0.f;
            for (int s = 0; s < split; ++s)
#pragma unroll
                for (int j = 0; j < V; ++j) f[j] += tile[(s * mine + l) * C::PITCH + c0l + j];
            put(m0 + rank * mine + l, c, f);
        }
    }
}

template <int T, bool KCA, int WA, bool KCB, int WB, bool EQ>
ja_status_t launch(Params p, cudaStream_t st) {
    static std::atomic<int> places_of[64], sms_of[64];   // CTAs that an SM holds; SMs
    int dev = 0;
    cudaGetDevice(&dev);
    int places = places_of[dev & 63].load();
    if (!places) {
        JA_CUDA(cudaFuncSetAttribute(contract_f32_kernel<T, KCA, WA, KCB, WB, EQ>, cudaFuncAttributeMaxDynamicSharedMemorySize, Cfg<T>::SMEM));
        JA_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&places, contract_f32_kernel<T, KCA, WA, KCB, WB, EQ>, NT, Cfg<T>::SMEM));
        sms_of[dev & 63].store(ja_sm_count());
        places_of[dev & 63].store(places = std::max(places, 1));
    }
    p.let_next = ja_let_next_pays((int64_t)p.tiles_m * p.tiles_n * p.split * p.batch[0] * p.batch[1], sms_of[dev & 63].load(), places);
    const dim3 grid((unsigned)(p.tiles_m * p.tiles_n * p.split), (unsigned)p.batch[1], (unsigned)p.batch[0]);
    if (p.split > 1) JA_CUDA(ja_launch_kernel_after(contract_f32_kernel<T, KCA, WA, KCB, WB, EQ>, grid, NT, Cfg<T>::SMEM, (unsigned)p.split, st, p));
    else JA_CUDA(ja_launch_kernel(contract_f32_kernel<T, KCA, WA, KCB, WB, EQ>, grid, NT, Cfg<T>::SMEM, 1, st, p));
    return JA_OK;
}
template <int T, bool KCA, int WA, bool KCB, int WB>
ja_status_t launch_e(const Params& p, cudaStream_t st) {
    const bool eq = p.A.equal && p.B.equal;
    if constexpr (T == 128) return launch<T, KCA, WA, KCB, WB, true>(p, st);   // chosen for equal blocks alone (registers)
    else return eq ? launch<T, KCA, WA, KCB, WB, true>(p, st) : launch<T, KCA, WA, KCB, WB, false>(p, st);
}
template <int T, bool KCA, int WA>
ja_status_t launch_b(const Params& p, cudaStream_t st) {
    if (p.B.kc) return launch_e<T, KCA, WA, true, 1>(p, st);
    return p.B.g == 4 ? launch_e<T, KCA, WA, false, 4>(p, st) : launch_e<T, KCA, WA, false, 1>(p, st);
}
template <int T>
ja_status_t launch_a(const Params& p, cudaStream_t st) {
    if (p.A.kc) return launch_b<T, true, 1>(p, st);
    return p.A.g == 4 ? launch_b<T, false, 4>(p, st) : launch_b<T, false, 1>(p, st);
}

}  // namespace

struct ContractF32Plan {
    Params p;
    int tile;
};

ja_status_t ja_contract_f32_plan(const std::string& ta, const std::string& tb, const std::string& tc, const ja_relation* A, const ja_relation* B,
                                 const ja_relation* C, std::shared_ptr<ContractF32Plan>* out) {
    out->reset();
    if (A->dtype != JA_F32 || B->dtype != JA_F32) return JA_OK;
    ProductRoles roles;
    if (!product_roles(ta, tb, tc, &roles) || !fits_32_bits(A) || !fits_32_bits(B) || !fits_32_bits(C)) return JA_OK;
    std::shared_ptr<ContractF32Plan> plan(new ContractF32Plan());
    Params& p = plan->p;
    memset(&p, 0, sizeof p);
    const bool swap = tc.find(roles.m) > tc.find(roles.n);   // columns: the later of the output's two indices
    if (swap) std::swap(roles.m, roles.n);
    fill_rel(&p.A, swap ? B : A, swap ? tb : ta, roles.m, roles.k, roles.batch, 4);
    fill_rel(&p.B, swap ? A : B, swap ? ta : tb, roles.n, roles.k, roles.batch, 4);
    fill_rel(&p.C, C, tc, roles.m, roles.n, roles.batch, 4);
    p.M = p.A.r.extent;
    p.N = p.B.r.extent;
    p.K = p.A.k.extent;
    p.c_dtype = (int)C->dtype;
    for (int i = 0; i < MAX_BATCH; ++i) {
        const size_t at = roles.batch[i] ? tc.find(roles.batch[i]) : std::string::npos;
        p.batch[i] = at == std::string::npos ? 1 : (int)C->extent[at];
    }
    if (p.batch[0] > 65535 || p.batch[1] > 65535) return JA_OK;
    // The largest tile that still gives most SMs one, and slices of the contracted index (at least four stages each) while there are
    // too few even of the smallest.
    const int64_t nb = (int64_t)p.batch[0] * p.batch[1], sms = ja_sm_count(), chunks = (p.K + TK - 1) / TK;
    auto tiles = [&](int t) { return nb * ((p.M + t - 1) / t) * ((p.N + t - 1) / t); };
    int t = 32;
    if (tiles(64) >= sms) t = 64;
    if (p.A.equal && p.B.equal && tiles(128) >= sms) t = 128;
    p.split = 1;
    while (p.split < 8 && tiles(t) * p.split * 2 <= 2 * sms && chunks >= 8 * p.split) p.split *= 2;
    p.tiles_m = (p.M + t - 1) / t;
    p.tiles_n = (p.N + t - 1) / t;
    if ((int64_t)p.tiles_m * p.tiles_n * p.split >= (1ll << 31)) return JA_OK;
    plan->tile = t;
    *out = plan;
    return JA_OK;
}

ja_status_t ja_launch_contract_f32(const ContractF32Plan& plan, cudaStream_t st) {
    ja_status_t s = plan.tile == 128 ? launch_a<128>(plan.p, st) : plan.tile == 64 ? launch_a<64>(plan.p, st) : launch_a<32>(plan.p, st);
    if (s == JA_OK) ja_count_launch();
    return s;
}

// tc_gemm.cu -- tensor-core GEMM of the batched path (the block's
// projections, Sec. III-A, once B * n fed rows make them a dense contraction):
//
//   out[n][f] (+)= sum_k (a_hi[n][k] + a_lo[n][k]) * w[f][k]
//
// w: bf16 weights, K-major ([N_w][K]); a_hi + a_lo: the fp32 activations as
// two bf16 parts, K-major ([M][K]).  The weights are the MMA's M = 128 side
// (one 128-row tile per CTA) and the activation rows its N side (NT per
// tile), so a handful of fed rows still fills the tensor core.  The two parts
// of the activations lie one behind the other and are one operand of 2 NT
// columns, whose two halves of the accumulator are added when it is read: an
// MMA of N = 128 takes as long as one of N = 256 (W1 of 512 rows with two MMAs
// per k-step, one per part: 13.2 us; with one: 11.3; d = 1024, q|k|v, W_o, W1
// and W2 of 128 rows: 9.5 us on average, now 8.4).  Each accumulator truncates
// half as often, too: K = 4096 is off by 4.4e-6 of the result's scale, by
// 9.2e-6 with both parts in one accumulator.
//
// Per CTA: one elected thread streams 64-wide k-chunks of the weight tile
// and of both activation parts into a 4-stage shared-memory ring with TMA
// (128-byte swizzled tiles), a second elected thread issues tcgen05.mma
// into a TMEM accumulator (128 lanes x 2 NT fp32 columns) and releases each
// stage with tcgen05.commit.  8 or 16 warps read the accumulator back with
// tcgen05.ld and finish it from the registers (tc_epilogue.cuh): warps w, w + 4,
// .. share TMEM lanes 32 (w % 4) .., i.e. weight rows, and divide the columns.
// Staging the tile in shared memory first, to write float4 pieces of rows,
// took 0.65 us more and left the stores as long (512 rows,
// d = 1024: W2 12.0 -> 10.2 us); where K splits meet in a cluster it is the
// layout of the exchange (q|k|v and W1 of 128 rows: 8.0 -> 7.3 us).  Grid:
// (N_w / 128 weight tiles, K splits, activation tiles).  The weight copies of
// the first stages are issued before griddepcontrol.wait; the activation copies
// after it.
#include <cuda.h>

#include <condition_variable>
#include <cstdio>
#include <cstring>
#include <mutex>

#include "common.cuh"
#include "kernels.cuh"
#include "mtp.h"
#include "tc_epilogue.cuh"
#include "tcgen05.cuh"

namespace mtp {
namespace {

constexpr int TC_M = 128;      // weight rows per CTA (MMA M)
constexpr int TC_K = 64;       // k per stage: one 128-byte swizzle row of bf16
// ring stages per activation tile size: about 190 KB of copies in flight per CTA
__host__ __device__ constexpr int tc_stages(int nt) { return nt <= 32 ? 8 : (nt <= 64 ? 6 : 4); }
constexpr int TC_MAX_STAGES = 8;
// 8 or 16 warps: two elected lanes run the ring; the epilogue is instruction-latency bound (one warp per
// scheduler hid nothing).  16 where a thread of 8 would finish 64 rows with arithmetic or read-modify-write
// (d = 1024, 512 rows: q|k|v 10.1 -> 9.1 us, W1 10.2 -> 9.3, W_o 4.9 -> 4.5, W2 8.4 -> 7.9); plain stores
// gain nothing (W1 11.3 vs 11.7 us), nor do the halved tiles of a cluster.
__host__ __device__ constexpr int tc_threads(int nt, int epi, bool cluster) {
    return nt == 128 && epi != TC_STORE && !cluster ? 512 : 256;
}
constexpr uint32_t TC_W_BYTES = TC_M * TC_K * 2;

// ---- PTX wrappers (tcgen05, TMA) ----
__device__ __forceinline__ void tma_load_2d(void* dst, const CUtensorMap* map, int x, int y, uint64_t* bar) {
    asm volatile(
        "cp.async.bulk.tensor.2d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], [%4];" ::"r"(
            smem_addr(dst)),
        "l"(reinterpret_cast<uint64_t>(map)), "r"(x), "r"(y), "r"(smem_addr(bar))
        : "memory");
}
// Bulk copy of `bytes` from this CTA's shared memory to shared memory of a CTA of the cluster
// (dst, bar: shared::cluster addresses), completing on that CTA's barrier.  16-byte aligned.
__device__ __forceinline__ void bulk_copy_s2s_cluster(uint32_t dst, uint32_t src, uint32_t bytes, uint32_t bar) {
    asm volatile("cp.async.bulk.shared::cluster.shared::cta.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(dst),
                 "r"(src), "r"(bytes), "r"(bar)
                 : "memory");
}
// Shared-memory address `saddr` of this CTA mapped to the CTA of cluster rank `rank`.
__device__ __forceinline__ uint32_t mapa_rank(uint32_t saddr, int rank) {
    uint32_t r;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(saddr), "r"(rank));
    return r;
}

// Instruction descriptor of kind::f16: fp32 accumulator, bf16 A and B, both
// K-major, M = 128, N = n.
__host__ __device__ constexpr uint32_t tc_idesc(int n) {
    return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(n >> 3) << 17) | ((uint32_t)(TC_M >> 4) << 24);
}

template <int NT, int EPI, bool CLUSTER>
__global__ void __launch_bounds__(tc_threads(NT, EPI, CLUSTER), 1)
    tc_gemm_kernel(const __grid_constant__ CUtensorMap tw, const __grid_constant__ CUtensorMap tah,
                   const __grid_constant__ CUtensorMap tal, const TcGemmArgs a) {
    extern __shared__ __align__(1024) unsigned char smem_raw[];
    constexpr uint32_t A_BYTES = NT * TC_K * 2, STAGE = TC_W_BYTES + 2 * A_BYTES;
    constexpr uint32_t TMEM_COLS = 2 * NT;  // the products with the hi parts, then with the lo parts
    constexpr int TC_STAGES = tc_stages(NT), THREADS = tc_threads(NT, EPI, CLUSTER), PARTS = THREADS / 128;
    __shared__ uint64_t full[TC_MAX_STAGES], empty[TC_MAX_STAGES], done, red_bar;
    __shared__ uint32_t tmem_base;
    __shared__ int s_ok;
    __shared__ long long s_rowbase[NT];  // TC_QKV: element offset of the row's key row in its page (-1: none)
    __shared__ int s_rowt[NT];           // TC_QKV: key row within the page; TC_GELU_PACK: row of a sequence
    unsigned char* smem = reinterpret_cast<unsigned char*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
    TraceEnd trace_guard(a.trace);
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int tile = blockIdx.x, split = blockIdx.y, ntile = blockIdx.z;
    const int chunks = a.k_chunks;
    const int kc0 = split * chunks;
    const int arow = ntile * NT;

    if (warp == 0) {
        tmem_alloc(&tmem_base, TMEM_COLS);
        tmem_relinquish();
    }
    if (tid == 32) {
        for (int s = 0; s < TC_STAGES; ++s) {
            mbar_init(&full[s], 1);
            mbar_init(&empty[s], 1);
        }
        mbar_init(&done, 1);
        mbar_init(&red_bar, 1);
        fence_barrier_init();
        s_ok = 1;
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = tmem_base;

    // weights of the first stages: independent of the previous kernel
    auto w_coords = [&](int c, int& x, int& y) {
        const int kc = kc0 + c;
        if (a.w_rows_per_kchunk) {  // k-chunk kc is a block of rows (W_o stored per head)
            x = 0;
            y = kc * a.w_rows_per_kchunk + tile * TC_M;
        } else {
            x = kc * TC_K;
            y = tile * TC_M;
        }
    };
    const int pre = chunks < TC_STAGES ? chunks : TC_STAGES;
    if (tid == 0) {
        for (int c = 0; c < pre; ++c) {
            unsigned char* st = smem + (size_t)c * STAGE;
            mbar_arrive_expect_tx(&full[c], STAGE);
            int x, y;
            w_coords(c, x, y);
            tma_load_2d(st, &tw, x, y, &full[c]);
        }
    }
    pdl_launch_dependents();
    pdl_wait();
    trace_wait(a.trace);

    // The elected lanes run the ring; the rest of warps 0 and 1 wait at __syncwarp
    // (not in the barrier poll below, which would hold up their elected lane).
    if (tid == 0) {  // producer: activations of the first stages, then the rest of the ring
        for (int c = 0; c < chunks; ++c) {
            const int s = c % TC_STAGES;
            unsigned char* st = smem + (size_t)s * STAGE;
            if (c >= TC_STAGES) {
                if (!mbar_wait(&empty[s], (uint32_t)((c / TC_STAGES) - 1) & 1, a.err)) {
                    s_ok = 0;
                    break;
                }
                mbar_arrive_expect_tx(&full[s], STAGE);
                int x, y;
                w_coords(c, x, y);
                tma_load_2d(st, &tw, x, y, &full[s]);
            }
            const int kx = (kc0 + c) * TC_K;
            tma_load_2d(st + TC_W_BYTES, &tah, kx, arow, &full[s]);
            tma_load_2d(st + TC_W_BYTES + A_BYTES, &tal, kx, arow, &full[s]);
        }
    } else if (tid == 32) {  // MMA issuer
        constexpr uint32_t IDESC = tc_idesc(2 * NT);  // the stage's hi and lo rows are one operand
        int c = 0;
        for (; c < chunks; ++c) {
            const int s = c % TC_STAGES;
            if (!mbar_wait(&full[s], (uint32_t)(c / TC_STAGES) & 1, a.err)) break;
            tc_fence_after();
            const uint32_t wb = smem_addr(smem + (size_t)s * STAGE);
            const uint32_t ab = wb + TC_W_BYTES;
#pragma unroll
            for (int kk = 0; kk < TC_K / 16; ++kk)
                tc_mma(tmem, sw128_desc(wb + kk * 32), sw128_desc(ab + kk * 32), IDESC, (c | kk) != 0);
            tc_commit(&empty[s]);  // stage s is free once these MMAs have read it
        }
        if (c < chunks) s_ok = 0;
        tc_commit(&done);  // every MMA issued above has completed
    } else if (warp >= 2 && (EPI == TC_QKV || EPI == TC_GELU_PACK)) {
        // per-row facts of the epilogue, gathered by the two idle warps while the ring runs
        for (int j = tid - 64; j < NT; j += THREADS - 64) {
            const int n = arow + j;
            const int seq = n < a.m ? a.row_seq[n] : -1;
            long long base = -1;
            int t = 0;
            if (EPI == TC_QKV && seq >= 0) {
                const int pos = a.row_pos[n];
                t = pos % a.page_size;
                const int page = a.block_table[(size_t)seq * a.bt_stride + pos / a.page_size];
                if (page < 0)
                    atomicOr(a.err, ERR_BOUNDS);
                else
                    base = (long long)page * a.page_elems + a.layer_off + (long long)t * HEAD_DIM;
            }
            s_rowbase[j] = seq >= 0 ? base : -2;  // -2: no sequence
            s_rowt[j] = EPI == TC_QKV ? t : (seq >= 0);
        }
    }
    if (warp < 2) __syncwarp();

    // epilogue: lane = weight row f (TMEM lane of the warp's quarter), 32 activation rows per load
    // one thread polls (a poll costs each polling thread, even on a completed phase); the block
    // barrier hands the result to the others
    const bool fin = __syncthreads_and(tid == 0 ? mbar_wait(&done, 0, a.err) : true) != 0;
    tc_fence_after();
    trace_mark(a.trace, 0);  // accumulator complete
    const bool good = fin && s_ok;
    const int quarter = warp & 3, part = warp >> 2;  // the TMEM lanes (weight rows) this warp may read, its columns
    const int f = tile * TC_M + quarter * 32 + lane;
    const uint32_t acc = tmem + ((uint32_t)(quarter * 32) << 16);
    const int rows = min(NT, a.m - arow);  // activation rows of the tile
    if constexpr (CLUSTER) {
        // K splits reduced in a cluster: Sc consecutive splits of this tile are one cluster, and each
        // finishes an Sc-th of the activation rows.  A thread reads its weight row's columns at once and
        // leaves them in the layout in which their finishers read them, [128 weight rows][rows of a share];
        // a peer's share goes there in one bulk copy (into the space of its ring: the cluster barrier says
        // that everyone's MMAs are done, and is waited for behind the staging).  Then each thread adds the
        // Sc partials of its weight row in rank order.  (16-byte st.async pushes from the registers: 4.8 us
        // for the 48 KB of a CTA at 128 rows, the copies 1.9 us.)
        const int Sc = a.cluster_reduce, rank = split % Sc, R = NT / Sc;  // rows of a share
        constexpr int N = NT / 8;             // four units of N rows per thread: half of every share
        const int pitch = R + 4;              // floats per (sender, weight row): 16-byte rows, spread banks
        const uint32_t part_bytes = (uint32_t)(TC_M * pitch * 4);
        float* recv = reinterpret_cast<float*>(smem);  // parts by sender, then the staged ones by receiver
        float* staged = recv + (size_t)Sc * TC_M * pitch;
        const int fl = quarter * 32 + lane;
        if (tid == 0) mbar_arrive_expect_tx(&red_bar, part_bytes * (uint32_t)(Sc - 1));
        __syncthreads();
        cluster_arrive_release();  // this CTA's ring is free and its barrier armed
        float v[4][N], w[4][N];
        // unit u: rows r0(u) .. + N of share p(u)
        auto share = [&](int u) { return Sc == 4 ? u : u >> 1; };
        auto first = [&](int u) { return part * (R / 2) + (Sc == 4 ? 0 : (u & 1) * N); };
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            tmem_ld_issue<N>(acc + (uint32_t)(share(u) * R + first(u)), v[u]);
            tmem_ld_issue<N>(acc + (uint32_t)(NT + share(u) * R + first(u)), w[u]);
        }
        tmem_ld_wait();
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            tmem_ld_done(v[u]);
            tmem_ld_done(w[u]);
#pragma unroll
            for (int e = 0; e < N; ++e) v[u][e] += w[u][e];
        }
        if (good) {
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const int p = share(u);
                float* dst = (p == rank ? recv : staged) + ((size_t)p * TC_M + fl) * pitch + first(u);
#pragma unroll
                for (int e = 0; e < N; e += 4)
                    *reinterpret_cast<float4*>(dst + e) = make_float4(v[u][e], v[u][e + 1], v[u][e + 2], v[u][e + 3]);
            }
        }
        fence_proxy_async();  // (read by the copies)
        trace_mark(a.trace, 1);  // thread 0's rows staged
        cluster_wait();
        __syncthreads();
        trace_mark(a.trace, 2);  // every ring free, every row staged
        if (tid < Sc - 1 && good) {  // one copy per issuing thread, receivers in rotated order
            const int p = (rank + 1 + tid) % Sc;
            bulk_copy_s2s_cluster(mapa_rank(smem_addr(recv + (size_t)rank * TC_M * pitch), p),
                                  smem_addr(staged + (size_t)p * TC_M * pitch), part_bytes,
                                  mapa_rank(smem_addr(&red_bar), p));
        }
        const bool got = __syncthreads_and(tid == 0 ? mbar_wait(&red_bar, 0, a.err) : true) != 0;
        cluster_arrive_relaxed();  // (waited for before leaving)
        trace_mark(a.trace, 3);  // the peers' partial rows received
        if (good && got) {
            const float bias = a.bias ? __ldg(a.bias + f) : 0.f;
            for (int r0 = part * (R / 2); r0 < (part + 1) * (R / 2); r0 += N) {
                float y[N];
#pragma unroll
                for (int e = 0; e < N; ++e) y[e] = 0.f;
#pragma unroll
                for (int src = 0; src < TC_CLUSTER_SPLITS; ++src) {  // every split's partial, in rank order
                    if (src >= Sc) break;
                    const float4* part = reinterpret_cast<const float4*>(recv + ((size_t)src * TC_M + fl) * pitch + r0);
#pragma unroll
                    for (int e = 0; e < N; e += 4) {
                        const float4 x = part[e / 4];
                        y[e] += x.x;
                        y[e + 1] += x.y;
                        y[e + 2] += x.z;
                        y[e + 3] += x.w;
                    }
                }
                const int j0 = rank * R + r0;
                tc_epilogue<EPI, false>(a, y, arow + j0, j0, rows - j0, f, bias, s_rowbase, s_rowt);
            }
            trace_mark(a.trace, 5);  // thread 0's stores issued
        }
    } else if (good) {
        constexpr int COLS = NT / PARTS, N = COLS < 32 ? COLS : 32;
        // the tile's first split adds the bias (heads: rows past n_valid have none)
        const float bias = a.bias && split == 0 && (!a.n_valid || f < a.n_valid) ? __ldg(a.bias + f) : 0.f;
        for (int j0 = part * COLS; j0 < (part + 1) * COLS && j0 < rows; j0 += N) {
            float v[N], w[N];
            tmem_ld_issue<N>(acc + (uint32_t)j0, v);
            tmem_ld_issue<N>(acc + (uint32_t)(NT + j0), w);
            tmem_ld_wait();
            tmem_ld_done(v);
            tmem_ld_done(w);
#pragma unroll
            for (int e = 0; e < N; ++e) v[e] += w[e];
            tc_epilogue<EPI, true>(a, v, arow + j0, j0, rows - j0, f, bias, s_rowbase, s_rowt);
        }
        trace_mark(a.trace, 5);  // thread 0's stores issued
    }
    // the MMAs may still be running: wait for them (bounded) before freeing TMEM
    if (!fin) mbar_wait(&done, 0, nullptr);
    if constexpr (CLUSTER) cluster_wait();  // no peer still pushes into this CTA
    tc_fence_before();
    __syncthreads();
    if (warp == 0) tmem_dealloc(tmem, TMEM_COLS);
}

// ---- tensor maps ----
using EncodeTiled = CUresult (*)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                 const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                                 CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

EncodeTiled encode_fn() {
    static EncodeTiled fn = nullptr;
    static std::once_flag once;
    std::call_once(once, [] {
        void* p = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault, &q) ==
                cudaSuccess &&
            q == cudaDriverEntryPointSuccess)
            fn = reinterpret_cast<EncodeTiled>(p);
    });
    return fn;
}

template <int NT>
size_t tc_smem() {
    return (size_t)tc_stages(NT) * (TC_W_BYTES + 2u * NT * TC_K * 2) + 1024;
}

template <int NT, typename K>
cudaError_t launch_kern(K kern, int threads, const TcGemm& g, cudaStream_t s, bool pdl) {
    const size_t smem = tc_smem<NT>();
    cudaError_t e = ensure_kernel_smem(reinterpret_cast<const void*>(kern), smem);
    if (e != cudaSuccess) return e;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(g.n_w / TC_M, g.splits, (g.args.m + NT - 1) / NT);
    cfg.blockDim = dim3(threads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = pdl ? 1 : 0;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    if (g.args.cluster_reduce > 1) {  // consecutive K splits of a tile form one cluster
        attr[1].id = cudaLaunchAttributeClusterDimension;
        attr[1].val.clusterDim.x = 1;
        attr[1].val.clusterDim.y = g.args.cluster_reduce;
        attr[1].val.clusterDim.z = 1;
        cfg.numAttrs = 2;
    }
    return cudaLaunchKernelEx(&cfg, kern, g.w, g.a_hi, g.a_lo, g.args);
}

template <int NT>
cudaError_t launch_nt(const TcGemm& g, cudaStream_t s, bool pdl) {
    const bool cluster = g.args.cluster_reduce > 1;
    switch (g.args.epilogue) {
        case TC_STORE: return launch_kern<NT>(tc_gemm_kernel<NT, TC_STORE, false>, tc_threads(NT, TC_STORE, false), g, s, pdl);
        case TC_ACCUM: return launch_kern<NT>(tc_gemm_kernel<NT, TC_ACCUM, false>, tc_threads(NT, TC_ACCUM, false), g, s, pdl);
        case TC_QKV:
            if (cluster) return launch_kern<NT>(tc_gemm_kernel<NT, TC_QKV, true>, tc_threads(NT, TC_QKV, true), g, s, pdl);
            return launch_kern<NT>(tc_gemm_kernel<NT, TC_QKV, false>, tc_threads(NT, TC_QKV, false), g, s, pdl);
        case TC_GELU_PACK:
            if (cluster) return launch_kern<NT>(tc_gemm_kernel<NT, TC_GELU_PACK, true>, tc_threads(NT, TC_GELU_PACK, true), g, s, pdl);
            return launch_kern<NT>(tc_gemm_kernel<NT, TC_GELU_PACK, false>, tc_threads(NT, TC_GELU_PACK, false), g, s, pdl);
        default: return cudaErrorInvalidValue;
    }
}

}  // namespace

int tc_encode_2d(CUtensorMap* map, const void* base, uint64_t inner, uint64_t rows, uint32_t box_rows,
                 bool pre_swizzled) {
    EncodeTiled fn = encode_fn();
    if (!fn) return -1;
    if ((reinterpret_cast<uintptr_t>(base) & 15) || (inner * 2) % 16 || box_rows == 0 || box_rows > 256) return -2;
    const cuuint64_t dims[2] = {inner, rows};
    const cuuint64_t strides[1] = {inner * 2};
    const cuuint32_t box[2] = {(cuuint32_t)TC_K, box_rows};
    const cuuint32_t estr[2] = {1, 1};
    // pre-swizzled tensors already hold chunk c of row r at c ^ (r & 7): copy them verbatim
    const CUresult r = fn(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void*>(base), dims, strides, box, estr,
                          CU_TENSOR_MAP_INTERLEAVE_NONE,
                          pre_swizzled ? CU_TENSOR_MAP_SWIZZLE_NONE : CU_TENSOR_MAP_SWIZZLE_128B,
                          CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    return r == CUDA_SUCCESS ? 0 : -3;
}

int tc_encode_rows(CUtensorMap* map, const void* base, uint64_t rows_per_block, uint32_t box_rows) {
    EncodeTiled fn = encode_fn();
    if (!fn) return -1;
    const cuuint64_t dims[3] = {TC_K, rows_per_block, (cuuint64_t)1 << 31};
    const cuuint64_t strides[2] = {TC_K * 2, rows_per_block * TC_K * 2};
    const cuuint32_t box[3] = {(cuuint32_t)TC_K, box_rows, 1}, estr[3] = {1, 1, 1};
    const CUresult r = fn(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, const_cast<void*>(base), dims, strides, box, estr,
                          CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
                          CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    return r == CUDA_SUCCESS ? 0 : -3;
}

int tc_tile_rows(int m) { return m <= 32 ? 32 : (m <= 64 ? 64 : 128); }

cudaError_t launch_tc_gemm(const TcGemm& g, cudaStream_t s, bool pdl) {
    if (g.n_w % TC_M || g.args.k_chunks < 1 || g.splits < 1 || g.args.m < 1) return cudaErrorInvalidValue;
    const int sc = g.args.cluster_reduce > 1 ? g.args.cluster_reduce : 1;
    // one cluster (2 or 4 splits) finishes a tile; accumulated outputs take their splits by atomics
    if (g.args.epilogue == TC_ACCUM ? sc != 1 : g.splits != sc) return cudaErrorInvalidValue;
    if ((sc != 1 && sc != 2 && sc != TC_CLUSTER_SPLITS) ||
        (sc > 1 && g.args.epilogue != TC_QKV && g.args.epilogue != TC_GELU_PACK))
        return cudaErrorInvalidValue;
    switch (g.nt) {
        case 32: return launch_nt<32>(g, s, pdl);
        case 64: return launch_nt<64>(g, s, pdl);
        case 128: return launch_nt<128>(g, s, pdl);
        default: return cudaErrorInvalidValue;
    }
}

}  // namespace mtp

using namespace mtp;

namespace {
// Error words of mtp_gemm_bf16x2's calls in flight: pinned host memory that the kernels reach directly, so
// a call needs no device allocation, memset or copy of its own (with them, 512 rows of W1: 39 us a call,
// 250 when the device was idle in between and the allocator had given its pool back; without: 33).  At
// most ERR_SLOTS calls hold one at a time, each on its own; more at once wait for one to come back.  A word
// is zero while it is free.
constexpr int ERR_SLOTS = 64;
class ErrorWords {
public:
    int take() {  // a free slot, -1 without the memory
        std::unique_lock<std::mutex> lock(mu_);
        if (!words_) {
            void* p = nullptr;
            if (cudaHostAlloc(&p, ERR_SLOTS * sizeof(int), cudaHostAllocMapped | cudaHostAllocPortable) != cudaSuccess) {
                cudaGetLastError();
                return -1;
            }
            std::memset(p, 0, ERR_SLOTS * sizeof(int));
            words_ = static_cast<int*>(p);
        }
        back_.wait(lock, [&] { return free_ != 0; });
        const int slot = __builtin_ctzll(free_);
        free_ &= free_ - 1;
        return slot;
    }
    void give(int slot) {
        std::lock_guard<std::mutex> lock(mu_);
        free_ |= 1ull << slot;
        back_.notify_one();
    }
    volatile int* host(int slot) { return words_ + slot; }
    int* device(int slot) {  // the address of the word on the current device, or null
        void* p = nullptr;
        return cudaHostGetDevicePointer(&p, words_, 0) == cudaSuccess ? static_cast<int*>(p) + slot : nullptr;
    }

private:
    std::mutex mu_;
    std::condition_variable back_;
    unsigned long long free_ = ~0ull;
    int* words_ = nullptr;  // kept until the process exits
};
ErrorWords g_error_words;

int gemm_fail(int code, const char* fmt, int a = 0, int b = 0, int c = 0, int d = 0, int e = 0) {
    char buf[256];
    snprintf(buf, sizeof(buf), fmt, a, b, c, d, e);
    return report_error(code, buf);
}
}  // namespace

extern "C" MTP_API int mtp_gemm_bf16x2(const void* w, const void* a_hi, const void* a_lo, float* out, int n_w, int k,
                                       int m, int splits, int accumulate, void* stream) {
    clear_error();
    if (!w || !a_hi || !a_lo || !out) return gemm_fail(MTP_ERR_INVALID, "mtp_gemm_bf16x2: null pointer");
    if (n_w < TC_M || n_w % TC_M || k < TC_K || k % TC_K || m < 1 || m > 4096 || splits < 1 ||
        (k / TC_K) % splits || (!accumulate && splits != 1))
        return gemm_fail(MTP_ERR_INVALID, "mtp_gemm_bf16x2: n_w=%d k=%d m=%d splits=%d accumulate=%d", n_w, k, m,
                         splits, accumulate);
    TcGemm g;
    std::memset(&g, 0, sizeof(g));
    g.n_w = n_w;
    g.splits = splits;
    g.nt = tc_tile_rows(m);
    g.args.out = out;
    g.args.ldo = n_w;
    g.args.bias = nullptr;
    g.args.m = m;
    g.args.k_chunks = k / TC_K / splits;
    g.args.w_rows_per_kchunk = 0;
    g.args.epilogue = accumulate ? TC_ACCUM : TC_STORE;
    int dev = 0, sms = 0;
    if (cudaGetDevice(&dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess)
        return gemm_fail(MTP_ERR_CUDA, "mtp_gemm_bf16x2: no usable CUDA device");
    const bool pairs = tc_gemm_pair_fits(n_w, m, k / TC_K, splits, sms);  // many rows: tiles of CTA pairs
    if (pairs) {  // whole-K tiles: nothing is added by another CTA
        g.splits = 1;
        g.args.k_chunks = k / TC_K;
    }
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    const int slot = g_error_words.take();
    if (slot < 0 || !(g.args.err = g_error_words.device(slot))) {
        if (slot >= 0) g_error_words.give(slot);
        return gemm_fail(MTP_ERR_CUDA, "mtp_gemm_bf16x2: error word allocation failed");
    }
    int rc = 0;
    if (tc_encode_2d(&g.w, w, (uint64_t)k, (uint64_t)n_w, TC_M, false) ||
        tc_encode_2d(&g.a_hi, a_hi, (uint64_t)k, (uint64_t)m, (uint32_t)g.nt, false) ||
        tc_encode_2d(&g.a_lo, a_lo, (uint64_t)k, (uint64_t)m, (uint32_t)g.nt, false)) {
        rc = gemm_fail(MTP_ERR_INVALID, "mtp_gemm_bf16x2: tensor map encoding failed (alignment?)");
    } else {
        const cudaError_t e = pairs ? launch_tc_gemm_pair(g, sms, st, false) : launch_tc_gemm(g, st, false);
        if (e != cudaSuccess) rc = report_error(MTP_ERR_CUDA, cudaGetErrorString(e));
    }
    const cudaError_t es = cudaStreamSynchronize(st);
    const int err = *g_error_words.host(slot);
    *g_error_words.host(slot) = 0;
    g_error_words.give(slot);
    if (rc) return rc;
    if (es != cudaSuccess) return report_error(MTP_ERR_CUDA, cudaGetErrorString(es));
    if (err) return gemm_fail(MTP_ERR_DEVICE, "mtp_gemm_bf16x2: device error word 0x%x", err);
    return MTP_OK;
}

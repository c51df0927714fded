// tc_gemm_pair.cu -- the batched path's projections over many rows (prefill
// passes): the same product and epilogues as tc_gemm.cu,
//
//   out[n][f] (+)= sum_k (a_hi[n][k] + a_lo[n][k]) * w[f][k],
//
// as a persistent kernel of CTA pairs (tcgen05 cta_group::2).
//
// What bounds it: at 128 x 128 tiles, one CTA each, every 64-wide k-chunk
// moves 48 KB from L2 into shared memory for 512 cycles of MMA (the two
// activation parts make the operand traffic 1.5 times a plain bf16 GEMM's),
// and nothing ran while a CTA wrote its tile out.  A pair of CTAs owns 256
// weight rows x 256 activation rows: each CTA holds its own 128 weight rows
// and half of the activation rows (hi and lo), the MMA reads the other half
// from the peer, so the same 48 KB feed 1024 cycles.  Two accumulators of 256
// TMEM columns let the epilogue warps write one tile out while the next
// one is multiplied.  4096 rows, d = 1024, device time against 128 x 128
// tiles: q|k|v 40 vs 74 us (1.29 PFLOP/s of MMA), W1 with GELU 59 vs 101,
// W_o 22 vs 24, W2 52 vs 81.
//
// Per CTA, 20 warps: warp 0 copies (one lane, TMA into a four-stage ring; both
// CTAs' copies complete on the leader's barrier), warp 1 of the leader issues
// the MMAs (one lane), warps 4 and up read the accumulator back and write it out
// (TMEM lane = weight row f, so a warp's store of one activation row is 32
// consecutive features).  Clusters stride over the tiles, the feature tiles of
// one block of activation rows first: W2's activations of 14592 rows are 239
// MB, and with the rows first they came from memory once per feature tile
// (W_o and W2 86 us on average, now 78; W1 137, now 131).
//
// The tensor core's accumulator truncates at every MMA, so the error of a
// product grows with the K of one accumulation (1024 and 4096: 2.2e-6 and
// 9.2e-6 from 64 bits).  K is therefore accumulated in segments of 512, which
// the epilogue warps add up in fp32 registers while the next one is multiplied
// (64 sums per thread; segments of 256 leave the MMAs waiting for the stores:
// W1 86 us).
#include <cuda.h>

#include <algorithm>

#include "common.cuh"
#include "kernels.cuh"
#include "tc_epilogue.cuh"
#include "tcgen05.cuh"

namespace mtp {
namespace {

constexpr int TP_F = 128;         // weight rows per CTA (the pair's tile has 256)
constexpr int TP_N = 256;         // activation rows per tile
constexpr int TP_K = 64;          // k per stage: one 128-byte swizzle row of bf16
constexpr int TP_STAGES = 4;
constexpr int TP_SEG = 8;         // k-chunks of one accumulation (K = 512)
constexpr int TP_EPI_WARP = 4;    // first epilogue warp (warp % 4 = its TMEM lane quarter)
// epilogue warps: a quarter of the lanes and 64 columns each (their sums stay in registers; GELU's erf
// is a chain of dependent, partly divergent instructions, which four warps per scheduler hide better
// than two)
constexpr int TP_EPI_WARPS = 16;
constexpr int TP_COLS = TP_N / (TP_EPI_WARPS / 4);
constexpr int TP_THREADS = 32 * (TP_EPI_WARP + TP_EPI_WARPS);
constexpr uint32_t TP_W_BYTES = TP_F * TP_K * 2;
constexpr uint32_t TP_A_BYTES = (TP_N / 2) * TP_K * 2;       // one part's half of the activation rows
constexpr uint32_t TP_STAGE = TP_W_BYTES + 2 * TP_A_BYTES;   // 48 KB
constexpr uint32_t TP_SMEM = TP_STAGES * TP_STAGE + 1024;
constexpr uint32_t TP_TMEM = 512;  // two accumulators of 256 columns

__device__ __forceinline__ void tmem_alloc2(uint32_t* dst, uint32_t ncols) {  // one warp of each CTA of the pair
    asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_addr(dst)), "r"(ncols)
                 : "memory");
}
__device__ __forceinline__ void tmem_relinquish2() {
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
}
__device__ __forceinline__ void tmem_dealloc2(uint32_t taddr, uint32_t ncols) {
    asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(taddr), "r"(ncols) : "memory");
}
__device__ __forceinline__ void tc_mma2(uint32_t d_tmem, uint64_t adesc, uint64_t bdesc, uint32_t idesc, uint32_t acc) {
    asm volatile(
        "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::2.kind::f16 [%0], %1, %2, %3, p;\n\t}" ::"r"(d_tmem),
        "l"(adesc), "l"(bdesc), "r"(idesc), "r"(acc)
        : "memory");
}
// Arrive on `bar` (the same shared-memory offset) in both CTAs once every MMA issued so far is done.
__device__ __forceinline__ void tc_commit2(uint64_t* bar) {
    asm volatile(
        "tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.multicast::cluster.b64 [%0], %1;" ::"r"(
            smem_addr(bar)),
        "h"((uint16_t)3)
        : "memory");
}
// 2-D TMA load into this CTA's shared memory; `bar`: a shared::cluster address in either CTA of the pair.
__device__ __forceinline__ void tma_load_2d_pair(void* dst, const CUtensorMap* map, int x, int y, uint32_t bar) {
    asm volatile(
        "cp.async.bulk.tensor.2d.cta_group::2.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, "
        "%3}], [%4];" ::"r"(smem_addr(dst)),
        "l"(reinterpret_cast<uint64_t>(map)), "r"(x), "r"(y), "r"(bar)
        : "memory");
}
__device__ __forceinline__ void mbar_arrive_cluster(uint32_t bar) {  // bar: shared::cluster address
    asm volatile("mbarrier.arrive.release.cluster.shared::cluster.b64 _, [%0];" ::"r"(bar) : "memory");
}
// Bounded wait that also acquires arrivals of the peer CTA.
__device__ __forceinline__ bool mbar_wait_cluster(uint64_t* bar, uint32_t parity, int* err) {
    for (uint32_t i = 0; i < MBAR_MAX_POLLS; ++i) {
        uint32_t done;
        asm volatile(
            "{\n\t.reg .pred p;\n\t"
            "mbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2;\n\t"
            "selp.u32 %0, 1, 0, p;\n\t}"
            : "=r"(done)
            : "r"(smem_addr(bar)), "r"(parity)
            : "memory");
        if (done) return true;
    }
    if (err) atomicOr(err, ERR_WAIT_TIMEOUT);
    return false;
}
__device__ __forceinline__ void epi_barrier() { asm volatile("bar.sync 1, %0;" ::"n"(32 * TP_EPI_WARPS) : "memory"); }

template <int EPI>
__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(TP_THREADS, 1)
    tc_gemm_pair_kernel(const __grid_constant__ CUtensorMap tw, const __grid_constant__ CUtensorMap tah,
                        const __grid_constant__ CUtensorMap tal, const TcGemmArgs a, const int tiles_f,
                        const int tiles_n) {
    extern __shared__ __align__(1024) unsigned char smem_raw[];
    __shared__ uint64_t full[TP_STAGES], empty[TP_STAGES], acc_full[2], acc_empty[2], drained;
    __shared__ uint32_t tmem_base;
    __shared__ int s_staged, s_failed;  // stages filled when a wait of the copies ran out; a wait of the MMAs did
    __shared__ long long s_rowbase[2][TP_N];  // TC_QKV: element offset of the row's key row in its page
                                              // (-1: unreserved page, -2: row of no sequence)
    __shared__ int s_rowt[2][TP_N];           // TC_QKV: key row within the page; TC_GELU_PACK: row of a sequence
    unsigned char* smem = reinterpret_cast<unsigned char*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
    TraceEnd trace_guard(a.trace);
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int rank = blockIdx.x & 1, pair = blockIdx.x >> 1, pairs = gridDim.x >> 1;
    const int tiles = tiles_f * tiles_n;
    const int chunks = a.k_chunks, segs = (chunks + TP_SEG - 1) / TP_SEG;
    const int work = pair < tiles ? (tiles - pair + pairs - 1) / pairs * segs : 0;  // accumulations of this pair

    if (warp == 0) {
        tmem_alloc2(&tmem_base, TP_TMEM);
        tmem_relinquish2();
    }
    if (tid == 32) {
        for (int s = 0; s < TP_STAGES; ++s) {
            mbar_init(&full[s], 1);
            mbar_init(&empty[s], 1);
        }
        for (int b = 0; b < 2; ++b) {
            mbar_init(&acc_full[b], 1);
            mbar_init(&acc_empty[b], 2 * TP_EPI_WARPS);  // the epilogue warps of both CTAs
        }
        mbar_init(&drained, 1);
        fence_barrier_init();
        s_staged = s_failed = 0;
    }
    tc_fence_before();
    __syncthreads();
    cluster_arrive_release();  // the peer's barriers are initialised before anything signals them
    cluster_wait();
    tc_fence_after();
    const uint32_t tmem = tmem_base;

    // tiles in order of the activation tile: the pairs at work at one time share weight tiles
    auto load_w = [&](int tile, int c, int s) {
        const int f0 = (tile % tiles_f) * 2 * TP_F + rank * TP_F;
        const int x = a.w_rows_per_kchunk ? 0 : c * TP_K;
        const int y = a.w_rows_per_kchunk ? c * a.w_rows_per_kchunk + f0 : f0;
        if (rank == 0) mbar_arrive_expect_tx(&full[s], 2 * TP_STAGE);  // both CTAs' copies of the stage
        tma_load_2d_pair(smem + (size_t)s * TP_STAGE, &tw, x, y, dsmem_addr(&full[s], 0));
    };
    auto load_a = [&](int tile, int c, int s) {
        const int n0 = (tile / tiles_f) * TP_N + rank * (TP_N / 2);
        unsigned char* st = smem + (size_t)s * TP_STAGE + TP_W_BYTES;
        const uint32_t bar = dsmem_addr(&full[s], 0);
        tma_load_2d_pair(st, &tah, c * TP_K, n0, bar);
        tma_load_2d_pair(st + TP_A_BYTES, &tal, c * TP_K, n0, bar);
    };
    const int pre = pair < tiles ? min(chunks, TP_STAGES) : 0;
    if (tid == 0)  // weights of the first stages: independent of the previous kernel
        for (int c = 0; c < pre; ++c) load_w(pair, c, c);
    pdl_launch_dependents();
    pdl_wait();
    trace_wait(a.trace);

    if (tid == 0) {  // ---- producer ----
        int it = 0;
        bool ok = true;
        for (int tile = pair; tile < tiles && ok; tile += pairs)
            for (int c = 0; c < chunks; ++c, ++it) {
                const int s = it % TP_STAGES;
                if (it >= pre) {
                    if (it >= TP_STAGES && !mbar_wait_cluster(&empty[s], (uint32_t)(it / TP_STAGES - 1) & 1, a.err)) {
                        ok = false;
                        break;
                    }
                    load_w(tile, c, s);
                }
                load_a(tile, c, s);
            }
        if (!ok) s_staged = it;
    } else if (tid == 32 && rank == 0) {  // ---- MMA issuer (the pair's leader) ----
        constexpr uint32_t IDESC = f16_idesc(2 * TP_F, TP_N, false);
        int it = 0;
        bool ok = true;
        for (int t = 0; t < work && ok; ++t) {
            const int b = t & 1, c0 = t % segs * TP_SEG, c1 = min(chunks, c0 + TP_SEG);
            if (t >= 2 && !mbar_wait_cluster(&acc_empty[b], (uint32_t)(t / 2 - 1) & 1, a.err)) {
                ok = false;
                break;
            }
            tc_fence_after();
            const uint32_t acc = tmem + (uint32_t)b * TP_N;
            for (int c = c0; c < c1; ++c, ++it) {
                const int s = it % TP_STAGES;
                if (!mbar_wait_cluster(&full[s], (uint32_t)(it / TP_STAGES) & 1, a.err)) {
                    ok = false;
                    break;
                }
                tc_fence_after();
                const uint32_t wb = smem_addr(smem + (size_t)s * TP_STAGE);
                const uint32_t hb = wb + TP_W_BYTES, lb = hb + TP_A_BYTES;
#pragma unroll
                for (int kk = 0; kk < TP_K / 16; ++kk) {
                    const uint64_t dw = sw128_desc(wb + kk * 32);
                    tc_mma2(acc, dw, sw128_desc(hb + kk * 32), IDESC, c != c0 || kk != 0);
                    tc_mma2(acc, dw, sw128_desc(lb + kk * 32), IDESC, 1u);
                }
                tc_commit2(&empty[s]);
            }
            if (ok) tc_commit2(&acc_full[b]);
        }
        if (!ok) {  // the MMAs that were issued end before TMEM is freed
            s_failed = 1;
            tc_commit2(&drained);
            mbar_wait_cluster(&drained, 0, nullptr);
        }
    } else if (warp >= TP_EPI_WARP) {  // ---- epilogue ----
        const int et = tid - TP_EPI_WARP * 32, quarter = warp & 3, j0 = ((warp - TP_EPI_WARP) >> 2) * TP_COLS;
        const int P = a.page_size;
        constexpr bool FACTS = EPI == TC_QKV || EPI == TC_GELU_PACK;
        float sum[TP_COLS];
        bool ok = true;
        for (int t = 0; t < work && ok; ++t) {
            const int b = t & 1, seg = t % segs, i = t / segs, tile = pair + i * pairs, fb = i & 1;
            const int row0 = (tile / tiles_f) * TP_N;
            if (FACTS && seg == 0) {  // per-row facts of the tile, one row per thread
                const int n = row0 + et;
                const int seq = et < TP_N && n < a.m ? a.row_seq[n] : -1;
                if (EPI == TC_GELU_PACK) {
                    if (et < TP_N) s_rowt[fb][et] = seq >= 0;
                } else if (et < TP_N) {
                    long long base = -2;
                    int tr = 0;
                    if (seq >= 0) {
                        const int pos = a.row_pos[n];
                        tr = pos % P;
                        const int page = a.block_table[(size_t)seq * a.bt_stride + pos / P];
                        base = page < 0 ? -1 : (long long)page * a.page_elems + a.layer_off + (long long)tr * HEAD_DIM;
                        if (page < 0) atomicOr(a.err, ERR_BOUNDS);
                    }
                    s_rowbase[fb][et] = base;
                    s_rowt[fb][et] = tr;
                }
                epi_barrier();
            }
            const int got_acc = lane == 0 ? mbar_wait_cluster(&acc_full[b], (uint32_t)(t / 2) & 1, a.err) : 1;
            ok = __all_sync(FULL_MASK, got_acc) != 0;
            if (!ok) {  // the row facts' barrier counts every epilogue warp: keep meeting it
                if (FACTS)
                    for (int rest = i + 1; rest < work / segs; ++rest) epi_barrier();
                break;
            }
            tc_fence_after();
            if (seg == 0) {
#pragma unroll
                for (int e = 0; e < TP_COLS; ++e) sum[e] = 0.f;
            }
            const uint32_t src = tmem + ((uint32_t)(quarter * 32) << 16) + (uint32_t)(b * TP_N + j0);
#pragma unroll
            for (int c = 0; c < TP_COLS; c += 16) {
                float v[16];
                tmem_ld16(src + (uint32_t)c, v);
#pragma unroll
                for (int e = 0; e < 16; ++e) sum[c + e] += v[e];
            }
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive_cluster(dsmem_addr(&acc_empty[b], 0));  // the leader may reuse the buffer
            if (seg + 1 < segs) continue;

            const int f = (tile % tiles_f) * 2 * TP_F + rank * TP_F + quarter * 32 + lane;
            const int n0 = row0 + j0, rows = min(TP_COLS, a.m - n0);  // this warp's rows
            if (rows <= 0) continue;
            const float bias = a.bias ? __ldg(a.bias + f) : 0.f;
            tc_epilogue<EPI, false>(a, sum, n0, j0, rows, f, bias, s_rowbase[fb], s_rowt[fb]);
        }
    }
    // nothing signals a CTA that has left, and TMEM is freed once both are done with it
    tc_fence_before();
    __syncthreads();
    // where a wait ran out, both CTAs' copies in flight land before the pair leaves (they complete on the leader).
    // (An epilogue wait runs out only where the issuer's did; a flag of its own cost W1's epilogue 3 %.)
    if ((s_failed || s_staged) && tid == 0 && rank == 0)
        for (int n = s_staged ? s_staged : work / segs * chunks, j = max(0, n - TP_STAGES); j < n; ++j)
            mbar_wait_cluster(&full[j % TP_STAGES], (uint32_t)(j / TP_STAGES) & 1, nullptr);
    cluster_arrive_release();
    cluster_wait();
    tc_fence_after();
    if (warp == 0) tmem_dealloc2(tmem, TP_TMEM);
}

template <int EPI>
cudaError_t launch_epi(const TcGemm& g, int pairs, cudaStream_t s, bool pdl) {
    auto kern = tc_gemm_pair_kernel<EPI>;
    cudaError_t e = ensure_kernel_smem(reinterpret_cast<const void*>(kern), TP_SMEM);
    if (e != cudaSuccess) return e;
    const int tiles_f = g.n_w / (2 * TP_F), tiles_n = (g.args.m + TP_N - 1) / TP_N;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(2 * std::min(pairs, tiles_f * tiles_n));
    cfg.blockDim = dim3(TP_THREADS);
    cfg.dynamicSmemBytes = TP_SMEM;
    cfg.stream = s;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = pdl ? 1 : 0;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kern, g.w, g.a_hi, g.a_lo, g.args, tiles_f, tiles_n);
}

}  // namespace

// This kernel takes about 0.66 us per 64-wide k-chunk and wave of tiles and 7 us around that (filling the
// ring, the last tile's epilogue), tc_gemm.cu 0.6 and under 2: in chunks, 11 and less than 4.  Measured at
// K = 1024, us by waves: here 17.5 / 28.3 / 39.2 / 49.5 for 1-4 waves of 256 x 256 tiles, tc_gemm.cu
// 11.2 / 20.8 / 30.0 / 39.7 for 1-4 waves of 128 x 128, of which there are twice as many where no tile is
// ragged.  So one wave there stays there, and two do where two are needed here.
bool tc_gemm_pair_fits(int n_w, int m, int k_chunks, int splits, int num_sms) {
    if (n_w % (2 * TP_F) || m <= TP_N / 2) return false;
    const int tiles = n_w / (2 * TP_F) * ((m + TP_N - 1) / TP_N), pairs = std::max(1, num_sms / 2);
    const int single = n_w / 128 * ((m + 127) / 128) * splits;
    const int here = (tiles + pairs - 1) / pairs * k_chunks + 11;
    const int there = (single + num_sms - 1) / num_sms * (k_chunks / splits) + 4;
    return here < there;
}

cudaError_t launch_tc_gemm_pair(const TcGemm& g, int num_sms, cudaStream_t s, bool pdl) {
    if (g.n_w % (2 * TP_F) || g.args.k_chunks < 1 || g.args.m < 1 || g.nt != TP_N / 2 || g.args.n_valid ||
        g.splits != 1)
        return cudaErrorInvalidValue;
    const int pairs = std::max(1, num_sms / 2);
    switch (g.args.epilogue) {
        case TC_STORE: return launch_epi<TC_STORE>(g, pairs, s, pdl);
        case TC_ACCUM: return launch_epi<TC_ACCUM>(g, pairs, s, pdl);
        case TC_QKV: return launch_epi<TC_QKV>(g, pairs, s, pdl);
        case TC_GELU_PACK: return launch_epi<TC_GELU_PACK>(g, pairs, s, pdl);
        default: return cudaErrorInvalidValue;
    }
}

}  // namespace mtp

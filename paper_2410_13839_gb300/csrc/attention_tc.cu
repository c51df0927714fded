// attention_tc.cu -- causal attention of prompt rows on the tensor cores
// (tcgen05), the attention of each block during prefill (Sec. III-A: the
// concatenated phoneme + acoustic prompt runs through the blocks as one
// sequence, every position attending to itself and the positions before it).
//
// Grid (split, head, tile).  A tile is 128 rows of the pass, the MMA's M side
// and the 128 TMEM lanes; its rows may belong to several slots (a prefill pass
// packs the prompts of many slots), in any order.  The tile's rows of one slot are
// a segment; the segment's keys 0 .. (its largest position) are cut into items of
// 128 keys, and split s takes items s, s + S, ... of every segment.
// Per item, with the cached keys and values of the item's pages copied by
// cp.async.bulk into a two-stage ring (the cache stores chunk c of key row t
// at c ^ (t & 7): exactly the 128-byte-swizzled tile the MMA reads):
//
//   S  = (Q_hi + Q_lo) K^T       two MMAs per 16 dims, 128 x 128 fp32 in TMEM
//   P  = 2^(S log2 e - m)        one thread per row (TMEM lane), masked to the
//                                segment's rows and keys <= the row's position;
//                                written to TMEM as bf16 hi + lo, 64 keys at a time
//   O += (P_hi + P_lo) V         two MMAs per 16 keys with P read from TMEM,
//                                128 x 64 fp32 in TMEM per 64 keys (V read as an
//                                MN-major operand), added up in registers
//
// m is a row's running maximum; where no row of a warp has a new one, nothing is
// rescaled.  (A reference that may lag behind by up to 2^8 costs no less time but
// 2.80e-6 instead of 2.73e-6 from 64 bits.)
//
// O is accumulated in TMEM over 64 keys only; the row threads add these products
// up in registers, in fp32, and rescale them there.  The tensor core truncates its
// accumulator at every MMA, so a sum over all of a row's keys drifts: with values
// of mean 1, rows of one prompt of 2000 keys are 3.5e-7 from 64 bits, and 1.4e-6
// with one accumulation per row (4.2e-7 with one per 128 keys; mean 0: 2.84e-6,
// 2.92e-6 and 2.87e-6).  It costs no time: the rescaling in TMEM, which reads and
// writes O, was needed for most halves, and goes.
//
// What bounds it: the softmax's instructions, about 8 per score with one warp per
// scheduler and CTA (fp32 additions and multiplications two at a time).  S is
// read into registers at once, so the next item's S = Q K^T runs under this one's
// softmax, P V of each half under the other half's, and two CTAs share an SM (97
// KB of shared memory, 256 TMEM columns each).
// Q and P enter as bf16 hi + lo pairs (hi + lo = x to about 2^-16 relative),
// so the products keep fp32 accuracy; the keys and values are the cache's bf16.
// One elected thread of the fifth warp issues the copies and the MMAs; the
// four other warps own one row each per thread.  Splits leave (maximum, sum,
// unnormalised output) per row in the workspace and the CTA that finishes
// last merges them (an atomic counter per tile and head, reset by that CTA).
#include <float.h>
#include <math.h>

#include <algorithm>

#include "common.cuh"
#include "kernels.cuh"
#include "mtp.h"
#include "tcgen05.cuh"

namespace mtp {
namespace {

constexpr int PA_ROWS = 128;     // query rows per tile: MMA M, TMEM lanes
constexpr int PA_KEYS = 128;     // keys per item: N of Q K^T, K of P V
constexpr int PA_SPLIT_ITEMS = 4;  // fewest items of a key split (a split costs its partials and their merge)
constexpr int PA_THREADS = 160;  // four row warps + the issuing warp
constexpr int PA_PART = 4 + HEAD_DIM;  // (max, sum, -, -, out[64]): out 16-byte aligned for float4 access
constexpr uint32_t PA_TILE = PA_ROWS * 128;  // 128 rows of 128 bytes
// shared memory (1024-byte aligned): Q hi | Q lo | stage 0 K | V | stage 1 K | V
constexpr uint32_t OFF_Q = 0, OFF_KV = 2 * PA_TILE;
constexpr uint32_t PA_SMEM = 6 * PA_TILE + 1024;
constexpr int PA_HALF = PA_KEYS / 2;  // keys whose weights P holds at a time
// TMEM columns: S [128) | P hi [32) | P lo [32) of half an item | O [64)
constexpr uint32_t TM_S = 0, TM_P = 128, TM_PLO = TM_P + PA_HALF / 2, TM_O = 192, TM_COLS = 256;
constexpr float LOG2E = 1.4426950408889634f;

__device__ __forceinline__ float ex2(float x) {
    float y;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}
// Two fp32 operations in one instruction, each rounded on its own.
__device__ __forceinline__ float2 fma2(float2 a, float2 b, float2 c) {
    float2 d;
    asm("{\n\t.reg .b64 a, b, c, d;\n\tmov.b64 a, {%2, %3};\n\tmov.b64 b, {%4, %5};\n\tmov.b64 c, {%6, %7};\n\t"
        "fma.rn.f32x2 d, a, b, c;\n\tmov.b64 {%0, %1}, d;\n\t}"
        : "=f"(d.x), "=f"(d.y)
        : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y), "f"(c.x), "f"(c.y));
    return d;
}
__device__ __forceinline__ float2 add2(float2 a, float2 b) {
    float2 d;
    asm("{\n\t.reg .b64 a, b, d;\n\tmov.b64 a, {%2, %3};\n\tmov.b64 b, {%4, %5};\n\t"
        "add.rn.f32x2 d, a, b;\n\tmov.b64 {%0, %1}, d;\n\t}"
        : "=f"(d.x), "=f"(d.y)
        : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y));
    return d;
}
__device__ __forceinline__ float2 mul2(float2 a, float2 b) {
    float2 d;
    asm("{\n\t.reg .b64 a, b, d;\n\tmov.b64 a, {%2, %3};\n\tmov.b64 b, {%4, %5};\n\t"
        "mul.rn.f32x2 d, a, b;\n\tmov.b64 {%0, %1}, d;\n\t}"
        : "=f"(d.x), "=f"(d.y)
        : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y));
    return d;
}
// D = A B (+ D) with A (bf16, K-major) read from TMEM: lane = row, two K elements per column
__device__ __forceinline__ void tc_mma_ta(uint32_t d_tmem, uint32_t a_tmem, uint64_t bdesc, uint32_t idesc,
                                          uint32_t acc) {
    asm volatile(
        "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], [%1], %2, %3, p;\n\t}" ::"r"(d_tmem),
        "r"(a_tmem), "l"(bdesc), "r"(idesc), "r"(acc)
        : "memory");
}
// 16 consecutive 32-bit columns of this warp's 32 TMEM lanes (thread i: lane i)
__device__ __forceinline__ void tmem_st16(uint32_t taddr, const uint32_t (&r)[16]) {
    asm volatile(
        "tcgen05.st.sync.aligned.32x32b.x16.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, "
        "%15, %16};" ::"r"(taddr),
        "r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7]), "r"(r[8]), "r"(r[9]),
        "r"(r[10]), "r"(r[11]), "r"(r[12]), "r"(r[13]), "r"(r[14]), "r"(r[15])
        : "memory");
}
__device__ __forceinline__ void tmem_st_wait() { asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory"); }
// (x0, x1) as one register of bf16 hi parts and one of bf16 lo parts (x0 in the low half)
__device__ __forceinline__ void split_pair(float x0, float x1, uint32_t& hi, uint32_t& lo) {
    const __nv_bfloat162 h = __floats2bfloat162_rn(x0, x1);
    hi = *reinterpret_cast<const uint32_t*>(&h);
    const float2 r = add2(make_float2(x0, x1), make_float2(-bf16_lo(hi), -bf16_hi(hi)));
    const __nv_bfloat162 l = __floats2bfloat162_rn(r.x, r.y);
    lo = *reinterpret_cast<const uint32_t*>(&l);
}

__device__ __forceinline__ void mbar_arrive(uint64_t* bar) {
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_addr(bar)) : "memory");
}

struct TileRows {
    int seq[PA_ROWS];                  // the rows' slots
    int slot[PA_ROWS], kmax[PA_ROWS];  // segments: the tile's rows of one slot, the keys they see
    int count[PA_ROWS / 32];           // run starts per warp
    int number[PA_ROWS];               // a slot's first run -> its segment
};

// Runs 0 .. nseg - 1 joined to a segment per slot, in order of the slots' first runs; leaves the number of
// segments in rows.count[0] and every row's in rows.seq (my_seg: the run of this thread's row, < 0: none).  The
// whole block calls it.  (Not inlined, and nothing returned in registers: inlined it costs the softmax 8 %.)
__device__ __noinline__ void join_runs(TileRows& rows, int nseg, int my_seg) {
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, runs = nseg;
    int slot = -1, kmax = 0, first = 0;
    if (tid < runs) {
        slot = rows.slot[tid];
        kmax = rows.kmax[tid];
        while (rows.slot[first] != slot) ++first;
    }
    const bool own = tid < runs && first == tid;
    const unsigned owners = __ballot_sync(FULL_MASK, own);
    if (tid < PA_ROWS) {
        rows.seq[tid] = first;  // a run's first run of the same slot
        if (lane == 0) rows.count[warp] = __popc(owners);
    }
    __syncthreads();
    int number = __popc(owners & ((1u << lane) - 1));
    nseg = 0;
    for (int w = 0; w < PA_ROWS / 32; ++w) {
        if (w == warp) number += nseg;
        nseg += rows.count[w];
    }
    if (own) {
        rows.number[tid] = number;
        rows.slot[number] = slot;
    }
    if (tid < PA_ROWS) rows.kmax[tid] = 0;
    __syncthreads();
    if (tid < runs) atomicMax(&rows.kmax[rows.number[first]], kmax);
    if (my_seg >= 0) my_seg = rows.number[rows.seq[my_seg]];
    __syncthreads();
    if (tid < PA_ROWS) rows.seq[tid] = my_seg;
    if (tid == 0) rows.count[0] = nseg;
    __syncthreads();
}

__global__ void __launch_bounds__(PA_THREADS, 2) attn_tc_kernel(const AttnArgs a) {
    extern __shared__ __align__(1024) unsigned char pa_raw[];
    __shared__ uint64_t kv_full[2], s_full, s_read, p_full[2], pv_done[2];  // p, pv: the item's halves
    __shared__ uint32_t tmem_base;
    __shared__ TileRows rows;
    __shared__ int s_abort, s_last;
    unsigned char* sm = reinterpret_cast<unsigned char*>((reinterpret_cast<uintptr_t>(pa_raw) + 1023) & ~(uintptr_t)1023);
    TraceEnd trace_guard(a.trace);
    const int sp = blockIdx.x, h = blockIdx.y, tile = blockIdx.z;
    const int S = a.n_splits, H = a.n_heads, P = a.page_size;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int row0 = tile * PA_ROWS;

    // ---- independent of the previous kernel ----
    if (warp == 4) {
        tmem_alloc(&tmem_base, TM_COLS);
        tmem_relinquish();
    }
    if (tid == 0) {
        mbar_init(&kv_full[0], 1);
        mbar_init(&kv_full[1], 1);
        mbar_init(&s_full, 1);
        mbar_init(&s_read, PA_ROWS / 32);  // one arrival per row warp
        for (int i = 0; i < 2; ++i) {
            mbar_init(&p_full[i], PA_ROWS / 32);
            mbar_init(&pv_done[i], 1);
        }
        fence_barrier_init();
        s_abort = 0;
    }
    // values past a segment's pages enter with weight zero: keep them finite (scores of such keys are
    // masked by selection)
    for (int st = 0; st < 2; ++st) {
        uint4* v = reinterpret_cast<uint4*>(sm + OFF_KV + (uint32_t)(2 * st + 1) * PA_TILE);
        for (int i = tid; i < (int)(PA_TILE / 16); i += PA_THREADS) v[i] = make_uint4(0u, 0u, 0u, 0u);
    }
    fence_proxy_async();
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = tmem_base;
    pdl_launch_dependents();
    pdl_wait();
    trace_wait(a.trace);

    // Q of this head, 16 lanes per row: on its way while the rows' runs are found
    constexpr int PER = 32 * (HEAD_DIM / 4) / 32;
    float4 x[PER];
    if (tid < PA_ROWS) {
#pragma unroll
        for (int u = 0; u < PER; ++u) {  // (rows past the pass read its last one)
            const int r = min(row0 + warp * 32 + u * 2 + (lane >> 4), a.rows - 1);
            x[u] = *reinterpret_cast<const float4*>(a.q + (size_t)r * a.ldq + h * HEAD_DIM + (lane & 15) * 4);
        }
    }

    // ---- the tile's rows and their runs ----
    int my_seq = -1, my_pos = -1;
    if (tid < PA_ROWS) {
        const int r = row0 + tid;
        if (r < a.rows) {  // one round of independent loads
            my_seq = a.row_seq[r];
            my_pos = a.row_pos[r];
        }
        rows.seq[tid] = my_seq;
        rows.kmax[tid] = 0;
    }
    __syncthreads();
    bool head = false;
    unsigned heads = 0, live = 0;  // the warp's rows that start a run, and those of a sequence
    if (tid < PA_ROWS) {
        live = __ballot_sync(FULL_MASK, my_seq >= 0);
        head = my_seq >= 0 && (tid == 0 || rows.seq[tid - 1] != my_seq);
        heads = __ballot_sync(FULL_MASK, head);
        if (lane == 0) rows.count[warp] = __popc(heads);
    }
    __syncthreads();
    int nseg = 0, my_seg = -1;
#pragma unroll
    for (int w = 0; w < PA_ROWS / 32; ++w) {
        if (w == warp) my_seg = nseg + __popc(heads & (0xffffffffu >> (31 - lane))) - 1;  // run of this row
        nseg += rows.count[w];
    }
    if (tid < PA_ROWS && my_seq >= 0) {
        if (head) rows.slot[my_seg] = my_seq;
        atomicMax(&rows.kmax[my_seg], my_pos + 1);
    }
    __syncthreads();
    // a slot whose rows lie in several runs is one segment (runs of ascending slots, as packed prompts are, need
    // no look)
    if (nseg > 1 && __syncthreads_or(tid > 0 && tid < nseg && rows.slot[tid] <= rows.slot[tid - 1])) {
        join_runs(rows, nseg, my_seg);
        nseg = rows.count[0];
        if (tid < PA_ROWS) my_seg = rows.seq[tid];
    }
    // this split's items in order: segment g, key tiles j = sp, sp + S, ... below the segment's end
    auto skip_empty = [&](int2 t) {
        while (t.x < nseg && t.y * PA_KEYS >= rows.kmax[t.x]) {
            ++t.x;
            t.y = sp;
        }
        return t;
    };
    auto next_item = [&](int2 t) {
        t.y += S;
        return skip_empty(t);
    };
    const int2 first = skip_empty(make_int2(0, sp));

    float m_run = -INFINITY, l_run = 0.f;  // m_run in log2 units
    float o[HEAD_DIM];  // this row's unnormalised output, without the last half's product
#pragma unroll
    for (int c = 0; c < HEAD_DIM; ++c) o[c] = 0.f;
    // adds the last half's product (complete) to it
    auto add_product = [&]() {
#pragma unroll
        for (int c0 = 0; c0 < HEAD_DIM; c0 += 16) {
            float v[16];
            tmem_ld16(tmem + ((uint32_t)(warp * 32) << 16) + TM_O + c0, v);
#pragma unroll
            for (int e = 0; e < 16; e += 2) {
                const float2 y = add2(make_float2(o[c0 + e], o[c0 + e + 1]), make_float2(v[e], v[e + 1]));
                o[c0 + e] = y.x;
                o[c0 + e + 1] = y.y;
            }
        }
    };
    bool seen = false;  // a row of the warp sees keys of the last half
    int items = 0;
    bool fine = true;
    if (warp == 4) {  // ---- the issuing warp: copies (a lane per page) and MMAs (lane 0) ----
        constexpr uint32_t IDESC_S = f16_idesc(PA_ROWS, PA_KEYS, false);
        constexpr uint32_t IDESC_O = f16_idesc(PA_ROWS, HEAD_DIM, true);
        const uint32_t q_hi = smem_addr(sm + OFF_Q), q_lo = q_hi + PA_TILE;
        const long long kv_head = (long long)h * P * HEAD_DIM, v_off = (long long)H * P * HEAD_DIM;
        // lane q: page q of the item (-2: none; -1: unreserved, as are pages past the slot's table row)
        auto item_page = [&](int2 t) {
            if (t.x >= nseg) return -2;
            const int p = t.y * (PA_KEYS / P) + lane;
            if (lane >= PA_KEYS / P || p * P >= rows.kmax[t.x]) return -2;
            return p < a.bt_stride ? max(-1, a.block_table[(size_t)rows.slot[t.x] * a.bt_stride + p]) : -1;
        };
        // copies of item i into stage i & 1
        auto stage_item = [&](int i, int page) {
            const uint32_t blk = (uint32_t)P * 128;
            uint64_t* bar = &kv_full[i & 1];
            unsigned char* ks = sm + OFF_KV + (uint32_t)(i & 1) * 2 * PA_TILE + (uint32_t)(lane * P) * 128;
            const unsigned have = __ballot_sync(FULL_MASK, page >= 0);
            if (lane == 0) mbar_arrive_expect_tx(bar, 2 * blk * __popc(have));
            __syncwarp();
            if (page >= 0) {
                const __nv_bfloat16* base = a.kv_pool + (long long)page * a.page_elems + a.layer_off + kv_head;
                bulk_copy_g2s(ks, base, blk, bar);
                bulk_copy_g2s(ks + PA_TILE, base + v_off, blk, bar);
            } else if (page == -1 && a.err) {  // unreserved page: report, never read
                atomicOr(a.err, ERR_BOUNDS);
            }
        };
        auto wait = [&](uint64_t* bar, uint32_t parity) {  // one lane polls
            return __all_sync(FULL_MASK, lane != 0 || mbar_wait(bar, parity, a.err)) != 0;
        };
        int staged = 0;  // items staged so far
        int2 ahead = first;
        {
            const int p0 = item_page(ahead);
            const bool any0 = ahead.x < nseg;
            ahead = any0 ? next_item(ahead) : ahead;
            const int p1 = item_page(ahead);
            if (any0) stage_item(staged++, p0);
            if (ahead.x < nseg) {
                stage_item(staged++, p1);
                ahead = next_item(ahead);
            }
        }
        int ahead_page = item_page(ahead);
        asm volatile("bar.sync 1, %0;" ::"n"(PA_THREADS) : "memory");  // Q is in shared memory
        bool ok = true;
        auto issue_s = [&](int i) {  // S of item i, once its keys are in
            ok = wait(&kv_full[i & 1], (uint32_t)(i >> 1) & 1);
            if (!ok) return;
            tc_fence_after();
            if (lane == 0) {
                const uint32_t kb = smem_addr(sm + OFF_KV + (uint32_t)(i & 1) * 2 * PA_TILE);
#pragma unroll
                for (int kk = 0; kk < HEAD_DIM / 16; ++kk) {
                    const uint64_t bk = sw128_desc(kb + kk * 32);
                    tc_mma(tmem + TM_S, sw128_desc(q_hi + kk * 32), bk, IDESC_S, kk != 0);
                    tc_mma(tmem + TM_S, sw128_desc(q_lo + kk * 32), bk, IDESC_S, 1u);
                }
                tc_commit(&s_full);
            }
            __syncwarp();
        };
        int i = 0, s_issued = 0, pv_issued = 0;
        if (staged > 0) {
            issue_s(0);
            s_issued = ok;
        }
        for (int2 t = first; ok && t.x < nseg; ++i) {
            const int keys = rows.kmax[t.x] - t.y * PA_KEYS;  // of the item that some row of the tile sees
            t = next_item(t);
            const uint32_t vb = smem_addr(sm + OFF_KV + (uint32_t)(2 * (i & 1) + 1) * PA_TILE);
#pragma unroll
            for (int half = 0; half < 2; ++half) {
                if (half) {  // S is in the rows' registers: the next item's overwrites it
                    ok = wait(&s_read, (uint32_t)i & 1);
                    if (!ok) break;
                    if (t.x < nseg) {
                        issue_s(i + 1);
                        if (!ok) break;
                        ++s_issued;
                    }
                }
                ok = wait(&p_full[half], (uint32_t)i & 1);
                if (!ok) break;
                tc_fence_after();
                if (lane == 0 && half * PA_HALF < keys) {
#pragma unroll
                    for (int kk = 0; kk < PA_HALF / 16; ++kk) {
                        const uint64_t bv = sw128_mn_desc(vb + (half * (PA_HALF / 16) + kk) * 2048);
                        tc_mma_ta(tmem + TM_O, tmem + TM_P + kk * 8, bv, IDESC_O, kk != 0);
                        tc_mma_ta(tmem + TM_O, tmem + TM_PLO + kk * 8, bv, IDESC_O, 1u);
                    }
                }
                if (lane == 0) tc_commit(&pv_done[half]);
                __syncwarp();
                ++pv_issued;
            }
            if (!ok) break;
            if (ahead.x < nseg) {  // this item's stage is free once its MMAs have read it
                ok = wait(&pv_done[1], (uint32_t)i & 1);
                if (!ok) break;
                stage_item(staged++, ahead_page);
                ahead = next_item(ahead);
                ahead_page = item_page(ahead);
            }
        }
        if (!ok && lane == 0) {
            s_abort = 1;
            // copies still in flight land, and issued MMAs end (bounded), before the CTA leaves
            for (int j = s_issued; j < staged; ++j) mbar_wait(&kv_full[j & 1], (uint32_t)(j >> 1) & 1, nullptr);
            const int half = pv_issued & 1;  // the next commit to come on this barrier follows every MMA
            tc_commit(&pv_done[half]);
            mbar_wait(&pv_done[half], (uint32_t)(pv_issued >> 1) & 1, nullptr);
        }
        __syncwarp();
    } else {  // ---- one row per thread: Q, then softmax ----
        {
            // Q: rows pre-scaled by 1/sqrt(64), zero without a sequence, bf16 hi | lo, swizzled
#pragma unroll
            for (int u = 0; u < PER; ++u) {
                const int q = warp * 32 + u * 2 + (lane >> 4), c4 = lane & 15;
                if (!(live >> (q & 31) & 1)) x[u] = make_float4(0.f, 0.f, 0.f, 0.f);
                uint2 hi, lo;
                split_pair(x[u].x * 0.125f, x[u].y * 0.125f, hi.x, lo.x);
                split_pair(x[u].z * 0.125f, x[u].w * 0.125f, hi.y, lo.y);
                unsigned char* at = sm + OFF_Q + q * 128 + (((c4 >> 1) ^ (q & 7)) << 4) + (c4 & 1) * 8;
                *reinterpret_cast<uint2*>(at) = hi;
                *reinterpret_cast<uint2*>(at + PA_TILE) = lo;
            }
        }
        fence_proxy_async();  // Q is read by the tensor cores
        asm volatile("bar.sync 1, %0;" ::"n"(PA_THREADS) : "memory");
        const uint32_t base = tmem + ((uint32_t)(warp * 32) << 16);
        for (int2 t = first; t.x < nseg; t = next_item(t), ++items) {
            // keys of the item this row sees: columns 0 .. lim
            const int lim = my_seq >= 0 && t.x == my_seg ? my_pos - t.y * PA_KEYS : -1;
            // one lane polls (a poll costs every polling thread); tcgen05.ld is issued by whole warps
            if (!__all_sync(FULL_MASK, lane != 0 || mbar_wait(&s_full, (uint32_t)items & 1, a.err))) {
                s_abort = 1;
                fine = false;
                break;
            }
            tc_fence_after();
            // two halves of 64 keys, each with its own look at the maximum; a half of which no row of the
            // warp sees a key (another run's rows, keys past every row) has weight zero without any work
            bool done = true;
#pragma unroll 1
            for (int half = 0; half < 2; ++half) {
                const int hl = lim - half * PA_HALF;  // columns 0 .. hl of this half
                const bool need = __any_sync(FULL_MASK, hl >= 0) != 0;
                uint32_t hi[PA_HALF / 2], lo[PA_HALF / 2];
                float corr = 1.f;
                bool move = false;
                if (need) {
                    float sv[PA_HALF];
                    tmem_ld_issue<32>(base + TM_S + half * PA_HALF, *reinterpret_cast<float(*)[32]>(&sv[0]));
                    tmem_ld_issue<32>(base + TM_S + half * PA_HALF + 32, *reinterpret_cast<float(*)[32]>(&sv[32]));
                    tmem_ld_wait();
                    tmem_ld_done(*reinterpret_cast<float(*)[32]>(&sv[0]));
                    tmem_ld_done(*reinterpret_cast<float(*)[32]>(&sv[32]));
                    if (half) {
                        tc_fence_before();
                        __syncwarp();
                        if (lane == 0) mbar_arrive(&s_read);
                    }
                    if (!__all_sync(FULL_MASK, hl >= PA_HALF - 1)) {
#pragma unroll
                        for (int c = 0; c < PA_HALF; ++c) sv[c] = c <= hl ? sv[c] : -INFINITY;
                    }
                    float mx[4] = {-INFINITY, -INFINITY, -INFINITY, -INFINITY};
#pragma unroll
                    for (int c = 0; c < PA_HALF; ++c) mx[c & 3] = fmaxf(mx[c & 3], sv[c]);
                    const float top = fmaxf(fmaxf(mx[0], mx[1]), fmaxf(mx[2], mx[3])) * LOG2E;
                    // a row's first keys set its maximum; a later one above it moves it
                    const bool fresh = m_run == -INFINITY;
                    move = !fresh && top > m_run;
                    if (move) corr = ex2(m_run - top);
                    if (fresh || move) m_run = top;
                    const float ref = m_run == -INFINITY ? 0.f : m_run;  // a row that has seen no key: every weight 0
                    float2 sum[2] = {{0.f, 0.f}, {0.f, 0.f}};
#pragma unroll
                    for (int e = 0; e < PA_HALF / 2; ++e) {
                        const float2 x = fma2(make_float2(sv[2 * e], sv[2 * e + 1]), make_float2(LOG2E, LOG2E),
                                              make_float2(-ref, -ref));
                        const float2 p = make_float2(ex2(x.x), ex2(x.y));
                        sum[e & 1] = add2(sum[e & 1], p);
                        split_pair(p.x, p.y, hi[e], lo[e]);
                    }
                    l_run = fmaf(l_run, corr, (sum[0].x + sum[0].y) + (sum[1].x + sum[1].y));
                } else {
                    if (half) {
                        __syncwarp();
                        if (lane == 0) mbar_arrive(&s_read);
                    }
#pragma unroll
                    for (int e = 0; e < PA_HALF / 2; ++e) hi[e] = lo[e] = 0u;
                }
                // the previous half's weights have been read, and its product is complete
                if (half || items > 0)
                    done = __all_sync(FULL_MASK, lane != 0 || mbar_wait(&pv_done[half ^ 1],
                                                                        (uint32_t)(half ? items : items - 1) & 1, a.err));
                if (!done) break;
                tc_fence_after();
                if (seen) add_product();  // the next product overwrites it
                if (__any_sync(FULL_MASK, move)) {
#pragma unroll
                    for (int c = 0; c < HEAD_DIM; ++c) o[c] *= corr;
                }
                seen = need;
#pragma unroll
                for (int q = 0; q < PA_HALF / 2; q += 16) {
                    tmem_st16(base + TM_P + q, *reinterpret_cast<const uint32_t(*)[16]>(&hi[q]));
                    tmem_st16(base + TM_PLO + q, *reinterpret_cast<const uint32_t(*)[16]>(&lo[q]));
                }
                tmem_st_wait();
                tc_fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive(&p_full[half]);
            }
            if (!done) {
                s_abort = 1;
                fine = false;
                break;
            }
        }
    }
    if (tid < PA_ROWS && items > 0 && fine) {
        if (__all_sync(FULL_MASK, lane != 0 || mbar_wait(&pv_done[1], (uint32_t)(items - 1) & 1, a.err))) {
            tc_fence_after();
            if (seen) add_product();
        } else {
            s_abort = 1;
        }
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 4) tmem_dealloc(tmem, TM_COLS);
    if (s_abort) return;  // error word set

    // ---- results: rows of this tile, through shared memory (Q's space is free), 16 lanes per row ----
    const int r = row0 + tid;
    float4* ost = reinterpret_cast<float4*>(sm + OFF_Q);  // [128][16], chunk c of row q at c ^ (q & 15)
    // v / sum: the product with the reciprocal, corrected by its remainder (q + r (v - q sum); 64 divisions
    // are 2 us of instructions that every tile fetches and runs once).  An infinite q has no remainder: any
    // finite value leaves it as it is.
    auto stage_row = [&](const float* v, float sum) {
        const float r = 1.f / sum;
        auto quotients = [&](const float* x) {
            const float2 y = make_float2(x[0], x[1]), r2 = make_float2(r, r);
            const float2 q = mul2(y, r2), rem = fma2(q, make_float2(-sum, -sum), y);
            return fma2(make_float2(fmaxf(rem.x, -FLT_MAX), fmaxf(rem.y, -FLT_MAX)), r2, q);
        };
#pragma unroll
        for (int c = 0; c < HEAD_DIM / 4; ++c) {
            const float2 a0 = quotients(v + 4 * c), a1 = quotients(v + 4 * c + 2);
            ost[tid * 16 + (c ^ (tid & 15))] = make_float4(a0.x, a0.y, a1.x, a1.y);
        }
    };
    auto write_rows = [&]() {  // every warp writes the rows its own threads staged, 8 lanes and dims each
        __syncwarp();
        float4 y[16];
#pragma unroll
        for (int u = 0; u < 8; ++u) {
            const int q = warp * 32 + u * 4 + (lane >> 3);
            const bool on = live >> (q & 31) & 1;
#pragma unroll
            for (int e = 0; e < 2; ++e) {
                const int c4 = 2 * (lane & 7) + e;
                y[2 * u + e] = ost[q * 16 + (c4 ^ (q & 15))];
                if (!on) y[2 * u + e] = make_float4(0.f, 0.f, 0.f, 0.f);
            }
        }
        const int c = h * HEAD_DIM + (lane & 7) * 8, q0 = warp * 32 + (lane >> 3);
        if (a.out) {
#pragma unroll
            for (int u = 0; u < 8; ++u)
                if (live >> ((q0 + u * 4) & 31) & 1) {
                    float4* o = reinterpret_cast<float4*>(a.out + (size_t)(row0 + q0 + u * 4) * a.ldo + c);
                    o[0] = y[2 * u];
                    o[1] = y[2 * u + 1];
                }
        }
        if (a.out_hi) {
#pragma unroll
            for (int u = 0; u < 8; ++u) {
                if (row0 + q0 + u * 4 >= a.rows) continue;
                uint4 hi, lo;
                split_pair(y[2 * u].x, y[2 * u].y, hi.x, lo.x);
                split_pair(y[2 * u].z, y[2 * u].w, hi.y, lo.y);
                split_pair(y[2 * u + 1].x, y[2 * u + 1].y, hi.z, lo.z);
                split_pair(y[2 * u + 1].z, y[2 * u + 1].w, hi.w, lo.w);
                const size_t at = (size_t)(row0 + q0 + u * 4) * a.ldb + c;
                *reinterpret_cast<uint4*>(a.out_hi + at) = hi;
                *reinterpret_cast<uint4*>(a.out_lo + at) = lo;
            }
        }
    };
    const bool active = tid < PA_ROWS && r < a.rows && my_seq >= 0;
    if (S == 1) {
        if (tid >= PA_ROWS) return;
        if (active) stage_row(o, l_run);
        write_rows();
        return;
    }
    float* part = a.ws_part + (((size_t)(tile * H + h) * S + sp) * PA_ROWS) * PA_PART;
    if (tid < PA_ROWS) {
        float* pj = part + (size_t)tid * PA_PART;
        pj[0] = m_run;
        pj[1] = l_run;
#pragma unroll
        for (int c = 0; c < HEAD_DIM; c += 4)
            *reinterpret_cast<float4*>(pj + 4 + c) = make_float4(o[c], o[c + 1], o[c + 2], o[c + 3]);
    }
    __threadfence();
    __syncthreads();
    if (tid == 0) s_last = atomicAdd(a.ws_count + tile * H + h, 1) == S - 1;
    __syncthreads();
    if (!s_last) return;
    __threadfence();
    if (tid == 0) a.ws_count[tile * H + h] = 0;
    if (tid >= PA_ROWS) return;
    if (active) {
        // merge the splits in split order: M = max m_s, L = sum 2^(m_s - M) l_s, out = sum 2^(m_s - M) o_s / L
        const float* base = a.ws_part + ((size_t)(tile * H + h) * S * PA_ROWS + tid) * PA_PART;
        const size_t sstride = (size_t)PA_ROWS * PA_PART;
        float M = -INFINITY;
        for (int s = 0; s < S; ++s) M = fmaxf(M, __ldcg(base + s * sstride));
        float L = 0.f;
#pragma unroll
        for (int c = 0; c < HEAD_DIM; ++c) o[c] = 0.f;
        for (int s = 0; s < S; ++s) {
            const float* ps = base + s * sstride;
            const float ms = __ldcg(ps);
            const float w = ms == -INFINITY ? 0.f : ex2(ms - M);
            L = fmaf(w, __ldcg(ps + 1), L);
#pragma unroll
            for (int c = 0; c < HEAD_DIM; c += 4) {
                const float4 v = __ldcg(reinterpret_cast<const float4*>(ps + 4 + c));
                o[c] = fmaf(w, v.x, o[c]);
                o[c + 1] = fmaf(w, v.y, o[c + 1]);
                o[c + 2] = fmaf(w, v.z, o[c + 2]);
                o[c + 3] = fmaf(w, v.w, o[c + 3]);
            }
        }
        stage_row(o, L);
    }
    write_rows();
}

}  // namespace

size_t attn_tc_workspace_floats(int tiles, int n_heads, int n_splits) {
    return (size_t)tiles * n_heads * n_splits * PA_ROWS * PA_PART;
}

int attn_tc_tiles(int rows) { return (rows + PA_ROWS - 1) / PA_ROWS; }

int attn_tc_splits_for(int tiles, int n_heads, int max_keys, int num_sms) {
    const int key_tiles = (max_keys + PA_KEYS - 1) / PA_KEYS;
    int s = num_sms / std::max(1, tiles * n_heads);
    return std::max(1, std::min(s, key_tiles / PA_SPLIT_ITEMS));
}

cudaError_t launch_attention_tc(const AttnArgs& a, cudaStream_t s, bool pdl) {
    if (a.rows < 1 || a.n_splits < 1 || a.n_splits > 0xffff || (a.page_size & 7) ||
        PA_KEYS % a.page_size || (a.ldq & 3) || (a.out && (a.ldo & 3)) || (a.out_hi && (a.ldb & 7)) ||
        (reinterpret_cast<uintptr_t>(a.q) & 15))
        return cudaErrorInvalidValue;
    cudaError_t e = ensure_kernel_smem(reinterpret_cast<const void*>(attn_tc_kernel), PA_SMEM);
    if (e != cudaSuccess) return e;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(a.n_splits, a.n_heads, attn_tc_tiles(a.rows));
    cfg.blockDim = dim3(PA_THREADS);
    cfg.dynamicSmemBytes = PA_SMEM;
    cfg.stream = s;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = pdl ? 1 : 0;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, attn_tc_kernel, a);
}

}  // namespace mtp

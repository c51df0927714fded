// attention.cu -- causal attention of the fed rows over the paged bf16 KV cache
// (the attention of each block, Sec. III-A), split along the key axis.
//
// A group is the rows of one slot (the n tokens fed this step, or 8
// consecutive positions of a prefill chunk).  Each head's work is the stream of
// every group's cached keys, in batches of 64 (one page of 128): grid (J, H),
// CTA j of head h takes batches [j T / J, (j + 1) T / J) of the T, whatever
// groups they belong to.  With J chosen for one wave (four CTAs per SM), all
// CTAs do the same work whether the contexts are ragged or not, and a CTA's
// fixed costs (plan, first copies, merges: about 5 us) are paid once per wave.
// Splitting every group's keys in the same number of parts left the longest
// contexts to set the time (one part) or paid those costs over and over (three
// parts, 2.5 waves).  32 slots of 180-2000 keys, 16 heads: 35 vs 51 us alone (one
// part), and per launch of a decode step at about 450 keys 18.6 vs 29 us (32
// slots, three parts) and 45 vs 57 us (128 slots, one part).
//
// A CTA finds its first group by a scan over the groups' batch counts, and then
// walks the stream: warp 0 keeps the next batches of keys and values on their
// way into a ring of three shared-memory slots with cp.async.bulk (a lane per
// page; plain pools, the stand-alone operator's, with tensor copies that
// swizzle the rows like the cache: at their plain 128-byte pitch every ldmatrix
// of eight rows was an 8-way bank conflict, 86 vs 51 us for 32 slots of about
// 1,100 keys).  Each warp takes 16-key tiles on the tensor cores (mma.sync)
// with the keys as the M side: S^T = K Q^T and O^T += V^T P^T, the fed rows' Q
// and P entering as bf16 hi + lo pairs (two N = 8 operands), which keeps them
// to fp32 accuracy, and its online-softmax state in registers; the warps'
// states are merged in shared memory at the end of the group.  A group that
// several CTAs share leaves partial results (max, sum, unnormalised output) in
// the workspace, and the CTA that finishes last (an atomic counter of the
// group's first CTA and head, reset by that CTA) merges them in stream order, so
// no second kernel is needed.
//
// Under programmatic dependent launch the plan and the first batches that hold
// only keys cached by earlier steps are fetched before griddepcontrol.wait.
#include <math.h>

#include <cstdio>

#include "common.cuh"
#include "kernels.cuh"
#include "mtp.h"

namespace mtp {
namespace {

constexpr int ATT_THREADS = 128;  // four warps: four CTAs per SM
constexpr int ATT_STAGES = 3;    // staging slots of the key/value ring (three 64-key slots keep ~48 KB in flight)
constexpr int RPG = MAX_ROWS;    // rows per group, upper bound
constexpr int PART = 2 + HEAD_DIM;  // (max, sum, out[64]) per row and split
constexpr float LOG2E = 1.4426950408889634f;
constexpr int NW = ATT_THREADS / 32;
constexpr int MROWS = 4;         // rows whose warp states are merged at a time (one per warp)
static_assert(HEAD_DIM == 64, "score scale 0.125 assumes 64-wide heads");



// keys per staging half: 64, or a whole page when pages are longer
__host__ __device__ constexpr int half_keys(int page_size) { return page_size > 64 ? page_size : 64; }

__device__ __forceinline__ float ex2(float x) {
    float y;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}
__device__ __forceinline__ void ldsm_x4(uint32_t (&r)[4], uint32_t addr) {
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0, %1, %2, %3}, [%4];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
                 : "r"(addr));
}
__device__ __forceinline__ void ldsm_x4_t(uint32_t (&r)[4], uint32_t addr) {
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0, %1, %2, %3}, [%4];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
                 : "r"(addr));
}
__device__ __forceinline__ void mma_bf16(float (&d)[4], const uint32_t (&a)[4], const uint32_t (&b)[2]) {
    asm volatile(
        "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, "
        "{%0, %1, %2, %3};"
        : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
        : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b[0]), "r"(b[1]));
}
// The transpose of the 8 x 8 b16 matrix whose row lane / 4, columns 2 (lane % 4) and + 1, this
// lane holds in r: returns the same elements of the transposed matrix.
__device__ __forceinline__ uint32_t movmatrix_trans(uint32_t r) {
    uint32_t d;
    asm volatile("movmatrix.sync.aligned.m8n8.trans.b16 %0, %1;" : "=r"(d) : "r"(r));
    return d;
}
// x0, x1 as bf16 pairs hi + lo (hi + lo = x to about 2^-16 relative; low halves hold x0)
__device__ __forceinline__ void split2(float x0, float x1, uint32_t& hi, uint32_t& lo) {
    const __nv_bfloat162 h = __floats2bfloat162_rn(x0, x1);
    hi = *reinterpret_cast<const uint32_t*>(&h);
    const __nv_bfloat162 l = __floats2bfloat162_rn(x0 - bf16_lo(hi), x1 - bf16_hi(hi));
    lo = *reinterpret_cast<const uint32_t*>(&l);
}

// PLAIN: the pool holds plain rows; a tensor copy with the 128-byte swizzle lays them out as the
// cache stores them (chunk c of row t at c ^ (t & 7)).
__device__ __forceinline__ void tma_page(void* dst, const CUtensorMap* map, int row, int page, uint64_t* bar) {
    asm volatile(
        "cp.async.bulk.tensor.3d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4}], [%5];" ::"r"(
            smem_addr(dst)),
        "l"(reinterpret_cast<uint64_t>(map)), "r"(0), "r"(row), "r"(page), "r"(smem_addr(bar))
        : "memory");
}

// What the plan needs of a group: the keys its rows see (0: no active row), its slot, and (PLAN_DEVICE)
// how many rows it has: row j at position keys - rows + j.
struct Group {
    int keys, seq, rows;
};
// PLAN_DEVICE: from the slot state left by earlier steps (the rule the embedding applies), so it is known
// before the dependency wait.
__device__ __forceinline__ Group load_group(const AttnArgs& a, int g) {
    Group x = {0, g, 0};
    if (a.plan == PLAN_DEVICE) {  // one round of independent loads
        const int act = a.active[g], dn = a.done[g], np = a.seq_new[g], len = a.seq_len[g];
        if (act && !dn && np > 0) {
            x.keys = len + np;
            x.rows = np;
        }
        return x;
    }
#pragma unroll
    for (int j = 0; j < RPG; ++j) {
        if (j >= a.rows_per_group) break;
        const int r = g * a.rows_per_group + j;
        const int rs = r < a.rows ? a.row_seq[r] : -1, rp = r < a.rows ? a.row_pos[r] : 0;
        if (rs >= 0) {
            x.seq = rs;
            x.keys = max(x.keys, rp + 1);
        }
    }
    return x;
}

template <bool PLAIN>
__global__ void __launch_bounds__(ATT_THREADS, 4)
    attn_kernel(const AttnArgs a, const __grid_constant__ CUtensorMap plain_map) {
    extern __shared__ __align__(1024) unsigned char smem_raw[];
    // the tensor copy's swizzle goes by the address: 1024-byte aligned slots
    unsigned char* smem = reinterpret_cast<unsigned char*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
    __shared__ uint64_t bar[ATT_STAGES];
    __shared__ int s_sum[NW], s_g0, s_off;
    __shared__ Group s_group[ATT_THREADS];  // the groups' facts, where they are at most that many
    __shared__ int s_share[2][4];           // groups shared with other CTAs: group, first CTA, parts, active rows
    __shared__ int s_last[2];

    const int jc = blockIdx.x, h = blockIdx.y;
    TraceEnd trace_guard(a.trace);
    const int H = a.n_heads, P = a.page_size, rpg = a.rows_per_group;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int KB = half_keys(P);       // keys per batch
    const int ppb = KB / P;            // pages per batch
    __nv_bfloat16* Ks = reinterpret_cast<__nv_bfloat16*>(smem);
    __nv_bfloat16* Vs = Ks + ATT_STAGES * KB * HEAD_DIM;
    float* wst = reinterpret_cast<float*>(Vs + ATT_STAGES * KB * HEAD_DIM);  // [NW][MROWS][PART] warp states
    const long long kv_head_off = (long long)h * P * HEAD_DIM;
    const long long v_off = (long long)H * P * HEAD_DIM;

    if (tid == 0) {
        if (PLAIN) asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(&plain_map)) : "memory");
        for (int i = 0; i < ATT_STAGES; ++i) mbar_init(&bar[i], 1);
        s_share[0][2] = s_share[1][2] = 0;
        fence_barrier_init();
    }
    if (a.plan != PLAN_DEVICE) {  // the rows' plan is written by an earlier kernel of this pass
        pdl_launch_dependents();
        pdl_wait();
        trace_wait(a.trace);
    }

    // ---- this CTA's share of the head's stream of batches ----
    // the groups' facts in shared memory: of all of them, or (whole) of this CTA's
    const bool few = a.groups <= ATT_THREADS || a.whole;
    auto group_of = [&](int g) { return few ? s_group[a.whole ? 0 : g] : load_group(a, g); };
    auto batches = [&](const Group& x) { return (x.keys + KB - 1) / KB; };
    // inclusive sum of v over the block's threads before and including this one; total: of all
    auto block_scan = [&](int v, int& total) {
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int u = __shfl_up_sync(FULL_MASK, v, o);
            if (lane >= o) v += u;
        }
        __syncthreads();  // s_sum's last readers are done
        if (lane == 31) s_sum[warp] = v;
        __syncthreads();
        total = 0;
#pragma unroll
        for (int w = 0; w < NW; ++w) {
            if (w < warp) v += s_sum[w];
            total += s_sum[w];
        }
        return v;
    };
    int T, J, x0, x1;  // batches of the head, CTAs that take part (each has a batch), this CTA's range
    if (a.whole) {  // group jc, all of it
        T = J = x0 = 0;
        const Group x = load_group(a, jc);
        x1 = batches(x);
        if (tid == 0) {
            s_group[0] = x;
            s_g0 = jc;
            s_off = 0;
        }
    } else {
        int nb0 = 0;  // of the first 128 groups
        if (tid < a.groups) {
            const Group x = load_group(a, tid);
            s_group[tid] = x;
            nb0 = batches(x);
        }
        const int incl0 = block_scan(nb0, T);
        for (int base = ATT_THREADS; base < a.groups; base += ATT_THREADS) {
            int t;
            block_scan(base + tid < a.groups ? batches(load_group(a, base + tid)) : 0, t);
            T += t;
        }
        J = max(1, min((int)gridDim.x, T));
        x0 = jc < J ? (int)((long long)jc * T / J) : T;
        x1 = jc < J ? (int)((long long)(jc + 1) * T / J) : T;
        if (x0 < x1) {  // the group that holds batch x0
            int before = 0;
            for (int base = 0; base < a.groups; base += ATT_THREADS) {
                int nb = nb0, incl = incl0, t = 0;
                if (!few) {
                    nb = base + tid < a.groups ? batches(load_group(a, base + tid)) : 0;
                    incl = block_scan(nb, t);
                }
                if (before + incl - nb <= x0 && x0 < before + incl) {
                    s_g0 = base + tid;
                    s_off = x0 - (before + incl - nb);
                }
                before += t;
                if (x0 < before) break;
            }
        }
    }
    __syncthreads();

    // ---- copies: warp 0 walks the stream ahead of the tiles ----
    int pg = 0, pb = 0, pnb = 0, pseq = -1, pkeys = 0, ppages = 0, pold = 0, staged = 0;  // group, its next batch, ...
    auto next_group = [&]() {  // the next group with keys, from pg on
        for (;; ++pg) {
            const Group x = group_of(pg);
            pnb = batches(x);
            pseq = x.seq;
            pkeys = x.keys;
            ppages = (x.keys + P - 1) / P;
            pold = a.plan == PLAN_DEVICE ? (x.keys - x.rows) / P : ppages;  // pages of earlier steps' keys only
            if (pnb > 0) return;
        }
    };
    auto stage_next = [&]() {  // the stream's next batch into the ring (warp 0)
        const int slot = staged % ATT_STAGES, p = pb * ppb + lane;
        const bool mine = lane < ppb && p < ppages;
        const int phys = mine ? a.block_table[(size_t)pseq * a.bt_stride + p] : -1;
        if (mine && phys < 0 && a.err) atomicOr(a.err, ERR_BOUNDS);  // unreserved page: report, never read
        // of the group's last page only the 16-key tiles that hold a key (tensor copies: whole pages)
        const int rows = PLAIN ? P : min(P, (pkeys - p * P + 15) & ~15);
        const uint32_t blk = phys >= 0 ? (uint32_t)rows * HEAD_DIM * 2 : 0u;
        const uint32_t bytes = 2 * __reduce_add_sync(FULL_MASK, blk);
        fence_proxy_async();  // the slot was last read by this CTA's threads
        if (lane == 0) mbar_arrive_expect_tx(&bar[slot], bytes);
        __syncwarp();
        if (phys >= 0) {
            __nv_bfloat16* kd = Ks + ((size_t)slot * KB + lane * P) * HEAD_DIM;
            __nv_bfloat16* vd = Vs + ((size_t)slot * KB + lane * P) * HEAD_DIM;
            if (PLAIN) {
                const int row = (int)((a.layer_off + kv_head_off) / HEAD_DIM);
                tma_page(kd, &plain_map, row, phys, &bar[slot]);
                tma_page(vd, &plain_map, row + (int)(v_off / HEAD_DIM), phys, &bar[slot]);
            } else {
                const __nv_bfloat16* base = a.kv_pool + (long long)phys * a.page_elems + a.layer_off + kv_head_off;
                bulk_copy_g2s(kd, base, blk, &bar[slot]);
                bulk_copy_g2s(vd, base + v_off, blk, &bar[slot]);
            }
        }
        ++staged;
        if (++pb == pnb && x0 + staged < x1) {
            ++pg;
            next_group();
            pb = 0;
        }
    };
    const int n = x1 - x0;
    int g = 0, cb = 0;  // group and batch within it
    if (n > 0) {
        g = s_g0;
        cb = s_off;
        if (warp == 0) {
            pg = g;
            next_group();
            pb = cb;
            if (a.plan == PLAN_DEVICE)
                while (staged < min(n, ATT_STAGES) && min((pb + 1) * ppb, ppages) <= pold) stage_next();
        }
    }
    if (a.plan == PLAN_DEVICE) {
        pdl_launch_dependents();
        pdl_wait();
        trace_wait(a.trace);
    }
    if (warp == 0)
        while (staged < min(n, ATT_STAGES)) stage_next();

    // output pair (2 lane, 2 lane + 1) of head h in row row_j of group gr
    auto put = [&](int gr, int row_j, float v0, float v1) {
        const size_t r = (size_t)gr * rpg + row_j;
        if (a.out) {
            float* o = a.out + r * a.ldo + h * HEAD_DIM + 2 * lane;
            o[0] = v0;
            o[1] = v1;
        }
        if (a.out_hi) {
            uint32_t hi, lo;
            split2(v0, v1, hi, lo);
            *reinterpret_cast<uint32_t*>(a.out_hi + r * a.ldb + h * HEAD_DIM + 2 * lane) = hi;
            *reinterpret_cast<uint32_t*>(a.out_lo + r * a.ldb + h * HEAD_DIM + 2 * lane) = lo;
        }
    };
    if (a.out_hi)  // groups without keys: zero operand rows, a warp per group
        for (int gr = jc + warp * gridDim.x; gr < a.groups; gr += NW * gridDim.x)
            if (group_of(gr).keys == 0)
                for (int row_j = 0; row_j < rpg; ++row_j) {
                    const size_t o = ((size_t)gr * rpg + row_j) * a.ldb + h * HEAD_DIM + 2 * lane;
                    *reinterpret_cast<uint32_t*>(a.out_hi + o) = 0u;
                    *reinterpret_cast<uint32_t*>(a.out_lo + o) = 0u;
                }

    // per-warp tensor-core tiles with the keys as the M side: S^T = K Q^T (16 keys x the 8 query
    // rows; the queries' bf16 hi and lo parts are two N = 8 operands) and O^T += V^T P^T (head
    // dims x query rows, P^T's hi and lo parts added into the same accumulator).  Lane (g8, c2):
    // keys g8, g8 + 8 of a tile and queries c2, c2 + 1 in S^T; head dims g8, g8 + 8 of each 16-dim
    // block and queries c2, c2 + 1 in O^T.
    const int g8 = lane >> 2, c2 = (lane & 3) * 2;
    // partials: a CTA shares at most its first group (slot 0) and its last (slot 1: begun here)
    // (a CTA is the first of one shared group at most: its counter is that group's)
    auto count_of = [&](int c_first) { return a.ws_count + (size_t)h * J + c_first; };
    auto part_of = [&](int cta, int c_first) {
        return a.ws_part + (((size_t)(h * J + cta) * 2 + (cta == c_first ? 1 : 0)) * RPG) * PART;
    };
    bool ok = true;
    for (int i = 0; i < n && ok; ++g, cb = 0) {
        const Group x = group_of(g);
        if (x.keys == 0) continue;
        const int gpages = (x.keys + P - 1) / P, gnb = batches(x);
        // ---- the group's rows (lanes 0..7 of every warp) and its queries, loaded together ----
        int row_pos = -1;
        if (a.plan == PLAN_DEVICE) {
            if (lane < x.rows) row_pos = x.keys - x.rows + lane;
        } else if (lane < rpg && g * rpg + lane < a.rows) {
            const int rs = a.row_seq[g * rpg + lane], rp = a.row_pos[g * rpg + lane];
            row_pos = rs >= 0 ? rp : -1;
        }
        uint32_t qhi[4][2], qlo[4][2];  // B operand of S^T: query row g8, dims ks * 16 + 8 hh + c2, + 1
        int qpos[2];
        unsigned act;
        {
            const bool in = g8 < rpg && g * rpg + g8 < a.rows;
            const float* qr = a.q + (size_t)(g * rpg + (in ? g8 : 0)) * a.ldq + h * HEAD_DIM + c2;
            float2 v[4][2];
#pragma unroll
            for (int ks = 0; ks < 4; ++ks)
#pragma unroll
                for (int hh = 0; hh < 2; ++hh)
                    v[ks][hh] = make_float2(qr[ks * 16 + hh * 8], qr[ks * 16 + hh * 8 + 1]);
            act = __ballot_sync(FULL_MASK, row_pos >= 0);
            const float scale = in && (act >> g8 & 1) ? 0.125f : 0.f;  // 1/sqrt(64): bf16-valued queries stay exact
#pragma unroll
            for (int j = 0; j < 2; ++j) qpos[j] = __shfl_sync(FULL_MASK, row_pos, c2 + j);
#pragma unroll
            for (int ks = 0; ks < 4; ++ks)
#pragma unroll
                for (int hh = 0; hh < 2; ++hh)
                    split2(scale != 0.f ? v[ks][hh].x * scale : 0.f, scale != 0.f ? v[ks][hh].y * scale : 0.f,
                           qhi[ks][hh], qlo[ks][hh]);
        }
        float m_w[2] = {-INFINITY, -INFINITY} /* log2 units */, l_w[2] = {0.f, 0.f};
        float o[4][4];  // O^T block dp: dims dp * 16 + g8 (0, 1) and + 8 (2, 3), queries c2 + (i & 1)
#pragma unroll
        for (int j = 0; j < 4; ++j)
#pragma unroll
            for (int e = 0; e < 4; ++e) o[j][e] = 0.f;
        const int gs = x0 + i - cb;  // the group's first batch in the stream
        const int cend = min(gnb, cb + n - i);
        for (; cb < cend; ++cb, ++i) {
            const int slot = i % ATT_STAGES, key0 = cb * KB;
            const int nk = min(min(ppb, gpages - cb * ppb) * P, (x.keys - key0 + 15) & ~15);
            ok = mbar_wait(&bar[slot], (uint32_t)(i / ATT_STAGES) & 1, a.err) && ok;
            const uint32_t kb = smem_addr(Ks + (size_t)slot * KB * HEAD_DIM);
            const uint32_t vb = smem_addr(Vs + (size_t)slot * KB * HEAD_DIM);
            for (int kt = warp * 16; kt < nk && ok; kt += NW * 16) {
                float sh[4] = {0.f, 0.f, 0.f, 0.f}, sl[4] = {0.f, 0.f, 0.f, 0.f};  // hi and lo parts: own chains
                {
                    // A = K rows kt..kt+15: matrices (keys 0-7 | 8-15) x (dims 0-7 | 8-15) of the k-step
                    const int key = kt + (lane & 7) + (((lane >> 3) & 1) << 3), chalf = lane >> 4;
#pragma unroll
                    for (int ks = 0; ks < 4; ++ks) {
                        uint32_t ka[4];
                        ldsm_x4(ka, kb + key * 128 + ((uint32_t)((2 * ks + chalf) ^ (key & 7)) << 4));
                        const uint32_t bh[2] = {qhi[ks][0], qhi[ks][1]}, bl[2] = {qlo[ks][0], qlo[ks][1]};
                        mma_bf16(sh, ka, bh);
                        mma_bf16(sl, ka, bl);
                    }
                }
                // this lane's scores: keys kt + g8 (e = 0, 1) and kt + g8 + 8 (e = 2, 3), query c2 + (e & 1)
                float sv[4];
#pragma unroll
                for (int e = 0; e < 4; ++e)
                    sv[e] = key0 + kt + g8 + (e >> 1) * 8 <= qpos[e & 1] ? sh[e] + sl[e] : -INFINITY;
                // weights are taken relative to the row's running maximum m_w; where no lane's score exceeds it,
                // the maximum over the lanes and the rescaling are skipped.  (A reference that may lag behind by
                // up to 2^8 moves less often, 0.5 % faster, but 32 slots of 180-2000 keys are then 3.4e-6 from
                // 64 bits instead of 3.1e-6.)
                float t0 = fmaxf(sv[0], sv[2]) * LOG2E, t1 = fmaxf(sv[1], sv[3]) * LOG2E;
                if (__any_sync(FULL_MASK, t0 > m_w[0] || t1 > m_w[1])) {
#pragma unroll
                    for (int off = 4; off < 32; off <<= 1) {  // over the tile's keys: lanes g8
                        t0 = fmaxf(t0, __shfl_xor_sync(FULL_MASK, t0, off));
                        t1 = fmaxf(t1, __shfl_xor_sync(FULL_MASK, t1, off));
                    }
                    const float mn[2] = {fmaxf(m_w[0], t0), fmaxf(m_w[1], t1)};
#pragma unroll
                    for (int j = 0; j < 2; ++j) {
                        const float corr = m_w[j] == -INFINITY ? 1.f : ex2(m_w[j] - mn[j]);  // (no sums yet)
                        l_w[j] *= corr;
                        m_w[j] = mn[j];
#pragma unroll
                        for (int dp = 0; dp < 4; ++dp) {
                            o[dp][j] *= corr;
                            o[dp][2 + j] *= corr;
                        }
                    }
                }
                float pv[4];
#pragma unroll
                for (int e = 0; e < 4; ++e) pv[e] = sv[e] == -INFINITY ? 0.f : ex2(fmaf(sv[e], LOG2E, -m_w[e & 1]));
                l_w[0] += pv[0] + pv[2];
                l_w[1] += pv[1] + pv[3];
                // P^T as the B operand (keys x queries): this lane holds rows g8 (keys) and columns c2
                // (queries) of each 8 x 8 block; its transpose is the operand's layout (query g8, keys c2, + 1)
                uint32_t ph0, pl0, ph1, pl1;
                split2(pv[0], pv[1], ph0, pl0);  // keys g8
                split2(pv[2], pv[3], ph1, pl1);  // keys g8 + 8
                const uint32_t bph[2] = {movmatrix_trans(ph0), movmatrix_trans(ph1)};
                const uint32_t bpl[2] = {movmatrix_trans(pl0), movmatrix_trans(pl1)};
                // A = V^T: matrices (dims 0-7 | 8-15 of block dp) x (keys 0-7 | 8-15), from the key rows
                const int vkey = kt + (lane & 7) + ((lane >> 4) << 3), vhalf = (lane >> 3) & 1;
#pragma unroll
                for (int dp = 0; dp < 4; ++dp) {
                    uint32_t va[4];
                    ldsm_x4_t(va, vb + vkey * 128 + ((uint32_t)((2 * dp + vhalf) ^ (vkey & 7)) << 4));
                    mma_bf16(o[dp], va, bph);
                    mma_bf16(o[dp], va, bpl);
                }
            }
            __syncthreads();  // every warp is done with this slot
            if (warp == 0 && staged < n) stage_next();
        }
        ok = __syncthreads_and(ok) != 0;
        if (!ok) break;

        // ---- the group's keys of this CTA are done: merge the warps' (max, sum, out) per row ----
#pragma unroll
        for (int j = 0; j < 2; ++j)  // each lane summed its own keys; the query's keys span lanes g8
#pragma unroll
            for (int off = 4; off < 32; off <<= 1) l_w[j] += __shfl_xor_sync(FULL_MASK, l_w[j], off);
        // the CTAs that share the group: those of its first and last batch
        const int c_first = a.whole ? jc : (int)(((long long)(gs + 1) * J - 1) / T);
        const int parts = a.whole ? 1 : (int)(((long long)(gs + gnb) * J - 1) / T) - c_first + 1;
#pragma unroll 1
        for (int r0 = 0; r0 < rpg; r0 += MROWS) {
            if ((c2 & ~(MROWS - 1)) == r0) {
#pragma unroll
                for (int j = 0; j < 2; ++j) {
                    float* ws = wst + ((size_t)warp * MROWS + (c2 & (MROWS - 1)) + j) * PART;
                    if (g8 == 0) {
                        ws[0] = m_w[j];
                        ws[1] = l_w[j];
                    }
#pragma unroll
                    for (int dp = 0; dp < 4; ++dp) {
                        ws[2 + dp * 16 + g8] = o[dp][j];
                        ws[2 + dp * 16 + g8 + 8] = o[dp][2 + j];
                    }
                }
            }
            __syncthreads();
            const int row_j = r0 + warp;  // warp w merges row r0 + w: output dims 2 lane, 2 lane + 1
            if (row_j < rpg) {
                float M = -INFINITY, L = 0.f, y0 = 0.f, y1 = 0.f;
#pragma unroll
                for (int w = 0; w < NW; ++w) M = fmaxf(M, wst[((size_t)w * MROWS + warp) * PART]);
#pragma unroll
                for (int w = 0; w < NW; ++w) {
                    const float* ws = wst + ((size_t)w * MROWS + warp) * PART;
                    const float sc = ws[0] == -INFINITY ? 0.f : ex2(ws[0] - M);
                    L = fmaf(sc, ws[1], L);
                    y0 = fmaf(sc, ws[2 + 2 * lane], y0);
                    y1 = fmaf(sc, ws[3 + 2 * lane], y1);
                }
                if (parts > 1) {
                    float* pj = part_of(jc, c_first) + row_j * PART;
                    if (lane == 0) {
                        pj[0] = M;
                        pj[1] = L;
                    }
                    pj[2 + 2 * lane] = y0;
                    pj[3 + 2 * lane] = y1;
                } else if (act >> row_j & 1) {
                    put(g, row_j, y0 / L, y1 / L);
                } else if (a.out_hi) {
                    put(g, row_j, 0.f, 0.f);
                }
            }
            __syncthreads();  // wst may be written again
        }
        if (parts > 1 && tid == 0) {
            int* sh = s_share[jc == c_first ? 1 : 0];
            sh[0] = g;
            sh[1] = c_first;
            sh[2] = parts;
            sh[3] = (int)act;
        }
    }
    // ---- the shared groups (at most the CTA's first and its last): the CTA that finishes one last merges
    // its parts; both counters are asked at once, after the stream ----
    __threadfence();
    __syncthreads();
    trace_mark(a.trace, 2);  // partials written
    if (tid < 2) {
        const int* sh = s_share[tid];
        s_last[tid] = ok && sh[2] > 0 ? atomicAdd(count_of(sh[1]), 1) == sh[2] - 1 : 0;
    }
    __syncthreads();
#pragma unroll 1
    for (int k = 0; k < 2; ++k) {
        if (!s_last[k]) continue;
        __threadfence();
        const int sg = s_share[k][0], c_first = s_share[k][1], parts = s_share[k][2];
        const unsigned act = (unsigned)s_share[k][3];
        for (int row_j = warp; row_j < rpg; row_j += NW) {
            if (!(act >> row_j & 1)) {
                if (a.out_hi) put(sg, row_j, 0.f, 0.f);
                continue;
            }
            // the parts in stream order, four loaded at a time
            float M = -INFINITY, L = 0.f, y0 = 0.f, y1 = 0.f;
            for (int p0 = 0; p0 < parts; p0 += 4) {
                float m[4], l[4], v0[4], v1[4];
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    const bool have = p0 + q < parts;
                    const float* pj = part_of(c_first + (have ? p0 + q : 0), c_first) + row_j * PART;
                    m[q] = have ? __ldcg(pj) : -INFINITY;
                    l[q] = have ? __ldcg(pj + 1) : 0.f;
                    v0[q] = have ? __ldcg(pj + 2 + 2 * lane) : 0.f;
                    v1[q] = have ? __ldcg(pj + 3 + 2 * lane) : 0.f;
                }
                const float Mn = fmaxf(fmaxf(M, fmaxf(m[0], m[1])), fmaxf(m[2], m[3]));
                const float old = M == -INFINITY ? 0.f : ex2(M - Mn);
                L *= old;
                y0 *= old;
                y1 *= old;
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    const float w = m[q] == -INFINITY ? 0.f : ex2(m[q] - Mn);
                    L = fmaf(w, l[q], L);
                    y0 = fmaf(w, v0[q], y0);
                    y1 = fmaf(w, v1[q], y1);
                }
                M = Mn;
            }
            put(sg, row_j, y0 / L, y1 / L);
        }
        if (tid == 0) *count_of(c_first) = 0;
    }
    if (!ok && warp == 0) {  // error word set; let copies in flight land before leaving
        for (int i = max(0, staged - ATT_STAGES); i < staged; ++i)
            mbar_wait(&bar[i % ATT_STAGES], (uint32_t)(i / ATT_STAGES) & 1, nullptr);
    }
}

}  // namespace

size_t attn_workspace_floats(int n_heads, int ctas) {
    return ctas > 1 ? (size_t)n_heads * ctas * 2 * RPG * PART : 0;
}

size_t attn_smem_bytes(int page_size) {
    return (size_t)2 * ATT_STAGES * half_keys(page_size) * HEAD_DIM * 2 + (size_t)NW * MROWS * PART * 4 + 1024;
}

int attn_ctas_per_sm(int page_size) { return page_size > 64 ? ATTN_CTAS_PER_SM / 2 : ATTN_CTAS_PER_SM; }

int attn_ctas_for(int groups, int n_heads, int page_size, int max_keys, int num_sms) {
    // one wave of resident CTAs while they have batches: a batch each (5 slots of 100-600 keys, 8 heads: 10.5 us,
    // 12.7 with two), of contexts over 1024 keys more, since every CTA of a group leaves partials that its last
    // one merges (1 slot of 2000 keys, 16 heads: 20.8, 14.6 and 12.6 us with 32, 16 and 8 CTAs a head; with few
    // heads the merges do not meet in time: 2 slots, 1 head: 12.5, 11.0 and 12.5)
    const int kb = half_keys(page_size), nb = (max_keys + kb - 1) / kb;  // keys of a batch, batches per group
    const int each = max_keys <= 1024 ? 1 : (n_heads <= 4 ? 128 : 256) / kb;
    const long long want = (long long)groups * ((nb + each - 1) / each);
    return (int)max(1ll, min(want, (long long)max(1, attn_ctas_per_sm(page_size) * num_sms / n_heads)));
}

bool attn_whole_groups(int groups, int n_heads, int page_size, int max_keys, int num_sms) {
    // contexts of a batch or two: a plan and a merge would cost more than they share out (1 slot of 33 keys: 6.6 vs
    // 8.4 us; 20 slots of 33-99 keys, 16 heads: 8.5 vs 10.4).  Longer ones where the groups are most of a wave, and
    // no more: 20 slots of 200-400 keys, 8 heads: 12.6 vs 18.9 us, 10 slots of 300-600, 12 heads: 12.6 vs 14.6 (with
    // 8 heads, 80 groups, 14.5 vs 12.5; 32 slots of 180-2000 keys, 8 heads: 28.4 vs 20.7).
    const long long ctas = (long long)groups * n_heads;
    return max_keys <= 2 * half_keys(page_size) ||
           (max_keys <= 640 && 4 * ctas >= 3ll * num_sms && ctas <= (long long)attn_ctas_per_sm(page_size) * num_sms);
}

template <bool PLAIN>
static cudaError_t launch_attn_t(const AttnArgs& a, const CUtensorMap& map, cudaStream_t s, bool pdl) {
    if (a.rows_per_group < 1 || a.rows_per_group > RPG || half_keys(a.page_size) % a.page_size != 0 || a.groups < 1 ||
        (!a.whole && a.ctas < 1) || (a.plan != PLAN_ROWS && a.plan != PLAN_DEVICE))
        return cudaErrorInvalidValue;
    const size_t smem = attn_smem_bytes(a.page_size);
    auto kern = attn_kernel<PLAIN>;
    cudaError_t e = ensure_kernel_smem(reinterpret_cast<const void*>(kern), smem);
    if (e != cudaSuccess) return e;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(a.whole ? a.groups : a.ctas, a.n_heads);
    cfg.blockDim = dim3(ATT_THREADS);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = pdl ? 1 : 0;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kern, a, map);
}

cudaError_t launch_attention(const AttnArgs& a, cudaStream_t s, bool pdl) {
    return launch_attn_t<false>(a, CUtensorMap{}, s, pdl);
}

cudaError_t launch_attention_plain(const AttnArgs& a, cudaStream_t s) {
    if (a.plan != PLAN_ROWS) return cudaErrorInvalidValue;
    // [page][row of the page (layer, keys | values, head, key)][64]; the number of pages is not known here
    // (the kernel reads only pages of the block table)
    CUtensorMap map;
    if (tc_encode_rows(&map, a.kv_pool, (uint64_t)a.page_elems / HEAD_DIM, (uint32_t)a.page_size) != 0)
        return cudaErrorInvalidValue;
    return launch_attn_t<true>(a, map, s, false);
}

}  // namespace mtp

// ---- allocation-free attention (mtp_attention_noalloc) ----------------------
// For callers that may not allocate GPU memory while they run (a real-time
// audio callback, where cudaMalloc/cudaFree can block or synchronise the
// device; a host that owns all GPU memory): the split-merge scratch of the
// attention kernel is this fixed array, one per GPU that loads the library,
// held until the process exits and shared by every call on that GPU.
static __device__ __align__(256) unsigned char g_attention_scratch[MTP_ATTENTION_NOALLOC_SCRATCH_BYTES];

extern "C" MTP_API int mtp_attention_noalloc(const mtp_attention_args* args, void* cuda_stream) {
    mtp::clear_error();
    mtp::AttnStandalonePlan p;
    const int r = mtp::attention_standalone_plan(args, true, &p);  // checked before anything is queued
    if (r != MTP_OK) return r;
    if (p.need > MTP_ATTENTION_NOALLOC_SCRATCH_BYTES) {
        char msg[256];
        std::snprintf(msg, sizeof(msg),
                      "attention: this call needs %zu bytes of scratch, the fixed scratch array holds %u", p.need,
                      (unsigned)MTP_ATTENTION_NOALLOC_SCRATCH_BYTES);
        return mtp::report_error(MTP_ERR_INVALID, msg);
    }
    // The array's name is only a host-side stand-in for it; its device address
    // is looked up on every call (no allocation), so it stays right after the
    // context of the device is torn down and made again.
    void* scratch = nullptr;
    cudaError_t e = cudaGetSymbolAddress(&scratch, g_attention_scratch);
    if (e != cudaSuccess || !scratch) {
        char msg[256];
        std::snprintf(msg, sizeof(msg), "attention scratch address lookup failed: %s", cudaGetErrorString(e));
        return mtp::report_error(MTP_ERR_CUDA, msg);
    }
    const cudaStream_t s = static_cast<cudaStream_t>(cuda_stream);
    e = cudaMemsetAsync(scratch, 0, p.count_bytes, s);  // merge counters
    if (e != cudaSuccess) return mtp::report_error(MTP_ERR_CUDA, cudaGetErrorString(e));
    return mtp::attention_standalone_launch(args, p, scratch, MTP_ATTENTION_NOALLOC_SCRATCH_BYTES, s);
}

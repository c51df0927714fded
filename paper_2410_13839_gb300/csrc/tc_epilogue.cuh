// tc_epilogue.cuh -- what the tensor-core projections (tc_gemm.cu,
// tc_gemm_pair.cu) do with N consecutive activation rows of one weight row per
// lane, straight from the accumulator's registers: a lane holds weight row f,
// so a warp's store of one activation row is 32 consecutive features (128
// bytes of fp32).  bf16 outputs go out in pairs: lanes 2i and 2i + 1 exchange
// one value, then the even lane writes features (f, f + 1) of row e and the odd
// lane those of row e + 1.
#pragma once

#include "common.cuh"
#include "kernels.cuh"

namespace mtp {

__device__ __forceinline__ uint32_t pack_bf16(float lo, float hi) {
    const __nv_bfloat162 p = __floats2bfloat162_rn(lo, hi);
    return *reinterpret_cast<const uint32_t*>(&p);
}

// v[e]: the product of activation row n0 + e (tile row j0 + e; rows of them
// exist) and weight row f; bias is f's.  rowbase / rowt: the tile's row facts
// (TC_QKV: element offset of the row's key row in its page, -1 unreserved page,
// -2 row of no sequence, and the key row within the page; TC_GELU_PACK: rowt
// nonzero for a row of a sequence).  SHARED: other CTAs add to the same outputs
// (TC_ACCUM by atomics).  Called by whole warps.
template <int EPI, bool SHARED, int N>
__device__ __forceinline__ void tc_epilogue(const TcGemmArgs& a, const float (&v)[N], int n0, int j0, int rows, int f,
                                            float bias, const long long* rowbase, const int* rowt) {
    const int lane = threadIdx.x & 31, odd = lane & 1;
    if (EPI == TC_STORE) {
        float* o = a.out + (size_t)n0 * a.ldo + f;
#pragma unroll
        for (int e = 0; e < N; ++e)
            if (e < rows) o[(size_t)e * a.ldo] = v[e] + bias;
    } else if (EPI == TC_ACCUM && SHARED) {
        if (a.n_valid && f >= a.n_valid) return;
        float* o = a.out + (size_t)n0 * a.ldo + f;
#pragma unroll
        for (int e = 0; e < N; ++e)
            if (e < rows) atomicAdd(o + (size_t)e * a.ldo, v[e] + bias);
    } else if (EPI == TC_ACCUM) {
        float* o = a.out + (size_t)n0 * a.ldo + f;
#pragma unroll
        for (int e0 = 0; e0 < N; e0 += 8) {
            float x[8];
#pragma unroll
            for (int e = 0; e < 8; ++e) x[e] = e0 + e < rows ? o[(size_t)(e0 + e) * a.ldo] : 0.f;
#pragma unroll
            for (int e = 0; e < 8; ++e)
                if (e0 + e < rows) o[(size_t)(e0 + e) * a.ldo] = x[e] + (v[e0 + e] + bias);
        }
    } else if (EPI == TC_GELU_PACK) {
        uint32_t act[(N + 31) / 32];  // rows of a sequence (the others are written as zeros)
#pragma unroll
        for (int q = 0; q < N; q += 32) act[q / 32] = __ballot_sync(FULL_MASK, q + lane < N && rowt[j0 + q + lane]);
        const size_t at = (size_t)(n0 + odd) * a.ldo + (f - odd);
        __nv_bfloat16 *ph = a.pack_hi + at, *pl = a.pack_lo + at;
        const int mine = rows - odd;  // this lane writes rows e + odd < rows
#pragma unroll
        for (int e = 0; e < N; e += 2) {
            const float u0 = gelu_erf(v[e] + bias), u1 = gelu_erf(v[e + 1] + bias);
            const float g0 = act[e >> 5] >> (e & 31) & 1 ? u0 : 0.f;
            const float g1 = act[e >> 5] >> ((e & 31) + 1) & 1 ? u1 : 0.f;
            const float got = __shfl_xor_sync(FULL_MASK, odd ? g0 : g1, 1);
            const float y0 = odd ? got : g0, y1 = odd ? g1 : got;
            const uint32_t hi = pack_bf16(y0, y1);
            const uint32_t lo = pack_bf16(y0 - bf16_lo(hi), y1 - bf16_hi(hi));
            if (e < mine) {
                *reinterpret_cast<uint32_t*>(ph) = hi;
                *reinterpret_cast<uint32_t*>(pl) = lo;
            }
            ph += 2 * (size_t)a.ldo;
            pl += 2 * (size_t)a.ldo;
        }
    } else {  // TC_QKV: features h * 192 + {q, k, v} * 64 + dd (one head and part per warp)
        const int H = a.n_heads, P = a.page_size, d = H * HEAD_DIM;
        const int h = f / (3 * HEAD_DIM), sec = (f / HEAD_DIM) % 3, dd = f % HEAD_DIM;
        if (sec == 0) {
            float* o = a.out + (size_t)n0 * d + h * HEAD_DIM + dd;
#pragma unroll
            for (int e = 0; e < N; ++e)
                if (rowbase[j0 + e] != -2) o[(size_t)e * d] = v[e] + bias;
        } else {
            const int de = dd - odd;
            const long long off = (long long)(sec - 1) * H * P * HEAD_DIM + (long long)h * P * HEAD_DIM;
#pragma unroll
            for (int e = 0; e < N; e += 2) {
                const float g0 = v[e] + bias, g1 = v[e + 1] + bias;
                const float got = __shfl_xor_sync(FULL_MASK, odd ? g0 : g1, 1);
                const uint32_t pk = odd ? pack_bf16(got, g1) : pack_bf16(g0, got);
                const long long base = rowbase[j0 + e + odd];
                const int tr = rowt[j0 + e + odd];
                if (base >= 0)
                    *reinterpret_cast<uint32_t*>(reinterpret_cast<uint16_t*>(a.kv_pool) + base + off +
                                                 ((((de >> 3) ^ (tr & 7)) << 3) | (de & 7))) = pk;
            }
        }
    }
}

}  // namespace mtp

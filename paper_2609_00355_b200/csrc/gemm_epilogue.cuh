// Pieces that the GEMM kernels' epilogues share: the sampling mode's noise field and the end of an arg-max launch.
#pragma once
#include "gemm_tc.cuh"
#include "tc_ptx.cuh"

namespace glance {
namespace {

// Philox4x32-10 (Salmon et al., SC 2011): the counter-based generator behind the sampling mode's noise field.
__device__ __forceinline__ uint4 philox4x32_10(uint4 c, uint2 k) {
#pragma unroll
    for (int r = 0; r < 10; ++r) {
        const uint32_t hi0 = __umulhi(0xD2511F53u, c.x), lo0 = 0xD2511F53u * c.x;
        const uint32_t hi1 = __umulhi(0xCD9E8D57u, c.z), lo1 = 0xCD9E8D57u * c.z;
        c = make_uint4(hi1 ^ c.y ^ k.x, lo1, hi0 ^ c.w ^ k.y, lo0);
        k.x += 0x9E3779B9u;
        k.y += 0xBB67AE85u;
    }
    return c;
}
// standard Gumbel noise from one 32-bit word: u = ((w >> 9) + 0.5) 2^-23 lies strictly inside (0,1)
__device__ __forceinline__ float gumbel_from_word(uint32_t w) {
    const float u = ((float)(w >> 9) + 0.5f) * 1.1920928955078125e-07f;
    return -logf(-logf(u));
}

// End of an arg-max launch, called by all NT threads of every CTA: the last CTA to finish decodes the merged keys and, with
// the entropy log on, merges the `ent_tiles` soft-max parts of every root row.
template <int NT>
__device__ __forceinline__ void finish_argmax(const TcGemmArgs &a, int ent_tiles) {
    // the last CTA to finish turns the merged keys into token ids and re-arms keys and counter
    __shared__ int is_last;
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0) is_last = (atomicAdd(a.counter, 1) == (int)(gridDim.x * gridDim.y * gridDim.z) - 1);
    __syncthreads();
    if (is_last) {
        __threadfence();
        for (int r = threadIdx.x; r < a.R; r += blockDim.x) {
            const unsigned long long k = __ldcg(a.keys + r);
            a.argmax[r] = unpack_id(k);
            a.keys[r] = 0ull;
        }
        if (threadIdx.x == 0) *a.counter = 0;
        if (a.ent_out) {
            // entropy of every root row from the per-part statistics: H = (M + log L) - T / L, merged in a fixed order
            __shared__ float red_m[NT / 32], red_l[NT / 32], red_t[NT / 32];
            const int wid = threadIdx.x >> 5, ln = threadIdx.x & 31;
            for (int sq = 0; sq < a.ent_batch && sq * a.ent_N < a.R; ++sq) {
                float M = -INFINITY, L = 0.f, T = 0.f;
                for (int tl = threadIdx.x; tl < ent_tiles; tl += blockDim.x) {
                    const float *src = a.ent_part + ((size_t)tl * a.ent_batch + sq) * 3;
                    const float m = __ldcg(src), l = __ldcg(src + 1), t = __ldcg(src + 2);
                    const float nm = fmaxf(M, m);
                    const float c0 = (M == -INFINITY) ? 0.f : __expf(M - nm), c1 = (m == -INFINITY) ? 0.f : __expf(m - nm);
                    L = L * c0 + l * c1;
                    T = T * c0 + t * c1;
                    M = nm;
                }
#pragma unroll
                for (int o = 16; o > 0; o >>= 1) {
                    const float m = __shfl_xor_sync(0xffffffffu, M, o), l = __shfl_xor_sync(0xffffffffu, L, o);
                    const float t = __shfl_xor_sync(0xffffffffu, T, o);
                    const float nm = fmaxf(M, m);
                    const float c0 = (M == -INFINITY) ? 0.f : __expf(M - nm), c1 = (m == -INFINITY) ? 0.f : __expf(m - nm);
                    L = L * c0 + l * c1;
                    T = T * c0 + t * c1;
                    M = nm;
                }
                if (ln == 0) { red_m[wid] = M; red_l[wid] = L; red_t[wid] = T; }
                __syncthreads();
                if (threadIdx.x == 0) {
                    float gm = -INFINITY;
                    for (int w = 0; w < NT / 32; ++w) gm = fmaxf(gm, red_m[w]);
                    float gl = 0.f, gt = 0.f;
                    for (int w = 0; w < NT / 32; ++w) {
                        const float c = (red_m[w] == -INFINITY) ? 0.f : __expf(red_m[w] - gm);
                        gl += red_l[w] * c;
                        gt += red_t[w] * c;
                    }
                    a.ent_out[sq] = (gm + logf(gl)) - gt / gl;
                }
                __syncthreads();
            }
        }
    }
}

}  // namespace
}  // namespace glance

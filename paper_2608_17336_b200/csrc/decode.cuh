// Launch parameters of the decode step, shared by its two kernels (decode.cu: warp-level MMAs, every supported
// shape; decode_umma.cu: tcgen05 MMAs, head dimension 128 with 128-key tiles).  Not part of the public ABI.
#pragma once

#include <cuda_fp16.h>
#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>

namespace tilemix {

struct DecodeParams {
    int B, Hq, Hk, max_len, G, nb, W, n_splits, n_blk;
    int n_parts;     // partial results per query head in the workspace
    // tcgen05 form, automatic split count: n_ctas CTAs (one wave or two) are shared out over the n_rows = B * Hk rows by
    // their cost, at most split_cap to a row (n_parts = 2 * split_cap); n_splits is then not used
    int balanced, n_rows, n_ctas, split_cap;
    int by_length;   // warp-level form: the grid takes the sequences longest first
    float scale_log2;
    const __half* q;
    const __half* k16;
    const int8_t* k8;
    const float* k_scale;
    const int8_t* v8;
    const float* v_scale;
    const uint32_t* words;
    const int32_t* cache_len;       // the caller's array (device memory; read with a clamp to [0, max_len])
    float* o_part;   // [B, Hq, n_parts, D]
    float* m_part;   // [B, Hq, n_parts]
    float* z_part;
    int8_t* q8_out;
    float* qs_out;
    __half* out;     // [B, Hq, D]
    float* lse;      // nullable [B, Hq]
    // 16 bits per (sequence, KV head) row, 0 before the step: CTAs of the row that have written their partial results.  The
    // last one merges them.  (Not used by a row with one CTA, which writes the output itself.)
    uint32_t* arrived;
    int fused;       // 1: merged by the step, 0: by a kernel of its own
    int* status;     // 4 ints at the start of the workspace (same record as the attention kernel's)
    unsigned long long wait_limit_ns;   // limit of the bounded waits
    int test_drop_tile;                 // testing aid: the producer leaves out the copies of this tile of every split (-1: none)
};

// Merge of partial results: m = max m_s, z = sum z_s 2^(m_s - m), O = sum O~_s 2^(m_s - m) / z for the query head `row` of
// [B, Hq] and the C output columns from e on; a whole warp with consecutive columns.  The parts are taken 32 at a time: lane
// s loads (m_s, z_s) and the weights are shared by shuffles, so that the loads of O~_s depend on one round trip only and are
// in flight together (a part that nobody wrote has m_s = -inf, weight 0, and is not loaded).
template <int D, int C>
__device__ __forceinline__ void merge_columns(const DecodeParams& prm, int64_t row, int n_parts, int e) {
    static_assert(C == 1 || C == 2 || C == 4, "one load per part");
    constexpr float kLn2f = 0.6931471805599453f;
    const int lane = threadIdx.x & 31;
    const int64_t first = row * prm.n_parts;
    float m = -INFINITY, z = 0.f, o[C];
#pragma unroll
    for (int c = 0; c < C; ++c) o[c] = 0.f;
    for (int s0 = 0; s0 < n_parts; s0 += 32) {
        const int s = s0 + lane;
        const float ms = s < n_parts ? __ldcg(prm.m_part + first + s) : -INFINITY;
        const float zs = s < n_parts ? __ldcg(prm.z_part + first + s) : 0.f;
        float mc = ms;
#pragma unroll
        for (int d = 16; d > 0; d >>= 1) mc = fmaxf(mc, __shfl_xor_sync(0xffffffffu, mc, d));
        const float m_new = fmaxf(m, mc);
        if (m_new == -INFINITY) continue;                    // (the same in every lane)
        const float back = m == -INFINITY ? 0.f : exp2f(m - m_new);
        const float w = ms == -INFINITY ? 0.f : exp2f(ms - m_new);
        const float zw = ms == -INFINITY ? 0.f : zs * w;
        z *= back; m = m_new;
#pragma unroll
        for (int c = 0; c < C; ++c) o[c] *= back;
        const float* src = prm.o_part + (first + s0) * D + e;
        // eight at a time, the last group too: the lanes past the last part hold weight 0 (one part after the other at the
        // end is a chain of round trips, and a row of a few splits has nothing else)
        for (int i0 = 0; i0 < min(32, n_parts - s0); i0 += 8) {
#pragma unroll
            for (int k = 0; k < 8; ++k) {
                const float wi = __shfl_sync(0xffffffffu, w, i0 + k);
                z += __shfl_sync(0xffffffffu, zw, i0 + k);
                if (wi != 0.f) {
                    alignas(16) float x[C];
                    const float* at = src + static_cast<int64_t>(i0 + k) * D;
                    if constexpr (C == 4) *reinterpret_cast<float4*>(x) = __ldcg(reinterpret_cast<const float4*>(at));
                    else if constexpr (C == 2) *reinterpret_cast<float2*>(x) = __ldcg(reinterpret_cast<const float2*>(at));
                    else x[0] = __ldcg(at);
#pragma unroll
                    for (int c = 0; c < C; ++c) o[c] += x[c] * wi;
                }
            }
        }
    }
    alignas(8) __half h[C];
#pragma unroll
    for (int c = 0; c < C; ++c) h[c] = __float2half_rn(z > 0.f ? o[c] / z : 0.f);
    __half* dst = prm.out + row * D + e;
    if constexpr (C == 4) *reinterpret_cast<uint2*>(dst) = *reinterpret_cast<const uint2*>(h);
    else if constexpr (C == 2) *reinterpret_cast<__half2*>(dst) = *reinterpret_cast<const __half2*>(h);
    else dst[0] = h[0];
    if (e == 0 && prm.lse != nullptr) prm.lse[row] = z > 0.f ? (m + log2f(z)) * kLn2f : -INFINITY;
}

// At the end of a step's CTA of THREADS threads, by all of them, when the partial results that it owes have been stored: the
// last CTA of row (b, hk) -- `ctas` of them, two or more -- merges the n_parts parts of its R query heads.  A thread takes as
// many adjacent columns as let one pass do: another pass is two more round trips to L2 behind the first (8 query heads of 128 in
// 64-key tiles, one sequence of 8000 keys: four passes 29.4 us, one 15.5, merge kernel 22.9).
template <int D, int R, int THREADS>
__device__ __forceinline__ void merge_if_last(const DecodeParams& prm, int b, int hk, int ctas, int n_parts) {
    constexpr int C = R * D <= THREADS ? 1 : R * D <= 2 * THREADS ? 2 : 4;
    static_assert(R * D <= C * THREADS && D % (32 * C) == 0, "one pass, a warp inside one row");
    __shared__ int last_s;
    __threadfence();        // this thread's partial results, before the arrival
    __syncthreads();
    if (threadIdx.x == 0) {
        const int row = b * prm.Hk + hk;
        const uint32_t before = atomicAdd(prm.arrived + (row >> 1), 1u << (16 * (row & 1)));
        last_s = static_cast<int>((before >> (16 * (row & 1))) & 0xffffu) == ctas - 1;
    }
    __syncthreads();
    if (!last_s) return;
    __threadfence();
    const int i = C * threadIdx.x;
    if (i < R * D) merge_columns<D, C>(prm, static_cast<int64_t>(b) * prm.Hq + hk * R + i / D, n_parts, i % D);
}

// The tcgen05 form of the step for head_dim 128, tile_n 128 (R = Hq / Hk in {1, 2, 4, 8}): enqueues the kernel
// that writes the output (prm.fused) or (m, z, O~) of every split to the workspace, for the caller's merge kernel.  Returns a cudaError_t
// or a TILEMIX_ERR_* code.
int launch_decode_umma(int R, const DecodeParams& prm, cudaStream_t stream);

}  // namespace tilemix

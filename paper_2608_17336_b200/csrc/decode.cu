// Decode step over an INT8 key/value cache (App. C, "Additional Execution Interfaces"): one query
// token per sequence, keys split over CTAs, the H_q/H_k query heads of a KV head served together.
// HBM-bound: a cached token costs d bytes of K8 (or 2d of FP16 K on the FP16 route) plus d bytes of
// V8, each read once.  This file holds the host entry points, the preparation and merge kernels, and the
// warp-level form of the step for head_dim 64 or 64-key tiles: the tiles are streamed into a shared-memory
// ring by untiled bulk copies, and the H_q/H_k query rows of a KV head are the
// rows of a 16-row warp-level tensor-core operand.  head_dim 128 with 128-key tiles runs the tcgen05 form
// (decode_umma.cu), where the KEYS are the MMA rows.
#include <cuda_fp16.h>
#include <math.h>

#include "common.cuh"
#include "decode.cuh"
#include "ptx_sm100.cuh"

namespace tilemix {

namespace {

constexpr float kLog2e = 1.4426950408889634f;
constexpr float kLn2 = 0.6931471805599453f;

// Keys per kernel tile.  Head dimension 64: 128, i.e. one routing tile of 128 keys or two of 64 (each of the eight warps
// has a 16-key step of its own).  Head dimension 128 (64-key routing tiles): 64, two warps per step with half of the
// output columns each; a warp with all 128 columns needs more than its 128 registers (8 x 16K keys: 97 us, 118 that way).
template <int D>
constexpr int kChunk = D == 64 ? 128 : 64;

// Ring of kernel tiles in shared memory.  What bounds the step is the data in flight: two CTAs per SM with 96 KB each keep
// what the HBM latency asks for on the way (two stages before, 24 KB with 64-key tiles of dimension 64; that, two such
// tiles per kernel tile and the shares below: 16 sequences of up to 8K keys, 32 / 8 heads of 64, 67 -> 42 us).
constexpr int kRingBytes = 96 * 1024;
template <int D, bool F16K>
struct Stage {
    static constexpr int kK = kChunk<D> * D * (F16K ? 2 : 1);   // room for the FP16 copy of the keys, if there is one
    static constexpr int kV = kChunk<D> * D;
    static constexpr int kBytes = kK + kV;
    static constexpr int kStages = kRingBytes / kBytes;
};
constexpr int kMaxStages = 6;

// Sequence number n of the batch (0: the longest) by cache length in kernel tiles, equal ones in their order.  The grid
// takes the sequences in this order, so that it ends with the shortest CTAs; which keys a CTA gets does not depend on it.
// (Up to 8K keys each, 32 / 8 heads of 64: 16 sequences of four splits 50 us in the order of the batch, 42 so; 64 of up to
// 4K keys, one split each, 77 and 65.)
// Lane l holds the lengths of sequences l, l + 32, ...; a radix selection on (tiles, ~sequence), the same in every warp.
constexpr int kSortRows = 8, kMaxSorted = 32 * kSortRows;
template <int T>
__device__ __forceinline__ int nth_longest(const int32_t* __restrict__ cache_len, int B, int max_len, int n) {
    const int lane = threadIdx.x & 31, index_bits = B <= 32 ? 5 : 8, last = (1 << index_bits) - 1;
    uint32_t key[kSortRows], most = 0u, least = 0xffffffffu;      // (key 0: no such sequence)
#pragma unroll
    for (int k = 0; k < kSortRows; ++k) {
        const int b = lane + 32 * k;
        key[k] = 0u;
        if (b < B) {
            const uint32_t tiles = min((min(max(cache_len[b], 0), max_len) + T - 1) / T, (1 << 23) - 2);
            key[k] = (tiles + 1) << index_bits | static_cast<uint32_t>(last - b);
            most = max(most, key[k]);
            least = min(least, key[k]);
        }
    }
    most = __reduce_max_sync(0xffffffffu, most);
    least = __reduce_min_sync(0xffffffffu, least);
    if (most >> index_bits == least >> index_bits) return n;     // all of one length
    uint32_t found = 0u;
    for (int bit = 31 - __clz(most); bit >= 0; --bit) {
        const uint32_t want = (found >> bit) | 1u;
        int with_bit = (key[0] >> bit) == want ? 1 : 0;
        if (index_bits > 5) {
#pragma unroll
            for (int k = 1; k < kSortRows; ++k) with_bit += (key[k] >> bit) == want ? 1 : 0;
            with_bit = __reduce_add_sync(0xffffffffu, with_bit);
        } else {
            with_bit = __popc(__ballot_sync(0xffffffffu, with_bit));
        }
        if (n < with_bit) found |= 1u << bit; else n -= with_bit;
    }
    return last - static_cast<int>(found & static_cast<uint32_t>(last));
}

// ---- warp-level tensor-core MMAs (m16n8k32 INT8 / m16n8k16 FP16, FP32 or INT32 accumulators) ----------
// Lane l holds, with g = l / 4 and t = l % 4: A rows g (a0, a2) and g + 8 (a1, a3), B column g, C rows g
// (c0, c1) and g + 8 (c2, c3) at columns 2t, 2t + 1.  Only rows 0..R-1 of A are query rows here, so a1 and
// a3 are always zero and c2, c3 stay zero.
__device__ __forceinline__ void mma_s8(int (&c)[4], uint32_t a0, uint32_t a2, uint32_t b0, uint32_t b1) {
    asm volatile("mma.sync.aligned.m16n8k32.row.col.s32.s8.s8.s32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
                 : "+r"(c[0]), "+r"(c[1]), "+r"(c[2]), "+r"(c[3])
                 : "r"(a0), "r"(0u), "r"(a2), "r"(0u), "r"(b0), "r"(b1));
}
__device__ __forceinline__ void mma_f16(float (&c)[4], uint32_t a0, uint32_t a2, uint32_t b0, uint32_t b1) {
    asm volatile("mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
                 : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
                 : "r"(a0), "r"(0u), "r"(a2), "r"(0u), "r"(b0), "r"(b1));
}

// D: head dim; R: query heads per KV head; RT: keys per routing tile (= scale block); a kernel tile is T keys.
// Tiles are contiguous in the cache, so they are streamed into a ring of shared-memory stages with
// untiled bulk copies ("full" / "empty" mbarriers per stage), issued by one lane of the last warp
// before it turns to its own share of a tile.  The eight warps never synchronise with one another
// inside the loop: each one owns 16 keys of every tile and runs its own flash-decoding recurrence on them --
//  (1) scores S[R x 16] = Q K^T on the tensor cores, the R query rows being rows 0..R-1 of a 16-row A
//      operand.  The contraction index may be permuted freely as long as Q and K use the same
//      permutation, so lane t simply takes the 16-byte chunks t, t+4, ... of a row;
//  (2) running maximum and sum of its own keys (two shuffles per row), P = 2^(s - m) times delta_V,
//      rounded to FP16 -- the score fragment is already laid out as the A operand of the next product;
//  (3) O~[R x D] += P V8 on the tensor cores.  V8 is converted to FP16 in registers (exactly); the
//      output columns are permuted (column n of block nb is d = (D/8) n + nb) so that the bytes a
//      lane needs from a cached row are contiguous.
// After the loop the eight (m, z, O~) are merged in shared memory like splits.
constexpr int kConsumerWarps = 8;
constexpr int kDecodeThreads = kConsumerWarps * 32;   // 2 CTAs/SM = 4 warps per scheduler: 128 registers each

template <int D, int R, int RT, bool F16K>
__global__ void __launch_bounds__(kDecodeThreads, 2)
decode_kernel(const DecodeParams prm) {
    constexpr int T = kChunk<D>, SUBN = T / RT;   // routing tiles of a kernel tile
    using St = Stage<D, F16K>;
    constexpr int W8 = D / 16, W16 = D / 8;       // 32-bit words per lane and row: INT8 / FP16 operand
    constexpr int KS3 = T / 16;                   // 16-key steps of a tile
    constexpr int NSPLIT = kConsumerWarps / KS3;  // warps sharing one step (each takes some column blocks)
    constexpr int NBLK = D / 8 / NSPLIT;          // column blocks of 8 per warp
    constexpr int BPG = D / 8;                    // bytes of a cached V row per lane group
    static_assert(KS3 <= kConsumerWarps && kConsumerWarps % KS3 == 0, "tile shape vs warps");
    static_assert(kRingBytes >= static_cast<int>(kConsumerWarps * R * (D + 2) * sizeof(float)), "the final merge reuses the ring");
    static_assert(St::kStages <= kMaxStages, "barriers of the ring");
    const int hk = blockIdx.y;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int g = lane >> 2, t = lane & 3;
    const int split = blockIdx.x;
    // (lengths live on the device and cannot be checked by the host: out-of-range values are clamped.  This grid may run
    // beside the prepare kernel, so it clamps the caller's array itself, and waits for that kernel before it writes the
    // status record or ends.)
    const int b = prm.by_length ? nth_longest<T>(prm.cache_len, prm.B, prm.max_len, blockIdx.z) : blockIdx.z;
    const int len = min(max(prm.cache_len[b], 0), prm.max_len);
    const int n_tiles = (len + T - 1) / T;
    const int per_split = (n_tiles + prm.n_splits - 1) / prm.n_splits;
    const int t0 = split * per_split, t1 = min(n_tiles, t0 + per_split);

    extern __shared__ __align__(128) uint8_t ring[];   // n_stages x (K tile | V tile)
    constexpr int n_stages = St::kStages, k_slot = St::kK, stage_bytes = St::kBytes;
    __shared__ __align__(16) uint32_t qh[R][D / 2];   // query rows, FP16 pairs (FP16 route)
    __shared__ __align__(16) uint32_t q8w[R][D / 4];  // quantised query rows, 4 bytes per word (INT8 route)
    __shared__ float dq_s[R];
    __shared__ __align__(8) uint64_t full_bar[kMaxStages], empty_bar[kMaxStages];
    __shared__ int abort_flag;
    // route bit (sign) and the two block scales of the first kMetaTiles tiles of this split, staged once
    constexpr int kMetaTiles = 256;
    __shared__ float2 meta[kMetaTiles];   // x = delta_K (negative zero / negated: FP16 route), y = delta_V

    const uint32_t ring_u32 = ptx::smem_u32(ring);
    if (tid == 0) {
        for (int s = 0; s < n_stages; ++s) {
            ptx::mbar_init(ptx::smem_u32(&full_bar[s]), 1);
            ptx::mbar_init(ptx::smem_u32(&empty_bar[s]), kConsumerWarps);
        }
        abort_flag = 0;
        ptx::fence_mbar_init();
    }

    // ---- the query rows of this KV head: FP16 copy and blockwise INT8 (block = the row) ----------
    if (warp < R) {
        const int hq = hk * R + warp;
        const __half* qrow = prm.q + (static_cast<int64_t>(b) * prm.Hq + hq) * D;
        float v[D / 32];
        float amax = 0.f;
#pragma unroll
        for (int x = 0; x < D / 32; ++x) {
            v[x] = __half2float(qrow[lane + 32 * x]);
            amax = fmaxf(amax, fabsf(v[x]));
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) amax = fmaxf(amax, __shfl_xor_sync(0xffffffffu, amax, o));
        const float delta = __fdiv_rn(amax, 127.f);
#pragma unroll
        for (int x = 0; x < D / 32; ++x) {
            const int e = lane + 32 * x;
            int q8 = 0;
            if (amax > 0.f) q8 = max(-127, min(127, __float2int_rn(__fdiv_rn(v[x], delta))));
            reinterpret_cast<__half*>(&qh[warp][0])[e] = qrow[e];
            reinterpret_cast<int8_t*>(&q8w[warp][0])[e] = static_cast<int8_t>(q8);
            if (split == 0 && prm.q8_out != nullptr)
                prm.q8_out[(static_cast<int64_t>(b) * prm.Hq + hq) * D + e] = static_cast<int8_t>(q8);
        }
        if (lane == 0) {
            dq_s[warp] = delta;
            if (split == 0 && prm.qs_out != nullptr) prm.qs_out[static_cast<int64_t>(b) * prm.Hq + hq] = delta;
        }
    }

    const int64_t row_base = (static_cast<int64_t>(b) * prm.Hk + hk) * prm.max_len;
    const float* dk = prm.k_scale + (static_cast<int64_t>(b) * prm.Hk + hk) * prm.n_blk;
    const float* dv = prm.v_scale + (static_cast<int64_t>(b) * prm.Hk + hk) * prm.n_blk;
    const uint32_t* wrow = prm.words != nullptr
        ? prm.words + (static_cast<int64_t>(prm.nb == 1 ? 0 : b) * prm.Hk + hk) * prm.W : nullptr;
    auto route_of = [&](int rt) -> bool {      // of a routing tile
        if (wrow == nullptr) return false;
        const int grp = rt / prm.G;
        return (wrow[grp >> 5] >> (grp & 31)) & 1u;
    };
    // Bounded wait on a ring barrier; false when the CTA is giving up.
    auto wait_ring = [&](uint64_t* bar, uint32_t parity) -> bool {
        const uint32_t addr = ptx::smem_u32(bar);
        if (ptx::mbar_try_wait(addr, parity)) return true;
        const uint64_t start = ptx::globaltimer_ns();
        uint32_t spins = 0;
        while (!ptx::mbar_try_wait(addr, parity)) {
            if ((++spins & 63u) == 0u) {
                if (*reinterpret_cast<volatile int*>(&abort_flag)) return false;
                if (ptx::globaltimer_ns() - start > prm.wait_limit_ns) {
                    *reinterpret_cast<volatile int*>(&abort_flag) = 1;
                    return false;
                }
            }
        }
        return true;
    };
    // routing tiles of this split (the last kernel tile of a row may have one only)
    const int rt0 = t0 * SUBN, rt1 = min(t1 * SUBN, (len + RT - 1) / RT);
    for (int i = tid; i < kMetaTiles && rt0 + i < rt1; i += kDecodeThreads) {
        const int rt = rt0 + i;
        // delta_K >= 0; the FP16 route is marked by a negative x (its delta_K is not used)
        meta[i] = make_float2(route_of(rt) ? dk[rt] : -1.f, dv[rt]);
    }
    if constexpr (!F16K) {
        // This instance was chosen because no FP16 key cache was passed: every group inside the cache length has
        // to be INT8-routed.  A 0 bit is found here, before any copy is started; the CTA records it and leaves
        // (no access is made, nothing is in flight).
        int fp16_group = 0;
        for (int rt = rt0 + tid; rt < rt1; rt += kDecodeThreads) fp16_group |= route_of(rt) ? 0 : 1;
        if (__syncthreads_or(fp16_group)) {
            ptx::griddep_wait();
            if (tid == 0 && atomicCAS(&prm.status[0], 0, TILEMIX_ERR_NULL) == 0) {
                prm.status[1] = 16; prm.status[2] = t0; prm.status[3] = 1;
            }
            return;
        }
    } else {
        __syncthreads();   // barriers initialised, query rows and tile metadata staged
    }
    ptx::griddep_launch_dependents();     // a merge kernel may be brought in; it waits for this grid to finish

    // per-warp flash-decoding state: rows g (< R) of this warp's keys
    float m_run = -INFINITY, z_part = 0.f;          // z_part: this lane's share of the row sum
    float acc[NBLK][2];                             // O~ rows g, columns 2t, 2t+1 of this warp's blocks
#pragma unroll
    for (int nb = 0; nb < NBLK; ++nb) acc[nb][0] = acc[nb][1] = 0.f;

    // Refill of the ring by one lane (of the last warp): tile `tile` into its stage, after every warp
    // has handed that stage back.  Returns false when the CTA is giving up.
    const int8_t* k8 = prm.k8 + row_base * D;
    const int8_t* v8 = prm.v8 + row_base * D;
    const __half* k16 = prm.k16 != nullptr ? prm.k16 + row_base * D : nullptr;
    int last_produced = -1;   // (producer lane) the last tile whose copies were started
    auto produce = [&](int tile) -> bool {
        const int it = tile - t0, stage = it % n_stages;
        if (it == prm.test_drop_tile) return true;   // testing aid: this tile never lands, the consumers' bounded wait runs out
        // the first pass over the ring finds every stage free
        if (it >= n_stages && !wait_ring(&empty_bar[stage], ((it / n_stages) - 1) & 1)) return false;
        const int rows = min(T, len - tile * T);   // only rows that exist
        const uint32_t bar = ptx::smem_u32(&full_bar[stage]);
        const uint32_t dst = ring_u32 + stage * stage_bytes;
        uint32_t kbytes[SUBN], bytes = rows * D;
        bool int8[SUBN];
#pragma unroll
        for (int i = 0; i < SUBN; ++i) {
            const int r = max(0, min(RT, rows - i * RT));
            int8[i] = r > 0 && route_of(tile * SUBN + i);
            kbytes[i] = r * D * (int8[i] ? 1 : 2);
            bytes += kbytes[i];
        }
        ptx::mbar_arrive_expect_tx(bar, bytes);
#pragma unroll
        for (int i = 0; i < SUBN; ++i) {
            const int64_t at = static_cast<int64_t>(tile * SUBN + i) * RT * D;
            const uint32_t kdst = dst + i * (k_slot / SUBN);
            if (kbytes[i] == 0u) continue;
            if (int8[i]) ptx::bulk_load_1d(kdst, k8 + at, kbytes[i], bar);
            else ptx::bulk_load_1d(kdst, k16 + at, kbytes[i], bar);
        }
        ptx::bulk_load_1d(dst + k_slot, v8 + static_cast<int64_t>(tile) * T * D, rows * D, bar);
        last_produced = tile;
        return true;
    };
    const bool producer = warp == kConsumerWarps - 1 && lane == 0;
    // tiles asked for ahead of the one in work: with a deep ring one less than fits, so that the producing warp does
    // not wait for the slowest warp to hand back the tile it has itself just finished
    constexpr int kAhead = n_stages > 3 ? n_stages - 2 : n_stages - 1;
    if (producer)
        for (int s = 0; s < kAhead && t0 + s < t1; ++s) produce(t0 + s);
    {
        // ================================================================ consumers
        const int ks = warp / NSPLIT, nb0 = (warp % NSPLIT) * NBLK;   // this warp's keys (16 ks ..) and column blocks
        const bool counts_z = (warp % NSPLIT) == 0;                    // one warp per key step sums z
        const int sub = 16 * ks / RT, key_in_rt = 16 * ks - sub * RT;  // the keys' routing tile of the kernel tile
        // A fragments of the INT8 route: lane t's words of query row g, in the order the K words are used
        uint32_t qa8[W8];
#pragma unroll
        for (int wi = 0; wi < W8; ++wi) qa8[wi] = g < R ? q8w[g < R ? g : 0][4 * (t + 4 * (wi / 4)) + (wi % 4)] : 0u;
        const float dq = g < R ? dq_s[g < R ? g : 0] : 0.f;

        for (int tile = t0; tile < t1; ++tile) {
            const int it = tile - t0, stage = it % n_stages;
            if (producer && tile + kAhead < t1) produce(tile + kAhead);   // keeps the ring full
            // route bit and block scales: from shared memory (global loads for tiles beyond the staged ones)
            bool int8;
            float dkt, dvt;
            const int rt = tile * SUBN + sub;
            if (rt >= rt1) {               // (no such keys: all are masked below)
                int8 = true;
                dkt = dvt = 0.f;
            } else if (rt - rt0 < kMetaTiles) {
                const float2 mt = meta[rt - rt0];
                int8 = mt.x >= 0.f;
                dkt = mt.x;
                dvt = mt.y;
            } else {
                int8 = route_of(rt);
                dkt = int8 ? dk[rt] : 0.f;
                dvt = dv[rt];
            }
            if (!wait_ring(&full_bar[stage], (it / n_stages) & 1)) break;
            const uint8_t* vst = ring + stage * stage_bytes + k_slot;
            const uint8_t* kst = ring + stage * stage_bytes + sub * (k_slot / SUBN);
            // ---- (1) scores of this warp's 16 keys, rows g: s[nb][0..1] = keys 8 nb + 2t, 2t + 1 ----------
            float sc[2][2];
            if (int8) {
                const float a = prm.scale_log2 * dq * dkt;
#pragma unroll
                for (int nb = 0; nb < 2; ++nb) {
                    const uint8_t* krow = kst + (key_in_rt + 8 * nb + g) * D;       // B column g = that key
                    uint32_t kw[W8];
#pragma unroll
                    for (int ch = 0; ch < W8 / 4; ++ch) {
                        const uint4 q = *reinterpret_cast<const uint4*>(krow + 16 * (t + 4 * ch));
                        kw[4 * ch] = q.x; kw[4 * ch + 1] = q.y; kw[4 * ch + 2] = q.z; kw[4 * ch + 3] = q.w;
                    }
                    int c[4] = {0, 0, 0, 0};
#pragma unroll
                    for (int k = 0; k < W8 / 2; ++k) mma_s8(c, qa8[2 * k], qa8[2 * k + 1], kw[2 * k], kw[2 * k + 1]);
                    sc[nb][0] = static_cast<float>(c[0]) * a;
                    sc[nb][1] = static_cast<float>(c[1]) * a;
                }
            } else {
                uint32_t qa16[W16];
#pragma unroll
                for (int ch = 0; ch < W16 / 4; ++ch) {
                    uint4 q = make_uint4(0u, 0u, 0u, 0u);
                    if (g < R) q = *reinterpret_cast<const uint4*>(&qh[g < R ? g : 0][4 * (t + 4 * ch)]);
                    qa16[4 * ch] = q.x; qa16[4 * ch + 1] = q.y; qa16[4 * ch + 2] = q.z; qa16[4 * ch + 3] = q.w;
                }
#pragma unroll
                for (int nb = 0; nb < 2; ++nb) {
                    const uint8_t* krow = kst + (key_in_rt + 8 * nb + g) * D * 2;
                    float c[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
                    for (int ch = 0; ch < W16 / 4; ++ch) {
                        const uint4 q = *reinterpret_cast<const uint4*>(krow + 16 * (t + 4 * ch));
                        mma_f16(c, qa16[4 * ch], qa16[4 * ch + 1], q.x, q.y);
                        mma_f16(c, qa16[4 * ch + 2], qa16[4 * ch + 3], q.z, q.w);
                    }
                    sc[nb][0] = c[0] * prm.scale_log2;
                    sc[nb][1] = c[1] * prm.scale_log2;
                }
            }
            // keys beyond the cached length (stale shared memory) do not exist
            const int j0 = tile * T + 16 * ks + 2 * t;
#pragma unroll
            for (int nb = 0; nb < 2; ++nb) {
                if (j0 + 8 * nb >= len) sc[nb][0] = -INFINITY;
                if (j0 + 8 * nb + 1 >= len) sc[nb][1] = -INFINITY;
            }
            // ---- (2) this warp's online softmax over its own keys ------------------------------------------
            float tmax = fmaxf(fmaxf(sc[0][0], sc[0][1]), fmaxf(sc[1][0], sc[1][1]));
            tmax = fmaxf(tmax, __shfl_xor_sync(0xffffffffu, tmax, 1));
            tmax = fmaxf(tmax, __shfl_xor_sync(0xffffffffu, tmax, 2));
            const float m_new = fmaxf(m_run, tmax);
            // a warp whose 16 keys of this tile all lie beyond the cache keeps its state (m_new may be -inf)
            const float m_use = m_new == -INFINITY ? 0.f : m_new;
            const float alpha = exp2f(m_run - m_use);        // 0 on the first keys, 1 if the maximum stands
            float p[2][2];
#pragma unroll
            for (int nb = 0; nb < 2; ++nb) {
                p[nb][0] = exp2f(sc[nb][0] - m_use);
                p[nb][1] = exp2f(sc[nb][1] - m_use);
            }
            z_part = z_part * alpha + ((p[0][0] + p[0][1]) + (p[1][0] + p[1][1]));
            m_run = m_new;
            if (__any_sync(0xffffffffu, alpha != 1.f)) {
#pragma unroll
                for (int nb = 0; nb < NBLK; ++nb) { acc[nb][0] *= alpha; acc[nb][1] *= alpha; }
            }
            // P x delta_V, FP16: the score fragment (row g, keys 2t, 2t+1 of each 8-key block) is the A
            // fragment of the PV product over these 16 keys
            const __half2 h0 = __floats2half2_rn(p[0][0] * dvt, p[0][1] * dvt);
            const __half2 h2 = __floats2half2_rn(p[1][0] * dvt, p[1][1] * dvt);
            const uint32_t pa0 = g < R ? *reinterpret_cast<const uint32_t*>(&h0) : 0u;
            const uint32_t pa2 = g < R ? *reinterpret_cast<const uint32_t*>(&h2) : 0u;
            // ---- (3) O~ += P V8 ------------------------------------------------------------------------------
            // the four cached rows whose pairs this lane feeds: keys 2t, 2t+1 and 2t+8, 2t+9 of the step,
            // at this lane group's columns of this warp's blocks
            const uint8_t* vbase = vst + (16 * ks + 2 * t) * D + BPG * g + nb0;
            const __half2 off = __floats2half2_rn(1152.f, 1152.f);
#pragma unroll
            for (int w = 0; w < NBLK / 4; ++w) {
                // four column blocks at a time: one 32-bit word of each of the four rows
                uint32_t u[4];
#pragma unroll
                for (int r4 = 0; r4 < 4; ++r4)
                    u[r4] = *reinterpret_cast<const uint32_t*>(vbase + ((r4 & 1) + (r4 >> 1) * 8) * D + 4 * w) ^ 0x80808080u;
                if (w == NBLK / 4 - 1) {
                    // last read of this stage by this warp: hand the stage back
                    __syncwarp();
                    if (lane == 0) ptx::mbar_arrive(ptx::smem_u32(&empty_bar[stage]));
                }
                // bytes of rows (k0, k1) and (k2, k3) interleaved: {k0[e], k1[e]} pairs for e = 0..3
                const uint32_t lo01 = __byte_perm(u[0], u[1], 0x5140), hi01 = __byte_perm(u[0], u[1], 0x7362);
                const uint32_t lo23 = __byte_perm(u[2], u[3], 0x5140), hi23 = __byte_perm(u[2], u[3], 0x7362);
#pragma unroll
                for (int e = 0; e < 4; ++e) {
                    const uint32_t s01 = e < 2 ? lo01 : hi01, s23 = e < 2 ? lo23 : hi23;
                    const uint32_t sel = (e & 1) ? 0x4342u : 0x4140u;
                    // half2(1024 + (x + 128)) - 1152 = half2(x), exactly
                    uint32_t b0 = __byte_perm(s01, 0x64646464u, sel), b1 = __byte_perm(s23, 0x64646464u, sel);
                    const __half2 v0 = __hsub2(*reinterpret_cast<const __half2*>(&b0), off);
                    const __half2 v1 = __hsub2(*reinterpret_cast<const __half2*>(&b1), off);
                    // rows g + 8 of the product do not exist: their accumulators start at 0 and are dropped, so
                    // that the MMAs of different column blocks do not depend on one another
                    float c[4] = {acc[4 * w + e][0], acc[4 * w + e][1], 0.f, 0.f};
                    mma_f16(c, pa0, pa2, *reinterpret_cast<const uint32_t*>(&v0), *reinterpret_cast<const uint32_t*>(&v1));
                    acc[4 * w + e][0] = c[0]; acc[4 * w + e][1] = c[1];
                }
            }
            if (!counts_z) z_part = 0.f;   // the row sum of a key step is counted by one of its warps
        }
    }

    // ---- merge of the eight warps; the row's only split writes the output, others (m, z, O~) to the workspace -----
    __syncthreads();   // every warp is out of the ring (all copies it waited for have landed)
    // The prepare kernel has completed before this grid does, and before the row's counter is used: a merge kernel waits for
    // this grid only, and what the stream runs behind it may read the status record or use the workspace again.
    ptx::griddep_wait();
    if (*reinterpret_cast<volatile int*>(&abort_flag)) {
        if (tid == 0 && atomicCAS(&prm.status[0], 0, TILEMIX_ERR_DEVICE_TIMEOUT) == 0) {
            prm.status[1] = 16; prm.status[2] = t0; prm.status[3] = 0;
        }
        // the copies still in flight land before this CTA's shared memory is given back (each stage's latest one)
        if (producer) {
            for (int tile = max(t0, last_produced - n_stages + 1); tile <= last_produced; ++tile) {
                const int it = tile - t0;
                if (it == prm.test_drop_tile) continue;
                for (int spin = 0; spin < (1 << 16); ++spin)
                    if (ptx::mbar_try_wait(ptx::smem_u32(&full_bar[it % n_stages]), (it / n_stages) & 1)) break;
            }
        }
        return;
    }
    float (*red)[R][D + 2] = reinterpret_cast<float (*)[R][D + 2]>(ring);   // per warp and row: O~[D], m, z
    {
        const int nb0 = (warp % NSPLIT) * NBLK;
        if constexpr (NSPLIT > 1) {
            // warps of one key step hold disjoint column blocks: zero the rest of this warp's plane first
            for (int idx = lane; idx < R * D; idx += 32) red[warp][idx / D][idx % D] = 0.f;
            __syncwarp();
        }
        float z = z_part;
        z += __shfl_xor_sync(0xffffffffu, z, 1);
        z += __shfl_xor_sync(0xffffffffu, z, 2);
        if (g < R) {
#pragma unroll
            for (int nb = 0; nb < NBLK; ++nb) {
                // column n of block nb is d = (D/8) n + nb; this lane holds n = 2t, 2t+1
                red[warp][g][BPG * (2 * t) + nb0 + nb] = acc[nb][0];
                red[warp][g][BPG * (2 * t + 1) + nb0 + nb] = acc[nb][1];
            }
            if (t == 0) { red[warp][g][D] = m_run; red[warp][g][D + 1] = z; }
        }
    }
    __syncthreads();
    for (int idx = tid; idx < R * D; idx += kDecodeThreads) {
        const int r = idx / D, e = idx - r * D;
        float m = -INFINITY;
#pragma unroll
        for (int w = 0; w < kConsumerWarps; ++w) m = fmaxf(m, red[w][r][D]);
        float o = 0.f, z = 0.f;
        if (m > -INFINITY) {
#pragma unroll
            for (int w = 0; w < kConsumerWarps; ++w) {
                const float mw = red[w][r][D];
                if (mw == -INFINITY) continue;
                const float wgt = exp2f(mw - m);
                o += red[w][r][e] * wgt;
                z += red[w][r][D + 1] * wgt;
            }
        }
        const int64_t head = static_cast<int64_t>(b) * prm.Hq + hk * R + r, part = head * prm.n_splits + split;
        if (prm.n_splits == 1) {
            prm.out[head * D + e] = __float2half_rn(z > 0.f ? o / z : 0.f);
            if (e == 0 && prm.lse != nullptr) prm.lse[head] = z > 0.f ? (m + log2f(z)) * kLn2 : -INFINITY;
        } else {
            prm.o_part[part * D + e] = o;
            if (e == 0) { prm.m_part[part] = m; prm.z_part[part] = z; }
        }
    }
    if (prm.fused && prm.n_splits > 1) merge_if_last<D, R, kDecodeThreads>(prm, b, hk, prm.n_splits, prm.n_splits);
}

// Merge as a kernel of its own (grids of several waves, see tilemix_decode_int8kv): one block per query head, one thread per
// output column.
template <int D>
__global__ void __launch_bounds__(D)
decode_merge_kernel(const DecodeParams prm) {
    ptx::griddep_wait();   // (when launched as a programmatic dependent of the step kernel)
    merge_columns<D, 1>(prm, blockIdx.x, prm.n_parts, threadIdx.x);
}

// Step and merge overlap the tail of the kernel before them (programmatic dependent launch).
template <int D>
int launch_merge(const DecodeParams& prm, cudaStream_t stream) {
    if (prm.fused) return TILEMIX_OK;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(prm.B * prm.Hq); cfg.blockDim = dim3(D); cfg.stream = stream;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr; cfg.numAttrs = 1;
    const cudaError_t e = cudaLaunchKernelEx(&cfg, decode_merge_kernel<D>, prm);
    g_launch_count.fetch_add(1);
    return static_cast<int>(e);
}

template <int D, int R, int RT>
int launch_cfg(const DecodeParams& prm, cudaStream_t stream) {
    // no FP16 key cache: the instance whose ring holds INT8 keys only
    auto kernel = prm.k16 != nullptr ? decode_kernel<D, R, RT, true> : decode_kernel<D, R, RT, false>;
    cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kRingBytes);
    if (e != cudaSuccess) return static_cast<int>(e);
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(prm.n_splits, prm.Hk, prm.B);
    cfg.blockDim = dim3(kDecodeThreads); cfg.dynamicSmemBytes = kRingBytes; cfg.stream = stream;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr; cfg.numAttrs = 1;
    e = cudaLaunchKernelEx(&cfg, kernel, prm);
    g_launch_count.fetch_add(1);
    if (e != cudaSuccess) return static_cast<int>(e);
    return launch_merge<D>(prm, stream);
}

template <int D, int RT>
int launch_r(int R, const DecodeParams& prm, cudaStream_t stream) {
    switch (R) {
        case 1: return launch_cfg<D, 1, RT>(prm, stream);
        case 2: return launch_cfg<D, 2, RT>(prm, stream);
        case 4: return launch_cfg<D, 4, RT>(prm, stream);
        case 8: return launch_cfg<D, 8, RT>(prm, stream);
        default: return TILEMIX_ERR_UNSUPPORTED;
    }
}

constexpr size_t kDecodeStatusBytes = 256;   // status record of the bounded waits
constexpr int kDecodeWave = 148;             // CTAs of one wave of the tcgen05 form (one per SM)
constexpr int kDecodeBalanceRows = 160;      // rows of a batch whose splits that kernel can balance

// Before the step: clears the status record and the rows' counters behind it.  (The cache lengths live on the device, so the
// host cannot check them: the step clamps each to [0, max_len] as it reads it.)
__global__ void decode_prepare_kernel(int* status, int n) {
    ptx::griddep_launch_dependents();   // the step kernel may start meanwhile; it waits before it uses either or ends
    for (int i = threadIdx.x; i < n; i += blockDim.x) status[i] = 0;
}

// Behind the status record (it held a copy of the lengths): room for counters.  The size of a workspace stays what it was.
size_t decode_len_bytes(int B) { return (static_cast<size_t>(B) * sizeof(int32_t) + 255) / 256 * 256; }

struct DecodeGeometry {
    int n_blk, T_mask, W, n_splits;
    int k_tiles;            // kernel tiles of a row of max_len keys
    int n_parts;            // partial results per query head in the workspace (the tcgen05 form writes two per split)
    int balanced, n_ctas, split_cap;   // tcgen05 form with an automatic split count: see DecodeParams
    size_t o_bytes, mz_bytes;
};

int resolve_decode(const tilemix_decode_t* p, DecodeGeometry* g) {
    if (p == nullptr) return TILEMIX_ERR_NULL;
    if (p->batch <= 0 || p->heads_q <= 0 || p->heads_kv <= 0 || p->head_dim <= 0 || p->max_len <= 0 ||
        p->tile_n <= 0 || p->group <= 0 || p->n_splits < -1)
        return TILEMIX_ERR_SHAPE;
    if (p->heads_q % p->heads_kv != 0) return TILEMIX_ERR_SHAPE;
    if (p->mask_batch != 1 && p->mask_batch != p->batch) return TILEMIX_ERR_SHAPE;
    const int R = p->heads_q / p->heads_kv;
    if ((p->head_dim != 64 && p->head_dim != 128) || (p->tile_n != 64 && p->tile_n != 128) ||
        (R != 1 && R != 2 && R != 4 && R != 8))
        return TILEMIX_ERR_UNSUPPORTED;
    g->n_blk = static_cast<int>(ceil_div(p->max_len, p->tile_n));
    g->T_mask = static_cast<int>(ceil_div(p->max_len, static_cast<int64_t>(p->group) * p->tile_n));
    g->W = static_cast<int>(ceil_div(g->T_mask, 32));
    // n_splits: > 0 as given, 0 chosen here (the same for every row), -1 chosen here and, where the kernel can do
    // it, shared out over the rows by the kernel
    const bool balance = p->n_splits == -1;
    int splits = balance ? 0 : p->n_splits;
    const bool umma = p->head_dim == 128 && p->tile_n == 128;   // the tcgen05 form of the step (decode_umma.cu)
    const int k_tiles = umma ? g->n_blk : static_cast<int>(ceil_div(p->max_len, p->head_dim == 64 ? kChunk<64> : kChunk<128>));
    g->balanced = 0; g->n_ctas = 0; g->split_cap = 0;
    if (splits == 0) {
        if (umma) {
            // one CTA per SM, HBM-bound once every SM streams: a single wave, as many splits as fit into it
            // (measured at 8 x 8 KV heads and 32K keys: 2 splits = 128 CTAs 104 us, 9 splits = 3.9 waves 123 us),
            // at least four key tiles per split
            const int64_t n_rows = static_cast<int64_t>(p->batch) * p->heads_kv;
            const int64_t want = kDecodeWave / n_rows;
            splits = static_cast<int>(want < 1 ? 1 : want);
            const int cap = g->n_blk / 4 > 0 ? g->n_blk / 4 : 1;
            if (splits > cap) splits = cap;
            // On request, for a batch whose rows fit one wave: the kernel shares the wave's CTAs out by the rows'
            // cost (cache length, FP16-routed groups), up to split_cap to a row; the workspace has room for that
            // many.  Not the default: rows of one length get the same number of CTAs that way, or two waves of them, and
            // pay for the sharing out (us uniform / shared out: 8 x 8 rows of 32K keys 110 / 118, of 8K 39 / 45, 4 x 8 of 32K
            // 63 / 71, 16 x 8 of 12K 80 / 107, one sequence of 64K 43 / 49); and which keys a CTA gets then depends on the
            // lengths beside it.
            if (balance && n_rows <= kDecodeWave && n_rows <= kDecodeBalanceRows) {
                int row_cap = 8 * splits < 16 ? 16 : 8 * splits;
                if (row_cap > cap) row_cap = cap;
                // With more rows than half a wave a single wave cannot split the long ones: two waves then.
                // (16 x 8 rows, lengths uniform in [0, 12K]: 82.7 us in one wave, 76.5 in two; the warp-level form 85.)
                const int64_t most = 2 * n_rows > kDecodeWave ? 2 * kDecodeWave : kDecodeWave;
                const int64_t ctas = n_rows * row_cap < most ? n_rows * row_cap : most;
                g->balanced = 1; g->n_ctas = static_cast<int>(ctas); g->split_cap = row_cap;
            }
        } else {
            // Two CTAs per SM, in one wave or -- batches of long sequences -- two (a third, partial one idles a quarter of the
            // GPU), with at least two kernel tiles per split.  A CTA costs its set-up, drain and partial result, which one
            // wave pays once; two waves of shorter CTAs even out unequal lengths.  The line is where a CTA of the second
            // form has twelve kernel tiles.  us in one wave and in two, lengths equal / uniform in [0, max]: d = 64,
            // 50 rows x 5000 keys (3.6 tiles) 28 / 26 and 32 / 30; 72 x 8000 (7.9) 36 / 32 and 42 / 32; 200 x 3000 (12)
            // 46 / 42 and 50 / 30; 64 x 16384 (14) 60 / 48 and 64 / 40; 128 x 8192 (16) 58 / 52 and 64 / 42; d = 128:
            // 48 x 4000 (5.2) 32 / 26 and 38 / 30; 32 x 12000 (10) 46 / 36 and 56 / 38; 64 x 16384 (28) 101 / 75 and
            // 101 / 60.  One sequence has nothing to even out: 8 rows x 65536 keys 44 and 56.
            const int64_t rows = static_cast<int64_t>(p->batch) * p->heads_kv, wave = 2 * kDecodeWave;
            int64_t want = 2 * wave / rows;
            if (p->batch == 1 || k_tiles < 12 * (want < 1 ? 1 : want)) want = wave / rows;
            const int cap = k_tiles / 2 > 0 ? k_tiles / 2 : 1;
            if (want > cap) want = cap;
            splits = static_cast<int>(want < 1 ? 1 : want);
        }
    }
    if (splits > g->n_blk) splits = g->n_blk;
    if (splits > 65535) return TILEMIX_ERR_UNSUPPORTED;
    if (splits > k_tiles) splits = k_tiles;      // a split is whole kernel tiles: more of them would only be empty CTAs
    g->n_splits = splits;
    g->k_tiles = k_tiles;
    g->n_parts = umma ? 2 * (g->balanced ? g->split_cap : splits) : splits;
    const size_t rows = static_cast<size_t>(p->batch) * p->heads_q * g->n_parts;
    g->o_bytes = (rows * p->head_dim * sizeof(float) + 255) / 256 * 256;
    g->mz_bytes = (rows * sizeof(float) + 255) / 256 * 256;
    return TILEMIX_OK;
}

}  // namespace
}  // namespace tilemix

using namespace tilemix;

extern "C" {

size_t tilemix_decode_workspace_size(const tilemix_decode_t* p) {
    DecodeGeometry g;
    if (resolve_decode(p, &g)) return 0;
    return kDecodeStatusBytes + decode_len_bytes(p->batch) + g.o_bytes + 2 * g.mz_bytes;
}

int tilemix_decode_int8kv(const tilemix_decode_t* p, const void* q_f16, const void* k_f16, const int8_t* k_i8,
                          const float* k_scale, const int8_t* v_i8, const float* v_scale,
                          const uint32_t* mask_words, const int32_t* cache_len, void* out_f16, float* lse,
                          int8_t* q_i8_out, float* q_scale_out, void* workspace, size_t workspace_bytes,
                          void* stream) {
    DecodeGeometry g;
    int rc = resolve_decode(p, &g);
    if (rc) return rc;
    if (!q_f16 || !k_i8 || !k_scale || !v_i8 || !v_scale || !cache_len || !out_f16 || !workspace) return TILEMIX_ERR_NULL;
    if (mask_words == nullptr && k_f16 == nullptr) return TILEMIX_ERR_NULL;   // all FP16 needs the FP16 cache
    if (!aligned16(q_f16) || !aligned16(k_i8) || !aligned16(v_i8) || !aligned16(out_f16) || !aligned16(workspace) ||
        (k_f16 && !aligned16(k_f16)))
        return TILEMIX_ERR_ALIGN;
    if (workspace_bytes < kDecodeStatusBytes + decode_len_bytes(p->batch) + g.o_bytes + 2 * g.mz_bytes) return TILEMIX_ERR_WORKSPACE;
    DecodeParams prm{};
    prm.B = p->batch; prm.Hq = p->heads_q; prm.Hk = p->heads_kv; prm.max_len = p->max_len; prm.G = p->group;
    prm.nb = p->mask_batch; prm.W = g.W; prm.n_splits = g.n_splits; prm.n_blk = g.n_blk;
    prm.n_parts = g.n_parts; prm.balanced = g.balanced; prm.n_rows = p->batch * p->heads_kv;
    prm.n_ctas = g.n_ctas; prm.split_cap = g.split_cap;
    prm.by_length = p->batch > 1 && p->batch <= kMaxSorted ? 1 : 0;
    const float scale = p->softmax_scale > 0.f ? p->softmax_scale : 1.0f / sqrtf(static_cast<float>(p->head_dim));
    prm.scale_log2 = scale * kLog2e;
    prm.q = static_cast<const __half*>(q_f16);
    prm.k16 = static_cast<const __half*>(k_f16);
    prm.k8 = k_i8; prm.k_scale = k_scale; prm.v8 = v_i8; prm.v_scale = v_scale;
    prm.words = mask_words;
    prm.status = static_cast<int*>(workspace);
    prm.wait_limit_ns = g_wait_limit_ns.load();
    prm.test_drop_tile = g_test_drop.load() == 2 ? 1 : -1;
    prm.cache_len = cache_len;
    uint8_t* ws = static_cast<uint8_t*>(workspace) + kDecodeStatusBytes + decode_len_bytes(p->batch);
    prm.o_part = reinterpret_cast<float*>(ws);
    prm.m_part = reinterpret_cast<float*>(ws + g.o_bytes);
    prm.z_part = reinterpret_cast<float*>(ws + g.o_bytes + g.mz_bytes);
    prm.q8_out = q_i8_out; prm.qs_out = q_scale_out;
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    const int R = p->heads_q / p->heads_kv;
    prm.out = static_cast<__half*>(out_f16);
    prm.lse = lse;
    // A row with one CTA needs no merge: that CTA writes the output, out of shared memory (warp-level form) or tensor memory
    // (with partial results and a merge kernel / so, us: 64 x 500 keys, 8 heads of 64 25.4 / 23.3; 40 x 3000, 64 / 32 heads of
    // 64 97 / 94; 48 x 1500, 32 / 8 heads of 128 in 64-key tiles 43.8 / 41.0; in 128-key tiles 64 x 2000 60.4 / 58.2, 16 x
    // 16000 111.5 / 109.6).
    // Of a row with more CTAs the last one merges at its end, where they start together (one wave; the shared-out form, in
    // its two waves too: 16 ragged sequences 76.5 / 74.6) and are more than two: no third kernel behind the end of the grid.
    // us with the merge kernel and so (calls in one CUDA graph), 128-key tiles of 128: one sequence, 8 KV heads, four query
    // heads each, 8000 keys 19.6 / 19.1, 40000 keys 35.5 / 34.7, eight each 42.2 / 40.6; 12 x 2500 keys, 4 KV heads 20.5 /
    // 20.0; heads of 64: one sequence, 3072 keys 9.7 / 9.1, 42 rows x 5000 keys, eight query heads 18.6 / 17.6.  Two splits:
    // 64 rows x 2048 keys, 128-key tiles of 128 19.5 / 18.6, x 4096 28.3 / 28.2, 128 rows x 2048 keys of 64 17.75 / 18.1, x
    // 8192 48.3 / 48.3: those keep the kernel.  So do three and four splits of two kernel tiles in the warp-level form: so
    // short a step ends before the merge has got under way (one sequence, 384 keys of 128 in 64-key tiles 8.7 / 9.6, 768
    // keys of 64 8.2 / 9.0).  In a grid of several waves the merge at the end of a CTA holds up the one behind it: 64 x 2000
    // keys 60.4 / 62.7, 32 x 4000, 32 KV heads 137 / 146.  Every row merged so has a counter behind the status record.
    const bool umma = p->head_dim == 128 && p->tile_n == 128;
    const int64_t ctas = static_cast<int64_t>(g.n_splits) * prm.n_rows, wave = umma ? kDecodeWave : 2 * kDecodeWave;
    const bool in_step = g.n_splits > 2 && ctas <= wave && (umma || g.n_splits > 4 || g.k_tiles > 2 * g.n_splits);
    const bool counted = g.balanced || in_step;
    // 16 bits a row, of at most one wave's rows: the shared-out form has no more, more than two splits in two waves are 98
    static_assert(4 + (kDecodeWave + 1) / 2 <= static_cast<int>(kDecodeStatusBytes + 256) / 4, "the counters lie behind the status record");
    const int n_words = (prm.n_rows + 1) / 2;
    prm.fused = counted || (!g.balanced && g.n_splits == 1) ? 1 : 0;
    prm.arrived = reinterpret_cast<uint32_t*>(prm.status) + 4;
    decode_prepare_kernel<<<1, counted ? 128 : 32, 0, s>>>(prm.status, counted ? 4 + n_words : 4);
    g_launch_count.fetch_add(1);
    cudaError_t pe = cudaGetLastError();
    if (pe != cudaSuccess) return static_cast<int>(pe);
    if (umma) {
        // the tcgen05 form of the step (decode_umma.cu); a step that has written its outputs gets no merge kernel
        rc = launch_decode_umma(R, prm, s);
        if (rc) return rc;
        return launch_merge<128>(prm, s);
    }
    if (p->head_dim == 128 && p->tile_n == 64) return launch_r<128, 64>(R, prm, s);
    if (p->head_dim == 64 && p->tile_n == 128) return launch_r<64, 128>(R, prm, s);
    if (p->head_dim == 64 && p->tile_n == 64) return launch_r<64, 64>(R, prm, s);
    return TILEMIX_ERR_UNSUPPORTED;
}

}  // extern "C"

// Routing-mask packer (Sec. 4.2, "Bitmask packing"; App. B, "Coverage Accounting"): turns the
// byte map R[nb, h_k, m, g] into rows of W little-endian uint32 words with bit g = R, and
// counts legal and INT8-routed groups per (nb, h_k).  Causal legality is applied here so the
// packed form is canonical: groups with no legal pair, pad bits and (optionally) diagonal
// groups are written as 0.
#include <cooperative_groups.h>

#include "common.cuh"

namespace tilemix {

namespace {

constexpr int kThreads = 512;
constexpr int kUnroll = 4;         // words per warp and round
constexpr int kStagedSeqs = 512;   // sequences (and one) whose offsets are staged in shared memory

// One warp makes a word: lane t reads the byte of group 32 w + t (a coalesced piece of the row), one vote is the word.
// Bound by the latency of those reads, so a (mask batch, KV head) gets a cluster of up to eight CTAs, kUnroll words per
// warp are in flight together, and words above the diagonal are not read.  The counts of a cluster meet in its first
// CTA's shared memory.  (One thread per word, 32 dependent byte loads each, and one CTA per head: 69 us for 8 heads of
// 1024 x 128 groups; now 24.)
template <bool CLUSTER>
__global__ void __launch_bounds__(kThreads)
pack_kernel(const uint8_t* __restrict__ route, int L_dense, int tile_m, int tile_n, int G, int T_m,
            int T_mask, int W, int pin_diag, uint32_t* __restrict__ words,
            unsigned long long* __restrict__ counts, const int32_t* tok, const int32_t* tile_off, int n_seqs) {
    namespace cg = cooperative_groups;
    cg::cluster_group cluster = cg::this_cluster();
    const int n_ctas = CLUSTER ? static_cast<int>(cluster.num_blocks()) : 1, rank = CLUSTER ? static_cast<int>(cluster.block_rank()) : 0;
    __shared__ unsigned int s_count[2];        // legal, INT8-routed
    __shared__ int32_t s_off[2 * kStagedSeqs];
    if (threadIdx.x < 2) s_count[threadIdx.x] = 0u;
    if (tok != nullptr && n_seqs < kStagedSeqs) {   // the look-up of a row's sequence is a chain of dependent reads
        for (int i = threadIdx.x; i <= n_seqs; i += kThreads) { s_off[i] = tile_off[i]; s_off[kStagedSeqs + i] = tok[i]; }
        tile_off = s_off;
        tok = s_off + kStagedSeqs;
    }
    if constexpr (CLUSTER) cluster.sync(); else __syncthreads();
    const int64_t bh = blockIdx.x / n_ctas;
    const uint8_t* r_in = route + bh * T_m * static_cast<int64_t>(T_mask);
    uint32_t* w_out = words + bh * T_m * static_cast<int64_t>(W);
    const int lane = threadIdx.x & 31, n_warps = n_ctas * (kThreads / 32);
    const int64_t total = static_cast<int64_t>(T_m) * W;
    unsigned int n_legal = 0, n_int8 = 0;
    for (int64_t base = rank * (kThreads / 32) + (threadIdx.x >> 5); base < total; base += static_cast<int64_t>(kUnroll) * n_warps) {
        uint32_t legal[kUnroll], bit[kUnroll];
#pragma unroll
        for (int u = 0; u < kUnroll; ++u) {
            const int64_t idx = base + static_cast<int64_t>(u) * n_warps;
            legal[u] = bit[u] = 0u;
            if (idx >= total) continue;
            const int m_row = static_cast<int>(idx / W), w = static_cast<int>(idx - static_cast<int64_t>(m_row) * W);
            // variable-length batch: row m_row of the packed batch is row m of its own sequence of length L
            int m = m_row, L = L_dense;
            if (tok != nullptr) {
                const int s = find_seq(tile_off, n_seqs, m_row);
                m = m_row - tile_off[s];
                L = tok[s + 1] - tok[s];
            }
            const int64_t last_row = min(static_cast<int64_t>(m + 1) * tile_m, static_cast<int64_t>(L)) - 1;
            // key tiles that straddle the diagonal of row m: [n_lo, n_hi]
            const int64_t n_lo = static_cast<int64_t>(m) * tile_m / tile_n;
            const int64_t n_hi = last_row / tile_n;
            const int64_t g = 32ll * w + lane, first_tile = g * G;
            if (g < T_mask && first_tile * tile_n <= last_row) {   // (groups beyond that hold no legal pair)
                legal[u] = 1u;
                const bool diag = first_tile <= n_hi && first_tile + G - 1 >= n_lo;
                if (!(pin_diag && diag)) bit[u] = r_in[static_cast<int64_t>(m_row) * T_mask + g];
            }
        }
#pragma unroll
        for (int u = 0; u < kUnroll; ++u) {
            const int64_t idx = base + static_cast<int64_t>(u) * n_warps;
            const uint32_t word = __ballot_sync(0xffffffffu, bit[u] != 0u);
            n_legal += __popc(__ballot_sync(0xffffffffu, legal[u] != 0u));
            n_int8 += __popc(word);
            if (lane == 0 && idx < total) w_out[idx] = word;
        }
    }
    if (lane == 0 && counts != nullptr) {
        unsigned int* first = CLUSTER ? cluster.map_shared_rank(s_count, 0) : s_count;
        atomicAdd(&first[0], n_legal);
        atomicAdd(&first[1], n_int8);
    }
    if constexpr (CLUSTER) cluster.sync(); else __syncthreads();
    if (rank == 0 && threadIdx.x < 2 && counts != nullptr) counts[bh * 2 + threadIdx.x] = s_count[threadIdx.x];
}

}  // namespace

int launch_pack(const Geometry& g, const uint8_t* route, uint32_t pack_flags, uint32_t* words,
                unsigned long long* counts, cudaStream_t stream, const VarlenDev* vl) {
    // about two rounds of words per warp, up to the portable cluster size
    int cluster = 1;
    const int64_t total = static_cast<int64_t>(g.T_m) * g.W;
    while (cluster < 8 && total > 2ll * kUnroll * (kThreads / 32) * cluster) cluster *= 2;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(static_cast<unsigned>(g.nb * g.Hk * cluster));
    cfg.blockDim = dim3(kThreads);
    cfg.stream = stream;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = static_cast<unsigned>(cluster);
    attr[0].val.clusterDim.y = attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = cluster > 1 ? 1 : 0;
    const cudaError_t e = cudaLaunchKernelEx(&cfg, cluster > 1 ? pack_kernel<true> : pack_kernel<false>, route, g.L, g.tile_m, g.tile_n, g.G, g.T_m, g.T_mask, g.W,
                                             (pack_flags & TILEMIX_PIN_DIAGONAL_FP16) ? 1 : 0, words, counts,
                                             vl ? vl->tok : static_cast<const int32_t*>(nullptr),
                                             vl ? vl->tile : static_cast<const int32_t*>(nullptr), vl ? vl->n : 0);
    g_launch_count.fetch_add(1);
    return static_cast<int>(e);
}

}  // namespace tilemix

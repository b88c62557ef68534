// Distance table of the core (the partial hierarchy's top, Sec. 3's
// candidate-bounded contraction): for every pair of core vertices, the
// length of the shortest path between them, so that a query stops its two
// upward searches at the core and joins them through the table instead of
// searching inside the core.
//
// The core vertices are the last core_size ranks; their E_up rows hold the
// core's own edges (a core vertex keeps its overlay out-edges, all to other
// core vertices). One block per core source runs a label-correcting search
// over those rows: a level expands the vertices whose label dropped in the
// level before, each queued once (a bitmap). Distances between
// surviving vertices are those of the input graph, so row i is the
// shortest-path distance from core vertex i to every core vertex.
#include <algorithm>

#include "handle.cuh"

namespace gbch {
namespace {

constexpr uint32_t CORE_ERR_BOUND = 2u;

// Threads of a source's block, at most, and the largest core whose labels are
// kept in shared memory (label and two queue bits a vertex: 212 KB).
constexpr int CT_THREADS = 1024;
constexpr uint32_t CT_SMEM_CORE = 51200;

// One block per core source: a label-correcting search over the core's rows.
// The vertices whose label dropped are bits of a queue bitmap; a warp takes
// the next word of the level's bitmap (a shared counter, so that a word with a
// hub holds up one warp only), clears it, spreads the out-edges of its up to
// 32 vertices over its lanes and sets the heads' bits in the next level's.
// With LSMEM the labels are in shared memory and the row is written once at
// the end; cores above CT_SMEM_CORE use the row itself (atomics in L2).
// Bound by the shared-memory atomics and the edge loads from L2. RMAT 2^14
// (3,320 core vertices): 7.4 ms; a thread per queued vertex walking its
// row, labels in L2, took 100 ms.
template <bool LSMEM>
__global__ void __launch_bounds__(CT_THREADS) k_core_table(const uint32_t *up_off, const uint2 *up_adj, uint32_t n,
                                                           uint32_t n_up, uint32_t core_lo, uint32_t C,
                                                           uint32_t *tab, uint32_t *work, uint32_t *err) {
    extern __shared__ uint32_t ct_smem[];
    __shared__ uint32_t s_item, s_next, s_any[2];
    const uint32_t W = (C + 31) / 32;
    uint32_t *const bits = ct_smem;  // two bitmaps of W words
    const uint32_t tid = threadIdx.x, lane = lane_id();
    for (uint32_t j = tid; j < 2 * W; j += blockDim.x) ct_smem[j] = 0;
    while (true) {
        __syncthreads();
        if (tid == 0) s_item = atomicAdd(work, 1u);
        __syncthreads();
        const uint32_t src = s_item;
        if (src >= C) break;
        uint32_t *row = tab + (size_t)src * C;
        uint32_t *lab = LSMEM ? ct_smem + 2 * W : row;
        auto label = [&](uint32_t v) { return LSMEM ? *(volatile uint32_t *)(lab + v) : __ldcg(lab + v); };
        for (uint32_t j = tid; j < C; j += blockDim.x) lab[j] = INF;
        __syncthreads();
        if (tid == 0) {
            lab[src] = 0;
            bits[src / 32] = 1u << (src % 32);
            s_next = 0;
            s_any[0] = 1;
            s_any[1] = 0;
        }
        for (uint32_t cur = 0;; cur ^= 1) {
            __syncthreads();
            if (!s_any[cur]) break;
            bool any = false;
            while (true) {
                uint32_t w = 0;
                if (lane == 0) w = atomicAdd(&s_next, 1u);
                w = __shfl_sync(FULL, w, 0);
                if (w >= W) break;
                uint32_t word = 0;
                if (lane == 0) word = atomicExch(&bits[cur * W + w], 0u);
                word = __shfl_sync(FULL, word, 0);
                if (!word) continue;
                const uint32_t x = 32 * w + lane;
                uint32_t b = 0, cnt = 0, dx = INF;
                if (((word >> lane) & 1u) && x < C) {
                    b = up_off[core_lo + x];
                    const uint32_t e = up_off[core_lo + x + 1];
                    if (b <= e && e <= n_up) cnt = e - b;
                    else atomicOr(err, CORE_ERR_BOUND);
                    dx = label(x);
                }
                const uint32_t incl = warp_incl_scan(cnt);
                const uint32_t total = __shfl_sync(FULL, incl, 31);
                const uint32_t excl = incl - cnt;
                for (uint32_t base = 0; base < total; base += 32) {
                    const uint32_t idx = base + lane;
                    const uint32_t o = warp_owner(excl, idx);
                    const uint32_t ob = __shfl_sync(FULL, b, o);
                    const uint32_t oex = __shfl_sync(FULL, excl, o);
                    const uint32_t odx = __shfl_sync(FULL, dx, o);
                    if (idx >= total) continue;
                    const uint2 a = up_adj[ob + (idx - oex)];
                    if (a.x < core_lo || a.x >= n) {
                        atomicOr(err, CORE_ERR_BOUND);
                        continue;
                    }
                    const uint32_t y = a.x - core_lo;
                    const uint32_t nd = sat_add(odx, a.y);
                    if (nd >= label(y)) continue;
                    if (atomicMin(&lab[y], nd) <= nd) continue;
                    atomicOr(&bits[(cur ^ 1) * W + y / 32], 1u << (y % 32));
                    any = true;
                }
            }
            if (any) s_any[cur ^ 1] = 1;
            __syncthreads();
            if (tid == 0) {
                s_next = 0;
                s_any[cur] = 0;
            }
        }
        if (LSMEM)
            for (uint32_t j = tid; j < C; j += blockDim.x) row[j] = lab[j];
    }
}

}  // namespace

void core_table(ch_s *h, uint64_t max_bytes, cudaStream_t st) {
    const uint64_t C = h->core_size;
    h->core_tab.release();
    h->core_n = 0;
    h->core_lo = h->n;
    if (C == 0) return;
    if (C >= (1ull << 32) || C > max_bytes / 4 / C)  // C^2 * 4 > max_bytes, without overflow
        throw Error{CH_ERANGE, "core distance table of " + std::to_string(C) + "^2 entries exceeds the byte limit"};
    const uint32_t n = h->n;
    const uint32_t core_lo = (uint32_t)(n - C);
    DevBuf<uint32_t> tab, ctl;
    tab.alloc(C * C);
    ctl.alloc(2);  // [0] work counter, [1] error word
    ctl.zero(st);
    // Small cores leave room for several blocks an SM, which hide each other's
    // barriers; a core that fills the SM gets all of its threads.
    const bool lsmem = C <= CT_SMEM_CORE;
    auto *kern = lsmem ? k_core_table<true> : k_core_table<false>;
    const size_t smem = ((C + 31) / 32 * 2 + (lsmem ? C : 0)) * sizeof(uint32_t);
    if (smem > 227u * 1024 - 1024) throw Error{CH_ERANGE, "core of " + std::to_string(C) + " vertices is too large for a distance table"};
    CH_CUDA_TRY(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
    int per_sm = 0, threads = 512;
    CH_CUDA_TRY(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, threads, smem));
    if (per_sm < 2) {
        threads = CT_THREADS;
        per_sm = 1;
    }
    const int grid = (int)std::min<uint64_t>(C, (uint64_t)device_sm_count() * per_sm);
    kern<<<grid, threads, smem, st>>>(h->up_off.ptr, h->up_adj.ptr, n, (uint32_t)h->n_up, core_lo, (uint32_t)C,
                                      tab.ptr, ctl.ptr, ctl.ptr + 1);
    CH_CHECK_LAUNCH();
    uint32_t err = 0;
    CH_CUDA_TRY(cudaMemcpyAsync(&err, ctl.ptr + 1, 4, cudaMemcpyDeviceToHost, st));
    CH_CUDA_TRY(cudaStreamSynchronize(st));
    if (err) throw Error{CH_ECUDA, "internal index check failed in the core table"};
    h->core_tab = std::move(tab);
    h->core_lo = core_lo;
    h->core_n = (uint32_t)C;
}

}  // namespace gbch

// One-to-all distances on a built hierarchy (ch_one_to_all), the PHAST scheme
// the paper cites for single-source distances on a CH (Sec. 5).
//
// A vertex's distance from s is the least d_up(x) + (a downward path x -> v)
// over the vertices x of s's upward search. Both parts follow the rank order,
// whose levels are contiguous rank ranges (rank sorts by level first):
//   upward    s's search space is a few hundred vertices: a queue below the
//             top levels (phast_climb), then those levels ascending. A level's
//             labels are final once every lower level has pushed along its
//             E_up edges, because an E_up edge leaves a vertex for a
//             later-contracted one (its live neighbours were outside the
//             independent set V_F). The core, whose E_up holds the edges
//             among its own vertices, repeats its pushes until a pass changes
//             nothing (Bellman-Ford, at most core-size passes).
//   downward  levels descending, core excluded (its labels are exact after
//             the upward part). d(u) = min(d(u), d(x) + w) over u's E_down
//             edges (x, u); x lies in a higher level, so d(x) is final. No
//             atomics: each vertex is written by its own thread.
//
// Layout: the labels of PK sources (4, 16 or 64, the least that holds the rest
// of the batch) are interleaved per vertex in rank order, D[r * PK + i], so that
// PK / 4 threads serve a vertex with 16-byte loads and a gather along an edge
// reads one row. Levels with more than TOP_LEVEL vertices get a launch each
// (overlapped, a level waits for the one before). The run of smaller levels at
// the top of the hierarchy, where levels hold a handful of vertices, is walked
// by a block a source with the labels in shared memory (k_phast_top). The
// result leaves D through one permuting pass, out[i * n + v] =
// D[rank[v] * PK + i].
//
// 64 sources on a 1M-vertex geometric graph: 0.76 ms. (One block walked
// the upper levels of all 64 sources through global memory: 3.3 of 4.2 ms.)
//
// Algorithmic bytes per pass, both sweeps: the label rows (4 * PK B read and
// written per vertex and sweep), 8 B per E_up / E_down entry plus a 4 * PK-B
// label row per entry, and the offsets; then 4 * PK B read and 4 * PK B written
// per vertex for the output.

#include <algorithm>
#include <vector>

#include "handle.cuh"

namespace gbch {
namespace {

constexpr uint32_t TOP_LEVEL = 256;     // largest level k_phast_top walks (128 or 512: 5% slower)
constexpr uint32_t TOP_WORDS = 50000;   // its shared memory: labels, both CSRs' offsets, level bounds
constexpr int TOP_THREADS = 1024;
constexpr uint32_t CLIMB_CAP = 2048;    // queue entries of a source's climb to the top levels, per step
constexpr uint32_t PERR_RANGE = 1u;    // a source id >= n (same bit as the query kernels)
constexpr uint32_t PERR_BOUND = 2u;    // an index check failed; the access was skipped

// One pass over the core (ranks [r0, r1)): its vertices' finite labels are
// pushed along their E_up edges, Q threads a vertex, 4 sources each. A stale
// read of a target only costs an extra atomicMin: labels only ever decrease.
template <uint32_t Q>
__global__ void k_phast_core(uint32_t *D, uint32_t r0, uint32_t r1, const uint32_t *up_off, const uint2 *up_adj,
                           uint32_t n, uint32_t *changed, uint32_t *err) {
    bool lowered = false;
    const uint64_t total = (uint64_t)(r1 - r0) * Q;
    for (uint64_t t = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; t < total;
         t += (uint64_t)gridDim.x * blockDim.x) {
        const uint32_t r = r0 + (uint32_t)(t / Q), q = (uint32_t)(t % Q);
        const uint4 d = __ldcg(reinterpret_cast<const uint4 *>(D) + (uint64_t)r * Q + q);
        if ((d.x & d.y & d.z & d.w) == INF) continue;
        const uint32_t lab[4] = {d.x, d.y, d.z, d.w};
        const uint32_t e1 = up_off[r + 1];
        for (uint32_t e = up_off[r]; e < e1; ++e) {
            const uint2 a = up_adj[e];
            if (a.x >= n) {
                atomicOr(err, PERR_BOUND);
                continue;
            }
            uint32_t *p = D + ((uint64_t)a.x * Q + q) * 4;
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const uint32_t nd = sat_add(lab[i], a.y);
                if (nd < __ldcg(p + i) && atomicMin(p + i, nd) > nd) lowered = true;
            }
        }
    }
    if (lowered) *changed = 1u;
}

// One level [r0, r1) of the downward sweep: pulls over E_down.
template <uint32_t Q>
__global__ void k_phast_down(uint32_t *D, uint32_t r0, uint32_t r1, const uint32_t *dn_off, const uint2 *dn_adj,
                             uint32_t n, uint32_t *err) {
    const uint64_t total = (uint64_t)(r1 - r0) * Q;
    uint4 *D4 = reinterpret_cast<uint4 *>(D);
    pdl_wait();
    pdl_launch();
    for (uint64_t t = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; t < total;
         t += (uint64_t)gridDim.x * blockDim.x) {
        const uint32_t r = r0 + (uint32_t)(t / Q), q = (uint32_t)(t % Q);
        uint4 d = __ldcg(D4 + (uint64_t)r * Q + q);
        const uint32_t b = dn_off[r], e1 = dn_off[r + 1];
        constexpr uint32_t U = 4;  // edges in flight
        for (uint32_t e = b; e < e1; e += U) {
            uint2 a[U];
            uint4 x[U];
#pragma unroll
            for (uint32_t u = 0; u < U; ++u) {
                a[u] = e + u < e1 ? dn_adj[e + u] : make_uint2(INF, INF);
                if (a[u].x >= n) {
                    if (e + u < e1) atomicOr(err, PERR_BOUND);
                    a[u] = make_uint2(0, INF);  // adds nothing
                }
            }
#pragma unroll
            for (uint32_t u = 0; u < U; ++u)
                x[u] = a[u].y != INF ? __ldcg(D4 + (uint64_t)a[u].x * Q + q) : make_uint4(INF, INF, INF, INF);
#pragma unroll
            for (uint32_t u = 0; u < U; ++u) {
                d.x = min(d.x, sat_add(x[u].x, a[u].y));
                d.y = min(d.y, sat_add(x[u].y, a[u].y));
                d.z = min(d.z, sat_add(x[u].z, a[u].y));
                d.w = min(d.w, sat_add(x[u].w, a[u].y));
            }
        }
        D4[(uint64_t)r * Q + q] = d;
    }
}

// A block a source: with src, its whole upward part (the climb to the top
// levels, then those levels ascending); with down, the top levels descending.
// The top levels are the small ones, [l0, l1) = ranks [base, top), a barrier
// between levels.
// Labels, both CSRs' offsets and the level bounds are in shared memory; a warp
// takes every 32nd vertex of a level, its row's first 64 edges from registers.
// The rows do not depend on the labels, so a warp has the rows of its next
// TOP_AHEAD vertices in flight: a level of up to 32 vertices costs a barrier
// and a few shared-memory accesses instead of two round trips to L2. Edges to
// the core (ranks from top on) go to D.
constexpr int TOP_AHEAD = 6;

template <bool UP>
__device__ void phast_top_sweep(uint32_t *lab, const uint32_t *off, const uint32_t *lv, uint32_t nl, uint32_t base,
                                uint32_t top, const uint2 *adj, uint32_t *D, uint32_t pk, uint32_t i, uint32_t n,
                                uint32_t *err) {
    const uint32_t lane = lane_id(), warp = threadIdx.x >> 5;
    constexpr uint32_t W = TOP_THREADS / 32;
    // position: level k of nl in sweep order, first vertex r of the warps' next 32
    struct Pos {
        uint32_t k, r;
    };
    auto level = [&](uint32_t k) { return UP ? k : nl - 1 - k; };
    auto skip_empty = [&](Pos &p) {
        while (p.k < nl && p.r >= lv[level(p.k) + 1])
            if (++p.k < nl) p.r = lv[level(p.k)];
    };
    auto start = [&] {
        Pos p{0, lv[level(0)]};
        skip_empty(p);
        return p;
    };
    uint2 e0[TOP_AHEAD], e1[TOP_AHEAD];
    auto fetch = [&](Pos &p, uint2 &a0, uint2 &a1) {
        a0 = a1 = make_uint2(INF, INF);
        if (p.k >= nl) return;
        const uint32_t r = p.r + warp;
        if (r < lv[level(p.k) + 1]) {
            const uint32_t b = off[r - base], m = off[r - base + 1] - b;
            if (lane < m) a0 = adj[b + lane];
            if (lane + 32 < m) a1 = adj[b + lane + 32];
        }
        p.r += W;
        skip_empty(p);
    };
    // an edge whose other end is x: its label, or the push of d + w to it
    auto pull = [&](uint2 e) {
        if (e.x < top && e.x >= base) return sat_add(lab[e.x - base], e.y);
        if (e.x < n && e.x >= top) return sat_add(__ldcg(D + (uint64_t)e.x * pk + i), e.y);
        if (e.x != INF) atomicOr(err, PERR_BOUND);
        return INF;
    };
    auto push = [&](uint2 e, uint32_t d) {
        const uint32_t nd = sat_add(d, e.y);
        if (nd == INF) return;
        if (e.x < top && e.x >= base) atomicMin(&lab[e.x - base], nd);
        else if (e.x < n && e.x >= top) atomicMin(D + (uint64_t)e.x * pk + i, nd);
        else atomicOr(err, PERR_BOUND);
    };
    Pos ahead = start(), at = ahead;
#pragma unroll
    for (int u = 0; u < TOP_AHEAD; ++u) fetch(ahead, e0[u], e1[u]);
    while (at.k < nl) {
#pragma unroll
        for (int u = 0; u < TOP_AHEAD; ++u) {
            if (at.k >= nl) break;
            const uint32_t r = at.r + warp;
            if (r < lv[level(at.k) + 1]) {
                const uint32_t b = off[r - base], m = off[r - base + 1] - b;
                uint32_t d = lab[r - base];
                if (UP) {
                    if (d != INF) {
                        if (lane < m) push(e0[u], d);
                        if (lane + 32 < m) push(e1[u], d);
                        for (uint32_t j = lane + 64; j < m; j += 32) push(adj[b + j], d);
                    }
                } else {
                    d = min(d, min(pull(e0[u]), pull(e1[u])));
                    for (uint32_t j = lane + 64; j < m; j += 32) d = min(d, pull(adj[b + j]));
                    d = __reduce_min_sync(FULL, d);
                    if (lane == 0) lab[r - base] = d;
                }
            }
            fetch(ahead, e0[u], e1[u]);
            const uint32_t k = at.k;
            at.r += W;
            skip_empty(at);
            if (at.k != k) __syncthreads();
        }
    }
    __syncthreads();
}

// The upward search of source i (rank r0) below the top levels: a queue of
// lowered vertices, a warp a row, until none is left; labels in D, those of the
// top levels in lab. Entered twice in a step, a vertex is only expanded twice.
// If the queue overflows, the block goes over every lower vertex in rank order
// instead (levels are rank ranges, so a level's labels are final when it is
// reached).
__device__ void phast_climb(uint32_t *lab, uint32_t (*queue)[CLIMB_CAP], uint32_t *cnt3, uint32_t base, uint32_t top,
                            const uint32_t *up_off, const uint2 *up_adj, uint32_t n_up, const uint32_t *lv,
                            uint32_t levels, uint32_t *D, uint32_t pk, uint32_t i, uint32_t n, uint32_t r0,
                            uint32_t *err) {
    const uint32_t lane = lane_id(), warp = threadIdx.x >> 5;
    // lowers x's label; whether x has to be expanded
    auto lower = [&](uint32_t x, uint32_t nd) {
        if (nd == INF) return false;
        if (x >= base && x < top) {
            atomicMin(&lab[x - base], nd);
            return false;
        }
        if (x >= n) {
            atomicOr(err, PERR_BOUND);
            return false;
        }
        return atomicMin(D + (uint64_t)x * pk + i, nd) > nd && x < base;
    };
    auto row = [&](uint32_t x, uint32_t &b, uint32_t &e) {
        b = up_off[x];
        e = up_off[x + 1];
        if (b > e || e > n_up) {
            atomicOr(err, PERR_BOUND);
            b = e = 0;
        }
    };
    if (threadIdx.x == 0) {
        queue[0][0] = r0;
        cnt3[0] = r0 < base;
        cnt3[1] = 0;
        if (r0 < base || r0 >= top) D[(uint64_t)r0 * pk + i] = 0;
        else lab[r0 - base] = 0;
    }
    for (uint32_t step = 0;; ++step) {
        __syncthreads();
        const uint32_t nq = cnt3[step % 3];
        if (nq == 0) return;
        if (nq > CLIMB_CAP) break;
        if (threadIdx.x == 0) cnt3[(step + 2) % 3] = 0;
        const uint32_t *cur = queue[step & 1u];
        uint32_t *nxt = queue[(step & 1u) ^ 1u], *ncnt = &cnt3[(step + 1) % 3];
        for (uint32_t f = warp; f < nq; f += TOP_THREADS / 32) {
            const uint32_t x = cur[f];
            const uint32_t d = __ldcg(D + (uint64_t)x * pk + i);
            uint32_t b, e;
            row(x, b, e);
            for (uint32_t j = b + lane; j < e; j += 32) {
                const uint2 a = up_adj[j];
                if (!lower(a.x, sat_add(d, a.y))) continue;
                const uint32_t p = atomicAdd(ncnt, 1u);
                if (p < CLIMB_CAP) nxt[p] = a.x;
            }
        }
    }
    for (uint32_t l = 0; l < levels; ++l) {
        for (uint32_t x = lv[l] + threadIdx.x; x < lv[l + 1] && x < base; x += TOP_THREADS) {
            const uint32_t d = __ldcg(D + (uint64_t)x * pk + i);
            if (d == INF) continue;
            uint32_t b, e;
            row(x, b, e);
            for (uint32_t j = b; j < e; ++j) {
                const uint2 a = up_adj[j];
                lower(a.x, sat_add(d, a.y));
            }
        }
        __syncthreads();
    }
}

__global__ void __launch_bounds__(TOP_THREADS)
k_phast_top(uint32_t *D, uint32_t pk, const uint32_t *lv, uint32_t l0, uint32_t l1, uint32_t base, uint32_t top,
            const uint32_t *src, const uint32_t *rank, bool down, const uint32_t *up_off, const uint2 *up_adj, uint32_t n_up, const uint32_t *dn_off,
            const uint2 *dn_adj, uint32_t n_dn, uint32_t n, uint32_t *err) {
    extern __shared__ uint32_t top_smem[];
    const uint32_t tid = threadIdx.x, T = top - base, nl = l1 - l0, i = blockIdx.x;
    uint32_t *lab = top_smem, *uo = lab + T, *dof = uo + T + 1, *slv = dof + T + 1;
    bool ok = true;
    for (uint32_t j = tid; j <= T; j += TOP_THREADS) {
        uo[j] = up_off[base + j];
        dof[j] = dn_off[base + j];
        ok &= uo[j] <= n_up && dof[j] <= n_dn &&
              (j == 0 || (up_off[base + j - 1] <= uo[j] && dn_off[base + j - 1] <= dof[j]));
    }
    for (uint32_t j = tid; j <= nl; j += TOP_THREADS) {
        slv[j] = lv[l0 + j];
        ok &= slv[j] >= base && slv[j] <= top && (j == 0 || lv[l0 + j - 1] <= slv[j]);
    }
    pdl_wait();
    pdl_launch();
    if (!__syncthreads_and(ok)) {
        if (tid == 0) atomicOr(err, PERR_BOUND);
        return;
    }
    for (uint32_t j = tid; j < T; j += TOP_THREADS) lab[j] = src ? INF : __ldcg(D + (uint64_t)(base + j) * pk + i);
    __syncthreads();
    if (src) {
        __shared__ uint32_t queue[2][CLIMB_CAP], cnt3[3];
        const uint32_t s = src[i], r = s < n ? rank[s] : INF;
        if (r < n) {
            phast_climb(lab, queue, cnt3, base, top, up_off, up_adj, n_up, lv, l0, D, pk, i, n, r, err);
            if (nl) phast_top_sweep<true>(lab, uo, slv, nl, base, top, up_adj, D, pk, i, n, err);
        } else if (tid == 0) {
            atomicOr(err, s < n ? PERR_BOUND : PERR_RANGE);  // its row stays INF
        }
        __syncthreads();
    }
    if (down && nl) phast_top_sweep<false>(lab, dof, slv, nl, base, top, dn_adj, D, pk, i, n, err);
    for (uint32_t j = tid; j < T; j += TOP_THREADS) D[(uint64_t)(base + j) * pk + i] = lab[j];
}

// out[i * n + v] = D[rank[v] * PK + i] for the batch's nsrc sources: a tile of
// 64 vertices goes through shared memory, so that whole label rows are read and
// runs of 64 vertices written (1M vertices, 64 sources: 96 us for 512 MB;
// 137 with a thread a vertex reading its row in 16-byte pieces).
constexpr uint32_t OUT_TILE = 64;

template <uint32_t Q>
__global__ void __launch_bounds__(256) k_phast_out(const uint32_t *D, const uint32_t *rank, uint32_t n, uint32_t nsrc,
                                                   uint32_t *out, uint32_t *err) {
    __shared__ uint32_t tile[4 * Q][OUT_TILE + 1];
    pdl_wait();
    const uint4 *D4 = reinterpret_cast<const uint4 *>(D);
    for (uint64_t v0 = blockIdx.x * (uint64_t)OUT_TILE; v0 < n; v0 += (uint64_t)gridDim.x * OUT_TILE) {
        const uint32_t m = (uint32_t)min((unsigned long long)OUT_TILE, (unsigned long long)(n - v0));
        for (uint32_t t = threadIdx.x; t < m * Q; t += blockDim.x) {
            const uint32_t v = t / Q, q = t % Q;
            const uint32_t r = rank[v0 + v];
            uint4 x = make_uint4(INF, INF, INF, INF);
            if (r < n) x = __ldcg(D4 + (uint64_t)r * Q + q);
            else atomicOr(err, PERR_BOUND);
            tile[4 * q][v] = x.x;
            tile[4 * q + 1][v] = x.y;
            tile[4 * q + 2][v] = x.z;
            tile[4 * q + 3][v] = x.w;
        }
        __syncthreads();
        for (uint32_t t = threadIdx.x; t < nsrc * OUT_TILE; t += blockDim.x) {
            const uint32_t i = t / OUT_TILE, v = t % OUT_TILE;
            if (v < m) out[(uint64_t)i * n + v0 + v] = tile[i][v];
        }
        __syncthreads();
    }
}

// The levels of one pass: what k_phast_top walks.
struct Top {
    uint32_t l0, l1, base, top;
};

// One pass of up to PK = 4 Q sources.
template <uint32_t Q>
void phast_pass(ch_s *h, const std::vector<uint32_t> &lv, const Top &t, const uint32_t *src, uint32_t nsrc,
                uint32_t *out, cudaStream_t st) {
    const uint32_t n = h->n, PK = 4 * Q;
    uint32_t *D = h->phast_d.ptr, *err = h->qerr.ptr;
    const int sms = device_sm_count();
    auto grid = [&](uint64_t threads) { return grid_for(threads, 256, sms * 8); };
    CH_CUDA_TRY(cudaMemsetAsync(D, 0xFF, (size_t)n * PK * sizeof(uint32_t), st));
    auto walk = [&](bool upward, bool downward) {
        const size_t words = 3ull * (t.top - t.base) + 2 + (t.l1 - t.l0) + 1;
        launch_pdl(k_phast_top, nsrc, TOP_THREADS, words * sizeof(uint32_t), st, D, PK, h->phast_lv.ptr, t.l0, t.l1,
                   t.base, t.top, upward ? src : nullptr, h->rank.ptr, downward, h->up_off.ptr, h->up_adj.ptr,
                   (uint32_t)h->n_up, h->dn_off.ptr, h->dn_adj.ptr, (uint32_t)h->n_down, n, err);
    };
    const uint32_t core_lo = t.top;
    if (core_lo == n) {
        walk(true, true);
    } else {
        walk(true, false);
        // at most (core size) passes change a label; one more finds none
        for (uint64_t pass = 0; pass <= (uint64_t)(n - core_lo); ++pass) {
            uint32_t changed = 0;
            CH_CUDA_TRY(cudaMemsetAsync(h->phast_flag.ptr, 0, sizeof(uint32_t), st));
            k_phast_core<Q><<<grid((uint64_t)(n - core_lo) * Q), 256, 0, st>>>(
                D, core_lo, n, h->up_off.ptr, h->up_adj.ptr, n, h->phast_flag.ptr, err);
            CH_CHECK_LAUNCH();
            CH_CUDA_TRY(cudaMemcpyAsync(&changed, h->phast_flag.ptr, sizeof(uint32_t), cudaMemcpyDeviceToHost, st));
            CH_CUDA_TRY(cudaStreamSynchronize(st));
            if (!changed) break;
        }
        walk(false, true);
    }
    for (uint32_t l = t.l0; l-- > 0;)
        if (lv[l + 1] > lv[l])
            launch_pdl(k_phast_down<Q>, grid((uint64_t)(lv[l + 1] - lv[l]) * Q), 256, 0, st, D, lv[l], lv[l + 1],
                       h->dn_off.ptr, h->dn_adj.ptr, n, err);
    launch_pdl(k_phast_out<Q>, grid_for(n, OUT_TILE, sms * 8), 256, 0, st, D, h->rank.ptr, n, nsrc, out, err);
}

}  // namespace

bool rank_levels(const ch_s *h, std::vector<uint32_t> &lv) {
    const size_t L = h->round_stats.size();
    lv.resize(L + 2);
    uint64_t acc = 0;
    for (size_t l = 0; l < L; ++l) {
        lv[l] = (uint32_t)std::min<uint64_t>(acc, h->n);
        acc += h->round_stats[l][2];  // |V_F| of round l
    }
    lv[L] = (uint32_t)std::min<uint64_t>(acc, h->n);
    lv[L + 1] = h->n;
    return acc + h->core_size == h->n;
}

void one_to_all(ch_s *h, const uint32_t *src, uint64_t k, uint32_t *dist_out, cudaStream_t st) {
    if (k == 0 || h->n == 0) return;
    const uint32_t n = h->n;
    const size_t L = h->round_stats.size();
    std::vector<uint32_t> lv;
    if (!rank_levels(h, lv)) throw Error{CH_EINVAL, "the hierarchy's level sizes do not add up to n"};
    // What k_phast_top walks: the longest run of small levels right below the
    // core that its shared memory holds.
    Top t{(uint32_t)L, (uint32_t)L, lv[L], lv[L]};
    while (t.l0 > 0 && lv[t.l0] - lv[t.l0 - 1] <= TOP_LEVEL &&
           3ull * (lv[L] - lv[t.l0 - 1]) + 3 + (L - t.l0 + 1) <= TOP_WORDS)
        --t.l0;
    t.base = lv[t.l0];
    const uint32_t PK = k > 16 ? 64 : (k > 4 ? 16 : 4);
    if (h->phast_d.count < (size_t)n * PK) h->phast_d.alloc((size_t)n * PK);
    if (h->phast_lv.count < L + 2) h->phast_lv.alloc(L + 2);
    if (h->phast_flag.count < 1) h->phast_flag.alloc(1);
    CH_CUDA_TRY(cudaFuncSetAttribute(k_phast_top, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                     (int)(TOP_WORDS * sizeof(uint32_t))));
    CH_CUDA_TRY(cudaMemcpyAsync(h->phast_lv.ptr, lv.data(), (L + 2) * sizeof(uint32_t),
                                cudaMemcpyHostToDevice, st));
    for (uint64_t b = 0; b < k;) {
        const uint64_t left = k - b;
        uint32_t *out = dist_out + b * (uint64_t)n;
        const uint32_t nsrc = (uint32_t)std::min<uint64_t>(left, 64);
        if (left > 16) phast_pass<16>(h, lv, t, src + b, nsrc, out, st);
        else if (left > 4) phast_pass<4>(h, lv, t, src + b, nsrc, out, st);
        else phast_pass<1>(h, lv, t, src + b, nsrc, out, st);
        b += nsrc;
    }
}

}  // namespace gbch

// Large query batches by hub labels (not in the paper, whose queries search
// one at a time): the upward searches of a batch share nearly all of their
// work, because the vertices that many searches climb through have the same
// labels for all of them. So the batch computes, for every vertex that a
// search can climb through and for both directions, the set of (hub, distance)
// pairs of its upward search space, from the highest level down: the label of
// v is {(v, 0)} and the labels of its upward neighbours, each entry plus the
// edge's weight, the least distance per hub. A query is then the least
// d_s(h) + d_t(h) over the hubs that the labels of s and t share.
//
// Pruning: an entry (h, d) is dropped when some entry (y, d') of the same label
// and an edge y -> h of the opposite CSR give d' + w < d (stall on demand). Its
// distance then exceeds the true one, so h with it is the top of no shortest
// path, while an exact entry is never dropped; the answers stay exact. Only
// the top 1/HL_PRUNE_PART of the ranks test it: every label inherits from
// theirs (200K-vertex geometric graph: 391 entries a label unpruned, 142 with
// the test on the top 1/20, 128 with it everywhere, at 20 times the work).
//
// Labels are made by each call from its own batch; only the memory is kept.
#include <algorithm>
#include <cmath>

#include "handle.cuh"
#include "qsearch.cuh"

namespace gbch {
namespace {

// The line from which a batch uses labels. A search costs the same for every
// query; labels cost a launch or two a level (8 to 10 us), and the merges of what
// the batch climbs through. A label holds about 0.13 row^2 hubs a level (row: mean
// length of a CSR row; measured 1.1 to 1.2 x the levels at row 3, 2.0 at 3.9), and
// once the arena outgrows the L2 its merges run at HBM latency, so the line also
// grows with n x levels x row^4. Rows above 4.5 count as 4.5: longer ones were
// measured on small, dense graphs only, where the labels stay in the L2.
// Measured, ms (labels / searches):
//   geometric (row 3)  20K vertices, 56 levels: 16K queries 0.72 / 0.78; 100K, 107:
//         25K 1.54 / 1.89; 256K, 135: 40K 2.7 / 4.0; 1M, 218: 80K 9.3 / 14.4, 1M
//         17.0 / 186.6; 3M, 325: 139K 52.9 / 52.5, 400K 63 / 151
//   grids (3.8 to 3.9) 128^2, 71: 16K 0.99 / 0.98; 300^2, 114: 24K 2.5 / 2.7; 600^2,
//         187: 48K 9.2 / 10.5; 1000^2, 241: 80K 39.4 / 30.8, 400K 66 / 151; 1400^2,
//         302: 112K 139 / 70, 400K 203 / 247; 1800^2, 344: 144K 304 / 140, 400K 401 /
//         387
//   digraphs           2.5K vertices, 224: 16K 1.8 / 1.3, 66K 1.9 / 4.7; 20K (m = 1.5
//         n), 198: 16K 1.9 / 1.0, 66K 2.0 / 3.7; 20K (m = 2 n), 514: 16K 11.5 / 5.7,
//         66K 17.3 / 20.4; 9K (m = 3.4 n), 726: 16K 24.0 / 11.1, 66K 47.1 / 42.0,
//         400K 203 / 251 (and 60% of its queries are searched all the same)
// Every losing one is below the line. (Not so RMAT 2^12 contracted whole, 100
// levels, half of whose searches end at once: 22K queries 0.94 / 0.55.)
constexpr uint64_t HL_MIN_K = 1u << 14;
constexpr double HL_MIN_SQRT = 80, HL_MIN_LEVEL = 224, HL_ROW_MAX = 4.5, HL_WORK = 566e3;
bool batch_is_large(const ch_s *h, uint64_t k) {
    const double n = (double)h->n, levels = (double)h->round_stats.size();
    const double row = std::min(HL_ROW_MAX, 0.5 * (double)(h->n_up + h->n_down) / n);
    return k >= HL_MIN_K && (double)k >= HL_MIN_SQRT * std::sqrt(n) && (double)k >= HL_MIN_LEVEL * levels &&
           (double)k * HL_WORK >= n * levels * row * row * row * row;
}
constexpr uint32_t HL_PRUNE_PART = 16;
// Levels of at most this many vertices are merged by a block a label.
constexpr uint32_t HL_BLOCK_LEVEL = 2048;
// Arena entries per vertex and direction, on average, and its largest size
// (1M-vertex geometric graph: 271 entries a label, labels for two thirds of
// the vertices and directions of a batch of 1M queries).
constexpr uint64_t HL_AVG = 384;
constexpr uint64_t HL_MAX_BYTES = 24ull << 30;
constexpr size_t Q_CHUNK_MAX = 1u << 22;  // queries of one call at most

constexpr uint32_t HL_NONE = 0xFFFFFFFFu;  // size of a label that was not computed

struct HlArgs {
    uint32_t n, n_up, n_dn;
    const uint32_t *rank;
    const uint32_t *up_off, *dn_off;
    const uint2 *up_adj, *dn_adj;
    uint8_t *mark;           // [2 n] direction-major: the label is needed
    uint32_t *off, *size;    // [2 n] arena position and entries of each label
    uint2 *arena;            // (hub rank, distance)
    uint64_t cap;            // arena entries
    unsigned long long *cursor;
    uint32_t *err;
    unsigned long long *stats;  // [0] labels merged, [1] entries read
};

struct HlDir {
    const uint32_t *off;   // rows to higher ranks
    const uint2 *adj;
    uint32_t m;
    const uint32_t *soff;  // the opposite CSR, for the stall test
    const uint2 *sadj;
    uint32_t sm;
};

__device__ __forceinline__ HlDir hl_dir(const HlArgs &a, uint32_t dir) {
    return dir ? HlDir{a.dn_off, a.dn_adj, a.n_dn, a.up_off, a.up_adj, a.n_up}
               : HlDir{a.up_off, a.up_adj, a.n_up, a.dn_off, a.dn_adj, a.n_dn};
}

// Row [b, e) of vertex v, empty (and an error recorded) if it is malformed.
__device__ __forceinline__ void hl_row(const HlArgs &a, const uint32_t *off, uint32_t m, uint32_t v, uint32_t &b,
                                       uint32_t &e) {
    b = off[v];
    e = off[v + 1];
    if (b > e || e > m) {
        atomicOr(a.err, QERR_BOUND);
        b = e = 0;
    }
}

// A label under construction in shared memory: an open-addressing table of T
// hubs and, with LIST, the list of its used slots. A label may hold LIMIT hubs;
// the table has room for what the threads at work (a warp, or a block with
// BLOCK) insert before they see that. T is any number (the hash is a
// multiply-high), so that the small table is no larger than labels need: at
// 768 slots 28 merging warps and 36 querying ones fit an SM, against 16 at
// 1024 slots with a list.
template <uint32_t T_, bool LIST, bool BLOCK>
struct alignas(16) HlTab {
    static constexpr uint32_t T = T_, LIMIT = T - (BLOCK ? T / 4 : T / 6);
    static constexpr uint32_t NLIST = LIST ? (BLOCK ? T : LIMIT + 32) : 1;
    static constexpr bool list_kept = LIST, by_block = BLOCK;
    static constexpr uint16_t STALLED = 0x8000u;
    static_assert(T <= 0x7FFF && LIMIT + 32 < T, "slot numbers and head room");
    uint32_t key[T];
    uint32_t val[T];
    uint16_t list[NLIST];
    uint32_t cnt;   // BLOCK: used slots
    uint32_t bad;   // BLOCK: 1 = a part of the label is missing, 2 = too large
    uint32_t kept, base;
};

template <class Tab>
__device__ __forceinline__ uint32_t hl_hash(uint32_t v) {
    return __umulhi(v * 2654435761u, Tab::T);
}
template <class Tab>
__device__ __forceinline__ uint32_t hl_next(uint32_t h) {
    return h + 1 == Tab::T ? 0 : h + 1;
}

// Empties the table with the group's threads (gt of GT).
template <class Tab>
__device__ __forceinline__ void hl_clear(Tab &t, uint32_t gt, uint32_t GT) {
    static_assert(Tab::T % 4 == 0, "cleared by 16-byte stores");
    uint4 *k4 = reinterpret_cast<uint4 *>(t.key), *v4 = reinterpret_cast<uint4 *>(t.val);
    for (uint32_t j = gt; j < Tab::T / 4; j += GT) {
        k4[j] = make_uint4(EMPTY, EMPTY, EMPTY, EMPTY);
        v4[j] = make_uint4(INF, INF, INF, INF);
    }
}

// Distance of hub v in the table, INF if it has none.
template <class Tab>
__device__ __forceinline__ uint32_t hl_find(const Tab &t, uint32_t v) {
    uint32_t h = hl_hash<Tab>(v);
    for (uint32_t p = 0; p < Tab::T; ++p) {
        const uint32_t k = t.key[h];
        if (k == v) return t.val[h];
        if (k == EMPTY) return INF;
        h = hl_next<Tab>(h);
    }
    return INF;
}

// Lowers hub v's distance to d, for each lane with on set; every lane of the
// warp calls it. Counts new hubs (in the table for a block's, else in cnt, the
// same in every lane) and lists their slots.
template <class Tab>
__device__ __forceinline__ void hl_lower(Tab &t, bool on, uint32_t v, uint32_t d, uint32_t &cnt) {
    uint32_t h = hl_hash<Tab>(v);
    bool created = false;
    if (on) {
        for (uint32_t p = 0; p < Tab::T; ++p) {
            uint32_t k = t.key[h];
            if (k == EMPTY) {
                k = atomicCAS(&t.key[h], EMPTY, v);
                created = k == EMPTY;
                if (created) k = v;
            }
            if (k == v) break;
            h = hl_next<Tab>(h);
        }
        atomicMin(&t.val[h], d);
    }
    const uint32_t m = __ballot_sync(FULL, created);
    if (!m) return;
    uint32_t p = cnt;
    if (Tab::by_block) {
        const uint32_t leader = __ffs(m) - 1;
        if (lane_id() == leader) p = atomicAdd(&t.cnt, (uint32_t)__popc(m));
        p = __shfl_sync(FULL, p, leader);
    } else {
        cnt += __popc(m);
    }
    if (Tab::list_kept && created) t.list[p + __popc(m & ((1u << lane_id()) - 1u))] = (uint16_t)h;
}

// Whether the label outgrew its table (one answer for the warp: lanes may read
// a block's count at different times).
template <class Tab>
__device__ __forceinline__ bool hl_full(const Tab &t, uint32_t cnt) {
    if (!Tab::by_block) return cnt > Tab::LIMIT;
    return __any_sync(FULL, *(const volatile uint32_t *)&t.cnt > Tab::LIMIT);
}

using HlWarp = HlTab<768, true, false>;     // merges by a warp
using HlBlock = HlTab<4096, true, true>;    // by a block
using HlQuery = HlTab<768, false, false>;   // queries by a warp
using HlQueryBlock = HlTab<4096, false, true>;

constexpr int HL_UNROLL = 4;  // entries of a label a lane reads at once

// Runs f(on, hub, distance) over the label of every neighbour in row [b, e),
// distances through the neighbour's edge, a warp's 32 lanes at a time, until
// it returns false; warp w of W takes every W-th neighbour. Returns false if
// f did or if a label is missing. Counts the entries read.
template <class F>
__device__ __forceinline__ bool hl_row_labels(const HlArgs &a, const HlDir &d, uint32_t dir, uint32_t b, uint32_t e,
                                              uint32_t w, uint32_t W, QStat &stat, F &&f) {
    const uint32_t lane = lane_id();
    const uint32_t *size = a.size + (size_t)dir * a.n, *off = a.off + (size_t)dir * a.n;
    for (uint32_t j0 = b; j0 < e; j0 += 32 * W) {
        const uint32_t j = j0 + w + W * lane;
        uint32_t wt = 0, sz = 0, of = 0;
        bool ok = true;
        if (j < e) {
            const uint2 x = d.adj[j];
            if (x.x < a.n) {
                wt = x.y;
                sz = size[x.x];
                of = off[x.x];
                ok = sz != HL_NONE && (uint64_t)of + sz <= a.cap;
            } else {
                atomicOr(a.err, QERR_BOUND);
                ok = false;
            }
        }
        if (!__all_sync(FULL, ok)) return false;
        stat.edges += sz;
        const uint32_t left = e - j0, m = left <= w ? 0 : min(32u, (left - w + W - 1) / W);
        for (uint32_t q = 0; q < m; ++q) {
            const uint32_t qn = __shfl_sync(FULL, sz, q), qo = __shfl_sync(FULL, of, q),
                           qw = __shfl_sync(FULL, wt, q);
            for (uint32_t p0 = 0; p0 < qn; p0 += 32 * HL_UNROLL) {
                uint2 en[HL_UNROLL];
#pragma unroll
                for (int u = 0; u < HL_UNROLL; ++u) {
                    const uint32_t p = p0 + 32 * u + lane;
                    en[u] = p < qn ? __ldcg(a.arena + qo + p) : make_uint2(0, INF);
                }
#pragma unroll
                for (int u = 0; u < HL_UNROLL; ++u) {
                    if (p0 + 32 * u >= qn) break;
                    const uint32_t nd = sat_add(en[u].y, qw);
                    if (!f(nd != INF, en[u].x, nd)) return false;
                }
            }
        }
    }
    return true;
}

// Marks what the batch's endpoints climb to first: the upward neighbours of
// every source (direction 0) and target (direction 1), or the endpoints
// themselves when the batch asks for each vertex more than once on average.
__global__ void k_hl_mark(HlArgs a, const uint32_t *src, const uint32_t *dst, uint64_t k, bool self) {
    for (uint64_t t = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; t < 2 * k;
         t += (uint64_t)gridDim.x * blockDim.x) {
        const uint32_t dir = t >= k;
        const uint32_t v = dir ? dst[t - k] : src[t];
        const uint32_t r = v < a.n ? a.rank[v] : INF;
        if (r >= a.n) continue;  // reported by k_hl_query
        uint8_t *mark = a.mark + (size_t)dir * a.n;
        if (self) {
            mark[r] = 1;
            continue;
        }
        const HlDir d = hl_dir(a, dir);
        uint32_t b, e;
        hl_row(a, d.off, d.m, r, b, e);
        for (uint32_t j = b; j < e; ++j) {
            const uint32_t x = d.adj[j].x;
            if (x < a.n) mark[x] = 1;
            else atomicOr(a.err, QERR_BOUND);
        }
    }
}

// Levels ascending: the upward neighbours of the marked vertices of ranks
// [r0, r1) are marked too.
__global__ void k_hl_close(HlArgs a, uint32_t r0, uint32_t r1) {
    pdl_wait();
    pdl_launch();
    const uint32_t range = r1 - r0;
    for (uint64_t t = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; t < 2ull * range;
         t += (uint64_t)gridDim.x * blockDim.x) {
        const uint32_t dir = t >= range, r = r0 + (uint32_t)(dir ? t - range : t);
        uint8_t *mark = a.mark + (size_t)dir * a.n;
        if (!mark[r]) continue;
        const HlDir d = hl_dir(a, dir);
        uint32_t b, e;
        hl_row(a, d.off, d.m, r, b, e);
        for (uint32_t j = b; j < e; ++j) {
            const uint32_t x = d.adj[j].x;
            if (x < a.n) mark[x] = 1;
            else atomicOr(a.err, QERR_BOUND);
        }
    }
}

// Merges the labels of a level, ranks [r0, r1), both directions; the levels
// above are done. A warp merges a label, where marked, and appends those that
// outgrow its table to list (count in *list_cnt); a block merges every label of
// the level, or with `listed` those of the list. Blocks take the upper levels
// (few vertices with up to hundreds of neighbours each, where the time of one
// merge decides) and the listed ones.
//
// A warp's merge is bound by the shared-memory table (about 40 instructions
// per 32 entries read) and by the latency of the entries, which HL_UNROLL
// loads in flight a lane hide; labels are read and written once, coalesced.
template <class Tab, int THREADS>
__global__ void __launch_bounds__(THREADS, Tab::by_block ? 1 : 7)
k_hl_merge(HlArgs a, uint32_t r0, uint32_t r1, uint32_t prune_from, uint32_t *list, uint32_t *list_cnt, bool listed) {
    extern __shared__ __align__(16) unsigned char hl_raw[];
    constexpr bool BLOCK = Tab::by_block;
    constexpr uint32_t W = BLOCK ? THREADS / 32 : 1;  // warps a label
    constexpr uint32_t GT = W * 32;                   // threads a label
    const uint32_t lane = lane_id(), warp = threadIdx.x >> 5;
    Tab &t = reinterpret_cast<Tab *>(hl_raw)[BLOCK ? 0 : warp];
    const uint32_t gt = BLOCK ? threadIdx.x : lane, gw = BLOCK ? warp : 0;
    auto sync = [] {
        if (BLOCK) __syncthreads();
        else __syncwarp();
    };
    if (!listed) hl_clear(t, gt, GT);  // while the launch before this one ends
    pdl_wait();
    pdl_launch();
    QStat stat;
    const uint32_t range = r1 - r0, items = listed ? min(*list_cnt, 2 * range) : 2 * range;
    const uint32_t groups = BLOCK ? gridDim.x : gridDim.x * (THREADS / 32);
    if (listed) {  // usually nothing
        if (blockIdx.x >= items) return;
        hl_clear(t, gt, GT);
    }
    for (uint32_t q = BLOCK ? blockIdx.x : blockIdx.x * (THREADS / 32) + warp; q < items; q += groups) {
        const uint32_t it = listed ? list[q] : q;
        const uint32_t dir = it >= range, r = r0 + (dir ? it - range : it);
        if (r >= r1) continue;
        if (!BLOCK && !a.mark[(size_t)dir * a.n + r]) continue;
        const HlDir d = hl_dir(a, dir);
        sync();
        uint32_t cnt = 1;
        if (gt == 0) {
            const uint32_t h = hl_hash<Tab>(r);
            t.key[h] = r;
            t.val[h] = 0;
            t.list[0] = (uint16_t)h;
            if (BLOCK) {
                t.cnt = 1;
                t.bad = 0;
                t.kept = 0;
            }
        }
        sync();
        uint32_t b, e;
        hl_row(a, d.off, d.m, r, b, e);
        bool full = false;
        bool good = hl_row_labels(a, d, dir, b, e, gw, W, stat, [&](bool on, uint32_t v, uint32_t nd) {
            full = hl_full(t, cnt);
            if (full) return false;
            hl_lower(t, on, v, nd, cnt);
            return true;
        });
        if (BLOCK) {
            if (!good) t.bad = 1;
            sync();
            cnt = t.cnt;
            good = !t.bad;
        } else if (full && lane == 0) {
            const uint32_t p = atomicAdd(list_cnt, 1u);
            if (p < 2 * a.n) list[p] = it;
        }
        __syncwarp();
        uint32_t kept = 0;  // this warp's part of the list
        if (good) {
            // a block deals its hubs to all of its warps, so that their rows
            // are in flight at once
            const uint32_t part = BLOCK ? min(32u, (cnt + W - 1) / W) : 32u;
            for (uint32_t l0 = gw * part; l0 < cnt; l0 += W * part) {
                const uint32_t i = lane < part ? l0 + lane : cnt;
                const uint32_t slot = i < cnt ? t.list[i] : 0;
                bool stalled = false;
                if (r >= prune_from) {
                    // the row of each lane's hub in the opposite CSR
                    uint32_t sb = 0, se = 0;
                    const uint32_t h = t.key[slot], dh = t.val[slot];
                    if (i < cnt) hl_row(a, d.soff, d.sm, h, sb, se);
                    const uint32_t incl = warp_incl_scan(se - sb);
                    const uint32_t total = __shfl_sync(FULL, incl, 31);
                    const uint32_t excl = incl - (se - sb);
                    constexpr uint32_t U = BLOCK ? 4 : 2;  // edges a lane has in flight
                    for (uint32_t base = 0; base < total; base += 32 * U) {
                        uint2 y[U];
                        uint32_t od[U];
#pragma unroll
                        for (uint32_t u = 0; u < U; ++u) {
                            const uint32_t idx = base + 32 * u + lane;
                            const uint32_t o = warp_owner(excl, idx);
                            const uint32_t ob = __shfl_sync(FULL, sb, o), oex = __shfl_sync(FULL, excl, o);
                            od[u] = __shfl_sync(FULL, dh, o);
                            y[u] = idx < total ? d.sadj[ob + (idx - oex)] : make_uint2(EMPTY, INF);
                        }
#pragma unroll
                        for (uint32_t u = 0; u < U; ++u) {
                            const uint32_t first = base + 32 * u;
                            const bool st = y[u].x != EMPTY && sat_add(hl_find(t, y[u].x), y[u].y) < od[u];
                            const uint32_t B = __ballot_sync(FULL, st);
                            const uint32_t lo = max(excl, first), hi = min(incl, first + 32);
                            if (hi > lo && (B & qb_lane_range(lo - first, hi - first))) stalled = true;
                        }
                    }
                    stat.edges += se - sb;
                }
                if (stalled) t.list[i] = (uint16_t)(slot | Tab::STALLED);
                kept += __popc(__ballot_sync(FULL, i < cnt && !stalled));
            }
            unsigned long long base = 0;
            if (BLOCK) {
                if (lane == 0 && kept) atomicAdd(&t.kept, kept);
                sync();
                if (gt == 0) {
                    base = atomicAdd(a.cursor, (unsigned long long)t.kept);
                    const bool fits = base + t.kept <= a.cap;
                    if (fits) {
                        a.off[(size_t)dir * a.n + r] = (uint32_t)base;
                        a.size[(size_t)dir * a.n + r] = t.kept;
                    }
                    t.base = (uint32_t)base;
                    t.bad = !fits;
                    t.kept = 0;
                }
                sync();
                good = !t.bad;
                base = t.base;
            } else {
                if (lane == 0) base = atomicAdd(a.cursor, (unsigned long long)kept);
                base = __shfl_sync(FULL, base, 0);
                good = base + kept <= a.cap;
                if (good && lane == 0) {
                    a.off[(size_t)dir * a.n + r] = (uint32_t)base;
                    a.size[(size_t)dir * a.n + r] = kept;
                }
            }
            uint32_t run = 0;
            for (uint32_t l0 = gw * 32; good && l0 < cnt; l0 += GT) {
                const uint32_t i = l0 + lane;
                const uint32_t en = i < cnt ? t.list[i] : Tab::STALLED;
                const bool keep = !(en & Tab::STALLED);
                const uint32_t m = __ballot_sync(FULL, keep);
                if (BLOCK && m) {
                    const uint32_t leader = __ffs(m) - 1;
                    if (lane == leader) run = atomicAdd(&t.kept, (uint32_t)__popc(m));
                    run = __shfl_sync(FULL, run, leader);
                }
                if (keep)
                    a.arena[base + run + __popc(m & ((1u << lane) - 1u))] = make_uint2(t.key[en], t.val[en]);
                if (!BLOCK) run += __popc(m);
            }
        }
        sync();
        // empty the table again
        for (uint32_t i = gt; i < cnt; i += GT) {
            const uint32_t slot = t.list[i] & 0x7FFFu;
            t.key[slot] = EMPTY;
            t.val[slot] = INF;
        }
        stat.exp += gt == 0;
    }
    qb_flush_stat(stat, a.stats);
}

// Runs f over the label of the endpoint of rank r in direction dir: its own
// where it was computed, else its upward neighbours' and itself; warp w of W
// takes its share.
template <class F>
__device__ __forceinline__ bool hl_endpoint(const HlArgs &a, uint32_t dir, uint32_t r, uint32_t w, uint32_t W,
                                            QStat &stat, F &&f) {
    const uint32_t lane = lane_id();
    const uint32_t n = a.size[(size_t)dir * a.n + r];
    if (n != HL_NONE) {
        const uint32_t o = a.off[(size_t)dir * a.n + r];
        if ((uint64_t)o + n > a.cap) return false;
        stat.edges += lane == 0 && w == 0 ? n : 0;
        for (uint32_t p0 = w * 32 * HL_UNROLL; p0 < n; p0 += W * 32 * HL_UNROLL) {
            uint2 en[HL_UNROLL];
#pragma unroll
            for (int u = 0; u < HL_UNROLL; ++u) {
                const uint32_t p = p0 + 32 * u + lane;
                en[u] = p < n ? __ldcg(a.arena + o + p) : make_uint2(0, INF);
            }
#pragma unroll
            for (int u = 0; u < HL_UNROLL; ++u) {
                if (p0 + 32 * u >= n) break;
                if (!f(en[u].y != INF, en[u].x, en[u].y)) return false;
            }
        }
        return true;
    }
    if (w == 0 && !f(lane == 0, r, 0u)) return false;
    const HlDir d = hl_dir(a, dir);
    uint32_t b, e;
    hl_row(a, d.off, d.m, r, b, e);
    return hl_row_labels(a, d, dir, b, e, w, W, stat, f);
}

// Answers queries by labels: the label of s goes into the table, the label of
// t is looked up in it. A warp a query of the batch, those that outgrow its
// table appended to list (count in *list_cnt); then a block a query of that
// list. A query whose labels are missing, or outgrow a block's table, is
// appended to ovf (counted in *ovf_cnt) for the search kernels.
template <class Tab, int THREADS>
__global__ void __launch_bounds__(THREADS)
k_hl_query(HlArgs a, const uint32_t *src, const uint32_t *dst, uint64_t k, uint32_t *out, uint32_t *list,
           uint32_t *list_cnt, uint32_t *ovf, uint32_t *ovf_cnt) {
    extern __shared__ __align__(16) unsigned char hl_raw[];
    constexpr bool BLOCK = Tab::by_block;
    constexpr uint32_t W = BLOCK ? THREADS / 32 : 1, GT = W * 32;
    const uint32_t lane = lane_id(), warp = threadIdx.x >> 5;
    Tab &t = reinterpret_cast<Tab *>(hl_raw)[BLOCK ? 0 : warp];
    const uint32_t gt = BLOCK ? threadIdx.x : lane, gw = BLOCK ? warp : 0;
    auto sync = [] {
        if (BLOCK) __syncthreads();
        else __syncwarp();
    };
    pdl_wait();
    pdl_launch();
    QStat stat;
    const uint64_t items = BLOCK ? min((unsigned long long)*list_cnt, (unsigned long long)k) : k;
    const uint64_t groups = BLOCK ? gridDim.x : (uint64_t)gridDim.x * (THREADS / 32);
    for (uint64_t q = BLOCK ? blockIdx.x : blockIdx.x * (uint64_t)(THREADS / 32) + warp; q < items; q += groups) {
        const uint64_t i = BLOCK ? list[q] : q;
        const uint32_t s = src[i], v = dst[i];
        if (s >= a.n || v >= a.n) {
            if (gt == 0) {
                atomicOr(a.err, QERR_RANGE);
                out[i] = INF;
            }
            continue;
        }
        const uint32_t rs = a.rank[s], rt = a.rank[v];
        if (rs >= a.n || rt >= a.n) {
            if (gt == 0) {
                atomicOr(a.err, QERR_BOUND);
                out[i] = INF;
            }
            continue;
        }
        sync();
        hl_clear(t, gt, GT);
        if (BLOCK && gt == 0) {
            t.cnt = 0;
            t.bad = 0;
            t.kept = INF;  // the answer
        }
        sync();
        uint32_t cnt = 0;
        bool full = false;
        bool good = hl_endpoint(a, 0, rs, gw, W, stat, [&](bool on, uint32_t h, uint32_t d) {
            full = hl_full(t, cnt);
            if (full) return false;
            hl_lower(t, on, h, d, cnt);
            return true;
        });
        if (BLOCK && !good) t.bad = 1;
        sync();
        if (BLOCK) good = !t.bad;
        uint32_t mu = INF;
        if (good)
            good = hl_endpoint(a, 1, rt, gw, W, stat, [&](bool on, uint32_t h, uint32_t d) {
                if (on) mu = min(mu, sat_add(hl_find(t, h), d));
                return true;
            });
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) mu = min(mu, __shfl_xor_sync(FULL, mu, o));
        if (BLOCK) {
            if (!good) t.bad = 1;
            if (lane == 0 && mu != INF) atomicMin(&t.kept, mu);
            sync();
            good = !t.bad;
            mu = t.kept;
        }
        if (gt == 0) {
            if (good) out[i] = mu;
            else if (!BLOCK && full) list[atomicAdd(list_cnt, 1u)] = (uint32_t)i;
            else ovf[atomicAdd(ovf_cnt, 1u)] = (uint32_t)i;
        }
    }
    qb_flush_stat(stat, a.stats);
}

constexpr int HLW_THREADS = 128, HLB_THREADS = 1024, HLQ_THREADS = 128, HLQB_THREADS = 256;
constexpr size_t HLW_SMEM = sizeof(HlWarp) * (HLW_THREADS / 32);
constexpr size_t HLQ_SMEM = sizeof(HlQuery) * (HLQ_THREADS / 32);
constexpr auto hl_merge_warp = k_hl_merge<HlWarp, HLW_THREADS>;
constexpr auto hl_merge_block = k_hl_merge<HlBlock, HLB_THREADS>;
constexpr auto hl_query_warp = k_hl_query<HlQuery, HLQ_THREADS>;
constexpr auto hl_query_block = k_hl_query<HlQueryBlock, HLQB_THREADS>;
static_assert(sizeof(HlWarp) % 16 == 0 && sizeof(HlQuery) % 16 == 0, "a block's tables start on 16 bytes");

// The batch's labels fit this handle's hierarchy: no core (its rows are not
// acyclic), level sizes that add up, and an arena within the limit.
bool labels_possible(const ch_s *h) {
    return !h->hl_off && h->core_size == 0 && h->n >= 2 && h->n_up && h->n_down &&
           2ull * h->n * HL_AVG * sizeof(uint2) <= HL_MAX_BYTES;
}

}  // namespace

bool query_labels_prepare(ch_s *h, uint64_t k) {
    if (!labels_possible(h) || !batch_is_large(h, k)) return false;
    if (h->hl_arena.ptr) return true;
    std::vector<uint32_t> lv;
    if (!rank_levels(h, lv)) {
        h->hl_off = true;
        return false;
    }
    const size_t n = h->n;
    const size_t entries = std::max<size_t>(2 * n * HL_AVG, 1u << 16);
    // Labels only make the batch faster, and the arena is far larger than the
    // hierarchy: it takes at most a quarter of what the device has left, so that
    // what the caller allocates next fits as it would with searches.
    if (entries * sizeof(uint2) > dev_available() / 4) return false;
    try {
        DevBuf<uint2> arena;
        DevBuf<uint32_t> label;
        DevBuf<uint8_t> mark;
        DevBuf<unsigned long long> cursor;
        DevBuf<uint32_t> list;
        // labels of a level (2 n) or queries of a batch for the block kernels,
        // then their counts: one a level, and the batch's
        list.alloc(std::max<size_t>(2 * n, Q_CHUNK_MAX) + h->round_stats.size() + 1);
        label.alloc(4 * n);
        mark.alloc(2 * n);
        cursor.alloc(1);
        arena.alloc(entries);
        h->hl_label = std::move(label);
        h->hl_mark = std::move(mark);
        h->hl_list = std::move(list);
        h->hl_cursor = std::move(cursor);
        h->hl_arena = std::move(arena);
    } catch (const Error &e) {
        // no memory for labels: the searches need none of it
        if (!out_of_memory(e)) throw;
        h->hl_off = true;
        return false;
    }
    CH_CUDA_TRY(cudaFuncSetAttribute(hl_merge_warp, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)HLW_SMEM));
    CH_CUDA_TRY(cudaFuncSetAttribute(hl_merge_block, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                     (int)sizeof(HlBlock)));
    CH_CUDA_TRY(cudaFuncSetAttribute(hl_query_warp, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)HLQ_SMEM));
    CH_CUDA_TRY(cudaFuncSetAttribute(hl_query_block, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                     (int)sizeof(HlQueryBlock)));
    return true;
}

bool query_batch_labels(ch_s *h, const uint32_t *src, const uint32_t *dst, uint64_t k, uint32_t *dist_out,
                        uint32_t *ovf, uint32_t *ovf_cnt, cudaStream_t st) {
    if (!h->hl_arena.ptr) {
        // a capture must not allocate: it takes the searches unless an
        // earlier batch (or query_graph_create) has made the arena
        cudaStreamCaptureStatus cs = cudaStreamCaptureStatusNone;
        CH_CUDA_TRY(cudaStreamIsCapturing(st, &cs));
        if (cs != cudaStreamCaptureStatusNone) return false;
    }
    if (!query_labels_prepare(h, k)) return false;
    std::vector<uint32_t> lv;
    if (!rank_levels(h, lv)) return false;
    const uint32_t n = h->n;
    const size_t L = h->round_stats.size();
    HlArgs a;
    a.n = n;
    a.n_up = (uint32_t)h->n_up;
    a.n_dn = (uint32_t)h->n_down;
    a.rank = h->rank.ptr;
    a.up_off = h->up_off.ptr;
    a.dn_off = h->dn_off.ptr;
    a.up_adj = h->up_adj.ptr;
    a.dn_adj = h->dn_adj.ptr;
    a.mark = h->hl_mark.ptr;
    a.off = h->hl_label.ptr;
    a.size = h->hl_label.ptr + 2 * (size_t)n;
    a.arena = h->hl_arena.ptr;
    a.cap = std::min<uint64_t>(h->hl_arena.count, 0xFFFFFFFFull);
    a.cursor = h->hl_cursor.ptr;
    a.err = h->qerr.ptr;
    a.stats = h->q_stats.ptr;
    const int sms = device_sm_count();
    CH_CUDA_TRY(cudaMemsetAsync(a.mark, 0, 2 * (size_t)n, st));
    CH_CUDA_TRY(cudaMemsetAsync(a.size, 0xFF, 2 * (size_t)n * sizeof(uint32_t), st));
    CH_CUDA_TRY(cudaMemsetAsync(a.cursor, 0, sizeof(unsigned long long), st));
    uint32_t *list = h->hl_list.ptr, *counts = list + std::max<size_t>(2 * (size_t)n, Q_CHUNK_MAX);
    CH_CUDA_TRY(cudaMemsetAsync(counts, 0, (L + 1) * sizeof(uint32_t), st));
    k_hl_mark<<<grid_for(2 * k, 256, sms * 8), 256, 0, st>>>(a, src, dst, k, k >= 2ull * n);
    CH_CHECK_LAUNCH();
    // the run of small levels at the top: all of their labels, a block each
    size_t top = L;
    while (top > 0 && lv[top] - lv[top - 1] <= HL_BLOCK_LEVEL) --top;
    for (size_t l = 0; l < top; ++l)
        if (lv[l + 1] > lv[l])
            launch_pdl(k_hl_close, grid_for(2ull * (lv[l + 1] - lv[l]), 256, sms * 8), 256, 0, st, a, lv[l],
                       lv[l + 1]);
    const uint32_t prune_from = n - n / HL_PRUNE_PART;
    for (size_t l = L; l-- > 0;) {
        const uint32_t r0 = lv[l], r1 = lv[l + 1];
        if (r0 == r1) continue;
        if (l < top)
            launch_pdl(hl_merge_warp, grid_for(2ull * (r1 - r0), HLW_THREADS / 32, sms * 7), HLW_THREADS, HLW_SMEM,
                       st, a, r0, r1, prune_from, list, counts + l, false);
        launch_pdl(hl_merge_block, (unsigned)std::min<uint64_t>(2ull * (r1 - r0), sms * 2), HLB_THREADS,
                   sizeof(HlBlock), st, a, r0, r1, prune_from, list, counts + l, l < top);
    }
    launch_pdl(hl_query_warp, grid_for(k, HLQ_THREADS / 32, sms * 9), HLQ_THREADS, HLQ_SMEM, st, a, src, dst, k,
               dist_out, list, counts + L, ovf, ovf_cnt);
    launch_pdl(hl_query_block, sms * 6, HLQB_THREADS, sizeof(HlQueryBlock), st, a, src, dst, k, dist_out, list,
               counts + L, ovf, ovf_cnt);
    return true;
}

}  // namespace gbch

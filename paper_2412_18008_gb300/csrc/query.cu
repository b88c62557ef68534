// Batched CH s-t queries (Sec. 5 of arXiv 2412.18008): an upward search
// from s over E_up and an upward search from t over reversed E_down; the
// answer is the least d_s(v) + d_t(v) over the vertices both searches reach.
//
// The hierarchy is stored in rank order, so both searches run on a DAG whose
// edges all point to higher ranks. Each search is label-correcting: a
// frontier of improved vertices is expanded until no label changes, which
// gives exact shortest distances on any graph with positive weights, and
// the result cannot depend on the order of the relaxations.
//
// One block serves one query at a time and pulls the next index from a
// counter (persistent grid, three blocks per SM). Its labels live in a
// shared-memory hash table whose entries carry both directions' distances,
// so the meeting minimum is one pass over the table. A query whose search
// spaces do not fit is redone by a second kernel that keeps labels in dense
// per-vertex arrays in global memory (one block per array slot); so is every
// query of a hierarchy with a core that no table would hold.

#include <algorithm>
#include <mutex>
#include <vector>

#include "handle.cuh"
#include "qsearch.cuh"

namespace gbch {
namespace {

constexpr uint64_t Q_CHUNK = 1u << 22;  // queries per launch pair
// Counters of a batch, cleared at its start: what an earlier batch left behind,
// whole or not, does not matter to the next. (Small batches have none.)
constexpr uint32_t QWORK = 8;

// (The stalling variants are held to six resident blocks per SM, about 40
// registers a thread, so that six 2^11-slot blocks fit an SM.)
template <bool PRUNE, bool WARP, int TB, bool STALL, bool DELTA = false>
__global__ void __launch_bounds__(QB_THREADS, (STALL || DELTA) ? 6 : 1) k_query_block(QArgs a) {
    extern __shared__ __align__(16) unsigned char qb_raw[];
    QBSmem<TB> &q = *reinterpret_cast<QBSmem<TB> *>(qb_raw);
    const uint32_t tid = threadIdx.x;
    QStat stat;
    const uint64_t nitems = a.in_list ? a.work[a.in_cnt] : a.k;
    if (nitems == 0) return;
    qb_clear(q);
    while (true) {
        __syncthreads();
        if (tid == 0) q.item = atomicAdd(&a.work[a.ctr], 1u);
        __syncthreads();
        const uint32_t j = q.item;
        if (j >= nitems) break;
        const uint32_t i = a.in_list ? a.in_list[j] : j;
        if (i >= a.k) {
            if (tid == 0) atomicOr(a.err, QERR_BOUND);
            continue;
        }
        const uint32_t s = a.src[i], t = a.dst[i];
        if (s >= a.n || t >= a.n) {
            if (tid == 0) {
                atomicOr(a.err, QERR_RANGE);
                a.out[i] = INF;
                if (a.settled) a.settled[i] = 0;
            }
            continue;
        }
        const uint32_t rs = a.rank[s], rt = a.rank[t];
        if (rs >= a.n || rt >= a.n) {
            if (tid == 0) {
                atomicOr(a.err, QERR_BOUND);
                a.out[i] = INF;
            }
            continue;
        }
        uint32_t mu, cnt;
        if (!block_query<PRUNE, WARP, TB, STALL, DELTA>(q, a, rs, rt, mu, cnt, stat)) {
            if (tid == 0) a.ovf[atomicAdd(&a.work[a.ovf_cnt], 1u)] = i;
            continue;
        }
        if (tid == 0) {
            a.out[i] = mu;
            if (a.settled) a.settled[i] = cnt;
        }
    }
    qb_flush_stat(stat, a.stats);
}

// Queries on per-vertex label arrays in global memory (no capacity limit),
// one block per slot: those that overflow the shared tables, and every query
// of a hierarchy whose core is larger than a table (dense_first).
struct QDense {
    uint32_t *df, *db;   // labels, INF between queries
    uint32_t *queued;    // bit d: the vertex is in direction d's queue; 0 between queries
    uint32_t *fa, *fb;   // two frontiers of up to 2 n entries (vertex | direction << 31)
    uint32_t *touched;   // labels set, up to 2 n vertices
    uint32_t nslots;
};

constexpr int QD_THREADS = 1024;
constexpr uint32_t QD_WORDS = 9;  // uint32 per vertex of a slot
// Edges a level should expand: with fewer than the low mark the next level's
// bucket doubles, with more than the high mark it halves.
constexpr uint32_t QD_EDGES_LOW = 4096, QD_EDGES_HIGH = 32768;

struct QDSmem {
    // one tile of frontier entries: exclusive prefix of their out-degrees,
    // first edge index, label, direction
    uint32_t excl[QD_THREADS], beg[QD_THREADS], lab[QD_THREADS];
    uint8_t dir[QD_THREADS];
    uint32_t wtot[QD_THREADS / 32];
    uint32_t cnt3[3], lmin3[3][2];  // queue sizes and least queued labels per level (mod 3)
    uint32_t item, nt, mu, delta, edges;
};

// Both searches of a query at once, label-correcting, in levels like the
// shared-table search's (block_search): a level expands the queued vertices
// within `delta` of their direction's least queued label, keeps the others
// and drops those whose label is not below the best meeting sum mu. Inside the
// core, whose edges both directions hold, a search need not reach past the
// middle of the path: a core vertex x is dropped when its label plus the other
// direction's least queued label is not below mu. (A path through x shorter
// than mu then has its remainder at labels the other direction has settled,
// x among them, so x already holds both labels and mu counts their sum.
// Vertices below the core are never dropped for this: only their own
// direction climbs to the core.) Exhaustive searches (not PRUNE) expand
// everything at once.
//
// mu_out and cnt_out are, in every thread, the answer and the labels set.
//
// Bound by the level chain's round trips to L2 (queue, label, offsets, edge,
// label): the edges of a tile of 1024 entries are spread over all 1024 threads
// by a block-wide scan, so that a hub's row costs no more than as many edges
// of small rows, and the bucket width follows the work of the level before
// (a fixed one is wrong by orders of magnitude from one graph to the next).
// RMAT 2^15 (5,648 core vertices), 96 queries: 1.0 ms; a thread per
// frontier vertex, both searches exhaustive and one after the other, after
// two passes of overflowing table searches: 445 ms.
template <bool PRUNE>
__device__ void dense_query(QDSmem &q, const QArgs &a, const QDense &dn, uint32_t rs, uint32_t rt, uint32_t &mu_out,
                            uint32_t &cnt_out, QStat &stat) {
    const uint32_t tid = threadIdx.x, lane = lane_id(), warp = tid >> 5;
    const size_t base = (size_t)blockIdx.x * a.n;
    uint32_t *df = dn.df + base, *db = dn.db + base, *queued = dn.queued + base;
    uint32_t *const fra = dn.fa + 2 * base, *const frb = dn.fb + 2 * base;
    uint32_t *touched = dn.touched + 2 * base;
    __syncthreads();
    if (tid == 0) {
        df[rs] = 0;
        db[rt] = 0;
        queued[rs] = rs == rt ? 3u : 1u;
        if (rs != rt) queued[rt] = 2u;
        touched[0] = rs;
        touched[1] = rt;
        fra[0] = rs;
        fra[1] = rt | 0x80000000u;
        q.nt = 2;
        q.mu = rs == rt ? 0u : INF;
        q.cnt3[0] = 2;
        q.cnt3[1] = 0;
        q.lmin3[0][0] = q.lmin3[0][1] = 0;
        q.lmin3[1][0] = q.lmin3[1][1] = INF;
        q.delta = a.dense_delta;
        q.edges = 0;
    }
    for (uint32_t lvl = 0;; ++lvl) {
        __syncthreads();
        const uint32_t nfront = q.cnt3[lvl % 3];
        const uint32_t mu0 = q.mu, minf = q.lmin3[lvl % 3][0], minb = q.lmin3[lvl % 3][1];
        uint32_t delta = q.delta;
        const uint32_t did = q.edges;
        if (nfront == 0) break;
        if (lvl >= (1u << 30)) {  // the least label grows every other level at the latest
            if (tid == 0) atomicOr(a.err, QERR_BOUND);
            break;
        }
        if (lvl && did < QD_EDGES_LOW) delta = min(2u * delta, 1u << 30);
        else if (did > QD_EDGES_HIGH) delta = max(delta / 2u, 1u);
        const uint32_t thrf = sat_add(minf, delta), thrb = sat_add(minb, delta);
        __syncthreads();
        if (tid == 0) {
            q.cnt3[(lvl + 2) % 3] = 0;
            q.lmin3[(lvl + 2) % 3][0] = q.lmin3[(lvl + 2) % 3][1] = INF;
            q.delta = delta;
            q.edges = 0;
        }
        const uint32_t *cur = lvl & 1u ? frb : fra;
        uint32_t *nxt = lvl & 1u ? fra : frb;
        uint32_t *ncnt = &q.cnt3[(lvl + 1) % 3];
        uint32_t lmf = INF, lmb = INF;  // least labels this thread queues
        for (uint32_t t0 = 0; t0 < nfront; t0 += QD_THREADS) {
            // Barriers keep this part of a tile, which reads labels and takes
            // vertices out of the queue, apart from the relaxations of this
            // tile and of the one before: a label read here is current, and one
            // lowered later finds the vertex's bit clear and queues it again.
            const uint32_t fi = t0 + tid;
            const uint32_t ent = fi < nfront ? __ldcg(cur + fi) : 0;
            const uint32_t x = ent & 0x7FFFFFFFu, dir = ent >> 31;
            bool ok = fi < nfront && x < a.n;
            if (fi < nfront && !ok) atomicOr(a.err, QERR_BOUND);
            uint32_t *dist = dir ? db : df;
            const uint32_t lab = ok ? __ldcg(dist + x) : INF;
            bool keep = false;
            if (PRUNE) {
                const bool drop = ok && (lab >= mu0 || (x >= a.core_first &&
                                                        sat_add(lab, dir ? minf : minb) >= mu0));
                keep = ok && !drop && lab > (dir ? thrb : thrf);
                if (drop) {
                    atomicAnd(&queued[x], ~(1u << dir));
                    ok = false;
                }
                const uint32_t m = __ballot_sync(FULL, keep);
                if (m) {
                    uint32_t p = 0;
                    const uint32_t leader = __ffs(m) - 1;
                    if (lane == leader) p = atomicAdd(ncnt, (uint32_t)__popc(m));
                    p = __shfl_sync(FULL, p, leader) + __popc(m & ((1u << lane) - 1u));
                    if (keep) {
                        if (p < 2u * a.n) nxt[p] = ent;
                        else atomicOr(a.err, QERR_BOUND);
                        if (dir) lmb = min(lmb, lab);
                        else lmf = min(lmf, lab);
                    }
                }
                if (keep) ok = false;
            }
            uint32_t b = 0, cnt = 0;
            if (ok) {
                atomicAnd(&queued[x], ~(1u << dir));
                const uint32_t *off = dir ? a.dn_off : a.up_off;
                b = off[x];
                const uint32_t e = off[x + 1];
                if (b <= e && e <= (dir ? a.n_dn : a.n_up)) cnt = e - b;
                else atomicOr(a.err, QERR_BOUND);
            }
            stat.exp += cnt ? 1u : 0u;
            const uint32_t incl = warp_incl_scan(cnt);
            if (lane == 31) q.wtot[warp] = incl;
            q.beg[tid] = b;
            q.lab[tid] = lab;
            q.dir[tid] = (uint8_t)dir;
            __syncthreads();
            const uint32_t wt = q.wtot[lane];
            const uint32_t wincl = warp_incl_scan(wt);
            const uint32_t total = __shfl_sync(FULL, wincl, 31);
            q.excl[tid] = __shfl_sync(FULL, wincl - wt, warp) + incl - cnt;
            if (tid == 0) q.edges += total;
            __syncthreads();
            for (uint32_t e0 = tid; e0 < total; e0 += QD_THREADS) {
                // owner entry: the largest k with excl[k] <= e0
                uint32_t k = 0;
#pragma unroll
                for (uint32_t step = QD_THREADS / 2; step > 0; step >>= 1)
                    if (q.excl[k + step] <= e0) k += step;
                ++stat.edges;
                const uint32_t edir = q.dir[k];
                const uint2 e = (edir ? a.dn_adj : a.up_adj)[q.beg[k] + (e0 - q.excl[k])];
                const uint32_t nd = sat_add(q.lab[k], e.y);
                if (e.x >= a.n) {
                    atomicOr(a.err, QERR_BOUND);
                    continue;
                }
                if (nd == INF) continue;
                if (PRUNE && nd >= *(volatile uint32_t *)&q.mu) continue;
                uint32_t *ed = edir ? db : df;
                if (nd >= __ldcg(ed + e.x)) continue;
                const uint32_t old = atomicMin(&ed[e.x], nd);
                if (nd >= old) continue;
                if (old == INF) {
                    const uint32_t p = atomicAdd(&q.nt, 1u);
                    if (p < 2u * a.n) touched[p] = e.x;
                    else atomicOr(a.err, QERR_BOUND);
                }
                if (edir) lmb = min(lmb, nd);
                else lmf = min(lmf, nd);
                if (PRUNE) {
                    const uint32_t other = __ldcg((edir ? df : db) + e.x);
                    if (other != INF) atomicMin(&q.mu, sat_add(nd, other));
                }
                if (!(atomicOr(&queued[e.x], 1u << edir) & (1u << edir))) {
                    const uint32_t p = atomicAdd(ncnt, 1u);
                    if (p < 2u * a.n) nxt[p] = e.x | (edir << 31);
                    else atomicOr(a.err, QERR_BOUND);
                }
            }
            __syncthreads();
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            lmf = min(lmf, __shfl_xor_sync(FULL, lmf, o));
            lmb = min(lmb, __shfl_xor_sync(FULL, lmb, o));
        }
        if (lane == 0) {
            if (lmf != INF) atomicMin(&q.lmin3[(lvl + 1) % 3][0], lmf);
            if (lmb != INF) atomicMin(&q.lmin3[(lvl + 1) % 3][1], lmb);
        }
    }
    __syncthreads();
    // the answer: the least meeting sum over the vertices reached
    const uint32_t nt = min(q.nt, 2u * a.n);
    if (tid == 0) q.mu = INF;
    __syncthreads();
    uint32_t mu = INF;
    for (uint32_t p = tid; p < nt; p += QD_THREADS) {
        const uint32_t v = __ldcg(touched + p);
        mu = min(mu, sat_add(__ldcg(df + v), __ldcg(db + v)));
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) mu = min(mu, __shfl_xor_sync(FULL, mu, o));
    if (lane == 0 && mu != INF) atomicMin(&q.mu, mu);
    __syncthreads();
    mu_out = q.mu;
    cnt_out = nt;
    for (uint32_t p = tid; p < nt; p += QD_THREADS) {
        const uint32_t v = __ldcg(touched + p);
        df[v] = INF;
        db[v] = INF;
        queued[v] = 0;
    }
}

// Query i's endpoints as ranks; false (in every thread), with the error
// recorded and the answer INF, when an id is out of range.
__device__ __forceinline__ bool query_ranks(const QArgs &a, uint32_t i, uint32_t &rs, uint32_t &rt) {
    const uint32_t s = a.src ? a.src[i] : a.one_src, t = a.dst[i];
    rs = s < a.n ? a.rank[s] : INF;
    rt = t < a.n ? a.rank[t] : INF;
    if (rs < a.n && rt < a.n) return true;
    if (threadIdx.x == 0) {
        atomicOr(a.err, s >= a.n || t >= a.n ? QERR_RANGE : QERR_BOUND);
        a.out[i] = INF;
        if (a.settled) a.settled[i] = 0;
    }
    return false;
}

template <bool PRUNE>
__global__ void __launch_bounds__(QD_THREADS) k_query_dense(QArgs a, QDense dn) {
    __shared__ QDSmem q;
    const uint32_t tid = threadIdx.x;
    pdl_wait();
    const uint32_t nitems = a.ovf_flags || a.dense_first ? (uint32_t)a.k : a.work[a.ovf_cnt];
    QStat stat;
    bool worked = false;
    for (uint32_t next = blockIdx.x; nitems;) {
        uint32_t i;
        if (a.ovf_flags) {
            if (next >= nitems) break;
            i = next;
            next += gridDim.x;
            if (!a.ovf[i]) continue;
        } else {
            __syncthreads();
            if (tid == 0) q.item = atomicAdd(&a.work[1], 1u);
            __syncthreads();
            if (q.item >= nitems) break;
            i = a.dense_first ? q.item : a.ovf[q.item];
        }
        worked = true;
        if (i >= a.k) {
            if (tid == 0) atomicOr(a.err, QERR_BOUND);
            continue;
        }
        uint32_t rs, rt, mu, cnt;
        if (!query_ranks(a, i, rs, rt)) continue;
        dense_query<PRUNE>(q, a, dn, rs, rt, mu, cnt, stat);
        if (tid == 0) {
            a.out[i] = mu;
            if (a.settled) a.settled[i] = cnt;
        }
    }
    if (worked) qb_flush_stat(stat, a.stats);
}

// Small batches: a block of 1024 threads a query, in one launch; queries that
// outgrow the table are flagged for the dense kernel behind it (a flag a query
// in place of a list, so that there is no counter to clear). With that few
// queries the time of one counts: the chain of round trips of its levels, and
// how fast one SM issues their instructions. The levels are block_search's,
// with stalling and buckets, but a warp takes whole rows: a level's entries
// are dealt to 32 warps, most of which hold one or two, and each row's lanes
// read its stall edges and its out-edges together, without the scans and owner
// searches of flattened rows. An entry found stalled drops the out-edges it has
// read. Geometric graph of 1M vertices, back to back: 63 us for a query, 114 for
// 152, against 122 and 216 by the launches that larger batches take (a query
// that is waited for takes 80 us, launch and wait included). (Rows
// flattened over the whole block: 80 and 133 us. Whole rows in the blocks of
// 256 threads that larger batches use, several rows a warp: slower, 302 us for
// 777 queries against 254.)
constexpr int QS_THREADS = 1024;

template <int TB>
__device__ bool row_search(QBSmem<TB> &q, const QArgs &a, QStat &stat) {
    constexpr uint32_t FC = QBSmem<TB>::FC, CW = QBSmem<TB>::CW;
    const uint32_t tid = threadIdx.x, lane = lane_id(), warp = tid >> 5;
    constexpr uint32_t W = QS_THREADS / 32;
    for (uint32_t lvl = 1;; ++lvl) {
        __syncthreads();
        const uint32_t cur = (lvl - 1) & 1u;
        const uint32_t nfront = q.cnt3[(lvl - 1) % 3];
        if (nfront > FC) return false;
        if (nfront == 0) return true;
        if (lvl >= 0xFFFFu) {
            if (tid == 0) atomicOr(a.err, QERR_BOUND);
            return false;
        }
        const uint32_t thr_f = sat_add(q.lmin3[(lvl - 1) % 3][0], a.delta),
                       thr_b = sat_add(q.lmin3[(lvl - 1) % 3][1], a.delta);
        if (tid == 0) {
            q.cnt3[(lvl + 1) % 3] = 0;
            q.lmin3[(lvl + 1) % 3][0] = q.lmin3[(lvl + 1) % 3][1] = INF;
        }
        for (uint32_t j = tid; j < 2u * CW; j += QS_THREADS) (&q.claim[(lvl + 1) & 1u][0][0])[j] = 0;
        const uint32_t nxt_cnt = lvl % 3;
        uint32_t *next_front = q.front[cur ^ 1u];
        uint32_t lmf = INF, lmb = INF;
        for (uint32_t p0 = 0; p0 + warp < nfront; p0 += QS_THREADS) {
            const uint32_t fi = p0 + warp + W * lane;
            bool fv = fi < nfront && fi < FC;
            const uint32_t ent = fv ? q.front[cur][fi] : 0;
            const uint32_t dir = ent >> 31, slot = ent & 0x7FFFFFFFu;
            const uint32_t lab = fv && slot < QBSmem<TB>::T ? (dir ? q.db[slot] : q.df[slot]) : INF;
            if (fv && lab >= q.mu) {
                fv = false;  // cannot improve the answer
            } else if (fv && lab > (dir ? thr_b : thr_f)) {
                // stays queued
                if (qb_claim(q, slot, dir, lvl)) {
                    const uint32_t p = atomicAdd(&q.cnt3[nxt_cnt], 1u);
                    if (p < FC) next_front[p] = ent;
                    if (dir) lmb = min(lmb, lab);
                    else lmf = min(lmf, lab);
                }
                fv = false;
            }
            uint32_t b, cnt, dx, sb, se;
            qb_entry_both(q, a, fv, ent, b, cnt, dx, sb, se);
            uint32_t scnt = 0;
            if (cnt && sb <= se && se <= (dir ? a.n_up : a.n_dn)) scnt = se - sb;
            else if (cnt) atomicOr(a.err, QERR_BOUND);
            stat.exp += cnt ? 1u : 0u;
            stat.edges += scnt;
            for (uint32_t m = __ballot_sync(FULL, cnt != 0); m; m &= m - 1) {
                const uint32_t o = __ffs(m) - 1;
                const uint32_t ob = __shfl_sync(FULL, b, o), oc = __shfl_sync(FULL, cnt, o),
                               od = __shfl_sync(FULL, dx, o), osb = __shfl_sync(FULL, sb, o),
                               osc = __shfl_sync(FULL, scnt, o), odir = __shfl_sync(FULL, ent, o) >> 31;
                const uint2 *oadj = (odir ? a.dn_adj : a.up_adj) + ob, *sadj = (odir ? a.up_adj : a.dn_adj) + osb;
                uint2 y = lane < oc ? oadj[lane] : make_uint2(0, 0);
                bool stalled = false;
                for (uint32_t j = lane; j < osc; j += 32) {
                    const uint2 z = sadj[j];
                    const uint32_t at = z.x < a.n ? qb_find<TB>(q.key, z.x) : EMPTY;
                    stalled |= at != EMPTY && sat_add(odir ? q.db[at] : q.df[at], z.y) < od;
                }
                if (__any_sync(FULL, stalled)) continue;
                stat.edges += lane == 0 ? oc : 0;
                for (uint32_t j = lane; j < oc;) {
                    qb_relax<true, TB, true>(q, a, odir, y, od, lvl, nxt_cnt, next_front, lmf, lmb);
                    j += 32;
                    if (j < oc) y = oadj[j];
                }
            }
        }
        lmf = __reduce_min_sync(FULL, lmf);
        lmb = __reduce_min_sync(FULL, lmb);
        if (lane == 0) {
            if (lmf != INF) atomicMin(&q.lmin3[nxt_cnt][0], lmf);
            if (lmb != INF) atomicMin(&q.lmin3[nxt_cnt][1], lmb);
        }
    }
}

__global__ void __launch_bounds__(QS_THREADS, 1) k_query_small(QArgs a) {
    extern __shared__ __align__(16) unsigned char qb_raw[];
    QBSmem<12> &q = *reinterpret_cast<QBSmem<12> *>(qb_raw);
    QStat stat;
    pdl_launch();
    qb_clear(q);
    for (uint32_t i = blockIdx.x; i < a.k; i += gridDim.x) {
        uint32_t rs, rt, mu, cnt;
        bool ok = true;
        if (query_ranks(a, i, rs, rt)) {
            ok = block_query_by(q, a, rs, rt, mu, cnt, [&] { return row_search<12>(q, a, stat); });
            if (threadIdx.x == 0 && ok) a.out[i] = mu;
        }
        if (threadIdx.x == 0) a.ovf[i] = !ok;
    }
    qb_flush_stat(stat, a.stats);
}

// Resident blocks per SM of each block-kernel configuration
// [table bits == 11][block-flat, warp-flat, warp-flat with stalling,
// the same with delta-stepping levels][threads == 256], resolved once.
int g_qb_bps[2][4][2] = {{{-1, -1}, {-1, -1}, {-1, -1}, {-1, -1}}, {{-1, -1}, {-1, -1}, {-1, -1}, {-1, -1}}};

template <int TB>
void qb_resolve(int s) {
    const int smem = (int)sizeof(QBSmem<TB>);
    CH_CUDA_TRY(cudaFuncSetAttribute(k_query_block<true, true, TB, true, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem));
    CH_CUDA_TRY(cudaFuncSetAttribute(k_query_block<true, false, TB, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem));
    CH_CUDA_TRY(cudaFuncSetAttribute(k_query_block<false, false, TB, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem));
    CH_CUDA_TRY(cudaFuncSetAttribute(k_query_block<true, true, TB, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem));
    CH_CUDA_TRY(cudaFuncSetAttribute(k_query_block<false, true, TB, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem));
    CH_CUDA_TRY(cudaFuncSetAttribute(k_query_block<true, true, TB, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem));
    for (int l = 0; l < 4; ++l)
        for (int t = 0; t < 2; ++t) {
            int b = 0;
            const int threads = t ? 256 : 128;
            if (l == 3) CH_CUDA_TRY(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&b, k_query_block<true, true, TB, true, true>, threads, smem));
            else if (l == 2) CH_CUDA_TRY(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&b, k_query_block<true, true, TB, true>, threads, smem));
            else if (l == 1) CH_CUDA_TRY(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&b, k_query_block<true, true, TB, false>, threads, smem));
            else CH_CUDA_TRY(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&b, k_query_block<true, false, TB, false>, threads, smem));
            g_qb_bps[s][l][t] = std::max(1, b);
        }
}

void qb_resolve_occupancy() {
    if (g_qb_bps[0][0][0] >= 0) return;
    qb_resolve<12>(0);
    CH_CUDA_TRY(cudaFuncSetAttribute(k_query_small, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(QBSmem<12>)));
    qb_resolve<11>(1);
}

template <int TB>
void launch_tb(const QArgs &a, bool prune, bool warp, bool stall, bool delta, int blocks, int threads,
               cudaStream_t st) {
    const size_t smem = sizeof(QBSmem<TB>);
    if (warp) {
        if (prune && stall && delta) k_query_block<true, true, TB, true, true><<<blocks, threads, smem, st>>>(a);
        else if (prune && stall) k_query_block<true, true, TB, true><<<blocks, threads, smem, st>>>(a);
        else if (prune) k_query_block<true, true, TB, false><<<blocks, threads, smem, st>>>(a);
        else k_query_block<false, true, TB, false><<<blocks, threads, smem, st>>>(a);
    } else {
        if (prune) k_query_block<true, false, TB, false><<<blocks, threads, smem, st>>>(a);
        else k_query_block<false, false, TB, false><<<blocks, threads, smem, st>>>(a);
    }
    CH_CHECK_LAUNCH();
}

// Launches one block-kernel pass in the handle's layout and block size: a
// persistent grid of as many blocks as are resident at once (no more than
// the items), with 2^11-slot tables when small is set, else 2^12. Stall on
// demand applies to pruned searches in the warp layout only, and
// delta-stepping levels to those with stalling.
void launch_query_block(const ch_s *h, const QArgs &a, bool prune, bool small, uint64_t items,
                        cudaStream_t st) {
    const bool warp = h->q_layout == CH_QUERY_WARP_FLAT;
    const bool stall = warp && prune && h->q_stall;
    const bool delta = stall && h->q_delta != 0;
    const int l = delta ? 3 : (stall ? 2 : (warp ? 1 : 0));
    const int t = h->q_threads == 256 ? 1 : 0;
    const int threads = t ? 256 : 128;
    const int blocks = (int)std::max<uint64_t>(
        1, std::min<uint64_t>(items, (uint64_t)device_sm_count() * g_qb_bps[small ? 1 : 0][l][t]));
    if (small) launch_tb<11>(a, prune, warp, stall, delta, blocks, threads, st);
    else launch_tb<12>(a, prune, warp, stall, delta, blocks, threads, st);
}

// Weights of `cnt` evenly spaced entries of an adjacency array.
__global__ void k_sample_weights(const uint2 *adj, uint64_t m, uint32_t *out, uint32_t cnt) {
    const uint32_t i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < cnt) out[i] = adj[(uint64_t)i * m / cnt].y;
}

constexpr uint32_t WSCALE_SAMPLE = 1024;
constexpr uint32_t DELTA_DEFAULT_MULT = 128;         // default delta, in weight scales
constexpr uint32_t DELTA_TUNE_MULT[3] = {64, 128, 256};  // autotuner candidates 12-14

// mult x the weight scale, at least 1 and below INF.
uint32_t delta_of(const ch_s *h, uint32_t mult) {
    const uint64_t d = (uint64_t)mult * h->q_wscale;
    return (uint32_t)std::max<uint64_t>(1, std::min<uint64_t>(d, INF - 1));
}

}  // namespace

void query_init(ch_s *h) {
    const uint32_t n = h->n;
    h->qerr.alloc(1);
    h->qerr.zero(0);
    h->qwork.alloc(QWORK);
    h->q_ovf_cap = Q_CHUNK;
    h->q_ovf_list.alloc(2 * Q_CHUNK);  // overflow lists of the two block-kernel passes
    // as many slots as the chip runs blocks of the dense kernel at once (two
    // an SM), within 1 GiB
    const uint64_t per_slot = (uint64_t)std::max<uint32_t>(n, 1) * QD_WORDS * 4;
    h->q_slots = (uint32_t)std::max<uint64_t>(
        2, std::min<uint64_t>(2 * (uint64_t)device_sm_count(), (1024ull << 20) / per_slot));
    const size_t sn = (size_t)h->q_slots * std::max<uint32_t>(n, 1);
    h->q_dense.alloc(sn * QD_WORDS);
    // df, db: INF; queue bits: 0; the rest need no initial value
    CH_CUDA_TRY(cudaMemset(h->q_dense.ptr, 0xFF, sn * 2 * 4));
    CH_CUDA_TRY(cudaMemset(h->q_dense.ptr + 2 * sn, 0, sn * 4));
    h->q_stats.alloc(2);
    h->q_stats.zero(0);
    qb_resolve_occupancy();
    // weight scale of the hierarchy (the median of sampled E_up weights) and
    // the default delta
    h->q_wscale = 1;
    if (h->n_up > 0) {
        DevBuf<uint32_t> wb;
        wb.alloc(WSCALE_SAMPLE);
        k_sample_weights<<<(WSCALE_SAMPLE + 255) / 256, 256>>>(h->up_adj.ptr, h->n_up, wb.ptr, WSCALE_SAMPLE);
        CH_CHECK_LAUNCH();
        std::vector<uint32_t> w(WSCALE_SAMPLE);
        CH_CUDA_TRY(cudaMemcpy(w.data(), wb.ptr, WSCALE_SAMPLE * sizeof(uint32_t), cudaMemcpyDeviceToHost));
        std::nth_element(w.begin(), w.begin() + WSCALE_SAMPLE / 2, w.end());
        h->q_wscale = std::max<uint32_t>(1, w[WSCALE_SAMPLE / 2]);
    }
    // Without delta when the hierarchy has a core: its queries search the
    // core, outgrow the shared tables and are redone on the dense kernel;
    // delta-stepping levels only delay that overflow.
    h->q_delta = h->core_size ? 0 : delta_of(h, DELTA_DEFAULT_MULT);
    CH_CUDA_TRY(cudaDeviceSynchronize());
}

namespace {

// The label arrays of the dense kernel's slots.
QDense dense_slots(const ch_s *h) {
    const size_t sn = (size_t)h->q_slots * std::max<uint32_t>(h->n, 1);
    QDense dn;
    dn.df = h->q_dense.ptr;
    dn.db = dn.df + sn;
    dn.queued = dn.df + 2 * sn;
    dn.fa = dn.df + 3 * sn;
    dn.fb = dn.df + 5 * sn;
    dn.touched = dn.df + 7 * sn;
    dn.nslots = h->q_slots;
    return dn;
}

// Searches of a core larger than this reach more vertices than a table of
// 2^12 slots takes, so their queries go to the dense kernel at once (without
// a core table, which keeps the searches out of the core). Half the table:
// the searches below the core need room too. 96 queries of RMAT 2^15 (core
// 5,648): 320 ms of the 445 were the two passes that overflowed.
constexpr uint64_t DENSE_FIRST_CORE = 2048;

// What every kernel of a batch needs of the hierarchy.
QArgs hierarchy_args(const ch_s *h) {
    QArgs a;
    a.n = h->n;
    a.n_up = (uint32_t)h->n_up;
    a.n_dn = (uint32_t)h->n_down;
    a.rank = h->rank.ptr;
    a.up_off = h->up_off.ptr;
    a.dn_off = h->dn_off.ptr;
    a.up_adj = h->up_adj.ptr;
    a.dn_adj = h->dn_adj.ptr;
    a.err = h->qerr.ptr;
    a.stats = h->q_stats.ptr;
    a.core_tab = h->core_n ? h->core_tab.ptr : nullptr;
    a.core_lo = h->core_lo;
    a.core_n = h->core_n;
    a.core_first = (uint32_t)(h->n - h->core_size);
    a.dense_delta = std::max<uint32_t>(1, h->q_wscale / 8);
    a.dense_first = !h->core_n && h->core_size > DENSE_FIRST_CORE;
    a.delta = h->q_delta ? h->q_delta : INF;
    return a;
}

// The dense kernel over a batch's overflowed queries (or all of them).
void launch_query_dense(const ch_s *h, const QArgs &a, bool prune, uint64_t k, cudaStream_t st) {
    const QDense dn = dense_slots(h);
    const unsigned blocks = (unsigned)std::min<uint64_t>(dn.nslots, k);
    launch_pdl(prune ? k_query_dense<true> : k_query_dense<false>, blocks, QD_THREADS, 0, st, a, dn);
}

}  // namespace

namespace {

// A batch with at most one query an SM is small: two of its 1024-thread
// blocks do not fit an SM (60 registers a thread), and at two queries an SM
// both ways take the same time (1M vertices, 304 queries: 182 and 212 us; 256K
// vertices: 126 and 120 us). Not for queries that need the dense kernel.
bool small_batch(const QArgs &a, uint64_t k) { return k <= (uint64_t)device_sm_count() && !a.dense_first; }

// (a.ovf: room for k flags)
void launch_query_small(const ch_s *h, QArgs &a, cudaStream_t st) {
    a.ovf_flags = true;
    k_query_small<<<(unsigned)a.k, QS_THREADS, sizeof(QBSmem<12>), st>>>(a);
    CH_CHECK_LAUNCH();
    launch_query_dense(h, a, true, a.k, st);
}

}  // namespace

bool query_batch_small(ch_s *h, const uint32_t *src, uint32_t one_src, const uint32_t *dst, uint64_t k,
                       uint32_t *dist_out, cudaStream_t st) {
    QArgs a = hierarchy_args(h);
    if (!small_batch(a, k)) return false;
    a.src = src;
    a.one_src = one_src;
    a.dst = dst;
    a.out = dist_out;
    a.settled = nullptr;
    a.k = k;
    a.ovf = h->q_ovf_list.ptr;
    launch_query_small(h, a, st);
    return true;
}

void query_batch(ch_s *h, const uint32_t *src, const uint32_t *dst, uint64_t k,
                 uint32_t *dist_out, uint32_t *settled_out, cudaStream_t st, bool searches_only) {
    if (k == 0) return;
    if (!settled_out && !searches_only && query_batch_small(h, src, 0, dst, k, dist_out, st)) return;
    for (uint64_t c0 = 0; c0 < k; c0 += Q_CHUNK) {
        const uint64_t kc = std::min<uint64_t>(Q_CHUNK, k - c0);
        QArgs a = hierarchy_args(h);
        a.src = src + c0;
        a.dst = dst + c0;
        a.out = dist_out + c0;
        a.settled = settled_out ? settled_out + c0 : nullptr;
        a.k = kc;
        a.work = h->qwork.ptr;
        a.in_list = nullptr;
        a.in_cnt = 0;
        CH_CUDA_TRY(cudaMemsetAsync(a.work, 0, QWORK * sizeof(uint32_t), st));
        // Pruned searches unless the caller asked for search-space sizes,
        // which are defined by the exhaustive upward searches.
        const bool prune = settled_out == nullptr;
        if (a.dense_first) {
            launch_query_dense(h, a, prune, kc, st);
            continue;
        }
        uint32_t *const list = h->q_ovf_list.ptr, *const list2 = list + Q_CHUNK;
        if (prune && !searches_only && query_batch_labels(h, a.src, a.dst, kc, a.out, list, a.work + 4, st)) {
            // the queries that the labels could not answer, by searches
            a.in_list = list;
            a.in_cnt = 4;
        }
        if (h->q_small_first) {
            // pass 1 on small tables (twice the resident queries); the
            // queries that overflow them are redone on the large tables
            a.ctr = 0;
            a.ovf = list2;
            a.ovf_cnt = 5;
            launch_query_block(h, a, prune, true, kc, st);
            a.in_list = list2;
            a.in_cnt = 5;
        }
        a.ctr = 3;
        a.ovf = a.in_list == list ? list2 : list;  // (the list that is used up)
        a.ovf_cnt = 2;
        launch_query_block(h, a, prune, false, kc, st);
        launch_query_dense(h, a, prune, kc, st);
    }
}

// ---------------------------------------------------------------------------
// Configuration, autotuning, work counters, CUDA graphs
// ---------------------------------------------------------------------------

namespace {

// Seeded uniform pairs for the autotuner's sample (MurmurHash3 finaliser of
// a counter, reduced modulo n).
__global__ void k_sample_pairs(uint32_t *s, uint32_t *t, uint64_t k, uint32_t n, uint32_t seed) {
    for (uint64_t i = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; i < k;
         i += (uint64_t)gridDim.x * blockDim.x) {
        const uint32_t a = murmur_fmix32((uint32_t)(2 * i) ^ murmur_fmix32(seed));
        const uint32_t b = murmur_fmix32((uint32_t)(2 * i + 1) ^ murmur_fmix32(seed + 0x9e3779b9u));
        s[i] = a % n;
        t[i] = b % n;
    }
}

}  // namespace

void query_set_config(ch_s *h, uint32_t layout, uint32_t threads, uint32_t small_first, uint32_t stall,
                      uint32_t delta) {
    if ((layout != CH_QUERY_BLOCK_FLAT && layout != CH_QUERY_WARP_FLAT) || (threads != 128 && threads != 256) ||
        small_first > 1 || stall > 1 || (stall && layout != CH_QUERY_WARP_FLAT) || (delta && !stall) ||
        delta == INF)
        throw Error{CH_EINVAL, "query configuration: layout BLOCK_FLAT or WARP_FLAT, threads 128 or 256, "
                               "small_first 0 or 1, stall 0 or 1 (WARP_FLAT only), delta below 2^32 - 1 "
                               "(with stall 1 only when not 0)"};
    h->q_layout = layout;
    h->q_threads = threads;
    h->q_small_first = small_first;
    h->q_stall = stall;
    h->q_delta = delta;
    h->q_fits_small = -1;
}

bool query_fits_small(ch_s *h, cudaStream_t st) {
    constexpr uint32_t SAMPLE = 512, MOST = SAMPLE / 32;  // (see server_start for the line)
    if (h->q_fits_small >= 0) return h->q_fits_small;
    if (h->n == 0) return true;
    // buffers of its own: a batch may be in flight on another stream
    DevBuf<uint32_t> buf;
    buf.alloc(QWORK + 4 * SAMPLE);
    CH_CUDA_TRY(cudaMemsetAsync(buf.ptr, 0, QWORK * sizeof(uint32_t), st));
    uint32_t *s = buf.ptr + QWORK, *t = s + SAMPLE;
    k_sample_pairs<<<(SAMPLE + 255) / 256, 256, 0, st>>>(s, t, SAMPLE, h->n, 1u);
    CH_CHECK_LAUNCH();
    QArgs a = hierarchy_args(h);
    a.core_tab = nullptr;  // (the server's searches do not use it)
    a.stats = nullptr;
    a.settled = nullptr;
    a.src = s;
    a.dst = t;
    a.out = t + SAMPLE;
    a.k = SAMPLE;
    a.work = buf.ptr;
    a.in_list = nullptr;
    a.ctr = 0;
    a.ovf = a.out + SAMPLE;
    a.ovf_cnt = 2;
    launch_query_block(h, a, true, true, SAMPLE, st);
    uint32_t over = 0;
    CH_CUDA_TRY(cudaMemcpyAsync(&over, a.work + a.ovf_cnt, sizeof over, cudaMemcpyDeviceToHost, st));
    CH_CUDA_TRY(cudaStreamSynchronize(st));
    h->q_fits_small = over <= MOST;
    return h->q_fits_small;
}

void query_autotune(ch_s *h, uint64_t sample, uint32_t seed, cudaStream_t st, ch_query_config_t *chosen,
                    double *ms_out) {
    if (sample == 0 || h->n == 0) throw Error{CH_EINVAL, "autotune needs a sample and a non-empty graph"};
    DevBuf<uint32_t> buf;
    buf.alloc(3 * sample);
    uint32_t *s = buf.ptr, *t = buf.ptr + sample, *out = buf.ptr + 2 * sample;
    k_sample_pairs<<<grid_for(sample, 256, device_sm_count() * 4), 256, 0, st>>>(s, t, sample, h->n, seed);
    CH_CHECK_LAUNCH();
    const uint32_t keep_l = h->q_layout, keep_t = h->q_threads, keep_s = h->q_small_first,
                   keep_st = h->q_stall, keep_d = h->q_delta;
    cudaEvent_t e0, e1;
    CH_CUDA_TRY(cudaEventCreate(&e0));
    CH_CUDA_TRY(cudaEventCreate(&e1));
    // candidates 0-7: 4 * small_first + 2 * warp layout + (threads == 256);
    // 8-11: warp layout with stalling, 8 + 2 * small_first + (threads == 256);
    // 12-14: warp layout, 256 threads, small tables first, stalling, delta
    // at three multiples of the weight scale
    auto apply = [&](int i) {
        if (i < 8)
            query_set_config(h, (i & 2) ? CH_QUERY_WARP_FLAT : CH_QUERY_BLOCK_FLAT, (i & 1) ? 256 : 128,
                             (i & 4) ? 1 : 0, 0, 0);
        else if (i < 12)
            query_set_config(h, CH_QUERY_WARP_FLAT, (i & 1) ? 256 : 128, (i & 2) ? 1 : 0, 1, 0);
        else
            query_set_config(h, CH_QUERY_WARP_FLAT, 256, 1, 1, delta_of(h, DELTA_TUNE_MULT[i - 12]));
    };
    double best = 0;
    int best_i = -1;
    try {
        for (int i = 0; i < CH_QUERY_AUTOTUNE_CONFIGS; ++i) {
            apply(i);
            query_batch(h, s, t, sample, out, nullptr, st, true);  // warm-up
            CH_CUDA_TRY(cudaEventRecord(e0, st));
            query_batch(h, s, t, sample, out, nullptr, st, true);
            CH_CUDA_TRY(cudaEventRecord(e1, st));
            CH_CUDA_TRY(cudaEventSynchronize(e1));
            float ms = 0;
            CH_CUDA_TRY(cudaEventElapsedTime(&ms, e0, e1));
            if (ms_out) ms_out[i] = ms;
            if (best_i < 0 || ms < best) {
                best = ms;
                best_i = i;
            }
        }
    } catch (...) {
        h->q_layout = keep_l;
        h->q_threads = keep_t;
        h->q_small_first = keep_s;
        h->q_stall = keep_st;
        h->q_delta = keep_d;
        cudaEventDestroy(e0);
        cudaEventDestroy(e1);
        throw;
    }
    cudaEventDestroy(e0);
    cudaEventDestroy(e1);
    apply(best_i);
    if (chosen) {
        chosen->layout = h->q_layout;
        chosen->threads = h->q_threads;
        chosen->small_first = h->q_small_first;
        chosen->stall = h->q_stall;
        chosen->delta = h->q_delta;
    }
    // the sample's work is not the caller's: clear the counters
    CH_CUDA_TRY(cudaMemsetAsync(h->q_stats.ptr, 0, 2 * sizeof(unsigned long long), st));
    CH_CUDA_TRY(cudaStreamSynchronize(st));
}

double query_time_sample(ch_s *h, uint64_t sample, uint32_t seed, cudaStream_t st) {
    if (sample == 0 || h->n == 0) return 0.0;
    DevBuf<uint32_t> buf;
    buf.alloc(3 * sample);
    uint32_t *s = buf.ptr, *t = buf.ptr + sample, *out = buf.ptr + 2 * sample;
    k_sample_pairs<<<grid_for(sample, 256, device_sm_count() * 4), 256, 0, st>>>(s, t, sample, h->n, seed);
    CH_CHECK_LAUNCH();
    cudaEvent_t e0, e1;
    CH_CUDA_TRY(cudaEventCreate(&e0));
    CH_CUDA_TRY(cudaEventCreate(&e1));
    float ms = 0;
    cudaError_t e = cudaSuccess;
    try {
        query_batch(h, s, t, sample, out, nullptr, st);  // warm-up
        CH_CUDA_TRY(cudaEventRecord(e0, st));
        query_batch(h, s, t, sample, out, nullptr, st);
        CH_CUDA_TRY(cudaEventRecord(e1, st));
        CH_CUDA_TRY(cudaEventSynchronize(e1));
        e = cudaEventElapsedTime(&ms, e0, e1);
    } catch (...) {
        cudaEventDestroy(e0);
        cudaEventDestroy(e1);
        throw;
    }
    cudaEventDestroy(e0);
    cudaEventDestroy(e1);
    if (e != cudaSuccess) throw Error{CH_ECUDA, cudaGetErrorString(e)};
    CH_CUDA_TRY(cudaMemsetAsync(h->q_stats.ptr, 0, 2 * sizeof(unsigned long long), st));
    CH_CUDA_TRY(cudaStreamSynchronize(st));
    return ms;
}

void query_work(ch_s *h, cudaStream_t st, uint64_t out[2]) {
    unsigned long long v[2] = {0, 0};
    CH_CUDA_TRY(cudaMemcpyAsync(v, h->q_stats.ptr, sizeof(v), cudaMemcpyDeviceToHost, st));
    CH_CUDA_TRY(cudaMemsetAsync(h->q_stats.ptr, 0, sizeof(v), st));
    CH_CUDA_TRY(cudaStreamSynchronize(st));
    out[0] = v[0];
    out[1] = v[1];
}

}  // namespace gbch

struct ch_query_graph_s {
    cudaGraphExec_t exec = nullptr;
    uint64_t kernels = 0;  // kernel launches one replay makes
};

namespace gbch {

ch_query_graph_s *query_graph_create(ch_s *h, const uint32_t *src, const uint32_t *dst, uint64_t k,
                                     uint32_t *dist_out) {
    query_labels_prepare(h, std::min<uint64_t>(k, Q_CHUNK));  // a capture must not allocate
    cudaStream_t st = nullptr;
    CH_CUDA_TRY(cudaStreamCreateWithFlags(&st, cudaStreamNonBlocking));
    cudaGraph_t graph = nullptr;
    try {
        CH_CUDA_TRY(cudaStreamBeginCapture(st, cudaStreamCaptureModeThreadLocal));
        try {
            query_batch(h, src, dst, k, dist_out, nullptr, st);
        } catch (...) {
            cudaStreamEndCapture(st, &graph);
            if (graph) cudaGraphDestroy(graph);
            cudaGetLastError();
            throw;
        }
        CH_CUDA_TRY(cudaStreamEndCapture(st, &graph));
    } catch (...) {
        cudaStreamDestroy(st);
        throw;
    }
    cudaStreamDestroy(st);
    auto *g = new ch_query_graph_s();
    cudaError_t e = cudaSuccess;
    if (graph) {
        // the launches were counted at capture; count them when replays run them
        size_t nn = 0;
        e = cudaGraphGetNodes(graph, nullptr, &nn);
        std::vector<cudaGraphNode_t> nodes(nn);
        if (e == cudaSuccess && nn) e = cudaGraphGetNodes(graph, nodes.data(), &nn);
        for (size_t i = 0; e == cudaSuccess && i < nn; ++i) {
            cudaGraphNodeType ty;
            e = cudaGraphNodeGetType(nodes[i], &ty);
            if (e == cudaSuccess && ty == cudaGraphNodeTypeKernel) ++g->kernels;
        }
        kernel_launch_add(-(int64_t)g->kernels);
        if (e == cudaSuccess) e = cudaGraphInstantiate(&g->exec, graph, 0);
    }
    if (graph) cudaGraphDestroy(graph);
    if (e != cudaSuccess) {
        delete g;
        cudaGetLastError();
        throw Error{CH_ECUDA, std::string("graph instantiation: ") + cudaGetErrorString(e)};
    }
    return g;
}

void query_graph_launch(ch_query_graph_s *g, cudaStream_t st) {
    if (!g->exec) return;  // k = 0: nothing was captured
    CH_CUDA_TRY(cudaGraphLaunch(g->exec, st));
    kernel_launch_add((int64_t)g->kernels);
}

void query_graph_free(ch_query_graph_s *g) {
    if (g->exec) cudaGraphExecDestroy(g->exec);
    delete g;
}

// ---------------------------------------------------------------------------
// Query batches that allocate nothing (ch_query_batch_static)
// ---------------------------------------------------------------------------
//
// Same kernels as query_batch; the only difference is where the per-call
// scratch lives (the work counters and the list of queries handed to the
// dense kernel). Here it is one file-scope device array, so a call needs no
// allocation at all; every GPU that loads the library holds the array
// (about 1 MiB) until the process exits. The array is shared by all calls
// and all handles on a device: calls whose work overlaps on the GPU race on
// it and must be serialised by the caller (one stream, or events).

namespace {

constexpr uint32_t kStaticScratchHead = 4;  // [0] block counter, [1] dense counter, [2] overflow count
__device__ __align__(256) uint32_t g_static_query_scratch[kStaticScratchHead + CH_STATIC_QUERY_MAX];

std::mutex g_static_mu;
uint32_t *g_static_ptr[64] = {nullptr};

// Device address of the scratch array for the current device. The first call
// on a device resolves it (cudaGetSymbolAddress) with that device current;
// later calls reuse it.
uint32_t *static_scratch() {
    int dev = 0;
    CH_CUDA_TRY(cudaGetDevice(&dev));
    if (dev < 0 || dev >= 64) throw Error{CH_ERANGE, "device ordinal above 63"};
    std::lock_guard<std::mutex> lock(g_static_mu);
    if (!g_static_ptr[dev]) {
        void *p = nullptr;
        CH_CUDA_TRY(cudaGetSymbolAddress(&p, g_static_query_scratch));
        g_static_ptr[dev] = static_cast<uint32_t *>(p);
    }
    return g_static_ptr[dev];
}

}  // namespace

void query_batch_static(ch_s *h, const uint32_t *src, const uint32_t *dst, uint64_t k,
                        uint32_t *dist_out, cudaStream_t st) {
    if (k > CH_STATIC_QUERY_MAX)
        throw Error{CH_ERANGE, "batch larger than CH_STATIC_QUERY_MAX queries"};
    if (k == 0) return;
    int dev = 0;
    CH_CUDA_TRY(cudaGetDevice(&dev));
    if (dev != h->device)
        throw Error{CH_EINVAL, "the current device is not the hierarchy's device"};
    uint32_t *scratch = static_scratch();
    QArgs a = hierarchy_args(h);
    a.src = src;
    a.dst = dst;
    a.out = dist_out;
    a.settled = nullptr;
    a.k = k;
    a.work = scratch;
    a.in_list = nullptr;
    a.in_cnt = 0;
    a.ctr = 0;
    a.ovf = scratch + kStaticScratchHead;
    a.ovf_cnt = 2;
    if (small_batch(a, k)) return launch_query_small(h, a, st);
    // the counters keep the previous call's values: clear them
    CH_CUDA_TRY(cudaMemsetAsync(scratch, 0, kStaticScratchHead * sizeof(uint32_t), st));
    // one block-kernel pass (large tables): the scratch holds one list
    if (!a.dense_first) launch_query_block(h, a, true, false, k, st);
    launch_query_dense(h, a, true, k, st);
}

}  // namespace gbch

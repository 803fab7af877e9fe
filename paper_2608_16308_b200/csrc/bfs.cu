// DB-BFS (Section 4.2, Algorithm 5): level-synchronous BFS where every level is one Boolean
// SpMSpV.  The frontier lives directly in the vector-block masks, visited vertices are stripped
// with a second set of masks, and push or pull is chosen per level from the ratio of nonempty
// frontier blocks (Section 3.3.1) without rebuilding anything.  The whole traversal is ONE
// cooperative launch: levels are separated by grid-wide barriers (co-residency is guaranteed
// by the cooperative launch), so there is no host round trip per level.
#include <cooperative_groups.h>
#include <cstddef>

#include "internal.cuh"
#include "microkernels.cuh"
#include "push_direct.cuh"
#include "worklist.cuh"

namespace cg = cooperative_groups;

namespace dbs {

constexpr int BFS_CTA = BFS_LIST;   // one thread block per SM (a grid barrier over 148 blocks costs far less than over a thousand), a thread per listed vertex

// Rows of one hypersparse block reached from the active columns (one lane per block).
template <int DT>
__device__ __forceinline__ uint32_t lane_block_bool(int type, uint32_t w, uint32_t aux, uint32_t xm,
                                                    const uint8_t *payload) {
    uint32_t hit = 0;
    if (type == DBSPMSPV_BLK_INLINE) {
        hit = ((xm >> (aux & 15)) & 1u) << (aux >> 4);
    } else {
        const uint8_t *blk = payload + (size_t)w * 4;
        for (uint32_t k = 0; k <= aux; ++k) {
            const uint32_t rc = blk[k];
            if ((xm >> (rc & 15)) & 1u) hit |= 1u << (rc >> 4);
        }
    }
    return hit;
}

__device__ __forceinline__ void write_levels(int32_t *levels, int rb, uint32_t fresh, int depth) {
    while (fresh) {
        const int r = __ffs(fresh) - 1;
        fresh &= fresh - 1;
        levels[rb * 16 + r] = depth;
    }
}

// The threads that share a level's work (the whole cooperative grid).
struct Scope {
    int tid, nthreads;      // thread index / count in the scope
    int gwarp, nwarps;      // warp index / count in the scope
};

// Where a level puts what it finds: the next level's frontier.
struct NextLevel {
    uint32_t *N;                 // masks
    int32_t *words, *verts;      // lists of the words that became nonzero and of the first BFS_LIST vertices
    Counters::BfsSet *set;
    bool counts;                 // the elements of the frontier's columns are counted (see BFS_LARGE_WORDS)
};
// Appends what the lanes of a warp found: `mine` vertices each, which put(k, place) writes for k < mine, and (new_word) a mask word that became nonzero.  One atomic for both lists.
template <typename Put>
__device__ __forceinline__ void append_found(const NextLevel &nx, int word, bool new_word, int mine, int lane, Put put) {
    const uint32_t m = __ballot_sync(FULL, new_word);
    int incl = mine;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) { const int t = __shfl_up_sync(FULL, incl, o); if (lane >= o) incl += t; }
    unsigned long long base = 0;
    if (lane == 31) base = atomicAdd(reinterpret_cast<unsigned long long *>(&nx.set->n_verts), (unsigned long long)__popc(m) << 32 | (unsigned)incl);
    base = __shfl_sync(FULL, base, 31);
    if (new_word) nx.words[(int)(base >> 32) + __popc(m & ((1u << lane) - 1u))] = word;
    const int at = (int)(uint32_t)base + incl - mine;
    for (int k = 0; k < mine && at + k < BFS_LIST; ++k) put(k, at + k);
}
// ... the set bits of a word each
__device__ __forceinline__ void append_words(const NextLevel &nx, int word, uint32_t mask, bool new_word, int lane) {
    uint32_t left = mask;
    append_found(nx, word, new_word, __popc(mask), lane, [&](int, int place) { nx.verts[place] = word * 32 + __ffs(left) - 1; left &= left - 1; });
}
// What the lanes of a warp counted: vector blocks that became nonempty, and elements -- of vertices in other warps' blocks too -- in one atomic.
__device__ __forceinline__ void add_counts(const NextLevel &nx, int blocks, int edges, int lane) {
    static_assert(offsetof(Counters::BfsSet, edges) == offsetof(Counters::BfsSet, n_blocks) + 4 && offsetof(Counters::BfsSet, n_blocks) % 8 == 0, "one 8-byte word");
    blocks = __reduce_add_sync(FULL, blocks);
    if (nx.counts) edges = __reduce_add_sync(FULL, edges);
    if (lane == 0 && (blocks | edges)) atomicAdd(reinterpret_cast<unsigned long long *>(&nx.set->n_blocks), (unsigned long long)(unsigned)edges << 32 | (unsigned)blocks);
}
// Up to this many warp steps the bookkeeping is the claiming lanes': a second atomic per vertex found, but neither a pass nor a barrier
// behind the level.  Larger levels leave it to a pass over the words that became nonzero, one update for up to 32 vertices: levels of 2^22
// vertices that reach most of them through a few thousand hubs took 78 - 150 us with an atomic each, 59 - 116 with the pass, and 37 - 71 since the pass writes
// the levels too and nobody waits for an atomic's reply.  (Limit 512:
// levels of a few thousand steps 2 - 5 us longer; 4096 to 65536: no difference on graphs of 17,000 to 2^22 vertices.)
constexpr int BFS_MARK_STEPS = 16384;

// Words that a warp takes at a time so that one pass of all warps covers the n_words: 32, or -- on a graph with fewer mask words than that keeps every
// warp busy -- the smallest power of two that does.  (With 32 words each a graph of 2^18 vertices gave work to 256 of 4736 warps.)
__device__ __forceinline__ int words_per_warp(int n_words, int nwarps) {
    int W = 32;
    while (W > 1 && (int64_t)nwarps * (W / 2) >= n_words) W >>= 1;
    return W;
}
// Graphs of that many words per warp or more (on 148 SMs: above 606,208 vertices) count the elements of a pushed frontier and look at the first element of
// every wanted row before its run.  Below, where the index stays in L2 and worklists are short, both are only links of a chain of loads: six sources each, with / without them,
// 65 K vertices 55.3 / 53.0 us, in scattered order 57.6 / 55.1; 262 K 67.6 / 65.2 and 66.8 / 64.5; 500 K 81.5 / 77.9 and 75.6 / 75.1.  Above, with / without: the count 700 K 84.4 / 83.9
// and 68.5 / 67.6, 2^20 92.1 / 92.1 and 86.8 / 87.8, 2^22 148.9 / 153.4 and 128.6 / 127.0 (single sources lose 10 us without it); the look 700 K 84.4 / 85.2 and
// 68.5 / 72.4, 2^22 148.9 / 167.0 and 128.6 / 151.7.  (The degrees asked for beside the atomic in place of behind it: no gain.  The look under wide frontiers only: none in small graphs, 2^22 162.)
constexpr int BFS_LARGE_WORDS = 8;

// Boolean push: tasks of the active frontier blocks (a task is at most PUSH_CHUNK = 32 view
// entries: one warp step); newly reached rows are claimed with one atomicOr per entry on the
// next-frontier masks.  Like the pull, the loop is software-
// pipelined: while task k is evaluated, the visited masks of k+1, the view entries of k+2 and
// the task record of k+3 (in this warp's stride) are in flight.
// With MARK the winner does the level's bookkeeping for the vertex: it writes its level, marks it visited, lists it and the word it turned nonzero.
// Without it nobody looks at a reply: all that is the pass behind the level.
template <int DT, bool MARK>
__device__ void bfs_push(const Device &d, const Scope &sc, const uint32_t *F, const uint2 *tasks, int n_recs, const int4 *hubs, int n_hubs,
                         int32_t *levels, int depth, const NextLevel &nx) {
    static_assert(PUSH_CHUNK == 32, "one warp step per task");
    const int lane = threadIdx.x & 31;
    const int gwarp = sc.gwarp, nwarps = sc.nwarps;
    const HubTable table = load_hub_table(hubs, n_hubs, lane);
    const int n_tasks = n_recs + table.total;                    // task records, then the steps of the hub runs
    auto item = [&](int i) { return worklist_item(tasks, n_recs, table, i); };
    const uint2 none = make_uint2(0u, 0u);
    int blocks = 0, edges = 0;
    // claims the rows `hit` of row block `brow` (called by a full warp; hit = 0: nothing in this lane)
    auto publish = [&](int brow, uint32_t hit) {
        if (!MARK) {                                   // (nobody waits for a reply: levels, list and counts are the pass behind the level)
            if (hit) atomicOr(&nx.N[brow >> 1], hit << ((brow & 1) * 16));
            return;
        }
        uint32_t old = 0, fresh = 0;
        const int sh = (brow & 1) * 16;
        if (hit) {
            old = atomicOr(&nx.N[brow >> 1], hit << sh);
            fresh = hit & ~(old >> sh);
        }
        if (!__any_sync(FULL, fresh != 0u)) return;
        const bool newly = fresh && ((old >> sh) & 0xFFFFu) == 0;
        if (fresh) {
            write_levels(levels, brow, fresh, depth);
            atomicOr(&d.ws.visited32[brow >> 1], fresh << sh);
            blocks += newly;
            if (nx.counts) for (uint32_t f = fresh; f; f &= f - 1) edges += (int)degree_of_code(d.col_degree[brow * 16 + __ffs(f) - 1]);
        }
        append_words(nx, brow >> 1, fresh << sh, fresh && !old, lane);
    };
    struct Entries { uint32_t idx, aux, xm; int n, start; };   // n: entries of the task (0 = no task)
    auto entries_of = [&](int t, const uint2 &task) {
        Entries e{0u, 0u, 0u, 0, 0};
        if (t < n_tasks) {
            const int jb = (int)(task.x & IDX_MASK), start = (int)task.y;
            e.n = (int)(task.x >> 27) + 1;
            e.start = start;
            if (lane < e.n && DBS_CHK_RANGE(d, start, e.n) && DBS_CHK_INDEX(d, jb, d.nb)) {
                e.idx = d.csc.idx[start + lane]; e.aux = d.csc.aux[start + lane];
#ifdef DBS_BOUNDS_CHECK
                uint32_t w_ = d.csc.w[start + lane];
                DBS_CHK_ENTRY(d, false, e.idx, w_, e.aux);
#endif
            }
            e.xm = mask_of(F, jb);
        }
        return e;
    };
    auto need_of = [&](const Entries &e) { return lane < e.n ? ~mask_of(d.ws.visited32, e.idx & IDX_MASK) & 0xFFFFu : 0u; };
    uint2 t1 = gwarp + nwarps < n_tasks ? item(gwarp + nwarps) : none;
    uint2 t2 = gwarp + 2 * nwarps < n_tasks ? item(gwarp + 2 * nwarps) : none;
    uint2 t0 = gwarp < n_tasks ? item(gwarp) : none;
    Entries e0 = entries_of(gwarp, t0);
    Entries e1 = entries_of(gwarp + nwarps, t1);
    uint32_t need0 = need_of(e0);
    for (int t = gwarp; t < n_tasks; t += nwarps) {
        const uint2 t3 = t + 3 * nwarps < n_tasks ? item(t + 3 * nwarps) : none;          // stage 1
        const Entries e2 = entries_of(t + 2 * nwarps, t2);                                // stage 2
        const uint32_t need1 = need_of(e1);                                               // stage 3
        // stage 4: evaluate task t
        {
            const uint32_t idx = e0.idx, aux = e0.aux, xm = e0.xm;
            const int type = idx >> TYPE_SHIFT, brow = idx & IDX_MASK;
            bool heavy = false;
            uint32_t w = 0;
            uint32_t hit = 0;
            if (need0) {
                if (type == DBSPMSPV_BLK_INLINE) {
                    hit = ((xm >> (aux & 15)) & 1u) << (aux >> 4);
                } else {
                    w = d.csc.w[e0.start + lane];
                    if (type == DBSPMSPV_BLK_COO) {
                        if (aux < COO_SERIAL_MAX) hit = lane_block_bool<DT>(type, w, aux, xm, d.payload);
                        else heavy = true;
                    } else {
                        hit = lane_heavy_bool(type, d.payload + (size_t)w * 4, xm);
                    }
                }
                hit &= need0;
            }
            publish(brow, hit);
            uint32_t hv = __ballot_sync(FULL, heavy);
            while (hv) {
                const int src = __ffs(hv) - 1;
                hv &= hv - 1;
                const uint32_t bidx = __shfl_sync(FULL, idx, src);
                const uint32_t bw = __shfl_sync(FULL, w, src);
                const int nnz = (int)__shfl_sync(FULL, aux, src) + 1;
                const int btype = bidx >> TYPE_SHIFT, bbrow = bidx & IDX_MASK;
                uint32_t hits = warp_block_bool<DT>(btype, d.payload + (size_t)bw * 4, nnz, xm, lane);
                hits &= ~mask_of(d.ws.visited32, bbrow);
                publish(bbrow, lane == 0 ? hits : 0u);
            }
        }
        // rotate the pipeline
        e0 = e1; e1 = e2; need0 = need1; t2 = t3;
    }
    if (MARK) add_counts(nx, blocks, edges, lane);
}

// A short listed frontier, pushed without a worklist: every thread block lays the vertices' runs of INLINE elements and of the payload entries of their column blocks end to end in chunks, the
// warps of the grid share them out, and the claiming lanes do the bookkeeping.  Such a level moves next to nothing; it is the chain list -> column pointers -> entries -> visited -> claim -> list, one
// barrier behind it (a worklist is one more phase and barrier in front).  Every frontier of at most BFS_LIST vertices has its list, whichever way its level went.  Searches, symmetrised R-MAT, eight
// sources each, with worklists / so, in brackets in scattered order: 16 K vertices 45.6 / 40.2 us (42.2 / 39.4), 65 K 54.7 / 48.2 (50.3 / 43.0), 262 K 53.4 / 42.8 (57.7 / 46.6), 2^20 75.3 / 61.6
// (75.7 / 67.2), 2^22 138.8 / 130.2 (112.6 / 110.2); part of it are the counters of a level, one 16-byte load behind its last barrier in place of four to seven loads one after the other.
// (Only the scan is kept: a chunk's warp fetches its vertex and the places of its runs once more, from L1.  With those in shared memory too, 25 KB in place of 4, the pull levels of large graphs, whose
// gathers of frontier masks live in the L1 that this takes away, were longer: searches on 2 M uniform rows of eight 233 us, 225 so.)
struct BfsListShared {
    int pre[BFS_LIST + 1];                            // chunks before a vertex
    int sum[BFS_CTA / 32], elems[BFS_CTA / 32];
};
// Lays the chunks out; returns their number, and the elements behind them (the same in every thread).
__device__ int bfs_list_layout(const Device &d, const int32_t *verts, int cnt, BfsListShared &sh, int &n_elems) {
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    int first, deg = 0, pdeg = 0;
    if (tid < cnt) {
        int j = verts[tid];
        if (!DBS_CHK_INDEX(d, j, d.n)) j = 0;
        column_run(d, j, first, deg);
        payload_run(d, j >> 4, first, pdeg);
    }
    const int mine = (deg + PD_CHUNK - 1) / PD_CHUNK + (pdeg + PD_PAYLOAD - 1) / PD_PAYLOAD;
    int incl = mine;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) { const int t = __shfl_up_sync(FULL, incl, o); if (lane >= o) incl += t; }
    const int elems = __reduce_add_sync(FULL, deg + pdeg);
    if (lane == 31) { sh.sum[warp] = incl; sh.elems[warp] = elems; }
    __syncthreads();
    const int v = sh.sum[lane], total = __reduce_add_sync(FULL, v);
    n_elems = __reduce_add_sync(FULL, sh.elems[lane]);
    sh.pre[tid] = incl - mine + __reduce_add_sync(FULL, lane < warp ? v : 0);
    if (tid == 0) sh.pre[BFS_LIST] = total;
    __syncthreads();
    return total;
}
template <int DT>
__device__ void bfs_push_list(const Device &d, const int32_t *verts, int total, const BfsListShared &sh, int32_t *levels, int depth, const NextLevel &nx) {
    constexpr int U = PD_CHUNK / 32;
    static_assert(PD_PAYLOAD / 2 == U, "one element per lane and step either way");
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    int blocks = 0, edges = 0;
    // (neighbouring chunks on different SMs)
    for (int c = warp * (int)gridDim.x + (int)blockIdx.x; c < total; c += (int)gridDim.x * (BFS_CTA / 32)) {
        int o = 0;                                     // the last vertex with at most c chunks before it
#pragma unroll
        for (int st = BFS_LIST / 2; st; st >>= 1) if (sh.pre[o + st] <= c) o += st;
        int j = verts[o], first, deg, pfirst, pdeg;
        if (!DBS_CHK_INDEX(d, j, d.n)) j = 0;
        column_run(d, j, first, deg);
        payload_run(d, j >> 4, pfirst, pdeg);
        const int k = c - sh.pre[o], n_inline = (deg + PD_CHUNK - 1) / PD_CHUNK;
        int target[U];
        if (k < n_inline) {                            // warp-uniform
            const int at = k * PD_CHUNK + lane;
            uint32_t idx[U], w[U], aux[U];
#pragma unroll
            for (int u = 0; u < U; ++u) {
                idx[u] = PAD_IDX; w[u] = 0u; aux[u] = 0u;
                if (at + u * 32 < deg) push_entry<false>(d, first + at + u * 32, idx[u], w[u], aux[u]);
            }
#pragma unroll
            for (int u = 0; u < U; ++u) target[u] = idx[u] < (1u << TYPE_SHIFT) ? (int)((idx[u] & IDX_MASK) * 16u + (aux[u] >> 4)) : -1;
        } else {
            const int at = (k - n_inline) * PD_PAYLOAD;
            bool in[U];
            float value[U];
            uint32_t rb[U];
            payload_elements<DBSPMSPV_PATTERN, U>(d, pfirst + at, min(PD_PAYLOAD, pdeg - at), j & 15, lane, in, value, rb);
#pragma unroll
            for (int u = 0; u < U; ++u) target[u] = in[u] ? (int)(rb[u] * 16u) + (lane & 15) : -1;
        }
        uint32_t seen[U], old[U], fresh = 0u, opened = 0u;
#pragma unroll
        for (int u = 0; u < U; ++u) seen[u] = target[u] >= 0 ? __ldcg(d.ws.visited32 + (target[u] >> 5)) : 0xFFFFFFFFu;
#pragma unroll
        for (int u = 0; u < U; ++u) {
            old[u] = 0xFFFFFFFFu;
            if (!((seen[u] >> (target[u] & 31)) & 1u)) old[u] = atomicOr(nx.N + (target[u] >> 5), 1u << (target[u] & 31));
        }
#pragma unroll
        for (int u = 0; u < U; ++u)
            if (!((old[u] >> (target[u] & 31)) & 1u)) {
                fresh |= 1u << u;
                levels[target[u]] = depth;
                atomicOr(d.ws.visited32 + (target[u] >> 5), 1u << (target[u] & 31));
                blocks += ((old[u] >> (target[u] & 16)) & 0xFFFFu) == 0u;
                if (!old[u]) opened |= 1u << u;
            }
        if (!__any_sync(FULL, fresh != 0u)) continue;
        // both lists with one scan and one atomic (vertices in the low half of each)
        const int mine = __popc(fresh) | __popc(opened) << 16;
        int incl = mine;
#pragma unroll
        for (int st = 1; st < 32; st <<= 1) { const int t = __shfl_up_sync(FULL, incl, st); if (lane >= st) incl += t; }
        unsigned long long base = 0;
        if (lane == 31) base = atomicAdd(reinterpret_cast<unsigned long long *>(&nx.set->n_verts), (unsigned long long)(unsigned)(incl >> 16) << 32 | (unsigned)(incl & 0xFFFF));
        if (nx.counts)
#pragma unroll
            for (int u = 0; u < U; ++u) if ((fresh >> u) & 1u) edges += (int)degree_of_code(d.col_degree[target[u]]);
        base = __shfl_sync(FULL, base, 31);
        int v = (int)(uint32_t)base + ((incl - mine) & 0xFFFF), w = (int)(base >> 32) + ((incl - mine) >> 16);
#pragma unroll
        for (int u = 0; u < U; ++u) {
            if ((fresh >> u) & 1u) { if (v < BFS_LIST) nx.verts[v] = target[u]; ++v; }
            if ((opened >> u) & 1u) nx.words[w++] = target[u] >> 5;
        }
    }
    add_counts(nx, blocks, edges, lane);
}

// Boolean pull: one warp per row-block segment (a segment has at most MAX_SEG_ENTRIES = 4 x 32
// view entries, so one round of four warp steps covers it); row blocks with nothing left to
// discover are skipped.  A segment costs a chain of dependent loads (descriptor -> visited mask
// -> view entries -> frontier masks); the loop is software-pipelined four deep so that only the
// last link is waited for: while segment k is evaluated, the entries of k+1, the visited mask
// of k+2 and the descriptor of k+3 (k counted in this warp's stride) are already in flight.
template <int DT>
__device__ void bfs_pull(const Device &d, const Scope &sc, const uint32_t *F, uint32_t *N, int32_t *levels, int depth) {
    constexpr int U = MAX_SEG_ENTRIES / 32;
    const int lane = threadIdx.x & 31;
    const int gwarp = sc.gwarp, nwarps = sc.nwarps;
    const int nseg = d.n_segments;
    const Segment none = Segment{0, 0, 0, 0};
    auto need_of = [&](const Segment &sg) { return (sg.count & 0x7FFFFFFF) ? ~mask_of(d.ws.visited32, sg.row_block) & 0xFFFFu : 0u; };
    // prologue: fill the pipeline
    Segment s0 = gwarp < nseg ? d.segments[gwarp] : none;
    Segment s1 = gwarp + nwarps < nseg ? d.segments[gwarp + nwarps] : none;
    Segment s2 = gwarp + 2 * nwarps < nseg ? d.segments[gwarp + 2 * nwarps] : none;
    uint32_t need0 = need_of(s0), need1 = need_of(s1);
    // the entries of a segment: lane l takes positions l, l + 32, ... (constant offsets from one
    // pointer per array, one comparison per step)
    auto fetch = [&](const Segment &sg, uint32_t need, uint32_t (&idx)[U], uint32_t (&aux)[U]) {
        const uint32_t *ip = d.csr.idx + sg.start + lane;
        const uint8_t *ap = d.csr.aux + sg.start + lane;
        const int rem = need && DBS_CHK_RANGE(d, sg.start, sg.count & 0x7FFFFFFF) ? (sg.count & 0x7FFFFFFF) - lane : 0;
#pragma unroll
        for (int u = 0; u < U; ++u) {
            idx[u] = 0; aux[u] = 0;
            if (rem > u * 32) { idx[u] = ip[u * 32]; aux[u] = ap[u * 32]; }
        }
    };
    uint32_t idx0[U], aux0[U];
    fetch(s0, need0, idx0, aux0);
    for (int sg = gwarp; sg < nseg; sg += nwarps) {
        // stage 1: descriptor three strides ahead
        const Segment s3 = sg + 3 * nwarps < nseg ? d.segments[sg + 3 * nwarps] : none;
        // stage 2: visited mask two strides ahead
        const uint32_t need2 = need_of(s2);
        // stage 3: view entries one stride ahead
        uint32_t idx1[U], aux1[U];
        fetch(s1, need1, idx1, aux1);
        // stage 4: evaluate this segment
        if (need0) {
            const int cnt0 = s0.count & 0x7FFFFFFF;
            const int rb = s0.row_block;
            // frontier masks: only for entries that can still contribute -- past-the-end entries
            // are all-zero (INLINE, row 0); an INLINE entry whose row is not wanted is skipped
            // (late pull levels want one or two rows of a row block: most gathers fall away)
            const int rem0 = cnt0 - lane;
            uint32_t xm[U];
            bool heavy_any = false;
#pragma unroll
            for (int u = 0; u < U; ++u) {
                const bool inl = (idx0[u] >> TYPE_SHIFT) == DBSPMSPV_BLK_INLINE;
                const bool want = rem0 > u * 32 && (!inl || ((need0 >> (aux0[u] >> 4)) & 1u));
                xm[u] = want ? mask_of(F, idx0[u] & IDX_MASK) : 0u;
                heavy_any |= want && !inl;
            }
            uint32_t hit = 0;
#pragma unroll
            for (int u = 0; u < U; ++u)        // INLINE entries: branch-free (xm is 0 where not wanted)
                hit |= ((idx0[u] >> TYPE_SHIFT) == DBSPMSPV_BLK_INLINE ? (xm[u] >> (aux0[u] & 15)) & 1u : 0u) << (aux0[u] >> 4);
            if (__any_sync(FULL, heavy_any)) {   // rare: packed-COO and mask-based blocks
#pragma unroll
                for (int u = 0; u < U; ++u) {
                    if (u * 32 >= cnt0) break;      // warp-uniform
                    const int type = idx0[u] >> TYPE_SHIFT;
                    bool heavy = false;
                    uint32_t w = 0;
                    if (xm[u] && type != DBSPMSPV_BLK_INLINE) {
                        w = d.csr.w[s0.start + u * 32 + lane];
                        if (type == DBSPMSPV_BLK_COO) {
                            if (aux0[u] < COO_SERIAL_MAX) hit |= lane_block_bool<DT>(type, w, aux0[u], xm[u], d.payload);
                            else heavy = true;
                        } else {
                            hit |= lane_heavy_bool(type, d.payload + (size_t)w * 4, xm[u]);
                        }
                    }
                    uint32_t hv = __ballot_sync(FULL, heavy);
                    while (hv) {
                        const int src = __ffs(hv) - 1;
                        hv &= hv - 1;
                        const uint32_t bidx = __shfl_sync(FULL, idx0[u], src);
                        const uint32_t bw = __shfl_sync(FULL, w, src);
                        const int nnz = (int)__shfl_sync(FULL, aux0[u], src) + 1;
                        const uint32_t bxm = __shfl_sync(FULL, xm[u], src);
                        hit |= warp_block_bool<DT>(bidx >> TYPE_SHIFT, d.payload + (size_t)bw * 4, nnz, bxm, lane);
                    }
                }
            }
            hit = __reduce_or_sync(FULL, hit) & need0;
            if (hit) {
                if (s0.count < 0) {          // the segment is its whole row block: plain stores
                    if (lane == 0) reinterpret_cast<uint16_t *>(N)[rb] = (uint16_t)hit;
                    if (lane < 16 && ((hit >> lane) & 1u)) levels[rb * 16 + lane] = depth;
                } else if (lane == 0) {
                    const int sh = (rb & 1) * 16;
                    const uint32_t old = atomicOr(&N[rb >> 1], hit << sh);
                    write_levels(levels, rb, hit & ~(old >> sh), depth);
                }
            }
        }
        // rotate the pipeline
        s0 = s1; s1 = s2; s2 = s3;
        need0 = need1; need1 = need2;
#pragma unroll
        for (int u = 0; u < U; ++u) { idx0[u] = idx1[u]; aux0[u] = aux1[u]; }
    }
}

// Boolean pull over the row-run index (square matrices, unless the index was switched off).
// What bounds it is DRAM: a sector per row that is not settled by its first element (R-MAT scale 22, a frontier of 160 K vector blocks: 38 us without the
// look at the first elements, 26 with it; in scattered order, where the runs used to begin anywhere, 40 -> 22), and the whole runs of rows with no frontier neighbour.
// Entries with a payload are evaluated first, from the per-row-block position list, and a row
// block is left as soon as each of its wanted rows has a parent; then every row that is still
// wanted walks its own INLINE run and stops at its first frontier neighbour -- the early exit of
// Algorithm 5 per row instead of per row block: in the big levels a row finds a parent within a
// few entries, so a fraction of the edges is read at all.
// A warp takes a block of W = 32 consecutive mask words (1024 rows; fewer on small graphs) and lane l walks one row of
// every word (row (l + k) mod 32 of the block's word k), one row after the other, each lane at its own pace.  (With lane = row inside ONE word a
// word costs as many dependent rounds as its slowest row -- and at the levels with a small
// frontier almost every word holds a row without a frontier neighbour, which is walked to its
// end -- so a warp's time would be the sum over its words of the maximum; here it is the maximum
// over the lanes of the sum, about a third of the rounds.)  Four entries are fetched per round
// and lane (eight when the frontier is small), then their frontier masks; the run of the lane's
// next row is fetched meanwhile.  A row that has not finished after eight rounds is long (a hub
// with no frontier neighbour so far) and is finished by the whole warp, 32 * 8 entries per step.
// Found rows are collected as one bit per (lane, word) and transposed back with ballots, so the
// warp owns its mask words: plain stores, no atomics.
// a pull level over a frontier that fills fewer than this share of the vector blocks reads two groups of four entries per round
#ifndef DBS_BFS_WIDE_PULL
#define DBS_BFS_WIDE_PULL 0.3f
#endif
constexpr float BFS_WIDE_PULL = DBS_BFS_WIDE_PULL;

template <int DT>
__device__ void bfs_pull_rows(const Device &d, const uint32_t *F, uint32_t *Z, const NextLevel &nx, int32_t *levels, int depth, bool wide, uint32_t *s_need) {
    uint32_t *const N = nx.N;
    const int lane = threadIdx.x & 31;
    // (neighbouring words on different SMs: on an R-MAT graph that was not relabelled they are heavy together)
    const int gwarp = (threadIdx.x >> 5) * gridDim.x + blockIdx.x;
    const int nwarps = (gridDim.x * blockDim.x) >> 5;
    const int n_words = (d.mb + 1) / 2;
    constexpr uint32_t NONE = 0xFFFFFFFFu;          // no entry: local column 31 never matches a 16-bit mask
    constexpr int LONG_UNROLL = 8, MAX_ROUNDS = 8;
    const int per_round = wide ? 8 : 4;
    int n_nz = 0;
    const int W = words_per_warp(n_words, nwarps);  // (a lane walks W rows)
    for (int w0 = gwarp * W; w0 < n_words; w0 += nwarps * W) {
        const int wd = w0 + lane;                    // this lane's word (bookkeeping); rows: lane = row of every word
        const bool in = lane < W && wd < n_words;
        const uint32_t need = in ? ~d.ws.visited32[wd] : 0u;   // (rows without stored elements and rows past m count as visited)
        if (in) Z[wd] = 0u;
        if (!__any_sync(FULL, need != 0u)) { if (in) N[wd] = 0u; continue; }
        uint32_t found = 0u;
        // entries with a payload: the words that have any (their two row blocks' ranges), one word at a time
        {
            int pb0 = 0, pe0 = 0, pb1 = 0, pe1 = 0;
            if (need) {
                const int rb = 2 * wd;
                if (rb < d.mb) { pb0 = d.csr.ptr[rb]; pe0 = d.csr_inl[rb]; }
                if (rb + 1 < d.mb) { pb1 = d.csr.ptr[rb + 1]; pe1 = d.csr_inl[rb + 1]; }
            }
            uint32_t todo = __ballot_sync(FULL, need && (pe0 > pb0 || pe1 > pb1));
            while (todo) {
                const int k = __ffs(todo) - 1;
                todo &= todo - 1;
                // (Up to 16 entries a row block: a half-warp for each of the two, one chain of loads per word; more: the whole warp for one after the other.  Searches on 27-point operators, 100^3 / 150^3 cells,
                // the row blocks one after the other 1535 / 7130 us, so 1420 / 6530; half-warps whatever the length: 1 % less there, R-MAT of 700 K vertices, whose hub row blocks have hundreds, 81 -> 87.)
                const uint32_t need_k = __shfl_sync(FULL, need, k);
                const int beg0 = __shfl_sync(FULL, pb0, k), end0 = __shfl_sync(FULL, pe0, k), beg1 = __shfl_sync(FULL, pb1, k), end1 = __shfl_sync(FULL, pe1, k);
                uint32_t fk = 0u;
                const int step = max(end0 - beg0, end1 - beg1) <= 16 ? 16 : 32;
#pragma unroll 1
                for (int part = step & 16 ? lane & 16 : 0; ; part += 16) {
                    const uint32_t need_part = need_k & (0xFFFFu << part);
                    const int pend = part ? end1 : end0;
                    for (int pos = (part ? beg1 : beg0) + (lane & (step - 1)); __any_sync(FULL, pos < pend && (need_part & ~fk)); pos += step) {      // (until every wanted row has a parent)
                        uint32_t hit = 0;
                        if (pos < pend && (need_part & ~fk)) {
                            uint32_t idx = d.csr.idx[pos], aux = d.csr.aux[pos];
#ifdef DBS_BOUNDS_CHECK
                            { uint32_t w_ = d.csr.w[pos]; DBS_CHK_ENTRY(d, true, idx, w_, aux); }
#endif
                            const uint32_t xm = mask_of(F, idx & IDX_MASK);
                            if (xm) {
                                const int type = idx >> TYPE_SHIFT;
                                const uint32_t w = d.csr.w[pos];
                                hit = type == DBSPMSPV_BLK_COO ? lane_block_bool<DT>(type, w, aux, xm, d.payload)
                                                               : lane_heavy_bool(type, d.payload + (size_t)w * 4, xm);
                            }
                        }
                        fk |= __reduce_or_sync(FULL, hit << part) & need_k;
                    }
                    if (step == 16 || part) break;
                }
                if ((fk >> lane) & 1u) levels[(size_t)(w0 + k) * 32 + lane] = depth;
                if (lane == k) found |= fk;
            }
        }
        // The first column of every wanted row's run, the one with the highest degree, from an array of their own: lane = row, eight words at a time.
        // Under a frontier that holds the hubs most rows end here, with neither their run's place nor its first sector fetched.
        if (W >= BFS_LARGE_WORDS) {
            constexpr int U = 8;
            const uint32_t wanted = need & ~found;
            uint32_t todo = __ballot_sync(FULL, wanted != 0u);
            while (todo) {
                int k[U];
                uint32_t v[U], xm[U];
#pragma unroll
                for (int u = 0; u < U; ++u) {
                    k[u] = __ffs(todo) - 1;                   // (-1: no more words)
                    todo &= todo - 1;
                    const uint32_t word = __shfl_sync(FULL, wanted, k[u] & 31);
                    v[u] = k[u] >= 0 && ((word >> lane) & 1u) ? __ldcs(d.row_first + (size_t)(w0 + k[u]) * 32 + lane) : NONE;
                    if (v[u] != NONE && !DBS_CHK_INDEX(d, v[u] & IDX_MASK, d.nb)) v[u] = NONE;
                }
#pragma unroll
                for (int u = 0; u < U; ++u) xm[u] = v[u] != NONE ? mask_of(F, v[u] & IDX_MASK) : 0u;
#pragma unroll
                for (int u = 0; u < U; ++u) {
                    const bool got = (xm[u] >> (v[u] >> 27)) & 1u;
                    const uint32_t fk = __ballot_sync(FULL, got);
                    if (got) levels[(size_t)(w0 + k[u]) * 32 + lane] = depth;
                    if (lane == k[u]) found |= fk;
                }
            }
        }
        // rows: bit k of `mine` = row (lane + k) mod 32 of word w0 + k is still wanted.  (The rotation matters where
        // the degree goes with the low bits of the row number, as in an R-MAT graph that was not relabelled: with
        // row = lane, lane 0 would own the heaviest row of every word.)
        __syncwarp();
        s_need[lane] = need & ~found;
        __syncwarp();
        uint32_t mine = 0u;
#pragma unroll 8
        for (int k = 0; k < 32; ++k) mine |= ((s_need[k] >> ((lane + k) & 31)) & 1u) << k;
        uint32_t res = 0u, longm = 0u;
        int k = 0, p = 0, e = 0, rounds = 0;
        bool active = false;
        // (the run of the lane's next row is fetched while the current one is walked)
        int kn = 0, pn = 0, en = 0;
        bool have_next = false;
        auto fetch_next = [&]() {
            have_next = mine != 0u;
            if (have_next) {
                kn = __ffs(mine) - 1;
                mine &= mine - 1;
                const size_t row = (size_t)(w0 + kn) * 32 + ((lane + kn) & 31);
                pn = d.rowrun_ptr[row];
                en = d.rowrun_ptr[row + 1];
            }
        };
        fetch_next();
        while (__any_sync(FULL, active || have_next)) {
            if (!active && have_next) {               // next row of this lane
                k = kn; p = pn; e = en;
                active = p < e;
                rounds = 0;
                fetch_next();
            }
            // (one form with the second group's loads left out: 150^3 cells 7400 us, 8 M uniform rows of four 866; a form each 6530 and 823)
            if (active && !wide) {
                // a round = the aligned group of four entries from position p on: one 16-byte load
                const int q0 = p & ~3;
                const uint4 v4 = __ldcs(reinterpret_cast<const uint4 *>(d.rowrun_idx + q0));       // (the array has slack behind its end)
                uint32_t v[4] = {v4.x, v4.y, v4.z, v4.w}, xm[4];
#pragma unroll
                for (int j = 0; j < 4; ++j) if (q0 + j < p || q0 + j >= e || (v[j] != NONE && !DBS_CHK_INDEX(d, v[j] & IDX_MASK, d.nb))) v[j] = NONE;
#pragma unroll
                for (int j = 0; j < 4; ++j) xm[j] = v[j] != NONE ? mask_of(F, v[j] & IDX_MASK) : 0u;
                bool got = false;
#pragma unroll
                for (int j = 0; j < 4; ++j) got |= ((xm[j] >> (v[j] >> 27)) & 1u) != 0;
                p = q0 + 4;
                if (got) { res |= 1u << k; levels[(size_t)(w0 + k) * 32 + ((lane + k) & 31)] = depth; active = false; }
                else if (p >= e) active = false;
                else if (++rounds == MAX_ROUNDS) { longm |= 1u << k; active = false; }     // a long row: finished by the whole warp below
            } else if (active) {
                // under a small frontier, two groups a round
                const int q0 = p & ~3;
                uint4 v4 = __ldcs(reinterpret_cast<const uint4 *>(d.rowrun_idx + q0)), w4 = make_uint4(NONE, NONE, NONE, NONE);   // (the array has slack behind its end)
                if (q0 + 4 < e) w4 = __ldcs(reinterpret_cast<const uint4 *>(d.rowrun_idx + q0 + 4));
                uint32_t v[8] = {v4.x, v4.y, v4.z, v4.w, w4.x, w4.y, w4.z, w4.w}, xm[8];
#pragma unroll
                for (int j = 0; j < 8; ++j) if (q0 + j < p || q0 + j >= e || (v[j] != NONE && !DBS_CHK_INDEX(d, v[j] & IDX_MASK, d.nb))) v[j] = NONE;
#pragma unroll
                for (int j = 0; j < 8; ++j) xm[j] = v[j] != NONE ? mask_of(F, v[j] & IDX_MASK) : 0u;
                bool got = false;
#pragma unroll
                for (int j = 0; j < 8; ++j) got |= ((xm[j] >> (v[j] >> 27)) & 1u) != 0;
                p = q0 + 8;
                if (got) { res |= 1u << k; levels[(size_t)(w0 + k) * 32 + ((lane + k) & 31)] = depth; active = false; }
                else if (p >= e) active = false;
                else if (++rounds == MAX_ROUNDS) { longm |= 1u << k; active = false; }     // a long row: finished by the whole warp below
            }
        }
        // long rows (hubs with no frontier neighbour among their first entries): the whole warp, 32 * LONG_UNROLL entries per round
        uint32_t lanes_long = __ballot_sync(FULL, longm != 0u);
        while (lanes_long) {
            const int src = __ffs(lanes_long) - 1;
            lanes_long &= lanes_long - 1;
            uint32_t lm = __shfl_sync(FULL, longm, src);
            while (lm) {
                const int kk = __ffs(lm) - 1;
                lm &= lm - 1;
                const size_t row = (size_t)(w0 + kk) * 32 + ((src + kk) & 31);
                const int lp = (d.rowrun_ptr[row] & ~3) + MAX_ROUNDS * per_round, le = d.rowrun_ptr[row + 1];
                bool hit = false;
                for (int q = lp; q < le && !hit; q += 32 * LONG_UNROLL) {
                    uint32_t v[LONG_UNROLL], xm[LONG_UNROLL];
#pragma unroll
                    for (int u = 0; u < LONG_UNROLL; ++u) {
                        const int p_ = q + 32 * u + lane;
                        v[u] = p_ < le ? d.rowrun_idx[p_] : NONE;
                        if (v[u] != NONE && !DBS_CHK_INDEX(d, v[u] & IDX_MASK, d.nb)) v[u] = NONE;
                    }
#pragma unroll
                    for (int u = 0; u < LONG_UNROLL; ++u) xm[u] = v[u] != NONE ? mask_of(F, v[u] & IDX_MASK) : 0u;
                    bool m1 = false;
#pragma unroll
                    for (int u = 0; u < LONG_UNROLL; ++u) m1 |= ((xm[u] >> (v[u] >> 27)) & 1u) != 0;
                    hit = __any_sync(FULL, m1);
                }
                if (hit && lane == src) { res |= 1u << kk; levels[row] = depth; }
            }
        }
        // back to one word per lane: bit (l + k) mod 32 of word w0 + k <- bit k of lane l's result
        for (int kk = 0; kk < W; ++kk) {
            const uint32_t fk = __ballot_sync(FULL, (res >> kk) & 1u);
            if (lane == kk) found |= __funnelshift_l(fk, fk, kk);
        }
        found &= need;
        if (in) N[wd] = found;
        if (found) d.ws.visited32[wd] |= found;
        n_nz += ((found & 0xFFFFu) != 0) + ((found >> 16) != 0);
        if (__any_sync(FULL, found != 0u)) append_words(nx, wd, found, found != 0u, lane);
    }
    n_nz = __reduce_add_sync(FULL, n_nz);
    if (lane == 0 && n_nz) atomicAdd(&nx.set->n_blocks, n_nz);
}

// Per-level selector (Section 3.3.1): push iff N_nzblk / N_blk < th3.  Monotone in n_nzblk.
__device__ __forceinline__ int bfs_path(int n_nzblk, int nb, float th3, int force_path) {
    if (force_path == DBSPMSPV_PATH_PUSH || force_path == DBSPMSPV_PATH_PULL) return force_path;
    return ((float)n_nzblk / (float)nb < th3) ? DBSPMSPV_PATH_PUSH : DBSPMSPV_PATH_PULL;
}

// Worklist of the frontier F from the listed nonzero words of its masks: a warp takes one word
// (two vector blocks) at a time, lane = column; frontier columns emit their INLINE runs (adjacent
// ones merged), lanes 0 and 16 the payload runs of the two blocks.  (With the words in index
// order, the few warps that held the hub blocks of an early frontier wrote almost the whole
// worklist.)
__device__ void bfs_worklist(const Device &d, const Scope &sc, const uint32_t *F, const int32_t *words, int n_listed,
                             int32_t *n_tasks, int32_t *n_hubs, int4 *hubs, uint2 *tasks) {
    const int lane = threadIdx.x & 31;
    Counters *ctr = d.ws.ctr;
    for (int i = sc.gwarp; i < n_listed; i += sc.nwarps) {
        const int wd = words[i];
        const uint32_t word = F[wd];
        const int jb = 2 * wd + (lane >> 4), j = jb * 16 + (lane & 15);
        const bool listed = (word >> lane) & 1u;
        int first = 0, deg = 0;
        if (listed) column_run(d, j, first, deg);
        merge_column_runs(listed, j, first, deg, lane);
        emit_tasks(d, false, jb, first, deg, lane, n_tasks, &ctr->pad, PUSH_CHUNK, n_hubs, hubs, tasks);
        first = 0; deg = 0;
        if ((lane & 15) == 0 && ((word >> lane) & 0xFFFFu)) payload_run(d, jb, first, deg);
        if (__any_sync(FULL, deg > 0)) emit_tasks(d, false, jb, first, deg, lane, n_tasks, &ctr->pad, d.payload_chunk, nullptr, nullptr, tasks);
    }
}

// Path of a level (Section 3.3.1): push iff the ratio of nonempty
// frontier blocks is below th3 -- and, the worklist of a push level being built by then, iff that
// worklist is short: a frontier of a few hub vertices fills few vector blocks but owns a good
// part of all stored elements, and a pull, which stops every row at its first frontier
// neighbour, reads less than the push of all those elements would (edge_frac = the share of
// the view's entries above which the push is given up; 0 = block ratio only).  `steps`: warp steps of the worklist;
// `edges`: elements it would hold at least, where they were counted (such a frontier's worklist is not built at all: a few thousand hubs make hundreds of
// thousands of records, 10 us on 2^22 vertices).
__device__ __forceinline__ int bfs_level_path(const Device &d, int n_nzblk, int steps, int edges, float th3, float edge_frac, int force_path) {
    int path = bfs_path(n_nzblk, d.nb, th3, force_path);
    if (path == DBSPMSPV_PATH_PUSH && force_path == DBSPMSPV_PATH_AUTO && edge_frac > 0.f && d.rowrun_ptr != nullptr &&
        ((float)edges > edge_frac * (float)d.n_entries || (float)steps * (float)PUSH_CHUNK > edge_frac * (float)d.n_entries)) path = DBSPMSPV_PATH_PULL;
    return path;
}

// (a level uses one or the other; behind a layout that is given up nobody looks at it any more)
union BfsShared {
    uint32_t need[BFS_CTA];                           // per warp: the wanted rows of its 32 words (transposed pull)
    BfsListShared list;
};

// One level of the search: the expansion of the frontier of level lv.  Three mask buffers rotate:
// F holds the frontier, N receives the next one, Z (the frontier before) is cleared meanwhile and
// becomes N of the next level.  Four lists of nonzero mask words and of vertices rotate with them -- the lists of
// the frontier produced by level L are number L % 4 -- and three sets of per-level counters, so
// that nothing is moved or reset behind an extra barrier.  `now`: the counters of the frontier (in: this level's, out: the next one's, fetched once behind the last barrier);
// z_words: mask words of Z.
template <int DT>
__device__ void bfs_level(const Device &d, cg::grid_group &grid, const Scope &sc, int lv, Counters::BfsSet &now, int z_words, int32_t *levels, float th3,
                          float edge_frac, int force_path, BfsShared &sh) {
    Counters *ctr = d.ws.ctr;
    const int lane = threadIdx.x & 31;
    const int n_words = (d.mb + 1) / 2;
    uint32_t *const buf[3] = {d.ws.x_mask32, d.ws.y_mask32, d.ws.z_mask32};
    const int cur = lv % 3, nxt = (lv + 1) % 3, spare = (lv + 2) % 3;
    const uint32_t *F = buf[cur];
    uint32_t *N = buf[nxt], *Z = buf[spare];
    const int q_in = (lv + 3) & 3, q_out = lv & 3, q_z = (lv + 2) & 3;      // lists: of the frontier / produced now / of Z
    const int32_t *words_z = d.ws.bfs_words + (size_t)q_z * d.ws.bfs_words_stride;
    const int depth = lv + 1;
    const bool counts = d.col_degree && words_per_warp(n_words, sc.nwarps) >= BFS_LARGE_WORDS;
    const NextLevel nx{N, d.ws.bfs_words + (size_t)q_out * d.ws.bfs_words_stride, d.ws.bfs_verts + q_out * BFS_LIST, &ctr->bfs_set[nxt], counts};
    // counters that come into use at the next level are reset now: nobody reads or writes them
    // during this one (the previous level was their last reader, behind a barrier)
    if (sc.tid == 0) {
        ctr->bfs_set[spare] = Counters::BfsSet{0, 0, 0, 0};
        ctr->bfs_work[nxt][0] = 0;
        ctr->bfs_work[nxt][1] = 0;
        if (depth <= DBSPMSPV_MAX_BFS_LEVELS_RECORDED) {
            ctr->bfs_level_nzblk[depth - 1] = now.n_blocks;
            ctr->bfs_stamp[depth] = global_timer_ns();
        }
    }
    auto took = [&](int path) { if (sc.tid == 0 && depth <= DBSPMSPV_MAX_BFS_LEVELS_RECORDED) ctr->bfs_level_path[depth - 1] = path; };
    auto next = [&]() {
        grid.sync();
        const int4 v = __ldcg(reinterpret_cast<const int4 *>(&ctr->bfs_set[nxt]));
        now = Counters::BfsSet{v.x, v.y, v.z, v.w};
    };
    int path = bfs_level_path(d, now.n_blocks, 0, now.edges, th3, edge_frac, force_path);
    if (path == DBSPMSPV_PATH_PUSH && now.n_verts <= BFS_LIST) {
        int elems;
        const int32_t *const verts = d.ws.bfs_verts + q_in * BFS_LIST;
        const int total = bfs_list_layout(d, verts, now.n_verts, sh.list, elems);
        path = bfs_level_path(d, now.n_blocks, 0, elems, th3, edge_frac, force_path);
        if (path == DBSPMSPV_PATH_PUSH && elems <= BFS_MARK_STEPS * PUSH_CHUNK) {
            took(path);
            for (int i = sc.tid; i < z_words; i += sc.nthreads) Z[words_z[i]] = 0u;
            bfs_push_list<DT>(d, verts, total, sh.list, levels, depth, nx);
            next();
            return;
        }
    }
    int n_tasks = 0, n_hubs = 0, steps = 0;
    int4 *const hubs = d.ws.hubs + cur * HUB_CAP;
    if (path == DBSPMSPV_PATH_PUSH) {
        // (the level may still turn to a pull when the worklist is long)
        bfs_worklist(d, sc, F, d.ws.bfs_words + (size_t)q_in * d.ws.bfs_words_stride, now.n_words, &ctr->bfs_work[cur][0], &ctr->bfs_work[cur][1], hubs, d.ws.tasks);
        grid.sync();
        n_tasks = __ldcg(&ctr->bfs_work[cur][0]);
        n_hubs = min(__ldcg(&ctr->bfs_work[cur][1]), HUB_CAP);
        steps = n_tasks;                                // the task records plus the steps of the listed hub runs
        for (int k = 0; k < n_hubs; ++k) steps += (hubs[k].z + PUSH_CHUNK - 1) / PUSH_CHUNK;
        path = bfs_level_path(d, now.n_blocks, steps, now.edges, th3, edge_frac, force_path);
    }
    took(path);
    if (path != DBSPMSPV_PATH_PUSH && d.rowrun_ptr != nullptr) {
        // a pull over the row-run index does its own bookkeeping (it owns the mask words it writes)
        bfs_pull_rows<DT>(d, F, Z, nx, levels, depth, (float)now.n_blocks < BFS_WIDE_PULL * (float)d.nb, sh.need + (threadIdx.x >> 5) * 32);
        next();
        return;
    }
    const bool mark = path == DBSPMSPV_PATH_PUSH && steps <= BFS_MARK_STEPS;
    if (path == DBSPMSPV_PATH_PUSH) {
        // Z (the frontier before this one) is cleared through its list
        for (int i = sc.tid; i < z_words; i += sc.nthreads) Z[words_z[i]] = 0u;
        if (mark) bfs_push<DT, true>(d, sc, F, d.ws.tasks, n_tasks, hubs, n_hubs, levels, depth, nx);
        else bfs_push<DT, false>(d, sc, F, d.ws.tasks, n_tasks, hubs, n_hubs, levels, depth, nx);
    } else bfs_pull<DT>(d, sc, F, N, levels, depth);    // over the row-block segments (no row-run index)
    if (mark) { next(); return; }
    grid.sync();
    // Levels, visited, the lists and the counts: a warp takes its words, then writes the levels of one nonzero word after the other, lane = row
    // (32 words each kept 684 of 4736 warps busy on 700 K vertices: a search with such a level 107 us, 104 with the words spread).  (A pull over segments has written its levels, and left Z.)
    const bool pulled = path != DBSPMSPV_PATH_PUSH;
    int nz = 0, edges = 0;
    const int W = words_per_warp(n_words, sc.nwarps);
    for (int k0 = sc.gwarp * W; k0 < n_words; k0 += sc.nwarps * W) {
        const int k = k0 + lane;
        const bool in = lane < W && k < n_words;
        const uint32_t nm = in ? __ldcg(N + k) : 0u;
        if (nm) {
            d.ws.visited32[k] |= nm;
            nz += ((nm & 0xFFFFu) != 0) + ((nm >> 16) != 0);
        }
        if (pulled && in) Z[k] = 0u;
        if (__any_sync(FULL, nm != 0u)) append_words(nx, k, nm, nm != 0u, lane);
        if (!pulled)
            for (uint32_t todo = __ballot_sync(FULL, nm != 0u); todo; todo &= todo - 1) {
                const int q = __ffs(todo) - 1;
                if ((__shfl_sync(FULL, nm, q) >> lane) & 1u) {
                    const size_t row = (size_t)(k0 + q) * 32 + lane;
                    levels[row] = depth;
                    if (counts) edges += (int)degree_of_code(d.col_degree[row]);
                }
            }
    }
    add_counts(nx, nz, edges, lane);
    next();
}

template <int DT>
__global__ void __launch_bounds__(BFS_CTA) k_bfs(Device d, int32_t src, int32_t *levels, float th3, float edge_frac,
                                                 int force_path, int max_levels) {
    __shared__ BfsShared sh;
    cg::grid_group grid = cg::this_grid();
    const int tid = blockIdx.x * blockDim.x + threadIdx.x;
    const int nthreads = gridDim.x * blockDim.x;
    const int n_words = (d.mb + 1) / 2;
    Counters *ctr = d.ws.ctr;
    const Scope sc{tid, nthreads, tid >> 5, nthreads >> 5};
    if (tid == 0) ctr->bfs_stamp[0] = global_timer_ns();

    // levels = -1 (16-byte stores over the aligned middle, the ragged ends one by one)
    {
        const uintptr_t addr = reinterpret_cast<uintptr_t>(levels);
        int64_t head = (int64_t)((16 - (addr & 15)) & 15) / 4;
        if (head > d.n) head = d.n;
        const int64_t n4 = (d.n - head) / 4;
        int4 *mid = reinterpret_cast<int4 *>(levels + head);
        const int64_t at = (int64_t)src - head;            // the source's place in the middle
        for (int64_t v = tid; v < n4; v += nthreads) mid[v] = v == (at >> 2) && at >= 0 ? make_int4((at & 3) ? -1 : 0, (at & 3) == 1 ? 0 : -1, (at & 3) == 2 ? 0 : -1, (at & 3) == 3 ? 0 : -1) : make_int4(-1, -1, -1, -1);
        for (int64_t v = tid; v < head; v += nthreads) levels[v] = v == src ? 0 : -1;
        for (int64_t v = head + n4 * 4 + tid; v < d.n; v += nthreads) levels[v] = v == src ? 0 : -1;
    }
    // rows without a stored element can never be reached through a pull: they start out as
    // "visited", so that a row block is skipped (and a segment left early) once every row that
    // can be found has been found
    // The source is the first frontier: whoever initialises its word and its level sets them right, so one barrier is enough.
    const int src_word = src >> 5;
    const uint32_t src_bit = 1u << (src & 31);
    for (int k = tid; k < n_words; k += nthreads) {
        const bool mine = k == src_word;
        d.ws.visited32[k] = ~d.row_present32[k] | (mine ? src_bit : 0u);
        d.ws.x_mask32[k] = mine ? src_bit : 0u; d.ws.y_mask32[k] = 0u; d.ws.z_mask32[k] = 0u;
    }
    if (tid == 0) {
        for (int k = 0; k < 3; ++k) { ctr->bfs_set[k] = Counters::BfsSet{k == 0, k == 0, k == 0, 0}; ctr->bfs_work[k][0] = 0; ctr->bfs_work[k][1] = 0; }
        d.ws.bfs_words[(size_t)3 * d.ws.bfs_words_stride] = src_word;        // (the source's lists are number 3 = "produced by level -1")
        d.ws.bfs_verts[3 * BFS_LIST] = src;
    }
    grid.sync();
    int lv = 0, z_words = 0;
    int64_t reached = 1;
    Counters::BfsSet now{1, 1, 1, 0};
    while (lv < max_levels && now.n_blocks != 0) {
        const int f_words = now.n_words;
        bfs_level<DT>(d, grid, sc, lv, now, z_words, levels, th3, edge_frac, force_path, sh);    // ends with a grid barrier
        z_words = f_words;
        reached += now.n_verts;
        ++lv;
    }
    // leave the shared workspace as dbspmspv_run expects it: all masks clear.  The frontier before
    // the last one (buffer (lv + 2) % 3) is cleared through its list; the last frontier is empty
    // unless the level cap ended the search; the third buffer is clear.
    {
        uint32_t *const buf[3] = {d.ws.x_mask32, d.ws.y_mask32, d.ws.z_mask32};
        uint32_t *Z = buf[(lv + 2) % 3], *F = buf[lv % 3];
        const int32_t *wz = d.ws.bfs_words + (size_t)((lv + 2) & 3) * d.ws.bfs_words_stride;
        for (int i = tid; i < z_words; i += nthreads) Z[wz[i]] = 0u;
        if (now.n_blocks != 0)
            for (int k = tid; k < n_words; k += nthreads) F[k] = 0u;
    }
    if (tid == 0) {
        ctr->bfs_levels = lv;
        ctr->bfs_reached = (int32_t)reached;
        if (lv < DBSPMSPV_MAX_BFS_LEVELS_RECORDED + 1) ctr->bfs_stamp[lv + 1] = global_timer_ns();
    }
}

template <int DT>
static int bfs_typed(dbspmspv_handle_s *h, int32_t src, int32_t *levels, cudaStream_t st) {
    Device d = h->d;
    if (!h->bfs_grid) {
        int per_sm = 0;
        if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_bfs<DT>, BFS_CTA, 0) != cudaSuccess || per_sm < 1) return DBSPMSPV_ERR_CUDA;
        h->bfs_grid = per_sm * h->sm_count;
    }
    float th3 = h->ropts.th3_bfs;
    float edge_frac = h->ropts.bfs_push_max_edge_frac;
    int force = h->ropts.force_path;
    int max_levels = d.n > 0x7FFFFFFF ? 0x7FFFFFFF : (int)d.n;
    void *args[] = {&d, &src, &levels, &th3, &edge_frac, &force, &max_levels};
    DBS_CUDA(cudaLaunchCooperativeKernel((void *)k_bfs<DT>, dim3(h->bfs_grid), dim3(BFS_CTA), args, 0, st));
    ++h->kernel_launches;
    return DBSPMSPV_OK;
}

}  // namespace dbs

extern "C" int db_bfs(dbspmspv_handle_t h, int32_t src, int32_t *levels, dbspmspv_stream_t stream) {
    if (!h || !levels) return DBSPMSPV_ERR_INVALID_ARG;
    if (h->d.m != h->d.n) return DBSPMSPV_ERR_UNSUPPORTED;
    if (src < 0 || src >= h->d.n) return DBSPMSPV_ERR_INVALID_ARG;
    if (!dbs::on_handle_device(h)) return DBSPMSPV_ERR_INVALID_ARG;
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    h->last_stream = st;
    switch (h->d.dtype) {
        case DBSPMSPV_F32: return dbs::bfs_typed<DBSPMSPV_F32>(h, src, levels, st);
        case DBSPMSPV_BF16: return dbs::bfs_typed<DBSPMSPV_BF16>(h, src, levels, st);
        default: return dbs::bfs_typed<DBSPMSPV_PATTERN>(h, src, levels, st);
    }
}

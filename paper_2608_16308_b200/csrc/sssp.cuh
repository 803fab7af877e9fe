// db_sssp on hypersparse handles: the whole search in one cooperative launch, no accumulator and no sparse vectors in between.
//
// The search is the synchronous iteration of (min, +) products: step t relaxes the out-edges of the
// vertices whose distance improved in step t - 1, with the distances they had at the end of that step.  As a host loop over
// dbspmspv_run it paid, per step, a blocking of x, an accumulator that was filled and compacted, a relaxation pass and a
// round trip to the host (R-MAT scale 20: 9 steps, 1.17 ms, of which 0.2 ms an idle GPU).  Here a step reads the distances from one of two arrays of words, which nobody writes meanwhile, and lowers the
// words of the other one, which then holds the distances:
//   expand   the columns of the frontier (a bitmap) laid end to end per thread block as in the direct push (push_direct.cuh); a candidate
//            distance goes straight into the target's word with an atomic minimum, and the thread whose atomic is the first to bring
//            it below the distance marks the target in the next frontier and counts it;
//   long     the listed long runs and payload runs, a warp per chunk (only if there are any);
// with a grid barrier after each.  The other array has the distances of two steps ago: they differ from the present ones in the vertices of the frontier, which whoever expands them brings down
// as well, in whatever order.  (With one array a pass behind every step copied and counted what was marked, one more barrier and 5 - 10 us a step.)
// A large step is pulled (sssp_pull), row by row.  A step that reaches few edges (of INLINE runs, which is what is counted: steps of a 27-point operator list a little longer, and gain by it
// like the others) also lists what it marks; a frontier that is listed and short is expanded
// from its list in one phase, long runs and payload entries included (sssp_expand_list).  A step finds the same improvements, distance for distance, as the product did: a vertex is marked iff its word
// went below the distance it had before the step.  The caller's distances are written at the end.
//
// What a small step costs is its trips to L2, one after the other, 0.6 us each with what surrounds it: the counters that decide the next step lie in one 16-byte word (SsspSet), fetched once behind the barrier.
// (As five words fetched one by one, with a pass that settled the marked vertices: 16 K vertices 119 -> 102 us a search, 131 K 165 -> 139 (124 -> 104), 300 K 141 -> 126 (140 -> 121), 2^20 305 -> 290 (288 -> 260);
// with the marked vertices settled behind the pulled steps too: 152, 195 (168), 180 (142 with other sources), 364 (306).)
//
// What bounds a large step is the gather of one target distance per edge.  It goes through L1 (a candidate that does not beat the distance is done); only one that does looks at the word
// in L2, and only one that beats that too pays an atomic: the words of hub rows, which thousands of edges reach, settle after a few atomics.
#pragma once

#include <cooperative_groups.h>

#include "internal.cuh"
#include "minplus.cuh"
#include "push_direct.cuh"

namespace dbs {

constexpr int SSSP_CTA = 1024;
constexpr int SSSP_WARPS = SSSP_CTA / 32;
constexpr int SSSP_WORDS = SSSP_CTA / 8;          // frontier words of a thread block's round: eight threads per word, four columns each
constexpr int SSSP_COLS = SSSP_CTA * 4;
constexpr int SSSP_ILP = 4;                       // warp steps in flight
// A step whose frontier reaches more than this share of the stored elements is pulled.  Shares of 5 / 10 / 15 / 20 %, symmetrised R-MAT, means of twelve sources, in brackets with the
// vertices in scattered order: 131 K vertices 172 / 169 / 167 / 168 us a search (128 / 127 / 127 / 128), 300 K 142 / 142 / 143 / 142 (146 / 144 / 143 / 142), 500 K 232 / 229 / 229 / 229,
// 2^20 315 / 307 / 309 / 308 (291 / 286 / 286 / 286).
constexpr float SSSP_PULL_SHARE = 0.1f;
// ... on handles of weights with many payload blocks (payload_rich), whose entries a push takes one by one, while their rows are shared among lanes, which makes a pulled step cheap: 27-point operators, weights
// of one size / in [0.05, 1.05), which improve a vertex more often, four sources, 5 -> 10 %: 40^3 cells 408 -> 568 / 493 -> 540 us a search, 90^3 2493 -> 2517 / 5000 -> 4863, 120^3 4971 -> 5006 / 12181 -> 11725,
// 150^3 10084 -> 10356 / 28964 -> 27580 (before the rules on shares 11517 / 27904).
constexpr float SSSP_PULL_SHARE_PAYLOAD = 0.05f;
// Once a step has been pulled the rows have bests that prune, and a pulled step that finds little costs a pass over the rows: the share for the steps behind it.  5 / 0.5 / 0.2 / 0.05 %, six
// sources: 131 K vertices 180 / 174 / 173 / 172 (156 / 149 / 149 / 149), 300 K 175 / 168 / 167 / 167 (136 / 133 / 133 / 134), 500 K 253 / 242 / 240 / 239, 2^20 371 / 362 / 362 / 356 (307 / 296 / 294 / 301).
constexpr float SSSP_LATE_SHARE = 0.002f;
// With weights that pass is what the step costs on large graphs: it has to be worth an edge for so many rows too -- an eighth of them at 2^20, rising with the square to all of them, the more of the rows' words no longer
// stay in L2 (and with fewer elements a row than R-MAT's 32 the share of the elements says little about it).  A share of 0.2 % alone / an eighth / a quarter / a half / all of the rows, uniform rows of 4 or 8:
// 2 M x 4 1135 / 1004 / 931 / 896 / 896 us a search, x 8 1483 / 1399 / 1347 / 1290 / 1239, 8 M x 4 4123 / 3620 / 3480 / 3393 / 3393, x 8 5514 / 5157 / 4969 / 4781 / 4602; R-MAT 2^20 286 / 287 / 288 / 291 / 294 (251 / 252 / 253 / 254 /
// 260); on handles with many payload blocks no more than that eighth, 150^3 cells, weights in [0.05, 1.05), an eighth / a half 27580 / 27754.  (Unit weights: the share alone is the better rule, 8 M uniform rows x 8 764 / 776 / 775 / 791 / 793, R-MAT of 4 M vertices x 8 234 / 242 / 249 / 258 / 259.)
constexpr float SSSP_LATE_ROWS = 0.125f;
// Rounds of four elements that a lane walks of a row.  6 / 8 / 12, the same six: 131 K vertices 177 / 173 / 180 (153 / 149 / 158), 300 K 172 / 167 / 175 (137 / 133 / 136), 500 K 246 / 240 / 240,
// 2^20 373 / 362 / 363 (300 / 294 / 299).
constexpr int SSSP_ROUNDS = 8;
constexpr int SSSP_CHUNK = 512;                   // elements of a listed chunk of a longer row
// A step whose frontier reaches at most so many edges lists the vertices it marks; a list of at most SSSP_LIST vertices serves the next step.
// (The bitmap of 2^20 vertices is two rounds of every thread block, whatever it holds: a step of a few vertices took 14 us, 26 with a long run.)
constexpr int SSSP_LIST = SSSP_CTA;
constexpr unsigned SSSP_LIST_EDGES = 1u << 17;
constexpr int SSSP_STARTS = 1, SSSP_LATE = 2, SSSP_BELOW_ZERO = 4;      // a launch: the first of its search, or one behind it (a step has been pulled before; a distance has been below zero)
constexpr int SSSP_MAX_STEPS = 1024;              // steps of one launch, at most: a cycle of negative weight ends on the host

// What a step leaves to the next one, in one 16-byte word: a barrier is followed by one trip to L2.
struct alignas(16) SsspSet {
    unsigned edges, found;    // out-edges of the frontier in INLINE runs (to an eighth); its vertices
    int low;                  // its smallest word
    int n_long;               // chunks of long runs or rows that the step itself listed
};
struct SsspState {
    int *word[2];             // distances (ordered words): a step reads them from one array, which nobody writes meanwhile, and lowers them in the other
    uint32_t *bits[3];        // frontiers, one bit per vertex: the step's, the one it marks, the one before (being cleared), in turn
    SsspSet *set;             // three of them, in turn
    int32_t *ctr;             // [0] steps made, [1] array of the distances, [2..4] places taken in the step's list
    int4 *chunks;             // {row, first, end, -} of the listed chunks of long rows
    int32_t *list[2];         // the vertices marked by alternating steps, SSSP_LIST at most
    int32_t *report;          // page-locked host words: steps made, vertices of the frontier that was left, SSSP_LATE, SSSP_BELOW_ZERO of what came before
    int32_t n_words;
};

// ordered(v): monotone in v, and the bits themselves where v >= 0
__device__ __forceinline__ int sssp_word(float v) { return ordered_word(__float_as_int(v)); }
__device__ __forceinline__ float sssp_value(int w) { return __int_as_float(ordered_word(w)); }

struct SsspShared {
    int pre[SSSP_COLS + 1];                       // elements before a column of the round
    int2 run[SSSP_COLS];                          // position of its first entry minus that; its distance
    uint16_t own[SSSP_COLS * PD_LONG / 32];       // column that owns the first element of a step of 32
    int cnt[SSSP_WARPS], sum[SSSP_WARPS], rec[SSSP_WARPS], base;
};

// What a step finds: vertices that it lowers, the smallest of their words, their out-edges (fewer than 2^32 together).  Every thread keeps its own.
struct SsspTally {
    int found = 0, low = 0x7F800000;
    unsigned edges = 0;
};
// Into the next step's counters, summed up per thread block.  Called by all of its threads.
struct SsspSums { int found[SSSP_WARPS], low[SSSP_WARPS]; unsigned edges[SSSP_WARPS]; };
__device__ __forceinline__ void sssp_count(const SsspState &s, SsspSums &sums, int set, const SsspTally &tally) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    int found = __reduce_add_sync(FULL, tally.found), low = __reduce_min_sync(FULL, tally.low);
    unsigned edges = __reduce_add_sync(FULL, tally.edges);
    if (lane == 0) { sums.found[warp] = found; sums.low[warp] = low; sums.edges[warp] = edges; }
    __syncthreads();
    if (warp != 0) return;
    found = __reduce_add_sync(FULL, sums.found[lane]);
    low = __reduce_min_sync(FULL, sums.low[lane]);
    edges = __reduce_add_sync(FULL, sums.edges[lane]);
    if (lane != 0) return;
    // (a thread block may have lowered vertices further that all had been counted elsewhere: the smallest word can be one of theirs)
    if (found) atomicAdd(reinterpret_cast<unsigned long long *>(&s.set[set].edges), (unsigned long long)(unsigned)found << 32 | edges);
    if (low < 0x7F800000) atomicMin(&s.set[set].low, low);
}
__device__ __forceinline__ unsigned sssp_degree(const Device &d, int j) {
    if (d.col_degree) return degree_of_code(d.col_degree[j]);
    int first, deg;
    column_run(d, j, first, deg);
    return degree_of_code(degree_code((uint32_t)deg));
}

// A pushed step reads the distances, `was`, lowers the words of the other array and marks what it lowers: bits, and (list not null) a list.
struct SsspNext {
    const int *was;
    int *word;
    uint32_t *bits;
    int32_t *list, *n_list;
};

// The candidates of up to U targets per lane (target < 0: none); called by a whole warp.  The one that brings a word below the distance is the vertex's first.  (A vertex of the frontier itself
// may still have its word of two steps ago when it is met, a larger one: it is brought down to the distance by whoever expands it, before or after.)
template <int U>
__device__ __forceinline__ void sssp_relax(const Device &d, const SsspNext &next, const int (&target)[U], const float (&cand)[U], SsspTally &tally) {
    int was[U], seen[U];
    if (!next.list) {
        // (the distances come through L1: nobody writes them in this step.  Looks at the words, atomics and marks side by side: one candidate after the other, searches on a 27-point operator, 90^3 / 150^3 cells,
        // two sources, took 2330 / 11245 us in place of 2286 / 10960; R-MAT within 1 % either way.)
#pragma unroll
        for (int u = 0; u < U; ++u) was[u] = target[u] >= 0 ? __ldca(next.was + target[u]) : (int)0x80000000;
#pragma unroll
        for (int u = 0; u < U; ++u) seen[u] = sssp_word(cand[u]) < was[u] ? __ldcg(next.word + target[u]) : (int)0x80000000;
        uint32_t tried = 0u;
#pragma unroll
        for (int u = 0; u < U; ++u)
            if (sssp_word(cand[u]) < seen[u]) { seen[u] = atomicMin(next.word + target[u], sssp_word(cand[u])); tried |= 1u << u; }
#pragma unroll
        for (int u = 0; u < U; ++u) {
            if (!((tried >> u) & 1u)) continue;
            tally.low = min(tally.low, sssp_word(cand[u]));
            if (seen[u] < was[u]) continue;
            atomicOr(next.bits + (target[u] >> 5), 1u << (target[u] & 31));
            ++tally.found;
            tally.edges += sssp_degree(d, target[u]);
        }
        return;
    }
    // few edges: what counts is the chain.  The atomics go out with no look at the words in front.
    uint32_t fresh = 0u;
#pragma unroll
    for (int u = 0; u < U; ++u)
        if (target[u] >= 0) { was[u] = __ldcg(next.was + target[u]); seen[u] = atomicMin(next.word + target[u], sssp_word(cand[u])); }
#pragma unroll
    for (int u = 0; u < U; ++u) {
        if (target[u] < 0 || sssp_word(cand[u]) >= was[u]) continue;
        tally.low = min(tally.low, sssp_word(cand[u]));
        if (seen[u] < was[u]) continue;
        atomicOr(next.bits + (target[u] >> 5), 1u << (target[u] & 31));
        fresh |= 1u << u;
    }
    if (!__any_sync(FULL, fresh != 0u)) return;
    const int lane = threadIdx.x & 31, mine = __popc(fresh);
    int incl = mine;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) { const int t = __shfl_up_sync(FULL, incl, o); if (lane >= o) incl += t; }
    int base = 0;
    if (lane == 31) base = atomicAdd(next.n_list, incl);
    unsigned edges = 0;                                // (their degrees arrive beside the place in the list)
#pragma unroll
    for (int u = 0; u < U; ++u) if ((fresh >> u) & 1u) edges += sssp_degree(d, target[u]);
    int at = __shfl_sync(FULL, base, 31) + incl - mine;
#pragma unroll
    for (int u = 0; u < U; ++u)
        if ((fresh >> u) & 1u) { if (at < SSSP_LIST) next.list[at] = target[u]; ++at; }
    tally.found += mine;
    tally.edges += edges;
}

template <int DT>
__device__ void sssp_expand(const Device &d, const SsspState &s, const uint32_t *F, const SsspNext &next, int32_t *n_long, SsspShared &sh, SsspTally &tally) {
    constexpr bool VAL = DT != DBSPMSPV_PATTERN;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int rounds = (s.n_words + SSSP_WORDS * (int)gridDim.x - 1) / (SSSP_WORDS * (int)gridDim.x);
    for (int round = 0; round < rounds; ++round) {
        int first[4], deg[4], pfirst = 0, pdeg = 0, col0 = 0;
        float xv[4];
        uint32_t listed = 0;
#pragma unroll
        for (int k = 0; k < 4; ++k) { first[k] = 0; deg[k] = 0; xv[k] = 0.f; }
        const int64_t wi = (int64_t)(round * SSSP_WORDS + (tid >> 3)) * gridDim.x + blockIdx.x;
        if (wi < s.n_words) listed = (__ldcg(F + wi) >> (4 * (tid & 7))) & 15u;
        if (!__syncthreads_or(listed != 0u)) continue;
        int n_rec = 0;
        if (listed) {
            const int j0 = (int)wi * 32 + 4 * (tid & 7);
            col0 = j0 & 15;
            const int32_t *cp = d.csc.colptr + 17 * (j0 >> 4) + col0;
            int c[5];
#pragma unroll
            for (int k = 0; k < 5; ++k) c[k] = cp[k];
#pragma unroll
            for (int k = 0; k < 4; ++k)
                if ((listed >> k) & 1u) {
                    first[k] = c[k]; deg[k] = c[k + 1] - c[k];
                    const int w = __ldcg(next.was + j0 + k);
                    xv[k] = sssp_value(w);
                    atomicMin(next.word + j0 + k, w);
                    if (!DBS_CHK_RANGE(d, first[k], deg[k])) deg[k] = 0;
                }
            if (d.n_payload) payload_run(d, j0 >> 4, pfirst, pdeg);
            // long runs and runs of payload entries: chunks for the second half of the step
#pragma unroll
            for (int k = 0; k < 4; ++k)
                if (deg[k] > PD_LONG) { n_rec += (deg[k] + PD_CHUNK - 1) / PD_CHUNK; deg[k] = -deg[k]; }      // (negative: listed)
            if (pdeg > 0) n_rec += __popc(listed) * ((pdeg + PD_PAYLOAD - 1) / PD_PAYLOAD);
        }
        int n_cols = 0, n_elems = 0;
#pragma unroll
        for (int k = 0; k < 4; ++k) { n_cols += deg[k] > 0; n_elems += max(deg[k], 0); }
        int ic = n_cols, is = n_elems, ir = n_rec;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int a = __shfl_up_sync(FULL, ic, o), b = __shfl_up_sync(FULL, is, o), c = __shfl_up_sync(FULL, ir, o);
            if (lane >= o) { ic += a; is += b; ir += c; }
        }
        if (lane == 31) { sh.cnt[warp] = ic; sh.sum[warp] = is; sh.rec[warp] = ir; }
        __syncthreads();
        // (a lane per warp: the sums before it and the totals)
        const int vc = sh.cnt[lane], vs = sh.sum[lane], vr = sh.rec[lane];
        const int tot_c = __reduce_add_sync(FULL, vc), tot_e = __reduce_add_sync(FULL, vs), tot_r = __reduce_add_sync(FULL, vr);
        int c = ic - n_cols + __reduce_add_sync(FULL, lane < warp ? vc : 0), e = is - n_elems + __reduce_add_sync(FULL, lane < warp ? vs : 0);
        int at = ir - n_rec + __reduce_add_sync(FULL, lane < warp ? vr : 0);
        if (tid == 0) {
            sh.base = tot_r ? atomicAdd(n_long, tot_r) : 0;
            sh.pre[tot_c] = tot_e;
        }
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            if (deg[k] <= 0) continue;
            sh.pre[c] = e;
            sh.run[c] = make_int2(first[k] - e, __float_as_int(xv[k]));
            for (int q = (e + 31) >> 5; q * 32 < e + deg[k]; ++q) sh.own[q] = (uint16_t)c;
            ++c;
            e += deg[k];
        }
        __syncthreads();
        if (tot_r) {                                   // block-uniform; a thread's runs are written by its whole warp
            at += sh.base;
#pragma unroll
            for (int k = 0; k < 4; ++k)
                for (uint32_t todo = __ballot_sync(FULL, deg[k] < 0); todo; todo &= todo - 1) {
                    const int src = __ffs(todo) - 1;
                    const int f = __shfl_sync(FULL, first[k], src), n = -__shfl_sync(FULL, deg[k], src), o = __shfl_sync(FULL, at, src);
                    const int xb = __shfl_sync(FULL, __float_as_int(xv[k]), src);
                    const int n_chunks = (n + PD_CHUNK - 1) / PD_CHUNK;
                    for (int q = lane; q < n_chunks; q += 32) d.ws.long_runs[o + q] = make_int4(f + q * PD_CHUNK, min(PD_CHUNK, n - q * PD_CHUNK), xb, 0);
                    if (lane == src) at += n_chunks;
                }
            if (pdeg > 0)
#pragma unroll
                for (int k = 0; k < 4; ++k)
                    if ((listed >> k) & 1u)
                        for (int q = 0; q < pdeg; q += PD_PAYLOAD) d.ws.long_runs[at++] = make_int4(pfirst + q, min(PD_PAYLOAD, pdeg - q), __float_as_int(xv[k]), 0x100 | (col0 + k));
        }
        // 32 elements per warp step, SSSP_ILP steps at a time; the entries of the next ones are fetched before these are relaxed
        uint32_t idx[SSSP_ILP], w[SSSP_ILP], aux[SSSP_ILP];
        float x[SSSP_ILP];
        auto fetch = [&](int s0) {
#pragma unroll
            for (int u = 0; u < SSSP_ILP; ++u) {
                const int e0 = s0 + u * SSSP_CTA;
                idx[u] = PAD_IDX; w[u] = 0u; aux[u] = 0u; x[u] = 0.f;
                if (e0 < tot_e) {                      // warp-uniform; the step's first owner, then every lane's own (see k_push_direct)
                    const int lo = sh.own[e0 >> 5];
                    const uint32_t b = (uint32_t)(sh.pre[min(lo + 1 + lane, tot_c)] - e0);
                    const uint32_t m = __reduce_or_sync(FULL, b < 32u ? 1u << b : 0u);
                    if (e0 + lane < tot_e) {
                        const int2 run = sh.run[lo + __popc(m & ((2u << lane) - 1u))];
                        x[u] = __int_as_float(run.y);
                        push_entry<VAL>(d, run.x + e0 + lane, idx[u], w[u], aux[u]);
                    }
                }
            }
        };
        if (warp * 32 < tot_e) fetch(warp * 32);
        for (int s0 = warp * 32; s0 < tot_e; s0 += SSSP_CTA * SSSP_ILP) {
            float cand[SSSP_ILP];
            int target[SSSP_ILP];
#pragma unroll
            for (int u = 0; u < SSSP_ILP; ++u) {
                target[u] = idx[u] < (1u << TYPE_SHIFT) ? (int)((idx[u] & IDX_MASK) * 16u + (aux[u] >> 4)) : -1;
                cand[u] = x[u] + Val<DT>::inline_value(w[u]);
            }
            if (s0 + SSSP_CTA * SSSP_ILP < tot_e) fetch(s0 + SSSP_CTA * SSSP_ILP);
            sssp_relax<SSSP_ILP>(d, next, target, cand, tally);
        }
        __syncthreads();                               // (the next round overwrites the layout)
    }
}

template <int DT>
__device__ void sssp_long(const Device &d, const SsspNext &next, int n, SsspTally &tally) {
    constexpr bool VAL = DT != DBSPMSPV_PATTERN;
    constexpr int U = PD_CHUNK / 32;
    const int lane = threadIdx.x & 31;
    const int gwarp = (int)(blockIdx.x * SSSP_CTA + threadIdx.x) >> 5, nwarps = (int)(gridDim.x * SSSP_CTA) >> 5;
    // a chunk's record two rounds ahead, its entries one
    uint32_t idx[U], w[U], aux[U];
    auto record = [&](int i) { return i < n ? __ldcg(d.ws.long_runs + i) : make_int4(0, 0, 0, 0); };
    auto fetch = [&](const int4 &run) {
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const int k = u * 32 + lane;
            idx[u] = PAD_IDX; w[u] = 0u; aux[u] = 0u;
            if (!run.w && k < run.y && DBS_CHK_RANGE(d, run.x, run.y)) push_entry<VAL>(d, run.x + k, idx[u], w[u], aux[u]);
        }
    };
    int4 run = record(gwarp), ahead = record(gwarp + nwarps);
    fetch(run);
    for (int i = gwarp; i < n; i += nwarps) {
        const float x = __int_as_float(run.z);
        float cand[U];
        int target[U];
#pragma unroll
        for (int u = 0; u < U; ++u) {
            target[u] = idx[u] < (1u << TYPE_SHIFT) ? (int)((idx[u] & IDX_MASK) * 16u + (aux[u] >> 4)) : -1;
            cand[u] = x + Val<DT>::inline_value(w[u]);
        }
        if (run.w && DBS_CHK_RANGE(d, run.x, run.y)) { // payload entries: a half-warp each
            static_assert(PD_PAYLOAD / 2 == U, "one element per lane and step either way");
            bool in[U];
            uint32_t rb[U];
            payload_elements<DT, U>(d, run.x, run.y, run.w & 15, lane, in, cand, rb);
#pragma unroll
            for (int u = 0; u < U; ++u) { target[u] = in[u] ? (int)(rb[u] * 16u) + (lane & 15) : -1; cand[u] += x; }
        }
        run = ahead;
        ahead = record(i + 2 * nwarps);
        fetch(run);
        sssp_relax<U>(d, next, target, cand, tally);
    }
}

// A short listed frontier: every thread block lays the vertices' chunks (of their INLINE runs and of the payload entries of their column
// blocks) end to end, the warps of the grid share them out.
struct SsspListShared {
    int pre[SSSP_LIST + 1];                       // chunks before a vertex
    int vertex[SSSP_LIST], first[SSSP_LIST], deg[SSSP_LIST], pfirst[SSSP_LIST], pdeg[SSSP_LIST];
    float x[SSSP_LIST];
    int sum[SSSP_WARPS];
};
template <int DT>
__device__ void sssp_expand_list(const Device &d, const int32_t *list, int cnt, const SsspNext &next, SsspListShared &sh, SsspTally &tally) {
    constexpr bool VAL = DT != DBSPMSPV_PATTERN;
    constexpr int U = PD_CHUNK / 32;
    static_assert(PD_PAYLOAD / 2 == U, "one element per lane and step either way");
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    int j = 0, first = 0, deg = 0, pfirst = 0, pdeg = 0;
    if (tid < cnt) {
        j = __ldcg(list + tid);
        const int w = __ldcg(next.was + j);
        sh.x[tid] = sssp_value(w);
        if (blockIdx.x == 0) atomicMin(next.word + j, w);
        column_run(d, j, first, deg);
        if (d.n_payload) payload_run(d, j >> 4, pfirst, pdeg);
        if (!DBS_CHK_RANGE(d, first, deg)) deg = 0;
        if (!DBS_CHK_RANGE(d, pfirst, pdeg)) pdeg = 0;
    }
    sh.vertex[tid] = j; sh.first[tid] = first; sh.deg[tid] = deg; sh.pfirst[tid] = pfirst; sh.pdeg[tid] = pdeg;
    const int mine = (deg + PD_CHUNK - 1) / PD_CHUNK + (pdeg + PD_PAYLOAD - 1) / PD_PAYLOAD;
    int incl = mine;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) { const int t = __shfl_up_sync(FULL, incl, o); if (lane >= o) incl += t; }
    if (lane == 31) sh.sum[warp] = incl;
    __syncthreads();
    const int v = sh.sum[lane], total = __reduce_add_sync(FULL, v);
    sh.pre[tid] = incl - mine + __reduce_add_sync(FULL, lane < warp ? v : 0);
    if (tid == 0) sh.pre[SSSP_LIST] = total;
    __syncthreads();
    // (neighbouring chunks on different SMs)
    for (int c = warp * (int)gridDim.x + (int)blockIdx.x; c < total; c += (int)gridDim.x * SSSP_WARPS) {
        int o = 0;                                     // the last vertex with at most c chunks before it
#pragma unroll
        for (int st = SSSP_LIST / 2; st; st >>= 1) if (sh.pre[o + st] <= c) o += st;
        const int k = c - sh.pre[o], n_inline = (sh.deg[o] + PD_CHUNK - 1) / PD_CHUNK;
        const float x = sh.x[o];
        float cand[U];
        int target[U];
        if (k < n_inline) {                            // warp-uniform
            const int at = k * PD_CHUNK + lane;
            uint32_t idx[U], w[U], aux[U];
#pragma unroll
            for (int u = 0; u < U; ++u) {
                idx[u] = PAD_IDX; w[u] = 0u; aux[u] = 0u;
                if (at + u * 32 < sh.deg[o]) push_entry<VAL>(d, sh.first[o] + at + u * 32, idx[u], w[u], aux[u]);
            }
#pragma unroll
            for (int u = 0; u < U; ++u) {
                target[u] = idx[u] < (1u << TYPE_SHIFT) ? (int)((idx[u] & IDX_MASK) * 16u + (aux[u] >> 4)) : -1;
                cand[u] = x + Val<DT>::inline_value(w[u]);
            }
        } else {
            const int at = (k - n_inline) * PD_PAYLOAD;
            bool in[U];
            uint32_t rb[U];
            payload_elements<DT, U>(d, sh.pfirst[o] + at, min(PD_PAYLOAD, sh.pdeg[o] - at), sh.vertex[o] & 15, lane, in, cand, rb);
#pragma unroll
            for (int u = 0; u < U; ++u) { target[u] = in[u] ? (int)(rb[u] * 16u) + (lane & 15) : -1; cand[u] += x; }
        }
        sssp_relax<U>(d, next, target, cand, tally);
    }
}

// Elements k0 .. k0 + 3 (k0 a multiple of four) of the runs: columns and weights, one 32-byte sector in one load.
template <bool VAL>
__device__ __forceinline__ void sssp_four(const Device &d, int k0, uint32_t (&col)[4], float (&w)[4]) {
    if (VAL) {
        asm volatile("ld.global.cs.v8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
                     : "=r"(col[0]), "=f"(w[0]), "=r"(col[1]), "=f"(w[1]), "=r"(col[2]), "=f"(w[2]), "=r"(col[3]), "=f"(w[3]) : "l"(d.weightrun + k0));
    } else {
        const uint4 a = __ldcs(reinterpret_cast<const uint4 *>(d.rowrun_idx + k0));
        const uint32_t v[4] = {a.x, a.y, a.z, a.w};
#pragma unroll
        for (int j = 0; j < 4; ++j) { col[j] = (v[j] & IDX_MASK) * 16u + (v[j] >> 27); w[j] = 1.0f; }
    }
}
// No element behind one of weight w can do better than this (the order goes by the upper bits).  The lower bits of an infinite or NaN weight
// must not be cut off: below -infinity in the order of words there are only NaNs, and the bound of a NaN would end the row.
template <bool VAL>
__device__ __forceinline__ float sssp_bound(float xmin, float w) {
    constexpr int least = (int)0x807FFFFFu;        // sssp_word(-infinity)
    return xmin + (VAL ? sssp_value(max(sssp_word(w) & ~((1 << (32 - SSSP_WEIGHT_BITS)) - 1), least)) : w);
}

// A large step pulled.  Every row walks its own elements, which lie by weight (Device::weightrun), and stops at the first that
// cannot improve it: smallest distance of the frontier + weight >= the row's best.  In the late large steps of an R-MAT search that leaves a
// seventh of the elements, and a row reached for the first time soon has a best of its own.  Columns outside the
// frontier improve nothing (their edges were relaxed when they entered it), so they need no test.
// Rows that their lightest element (Device::row_lightest) cannot improve are sorted out 32 at a time; the others go to a queue of the warp, from which
// a lane takes the next one as soon as it has finished a row, four elements (one 32-byte sector) a round.  What is left of a row that has not
// stopped after SSSP_ROUNDS rounds is listed in chunks, which all warps share out behind a grid barrier (walked by the warp that met them, the
// hub rows of an R-MAT graph, neighbours all, took one warp 300 us); of a row of several chunks only those whose first weight can still improve it.
// Handles of unit weights walk the row-run index.
// The sums of a walk are compared as floats (a distance is never -0, and fminf leaves NaNs out like the order of words does), and a gathered word is taken for its bits until a distance has been below zero:
// where most rows are walked to their end, instructions bound the step.  Every sum turned into a word and every distance back / sums as floats / so: 27-point operator, weights in [0.05, 1.05), four sources,
// 90^3 cells 6180 / 5180 / 5000 us a search, 120^3 15040 / 12580 / 12180, 150^3 35290 / 29620 / 28960; R-MAT 131 K vertices 117 / 110 / 110, 300 K 157 / 147 / 147, 2^20 183 / 171 / 168.
// What bounds it: a distance gathered per element, one a clock and SM at most (12 M in the first pulled step of R-MAT scale 20: 41 of its 80 us), then the rows that come last, while
// most warps stand at the barrier (the L1 is 11 % busy over a whole search).  That step took 156 us when a lane walked seven rows of its own and the blocks with a payload followed, a warp
// at a time; the whole search 670, 560 and 530 us from three sources, 400, 328 and 312 now; in scattered order 354 - 466, 270 - 367 now.  A frontier bitmap in shared memory in front of the gathers: 80 -> 103 (L1 is what it
// takes away); less shared memory by half the columns a round in sssp_expand: within 2 %.
struct SsspPullShared {
    int4 queue[SSSP_WARPS][64];       // {row, first, end, best so far} of the rows that wait for a lane
    int4 longs[SSSP_WARPS][32];                   // {row, first, end, best} of what is left of long rows
    int queue_degree[SSSP_WARPS][64];             // their columns' elements, at least
    int cursor;                                   // groups of rows taken by the thread block's warps
};

// A row lowered to `best`, below its distance `had`, by one of several threads that may.
__device__ __forceinline__ void sssp_lower(const Device &d, int *word, uint32_t *next, int row, int best, int had, SsspTally &tally) {
    tally.low = min(tally.low, best);
    if (atomicMin(word + row, best) < had) return;     // (not the first)
    atomicOr(next + (row >> 5), 1u << (row & 31));
    ++tally.found;
    tally.edges += sssp_degree(d, row);
}
// Chunks of the n <= 32 long rows that a warp has met.
template <bool VAL>
__device__ __forceinline__ void sssp_list_long(const Device &d, const SsspState &s, const int4 *longs, int n, float xmin, int32_t *n_long, int lane) {
    const int4 r = lane < n ? longs[lane] : make_int4(0, 0, 0, 0);
    int chunks = (r.z - r.y + SSSP_CHUNK - 1) / SSSP_CHUNK;
    if (VAL)
        for (uint32_t todo = __ballot_sync(FULL, chunks > 1); todo; todo &= todo - 1) {      // the warp looks at 32 chunks of a row at a time
            const int src = __ffs(todo) - 1, first = __shfl_sync(FULL, r.y, src), all = __shfl_sync(FULL, chunks, src);
            const float best = sssp_value(__shfl_sync(FULL, r.w, src));
            int kept = 0;
            while (kept < all) {
                const int c = kept + lane;
                const bool in = c < all && (c == 0 || sssp_bound<VAL>(xmin, __uint_as_float(d.weightrun[first + c * SSSP_CHUNK].y)) < best);
                const uint32_t m = __ballot_sync(FULL, in);
                if (m != FULL) { kept += __ffs(~m) - 1; break; }
                kept += 32;
            }
            if (lane == src) chunks = kept;
        }
    int incl = chunks;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) { const int t = __shfl_up_sync(FULL, incl, o); if (lane >= o) incl += t; }
    int base = 0;
    if (lane == 31) base = atomicAdd(n_long, incl);
    int at = __shfl_sync(FULL, base, 31) + incl - chunks;
    for (int c = 0; c < chunks; ++c) s.chunks[at++] = make_int4(r.x, r.y + c * SSSP_CHUNK, min(r.z, r.y + (c + 1) * SSSP_CHUNK), 0);
}

// A pulled step of a graph with no more rows than the GPU has lanes (handles with weights): 1 << share lanes share a row, four elements each a round, so that a row is a round or two instead of up to
// eight one after the other; what is left of it after SSSP_SHARED_ROUNDS of them is listed.  What bounds the step there is that chain (a round takes 2 us whatever it holds) with most warps idle.
// A lane per row / so: 16 K vertices 102 / 78 us a search, in scattered order 113 / 88, 40 K 113 / 95, 65 K 104 / 86 in scattered order, 131 K 140 / 129 (104 / 96); two lanes per row also on 300 K
// 125 / 121 (120 / 124), on 500 K 205 / 232: not above the number of lanes.  Four lanes on 65 K 96 in place of 87, on 40 K the same: as many as there are for every row.  Eight rounds: 83, 93, 100, 102, 137 (102).
constexpr int SSSP_SHARED_ROUNDS = 4;
static_assert(8 * SSSP_SHARED_ROUNDS - 3 > 4 * (SSSP_ROUNDS - 1), "the list of chunks has room for rows of that length (run.cu)");
__device__ __forceinline__ int sssp_row_share(int64_t n, int nthreads) {
    int share = n <= nthreads ? 1 : 0;
    while (share && share < 3 && n << (share + 1) <= nthreads) ++share;
    return share;
}
__device__ void sssp_pull_shared(const Device &d, const SsspState &s, int c, uint32_t *next, int share, int low, int32_t *n_long, SsspPullShared &sh, SsspTally &tally) {
    constexpr int NONE = 0x7F800000;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, sub = lane & ((1 << share) - 1), rows = 32 >> share;
    const int nwarps = (int)(gridDim.x * SSSP_CTA) >> 5;
    const float xmin = sssp_value(low);
    const int *const dist = s.word[c];
    int *const word = s.word[c ^ 1];
    // (neighbouring rows on different SMs: they are heavy together on an R-MAT graph that was not relabelled)
    for (int64_t r0 = (int64_t)(warp * (int)gridDim.x + (int)blockIdx.x) * rows; r0 < d.n; r0 += (int64_t)nwarps * rows) {
        const int64_t r = r0 + (lane >> share);
        int p = 0, e = 0, have = 0, degree = 0;
        float lightest = 0.f;
        if (r < d.n) { p = d.weight_ptr[r]; e = d.weight_ptr[r + 1]; have = __ldcg(dist + r); lightest = d.row_lightest[r]; degree = (int)d.col_degree[r]; }
        float best = sssp_value(have);
        bool walks = p < e && xmin + lightest < best;
        for (int round = 0; round < SSSP_SHARED_ROUNDS && __any_sync(FULL, walks); ++round) {
            const int q = (p & ~3) + 4 * sub;
            uint32_t col[4];
            float w[4] = {0.f, 0.f, 0.f, 0.f};
            int x[4] = {NONE, NONE, NONE, NONE};
            if (walks && q < e) {
                sssp_four<true>(d, q, col, w);
#pragma unroll
                for (int j = 0; j < 4; ++j)
                    if (q + j >= p && q + j < e && xmin + w[j] < best && DBS_CHK_INDEX(d, col[j], d.n)) x[j] = __ldca(dist + col[j]);
            }
            float mine = best;
#pragma unroll
            for (int j = 0; j < 4; ++j) mine = fminf(mine, sssp_value(x[j]) + w[j]);
            for (int o = 1; o < 1 << share; o <<= 1) mine = fminf(mine, __shfl_xor_sync(FULL, mine, o));
            const float last = __shfl_sync(FULL, w[3], lane | ((1 << share) - 1));      // (the largest weight of the round)
            best = mine;
            p = (p & ~3) + (4 << share);
            walks = walks && p < e && sssp_bound<true>(xmin, last) < best;
        }
        if (sub == 0 && r < d.n) {
            const int now = sssp_word(best);
            __stcg(word + r, now);
            if (now < have) {
                atomicOr(next + (r >> 5), 1u << (r & 31));
                ++tally.found; tally.low = min(tally.low, now); tally.edges += degree_of_code((uint32_t)degree);
            }
        }
        const uint32_t left = __ballot_sync(FULL, walks && sub == 0);
        if (left) {
            int4 *longs = sh.longs[warp];
            if (walks && sub == 0) longs[__popc(left & ((1u << lane) - 1u))] = make_int4((int)r, p, e, sssp_word(best));
            __syncwarp();
            sssp_list_long<true>(d, s, longs, __popc(left), xmin, n_long, lane);
            __syncwarp();
        }
    }
}

// The words of the other array are written, all of them; with weights a row has one writer until the chunks, without (payload entries lower it too) they are lowered by atomics.  What is counted of a row (its column's degree) comes with
// the row's own words, 32 rows at a time: fetched where a row ends, a whole warp waits for it in most rounds (2^20 vertices 358 -> 400 us a search), and so it does for a look at the old frontier's
// marks that would spare the words that do not change (358 -> 405).  The distances of the 4 to 32 K columns of the highest degree in shared memory, where 34 to 69 % of the elements lie: nothing
// gained with 4 K of them (before what it costs to bring them there), slower with more -- what they take from the L1 are the lines that the other gathers wait in.
template <int DT>
__device__ void sssp_pull(const Device &d, const SsspState &s, int c, const uint32_t *F, uint32_t *next, int low, bool below_zero, int32_t *n_long, SsspPullShared &sh, SsspTally &tally) {
    constexpr bool VAL = DT != DBSPMSPV_PATTERN;
    constexpr int NONE = 0x7F800000;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int gwarp = (int)(blockIdx.x * SSSP_CTA + threadIdx.x) >> 5, nwarps = (int)(gridDim.x * SSSP_CTA) >> 5;
    const uint32_t lt = (1u << lane) - 1u;
    const float xmin = sssp_value(low);
    const int *const dist = s.word[c];
    int *const word = s.word[c ^ 1];
    const int32_t *ptr = VAL ? d.weight_ptr : d.rowrun_ptr;
    auto bound = [&](float w) { return sssp_bound<VAL>(xmin, w); };
    // The thread block's groups of rows, spread over the matrix, are taken by its warps in turn.  (On an R-MAT graph that was not relabelled neighbouring rows are
    // heavy together, and so are rows with the same low bits: group i of block b is number b + i of the i-th stretch.  Groups dealt out by the elements they hold,
    // the heaviest first, from a table: no gain there, 5 % longer on graphs in scattered order.)
    const int n_groups = (int)((d.n + 31) / 32), per_block = (n_groups + (int)gridDim.x - 1) / (int)gridDim.x;
    if (threadIdx.x == 0) sh.cursor = 0;
    __syncthreads();
    int4 *queue = sh.queue[warp], *longs = sh.longs[warp];
    int *queue_degree = sh.queue_degree[warp];
    int row_g = 0, p_g = 0, e_g = 0, have_g = 0;       // a row of the next group
    uint32_t code_g = 0u;
    float w_g = 1.0f;
    bool more = true;
    auto fetch = [&]() {
        int i = 0;
        if (lane == 0) i = atomicAdd(&sh.cursor, 1);
        i = __shfl_sync(FULL, i, 0);
        more = i < per_block;
        if (!more) return;
        const int64_t g = (int64_t)i * gridDim.x + (blockIdx.x + i) % gridDim.x, r = g * 32 + lane;
        row_g = (int)(r < d.n ? r : d.n); p_g = 0; e_g = 0; have_g = 0;
        if (r < d.n) { p_g = ptr[r]; e_g = ptr[r + 1]; have_g = __ldcg(dist + r); if (VAL) { w_g = d.row_lightest[r]; code_g = d.col_degree[r]; } }
    };
    fetch();
    int head = 0, cnt = 0, n_listed = 0;
    int row = -1, p = 0, e = 0, q_long = 0;            // the row being walked: elements [p, e), from q_long on it is long
    float have = 0.f, best = __int_as_float(NONE);     // its distance before the step, and now
    int degree = 0;
    for (;;) {
        while (more && cnt < 32) {                     // (no more than that: what a warp has claimed no other one can take)
            const bool pass = p_g < e_g && sssp_word(xmin + w_g) < have_g;
            const uint32_t m = __ballot_sync(FULL, pass);
            if (pass) {
                const int at = (head + cnt + __popc(m & lt)) & 63;
                queue[at] = make_int4(row_g, p_g, e_g, have_g);
                if (VAL) queue_degree[at] = (int)degree_of_code(code_g);
            }
            if (row_g < d.n) {                         // (what the row's walk finds comes on top, from this warp too)
                if (VAL) __stcg(word + row_g, have_g); else atomicMin(word + row_g, have_g);
            }
            cnt += __popc(m);
            fetch();
        }
        __syncwarp();
        const uint32_t idle = __ballot_sync(FULL, row < 0);
        if (idle == FULL && cnt == 0) break;
        if (idle && cnt) {
            const int k = __popc(idle & lt);
            if (row < 0 && k < cnt) {
                const int4 q = queue[(head + k) & 63];
                row = q.x; p = q.y; e = q.z; have = best = sssp_value(q.w); q_long = (p & ~3) + SSSP_ROUNDS * 4;
                if (VAL) degree = queue_degree[(head + k) & 63];
            }
            const int took = min(__popc(idle), cnt);
            head += took; cnt -= took;
        }
        bool left = false;                             // a long row: what has been found so far counts, the rest is listed
        if (row >= 0) {
            // (a row that was never reached needs several rounds: two groups at a time until something is found)
            uint32_t col[8];
            float w[8];
            int x[8];
            const int q0 = p & ~3;
            const bool two = best == __int_as_float(NONE) && q0 + 4 < e;
            sssp_four<VAL>(d, q0, reinterpret_cast<uint32_t (&)[4]>(col[0]), reinterpret_cast<float (&)[4]>(w[0]));
            if (two) sssp_four<VAL>(d, q0 + 4, reinterpret_cast<uint32_t (&)[4]>(col[4]), reinterpret_cast<float (&)[4]>(w[4]));
#pragma unroll
            for (int j = 0; j < 8; ++j) {
                x[j] = NONE;
                const bool go = (j < 4 || two) && q0 + j >= p && q0 + j < e && xmin + w[j] < best;
                if (go && DBS_CHK_INDEX(d, col[j], d.n)) x[j] = __ldca(dist + col[j]);
            }
            float last = w[3];
            if (VAL && below_zero)
#pragma unroll
                for (int j = 0; j < 8; ++j) x[j] = __float_as_int(sssp_value(x[j]));
#pragma unroll
            for (int j = 0; j < 8; ++j)
                if (j < 4 || two) { best = fminf(best, __int_as_float(x[j]) + w[j]); last = w[j]; }
            p = q0 + (two ? 8 : 4);
            const bool over = p >= e || !(bound(last) < best);
            left = !over && p >= q_long;
            if ((over || left) && best < have) {
                const int now = sssp_word(best);
                if (VAL) {
                    __stcg(word + row, now);
                    atomicOr(next + (row >> 5), 1u << (row & 31));
                    ++tally.found; tally.low = min(tally.low, now); tally.edges += (unsigned)degree;
                } else sssp_lower(d, word, next, row, now, sssp_word(have), tally);
            }
            if (over) row = -1;
        }
        const uint32_t lm = __ballot_sync(FULL, left);
        if (lm) {
            if (n_listed + __popc(lm) > 32) { __syncwarp(); sssp_list_long<VAL>(d, s, longs, n_listed, xmin, n_long, lane); n_listed = 0; __syncwarp(); }
            if (left) { longs[n_listed + __popc(lm & lt)] = make_int4(row, p, e, sssp_word(best)); row = -1; }
            n_listed += __popc(lm);
        }
    }
    __syncwarp();
    if (n_listed) sssp_list_long<VAL>(d, s, longs, n_listed, xmin, n_long, lane);
    if (VAL) return;
    // entries with a payload (unit weights): one block per warp at a time, columns of the frontier only (the blocks sit where a power-law graph is dense, among
    // the vertices that settle first: late large steps skip most of them); the next entry is fetched meanwhile
    struct Entry { uint32_t idx, w, aux; int rb; };
    auto entry = [&](int pos) {
        Entry e{0u, 0u, 0u, 0};
        if (pos >= 0 && DBS_CHK_INDEX(d, pos, d.n_entries)) {
            e = Entry{d.csr.idx[pos], d.csr.w[pos], d.csr.aux[pos], d.entry_row[pos]};
            DBS_CHK_ENTRY(d, true, e.idx, e.w, e.aux);
        }
        return e;
    };
    auto position = [&](int q) { return q < d.n_payload ? d.payload_pos[q] : -1; };
    Entry ahead = entry(position(gwarp));
    int pos = position(gwarp + nwarps);
    for (int q = gwarp; q < d.n_payload; q += nwarps) {
        const Entry e = ahead;
        ahead = entry(pos);
        pos = position(q + 2 * nwarps);
        const int type = (int)(e.idx >> TYPE_SHIFT), cb = (int)(e.idx & IDX_MASK);
        if (type == DBSPMSPV_BLK_INLINE || !DBS_CHK_INDEX(d, e.rb, d.mb)) continue;      // (only a replaced entry is INLINE here; warp-uniform)
        const uint32_t xm = mask_of(F, cb);
        if (!xm) continue;                                                               // warp-uniform
        block_rows_min_warp<DT>(type, e.w, e.aux, xm, reinterpret_cast<const float *>(dist) + (size_t)cb * 16, d.payload, lane, [&](int r, uint32_t key) {
            const int v = sssp_word(minplus_value(key)), row = e.rb * 16 + r, had = __ldcg(dist + row);
            if (v < had) sssp_lower(d, word, next, row, v, had, tally);
        });
    }
}

// The listed chunks of long rows, a warp per chunk, four elements per lane and step.  The next chunk's record, best and first elements are
// fetched while this one's distances arrive.
template <int DT>
__device__ void sssp_pull_long(const Device &d, const SsspState &s, int c, uint32_t *next, int low, int n, SsspTally &tally) {
    constexpr bool VAL = DT != DBSPMSPV_PATTERN;
    constexpr int NONE = 0x7F800000;
    const int lane = threadIdx.x & 31;
    const int gwarp = (int)(blockIdx.x * SSSP_CTA + threadIdx.x) >> 5, nwarps = (int)(gridDim.x * SSSP_CTA) >> 5;
    const float xmin = sssp_value(low);
    const int *const dist = s.word[c];
    int *const word = s.word[c ^ 1];
    auto record = [&](int i) { return i < n ? __ldcg(s.chunks + i) : make_int4(0, 0, 0, 0); };
    int4 now_c = record(gwarp), ahead = record(gwarp + nwarps);
    uint32_t col[4] = {0u, 0u, 0u, 0u};
    float w[4] = {0.f, 0.f, 0.f, 0.f};
    int had = 0;
    auto first = [&](const int4 &r) {
        const int k0 = (r.y & ~3) + 4 * lane;
        if (k0 < r.z) { had = __ldcg(word + r.x); sssp_four<VAL>(d, k0, col, w); }
    };
    first(now_c);
    for (int i = gwarp; i < n; i += nwarps) {
        had = __shfl_sync(FULL, had, 0);               // (lane 0 of a chunk always has elements)
        const int start = had, row = now_c.x, p = now_c.y, e = now_c.z;
        int now = had;
        for (int q = (p & ~3) + 4 * lane;; q += 128) {
            const float best = sssp_value(now);
            float wq[4];
            int x[4];
            const bool in = q < e, more = q - 4 * lane + 128 < e;             // (warp-uniform: the chunk goes on)
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                x[j] = NONE;
                wq[j] = w[j];
                const bool go = in && q + j >= p && q + j < e && xmin + w[j] < best;
                if (go && DBS_CHK_INDEX(d, col[j], d.n)) x[j] = __ldca(dist + col[j]);
            }
            if (more) { if (q + 128 < e) sssp_four<VAL>(d, q + 128, col, w); }
            else { now_c = ahead; ahead = record(i + 2 * nwarps); first(now_c); }
            float mine = best;
            if (in)
#pragma unroll
                for (int j = 0; j < 4; ++j) mine = fminf(mine, sssp_value(x[j]) + wq[j]);
            now = __reduce_min_sync(FULL, sssp_word(mine));
            if (!more) break;
            const bool over = !(sssp_bound<VAL>(xmin, wq[3]) < sssp_value(now));
            if (__shfl_sync(FULL, (int)over, 31)) {    // (the last lane's weight is the largest of the step)
                now_c = ahead; ahead = record(i + 2 * nwarps); first(now_c);
                break;
            }
        }
        if (lane == 0 && now < start) {
            // (a row of several chunks is counted by the one that marks it)
            const uint32_t bit = 1u << (row & 31);
            atomicMin(word + row, now);
            tally.low = min(tally.low, now);
            if (!(atomicOr(next + (row >> 5), bit) & bit)) { ++tally.found; tally.edges += sssp_degree(d, row); }
        }
    }
}

constexpr int SSSP_SMEM = (int)(sizeof(SsspShared) > sizeof(SsspPullShared) ? sizeof(SsspShared) : sizeof(SsspPullShared));
static_assert(sizeof(SsspListShared) <= sizeof(SsspShared), "the phases share one allocation");
// The arguments stay in the constant bank: the lists and bitmaps are taken by the step's number, for which every thread kept a copy of its own in local memory, that
// spilled more besides (then 216 -> 88 bytes of stack, 144 by now; R-MAT 300 K / 500 K / 2^20 vertices 242 / 252 / 359 -> 222 / 227 / 331 us a search, in scattered order 202 / 237 / 333 -> 186 / 217 / 306; 27-point
// operator on 90^3 cells, an inner source, 3029 -> 2947).  The phases as functions of their own, which share no registers: 233 / 239 / 343 us.  No phase holds the spills alone (each of them left out takes at most 40 of 120
// bytes away): a kernel without the rows shared among lanes needs 120 all the same, and with what a row's walk keeps moved to shared memory large searches were up to 4 % longer.
template <int DT>
__global__ void __launch_bounds__(SSSP_CTA, 1) k_sssp(const __grid_constant__ Device d, const __grid_constant__ SsspState s, int32_t src, float *dist_out, int start, int max_steps, unsigned pull_edges, unsigned late_edges) {
    namespace cg = cooperative_groups;
    extern __shared__ __align__(16) uint8_t s_dyn[];
    __shared__ SsspSums sums;
    SsspShared &sh = *reinterpret_cast<SsspShared *>(s_dyn);
    cg::grid_group grid = cg::this_grid();
    const int tid = blockIdx.x * SSSP_CTA + threadIdx.x, nthreads = gridDim.x * SSSP_CTA;
    if (start == SSSP_STARTS) {                        // (a later launch of the same search continues where the one before stopped)
        const int64_t n = (int64_t)s.n_words * 32;
        for (int64_t v = tid; v < n; v += nthreads) s.word[0][v] = s.word[1][v] = v == src ? 0 : 0x7F800000;
        for (int k = tid; k < s.n_words; k += nthreads) { s.bits[0][k] = k == src >> 5 ? 1u << (src & 31) : 0u; s.bits[1][k] = 0u; }       // (the third is cleared by the first step)
        if (tid == 0) {
            int first, deg;
            column_run(d, src, first, deg);
            for (int k = 0; k < 5; ++k) s.ctr[k] = 0;
            for (int k = 0; k < 3; ++k) s.set[k] = SsspSet{k == 0 ? (unsigned)deg : 0u, k == 0 ? 1u : 0u, k == 0 ? 0 : 0x7F800000, 0};
            s.list[1][0] = src;
        }
        grid.sync();
    }
    auto read = [&](int k) {
        const int4 v = __ldcg(reinterpret_cast<const int4 *>(s.set + k));
        return SsspSet{(unsigned)v.x, (unsigned)v.y, v.z, v.w};
    };
    int t = __ldcg(s.ctr), c = __ldcg(s.ctr + 1);      // array c holds the distances; so does the other one, but for the frontier, of which it has larger ones
    bool late = (start & SSSP_LATE) != 0;              // a step has been pulled, in this launch or one before
    constexpr bool VAL = DT != DBSPMSPV_PATTERN;
    bool below_zero = VAL && (start & SSSP_BELOW_ZERO);      // a distance has been below zero, likewise: its word is not its bits
    bool lists = start == SSSP_STARTS;                 // the step before listed what it marked, in list[(t + 1) & 1]
    SsspSet now = read(t % 3);                         // grid-uniform, as all that is decided from it
    for (int made = 0; made < max_steps && now.found; ++made, ++t, c ^= 1) {
        const uint32_t *F = s.bits[t % 3];
        uint32_t *N = s.bits[(t + 1) % 3], *Z = s.bits[(t + 2) % 3];
        const int nxt = (t + 1) % 3;
        int32_t *n_long = &s.set[nxt].n_long, *n_list = s.ctr + 2 + t % 3;
        const bool listed = lists && now.found <= SSSP_LIST, pulled = now.edges > (late ? late_edges : pull_edges);
        late = late || pulled;
        if (VAL) below_zero = below_zero || now.low < 0;
        lists = !pulled && now.edges <= SSSP_LIST_EDGES;
        if (tid == 0) { s.ctr[2 + nxt] = 0; s.set[(t + 2) % 3] = SsspSet{0u, 0u, 0x7F800000, 0}; }      // (their last readers were the steps t - 2 and t - 1)
        const SsspNext next{s.word[c], s.word[c ^ 1], N, lists ? s.list[t & 1] : nullptr, n_list};
        SsspTally tally;
        const int share = DT != DBSPMSPV_PATTERN ? sssp_row_share(d.n, nthreads) : 0;
        if (pulled && share) sssp_pull_shared(d, s, c, N, share, now.low, n_long, *reinterpret_cast<SsspPullShared *>(s_dyn), tally);
        else if (pulled) sssp_pull<DT>(d, s, c, F, N, now.low, below_zero, n_long, *reinterpret_cast<SsspPullShared *>(s_dyn), tally);
        else if (listed) sssp_expand_list<DT>(d, s.list[(t + 1) & 1], (int)now.found, next, *reinterpret_cast<SsspListShared *>(s_dyn), tally);
        else sssp_expand<DT>(d, s, F, next, n_long, sh, tally);
        for (int k = tid; k < s.n_words; k += nthreads) Z[k] = 0u;
        sssp_count(s, sums, nxt, tally);
        grid.sync();
        const int low = now.low;
        now = read(nxt);
        if (now.n_long > 0) {                          // chunks of long runs or rows
            SsspTally more;
            if (pulled) sssp_pull_long<DT>(d, s, c, N, low, now.n_long, more);
            else sssp_long<DT>(d, next, now.n_long, more);
            sssp_count(s, sums, nxt, more);
            grid.sync();
            now = read(nxt);
        }
    }
    // the distances themselves
    for (int64_t v = tid; v < d.n; v += nthreads) dist_out[v] = sssp_value(__ldcg(s.word[c] + v));
    // (everyone read the counters before the first barrier, or leaves without a step)
    if (tid == 0) { s.ctr[0] = t; s.ctr[1] = c; s.report[0] = t; s.report[1] = (int)now.found; s.report[2] = (late ? SSSP_LATE : 0) | (below_zero ? SSSP_BELOW_ZERO : 0); }
}

}  // namespace dbs

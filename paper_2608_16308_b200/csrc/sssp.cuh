// db_sssp on hypersparse handles: the whole search in one cooperative launch, no accumulator and no sparse vectors in between.
//
// The search is the synchronous iteration of (min, +) products: step t relaxes the out-edges of the
// vertices whose distance improved in step t - 1, with the distances they had at the end of that step.  As a host loop over
// dbspmspv_run it paid, per step, a blocking of x, an accumulator that was filled and compacted, a relaxation pass and a
// round trip to the host (R-MAT scale 20: 9 steps, 1.17 ms, of which 0.2 ms an idle GPU).  Here a step is
//   expand   the columns of the frontier (a bitmap) laid end to end per thread block as in the direct push (push_direct.cuh); a candidate
//            distance goes straight into the target's word with an atomic minimum, and the thread whose atomic lowered
//            it marks the target in the next frontier;
//   long     the listed long runs and payload runs, a warp per chunk (only if there are any);
//   settle   the marked vertices copy their word into the caller's distances -- the values the next
//            step starts from, which no one lowers meanwhile -- and are counted;
// with a grid barrier after each.  A step finds the same improvements, distance for distance, as the product did: `word`
// holds the minimum over everything seen so far, a vertex is marked iff its word went below the distance it had before the step.
//
// What bounds a large step is the gather of one target word per edge.  It goes through L1 first (a stale word is never too small,
// so a candidate that does not beat it is done); only a candidate that does looks at L2, and only one that beats that too pays an atomic:
// the words of hub rows, which thousands of edges reach, settle after a few atomics.
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
// A step whose frontier reaches more than this share of the stored elements is pulled.  Shares of 2 / 5 / 10 / 20 %: symmetrised R-MAT scale 20,
// three sources, 559 - 661 / 561 - 670 / 571 - 664 / 575 - 665 us a search, with its vertices in scattered order 354 - 415 / 355 - 415 / 316 - 372 / 353 - 372;
// scale 17 within 7 % of each other.
constexpr float SSSP_PULL_SHARE = 0.05f;
constexpr int SSSP_ROUNDS = 8;                    // rounds of four elements that a lane walks of a row
constexpr int SSSP_CHUNK = 512;                   // elements of a listed chunk of a longer row
constexpr int SSSP_MAX_STEPS = 1024;              // steps of one launch, at most: a cycle of negative weight ends on the host

struct SsspState {
    int *word;                // n: ordered words of the smallest distance seen
    uint32_t *bits[2];        // frontiers of alternating steps, one bit per vertex
    int32_t *ctr;             // [0..2] vertices of the frontier, [3..5] listed chunks (sets rotate by step), [6] steps made
    int *low;                 // smallest word of the frontier, rotating with the counters
    unsigned long long *edges;   // out-edges of the frontier in INLINE runs, likewise
    int4 *chunks;             // {row, first, end, -} of the listed chunks of long rows
    int32_t *report;          // page-locked host words: steps made, vertices of the frontier that was left
    int32_t n_words;
};

// ordered(v): monotone in v, and the bits themselves where v >= 0
__device__ __forceinline__ int sssp_word(float v) { return ordered_word(__float_as_int(v)); }
__device__ __forceinline__ float sssp_value(int w) { return __int_as_float(ordered_word(w)); }

struct SsspShared {
    unsigned long long edges[SSSP_WARPS];
    int pre[SSSP_COLS + 1];                       // elements before a column of the round
    int2 run[SSSP_COLS];                          // position of its first entry minus that; its distance
    uint16_t own[SSSP_COLS * PD_LONG / 32];       // column that owns the first element of a step of 32
    int cnt[SSSP_WARPS], sum[SSSP_WARPS], rec[SSSP_WARPS], base;
};

// The candidates of up to U targets per lane (target < 0: none).
template <int U>
__device__ __forceinline__ void sssp_relax(const SsspState &s, uint32_t *next, const int (&target)[U], const float (&cand)[U]) {
    int seen[U];
#pragma unroll
    for (int u = 0; u < U; ++u) seen[u] = target[u] >= 0 ? __ldca(s.word + target[u]) : 0;
#pragma unroll
    for (int u = 0; u < U; ++u) {
        if (target[u] < 0) continue;
        const int c = sssp_word(cand[u]);
        if (c >= seen[u] || c >= __ldcg(s.word + target[u])) continue;
        if (c < atomicMin(s.word + target[u], c)) atomicOr(next + (target[u] >> 5), 1u << (target[u] & 31));
    }
}

template <int DT>
__device__ void sssp_expand(const Device &d, const SsspState &s, const float *dist, const uint32_t *F, uint32_t *next, int32_t *n_long, SsspShared &sh) {
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
                if ((listed >> k) & 1u) { first[k] = c[k]; deg[k] = c[k + 1] - c[k]; xv[k] = __ldcg(dist + j0 + k); if (!DBS_CHK_RANGE(d, first[k], deg[k])) deg[k] = 0; }
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
            sssp_relax<SSSP_ILP>(s, next, target, cand);
        }
        __syncthreads();                               // (the next round overwrites the layout)
    }
}

template <int DT>
__device__ void sssp_long(const Device &d, const SsspState &s, uint32_t *next, int n) {
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
        sssp_relax<U>(s, next, target, cand);
    }
}

// A row's new best.
__device__ __forceinline__ void sssp_lower(const SsspState &s, uint32_t *next, int row, int best) {
    if (best < atomicMin(s.word + row, best)) atomicOr(next + (row >> 5), 1u << (row & 31));
}
// Elements k0 .. k0 + 3 (k0 a multiple of four) of the runs: columns and weights.
template <bool VAL>
__device__ __forceinline__ void sssp_four(const Device &d, int k0, uint32_t (&col)[4], float (&w)[4]) {
    if (VAL) {
        const uint4 a = __ldcs(reinterpret_cast<const uint4 *>(d.weightrun + k0)), b = __ldcs(reinterpret_cast<const uint4 *>(d.weightrun + k0 + 2));
        col[0] = a.x; w[0] = __uint_as_float(a.y); col[1] = a.z; w[1] = __uint_as_float(a.w);
        col[2] = b.x; w[2] = __uint_as_float(b.y); col[3] = b.z; w[3] = __uint_as_float(b.w);
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
__device__ __forceinline__ int sssp_bound(float xmin, float w) {
    constexpr int least = (int)0x807FFFFFu;        // sssp_word(-infinity)
    return sssp_word(xmin + (VAL ? sssp_value(max(sssp_word(w) & ~((1 << (32 - SSSP_WEIGHT_BITS)) - 1), least)) : w));
}

// A large step pulled.  Every row walks its own elements, which lie by weight (Device::weightrun), and stops at the first that
// cannot improve it: smallest distance of the frontier + weight >= the row's best.  In the late large steps of an R-MAT search that leaves a
// seventh of the elements, and a row reached for the first time soon has a best of its own.  Columns outside the
// frontier improve nothing (their edges were relaxed when they entered it), so they need no test.
// A lane walks the rows of its own, four elements (one 32-byte sector) a round, row after row, the next row's place fetched meanwhile; what is left of a row that has not
// stopped after SSSP_ROUNDS rounds is listed in chunks, which all warps share out behind a grid barrier (walked by the warp that met them, the
// hub rows of an R-MAT graph, neighbours all, took one warp 300 us).  Handles of unit weights walk the row-run index.
template <int DT>
__device__ void sssp_pull(const Device &d, const SsspState &s, const float *dist, const uint32_t *F, uint32_t *next, int low, int32_t *n_long) {
    constexpr bool VAL = DT != DBSPMSPV_PATTERN;
    constexpr int NONE = 0x7F800000;
    const int lane = threadIdx.x & 31;
    const int gwarp = (int)(blockIdx.x * SSSP_CTA + threadIdx.x) >> 5, nwarps = (int)(gridDim.x * SSSP_CTA) >> 5;
    const float xmin = sssp_value(low);
    auto lower = [&](int row, int best) { sssp_lower(s, next, row, best); };
    auto bound = [&](float w) { return sssp_bound<VAL>(xmin, w); };
    // Up to 32 groups of 32 rows per warp, spread over the matrix: on an R-MAT graph that was not relabelled neighbouring rows are heavy together
    // (a warp that took eight neighbouring groups of hubs: 136 us where the step takes 60).
    const int n_groups = (int)((d.n + 31) / 32);
    for (int64_t g0 = gwarp; g0 < n_groups; g0 += 32ll * nwarps) {
        int k = 0, row = -1, p = 0, e = 0, have = 0, best = NONE, q_long = 0;      // the row being walked: elements [p, e), from q_long on it is long
        int k_row = 0, k_n = 0, row_n = -1, p_n = 0, e_n = 0, have_n = 0;                              // the next one
        uint32_t longm = 0u;
        int n_chunks = 0;
        // (row lane + k mod 32 of the k-th group, so that no lane gets the heavy rows of every group)
        auto fetch = [&]() {
            row_n = -1;
            if (k < 32 && g0 + (int64_t)k * nwarps < n_groups) {
                const int64_t r = (g0 + (int64_t)k * nwarps) * 32 + ((lane + k) & 31);
                k_n = k;
                if (r < d.n) { row_n = (int)r; p_n = d.rowrun_ptr[r]; e_n = d.rowrun_ptr[r + 1]; have_n = __ldcg(s.word + r); }
                else row_n = -2;                       // no such row, but the walk goes on
                ++k;
            }
        };
        fetch();
        while (__any_sync(FULL, row >= 0 || row_n != -1)) {
            if (row < 0 && row_n != -1) {
                row = row_n; k_row = k_n; p = p_n; e = e_n; have = have_n; best = have_n; q_long = (p & ~3) + SSSP_ROUNDS * 4;
                if (row < 0 || p >= e) row = -1;
                fetch();
            }
            if (row >= 0) {
                // (a row that was never reached needs several rounds: two groups at a time until something is found)
                uint32_t col[8];
                float w[8], x[8];
                const int q0 = p & ~3;
                const bool two = best == NONE && q0 + 4 < e;
                sssp_four<VAL>(d, q0, reinterpret_cast<uint32_t (&)[4]>(col[0]), reinterpret_cast<float (&)[4]>(w[0]));
                if (two) sssp_four<VAL>(d, q0 + 4, reinterpret_cast<uint32_t (&)[4]>(col[4]), reinterpret_cast<float (&)[4]>(w[4]));
#pragma unroll
                for (int j = 0; j < 8; ++j) {
                    x[j] = __int_as_float(NONE);
                    if ((j < 4 || two) && q0 + j >= p && q0 + j < e && sssp_word(xmin + w[j]) < best && DBS_CHK_INDEX(d, col[j], d.n)) x[j] = __ldca(dist + col[j]);
                }
                float last = w[3];
#pragma unroll
                for (int j = 0; j < 8; ++j)
                    if (j < 4 || two) { best = min(best, sssp_word(x[j] + w[j])); last = w[j]; }
                p = q0 + (two ? 8 : 4);
                if (p >= e || bound(last) >= best) { if (best < have) lower(row, best); row = -1; }
                else if (p >= q_long) {     // a long row: what has been found so far counts, the rest below
                    if (best < have) lower(row, best);
                    longm |= 1u << k_row;
                    n_chunks += (e - q_long + SSSP_CHUNK - 1) / SSSP_CHUNK;
                    row = -1;
                }
            }
        }
        if (__any_sync(FULL, n_chunks > 0)) {
            int incl = n_chunks;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) { const int t = __shfl_up_sync(FULL, incl, o); if (lane >= o) incl += t; }
            int base = 0;
            if (lane == 31) base = atomicAdd(n_long, incl);
            int at = __shfl_sync(FULL, base, 31) + incl - n_chunks;
            for (; longm; longm &= longm - 1) {
                const int kk = __ffs(longm) - 1;
                const int r = (int)((g0 + (int64_t)kk * nwarps) * 32 + ((lane + kk) & 31)), end = d.rowrun_ptr[r + 1];
                for (int q = (d.rowrun_ptr[r] & ~3) + SSSP_ROUNDS * 4; q < end; q += SSSP_CHUNK) s.chunks[at++] = make_int4(r, q, min(end, q + SSSP_CHUNK), 0);
            }
        }
    }
    // entries with a payload: one block per warp at a time, columns of the frontier only (the blocks sit where a power-law graph is dense, among
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
        block_rows_min_warp<DT>(type, e.w, e.aux, xm, dist + (size_t)cb * 16, d.payload, lane, [&](int r, uint32_t key) {
            const int c = sssp_word(minplus_value(key)), row = e.rb * 16 + r;
            if (c < __ldcg(s.word + row)) lower(row, c);
        });
    }
}

// The listed chunks of long rows, a warp per chunk, four elements per lane and step.
template <int DT>
__device__ void sssp_pull_long(const Device &d, const SsspState &s, const float *dist, uint32_t *next, int low, int n) {
    constexpr bool VAL = DT != DBSPMSPV_PATTERN;
    const int lane = threadIdx.x & 31;
    const int gwarp = (int)(blockIdx.x * SSSP_CTA + threadIdx.x) >> 5, nwarps = (int)(gridDim.x * SSSP_CTA) >> 5;
    const float xmin = sssp_value(low);
    int4 ahead = gwarp < n ? __ldcg(s.chunks + gwarp) : make_int4(0, 0, 0, 0);
    for (int i = gwarp; i < n; i += nwarps) {
        const int4 c = ahead;
        if (i + nwarps < n) ahead = __ldcg(s.chunks + i + nwarps);
        const int had = __ldcg(s.word + c.x);
        int now = had;
        uint32_t col[4], col_n[4];
        float w[4], w_n[4];
        const int k0 = c.y + 4 * lane;
        if (k0 < c.z) sssp_four<VAL>(d, k0, col, w);
        for (int q = k0; q - 4 * lane < c.z; q += 128) {
            if (q + 128 < c.z) sssp_four<VAL>(d, q + 128, col_n, w_n);
            float x[4];
            int mine = now;
            bool over = true;
            if (q < c.z) {
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    x[j] = __int_as_float(0x7F800000);
                    if (q + j < c.z && sssp_word(xmin + w[j]) < now && DBS_CHK_INDEX(d, col[j], d.n)) x[j] = __ldca(dist + col[j]);
                }
#pragma unroll
                for (int j = 0; j < 4; ++j) mine = min(mine, sssp_word(x[j] + w[j]));
            }
            now = __reduce_min_sync(FULL, mine);
            if (q < c.z) over = sssp_bound<VAL>(xmin, w[3]) >= now;
            if (__shfl_sync(FULL, (int)over, 31)) break;               // (the last lane's weight is the largest of the step; past the end: done)
#pragma unroll
            for (int j = 0; j < 4; ++j) { col[j] = col_n[j]; w[j] = w_n[j]; }
        }
        if (lane == 0 && now < had) sssp_lower(s, next, c.x, now);
    }
}

template <int DT>
__global__ void __launch_bounds__(SSSP_CTA, 1) k_sssp(Device d, SsspState s, int32_t src, float *dist, int start, int max_steps, unsigned long long pull_edges) {
    namespace cg = cooperative_groups;
    extern __shared__ __align__(16) uint8_t s_dyn[];
    SsspShared &sh = *reinterpret_cast<SsspShared *>(s_dyn);
    cg::grid_group grid = cg::this_grid();
    const int tid = blockIdx.x * SSSP_CTA + threadIdx.x, nthreads = gridDim.x * SSSP_CTA, lane = threadIdx.x & 31;
    if (start) {                                       // (a later launch of the same search continues where the one before stopped)
        const int64_t n = d.n;
        for (int64_t v = tid; v < n; v += nthreads) { s.word[v] = v == src ? 0 : 0x7F800000; dist[v] = v == src ? 0.0f : __int_as_float(0x7F800000); }
        for (int k = tid; k < s.n_words; k += nthreads) { s.bits[0][k] = k == src >> 5 ? 1u << (src & 31) : 0u; s.bits[1][k] = 0u; }
        if (tid < 6) s.ctr[tid] = tid == 0 ? 1 : 0;
        if (tid == 6) { s.ctr[6] = 0; for (int k = 0; k < 3; ++k) { s.low[k] = k == 0 ? 0 : 0x7F800000; s.edges[k] = 0ull; } }
        grid.sync();
    }
    int t = s.ctr[6];
    for (int made = 0; made < max_steps && __ldcg(s.ctr + t % 3) != 0; ++made, ++t) {
        uint32_t *F = s.bits[t & 1], *next = s.bits[(t + 1) & 1];
        int32_t *n_long = s.ctr + 3 + t % 3;
        if (tid == 0) s.ctr[3 + (t + 1) % 3] = 0;      // (its last reader was step t - 2)
        if (__ldcg(s.edges + t % 3) > pull_edges) {    // grid-uniform
            const int low = __ldcg(s.low + t % 3);
            sssp_pull<DT>(d, s, dist, F, next, low, n_long);
            grid.sync();
            const int n = __ldcg(n_long);
            if (n > 0) {                               // grid-uniform
                sssp_pull_long<DT>(d, s, dist, next, low, n);
                grid.sync();
            }
        } else {
            sssp_expand<DT>(d, s, dist, F, next, n_long, sh);
            grid.sync();
            const int n = __ldcg(n_long);
            if (n > 0) {                               // grid-uniform
                sssp_long<DT>(d, s, next, n);
                grid.sync();
            }
        }
        if (tid == 0) { s.ctr[(t + 2) % 3] = 0; s.low[(t + 2) % 3] = 0x7F800000; s.edges[(t + 2) % 3] = 0ull; }
        int found = 0, low = 0x7F800000;
        unsigned long long edges = 0;
        const int gwarp = tid >> 5, nwarps = nthreads >> 5;
        for (int w0 = gwarp; w0 < s.n_words; w0 += 8 * nwarps) {
            uint32_t b[8];
            int v[8], deg[8];
#pragma unroll
            for (int q = 0; q < 8; ++q) { const int w = w0 + q * nwarps; b[q] = w < s.n_words ? __ldcg(next + w) : 0u; }
#pragma unroll
            for (int q = 0; q < 8; ++q) {
                v[q] = 0x7F800000; deg[q] = 0;
                if ((b[q] >> lane) & 1u) {
                    const int j = (w0 + q * nwarps) * 32 + lane;
                    v[q] = __ldcg(s.word + j);
                    const int32_t *cp = d.csc.colptr + 17 * (j >> 4) + (j & 15);
                    deg[q] = cp[1] - cp[0];
                }
            }
#pragma unroll
            for (int q = 0; q < 8; ++q) {
                const int w = w0 + q * nwarps;
                if (w >= s.n_words) break;
                if ((b[q] >> lane) & 1u) dist[(int64_t)w * 32 + lane] = sssp_value(v[q]);
                if (lane == 0) F[w] = 0u;
                found += __popc(b[q]);
                low = min(low, v[q]);
                edges += (unsigned)deg[q];
            }
        }
        low = __reduce_min_sync(FULL, low);
#pragma unroll
        for (int o = 16; o; o >>= 1) edges += __shfl_xor_sync(FULL, edges, o);
        if (lane == 0) { sh.cnt[threadIdx.x >> 5] = found; sh.sum[threadIdx.x >> 5] = low; sh.edges[threadIdx.x >> 5] = edges; }
        __syncthreads();
        if (threadIdx.x < 32) {
            found = __reduce_add_sync(FULL, sh.cnt[lane]);
            low = __reduce_min_sync(FULL, sh.sum[lane]);
            edges = sh.edges[lane];
#pragma unroll
            for (int o = 16; o; o >>= 1) edges += __shfl_xor_sync(FULL, edges, o);
            if (lane == 0 && found) { atomicAdd(s.ctr + (t + 1) % 3, found); atomicMin(s.low + (t + 1) % 3, low); atomicAdd(s.edges + (t + 1) % 3, edges); }
        }
        grid.sync();
    }
    // (everyone read ctr[6] before the first barrier, or leaves without a step)
    if (tid == 0) { s.ctr[6] = t; s.report[0] = t; s.report[1] = __ldcg(s.ctr + t % 3); }
}

}  // namespace dbs

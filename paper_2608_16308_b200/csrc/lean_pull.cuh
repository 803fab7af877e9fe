// Streaming pull for hypersparse handles (Sections 3.3.2, 3.3.3): almost every stored element of
// such a matrix is an INLINE entry of the block-CSR view, and that view keeps the elements of a
// row adjacent, so y = A x is a segmented sum over one stream.
//
//   * The view is cut into chunks of LEAN_CHUNK consecutive entries, whatever row they belong to
//     (equal bytes per chunk: no weights, no segment table).  A lane reads its eight entries of
//     a chunk with 16-byte streaming loads, and the loads of the warp's NEXT chunk are issued
//     before the current one is worked on: the registers are the staging buffer (Section 3.3.3's
//     double buffering), which leaves the shared memory to the filter below and the rest of the
//     SM's on-chip memory to the L1 that serves the hot columns of a power-law matrix.
//   * One thread block per SM keeps the presence bitmap of x (the vector-block masks, one bit per
//     column) in shared memory and tests it before every gather: an absent x_j costs a
//     shared-memory load instead of a trip through the L1 tag stage, which is what bounds this
//     kernel (one 4-byte gather per stored element, one cache line each).
//   * A warp pass covers one chunk, eight CONSECUTIVE entries per lane.  A lane gathers the x
//     entries that pass the filter (one load each: the dense copy of x carries a "not listed"
//     marker), multiplies, and sums runs of equal row inside its eight entries in registers;
//     ROW_FLAG in the entry marks where a row starts.
//   * Across the lanes a segmented shuffle scan adds up the pieces of every row that spans
//     several lanes (Section 3.3.3: registers, then warp shuffle), and one lane per row adds the
//     sum to global memory -- a row cut by a pass or chunk boundary simply contributes one atomic
//     per piece.  The row a sum belongs to comes from the row list (lean_rows), indexed by the
//     running count of ROW_FLAGs; structural hits are tracked as bit masks beside the sums.
//   * The few entries with a payload are skipped by the stream and taken before it, one block
//     per warp at a time, from the list of their positions.
//   * Bounds, 16 M fp32 entries, half of x listed: 58 us (73 before the filter's loads were spread and the payload entries
//     moved to the front), L1 data path 76 % busy (gathers, filter look-ups and the stream share it), issue slots 52 %.
//   * The same kernel serves the (min, +) semiring (Out::MINPLUS): products become sums, sums
//     minima with identity +infinity, and the writeback keeps the smaller value (minplus.cuh).
#pragma once

#include "internal.cuh"
#include "microkernels.cuh"
#include "minplus.cuh"
#include "push_direct.cuh"

namespace dbs {

constexpr int LEAN_WARPS = 32;     // warps per thread block; one thread block per SM
constexpr int LEAN_CTA = LEAN_WARPS * 32;
// Presence filter of x in shared memory: one bit per column (folded modulo the filter size when
// x has more columns than bits), tested before every gather.
constexpr int LEAN_FILTER_MAX_WORDS = 32768;   // 128 KB: exact up to 1,048,576 columns

constexpr int LEAN_ROWS_CACHED = 64;
constexpr int LEAN_PER_LANE = LEAN_CHUNK / 32;
static_assert(LEAN_PER_LANE == 8, "a lane takes two 16-byte loads of view indices");

// A lane's eight consecutive entries of one chunk: view indices, packed coordinates, values.
struct LeanEntries { uint4 i0, i1; uint2 a; uint4 w0, w1; };
template <bool VAL>
__device__ __forceinline__ LeanEntries lean_fetch(const Device &d, int c, int lane) {
    // (always a whole chunk: the view arrays have that much slack behind the last entry, filled
    // with PAD_IDX entries; streaming loads: the bytes are never read again)
    const size_t e = (size_t)c * LEAN_CHUNK + (size_t)LEAN_PER_LANE * lane;
    LeanEntries r;
    r.i0 = __ldcs(reinterpret_cast<const uint4 *>(d.csr.idx + e));
    r.i1 = __ldcs(reinterpret_cast<const uint4 *>(d.csr.idx + e + 4));
    r.a = __ldcs(reinterpret_cast<const uint2 *>(d.csr.aux + e));
    r.w0 = r.w1 = make_uint4(0u, 0u, 0u, 0u);
    if (VAL) {
        r.w0 = __ldcs(reinterpret_cast<const uint4 *>(d.csr.w + e));
        r.w1 = __ldcs(reinterpret_cast<const uint4 *>(d.csr.w + e + 4));
    }
    return r;
}
// A chunk whose dependent loads are in flight: the x entries, the values, the slice of the row list.
struct LeanWork {
    float xin[LEAN_PER_LANE];
    uint4 w0, w1;
    int rowp0, rowp1;
    int ord;             // ROW_FLAGs before the chunk (lean_rows[ord - 1] is the row that runs into it)
    uint32_t meta;       // bits 0-7: entry k starts a row; 8-16: row starts in the lanes below; 17: some lane holds several
};

template <int DT, typename Out>
__device__ __forceinline__ void lean_add(Out out, int row, float v) {
    if (Out::MINPLUS) {          // keep the smaller sum (an atomic whose reply nobody waits for)
        atomicMax(reinterpret_cast<int *>(out.acc) + row, minplus_word(v));
        return;
    }
    out_add(out, row, DT != DBSPMSPV_PATTERN ? v : 1.0f);
}
// The semiring of the segmented reduction: (+, *) or, for Out::MINPLUS, (min, +).
template <typename Out> __device__ __forceinline__ float lean_identity() { return Out::MINPLUS ? __int_as_float(0x7F800000) : 0.f; }
template <typename Out> __device__ __forceinline__ float lean_mul(float a, float x) { return Out::MINPLUS ? a + x : a * x; }
template <typename Out> __device__ __forceinline__ float lean_sum(float s, float p) { return Out::MINPLUS ? fminf(s, p) : s + p; }

// First half of a chunk: what needs the entries only (the row-start bits and, from a ballot of them, how many rows start
// in the lanes below), then all dependent global loads at once -- nothing here waits for them.
__device__ __forceinline__ void lean_issue(const Device &d, LeanWork &q, const LeanEntries &r, int ord, const uint32_t *filter, uint32_t filter_mask, int lane) {
    constexpr int K = LEAN_PER_LANE;
    const uint32_t lt = (1u << lane) - 1u;
    const uint32_t idx[K] = {r.i0.x, r.i0.y, r.i0.z, r.i0.w, r.i1.x, r.i1.y, r.i1.z, r.i1.w};
#pragma unroll
    for (int k = 0; k < K; ++k) {
        // INLINE is class 0: any other entry (a block with a payload, the slack) is skipped here
        bool go = idx[k] < (1u << TYPE_SHIFT) && DBS_CHK_INDEX(d, idx[k] & IDX_MASK, d.nb);
        const uint32_t a = k < 4 ? r.a.x : r.a.y;
        const uint32_t col = (idx[k] & IDX_MASK) * 16u + ((a >> (8 * (k & 3))) & 15u);
        // (a set filter bit may belong to another column when the filter is folded: the gather
        // then returns the "not listed" marker, as it would without the filter)
        go = go && ((filter[(col >> 5) & filter_mask] >> (col & 31u)) & 1u);
        // (through L1: on a power-law matrix a few hundred columns draw a third of all gathers, and with L2-only
        // loads those lines saturate single L2 slices)
        q.xin[k] = go ? __ldg(d.ws.x_dense + col) : __uint_as_float(X_ABSENT);
    }
    q.w0 = r.w0; q.w1 = r.w1;
    uint32_t hb = 0u;            // bit k: entry k starts a row
#pragma unroll
    for (int k = 0; k < K; ++k) hb |= ((idx[k] >> 27) & 1u) << k;
    const int cnt = __popc(hb);
    const uint32_t hm = __ballot_sync(FULL, hb != 0u);      // lanes in which a row starts
    const bool multi = __any_sync(FULL, cnt > 1);           // some lane holds several row starts
    int excl, total;                                         // row starts in the lanes below / in the chunk
    if (multi) {
        int incl = cnt;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int t = __shfl_up_sync(FULL, incl, o);
            if (lane >= o) incl += t;
        }
        excl = incl - cnt;
        total = __shfl_sync(FULL, incl, 31);
    } else {
        excl = __popc(hm & lt);
        total = __popc(hm);
    }
    // the rows this chunk adds to (lean_rows[ord - 1 .. ord + total - 1]: a lane fetches numbers l and 32 + l of
    // them; a chunk of rows of one to three entries has more than 64 and reads the rest from the list directly)
    const int o = ord - 1 + lane;
    q.rowp0 = lane <= total && o >= 0 && o < d.n_lean_rows ? __ldg(d.lean_rows + o) : 0;
    q.rowp1 = lane + 32 <= total && o + 32 < d.n_lean_rows ? __ldg(d.lean_rows + o + 32) : 0;
    q.ord = ord;
    q.meta = hb | (uint32_t)excl << 8 | (multi ? 1u << 17 : 0u);
}

// Second half: the sums.
template <int DT, typename Out>
__device__ __forceinline__ void lean_sums(const Device &d, Out out, const LeanWork &q, int *s_rows, int lane) {
    constexpr bool VAL = DT != DBSPMSPV_PATTERN;
    constexpr int K = LEAN_PER_LANE;
    const uint32_t lt = (1u << lane) - 1u;
    const uint32_t wv[K] = {q.w0.x, q.w0.y, q.w0.z, q.w0.w, q.w1.x, q.w1.y, q.w1.z, q.w1.w};
    const float (&xin)[K] = q.xin;
    const uint32_t hb = q.meta & 0xFFu;
    const int excl = (int)(q.meta >> 8) & 0x1FF, cnt = __popc(hb), ord = q.ord;
    const bool multi = (q.meta >> 17) & 1u;
    const uint32_t hm = __ballot_sync(FULL, hb != 0u);
    // row of the chunk's row start number k (k = 0: the row that runs into the chunk)
    auto row_of = [&](int k) { return k < LEAN_ROWS_CACHED ? s_rows[k] : d.lean_rows[ord - 1 + k]; };
    __syncwarp();                // (the previous chunk's look-ups are over)
    s_rows[lane] = q.rowp0;
    s_rows[lane + 32] = q.rowp1;
    __syncwarp();
    // ---- sums.  Thread-serial part: `lead` = sum of the lane's entries before its first row
    // start (they belong to the row that was open when the lane began), `seg` = sum from its last
    // row start on; rows that lie wholly inside the lane are added to global memory by the lane.
    const float ID = lean_identity<Out>();
    float lead = ID, seg = ID;
    uint32_t lead_hit = 0u, seg_hit = 0u;
    if (!multi) {
        // at most one row start per lane (the usual case): entries below it, entries from it on
        const int f = hb ? __ffs(hb) - 1 : K;
        uint32_t pb = 0u;
#pragma unroll
        for (int k = 0; k < K; ++k) {
            if (__float_as_uint(xin[k]) != X_ABSENT) {
                pb |= 1u << k;
                if (VAL) {
                    const float p = lean_mul<Out>(Val<DT>::inline_value(wv[k]), xin[k]);
                    if (k < f) lead = lean_sum<Out>(lead, p); else seg = lean_sum<Out>(seg, p);
                }
            }
        }
        const uint32_t below = (1u << f) - 1u;
        lead_hit = pb & below;
        seg_hit = pb & ~below;
    } else {
        int nh = 0;
#pragma unroll
        for (int k = 0; k < K; ++k) {
            if ((hb >> k) & 1u) {
                if (nh == 0) { lead = seg; lead_hit = seg_hit; }
                else if (seg_hit) lean_add<DT>(out, row_of(excl + nh), seg);   // a whole row inside the lane
                ++nh;
                seg = ID; seg_hit = 0u;
            }
            if (__float_as_uint(xin[k]) != X_ABSENT) {
                if (VAL) seg = lean_sum<Out>(seg, lean_mul<Out>(Val<DT>::inline_value(wv[k]), xin[k]));
                seg_hit = 1u;
            }
        }
        if (nh == 0) { lead = seg; lead_hit = seg_hit; seg = ID; seg_hit = 0u; }
    }
    // Warp part.  A lane with a row start closes the row that was open before it.  S = inclusive
    // sum of `lead` over the lanes since the last lane with a row start (exclusive): at a lane with
    // a row start, or at lane 31, S is the whole tail of the row that started before.
    const uint32_t lh = __ballot_sync(FULL, lead_hit != 0u);
    float S = lead;
    if (VAL) {
        const int reach = lane - (32 - __clz(hm & lt));       // lanes to my left in my run
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const float t = __shfl_up_sync(FULL, S, o);
            if (reach >= o) S = lean_sum<Out>(S, t);
        }
    }
    // (a) the row that runs into the chunk: closed by the first lane with a row start (lane 31 if none)
    const int wl = hm ? __ffs(hm) - 1 : 31;
    if (lane == wl && (lh & ((2u << wl) - 1u))) lean_add<DT>(out, row_of(0), S);
    // (b) the row that starts at a lane's last row start: its piece here, plus the leads of the
    // lanes up to and including the next lane with a row start (or lane 31)
    const uint32_t above = hm & ~lt & ~(1u << lane);
    const int nx = above ? __ffs(above) - 1 : 31;
    float tail = ID;
    if (VAL) { tail = __shfl_sync(FULL, S, nx); if (lane == 31) tail = ID; }
    if (cnt) {
        const uint32_t tail_hit = ((lh >> 1) >> lane) & ((1u << (nx - lane)) - 1u);
        if (seg_hit | tail_hit) lean_add<DT>(out, row_of(excl + cnt), lean_sum<Out>(seg, tail));
    }
}

struct LeanScratch {        // per warp
    int rows[LEAN_ROWS_CACHED];   // the slice of the row list the current chunk adds to
    float sx[16];                 // the microkernels of the entries with a payload
    float stmp[32];
};

template <int DT, typename Out, bool LONG>
__global__ void __launch_bounds__(LEAN_CTA, 1)
k_pull_lean(Device d, Out out, float th3, int force_path, int popc_threshold, int filter_words, int boolean_push) {
    extern __shared__ __align__(128) uint8_t s_lean[];
    constexpr bool VAL = DT != DBSPMSPV_PATTERN;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    uint32_t *filter = reinterpret_cast<uint32_t *>(s_lean);
    LeanScratch *ls = reinterpret_cast<LeanScratch *>(s_lean + (size_t)filter_words * 4) + warp;
    pdl_wait();
    if (select_path(d, th3, force_path) != DBSPMSPV_PATH_PULL) {
        if constexpr (LONG) {                          // the push's listed chunks (see k_push_long)
            const int gw = warp * gridDim.x + blockIdx.x, nw = gridDim.x * LEAN_WARPS;
            constexpr int MODE = Out::MINPLUS ? 2 : DT == DBSPMSPV_PATTERN ? 1 : 0;
            if (MODE == 0 && boolean_push) push_long_chunks<DT, 1, false>(d, gw, nw);
            else push_long_chunks<DT, MODE, false>(d, gw, nw);
        }
        return;
    }
    if (blockIdx.x == 0 && threadIdx.x == 0) d.ws.ctr->path = DBSPMSPV_PATH_PULL;
    const int gwarp = warp * gridDim.x + blockIdx.x;      // (neighbouring chunks on different SMs: the last, partial round of chunks is spread over all of them)
    const int nwarps = gridDim.x * LEAN_WARPS;
    LeanEntries nxt = {};
    int ord_next = 0;
    if (gwarp < d.n_lean_chunks) { nxt = lean_fetch<VAL>(d, gwarp, lane); ord_next = d.lean_chunk_ord[gwarp]; }
    // the filter: the vector-block masks are the presence bitmap of x (bit j of the array = column
    // j); folded by OR when x has more columns than the filter has bits
    {
        const int n_words = (d.nb + 1) / 2;
        if (n_words <= filter_words && filter_words >= 4 * LEAN_CTA) {
            // Every thread block reads the same words: four 16-byte loads in flight per thread, and the blocks start at different places.
            // (One dependent word after the other, all blocks on the same L2 slice at a time, took 14 us of a kernel of 73.)
            const int n16 = filter_words / 4;
            for (int k0 = 0; k0 < n16; k0 += 4 * LEAN_CTA) {
                uint4 v[4];
                int at[4];
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                    const int k = k0 + u * LEAN_CTA + threadIdx.x;
                    at[u] = k < n16 ? (int)((k + blockIdx.x * 64u) & (n16 - 1)) : -1;
                    v[u] = make_uint4(0u, 0u, 0u, 0u);
                    if (at[u] >= 0 && at[u] * 4 + 3 < n_words) v[u] = __ldcg(reinterpret_cast<const uint4 *>(d.ws.x_mask32) + at[u]);
                    else if (at[u] >= 0 && at[u] * 4 < n_words) {
                        v[u].x = d.ws.x_mask32[at[u] * 4];
                        if (at[u] * 4 + 1 < n_words) v[u].y = d.ws.x_mask32[at[u] * 4 + 1];
                        if (at[u] * 4 + 2 < n_words) v[u].z = d.ws.x_mask32[at[u] * 4 + 2];
                    }
                }
#pragma unroll
                for (int u = 0; u < 4; ++u) if (at[u] >= 0) reinterpret_cast<uint4 *>(filter)[at[u]] = v[u];
            }
        } else
        for (int f = threadIdx.x; f < filter_words; f += LEAN_CTA) {
            uint32_t v = 0u;
            for (int q = f; q < n_words; q += filter_words) v |= d.ws.x_mask32[q];
            filter[f] = v;
        }
    }
    __syncthreads();
    const uint32_t filter_mask = (uint32_t)filter_words - 1u;
    // Entries with a payload: one block per warp at a time (they are the exception in these handles).  Before the stream, with its first
    // chunk in flight: a block is a chain of six dependent loads, which cost 11 us at the end of a kernel of 60 (5.5 K blocks, 16 M
    // entries), where nothing else was left to run.  From the last warp on: the last ones have a chunk less in the stream.
    for (int q = nwarps - 1 - gwarp; q < d.n_payload; q += nwarps) {
        const int pos = d.payload_pos[q];
        if (!DBS_CHK_INDEX(d, pos, d.n_entries)) continue;            // warp-uniform
        uint32_t idx = d.csr.idx[pos];
#ifdef DBS_BOUNDS_CHECK
        {
            uint32_t w_ = d.csr.w[pos], a_ = d.csr.aux[pos];
            DBS_CHK_ENTRY(d, true, idx, w_, a_);
            if ((idx >> TYPE_SHIFT) == DBSPMSPV_BLK_INLINE || !DBS_CHK_INDEX(d, d.entry_row[pos], d.mb)) continue;   // (only a replaced entry is INLINE here)
        }
#endif
        const int cb = idx & IDX_MASK, type = idx >> TYPE_SHIFT;
        const uint32_t xm = mask_of(d.ws.x_mask32, cb);
        if (!xm) continue;                                            // warp-uniform
        const uint8_t *blk = d.payload + (size_t)d.csr.w[pos] * 4;
        const int nnz = (int)d.csr.aux[pos] + 1;
        const int rb = d.entry_row[pos];
        if (Out::MINPLUS) {
            block_rows_min_warp<DT>(type, d.csr.w[pos], d.csr.aux[pos], xm, d.ws.x_dense + (size_t)cb * 16, d.payload, lane, [&](int r, uint32_t key) {
                atomicMax(reinterpret_cast<int *>(out.acc) + (size_t)rb * 16 + r, minplus_word_of_key(key));
            });
            continue;
        }
        uint32_t hits;
        float sum = 0.f;
        if (DT == DBSPMSPV_PATTERN) {
            hits = warp_block_bool<DT>(type, blk, nnz, xm, lane);
        } else {
            __syncwarp();
            if (lane < 16) ls->sx[lane] = d.ws.x_dense[(size_t)cb * 16 + lane];
            __syncwarp();
            sum = warp_block<DT>(type, blk, nnz, xm, ls->sx, ls->stmp, lane, popc_threshold, hits);
        }
        if (lane < 16 && ((hits >> lane) & 1u)) out_add(out, (size_t)rb * 16 + lane, DT != DBSPMSPV_PATTERN ? sum : 1.0f);
    }
    // Without values the gathers of a chunk are issued before the sums of the chunk before it (79 us to 61 on 29 M entries, 30 % of x
    // listed).  With values the registers for two chunks are not there (and 53 us in place of 45 on 16 M entries): the next
    // chunk's entries fly during the sums, its gathers follow.
    constexpr int AHEAD = VAL ? 0 : 1;
    LeanWork cur = {};
    auto fetch = [&](int c) { if (c < d.n_lean_chunks) { nxt = lean_fetch<VAL>(d, c, lane); ord_next = d.lean_chunk_ord[c]; } };
    if (AHEAD && gwarp < d.n_lean_chunks) {
        lean_issue(d, cur, nxt, ord_next, filter, filter_mask, lane);
        fetch(gwarp + nwarps);
    }
    for (int c = gwarp; c < d.n_lean_chunks; c += nwarps) {
        if (AHEAD) {
            LeanWork ahead = {};
            if (c + nwarps < d.n_lean_chunks) lean_issue(d, ahead, nxt, ord_next, filter, filter_mask, lane);
            fetch(c + 2 * nwarps);
            lean_sums<DT, Out>(d, out, cur, ls->rows, lane);
            cur = ahead;
        } else {
            const LeanEntries now = nxt;
            const int ord = ord_next;
            fetch(c + nwarps);
            lean_issue(d, cur, now, ord, filter, filter_mask, lane);
            lean_sums<DT, Out>(d, out, cur, ls->rows, lane);
        }
    }
}

}  // namespace dbs

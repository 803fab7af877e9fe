// dbspmspv_run for a short x on a hypersparse handle, as ONE kernel of ONE thread-block cluster
// (Section 4.1: vector-metadata construction fused with the SpMSpV kernel, no extra launch, no
// host round trip).  The chain of the general path -- push, listed chunks, finishing
// kernel -- costs up to three dependent launches, each with its own cold first loads, whatever x
// holds; for up to a few hundred listed columns that chain IS the call (18 - 26 us for 10 .. 100
// nonzeros on a matrix with a million rows, cold; 11 - 18 us here).  Here nothing of x is staged at all:
//   * a warp takes one listed column j (consecutive columns in different thread blocks): its
//     value stays in a register, its run of INLINE
//     elements comes from the column pointers of the block-CSC view, four of them
//     fetched per lane before the first is used, the column block's few
//     entries with a payload are taken eight at a time, a half-warp each; hub columns and longer runs of payload entries are listed and
//     shared out over the whole cluster in chunks (a lane per payload entry, a run by one warp: R-MAT matrices, not relabelled, 64 K .. 256 K rows, 96 / 250 columns 11 - 14 / 14 - 16 us a call, 9 - 11 / 12 - 13 so);
//   * a product goes to the handle's dense accumulator with a reply-free atomic, and sets the
//     row's bit in a bitmap of ALL rows that the cluster's thread blocks hold together in their
//     shared memories (4 bytes per 32 rows, an eighth of the rows per thread block; remote bits
//     are set through distributed shared memory) -- the structural-hit record, exact whatever
//     the sums are;
//   * after one cluster barrier the bitmap is the list of the result's rows: every thread block counts
//     its slice, the eight totals are exchanged through distributed shared memory, the set bits
//     become the slice's row list in shared memory, and the thread block gathers the sums, clears them and writes its part of y.  (Where a slice
//     holds more than SMALL_ROWS rows the list is parked in the unused task array and all threads of the cluster take result positions in turn.)
// What bounds it is the chain of trips, 0.6 - 0.9 us each: x -> column pointers -> entries -> sums and bits, a cluster barrier, counts, a cluster barrier, sums -> y.  The trips as far as the entries
// are made while the cluster meets for the first time and clears its bitmap; nothing is read back from global memory but the sums.  (Met first, then walked, the row list written to global memory and read
// again behind two more cluster barriers: uniform rows, 16 K of them, 16 columns 6.8 -> 5.2 us a call, a million, 16 / 160 columns 7.7 / 9.7 -> 6.1 / 6.6; R-MAT in scattered order, 64 K rows,
// 48 columns 7.8 -> 6.1, a million, 96 columns 9.4 -> 7.2; not relabelled, 131 K, 16 / 96 columns 9.5 / 13.4 -> 7.1 / 9.4, a million 8.0 / 9.9 -> 6.5 / 7.8; 27-point operator on 90^3 cells, 64 scattered columns 13.2 -> 8.1.)
// The dense copy of x, the vector-block masks and the worklist are never
// written, so there is nothing to clean up.  Used when x is short, the selector is certain to
// say push, the bitmap fits, and no option asks for the general path; results are identical
// to the general path's up to the order of the fp32 additions.  The cluster barriers are the
// hardware's (all thread blocks of a cluster are co-resident by construction): no spin-waits.
#pragma once

#include <cooperative_groups.h>

#include "internal.cuh"
#include "minplus.cuh"
#include "push_direct.cuh"
#include "worklist.cuh"

namespace dbs {

constexpr int SMALL_CTA = 1024;
constexpr int SMALL_CLUSTER = 8;               // thread blocks of the cluster (the portable maximum)
// One warp per listed column: small_call_limit in run.cu says where a handle's calls change over to the chain of kernels, with both sides measured.
constexpr int SMALL_MAX_NNZ_X = 256;
constexpr int SMALL_HUB_RUN = 512;             // a run from this length on is walked by the whole cluster
constexpr int SMALL_HUB_PAYLOAD = 17;          // ... and one of so many entries with a payload
constexpr int SMALL_HUB_CAP = 128;
constexpr int SMALL_ILP = 4;                   // view entries a thread fetches before it works on them
constexpr size_t SMALL_MAX_SMEM = 40 * 1024;   // bitmap slices of one thread block (dynamic shared memory)
constexpr int SMALL_ROWS = 8192;               // rows of a slice's result that are listed in shared memory (behind the slices)

struct SmallShared {
    int wsum[SMALL_CTA / 32];
    int total[SMALL_CLUSTER];      // result entries of every thread block's slice (each block holds a full copy)
    int nzblk;                     // (thread block 0) nonempty vector blocks
    int n_hubs;                    // (thread block 0) listed hub runs
    int4 hubs[SMALL_HUB_CAP];      // (thread block 0) first position, entries, x value bits, local column | payload flag << 8
    int4 run[SMALL_HUB_CAP];       // the list once more, in every thread block, and the chunks before each run
    int pre[SMALL_HUB_CAP + 1];
};

// mode: 0 = (+, *), 1 = Boolean, 2 = (min, +)
template <int DT>
__global__ void __cluster_dims__(SMALL_CLUSTER, 1, 1) __launch_bounds__(SMALL_CTA, 1)
k_run_small(Device d, const int32_t *__restrict__ x_idx, const void *__restrict__ x_val, int32_t nnz_x, int mode,
            int32_t *__restrict__ y_idx, float *__restrict__ y_val, int64_t y_capacity, int32_t *__restrict__ y_nnz,
            const uint32_t *__restrict__ row_mask, int complement) {
    namespace cg = cooperative_groups;
    cg::cluster_group cluster = cg::this_cluster();
    extern __shared__ __align__(16) uint32_t s_small[];
    __shared__ SmallShared sh;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int rank = (int)cluster.block_rank();
    const int ywords = (d.mb + 1) / 2, cbwords = (d.nb + 31) / 32;
    const int yper = (ywords + SMALL_CLUSTER - 1) / SMALL_CLUSTER, cper = (cbwords + SMALL_CLUSTER - 1) / SMALL_CLUSTER;
    // this block's slices: row words [rank * yper, ...), vector-block words [rank * cper, ...)
    for (int k = tid; k < yper + cper; k += SMALL_CTA) s_small[k] = 0u;
    if (tid == 0) { sh.nzblk = 0; sh.n_hubs = 0; }
    asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
    pdl_wait();
    // A warp per listed column (256 warps in the cluster); consecutive columns go
    // to different thread blocks.  (Several columns per warp were measured too: from about a
    // thousand columns on, the tails of the longer runs make the slowest warp take longer than
    // the general path's whole chain of kernels, which spreads them over the GPU.)
    // Its x, its column's place and its first entries are fetched before the cluster has met.
    static_assert(SMALL_MAX_NNZ_X * 32 <= SMALL_CLUSTER * SMALL_CTA, "every listed column has its own warp");
    const int k = warp * SMALL_CLUSTER + rank;
    bool have = k < nnz_x;                         // warp-uniform
    const int j = have ? x_idx[k] : 0;
    if (have && (j < 0 || j >= d.n)) { if (lane == 0) d.ws.ctr->status = DBSPMSPV_ERR_BOUNDS; have = false; }
    float xv = 1.0f;
    int first = 0, deg = 0, pfirst = 0, pdeg = 0;
    uint32_t ix[SMALL_ILP], wv[SMALL_ILP], ax[SMALL_ILP];
#pragma unroll
    for (int u = 0; u < SMALL_ILP; ++u) { ix[u] = 0xFFFFFFFFu; wv[u] = 0u; ax[u] = 0u; }
    if (have) {
        if (mode != 1 && x_val) {
            if (DT == DBSPMSPV_BF16) xv = __bfloat162float(static_cast<const __nv_bfloat16 *>(x_val)[k]);
            else xv = static_cast<const float *>(x_val)[k];
        }
        column_run(d, j, first, deg);
        payload_run(d, j >> 4, pfirst, pdeg);
        if (deg < SMALL_HUB_RUN)
#pragma unroll
            for (int u = 0; u < SMALL_ILP; ++u) {
                const int q = lane + 32 * u;
                if (q < deg) { ix[u] = d.csc.idx[first + q]; wv[u] = d.csc.w[first + q]; ax[u] = d.csc.aux[first + q]; }
            }
    }
    asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
    SmallShared *sh0 = cluster.map_shared_rank(&sh, 0);
    // wi / yper: a slice has at most 10240 words (SMALL_MAX_SMEM), so wi * yper < 2^32 and the quotient by the rounded-up reciprocal is exact (a slice of one word: the word's number itself)
    const unsigned ymagic = 0xFFFFFFFFu / (unsigned)yper + 1u;
    int *words = reinterpret_cast<int *>(d.ws.y_acc);
    auto add = [&](int row, float a, float xv) {
        if (mode == 2) atomicMax(words + row, minplus_word(a + xv));
        else if (mode == 0 && DT != DBSPMSPV_PATTERN) atomicAdd(d.ws.y_acc + row, a * xv);
        const int wi = row >> 5, owner = yper > 1 ? (int)__umulhi((unsigned)wi, ymagic) : wi;
        atomicOr(cluster.map_shared_rank(s_small, owner) + (wi - owner * yper), 1u << (row & 31));
    };
    auto add_entry = [&](uint32_t idx, uint32_t w, uint32_t aux, float xv) {
        if (idx == 0xFFFFFFFFu || !DBS_CHK_INDEX(d, idx & IDX_MASK, d.mb)) return;
        add((int)(idx & IDX_MASK) * 16 + (int)(aux >> 4), Val<DT>::inline_value(w), xv);
    };
    // INLINE entries p, p + step, ... below `end`: SMALL_ILP of them are fetched before the first is used
    // (a run is a chain of cold loads otherwise: the address of an entry's atomic depends on the entry)
    auto inline_run = [&](int p, int end, int step, float xv) {
        for (; p < end; p += SMALL_ILP * step) {
            uint32_t ix[SMALL_ILP], wv[SMALL_ILP], ax[SMALL_ILP];
#pragma unroll
            for (int u = 0; u < SMALL_ILP; ++u) {
                const int q = p + u * step;
                ix[u] = 0xFFFFFFFFu; wv[u] = 0u; ax[u] = 0u;
                if (q < end) { ix[u] = d.csc.idx[q]; wv[u] = d.csc.w[q]; ax[u] = d.csc.aux[q]; }
            }
#pragma unroll
            for (int u = 0; u < SMALL_ILP; ++u) add_entry(ix[u], wv[u], ax[u], xv);
        }
    };
    // `count` <= PD_PAYLOAD entries with a payload, local column c, by one warp: a half-warp each (push_direct.cuh)
    auto payload_chunk = [&](int p, int count, int c, float xv) {
        constexpr int U = PD_PAYLOAD / 2;
        bool in[U];
        float a[U];
        uint32_t rb[U];
        payload_elements<DT, U>(d, p, count, c, lane, in, a, rb);
#pragma unroll
        for (int u = 0; u < U; ++u) if (in[u] && DBS_CHK_INDEX(d, rb[u], d.mb)) add((int)(rb[u] * 16u) + (lane & 15), a[u], xv);
    };
    // a run that the whole cluster should share: listed in thread block 0 (true), or left to the warp
    auto list_hub = [&](int first, int deg, float xv, int tag) {
        int slot = 0;
        if (lane == 0) slot = atomicAdd(&sh0->n_hubs, 1);
        slot = __shfl_sync(FULL, slot, 0);
        if (slot >= SMALL_HUB_CAP) return false;
        if (lane == 0) sh0->hubs[slot] = make_int4(first, deg, __float_as_int(xv), tag);
        return true;
    };
    // ---- traversal
    if (have) {
        if (lane == 0) {
            const int cw = j >> 9, owner = cw / cper;
            const uint32_t bit = 1u << ((j >> 4) & 31);
            if (!(atomicOr(cluster.map_shared_rank(s_small, owner) + yper + (cw - owner * cper), bit) & bit)) atomicAdd(&sh0->nzblk, 1);
        }
#pragma unroll
        for (int u = 0; u < SMALL_ILP; ++u) add_entry(ix[u], wv[u], ax[u], xv);
        if (deg >= SMALL_HUB_RUN) { if (!list_hub(first, deg, xv, 0)) inline_run(first + lane, first + deg, 32, xv); }
        else inline_run(first + 32 * SMALL_ILP + lane, first + deg, 32, xv);
        if (pdeg > 0 && (pdeg < SMALL_HUB_PAYLOAD || !list_hub(pfirst, pdeg, xv, (j & 15) | 256)))
            for (int p = 0; p < pdeg; p += PD_PAYLOAD) payload_chunk(pfirst + p, min(PD_PAYLOAD, pdeg - p), j & 15, xv);
    }
    cluster.sync();
    // listed runs: every thread block lays their chunks end to end, the warps of the cluster share them out
    const int n_hubs = min(sh0->n_hubs, SMALL_HUB_CAP);
    if (n_hubs) {                              // (cluster-uniform: every block read the same count)
        constexpr int CHUNK = 32 * SMALL_ILP;
        if (tid < n_hubs) sh.run[tid] = sh0->hubs[tid];
        __syncthreads();
        if (warp == 0) {
            int before = 0;
            for (int q0 = 0; q0 < n_hubs; q0 += 32) {
                const int q = q0 + lane;
                const int chunks = q >= n_hubs ? 0 : sh.run[q].w & 256 ? (sh.run[q].y + PD_PAYLOAD - 1) / PD_PAYLOAD : (sh.run[q].y + CHUNK - 1) / CHUNK;
                int incl = chunks;
#pragma unroll
                for (int o = 1; o < 32; o <<= 1) { const int t = __shfl_up_sync(FULL, incl, o); if (lane >= o) incl += t; }
                if (q < n_hubs) sh.pre[q] = before + incl - chunks;
                before += __shfl_sync(FULL, incl, 31);
            }
            if (lane == 0) sh.pre[n_hubs] = before;
        }
        __syncthreads();
        const int all = sh.pre[n_hubs];
        for (int c = warp * SMALL_CLUSTER + rank; c < all; c += SMALL_CLUSTER * SMALL_CTA / 32) {
            int o = 0;                         // the last run with at most c chunks before it
#pragma unroll
            for (int st = SMALL_HUB_CAP / 2; st; st >>= 1) if (o + st < n_hubs && sh.pre[o + st] <= c) o += st;
            const int4 hb = sh.run[o];
            const int at = c - sh.pre[o];
            const float xs = __int_as_float(hb.z);
            if (hb.w & 256) payload_chunk(hb.x + at * PD_PAYLOAD, min(PD_PAYLOAD, hb.y - at * PD_PAYLOAD), hb.w & 15, xs);
            else inline_run(hb.x + at * CHUNK + lane, hb.x + min(hb.y, (at + 1) * CHUNK), 32, xs);
        }
        cluster.sync();
    }
    // ---- result from the bitmap.  This block's slice; thread t owns the words [t * per, (t + 1) * per).
    const int my_words = max(0, min(yper, ywords - rank * yper));
    const int per = (yper + SMALL_CTA - 1) / SMALL_CTA;
    const int w0 = min(tid * per, my_words), w1 = min(w0 + per, my_words);
    const int wbase = rank * yper;
    auto keep_of = [&](int wi) { return row_mask ? (complement ? ~row_mask[wi] : row_mask[wi]) : 0xFFFFFFFFu; };
    int cnt = 0;
    for (int wi = w0; wi < w1; ++wi) {
        const uint32_t word = s_small[wi];
        if (word) cnt += __popc(word & keep_of(wbase + wi));
    }
    int incl = cnt;
    for (int o = 1; o < 32; o <<= 1) {
        const int t = __shfl_up_sync(0xFFFFFFFFu, incl, o);
        if (lane >= o) incl += t;
    }
    if (lane == 31) sh.wsum[warp] = incl;
    __syncthreads();
    if (warp == 0) {
        int v = sh.wsum[lane], s = v;
        for (int o = 1; o < 32; o <<= 1) {
            const int t = __shfl_up_sync(0xFFFFFFFFu, s, o);
            if (lane >= o) s += t;
        }
        sh.wsum[lane] = s - v;
        // this block's total goes into every block's table
        if (lane == 31)
            for (int r = 0; r < SMALL_CLUSTER; ++r) cluster.map_shared_rank(&sh, r)->total[rank] = s;
    }
    cluster.sync();
    int before = 0, total = 0, most = 0;
#pragma unroll
    for (int r = 0; r < SMALL_CLUSTER; ++r) { if (r < rank) before += sh.total[r]; total += sh.total[r]; most = max(most, sh.total[r]); }
    if (rank == 0 && tid == 0) {
        Counters *c = d.ws.ctr;
        *y_nnz = total;
        if ((int64_t)total > y_capacity) c->status = DBSPMSPV_ERR_CAPACITY;
        c->last_y_nnz = total;
        c->last_n_nzblk = sh.nzblk;
        c->last_n_tasks = 0;
        c->last_path = DBSPMSPV_PATH_PUSH;
        c->path = DBSPMSPV_PATH_PUSH;
    }
    auto write = [&](int64_t q, int row, float v) {
        y_idx[q] = row;
        if (y_val) y_val[q] = mode == 1 || (mode == 0 && DT == DBSPMSPV_PATTERN) ? 1.0f : mode == 2 ? minplus_of_word(__float_as_uint(v)) : v + 0.0f;      // (+ 0: a row of -0 products is 0)
    };
    if (most <= SMALL_ROWS) {                      // (cluster-uniform) this slice's rows, in order; those masked out are cleared here
        int *list = reinterpret_cast<int *>(s_small) + yper + cper;
        int at = sh.wsum[warp] + incl - cnt;
        for (int wi = w0; wi < w1; ++wi) {
            const uint32_t word = s_small[wi];
            if (!word) continue;
            const uint32_t keep = keep_of(wbase + wi);
            for (uint32_t bb = word; bb; bb &= bb - 1) {
                const int bit = __ffs(bb) - 1, row = (wbase + wi) * 32 + bit;
                if ((keep >> bit) & 1u) list[at++] = row;
                else d.ws.y_acc[row] = __uint_as_float(ACC_CLEAR);
            }
        }
        __syncthreads();
        const int mine = sh.total[rank];
        for (int p0 = tid; p0 < mine; p0 += SMALL_ILP * SMALL_CTA) {
            int r[SMALL_ILP];
            float v[SMALL_ILP];
#pragma unroll
            for (int u = 0; u < SMALL_ILP; ++u) {
                const int q = p0 + u * SMALL_CTA;
                r[u] = q < mine ? list[q] : -1;
                v[u] = r[u] >= 0 ? __ldcg(d.ws.y_acc + r[u]) : 0.f;              // (the sums were made by atomics in L2)
            }
#pragma unroll
            for (int u = 0; u < SMALL_ILP; ++u) {
                if (r[u] < 0) continue;
                const int64_t q = (int64_t)before + p0 + u * SMALL_CTA;
                d.ws.y_acc[r[u]] = __uint_as_float(ACC_CLEAR);
                if (q < y_capacity) write(q, r[u], v[u]);
            }
        }
        return;                                    // (nobody reads another block's shared memory any more)
    }
    int pos = before + sh.wsum[warp] + incl - cnt;
    const int64_t room = y_capacity < (int64_t)total ? y_capacity : (int64_t)total;
    // the result's rows, in order, parked in the (unused) task array; rows that do not go to y
    // (masked out, or beyond the capacity) are cleared here
    int32_t *rows = reinterpret_cast<int32_t *>(d.ws.tasks);
    for (int wi = w0; wi < w1; ++wi) {
        const uint32_t word = s_small[wi];
        if (!word) continue;
        const uint32_t keep = keep_of(wbase + wi);
        for (uint32_t bb = word; bb; bb &= bb - 1) {
            const int bit = __ffs(bb) - 1, row = (wbase + wi) * 32 + bit;
            if (((keep >> bit) & 1u) && pos < room) rows[pos++] = row;
            else { if ((keep >> bit) & 1u) ++pos; d.ws.y_acc[row] = __uint_as_float(ACC_CLEAR); }
        }
    }
    cluster.sync();          // (release / acquire at cluster scope: the row list is visible to every block)
    // every thread of the cluster takes result positions in turn: the gathers of a round are independent
    for (int64_t p0 = rank * SMALL_CTA + tid; p0 < room; p0 += (int64_t)SMALL_ILP * SMALL_CLUSTER * SMALL_CTA) {
        int r[SMALL_ILP];
        float v[SMALL_ILP];
#pragma unroll
        for (int u = 0; u < SMALL_ILP; ++u) {
            const int64_t q = p0 + (int64_t)u * SMALL_CLUSTER * SMALL_CTA;
            r[u] = q < room ? __ldcg(rows + q) : -1;
        }
#pragma unroll
        for (int u = 0; u < SMALL_ILP; ++u) v[u] = r[u] >= 0 ? __ldcg(d.ws.y_acc + r[u]) : 0.f;      // (the sums were made by atomics in L2)
#pragma unroll
        for (int u = 0; u < SMALL_ILP; ++u) {
            if (r[u] < 0) continue;
            const int64_t q = p0 + (int64_t)u * SMALL_CLUSTER * SMALL_CTA;
            d.ws.y_acc[r[u]] = __uint_as_float(ACC_CLEAR);
            write(q, r[u], v[u]);
        }
    }
}

}  // namespace dbs

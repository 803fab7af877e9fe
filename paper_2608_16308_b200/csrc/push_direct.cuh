// Push of hypersparse handles: y = A x straight from the listed columns, no worklist in between.
//
// Almost every stored element of such a matrix is an INLINE entry of the block-CSC view, column by
// column, so a push is: for every listed column, its run of entries; for every entry, one atomic
// on the dense accumulator.  Cutting the runs into a worklist in one kernel and walking it in the
// next cost a round trip through global memory, a kernel boundary and the staging of x (R-MAT
// scale 20, x = 1 %: 16 us of a 24.6 us call; this kernel: 5).  Here a thread block takes a share of the listed
// columns, lays their runs end to end with one scan in shared memory and deals the elements out
// evenly over its warps, 32 consecutive ones per warp step and PD_ILP steps in flight: what
// bounds it is the chain x -> column pointers -> entries -> atomic, walked once.
//
//   * LIST: the columns come from the x list itself, in groups of eight spread over the grid (sorted lists
//     put the hub columns side by side); the vector-block masks are set here (structure of x:
//     duplicates, count of nonempty blocks), x is not staged.  Used when the selector is certain to say push.
//   * MASKS: the columns come from the finished vector-block masks and the dense copy of x, 32 words
//     per thread block and round; used when the path is decided on the device (the blocking
//     kernel ran before) and returns at once if the decision was the pull.
//
// A run longer than PD_LONG entries (a hub column of an R-MAT matrix has tens of thousands; left to one
// thread block it was the whole kernel's time) is cut into chunks that go to a list instead, and so is the run of payload entries of a
// listed column's block, a chain of three or four dependent loads each: once per listed column, or, for a longer x on a handle with many of
// them, once per group of four columns (GROUPS; a form of its own: as a branch it cost calls of two short kernels 0.2 us), whose listed ones the second kernel takes from the finished masks; a second kernel, launched
// only on handles that have such runs, deals the chunks out over the warps of the GPU.  Space in the list is claimed with one
// atomic per thread block: an atomic per run was up to eight round trips in one thread, and atomics on one word take
// 1.4 ns each.  (Taking chunks dynamically at the end of the first kernel, from a ticket
// counter or by claiming them one by one, took 10 us longer: 888 thread blocks queueing for 35 chunks.)
//
// The semirings differ in the last line only: (+, *) adds the product, the Boolean one adds 1, (min, +) keeps
// the larger key (minplus.cuh).  Products into hub row blocks go to one of HUB_COPIES private
// accumulators, folded by the finishing kernel (see Device::hub_acc).
#pragma once

#include "internal.cuh"
#include "minplus.cuh"
#include "worklist.cuh"

namespace dbs {

constexpr int PD_WARPS = PD_CTA / 32;
constexpr int PD_ILP = 4;            // warp steps in flight
static_assert(PD_CHUNK % 32 == 0, "whole entries per lane");
constexpr int pd_per_sm(bool masks) { return masks ? 5 : 6; }   // resident thread blocks per SM (registers)
// Mask words of a thread block's round (MASKS): eight threads per word, four columns each.  (Eight columns, four thread blocks per SM: R-MAT scale 20, x = 10 %, 39.7 -> 42.8 us a call.)
constexpr int PD_MASK_WORDS = 32;

// MODE 0: (+, *), 1: Boolean, 2: (min, +)
template <int DT, int MODE>
__device__ __forceinline__ void push_product(const Device &d, uint32_t idx, int r, float a, float xv) {
    const size_t row = (size_t)(idx & IDX_MASK) * 16 + r;
    const bool hub = d.hub_on && (idx & HUB_FLAG);
    float *acc = d.ws.y_acc + row;
    if (hub) {
        const int slot = d.hub_slot[idx & IDX_MASK];
        if (!DBS_CHK_INDEX(d, slot, d.n_hub_blocks)) return;
        acc = d.hub_acc + ((size_t)(blockIdx.x & (d.hub_on - 1)) * d.n_hub_blocks + slot) * 16 + r;
    }
    if (MODE == 2) { atomicMax(reinterpret_cast<int *>(acc), minplus_word(a + xv)); return; }
    const float v = MODE == 1 ? 1.0f : a * xv;
    atomicAdd(acc, v);
    if (MODE == 0 && acc_needs_flag(v)) atomicOr(&d.ws.y_mask32[row >> 5], 1u << (row & 31));
}

template <bool VAL>
__device__ __forceinline__ void push_entry(const Device &d, int p, uint32_t &idx, uint32_t &w, uint32_t &aux) {
    idx = d.csc.idx[p];
    aux = d.csc.aux[p];
    w = VAL ? d.csc.w[p] : 0u;
    DBS_CHK_ENTRY(d, false, idx, w, aux);
}

// Elements (row, col) of the blocks with a payload behind the CSC-view entries first .. first + count - 1: value and row block
// where one is stored.  A half-warp takes an entry, lane = row, U of them side by side: entry, header and
// value are one trip each, for all rows and all entries at once.
template <int DT, int U>
__device__ __forceinline__ void payload_elements(const Device &d, int first, int count, int col, int lane, bool (&in)[U], float (&value)[U], uint32_t (&rb)[U]) {
    const int row = lane & 15;
    uint32_t idx[U], w[U], aux[U];
#pragma unroll
    for (int u = 0; u < U; ++u) {
        const int k = 2 * u + (lane >> 4), p = first + (k < count ? k : 0);
        in[u] = k < count;
        idx[u] = d.csc.idx[p]; w[u] = d.csc.w[p]; aux[u] = d.csc.aux[p];
        DBS_CHK_ENTRY(d, false, idx[u], w[u], aux[u]);
        rb[u] = idx[u] & IDX_MASK;
        value[u] = 1.0f;
    }
    uint32_t m[U], start[U];
#pragma unroll
    for (int u = 0; u < U; ++u) {
        const int type = (int)(idx[u] >> TYPE_SHIFT);
        m[u] = 0u; start[u] = 0u;
        if (type > DBSPMSPV_BLK_COO) {
            const uint8_t *blk = d.payload + (size_t)w[u] * 4;
            const int major = is_row_major(type) ? row : col;
            m[u] = reinterpret_cast<const uint16_t *>(blk)[major];
            if (DT != DBSPMSPV_PATTERN && type != DBSPMSPV_BLK_DENSE) start[u] = blk[32 + major];
        }
    }
#pragma unroll
    for (int u = 0; u < U; ++u) {
        const int type = (int)(idx[u] >> TYPE_SHIFT), minor = is_row_major(type) ? col : row;
        const uint8_t *blk = d.payload + (size_t)w[u] * 4;
        if (type > DBSPMSPV_BLK_COO) {
            in[u] = in[u] && ((m[u] >> minor) & 1u);
            if (DT != DBSPMSPV_PATTERN && in[u])
                value[u] = type == DBSPMSPV_BLK_DENSE ? Val<DT>::load(blk + 32, col * 16 + row)
                                                      : Val<DT>::load(blk + HDR_BYTES, start[u] + __popc(m[u] & ((1u << minor) - 1u)));
        } else if (type == DBSPMSPV_BLK_COO) {             // (only with forced formats)
            const int nnz = (int)aux[u] + 1;
            bool found = false;
            for (int k = 0; k < nnz && in[u]; ++k)
                if (blk[k] == (uint32_t)(row << 4 | col)) { value[u] = Val<DT>::load(blk + ((nnz + 3) & ~3), k); found = true; break; }
            in[u] = in[u] && found;
        } else {                                           // (only in the range-checked build: a replaced entry)
            value[u] = Val<DT>::inline_value(w[u]);
            in[u] = in[u] && (int)(aux[u] & 15) == col && (int)(aux[u] >> 4) == row;
        }
    }
}

// The blocks with a payload behind the CSC-view entries first .. first + count - 1 (at most 2 U, all of one column block) against
// the listed ones of four of its columns, 4 group .. 4 group + 3.  A half-warp takes an entry, lane = row, U of them side by side: entry, header
// and (two columns at a time) values are one trip each for all rows and all entries; a lane's products end in one atomic.
template <int DT, int MODE, int U>
__device__ __forceinline__ void payload_rows(const Device &d, int first, int count, int group, int lane) {
    constexpr bool VAL = DT != DBSPMSPV_PATTERN && MODE != 1;
    const int row = lane & 15, c0 = 4 * (group & 3);
    const uint32_t xm = (mask_of(d.ws.x_mask32, group >> 2) >> c0) & 15u;           // warp-uniform
    const float4 x4 = MODE == 1 ? make_float4(1.f, 1.f, 1.f, 1.f) : *reinterpret_cast<const float4 *>(d.ws.x_dense + 4 * (size_t)group);
    const float x[4] = {x4.x, x4.y, x4.z, x4.w};
    uint32_t idx[U], w[U], off[U];               // off: place of the row's value of the four columns, a byte each (before: the entry's aux byte)
    float acc[U];
#pragma unroll
    for (int u = 0; u < U; ++u) {
        const int k = 2 * u + (lane >> 4), p = first + (k < count ? k : 0);
        uint32_t aux = d.csc.aux[p];
        idx[u] = d.csc.idx[p]; w[u] = d.csc.w[p];
        DBS_CHK_ENTRY(d, false, idx[u], w[u], aux);
        off[u] = aux;
        if (k >= count) idx[u] = PAD_IDX;
    }
    uint32_t have = 0u;                          // bits 4 u + k: the row has an element in listed column k of entry u
#pragma unroll
    for (int u = 0; u < U; ++u) {
        const int type = (int)(idx[u] >> TYPE_SHIFT);
        acc[u] = MODE == 2 ? __uint_as_float(ACC_CLEAR) : 0.f;
        if (type <= DBSPMSPV_BLK_COO || type > BLK_CSR_ROWMAJOR) continue;
        const uint8_t *blk = d.payload + (size_t)w[u] * 4;
        const uint16_t *masks = reinterpret_cast<const uint16_t *>(blk);
        uint32_t in = 0u, o = 0u;
        if (is_row_major(type)) {
            const uint32_t m = masks[row], s = VAL ? blk[32 + row] : 0u;
            in = (m >> c0) & 15u;
            o = s + __popc(m & ((1u << c0) - 1u));
            o = (o & 0xFFu) | (o + (in & 1u)) << 8 | (o + __popc(in & 3u)) << 16 | (o + __popc(in & 7u)) << 24;
        } else {
            const uint2 m2 = *reinterpret_cast<const uint2 *>(masks + c0);
            const uint32_t m[4] = {m2.x & 0xFFFFu, m2.x >> 16, m2.y & 0xFFFFu, m2.y >> 16};
            const uint32_t s = VAL && type != DBSPMSPV_BLK_DENSE ? *reinterpret_cast<const uint32_t *>(blk + 32 + c0) : 0u;
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                in |= ((m[k] >> row) & 1u) << k;
                const uint32_t at = type == DBSPMSPV_BLK_DENSE ? (uint32_t)((c0 + k) * 16 + row) : ((s >> (8 * k)) & 0xFFu) + __popc(m[k] & ((1u << row) - 1u));
                o |= (at & 0xFFu) << (8 * k);
            }
        }
        off[u] = o;
        have |= (in & xm) << (4 * u);
        w[u] += (type == DBSPMSPV_BLK_DENSE ? 32 : HDR_BYTES) / 4;
    }
#pragma unroll
    for (int k0 = 0; k0 < 4; k0 += 2) {
        if (!((xm >> k0) & 3u)) continue;        // warp-uniform
        float a[U][2];
        if (VAL)
#pragma unroll
            for (int u = 0; u < U; ++u)
#pragma unroll
                for (int k = 0; k < 2; ++k) {
                    a[u][k] = 0.f;
                    if ((have >> (4 * u + k0 + k)) & 1u) a[u][k] = Val<DT>::load(d.payload + (size_t)w[u] * 4, (off[u] >> (8 * (k0 + k))) & 0xFFu);
                }
        if (MODE != 1)
#pragma unroll
            for (int u = 0; u < U; ++u)
#pragma unroll
                for (int k = 0; k < 2; ++k)
                    if ((have >> (4 * u + k0 + k)) & 1u) {
                        if (MODE == 2) acc[u] = __int_as_float(max(__float_as_int(acc[u]), minplus_word((VAL ? a[u][k] : 1.0f) + x[k0 + k])));
                        else acc[u] += a[u][k] * x[k0 + k];
                    }
    }
    auto put = [&](size_t r, float v) {
        if (MODE == 2) { atomicMax(reinterpret_cast<int *>(d.ws.y_acc) + r, __float_as_int(v)); return; }
        atomicAdd(d.ws.y_acc + r, MODE == 1 ? 1.0f : v);
        if (MODE == 0 && acc_needs_flag(v)) atomicOr(&d.ws.y_mask32[r >> 5], 1u << (r & 31));
    };
#pragma unroll
    for (int u = 0; u < U; ++u) {
        const size_t r0 = (size_t)(idx[u] & IDX_MASK) * 16;
        if ((have >> (4 * u)) & 15u) put(r0 + row, acc[u]);
        if ((int)(idx[u] >> TYPE_SHIFT) != DBSPMSPV_BLK_COO) continue;
        // packed coordinate lists (only with forced formats): the half-warp's lanes share the elements out
        const uint8_t *blk = d.payload + (size_t)w[u] * 4;
        const int nnz = (int)off[u] + 1;
        for (int k = row; k < nnz; k += 16) {
            const int c = (blk[k] & 15) - c0;
            if (c < 0 || c > 3 || !((xm >> c) & 1u)) continue;
            const float v = VAL ? Val<DT>::load(blk + ((nnz + 3) & ~3), k) : 1.0f, xv = c == 0 ? x[0] : c == 1 ? x[1] : c == 2 ? x[2] : x[3];
            put(r0 + (blk[k] >> 4), MODE == 2 ? __int_as_float(minplus_word(v + xv)) : v * xv);
        }
    }
}

template <int DT, int MODE, bool MASKS, bool GROUPS>
__global__ void __launch_bounds__(PD_CTA, pd_per_sm(MASKS))
k_push_direct(Device d, const int32_t *__restrict__ x_idx, const void *__restrict__ x_val, int32_t nnz_x, int validate, float th3,
              int force_path, int cols, int rounds) {
    constexpr int PER = MASKS ? 4 : 1;                 // columns per thread and round
    constexpr int NC = PD_CTA * PER;
    constexpr bool VAL = DT != DBSPMSPV_PATTERN && MODE != 1;
    __shared__ int s_pre[NC + 1];                      // elements before a column of the round
    __shared__ int2 s_run[NC];                         // position of its first entry minus that; its x value
    __shared__ uint16_t s_own[NC * PD_LONG / 32];      // column that owns the first element of a step of 32
    __shared__ int s_cnt[PD_WARPS], s_sum[PD_WARPS], s_rec[PD_WARPS], s_base;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    pdl_wait();
    if (MASKS && select_path(d, th3, force_path) != DBSPMSPV_PATH_PUSH) return;
    Counters *ctr = d.ws.ctr;
    if (blockIdx.x == 0 && tid == 0) ctr->path = DBSPMSPV_PATH_PUSH;
    for (int round = 0; round < rounds; ++round) {
        int first[PER], deg[PER], pfirst = 0, pdeg = 0, col0 = 0;     // INLINE runs of the thread's columns (the first one is col0); payload run of their block
        float xv[PER];
        uint32_t listed = 0;                           // bit k: column col0 + k is listed
        bool newly = false;
#pragma unroll
        for (int k = 0; k < PER; ++k) { first[k] = 0; deg[k] = 0; xv[k] = 1.0f; }
        if (MASKS) {
            const int n_words = (d.nb + 1) / 2;
            const int64_t wi = (int64_t)(round * PD_MASK_WORDS + (tid >> 3)) * gridDim.x + blockIdx.x;
            if (wi < n_words) listed = (d.ws.x_mask32[wi] >> (4 * (tid & 7))) & 15u;
            if (listed) {
                const int j0 = (int)wi * 32 + 4 * (tid & 7);
                const int32_t *cp = d.csc.colptr + 17 * (j0 >> 4) + (j0 & 15);
                int c[5];
#pragma unroll
                for (int k = 0; k < 5; ++k) c[k] = cp[k];
                const float4 v = MODE == 1 ? make_float4(1.f, 1.f, 1.f, 1.f) : *reinterpret_cast<const float4 *>(d.ws.x_dense + j0);
                const float vv[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
                for (int k = 0; k < PER; ++k)
                    if ((listed >> k) & 1u) { first[k] = c[k]; deg[k] = c[k + 1] - c[k]; xv[k] = vv[k]; if (!DBS_CHK_RANGE(d, first[k], deg[k])) deg[k] = 0; }
                if (d.n_payload) { payload_run(d, j0 >> 4, pfirst, pdeg); col0 = j0; }
            }
        } else {
            const int g = tid >> 3;
            const int64_t i = ((int64_t)(round * (cols >> 3) + g) * gridDim.x + blockIdx.x) * 8 + (tid & 7);
            if (g < (cols >> 3) && i < nnz_x) {
                const int j = x_idx[i];
                if (j < 0 || j >= d.n) {
                    ctr->status = DBSPMSPV_ERR_BOUNDS;
                } else {
                    if (MODE != 1 && x_val) {
                        if (DT == DBSPMSPV_BF16) xv[0] = __bfloat162float(static_cast<const __nv_bfloat16 *>(x_val)[i]);
                        else xv[0] = static_cast<const float *>(x_val)[i];
                    }
                    column_run(d, j, first[0], deg[0]);
                    if (d.n_payload) payload_run(d, j >> 4, pfirst, pdeg);
                    const int sh = ((j >> 4) & 1) * 16;
                    const uint32_t old = atomicOr(&d.ws.x_mask32[j >> 5], 1u << (j & 31));
                    newly = ((old >> sh) & 0xFFFFu) == 0;
                    col0 = j;
                    listed = 1u;
                    if ((old >> (j & 31)) & 1u) {         // listed before: contributes once
                        deg[0] = 0; pdeg = 0; listed = 0u;
                        if (validate) ctr->status = DBSPMSPV_ERR_INVALID_ARG;
                    } else if (GROUPS) {
                        if ((old >> (j & 28)) & 15u) pdeg = 0;               // (listed by the thread that came to these four columns first)
                        if (MODE != 1) d.ws.x_dense[j] = xv[0];              // (k_push_long takes x from there)
                    }
                }
            }
        }
        // long runs and the columns' runs of payload entries: chunks for the second kernel
        int n_rec = 0;
        if (d.long_cap) {
#pragma unroll
            for (int k = 0; k < PER; ++k)
                if (deg[k] > PD_LONG) { n_rec += (deg[k] + PD_CHUNK - 1) / PD_CHUNK; deg[k] = -deg[k]; }      // (negative: listed)
            if (pdeg > 0) n_rec += (GROUPS ? 1 : __popc(listed)) * ((pdeg + PD_PAYLOAD - 1) / PD_PAYLOAD);
        }
        // lay the nonempty short runs end to end
        int n_cols = 0, n_elems = 0;
#pragma unroll
        for (int k = 0; k < PER; ++k) { n_cols += deg[k] > 0; n_elems += max(deg[k], 0); }
        int ic = n_cols, is = n_elems, ir = n_rec;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int a = __shfl_up_sync(FULL, ic, o), b = __shfl_up_sync(FULL, is, o), c = __shfl_up_sync(FULL, ir, o);
            if (lane >= o) { ic += a; is += b; ir += c; }
        }
        if (lane == 31) { s_cnt[warp] = ic; s_sum[warp] = is; s_rec[warp] = ir; }
        const int n_new = __syncthreads_count(newly);          // (also: the element loop of the round before is over)
        int c = ic - n_cols, e = is - n_elems, tot_c = 0, tot_e = 0, rec = ir - n_rec, tot_r = 0;
#pragma unroll
        for (int q = 0; q < PD_WARPS; ++q) {
            if (q < warp) { c += s_cnt[q]; e += s_sum[q]; rec += s_rec[q]; }
            tot_c += s_cnt[q];
            tot_e += s_sum[q];
            tot_r += s_rec[q];
        }
        if (tid == 0) {
            if (n_new) atomicAdd(&ctr->n_nzblk, n_new);
            if (tot_e | tot_r) atomicAdd(&ctr->n_tasks, ((tot_e + 31) >> 5) + tot_r);
            s_base = tot_r ? atomicAdd(&ctr->n_long, tot_r) : 0;
            s_pre[tot_c] = tot_e;
        }
#pragma unroll
        for (int k = 0; k < PER; ++k) {
            if (deg[k] <= 0) continue;
            s_pre[c] = e;
            s_run[c] = make_int2(first[k] - e, __float_as_int(xv[k]));
            for (int q = (e + 31) >> 5; q * 32 < e + deg[k]; ++q) s_own[q] = (uint16_t)c;
            ++c;
            e += deg[k];
        }
        __syncthreads();
        if (tot_r) {                                   // block-uniform; a thread's runs are written by its whole warp
            int at = s_base + rec;
#pragma unroll
            for (int k = 0; k < PER; ++k)
                for (uint32_t todo = __ballot_sync(FULL, deg[k] < 0); todo; todo &= todo - 1) {
                    const int src = __ffs(todo) - 1;
                    const int f = __shfl_sync(FULL, first[k], src), n = -__shfl_sync(FULL, deg[k], src), o = __shfl_sync(FULL, at, src);
                    const int xb = __shfl_sync(FULL, __float_as_int(xv[k]), src);
                    const int n_chunks = (n + PD_CHUNK - 1) / PD_CHUNK;
                    for (int q = lane; q < n_chunks; q += 32) d.ws.long_runs[o + q] = make_int4(f + q * PD_CHUNK, min(PD_CHUNK, n - q * PD_CHUNK), xb, 0);
                    if (lane == src) at += n_chunks;
                }
            if (pdeg > 0 && GROUPS)
                for (int q = 0; q < pdeg; q += PD_PAYLOAD) d.ws.long_runs[at++] = make_int4(pfirst + q, min(PD_PAYLOAD, pdeg - q), col0 >> 2, 0x100);
            else if (pdeg > 0)
#pragma unroll
                for (int k = 0; k < PER; ++k)
                    if ((listed >> k) & 1u)
                        for (int q = 0; q < pdeg; q += PD_PAYLOAD) d.ws.long_runs[at++] = make_int4(pfirst + q, min(PD_PAYLOAD, pdeg - q), __float_as_int(xv[k]), 0x100 | ((col0 + k) & 15));
        }
        for (int s0 = warp * 32; s0 < tot_e; s0 += PD_CTA * PD_ILP) {
            uint32_t idx[PD_ILP], w[PD_ILP], aux[PD_ILP];
            float xs[PD_ILP];
#pragma unroll
            for (int u = 0; u < PD_ILP; ++u) {
                const int e0 = s0 + u * PD_CTA;
                idx[u] = PAD_IDX; w[u] = 0u; aux[u] = 0u; xs[u] = 0.f;
                if (e0 < tot_e) {                   // warp-uniform
                    // the step's first owner, then every lane's own from the run boundaries inside the step (the runs are not empty)
                    const int lo = s_own[e0 >> 5];
                    const uint32_t b = (uint32_t)(s_pre[min(lo + 1 + lane, tot_c)] - e0);
                    const uint32_t m = __reduce_or_sync(FULL, b < 32u ? 1u << b : 0u);
                    if (e0 + lane < tot_e) {
                        const int2 run = s_run[lo + __popc(m & ((2u << lane) - 1u))];
                        xs[u] = __int_as_float(run.y);
                        push_entry<VAL>(d, run.x + e0 + lane, idx[u], w[u], aux[u]);
                    }
                }
            }
#pragma unroll
            for (int u = 0; u < PD_ILP; ++u)
                if (idx[u] < (1u << TYPE_SHIFT)) push_product<DT, MODE>(d, idx[u], (int)(aux[u] >> 4), Val<DT>::inline_value(w[u]), xs[u]);
        }
    }
}

// The listed chunks, a warp at a time; the next chunk's record is fetched a round ahead.
// (Nothing is listed when the path decided on the device is the pull.)
// Where the path is decided on the device and the matrix is small, the streaming pull, launched in any case, takes them when the decision was the push: a launch less
// (R-MAT 20 K rows, x = 30 %: 14.5 -> 12.6 us a call; 40 K vertices, masked, 10 %: 15.7 -> 15.0; 256 K rows, 10 %: 22.1 -> 21.1; with 16 to 31 M entries, where
// the warps of its one thread block per SM are too few, up to 1 % longer, and payload runs of four columns 8 %).
constexpr int LONG_IN_PULL_ENTRIES = 8 << 20;
template <int DT, int MODE, bool GROUPS>
__device__ __forceinline__ void push_long_chunks(const Device &d, int gwarp, int nwarps) {
    constexpr bool VAL = DT != DBSPMSPV_PATTERN && MODE != 1;
    constexpr int U = PD_CHUNK / 32;
    const int lane = threadIdx.x & 31;
    const int n = min(d.ws.ctr->n_long, d.long_cap);
    int4 next = gwarp < n ? d.ws.long_runs[gwarp] : make_int4(0, 0, 0, 0);
    for (int i = gwarp; i < n; i += nwarps) {
        const int4 run = next;
        if (i + nwarps < n) next = d.ws.long_runs[i + nwarps];
        if (!DBS_CHK_RANGE(d, run.x, run.y)) continue;
        const float xs = __int_as_float(run.z);
        if (GROUPS && run.w) {                         // payload entries, four columns (warp-uniform)
            if (DBS_CHK_INDEX(d, run.z, 4 * (int64_t)d.nb)) payload_rows<DT, MODE, PD_PAYLOAD / 2>(d, run.x, run.y, run.z, lane);
            continue;
        }
        if (!GROUPS && run.w) {                        // payload entries, one column: a half-warp each
            bool in[PD_PAYLOAD / 2];
            float a[PD_PAYLOAD / 2];
            uint32_t rb[PD_PAYLOAD / 2];
            payload_elements<DT, PD_PAYLOAD / 2>(d, run.x, run.y, run.w & 15, lane, in, a, rb);
#pragma unroll
            for (int u = 0; u < PD_PAYLOAD / 2; ++u)
                if (in[u]) push_product<DT, MODE>(d, rb[u], lane & 15, a[u], xs);
            continue;
        }
        uint32_t idx[U], w[U], aux[U];
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const int k = u * 32 + lane;
            idx[u] = PAD_IDX; w[u] = 0u; aux[u] = 0u;
            if (k < run.y) push_entry<VAL>(d, run.x + k, idx[u], w[u], aux[u]);
        }
#pragma unroll
        for (int u = 0; u < U; ++u)
            if (idx[u] < (1u << TYPE_SHIFT)) push_product<DT, MODE>(d, idx[u], (int)(aux[u] >> 4), Val<DT>::inline_value(w[u]), xs);
    }
}

template <int DT, int MODE, bool GROUPS>
__global__ void __launch_bounds__(PD_CTA, 6) k_push_long(Device d) {
    pdl_wait();
    push_long_chunks<DT, MODE, GROUPS>(d, (int)(blockIdx.x * PD_CTA + threadIdx.x) >> 5, (int)(gridDim.x * PD_CTA) >> 5);
}

}  // namespace dbs

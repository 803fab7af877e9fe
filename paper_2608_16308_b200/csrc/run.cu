// One SpMSpV call (Sections 3.3 and 4.1): vector blocking, device-side path selection, push / pull
// traversal with per-block microkernels, hierarchical writeback, and one finishing kernel that turns
// the dense accumulator into a sorted sparse y.  (Hypersparse handles push straight from the listed columns,
// push_direct.cuh; the others through a worklist.)  Also the dense-in / dense-out
// decode entry (Section 4.3).  Nothing here allocates device memory or synchronises, except db_sssp
// (one launch, sssp.cuh, or a host loop over (min, +) products, at the end of the file).
#include "internal.cuh"
#include "call_graph.cuh"
#include "microkernels.cuh"
#include "staging.cuh"
#include "worklist.cuh"
#include "mma_block.cuh"

namespace dbs {

// ------------------------------------------------------------------------------------------
// Output of a traversal.  The sparse path accumulates into the handle's dense accumulator (see
// ACC_CLEAR); the decode path adds straight into the caller's y.
// ------------------------------------------------------------------------------------------
struct OutSparse {
    float *acc;
    uint32_t *flag32;  // bits of the rows that a tiny sum reached
    static constexpr bool MASKS = true;
    static constexpr bool MINPLUS = false;
};
struct OutDense {
    float *acc;
    uint32_t *flag32;
    static constexpr bool MASKS = false;
    static constexpr bool MINPLUS = false;
};
// (min, +) semiring: the accumulator holds words of the smallest sum so far (minplus.cuh)
struct OutSparseMin {
    float *acc;
    uint32_t *flag32;
    static constexpr bool MASKS = true;
    static constexpr bool MINPLUS = true;
};
template <typename Out> __device__ __forceinline__ void out_add(Out out, size_t row, float v) {
    atomicAdd(out.acc + row, v);
    if (Out::MASKS && acc_needs_flag(v)) atomicOr(out.flag32 + (row >> 5), 1u << (row & 31));
}
}
#include "lean_pull.cuh"
#include "push_direct.cuh"

namespace dbs {

constexpr int CTA = 128;            // four warps per thread block (Section 3.3.2)
constexpr int WARPS = CTA / 32;
constexpr int XB_TPB = 512;         // vector blocking of a sparse x: threads per block
constexpr int CMP_TPB = 256;        // finishing kernel: threads per tile
constexpr int TILE_WORDS = CMP_TPB / 4;  // a tile: 64 mask words = 2048 rows, 8 rows per thread

// ------------------------------------------------------------------------------------------
// Vector blocking (Section 3.2.2) of a sparse x: one thread per listed nonzero scatters the value
// into the dense copy and sets its mask bit.
// EMIT (handles whose elements sit mostly in blocks with a payload: banded matrices, pruned
// layers): fused with the push worklist (Section 3.3.2) -- the thread that turns a vector block from
// empty to nonempty emits the push tasks of its whole block-CSC column (runs of <= 32 entries; the
// INLINE elements among them are filtered by the mask in the traversal).  Space in the worklist is
// claimed with a warp scan, a sum over the thread block's warps and one atomic per thread
// block; the count of nonempty vector blocks is aggregated the same way (Section 4.1).
// Without EMIT: the dense copy, the masks and the count only -- hypersparse handles whose path is
// decided on the device; the direct push then takes its columns from the masks.
// ------------------------------------------------------------------------------------------
template <int DT, bool EMIT>
__global__ void k_xblock_sparse(Device d, const int32_t *__restrict__ x_idx, const void *__restrict__ x_val,
                                int32_t nnz_x, int validate) {
    pdl_wait();
    const int t = blockIdx.x * blockDim.x + threadIdx.x;
    const int lane = threadIdx.x & 31;
    bool newly = false;
    int jb = 0, first = 0, end = 0;
    if (t < nnz_x) {
        const int j = x_idx[t];
        // an index outside [0, n) is never written through: the entry is skipped and the call
        // reports ERR_BOUNDS (the compare is free next to the dependent scatter)
        if (j < 0 || j >= d.n) {
            d.ws.ctr->status = DBSPMSPV_ERR_BOUNDS;
        } else {
            float v = 1.0f;
            if (x_val) {
                if (DT == DBSPMSPV_BF16) v = __bfloat162float(static_cast<const __nv_bfloat16 *>(x_val)[t]);
                else v = static_cast<const float *>(x_val)[t];
            }
            // a listed NaN that happens to carry the marker's bit pattern is stored as the
            // canonical quiet NaN, so the marker itself never appears as data
            d.ws.x_dense[j] = __float_as_uint(v) == X_ABSENT ? __uint_as_float(0x7FC00000u) : v;
            jb = j >> 4;
            // (fetched before the atomic whose result decides whether it is needed)
            if (EMIT) { first = d.csc.ptr[jb]; end = d.csc.ptr[jb + 1]; }
            const int sh = (jb & 1) * 16;
            const uint32_t old = atomicOr(&d.ws.x_mask32[j >> 5], 1u << ((j & 15) + sh));
            newly = ((old >> sh) & 0xFFFFu) == 0;
            if (validate && ((old >> ((j & 15) + sh)) & 1u)) d.ws.ctr->status = DBSPMSPV_ERR_INVALID_ARG;   // optional check: duplicate index
        }
    }
    emit_tasks<true>(d, newly, jb, first, EMIT && newly ? end - first : 0, lane, &d.ws.ctr->n_tasks, &d.ws.ctr->n_nzblk, PUSH_CHUNK,
                     EMIT ? &d.ws.ctr->n_hubs : nullptr, d.ws.hubs);
}


// Dense input (Sections 4.1, 4.3): every warp reads 32 elements, one ballot gives the two
// 16-bit masks of its two vector blocks.  Also clears the dense output.
// Which entries of a dense activation vector take part in a decode call: |x_j| > tau, or, with
// the ReLU fused in, x_j > tau (tau = 0: x_j not zero / positive).  A NaN always takes part.
__device__ __forceinline__ bool decode_takes_part(const Device &d, float v) {
    return d.decode_relu ? !(v <= d.decode_tau) : !(fabsf(v) <= d.decode_tau);
}

template <int DT>
__global__ void k_xblock_dense(Device d, const void *__restrict__ x, float *__restrict__ y) {
    pdl_wait();
    const int lane = threadIdx.x & 31;
    const int64_t padded = (int64_t)((d.nb + 1) / 2) * 32;
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t j = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; j < padded; j += stride) {
        float v = 0.f;
        if (j < d.n) {
            if (DT == DBSPMSPV_BF16 && !d.decode_x_f32) v = __bfloat162float(static_cast<const __nv_bfloat16 *>(x)[j]);
            else v = static_cast<const float *>(x)[j];
            if (DT == DBSPMSPV_BF16 && d.decode_x_f32) v = __bfloat162float(__float2bfloat16_rn(v));
        }
        const bool in = j < d.n && decode_takes_part(d, v);
        if (j < (int64_t)d.nb * 16)
            d.ws.x_dense[j] = in ? (__float_as_uint(v) == X_ABSENT ? __uint_as_float(0x7FC00000u) : v)
                                 : __uint_as_float(X_ABSENT);
        const uint32_t bits = __ballot_sync(FULL, in);
        if (lane == 0) d.ws.x_mask32[j >> 5] = bits;
        const bool newly = (lane == 0 && (bits & 0xFFFFu)) || (lane == 16 && (bits >> 16));
        int first = 0, deg = 0;
        const bool listed = in && j < d.n;
        if (d.payload_chunk == PUSH_CHUNK) {                 // whole column blocks, as in the sparse-x kernel
            if (newly) { first = d.csc.ptr[j >> 4]; deg = d.csc.ptr[(j >> 4) + 1] - first; }
            emit_tasks(d, newly, (int)(j >> 4), first, deg, lane, &d.ws.ctr->n_tasks, &d.ws.ctr->n_nzblk, PUSH_CHUNK, &d.ws.ctr->n_hubs, d.ws.hubs);
            continue;
        }
        if (listed) column_run(d, (int)j, first, deg);
        merge_column_runs(listed, (int)j, first, deg, lane);
        emit_tasks(d, newly, (int)(j >> 4), first, deg, lane, &d.ws.ctr->n_tasks, &d.ws.ctr->n_nzblk, PUSH_CHUNK, &d.ws.ctr->n_hubs, d.ws.hubs);
        first = 0; deg = 0;
        if (newly) payload_run(d, (int)(j >> 4), first, deg);
        if (__any_sync(FULL, deg > 0))
            emit_tasks(d, false, (int)(j >> 4), first, deg, lane, &d.ws.ctr->n_tasks, &d.ws.ctr->n_nzblk, d.payload_chunk);
    }
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < d.m; i += stride) y[i] = 0.f;
}

// ------------------------------------------------------------------------------------------
// Traversal.
// ------------------------------------------------------------------------------------------
// One lane owns one hypersparse block (INLINE or COO).  `emit(r, v)` receives the products,
// already summed per row where the entries of a row are adjacent (COO is stored row-major);
// `xin` is the x entry of an INLINE block's single column (fetched by the caller in parallel
// with the mask); `xb` points at the 16 x entries of the block's vector block.  Returns the
// structural-hit row mask.
template <int DT, typename Emit>
__device__ __forceinline__ uint32_t lane_block(int type, uint32_t w, uint32_t aux, uint32_t xm,
                                               float xin, const float *xb, const uint8_t *payload,
                                               Emit emit) {
    uint32_t hit = 0;
    if (type == DBSPMSPV_BLK_INLINE) {
        if ((xm >> (aux & 15)) & 1u) {
            if (DT != DBSPMSPV_PATTERN) emit((int)(aux >> 4), Val<DT>::inline_value(w) * xin);
            hit = 1u << (aux >> 4);
        }
    } else {
        const int nnz = (int)aux + 1;
        const uint8_t *blk = payload + (size_t)w * 4;
        const uint32_t *cw = reinterpret_cast<const uint32_t *>(blk);
        const uint8_t *vals = blk + ((nnz + 3) & ~3);
        int cur = -1;
        float s = 0.f;
        for (int k0 = 0; k0 < nnz; k0 += 4) {
            uint32_t word = cw[k0 >> 2];
            const int lim = min(4, nnz - k0);
            for (int j = 0; j < lim; ++j, word >>= 8) {
                const int c = word & 15, r = (word >> 4) & 15;
                if ((xm >> c) & 1u) {
                    if (DT != DBSPMSPV_PATTERN) {
                        if (r != cur) { if (cur >= 0) emit(cur, s); cur = r; s = 0.f; }
                        s += Val<DT>::load(vals, k0 + j) * xb[c];
                    }
                    hit |= 1u << r;
                }
            }
        }
        if (DT != DBSPMSPV_PATTERN && cur >= 0) emit(cur, s);
    }
    return hit;
}

// The COO blocks held by the 32 lanes of a warp, processed as ONE flat list of stored entries:
// a warp scan of the per-lane entry counts lays the entries out, then every lane takes one
// entry per step and finds its owner block by a shuffle binary search over the scan.  This
// keeps all lanes busy whatever the mix of block sizes (a lane looping over its own block
// would make the whole warp wait for the largest block).  `cnt` is the lane's entry count
// (0 = no COO block here); `tag0`, `tag1` are per-block values handed back to
// `emit(tag0, tag1, r, c, value, owner_lane)` for every entry whose column is active.
template <int DT, typename Emit>
__device__ __forceinline__ void warp_flat_coo(int cnt, uint32_t w, uint32_t xm, uint32_t tag0, uint32_t tag1,
                                              const uint8_t *payload, int lane, Emit emit) {
    int incl = cnt;
    for (int o = 1; o < 32; o <<= 1) {
        int t = __shfl_up_sync(FULL, incl, o);
        if (lane >= o) incl += t;
    }
    const int total = __shfl_sync(FULL, incl, 31);
    for (int e0 = 0; e0 < total; e0 += 32) {
        const int e = e0 + lane;
        int o = 0;
#pragma unroll
        for (int s = 16; s; s >>= 1) {
            const int v = __shfl_sync(FULL, incl, o + s - 1);
            if (v <= e) o += s;
        }
        const int bn = __shfl_sync(FULL, cnt, o);
        const int k = e - (__shfl_sync(FULL, incl, o) - bn);
        const uint32_t bw = __shfl_sync(FULL, w, o);
        const uint32_t bxm = __shfl_sync(FULL, xm, o);
        const uint32_t bt0 = __shfl_sync(FULL, tag0, o);
        const uint32_t bt1 = __shfl_sync(FULL, tag1, o);
        if (e < total) {
            const uint8_t *blk = payload + (size_t)bw * 4;
            const uint32_t rc = blk[k];
            const int c = rc & 15, r = rc >> 4;
            if ((bxm >> c) & 1u) emit(bt0, bt1, r, c, Val<DT>::load(blk + ((bn + 3) & ~3), k), o);
        }
    }
}

// Structural hits of a pattern block: a count per row instead of a sum.
template <typename Out>
__device__ __forceinline__ void mark_rows(Out out, int rb, uint32_t rows16) {
    for (; rows16; rows16 &= rows16 - 1) out_add(out, (size_t)rb * 16 + __ffs(rows16) - 1, 1.0f);
}

// Writeback of one block handled outside the shared-memory accumulator: lanes 0..15 own the 16
// rows; one global atomic per touched row.
template <int DT, typename Out>
__device__ __forceinline__ void flush_rows(Out out, int rb, uint32_t hits, float v, int lane) {
    if (lane < 16 && ((hits >> lane) & 1u)) out_add(out, (size_t)rb * 16 + lane, DT != DBSPMSPV_PATTERN ? v : 1.0f);
}

// Per-warp staging area in shared memory: two stages of view entries for the pull; the push
// uses the same bytes as one stage for the payload of a task's blocks.
struct PullStage {
    uint32_t idx[STAGE_CAP];
    uint32_t w[STAGE_CAP];
    uint8_t aux[STAGE_CAP];
};
struct PullWarp {
    PullStage stage[2];
    uint64_t bar[2];
};

// Push (Section 3.3.2): every warp takes one task = up to PUSH_CHUNK consecutive block-CSC
// entries of one active column block (32 per step, all fetched up front); the vector block is staged once per task (Section 3.3.3).  Lanes
// own hypersparse blocks; heavier blocks are then processed by the whole warp one at a time.
// Writeback: warp-level reduction, then one global atomic per touched row and one atomicOr on
// the row block's hit mask.  The task record carries its length, so the view entries, the mask
// and the x block are all fetched in one round of independent loads.
template <int DT, typename Out, bool HV>
__device__ void push_body(const Device &d, Out out, int popc_threshold, float *s_x, float *s_tmp, float *s_lacc, PullWarp *pw) {
    constexpr int U = PUSH_CHUNK / 32;
    const int lane = threadIdx.x & 31;
    const int gwarp = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int nwarps = (gridDim.x * blockDim.x) >> 5;
    static_assert(U == 1, "one warp step per task");
    const int n_recs = d.ws.ctr->n_tasks, n_hubs = min(d.ws.ctr->n_hubs, HUB_CAP);
    const HubTable hubs = load_hub_table(d.ws.hubs, n_hubs, lane);
    const int n_tasks = n_recs + hubs.total;                       // task records, then the steps of the hub runs
    auto item = [&](int i) { return worklist_item(d.ws.tasks, n_recs, hubs, i); };
    // A task is a chain of dependent loads (record -> entries, column end, mask, x block); the
    // loop is software-pipelined: while task k is evaluated, the loads of k+1 and the record of
    // k+2 (in this warp's stride) are in flight.
    struct Loads { uint32_t idx, w, aux, xm; float xv; int start, end, jb; };
    auto loads_of = [&](int t, const uint2 &task) {
        Loads l{0u, 0u, 0u, 0u, 0.f, 0, 0, 0};
        if (t < n_tasks) {
            const int jb = (int)(task.x & IDX_MASK);
            l.jb = jb;
            const int cnt = (int)(task.x >> 27) + 1;              // entries of the task
            l.start = (int)task.y;
            if (lane < cnt && DBS_CHK_RANGE(d, l.start, cnt) && DBS_CHK_INDEX(d, jb, d.nb)) {
                const int p = l.start + lane; l.idx = d.csc.idx[p]; l.w = d.csc.w[p]; l.aux = d.csc.aux[p];
                DBS_CHK_ENTRY(d, false, l.idx, l.w, l.aux);
            }
            l.end = l.start + cnt;
            l.xm = mask_of(d.ws.x_mask32, jb);
            if (lane < 16) l.xv = d.ws.x_dense[jb * 16 + lane];
        }
        return l;
    };
    const uint2 none = make_uint2(0u, 0u);
    uint2 rec1 = gwarp + nwarps < n_tasks ? item(gwarp + nwarps) : none;
    Loads cur = loads_of(gwarp, gwarp < n_tasks ? item(gwarp) : none);
    // Payload staging (Section 3.3.3) on handles whose elements sit mostly in blocks with a payload:
    // when the payload of all blocks of a task fits the warp's staging area, every lane moves its
    // block there with one bulk copy and the microkernels read shared memory.  The point is the
    // bytes in flight: 32 blocks per warp at once instead of the two a half-warp pair walks
    // (header -> values, two dependent trips each) -- at 14 warps per SM the latter keeps about
    // 6 KB per SM in flight where the memory system wants 35.  (A second area per warp, so that
    // the next task's copies fly while this one is computed, was measured slower: the shared
    // memory it takes costs a resident thread block per SM.)
    constexpr int STAGE_AREA = (int)sizeof(PullStage) * 2;
    uint32_t stage_parity = 0u;
    // issues the copies of one task; returns the lane's byte offset in the area, or -1 (not staged)
    auto stage_issue = [&](const Loads &l) {
        const bool have = l.start + lane < l.end;
        const int type = l.idx >> TYPE_SHIFT;
        const int bytes = have && type != DBSPMSPV_BLK_INLINE ? payload_words(type, (int)l.aux + 1, Val<DT>::SIZE) * 4 : 0;
        int incl = bytes;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int v = __shfl_up_sync(FULL, incl, o);
            if (lane >= o) incl += v;
        }
        const int total = __shfl_sync(FULL, incl, 31);
        if (total <= 0 || total > STAGE_AREA) return -1;          // warp-uniform
        uint8_t *area = reinterpret_cast<uint8_t *>(pw->stage);
        if (lane == 0) mbar_arrive_expect_tx(&pw->bar[0], (uint32_t)total);
        __syncwarp();
        if (bytes) bulk_copy_g2s(area + incl - bytes, d.payload + (size_t)l.w * 4, (uint32_t)bytes, &pw->bar[0]);
        return incl - bytes;
    };
    if (HV) {
        if (lane == 0) { mbar_init(&pw->bar[0], 1); fence_barrier_init(); }
        __syncwarp();
    }
    for (int t = gwarp; t < n_tasks; t += nwarps) {
        const uint2 rec2 = t + 2 * nwarps < n_tasks ? item(t + 2 * nwarps) : none;
        const Loads nxt = loads_of(t + nwarps, rec1);
        rec1 = rec2;
        const int off_cur = HV ? stage_issue(cur) : -1;         // (the area is free: the last task's reads ended at the warp barrier)
        uint32_t idx[U] = {cur.idx}, w[U] = {cur.w}, aux[U] = {cur.aux};
        const int start = cur.start, end = cur.end, jb = cur.jb;
        const uint32_t xm = cur.xm;
        if (lane < 16) s_x[lane] = cur.xv;
        cur = nxt;
        __syncwarp();
#pragma unroll
        for (int u = 0; u < U; ++u) {
            if (start + u * 32 >= end) break;                 // warp-uniform
            const bool have = start + u * 32 + lane < end;
            bool heavy = false;
            int coo_cnt = 0;
            const int type = idx[u] >> TYPE_SHIFT;
            const int brow = idx[u] & IDX_MASK;
            const uint8_t *pl = d.payload;        // where this task's payload is read from (w[u] counts 4-byte words from it)
            if (HV && off_cur >= 0) {            // warp-uniform: this task's payload was staged
                if (!mbar_wait_bounded(&pw->bar[0], stage_parity)) {
                    // (never seen; the copies in flight get a second, equally bounded chance to land before the warp leaves)
                    d.ws.ctr->status = DBSPMSPV_ERR_TIMEOUT;
                    mbar_wait_bounded(&pw->bar[0], stage_parity);
                    return;
                }
                stage_parity ^= 1u;
                pl = reinterpret_cast<const uint8_t *>(pw->stage);
                if (have && type != DBSPMSPV_BLK_INLINE) w[u] = (uint32_t)off_cur >> 2;
            }
            if (have) {
                if (type == DBSPMSPV_BLK_INLINE) {
                    const uint32_t hit = lane_block<DT>(type, w[u], aux[u], xm, s_x[aux[u] & 15], s_x, pl,
                                                        [&](int r, float v) { out_add(out, (size_t)brow * 16 + r, v); });
                    if (DT == DBSPMSPV_PATTERN) mark_rows(out, brow, hit);
                } else if (type == DBSPMSPV_BLK_COO && aux[u] < COO_SERIAL_MAX) {
                    coo_cnt = (int)aux[u] + 1;
                } else {
                    heavy = true;
                }
            }
            if (__any_sync(FULL, coo_cnt)) {
                warp_flat_coo<DT>(coo_cnt, w[u], xm, (uint32_t)brow, 0u, pl, lane,
                                  [&](uint32_t tag, uint32_t, int r, int c, float a, int) {
                                      out_add(out, (size_t)tag * 16 + r, DT != DBSPMSPV_PATTERN ? a * s_x[c] : 1.0f);
                                  });
                __syncwarp();
            }
            // dense vector block and several mask-based blocks in the step: half-warp streaming
            // form (two blocks per warp at a time, next pair prefetched; a warp that takes one
            // block at a time waits out two dependent loads per block)
            if (HV && DT != DBSPMSPV_PATTERN && __popc(xm) >= popc_threshold) {
                const bool mk = heavy && type != DBSPMSPV_BLK_COO;
                const uint32_t cs = __ballot_sync(FULL, mk);
                if (__popc(cs) >= HEAVY_LANE_MIN) {
                    auto emit = [&](int erb, int erow, float esum) {
                        out_add(out, (size_t)erb * 16 + erow, esum);
                    };
                    const uint32_t rows = __ballot_sync(FULL, mk && is_row_major(type));
                    const uint32_t tagged = (idx[u] & ~IDX_MASK) | (uint32_t)jb;     // class bits + the task's column block
                    if (cs & ~rows) half_stream<DT, false>(pl, d.ws.x_dense, tagged, w[u], xm, brow, cs & ~rows, lane, emit);
                    if (rows) half_stream<DT, true>(pl, d.ws.x_dense, tagged, w[u], xm, brow, rows, lane, emit);
                    if (mk) heavy = false;
                    __syncwarp();
                }
            }
            uint32_t hv = __ballot_sync(FULL, heavy);
            // sparse local mask -> lane-owned form; dense local mask -> warp form (Section 3.3.3:
            // the number of active entries of the vector block picks the microkernel)
            const bool lane_form = heavy && type != DBSPMSPV_BLK_COO && __popc(xm) < popc_threshold;
            const uint32_t hv_mask = HV ? __ballot_sync(FULL, lane_form) : 0u;
            if (HV && __popc(hv_mask) >= HEAVY_LANE_MIN) {
                // many mask-based blocks side by side: every lane walks its own block
                if (lane_form) {
                    const uint8_t *blk = pl + (size_t)w[u] * 4;
                    float *acc = s_lacc + lane;
                    uint32_t hits;
                    if (DT == DBSPMSPV_PATTERN) {
                        hits = lane_heavy_bool(type, blk, xm);
                    } else {
#pragma unroll
                        for (int r = 0; r < 16; ++r) acc[r * LANE_ACC_STRIDE] = 0.f;
                        hits = lane_heavy<DT>(type, blk, xm, s_x, acc);
                    }
                    for (uint32_t hh = hits; hh; hh &= hh - 1) {
                        const int r = __ffs(hh) - 1;
                        out_add(out, (size_t)brow * 16 + r, DT != DBSPMSPV_PATTERN ? acc[r * LANE_ACC_STRIDE] : 1.0f);
                    }
                }
                __syncwarp();
                hv &= ~hv_mask;   // oversized COO blocks (forced format) stay with the warp form
            }
            while (hv) {
                const int src = __ffs(hv) - 1;
                hv &= hv - 1;
                const uint32_t bidx = __shfl_sync(FULL, idx[u], src);
                const uint32_t bw = __shfl_sync(FULL, w[u], src);
                const int nnz = (int)__shfl_sync(FULL, aux[u], src) + 1;
                const int btype = bidx >> TYPE_SHIFT;
                const int bbrow = bidx & IDX_MASK;
                const uint8_t *blk = pl + (size_t)bw * 4;
                uint32_t hits;
                float sum = 0.f;
                if (DT == DBSPMSPV_PATTERN) hits = warp_block_bool<DT>(btype, blk, nnz, xm, lane);
                else sum = warp_block<DT>(btype, blk, nnz, xm, s_x, s_tmp, lane, popc_threshold, hits);
                flush_rows<DT>(out, bbrow, hits, sum, lane);
            }
        }
        __syncwarp();
    }
}

// Pull (Section 3.3.2).  The block-CSR view is streamed through shared memory: every warp owns
// a double-buffered stage (Section 3.3.3) that one lane fills with three bulk copies (index,
// word and aux arrays of one chunk of consecutive segments) while the warp works on the other
// stage.  Inside a chunk the lanes run over the entries 32 at a time, whatever segment they
// belong to: the first entry of every segment carries a flag bit, so a ballot and a popcount
// give each lane its segment, hence its row block.  Writeback is hierarchical where it pays:
// the segment the warp is currently "in" accumulates its 16 partial sums in shared memory
// (long hub row blocks stay there over many steps); products of the other, short segments met
// in the same step go straight to global atomics.  INLINE entries need one gather only: the
// dense copy of x carries a "not listed" marker, so presence and value come from one load.
#ifndef DBS_PULL_UNROLL
#define DBS_PULL_UNROLL 2
#endif
constexpr int PULL_UNROLL = DBS_PULL_UNROLL;
#ifndef DBS_SY_COPIES
#define DBS_SY_COPIES 4
#endif
constexpr int SY_COPIES = DBS_SY_COPIES;  // copies of the pull accumulator per warp (power of two, <= 32)
constexpr uint32_t SEG_FLAG = 1u << 28;   // view entry starts a pull segment (block-CSR view only)

// lane 0 issues the copies of the chunk [e0, e1) into stage st
__device__ __forceinline__ void pull_issue(const Device &d, int e0, int e1, PullStage *st, uint64_t *bar, int lane) {
    const int a0 = e0 & ~15, a1 = (e1 + 15) & ~15;
    if (lane == 0 && e1 > e0 && DBS_CHK_RANGE(d, e0, e1 - e0)) {      // same condition as the consumer's wait
        const uint32_t n = (uint32_t)(a1 - a0);
        fence_proxy_async_smem();
        mbar_arrive_expect_tx(bar, n * 9u);
        bulk_copy_g2s(st->idx, d.csr.idx + a0, n * 4u, bar);
        bulk_copy_g2s(st->w, d.csr.w + a0, n * 4u, bar);
        bulk_copy_g2s(st->aux, d.csr.aux + a0, n, bar);
    }
}

template <int DT, typename Out, bool HV>
__device__ void pull_body(const Device &d, Out out, int popc_threshold, float *s_x, float *s_tmp,
                          float *s_y, float *s_lacc, PullWarp *pw) {
    const int lane = threadIdx.x & 31;
    const uint32_t le_mask = 0xFFFFFFFFu >> (31 - lane);
    const int gwarp = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int nwarps = (gridDim.x * blockDim.x) >> 5;
    if (lane == 0) { mbar_init(&pw->bar[0], 1); mbar_init(&pw->bar[1], 1); fence_barrier_init(); }
    // the shared accumulator is kept in SY_COPIES copies, each fed by its own group of lanes:
    // fewer lanes per address means fewer retries of the shared-memory fp32 atomic
    for (int k = lane; k < 16 * SY_COPIES; k += 32) s_y[k] = 0.f;
    float *const my_y = s_y + (lane / (32 / SY_COPIES)) * 16;
    __syncwarp();
    uint32_t parity = 0u;             // bit s: phase parity of stage s
    int cur = 0;
    bool next_in_flight = false;
    int2 c0 = make_int2(0, 0), c1 = c0, n0 = c0, n1 = c0;
    if (gwarp < d.n_chunks) {
        c0 = d.chunks[gwarp]; c1 = d.chunks[gwarp + 1];
        pull_issue(d, c0.y, c1.y, &pw->stage[0], &pw->bar[0], lane);
    }
    if (gwarp + nwarps < d.n_chunks) { n0 = d.chunks[gwarp + nwarps]; n1 = d.chunks[gwarp + nwarps + 1]; }
    for (int c = gwarp; c < d.n_chunks; c += nwarps) {
        const int e0 = c0.y, e1 = c1.y, a0 = e0 & ~15;
        int ord_base = c0.x - 1;          // segment of the entry just before the current step
        // prefetch: next chunk's copies, and the descriptor of the one after
        const int cn = c + nwarps;
        next_in_flight = cn < d.n_chunks;
        if (next_in_flight) pull_issue(d, n0.y, n1.y, &pw->stage[cur ^ 1], &pw->bar[cur ^ 1], lane);
        c0 = n0; c1 = n1;
        if (cn + nwarps < d.n_chunks) { n0 = d.chunks[cn + nwarps]; n1 = d.chunks[cn + nwarps + 1]; }
        if (e1 > e0) {
            if (!mbar_wait_bounded(&pw->bar[cur], (parity >> cur) & 1u)) {
                d.ws.ctr->status = DBSPMSPV_ERR_TIMEOUT;
                break;
            }
            parity ^= 1u << cur;
        }
        const PullStage *st = &pw->stage[cur];
        int cur_rb = -1;                  // row block held in the shared accumulator
        int last_rb = -1;                 // row block of segment ord_base
        uint32_t hit = 0;
        for (int base = e0; base < e1; base += 32 * PULL_UNROLL) {
            uint32_t idx[PULL_UNROLL], w[PULL_UNROLL], aux[PULL_UNROLL];
            float xin[PULL_UNROLL];
#pragma unroll
            for (int u = 0; u < PULL_UNROLL; ++u) {
                const int p = base + u * 32 + lane;
                idx[u] = 0; w[u] = 0; aux[u] = 0;
                if (p < e1) { const int o = p - a0; idx[u] = st->idx[o]; w[u] = st->w[o]; aux[u] = st->aux[o]; DBS_CHK_ENTRY(d, true, idx[u], w[u], aux[u]); }
            }
#pragma unroll
            for (int u = 0; u < PULL_UNROLL; ++u) {
                const bool have = base + u * 32 + lane < e1;
                // (L2-only load: the 4-byte gathers hit L1 one time in ten and only evict each other there)
                xin[u] = have ? __ldcg(&d.ws.x_dense[(size_t)(idx[u] & IDX_MASK) * 16 + (aux[u] & 15)])
                             : __uint_as_float(X_ABSENT);
            }
#pragma unroll
            for (int u = 0; u < PULL_UNROLL; ++u) {
                if (base + u * 32 >= e1) break;   // warp-uniform
                const bool have = base + u * 32 + lane < e1;
                const uint32_t fb = __ballot_sync(FULL, (idx[u] & SEG_FLAG) != 0u);   // idx is 0 past the end
                // Most steps lie inside one segment (long row blocks are cut into segments of whole
                // steps): then the row block is warp-uniform and known without a per-lane lookup.
                const bool one_seg = (fb & ~1u) == 0u;
                int rb, rb0;
                if (one_seg) {
                    if (fb) last_rb = d.seg_rb[++ord_base];
                    rb = rb0 = last_rb;
                } else {
                    const int ord = ord_base + __popc(fb & le_mask);
                    ord_base += __popc(fb);
                    rb = have ? d.seg_rb[ord] : 0;
                    rb0 = __shfl_sync(FULL, rb, 0);
                    last_rb = __shfl_sync(FULL, rb, 31);   // (past the end only in the chunk's last step)
                }
                // the shared accumulator follows the row block of the step's first entry (a long
                // row block keeps it over all its segments of the chunk)
                if (rb0 != cur_rb) {
                    hit = __reduce_or_sync(FULL, hit);
                    __syncwarp();
                    if (lane < 16) {
                        if ((hit >> lane) & 1u) {
                            float t = DT != DBSPMSPV_PATTERN ? 0.f : 1.0f;
                            if (DT != DBSPMSPV_PATTERN) {
#pragma unroll
                                for (int k = 0; k < SY_COPIES; ++k) { t += s_y[k * 16 + lane]; s_y[k * 16 + lane] = 0.f; }
                            }
                            out_add(out, (size_t)cur_rb * 16 + lane, t);
                        }
                    }
                    hit = 0;
                    cur_rb = rb0;
                    __syncwarp();
                }
                const int type = idx[u] >> TYPE_SHIFT;
                const bool inl = type == DBSPMSPV_BLK_INLINE;
                if (inl && __float_as_uint(xin[u]) != X_ABSENT) {    // absent also covers "past the end"
                    const float v = Val<DT>::inline_value(w[u]) * xin[u];
                    const int r = aux[u] >> 4;
                    if (one_seg || rb == cur_rb) {
                        if (DT != DBSPMSPV_PATTERN) atomicAdd(&my_y[r], v);
                        hit |= 1u << r;
                    } else {
                        out_add(out, (size_t)rb * 16 + r, DT != DBSPMSPV_PATTERN ? v : 1.0f);
                    }
                }
                const bool other = have && !inl;
                if (!__any_sync(FULL, other)) continue;
                // classes that go through the vector-block mask; they write straight to global
                const int bcol_l = idx[u] & IDX_MASK;
                const uint32_t xm = other ? mask_of(d.ws.x_mask32, bcol_l) : 0u;
                bool heavy = false;
                int coo_cnt = 0;
                if (xm) {
                    if (type == DBSPMSPV_BLK_COO && aux[u] < COO_SERIAL_MAX) {
                        coo_cnt = (int)aux[u] + 1;
                    } else {
                        heavy = true;
                    }
                }
                if (__any_sync(FULL, coo_cnt)) {
                    warp_flat_coo<DT>(coo_cnt, w[u], xm, (uint32_t)rb, (uint32_t)bcol_l, d.payload, lane,
                                      [&](uint32_t trb, uint32_t tcol, int r, int c, float a, int) {
                                          out_add(out, (size_t)trb * 16 + r, DT != DBSPMSPV_PATTERN ? a * d.ws.x_dense[(size_t)tcol * 16 + c] : 1.0f);
                                      });
                    __syncwarp();
                }
                // runs of mask-based blocks (pruned layers, banded matrices): half-warp streaming form
                if (HV && DT != DBSPMSPV_PATTERN) {
                    const bool mk = heavy && type != DBSPMSPV_BLK_COO;
                    const uint32_t cs = __ballot_sync(FULL, mk);
                    if (__popc(cs) >= HEAVY_LANE_MIN) {
                        auto emit = [&](int erb, int erow, float esum) {
                            if (erb == cur_rb) {
                                atomicAdd(&my_y[erow], esum);
                                hit |= 1u << erow;
                            } else {
                                out_add(out, (size_t)erb * 16 + erow, esum);
                            }
                        };
                        const uint32_t rows = __ballot_sync(FULL, mk && is_row_major(type));
                        if (cs & ~rows) half_stream<DT, false>(d.payload, d.ws.x_dense, idx[u], w[u], xm, rb, cs & ~rows, lane, emit);
                        if (rows) half_stream<DT, true>(d.payload, d.ws.x_dense, idx[u], w[u], xm, rb, rows, lane, emit);
                        if (mk) heavy = false;
                        __syncwarp();
                    }
                }
                uint32_t hv = __ballot_sync(FULL, heavy);
                // sparse local mask -> lane-owned form; dense local mask -> warp form
                const bool lane_form = heavy && type != DBSPMSPV_BLK_COO && __popc(xm) < popc_threshold;
                const uint32_t hv_mask = HV ? __ballot_sync(FULL, lane_form) : 0u;
                if (HV && __popc(hv_mask) >= HEAVY_LANE_MIN) {
                    // Mask-based blocks side by side under sparse local masks (banded matrices at
                    // run ends): every lane walks its own block and leaves 16 partial sums in its
                    // private scratch column, so the warp keeps up to 32 blocks going.  Blocks of
                    // the row block held in the shared accumulator are then summed across lanes
                    // by 16 lanes (no atomics); blocks of other row blocks go straight to global.
                    float *acc = s_lacc + lane;
                    uint32_t hits = 0;
                    if (lane_form) {
                        const uint8_t *blk = d.payload + (size_t)w[u] * 4;
                        if (DT == DBSPMSPV_PATTERN) {
                            hits = lane_heavy_bool(type, blk, xm);
                        } else {
#pragma unroll
                            for (int r = 0; r < 16; ++r) acc[r * LANE_ACC_STRIDE] = 0.f;
                            hits = lane_heavy<DT>(type, blk, xm, d.ws.x_dense + (size_t)bcol_l * 16, acc);
                        }
                    }
                    const bool in_cur = lane_form && rb == cur_rb;
                    const uint32_t members = __ballot_sync(FULL, in_cur);
                    __syncwarp();
                    if (in_cur) hit |= hits;
                    if (DT != DBSPMSPV_PATTERN && members && lane < 16) {
                        float t = 0.f;
                        for (uint32_t mm = members; mm; mm &= mm - 1) t += s_lacc[lane * LANE_ACC_STRIDE + __ffs(mm) - 1];
                        s_y[lane] += t;
                    }
                    if (lane_form && !in_cur) {
                        for (uint32_t hh = hits; hh; hh &= hh - 1) {
                            const int r = __ffs(hh) - 1;
                            out_add(out, (size_t)rb * 16 + r, DT != DBSPMSPV_PATTERN ? acc[r * LANE_ACC_STRIDE] : 1.0f);
                        }
                    }
                    __syncwarp();
                    hv &= ~hv_mask;
                }
                while (hv) {
                    const int src = __ffs(hv) - 1;
                    hv &= hv - 1;
                    const uint32_t bidx = __shfl_sync(FULL, idx[u], src);
                    const uint32_t bw = __shfl_sync(FULL, w[u], src);
                    const int nnz = (int)__shfl_sync(FULL, aux[u], src) + 1;
                    const uint32_t bxm = __shfl_sync(FULL, xm, src);
                    const int brb = __shfl_sync(FULL, rb, src);
                    const int btype = bidx >> TYPE_SHIFT;
                    const int bcol = bidx & IDX_MASK;
                    const uint8_t *blk = d.payload + (size_t)bw * 4;
                    uint32_t hits;
                    float sum = 0.f;
                    if (DT == DBSPMSPV_PATTERN) {
                        hits = warp_block_bool<DT>(btype, blk, nnz, bxm, lane);
                    } else {
                        __syncwarp();
                        if (lane < 16) s_x[lane] = d.ws.x_dense[(size_t)bcol * 16 + lane];
                        __syncwarp();
                        sum = warp_block<DT>(btype, blk, nnz, bxm, s_x, s_tmp, lane, popc_threshold, hits);
                    }
                    flush_rows<DT>(out, brb, hits, sum, lane);
                }
            }
        }
        // end of the chunk: flush what the shared accumulator still holds
        hit = __reduce_or_sync(FULL, hit);
        __syncwarp();
        if (lane < 16) {
            if ((hit >> lane) & 1u) {
                float t = DT != DBSPMSPV_PATTERN ? 0.f : 1.0f;
                if (DT != DBSPMSPV_PATTERN) {
#pragma unroll
                    for (int k = 0; k < SY_COPIES; ++k) { t += s_y[k * 16 + lane]; s_y[k * 16 + lane] = 0.f; }
                }
                out_add(out, (size_t)cur_rb * 16 + lane, t);
            }
        }
        __syncwarp();
        cur ^= 1;
        next_in_flight = false;
    }
    // left early on a timeout: let the copy still in flight land before the stage memory is
    // given back (bounded, like every wait here)
    if (next_in_flight) mbar_wait_bounded(&pw->bar[cur ^ 1], (parity >> (cur ^ 1)) & 1u);
}
#ifndef DBS_MIN_CTAS
#define DBS_MIN_CTAS 1
#endif
// (MODE 1: five resident thread blocks per SM -- a cap of 102 registers -- measured 7 - 10 % faster
// than the compiler's own 107 registers and four thread blocks once the push stages its payload)
#ifndef DBS_MIN_CTAS_HEAVY
#define DBS_MIN_CTAS_HEAVY 5
#endif
// Variants of the traversal kernel, chosen per handle from the class census at create:
//   MODE 0  hypersparse matrices (power-law graphs): the push only -- their pull is the
//           streaming kernel k_pull_lean, launched next in the stream
//   MODE 1  matrices whose elements sit mostly in mask-based blocks (pruned layers, banded
//           matrices): half-warp streaming and lane-owned microkernels
// Dynamic shared memory: per-warp pull stages (the push stages payload there) | lane scratch of the lane-owned form (MODE 1).
template <int MODE> constexpr size_t compute_dyn_smem() {
    return MODE >= 1 ? WARPS * sizeof(PullWarp) + WARPS * 16 * LANE_ACC_STRIDE * sizeof(float) : 0;
}

template <int DT, typename Out, int MODE>
__global__ void __launch_bounds__(CTA, MODE >= 1 ? DBS_MIN_CTAS_HEAVY : DBS_MIN_CTAS) k_compute(Device d, Out out, float th3, int force_path, int popc_threshold, int pull_done) {
    constexpr bool HV = MODE >= 1;
    __shared__ float s_x[WARPS][16], s_tmp[WARPS][32], s_y[HV ? WARPS : 1][16 * SY_COPIES];
    extern __shared__ __align__(128) uint8_t s_dyn[];
    PullWarp *s_pull = reinterpret_cast<PullWarp *>(s_dyn);
    float *s_lacc = reinterpret_cast<float *>(s_dyn + WARPS * sizeof(PullWarp));
    const int warp = threadIdx.x >> 5;
    pdl_wait();
    const int path = select_path(d, th3, force_path);
    if (blockIdx.x == 0 && threadIdx.x == 0) d.ws.ctr->path = path;
    float *lacc = HV ? s_lacc + warp * 16 * LANE_ACC_STRIDE : nullptr;
    if (pull_done && path == DBSPMSPV_PATH_PULL) return;     // (the decode entry's own pull kernel has run)
    if (path == DBSPMSPV_PATH_PUSH) push_body<DT, Out, HV>(d, out, popc_threshold, s_x[warp], s_tmp[warp], lacc, HV ? &s_pull[warp] : nullptr);
    else if (HV) pull_body<DT, Out, HV>(d, out, popc_threshold, s_x[warp], s_tmp[warp], s_y[warp], lacc, &s_pull[warp]);
    // (MODE 0: the pull is k_pull_lean's)
}

// Pull of the decode entry for matrices whose elements sit mostly in mask-based blocks (pruned
// layers).  A warp takes 32 consecutive entries of the block-CSR view, one block per lane.  A
// lane walks the active columns of its own column-major or Dense block and keeps the 16 row sums
// in registers (a Dense column is two 16-byte loads for bf16); with activations 10 % dense a block
// has one or two active columns, and a step serves 32 blocks with the instructions the half-warp
// form spends on two.  When the 32 entries share a row block -- always, for the layer shapes of
// Section 4.3 -- the 32 x 16 sums are folded by 16 shuffles into one atomic per row; otherwise every
// lane adds its own.  Row-major blocks take the half-warp streaming form, the odd COO/INLINE
// entry its own lane.  Does nothing unless the selector says pull; the general
// kernel, launched next, then only runs the push.
#ifndef DBS_LBC
#define DBS_LBC 3
#endif
constexpr int LBC = DBS_LBC;              // columns of a lane's block per pass of lane_block_columns
constexpr int LBC_SLOT_BYTES = 48;  // staging slot of a lane: 32 bytes used; the stride keeps 16-byte stores conflict-free

// Active columns of one column-major (or Dense) block, by the lane that owns it: acc[r] += A[r][c] x[c].
// The loads of up to LBC columns are issued together, level by level (x and header, then the
// values), so a pass costs two memory latencies whatever the number of columns.  bf16 values
// come in as two 16-byte loads per column -- with 32 lanes on 32 different cache lines a load
// instruction costs the same whatever its width, so element-wise loads were 8 times the L1 work.
// A compressed column (its values packed in row order from a 2-byte aligned start) is then
// expanded to its rows through the lane's own 48 bytes of shared memory: the 32 aligned bytes
// that hold it are stored there and each row with a set mask bit reads the next 2 bytes.  No
// other lane touches the slot, so no barrier is involved.
template <int DT>
__device__ __forceinline__ void lane_block_columns(const uint8_t *blk, bool dense, uint32_t xm, const float *xb,
                                                   float (&acc)[16], uint4 *slot) {
    const uint16_t *masks = reinterpret_cast<const uint16_t *>(blk);
    for (uint32_t a = xm; a;) {
        int c[LBC];
        bool on[LBC];
        float xs[LBC];
        uint32_t mc[LBC];
        int pos[LBC];
#pragma unroll
        for (int j = 0; j < LBC; ++j) { on[j] = a != 0; c[j] = on[j] ? __ffs(a) - 1 : 0; a &= a - 1; }
#pragma unroll
        for (int j = 0; j < LBC; ++j) {
            xs[j] = 0.f; mc[j] = 0u; pos[j] = 0;
            if (on[j]) {
                xs[j] = xb[c[j]];
                if (!dense) { mc[j] = masks[c[j]]; pos[j] = blk[32 + c[j]]; }
            }
        }
        if (DT == DBSPMSPV_BF16) {
            uint4 lo[LBC], hi[LBC];
            int off[LBC];          // halfword offset of the column's first value inside lo|hi
#pragma unroll
            for (int j = 0; j < LBC; ++j) {
                lo[j] = make_uint4(0u, 0u, 0u, 0u); hi[j] = lo[j]; off[j] = 0;
                if (on[j]) {
                    const int byte0 = dense ? 32 + c[j] * 32 : HDR_BYTES + ((pos[j] * 2) & ~15);
                    off[j] = dense ? 0 : pos[j] & 7;
                    const uint4 *src = reinterpret_cast<const uint4 *>(blk + byte0);
                    lo[j] = src[0]; hi[j] = src[1];       // (the payload has slack behind its last block)
                }
            }
#pragma unroll
            for (int j = 0; j < LBC; ++j) {
                if (!on[j]) continue;
                if (dense) {
                    // absent elements are stored as zeros: only a non-finite x needs the mask
                    uint32_t gate = 0xFFFFu;
                    if ((__float_as_uint(xs[j]) & 0x7F800000u) == 0x7F800000u) gate = masks[c[j]];
                    const uint32_t u[8] = {lo[j].x, lo[j].y, lo[j].z, lo[j].w, hi[j].x, hi[j].y, hi[j].z, hi[j].w};
#pragma unroll
                    for (int q = 0; q < 8; ++q) {
                        const float v0 = __uint_as_float(u[q] << 16), v1 = __uint_as_float(u[q] & 0xFFFF0000u);
                        if ((gate >> (2 * q)) & 1u) acc[2 * q] += v0 * xs[j];
                        if ((gate >> (2 * q + 1)) & 1u) acc[2 * q + 1] += v1 * xs[j];
                    }
                } else if (off[j] + __popc(mc[j]) <= 16) {
                    slot[0] = lo[j]; slot[1] = hi[j];
                    asm volatile("" ::: "memory");
                    const uint16_t *sv = reinterpret_cast<const uint16_t *>(slot) + off[j];
                    int i = 0;
#pragma unroll
                    for (int r = 0; r < 16; ++r)
                        if ((mc[j] >> r) & 1u) { acc[r] += __uint_as_float((uint32_t)sv[i] << 16) * xs[j]; ++i; }
                    asm volatile("" ::: "memory");
                } else {
                    // the column straddles the 32 staged bytes: element-wise
                    const uint8_t *vals = blk + HDR_BYTES;
                    int i = pos[j];
#pragma unroll
                    for (int r = 0; r < 16; ++r)
                        if ((mc[j] >> r) & 1u) { acc[r] += Val<DT>::load(vals, i) * xs[j]; ++i; }
                }
            }
        } else {
            const uint8_t *vals = blk + (dense ? 32 : HDR_BYTES);
#pragma unroll
            for (int j = 0; j < LBC; ++j) {
                if (!on[j]) continue;
                if (dense) {
                    uint32_t gate = 0xFFFFu;
                    if ((__float_as_uint(xs[j]) & 0x7F800000u) == 0x7F800000u) gate = masks[c[j]];
#pragma unroll
                    for (int r = 0; r < 16; ++r)
                        if ((gate >> r) & 1u) acc[r] += Val<DT>::load(vals, c[j] * 16 + r) * xs[j];
                } else {
                    int i = pos[j];
#pragma unroll
                    for (int r = 0; r < 16; ++r)
                        if ((mc[j] >> r) & 1u) { acc[r] += Val<DT>::load(vals, i) * xs[j]; ++i; }
                }
            }
        }
    }
}

// Sum of acc[r] over the 32 lanes, for all 16 rows: afterwards the lane pair (2k, 2k + 1) holds
// the total of row folded_row(lane).
__device__ __forceinline__ float fold_rows(const float (&acc)[16], int lane) {
    float a8[8], a4[4], a2[2];
    const bool u16 = lane & 16, u8 = lane & 8, u4 = lane & 4, u2 = lane & 2;
#pragma unroll
    for (int i = 0; i < 8; ++i) a8[i] = (u16 ? acc[i + 8] : acc[i]) + __shfl_xor_sync(FULL, u16 ? acc[i] : acc[i + 8], 16);
#pragma unroll
    for (int i = 0; i < 4; ++i) a4[i] = (u8 ? a8[i + 4] : a8[i]) + __shfl_xor_sync(FULL, u8 ? a8[i] : a8[i + 4], 8);
#pragma unroll
    for (int i = 0; i < 2; ++i) a2[i] = (u4 ? a4[i + 2] : a4[i]) + __shfl_xor_sync(FULL, u4 ? a4[i] : a4[i + 2], 4);
    const float a1 = (u2 ? a2[1] : a2[0]) + __shfl_xor_sync(FULL, u2 ? a2[0] : a2[1], 2);
    return a1 + __shfl_xor_sync(FULL, a1, 1);
}
__device__ __forceinline__ int folded_row(int lane) { return ((lane >> 4) & 1) * 8 + ((lane >> 3) & 1) * 4 + ((lane >> 2) & 1) * 2 + ((lane >> 1) & 1); }

template <int DT>
__global__ void __launch_bounds__(CTA) k_decode_pull(Device d, const int32_t *__restrict__ entry_row,
                                                     float *__restrict__ y, float th3, int force_path) {
    __shared__ __align__(16) uint8_t s_slots[CTA * LBC_SLOT_BYTES];
    pdl_wait();
    if (select_path(d, th3, force_path) != DBSPMSPV_PATH_PULL) return;
    if (blockIdx.x == 0 && threadIdx.x == 0) d.ws.ctr->path = DBSPMSPV_PATH_PULL;
    const int lane = threadIdx.x & 31;
    uint4 *slot = reinterpret_cast<uint4 *>(s_slots + threadIdx.x * LBC_SLOT_BYTES);
    const int gwarp = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int nwarps = (gridDim.x * blockDim.x) >> 5;
    const int n_tasks = (d.n_entries + 31) >> 5;
    auto emit = [&](int erb, int erow, float esum) { atomicAdd(y + (size_t)erb * 16 + erow, esum); };
    for (int task = gwarp; task < n_tasks; task += nwarps) {
        const int p = task * 32 + lane;
        const bool have = p < d.n_entries;
        uint32_t idx = 0, w = 0, aux = 0, xm = 0;
        int rb = -1;
        if (have) {
            idx = d.csr.idx[p]; w = d.csr.w[p]; aux = d.csr.aux[p]; rb = entry_row[p];
            DBS_CHK_ENTRY(d, true, idx, w, aux);
            if (!DBS_CHK_INDEX(d, rb, d.mb)) rb = 0;
            xm = mask_of(d.ws.x_mask32, idx & IDX_MASK);
        }
        const int type = idx >> TYPE_SHIFT;
        const bool mk = have && xm && type > DBSPMSPV_BLK_COO;
        const bool rowm = mk && is_row_major(type);
        const float *xb = d.ws.x_dense + (size_t)(idx & IDX_MASK) * 16;
        float acc[16];
#pragma unroll
        for (int r = 0; r < 16; ++r) acc[r] = 0.f;
        if (mk && !rowm) lane_block_columns<DT>(d.payload + (size_t)w * 4, type == DBSPMSPV_BLK_DENSE, xm, xb, acc, slot);
        __syncwarp();
        const int rb0 = __shfl_sync(FULL, rb, 0);
        if (__all_sync(FULL, rb == rb0)) {
            const float total = fold_rows(acc, lane);
            if (!(lane & 1) && total != 0.f) atomicAdd(y + (size_t)rb0 * 16 + folded_row(lane), total);
        } else if (mk && !rowm) {
#pragma unroll
            for (int r = 0; r < 16; ++r)
                if (acc[r] != 0.f) atomicAdd(y + (size_t)rb * 16 + r, acc[r]);
        }
        const uint32_t rows = __ballot_sync(FULL, rowm);
        if (rows) half_stream<DT, true>(d.payload, d.ws.x_dense, idx, w, xm, rb, rows, lane, emit);
        if (have && xm && type <= DBSPMSPV_BLK_COO) {       // the odd hypersparse block: its own lane
            float *row0 = y + (size_t)rb * 16;
            if (type == DBSPMSPV_BLK_INLINE) {
                if ((xm >> (aux & 15)) & 1u) atomicAdd(row0 + (aux >> 4), Val<DT>::inline_value(w) * xb[aux & 15]);
            } else {
                const int nnz = (int)aux + 1;
                const uint8_t *blk = d.payload + (size_t)w * 4, *vals = blk + ((nnz + 3) & ~3);
                for (int k = 0; k < nnz; ++k) {
                    const int c = blk[k] & 15, r = blk[k] >> 4;
                    if ((xm >> c) & 1u) atomicAdd(row0 + r, Val<DT>::load(vals, k) * xb[c]);
                }
            }
        }
    }
}

// Active columns of the column-major and Dense blocks of one warp step, when all 32 blocks lie in
// ONE row block: then any lane may take any (block, column) pair -- its 16 sums go into the
// same rows -- and the pairs are dealt out evenly, 32 per round, instead of every lane walking
// the columns of its own block (with activations 10 % dense a block has 1.6 active columns on
// average but the busiest of 32 has five).  `cols` is the lane's own block's active-column mask
// (0: not a block of these classes).  Column values are fetched and expanded as in
// lane_block_columns, Dense columns through the same staged form.
// WC_ILP = (block, column) pairs a lane works on at a time: 2 where a warp has several steps per
// row block (wide layers: measured 45 -> 41 us on 4096 x 11008), 1 where it has one or two
// (12288 x 4096: 2 measured 10 % slower).
__host__ __device__ constexpr int wc_ilp(int warps_per_block) { return warps_per_block >= 8 ? 2 : 1; }
// staging bytes per lane; the stride keeps 16-byte stores conflict-free
__host__ __device__ constexpr int wc_slot_bytes(int ilp) { return 48 * ilp + (ilp > 1 ? 16 : 0); }

// DIRECT: the payload lies in shared memory, so the values are indexed where they are (no staging slot).
template <int DT, int WC_ILP, bool DIRECT = false>
__device__ __forceinline__ void warp_columns(const uint8_t *payload, const float *x_blocks, uint32_t idx, uint32_t w,
                                             uint32_t cols, int lane, float (&acc)[16], uint4 *slot) {
    int incl = __popc(cols);
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int t = __shfl_up_sync(FULL, incl, o);
        if (lane >= o) incl += t;
    }
    const int excl = incl - __popc(cols);
    const int total = __shfl_sync(FULL, incl, 31);
    for (int k0 = 0; k0 < total; k0 += 32 * WC_ILP) {
        // WC_ILP pairs per lane and round, worked on side by side: their dependent loads (header ->
        // values -> staged expansion) overlap
        bool on[WC_ILP], dense[WC_ILP];
        uint32_t m[WC_ILP], bidx[WC_ILP], bw[WC_ILP], gate[WC_ILP];
        int j[WC_ILP], pos[WC_ILP];
        float xv[WC_ILP];
        const uint8_t *blk[WC_ILP];
#pragma unroll
        for (int u = 0; u < WC_ILP; ++u) {
            const int k = k0 + 32 * u + lane;
            int b = 0;                   // owner of pair k: the last lane whose exclusive prefix is <= k
#pragma unroll
            for (int s = 16; s; s >>= 1) {
                const int t = __shfl_sync(FULL, excl, b + s);
                if (t <= k) b += s;
            }
            m[u] = __shfl_sync(FULL, cols, b);
            j[u] = k - __shfl_sync(FULL, excl, b);
            bidx[u] = __shfl_sync(FULL, idx, b);
            bw[u] = __shfl_sync(FULL, w, b);
            on[u] = k < total;
        }
#pragma unroll
        for (int u = 0; u < WC_ILP; ++u) {
            gate[u] = 0u; pos[u] = 0; xv[u] = 0.f; dense[u] = false; blk[u] = payload;
            if (on[u]) {
                uint32_t mm = m[u];
                for (int t = 0; t < j[u]; ++t) mm &= mm - 1;
                const int c = __ffs(mm) - 1;   // the j-th active column of that block
                dense[u] = (bidx[u] >> TYPE_SHIFT) == DBSPMSPV_BLK_DENSE;
                blk[u] = payload + (size_t)bw[u] * 4;
                xv[u] = x_blocks[(size_t)(bidx[u] & IDX_MASK) * 16 + c];
                // absent elements of a Dense block are stored as zeros: only a non-finite x needs its mask
                const bool finite = (__float_as_uint(xv[u]) & 0x7F800000u) != 0x7F800000u;
                gate[u] = dense[u] && finite ? 0xFFFFu : reinterpret_cast<const uint16_t *>(blk[u])[c];
                pos[u] = dense[u] ? c * 16 : blk[u][32 + c];
            }
        }
        if (DT == DBSPMSPV_BF16 && !DIRECT) {
            int off[WC_ILP];
#pragma unroll
            for (int u = 0; u < WC_ILP; ++u) {
                off[u] = pos[u] & 7;
                if (on[u]) {
                    const int nvals = dense[u] ? 16 : __popc(gate[u]);
                    const uint4 *src = reinterpret_cast<const uint4 *>(blk[u] + (dense[u] ? 32 : HDR_BYTES) + ((pos[u] * 2) & ~15));
                    const uint4 zero = make_uint4(0u, 0u, 0u, 0u);
                    const uint4 q0 = src[0], q1 = off[u] + nvals > 8 ? src[1] : zero, q2 = off[u] + nvals > 16 ? src[2] : zero;
                    slot[3 * u] = q0; slot[3 * u + 1] = q1; slot[3 * u + 2] = q2;
                }
            }
            asm volatile("" ::: "memory");
            int i[WC_ILP];
#pragma unroll
            for (int u = 0; u < WC_ILP; ++u) i[u] = 0;
#pragma unroll
            for (int r = 0; r < 16; ++r) {
#pragma unroll
                for (int u = 0; u < WC_ILP; ++u) {
                    const uint16_t *sv = reinterpret_cast<const uint16_t *>(slot + 3 * u) + off[u];
                    const uint32_t bit = (gate[u] >> r) & 1u;
                    if (bit) acc[r] += __uint_as_float((uint32_t)sv[i[u]] << 16) * xv[u];
                    i[u] += (int)bit | (dense[u] ? 1 : 0);
                }
            }
            asm volatile("" ::: "memory");
        } else {
#pragma unroll
            for (int u = 0; u < WC_ILP; ++u) {
                const uint8_t *vals = blk[u] + (dense[u] ? 32 : HDR_BYTES);
                int i = pos[u];
#pragma unroll
                for (int r = 0; r < 16; ++r) {
                    const uint32_t bit = (gate[u] >> r) & 1u;
                    if (bit) acc[r] += Val<DT>::load(vals, i) * xv[u];
                    i += (int)bit | (dense[u] ? 1 : 0);
                }
            }
        }
    }
}

// x -> 16-bit masks and fp32 blocks in shared memory (absent entries carry the marker), by all
// `threads` threads of the block; s_cnt[0] and s_cnt[1] (zeroed by the caller, barrier in
// between) receive the numbers of nonzero vector blocks and of nonzero elements.  The caller synchronises afterwards.
template <int DT>
__device__ __forceinline__ void stage_x_blocks(const Device &d, const void *__restrict__ x, float *s_x, uint16_t *s_xm,
                                               int *s_cnt, int tid, int T) {
    const int lane = tid & 31;
    const bool aligned = (reinterpret_cast<uintptr_t>(x) & 15u) == 0;
    // (a bf16 handle may be given its x in fp32 -- the fp32 output of the layer before --, which
    // is rounded to bf16 here, to nearest even, so that the products stay exact)
    const bool x16 = DT == DBSPMSPV_BF16 && !d.decode_x_f32;
    int mine = 0;
    for (int cb = tid; cb < d.nb; cb += T) {
        const int64_t j0 = (int64_t)cb * 16;
        float v[16];
        if (aligned && j0 + 16 <= d.n) {
            if (x16) {
                const uint4 *src = reinterpret_cast<const uint4 *>(static_cast<const uint16_t *>(x) + j0);
                const uint4 a = src[0], b = src[1];
                const uint32_t u[8] = {a.x, a.y, a.z, a.w, b.x, b.y, b.z, b.w};
#pragma unroll
                for (int q = 0; q < 8; ++q) { v[2 * q] = __uint_as_float(u[q] << 16); v[2 * q + 1] = __uint_as_float(u[q] & 0xFFFF0000u); }
            } else {
                const float4 *src = reinterpret_cast<const float4 *>(static_cast<const float *>(x) + j0);
#pragma unroll
                for (int q = 0; q < 4; ++q) { const float4 f = src[q]; v[4 * q] = f.x; v[4 * q + 1] = f.y; v[4 * q + 2] = f.z; v[4 * q + 3] = f.w; }
            }
        } else {
#pragma unroll
            for (int k = 0; k < 16; ++k) {
                v[k] = 0.f;
                if (j0 + k < d.n) v[k] = x16 ? __uint_as_float((uint32_t) static_cast<const uint16_t *>(x)[j0 + k] << 16)
                                             : static_cast<const float *>(x)[j0 + k];
            }
        }
        uint32_t bits = 0;
#pragma unroll
        for (int k = 0; k < 16; ++k) {
            if (DT == DBSPMSPV_BF16 && !x16) v[k] = __bfloat162float(__float2bfloat16_rn(v[k]));
            const bool nz = decode_takes_part(d, v[k]);
            bits |= (nz ? 1u : 0u) << k;
            // (a widened bf16 has zero low bits: it cannot collide with the marker)
            if (DT != DBSPMSPV_BF16 && __float_as_uint(v[k]) == X_ABSENT) v[k] = __uint_as_float(0x7FC00000u);
            v[k] = nz ? v[k] : __uint_as_float(X_ABSENT);
        }
        float4 *dst = reinterpret_cast<float4 *>(s_x + j0);
#pragma unroll
        for (int q = 0; q < 4; ++q) dst[q] = make_float4(v[4 * q], v[4 * q + 1], v[4 * q + 2], v[4 * q + 3]);
        s_xm[cb] = (uint16_t)bits;
        mine += (bits != 0) | (__popc(bits) << 16);           // nonzero blocks, nonzero elements
    }
    mine = __reduce_add_sync(FULL, mine);
    if (lane == 0 && mine) { atomicAdd(&s_cnt[0], mine & 0xFFFF); atomicAdd(&s_cnt[1], mine >> 16); }
}

// Streaming reads the whole payload whatever x holds; the single-kernel form above fetches only
// the columns x reaches, which is less than half of the bytes once x has fewer nonzero elements
// than this share (measured on the three layer shapes: 22.6 against 27.6 us at 10 %, 37.9
// against 33.8 us at 30 %).  The choice follows the x of the handle's previous decode call --
// both kernels report the number of nonzero elements they saw through a word of mapped host
// memory, read without waiting: activations of one layer keep their sparsity from token to token.
constexpr float STREAM_MIN_X_DENSITY = 0.15f;

// The whole decode call in one kernel, for payload-dominated handles whose x fits in shared
// memory (Section 4.3: one layer, one token).  One thread block per row block.  Every block
// first reads the dense activation vector itself -- a few KB -- into shared memory as the
// vector-block masks and the fp32 x blocks the microkernels expect, counts the nonzero vector
// blocks and evaluates the selector; nothing of that touches the handle's workspace, so there
// is no blocking kernel before and no cleanup after.
//   pull: the warps take the row block's view entries 32 at a time, one block per lane (see
//         k_decode_pull);
//   push: the lanes take the nonzero vector blocks instead and look their column block up in
//         the row block's entries (sorted by column block) by bisection, so only blocks under a
//         nonzero vector block are fetched.
// The 16 row sums are folded over the warp, added up over the warps in shared memory and
// stored: a thread block owns its rows, so y needs neither zeroing nor atomics.
struct FusedLayout {
    int x_bytes, slot_off, part_off, y_off, cnt_off, active_off, xm_off, total;
    __host__ __device__ FusedLayout(int nb, int threads) {
        x_bytes = nb * 64;
        slot_off = x_bytes;
        part_off = slot_off + threads * wc_slot_bytes(wc_ilp(threads / 32));
        y_off = part_off + (threads / 32) * 64;
        cnt_off = y_off + 64;
        active_off = cnt_off + 16;
        xm_off = active_off + nb * 4;
        total = (xm_off + nb * 2 + 15) & ~15;
    }
};
constexpr int FUSED_MAX_SMEM = 200 * 1024;   // of the 227 KB a thread block may have

template <int DT, int NW>
__global__ void __launch_bounds__(NW * 32, 768 / (NW * 32))
k_decode_fused(Device d, const void *__restrict__ x, float *__restrict__ y, float th3, int force_path) {
    extern __shared__ __align__(16) uint8_t s_dyn[];
    constexpr int T = NW * 32;
    const FusedLayout lay(d.nb, T);
    float *s_x = reinterpret_cast<float *>(s_dyn);
    float *s_part = reinterpret_cast<float *>(s_dyn + lay.part_off);
    float *s_y = reinterpret_cast<float *>(s_dyn + lay.y_off);
    int *s_cnt = reinterpret_cast<int *>(s_dyn + lay.cnt_off);       // [0] nonzero vector blocks
    int *s_active = reinterpret_cast<int *>(s_dyn + lay.active_off);  // their indices, ascending (push)
    uint16_t *s_xm = reinterpret_cast<uint16_t *>(s_dyn + lay.xm_off);
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    uint4 *slot = reinterpret_cast<uint4 *>(s_dyn + lay.slot_off + tid * wc_slot_bytes(wc_ilp(NW)));
    pdl_wait();
    if (tid == 0) { s_cnt[0] = 0; s_cnt[1] = 0; }
    if (tid < 16) s_y[tid] = 0.f;
    __syncthreads();

    stage_x_blocks<DT>(d, x, s_x, s_xm, s_cnt, tid, T);
    __syncthreads();
    const int n_nzblk = s_cnt[0];
    int path = force_path;
    if (path != DBSPMSPV_PATH_PUSH && path != DBSPMSPV_PATH_PULL)
        path = (float)n_nzblk / (float)d.nb < th3 ? DBSPMSPV_PATH_PUSH : DBSPMSPV_PATH_PULL;
    if (blockIdx.x == 0 && tid == 0) {
        Counters *c = d.ws.ctr;
        c->last_n_nzblk = n_nzblk; c->last_n_tasks = 0; c->last_path = path; c->last_y_nnz = (int32_t)d.m;
        // (a store to host memory: only when it changes what the host goes by)
        if (d.x_nnz_seen && ((float)s_cnt[1] < STREAM_MIN_X_DENSITY * (float)d.n) != (d.x_sparse_believed != 0)) *d.x_nnz_seen = s_cnt[1];
    }
    if (path == DBSPMSPV_PATH_PUSH) {
        if (warp == 0) {
            int count = 0;
            for (int base = 0; base < d.nb; base += 32) {
                const bool on = base + lane < d.nb && s_xm[base + lane] != 0;
                const uint32_t m = __ballot_sync(FULL, on);
                if (on) s_active[count + __popc(m & below(lane))] = base + lane;
                count += __popc(m);
            }
        }
        __syncthreads();
    }

    const int rb = blockIdx.x;
    const int begin = d.csr.ptr[rb], end = d.csr.ptr[rb + 1];
    float acc[16];
#pragma unroll
    for (int r = 0; r < 16; ++r) acc[r] = 0.f;
    auto emit = [&](int, int erow, float esum) { atomicAdd(&s_y[erow], esum); };
    // one step: the lane's entry (idx, w, aux), if `have`
    auto step = [&](uint32_t idx, uint32_t w, uint32_t aux, bool have) {
        const uint32_t xm = have ? s_xm[idx & IDX_MASK] : 0u;
        const int type = idx >> TYPE_SHIFT;
        const bool mk = have && xm && type > DBSPMSPV_BLK_COO;
        const bool rowm = mk && is_row_major(type);
        const float *xb = s_x + (size_t)(idx & IDX_MASK) * 16;
        warp_columns<DT, wc_ilp(NW)>(d.payload, s_x, idx, w, mk && !rowm ? xm : 0u, lane, acc, slot);
        __syncwarp();
        const uint32_t rows = __ballot_sync(FULL, rowm);
        if (rows) half_stream<DT, true>(d.payload, s_x, idx, w, xm, rb, rows, lane, emit);
        if (have && xm && type <= DBSPMSPV_BLK_COO) {       // the odd hypersparse block: its own lane
            if (type == DBSPMSPV_BLK_INLINE) {
                if ((xm >> (aux & 15)) & 1u) atomicAdd(&s_y[aux >> 4], Val<DT>::inline_value(w) * xb[aux & 15]);
            } else {
                const int nnz = (int)aux + 1;
                const uint8_t *blk = d.payload + (size_t)w * 4, *vals = blk + ((nnz + 3) & ~3);
                for (int k = 0; k < nnz; ++k) {
                    const int c = blk[k] & 15, r = blk[k] >> 4;
                    if ((xm >> c) & 1u) atomicAdd(&s_y[r], Val<DT>::load(vals, k) * xb[c]);
                }
            }
        }
    };
    auto fetch = [&](int p, bool have, uint32_t &idx, uint32_t &w, uint32_t &aux) {
        idx = 0; w = 0; aux = 0;
        if (have && DBS_CHK_INDEX(d, p, d.n_entries)) { idx = d.csr.idx[p]; w = d.csr.w[p]; aux = d.csr.aux[p]; DBS_CHK_ENTRY(d, true, idx, w, aux); }
    };
    if (path == DBSPMSPV_PATH_PULL) {
        // the next step's entries are fetched before this step's blocks are worked on
        uint32_t idx, w, aux, n_idx, n_w, n_aux;
        int base = begin + warp * 32;
        fetch(base + lane, base + lane < end, idx, w, aux);
        for (; base < end; base += T) {
            const int nb_ = base + T;
            fetch(nb_ + lane, nb_ + lane < end, n_idx, n_w, n_aux);
            step(idx, w, aux, base + lane < end);
            idx = n_idx; w = n_w; aux = n_aux;
        }
    } else {
        // the row block's entries with a payload are sorted by column block: [begin, pend)
        const int pend = d.csr_inl[rb];
        for (int i0 = warp * 32; i0 < n_nzblk; i0 += T) {
            int lo = 0, hi = 0;
            if (i0 + lane < n_nzblk) {
                const uint32_t cb = (uint32_t)s_active[i0 + lane];
                int a = begin, b = pend;          // first entry with column block >= cb
                while (a < b) { const int mid = a + ((b - a) >> 1); if ((d.csr.idx[mid] & IDX_MASK) < cb) a = mid + 1; else b = mid; }
                lo = a; b = pend;                 // first entry with column block > cb
                while (a < b) { const int mid = a + ((b - a) >> 1); if ((d.csr.idx[mid] & IDX_MASK) <= cb) a = mid + 1; else b = mid; }
                hi = a;
            }
            for (int t = 0; __any_sync(FULL, lo + t < hi); ++t) {
                uint32_t idx, w, aux;
                fetch(lo + t, lo + t < hi, idx, w, aux);
                step(idx, w, aux, lo + t < hi);
            }
        }
        // its INLINE elements (row by row, rare in these handles): each tested against its mask
        for (int base = pend + warp * 32; base < end; base += T) {
            uint32_t idx, w, aux;
            fetch(base + lane, base + lane < end, idx, w, aux);
            step(idx, w, aux, base + lane < end);
        }
    }
    {
        const float total = fold_rows(acc, lane);
        if (!(lane & 1)) s_part[warp * 16 + folded_row(lane)] = total;
    }
    __syncthreads();
    if (tid < 16) {
        float sum = s_y[tid];
#pragma unroll
        for (int k = 0; k < NW; ++k) sum += s_part[k * 16 + tid];
        const int64_t row = (int64_t)rb * 16 + tid;
        if (row < d.m) y[row] = sum;
    }
}

// ------------------------------------------------------------------------------------------
// Streaming decode (Section 4.3: one layer, one token) for payload-dominated handles: the whole
// call in one persistent kernel that reads the payload as a stream.
//   * The payload of a row block is one contiguous byte range; at create it is cut into chunks
//     of whole blocks (a few KB, at most 32 blocks).  The chunk list is split evenly over all
//     warps of the grid, every warp taking a contiguous piece.
//   * Every warp runs its own ring of STREAM_DEPTH stages in shared memory: one lane moves a
//     chunk's payload bytes with one bulk copy while the warp works on an earlier chunk (the
//     chunk's view entries, 9 bytes per block, are loaded into registers a round ahead).  The microkernels' chains of
//     dependent loads (entry -> header -> column start -> values) then cost shared-memory
//     latency, no load goes through the L1 tag stage one sector at a time, and HBM sees
//     sequential reads whatever the activation sparsity.
//   * x is read once per thread block (a few KB) into masks and fp32 blocks, as in the
//     single-kernel form above; the 16 row sums of a warp stay in registers while its chunks
//     belong to one row block and go to y with one atomic per row when the row block changes
//     (y is zeroed by a memset in front of the kernel).
// A call whose x fills few vector blocks (push) walks the row blocks' entries by bisection
// straight from global memory, as the single-kernel form does.
#ifndef DBS_STREAM_WARPS
#define DBS_STREAM_WARPS 16
#endif
#ifndef DBS_STREAM_BUDGET
#define DBS_STREAM_BUDGET (220 * 1024)
#endif
constexpr int STREAM_WARPS = DBS_STREAM_WARPS;
constexpr int STREAM_CTA = STREAM_WARPS * 32;
#ifndef DBS_STREAM_DEPTH
#define DBS_STREAM_DEPTH 2
#endif
constexpr int STREAM_DEPTH = DBS_STREAM_DEPTH;
constexpr int STREAM_MAX_SMEM = 227 * 1024;   // all a thread block may have
constexpr int DCB_MAX_SMEM = STREAM_MAX_SMEM - 256;   // (static shared memory of k_decode_cols_batch)
__host__ __device__ constexpr int stream_stride(int stage_bytes) { return (stage_bytes + 127) & ~127; }
struct StreamLayout {
    int xm_off, cnt_off, active_off, bar_off, ring_off, total;
    __host__ __device__ StreamLayout(int nb, int stage_bytes) {
        xm_off = nb * 64;
        cnt_off = (xm_off + nb * 2 + 15) & ~15;
        active_off = cnt_off + 16;
        bar_off = (active_off + nb * 4 + 15) & ~15;
        ring_off = (bar_off + STREAM_WARPS * STREAM_DEPTH * 8 + 127) & ~127;
        total = ring_off + STREAM_WARPS * STREAM_DEPTH * stream_stride(stage_bytes);
    }
};

template <int DT>
__global__ void __launch_bounds__(STREAM_CTA, STREAM_WARPS <= 8 ? 2 : 1)
k_decode_stream(Device d, const void *__restrict__ x, float *__restrict__ y, float th3, int force_path) {
    extern __shared__ __align__(128) uint8_t s_dyn[];
    constexpr int T = STREAM_CTA, NW = STREAM_WARPS;
    const StreamLayout lay(d.nb, d.stage_bytes);
    float *s_x = reinterpret_cast<float *>(s_dyn);
    uint16_t *s_xm = reinterpret_cast<uint16_t *>(s_dyn + lay.xm_off);
    int *s_cnt = reinterpret_cast<int *>(s_dyn + lay.cnt_off);
    int *s_active = reinterpret_cast<int *>(s_dyn + lay.active_off);
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int stride = stream_stride(d.stage_bytes);
    uint64_t *s_bar = reinterpret_cast<uint64_t *>(s_dyn + lay.bar_off) + warp * STREAM_DEPTH;
    uint8_t *s_ring = s_dyn + lay.ring_off + (size_t)warp * STREAM_DEPTH * stride;
    if (tid == 0) { s_cnt[0] = 0; s_cnt[1] = 0; }

    // this warp's piece of the chunk list; lane i keeps the descriptor of its i-th chunk (32 at a time)
    const int gw = blockIdx.x * NW + warp, W = gridDim.x * NW;
    const int lo = (int)((int64_t)d.n_stage_chunks * gw / W), hi = (int)((int64_t)d.n_stage_chunks * (gw + 1) / W);
    const int n_mine = hi - lo;
    int4 my_desc = make_int4(0, 0, 0, 0);
    if (lane < n_mine) my_desc = d.stage_chunks[lo + lane];
    auto desc_of = [&](int k) {                               // (whole warp)
        return make_int4(__shfl_sync(FULL, my_desc.x, k & 31), __shfl_sync(FULL, my_desc.y, k & 31),
                         __shfl_sync(FULL, my_desc.z, k & 31), __shfl_sync(FULL, my_desc.w, k & 31));
    };
    // descriptor: x = first view entry, y = row block, z = payload offset in words, w = words | entries << 24
    auto issue = [&](const int4 &ch, int st) {               // lane 0 only
        uint8_t *base = s_ring + (size_t)st * stride;
        uint32_t pb = ((uint32_t)ch.w & 0xFFFFFFu) * 4u;
        if (!DBS_CHK_INDEX(d, pb, d.stage_bytes + 1) || !DBS_CHK_INDEX(d, (uint64_t)(uint32_t)ch.z + (pb >> 2), (uint64_t)d.payload_words + 1)) pb = 0u;
        fence_proxy_async_smem();
        mbar_arrive_expect_tx(&s_bar[st], pb);
        if (pb) bulk_copy_g2s(base, d.payload + (size_t)(uint32_t)ch.z * 4, pb, &s_bar[st]);
    };
    // the chunk's view entries, one per lane, by plain loads a round ahead of their use (they
    // are 9 bytes per block; bulk copies of 48-256 bytes cost the copy engine as much as the payload's)
    auto entries_of = [&](const int4 &ch, uint32_t &idx, uint32_t &w, uint32_t &aux) {
        idx = 0; w = 0; aux = 0;
        if (lane < (int)((uint32_t)ch.w >> 24) && DBS_CHK_RANGE(d, ch.x, (uint32_t)ch.w >> 24)) {
            const int p_ = ch.x + lane; idx = d.csr.idx[p_]; w = d.csr.w[p_]; aux = d.csr.aux[p_];
            DBS_CHK_ENTRY(d, true, idx, w, aux);
            // (the staged copy holds exactly the chunk's words: the block must start inside them)
            if ((idx >> TYPE_SHIFT) != DBSPMSPV_BLK_INLINE && !DBS_CHK_INDEX(d, (int64_t)w - (uint32_t)ch.z, (uint32_t)ch.w & 0xFFFFFFu)) { idx = 0u; w = 0u; aux = 0u; }
        }
    };
    int issued = 0;                                           // chunks of mine whose copies were started
    if (lane == 0) {
#pragma unroll
        for (int k = 0; k < STREAM_DEPTH; ++k) mbar_init(&s_bar[k], 1);
        fence_barrier_init();
    }
    __syncwarp();
    // the first copies start before x is even looked at
    for (; issued < STREAM_DEPTH - 1 && issued < n_mine; ++issued) {
        const int4 ch = desc_of(issued);
        if (lane == 0) issue(ch, issued);
    }
    __syncthreads();
    stage_x_blocks<DT>(d, x, s_x, s_xm, s_cnt, tid, T);
    __syncthreads();
    const int n_nzblk = s_cnt[0];
    int path = force_path;
    if (path != DBSPMSPV_PATH_PUSH && path != DBSPMSPV_PATH_PULL)
        path = (float)n_nzblk / (float)d.nb < th3 ? DBSPMSPV_PATH_PUSH : DBSPMSPV_PATH_PULL;
    if (blockIdx.x == 0 && tid == 0) {
        Counters *c = d.ws.ctr;
        c->last_n_nzblk = n_nzblk; c->last_n_tasks = 0; c->last_path = path; c->last_y_nnz = (int32_t)d.m;
        // (a store to host memory: only when it changes what the host goes by)
        if (d.x_nnz_seen && ((float)s_cnt[1] < STREAM_MIN_X_DENSITY * (float)d.n) != (d.x_sparse_believed != 0)) *d.x_nnz_seen = s_cnt[1];
    }

    // y is zeroed by the kernel in front, which this one may overlap up to here
    pdl_wait();

    float acc[16];
#pragma unroll
    for (int r = 0; r < 16; ++r) acc[r] = 0.f;
    int cur_rb = -1;
    // the warp's 16 row sums -> y (rows past m hold nothing: their sums are exact zeros)
    auto flush = [&]() {
        if (cur_rb >= 0) {
            const float total = fold_rows(acc, lane);
            if (!(lane & 1) && total != 0.f) atomicAdd(y + (size_t)cur_rb * 16 + folded_row(lane), total);
#pragma unroll
            for (int r = 0; r < 16; ++r) acc[r] = 0.f;
        }
    };
    auto emit = [&](int erb, int erow, float esum) { atomicAdd(y + (size_t)erb * 16 + erow, esum); };
    // one step: the lane's entry (idx, w, aux) of row block cur_rb, if `have`; the payload pointer
    // is the staged copy (shifted so that the entry's offset applies) or, on the rare paths that
    // read global memory, the payload itself -- the values are indexed where they are either way
    auto step = [&](const uint8_t *payload, uint32_t idx, uint32_t w, uint32_t aux, bool have) {
        const uint32_t xm = have ? s_xm[idx & IDX_MASK] : 0u;
        const int type = idx >> TYPE_SHIFT;
        const bool mk = have && xm && type > DBSPMSPV_BLK_COO;
        const bool rowm = mk && is_row_major(type);
        const float *xb = s_x + (size_t)(idx & IDX_MASK) * 16;
        warp_columns<DT, 2, true>(payload, s_x, idx, w, mk && !rowm ? xm : 0u, lane, acc, static_cast<uint4 *>(nullptr));
        __syncwarp();
        const uint32_t rows = __ballot_sync(FULL, rowm);
        if (rows) half_stream<DT, true>(payload, s_x, idx, w, xm, cur_rb, rows, lane, emit);
        if (have && xm && type <= DBSPMSPV_BLK_COO) {       // the odd hypersparse block: its own lane
            float *row0 = y + (size_t)cur_rb * 16;
            if (type == DBSPMSPV_BLK_INLINE) {
                if ((xm >> (aux & 15)) & 1u) atomicAdd(row0 + (aux >> 4), Val<DT>::inline_value(w) * xb[aux & 15]);
            } else {
                const int nnz = (int)aux + 1;
                const uint8_t *blk = payload + (size_t)w * 4, *vals = blk + ((nnz + 3) & ~3);
                for (int k = 0; k < nnz; ++k) {
                    const int c = blk[k] & 15, r = blk[k] >> 4;
                    if ((xm >> c) & 1u) atomicAdd(row0 + r, Val<DT>::load(vals, k) * xb[c]);
                }
            }
        }
    };
    auto fetch = [&](int p, bool have, uint32_t &idx, uint32_t &w, uint32_t &aux) {
        idx = 0; w = 0; aux = 0;
        if (have && DBS_CHK_INDEX(d, p, d.n_entries)) { idx = d.csr.idx[p]; w = d.csr.w[p]; aux = d.csr.aux[p]; DBS_CHK_ENTRY(d, true, idx, w, aux); }
    };

    if (path == DBSPMSPV_PATH_PULL) {
        bool timed_out = false;
        uint32_t idx = 0, w = 0, aux = 0, n_idx, n_w, n_aux;
        if (n_mine > 0) entries_of(desc_of(0), idx, w, aux);
        for (int k = 0; k < n_mine; ++k) {
            // keep STREAM_DEPTH - 1 chunks in flight beside this one: chunk i goes into the stage
            // that chunk i - STREAM_DEPTH was read from, in a round before this one
            for (const int lim = min(n_mine, min(k + STREAM_DEPTH, (k & ~31) + 32)); issued < lim; ++issued) {
                const int4 nch = desc_of(issued);
                if (lane == 0) issue(nch, issued % STREAM_DEPTH);
            }
            const int st = k % STREAM_DEPTH;
            const int4 ch = desc_of(k);
            n_idx = 0; n_w = 0; n_aux = 0;
            if (k + 1 < n_mine && ((k + 1) & 31)) entries_of(desc_of(k + 1), n_idx, n_w, n_aux);
            if (!mbar_wait_bounded(&s_bar[st], (uint32_t)(k / STREAM_DEPTH) & 1u)) { timed_out = true; break; }
            if (ch.y != cur_rb) { flush(); cur_rb = DBS_CHK_INDEX(d, ch.y, d.mb) ? ch.y : 0; }
            const uint8_t *base = s_ring + (size_t)st * stride;
            step(base - (size_t)(uint32_t)ch.z * 4, idx, w, aux, lane < (int)((uint32_t)ch.w >> 24));
            __syncwarp();
            idx = n_idx; w = n_w; aux = n_aux;
            if (k + 1 < n_mine && !((k + 1) & 31)) {           // first chunk of the next descriptor batch: fetched late
                my_desc = make_int4(0, 0, 0, 0);
                if (k + 1 + lane < n_mine) my_desc = d.stage_chunks[lo + k + 1 + lane];
                entries_of(desc_of(k + 1), idx, w, aux);
            }
        }
        flush();
        if (timed_out) { d.ws.ctr->status = DBSPMSPV_ERR_TIMEOUT; return; }
        // the INLINE elements of the row blocks (row by row, rare in these handles)
        for (int rb = gw; rb < d.mb && d.has_inline; rb += W) {
            const int b0 = d.csr_inl[rb], b1 = d.csr.ptr[rb + 1];
            cur_rb = rb;
            for (int base = b0; base < b1; base += 32) {
                uint32_t idx, w, aux;
                fetch(base + lane, base + lane < b1, idx, w, aux);
                step(d.payload, idx, w, aux, base + lane < b1);
            }
            if (b1 > b0) flush();
        }
    } else {
        // copies of the first chunks are in flight: they must have landed before the block ends
        for (int k = 0; k < issued; ++k) mbar_wait_bounded(&s_bar[k], 0u);
        if (warp == 0) {
            int count = 0;
            for (int base = 0; base < d.nb; base += 32) {
                const bool on = base + lane < d.nb && s_xm[base + lane] != 0;
                const uint32_t m = __ballot_sync(FULL, on);
                if (on) s_active[count + __popc(m & below(lane))] = base + lane;
                count += __popc(m);
            }
        }
        __syncthreads();
        for (int rb = blockIdx.x; rb < d.mb; rb += gridDim.x) {
            const int begin = d.csr.ptr[rb], pend = d.csr_inl[rb], end = d.csr.ptr[rb + 1];
            cur_rb = rb;
            // the row block's entries with a payload are sorted by column block: [begin, pend)
            for (int i0 = warp * 32; i0 < n_nzblk; i0 += T) {
                int lo_ = 0, hi_ = 0;
                if (i0 + lane < n_nzblk) {
                    const uint32_t cb = (uint32_t)s_active[i0 + lane];
                    int a = begin, b = pend;          // first entry with column block >= cb
                    while (a < b) { const int mid = a + ((b - a) >> 1); if ((d.csr.idx[mid] & IDX_MASK) < cb) a = mid + 1; else b = mid; }
                    lo_ = a; b = pend;                // first entry with column block > cb
                    while (a < b) { const int mid = a + ((b - a) >> 1); if ((d.csr.idx[mid] & IDX_MASK) <= cb) a = mid + 1; else b = mid; }
                    hi_ = a;
                }
                for (int t = 0; __any_sync(FULL, lo_ + t < hi_); ++t) {
                    uint32_t idx, w, aux;
                    fetch(lo_ + t, lo_ + t < hi_, idx, w, aux);
                    step(d.payload, idx, w, aux, lo_ + t < hi_);
                }
            }
            for (int base = pend + warp * 32; base < end; base += T) {
                uint32_t idx, w, aux;
                fetch(base + lane, base + lane < end, idx, w, aux);
                step(d.payload, idx, w, aux, base + lane < end);
            }
            flush();
        }
    }
}

}  // namespace dbs
#include "decode_batch.cuh"
#include "small_call.cuh"
#include "decode_columns.cuh"
#include "sssp.cuh"
namespace dbs {

// ------------------------------------------------------------------------------------------
// The end of a call: the rows that were hit, in order, become y; the accumulator and the vector-block
// state of this call's x are cleared, and the counters are rolled over.
// ------------------------------------------------------------------------------------------

// Fold of the private accumulators of eight rows of a hub row block into the accumulator proper, by the
// thread that owns the rows: the copies are fetched four at a time (all at once took the kernel to 128
// registers, two thread blocks per SM) and added up in a fixed order; (min, +)
// words are folded by their maximum.  Touched copies are put back to HUB_CLEAR.
__device__ __forceinline__ void fold_hub_rows(const Device &d, int slot, int half, int minplus, uint32_t (&acc)[8]) {
#pragma unroll 1
    for (int c0 = 0; c0 < d.hub_on; c0 += 4) {
        uint4 *p = reinterpret_cast<uint4 *>(d.hub_acc + ((size_t)c0 * d.n_hub_blocks + slot) * 16 + 8 * half);
        const size_t next = (size_t)d.n_hub_blocks * 4;          // 16-byte words from copy to copy
        uint4 v[4][2];
#pragma unroll
        for (int k = 0; k < 4; ++k) { v[k][0] = __ldcg(p + k * next); v[k][1] = __ldcg(p + k * next + 1); }
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const uint32_t w[8] = {v[k][0].x, v[k][0].y, v[k][0].z, v[k][0].w, v[k][1].x, v[k][1].y, v[k][1].z, v[k][1].w};
            uint32_t touched = 0u;
#pragma unroll
            for (int r = 0; r < 8; ++r) {
                touched |= w[r] ^ HUB_CLEAR;
                // (an untouched -0.0f adds nothing)
                if (minplus) acc[r] = (uint32_t)max((int)acc[r], (int)w[r]);
                else acc[r] = __float_as_uint(__uint_as_float(acc[r]) + __uint_as_float(w[r]));
            }
            if (touched) {
                p[k * next] = make_uint4(HUB_CLEAR, HUB_CLEAR, HUB_CLEAR, HUB_CLEAR);
                p[k * next + 1] = make_uint4(HUB_CLEAR, HUB_CLEAR, HUB_CLEAR, HUB_CLEAR);
            }
        }
    }
}

// What the last kernel of a call clears of the vector-block state of its x.
enum { CLEAR_MASKS = 1, CLEAR_DENSE = 2, CLEAR_SWEEP = 4 };   // SWEEP: whole arrays instead of entry by entry

constexpr int TILE_WAIT_LIMIT = 1 << 20;
constexpr int FINISH_PARITY = 1 << 30;
constexpr int FINISH_GROUP = 32;          // tiles per group
__device__ __forceinline__ unsigned long long load_relaxed64(const unsigned long long *p) {
    unsigned long long v;
    asm volatile("ld.relaxed.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
    return v;
}
__device__ __forceinline__ int load_relaxed32(const int32_t *p) {
    int v;
    asm volatile("ld.relaxed.gpu.global.s32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}
// Result entries in all tiles before `tile`, by one warp (see k_finish): the sums of the complete groups before its
// own, the status words of the tiles before it in its group.  -1 when a wait ran out.
__device__ __forceinline__ int entries_before(const Device &d, int tile, int parity, int lane) {
    const int g = tile / FINISH_GROUP, r = tile % FINISH_GROUP;
    const unsigned long long *groups = d.ws.tile_group + parity * d.ws.n_tile_groups;
    int sum = 0;
    bool ok = true;
    if (lane < r) {
        int v = 0, i = 0;
        do v = load_relaxed32(d.ws.tile_status + g * FINISH_GROUP + lane); while ((v & 1) != parity && ++i < TILE_WAIT_LIMIT);
        ok = i < TILE_WAIT_LIMIT;
        sum = v >> 1;
    }
    for (int k = lane; k < g; k += 32) {
        unsigned long long v = 0;
        int i = 0;
        do v = load_relaxed64(groups + k); while ((int)(v >> 32) != FINISH_GROUP && ++i < TILE_WAIT_LIMIT);
        ok = ok && i < TILE_WAIT_LIMIT;
        sum += (int)(uint32_t)v;
    }
    sum = __reduce_add_sync(FULL, sum);
    return __all_sync(FULL, ok) ? sum : -1;
}

// The counters of the call, by the thread that knows the length of y.
__device__ __forceinline__ void finish_counters(const Device &d, int total, int64_t y_capacity, int32_t *y_nnz) {
    Counters *ctr = d.ws.ctr;
    *y_nnz = total;
    if (total > y_capacity) ctr->status = DBSPMSPV_ERR_CAPACITY;
    ctr->last_y_nnz = total;
    ctr->last_n_nzblk = ctr->n_nzblk;
    ctr->last_n_tasks = ctr->n_tasks;
    ctr->last_path = ctr->path;
    ctr->n_nzblk = 0;
    ctr->n_tasks = 0;
    ctr->n_hubs = 0;
    ctr->n_long = 0;
}
// Vector-block state of this call's x: clear the masks and put the "not listed" marker back -- entry by entry, or,
// for an x that lists a good part of all columns, by streaming over the whole arrays (full-line stores instead of scattered
// 4-byte ones).  `at`: the thread's number in the grid, `j0`: x_idx[at], fetched ahead (-1: none).
__device__ __forceinline__ void finish_clear_x(const Device &d, const int32_t *__restrict__ x_idx, int32_t nnz_x, int clear, int at, int stride, int j0) {
    if (clear & CLEAR_SWEEP) {
        const int n_words = (d.nb + 1) / 2;
        if (clear & CLEAR_DENSE) {
            uint4 *xd4 = reinterpret_cast<uint4 *>(d.ws.x_dense);
            for (int k = at; k < n_words * 8; k += stride) xd4[k] = make_uint4(X_ABSENT, X_ABSENT, X_ABSENT, X_ABSENT);
        }
        for (int k = at; k < n_words; k += stride) d.ws.x_mask32[k] = 0u;
        return;
    }
    auto drop = [&](int j) {
        if (j < 0 || j >= d.n) return;
        d.ws.x_mask32[j >> 5] = 0u;
        if (clear & CLEAR_DENSE) d.ws.x_dense[j] = __uint_as_float(X_ABSENT);
    };
    drop(j0);
    for (int k = at + stride; k < nnz_x; k += stride) drop(x_idx[k]);
}

// The end of a call in one kernel: which rows were hit (see ACC_CLEAR), their order, y, and everything
// put back.  A thread block takes a tile of 2048 rows, a thread eight of them in two 16-byte loads that
// stay in registers; the tile publishes its count -- in a status word and, added up, in the word of its group of
// 32 tiles -- and one warp adds up the words of the groups and tiles before it (no chain from tile to
// tile), so y comes out sorted.  (With every thread polling a word of every earlier tile the polls
// queued up on the lines that the counts had to get into: 16 us.)
// A tile only waits for tiles with a lower ticket, and a ticket is taken when the thread block starts:
// the blocks it waits for are running.  The status of a tile carries the parity of the call
// (every call rewrites every tile), so nothing has to be reset.
// It replaces a counting pass and a placing pass: as two kernels they were two waits for the
// predecessor's last store and the accumulator was fetched twice (9.3 us exposed behind the traversal on a
// million rows; 5 here).
// FOLD: the call's push used private accumulators (more registers: a kernel of its own, so that the other keeps eight
// thread blocks per SM -- on four million rows the tiles come in waves).
template <bool FOLD>
__global__ void __launch_bounds__(CMP_TPB, FOLD ? 5 : 8) k_finish(Device d, int32_t *__restrict__ y_idx, float *__restrict__ y_val,
                                                    int64_t y_capacity, int32_t *__restrict__ y_nnz, int boolean,
                                                    const int32_t *__restrict__ x_idx, int32_t nnz_x, int clear, int fold,
                                                    const uint32_t *__restrict__ row_mask, int complement) {
    __shared__ int s_cnt[CMP_TPB / 32], s_ticket, s_parity, s_base;
    __shared__ int32_t s_oidx[CMP_TPB * 8];
    __shared__ float s_oval[CMP_TPB * 8];
    Counters *ctr = d.ws.ctr;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    // Ticket and parity of the call come from one word.  They are taken before the wait for the predecessor: the kernels in front of this
    // one in the call were let go only after the call before had ended.  (An empty x has no such kernel.)
    if (nnz_x == 0) pdl_wait();
    if (threadIdx.x == 0) { const int w = atomicAdd(&ctr->finish_ticket, 1); s_ticket = w & (FINISH_PARITY - 1); s_parity = w & FINISH_PARITY ? 1 : 0; }
    __syncthreads();
    const int tile = s_ticket, parity = s_parity, n_tiles = d.ws.n_tiles;
    const int stride = gridDim.x * CMP_TPB;
    const int bi = tile * CMP_TPB + threadIdx.x;      // byte of the hit mask: rows 8 bi .. 8 bi + 7
    const int j0 = (!(clear & CLEAR_SWEEP) && bi < nnz_x) ? x_idx[bi] : -1;      // (x is the caller's: nothing of this call writes it)
    pdl_wait();
    if (tile < n_tiles) {
        const int n_bytes = (d.mb + 1) / 2 * 4;
        uint8_t *mask8 = reinterpret_cast<uint8_t *>(d.ws.y_mask32);
        uint32_t hits = 0, keep = 0xFFu;                // rows to clear; rows that may go to y
        uint32_t v[8];
        if (bi < n_bytes) {
            uint4 *acc4 = reinterpret_cast<uint4 *>(d.ws.y_acc + (size_t)bi * 8);
            const uint4 a = __ldcg(acc4), b = __ldcg(acc4 + 1);
            const uint32_t flags = mask8[bi];
            const int path = FOLD ? ctr->path : 0;      // (a pull leaves the private accumulators alone)
            if (row_mask) keep = reinterpret_cast<const uint8_t *>(row_mask)[bi] ^ (complement ? 0xFFu : 0u);
            v[0] = a.x; v[1] = a.y; v[2] = a.z; v[3] = a.w; v[4] = b.x; v[5] = b.y; v[6] = b.z; v[7] = b.w;
            hits = flags;
#pragma unroll
            for (int r = 0; r < 8; ++r) hits |= (v[r] != ACC_CLEAR ? 1u : 0u) << r;
            if (hits) {
                acc4[0] = make_uint4(ACC_CLEAR, ACC_CLEAR, ACC_CLEAR, ACC_CLEAR);
                acc4[1] = make_uint4(ACC_CLEAR, ACC_CLEAR, ACC_CLEAR, ACC_CLEAR);
            }
            if (flags) mask8[bi] = 0;
            if (FOLD) {
                const int slot = d.hub_slot[bi >> 1];
                if (slot != HUB_NONE && path != DBSPMSPV_PATH_PULL && DBS_CHK_INDEX(d, slot, d.n_hub_blocks)) {
                    fold_hub_rows(d, slot, bi & 1, fold == 2, v);
#pragma unroll
                    for (int r = 0; r < 8; ++r) hits |= (v[r] != ACC_CLEAR ? 1u : 0u) << r;
                }
            }
        }
        const uint32_t bits = hits & keep;
        const int c = __popc(bits);
        int incl = c;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int t = __shfl_up_sync(FULL, incl, o);
            if (lane >= o) incl += t;
        }
        if (lane == 31) s_cnt[warp] = incl;
        __syncthreads();
        int local = 0, tile_total = 0;
#pragma unroll
        for (int k = 0; k < CMP_TPB / 32; ++k) {
            if (k < warp) local += s_cnt[k];
            tile_total += s_cnt[k];
        }
        if (threadIdx.x == 0) {
            asm volatile("st.relaxed.gpu.global.s32 [%0], %1;" ::"l"(d.ws.tile_status + tile), "r"(tile_total * 2 + parity) : "memory");
            atomicAdd(d.ws.tile_group + parity * d.ws.n_tile_groups + tile / FINISH_GROUP, (1ull << 32) + (unsigned)tile_total);
        }
        // (the group words of the other parity served the call before: cleared for the next one)
        if (tile == 0)
            for (int k = threadIdx.x; k < d.ws.n_tile_groups; k += CMP_TPB) d.ws.tile_group[(parity ^ 1) * d.ws.n_tile_groups + k] = 0ull;
        // the tile's entries are gathered in shared memory (while the other tiles' counts arrive), then written out in whole lines
        if (bits) {
            int pos = local + incl - c;
#pragma unroll
            for (int bit = 0; bit < 8; ++bit) {
                if ((bits >> bit) & 1u) {
                    s_oidx[pos] = bi * 8 + bit;
                    // boolean 1: a Boolean result; 2: the accumulator holds (min, +) words; else a sum (a row of -0 products is 0)
                    s_oval[pos] = boolean == 1 ? 1.0f : boolean == 2 ? minplus_of_word(v[bit]) : __uint_as_float(v[bit]) + 0.0f;
                    ++pos;
                }
            }
        }
        if (warp == 0) {
            const int before = entries_before(d, tile, parity, lane);
            if (lane == 0) { s_base = before; if (before < 0) ctr->status = DBSPMSPV_ERR_TIMEOUT; }
        }
        __syncthreads();
        const int base = max(s_base, 0);
        for (int k = threadIdx.x; k < tile_total; k += CMP_TPB) {
            const int64_t pos = (int64_t)base + k;
            if (pos < y_capacity) {
                y_idx[pos] = s_oidx[k];
                if (y_val) y_val[pos] = s_oval[k];
            }
        }
        if (tile == n_tiles - 1 && threadIdx.x == 0) finish_counters(d, base + tile_total, y_capacity, y_nnz);
    }
    // the block with the last ticket: all tickets are taken
    if (tile == (int)gridDim.x - 1 && threadIdx.x == 0) ctr->finish_ticket = parity ? 0 : FINISH_PARITY;
    finish_clear_x(d, x_idx, nnz_x, clear, bi, stride, j0);
}

// The same over two tiles per thread block, for accumulators of more tiles than fit on the GPU at once behind a push of blocks: the second tile waits in shared memory, so
// that a thread block needs no more registers, the two are counted and lined up as one, and most of the second wave with its ticket, loads, count and wait is spared.
// What it gains is the tiles that hold nothing, so it is kept to handles whose elements sit in blocks, which x in runs reaches in stretches; one tile / two, us a call at x = 2 / 3 / 4.5 %:
// 27-point operators, x in runs, 140^3 cells 36.2 / 42.0 / 50.7 and 33.9 / 40.0 / 48.9, 150^3 35.1 / 42.7 / 53.8 and 31.5 / 39.7 / 50.7, 160^3 33.4 / 38.1 / 46.5 and 30.1 / 35.7 / 45.0; bands of 48
// elements, 4 M rows, 43.1 / 50.1 / 62.2 and 38.5 / 45.2 / 57.0; scattered x within 1 % of each other.  With results in every tile half as many thread blocks are the slower form
// (uniform rows of 8, 2.5 M of them 15.3 / 17.0 / 20.1 and 17.5 / 19.6 / 22.9, 3.2 M 18.5 / 21.2 / 26.2 and 19.6 / 22.4 / 27.1), also just past the first wave (136^3 scattered 49.4 / 66.8 / 90.9 and
// 50.6 / 69.0 / 92.7), and in nearly all rows the second tile's way through shared memory costs more than the wave (144^3, 30 %, 149 and 154).
__global__ void __launch_bounds__(CMP_TPB, 8) k_finish_pair(Device d, int32_t *__restrict__ y_idx, float *__restrict__ y_val,
                                                           int64_t y_capacity, int32_t *__restrict__ y_nnz, int boolean,
                                                           const int32_t *__restrict__ x_idx, int32_t nnz_x, int clear,
                                                           const uint32_t *__restrict__ row_mask, int complement) {
    __shared__ __align__(16) uint4 s_second[2][CMP_TPB];
    __shared__ int s_cnt[CMP_TPB / 32], s_ticket, s_parity, s_base;
    __shared__ int32_t s_oidx[CMP_TPB * 8];
    __shared__ float s_oval[CMP_TPB * 8];
    Counters *ctr = d.ws.ctr;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    if (nnz_x == 0) pdl_wait();
    if (tid == 0) { const int w = atomicAdd(&ctr->finish_ticket, 1); s_ticket = w & (FINISH_PARITY - 1); s_parity = w & FINISH_PARITY ? 1 : 0; }
    __syncthreads();
    const int unit = s_ticket, parity = s_parity, n_units = (d.ws.n_tiles + 1) / 2;
    const int stride = gridDim.x * CMP_TPB, at = unit * CMP_TPB + tid;
    const int j0 = (!(clear & CLEAR_SWEEP) && at < nnz_x) ? x_idx[at] : -1;
    pdl_wait();
    if (unit < n_units) {
        const int n_bytes = (d.mb + 1) / 2 * 4;
        uint8_t *mask8 = reinterpret_cast<uint8_t *>(d.ws.y_mask32);
        const int bi = unit * 2 * CMP_TPB + tid, bj = bi + CMP_TPB;         // bytes of the hit mask: rows 8 bi .. 8 bi + 7 and 8 bj .. 8 bj + 7
        const uint4 untouched = make_uint4(ACC_CLEAR, ACC_CLEAR, ACC_CLEAR, ACC_CLEAR);
        uint4 *acc_i = reinterpret_cast<uint4 *>(d.ws.y_acc + (size_t)bi * 8), *acc_j = reinterpret_cast<uint4 *>(d.ws.y_acc + (size_t)bj * 8);
        uint32_t v[8], bits_i = 0u, bits_j = 0u;
        uint32_t flags_j = 0u;
        if (bj < n_bytes) {                            // (every thread reads back what it copied itself)
#pragma unroll
            for (int h = 0; h < 2; ++h) asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(smem_addr(&s_second[h][tid])), "l"(acc_j + h) : "memory");
            flags_j = mask8[bj];
        }
        if (bi < n_bytes) {
            const uint4 a = __ldcg(acc_i), b = __ldcg(acc_i + 1);
            const uint32_t flags = mask8[bi];
            v[0] = a.x; v[1] = a.y; v[2] = a.z; v[3] = a.w; v[4] = b.x; v[5] = b.y; v[6] = b.z; v[7] = b.w;
            uint32_t hits = flags;
#pragma unroll
            for (int r = 0; r < 8; ++r) hits |= (v[r] != ACC_CLEAR ? 1u : 0u) << r;
            if (hits) { acc_i[0] = untouched; acc_i[1] = untouched; }
            if (flags) mask8[bi] = 0;
            bits_i = row_mask ? hits & (reinterpret_cast<const uint8_t *>(row_mask)[bi] ^ (complement ? 0xFFu : 0u)) : hits;
        }
        auto second = [&](uint32_t (&w)[8]) {
            const uint4 a = s_second[0][tid], b = s_second[1][tid];
            w[0] = a.x; w[1] = a.y; w[2] = a.z; w[3] = a.w; w[4] = b.x; w[5] = b.y; w[6] = b.z; w[7] = b.w;
        };
        asm volatile("cp.async.wait_all;" ::: "memory");
        if (bj < n_bytes) {
            uint32_t w[8], hits = flags_j;
            second(w);
#pragma unroll
            for (int r = 0; r < 8; ++r) hits |= (w[r] != ACC_CLEAR ? 1u : 0u) << r;
            if (hits) { acc_j[0] = untouched; acc_j[1] = untouched; }
            if (flags_j) mask8[bj] = 0;
            bits_j = row_mask ? hits & (reinterpret_cast<const uint8_t *>(row_mask)[bj] ^ (complement ? 0xFFu : 0u)) : hits;
        }
        const int c = __popc(bits_i) | __popc(bits_j) << 16;               // (2048 at most: both counts in one scan)
        int incl = c;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int t = __shfl_up_sync(FULL, incl, o);
            if (lane >= o) incl += t;
        }
        if (lane == 31) s_cnt[warp] = incl;
        __syncthreads();
        int before = incl - c, total = 0;
#pragma unroll
        for (int k = 0; k < CMP_TPB / 32; ++k) {
            if (k < warp) before += s_cnt[k];
            total += s_cnt[k];
        }
        const int total_i = total & 0xFFFF, total_j = total >> 16;
        // (every call rewrites every tile's word, read or not: the next call may take one tile per thread block)
        if (tid == 1 && unit + n_units < d.ws.n_tiles) d.ws.tile_status[unit + n_units] = parity;
        if (tid == 0) {
            asm volatile("st.relaxed.gpu.global.s32 [%0], %1;" ::"l"(d.ws.tile_status + unit), "r"((total_i + total_j) * 2 + parity) : "memory");
            atomicAdd(d.ws.tile_group + parity * d.ws.n_tile_groups + unit / FINISH_GROUP, (1ull << 32) + (unsigned)(total_i + total_j));
        }
        if (unit == 0)
            for (int k = tid; k < d.ws.n_tile_groups; k += CMP_TPB) d.ws.tile_group[(parity ^ 1) * d.ws.n_tile_groups + k] = 0ull;
        auto gather = [&](uint32_t bits, int first_row, const uint32_t (&w)[8], int pos) {
#pragma unroll
            for (int bit = 0; bit < 8; ++bit) {
                if ((bits >> bit) & 1u) {
                    s_oidx[pos] = first_row + bit;
                    s_oval[pos] = boolean == 1 ? 1.0f : boolean == 2 ? minplus_of_word(w[bit]) : __uint_as_float(w[bit]) + 0.0f;
                    ++pos;
                }
            }
        };
        auto write = [&](int64_t base, int n) {
            for (int k = tid; k < n; k += CMP_TPB) {
                const int64_t pos = base + k;
                if (pos < y_capacity) {
                    y_idx[pos] = s_oidx[k];
                    if (y_val) y_val[pos] = s_oval[k];
                }
            }
        };
        if (bits_i) gather(bits_i, bi * 8, v, before & 0xFFFF);
        if (warp == 0) {
            const int sum = entries_before(d, unit, parity, lane);
            if (lane == 0) { s_base = sum; if (sum < 0) ctr->status = DBSPMSPV_ERR_TIMEOUT; }
        }
        __syncthreads();
        const int base = max(s_base, 0);
        write(base, total_i);
        __syncthreads();
        if (bits_j) {
            uint32_t w[8];
            second(w);
            gather(bits_j, bj * 8, w, before >> 16);
        }
        __syncthreads();
        write((int64_t)base + total_i, total_j);
        if (unit == n_units - 1 && tid == 0) finish_counters(d, base + total_i + total_j, y_capacity, y_nnz);
    }
    if (unit == (int)gridDim.x - 1 && tid == 0) ctr->finish_ticket = parity ? 0 : FINISH_PARITY;
    finish_clear_x(d, x_idx, nnz_x, clear, at, stride, j0);
}

// The same over FINISH_WIDE tiles at most per thread block, for accumulators of more tiles than fit on the GPU at once (in waves, each tile
// with its ticket, loads, count and wait: 16 us on four million rows even for an empty result; 8 here).  First all tiles are
// counted, their loads side by side; then the rows that hold results are fetched again, from L2, and written.  (Four million
// rows, x = 1 %: 13.9 us, 16.6 in waves.  Lining up results per warp, or writing few of them straight to y, took 15.)
constexpr int FINISH_WIDE = 4;
template <bool FOLD>
__global__ void __launch_bounds__(CMP_TPB, FOLD ? 4 : 8) k_finish_wide(Device d, int per_block, int32_t *__restrict__ y_idx, float *__restrict__ y_val,
                                                    int64_t y_capacity, int32_t *__restrict__ y_nnz, int boolean,
                                                    const int32_t *__restrict__ x_idx, int32_t nnz_x, int clear, int fold,
                                                    const uint32_t *__restrict__ row_mask, int complement) {
    __shared__ int s_cnt[FINISH_WIDE][CMP_TPB / 32], s_ticket, s_parity, s_base;
    __shared__ int32_t s_oidx[CMP_TPB * 8];
    __shared__ float s_oval[CMP_TPB * 8];
    Counters *ctr = d.ws.ctr;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    if (nnz_x == 0) pdl_wait();
    if (threadIdx.x == 0) { const int w = atomicAdd(&ctr->finish_ticket, 1); s_ticket = w & (FINISH_PARITY - 1); s_parity = w & FINISH_PARITY ? 1 : 0; }
    __syncthreads();
    const int unit = s_ticket, parity = s_parity, n_units = (d.ws.n_tiles + per_block - 1) / per_block;
    const int stride = gridDim.x * CMP_TPB, at = unit * CMP_TPB + threadIdx.x;
    const int j0 = (!(clear & CLEAR_SWEEP) && at < nnz_x) ? x_idx[at] : -1;
    pdl_wait();
    if (unit < n_units) {
        const int n_bytes = (d.mb + 1) / 2 * 4;
        uint8_t *mask8 = reinterpret_cast<uint8_t *>(d.ws.y_mask32);
        const int first = unit * per_block * CMP_TPB + threadIdx.x;          // byte of the hit mask in the unit's first tile
        const int path = FOLD ? ctr->path : 0;
        uint32_t kept = 0u;                       // per tile: rows of this thread that go to y
        uint32_t before[2] = {0u, 0u};            // per tile, 16 bits: such rows in the lanes up to this one
        const uint4 untouched = make_uint4(ACC_CLEAR, ACC_CLEAR, ACC_CLEAR, ACC_CLEAR);
#pragma unroll
        for (int t0 = 0; t0 < FINISH_WIDE; t0 += 2) {
            uint4 a[2], b[2];
            uint32_t flags[2];
#pragma unroll
            for (int u = 0; u < 2; ++u) {
                const int bi = first + (t0 + u) * CMP_TPB;
                a[u] = b[u] = untouched;
                flags[u] = 0u;
                if (t0 + u < per_block && bi < n_bytes) {
                    const uint4 *acc4 = reinterpret_cast<const uint4 *>(d.ws.y_acc + (size_t)bi * 8);
                    a[u] = __ldcg(acc4); b[u] = __ldcg(acc4 + 1);
                    flags[u] = mask8[bi];
                }
            }
#pragma unroll
            for (int u = 0; u < 2; ++u) {
                const int t = t0 + u, bi = first + t * CMP_TPB;
                const bool mine = t < per_block && bi < n_bytes;
                uint4 *acc4 = reinterpret_cast<uint4 *>(d.ws.y_acc + (size_t)bi * 8);
                uint32_t v[8] = {a[u].x, a[u].y, a[u].z, a[u].w, b[u].x, b[u].y, b[u].z, b[u].w};
                uint32_t hits = flags[u];
                bool folded = false;
                if (FOLD && mine) {
                    const int slot = d.hub_slot[bi >> 1];
                    if (slot != HUB_NONE && path != DBSPMSPV_PATH_PULL && DBS_CHK_INDEX(d, slot, d.n_hub_blocks)) {
                        fold_hub_rows(d, slot, bi & 1, fold == 2, v);
                        folded = true;
                    }
                }
                uint32_t differ = 0u;
#pragma unroll
                for (int r = 0; r < 8; ++r) differ |= v[r] ^ ACC_CLEAR;
                if (differ) {                                              // (most rows of a wide accumulator are untouched)
#pragma unroll
                    for (int r = 0; r < 8; ++r) hits |= (v[r] != ACC_CLEAR ? 1u : 0u) << r;
                }
                uint32_t bits = hits;
                if (hits && row_mask) bits &= reinterpret_cast<const uint8_t *>(row_mask)[bi] ^ (complement ? 0xFFu : 0u);
                if (flags[u]) mask8[bi] = 0;
                if (bits && folded) { acc4[0] = make_uint4(v[0], v[1], v[2], v[3]); acc4[1] = make_uint4(v[4], v[5], v[6], v[7]); }      // (fetched again below)
                else if (hits && !bits) { acc4[0] = untouched; acc4[1] = untouched; }
                kept |= bits << (8 * t);
                int incl = __popc(bits);
                if (__any_sync(FULL, bits != 0u)) {
#pragma unroll
                    for (int o = 1; o < 32; o <<= 1) {
                        const int q = __shfl_up_sync(FULL, incl, o);
                        if (lane >= o) incl += q;
                    }
                }
                before[t >> 1] |= (uint32_t)incl << (16 * (t & 1));
                if (lane == 31) s_cnt[t][warp] = incl;
            }
        }
        __syncthreads();
        int unit_total = 0;
        for (int t = 0; t < per_block; ++t)
            for (int k = 0; k < CMP_TPB / 32; ++k) unit_total += s_cnt[t][k];
        // (every call rewrites every tile's word, read or not: the next call may take one tile per thread block)
        if (threadIdx.x > 0 && threadIdx.x < per_block && unit + threadIdx.x * n_units < d.ws.n_tiles) d.ws.tile_status[unit + threadIdx.x * n_units] = parity;
        if (threadIdx.x == 0) {
            asm volatile("st.relaxed.gpu.global.s32 [%0], %1;" ::"l"(d.ws.tile_status + unit), "r"(unit_total * 2 + parity) : "memory");
            atomicAdd(d.ws.tile_group + parity * d.ws.n_tile_groups + unit / FINISH_GROUP, (1ull << 32) + (unsigned)unit_total);
        }
        if (unit == 0)
            for (int k = threadIdx.x; k < d.ws.n_tile_groups; k += CMP_TPB) d.ws.tile_group[(parity ^ 1) * d.ws.n_tile_groups + k] = 0ull;
        int base = 0;
        if (unit_total > 0 || unit == n_units - 1) {                      // (an empty unit has nothing to place)
            for (int t = 0; t < per_block; ++t) {
                int local = 0, tile_total = 0;
#pragma unroll
                for (int k = 0; k < CMP_TPB / 32; ++k) {
                    if (k < warp) local += s_cnt[t][k];
                    tile_total += s_cnt[t][k];
                }
                if (tile_total == 0 && t > 0) continue;                    // block-uniform
                const uint32_t bits = (kept >> (8 * t)) & 0xFFu;
                if (bits) {
                    const int bi = first + t * CMP_TPB;
                    uint4 *acc4 = reinterpret_cast<uint4 *>(d.ws.y_acc + (size_t)bi * 8);
                    const uint4 a = __ldcg(acc4), b = __ldcg(acc4 + 1);
                    acc4[0] = untouched; acc4[1] = untouched;
                    const uint32_t v[8] = {a.x, a.y, a.z, a.w, b.x, b.y, b.z, b.w};
                    int pos = local + (int)((before[t >> 1] >> (16 * (t & 1))) & 0xFFFFu) - __popc(bits);
#pragma unroll
                    for (int bit = 0; bit < 8; ++bit) {
                        if ((bits >> bit) & 1u) {
                            s_oidx[pos] = bi * 8 + bit;
                            s_oval[pos] = boolean == 1 ? 1.0f : boolean == 2 ? minplus_of_word(v[bit]) : __uint_as_float(v[bit]) + 0.0f;
                            ++pos;
                        }
                    }
                }
                if (t == 0 && warp == CMP_TPB / 32 - 1) {                  // (while the other tiles' counts arrive the first tile is gathered)
                    const int sum = entries_before(d, unit, parity, lane);
                    if (lane == 0) { s_base = sum; if (sum < 0) ctr->status = DBSPMSPV_ERR_TIMEOUT; }
                }
                __syncthreads();
                if (t == 0) base = max(s_base, 0);
                for (int k = threadIdx.x; k < tile_total; k += CMP_TPB) {
                    const int64_t pos = (int64_t)base + k;
                    if (pos < y_capacity) {
                        y_idx[pos] = s_oidx[k];
                        if (y_val) y_val[pos] = s_oval[k];
                    }
                }
                base += tile_total;
                __syncthreads();
            }
            if (unit == n_units - 1 && threadIdx.x == 0) finish_counters(d, base, y_capacity, y_nnz);
        }
    }
    if (unit == (int)gridDim.x - 1 && threadIdx.x == 0) ctr->finish_ticket = parity ? 0 : FINISH_PARITY;
    finish_clear_x(d, x_idx, nnz_x, clear, at, stride, j0);
}

__global__ void k_decode_cleanup(Device d) {
    pdl_wait();
    const int n_words = (d.nb + 1) / 2;
    const int stride = gridDim.x * blockDim.x;
    for (int k = blockIdx.x * blockDim.x + threadIdx.x; k < n_words; k += stride) d.ws.x_mask32[k] = 0u;
    for (int64_t j = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; j < (int64_t)d.nb * 16; j += stride)
        d.ws.x_dense[j] = __uint_as_float(X_ABSENT);
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        Counters *c = d.ws.ctr;
        c->last_n_nzblk = c->n_nzblk;
        c->last_n_tasks = c->n_tasks;
        c->last_path = c->path;
        c->last_y_nnz = (int32_t)d.m;
        c->n_nzblk = 0;
        c->n_tasks = 0;
        c->n_hubs = 0;
    }
}

// Test hook: the bounded wait of the staging code on a barrier that nothing will ever arrive on
// (no copy is in flight, so there is nothing to drain): the wait gives up after `max_tries`
// tries and the kernel records DBSPMSPV_ERR_TIMEOUT, exactly as the pull traversal would.
__global__ void k_wait_probe(Device d, int max_tries) {
    __shared__ uint64_t bar;
    if (threadIdx.x == 0) {
        mbar_init(&bar, 1);
        fence_barrier_init();
        if (!mbar_wait_bounded(&bar, 0u, max_tries)) d.ws.ctr->status = DBSPMSPV_ERR_TIMEOUT;
    }
}

__global__ void k_fill_u32(uint32_t *p, int64_t n, uint32_t v) {
    pdl_wait();
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) p[i] = v;
}

// ------------------------------------------------------------------------------------------
// Host side
// ------------------------------------------------------------------------------------------
template <typename T> static int dev_alloc_zero(T **p, size_t count, int64_t *total) {
    void *q = nullptr;
    size_t bytes = (count ? count : 1) * sizeof(T);
    if (cudaMalloc(&q, bytes) != cudaSuccess) return DBSPMSPV_ERR_ALLOC;
    if (cudaMemset(q, 0, bytes) != cudaSuccess) return DBSPMSPV_ERR_CUDA;
    *p = static_cast<T *>(q);
    *total += (int64_t)bytes;
    return DBSPMSPV_OK;
}

// Persistent grid of the traversal kernel: as many thread blocks as fit (0 on error).
template <int DT, typename Out, int MODE> static int compute_grid(int sm_count) {
    const size_t smem = compute_dyn_smem<MODE>();
    if (cudaFuncSetAttribute(k_compute<DT, Out, MODE>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem) != cudaSuccess) return 0;
    int per_sm = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_compute<DT, Out, MODE>, CTA, smem) != cudaSuccess || per_sm < 1) return 0;
    return sm_count * per_sm;
}

template <int DT, typename Out, int MODE>
static int launch_compute(dbspmspv_handle_s *h, CallList &calls, Out out, float th3, int pull_done = 0) {
    // (one handle launches one instantiation per output kind; the decode entry of a handle and its
    // run entry differ in Out, hence the two slots)
    int &grid = Out::MASKS ? h->grid_compute : h->grid_compute_dense;
    if (!grid) grid = compute_grid<DT, Out, MODE>(h->sm_count);
    if (!grid) return DBSPMSPV_ERR_CUDA;
    const size_t smem = compute_dyn_smem<MODE>();
    calls.add(k_compute<DT, Out, MODE>, grid, CTA, smem, true, h->d, out, th3, h->ropts.force_path, h->ropts.popc_threshold, pull_done);
    return DBSPMSPV_OK;
}

// The streaming pull of hypersparse handles (lean_pull.cuh), launched behind k_compute.
template <int DT, typename Out, bool LONG = false>
static int launch_lean(dbspmspv_handle_s *h, CallList &calls, Out out, float th3, int boolean_push = 0) {
    bool &configured = (Out::MINPLUS ? h->lean_configured_min : Out::MASKS ? h->lean_configured : h->lean_configured_dense)[LONG];
    // filter size: the power of two that holds one bit per column, capped
    const int n_words = (h->d.nb + 1) / 2;
    int filter_words = 32;
    while (filter_words < n_words && filter_words < LEAN_FILTER_MAX_WORDS) filter_words <<= 1;
    const size_t smem = (size_t)filter_words * 4 + LEAN_WARPS * sizeof(LeanScratch);
    if (!configured) {
        // (the attribute belongs to the kernel, not to the handle: the largest size, or a handle with few columns would lower it
        // below what one with many, configured before, asks for)
        constexpr int most = LEAN_FILTER_MAX_WORDS * 4 + LEAN_WARPS * (int)sizeof(LeanScratch);
        auto kernel = k_pull_lean<DT, Out, LONG>;
        if (cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, most) != cudaSuccess) return DBSPMSPV_ERR_CUDA;
        configured = true;
    }
    calls.add(k_pull_lean<DT, Out, LONG>, h->sm_count, LEAN_CTA, smem, true, h->d, out, th3, h->ropts.force_path, h->ropts.popc_threshold, filter_words, boolean_push);
    return DBSPMSPV_OK;
}

// Upper bound of the selector's ratio known on the host: with at most `nnz_x` listed columns no
// more than min(nnz_x, nb) vector blocks are nonempty.  When even that stays below th3 the push
// is certain and the pull kernel need not be launched.
static bool pull_possible(const dbspmspv_handle_s *h, int64_t nnz_x, float th3) {
    if (h->ropts.force_path == DBSPMSPV_PATH_PUSH) return false;
    if (h->ropts.force_path == DBSPMSPV_PATH_PULL) return true;
    const int64_t most = nnz_x < h->d.nb ? nnz_x : h->d.nb;
    return !((float)most / (float)h->d.nb < th3);
}

int allocate_workspace(dbspmspv_handle_s *h) {
    Device &d = h->d;
    Workspace &ws = d.ws;
    int64_t total = 0;
    const size_t xwords = (size_t)(d.nb + 1) / 2 + 4, ywords = (size_t)(d.mb + 1) / 2 + 4;
    // Entries with a payload per push task: a full warp step where such blocks are the bulk of
    // the matrix (the lanes then share them out); a few where they are the exception and a warp
    // takes them one at a time (32 of them in one task would keep one warp busy for tens of
    // microseconds while the others have long finished).
    d.payload_chunk = h->heavy_stage ? PUSH_CHUNK : 4;
    // one partial task at most per column (INLINE run) and per column block (payload run)
    // (Handles whose elements sit mostly in blocks with a payload take a column block as one run; elsewhere its entries with a payload
    // and its columns are runs of their own.)
    ws.task_capacity = h->heavy_stage ? (int64_t)d.n_entries / PUSH_CHUNK + 17 * (int64_t)d.nb + 32
                                      : (int64_t)d.n_entries / PUSH_CHUNK + (int64_t)d.n_payload / d.payload_chunk + 17 * (int64_t)d.nb + 32;
    if (ws.task_capacity < (d.m + 1) / 2 + 32) ws.task_capacity = (d.m + 1) / 2 + 32;      // (the short call parks the result's rows there)
    ws.n_tiles = (int32_t)ceil_div<int64_t>((d.mb + 1) / 2, TILE_WORDS);
    if (ws.n_tiles < 1) ws.n_tiles = 1;
    // One allocation for the whole workspace, carved at 512-byte boundaries (a dozen cudaMalloc
    // calls fewer per handle).  Where the driver places its pages still matters: the same push
    // kernel measured 68 .. 83 us on the same data from one allocation history to the next.
    size_t off = 0;
    // (arrays of a megabyte or more start on a 2 MB boundary, the others on a 512-byte one)
    auto carve = [&](size_t bytes) {
        const size_t a = bytes >= ((size_t)1 << 20) ? ((size_t)2 << 20) : 512;
        off = (off + a - 1) / a * a;
        const size_t o = off;
        off += (bytes + 511) & ~(size_t)511;
        return o;
    };
    const size_t zwords = xwords > ywords ? xwords : ywords;
    const size_t o_xd = carve(xwords * 32 * sizeof(float)), o_yacc = carve(ywords * 32 * sizeof(float)),
                 o_long = carve((size_t)d.long_cap * sizeof(*ws.long_runs)), o_tasks = carve((size_t)ws.task_capacity * sizeof(*ws.tasks)),
                 o_verts = carve((d.m == d.n ? 4 * BFS_LIST : 1) * sizeof(*ws.bfs_verts)),
                 o_xm = carve(xwords * 4), o_ym = carve(ywords * 4), o_zm = carve(zwords * 4),
                 o_words = carve(4 * zwords * sizeof(*ws.bfs_words)), o_vis = carve((d.m == d.n ? ywords : 1) * 4),
                 o_hubs = carve((size_t)3 * HUB_CAP * sizeof(*ws.hubs)), o_tile = carve((size_t)ws.n_tiles * sizeof(*ws.tile_status)),
                 o_group = carve((size_t)2 * ((ws.n_tiles + FINISH_GROUP - 1) / FINISH_GROUP) * sizeof(*ws.tile_group)),
                 o_ctr = carve(sizeof(*ws.ctr));
    void *arena = nullptr;
    if (cudaMalloc(&arena, off) != cudaSuccess) return DBSPMSPV_ERR_ALLOC;
    h->ws_arena = arena;
    if (cudaMemset(arena, 0, off) != cudaSuccess) return DBSPMSPV_ERR_CUDA;
    uint8_t *base = static_cast<uint8_t *>(arena);
    ws.x_dense = reinterpret_cast<decltype(ws.x_dense)>(base + o_xd);
    ws.y_acc = reinterpret_cast<decltype(ws.y_acc)>(base + o_yacc);
    ws.long_runs = reinterpret_cast<decltype(ws.long_runs)>(base + o_long);
    ws.bfs_verts = reinterpret_cast<decltype(ws.bfs_verts)>(base + o_verts);
    ws.tasks = reinterpret_cast<decltype(ws.tasks)>(base + o_tasks);
    ws.x_mask32 = reinterpret_cast<decltype(ws.x_mask32)>(base + o_xm);
    ws.y_mask32 = reinterpret_cast<decltype(ws.y_mask32)>(base + o_ym);
    ws.z_mask32 = reinterpret_cast<decltype(ws.z_mask32)>(base + o_zm);
    ws.bfs_words = reinterpret_cast<decltype(ws.bfs_words)>(base + o_words);
    ws.bfs_words_stride = (int32_t)zwords;
    ws.visited32 = reinterpret_cast<decltype(ws.visited32)>(base + o_vis);
    ws.hubs = reinterpret_cast<decltype(ws.hubs)>(base + o_hubs);
    ws.tile_status = reinterpret_cast<decltype(ws.tile_status)>(base + o_tile);
    ws.tile_group = reinterpret_cast<decltype(ws.tile_group)>(base + o_group);
    ws.n_tile_groups = (ws.n_tiles + FINISH_GROUP - 1) / FINISH_GROUP;
    ws.ctr = reinterpret_cast<decltype(ws.ctr)>(base + o_ctr);
    total = (int64_t)off;
    h->stats.workspace_bytes = total;
    // (status words of parity 1: the first call waits for words of parity 0)
    if (cudaMemset(ws.tile_status, 0xFF, (size_t)ws.n_tiles * sizeof(*ws.tile_status)) != cudaSuccess) return DBSPMSPV_ERR_CUDA;
    if (cudaMemset(ws.x_dense, 0xFF, xwords * 32 * sizeof(float)) != cudaSuccess) return DBSPMSPV_ERR_CUDA;
    {   // 0xFFFFFFFF -> the marker pattern 0x7FFFFFFF needs a kernel; a tiny fill does it
        uint32_t *p = reinterpret_cast<uint32_t *>(ws.x_dense);
        k_fill_u32<<<256, 256>>>(p, (int64_t)xwords * 32, X_ABSENT);
        k_fill_u32<<<256, 256>>>(reinterpret_cast<uint32_t *>(ws.y_acc), (int64_t)ywords * 32, ACC_CLEAR);
        if (cudaDeviceSynchronize() != cudaSuccess) return DBSPMSPV_ERR_CUDA;
    }
    // events for the optional kernel timing are made here so that run-time calls create nothing
    if (cudaEventCreate(&h->ev[0]) != cudaSuccess || cudaEventCreate(&h->ev[1]) != cudaSuccess) return DBSPMSPV_ERR_CUDA;
    return DBSPMSPV_OK;
}

// Columns up to which a call takes its one-kernel form (small_call.cuh).  It is the faster one up to all of these lines, and by now beyond them: uniform rows, 48 / 96 / 160 / 250 columns, one kernel
// against the chain of two, whose launches the host is bound by: 16 K rows 5.3 / 5.4 / 5.7 / 6.4 against 6.3 us a call, 128 K 5.5 / 5.6 / 6.2 / 6.5 against 6.5, 256 K 5.6 / 5.6 / 5.9 / 6.3 against 8.2 / 6.6 /
// 6.5 / 6.5, 512 K 5.7 / 6.0 / 6.2 / 6.5 against 8.9 / 8.6 / 8.1 / 7.8, a million 6.3 / 6.5 / 6.6 / 7.0 against 10.  With long columns, R-MAT in scattered order, against the chain of three: 16 K rows
// 5.7 / 6.1 / 7.2 / 7.6 against 8.5 - 9.6, 256 K 7.3 / 6.1 / 6.7 / 7.2 against 8.7 - 9.3, 512 K 5.8 / 6.7 / 8.5 / 9.0 against 10, a million 7.1 / 7.2 / 8.6 / 8.5 against 13.7.  Not relabelled (more payload
// blocks) both vary by half with the columns that x lists: 16 K 7.8 / 9.2 / 10.4 / 13.3 against 9.4 / 9.8 / 9.9 / 10.2, 256 K 9.4 / 10.8 / 11.3 / 12.4 against 10.4 - 10.8, a million 6.9 / 7.8 / 13.1 / 13.7
// against 13.5 - 14.2.  The lines are those of an earlier, slower one-kernel form (7.5 us where it is 5.5 now) and stay because callers' launch counts are tested on both sides of them.
static int small_call_limit(const dbspmspv_handle_s *h) {
    const Device &d = h->d;
    if (d.long_cap == 0) return d.m <= (1 << 17) ? 48 : d.m <= 5 << 16 ? 64 : d.m <= 5 << 17 ? 96 : d.m <= 7 << 17 ? 144 : 224;
    if ((int64_t)d.n_payload * 2048 > d.n_entries) return SMALL_MAX_NNZ_X;
    return d.m <= (1 << 19) ? 96 : 160;
}

template <int DT>
static int run_typed(dbspmspv_handle_s *h, const int32_t *x_idx, const void *x_val, int32_t nnz_x,
                     int semiring, int32_t *y_idx, float *y_val, int64_t y_capacity, int32_t *y_nnz,
                     cudaStream_t st, const uint32_t *row_mask = nullptr, int complement = 0) {
    const Device &d = h->d;
    CallList calls;
    // a short x on a hypersparse handle: the whole call as one kernel of one thread-block cluster (small_call.cuh)
    {
        const size_t ywords = (size_t)(d.mb + 1) / 2, cbwords = (size_t)(d.nb + 31) / 32;
        const size_t smem = ((ywords + SMALL_CLUSTER - 1) / SMALL_CLUSTER + (cbwords + SMALL_CLUSTER - 1) / SMALL_CLUSTER) * sizeof(uint32_t);
        if (nnz_x > 0 && nnz_x <= small_call_limit(h) && d.n_entries > 0 && !h->heavy_stage && !h->ropts.validate && !h->ropts.timing &&
            !h->ropts.no_small_call && h->ropts.force_path != DBSPMSPV_PATH_PULL && !pull_possible(h, nnz_x, h->ropts.th3) &&
            smem <= SMALL_MAX_SMEM && (int64_t)ywords * 32 * (int64_t)sizeof(int32_t) <= d.ws.task_capacity * (int64_t)sizeof(*d.ws.tasks)) {
            const int mode = semiring == DBSPMSPV_OR_AND ? 1 : semiring == DBSPMSPV_MIN_PLUS ? 2 : 0;
            if (!h->small_configured) {
                // (the attribute belongs to the kernel, not to the handle: the largest size)
                DBS_CUDA(cudaFuncSetAttribute(k_run_small<DT>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)SMALL_MAX_SMEM + SMALL_ROWS * (int)sizeof(int)));
                h->small_configured = true;
            }
            calls.add(k_run_small<DT>, SMALL_CLUSTER, SMALL_CTA, smem + SMALL_ROWS * sizeof(int), false, d, x_idx, x_val, nnz_x, mode, y_idx, y_val, y_capacity, y_nnz, row_mask, complement);
            return submit_calls(h, calls, st);
        }
    }
    const bool minplus = semiring == DBSPMSPV_MIN_PLUS, boolean = semiring == DBSPMSPV_OR_AND || (DT == DBSPMSPV_PATTERN && !minplus);
    const void *xv = semiring == DBSPMSPV_OR_AND ? nullptr : x_val;
    const bool any = nnz_x > 0 && d.n_entries > 0;
    const int fp = h->ropts.force_path;
    int clear = CLEAR_MASKS | CLEAR_DENSE;
    h->d.hub_on = 0;
    if (!h->heavy_stage) {
        // Hypersparse handles: direct push, pull by the streaming kernel.  (min, +) pulls only on valued handles.
        const bool may_pull = (!minplus || DT != DBSPMSPV_PATTERN) && pull_possible(h, nnz_x, h->ropts.th3);
        const bool may_push = !may_pull || fp != DBSPMSPV_PATH_PULL;
        const int mode = boolean ? 1 : minplus ? 2 : 0;
        const bool groups = h->payload_rich && nnz_x >= PD_GROUPS_MIN_NNZ_X;
        const bool long_in_pull = any && may_pull && may_push && d.long_cap && !groups && d.n_entries <= LONG_IN_PULL_ENTRIES;
        // private accumulators for the hub row blocks, when x is long enough for their atomics to queue up
        const int hub_min = h->ropts.hub_min_nnz_x ? h->ropts.hub_min_nnz_x : HUB_MIN_NNZ_X;
        h->d.hub_on = may_push && d.n_hub_blocks > 0 && hub_min > 0 && nnz_x >= hub_min ? (nnz_x < HUB_ALL_NNZ_X ? 4 : HUB_COPIES) : 0;
        if (may_pull && nnz_x > 0) calls.add(k_xblock_sparse<DT, false>, (nnz_x + XB_TPB - 1) / XB_TPB, XB_TPB, 0, false, d, x_idx, xv, nnz_x, h->ropts.validate);
        if (h->ropts.timing) calls.ev_before = calls.n;
        if (nnz_x > 0 && may_push) {
            auto push = [&](auto list_kernel, auto mask_kernel, auto long_kernel) {
                if (may_pull) {
                    // (decided on the device) 32 mask words per thread block and round
                    const int n_words = (d.nb + 1) / 2;
                    int g = (n_words + PD_MASK_WORDS - 1) / PD_MASK_WORDS;
                    // (fewer words each where there would not be a thread block for every place on the GPU: 63 of them took 21 us over 64 K columns)
                    const int places = pd_per_sm(true) * h->sm_count;
                    if (g < places) g = n_words < places ? n_words : places;
                    if (g > 65536) g = 65536;
                    calls.add(mask_kernel, g, PD_CTA, 0, true, d, x_idx, xv, nnz_x, 0, h->ropts.th3, fp, 0, (n_words + PD_MASK_WORDS * g - 1) / (PD_MASK_WORDS * g));
                } else {
                    // columns per thread block: few enough to fill the GPU, at least eight
                    const int most = pd_per_sm(false) * h->sm_count;
                    int cols = (nnz_x + most - 1) / most;
                    cols = cols <= 8 ? 8 : cols >= PD_CTA ? PD_CTA : (cols + 7) & ~7;
                    int g = (nnz_x + cols - 1) / cols;
                    if (g > most) g = most;
                    calls.add(list_kernel, g, PD_CTA, 0, false, d, x_idx, xv, nnz_x, (int)h->ropts.validate, h->ropts.th3, fp, cols, (nnz_x + cols * g - 1) / (cols * g));
                }
                if (d.long_cap && !long_in_pull) calls.add(long_kernel, 6 * h->sm_count, PD_CTA, 0, true, d);
            };
            constexpr int VT = DT == DBSPMSPV_PATTERN ? DBSPMSPV_F32 : DT;       // (pattern handles have no (+, *))
            if (mode == 1 && groups) push(k_push_direct<DT, 1, false, true>, k_push_direct<DT, 1, true, true>, k_push_long<DT, 1, true>);
            else if (mode == 1) push(k_push_direct<DT, 1, false, false>, k_push_direct<DT, 1, true, false>, k_push_long<DT, 1, false>);
            else if (mode == 2 && groups) push(k_push_direct<DT, 2, false, true>, k_push_direct<DT, 2, true, true>, k_push_long<DT, 2, true>);
            else if (mode == 2) push(k_push_direct<DT, 2, false, false>, k_push_direct<DT, 2, true, false>, k_push_long<DT, 2, false>);
            else if (DT != DBSPMSPV_PATTERN && groups) push(k_push_direct<VT, 0, false, true>, k_push_direct<VT, 0, true, true>, k_push_long<VT, 0, true>);
            else if (DT != DBSPMSPV_PATTERN) push(k_push_direct<VT, 0, false, false>, k_push_direct<VT, 0, true, false>, k_push_long<VT, 0, false>);
        }
        if (any && may_pull) {
            const OutSparse out{d.ws.y_acc, d.ws.y_mask32};
            const OutSparseMin out_min{d.ws.y_acc, d.ws.y_mask32};
            const int s = minplus ? (long_in_pull ? launch_lean<DT, OutSparseMin, true>(h, calls, out_min, h->ropts.th3) : launch_lean<DT, OutSparseMin>(h, calls, out_min, h->ropts.th3))
                                  : (long_in_pull ? launch_lean<DT, OutSparse, true>(h, calls, out, h->ropts.th3, mode == 1) : launch_lean<DT, OutSparse>(h, calls, out, h->ropts.th3));
            if (s != DBSPMSPV_OK) return s;
        }
        if (!may_pull && (mode == 1 || !groups)) clear = CLEAR_MASKS;      // (x was staged for the payload entries only)
    } else {
        if (nnz_x > 0) calls.add(k_xblock_sparse<DT, true>, (nnz_x + XB_TPB - 1) / XB_TPB, XB_TPB, 0, false, d, x_idx, xv, nnz_x, h->ropts.validate);
        if (h->ropts.timing) calls.ev_before = calls.n;
        if (any && minplus) {
            calls.add(k_minplus_push<DT>, 4 * h->sm_count, MINPLUS_CTA, 0, true, d, h->ropts.th3, (int)DBSPMSPV_PATH_PUSH);
        } else if (any) {
            const int s = launch_compute<DT, OutSparse, 1>(h, calls, OutSparse{d.ws.y_acc, d.ws.y_mask32}, h->ropts.th3);
            if (s != DBSPMSPV_OK) return s;
        }
    }
    if (h->ropts.timing) { calls.ev_after = calls.n; h->timed = true; }
    const int nt = d.ws.n_tiles;
    int extra = (nnz_x + CMP_TPB * 8 - 1) / (CMP_TPB * 8);
    if (extra > 4 * h->sm_count) extra = 4 * h->sm_count;
    // scattered clears cost more than a full sweep once x lists a good part of the columns (a sweep of the masks alone is 32 times shorter)
    if ((int64_t)nnz_x * (clear & CLEAR_DENSE ? 8 : 128) > d.n) clear |= CLEAR_SWEEP;
    // several tiles per thread block where they would come in waves (eight thread blocks per SM); behind a short push of whole blocks, which
    // leaves most tiles untouched, from two thread blocks per SM on (27-point operator on 97^3, 110^3, 128^3, 130^3 cells, x = 0.03 %: 17.3, 18.0, 18.0, 19.9 us
    // a call with a tile each, 14.6, 15.7, 14.6, 16.6 so; at 0.5 % the same, at 1 % up to 1.5 slower.  Behind a direct push, whose results lie everywhere,
    // it is the slower form in one wave: R-MAT scale 20, 0.2 %, 13.2 against 15.0)
    const int wave = (h->heavy_stage && (int64_t)nnz_x * 128 <= d.n ? 2 : 8) * h->sm_count;
    int per_block = (nt + wave - 1) / wave;
    if (per_block > FINISH_WIDE) per_block = FINISH_WIDE;
    // (results in good part of the rows: fetching them twice costs more than the waves, 24 us against 19 with nearly all rows)
    if ((int64_t)nnz_x * 64 > d.n) per_block = 1;
    if (per_block > 1)
        calls.add(d.hub_on ? k_finish_wide<true> : k_finish_wide<false>, (nt + per_block - 1) / per_block + extra, CMP_TPB, 0, calls.n > 0, d, per_block, y_idx, y_val, y_capacity, y_nnz,
                  minplus ? 2 : (int)boolean, x_idx, nnz_x, clear, d.hub_on ? (minplus ? 2 : 1) : 0, row_mask, complement);
    else if ((h->heavy_stage || h->payload_rich) && nt > 9 * h->sm_count && !d.hub_on && (int64_t)nnz_x * 16 <= d.n)      // (see k_finish_pair)
        calls.add(k_finish_pair, (nt + 1) / 2 + extra, CMP_TPB, 0, calls.n > 0, d, y_idx, y_val, y_capacity, y_nnz, minplus ? 2 : (int)boolean, x_idx, nnz_x, clear, row_mask, complement);
    else
        calls.add(d.hub_on ? k_finish<true> : k_finish<false>, nt + extra, CMP_TPB, 0, calls.n > 0, d, y_idx, y_val, y_capacity, y_nnz, minplus ? 2 : (int)boolean, x_idx, nnz_x, clear,
                  d.hub_on ? (minplus ? 2 : 1) : 0, row_mask, complement);
    return submit_calls(h, calls, st);
}

// payload bytes of one stage of a warp's ring in the streaming decode: what shared memory leaves
// when two thread blocks share an SM (else one), at most STAGE_BYTES; 0 = no room (a block must fit)
int decode_stage_bytes(const Device &d) {
    const StreamLayout lay(d.nb, 0);
    for (int budget : {DBS_STREAM_BUDGET, STREAM_MAX_SMEM}) {
        const int room = budget - lay.ring_off;
        if (room <= 0) continue;
        int sb = (room / (STREAM_WARPS * STREAM_DEPTH)) & ~511;
        if (sb > STAGE_BYTES) sb = STAGE_BYTES;
        if (sb >= 2048) return sb;
    }
    return 0;
}

// Decode over columns: `nvec` vectors (1, or at most as many as decode_columns_group says).
template <int C>
static int decode_columns_c(dbspmspv_handle_s *h, CallList &calls, const void *x, float *y) {
    const Device &d = h->d;
    const int strips = (int)((d.m + DC_ROWS - 1) / DC_ROWS);
    if (!h->cols_configured) {
        DBS_CUDA(cudaFuncSetAttribute(k_decode_cols<C>, cudaFuncAttributeMaxDynamicSharedMemorySize, FUSED_MAX_SMEM));
        h->cols_configured = true;
    }
    calls.add(k_decode_cols<C>, strips * C, DC_CTA, (size_t)DC_WARPS * dc_warp_entries(d.nb, C) * sizeof(float2), false, d, x, y, h->ropts.th3_decode, h->ropts.force_path);
    return DBSPMSPV_OK;
}
static int decode_columns(dbspmspv_handle_s *h, const void *x, int64_t ldx, float *y, int64_t ldy, int nvec, cudaStream_t st) {
    CallList calls;
    const Device &d = h->d;
    int s = DBSPMSPV_OK;
    if (nvec == 1) {
        switch (dc_cluster(d.m, h->sm_count)) {
            case 1: s = decode_columns_c<1>(h, calls, x, y); break;
            case 2: s = decode_columns_c<2>(h, calls, x, y); break;
            case 4: s = decode_columns_c<4>(h, calls, x, y); break;
            default: s = decode_columns_c<8>(h, calls, x, y); break;
        }
        if (s != DBSPMSPV_OK) return s;
    } else {
        const int nv = nvec <= 4 ? 4 : 8;
        auto kernel = nv == 4 ? k_decode_cols_batch<4> : k_decode_cols_batch<8>;
        if (!h->cols_batch_configured[nv / 8]) {
            // (the attribute belongs to the kernel, not to the handle: the largest size)
            DBS_CUDA(cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, DCB_MAX_SMEM));
            h->cols_batch_configured[nv / 8] = true;
        }
        calls.add(k_zero_rows, (int)((d.m + 255) / 256), 256, 0, false, y, ldy, d.m, nvec);
        calls.add(kernel, h->sm_count, DCB_CTA, (size_t)DcBatchLayout(d.nb, nv).total, true, d, x, ldx, y, ldy, nvec, h->ropts.th3_decode, h->ropts.force_path);
    }
    if (h->ropts.timing) { calls.ev_before = 0; calls.ev_after = calls.n; h->timed = true; }
    return submit_calls(h, calls, st);
}
// vectors of one batched call over columns, at most (1: the lists of several do not fit in shared memory)
static int decode_columns_group(const dbspmspv_handle_s *h) {
    for (int nv : {8, 4})
        if (DcBatchLayout(h->d.nb, nv).total <= DCB_MAX_SMEM) return nv;
    return 1;
}

template <int DT>
static int decode_typed(dbspmspv_handle_s *h, const void *x, float *y, cudaStream_t st) {
    const Device &d = h->d;
    CallList calls;
    h->d.decode_tau = h->ropts.decode_threshold;
    h->d.decode_relu = h->ropts.decode_relu != 0;
    h->d.decode_x_f32 = h->ropts.decode_x_f32 != 0;
    if (DT == DBSPMSPV_BF16 && d.cols && h->ropts.no_fused_decode == 0) return decode_columns(h, x, 0, y, 0, 1, st);
    // (-1: no decode call has reported yet)
    const int seen = h->x_nnz_seen_host ? *const_cast<volatile int32_t *>(h->x_nnz_seen_host) : -1;
    const bool sparse_x = seen >= 0 && (float)seen < STREAM_MIN_X_DENSITY * (float)d.n;
    h->d.x_sparse_believed = sparse_x;
    if (h->heavy_stage && d.stage_chunks != nullptr && (h->ropts.no_fused_decode == 3 || (h->ropts.no_fused_decode == 0 && !sparse_x))) {
        // the streaming form: one persistent kernel behind a memset of y
        const StreamLayout lay(d.nb, d.stage_bytes);
        if (!h->stream_grid) {
            // (the attribute belongs to the kernel, not to the handle: always the largest size)
            DBS_CUDA(cudaFuncSetAttribute(k_decode_stream<DT>, cudaFuncAttributeMaxDynamicSharedMemorySize, STREAM_MAX_SMEM));
            int per_sm = 0;
            DBS_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_decode_stream<DT>, STREAM_CTA, lay.total));
            if (per_sm < 1) return DBSPMSPV_ERR_CUDA;
            h->stream_grid = per_sm * h->sm_count;
        }
        if (h->ropts.timing) { calls.ev_before = 0; calls.ev_after = 2; h->timed = true; }
        calls.add(k_fill_u32, (int)((d.m + 1023) / 1024), 256, 0, false, reinterpret_cast<uint32_t *>(y), d.m, 0u);
        calls.add(k_decode_stream<DT>, h->stream_grid, STREAM_CTA, (size_t)lay.total, true, d, x, y, h->ropts.th3_decode, h->ropts.force_path);
        return submit_calls(h, calls, st);
    }
    if (h->heavy_stage && h->ropts.no_fused_decode != 1) {
        // one kernel for the whole call, when x fits in shared memory
        const int per_rb = d.mb ? d.n_entries / d.mb : 0;
        // warps per thread block from the entries per row block (measured on the three layer
        // shapes: more, smaller warps-per-block steps were 5-30 % slower)
        const int nw = per_rb <= 384 ? 4 : per_rb <= 1024 ? 8 : 16;
        const FusedLayout lay(d.nb, nw * 32);
        if (lay.total <= FUSED_MAX_SMEM) {
            auto kernel = nw == 4 ? k_decode_fused<DT, 4> : nw == 8 ? k_decode_fused<DT, 8> : k_decode_fused<DT, 16>;
            bool &done = h->fused_configured[nw == 4 ? 0 : nw == 8 ? 1 : 2];
            if (!done) {
                DBS_CUDA(cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, FUSED_MAX_SMEM));
                done = true;
            }
            if (h->ropts.timing) { calls.ev_before = 0; calls.ev_after = 1; h->timed = true; }
            calls.add(kernel, d.mb, nw * 32, (size_t)lay.total, false, d, x, y, h->ropts.th3_decode, h->ropts.force_path);
            return submit_calls(h, calls, st);
        }
    }
    const int64_t padded = (int64_t)((d.nb + 1) / 2) * 32;
    int64_t work = padded > d.m ? padded : d.m;
    int g = (int)((work + 255) / 256);
    if (g > 8 * h->sm_count) g = 8 * h->sm_count;
    calls.add(k_xblock_dense<DT>, g, 256, 0, false, d, x, y);
    OutDense out{y, nullptr};
    if (h->ropts.timing) calls.ev_before = calls.n;
    if (d.n_entries > 0) {
        int s;
        if (h->heavy_stage) {
            // pull by the lean kernel of its own; the general kernel then only runs a push
            int &grid = h->grid_decode_pull;
            if (!grid) {
                int per_sm = 0;
                if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_decode_pull<DT>, CTA, 0) != cudaSuccess || per_sm < 1) return DBSPMSPV_ERR_CUDA;
                grid = per_sm * h->sm_count;
            }
            calls.add(k_decode_pull<DT>, grid, CTA, 0, true, d, (const int32_t *)h->block_row, y, h->ropts.th3_decode, h->ropts.force_path);
            s = launch_compute<DT, OutDense, 1>(h, calls, out, h->ropts.th3_decode, 1);
        } else {
            s = DBSPMSPV_OK;
            if (h->ropts.force_path != DBSPMSPV_PATH_PULL) s = launch_compute<DT, OutDense, 0>(h, calls, out, h->ropts.th3_decode);
            if (s == DBSPMSPV_OK && pull_possible(h, d.n, h->ropts.th3_decode)) s = launch_lean<DT, OutDense>(h, calls, out, h->ropts.th3_decode);
        }
        if (s != DBSPMSPV_OK) return s;
    }
    if (h->ropts.timing) { calls.ev_after = calls.n; h->timed = true; }
    int gc = ((d.nb + 1) / 2 + 255) / 256;
    if (gc > h->sm_count) gc = h->sm_count;
    calls.add(k_decode_cleanup, gc, 256, 0, true, d);
    return submit_calls(h, calls, st);
}

// dbspmspv_decode_batch: where the handle has the streaming form, groups of vectors share one
// pass over the payload -- bf16 handles: up to eight per group on the tensor cores
// (k_decode_batch_mma), with the per-column kernel launched behind it as the fallback for
// non-finite activations; fp32 handles: up to four per group in the per-column kernel.  What is
// left over (and every vector of a handle without the streaming form) goes through decode_typed.
template <int DT>
static int decode_batch_typed(dbspmspv_handle_s *h, const void *x, int64_t ldx, float *y, int64_t ldy, int32_t batch,
                              cudaStream_t st) {
    const Device &d = h->d;
    const size_t esize = (DT == DBSPMSPV_BF16 && !h->ropts.decode_x_f32) ? 2 : 4;
    const bool stream_ok = h->heavy_stage && d.stage_chunks != nullptr && (h->ropts.no_fused_decode == 0 || h->ropts.no_fused_decode == 3);
    int max_nb = 1, max_mma = 1;
    if (stream_ok) {
        for (int nb : {2, 4})
            if (BatchLayout(d.nb, nb, d.stage_bytes).total <= STREAM_MAX_SMEM) max_nb = nb;
        if (DT == DBSPMSPV_BF16)
            for (int nb : {2, 4, 8})
                if (max_nb >= (nb < 4 ? nb : 4) && BatchMmaLayout(d.nb, nb, d.stage_bytes).total <= STREAM_MAX_SMEM) max_mma = nb;
    }
    h->d.decode_tau = h->ropts.decode_threshold;
    h->d.decode_relu = h->ropts.decode_relu != 0;
    h->d.decode_x_f32 = h->ropts.decode_x_f32 != 0;
    const int cols_group = DT == DBSPMSPV_BF16 && d.cols && h->ropts.no_fused_decode == 0 ? decode_columns_group(h) : 0;
    // the per-column kernel on vectors [b0, b0 + g), g <= 4
    auto scalar_group = [&](CallList &calls, const void *xg, float *yg, int g, int only_as_fallback) -> int {
        const int nb = g <= 2 ? 2 : 4;
        const BatchLayout lay(d.nb, nb, d.stage_bytes);
        auto kernel = nb == 2 ? k_decode_stream_batch<DT, 2> : k_decode_stream_batch<DT, 4>;
        bool &done = h->batch_configured[nb == 2 ? 0 : 1];
        if (!done) {
            DBS_CUDA(cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, STREAM_MAX_SMEM));
            done = true;
        }
        calls.add(kernel, h->sm_count, BATCH_CTA, (size_t)lay.total, true, d, xg, ldx, yg, ldy, g, only_as_fallback);
        return DBSPMSPV_OK;
    };
    // (Over columns, 50 % pruned, 30 % active, two vectors in one pass against two single calls: 2048 x 2048 9.1 against 13.0 us, 4096 x 4096 12.3 / 13.3,
    // 8192 x 4096 16.6 / 13.4, 12288 x 4096 21.4 / 16.3, 8192 x 12288 34.6 / 38.7; three vectors 19 - 40 against 20 - 58.)
    for (int32_t b0 = 0; b0 < batch;) {
        const int left = batch - b0;
        const void *xg = static_cast<const uint8_t *>(x) + (size_t)b0 * (size_t)ldx * esize;
        float *yg = y + (size_t)b0 * (size_t)ldy;
        const int cap = cols_group > 1 ? cols_group : DT == DBSPMSPV_BF16 && max_mma > 1 ? max_mma : max_nb;
        const int g = left < cap ? left : cap;
        if (g == 1) {
            const int s = decode_typed<DT>(h, xg, yg, st);
            if (s != DBSPMSPV_OK) return s;
            b0 += 1;
            continue;
        }
        if (cols_group > 1) {
            const int s = decode_columns(h, xg, ldx, yg, ldy, g, st);
            if (s != DBSPMSPV_OK) return s;
            b0 += g;
            continue;
        }
        CallList calls;
        if (h->ropts.timing) calls.ev_before = 0;
        calls.add(k_zero_rows, (int)((d.m + 255) / 256), 256, 0, false, yg, ldy, d.m, g);
        if (DT == DBSPMSPV_BF16 && max_mma > 1) {
            const int nb = g <= 2 ? 2 : g <= 4 ? 4 : 8;
            const BatchMmaLayout lay(d.nb, nb, d.stage_bytes);
            auto kernel = nb == 2 ? k_decode_batch_mma<2> : nb == 4 ? k_decode_batch_mma<4> : k_decode_batch_mma<8>;
            bool &done = h->batch_mma_configured[nb == 2 ? 0 : nb == 4 ? 1 : 2];
            if (!done) {
                DBS_CUDA(cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, STREAM_MAX_SMEM));
                done = true;
            }
            calls.add(kernel, h->sm_count, BATCH_MMA_CTA, (size_t)lay.total, true, d, xg, ldx, yg, ldy, g);
            // the fallback for non-finite activations: returns at once unless the kernel above asked for it
            for (int q = 0; q < g; q += 4) {
                const int gq = g - q < 4 ? g - q : 4;
                const int s = scalar_group(calls, static_cast<const uint8_t *>(xg) + (size_t)q * (size_t)ldx * esize, yg + (size_t)q * (size_t)ldy, gq, 1);
                if (s != DBSPMSPV_OK) return s;
            }
        } else {
            const int s = scalar_group(calls, xg, yg, g, 0);
            if (s != DBSPMSPV_OK) return s;
        }
        if (h->ropts.timing) { calls.ev_after = calls.n; h->timed = true; }
        const int s = submit_calls(h, calls, st);
        if (s != DBSPMSPV_OK) return s;
        b0 += g;
    }
    return DBSPMSPV_OK;
}

// ------------------------------------------------------------------------------------------
// db_sssp: single-source shortest paths as the iteration of (min, +) products (Sections 1, 6:
// SpMSpV as the primitive of GraphBLAS-style graph algorithms).  x = the vertices whose
// distance improved in the last step, with their distances; y = A (min,+) x; every y_i below
// dist_i replaces it and puts i on the next x.  The rows of y are distinct, so the relaxation
// needs no atomics on dist.
// ------------------------------------------------------------------------------------------
__global__ void k_sssp_init(float *dist, int64_t n, int32_t src, int32_t *x_idx, float *x_val, int32_t *count) {
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t v = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; v < n; v += stride) dist[v] = v == src ? 0.0f : __int_as_float(0x7F800000);
    if (blockIdx.x == 0 && threadIdx.x == 0) { x_idx[0] = src; x_val[0] = 0.0f; count[0] = 0; }
}

// count[0]: entries of the next x
__global__ void k_sssp_relax(const int32_t *__restrict__ y_idx, const float *__restrict__ y_val, const int32_t *__restrict__ y_nnz,
                             float *__restrict__ dist, int32_t *__restrict__ x_idx, float *__restrict__ x_val, int32_t *count) {
    const int n = *y_nnz;
    const int lane = threadIdx.x & 31;
    const int stride = gridDim.x * blockDim.x;
    for (int k0 = (blockIdx.x * blockDim.x + threadIdx.x) - lane; k0 < n; k0 += stride) {     // warp-uniform trip count
        const int k = k0 + lane;
        bool better = false;
        int i = 0;
        float v = 0.f;
        if (k < n) { i = y_idx[k]; v = y_val[k]; better = v < dist[i]; }
        const uint32_t m = __ballot_sync(0xFFFFFFFFu, better);
        if (!m) continue;
        int base = 0;
        if (lane == 0) base = atomicAdd(count, __popc(m));
        base = __shfl_sync(0xFFFFFFFFu, base, 0);
        if (better) {
            const int pos = base + __popc(m & ((1u << lane) - 1u));
            dist[i] = v;
            x_idx[pos] = i;
            x_val[pos] = v;
        }
    }
}

// The whole search as one cooperative launch (sssp.cuh).
template <int DT>
static int sssp_one_launch(dbspmspv_handle_s *h, int32_t src, float *dist, int32_t *n_steps, cudaStream_t st) {
    const Device &d = h->d;
    SsspState s;
    s.n_words = (int32_t)((d.n + 31) / 32);
    const size_t word_bytes = ((size_t)s.n_words * 32 * sizeof(int) + 255) & ~(size_t)255, bit_bytes = ((size_t)s.n_words * 4 + 255) & ~(size_t)255;
    if (!h->sssp_host && cudaHostAlloc(reinterpret_cast<void **>(&h->sssp_host), 4 * sizeof(int32_t), cudaHostAllocDefault) != cudaSuccess) { h->sssp_host = nullptr; return DBSPMSPV_ERR_ALLOC; }
    // chunks of long rows: a row has more than 4 (SSSP_ROUNDS - 1) elements before any of it is listed
    const size_t chunk_bytes = ((size_t)h->nnz / (4 * (SSSP_ROUNDS - 1)) + (size_t)h->nnz / SSSP_CHUNK + 64) * sizeof(int4);
    if (!h->sssp_state) {
        if (cudaMalloc(&h->sssp_state, 2 * word_bytes + 3 * bit_bytes + 256 + 2 * SSSP_LIST * sizeof(int32_t) + chunk_bytes) != cudaSuccess) { h->sssp_state = nullptr; return DBSPMSPV_ERR_ALLOC; }
        DBS_CUDA(cudaFuncSetAttribute(k_sssp<DT>, cudaFuncAttributeMaxDynamicSharedMemorySize, SSSP_SMEM));
    }
    uint8_t *p = static_cast<uint8_t *>(h->sssp_state);
    for (int k = 0; k < 2; ++k) { s.word[k] = reinterpret_cast<int *>(p); p += word_bytes; }
    for (int k = 0; k < 3; ++k) { s.bits[k] = reinterpret_cast<uint32_t *>(p); p += bit_bytes; }
    s.set = reinterpret_cast<SsspSet *>(p);
    s.ctr = reinterpret_cast<int32_t *>(p + 3 * sizeof(SsspSet)); p += 256;
    for (int k = 0; k < 2; ++k) { s.list[k] = reinterpret_cast<int32_t *>(p); p += SSSP_LIST * sizeof(int32_t); }
    s.chunks = reinterpret_cast<int4 *>(p);
    s.report = h->sssp_host;
    // edges from which a step is pulled, the first one and those behind it (sssp.cuh)
    const bool weights = DT != DBSPMSPV_PATTERN;
    const bool rich = weights && h->payload_rich;
    const float rows = (float)d.n, pull = rich && d.n <= (int64_t)h->sm_count * SSSP_CTA ? SSSP_PULL_SHARE_PAYLOAD : SSSP_PULL_SHARE;
    float late = SSSP_LATE_SHARE * (float)d.n_entries;
    if (weights) late = fmaxf(late, rows * fminf(SSSP_LATE_ROWS * (rows / (1 << 20)) * (rows / (1 << 20)), rich ? SSSP_LATE_ROWS : 1.0f));
    Device dev = d;
    int start = SSSP_STARTS;
    for (int64_t made = 0;; start = h->sssp_host[2]) {
        int max_steps = (int)(d.n + 1 - made < SSSP_MAX_STEPS ? d.n + 1 - made : SSSP_MAX_STEPS);
        const bool can_pull = DT == DBSPMSPV_PATTERN ? d.rowrun_ptr != nullptr : d.weightrun != nullptr && d.col_degree != nullptr;
        unsigned pull_edges = can_pull ? (unsigned)(pull * (float)d.n_entries) : ~0u, late_edges = can_pull ? (unsigned)fminf(late, pull * (float)d.n_entries) : ~0u;
        void *args[] = {&dev, &s, &src, &dist, &start, &max_steps, &pull_edges, &late_edges};
        DBS_CUDA(cudaLaunchCooperativeKernel((void *)k_sssp<DT>, dim3(h->sm_count), dim3(SSSP_CTA), args, SSSP_SMEM, st));
        ++h->kernel_launches;
        DBS_CUDA(cudaStreamSynchronize(st));
        made = h->sssp_host[0];
        if (h->sssp_host[1] == 0) { if (n_steps) *n_steps = (int32_t)made; return DBSPMSPV_OK; }
        if (made >= d.n + 1) return DBSPMSPV_ERR_UNSUPPORTED;          // a cycle of negative weight
    }
}

template <int DT>
static int sssp_typed(dbspmspv_handle_s *h, int32_t src, float *dist, int32_t *n_steps, cudaStream_t st) {
    const Device &d = h->d;
    const int64_t n = d.n;
    if (!h->heavy_stage && h->ropts.force_path == DBSPMSPV_PATH_AUTO) return sssp_one_launch<DT>(h, src, dist, n_steps, st);
    // handles whose elements sit mostly in blocks with a payload, and forced directions: (min, +) products in a host loop
    if (!h->sssp_arena) {
        // two x lists (the relaxation writes the one the running product does not read), y, two counters
        const size_t bytes = (size_t)n * (4 * sizeof(int32_t) + 2 * sizeof(float)) + 64;
        if (cudaMalloc(&h->sssp_arena, bytes) != cudaSuccess) { h->sssp_arena = nullptr; return DBSPMSPV_ERR_ALLOC; }
        if (!h->sssp_host && cudaHostAlloc(reinterpret_cast<void **>(&h->sssp_host), 4 * sizeof(int32_t), cudaHostAllocDefault) != cudaSuccess) return DBSPMSPV_ERR_ALLOC;
    }
    int32_t *xi[2], *y_idx, *ctr;
    float *xv[2], *y_val;
    {
        uint8_t *p = static_cast<uint8_t *>(h->sssp_arena);
        xi[0] = reinterpret_cast<int32_t *>(p); p += n * sizeof(int32_t);
        xi[1] = reinterpret_cast<int32_t *>(p); p += n * sizeof(int32_t);
        y_idx = reinterpret_cast<int32_t *>(p); p += n * sizeof(int32_t);
        xv[0] = reinterpret_cast<float *>(p); p += n * sizeof(float);
        xv[1] = reinterpret_cast<float *>(p); p += n * sizeof(float);
        y_val = reinterpret_cast<float *>(p); p += n * sizeof(float);
        ctr = reinterpret_cast<int32_t *>(p);                 // [0] next x count, [1] y_nnz
    }
    k_sssp_init<<<4 * h->sm_count, 256, 0, st>>>(dist, n, src, xi[0], xv[0], ctr);
    ++h->kernel_launches;
    int32_t nnz_x = 1;
    int steps = 0, cur = 0, status = DBSPMSPV_OK;
    while (nnz_x > 0) {
        if (++steps > n + 1) { status = DBSPMSPV_ERR_UNSUPPORTED; break; }          // a cycle of negative weight
        status = run_typed<DT>(h, xi[cur], xv[cur], nnz_x, DBSPMSPV_MIN_PLUS, y_idx, y_val, n, ctr + 1, st);
        if (status != DBSPMSPV_OK) break;
        k_sssp_relax<<<2 * h->sm_count, 256, 0, st>>>(y_idx, y_val, ctr + 1, dist, xi[cur ^ 1], xv[cur ^ 1], ctr);
        ++h->kernel_launches;
        if (cudaMemcpyAsync(h->sssp_host, ctr, sizeof(int32_t), cudaMemcpyDeviceToHost, st) != cudaSuccess ||
            cudaMemsetAsync(ctr, 0, sizeof(int32_t), st) != cudaSuccess || cudaStreamSynchronize(st) != cudaSuccess) {
            status = DBSPMSPV_ERR_CUDA;
            break;
        }
        nnz_x = h->sssp_host[0];
        cur ^= 1;
    }
    if (status != DBSPMSPV_OK) return status;
    if (n_steps) *n_steps = steps;
    return DBSPMSPV_OK;
}

}  // namespace dbs

extern "C" {

void dbspmspv_default_run_opts(dbspmspv_run_opts *o) {
    if (!o) return;
    *o = dbspmspv_run_opts();
    o->th3 = 0.95f;
    o->th3_bfs = 0.05f;
    o->th3_decode = 0.01f;
    o->bfs_push_max_edge_frac = 0.08f;
    o->force_path = DBSPMSPV_PATH_AUTO;
    o->popc_threshold = 8;
    o->validate = 0;
}

int dbspmspv_set_run_opts(dbspmspv_handle_t h, const dbspmspv_run_opts *opts) {
    if (!h || !opts) return DBSPMSPV_ERR_INVALID_ARG;
    if (opts->force_path < DBSPMSPV_PATH_AUTO || opts->force_path > DBSPMSPV_PATH_PULL) return DBSPMSPV_ERR_INVALID_ARG;
    if (!(opts->th3 >= 0.f) || !(opts->th3_bfs >= 0.f) || !(opts->th3_decode >= 0.f) || !(opts->bfs_push_max_edge_frac >= 0.f) ||
        !(opts->decode_threshold >= 0.f)) return DBSPMSPV_ERR_INVALID_ARG;
    h->ropts = *opts;
    return DBSPMSPV_OK;
}

static int run_checked(dbspmspv_handle_t h, const int32_t *x_idx, const void *x_val, int32_t nnz_x,
                       int semiring, int32_t *y_idx, float *y_val, int64_t y_capacity, int32_t *y_nnz,
                       dbspmspv_stream_t stream, const uint32_t *row_mask, int complement) {
    if (!h || nnz_x < 0 || y_capacity < 0 || !y_nnz) return DBSPMSPV_ERR_INVALID_ARG;
    if (nnz_x > 0 && !x_idx) return DBSPMSPV_ERR_INVALID_ARG;
    if (y_capacity > 0 && !y_idx) return DBSPMSPV_ERR_INVALID_ARG;
    if (semiring != DBSPMSPV_PLUS_TIMES && semiring != DBSPMSPV_OR_AND && semiring != DBSPMSPV_MIN_PLUS) return DBSPMSPV_ERR_INVALID_ARG;
    if (semiring == DBSPMSPV_PLUS_TIMES && h->d.dtype == DBSPMSPV_PATTERN) return DBSPMSPV_ERR_UNSUPPORTED;
    if (semiring != DBSPMSPV_OR_AND && ((nnz_x > 0 && !x_val) || (y_capacity > 0 && !y_val))) return DBSPMSPV_ERR_INVALID_ARG;
    if ((int64_t)nnz_x > h->d.n) return DBSPMSPV_ERR_INVALID_ARG;
    if (!dbs::on_handle_device(h)) return DBSPMSPV_ERR_INVALID_ARG;
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    h->last_stream = st;
    switch (h->d.dtype) {
        case DBSPMSPV_F32: return dbs::run_typed<DBSPMSPV_F32>(h, x_idx, x_val, nnz_x, semiring, y_idx, y_val, y_capacity, y_nnz, st, row_mask, complement);
        case DBSPMSPV_BF16: return dbs::run_typed<DBSPMSPV_BF16>(h, x_idx, x_val, nnz_x, semiring, y_idx, y_val, y_capacity, y_nnz, st, row_mask, complement);
        default: return dbs::run_typed<DBSPMSPV_PATTERN>(h, x_idx, x_val, nnz_x, semiring, y_idx, y_val, y_capacity, y_nnz, st, row_mask, complement);
    }
}

int dbspmspv_run(dbspmspv_handle_t h, const int32_t *x_idx, const void *x_val, int32_t nnz_x,
                 int semiring, int32_t *y_idx, float *y_val, int64_t y_capacity, int32_t *y_nnz,
                 dbspmspv_stream_t stream) {
    return run_checked(h, x_idx, x_val, nnz_x, semiring, y_idx, y_val, y_capacity, y_nnz, stream, nullptr, 0);
}

int dbspmspv_run_masked(dbspmspv_handle_t h, const int32_t *x_idx, const void *x_val, int32_t nnz_x,
                        int semiring, const uint32_t *row_mask, int complement, int32_t *y_idx, float *y_val,
                        int64_t y_capacity, int32_t *y_nnz, dbspmspv_stream_t stream) {
    if (!row_mask || (complement != 0 && complement != 1)) return DBSPMSPV_ERR_INVALID_ARG;
    return run_checked(h, x_idx, x_val, nnz_x, semiring, y_idx, y_val, y_capacity, y_nnz, stream, row_mask, complement);
}

int db_sssp(dbspmspv_handle_t h, int32_t src, float *dist, int32_t *n_steps, dbspmspv_stream_t stream) {
    if (!h || !dist) return DBSPMSPV_ERR_INVALID_ARG;
    if (h->d.m != h->d.n) return DBSPMSPV_ERR_UNSUPPORTED;
    if (h->d.dtype == DBSPMSPV_BF16) return DBSPMSPV_ERR_UNSUPPORTED;    // distances are fp32; x would have to be bf16
    if (src < 0 || src >= h->d.n) return DBSPMSPV_ERR_INVALID_ARG;
    if (!dbs::on_handle_device(h)) return DBSPMSPV_ERR_INVALID_ARG;
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    h->last_stream = st;
    return h->d.dtype == DBSPMSPV_F32 ? dbs::sssp_typed<DBSPMSPV_F32>(h, src, dist, n_steps, st)
                                      : dbs::sssp_typed<DBSPMSPV_PATTERN>(h, src, dist, n_steps, st);
}

int dbspmspv_test_bounded_wait(dbspmspv_handle_t h, int32_t max_tries, dbspmspv_stream_t stream) {
    if (!h || max_tries < 1 || max_tries > 4096) return DBSPMSPV_ERR_INVALID_ARG;
    if (!dbs::on_handle_device(h)) return DBSPMSPV_ERR_INVALID_ARG;
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    h->last_stream = st;
    dbs::k_wait_probe<<<1, 32, 0, st>>>(h->d, max_tries);
    ++h->kernel_launches;
    DBS_CUDA(cudaGetLastError());
    return DBSPMSPV_OK;
}

int dbspmspv_decode_batch(dbspmspv_handle_t h, const void *x, int64_t ldx, float *y, int64_t ldy, int32_t batch,
                          dbspmspv_stream_t stream) {
    if (!h || !x || !y || batch < 1 || ldx < h->d.n || ldy < h->d.m) return DBSPMSPV_ERR_INVALID_ARG;
    if (!dbs::on_handle_device(h)) return DBSPMSPV_ERR_INVALID_ARG;
    if (h->d.dtype == DBSPMSPV_PATTERN) return DBSPMSPV_ERR_UNSUPPORTED;
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    h->last_stream = st;
    return h->d.dtype == DBSPMSPV_F32 ? dbs::decode_batch_typed<DBSPMSPV_F32>(h, x, ldx, y, ldy, batch, st)
                                      : dbs::decode_batch_typed<DBSPMSPV_BF16>(h, x, ldx, y, ldy, batch, st);
}

int dbspmspv_test_corrupt_entry(dbspmspv_handle_t h, int32_t position, uint32_t block_index) {
#ifdef DBS_BOUNDS_CHECK
    if (!h || position < 0 || position >= h->d.n_entries || block_index > dbs::IDX_MASK) return DBSPMSPV_ERR_INVALID_ARG;
    if (!dbs::on_handle_device(h)) return DBSPMSPV_ERR_INVALID_ARG;
    uint32_t v = 0;
    DBS_CUDA(cudaMemcpy(&v, h->d.csr.idx + position, 4, cudaMemcpyDeviceToHost));
    v = (v & ~dbs::IDX_MASK) | block_index;
    DBS_CUDA(cudaMemcpy(h->d.csr.idx + position, &v, 4, cudaMemcpyHostToDevice));
    return DBSPMSPV_OK;
#else
    (void)h; (void)position; (void)block_index;
    return DBSPMSPV_ERR_UNSUPPORTED;
#endif
}

int dbspmspv_decode(dbspmspv_handle_t h, const void *x, float *y, dbspmspv_stream_t stream) {
    if (!h || !x || !y) return DBSPMSPV_ERR_INVALID_ARG;
    if (!dbs::on_handle_device(h)) return DBSPMSPV_ERR_INVALID_ARG;
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    h->last_stream = st;
    switch (h->d.dtype) {
        case DBSPMSPV_F32: return dbs::decode_typed<DBSPMSPV_F32>(h, x, y, st);
        case DBSPMSPV_BF16: return dbs::decode_typed<DBSPMSPV_BF16>(h, x, y, st);
        default: return DBSPMSPV_ERR_UNSUPPORTED;
    }
}

}  // extern "C"

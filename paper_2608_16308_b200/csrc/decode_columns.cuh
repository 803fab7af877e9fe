// Decode over columns (Section 4.3: one layer, one token or a few) for bf16 layers that are pruned, but
// not to a small fraction: y = W x as a sum over the columns that x reaches.
//
// What such a call cannot do without is the surviving weights of the active columns; the block
// payload holds them in pieces of 15 - 32 bytes behind 48-byte headers, so that a call either read
// everything (12288 x 4096 pruned by half: 84 MB whatever x holds, 27 us) or fetched the pieces in chains of dependent loads.  Here the
// weights lie once more, column by column: strips of DC_ROWS = 32 rows, [strip][column][row], 64 contiguous
// bytes per column and strip, absent elements as DC_ABSENT (a -0.0 that no stored weight uses: a
// stored -0 is kept as +0, which gives the same products up to the sign of a zero).  A call then reads the
// active columns only, every lane 16 bytes at a time, all loads independent of each other, and the arithmetic is one shift
// or mask and one FMA per weight: what bounds it is HBM (active share x 2 bytes per weight) plus about 5 us of
// launch, blocking of x and reduction.  The copy costs 2 bytes per matrix entry; it is built where that is at most DC_MAX_RATIO times the payload
// (up to about 80 % pruned) and where the matrix has the rows to fill the GPU with strips.
//
//   * A thread block owns a strip (a cluster of C blocks where the matrix has too few strips: each
//     takes every C-th vector block of x, the sums meet in the first block's shared memory), so y
//     needs neither zeroing nor atomics.
//   * x is blocked by every thread block for itself (a few KB, from L2): the entries that take part become a list of
//     (column, value) in shared memory.
//   * Several vectors (k_decode_cols_batch) share one pass over the union of their columns on the tensor cores: D[vector][row] += X[vector][k] W[k][row],
//     16 columns per mma.sync m16n8k16, the W fragments straight from global memory -- a lane loads four rows of the four columns its fragment
//     holds and pairs the columns with byte permutes, no shared memory and no expansion in between.
//   * A non-finite x entry may only meet stored elements: such calls (checked while x is blocked) take a plain loop that tests every element.
#pragma once

#include <cooperative_groups.h>

namespace dbs {

constexpr int DC_SLOW_FLAG = 1 << 30;

// x entry j of vector `b` as the products see it
__device__ __forceinline__ float dc_x(const Device &d, const void *x, int64_t ldx, int b, int64_t j) {
    if (d.decode_x_f32) return __bfloat162float(__float2bfloat16_rn(static_cast<const float *>(x)[b * ldx + j]));
    return __bfloat162float(static_cast<const __nv_bfloat16 *>(x)[b * ldx + j]);
}
// eight consecutive entries j0 .. j0 + 7 (j0 a multiple of 8; entries past n are 0 and never take part)
__device__ __forceinline__ void dc_load8(const Device &d, const void *x, int64_t ldx, int b, int64_t j0, bool aligned, float (&v)[8]) {
    if (aligned && j0 + 8 <= d.n) {
        if (d.decode_x_f32) {
            const float4 *p = reinterpret_cast<const float4 *>(static_cast<const float *>(x) + b * ldx + j0);
            const float4 f = p[0], g = p[1];
            const float w[8] = {f.x, f.y, f.z, f.w, g.x, g.y, g.z, g.w};
#pragma unroll
            for (int k = 0; k < 8; ++k) v[k] = __bfloat162float(__float2bfloat16_rn(w[k]));
        } else {
            const uint4 u = *reinterpret_cast<const uint4 *>(static_cast<const uint16_t *>(x) + b * ldx + j0);
            const uint32_t w[4] = {u.x, u.y, u.z, u.w};
#pragma unroll
            for (int k = 0; k < 4; ++k) { v[2 * k] = __uint_as_float(w[k] << 16); v[2 * k + 1] = __uint_as_float(w[k] & 0xFFFF0000u); }
        }
        return;
    }
#pragma unroll
    for (int k = 0; k < 8; ++k) v[k] = j0 + k < d.n ? dc_x(d, x, ldx, b, j0 + k) : 0.f;
}
__device__ __forceinline__ bool dc_finite(float v) { return (__float_as_uint(v) & 0x7F800000u) != 0x7F800000u; }

// The calls with a non-finite x entry: lane = row, a column at a time, every element tested.
template <int NV>
__device__ __forceinline__ void dc_slow(const Device &d, const void *x, int64_t ldx, int nvec, int strip, int warp, int step, int lane, float (&acc)[NV]) {
    const uint16_t *w = reinterpret_cast<const uint16_t *>(d.cols) + (size_t)strip * d.n * DC_ROWS + lane;
#pragma unroll
    for (int b = 0; b < NV; ++b) acc[b] = 0.f;
    for (int64_t j = warp; j < d.n; j += step) {
        const uint32_t u = w[j * DC_ROWS];
#pragma unroll
        for (int b = 0; b < NV; ++b) {
            if (b >= nvec) break;
            const float v = dc_x(d, x, ldx, b, j);
            if (u != DC_ABSENT && decode_takes_part(d, v)) acc[b] += __uint_as_float(u << 16) * v;
        }
    }
}

// What the first thread of a call writes down about it.
__device__ __forceinline__ void dc_record(const Device &d, int n_nzblk, float th3, int force_path) {
    Counters *c = d.ws.ctr;
    c->last_n_nzblk = n_nzblk;
    c->last_n_tasks = 0;
    c->last_path = force_path == DBSPMSPV_PATH_PUSH || force_path == DBSPMSPV_PATH_PULL ? force_path
                 : (float)n_nzblk / (float)d.nb < th3 ? DBSPMSPV_PATH_PUSH : DBSPMSPV_PATH_PULL;
    c->last_y_nnz = (int32_t)d.m;
}

constexpr int DC_WARPS = 8;
constexpr int DC_CTA = DC_WARPS * 32;
constexpr int DC_ILP = 8;            // 16-byte loads in flight per lane: 4 KB per warp

// One vector.  Lane (q, p) = (lane / 4, lane % 4): rows 8 p .. 8 p + 7 of the strip, every eighth column of the list.
template <int C>
__global__ void __cluster_dims__(C, 1, 1) __launch_bounds__(DC_CTA)
k_decode_cols(Device d, const void *__restrict__ x, float *__restrict__ y, float th3, int force_path) {
    namespace cg = cooperative_groups;
    extern __shared__ __align__(16) uint8_t s_dyn[];
    float2 *s_list = reinterpret_cast<float2 *>(s_dyn);              // (column bits, value)
    __shared__ float s_part[DC_WARPS][DC_ROWS], s_sum[C][DC_ROWS];
    __shared__ int s_n, s_nz, s_seen[C];                             // entries; nonzero vector blocks; those of every rank, plus DC_SLOW_FLAG if it met a non-finite entry
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int rank = C > 1 ? (int)cg::this_cluster().block_rank() : 0, strip = blockIdx.x / C;
    if (tid == 0) { s_n = 0; s_nz = 0; }
    pdl_wait();
    if (C > 1) cg::this_cluster().sync(); else __syncthreads();       // (a cluster: every block has started before its shared memory is written)
    bool odd = false;                                                 // some entry is not finite
    // ---- the list of the entries that take part: eight consecutive ones per thread and round, this rank's vector blocks only
    {
        const bool aligned = (reinterpret_cast<uintptr_t>(x) & 15u) == 0;
        const int units = (d.nb - rank + C - 1) / C * 2;             // halves of this rank's vector blocks
        int nz = 0;
        for (int u0 = warp * 32; u0 < units; u0 += DC_CTA) {
            const int u = u0 + lane;
            const int64_t j0 = ((int64_t)(u >> 1) * C + rank) * 16 + (u & 1) * 8;
            float v[8];
            uint32_t bits = 0;
            if (u < units) {
                dc_load8(d, x, 0, 0, j0, aligned, v);
#pragma unroll
                for (int k = 0; k < 8; ++k) { bits |= (j0 + k < d.n && decode_takes_part(d, v[k]) ? 1u : 0u) << k; }
            }
            const int cnt = __popc(bits);
            int incl = cnt;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) { const int t = __shfl_up_sync(FULL, incl, o); if (lane >= o) incl += t; }
            int base = 0;
            if (lane == 31 && incl) base = atomicAdd(&s_n, incl);
            int at = __shfl_sync(FULL, base, 31) + incl - cnt;
#pragma unroll
            for (int k = 0; k < 8; ++k)
                if ((bits >> k) & 1u) { s_list[at++] = make_float2(__int_as_float((int)j0 + k), v[k]); odd |= !dc_finite(v[k]); }
            nz += __popc(__ballot_sync(FULL, bits | __shfl_xor_sync(FULL, bits, 1)) & 0x55555555u);
        }
        if (lane == 0 && nz) atomicAdd(&s_nz, nz);
        odd = __syncthreads_or(odd);
        if (C > 1) {
            // (every rank has to know whether any met a non-finite entry)
            cg::cluster_group cluster = cg::this_cluster();
            if (tid < C) cluster.map_shared_rank(s_seen, tid)[rank] = s_nz | (odd ? DC_SLOW_FLAG : 0);
            cluster.sync();
#pragma unroll
            for (int r = 0; r < C; ++r) odd |= (s_seen[r] & DC_SLOW_FLAG) != 0;
        } else if (tid == 0) {
            s_seen[0] = s_nz;
        }
        if (strip == 0 && rank == 0 && tid == 0) {
            int total = 0;
#pragma unroll
            for (int r = 0; r < C; ++r) total += s_seen[r] & (DC_SLOW_FLAG - 1);
            dc_record(d, total, th3, force_path);
        }
        if (odd) {
            float a[1];
            dc_slow<1>(d, x, 0, 1, strip, warp * C + rank, DC_WARPS * C, lane, a);
            s_part[warp][lane] = a[0];
        } else s_part[warp][lane] = 0.f;
    }
    __syncthreads();
    const int n = odd ? 0 : s_n;
    if (n > 0) {                                                      // block-uniform
        const uint4 *w = d.cols + (size_t)strip * d.n * (DC_ROWS / 8) + (lane & 3);
        float acc[8];
#pragma unroll
        for (int r = 0; r < 8; ++r) acc[r] = 0.f;
        for (int k0 = warp * 8 + (lane >> 2); k0 - (lane >> 2) < n; k0 += DC_WARPS * 8 * DC_ILP) {
            uint4 v[DC_ILP];
            float xv[DC_ILP];
#pragma unroll
            for (int u = 0; u < DC_ILP; ++u) {
                const int k = k0 + u * DC_WARPS * 8;
                v[u] = make_uint4(0u, 0u, 0u, 0u);
                xv[u] = 0.f;
                if (k < n) { const float2 e = s_list[k]; xv[u] = e.y; v[u] = __ldcs(w + (size_t)__float_as_int(e.x) * (DC_ROWS / 8)); }
            }
#pragma unroll
            for (int u = 0; u < DC_ILP; ++u) {
                const uint32_t q[4] = {v[u].x, v[u].y, v[u].z, v[u].w};
#pragma unroll
                for (int r = 0; r < 4; ++r) {
                    acc[2 * r] += __uint_as_float(q[r] << 16) * xv[u];
                    acc[2 * r + 1] += __uint_as_float(q[r] & 0xFFFF0000u) * xv[u];
                }
            }
        }
        // sums over the eight column slots of the warp: three halving exchanges leave one row per lane
        const bool h16 = lane & 16, h8 = lane & 8, h4 = lane & 4;
        float a4[4], a2[2];
#pragma unroll
        for (int i = 0; i < 4; ++i) a4[i] = (h16 ? acc[i + 4] : acc[i]) + __shfl_xor_sync(FULL, h16 ? acc[i] : acc[i + 4], 16);
#pragma unroll
        for (int i = 0; i < 2; ++i) a2[i] = (h8 ? a4[i + 2] : a4[i]) + __shfl_xor_sync(FULL, h8 ? a4[i] : a4[i + 2], 8);
        const float a1 = (h4 ? a2[1] : a2[0]) + __shfl_xor_sync(FULL, h4 ? a2[0] : a2[1], 4);
        s_part[warp][(lane & 3) * 8 + (h16 ? 4 : 0) + (h8 ? 2 : 0) + (h4 ? 1 : 0)] = a1;
    }
    __syncthreads();
    float sum = 0.f;
    if (tid < DC_ROWS) {
#pragma unroll
        for (int k = 0; k < DC_WARPS; ++k) sum += s_part[k][tid];
    }
    if (C > 1) {
        cg::cluster_group cluster = cg::this_cluster();
        if (tid < DC_ROWS) cluster.map_shared_rank(&s_sum[0][0], 0)[rank * DC_ROWS + tid] = sum;
        cluster.sync();
        if (rank == 0 && tid < DC_ROWS) {
            sum = 0.f;
#pragma unroll
            for (int r = 0; r < C; ++r) sum += s_sum[r][tid];
        }
    }
    const int64_t row = (int64_t)strip * DC_ROWS + tid;
    if (rank == 0 && tid < DC_ROWS && row < d.m) y[row] = sum;
}

constexpr int DCB_WARPS = 16;
constexpr int DCB_CTA = DCB_WARPS * 32;
constexpr int DCB_ILP = 2;           // steps of 16 columns in flight per warp: 2 KB
static_assert(DCB_WARPS * 32 >= 8 * DC_ROWS, "a thread per vector and row");

// Shared memory of a batched call: values by pairs of list entries, [pair][vector][2] bf16; columns; partial sums.
struct DcBatchLayout {
    int cap, col_off, red_off, total;
    __host__ __device__ DcBatchLayout(int nb, int nv, int c) {
        cap = (nb + c - 1) / c * 16 + 16;                             // entries of a rank, padded to whole steps
        col_off = cap * nv * 2;
        red_off = (col_off + cap * 2 + 15) & ~15;
        total = red_off + DCB_WARPS / 2 * nv * DC_ROWS * 4;
    }
};

static_assert(DC_MAX_COLUMNS < 65536, "16-bit columns");
// its static shared memory (the sums of the ranks, a few words), rounded up
__host__ __device__ constexpr int dcb_static(int nv, int c) { return (c > 1 ? c : 1) * nv * DC_ROWS * 4 + 256; }

// Up to NV vectors.  Fragment lane (g, t) = (lane / 4, lane % 4) of a step: rows 4 g .. 4 g + 3 of columns 2 t, 2 t + 1, 2 t + 8, 2 t + 9.  N tile i
// holds the rows 4 g' + i, g' = 0 .. 7, so that a lane's four rows of a column are its elements of the four tiles.
template <int NV, int C>
__global__ void __cluster_dims__(C, 1, 1) __launch_bounds__(DCB_CTA, 2)
k_decode_cols_batch(Device d, const void *__restrict__ x, int64_t ldx, float *__restrict__ y, int64_t ldy, int nvec, float th3, int force_path) {
    namespace cg = cooperative_groups;
    extern __shared__ __align__(16) uint8_t s_dyn[];
    const DcBatchLayout lay(d.nb, NV, C);
    uint16_t *s_x = reinterpret_cast<uint16_t *>(s_dyn);
    uint16_t *s_col = reinterpret_cast<uint16_t *>(s_dyn + lay.col_off);
    float *s_red = reinterpret_cast<float *>(s_dyn + lay.red_off);
    __shared__ float s_sum[C > 1 ? C : 1][NV * DC_ROWS];
    __shared__ int s_n, s_nz, s_seen[C];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int rank = C > 1 ? (int)cg::this_cluster().block_rank() : 0;
    if (tid == 0) { s_n = 0; s_nz = 0; }
    pdl_wait();
    if (C > 1) cg::this_cluster().sync(); else __syncthreads();
    bool odd = false;
    {
        const bool aligned = (reinterpret_cast<uintptr_t>(x) & 15u) == 0 && (ldx & 7) == 0;
        const int units = (d.nb - rank + C - 1) / C * 2;
        int nz = 0;
        for (int u0 = warp * 32; u0 < units; u0 += DCB_CTA) {
            const int u = u0 + lane;
            const int64_t j0 = ((int64_t)(u >> 1) * C + rank) * 16 + (u & 1) * 8;
            uint32_t h[NV][4];                                        // the entries as bf16 pairs, 0 where one does not take part
            uint32_t bits = 0;
#pragma unroll
            for (int b = 0; b < NV; ++b) {
                h[b][0] = h[b][1] = h[b][2] = h[b][3] = 0u;
                if (u < units && b < nvec) {
                    float v[8];
                    dc_load8(d, x, ldx, b, j0, aligned, v);
#pragma unroll
                    for (int k = 0; k < 8; ++k) {
                        const bool in = j0 + k < d.n && decode_takes_part(d, v[k]);
                        odd |= in && !dc_finite(v[k]);
                        bits |= (in ? 1u : 0u) << k;
                        if (in) h[b][k >> 1] |= (__float_as_uint(v[k]) >> 16) << (16 * (k & 1));
                    }
                }
            }
            const int cnt = __popc(bits);
            int incl = cnt;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) { const int t = __shfl_up_sync(FULL, incl, o); if (lane >= o) incl += t; }
            int base = 0;
            if (lane == 31 && incl) base = atomicAdd(&s_n, incl);
            int at = __shfl_sync(FULL, base, 31) + incl - cnt;
#pragma unroll
            for (int k = 0; k < 8; ++k) {
                if (!((bits >> k) & 1u)) continue;
                s_col[at] = (uint16_t)(j0 + k);
#pragma unroll
                for (int b = 0; b < NV; ++b) s_x[((at >> 1) * NV + b) * 2 + (at & 1)] = (uint16_t)(h[b][k >> 1] >> (16 * (k & 1)));
                ++at;
            }
            nz += __popc(__ballot_sync(FULL, bits | __shfl_xor_sync(FULL, bits, 1)) & 0x55555555u);
        }
        if (lane == 0 && nz) atomicAdd(&s_nz, nz);
        odd = __syncthreads_or(odd);
        if (C > 1) {
            cg::cluster_group cluster = cg::this_cluster();
            if (tid < C) cluster.map_shared_rank(s_seen, tid)[rank] = s_nz | (odd ? DC_SLOW_FLAG : 0);
            cluster.sync();
#pragma unroll
            for (int r = 0; r < C; ++r) odd |= (s_seen[r] & DC_SLOW_FLAG) != 0;
        } else if (tid == 0) {
            s_seen[0] = s_nz;
        }
        if (blockIdx.x == 0 && tid == 0) {
            int total = 0;
#pragma unroll
            for (int r = 0; r < C; ++r) total += s_seen[r] & (DC_SLOW_FLAG - 1);
            dc_record(d, total, th3, force_path);
        }
    }
    const int n = s_n, n_steps = (n + 15) >> 4;
    if (tid < 16 && n + tid < n_steps * 16) {                         // the last step is filled up with column 0 times 0
        const int at = n + tid;
        s_col[at] = 0;
        for (int b = 0; b < NV; ++b) s_x[((at >> 1) * NV + b) * 2 + (at & 1)] = 0;
    }
    __syncthreads();
    const int g = lane >> 2, t = lane & 3;
    const uint32_t *xw = reinterpret_cast<const uint32_t *>(s_x);
    for (int strip = blockIdx.x / C; strip * DC_ROWS < d.m; strip += gridDim.x / C) {
        float acc[4][4];
#pragma unroll
        for (int i = 0; i < 4; ++i) acc[i][0] = acc[i][1] = acc[i][2] = acc[i][3] = 0.f;
        const uint2 *w = reinterpret_cast<const uint2 *>(d.cols) + (size_t)strip * d.n * (DC_ROWS / 4) + g;
        for (int s0 = odd ? n_steps : warp; s0 < n_steps; s0 += DCB_WARPS * DCB_ILP) {
            uint2 v[DCB_ILP][4];
#pragma unroll
            for (int u = 0; u < DCB_ILP; ++u) {
                const int s = s0 + u * DCB_WARPS;
                if (s < n_steps) {                                    // warp-uniform
                    const uint32_t lo = *reinterpret_cast<const uint32_t *>(s_col + s * 16 + 2 * t), hi = *reinterpret_cast<const uint32_t *>(s_col + s * 16 + 8 + 2 * t);
                    v[u][0] = __ldcs(w + (size_t)(lo & 0xFFFFu) * (DC_ROWS / 4));
                    v[u][1] = __ldcs(w + (size_t)(lo >> 16) * (DC_ROWS / 4));
                    v[u][2] = __ldcs(w + (size_t)(hi & 0xFFFFu) * (DC_ROWS / 4));
                    v[u][3] = __ldcs(w + (size_t)(hi >> 16) * (DC_ROWS / 4));
                }
            }
#pragma unroll
            for (int u = 0; u < DCB_ILP; ++u) {
                const int s = s0 + u * DCB_WARPS;
                if (s >= n_steps) break;
                const uint32_t a0 = g < NV ? xw[(s * 8 + t) * NV + g] : 0u, a2 = g < NV ? xw[(s * 8 + t + 4) * NV + g] : 0u;
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    const uint32_t sel = i & 1 ? 0x7632u : 0x5410u;
                    const uint32_t b0 = __byte_perm(i < 2 ? v[u][0].x : v[u][0].y, i < 2 ? v[u][1].x : v[u][1].y, sel);
                    const uint32_t b1 = __byte_perm(i < 2 ? v[u][2].x : v[u][2].y, i < 2 ? v[u][3].x : v[u][3].y, sel);
                    mma_bf16_m16n8k16(acc[i], a0, 0u, a2, 0u, b0, b1);
                }
            }
        }
        // sums over the warps: the upper half hands its sums to the lower half, then a thread per (vector, row) adds up.
        // acc[i][0], acc[i][1]: vector g, rows 8 t + i and 8 t + 4 + i
        float *red = s_red + (warp % (DCB_WARPS / 2)) * NV * DC_ROWS;
        if (odd) {
            float a[NV];
            dc_slow<NV>(d, x, ldx, nvec, strip, warp * C + rank, DCB_WARPS * C, lane, a);
            if (warp >= DCB_WARPS / 2)
#pragma unroll
                for (int b = 0; b < NV; ++b) red[b * DC_ROWS + lane] = a[b];
            __syncthreads();
            if (warp < DCB_WARPS / 2)
#pragma unroll
                for (int b = 0; b < NV; ++b) red[b * DC_ROWS + lane] += a[b];
        } else {
            if (warp >= DCB_WARPS / 2 && g < NV)
#pragma unroll
                for (int i = 0; i < 4; ++i) { red[g * DC_ROWS + 8 * t + i] = acc[i][0]; red[g * DC_ROWS + 8 * t + 4 + i] = acc[i][1]; }
            __syncthreads();
            if (warp < DCB_WARPS / 2 && g < NV)
#pragma unroll
                for (int i = 0; i < 4; ++i) { red[g * DC_ROWS + 8 * t + i] += acc[i][0]; red[g * DC_ROWS + 8 * t + 4 + i] += acc[i][1]; }
        }
        __syncthreads();
        float sum = 0.f;
        if (tid < NV * DC_ROWS) {
#pragma unroll
            for (int k = 0; k < DCB_WARPS / 2; ++k) sum += s_red[k * NV * DC_ROWS + tid];
        }
        if (C > 1) {
            cg::cluster_group cluster = cg::this_cluster();
            if (tid < NV * DC_ROWS) cluster.map_shared_rank(&s_sum[0][0], 0)[rank * NV * DC_ROWS + tid] = sum;
            cluster.sync();
            if (rank == 0 && tid < NV * DC_ROWS) {
                sum = 0.f;
#pragma unroll
                for (int r = 0; r < C; ++r) sum += s_sum[C > 1 ? r : 0][tid];
            }
            cluster.sync();                                           // (the next strip overwrites the sums)
        }
        const int b = tid / DC_ROWS;
        const int64_t row = (int64_t)strip * DC_ROWS + tid % DC_ROWS;
        if (rank == 0 && b < nvec && b < NV && row < d.m) y[b * ldy + row] = sum;
        __syncthreads();
    }
}

// Thread blocks of a cluster: as many as it takes to give every SM one (one where the strips alone do).
inline int dc_cluster(int64_t m, int sm_count) {
    const int64_t strips = (m + DC_ROWS - 1) / DC_ROWS;
    int c = 1;
    while (c < 8 && strips * c * 2 <= sm_count) c *= 2;
    return c;
}

}  // namespace dbs

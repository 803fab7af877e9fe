// Decode over columns (Section 4.3: one layer, one token or a few) for bf16 layers that are pruned, but
// not to a small fraction: y = W x as a sum over the columns that x reaches.
//
// What such a call cannot do without is the surviving weights of the active columns; the block
// payload holds them in pieces of 15 - 32 bytes behind 48-byte headers, so that a call either read
// everything (12288 x 4096 pruned by half: 84 MB whatever x holds, 27 us) or fetched the pieces in chains of dependent loads.  Here the
// weights lie once more, column by column: strips of DC_ROWS = 64 rows, [strip][column][row], 128 contiguous
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
//     16 columns per mma.sync m16n8k16, the W fragments straight from global memory -- a lane loads eight rows of the four columns its fragment
//     holds and pairs the columns with byte permutes, no shared memory and no expansion in between.
//   * A non-finite x entry may only meet stored elements: what met one while x was blocked -- the warp, of a single vector; the whole call, of several -- takes a plain
//     loop that tests every element.
#pragma once

#include <cooperative_groups.h>

namespace dbs {

// x entry j of vector `b` as the products see it
__device__ __forceinline__ float dc_x(const Device &d, const void *x, int64_t ldx, int b, int64_t j) {
    if (d.decode_x_f32) return __bfloat162float(__float2bfloat16_rn(static_cast<const float *>(x)[b * ldx + j]));
    return __bfloat162float(static_cast<const __nv_bfloat16 *>(x)[b * ldx + j]);
}
// eight consecutive entries j0 .. j0 + 7 (j0 a multiple of 8) as bf16; entries past n are 0
__device__ __forceinline__ uint4 dc_load8(const Device &d, const void *x, int64_t ldx, int b, int64_t j0, bool aligned) {
    uint32_t w[4] = {0u, 0u, 0u, 0u};
    if (aligned && !d.decode_x_f32 && j0 + 8 <= d.n) return *reinterpret_cast<const uint4 *>(static_cast<const uint16_t *>(x) + b * ldx + j0);
    if (aligned && j0 + 8 <= d.n) {
        const float4 *p = reinterpret_cast<const float4 *>(static_cast<const float *>(x) + b * ldx + j0);
        const float4 f = p[0], g = p[1];
        const float v[8] = {f.x, f.y, f.z, f.w, g.x, g.y, g.z, g.w};
#pragma unroll
        for (int k = 0; k < 8; ++k) w[k >> 1] |= (__float_as_uint(__bfloat162float(__float2bfloat16_rn(v[k]))) >> 16) << (16 * (k & 1));
    } else {
#pragma unroll
        for (int k = 0; k < 8; ++k)
            if (j0 + k < d.n) w[k >> 1] |= (__float_as_uint(dc_x(d, x, ldx, b, j0 + k)) >> 16) << (16 * (k & 1));
    }
    return make_uint4(w[0], w[1], w[2], w[3]);
}
__device__ __forceinline__ float dc_entry(const uint4 &u, int k) {       // entry k of eight
    const uint32_t w = k < 2 ? u.x : k < 4 ? u.y : k < 6 ? u.z : u.w;
    return __uint_as_float(k & 1 ? w & 0xFFFF0000u : w << 16);
}

// Which entries of a pair of bf16 take part (see decode_takes_part), two at a time: magnitude bits compared by a carry
// into the halfword's top bit.  |v| > tau is a comparison of magnitude bits (tau's own low half can be dropped); with the
// ReLU a negative entry takes part only if it is a NaN.
struct DcTest {
    uint32_t k, s;
    __device__ __forceinline__ explicit DcTest(const Device &d) {
        k = (0x7FFFu - (__float_as_uint(d.decode_tau) >> 16)) * 0x10001u;
        s = d.decode_relu ? 0u : 0xFFFFFFFFu;
    }
    __device__ __forceinline__ uint32_t operator()(uint32_t w) const {       // bits 15 and 31
        const uint32_t a = w & 0x7FFF7FFFu;
        return (a + k) & (~w | s | (a + 0x007F007Fu)) & 0x80008000u;
    }
};
__device__ __forceinline__ uint32_t dc_odd(uint32_t w) { return ((w & 0x7FFF7FFFu) + 0x00800080u) & 0x80008000u; }     // infinite or NaN
__device__ __forceinline__ uint32_t dc_pair_bits(uint32_t m) { return ((m >> 15) & 1u) | ((m >> 30) & 2u); }
__device__ __forceinline__ uint32_t dc_pair_mask(uint32_t m) { return ((m >> 15) & 0x00010001u) * 0xFFFFu; }

// The calls with a non-finite x entry: a lane takes the rows lane, lane + 32 of the strip, a column at a time, every element tested.
constexpr int DC_PER_LANE = DC_ROWS / 32;
template <int NV>
__device__ __forceinline__ void dc_slow(const Device &d, const void *x, int64_t ldx, int nvec, int strip, int warp, int step, int lane, float (&acc)[NV][DC_PER_LANE]) {
    const uint16_t *w = reinterpret_cast<const uint16_t *>(d.cols) + (size_t)strip * d.n * DC_ROWS + lane;
#pragma unroll
    for (int b = 0; b < NV; ++b)
#pragma unroll
        for (int h = 0; h < DC_PER_LANE; ++h) acc[b][h] = 0.f;
    for (int64_t j = warp; j < d.n; j += step) {
#pragma unroll
        for (int b = 0; b < NV; ++b) {
            if (b >= nvec) break;
            const float v = dc_x(d, x, ldx, b, j);
            if (!decode_takes_part(d, v)) continue;
#pragma unroll
            for (int h = 0; h < DC_PER_LANE; ++h) {
                const uint32_t u = w[j * DC_ROWS + 32 * h];
                if (u != DC_ABSENT) acc[b][h] += __uint_as_float(u << 16) * v;
            }
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

constexpr int DC_WARPS = 16;
constexpr int DC_CTA = DC_WARPS * 32;
constexpr int DC_ILP = 8;            // 16-byte loads in flight per lane: 4 KB per warp
constexpr int DC_LANES = DC_ROWS / 8;    // lanes that share a column (eight rows each)
constexpr int DC_SLOTS = 32 / DC_LANES;  // columns of a warp's load
constexpr int DC_XILP = 2;           // groups of eight x entries a lane fetches at once
static_assert(DC_ROWS == 64, "two halving exchanges over the column slots");

// Vector blocks of x that rank `rank` of C takes; its warps take them in turn, four neighbours at a time.  Entries of a warp's list, at most.
__host__ __device__ inline int dc_blocks(int nb, int c, int rank) { return (nb - rank + c - 1) / c; }
__host__ __device__ inline int dc_warp_entries(int nb, int c) { return (dc_blocks(nb, c, 0) + 4 * DC_WARPS - 1) / (4 * DC_WARPS) * 64; }

// One vector.  A warp blocks a share of x for itself -- pieces of 64 entries spread over x, so that longer active runs meet all warps -- and goes on to the columns it
// found: nobody waits for a list of the whole thread block.  (With one, three barriers and an atomic per warp stood between x and the first weight, and clusters
// met twice more.  4096 x 11008, 10 / 50 % active: 6.4 / 12.4 -> 5.1 / 11.4 us; 2000 x 2000 4.8 -> 3.8; 12288 x 4096, 30 %: 8.1 -> 7.9.)
// Lane (q, p) = (lane / 8, lane % 8): rows 8 p .. 8 p + 7 of the strip, every fourth column of the list.
template <int C>
__global__ void __cluster_dims__(C, 1, 1) __launch_bounds__(DC_CTA, 2)
k_decode_cols(Device d, const void *__restrict__ x, float *__restrict__ y, float th3, int force_path) {
    namespace cg = cooperative_groups;
    extern __shared__ __align__(16) uint8_t s_dyn[];
    __shared__ __align__(8) float s_part[DC_WARPS][DC_ROWS];
    __shared__ float s_sum[C][DC_ROWS];
    __shared__ int s_nz[DC_WARPS], s_seen[C];                         // nonzero vector blocks of every warp; of every rank
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int rank = C > 1 ? (int)cg::this_cluster().block_rank() : 0, strip = blockIdx.x / C;
    // (a cluster: every block has started before its shared memory is written; met again behind the weights)
    if (C > 1) asm volatile("barrier.cluster.arrive.relaxed.aligned;" ::: "memory");
    pdl_wait();
    const int blocks = dc_blocks(d.nb, C, rank);
    float2 *list = reinterpret_cast<float2 *>(s_dyn) + warp * dc_warp_entries(d.nb, C);              // (column bits, value)
    bool odd = false;                                                 // some entry is not finite
    int n = 0, nz = 0;
    {
        const bool aligned = (reinterpret_cast<uintptr_t>(x) & 15u) == 0;
        const DcTest test(d);
        for (int b0 = 4 * warp; b0 < blocks; b0 += 16 * DC_WARPS * DC_XILP) {    // two lanes per vector block, eight entries each
            uint4 v[DC_XILP];
            int j0[DC_XILP];
#pragma unroll
            for (int q = 0; q < DC_XILP; ++q) {
                const int b = b0 + (q * 4 + (lane >> 3)) * 4 * DC_WARPS + ((lane >> 1) & 3);
                j0[q] = (b * C + rank) * 16 + (lane & 1) * 8;
                v[q] = make_uint4(0u, 0u, 0u, 0u);
                if (b < blocks) v[q] = dc_load8(d, x, 0, 0, j0[q], aligned);
            }
            uint32_t bits = 0;                                        // eight per load
#pragma unroll
            for (int q = 0; q < DC_XILP; ++q) {
                const uint32_t w[4] = {v[q].x, v[q].y, v[q].z, v[q].w};          // (entries past n are 0: they never take part)
#pragma unroll
                for (int k = 0; k < 4; ++k) {
                    const uint32_t m = test(w[k]);
                    bits |= dc_pair_bits(m) << (8 * q + 2 * k);
                    odd |= (m & dc_odd(w[k])) != 0u;
                }
            }
            const int cnt = __popc(bits);
            int incl = cnt;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) { const int t = __shfl_up_sync(FULL, incl, o); if (lane >= o) incl += t; }
            int at = n + incl - cnt;
            n += __shfl_sync(FULL, incl, 31);
            const uint32_t both = bits | __shfl_xor_sync(FULL, bits, 1);
#pragma unroll
            for (int q = 0; q < DC_XILP; ++q) {
#pragma unroll
                for (int k = 0; k < 8; ++k)
                    if ((bits >> (8 * q + k)) & 1u) list[at++] = make_float2(__int_as_float(j0[q] + k), dc_entry(v[q], k));
                nz += __popc(__ballot_sync(FULL, (both >> (8 * q)) & 0xFFu) & 0x55555555u);
            }
        }
        __syncwarp();
    }
    if (__any_sync(FULL, odd)) {                                      // this warp's columns, every element tested
        float a[DC_PER_LANE] = {};
        const uint16_t *w = reinterpret_cast<const uint16_t *>(d.cols) + (size_t)strip * d.n * DC_ROWS + lane;
        for (int k = 0; k < n; ++k) {
            const float2 e = list[k];
#pragma unroll
            for (int h = 0; h < DC_PER_LANE; ++h) {
                const uint32_t u = w[(size_t)__float_as_int(e.x) * DC_ROWS + 32 * h];
                if (u != DC_ABSENT) a[h] += __uint_as_float(u << 16) * e.y;
            }
        }
#pragma unroll
        for (int h = 0; h < DC_PER_LANE; ++h) s_part[warp][lane + 32 * h] = a[h];
    } else {
        const uint4 *w = d.cols + (size_t)strip * d.n * (DC_ROWS / 8) + (lane & (DC_LANES - 1));
        float acc[8];
#pragma unroll
        for (int r = 0; r < 8; ++r) acc[r] = 0.f;
        for (int k0 = 0; k0 < n; k0 += DC_SLOTS * DC_ILP) {
            uint4 v[DC_ILP];
            float xv[DC_ILP];
#pragma unroll
            for (int u = 0; u < DC_ILP; ++u) {
                const int k = k0 + u * DC_SLOTS + lane / DC_LANES;
                v[u] = make_uint4(0u, 0u, 0u, 0u);
                xv[u] = 0.f;
                if (k < n) { const float2 e = list[k]; xv[u] = e.y; v[u] = __ldcs(w + (size_t)__float_as_int(e.x) * (DC_ROWS / 8)); }
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
        // sums over the four column slots of the warp: two halving exchanges leave two rows per lane
        const bool h16 = lane & 16, h8 = lane & 8;
        float a4[4], a2[2];
#pragma unroll
        for (int i = 0; i < 4; ++i) a4[i] = (h16 ? acc[i + 4] : acc[i]) + __shfl_xor_sync(FULL, h16 ? acc[i] : acc[i + 4], 16);
#pragma unroll
        for (int i = 0; i < 2; ++i) a2[i] = (h8 ? a4[i + 2] : a4[i]) + __shfl_xor_sync(FULL, h8 ? a4[i] : a4[i + 2], 8);
        *reinterpret_cast<float2 *>(&s_part[warp][(lane & 7) * 8 + (h16 ? 4 : 0) + (h8 ? 2 : 0)]) = make_float2(a2[0], a2[1]);
    }
    if (lane == 0) s_nz[warp] = nz;
    __syncthreads();
    float sum = 0.f;
    if (tid < DC_ROWS) {
#pragma unroll
        for (int k = 0; k < DC_WARPS; ++k) sum += s_part[k][tid];
    }
    int seen = 0;
    if (tid == 0) {
#pragma unroll
        for (int k = 0; k < DC_WARPS; ++k) seen += s_nz[k];
    }
    if (C > 1) {
        cg::cluster_group cluster = cg::this_cluster();
        asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
        if (tid < DC_ROWS) cluster.map_shared_rank(&s_sum[0][0], 0)[rank * DC_ROWS + tid] = sum;
        if (tid == 0) cluster.map_shared_rank(s_seen, 0)[rank] = seen;
        cluster.sync();
        if (rank == 0 && tid < DC_ROWS) {
            sum = 0.f;
#pragma unroll
            for (int r = 0; r < C; ++r) sum += s_sum[r][tid];
        }
        if (rank == 0 && tid == 0) {
            seen = 0;
#pragma unroll
            for (int r = 0; r < C; ++r) seen += s_seen[r];
        }
    }
    const int64_t row = (int64_t)strip * DC_ROWS + tid;
    if (rank == 0 && tid < DC_ROWS && row < d.m) y[row] = sum;
    if (strip == 0 && rank == 0 && tid == 0) dc_record(d, seen, th3, force_path);
}

constexpr int DCB_WARPS = 16;
constexpr int DCB_CTA = DCB_WARPS * 32;
constexpr int DCB_ILP = 2;           // steps of 16 columns in flight per warp: 4 KB
constexpr int DCB_SLOTS = 4;         // partial sums kept in shared memory: four warps at a time add theirs
constexpr int DCB_PREFETCH = 16384;  // bytes of one prefetch into L2
constexpr int64_t DCB_PREFETCH_MIN = 32ll << 20;   // bytes of a layer from which on its pieces are prefetched
constexpr int DCB_ROUNDS = 8;        // groups of eight x entries a thread may own (a byte of its mask each)
static_assert(DCB_CTA >= 8 * DC_ROWS, "a thread per vector and row");
static_assert(DC_MAX_COLUMNS < 65536 && DC_MAX_COLUMNS <= DCB_CTA * DCB_ROUNDS * 8, "16-bit columns; every entry has an owner");

// Shared memory of a batched call: values by pairs of list entries, [pair][vector] 2 x bf16; columns; partial sums.
struct DcBatchLayout {
    int col_off, red_off, total;
    __host__ __device__ DcBatchLayout(int nb, int nv) {
        const int cap = nb * 16 + 16;
        col_off = cap * nv * 2;
        red_off = (col_off + cap * 2 + 15) & ~15;
        total = red_off + DCB_SLOTS * nv * DC_ROWS * 4;
    }
};

// Up to NV vectors, one thread block per SM; y is zeroed in front.  The work -- strips times steps of 16 columns of the
// list -- is cut into equal pieces, one per thread block, whatever strip they begin in; a piece ends in one atomic per row and vector for every strip it
// touches.  (A thread block per strip left 172 strips to 148 SMs: 42 us for 11008 x 4096 and eight vectors.)
// Every thread block builds the same list (counts and scans, no atomics).
// Fragment lane (g, t) = (lane / 4, lane % 4) of a step: rows 8 g .. 8 g + 7 of columns 2 t, 2 t + 1, 2 t + 8, 2 t + 9.  N tile i
// holds the rows 8 g' + i, g' = 0 .. 7, so that a lane's eight rows of a column are its elements of the eight tiles.
template <int NV>
__global__ void __launch_bounds__(DCB_CTA, 1)
k_decode_cols_batch(Device d, const void *__restrict__ x, int64_t ldx, float *__restrict__ y, int64_t ldy, int nvec, float th3, int force_path) {
    extern __shared__ __align__(16) uint8_t s_dyn[];
    const DcBatchLayout lay(d.nb, NV);
    uint32_t *s_x = reinterpret_cast<uint32_t *>(s_dyn);
    uint16_t *s_col = reinterpret_cast<uint16_t *>(s_dyn + lay.col_off);
    float *s_red = reinterpret_cast<float *>(s_dyn + lay.red_off);
    __shared__ int s_cnt[DCB_WARPS], s_nz[DCB_WARPS];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    // While x is staged nothing else asks for weights: the beginning of this block's piece, as it lies when most columns are reached, goes to L2 meanwhile.
    // (Large layers and three vectors or more.  Five layers in turn, so that none waits in L2, without / with it: 12288 x 4096, three vectors with 2 / 5 / 15 / 30 % active entries 12.0 / 14.4 /
    // 19.2 / 24.4 and 11.5 / 13.8 / 18.4 / 23.3 us, eight 18.0 / 21.8 / 29.1 / 27.7 and 17.6 / 21.2 / 28.2 / 27.0; 9000 x 2000, three 9.0 / 9.7 / 12.1 / 14.7 and 9.1 / 9.7 / 11.8 / 14.1.  It pays with few
    // active entries too.  3000 x 3000 no gain, 1500 x 1500 0.3 longer.)
    {
        const int64_t total = (d.m + DC_ROWS - 1) / DC_ROWS * d.n * DC_ROWS * 2, from = (int64_t)((double)total * blockIdx.x / gridDim.x) / 128 * 128 + (int64_t)tid * DCB_PREFETCH;
        if (total >= DCB_PREFETCH_MIN && nvec > 2 && tid < 8 && from + DCB_PREFETCH <= total)
            asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(reinterpret_cast<const uint8_t *>(d.cols) + from), "r"(DCB_PREFETCH) : "memory");
    }
    // (x may be read before the wait: the kernel in front zeroes y, and let this one start when everything before it had ended)
    // ---- x into shared memory: the entries that take part, by pairs of columns, and the union of the vectors' columns.
    // A warp owns consecutive groups of eight columns; the 16-byte pieces (pair, four vectors) are permuted inside their row of 32 words so that neither the
    // writes (a piece each) nor the fragment reads (four pairs, NV vectors) meet in a bank.
    constexpr int PAIRS = 32 / NV;                                     // pairs per row
    auto place = [&](int p, int b) { return p / PAIRS * 32 + (((p % PAIRS) * NV + b) ^ ((p / PAIRS & 7) << 2)); };
    auto store = [&](int p, const uint32_t (&w)[NV]) {
#pragma unroll
        for (int b = 0; b < NV; b += 4) *reinterpret_cast<uint4 *>(s_x + place(p, b)) = make_uint4(w[b], w[b + 1], w[b + 2], w[b + 3]);
    };
    // Without a cut every entry that is not zero takes part, and a zero may as well (the absent weights are zeros, too): nothing is masked.  (What bounded this phase is its instructions, five times as many
    // with the general test and a word at a time: five layers in turn, eight vectors, 11008 x 4096, 30 % active 25.3 -> 23.5 us a call, 3000 x 3000, 5 / 50 % 14.3 / 15.4 -> 12.3 / 13.4, 1024 x 12288, 5 %
    // 20.6 -> 15.0, 4096 x 11008, 30 % 32.1 -> 26.9; two vectors 20.3 -> 19.2, 8.8 / 11.9 -> 8.0 / 11.1, 12.6 -> 9.9, 24.0 -> 21.2)
    const bool plain = d.decode_tau == 0.f && !d.decode_relu;
    bool odd = false;
    uint64_t bits = 0;
    const int groups = d.nb * 2, rounds = (groups + DCB_CTA - 1) / DCB_CTA, u0 = warp * rounds * 32 + lane;
    const DcTest test(d);
    {
        const bool aligned = (reinterpret_cast<uintptr_t>(x) & 15u) == 0 && (ldx & 7) == 0;
        int nz = 0;
        for (int r = 0; r < rounds; ++r) {
            const int u = u0 + 32 * r;
            uint4 h[NV];
#pragma unroll
            for (int b = 0; b < NV; ++b) {
                h[b] = make_uint4(0u, 0u, 0u, 0u);
                if (u < groups && b < nvec) h[b] = dc_load8(d, x, ldx, b, (int64_t)u * 8, aligned);
            }
            uint32_t any[4] = {0u, 0u, 0u, 0u}, strange = 0u;
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                uint32_t w[NV];
#pragma unroll
                for (int b = 0; b < NV; ++b) w[b] = k == 0 ? h[b].x : k == 1 ? h[b].y : k == 2 ? h[b].z : h[b].w;
                if (plain) {
#pragma unroll
                    for (int b = 0; b < NV; ++b) {
                        const uint32_t a = w[b] & 0x7FFF7FFFu;
                        any[k] |= a + 0x7FFF7FFFu;                     // (bits 15 and 31)
                        strange |= a + 0x00800080u;
                    }
                    any[k] &= 0x80008000u;
                } else {
#pragma unroll
                    for (int b = 0; b < NV; ++b) {
                        const uint32_t m = test(w[b]);
                        any[k] |= m;
                        strange |= m & dc_odd(w[b]);
                        w[b] &= dc_pair_mask(m);
                    }
                }
                if (u < groups) store(u * 4 + k, w);
            }
            strange &= 0x80008000u;
            odd |= strange != 0u;
            uint32_t in = 0;
#pragma unroll
            for (int k = 0; k < 4; ++k) in |= dc_pair_bits(any[k]) << (2 * k);
            bits |= (uint64_t)in << (8 * r);
            nz += __popc(__ballot_sync(FULL, in | __shfl_xor_sync(FULL, in, 1)) & 0x55555555u);
        }
        if (lane == 31) s_nz[warp] = nz;
    }
    const int cnt = __popcll(bits);
    int incl = cnt;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) { const int t = __shfl_up_sync(FULL, incl, o); if (lane >= o) incl += t; }
    if (lane == 31) s_cnt[warp] = incl;
    odd = __syncthreads_or(odd);
    int n = 0;
#pragma unroll
    for (int k = 0; k < DCB_WARPS; ++k) n += s_cnt[k];
    if (blockIdx.x == 0 && tid == 0) {
        int nz = 0;
        for (int k = 0; k < DCB_WARPS; ++k) nz += s_nz[k];
        dc_record(d, nz, th3, force_path);
    }
    // Most columns reached: all of them are taken, as they lie.  Else the union becomes a list, and the values are staged once more, by list entry.
    const bool all = (int64_t)n * 4 >= d.n * 3;
    const int n_steps = all ? d.nb : (n + 15) >> 4, strips = (int)((d.m + DC_ROWS - 1) / DC_ROWS);
    // this block's piece; a non-finite entry: whole strips instead, element by element
    const int64_t work = (int64_t)strips * (odd ? 1 : n_steps);
    const int64_t lo = work * blockIdx.x / gridDim.x, hi = work * (blockIdx.x + 1) / gridDim.x;
    if (lo >= hi) { pdl_wait(); return; }                             // block-uniform; (no entry in any vector: nobody has a piece, and y is zeroed all the same before this kernel ends)
    if (!odd && !all) {
        int at = incl - cnt;
        for (int k = 0; k < warp; ++k) at += s_cnt[k];
        for (int r = 0; r < rounds; ++r)
            for (uint32_t m = (uint32_t)(bits >> (8 * r)) & 0xFFu; m; m &= m - 1) s_col[at++] = (uint16_t)((u0 + 32 * r) * 8 + __ffs(m) - 1);
        if (n + tid < n_steps * 16) s_col[n + tid] = 0;               // (at most 15: the last step is filled up with column 0 times 0)
        __syncthreads();
        const int first = (int)(lo % n_steps), last = (int)((hi - 1) % n_steps);
        const bool whole = hi - lo >= n_steps;
        for (int p = tid; p < n_steps * 8; p += DCB_CTA) {
            const int s = p >> 3;
            if (!whole && (first <= last ? s < first || s > last : s < first && s > last)) continue;      // (a step this block does not visit)
            // (the places behind the list hold column 0: fetched, and dropped)
            const uint32_t c2 = reinterpret_cast<const uint32_t *>(s_col)[p];
            uint32_t v[NV];
            if (d.decode_x_f32) {
                const float *xf = static_cast<const float *>(x);
                float f[NV][2];
#pragma unroll
                for (int b = 0; b < NV; ++b) { const float *row = xf + (b < nvec ? b : 0) * ldx; f[b][0] = row[c2 & 0xFFFFu]; f[b][1] = row[c2 >> 16]; }
#pragma unroll
                for (int b = 0; b < NV; ++b)
                    v[b] = (__float_as_uint(__bfloat162float(__float2bfloat16_rn(f[b][0]))) >> 16) | (__float_as_uint(__bfloat162float(__float2bfloat16_rn(f[b][1]))) & 0xFFFF0000u);
            } else {
                const uint16_t *xh = static_cast<const uint16_t *>(x);
                uint16_t f[NV][2];
#pragma unroll
                for (int b = 0; b < NV; ++b) { const uint16_t *row = xh + (b < nvec ? b : 0) * ldx; f[b][0] = row[c2 & 0xFFFFu]; f[b][1] = row[c2 >> 16]; }
#pragma unroll
                for (int b = 0; b < NV; ++b) v[b] = (uint32_t)f[b][0] | (uint32_t)f[b][1] << 16;
            }
            const uint32_t there = 2 * p + 1 < n ? 0xFFFFFFFFu : 2 * p < n ? 0xFFFFu : 0u;
#pragma unroll
            for (int b = 0; b < NV; ++b) {
                v[b] = b < nvec ? v[b] & there : 0u;
                if (!plain) v[b] &= dc_pair_mask(test(v[b]));
            }
            store(p, v);
        }
        __syncthreads();
    }
    const int g = lane >> 2, t = lane & 3;
    for (int64_t pos = lo; pos < hi;) {
        const int per = odd ? 1 : n_steps, strip = (int)(pos / per), sa = (int)(pos % per);
        const int sb = (int)(hi - pos < per - sa ? sa + (hi - pos) : per);
        float *red = s_red + (warp % DCB_SLOTS) * NV * DC_ROWS;
        if (odd) {
            float a[NV][DC_PER_LANE];
            dc_slow<NV>(d, x, ldx, nvec, strip, warp, DCB_WARPS, lane, a);
            for (int q = DCB_WARPS / DCB_SLOTS - 1; q >= 0; --q) {
                if (warp / DCB_SLOTS == q)
#pragma unroll
                    for (int k = 0; k < NV * DC_PER_LANE; ++k) red[k * 32 + lane] = a[k / DC_PER_LANE][k % DC_PER_LANE] + (q == DCB_WARPS / DCB_SLOTS - 1 ? 0.f : red[k * 32 + lane]);
                __syncthreads();
            }
        } else {
            float acc[8][4];
#pragma unroll
            for (int i = 0; i < 8; ++i) acc[i][0] = acc[i][1] = acc[i][2] = acc[i][3] = 0.f;
            const uint4 *w = d.cols + (size_t)strip * d.n * (DC_ROWS / 8) + g;
            for (int s0 = sa + warp; s0 < sb; s0 += DCB_WARPS * DCB_ILP) {
                uint4 v[DCB_ILP][4];
#pragma unroll
                for (int u = 0; u < DCB_ILP; ++u) {
                    const int s = s0 + u * DCB_WARPS;
                    if (s < sb) {                                     // warp-uniform
                        uint32_t c[4];
                        if (all) {                                    // (a column past n has no values: any address will do)
#pragma unroll
                            for (int k = 0; k < 4; ++k) c[k] = min((uint32_t)(s * 16 + 2 * t + (k & 1) + 4 * (k & 2)), (uint32_t)d.n - 1u);
                        } else {
                            const uint32_t c01 = *reinterpret_cast<const uint32_t *>(s_col + s * 16 + 2 * t), c89 = *reinterpret_cast<const uint32_t *>(s_col + s * 16 + 8 + 2 * t);
                            c[0] = c01 & 0xFFFFu; c[1] = c01 >> 16; c[2] = c89 & 0xFFFFu; c[3] = c89 >> 16;
                        }
#pragma unroll
                        for (int k = 0; k < 4; ++k) v[u][k] = __ldcs(w + (size_t)c[k] * (DC_ROWS / 8));
                    }
                }
#pragma unroll
                for (int u = 0; u < DCB_ILP; ++u) {
                    const int s = s0 + u * DCB_WARPS;
                    if (s >= sb) break;
                    uint32_t a0 = 0u, a2 = 0u;
                    if (g < NV) {
                        const int p = s * 8 + t;
                        a0 = s_x[place(p, g)];
                        a2 = s_x[place(p + 4, g)];
                    }
                    const uint32_t q[4][4] = {{v[u][0].x, v[u][0].y, v[u][0].z, v[u][0].w}, {v[u][1].x, v[u][1].y, v[u][1].z, v[u][1].w},
                                              {v[u][2].x, v[u][2].y, v[u][2].z, v[u][2].w}, {v[u][3].x, v[u][3].y, v[u][3].z, v[u][3].w}};
#pragma unroll
                    for (int i = 0; i < 8; ++i) {
                        const uint32_t sel = i & 1 ? 0x7632u : 0x5410u;
                        mma_bf16_m16n8k16(acc[i], a0, 0u, a2, 0u, __byte_perm(q[0][i >> 1], q[1][i >> 1], sel), __byte_perm(q[2][i >> 1], q[3][i >> 1], sel));
                    }
                }
            }
            // sums over the warps, four at a time.  acc[i][0], acc[i][1]: vector g, rows 16 t + i and 16 t + 8 + i
            for (int q = DCB_WARPS / DCB_SLOTS - 1; q >= 0; --q) {
                if (warp / DCB_SLOTS == q && g < NV)
#pragma unroll
                    for (int i = 0; i < 8; ++i) {
                        float *o = red + g * DC_ROWS + 16 * t + i;
                        const bool add = q != DCB_WARPS / DCB_SLOTS - 1;
                        o[0] = acc[i][0] + (add ? o[0] : 0.f);
                        o[8] = acc[i][1] + (add ? o[8] : 0.f);
                    }
                __syncthreads();
            }
        }
        pdl_wait();                                                   // (y has been zeroed)
        if (tid < nvec * DC_ROWS) {
            float sum = 0.f;
#pragma unroll
            for (int k = 0; k < DCB_SLOTS; ++k) sum += s_red[k * NV * DC_ROWS + tid];
            const int64_t row = (int64_t)strip * DC_ROWS + tid % DC_ROWS;
            if (row < d.m) atomicAdd(y + (tid / DC_ROWS) * ldy + row, sum);
        }
        __syncthreads();
        pos += sb - sa;
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

// Layers of a batch as small dense products (the batch formulation the paper leaves open in Sec. 7).
//
// The rankings of all buckets start with much the same nodes, so queries that hash alike select almost the same
// nodes and hand almost the same nodes on.  G queries with neighbouring (budget, keys) form a group; for a group
//   - the inputs at least one of its queries has nonzero, and
//   - the nodes at least one of its queries selected
// are listed once, and (inputs) x (nodes) x (G queries) is evaluated as a dense product on the FMA pipes: every
// weight is loaded and widened once for G queries, two queries' multiply-adds per instruction.  Products that no
// query asked for are dropped at the end; an input that is 0 for a query adds w * 0 to its sums, which leaves them
// as they are.  The summation order is the library's fixed one: the listed inputs are grouped by partial sum
// ((j / V) mod 32), ascending inside a group, each (query, node) partial sum is one chain of fused multiply-adds,
// and the 32 partial sums meet in the tree 16, 8, 4, 2, 1.
//
//   tile_order_kernel   queries -> groups (sorted by budget, then keys)
//   tile_prep_kernel    per group: union of inputs, staged values [entry][query], union of nodes, work items
//   tile_rows_kernel, tile_rows_wide_kernel
//                       per work item (group, 128 or 256 columns): the product, bias, ReLU, scatter to the lists
#pragma once
#include "slonn_common.cuh"

#define SLONN_TILE_G 16         // queries per group
#define SLONN_TILE_WARPS 16     // warps of tile_rows_kernel: two partial sums each
#define SLONN_TILE_NN 4         // columns per lane
#define SLONN_TILE_COLS (32 * SLONN_TILE_NN)
#define SLONN_WIDE_WARPS 8      // the same of tile_rows_wide_kernel: four partial sums each
#define SLONN_WIDE_NN 8
#define SLONN_WIDE_COLS (32 * SLONN_WIDE_NN)
#define SLONN_TILE_CHUNK 8192u  // most queries sorted and staged at a time
#define SLONN_TILE_MAX_N 32768u // widest layer: the group's G node bitmaps are built in shared memory
#define SLONN_TILE_TAKEN 4      // place of the counts of taken items behind those of items
#define SLONN_TILE_WORK 6u      // words of counts
#define SLONN_TILE_SLACK 64u    // entries past a group's list that a pipelined load may touch

// Position of partial sum p in the entry order, and back.  Four in a row are those of a warp of eight, in bit-reversed order
// (w, w + 16, w + 8, w + 24), so that the operands of an addition of the tree follow each other; a warp of sixteen has two of them.
__host__ __device__ __forceinline__ uint32_t tile_slot(uint32_t p) { return (p & 7u) * 4u + ((p >> 4) | ((p >> 2) & 2u)); }
__host__ __device__ __forceinline__ uint32_t tile_partial(uint32_t slot) { return (slot >> 2) + ((slot & 1u) << 4) + ((slot & 2u) << 2); }

// ---------------------------------------------------------------------------
// groups: queries in the order of (budget, keys)
// ---------------------------------------------------------------------------
struct slonn_order_params {
    const uint64_t *key;     // [n] sort key of each query (all different)
    const uint16_t *budget_bp;
    uint32_t bp_lo;          // queries with a smaller budget are left out
    uint32_t skip_full;      // 1: and those at exactly 10000 bp
    uint32_t q0, n;          // queries [q0, q0 + n), n <= SLONN_TILE_CHUNK
    uint32_t *order;         // out: the first entries; the rest keep the 0xffffffff (no query) they were set to
    uint32_t *work;          // [SLONN_TILE_WORK] cleared for the tile_prep_kernel that follows
};

// Rank by counting: a query's place is the number of smaller keys of its chunk.  n^2 compares (17 M for 4096
// queries) spread over the GPU, less than the launches of a radix sort.  A warp ranks four queries.  What bounds it is the
// latency of the two rounds of loads in front of the compares: all of a round's are issued at once (4096 queries: one
// after another, each key behind its budget, 15.8 us; at once 9.7 us).
__global__ void __launch_bounds__(256) tile_order_kernel(slonn_order_params P)
{
    slonn_enter();
    __shared__ uint64_t s[2048];
    const uint32_t lane = threadIdx.x & 31u, warp = threadIdx.x >> 5;
    const uint32_t e0 = (blockIdx.x * 8u + warp) * 4u;
    uint64_t mine[4];
    uint32_t rank[4] = {0u, 0u, 0u, 0u};
    if (blockIdx.x == 0 && threadIdx.x < SLONN_TILE_WORK) P.work[threadIdx.x] = 0u;
    // ~0: left out.  The key of a query that is left out may never have been written; it is loaded beside the budget all the
    // same, so that neither load waits for the other.
    auto key_of = [&](uint32_t e) -> uint64_t {
        const uint32_t q = P.q0 + min(e, P.n - 1u);
        const uint32_t bp = P.budget_bp[q];
        const uint64_t key = P.key[q];
        return e >= P.n || bp < P.bp_lo || (P.skip_full && bp == 10000u) ? ~0ull : key;
    };
    bool any = false;
#pragma unroll
    for (int k = 0; k < 4; ++k) { mine[k] = key_of(e0 + k); any |= mine[k] != ~0ull; }
    if (!__syncthreads_or(any)) return; // none of the block's queries is served
    for (uint32_t base = 0; base < P.n; base += 2048u) {
        const uint32_t m = min(2048u, P.n - base);
        __syncthreads();
        uint64_t mykey[8];
#pragma unroll
        for (int u = 0; u < 8; ++u) mykey[u] = key_of(base + threadIdx.x + u * 256u);
#pragma unroll
        for (int u = 0; u < 8; ++u) s[threadIdx.x + u * 256u] = mykey[u];
        __syncthreads();
        if (any) // uniform for the warp
            for (uint32_t i = lane; i < m; i += 32) {
                const uint64_t v = s[i];
#pragma unroll
                for (int k = 0; k < 4; ++k) rank[k] += v < mine[k] ? 1u : 0u;
            }
    }
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        const uint32_t r = __reduce_add_sync(SLONN_FULL_MASK, rank[k]);
        if (lane == 0 && mine[k] != ~0ull) P.order[r] = P.q0 + e0 + k;
    }
}

// ---------------------------------------------------------------------------
// what a layer's product needs, per group
// ---------------------------------------------------------------------------
struct slonn_tile_params {
    // queries: slot s of the chunk is order[s], or q0 + s without an order; slots past *count hold none
    const uint32_t *order;    // nullable
    const uint32_t *count;    // nullable: entries of `order` that are queries (s0 + s < *count)
    const uint16_t *skip_bp;  // nullable, only without an order: queries with this budget == 10000 are left out
    uint32_t q0, n, s0;       // first query (no order); slots of this chunk; first slot (with count)
    slonn_input in;
    uint32_t D, N, V;         // V: inputs per 16-byte weight chunk
    uint32_t kcap, wps;       // entries staged per group at most; 32-bit words per partial sum of the input bitmap
    const void *WT;
    uint32_t ldb;             // bytes per row of WT
    const uint32_t *colpos, *colnode; // nullable = identity
    const float *bias;
    uint32_t relu;
    // outputs
    uint32_t select;          // 1: the nodes listed in ids for (q, a); 0: every node
    uint32_t n_act, a;
    const uint64_t *indptr;
    uint32_t *ids;            // CSR payload (read when select; written when every node of an activator layer is computed)
    uint32_t write_ids;
    float *out_vals;          // CSR payload, nullable
    float *out_dense;         // [n][out_stride], nullable
    uint32_t *out_dense_ids;  // nullable
    uint32_t out_stride;
    // scratch
    uint32_t groups;
    uint32_t nwords;          // (N + 31) / 32
    uint32_t cols;            // columns of a work item: SLONN_TILE_COLS or SLONN_WIDE_COLS, or 0: tile_prep_kernel decides
    uint32_t *work;           // number of work items of SLONN_TILE_COLS and of SLONN_WIDE_COLS columns; one of them stays 0; and at SLONN_TILE_TAKEN how many the blocks have taken
    uint32_t *items;          // group << 16 | tile (groups <= 1024 * 8, tiles <= N / 128)
    uint32_t *kseg;           // [groups][33] first entry of each partial sum's stretch, total
    uint32_t *krow;           // [groups][kcap] byte offset of the entry's row of WT
    float *xt;                // [groups][kcap][G] staged values
    uint2 *ucol;              // [groups][N] listed columns of WT, ascending, and their nodes (select)
    uint32_t *ucount;         // [groups] how many
    uint32_t *bm;             // [groups][nwords][G] node bitmap of each query (select)
    uint32_t *pre;            // [groups][nwords][G] nodes of the query below the word
};

__device__ __forceinline__ uint32_t tile_query(const slonn_tile_params &P, uint32_t slot)
{
    if (P.order) return P.count && P.s0 + slot >= *P.count ? 0xffffffffu : P.order[slot];
    if (slot >= P.n) return 0xffffffffu;
    const uint32_t q = P.q0 + slot;
    return P.skip_bp && P.skip_bp[q] == 10000u ? 0xffffffffu : q;
}

// Whether work items of a layer take 256 columns, for `groups` groups that have queries; `listed`: items of 256 columns that the first
// queries of these groups alone fill (selected nodes; a group's union holds at least those).  Nowhere if the layer has more than
// 40 MiB of weights (fp32 4096 x 4096, 128 and 256 columns, every node, 1300 queries 1213 and 1280 us, 656 queries 744 and 861; 90 %
// of the nodes, 4000 queries, 3570 and 3813).
// Every node computed (only where one load brings a lane's eight columns; 2048 x 500, 1000 queries, 91 and 101): 148 items are worked on
// at a time, and 256 columns take 1.8 times as long as 128.  bf16 1536 x 1536, 13 groups 60 and 54, 49 groups 110 and 95, 82
// groups (4 and 7 rounds) 177 and 171; 4096 x 4096, 256 groups, 3157 and 2763.  With more than 10 MiB the first of them start later:
// 4096 x 4096, 7 groups (1 and 2 rounds) 142 and 155, 16 groups 249 and 245, 41 groups (5 and 9) 515 either way; fp32 4096 x 2048, 29
// groups (2 and 4) 261 and 269, 49 groups 370 and 366.  even: the groups' inputs are about equally many.  Behind lists of mixed budgets
// the last items are the longest, and all but a few SMs wait for them: 4096 x 1000, one query in 100 at 35 %, the others at 5 %, 1024
// queries 90 and 106, 2100 queries (4 and 8 rounds) 118 and 140, 4096 queries (7 and 14) 180 and 181 (all at 5 %: 145 and 129).
// Selected nodes: from 2048 items on.  bf16 4096 x 2048, 40 %, 1000 items 946 and 1009, 1628 items 1446 and 1440, 50 %, 1252 items
// 1420 and 1460, 90 %, 2504 items 2210 and 2134; 4096 x 4096, 75 %, 1200 items 1281 and 1349, 3000 items 2910 and 2783; fp32 3072 x 3072,
// 40 %, 2035 items 1496 and 1400.
__host__ __device__ __forceinline__ bool tile_wide_layer(uint32_t D, uint32_t N, uint32_t V, bool select)
{
    return (uint64_t)D * N * (16u / V) <= (40ull << 20) && (select || N % SLONN_WIDE_NN == 0u);
}
__host__ __device__ __forceinline__ bool tile_wide(uint32_t groups, uint32_t D, uint32_t N, uint32_t V, bool select, uint32_t listed, bool even)
{
    if (!tile_wide_layer(D, N, V, select)) return false;
    if (select) return listed >= 2048u;
    const uint32_t wide = (groups * ((N + SLONN_WIDE_COLS - 1) / SLONN_WIDE_COLS) + 147u) / 148u; // rounds
    const uint32_t narrow = (groups * ((N + SLONN_TILE_COLS - 1) / SLONN_TILE_COLS) + 147u) / 148u;
    const uint32_t start = (uint64_t)D * N * (16u / V) <= (10ull << 20) ? 0u : V == 8u ? 2u : 3u;
    return wide * 9u + start <= narrow * 5u && (even || wide >= 7u);
}

static_assert(SLONN_TILE_CHUNK / SLONN_TILE_G <= 512, "a thread of tile_prep_kernel per group");
// Two blocks per group that share nothing: block (g, 0) lists the inputs and stages their values, block (g, 1) lists the
// nodes and adds the group's work items.  One warp per query; a warp's list reads are issued eight at a time.
__global__ void __launch_bounds__(512) tile_prep_kernel(slonn_tile_params P)
{
    slonn_enter();
    extern __shared__ uint32_t smem_u[];
    constexpr int G = SLONN_TILE_G;
    __shared__ uint32_t slotcnt[32];
    __shared__ uint32_t slotstart[33];
    __shared__ uint32_t s_q[G];
    __shared__ uint64_t s_begin[G];
    __shared__ uint32_t s_len[G];
    __shared__ uint32_t wsum[16];
    __shared__ uint2 wcount[16]; // per warp: groups that have queries, items their first queries fill
    const uint32_t g = blockIdx.x;
    const uint32_t tid = threadIdx.x, lane = tid & 31u, warp = tid >> 5; // warp: the query this warp reads the list of
    const bool nodes = blockIdx.y != 0u;
    const bool lists = nodes ? P.select != 0u : P.in.kind == SLONN_IN_LIST;

    bool any = false;
    if (tid < (uint32_t)G) {
        const uint32_t slot = g * G + tid;
        const uint32_t q = slot < P.n ? tile_query(P, slot) : 0xffffffffu;
        uint64_t begin = 0;
        uint32_t len = 0;
        if (q != 0xffffffffu) {
            any = true;
            if (lists) {
                const uint64_t *ip = nodes ? P.indptr + (uint64_t)q * P.n_act + P.a : P.in.indptr + (uint64_t)q * P.in.ip_mul + P.in.ip_add;
                begin = ip[0];
                len = (uint32_t)(ip[1] - begin);
            }
        }
        s_q[tid] = q; s_begin[tid] = begin; s_len[tid] = len;
    }

    if (nodes) {
        uint32_t *nbits = smem_u;          // [nwords] listed columns of WT
        uint32_t *bm = nbits + P.nwords;   // [G][nwords] the queries' nodes
        uint32_t ncols = P.N;
        if (P.select) for (uint32_t i = tid; i < (G + 1u) * P.nwords; i += blockDim.x) nbits[i] = 0u;
        if (!__syncthreads_or(any)) return;
        // Which queries a launch serves only the device knows (those of a budget range, of a list): the width of the work items is
        // decided here, by every group alike, from one query of each group (a thread's; at most 512 groups).
        if (P.cols == 0u) {
            uint32_t q = 0xffffffffu;
            if (tid < P.groups) // with an order a group's queries come first
                for (uint32_t k = 0; k < (P.order ? 1u : (uint32_t)G) && q == 0xffffffffu; ++k) q = tid * G + k < P.n ? tile_query(P, tid * G + k) : 0xffffffffu;
            uint32_t items = 0;
            if (P.select && q != 0xffffffffu) {
                const uint64_t *ip = P.indptr + (uint64_t)q * P.n_act + P.a;
                items = ((uint32_t)(ip[1] - ip[0]) + SLONN_WIDE_COLS - 1) / SLONN_WIDE_COLS;
            }
            const uint32_t have = __popc(__ballot_sync(SLONN_FULL_MASK, q != 0xffffffffu));
            items = __reduce_add_sync(SLONN_FULL_MASK, items);
            if (lane == 0) wcount[warp] = make_uint2(have, items); // read behind the next barrier
            if (!P.select) __syncthreads();
        }
        if (P.select) {
            const uint32_t *ids = P.ids + s_begin[warp];
            const uint32_t len = s_len[warp];
            for (uint32_t i0 = 0; i0 < len; i0 += 256u) {
                uint32_t id[8], col[8];
#pragma unroll
                for (int u = 0; u < 8; ++u) id[u] = i0 + u * 32u + lane < len ? min(ids[i0 + u * 32u + lane], P.N - 1u) : 0xffffffffu;
#pragma unroll
                for (int u = 0; u < 8; ++u) col[u] = id[u] != 0xffffffffu && P.colpos ? __ldg(P.colpos + id[u]) : id[u];
#pragma unroll
                for (int u = 0; u < 8; ++u)
                    if (id[u] != 0xffffffffu) {
                        atomicOr(&bm[warp * P.nwords + (id[u] >> 5)], 1u << (id[u] & 31u));
                        atomicOr(&nbits[col[u] >> 5], 1u << (col[u] & 31u));
                    }
            }
            __syncthreads();
            // each query's bitmap and the nodes below each word
            {
                uint32_t base = 0;
                for (uint32_t w0 = 0; w0 < P.nwords; w0 += 32u) {
                    const uint32_t w = w0 + lane;
                    const uint32_t bits = w < P.nwords ? bm[warp * P.nwords + w] : 0u;
                    const uint32_t c = __popc(bits);
                    uint32_t incl = c;
#pragma unroll
                    for (int off = 1; off < 32; off <<= 1) {
                        const uint32_t t = __shfl_up_sync(SLONN_FULL_MASK, incl, off);
                        if (lane >= (uint32_t)off) incl += t;
                    }
                    if (w < P.nwords) {
                        const uint64_t at = ((uint64_t)g * P.nwords + w) * G + warp;
                        P.bm[at] = bits;
                        P.pre[at] = base + incl - c;
                    }
                    base += __shfl_sync(SLONN_FULL_MASK, incl, 31);
                }
            }
            // listed columns, ascending
            const uint32_t wpt = (P.nwords + blockDim.x - 1) / blockDim.x;
            const uint32_t w0 = tid * wpt, w1 = min(w0 + wpt, P.nwords);
            uint32_t c = 0;
            for (uint32_t w = w0; w < w1; ++w) c += __popc(nbits[w]);
            uint32_t incl = c;
#pragma unroll
            for (int off = 1; off < 32; off <<= 1) {
                const uint32_t t = __shfl_up_sync(SLONN_FULL_MASK, incl, off);
                if (lane >= (uint32_t)off) incl += t;
            }
            if (lane == 31) wsum[warp] = incl;
            __syncthreads();
            uint32_t before = 0, all = 0;
            for (uint32_t w = 0; w < 16u; ++w) {
                if (w < warp) before += wsum[w];
                all += wsum[w];
            }
            uint32_t o = before + incl - c;
            for (uint32_t w = w0; w < w1; ++w) {
                uint32_t bits = nbits[w];
                while (bits) {
                    const uint32_t t = __ffs(bits) - 1;
                    bits &= bits - 1;
                    const uint32_t col = (w << 5) + t;
                    P.ucol[(uint64_t)g * P.N + o++] = make_uint2(col, P.colnode ? __ldg(P.colnode + col) : col);
                }
            }
            ncols = all;
        }
        if (tid < 32u) {
            bool wide = P.cols == SLONN_WIDE_COLS;
            if (P.cols == 0u) {
                const uint2 c = tid < 16u ? wcount[tid] : make_uint2(0u, 0u);
                const uint32_t have = __reduce_add_sync(SLONN_FULL_MASK, c.x), items = __reduce_add_sync(SLONN_FULL_MASK, c.y);
                wide = tile_wide(have, P.D, P.N, P.V, P.select != 0u, items, P.in.kind != SLONN_IN_LIST || P.count);
            }
            const uint32_t cols = wide ? SLONN_WIDE_COLS : SLONN_TILE_COLS;
            const uint32_t tiles = (ncols + cols - 1) / cols;
            uint32_t base = 0;
            if (tid == 0) {
                P.ucount[g] = ncols;
                base = atomicAdd(P.work + (wide ? 1 : 0), tiles);
            }
            base = __shfl_sync(SLONN_FULL_MASK, base, 0);
            for (uint32_t t = tid; t < tiles; t += 32u) P.items[base + t] = (g << 16) | t;
        }
        return;
    }

    uint32_t *kbits = smem_u;              // [32 * wps] listed inputs, by partial sum
    uint32_t *kpre = kbits + 32u * P.wps;  // listed inputs of the partial sum below the word
    for (uint32_t i = tid; i < 32u * P.wps; i += blockDim.x) kbits[i] = 0u;
    if (!__syncthreads_or(any)) return;
    // input j: chunk c = j / V belongs to partial sum c mod 32 and is its chunk number c / 32
    auto bit_of = [&](uint32_t j, uint32_t &slot, uint32_t &pos) {
        const uint32_t c = P.V == 8u ? j >> 3 : j >> 2;
        slot = tile_slot(c & 31u);
        pos = P.V == 8u ? ((c >> 5) << 3) + (j & 7u) : ((c >> 5) << 2) + (j & 3u);
    };
    auto place_of = [&](uint32_t j) -> uint32_t {
        uint32_t slot, pos;
        bit_of(j, slot, pos);
        const uint32_t w = slot * P.wps + (pos >> 5);
        return slotstart[slot] + kpre[w] + __popc(kbits[w] & ((1u << (pos & 31u)) - 1u));
    };
    // the nonzero inputs of this warp's query, eight loads at a time
    auto for_inputs = [&](auto &&f) {
        const uint32_t *ids = P.in.ids + s_begin[warp];
        const float *vals = P.in.vals + s_begin[warp];
        const uint32_t len = s_len[warp];
        for (uint32_t i0 = 0; i0 < len; i0 += 256u) {
            uint32_t j[8];
            float v[8];
#pragma unroll
            for (int u = 0; u < 8; ++u) {
                const bool in = i0 + u * 32u + lane < len;
                j[u] = in ? ids[i0 + u * 32u + lane] : 0xffffffffu;
                v[u] = in ? vals[i0 + u * 32u + lane] : 0.0f;
            }
#pragma unroll
            for (int u = 0; u < 8; ++u)
                if (v[u] != 0.0f && j[u] < P.D) f(j[u], v[u]);
        }
    };
    if (lists) {
        for_inputs([&](uint32_t j, float) {
            uint32_t slot, pos;
            bit_of(j, slot, pos);
            atomicOr(&kbits[slot * P.wps + (pos >> 5)], 1u << (pos & 31u));
        });
    } else {
        for (uint32_t j = tid; j < P.D; j += blockDim.x) {
            uint32_t slot, pos;
            bit_of(j, slot, pos);
            atomicOr(&kbits[slot * P.wps + (pos >> 5)], 1u << (pos & 31u));
        }
    }
    __syncthreads();

    // places of the listed inputs: stretches of an even number of entries, one per partial sum
    for (uint32_t s = warp; s < 32u; s += 16u) {
        uint32_t base = 0;
        for (uint32_t w0 = 0; w0 < P.wps; w0 += 32u) {
            const uint32_t c = w0 + lane < P.wps ? __popc(kbits[s * P.wps + w0 + lane]) : 0u;
            uint32_t incl = c;
#pragma unroll
            for (int off = 1; off < 32; off <<= 1) {
                const uint32_t t = __shfl_up_sync(SLONN_FULL_MASK, incl, off);
                if (lane >= (uint32_t)off) incl += t;
            }
            if (w0 + lane < P.wps) kpre[s * P.wps + w0 + lane] = base + incl - c;
            base += __shfl_sync(SLONN_FULL_MASK, incl, 31);
        }
        if (lane == 0) slotcnt[s] = base;
    }
    __syncthreads();
    if (warp == 0) {
        const uint32_t c = (slotcnt[lane] + 1u) & ~1u;
        uint32_t incl = c;
#pragma unroll
        for (int off = 1; off < 32; off <<= 1) {
            const uint32_t t = __shfl_up_sync(SLONN_FULL_MASK, incl, off);
            if (lane >= (uint32_t)off) incl += t;
        }
        slotstart[lane] = incl - c;
        P.kseg[g * 33u + lane] = incl - c;
        if (lane == 31) { slotstart[32] = incl; P.kseg[g * 33u + 32u] = incl; }
    }
    __syncthreads();
    uint32_t *krow = P.krow + (uint64_t)g * P.kcap;
    float *xt = P.xt + (uint64_t)g * P.kcap * G;
    float4 *xt4 = reinterpret_cast<float4 *>(xt);
    const uint32_t total = slotstart[32];
    if (tid < SLONN_TILE_SLACK - 32u) krow[total + tid] = 0u; // loaded ahead by the walk, never used: a valid row
    if (lists) {
        const float4 z = make_float4(0.f, 0.f, 0.f, 0.f);
        for (uint32_t i = tid; i < total * (G / 4); i += blockDim.x) xt4[i] = z;
        for (uint32_t i = tid; i < 32u * P.wps; i += blockDim.x) { // the listed inputs' rows, word by word
            const uint32_t slot = i / P.wps, w = i - slot * P.wps;
            const uint32_t p = tile_partial(slot);
            uint32_t bits = kbits[i], at = slotstart[slot] + kpre[i];
            while (bits) {
                const uint32_t t = __ffs(bits) - 1;
                bits &= bits - 1;
                const uint32_t pos = (w << 5) + t;
                const uint32_t j = P.V == 8u ? (((pos >> 3) * 32u + p) << 3) + (pos & 7u) : (((pos >> 2) * 32u + p) << 2) + (pos & 3u);
                krow[at++] = j * P.ldb;
            }
        }
        if (tid < 32u && (slotcnt[tid] & 1u)) krow[slotstart[tid] + slotcnt[tid]] = 0u; // an odd stretch: one entry of zeros
        __syncthreads();
        for_inputs([&](uint32_t j, float v) { xt[(uint64_t)place_of(j) * G + warp] = v; });
    } else {
        for (uint32_t j = tid; j < P.D; j += blockDim.x) {
            const uint32_t at = place_of(j);
            krow[at] = j * P.ldb;
            float v[G];
#pragma unroll
            for (int i = 0; i < G; ++i) v[i] = s_q[i] != 0xffffffffu ? P.in.dense[(uint64_t)s_q[i] * P.D + j] : 0.0f;
#pragma unroll
            for (int i = 0; i < G; i += 4) xt4[((uint64_t)at * G + i) / 4] = make_float4(v[i], v[i + 1], v[i + 2], v[i + 3]);
        }
        if (tid < 32u && (slotcnt[tid] & 1u)) {
            const uint32_t at = slotstart[tid] + slotcnt[tid];
            krow[at] = 0u;
            for (int i = 0; i < G; ++i) xt[(uint64_t)at * G + i] = 0.0f;
        }
    }
}

// ---------------------------------------------------------------------------
// the product
// ---------------------------------------------------------------------------
template <int BYTES>
__device__ __forceinline__ void tile_cp_async(uint32_t dst, const void *src)
{
    if constexpr (BYTES == 16) asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst), "l"(src) : "memory");
    else asm volatile("cp.async.ca.shared.global [%0], [%1], %2;" ::"r"(dst), "l"(src), "n"(BYTES) : "memory");
}


// shared memory of tile_rows_kernel
#define SLONN_TILE_BLOCK 16                    // entries a warp copies ahead at a time
#define SLONN_TILE_RING (3 * SLONN_TILE_BLOCK) // entries in a warp's ring
#define SLONN_TILE_ROWS_AT (SLONN_TILE_RING * SLONN_TILE_G * 4) // values, then row offsets
#define SLONN_TILE_RING_BYTES (SLONN_TILE_ROWS_AT + SLONN_TILE_RING * 4 + 16) // the first row offsets again behind the last
#define SLONN_TILE_PART (SLONN_TILE_COLS * SLONN_TILE_G) // floats of a warp's sums
#define SLONN_TILE_SMEM ((size_t)SLONN_TILE_WARPS * (SLONN_TILE_RING_BYTES + SLONN_TILE_PART * 4))
#define SLONN_TILE_STATIC (2 * SLONN_TILE_COLS * 8 + 2 * SLONN_TILE_WARPS * 32 + 2 * SLONN_TILE_G * 12 + 8) // s_col, s_item, s_q, s_off, s_next and s_items
static_assert(SLONN_TILE_SMEM > 46 * 1024 && SLONN_TILE_SMEM + SLONN_TILE_STATIC <= 227 * 1024,
              "tile_rows_kernel must opt in to its shared memory and fit a block's 227 KB with its static part");

// The four weights of a lane for one entry, as loaded from p[j] + row.  QUAD: four neighbouring columns, one load; else
// one load each.
template <bool BF16, bool QUAD> struct tile_weights {
    uint32_t r[(BF16 && QUAD) ? 2 : 4];
    __device__ __forceinline__ void load(const unsigned char *const (&p)[QUAD ? 1 : SLONN_TILE_NN], uint32_t row)
    {
        if constexpr (QUAD && BF16) {
            const uint2 v = __ldg(reinterpret_cast<const uint2 *>(p[0] + row));
            r[0] = v.x; r[1] = v.y;
        } else if constexpr (QUAD) {
            const uint4 v = __ldg(reinterpret_cast<const uint4 *>(p[0] + row));
            r[0] = v.x; r[1] = v.y; r[2] = v.z; r[3] = v.w;
        } else {
#pragma unroll
            for (int j = 0; j < SLONN_TILE_NN; ++j)
                r[j] = BF16 ? (uint32_t)__ldg(reinterpret_cast<const uint16_t *>(p[j] + row))
                            : __ldg(reinterpret_cast<const uint32_t *>(p[j] + row));
        }
    }
    // columns 2 i and 2 i + 1, widened.  bf16 through the permute unit: shifts left to the compiler become integer
    // multiply-adds on the FMA pipe, which is the busy one.
    __device__ __forceinline__ float2 pair(int i) const
    {
        if constexpr (!BF16) return make_float2(__uint_as_float(r[2 * i]), __uint_as_float(r[2 * i + 1]));
        else if constexpr (QUAD) return make_float2(__uint_as_float(__byte_perm(r[i], 0u, 0x1044)), __uint_as_float(__byte_perm(r[i], 0u, 0x3244)));
        else return make_float2(__uint_as_float(__byte_perm(r[2 * i], 0u, 0x1044)), __uint_as_float(__byte_perm(r[2 * i + 1], 0u, 0x1044)));
    }
};

// One block of 16 warps per SM takes work items (group, 128 columns) until none is left.  A warp walks the entries of
// two partial sums (p and p + 16); a lane holds the 16 queries' sums of four columns (64 accumulators).  Per entry: 16
// values broadcast from the warp's ring in shared memory, four weights loaded two entries ahead into registers, 32
// packed multiply-adds (one value times two columns' weights; each half rounded on its own, as fmaf does).  What the
// next item needs first (its entry stretches, its columns, the first values and weights) is fetched while the block
// finishes the one at hand.
// QUAD: a lane's columns are neighbours and one load fetches their weights (every node computed, N a multiple of 4).
template <bool BF16, bool QUAD>
__global__ void __launch_bounds__(SLONN_TILE_WARPS * 32, 1) tile_rows_kernel(slonn_tile_params P)
{
    slonn_enter();
    constexpr int G = SLONN_TILE_G, NN = SLONN_TILE_NN, W = SLONN_TILE_WARPS;
    constexpr uint32_t ESZ = BF16 ? 2u : 4u;
    constexpr uint32_t BLOCK_STEPS = SLONN_TILE_BLOCK / 2;
    extern __shared__ __align__(16) unsigned char smem_b[];
    __shared__ __align__(8) uint2 s_col[2][SLONN_TILE_COLS]; // column and node of each slot (select)
    __shared__ __align__(16) uint32_t s_item[2][W][8]; // per warp: its three kseg values, column count, item
    __shared__ uint32_t s_q[2][G];
    __shared__ uint64_t s_off[2][G];
    const uint32_t tid = threadIdx.x, lane = tid & 31u, warp = tid >> 5;
    unsigned char *ring = smem_b + warp * SLONN_TILE_RING_BYTES;
    const uint32_t ring_s = (uint32_t)__cvta_generic_to_shared(ring);
    float *part = reinterpret_cast<float *>(smem_b + W * SLONN_TILE_RING_BYTES); // [warp][query][column slot]
    // this lane's column slots: 64 i + 2 lane + {0, 1}
    float *mypart = part + warp * SLONN_TILE_PART + 2u * lane;
    // union index of column slot s of a tile
    auto slot_index = [&](uint32_t tile, uint32_t s) -> uint32_t {
        return tile * SLONN_TILE_COLS + (QUAD ? ((s & 63u) >> 1) * 4u + (s >> 6) * 2u + (s & 1u) : s);
    };
    __shared__ uint32_t s_next, s_items; // the item after next; items in all, which is read from here so that it holds no register in the loop
    auto n_items = [&]() { return *reinterpret_cast<volatile uint32_t *>(&s_items); };

    // the item at hand: the steps of the warp's two partial sums, the lane's columns in row 0
    uint32_t nA = 0, nst = 0; // steps of two entries: of the first partial sum, of both
    const unsigned char *p[QUAD ? 1 : NN];
    tile_weights<BF16, QUAD> wn[2];
    uint32_t copied = 0;      // steps whose copies have been issued
    uint32_t at_copy = 0;     // ring block (0, 1, 2) the next copies go to
    const uint32_t *krow = nullptr;
    const unsigned char *xsrc = nullptr;
    auto copy_block = [&]() {
        if (copied < nst) {
            const uint32_t dst = ring_s + at_copy * (SLONN_TILE_BLOCK * G * 4);
            tile_cp_async<16>(dst + lane * 16u, xsrc + lane * 16u);
            tile_cp_async<16>(dst + 512u + lane * 16u, xsrc + 512u + lane * 16u);
            if (lane < 8u) tile_cp_async<8>(ring_s + SLONN_TILE_ROWS_AT + at_copy * (SLONN_TILE_BLOCK * 4) + lane * 8u, krow + lane * 2u);
            if (lane == 8u && at_copy == 0u) tile_cp_async<8>(ring_s + SLONN_TILE_ROWS_AT + SLONN_TILE_RING * 4, krow);
            xsrc += SLONN_TILE_BLOCK * G * 4;
            krow += SLONN_TILE_BLOCK;
            copied += BLOCK_STEPS;
            at_copy = at_copy == 2u ? 0u : at_copy + 1u;
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
    };
    // fetches what a warp needs to know of an item into s_item[buf][warp]
    // (and, between the block's threads, the item's columns into s_col[buf])
    auto look_up = [&](uint32_t index, uint32_t buf) {
        const uint32_t item = P.items[index];
        if (P.select && tid < SLONN_TILE_COLS) // entries behind the group's last are not used, but stay inside the scratch
            tile_cp_async<8>((uint32_t)__cvta_generic_to_shared(&s_col[buf][tid]),
                             P.ucol + (uint64_t)(item >> 16) * P.N + min((item & 0xffffu) * SLONN_TILE_COLS + tid, P.N - 1u));
        if (lane == 4u) s_item[buf][warp][4] = item;
        if (lane < 4u)
            tile_cp_async<4>((uint32_t)__cvta_generic_to_shared(&s_item[buf][warp][lane]),
                             lane < 3u ? P.kseg + (item >> 16) * 33u + (warp & 7u) * 4u + (warp >> 3) * 2u + lane : P.ucount + (item >> 16));
    };
    // makes the item looked up in s_item[buf] the item at hand and starts the copies of its first blocks
    auto start_copies = [&](uint32_t buf) {
        const uint4 m = *reinterpret_cast<const uint4 *>(s_item[buf][warp]);
        const uint32_t item = s_item[buf][warp][4], g = item >> 16;
        nA = (m.y - m.x) >> 1; nst = (m.z - m.x) >> 1;
        krow = P.krow + (uint64_t)g * P.kcap + m.x;
        xsrc = reinterpret_cast<const unsigned char *>(P.xt + ((uint64_t)g * P.kcap + m.x) * G);
        copied = 0; at_copy = 0;
        copy_block(); copy_block();
        if (tid < (uint32_t)G) {
            const uint32_t slot = g * G + tid;
            const uint32_t q = slot < P.n ? tile_query(P, slot) : 0xffffffffu;
            s_q[buf][tid] = q;
            s_off[buf][tid] = (q != 0xffffffffu && P.indptr) ? P.indptr[(uint64_t)q * P.n_act + P.a] : 0;
        }
    };
    // and, behind a barrier of the block, its first weights
    auto start_weights = [&](uint32_t buf) {
        const uint32_t tile = s_item[buf][warp][4] & 0xffffu, last = s_item[buf][warp][3] - tile * SLONN_TILE_COLS - 1u;
        const unsigned char *WT = reinterpret_cast<const unsigned char *>(P.WT);
        if constexpr (QUAD) {
            p[0] = WT + (uint64_t)min(tile * SLONN_TILE_COLS + lane * 4u, P.N - 4u) * ESZ;
        } else {
#pragma unroll
            for (int j = 0; j < NN; ++j) {
                const uint32_t s = min((j >> 1) * 64u + lane * 2u + (j & 1), last); // slots behind the last column repeat it
                p[j] = WT + (uint64_t)(P.select ? s_col[buf][s].x : tile * SLONN_TILE_COLS + s) * ESZ;
            }
        }
        asm volatile("cp.async.wait_group 1;" ::: "memory");
        __syncwarp();
        if (nst) {
            const uint2 r = *reinterpret_cast<const uint2 *>(ring + SLONN_TILE_ROWS_AT);
            wn[0].load(p, r.x);
            wn[1].load(p, r.y);
        }
    };

    // Items differ (unions, budgets), so beyond the first two a block takes the next one nobody has (dealt out in turn, second layer of
    // 8192 queries of 5 to 100 % on 4096 x 4096 1338 us, now 1280; 4096 queries at 10 % on as many, sort and staging included, 182
    // and 177; from the end of the list, where the highest budgets are, 1292).
    uint32_t next = blockIdx.x + gridDim.x;
    {
        const uint32_t n = P.work[0];
        if (blockIdx.x >= n) return;
        if (tid == 0) s_items = n;
    }
    for (uint32_t i = lane; i < SLONN_TILE_RING_BYTES / 4; i += 32) reinterpret_cast<uint32_t *>(ring)[i] = 0u; // row offsets that exist
    look_up(blockIdx.x, 0u);
    asm volatile("cp.async.wait_all;" ::: "memory");
    __syncthreads();
    start_copies(0u);
    start_weights(0u);

    for (uint32_t buf = 0;; buf ^= 1u) {
        uint32_t taken = 0;
        if (tid == 0 && next < n_items()) taken = 2u * gridDim.x + atomicAdd(P.work + SLONN_TILE_TAKEN, 1u);
        float2 acc[G][NN / 2];
#pragma unroll
        for (int i = 0; i < G; ++i)
#pragma unroll
            for (int j = 0; j < NN / 2; ++j) acc[i][j] = make_float2(0.0f, 0.0f);
        uint32_t st = 0, block_end = 0;                                   // step at hand, first step of the next ring block
        const float4 *x4 = reinterpret_cast<const float4 *>(ring);        // its values
        const uint2 *rows = reinterpret_cast<const uint2 *>(ring + SLONN_TILE_ROWS_AT); // its rows
#pragma unroll 1
        for (uint32_t half = 0; half < 2; ++half) { // the warp's two partial sums
            const uint32_t end = half ? nst : nA;
#pragma unroll 1
            while (st < end) {
                if (st == block_end) { // a new ring block: the one after it must have landed too, the one before is free
                    asm volatile("cp.async.wait_group 0;" ::: "memory");
                    __syncwarp();
                    copy_block();
                    block_end += BLOCK_STEPS;
                    if (x4 == reinterpret_cast<const float4 *>(ring + SLONN_TILE_ROWS_AT)) {
                        x4 = reinterpret_cast<const float4 *>(ring);
                        rows = reinterpret_cast<const uint2 *>(ring + SLONN_TILE_ROWS_AT);
                    }
                }
                const uint32_t stop = min(end, block_end);
#pragma unroll 1
                do {
                    float2 w[2][NN / 2];
#pragma unroll
                    for (int e = 0; e < 2; ++e)
#pragma unroll
                        for (int j = 0; j < NN / 2; ++j) w[e][j] = wn[e].pair(j);
                    const uint2 r = *++rows; // the next step's rows (behind the last step: rows that exist, not used)
                    wn[0].load(p, r.x);
                    wn[1].load(p, r.y);
                    constexpr int RUN = 8; // neighbouring multiply-adds that share the weight pair
#pragma unroll
                    for (int e = 0; e < 2; ++e)
#pragma unroll
                        for (int i0 = 0; i0 < G; i0 += RUN) {
                            float x[RUN];
#pragma unroll
                            for (int i = 0; i < RUN; i += 4) {
                                const float4 v = x4[e * (G / 4) + (i0 + i) / 4];
                                x[i] = v.x; x[i + 1] = v.y; x[i + 2] = v.z; x[i + 3] = v.w;
                            }
#pragma unroll
                            for (int j = 0; j < NN / 2; ++j)
#pragma unroll
                                for (int i = 0; i < RUN; ++i) acc[i0 + i][j] = __ffma2_rn(make_float2(x[i], x[i]), w[e][j], acc[i0 + i][j]);
                        }
                    x4 += 2 * G / 4;
                } while (++st < stop);
            }
            if (half == 0) { // the first partial sum is complete: put it aside
#pragma unroll
                for (int i = 0; i < G; ++i)
#pragma unroll
                    for (int j = 0; j < NN / 2; ++j) {
                        *reinterpret_cast<float2 *>(mypart + i * SLONN_TILE_COLS + j * 64) = acc[i][j];
                        acc[i][j] = make_float2(0.0f, 0.0f);
                    }
                if (next < n_items()) look_up(next, buf ^ 1u);
            }
        }
#pragma unroll
        for (int i = 0; i < G; ++i)
#pragma unroll
            for (int j = 0; j < NN / 2; ++j) {
                float2 *p = reinterpret_cast<float2 *>(mypart + i * SLONN_TILE_COLS + j * 64);
                *p = __fadd2_rn(*p, acc[i][j]);
            }
        asm volatile("cp.async.wait_all;" ::: "memory");
        __syncwarp();

        const bool more = next < n_items();
        if (tid == 0) s_next = taken;
        // the item's own end, one column and four queries per thread
        const uint32_t g = s_item[buf][warp][4] >> 16, tile = s_item[buf][warp][4] & 0xffffu, cnt = s_item[buf][warp][3];
        const uint32_t s = tid % SLONN_TILE_COLS, quad = tid / SLONN_TILE_COLS;
        const uint32_t u = slot_index(tile, s);
        const bool mine = u < cnt;
        uint32_t nd = 0;
        float b = 0.0f;
        uint4 word = make_uint4(~0u, ~0u, ~0u, ~0u), below = make_uint4(0u, 0u, 0u, 0u);
        if (mine) {
            nd = P.select ? s_col[buf][s].y : P.colnode ? __ldg(P.colnode + u) : u;
            b = __ldg(P.bias + nd);
            if (P.select) {
                const uint64_t at = (((uint64_t)g * P.nwords + (nd >> 5)) * G + quad * 4u) / 4u;
                word = reinterpret_cast<const uint4 *>(P.bm)[at];
                below = reinterpret_cast<const uint4 *>(P.pre)[at];
            }
        }
        if (more) start_copies(buf ^ 1u);
        __syncthreads();
        next = s_next;
        if (more) start_weights(buf ^ 1u);
        if (mine) {
            // the sixteen warps' sums, strides 8, 4, 2, 1 of the tree; then bias, ReLU and the query's list
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const uint32_t q = s_q[buf][quad * 4u + i];
                float v[W];
#pragma unroll
                for (int w = 0; w < W; ++w) v[w] = part[w * SLONN_TILE_PART + (quad * 4u + i) * SLONN_TILE_COLS + s];
#pragma unroll
                for (int off = W / 2; off >= 1; off >>= 1)
#pragma unroll
                    for (int w = 0; w < off; ++w) v[w] = v[w] + v[w + off];
                if (q == 0xffffffffu) continue;
                float z = v[0] + b;
                if (P.relu) z = z > 0.0f ? z : 0.0f;
                uint32_t pos = nd;
                if (P.select) {
                    const uint32_t wd = i == 0 ? word.x : i == 1 ? word.y : i == 2 ? word.z : word.w;
                    const uint32_t bl = i == 0 ? below.x : i == 1 ? below.y : i == 2 ? below.z : below.w;
                    const uint32_t bit = 1u << (nd & 31u);
                    if (!(wd & bit)) continue;
                    pos = bl + __popc(wd & (bit - 1u));
                }
                const uint64_t off = s_off[buf][quad * 4u + i];
                if (P.out_vals) P.out_vals[off + pos] = z;
                if (P.write_ids) P.ids[off + pos] = nd;
                if (P.out_dense) {
                    P.out_dense[(uint64_t)q * P.out_stride + pos] = z;
                    if (P.out_dense_ids) P.out_dense_ids[(uint64_t)q * P.out_stride + pos] = nd;
                }
            }
        }
        if (!more) return;
        __syncthreads(); // the sums have been read
    }
}

// ---------------------------------------------------------------------------
// the product, 256 columns at a time
// ---------------------------------------------------------------------------
// shared memory of tile_rows_wide_kernel
#define SLONN_WIDE_STEP (2 * SLONN_TILE_G * 4 + 16) // bytes of a step in a warp's ring: two entries' values, their row offsets, padding
#define SLONN_WIDE_BLOCK 8                          // steps a warp copies ahead at a time
#define SLONN_WIDE_RING (3 * SLONN_WIDE_BLOCK)      // steps in a warp's ring
#define SLONN_WIDE_ROWS_AT (2 * SLONN_TILE_G * 4)   // row offsets within a step
#define SLONN_WIDE_RING_BYTES ((SLONN_WIDE_RING + 1) * SLONN_WIDE_STEP) // the first step's row offsets again behind the last step
#define SLONN_WIDE_SMEM ((size_t)SLONN_WIDE_WARPS * (SLONN_WIDE_RING_BYTES + SLONN_WIDE_COLS * SLONN_TILE_G * 4))
#define SLONN_WIDE_STATIC (2 * SLONN_WIDE_COLS * 8 + 2 * SLONN_TILE_G * 12 + 2 * SLONN_WIDE_WARPS * 32 + 16) // s_col, s_q, s_off, s_item, s_tmem
#define SLONN_WIDE_TMEM 256 // columns of tensor memory: 128 sums per lane, two warps on the same lanes
static_assert(SLONN_WIDE_SMEM > 46 * 1024 && SLONN_WIDE_SMEM + SLONN_WIDE_STATIC <= 227 * 1024,
              "tile_rows_wide_kernel must opt in to its shared memory and fit a block's 227 KB with its static part");

// N values of every lane of a warp, value(0) to value(N - 1), to its own 32 lanes of tensor memory, 16 columns at a time, and back: take(k,
// v).  All lanes have to execute these instructions together, and the code in front of them branches by lane: the warp meets first.
template <int N, typename F>
__device__ __forceinline__ void tile_tmem_store(uint32_t at, F value)
{
    __syncwarp();
#pragma unroll
    for (int h = 0; h < N; h += 16) {
        uint32_t r[16];
#pragma unroll
        for (int k = 0; k < 16; ++k) r[k] = __float_as_uint(value(h + k));
        asm volatile("tcgen05.st.sync.aligned.32x32b.x16.b32 [%0], "
                     "{%1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, %16};"
                     ::"r"(at + h), "r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7]), "r"(r[8]),
                     "r"(r[9]), "r"(r[10]), "r"(r[11]), "r"(r[12]), "r"(r[13]), "r"(r[14]), "r"(r[15])
                     : "memory");
    }
    asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
}
template <int N, typename F>
__device__ __forceinline__ void tile_tmem_load(uint32_t at, F take)
{
    __syncwarp();
#pragma unroll
    for (int h = 0; h < N; h += 16) {
        uint32_t r[16];
        asm volatile("tcgen05.ld.sync.aligned.32x32b.x16.b32 "
                     "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15}, [%16];\n\t"
                     "tcgen05.wait::ld.sync.aligned;"
                     : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]),
                       "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
                     : "r"(at + h)
                     : "memory");
#pragma unroll
        for (int k = 0; k < 16; ++k) take(h + k, __uint_as_float(r[k]));
    }
}

// The eight weights of a lane for one entry, as loaded from p[j] + row.  VEC: neighbouring columns, 16 bytes per load; else one
// load each.
template <bool BF16, bool VEC> struct wide_weights {
    uint32_t r[(BF16 && VEC) ? 4 : 8];
    __device__ __forceinline__ void load(const unsigned char *const (&p)[VEC ? 1 : SLONN_WIDE_NN], uint32_t row)
    {
        if constexpr (VEC) {
#pragma unroll
            for (int i = 0; i < (BF16 ? 1 : 2); ++i) {
                const uint4 v = __ldg(reinterpret_cast<const uint4 *>(p[0] + row) + i);
                r[4 * i] = v.x; r[4 * i + 1] = v.y; r[4 * i + 2] = v.z; r[4 * i + 3] = v.w;
            }
        } else {
#pragma unroll
            for (int j = 0; j < SLONN_WIDE_NN; ++j)
                r[j] = BF16 ? (uint32_t)__ldg(reinterpret_cast<const uint16_t *>(p[j] + row))
                            : __ldg(reinterpret_cast<const uint32_t *>(p[j] + row));
        }
    }
    __device__ __forceinline__ float2 pair(int i) const // columns 2 i and 2 i + 1, widened (see tile_weights)
    {
        if constexpr (!BF16) return make_float2(__uint_as_float(r[2 * i]), __uint_as_float(r[2 * i + 1]));
        else if constexpr (VEC) return make_float2(__uint_as_float(__byte_perm(r[i], 0u, 0x1044)), __uint_as_float(__byte_perm(r[i], 0u, 0x3244)));
        else return make_float2(__uint_as_float(__byte_perm(r[2 * i], 0u, 0x1044)), __uint_as_float(__byte_perm(r[2 * i + 1], 0u, 0x1044)));
    }
};

// tile_rows_kernel with twice the columns per lane (128 accumulators) and half the warps, one block of 8 warps per SM.  What is not
// a multiply-add takes issue slots and register writes from them (every value and weight loaded costs a cycle of the
// scheduler): per multiply-add the 16 broadcast values, the loop and the waits are halved here.  A warp walks the entries of four
// partial sums, w, w + 16, w + 8, w + 24; a finished one meets its partner of the tree as soon as both exist: the first of two
// waits in tensor memory (128 registers per lane), the sum of the first two in shared memory, where the warps' sums meet in the
// end.  VEC: a lane's columns are neighbours (every node computed, N a multiple of 8).
template <bool BF16, bool VEC>
__global__ void __launch_bounds__(SLONN_WIDE_WARPS * 32, 1) tile_rows_wide_kernel(slonn_tile_params P)
{
    slonn_enter();
    constexpr int G = SLONN_TILE_G, NN = SLONN_WIDE_NN, W = SLONN_WIDE_WARPS, SEGS = 32 / W;
    constexpr uint32_t ESZ = BF16 ? 2u : 4u, STEP = SLONN_WIDE_STEP, COLS = SLONN_WIDE_COLS, PART = COLS * G;
    extern __shared__ __align__(16) unsigned char smem_b[];
    __shared__ __align__(8) uint2 s_col[2][COLS]; // column and node of each slot (select)
    __shared__ __align__(16) uint32_t s_item[2][W][8]; // per warp: its SEGS + 1 kseg values; column count at 5, item at 6
    __shared__ uint64_t s_off[2][G];
    __shared__ uint32_t s_q[2][G];
    __shared__ uint32_t s_tmem;
    const uint32_t n_items = P.work[1];
    uint32_t it = blockIdx.x;
    if (it >= n_items) return;
    const uint32_t tid = threadIdx.x, lane = tid & 31u, warp = tid >> 5;
    const uint32_t ring = warp * SLONN_WIDE_RING_BYTES; // offset in smem_b
    const uint32_t ring_s = (uint32_t)__cvta_generic_to_shared(smem_b) + ring;
    float *part = reinterpret_cast<float *>(smem_b + W * SLONN_WIDE_RING_BYTES); // [warp][query][column slot]
    // this lane's column slots: 64 i + 2 lane + {0, 1}
    float *mypart = part + warp * PART + 2u * lane;
    // union index of column slot s of a tile
    auto slot_index = [&](uint32_t tile, uint32_t s) -> uint32_t {
        return tile * COLS + (VEC ? ((s & 63u) >> 1) * NN + (s >> 6) * 2u + (s & 1u) : s);
    };

    // the item at hand: the lane's columns in row 0
    const unsigned char *p[VEC ? 1 : NN];
    wide_weights<BF16, VEC> wn[2];
    uint32_t at_copy = 0;              // ring block (0, 1, 2) the next copies go to
    uint32_t src = 0, src_end = 0;     // the entry they start with, and the warp's last, of all groups' entries
    auto copy_block = [&]() {
        if (src < src_end) {
            const uint32_t *krow = P.krow + src;
            const unsigned char *xsrc = reinterpret_cast<const unsigned char *>(P.xt + (uint64_t)src * G);
            const uint32_t dst = ring_s + at_copy * (SLONN_WIDE_BLOCK * STEP);
            const uint32_t to = dst + (lane >> 3) * STEP + (lane & 7u) * 16u; // eight lanes copy a step's values
            tile_cp_async<16>(to, xsrc + lane * 16u);
            tile_cp_async<16>(to + 4u * STEP, xsrc + 512u + lane * 16u);
            if (lane < 8u) tile_cp_async<8>(dst + lane * STEP + SLONN_WIDE_ROWS_AT, krow + lane * 2u);
            if (lane == 8u && at_copy == 0u) tile_cp_async<8>(ring_s + SLONN_WIDE_RING * STEP + SLONN_WIDE_ROWS_AT, krow);
            src += SLONN_WIDE_BLOCK * 2;
            at_copy = at_copy == 2u ? 0u : at_copy + 1u;
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
    };
    // fetches what a warp needs to know of an item into s_item[buf][warp]
    // (and, between the block's threads, the item's columns into s_col[buf])
    auto look_up = [&](uint32_t index, uint32_t buf) {
        const uint32_t item = P.items[index];
        if (P.select) // entries behind the group's last are not used, but stay inside the scratch
            tile_cp_async<8>((uint32_t)__cvta_generic_to_shared(&s_col[buf][tid]),
                             P.ucol + (uint64_t)(item >> 16) * P.N + min((item & 0xffffu) * COLS + tid, P.N - 1u));
        if (lane == 6u) s_item[buf][warp][6] = item;
        if (lane <= (uint32_t)SEGS || lane == 5u)
            tile_cp_async<4>((uint32_t)__cvta_generic_to_shared(&s_item[buf][warp][lane]),
                             lane <= (uint32_t)SEGS ? P.kseg + (item >> 16) * 33u + warp * SEGS + lane : P.ucount + (item >> 16));
    };
    // makes the item looked up in s_item[buf] the item at hand and starts the copies of its first blocks
    auto start_copies = [&](uint32_t buf) {
        const uint32_t g = s_item[buf][warp][6] >> 16;
        src = g * P.kcap + s_item[buf][warp][0];
        src_end = g * P.kcap + s_item[buf][warp][SEGS];
        at_copy = 0;
        copy_block(); copy_block();
        if (tid < (uint32_t)G) {
            const uint32_t slot = g * G + tid;
            const uint32_t q = slot < P.n ? tile_query(P, slot) : 0xffffffffu;
            s_q[buf][tid] = q;
            s_off[buf][tid] = (q != 0xffffffffu && P.indptr) ? P.indptr[(uint64_t)q * P.n_act + P.a] : 0;
        }
    };
    // and, behind a barrier of the block, its first weights
    auto start_weights = [&](uint32_t buf) {
        const uint32_t tile = s_item[buf][warp][6] & 0xffffu, last = s_item[buf][warp][5] - tile * COLS - 1u;
        const unsigned char *WT = reinterpret_cast<const unsigned char *>(P.WT);
        if constexpr (VEC) {
            p[0] = WT + (uint64_t)min(tile * COLS + lane * NN, P.N - NN) * ESZ;
        } else {
#pragma unroll
            for (int j = 0; j < NN; ++j) {
                const uint32_t s = min((j >> 1) * 64u + lane * 2u + (j & 1), last); // slots behind the last column repeat it
                p[j] = WT + (uint64_t)(P.select ? s_col[buf][s].x : tile * COLS + s) * ESZ;
            }
        }
        asm volatile("cp.async.wait_group 1;" ::: "memory");
        __syncwarp();
        if (s_item[buf][warp][SEGS] != s_item[buf][warp][0]) {
            const uint2 r = *reinterpret_cast<const uint2 *>(smem_b + ring + SLONN_WIDE_ROWS_AT);
            wn[0].load(p, r.x);
            wn[1].load(p, r.y);
        }
    };

    // items are dealt out in turn: neighbours in the list are of neighbouring groups and cost about the same (whoever is free takes the next,
    // as in tile_rows_kernel: two more registers across the loop than there are, every node of 4096 x 2048 for 1638 queries 1202 -> 1257 us)
    if (warp == 0) {
        __syncwarp();
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"((uint32_t)__cvta_generic_to_shared(&s_tmem)), "r"(SLONN_WIDE_TMEM) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    for (uint32_t i = lane; i < SLONN_WIDE_RING_BYTES / 4; i += 32) reinterpret_cast<uint32_t *>(smem_b + ring)[i] = 0u; // row offsets that exist
    look_up(it, 0u);
    asm volatile("cp.async.wait_all;" ::: "memory");
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const uint32_t tmem = s_tmem + (((warp & 3u) * 32u) << 16) + (warp >> 2) * 128u; // this warp's 32 lanes, 128 columns
    start_copies(0u);
    start_weights(0u);

    for (uint32_t buf = 0;; buf ^= 1u) {
        float2 acc[G][NN / 2];
        uint32_t left = 0; // steps of the ring block ahead
        uint32_t at = ring; // the step at hand, in smem_b
#pragma unroll 1
        for (uint32_t seg = 0; seg < (uint32_t)SEGS; ++seg) { // the warp's partial sums
#pragma unroll
            for (int i = 0; i < G; ++i)
#pragma unroll
                for (int j = 0; j < NN / 2; ++j) acc[i][j] = make_float2(0.0f, 0.0f);
            uint32_t todo = (s_item[buf][warp][seg + 1u] - s_item[buf][warp][seg]) >> 1; // steps of two entries
#pragma unroll 1
            while (todo) {
                if (left == 0) { // a new ring block: the one after it must have landed too, the one before is free
                    asm volatile("cp.async.wait_group 0;" ::: "memory");
                    __syncwarp();
                    copy_block();
                    left = SLONN_WIDE_BLOCK;
                    if (at == ring + SLONN_WIDE_RING * STEP) at = ring;
                }
                const uint32_t now = min(todo, left), at_stop = at + now * STEP;
                todo -= now;
                left -= now;
#pragma unroll 1
                do {
                    float2 w[2][NN / 2];
#pragma unroll
                    for (int e = 0; e < 2; ++e)
#pragma unroll
                        for (int j = 0; j < NN / 2; ++j) w[e][j] = wn[e].pair(j);
                    const uint2 r = *reinterpret_cast<const uint2 *>(smem_b + at + STEP + SLONN_WIDE_ROWS_AT); // the next step's rows (behind the last step: rows that exist, not used)
                    wn[0].load(p, r.x);
                    wn[1].load(p, r.y);
                    constexpr int RUN = 8; // neighbouring multiply-adds that share the weight pair
#pragma unroll
                    for (int e = 0; e < 2; ++e)
#pragma unroll
                        for (int i0 = 0; i0 < G; i0 += RUN) {
                            float x[RUN];
#pragma unroll
                            for (int i = 0; i < RUN; i += 4) {
                                const float4 v = *reinterpret_cast<const float4 *>(smem_b + at + (e * G + i0 + i) * 4);
                                x[i] = v.x; x[i + 1] = v.y; x[i + 2] = v.z; x[i + 3] = v.w;
                            }
#pragma unroll
                            for (int j = 0; j < NN / 2; ++j)
#pragma unroll
                                for (int i = 0; i < RUN; ++i) acc[i0 + i][j] = __ffma2_rn(make_float2(x[i], x[i]), w[e][j], acc[i0 + i][j]);
                        }
                    at += STEP;
                } while (at != at_stop);
            }
            // the partial sum is complete: it waits for its partner, or meets it
            auto sums = [&](int k) -> float & { float2 &v = acc[k / NN][(k % NN) >> 1]; return (k & 1) ? v.y : v.x; };
            if (!(seg & 1u)) {
                tile_tmem_store<G * NN>(tmem, sums);
                continue;
            }
            tile_tmem_load<G * NN>(tmem, [&](int k, float first) { sums(k) = first + sums(k); });
            const bool later = seg >= (uint32_t)SEGS / 2u;
            if (!later) {
                __syncthreads(); // the block has read the sums of the item before
                if (it + gridDim.x < n_items) look_up(it + gridDim.x, buf ^ 1u);
            }
#pragma unroll
            for (int i = 0; i < G; ++i)
#pragma unroll
                for (int j = 0; j < NN / 2; ++j) {
                    float2 *s = reinterpret_cast<float2 *>(mypart + i * COLS + j * 64);
                    *s = later ? __fadd2_rn(*s, acc[i][j]) : acc[i][j];
                }
        }
        asm volatile("cp.async.wait_all;" ::: "memory");
        __syncwarp();

        it += gridDim.x;
        const bool more = it < n_items;
        // the item's own end, one column per thread
        const uint32_t g = s_item[buf][warp][6] >> 16, tile = s_item[buf][warp][6] & 0xffffu, cnt = s_item[buf][warp][5];
        const uint32_t u = slot_index(tile, tid);
        const bool mine = u < cnt;
        uint32_t nd = 0;
        float b = 0.0f;
        uint4 word[G / 4], below[G / 4];
        if (mine) {
            nd = P.select ? s_col[buf][tid].y : P.colnode ? __ldg(P.colnode + u) : u;
            b = __ldg(P.bias + nd);
            if (P.select) {
                const uint64_t from = (((uint64_t)g * P.nwords + (nd >> 5)) * G) / 4u;
#pragma unroll
                for (int i = 0; i < G / 4; ++i) {
                    word[i] = reinterpret_cast<const uint4 *>(P.bm)[from + i];
                    below[i] = reinterpret_cast<const uint4 *>(P.pre)[from + i];
                }
            }
        }
        if (more) start_copies(buf ^ 1u);
        __syncthreads();
        if (more) start_weights(buf ^ 1u);
        if (mine) {
            // the warps' sums, strides W / 2 .. 1 of the tree; then bias, ReLU and the query's list
            auto emit = [&](uint32_t k, uint32_t wd, uint32_t bl) {
                float v[W];
#pragma unroll
                for (int w = 0; w < W; ++w) v[w] = part[w * PART + k * COLS + tid];
#pragma unroll
                for (int off = W / 2; off >= 1; off >>= 1)
#pragma unroll
                    for (int w = 0; w < off; ++w) v[w] = v[w] + v[w + off];
                const uint32_t q = s_q[buf][k];
                if (q == 0xffffffffu) return;
                float z = v[0] + b;
                if (P.relu) z = z > 0.0f ? z : 0.0f;
                uint32_t pos = nd;
                if (P.select) {
                    const uint32_t bit = 1u << (nd & 31u);
                    if (!(wd & bit)) return;
                    pos = bl + __popc(wd & (bit - 1u));
                }
                const uint64_t off = s_off[buf][k];
                if (P.out_vals) P.out_vals[off + pos] = z;
                if (P.write_ids) P.ids[off + pos] = nd;
                if (P.out_dense) {
                    P.out_dense[(uint64_t)q * P.out_stride + pos] = z;
                    if (P.out_dense_ids) P.out_dense_ids[(uint64_t)q * P.out_stride + pos] = nd;
                }
            };
#pragma unroll
            for (int i = 0; i < G / 4; ++i) {
                emit(4 * i, word[i].x, below[i].x);
                emit(4 * i + 1, word[i].y, below[i].y);
                emit(4 * i + 2, word[i].z, below[i].z);
                emit(4 * i + 3, word[i].w, below[i].w);
            }
        }
        if (!more) break;
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    if (warp == 0) {
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        __syncwarp();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(s_tmem), "r"(SLONN_WIDE_TMEM) : "memory");
    }
}

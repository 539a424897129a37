// List-fed layers of batches of tens of queries, input-stationary, in two launches: with so few queries a layer has too
// little work for a block per query (layer_cols_kernel) and too much of it is the same for all blocks of a query to be repeated
// in each (its split form: grouping the list, the hash functions, the selection and the order of the nodes are two thirds of
// a block's time at 10 %).
//   few_select_kernel   one block per query: groups the nonzero inputs, hash functions, keys, selection, nodes in column order;
//                       what the other launch needs of it goes to scratch (a layer without activator: the grouped inputs only)
//   few_nodes_kernel    one block per (query, 32 runs of four columns): its warps share the 32 partial sums, as gather_cols_kernel's split form
// 64 queries at 25 % on nine layers of 4096 nodes: 495 us a pass with hash_select_kernel and whole rows, 327 with these.  Launch by launch
// between events a layer takes 17 and 50 us (rows at 11.7 TB/s from L2), with these 17 and 30.
#pragma once
#include "slonn_cluster_lists.cuh"

#ifndef SLONN_FEW_BLOCKS
#define SLONN_FEW_BLOCKS 5 // 48 registers.  64 queries at 25 % on nine layers of 4096 nodes, 4 / 5 / 6: 378 / 334 / 364 us, 24 at 25 % 277 / 278 / 317, 64 at 10 % 175 / 176 / 180
#endif
#define SLONN_FEW_SEG 36 // words of scratch for a query's borders of partial sums and number of quads

struct slonn_few_params {
    slonn_gather_params G;      // in, WT, colpos, bias, D, N, n_act, a, indptr, ids (= out of the selection), outputs, filters, rows_cap, in_cap
    const void *WH;
    const uint32_t *hash_nodes;
    const void *tables;
    uint32_t cap, K, L, pre, layer;
    uint16_t *codes;            // nullable
    uint32_t *status;
    // scratch, per query
    uint2 *ent;                 // [ent_stride] grouped inputs (j, bits of x_j), each partial sum filled up to a multiple of four
    uint32_t *seg;              // [SLONN_FEW_SEG] where each partial sum begins, how many in all; number of quads
    uint2 *nodes;               // [rows_cap] in column order: place in the id-ascending list, node
    uint2 *quads;               // [quad_stride] runs of four columns that hold a node: first column | which of the four << 16, place of the first in `nodes`
    uint32_t ent_stride;
    uint32_t quad_stride;
    uint32_t scratch_bytes;     // few_select_kernel's shared memory for the grouped inputs
};

template <bool BF16>
__global__ void __launch_bounds__(SLONN_CLUSTER_THREADS, 2) few_select_kernel(const __grid_constant__ slonn_few_params Q)
{
    slonn_enter();
    constexpr uint32_t T = SLONN_CLUSTER_THREADS, W = T / 32u, V = BF16 ? 8u : 4u;
    const slonn_gather_params &P = Q.G;
    extern __shared__ float4 smem4[];
    __shared__ uint32_t counts[SLONN_LISTS_SELECT * W];
    __shared__ uint32_t s_cnt[32];
    __shared__ float part[W * 64u];
    const uint32_t q = blockIdx.x;
    if (P.skip_bp && P.skip_bp[q] == 10000u) return;
    if (!bp_in_range(P.range_bp, P.bp_lo, P.bp_hi, q)) return;
    const uint32_t tid = threadIdx.x, lane = tid & 31u, warp = tid >> 5;
    const uint32_t H = Q.K * Q.L, smax = cols_smax(P.D, V), pitch = (smax + 3u) & ~3u, xfloats = (max(32u * smax, P.N) + 3u) & ~3u;

    // shared memory: inputs by partial sum, then the selection's marks | grouped inputs | the active set
    float *x = reinterpret_cast<float *>(smem4);
    uint2 *ent = reinterpret_cast<uint2 *>(x + xfloats);
    lists_set S;
    S.words = (P.N + 31u) >> 5;
    S.bits = reinterpret_cast<uint32_t *>(reinterpret_cast<char *>(ent) + Q.scratch_bytes);
    S.below = S.bits + S.words; S.idbits = S.below + S.words; S.idbelow = S.idbits + S.words;
    S.node = reinterpret_cast<uint16_t *>(S.idbelow + S.words);
    S.col = S.node + P.rows_cap; S.pos = S.col + P.rows_cap;

    {
        const uint64_t s0 = P.in.indptr[(uint64_t)q * P.in.ip_mul + P.in.ip_add];
        const uint32_t len = min((uint32_t)(P.in.indptr[(uint64_t)q * P.in.ip_mul + P.in.ip_add + 1] - s0), P.in_cap);
        const float4 z = make_float4(0.f, 0.f, 0.f, 0.f);
        for (uint32_t i = tid; i < xfloats / 4u; i += T) smem4[i] = z;
        __syncthreads();
#pragma unroll 2
        for (uint32_t i = tid; i < len; i += T) {
            const uint32_t j = P.in.ids[s0 + i], c = j / V;
            const float v = P.in.vals[s0 + i];
            if (j < P.D) x[(c & 31u) * smax + (c >> 5) * V + (j & (V - 1u))] = v;
        }
        __syncthreads();
    }
    // the warp's two partial sums: grouped inputs, and the hash functions' (two per lane of a half warp)
    uint2 *e0 = ent + warp * pitch, *e1 = e0 + 16u * pitch;
    uint32_t n0, n1;
    const uint32_t m = lists_group<V>(x, smax, warp, lane, e0, e1, n0, n1);
    const bool hash = P.use_list != 0u; // a layer without activator: only its grouped inputs are wanted
    if (lane == 0) { s_cnt[warp] = (n0 + 3u) & ~3u; s_cnt[warp + 16u] = (n1 + 3u) & ~3u; }
    float hb = 0.0f;
    if (hash) {
        const float2 a = lists_hash<BF16>(e0, e1, m, Q.WH, lane);
        if (lane < 16u) *reinterpret_cast<float2 *>(part + warp * 64u + 2u * lane) = a;
        if (lane < H) hb = __ldg(P.bias + __ldg(Q.hash_nodes + lane));
    }
    __syncthreads(); // also: the inputs have been grouped
    { // the grouped inputs, one partial sum behind the other
        const uint32_t c = s_cnt[lane];
        uint32_t incl = c;
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) {
            const uint32_t t = __shfl_up_sync(SLONN_FULL_MASK, incl, d);
            if (lane >= (uint32_t)d) incl += t;
        }
        uint32_t *seg = Q.seg + (uint64_t)q * SLONN_FEW_SEG;
        if (warp == 0) {
            seg[lane] = incl - c;
            if (lane == 31u) seg[32] = incl;
        }
        uint2 *out = Q.ent + (uint64_t)q * Q.ent_stride;
        const uint32_t at0 = __shfl_sync(SLONN_FULL_MASK, incl - c, warp), at1 = __shfl_sync(SLONN_FULL_MASK, incl - c, warp + 16u);
        for (uint32_t i = lane; i < ((n0 + 3u) & ~3u); i += 32u) out[at0 + i] = e0[i];
        for (uint32_t i = lane; i < ((n1 + 3u) & ~3u); i += 32u) out[at1 + i] = e1[i];
    }
    if (!hash) return;
    const uint32_t signs = __ballot_sync(SLONN_FULL_MASK, lane < H && lists_tree(part, lane) + hb > 0.0f);
    auto key = [&](uint32_t b) { return (signs >> (b * Q.K)) & ((1u << Q.K) - 1u); };
    if (Q.codes && tid < Q.L) Q.codes[((uint64_t)q * P.n_act + P.a) * Q.L + tid] = (uint16_t)key(tid);
    const uint64_t off = P.indptr[(uint64_t)q * P.n_act + P.a];
    const uint32_t B = min((uint32_t)(P.indptr[(uint64_t)q * P.n_act + P.a + 1] - off), P.rows_cap);
    const lists_layer ly = {Q.tables, Q.hash_nodes, P.colpos, P.N, Q.cap};
    uint32_t *first = reinterpret_cast<uint32_t *>(x), *ids = const_cast<uint32_t *>(P.ids) + off;
    auto run = [&](auto u) { return lists_select<uint16_t, u.value>(ly, Q.K, Q.L, B, Q.pre, key, first, S, true, counts, ids); };
    const bool ok = (B - Q.pre) * Q.L <= 4u * T ? run(std::integral_constant<int, 4>()) : run(std::integral_constant<int, SLONN_LISTS_SELECT>());
    if (!ok && tid == 0) slonn_report(Q.status, SLONN_ERR_ARG, q, Q.layer);
    __syncthreads();
    for (uint32_t i = tid; i < B; i += T) Q.nodes[(uint64_t)q * P.rows_cap + i] = make_uint2(S.pos[i], S.node[i]);
    // the runs of four columns that hold a node (a warp: four words of the bitmap)
    const uint32_t rounds = (P.N / 4u + T - 1u) / T; // at most four
    auto held = [&](uint32_t r) -> uint32_t {
        const uint32_t c = (r * T + tid) * 4u;
        return c < P.N ? (S.bits[c >> 5] >> (c & 31u)) & 15u : 0u;
    };
    for (uint32_t r = 0; r < rounds; ++r) {
        const uint32_t c = __popc(__ballot_sync(SLONN_FULL_MASK, held(r) != 0u));
        if (lane == 0) counts[r * W + warp] = c;
    }
    __syncthreads();
    for (uint32_t r = 0; r < rounds; ++r) {
        uint32_t before = 0;
        for (uint32_t i = lane; i < r * W + warp; i += 32u) before += counts[i];
        before = __reduce_add_sync(SLONN_FULL_MASK, before);
        const uint32_t h = held(r), some = __ballot_sync(SLONN_FULL_MASK, h != 0u), c = (r * T + tid) * 4u;
        if (h) {
            const uint32_t at = S.below[c >> 5] + __popc(S.bits[c >> 5] & ((1u << (c & 31u)) - 1u));
            Q.quads[(uint64_t)q * Q.quad_stride + before + __popc(some & ((1u << lane) - 1u))] = make_uint2(c | (h << 16), at);
        }
        if (r + 1u == rounds && tid == T - 1u) Q.seg[(uint64_t)q * SLONN_FEW_SEG + 33] = before + __popc(some);
    }
}

// The four weights of a run of columns of one input, `off` bytes into WT (a multiple of four element sizes).
template <bool BF16>
__device__ __forceinline__ void few_load(const void *WT, uint32_t off, uint32_t (&w)[BF16 ? 2 : 4])
{
    const char *p = reinterpret_cast<const char *>(WT) + off;
    if constexpr (BF16) {
        const uint2 v = __ldg(reinterpret_cast<const uint2 *>(p));
        w[0] = v.x; w[1] = v.y;
    } else {
        const uint4 v = __ldg(reinterpret_cast<const uint4 *>(p));
        w[0] = v.x; w[1] = v.y; w[2] = v.z; w[3] = v.w;
    }
}
template <bool BF16>
__device__ __forceinline__ void few_add(const uint32_t (&w)[BF16 ? 2 : 4], uint32_t xbits, float2 (&a)[2])
{
    const float x = __uint_as_float(xbits);
#pragma unroll
    for (int i = 0; i < 2; ++i) {
        float2 v;
        if constexpr (BF16) v = make_float2(bf16_lo(w[i]), bf16_hi(w[i]));
        else v = make_float2(__uint_as_float(w[2 * i]), __uint_as_float(w[2 * i + 1]));
        a[i] = __ffma2_rn(v, make_float2(x, x), a[i]);
    }
}

// What bounds it is the way from L2: a query's columns in sectors, 8.6 TB/s under the profiler, the L1 68 % busy.  Lane = run of four columns: in column
// order most of a run's columns are selected, and a request brings 32 of them instead of 32 columns (64 queries at 25 %, 4096 x
// 4096, without events: 37 us a layer with a column or two per lane, 26 with runs; blocks of one SM on neighbouring queries' same
// columns, for L1 hits, measured with two columns per lane: 42).
template <bool BF16>
__global__ void __launch_bounds__(SLONN_THREADS, SLONN_FEW_BLOCKS) few_nodes_kernel(const __grid_constant__ slonn_few_params Q)
{
    slonn_enter();
    constexpr uint32_t ESZ = BF16 ? 2u : 4u;
    const slonn_gather_params &P = Q.G;
    extern __shared__ float4 smem4[];
    __shared__ uint32_t seg[33];
    // Fewer than 96 queries: all queries' first runs, then all second ones, so that the blocks behind a query's last run, which the host does
    // not know, come last and the SMs work on the same columns (nine layers of 4096, 25 %: 24 queries 278 -> 270 us, 64 347 -> 331, 35 %:
    // 358 -> 327; but 100 queries 434 -> 444, 140 at 35 % 763 -> 787: the queries' own inputs then miss L1).
    const uint32_t n = gridDim.x / P.ctas_per_query;
    const uint32_t q = n < 96u ? blockIdx.x % n : blockIdx.x / P.ctas_per_query, chunk = n < 96u ? blockIdx.x / n : blockIdx.x - q * P.ctas_per_query, r0 = chunk * 32u;
    if (P.skip_bp && P.skip_bp[q] == 10000u) return;
    if (!bp_in_range(P.range_bp, P.bp_lo, P.bp_hi, q)) return;
    const uint32_t *gseg = Q.seg + (uint64_t)q * SLONN_FEW_SEG;
    const uint32_t nquads = P.use_list ? min(gseg[33], Q.quad_stride) : P.N / 4u;
    if (r0 >= nquads) return;
    const uint32_t tid = threadIdx.x, lane = tid & 31u, warp = tid >> 5, nwarps = SLONN_THREADS / 32u;
    // shared memory: the partial sums [32][4][32], lane innermost | grouped inputs
    float *zpart = reinterpret_cast<float *>(smem4);
    uint2 *ent = reinterpret_cast<uint2 *>(zpart + 32 * 4 * 32);
    const uint32_t total = min(gseg[32], Q.ent_stride);
    if (tid < 33u) seg[tid] = gseg[tid];
    const uint4 *src = reinterpret_cast<const uint4 *>(Q.ent + (uint64_t)q * Q.ent_stride);
    for (uint32_t i = tid; i < total / 2u; i += SLONN_THREADS) reinterpret_cast<uint4 *>(ent)[i] = src[i];
    uint2 quad = make_uint2(min(r0 + lane, nquads - 1u) * 4u | (15u << 16), 0u);
    if (P.use_list) quad = Q.quads[(uint64_t)q * Q.quad_stride + min(r0 + lane, nquads - 1u)];
    const uint32_t cb = (quad.x & 0xffffu) * ESZ, ldb = P.N * ESZ;
    __syncthreads();
    for (uint32_t p = warp; p < 32u; p += nwarps) {
        float2 a[2] = {make_float2(0.0f, 0.0f), make_float2(0.0f, 0.0f)};
        uint32_t k = seg[p];
        const uint32_t e = seg[p + 1];
        auto walk = [&](auto count) { // entries k .. k + count - 1, all loads first
            constexpr int C = count.value;
            uint32_t w[C][BF16 ? 2 : 4];
#pragma unroll
            for (int i = 0; i < C; i += 2) {
                const uint4 v = *reinterpret_cast<const uint4 *>(ent + k + i);
                few_load<BF16>(P.WT, v.x * ldb + cb, w[i]);
                few_load<BF16>(P.WT, v.z * ldb + cb, w[i + 1]);
            }
#pragma unroll
            for (int i = 0; i < C; i += 2) {
                const uint4 v = *reinterpret_cast<const uint4 *>(ent + k + i);
                few_add<BF16>(w[i], v.y, a);
                few_add<BF16>(w[i + 1], v.w, a);
            }
            k += C;
        };
        while (k + 8u <= e) walk(std::integral_constant<int, 8>());
        if (k < e) walk(std::integral_constant<int, 4>());
        float *z = zpart + p * 128u + lane;
        z[0] = a[0].x; z[32] = a[0].y; z[64] = a[1].x; z[96] = a[1].y;
    }
    __syncthreads();
    if (warp >= 4u || r0 + lane >= nquads || !((quad.x >> (16u + warp)) & 1u)) return; // warp c finishes the runs' column c
    uint2 mine; // place in the id-ascending list, node
    if (P.use_list) mine = Q.nodes[(uint64_t)q * P.rows_cap + quad.y + __popc((quad.x >> 16) & ((1u << warp) - 1u))];
    else mine.x = mine.y = (quad.x & 0xffffu) + warp;
    const float b = __ldg(P.bias + mine.y);
    float acc[32];
#pragma unroll
    for (int p = 0; p < 32; ++p) acc[p] = zpart[p * 128u + warp * 32u + lane];
    float z = cols_tree(acc) + b;
    if (P.relu) z = z > 0.0f ? z : 0.0f;
    const uint32_t pos = mine.x;
    if (P.use_list && P.out_vals) P.out_vals[P.indptr[(uint64_t)q * P.n_act + P.a] + pos] = z;
    if (P.out_dense) {
        P.out_dense[(uint64_t)q * P.out_stride + pos] = z;
        if (P.out_dense_ids) P.out_dense_ids[(uint64_t)q * P.out_stride + pos] = mine.y;
    }
}

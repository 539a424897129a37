// The latency path for networks with list-fed layers: as cluster_network_kernel, one cluster of 16 blocks per query, but a
// layer that is fed by an activator layer's list and has its transposed copies runs INPUT-STATIONARY.  What bounds this path
// is the chain of dependent round trips per layer, and this form has the shortest:
//   1. every block groups the nonzero inputs by partial sum for itself (warp w those of w and w + 16: no barrier);
//   2. block r computes the hash functions' partial sums r and r + 16 from the side-by-side hash rows (one 64-byte line per nonzero
//      input) and sends them to all;                                                                 cluster barrier
//   3. every block runs the selection: each list position marks its node with the lowest position that names it, the
//      positions that find their own mark are the first ones of their nodes, and one count over them in position order
//      cuts the list at the budget (a handful of block barriers whatever the overlap of the lists);
//   4. the block evaluates its share of the nodes, lane = node, in column order, a warp its two partial sums of all of them, 16
//      loads per lane in flight; activations go to every block's copy of the next input.      cluster barrier
// Two cluster barriers per layer as before, but B_out * B_in weights instead of B_out rows.  Nine layers of 4096 nodes, one query at
// 10 %, whole rows and this form: 64 different queries in turn 121 and 88 us a pass, three models in turn 156 and 87, weights and code
// from HBM 176 and 127.  Of a layer's 9.2 us (clock stamps): grouping 0.9, hash 2.1, selection 2.7 (list loads 1.0 of it),
// nodes 1.8, delivery and barrier 1.7; a layer run by rows takes 13.
// Every phase is short enough that its instruction count, times the four warps of a scheduler, is what it takes: all loads
// in flight at once cost more in spills than they saved (lists_walk with 16 entries of both partial sums in flight 3.7 us, 8: 1.8).
// Other clusters bringing the weights into L2 ahead of time: 104 us where queries follow one another (not measured from HBM).
// Layers whose input is dense run as in cluster_network_kernel.  They share the selection's code with the others: fetched from HBM,
// a second copy of it took 8 us of a pass (three layers of 1024 at 3 %: 43 us, now 34; by rows 35).
#pragma once
#include "slonn_cluster_kernel.cuh"

#define SLONN_LISTS_SELECT 8 // list positions per thread, most
#define SLONN_LISTS_POSITIONS (SLONN_LISTS_SELECT * SLONN_CLUSTER_THREADS)
#define SLONN_LISTS_DEPTH 4  // 16-byte chunks of a weight row in flight per lane (8: the first layer takes as long, the others 3 % longer: spills)

// ---- selection ----------------------------------------------------------------------

// Where a block keeps a layer's active set: per place (by column where the layer runs input-stationary, else by id) the node,
// its column and its place by id.
struct lists_set {
    uint32_t *bits, *below;     // [words] marked columns, and how many lie below each word
    uint32_t *idbits, *idbelow; // the same by id, where the places differ and somebody asks for them
    uint16_t *node, *col, *pos;
    uint32_t words;
};

// What the selection reads of a layer.  colpos: places are by column of this order; NULL: by id.
struct lists_layer {
    const void *tables;
    const uint32_t *hash_nodes, *colpos;
    uint32_t N, cap;
};

// The layer's active set by the rule of block_select, for at most SLONN_LISTS_POSITIONS list positions.  A whole block of
// SLONN_CLUSTER_THREADS; key(b): table b's; `first`: N words of scratch, a multiple of four.  by_id: places by id are wanted.  ids_out: nullable, the id-ascending
// list.  Ends without a barrier.  Every place below B is filled whatever the lists hold (a saved model's entries are not checked on
// loading); returns false when they did not hold enough distinct ids beside the hash nodes.
// U: positions per thread.
template <typename IDT, int U, typename KEY>
__device__ __forceinline__ bool lists_select(const lists_layer &ly, uint32_t K, uint32_t L, uint32_t B, uint32_t pre,
                                             KEY &&key, uint32_t *first, const lists_set &S, bool by_id,
                                             uint32_t *counts /* [SELECT * 16] shared */, uint32_t *ids_out)
{
    constexpr uint32_t T = SLONN_CLUSTER_THREADS, W = T / 32u;
    static_assert(W == 16u, "a warp reads the counts of a row of positions with half of its lanes");
    const uint32_t tid = threadIdx.x, lane = tid & 31u, warp = tid >> 5;
    const uint32_t *colpos = ly.colpos;
    by_id = by_id && colpos;
    const uint32_t want = B - pre, npos = want * L;
    bool ok = true, listed = B != ly.N && want <= ly.cap; // not listed: nodes 0 .. B - 1 (all, or more than the lists hold, which the plan reports)

    uint32_t id[U], col[U];
    {
        uint32_t r = tid / L, b = tid - r * L; // rank and table of the thread's first position
        const uint32_t rs = T / L, bs = T - rs * L;
        if (bs == 0u) { // the others are of the same list
            const uint64_t bucket = ((uint64_t)b << K) + key(b);
            const IDT *ranked = reinterpret_cast<const IDT *>(ly.tables) + bucket * ly.cap + r;
#pragma unroll
            for (int u = 0; u < U; ++u) id[u] = listed && u * T + tid < npos ? (uint32_t)__ldg(ranked + u * rs) : 0xffffffffu;
        } else {
#pragma unroll
            for (int u = 0; u < U; ++u) {
                id[u] = listed && u * T + tid < npos ? table_entry<IDT>(ly.tables, ly.cap, K, b, key(b), r) : 0xffffffffu;
                r += rs; b += bs;
                if (b >= L) { b -= L; ++r; }
            }
        }
    }
    uint32_t hnode = tid < pre ? __ldg(ly.hash_nodes + tid) : 0xffffffffu, hcol = hnode; // always active
    for (uint32_t i = tid; i < (ly.N + 3u) / 4u; i += T) reinterpret_cast<uint4 *>(first)[i] = make_uint4(~0u, ~0u, ~0u, ~0u);
    for (uint32_t i = tid; i < S.words; i += T) { S.bits[i] = 0u; S.idbits[i] = 0u; }
    __syncthreads();
#pragma unroll
    for (int u = 0; u < U; ++u)
        if (id[u] < ly.N) atomicMin(&first[id[u]], u * T + tid + 1u);
    if (tid < pre) atomicMin(&first[hnode], 0u); // below every list position: an entry that names a hash node is not counted
#pragma unroll
    for (int u = 0; u < U; ++u) col[u] = id[u] < ly.N && colpos ? __ldg(colpos + id[u]) : id[u];
    if (tid < pre && colpos) hcol = __ldg(colpos + hnode);
    __syncthreads();
    uint32_t own[U]; // the warp's positions that are the first of their node
#pragma unroll
    for (int u = 0; u < U; ++u) {
        own[u] = 0u;
        if (u * T >= npos) continue; // uniform
        own[u] = __ballot_sync(SLONN_FULL_MASK, id[u] < ly.N && first[min(id[u], ly.N - 1u)] == u * T + tid + 1u);
        if (lane == 0) counts[u * W + warp] = __popc(own[u]);
    }
    __syncthreads();
    uint32_t total = 0, taken = 0; // taken: bit u = this thread's position u is in the active set
#pragma unroll
    for (int u = 0; u < U; ++u) {
        if (u * T >= npos) continue;
        const uint32_t c = lane < W ? counts[u * W + lane] : 0u;
        const uint32_t sum = __reduce_add_sync(SLONN_FULL_MASK, c | (lane < warp ? c << 16 : 0u)); // all warps' | those below this one
        if (((own[u] >> lane) & 1u) && total + (sum >> 16) + __popc(own[u] & ((1u << lane) - 1u)) < want) taken |= 1u << u;
        total += sum & 0xffffu;
    }
    if (listed && total < want) ok = listed = false; // uniform
    auto mark = [&](uint32_t node, uint32_t c) {
        atomicOr(&S.bits[c >> 5], 1u << (c & 31u));
        if (by_id) atomicOr(&S.idbits[node >> 5], 1u << (node & 31u));
    };
    auto each = [&](auto &&f) { // the thread's share of the set: f(node, column)
        if (!listed) {
            for (uint32_t i = tid; i < B; i += T) f(i, colpos ? __ldg(colpos + i) : i);
            return;
        }
#pragma unroll
        for (int u = 0; u < U; ++u)
            if ((taken >> u) & 1u) f(id[u], col[u]);
        if (tid < pre) f(hnode, hcol);
    };
    each(mark);
    __syncthreads();
    if (warp < (by_id ? 2u : 1u)) { // what lies below each word: warp 0 by column, warp 1 by id
        const uint32_t *bits = warp ? S.idbits : S.bits;
        uint32_t *below = warp ? S.idbelow : S.below;
        const uint32_t per = (S.words + 31u) >> 5, w0 = min(lane * per, S.words), w1 = min(w0 + per, S.words);
        uint32_t c = 0;
        for (uint32_t w = w0; w < w1; ++w) c += __popc(bits[w]);
        uint32_t run = c;
#pragma unroll
        for (int off = 1; off < 32; off <<= 1) {
            const uint32_t t = __shfl_up_sync(SLONN_FULL_MASK, run, off);
            if (lane >= (uint32_t)off) run += t;
        }
        run -= c;
        for (uint32_t w = w0; w < w1; ++w) { below[w] = run; run += __popc(bits[w]); }
    }
    __syncthreads();
    auto place = [&](uint32_t node, uint32_t c) {
        const uint32_t at = S.below[c >> 5] + __popc(S.bits[c >> 5] & ((1u << (c & 31u)) - 1u));
        const uint32_t by = by_id ? S.idbelow[node >> 5] + __popc(S.idbits[node >> 5] & ((1u << (node & 31u)) - 1u)) : at;
        S.node[at] = (uint16_t)node; S.col[at] = (uint16_t)c; S.pos[at] = (uint16_t)by;
        if (ids_out) ids_out[by] = node;
    };
    each(place);
    return ok;
}

// ---- input-stationary sums ------------------------------------------------------------

// a[r] = sum of a warp's two partial sums (w and w + 16) for the weights cb[r] bytes into the rows (of ldb bytes) of WT: entries
// e0[0 .. m) of the one and e1[0 .. m) of the other, each in order, m a multiple of 4.  All loads of G groups of four are issued
// before the first is waited for.
template <bool BF16, int R>
__device__ __forceinline__ void lists_walk(const uint2 *e0, const uint2 *e1, uint32_t m, const void *WT, uint32_t ldb, const uint32_t (&cb)[R], float (&a)[R])
{
    constexpr int G = R == 1 ? 2 : 1;
    float b[R];
#pragma unroll
    for (int r = 0; r < R; ++r) a[r] = b[r] = 0.0f;
#pragma unroll 1
    for (uint32_t k = 0; k < m; k += 4u * G) {
        float w[G][2][R][4];
#pragma unroll
        for (int g = 0; g < G; ++g)
            if (k + 4u * g < m) {
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    const uint4 *e = reinterpret_cast<const uint4 *>((h ? e1 : e0) + k + 4u * g);
                    const uint32_t j[4] = {e[0].x, e[0].z, e[1].x, e[1].z};
#pragma unroll
                    for (int i = 0; i < 4; ++i)
#pragma unroll
                        for (int r = 0; r < R; ++r) w[g][h][r][i] = cols_weight_at<BF16>(WT, j[i] * ldb + cb[r]);
                }
            }
#pragma unroll
        for (int g = 0; g < G; ++g)
            if (k + 4u * g < m) {
                const uint4 *f0 = reinterpret_cast<const uint4 *>(e0 + k + 4u * g), *f1 = reinterpret_cast<const uint4 *>(e1 + k + 4u * g);
                const uint32_t x0[4] = {f0[0].y, f0[0].w, f0[1].y, f0[1].w}, x1[4] = {f1[0].y, f1[0].w, f1[1].y, f1[1].w};
#pragma unroll
                for (int i = 0; i < 4; ++i)
#pragma unroll
                    for (int r = 0; r < R; ++r) {
                        a[r] = fmaf(w[g][0][r][i], __uint_as_float(x0[i]), a[r]);
                        b[r] = fmaf(w[g][1][r][i], __uint_as_float(x1[i]), b[r]);
                    }
            }
    }
#pragma unroll
    for (int r = 0; r < R; ++r) a[r] = a[r] + b[r];
}

// The hash functions' sums of the partial sums of e0 and e1 for the inputs both list (as lists_walk), functions 2 (lane mod 16) and
// the one behind it: half of the warp walks e0, the other e1, a load brings two functions' weights.
template <bool BF16>
__device__ __forceinline__ float2 lists_hash(const uint2 *e0, const uint2 *e1, uint32_t m, const void *WH, uint32_t lane)
{
    constexpr uint32_t ESZ = BF16 ? 2u : 4u;
    const uint4 *e = reinterpret_cast<const uint4 *>(lane & 16u ? e1 : e0);
    const uint32_t cb = (lane & 15u) * 2u * ESZ;
    float2 a = make_float2(0.0f, 0.0f);
#pragma unroll 1
    for (uint32_t k = 0; k < m; k += 16u, e += 8) {
        float w[16][2];
#pragma unroll
        for (int i = 0; i < 8; ++i)
            if (k + 2u * i < m) {
                const uint4 v = e[i];
                cols_weight2_at<BF16>(WH, v.x * (32u * ESZ) + cb, w[2 * i][0], w[2 * i][1]);
                cols_weight2_at<BF16>(WH, v.z * (32u * ESZ) + cb, w[2 * i + 1][0], w[2 * i + 1][1]);
            }
#pragma unroll
        for (int i = 0; i < 8; ++i)
            if (k + 2u * i < m) {
                const uint4 v = e[i];
                a.x = fmaf(w[2 * i][0], __uint_as_float(v.y), a.x);
                a.y = fmaf(w[2 * i][1], __uint_as_float(v.y), a.y);
                a.x = fmaf(w[2 * i + 1][0], __uint_as_float(v.w), a.x);
                a.y = fmaf(w[2 * i + 1][1], __uint_as_float(v.w), a.y);
            }
    }
    a.x = a.x + __shfl_xor_sync(SLONN_FULL_MASK, a.x, 16);
    a.y = a.y + __shfl_xor_sync(SLONN_FULL_MASK, a.y, 16);
    return a;
}

// The nonzero inputs of partial sums `warp` and `warp + 16` of a layer's inputs x (by partial sum, smax each: lists_index) to e0 and
// e1, in order: n0 and n1 of them, and both filled up to the returned multiple of four with inputs that are listed anyway, at
// the value 0.  One warp.
template <uint32_t V>
__device__ __forceinline__ uint32_t lists_group(const float *x, uint32_t smax, uint32_t warp, uint32_t lane, uint2 *e0, uint2 *e1, uint32_t &n0, uint32_t &n1)
{
    const uint32_t lower = (1u << lane) - 1u;
    n0 = n1 = 0;
    for (uint32_t i0 = 0; i0 < smax; i0 += 128u) { // four neighbours per lane, of one chunk
        const uint32_t i = i0 + 4u * lane;
        const bool in = i < smax;
        auto group = [&](uint32_t p, uint2 *e, uint32_t &n) {
            const float4 v = in ? *reinterpret_cast<const float4 *>(x + p * smax + i) : make_float4(0.f, 0.f, 0.f, 0.f);
            const uint32_t b0 = __ballot_sync(SLONN_FULL_MASK, v.x != 0.0f), b1 = __ballot_sync(SLONN_FULL_MASK, v.y != 0.0f);
            const uint32_t b2 = __ballot_sync(SLONN_FULL_MASK, v.z != 0.0f), b3 = __ballot_sync(SLONN_FULL_MASK, v.w != 0.0f);
            uint2 *at = e + n + __popc(b0 & lower) + __popc(b1 & lower) + __popc(b2 & lower) + __popc(b3 & lower);
            const uint32_t j = ((i / V) * 32u + p) * V + (i & (V - 1u));
            if (v.x != 0.0f) *at++ = make_uint2(j, __float_as_uint(v.x));
            if (v.y != 0.0f) *at++ = make_uint2(j + 1u, __float_as_uint(v.y));
            if (v.z != 0.0f) *at++ = make_uint2(j + 2u, __float_as_uint(v.z));
            if (v.w != 0.0f) *at++ = make_uint2(j + 3u, __float_as_uint(v.w));
            n += __popc(b0) + __popc(b1) + __popc(b2) + __popc(b3);
        };
        group(warp, e0, n0);
        group(warp + 16u, e1, n1);
    }
    __syncwarp();
    const uint32_t m = (max(n0, n1) + 3u) & ~3u;
    const uint32_t j = n0 ? e0[0].x : e1[0].x; // m == 0: not used
    __syncwarp();
    for (uint32_t i = n0 + lane; i < m; i += 32u) e0[i] = make_uint2(j, 0u);
    for (uint32_t i = n1 + lane; i < m; i += 32u) e1[i] = make_uint2(j, 0u);
    __syncwarp();
    return m;
}

// The sums of the 16 warps (part[warp][64]) of slot s, strides 8, 4, 2, 1 of the tree.
__device__ __forceinline__ float lists_tree(const float *part, uint32_t s)
{
    float v[16];
#pragma unroll
    for (int w = 0; w < 16; ++w) v[w] = part[w * 64 + s];
#pragma unroll
    for (int off = 8; off >= 1; off >>= 1)
#pragma unroll
        for (int w = 0; w < off; ++w) v[w] = v[w] + v[w + off];
    return v[0];
}

// Where input j of a layer lies in a block's copy: as warp_dot_row1 reads it, or, for a layer that runs input-stationary, by
// partial sum (D / V chunks of V inputs; chunk c belongs to partial sum c mod 32).
template <bool BF16>
__device__ __forceinline__ uint32_t lists_index(const slonn_cluster_layer &ly, uint32_t j)
{
    constexpr uint32_t V = BF16 ? 8u : 4u;
    if (!ly.by_input) return xs_index<BF16>(j, ly.nchunks);
    const uint32_t c = j / V;
    return (c & 31u) * cols_smax(ly.D, V) + (c >> 5) * V + (j & (V - 1u));
}

template <bool BF16>
__global__ void __launch_bounds__(SLONN_CLUSTER_THREADS, 1) cluster_lists_kernel(const __grid_constant__ slonn_cluster_params P)
{
    slonn_enter();
    namespace cg = cooperative_groups;
    cg::cluster_group cluster = cg::this_cluster();
    constexpr uint32_t T = SLONN_CLUSTER_THREADS, W = T / 32u, V = BF16 ? 8u : 4u, ESZ = BF16 ? 2u : 4u;
    static_assert(SLONN_CLUSTER_SIZE == 16 && W == 16u, "warp r of block r computes the hash functions' partial sums r and r + 16");
    extern __shared__ float4 smem4[];
    __shared__ float zh[128];
    __shared__ uint32_t keys[8];
    __shared__ uint32_t counts[SLONN_LISTS_SELECT * W];
    __shared__ uint64_t s_off[SLONN_MAX_LAYERS];
    __shared__ uint32_t s_cnt[SLONN_MAX_LAYERS], s_at[4];
    __shared__ float s_hbias[SLONN_MAX_LAYERS][32]; // biases of the hash nodes where the layer runs input-stationary
    __shared__ slonn_cluster_layer s_layer[SLONN_MAX_LAYERS]; // a layer's constants would each be fetched from L2 on their first use

    const uint32_t C = P.cluster;
    const uint32_t rank = cluster.block_rank();
    const uint32_t q = blockIdx.x / C;
    const uint32_t tid = threadIdx.x, lane = tid & 31u, warp = tid >> 5;
    const uint32_t gwarp = warp * C + rank, gwarps = C * W; // rows are dealt out to the blocks in turn
    const uint32_t H = P.K * P.L;

    // shared memory: two inputs | grouped inputs, or the selection's marks where a layer runs by rows | two sets of the warps'
    // sums | the active set
    float *xin = reinterpret_cast<float *>(smem4), *xout = xin + P.xbuf_floats; // they change places from layer to layer
    // where the rest begins is kept in shared memory too: registers that live through the whole kernel cost spills
    char *const smem_c = reinterpret_cast<char *>(smem4);
    if (tid == 0) {
        s_at[0] = P.xbuf_floats * 8u;
        s_at[1] = s_at[0] + P.scratch_bytes;
        s_at[2] = s_at[1] + 2u * W * 64u * 4u;
    }
    auto entries = [&]() { return reinterpret_cast<uint2 *>(smem_c + s_at[0]); };
    auto sums = [&]() { return reinterpret_cast<float *>(smem_c + s_at[1]); };
    auto active_set = [&]() {
        lists_set S;
        S.bits = reinterpret_cast<uint32_t *>(smem_c + s_at[2]);
        S.below = S.bits + P.bitmap_words; S.idbits = S.below + P.bitmap_words; S.idbelow = S.idbits + P.bitmap_words;
        S.node = reinterpret_cast<uint16_t *>(S.idbelow + P.bitmap_words);
        S.col = S.node + P.ids_cap; S.pos = S.col + P.ids_cap;
        S.words = 0;
        return S;
    };

    if (tid == 0) cluster_plan(P, q, rank, s_off, s_cnt);
    static_assert(sizeof(slonn_cluster_layer) % 8 == 0, "copied in 64-bit words");
    for (uint32_t i = tid; i < P.n_layers * (uint32_t)(sizeof(slonn_cluster_layer) / 8); i += T)
        reinterpret_cast<uint64_t *>(s_layer)[i] = reinterpret_cast<const uint64_t *>(P.layer)[i];
    for (uint32_t l = warp; l < P.n_layers; l += W)
        if (P.layer[l].by_input && P.layer[l].has_act && lane < H) s_hbias[l][lane] = __ldg(P.layer[l].bias + __ldg(P.layer[l].hash_nodes + lane));
    auto clear = [&](float *x) {
        const float4 z = make_float4(0.f, 0.f, 0.f, 0.f);
        for (uint32_t i = tid; i < (P.xbuf_floats >> 2); i += T) reinterpret_cast<float4 *>(x)[i] = z;
    };
    { // input := x (every block its own copy; the first layer runs by rows)
        const slonn_cluster_layer &l0 = P.layer[0];
        const float4 *src = reinterpret_cast<const float4 *>(P.x + (uint64_t)q * l0.D);
        float4 *dst = smem4;
#pragma unroll 4
        for (uint32_t i = tid; i < (l0.D >> 2); i += T) {
            const float4 v = __ldg(src + i);
            if (BF16) dst[(i & 1u) * l0.nchunks + (i >> 1)] = v;
            else dst[i] = v;
        }
    }
    clear(xout);
    cluster.sync(); // every block runs, and the buffer the first layer's activations go to is zero

    for (uint32_t l = 0; l < P.n_layers; ++l) {
        const slonn_cluster_layer &ly = s_layer[l];
        const bool is_last = l + 1 == P.n_layers;
        // xout is all zero here, in every block
        const uint64_t off = ly.has_act ? s_off[l] : 0;
        const uint32_t B = ly.has_act ? s_cnt[l] : ly.N;
        uint32_t *ids_out = rank == 0 && P.out_ids ? P.out_ids + off : nullptr;
        const bool by_id = is_last || P.out_vals || ids_out;
        auto select = [&](uint32_t *first, auto &&key) {
            lists_set S = active_set();
            S.words = (ly.N + 31u) >> 5;
            // nodes of a layer number at most SLONN_CLUSTER_MAX_N: 16-bit ids
            const uint32_t npos = (B - P.pre) * P.L;
            const lists_layer sl = {ly.tables, ly.hash_nodes, ly.by_input ? ly.colpos : nullptr, ly.N, ly.cap};
            auto run = [&](auto u) { return lists_select<uint16_t, u.value>(sl, P.K, P.L, B, P.pre, key, first, S, by_id, counts, ids_out); };
            const bool ok = npos <= 2 * T ? run(std::integral_constant<int, 2>()) : npos <= 4 * T ? run(std::integral_constant<int, 4>())
                                                                                  : run(std::integral_constant<int, SLONN_LISTS_SELECT>());
            if (!ok && rank == 0 && tid == 0) slonn_report(P.status, SLONN_ERR_ARG, q, l);
            __syncthreads();
        };
        // sum z of node nd, place `by` in the id-ascending list, to block `to`
        auto deliver = [&](uint32_t to, uint32_t nd, uint32_t by, float z) {
            if (ly.relu) z = z > 0.0f ? z : 0.0f;
            if (to == 0) {
                if (ly.has_act && P.out_vals) P.out_vals[off + by] = z;
                if (is_last) {
                    P.logits[(uint64_t)q * P.logit_stride + by] = z;
                    if (ly.has_act) P.logit_ids[(uint64_t)q * P.logit_stride + by] = nd;
                }
            }
            // the next layer's input or, after the last, the logits by place for the prediction
            if (!is_last) *cluster.map_shared_rank(&xout[lists_index<BF16>(s_layer[l + 1], nd)], to) = z;
            else if (to == 0) *cluster.map_shared_rank(&xout[by], 0) = z;
        };

        uint2 *e0 = nullptr, *e1 = nullptr; // input-stationary: the grouped inputs of the warp's two partial sums
        uint32_t m = 0, signs = 0;
        if (!ly.by_input) {
            if (ly.has_act) {
                // FreeHash rows, spread over the cluster; each sum goes to every block
                for (uint32_t h = gwarp; h < H; h += gwarps) {
                    const uint32_t nd = __ldg(ly.hash_nodes + h);
                    const float b = __ldg(ly.bias + nd);
                    const float z = warp_dot_row1<BF16, SLONN_LISTS_DEPTH>(reinterpret_cast<const uint4 *>(ly.W) + (uint64_t)nd * ly.nchunks, reinterpret_cast<const float4 *>(xin), ly.nchunks, lane) + b;
                    if (lane < C) *cluster.map_shared_rank(&zh[h], lane) = z;
                }
                cluster.sync();
                if (tid < P.L) {
                    uint32_t key = 0;
                    for (uint32_t j = 0; j < P.K; ++j)
                        if (zh[tid * P.K + j] > 0.0f) key |= (1u << j);
                    keys[tid] = key;
                }
                __syncthreads();
            }
        } else {
            const uint32_t smax = cols_smax(ly.D, V), pitch = (smax + 3u) & ~3u;
            e0 = entries() + warp * pitch; e1 = e0 + 16u * pitch;
            uint32_t n0, n1;
            m = lists_group<V>(xin, smax, warp, lane, e0, e1, n0, n1);
            if (ly.has_act) {
                // the hash functions' partial sums rank and rank + 16, to every block
                if (warp == rank) {
                    const float2 a = lists_hash<BF16>(e0, e1, m, P.layer[l].WH, lane);
                    float *at = sums() + rank * 64u + (lane & 15u) * 2u;
                    for (uint32_t to = lane >> 4; to < C; to += 2u) *cluster.map_shared_rank(reinterpret_cast<float2 *>(at), to) = a;
                }
                cluster.sync(); // also: the block has grouped its inputs
                signs = __ballot_sync(SLONN_FULL_MASK, lane < H && lists_tree(sums(), lane) + s_hbias[l][lane] > 0.0f);
            } else {
                __syncthreads();
            }
        }
        if (ly.has_act) {
            auto key = [&](uint32_t b) { return ly.by_input ? (signs >> (b * P.K)) & ((1u << P.K) - 1u) : keys[b]; };
            if (rank == 0 && P.codes && tid < P.L) P.codes[((uint64_t)q * P.n_act + ly.a) * P.L + tid] = (uint16_t)key(tid);
            // the marks lie where the input was, or the grouped inputs would be; as an offset, so that it stays an address of shared memory
            // (a choice of two pointers: 1 % slower)
            select(reinterpret_cast<uint32_t *>(smem_c + (!ly.by_input ? s_at[0] : l & 1u ? P.xbuf_floats * 4u : 0u)), key);
        }
        if (!ly.by_input) {
            for (uint32_t r = gwarp; r < B; r += gwarps) {
                const uint32_t nd = ly.has_act ? active_set().node[r] : r;
                const float b = __ldg(ly.bias + nd);
                const float z = warp_dot_row1<BF16, SLONN_LISTS_DEPTH>(reinterpret_cast<const uint4 *>(ly.W) + (uint64_t)nd * ly.nchunks, reinterpret_cast<const float4 *>(xin), ly.nchunks, lane) + b;
                if (lane < C) deliver(lane, nd, r, z);
            }
            __syncthreads();
            clear(xin);
        } else {
            uint32_t buf = ly.has_act; // the set of sums that the hash functions' have left free
            if (!is_last) clear(xin);
            // the block's share of the nodes, up to 64 at a time
            const uint32_t per = (B + C - 1u) / C, r0 = min(rank * per, B), r1 = min(r0 + per, B);
            auto nodes = [&](uint32_t r, auto two) {
                constexpr int R = two.value;
                uint32_t nd[R], by[R], cb[R];
                float b[R], a[R];
#pragma unroll
                for (int k = 0; k < R; ++k) {
                    const uint32_t s = min(r + k * 32u + lane, r1 - 1u);
                    nd[k] = by[k] = s;
                    uint32_t col = s;
                    if (ly.has_act) { const lists_set S = active_set(); nd[k] = S.node[s]; by[k] = S.pos[s]; col = S.col[s]; }
                    cb[k] = col * ESZ;
                    b[k] = __ldg(ly.bias + nd[k]);
                }
                lists_walk<BF16, R>(e0, e1, m, P.layer[l].WT, ly.N * ESZ, cb, a);
                float *mine = sums() + buf * (W * 64u);
#pragma unroll
                for (int k = 0; k < R; ++k) mine[warp * 64u + k * 32u + lane] = a[k];
                __syncthreads(); // the other set of sums is free behind this
#pragma unroll
                for (int k = 0; k < R; ++k) {
                    const float z = lists_tree(mine, k * 32u + lane) + b[k];
                    if (r + k * 32u + lane < r1)
                        for (uint32_t to = warp; to < C; to += W) deliver(to, nd[k], by[k], z);
                }
                buf ^= 1u;
            };
            for (uint32_t r = r0; r < r1; r += 64u) { // uniform for the block
                if (r1 - r > 32u) nodes(r, std::integral_constant<int, 2>());
                else nodes(r, std::integral_constant<int, 1>());
            }
        }
        cluster.sync(); // every activation of this layer delivered, the input it read zeroed

        if (is_last && rank == 0 && P.pred) {
            const uint32_t bi = cluster_argmax(xout, B);
            if (tid == 0 && bi != 0xffffffffu)
                P.pred[q] = ly.has_act ? *reinterpret_cast<volatile uint32_t *>(P.logit_ids + (uint64_t)q * P.logit_stride + bi) : bi; // written within the cluster
        }
        float *const t = xin;
        xin = xout; xout = t;
    }
}

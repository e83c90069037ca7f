// Which slots of a regular patch's tile hold a value (sww_tile.cuh), one bit each, taken
// from the flags when the active lists are built (the flags of a grid do not change
// until its next adaptation, the trend runs four times a step).  With the flags of the
// 121 nodes and 363 edges of an 8 x 8 tile staged byte by byte, half of a tile's copies
// and a sixth of its instructions went to them.
//
// Included inside an anonymous namespace after sww_bodies.cuh (tile.h at file scope).
#pragma once

// Words of a patch's block (thread t of a tile reads bit t % 32 of word t / 32: one word a
// warp): F at edge slots, q at triangle slots, div F, K and B at own nodes, q F^perp at own
// edges (o P^2 + i); a multiple of 16 bytes (a bulk copy).
template <int P>
struct TileValid {
    static constexpr int W = P + 3, NN = W * W, PP = P * P;
    static constexpr int F = 0, Q = F + (3 * NN + 31) / 32, N = Q + (2 * NN + 31) / 32, E = N + (PP + 31) / 32;
    static constexpr int WORDS = (E + (3 * PP + 31) / 32 + 3) / 4 * 4;
    static constexpr uint32_t BYTES = 4u * uint32_t(WORDS);
    static constexpr int SCRATCH = (NN + 31) / 32 + (3 * NN + 31) / 32;   // words a warp needs to build one
};

// the structured path applies: a regular tile of a level with tiles, inviscid and
// with the velocity free (the viscous and advection forms take the tabulated path)
template <class R>
__device__ __forceinline__ bool tile_regular(const DevLevelT<R>& L, int64_t pat) {
    return pat < L.npatch && L.thalo != nullptr && L.tirr[pat] == 0 && !viscous(L) && !L.advect;
}

// bits pos .. pos + 31 of the bits in w[0..n) (zero outside them)
__device__ __forceinline__ uint32_t bits_at(const uint32_t* w, int n, int pos) {
    const int i = pos >> 5;
    const uint32_t lo = unsigned(i) < unsigned(n) ? w[i] : 0u, hi = unsigned(i + 1) < unsigned(n) ? w[i + 1] : 0u;
    return __funnelshift_r(lo, hi, unsigned(pos) & 31u);
}

// The tile's node and edge slots lane, lane + 32, ...: own points as -(offset) - 1, halo
// points as their index in the halo table, other positions as NONE (as TilePlan); the same
// for every patch, kept in registers where they are few enough.
template <int P>
struct ValidPlan {
    using V = TileValid<P>;
    static constexpr int W = V::W, NN = V::NN, GN = (NN + 31) / 32, GE = (3 * NN + 31) / 32;
    static constexpr int NONE = -(1 << 30);
    __device__ static int node(int x) {
        const int a = x / W - 1, b = x % W - 1;
        return x >= NN ? NONE : (a >= 0 && a < P && b >= 0 && b < P) ? -(a * P + b) - 1 : tile::slot(P, P + 1, a, b);
    }
    __device__ static int edge(int y) {
        constexpr tile::Shape S{P};
        const int o = y / NN, x = y - o * NN, a = x / W - 1, b = x % W - 1;
        return (y >= 3 * NN || a > S.eA(o) || b > S.eB(o)) ? NONE
               : (a >= 0 && a < P && b >= 0 && b < P)      ? -(o * P * P + a * P + b) - 1
                                                           : S.off_edge(o) + tile::slot(P, S.eB(o), a, b);
    }
};

// patch `pat`'s block, by one warp (sh: SCRATCH words of its own; node(g), edge(g): the plan
// of this lane's slot of group g).  The flags are read with all their loads in flight, and
// the bits of F and q are combined a word a lane: at a slot's bit, its nodes' and edges'
// bits lie at constant offsets, and bits outside the tile's ranges are zero.
template <class R, int P, class Node, class Edge>
__device__ __forceinline__ void tile_valid_build(const DevLevelT<R>& L, int64_t pat, uint32_t* sh, Node node, Edge edge) {
    using V = TileValid<P>;
    using VP = ValidPlan<P>;
    constexpr tile::Shape S{P};
    constexpr int W = V::W, NN = V::NN, PP = V::PP, GN = VP::GN, GE = VP::GE, GL = (3 * PP + 31) / 32;
    constexpr int U = P <= 8 ? GE : 4;   // groups in flight
    const int lane = threadIdx.x & 31;
    const int32_t* __restrict__ halo = L.thalo + pat * S.halo();
    const int32_t nelem = int32_t(L.nelem), base = int32_t(pat) * PP;
    uint32_t* __restrict__ out = L.tvalid + pat * V::WORDS;
    uint32_t *nodes = sh, *edges = sh + GN;   // availability at node and edge slots
    __syncwarp();
#pragma unroll
    for (int g0 = 0; g0 < GN; g0 += U) {
        uint8_t f[U];
#pragma unroll
        for (int i = 0; i < U; ++i) {
            const int c = g0 + i < GN ? node(g0 + i) : VP::NONE;
            f[i] = c == VP::NONE ? 0 : L.nflag[c < 0 ? base + (-c - 1) : halo[c]];
        }
#pragma unroll
        for (int i = 0; i < U; ++i)
            if (g0 + i < GN) {
                const uint32_t m = __ballot_sync(0xffffffffu, (f[i] & AVAIL) != 0);
                if (lane == 0) nodes[g0 + i] = m;
            }
    }
#pragma unroll
    for (int g0 = 0; g0 < GE; g0 += U) {
        uint8_t f[U];
#pragma unroll
        for (int i = 0; i < U; ++i) {
            const int c = g0 + i < GE ? edge(g0 + i) : VP::NONE;
            int32_t e = 0;
            if (c >= 0) {
                e = halo[c] >> 1;
            } else if (c != VP::NONE) {
                const int k = -c - 1, o = k / PP;
                e = o * nelem + base + (k - o * PP);
            }
            f[i] = c == VP::NONE ? 0 : L.eflag[e];
        }
#pragma unroll
        for (int i = 0; i < U; ++i)
            if (g0 + i < GE) {
                const uint32_t m = __ballot_sync(0xffffffffu, (f[i] & AVAIL) != 0);
                if (lane == 0) edges[g0 + i] = m;
            }
    }
    uint8_t lf[GL];   // own edges
#pragma unroll
    for (int g = 0; g < GL; ++g) {
        const int w = g * 32 + lane, o = w / PP;
        lf[g] = w < 3 * PP ? L.eflag[o * nelem + base + (w - o * PP)] : 0;
    }
    __syncwarp();
    for (int g = lane; g < V::Q - V::F; g += 32) {
        uint32_t m = 0u;
#pragma unroll
        for (int o = 0; o < 3; ++o) {
            const int x = g * 32 - o * NN;
            m |= bits_at(nodes, GN, x) & bits_at(nodes, GN, x + (o == 0 ? W : o == 1 ? W + 1 : 1));
        }
        out[V::F + g] = m & edges[g];
    }
    for (int g = lane; g < V::N - V::Q; g += 32) {
        uint32_t m = 0u;
#pragma unroll
        for (int t = 0; t < 2; ++t) {
            const int x = g * 32 - t * NN;
            // vertices and sides as in tile_trend
            const int n1 = t == 0 ? x + W : x + W + 1, n2 = t == 0 ? x + W + 1 : x + 1;
            const int s0 = t == 0 ? x : NN + x, s1 = t == 0 ? 2 * NN + x + W : x + 1, s2 = t == 0 ? NN + x : 2 * NN + x;
            m |= bits_at(nodes, GN, x) & bits_at(nodes, GN, n1) & bits_at(nodes, GN, n2) & bits_at(edges, GE, s0) &
                 bits_at(edges, GE, s1) & bits_at(edges, GE, s2);
        }
        out[V::Q + g] = m;
    }
#pragma unroll
    for (int g = 0; g < V::E - V::N; ++g) {
        const int i = g * 32 + lane, x = (i / P + 1) * W + i % P + 1;
        auto get = [&](const uint32_t* w, int k) { return w[k >> 5] >> (k & 31); };
        uint32_t ok = 0u;
        if (i < PP)   // the node and its ring: its own edges, and those coming in
            ok = get(nodes, x) & get(edges, x) & get(edges, NN + x) & get(edges, 2 * NN + x) & get(edges, x - W) &
                 get(edges, NN + x - W - 1) & get(edges, 2 * NN + x - 1);
        const uint32_t m = __ballot_sync(0xffffffffu, ok & 1u);
        if (lane == 0) out[V::N + g] = m;
    }
#pragma unroll
    for (int g = 0; g < GL; ++g) {
        const uint32_t m = __ballot_sync(0xffffffffu, (lf[g] & LIVE) != 0);
        if (lane == 0) out[V::E + g] = m;
    }
}

// the blocks of the regular patches of a core list, a warp an entry (sh: SCRATCH words of
// patch side P for each warp of the block)
template <class R, int P>
__device__ __forceinline__ void tile_valid_entries(const DevLevelT<R>* __restrict__ lvs, const int32_t* __restrict__ list,
                                                   int count, int w, int nw, uint32_t* sh) {
    using VP = ValidPlan<P>;
    const int lane = threadIdx.x & 31;
    uint32_t* own = sh + (threadIdx.x >> 5) * TileValid<P>::SCRATCH;
    if constexpr (P <= 8) {
        int n[VP::GN], e[VP::GE];
#pragma unroll
        for (int g = 0; g < VP::GN; ++g) n[g] = VP::node(g * 32 + lane);
#pragma unroll
        for (int g = 0; g < VP::GE; ++g) e[g] = VP::edge(g * 32 + lane);
        for (int t = w; t < count; t += nw) {
            const int32_t ent = list[t];
            const DevLevelT<R>& L = lvs[ent >> LVL_SHIFT];
            if (tile_regular(L, int64_t(ent & PATCH_MASK)))
                tile_valid_build<R, P>(L, int64_t(ent & PATCH_MASK), own, [&](int g) { return n[g]; },
                                       [&](int g) { return e[g]; });
        }
    } else {
        for (int t = w; t < count; t += nw) {
            const int32_t ent = list[t];
            const DevLevelT<R>& L = lvs[ent >> LVL_SHIFT];
            if (tile_regular(L, int64_t(ent & PATCH_MASK)))
                tile_valid_build<R, P>(L, int64_t(ent & PATCH_MASK), own, [&](int g) { return VP::node(g * 32 + lane); },
                                       [&](int g) { return VP::edge(g * 32 + lane); });
        }
    }
}
// resident blocks of 256 threads per SM the builder is built for (its plan and the flags
// in flight take up to 80 registers)
template <int P>
constexpr int valid_blocks() { return P <= 8 ? 3 : 2; }

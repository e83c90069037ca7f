// Persistent RK stage: one cooperative launch runs every phase of a trend
// evaluation and its stage update (Sec. 3.1), the phases separated by grid
// barriers instead of kernel boundaries:
//
//   ghosts of levels Jmin+1..top (coarse to fine, one phase per level)
//   -> the trend of every active patch: the structured tile of a regular patch
//      (F, q, div F, K, B, q F^perp), F and q from the tabulated bodies elsewhere
//   -> div, K, B and q F^perp at the points of the irregular patches
//   -> restriction of B, F, q F^perp and div, top-1 down to Jmin (two phases a level)
//   -> RK stage update of the live points (all levels)
//
// One block of 512 threads per SM, up to 128 registers a thread (with 1024 threads of 64
// the ids read ahead spill: 75 us a stage instead of 69 on the jet below in FP32, 118
// instead of 101 in FP64).  The phases of a small grid are bound by latency: a barrier,
// then a chain of dependent gathers.  So the level-serial phases run over the point work
// lists (their lengths staged once per block) with the ids of each thread's first item
// read ahead while its block waits (ListPhase); consecutive warps of a list go to
// different SMs, which also spreads the FP64 work (the FP64 pipe starts one warp
// instruction per 16 clocks and SM); and the block's teams (Team) each work on a patch
// of their own in the trend.  On the jet of 23 400 live cells on five levels a stage took
// 206 us (FP64) and 134 us (FP32) with the patches' items dealt out in whole blocks, one
// patch per block at a time and a barrier of 304 blocks; 101 and 69 us now.  The barrier
// itself costs 1.4 us.
//
// Values written by other blocks in one phase are read in the next: the barrier's
// release and acquire at GPU scope, between two block barriers, order them (the acquire
// also drops the SM's stale L1 lines), so loads may use L1, where the gathers of
// neighbouring items meet (with L1 bypassed a stage of that jet took 3 to 5 % longer).
//
// Every barrier wait is bounded: after about two seconds a block sets the error flag and
// the kernel returns; so does the wait for a patch's geometry block (a bulk copy).
#include <cuda_runtime.h>

#include <algorithm>
#include <cstdint>

#include "sww_core.cuh"
#include "sww_kernels.h"
#include "sww_stage.h"
#include "tile.h"

namespace sww {

namespace {

#include "bulk.cuh"
#include "sww_bodies.cuh"
#include "sww_tile.cuh"

constexpr int STAGE_TPB = 512;
constexpr int MAXL = 12;
constexpr long long SPIN_CYCLES = 4000000000ll;   // ~2 s at 2 GHz

// threads of one team of the trend: a tile's 4 p^2 own points, and teams that fit
// the block's shared memory
template <class R, int P>
struct Teams {
    static constexpr int NT = P == 4 ? 128 : P == 8 ? 256 : 512;
    static constexpr size_t FIT = (227 * 1024 - 12 * 1024) / Tile<R, P>::BYTES;   // 12 KB: the level records
    static constexpr int N = FIT < size_t(STAGE_TPB / NT) ? int(FIT) : STAGE_TPB / NT;
    static_assert(N >= 1 && N < 16, "named barriers 1..15");
};

__device__ __forceinline__ unsigned ld_acquire(const unsigned* p) {
    unsigned v;
    asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}
__device__ __forceinline__ void red_release(unsigned* p) {
    asm volatile("red.release.gpu.global.add.u32 [%0], 1;" ::"l"(p) : "memory");
}

// Grid-wide barrier of the cooperative launch.  bar[0] counts arrivals and is never
// reset; bar[BASE] holds its value when the launch began (written by the launch before
// it, at its end), so the n-th barrier of a launch is complete when the count has
// reached base + n * blocks, in arithmetic modulo 2^32.  One counter: the arrivals
// need no answer, so a barrier costs one trip to the L2 and the polls (a two-level
// barrier with its two dependent atomics and sleeping waits took about 2 us longer).
struct GridBarrier {
    static constexpr int BASE = 32;
    unsigned* bar;
    int* err;
    long long limit;
    int skip;
    unsigned target;

    bool left = false;   // thread 0 of a block that did not arrive

    // The block arrives (its writes of the phase before are released).  Between arriving and
    // waiting a thread may read what does not change during a stage.
    __device__ void arrive() {
        __syncthreads();
        if (threadIdx.x == 0) {
            if (int(blockIdx.x) == skip) {
                left = true;
            } else {
                __threadfence();
                red_release(bar);
                target += gridDim.x;
            }
        }
    }

    // waits for all blocks: false, for every thread of the block, when the wait timed out
    // (after `limit` cycles; the error flag is set), another block has reported an error,
    // or the block is the one told to leave without arriving (fault injection).  A block
    // that leaves arrives nowhere again, so no block passes a later barrier.
    __device__ bool wait() {
        bool ok = true;
        if (threadIdx.x == 0) {
            if (left) {
                ok = false;
            } else {
                const long long t0 = clock64();
                unsigned polls = 0;
                while (int(ld_acquire(bar) - target) < 0) {
                    if ((++polls & 15u) == 0 && *reinterpret_cast<volatile int*>(err)) {
                        ok = false;
                        break;
                    }
                    if (clock64() - t0 > limit) {
                        atomicExch(err, 1);
                        ok = false;
                        break;
                    }
                }
                __threadfence();
            }
        }
        return __syncthreads_and(ok);
    }
    __device__ bool sync() {
        arrive();
        return wait();
    }
};

// This thread's first item of a phase: consecutive warps of items go to consecutive
// blocks, so that a short list reaches every SM.  The next item is gridDim.x *
// blockDim.x further on.
__device__ __forceinline__ int first_item() {
    return int(((threadIdx.x >> 5) * gridDim.x + blockIdx.x) * 32 + (threadIdx.x & 31));
}

// One level-serial phase over work lists k0 and (k1 >= 0) k1 of level L, item i < n0 of
// the first, then the second; a thread's first item is read ahead of the phase: its id and
// the ids it gathers through (lists, tables and flags do not change during a stage), between
// the block's arrival at the barrier before the phase and its wait.  Then the phase is one
// round of gathers instead of three or four rounds of dependent loads.  Items further on
// (grids beyond one item a thread) take the general bodies, whose arithmetic is the same.
template <class R>
struct ListPhase {
    const DevLevelT<R>* L = nullptr;
    int n0 = 0, n1 = 0, k0 = 0, k1 = -1;
    // read ahead (by the phase's own functions below)
    int32_t id = -1, a = 0, b = 0, s[24];
    uint32_t f = 0;

    __device__ __forceinline__ int32_t load(int i) const {
        return i < n0 ? L->wl[wl_off(*L, k0) + i] : L->wl[wl_off(*L, k1) + (i - n0)];
    }
    __device__ __forceinline__ bool first(const DevLevelT<R>& lev, const int (&cnt)[MAXL][WL_KINDS], int j, int ka, int kb) {
        L = &lev, k0 = ka, k1 = kb;
        n0 = cnt[j][ka], n1 = kb >= 0 ? cnt[j][kb] : 0;
        const int i = first_item();
        id = i < n0 + n1 ? load(i) : -1;
        return i < n0;
    }
    // the items after the thread's first
    template <class Body>
    __device__ __forceinline__ void rest(Body body) const {
        const int stride = int(gridDim.x * blockDim.x);
        for (int i = first_item() + stride; i < n0 + n1; i += stride) body(i < n0 ? 0 : 1, int64_t(load(i)));
    }

    // ---- ghosts of L (WL_GN, WL_GE) from C, as fill_node and fill_edge
    __device__ __forceinline__ void ahead_fill(const DevLevelT<R>& F, const int (&cnt)[MAXL][WL_KINDS], int j) {
        const bool node = first(F, cnt, j, WL_GN, WL_GE);
        if (id < 0) return;
        f = 0u;
        if (node) {
            a = F.f2c[id];
            if (a >= 0) return;
#pragma unroll
            for (int q = 0; q < 4; ++q) s[q] = F.par[q * F.N + id];
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                s[4 + q] = F.f2c[s[q]];
                if (F.nflag[s[q]] & LIVE) f |= 1u << q;
            }
        } else {
            a = F.fe_ot[id], b = F.fe_ce[id];
#pragma unroll
            for (int k = 0; k < 12; ++k) s[k] = F.vst[k * F.E + id];
            if (a >= 0) {
                f = F.eflag[a];
#pragma unroll
                for (int k = 0; k < 12; ++k) s[12 + k] = F.vst[k * F.E + a];
            }
        }
    }
    __device__ __forceinline__ void run_fill(const DevLevelT<R>& F, const DevLevelT<R>& C) {
        if (id >= 0 && first_item() < n0) {
            if (a >= 0) {
                F.dh[id] = C.dh[a];
            } else {
                R w[4], v[4];
#pragma unroll
                for (int q = 0; q < 4; ++q) w[q] = F.ptw[q * F.N + id], v[q] = (f >> q & 1u) ? F.dh[s[q]] : C.dh[s[4 + q]];
                R sum = R(0);
#pragma unroll
                for (int q = 0; q < 4; ++q) sum += w[q] * v[q];
                F.dh[id] = sum;
            }
        } else if (id >= 0 && !F.advect) {
            const R P = predict_from(F, C.u, id, s);
            if (a < 0) {
                F.u[id] = P;
            } else {
                const R uc = C.u[b];
                if (f & LIVE) {
                    F.u[id] = R(2) * uc - F.u[a];
                } else {
                    const R Po = predict_from(F, C.u, a, s + 12);
                    F.u[id] = half_value(P, Po, uc);
                    if (f & GHOST) F.u[a] = half_value(Po, P, uc);
                }
            }
        }
        rest([&](int k, int64_t x) {
            if (k == 0)
                fill_node(F, C, x);
            else
                fill_edge(F, C, x);
        });
    }

    // ---- restriction to L (WL_CN, WL_RE) from F, as restrict_node and restrict_edge
    __device__ __forceinline__ void ahead_restrict(const DevLevelT<R>& C, const int (&cnt)[MAXL][WL_KINDS], int j) {
        const bool node = first(C, cnt, j, WL_CN, WL_RE);
        if (id < 0) return;
        if (node) {
            a = C.c2f[id];
        } else {
            const int32_t na = C.en[id], nb = C.en[C.E + id];
#pragma unroll
            for (int k = 0; k < 12; ++k) s[k] = C.rf_fi[k * C.E + id];
#pragma unroll
            for (int k = 0; k < 11; ++k) s[12 + k] = C.rf_ci[k * C.E + id];
            a = C.half[id], b = C.half[C.E + id];
            f = C.nflag[na] & C.nflag[nb];
        }
    }
    __device__ __forceinline__ void run_restrict(const DevLevelT<R>& C, const DevLevelT<R>& F) {
        if (id >= 0 && first_item() < n0) {
            if (!C.advect) C.B[id] = F.B[a];
        } else if (id >= 0) {
            const bool visc = viscous(C);
            R sum = R(0);
#pragma unroll
            for (int k = 0; k < 12; ++k) sum += C.rf_fw[k * C.E + id] * (visc ? F.F[s[k]] + F.Fd[s[k]] : F.F[s[k]]);
#pragma unroll
            for (int k = 0; k < 11; ++k) sum += C.rf_cw[k * C.E + id] * F.c[s[12 + k]];
            C.F[id] = sum / geo<R>(C.l_e, id);
            if (visc) C.Fd[id] = R(0);
            if ((f & COVERED) && !C.advect) C.Q[id] = R(0.5) * (F.Q[a] + F.Q[b]);
        }
        rest([&](int k, int64_t x) {
            if (k == 0)
                restrict_node(C, F, x);
            else
                restrict_edge(C, F, x);
        });
    }

    // ---- divergence of the restricted fluxes of L (WL_DN), as div_at
    __device__ __forceinline__ void ahead_div(const DevLevelT<R>& C, const int (&cnt)[MAXL][WL_KINDS], int j) {
        first(C, cnt, j, WL_DN, -1);
        if (id < 0) return;
        const uint8_t fv = C.nflag[id];
        a = C.deg[id];
#pragma unroll
        for (int k = 0; k < 6; ++k) s[k] = C.ring_e[k * C.N + id];
        uint8_t ok = 0xff;
#pragma unroll
        for (int k = 0; k < 6; ++k)
            if (k < a) ok = (C.eflag[s[k] >> 1] & AVAIL) ? ok : 0;
        f = (fv & AVAIL) ? ok : 0;
    }
    __device__ __forceinline__ void run_div(const DevLevelT<R>& C) {
        if (id >= 0 && f) {
            const bool visc = viscous(C);
            R F[6];
            double le[6];
#pragma unroll
            for (int k = 0; k < 6; ++k) {
                const int64_t e = s[k] < 0 ? 0 : s[k] >> 1;   // slot 5 of a pentagon: -1, not used
                F[k] = C.F[e], le[k] = C.l_e[e];
                if (visc) F[k] = F[k] + C.Fd[e];
            }
            const double A = C.A_i[id];
            R div = R(0);
#pragma unroll
            for (int k = 0; k < 6; ++k)
                if (k < a) div += esign<R>(s[k]) * F[k] * to_r<R>(le[k]);
            C.c[id] = div / to_r<R>(A);
        }
        rest([&](int, int64_t x) { div_at(C, x); });
    }
};

// items of `count` entries of `list` (NS slots of P items an entry): body(entry, item)
template <class Body>
__device__ __forceinline__ void entry_items(const int32_t* __restrict__ list, int count, uint32_t NS, int P, Body body) {
    const int lp = __ffs(P) - 1;
    const uint32_t n = uint32_t(count) * (NS << lp);
    for (uint32_t it = uint32_t(first_item()); it < n; it += gridDim.x * blockDim.x) {
        const uint32_t e = (it >> lp) / NS;
        body(list[e], it - ((e * NS) << lp));
    }
}

template <class R, int P>
__global__ void __launch_bounds__(STAGE_TPB, 1) k_stage(const __grid_constant__ StageArgs<R> a) {
    extern __shared__ __align__(16) unsigned char smem[];
    __shared__ DevLevelT<R> sl[MAXL];
    __shared__ int cnt[MAXL][WL_KINDS];
    __shared__ LiveItems live;
    __shared__ int n_core, n_irr, start_ok;
    __shared__ unsigned start_base;
    {
        const int words = int((a.jmax + 1) * sizeof(DevLevelT<R>) / sizeof(int));
        const int* src = reinterpret_cast<const int*>(a.lvs);
        int* dst = reinterpret_cast<int*>(sl);
        for (int k = threadIdx.x; k < words; k += blockDim.x) dst[k] = src[k];
        if (threadIdx.x == 0) {
            // a launch that follows a failed one leaves at once (its barrier count is stale)
            start_ok = *reinterpret_cast<volatile int*>(a.err) == 0;
            start_base = a.bar[GridBarrier::BASE];
            n_core = a.lists.count[1], n_irr = a.lists.count[2];
        }
        __syncthreads();
        if (!start_ok) return;
        live.init(sl, a.jmin, a.jtop);
        for (int k = threadIdx.x; k < (a.jtop + 1) * WL_KINDS; k += blockDim.x)
            if (k / WL_KINDS >= a.jmin) cnt[k / WL_KINDS][k % WL_KINDS] = sl[k / WL_KINDS].wl_n[k % WL_KINDS];
        __syncthreads();
    }
    const long long limit = a.spin > 0 ? a.spin : SPIN_CYCLES;
    GridBarrier gb{a.bar, a.err, limit, a.skip, start_base};
    const DevLevelT<R>* lv = sl;
    const R H = a.H, g = a.g;
    ListPhase<R> ph;
    // ghosts, coarse to fine
    if (a.jtop > a.jmin) ph.ahead_fill(lv[a.jmin + 1], cnt, a.jmin + 1);
    for (int j = a.jmin + 1; j <= a.jtop; ++j) {
        ph.run_fill(lv[j], lv[j - 1]);
        gb.arrive();
        if (j < a.jtop) ph.ahead_fill(lv[j + 1], cnt, j + 1);
        if (!gb.wait()) return;
    }
    // the trend: the irregular patches' F and q one thread an item, then a regular patch
    // a team at a time (patches dealt out over the SMs first)
    entry_items(a.lists.irr, n_irr, 5, a.P, [&](int32_t ent, uint32_t local) {
        irregular_fq(lv[ent >> LVL_SHIFT], int64_t(ent & PATCH_MASK), local, a.P, H);
    });
    {
        using TM = Teams<R, P>;
        const int team = int(threadIdx.x) / TM::NT;
        bool ok = true;
        if (team < TM::N)
            ok = tile_sweep<R, P, TM::NT>(Team<TM::NT>{int(threadIdx.x) % TM::NT, unsigned(team + 1)}, lv, a.lists.core, n_core,
                                          int(team * gridDim.x + blockIdx.x), int(TM::N * gridDim.x), H, g,
                                          smem + team * Tile<R, P>::BYTES, a.err, limit);
        if (!__syncthreads_and(ok)) return;
    }
    if (!gb.sync()) return;
    entry_items(a.lists.irr, n_irr, 4, a.P, [&](int32_t ent, uint32_t local) {
        auto body = [&](const DevLevelT<R>& L, int kind, int64_t id, int64_t) {
            if (kind == K_NODE)
                node_at(L, id, g);
            else
                coriolis_at(L, id);
        };
        visit_item<K_NODE | K_EDGE>(lv[ent >> LVL_SHIFT], int64_t(ent & PATCH_MASK), local, a.P, body);
    });
    // restriction, fine to coarse; then the update
    gb.arrive();
    if (a.jtop > a.jmin) ph.ahead_restrict(lv[a.jtop - 1], cnt, a.jtop - 1);
    if (!gb.wait()) return;
    for (int j = a.jtop - 1; j >= a.jmin; --j) {
        ph.run_restrict(lv[j], lv[j + 1]);
        gb.arrive();
        ph.ahead_div(lv[j], cnt, j);
        if (!gb.wait()) return;
        ph.run_div(lv[j]);
        gb.arrive();
        if (j > a.jmin) ph.ahead_restrict(lv[j - 1], cnt, j - 1);
        if (!gb.wait()) return;
    }
    // every block has read the barrier's base: the next launch's is this one's last target
    if (blockIdx.x == 0 && threadIdx.x == 0) a.bar[GridBarrier::BASE] = gb.target;
    const R dt = to_r<R>(a.dt ? *a.dt : 0.0);
    live.run(lv, a.jmin, a.jtop, first_item(), int(gridDim.x * blockDim.x), [&](const DevLevelT<R>& L, int kind, int64_t id) {
        if (kind == K_NODE)
            update_node(L, id, a.st, dt);
        else
            update_edge(L, id, a.st, dt);
    });
}

template <class R, int P>
unsigned stage_grid_p(int nsm) {
    constexpr size_t smem = Teams<R, P>::N * Tile<R, P>::BYTES;
    // the dynamic tile and the static level records together may pass the default
    // 48 KB: the dynamic size is always declared
    if (cudaFuncSetAttribute(k_stage<R, P>, cudaFuncAttributeMaxDynamicSharedMemorySize, int(smem)) != cudaSuccess)
        return 0;
    int per_sm = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_stage<R, P>, STAGE_TPB, smem) != cudaSuccess) return 0;
    return unsigned(std::max(per_sm, 0) * nsm);
}

template <class R, int P>
cudaError_t launch_stage_p(const StageArgs<R>& a, unsigned grid, cudaStream_t s) {
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3(grid);
    cfg.blockDim = dim3(STAGE_TPB);
    cfg.dynamicSmemBytes = Teams<R, P>::N * Tile<R, P>::BYTES;
    cfg.stream = s;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeCooperative;
    attr[0].val.cooperative = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    count_launch(1);
    return cudaLaunchKernelEx(&cfg, k_stage<R, P>, a);
}

}  // namespace

// patch area -> tile side of the stage kernel (sides 1 and 2 have no regular tile)
template <class R>
unsigned stage_grid(int P, int nsm) {
    return P == 64 ? stage_grid_p<R, 8>(nsm) : P == 256 ? stage_grid_p<R, 16>(nsm) : stage_grid_p<R, 4>(nsm);
}

template <class R>
cudaError_t launch_stage(const StageArgs<R>& a, unsigned grid, cudaStream_t s) {
    if (a.jmax + 1 > MAXL) return cudaErrorInvalidValue;
    return a.P == 64 ? launch_stage_p<R, 8>(a, grid, s) : a.P == 256 ? launch_stage_p<R, 16>(a, grid, s)
                                                                    : launch_stage_p<R, 4>(a, grid, s);
}

template unsigned stage_grid<double>(int, int);
template unsigned stage_grid<float>(int, int);
template cudaError_t launch_stage<double>(const StageArgs<double>&, unsigned, cudaStream_t);
template cudaError_t launch_stage<float>(const StageArgs<float>&, unsigned, cudaStream_t);

}  // namespace sww

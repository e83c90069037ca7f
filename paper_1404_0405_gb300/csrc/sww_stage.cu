// Persistent step: one cooperative launch runs the time step, every stage's trend and
// update (Sec. 3.1), the partial transform and the coefficients of a step, another its
// inverse transform, their phases separated by grid barriers instead of kernel boundaries:
//
//   the largest frequency and velocities of the live points, the time step from them
//   per stage: ghosts of levels Jmin+1..top (coarse to fine, one phase per level)
//   -> the trend of every active patch: the structured tile of a regular patch
//      (F, q, div F, K, B, q F^perp), F and q from the tabulated bodies elsewhere
//   -> div, K, B and q F^perp at the points of the irregular patches
//   -> restriction of B, F, q F^perp and div, top-1 down to Jmin (two phases a level)
//   -> RK stage update of the live points (all levels)
//   then the partial transform top-1 down to Jmin, the ghosts, the coefficients with the
//   live maxima, the thresholds.
//
// A trend evaluation alone is one stage of the same kernel.  A step of the jet with 21 550
// live cells on five levels takes 950 us (FP64) and 577 us (FP32) as a launch per phase,
// 720 and 504 so.
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
// patch per block at a time and a barrier of 304 blocks; 101 and 69 us so.  The barrier
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
    unsigned* target;   // shared memory, thread 0's
    bool* left;         // thread 0 of a block that did not arrive

    // The block arrives (its writes of the phase before are released).  Between arriving and
    // waiting a thread may read what does not change during a stage.
    __device__ void arrive() {
        __syncthreads();
        if (threadIdx.x == 0) {
            if (int(blockIdx.x) == skip) {
                *left = true;
            } else {
                __threadfence();
                red_release(bar);
                *target += gridDim.x;
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
            if (*left) {
                ok = false;
            } else {
                const long long t0 = clock64();
                const unsigned want = *target;
                unsigned polls = 0;
                while (int(ld_acquire(bar) - want) < 0) {
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

// One level-serial phase over work lists k0 and (k1 >= 0) k1 of level L, one after the
// other; a thread's first item is read ahead of the phase: its id and
// the ids it gathers through (lists, tables and flags do not change during a stage), between
// the block's arrival at the barrier before the phase and its wait.  Then the phase is one
// round of gathers instead of three or four rounds of dependent loads.  Items further on
// (grids beyond one item a thread) take the general bodies, whose arithmetic is the same.
template <class R>
struct ListPhase {
    const DevLevelT<R>* L = nullptr;
    int n0 = 0, n1 = 0, k0 = 0, k1 = -1;
    // read ahead (by the phase's own functions below)
    int32_t id = -1, a = 0, b = 0, s[24] = {};
    uint32_t f = 0;

    // what was read ahead before is dead (held through the trend otherwise)
    __device__ __forceinline__ void reset() { *this = ListPhase(); }

    // list (0, 1) of item i
    __device__ __forceinline__ int list_of(int i) const { return i < n0 ? 0 : 1; }
    __device__ __forceinline__ int32_t load(int i) const {
        return i < n0 ? L->wl[wl_off(*L, k0) + i] : L->wl[wl_off(*L, k1) + (i - n0)];
    }
    __device__ __forceinline__ int first(const DevLevelT<R>& lev, const int (&cnt)[MAXL][WL_KINDS], int j, int ka, int kb) {
        reset();
        L = &lev, k0 = ka, k1 = kb;
        n0 = cnt[j][ka], n1 = kb >= 0 ? cnt[j][kb] : 0;
        const int i = first_item();
        id = i < n0 + n1 ? load(i) : -1;
        return list_of(i);
    }
    // the items after the thread's first
    template <class Body>
    __device__ __forceinline__ void rest(Body body) const {
        const int stride = int(gridDim.x * blockDim.x);
        for (int i = first_item() + stride; i < n0 + n1; i += stride) body(list_of(i), int64_t(load(i)));
    }

    // ---- ghosts of L (WL_GN, WL_GE) from C, as fill_node and fill_edge
    // the stencil ids of fine edge e into s[at..at + 11]
    __device__ __forceinline__ void stencil(const DevLevelT<R>& F, int64_t e, int at) {
#pragma unroll
        for (int k = 0; k < 12; ++k) s[at + k] = F.vst[k * F.E + e];
    }
    __device__ __forceinline__ void ahead_fill(const DevLevelT<R>& F, const int (&cnt)[MAXL][WL_KINDS], int j) {
        const int k = first(F, cnt, j, WL_GN, WL_GE);
        if (id < 0) return;
        if (k == 0) {
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
            stencil(F, id, 0);
            if (a >= 0) {
                f = F.eflag[a];
                stencil(F, a, 12);
            }
        }
    }
    __device__ __forceinline__ void run_fill(const DevLevelT<R>& F, const DevLevelT<R>& C) {
        const int k = list_of(first_item());
        if (id >= 0 && k == 0) {
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
        } else if (id >= 0 && k == 1 && !F.advect) {
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

    // ---- inverse transform at the live points of L (WL_LN, WL_LE) from C, as inverse_a_item
    __device__ __forceinline__ void ahead_inverse(const DevLevelT<R>& F, const DevLevelT<R>& C, const int (&cnt)[MAXL][WL_KINDS],
                                                  int j) {
        const int k = first(F, cnt, j, WL_LN, WL_LE);
        if (id < 0) return;
        if (k == 0) {
            a = F.f2c[id];
            if (a < 0) return;
#pragma unroll
            for (int q = 0; q < 12; ++q) {
                const int32_t m = C.mk_i[q * C.N + a];
                s[q] = m < 0 ? 0 : m;   // padded with -1 at the pentagons
                f |= m < 0 ? 0u : 1u << q;
            }
            uint8_t fl[12];
#pragma unroll
            for (int q = 0; q < 12; ++q) fl[q] = F.nflag[s[q]];
#pragma unroll
            for (int q = 0; q < 12; ++q)
                if ((fl[q] & (LIVE | WASLIVE)) != (LIVE | WASLIVE)) f &= ~(1u << q);
        } else if (!F.advect) {
            a = F.fe_ot[id], b = F.fe_ce[id];
            f = F.eflag[id] | (uint32_t(F.fe_kind[id]) << 16);
            stencil(F, id, 0);
            if (a >= 0) {
                f |= uint32_t(F.eflag[a]) << 8;
                stencil(F, a, 12);
            }
        }
    }
    __device__ __forceinline__ void run_inverse(const DevLevelT<R>& F, const DevLevelT<R>& C) {
        const int k = list_of(first_item());
        if (id >= 0 && k == 0 && a >= 0) {
            R w[12], d[12];
#pragma unroll
            for (int q = 0; q < 12; ++q) w[q] = C.mk_w[q * C.N + a], d[q] = F.hdet[s[q]];
            R sum = C.dh[a];
#pragma unroll
            for (int q = 0; q < 12; ++q)
                if (f >> q & 1u) sum -= w[q] * d[q];
            F.dh[id] = sum;
        } else if (id >= 0 && k == 1 && !F.advect) {
            if (a < 0) {
                const R Pr = predict_from(F, C.u, id, s), d = F.ui[id];
                F.u[id] = Pr + ((f & WASLIVE) ? d : R(0));
            } else {
                const uint32_t fo = f >> 8 & 0xffu, kind = f >> 16;
                // the first half's item writes both when both are live
                if (!((kind == 1) & ((fo & LIVE) != 0))) {
                    const R Pr = predict_from(F, C.u, id, s), Po = predict_from(F, C.u, a, s + 12);
                    const R uc = C.u[b], de = F.ue[b];
                    const R d = ((f | fo) & WASLIVE) ? de : R(0);
                    {
                        const R delta = R(0.5) * (R(2) * uc - Pr - Po);
                        F.u[id] = Pr + delta + (kind == 0 ? d : -d);
                    }
                    if (fo & LIVE) {
                        const R delta = R(0.5) * (R(2) * uc - Po - Pr);
                        F.u[a] = Po + delta - d;
                    }
                }
            }
        }
        rest([&](int k, int64_t x) { inverse_a_item(F, C, k == 0 ? K_NODE : K_EDGE, x); });
    }

    // ---- its odd nodes from the even ones (WL_LN), as inverse_b_item
    __device__ __forceinline__ void ahead_odd(const DevLevelT<R>& F, const int (&cnt)[MAXL][WL_KINDS], int j) {
        first(F, cnt, j, WL_LN, -1);
    }
    __device__ __forceinline__ void run_odd(const DevLevelT<R>& F) {
        if (id >= 0) inverse_b_item(F, id);
        rest([&](int, int64_t x) { inverse_b_item(F, x); });
    }

    // ---- restriction to L (WL_CN, WL_RE) from F, as restrict_node and restrict_edge
    __device__ __forceinline__ void ahead_restrict(const DevLevelT<R>& C, const int (&cnt)[MAXL][WL_KINDS], int j) {
        const int k = first(C, cnt, j, WL_CN, WL_RE);
        if (id < 0) return;
        if (k == 0) {
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

    // ---- partial transform at the covered nodes of L (WL_CN) from F
    __device__ __forceinline__ void ahead_partial(const DevLevelT<R>& C, const int (&cnt)[MAXL][WL_KINDS], int j) {
        first(C, cnt, j, WL_CN, -1);
    }
    __device__ __forceinline__ void run_partial(const DevLevelT<R>& C, const DevLevelT<R>& F) {
        if (id >= 0) partial_node(C, F, id);
        rest([&](int, int64_t x) { partial_node(C, F, x); });
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

// What a block keeps in shared memory: the level records, the work lists' lengths, the
// live points' offsets, and the barrier's state (thread 0's).
template <class R>
struct BlockState {
    DevLevelT<R> sl[MAXL];
    int cnt[MAXL][WL_KINDS];
    LiveItems live;
    int n_core, n_irr, start_ok;
    unsigned target;
    bool left;

    // by the whole block; false when a launch before this one failed (its barrier count is
    // stale): the block leaves at once
    __device__ __forceinline__ bool init(const StageArgs<R>& a) {
        const int words = int((a.jmax + 1) * sizeof(DevLevelT<R>) / sizeof(int));
        const int* src = reinterpret_cast<const int*>(a.lvs);
        int* dst = reinterpret_cast<int*>(sl);
        for (int k = threadIdx.x; k < words; k += blockDim.x) dst[k] = src[k];
        if (threadIdx.x == 0) {
            start_ok = *reinterpret_cast<volatile int*>(a.err) == 0;
            target = a.bar[GridBarrier::BASE], left = false;
            n_core = a.lists.count[1], n_irr = a.lists.count[2];
        }
        __syncthreads();
        if (!start_ok) return false;
        live.init(sl, a.jmin, a.jtop);
        for (int k = threadIdx.x; k < (a.jtop + 1) * WL_KINDS; k += blockDim.x)
            if (k / WL_KINDS >= a.jmin) cnt[k / WL_KINDS][k % WL_KINDS] = sl[k / WL_KINDS].wl_n[k % WL_KINDS];
        __syncthreads();
        return true;
    }
    __device__ __forceinline__ GridBarrier barrier(const StageArgs<R>& a) {
        return GridBarrier{a.bar, a.err, a.spin > 0 ? a.spin : SPIN_CYCLES, a.skip, &target, &left};
    }
    // after the block's last wait: the next launch's count begins at this one's last target
    // (every block has read the base)
    __device__ __forceinline__ void done(const StageArgs<R>& a) const {
        if (blockIdx.x == 0 && threadIdx.x == 0) a.bar[GridBarrier::BASE] = target;
    }
};

template <class R, int P>
__global__ void __launch_bounds__(STAGE_TPB, 1) k_stage(const __grid_constant__ StageArgs<R> a) {
    extern __shared__ __align__(16) unsigned char smem[];
    __shared__ BlockState<R> bs;
    __shared__ unsigned long long sh[STAGE_TPB / 32], slev[RED_WORDS - RED_LEVEL];
    __shared__ double dt_s;
    if (!bs.init(a)) return;
    const auto& cnt = bs.cnt;
    const LiveItems& live = bs.live;
    GridBarrier gb = bs.barrier(a);
    const DevLevelT<R>* lv = bs.sl;
    const R H = a.H, g = a.g;
    // the time step: every block takes it from the grid's maxima; block 0 keeps it
    if (a.pre == 1) {
        cfl_maxima(live, lv, a.jmin, a.jtop, first_item(), int(gridDim.x * blockDim.x), a.Hd, a.gd, a.red, sh, slev);
        if (!gb.sync()) return;
        if (threadIdx.x < 32) {
            const double d = cfl_step<R>(lv, a.red, a.cfl);
            if (threadIdx.x == 0) dt_s = d;
        }
    } else if (threadIdx.x == 0) {
        dt_s = a.pre == 2 ? a.dt_given : a.dt ? *a.dt : 0.0;
    }
    __syncthreads();
    if (a.pre && blockIdx.x == 0 && threadIdx.x == 0) *a.dt = dt_s;
    ListPhase<R> ph;
    // the ghosts, coarse to fine (the first level's ids read ahead); the barrier after the
    // last level unless `open`
    auto ghosts = [&](bool open) -> bool {
        for (int j = a.jmin + 1; j <= a.jtop; ++j) {
            ph.run_fill(lv[j], lv[j - 1]);
            if (open && j == a.jtop) return true;
            gb.arrive();
            if (j < a.jtop) ph.ahead_fill(lv[j + 1], cnt, j + 1);
            if (!gb.wait()) return false;
        }
        return true;
    };
    if (a.jtop > a.jmin) ph.ahead_fill(lv[a.jmin + 1], cnt, a.jmin + 1);
#pragma unroll 1
    for (int k = 0; k < a.ns; ++k) {
        if (!ghosts(false)) return;
        ph.reset();
        // the trend: the irregular patches' F and q one thread an item, then a regular patch
        // a team at a time (patches dealt out over the SMs first)
        entry_items(a.lists.irr, bs.n_irr, 5, a.P, [&](int32_t ent, uint32_t local) {
            irregular_fq(lv[ent >> LVL_SHIFT], int64_t(ent & PATCH_MASK), local, a.P, H);
        });
        {
            using TM = Teams<R, P>;
            const int team = int(threadIdx.x) / TM::NT;
            bool ok = true;
            if (team < TM::N)
                ok = tile_sweep<R, P, TM::NT>(Team<TM::NT>{int(threadIdx.x) % TM::NT, unsigned(team + 1)}, lv, a.lists.core, bs.n_core,
                                              int(team * gridDim.x + blockIdx.x), int(TM::N * gridDim.x), H, g,
                                              smem + team * Tile<R, P>::BYTES, a.err, gb.limit);
            if (!__syncthreads_and(ok)) return;
        }
        if (!gb.sync()) return;
        // every block has taken the time step: the words back to zero for the maxima below and
        // the next step
        if (a.pre && k == 0 && blockIdx.x == 0 && threadIdx.x < RED_WORDS) a.red[threadIdx.x] = 0ull;
        entry_items(a.lists.irr, bs.n_irr, 4, a.P, [&](int32_t ent, uint32_t local) {
            auto body = [&](const DevLevelT<R>& L, int kind, int64_t id, int64_t) {
                if (kind == K_NODE)
                    node_at(L, id, g);
                else
                    coriolis_at(L, id);
            };
            visit_item<K_NODE | K_EDGE>(lv[ent >> LVL_SHIFT], int64_t(ent & PATCH_MASK), local, a.P, body);
        });
        // restriction, fine to coarse
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
        // the update; then the next stage, or what follows the last
        ph.reset();
        const R dt = to_r<R>(dt_s);
        live.run(lv, a.jmin, a.jtop, first_item(), int(gridDim.x * blockDim.x), [&](const DevLevelT<R>& L, int kind, int64_t id) {
            if (kind == K_NODE)
                update_node(L, id, a.st[k], dt);
            else
                update_edge(L, id, a.st[k], dt);
        });
        const bool last = k + 1 == a.ns;
        if (last && !(a.post && a.jtop > a.jmin) && !a.details) break;
        gb.arrive();
        if (a.jtop > a.jmin && !last) ph.ahead_fill(lv[a.jmin + 1], cnt, a.jmin + 1);
        if (a.jtop > a.jmin && last) ph.ahead_partial(lv[a.jtop - 1], cnt, a.jtop - 1);
        if (!gb.wait()) return;
    }
    if (a.post && a.jtop > a.jmin) {
        for (int j = a.jtop - 1; j >= a.jmin; --j) {
            ph.run_partial(lv[j], lv[j + 1]);
            gb.arrive();
            if (j > a.jmin)
                ph.ahead_partial(lv[j - 1], cnt, j - 1);
            else
                ph.ahead_fill(lv[a.jmin + 1], cnt, a.jmin + 1);
            if (!gb.wait()) return;
        }
        if (!ghosts(!a.details)) return;
    }
    if (a.details) {
        details_and_maxima(live, lv, a.jmin, a.jtop, first_item(), int(gridDim.x * blockDim.x), a.red, sh);
        if (!gb.sync()) return;
        if (blockIdx.x == 0 && threadIdx.x == 0) thresholds(a.thr, a.red, -1.0, -1.0, a.eps_c, a.advect);
    }
    bs.done(a);
}

// The inverse transform of the retained coefficients over the new lists, levels jmin + 1 up
// to a.jtop, with the ghosts: per level the even nodes and the edges from the level below,
// then the odd nodes from the even ones, then the ghosts.  The ghosts stay behind the odd
// nodes: at the rim of a proposed patch an odd node may have a parent that is not live, and
// takes the parent's value of before.
template <class R>
__global__ void __launch_bounds__(STAGE_TPB, 1) k_inverse(const __grid_constant__ StageArgs<R> a) {
    __shared__ BlockState<R> bs;
    if (!bs.init(a)) return;
    GridBarrier gb = bs.barrier(a);
    ListPhase<R> ph;
    if (a.jtop > a.jmin) ph.ahead_inverse(bs.sl[a.jmin + 1], bs.sl[a.jmin], bs.cnt, a.jmin + 1);
    for (int j = a.jmin + 1; j <= a.jtop; ++j) {
        const DevLevelT<R>& F = bs.sl[j];
        const DevLevelT<R>& C = bs.sl[j - 1];
        ph.run_inverse(F, C);
        gb.arrive();
        ph.ahead_odd(F, bs.cnt, j);
        if (!gb.wait()) return;
        ph.run_odd(F);
        gb.arrive();
        ph.ahead_fill(F, bs.cnt, j);
        if (!gb.wait()) return;
        ph.run_fill(F, C);
        if (j == a.jtop) break;
        gb.arrive();
        ph.ahead_inverse(bs.sl[j + 1], F, bs.cnt, j + 1);
        if (!gb.wait()) return;
    }
    bs.done(a);
}

template <class R, int P>
unsigned stage_grid_p(int nsm) {
    constexpr size_t smem = Teams<R, P>::N * Tile<R, P>::BYTES;
    // the dynamic tile and the static level records together may pass the default
    // 48 KB: the dynamic size is always declared
    if (cudaFuncSetAttribute(k_stage<R, P>, cudaFuncAttributeMaxDynamicSharedMemorySize, int(smem)) != cudaSuccess)
        return 0;
    int per_sm = 0, inv = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_stage<R, P>, STAGE_TPB, smem) != cudaSuccess) return 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&inv, k_inverse<R>, STAGE_TPB, 0) != cudaSuccess) return 0;
    return unsigned(std::max(std::min(per_sm, inv), 0) * nsm);
}

template <class R, class K>
cudaError_t launch_coop(K kernel, const StageArgs<R>& a, unsigned grid, size_t smem, cudaStream_t s) {
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3(grid);
    cfg.blockDim = dim3(STAGE_TPB);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeCooperative;
    attr[0].val.cooperative = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    count_launch(1);
    return cudaLaunchKernelEx(&cfg, kernel, a);
}

template <class R, int P>
cudaError_t launch_stage_p(const StageArgs<R>& a, unsigned grid, cudaStream_t s) {
    return launch_coop(k_stage<R, P>, a, grid, Teams<R, P>::N * Tile<R, P>::BYTES, s);
}

}  // namespace

// patch area -> tile side of the stage kernel (sides 1 and 2 have no regular tile)
template <class R>
unsigned stage_grid(int P, int nsm) {
    return P == 64 ? stage_grid_p<R, 8>(nsm) : P == 256 ? stage_grid_p<R, 16>(nsm) : stage_grid_p<R, 4>(nsm);
}

template <class R>
cudaError_t launch_stage(const StageArgs<R>& a, unsigned grid, cudaStream_t s) {
    if (a.jmax + 1 > MAXL || a.ns < 1 || a.ns > STEP_STAGES) return cudaErrorInvalidValue;
    return a.P == 64 ? launch_stage_p<R, 8>(a, grid, s) : a.P == 256 ? launch_stage_p<R, 16>(a, grid, s)
                                                                    : launch_stage_p<R, 4>(a, grid, s);
}

template <class R>
cudaError_t launch_inverse(const StageArgs<R>& a, unsigned grid, cudaStream_t s) {
    if (a.jmax + 1 > MAXL || a.jtop > a.jmax) return cudaErrorInvalidValue;
    return launch_coop(k_inverse<R>, a, grid, 0, s);
}

template cudaError_t launch_inverse<double>(const StageArgs<double>&, unsigned, cudaStream_t);
template cudaError_t launch_inverse<float>(const StageArgs<float>&, unsigned, cudaStream_t);
template unsigned stage_grid<double>(int, int);
template unsigned stage_grid<float>(int, int);
template cudaError_t launch_stage<double>(const StageArgs<double>&, unsigned, cudaStream_t);
template cudaError_t launch_stage<float>(const StageArgs<float>&, unsigned, cudaStream_t);

}  // namespace sww

// The phases of a step as one regular launch each, for every member of an ensemble or
// for one handle: time step; each stage's trend and update (Sec. 3.1, in
// the order of the persistent stage): ghosts level by level, the structured trend and
// the irregular patches (sww_tile.cu), the restrictions level by level, the update; the
// partial transform and ghosts; coefficients, maxima and thresholds; the inverse
// transform; the read-back records.  The kernel boundary is the barrier.
//
// Blocks come in groups, one group per member: a block copies the level records of
// its member that the phase touches into shared memory once, then strides over
// that member's items only (no search for the member of an item, and every field
// address from shared memory).
//
// Each phase is a kernel of its own.  The phases are chains of gathers whose latency is
// hidden by resident warps and by loads in flight per thread.  The stencil phases (up to
// 24 entries an item) are built for four blocks per SM (64 registers: measured 3-25 %
// faster per phase than five blocks, and six are slower still), the others for eight; one
// kernel for all phases had to take 32 registers for every phase and spilled 228 bytes.
// Ghosts of the 64-member jet ensemble (Jmax 6..9, per level and stage): 47 -> 35 us,
// restriction 33 -> 21, partial transform 76 -> 27, inverse transform 107 -> 70.
#include <cuda_runtime.h>

#include <algorithm>
#include <cstdint>

#include "pdl.cuh"
#include "sww_core.cuh"
#include "sww_kernels.h"
#include "sww_stage.h"

namespace sww {

namespace {

#include "sww_bodies.cuh"

constexpr int BATCH_TPB = 256;
constexpr int MAXL = 12;
constexpr int MAXM = 128;
enum {
    PH_FILL = 0, PH_RESTRICT, PH_DIV, PH_UPDATE, PH_SET_DT, PH_DT, PH_DT_FINAL, PH_PARTIAL,
    PH_DETAILS, PH_THRESH, PH_INV_A, PH_INV_B, PH_INV_FILL, PH_OUT
};

// items of work lists k0 and k1 (k1 < 0: none) of level L, block b of the
// member's bpm blocks: body(0, id) for list k0, body(1, id) for list k1
template <class R, class Body>
__device__ __forceinline__ void member_wl(const DevLevelT<R>& L, int k0, int k1, int b, int bpm, Body body) {
    const int n0 = L.wl_n[k0], n1 = k1 >= 0 ? L.wl_n[k1] : 0;
    const int32_t* __restrict__ l0 = L.wl + wl_off(L, k0);
    const int32_t* __restrict__ l1 = k1 >= 0 ? L.wl + wl_off(L, k1) : l0;
    for (int i = b * int(blockDim.x) + int(threadIdx.x); i < n0 + n1; i += bpm * int(blockDim.x)) {
        if (i < n0)
            body(0, int64_t(l0[i]));
        else
            body(1, int64_t(l1[i - n0]));
    }
}

template <int PH>
constexpr int phase_blocks() {
    return PH == PH_FILL || PH == PH_INV_FILL || PH == PH_RESTRICT || PH == PH_PARTIAL || PH == PH_DETAILS || PH == PH_INV_A || PH == PH_DIV
               ? 4
               : PH == PH_INV_B ? 6 : 8;
}

template <class R, int PH>
__global__ void __launch_bounds__(BATCH_TPB, phase_blocks<PH>()) k_phase(const __grid_constant__ BatchArgs<R> a, int j, int bpm) {
    chain_wait();
    const int m = blockIdx.x / bpm, b = blockIdx.x % bpm;
    const MemberRef<R>* mr = a.m ? a.m + m : &a.one;
    // one block per member
    if constexpr (PH == PH_DT_FINAL || PH == PH_SET_DT) {
        // the step, CFL or given; the reduction words are left at zero for the step's maxima
        // and the next step
        if (threadIdx.x < 32) {
            const double dt = PH == PH_SET_DT ? a.dt_given : cfl_step<R>(mr->lvs, mr->red, mr->cfl);
            __syncwarp();
            if (threadIdx.x == 0) *mr->dt = dt;
            if (threadIdx.x < RED_WORDS) mr->red[threadIdx.x] = 0ull;
        }
        return;
    }
    if constexpr (PH == PH_THRESH) {   // given, or relative to the live maxima (a prescribed velocity has no threshold)
        if (threadIdx.x == 0) thresholds(mr->thr, mr->red, a.eps_h, a.eps_u, mr->eps_c, mr->advect != 0);
        return;
    }
    if constexpr (PH == PH_OUT) {
        BatchOut* o = reinterpret_cast<BatchOut*>(a.out) + m;
        const int t = threadIdx.x;
        if (t < 16) {
            const bool in = t >= a.jmin && t <= mr->jmax;
            o->counts[t] = in ? *mr->lvs[t].npatches : 0;
            o->live[t] = in ? mr->lvs[t].wl_n[WL_LN] : 0;
        }
        if (t == 0) {
            o->dt = *mr->dt;
            o->err = *mr->err;
        }
        return;
    }
    const int jtop = mr->jtop;
    // level-serial phases skip the members that do not reach the level
    constexpr bool inv = PH == PH_INV_A || PH == PH_INV_B || PH == PH_INV_FILL;
    constexpr bool down = PH == PH_RESTRICT || PH == PH_DIV || PH == PH_PARTIAL;
    if (PH == PH_FILL && j > jtop) return;
    if (down && j > jtop - 1) return;
    if (inv && j > mr->j1) return;
    // the member's records of the levels the phase reads (the inverse transform
    // reaches one level above the top)
    __shared__ DevLevelT<R> sl[MAXL];
    {
        const int lo = (PH == PH_FILL || inv) ? j - 1 : down ? j : a.jmin;
        const int hi = (PH == PH_RESTRICT || PH == PH_PARTIAL) ? j + 1 : (PH == PH_FILL || PH == PH_DIV || inv) ? j : jtop;
        const int words = int((hi - lo + 1) * sizeof(DevLevelT<R>) / sizeof(int));
        const int* src = reinterpret_cast<const int*>(mr->lvs + lo);
        int* dst = reinterpret_cast<int*>(sl + lo);
        for (int k = threadIdx.x; k < words; k += blockDim.x) dst[k] = src[k];
    }
    __syncthreads();
    // the live points of every level
    constexpr bool all_live = PH == PH_UPDATE || PH == PH_DT || PH == PH_DETAILS;
    __shared__ LiveItems live;
    const int first = b * int(blockDim.x) + int(threadIdx.x), stride = bpm * int(blockDim.x);
    if constexpr (all_live) {
        live.init(sl, a.jmin, jtop);
        __syncthreads();
    }
    if constexpr (PH == PH_FILL || PH == PH_INV_FILL) {
        // ghost nodes and edges of level j from level j - 1 (of the inverse transform: a phase
        // behind its odd nodes, which at the rim of a proposed patch may have a parent that is
        // not live and take its value of before)
        member_wl(sl[j], WL_GN, WL_GE, b, bpm, [&](int k, int64_t id) {
            if (k == 0)
                fill_node(sl[j], sl[j - 1], id);
            else
                fill_edge(sl[j], sl[j - 1], id);
        });
    } else if constexpr (PH == PH_RESTRICT) {
        // covered nodes and the edges with a covered end of level j
        member_wl(sl[j], WL_CN, WL_RE, b, bpm, [&](int k, int64_t id) {
            if (k == 0)
                restrict_node(sl[j], sl[j + 1], id);
            else
                restrict_edge(sl[j], sl[j + 1], id);
        });
    } else if constexpr (PH == PH_DIV) {
        member_wl(sl[j], WL_DN, -1, b, bpm, [&](int, int64_t id) { div_at(sl[j], id); });
    } else if constexpr (PH == PH_PARTIAL) {
        // R_h at covered nodes of level j from level j + 1 (Eq. Rh)
        member_wl(sl[j], WL_CN, -1, b, bpm, [&](int, int64_t id) { partial_node(sl[j], sl[j + 1], id); });
    } else if constexpr (PH == PH_DT) {
        __shared__ unsigned long long sh[BATCH_TPB / 32], slev[RED_WORDS - RED_LEVEL];
        cfl_maxima(live, sl, a.jmin, jtop, first, stride, a.H, a.g, mr->red, sh, slev);   // the step in PH_DT_FINAL
    } else if constexpr (PH == PH_DETAILS) {
        __shared__ unsigned long long shm[BATCH_TPB / 32];
        details_and_maxima(live, sl, a.jmin, jtop, first, stride, mr->red, shm);
    } else if constexpr (PH == PH_INV_A) {
        member_wl(sl[j], WL_LN, WL_LE, b, bpm,
                  [&](int k, int64_t id) { inverse_a_item(sl[j], sl[j - 1], k == 0 ? K_NODE : K_EDGE, id); });
    } else if constexpr (PH == PH_INV_B) {
        member_wl(sl[j], WL_LN, -1, b, bpm, [&](int, int64_t id) { inverse_b_item(sl[j], id); });
    } else {
        static_assert(PH == PH_UPDATE || PH == PH_SET_DT || PH == PH_DT_FINAL || PH == PH_THRESH || PH == PH_OUT, "phase");
        const R dt = to_r<R>(mr->dt ? *mr->dt : 0.0);
        live.run(sl, a.jmin, jtop, first, stride, [&](const DevLevelT<R>& L, int kind, int64_t id) {
            if (kind == K_NODE)
                update_node(L, id, a.st, dt);
            else
                update_edge(L, id, a.st, dt);
        });
    }
}

// blocks per member: enough for the member's share of the bound, at most two waves of
// 8 blocks of 256 per SM over all members (measured a little faster than one wave:
// the members' shares are uneven)
template <class R>
int batch_bpm(const BatchArgs<R>& a, int64_t entries, int slots, int nsm) {
    const int cap = std::max(1, 16 * nsm / a.nm);
    const int64_t per = (entries + a.nm - 1) / a.nm * a.P * slots;
    return int(std::max<int64_t>(1, std::min<int64_t>((per + BATCH_TPB - 1) / BATCH_TPB, cap)));
}

template <int PH, class R>
cudaError_t batch_go(const BatchArgs<R>& a, int j, int bpm, cudaStream_t s) {
    count_launch(1);
    return launch_chain(a.chain, k_phase<R, PH>, dim3(unsigned(a.nm * bpm)), dim3(BATCH_TPB), 0, s, a, j, bpm);
}

template <class R>
bool batch_ok(const BatchArgs<R>& a, int top) {
    return a.nm >= 1 && a.nm <= MAXM && (a.m || a.nm == 1) && top + 1 <= MAXL;
}
template <class R>
int64_t entries_to(const BatchArgs<R>& a, const int64_t* level_entries) {
    int64_t all = 0;
    for (int j = a.jmin; j <= a.jtop_max; ++j) all += level_entries[j];
    return all;
}

}  // namespace

template <class R>
cudaError_t launch_batch_restrict(const BatchArgs<R>& a, const int64_t* level_entries, int j, int nsm, cudaStream_t s) {
    if (!batch_ok(a, j + 1)) return cudaErrorInvalidValue;
    return batch_go<PH_RESTRICT>(a, j, batch_bpm(a, level_entries[j], 4, nsm), s);
}

template <class R>
cudaError_t launch_batch_div(const BatchArgs<R>& a, const int64_t* level_entries, int j, int nsm, cudaStream_t s) {
    if (!batch_ok(a, j)) return cudaErrorInvalidValue;
    return batch_go<PH_DIV>(a, j, batch_bpm(a, level_entries[j], 1, nsm), s);
}

template <class R>
cudaError_t launch_stage_batch_part(const BatchArgs<R>& a, const int64_t* level_entries, int64_t irr_entries, int nsm,
                                    int part, cudaStream_t s) {
    if (!batch_ok(a, a.jtop_max)) return cudaErrorInvalidValue;
    const int64_t all = entries_to(a, level_entries);
    cudaError_t e = cudaSuccess;
    switch (part) {
        case 0:
            for (int j = a.jmin + 1; j <= a.jtop_max && e == cudaSuccess; ++j)
                e = batch_go<PH_FILL>(a, j, batch_bpm(a, level_entries[j], 4, nsm), s);
            break;
        case 1:
        case 2:
            e = launch_tile_trend(a, all, irr_entries, nsm, part, s);
            break;
        case 3:
            for (int j = a.jtop_max - 1; j >= a.jmin && e == cudaSuccess; --j) {
                e = launch_batch_restrict(a, level_entries, j, nsm, s);
                if (e == cudaSuccess) e = launch_batch_div(a, level_entries, j, nsm, s);
            }
            break;
        default:
            e = batch_go<PH_UPDATE>(a, 0, batch_bpm(a, all, 4, nsm), s);
    }
    return e;
}

template <class R>
cudaError_t launch_batch_pre(const BatchArgs<R>& a, const int64_t* level_entries, int nsm, double dt, cudaStream_t s) {
    if (!batch_ok(a, a.jtop_max)) return cudaErrorInvalidValue;
    const int64_t all = entries_to(a, level_entries);
    BatchArgs<R> b = a;
    b.dt_given = dt;
    if (dt > 0) return batch_go<PH_SET_DT>(b, 0, 1, s);
    cudaError_t e = batch_go<PH_DT>(b, 0, batch_bpm(b, all, 4, nsm), s);
    return e == cudaSuccess ? batch_go<PH_DT_FINAL>(b, 0, 1, s) : e;
}

template <class R>
cudaError_t launch_batch_fill(const BatchArgs<R>& a, const int64_t* level_entries, int nsm, cudaStream_t s) {
    return launch_stage_batch_part(a, level_entries, 0, nsm, 0, s);
}

template <class R>
cudaError_t launch_batch_partial(const BatchArgs<R>& a, const int64_t* level_entries, int nsm, cudaStream_t s) {
    if (!batch_ok(a, a.jtop_max)) return cudaErrorInvalidValue;
    cudaError_t e = cudaSuccess;
    for (int j = a.jtop_max - 1; j >= a.jmin && e == cudaSuccess; --j)
        e = batch_go<PH_PARTIAL>(a, j, batch_bpm(a, level_entries[j], 1, nsm), s);
    return e;
}

template <class R>
cudaError_t launch_batch_details(const BatchArgs<R>& a, const int64_t* level_entries, int nsm, cudaStream_t s) {
    if (!batch_ok(a, a.jtop_max)) return cudaErrorInvalidValue;
    return batch_go<PH_DETAILS>(a, 0, batch_bpm(a, entries_to(a, level_entries), 4, nsm), s);
}

template <class R>
cudaError_t launch_batch_thresholds(const BatchArgs<R>& a, cudaStream_t s) {
    if (!batch_ok(a, 0)) return cudaErrorInvalidValue;
    return batch_go<PH_THRESH>(a, 0, 1, s);
}

template <class R>
cudaError_t launch_batch_inverse(const BatchArgs<R>& a, const int64_t* level_entries, int j, int nsm, cudaStream_t s) {
    if (!batch_ok(a, j)) return cudaErrorInvalidValue;
    cudaError_t e = batch_go<PH_INV_A>(a, j, batch_bpm(a, level_entries[j], 4, nsm), s);
    return e == cudaSuccess ? batch_go<PH_INV_B>(a, j, batch_bpm(a, level_entries[j], 1, nsm), s) : e;
}

template <class R>
cudaError_t launch_batch_inverse_fill(const BatchArgs<R>& a, const int64_t* level_entries, int j, int nsm, cudaStream_t s) {
    if (!batch_ok(a, j)) return cudaErrorInvalidValue;
    return batch_go<PH_INV_FILL>(a, j, batch_bpm(a, level_entries[j], 4, nsm), s);
}

template <class R>
cudaError_t launch_batch_out(const BatchArgs<R>& a, cudaStream_t s) {
    if (!batch_ok(a, 0)) return cudaErrorInvalidValue;
    return batch_go<PH_OUT>(a, 0, 1, s);
}

#define BATCH_INST(R)                                                                                          \
    template cudaError_t launch_batch_restrict<R>(const BatchArgs<R>&, const int64_t*, int, int, cudaStream_t); \
    template cudaError_t launch_batch_div<R>(const BatchArgs<R>&, const int64_t*, int, int, cudaStream_t);     \
    template cudaError_t launch_batch_pre<R>(const BatchArgs<R>&, const int64_t*, int, double, cudaStream_t);  \
    template cudaError_t launch_batch_fill<R>(const BatchArgs<R>&, const int64_t*, int, cudaStream_t);         \
    template cudaError_t launch_batch_partial<R>(const BatchArgs<R>&, const int64_t*, int, cudaStream_t);      \
    template cudaError_t launch_batch_details<R>(const BatchArgs<R>&, const int64_t*, int, cudaStream_t);      \
    template cudaError_t launch_batch_thresholds<R>(const BatchArgs<R>&, cudaStream_t);                        \
    template cudaError_t launch_batch_inverse<R>(const BatchArgs<R>&, const int64_t*, int, int, cudaStream_t); \
    template cudaError_t launch_batch_inverse_fill<R>(const BatchArgs<R>&, const int64_t*, int, int, cudaStream_t); \
    template cudaError_t launch_batch_out<R>(const BatchArgs<R>&, cudaStream_t);                               \
    template cudaError_t launch_stage_batch_part<R>(const BatchArgs<R>&, const int64_t*, int64_t, int, int, cudaStream_t);
BATCH_INST(double)
BATCH_INST(float)

}  // namespace sww

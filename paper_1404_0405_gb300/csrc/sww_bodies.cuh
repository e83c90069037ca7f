// Device-side helpers shared by the kernel translation units: the work-list item
// loop and the per-item bodies of the trend, the RK stage and the prolongation.
// Included inside an anonymous namespace of each translation unit.
#pragma once

#include "f64conv.cuh"

__device__ __forceinline__ int64_t gid() { return int64_t(blockIdx.x) * blockDim.x + threadIdx.x; }
template <class R>
__device__ __forceinline__ R esign(int32_t code) { return (code & 1) ? R(-1) : R(1); }
// an FP64 geometry value entering arithmetic of the working precision (FP32: the
// integer-pipe rounding of f64conv.cuh)
template <class R>
__device__ __forceinline__ R to_r(double x);
template <>
__device__ __forceinline__ double to_r<double>(double x) { return x; }
template <>
__device__ __forceinline__ float to_r<float>(double x) { return f64_to_f32_rn(x); }
template <class R>
__device__ __forceinline__ R geo(const double* __restrict__ p, int64_t i) { return to_r<R>(p[i]); }


template <class R>
__device__ __forceinline__ R predict(const DevLevelT<R>& F, const R* __restrict__ uc, int64_t fe) {
    R s = R(0);
#pragma unroll
    for (int k = 0; k < 12; ++k) s += F.vw[k * F.E + fe] * uc[F.vst[k * F.E + fe]];
    return s;
}

// the same through stencil ids already read
template <class R>
__device__ __forceinline__ R predict_from(const DevLevelT<R>& F, const R* __restrict__ uc, int64_t fe, const int32_t* st) {
    R s = R(0);
#pragma unroll
    for (int k = 0; k < 12; ++k) s += F.vw[k * F.E + fe] * uc[st[k]];
    return s;
}

template <class R>
__device__ __forceinline__ R height_detail(const DevLevelT<R>& F, int64_t x) {
    R s = F.dh[x];
#pragma unroll
    for (int k = 0; k < 4; ++k) s -= F.ptw[k * F.N + x] * F.dh[F.par[k * F.N + x]];
    return s;
}

__device__ __forceinline__ unsigned long long dbits(double x) {
    return static_cast<unsigned long long>(__double_as_longlong(x));
}

// the viscous form (nu != 0), tested on the bits of nu (either sign of zero is
// zero) on the integer pipe: the per-point bodies ask at every point
template <class Lv>
__device__ __forceinline__ bool viscous(const Lv& L) {
    return (dbits(L.nu) << 1) != 0;
}

// ---------------------------------------------------------------------------- CFL step and field maxima

// |x| as an unsigned key ordered like |x|: with the sign bit cleared, IEEE numbers
// order like their bit patterns, and NaN keys lie above the key of +infinity
__device__ __forceinline__ unsigned long long abs_key(float x) { return __float_as_uint(x) & 0x7fffffffu; }
__device__ __forceinline__ unsigned long long abs_key(double x) { return dbits(x) & 0x7fffffffffffffffull; }
template <class R>
__device__ __forceinline__ unsigned long long inf_key() {
    return sizeof(R) == 4 ? 0x7f800000ull : 0x7ff0000000000000ull;
}
// the magnitude a key stands for, as a double (exact: widening keeps the value)
template <class R>
__device__ __forceinline__ double key_value(unsigned long long k) {
    return sizeof(R) == 4 ? double(__uint_as_float(unsigned(k))) : __longlong_as_double(static_cast<long long>(k));
}

// squared CFL frequency f^2 + g h (pi/dx)^2 at node id, in FP64 with the products
// and sums rounded in the written order (no contraction).  The time step takes the
// square root of the maximum only: a correctly rounded square root is monotone, so
// that equals the maximum of the roots.
template <class R>
__device__ __forceinline__ double omega2_at(const DevLevelT<R>& L, int64_t id, double H, double g) {
    const double f = L.f_n[id];
    return __dadd_rn(__dmul_rn(f, f), __dmul_rn(__dmul_rn(g, __dadd_rn(H, double(L.dh[id]))), L.kx2));
}

// Running maximum of a key per level over one thread's items, flushed into the
// block's per-level words (shared memory) when the level changes: a thread meets
// its items in list order, which is level order, so it flushes a few times.
struct LevelMax {
    int j = -1;
    unsigned long long k = 0;
    __device__ __forceinline__ void flush(unsigned long long* sm) {
        if (k) atomicMax(sm + j, k);
    }
    __device__ __forceinline__ void add(int jj, unsigned long long key, unsigned long long* sm) {
        if (jj != j) {
            flush(sm);
            j = jj;
            k = 0;
        }
        k = key > k ? key : k;
    }
};

// Advective bound min over live edges of dx_j / |u| (Sec. 3.1's CFL condition):
// for one level, a correctly rounded dx_j / a falls as a grows, so the minimum is
// dx_j over the level's largest |u|; then the step cfl * min(1/omega, that bound).  By
// one warp, a level a lane; the value is lane 0's.
template <class R>
__device__ __forceinline__ double cfl_step(const DevLevelT<R>* lvs, const unsigned long long* red, double cfl) {
    const int lane = threadIdx.x & 31;
    const unsigned long long k = lane < RED_WORDS - RED_LEVEL ? red[RED_LEVEL + lane] : 0ull;
    double r = k ? lvs[lane].dx / key_value<R>(k) : INFINITY;
    for (int o = 16; o > 0; o >>= 1) r = fmin(r, __shfl_xor_sync(0xffffffffu, r, o));
    const double w = sqrt(__longlong_as_double(static_cast<long long>(red[0])));
    return cfl * fmin(1.0 / w, r);
}

// patch of node x (the poles: npatch); the patch side is a power of two
template <class Lv>
__device__ __forceinline__ int64_t patch_of(const Lv& L, int64_t x) {
    return x < L.nelem ? int64_t(uint32_t(x) >> (2 * (__ffs(int(L.p)) - 1))) : L.npatch;
}

// Item kinds of a work-list entry, in slot order.
constexpr int K_NODE = 1, K_EDGE = 2, K_TRI = 4;

template <int KINDS>
__host__ __device__ constexpr int slots_of() {
    return ((KINDS & K_NODE) ? 1 : 0) + ((KINDS & K_EDGE) ? 3 : 0) + ((KINDS & K_TRI) ? 2 : 0);
}

// Visit the items of the entries of a work list, one thread per item:
// body(L, kind, id, elem).  An entry covers slots x P threads (P = configured patch
// area): one slot of nodes, three of edges (orientation 0, 1, 2) and two of triangles,
// as KINDS selects.  A pole entry yields the two pole nodes with
// elem = -1.  Entries name their level in `lvs` (multi-level lists) or all belong
// to `one` when lvs is null.
// Item `local` (0 <= local < slots x P) of work-list entry patch `pat` of level L:
// body(L, kind, id, elem) when the slot holds an item (see for_items).
// P is a power of two (the patch side is), so slot and index are a shift and a mask.
template <int KINDS, class Lv, class Body>
__device__ __forceinline__ void visit_item(const Lv& L, int64_t pat, uint32_t local, int P, Body& body) {
    int slot = int(local >> (__ffs(P) - 1));
    const int64_t idx = int64_t(local & uint32_t(P - 1));
    if (pat == L.npatch) {
        if ((KINDS & K_NODE) && slot == 0 && idx < 2) body(L, K_NODE, L.nelem + idx, int64_t(-1));
        return;
    }
    const int64_t pp = L.p * L.p;
    if (idx >= pp) return;
    const int64_t el = pat * pp + idx;
    if (KINDS & K_NODE) {
        if (slot == 0) {
            body(L, K_NODE, el, el);
            return;
        }
        slot -= 1;
    }
    if (KINDS & K_EDGE) {
        if (slot < 3) {
            body(L, K_EDGE, slot * L.nelem + el, el);
            return;
        }
        slot -= 3;
    }
    if (KINDS & K_TRI) {
        if (slot < 2) {
            body(L, K_TRI, slot * L.nelem + el, el);
            return;
        }
    }
}

template <int KINDS, class Lv, class Body>
__device__ __forceinline__ void for_items(const Lv* __restrict__ lvs, const Lv& one,
                                          const int32_t* __restrict__ list, const int32_t* __restrict__ count, int P,
                                          Body body) {
    // 32-bit item numbers: a list holds fewer than 2^31 items up to level 11
    constexpr uint32_t NS = slots_of<KINDS>();
    const int lp = __ffs(P) - 1;
    const uint32_t n = uint32_t(*count) * (NS << lp);
    const uint32_t stride = gridDim.x * blockDim.x;
    for (uint32_t it = blockIdx.x * blockDim.x + threadIdx.x; it < n; it += stride) {
        const uint32_t e = (it >> lp) / NS;
        const int32_t ent = list[e];
        const Lv& L = lvs ? lvs[ent >> LVL_SHIFT] : one;
        visit_item<KINDS>(L, int64_t(ent & PATCH_MASK), it - ((e * NS) << lp), P, body);
    }
}

// ---------------------------------------------------------------------------- trend bodies (Sec. 3.1)

// The bodies below load what they need in groups issued together and test the flags
// afterwards: a short-circuit test per neighbour makes each load wait for the one before
// (a divergence's six ring edges took 4 us of a stage's phase that way, 2 us now).

// potential vorticity q = (curl u + f)/h at a triangle (dual cell)
template <class R>
__device__ __forceinline__ void pv_at(const DevLevelT<R>& L, int64_t t, R H) {
    if (L.advect) return;   // no velocity trend, no q
    int32_t n[3], c[3];
#pragma unroll
    for (int k = 0; k < 3; ++k) n[k] = L.tn[k * L.T + t], c[k] = L.te[k * L.T + t];
    uint8_t nf[3], ef[3];
    R dh[3], u[3];
    double de[3];
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        nf[k] = L.nflag[n[k]], ef[k] = L.eflag[c[k] >> 1];
        dh[k] = L.dh[n[k]], u[k] = L.u[c[k] >> 1], de[k] = L.d_e[c[k] >> 1];
    }
    bool ok = true;
#pragma unroll
    for (int k = 0; k < 3; ++k) ok = ok & ((nf[k] & AVAIL) != 0) & ((ef[k] & AVAIL) != 0);
    if (!ok) return;
    R circ = esign<R>(c[0]) * u[0] * to_r<R>(de[0]) + esign<R>(c[1]) * u[1] * to_r<R>(de[1]) +
             esign<R>(c[2]) * u[2] * to_r<R>(de[2]);
    R hv = geo<R>(L.kite, t) * (H + dh[0]) + geo<R>(L.kite, L.T + t) * (H + dh[1]) + geo<R>(L.kite, 2 * L.T + t) * (H + dh[2]);
    R Av = geo<R>(L.A_v, t);
    if (viscous(L)) L.zeta[t] = circ / Av;
    // one division in the FP64 form (the FP64 pipe is narrow)
    if constexpr (sizeof(R) == 8)
        L.q[t] = (circ + geo<R>(L.f_v, t) * Av) / hv;
    else
        L.q[t] = (circ / Av + geo<R>(L.f_v, t)) / (hv / Av);
}

// thickness flux F = h_e u at an edge
template <class R>
__device__ __forceinline__ void flux_at(const DevLevelT<R>& L, int64_t e, R H) {
    const uint8_t fe = L.eflag[e];
    const int32_t a = L.en[e], b = L.en[L.E + e];
    const R u = L.u[e];
    const uint8_t fa = L.nflag[a], fb = L.nflag[b];
    const R ha = L.dh[a], hb = L.dh[b];
    if (!(((fe & AVAIL) != 0) & ((fa & AVAIL) != 0) & ((fb & AVAIL) != 0))) return;
    L.F[e] = R(0.5) * ((H + ha) + (H + hb)) * u;
    // viscous form: diffusive height flux -nu grad(dh) (joins F in the divergence)
    if (viscous(L)) L.Fd[e] = -R(L.nu) * (hb - ha) / geo<R>(L.d_e, e);
}

// the ring of node v: its edges' codes, and their flags, total height flux and lengths
template <class R>
struct Ring {
    int32_t code[6];
    uint8_t ef[6];
    R F[6];
    double le[6];
    __device__ __forceinline__ Ring(const DevLevelT<R>& L, int64_t v) {
#pragma unroll
        for (int k = 0; k < 6; ++k) code[k] = L.ring_e[k * L.N + v];
#pragma unroll
        for (int k = 0; k < 6; ++k) {
            const int64_t e = edge(k);
            ef[k] = L.eflag[e], F[k] = L.F[e], le[k] = L.l_e[e];
        }
        if (viscous(L)) {
#pragma unroll
            for (int k = 0; k < 6; ++k) F[k] = F[k] + L.Fd[edge(k)];
        }
    }
    // ring slot 5 of a pentagon is padded with -1: edge 0 is read and not used
    __device__ __forceinline__ int64_t edge(int k) const { return code[k] < 0 ? 0 : code[k] >> 1; }
};

// divergence of the height flux (with the diffusive flux of the viscous form) at a node
template <class R>
__device__ __forceinline__ void div_at(const DevLevelT<R>& L, int64_t v) {
    const uint8_t fv = L.nflag[v];
    const int dg = L.deg[v];
    const double Av = L.A_i[v];
    if (!(fv & AVAIL)) return;
    const Ring<R> g(L, v);
    R div = R(0);
    bool ok = true;   // every ring edge available (else nothing is written)
#pragma unroll
    for (int k = 0; k < 6; ++k)
        if (k < dg) {
            ok = ok & ((g.ef[k] & AVAIL) != 0);
            div += esign<R>(g.code[k]) * g.F[k] * to_r<R>(g.le[k]);
        }
    if (!ok) return;
    L.c[v] = div / to_r<R>(Av);
}

// a node whose divergence the restricted fluxes change: available, with a covered
// node among itself and its neighbours (an edge is restricted when an end is
// covered).  The work list WL_DN holds exactly these nodes.
template <class R>
__device__ __forceinline__ bool restricted_div_node(const DevLevelT<R>& L, int64_t v) {
    const uint8_t f = L.nflag[v];
    if (!(f & AVAIL)) return false;
    if (f & COVERED) return true;
    // the neighbours' flags, their loads issued together (no early exit)
    const int dg = L.deg[v];
    uint8_t acc = 0;
#pragma unroll
    for (int k = 0; k < 6; ++k)
        if (k < dg) acc |= L.nflag[L.ring_n[k * L.N + v]];
    return (acc & COVERED) != 0;
}

// divergence, kinetic energy and Bernoulli function at a node
template <class R>
__device__ __forceinline__ void node_at(const DevLevelT<R>& L, int64_t v, R g) {
    if (L.advect) return div_at(L, v);   // prescribed velocity: no Bernoulli function
    const uint8_t fv = L.nflag[v];
    const int dg = L.deg[v];
    if (!(fv & AVAIL)) return;
    const Ring<R> r(L, v);
    R u[6];
    double de[6];
#pragma unroll
    for (int k = 0; k < 6; ++k) u[k] = L.u[r.edge(k)], de[k] = L.d_e[r.edge(k)];
    R div = R(0), ke = R(0), du = R(0);
    bool ok = true;   // every ring edge available (else nothing is written)
    const bool visc = viscous(L);
#pragma unroll
    for (int k = 0; k < 6; ++k)
        if (k < dg) {
            ok = ok & ((r.ef[k] & AVAIL) != 0);
            const R le = to_r<R>(r.le[k]);
            div += esign<R>(r.code[k]) * r.F[k] * le;
            if (visc) du += esign<R>(r.code[k]) * u[k] * le;
            ke += R(0.25) * le * to_r<R>(de[k]) * u[k] * u[k];
        }
    if (!ok) return;
    R A = geo<R>(L.A_i, v);
    // viscous form: -nu div u joins B (so that -grad B gains +nu grad div u)
    if (visc) ke -= R(L.nu) * du;
    L.c[v] = div / A;
    L.B[v] = g * L.dh[v] + ke / A;
}

// energy-conserving Coriolis tendency +q F.n_left at a live edge (TRiSK)
template <class R>
__device__ __forceinline__ void coriolis_at(const DevLevelT<R>& L, int64_t e) {
    if (L.advect || !(L.eflag[e] & LIVE)) return;
    // FP64: the factors 1/2 of the q averages out of the sum (powers of two).  Not in FP32,
    // where the products of a field that dies away reach the subnormals and would round
    // elsewhere
    constexpr R hq = sizeof(R) == 8 ? R(1) : R(0.5);
    R qe = hq * (L.q[L.et[e]] + L.q[L.et[L.E + e]]);
    R s = R(0);
#pragma unroll
    for (int k = 0; k < 10; ++k) {
        int32_t e2 = L.cor_i[k * L.E + e];
        R w = geo<R>(L.cor_w, k * L.E + e);
        R q2 = hq * (L.q[L.et[e2]] + L.q[L.et[L.E + e2]]);
        s += w * L.F[e2] * hq * (qe + q2);
    }
    if constexpr (sizeof(R) == 8) s *= R(0.25);
    // viscous form: -nu grad^perp curl u, grad^perp zeta = (1/l_e) sum_{v at e} t_{e,v} zeta_v
    if (viscous(L)) {
        R gp = R(0);
        for (int side = 0; side < 2; ++side) {
            const int32_t t = L.et[side * L.E + e];
            for (int k = 0; k < 3; ++k) {
                const int32_t code = L.te[k * L.T + t];
                if ((code >> 1) == e) gp += esign<R>(code) * L.zeta[t];
            }
        }
        s -= R(L.nu) * gp / geo<R>(L.l_e, e);
    }
    L.Q[e] = s;
}

// trend and one Runge-Kutta stage at a live point (terms with a zero coefficient
// are skipped, so stale storage never enters):
//   y <- a*y0 + b*y + (cdt*dt)*k + (ddt*dt)*acc,   acc <- al*acc + be*k
template <class R>
__device__ __forceinline__ void rk_apply(const StageCoef<R>& st, R dt, R k, R* y, R* y0, R* acc) {
    R v = st.cdt * dt * k;
    R b = R(0);
    if (st.base) {
        b = *y;
        *y0 = b;
    } else if (st.ha) {
        b = *y0;
    }
    if (st.ha) v += st.a * b;
    if (st.hb) v += st.b * *y;
    if (st.hddt) v += st.ddt * dt * *acc;
    if (st.hacc) *acc = (st.hal ? st.al * *acc : R(0)) + st.be * k;
    *y = v;
}

template <class R>
__device__ __forceinline__ void update_node(const DevLevelT<R>& L, int64_t v, const StageCoef<R>& st, R dt) {
    R k = -L.c[v];
    if (st.trend) L.dht[v] = k;
    if (st.apply) rk_apply(st, dt, k, &L.dh[v], &L.dh0[v], &L.dha[v]);
}

template <class R>
__device__ __forceinline__ void update_edge(const DevLevelT<R>& L, int64_t e, const StageCoef<R>& st, R dt) {
    if (L.advect) {   // prescribed velocity: zero trend, u untouched
        if (st.trend) L.ut[e] = R(0);
        return;
    }
    R k = L.Q[e] - (L.B[L.en[L.E + e]] - L.B[L.en[e]]) / geo<R>(L.d_e, e);
    if (st.trend) L.ut[e] = k;
    if (st.apply) rk_apply(st, dt, k, &L.u[e], &L.u0[e], &L.ua[e]);
}

// ---------------------------------------------------------------------------- prolongation (Eqs. 1-2)

// ghost node i of level F (of its list WL_GN) from level C: inverse transform with zero
// coefficients
template <class R>
__device__ __forceinline__ void fill_node(const DevLevelT<R>& F, const DevLevelT<R>& C, int64_t i) {
    const int32_t k = F.f2c[i];
    if (k >= 0) {
        F.dh[i] = C.dh[k];
        return;
    }
    int32_t p[4], c[4];
    R w[4], a[4], b[4];
    uint8_t f[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) p[q] = F.par[q * F.N + i], w[q] = F.ptw[q * F.N + i];
    // the parents of an odd node are even: each has a coarse node
#pragma unroll
    for (int q = 0; q < 4; ++q) f[q] = F.nflag[p[q]], a[q] = F.dh[p[q]], c[q] = F.f2c[p[q]];
#pragma unroll
    for (int q = 0; q < 4; ++q) b[q] = C.dh[c[q]];
    R s = R(0);
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        const R v = (f[q] & LIVE) ? a[q] : b[q];
        s += w[q] * v;
    }
    F.dh[i] = s;
}

// the half of a coarse edge with coarse velocity uc, from its own prediction and the
// other half's, when neither is live
template <class R>
__device__ __forceinline__ R half_value(R P, R Po, R uc) { return P + R(0.5) * (R(2) * uc - P - Po); }

// ghost edge i of level F (of its list WL_GE) from level C.  Both halves of a coarse edge
// need both predictions, so the item of the first half writes the second too when that
// is a ghost as well (then the list does not hold the second, see wl_item): 24
// stencil entries a pair instead of 48.
template <class R>
__device__ __forceinline__ void fill_edge(const DevLevelT<R>& F, const DevLevelT<R>& C, int64_t i) {
    if (F.advect) return;   // prescribed velocity is kept everywhere
    const int32_t o = F.fe_ot[i];
    const int32_t E = F.fe_ce[i];
    const R P = predict(F, C.u, i);
    if (o < 0) {
        F.u[i] = P;
        return;
    }
    const uint8_t fo = F.eflag[o];
    const R uo = F.u[o], uc = C.u[E];
    if (fo & LIVE) {
        F.u[i] = R(2) * uc - uo;
    } else {
        const R Po = predict(F, C.u, o);
        F.u[i] = half_value(P, Po, uc);
        // only the first half reaches here when both are ghosts
        if (fo & GHOST) F.u[o] = half_value(Po, P, uc);
    }
}


// ---------------------------------------------------------------------------- transforms (Eqs. 1-2)

// A coarse edge has a coefficient when one of its halves is live; it is taken at the first
// half (kind 0) when that is live, else at the second.  Live half i of the other half o,
// kind k: whether i is the one.
__device__ __forceinline__ bool pair_at(int k, uint8_t other_flag) { return k == 0 || !(other_flag & LIVE); }

// wavelet coefficients at a live point of F > Jmin from C = the level below
// (Eqs. 1-2; velocity transform of Sec. 4.1): h~ at odd nodes, u~ at interior fine
// edges, u~_E of a coarse edge at one of its live halves
template <class R>
__device__ __forceinline__ void details_item(const DevLevelT<R>& L, const DevLevelT<R>& C, int kind, int64_t id) {
    if (kind == K_NODE) {
        if (L.f2c[id] < 0) L.hdet[id] = height_detail(L, id);
        return;
    }
    const int32_t o = L.fe_ot[id];
    const int fk = L.fe_kind[id];
    if (o >= 0 && !pair_at(fk, L.eflag[o])) return;
    const R di = L.u[id] - predict(L, C.u, id);
    if (o < 0) {
        L.ui[id] = di;
    } else {
        const R d_o = L.u[o] - predict(L, C.u, o);
        L.ue[L.fe_ce[id]] = fk == 0 ? R(0.5) * (di - d_o) : R(0.5) * (d_o - di);
    }
}

// inverse transform of the retained coefficients at a live point of F from C:
// (a) even nodes and edges; coefficients count only where the point was live
// before the adaptation (WASLIVE)
template <class R>
__device__ __forceinline__ void inverse_a_item(const DevLevelT<R>& L, const DevLevelT<R>& C, int kind, int64_t id) {
    if (kind == K_NODE) {
        const int32_t k = L.f2c[id];
        if (k < 0) return;
        R s = C.dh[k];
#pragma unroll
        for (int g = 0; g < 12; g += 6) {
            int32_t m[6];
            R w[6], d[6];
            uint8_t mf[6];
#pragma unroll
            for (int q = 0; q < 6; ++q) m[q] = C.mk_i[(g + q) * C.N + k], w[q] = C.mk_w[(g + q) * C.N + k];
#pragma unroll
            for (int q = 0; q < 6; ++q) {
                const int64_t x = m[q] < 0 ? 0 : m[q];   // padded with -1 at the pentagons
                mf[q] = L.nflag[x], d[q] = L.hdet[x];
            }
#pragma unroll
            for (int q = 0; q < 6; ++q)
                if ((m[q] >= 0) & ((mf[q] & (LIVE | WASLIVE)) == (LIVE | WASLIVE))) s -= w[q] * d[q];
        }
        L.dh[id] = s;
        return;
    }
    const int64_t i = id;
    if (L.advect) return;   // a prescribed velocity is kept as set
    const uint8_t fi = L.eflag[i];
    const int32_t o = L.fe_ot[i], E = L.fe_ce[i];
    const int fk = L.fe_kind[i];
    if (o < 0) {
        const R Pr = predict(L, C.u, i), d = L.ui[i];
        L.u[i] = Pr + ((fi & WASLIVE) ? d : R(0));
        return;
    }
    // the halves of a coarse edge share their predictions: the first half's item writes
    // both when both are live
    const uint8_t fo = L.eflag[o];
    if ((fk == 1) & ((fo & LIVE) != 0)) return;
    const R Pr = predict(L, C.u, i), Po = predict(L, C.u, o);
    const R uc = C.u[E], de = L.ue[E];
    const R d = ((fi | fo) & WASLIVE) ? de : R(0);
    {
        const R delta = R(0.5) * (R(2) * uc - Pr - Po);
        L.u[i] = Pr + delta + (fk == 0 ? d : -d);
    }
    if (fo & LIVE) {
        const R delta = R(0.5) * (R(2) * uc - Po - Pr);
        L.u[o] = Po + delta - d;
    }
}

// (b) odd nodes from the even ones
template <class R>
__device__ __forceinline__ void inverse_b_item(const DevLevelT<R>& L, int64_t id) {
    const uint8_t f = L.nflag[id];
    const int32_t k = L.f2c[id];
    if (k >= 0) return;
    R s = (f & WASLIVE) ? L.hdet[id] : R(0);
#pragma unroll
    for (int q = 0; q < 4; ++q) s += L.ptw[q * L.N + id] * L.dh[L.par[q * L.N + id]];
    L.dh[id] = s;
}

#define ITEMS(KINDS, lvs, one, list, count, P) \
    for_items<KINDS>(lvs, one, list, count, P, [&](const auto& L, int kind, int64_t id, int64_t el)

// restriction from F = level j+1 to C = level j (Sec. 3.1), at a covered node (list
// WL_CN): B by injection
template <class R>
__device__ __forceinline__ void restrict_node(const DevLevelT<R>& L, const DevLevelT<R>& F, int64_t id) {
    if (!L.advect) L.B[id] = F.B[L.c2f[id]];
}

// at an edge with a covered end (list WL_RE): flux by R_F, Coriolis tendency by R_u where
// both ends are covered
template <class R>
__device__ __forceinline__ void restrict_edge(const DevLevelT<R>& L, const DevLevelT<R>& F, int64_t i) {
    const uint8_t both = L.nflag[L.en[i]] & L.nflag[L.en[L.E + i]];
    // the restricted total height flux (mass flux plus the viscous form's diffusive
    // flux) goes to F; the coarse diffusive flux is then zero
    const bool visc = viscous(L);
    R s = R(0);
#pragma unroll
    for (int k = 0; k < 12; ++k) {
        const int32_t f = L.rf_fi[k * L.E + i];
        s += L.rf_fw[k * L.E + i] * (visc ? F.F[f] + F.Fd[f] : F.F[f]);
    }
#pragma unroll
    for (int k = 0; k < 11; ++k) s += L.rf_cw[k * L.E + i] * F.c[L.rf_ci[k * L.E + i]];
    L.F[i] = s / geo<R>(L.l_e, i);
    if (visc) L.Fd[i] = R(0);
    if ((both & COVERED) && !L.advect) L.Q[i] = R(0.5) * (F.Q[L.half[i]] + F.Q[L.half[L.E + i]]);
}

// partial height transform (Eq. Rh) at a covered node of C (list WL_CN) from F = the level
// above: the details of M_k, all live, four at a time (the twelve one after another
// are a chain of 36 loads)
template <class R>
__device__ __forceinline__ void partial_node(const DevLevelT<R>& C, const DevLevelT<R>& F, int64_t id) {
    R s = F.dh[C.c2f[id]];
#pragma unroll
    for (int g = 0; g < 12; g += 4) {
        int32_t m[4];
        R w[4], d[4];
        uint8_t mf[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) m[q] = C.mk_i[(g + q) * C.N + id], w[q] = C.mk_w[(g + q) * C.N + id];
        // a pentagon's padded -1 reads M_k's first node instead, unused
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const int64_t x = m[q] < 0 ? C.mk_i[id] : m[q];
            mf[q] = F.nflag[x], d[q] = height_detail(F, x);
        }
#pragma unroll
        for (int q = 0; q < 4; ++q)
            if ((m[q] >= 0) & ((mf[q] & LIVE) != 0)) s += w[q] * d[q];
    }
    C.dh[id] = s;
}

// ---------------------------------------------------------------------------- mask items (Sec. 2.3)

// significance at level F (Sec. 2.3): odd node with |h~| >= eps_h; both ends of an
// interior edge with |u~| >= eps_u; both ends and the midpoint of a coarse edge with
// |u~_E| >= eps_u; only points live before the adaptation carry coefficients
// The significance threshold e (FP64) as a threshold of the field type: the least
// R value >= e, so that |x| >= e and |x| >= sig_thr<R>(e) agree for every x of type
// R (infinity and NaN included); the tests below then compare in R.
template <class R>
__device__ __forceinline__ R sig_thr(double e);
template <>
__device__ __forceinline__ double sig_thr<double>(double e) { return e; }
template <>
__device__ __forceinline__ float sig_thr<float>(double e) { return __double2float_ru(e); }

// at a live node
template <class R>
__device__ __forceinline__ bool sig_node(const DevLevelT<R>& F, int64_t i, R eh) {
    const int32_t k = F.f2c[i];
    const R d = F.hdet[i];
    if ((k < 0) & (fabs(d) >= eh)) {
        F.sig[i] = 1;
        return true;
    }
    return false;
}

// at a live edge: its own coefficient, or its coarse edge's (pair_at)
template <class R>
__device__ __forceinline__ bool sig_edge(const DevLevelT<R>& F, const DevLevelT<R>& C, int64_t i, R eu) {
    const int32_t o = F.fe_ot[i], E = F.fe_ce[i];
    const int k = F.fe_kind[i];
    if (o < 0) {
        if (!(fabs(F.ui[i]) >= eu)) return false;
        F.sig[F.en[i]] = 1;
        F.sig[F.en[F.E + i]] = 1;
        return true;
    }
    const uint8_t fo = F.eflag[o];
    const R d = F.ue[E];
    if (!(pair_at(k, fo) & (fabs(d) >= eu))) return false;
    F.sig[C.c2f[C.en[E]]] = 1;
    F.sig[C.c2f[C.en[C.E + E]]] = 1;
    F.sig[C.mid[E]] = 1;
    return true;
}

// T = S + same-level neighbours of S + children of the coarser significance set; a
// patch the learned proposal names joins T as a whole (the exact rules' own set is
// recorded per patch for the proposal's statistics)
template <class R>
__device__ __forceinline__ void adjacent_node(const DevLevelT<R>& F, const DevLevelT<R>& C, bool children, int64_t x) {
    // significance bytes are 0 or 1; each group of loads is issued together
    uint8_t t = F.sig[x];
    if (!t) {
        const int dg = F.deg[x];
        int32_t y[6];
#pragma unroll
        for (int k = 0; k < 6; ++k) y[k] = k < dg ? F.ring_n[k * F.N + x] : int32_t(x);
#pragma unroll
        for (int k = 0; k < 6; ++k) t |= F.sig[y[k]];
        if (!t && children) {
            int32_t cy[7];
            cy[6] = F.f2c[x];
#pragma unroll
            for (int k = 0; k < 6; ++k) cy[k] = F.f2c[y[k]];
#pragma unroll
            for (int k = 0; k < 7; ++k)
                if (cy[k] >= 0) t |= C.sig[cy[k]];
        }
    }
    const int64_t P = patch_of(F, x);
    if (t)
        F.pexact[P] = 1;
    else if (F.prop[P])
        t = 1;
    F.tmask[x] = t;
}

// graded closure at level F: coarse node of a live node of the finer level Fp, and
// the prediction parents of every live odd node (only ever sets bytes to 1)
template <class R>
__device__ __forceinline__ void close_node(const DevLevelT<R>& F, const DevLevelT<R>& Fp, bool has_finer, int64_t x) {
    uint8_t t = F.tmask[x];
    if (has_finer && Fp.tmask[F.c2f[x]]) t = 1;
    if (!t) return;
    F.tmask[x] = 1;
    if (F.f2c[x] < 0) {
#pragma unroll
        for (int q = 0; q < 4; ++q) F.tmask[F.par[q * F.N + x]] = 1;
    }
}

// live flag (every node when `all`, else the mask), remembering whether it was live
template <class R>
__device__ __forceinline__ uint8_t live_node(const DevLevelT<R>& L, int64_t i, bool all) {
    const uint8_t lv = all ? 1 : L.tmask[i];
    L.nflag[i] = uint8_t((lv ? LIVE : 0) | ((L.nflag[i] & LIVE) ? WASLIVE : 0));
    L.band0[i] = lv;
    return lv;
}

// An edge is live when an end node is: from the closure marks (every node when `all`), not
// from the node flags, so that nodes and edges take their flags in one pass.  counts(x):
// whether the mark of node x makes it live (asked at marked ends only).
template <class R, class Counts>
__device__ __forceinline__ void live_edge(const DevLevelT<R>& L, int64_t e, bool all, Counts counts) {
    const uint8_t was = (L.eflag[e] & LIVE) ? WASLIVE : 0;
    const int32_t a = L.en[e], b = L.en[L.E + e];
    const uint8_t ma = L.tmask[a], mb = L.tmask[b];
    const bool lv = all || (ma && counts(a)) || (mb && counts(b));
    L.eflag[e] = uint8_t((lv ? LIVE : 0) | was);
}

// one neighbour hop of the ghost band: band1 <- dilate(band0) when `forward`,
// band0 <- dilate(band1) otherwise
template <class R>
__device__ __forceinline__ uint8_t dilate_node(const DevLevelT<R>& L, int64_t x, bool forward) {
    const uint8_t* __restrict__ in = forward ? L.band0 : L.band1;
    uint8_t* __restrict__ out = forward ? L.band1 : L.band0;
    // band bytes are 0 or 1; the neighbours' loads are issued together
    uint8_t t = in[x];
    if (!t) {
        const int dg = L.deg[x];
#pragma unroll
        for (int k = 0; k < 6; ++k)
            if (k < dg) t |= in[L.ring_n[k * L.N + x]];
    }
    out[x] = t;
    return t;
}

template <class R>
__device__ __forceinline__ void ghost_node(const DevLevelT<R>& L, int64_t i, const uint8_t* band) {
    if (!(L.nflag[i] & LIVE) && band[i]) L.nflag[i] |= GHOST;
}

template <class R>
__device__ __forceinline__ void ghost_edge(const DevLevelT<R>& L, int64_t e, const uint8_t* band) {
    if (!(L.eflag[e] & LIVE) && band[L.en[e]] && band[L.en[L.E + e]]) L.eflag[e] |= GHOST;
}

// covered coarse node: the fine node at the same place and all of M_k live
template <class R>
__device__ __forceinline__ void covered_node(const DevLevelT<R>& C, const DevLevelT<R>& F, int64_t k) {
    if (!(F.nflag[C.c2f[k]] & LIVE)) return;
    bool all = true;   // the loads issued together (no early exit)
#pragma unroll
    for (int q = 0; q < 12; ++q) {
        const int32_t m = C.mk_i[q * C.N + k];
        if (m >= 0 && !(F.nflag[m] & LIVE)) all = false;
    }
    if (all) C.nflag[k] |= COVERED;
}

// ---------------------------------------------------------------------------- patch lists (Sec. 5.2)

// the 32 bytes flag[i0..) (those below n) as bits; flag + i0 is 16-byte aligned
__device__ __forceinline__ unsigned flag_bits(const uint8_t* __restrict__ flag, int64_t i0, int64_t n) {
    unsigned bits = 0u;
    if (i0 + 32 <= n) {
        const uint4 a = *reinterpret_cast<const uint4*>(flag + i0);
        const uint4 b = *reinterpret_cast<const uint4*>(flag + i0 + 16);
        const unsigned words[8] = {a.x, a.y, a.z, a.w, b.x, b.y, b.z, b.w};
#pragma unroll
        for (int q = 0; q < 8; ++q)
#pragma unroll
            for (int k = 0; k < 4; ++k) bits |= (((words[q] >> (8 * k)) & 0xffu) ? 1u : 0u) << (4 * q + k);
    } else {
        for (int k = 0; k < 32 && i0 + k < n; ++k) bits |= (flag[i0 + k] ? 1u : 0u) << k;
    }
    return bits;
}

// The indices of the nonzero bytes of flag[0..n) into out (tag | index), in
// ascending order, by one block: each thread takes 32 consecutive flags per pass
// (two 16-byte loads), the block forms an exclusive prefix of the counts, and each
// thread writes its entries, to out and to out2.  flag must be 16-byte aligned.  Returns
// the count (in every thread).
__device__ int compact_flags(const uint8_t* __restrict__ flag, int64_t n, int32_t tag, int32_t* __restrict__ out,
                             int32_t* __restrict__ out2) {
    __shared__ int wsum[32];
    __shared__ int total;
    if (threadIdx.x == 0) total = 0;
    __syncthreads();
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, nw = blockDim.x >> 5;
    for (int64_t start = 0; start < n; start += 32 * int64_t(blockDim.x)) {
        const int64_t i0 = start + 32 * int64_t(threadIdx.x);
        unsigned bits = flag_bits(flag, i0, n);
        const int cnt = __popc(bits);
        int incl = cnt;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int v = __shfl_up_sync(0xffffffffu, incl, o);
            if (lane >= o) incl += v;
        }
        if (lane == 31) wsum[w] = incl;
        __syncthreads();
        if (w == 0) {
            int v = lane < nw ? wsum[lane] : 0, iv = v;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int t = __shfl_up_sync(0xffffffffu, iv, o);
                if (lane >= o) iv += t;
            }
            if (lane < nw) wsum[lane] = iv - v;   // exclusive prefix over warps
        }
        __syncthreads();
        int pos = total + wsum[w] + incl - cnt;
        while (bits) {
            const int k = __ffs(bits) - 1;
            out[pos] = out2[pos] = tag | int32_t(i0 + k);
            ++pos;
            bits &= bits - 1u;
        }
        __syncthreads();
        if (threadIdx.x == blockDim.x - 1) total += wsum[w] + incl;
        __syncthreads();
    }
    return total;
}

// Level L's three ascending lists from its patch flags, by one block of any width: the
// active patches (pflag), of these the core (kflag; `whole`: every active patch, as on
// Jmin, which is live in full), and of the core the patches whose tile is not regular;
// each with the pole entry last when a pole is live or ghost.  A thread takes 32 flags
// a pass, and the three counts are prefix-summed together.  The flag arrays are
// 16-byte aligned.
template <class R>
__device__ void patch_scan_level(const DevLevelT<R>& L, bool whole) {
    using U64 = unsigned long long;
    __shared__ U64 wsum[32], total;      // active patches in the low half, core in the high half
    __shared__ unsigned wsum_i[32], total_i;
    const int32_t tag = int32_t(L.J) << LVL_SHIFT;
    const bool all_irr = viscous(L) || L.advect || L.thalo == nullptr;
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, nw = blockDim.x >> 5;
    if (threadIdx.x == 0) total = 0, total_i = 0;
    __syncthreads();
    for (int64_t start = 0; start < L.npatch; start += 32 * int64_t(blockDim.x)) {
        const int64_t i0 = start + 32 * int64_t(threadIdx.x);
        // the three arrays' loads issued together
        const unsigned a = flag_bits(L.pflag, i0, L.npatch);
        const unsigned core = whole ? ~0u : flag_bits(L.kflag, i0, L.npatch);
        const unsigned irr = all_irr ? ~0u : flag_bits(L.tirr, i0, L.npatch);
        const unsigned c = a & core, r = c & irr;
        const U64 cnt = U64(__popc(a)) | U64(__popc(c)) << 32;
        const unsigned cnt_i = __popc(r);
        U64 incl = cnt;
        unsigned incl_i = cnt_i;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const U64 v = __shfl_up_sync(0xffffffffu, incl, o);
            const unsigned vi = __shfl_up_sync(0xffffffffu, incl_i, o);
            if (lane >= o) incl += v, incl_i += vi;
        }
        if (lane == 31) wsum[w] = incl, wsum_i[w] = incl_i;
        __syncthreads();
        if (w == 0) {
            const U64 v = lane < nw ? wsum[lane] : 0;
            const unsigned vi = lane < nw ? wsum_i[lane] : 0;
            U64 iv = v;
            unsigned ii = vi;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const U64 t = __shfl_up_sync(0xffffffffu, iv, o);
                const unsigned ti = __shfl_up_sync(0xffffffffu, ii, o);
                if (lane >= o) iv += t, ii += ti;
            }
            if (lane < nw) wsum[lane] = iv - v, wsum_i[lane] = ii - vi;   // exclusive prefix over warps
        }
        __syncthreads();
        const U64 before = total + wsum[w] + incl - cnt;
        const unsigned before_i = total_i + wsum_i[w] + incl_i - cnt_i;
        auto put = [&](unsigned bits, int32_t* __restrict__ out, unsigned pos) {
            while (bits) {
                out[pos++] = tag | int32_t(i0 + __ffs(bits) - 1);
                bits &= bits - 1u;
            }
        };
        put(a, L.patches, unsigned(before));
        put(c, L.clist, unsigned(before >> 32));
        put(r, L.ilist, before_i);
        __syncthreads();
        if (threadIdx.x == blockDim.x - 1) total = before + cnt, total_i = before_i + cnt_i;
        __syncthreads();
    }
    if (threadIdx.x == 0) {
        int n[LIST_COUNTS] = {int(unsigned(total)), int(total >> 32), int(total_i)};
        if ((L.nflag[L.nelem] | L.nflag[L.nelem + 1]) & AVAIL) {
            const int32_t pole = tag | int32_t(L.npatch);
            L.patches[n[0]++] = pole, L.clist[n[1]++] = pole, L.ilist[n[2]++] = pole;
        }
        for (int q = 0; q < LIST_COUNTS; ++q) L.npatches[q] = n[q];
    }
}

// The all-level lists of levels jmin..jmax from the levels' lists (in level order):
// block j - jmin copies level j's entries behind those of the levels below it, and
// clears the level's work-list counts (the point work lists are rebuilt next).
template <class R>
__device__ void concat_lists(const DevLevelT<R>* __restrict__ lvs, int jmin, int jmax, const GridLists& g) {
    const int j = jmin + int(blockIdx.x);
    if (j > jmax) return;
    int base[LIST_COUNTS] = {0, 0, 0};
    for (int i = jmin; i < j; ++i)
        for (int q = 0; q < LIST_COUNTS; ++q) base[q] += lvs[i].npatches[q];
    const DevLevelT<R>& L = lvs[j];
    const int32_t* src[LIST_COUNTS] = {L.patches, L.clist, L.ilist};
    int32_t* dst[LIST_COUNTS] = {g.all, g.core, g.irr};
    for (int q = 0; q < LIST_COUNTS; ++q) {
        const int n = L.npatches[q];
        for (int i = threadIdx.x; i < n; i += blockDim.x) dst[q][base[q] + i] = src[q][i];
        if (j == jmax && threadIdx.x == 0) g.count[q] = base[q] + n;
    }
    if (threadIdx.x < WL_KINDS && L.wl_n) L.wl_n[threadIdx.x] = 0;
}

// offset of work list k of a level in wl
template <class R>
__device__ __forceinline__ int64_t wl_off(const DevLevelT<R>& L, int k) {
    const int edges = k <= WL_GE ? 0 : k <= WL_RE ? 1 : 2;   // lists of edges before list k
    return (k - edges) * L.N + edges * L.E;
}

// The live points of levels ja..jb of one block's shared copy of the level records, item i
// of n(): off[j - ja] the items before level j.  A thread's items rise, so it steps its
// level up as it goes.  Passes over live points that visited every item of the core
// patches kept under half of their threads busy (41 % of the core's nodes are live on
// the jet at eps 1e-2, 31 % on a 64-member ensemble).
struct LiveItems {
    int off[14], nodes[14];

    // by the whole block, then a block barrier by the caller
    template <class R>
    __device__ void init(const DevLevelT<R>* lv, int ja, int jb) {
        if (threadIdx.x < 32) {
            const int lane = threadIdx.x, j = ja + lane;
            const int nn = j <= jb ? lv[j].wl_n[WL_LN] : 0, n = j <= jb ? nn + lv[j].wl_n[WL_LE] : 0;
            int incl = n;
#pragma unroll
            for (int o = 1; o < 16; o <<= 1) {
                const int v = __shfl_up_sync(0xffffffffu, incl, o);
                if (lane >= o) incl += v;
            }
            if (lane < 14) off[lane] = incl - n, nodes[lane] = nn;
        }
    }
    // items first, first + stride, ...: body(L, kind, id)
    template <class R, class Body>
    __device__ __forceinline__ void run(const DevLevelT<R>* lv, int ja, int jb, int first, int stride, Body body) const {
        int j = ja;
        const int n = off[jb + 1 - ja];
        for (int i = first; i < n; i += stride) {
            while (i >= off[j + 1 - ja]) ++j;
            const DevLevelT<R>& L = lv[j];
            const int nn = nodes[j - ja], k = i - off[j - ja];
            if (k < nn)
                body(L, K_NODE, int64_t(L.wl[wl_off(L, WL_LN) + k]));
            else
                body(L, K_EDGE, int64_t(L.wl[wl_off(L, WL_LE) + (k - nn)]));
        }
    }
};

struct MaxU64 {
    __device__ unsigned long long operator()(unsigned long long x, unsigned long long y) const { return x > y ? x : y; }
};

// block reduction of one word per thread (every thread returns the block's value); sh: a
// word per warp
template <class Op>
__device__ unsigned long long block_reduce_u64(unsigned long long v, Op op, unsigned long long* sh) {
    for (int o = 16; o > 0; o >>= 1) v = op(v, __shfl_down_sync(0xffffffffu, v, o));
    const int w = threadIdx.x >> 5, l = threadIdx.x & 31, nw = blockDim.x >> 5;
    __syncthreads();
    if (l == 0) sh[w] = v;
    __syncthreads();
    if (threadIdx.x == 0) {
        for (int k = 1; k < nw; ++k) v = op(v, sh[k]);
        sh[0] = v;
    }
    __syncthreads();
    return sh[0];
}

// Into red: the largest omega^2 over live nodes (none with a prescribed velocity) and, per
// level, the largest |u| over live edges with u != 0 (NaN left out, as dx/|u| with u NaN
// takes no part).  By whole blocks; sh as above, slev: a word per level.
template <class R>
__device__ __forceinline__ void cfl_maxima(const LiveItems& live, const DevLevelT<R>* lv, int jmin, int jtop, int first, int stride,
                                           double H, double g, unsigned long long* red, unsigned long long* sh,
                                           unsigned long long* slev) {
    if (threadIdx.x < RED_WORDS - RED_LEVEL) slev[threadIdx.x] = 0ull;
    __syncthreads();
    unsigned long long wmax = 0;
    LevelMax um;
    live.run(lv, jmin, jtop, first, stride, [&](const DevLevelT<R>& L, int kind, int64_t id) {
        if (kind == K_NODE) {
            if (!L.advect) wmax = max(wmax, dbits(omega2_at(L, id, H, g)));
        } else {
            const unsigned long long k = abs_key(L.u[id]);
            if (k && k <= inf_key<R>()) um.add(L.J, k, slev);
        }
    });
    um.flush(slev);
    wmax = block_reduce_u64(wmax, MaxU64(), sh);   // synchronises the block: slev is complete
    if (threadIdx.x == 0 && wmax) atomicMax(&red[0], wmax);
    if (threadIdx.x < RED_WORDS - RED_LEVEL && slev[threadIdx.x]) atomicMax(&red[RED_LEVEL + threadIdx.x], slev[threadIdx.x]);
}

// The wavelet coefficients (levels above Jmin) and, in the same pass, max |dh| over live
// nodes and max |u| over live edges of every level into red[2..3]: compared as keys of the
// field type, widened to FP64 once per block (bit patterns of non-negative doubles); the
// details only read dh and u
template <class R>
__device__ __forceinline__ void details_and_maxima(const LiveItems& live, const DevLevelT<R>* lv, int jmin, int jtop, int first,
                                                   int stride, unsigned long long* red, unsigned long long* sh) {
    unsigned long long hmax = 0, umax = 0;
    live.run(lv, jmin, jtop, first, stride, [&](const DevLevelT<R>& L, int kind, int64_t id) {
        if (kind == K_NODE)
            hmax = max(hmax, abs_key(L.dh[id]));
        else
            umax = max(umax, abs_key(L.u[id]));
        if (L.J > jmin) details_item(L, (&L)[-1], kind, id);
    });
    hmax = block_reduce_u64(hmax, MaxU64(), sh);
    umax = block_reduce_u64(umax, MaxU64(), sh);
    if (threadIdx.x == 0) {
        if (hmax) atomicMax(&red[2], dbits(key_value<R>(hmax)));
        if (umax) atomicMax(&red[3], dbits(key_value<R>(umax)));
    }
}

// the thresholds: given (> 0), or relative to the maxima (a prescribed velocity has none)
__device__ __forceinline__ void thresholds(double* thr, const unsigned long long* red, double eps_h, double eps_u, double eps_c,
                                           bool advect) {
    const double h = __longlong_as_double(static_cast<long long>(red[2]));
    const double u = __longlong_as_double(static_cast<long long>(red[3]));
    thr[0] = eps_h > 0 ? eps_h : eps_c * h;
    thr[1] = eps_u > 0 ? eps_u : advect ? INFINITY : eps_c * u;
}

// The point work lists of the entries of `list`, a warp an entry (warp w of nw warps):
// live points, ghost points, covered nodes, edges with a covered end, and
// available nodes with a covered node among themselves and their neighbours (their
// divergence changes with the restricted fluxes).  The warp goes through the entry's
// node and edge slots 256 items at a time, keeps in which lists each belongs, and then
// reserves its room with one addition per list, by a lane each.  (With one addition per
// 32 items they queued on the lists' counters: 260 us for the 52 632 patches of
// turbulence at Jmax 9, 136 us now, the lists of live points included.)  The order of
// the lists is not fixed; every item's work is independent of it.
template <class R>
__device__ __forceinline__ unsigned wl_member(const DevLevelT<R>& L, int kind, int64_t id) {
    if (kind == K_NODE) {
        const uint8_t f = L.nflag[id];
        return ((f & LIVE) ? 1u << WL_LN : 0u) | ((f & GHOST) ? 1u << WL_GN : 0u) | ((f & COVERED) ? 1u << WL_CN : 0u) |
               (restricted_div_node(L, id) ? 1u << WL_DN : 0u);
    }
    const uint8_t f = L.eflag[id];
    const int32_t na = L.en[id], nb = L.en[L.E + id];
    // the first half of a coarse edge fills a ghost second half too (fill_edge)
    bool ge = (f & GHOST) != 0;
    if (ge && L.fe_kind[id] == 1 && (L.eflag[L.fe_ot[id]] & GHOST)) ge = false;
    return ((f & LIVE) ? 1u << WL_LE : 0u) | (ge ? 1u << WL_GE : 0u) | (((L.nflag[na] | L.nflag[nb]) & COVERED) ? 1u << WL_RE : 0u);
}

// one entry of patch area P: its G groups of 32 items from g0 on
template <int P, int G, class R>
__device__ __forceinline__ void wl_groups(const DevLevelT<R>& L, int64_t pat, int g0, int lane) {
    const unsigned below = (1u << lane) - 1u;
    // a group holds nodes (its items below P), edges, or for P = 16 both
    auto holds = [](int g, int k) {
        const bool node = k == WL_GN || k == WL_CN || k == WL_DN || k == WL_LN;
        return node ? g * 32 < P : (g + 1) * 32 > P;
    };
    int32_t id[G];
    unsigned in[G], m[G][WL_KINDS];
    int n = 0;   // lane k: entries of list k
#pragma unroll
    for (int g = 0; g < G; ++g) {
        in[g] = 0u, id[g] = 0;
        auto body = [&](const DevLevelT<R>& LL, int kind, int64_t i, int64_t) {
            id[g] = int32_t(i);
            in[g] = wl_member(LL, kind, i);
        };
        visit_item<K_NODE | K_EDGE>(L, pat, uint32_t((g0 + g) * 32 + lane), P, body);
    }
    __syncwarp();
#pragma unroll
    for (int g = 0; g < G; ++g)
#pragma unroll
        for (int k = 0; k < WL_KINDS; ++k)
            if (holds(g0 + g, k)) {
                m[g][k] = __ballot_sync(0xffffffffu, in[g] >> k & 1u);
                if (lane == k) n += __popc(m[g][k]);
            }
    int at = 0;
    if (lane < WL_KINDS && n) at = atomicAdd(&L.wl_n[lane], n);
#pragma unroll
    for (int k = 0; k < WL_KINDS; ++k) {
        int pos = __shfl_sync(0xffffffffu, at, k);
        int32_t* __restrict__ out = L.wl + wl_off(L, k);
#pragma unroll
        for (int g = 0; g < G; ++g)
            if (holds(g0 + g, k)) {
                if (in[g] >> k & 1u) out[pos + __popc(m[g][k] & below)] = id[g];
                pos += __popc(m[g][k]);
            }
    }
}

template <int P, class R>
__device__ __forceinline__ void wl_entries(const DevLevelT<R>* __restrict__ lvs, const int32_t* __restrict__ list,
                                           int count, int w, int nw) {
    constexpr int NG = 4 * P / 32, G = NG < 8 ? NG : 8;
    for (int t = w; t < count; t += nw) {
        const int32_t ent = list[t];
        const DevLevelT<R>& L = lvs[ent >> LVL_SHIFT];
#pragma unroll
        for (int g0 = 0; g0 < NG; g0 += G) wl_groups<P, G>(L, int64_t(ent & PATCH_MASK), g0, int(threadIdx.x & 31));
    }
}

template <class R>
__device__ __forceinline__ void wl_build(const DevLevelT<R>* __restrict__ lvs, const int32_t* __restrict__ list, int count,
                                         int P, int w, int nw) {
    if (P == 64)
        wl_entries<64>(lvs, list, count, w, nw);
    else if (P == 16)
        wl_entries<16>(lvs, list, count, w, nw);
    else
        wl_entries<256>(lvs, list, count, w, nw);
}

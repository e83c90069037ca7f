// Host-side launchers of the kernels in sww_kernels.cu.
#pragma once
#include <cuda_runtime.h>

#include <cstdint>

#include "sww_core.cuh"

namespace sww {

// One Runge-Kutta stage: y <- a*y0 + b*y + (cdt*dt)*k + (ddt*dt)*acc, acc <- al*acc + be*k
// (nothing written to acc when both are 0).  apply == 0 only stores the trend k.  base:
// the base y0 is this stage's y (the first stage stores it).  trend: k is stored (the last
// stage of a step, whose trend stays readable).
struct RKStage {
    int apply;
    double a, b, cdt, ddt, al, be;
    int base, trend;
};

// The same in the working precision with its tests taken: made on the host and passed
// with the launch.  (Made by each thread, its six conversions and six FP64 comparisons
// held the FP64 pipe, one warp instruction per 16 clocks, for 13 us of an update over
// 13 640 patches and 3 us of a persistent stage.)
template <class R>
struct StageCoef {
    R a, b, cdt, ddt, al, be;
    bool apply, ha, hb, hddt, hacc, hal, base, trend;
    StageCoef() = default;
    StageCoef(const RKStage& s)
        : a(R(s.a)), b(R(s.b)), cdt(R(s.cdt)), ddt(R(s.ddt)), al(R(s.al)), be(R(s.be)), apply(s.apply != 0),
          ha(s.a != 0.0), hb(s.b != 0.0), hddt(s.ddt != 0.0), hacc(s.al != 0.0 || s.be != 0.0), hal(s.al != 0.0),
          base(s.base != 0), trend(s.trend != 0) {}
};

// A work list on the device: entries (level-tagged patches), their count, the
// device array of levels (for multi-level lists; null for a single level's list),
// threads per entry S (the configured patch area) and the fixed grid size.
template <class R>
struct WorkT {
    const DevLevelT<R>* lvs;
    const int32_t* list;
    const int32_t* count;
    int S;
    unsigned grid;
};

// The all-level lists of a handle (level order, ascending patches): every active patch,
// the core (CORE_HOPS), and of the core the entries whose tile is not regular, with their
// lengths in count[0..2].
struct GridLists {
    int32_t *all, *core, *irr;
    int32_t* count;
};

// Levels ja..jb of a multi-level dense launch; off[j - ja] is the first thread of
// level j and off[jb + 1 - ja] the total.  Level tail_j (-1: none; only ever jb) is a
// tail level of tail_n items covered by a fixed number of striding threads.
struct Span {
    int ja, jb;
    int64_t off[14];
    int tail_j;
    int64_t tail_n;
};

// Arguments of the mask construction over levels ja..jb (ja = Jmin).
template <class R>
struct MaskArgsT {
    const DevLevelT<R>* lvs;    // device array of levels
    const DevLevelT<R>* host;   // the same levels on the host
    int ja, jb, hops;
    const double* thr;          // eps_h, eps_u on the device
    Span nodes_f, edges_f;      // levels ja+1..jb: nodes, edges
    Span nodes, edges;          // levels ja..jb
    Span nodes_c;               // levels ja..jb-1: nodes
    Span patches;               // levels ja..jb: patches
    int32_t* sig_any;           // [sig_any_len] per level: any significant point (device)
    int sig_any_len;
    unsigned tail_blocks;       // blocks of a per-level launch on the tail level
    unsigned long long* lstat;  // learned-proposal counters (misses, over, proposed) or null
};

// Launchers; R = double (FP64 form) or float (FP32 form), instantiated for both.
// dense level kernels (masks, initialisation, diagnostics)
template <class R> void launch_restrict_full(const DevLevelT<R>& C, const DevLevelT<R>& F, cudaStream_t s);
// full level F from the full level below (zero coefficients away from live points)
template <class R>
void launch_uniform(const DevLevelT<R>& F, const DevLevelT<R>& C, const R* cdh, const R* cu, R* odh, R* ou,
                    cudaStream_t s);
// WASLIVE := LIVE on the listed patches (inverse transform of the stored coefficients)
template <class R> void launch_mark_support(const WorkT<R>& W, cudaStream_t s);
// significance, adjacency, closure, live flags, ghost band, covered nodes and
// patch lists of levels a.ja..a.jb
template <class R> void launch_mask(const MaskArgsT<R>& a, cudaStream_t s);
// every point of levels edges.ja..edges.jb live; covered flags; patch lists
template <class R> void launch_live_all(const DevLevelT<R>* lvs, const Span& edges, cudaStream_t s);
template <class R> void launch_covered_all(const DevLevelT<R>* lvs, const Span& nodes_c, cudaStream_t s);
template <class R> void launch_patches_all(const DevLevelT<R>* lvs, const Span& patches, cudaStream_t s);
// the all-level lists from the levels' lists, and the levels' point work lists (patch
// area P; grid: blocks of the list launch)
template <class R>
void launch_concat(const DevLevelT<R>* lvs, int jmin, int jmax, const GridLists& lists, int P, unsigned grid,
                   cudaStream_t s);
template <class R> int sums_blocks(const DevLevelT<R>& L);
template <class R>
void launch_sums(const DevLevelT<R>& L, double H, double g, double* part, double* out, cudaStream_t s);
template <class R> void launch_count(const DevLevelT<R>& L, unsigned long long* cnt, cudaStream_t s);
// y[i] = B(x[i]) (double <-> float)
template <class A, class B> void launch_convert(const A* x, B* y, int64_t n, cudaStream_t s);

// Process-wide number of library kernel launches (count_launch adds launches made
// outside the launchers above).
int64_t kernel_launches();
void count_launch(int64_t n);

}  // namespace sww

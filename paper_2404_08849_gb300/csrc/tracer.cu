// tracer.cu - tracer transport, Eq. 10 (horizontal part), Sec. 2.1:
// third-order upwind edge flux, Wicker-Skamarock RK3, Zalesak FCT on the
// final stage; FP64 or single-precision tracers (Sec. 2.3) with an FP64
// mass flux and FP64 layer mass.
//
// Batching (ensembles of uneven members, Sec. 4.3 ensemble runs): every
// phase of the step is one pass over a flat work list that concatenates,
// for each member m and tracer group g (tracers_per_thread tracers), the
// (entity, level) index space of that member; a segment table maps a flat
// index to (m, g) by binary search, cached per thread across grid-stride
// iterations.  The phases run either as one launch each or inside one
// persistent cooperative kernel separated by bounded grid barriers.
//
// In binary32 these kernels are bound by instruction issue, the L1 data pipe and
// latency, in binary64 by the FP64 pipe; conversions run in integers (cv), as
// the hardware's issue on that pipe.
//
// Data layout: q [T][nC][ld], dpi [nC][ld], mass flux [nE][ld], edge
// fluxes [T][nE][ld]; consecutive threads take consecutive levels of one
// entity (coalesced rows), neighbour rows are gathered through L1/L2.
//
// A work item is a vector of 4 or 2 binary32 or 2 binary64 levels where the
// member's rows allow it (vec_class): with one level per 4-byte access the
// L1 data pipe (79 % of its wavefronts) and the latency of many small gathers
// bounded the binary32 phases.  Level-7 mesh, 4 tracers, 60 levels, binary32,
// us per launch, one level / vectors: div 231 / 145, edge 365 / 231, update
// 226 / 148 (then at the DRAM rate), ratios 545 / 345 (half of it the
// division's slow path, see fct_ratio), final 440 / 307, low-order 270 / 128
// more in the first edge phase; the step 3316 / 2001 with the vertical transport
// as it stands.  binary64 is bound by the FP64 pipe and gains little from the
// width.
#include <algorithm>
#include <cmath>
#include <cstring>
#include <vector>

#include "common.cuh"
#include "forms.cuh"

#define PN(n) (sizeof(TC) == 4 ? n "/mix" : n "/fp64")

namespace grist {

struct MemberDev {
    void *q;                // [T][nC][ld] caller's tracers (q^n in, q^{n+1} out)
    const double *dpi;      // [nC][ld]
    const double *F;        // [nE][ld]
    void *qA, *qB;          // scratch stage tracers [T][nC][ld]
    void *FH;               // scratch edge fluxes [T][nE][ld]; A = F^H - F^L in a limited final stage
    void *R2;               // scratch FCT ratios {R+, R-} [T][nC][ld] pairs in the compute type
    void *X2;               // scratch FCT local bounds {max, min}(q^n, q^td) [T][nC][ld] pairs
    void *DFL;              // scratch FCT div F^L [T][nC][ld] in the compute type
    const void *Ff;         // mass flux in the compute type [nE][ld]: a binary32 copy (scratch) or F itself
    void *DV;               // scratch {dpi, div F} pairs in the compute type [nC][ld]
    int L, T, ld, pad;
    const double *Mv;       // time-mean vertical mass flux [nC][ldi] or null (no vertical step)
    int ldi;
    LevelDiv DL;            // division by Lg
    int Lg;                 // level groups of a thread: V consecutive levels from g V, or levels g, g + Lg, ...
    unsigned long long qs, fs;  // nC*ld, nE*ld
};

// A flat work space: segment s covers [start[s], start[s+1]) and belongs to
// member mg[s].x, tracer group mg[s].y; within a segment the local index r
// is entity * L + level.
struct Space {
    const unsigned long long *start;  // [nseg + 1]
    const int2 *mg;                   // [nseg]
    int nseg;
    unsigned long long total;
};

// Tiles of consecutive (space-filling-curve) cells for the fused stage
// kernel: per tile the halo cells its edge fluxes read (the tile, its
// neighbours and theirs), its edges, and for every tile edge the halo-local
// indices of c1, c2 and the two deriv-two stencils; per tile cell the
// tile-local index of each of its six edges.
constexpr int kTileCells = 32;

struct TileMesh {
    int ntiles, Hmax, Emax;
    const int *hoff;           // [ntiles + 1]
    const int *halo;           // global cell ids
    const int *eoff;           // [ntiles + 1]
    const int *tedge;          // global edge ids
    const uint16_t *eloc;      // [edges][16]: c1, c2, stencil side 0 (7), side 1 (7)
    const uint16_t *cle;       // [ntiles * kTileCells][6]
};

struct TracerCtx {
    grist_tracer_tuning tune{128, 4, 0, 0, 0, 2, 1};
    // tile tables (built on first use)
    char *dtile = nullptr;
    TileMesh tiles{};
    // work-list tables (member descriptors, segment tables), one device copy
    // per distinct batch, never rewritten: a step recorded in a graph keeps
    // reading the table it was recorded with, whatever other batches run
    // in between.  cur: the table of the last planned batch.
    struct Table {
        std::vector<char> host;
        char *dev = nullptr;
    };
    std::vector<Table> tabs;
    int cur = -1;
    unsigned *barrier = nullptr;  // [0] arrival count, [1] generation, [2] abort, [3] self-test word
    // graph cache: the last few captured steps, keyed by their signature
    // (buffers, sizes, dt, tuning, stream) - alternating buffer sets, as in
    // a pipelined caller, each keep their graph
    struct GraphEntry {
        std::vector<unsigned long long> sig;
        cudaGraph_t graph = nullptr;
        cudaGraphExec_t exec = nullptr;
    };
    std::vector<GraphEntry> graphs;
    bool graph_failed = false;
    std::vector<unsigned long long> failed_sig;

    void drop_graphs() {
        for (auto &g : graphs) {
            if (g.exec) cudaGraphExecDestroy(g.exec);
            if (g.graph) cudaGraphDestroy(g.graph);
        }
        graphs.clear();
    }
};

constexpr size_t kGraphCache = 4;
constexpr size_t kTableCache = 64;   // distinct batches whose tables a handle keeps

void tracer_ctx_free(TracerCtx *c) {
    if (!c) return;
    c->drop_graphs();
    for (auto &t : c->tabs)
        if (t.dev) cudaFree(t.dev);
    if (c->dtile) cudaFree(c->dtile);
    if (c->barrier) cudaFree(c->barrier);
    delete c;
}

namespace {

constexpr long long kBarrierSpinLimit = 20000000;  // x ~64 ns sleep: about a second
constexpr int kVertMaxL = 128;   // levels supported by the vertical transport
// Largest block of the work-list kernels (their register use, at most 128
// per thread, lets every block up to this size launch).
constexpr int kTracerMaxBlock = 512;
// Widths of a work item's level vector: 1, 2 or 4 consecutive levels.
constexpr int kVecClasses = 3;

struct Batch {
    const MemberDev *mem;
    int nm;
    // D: cell x level (no groups); C: cell x level x group; E: edge x level x
    // group; each by the members' vector width (class c: 2^c levels)
    Space D[kVecClasses], C[kVecClasses], E[kVecClasses];
    Space T;        // blocks of the fused stage kernel: segment start = first block of (member, group)
    int tpt;
    int lpt;        // levels per thread of the work-list phases (1 or 2; the persistent launch takes 1)
    double dt;
    double dt3;     // dt / 3, the first RK stage (formed on the host)
    int fct;
    int beta1;
    int ring;       // the edge phases run cell-centrically (item_edge_ring) over the space C
    double beta;
    double cmax;    // vertical transport: largest explicit Courant number
};

// Cached segment lookup: returns the segment of flat index n, reusing seg
// when n still lies inside it.
__device__ __forceinline__ int find_seg(const Space &S, unsigned long long n, int seg) {
    if (seg >= 0 && n >= S.start[seg] && n < S.start[seg + 1]) return seg;
    int lo = 0, hi = S.nseg - 1;
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (S.start[mid] <= n) lo = mid;
        else hi = mid - 1;
    }
    return lo;
}

// Loads of arrays that a phase writes and a later phase reads.  Inside the
// persistent kernel such data changes during the launch, so it is read
// coherently at L2 (ld.global.cg); across separate launches the read-only
// path is safe.
template <bool PERS, typename T> __device__ __forceinline__ T lds(const T *p) {
    return PERS ? __ldcg(p) : __ldg(p);
}

template <typename TC> __device__ __forceinline__ TC tiny_of();
template <> __device__ __forceinline__ double tiny_of<double>() { return 2.2250738585072014e-308; }
template <> __device__ __forceinline__ float tiny_of<float>() { return 1.17549435e-38f; }

// ---------------------------------------------------------------------------
// phase bodies (one work item each)

// {dpi, div F} pair in the compute type.
template <typename TC> struct Vec2;
template <> struct Vec2<float> { using T = float2; };
template <> struct Vec2<double> { using T = double2; };

// Stage ratios r1 = dpi^n / dpi^(s) and r2 = dt_s / dpi^(s) of the update
// q^(s) = r1 q^n - r2 div F^H, with dpi^(s) = dpi^n - dt_s div F: FP64 in the
// FP64 policy (the oracle's arithmetic); in the binary32 policy in binary32
// from the rounded pair, so the binary32 phases issue no FP64 instruction
// (the ratios are rounded to binary32 either way).
__device__ __forceinline__ void stage_ratios(double2 dv, double dts, float, double &r1, double &r2) {
    const double rinv = rcp(dv.x - dts * dv.y);
    r1 = dv.x * rinv;
    r2 = dts * rinv;
}
__device__ __forceinline__ void stage_ratios(float2 dv, double, float dtsf, float &r1, float &r2) {
    const float rinv = __frcp_rn(fmaf(-dtsf, dv.y, dv.x));
    r1 = dv.x * rinv;
    r2 = dtsf * rinv;
}
// Layer mass at the end of the step, dpi^n - dt div F, in the compute type.
__device__ __forceinline__ double end_mass(double2 dv, double dt, float) { return dv.x - dt * dv.y; }
__device__ __forceinline__ float end_mass(float2 dv, double, float dtf) { return fmaf(-dtf, dv.y, dv.x); }

// Vectors of V consecutive levels (V * sizeof(T) up to 32 bytes), moved as 8-
// or 16-byte accesses; plan_batch gives a member only a V that its rows and
// pointers are aligned to.  PERS as in lds().
template <bool PERS, int V, typename T> __device__ __forceinline__ void ldv(const T *p, T (&o)[V]) {
    if constexpr (V == 1) {
        o[0] = lds<PERS>(p);
    } else if constexpr (sizeof(T) * V == 8) {
        const float2 a = lds<PERS>((const float2 *)p);
        o[0] = a.x; o[1] = a.y;
    } else if constexpr (sizeof(T) == 4) {
#pragma unroll
        for (int j = 0; j < V; j += 4) {
            const float4 a = lds<PERS>((const float4 *)(p + j));
            o[j] = a.x; o[j + 1] = a.y; o[j + 2] = a.z; o[j + 3] = a.w;
        }
    } else {
#pragma unroll
        for (int j = 0; j < V; j += 2) {
            const double2 a = lds<PERS>((const double2 *)(p + j));
            o[j] = a.x; o[j + 1] = a.y;
        }
    }
}
template <int V, typename T> __device__ __forceinline__ void stv(T *p, const T (&o)[V]) {
    if constexpr (V == 1) {
        *p = o[0];
    } else if constexpr (sizeof(T) * V == 8) {
        *(float2 *)p = make_float2(o[0], o[1]);
    } else if constexpr (sizeof(T) == 4) {
#pragma unroll
        for (int j = 0; j < V; j += 4) *(float4 *)(p + j) = make_float4(o[j], o[j + 1], o[j + 2], o[j + 3]);
    } else {
#pragma unroll
        for (int j = 0; j < V; j += 2) *(double2 *)(p + j) = make_double2(o[j], o[j + 1]);
    }
}
// The caller's q^n where the same launch overwrites it in place (each thread
// its own levels): an ordinary load.
template <int V, typename T> __device__ __forceinline__ void ldv_own(const T *p, T (&o)[V]) {
    if constexpr (V == 1) {
        o[0] = *p;
    } else if constexpr (sizeof(T) * V == 8) {
        const float2 a = *(const float2 *)p;
        o[0] = a.x; o[1] = a.y;
    } else if constexpr (sizeof(T) == 4) {
#pragma unroll
        for (int j = 0; j < V; j += 4) {
            const float4 a = *(const float4 *)(p + j);
            o[j] = a.x; o[j + 1] = a.y; o[j + 2] = a.z; o[j + 3] = a.w;
        }
    } else {
#pragma unroll
        for (int j = 0; j < V; j += 2) {
            const double2 a = *(const double2 *)(p + j);
            o[j] = a.x; o[j + 1] = a.y;
        }
    }
}

// The {dpi, div F} pairs of V levels: d[2 v], d[2 v + 1].
template <bool PERS, typename TC, int V>
__device__ __forceinline__ void dv_at(const MemberDev &mb, size_t x, typename Vec2<TC>::T (&o)[V]) {
    TC d[2 * V];
    ldv<PERS, 2 * V>((const TC *)mb.DV + 2 * x, d);
#pragma unroll
    for (int v = 0; v < V; v++) o[v] = typename Vec2<TC>::T{d[2 * v], d[2 * v + 1]};
}

// A cell's edges, neighbours and divergence weights, read once per work
// item (rows of 8, 16-byte vectors) and shared by its levels.
static_assert(GRIST_MAXE == 6, "cell rows hold 6 entries");
template <typename TW> struct CellRow {
    int e[GRIST_MAXE], nb[GRIST_MAXE];
    TW cw[GRIST_MAXE];
};
template <bool NB, typename TW>
__device__ __forceinline__ void load_cell_row(const DevMesh &m, int i, CellRow<TW> &r) {
    load_row6(m.eoc8, i, r.e);
    if (NB) load_row6(m.coc8, i, r.nb);
    load_row6(Coef<TW>::cdiv8(m), i, r.cw);
}

// Tracer continuity of the member: div F of the FP64 time-mean mass flux,
// summed in FP64, stored with dpi^n as the {dpi, div F} pair of the later
// phases (rounded to binary32 in the binary32 policy).  In that policy each
// edge's flux is also rounded once to binary32 for the later phases (by the
// cell it leaves: positive divergence coefficient), so they read 4 bytes
// per edge-level instead of 8.
template <typename TC, int V>
__device__ __forceinline__ void item_div(const MemberDev &mb, const CellRow<double> &r, int i, int k) {
    double s[V];
#pragma unroll
    for (int v = 0; v < V; v++) s[v] = 0.0;
#pragma unroll
    for (int j = 0; j < GRIST_MAXE; j++) {
        const size_t y = (size_t)r.e[j] * mb.ld + k;
        const double cw = r.cw[j];
        double f[V];
        ldv<false, V>(mb.F + y, f);
#pragma unroll
        for (int v = 0; v < V; v++) s[v] += cw * f[v];
        if constexpr (sizeof(TC) == 4) {
            if (cw > 0.0) {
                float g[V];
#pragma unroll
                for (int v = 0; v < V; v++) g[v] = cv<float>(f[v]);
                stv<V>((float *)mb.Ff + y, g);
            }
        }
    }
    const size_t x = (size_t)i * mb.ld + k;
    double dp[V];
    ldv<false, V>(mb.dpi + x, dp);
    TC d[2 * V];
#pragma unroll
    for (int v = 0; v < V; v++) {
        d[2 * v] = cv<TC>(dp[v]);
        d[2 * v + 1] = cv<TC>(s[v]);
    }
    stv<2 * V>((TC *)mb.DV + 2 * x, d);
}

// Mass flux of V levels from edge-level x in the compute type: the binary32
// copy made by the continuity phase (read coherently inside the persistent
// launch, which wrote it), or the caller's FP64 array.
template <bool PERS, int V, typename TC>
__device__ __forceinline__ void flux_at(const MemberDev &mb, size_t x, TC (&f)[V]) {
    if constexpr (sizeof(TC) == 4) ldv<PERS, V>((const float *)mb.Ff + x, f);
    else ldv<false, V>(mb.F + x, f);
}

// Products and sums of the limiter written with explicit rounding, so the
// edge-centric and cell-centric forms (different kernels) give the same
// bits: F^L = F q^n_upwind, A = F^H - F^L = F (q_e - q^n_upwind), div F^L
// summed by fused multiply-adds in edge order, q^td = r1 q^n - r2 div F^L.
__device__ __forceinline__ float mul_rn(float a, float b) { return __fmul_rn(a, b); }
__device__ __forceinline__ double mul_rn(double a, double b) { return __dmul_rn(a, b); }
__device__ __forceinline__ float sub_rn(float a, float b) { return __fsub_rn(a, b); }
__device__ __forceinline__ double sub_rn(double a, double b) { return __dsub_rn(a, b); }
__device__ __forceinline__ float fma_rn(float a, float b, float c) { return __fmaf_rn(a, b, c); }
__device__ __forceinline__ double fma_rn(double a, double b, double c) { return __fma_rn(a, b, c); }
template <typename TC> __device__ __forceinline__ TC antidiff(TC f, TC qe, TC qup) { return mul_rn(f, sub_rn(qe, qup)); }
template <typename TC> __device__ __forceinline__ TC lowres_value(TC r1, TC r2, TC qn, TC divl) {
    return fma_rn(r1, qn, -mul_rn(r2, divl));
}

// Third-order upwind edge flux (Skamarock-Gassmann form):
//   q_e = (q1 + q2)/2 - (dc^2/12)(q''1 + q''2) + sgn(F) beta (dc^2/12)(q''2 - q''1)
// F^H = F q_e, on V levels of one edge.  With beta = 1 only the upwind side's
// second derivative survives: q_e = (q1 + q2)/2 - 2 (dc^2/12) q''_upwind
// (V = 1 here: the levels of a vector may have different upwind sides).
// In the final stage of a limited step (qn = q^n) the phase stores the
// antidiffusive flux A = F^H - F^L instead of F^H.
template <bool PERS, typename TQ, typename TC, int V>
__device__ __forceinline__ void item_edge(const DevMesh &m, const MemberDev &mb, const TQ *q, const TQ *qn, int t0,
                                          int t1, int e, int k, bool beta1, TC beta) {
    const int ld = mb.ld;
    const int2 c = ldg(m.coe + e);
    TC f[V];
    flux_at<PERS, V>(mb, (size_t)e * ld + k, f);
    const TC dc2 = ldg(Coef<TC>::dc2(m) + e);
    const int32_t *st = m.d2i + (size_t)e * 14;
    const TC *cf = Coef<TC>::d2c(m) + (size_t)e * 14;
    TC *FH = (TC *)mb.FH;
    for (int t = t0; t < t1; t++) {
        const TQ *qt = q + (size_t)t * mb.qs + k;
        TC q1[V], q2[V], qe[V], a[V], b[V];
        ldv<PERS, V>(qt + (size_t)c.x * ld, q1);
        ldv<PERS, V>(qt + (size_t)c.y * ld, q2);
        if (V == 1 && beta1) {
            const int side = f[0] >= (TC)0 ? 0 : 1;
            TC d = 0;
#pragma unroll
            for (int j = 0; j < GRIST_D2P; j++) {
                ldv<PERS, V>(qt + (size_t)ldg(st + side * GRIST_D2P + j) * ld, a);
                d += ldg(cf + side * GRIST_D2P + j) * a[0];
            }
            qe[0] = (TC)0.5 * (q1[0] + q2[0]) - (TC)2 * dc2 * d;
        } else {
            TC d1[V], d2[V];
#pragma unroll
            for (int v = 0; v < V; v++) d1[v] = d2[v] = 0;
#pragma unroll
            for (int j = 0; j < GRIST_D2P; j++) {
                ldv<PERS, V>(qt + (size_t)ldg(st + j) * ld, a);
                ldv<PERS, V>(qt + (size_t)ldg(st + GRIST_D2P + j) * ld, b);
                const TC w1 = ldg(cf + j), w2 = ldg(cf + GRIST_D2P + j);
#pragma unroll
                for (int v = 0; v < V; v++) {
                    d1[v] += w1 * a[v];
                    d2[v] += w2 * b[v];
                }
            }
#pragma unroll
            for (int v = 0; v < V; v++) {
                const TC sgn = f[v] >= (TC)0 ? (TC)1 : (TC)-1;
                qe[v] = (TC)0.5 * (q1[v] + q2[v]) - dc2 * (d1[v] + d2[v]) + sgn * beta * dc2 * (d2[v] - d1[v]);
            }
        }
        if (qn) {
            ldv<PERS, V>(qn + (size_t)t * mb.qs + (size_t)c.x * ld + k, a);
            ldv<PERS, V>(qn + (size_t)t * mb.qs + (size_t)c.y * ld + k, b);
        }
#pragma unroll
        for (int v = 0; v < V; v++) qe[v] = qn ? antidiff(f[v], qe[v], f[v] >= (TC)0 ? a[v] : b[v]) : f[v] * qe[v];
        stv<V>(FH + (size_t)t * mb.fs + (size_t)e * ld + k, qe);
    }
}

// The combined-weight edge flux (beta = 1) of one edge on V levels whose
// fluxes all run to the side whose stencil row (idx, w) is given.
template <bool PERS, typename TQ, typename TC, int V>
__device__ __forceinline__ void edge_combined(const MemberDev &mb, const TQ *q, const TQ *qn, int t0, int t1, int e,
                                              int k, const TC (&f)[V], const int (&idx)[GRIST_D2P],
                                              const TC (&w)[GRIST_D2P]) {
    const int ld = mb.ld;
    TC *FH = (TC *)mb.FH;
    for (int t = t0; t < t1; t++) {
        const TQ *qt = q + (size_t)t * mb.qs + k;
        TC s[V], a[V];
#pragma unroll
        for (int v = 0; v < V; v++) s[v] = 0;
#pragma unroll
        for (int j = 0; j < GRIST_D2P; j++) {
            ldv<PERS, V>(qt + (size_t)idx[j] * ld, a);
#pragma unroll
            for (int v = 0; v < V; v++) s[v] += w[j] * a[v];
        }
        if (qn) ldv<PERS, V>(qn + (size_t)t * mb.qs + (size_t)idx[0] * ld + k, a);
#pragma unroll
        for (int v = 0; v < V; v++) s[v] = qn ? antidiff(f[v], s[v], a[v]) : f[v] * s[v];
        stv<V>(FH + (size_t)t * mb.fs + (size_t)e * ld + k, s);
    }
}

// The edge item over a thread's levels (edge-centric form).  With the
// combined weights, the upwind side's stencil (4 vector loads) is read once
// and read again only for a level whose flux runs the other way; a vector
// whose levels disagree on the side takes them one by one.
template <bool PERS, typename TQ, typename TC, int LPT, int V>
__device__ __forceinline__ void item_edge_levels(const DevMesh &m, const MemberDev &mb, const TQ *q, const TQ *qn,
                                                 int t0, int t1, int e, int kg, bool beta1, TC beta) {
    if (!(beta1 && m.d2w_ok)) {
        if (V > 1 && !beta1) {
            item_edge<PERS, TQ, TC, V>(m, mb, q, qn, t0, t1, e, kg * V, beta1, beta);
            return;
        }
#pragma unroll 1
        for (int u = 0; u < LPT * V; u++) {
            const int k = V > 1 ? kg * V + u : kg + u * mb.Lg;
            if (LPT > 1 && k >= mb.L) break;
            item_edge<PERS, TQ, TC, 1>(m, mb, q, qn, t0, t1, e, k, beta1, beta);
        }
        return;
    }
    const size_t row = (size_t)e * mb.ld;
    int idx[GRIST_D2P];
    TC w[GRIST_D2P];
    if constexpr (V > 1) {
        TC f[V];
        flux_at<PERS, V>(mb, row + kg * V, f);
        const int side = f[0] >= (TC)0 ? 0 : 1;
        bool same = true;
#pragma unroll
        for (int v = 1; v < V; v++) same &= (f[v] >= (TC)0 ? 0 : 1) == side;
        if (same) {
            load_d2w(m, e, side, idx, w);
            edge_combined<PERS, TQ, TC, V>(mb, q, qn, t0, t1, e, kg * V, f, idx, w);
            return;
        }
    }
    int loaded = -1;
#pragma unroll(V > 1 ? 1 : LPT)
    for (int u = 0; u < LPT * V; u++) {
        const int k = V > 1 ? kg * V + u : kg + u * mb.Lg;
        if (LPT > 1 && k >= mb.L) break;
        TC f[1];
        flux_at<PERS, 1>(mb, row + k, f);
        const int side = f[0] >= (TC)0 ? 0 : 1;
        if (side != loaded) {
            load_d2w(m, e, side, idx, w);
            loaded = side;
        }
        edge_combined<PERS, TQ, TC, 1>(mb, q, qn, t0, t1, e, k, f, idx, w);
    }
}

// The low-order results of V levels at cell-level y of the tracer arrays: the
// local bounds {max, min}(q^n, q^td) and div F^L.
template <typename TC, int V>
__device__ __forceinline__ void store_lowres(const MemberDev &mb, size_t y, const TC (&r1)[V], const TC (&r2)[V],
                                             const TC (&qi)[V], const TC (&divl)[V]) {
    TC b[2 * V];
#pragma unroll
    for (int v = 0; v < V; v++) {
        const TC qd = lowres_value(r1[v], r2[v], qi[v], divl[v]);
        Bounds<TC> bd(qi[v], qi[v]);
        bd.take(qd, qd);
        b[2 * v] = bd.max();
        b[2 * v + 1] = bd.min();
    }
    stv<2 * V>((TC *)mb.X2 + 2 * y, b);
    stv<V>((TC *)mb.DFL + y, divl);
}

template <typename TC, int V, bool LOW> constexpr int ring_tracers() {
    return sizeof(TC) * V <= 8 || (LOW && sizeof(TC) == 4) ? 2 : 1;
}
// Cell-centric form of the edge flux (beta = 1, combined weights, every
// stencil the upwind cell's ring {i, neighbours} in the order of the cell's
// neighbour list): the thread of cell i gathers q over its ring and forms
// the flux of each edge whose flux leaves the cell, so each edge-level is
// written once, by its upwind cell, with the weights and the summation
// order of the edge-centric form (bit-identical), from 7 gathers per
// cell-level instead of 7 per edge-level.  The ring values of up to
// ring_tracers() tracers are gathered first, so each drained edge's weights
// are read once for them.  The drained edge-levels are kept as a mask (bit
// 8 v + j: level v, edge j), and each thread walks its own drained edges: a
// warp's cells drain different edges, so a walk over all six would spend 4.6
// passes on the three that each thread has.  An edge whose V levels all
// drain this cell is stored as one vector.  In the final stage of a limited
// step (qn = q^n) the phase stores A = F^H - F^L, F^L = F q^n_i.
//
// LOW (the first stage of a limited step, q = q^n): the ring and the fluxes
// are all that the low-order solution needs, so its phase (item_lowres, the
// same operations) is done here, without gathering them again.
template <bool PERS, typename TQ, typename TC, int LPT, int V, bool LOW>
__device__ __forceinline__ void item_edge_ring(const DevMesh &m, const MemberDev &mb, const TQ *q, const TQ *qn, int t0,
                                               int t1, int i, int kg, double dt, float dtf) {
    constexpr int RT = ring_tracers<TC, V, LOW>();
    const int ld = mb.ld;
    TC *FH = (TC *)mb.FH;
    int nb[GRIST_MAXE];
    load_row6(m.coc8, i, nb);
#pragma unroll
    for (int u = 0; u < LPT; u++) {
        const int k = (kg + u * mb.Lg) * V;
        if (LPT > 1 && k >= mb.L) break;
        unsigned out = 0, c1 = 0;
        {
            int e[GRIST_MAXE];
            TC cw[GRIST_MAXE];
            load_row6(m.eoc8, i, e);
            load_row6(Coef<TC>::cdiv8(m), i, cw);
#pragma unroll
            for (int j = 0; j < GRIST_MAXE; j++) {
                TC f[V];
                flux_at<PERS, V>(mb, (size_t)e[j] * ld + k, f);
                if (pos(cw[j])) c1 |= 1u << j;
                if (nonzero(cw[j])) {   // a real edge
#pragma unroll
                    for (int v = 0; v < V; v++)
                        if (nonneg(f[v]) == pos(cw[j])) out |= 1u << (8 * v + j);
                }
            }
        }
        unsigned any = out;
        if (V > 2) any |= any >> 16;
        if (V > 1) any |= any >> 8;
        any &= 0x3fu;
        const size_t x = (size_t)i * ld + k;
        TC r1[V], r2[V];
        if constexpr (LOW) {
            typename Vec2<TC>::T dv[V];
            dv_at<PERS, TC, V>(mb, x, dv);
#pragma unroll
            for (int v = 0; v < V; v++) stage_ratios(dv[v], dt, dtf, r1[v], r2[v]);
        }
        for (int tb = t0; tb < t1; tb += RT) {
            const int nt = min(RT, t1 - tb);
            TC qr[RT][GRIST_D2P][V], qup[RT][V];
#pragma unroll
            for (int a = 0; a < RT; a++) {
                if (a >= nt) break;
                const TQ *qt = q + (size_t)(tb + a) * mb.qs;
                ldv<PERS, V>(qt + (size_t)i * ld + k, qr[a][0]);
#pragma unroll
                for (int j = 0; j < GRIST_MAXE; j++) ldv<PERS, V>(qt + (size_t)nb[j] * ld + k, qr[a][1 + j]);
                if (qn) ldv_own<V>(qn + (size_t)(tb + a) * mb.qs + x, qup[a]);
            }
            if constexpr (LOW) {
                TC divl[RT][V];
#pragma unroll
                for (int a = 0; a < RT; a++)
#pragma unroll
                    for (int v = 0; v < V; v++) divl[a][v] = 0;
                int e[GRIST_MAXE];
                TC cw[GRIST_MAXE];
                load_row6(m.eoc8, i, e);
                load_row6(Coef<TC>::cdiv8(m), i, cw);
#pragma unroll
                for (int j = 0; j < GRIST_MAXE; j++) {
                    TC f[V];
                    flux_at<PERS, V>(mb, (size_t)e[j] * ld + k, f);
#pragma unroll
                    for (int v = 0; v < V; v++) {
                        const TC cf = mul_rn(cw[j], f[v]);
#pragma unroll
                        for (int a = 0; a < RT; a++)
                            divl[a][v] = fma_rn(cf, (out >> (8 * v + j)) & 1u ? qr[a][0][v] : qr[a][1 + j][v], divl[a][v]);
                    }
                }
#pragma unroll
                for (int a = 0; a < RT; a++) {
                    if (a >= nt) break;
                    store_lowres<TC, V>(mb, (size_t)(tb + a) * mb.qs + x, r1, r2, qr[a][0], divl[a]);
                }
            }
#pragma unroll 1
            for (unsigned left = any; left; left &= left - 1) {
                const int j = __ffs((int)left) - 1;
                const int e = ldg(m.eoc8 + (size_t)i * 8 + j);
                TC w[GRIST_D2P], f[V];
                load_d2w_weights(m, e, ((c1 >> j) & 1u) ? 0 : 1, w);
                flux_at<PERS, V>(mb, (size_t)e * ld + k, f);
                const unsigned oj = out >> j;
                bool all = true;
#pragma unroll
                for (int v = 0; v < V; v++) all &= ((oj >> (8 * v)) & 1u) != 0;
#pragma unroll
                for (int a = 0; a < RT; a++) {
                    if (a >= nt) break;
                    TC g[V];
#pragma unroll
                    for (int v = 0; v < V; v++) {
                        TC s = 0;
#pragma unroll
                        for (int p = 0; p < GRIST_D2P; p++) s += w[p] * qr[a][p][v];
                        g[v] = qn ? antidiff(f[v], s, qup[a][v]) : f[v] * s;
                    }
                    TC *dst = FH + (size_t)(tb + a) * mb.fs + (size_t)e * ld + k;
                    if (all) {
                        stv<V>(dst, g);
                    } else {
#pragma unroll
                        for (int v = 0; v < V; v++)
                            if ((oj >> (8 * v)) & 1u) dst[v] = g[v];
                    }
                }
            }
        }
    }
}

// RK stage update: q^(s) = (dpi^n q^n - dt_s div F^H) / dpi^(s),
// written as r1 q^n - r2 div with r1 = dpi^n/dpi^(s), r2 = dt_s/dpi^(s)
// taken once per (cell, level) in FP64 and rounded to the tracer type
// (Sec. 2.2 (ii): no mixed-kind products inside the tracer loop).
template <bool PERS, typename TQ, typename TC, int V>
__device__ __forceinline__ bool item_update(const CellRow<TC> &r, const MemberDev &mb, TQ *qout, int t0, int t1, int i,
                                            int k, double dts, float dtsf) {
    const int ld = mb.ld;
    const size_t x = (size_t)i * ld + k;
    typename Vec2<TC>::T dv[V];
    TC r1[V], r2[V];
    dv_at<PERS, TC, V>(mb, x, dv);
#pragma unroll
    for (int v = 0; v < V; v++) stage_ratios(dv[v], dts, dtsf, r1[v], r2[v]);
    const TQ *qn = (const TQ *)mb.q;
    const TC *FH = (const TC *)mb.FH;
    bool bad = false;
    for (int t = t0; t < t1; t++) {
        const TC *ft = FH + (size_t)t * mb.fs + k;
        TC div[V], qv[V];
        ldv_own<V>(qn + (size_t)t * mb.qs + x, qv);
#pragma unroll
        for (int v = 0; v < V; v++) div[v] = 0;
#pragma unroll
        for (int j = 0; j < GRIST_MAXE; j++) {
            TC a[V];
            ldv<PERS, V>(ft + (size_t)r.e[j] * ld, a);
#pragma unroll
            for (int v = 0; v < V; v++) div[v] += r.cw[j] * a[v];
        }
#pragma unroll
        for (int v = 0; v < V; v++) {
            qv[v] = r1[v] * qv[v] - r2[v] * div[v];
            bad |= !isfinite(qv[v]);
        }
        stv<V>(qout + (size_t)t * mb.qs + x, qv);
    }
    return bad;
}

// FCT 1: low-order solution q^td = (dpi^n q^n - dt div F^L) / dpi^(3),
// with F^L the first-order upwind flux of q^n (the upwind cell is c1 when
// F >= 0, c2 otherwise; cell i is c1 of its edge exactly when its
// divergence coefficient is positive), stored as the cell's local bounds
// {max, min}(q^n, q^td) (X2: q^td is the member of the pair that is not
// q^n, or q^n itself), and div F^L (DFL) for the later phases.
template <bool PERS, typename TQ, typename TC, int V>
__device__ __forceinline__ void item_lowres(const CellRow<TC> &r, const MemberDev &mb, int t0, int t1, int i, int k,
                                            double dt, float dtf) {
    const int ld = mb.ld;
    const size_t x = (size_t)i * ld + k;
    typename Vec2<TC>::T dv[V];
    TC r1[V], r2[V];
    dv_at<PERS, TC, V>(mb, x, dv);
#pragma unroll
    for (int v = 0; v < V; v++) stage_ratios(dv[v], dt, dtf, r1[v], r2[v]);
    // s dv/A F of the cell's edges; a level drains this cell through edge j
    // where bit j V + v is set
    TC cf[GRIST_MAXE][V];
    unsigned out = 0;
#pragma unroll
    for (int j = 0; j < GRIST_MAXE; j++) {
        flux_at<PERS, V>(mb, (size_t)r.e[j] * ld + k, cf[j]);
#pragma unroll
        for (int v = 0; v < V; v++) {
            if (nonneg(cf[j][v]) == pos(r.cw[j])) out |= 1u << (j * V + v);
            cf[j][v] = mul_rn(r.cw[j], cf[j][v]);
        }
    }
    const TQ *qn = (const TQ *)mb.q;
    for (int t = t0; t < t1; t++) {
        const TQ *qt = qn + (size_t)t * mb.qs + k;
        TC divl[V], qi[V];
        ldv<PERS, V>(qt + (size_t)i * ld, qi);
#pragma unroll
        for (int v = 0; v < V; v++) divl[v] = 0;
#pragma unroll
        for (int j = 0; j < GRIST_MAXE; j++) {
            TC a[V];
            ldv<PERS, V>(qt + (size_t)r.nb[j] * ld, a);
#pragma unroll
            for (int v = 0; v < V; v++) divl[v] = fma_rn(cf[j][v], (out >> (j * V + v)) & 1u ? qi[v] : a[v], divl[v]);
        }
        store_lowres<TC, V>(mb, (size_t)t * mb.qs + x, r1, r2, qi, divl);
    }
}

// FCT 2: bounds over the cell and its neighbours of {q^n, q^td} (from the
// cells' local bounds); antidiffusive in/out sums P+- of A = F^H - F^L (as
// the final edge phase stored it); allowed changes Q+-; ratios
// R+- = min(1, Q / (P + TINY)) (Sec. 2.2 (iii): TINY of the working type),
// stored as the pair {R+, R-}.
template <bool PERS, typename TQ, typename TC, int V>
__device__ __forceinline__ void item_ratios(const CellRow<TC> &r, const MemberDev &mb, int t0, int t1, int i, int k,
                                            double dt, float dtf) {
    const int ld = mb.ld;
    const size_t x = (size_t)i * ld + k;
    typename Vec2<TC>::T dv[V];
    TC dp3[V];
    dv_at<PERS, TC, V>(mb, x, dv);
#pragma unroll
    for (int v = 0; v < V; v++) dp3[v] = static_cast<TC>(end_mass(dv[v], dt, dtf));
    const TC dtc = sizeof(TC) == 4 ? (TC)dtf : (TC)dt;
    const TC *X2 = (const TC *)mb.X2;
    const TQ *qn = (const TQ *)mb.q;
    const TC *A = (const TC *)mb.FH;
    TC *R2 = (TC *)mb.R2;
    for (int t = t0; t < t1; t++) {
        const TC *xt = X2 + 2 * ((size_t)t * mb.qs + k);
        const TC *at = A + (size_t)t * mb.fs + k;
        TC bi[2 * V], pp[V], pm[V], qi[V];
        ldv<PERS, 2 * V>(xt + 2 * (size_t)i * ld, bi);
        ldv<PERS, V>(qn + (size_t)t * mb.qs + x, qi);
        Bounds<TC> bd[V];
#pragma unroll
        for (int v = 0; v < V; v++) {
            bd[v] = Bounds<TC>(bi[2 * v], bi[2 * v + 1]);
            pp[v] = pm[v] = 0;
        }
#pragma unroll
        for (int j = 0; j < GRIST_MAXE; j++) {
            TC bn[2 * V], a[V];
            ldv<PERS, 2 * V>(xt + 2 * (size_t)r.nb[j] * ld, bn);
            ldv<PERS, V>(at + (size_t)r.e[j] * ld, a);
#pragma unroll
            for (int v = 0; v < V; v++) {
                bd[v].take(bn[2 * v], bn[2 * v + 1]);
                add_signed(r.cw[j] * a[v], pp[v], pm[v]);  // outward A / A_i
            }
        }
        TC rr[2 * V];
#pragma unroll
        for (int v = 0; v < V; v++) {
            const TC qtd = same_num(bi[2 * v], qi[v]) ? bi[2 * v + 1] : bi[2 * v];
            const TC Qp = (bd[v].max() - qtd) * dp3[v], Qm = (qtd - bd[v].min()) * dp3[v];
            rr[2 * v] = fct_ratio(Qp, pp[v] * dtc + tiny_of<TC>());
            rr[2 * v + 1] = fct_ratio(Qm, pm[v] * dtc + tiny_of<TC>());
        }
        stv<2 * V>(R2 + 2 * ((size_t)t * mb.qs + x), rr);
    }
}

// FCT 3: limited flux F^L + C A with C = min(R-(c1), R+(c2)) when A runs
// c1 -> c2 (A >= 0), min(R+(c1), R-(c2)) else; q^{n+1} = (dpi^n q^n - dt
// div(F^L + C A)) / dpi^(3), with div F^L from the low-order phase, written
// over q^n in place (each thread reads only its own cell's q^n).
template <bool PERS, typename TQ, typename TC, int V>
__device__ __forceinline__ bool item_final(const CellRow<TC> &r, const MemberDev &mb, int t0, int t1, int i, int k,
                                           double dt, float dtf) {
    const int ld = mb.ld;
    const size_t x = (size_t)i * ld + k;
    typename Vec2<TC>::T dv[V];
    TC r1[V], r2[V];
    dv_at<PERS, TC, V>(mb, x, dv);
#pragma unroll
    for (int v = 0; v < V; v++) stage_ratios(dv[v], dt, dtf, r1[v], r2[v]);
    TQ *q = (TQ *)mb.q;
    const TC *A = (const TC *)mb.FH, *DFL = (const TC *)mb.DFL;
    const TC *R2 = (const TC *)mb.R2;
    bool bad = false;
    for (int t = t0; t < t1; t++) {
        const TC *at = A + (size_t)t * mb.fs + k;
        const TC *rt = R2 + 2 * ((size_t)t * mb.qs + k);
        TC ri[2 * V], div[V], qv[V];
        ldv<PERS, 2 * V>(rt + 2 * (size_t)i * ld, ri);
        ldv<PERS, V>(DFL + (size_t)t * mb.qs + x, div);
        ldv_own<V>(q + (size_t)t * mb.qs + x, qv);
#pragma unroll
        for (int j = 0; j < GRIST_MAXE; j++) {
            TC ae[V], rn[2 * V];
            ldv<PERS, V>(at + (size_t)r.e[j] * ld, ae);
            ldv<PERS, 2 * V>(rt + 2 * (size_t)r.nb[j] * ld, rn);
            const bool i_is_c1 = pos(r.cw[j]);
#pragma unroll
            for (int v = 0; v < V; v++) {
                // A leaves cell i: its R- and the neighbour's R+; A enters it: the other two
                const bool leaves = nonneg(ae[v]) == i_is_c1;
                const TC c = leaves ? min_num(ri[2 * v + 1], rn[2 * v]) : min_num(ri[2 * v], rn[2 * v + 1]);
                div[v] += r.cw[j] * (c * ae[v]);
            }
        }
#pragma unroll
        for (int v = 0; v < V; v++) {
            qv[v] = r1[v] * qv[v] - r2[v] * div[v];
            bad |= !isfinite(qv[v]);
        }
        stv<V>(q + (size_t)t * mb.qs + x, qv);
    }
    return bad;
}

// ---------------------------------------------------------------------------
// phases: grid-stride loops over a work space

enum Phase { P_DIV = 0, P_EDGE0, P_UPD0, P_EDGE1, P_UPD1, P_EDGE2, P_UPD2, P_LOWRES, P_RATIOS, P_FINAL, P_NPHASE };

// One pass over a work space.  A work item is (entity, level group g) of a
// member and tracer group.  V > 1: the thread takes the V consecutive levels
// g V, ..., g V + V - 1 as one vector.  V = 1: it takes the LPT levels g,
// g + Lg, ... (Lg = ceil(L / LPT)).  Either way consecutive threads touch
// consecutive memory, and the entity's tables are read once for its levels.
// RING: the form of an edge phase, -1 = as B.ring says (the persistent
// launch), 0 / 1 = compiled for one form (the per-phase kernels, so that a
// kernel's registers serve the form it runs), 2 = the cell-centric form with
// the low-order solution.
template <bool PERS, typename TQ, typename TC, int PH, int LPT = 1, int V = 1, int RING = -1>
__device__ void run_phase(const DevMesh &m, const Batch &B, const Space &S, uint32_t *status) {
    static_assert(V == 1 || LPT == 1, "a vector item has one level group");
    const bool ring = RING < 0 ? (B.ring != 0) : (RING >= 1);
    const unsigned long long stride = (unsigned long long)gridDim.x * blockDim.x;
    int seg = -1;
    bool bad = false;
    const double dts = PH <= P_UPD0 ? B.dt3 : (PH <= P_UPD1 ? 0.5 * B.dt : B.dt);
    const float dtsf = cv<float>(dts), dtf = cv<float>(B.dt);
    const TC beta = static_cast<TC>(B.beta);
    for (unsigned long long n = (unsigned long long)blockIdx.x * blockDim.x + threadIdx.x; n < S.total; n += stride) {
        seg = find_seg(S, n, seg);
        const int2 mg = S.mg[seg];
        const MemberDev &mb = B.mem[mg.x];
        int ent, kg;
        split_index((uint32_t)(n - S.start[seg]), mb.DL, ent, kg);
        const int t0 = mg.y * B.tpt;
        const int t1 = min(mb.T, t0 + B.tpt);
        if constexpr (PH == P_EDGE0 || PH == P_EDGE1 || PH == P_EDGE2) {
            const TQ *qs = (const TQ *)(PH == P_EDGE0 ? mb.q : (PH == P_EDGE1 ? mb.qA : mb.qB));
            // the final stage of a limited step stores A = F^H - F^L
            const TQ *qn = (PH == P_EDGE2 && B.fct) ? (const TQ *)mb.q : nullptr;
            if (ring) {
                item_edge_ring<PERS, TQ, TC, LPT, V, RING == 2>(m, mb, qs, qn, t0, t1, ent, kg, B.dt, dtf);
            } else {
                item_edge_levels<PERS, TQ, TC, LPT, V>(m, mb, qs, qn, t0, t1, ent, kg, B.beta1, beta);
            }
            continue;
        }
        // the cell's row, once for its levels (FP64 weights for the
        // continuity phase); the limited-flux phase, the one with the most
        // live values per level, reads it again for each strided level
        using TW = typename std::conditional<PH == P_DIV, double, TC>::type;
        constexpr bool kNb = PH == P_LOWRES || PH == P_RATIOS || PH == P_FINAL;
        constexpr bool kRowPerLevel = PH == P_FINAL && LPT > 1;
        CellRow<TW> r;
        if (!kRowPerLevel) load_cell_row<kNb>(m, ent, r);
#pragma unroll
        for (int u = 0; u < LPT; u++) {
        const int k = (kg + u * mb.Lg) * V;
        if (LPT > 1 && k >= mb.L) break;
        if (kRowPerLevel) load_cell_row<kNb>(m, ent, r);
        if constexpr (PH == P_DIV) item_div<TC, V>(mb, r, ent, k);
        if constexpr (PH == P_UPD0) bad |= item_update<PERS, TQ, TC, V>(r, mb, (TQ *)mb.qA, t0, t1, ent, k, dts, dtsf);
        if constexpr (PH == P_UPD1) bad |= item_update<PERS, TQ, TC, V>(r, mb, (TQ *)mb.qB, t0, t1, ent, k, dts, dtsf);
        if constexpr (PH == P_UPD2) bad |= item_update<PERS, TQ, TC, V>(r, mb, (TQ *)mb.q, t0, t1, ent, k, dts, dtsf);
        if constexpr (PH == P_LOWRES) item_lowres<PERS, TQ, TC, V>(r, mb, t0, t1, ent, k, B.dt, dtf);
        if constexpr (PH == P_RATIOS) item_ratios<PERS, TQ, TC, V>(r, mb, t0, t1, ent, k, B.dt, dtf);
        if constexpr (PH == P_FINAL) bad |= item_final<PERS, TQ, TC, V>(r, mb, t0, t1, ent, k, B.dt, dtf);
        }
    }
    if (bad) atomicOr(status, GRIST_FLAG_NONFINITE);
}

// Register cap of a work-list phase kernel in the binary32 policy.  These
// kernels are bound by the latency of their neighbour gathers: a cap trades
// the loads each thread keeps in flight against resident warps, and the best
// point differs per phase (measured on the level-9 mesh, 60 levels, 4
// tracers).  Compile-time, per phase; 0 = only the limit that lets a block
// of kTracerMaxBlock threads launch (65536 registers per SM), which is also
// the FP64 policy's cap.
#ifndef GRIST_TR_REGS_EDGE   // edge fluxes, edge-centric form
#define GRIST_TR_REGS_EDGE 56
#endif
#ifndef GRIST_TR_REGS_RING   // edge fluxes, cell-centric form
#define GRIST_TR_REGS_RING 72
#endif
#ifndef GRIST_TR_REGS_UPD
#define GRIST_TR_REGS_UPD 64
#endif
#ifndef GRIST_TR_REGS_LOWRES
#define GRIST_TR_REGS_LOWRES 64
#endif
#ifndef GRIST_TR_REGS_RATIOS
#define GRIST_TR_REGS_RATIOS 72
#endif
#ifndef GRIST_TR_REGS_FINAL
#define GRIST_TR_REGS_FINAL 0
#endif
constexpr int kTracerRegLimit = 65536 / kTracerMaxBlock;
constexpr int cap_or_none(int r) { return r > 0 && r < kTracerRegLimit ? r : kTracerRegLimit; }
template <typename TC, int PH, int V, int RING> constexpr int tracer_phase_regs() {
    constexpr bool edge = PH == P_EDGE0 || PH == P_EDGE1 || PH == P_EDGE2;
    constexpr bool upd = PH == P_UPD0 || PH == P_UPD1 || PH == P_UPD2;
    if (sizeof(TC) != 4) return kTracerRegLimit;
    // vector items: bytes in flight come from the width of their loads, so more
    // registers and fewer warps do better than for single levels
    if (V > 1)
        return cap_or_none(edge             ? (RING == 2 ? (V == 4 ? 0 : 80) : (RING == 1 ? 72 : 0))
                           : PH == P_LOWRES ? 72
                                            : 0);
    return cap_or_none(edge             ? (RING >= 1 ? GRIST_TR_REGS_RING : GRIST_TR_REGS_EDGE)
                       : upd            ? GRIST_TR_REGS_UPD
                       : PH == P_LOWRES ? GRIST_TR_REGS_LOWRES
                       : PH == P_RATIOS ? GRIST_TR_REGS_RATIOS
                       : PH == P_FINAL  ? GRIST_TR_REGS_FINAL
                                        : 0);
}

// The space a phase runs over: cells without groups, edges (edge-centric
// fluxes) or cells with tracer groups.
constexpr bool is_edge_phase(int ph) { return ph == P_EDGE0 || ph == P_EDGE1 || ph == P_EDGE2; }
__host__ __device__ __forceinline__ const Space &phase_space(const Batch &B, int ph, bool ring, int cls) {
    return ph == P_DIV ? B.D[cls] : (is_edge_phase(ph) && !ring) ? B.E[cls] : B.C[cls];
}

template <typename TQ, typename TC, int PH, int LPT, int V, int RING>
__global__ void __maxnreg__((tracer_phase_regs<TC, PH, V, RING>())) k_tracer_phase(DevMesh m, Batch B, uint32_t *status) {
    constexpr int cls = V == 4 ? 2 : (V == 2 ? 1 : 0);
    run_phase<false, TQ, TC, PH, LPT, V, RING>(m, B, phase_space(B, PH, RING >= 1, cls), status);
}

// Fused RK stage (no limiter) on one tile x 32 levels x the tracers of one
// group: the stage input on the tile's halo goes to shared memory, every
// tile edge's third-order flux is computed once into shared memory, and the
// cell update gathers from there (boundary edges of a tile are computed by
// both tiles that share them).  Same arithmetic as item_edge + item_update.
template <typename TQ, typename TC, bool BETA1>
__global__ void __launch_bounds__(256) k_tr_tile_stage(DevMesh m, TileMesh tm, Batch B, int stage,
                                                       uint32_t *status) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    TC *qs = (TC *)smem_raw;              // [Hmax][32]
    TC *fs = qs + (size_t)tm.Hmax * 32;   // [Emax][32]
    __shared__ int s_seg;
    if (threadIdx.x == 0) s_seg = find_seg(B.T, blockIdx.x, -1);
    __syncthreads();
    const int seg = s_seg;
    const int2 mg = B.T.mg[seg];
    const MemberDev &mb = B.mem[mg.x];
    const unsigned r = blockIdx.x - (unsigned)B.T.start[seg];
    const int nch = (mb.L + 31) >> 5;
    const int tile = (int)(r / nch), chunk = (int)(r % nch);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
    const int k = chunk * 32 + lane;
    const bool kin = k < mb.L;
    const int ld = mb.ld;
    const int h0 = tm.hoff[tile], H = tm.hoff[tile + 1] - h0;
    const int e0 = tm.eoff[tile], E = tm.eoff[tile + 1] - e0;
    const int c0 = tile * kTileCells;
    const int nc = min(kTileCells, m.nC - c0);
    const TQ *qin = stage == 0 ? (const TQ *)mb.q : (stage == 1 ? (const TQ *)mb.qA : (const TQ *)mb.qB);
    TQ *qout = stage == 0 ? (TQ *)mb.qA : (stage == 1 ? (TQ *)mb.qB : (TQ *)mb.q);
    const TQ *qn = (const TQ *)mb.q;
    const double dts = stage == 0 ? B.dt3 : (stage == 1 ? 0.5 * B.dt : B.dt);
    const TC beta = static_cast<TC>(B.beta);
    // stage ratios of this warp's cells (same for every tracer)
    constexpr int kCpw = kTileCells / 4;   // cells per warp for blocks of >= 4 warps
    TC r1v[kCpw], r2v[kCpw];
#pragma unroll
    for (int idx = 0; idx < kCpw; idx++) {
        const int ci = warp + idx * nw;
        r1v[idx] = r2v[idx] = (TC)0;
        if (ci < nc && kin) {
            const size_t x = (size_t)(c0 + ci) * ld + k;
            stage_ratios(((const typename Vec2<TC>::T *)mb.DV)[x], dts, cv<float>(dts), r1v[idx], r2v[idx]);
        }
    }
    const int t0 = mg.y * B.tpt, t1 = min(mb.T, t0 + B.tpt);
    bool bad = false;
    for (int t = t0; t < t1; t++) {
        const TQ *qt = qin + (size_t)t * mb.qs;
        for (int hh = warp; hh < H; hh += nw)
            qs[hh * 32 + lane] = kin ? static_cast<TC>(ldg(qt + (size_t)ldg(tm.halo + h0 + hh) * ld + k)) : (TC)0;
        __syncthreads();
        for (int j = warp; j < E; j += nw) {
            if (kin) {
                const int e = ldg(tm.tedge + e0 + j);
                const uint16_t *loc = tm.eloc + (size_t)(e0 + j) * 16;
                const TC f = static_cast<TC>(ldg(mb.F + (size_t)e * ld + k));
                const TC dc2 = ldg(Coef<TC>::dc2(m) + e);
                const TC *cf = Coef<TC>::d2c(m) + (size_t)e * 14;
                const TC q1 = qs[loc[0] * 32 + lane], q2 = qs[loc[1] * 32 + lane];
                TC qe;
                if (BETA1) {
                    const int side = f >= (TC)0 ? 0 : 1;
                    TC d = 0;
#pragma unroll
                    for (int i = 0; i < GRIST_D2P; i++)
                        d += ldg(cf + side * GRIST_D2P + i) * qs[loc[2 + side * GRIST_D2P + i] * 32 + lane];
                    qe = (TC)0.5 * (q1 + q2) - (TC)2 * dc2 * d;
                } else {
                    const TC sgn = f >= (TC)0 ? (TC)1 : (TC)-1;
                    TC d1 = 0, d2 = 0;
#pragma unroll
                    for (int i = 0; i < GRIST_D2P; i++) {
                        d1 += ldg(cf + i) * qs[loc[2 + i] * 32 + lane];
                        d2 += ldg(cf + GRIST_D2P + i) * qs[loc[2 + GRIST_D2P + i] * 32 + lane];
                    }
                    qe = (TC)0.5 * (q1 + q2) - dc2 * (d1 + d2) + sgn * beta * dc2 * (d2 - d1);
                }
                fs[j * 32 + lane] = f * qe;
            }
        }
        __syncthreads();
#pragma unroll
        for (int idx = 0; idx < kCpw; idx++) {
            const int ci = warp + idx * nw;
            if (ci < nc && kin) {
                const int cell = c0 + ci;
                const uint16_t *le = tm.cle + (size_t)cell * 6;
                TC div = 0;
#pragma unroll
                for (int j = 0; j < GRIST_MAXE; j++) div += ldg(Coef<TC>::cdiv(m) + cell * 6 + j) * fs[le[j] * 32 + lane];
                const size_t x = (size_t)cell * ld + k;
                const TC v = r1v[idx] * static_cast<TC>(qn[(size_t)t * mb.qs + x]) - r2v[idx] * div;
                bad |= !isfinite(v);
                qout[(size_t)t * mb.qs + x] = static_cast<TQ>(v);
            }
        }
        __syncthreads();
    }
    if (bad) atomicOr(status, GRIST_FLAG_NONFINITE);
}

// ---------------------------------------------------------------------------
// Vertical transport, the delta(M q) term of Eq. 10, by an adaptively
// implicit upwind scheme (Sec. 2.1; the reading): at interior interface j
// (between layers j-1 above and j below, M_j > 0 carrying mass downward)
// the donor layer is j-1 if M_j > 0, else j, with Courant number
// c_j = |M_j| dt / dpi*_donor; the share Me_j = min(1, cmax / c_j) M_j moves
// explicitly (first-order upwind from q at the start), the rest
// Mi_j = M_j - Me_j by backward-Euler upwind, so per column
//   dpi+_k q+_k + dt (Fi_{k+1} - Fi_k) = dpi*_k q_k - dt (Fe_{k+1} - Fe_k),
//   dpi*_k = dpi_k - dt div(F)_k (the horizontal step's end),
//   dpi+_k = dpi*_k - dt (M_{k+1} - M_k),
// a tridiagonal M-matrix system solved by the Thomas algorithm.  Arithmetic
// in the tracer compute type.
__device__ __forceinline__ double vinv(double x) { return rcp(x); }   // correctly rounded, as 1.0 / x
__device__ __forceinline__ float vinv(float x) { return 1.0f / x; }

// One warp per column; lane l holds the K consecutive levels from l K (K =
// ceil(L / 32)) and the interfaces above them, so the neighbours it needs
// come from the next lanes by shuffles, a tracer's column is read once, and
// each interface's flux is formed once.  Whether the interface moves explicitly
// is decided by |M| dt <= cmax dpi*_donor (no division); only an interface
// beyond that takes the Courant number and its share.  When no interface of
// the column has an implicit share (the usual case) the tridiagonal system is
// diagonal: the Thomas sweep then reduces to q+_k = rhs_k * (1 / b_k), which
// every lane evaluates for its own levels.  Otherwise the rows go through
// shared memory and one lane runs the sweep.  Up to kVertT tracers' columns
// are loaded before the first is used.  Level 7, 4 tracers, 60 levels, us a
// launch against a split by both neighbours with a division each and lanes
// over every 32nd level: binary64 1946 -> 585 (FP64 pipe, 26.7 -> 8
// instructions a tracer-level), binary32 246 -> 125 (memory latency).
constexpr int kVertWarps = 8;
constexpr int kVertT = 4;

template <typename TQ, typename TC, int K, bool VEC>
__global__ void __launch_bounds__(kVertWarps * 32) k_tr_vertical(DevMesh m, MemberDev mb, double dt, double cmax,
                                                                uint32_t *status) {
    __shared__ TC sA[kVertWarps][K * 32], sB[kVertWarps][K * 32], sC[kVertWarps][K * 32], sD[kVertWarps][K * 32],
        sE[kVertWarps][K * 32];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int i = blockIdx.x * kVertWarps + warp;
    if (i >= m.nC) return;   // whole warps only: no block barrier below
    const int L = mb.L, k0 = lane * K;
    const TC dtc = cv<TC>(dt), cm = cv<TC>(cmax);
    const size_t row = (size_t)i * mb.ld + k0, irow = (size_t)i * mb.ldi + k0;
    constexpr unsigned kAllLanes = 0xffffffffu;
    // a lane's levels as one vector (VEC: whole vectors, aligned), else one by one
    auto load = [&](const auto *p, auto (&o)[K]) {
#pragma unroll
        for (int r = 0; r < K; r++) o[r] = 0;
        if constexpr (VEC) {
            if (k0 < L) ldv_own<K>(p, o);
        } else {
#pragma unroll
            for (int r = 0; r < K; r++)
                if (k0 + r < L) o[r] = p[r];
        }
    };
    // start layer mass of the vertical step (the end of the horizontal one),
    // that of the layer above the lane's first, interface fluxes
    TC dps[K], Mt[K];
    const float dtf = cv<float>(dt);
    {
        const typename Vec2<TC>::T *DV = (const typename Vec2<TC>::T *)mb.DV + row;
#pragma unroll
        for (int r = 0; r < K; r++) {
            const int k = k0 + r;
            dps[r] = (TC)1;
            Mt[r] = (TC)0;
            if (k < L) {
                dps[r] = (TC)end_mass(DV[r], dt, dtf);
                if (k > 0) Mt[r] = cv<TC>(mb.Mv[irow + r]);
            }
        }
    }
    const TC above0 = __shfl_up_sync(kAllLanes, dps[K - 1], 1);
    // dt times the explicit and implicit shares of the flux at the lane's
    // interfaces; bit r of up: its donor is the layer above
    TC me[K], mi[K];
    unsigned up = 0;
    bool implicit = false;
#pragma unroll
    for (int r = 0; r < K; r++) {
        me[r] = dtc * Mt[r];
        mi[r] = (TC)0;
        if (pos(Mt[r])) up |= 1u << r;
        const TC donor = (up >> r) & 1u ? (r ? dps[r - 1] : above0) : dps[r];
        if (nonzero(Mt[r]) && !le_num(abs_num(me[r]), cm * donor)) {
            const TC cour = fabs(Mt[r]) * dtc / donor;
            const TC f = cour <= cm ? (TC)1 : cm / cour;
            const TC e = f * Mt[r];
            mi[r] = dtc * (Mt[r] - e);
            me[r] = dtc * e;
            implicit |= mi[r] != (TC)0;
        }
    }
    implicit = __any_sync(kAllLanes, implicit);
    // shares at the interface below the lane's last layer (none at the ground)
    TC meb = __shfl_down_sync(kAllLanes, me[0], 1), mib = (TC)0;
    unsigned upb = __shfl_down_sync(kAllLanes, up, 1);
    if (implicit) mib = __shfl_down_sync(kAllLanes, mi[0], 1);
    if (lane == 31) {
        meb = mib = (TC)0;
        upb = 1;   // no flux times its own last level: there is no next lane
    }
    TC rb[K];
#pragma unroll
    for (int r = 0; r < K; r++) {
        const TC et = me[r], eb = r + 1 < K ? me[(r + 1) % K] : meb;
        TC b = dps[r] - (eb - et);
        if (implicit) {
            const TC it = mi[r], ib = r + 1 < K ? mi[(r + 1) % K] : mib;
            b = dps[r] - ((eb + ib) - (et + it)) + (fmax_((TC)0, ib) - fmin_((TC)0, it));
            const int k = k0 + r;
            sA[warp][k] = -fmax_((TC)0, it);
            sB[warp][k] = b;
            sC[warp][k] = fmin_((TC)0, ib);
        }
        rb[r] = vinv(b);
    }
    bool bad = false;
    for (int tb = 0; tb < mb.T; tb += kVertT) {
        TC q[kVertT][K];
#pragma unroll
        for (int a = 0; a < kVertT; a++)
            if (tb + a < mb.T) load((const TQ *)mb.q + (size_t)(tb + a) * mb.qs + row, q[a]);
#pragma unroll
        for (int a = 0; a < kVertT; a++) {
            if (tb + a >= mb.T) break;
            TQ *qt = (TQ *)mb.q + (size_t)(tb + a) * mb.qs + row;
            const TC qm = __shfl_up_sync(kAllLanes, q[a][K - 1], 1), qp = __shfl_down_sync(kAllLanes, q[a][0], 1);
            TC x[K], fl = me[0] * ((up & 1u) ? qm : q[a][0]);
            // the lane's last interface: the flux of the next lane's first
            const TC flb = meb * ((upb & 1u) ? q[a][K - 1] : qp);
#pragma unroll
            for (int r = 0; r < K; r++) {
                const TC fb = r + 1 < K ? me[(r + 1) % K] * ((up >> (r + 1)) & 1u ? q[a][r] : q[a][(r + 1) % K]) : flb;
                x[r] = dps[r] * q[a][r] - (fb - fl);
                fl = fb;
            }
            if (!implicit) {
#pragma unroll
                for (int r = 0; r < K; r++) x[r] *= rb[r];
            } else {
#pragma unroll
                for (int r = 0; r < K; r++) sD[warp][k0 + r] = x[r];
                __syncwarp();
                if (lane == 0) {
                    // Thomas sweep: forward elimination into sE and sD, back
                    // substitution into sD
                    TC cpk = (TC)0, dk = (TC)0;
                    for (int k = 0; k < L; k++) {
                        const TC ak = sA[warp][k];
                        const TC rden = vinv(k == 0 ? sB[warp][k] : sB[warp][k] - ak * cpk);
                        cpk = sC[warp][k] * rden;
                        dk = (k == 0 ? sD[warp][k] : sD[warp][k] - ak * dk) * rden;
                        sE[warp][k] = cpk;
                        sD[warp][k] = dk;
                    }
                    TC qb = (TC)0;
                    for (int k = L - 1; k >= 0; k--) {
                        qb = (k == L - 1) ? sD[warp][k] : sD[warp][k] - sE[warp][k] * qb;
                        sD[warp][k] = qb;
                    }
                }
                __syncwarp();
#pragma unroll
                for (int r = 0; r < K; r++) x[r] = sD[warp][k0 + r];
                __syncwarp();   // the next tracer reuses the rows
            }
#pragma unroll
            for (int r = 0; r < K; r++) bad |= k0 + r < L && !isfinite(x[r]);
            if constexpr (VEC) {
                if (k0 < L) stv<K>(qt, x);
            } else {
#pragma unroll
                for (int r = 0; r < K; r++)
                    if (k0 + r < L) qt[r] = (TQ)x[r];
            }
        }
    }
    if (bad) atomicOr(status, GRIST_FLAG_NONFINITE);
}

// Bounded wait until *gen differs from g: at most `limit` polls (~64 ns
// apart); on giving up (or when another block already gave up) raises
// GRIST_FLAG_TIMEOUT and returns false.
__device__ bool bounded_wait_change(volatile unsigned *gen, unsigned g, long long limit, unsigned *abort_word,
                                    uint32_t *status) {
    long long it = 0;
    while (*gen == g) {
        if (++it > limit || *(volatile unsigned *)abort_word) {
            atomicExch(abort_word, 1u);
            atomicOr(status, GRIST_FLAG_TIMEOUT);
            return false;
        }
        __nanosleep(64);
    }
    return true;
}

// Grid barrier for a cooperative launch (all blocks co-resident).  bar[0]
// counts arrivals, bar[1] is the generation, bar[2] the launch's abort word
// (both bar[0] and bar[2] are zeroed before every launch).  Thread 0 of each
// block arrives on the counter; the last arrival resets it and bumps the
// generation.  The wait is bounded (bounded_wait_change), so the kernel
// always ends; after a timeout every block returns false.
__device__ bool grid_sync(unsigned *bar, uint32_t *status) {
    __shared__ int ok;
    __syncthreads();
    if (threadIdx.x == 0) {
        ok = 1;
        volatile unsigned *gen = bar + 1;
        const unsigned g = *gen;
        __threadfence();
        const unsigned arrived = atomicAdd(bar, 1u);
        if (arrived == gridDim.x - 1) {
            atomicExch(bar, 0u);
            __threadfence();
            atomicAdd(bar + 1, 1u);
        } else if (!bounded_wait_change(gen, g, kBarrierSpinLimit, bar + 2, status)) {
            ok = 0;
        }
        __threadfence();
    }
    __syncthreads();
    return ok != 0;
}

// Self-test of the bounded wait: one thread waits on a word nothing writes.
__global__ void k_wait_selftest(unsigned *word, unsigned *abort_word, long long limit, uint32_t *status) {
    if (threadIdx.x == 0 && blockIdx.x == 0)
        bounded_wait_change(word, *(volatile unsigned *)word, limit, abort_word, status);
}

// One cooperative launch for the whole step: the phases in order with a
// grid barrier between consecutive ones.
template <typename TQ, typename TC>
__global__ void k_tracer_persistent(DevMesh m, Batch B, unsigned *bar, uint32_t *status) {
    run_phase<true, TQ, TC, P_DIV>(m, B, phase_space(B, P_DIV, B.ring != 0, 0), status);
    if (!grid_sync(bar, status)) return;
    run_phase<true, TQ, TC, P_EDGE0>(m, B, phase_space(B, P_EDGE0, B.ring != 0, 0), status);
    if (!grid_sync(bar, status)) return;
    run_phase<true, TQ, TC, P_UPD0>(m, B, phase_space(B, P_UPD0, B.ring != 0, 0), status);
    if (!grid_sync(bar, status)) return;
    run_phase<true, TQ, TC, P_EDGE1>(m, B, phase_space(B, P_EDGE1, B.ring != 0, 0), status);
    if (!grid_sync(bar, status)) return;
    run_phase<true, TQ, TC, P_UPD1>(m, B, phase_space(B, P_UPD1, B.ring != 0, 0), status);
    if (!grid_sync(bar, status)) return;
    run_phase<true, TQ, TC, P_EDGE2>(m, B, phase_space(B, P_EDGE2, B.ring != 0, 0), status);
    if (!grid_sync(bar, status)) return;
    if (!B.fct) {
        run_phase<true, TQ, TC, P_UPD2>(m, B, phase_space(B, P_UPD2, B.ring != 0, 0), status);
        return;
    }
    run_phase<true, TQ, TC, P_LOWRES>(m, B, phase_space(B, P_LOWRES, B.ring != 0, 0), status);
    if (!grid_sync(bar, status)) return;
    run_phase<true, TQ, TC, P_RATIOS>(m, B, phase_space(B, P_RATIOS, B.ring != 0, 0), status);
    if (!grid_sync(bar, status)) return;
    run_phase<true, TQ, TC, P_FINAL>(m, B, phase_space(B, P_FINAL, B.ring != 0, 0), status);
}

// ---------------------------------------------------------------------------
// host side

size_t al256(size_t b) { return (b + 255) & ~size_t(255); }

struct HostPlan {
    std::vector<MemberDev> mem;
    struct Seg {
        std::vector<unsigned long long> start;   // closed by the total
        std::vector<int2> mg;
        size_t o_start = 0, o_mg = 0;            // offsets in the device table
    };
    Seg D[kVecClasses], C[kVecClasses], E[kVecClasses], T;
    size_t scratch_bytes = 0;
};

// The widest vector of consecutive levels, as a power of two, that the
// member's rows and pointers allow: up to 16 bytes of q and of its binary32
// scratch, whole vectors only (L and ld multiples of it).
template <typename TQ> int vec_class(const grist_tracer_member &u) {
    auto at = [](const void *p, size_t a) { return ((uintptr_t)p) % a == 0; };
    for (int c = sizeof(TQ) == 4 ? 2 : 1; c > 0; c--) {
        const int V = 1 << c;
        if (u.n_levels % V == 0 && u.ld % V == 0 && at(u.q, V * sizeof(TQ)) && at(u.dpi, 16) && at(u.mass_flux, 16))
            return c;
    }
    return 0;
}

template <typename TQ, typename TC>
int plan_batch(const DevMesh &m, const grist_tracer_batch *b, int tpt, int lpt, HostPlan &P) {
    P = HostPlan();
    size_t off = 0;
    unsigned long long tD[kVecClasses] = {0}, tC[kVecClasses] = {0}, tE[kVecClasses] = {0}, tT = 0;
    const unsigned long long ntiles = ((unsigned long long)m.nC + kTileCells - 1) / kTileCells;
    for (int i = 0; i < b->n_members; i++) {
        const grist_tracer_member &u = b->members[i];
        if (u.n_levels == 0 || u.n_tracers == 0) continue;
        MemberDev d{};
        d.q = u.q;
        d.dpi = u.dpi;
        d.F = u.mass_flux;
        d.L = u.n_levels;
        d.T = u.n_tracers;
        d.ld = u.ld;
        d.Mv = u.vmass_flux;
        d.ldi = u.ld_int;
        // levels_per_thread 1 is one level; 2 is a vector where the layout
        // allows one, else two levels Lg apart
        const int vc = lpt > 1 ? vec_class<TQ>(u) : 0;
        d.Lg = vc ? u.n_levels >> vc : (u.n_levels + lpt - 1) / lpt;
        d.DL = make_div((uint32_t)d.Lg);
        d.qs = (unsigned long long)m.nC * u.ld;
        d.fs = (unsigned long long)m.nE * u.ld;
        // scratch offsets (relative, resolved after allocation)
        const size_t bq = (size_t)d.T * d.qs * sizeof(TQ), bf = (size_t)d.T * d.fs * sizeof(TC),
                     br = (size_t)d.T * d.qs * sizeof(TC);
        d.qA = (void *)(uintptr_t)off; off += al256(bq);
        d.qB = (void *)(uintptr_t)off; off += al256(bq);
        d.FH = (void *)(uintptr_t)off; off += al256(bf);
        d.R2 = (void *)(uintptr_t)off; off += al256(2 * br);
        d.X2 = (void *)(uintptr_t)off; off += al256(2 * br);
        d.DFL = (void *)(uintptr_t)off; off += al256(br);
        if (sizeof(TC) == 4) { d.Ff = (const void *)(uintptr_t)off; off += al256(d.fs * sizeof(float)); }
        d.DV = (void *)(uintptr_t)off; off += al256(d.qs * 2 * sizeof(TC));
        const int idx = (int)P.mem.size();
        const int G = (d.T + tpt - 1) / tpt;
        auto add = [&](HostPlan::Seg &S, unsigned long long &tot, int g, unsigned long long n) {
            S.start.push_back(tot);
            S.mg.push_back(make_int2(idx, g));
            tot += n;
        };
        add(P.D[vc], tD[vc], 0, (unsigned long long)m.nC * d.Lg);
        for (int g = 0; g < G; g++) {
            add(P.C[vc], tC[vc], g, (unsigned long long)m.nC * d.Lg);
            add(P.E[vc], tE[vc], g, (unsigned long long)m.nE * d.Lg);
            add(P.T, tT, g, ntiles * (unsigned long long)((d.L + 31) / 32));
        }
        P.mem.push_back(d);
    }
    for (int c = 0; c < kVecClasses; c++) {
        P.D[c].start.push_back(tD[c]);
        P.C[c].start.push_back(tC[c]);
        P.E[c].start.push_back(tE[c]);
    }
    P.T.start.push_back(tT);
    P.scratch_bytes = off;
    return GRIST_OK;
}

// Upload the plan's tables (member descriptors with resolved scratch
// pointers, segment tables) into the context's device table; returns the
// Batch with device pointers.  Synchronous when the tables change.
template <typename TQ, typename TC>
int upload_plan(grist_mesh_s *h, TracerCtx *c, HostPlan &P, const grist_tracer_batch *b, double dt, Batch &B,
                cudaStream_t st) {
    char *scr = (char *)scratch(h, 0, P.scratch_bytes + 256);
    if (!scr) return GRIST_ENOMEM;
    for (auto &d : P.mem) {
        d.qA = scr + (uintptr_t)d.qA;
        d.qB = scr + (uintptr_t)d.qB;
        d.FH = scr + (uintptr_t)d.FH;
        d.R2 = scr + (uintptr_t)d.R2;
        d.X2 = scr + (uintptr_t)d.X2;
        d.DFL = scr + (uintptr_t)d.DFL;
        d.Ff = sizeof(TC) == 4 ? (const void *)(scr + (uintptr_t)d.Ff) : (const void *)d.F;
        d.DV = scr + (uintptr_t)d.DV;
    }
    const size_t nm = P.mem.size();
    size_t o = 0;
    const size_t o_mem = o; o += al256(nm * sizeof(MemberDev));
    auto each = [&](auto &&fn) {
        for (int k = 0; k < kVecClasses; k++) {
            fn(P.D[k], B.D[k]);
            fn(P.C[k], B.C[k]);
            fn(P.E[k], B.E[k]);
        }
        fn(P.T, B.T);
    };
    each([&](HostPlan::Seg &S, Space &) {
        S.o_start = o; o += al256(S.start.size() * 8);
        S.o_mg = o; o += al256(S.mg.size() * sizeof(int2));
    });
    std::vector<char> ht(o, 0);
    std::memcpy(ht.data() + o_mem, P.mem.data(), nm * sizeof(MemberDev));
    each([&](HostPlan::Seg &S, Space &) {
        std::memcpy(ht.data() + S.o_start, S.start.data(), S.start.size() * 8);
        if (!S.mg.empty()) std::memcpy(ht.data() + S.o_mg, S.mg.data(), S.mg.size() * sizeof(int2));
    });
    int ti = -1;
    for (size_t x = 0; x < c->tabs.size() && ti < 0; x++)
        if (c->tabs[x].host.size() == o && std::memcmp(c->tabs[x].host.data(), ht.data(), o) == 0) ti = (int)x;
    if (ti < 0) {
        // a batch not seen before: its table is made outside any stream
        // capture (a recorded step must have run once without capture)
        cudaStreamCaptureStatus cs = cudaStreamCaptureStatusNone;
        GRIST_CUDA_TRY(cudaStreamIsCapturing(st, &cs));
        if (cs != cudaStreamCaptureStatusNone) return GRIST_EUNSUPPORTED;
        if (c->tabs.size() >= kTableCache) {
            // drop the oldest table (and the tracer graphs, which may read it)
            GRIST_CUDA_TRY(cudaDeviceSynchronize());
            c->drop_graphs();
            cudaFree(c->tabs.front().dev);
            c->tabs.erase(c->tabs.begin());
        }
        TracerCtx::Table t;
        if (cudaMalloc(&t.dev, o) != cudaSuccess) return GRIST_ENOMEM;
        if (cudaMemcpy(t.dev, ht.data(), o, cudaMemcpyHostToDevice) != cudaSuccess) {
            cudaFree(t.dev);
            return GRIST_ECUDA;
        }
        t.host = ht;
        c->tabs.push_back(std::move(t));
        ti = (int)c->tabs.size() - 1;
    }
    c->cur = ti;
    char *dtab = c->tabs[ti].dev;
    if (!c->barrier) {
        if (cudaMalloc(&c->barrier, 4 * sizeof(unsigned)) != cudaSuccess) return GRIST_ENOMEM;
        GRIST_CUDA_TRY(cudaMemset(c->barrier, 0, 4 * sizeof(unsigned)));
    }
    B.mem = (const MemberDev *)(dtab + o_mem);
    B.nm = (int)nm;
    each([&](HostPlan::Seg &S, Space &D) {
        D = Space{(const unsigned long long *)(dtab + S.o_start), (const int2 *)(dtab + S.o_mg), (int)S.mg.size(),
                  S.start.back()};
    });
    B.tpt = c->tune.tracers_per_thread;
    B.lpt = c->tune.persistent ? 1 : c->tune.levels_per_thread;
    B.dt = dt;
    B.dt3 = dt / 3.0;
    B.fct = b->limiter ? 1 : 0;
    B.beta1 = b->beta_upwind == 1.0 ? 1 : 0;
    B.ring = (c->tune.cell_edges && B.beta1 && dev_mesh(h).ring_ok) ? 1 : 0;
    B.beta = b->beta_upwind;
    B.cmax = b->vertical_courant_max;
    return GRIST_OK;
}

int sm_count(int dev) {
    int n = 0;
    cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev);
    return n > 0 ? n : 1;
}

int build_tiles(grist_mesh_s *h, TracerCtx *c);

// Enqueue the horizontal phases (no host synchronisation: capturable).
template <typename TQ, typename TC>
int enqueue_horizontal(grist_mesh_s *h, TracerCtx *c, const Batch &B, cudaStream_t st) {
    const DevMesh &m = dev_mesh(h);
    uint32_t *status = status_word(h);
    const int block = c->tune.block;
    const int dev = mesh_device(h);
    if (B.nm == 0) return GRIST_OK;
    if (c->tune.persistent) {
        int per_sm = 0;
        GRIST_CUDA_TRY(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_tracer_persistent<TQ, TC>, block, 0));
        if (per_sm < 1) return GRIST_EUNSUPPORTED;
        const int grid = per_sm * sm_count(dev);
        DevMesh mm = m;
        Batch bb = B;
        unsigned *bar = c->barrier;
        GRIST_CUDA_TRY(cudaMemsetAsync(bar, 0, 3 * sizeof(unsigned), st));
        void *args[] = {&mm, &bb, &bar, &status};
        GRIST_LAUNCH(h, PN("k_tracer_persistent"), st,
                     GRIST_CUDA_TRY(cudaLaunchCooperativeKernel((const void *)k_tracer_persistent<TQ, TC>, grid, block,
                                                                args, 0, st)));
        return GRIST_OK;
    }
    static const char *names_f[] = {"k_tr_div/mix", "k_tr_edge/mix", "k_tr_update/mix", "k_tr_edge/mix",
                                    "k_tr_update/mix", "k_tr_edge/mix", "k_tr_update/mix", "k_tr_lowres/mix",
                                    "k_tr_ratios/mix", "k_tr_final/mix"};
    static const char *names_d[] = {"k_tr_div/fp64", "k_tr_edge/fp64", "k_tr_update/fp64", "k_tr_edge/fp64",
                                    "k_tr_update/fp64", "k_tr_edge/fp64", "k_tr_update/fp64", "k_tr_lowres/fp64",
                                    "k_tr_ratios/fp64", "k_tr_final/fp64"};
    const int sms = sm_count(dev);
    const bool fused = c->tune.fused != 0;
    if (fused) {
        int rc = build_tiles(h, c);
        if (rc != GRIST_OK) return rc;
    }
    const size_t tile_smem = (size_t)(c->tiles.Hmax + c->tiles.Emax) * 32 * sizeof(TC);
    auto launch_tile = [&](int stage) -> int {
        if (B.T.total == 0) return GRIST_OK;
        const unsigned grid = (unsigned)B.T.total;
        if (B.beta1) {
            GRIST_CUDA_TRY(cudaFuncSetAttribute(k_tr_tile_stage<TQ, TC, true>,
                                                cudaFuncAttributeMaxDynamicSharedMemorySize, (int)tile_smem));
            GRIST_LAUNCH(h, sizeof(TC) == 4 ? "k_tr_tile_stage/mix" : "k_tr_tile_stage/fp64", st,
                         k_tr_tile_stage<TQ, TC, true><<<grid, 256, tile_smem, st>>>(m, c->tiles, B, stage, status));
        } else {
            GRIST_CUDA_TRY(cudaFuncSetAttribute(k_tr_tile_stage<TQ, TC, false>,
                                                cudaFuncAttributeMaxDynamicSharedMemorySize, (int)tile_smem));
            GRIST_LAUNCH(h, sizeof(TC) == 4 ? "k_tr_tile_stage/mix" : "k_tr_tile_stage/fp64", st,
                         k_tr_tile_stage<TQ, TC, false><<<grid, 256, tile_smem, st>>>(m, c->tiles, B, stage, status));
        }
        return GRIST_OK;
    };
    for (int ph = P_DIV; ph < P_NPHASE; ph++) {
        if (!B.fct && ph > P_UPD2) break;
        if (B.fct && ph == P_UPD2) continue;
        // the cell-centric first edge phase of a limited step does the
        // low-order phase too (a fused stage has no such edge phase)
        const bool with_low = B.fct && B.ring && !fused;
        if (ph == P_LOWRES && with_low) continue;
        if (fused && (ph == P_EDGE0 || ph == P_EDGE1 || (!B.fct && ph == P_EDGE2))) continue;
        if (fused && (ph == P_UPD0 || ph == P_UPD1 || ph == P_UPD2)) {
            const int rc = launch_tile(ph == P_UPD0 ? 0 : (ph == P_UPD1 ? 1 : 2));
            if (rc != GRIST_OK) return rc;
            continue;
        }
        const char *nm = ph == P_EDGE0 && with_low ? (sizeof(TC) == 4 ? "k_tr_edge_low/mix" : "k_tr_edge_low/fp64")
                         : sizeof(TC) == 4         ? names_f[ph]
                                                   : names_d[ph];
        for (int cls = 0; cls < kVecClasses; cls++) {
            const unsigned long long total = phase_space(B, ph, B.ring != 0, cls).total;
            if (total == 0) continue;
            const long long want = (long long)((total + block - 1) / block);
            const long long cap = (long long)sms * 2048 * 32 / block;  // enough blocks to fill every SM many times
            const unsigned grid = (unsigned)(want > cap ? cap : want);
            switch (ph) {
#define GRIST_PHASE_LAUNCH(P_, R_)                                                                              \
    if constexpr (sizeof(TC) == 4) {                                                                            \
        if (cls == 2)                                                                                           \
            GRIST_LAUNCH(h, nm, st, (k_tracer_phase<TQ, TC, P_, 1, 4, R_><<<grid, block, 0, st>>>(m, B, status))); \
    }                                                                                                           \
    if (cls == 1)                                                                                               \
        GRIST_LAUNCH(h, nm, st, (k_tracer_phase<TQ, TC, P_, 1, 2, R_><<<grid, block, 0, st>>>(m, B, status)));  \
    else if (cls == 0 && B.lpt == 2)                                                                            \
        GRIST_LAUNCH(h, nm, st, (k_tracer_phase<TQ, TC, P_, 2, 1, R_><<<grid, block, 0, st>>>(m, B, status)));  \
    else if (cls == 0)                                                                                          \
        GRIST_LAUNCH(h, nm, st, (k_tracer_phase<TQ, TC, P_, 1, 1, R_><<<grid, block, 0, st>>>(m, B, status)));
#define GRIST_PHASE_CASE(P_)                     \
    case P_:                                     \
        if constexpr (is_edge_phase(P_)) {       \
            if (P_ == P_EDGE0 && with_low) {     \
                GRIST_PHASE_LAUNCH(P_, P_ == P_EDGE0 ? 2 : 1) \
            } else if (B.ring) {                 \
                GRIST_PHASE_LAUNCH(P_, 1)        \
            } else {                             \
                GRIST_PHASE_LAUNCH(P_, 0)        \
            }                                    \
        } else {                                 \
            GRIST_PHASE_LAUNCH(P_, 0)            \
        }                                        \
        break;
                GRIST_PHASE_CASE(P_DIV)
                GRIST_PHASE_CASE(P_EDGE0)
                GRIST_PHASE_CASE(P_UPD0)
                GRIST_PHASE_CASE(P_EDGE1)
                GRIST_PHASE_CASE(P_UPD1)
                GRIST_PHASE_CASE(P_EDGE2)
                GRIST_PHASE_CASE(P_UPD2)
                GRIST_PHASE_CASE(P_LOWRES)
                GRIST_PHASE_CASE(P_RATIOS)
                GRIST_PHASE_CASE(P_FINAL)
#undef GRIST_PHASE_CASE
#undef GRIST_PHASE_LAUNCH
            }
        }
    }
    return cudaGetLastError() == cudaSuccess ? GRIST_OK : GRIST_ECUDA;
}

// The step: the horizontal phases, then the vertical transport of every
// member that has a vertical mass flux (one launch per such member; the
// members' resolved descriptors are the host mirror of the device table).
template <typename TQ, typename TC>
int enqueue_step(grist_mesh_s *h, TracerCtx *c, const Batch &B, cudaStream_t st) {
    int rc = enqueue_horizontal<TQ, TC>(h, c, B, st);
    if (rc != GRIST_OK) return rc;
    const DevMesh &m = dev_mesh(h);
    const MemberDev *hm = reinterpret_cast<const MemberDev *>(c->tabs[c->cur].host.data());
    for (int j = 0; j < B.nm; j++) {
        if (!hm[j].Mv) continue;
        const unsigned gv = grid_for(m.nC, kVertWarps);
        const int K = (hm[j].L + 31) / 32;
        const bool vec = hm[j].L % K == 0 && hm[j].ld % K == 0 && (uintptr_t)hm[j].q % std::min<size_t>(16, K * sizeof(TQ)) == 0;
        auto go = [&](auto kern) {
            GRIST_LAUNCH(h, sizeof(TC) == 4 ? "k_tr_vertical/mix" : "k_tr_vertical/fp64", st,
                         (kern<<<gv, kVertWarps * 32, 0, st>>>(m, hm[j], B.dt, B.cmax, status_word(h))));
        };
        if (K == 1) go(k_tr_vertical<TQ, TC, 1, false>);
        else if (K == 2 && vec) go(k_tr_vertical<TQ, TC, 2, true>);
        else if (K == 2) go(k_tr_vertical<TQ, TC, 2, false>);
        else if (K == 3) go(k_tr_vertical<TQ, TC, 3, false>);
        else if (vec) go(k_tr_vertical<TQ, TC, 4, true>);
        else go(k_tr_vertical<TQ, TC, 4, false>);
    }
    return cudaGetLastError() == cudaSuccess ? GRIST_OK : GRIST_ECUDA;
}

// Build the tile tables of the mesh (once per handle) and upload them.
int build_tiles(grist_mesh_s *h, TracerCtx *c) {
    if (c->dtile) return GRIST_OK;
    const HostTables &ht = host_tables(h);
    const int nC = ht.nC;
    const int nt = (nC + kTileCells - 1) / kTileCells;
    std::vector<int> hoff(nt + 1, 0), eoff(nt + 1, 0), halo, tedge;
    std::vector<uint16_t> eloc, cle((size_t)nt * kTileCells * 6, 0);
    int Hmax = 0, Emax = 0;
    std::vector<int> cells, edges;
    for (int t = 0; t < nt; t++) {
        const int c0 = t * kTileCells, c1 = std::min(nC, c0 + kTileCells);
        edges.clear();
        for (int i = c0; i < c1; i++)
            for (int j = 0; j < 6; j++) edges.push_back(ht.eoc[(size_t)i * 6 + j]);
        std::sort(edges.begin(), edges.end());
        edges.erase(std::unique(edges.begin(), edges.end()), edges.end());
        cells.clear();
        for (int e : edges) {
            cells.push_back(ht.coe[e].x);
            cells.push_back(ht.coe[e].y);
            for (int q = 0; q < 14; q++) cells.push_back(ht.d2i[(size_t)e * 14 + q]);
        }
        std::sort(cells.begin(), cells.end());
        cells.erase(std::unique(cells.begin(), cells.end()), cells.end());
        if (cells.size() > 65535 || edges.size() > 65535) return GRIST_EUNSUPPORTED;
        auto loc = [&](int cell) {
            return (uint16_t)(std::lower_bound(cells.begin(), cells.end(), cell) - cells.begin());
        };
        for (int e : edges) {
            eloc.push_back(loc(ht.coe[e].x));
            eloc.push_back(loc(ht.coe[e].y));
            for (int q = 0; q < 14; q++) eloc.push_back(loc(ht.d2i[(size_t)e * 14 + q]));
        }
        for (int i = c0; i < c1; i++)
            for (int j = 0; j < 6; j++)
                cle[(size_t)i * 6 + j] = (uint16_t)(std::lower_bound(edges.begin(), edges.end(),
                                                                     ht.eoc[(size_t)i * 6 + j]) - edges.begin());
        halo.insert(halo.end(), cells.begin(), cells.end());
        tedge.insert(tedge.end(), edges.begin(), edges.end());
        hoff[t + 1] = (int)halo.size();
        eoff[t + 1] = (int)tedge.size();
        Hmax = std::max(Hmax, (int)cells.size());
        Emax = std::max(Emax, (int)edges.size());
    }
    size_t o = 0;
    const size_t o_hoff = o; o += al256(hoff.size() * 4);
    const size_t o_halo = o; o += al256(halo.size() * 4);
    const size_t o_eoff = o; o += al256(eoff.size() * 4);
    const size_t o_tedge = o; o += al256(tedge.size() * 4);
    const size_t o_eloc = o; o += al256(eloc.size() * 2);
    const size_t o_cle = o; o += al256(cle.size() * 2);
    std::vector<char> hb(o, 0);
    std::memcpy(hb.data() + o_hoff, hoff.data(), hoff.size() * 4);
    std::memcpy(hb.data() + o_halo, halo.data(), halo.size() * 4);
    std::memcpy(hb.data() + o_eoff, eoff.data(), eoff.size() * 4);
    std::memcpy(hb.data() + o_tedge, tedge.data(), tedge.size() * 4);
    std::memcpy(hb.data() + o_eloc, eloc.data(), eloc.size() * 2);
    std::memcpy(hb.data() + o_cle, cle.data(), cle.size() * 2);
    char *d = nullptr;
    if (cudaMalloc(&d, o) != cudaSuccess) return GRIST_ENOMEM;
    if (cudaMemcpy(d, hb.data(), o, cudaMemcpyHostToDevice) != cudaSuccess) {
        cudaFree(d);
        return GRIST_ECUDA;
    }
    c->dtile = d;
    TileMesh &T = c->tiles;
    T.ntiles = nt;
    T.Hmax = Hmax;
    T.Emax = Emax;
    T.hoff = (const int *)(d + o_hoff);
    T.halo = (const int *)(d + o_halo);
    T.eoff = (const int *)(d + o_eoff);
    T.tedge = (const int *)(d + o_tedge);
    T.eloc = (const uint16_t *)(d + o_eloc);
    T.cle = (const uint16_t *)(d + o_cle);
    return GRIST_OK;
}

TracerCtx *ctx_of(grist_mesh_s *h) {
    TracerCtx *&c = tracer_ctx(h);
    if (!c) c = new TracerCtx();
    return c;
}

template <typename TQ, typename TC>
int tracer_step_t(grist_mesh_s *h, const grist_tracer_batch *b, double dt, cudaStream_t st) {
    TracerCtx *c = ctx_of(h);
    const DevMesh &m = dev_mesh(h);
    HostPlan P;
    int rc = plan_batch<TQ, TC>(m, b, c->tune.tracers_per_thread, c->tune.persistent ? 1 : c->tune.levels_per_thread, P);
    if (rc != GRIST_OK) return rc;
    Batch B;
    rc = upload_plan<TQ, TC>(h, c, P, b, dt, B, st);
    if (rc != GRIST_OK) return rc;
    if (!c->tune.use_graph || profiling(h)) return enqueue_step<TQ, TC>(h, c, B, st);
    // graph path: signature = batch contents + tuning + dt + stream
    std::vector<unsigned long long> sig;
    sig.push_back((unsigned long long)b->prec);
    sig.push_back((unsigned long long)b->limiter);
    unsigned long long u;
    std::memcpy(&u, &b->beta_upwind, 8); sig.push_back(u);
    std::memcpy(&u, &dt, 8); sig.push_back(u);
    std::memcpy(&u, &b->vertical_courant_max, 8); sig.push_back(u);
    sig.push_back((unsigned long long)(uintptr_t)st);
    sig.push_back(((unsigned long long)c->tune.block << 32) | (unsigned)c->tune.tracers_per_thread);
    sig.push_back((unsigned long long)c->tune.persistent | ((unsigned long long)c->tune.levels_per_thread << 8) |
                  ((unsigned long long)c->tune.fused << 16) | ((unsigned long long)c->tune.cell_edges << 24));
    for (int i = 0; i < b->n_members; i++) {
        const grist_tracer_member &mm = b->members[i];
        sig.push_back((unsigned long long)(uintptr_t)mm.q);
        sig.push_back((unsigned long long)(uintptr_t)mm.dpi);
        sig.push_back((unsigned long long)(uintptr_t)mm.mass_flux);
        sig.push_back(((unsigned long long)mm.n_levels << 40) | ((unsigned long long)mm.n_tracers << 20) |
                      (unsigned long long)mm.ld);
        sig.push_back((unsigned long long)(uintptr_t)mm.vmass_flux);
        sig.push_back((unsigned long long)mm.ld_int);
    }
    sig.push_back((unsigned long long)(uintptr_t)c->tabs[c->cur].dev);
    // inside a caller's capture (a whole-step graph) the kernels are
    // recorded directly into that graph
    cudaStreamCaptureStatus cs;
    GRIST_CUDA_TRY(cudaStreamIsCapturing(st, &cs));
    if (cs != cudaStreamCaptureStatusNone || st == nullptr) return enqueue_step<TQ, TC>(h, c, B, st);
    for (auto &ge : c->graphs)
        if (ge.sig == sig) {
            GRIST_CUDA_TRY(cudaGraphLaunch(ge.exec, st));
            return GRIST_OK;
        }
    if (c->graph_failed && sig == c->failed_sig) return enqueue_step<TQ, TC>(h, c, B, st);
    GRIST_CUDA_TRY(cudaStreamBeginCapture(st, cudaStreamCaptureModeThreadLocal));
    int erc = enqueue_step<TQ, TC>(h, c, B, st);
    cudaGraph_t g = nullptr;
    cudaGraphExec_t ex = nullptr;
    cudaError_t ce = cudaStreamEndCapture(st, &g);
    if (erc != GRIST_OK || ce != cudaSuccess || !g || cudaGraphInstantiate(&ex, g, 0) != cudaSuccess) {
        // this batch cannot be captured (e.g. the cooperative launch): run
        // it directly and remember not to retry the capture
        if (g) cudaGraphDestroy(g);
        cudaGetLastError();
        c->graph_failed = true;
        c->failed_sig = sig;
        return enqueue_step<TQ, TC>(h, c, B, st);
    }
    if (c->graphs.size() >= kGraphCache) {
        // evict the oldest; its last replay may still be queued on a stream
        GRIST_CUDA_TRY(cudaDeviceSynchronize());
        cudaGraphExecDestroy(c->graphs.front().exec);
        cudaGraphDestroy(c->graphs.front().graph);
        c->graphs.erase(c->graphs.begin());
    }
    TracerCtx::GraphEntry ge;
    ge.sig = sig;
    ge.graph = g;
    ge.exec = ex;
    c->graphs.push_back(ge);
    GRIST_CUDA_TRY(cudaGraphLaunch(ex, st));
    return GRIST_OK;
}

int validate(const grist_tracer_batch *b, double dt) {
    if (!b || (b->n_members > 0 && !b->members) || b->n_members < 0) return GRIST_EINVAL;
    if (b->n_members > GRIST_MAX_MEMBERS) return GRIST_EUNSUPPORTED;
    if (!(dt > 0) || !std::isfinite(dt)) return GRIST_EINVAL;
    if (b->prec != GRIST_FP64 && b->prec != GRIST_MIX && b->prec != GRIST_MIX_DBL_MASS && b->prec != GRIST_MIX_DF)
        return GRIST_EINVAL;
    if (!std::isfinite(b->beta_upwind)) return GRIST_EINVAL;
    for (int i = 0; i < b->n_members; i++) {
        const grist_tracer_member &mb = b->members[i];
        if (mb.n_levels < 0 || mb.n_tracers < 0 || mb.n_levels > GRIST_MAXL || mb.ld < mb.n_levels) return GRIST_EINVAL;
        if (mb.n_levels > 0 && mb.n_tracers > 0 && (!mb.q || !mb.dpi || !mb.mass_flux)) return GRIST_EINVAL;
        if (mb.vmass_flux && mb.ld_int < mb.n_levels + 1) return GRIST_EINVAL;
        if (mb.vmass_flux && mb.n_levels > kVertMaxL) return GRIST_EUNSUPPORTED;
    }
    if (!(b->vertical_courant_max >= 0.0)) return GRIST_EINVAL;   // NaN and negatives; +inf: explicit only
    return GRIST_OK;
}

int dispatch(grist_mesh_s *h, const grist_tracer_batch *b, double dt, cudaStream_t st) {
    return b->prec == GRIST_FP64 ? tracer_step_t<double, double>(h, b, dt, st) : tracer_step_t<float, float>(h, b, dt, st);
}

int check_tuning(const grist_tracer_tuning *t) {
    if (!t) return GRIST_EINVAL;
    if (t->block < 64 || t->block > kTracerMaxBlock || t->block % 32) return GRIST_EINVAL;
    if (t->tracers_per_thread < 1 || t->tracers_per_thread > 64) return GRIST_EINVAL;
    if (t->persistent != 0 && t->persistent != 1) return GRIST_EINVAL;
    if (t->use_graph != 0 && t->use_graph != 1) return GRIST_EINVAL;
    if (t->fused != 0 && t->fused != 1) return GRIST_EINVAL;
    if (t->levels_per_thread != 1 && t->levels_per_thread != 2) return GRIST_EINVAL;
    if (t->cell_edges != 0 && t->cell_edges != 1) return GRIST_EINVAL;
    return GRIST_OK;
}

}  // namespace
}  // namespace grist

using namespace grist;

extern "C" int grist_tracer_step(grist_mesh h, const grist_tracer_batch *b, double dt, void *stream) {
    if (!h) return GRIST_EINVAL;
    int rc = validate(b, dt);
    if (rc != GRIST_OK) return rc;
    if (cudaSetDevice(mesh_device(h)) != cudaSuccess) return GRIST_ECUDA;
    return dispatch(h, b, dt, (cudaStream_t)stream);
}

extern "C" int grist_selftest_bounded_wait(grist_mesh h, int64_t spin_limit, void *stream) {
    if (!h || spin_limit < 1 || spin_limit > 100000000) return GRIST_EINVAL;
    if (cudaSetDevice(mesh_device(h)) != cudaSuccess) return GRIST_ECUDA;
    TracerCtx *c = ctx_of(h);
    if (!c->barrier) {
        if (cudaMalloc(&c->barrier, 4 * sizeof(unsigned)) != cudaSuccess) return GRIST_ENOMEM;
        GRIST_CUDA_TRY(cudaMemset(c->barrier, 0, 4 * sizeof(unsigned)));
    }
    // word 3 is written by no kernel; word 2 is cleared first so the wait
    // runs to its own limit
    cudaStream_t st = (cudaStream_t)stream;
    GRIST_CUDA_TRY(cudaMemsetAsync(c->barrier + 2, 0, sizeof(unsigned), st));
    k_wait_selftest<<<1, 32, 0, st>>>(c->barrier + 3, c->barrier + 2, (long long)spin_limit, status_word(h));
    return cudaGetLastError() == cudaSuccess ? GRIST_OK : GRIST_ECUDA;
}

extern "C" int grist_tracer_set_tuning(grist_mesh h, const grist_tracer_tuning *t) {
    if (!h) return GRIST_EINVAL;
    int rc = check_tuning(t);
    if (rc != GRIST_OK) return rc;
    TracerCtx *c = ctx_of(h);
    c->tune = *t;
    return GRIST_OK;
}

extern "C" int grist_tracer_get_tuning(grist_mesh h, grist_tracer_tuning *t) {
    if (!h || !t) return GRIST_EINVAL;
    *t = ctx_of(h)->tune;
    return GRIST_OK;
}

extern "C" int grist_tracer_autotune(grist_mesh h, const grist_tracer_batch *b, double dt, int32_t steps,
                                     void *stream, grist_tracer_tuning *best, double *best_ms) {
    if (!h || !best || steps < 1) return GRIST_EINVAL;
    int rc = validate(b, dt);
    if (rc != GRIST_OK) return rc;
    if (cudaSetDevice(mesh_device(h)) != cudaSuccess) return GRIST_ECUDA;
    cudaStream_t st = (cudaStream_t)stream;
    TracerCtx *c = ctx_of(h);
    const grist_tracer_tuning saved = c->tune;
    const DevMesh &m = dev_mesh(h);
    // private copies of the tracers
    std::vector<grist_tracer_member> mem(b->members, b->members + b->n_members);
    std::vector<void *> copies;
    const size_t es = b->prec == GRIST_FP64 ? 8 : 4;
    int maxT = 1;
    for (auto &mb : mem) {
        if (mb.n_levels == 0 || mb.n_tracers == 0) continue;
        maxT = mb.n_tracers > maxT ? mb.n_tracers : maxT;
        const size_t bytes = (size_t)mb.n_tracers * m.nC * mb.ld * es;
        void *p = nullptr;
        if (cudaMalloc(&p, bytes) != cudaSuccess) {
            for (void *q : copies) cudaFree(q);
            return GRIST_ENOMEM;
        }
        cudaMemcpyAsync(p, mb.q, bytes, cudaMemcpyDeviceToDevice, st);
        copies.push_back(p);
        mb.q = p;
    }
    grist_tracer_batch bb = *b;
    bb.members = mem.data();
    cudaEvent_t e0, e1;
    cudaEventCreate(&e0);
    cudaEventCreate(&e1);
    auto time_cfg = [&](const grist_tracer_tuning &t, double *ms) -> int {
        c->tune = t;
        int r = dispatch(h, &bb, dt, st);  // warm-up (and graph capture)
        if (r != GRIST_OK) return r;
        cudaEventRecord(e0, st);
        for (int i = 0; i < steps; i++) {
            r = dispatch(h, &bb, dt, st);
            if (r != GRIST_OK) return r;
        }
        cudaEventRecord(e1, st);
        if (cudaEventSynchronize(e1) != cudaSuccess) return GRIST_ECUDA;
        float f = 0.f;
        cudaEventElapsedTime(&f, e0, e1);
        *ms = f / steps;
        return GRIST_OK;
    };
    grist_tracer_tuning bestt = saved;
    double bestms = 1e300;
    const int blocks[] = {128, 256, 512};
    const int tpts[] = {1, 2, 4, 8};
    for (int fu = 0; fu <= 1; fu++) {
        for (int bl : blocks) {
            for (int tp : tpts) {
                if (tp > 1 && tp / 2 >= maxT) continue;
                grist_tracer_tuning t{bl, tp, 0, 0, fu, 1, 1};
                double ms = 0;
                if (time_cfg(t, &ms) == GRIST_OK && ms < bestms) { bestms = ms; bestt = t; }
            }
        }
    }
    // two levels per thread (work-list phases) at the best tracers per
    // thread, every block size
    {
        const int tp = bestt.tracers_per_thread, fu = bestt.fused;
        for (int bl : blocks) {
            grist_tracer_tuning t{bl, tp, 0, 0, fu, 2, 1};
            double ms = 0;
            if (time_cfg(t, &ms) == GRIST_OK && ms < bestms) { bestms = ms; bestt = t; }
        }
    }
    // the edge-centric form of the edge fluxes at the best so far
    {
        grist_tracer_tuning t = bestt;
        t.cell_edges = 0;
        double ms = 0;
        if (time_cfg(t, &ms) == GRIST_OK && ms < bestms) { bestms = ms; bestt = t; }
    }
    for (int pers = 0; pers <= 1; pers++) {
        for (int gr = 0; gr <= 1; gr++) {
            if (pers == 0 && gr == 0) continue;
            grist_tracer_tuning t = bestt;
            t.persistent = pers;
            t.use_graph = gr;
            if (pers) {
                t.fused = 0;
                t.levels_per_thread = 1;
            }
            double ms = 0;
            if (time_cfg(t, &ms) == GRIST_OK && ms < bestms) { bestms = ms; bestt = t; }
        }
    }
    cudaEventDestroy(e0);
    cudaEventDestroy(e1);
    cudaStreamSynchronize(st);
    for (void *q : copies) cudaFree(q);
    // the cached graphs may refer to the freed copies: drop them
    c->drop_graphs();
    c->tune = bestt;
    *best = bestt;
    if (best_ms) *best_ms = bestms;
    uint32_t flags = 0;
    cudaMemcpy(&flags, status_word(h), sizeof(uint32_t), cudaMemcpyDeviceToHost);
    if (flags & GRIST_FLAG_TIMEOUT) return GRIST_ETIMEOUT;
    return GRIST_OK;
}

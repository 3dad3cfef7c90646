// dycore.cu - GRIST dry dynamical core steps (Eqs. 3-9, Sec. 2.1):
// hydrostatic (RK3 + Mesinger forward-backward) and non-hydrostatic
// (horizontally explicit, vertically implicit) on the Voronoi C-grid, in
// FP64 or the paper's mixed precision (Sec. 2.3): advective terms in the
// policy's single-precision type, pressure gradient / gravity, vertical
// integrals, the equation of state, the column solve, surface pressure and
// layer mass in FP64.
//
// Layer fields [entity][ld], interface fields [cell][ld_int]; one thread per
// (entity, level) or vector of levels for the horizontal stencils, a warp's
// lanes over the levels of a column for the vertical scans (continuity prefix,
// hydrostatic integral) and one thread per column for the tridiagonal solve.
//
// FP64 arithmetic is the scarce resource on this GPU (about 1/60 of the FP32
// rate: an FP64 instruction of a warp holds its scheduler's pipe for 64
// cycles), so divisions by layer masses are replaced by products with
// reciprocals formed once per column / edge / vertex (1/(ps - pi_top)) and
// once per level (1/dB), the equation of state inside a stage is evaluated
// relative to the stage-input state (see pow1p_near0), and exact differences
// and products are taken in integers (sub_near, MulF32).
#include <cmath>
#include <type_traits>
#include <vector>

#include "common.cuh"
#include "forms.cuh"
#include "series.cuh"

#define PN(n) (P::DF ? n "/mixdf" : (sizeof(TA) == 4 ? (sizeof(TM) == 8 ? n "/mixdbl" : n "/mix") : n "/fp64"))

namespace grist {
namespace {

constexpr int kBlock = 256;
constexpr int kNHMax = 128;  // levels supported by the column solver
// Edges or cells that a warp of the mass kernels walks.  The per-entity FP64
// scalars run one entity per lane, so fewer entities waste more of the FP64
// pipe; but with 32 a 10,242-cell mesh has two warps an SM.  8 against 32, us a
// launch: level 5, 30 levels, mass_col 67 / 24, mass_edge 38 / 16; level 8, 60
// levels, 699 / 696 and 595 / 306.
constexpr int kMassGroup = 8;

struct DyPar {
    int L, ld, ldi;
    double pi_top, p0, rd, cp, g, beta, kappa, gamma;
    double obeta, obetag;  // 1 - beta, (1 - beta) g
    double rp0;            // 1/p0, or 0 where p/p0 has to be divided
    const double *B;      // [L+1] interface coordinate
    const double *dB;     // [L]   layer thickness in B
    const double *rdB;    // [L]   1/dB
    const double *hrdBi;  // [L+1] 1/(dB[j-1] + dB[j]) at interior interfaces j (half the reciprocal mean)
    const double *dBi;    // [L+1] (dB[j-1] + dB[j])/2 at interior interfaces j
    const double *Bm;     // [L]   (B[k] + B[k+1])/2, mid-layer coordinate, rounded,
    const double *Bml;    // [L]   and the rest of it
    const float *dBf;     // [L]   dB rounded to single precision
    const double *phis;   // [nC]  surface geopotential
    uint32_t emu;         // GRIST_ROW_* rows rounded to binary32 (precision search)
};

// Whether the pressure, geopotential and column kernels take forms that round
// differently from the first ones (tabled reference columns, dphi/th as one
// field, the PV flux in two sums): the FP64 policy only.  In the mixed policies these fields feed binary32
// values (u, the mass flux, the advection of w and phi) by differences, and
// an ulp of phi moves some of those by a whole binary32 rounding; there the
// kernels keep every bit.  (The emulating FP64 variant equals the FP64 policy
// bit for bit where no emulated row is involved, so it takes them too.)
template <class P> constexpr bool short_forms() { return sizeof(typename P::TA) == 8; }

// Storage-rounding emulation of a single-precision row (precision search,
// Sec. 2.2 Eqs. 1-2): in the emulating FP64 policy (E) a double value of a
// row whose bit is set is rounded to binary32 where it is produced; the
// production policies compile to the plain value.
template <bool E> __device__ __forceinline__ double emu(double x, uint32_t mask, uint32_t bit) {
    if (E) return (mask & bit) ? (double)(float)x : x;
    return x;
}
template <bool E> __device__ __forceinline__ float emu(float x, uint32_t, uint32_t) { return x; }

// GRIST_MIX_DF: a double field that the momentum equation only differences
// (layer phi, K) is stored as its double-float split (h, l) in the same
// 8-byte slot, read back as a float2.
__device__ __forceinline__ double pack_split(double x) {
    float h, l;
    split_df(x, h, l);
    return __hiloint2double(__float_as_int(l), __float_as_int(h));
}

// Compensated single-precision accumulation (Knuth's TwoSum): a value is
// hi + lo with |lo| <= ulp(hi)/2, so a sum of FP32 terms carries about 48
// significant bits - as accurate as FP64 accumulation of the same FP32
// terms - while running on the FP32 pipe (FP64 instructions, conversions
// included, are the scarce resource on this GPU).
struct F2 {
    float hi, lo;
};
__device__ __forceinline__ F2 f2_add(F2 a, F2 b) {
    const float s = a.hi + b.hi;
    const float bb = s - a.hi;
    const float e = (a.hi - (s - bb)) + (b.hi - bb);
    const float lo = e + a.lo + b.lo;
    const float hi = s + lo;
    return F2{hi, lo - (hi - s)};
}
__device__ __forceinline__ F2 f2_shfl_xor(F2 v, int o) {
    return F2{__shfl_xor_sync(0xffffffffu, v.hi, o), __shfl_xor_sync(0xffffffffu, v.lo, o)};
}
__device__ __forceinline__ F2 f2_shfl_up(F2 v, int o) {
    return F2{__shfl_up_sync(0xffffffffu, v.hi, o), __shfl_up_sync(0xffffffffu, v.lo, o)};
}

// Sums over a warp's lanes of G values per lane (one column sum per entity),
// lane l ending with the sum of entity l mod G.  The sums add in the order of
// a butterfly (xor 16, 8, 4, 2, 1, own value first) that each entity would
// do for itself, but once a step tells two entities apart a lane keeps the
// partial sum of one and sends that of the other: 31 additions for 32
// entities instead of 5 each.  Entities are visited in bit-reversed order, so
// at most log2(G) partial sums are held.  leaf(j): entity j's value in this
// lane.  FP64 terms are added in FP64, FP32 terms in compensated FP32.
__device__ __forceinline__ double lane_add(double a, double b) { return a + b; }
__device__ __forceinline__ F2 lane_add(F2 a, F2 b) { return f2_add(a, b); }
__device__ __forceinline__ double lane_xor(double v, int o) { return __shfl_xor_sync(0xffffffffu, v, o); }
__device__ __forceinline__ F2 lane_xor(F2 v, int o) { return f2_shfl_xor(v, o); }
__device__ __forceinline__ double lane_pick(bool c, double a, double b) { return c ? a : b; }
__device__ __forceinline__ F2 lane_pick(bool c, F2 a, F2 b) { return F2{c ? a.hi : b.hi, c ? a.lo : b.lo}; }

// Pieces of the column prefix (k_mass_col): lane_carry adds the earlier chunks'
// total, lane_next is the total for the next chunk.
template <class S> __device__ __forceinline__ S lane_zero();
template <> __device__ __forceinline__ double lane_zero<double>() { return 0.0; }
template <> __device__ __forceinline__ F2 lane_zero<F2>() { return F2{0.f, 0.f}; }
template <class S> __device__ __forceinline__ S lane_value(double x) {
    if constexpr (sizeof(S) == 8 && std::is_same<S, double>::value) return x;
    else return F2{cv<float>(x), 0.f};
}
template <class S> __device__ __forceinline__ S lane_value(float x) {
    if constexpr (std::is_same<S, double>::value) return (double)x;
    else return F2{x, 0.f};
}
__device__ __forceinline__ double lane_up(double v, int o) { return __shfl_up_sync(0xffffffffu, v, o); }
__device__ __forceinline__ F2 lane_up(F2 v, int o) { return f2_shfl_up(v, o); }
__device__ __forceinline__ double lane_carry(double run, double v) { return run + v; }
__device__ __forceinline__ F2 lane_carry(F2 run, F2 v) { return f2_add(v, run); }
__device__ __forceinline__ double lane_total(double v) { return v; }
__device__ __forceinline__ double lane_total(F2 v) { return f2d(v.hi) + f2d(v.lo); }
__device__ __forceinline__ double lane_next(double run, double v, double) { return run + __shfl_sync(0xffffffffu, v, 31); }
__device__ __forceinline__ F2 lane_next(F2, F2, F2 pre) {
    return F2{__shfl_sync(0xffffffffu, pre.hi, 31), __shfl_sync(0xffffffffu, pre.lo, 31)};
}

template <int G, int O, class Leaf>   // O: the step that tells this call's two halves apart; 2 G > O >= 1
__device__ __forceinline__ auto entity_sums(Leaf &leaf, int j, int lane) {
    if constexpr (O >= G) {
        auto v = leaf(j);
#pragma unroll
        for (int o = 16; o >= G; o >>= 1) v = lane_add(v, lane_xor(v, o));
        return v;
    } else {
        const auto a = entity_sums<G, 2 * O>(leaf, j, lane);
        const auto b = entity_sums<G, 2 * O>(leaf, j | O, lane);
        const bool up = (lane & O) != 0;
        return lane_add(lane_pick(up, b, a), lane_xor(lane_pick(up, a, b), O));
    }
}

// GRIST_MIX_DF form of p (1 + x)^g for |x| <= 2^-6: the increment
// (1 + x)^g - 1 = x (C1 + x (C2 + ... + x C5)) in binary32 (the omitted
// terms are below 2^-30 of it), added to p in FP64 - the increment's
// binary32 rounding, about 2^-23 |g x|, is ~1e-10 of p for |x| ~ 1e-3.
// Larger |x| (none in a stable step) falls back to the FP64 pow.
__device__ __forceinline__ double scale_near1_df(double p, double x, double g, const Binom &B) {
    const unsigned hx = (unsigned)__double2hiint(x) & 0x7fffffffu;
    if (hx > 0x3f900000u) return p * pow(1.0 + x, g);
    const float xf = d2f(x);
    float s = B.f[5];
#pragma unroll
    for (int n = 4; n >= 1; n--) s = fmaf(s, xf, B.f[n]);
    return fma(p, f2d(s * xf), p);
}

// ---------------------------------------------------------------------------
// Eq. 3: mass flux at edges F = dpi_e u, dpi_e = mean of the two cells'
// layer mass = dB_k (ps1 + ps2 - 2 pi_top)/2.  One warp takes G edges: the
// per-edge FP64 work (column factor, the reciprocal 1/(ps1 + ps2 - 2 pi_top)
// for the momentum equation) runs one edge per lane - an FP64 instruction
// costs the FP64 pipe a full warp slot however few lanes are active - then
// the warp walks its edges with the lanes over levels, forming the product
// in the mass-flux type and the edges' column sums sum_k F_k (entity_sums;
// both cells of the edge later use the same value, so the global mass change
// cancels to round-off).  In the final stage fscale times the flux is
// accumulated for the tracer solver (Sec. 2.3: single computed, saved double).
// Against one edge at a time (its load, product and butterfly of five
// compensated additions in turn, 32 edges a warp), mixed: level 8, 60 levels
// 417 -> 306 us a launch (139 at the DRAM rate), level 5, 30 levels 34 -> 16.
template <class P>
__global__ void __launch_bounds__(kBlock) k_mass_edge(DevMesh m, DyPar d, const double *__restrict__ ps_s,
                            const typename P::TU *__restrict__ u_s, typename P::TM *__restrict__ F,
                            double *__restrict__ Facc, double fscale, double *__restrict__ rsum_e,
                            double *__restrict__ Fcol) {
    const bool scaled = fscale != 1.0;
    using TM = typename P::TM;
    constexpr int G = kMassGroup;
    const int e0 = (int)((blockIdx.x * blockDim.x + threadIdx.x) >> 5) * G;
    const int lane = threadIdx.x & 31;
    if (e0 >= m.nE) return;
    const int ne = min(G, m.nE - e0);
    TM hs_l = 0;
    if (lane < ne) {
        const int2 c = ldg(m.coe + e0 + lane);
        const double sum = (ldg(ps_s + c.x) - d.pi_top) + (ldg(ps_s + c.y) - d.pi_top);
        hs_l = cv<TM>(0.5 * sum);
        rsum_e[e0 + lane] = 0.5 * rcp(sum);   // 1 / (2 dpi_e / dB)
    }
    // two 32-level chunks of all the warp's edges are loaded before the first
    // is used; past the last edge its loads are repeated and nothing is stored
    using Sum = typename std::conditional<sizeof(TM) == 8, double, F2>::type;
    Sum part[G];
    TM hs[G];
#pragma unroll
    for (int j = 0; j < G; j++) {
        part[j] = lane_zero<Sum>();
        hs[j] = __shfl_sync(0xffffffffu, hs_l, j);
    }
    for (int k0 = lane; k0 < d.L; k0 += 64) {
        const bool two = k0 + 32 < d.L;
        typename P::TU u[G][2];
#pragma unroll
        for (int j = 0; j < G; j++) {
            const size_t x = (size_t)(e0 + min(j, ne - 1)) * d.ld + k0;
            u[j][0] = u_s[x];
            u[j][1] = two ? u_s[x + 32] : (typename P::TU)0;
        }
#pragma unroll
        for (int h = 0; h < 2; h++) {
            const int k = k0 + 32 * h;
            if (k >= d.L) break;
            const TM dB = sizeof(TM) == 8 ? (TM)ldg(d.dB + k) : (TM)ldg(d.dBf + k);
#pragma unroll
            for (int j = 0; j < G; j++) {
                if (j >= ne) break;
                const size_t x = (size_t)(e0 + j) * d.ld + k;
                const TM f = emu<P::EMU>(dB * hs[j] * cv<TM>(u[j][h]), d.emu, GRIST_ROW_MASS_FLUX);
                F[x] = f;
                part[j] = lane_add(part[j], lane_value<Sum>(f));
                if (Facc) Facc[x] += scaled ? fscale * cv<double>(f) : cv<double>(f);
            }
        }
    }
    auto leaf = [&](int j) { return part[j]; };
    // lane l ends with edge l mod G; the butterfly of edge j (counted from a
    // multiple of 32) is the one that ends in lane j mod 32
    const auto col = entity_sums<G, 1>(leaf, 0, lane);
    const int at = e0 & 31;
    if (lane >= at && lane < at + ne) {
        if constexpr (sizeof(TM) == 8) Fcol[e0 + lane - at] = col;
        else Fcol[e0 + lane - at] = f2d(col.hi) + f2d(col.lo);
    }
}

// Eq. 3 column part.  One warp takes G cells; the per-cell FP64 work (the
// surface pressure tendency -sum_j s dv/A (column sum of edge j), its stage
// update, 1/(ps - pi_top)) runs one cell per lane, then the warp walks its
// cells with the lanes over levels: layer divergence D_k (mass-flux type),
// vertical mass flux M_{k+1/2} = -B_{k+1/2} dps/dt - sum_{l<=k} D_l by a
// warp scan, theta = (dpi theta)/dpi of the stage input for Eq. 4.  In the
// first stage of the NH core also the t^n state that the column solve's
// equation of state is taken relative to: 1/(dpi theta) and dphi, or their
// product (short_forms).
//
// The two 32-level chunks of a pair are loaded and scanned together (the scans
// are independent until the carry is added), which hides half the shuffles'
// latency.  The scan keeps the order of one 32-lane scan per chunk: M, and so
// the mixed policies, keep their bits.  FP64 policy, level 7, 60 levels
// 528 -> 399 us a launch; mixed, level 8 730 -> 696 (the correctly rounded
// 1/(dpi theta) of the first stage holds the FP64 pipe 80 % there), level 6,
// 30 levels 65 -> 40.
template <class P>
__global__ void __launch_bounds__(kBlock) k_mass_col(DevMesh m, DyPar d, const typename P::TM *__restrict__ F,
                           const double *__restrict__ Fcol, const double *__restrict__ ps_s,
                           const double *__restrict__ ps_n, double *__restrict__ ps_out,
                           const double *__restrict__ th_s, typename P::TA *__restrict__ theta,
                           double *__restrict__ Mv, double dts, double *__restrict__ dpi_out,
                           double *__restrict__ rdps_out, double *__restrict__ rth_out,
                           double *__restrict__ dphi_out, const double *__restrict__ phi_n,
                           double *__restrict__ Macc, double fscale) {
    using TM = typename P::TM;
    using TA = typename P::TA;
    constexpr int G = kMassGroup;
    const int i0 = (int)((blockIdx.x * blockDim.x + threadIdx.x) >> 5) * G;
    const int lane = threadIdx.x & 31;
    if (i0 >= m.nC) return;
    const int nci = min(G, m.nC - i0);
    double pst_l = 0.0, dps_l = 0.0, rdps_l = 0.0;
    if (lane < nci) {
        const int i = i0 + lane;
#pragma unroll
        for (int j = 0; j < GRIST_MAXE; j++) pst_l -= ldg(m.cdiv + i * 6 + j) * ldg(Fcol + ldg(m.eoc + i * 6 + j));
        dps_l = ldg(ps_s + i) - d.pi_top;
        rdps_l = rcp(dps_l);
        ps_out[i] = ps_n[i] + dts * pst_l;
        rdps_out[i] = rdps_l;
        Mv[(size_t)i * d.ldi] = 0.0;
        Mv[(size_t)i * d.ldi + d.L] = 0.0;
    }
    const int nch = (d.L + 31) >> 5;
    using Sum = typename std::conditional<sizeof(TM) == 8, double, F2>::type;
#pragma unroll 1
    for (int c = 0; c < nci; c++) {
        const int i = i0 + c;
        const double pst = __shfl_sync(0xffffffffu, pst_l, c);
        const double dps = __shfl_sync(0xffffffffu, dps_l, c);
        const double rdps = __shfl_sync(0xffffffffu, rdps_l, c);
        int eidx[GRIST_MAXE];
        TM cw[GRIST_MAXE];
        load_row6(m.eoc8, i, eidx);
        load_row6(Coef<TM>::cdiv8(m), i, cw);
        Sum run = lane_zero<Sum>();
        auto chunks = [&](auto count, int ch) {
            constexpr int H = decltype(count)::value;
            Sum v[H];
#pragma unroll
            for (int h = 0; h < H; h++) {
                const int k = (ch + h) * 32 + lane;
                TM s = 0;
                if (k < d.L) {
#pragma unroll
                    for (int j = 0; j < GRIST_MAXE; j++) s += cw[j] * ldg(F + (size_t)eidx[j] * d.ld + k);
                    s = emu<P::EMU>(s, d.emu, GRIST_ROW_MASS_FLUX);
                    const size_t x = (size_t)i * d.ld + k;
                    theta[x] = emu<P::EMU>(cv<TA>(th_s[x] * ldg(d.rdB + k) * rdps), d.emu, GRIST_ROW_THETA);
                    if (dpi_out) dpi_out[x] = ldg(d.dB + k) * dps;
                    if (rth_out) {
                        const size_t y = (size_t)i * d.ldi + k;
                        const double dphi = phi_n[y] - phi_n[y + 1];
                        if constexpr (short_forms<P>()) {
                            rth_out[x] = dphi * rcp(th_s[x]);
                        } else {
                            rth_out[x] = rcp(th_s[x]);
                            dphi_out[x] = dphi;
                        }
                    }
                }
                v[h] = lane_value<Sum>(s);
            }
            // inclusive prefix of D over each chunk, carried across chunks: FP64
            // terms in FP64, FP32 terms in compensated FP32 (the earlier
            // chunks' total too, so the prefix reaches FP64 once, at M)
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
#pragma unroll
                for (int h = 0; h < H; h++) {
                    const Sum t = lane_up(v[h], o);
                    if (lane >= o) v[h] = lane_add(v[h], t);
                }
            }
#pragma unroll
            for (int h = 0; h < H; h++) {
                const int k = (ch + h) * 32 + lane;
                const Sum pre = lane_carry(run, v[h]);
                if (k < d.L - 1) {
                    const double mk = -ldg(d.B + k + 1) * pst - lane_total(pre);
                    Mv[(size_t)i * d.ldi + k + 1] = mk;
                    if (Macc) Macc[(size_t)i * d.ldi + k + 1] += fscale * mk;
                }
                run = lane_next(run, v[h], pre);
            }
        };
        int ch = 0;
#pragma unroll 1
        for (; ch + 1 < nch; ch += 2) chunks(std::integral_constant<int, 2>(), ch);
        if (ch < nch) chunks(std::integral_constant<int, 1>(), ch);
    }
}

// Eq. 4 horizontal flux: third-order upwind (beta = 1) edge value of theta
// times the mass flux.  V = 4 (binary32): a thread takes four consecutive levels
// of one edge as vectors, with one read of the upwind stencil row (4 vector
// loads) where their fluxes run the same way, else level by level; V = 1:
// levels kg and kg + Lh (Lh = ceil(L/2)).  Gathers of 4-byte values are
// latency-bound: level 8, 60 levels, mixed 648 -> 435 us a launch (162 at the
// DRAM rate).  Pairs were not faster: binary32, 30 levels, level 6 25 -> 27;
// FP64 (bound by its pipe), level 7 501 -> 520.
template <class P, int V>
__global__ void __launch_bounds__(kBlock) k_theta_flux(DevMesh m, DyPar d, LevelDiv Dh, const typename P::TM *__restrict__ F,
                             const typename P::TA *__restrict__ th, typename P::TA *__restrict__ Fth) {
    using TA = typename P::TA;
    const int Lh = (int)Dh.d;
    uint32_t n = blockIdx.x * blockDim.x + threadIdx.x;
    if (n >= (uint32_t)m.nE * (uint32_t)Lh) return;
    int e, kg;
    split_index(n, Dh, e, kg);
    int c[GRIST_D2P];
    TA w[GRIST_D2P];
    int loaded = -1;
    auto level = [&](int k) {
        const size_t x = (size_t)e * d.ld + k;
        const TA f = cv<TA>(F[x]);
        const int side = nonneg(f) ? 0 : 1;
        TA te;
        if (m.d2w_ok) {
            // one weighted sum over the upwind side's stencil (the mean of
            // the edge's two cells folded into the weights)
            if (side != loaded) {
                load_d2w(m, e, side, c, w);
                loaded = side;
            }
            te = 0;
#pragma unroll
            for (int j = 0; j < GRIST_D2P; j++) te += w[j] * ldg(th + (size_t)c[j] * d.ld + k);
        } else {
            const int32_t *st = m.d2i + (size_t)e * 14 + side * GRIST_D2P;
            const int2 ce = ldg(m.coe + e);
            const TA *cf = Coef<TA>::d2c(m) + (size_t)e * 14 + side * GRIST_D2P;
            TA sm = 0;
#pragma unroll
            for (int j = 0; j < GRIST_D2P; j++) sm += ldg(cf + j) * ldg(th + (size_t)ldg(st + j) * d.ld + k);
            te = (TA)0.5 * (ldg(th + (size_t)ce.x * d.ld + k) + ldg(th + (size_t)ce.y * d.ld + k)) -
                 (TA)2 * ldg(Coef<TA>::dc2(m) + e) * sm;
        }
        Fth[x] = emu<P::EMU>(f * te, d.emu, GRIST_ROW_THETA);
    };
    if constexpr (V > 1) {
        const size_t x = (size_t)e * d.ld + kg * V;
        typename P::TM fm[V];
        ldgv<V>(F + x, fm);
        TA f[V], q[V], te[V];
        unsigned back = 0;   // bit t: level t's flux runs from c2
#pragma unroll
        for (int t = 0; t < V; t++) {
            f[t] = cv<TA>(fm[t]);
            if (!(f[t] >= (TA)0)) back |= 1u << t;
            te[t] = 0;
        }
        if (m.d2w_ok && (back == 0u || back == (1u << V) - 1u)) {
            load_d2w(m, e, back ? 1 : 0, c, w);
#pragma unroll
            for (int j = 0; j < GRIST_D2P; j++) {
                ldgv<V>(th + (size_t)c[j] * d.ld + kg * V, q);
#pragma unroll
                for (int t = 0; t < V; t++) te[t] += w[j] * q[t];
            }
#pragma unroll
            for (int t = 0; t < V; t++) te[t] *= f[t];
            stgv<V>(Fth + x, te);
        } else {
#pragma unroll 1
            for (int t = 0; t < V; t++)
                if (kg * V + t < d.L) level(kg * V + t);
        }
    } else {
        level(kg);
        if (kg + Lh < d.L) level(kg + Lh);
    }
}

// Eq. 4 update: dpi theta^(s) = dpi theta^n + dt_s (-div F_theta - delta(M theta)),
// V consecutive levels a thread (V > 1), or levels kg and kg + Lh.  th_n and
// th_out may be the caller's rows, moved level by level where those are not
// aligned.  Level 8, 60 levels, mixed: 420 -> 264 us a launch (233 at the DRAM
// rate); level 6, 30 levels (pairs) 17 -> 13; FP64, level 7, 276 -> 248.
template <class P, int V>
__global__ void __launch_bounds__(kBlock) k_theta_update(DevMesh m, DyPar d, LevelDiv Dh, const typename P::TA *__restrict__ Fth,
                               const typename P::TA *__restrict__ th, const double *__restrict__ Mv,
                               const double *__restrict__ th_n, double *__restrict__ th_out, double dts) {
    using TA = typename P::TA;
    const int Lh = (int)Dh.d;
    uint32_t n = blockIdx.x * blockDim.x + threadIdx.x;
    if (n >= (uint32_t)m.nC * (uint32_t)Lh) return;
    int i, kg;
    split_index(n, Dh, i, kg);
    // the cell's row once for the thread's levels
    int eidx[GRIST_MAXE];
    TA cw[GRIST_MAXE];
    load_row6(m.eoc8, i, eidx);
    load_row6(Coef<TA>::cdiv8(m), i, cw);
    if constexpr (V > 1) {
        const int k = kg * V;
        const size_t x = (size_t)i * d.ld + k, y = (size_t)i * d.ldi + k;
        TA div[V], a[V], tk[V], fl[V + 1];
        double o[V];
#pragma unroll
        for (int t = 0; t < V; t++) div[t] = 0;
#pragma unroll
        for (int j = 0; j < GRIST_MAXE; j++) {
            ldgv<V>(Fth + (size_t)eidx[j] * d.ld + k, a);
#pragma unroll
            for (int t = 0; t < V; t++) div[t] += cw[j] * a[t];
        }
        const bool whole = k + V <= d.L;
        ldgv<V>(th + x, tk);
        if (whole) {
            ldgv<V>(th_n + x, o);
        } else {
#pragma unroll
            for (int t = 0; t < V; t++) o[t] = k + t < d.L ? ldg(th_n + x + t) : 0.0;
        }
        const TA above = k > 0 ? ldg(th + x - 1) : (TA)0, below = k + V < d.L ? ldg(th + x + V) : (TA)0;
#pragma unroll
        for (int t = 0; t <= V; t++) {
            const TA q0 = t > 0 ? tk[t > 0 ? t - 1 : 0] : above, q1 = t < V ? tk[t < V ? t : 0] : below;
            fl[t] = (k + t > 0 && k + t < d.L) ? cv<TA>(ldg(Mv + y + t)) * ((TA)0.5 * (q0 + q1)) : (TA)0;
        }
#pragma unroll
        for (int t = 0; t < V; t++) {
            const TA tend = -div[t] - (fl[t + 1] - fl[t]);
            o[t] = o[t] + dts * cv<double>(tend);
        }
        if (whole) {
            stgv<V>(th_out + x, o);
        } else {
#pragma unroll
            for (int t = 0; t < V; t++)
                if (k + t < d.L) th_out[x + t] = o[t];
        }
    } else {
#pragma unroll
        for (int u = 0; u < 2; u++) {
            const int k = kg + u * Lh;
            if (k >= d.L) break;
            TA div = 0;
#pragma unroll
            for (int j = 0; j < GRIST_MAXE; j++) div += cw[j] * ldg(Fth + (size_t)eidx[j] * d.ld + k);
            const size_t x = (size_t)i * d.ld + k;
            const TA tk = th[x];
            TA top = 0, bot = 0;
            if (k > 0) top = cv<TA>(Mv[(size_t)i * d.ldi + k]) * ((TA)0.5 * (th[x - 1] + tk));
            if (k < d.L - 1) bot = cv<TA>(Mv[(size_t)i * d.ldi + k + 1]) * ((TA)0.5 * (tk + th[x + 1]));
            const TA tend = -div - (bot - top);
            th_out[x] = th_n[x] + dts * cv<double>(tend);
        }
    }
}

// The table of the hydrostatic equation of state (exner_entry, series.cuh):
// 256 bins x L entries of 16 bytes, of which a run touches the bins its surface
// pressures span (a few tens of kB).
constexpr int kExnerBins = 256;
struct Exner {
    const double2 *tab;
    int base;   // (high word of dps) >> 13 of bin 0
};

__global__ void k_exner_table(DyPar d, int base, double2 *__restrict__ tab) {
    const int n = blockIdx.x * blockDim.x + threadIdx.x;
    if (n >= kExnerBins * d.L) return;
    const int bin = n / d.L, k = n - bin * d.L;
    tab[n] = exner_entry(d.pi_top, d.Bm[k], d.Bml[k], exner_centre(base, bin), d.p0, d.rd, d.kappa);
}

// Eq. 8 (hydrostatic diagnostics), one warp per column: mid-layer pressure,
// alpha = Rd theta (p/p0)^kappa / p, geopotential integrated upward from
// phi_s by a suffix scan, layer geopotential = mean of its interfaces.
// Bound by the FP64 pipe: 29 instructions a cell-level with the table
// above (SHORT, see short_forms) against about 130 with pow(); level-6 mesh,
// 30 levels: 323 -> 73 us a launch, plus 11 us a step for the table.
// A warp takes two columns, so that the correctly rounded 1/dps runs one column
// per lane.  Level 6, 30 levels, us a step by columns, 1, 2, 4: FP64 1833, 1807,
// 1805; mixed 1551, 1518, 1557.  With pow(), p/p0 is the product with 1/p0
// corrected by its remainder (the correctly rounded quotient: rp0 is correctly
// rounded and p0's significand not all ones, which the host checks) and the
// pressure below is the next lane's above: the bits of the division.
constexpr int kDiagCols = 2;
template <bool EMU, bool DF, bool SHORT>
__global__ void __launch_bounds__(kBlock) k_hydro_diag(DevMesh m, DyPar d, Exner ex, Binom bk, const double *__restrict__ ps,
                             const double *__restrict__ th, double *__restrict__ p, double *__restrict__ al,
                             double *__restrict__ phl) {
    constexpr int C = kDiagCols;
    const int i0 = (int)((blockIdx.x * blockDim.x + threadIdx.x) >> 5) * C;
    const int lane = threadIdx.x & 31;
    if (i0 >= m.nC) return;
    double dps_l = 0.0, rdps_l = 0.0;
    if (i0 + lane < m.nC && lane < C) {
        dps_l = ps[i0 + lane] - d.pi_top;
        rdps_l = rcp(dps_l);
    }
    const int nch = (d.L + 31) >> 5, ncol = min(C, m.nC - i0);
#pragma unroll 1
    for (int c = 0; c < ncol; c++) {
        const int i = i0 + c;
        const double dps = __shfl_sync(0xffffffffu, dps_l, c), rdps = __shfl_sync(0xffffffffu, rdps_l, c);
        const int bin = SHORT ? (__double2hiint(dps) >> 13) - ex.base : -1;
        const bool tabled = bin >= 0 && bin < kExnerBins;   // the same for the whole warp
        const double off = SHORT ? dps - exner_centre(ex.base, bin) : 0.0;
        const double2 *row = ex.tab + (size_t)(tabled ? bin : 0) * d.L;
        double carry = ldg(d.phis + i);
        for (int ch = nch - 1; ch >= 0; ch--) {
            const int k = ch * 32 + lane;
            double contrib = 0.0, a = 0.0, pk = 0.0;
            if (tabled) {
                if (k < d.L) {
                    const double2 r = ldg(row + k);
                    pk = fma(ldg(d.Bm + k), dps, fma(ldg(d.Bml + k), dps, d.pi_top));
                    contrib = th[(size_t)i * d.ld + k] * exner_at(r, off, bk);   // alpha dpi
                    a = contrib * (ldg(d.rdB + k) * rdps);
                }
            } else {
                const double pt = d.pi_top + ldg(d.B + min(k, d.L)) * dps;
                double pb = __shfl_down_sync(0xffffffffu, pt, 1);
                if (lane == 31 && k < d.L) pb = d.pi_top + ldg(d.B + k + 1) * dps;
                if (k < d.L) {
                    const double dp = sub_near(pb, pt);
                    pk = 0.5 * (pt + pb);
                    double q;
                    if (d.rp0 != 0.0) {
                        q = pk * d.rp0;
                        q = fma(fma(-q, d.p0, pk), d.rp0, q);
                    } else {
                        q = pk / d.p0;
                    }
                    a = d.rd * (th[(size_t)i * d.ld + k] * ldg(d.rdB + k) * rdps) * pow(q, d.kappa) / pk;
                    contrib = a * dp;
                }
            }
            // inclusive suffix sum within the chunk
            double v = contrib;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                double t = __shfl_down_sync(0xffffffffu, v, o);
                if (lane + o < 32) v += t;
            }
            if (k < d.L) {
                const size_t x = (size_t)i * d.ld + k;
                p[x] = emu<EMU>(pk, d.emu, GRIST_ROW_EOS);
                al[x] = emu<EMU>(a, d.emu, GRIST_ROW_EOS);
                const double ph = SHORT ? carry + fma(-0.5, contrib, v) : carry + (v - contrib) + 0.5 * contrib;
                phl[x] = DF ? pack_split(ph) : emu<EMU>(ph, d.emu, GRIST_ROW_EOS);
            }
            carry += __shfl_sync(0xffffffffu, v, 0);
        }
    }
}

// Column reciprocal of the kite-remapped vertex layer mass:
// 1 / sum_i kite(i,v)/A_v (ps_i - pi_top); the layer value is dB_k times it.
template <bool EMU>
__global__ void k_vertex_mass(DevMesh m, DyPar d, const double *__restrict__ ps_s, double *__restrict__ rdpv) {
    const int v = blockIdx.x * blockDim.x + threadIdx.x;
    if (v >= m.nV) return;
    double s = 0.0;
#pragma unroll
    for (int j = 0; j < 3; j++) s += ldg(m.ckite + v * 3 + j) * (ldg(ps_s + ldg(m.cov + v * 3 + j)) - d.pi_top);
    rdpv[v] = emu<EMU>(rcp(s), d.emu, GRIST_ROW_DPI_PV);
}

// Vertex PV, Sec. 2.3: zeta_p = (zeta + f) / dpi_v, the relative vorticity
// from the circulation of u (advective type), dpi_v the kite-weighted remap
// of the FP64 layer mass (dpi must be double for zeta_p).  In a binary32
// advective type the FP64 factor 1/dpi_v = (1/dB_k)(1/dpi_col) is formed
// first and rounded once, then the rest is binary32 arithmetic (Sec. 2.2
// (ii): no mixed-kind expression): one FP64 product per vertex-level.
template <class P>
__global__ void k_vort(DevMesh m, DyPar d, LevelDiv Dh, const typename P::TU *__restrict__ u,
                       const double *__restrict__ rdpv, typename P::TA *__restrict__ qv) {
    using TA = typename P::TA;
    const int Lh = (int)Dh.d;
    uint32_t n = blockIdx.x * blockDim.x + threadIdx.x;
    if (n >= (uint32_t)m.nV * (uint32_t)Lh) return;
    int v, kg;
    split_index(n, Dh, v, kg);
    // the vertex's edges and weights once for its two levels kg and kg + Lh
    int ev[3];
    TA cc[3];
#pragma unroll
    for (int j = 0; j < 3; j++) {
        ev[j] = ldg(m.eov + v * 3 + j);
        cc[j] = ldg(Coef<TA>::ccurl(m) + v * 3 + j);
    }
    const double rv = ldg(rdpv + v);
#pragma unroll
    for (int w = 0; w < 2; w++) {
        const int k = kg + w * Lh;
        if (k >= d.L) break;
        TA z = 0;
#pragma unroll
        for (int j = 0; j < 3; j++) z += cc[j] * cv<TA>(ldg(u + (size_t)ev[j] * d.ld + k));
        if constexpr (sizeof(TA) == 4) {
            qv[(size_t)v * d.ld + k] = (z + ldg(m.fv_f + v)) * d2f(ldg(d.rdB + k) * rv);
        } else {
            qv[(size_t)v * d.ld + k] = emu<P::EMU>(cv<TA>((cv<double>(z) + ldg(m.fv + v)) * (ldg(d.rdB + k) * rv)),
                                                   d.emu, GRIST_ROW_PV_FLUX);
        }
    }
}

__device__ __forceinline__ double f2d_normal(float f) {   // a normal number or zero
    const uint32_t u = __float_as_uint(f), a = u & 0x7fffffffu;
    const uint32_t hi = a < 0x00800000u ? 0u : (a >> 3) + 0x38000000u;
    return __hiloint2double((int)(hi | (u & 0x80000000u)), (int)(a << 29));
}

// Cell kinetic energy, stored doubled: 2K = sum (dc dv / 2A) u^2 (FP64:
// boxed term of Eq. 5), V consecutive levels a thread.  Bound by the FP64 pipe
// (89 %): with a binary32 wind the product of the weight and u, half of the
// FP64 instructions, is formed in integers bit for bit (MulF32; the weight is
// unpacked once for the V levels).  Level 8, 60 levels, mixed: 846 -> 534 us a
// launch.
template <class P, int V>
__global__ void __launch_bounds__(kBlock) k_ke(DevMesh m, DyPar d, LevelDiv Dg, const typename P::TU *__restrict__ u,
                                               double *__restrict__ K) {
    const uint32_t n = blockIdx.x * blockDim.x + threadIdx.x;
    if (n >= (uint32_t)m.nC * Dg.d) return;
    int i, kg;
    split_index(n, Dg, i, kg);
    const int k = kg * V;
    int e[GRIST_MAXE];
    load_row6(m.eoc8, i, e);
    double s[V];
    bool ok[V];
#pragma unroll
    for (int t = 0; t < V; t++) {
        s[t] = 0.0;
        ok[t] = true;
    }
#pragma unroll
    for (int j = 0; j < GRIST_MAXE; j++) {
        const double w = ldg(m.kec2 + i * 6 + j);
        typename P::TU ue[V];
        const typename P::TU *uj = u + (size_t)e[j] * d.ld + k;
        if (V == 1 || k + V <= d.L) {
            ldgv<V>(uj, ue);
        } else {
#pragma unroll
            for (int t = 0; t < V; t++) ue[t] = k + t < d.L ? ldg(uj + t) : (typename P::TU)0;
        }
        if constexpr (sizeof(typename P::TU) == 4) {
            const MulF32 wm(w);
            if ((__double_as_longlong(w) << 1) == 0) continue;   // padding of a pentagon
#pragma unroll
            for (int t = 0; t < V; t++) s[t] = fma(wm.times(ue[t], ok[t]), f2d_normal(ue[t]), s[t]);
        } else {
#pragma unroll
            for (int t = 0; t < V; t++) s[t] += w * ue[t] * ue[t];
        }
    }
#pragma unroll
    for (int t = 0; t < V; t++) {
        if (!ok[t]) {   // a subnormal or non-finite wind
            s[t] = 0.0;
            for (int j = 0; j < GRIST_MAXE; j++) {
                const double ue = cv<double>(u[(size_t)e[j] * d.ld + k + t]);
                s[t] += ldg(m.kec2 + i * 6 + j) * ue * ue;
            }
        }
        s[t] = P::DF ? pack_split(s[t]) : emu<P::EMU>(s[t], d.emu, GRIST_ROW_KE_GRAD);
    }
    stgv<V>(K + (size_t)i * d.ld + k, s);
}

// Twice the PV at an edge from the sum of its vertices' (the mean is the value
// that the precision search rounds).
template <class P> __device__ __forceinline__ typename P::TA twice_pv(typename P::TA sum, const DyPar &d) {
    using TA = typename P::TA;
    if constexpr (P::EMU) return (TA)2 * emu<true>((TA)0.5 * sum, d.emu, GRIST_ROW_PV_FLUX);
    return sum;
}

// What the momentum equation needs of the PV at edges, q_e the mean of the
// edge's two vertices: q_e itself, so that a neighbour is one load instead of two
// and an index; in the FP64 policy 2 F q_e, with which the PV flux
// sum_e' w F' (q_e + q_e')/2 is (q_e sum w F' + sum w F' q_e')/2, two FP64
// instructions a neighbour instead of six (short_forms).  V consecutive levels
// a thread, 16 bytes: the vertex rows are gathers, and with single levels the
// pass took 492 us, with vectors 170 (level 8, 60 levels, mixed).
template <class P, int V>
__global__ void __launch_bounds__(kBlock) k_pv_edge(DevMesh m, DyPar d, LevelDiv Dg, const typename P::TM *__restrict__ F,
                                                    const typename P::TA *__restrict__ qv, typename P::TA *__restrict__ G) {
    using TA = typename P::TA;
    const uint32_t n = blockIdx.x * blockDim.x + threadIdx.x;
    if (n >= (uint32_t)m.nE * Dg.d) return;
    int e, kg;
    split_index(n, Dg, e, kg);
    const int2 v = ldg(m.voe + e);
    const size_t x = (size_t)e * d.ld + kg * V;
    TA a[V], b[V];
    ldgv<V>(qv + (size_t)v.x * d.ld + kg * V, a);
    ldgv<V>(qv + (size_t)v.y * d.ld + kg * V, b);
    if constexpr (short_forms<P>()) {
        TA f[V];
        ldgv<V>(F + x, f);
#pragma unroll
        for (int t = 0; t < V; t++) a[t] = f[t] * twice_pv<P>(a[t] + b[t], d);
    } else {
#pragma unroll
        for (int t = 0; t < V; t++) a[t] = (TA)0.5 * (a[t] + b[t]);
    }
    stgv<V>(G + x, a);
}

// Eq. 5 momentum tendency and stage update:
//   PV flux (1/dc) sum w dv' F' (q_e + q_e')/2          [advective type]
//   - dK/dn - eta-dot du/deta                              [FP64, boxed]
//   - alpha_e dp/dn - (dp/dpi)_e dphi/dn                   [FP64]
// with the tendency rounded to the wind's type (Sec. 2.3: boxed terms are
// computed in double, their tendency saved in single).  The edge layer mass
// in the vertical advection is dB_k (ps1 + ps2 - 2 pi_top)/2, entered as
// the product of the per-level and per-edge reciprocals.
// Bound by the FP64 pipe: the differences of p, phi and K between the edge's
// cells and of u between levels are taken off it without changing a bit
// (sub_near, wind_diff), 16 -> 11 FP64 instructions an edge-level in the mixed
// policies; then the loads' latency is what is left, so every load is issued
// before the first use, none behind a branch (2897 -> 2580 us below), with
// six blocks of 256 an SM (4: 3079, 5: 2606, 7: 2784; GRIST_MIX_DF, without
// FP64, eight: 110 -> 97 at level 6, 41 levels).  Level 8, 60 levels, us a launch
// with k_pv_edge's: mixed 3457 -> 2750; FP64, level 7, 3886 -> 1990.  Two or
// four levels a thread (shared indices and M sums) were slower: 2752 and 3370.
template <class P, bool NH>
__global__ void __launch_bounds__(kBlock, P::DF ? 8 : 6) k_momentum(DevMesh m, DyPar d, LevelDiv Dv, const typename P::TU *__restrict__ u_s,
                           const typename P::TU *u_n, typename P::TU *u_out, const typename P::TM *__restrict__ F,
                           const typename P::TA *__restrict__ qv, const typename P::TA *__restrict__ G,
                           const double *__restrict__ K,
                           const double *__restrict__ Mv, const double *__restrict__ rsum_e,
                           const double *__restrict__ p, const double *__restrict__ al,
                           const double *__restrict__ phl, const double *__restrict__ dpp, double dts,
                           uint32_t *status) {
    using TA = typename P::TA;
    using TU = typename P::TU;
    uint32_t n = blockIdx.x * blockDim.x + threadIdx.x;
    if (n >= (uint32_t)m.nE * (uint32_t)d.L) return;
    int e, k;
    split_index(n, Dv, e, k);
    const size_t x = (size_t)e * d.ld + k;
    const int2 c = ldg(m.coe + e);
    TA pv = 0;
    if constexpr (short_forms<P>()) {
        const int2 ve = ldg(m.voe + e);
        const TA q2 = twice_pv<P>(ldg(qv + (size_t)ve.x * d.ld + k) + ldg(qv + (size_t)ve.y * d.ld + k), d);
        TA s = 0;
#pragma unroll
        for (int j = 0; j < GRIST_MAXEOE; j++) {
            const size_t y = (size_t)ldg(m.eoe + e * 10 + j) * d.ld + k;
            const TA w = ldg(Coef<TA>::wpv(m) + e * 10 + j);
            s += w * ldg(F + y);
            pv += w * ldg(G + y);
        }
        pv = fma(q2, s, pv);   // 2 q_e sum w F' + sum w F' 2 q_e': four times the flux
    } else {
        const TA qee = ldg(G + x);
#pragma unroll
        for (int j = 0; j < GRIST_MAXEOE; j++) {
            const size_t y = (size_t)ldg(m.eoe + e * 10 + j) * d.ld + k;
            pv += ldg(Coef<TA>::wpv(m) + e * 10 + j) * cv<TA>(ldg(F + y)) * ((TA)0.5 * (qee + ldg(G + y)));
        }
    }
    const size_t a1 = (size_t)c.x * d.ld + k, a2 = (size_t)c.y * d.ld + k;
    if (P::DF) {
        // GRIST_MIX_DF: the slow tendency in binary32; the differences of the
        // double fields p, layer phi and K from their double-float splits
        // (p split here, phi and K stored split), the factors that are only
        // multiplied truncated to binary32, every other operation in binary32
        // - no FP64 instruction
        const float uk = (float)ldg(u_s + x);
        float va32 = 0.f;
        if (k < d.L - 1)
            va32 = (d2f_trunc(ldg(Mv + (size_t)c.x * d.ldi + k + 1)) +
                    d2f_trunc(ldg(Mv + (size_t)c.y * d.ldi + k + 1))) *
                   ((float)ldg(u_s + x + 1) - uk);
        if (k > 0)
            va32 = fmaf(d2f_trunc(ldg(Mv + (size_t)c.x * d.ldi + k)) + d2f_trunc(ldg(Mv + (size_t)c.y * d.ldi + k)),
                        uk - (float)ldg(u_s + x - 1), va32);
        va32 *= d2f_trunc(ldg(d.rdB + k)) * d2f_trunc(ldg(rsum_e + e));
        float p1h, p1l, p2h, p2l;
        split_df(ldg(p + a1), p1h, p1l);
        split_df(ldg(p + a2), p2h, p2l);
        const float2 f1 = ldg(reinterpret_cast<const float2 *>(phl) + a1);
        const float2 f2 = ldg(reinterpret_cast<const float2 *>(phl) + a2);
        const float2 k1 = ldg(reinterpret_cast<const float2 *>(K) + a1);
        const float2 k2 = ldg(reinterpret_cast<const float2 *>(K) + a2);
        const float de = NH ? d2f_trunc(ldg(dpp + a1)) + d2f_trunc(ldg(dpp + a2)) : 2.f;
        const float grad = fmaf(d2f_trunc(ldg(al + a1)) + d2f_trunc(ldg(al + a2)), diff_df(p2h, p2l, p1h, p1l),
                                fmaf(de, diff_df(f2.x, f2.y, f1.x, f1.y), diff_df(k2.x, k2.y, k1.x, k1.y)));
        const float tend = (float)pv + fmaf(d2f_trunc(ldg(m.hrdc + e)), grad, -va32);
        const float v = (float)u_n[x] + d2f(dts) * tend;
        if (!isfinite(v)) atomicOr(status, GRIST_FLAG_NONFINITE);
        u_out[x] = (TU)v;
        return;
    }
    // every load before the first use, none behind a branch
    const bool low = k < d.L - 1, high = k > 0;
    const TU uk = ldg(u_s + x), ub = ldg(u_s + x + (low ? 1 : 0)), ut = ldg(u_s + x - (high ? 1 : 0)), un = u_n[x];
    const double *M1 = Mv + (size_t)c.x * d.ldi + k, *M2 = Mv + (size_t)c.y * d.ldi + k;
    const double mb1 = ldg(M1 + 1), mb2 = ldg(M2 + 1), mt1 = ldg(M1), mt2 = ldg(M2);
    const double p1 = ldg(p + a1), p2 = ldg(p + a2), f1 = ldg(phl + a1), f2 = ldg(phl + a2), k1 = ldg(K + a1),
                 k2 = ldg(K + a2), al1 = ldg(al + a1), al2 = ldg(al + a2);
    const double d1 = NH ? ldg(dpp + a1) : 1.0, d2 = NH ? ldg(dpp + a2) : 1.0;
    double va = 0.0;
    if (low) va = (mb1 + mb2) * wind_diff(ub, uk);
    if (high) va = fma(mt1 + mt2, wind_diff(uk, ut), va);
    // [M sums](du) / (2 dpi_e) with dpi_e = dB (sum)/2, M_e = (M1 + M2)/2;
    // rsum_e holds 1/(2 sum)
    va *= ldg(d.rdB + k) * ldg(rsum_e + e);
    va = emu<P::EMU>(va, d.emu, GRIST_ROW_VADV_U);
    // dK/dn + alpha_e dp/dn + (dp/dpi)_e dphi/dn with the two means folded
    // into -1/(2 dc) (hrdc) and K stored doubled
    double grad;
    if (!P::EMU || !(d.emu & GRIST_ROW_PGF)) {
        const double de = NH ? d1 + d2 : 2.0;
        grad = fma(al1 + al2, sub_near(p2, p1), fma(de, sub_near(f2, f1), sub_near(k2, k1)));
    } else {
        // pressure gradient and gravity from binary32 inputs, summed and
        // rounded to binary32 (precision search)
        const uint32_t r = GRIST_ROW_PGF;
        const double de = NH ? emu<P::EMU>(d1, d.emu, r) + emu<P::EMU>(d2, d.emu, r) : 2.0;
        const double pgf = emu<P::EMU>(fma(emu<P::EMU>(al1, d.emu, r) + emu<P::EMU>(al2, d.emu, r),
                                           emu<P::EMU>(p2, d.emu, r) - emu<P::EMU>(p1, d.emu, r),
                                           de * (emu<P::EMU>(f2, d.emu, r) - emu<P::EMU>(f1, d.emu, r))),
                                       d.emu, r);
        grad = pgf + (k2 - k1);
    }
    const double slow = fma(ldg(m.hrdc + e), grad, -va);
    const TA tend = P::EMU             ? emu<P::EMU>((TA)0.25 * pv, d.emu, GRIST_ROW_PV_FLUX) + cv<TA>(slow)
                    : short_forms<P>() ? fma((TA)0.25, pv, cv<TA>(slow))
                                       : pv + cv<TA>(slow);
    const TU v = emu<P::EMU>(cv<TU>(cv<TA>(un) + cv<TA>(dts) * tend), d.emu, GRIST_ROW_WIND);
    if (!isfinite(v)) atomicOr(status, GRIST_FLAG_NONFINITE);
    u_out[x] = v;
}

// ---------------------------------------------------------------------------
// Non-hydrostatic pieces (Eqs. 6, 7, 9)

// Eq. 9 at time level n: p = p0 (Rd dpi_theta / (p0 dphi))^gamma, as
// p0 exp(gamma log(.)).
template <bool EMU>
__global__ void k_eos(DevMesh m, DyPar d, LevelDiv Dv, const double *__restrict__ th, const double *__restrict__ phi,
                      double *__restrict__ p) {
    uint32_t n = blockIdx.x * blockDim.x + threadIdx.x;
    if (n >= (uint32_t)m.nC * (uint32_t)d.L) return;
    int i, k;
    split_index(n, Dv, i, k);
    const double dphi = phi[(size_t)i * d.ldi + k] - phi[(size_t)i * d.ldi + k + 1];
    p[(size_t)i * d.ld + k] =
        emu<EMU>(d.p0 * exp(d.gamma * log(d.rd * th[(size_t)i * d.ld + k] / (d.p0 * dphi))), d.emu, GRIST_ROW_EOS);
}

// A binary32 advective type takes the differences of the FP64 fields from
// their truncating double-float splits (split_trunc; accurate to about 2^-24
// of the difference before its binary32 rounding) instead of FP64
// subtractions, so the binary32 advection issues no FP64 instruction.
template <typename TA> struct AdvVal;
template <> struct AdvVal<double> {
    double v;
    __device__ __forceinline__ explicit AdvVal(double x) : v(x) {}
};
template <> struct AdvVal<float> {
    float h, l;
    __device__ __forceinline__ explicit AdvVal(double x) { split_trunc(x, h, l); }
};
__device__ __forceinline__ double adv_diff(const AdvVal<double> &a, const AdvVal<double> &b) { return a.v - b.v; }
// of phi, whose neighbours are close: the same bits off the FP64 pipe
__device__ __forceinline__ double adv_diff_near(const AdvVal<double> &a, const AdvVal<double> &b) { return sub_near(a.v, b.v); }
__device__ __forceinline__ float adv_diff(const AdvVal<float> &a, const AdvVal<float> &b) {
    return diff_df(a.h, a.l, b.h, b.l);
}
__device__ __forceinline__ float adv_diff_near(const AdvVal<float> &a, const AdvVal<float> &b) { return adv_diff(a, b); }

// Explicit parts of Eqs. 6-7 at every interface: horizontal advection
// V.grad(x) = (1/A) sum s dv u^int (x_nb - x)/2 and vertical advection
// M (x_{j+1} - x_{j-1}) / (dpi_{j-1} + dpi_j) of w and phi from the stage
// input (advective type; the differences of the FP64 fields are formed to
// about 2^-24 of themselves before the rounding to that type), plus the (1 - beta) share of g (dp/dpi - 1) and g w at t^n.  The
// t^n forcing g (dp/dpi - 1) is formed in the first stage (FIRST) from the
// t^n pressure and kept for the later stages.  The binary32 form is bound by
// the integer pipe (the splits), the FP64 form by the FP64 pipe; the cell's row
// is read as vectors and the factors 1/2 of u and of the difference are taken
// out of the sums.  Level 8, 60 levels, mixed 1107 -> 1042 us a launch (five
// blocks of 256 an SM; 4: 1176, 6: 1218); FP64, level 7, 1184 -> 888.
template <class P, bool FIRST>
__global__ void __launch_bounds__(kBlock, 5) k_nh_explicit(DevMesh m, DyPar d, LevelDiv Dv, const typename P::TU *__restrict__ u_s,
                              const double *__restrict__ rdps_s, const double *__restrict__ Mv,
                              const double *__restrict__ w_s, const double *__restrict__ phi_s,
                              const double *__restrict__ w_n, const double *__restrict__ phi_n,
                              const double *__restrict__ p_n, double *__restrict__ fw_n, double *__restrict__ wst,
                              double *__restrict__ phst, double dts) {
    using TA = typename P::TA;
    uint32_t n = blockIdx.x * blockDim.x + threadIdx.x;
    const int Li = d.L + 1;
    if (n >= (uint32_t)m.nC * (uint32_t)Li) return;
    int i, j;
    split_index(n, Dv, i, j);
    const size_t xi = (size_t)i * d.ldi + j;
    if (j == d.L) {
        wst[xi] = 0.0;
        phst[xi] = ldg(d.phis + i);
        return;
    }
    const AdvVal<TA> wi(w_s[xi]), pi(phi_s[xi]);
    // sums of cdiv (u_{j-1} + u_j) dx: four times the advection (exact scalings
    // of its terms, taken out of the loop)
    TA hw = 0, hp = 0;
    int e[GRIST_MAXE], nb[GRIST_MAXE];
    TA cw[GRIST_MAXE];
    load_row6(m.eoc8, i, e);
    load_row6(m.coc8, i, nb);
    load_row6(Coef<TA>::cdiv8(m), i, cw);
#pragma unroll
    for (int s = 0; s < GRIST_MAXE; s++) {
        const size_t ue = (size_t)e[s] * d.ld + j, y = (size_t)nb[s] * d.ldi + j;
        const TA ub = cv<TA>(ldg(u_s + ue)), ut = j == 0 ? ub : cv<TA>(ldg(u_s + ue - 1));
        const TA cu = cw[s] * (ut + ub);
        hw += cu * adv_diff(AdvVal<TA>(ldg(w_s + y)), wi);
        hp += cu * adv_diff_near(AdvVal<TA>(ldg(phi_s + y)), pi);
    }
    TA vw = 0, vp = 0;
    double fw = 0.0;
    if (j > 0) {
        const double rd2 = ldg(d.hrdBi + j) * ldg(rdps_s + i);   // 1/(dpi_{j-1} + dpi_j)
        const TA r = cv<TA>(Mv[(size_t)i * d.ldi + j] * rd2);
        vw = r * adv_diff(AdvVal<TA>(w_s[xi + 1]), AdvVal<TA>(w_s[xi - 1]));
        vp = r * adv_diff_near(AdvVal<TA>(phi_s[xi + 1]), AdvVal<TA>(phi_s[xi - 1]));
        if (FIRST) {
            // first stage: the stage input is t^n, so rdps_s is 1/(ps^n - pi_top)
            fw = d.g * fma(p_n[(size_t)i * d.ld + j] - p_n[(size_t)i * d.ld + j - 1], 2.0 * rd2, -1.0);
            fw_n[xi] = fw;
        } else {
            fw = fw_n[xi];
        }
    }
    const TA q = (TA)0.25;
    wst[xi] = w_n[xi] + dts * (cv<double>(emu<P::EMU>(-q * hw - vw, d.emu, GRIST_ROW_NH_ADV)) + d.obeta * fw);
    phst[xi] = phi_n[xi] + dts * (cv<double>(emu<P::EMU>(-q * hp - vp, d.emu, GRIST_ROW_NH_ADV)) + d.obetag * w_n[xi]);
}

// Staging of a [32 columns][kSolveKC levels] tile between global memory
// (rows of stride S, one row per column) and shared memory
// sm[level * 33 + column]: each step moves kSolveKC consecutive levels
// (32 bytes, one sector) of 32 / kSolveKC columns, so every global sector
// is used whole; the 33-wide rows keep the shared-memory side free of bank
// conflicts.  Four-level chunks keep a block's shared memory at 6.6 KB so
// that 20 one-warp blocks fit on an SM (level 8, 60 levels, us a launch by blocks
// the registers must allow: 16 3539, 18 3368, 20 3346, 22 3451, 24 3475; chunks of
// 2 or 8 levels 3983, 4177).
#ifndef GRIST_SOLVE_KC
#define GRIST_SOLVE_KC 4          // levels per staged chunk (1, 2, 4 or 8)
#endif
#ifndef GRIST_SOLVE_MIN_BLOCKS
#define GRIST_SOLVE_MIN_BLOCKS 20 // resident one-warp blocks per SM the registers must allow
#endif
constexpr int kSolveCols = 32;
constexpr int kSolveKC = GRIST_SOLVE_KC;
constexpr int kSolveColsPerStep = 32 / kSolveKC;
constexpr int kRow = 33;
constexpr int kStage = kSolveKC * kRow;
constexpr int kSolveMinBlocks = GRIST_SOLVE_MIN_BLOCKS;
static_assert(kSolveKC == 1 || kSolveKC == 2 || kSolveKC == 4 || kSolveKC == 8, "chunk of 1, 2, 4 or 8 levels");

__device__ __forceinline__ void stage_in(const double *X, size_t S, int col0, int ncol, int k0, int nk, double *sm) {
    const int lane = threadIdx.x & 31, kk = lane % kSolveKC;
#pragma unroll
    for (int it = 0; it < kSolveKC; it++) {
        const int col = it * kSolveColsPerStep + lane / kSolveKC;
        double v = 0.0;
        if (col < ncol && kk < nk) v = X[(size_t)(col0 + col) * S + k0 + kk];
        sm[kk * kRow + col] = v;
    }
}

__device__ __forceinline__ void stage_out(double *X, size_t S, int col0, int ncol, int k0, int nk, const double *sm) {
    const int lane = threadIdx.x & 31, kk = lane % kSolveKC;
#pragma unroll
    for (int it = 0; it < kSolveKC; it++) {
        const int col = it * kSolveColsPerStep + lane / kSolveKC;
        if (col < ncol && kk < nk) X[(size_t)(col0 + col) * S + k0 + kk] = sm[kk * kRow + col];
    }
}

// Implicit part of Eqs. 6-7 and Eq. 9, FP64; two kernels with the same
// arithmetic.  k_nh_solve: one thread per column, a block is one warp of 32
// consecutive columns; column data moves through shared memory in
// kSolveKC-level chunks (whole-sector global access).  k_nh_solve_block, below:
// a block of 8 warps takes 32 columns.
// Equation of state relative to the t^n state (1/th_r, phi_r, p_r):
//   p** = p_r ((th dphi_r) / (th_r dphi**))^gamma     (pow1p_near0; dphi_r
//   of t^n is formed once per step)
// linearised about phi**: p_k = p**_k - C_k (w_k - w_{k+1}),
// C_k = gamma p**_k beta dt g / dphi**_k; tridiagonal rows for interior
// interfaces j = 1..L-1 (w = 0 at top and ground),
//   -a_j C_{j-1} w_{j-1} + (1 + a_j (C_{j-1} + C_j)) w_j - a_j C_j w_{j+1}
//       = w**_j + a_j (p**_j - p**_{j-1}) - beta dt g,
// a_j = beta dt g / dpi_j at the interface; each row is divided by a_j
// (off-diagonals -C, no product per row) and the system solved by the
// Thomas algorithm; phi = phi** + beta dt g w; the full EOS then gives
//   p = p** (dphi / dphi**)^(-gamma),  dphi = dphi** + beta dt g (w_k - w_{k+1});
// finally alpha = dphi/dpi, layer phi and dp/dpi averaged to layers
// (interface value 1 at top and bottom) for the momentum equation.  p may be
// p_r (the last stage writes the state in place): each block reads all
// reference values of its columns before writing them.
template <bool EMU, bool DF, bool SHORT>
__global__ void __launch_bounds__(32, kSolveMinBlocks) k_nh_solve(DevMesh m, DyPar d, const double *__restrict__ wst,
                                                 const double *__restrict__ phst, const double *__restrict__ th,
                                                 const double *__restrict__ rth_r, const double *__restrict__ dphi_r,
                                                 const double *p_r, const double *__restrict__ ps, double dts,
                                                 double *w_out, double *phi_out, double *p, double *__restrict__ al,
                                                 double *__restrict__ phl, double *__restrict__ dpp, Binom bg_pos,
                                                 Binom bg_neg) {
    __shared__ double sA[6 * kStage + kRow];
    const int lane = threadIdx.x;
    const int col0 = blockIdx.x * kSolveCols;
    const int ncol = min(kSolveCols, m.nC - col0);
    const int i = col0 + lane;
    const bool act = lane < ncol;
    const int L = d.L;
    const double bg = d.beta * dts * d.g;
    const double gbg = d.gamma * bg;
    const double dps = act ? ps[i] - d.pi_top : 1.0;
    const double rdps = rcp(dps);
    const double psg = dps * rcp(bg);   // 1/a_j = dBi_j psg
    const unsigned amask = __ballot_sync(0xffffffffu, act);
    double cp[kNHMax], dd[kNHMax], pst[kNHMax], rdf[kNHMax];
    double ftop = act ? phst[(size_t)i * d.ldi] : 0.0;
    const double phi_top0 = ftop;
    double pst_prev = 0.0, C_prev = 0.0;
    // forward sweep
    for (int k0 = 0; k0 < L; k0 += kSolveKC) {
        const int nk = min(kSolveKC, L - k0);
        __syncwarp();
        stage_in(phst, d.ldi, col0, ncol, k0 + 1, nk, sA + 0 * kStage);
        if (!SHORT) stage_in(dphi_r, d.ld, col0, ncol, k0, nk, sA + 1 * kStage);
        stage_in(th, d.ld, col0, ncol, k0, nk, sA + 2 * kStage);
        stage_in(rth_r, d.ld, col0, ncol, k0, nk, sA + 3 * kStage);
        stage_in(p_r, d.ld, col0, ncol, k0, nk, sA + 4 * kStage);
        stage_in(wst, d.ldi, col0, ncol, k0, nk, sA + 5 * kStage);
        __syncwarp();
        if (act) {
            for (int kk = 0; kk < nk; kk++) {
                const int j = k0 + kk;
                const int o = kk * kRow + lane;
                const double fbot = sA[0 * kStage + o];
                const double rdfj = rcp_nr(ftop - fbot);
                // x = th dphi_r / (th_r dphi**) - 1, the ratio's offset from 1
                const double tr = sA[2 * kStage + o] * sA[3 * kStage + o];
                const double x = SHORT ? fma(tr, rdfj, -1.0) : fma(tr, sA[1 * kStage + o] * rdfj, -1.0);
                const double pstj = DF ? scale_near1_df(sA[4 * kStage + o], x, d.gamma, bg_pos)
                                       : sA[4 * kStage + o] * pow1p_near0(x, d.gamma, bg_pos, amask);
                pst[j] = pstj;
                rdf[j] = rdfj;
                const double C = gbg * pstj * rdfj;
                if (j >= 1) {
                    // row j / a_j: -C_{j-1} w_{j-1} + (1/a_j + C_{j-1} + C_j) w_j - C_j w_{j+1}
                    //            = (w**_j - beta dt g)/a_j + p**_j - p**_{j-1}
                    // (no w_{j+1} term in the last row: w_L = 0)
                    const double sj = ldg(d.dBi + j) * psg;
                    const double b = sj + (C_prev + C);
                    const double rhs = fma(sA[5 * kStage + o] - bg, sj, pstj - pst_prev);
                    const double cq = (j == L - 1) ? 0.0 : C;
                    const int r = j - 1;
                    if (r == 0) {
                        const double rb = rcp_nr(b);
                        cp[0] = -cq * rb;
                        dd[0] = rhs * rb;
                    } else {
                        const double rden = rcp_nr(fma(C_prev, cp[r - 1], b));
                        cp[r] = -cq * rden;
                        dd[r] = fma(C_prev, dd[r - 1], rhs) * rden;
                    }
                }
                pst_prev = pstj;
                C_prev = C;
                ftop = fbot;
            }
        }
    }
    // back substitution, bottom to top, w written chunk by chunk
    // (interfaces 0..L; w = 0 at 0 and L)
    double wn = 0.0;
    for (int k0 = (L / kSolveKC) * kSolveKC; k0 >= 0; k0 -= kSolveKC) {
        const int nk = min(kSolveKC, L + 1 - k0);
        __syncwarp();
        for (int kk = nk - 1; kk >= 0; kk--) {
            const int jf = k0 + kk;
            double wv = 0.0;
            if (act && jf >= 1 && jf <= L - 1) {
                wn = fma(-cp[jf - 1], wn, dd[jf - 1]);
                wv = wn;
            }
            sA[kk * kRow + lane] = wv;
        }
        __syncwarp();
        stage_out(w_out, d.ldi, col0, ncol, k0, nk, sA);
    }
    // phi, EOS and momentum diagnostics, top to bottom
    if (act) phi_out[(size_t)i * d.ldi] = phi_top0;
    // halves of dp/dpi at the interfaces (1 at top and ground), so that the
    // layer mean is one addition
    double phi_top = phi_top0, htop = 0.5, pprev = 0.0;
    for (int k0 = 0; k0 < L; k0 += kSolveKC) {
        const int nk = min(kSolveKC, L - k0);
        __syncwarp();
        stage_in(phst, d.ldi, col0, ncol, k0 + 1, nk, sA + 0 * kStage);
        stage_in(w_out, d.ldi, col0, ncol, k0, nk, sA + 1 * kStage);   // w at interfaces k0..k0+nk-1
        if (lane < ncol) sA[6 * kStage + lane] = w_out[(size_t)i * d.ldi + k0 + nk];   // interface k0+nk
        __syncwarp();
        if (act) {
            for (int kk = 0; kk < nk; kk++) {
                const int k = k0 + kk;
                const int o = kk * kRow + lane;
                const double w_top = sA[1 * kStage + o];
                const double w_bot = (kk + 1 < nk) ? sA[1 * kStage + o + kRow] : sA[6 * kStage + lane];
                const double phi_bot = (k + 1 < L) ? fma(bg, w_bot, sA[o]) : ldg(d.phis + i);
                const double xk = bg * (w_top - w_bot) * rdf[k];
                const double pk = DF ? scale_near1_df(pst[k], xk, -d.gamma, bg_neg)
                                     : pst[k] * pow1p_near0(xk, -d.gamma, bg_neg, amask);
                double hcur = 0.5;
                if (k > 0) {
                    hcur = (pk - pprev) * (ldg(d.hrdBi + k) * rdps);
                    const double dv = htop + hcur;
                    if (kk > 0) sA[5 * kStage + o - kRow] = emu<EMU>(dv, d.emu, GRIST_ROW_EOS);   // layer k-1 of this chunk
                    else dpp[(size_t)i * d.ld + k - 1] = emu<EMU>(dv, d.emu, GRIST_ROW_EOS);        // of the previous chunk
                }
                sA[2 * kStage + o] = emu<EMU>(pk, d.emu, GRIST_ROW_EOS);
                const double dphi = phi_top - phi_bot;
                sA[3 * kStage + o] = emu<EMU>(dphi * (ldg(d.rdB + k) * rdps), d.emu, GRIST_ROW_EOS);
                const double phm = fma(0.5, dphi, phi_bot);   // layer mean (phi_top + phi_bot)/2
                sA[4 * kStage + o] = DF ? pack_split(phm) : emu<EMU>(phm, d.emu, GRIST_ROW_EOS);
                sA[1 * kStage + o] = phi_bot;   // w_top of this row is no longer needed
                htop = hcur;
                pprev = pk;
                phi_top = phi_bot;
            }
        }
        __syncwarp();
        stage_out(phi_out, d.ldi, col0, ncol, k0 + 1, nk, sA + 1 * kStage);
        stage_out(p, d.ld, col0, ncol, k0, nk, sA + 2 * kStage);
        stage_out(al, d.ld, col0, ncol, k0, nk, sA + 3 * kStage);
        stage_out(phl, d.ld, col0, ncol, k0, nk, sA + 4 * kStage);
        stage_out(dpp, d.ld, col0, ncol, k0, nk - 1, sA + 5 * kStage);
    }
    if (act) dpp[(size_t)i * d.ld + L - 1] = emu<EMU>(htop + 0.5, d.emu, GRIST_ROW_EOS);
}

// The same solve by blocks of 8 warps and 32 columns, the column arrays in
// shared memory ([level][33]).  Passes:
//   A   lanes = columns, a warp per level: p**, 1/dphi**, C;
//   B   Thomas sweep, one lane per column of one warp (on the scheduler
//       blockIdx mod 8 picks, so that resident blocks' sweeps spread);
//   C   lanes = columns, a warp per level: the new pressure;
//   D   the block's threads over the flat (column, level) index, so the
//       outputs are written as whole rows.
// The FP64 pipe bounds both kernels, 44 instructions a cell-level (SHORT: 43; the
// block form 46).
// One warp for 32 columns needs about 20 blocks an SM to keep the pipe busy
// (75 % then); with fewer columns than that the levels are the parallelism
// left (solve_by_blocks has the figures).
// SHORT: rth_r holds dphi_r / th_r.
constexpr int kSolveWarps = 8;

template <bool EMU, bool DF, bool SHORT>
__global__ void __launch_bounds__(kSolveWarps * 32) k_nh_solve_block(
    DevMesh m, DyPar d, LevelDiv Dv, const double *__restrict__ wst, const double *__restrict__ phst,
    const double *__restrict__ th, const double *__restrict__ rth_r, const double *__restrict__ dphi_r,
    const double *p_r, const double *__restrict__ ps, double dts, double *w_out, double *phi_out, double *p,
    double *__restrict__ al, double *__restrict__ phl, double *__restrict__ dpp, Binom bg_pos, Binom bg_neg) {
    extern __shared__ __align__(16) double sol[];
    const int L = d.L;
    double *sP = sol, *sD = sP + L * kRow, *sC = sD + L * kRow, *sW = sC + L * kRow;
    __shared__ double s_rdps[kSolveCols], s_psg[kSolveCols];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int col0 = blockIdx.x * kSolveCols;
    const int ncol = min(kSolveCols, m.nC - col0);
    const bool act = lane < ncol;
    const unsigned amask = __ballot_sync(0xffffffffu, act);
    const double bg = d.beta * dts * d.g;
    const double gbg = d.gamma * bg;
    if (warp == 0 && act) {
        const double dps = ps[col0 + lane] - d.pi_top;
        s_rdps[lane] = rcp(dps);
        s_psg[lane] = dps * rcp(bg);   // 1/a_j = dBi_j psg
    }
    // A
    if (act) {
        const size_t x0 = (size_t)(col0 + lane) * d.ld, y0 = (size_t)(col0 + lane) * d.ldi;
        for (int k = warp; k < L; k += kSolveWarps) {
            const double rdf = rcp_nr(phst[y0 + k] - phst[y0 + k + 1]);
            const double pr = p_r[x0 + k], tr = ldg(th + x0 + k) * ldg(rth_r + x0 + k);
            // th dphi_r / (th_r dphi**) - 1
            const double x = SHORT ? fma(tr, rdf, -1.0) : fma(tr, ldg(dphi_r + x0 + k) * rdf, -1.0);
            const double pst = DF ? scale_near1_df(pr, x, d.gamma, bg_pos)
                                  : pr * pow1p_near0(x, d.gamma, bg_pos, amask);
            const int o = k * kRow + lane;
            sP[o] = pst;
            sD[o] = rdf;
            sC[o] = gbg * pst * rdf;
            sW[o] = wst[y0 + k] - bg;
        }
    }
    __syncthreads();
    // B
    if (warp == (int)(blockIdx.x % kSolveWarps) && act) {
        const double psg = s_psg[lane];
        double Cp = sC[lane], pp = sP[lane], cp = 0.0, dd = 0.0;
        for (int j = 1; j < L; j++) {
            const int o = j * kRow + lane;
            const double C = sC[o], pj = sP[o];
            // row j / a_j, as in k_nh_solve
            const double sj = ldg(d.dBi + j) * psg;
            const double b = sj + (Cp + C);
            const double rhs = fma(sW[o], sj, pj - pp);
            const double rden = rcp_nr(fma(Cp, cp, b));
            cp = j == L - 1 ? -0.0 * rden : -C * rden;
            dd = fma(Cp, dd, rhs) * rden;
            sC[o] = cp;
            sW[o] = dd;
            Cp = C;
            pp = pj;
        }
        double wn = 0.0;
        for (int j = L - 1; j >= 1; j--) {
            const int o = j * kRow + lane;
            wn = fma(-sC[o], wn, sW[o]);
            sW[o] = wn;
        }
        sW[lane] = 0.0;
    }
    __syncthreads();
    // C
    if (act) {
        for (int k = warp; k < L; k += kSolveWarps) {
            const int o = k * kRow + lane;
            const double w_bot = k + 1 < L ? sW[o + kRow] : 0.0;
            const double xk = bg * (sW[o] - w_bot) * sD[o];
            sP[o] = DF ? scale_near1_df(sP[o], xk, -d.gamma, bg_neg)
                       : sP[o] * pow1p_near0(xk, -d.gamma, bg_neg, amask);
        }
    }
    __syncthreads();
    // D: a warp takes 31 items and the one after them (the interface below)
    const int items = ncol * L;
    for (int base = warp * 31; base < items; base += kSolveWarps * 31) {
        const int n = min(base + lane, items - 1);
        int c, k;
        split_index((uint32_t)n, Dv, c, k);
        const size_t x = (size_t)(col0 + c) * d.ld + k, y = (size_t)(col0 + c) * d.ldi + k;
        const int o = k * kRow + c;
        const double rdps = s_rdps[c], pk = sP[o], w = sW[o];
        const double phi_top = k > 0 ? fma(bg, w, phst[y]) : phst[y];
        double phi_bot = __shfl_down_sync(0xffffffffu, phi_top, 1);
        // halves of dp/dpi at the layer's interfaces (1 at top and ground)
        const double hc = k > 0 ? (pk - sP[o - kRow]) * (ldg(d.hrdBi + k) * rdps) : 0.5;
        double hb = __shfl_down_sync(0xffffffffu, hc, 1);
        if (k == L - 1) {
            hb = 0.5;
            phi_bot = ldg(d.phis + col0 + c);
        }
        if (lane < 31 && base + lane < items) {
            const double dphi = phi_top - phi_bot;
            w_out[y] = w;
            phi_out[y] = phi_top;
            if (k == L - 1) {
                w_out[y + 1] = 0.0;
                phi_out[y + 1] = phi_bot;
            }
            p[x] = emu<EMU>(pk, d.emu, GRIST_ROW_EOS);
            al[x] = emu<EMU>(dphi * (ldg(d.rdB + k) * rdps), d.emu, GRIST_ROW_EOS);
            const double phm = fma(0.5, dphi, phi_bot);   // layer mean (phi_top + phi_bot)/2
            phl[x] = DF ? pack_split(phm) : emu<EMU>(phm, d.emu, GRIST_ROW_EOS);
            dpp[x] = emu<EMU>(hc + hb, d.emu, GRIST_ROW_EOS);
        }
    }
}

// Which form, by columns and levels; both give the same bits
// (tests/test_gpu_solve_bits.py).  Mixed, us a launch, one warp / block:
//   levels            20         30         41         50         60         71
//   10,242 cells   57 /  35   91 /  49  128 /  65  156 /  95  184 /  91  216 / 138
//   40,962         93 / 100  142 / 138  201 / 185  237 / 279  274 / 260  342 / 373
//   163,842       326 / 317  518 / 458  754 / 620  878 / 864  938 / 975 1297 /1260
//   655,362                 1845 /1828                       3519 /3811
// 80 levels: 244 / 179, 364 / 455, 1246 / 1541; FP64 within 4 % of these.  So the
// block form while the one-warp form has less than a wave (20 resident blocks of
// 32 columns on 152 SMs) or columns are short, where three blocks' arrays fit an
// SM (70 levels; with fewer blocks an SM waits through every pass); above 70
// levels only for a few blocks per SM in all.  The line at 40 levels is on the safe
// side: at 163,842 cells the block form is the faster one up to 50.
inline bool solve_by_blocks(int nC, int L) {
    if (L > 70) return nC <= 152 * kSolveCols * 3;
    return nC < 152 * kSolveCols * kSolveMinBlocks || L <= 40;
}

template <bool EMU, bool DF, bool SHORT>
cudaError_t launch_solve(const DevMesh &m, const DyPar &d, LevelDiv Dv, const double *wst, const double *phst,
                         const double *th, const double *rth, const double *dphi, const double *p_r, const double *ps,
                         double dts, double *w_out, double *phi_out, double *p, double *al, double *phl, double *dpp,
                         const Binom &bp, const Binom &bn, bool blocks, cudaStream_t st) {
    const unsigned grid = grid_for(m.nC, kSolveCols);
    if (blocks) {
        const int bytes = 4 * d.L * kRow * 8;
        const cudaError_t e = cudaFuncSetAttribute(k_nh_solve_block<EMU, DF, SHORT>,
                                                   cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
        if (e != cudaSuccess) return e;
        k_nh_solve_block<EMU, DF, SHORT><<<grid, kSolveWarps * 32, bytes, st>>>(
            m, d, Dv, wst, phst, th, rth, dphi, p_r, ps, dts, w_out, phi_out, p, al, phl, dpp, bp, bn);
    } else {
        k_nh_solve<EMU, DF, SHORT><<<grid, kSolveCols, 0, st>>>(m, d, wst, phst, th, rth, dphi, p_r, ps, dts, w_out, phi_out, p,
                                                         al, phl, dpp, bp, bn);
    }
    return cudaSuccess;
}

// Relative vorticity at the vertices (diagnostic): zeta_v = sum_j ccurl u,
// ccurl = t(e,v) dc_e / A_v, in FP64; V consecutive levels a thread where rows
// are whole, aligned vectors.  A binary32 wind is converted in integers: the
// hardware conversions run on the FP64 pipe, which bounds the kernel.
// Level 7, 60 levels: binary32 wind 219 -> 107 us, binary64 124 -> 107 (62 at the
// DRAM rate).
template <typename TU, int V>
__global__ void __launch_bounds__(kBlock) k_diag_vort(DevMesh m, int ld, LevelDiv Dg, const TU *__restrict__ u,
                                                      double *__restrict__ vor) {
    const uint32_t n = blockIdx.x * blockDim.x + threadIdx.x;
    if (n >= (uint32_t)m.nV * Dg.d) return;
    int v, kg;
    split_index(n, Dg, v, kg);
    double z[V];
#pragma unroll
    for (int t = 0; t < V; t++) z[t] = 0.0;
#pragma unroll
    for (int j = 0; j < 3; j++) {
        const double c = ldg(m.ccurl + v * 3 + j);
        TU ue[V];
        ldgv<V>(u + (size_t)ldg(m.eov + v * 3 + j) * ld + kg * V, ue);
#pragma unroll
        for (int t = 0; t < V; t++) z[t] += c * cv<double>(ue[t]);
    }
    stgv<V>(vor + (size_t)v * ld + kg * V, z);
}

__global__ void k_add_scalar(double *x, double v) {
    if (threadIdx.x == 0 && blockIdx.x == 0) *x += v;
}

// Where the wind's diagnostics go in the NH core: beside the mass kernels from
// the start of the stage, or beside the column solve.  Small meshes leave SMs
// idle all along and gain from the early start (10,242 cells: 464 against 484
// us a step); on large ones every kernel fills the GPU and the solve, with a
// third of the warps and waiting for its chains, is what can take them
// (163,842 cells, FP64: 16953 against 17128; 655,362, mixed: 28667, 28775;
// 40,962 equal).
inline bool wind_beside_solve(int nC) { return nC > 100000; }

// One side stream of a dycore step: work on s after fork(k) follows what st has
// so far; join(k) makes st wait for all of s so far.  Every fork is joined
// before the step returns, also on an error, so that the caller's buffers are
// used on st's order only and a capture of st takes the side stream in and
// gives it back.  While kernels are timed one by one, or without the stream,
// s is st itself.
struct Side {
    cudaStream_t st, s;
    cudaEvent_t *ev;
    bool on, open = false;
    Side(grist_mesh_s *h, int which, cudaStream_t st_) : st(st_), s(st_), ev(nullptr), on(false) {
        if (!profiling(h)) on = side_stream(h, which, &s, &ev);
        if (!on) s = st;
    }
    ~Side() { if (open) join(); }
    void fork() {
        if (!on) return;
        cudaEventRecord(ev[0], st);
        cudaStreamWaitEvent(s, ev[0], 0);
        open = true;
    }
    void join() {
        if (!open) return;
        cudaEventRecord(ev[1], s);
        cudaStreamWaitEvent(st, ev[1], 0);
        open = false;
    }
};

template <class P, bool NH>
int dycore_step(grist_mesh_s *h, grist_dycore_state *S, const grist_dycore_params *prm, double dt, cudaStream_t st) {
    using TU = typename P::TU;
    using TA = typename P::TA;
    using TM = typename P::TM;
    const DevMesh &m = dev_mesh(h);
    const int L = prm->n_levels, ld = prm->ld, ldi = prm->ld_int;
    const size_t nCL = (size_t)m.nC * ld, nEL = (size_t)m.nE * ld, nVL = (size_t)m.nV * ld, nCI = (size_t)m.nC * ldi;

    // scratch layout
    auto al = [](size_t b) { return (b + 255) & ~size_t(255); };
    size_t off = 0;
    auto take = [&](size_t bytes) { size_t o = off; off += al(bytes); return o; };
    const size_t nvg = 7 * (size_t)L + 3 + ((size_t)L + 1) / 2;   // doubles, then L floats
    const size_t o_vg = take(sizeof(double) * nvg);
    const size_t o_uA = take(nEL * sizeof(TU)), o_uB = take(nEL * sizeof(TU));
    const size_t o_psA = take(m.nC * 8), o_psB = take(m.nC * 8), o_psN = take(m.nC * 8);
    const size_t o_rdps = take(m.nC * 8), o_rsum = take(m.nE * 8), o_rdpv = take(m.nV * 8),
                 o_fcol = take(m.nE * 8);
    const size_t o_thA = take(nCL * 8), o_thB = take(nCL * 8);
    const size_t o_F = take(nEL * sizeof(TM)), o_M = take(nCI * 8);
    const size_t o_theta = take(nCL * sizeof(TA)), o_Fth = take(nEL * sizeof(TA));
    const size_t o_p = take(nCL * 8), o_al = take(nCL * 8), o_phl = take(nCL * 8), o_dpp = take(nCL * 8);
    const size_t o_qv = take(nVL * sizeof(TA)), o_K = take(nCL * 8);
    // The edge PV takes the theta flux's array where it is formed after the theta
    // update: in the FP64 policy, which needs the mass flux for it anyway, and on
    // large meshes, where the array counts (level 9, 60 levels: 1.9 GB in
    // binary32).  By size alone, so that no choice of forms moves the scratch of a
    // recorded step.
    const bool pv_shares = short_forms<P>() || wind_beside_solve(m.nC);
    const size_t o_Gq = pv_shares ? o_Fth : take(nEL * sizeof(TA));
    size_t o_wA = 0, o_wB = 0, o_phA = 0, o_phB = 0, o_wst = 0, o_phst = 0, o_pn = 0, o_fw = 0, o_rth = 0, o_dph = 0;
    constexpr bool kTable = !NH && short_forms<P>();
    const size_t o_ex = take(kTable ? (size_t)kExnerBins * L * sizeof(double2) : 0);
    if (NH) {
        o_wA = take(nCI * 8); o_wB = take(nCI * 8); o_phA = take(nCI * 8); o_phB = take(nCI * 8);
        o_wst = take(nCI * 8); o_phst = take(nCI * 8); o_pn = take(nCL * 8); o_fw = take(nCI * 8);
        o_rth = take(nCL * 8);
        o_dph = take(short_forms<P>() ? 0 : nCL * 8);
    }
    char *s = (char *)scratch(h, 1, off);
    if (!s) return GRIST_ENOMEM;

    // vertical grid: B (L+1) | dB (L) | 1/dB (L) | 1/(dB[j-1]+dB[j]) (L+1) | (dB[j-1]+dB[j])/2 (L+1) |
    // (B[k]+B[k+1])/2 (L) | its rest (L) | dB in binary32 (L floats)
    std::vector<double> vg(nvg, 0.0);
    double *hB = vg.data(), *hdB = hB + L + 1, *hrdB = hdB + L, *hhrdBi = hrdB + L, *hdBi = hhrdBi + L + 1;
    for (int k = 0; k <= L; k++) hB[k] = prm->b_interface[k];
    for (int k = 0; k < L; k++) {
        hdB[k] = prm->b_interface[k + 1] - prm->b_interface[k];
        hrdB[k] = 1.0 / hdB[k];
    }
    for (int j = 1; j < L; j++) {
        hhrdBi[j] = 1.0 / (hdB[j - 1] + hdB[j]);
        hdBi[j] = 0.5 * (hdB[j - 1] + hdB[j]);
    }
    double *hBm = hdBi + L + 1;
    double *hBml = hBm + L;
    for (int k = 0; k < L; k++) {
        // the sum's rounding error by the larger summand (B increases)
        const double sum = hB[k] + hB[k + 1];
        hBm[k] = 0.5 * sum;
        hBml[k] = 0.5 * (hB[k] - (sum - hB[k + 1]));
    }
    float *hdBf = reinterpret_cast<float *>(hBml + L);
    for (int k = 0; k < L; k++) hdBf[k] = (float)hdB[k];
    double *dvg = (double *)(s + o_vg);
    if (vg_ptr(h) != dvg || vg_cache(h) != vg) {
        // ordered after this stream's earlier steps, which read the old table
        GRIST_CUDA_TRY(cudaMemcpyAsync(dvg, vg.data(), vg.size() * sizeof(double), cudaMemcpyHostToDevice, st));
        GRIST_CUDA_TRY(cudaStreamSynchronize(st));  // vg is a host temporary
        vg_cache(h) = vg;
        vg_ptr(h) = dvg;
    }

    DyPar d;
    d.L = L; d.ld = ld; d.ldi = ldi;
    d.pi_top = prm->pi_top; d.p0 = prm->p0; d.rd = prm->rd; d.cp = prm->cp; d.g = prm->g;
    {
        // p/p0 by the corrected product needs p0 and the quotient away from the
        // ends of the range, and a significand other than all ones
        int e2 = 0;
        const double f = std::isfinite(prm->p0) ? std::frexp(prm->p0, &e2) : 0.0;
        d.rp0 = std::isfinite(prm->p0) && std::abs(e2) < 200 && f != 1.0 - 0x1p-53 ? 1.0 / prm->p0 : 0.0;
    }
    d.beta = prm->offcentre_beta; d.obeta = 1.0 - d.beta; d.obetag = d.obeta * d.g; d.kappa = prm->rd / prm->cp; d.gamma = prm->cp / (prm->cp - prm->rd);
    d.B = dvg; d.dB = dvg + L + 1; d.rdB = dvg + 2 * L + 1; d.hrdBi = dvg + 3 * L + 1; d.dBi = dvg + 4 * L + 2;
    d.phis = prm->phi_surface;
    d.Bm = dvg + 5 * L + 3;
    d.Bml = dvg + 6 * L + 3;
    d.dBf = reinterpret_cast<const float *>(dvg + 7 * L + 3);
    d.emu = prm->emulate_fp32_rows;

    TU *uA = (TU *)(s + o_uA), *uB = (TU *)(s + o_uB);
    double *psA = (double *)(s + o_psA), *psB = (double *)(s + o_psB), *psN = (double *)(s + o_psN);
    double *rdps = (double *)(s + o_rdps), *rsum = (double *)(s + o_rsum), *rdpv = (double *)(s + o_rdpv),
           *fcol = (double *)(s + o_fcol);
    double *thA = (double *)(s + o_thA), *thB = (double *)(s + o_thB);
    TM *F = (TM *)(s + o_F);
    double *Mv = (double *)(s + o_M);
    TA *theta = (TA *)(s + o_theta), *Fth = (TA *)(s + o_Fth);
    double *p = (double *)(s + o_p), *alp = (double *)(s + o_al), *phl = (double *)(s + o_phl),
           *dpp = (double *)(s + o_dpp);
    TA *qv = (TA *)(s + o_qv), *Gq = (TA *)(s + o_Gq);
    double *K = (double *)(s + o_K);
    double *wA = (double *)(s + o_wA), *wB = (double *)(s + o_wB), *phA = (double *)(s + o_phA),
           *phB = (double *)(s + o_phB), *wst = (double *)(s + o_wst), *phst = (double *)(s + o_phst),
           *pn = (double *)(s + o_pn), *fwn = (double *)(s + o_fw), *rthn = (double *)(s + o_rth),
           *dphn = (double *)(s + o_dph);

    TU *u = (TU *)S->u;
    uint32_t *status = status_word(h);
    const LevelDiv DL = make_div((uint32_t)L), DI = make_div((uint32_t)(L + 1)), DH = make_div((uint32_t)(L + 1) / 2);
    const unsigned gC = grid_for((long long)m.nC * L, kBlock),
                   gV = grid_for((long long)m.nV * L, kBlock), gW = grid_for(((long long)m.nC + kDiagCols - 1) / kDiagCols * 32, kBlock),
                   gI = grid_for((long long)m.nC * (L + 1), kBlock),
                   gVx = grid_for(m.nV, kBlock), gEG = grid_for(((long long)m.nE + kMassGroup - 1) / kMassGroup * 32, kBlock),
                   gCG = grid_for(((long long)m.nC + kMassGroup - 1) / kMassGroup * 32, kBlock),
                   gVH = grid_for((long long)m.nV * DH.d, kBlock);
    // Vectors of levels where a row is whole, aligned vectors.  The last one may
    // reach past the levels into the row's padding: of the scratch arrays, which
    // have the caller's row length, it is read and written, of the caller's
    // arrays it is not.
    // Kinetic energy on 2 (binary32 wind: up to 4) levels
    constexpr int kKeV = sizeof(TU) == 4 ? 4 : 2;
    auto ke_fits = [&](int v) { return ld % v == 0 && (uintptr_t)u % (v * sizeof(TU)) == 0; };
    const int kev = kKeV == 4 && ke_fits(4) ? 4 : (ke_fits(2) ? 2 : 1);
    const LevelDiv DK = make_div((uint32_t)((L + kev - 1) / kev));
    const unsigned gK = grid_for((long long)m.nC * DK.d, kBlock);
    // edge PV on 16-byte vectors of levels, or 8-byte ones
    constexpr int kPvV = 16 / sizeof(TA), kPvH = sizeof(TA) == 4 ? 2 : 1;
    const int pvv = ld % kPvV == 0 ? kPvV : (ld % kPvH == 0 ? kPvH : 1);
    const LevelDiv DP = make_div((uint32_t)((L + pvv - 1) / pvv));
    // theta update on the same vectors, the flux on binary32 quads, or two levels
    // half a column apart
    const bool quad = pvv == 4;
    const int thv = ((uintptr_t)S->dpi_theta % 16) == 0 ? pvv : 1;
    const LevelDiv DT = quad ? DP : DH, DTU = thv > 1 ? DP : DH;
    const unsigned gEH = grid_for((long long)m.nE * DT.d, kBlock), gCT = grid_for((long long)m.nC * DTU.d, kBlock);
    const unsigned gE = grid_for((long long)m.nE * L, kBlock), gP = grid_for((long long)m.nE * DP.d, kBlock);
    const double dts[3] = {dt / 3.0, dt / 2.0, dt};
    const double ascale = S->accum_scale != 0.0 ? S->accum_scale : 1.0;

    GRIST_CUDA_TRY(cudaMemcpyAsync(psN, S->ps, m.nC * sizeof(double), cudaMemcpyDeviceToDevice, st));
    // t^n pressure: carried in the state when valid, else from the EOS
    const double *p_n = pn;
    if (NH) {
        if (S->p_nh && S->p_nh_valid) {
            p_n = S->p_nh;
        } else {
            double *dst = S->p_nh ? S->p_nh : pn;
            GRIST_LAUNCH(h, PN("k_eos"), st, k_eos<P::EMU><<<gC, kBlock, 0, st>>>(m, d, DL, S->dpi_theta, S->phi, dst));
            p_n = dst;
        }
    }
    const Binom bpos = binomial(d.gamma), bneg = binomial(-d.gamma), bkap = binomial(d.kappa - 1.0);
    Exner ex{(double2 *)(s + o_ex), 0};
    if (kTable) {
        // two octaves up to twice the power of two at or below p0 - pi_top;
        // bins that no column can fall in where the series' exponent would be
        // out of its range (kappa - 1 outside (-1, 0)).  Made in every step
        // (about 10 us): a step recorded in a graph then carries its own
        int e2 = 0;
        const double span = prm->p0 - prm->pi_top;
        if (std::isfinite(span)) std::frexp(span, &e2);   // |span| in [2^(e2-1), 2^e2)
        ex.base = d.kappa > 0.0 && d.kappa < 1.0 && e2 > -1000 ? (1023 + e2 - 2) << 7 : 1 << 20;
        GRIST_LAUNCH(h, PN("k_exner_table"), st, k_exner_table<<<grid_for((long long)kExnerBins * L, 32), 32, 0, st>>>(
            d, ex.base, (double2 *)(s + o_ex)));
    }

    auto edge_pv = [&](cudaStream_t sw) {
        GRIST_LAUNCH(h, PN("k_pv_edge"), sw, (pvv == kPvV   ? k_pv_edge<P, kPvV>
                                              : pvv == kPvH ? k_pv_edge<P, kPvH>
                                                            : k_pv_edge<P, 1>)<<<gP, kBlock, 0, sw>>>(m, d, DP, F, qv, Gq));
    };
    double *p_outs[3] = {p, p, (NH && S->p_nh) ? S->p_nh : p};

    const TU *u_in = u;
    const double *ps_in = psN, *th_in = S->dpi_theta, *w_in = S->w, *phi_in = S->phi;
    TU *u_outs[3] = {uA, uB, u};
    double *ps_outs[3] = {psA, psB, S->ps};
    double *th_outs[3] = {thA, thB, S->dpi_theta};
    double *w_outs[3] = {wA, wB, S->w};
    double *phi_outs[3] = {phA, phB, S->phi};
    // Two chains of a stage do not depend on each other until the column solve
    // or the momentum equation: mass -> theta (-> column), and the wind's
    // diagnostics (vertex PV, edge PV, kinetic energy) of the stage input; in
    // the NH core the advection of w and phi needs the mass kernels only.
    // They run on side streams of the handle, forked and joined by events.  us a
    // step in one chain / with them: level 5 coupled, 30 levels, recorded 506 /
    // 464; level 6 hydrostatic, 30 levels, mixed 1686 / 1589, FP64 1880 / 1802;
    // level 6 NH, 41 levels 1606 / 1446; level 7 FP64 NH 17277 / 16953; level 8
    // mixed NH 28962 / 28667.
    Side sw_(h, 0, st), sx_(h, 1, st);   // the wind's diagnostics, the advection
    const int place = dycore_tuning(h).wind_placement;
    const bool late = NH && (place == 2 || (place == 0 && wind_beside_solve(m.nC)));
    // the edge PV with the wind's chain; else on its stream once the theta
    // update is done, or (FP64 policy) on st after the join
    const bool pv_with_wind = !pv_shares || (late && !short_forms<P>());
    for (int s3 = 0; s3 < 3; s3++) {
        const double h3 = dts[s3];
        auto wind = [&](cudaStream_t sw) {
            GRIST_LAUNCH(h, PN("k_vertex_mass"), sw, k_vertex_mass<P::EMU><<<gVx, kBlock, 0, sw>>>(m, d, ps_in, rdpv));
            GRIST_LAUNCH(h, PN("k_vort"), sw, k_vort<P><<<gVH, kBlock, 0, sw>>>(m, d, DH, u_in, rdpv, qv));
            GRIST_LAUNCH(h, PN("k_ke"), sw, (kev == 4   ? k_ke<P, kKeV>
                                             : kev == 2 ? k_ke<P, 2>
                                                        : k_ke<P, 1>)<<<gK, kBlock, 0, sw>>>(m, d, DK, u_in, K));
            if (pv_with_wind) edge_pv(sw);
        };
        auto explicit_part = [&](cudaStream_t sw) {
            if (s3 == 0)
                GRIST_LAUNCH(h, PN("k_nh_explicit"), sw, k_nh_explicit<P, true><<<gI, kBlock, 0, sw>>>(
                    m, d, DI, u_in, rdps, Mv, w_in, phi_in, S->w, S->phi, p_n, fwn, wst, phst, h3));
            else
                GRIST_LAUNCH(h, PN("k_nh_explicit"), sw, k_nh_explicit<P, false><<<gI, kBlock, 0, sw>>>(
                    m, d, DI, u_in, rdps, Mv, w_in, phi_in, S->w, S->phi, p_n, fwn, wst, phst, h3));
        };
        if (!late || !NH) {
            sw_.fork();
            wind(sw_.s);
        }
        GRIST_LAUNCH(h, PN("k_mass_edge"), st, k_mass_edge<P><<<gEG, kBlock, 0, st>>>(
            m, d, ps_in, u_in, F, s3 == 2 ? S->mass_flux_accum : nullptr, ascale, rsum, fcol));
        GRIST_LAUNCH(h, PN("k_mass_col"), st, k_mass_col<P><<<gCG, kBlock, 0, st>>>(
            m, d, F, fcol, ps_in, psN, ps_outs[s3], th_in, theta, Mv, h3, s3 == 0 ? S->dpi_start : nullptr, rdps,
            (NH && s3 == 0) ? rthn : nullptr, dphn, S->phi, s3 == 2 ? S->vmass_flux_accum : nullptr, ascale));
        if (NH) {
            sx_.fork();
            explicit_part(sx_.s);
        }
        GRIST_LAUNCH(h, PN("k_theta_flux"), st, (quad ? k_theta_flux<P, sizeof(TA) == 4 ? 4 : 1> : k_theta_flux<P, 1>)<<<gEH, kBlock, 0, st>>>(m, d, DT, F, theta, Fth));
        GRIST_LAUNCH(h, PN("k_theta_update"), st, (thv == kPvV   ? k_theta_update<P, kPvV>
                                                   : thv == kPvH ? k_theta_update<P, kPvH>
                                                                 : k_theta_update<P, 1>)<<<gCT, kBlock, 0, st>>>(
            m, d, DTU, Fth, theta, Mv, S->dpi_theta, th_outs[s3], h3));
        if (!pv_with_wind && !short_forms<P>()) {
            sw_.fork();
            edge_pv(sw_.s);
        }
        if (NH) {
            sx_.join();
            if (late) {
                sw_.fork();
                wind(sw_.s);
            }
            cudaError_t se = cudaSuccess;
            const int form = dycore_tuning(h).column_solve;
            const bool blocks = form == 2 || (form == 0 && solve_by_blocks(m.nC, L));
            GRIST_LAUNCH(h, blocks ? PN("k_nh_solve_block") : PN("k_nh_solve"), st, se = (launch_solve<P::EMU, P::DF, short_forms<P>()>(
                m, d, DL, wst, phst, th_outs[s3], rthn, dphn, p_n, ps_outs[s3], h3, w_outs[s3], phi_outs[s3], p_outs[s3],
                alp, phl, dpp, bpos, bneg, blocks, st)));
            if (se != cudaSuccess) return GRIST_ECUDA;
        } else {
            GRIST_LAUNCH(h, PN("k_hydro_diag"), st, k_hydro_diag<P::EMU, P::DF, short_forms<P>()><<<gW, kBlock, 0, st>>>(
                m, d, ex, bkap, ps_outs[s3], th_outs[s3], p, alp, phl));
        }
        sw_.join();
        if (short_forms<P>()) edge_pv(st);
        GRIST_LAUNCH(h, PN("k_momentum"), st, k_momentum<P, NH><<<gE, kBlock, 0, st>>>(
            m, d, DL, u_in, u, u_outs[s3], F, qv, Gq, K, Mv, rsum, p_outs[s3], alp, phl, dpp, h3, status));
        u_in = u_outs[s3];
        ps_in = ps_outs[s3];
        th_in = th_outs[s3];
        w_in = w_outs[s3];
        phi_in = phi_outs[s3];
    }
    if (S->accum_weight) GRIST_LAUNCH(h, PN("k_add_scalar"), st, k_add_scalar<<<1, 32, 0, st>>>(S->accum_weight, ascale));
    if (cudaGetLastError() != cudaSuccess) return GRIST_ECUDA;
    if (NH && S->p_nh) S->p_nh_valid = 1;
    return GRIST_OK;
}

int check(grist_mesh h, grist_dycore_state *S, const grist_dycore_params *prm, grist_precision prec, double dt,
          bool nh) {
    if (!h || !S || !prm) return GRIST_EINVAL;
    if (!(dt > 0) || !std::isfinite(dt)) return GRIST_EINVAL;
    if (prec != GRIST_FP64 && prec != GRIST_MIX && prec != GRIST_MIX_DBL_MASS && prec != GRIST_MIX_DF)
        return GRIST_EINVAL;
    const int L = prm->n_levels;
    if (L < 2 || L > GRIST_MAXL || prm->ld < L || prm->ld_int < L + 1) return GRIST_EINVAL;
    if (nh && L > kNHMax) return GRIST_EUNSUPPORTED;
    if (!S->u || !S->ps || !S->dpi_theta || !prm->b_interface || !prm->phi_surface) return GRIST_EINVAL;
    if (nh && (!S->w || !S->phi)) return GRIST_EINVAL;
    if (prm->b_interface[0] != 0.0 || prm->b_interface[L] != 1.0) return GRIST_EINVAL;
    for (int k = 0; k < L; k++)
        if (!(prm->b_interface[k + 1] > prm->b_interface[k])) return GRIST_EINVAL;
    if (!(prm->pi_top >= 0) || !(prm->p0 > 0) || !(prm->rd > 0) || !(prm->cp > prm->rd) || !(prm->g > 0))
        return GRIST_EINVAL;
    if (nh && !(prm->offcentre_beta > 0 && prm->offcentre_beta <= 1)) return GRIST_EINVAL;
    if (!std::isfinite(S->accum_scale) || S->accum_scale < 0) return GRIST_EINVAL;
    if (prm->emulate_fp32_rows & ~GRIST_ROW_ALL) return GRIST_EINVAL;
    return GRIST_OK;
}

}  // namespace
}  // namespace grist

using namespace grist;

extern "C" int grist_dycore_step_hydro(grist_mesh h, grist_dycore_state *S, const grist_dycore_params *prm,
                                       grist_precision prec, double dt, void *stream) {
    int rc = check(h, S, prm, prec, dt, false);
    if (rc != GRIST_OK) return rc;
    if (cudaSetDevice(mesh_device(h)) != cudaSuccess) return GRIST_ECUDA;
    cudaStream_t st = (cudaStream_t)stream;
    if (prm->emulate_fp32_rows) {
        if (prec != GRIST_FP64) return GRIST_EUNSUPPORTED;
        return dycore_step<PolFP64EMU, false>(h, S, prm, dt, st);
    }
    switch (prec) {
        case GRIST_FP64: return dycore_step<PolFP64, false>(h, S, prm, dt, st);
        case GRIST_MIX: return dycore_step<PolMIX, false>(h, S, prm, dt, st);
        case GRIST_MIX_DF: return dycore_step<PolMIXDF, false>(h, S, prm, dt, st);
        default: return dycore_step<PolMIXDBL, false>(h, S, prm, dt, st);
    }
}

extern "C" int grist_dycore_step_nh(grist_mesh h, grist_dycore_state *S, const grist_dycore_params *prm,
                                    grist_precision prec, double dt, void *stream) {
    int rc = check(h, S, prm, prec, dt, true);
    if (rc != GRIST_OK) return rc;
    if (cudaSetDevice(mesh_device(h)) != cudaSuccess) return GRIST_ECUDA;
    cudaStream_t st = (cudaStream_t)stream;
    if (prm->emulate_fp32_rows) {
        if (prec != GRIST_FP64) return GRIST_EUNSUPPORTED;
        return dycore_step<PolFP64EMU, true>(h, S, prm, dt, st);
    }
    switch (prec) {
        case GRIST_FP64: return dycore_step<PolFP64, true>(h, S, prm, dt, st);
        case GRIST_MIX: return dycore_step<PolMIX, true>(h, S, prm, dt, st);
        case GRIST_MIX_DF: return dycore_step<PolMIXDF, true>(h, S, prm, dt, st);
        default: return dycore_step<PolMIXDBL, true>(h, S, prm, dt, st);
    }
}

extern "C" int grist_dycore_set_tuning(grist_mesh h, const grist_dycore_tuning *t) {
    if (!h || !t || t->column_solve < 0 || t->column_solve > 2) return GRIST_EINVAL;
    if (t->wind_placement < 0 || t->wind_placement > 2) return GRIST_EINVAL;
    dycore_tuning(h) = *t;
    return GRIST_OK;
}

extern "C" int grist_dycore_get_tuning(grist_mesh h, grist_dycore_tuning *t) {
    if (!h || !t) return GRIST_EINVAL;
    *t = dycore_tuning(h);
    return GRIST_OK;
}

extern "C" int grist_diag_vorticity(grist_mesh h, const void *u, grist_precision prec, int32_t n_levels, int32_t ld,
                                    double *vor, void *stream) {
    if (!h || !u || !vor || n_levels < 1 || n_levels > GRIST_MAXL || ld < n_levels) return GRIST_EINVAL;
    if (prec != GRIST_FP64 && prec != GRIST_MIX && prec != GRIST_MIX_DBL_MASS && prec != GRIST_MIX_DF)
        return GRIST_EINVAL;
    if (cudaSetDevice(mesh_device(h)) != cudaSuccess) return GRIST_ECUDA;
    const DevMesh &m = dev_mesh(h);
    cudaStream_t st = (cudaStream_t)stream;
    auto go = [&](auto kern, int v, const auto *w) {
        const LevelDiv Dg = make_div((uint32_t)(n_levels / v));
        kern<<<grid_for((long long)m.nV * Dg.d, kBlock), kBlock, 0, st>>>(m, ld, Dg, w, vor);
    };
    auto fits = [&](int v, size_t size) {
        return n_levels % v == 0 && ld % v == 0 && (uintptr_t)u % (v * size) == 0 && (uintptr_t)vor % 16 == 0;
    };
    if (prec == GRIST_FP64) {
        if (fits(2, 8)) go(k_diag_vort<double, 2>, 2, (const double *)u);
        else go(k_diag_vort<double, 1>, 1, (const double *)u);
    } else {
        if (fits(4, 4)) go(k_diag_vort<float, 4>, 4, (const float *)u);
        else if (fits(2, 4)) go(k_diag_vort<float, 2>, 2, (const float *)u);
        else go(k_diag_vort<float, 1>, 1, (const float *)u);
    }
    return cudaGetLastError() == cudaSuccess ? GRIST_OK : GRIST_ECUDA;
}

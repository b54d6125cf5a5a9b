// dugks_strip.cuh -- the step kernel of the central reconstruction: one warp marches up a strip of 32 columns.
//
// Each lane owns one column.  Per row it sums phi', forms the cell record (macros, psi-bar-plus of Eq. 29, the
// psi~+ partials of Eq. 30), the west x-face and the y-face to the row below, and finishes the row below with the
// flux update (Eq. 24).  What a row needs from the rows around it stays in the lane's registers; what it needs from
// the columns beside it comes by shuffles.  A grid is cut into strips of 28 columns and chunks of rows, as many as
// run at once (strip_plan); rows arrive by TMA two ahead of use (FP32 between walls three) and leave by TMA stores.
//
// Why a march: a tile of 32 x 8 cells computes a ring of 84 more records and 8 % of its faces twice, holds all of it
// in shared memory between four CTA barriers, and spends a fifth of its instructions on addresses.  A strip
// computes 32 records and 64 faces for 28 cells (14 % more than it needs; two record rows more per chunk) and
// meets no barrier at all.  What bounds it: FP32, issue slots (72 % active; any spill doubles the time, the first-level
// cache being what the shared memory leaves); FP64, the FP64 pipe (85 % active).  Wider strips exchange columns through
// shared memory behind CTA barriers: 64 to 224 columns are 5 to 80 % slower in FP32 and equal in FP64.
//
// Measured, tile kernel -> strip kernel: FP32 2048^2 287 -> 206 us a step, 4096^2 1,150 -> 794, 509 x 387 26.9 -> 16.6,
// 64^2 10.3 -> 5.0, 256 x 1024 between walls 28.9 -> 21.4; FP64 1024^2 2,464 -> 1,757.
#pragma once

#include "dugks_device.cuh"

namespace dugks {

// ---- pairs of FP64 values ----
template <typename Real> struct Pair;
template <> struct Pair<double> { using T = double2; };
template <typename Real> using V2 = typename Pair<Real>::T;

__device__ __forceinline__ double2 v2(double a, double b) { return make_double2(a, b); }
__device__ __forceinline__ double2 v2(double a) { return make_double2(a, a); }
__device__ __forceinline__ double2 vfma(double2 a, double2 b, double2 c) {
    return make_double2(fma(a.x, b.x, c.x), fma(a.y, b.y, c.y));
}
__device__ __forceinline__ double2 vmul(double2 a, double2 b) { return make_double2(a.x * b.x, a.y * b.y); }
__device__ __forceinline__ double2 vadd(double2 a, double2 b) { return make_double2(a.x + b.x, a.y + b.y); }
__device__ __forceinline__ double2 vsub(double2 a, double2 b) { return make_double2(a.x - b.x, a.y - b.y); }

// Directions in pairs: A = (1, 3) along +x, +y; B = (5, 7) their opposites; C = (2, 4) the diagonals with
// xi_y = +1; D = (6, 8) their opposites.  Components of xi: A (1,0) (0,1); C (1,1) (-1,1); B = -A; D = -C.
template <typename Real>
struct Dirs {
    V2<Real> A, B, C, D;
};

// What one cell hands to the faces around it.
template <typename Real, bool COUPLED>
struct CellRec {
    Dirs<Real> f, g;   // psi-bar-plus
    Real f0, L;
    V2<Real> G, E;     // 12 grad phi, dt d_t(phi u); L = 6 lap phi
};

// Sums of two cells' fields at a face: f0 of psi-bar-plus, 12 grad phi, dt d_t(phi u), 6 lap phi.
template <typename Real>
struct FaceSum {
    Real f0, L;
    V2<Real> G, E;
};

// The directions that cross a face, for both models: n = (A, B) components along the normal.
template <typename Real>
struct Flux {
    V2<Real> fC, fD, gC, gD, fn, gn;
};

// Geometry of the launch (host side and device side share it).
constexpr int kStripLanes = 32;   // columns of a strip with its halo: one warp
constexpr int kStripCtas = 8;     // CTAs the register allocation leaves room for on an SM: two warps a scheduler

// FP32 without walls keeps psi~+ and the south flux of the row below in shared memory (52 values a lane): 156
// registers instead of 225, three warps a scheduler instead of two (2048^2 212 -> 206 us, 4096^2 829 -> 794).  With
// walls the top wall's flux stays in registers too and the same cap spills.
template <typename Real, bool WALLY>
__host__ __device__ constexpr bool strip_keeps() {
    return sizeof(Real) == 4 && !WALLY;
}
template <typename Real, bool WALLY>
__host__ __device__ constexpr int strip_ctas() {
    return strip_keeps<Real, WALLY>() ? 12 : kStripCtas;
}

template <typename Real, bool COUPLED, bool SHF, bool KEEP>
struct StripShape {
    static constexpr int HX = 2;                   // phi halo: columns on each side of the strip's own
    static constexpr int NQ = COUPLED ? 18 : 9;
    static constexpr int S = sizeof(Real) == 4 && !KEEP ? 4 : 3;   // staged rows in flight or in use
    static constexpr int KG = COUPLED ? 13 : 8;    // kept groups of 4 values: psi~+ of two rows, one flux
    static constexpr int AL = 128 / int(sizeof(Real));
    static constexpr int RG = SHF ? 0 : 4;   // record groups of 4 values (exchanged by shuffles: none)
    __host__ __device__ static constexpr int up(int v) { return (v + AL - 1) / AL * AL; }
    // columns of a staged row: x0 - 4 .. x0 - 4 + box - 1
    __host__ __device__ static constexpr int box(int w) { return w + 4; }
    __host__ __device__ static constexpr int own(int w) { return w - 2 * HX; }
    __host__ __device__ static constexpr int hist_off(int w) { return up(NQ * box(w)); }
    __host__ __device__ static constexpr int slot(int w) { return hist_off(w) + up(2 * box(w)); }
    __host__ __device__ static constexpr int rec_rows(bool wally) { return wally ? 2 : 1; }
    // offsets in elements: staged rows, the finished row, records, fluxes, phi row or kept values, barriers
    __host__ __device__ static constexpr int off_out(int w) { return S * slot(w); }
    __host__ __device__ static constexpr int out_hist(int w) { return up(NQ * own(w)); }
    __host__ __device__ static constexpr int off_rec(int w) { return off_out(w) + out_hist(w) + up(2 * own(w)); }
    __host__ __device__ static constexpr int rec_stride(int w) { return up(RG * 4 * (w + 2)); }
    __host__ __device__ static constexpr int off_flux(int w, bool wally) {
        return off_rec(w) + rec_rows(wally) * rec_stride(w);
    }
    __host__ __device__ static constexpr int off_phi(int w, bool wally) {
        return off_flux(w, wally) + (SHF ? 0 : up(6 * (w + 1) + 4));
    }
    __host__ __device__ static constexpr int off_bar(int w, bool wally) { return off_phi(w, wally) + (SHF ? 0 : up(w + 2)) + (KEEP ? KG * 4 * w : 0); }
    __host__ __device__ static constexpr size_t smem_bytes(int w, bool wally) {
        return size_t(off_bar(w, wally)) * sizeof(Real) + S * 8 + 128;
    }
};

// Columns are exchanged by shuffles; in FP64 with walls (Allen-Cahn alone) through shared memory (the wall faces read
// the records of two rows from there).
template <typename Real, bool WALLY>
__host__ __device__ constexpr bool strip_shuffles() {
    return !WALLY || sizeof(Real) == 4;
}
__device__ __forceinline__ float from_west(float v) { return __shfl_up_sync(0xffffffffu, v, 1); }
__device__ __forceinline__ float from_east(float v) { return __shfl_down_sync(0xffffffffu, v, 1); }
__device__ __forceinline__ double from_west(double v) { return __shfl_up_sync(0xffffffffu, v, 1); }
__device__ __forceinline__ double from_east(double v) { return __shfl_down_sync(0xffffffffu, v, 1); }
__device__ __forceinline__ double2 from_west(double2 v) { return make_double2(from_west(v.x), from_west(v.y)); }
__device__ __forceinline__ double2 from_east(double2 v) { return make_double2(from_east(v.x), from_east(v.y)); }
__device__ __forceinline__ float2 from_west(float2 v) { return make_float2(from_west(v.x), from_west(v.y)); }
__device__ __forceinline__ float2 from_east(float2 v) { return make_float2(from_east(v.x), from_east(v.y)); }

// phi' of one row with its west-east difference and sum.
template <typename Real>
struct PhiRow {
    Real p, d, s;
};

// Constants of one problem folded for the strip kernel.  A cell keeps G = 12 grad phi, L = 6 lap phi and
// E = dt d_t(phi u) unscaled, a face the sums of its two cells' (24 grad phi, 12 lap phi, 2 dt d_t(phi u)); the
// factors sit in the constants of the point kind.
template <typename Real>
struct PointK {
    Real eps;              // 1e-16 in units of G^2
    Real drho;             // grad rho = drho G
    Real beta, kappa;      // mu_phi grad phi = (beta phi (1 - phi) (phi - 1/2) + kappa L) G
    Real step, half;       // dt and dt/2 at a cell, h and h/2 at a face
    Real hd;               // half * drho
    Real kP, kU, kN, kD;   // f: (c1 f_eq + c2 S) / 36 = kP phi' + xi . (kU phi u + kN phi (1 - phi) n + kD E)
    Real kb, kc;           // g: cb / 36 = kb / (2 tau + step), cc / 36 = kc tau / (3 (2 tau + step))
};
template <typename Real>
struct StripPhys {
    PointK<Real> cell, face;
    Real rho_l, drho, visc_a, visc_b, gx, gy, rho_ref, phi_ref, u0x, u0y;
    Real nb, ff_a;         // -pf_b, ff_a
    Real cp, cm, h2, ht;   // 1/2 + h, 1/2 - h, 2 h, h / 4
    Real dt, h;
    int visc_linear, grav_mode, vel_kind;
};
template <typename Real>
inline StripPhys<Real> strip_phys(const Phys<double> &p) {
    StripPhys<Real> o;
    auto point = [&](double sum, double c1, double c2, double step, double g) {   // sum: cells added up
        PointK<Real> k;
        k.eps = Real(1e-16 * 144.0 * sum * sum);
        k.drho = Real(p.drho / (12.0 * sum));
        k.beta = Real(-p.beta4 / (12.0 * sum));
        k.kappa = Real(-p.kappa / (6.0 * sum) / (12.0 * sum));
        k.step = Real(step);
        k.half = Real(0.5 * step);
        k.hd = Real(0.5 * step * p.drho / (12.0 * sum));
        k.kP = Real(c1 / 36.0);
        k.kU = Real(3.0 * c1 / 36.0);
        k.kN = Real(c2 * p.theta_k / 36.0);
        k.kD = Real(3.0 * c2 * p.inv_dt / (36.0 * sum));
        k.kb = Real(g / 36.0);
        k.kc = Real(3.0 * g / 36.0);
        return k;
    };
    o.cell = point(1.0, p.pf_b, p.pf_c, p.dt, 3.0 * p.h);
    o.face = point(2.0, p.ff_b, p.ff_c, p.h, p.h);
    o.rho_l = Real(p.rho_l);
    o.drho = Real(p.drho);
    o.visc_a = Real(p.visc_a);
    o.visc_b = Real(p.visc_b);
    o.gx = Real(p.gx);
    o.gy = Real(p.gy);
    o.rho_ref = Real(p.rho_ref);
    o.phi_ref = Real(p.phi_ref);
    o.u0x = Real(p.u0x);
    o.u0y = Real(p.u0y);
    o.nb = Real(-p.pf_b);
    o.ff_a = Real(p.ff_a);
    o.cp = Real(0.5 + p.h);
    o.cm = Real(0.5 - p.h);
    o.h2 = Real(2.0 * p.h);
    o.ht = Real(0.25 * p.h);
    o.dt = Real(p.dt);
    o.h = Real(p.h);
    o.visc_linear = p.visc_linear;
    o.grav_mode = p.grav_mode;
    o.vel_kind = p.vel_kind;
    return o;
}

// FP64: the hardware's 20-bit seed refined once at third order: with e = 1 - x y the series 1 / x = y (1 + e + e^2 +
// ...), with e = 1 - x y^2 the series 1 / sqrt(x) = y (1 + e / 2 + 3 e^2 / 8 + ...); what is left is of order e^3.
// Within 1 ulp for arguments of 2^-1021 to 2^1021.  Where the seed is 0, infinite or NaN (x infinite, zero, outside
// that range or NaN) it is the result, as of a division; the test is integer work, which the FP64 pipe does not see.
__device__ __forceinline__ bool seed_is_result(double y) {
#ifdef __CUDA_ARCH__
    const unsigned m = (unsigned)__double2hiint(y) & 0x7fffffffu;
    return m - 0x00100000u >= 0x7fe00000u;
#else
    return false;
#endif
}
__device__ __forceinline__ double rcp_s(double x) {
    double y = x;
#ifdef __CUDA_ARCH__
    asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(x));
#endif
    const double e = fma(-x, y, 1.0);
    return seed_is_result(y) ? y : fma(y, fma(e, e, e), y);
}
__device__ __forceinline__ double rsqrt_s(double x) {
    double y = x;
#ifdef __CUDA_ARCH__
    asm("rsqrt.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(x));
#endif
    const double e = fma(-(x * y), y, 1.0);
    return seed_is_result(y) ? y : fma(y, e * fma(0.375, e, 0.5), y);
}

// State at a cell or a face (units of G, L and E above).
template <typename Real>
struct StripPt {
    Real sphi, phi;               // phi - phi_ref, phi
    V2<Real> G, E;
    Real L, rho, irho, lin;
    Real inv, tin;                // 1 / (2 tau_g + step), tau_g / (3 (2 tau_g + step))
    V2<Real> F, u;
    Real tn;                      // phi (1 - phi) / |G|
    Real Q, usq;                  // p' = 0.6 Q; |u|^2
};

// Closures of Eqs. 3-4, 6, 9-10, 34-36.  With mu = num / den (linear rule lin / 1, reciprocal rule 1 / lin) and
// e = 6 num + step rho den, 1 / (2 tau_g + step) = rho den / e and tau_g / (2 tau_g + step) = 3 num / e;
// 1 / rho = den e / (rho den e) comes from the same reciprocal.
template <typename Real, bool COUPLED>
__device__ __forceinline__ void strip_closures(const StripPhys<Real> &ph, const PointK<Real> &k, StripPt<Real> &s,
                                               bool swapped = false) {
    const Real phi = s.phi;
    const Real t = phi * (Real(1) - phi);
    s.tn = t * rsqrt_s(s.G.x * s.G.x + (s.G.y * s.G.y + k.eps));
    if constexpr (COUPLED) {
        s.rho = ph.rho_l + ph.drho * phi;
        const Real M = k.kappa * s.L + (k.beta * t) * (phi - Real(0.5));
        s.lin = ph.visc_a * phi + ph.visc_b;
        const Real num = ph.visc_linear ? s.lin : Real(1), den = ph.visc_linear ? Real(1) : s.lin;
        const Real rd = s.rho * den, e = k.step * rd + Real(6) * num;
        const Real R = rcp_s(rd * e);
        s.irho = den * (e * R);
        const Real r = rd * R;
        s.inv = rd * r;
        s.tin = num * r;
        V2<Real> g = swapped ? v2(ph.gy, ph.gx) : v2(ph.gx, ph.gy);
        if (ph.grav_mode) g = vmul(v2(s.rho - ph.rho_ref), g);
        s.F = vfma(v2(M), s.G, g);
    }
}

template <typename Real>
__device__ __forceinline__ void strip_moments(const Dirs<Real> &g, V2<Real> &m, Real &sn) {
    const V2<Real> a = vsub(g.A, g.B), c = vsub(g.C, g.D);
    const V2<Real> t = vadd(vadd(g.A, g.B), vadd(g.C, g.D));
    m = vadd(a, v2(c.x - c.y, c.x + c.y));
    sn = t.x + t.y;
}

// u and p (Eqs. 32-33) from the g moments.
template <typename Real>
__device__ __forceinline__ void strip_velocity_pressure(const PointK<Real> &k, V2<Real> m, Real sn, StripPt<Real> &s) {
    s.u = vmul(vfma(v2(k.half), s.F, m), v2(s.irho));
    s.usq = s.u.x * s.u.x + s.u.y * s.u.y;
    s.Q = (k.hd * (s.u.x * s.G.x + s.u.y * s.G.y) + sn) - Real(2.0 / 3.0) * (s.rho * s.usq);
}

// (c1 f_eq + c2 S^f)_k = w_k 36 (P + xi_k . V) / 36: P and V carry the diagonal weight 1/36; the axes take four
// times that.
template <typename Real>
__device__ __forceinline__ void strip_f_lin(const PointK<Real> &k, const StripPt<Real> &s, V2<Real> phu, Real &P,
                                            V2<Real> &V) {
    P = k.kP * s.sphi;
    V = vfma(v2(k.kD), s.E, vfma(v2(k.kN * s.tn), s.G, vmul(v2(k.kU), phu)));
}

// cb g_eq + cc S^g of a direction k and its opposite are w_k (E + O) and w_k (E - O) with
//   o = 3 xi_k . u, q = o^2 / 2 - 1.5 |u|^2 (Gamma_k / w_k - 1 = q + o),
//   a = cc grad rho, b = 3 cc F, c0 = cb rho - u . (a + b), base = 3 cb p' - u . b,
//   E = base + q c0 + o xi_k.(a + b),  O = xi_k.b + q xi_k.(a + b) + o c0.
// base, c0, a and b carry the diagonal weight 1/36; the axes take four times that.
template <typename Real>
struct GTerms {
    Real base, c0, q0, P, cb;
    V2<Real> b, ec, o;
};
template <typename Real>
__device__ __forceinline__ GTerms<Real> strip_g_terms(const PointK<Real> &k, const StripPt<Real> &s) {
    GTerms<Real> t;
    t.cb = k.kb * s.inv;
    const Real cc = k.kc * s.tin;
    t.b = vmul(v2(Real(3) * cc), s.F);
    t.ec = vfma(v2(cc * k.drho), s.G, t.b);
    t.P = (Real(1.8) * t.cb) * s.Q;
    t.base = t.P - (s.u.x * t.b.x + s.u.y * t.b.y);
    t.c0 = t.cb * s.rho - (s.u.x * t.ec.x + s.u.y * t.ec.y);
    t.q0 = Real(-1.5) * s.usq;
    t.o = vmul(v2(Real(3)), s.u);
    return t;
}
template <typename Real>
__device__ __forceinline__ void strip_g_eo(V2<Real> o, V2<Real> b, V2<Real> ec, const GTerms<Real> &t, V2<Real> &E,
                                           V2<Real> &O) {
    const V2<Real> q = vfma(vmul(v2(Real(0.5)), o), o, v2(t.q0));
    E = vfma(q, v2(t.c0), vfma(o, ec, v2(t.base)));
    O = vfma(q, ec, vfma(o, v2(t.c0), b));
}
template <typename Real>
__device__ __forceinline__ void strip_g_eo1(Real o, Real b, Real ec, const GTerms<Real> &t, Real &E, Real &O) {
    const Real q = (Real(0.5) * o) * o + t.q0;
    E = q * t.c0 + (o * ec + t.base);
    O = q * ec + (o * t.c0 + b);
}
// The pair of diagonals (2, 4) of a vector: xi_2 . v, xi_4 . v.
template <typename T>
__device__ __forceinline__ T diag2(T v) { return v2(v.x + v.y, v.y - v.x); }

// The face state and the distributions crossing the face (Eq. 28) from psi-bar and the sums of the two cells'
// fields; XFACE selects the normal.  swapped: x and y have changed places, the body force follows.
template <typename Real, bool COUPLED, bool XFACE>
__device__ __forceinline__ Flux<Real> strip_face(const StripPhys<Real> &ph, const Dirs<Real> &f, const Dirs<Real> &g,
                                                 const FaceSum<Real> &m, bool wall, V2<Real> uf,
                                                 bool swapped = false) {
    const PointK<Real> &k = ph.face;
    StripPt<Real> s;
    const V2<Real> t = vadd(vadd(f.A, f.B), vadd(f.C, f.D));
    s.sphi = Real(0.5) * m.f0 + (t.x + t.y);
    s.phi = ph.phi_ref + s.sphi;
    s.G = m.G;
    s.E = m.E;
    s.L = m.L;
    strip_closures<Real, COUPLED>(ph, k, s, swapped);
    if constexpr (COUPLED) {
        V2<Real> mm;
        Real sn;
        strip_moments(g, mm, sn);
        if (wall) {
            s.u = v2(Real(0));
            s.usq = Real(0);
            s.Q = sn;
        } else {
            strip_velocity_pressure(k, mm, sn, s);
        }
    } else {
        s.u = wall ? v2(Real(0)) : uf;
    }
    Flux<Real> o;
    {
        Real P;
        V2<Real> V;
        strip_f_lin(k, s, vmul(v2(s.phi), s.u), P, V);
        const V2<Real> d = diag2(V), a = v2(ph.ff_a);
        o.fC = vfma(a, f.C, vadd(v2(P), d));
        o.fD = vfma(a, f.D, vsub(v2(P), d));
        const Real n = XFACE ? V.x : V.y;
        o.fn = vfma(v2(Real(4)), v2(P + n, P - n), vmul(a, XFACE ? v2(f.A.x, f.B.x) : v2(f.A.y, f.B.y)));
    }
    if constexpr (COUPLED) {
        const V2<Real> ga = v2(Real(6) * s.tin);   // 2 tau_g / (2 tau_g + h)
        const GTerms<Real> c = strip_g_terms(k, s);
        V2<Real> E, O;
        strip_g_eo(diag2(c.o), diag2(c.b), diag2(c.ec), c, E, O);
        o.gC = vfma(ga, g.C, vadd(E, O));
        o.gD = vfma(ga, g.D, vsub(E, O));
        Real e, d;
        strip_g_eo1(XFACE ? c.o.x : c.o.y, XFACE ? c.b.x : c.b.y, XFACE ? c.ec.x : c.ec.y, c, e, d);
        o.gn = vfma(v2(Real(4)), v2(e + d, e - d), vmul(ga, XFACE ? v2(g.A.x, g.B.x) : v2(g.A.y, g.B.y)));
    }
    return o;
}

// Adds the flux of one axis: dt xi_n (in - out), the difference first, so that a cell with equal fluxes on both
// sides keeps its value.
template <typename Real, bool COUPLED, bool XAXIS>
__device__ __forceinline__ void strip_add_flux(Real dt, const Flux<Real> &in, const Flux<Real> &out, Dirs<Real> &f,
                                               Dirs<Real> &g) {
    const V2<Real> sc = XAXIS ? v2(dt, -dt) : v2(dt), sd = XAXIS ? v2(-dt, dt) : v2(-dt);
    f.C = vfma(sc, vsub(in.fC, out.fC), f.C);
    f.D = vfma(sd, vsub(in.fD, out.fD), f.D);
    const V2<Real> n = vsub(in.fn, out.fn);
    Real &fa = XAXIS ? f.A.x : f.A.y, &fb = XAXIS ? f.B.x : f.B.y;
    fa += dt * n.x;
    fb -= dt * n.y;
    if constexpr (COUPLED) {
        g.C = vfma(sc, vsub(in.gC, out.gC), g.C);
        g.D = vfma(sd, vsub(in.gD, out.gD), g.D);
        const V2<Real> q = vsub(in.gn, out.gn);
        Real &ga = XAXIS ? g.A.x : g.A.y, &gb = XAXIS ? g.B.x : g.B.y;
        ga += dt * q.x;
        gb -= dt * q.y;
    }
}

// Are all three finite (0 x is NaN for an infinity or a NaN)?  FP64 looks at the exponents and signs with integer
// instructions, which its pipe does not see.
__device__ __forceinline__ bool all_finite(float a, float b, float c) { return a * 0.0f + b * 0.0f + c * 0.0f == 0.0f; }
__device__ __forceinline__ int hi_word(double v) {
#ifdef __CUDA_ARCH__
    return __double2hiint(v);
#else
    return 0;
#endif
}
__device__ __forceinline__ bool all_finite(double a, double b, double c) {
    const int m = 0x7ff00000;
    return (hi_word(a) & m) != m && (hi_word(b) & m) != m && (hi_word(c) & m) != m;
}
__device__ __forceinline__ bool positive(double a) {   // down to 2^-1042
    return hi_word(a) > 0 && hi_word(a) <= 0x7ff00000;
}

template <typename Real, bool COUPLED>
__device__ __forceinline__ V2<Real> strip_velocity(const StepArgs<Real> &a, const Phys<Real> &ph, Real x, Real y,
                                                   double t) {
    V2<Real> u = v2(Real(0));
    if constexpr (!COUPLED) prescribed_velocity(ph, x, y, t, u.x, u.y);
    return u;
}

// One cell (Eqs. 29-33) from phi' of three rows, its distributions and history: its record, psi~+ of every direction
// and the new phi u; u: the velocity of the Allen-Cahn-only model.  Returns status bits.
template <typename Real, bool COUPLED>
__device__ __forceinline__ unsigned strip_cell(const StripPhys<Real> &ph, const PhiRow<Real> &pm, const PhiRow<Real> &pc,
                                               const PhiRow<Real> &pn, const Dirs<Real> &d, Real d0, const Dirs<Real> &dg,
                                               Real d0g, V2<Real> hist, bool first, V2<Real> u, CellRec<Real, COUPLED> &nr,
                                               Dirs<Real> &tf, Dirs<Real> &tg, Real &t0f, Real &t0g, V2<Real> &pu) {
    const PointK<Real> &k = ph.cell;
    StripPt<Real> s;
    s.sphi = pc.p;
    s.phi = ph.phi_ref + pc.p;
    s.G = v2(Real(4) * pc.d + (pn.d + pm.d), Real(4) * (pn.p - pm.p) + (pn.s - pm.s));
    s.L = Real(4) * (pc.s + (pn.p + pm.p)) + ((pn.s + pm.s) - Real(20) * pc.p);
    strip_closures<Real, COUPLED>(ph, k, s);
    if constexpr (COUPLED) {
        V2<Real> m;
        Real sn;
        strip_moments(dg, m, sn);
        strip_velocity_pressure(k, m, sn, s);
    } else {
        s.u = u;
    }
    pu = vmul(v2(s.phi), s.u);
    s.E = vsub(pu, hist);
    if (first) s.E = v2(Real(0));
    nr.G = s.G;
    nr.E = s.E;
    nr.L = s.L;
    const Real k43 = Real(4.0 / 3.0);
    {   // f: psi-bar-plus = d + e with e = pf_b f_eq + pf_c S - pf_b d, psi~+ = d + 4/3 e; the rest
        // direction takes minus the sum of the others' e (all nine add up to zero)
        Real P;
        V2<Real> V;
        strip_f_lin(k, s, pu, P, V);
        const V2<Real> dv = diag2(V), nb = v2(ph.nb), four = v2(Real(4));
        const V2<Real> eA = vfma(four, vadd(v2(P), V), vmul(nb, d.A));
        const V2<Real> eB = vfma(four, vsub(v2(P), V), vmul(nb, d.B));
        const V2<Real> eC = vfma(nb, d.C, vadd(v2(P), dv));
        const V2<Real> eD = vfma(nb, d.D, vsub(v2(P), dv));
        nr.f.A = vadd(d.A, eA);
        nr.f.B = vadd(d.B, eB);
        nr.f.C = vadd(d.C, eC);
        nr.f.D = vadd(d.D, eD);
        tf.A = vfma(v2(k43), eA, d.A);
        tf.B = vfma(v2(k43), eB, d.B);
        tf.C = vfma(v2(k43), eC, d.C);
        tf.D = vfma(v2(k43), eD, d.D);
        const V2<Real> e4 = vadd(vadd(eC, eD), vadd(eA, eB));
        const Real e0 = -(e4.x + e4.y);
        nr.f0 = d0 + e0;
        t0f = d0 + k43 * e0;
    }
    if constexpr (COUPLED) {
        const GTerms<Real> t = strip_g_terms(k, s);
        const Real cb = Real(-36) * t.cb;
        const V2<Real> nb = v2(cb), four = v2(Real(4));
        V2<Real> E, O;
        strip_g_eo(t.o, t.b, t.ec, t, E, O);
        const V2<Real> eA = vfma(four, vadd(E, O), vmul(nb, dg.A));
        const V2<Real> eB = vfma(four, vsub(E, O), vmul(nb, dg.B));
        strip_g_eo(diag2(t.o), diag2(t.b), diag2(t.ec), t, E, O);
        const V2<Real> eC = vfma(nb, dg.C, vadd(E, O));
        const V2<Real> eD = vfma(nb, dg.D, vsub(E, O));
        nr.g.A = vadd(dg.A, eA);
        nr.g.B = vadd(dg.B, eB);
        nr.g.C = vadd(dg.C, eC);
        nr.g.D = vadd(dg.D, eD);
        tg.A = vfma(v2(k43), eA, dg.A);
        tg.B = vfma(v2(k43), eB, dg.B);
        tg.C = vfma(v2(k43), eC, dg.C);
        tg.D = vfma(v2(k43), eD, dg.D);
        const Real e0 = cb * d0g + (Real(16) * (t.base + t.q0 * t.c0) - Real(36) * t.P);
        t0g = d0g + k43 * e0;
    }
    const bool bad = !all_finite(s.phi, s.u.x, s.u.y);
    bool nonphys = false;
    if constexpr (COUPLED) nonphys = !positive(s.rho) || !positive(s.lin);
    return (bad ? STATUS_NONFINITE : 0u) | (nonphys ? STATUS_NONPHYSICAL : 0u);
}

// Central reconstruction (Eq. 27) of one model, v = (1/2 + h c_n) a + (1/2 - h c_n) b - h c_t s_t between the
// cells a and b of a face, in two halves, so that a row keeps one value per direction for the row above it.
//
// x-face: with P = a + b (west + own), v = (1/2 + h c_n) P - 2 h c_n b + ht c_t (P one row below - P one row
// above); strip_x_open takes all but the row above, strip_x_close adds it.
template <typename Real>
__device__ __forceinline__ Dirs<Real> strip_x_open(const StripPhys<Real> &ph, const Dirs<Real> &P, const Dirs<Real> &b,
                                                   const Dirs<Real> &S, Real ht) {
    const Real cp = ph.cp, cm = ph.cm, h2 = ph.h2;
    Dirs<Real> o;
    o.C = vfma(v2(ht), S.C, vfma(v2(-h2, h2), b.C, vmul(v2(cp, cm), P.C)));
    o.D = vfma(v2(-ht), S.D, vfma(v2(h2, -h2), b.D, vmul(v2(cm, cp), P.D)));
    o.A = v2(cp * P.A.x - h2 * b.A.x, Real(0.5) * P.A.y + ht * S.A.y);
    o.B = v2(cm * P.B.x + h2 * b.B.x, Real(0.5) * P.B.y - ht * S.B.y);
    return o;
}
template <typename Real>
__device__ __forceinline__ void strip_x_close(Dirs<Real> &o, const Dirs<Real> &N, Real ht) {
    o.C = vfma(v2(-ht), N.C, o.C);
    o.D = vfma(v2(ht), N.D, o.D);
    o.A.y -= ht * N.A.y;
    o.B.y += ht * N.B.y;
}
// y-face: strip_y_open takes the cell below (a and its east - west difference R), strip_y_close the one above.
template <typename Real>
__device__ __forceinline__ Dirs<Real> strip_y_open(const StripPhys<Real> &ph, const Dirs<Real> &a, const Dirs<Real> &R) {
    const Real cp = ph.cp, cm = ph.cm, ht = ph.ht;
    Dirs<Real> o;
    o.C = vfma(v2(-ht, ht), R.C, vmul(v2(cp), a.C));
    o.D = vfma(v2(ht, -ht), R.D, vmul(v2(cm), a.D));
    o.A = v2(Real(0.5) * a.A.x - ht * R.A.x, cp * a.A.y);
    o.B = v2(Real(0.5) * a.B.x + ht * R.B.x, cm * a.B.y);
    return o;
}
template <typename Real>
__device__ __forceinline__ void strip_y_close(const StripPhys<Real> &ph, Dirs<Real> &o, const Dirs<Real> &b,
                                              const Dirs<Real> &R) {
    const Real cp = ph.cp, cm = ph.cm, ht = ph.ht;
    o.C = vfma(v2(-ht, ht), R.C, vfma(v2(cm), b.C, o.C));
    o.D = vfma(v2(ht, -ht), R.D, vfma(v2(cp), b.D, o.D));
    o.A = v2((o.A.x + Real(0.5) * b.A.x) - ht * R.A.x, o.A.y + cm * b.A.y);
    o.B = v2((o.B.x + Real(0.5) * b.B.x) + ht * R.B.x, o.B.y + cp * b.B.y);
}

// ---- records in shared memory: groups of four values, one record per column ----
template <typename Real>
__device__ __forceinline__ void st_pairs(Real *p, V2<Real> a, V2<Real> b) { st4(p, a.x, a.y, b.x, b.y); }
template <typename Real>
__device__ __forceinline__ void ld_pairs(const Real *p, V2<Real> &a, V2<Real> &b) {
    Real v[4];
    ld4(p, v);
    a = v2(v[0], v[1]);
    b = v2(v[2], v[3]);
}

// One wall face from the records in shared memory (R9): `row` this column's record next to the wall, `into` the
// next one into the fluid; gcd, gab the offsets of the record groups.
template <typename Real, bool TOP>
__device__ __forceinline__ Dirs<Real> strip_wall(const Real *row, const Real *into, int gcd, int gab,
                                                 const StripPhys<Real> &ph, Real r0, Real i0, Real &rest) {
    const Real h = ph.h;
    const Real dyw = TOP ? Real(0.5) : Real(-0.5);
    Dirs<Real> c, e, w, n;
    ld_pairs(row + gcd, c.C, c.D);
    ld_pairs(row + gab, c.A, c.B);
    ld_pairs(row + gcd + 4, e.C, e.D);
    ld_pairs(row + gab + 4, e.A, e.B);
    ld_pairs(row + gcd - 4, w.C, w.D);
    ld_pairs(row + gab - 4, w.A, w.B);
    ld_pairs(into + gcd, n.C, n.D);
    ld_pairs(into + gab, n.A, n.B);
    auto sy = [&](Real b, Real i) { return TOP ? b - i : i - b; };
    auto sx = [&](Real ev, Real wv) { return Real(0.5) * (ev - wv); };
    const Real away = TOP ? dyw - h : dyw + h;   // directions leaving the fluid
    Dirs<Real> o;
    rest = r0 + dyw * sy(r0, i0);
    o.A.x = c.A.x + dyw * sy(c.A.x, n.A.x) - h * sx(e.A.x, w.A.x);
    o.B.x = c.B.x + dyw * sy(c.B.x, n.B.x) + h * sx(e.B.x, w.B.x);
    if (TOP) {   // 2, 3, 4 leave; 6, 7, 8 bounce back
        o.A.y = c.A.y + away * sy(c.A.y, n.A.y);
        o.C.x = c.C.x + away * sy(c.C.x, n.C.x) - h * sx(e.C.x, w.C.x);
        o.C.y = c.C.y + away * sy(c.C.y, n.C.y) + h * sx(e.C.y, w.C.y);
        o.B.y = o.A.y;
        o.D = o.C;
    } else {     // 6, 7, 8 leave; 2, 3, 4 bounce back
        o.B.y = c.B.y + away * sy(c.B.y, n.B.y);
        o.D.x = c.D.x + away * sy(c.D.x, n.D.x) + h * sx(e.D.x, w.D.x);
        o.D.y = c.D.y + away * sy(c.D.y, n.D.y) - h * sx(e.D.y, w.D.y);
        o.A.y = o.B.y;
        o.C = o.D;
    }
    return o;
}

// cp.async of one element (4 or 8 bytes).
__device__ __forceinline__ void cp_async_elt(float *dst, const float *src) {
#ifdef __CUDA_ARCH__
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(smem_u32(dst)), "l"(src) : "memory");
#endif
}
__device__ __forceinline__ void cp_async_elt(double *dst, const double *src) {
#ifdef __CUDA_ARCH__
    asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"(smem_u32(dst)), "l"(src) : "memory");
#endif
}
__device__ __forceinline__ void cp_async_arrive(uint64_t *bar) {
#ifdef __CUDA_ARCH__
    asm volatile("cp.async.mbarrier.arrive.noinc.shared::cta.b64 [%0];" ::"r"(smem_u32(bar)) : "memory");
#endif
}

// Both loads of a staged row, by the thread whose `p` is set (predicated: no branch).
__device__ __forceinline__ void tma_load_row(bool p, uint64_t *bar, uint32_t bytes, void *dst, const CUtensorMap *map,
                                             void *dst2, const CUtensorMap *map2, int x, int y) {
#ifdef __CUDA_ARCH__
    asm volatile(
        "{\n .reg .pred p;\n setp.ne.u32 p, %0, 0;\n"
        " @p mbarrier.arrive.expect_tx.shared::cta.b64 _, [%1], %2;\n"
        " @p cp.async.bulk.tensor.3d.shared::cluster.global.mbarrier::complete_tx::bytes [%3], [%4, {%7, %8, %9}], [%1];\n"
        " @p cp.async.bulk.tensor.3d.shared::cluster.global.mbarrier::complete_tx::bytes [%5], [%6, {%7, %8, %9}], [%1];\n}\n" ::"r"(
            (uint32_t)p),
        "r"(smem_u32(bar)), "r"(bytes), "r"(smem_u32(dst)), "l"(reinterpret_cast<uint64_t>(map)), "r"(smem_u32(dst2)),
        "l"(reinterpret_cast<uint64_t>(map2)), "r"(x), "r"(y), "r"(0)
        : "memory");
#endif
}
// Both stores of a finished row, likewise, as one group.
__device__ __forceinline__ void tma_store_row(bool p, const void *src, const CUtensorMap *map, const void *src2,
                                              const CUtensorMap *map2, int x, int y) {
#ifdef __CUDA_ARCH__
    asm volatile(
        "{\n .reg .pred p;\n setp.ne.u32 p, %0, 0;\n"
        " @p cp.async.bulk.tensor.3d.global.shared::cta.bulk_group [%2, {%5, %6, %7}], [%1];\n"
        " @p cp.async.bulk.tensor.3d.global.shared::cta.bulk_group [%4, {%5, %6, %7}], [%3];\n"
        " @p cp.async.bulk.commit_group;\n}\n" ::"r"((uint32_t)p),
        "r"(smem_u32(src)), "l"(reinterpret_cast<uint64_t>(map)), "r"(smem_u32(src2)),
        "l"(reinterpret_cast<uint64_t>(map2)), "r"(x), "r"(y), "r"(0)
        : "memory");
#endif
}
// The waits until the stores issued have read shared memory, and until they are done.
__device__ __forceinline__ void tma_store_wait_read() {
#ifdef __CUDA_ARCH__
    asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory");
#endif
}
__device__ __forceinline__ void tma_store_wait() {
#ifdef __CUDA_ARCH__
    asm volatile("cp.async.bulk.wait_group 0;" ::: "memory");
#endif
}
__device__ __forceinline__ void fence_proxy_async_smem() {
#ifdef __CUDA_ARCH__
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
#endif
}

// Programmatic dependent launch: the next step's CTAs start while this step drains, and wait here until it has
// finished and its writes are visible.
__device__ __forceinline__ void grid_dependency_wait() {
#ifdef __CUDA_ARCH__
    asm volatile("griddepcontrol.wait;" ::: "memory");
#endif
}
__device__ __forceinline__ void grid_launch_dependents() {
#ifdef __CUDA_ARCH__
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
#endif
}

// Row y of the domain for a row at most HX outside it (grids have at least three rows).
template <bool WALLY>
__device__ __forceinline__ int strip_row(int y, int ny) {
    if (WALLY) return map_row<true>(y, ny);
    return y < 0 ? y + ny : (y >= ny ? y - ny : y);
}

struct StripArgs {
    int nstrips;   // strips across the grid
    int rows;      // rows of a chunk
};

// Tensor maps of one step: the staged row of the source, the finished row of the destination.
struct StripMaps {
    CUtensorMap src_state, src_hist, dst_state, dst_hist;
};

// The march of one CTA over rows [ya, yb) of the strip whose first own column is x0.
template <typename Real, bool COUPLED, bool WALLY>
__device__ __forceinline__ void strip_march(const StripMaps &tm, const StepArgs<Real> &a, const StripPhys<Real> &ph,
                                            const Phys<Real> &pv, int x0, int ya, int yb) {
    constexpr bool SHF = strip_shuffles<Real, WALLY>();
    static_assert(SHF || !COUPLED, "shared memory holds the records of f alone");
    using S = StripShape<Real, COUPLED, SHF, false>;
    extern __shared__ __align__(128) unsigned char smem_raw[];
    Real *sm = reinterpret_cast<Real *>(smem_raw + ((128u - (smem_u32(smem_raw) & 127u)) & 127u));
    constexpr int W = kStripLanes;
    const int tid = threadIdx.x;
    constexpr int BW = S::box(W), SLOT = S::slot(W), HO = S::hist_off(W), OW = S::own(W);
    Real *ring = sm;
    Real *sout = sm + S::off_out(W);
    Real *srec = sm + S::off_rec(W);
    Real *sflx = sm + S::off_flux(W, WALLY) + 4 * tid;
    Real *sphi = sm + S::off_phi(W, WALLY) + tid;
    uint64_t *bar = reinterpret_cast<uint64_t *>(sm + S::off_bar(W, WALLY));
    const int nx = a.nx, ny = a.ny;
    const int x = x0 - S::HX + tid;
    const int xend = min(x0 + OW, nx);
    const bool inner = tid >= S::HX && tid < W - S::HX;
    const bool mine = inner && x < xend;
    int xw = x % nx;
    if (xw < 0) xw += nx;
    const int nrows = yb - ya + 2 * S::HX;   // staged rows: y = ya - HX + k

    grid_launch_dependents();
    grid_dependency_wait();
    // staging: TMA when every column needed lies inside the domain, else one cp.async per value
    const bool tma = x0 >= S::HX && xend + S::HX <= nx && !(*((volatile unsigned *)a.status) & STATUS_TIMEOUT);
    bool alive = true;   // no wait has run out
    if (tid == 0) {
        for (int s = 0; s < S::S; s++) mbar_init(bar + s, tma ? 1u : (uint32_t)W);
    }
    __syncwarp();
    auto load_row = [&](int k, int slot) {
        if (k >= nrows) return;
        Real *dst = ring + slot * SLOT;
        uint64_t *b = bar + slot;
        if (tma) {
            const int y = strip_row<WALLY>(ya - S::HX + k, ny);
            tma_load_row(tid == 0, b, (uint32_t)((S::NQ + 2) * BW * sizeof(Real)), dst, &tm.src_state, dst + HO,
                         &tm.src_hist, x0 - 4, y);
        } else {
            const int y = strip_row<WALLY>(ya - S::HX + k, ny);
            const long long g = (long long)y * a.pitch + xw;
            Real *d = dst + tid + 4 - S::HX;
            if (in_bounds(xw >= 0 && xw < nx && y >= 0 && y < ny, a.status)) {
                for (int q = 0; q < S::NQ; q++) cp_async_elt(d + q * BW, a.src + q * a.plane + g);
                cp_async_elt(d + HO, a.hsrc + g);
                cp_async_elt(d + HO + BW, a.hsrc + a.plane + g);
            }
            cp_async_arrive(b);
        }
    };
    for (int k = 0; k < S::S; k++) load_row(k, k);

    const Real *col = ring + tid + 4 - S::HX;
    int slot = 0;           // of the row whose phi' comes next
    uint32_t parity = 0;    // of its barrier
    auto phi_row = [&]() {
        if (!mbar_wait(bar + slot, parity, alive ? kPollLimit : 1)) {
            atomicOr(a.status, STATUS_TIMEOUT);
            alive = false;
        }
        const Real *c = col + slot * SLOT;
        // the smallest terms first: diagonals, axes, rest
        PhiRow<Real> r;
        const V2<Real> t = vadd(vadd(v2(c[2 * BW], c[4 * BW]), v2(c[6 * BW], c[8 * BW])),
                                vadd(v2(c[1 * BW], c[3 * BW]), v2(c[5 * BW], c[7 * BW])));
        r.p = (t.x + t.y) + c[0];
        Real w, e;
        if constexpr (SHF) {
            w = from_west(r.p);
            e = from_east(r.p);
        } else {
            sphi[1] = r.p;
            __syncwarp();
            w = sphi[0];
            e = sphi[2];
        }
        r.d = e - w;
        r.s = e + w;
        return r;
    };
    auto next = [&](int s) { return s + 1 == S::S ? 0 : s + 1; };
    auto advance = [&]() {
        slot = next(slot);
        parity ^= slot == 0 ? 1u : 0u;
    };

    // carried from row to row
    Dirs<Real> Xf, Xg, Sf, Sg;      // opened x-face of row r - 1; west + own sums of row r - 1 (tangential directions)
    Dirs<Real> Yf, Yg;              // opened y-face above row r - 1
    FaceSum<Real> Xm, Ym;           // their sums of the cell fields (Ym: the cell below alone)
    Dirs<Real> tf, tg;              // psi~+ of row r - 1
    Flux<Real> yS;                  // flux through the south face of row r - 1
    Real t0f = Real(0), t0g = Real(0);   // its rest directions, done
    V2<Real> pu = v2(Real(0));           // its phi u
    PhiRow<Real> pm = phi_row();
    advance();
    __syncwarp();
    load_row(S::S, 0);   // row 0 is needed for phi' only
    PhiRow<Real> pc = phi_row();
    int cslot = slot;    // of the row whose record comes next
    advance();
    __syncwarp();
    const int gCDf = 0, gABf = 4 * (W + 2), gAux = 8 * (W + 2), gRest = 12 * (W + 2);
    const int last = yb - ya + 1;
    for (int j = 0; j <= last; j++) {
        const int r = ya - 1 + j;
        const PhiRow<Real> pn = phi_row();
        advance();
        if constexpr (SHF) __syncwarp();
        // the row finished in the last iteration: every thread has written it
        tma_store_row(tid == 0 && j >= 3 && alive, sout, &tm.dst_state, sout + S::out_hist(W), &tm.dst_hist, x0, r - 2);
        const bool row_in = !WALLY || (r >= 0 && r < ny);
        CellRec<Real, COUPLED> nr;
        Dirs<Real> ntf, ntg;
        Real n0f = Real(0), n0g = Real(0);
        V2<Real> npu = v2(Real(0));
        Real *rec = srec + 4 * tid + (WALLY ? (j & 1) * S::rec_stride(W) : 0);   // the west neighbour's record
        if (row_in) {
            // ---- the cell of row r ----
            const Real *c = col + cslot * SLOT;
            Dirs<Real> df, dg;
            Real d0g = Real(0);
            df.A = v2(c[1 * BW], c[3 * BW]);
            df.B = v2(c[5 * BW], c[7 * BW]);
            df.C = v2(c[2 * BW], c[4 * BW]);
            df.D = v2(c[6 * BW], c[8 * BW]);
            V2<Real> u = v2(Real(0));
            if constexpr (COUPLED) {
                dg.A = v2(c[10 * BW], c[12 * BW]);
                dg.B = v2(c[14 * BW], c[16 * BW]);
                dg.C = v2(c[11 * BW], c[13 * BW]);
                dg.D = v2(c[15 * BW], c[17 * BW]);
                d0g = c[9 * BW];
            } else {
                const int yw = WALLY ? r : (r < 0 ? r + ny : (r >= ny ? r - ny : r));
                if (ph.vel_kind == 0) {
                    u = v2(ph.u0x, ph.u0y);
                } else if (ph.vel_kind == 4) {
                    const long long gv = (long long)yw * a.pitch + xw;
                    u = v2(a.vel[gv], a.vel[a.plane + gv]);
                } else {
                    u = strip_velocity<Real, COUPLED>(a, pv, Real(xw) + Real(0.5), Real(yw) + Real(0.5), a.t_n);
                }
            }
            const unsigned bad = strip_cell<Real, COUPLED>(ph, pm, pc, pn, df, c[0], dg, d0g, v2(c[HO], c[HO + BW]),
                                                           a.first_step != 0, u, nr, ntf, ntg, n0f, n0g, npu);
            if (bad && mine && r >= ya && r < yb) atomicOr(a.status, bad);
            if constexpr (!SHF) {
                st_pairs(rec + 4 + gCDf, nr.f.C, nr.f.D);
                st_pairs(rec + 4 + gABf, nr.f.A, nr.f.B);
                st_pairs(rec + 4 + gAux, nr.G, nr.E);
                st2(rec + 4 + gRest, nr.f0, nr.L);
            }
        }
        __syncwarp();
        load_row(j + 1 + S::S, cslot);   // the slot of row r is free: every thread has read it
        cslot = next(cslot);
        Dirs<Real> nSf, nSg;         // west + own sums of row r
        Dirs<Real> Rf, Rg;           // east - west differences of row r
        FaceSum<Real> nXm;
        if (row_in) {
            if constexpr (SHF) {
                auto split = [](const Dirs<Real> &o, Dirs<Real> &sum, Dirs<Real> &R) {
                    const V2<Real> c = from_west(o.C), d = from_west(o.D), a = from_west(o.A), b = from_west(o.B);
                    sum.C = vadd(c, o.C);
                    sum.D = vadd(d, o.D);
                    sum.A = vadd(a, o.A);
                    sum.B = vadd(b, o.B);
                    R.C = vsub(from_east(o.C), c);
                    R.D = vsub(from_east(o.D), d);
                    R.A.x = from_east(o.A.x) - a.x;
                    R.B.x = from_east(o.B.x) - b.x;
                };
                split(nr.f, nSf, Rf);
                nXm.f0 = from_west(nr.f0) + nr.f0;
                nXm.L = from_west(nr.L) + nr.L;
                nXm.G = vadd(from_west(nr.G), nr.G);
                nXm.E = vadd(from_west(nr.E), nr.E);
                if constexpr (COUPLED) split(nr.g, nSg, Rg);
            } else {
                Dirs<Real> q, e;
                V2<Real> u, v;
                Real z[2];
                ld_pairs(rec + gCDf, q.C, q.D);
                ld_pairs(rec + gABf, q.A, q.B);
                ld_pairs(rec + gAux, u, v);
                ld2(rec + gRest, z);
                nSf.A = vadd(q.A, nr.f.A);
                nSf.B = vadd(q.B, nr.f.B);
                nSf.C = vadd(q.C, nr.f.C);
                nSf.D = vadd(q.D, nr.f.D);
                nXm.f0 = z[0] + nr.f0;
                nXm.L = z[1] + nr.L;
                nXm.G = vadd(u, nr.G);
                nXm.E = vadd(v, nr.E);
                ld_pairs(rec + 8 + gCDf, e.C, e.D);
                ld_pairs(rec + 8 + gABf, e.A, e.B);
                Rf.C = vsub(e.C, q.C);
                Rf.D = vsub(e.D, q.D);
                Rf.A.x = e.A.x - q.A.x;
                Rf.B.x = e.B.x - q.B.x;
            }
        }
        const Real half = Real(0.5);
        Flux<Real> xf, yN;
        const bool finish = j >= 2;   // row r - 1 is one of the chunk's own
        if (finish) {
            // ---- the west x-face of row r - 1 ----
            Real ht = ph.ht;
            if (WALLY && (r - 1 == 0 || r == ny)) ht = Real(2) * ph.ht;
            if (WALLY && r == ny) {
                nSf = Sf;
                if constexpr (COUPLED) nSg = Sg;
            }
            strip_x_close(Xf, nSf, ht);
            if constexpr (COUPLED) strip_x_close(Xg, nSg, ht);
            V2<Real> uf = v2(Real(0));
            if constexpr (!COUPLED) {
                const int yw = WALLY ? r - 1 : (r - 1 >= ny ? r - 1 - ny : r - 1);
                if (ph.vel_kind == 4) {
                    const long long kr = (long long)yw * a.pitch + xw, kl = kr - xw + (xw > 0 ? xw - 1 : nx - 1);
                    uf.x = a.vel_faces ? a.vel[2 * a.plane + kl] : half * (a.vel[kl] + a.vel[kr]);
                    uf.y = half * (a.vel[a.plane + kl] + a.vel[a.plane + kr]);
                } else {
                    uf = strip_velocity<Real, COUPLED>(a, pv, Real(xw), Real(yw) + half, a.t_n + double(pv.h));
                }
            }
            xf = strip_face<Real, COUPLED, true>(ph, Xf, Xg, Xm, false, uf);
            if constexpr (!SHF) {
                st_pairs(sflx, xf.fC, xf.fD);
                st2(sflx + 4 * (W + 1) - 2 * tid, xf.fn.x, xf.fn.y);
            }
        }
        // the x-face of row r, opened (next to a wall the slope is one-sided: the row takes itself as the one
        // beyond the wall, and at the top wall closes with itself)
        if (row_in) {
            const bool edge = WALLY && (r == 0 || r == ny - 1);
            const Real ht = edge ? Real(2) * ph.ht : ph.ht;
            if (WALLY && r == 0) {
                Sf = nSf;
                if constexpr (COUPLED) Sg = nSg;
            }
            Xf = strip_x_open(ph, nSf, nr.f, Sf, ht);
            if constexpr (COUPLED) Xg = strip_x_open(ph, nSg, nr.g, Sg, ht);
            Xm = nXm;
            Sf = nSf;
            if constexpr (COUPLED) Sg = nSg;
        }
        if (j >= 1) {
            // ---- the y-face between rows r - 1 and r; with walls also the wall's own faces ----
            auto yface = [&]() {
                strip_y_close(ph, Yf, nr.f, Rf);
                if constexpr (COUPLED) strip_y_close(ph, Yg, nr.g, Rg);
                V2<Real> uf = v2(Real(0));
                if constexpr (!COUPLED) {
                    const int yu = WALLY ? r : (r >= ny ? r - ny : r), yd = yu > 0 ? yu - 1 : ny - 1;
                    if (ph.vel_kind == 4) {
                        const long long kd = (long long)yd * a.pitch + xw, ku = (long long)yu * a.pitch + xw;
                        uf.x = half * (a.vel[kd] + a.vel[ku]);
                        uf.y = a.vel_faces ? a.vel[3 * a.plane + ku] : half * (a.vel[a.plane + kd] + a.vel[a.plane + ku]);
                    } else {
                        uf = strip_velocity<Real, COUPLED>(a, pv, Real(xw) + half, Real(yu), a.t_n + double(pv.h));
                    }
                }
                FaceSum<Real> m;
                m.f0 = Ym.f0 + nr.f0;
                m.L = Ym.L + nr.L;
                m.G = vadd(Ym.G, nr.G);
                m.E = vadd(Ym.E, nr.E);
                return strip_face<Real, COUPLED, false>(ph, Yf, Yg, m, false, uf);
            };
            if constexpr (WALLY) {
                auto wall = [&](auto top) {
                    constexpr bool TOP = decltype(top)::value;
                    const int j0 = j - 1, j1 = TOP ? j - 2 : j;   // iterations whose records to take
                    const Real *row = srec + (j0 & 1) * S::rec_stride(W) + 4 * (tid + 1);
                    const Real *into = srec + (j1 & 1) * S::rec_stride(W) + 4 * (tid + 1);
                    Real rest;
                    const Dirs<Real> fb = strip_wall<Real, TOP>(row, into, gCDf, gABf, ph, row[gRest], into[gRest], rest), gb{};
                    FaceSum<Real> m;   // the cell and its mirror image
                    m.f0 = Real(2) * rest;
                    m.L = Real(2) * row[gRest + 1];
                    m.G = v2(Real(2) * row[gAux], Real(0));
                    m.E = v2(Real(2) * row[gAux + 2], Real(0));
                    return strip_face<Real, COUPLED, false>(ph, fb, gb, m, true, v2(Real(0)));
                };
                if (r - 1 == 0 && j >= 2) yS = wall(std::false_type{});
                if (r == ny) yN = wall(std::true_type{});
                else if (r > 0) yN = yface();
            } else {
                yN = yface();
            }
        }
        if (row_in) {   // the y-face above row r, opened
            Yf = strip_y_open(ph, nr.f, Rf);
            if constexpr (COUPLED) Yg = strip_y_open(ph, nr.g, Rg);
            Ym.f0 = nr.f0;
            Ym.L = nr.L;
            Ym.G = nr.G;
            Ym.E = nr.E;
        }
        if (finish) {
            tma_store_wait_read();   // (only the issuing thread has any)
            __syncwarp();
            Flux<Real> xe;
            const Real *p = sflx + 4;
            if constexpr (SHF) {
                xe.fC = from_east(xf.fC);
                xe.fD = from_east(xf.fD);
                xe.fn = from_east(xf.fn);
                if constexpr (COUPLED) {
                    xe.gC = from_east(xf.gC);
                    xe.gD = from_east(xf.gD);
                    xe.gn = from_east(xf.gn);
                }
            } else {
                ld_pairs(p, xe.fC, xe.fD);
                Real z[2];
                ld2(sflx + 4 * (W + 1) - 2 * tid + 2, z);
                xe.fn = v2(z[0], z[1]);
            }
            // ---- the flux update of row r - 1 ----
            strip_add_flux<Real, COUPLED, true>(ph.dt, xf, xe, tf, tg);
            strip_add_flux<Real, COUPLED, false>(ph.dt, yS, yN, tf, tg);
            if (inner) {
                Real *o = sout + tid - S::HX;
                o[0] = t0f;
                o[1 * OW] = tf.A.x; o[3 * OW] = tf.A.y; o[5 * OW] = tf.B.x; o[7 * OW] = tf.B.y;
                o[2 * OW] = tf.C.x; o[4 * OW] = tf.C.y; o[6 * OW] = tf.D.x; o[8 * OW] = tf.D.y;
                if constexpr (COUPLED) {
                    o[9 * OW] = t0g;
                    o[10 * OW] = tg.A.x; o[12 * OW] = tg.A.y; o[14 * OW] = tg.B.x; o[16 * OW] = tg.B.y;
                    o[11 * OW] = tg.C.x; o[13 * OW] = tg.C.y; o[15 * OW] = tg.D.x; o[17 * OW] = tg.D.y;
                }
                o[S::out_hist(W)] = pu.x;
                o[S::out_hist(W) + OW] = pu.y;
                fence_proxy_async_smem();
            }
        }
        yS = yN;
        tf = ntf;
        tg = ntg;
        t0f = n0f;
        t0g = n0g;
        pu = npu;
        pm = pc;
        pc = pn;
    }
    __syncwarp();
    tma_store_row(tid == 0 && alive, sout, &tm.dst_state, sout + S::out_hist(W), &tm.dst_hist, x0, yb - 1);
    tma_store_wait();
    if (!alive)   // let copies in flight land before the CTA's shared memory is given away
        for (int s = 0; s < S::S; s++) mbar_wait(bar + s, (uint32_t)((nrows - 1 - s) / S::S) & 1u, kPollLimit);
}

// ---------------------------------------------------------------------------
// FP32.  Every value comes from the operations of the tile kernels in their order (the functions of
// dugks_device.cuh, two lanes to an instruction where those pack them), so the two give the same bits: FP32
// round-off of phi decides the interface normal wherever grad phi nearly vanishes, and a reordered sum there
// moves single cells by 1e-3.  What the march saves is the halo: a record is computed once per strip and row, a
// y-face once, and sums over the two cells of an x-face serve the rows above and below.
//
// Pairs hold a direction k = 1..4 and its opposite k + 4.
// ---------------------------------------------------------------------------
struct Rec32 {
    float2 f[4], g[4];
    float f0;
    float2 dp, D;    // grad phi, d_t(phi u)
    float lap;
};

// Central reconstruction across a face of one pair (Eq. 27): (1/2 + h c) a + (1/2 - h c) b, lane 0 with c = C.
template <int C>
__device__ __forceinline__ float2 recon32(float2 a, float2 b, float cp, float cm) {
    const float2 ca = C == 0 ? f2(0.5f) : (C > 0 ? f2(cp, cm) : f2(cm, cp));
    const float2 cb = C == 0 ? f2(0.5f) : (C > 0 ? f2(cm, cp) : f2(cp, cm));
    return fma2(cb, b, mul2(ca, a));
}
// ... and its tangential part, -h c_t s_t with T = (n + n') - (s + s') as s_t, lane 0 with c_t = C.
template <int C>
__device__ __forceinline__ float2 tangent32(float2 v, float2 n, float2 s, float ht) {
    return fma2(C > 0 ? f2(-ht, ht) : f2(ht, -ht), sub2(n, s), v);
}
__device__ __forceinline__ void unpack32(const float2 v[4], float o[9]) {
#pragma unroll
    for (int p = 0; p < 4; p++) {
        o[1 + p] = v[p].x;
        o[5 + p] = v[p].y;
    }
}

// moments9 of pairs: the sums over 2, 3, 4 and 6, 7, 8, and the two halves of the non-rest sum, side by side.
__device__ __forceinline__ void moments32(const float2 g[4], float &mx, float &my, float &sn) {
    mx = ((g[0].x + g[1].x) + g[3].y) - ((g[3].x + g[0].y) + g[1].y);
    const float2 t = add2(add2(g[1], g[2]), g[3]);
    my = t.x - t.y;
    const float2 n = add2(add2(g[0], g[1]), add2(g[2], g[3]));
    sn = n.x + n.y;
}
// Fluxes of one axis: pairs that cross it (x: 1, 2, 4; y: 2, 3, 4).
struct Flux32 {
    float2 f[3], g[3];
};
template <bool XFACE>
__host__ __device__ constexpr int flux_pair(int i) {
    return XFACE ? (i == 2 ? 3 : i) : i + 1;
}
// face_flux on pairs (g direction by direction: its lanes in one instruction gained nothing).
template <bool COUPLED, bool XFACE>
__device__ __forceinline__ Flux32 face32(const Phys<float> &ph, const float2 f[4], float f0, const float2 g[4], float2 dp,
                                         float lap, float2 D, bool wall, float ux, float uy) {
    Pt<float> s;
    float sphi = f0;
#pragma unroll
    for (int p = 0; p < 4; p++) sphi += f[p].x;
#pragma unroll
    for (int p = 0; p < 4; p++) sphi += f[p].y;
    s.phi = ph.phi_ref + sphi;
    s.dpx = dp.x;
    s.dpy = dp.y;
    s.lap = lap;
    s.Dx = D.x;
    s.Dy = D.y;
    closures<float, COUPLED>(ph, s, ph.h);
    if constexpr (COUPLED) {
        float mx, my, sn;
        moments32(g, mx, my, sn);
        if (wall) {
            s.ux = 0.0f;
            s.uy = 0.0f;
            s.pd = 0.6f * sn;
        } else {
            velocity_pressure(mx, my, sn, ph.half_h, s);
        }
    } else {
        s.ux = wall ? 0.0f : ux;
        s.uy = wall ? 0.0f : uy;
    }
    Flux32 o;
    const FLin<float> lf = f_lin(ph, s, ph.ff_b, ph.ff_c);
    auto fpair = [&](auto ic) {
        constexpr int P = flux_pair<XFACE>(decltype(ic)::value), K = P + 1;
        const float e = edot(K, lf.Vx, lf.Vy);
        const float2 q = f2(lf.P + e, lf.P - e), w = f2(wq<float>(K));
        o.f[decltype(ic)::value] = fma2(f2(ph.ff_a), f[P], mul2(w, q));
    };
    fpair(std::integral_constant<int, 0>{});
    fpair(std::integral_constant<int, 1>{});
    fpair(std::integral_constant<int, 2>{});
    if constexpr (COUPLED) {
        const float inv = rcp_r(2.0f * s.taug + ph.h);
        const float a = 2.0f * s.taug * inv, bb = ph.h * inv, c = s.taug * ph.h * inv;
        const GLin<float> gl = g_lin(s, bb, c);
        auto gpair = [&](auto ic) {
            constexpr int P = flux_pair<XFACE>(decltype(ic)::value), K = P + 1;
            o.g[decltype(ic)::value] = f2(a * g[P].x + g_lin_k(K, gl), a * g[P].y + g_lin_k(K + 4, gl));
        };
        gpair(std::integral_constant<int, 0>{});
        gpair(std::integral_constant<int, 1>{});
        gpair(std::integral_constant<int, 2>{});
    }
    return o;
}
// Adds dt xi_n (in - out) of one axis.
template <bool COUPLED, bool XAXIS>
__device__ __forceinline__ void flux32(float dt, const Flux32 &in, const Flux32 &out, float2 f[4], float2 g[4]) {
#pragma unroll
    for (int i = 0; i < 3; i++) {
        const int p = flux_pair<XAXIS>(i), c = XAXIS ? cx(p + 1) : cy(p + 1);
        const float2 d = c > 0 ? f2(dt, -dt) : f2(-dt, dt);
        f[p] = fma2(d, sub2(in.f[i], out.f[i]), f[p]);
        if (COUPLED) g[p] = fma2(d, sub2(in.g[i], out.g[i]), g[p]);
    }
}

__device__ __forceinline__ float4 group32(float2 a, float2 b) { return make_float4(a.x, a.y, b.x, b.y); }
__device__ __forceinline__ void ungroup32(const float4 &v, float2 &a, float2 &b) {
    a = f2(v.x, v.y);
    b = f2(v.z, v.w);
}

// A wall face (R9) from the cell next to the wall, its east and west neighbours and the next cell into the fluid:
// recon_wall on registers.
template <bool TOP>
__device__ __forceinline__ void wall32(const float2 c[4], const float2 e[4], const float2 w[4], const float2 n[4],
                                       float c0, float n0, bool rest, float h, float2 o[4], float &o0) {
    const float dyw = TOP ? 0.5f : -0.5f;
    float C[9], E[9], W[9], N[9], out[9];
    unpack32(c, C);
    unpack32(e, E);
    unpack32(w, W);
    unpack32(n, N);
    C[0] = c0;
    N[0] = n0;
#pragma unroll
    for (int k = 0; k < 9; k++) {
        const bool keep = TOP ? (cy(k) >= 0) : (cy(k) <= 0);
        if (!keep || (k == 0 && !rest)) continue;
        const float b0 = C[k];
        const float sy = TOP ? (b0 - N[k]) : (N[k] - b0);
        float v = b0 + (cy(k) == 0 ? dyw : (cy(k) > 0 ? dyw - h : dyw + h)) * sy;
        if (cx(k) != 0) {
            const float sx = 0.5f * (E[k] - W[k]);
            v -= h * sgnmul(cx(k), sx);
        }
        out[k] = v;
    }
#pragma unroll
    for (int k = 0; k < 9; k++) {
        const bool enters = TOP ? (cy(k) < 0) : (cy(k) > 0);
        if (enters) out[k] = out[opp(k)];
    }
#pragma unroll
    for (int p = 0; p < 4; p++) o[p] = f2(out[1 + p], out[5 + p]);
    if (rest) o0 = out[0];
}

// One cell: the operations of cell_item.  s holds grad phi and lap phi, c points at the cell's column of the staged
// row (planes bw apart, the history at ho), p = phi'.  Returns the record; psi~+ (rest directions in t0), phi u.
template <bool COUPLED>
__device__ __forceinline__ Rec32 cell32(const Phys<float> &ph, const StepArgs<float> &a, Pt<float> &s, const float *c, int bw,
                                        int ho, float p, int xw, int yw, float2 tf[4], float2 tg[4], float2 &t0, float2 &pu,
                                        bool own) {
    Rec32 nr;
                s.phi = ph.phi_ref + p;
                closures<float, COUPLED>(ph, s, ph.dt);
                float2 dg[4];
                if (COUPLED) {
    #pragma unroll
                    for (int q = 0; q < 4; q++) dg[q] = f2(c[(10 + q) * bw], c[(14 + q) * bw]);
                    float mx, my, sn;
                    moments32(dg, mx, my, sn);
                    velocity_pressure(mx, my, sn, ph.half_dt, s);
                } else if (ph.vel_kind == 0) {
                    s.ux = ph.u0x;
                    s.uy = ph.u0y;
                } else if (ph.vel_kind == 4) {
                    const long long gv = (long long)yw * a.pitch + xw;
                    s.ux = a.vel[gv];
                    s.uy = a.vel[a.plane + gv];
                } else {
                    prescribed_velocity(ph, float(xw) + 0.5f, float(yw) + 0.5f, a.t_n, s.ux, s.uy);
                }
                const float phux = s.phi * s.ux, phuy = s.phi * s.uy;
                if (a.first_step) {
                    s.Dx = 0.0f;
                    s.Dy = 0.0f;
                } else {
                    s.Dx = mul_sub(s.phi, s.ux, c[ho]) * ph.inv_dt;
                    s.Dy = mul_sub(s.phi, s.uy, c[ho + bw]) * ph.inv_dt;
                }
                pu = f2(phux, phuy);
                nr.dp = f2(s.dpx, s.dpy);
                nr.D = f2(s.Dx, s.Dy);
                nr.lap = s.lap;
                {
                    const FLin<float> lf = f_lin(ph, s, ph.pf_b, ph.pf_c);
                    float2 bsum2 = f2(0.0f);
                    auto fpair = [&](auto kc) {
                        constexpr int K = decltype(kc)::value;
                        const float2 d = f2(c[K * bw], c[(K + 4) * bw]);
                        const float2 bp = add2(d, fma2(f2(-ph.pf_b), d, f_lin_pair<K>(lf)));
                        nr.f[K - 1] = bp;
                        bsum2 = add2(bsum2, bp);
                        tf[K - 1] = fma2(f2(1.0f / 3.0f), sub2(bp, d), bp);
                    };
                    fpair(std::integral_constant<int, 1>{});
                    fpair(std::integral_constant<int, 2>{});
                    fpair(std::integral_constant<int, 3>{});
                    fpair(std::integral_constant<int, 4>{});
                    const float d = c[0];
                    const float bp = p - (bsum2.x + bsum2.y);
                    nr.f0 = bp;
                    t0.x = bp + (bp - d) * float(1.0 / 3.0);
                }
                if (COUPLED) {
                    const float inv = rcp_r(2.0f * s.taug + ph.dt);
                    const float cb = 3.0f * ph.h * inv, cc = 3.0f * s.taug * ph.h * inv;
                    const GLin<float> gl = g_lin(s, cb, cc);
                    auto gpair = [&](auto kc) {
                        constexpr int K = decltype(kc)::value;
                        const float2 d = dg[K - 1];
                        const float2 bp = add2(d, fma2(f2(-cb), d, g_lin_pair<K>(gl)));
                        nr.g[K - 1] = bp;
                        tg[K - 1] = fma2(f2(1.0f / 3.0f), sub2(bp, d), bp);
                    };
                    gpair(std::integral_constant<int, 1>{});
                    gpair(std::integral_constant<int, 2>{});
                    gpair(std::integral_constant<int, 3>{});
                    gpair(std::integral_constant<int, 4>{});
                    const float d = c[9 * bw], bp = d + (g_lin_k(0, gl) - cb * d);
                    t0.y = bp + (bp - d) * float(1.0 / 3.0);
                }
                if (own) {
                    const bool bad = !all_finite(s.phi, s.ux, s.uy);
                    const bool nonphys = COUPLED && !(s.rho > 0.0f && s.taug > 0.0f);
                    if (bad || nonphys)
                        atomicOr(a.status, (bad ? STATUS_NONFINITE : 0u) | (nonphys ? STATUS_NONPHYSICAL : 0u));
                }
    return nr;
}

template <bool COUPLED, bool WALLY>
__device__ __forceinline__ void strip_march32(const StripMaps &tm, const StepArgs<float> &a, const Phys<float> &ph,
                                              int x0, int ya, int yb) {
    using Real = float;
    constexpr bool KEEP = strip_keeps<float, WALLY>();
    using S = StripShape<float, COUPLED, true, KEEP>;
    extern __shared__ __align__(128) unsigned char smem_raw[];
    float *sm = reinterpret_cast<float *>(smem_raw + ((128u - (smem_u32(smem_raw) & 127u)) & 127u));
    constexpr int W = kStripLanes;
    const int tid = threadIdx.x;
    constexpr int BW = S::box(W), SLOT = S::slot(W), HO = S::hist_off(W), OW = S::own(W);
    float *ring = sm;
    float *sout = sm + S::off_out(W);
    uint64_t *bar = reinterpret_cast<uint64_t *>(sm + S::off_bar(W, WALLY));
    float4 *keep = reinterpret_cast<float4 *>(sm + S::off_phi(W, WALLY)) + tid;   // this lane's groups, W apart
    const int nx = a.nx, ny = a.ny;
    const int x = x0 - S::HX + tid;
    const int xend = min(x0 + OW, nx);
    const bool inner = tid >= S::HX && tid < W - S::HX;
    const bool mine = inner && x < xend;
    int xw = x % nx;
    if (xw < 0) xw += nx;
    const int nrows = yb - ya + 2 * S::HX;   // staged rows: y = ya - HX + k

    grid_launch_dependents();
    grid_dependency_wait();
    // staging: TMA when every column needed lies inside the domain, else one cp.async per value
    const bool tma = x0 >= S::HX && xend + S::HX <= nx && !(*((volatile unsigned *)a.status) & STATUS_TIMEOUT);
    bool alive = true;   // no wait has run out
    if (tid == 0) {
        for (int s = 0; s < S::S; s++) mbar_init(bar + s, tma ? 1u : (uint32_t)W);
    }
    __syncwarp();
    auto load_row = [&](int k, int slot) {
        if (k >= nrows) return;
        float *dst = ring + slot * SLOT;
        uint64_t *b = bar + slot;
        const int y = strip_row<WALLY>(ya - S::HX + k, ny);
        if (tma) {
            tma_load_row(tid == 0, b, (uint32_t)((S::NQ + 2) * BW * sizeof(float)), dst, &tm.src_state, dst + HO,
                         &tm.src_hist, x0 - 4, y);
        } else {
            const long long g = (long long)y * a.pitch + xw;
            float *d = dst + tid + 4 - S::HX;
            if (in_bounds(xw >= 0 && xw < nx && y >= 0 && y < ny, a.status)) {
                for (int q = 0; q < S::NQ; q++) cp_async_elt(d + q * BW, a.src + q * a.plane + g);
                cp_async_elt(d + HO, a.hsrc + g);
                cp_async_elt(d + HO + BW, a.hsrc + a.plane + g);
            }
            cp_async_arrive(b);
        }
    };
    for (int k = 0; k < S::S; k++) load_row(k, k);

    const float *col = ring + tid + 4 - S::HX;
    int slot = 0;           // of the row whose phi' comes next
    uint32_t parity = 0;    // of its barrier
    struct Phi { float p, e, w; };
    auto phi_row = [&]() {
        if (!mbar_wait(bar + slot, parity, alive ? kPollLimit : 1)) {
            atomicOr(a.status, STATUS_TIMEOUT);
            alive = false;
        }
        const float *c = col + slot * SLOT;
        Phi r;
        r.p = c[0];
#pragma unroll
        for (int k = 1; k < 9; k++) r.p += c[k * BW];
        r.e = from_east(r.p);
        r.w = from_west(r.p);
        slot = slot + 1 == S::S ? 0 : slot + 1;
        parity ^= slot == 0 ? 1u : 0u;
        return r;
    };

    // carried from row to row (row m = r - 1)
    Rec32 cur;              // its record
    float2 Vf[4], Vg[4];    // its west x-face, normal part; and the means of the cell fields there
    float V0 = 0.0f, Vl = 0.0f;
    float2 Vd = f2(0.0f), VD = f2(0.0f);
    float2 P1f[4], P1g[4], P2f[4], P2g[4];   // west + own sums of rows m, m - 1 (pairs 1..3)
    float2 tf[4], tg[4];    // psi~+
    float t0f = 0.0f, t0g = 0.0f;
    float2 pu = f2(0.0f);   // phi u
    Flux32 yS, yTop;        // fluxes through its south face, through the top wall
    Phi pm = phi_row();
    __syncwarp();
    load_row(S::S, 0);      // row 0 is needed for phi' only
    int cslot = slot;       // of the row whose record comes next
    Phi pc = phi_row();
    const float cp = 0.5f + ph.h, cm = 0.5f - ph.h;
    const int last = yb - ya + 1;
    for (int j = 0; j <= last; j++) {
        const int r = ya - 1 + j;
        const Phi pn = phi_row();
        __syncwarp();
        // the row finished in the last iteration: every lane has written it
        tma_store_row(tid == 0 && j >= 3 && alive, sout, &tm.dst_state, sout + S::out_hist(W), &tm.dst_hist, x0, r - 2);
        const bool row_in = !WALLY || (r >= 0 && r < ny);
        const int yw = WALLY ? r : (r < 0 ? r + ny : (r >= ny ? r - ny : r));
        Rec32 nr;
        float2 ntf[4], ntg[4];
        float n0f = 0.0f, n0g = 0.0f;
        float2 npu = f2(0.0f);
        if (row_in) {
            // ---- the cell of row r ----
            const float *c = col + cslot * SLOT;
            Pt<float> s;
            {
                const float C = pc.p, E = pc.e, Wv = pc.w, N = pn.p, Sv = pm.p, NE = pn.e, NW = pn.w, SE = pm.e, SW = pm.w;
                s.dpx = (E - Wv) * Real(1.0 / 3.0) + ((NE + SE) - (NW + SW)) * Real(1.0 / 12.0);
                s.dpy = (N - Sv) * Real(1.0 / 3.0) + ((NE + NW) - (SE + SW)) * Real(1.0 / 12.0);
                s.lap = (Real(4) * ((E + Wv) + (N + Sv)) + ((NE + NW) + (SE + SW)) - Real(20) * C) * Real(1.0 / 6.0);
            }
            float2 nt0 = f2(0.0f);
            nr = cell32<COUPLED>(ph, a, s, c, BW, HO, pc.p, xw, yw, ntf, ntg, nt0, npu, mine && r >= ya && r < yb);
            n0f = nt0.x;
            n0g = nt0.y;
        }
        constexpr int TG = COUPLED ? 5 : 3;   // groups of one row's psi~+
        if (KEEP && row_in) {
            float4 *k = keep + (j & 1) * TG * W;
            k[0] = group32(ntf[0], ntf[1]);
            k[W] = group32(ntf[2], ntf[3]);
            k[2 * W] = group32(f2(n0f, n0g), npu);
            if (COUPLED) {
                k[3 * W] = group32(ntg[0], ntg[1]);
                k[4 * W] = group32(ntg[2], ntg[3]);
            }
        }
        __syncwarp();
        load_row(j + 1 + S::S, cslot);   // the slot of row r is free: every lane has read it
        cslot = cslot + 1 == S::S ? 0 : cslot + 1;
        // ---- the west x-face of row m = r - 1 ----
        float2 wf[4], wg[4];             // the west neighbour's record of row r
        float2 Nf[4], Ng[4];             // west + own sums of row r
        if (row_in) {
#pragma unroll
            for (int p = 0; p < 4; p++) {
                wf[p] = from_west(nr.f[p]);
                Nf[p] = add2(wf[p], nr.f[p]);
                if (COUPLED) {
                    wg[p] = from_west(nr.g[p]);
                    Ng[p] = add2(wg[p], nr.g[p]);
                }
            }
        }
        Flux32 xf, yN;
        const bool finish = j >= 2;      // row m is one of the chunk's own
        if (finish) {
            const bool bottom = WALLY && r - 1 == 0, top = WALLY && r == ny;
            const float ht = (bottom || top) ? 0.5f * ph.h : 0.25f * ph.h;
#pragma unroll
            for (int p = 1; p < 4; p++) {
                if (top) { Nf[p] = P1f[p]; if (COUPLED) Ng[p] = P1g[p]; }
                if (bottom) { P2f[p] = P1f[p]; if (COUPLED) P2g[p] = P1g[p]; }
                Vf[p] = tangent32<1>(Vf[p], Nf[p], P2f[p], ht);   // pairs 1..3: c_t = xi_y of lane 0 = 1
                if (COUPLED) Vg[p] = tangent32<1>(Vg[p], Ng[p], P2g[p], ht);
            }
            float2 u = f2(0.0f);
            if (!COUPLED) {
                const int ym = WALLY ? r - 1 : (r - 1 >= ny ? r - 1 - ny : r - 1);
                if (ph.vel_kind == 4) {
                    const long long kr = (long long)ym * a.pitch + xw, kl = kr - xw + (xw > 0 ? xw - 1 : nx - 1);
                    u.x = a.vel_faces ? a.vel[2 * a.plane + kl] : 0.5f * (a.vel[kl] + a.vel[kr]);
                    u.y = 0.5f * (a.vel[a.plane + kl] + a.vel[a.plane + kr]);
                } else {
                    prescribed_velocity(ph, float(xw), float(ym) + 0.5f, a.t_n + double(ph.h), u.x, u.y);
                }
            }
            xf = face32<COUPLED, true>(ph, Vf, V0, Vg, Vd, Vl, VD, false, u.x, u.y);
        }
        if (row_in) {   // the west x-face of row r, normal part
            Vf[0] = recon32<1>(wf[0], nr.f[0], cp, cm);
            Vf[1] = recon32<1>(wf[1], nr.f[1], cp, cm);
            Vf[2] = recon32<0>(wf[2], nr.f[2], cp, cm);
            Vf[3] = recon32<-1>(wf[3], nr.f[3], cp, cm);
            V0 = 0.5f * (from_west(nr.f0) + nr.f0);
            if (COUPLED) {
                Vg[0] = recon32<1>(wg[0], nr.g[0], cp, cm);
                Vg[1] = recon32<1>(wg[1], nr.g[1], cp, cm);
                Vg[2] = recon32<0>(wg[2], nr.g[2], cp, cm);
                Vg[3] = recon32<-1>(wg[3], nr.g[3], cp, cm);
            }
            Vd = mul2(f2(0.5f), add2(from_west(nr.dp), nr.dp));
            VD = mul2(f2(0.5f), add2(from_west(nr.D), nr.D));
            Vl = 0.5f * (from_west(nr.lap) + nr.lap);
#pragma unroll
            for (int p = 1; p < 4; p++) {
                P2f[p] = P1f[p];
                P1f[p] = Nf[p];
                if (COUPLED) {
                    P2g[p] = P1g[p];
                    P1g[p] = Ng[p];
                }
            }
        }
        // ---- the y-face between rows m and r; with walls also the walls' own faces ----
        if (j >= 1) {
            if (WALLY && r == ny) {
                yN = yTop;
            } else if (!WALLY || r > 0) {
                float2 vf[4], vg[4], ef[4], eg[4], lf[4], lg[4];   // east and west neighbours of row m
#pragma unroll
                for (int p = 0; p < 4; p++) {
                    if (p == 2) continue;
                    ef[p] = from_east(cur.f[p]);
                    lf[p] = from_west(cur.f[p]);
                    if (COUPLED) {
                        eg[p] = from_east(cur.g[p]);
                        lg[p] = from_west(cur.g[p]);
                    }
                }
                const float ht = 0.25f * ph.h;
                vf[0] = tangent32<1>(recon32<0>(cur.f[0], nr.f[0], cp, cm), add2(ef[0], from_east(nr.f[0])), add2(lf[0], wf[0]), ht);
                vf[1] = tangent32<1>(recon32<1>(cur.f[1], nr.f[1], cp, cm), add2(ef[1], from_east(nr.f[1])), add2(lf[1], wf[1]), ht);
                vf[2] = recon32<1>(cur.f[2], nr.f[2], cp, cm);
                vf[3] = tangent32<-1>(recon32<1>(cur.f[3], nr.f[3], cp, cm), add2(ef[3], from_east(nr.f[3])), add2(lf[3], wf[3]), ht);
                float v0 = 0.5f * (cur.f0 + nr.f0);
                if (COUPLED) {
                    vg[0] = tangent32<1>(recon32<0>(cur.g[0], nr.g[0], cp, cm), add2(eg[0], from_east(nr.g[0])), add2(lg[0], wg[0]), ht);
                    vg[1] = tangent32<1>(recon32<1>(cur.g[1], nr.g[1], cp, cm), add2(eg[1], from_east(nr.g[1])), add2(lg[1], wg[1]), ht);
                    vg[2] = recon32<1>(cur.g[2], nr.g[2], cp, cm);
                    vg[3] = tangent32<-1>(recon32<1>(cur.g[3], nr.g[3], cp, cm), add2(eg[3], from_east(nr.g[3])), add2(lg[3], wg[3]), ht);
                }
                const float2 md = mul2(f2(0.5f), add2(cur.dp, nr.dp)), mD = mul2(f2(0.5f), add2(cur.D, nr.D));
                float2 u = f2(0.0f);
                if (!COUPLED) {
                    if (ph.vel_kind == 4) {
                        const int yd = yw > 0 ? yw - 1 : ny - 1;
                        const long long kd = (long long)yd * a.pitch + xw, ku = (long long)yw * a.pitch + xw;
                        u.x = 0.5f * (a.vel[kd] + a.vel[ku]);
                        u.y = a.vel_faces ? a.vel[3 * a.plane + ku] : 0.5f * (a.vel[a.plane + kd] + a.vel[a.plane + ku]);
                    } else {
                        prescribed_velocity(ph, float(xw) + 0.5f, float(yw), a.t_n + double(ph.h), u.x, u.y);
                    }
                }
                yN = face32<COUPLED, false>(ph, vf, v0, vg, md, 0.5f * (cur.lap + nr.lap), mD, false, u.x, u.y);
                if (WALLY && r - 1 == 0 && j >= 2) {   // the bottom wall, below row m
                    float rest = 0.0f;
                    wall32<false>(cur.f, ef, lf, nr.f, cur.f0, nr.f0, true, ph.h, vf, v0);
                    if (COUPLED) wall32<false>(cur.g, eg, lg, nr.g, 0.0f, 0.0f, false, ph.h, vg, rest);
                    yS = face32<COUPLED, false>(ph, vf, v0, vg, f2(cur.dp.x, 0.0f), cur.lap, f2(cur.D.x, 0.0f), true, 0.0f, 0.0f);
                }
                if (WALLY && r == ny - 1) {            // the top wall, above row r
                    float rest = 0.0f;
#pragma unroll
                    for (int p = 0; p < 4; p++) {
                        if (p == 2) continue;
                        ef[p] = from_east(nr.f[p]);
                        if (COUPLED) eg[p] = from_east(nr.g[p]);
                    }
                    wall32<true>(nr.f, ef, wf, cur.f, nr.f0, cur.f0, true, ph.h, vf, v0);
                    if (COUPLED) wall32<true>(nr.g, eg, wg, cur.g, 0.0f, 0.0f, false, ph.h, vg, rest);
                    yTop = face32<COUPLED, false>(ph, vf, v0, vg, f2(nr.dp.x, 0.0f), nr.lap, f2(nr.D.x, 0.0f), true, 0.0f, 0.0f);
                }
            }
        }
        if (finish) {
            // ---- the flux update of row m ----
            Flux32 xe;
#pragma unroll
            for (int i = 0; i < 3; i++) {
                xe.f[i] = from_east(xf.f[i]);
                if (COUPLED) xe.g[i] = from_east(xf.g[i]);
            }
            if (KEEP) {
                const float4 *k = keep + ((j - 1) & 1) * TG * W;
                float2 t0;
                ungroup32(k[0], tf[0], tf[1]);
                ungroup32(k[W], tf[2], tf[3]);
                ungroup32(k[2 * W], t0, pu);
                t0f = t0.x;
                t0g = t0.y;
                if (COUPLED) {
                    ungroup32(k[3 * W], tg[0], tg[1]);
                    ungroup32(k[4 * W], tg[2], tg[3]);
                }
                k = keep + 2 * TG * W;
                float2 unused;
                ungroup32(k[0], yS.f[0], yS.f[1]);
                ungroup32(k[W], yS.f[2], COUPLED ? yS.g[0] : unused);
                if (COUPLED) ungroup32(k[2 * W], yS.g[1], yS.g[2]);
            }
            flux32<COUPLED, true>(ph.dt, xf, xe, tf, tg);
            flux32<COUPLED, false>(ph.dt, yS, yN, tf, tg);
            tma_store_wait_read();   // (only the issuing lane has any)
            __syncwarp();
            if (inner) {
                float *o = sout + tid - S::HX;
                o[0] = t0f;
                if (COUPLED) o[9 * OW] = t0g;
#pragma unroll
                for (int p = 0; p < 4; p++) {
                    o[(1 + p) * OW] = tf[p].x;
                    o[(5 + p) * OW] = tf[p].y;
                    if (COUPLED) {
                        o[(10 + p) * OW] = tg[p].x;
                        o[(14 + p) * OW] = tg[p].y;
                    }
                }
                o[S::out_hist(W)] = pu.x;
                o[S::out_hist(W) + OW] = pu.y;
                fence_proxy_async_smem();
            }
        }
        if (KEEP) {
            if (j >= 1) {
                float4 *k = keep + 2 * TG * W;
                k[0] = group32(yN.f[0], yN.f[1]);
                k[W] = group32(yN.f[2], COUPLED ? yN.g[0] : f2(0.0f));
                if (COUPLED) k[2 * W] = group32(yN.g[1], yN.g[2]);
            }
        } else {
            yS = yN;
#pragma unroll
            for (int p = 0; p < 4; p++) {
                tf[p] = ntf[p];
                tg[p] = ntg[p];
            }
            t0f = n0f;
            t0g = n0g;
            pu = npu;
        }
        cur = nr;
        pm = pc;
        pc = pn;
    }
    __syncwarp();
    tma_store_row(tid == 0 && alive, sout, &tm.dst_state, sout + S::out_hist(W), &tm.dst_hist, x0, yb - 1);
    tma_store_wait();
    if (!alive)   // let copies in flight land before the CTA's shared memory is given away
        for (int s = 0; s < S::S; s++) mbar_wait(bar + s, (uint32_t)((nrows - 1 - s) / S::S) & 1u, kPollLimit);
}

// The constants a march reads.
template <typename Real> struct StripConst;
template <> struct StripConst<float> { using T = Phys<float>; };
template <> struct StripConst<double> { using T = StripPhys<double>; };
template <bool COUPLED, bool WALLY>
__device__ __forceinline__ void strip_run(const StripMaps &tm, const StepArgs<float> &a, const Phys<float> &ph,
                                          const Phys<float> &, int x0, int ya, int yb) {
    strip_march32<COUPLED, WALLY>(tm, a, ph, x0, ya, yb);
}
template <bool COUPLED, bool WALLY>
__device__ __forceinline__ void strip_run(const StripMaps &tm, const StepArgs<double> &a, const StripPhys<double> &ph,
                                          const Phys<double> &pv, int x0, int ya, int yb) {
    strip_march<double, COUPLED, WALLY>(tm, a, ph, pv, x0, ya, yb);
}

template <typename Real, bool COUPLED, bool WALLY>
__global__ void __launch_bounds__(kStripLanes, (strip_ctas<Real, WALLY>()))
strip_step_kernel(const __grid_constant__ StripMaps tm, const __grid_constant__ StepArgs<Real> a,
                  const __grid_constant__ typename StripConst<Real>::T ph, const __grid_constant__ Phys<Real> pv,
                  const __grid_constant__ StripArgs g) {
    using S = StripShape<Real, COUPLED, strip_shuffles<Real, WALLY>(), strip_keeps<Real, WALLY>()>;
    const int strip = (int)blockIdx.x % g.nstrips, chunk = (int)blockIdx.x / g.nstrips;
    const int ya = chunk * g.rows;
    strip_run<COUPLED, WALLY>(tm, a, ph, pv, strip * S::own(kStripLanes), ya, min(ya + g.rows, a.ny));
}

// ---- several problems in one launch ----

// One member of a batch: its buffers and where it stands (advanced on the device after a run of steps).
template <typename Real>
struct StripInst {
    StripMaps maps[2];         // of a step from buffer 0 or 1
    Real *state[2], *hist[2];
    const Real *vel;
    unsigned *status;
    Phys<Real> pv;             // the prescribed velocity's constants
    long long plane, steps;
    int nx, ny, pitch, nstrips, vel_faces, cur;
};

// The members of one launch, in parameter space: the constants are read as uniform operands, like those of the
// single-problem kernel.
constexpr int kStripMembers = 64;
template <typename Real>
struct StripGroup {
    const StripInst<Real> *inst;
    int n, rows, step;                  // members; rows of a chunk; steps since the descriptors were advanced
    int first[kStripMembers + 1];       // first CTA of each member
    typename StripConst<Real>::T ph[kStripMembers];
};

template <typename Real, bool COUPLED, bool WALLY>
__global__ void __launch_bounds__(kStripLanes, (strip_ctas<Real, WALLY>()))
strip_batch_kernel(const __grid_constant__ StripGroup<Real> g) {
    using S = StripShape<Real, COUPLED, strip_shuffles<Real, WALLY>(), strip_keeps<Real, WALLY>()>;
    const int b = (int)blockIdx.x;
    int lo = 0, hi = g.n;   // the member whose CTAs hold b
    while (hi - lo > 1) {
        const int mid = (lo + hi) >> 1;
        if (b >= g.first[mid]) lo = mid;
        else hi = mid;
    }
    const StripInst<Real> &d = g.inst[lo];
    const int i = b - g.first[lo];
    const int cur = d.cur ^ (g.step & 1);
    const long long steps = d.steps + g.step;
    StepArgs<Real> a;
    a.src = d.state[cur];
    a.hsrc = d.hist[cur];
    a.dst = d.state[cur ^ 1];
    a.hdst = d.hist[cur ^ 1];
    a.nx = d.nx;
    a.ny = d.ny;
    a.pitch = d.pitch;
    a.plane = d.plane;
    a.first_step = steps == 0;
    a.t_n = double(steps) * double(g.ph[lo].dt);
    a.small = 0;
    a.use_tma = 1;
    a.vel = d.vel;
    a.vel_faces = d.vel_faces;
    a.status = d.status;
    const int strip = i % d.nstrips, ya = (i / d.nstrips) * g.rows;
    strip_run<COUPLED, WALLY>(d.maps[cur], a, g.ph[lo], d.pv, strip * S::own(kStripLanes), ya, min(ya + g.rows, a.ny));
}

// After k steps: buffers swap k times, step counts grow by k.
template <typename Real>
__global__ void strip_advance_kernel(StripInst<Real> *inst, int n, int k) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) {
        inst[i].cur ^= (k & 1);
        inst[i].steps += k;
    }
}

}  // namespace dugks

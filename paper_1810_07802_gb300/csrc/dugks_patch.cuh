// dugks_patch.cuh -- the FP64 step kernel of small grids, of the coupled model between walls and of the upwind
// reconstruction: one CTA per rectangle of cells.
//
// The FP64 pipe of an SM takes 16 cycles per warp instruction, whichever warps they come from, so a step lasts as
// long as the SM with the most of them.  A grid of a few thousand cells is cut into rectangles of a size chosen for
// it (patch_plan), one or a few per SM; each CTA forms its cell records with a one-cell halo (upwind: two), then every face, then
// the update, its warps taking 32 cells or faces at a time.  x- and y-faces are the same code: the scheme is
// unchanged by exchanging the axes, so a y-face takes its neighbours along the other axis and the directions by
// their normal and tangential components, and no warp holds two kinds of work.
//
// Measured, tile kernel -> rectangles: central 64^2 57.5 -> 21.1 us a step, 128^2 57.5 -> 35.7, channel 4 x 200
// 59.5 -> 23.1, Allen-Cahn 256^2 84 -> 55; upwind 64^2 110 -> 33, 128^2 111 -> 62, 300 x 200 375 -> 206, 1024^2
// 4,939 -> 3,698, 256 x 1024 between walls 936 -> 925; coupled central between walls, strips -> rectangles: 380^2 382 ->
// 255 (tiles 371), 1024^2 2,211 -> 1,844, 3000 x 200 1,453 -> 1,023.
#pragma once

#include "dugks_strip.cuh"

namespace dugks {

constexpr int kPatchThreads = 256;

// van Leer's limiter of two one-sided differences (R14).
__device__ __forceinline__ double limited64(double a, double b) {
    const double p = a * b;
    return p > 0.0 ? (p + p) * rcp_s(a + b) : 0.0;
}

struct PatchArgs {
    int tx, ty, tiles_x;   // cells of a rectangle, rectangles across
};

// Shared memory of a rectangle, in doubles: phi', record planes, flux planes, psi~+ of the own cells.
template <bool COUPLED, bool UPW>
struct PatchShape {
    static constexpr int H = UPW ? 2 : 1;          // record halo
    static constexpr int NR = COUPLED ? 22 : 13;   // f0, f1..f8, Gx, Gy, Ex, Ey; g1..g8, L
    static constexpr int NF = COUPLED ? 12 : 6;
    static constexpr int NT = COUPLED ? 16 : 8;
    __host__ __device__ static int phis(int tx, int ty) { return (tx + 2 * H + 2) * (ty + 2 * H + 2); }
    __host__ __device__ static int cells(int tx, int ty) { return (tx + 2 * H) * (ty + 2 * H); }
    __host__ __device__ static int faces(int tx, int ty) { return (tx + 1) * ty + tx * (ty + 1); }
    __host__ __device__ static size_t smem_bytes(int tx, int ty) {
        return sizeof(double) * ((size_t)phis(tx, ty) + (size_t)NR * cells(tx, ty) + (size_t)NF * faces(tx, ty) +
                                 (size_t)NT * tx * ty);
    }
};

template <bool COUPLED, bool WALLY, bool UPW>
__global__ void __launch_bounds__(kPatchThreads, 1)
patch_step_kernel(const __grid_constant__ StepArgs<double> a, const __grid_constant__ StripPhys<double> ph,
                  const __grid_constant__ Phys<double> pv, const __grid_constant__ PatchArgs g) {
    using P = PatchShape<COUPLED, UPW>;
    constexpr int H = P::H;
    using V = double2;
    extern __shared__ __align__(128) unsigned char smem_raw[];
    const int tx = g.tx, ty = g.ty, nx = a.nx, ny = a.ny, tid = threadIdx.x;
    const int x0 = ((int)blockIdx.x % g.tiles_x) * tx, y0 = ((int)blockIdx.x / g.tiles_x) * ty;
    const int wx = tx + 2 * H + 2, cxn = tx + 2 * H, ncell = P::cells(tx, ty), nface = P::faces(tx, ty), nfx = (tx + 1) * ty;
    double *sphi = reinterpret_cast<double *>(smem_raw);
    double *rec = sphi + P::phis(tx, ty);
    double *flux = rec + (size_t)P::NR * ncell;
    double *plus = flux + (size_t)P::NF * nface;
    const int R_G = 9 * ncell, R_E = 11 * ncell, R_g = 13 * ncell - ncell, R_L = 21 * ncell;   // R_g + k: g_k, k >= 1
    auto column = [&](int x) {
        x %= nx;
        return x < 0 ? x + nx : x;
    };

    grid_launch_dependents();
    grid_dependency_wait();
    // 1. phi', one cell beyond the records
    for (int i = tid; i < P::phis(tx, ty); i += kPatchThreads) {
        const int iy = i / wx, gx = column(x0 - H - 1 + i - iy * wx), gy = map_row<WALLY>(y0 - H - 1 + iy, ny);
        if (!in_bounds(gx >= 0 && gx < nx && gy >= 0 && gy < ny, a.status)) continue;
        const double *c = a.src + ((long long)gy * a.pitch + gx);
        double v[9];
#pragma unroll
        for (int k = 0; k < 9; k++) v[k] = c[k * a.plane];
        sphi[i] = (((v[2] + v[4]) + (v[6] + v[8])) + ((v[1] + v[3]) + (v[5] + v[7]))) + v[0];
    }
    __syncthreads();
    // 2. the cells with the record halo
    for (int i = tid; i < ncell; i += kPatchThreads) {
        const int iy = i / cxn, ix = i - iy * cxn;
        const int x = x0 - H + ix, y = y0 - H + iy;
        if (WALLY && (y < 0 || y >= ny)) continue;   // beyond a wall: no face reads it
        const int gx = column(x), gy = WALLY ? y : map_row<false>(y, ny);
        if (!in_bounds(gx >= 0 && gx < nx && gy >= 0 && gy < ny, a.status)) continue;
        const long long o = (long long)gy * a.pitch + gx;
        const double *c = a.src + o;
        auto pair = [&](int k, int l) { return v2(c[k * a.plane], c[l * a.plane]); };
        Dirs<double> df, dg;
        df.A = pair(1, 3); df.B = pair(5, 7); df.C = pair(2, 4); df.D = pair(6, 8);
        double d0g = 0.0;
        if constexpr (COUPLED) {
            dg.A = pair(10, 12); dg.B = pair(14, 16); dg.C = pair(11, 13); dg.D = pair(15, 17);
            d0g = c[9 * a.plane];
        }
        const V h = v2(a.hsrc[o], a.hsrc[a.plane + o]);
        const double *p = sphi + (iy + 1) * wx + ix + 1;
        PhiRow<double> m, z, n;
        auto row = [&](const double *q, PhiRow<double> &r) {
            r.p = q[0];
            r.d = q[1] - q[-1];
            r.s = q[1] + q[-1];
        };
        row(p - wx, m);
        row(p, z);
        row(p + wx, n);
        V u = v2(0.0);
        if constexpr (!COUPLED) {
            if (ph.vel_kind == 0) u = v2(ph.u0x, ph.u0y);
            else if (ph.vel_kind == 4) u = v2(a.vel[o], a.vel[a.plane + o]);
            else u = strip_velocity<double, COUPLED>(a, pv, double(gx) + 0.5, double(gy) + 0.5, a.t_n);
        }
        CellRec<double, COUPLED> nr;
        Dirs<double> tf, tg;
        double t0f, t0g = 0.0;
        V pu;
        const unsigned bad = strip_cell<double, COUPLED>(ph, m, z, n, df, c[0], dg, d0g, h, a.first_step != 0, u, nr, tf, tg,
                                                         t0f, t0g, pu);
        double *r = rec + i;
        r[0] = nr.f0;
        r[1 * ncell] = nr.f.A.x; r[3 * ncell] = nr.f.A.y; r[5 * ncell] = nr.f.B.x; r[7 * ncell] = nr.f.B.y;
        r[2 * ncell] = nr.f.C.x; r[4 * ncell] = nr.f.C.y; r[6 * ncell] = nr.f.D.x; r[8 * ncell] = nr.f.D.y;
        r[R_G] = nr.G.x; r[R_G + ncell] = nr.G.y;
        r[R_E] = nr.E.x; r[R_E + ncell] = nr.E.y;
        if constexpr (COUPLED) {
            double *q = r + R_g;
            q[1 * ncell] = nr.g.A.x; q[3 * ncell] = nr.g.A.y; q[5 * ncell] = nr.g.B.x; q[7 * ncell] = nr.g.B.y;
            q[2 * ncell] = nr.g.C.x; q[4 * ncell] = nr.g.C.y; q[6 * ncell] = nr.g.D.x; q[8 * ncell] = nr.g.D.y;
            r[R_L] = nr.L;
        }
        if (ix >= H && ix < tx + H && iy >= H && iy < ty + H && x < nx && y < ny) {
            const int own = tx * ty;
            double *t = plus + (iy - H) * tx + ix - H;
            t[0] = tf.A.x; t[own] = tf.A.y; t[2 * own] = tf.B.x; t[3 * own] = tf.B.y;
            t[4 * own] = tf.C.x; t[5 * own] = tf.C.y; t[6 * own] = tf.D.x; t[7 * own] = tf.D.y;
            if constexpr (COUPLED) {
                t += 8 * own;
                t[0] = tg.A.x; t[own] = tg.A.y; t[2 * own] = tg.B.x; t[3 * own] = tg.B.y;
                t[4 * own] = tg.C.x; t[5 * own] = tg.C.y; t[6 * own] = tg.D.x; t[7 * own] = tg.D.y;
                a.dst[9 * a.plane + o] = t0g;
            }
            a.dst[o] = t0f;
            a.hdst[o] = pu.x;
            a.hdst[a.plane + o] = pu.y;
            if (bad) atomicOr(a.status, bad);
        }
    }
    __syncthreads();
    // 3. the faces: n the normal, t the tangent; cells L (at -n) and R (at +n)
    for (int i = tid; i < nface; i += kPatchThreads) {
        const bool xf = i < nfx;
        const int j = xf ? i : i - nfx, w = xf ? tx + 1 : tx;
        const int fy = j / w, fx = j - fy * w;
        const int ns = xf ? 1 : cxn, ts = xf ? cxn : 1;
        const int L = xf ? (fy + H) * cxn + fx + H - 1 : (fy + H - 1) * cxn + fx + H;
        const int x = x0 + fx, y = y0 + fy;   // the cell at +n
        if ((xf ? y >= ny : x >= nx) || (xf ? x - 1 >= nx : y - 1 >= ny)) continue;
        const bool bottom = WALLY && !xf && y == 0, top = WALLY && !xf && y == ny;
        // planes by component: A (n+, t+), B (n-, t-), C ((n+,t+), (n-,t+)), D ((n-,t-), (n+,t-))
        const int kn = xf ? 1 : 3, kt = xf ? 3 : 1, kc = xf ? 4 : 8, kd = xf ? 8 : 4;
        auto get = [&](const double *q) {
            Dirs<double> d;
            d.A = v2(q[kn * ncell], q[kt * ncell]);
            d.B = v2(q[(kn + 4) * ncell], q[(kt + 4) * ncell]);
            d.C = v2(q[2 * ncell], q[kc * ncell]);
            d.D = v2(q[6 * ncell], q[kd * ncell]);
            return d;
        };
        auto sum = [&](const double *q) {   // over the two cells of the face
            Dirs<double> u = get(q), v = get(q + ns);
            u.A = vadd(u.A, v.A); u.B = vadd(u.B, v.B); u.C = vadd(u.C, v.C); u.D = vadd(u.D, v.D);
            return u;
        };
        auto vec = [&](const double *q) { return xf ? v2(q[0], q[ncell]) : v2(q[ncell], q[0]); };
        Dirs<double> fb, gb;
        FaceSum<double> m;
        const bool wall = bottom || top;
        if (wall) {
            const int c0 = top ? L : L + ns, into = top ? -ns : ns;
            const double *r = rec + c0;
            const double s = top ? 1.0 : -1.0, h = ph.h;
            // the value at x_w - xi h of a direction with components (cn, ct)
            auto at = [&](const double *q, int cn, int ct) {
                const double b0 = q[0], sn = s * (b0 - q[into]);
                double v = b0 + (0.5 * s - h * cn) * sn;
                if (ct) v -= h * ct * (UPW ? limited64(b0 - q[-ts], q[ts] - b0) : 0.5 * (q[ts] - q[-ts]));
                return v;
            };
            auto bars = [&](const double *q) {
                Dirs<double> d;
                d.A.y = at(q + kt * ncell, 0, 1);
                d.B.y = at(q + (kt + 4) * ncell, 0, -1);
                if (top) {
                    d.A.x = at(q + kn * ncell, 1, 0);
                    d.C.x = at(q + 2 * ncell, 1, 1);
                    d.D.y = at(q + kd * ncell, 1, -1);
                    d.B.x = d.A.x; d.D.x = d.C.x; d.C.y = d.D.y;
                } else {
                    d.B.x = at(q + (kn + 4) * ncell, -1, 0);
                    d.D.x = at(q + 6 * ncell, -1, -1);
                    d.C.y = at(q + kc * ncell, -1, 1);
                    d.A.x = d.B.x; d.C.x = d.D.x; d.D.y = d.C.y;
                }
                return d;
            };
            fb = bars(r);
            m.f0 = 2.0 * at(r, 0, 0);
            m.G = v2(0.0, 2.0 * r[R_G]);   // no normal component; the tangent is x
            m.E = v2(0.0, 2.0 * r[R_E]);
            m.L = 0.0;
            if constexpr (COUPLED) {
                gb = bars(r + R_g);
                m.L = 2.0 * r[R_L];
            }
        } else {
            const double *r = rec + L;
            const bool lo = WALLY && xf && y == 0, hi = WALLY && xf && y == ny - 1;
            if constexpr (UPW) {
                // next to a wall a slope across it is the one-sided difference into the fluid: along an x-face's
                // tangent (both cells), along a y-face's normal (the cell next to the wall)
                const bool wl = WALLY && !xf && y - 1 == 0, wr = WALLY && !xf && y == ny - 1;
                const double h = ph.h;
                // the profile of the cell at q, on side s (-1: R, +1: L) of the face, at x_f - xi h
                auto profile = [&](const double *q, int s, int cn, int ct) {
                    const double c = q[0];
                    const double sn = (s > 0 ? wl : wr) ? (s > 0 ? q[ns] - c : c - q[-ns]) : limited64(c - q[-ns], q[ns] - c);
                    double v = c + sn * (0.5 * s - h * cn);
                    if (ct) v -= h * ct * (lo ? q[ts] - c : hi ? c - q[-ts] : limited64(c - q[-ts], q[ts] - c));
                    return v;
                };
                auto along = [&](const double *q, int ct) { return 0.5 * (profile(q, 1, 0, ct) + profile(q + ns, -1, 0, ct)); };
                auto bars = [&](const double *q) {
                    Dirs<double> d;
                    d.A = v2(profile(q + kn * ncell, 1, 1, 0), along(q + kt * ncell, 1));
                    d.B = v2(profile(q + (kn + 4) * ncell + ns, -1, -1, 0), along(q + (kt + 4) * ncell, -1));
                    d.C = v2(profile(q + 2 * ncell, 1, 1, 1), profile(q + kc * ncell + ns, -1, -1, 1));
                    d.D = v2(profile(q + 6 * ncell + ns, -1, -1, -1), profile(q + kd * ncell, 1, 1, -1));
                    return d;
                };
                fb = bars(r);
                m.f0 = 2.0 * along(r, 0);
                if constexpr (COUPLED) gb = bars(r + R_g);
            } else {
                const double ht = (lo || hi) ? 2.0 * ph.ht : ph.ht;
                const int up = hi ? 0 : ts, down = lo ? 0 : ts;
                fb = strip_x_open(ph, sum(r), get(r + ns), sum(r - down), ht);
                strip_x_close(fb, sum(r + up), ht);
                m.f0 = r[0] + r[ns];
                if constexpr (COUPLED) {
                    const double *q = r + R_g;
                    gb = strip_x_open(ph, sum(q), get(q + ns), sum(q - down), ht);
                    strip_x_close(gb, sum(q + up), ht);
                }
            }
            m.G = vadd(vec(r + R_G), vec(r + R_G + ns));
            m.E = vadd(vec(r + R_E), vec(r + R_E + ns));
            m.L = COUPLED ? r[R_L] + r[R_L + ns] : 0.0;
        }
        V uf = v2(0.0);
        if constexpr (!COUPLED) {
            const int gx = column(x), gy = WALLY ? y : map_row<false>(y, ny);
            if (wall) {
            } else if (ph.vel_kind == 4) {
                const int gl = xf ? column(x - 1) : gx, gd = xf ? gy : (gy > 0 ? gy - 1 : ny - 1);
                const long long kl = (long long)gd * a.pitch + gl, kr = (long long)gy * a.pitch + gx;
                const V mean = v2(0.5 * (a.vel[kl] + a.vel[kr]), 0.5 * (a.vel[a.plane + kl] + a.vel[a.plane + kr]));
                if (xf) uf = v2(a.vel_faces ? a.vel[2 * a.plane + kl] : mean.x, mean.y);
                else uf = v2(a.vel_faces ? a.vel[3 * a.plane + kr] : mean.y, mean.x);
            } else {
                const V u = strip_velocity<double, COUPLED>(a, pv, double(gx) + (xf ? 0.0 : 0.5), double(gy) + (xf ? 0.5 : 0.0),
                                                            a.t_n + double(pv.h));
                uf = xf ? u : v2(u.y, u.x);
            }
        }
        const Flux<double> o = strip_face<double, COUPLED, true>(ph, fb, gb, m, wall, uf, !xf);
        double *q = flux + i;
        q[0] = o.fC.x; q[nface] = o.fC.y; q[2 * nface] = o.fD.x; q[3 * nface] = o.fD.y;
        q[4 * nface] = o.fn.x; q[5 * nface] = o.fn.y;
        if constexpr (COUPLED) {
            q += 6 * nface;
            q[0] = o.gC.x; q[nface] = o.gC.y; q[2 * nface] = o.gD.x; q[3 * nface] = o.gD.y;
            q[4 * nface] = o.gn.x; q[5 * nface] = o.gn.y;
        }
    }
    __syncthreads();
    // 4. the flux update
    for (int i = tid; i < tx * ty; i += kPatchThreads) {
        const int iy = i / tx, ix = i - iy * tx, x = x0 + ix, y = y0 + iy, own = tx * ty;
        if (x >= nx || y >= ny || !in_bounds(x >= 0 && y >= 0, a.status)) continue;
        const double *fw = flux + iy * (tx + 1) + ix, *fs = flux + nfx + i;
        const double dt = ph.dt;
#pragma unroll
        for (int md = 0; md < (COUPLED ? 2 : 1); md++) {
            const double *t = plus + md * 8 * own + i;
            const double *w = fw + md * 6 * nface, *s = fs + md * 6 * nface;
            double *d = a.dst + (md * 9 * a.plane + (long long)y * a.pitch + x);
            auto dx = [&](int k) { return w[k * nface] - w[k * nface + 1]; };
            auto dy = [&](int k) { return s[k * nface] - s[k * nface + tx]; };
            d[1 * a.plane] = t[0] + dt * dx(4);
            d[3 * a.plane] = t[own] + dt * dy(4);
            d[5 * a.plane] = t[2 * own] - dt * dx(5);
            d[7 * a.plane] = t[3 * own] - dt * dy(5);
            d[2 * a.plane] = (t[4 * own] + dt * dx(0)) + dt * dy(0);
            d[4 * a.plane] = (t[5 * own] - dt * dx(1)) + dt * dy(3);
            d[6 * a.plane] = (t[6 * own] - dt * dx(2)) - dt * dy(2);
            d[8 * a.plane] = (t[7 * own] + dt * dx(3)) - dt * dy(1);
        }
    }
}

}  // namespace dugks

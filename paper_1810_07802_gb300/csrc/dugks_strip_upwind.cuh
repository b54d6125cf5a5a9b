// dugks_strip_upwind.cuh -- the FP32 step kernel of the upwind reconstruction: the march of dugks_strip.cuh with
// van Leer-limited slopes.
//
// A cell's two slopes per direction (its limited x- and y-differences) serve every face around it, so they are formed
// once per cell: the value a direction carries to the face it leaves by is then the cell's own, and a face takes
// one value from each side.  The tile kernel forms four slopes per direction and face.  The operations are the tile
// kernel's, lane for lane, as in the central march.  26 of a strip's 32 columns are its own (records reach two cells
// from a face); rows leave by plain stores, 26 columns being no multiple of 16 bytes.
#pragma once

#include "dugks_strip.cuh"

namespace dugks {

// Slopes of every direction of one cell along one axis: pairs of f and g, the rest direction of f.
struct Slope32 {
    float2 f[4], g[4];
    float f0;
};
__device__ __forceinline__ float2 limited32(float2 c, float2 lo, float2 hi) { return van_leer2(sub2(c, lo), sub2(hi, c)); }
__device__ __forceinline__ float limited32(float c, float lo, float hi) { return van_leer(c - lo, hi - c); }
// c + sn (normal offsets a of lane 0, b of lane 1)
__device__ __forceinline__ float2 leave32(float2 c, float2 sn, float a, float b) { return fma2(sn, f2(a, b), c); }
// - h c_t s_t, lane 0 with c_t = C
template <int C>
__device__ __forceinline__ float2 drift32(float2 v, float2 st, float h) {
    return fma2(C > 0 ? f2(-h, h) : f2(h, -h), st, v);
}

// Values of one model's pairs at the faces of an axis: v the crossing pairs (each lane at the face its direction
// leaves by), lo and hi the pair along the faces, seen from the cell on the high and on the low side of it.
struct Leave32 {
    float2 v[3], lo, hi;
};
// XAXIS: crossing pairs 1, 2, 4, along 3; else crossing 2, 3, 4, along 1.
template <bool XAXIS>
__device__ __forceinline__ Leave32 leave_all32(const float2 c[4], const float2 n[4], const float2 t[4], float h) {
    const float a = 0.5f - h, b = h - 0.5f;
    Leave32 o;
    if (XAXIS) {
        o.v[0] = leave32(c[0], n[0], a, b);
        o.v[1] = drift32<1>(leave32(c[1], n[1], a, b), t[1], h);
        o.v[2] = drift32<1>(leave32(c[3], n[3], b, a), t[3], h);
        o.hi = drift32<1>(leave32(c[2], n[2], 0.5f, 0.5f), t[2], h);
        o.lo = drift32<1>(leave32(c[2], n[2], -0.5f, -0.5f), t[2], h);
    } else {
        o.v[0] = drift32<1>(leave32(c[1], n[1], a, b), t[1], h);
        o.v[1] = leave32(c[2], n[2], a, b);
        o.v[2] = drift32<-1>(leave32(c[3], n[3], a, b), t[3], h);
        o.hi = drift32<1>(leave32(c[0], n[0], 0.5f, 0.5f), t[0], h);
        o.lo = drift32<1>(leave32(c[0], n[0], -0.5f, -0.5f), t[0], h);
    }
    return o;
}

// A wall face (R17): the cell's own profile for directions leaving the fluid or running along the wall,
// bounce-back for the rest.
template <bool TOP>
__device__ __forceinline__ void wall_upwind32(const float2 c[4], const float2 sx[4], const float2 sy[4], float h,
                                              float2 o[4]) {
    const float dyw = TOP ? 0.5f : -0.5f;
    float C[9], X[9], Y[9], out[9];
    unpack32(c, C);
    unpack32(sx, X);
    unpack32(sy, Y);
#pragma unroll
    for (int k = 1; k < 9; k++) {
        const bool keep = TOP ? (cy(k) >= 0) : (cy(k) <= 0);
        if (!keep) continue;
        float v = C[k] + (cy(k) == 0 ? dyw : (cy(k) > 0 ? dyw - h : dyw + h)) * Y[k];
        if (cx(k) != 0) v -= h * sgnmul(cx(k), X[k]);
        out[k] = v;
    }
#pragma unroll
    for (int k = 1; k < 9; k++) {
        const bool enters = TOP ? (cy(k) < 0) : (cy(k) > 0);
        if (enters) out[k] = out[opp(k)];
    }
#pragma unroll
    for (int p = 0; p < 4; p++) o[p] = f2(out[1 + p], out[5 + p]);
}

constexpr int kUpwindOwn = 26;   // a strip's own columns
template <bool COUPLED>
struct UpwindShape {
    static constexpr int HX = 3, S = 4, NQ = COUPLED ? 18 : 9, BW = kStripLanes + 4;
    static constexpr int HO = (NQ * BW + 31) / 32 * 32, SLOT = HO + (2 * BW + 31) / 32 * 32;
    static constexpr size_t smem_bytes = size_t(S) * SLOT * sizeof(float) + S * 8 + 128;
};

template <bool COUPLED, bool WALLY>
__global__ void __launch_bounds__(kStripLanes, kStripCtas)
strip_upwind_kernel(const __grid_constant__ StripMaps tm, const __grid_constant__ StepArgs<float> a,
                    const __grid_constant__ Phys<float> ph, const __grid_constant__ StripArgs ga) {
    using Real = float;
    using S = UpwindShape<COUPLED>;
    extern __shared__ __align__(128) unsigned char smem_raw[];
    float *ring = reinterpret_cast<float *>(smem_raw + ((128u - (smem_u32(smem_raw) & 127u)) & 127u));
    uint64_t *bar = reinterpret_cast<uint64_t *>(ring + S::S * S::SLOT);
    constexpr int BW = S::BW, HO = S::HO;
    const int tid = threadIdx.x;
    const int x0 = ((int)blockIdx.x % ga.nstrips) * kUpwindOwn, ya = ((int)blockIdx.x / ga.nstrips) * ga.rows;
    const int nx = a.nx, ny = a.ny, yb = min(ya + ga.rows, ny);
    const int x = x0 - S::HX + tid;
    const int xend = min(x0 + kUpwindOwn, nx);
    const bool mine = tid >= S::HX && x < xend;
    int xw = x % nx;
    if (xw < 0) xw += nx;
    const int nrows = yb - ya + 2 * S::HX;   // staged rows: y = ya - HX + k
    const int xs = (x0 - S::HX) & ~3;        // a TMA load starts on 16 bytes
    const int shift = x0 - S::HX - xs;

    grid_launch_dependents();
    grid_dependency_wait();
    // staging: TMA when every column needed lies inside the domain, else one cp.async per value
    const bool tma = x0 >= S::HX && xend + S::HX <= nx && !(*((volatile unsigned *)a.status) & STATUS_TIMEOUT);
    bool alive = true;
    if (tid == 0) {
        for (int s = 0; s < S::S; s++) mbar_init(bar + s, tma ? 1u : (uint32_t)kStripLanes);
    }
    __syncwarp();
    auto row_of = [&](int k) {   // staged row k of the domain: at most HX rows outside
        const int y = ya - S::HX + k;
        return map_row<WALLY>(y, ny);
    };
    auto load_row = [&](int k, int slot) {
        if (k >= nrows) return;
        float *dst = ring + slot * S::SLOT;
        uint64_t *b = bar + slot;
        const int y = row_of(k);
        if (tma) {
            tma_load_row(tid == 0, b, (uint32_t)((S::NQ + 2) * BW * sizeof(float)), dst, &tm.src_state, dst + HO,
                         &tm.src_hist, xs, y);
        } else {
            const long long g = (long long)y * a.pitch + xw;
            float *d = dst + tid + shift;
            if (in_bounds(xw >= 0 && xw < nx && y >= 0 && y < ny, a.status)) {
                for (int q = 0; q < S::NQ; q++) cp_async_elt(d + q * BW, a.src + q * a.plane + g);
                cp_async_elt(d + HO, a.hsrc + g);
                cp_async_elt(d + HO + BW, a.hsrc + a.plane + g);
            }
            cp_async_arrive(b);
        }
    };
    for (int k = 0; k < S::S; k++) load_row(k, k);

    const float *col = ring + tid + shift;
    int slot = 0;
    uint32_t parity = 0;
    struct Phi { float p, e, w; };
    auto phi_row = [&]() {
        if (!mbar_wait(bar + slot, parity, alive ? kPollLimit : 1)) {
            atomicOr(a.status, STATUS_TIMEOUT);
            alive = false;
        }
        const float *c = col + slot * S::SLOT;
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

    // carried: records of rows m = r - 1 and m - 1, psi~+ of both, the values row m - 1 sends up, its south flux
    Rec32 cur, prev;
    Slope32 sy;
    float2 tf[4], tg[4], qf[4], qg[4];
    float2 t0 = f2(0.0f), q0 = f2(0.0f), pu = f2(0.0f), qu = f2(0.0f);   // rest directions and phi u of rows m, m - 1
    float2 Nf[3], Nhf, Ng[3], Nhg;       // (lane 0 of N counts)
    float N0 = 0.0f;
    Flux32 yS, yTop;
    Phi pm = phi_row();
    __syncwarp();
    load_row(S::S, 0);      // row 0 is needed for phi' only
    int cslot = slot;
    Phi pc = phi_row();
    const float h = ph.h;
    const int last = yb - ya + 3;
    for (int j = 0; j <= last; j++) {
        const int r = ya - 2 + j;
        const Phi pn = phi_row();
        const bool row_in = !WALLY || (r >= 0 && r < ny);
        const int yw = WALLY ? r : map_row<false>(r, ny);
        Rec32 nr;
        float2 ntf[4], ntg[4], nt0 = f2(0.0f), npu = f2(0.0f);
        if (row_in) {
            // ---- the cell of row r ----
            const float *c = col + cslot * S::SLOT;
            Pt<float> s;
            {
                const float C = pc.p, E = pc.e, Wv = pc.w, N = pn.p, Sv = pm.p, NE = pn.e, NW = pn.w, SE = pm.e, SW = pm.w;
                s.dpx = (E - Wv) * Real(1.0 / 3.0) + ((NE + SE) - (NW + SW)) * Real(1.0 / 12.0);
                s.dpy = (N - Sv) * Real(1.0 / 3.0) + ((NE + NW) - (SE + SW)) * Real(1.0 / 12.0);
                s.lap = (Real(4) * ((E + Wv) + (N + Sv)) + ((NE + NW) + (SE + SW)) - Real(20) * C) * Real(1.0 / 6.0);
            }
            nr = cell32<COUPLED>(ph, a, s, c, BW, HO, pc.p, xw, yw, ntf, ntg, nt0, npu,
                                 mine && r >= ya && r < yb);
        }
        __syncwarp();
        load_row(j + 1 + S::S, cslot);   // the slot of row r is free: every lane has read it
        cslot = cslot + 1 == S::S ? 0 : cslot + 1;
        if (j >= 2) {
            const bool has_m = !WALLY || (r - 1 >= 0 && r - 1 < ny);
            Flux32 yN;
            if (has_m) {
                // ---- the slopes of row m ----
                Slope32 sx, n;
                const bool bottom = WALLY && r - 1 == 0, top = WALLY && r == ny;
#pragma unroll
                for (int p = 0; p < 4; p++) {
                    sx.f[p] = limited32(cur.f[p], from_west(cur.f[p]), from_east(cur.f[p]));
                    n.f[p] = bottom ? sub2(nr.f[p], cur.f[p]) : top ? sub2(cur.f[p], prev.f[p]) : limited32(cur.f[p], prev.f[p], nr.f[p]);
                    if (COUPLED) {
                        sx.g[p] = limited32(cur.g[p], from_west(cur.g[p]), from_east(cur.g[p]));
                        n.g[p] = bottom ? sub2(nr.g[p], cur.g[p]) : top ? sub2(cur.g[p], prev.g[p]) : limited32(cur.g[p], prev.g[p], nr.g[p]);
                    }
                }
                sx.f0 = limited32(cur.f0, from_west(cur.f0), from_east(cur.f0));
                n.f0 = bottom ? nr.f0 - cur.f0 : top ? cur.f0 - prev.f0 : limited32(cur.f0, prev.f0, nr.f0);
                const int ym = WALLY ? r - 1 : map_row<false>(r - 1, ny);
                if (r - 1 >= ya && r - 1 < yb) {
                    // ---- the west x-face of row m, and its update along x ----
                    auto face = [&](const Leave32 &v, float2 o[4]) {
                        o[0] = f2(from_west(v.v[0].x), v.v[0].y);
                        o[1] = f2(from_west(v.v[1].x), v.v[1].y);
                        o[2] = mul2(f2(0.5f), add2(from_west(v.hi), v.lo));
                        o[3] = f2(v.v[2].x, from_west(v.v[2].y));
                    };
                    float2 fb[4], gb[4];
                    face(leave_all32<true>(cur.f, sx.f, n.f, h), fb);
                    if (COUPLED) face(leave_all32<true>(cur.g, sx.g, n.g, h), gb);
                    const float lo = leave32(f2(cur.f0), f2(sx.f0), -0.5f, -0.5f).x, hi = leave32(f2(cur.f0), f2(sx.f0), 0.5f, 0.5f).x;
                    const float f0 = 0.5f * (from_west(hi) + lo);
                    const float2 md = mul2(f2(0.5f), add2(from_west(cur.dp), cur.dp));
                    const float2 mD = mul2(f2(0.5f), add2(from_west(cur.D), cur.D));
                    const float ml = 0.5f * (from_west(cur.lap) + cur.lap);
                    float2 u = f2(0.0f);
                    if (!COUPLED) {
                        if (ph.vel_kind == 4) {
                            const long long kr = (long long)ym * a.pitch + xw, kl = kr - xw + (xw > 0 ? xw - 1 : nx - 1);
                            u.x = a.vel_faces ? a.vel[2 * a.plane + kl] : 0.5f * (a.vel[kl] + a.vel[kr]);
                            u.y = 0.5f * (a.vel[a.plane + kl] + a.vel[a.plane + kr]);
                        } else {
                            prescribed_velocity(ph, float(xw), float(ym) + 0.5f, a.t_n + double(ph.h), u.x, u.y);
                        }
                    }
                    const Flux32 xf = face32<COUPLED, true>(ph, fb, f0, gb, md, ml, mD, false, u.x, u.y);
                    Flux32 xe;
#pragma unroll
                    for (int i = 0; i < 3; i++) {
                        xe.f[i] = from_east(xf.f[i]);
                        if (COUPLED) xe.g[i] = from_east(xf.g[i]);
                    }
                    flux32<COUPLED, true>(ph.dt, xf, xe, tf, tg);
                }
                // ---- the y-face between rows m - 1 and m ----
                const Leave32 yf = leave_all32<false>(cur.f, n.f, sx.f, h);
                Leave32 yg;
                if (COUPLED) yg = leave_all32<false>(cur.g, n.g, sx.g, h);
                const float y0lo = leave32(f2(cur.f0), f2(n.f0), -0.5f, -0.5f).x, y0hi = leave32(f2(cur.f0), f2(n.f0), 0.5f, 0.5f).x;
                if (j >= 3 && (!WALLY || r - 1 > 0)) {
                    auto face = [&](const float2 N[3], float2 Nh, const Leave32 &v, float2 o[4]) {
                        o[0] = mul2(f2(0.5f), add2(Nh, v.lo));
#pragma unroll
                        for (int i = 0; i < 3; i++) o[1 + i] = f2(N[i].x, v.v[i].y);
                    };
                    float2 fb[4], gb[4];
                    face(Nf, Nhf, yf, fb);
                    if (COUPLED) face(Ng, Nhg, yg, gb);
                    const float f0 = 0.5f * (N0 + y0lo);
                    float2 u = f2(0.0f);
                    if (!COUPLED) {
                        if (ph.vel_kind == 4) {
                            const int yd = ym > 0 ? ym - 1 : ny - 1;
                            const long long kd = (long long)yd * a.pitch + xw, ku = (long long)ym * a.pitch + xw;
                            u.x = 0.5f * (a.vel[kd] + a.vel[ku]);
                            u.y = a.vel_faces ? a.vel[3 * a.plane + ku] : 0.5f * (a.vel[a.plane + kd] + a.vel[a.plane + ku]);
                        } else {
                            prescribed_velocity(ph, float(xw) + 0.5f, float(ym), a.t_n + double(ph.h), u.x, u.y);
                        }
                    }
                    yN = face32<COUPLED, false>(ph, fb, f0, gb, mul2(f2(0.5f), add2(prev.dp, cur.dp)), 0.5f * (prev.lap + cur.lap),
                                                mul2(f2(0.5f), add2(prev.D, cur.D)), false, u.x, u.y);
                }
                if (bottom || top) {
                    float2 fb[4], gb[4];
                    if (bottom) {
                        wall_upwind32<false>(cur.f, sx.f, n.f, h, fb);
                        if (COUPLED) wall_upwind32<false>(cur.g, sx.g, n.g, h, gb);
                    } else {
                        wall_upwind32<true>(cur.f, sx.f, n.f, h, fb);
                        if (COUPLED) wall_upwind32<true>(cur.g, sx.g, n.g, h, gb);
                    }
                    const float f0 = cur.f0 + (bottom ? -0.5f : 0.5f) * n.f0;
                    const Flux32 w = face32<COUPLED, false>(ph, fb, f0, gb, f2(cur.dp.x, 0.0f), cur.lap, f2(cur.D.x, 0.0f),
                                                            true, 0.0f, 0.0f);
                    if (bottom) yN = w;     // the south flux of row 0
                    else yTop = w;
                }
#pragma unroll
                for (int i = 0; i < 3; i++) {
                    Nf[i] = yf.v[i];
                    if (COUPLED) Ng[i] = yg.v[i];
                }
                Nhf = yf.hi;
                if (COUPLED) Nhg = yg.hi;
                N0 = y0hi;
            } else {
                yN = yTop;
            }
            if (j >= 4) {
                // ---- row m - 1 is done ----
                flux32<COUPLED, false>(ph.dt, yS, yN, qf, qg);
                if (mine && alive && in_bounds(x >= 0 && x < nx && r - 2 >= 0 && r - 2 < ny, a.status)) {
                    const long long g = (long long)(r - 2) * a.pitch + x;
                    float *d = a.dst + g;
                    d[0] = q0.x;
                    if (COUPLED) d[9 * a.plane] = q0.y;
#pragma unroll
                    for (int p = 0; p < 4; p++) {
                        d[(1 + p) * a.plane] = qf[p].x;
                        d[(5 + p) * a.plane] = qf[p].y;
                        if (COUPLED) {
                            d[(10 + p) * a.plane] = qg[p].x;
                            d[(14 + p) * a.plane] = qg[p].y;
                        }
                    }
                    a.hdst[g] = qu.x;
                    a.hdst[a.plane + g] = qu.y;
                }
            }
            yS = yN;
        }
        prev = cur;
        cur = nr;
#pragma unroll
        for (int p = 0; p < 4; p++) {
            qf[p] = tf[p];
            tf[p] = ntf[p];
            if (COUPLED) {
                qg[p] = tg[p];
                tg[p] = ntg[p];
            }
        }
        q0 = t0;
        t0 = nt0;
        qu = pu;
        pu = npu;
        pm = pc;
        pc = pn;
    }
    if (!alive)   // let copies in flight land before the CTA's shared memory is given away
        for (int s = 0; s < S::S; s++) mbar_wait(bar + s, (uint32_t)((nrows - 1 - s) / S::S) & 1u, kPollLimit);
}

}  // namespace dugks

// dugks_strip_launch.cuh -- host-side launcher of the strip kernel, one translation unit per precision.
#pragma once

#include "dugks_internal.h"
#include "dugks_strip.cuh"

#include <algorithm>

namespace dugks {

// FP64 has no strips for the coupled model between walls: the records that its wall faces read from shared memory leave
// room for one warp a scheduler, and the rectangles are faster at every size (380^2 255 us a step against the strips'
// 382 and the tiles' 371, 5000 x 40 348, 552 and 513, 1400^2 3,376, 3,993 and 4,620).
template <typename Real>
constexpr bool strip_compiled(bool coupled, bool wally) { return sizeof(Real) == 4 || !coupled || !wally; }

template <typename Real, typename F>
cudaError_t with_strip(bool coupled, bool wally, F &&f) {
    using T = std::true_type;
    using U = std::false_type;
    if (!coupled) return wally ? f(U{}, T{}) : f(U{}, U{});
    if constexpr (strip_compiled<Real>(true, true))
        if (wally) return f(T{}, T{});
    return wally ? cudaErrorInvalidValue : f(T{}, U{});
}

// Shared memory of a CTA of which 4 w and no more fit on an SM (228 KB, 1 KB of each CTA the system's).
inline size_t strip_share(int w) { return size_t(228 * 1024 / (4 * w) - 1024) & ~size_t(127); }

// Rows of a chunk.  All CTAs run at once, w warps on every scheduler; a chunk of r rows costs about r + 2.5 rows
// (two more records, one more y-face, the first loads), and a row of w warps 1.62 and 2.32 us for w = 2 and 3 (FP32
// coupled; Allen-Cahn alone, which waits more, 1 to 1.15; the other kernels' rows are shorter or longer by a common
// factor).  For each w the rows that fill it, of these the cheapest: 509 x 387 takes two warps and 7 rows (16.6 us)
// before three and 5 (17.7), 2048^2 three and 86 (206; two: 212), Allen-Cahn 512^2 three and 6 (13.8; two: 14.8).  One
// warp is never better: its rows are twice as many and hardly faster (256^2 16.9 us against 9.8).  Results do not
// depend on the rows.
template <typename Ctas>
inline int strip_rows(bool coupled, int max_warps, int sms, int ny, int *warps, Ctas &&ctas) {
    const double row[] = {1.0, 1.62, coupled ? 2.32 : 1.87};
    int best = ny;
    double cost = 0;
    *warps = max_warps;
    for (int w = std::min(2, max_warps); w <= max_warps && w <= 3; w++) {
        int lo = 1, hi = ny;   // the fewest rows whose CTAs run at once (or all of them: one chunk a strip)
        while (lo < hi) {
            const int mid = (lo + hi) / 2;
            if (ctas(mid) <= 4ll * sms * w) hi = mid;
            else lo = mid + 1;
        }
        const double c = (lo + 2.5) * row[w - 1];
        if (cost == 0 || c < cost || ctas(lo) > 4ll * sms * w) {
            cost = c;
            best = lo;
            *warps = w;
        }
    }
    return best;
}

template <typename Real>
cudaError_t strip_plan(bool coupled, bool wally, int nx, int ny, StripPlan *out) {
    int dev = 0, sms = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (e != cudaSuccess || !strip_compiled<Real>(coupled, wally)) return e;
    return with_strip<Real>(coupled, wally, [&](auto c, auto wl) {
        constexpr bool C = decltype(c)::value, W = decltype(wl)::value;
        using S = StripShape<Real, C, strip_shuffles<Real, W>(), strip_keeps<Real, W>()>;
        constexpr size_t bytes = S::smem_bytes(kStripLanes, W);
        static OncePerDevice<int> resident;   // CTAs that fit on an SM
        int per_sm = 0;
        const cudaError_t e = resident.get(dev, &per_sm, [&](int *out) {
            cudaError_t r = cudaFuncSetAttribute(strip_step_kernel<Real, C, W>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                                 (int)std::max(bytes, strip_share(1)));
            if (r == cudaSuccess)
                r = cudaFuncSetAttribute(strip_batch_kernel<Real, C, W>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         (int)std::max(bytes, strip_share(1)));
            if (r == cudaSuccess)
                r = cudaOccupancyMaxActiveBlocksPerMultiprocessor(out, strip_step_kernel<Real, C, W>, kStripLanes, bytes);
            return r;
        });
        if (e != cudaSuccess) return e;
        if (per_sm < 1) return cudaErrorInvalidConfiguration;
        const int own = S::own(kStripLanes);
        const int nstrips = (nx + own - 1) / own;
        const int warps = std::min(per_sm, strip_ctas<Real, W>()) / 4;   // a scheduler
        out->max_warps = warps > 0 ? warps : 1;
        int w = 1;
        const int rows = strip_rows(coupled, out->max_warps, sms, ny, &w, [&](int r) { return (long long)nstrips * ((ny + r - 1) / r); });
        // A step's CTAs come while the last one's run: where more of them fit than the plan wants, some SMs would take
        // a third more of them than others (509 x 387 22.0 us against 16.6, 700^2 40.8 against 30.4, Allen-Cahn 2048^2
        // 162 against 137).  Below one warp a scheduler there is nothing to even out (64^2 5.0 against 6.0).
        const bool even = per_sm > 4 * w && (long long)nstrips * ((ny + rows - 1) / rows) > 4ll * sms;
        out->smem = even ? std::max(bytes, strip_share(w)) : bytes;
        // FP64: below eight rows a chunk the rectangles are faster at every size measured, 1.2 to 1.9 times where the grid
        // fills the chip (380^2 257 us a step against 329, Allen-Cahn 116 against 145) and up to 4.1 on smaller ones
        if (sizeof(Real) == 8 && rows < 8) return cudaSuccess;
        out->threads = kStripLanes;
        out->box = S::box(kStripLanes);
        out->own = own;
        out->rows = rows;
        out->nstrips = nstrips;
        return cudaSuccess;
    });
}

template <typename Real>
cudaError_t launch_strip(const StripPlan &pl, const StripMaps &tm, const StepArgs<Real> &a, const typename StripConst<Real>::T &sp,
                         const Phys<Real> &ph, bool coupled, bool wally, cudaStream_t st) {
    return with_strip<Real>(coupled, wally, [&](auto c, auto wl) {
        constexpr bool C = decltype(c)::value, W = decltype(wl)::value;
        using S = StripShape<Real, C, strip_shuffles<Real, W>(), strip_keeps<Real, W>()>;
        const StripArgs g{pl.nstrips, pl.rows};
        cudaLaunchAttribute at[1];
        at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
        at[0].val.programmaticStreamSerializationAllowed = 1;
        cudaLaunchConfig_t cfg = {};
        cfg.gridDim = dim3((unsigned)(pl.nstrips * ((a.ny + pl.rows - 1) / pl.rows)));
        cfg.blockDim = dim3(kStripLanes);
        cfg.dynamicSmemBytes = pl.smem;
        cfg.stream = st;
        cfg.attrs = at;
        cfg.numAttrs = 1;
        return cudaLaunchKernelEx(&cfg, strip_step_kernel<Real, C, W>, tm, a, sp, ph, g);
    });
}

// The rows of a chunk for a group of members (strips and rows of each).
template <typename Real>
cudaError_t strip_group_rows(bool coupled, bool wally, const int2 *members, int n, int *rows) {
    int dev = 0, sms = 0, most = 1;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    StripPlan one;
    if (e == cudaSuccess) e = strip_plan<Real>(coupled, wally, 1 << 20, 1 << 20, &one);
    if (e != cudaSuccess) return e;
    for (int i = 0; i < n; i++) most = std::max(most, members[i].y);
    int w = 1;
    *rows = strip_rows(coupled, one.max_warps, sms, most, &w, [&](int r) {
        long long t = 0;
        for (int i = 0; i < n; i++) t += (long long)members[i].x * ((members[i].y + r - 1) / r);
        return t;
    });
    return cudaSuccess;
}

// One step of a group of members (at most kStripMembers), `step` steps after its descriptors were last advanced.
template <typename Real>
cudaError_t launch_strip_group(const StripInst<Real> *inst, const typename StripConst<Real>::T *ph, const int2 *members, int n,
                               int rows, int step, bool coupled, bool wally, bool overlap, cudaStream_t st) {
    StripGroup<Real> g;
    g.inst = inst;
    g.n = n;
    g.rows = rows;
    g.step = step;
    g.first[0] = 0;
    for (int i = 0; i < n; i++) {
        g.first[i + 1] = g.first[i] + members[i].x * ((members[i].y + rows - 1) / rows);
        g.ph[i] = ph[i];
    }
    return with_strip<Real>(coupled, wally, [&](auto c, auto wl) {
        constexpr bool C = decltype(c)::value, W = decltype(wl)::value;
        using S = StripShape<Real, C, strip_shuffles<Real, W>(), strip_keeps<Real, W>()>;
        cudaLaunchAttribute at[1];
        at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
        at[0].val.programmaticStreamSerializationAllowed = overlap ? 1 : 0;
        cudaLaunchConfig_t cfg = {};
        cfg.gridDim = dim3((unsigned)g.first[n]);
        cfg.blockDim = dim3(kStripLanes);
        cfg.dynamicSmemBytes = S::smem_bytes(kStripLanes, W);
        cfg.stream = st;
        cfg.attrs = at;
        cfg.numAttrs = 1;
        return cudaLaunchKernelEx(&cfg, strip_batch_kernel<Real, C, W>, g);
    });
}
template <typename Real>
cudaError_t launch_strip_advance(StripInst<Real> *inst, int n, int k, cudaStream_t st) {
    strip_advance_kernel<Real><<<(n + 127) / 128, 128, 0, st>>>(inst, n, k);
    return cudaGetLastError();
}

#define DUGKS_INSTANTIATE_STRIP(Real)                                                                              \
    template cudaError_t strip_plan<Real>(bool, bool, int, int, StripPlan *);                                      \
    template cudaError_t launch_strip<Real>(const StripPlan &, const StripMaps &, const StepArgs<Real> &,          \
                                            const StripConst<Real>::T &, const Phys<Real> &, bool, bool, cudaStream_t);  \
    template cudaError_t strip_group_rows<Real>(bool, bool, const int2 *, int, int *);                             \
    template cudaError_t launch_strip_group<Real>(const StripInst<Real> *, const StripConst<Real>::T *, const int2 *,  \
                                                  int, int, int, bool, bool, bool, cudaStream_t);                  \
    template cudaError_t launch_strip_advance<Real>(StripInst<Real> *, int, int, cudaStream_t);

}  // namespace dugks

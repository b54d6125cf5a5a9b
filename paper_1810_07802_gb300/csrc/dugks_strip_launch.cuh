// dugks_strip_launch.cuh -- host-side launcher of the strip kernel, one translation unit per precision.
#pragma once

#include "dugks_internal.h"
#include "dugks_strip.cuh"

namespace dugks {

template <typename F>
cudaError_t with_strip(bool coupled, bool wally, F &&f) {
    using T = std::true_type;
    using U = std::false_type;
    if (coupled) return wally ? f(T{}, T{}) : f(T{}, U{});
    return wally ? f(U{}, T{}) : f(U{}, U{});
}

template <typename Real>
cudaError_t strip_plan(bool coupled, bool wally, int nx, int ny, StripPlan *out) {
    int dev = 0, sms = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (e != cudaSuccess) return e;
    return with_strip(coupled, wally, [&](auto c, auto wl) {
        constexpr bool C = decltype(c)::value, W = decltype(wl)::value;
        using S = StripShape<Real, C, strip_shuffles<Real, W>()>;
        constexpr size_t bytes = S::smem_bytes(kStripLanes, W);
        static OncePerDevice<int> resident;   // CTAs that fit on an SM
        int per_sm = 0;
        const cudaError_t e = resident.get(dev, &per_sm, [&](int *out) {
            cudaError_t r = cudaFuncSetAttribute(strip_step_kernel<Real, C, W>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                                 (int)bytes);
            if (r == cudaSuccess)
                r = cudaFuncSetAttribute(strip_batch_kernel<Real, C, W>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         (int)bytes);
            if (r == cudaSuccess)
                r = cudaOccupancyMaxActiveBlocksPerMultiprocessor(out, strip_step_kernel<Real, C, W>, kStripLanes, bytes);
            return r;
        });
        if (e != cudaSuccess) return e;
        if (per_sm < 1) return cudaErrorInvalidConfiguration;
        const int own = S::own(kStripLanes);
        const int nstrips = (nx + own - 1) / own;
        // one wave: as many chunks as run at once, so that every scheduler holds two warps to the end
        const long long ctas = (long long)(per_sm < kStripCtas ? per_sm : kStripCtas) * sms;
        const long long chunks = ctas > nstrips ? ctas / nstrips : 1;
        const int rows = (int)((ny + chunks - 1) / chunks);
        out->ctas = (int)ctas;
        // FP64: below eight rows a chunk the tile kernel's halo costs less than the rows a chunk adds
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
    return with_strip(coupled, wally, [&](auto c, auto wl) {
        constexpr bool C = decltype(c)::value, W = decltype(wl)::value;
        using S = StripShape<Real, C, strip_shuffles<Real, W>()>;
        const StripArgs g{pl.nstrips, pl.rows};
        cudaLaunchAttribute at[1];
        at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
        at[0].val.programmaticStreamSerializationAllowed = 1;
        cudaLaunchConfig_t cfg = {};
        cfg.gridDim = dim3((unsigned)(pl.nstrips * ((a.ny + pl.rows - 1) / pl.rows)));
        cfg.blockDim = dim3(kStripLanes);
        cfg.dynamicSmemBytes = S::smem_bytes(kStripLanes, W);
        cfg.stream = st;
        cfg.attrs = at;
        cfg.numAttrs = 1;
        return cudaLaunchKernelEx(&cfg, strip_step_kernel<Real, C, W>, tm, a, sp, ph, g);
    });
}

// The largest CTA count that runs at once and the rows of a chunk that keep a group of members (strips and rows of
// each) within it: results do not depend on the rows of a chunk.
template <typename Real>
cudaError_t strip_group_rows(bool coupled, bool wally, const int2 *members, int n, int *rows) {
    StripPlan one;
    cudaError_t e = strip_plan<Real>(coupled, wally, 1 << 20, 1 << 20, &one);
    if (e != cudaSuccess) return e;
    auto ctas = [&](int r) {
        long long t = 0;
        for (int i = 0; i < n; i++) t += (long long)members[i].x * ((members[i].y + r - 1) / r);
        return t;
    };
    int lo = 1, hi = 1;
    for (int i = 0; i < n; i++) hi = members[i].y > hi ? members[i].y : hi;
    while (lo < hi) {
        const int mid = (lo + hi) / 2;
        if (ctas(mid) <= one.ctas) hi = mid;
        else lo = mid + 1;
    }
    *rows = lo;
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
    return with_strip(coupled, wally, [&](auto c, auto wl) {
        constexpr bool C = decltype(c)::value, W = decltype(wl)::value;
        using S = StripShape<Real, C, strip_shuffles<Real, W>()>;
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

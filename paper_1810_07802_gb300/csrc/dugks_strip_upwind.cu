// FP32 upwind strip kernel: launch.
#include "dugks_internal.h"
#include "dugks_strip_upwind.cuh"

namespace dugks {

namespace {
template <typename F>
cudaError_t with_upwind(bool coupled, bool wally, F &&f) {
    using T = std::true_type;
    using U = std::false_type;
    if (coupled) return wally ? f(T{}, T{}) : f(T{}, U{});
    return wally ? f(U{}, T{}) : f(U{}, U{});
}
}  // namespace

cudaError_t strip_upwind_plan(bool coupled, bool wally, int nx, int ny, StripPlan *out) {
    int dev = 0, sms = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (e != cudaSuccess) return e;
    return with_upwind(coupled, wally, [&](auto c, auto w) {
        constexpr bool C = decltype(c)::value, W = decltype(w)::value;
        constexpr size_t bytes = UpwindShape<C>::smem_bytes;
        static OncePerDevice<char> ready;
        const cudaError_t e = ready.get(dev, nullptr, [&](char *) {
            return cudaFuncSetAttribute(strip_upwind_kernel<C, W>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
        });
        if (e != cudaSuccess) return e;
        out->threads = kStripLanes;
        out->box = UpwindShape<C>::BW;
        out->own = kUpwindOwn;
        out->nstrips = (nx + kUpwindOwn - 1) / kUpwindOwn;
        const long long ctas = (long long)kStripCtas * sms, chunks = ctas > out->nstrips ? ctas / out->nstrips : 1;
        out->rows = (int)((ny + chunks - 1) / chunks);
        return cudaSuccess;
    });
}

cudaError_t launch_strip_upwind(const StripPlan &pl, const StripMaps &tm, const StepArgs<float> &a, const Phys<float> &ph,
                                bool coupled, bool wally, cudaStream_t st) {
    return with_upwind(coupled, wally, [&](auto c, auto w) {
        constexpr bool C = decltype(c)::value, W = decltype(w)::value;
        const StripArgs g{pl.nstrips, pl.rows};
        cudaLaunchAttribute at[1];
        at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
        at[0].val.programmaticStreamSerializationAllowed = 1;
        cudaLaunchConfig_t cfg = {};
        cfg.gridDim = dim3((unsigned)(pl.nstrips * ((a.ny + pl.rows - 1) / pl.rows)));
        cfg.blockDim = dim3(kStripLanes);
        cfg.dynamicSmemBytes = UpwindShape<C>::smem_bytes;
        cfg.stream = st;
        cfg.attrs = at;
        cfg.numAttrs = 1;
        return cudaLaunchKernelEx(&cfg, strip_upwind_kernel<C, W>, tm, a, ph, g);
    });
}

}  // namespace dugks

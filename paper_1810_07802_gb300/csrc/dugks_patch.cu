// The FP64 step kernel of rectangles: their sizes and launch.
#include "dugks_internal.h"
#include "dugks_patch.cuh"

namespace dugks {

namespace {
template <typename F>
cudaError_t with_patch(bool coupled, bool wally, bool upw, F &&f) {
    using T = std::true_type;
    using U = std::false_type;
    auto g = [&](auto c, auto w) { return upw ? f(c, w, T{}) : f(c, w, U{}); };
    if (coupled) return wally ? g(T{}, T{}) : g(T{}, U{});
    return wally ? g(U{}, T{}) : g(U{}, U{});
}
// FP64 instructions of a cell, a face and a row of 32 lanes' phi' and update (counted in the source; coupled, A-C)
struct PatchCost {
    double cell, face, other;
};
PatchCost patch_cost(bool coupled, bool upw) {
    PatchCost c = coupled ? PatchCost{212, 235, 56} : PatchCost{92, 90, 32};
    if (upw) c.face += coupled ? 320 : 160;   // 38 (19) limited slopes instead of the central sums
    return c;
}
constexpr double kPatchFixed = 400;   // launch, loads and barriers of one CTA, in FP64 instructions (about 3 us)
}  // namespace

// The rectangle that leaves the busiest SM the fewest FP64 instructions, and that number against the strip
// kernel's (rows of 28 columns a warp, strip_rows rows a chunk; 0: no strips for this problem).
cudaError_t patch_plan(bool coupled, bool wally, bool upw, int nx, int ny, int strip_rows, PatchPlan *out) {
    int dev = 0, sms = 0, most = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&most, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
    if (e != cudaSuccess) return e;
    const PatchCost c = patch_cost(coupled, upw);
    auto warps = [](long long n) { return double((n + 31) / 32); };
    double best = 0;
    // of the sizes that cut an axis into the same number of rectangles the smallest
    auto smallest = [](int t, int n) { return t == 1 || (n + t - 1) / t != (n + t - 2) / (t - 1); };
    for (int ty = 1; ty <= 64 && ty <= ny; ty++) {
        if (!smallest(ty, ny)) continue;
        for (int tx = 1; tx <= 64 && tx <= nx; tx++) {
            if (!smallest(tx, nx)) continue;
            const size_t bytes = coupled ? (upw ? PatchShape<true, true>::smem_bytes(tx, ty) : PatchShape<true, false>::smem_bytes(tx, ty))
                                         : (upw ? PatchShape<false, true>::smem_bytes(tx, ty) : PatchShape<false, false>::smem_bytes(tx, ty));
            const int halo = upw ? 4 : 2;
            if (bytes > (size_t)most) continue;
            const long long tiles = (long long)((nx + tx - 1) / tx) * ((ny + ty - 1) / ty);
            const double one = c.cell * warps((long long)(tx + halo) * (ty + halo)) +
                               c.face * warps((long long)(tx + 1) * ty + (long long)tx * (ty + 1)) +
                               c.other * warps((long long)tx * ty) + kPatchFixed;
            const double t = one * double((tiles + sms - 1) / sms);
            if (best == 0 || t < best) {
                best = t;
                out->tx = tx;
                out->ty = ty;
                out->smem = bytes;
            }
        }
    }
    if (strip_rows > 0) {
        const double strips = (nx + 27) / 28, chunks = (ny + strip_rows - 1) / strip_rows;
        const double rows = strips * (ny + 2 * chunks), ctas = strips * chunks;
        const double strip = (rows * c.cell + strips * ny * 2 * c.face + ctas * c.face) / sms;
        if (strip < best) out->tx = out->ty = 0;
    }
    if (out->tx == 0) return cudaSuccess;
    return with_patch(coupled, wally, upw, [&](auto cp, auto w, auto u) {
        constexpr bool C = decltype(cp)::value, W = decltype(w)::value, UP = decltype(u)::value;
        static OncePerDevice<char> ready;
        return ready.get(dev, nullptr, [&](char *) {
            return cudaFuncSetAttribute(patch_step_kernel<C, W, UP>, cudaFuncAttributeMaxDynamicSharedMemorySize, most);
        });
    });
}

cudaError_t launch_patch(const PatchPlan &pl, const StepArgs<double> &a, const StripPhys<double> &sp,
                         const Phys<double> &ph, bool coupled, bool wally, bool upw, cudaStream_t st) {
    return with_patch(coupled, wally, upw, [&](auto cp, auto w, auto u) {
        constexpr bool C = decltype(cp)::value, W = decltype(w)::value, UP = decltype(u)::value;
        const PatchArgs g{pl.tx, pl.ty, (a.nx + pl.tx - 1) / pl.tx};
        cudaLaunchAttribute at[1];
        at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
        at[0].val.programmaticStreamSerializationAllowed = 1;
        cudaLaunchConfig_t cfg = {};
        cfg.gridDim = dim3((unsigned)(g.tiles_x * ((a.ny + pl.ty - 1) / pl.ty)));
        cfg.blockDim = dim3(kPatchThreads);
        cfg.dynamicSmemBytes = pl.smem;
        cfg.stream = st;
        cfg.attrs = at;
        cfg.numAttrs = 1;
        return cudaLaunchKernelEx(&cfg, patch_step_kernel<C, W, UP>, a, sp, ph, g);
    });
}

}  // namespace dugks

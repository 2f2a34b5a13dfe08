// Ensemble variants of the step kernel (many parameter sets in one launch):
// per-set tallies in FP64 accumulators in global memory, their counts there too or per
// block in shared memory (all sets' bins), at 128 or 256 threads per
// block, for the cell or the pair record layout (compile-time, as for the
// single-set kernels).  The step arithmetic is the single-set kernel's (fte_step.cuh).
#include "fte_step.cuh"

namespace fte {

template <int MODE, int NT, int LAY>
static const void* pick(int kperp, int dtype)
{
    if (dtype == FTE_BF16)
        return kperp ? (const void*)advance_kernel<true, FTE_BF16, MODE, NT, LAY>
                     : (const void*)advance_kernel<false, FTE_BF16, MODE, NT, LAY>;
    if (dtype == FTE_F16)
        return kperp ? (const void*)advance_kernel<true, FTE_F16, MODE, NT, LAY>
                     : (const void*)advance_kernel<false, FTE_F16, MODE, NT, LAY>;
    return kperp ? (const void*)advance_kernel<true, FTE_F32, MODE, NT, LAY>
                 : (const void*)advance_kernel<false, FTE_F32, MODE, NT, LAY>;
}

template <int MODE, int NT>
static const void* pick_layout(int kperp, int dtype, int pair)
{
    return pair ? pick<MODE, NT, kLayPair>(kperp, dtype) : pick<MODE, NT, kLayCell>(kperp, dtype);
}

// global tally, cell records, no cross-field diffusion, options fixed (advance_opt); near: with
// the reach test of the observers (kShapeNear)
template <int DT, int NT>
static const void* pick_linear_dt(bool near)
{
    constexpr int shape = kShapeUnroll | kShapeNormals;
    return near ? (const void*)advance_kernel<false, DT, kModeGlobal, NT, kLayCell, 0, kOptLinear, shape | kShapeNear>
                : (const void*)advance_kernel<false, DT, kModeGlobal, NT, kLayCell, 0, kOptLinear, shape>;
}

template <int NT>
static const void* pick_linear(int dtype, bool near)
{
    if (dtype == FTE_BF16) return pick_linear_dt<FTE_BF16, NT>(near);
    if (dtype == FTE_F16) return pick_linear_dt<FTE_F16, NT>(near);
    return pick_linear_dt<FTE_F32, NT>(near);
}

const void* advance_fn_batched(int kperp, int dtype, int mode, int nt, int pair, int opt, bool near)
{
    if (opt == kOptLinear) {
        if (nt == 128) return pick_linear<128>(dtype, near);
        return nt == 256 ? pick_linear<256>(dtype, near) : nullptr;
    }
    if (mode == kModeShared) {
        if (nt == 128) return pick_layout<kModeShared, 128>(kperp, dtype, pair);
        if (nt == 256) return pick_layout<kModeShared, 256>(kperp, dtype, pair);
    } else if (mode == kModeGlobal) {
        if (nt == 128) return pick_layout<kModeGlobal, 128>(kperp, dtype, pair);
        if (nt == 256) return pick_layout<kModeGlobal, 256>(kperp, dtype, pair);
    }
    return nullptr;
}

cudaError_t launch_advance_batched(const AdvanceArgs& a, const BatchArgs& b, int kperp, int mode, int nt,
                                   int opt, bool near, int blocks, size_t smem, cudaStream_t s)
{
    const void* fn = advance_fn_batched(kperp, a.g.dtype, mode, nt, a.g.pair, opt, near);
    if (!fn) return cudaErrorInvalidValue;
    void* args[] = {(void*)&a, (void*)&b};
    return cudaLaunchKernel(fn, dim3(blocks), dim3(nt), args, smem, s);
}

}  // namespace fte

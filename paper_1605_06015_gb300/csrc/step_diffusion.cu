// Explicit instantiations of the fused step kernel for the diffusion model.
#include "bbx_device.cuh"

namespace bbx {

template <bool MA, int AN, int TY, bool PL, bool GE, bool FL>
static StepKernel make_diffusion() {
    using P = Plan<BBX_DIFFUSION, MA, AN, TY, false, GATES_F32, FL>;
    return StepKernel{reinterpret_cast<const void*>(&step_kernel<BBX_DIFFUSION, MA, AN, TY, false, PL, GE, GATES_F32, FL>), P::SMEM,
                      P::THREADS, TY, P::FLOW};
}

template <bool MA, int AN, int TY, bool FL>
static StepKernel pick_diffusion(bool planar, bool general) {
    if constexpr (TY == 28) {  // the general variants have 7- and 14-row tiles
        if (general) return StepKernel{nullptr, 0, 0, 0};
    } else {
        if (general) return planar ? make_diffusion<MA, AN, TY, true, true, FL>() : make_diffusion<MA, AN, TY, false, true, FL>();
    }
    return planar ? make_diffusion<MA, AN, TY, true, false, FL>() : make_diffusion<MA, AN, TY, false, false, FL>();
}

// planar: grids with nz = 1 (tiles marched along y); general: the variant
// for the Lie scheme or the RK4 solver; flow: the variant that may take
// several steps in one launch, for the grids that have one
StepKernel step_kernel_diffusion(bool masked, int aniso, int ty, bool planar, bool general, bool flow) {
    // unmasked grids whose W-tilde sums all vanish: no sums in the stage ring
    // (plain variants; the general ones read the sums, or skip their copies)
#define BBX_CASE_NS(T) \
    if (!masked && aniso == AN_NO_SUMS && ty == T) \
        return general || !flow ? StepKernel{nullptr, 0, 0, 0} \
                       : (planar ? make_diffusion<false, AN_NO_SUMS, T, true, false, true>() : make_diffusion<false, AN_NO_SUMS, T, false, false, true>());
    BBX_CASE_NS(7) BBX_CASE_NS(14) BBX_CASE_NS(28)
#undef BBX_CASE_NS
#define BBX_CASE(MA, AN, T) \
    if (masked == MA && aniso == AN && ty == T) \
        return !MA && flow ? pick_diffusion<MA, AN, T, !MA>(planar, general) : pick_diffusion<MA, AN, T, false>(planar, general);
    BBX_CASE(false, false, 7) BBX_CASE(false, false, 14) BBX_CASE(false, false, 28)
    BBX_CASE(false, true, 7) BBX_CASE(false, true, 14) BBX_CASE(false, true, 28)
    BBX_CASE(true, false, 7) BBX_CASE(true, false, 14) BBX_CASE(true, false, 28)
    BBX_CASE(true, true, 7) BBX_CASE(true, true, 14) BBX_CASE(true, true, 28)
#undef BBX_CASE
    return StepKernel{nullptr, 0, 0, 0};
}

}  // namespace bbx

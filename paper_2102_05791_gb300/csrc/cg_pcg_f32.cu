// The persistent CG solver with FP32 vectors (one translation unit a precision: they compile side by side).
#include "cg_pcg_kernel.cuh"

namespace softsim {

template bool pcg_configure<float>(const Ctx &, PcgDev &);
template cudaError_t launch_pcg<float>(const Ctx &, const PcgDev &, const double *, double, float *, double, int,
                                       cudaStream_t);

}  // namespace softsim

// The persistent CG solver with FP64 vectors (one translation unit a precision: they compile side by side).
#include "cg_pcg_kernel.cuh"

namespace softsim {

template bool pcg_configure<double>(const Ctx &, PcgDev &);
template cudaError_t launch_pcg<double>(const Ctx &, const PcgDev &, const double *, double, double *, double, int,
                                       cudaStream_t);

}  // namespace softsim

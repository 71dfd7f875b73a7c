// Binary64 time DFTs in registers (rfft.cuh).
#include "rfft.cuh"

namespace pd {

template void rfft_launch<double, double>(Ctx &, const double *, int64_t, int64_t, int, const cpx<double> *, cpx<double> *, int64_t,
    const double *, const RhsNorm &, const SlotScale &, const char *, double);
template void crfft_launch<double>(Ctx &, const cpx<double> *, int64_t, int64_t, int, const cpx<double> *, void *, int64_t, int,
    double *, int *, const StepFinish &, const double *, double *, const int *, int, const int *, const SlotScale &, const char *, double);

}  // namespace pd

// Binary32, inverse: time DFTs in registers (rfft.cuh).
#include "rfft.cuh"

namespace pd {

template void crfft_launch<float>(Ctx &, const cpx<float> *, int64_t, int64_t, int, const cpx<float> *, void *, int64_t, int,
    double *, int *, const StepFinish &, const float *, double *, const int *, int, const int *, const SlotScale &, const char *, double);

}  // namespace pd

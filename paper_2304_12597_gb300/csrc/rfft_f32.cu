// Binary32, forward: time DFTs in registers (rfft.cuh).
#include "rfft.cuh"

namespace pd {

template void rfft_launch<float, double>(Ctx &, const double *, int64_t, int64_t, int, const cpx<float> *, cpx<float> *, int64_t,
    const float *, const RhsNorm &, const SlotScale &, const char *, double);
template void rfft_launch<float, float>(Ctx &, const float *, int64_t, int64_t, int, const cpx<float> *, cpx<float> *, int64_t,
    const float *, const RhsNorm &, const SlotScale &, const char *, double);

}  // namespace pd

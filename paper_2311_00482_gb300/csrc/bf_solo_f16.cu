// Solo beamforming kernels of FP16 records.
#include "bf_solo.cuh"

namespace bfi {

BF_SOLO_INSTANTIATE(launch_solo_f16, kPrecF16)

}  // namespace bfi

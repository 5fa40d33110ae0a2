// Solo beamforming kernels of BF16 records.
#include "bf_solo.cuh"

namespace bfi {

BF_SOLO_INSTANTIATE(launch_solo_bf16, kPrecBF16)

}  // namespace bfi

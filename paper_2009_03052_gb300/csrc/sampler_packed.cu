// sampler_packed.cu -- the samplers' instantiations for packed (succinct)
// tables.
#include "sampler.cuh"

namespace mc {

template <typename CT, typename V> static SampleKernel pick(SampleMode mode)
{
    switch (mode) {
    case SampleMode::Split: return sample_kernel<CT, V, true, false, false, true>;
    case SampleMode::Warps: return sample_warp_kernel<CT, V, true>;
    default: return sample_kernel<CT, V, true, false, false, false>;
    }
}

SampleKernel sample_kernel_packed(SampleMode mode, int bits, bool narrow)
{
    if (bits == 128) return pick<u128, u128>(mode);
    return narrow ? pick<uint64_t, uint64_t>(mode) : pick<uint64_t, u128>(mode);
}

}  // namespace mc

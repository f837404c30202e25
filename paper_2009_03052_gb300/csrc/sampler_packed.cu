// sampler_packed.cu -- the samplers' instantiations for packed (succinct)
// tables.
#include "sampler.cuh"

namespace mc {

template <typename CT, typename V> static SampleKernel pick(SampleMode mode, bool few)
{
    switch (mode) {
    case SampleMode::Latency: return sample_kernel<CT, V, true, true, false, false>;
    case SampleMode::Warps: return sample_warp_kernel<CT, V, true>;
    case SampleMode::Split:
        if (few) return sample_kernel<CT, V, true, false, false, true, 0, true>;
        return sample_kernel<CT, V, true, false, false, true>;
    default:
        if (few) return sample_kernel<CT, V, true, false, false, false, 0, true>;
        return sample_kernel<CT, V, true, false, false, false>;
    }
}

SampleKernel sample_kernel_packed(SampleMode mode, int bits, bool narrow, bool few)
{
    if (bits == 128) return pick<u128, u128>(mode, few);
    return narrow ? pick<uint64_t, uint64_t>(mode, few) : pick<uint64_t, u128>(mode, few);
}

}  // namespace mc

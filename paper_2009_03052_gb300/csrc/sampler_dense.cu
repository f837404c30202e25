// sampler_dense.cu -- the samplers' instantiations for dense tables (a
// translation unit of their own, so the build compiles them in parallel).
#include "sampler.cuh"

namespace mc {

template <typename CT, typename V> static SampleKernel pick(SampleMode mode, int wide)
{
    if constexpr (sizeof(CT) == 16)
        if (wide) switch (mode) {
            case SampleMode::Lanes: return sample_kernel<CT, V, false, false, false, false, 4>;
            case SampleMode::Latency: return sample_kernel<CT, V, false, true, false, false, 4>;
            case SampleMode::Split:
                if (wide == 3) return sample_kernel<CT, V, false, false, false, true, 3>;
                return sample_kernel<CT, V, false, false, false, true, 4>;
            default: break;
            }
    switch (mode) {
    case SampleMode::Lanes: return sample_kernel<CT, V, false, false, false, false>;
    case SampleMode::Latency: return sample_kernel<CT, V, false, true, false, false>;
    case SampleMode::Counted: return sample_kernel<CT, V, false, false, true, false>;
    case SampleMode::Split: return sample_kernel<CT, V, false, false, false, true>;
    case SampleMode::Warps: return sample_warp_kernel<CT, V, false>;
    }
    return nullptr;
}

SampleKernel sample_kernel_dense(SampleMode mode, int bits, bool narrow, int wide)
{
    if (bits == 128) return pick<u128, u128>(mode, wide);
    return narrow ? pick<uint64_t, uint64_t>(mode, 0) : pick<uint64_t, u128>(mode, 0);
}

}  // namespace mc

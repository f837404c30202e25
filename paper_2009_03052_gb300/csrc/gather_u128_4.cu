// gather_u128_4.cu -- instantiations of the neighbour-sum kernel for u128
// counts with first planes of 4-byte counts, one per lane layout that a
// level of k = 3..8 colours has (translation units of their own, so the
// build compiles them in parallel).
#include "gather.cuh"

namespace mc {

GatherKernel gather_kernel_ptr_u128_4(int UB, int G, int NU, int P, int U, int MB)
{
    MC_GATHER_LAYOUT(u128, 4, 4, 1, 1, 8)
    MC_GATHER_LAYOUT(u128, 4, 4, 1, 1, 4)
    MC_GATHER_LAYOUT(u128, 4, 4, 4, 1, 2)
    MC_GATHER_LAYOUT(u128, 4, 4, 4, 1, 1)
    MC_GATHER_LAYOUT(u128, 4, 4, 8, 1, 1)
    MC_GATHER_LAYOUT(u128, 4, 4, 16, 1, 1)
    MC_GATHER_LAYOUT(u128, 4, 4, 32, 1, 1)
    MC_GATHER_LAYOUT(u128, 4, 4, 32, 2, 1)
    MC_GATHER_LAYOUT(u128, 4, 4, 32, 6, 1)
    MC_GATHER_LAYOUT(u128, 4, 8, 1, 1, 8)
    MC_GATHER_LAYOUT(u128, 4, 8, 1, 1, 4)
    MC_GATHER_LAYOUT(u128, 4, 8, 4, 1, 2)
    MC_GATHER_LAYOUT(u128, 4, 8, 4, 1, 1)
    MC_GATHER_LAYOUT(u128, 4, 8, 16, 1, 1)
    MC_GATHER_LAYOUT(u128, 4, 8, 32, 1, 1)
    MC_GATHER_LAYOUT(u128, 4, 8, 32, 2, 1)
    MC_GATHER_LAYOUT(u128, 4, 16, 1, 1, 8)
    MC_GATHER_LAYOUT(u128, 4, 16, 1, 1, 4)
    MC_GATHER_LAYOUT(u128, 4, 16, 8, 1, 1)
    MC_GATHER_LAYOUT(u128, 4, 16, 16, 1, 1)
    MC_GATHER_LAYOUT(u128, 4, 16, 32, 2, 1)
    MC_GATHER_FOLDED(u128, 4, 4, 4, 2, 2)
    MC_GATHER_FOLDED(u128, 4, 4, 4, 2, 1)
    MC_GATHER_FOLDED(u128, 4, 4, 8, 2, 1)
    MC_GATHER_FOLDED(u128, 4, 8, 8, 2, 1)
    MC_GATHER_FOLDED(u128, 4, 16, 4, 2, 2)
    MC_GATHER_FOLDED(u128, 4, 16, 4, 2, 1)
    MC_GATHER_FOLDED(u128, 4, 16, 8, 2, 1)
    MC_GATHER_FOLDED(u128, 4, 4, 2, 3, 4)
    MC_GATHER_FOLDED(u128, 4, 4, 2, 3, 2)
    MC_GATHER_FOLDED(u128, 4, 4, 4, 3, 2)
    MC_GATHER_FOLDED(u128, 4, 4, 4, 3, 1)
    MC_GATHER_FOLDED(u128, 4, 4, 4, 4, 2)
    MC_GATHER_FOLDED(u128, 4, 4, 4, 4, 1)
    MC_GATHER_FOLDED(u128, 4, 8, 4, 3, 2)
    MC_GATHER_FOLDED(u128, 4, 8, 4, 3, 1)
    return nullptr;
}

}  // namespace mc

// gather_u128_8.cu -- instantiations of the neighbour-sum kernel for u128
// counts with first planes of 8-byte counts, one per lane layout that a
// level of k = 4..8 colours has.
#include "gather.cuh"

namespace mc {

GatherKernel gather_kernel_ptr_u128_8(int UB, int G, int NU, int P, int U, int MB)
{
    MC_GATHER_LAYOUT(u128, 8, 8, 16, 1, 1)
    MC_GATHER_LAYOUT(u128, 8, 8, 32, 2, 1)
    MC_GATHER_LAYOUT(u128, 8, 8, 32, 6, 1)
    MC_GATHER_LAYOUT(u128, 8, 16, 1, 1, 8)
    MC_GATHER_LAYOUT(u128, 8, 16, 1, 1, 4)
    MC_GATHER_LAYOUT(u128, 8, 16, 2, 1, 4)
    MC_GATHER_LAYOUT(u128, 8, 16, 2, 1, 2)
    MC_GATHER_LAYOUT(u128, 8, 16, 4, 1, 2)
    MC_GATHER_LAYOUT(u128, 8, 16, 4, 1, 1)
    MC_GATHER_LAYOUT(u128, 8, 16, 16, 1, 1)
    MC_GATHER_LAYOUT(u128, 8, 16, 32, 1, 1)
    MC_GATHER_LAYOUT(u128, 8, 16, 32, 2, 1)
    MC_GATHER_LAYOUT(u128, 8, 16, 32, 3, 1)
    MC_GATHER_FOLDED(u128, 8, 8, 8, 2, 1)
    MC_GATHER_FOLDED(u128, 8, 16, 8, 2, 1)
    MC_GATHER_FOLDED(u128, 8, 8, 4, 3, 2)
    MC_GATHER_FOLDED(u128, 8, 8, 4, 3, 1)
    return nullptr;
}

}  // namespace mc

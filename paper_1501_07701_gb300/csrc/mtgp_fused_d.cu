// Instantiations of the fused generation + statistics kernel for dense visits
// (DENSE), M = ceil(N/32) in {10, 11, 20} and G = 8 warps per CTA (see mtgp_fused.cuh).
#include "mtgp_fused.cuh"

namespace mtgp {

const void* fused_ptr_group_d(int M, int G)
{
    switch (M * 16 + G) {
    case 10 * 16 + 8: return (const void*)mtgp_fused_kernel<10, 8, true>;
    case 11 * 16 + 8: return (const void*)mtgp_fused_kernel<11, 8, true>;
    case 20 * 16 + 8: return (const void*)mtgp_fused_kernel<20, 8, true>;
    default: return nullptr;
    }
}

}  // namespace mtgp

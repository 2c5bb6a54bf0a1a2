// Instantiations of the fused generation + statistics kernel for dense visits
// (DENSE), M = ceil(N/32) = 44 and G = 8 warps per CTA (see mtgp_fused.cuh).
#include "mtgp_fused.cuh"

namespace mtgp {

const void* fused_ptr_group_f(int M, int G)
{
    switch (M * 16 + G) {
    case 44 * 16 + 8: return (const void*)mtgp_fused_kernel<44, 8, true>;
    default: return nullptr;
    }
}

}  // namespace mtgp

// Instantiations of the fused generation + statistics kernel for dense visits
// (DENSE), M = ceil(N/32) in {22, 23} and G = 8 warps per CTA (see mtgp_fused.cuh).
#include "mtgp_fused.cuh"

namespace mtgp {

const void* fused_ptr_group_e(int M, int G)
{
    switch (M * 16 + G) {
    case 22 * 16 + 8: return (const void*)mtgp_fused_kernel<22, 8, true>;
    case 23 * 16 + 8: return (const void*)mtgp_fused_kernel<23, 8, true>;
    default: return nullptr;
    }
}

}  // namespace mtgp

// Instantiations of the symmetric integer-code kernel (batches of up to
// kMaxBatch tensors; one tensor is a batch of one) for one clamp-set size
// (QUASAR_SS = 8, 4, 2 or 1 candidates, or 3 for the sets 3-3-2); compiled once
// per size, in parallel.
#include "recon_sym.cuh"

#if !defined(QUASAR_SS)
#error "QUASAR_SS must be defined"
#endif

#define QUASAR_CAT2(a, b) a##b
#define QUASAR_NAME(s) QUASAR_CAT2(sym_kernel_ss, s)

namespace quasar {

// Kernel entry for group size 4*epl.
const void* QUASAR_NAME(QUASAR_SS)(int epl)
{
    switch (epl) {
    case 8: return reinterpret_cast<const void*>(&k_recon_sym<8, kMaxBatch, QUASAR_SS>);
    case 16: return reinterpret_cast<const void*>(&k_recon_sym<16, kMaxBatch, QUASAR_SS>);
    case 32: return reinterpret_cast<const void*>(&k_recon_sym<32, kMaxBatch, QUASAR_SS>);
    case 64: return reinterpret_cast<const void*>(&k_recon_sym<64, kMaxBatch, QUASAR_SS>);
    default: return nullptr;
    }
}

}  // namespace quasar

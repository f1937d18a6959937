// Instantiations of the integer-code kernel for one chunk of 8 candidates
// (QUASAR_NCH = 1) or up to four (2), and one clamp-set size (QUASAR_SS = 4, 2
// or 1 candidates; with a single chunk also 8, or 3 for the sets 3-3-2);
// compiled once per pair, in parallel.
#include "recon_int.cuh"

#if !defined(QUASAR_NCH) || !defined(QUASAR_SS)
#error "QUASAR_NCH and QUASAR_SS must be defined"
#endif

#define QUASAR_CAT4(a, b, c, d) a##b##c##d
#define QUASAR_NAME(n, s) QUASAR_CAT4(int_kernel_nch, n, _ss, s)

namespace quasar {

// Kernel entry for group size 4*epl: one tensor or a batch of up to kMaxBatch
// tensors per launch; the AdamW-fused variant and the option variants (var) are
// built for batches.  nullptr where not built.
const void* QUASAR_NAME(QUASAR_NCH, QUASAR_SS)(int epl, bool batch, bool adam, bool var)
{
    constexpr int C = QUASAR_NCH;
    constexpr int S = QUASAR_SS;
    constexpr int B = kMaxBatch;
    if ((adam || var) && !batch) return nullptr;
    switch (epl) {
#define QUASAR_EPL(E)                                                                             \
    case E:                                                                                       \
        if (adam && var) return reinterpret_cast<const void*>(&k_recon_int<E, C, B, true, true, S>); \
        if (adam) return reinterpret_cast<const void*>(&k_recon_int<E, C, B, true, false, S>);    \
        if (var) return reinterpret_cast<const void*>(&k_recon_int<E, C, B, false, true, S>);     \
        if (!batch) return reinterpret_cast<const void*>(&k_recon_int<E, C, 1, false, false, S>); \
        return reinterpret_cast<const void*>(&k_recon_int<E, C, B, false, false, S>);
    QUASAR_EPL(8)
    QUASAR_EPL(16)
    QUASAR_EPL(32)
    QUASAR_EPL(64)
#undef QUASAR_EPL
    default: return nullptr;
    }
}

}  // namespace quasar

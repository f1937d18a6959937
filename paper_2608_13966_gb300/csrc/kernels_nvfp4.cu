// Instantiations of the NVFP4 kernel and of the tensor-absmax kernels.
#include "recon_nvfp4.cuh"

namespace quasar {

const void* nvfp4_kernel(bool batch)
{
    return batch ? reinterpret_cast<const void*>(&k_recon_nvfp4<kMaxBatch, NoAhead>)
                 : reinterpret_cast<const void*>(&k_recon_nvfp4<1, NoAhead>);
}

const void* nvfp4_amax_ahead_kernel()
{
    return reinterpret_cast<const void*>(&k_recon_nvfp4<kMaxStage, AmaxBatch<kMaxStage>>);
}

const void* nvfp4_adamw_ahead_kernel()
{
    return reinterpret_cast<const void*>(&k_recon_nvfp4<kMaxStage, AdamwBatch<kMaxStage>>);
}

const void* amax_kernel(bool batch)
{
    return batch ? reinterpret_cast<const void*>(&k_amax<kMaxStage>)
                 : reinterpret_cast<const void*>(&k_amax<1>);
}

const void* adamw_amax_kernel() { return reinterpret_cast<const void*>(&k_adamw_amax<kMaxStage>); }

const void* amax_init_kernel(bool batch)
{
    return batch ? reinterpret_cast<const void*>(&k_amax_init<kMaxBatch>)
                 : reinterpret_cast<const void*>(&k_amax_init<1>);
}

const void* amax_to_scale_kernel(bool batch)
{
    return batch ? reinterpret_cast<const void*>(&k_amax_to_scale<kMaxBatch>)
                 : reinterpret_cast<const void*>(&k_amax_to_scale<1>);
}

}  // namespace quasar

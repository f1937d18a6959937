// Instantiations of the NVFP4 kernel and of the tensor-absmax kernels.
#include "recon_adamw.cuh"
#include "recon_nvfp4.cuh"

namespace quasar {

const void* nvfp4_kernel(bool batch)
{
    return batch ? reinterpret_cast<const void*>(&k_recon_nvfp4<kMaxBatch>)
                 : reinterpret_cast<const void*>(&k_recon_nvfp4<1>);
}

const void* amax_kernel(bool batch)
{
    return batch ? reinterpret_cast<const void*>(&k_amax<kMaxBatch>)
                 : reinterpret_cast<const void*>(&k_amax<1>);
}

const void* adamw_amax_kernel() { return reinterpret_cast<const void*>(&k_adamw_amax<kMaxBatch>); }

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

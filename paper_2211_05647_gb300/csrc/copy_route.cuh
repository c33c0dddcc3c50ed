// copy_route.cuh -- which copies between the solver's arrays and a caller's
// memory run as kernels (rows.cu).  Host code, standard library only.
#pragma once

#include <cstddef>
#include <cstdint>

namespace fp {

// the device the arrays live on and its number of SMs
struct CopyHome {
    int dev, sms;
};

// Whether kernels of the arrays' device may read and write the caller's memory: device memory of that very device,
// whichever device is current in the calling thread (a copy engine reaches other places).
inline bool kernel_reaches(bool is_device_memory, int their_dev, const CopyHome &home)
{
    return is_device_memory && their_dev == home.dev;
}

// blocks of a linear copy kernel: one pass while they fit, else eight a SM
inline uint32_t copy_blocks(uint32_t units, uint32_t units_per_block, const CopyHome &home)
{
    const uint32_t one_pass = (units + units_per_block - 1) / units_per_block, cap = 8u * (uint32_t)home.sms;
    return one_pass < cap ? one_pass : cap;
}

}  // namespace fp

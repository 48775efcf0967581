// The library's memory pool (pool.cu): where scratch and plans come from.
#pragma once

#include <cuda_runtime_api.h>
#include <stddef.h>

namespace rbffd {

// Stream-ordered allocations come from a memory pool of the library's own, one
// per device.  The device's default pool gives everything back to the driver at
// each synchronisation, so every call that ends with one - most here do - paid
// 100 to 200 us to map its scratch again: set-up of a 10k-node problem (supports,
// weights, plan, time step) 1.73 ms with it, 1.37 without.  The library's pool keeps at most
// POOL_KEEP bytes that are not in use; what is above goes back at each
// synchronisation, the rest when an allocation fails and when the library is unloaded.
// Safe from any thread and stream (the driver orders reuse between streams).
static constexpr unsigned long long POOL_KEEP = 128ull << 20;
cudaError_t pool_alloc(void** p, size_t bytes, cudaStream_t s);

// Frees up to n arrays of one device (null ones are skipped), whichever device is
// current, when all work on theirs is done, as cudaFree would; what the pool then
// holds above POOL_KEEP goes back before it returns.
void pool_free(void* const* p, int n);

}  // namespace rbffd

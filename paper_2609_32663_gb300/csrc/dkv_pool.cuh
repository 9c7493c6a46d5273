// Device memory of plans (dkv_pool.cu).
#pragma once

#include <cstddef>
#include <cuda_runtime.h>

namespace dkv {

// Process-unique ID of the calling thread's CUDA context.
cudaError_t current_context_id(unsigned long long* id);

// One allocation of a plan.
struct PlanMemory {
    void* ptr = nullptr;
    size_t bytes = 0;
    unsigned long long context = 0;
};

cudaError_t plan_alloc(PlanMemory* m, size_t bytes);
// No-op for none. idle: the device has finished all work that uses the memory (else it
// is not kept for another plan).
void plan_free(const PlanMemory& m, bool idle);

}  // namespace dkv

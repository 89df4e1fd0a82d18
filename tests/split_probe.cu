// The set-up sources with two additions for tests/test_gpu_split_table.py: device allocations
// that fail on request, and a device bucket table put out of order.
#include <cub/cub.cuh>

namespace {
int g_allocations_left = -1;   // -1: no limit
cudaError_t counted_malloc(void **p, size_t bytes)
{
    if (g_allocations_left == 0) return cudaErrorMemoryAllocation;
    if (g_allocations_left > 0) g_allocations_left--;
    return cudaMalloc(p, bytes);
}
}  // namespace
#define cudaMalloc(p, bytes) counted_malloc(reinterpret_cast<void **>(p), bytes)
#include "sci_setup.cu"
#undef cudaMalloc

extern "C" void probe_limit_allocations(int left) { g_allocations_left = left; }

// moves the last bucket of the full (N-2) table, as it is, before the first one
extern "C" int probe_last_bucket_first(sci_ctx *ctx)
{
    std::vector<uint32_t> pos(ctx->e2);
    if (cudaMemcpy(pos.data(), ctx->e2_pos, 4 * pos.size(), cudaMemcpyDeviceToHost) != cudaSuccess) return -1;
    std::rotate(pos.begin(), pos.end() - sci::pos_size(pos.back()), pos.end());
    return cudaMemcpy(ctx->e2_pos, pos.data(), 4 * pos.size(), cudaMemcpyHostToDevice) == cudaSuccess ? 0 : -1;
}

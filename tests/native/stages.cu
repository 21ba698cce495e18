// Single stages of the library behind C entries, for tests that run a stage
// with a status word of their choice.  Linked with the library's objects.
#include <cuda_runtime.h>

#include "compress.cuh"
#include "coop.cuh"
#include "msid.cuh"
#include "sort.cuh"

using namespace msc;

namespace {

// A barrier that waits for a block that does not exist: its wait runs out.
__global__ void k_lonely_barrier(uint32_t* count, int32_t* passed, int32_t* status) {
    GridBarrier bar{count, 2, 0};
    const bool ok = grid_barrier(bar, status);
    if (threadIdx.x == 0) *passed = ok;
}

template <typename F>
size_t sized(F f) {
    Sizer s;
    f(s);
    return s.used;
}

}  // namespace

extern "C" {

MSC_API size_t stage_order_bytes(int64_t n) {
    return sized([&](Sizer& s) {
        for (int i = 0; i < 4; ++i) s.take<int32_t>(n);
        size_sort_scratch(s, n);
    });
}

MSC_API int stage_order(const float* f, int64_t n, int32_t* order, void* ws, size_t bytes, int32_t* status, void* stream) {
    Carver c(ws, bytes);
    uint32_t* ka = c.take<uint32_t>(n);
    int32_t* ia = c.take<int32_t>(n);
    uint32_t* kb = c.take<uint32_t>(n);
    int32_t* ib = c.take<int32_t>(n);
    const SortScratch sc = carve_sort_scratch(c, n);
    return run_order(f, n, order, ka, ia, kb, ib, sc, status, static_cast<cudaStream_t>(stream));
}

MSC_API size_t stage_compress_bytes(int64_t n) {
    return sized([&](Sizer& s) { size_compress_scratch(s, n, 1); });
}

// Pointers as the stencil makes them: followed without tests.
MSC_API int stage_compress(int32_t* ptr, int32_t n, void* ws, size_t bytes, int32_t* status, void* stream) {
    Carver c(ws, bytes);
    const CompressScratch sc = carve_compress_scratch(c, n, 1);
    CompressTune tune;
    tune.trusted = true;
    return run_compress(&ptr, 1, n, sc, status, static_cast<cudaStream_t>(stream), tune);
}

MSC_API size_t stage_ms_id_bytes(int64_t n) {
    return sized([&](Sizer& s) { size_ms_scratch(s, n); });
}

MSC_API int stage_ms_id(const int32_t* asc, const int32_t* desc, int32_t n, int32_t* ms, int32_t* cells, void* ws,
                        size_t bytes, int32_t* status, void* stream) {
    Carver c(ws, bytes);
    const MsScratch sc = carve_ms_scratch(c, n);
    return run_ms_id(asc, desc, n, ms, cells, sc, false, status, static_cast<cudaStream_t>(stream));
}

MSC_API int stage_lonely_barrier(uint32_t* count, int32_t* passed, int32_t* status, void* stream) {
    k_lonely_barrier<<<1, 64, 0, static_cast<cudaStream_t>(stream)>>>(count, passed, status);
    return cudaPeekAtLastError() == cudaSuccess ? 0 : -1;
}

}  // extern "C"

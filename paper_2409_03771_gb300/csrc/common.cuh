// Internal helpers shared by the sm_103a kernels of the msc library.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include "msc.h"

namespace msc {

constexpr int kWarp = 32;

// ----------------------------------------------------------------------------
// device status word: the first error recorded wins, except that a wait that
// ran out (record_give_up) replaces any other
__device__ __forceinline__ void record_error(int32_t* status, int32_t code) {
    if (status) atomicCAS(status, MSC_OK, code);
}

// A bounded wait (grid barrier, look-back, bulk copy) that ran out leaves its
// stage's outputs unfinished: indices in them may be anything.  The call's
// later stages are already enqueued, so those that use such an index without
// a test of their own look here first and leave their work undone.
__device__ __forceinline__ void record_give_up(int32_t* status) {
    if (status) atomicExch(status, MSC_ERR_INTERNAL);
}

__device__ __forceinline__ bool stage_gave_up(const int32_t* status) {
    return status && __ldca(status) == MSC_ERR_INTERNAL;  // written by an earlier kernel: one L2 read per SM
}

// The same for every thread of the block (kernels with barriers of their own).
__device__ __forceinline__ bool stage_gave_up_block(const int32_t* status) {
    return __syncthreads_or(threadIdx.x == 0 && stage_gave_up(status)) != 0;
}

// Debug builds (-DMSC_DEBUG_BOUNDS) check data-dependent addresses before
// the access: a violation records `code` in the status word and skips the
// access.  Release builds compile the check away.
#if defined(MSC_DEBUG_BOUNDS) || defined(MSC_GUARDS)
#define MSC_GUARD(cond, status, code) if (!(cond)) record_error((status), (code)); else
#else
#define MSC_GUARD(cond, status, code)
#endif

__device__ __forceinline__ uint32_t lanemask_lt() {
    uint32_t m;
    asm volatile("mov.u32 %0, %%lanemask_lt;" : "=r"(m));
    return m;
}

__device__ __forceinline__ unsigned long long ld_volatile_u64(const unsigned long long* p) {
    unsigned long long v;
    asm volatile("ld.volatile.global.u64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
    return v;
}

__device__ __forceinline__ void st_volatile_u64(unsigned long long* p, unsigned long long v) {
    asm volatile("st.volatile.global.u64 [%0], %1;" ::"l"(p), "l"(v) : "memory");
}

__device__ __forceinline__ int32_t ld_cached_s32(const int32_t* p) {
    int32_t v;
    asm volatile("ld.global.ca.s32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}

__device__ __forceinline__ int32_t ld_volatile_s32(const int32_t* p) {
    int32_t v;
    asm volatile("ld.volatile.global.s32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}

// A block's walk over the tiles first, first + step, first + 2 step, ... of
// a tx x ty x .. grid of tiles (x fastest; counts fit 32 bits, as every tile
// holds a vertex): the coordinates advance by the step's own, so a tile
// costs a few additions instead of two divisions.
struct TileWalk {
    int32_t tx, ty;
    int32_t x, y, z;     // the current tile
    int32_t sx, sy, sz;  // the step
    __device__ __forceinline__ TileWalk(int32_t tx_, int32_t ty_, uint32_t first, uint32_t step) : tx(tx_), ty(ty_) {
        split(first, x, y, z);
        split(step, sx, sy, sz);
    }
    __device__ __forceinline__ void split(uint32_t t, int32_t& a, int32_t& b, int32_t& c) const {
        const uint32_t q = t / (uint32_t)tx;
        a = (int32_t)(t - q * (uint32_t)tx);
        c = (int32_t)(q / (uint32_t)ty);
        b = (int32_t)(q - (uint32_t)c * (uint32_t)ty);
    }
    __device__ __forceinline__ void advance() {
        x += sx;
        y += sy;
        z += sz;
        if (x >= tx) {
            x -= tx;
            ++y;
        }
        if (y >= ty) {
            y -= ty;
            ++z;
        }
    }
};

// ----------------------------------------------------------------------------
// host side
struct Device {
    int id = -1;
    int sms = 0;
    int max_smem_optin = 0;
};

// Counts one kernel launch and, while tracing is on, brackets it with CUDA
// events on its stream (see trace.cu).  Construct right before the launch
// and let it go out of scope right after.
class TraceScope {
   public:
    TraceScope(const char* label, cudaStream_t s);
    ~TraceScope();
    TraceScope(const TraceScope&) = delete;
    TraceScope& operator=(const TraceScope&) = delete;

   private:
    const char* label_;
    cudaStream_t stream_;
    cudaEvent_t a_ = nullptr, b_ = nullptr;
};

// Launch counter adjustments: kernels recorded into a CUDA graph are
// counted when the graph is replayed, not when they are captured.
void add_launches(long long k);
unsigned long long launch_count();

// Properties of the current device (cached per device id).
const Device& current_device();

// Resident blocks per SM of a kernel on the current device.  The runtime
// works this out anew on every call (1.5 us of host time, five to ten times
// per segmentation), so the answers are remembered per device.
cudaError_t max_blocks_per_sm(int* out, const void* kernel, int threads, size_t smem);

template <typename K>
cudaError_t max_blocks_per_sm(int* out, K* kernel, int threads, size_t smem) {
    return max_blocks_per_sm(out, reinterpret_cast<const void*>(kernel), threads, smem);
}

// SMs that kernels on a stream can use: those of the device, or of the
// stream's green context (a part of the SMs that a program has set aside).
int stream_sms(cudaStream_t s);

// Bump-pointer carving of a caller workspace (256-byte aligned pieces).
struct Carver {
    char* base;
    size_t used = 0;
    size_t cap;
    Carver(void* p, size_t bytes) : base(static_cast<char*>(p)), cap(bytes) {}
    template <typename T>
    T* take(size_t count) {
        size_t off = (used + 255) & ~size_t(255);
        used = off + count * sizeof(T);
        return reinterpret_cast<T*>(base + off);
    }
    bool ok() const { return used <= cap; }
};

// Size-only twin of Carver, used by msc_workspace_bytes.
struct Sizer {
    size_t used = 0;
    template <typename T>
    void take(size_t count) {
        size_t off = (used + 255) & ~size_t(255);
        used = off + count * sizeof(T);
    }
};

inline int ceil_log2(int64_t n) {
    int b = 0;
    while ((int64_t(1) << b) < n) ++b;
    return b;
}

inline int64_t ceil_div(int64_t a, int64_t b) { return (a + b - 1) / b; }

#define MSC_TRY(expr)                                  \
    do {                                               \
        if ((expr) != cudaSuccess) return MSC_ERR_CUDA; \
    } while (0)

#define MSC_LAUNCHED()                                    \
    do {                                                  \
        if (cudaPeekAtLastError() != cudaSuccess) {       \
            cudaGetLastError();                           \
            return MSC_ERR_CUDA;                          \
        }                                                 \
    } while (0)

}  // namespace msc

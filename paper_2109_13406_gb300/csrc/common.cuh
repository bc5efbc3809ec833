// Shared host/device utilities of libmpdd: per-thread stream and error state,
// CUDA error mapping, BLAS-style flag parsing, launch helpers.
#pragma once

#include <cuda_runtime.h>

#include <cstdarg>
#include <cstdint>
#include <cstdio>

#include "mpdd.h"

namespace mpdd {

// Per-thread library state: the stream calls are issued on and the text of
// the last error (mp_dd_set_stream / mp_dd_last_error).
struct ThreadState {
    cudaStream_t stream = nullptr;
    char msg[512] = {0};
};

ThreadState &tls();

// Record a formatted message for mp_dd_last_error and return `code`.
int fail(int code, const char *fmt, ...);

// Map a CUDA runtime error to MP_DD_ERR_CUDA_BASE + e, recording `what`.
int cuda_fail(cudaError_t e, const char *what);

// Check for a launch error right after a kernel launch.
inline int check_launch(const char *what) {
    cudaError_t e = cudaGetLastError();
    return e == cudaSuccess ? 0 : cuda_fail(e, what);
}

// Clear the per-thread error text at the start of a call.
inline void clear_error() { tls().msg[0] = 0; }

// Case-insensitive comparison of the first character of a BLAS flag.
inline bool flag_is(const char *f, char c) {
    if (f == nullptr) return false;
    char x = f[0];
    if (x >= 'a' && x <= 'z') x = (char)(x - 'a' + 'A');
    return x == c;
}

// 'N' -> 0, 'T' or 'C' -> 1, anything else -> -1.
inline int trans_flag(const char *f) {
    if (flag_is(f, 'N')) return 0;
    if (flag_is(f, 'T') || flag_is(f, 'C')) return 1;
    return -1;
}

// 'U' -> 1, 'L' -> 2, anything else -> -1.
inline int uplo_flag(const char *f) {
    if (flag_is(f, 'U')) return 1;
    if (flag_is(f, 'L')) return 2;
    return -1;
}

// Kernels of one call that follow one another are launched chained: the next
// one's blocks may start while the last blocks of this one still run, and
// every kernel of the chain begins with chain_begin(), which waits until the
// kernel before it has completed and its writes are visible (and that one
// waited for its own predecessor in the same way), then lets the next one
// start.  No kernel reads or writes memory before it.  A kernel launched any
// other way behind the chain waits for all of it as usual, and chain_begin()
// does nothing in a kernel that was not launched chained.  This hides the
// launch latency between kernels of 2 to 20 us: CRT Rgemm 512^3 87 -> 73 us,
// Rgemm 96 x 80 x 70 59.4 -> 58.0.  Launches of many short blocks
// stay unchained (the wait costs each of them more than it hides), and so do
// large ones that live on L1 behind a kernel that takes all of the shared
// memory: a block that starts under that kernel's configuration keeps its
// small L1 (an 8192 product's residues: 2.0 ms unchained, 2.15 chained).
__device__ __forceinline__ void chain_begin() {
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}

constexpr unsigned kChainBlocks = 4096;   // ~27 per SM

template <typename... P, typename... A>
inline cudaError_t launch_chained_if(bool chain, void (*f)(P...), dim3 grid, dim3 block,
                                     size_t smem, cudaStream_t st, A &&...args) {
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = grid;
    cfg.blockDim = block;
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = at;
    cfg.numAttrs = chain && (uint64_t)grid.x * grid.y * grid.z <= kChainBlocks ? 1 : 0;
    return cudaLaunchKernelEx(&cfg, f, static_cast<P>(args)...);
}

template <typename... P, typename... A>
inline cudaError_t launch_chained(void (*f)(P...), dim3 grid, dim3 block, size_t smem,
                                  cudaStream_t st, A &&...args) {
    return launch_chained_if(true, f, grid, block, smem, st, static_cast<P>(args)...);
}

// check_launch for launch_chained's result.
inline int chained_ok(cudaError_t e, const char *what) {
    if (e != cudaSuccess) {
        cudaGetLastError();
        return cuda_fail(e, what);
    }
    return check_launch(what);
}

inline int64_t imax(int64_t a, int64_t b) { return a > b ? a : b; }
inline int64_t ceil_div(int64_t a, int64_t b) { return (a + b - 1) / b; }

inline bool dd_is_zero(mp_dd x) { return x.hi == 0.0 && x.lo == 0.0; }
inline bool dd_is_one(mp_dd x) { return x.hi == 1.0 && x.lo == 0.0; }

// Verify once per process that a device of compute capability 10.3 is
// current; returns 0 or MP_DD_ERR_NO_DEVICE.
int require_device();

// Number of SMs of the current device (cached).
int sm_count();
// Stream-ordered allocation from the library's own pools; free with
// cudaFreeAsync.  kPoolHost (the host forms' buffers, small exchange buffers):
// freed memory stays mapped for later calls.  kPoolScratch (workspaces of the
// factorisations' and solves' tensor-core updates): at most kScratchKeep bytes
// of freed memory stay mapped past a synchronisation.
enum PoolKind { kPoolHost = 0, kPoolScratch = 1, kPoolKinds = 2 };
constexpr uint64_t kScratchKeep = 2ull << 30;
cudaError_t pool_alloc(void **ptr, size_t bytes, cudaStream_t st, PoolKind kind = kPoolHost);

}  // namespace mpdd

// tg_error.hpp -- errors of the host code of libtg.
#pragma once

#include <cstdio>
#include <cuda_runtime.h>

#include "tg.h"

namespace tg {

// Internal error carrying a tg_status; caught at every extern "C" entry.
struct Error {
    tg_status status;
    const char *what;
    bool from_cuda = false;     // message already recorded by throw_cuda
};

// Text of the calling thread's last failed entry (tg_last_error).
inline thread_local char tl_last_error[256] = "";

inline void throw_cuda(cudaError_t e, const char *what) {
    if (e == cudaSuccess) return;
    (void)cudaGetLastError();   // clear the sticky-free error state
    std::snprintf(tl_last_error, sizeof tl_last_error, "%s: %s", what, cudaGetErrorString(e));
    throw Error{e == cudaErrorMemoryAllocation ? TG_ERR_OOM : TG_ERR_CUDA, what, true};
}

// For calls of destructors, which may run because an earlier call failed: an
// error of theirs must not be what the next entry's cudaGetLastError finds.
inline void forget(cudaError_t e) {
    if (e != cudaSuccess) (void)cudaGetLastError();
}

}  // namespace tg

#define TG_CK(call) ::tg::throw_cuda((call), #call)

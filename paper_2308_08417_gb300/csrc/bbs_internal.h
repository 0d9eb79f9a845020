// Helpers the API translation unit offers to the library's other host code.
#pragma once

#include <cuda_runtime.h>

#include "../../include/bbs.h"

namespace bbs {
// Set the thread's last-error message and return s.
bbs_status record_error(bbs_status s, const char* msg);
// CUDA device a handle is bound to.
int handle_device(const bbs_handle* h);
// Lets fn use smem bytes of dynamic shared memory on the current device. The limit
// belongs to the function, which calls of other sizes, other objects and other
// threads use too, and a captured launch is checked against it later: it is only
// ever raised.
cudaError_t allow_smem(const void* fn, size_t smem);
}  // namespace bbs

// Host interface between the launchers of libframefb (framefb_cuda.cu) and
// the group-transform path (framefb_grp.cu).  Internal: not part of the C ABI.
#pragma once
#include <cuda_runtime.h>

#include "framefb.h"

namespace ffb_host {

// Whether a matrix of a call runs on the group-transform kernel.
bool grp_takes(const framefb_mat& M, int32_t ops, framefb_dtype dt);

// Validate the path's matrices and report the workspace they need (bytes;
// the launches run one after another and share it).
framefb_status grp_check(const framefb_mat* mats, int32_t nmats, int32_t ops, framefb_dtype dt, size_t* ws_need);

// Queue the path on `st` (after grp_check).
framefb_status grp_run(const framefb_mat* mats, int32_t nmats, int32_t ops, framefb_dtype dt, void* ws,
                       cudaStream_t st);

}  // namespace ffb_host

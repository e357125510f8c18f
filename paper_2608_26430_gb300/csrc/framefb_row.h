// Host interface between the launchers of libframefb (framefb_cuda.cu) and
// the row-transform path (framefb_row.cu).  Internal: not part of the C ABI.
#pragma once
#include <cuda_runtime.h>

#include <memory>
#include <string>
#include <vector>

#include "framefb.h"

namespace ffb_host {

// Whether a matrix of a call runs on the row-transform kernel.
bool row_takes(const framefb_mat& M, int32_t ops, framefb_dtype dt);

// The launches of a call, with their parameters filled.
struct RowLaunches;
using RowReady = std::shared_ptr<RowLaunches>;

// Validate the path's matrices, report the workspace they need (bytes; the
// launches run one after another and share it), and hand the prepared
// launches on through `keep`.
framefb_status row_check(const framefb_mat* mats, int32_t nmats, int32_t ops, framefb_dtype dt, size_t* ws_need,
                         RowReady* keep = nullptr);

// Queue the launches of row_check on `st` (none if `ready` is empty).
framefb_status row_run(const RowReady& ready, void* ws, cudaStream_t st);

// Kernels row_run launches for `ops` (appended to `out`, no duplicates).
framefb_status row_kernel_names(const framefb_mat* mats, int32_t nmats, int32_t ops, framefb_dtype dt,
                                std::vector<std::string>& out);

// Bounded waits of the row kernel that gave up on the current device.
framefb_status row_wait_timeouts(uint32_t* count);

}  // namespace ffb_host

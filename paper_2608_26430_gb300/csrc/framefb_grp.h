// Host interface between the launchers of libframefb (framefb_cuda.cu) and
// the group-transform path (framefb_grp.cu).  Internal: not part of the C ABI.
#pragma once
#include <cuda_runtime.h>

#include <memory>

#include "framefb.h"

namespace ffb_host {

// Whether a plan fits the group-transform kernel, with whole or compacted buffers,
// and whether a matrix of a call, of a plan of this kind, runs on it.
enum class GrpKind { none, whole, big };
GrpKind grp_kind(const framefb_plan* plan);
bool grp_takes(GrpKind kind, const framefb_mat& M, int32_t ops, framefb_dtype dt);

// The launches of a call, with their parameters filled.
struct GrpLaunches;
using GrpReady = std::shared_ptr<GrpLaunches>;

// Validate the path's matrices, report the workspace they need (bytes; the
// launches run one after another and share it), and hand the prepared
// launches on through `keep`.
framefb_status grp_check(const framefb_mat* mats, int32_t nmats, int32_t ops, framefb_dtype dt, size_t* ws_need,
                         GrpReady* keep = nullptr);

// Queue the launches of grp_check on `st` (none if `ready` is empty).
framefb_status grp_run(const GrpReady& ready, void* ws, cudaStream_t st);

}  // namespace ffb_host

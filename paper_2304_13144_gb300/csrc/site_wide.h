// FP64 and dual-number per-neighborhood pass with the fewest floating-point operations
// (site_wide.cu).
#pragma once

#include <cuda_runtime.h>

#include "mtp_internal.h"

namespace mtp {

// bytes of workspace the pass needs for n_work neighborhoods (moments, then their adjoints), 0 if
// the model's shape has no such pass
size_t wide_workspace(const mtp_model* m, int64_t n_work, bool fp64, bool tangent);

// Outputs as run_sites (o.wide = the workspace above): energies/forces/virials, FP64 rows, or with
// `tangent` the partial gradients, whose number of rows is returned in *n_part (at most max_part).
// Returns false (nothing launched) where it does not apply; the caller then takes the generic kernel.
bool run_sites_wide(mtp_model* m, const mtp_batch* b, const mtp_nbr* nb, bool fp64, const SiteOutputs& o, bool tangent,
                    int64_t max_part, int64_t* n_part, cudaStream_t s);

void wide_prepare(mtp_model* m);

}  // namespace mtp

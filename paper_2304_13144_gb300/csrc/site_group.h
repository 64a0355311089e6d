// Grouped contraction of the three-kernel mixed pass (site_group.cu): four neighborhoods side by
// side in the lanes' 128-bit shared-memory words.
#pragma once

#include <cuda_runtime.h>

#include "mtp_internal.h"

namespace mtp {

// the grouped contraction's part of the schedule fits this model (always, where upload_schedule
// packed it and one group's arrays fit shared memory beside the round headers)
bool contract_group_available(const DevSchedule& d);

// eqs. 2, 5-6 and their adjoint for n_work neighborhoods: moments mom[n_work x ldm] in slot order
// (slot_comp: slot -> value index) are overwritten by dV/dM; V_i and the basis part of the rows
// go to `o`.  Returns where the schedule's words were read from (1 shared, 2 global, 3 tensor
// memory, the numbering of mtp_get_split_shape).
int run_contract_group(const DevSchedule& d, const SiteOutputs& o, const int* type, int64_t n_work, float* mom,
                       int ldm, const int* slot_comp, cudaStream_t s);

}  // namespace mtp

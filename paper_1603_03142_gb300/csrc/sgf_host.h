// sgf_host.h -- host-side helpers shared by the translation units of the C ABI.
#pragma once
#include <cuda_runtime.h>
#include <string>

#include "../../include/sgf.h"

namespace sgf {
// Records a printf-style message as the calling thread's last error (sgf_last_error)
// and returns s.
sgf_status fail(sgf_status s, const char *fmt, ...);
// fail() for a CUDA runtime error: SGF_ENOMEM for an allocation failure, SGF_ECUDA otherwise.
sgf_status cuda_fail(cudaError_t e, const char *what);
// sgf_plan_create_ex and sgf_plan_estimate with the choice of passes for the cross-level
// pairs: whole_grid keeps the whole-grid passes (and their spectra) where block
// convolutions would run.
sgf_status nest_plan_create(const sgf_nest_desc *desc, sgf_precision precision, uint32_t flags, bool whole_grid,
                            sgf_plan **out);
sgf_status nest_plan_estimate(const sgf_nest_desc *desc, sgf_precision precision, uint32_t flags, bool whole_grid,
                              size_t *workspace_bytes, size_t *spectra_bytes, size_t *build_bytes);
}  // namespace sgf

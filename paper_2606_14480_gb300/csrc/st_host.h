// st_host.h -- host-side helpers shared by the library's translation units.
#pragma once

#include <string>

#include "st.h"
#include "st_device.cuh"
#include "st_kernels.cuh"

namespace st {

// CTAs of the seeding kernel: threads, whether with more registers each, what
// their shared memory holds, and how many an SM takes.
struct SeedShape {
    bool wide = false;
    int threads = 0, smem_hits = 0, tbl_smem = 0, key_smem = 0, velo_smem = 0;
    size_t smem = 0;
    int bps = 0;
};

// The shapes a configuration may run with: [0] as configured, then ever fewer
// CTAs per SM, for smaller batches.  Returns how many; with `bps`, how many CTAs
// of each an SM takes (after set_smem_limits).
int seed_shapes(const st_config& c, SeedShape out[kSeedShapes], bool bps);

// The shape for a batch of `items` (event, half) items when at most `max_ctas`
// CTAs may run (their scratch).
const SeedShape& pick_seed_shape(const SeedShape* shapes, int n, const st_config& c, int64_t items, int n_sms,
                                 int64_t max_ctas);

}  // namespace st

// Derive the device constants from a configuration (validates it; false and a
// message on an invalid configuration).
bool derive_params(const st_config& c, st::DevParams& P, std::string& err);

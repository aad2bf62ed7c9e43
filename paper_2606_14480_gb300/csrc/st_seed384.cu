// st_seed384.cu -- the seeding kernel for CTAs of up to 384 threads.
#include "st_seed.cuh"

namespace st {

SeedKernel seed_kernel_384(bool seq, bool fused) { return seed_kernel_of<384, kSeedRegs384>(seq, fused); }

}  // namespace st

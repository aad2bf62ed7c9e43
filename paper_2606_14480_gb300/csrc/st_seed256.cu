// st_seed256.cu -- the seeding kernel for CTAs of up to 256 threads.
#include "st_seed.cuh"

namespace st {

SeedKernel seed_kernel_256(bool seq, bool fused) { return seed_kernel_of<256, kSeedRegs256>(seq, fused); }

}  // namespace st

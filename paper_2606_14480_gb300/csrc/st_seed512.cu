// st_seed512.cu -- the seeding kernel for CTAs of up to 512 threads.
#include "st_seed.cuh"

namespace st {

SeedKernel seed_kernel_512(bool seq, bool fused) { return seed_kernel_of<512, kSeedRegs512>(seq, fused); }

}  // namespace st

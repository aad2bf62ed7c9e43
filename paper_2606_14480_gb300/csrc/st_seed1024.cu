// st_seed1024.cu -- the seeding kernel for CTAs of up to 1024 threads.
#include "st_seed.cuh"

namespace st {

SeedKernel seed_kernel_1024(bool seq, bool fused) { return seed_kernel_of<1024, kSeedRegs1024>(seq, fused); }

}  // namespace st

// st_seed448.cu -- the seeding kernel for CTAs of up to 448 threads.
#include "st_seed.cuh"

namespace st {

SeedKernel seed_kernel_448(bool seq, bool fused) { return seed_kernel_of<448, kSeedBlocks448>(seq, fused); }

}  // namespace st

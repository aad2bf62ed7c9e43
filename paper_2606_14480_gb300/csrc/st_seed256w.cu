// st_seed256w.cu -- the seeding kernel for CTAs of up to 256 threads, four to
// an SM.
#include "st_seed.cuh"

namespace st {

SeedKernel seed_kernel_256w(bool seq, bool fused) { return seed_kernel_of<256, kSeedRegs256w>(seq, fused); }

}  // namespace st

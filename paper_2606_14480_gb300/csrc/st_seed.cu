// st_seed.cu -- sizes of the seeding kernel's memory and the choice of its
// instantiation.
#include "st_seed.cuh"

namespace st {

size_t seed_smem_bytes(int threads, int smem_hits, int tbl_smem, int key_smem) {
    return seed_smem_size(threads, smem_hits, tbl_smem, key_smem);
}
size_t seed_slot_bytes(int cand_cap, int uv_cap, int tbl_cap, int max_hits) {
    return seed_slot_size(cand_cap, uv_cap, tbl_cap, max_hits);
}

// The shared memory and the scratch per CTA that a configuration is accepted
// by: what an earlier layout of the kernel took (9216 bytes of bucket tables, 12
// triplet keys per thread of 512, 40 bytes per stored UV combination, and so
// on), in which the interface states its limits, so that what is accepted and
// what is refused does not change with the layout.  The present one takes less
// of both wherever a limit is near, but can take more of a small configuration
// (512 threads without staged hits: 36 KB against 18): the callers take the
// larger of this and what is really needed.
size_t seed_smem_limit_bytes(int threads, int smem_hits, int tbl_smem, int key_smem) {
    return align16(sizeof(float) * smem_hits) + 9216 + sizeof(ull) * (tbl_smem + key_smem) +
           sizeof(float) * 6 * key_smem + sizeof(int) * 3 * threads + sizeof(int) * (36 + 16);
}
size_t seed_slot_limit_bytes(int cand_cap, int max_xhits) {
    return align16(sizeof(int) * 16 * size_t(cand_cap)) +
           sizeof(ull) * (size_t(max_xhits) + cand_cap + size_t(kTripPerCand) * cand_cap) +
           16 + (2 * sizeof(uint4) + sizeof(uint2)) * kUvStore + sizeof(float) * 6 * size_t(cand_cap) + 8 +
           sizeof(ull) * 12 * 512 + 9 * size_t(cand_cap) + 4 + sizeof(uint32_t) * ((size_t(max_xhits) + 31) / 32);
}

SeedKernel seed_kernel(int threads, bool wide, bool seq, bool fused) {
    return threads <= 256 ? (wide ? seed_kernel_256w(seq, fused) : seed_kernel_256(seq, fused))
           : threads <= 384 ? seed_kernel_384(seq, fused)
           : threads <= 512 ? seed_kernel_512(seq, fused) : seed_kernel_1024(seq, fused);
}

}  // namespace st

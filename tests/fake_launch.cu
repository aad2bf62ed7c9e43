// Stand-ins for the kernels' sizes, occupancies and launchers (see
// fake_cuda.cpp): a launch is an operation of its stream.
#include "st_host.h"
#include "st_kernels.cuh"
#include "st_ut.cuh"

cudaError_t fake_launch(const char* name, cudaStream_t s, cudaEvent_t started);

namespace st {
size_t build_smem_bytes(int bins, int hits) { return size_t(8) * 24 * bins + size_t(10) * hits; }
size_t seed_smem_bytes(int threads, int hits, int tbl, int key) { return size_t(4) * hits + 8 * tbl + 32 * key + 32 * threads; }
size_t seed_smem_limit_bytes(int threads, int hits, int tbl, int key) { return seed_smem_bytes(threads, hits, tbl, key); }
size_t seed_slot_bytes(int cands, int uv, int tbl, int hits) { return size_t(109) * cands + 32 * uv + 8 * tbl + hits / 8 + 64; }
size_t match_smem_bytes(int velo) { return size_t(36) * velo + 1024; }
int build_blocks_per_sm(int, size_t) { return 4; }
int seed_blocks_per_sm(int threads, bool wide, size_t) {
    return threads <= 256 ? (wide ? 4 : 5) : threads <= 384 ? 3 : threads <= 512 ? 2 : 1;
}
int match_blocks_per_sm(int threads, size_t, bool, bool many) { return threads > 256 ? 2 : many ? 6 : 4; }
cudaError_t set_smem_limits(size_t) { return cudaSuccess; }
cudaError_t launch_build(const DevParams&, const BuildArgs&, int, int, cudaStream_t s) { return fake_launch("build", s, nullptr); }
cudaError_t launch_build_large(const DevParams&, const BuildArgs&, int, cudaStream_t s, cudaEvent_t started) {
    return fake_launch("build_large", s, started);
}
cudaError_t launch_order(const BuildArgs&, cudaStream_t s, bool) { return fake_launch("order", s, nullptr); }
cudaError_t launch_seed(const DevParams&, const SeedArgs& a, int, int, bool, size_t, cudaStream_t s, bool,
                        cudaEvent_t started) {
    return fake_launch(a.part == 1 ? "seed_large" : "seed", s, started);
}
cudaError_t launch_gather(const GatherArgs&, cudaStream_t s, bool) { return fake_launch("gather", s, nullptr); }
cudaError_t launch_match(const DevParams&, const MatchArgs&, int, int, bool many, cudaStream_t s, bool) {
    return fake_launch(many ? "match_many" : "match", s, nullptr);
}
cudaError_t launch_ut(const UtParams&, const UtArgs&, int, cudaStream_t s, bool) { return fake_launch("ut", s, nullptr); }
}  // namespace st

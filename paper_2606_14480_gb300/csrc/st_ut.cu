// st_ut.cu -- UT hits of the Long tracks (Section 4.3), sm_103a.
//
// One CTA per event.  The event's UT hits are staged in shared memory grouped
// by (layer, 16 mm bucket of x) with a counting sort, so a search window of a
// few mm reads one or two buckets (the order within a bucket does not matter:
// every choice below breaks ties explicitly by x, then by the hit's index).  One thread per seed with a matched VELO segment: the
// segment is extrapolated with Eq. (velo_ut_extrapolation), gamma_x from Eq.
// (gamma_parametrisation) at the pair's q/p, through the four UT layers in
// order; until a hit is found each layer is searched in its loose window and
// the closest hit refits gamma_x through itself, later layers in their tight
// windows (closest hit attached).  A Long track with fewer than min_hits UT
// hits loses its VELO segment.
//
// What bounds it is the latency of an event's chain (offsets, hits, counting
// sort, seeds, their segments, four layers), so that a batch should run in one
// round: 192 threads of 40 registers and 26 KB each fit eight times on an SM,
// the loads of hits go four at a time, and a thread's first seed is fetched
// while the hits are sorted.  1000 Run-3-like events: 23 us of the step with 256
// threads of 48 registers (five per SM, two rounds), 16 us this way; in buckets
// of 32 mm instead of 16 mm 17 us, with 160 threads 18 us.
#include <algorithm>
#include <cfloat>

#include "st_common.cuh"
#include "st_device.cuh"
#include "st_ut.cuh"

namespace st {

constexpr int kUtThreads = 192;
constexpr int kUtBlocks = 8;   // CTAs per SM
constexpr int kUtSmem = 4096;  // UT hits of one event staged in shared memory
constexpr int kUtBins = 128;   // x buckets per layer over [-1024, 1024) mm (edge buckets extend)
constexpr float kUtRange = 1024.f;

__device__ __forceinline__ int ut_bin(float x) {
    const int b = __float2int_rd((x + kUtRange) * (kUtBins / (2.f * kUtRange)));
    return min(max(b, 0), kUtBins - 1);
}

__global__ void __launch_bounds__(kUtThreads, kUtBlocks)
k_ut(const __grid_constant__ UtParams U, const __grid_constant__ UtArgs A) {
    __shared__ float sx[kUtSmem];
    __shared__ uint16_t si[kUtSmem];
    // first the buckets' counts (of bucket k at k + 1), then their fill cursors
    // from their starts on; when all hits are placed, entry k is the start of
    // bucket k
    __shared__ int s_cur[4 * kUtBins + 1], s_nl;
    const int tid = threadIdx.x, T = blockDim.x;
    pdl_wait();  // the matching's results
    for (int64_t e = blockIdx.x; e < A.n_events; e += gridDim.x) {
        const int64_t u0 = A.ut_off[e];
        const int nu = static_cast<int>(A.ut_off[e + 1] - u0);
        const int64_t s0 = A.seed_off[e];
        const int ns = A.seed_off[e + 1] - static_cast<int>(s0);
        const int64_t v0 = A.velo_off[e];
        const bool staged = nu <= kUtSmem;
        for (int k = tid; k <= 4 * kUtBins; k += T) s_cur[k] = 0;
        if (tid == 0) s_nl = 0;
        int v_next = tid < ns ? A.velo_idx[s0 + tid] : -1;  // of the thread's next seed
        __syncthreads();
        // four hits per thread per round, their loads issued together
        auto each_hit = [&](auto&& f) {
            for (int i0 = tid; i0 < nu; i0 += 4 * T) {
                int l[4];
                float x[4];
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    const int i = i0 + q * T;
                    l[q] = i < nu ? A.ut_layer[u0 + i] : 0;
                    x[q] = i < nu ? A.ut_x[u0 + i] : 0.f;
                }
#pragma unroll
                for (int q = 0; q < 4; ++q)
                    if (i0 + q * T < nu) f(i0 + q * T, l[q], x[q]);
            }
        };
        bool bad = false;
        each_hit([&](int, int l, float x) {
            if (l < 0 || l > 3 || !isfinite(x)) bad = true;
            else if (staged) atomicAdd(&s_cur[l * kUtBins + ut_bin(x) + 1], 1);
        });
        // the thread's next seed's segment and slope
        float xV = 0.f, yV = 0.f, txV = 0.f, tyV = 0.f, txS = 0.f;
        auto fetch = [&](int s) {
            if (v_next < 0) return;
            const float* vs = A.velo + (v0 + v_next) * 4;
            xV = vs[0];
            yV = vs[1];
            txV = vs[2];
            tyV = vs[3];
            txS = A.seed_state[(s0 + s) * 4 + 2];
        };
        fetch(tid);
        // an event with an invalid UT hit gets ST_EINVAL and no UT hits
        const bool skip = __syncthreads_or(bad) != 0;
        if (skip && tid == 0) A.status[e] = -1;  // ST_EINVAL
        if (staged && !skip) {
            if (tid < 32) {  // exclusive scan of the bucket counts by one warp
                constexpr int kPer = 4 * kUtBins / 32;
                int* const sc = s_cur + 1 + kPer * tid;
                int t = 0;
#pragma unroll
                for (int q = 0; q < kPer; ++q) t += sc[q];
                int x = t;
#pragma unroll
                for (int o = 1; o < 32; o <<= 1) {
                    const int y = __shfl_up_sync(0xffffffffu, x, o);
                    if (tid >= o) x += y;
                }
                int run = x - t;
#pragma unroll
                for (int q = 0; q < kPer; ++q) {
                    const int c = sc[q];
                    sc[q] = run;
                    run += c;
                }
            }
            __syncthreads();
            each_hit([&](int i, int l, float x) {
                const int k = atomicAdd(&s_cur[l * kUtBins + ut_bin(x) + 1], 1);
                sx[k] = x;
                si[k] = static_cast<uint16_t>(i);
            });
            __syncthreads();
        }
        int kept = 0;
        for (int s = tid; s < ns; s += T) {
            const int64_t r = s0 + s;
            int hits[4] = {-1, -1, -1, -1};
            int n = 0;
            float g = 0.f;
            const int v = v_next;
            if (v >= 0 && !skip) {
                const float qop = (txS - txV) * U.inv_kick;
                const float inv_p = 1000.f * fabsf(qop);  // 1/p in (GeV/c)^-1
                g = fmaf(U.gB, qop, U.gA);
                bool found = false;
#pragma unroll
                for (int l = 0; l < 4; ++l) {
                    const float* w = found ? &U.tight[4 * l] : &U.loose[4 * l];
                    if (!(w[3] > 0.f)) continue;
                    const float win = fminf(fmaxf(fmaf(w[1], inv_p, w[0]), w[2]), w[3]);
                    // straight part of the extrapolation as a float-float, so
                    // that the refit of gamma below keeps its precision
                    float p, pe, lh, ll;
                    two_prod(txV, U.dz[l], p, pe);
                    two_sum(xV, p, lh, ll);
                    ll += pe;
                    const float yt = fmaf(tyV, U.dz[l], yV);
                    const float ys = yt * U.t[l];
                    const float xm = lh + (ll + fmaf(g, U.dz2[l], -ys));
                    int best = -1;
                    float bd = 0.f, bx = 0.f;
                    auto consider = [&](float xh, auto&& index) {
                        const float d = fabsf(xh - xm);
                        if (!(d <= win) || (best >= 0 && d > bd)) return;
                        const int idx = index();
                        if (best < 0 || d < bd || xh < bx || (xh == bx && idx < best)) {
                            best = idx;
                            bd = d;
                            bx = xh;
                        }
                    };
                    if (staged) {
                        const int k0 = s_cur[l * kUtBins + ut_bin(xm - win)];
                        const int k1 = s_cur[l * kUtBins + ut_bin(xm + win) + 1];
                        for (int k = k0; k < k1; ++k) consider(sx[k], [&] { return int(si[k]); });
                    } else {
                        for (int i = 0; i < nu; ++i)
                            if (A.ut_layer[u0 + i] == l) consider(A.ut_x[u0 + i], [&] { return i; });
                    }
                    if (best < 0) continue;
                    hits[l] = best;
                    ++n;
                    if (!found) {
                        // gamma_x through this hit: (x_hit + y t - x_V - tx_V dz) / dz^2
                        g = (((bx - lh) - ll) + ys) / U.dz2[l];
                        found = true;
                    }
                }
            }
#pragma unroll
            for (int l = 0; l < 4; ++l) A.ut_hits[r * 4 + l] = hits[l];
            A.ut_n[r] = static_cast<int8_t>(n);
            A.gamma[r] = g;
            if (v >= 0 && n < U.min_hits) {
                A.velo_idx[r] = -1;
                A.chi2[r] = 0.f;
            }
            kept += v >= 0 && n >= U.min_hits;
            if (s + T < ns) {
                v_next = A.velo_idx[r + T];
                fetch(s + T);
            }
        }
        kept = warp_sum(kept);
        if ((tid & 31) == 0 && kept) atomicAdd(&s_nl, kept);
        __syncthreads();
        if (tid == 0 && A.n_long) A.n_long[e] = s_nl;
        __syncthreads();
    }
}

cudaError_t launch_ut(const UtParams& U, const UtArgs& a, int n_sms, cudaStream_t s, bool chained) {
    const int64_t grid = std::min<int64_t>(a.n_events, int64_t(n_sms) * kUtBlocks);
    if (grid <= 0) return cudaSuccess;
    return launch_k(k_ut, static_cast<unsigned>(grid), kUtThreads, 0, s, chained, nullptr, U, a);
}

}  // namespace st

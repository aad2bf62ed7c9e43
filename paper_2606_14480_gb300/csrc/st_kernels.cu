// st_kernels.cu -- sm_103a kernels of the SciFi Seeding + VELO-SciFi Matching
// hot path.  A batch that fits the resident CTAs gives each the work item
// (event, or detector half) of its own number; for larger ones persistent CTAs
// pull items from a device counter.
//
//   k_build   one event per item: validate hits, sort them by (container
//             slot, x, index) with a bucketed rank sort in shared memory, write
//             the per-event container (x, original index) and slot offsets.
//   k_order   the seeding items sorted by cost class, costliest first, the
//             order in which k_seed's queue hands them out; left out where
//             every item has a CTA of its own.
//   k_seed    (st_seed.cuh) one detector half of one event per item (the
//             paper keeps the halves apart, Section 5.2).  In the batch path
//             the CTA that finishes an event's second half also matches the
//             event.
//   k_scan / k_gather   per-event CSR of the seed records (up to 2048 events
//             k_gather finds the events' places itself).
//   k_match   (st_match.cuh) one event per item: VELO segments bucketed by ty
//             in shared memory, up to eight lanes per seed for its lowest
//             chi2_match, then optionally the final selection (ghost network,
//             clones).
//
// k_order, k_seed, k_scan, k_gather and k_match are launched as programmatic
// dependents of the kernel before them in the stream: their CTAs may be
// scheduled while it finishes, and wait (griddepcontrol.wait) for its
// completion and its memory before they read or write anything it touches.
// Launched without that attribute, the wait returns at once.
#include <algorithm>
#include <cfloat>
#include <utility>

#include "st_kernels.cuh"
#include "st_match.cuh"

namespace st {

// Sum per-thread counters over the CTA (warp shuffles, then shared memory)
// and add them to the global counters with one atomic per counter per CTA.
// Every thread of the CTA must call it.
__device__ __forceinline__ void flush_counters(unsigned long long* dst, const ull* c, int n) {
    __shared__ ull s_acc[16];
    if (threadIdx.x < 16) s_acc[threadIdx.x] = 0;
    __syncthreads();
    for (int k = 0; k < n; ++k) {
        ull v = c[k];
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
        if ((threadIdx.x & 31) == 0 && v) atomicAdd(&s_acc[k], v);
    }
    __syncthreads();
    if (threadIdx.x < n && s_acc[threadIdx.x]) atomicAdd(dst + threadIdx.x, s_acc[threadIdx.x]);
}

// ===========================================================================
// container build
// ===========================================================================

constexpr float kBinRange = 3500.f;

// Seeding items are handed out costliest first (largest-processing-time
// order), so that no large item starts when the rest of the batch is nearly
// done.  The cost of a (event, half) item is the size of its two-hit search
// domain, sum over iterations of n(T1) n(T3), plus its hit count; its class
// is that cost on a quarter-octave scale.
constexpr int kCostClasses = 128;
static_assert(kCostClasses % 32 == 0, "one warp scans the classes");

__device__ __forceinline__ int cost_class(ull cost) {
    if (cost < 4u) return static_cast<int>(cost);
    const int oct = 63 - __clzll(static_cast<long long>(cost));
    return min(4 * oct + static_cast<int>((cost >> (oct - 2)) & 3u), kCostClasses - 1);
}

__device__ __forceinline__ void set_item_class(const BuildArgs& A, int64_t item, int c) {
    if (!A.order) return;  // one round of items: their order does not matter
    A.item_class[item] = c;
    atomicAdd(A.class_count + c, 1);
}

// shared memory of k_build: bucket counts / fill cursors and bucket starts,
// the block scan's scratch, then 10 bytes per hit (x, bucket, the hits
// grouped by bucket, the sorted order)
size_t build_smem_bytes(int bins, int smem_hits) {
    const int NB = kZones * bins;
    return align16(sizeof(int) * (2 * NB + 1 + kScanInts)) + align16(size_t(10) * smem_hits);
}

// Per event (one CTA): validate and bucket the hits by (container slot, x),
// place them bucket by bucket, rank each hit inside its bucket by (x, index)
// and write the sorted event out in order.  Per-hit arrays: x (hx), bucket
// (bk), the hits grouped by bucket (pm) and the sorted order (so), which the
// ranking fills directly.  Between two events of a CTA the bucket
// counts are cleared during the ranking and the next event's ticket and
// offsets are fetched during the placement, so the next event starts with
// its loads.  At most 32 registers: up to eight 256-thread CTAs per SM.
//
// A batch that may hold large events is shared by two launches side by side
// (BuildArgs::split_hits): kLarge takes the events above it in CTAs with most
// of an SM's shared memory (an event of 12,700 hits: 82 us in scratch memory
// before), the other the rest with little of it each.
template <bool kLarge>
__global__ void __launch_bounds__(kMaxThreads, kLarge ? 1 : 4)
k_build(const __grid_constant__ DevParams P, const __grid_constant__ BuildArgs A) {
    extern __shared__ __align__(16) unsigned char smem[];
    const int NBmax = kZones * A.bins, T = blockDim.x, tid = threadIdx.x;
    int* cnt = reinterpret_cast<int*>(smem);  // counts, then fill cursors, then cleared
    int* off = cnt + NBmax;
    int* tmp = off + NBmax + 1;
    unsigned char* harea = smem + align16(sizeof(int) * (2 * NBmax + 1 + kScanInts));
    // the CTA's next event and its hit range, published by thread 0
    __shared__ int s_item, s_bad;
    __shared__ long long s_h0, s_h1;
    // per-zone / per-layer constants indexed by each hit's zone: in shared
    // memory (reads of kernel parameters at lane-dependent indices serialise)
    __shared__ int s_slot[kZones];
    __shared__ float s_zl[kLayers], s_tl[kLayers];
    if (tid < kZones) s_slot[tid] = P.slot_of_zone[tid];
    if (tid < kLayers) {
        s_zl[tid] = P.zl[tid];
        s_tl[tid] = P.tl[tid];
    }
    ull ctr[2] = {0, 0};
    int spar = 0;  // which half of tmp the next block scan uses
    for (int k = tid; k < NBmax; k += T) cnt[k] = 0;
    // the first warp: the next event and its offsets.  Tickets, or the next
    // large one of every gridDim.x-th event, 32 of them looked at together.
    __shared__ long long s_scan;
    auto next_item = [&](bool first = false) {
        if constexpr (kLarge) {
            int64_t e = A.n_events;
            int64_t h0 = 0, h1 = 0;
            int64_t k = s_scan;
            for (; k < A.n_events; k += 32 * int64_t(gridDim.x)) {
                const int64_t c = k + tid * int64_t(gridDim.x);
                if (c < A.n_events) {
                    h0 = A.ev_off[c];
                    h1 = A.ev_off[c + 1];
                }
                const unsigned hit =
                    __ballot_sync(0xffffffffu, c < A.n_events && h1 - h0 > A.split_hits && h1 - h0 <= A.max_hits);
                if (hit) {
                    const int l = __ffs(hit) - 1;
                    e = k + l * int64_t(gridDim.x);
                    if (tid == l) {
                        s_h0 = h0;
                        s_h1 = h1;
                    }
                    break;
                }
            }
            __syncwarp();
            if (tid == 0) {
                s_scan = e + gridDim.x;
                s_item = static_cast<int>(e);
            }
            __syncwarp();
        } else if (tid == 0) {
            // its own number first, then tickets (one event by direct calls: 54
            // us with a ticket each, 53 us without)
            const int64_t q = first ? blockIdx.x
                              : gridDim.x < A.n_events ? gridDim.x + int64_t(atomicAdd(A.queue, 1))
                                                       : A.n_events;
            if (q < A.n_events) {
                s_h0 = A.ev_off[q];
                s_h1 = A.ev_off[q + 1];
            }
            s_item = static_cast<int>(q);
        }
    };
    if (tid == 0) {
        s_bad = 0;
        s_scan = blockIdx.x;
    }
    if (tid < 32) {
        __syncwarp();
        next_item(true);
    }

    for (;;) {
        __syncthreads();
        const int64_t e = s_item;
        if (e >= A.n_events) break;
        const int64_t h0 = s_h0;
        const int64_t n64 = s_h1 - h0;
        int32_t* zo = A.zoff + e * kZoffStride;
        const int64_t cb = cont_base(A.ev_off, e);
        const bool bad_size = n64 < 0 || n64 > A.max_hits || cb + n64 > A.cont_cap;
        if (kLarge ? bad_size : !bad_size && A.split_hits > 0 && n64 > A.split_hits) {
            __syncthreads();  // the other launch's
            if (tid < 32) next_item();
            continue;
        }
        if (bad_size) {
            // too large for max_hits, or an earlier oversized event pushed this
            // one past the container
            for (int k = tid; k < kZoffStride; k += T) zo[k] = 0;
            if (tid < 2) set_item_class(A, 2 * e + tid, 0);
            __syncthreads();  // every thread has read s_item
            if (tid == 0) A.status[e] = -3;  // ST_OVERFLOW
            if (tid < 32) next_item();
            continue;
        }
        const int n = static_cast<int>(n64);
        // about four hits per bucket
        int B = min(8, A.bins);
        while (B < A.bins && B * (4 * kZones) < n) B <<= 1;
        const int NB = kZones * B;
        const bool in_smem = n <= A.smem_hits;
        unsigned char* base = in_smem ? harea : A.big + int64_t(blockIdx.x) * A.big_stride;
        const int cap = in_smem ? A.smem_hits : A.max_hits;
        float* hx = reinterpret_cast<float*>(base);
        uint16_t* bk = reinterpret_cast<uint16_t*>(hx + cap);
        uint16_t* pm = bk + cap;
        uint16_t* so = pm + cap;
        const float binscale = B / (2.f * kBinRange);
        // count: four hits per thread per round, their loads issued together
        for (int i0 = tid; i0 < n; i0 += 4 * T) {
            float xs[4];
            int zs[4];
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const int i = i0 + q * T;
                xs[q] = i < n ? A.x[h0 + i] : 0.f;
                zs[q] = i < n ? A.zone[h0 + i] : 0;
            }
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const int i = i0 + q * T;
                if (i >= n) break;
                const float x = xs[q];
                const int zn = zs[q];
                bool bad = !(zn >= 0 && zn < kZones) || !isfinite(x);
                if (!bad) {
                    const int L = zn >> 1;
                    if (A.z && !(fabsf(A.z[h0 + i] - s_zl[L]) <= 1e-3f)) bad = true;
                    if (A.dxdy && !(fabsf(A.dxdy[h0 + i] - s_tl[L]) <= 1e-6f)) bad = true;
                }
                if (bad) {
                    s_bad = 1;
                    continue;
                }
                int bin = __float2int_rd((x + kBinRange) * binscale);
                bin = min(max(bin, 0), B - 1);
                const int b = s_slot[zn] * B + bin;
                hx[i] = x;
                bk[i] = static_cast<uint16_t>(b);
                atomicAdd(&cnt[b], 1);
            }
        }
        __syncthreads();
        if (s_bad) {
            for (int k = tid; k < kZoffStride; k += T) zo[k] = 0;
            for (int k = tid; k < NB; k += T) cnt[k] = 0;
            if (tid < 2) set_item_class(A, 2 * e + tid, 0);
            __syncthreads();  // s_bad read by every thread
            if (tid == 0) {
                A.status[e] = -1;  // ST_EINVAL
                s_bad = 0;
            }
            if (tid < 32) next_item();
            continue;
        }
        {   // exclusive scan of the bucket counts; the counts become fill cursors
            const int per = (NB + T - 1) / T;
            const int k0 = min(tid * per, NB), k1 = min(k0 + per, NB);
            int sum = 0;
            for (int k = k0; k < k1; ++k) sum += cnt[k];
            int tot;
            int ex = block_exscan1(sum, tmp, spar, tot);
            for (int k = k0; k < k1; ++k) {
                const int c = cnt[k];
                off[k] = ex;
                cnt[k] = ex;
                ex += c;
            }
            if (tid == 0) off[NB] = tot;
        }
        __syncthreads();
        if (tid < 32) next_item();  // read by the other threads after the next loop-top barrier
        for (int i = tid; i < n; i += T) pm[atomicAdd(&cnt[bk[i]], 1)] = static_cast<uint16_t>(i);
        __syncthreads();
        // rank of each hit in its bucket -> its place in the sorted event;
        // the cursors are cleared for the next event.  Threads take the hits
        // in bucket order, so the lanes of a warp mostly share a bucket: equal
        // loop lengths, and the bucket's reads are broadcasts.
        for (int k = tid; k < NB; k += T) cnt[k] = 0;
        for (int d = tid; d < n; d += T) {
            const int i = pm[d];
            const int b = bk[i], s = off[b], c = off[b + 1] - s;
            const float x = hx[i];
            int r = 0;
            for (int k = s; k < s + c; ++k) {
                const int j = pm[k];
                const float xj = hx[j];
                r += (xj < x) || (xj == x && j < i);
            }
            so[s + r] = static_cast<uint16_t>(i);
        }
        __syncthreads();
        // the CTA's last event is as good as done: the next kernel may be
        // scheduled (it waits for this grid).  Not earlier: its CTAs would take
        // their places while some SMs are full, and stay unevenly spread (250
        // Run-3-like events: 115 us with the signal at the start, 107 us here).
        if (s_item >= A.n_events) pdl_signal();
        // the sorted event goes out in order (coalesced stores)
        for (int d = tid; d < n; d += T) {
            const int i = so[d];
            A.cx[cb + d] = hx[i];
            A.corig[cb + d] = i;
        }
        for (int k = tid; k < kZoffStride; k += T) zo[k] = off[k * B];
        if (tid < 2) {
            auto nz = [&](int sl) { return ull(off[(sl + 1) * B] - off[sl * B]); };
            ull cost = ull(off[(12 * tid + 12) * B] - off[12 * tid * B]);
            for (int it = 0; it < P.n_iter; ++it) cost += nz(12 * tid + P.it[it].s1) * nz(12 * tid + P.it[it].s3);
            set_item_class(A, 2 * e + tid, cost_class(cost));
        }
        if (tid == 0) {
            A.status[e] = 0;
            ctr[0] += n;
            ctr[1] += 1;
        }
    }
    flush_counters(A.counters + C_HITS, ctr, 2);
}

// The seeding items in cost order (a counting sort by class, costliest class
// first), after k_build has counted the classes.  One thread per item; a
// CTA's items of one class take consecutive places from one global atomic.
// The order inside a class does not matter: items are independent and their
// results are gathered per event.
constexpr int kOrderThreads = 1024;
// The items for the larger CTAs of a split batch: those that cost this many
// times the mean (500 uneven events of 120 tracks on average at 4, 5, 6.5, 8
// times: 483, 492, 503, 534 us) and at least as much as a CTA's share of the
// batch; what costs less is done before the batch is in any CTA (10,000 uneven
// events with 5, 8 times the mean alone 2918, 2801 us; 2733 unsplit).
constexpr float kBigCost = 5.f;

__global__ void __launch_bounds__(kOrderThreads) k_order(const __grid_constant__ BuildArgs A) {
    __shared__ int pos[kCostClasses], s_cnt[kCostClasses];
    const int tid = threadIdx.x;
    pdl_signal();
    pdl_wait();  // k_build's class counts
    const unsigned lane = tid & 31;
    if (tid < 32) {  // first place of each class: exclusive scan from the top class down
        constexpr int kPer = kCostClasses / 32;
        int c[kPer], t = 0;
#pragma unroll
        for (int q = 0; q < kPer; ++q) {
            c[q] = A.class_count[kCostClasses - 1 - (kPer * tid + q)];
            t += c[q];
        }
        int x = t;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int y = __shfl_up_sync(0xffffffffu, x, o);
            if (tid >= o) x += y;
        }
        int run = x - t;
#pragma unroll
        for (int q = 0; q < kPer; ++q) {
            pos[kCostClasses - 1 - (kPer * tid + q)] = run;
            run += c[q];
        }
    }
    for (int k = tid; k < kCostClasses; k += kOrderThreads) s_cnt[k] = 0;
    __syncthreads();
    const int64_t items = 2 * A.n_events;
    if (A.n_big && blockIdx.x == 0 && tid < 32) {
        auto cost = [](int c) {  // the least cost of class c (cost_class)
            return c < 8 ? float(c) : ldexpf(float(4 + (c & 3)), (c >> 2) - 2);
        };
        float sum = 0.f;
        for (int c = tid; c < kCostClasses; c += 32) sum += cost(c) * float(A.class_count[c]);
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
        const float bar = fmaxf(kBigCost * sum / float(items), sum / float(A.n_ctas));
        int n = 0;
        for (int c = tid; c < kCostClasses; c += 32) n += cost(c) >= bar ? A.class_count[c] : 0;
        n = __reduce_add_sync(0xffffffffu, n);
        if (tid == 0) *A.n_big = n;
    }
    const int64_t i = int64_t(blockIdx.x) * kOrderThreads + tid;
    const int c = i < items ? A.item_class[i] : -1;
    const unsigned same = __match_any_sync(0xffffffffu, c);
    const int leader = __ffs(same) - 1;
    int r = 0;
    if (c >= 0 && static_cast<int>(lane) == leader) r = atomicAdd(&s_cnt[c], __popc(same));
    r = __shfl_sync(0xffffffffu, r, leader) + __popc(same & ((1u << lane) - 1u));
    __syncthreads();
    for (int k = tid; k < kCostClasses; k += kOrderThreads)
        if (s_cnt[k]) pos[k] += atomicAdd(A.class_fill + k, s_cnt[k]);
    __syncthreads();
    if (c >= 0) A.order[pos[c] + r] = static_cast<int32_t>(i);
}

// ===========================================================================
// per-event CSR of the seed records
// ===========================================================================

__global__ void __launch_bounds__(1024) k_scan(const __grid_constant__ GatherArgs A) {
    __shared__ int tmp[36];
    pdl_signal();
    pdl_wait();  // the seeding kernel's item counts
    int64_t carry = 0;
    for (int64_t b = 0; b < A.n_events; b += blockDim.x) {
        const int64_t e = b + threadIdx.x;
        const int c = e < A.n_events ? A.item_count[2 * e] + A.item_count[2 * e + 1] : 0;
        int tot;
        const int ex = block_exscan(c, tmp, tot);
        if (e < A.n_events) A.ev_off[e] = static_cast<int32_t>(carry + ex);
        carry += tot;
    }
    if (threadIdx.x == 0) A.ev_off[A.n_events] = static_cast<int32_t>(carry);
}

// One block per event: the event's records come from the pool ranges of its
// two (event, half) items and go to one contiguous range of each output
// array, so every array is copied as a flat run (16-byte words when all
// output arrays allow it).
// (at most 32 registers: eight CTAs per SM, a 1000-event batch in one round)
// kScan: a grid of one CTA per event that also finds the event's place, by
// adding up the counts before it, and writes the offsets; k_scan does that for
// larger batches.  (For 1000 events the counts are 8 KB, read from L2 by every
// CTA at once; the separate kernel took 2.5 us of its own.)
template <bool kVec, bool kScan>
__global__ void __launch_bounds__(256, 8) k_gather(const __grid_constant__ GatherArgs A) {
    __shared__ int s_before[8];
    pdl_signal();
    pdl_wait();  // the seed records (and k_scan's event offsets)
    const bool fault = A.fault && *A.fault;
    int64_t d_own = 0;
    for (int64_t e = blockIdx.x; e < A.n_events; e += gridDim.x) {
        if (kScan) {
            int sum = 0;
            const int2* c = reinterpret_cast<const int2*>(A.item_count);
            for (int64_t q = threadIdx.x; q < e; q += blockDim.x) sum += c[q].x + c[q].y;
            sum = __reduce_add_sync(0xffffffffu, sum);
            if ((threadIdx.x & 31) == 0) s_before[threadIdx.x >> 5] = sum;
            __syncthreads();
            sum = 0;
#pragma unroll
            for (int w = 0; w < 8; ++w) sum += s_before[w];
            if (threadIdx.x == 0) {
                A.ev_off[e] = sum;
                if (e == A.n_events - 1) A.ev_off[A.n_events] = sum + c[e].x + c[e].y;
            }
            d_own = sum;
        }
        if (fault && threadIdx.x == 0) A.status[e] = -4;  // ST_TIMEOUT: the fused matching gave up a wait
        const int c0 = A.item_count[2 * e], c1 = A.item_count[2 * e + 1];
        const int n = c0 + c1;
        if (n == 0) continue;
        const int64_t s0 = A.item_start[2 * e], s1 = A.item_start[2 * e + 1];
        const int64_t d0 = kScan ? d_own : A.ev_off[e];
        auto src = [&](int k) { return k < c0 ? s0 + k : s1 + (k - c0); };
        const int T = blockDim.x;
        if (kVec) {
            // the event's 16-byte words as one range: hits (3 per record),
            // params (2), state (1); a thread loads four words before it stores
            // them, so their latencies overlap
            const uint4* ph = reinterpret_cast<const uint4*>(A.pool_hits);
            const uint4* pp = reinterpret_cast<const uint4*>(A.pool_params);
            const uint4* ps = reinterpret_cast<const uint4*>(A.pool_state);
            uint4* oh = reinterpret_cast<uint4*>(A.hits);
            uint4* op = reinterpret_cast<uint4*>(A.params);
            uint4* os = reinterpret_cast<uint4*>(A.state);
            const int W = 6 * n;
            for (int w0 = threadIdx.x; w0 < W; w0 += 4 * T) {
                uint4 v[4];
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    const int w = w0 + j * T;
                    if (w < 3 * n) {
                        const int k = w / 3;
                        v[j] = ph[src(k) * 3 + (w - 3 * k)];
                    } else if (w < 5 * n) {
                        const int u = w - 3 * n;
                        v[j] = pp[src(u >> 1) * 2 + (u & 1)];
                    } else if (w < W) {
                        v[j] = ps[src(w - 5 * n)];
                    }
                }
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    const int w = w0 + j * T;
                    if (w < 3 * n) {
                        oh[d0 * 3 + w] = v[j];
                    } else if (w < 5 * n) {
                        op[d0 * 2 + (w - 3 * n)] = v[j];
                    } else if (w < W) {
                        os[d0 + (w - 5 * n)] = v[j];
                    }
                }
            }
            const uint16_t* pn = reinterpret_cast<const uint16_t*>(A.pool_n);
            uint16_t* on = reinterpret_cast<uint16_t*>(A.n_hits);
            for (int k = threadIdx.x; k < n; k += T) {
                const int64_t r = src(k);
                const uint16_t c = pn[r];
                if (A.pool_velo) {
                    const int32_t vi = A.pool_velo[r];
                    const float ch = A.pool_chi2[r];
                    A.velo_idx[d0 + k] = vi;
                    A.chi2[d0 + k] = ch;
                }
                on[d0 + k] = c;
            }
        } else {
            if (A.pool_velo) {
                for (int k = threadIdx.x; k < n; k += T) {
                    A.velo_idx[d0 + k] = A.pool_velo[src(k)];
                    A.chi2[d0 + k] = A.pool_chi2[src(k)];
                }
            }
            for (int i = threadIdx.x; i < 12 * n; i += blockDim.x) {
                const int k = i / 12, q = i - 12 * k;
                A.hits[(d0 + k) * 12 + q] = A.pool_hits[src(k) * 12 + q];
            }
            for (int i = threadIdx.x; i < 8 * n; i += blockDim.x) {
                const int k = i >> 3, q = i & 7;
                A.params[(d0 + k) * 8 + q] = A.pool_params[src(k) * 8 + q];
            }
            for (int i = threadIdx.x; i < 4 * n; i += blockDim.x) {
                const int k = i >> 2, q = i & 3;
                A.state[(d0 + k) * 4 + q] = A.pool_state[src(k) * 4 + q];
            }
            for (int i = threadIdx.x; i < 2 * n; i += blockDim.x) {
                const int k = i >> 1, q = i & 1;
                A.n_hits[(d0 + k) * 2 + q] = A.pool_n[src(k) * 2 + q];
            }
        }
    }
}

// ===========================================================================
// matching
// ===========================================================================

// One event per work item (match_event), for matching_run on seeds in the
// per-event CSR layout.
// kFinal: compiled with the final selection of Section 4.4 (the plain
// instantiation does not carry its registers).
// kMany: CTAs of up to 256 threads with 40 registers each, six to an SM, where
// the 51 registers otherwise taken leave room for four.
template <bool kFinal, bool kMany>
__global__ void __launch_bounds__(kMany ? kMatchManyThreads : kMaxThreads, kMany ? 6 : 0)
k_match(const __grid_constant__ DevParams P, const __grid_constant__ MatchArgs A) {
    extern __shared__ __align__(16) unsigned char smem[];
    const int tid = threadIdx.x;
    __shared__ int s_item, s_cnt;
    ull ctr[4] = {0, 0, 0, 0};  // grid pairs, preselected pairs, Long tracks, evaluated pairs
    const MatchIO M{A.velo, A.seed_state, A.seed_n, A.velo_idx, A.chi2, A.ghost_prob};
    pdl_wait();  // the seeds

    // the first event is the CTA's own number, the others come from the queue
    // (none without one: the grid covers the events)
    for (int64_t e = blockIdx.x; e < A.n_events;) {
        const int64_t v0 = A.velo_off[e];
        const int nv = static_cast<int>(A.velo_off[e + 1] - v0);
        const int64_t s0 = A.seed_off[e];
        const int ns = A.seed_off[e + 1] - static_cast<int>(s0);
        const int nl = match_event<kFinal>(P, M, A.velo_smem, smem, v0, nv, ns,
                                           [&](int s) { return s0 + s; }, &s_cnt, ctr[0], ctr[1], ctr[3]);
        if (tid == 0) {
            if (A.n_long) A.n_long[e] = nl;
            ctr[2] += nl;
        }
        if (!A.queue) break;
        if (tid == 0) s_item = gridDim.x + atomicAdd(A.queue, 1);
        __syncthreads();
        e = s_item;
        __syncthreads();
    }
    pdl_signal();
    flush_counters(A.counters + C_MATCH_PAIRS, ctr, 3);
    flush_counters(A.counters + C_MATCH_EVAL, ctr + 3, 1);
}

size_t match_smem_bytes(int velo_smem) { return match_smem_size(velo_smem); }

// ===========================================================================
// launchers
// ===========================================================================

typedef void (*MatchKernel)(const DevParams, const MatchArgs);
static MatchKernel match_kernel(bool final_sel, bool many) {
    return final_sel ? k_match<true, false> : many ? k_match<false, true> : k_match<false, false>;
}

// Raise each kernel's dynamic shared-memory ceiling to what the device allows
// next to the kernel's own static shared memory (opt-in maximum - static).
cudaError_t set_smem_limits(size_t optin) {
    const void* fns[5 + 3 * kSeedShapes] = {
        reinterpret_cast<const void*>(k_build<false>), reinterpret_cast<const void*>(k_build<true>),
        reinterpret_cast<const void*>(match_kernel(false, false)), reinterpret_cast<const void*>(match_kernel(true, false)),
        reinterpret_cast<const void*>(match_kernel(false, true))};
    int n = 5;
    for (int sh = 0; sh < kSeedShapes; ++sh)
        for (int mode = 0; mode < 3; ++mode)
            fns[n++] = reinterpret_cast<const void*>(seed_kernel(kSeedThreads[sh], kSeedWide[sh], mode == 1, mode == 2));
    for (const void* f : fns) {
        cudaFuncAttributes fa;
        cudaError_t err = cudaFuncGetAttributes(&fa, f);
        if (err != cudaSuccess) return err;
        const int dyn = static_cast<int>(optin) - static_cast<int>(fa.sharedSizeBytes);
        if ((err = cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, dyn)) != cudaSuccess)
            return err;
    }
    return cudaSuccess;
}

// Whether the ceilings set_smem_limits raises are still in place (a
// cudaDeviceReset drops them with the context): checked on the container
// kernel, the first one set_smem_limits raises.
cudaError_t smem_limits_hold(size_t optin, bool& hold) {
    cudaFuncAttributes fa;
    const cudaError_t err = cudaFuncGetAttributes(&fa, reinterpret_cast<const void*>(k_build<false>));
    hold = err == cudaSuccess &&
           fa.maxDynamicSharedSizeBytes >= static_cast<int>(optin) - static_cast<int>(fa.sharedSizeBytes);
    return err;
}

int build_blocks_per_sm(int threads, size_t smem) {
    int n = 0;
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, k_build<false>, threads, smem);
    return n;
}
int seed_blocks_per_sm(int threads, bool wide, size_t smem) {
    int n = 0;
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, seed_kernel(threads, wide, false, false), threads, smem);
    return n;
}
int match_blocks_per_sm(int threads, size_t smem, bool final_sel, bool many) {
    int n = 0;
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, match_kernel(final_sel, many), threads, smem);
    return n;
}

cudaError_t launch_build(const DevParams& P, const BuildArgs& a, int grid, int threads, cudaStream_t s) {
    return launch_k(k_build<false>, static_cast<unsigned>(grid), static_cast<unsigned>(threads),
                    build_smem_bytes(a.bins, a.smem_hits), s, false, nullptr, P, a);
}

cudaError_t launch_build_large(const DevParams& P, const BuildArgs& a, int grid, cudaStream_t s, cudaEvent_t started) {
    return launch_k(k_build<true>, static_cast<unsigned>(grid), kMaxThreads, build_smem_bytes(a.bins, a.smem_hits), s,
                    false, started, P, a);
}

cudaError_t launch_order(const BuildArgs& a, cudaStream_t s, bool chained) {
    const int64_t items = 2 * a.n_events;
    if (items <= 0 || !a.order) return cudaSuccess;
    return launch_k(k_order, static_cast<unsigned>((items + kOrderThreads - 1) / kOrderThreads), kOrderThreads, 0, s,
                    chained, nullptr, a);
}

cudaError_t launch_seed(const DevParams& P, const SeedArgs& a, int grid, int threads, bool wide, size_t smem,
                        cudaStream_t s, bool chained, cudaEvent_t started) {
    const bool sq = P.iter_mode == 1;
    const bool fused = a.ev_done != nullptr;  // (a batch without any VELO segment may have no array of them)
    if (fused && sq) return cudaErrorInvalidValue;  // the runtime asks for fused matching in the HLT1 mode only
    const SeedKernel k = seed_kernel(threads, wide, sq, fused);
    return launch_k(k, static_cast<unsigned>(grid), static_cast<unsigned>(threads), smem, s, chained, started, P, a);
}

cudaError_t launch_gather(const GatherArgs& a, cudaStream_t s, bool chained) {
    // one CTA per event finds its own offset, while the sums it repeats are
    // short against a kernel of their own
    const bool own = a.n_events <= 2048;
    if (!own) {
        cudaError_t err = launch_k(k_scan, 1, 1024, 0, s, chained, nullptr, a);
        if (err != cudaSuccess) return err;
    }
    const int grid = static_cast<int>(std::min<int64_t>(a.n_events, 8192));
    if (grid <= 0) return cudaSuccess;
    // pool arrays are 256-byte aligned; the caller's output arrays may not be
    const uintptr_t mis = (reinterpret_cast<uintptr_t>(a.hits) | reinterpret_cast<uintptr_t>(a.params) |
                           reinterpret_cast<uintptr_t>(a.state)) & 15u;
    const bool vec = mis == 0 && (reinterpret_cast<uintptr_t>(a.n_hits) & 1u) == 0;
    void (*k)(const GatherArgs) = own ? (vec ? k_gather<true, true> : k_gather<false, true>)
                                      : (vec ? k_gather<true, false> : k_gather<false, false>);
    return launch_k(k, static_cast<unsigned>(grid), 256, 0, s, own ? chained : true, nullptr, a);
}

cudaError_t launch_match(const DevParams& P, const MatchArgs& a, int grid, int threads, bool many, cudaStream_t s,
                         bool chained) {
    return launch_k(match_kernel(P.final_sel != 0, many), static_cast<unsigned>(grid), static_cast<unsigned>(threads),
                    match_smem_bytes(a.velo_smem), s, chained, nullptr, P, a);
}

}  // namespace st

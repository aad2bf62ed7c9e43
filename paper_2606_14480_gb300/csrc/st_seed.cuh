// st_seed.cuh -- the seeding kernel, k_seed: one detector half of one event per
// work item.  XZ seeding of the iterations (pairs, third hits, extension,
// compensated least-squares fit), O(n) clone killing with a 64-bit atomicMin
// table, UV seeding (iterative or Hough clusters) with a 64-bit atomicMin per
// seed, and the seed records; HLT2-style iterations run as passes with a
// taken-hit bitmask.
//
// What bounds it is instruction issue and the latency of each item's chain of
// phases, not memory.  Per Run-3-like half (1150 hits) there are 2530 pairs,
// 230 triplets, 150 candidates, 73 kept, 800 UV combinations and 160 valid
// ones; so few that how they are spread over the lanes decides.  The searches
// therefore number their items by a block scan and give consecutive ones to
// the lanes of a warp, reject most of them by one look at a bit map of the
// layer's hits (2 mm bins: 88% of the pairs, 60% of the UV combinations), and
// collect the rest before the expensive step, so that it runs with full warps.
// 1000 Run-3-like events in one graph, matching fused in: the step 263 us when
// every thread walked its own run of pairs and combinations to the end (k_seed
// 206 us, 158 M warp instructions), 233 us this way (k_seed 190 us), 213 us with
// the registers set as below (k_seed 171 us, 125 M warp instructions).
#pragma once

#include "st_common.cuh"
#include "st_match.cuh"

namespace st {

// Registers per thread of each shape, for five, four, three, two and one CTAs
// per SM.  Set outright next to the largest CTA: asked for as a number of CTAs per
// SM, or without the largest CTA, the same counts give code that is slower
// everywhere (1000 Run-3-like events 232 against 215 us, 301 by direct calls 107
// against 101, HLT2-style 250 events 137 against 129).  (nvcc takes the pair
// where both depend on a template's arguments; the two are not documented to go
// together, so the build checks the registers that come out.)
constexpr int kSeedRegs256 = 48;
constexpr int kSeedRegs256w = 64;
constexpr int kSeedRegs384 = 56;
constexpr int kSeedRegs512 = 64;
constexpr int kSeedRegs1024 = 48;  // leaves room for a smaller CTA beside it
SeedKernel seed_kernel_256(bool seq, bool fused);
SeedKernel seed_kernel_256w(bool seq, bool fused);
SeedKernel seed_kernel_384(bool seq, bool fused);
SeedKernel seed_kernel_512(bool seq, bool fused);
SeedKernel seed_kernel_1024(bool seq, bool fused);

// ---------------------------------------------------------------------------
// per-zone hit maps: one bit per 2 mm bin that holds a hit, and per word of 32
// bins the first hit at or after it.  A window is known to be empty from its
// bits alone; otherwise the first hit at or after a bin is no earlier than the
// word's first hit plus the bits below the bin (every such bin holds at least
// one), and the search starts there.
// ---------------------------------------------------------------------------

// The range covers the SciFi's x acceptance (|x| < 3200 mm) and the stereo
// layers' measured coordinate, offset from it by y tan(5 deg) for |y| < 2500 mm
// (hits outside it fall into the end bins, which stays correct but scans
// longer).
constexpr float kMapRange = 3456.f;
constexpr int kMapBins = 3456;  // 2 mm bins over [-3456, 3456) mm
constexpr int kMapWords = kMapBins / 32;
constexpr int kMapStride = kMapWords + 1;  // a zero word after the last, read by windows that start in it

__device__ __forceinline__ int map_bin(float v) {
    const int b = __float2int_rd(fmaf(v, kMapBins / (2.f * kMapRange), 0.5f * kMapBins));
    return min(max(b, 0), kMapBins - 1);
}

// the maps of one half: bits[12][kMapStride], first[12][kMapWords]
struct HitMap {
    const uint32_t* bits;
    const uint16_t* first;
    __device__ __forceinline__ HitMap zone(int z) const { return {bits + z * kMapStride, first + z * kMapWords}; }
    // a place at or before the first hit of bin b or later
    __device__ __forceinline__ int from(int b) const {
        return first[b >> 5] + __popc(bits[b >> 5] & ((1u << (b & 31)) - 1u));
    }
    // whether bins b0 .. b1 hold no hit
    __device__ __forceinline__ bool empty(int b0, int b1) const {
        const uint32_t v = __funnelshift_r(bits[b0 >> 5], bits[(b0 >> 5) + 1], b0 & 31);
        const int span = b1 - b0;
        return span < 32 && (v & (0xffffffffu >> (31 - span))) == 0u;
    }
};

// first index i in [0, n) with x[i] >= v (n if none)
__device__ __forceinline__ int zlo(const float* x, const HitMap m, int n, float v) {
    int i = m.from(map_bin(v));
    while (i < n && x[i] < v) ++i;
    return i;
}

// first index i in [0, n) with x[i] > v (n if none)
__device__ __forceinline__ int zhi(const float* x, const HitMap m, int n, float v) {
    int i = m.from(map_bin(v));
    while (i < n && !(v < x[i])) ++i;
    return i;
}

// hits taken by earlier iterations (HLT2-style mode), one bit per half-local
// hit position; null when every hit is free
__device__ __forceinline__ bool is_used(const uint32_t* used, int p) {
    return used && ((used[p >> 5] >> (p & 31)) & 1u);
}

// The closest hit to xp within tol in a sorted zone (xs, its map, n hits
// starting at half-local position st), ties to the smaller x (the first met),
// skipping hits taken by earlier iterations.  The search starts at the map's
// place for xp - tol: hits below xp - tol are passed over (the window start a
// zlo search would give), it ends at the first hit above xp + tol.  In two
// steps, so that the loads of several searches can be in flight together.
struct Near {
    float lo, hi, x0, x1;  // the window; the hits at k and k + 1
    int k;
    __device__ __forceinline__ static float at(const float* xs, int n, int k) {
        return k < n ? xs[k] : __int_as_float(0x7fffffff);  // past the zone's end every comparison is false
    }
    __device__ __forceinline__ void start(const float* xs, const HitMap m, int n, float xp, float tol) {
        lo = xp - tol;
        hi = xp + tol;
        k = m.from(map_bin(lo));
        x0 = at(xs, n, k);
        x1 = at(xs, n, k + 1);
    }
    // the hit's half-local position, or -1
    __device__ __forceinline__ int finish(const float* xs, int n, int st, float xp, float tol, const uint32_t* used) {
        while (x0 < lo) {
            ++k;
            x0 = x1;
            x1 = at(xs, n, k + 1);
        }
        int best = -1;
        if (x0 <= hi) {
            float bd = fabsf(x0 - xp);
            if (bd <= tol && !is_used(used, st + k)) best = st + k;
            while (x1 <= hi) {
                ++k;
                const float d = fabsf(x1 - xp);
                if (d <= tol && (best < 0 || d < bd) && !is_used(used, st + k)) {
                    best = st + k;
                    bd = d;
                }
                x1 = at(xs, n, k + 1);
            }
        }
        return best;
    }
};
__device__ __forceinline__ int closest_hit(const float* xs, const HitMap m, int n, int st, float xp, float tol,
                                           const uint32_t* used) {
    Near q;
    q.start(xs, m, n, xp, tol);
    return q.finish(xs, n, st, xp, tol, used);
}

constexpr int kGainRow = 20;  // floats per hit pattern in shared memory (18, padded to 16-byte words)

struct Trip {
    int pos[6];
    float th[3], dth[3];
    float chi2, score;
    int nx;
};

// Triplet -> exact 3-hit model, extension to the other x-layers (closest hit
// within ext_tol, ties to the smaller x), least-squares fit and chi2 cut.
// The fit is done on residuals y_j of the hits from the 3-hit model, formed
// with error-free transformations so that they keep ~1e-7 mm accuracy; the
// correction dth = G y and the chi2 are then computed from small numbers.
// Returns 0 (fewer than 5 hits), 1 (chi2 cut) or 2 (candidate).
__device__ __forceinline__ int do_triplet(const DevParams& P, const IterP& I, const float* X, const int* szl,
                                          const HitMap map, const float* sG, const int* sMask, const uint32_t* used,
                                          int k1, int k2, int k3, Trip& o) {
    const int p1 = szl[I.s1] + k1, p2 = szl[I.s2] + k2, p3 = szl[I.s3] + k3;
    const float x1 = X[p1], x2 = X[p2], x3 = X[p3];
    const float t13 = (x3 - x1) * I.inv_dz31;
    const float base = fmaf(I.dz21, t13, x1);
    const float c3 = (x2 - base) * I.inv_k3;
    const float b3 = fmaf(-c3, I.q31, t13);
    const float a3 = x1 - fmaf(c3, I.f1, b3 * I.zb1);
    int nx = 3, m = (1 << I.s1) | (1 << I.s2) | (1 << I.s3);
#pragma unroll
    for (int s = 0; s < 6; ++s) o.pos[s] = s == I.s1 ? p1 : s == I.s2 ? p2 : s == I.s3 ? p3 : -1;
    Near nr[3];
    float xp[3];
    int zs[3], zn[3];
#pragma unroll
    for (int e = 0; e < 3; ++e) {
        const int sx = I.ext[e];
        xp[e] = fmaf(c3, P.xf_hi[sx], fmaf(b3, P.xzb[sx], a3));
        zs[e] = szl[sx];
        zn[e] = szl[sx + 1] - zs[e];
        nr[e].start(X + zs[e], map.zone(sx), zn[e], xp[e], P.ext_tol);
    }
#pragma unroll
    for (int e = 0; e < 3; ++e) {
        const int sx = I.ext[e];
        const int p = nr[e].finish(X + zs[e], zn[e], zs[e], xp[e], P.ext_tol, used);
        nx += p >= 0;
        m |= (p >= 0) << sx;
#pragma unroll
        for (int s = 0; s < 6; ++s) o.pos[s] = s == sx ? p : o.pos[s];
    }
    if (nx < 5) return 0;
    // gain of this hit pattern, [3][6] in rows of kGainRow
    float G[kGainRow];
#pragma unroll
    for (int q = 0; q < kGainRow / 4; ++q) {
        const float4 g = reinterpret_cast<const float4*>(sG + kGainRow * sMask[m])[q];
        G[4 * q] = g.x, G[4 * q + 1] = g.y, G[4 * q + 2] = g.z, G[4 * q + 3] = g.w;
    }
    float y[6];
#pragma unroll
    for (int s = 0; s < 6; ++s) {
        y[s] = 0.f;
        if (o.pos[s] >= 0) {
            float d, e;
            two_sum(X[o.pos[s]], -a3, d, e);
            float v = fmaf(-b3, P.xzb[s], d);
            v = fmaf(-c3, P.xf_hi[s], v);
            y[s] = v + fmaf(-c3, P.xf_lo[s], e);
        }
    }
    float da = 0.f, db = 0.f, dc = 0.f;
#pragma unroll
    for (int s = 0; s < 6; ++s) {
        da = fmaf(G[s], y[s], da);
        db = fmaf(G[6 + s], y[s], db);
        dc = fmaf(G[12 + s], y[s], dc);
    }
    float chi2 = 0.f;
#pragma unroll
    for (int s = 0; s < 6; ++s) {
        if (o.pos[s] >= 0) {
            const float r = y[s] - fmaf(dc, P.xf_hi[s], fmaf(db, P.xzb[s], da));
            chi2 = fmaf(r, r, chi2);
        }
    }
    chi2 *= P.inv_sx2;
    if (chi2 > P.chi2x_max * static_cast<float>(nx - 3)) return 1;
    o.th[0] = a3; o.th[1] = b3; o.th[2] = c3;
    o.dth[0] = da; o.dth[1] = db; o.dth[2] = dc;
    o.chi2 = chi2;
    o.nx = nx;
    const float sc = fmaf(P.w_chi2, chi2, fabsf(c3 + dc));
    o.score = nx == 6 ? sc : P.w5 * sc;
    return 2;
}
// x(z) of a seed at stereo slot u (3-hit model plus fit correction)
__device__ __forceinline__ float x_at_uv(const DevParams& P, const float* th, const float* dth, int u) {
    return fmaf(th[2], P.uf_hi[u], fmaf(th[1], P.uzb[u], th[0])) +
           fmaf(dth[2], P.uf_hi[u], fmaf(dth[1], P.uzb[u], dth[0]));
}

struct UV {
    int pos[6];
    int n;
    float chi2, tyr, beta, wm, zm;
};

// The q-th stereo layer a UV combination searches, in increasing z: those
// other than the initial one ui (iterative variant), or all six (ui = 6).
__device__ __forceinline__ int uv_layer(int ui, int q) { return q < ui ? q : q + 1; }
__device__ __forceinline__ float uv_xp(const DevParams& P, float Xl, float ty, int u) {
    return Xl - P.ut[u] * ty * P.uz[u];
}

// Whether a combination fails for certain: it can miss 6 - n_uv_min layers,
// and more of those it searches have no hit in their window.  In the iterative
// variant ty stays as it is only until the first hit, so it is the first
// layers that must all be empty.  The layers' tests do not depend on each
// other.
__device__ __forceinline__ bool uv_hopeless(const DevParams& P, const HitMap map, const float* Xs, bool hough, int pass,
                                            float ty) {
    const int ui = hough ? 6 : P.uv_init[pass];
    const int need = hough ? 6 : 7 - P.n_uv_min;  // layers to look at
    int empty = 0;
#pragma unroll
    for (int q = 0; q < 6; ++q) {
        if (q >= need) break;
        // (slot 6 only with q = 5, where an initial layer leaves five to search)
        const bool up = q >= ui;
        const int u1 = q < 5 ? q + 1 : 5;
        const float ut = up ? P.ut[u1] : P.ut[q], uz = up ? P.uz[u1] : P.uz[q];
        const int u = up ? u1 : q;
        const float xp = Xs[u] - ut * ty * uz;
        empty += map.zone(6 + u).empty(map_bin(xp - P.uv_tol), map_bin(xp + P.uv_tol));
    }
    return empty > 6 - P.n_uv_min;
}

// The hits of one UV combination (Section 3.4).  Iterative variant: start from
// the hit at half-local position pi of the initial stereo layer of `pass`, ty
// from the origin, closest hit within uv_tol in each remaining stereo layer in
// increasing z with ty averaging.  Hough: the closest hit in every layer at
// the given ty (pi < 0).  Xs[u] is the seed's x at stereo slot u.  A
// combination that can no longer reach n_uv_min stops early (it cannot be
// selected).  Positions (plus one) of slots 0..3 in the 16-bit fields of o.x,
// o.y, of slots 4, 5 in o.z; o.w is ty's bits; returns the number of hits.
__device__ __forceinline__ int uv_hits(const DevParams& P, const float* X, const int* szl, const HitMap map,
                                       const uint32_t* used, const float* Xs, bool hough, int pass, int pi, float ty,
                                       uint4& o) {
    ull lo4 = 0;
    unsigned hi2 = 0;
    int n = 0;
    const int nq = hough ? 6 : 5;
    if (!hough) {
        const int ui = P.uv_init[pass];
        n = 1;
        if (ui < 4) lo4 = ull(pi + 1) << (16 * ui);
        else hi2 = unsigned(pi + 1) << (16 * (ui - 4));
    }
#pragma unroll 1
    for (int q = 0; q < nq; ++q) {
        const int u = uv_layer(hough ? 6 : P.uv_init[pass], q);
        const float Xl = Xs[u];
        const float xp = uv_xp(P, Xl, ty, u);
        const int st = szl[6 + u];
        const int best = closest_hit(X + st, map.zone(6 + u), szl[7 + u] - st, st, xp, P.uv_tol, used);
        if (best >= 0) {
            if (!hough) {
                const float yl = (Xl - X[best]) * P.uinv_t[u];
                ty = 0.5f * fmaf(yl, P.uinv_z[u], ty);
            }
            if (u < 4) lo4 |= ull(best + 1) << (16 * u);
            else hi2 |= unsigned(best + 1) << (16 * (u - 4));
            ++n;
        }
        if (n + (nq - 1 - q) < P.n_uv_min) break;
    }
    o = make_uint4(static_cast<unsigned>(lo4), static_cast<unsigned>(lo4 >> 32), hi2, __float_as_uint(ty));
    return n;
}

// ty of the hit at half-local position pi of the initial layer of `pass`
__device__ __forceinline__ float uv_ty0(const DevParams& P, const float* X, const float* Xs, int pass, int pi) {
    const int ui = P.uv_init[pass];
    const float yi = (Xs[ui] - X[pi]) * P.uinv_t[ui];
    return yi * P.uinv_z[ui];
}

__device__ __forceinline__ UV uv_unpack(const uint4 v) {
    const unsigned w[3] = {v.x, v.y, v.z};
    UV u;
    u.n = 0;
#pragma unroll
    for (int r = 0; r < 6; ++r) {
        u.pos[r] = static_cast<int>((w[r >> 1] >> (16 * (r & 1))) & 0xFFFFu) - 1;
        u.n += u.pos[r] >= 0;
    }
    u.tyr = __uint_as_float(v.w);
    return u;
}

// Hough-cluster variant (Section 3.4, second approach), step 1 for the seeds
// kb .. nk - 1: every stereo hit of the half whose y lies in the first-layer
// window goes to coarse bin floor((y/z - lo) / w) of its layer's 64-bit
// occupancy mask; a cluster b is bins (b, b+1), its population the number of
// layers with a hit in it, counted for all clusters at once with three bit
// planes.  The kept clusters (most populated first, at least n_uv_min, ties to
// the smaller b) go to hcl[8 j ..], their number to hn[j].  Six lanes per seed,
// one stereo layer each, whose masks they exchange; five seeds per warp.
__device__ __forceinline__ void hough_select_in(const DevParams& P, const float* X, const int* szl, const HitMap map,
                                                const uint32_t* used, const float* Xs, int h, int kb, int nk,
                                                uint8_t* hcl, uint8_t* hn) {
    const int lane = threadIdx.x & 31, g = lane / 6, u = lane - 6 * g;
    for (int j0 = kb + 5 * (threadIdx.x >> 5); j0 < nk; j0 += 5 * (blockDim.x >> 5)) {
        const int j = g < 5 ? j0 + g : nk;  // (two lanes of the warp have no seed)
        ull m = 0;
        if (j < nk) {
            const float Xl = Xs[6 * j + u], t = P.ut[u];
            const float xa = fmaf(-P.uv_yhi[h], t, Xl), xb = fmaf(-P.uv_ylo[h], t, Xl);
            const int st = szl[6 + u], n = szl[7 + u] - st;
            const HitMap mz = map.zone(6 + u);
            const int lo = zlo(X + st, mz, n, fminf(xa, xb)), hi = zhi(X + st, mz, n, fmaxf(xa, xb));
            for (int k = lo; k < hi; ++k) {
                if (is_used(used, st + k)) continue;
                const float ty = (Xl - X[st + k]) * P.uinv_t[u] * P.uinv_z[u];
                const int b = min(max(__float2int_rd((ty - P.h_lo[h]) * P.h_inv_w), 0), P.h_bins - 1);
                m |= 1ull << b;
            }
        }
        const ull c = m | (m >> 1);  // bit b: a hit in bin b or b + 1
        ull s0 = 0, s1 = 0, s2 = 0;
#pragma unroll
        for (int q = 0; q < 6; ++q) {
            const ull cq = __shfl_sync(0xffffffffu, c, min(6 * g + q, 31));
            const ull c0 = s0 & cq;
            s0 ^= cq;
            const ull c1 = s1 & c0;
            s1 ^= c0;
            s2 |= c1;
        }
        const ull valid = ~0ull >> (65 - P.h_bins);  // clusters 0 .. bins-2
        int ns = 0;                                  // clusters before the population at hand
        for (int p = 6; p >= P.n_uv_min && ns < P.h_clusters; --p) {
            ull e = valid & ((p & 1) ? s0 : ~s0) & ((p & 2) ? s1 : ~s1) & ((p & 4) ? s2 : ~s2);
            const int c = __popcll(e);
            // lane u finds the kept clusters u and u + 6
            for (int k = u, q = ns; j < nk && k < min(P.h_clusters, ns + c); k += 6) {
                if (k < ns) continue;
                for (; q < k; ++q) e &= e - 1;
                hcl[8 * j + k] = static_cast<uint8_t>(__ffsll(static_cast<long long>(e)) - 1);
            }
            ns += c;
        }
        if (j < nk && u == 0) hn[j] = static_cast<uint8_t>(min(ns, P.h_clusters));
    }
}

// The Hough selection and the cold paths of the UV step each come as an
// inlined body (_in) and a call that is not inlined (_out).  The seeding
// kernel calls the _out forms except in its HLT2-style instantiation: their
// code and registers then stay out of the hot phases of the iterative HLT1
// path, which never or rarely runs them.
static __device__ __noinline__ void hough_select_out(const DevParams& P, const float* X, const int* szl,
                                                     const HitMap map, const uint32_t* used, const float* Xs, int h,
                                                     int kb, int nk, uint8_t* hcl, uint8_t* hn) {
    hough_select_in(P, X, szl, map, used, Xs, h, kb, nk, hcl, hn);
}

__device__ __forceinline__ float hough_ty(const DevParams& P, int h, int b, int f) {
    return fmaf(P.h_w, static_cast<float>(b) + (static_cast<float>(f) + 0.5f) * P.h_step, P.h_lo[h]);
}

// Straight-line fit y = y0 + ty z of a complete chain (o.pos, o.n, o.tyr).
// The y of each hit is formed as a float-float from error-free
// transformations and fitted relative to the line y = tyr z, so chi2_y keeps
// ~1e-6 relative accuracy.
static __device__ void uv_fit(const DevParams& P, const float* X, const float* th, const float* dth, UV& o) {
    float w[6];
    float sw = 0.f, sz = 0.f;
    const float ty = o.tyr;
#pragma unroll
    for (int u = 0; u < 6; ++u) {
        w[u] = 0.f;
        if (o.pos[u] < 0) continue;
        const float xh = X[o.pos[u]];
        // D = x(z_u) - x_hit as hi + lo
        float s, e, p, pe, s2, e2, p2, pe2, s3, e3;
        two_sum(th[0], -xh, s, e);
        two_prod(th[1], P.uzb[u], p, pe);
        two_sum(s, p, s2, e2);
        two_prod(th[2], P.uf_hi[u], p2, pe2);
        two_sum(s2, p2, s3, e3);
        const float lo = ((e + pe) + (e2 + pe2)) + (e3 + fmaf(th[2], P.uf_lo[u],
                          fmaf(dth[2], P.uf_hi[u], fmaf(dth[1], P.uzb[u], dth[0]))));
        // y = D / t as hi + lo: the remainder of the rounded quotient is exact,
        // so a reciprocal multiply loses nothing
        const float t = P.ut[u], it = P.uinv_t[u];
        const float yh = s3 * it;
        const float rm = fmaf(-yh, t, s3);
        const float yl = (rm + lo) * it;
        w[u] = fmaf(-ty, P.uz[u], yh) + yl;
        sw += w[u];
        sz += P.uzt[u];
    }
    const float inv_n = 1.f / static_cast<float>(o.n);
    const float wm = sw * inv_n, zm = sz * inv_n;
    float szz = 0.f, szw = 0.f;
#pragma unroll
    for (int u = 0; u < 6; ++u) {
        if (o.pos[u] < 0) continue;
        const float dz = P.uzt[u] - zm;
        szz = fmaf(dz, dz, szz);
        szw = fmaf(dz, w[u] - wm, szw);
    }
    const float beta = szw / szz;
    float chi2 = 0.f;
#pragma unroll
    for (int u = 0; u < 6; ++u) {
        if (o.pos[u] < 0) continue;
        const float r = (w[u] - wm) - beta * (P.uzt[u] - zm);
        chi2 = fmaf(r, r, chi2);
    }
    o.chi2 = chi2 * P.inv_sy2;
    o.beta = beta;
    o.wm = wm;
    o.zm = zm;
}

// A selection key per UV combination: fewer missing hits, then smaller chi2_y,
// then pass A, then the earlier initial hit (the order of Section 3.4's
// choice); the lowest 13 bits carry where the combination's hits were stored
// (kUvNotStored if they were not) and never decide.
constexpr int kUvNotStored = 8191;

__device__ __forceinline__ ull uv_key(int n, float chi2, int pass, int kinit, int stored) {
    return (ull(6 - n) << 61) | (ull(__float_as_uint(chi2) & 0x7fffffffu) << 30) | (ull(pass) << 29) |
           (ull(kinit) << 13) | ull(stored);
}

// A candidate of the x-z search, as it lies in the scratch.
struct alignas(16) Cand {
    float4 th;    // 3-hit model, chi2
    float4 dth;   // fit correction, score
    int4 p, q;    // half-local hit positions per x slot (-1: none); q.z: hits, q.w unused
};
__device__ __forceinline__ int cand_pos(const int4 p, const int4 q, int s) {
    return s == 0 ? p.x : s == 1 ? p.y : s == 2 ? p.z : s == 3 ? p.w : s == 4 ? q.x : q.y;
}

// x-z model of a candidate: th (3-hit model) and dth (fit correction)
struct XzModel {
    float th[3], dth[3];
};
__device__ __forceinline__ XzModel xz_model(const Cand* c) {
    const float4 a = c->th, b = c->dth;
    return XzModel{{a.x, a.y, a.z}, {b.x, b.y, b.z}};
}

// A valid UV combination, as it lies in the scratch: its hits and ty
// (uv_hits), then (seed, pass | initial hit << 1), which the fit's (chi2_y,
// beta, wm, zm) replace.
struct alignas(16) UvRec {
    uint4 v;
    float4 f;
};

// Cold path of the UV step: a valid combination that found the chain store
// full is fitted where it was found and takes part in the seed's choice by
// its key alone (its hits are searched again if it wins).
__device__ __forceinline__ void uv_fit_unstored_in(const DevParams& P, const float* X, const Cand* c,
                                                   uint4 v, ull* ukey, int pass, int kinit) {
    const XzModel m = xz_model(c);
    UV u = uv_unpack(v);
    uv_fit(P, X, m.th, m.dth, u);
    atomicMin(ukey, uv_key(u.n, u.chi2, pass, kinit, kUvNotStored));
}
static __device__ __noinline__ void uv_fit_unstored_out(const DevParams& P, const float* X, const Cand* c,
                                                        uint4 v, ull* ukey, int pass, int kinit) {
    uv_fit_unstored_in(P, X, c, v, ukey, pass, kinit);
}

// Cold path of the output step: the winning combination of a seed whose
// hits were not stored, searched again (same chain, same result) and fitted.
__device__ __forceinline__ UV uv_redo_in(const DevParams& P, const float* X, const int* szl, const HitMap map,
                                         const uint32_t* used, const float* Xs, const Cand* c,
                                         int h, const uint8_t* hc, ull key) {
    const int kinit = static_cast<int>((key >> 13) & 0xFFFFu);
    uint4 v;
    if (P.uv_mode == 1) {
        const int r = kinit / P.h_fine;
        uv_hits(P, X, szl, map, used, Xs, true, 0, -1, hough_ty(P, h, hc[r], kinit - r * P.h_fine), v);
    } else {
        const int pass = static_cast<int>((key >> 29) & 1);
        const int pi = szl[6 + P.uv_init[pass]] + kinit;
        uv_hits(P, X, szl, map, used, Xs, false, pass, pi, uv_ty0(P, X, Xs, pass, pi), v);
    }
    const XzModel m = xz_model(c);
    UV u = uv_unpack(v);
    uv_fit(P, X, m.th, m.dth, u);
    return u;
}
static __device__ __noinline__ UV uv_redo_out(const DevParams& P, const float* X, const int* szl, const HitMap map,
                                       const uint32_t* used, const float* Xs, const Cand* c, int h,
                                              const uint8_t* hc, ull key) {
    return uv_redo_in(P, X, szl, map, used, Xs, c, h, hc, key);
}

// The third-hit window of one pair (Eq. invp and the k3 band); false if the
// pair has none.
__device__ __forceinline__ bool pair_band(const DevParams& P, const IterP& I, float x1, float x3, float& lo, float& hi) {
    const float t13 = (x3 - x1) * I.inv_dz31;
    const float x0 = fmaf(-I.z1, t13, x1);
    const float ip = fmaf(P.invp_b * x0, x0, P.invp_a * fabsf(x0));
    const float sg = x0 > 0.f ? 1.f : -1.f;
    const float ulo = fmaf(I.mlo_k, ip, -I.c0), uhi = fmaf(I.mhi_k, ip, I.c0);
    const float bs = fmaf(I.dz21, t13, x1);
    const float xa = fmaf(I.k3, -sg * ulo, bs), xb = fmaf(I.k3, -sg * uhi, bs);
    lo = fminf(xa, xb);
    hi = fmaxf(xa, xb);
    return ip > 0.f;
}

constexpr int kTripPerCand = 2;  // triplets of one round per candidate slot, above which the item overflows

// The warps of the x-z search first test 32 pairs at a time against the hit
// map and queue those that may succeed until they fill the lanes for the exact
// window; the triplets queue up per warp until the block has walked kWalk
// groups of 32 pairs per warp, and then go one to a thread.  The UV search
// tests kUvBlock combinations at a time and gives the ones left one to a
// thread likewise.
constexpr int kPairQueue = 64;
constexpr int kTripQueue = 128;
constexpr int kWalk = 24;
// Rounds with more pairs per first hit than kDensePairs, whose pairs find more
// triplets each, walk fewer groups, so that the queues seldom run over.  1000
// Run-3-like events (13 pairs per first hit): 220 us with 8 groups, 213 with 12,
// 211 with 16, 210 with 24; 300 events by direct calls 98, 98, 96, 94 us; 2000
// uneven events 642, 633, 650, 680 us, 627 with this rule.  Where a queue runs
// over all the same (wide bands), the walk is repeated with as many groups as the
// triplets found say, and the item's next walks follow their own counts: a
// quarter of the groups for the rest of a round, as before, made 300 events with
// the band up to 20 times the expected curvature 210 us, 167 this way, 5 times
// 133 and 121.
constexpr int kWalkDense = 12;
constexpr int kDensePairs = 24;
constexpr int kUvBlock = 1024;

// Shared memory that the phases of an item use in turn: the warps' queues of
// the x-z search; the clone table; the UV list with the UV keys and the seeds'
// x at the stereo layers.
static __host__ __device__ inline size_t seed_phase_bytes(int threads, int tbl_smem, int key_smem) {
    const size_t walk = (sizeof(uint32_t) * kPairQueue + sizeof(uint2) * kTripQueue) * (threads / 32);
    const size_t tbl = sizeof(ull) * tbl_smem;
    const size_t uv = sizeof(uint32_t) * kUvBlock + (sizeof(ull) + 6 * sizeof(float)) * key_smem;
    const size_t m = walk > uv ? walk : uv;
    return align16(m > tbl ? m : tbl);
}
constexpr size_t kMapBytes = 12 * (sizeof(uint32_t) * kMapStride + sizeof(uint16_t) * kMapWords);
static_assert(kMapBytes % 16 == 0, "16-byte aligned parts");

static __host__ __device__ inline size_t seed_smem_size(int threads, int smem_hits, int tbl_smem, int key_smem) {
    return align16(sizeof(float) * smem_hits) + kMapBytes + seed_phase_bytes(threads, tbl_smem, key_smem) +
           (sizeof(int2) + sizeof(int) + sizeof(uint16_t)) * threads + sizeof(int) * (2 * kScanInts + 16);
}

// max_hits: hits of a half (the taken-hit bits)
static __host__ __device__ inline size_t seed_slot_size(int cand_cap, int uv_cap, int tbl_cap, int max_hits) {
    return (sizeof(Cand) + sizeof(int)) * size_t(cand_cap) + sizeof(ull) * (size_t(tbl_cap) + cand_cap) + 16 +
           sizeof(UvRec) * size_t(uv_cap) + sizeof(float) * 6 * size_t(cand_cap) + 9 * size_t(cand_cap) + 4 +
           sizeof(uint32_t) * ((size_t(max_hits) + 31) / 32);
}

constexpr int kDeferRounds = 2;       // matching left to idle CTAs once fewer seeding items than this per CTA remain
// A wait for an announced event ends after SeedArgs::wait_ns of the global
// timer; the poll count is a second bound in case the timer stalls.
constexpr int kReadySpinsMax = 1 << 24;

__device__ __forceinline__ unsigned long long global_ns() {
    unsigned long long t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}

// A CTA's scratch in global memory (SeedArgs::slot).
struct SeedSlot {
    int CC;            // candidates an item may have
    int uv_cap;        // valid UV combinations stored
    Cand* cand;        // [CC] the candidates in the order of the search
    UvRec* uv;         // [uv_cap] the valid UV combinations
    ull* tbl;          // clone table, if it does not fit in shared memory
    ull* key;          // UV keys, if they do not
    float* xs;         // x at the stereo layers of the kept seeds, if not in shared memory
    int* kept;         // [CC] candidates left by the clone kill
    uint8_t* hcl;      // Hough variant: kept clusters per seed
    uint8_t* hn;       // and their count
    uint32_t* used;    // HLT2-style mode: bits of the half's hits taken by earlier iterations
    __device__ __forceinline__ SeedSlot(uint8_t* slot, int cc, int uvc, int tbl_cap) : CC(cc), uv_cap(uvc) {
        cand = reinterpret_cast<Cand*>(slot);
        uv = reinterpret_cast<UvRec*>(cand + CC);
        key = reinterpret_cast<ull*>(uv + uv_cap);
        tbl = key + CC;
        xs = reinterpret_cast<float*>(tbl + tbl_cap);
        kept = reinterpret_cast<int*>(xs + 6 * CC);
        hcl = reinterpret_cast<uint8_t*>(kept + CC);
        hn = hcl + 8 * CC;
        used = reinterpret_cast<uint32_t*>((reinterpret_cast<uintptr_t>(hn + CC) + 3) & ~uintptr_t(3));
    }
};

// A CTA's variables in shared memory.
struct SeedVars {
    ull start;         // pool place of the item's records
    ull ctr[8];        // work counters: pairs, triplets, extended, candidates, kept, UV initial hits, valid UV
                       // combinations, seeds
    ull mctr[4];       // grid pairs, preselected pairs, Long tracks, evaluated pairs
    ull mbar;          // the staging copies' barrier (one phase per staged item)
    int item, match, cnt;
    int nvalid, nlist;
    int seg[2];        // first pair or combination of a round's second and third part
    int wcnt[32];      // triplets found per warp
};

// What the phases of an item share.
struct SeedItem {
    int h;             // detector half
    int it_lo, it_hi;  // iterations of this pass
    bool hough;
};

// The shared-memory arrays, in the order of seed_smem_size.
struct SeedSm {
    float* sx;
    uint32_t* bits;
    uint16_t* first;
    unsigned char* phase;
    int2* sA;          // owner: .x + item number is where its hits are; .y the T1 hit's x, or the seed
    int* sPS;          // owner: number of its first pair or combination
    int* tmp;          // block scans
    int* nz;
    int* szl;          // first half-local position of each slot
    uint16_t* sB;      // owner: its T1 hit
    __device__ __forceinline__ SeedSm(unsigned char* smem, int T, int smem_hits, int tbl_smem, int key_smem) {
        unsigned char* sp = smem;
        sx = reinterpret_cast<float*>(sp);
        sp += align16(sizeof(float) * smem_hits);
        bits = reinterpret_cast<uint32_t*>(sp);
        first = reinterpret_cast<uint16_t*>(bits + 12 * kMapStride);
        sp += kMapBytes;
        phase = sp;
        sp += seed_phase_bytes(T, tbl_smem, key_smem);
        sA = reinterpret_cast<int2*>(sp);
        sPS = reinterpret_cast<int*>(sA + T);
        tmp = sPS + T;
        nz = tmp + kScanInts;
        szl = nz + kScanInts;
        sB = reinterpret_cast<uint16_t*>(szl + 16);
    }
};

// The owner of each of 32 consecutive items from p0 on, one per lane: `own` is
// the owner of item p0 (owners have at least one item and ascending first
// items sPS); a bit per owner that starts among the 32 is counted up to the
// lane's.  Moves `own` to the owner of item p0 + 32.
__device__ __forceinline__ int owner_of_lane(const int* sPS, int n_own, int p0, int lane, int& own) {
    const int d = own + 1 + lane < n_own ? sPS[own + 1 + lane] - p0 : 64;
    const unsigned starts = __reduce_or_sync(0xffffffffu, d < 32 ? 1u << d : 0u);
    const int o = own + __popc(starts & (0xffffffffu >> (31 - lane)));
    own += __popc(__ballot_sync(0xffffffffu, d <= 32));
    return o;
}
// the owner of item p0
__device__ __forceinline__ int owner_of_item(const int* sPS, int n_own, int p0, int lane) {
    int own = 0;
    for (int o = lane; o < n_own; o += 32) own += sPS[o] <= p0;
    return __reduce_add_sync(0xffffffffu, own) - 1;
}

// The x-z search of one pass (its iterations it_lo .. it_hi - 1): its
// candidates follow the ncand ones in the slot, in the order of the search
// (iteration, T1 hit, T3 hit, T2 hit).  Each round takes up to R <= T first
// hits (the iterations' T1 layers in order) and finds their T3 windows; a
// block scan numbers the pairs.  The warps walk contiguous shares of them
// (kWalk and kPairQueue above say how), so the queued triplets, warp after
// warp, are in order, and so are the candidates that a block scan numbers.
// False if the item has more triplets in a round or more candidates than it
// may.
template <bool kSeq>
__device__ __forceinline__ bool xz_search(const DevParams& P, const SeedItem& it_, const SeedSm& M, SeedVars& V,
                                          const SeedSlot& S, const float* X, const HitMap map, const float* sG,
                                          const int* sMask, int R, int& ncand, int& spar) {
    const int T = blockDim.x, tid = threadIdx.x, lane = tid & 31, wid = tid >> 5, n_warps = T >> 5;
    const int CC = S.CC, TC = kTripPerCand * CC;
    const int it_lo = it_.it_lo, it_hi = it_.it_hi;
    const int* szl = M.szl;
    const uint32_t* used = kSeq ? S.used : nullptr;
    uint2* const tqs = reinterpret_cast<uint2*>(M.phase);  // the warps' queues: triplets, then pairs
    uint2* const tq = tqs + kTripQueue * wid;
    uint32_t* const pq = reinterpret_cast<uint32_t*>(tqs + kTripQueue * n_warps) + kPairQueue * wid;
    int K = kWalk * n_warps;  // groups of a block's next walk
    int n_items = 0;
    for (int it = it_lo; it < it_hi; ++it) n_items += szl[P.it[it].s1 + 1] - szl[P.it[it].s1];
    for (int b1 = 0; b1 < n_items; b1 += R) {
        const int i = tid < R ? b1 + tid : n_items;
        int np = 0, p3 = 0, own1 = 0;
        float x1o = 0.f;
        if (i < n_items) {
            int it = it_lo, k1 = i;
#pragma unroll
            for (int q = 0; q < 2; ++q) {
                if (it + 1 < it_hi) {
                    const int n1 = szl[P.it[it].s1 + 1] - szl[P.it[it].s1];
                    if (k1 >= n1) {
                        k1 -= n1;
                        ++it;
                    }
                }
            }
            const IterP& I = P.it[it];
            x1o = X[szl[I.s1] + k1];
            const float xc = I.scale3 * x1o;
            const int st3 = szl[I.s3], n3 = szl[I.s3 + 1] - st3;
            const HitMap m3 = map.zone(I.s3);
            const int lo3 = zlo(X + st3, m3, n3, xc - I.dx3);
            // (a window may end before it starts: layers against the flight direction, a negative scale)
            np = max(zhi(X + st3, m3, n3, xc + I.dx3) - lo3, 0);
            if (is_used(used, szl[I.s1] + k1)) np = 0;
            p3 = st3 + lo3;
            own1 = k1;
        }
        int tot_p, rank, n_own;
        const int ps = block_exscan1_nz(np, M.tmp, M.nz, spar, tot_p, rank, n_own);
        if (np > 0) {  // T1 hits with an empty window take no place
            M.sPS[rank] = ps;
            M.sB[rank] = static_cast<uint16_t>(own1);
            M.sA[rank] = make_int2(p3 - ps, __float_as_int(x1o));  // pair p's T3 hit is at .x + p
        }
        // first pairs of the pass's second and third iteration in this round
        const int i1 = szl[P.it[it_lo].s1 + 1] - szl[P.it[it_lo].s1];
        const int i2 = it_lo + 1 < it_hi ? i1 + szl[P.it[it_lo + 1].s1 + 1] - szl[P.it[it_lo + 1].s1] : i1;
        if (tid < R && b1 + tid == i1) V.seg[0] = ps;
        if (tid < R && b1 + tid == i2) V.seg[1] = ps;
        if (tid == 0) V.ctr[0] += tot_p;
        __syncthreads();
        const int sg1 = i1 <= b1 ? 0 : i1 < b1 + R ? V.seg[0] : tot_p;
        const int sg2 = i2 <= b1 ? 0 : i2 < b1 + R ? V.seg[1] : tot_p;
        // groups of 32 pairs, none across two iterations
        const int G1 = (sg1 + 31) >> 5, G2 = G1 + ((sg2 - sg1 + 31) >> 5), G = G2 + ((tot_p - sg2 + 31) >> 5);
        int round_trips = 0;
        const int most = (tot_p <= kDensePairs * n_own ? kWalk : kWalkDense) * n_warps;
        K = min(K, most);
        int resume = 0;           // triplets already taken of a single group that has more than a queue holds
        for (int B = 0; B < G;) {
            const int nB = min(K, G - B);
            const int per = (nB + n_warps - 1) / n_warps;
            const int gb = B + min(per * wid, nB), ge = B + min(per * (wid + 1), nB);
            int all = 0;  // triplets found
#pragma unroll 1
            for (int it = it_lo; it < it_hi; ++it) {
                const int gs = it == it_lo ? 0 : it == it_lo + 1 ? G1 : G2, gt = it == it_lo ? G1 : it == it_lo + 1 ? G2 : G;
                const int g0 = max(gb, gs), g1 = min(ge, gt);
                if (g0 >= g1) continue;
                const IterP& I = P.it[it];
                const int st2 = szl[I.s2], n2 = szl[I.s2 + 1] - st2, st3 = szl[I.s3];
                const HitMap m2 = map.zone(I.s2);
                int p0 = (it == it_lo ? 0 : it == it_lo + 1 ? sg1 : sg2) + 32 * (g0 - gs);
                const int p1 = min(p0 + 32 * (g1 - g0), it == it_lo ? sg1 : it == it_lo + 1 ? sg2 : tot_p);
                int own = owner_of_item(M.sPS, n_own, p0, lane);
                int ph = 0, pn = 0;  // the pair queue's head and fill
                while (pn > 0 || p0 < p1) {
                    while (pn < 32 && p0 < p1) {  // 32 pairs against the hit map
                        const int o = owner_of_lane(M.sPS, n_own, p0, lane, own);
                        bool pass = false;
                        int k3 = 0;
                        if (p0 + lane < p1) {
                            const int2 a = M.sA[o];
                            k3 = a.x + p0 + lane;
                            float lo, hi;
                            pass = pair_band(P, I, __int_as_float(a.y), X[k3], lo, hi);
                            pass &= !m2.empty(map_bin(lo), map_bin(hi));
                            if (kSeq) pass &= !is_used(used, k3);
                        }
                        const unsigned some = __ballot_sync(0xffffffffu, pass);
                        if (pass)
                            pq[(ph + pn + __popc(some & ((1u << lane) - 1u))) & (kPairQueue - 1)] =
                                (unsigned(o) << 20) | unsigned(k3);
                        pn += __popc(some);
                        p0 += 32;
                    }
                    __syncwarp();
                    const int nb = min(pn, 32);  // the exact windows of the next 32 that remain
                    int c = 0, lo2 = 0;
                    unsigned k13 = 0;
                    if (lane < nb) {
                        const unsigned e = pq[(ph + lane) & (kPairQueue - 1)];
                        const int o = e >> 20, k3 = e & 0xFFFFF;
                        float lo, hi;
                        pair_band(P, I, __int_as_float(M.sA[o].y), X[k3], lo, hi);
                        k13 = (unsigned(M.sB[o]) << 16) | unsigned(k3 - st3);
                        for (int k = m2.from(map_bin(lo)); k < n2; ++k) {
                            const float x = X[st2 + k];
                            if (hi < x) break;
                            if (x < lo || is_used(used, st2 + k)) continue;
                            if (c == 0) lo2 = k;
                            ++c;
                        }
                    }
                    ph += nb;
                    pn -= nb;
                    const unsigned some = __ballot_sync(0xffffffffu, c > 0);
                    int ex = __popc(some & ((1u << lane) - 1u)), n = __popc(some);
                    if (__any_sync(0xffffffffu, c > 1)) {
                        ex = c;
#pragma unroll
                        for (int s = 1; s < 32; s <<= 1) {
                            const int y = __shfl_up_sync(0xffffffffu, ex, s);
                            if (lane >= s) ex += y;
                        }
                        n = __shfl_sync(0xffffffffu, ex, 31);
                        ex -= c;
                    }
                    for (int q = 0; q < c; ++q, ++lo2) {
                        while (is_used(used, st2 + lo2)) ++lo2;
                        const int r = all + ex + q - resume;
                        if (r >= 0 && r < kTripQueue) tq[r] = make_uint2(k13, (unsigned(it) << 16) | unsigned(lo2));
                    }
                    all += n;
                    __syncwarp();
                }
            }
            if (lane == 0) V.wcnt[wid] = max(all - resume, 0);
            const bool more = __syncthreads_or(all - resume > kTripQueue);  // some warp's queue was too short
            int wb = lane < n_warps ? V.wcnt[lane] : 0;
            if (more || K < most) {
                // the next walk takes as many groups as fill three quarters of
                // the queue of the warp with most triplets
                const int fit = per * (kTripQueue * 3 / 4) / max(__reduce_max_sync(0xffffffffu, wb), 1);
                K = more && per == 1 ? max(1, nB / 4) : min(max(fit, 1) * n_warps, most);
                if (more && nB > 1) {
                    __syncthreads();  // (the counts' last reads)
                    continue;
                }
                wb = min(wb, kTripQueue);
            }
            // the queued triplets, one to a thread
            const int nt = __reduce_add_sync(0xffffffffu, wb);
#pragma unroll
            for (int s = 1; s < 32; s <<= 1) {
                const int y = __shfl_up_sync(0xffffffffu, wb, s);
                if (lane >= s) wb += y;
            }
            round_trips += nt;
            if (round_trips > TC) return false;
            for (int b = 0; b < nt; b += T) {
                const int t = b + tid;
                int code = -1;
                Trip o;
                int w = 0;  // the warp whose queue holds triplet t
#pragma unroll 1
                for (int q = 0; q < n_warps; ++q) w += __shfl_sync(0xffffffffu, wb, q) <= t;
                const int w0 = __shfl_sync(0xffffffffu, wb, (w - 1) & 31);
                if (t < nt) {
                    const uint2 tk = tqs[kTripQueue * w + t - (w > 0 ? w0 : 0)];
                    code = do_triplet(P, P.it[tk.y >> 16], X, szl, map, sG, sMask, used, tk.x >> 16, tk.y & 0xFFFFu,
                                      tk.x & 0xFFFFu, o);
                }
                // candidates in the low 16 bits, extended triplets (code >= 1)
                // in the high ones: at most one each per thread, so no carry
                int tot;
                const int co =
                    block_exscan1((code == 2 ? 1 : 0) | (code >= 1 ? 0x10000 : 0), M.tmp, spar, tot) & 0xFFFF;
                if (tid == 0) V.ctr[2] += tot >> 16;
                if (code == 2 && ncand + co < CC) {
                    Cand* c = S.cand + (ncand + co);
                    c->th = make_float4(o.th[0], o.th[1], o.th[2], o.chi2);
                    c->dth = make_float4(o.dth[0], o.dth[1], o.dth[2], o.score);
                    c->p = make_int4(o.pos[0], o.pos[1], o.pos[2], o.pos[3]);
                    c->q = make_int4(o.pos[4], o.pos[5], o.nx, 0);
                }
                ncand += tot & 0xFFFF;
            }
            if (tid == 0) V.ctr[1] += nt;
            __syncthreads();  // the queues' last reads
            if (more) {
                resume += kTripQueue;
            } else {
                resume = 0;
                B += nB;
            }
        }
    }
    return ncand <= CC;
}

// Clone killing (Eq. seed_clone_score and the two-pass vote of Section 3.3.4)
// of the candidates numbered cb0 .. ncand - 1; the ones left go to S.kept from
// place nk on, in order.
__device__ __forceinline__ void clone_kill(const SeedSm& M, const SeedSlot& S, ull* tbl, int nxh, int cb0, int ncand,
                                           int& nk, int& spar) {
    const int T = blockDim.x, tid = threadIdx.x;
    for (int i = tid; i < nxh; i += T) tbl[i] = ~0ull;
    __syncthreads();
    for (int k = cb0 + tid; k < ncand; k += T) {
        const Cand* c = S.cand + k;
        const ull key = (ull(__float_as_uint(c->dth.w)) << 32) | unsigned(k);
        const int4 p = c->p, q = c->q;
#pragma unroll
        for (int s = 0; s < 6; ++s)
            if (cand_pos(p, q, s) >= 0) atomicMin(&tbl[cand_pos(p, q, s)], key);
    }
    __syncthreads();
    for (int b = cb0; b < ncand; b += T) {
        const int k = b + tid;
        int keep = 0;
        if (k < ncand) {
            const Cand* c = S.cand + k;
            const ull key = (ull(__float_as_uint(c->dth.w)) << 32) | unsigned(k);
            const int4 p = c->p, q = c->q;
            int owned = 0;
#pragma unroll
            for (int s = 0; s < 6; ++s) owned += cand_pos(p, q, s) >= 0 && tbl[cand_pos(p, q, s)] == key;
            keep = owned >= 3 || (owned >= 2 && q.z == 6);
        }
        int tot;
        const int o = block_exscan1(keep, M.tmp, spar, tot);
        if (keep) S.kept[nk + o] = k;
        nk += tot;
    }
    __syncthreads();
}

// UV seeding (Section 3.4) of the kept seeds kb .. nk - 1: their best
// combination's key in ukey (~0 for none), the combinations in the slot.  One
// owner per (seed, pass), numbered pass-major (iterative), or per seed with
// its hypotheses (Hough); a block scan numbers a round's combinations, the
// warps test them kUvBlock at a time against the hit maps, and the ones left
// go one to a thread, in any order (the key decides).
template <bool kSeq>
__device__ __forceinline__ void uv_search(const DevParams& P, const SeedItem& it_, const SeedSm& M, SeedVars& V,
                                          const SeedSlot& S, const float* X, const HitMap map, ull* ukey, float* Xs,
                                          int kb, int nk, int& spar) {
    constexpr bool kOut = !kSeq;  // the out-of-line forms of the rarely run functions
    const int T = blockDim.x, tid = threadIdx.x, lane = tid & 31, wid = tid >> 5, n_warps = T >> 5;
    const int h = it_.h;
    const bool hough = it_.hough;
    const int* szl = M.szl;
    const uint32_t* used = kSeq ? S.used : nullptr;
    uint32_t* const list = reinterpret_cast<uint32_t*>(M.phase);
    const int nkp = nk - kb;
    const int nvs0 = min(V.nvalid, S.uv_cap);
    if (tid == 0) V.nlist = 0;
    for (int j = kb + tid; j < nk; j += T) {
        ukey[j] = ~0ull;
        const XzModel m = xz_model(S.cand + S.kept[j]);
#pragma unroll
        for (int u = 0; u < 6; ++u) Xs[6 * j + u] = x_at_uv(P, m.th, m.dth, u);
    }
    __syncthreads();
    if (hough) {
        if constexpr (kOut)
            hough_select_out(P, X, szl, map, used, Xs, h, kb, nk, S.hcl, S.hn);
        else
            hough_select_in(P, X, szl, map, used, Xs, h, kb, nk, S.hcl, S.hn);
        __syncthreads();
    }
    const int nuv = hough ? nkp : 2 * nkp;
    // ty of combination kinit of seed j (iterative: from its initial hit)
    auto start_ty = [&](int j, int pass, int kinit) {
        if (hough) {
            const int r = kinit / P.h_fine;
            return hough_ty(P, h, S.hcl[8 * j + r], kinit - r * P.h_fine);
        }
        return uv_ty0(P, X, Xs + 6 * j, pass, szl[6 + P.uv_init[pass]] + kinit);
    };
    for (int b = 0; b < nuv; b += T) {
        const int i = b + tid;
        int cntc = 0, lo = 0;
        if (i < nuv && hough) {
            cntc = S.hn[kb + i] * P.h_fine;
        } else if (i < nuv) {
            const int pass = i >= nkp, j = kb + i - (pass ? nkp : 0);
            const int ui = P.uv_init[pass];
            const float Xi = Xs[6 * j + ui];
            const float t = P.ut[ui];
            const float xa = fmaf(-P.uv_yhi[h], t, Xi), xb = fmaf(-P.uv_ylo[h], t, Xi);
            const int st = szl[6 + ui], n = szl[7 + ui] - st;
            // the window holds a few hits: its end by a forward scan
            const float wlo = fminf(xa, xb), whi = fmaxf(xa, xb);
            const float* xs = X + st;
            lo = zlo(xs, map.zone(6 + ui), n, wlo);
            int e = lo;
            while (e < n && !(whi < xs[e])) ++e;
            cntc = e - lo;
        }
        int tot, rank, n_own;
        const int ps = block_exscan1_nz(cntc, M.tmp, M.nz, spar, tot, rank, n_own);
        if (tid == 0) V.ctr[5] += tot;
        if (cntc > 0) {
            M.sPS[rank] = ps;
            M.sA[rank] = make_int2(lo - ps, kb + i - (!hough && i >= nkp ? nkp : 0));
        }
        if (i == nkp) V.seg[0] = ps;
        __syncthreads();
        const int sg = nkp <= b ? 0 : nkp < b + T ? V.seg[0] : tot;  // first combination of pass B
        for (int B = 0; B < tot; B += kUvBlock) {
            const int nB = min(kUvBlock, tot - B);
            const int per = ((((nB + 31) >> 5) + n_warps - 1) / n_warps) << 5;
            int c0 = B + min(per * wid, nB);
            const int c1 = B + min(per * (wid + 1), nB);
            int own = c0 < c1 ? owner_of_item(M.sPS, n_own, c0, lane) : 0;
            for (; c0 < c1; c0 += 32) {  // 32 combinations against the hit maps
                const int o = owner_of_lane(M.sPS, n_own, c0, lane, own);
                bool go = false;
                unsigned entry = 0;
                if (c0 + lane < c1) {
                    const int2 a = M.sA[o];
                    const int kinit = a.x + c0 + lane, pass = c0 + lane >= sg;
                    // an initial hit taken by an earlier iteration does not count
                    go = (hough || !is_used(used, szl[6 + P.uv_init[pass]] + kinit)) &&
                         !uv_hopeless(P, map, Xs + 6 * a.y, hough, pass, start_ty(a.y, pass, kinit));
                    entry = (unsigned(o) << 17) | (unsigned(pass) << 16) | unsigned(kinit);
                }
                const unsigned some = __ballot_sync(0xffffffffu, go);
                if (some == 0u) continue;
                int at = 0;
                if (lane == 0) at = atomicAdd(&V.nlist, __popc(some));
                at = __shfl_sync(0xffffffffu, at, 0);
                if (go) list[at + __popc(some & ((1u << lane) - 1u))] = entry;
            }
            __syncthreads();
            const int nl = V.nlist;
            for (int q = tid; q < nl; q += T) {
                const unsigned en = list[q];
                const int j = M.sA[en >> 17].y, pass = (en >> 16) & 1, kinit = en & 0xFFFFu;
                uint4 v;
                const int n = uv_hits(P, X, szl, map, used, Xs + 6 * j, hough, pass,
                                      szl[6 + P.uv_init[pass]] + kinit, start_ty(j, pass, kinit), v);
                if (n >= P.n_uv_min) {
                    const int sidx = atomicAdd(&V.nvalid, 1);
                    if (sidx < S.uv_cap) {
                        S.uv[sidx].v = v;
                        reinterpret_cast<uint2&>(S.uv[sidx].f) = make_uint2(unsigned(j), unsigned(pass) | (unsigned(kinit) << 1));
                    } else {
                        // store full: fit here; the winner is searched again at output
                        if constexpr (kOut)
                            uv_fit_unstored_out(P, X, S.cand + S.kept[j], v, &ukey[j], pass, kinit);
                        else
                            uv_fit_unstored_in(P, X, S.cand + S.kept[j], v, &ukey[j], pass, kinit);
                    }
                }
            }
            __syncthreads();
            if (tid == 0) V.nlist = 0;  // (the next block's appends follow a barrier or its own)
            if (B + kUvBlock < tot) __syncthreads();
        }
        __syncthreads();
    }
    // the stored combinations' fits, one per thread
    const int nvs = min(V.nvalid, S.uv_cap);
    for (int q = nvs0 + tid; q < nvs; q += T) {
        UvRec* r = S.uv + q;
        const uint2 mt = reinterpret_cast<const uint2&>(r->f);
        UV u = uv_unpack(r->v);
        const int j = static_cast<int>(mt.x);
        const XzModel m = xz_model(S.cand + S.kept[j]);
        uv_fit(P, X, m.th, m.dth, u);
        r->f = make_float4(u.chi2, u.beta, u.wm, u.zm);
        atomicMin(&ukey[j], uv_key(u.n, u.chi2, static_cast<int>(mt.y & 1u), static_cast<int>(mt.y >> 1), q));
    }
    __syncthreads();
}

// kSeq: compiled with the HLT2-style pass loop and taken-hit checks; the HLT1
// instantiation has neither (they fold away).
// kFuse: the kernel also matches each event, where the pool holds its
// records (HLT1 instantiation only).  The CTA that finishes the second of an
// event's two halves (a per-event counter) matches the event before its next
// item.  With defer_match, once fewer than kDeferRounds seeding items per CTA
// are left it announces the event in a ready list instead, and CTAs that find
// no seeding item left take the announced events (short items at the end
// balance the CTAs' finishing times); such a CTA waits (bounded) only while
// some event is still being seeded by a running CTA.  Kernels that share the
// GPU with others (the serving pipeline) do not defer: a waiting CTA would
// hold resources the other kernels could use.
template <int kT, int kR, bool kSeq, bool kFuse>
__global__ void __launch_bounds__(kT) __maxnreg__(kR)
k_seed(const __grid_constant__ DevParams P, const __grid_constant__ SeedArgs A) {
    extern __shared__ __align__(16) unsigned char smem[];
    __shared__ SeedVars V;
    // the x-z fit gains, indexed per thread by hit pattern: kept in shared
    // memory (divergent reads of kernel parameters serialise)
    __shared__ __align__(16) float sG[kMasks * kGainRow];
    __shared__ int sMask[64];
    const int T = blockDim.x, tid = threadIdx.x;
    const SeedSm M(smem, T, A.smem_hits, A.tbl_smem, A.key_smem);
    const SeedSlot S(A.slot + int64_t(blockIdx.x) * A.slot_stride, A.cand_cap, A.uv_cap, A.tbl_cap);
    const HitMap map{M.bits, M.first};
    const int* szl = M.szl;
    for (int i = tid; i < kMasks * 18; i += T) sG[kGainRow * (i / 18) + i % 18] = (&P.G[0][0][0])[i];
    for (int i = tid; i < 64; i += T) sMask[i] = P.mask_index[i];
    constexpr bool seq = kSeq;
    constexpr bool kOut = !kSeq;
    const uint32_t* used = kSeq ? S.used : nullptr;
    if (tid < 4) V.mctr[tid] = 0;
    if (tid < 8) V.ctr[tid] = 0;
    if (tid == 0) mbar_init(&V.mbar, 1);
    int spar = 0;  // which half of the scans' buffers the next one uses
    unsigned mphase = 0;
    bool stage_ok = true;
    pdl_signal();
    pdl_wait();  // the containers and the item order

    int64_t fin = -1;   // fused: event of the half this CTA finished last
    bool first = true;  // no item taken yet (thread 0)
    for (;;) {
        if (kFuse && fin >= 0) __threadfence();  // the half's records, before its count
        __syncthreads();
        if (tid == 0) {
            V.match = -1;
            const int n2 = A.part == 1 ? *A.n_big : A.n_list ? *A.n_list : static_cast<int>(2 * A.n_events);
            if (kFuse && fin >= 0 && atomicAdd(A.ev_done + fin, 1) == 1) {
                // this CTA finished the event's second half (the other half's
                // records were released before its count; the fence orders
                // them before the reads of the matching)
                __threadfence();
                const int left = n2 - min(*reinterpret_cast<volatile int*>(A.queue), n2);
                if (!A.defer_match || left >= kDeferRounds * static_cast<int>(gridDim.x)) {
                    V.match = static_cast<int>(fin);  // matched by this CTA, now
                } else {
                    // near the end: left for whichever CTA runs out of seeding items first
                    atomicExch(A.ready + atomicAdd(A.ready_ctr, 1), static_cast<int>(fin) + 1);
                    __threadfence();
                }
                atomicAdd(A.done_ctr, 1);
            }
            if (V.match < 0) {
                const int q = A.order ? (A.part == 2 ? *A.n_big : 0) + atomicAdd(A.queue, 1) : first ? static_cast<int>(blockIdx.x) : n2;
                first = false;
                if (q < n2) {
                    V.item = A.order ? A.order[q] : q;
                } else if (kFuse && A.defer_match) {
                    // no seeding item left, and each is held by a running CTA:
                    // take the next announced event, or stop once every event
                    // is done and none is left for this slot
                    const int n = static_cast<int>(A.n_events);
                    const int m = atomicAdd(A.m_claim, 1);
                    const volatile int* vr = A.ready;
                    int v = 0;
                    bool gave_up = true;
                    const unsigned long long t_wait = global_ns();
                    for (int it = 0; it < kReadySpinsMax; ++it) {
                        // the time limit is checked first: with wait_ns = 0
                        // every wait gives up (the timeout path, for tests)
                        if (global_ns() - t_wait >= A.wait_ns) break;
                        if (m < n) v = vr[m];
                        if (v) {
                            gave_up = false;
                            break;
                        }
                        if (*reinterpret_cast<volatile int*>(A.done_ctr) >= n) {
                            __threadfence();
                            if (m < n) v = vr[m];
                            gave_up = false;
                            break;
                        }
                        __nanosleep(100);
                    }
                    if (gave_up) atomicExch(A.fault, 1);
                    __threadfence();
                    V.match = v - 1;
                    V.item = -1;
                } else {
                    V.item = -1;
                }
            }
        }
        __syncthreads();
        fin = -1;
        if (kFuse && V.match >= 0) {
            const int64_t em = V.match;
            const int c0 = __ldcg(A.item_count + 2 * em), c1 = __ldcg(A.item_count + 2 * em + 1);
            const int64_t r0 = c0 ? __ldcg(A.item_start + 2 * em) : 0;
            const int64_t r1 = c1 ? __ldcg(A.item_start + 2 * em + 1) : 0;
            const int64_t v0 = A.velo_off[em];
            const MatchIO MI{A.velo, A.pool_state, A.pool_n, A.pool_velo, A.pool_chi2, nullptr};
            ull ng = 0, np = 0, nev = 0;
            const int nl = match_event<false>(P, MI, A.velo_smem, smem, v0,
                                              static_cast<int>(A.velo_off[em + 1] - v0), c0 + c1,
                                              [&](int s) { return s < c0 ? r0 + s : r1 + (s - c0); },
                                              &V.cnt, ng, np, nev);
            ng = warp_sum(ng);
            np = warp_sum(np);
            nev = warp_sum(nev);
            if ((tid & 31) == 0) {
                atomicAdd(&V.mctr[0], ng);
                atomicAdd(&V.mctr[1], np);
                atomicAdd(&V.mctr[3], nev);
            }
            if (tid == 0) {
                atomicAdd(&V.mctr[2], ull(nl));
                if (A.n_long) A.n_long[em] = nl;
            }
            continue;
        }
        const int64_t item = V.item;
        if (item < 0) break;
        const int64_t e = item >> 1;
        const int h = static_cast<int>(item & 1);
        if (kFuse) fin = e;
        const int32_t* zo = A.zoff + e * kZoffStride + 12 * h;
        const int64_t cbh = cont_base(A.ev_off, e) + zo[0];
        const int nh = zo[12] - zo[0];
        if (tid <= 12) M.szl[tid] = zo[tid] - zo[0];
        // the half's hits are one contiguous slice: staged in shared memory by
        // one bulk copy of the 16-byte words that hold it (the container's
        // events start 16-byte aligned and are padded to a multiple of 16 bytes)
        const int64_t w0 = cbh & ~int64_t(3);
        const int lead = static_cast<int>(cbh - w0);
        const int nw = (lead + nh + 3) & ~3;
        bool staged = false;
        if (stage_ok && nh > 0 && nw <= A.smem_hits) {
            if (tid == 0) bulk_to_smem(M.sx, A.cx + w0, 4u * unsigned(nw), &V.mbar);
            const bool got = mbar_wait(&V.mbar, mphase, kStagePolls);
            mphase ^= 1u;
            if (__syncthreads_or(!got)) {
                // the copy did not land: global reads from here on, the launch
                // marked faulty (every event then gets ST_TIMEOUT)
                stage_ok = false;
                if (tid == 0 && A.fault) atomicExch(A.fault, 1);
            } else {
                staged = true;
            }
        }
        const float* const Xs_ = M.sx + lead;   // staged hits
        const float* const Xg = A.cx + cbh;     // the container's
        const float* const X = staged ? Xs_ : Xg;

        // ------------------------------------------------------------ hit maps
        // a warp per zone: the bits by atomics (hits of one bin are few), the
        // words' first hits by the hit that begins each
        for (int k = tid; k < 12 * kMapStride; k += T) M.bits[k] = 0u;
        __syncthreads();
        {
            const int lane = tid & 31;
            for (int z = tid >> 5; z < 12; z += T >> 5) {
                const int st = szl[z], n = szl[z + 1] - st;
                uint32_t* bz = M.bits + z * kMapStride;
                uint16_t* fz = M.first + z * kMapWords;
                int wl = -1;  // word of the last hit before this group
                for (int i0 = 0; i0 < n; i0 += 32) {
                    const int i = i0 + lane;
                    const int b = i < n ? map_bin(X[st + i]) : kMapBins;
                    const int w = b >> 5;
                    int wp = __shfl_up_sync(0xffffffffu, w, 1);
                    if (lane == 0) wp = wl;
                    wl = __shfl_sync(0xffffffffu, w, 31);
                    if (i < n) {
                        atomicOr(&bz[w], 1u << (b & 31));
                        for (int q = wp + 1; q <= w; ++q) fz[q] = static_cast<uint16_t>(i);
                        if (i == n - 1) wl = w;
                    }
                }
                // words after the last hit
                const int wn = n > 0 ? __shfl_sync(0xffffffffu, wl, (n - 1) & 31) : -1;
                for (int q = wn + 1 + lane; q < kMapWords; q += 32) fz[q] = static_cast<uint16_t>(n);
            }
        }
        // HLT1: one pass over all iterations, then one clone kill and one UV
        // step.  HLT2-style (seq): one pass per iteration, each with its own
        // clone kill and UV step; the hits of a pass's seeds are marked in
        // S.used before the next pass.  Candidates and kept seeds of all
        // passes are appended to the same lists; the output step takes them
        // all.
        if (seq) {
            for (int i = tid; i < (nh + 31) / 32; i += T) S.used[i] = 0u;
        }
        if (tid == 0) V.nvalid = 0;
        __syncthreads();

        int ncand = 0, nk = 0;
        const int n_pass = seq ? P.n_iter : 1;
        const int nxh = szl[6];
        const bool tbl_in = nxh <= A.tbl_smem;
        bool ok = tbl_in || nxh <= A.tbl_cap;
        for (int ipass = 0; ok && ipass < n_pass; ++ipass) {
            const SeedItem I{h, seq ? ipass : 0, seq ? ipass + 1 : P.n_iter, P.uv_mode == 1};
            // ------------------------------------------------------------ XZ
            const int cb0 = ncand, kb = nk;
            // (the common case on pointers the compiler knows to be in shared memory)
            if (staged)
                ok = xz_search<kSeq>(P, I, M, V, S, Xs_, map, sG, sMask, A.round_hits, ncand, spar);
            else
                ok = xz_search<kSeq>(P, I, M, V, S, Xg, map, sG, sMask, A.round_hits, ncand, spar);
            if (!ok) break;
            // ------------------------------------------------------------ clone kill
            if (tbl_in)
                clone_kill(M, S, reinterpret_cast<ull*>(M.phase), nxh, cb0, ncand, nk, spar);
            else
                clone_kill(M, S, S.tbl, nxh, cb0, ncand, nk, spar);
            if (tid == 0) V.ctr[4] += nk - kb;
            // ------------------------------------------------------------ UV
            // (kept seeds [kb, nk) of this pass; with several passes the keys and
            // stereo positions live in global scratch)
            ull* const skey = reinterpret_cast<ull*>(M.phase + sizeof(uint32_t) * kUvBlock);
            float* const sXs = reinterpret_cast<float*>(skey + A.key_smem);
            if (!seq && staged && nk <= A.key_smem)
                uv_search<kSeq>(P, I, M, V, S, Xs_, map, skey, sXs, kb, nk, spar);
            else
                uv_search<kSeq>(P, I, M, V, S, X, map, !seq && nk <= A.key_smem ? skey : S.key,
                                !seq && nk <= A.key_smem ? sXs : S.xs, kb, nk, spar);
            if (seq && ipass + 1 < n_pass) {
                // hit cleanup: this pass's seeds give their hits to no later pass.
                // Their stereo hits come from the chain store; a pass whose store
                // overflowed cannot be cleaned up and counts as an overflow.
                if (V.nvalid > S.uv_cap) {
                    ok = false;
                    break;
                }
                for (int j = kb + tid; j < nk; j += T) {
                    const ull key = S.key[j];
                    if (key == ~0ull) continue;
                    const Cand* c = S.cand + S.kept[j];
                    const int4 cp = c->p, cq = c->q;
#pragma unroll
                    for (int q = 0; q < 6; ++q) {
                        const int p = cand_pos(cp, cq, q);
                        if (p >= 0) atomicOr(&S.used[p >> 5], 1u << (p & 31));
                    }
                    const UV u = uv_unpack(S.uv[key & 0x1FFFu].v);
#pragma unroll
                    for (int q = 0; q < 6; ++q) {
                        const int p = u.pos[q];
                        if (p >= 0) atomicOr(&S.used[p >> 5], 1u << (p & 31));
                    }
                }
                __syncthreads();
            }
        }  // passes
        if (tid == 0) {
            V.ctr[3] += ncand;
            V.ctr[6] += V.nvalid;  // every valid UV chain of the item's passes
        }
        if (!ok || (seq && V.nvalid > S.uv_cap)) {
            if (tid == 0) {
                if (A.retry) {
                    A.retry[atomicAdd(A.retry_ctr, 1)] = static_cast<int32_t>(item);
                } else {
                    A.status[e] = -3;  // ST_OVERFLOW
                    A.item_count[item] = 0;
                }
            }
            continue;
        }
        ull* const skey = reinterpret_cast<ull*>(M.phase + sizeof(uint32_t) * kUvBlock);
        const bool key_in = !seq && nk <= A.key_smem;
        const ull* ukey = key_in ? skey : S.key;
        const float* Xs = key_in ? reinterpret_cast<float*>(skey + A.key_smem) : S.xs;

        // ------------------------------------------------------------ seeds
        int nseed = 0;
        for (int b = 0; b < nk; b += T) {
            const int j = b + tid;
            const int has = j < nk && ukey[j] != ~0ull;
            nseed += __syncthreads_count(has);
        }
        if (tid == 0) {
            ull st = ~0ull;
            if (nseed > 0) {
                st = atomicAdd(A.pool_ctr, ull(nseed));
                if (st + nseed > ull(A.pool_cap)) {
                    A.status[e] = -3;
                    st = ~0ull;
                }
            }
            V.start = st;
            A.item_start[item] = st == ~0ull ? 0 : static_cast<int32_t>(st);
            A.item_count[item] = st == ~0ull ? 0 : nseed;
            V.ctr[7] += st == ~0ull ? 0 : nseed;
        }
        __syncthreads();
        if (V.start == ~0ull) continue;
        int wbase = 0;
        for (int b = 0; b < nk; b += T) {
            const int j = b + tid;
            const int has = j < nk && ukey[j] != ~0ull;
            int tot;
            const int o = block_exscan1(has, M.tmp, spar, tot);
            if (has) {
                const int64_t r = int64_t(V.start) + wbase + o;
                const ull key = ukey[j];
                const int sidx = static_cast<int>(key & 0x1FFFu);
                const Cand* c = S.cand + S.kept[j];
                const XzModel m = xz_model(c);
                const int4 cp = c->p, cq = c->q;
                const float* th = m.th;
                const float* dth = m.dth;
                UV u;
                if (sidx != kUvNotStored) {
                    u = uv_unpack(S.uv[sidx].v);
                    const float4 f = S.uv[sidx].f;
                    u.chi2 = f.x;
                    u.beta = f.y;
                    u.wm = f.z;
                    u.zm = f.w;
                } else {
                    if constexpr (kOut)
                        u = uv_redo_out(P, X, szl, map, used, Xs + 6 * j, c, h, S.hcl + 8 * j, key);
                    else
                        u = uv_redo_in(P, X, szl, map, used, Xs + 6 * j, c, h, S.hcl + 8 * j, key);
                }
                // the record goes out as 16-byte stores (pool rows are 48 /
                // 32 / 16 bytes long and the pool is 256-byte aligned)
                // layers 0..11 are x u v x | x u v x | x u v x: x slot q and
                // stereo slot q in layer order
                auto hx = [&](int q) {
                    const int p = cand_pos(cp, cq, q);
                    return p >= 0 ? A.corig[cbh + p] : -1;
                };
                auto hu = [&](int q) { return u.pos[q] >= 0 ? A.corig[cbh + u.pos[q]] : -1; };
                int4* ho = reinterpret_cast<int4*>(A.pool_hits + r * 12);
                ho[0] = make_int4(hx(0), hu(0), hu(1), hx(1));
                ho[1] = make_int4(hx(2), hu(2), hu(3), hx(3));
                ho[2] = make_int4(hx(4), hu(4), hu(5), hx(5));
                const float a = th[0] + dth[0], bb = th[1] + dth[1], cc = th[2] + dth[2];
                // y(z) = tyr z + wm + beta (z - zc - zm)
                const float ty = u.tyr + u.beta;
                const float y0 = fmaf(-u.beta, P.zc_uv + u.zm, u.wm);
                const float yS = fmaf(u.tyr, P.zS, fmaf(u.beta, (P.zS - P.zc_uv) - u.zm, u.wm));
                float4* po = reinterpret_cast<float4*>(A.pool_params + r * 8);
                po[0] = make_float4(a, bb, cc, c->th.w);
                po[1] = make_float4(y0, ty, u.chi2, 0.f);
                reinterpret_cast<float4*>(A.pool_state)[r] =
                    make_float4(fmaf(th[2], P.fS, fmaf(th[1], P.zbS, th[0])) +
                                    fmaf(dth[2], P.fS, fmaf(dth[1], P.zbS, dth[0])),
                                yS, fmaf(cc, P.dfS, bb), ty);
                const unsigned short nn = static_cast<unsigned short>((cq.z & 0xFF) | ((u.n & 0xFF) << 8));
                reinterpret_cast<unsigned short*>(A.pool_n)[r] = nn;
            }
            wbase += tot;
        }
    }
    __syncthreads();
    // a copy given up on may still land: wait for it (bounded) before the
    // CTA's shared memory goes away
    if (!stage_ok) mbar_wait(&V.mbar, mphase ^ 1u, kStagePolls);
    if (tid < 8 && V.ctr[tid]) atomicAdd(A.counters + C_PAIRS + tid, V.ctr[tid]);
    if (kFuse && tid < 3 && V.mctr[tid]) atomicAdd(A.counters + C_MATCH_PAIRS + tid, V.mctr[tid]);
    if (kFuse && tid == 3 && V.mctr[3]) atomicAdd(A.counters + C_MATCH_EVAL, V.mctr[3]);
}

template <int kT, int kR>
SeedKernel seed_kernel_of(bool seq, bool fused) {
    return fused ? k_seed<kT, kR, false, true> : seq ? k_seed<kT, kR, true, false> : k_seed<kT, kR, false, false>;
}

}  // namespace st

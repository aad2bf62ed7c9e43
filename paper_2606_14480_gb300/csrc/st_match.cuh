// st_match.cuh -- VELO-SciFi matching of one event (Section 4), shared by
// k_match and the seeding kernel's fused matching.
#pragma once

#include <cfloat>

#include "st_common.cuh"

namespace st {

// What the matching of one event reads and writes.
struct MatchIO {
    const float* velo;         // x, y, tx, ty at z_velo
    const float* seed_state;   // x, y, tx, ty at z_state, per row
    const int8_t* seed_n;      // (nx, nuv) per row
    int32_t* velo_idx;         // per row
    float* chi2;               // per row
    float* ghost_prob;         // per row (final selection)
};
// Lanes that share a seed: as many as keep seeds x lanes within kMatchFill
// times the CTA's threads.  500 events of 272 seeds and 400 segments: 41 us
// with a thread per seed (two passes, the second nearly empty), 34 us with up
// to 4 x 256 lanes' worth, 30 us with the segments laid out as below.
constexpr int kMatchLanes = 8;
constexpr int kMatchFill = 4;
constexpr int kTyBins = 64;
constexpr float kTyRange = 0.32f;  // buckets of 0.01 over [-0.32, 0.32); outside values go to the end buckets

inline size_t match_smem_size(int velo_smem) {
    return (2 * sizeof(float4) + sizeof(int)) * size_t(velo_smem) + sizeof(int) * (2 * kTyBins + 8);
}

__device__ __forceinline__ int ty_bin(float ty) {
    const int b = __float2int_rd((ty + kTyRange) * (kTyBins / (2.f * kTyRange)));
    return min(max(b, 0), kTyBins - 1);  // NaN maps to bucket 0 and never passes the cuts
}

// One (VELO, seed) pair of Section 4: preselection, then chi2_match; updates
// the best (chi2, VELO index).  Position differences are formed from
// float-float extrapolations to z = A_x (x) and z = z_match_y (y).  The first
// half of the segment decides most pairs.
struct VeloHalf {
    float tx, ty, yh, yl;
};
struct VeloRest {
    float xh, xl, it;
    int v;
};
static_assert(sizeof(VeloHalf) == sizeof(float4) && sizeof(VeloRest) == sizeof(float4), "");
__device__ __forceinline__ int match_pair(const DevParams& P, const VeloHalf& a, const VeloRest* rest, float xh,
                                          float xl, float yh, float yl, float txS, float tyS, float dzx,
                                          float& best, int& bv) {
    const float dtx = a.tx - txS, dty = a.ty - tyS;
    if (!(fabsf(dty) < P.cut_ty) || !(fabsf(dtx) < P.cut_tx)) return 0;
    const float dy = (a.yh - yh) + (a.yl - yl);
    if (!(fabsf(dy) < P.cut_y)) return 0;
    const float4 q = *reinterpret_cast<const float4*>(rest);
    const float dz = fmaf(P.Bx, fabsf(dtx), fmaf(P.Cx, dtx * dtx, fmaf(P.Ex * a.tx, a.tx, dzx)));
    const float dx = fmaf(dz, dtx, (q.x - xh) + (q.y - xl));
    if (!(fabsf(dx) < P.cut_x)) return 0;
    const float tolx = fmaf(P.tolx_b, dtx * dtx, P.tolx_a);
    const float c2 = dx * dx / tolx + dy * dy * q.z + dtx * dtx * P.inv_toltx + dty * dty * P.inv_tolty;
    const int vg = __float_as_int(q.w);
    if (c2 < P.chi2m_max && (c2 < best || (c2 == best && vg < bv))) {
        best = c2;
        bv = vg;
    }
    return 1;
}

// The eight inputs of the ghost network (Section 4.4) for one pair: z_match_x,
// dx, dy, dtx, dty (formed like match_pair's), slot 5 left for chi2_match,
// the VELO segment's pseudorapidity asinh(1/|slope|) (= -ln tan(theta/2)),
// slot 7 left for the seed's hit count.
static __device__ void pair_features(const DevParams& P, const float* vs, const float* ss, float f[8]) {
    const float x = vs[0], y = vs[1], tx = vs[2], ty = vs[3];
    float p, pe, s, se;
    two_prod(P.dAV_hi, tx, p, pe);
    two_sum(x, p, s, se);
    const float vxh = s, vxl = se + fmaf(P.dAV_lo, tx, pe);
    two_prod(P.dMV_hi, ty, p, pe);
    two_sum(y, p, s, se);
    const float vyh = s, vyl = se + fmaf(P.dMV_lo, ty, pe);
    const float xS = ss[0], yS = ss[1], txS = ss[2], tyS = ss[3];
    float xh, xl, yh, yl;
    two_prod(P.dAS_hi, txS, p, pe);
    two_sum(xS, p, xh, xl);
    xl += fmaf(P.dAS_lo, txS, pe);
    two_prod(P.dMS_hi, tyS, p, pe);
    two_sum(yS, p, yh, yl);
    yl += fmaf(P.dMS_lo, tyS, pe);
    const float dtx = tx - txS, dty = ty - tyS;
    const float dz = fmaf(P.Bx, fabsf(dtx), fmaf(P.Cx, dtx * dtx, fmaf(P.Ex * tx, tx, P.Dx * fabsf(xS))));
    f[0] = P.A_hi + (P.A_lo + dz);
    f[1] = fmaf(dz, dtx, (vxh - xh) + (vxl - xl));
    f[2] = (vyh - yh) + (vyl - yl);
    f[3] = dtx;
    f[4] = dty;
    f[6] = asinhf(1.f / fmaxf(sqrtf(fmaf(tx, tx, ty * ty)), 1e-6f));
}

// The ghost network: standardised inputs, 32 ReLU nodes, sigmoid output.
// Every lane reads the same weight at the same time (uniform constant reads).
static __device__ float ghost_nn(const DevParams& P, const float f[8]) {
    float in[8];
#pragma unroll
    for (int i = 0; i < 8; ++i) in[i] = (f[i] - P.nn[i]) * P.nn[8 + i];
    float z = P.nn[336];
#pragma unroll 4
    for (int k = 0; k < 32; ++k) {
        float a = P.nn[272 + k];
#pragma unroll
        for (int i = 0; i < 8; ++i) a = fmaf(P.nn[16 + 8 * k + i], in[i], a);
        if (a > 0.f) z = fmaf(P.nn[304 + k], a, z);
    }
    return 1.f / (1.f + expf(-z));
}

// Matching of one event (Section 4): the event's VELO segments are staged in
// shared memory (msm, match_smem_bytes(VS) bytes), VS at a time, with their
// float-float extrapolations and laid out by ty bucket, so a seed only visits
// the buckets its |dty| cut can reach (every other pair fails that cut).  A few
// lanes share a seed, each taking every n-th segment of its buckets: an event
// has fewer seeds than the CTA threads, and the time is the longest lane's.
// What bounds it is the latency of that chain: a pair costs one 16-byte read
// until it passes the first cuts, a lane's next seed is fetched while it works
// on one, and pairs are counted where they are found.  1000 Run-3-like events
// with the final selection: 34.3 us before these, 31.7 us with.
// Seed s (0 .. ns-1, in the event's canonical seed order) reads its state and
// hit counts and writes its pair at index row(s) of M's arrays.  Returns the
// event's Long-track count; n_grid / n_presel accumulate this thread's pair
// counts.
template <bool kFinal, class Row>
__device__ int match_event(const DevParams& P, const MatchIO& M, int VS, unsigned char* msm, int64_t v0, int nv,
                           int ns, Row row, int* s_cnt, ull& n_grid, ull& n_presel, ull& n_eval) {
    const int T = blockDim.x, tid = threadIdx.x;
    VeloHalf* const va = reinterpret_cast<VeloHalf*>(msm);  // [VS] the chunk's segments grouped by ty bucket
    VeloRest* const vb = reinterpret_cast<VeloRest*>(va + VS);
    int* const tag = reinterpret_cast<int*>(vb + VS);       // [VS] a segment's bucket and place in it
    int* const bcnt = tag + VS;                             // [kTyBins]
    int* const boff = bcnt + kTyBins;                       // [kTyBins + 1]
    const bool vec = (reinterpret_cast<uintptr_t>(M.velo) & 15u) == 0;
    const float* const velo = M.velo + v0 * 4;
    if (tid == 0) *s_cnt = 0;
    int G = 1;
    while (G < kMatchLanes && 2 * G * ns <= kMatchFill * T) G *= 2;
    const int lane = tid & 31, sub = lane & (G - 1), step = (T >> 5) * (32 / G);
    // the state of the lane's next seed, fetched ahead (past L1: in the fused
    // kernel other CTAs wrote the rows during this launch)
    float xS = 0.f, yS = 0.f, txS = 0.f, tyS = 0.f;
    auto fetch = [&](int s) {
        if (s >= ns) return;
        const float* st = M.seed_state + row(s) * 4;
        xS = __ldcg(st);
        yS = __ldcg(st + 1);
        txS = __ldcg(st + 2);
        tyS = __ldcg(st + 3);
    };
    const int first = (tid >> 5) * (32 / G) + lane / G;
    const bool plain = !P.velo_unique && !(kFinal && P.final_sel);  // no step drops a pair later
    int nl = 0;
    for (int vc = 0; vc < nv; vc += VS) {
        const int m = min(VS, nv - vc);
        const bool last = vc + VS >= nv;
        for (int k = tid; k < kTyBins; k += T) bcnt[k] = 0;
        fetch(first);
        __syncthreads();
        for (int v = tid; v < m; v += T) {
            const int b = ty_bin(velo[4 * (vc + v) + 3]);
            tag[v] = atomicAdd(&bcnt[b], 1) << 8 | b;
        }
        __syncthreads();
        if (tid < 32) {  // exclusive scan of the bucket counts by one warp
            const int c0 = bcnt[2 * tid], c1 = bcnt[2 * tid + 1];
            int x = c0 + c1;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int y = __shfl_up_sync(0xffffffffu, x, o);
                if (tid >= o) x += y;
            }
            const int ex = x - c0 - c1;
            boff[2 * tid] = ex;
            boff[2 * tid + 1] = ex + c0;
            if (tid == 31) boff[kTyBins] = x;
        }
        __syncthreads();
        for (int v = tid; v < m; v += T) {
            float x, y, tx, ty;
            const float* st = velo + 4 * (vc + v);
            if (vec) {
                const float4 q = *reinterpret_cast<const float4*>(st);
                x = q.x, y = q.y, tx = q.z, ty = q.w;
            } else {
                x = st[0], y = st[1], tx = st[2], ty = st[3];
            }
            const int t = tag[v], k = boff[t & 255] + (t >> 8);
            float p, pe, s;
            VeloRest r;
            two_prod(P.dAV_hi, tx, p, pe);
            two_sum(x, p, r.xh, s);
            r.xl = s + fmaf(P.dAV_lo, tx, pe);
            r.it = 1.f / fmaf(P.toly_b, fmaf(tx, tx, ty * ty), P.toly_a);
            r.v = vc + v;
            VeloHalf a;
            two_prod(P.dMV_hi, ty, p, pe);
            two_sum(y, p, a.yh, s);
            a.yl = s + fmaf(P.dMV_lo, ty, pe);
            a.tx = tx;
            a.ty = ty;
            *reinterpret_cast<float4*>(va + k) = make_float4(a.tx, a.ty, a.yh, a.yl);
            *reinterpret_cast<float4*>(vb + k) = make_float4(r.xh, r.xl, r.it, __int_as_float(r.v));
        }
        __syncthreads();
        for (int s0 = (tid >> 5) * (32 / G); s0 < ns; s0 += step) {  // uniform over the warp
            const int s = s0 + lane / G;
            float best = FLT_MAX;
            int bv = 0x7fffffff, npre = 0;
            if (s < ns) {
                float p, pe, xh, xl, yh, yl;
                two_prod(P.dAS_hi, txS, p, pe);
                two_sum(xS, p, xh, xl);
                xl += fmaf(P.dAS_lo, txS, pe);
                two_prod(P.dMS_hi, tyS, p, pe);
                two_sum(yS, p, yh, yl);
                yl += fmaf(P.dMS_lo, tyS, pe);
                const float dzx = P.Dx * fabsf(xS), txs = txS, tys = tyS;
                fetch(s + step);
                if (vc > 0 && sub == 0) {
                    const int pv = M.velo_idx[row(s)];
                    if (pv >= 0) {
                        bv = pv;
                        best = M.chi2[row(s)];
                    }
                }
                // buckets that can hold |ty - tyS| < cut_ty (slightly widened;
                // the exact cut is applied per pair)
                const float w = P.cut_ty + 1e-6f * (fabsf(tys) + P.cut_ty);
                const int k0 = boff[ty_bin(tys - w)], k1 = boff[ty_bin(tys + w) + 1];
                if (sub == 0) {
                    n_eval += k1 - k0;
                    n_grid += m;
                }
                for (int k = k0 + sub; k < k1; k += G) {
                    const float4 q = *reinterpret_cast<const float4*>(va + k);
                    npre += match_pair(P, VeloHalf{q.x, q.y, q.z, q.w}, vb + k, xh, xl, yh, yl, txs, tys, dzx, best,
                                       bv);
                }
            }
            n_presel += npre;
            for (int o = 1; o < G; o <<= 1) {  // the lowest chi2 of the seed's lanes, ties to the lower index
                const float c = __shfl_xor_sync(0xffffffffu, best, o);
                const int v = __shfl_xor_sync(0xffffffffu, bv, o);
                if (c < best || (c == best && v < bv)) {
                    best = c;
                    bv = v;
                }
            }
            if (s < ns && sub == 0) {
                const bool found = best < FLT_MAX;
                M.velo_idx[row(s)] = found ? bv : -1;
                M.chi2[row(s)] = found ? best : 0.f;
                nl += last && found;
            }
        }
        __syncthreads();
    }
    if (nv == 0) {
        for (int s = tid; s < ns; s += T) {
            M.velo_idx[row(s)] = -1;
            M.chi2[row(s)] = 0.f;
        }
    }
    if (!plain) {
        nl = 0;
        __syncthreads();
    }
    if (P.velo_unique) {
        // a VELO segment keeps its best seed (lowest chi2, then lower seed
        // index); losers are marked -2 - v so that concurrent readers still
        // see which segment they held
        for (int s = tid; s < ns; s += T) {
            const int v = M.velo_idx[row(s)];
            if (v < 0) continue;
            const float c = M.chi2[row(s)];
            for (int t = 0; t < ns; ++t) {
                if (t == s) continue;
                int vt = M.velo_idx[row(t)];
                if (vt <= -2) vt = -2 - vt;
                if (vt != v) continue;
                const float ct = M.chi2[row(t)];
                if (ct < c || (ct == c && t < s)) {
                    M.velo_idx[row(s)] = -2 - v;
                    break;
                }
            }
        }
        __syncthreads();
        for (int s = tid; s < ns; s += T) {
            if (M.velo_idx[row(s)] <= -2) {
                M.velo_idx[row(s)] = -1;
                M.chi2[row(s)] = 0.f;
            }
        }
        __syncthreads();
    }
    if (kFinal && P.final_sel) {
        // Section 4.4: ghost probability of each best pair and the cut, then
        // clones: a kept pair whose VELO segment another kept pair holds with a
        // ghost probability lower by at least clone_margin (one pair per seed,
        // so no two pairs share a seed).  With clone_margin > 0 that is p -
        // (lowest p on the segment) >= clone_margin; the lowest p per segment
        // is an atomicMin of the probabilities' bits (non-negative floats order
        // as unsigned).
        const bool small = nv <= VS;
        unsigned* const vmin = reinterpret_cast<unsigned*>(tag);  // [VS] lowest ghost probability per segment
        if (small) {
            for (int v = tid; v < nv; v += T) vmin[v] = 0x7f800000u;
            __syncthreads();
        }
        for (int s = tid; s < ns; s += T) {
            const int v = M.velo_idx[row(s)];
            float p = 1.f;
            if (v >= 0) {
                float f[8];
                pair_features(P, M.velo + (v0 + v) * 4, M.seed_state + row(s) * 4, f);
                f[5] = M.chi2[row(s)];
                f[7] = static_cast<float>(M.seed_n[2 * row(s)] + M.seed_n[2 * row(s) + 1]);
                p = ghost_nn(P, f);
                if (!(p < P.ghost_max)) {
                    M.velo_idx[row(s)] = -1;
                    M.chi2[row(s)] = 0.f;
                } else if (small) {
                    atomicMin(&vmin[v], __float_as_uint(p));
                }
            }
            M.ghost_prob[row(s)] = p;
        }
        __syncthreads();
        if (small) {
            // (each thread's own rows)
            for (int s = tid; s < ns; s += T) {
                const int v = M.velo_idx[row(s)];
                const bool clone = v >= 0 && M.ghost_prob[row(s)] - __uint_as_float(vmin[v]) >= P.clone_margin;
                if (clone) {
                    M.velo_idx[row(s)] = -1;
                    M.chi2[row(s)] = 0.f;
                }
                nl += v >= 0 && !clone;
            }
        } else {
            // clones are marked -2 - v, so that concurrent readers still see
            // which segment they held
            for (int s = tid; s < ns; s += T) {
                const int v = M.velo_idx[row(s)];
                if (v < 0) continue;
                const float p = M.ghost_prob[row(s)];
                for (int t = 0; t < ns; ++t) {
                    if (t == s) continue;
                    int vt = M.velo_idx[row(t)];
                    if (vt <= -2) vt = -2 - vt;
                    if (vt == v && p - M.ghost_prob[row(t)] >= P.clone_margin) {
                        M.velo_idx[row(s)] = -2 - v;
                        break;
                    }
                }
            }
            __syncthreads();
            for (int s = tid; s < ns; s += T) {
                const int v = M.velo_idx[row(s)];
                if (v <= -2) {
                    M.velo_idx[row(s)] = -1;
                    M.chi2[row(s)] = 0.f;
                }
                nl += v >= 0;
            }
        }
    } else if (!plain) {
        for (int s = tid; s < ns; s += T) nl += M.velo_idx[row(s)] >= 0;
    }
    nl = warp_sum(nl);
    if ((tid & 31) == 0 && nl) atomicAdd(s_cnt, nl);
    __syncthreads();
    return *s_cnt;
}

}  // namespace st

// sf_knn.cu -- exact k-nearest-neighbour bandwidths h_j (the kNN bandwidth
// rule: h_j = distance from point j to its k-th nearest other point).
//
// Exactness contract: the neighbour set equals the one a brute-force FP64
// evaluation gives with d2 = ((dx*dx)+(dy*dy))+(dz*dz), dx = (double)x_i -
// (double)x_j, ties broken by the smaller original index; h = (float)sqrt(d2_k).
//
// Two kernels, both of persistent warps that take the next leaf of 32 Morton-consecutive
// query points from an atomic counter (no warp waits for another). k_knn_sel (below)
// computes the bandwidths; k_knn, which follows, takes the leaves that it leaves over
// and every call that asks for the neighbours' ids:
//  1. radius bound: per lane, the k-th smallest FP32 d2 among the points of
//     nearby leaves in sorted order (a bin edge above it, from 32-bin
//     histograms of 5 then 13 leaves at k = 64) -- an upper bound of the true
//     k-th distance;
//  2. candidates: the index walk keeps the leaves within that radius of at
//     least one lane's point, and records them in a per-warp leaf list in
//     global memory; their points inside the warp's envelope box are the
//     candidates (every pass reloads them leaf by leaf);
//  3. histogram while collecting: per lane, 32 bins of FP32 d2 over [0, T];
//     the bin holding the k-th is found;
//  4. band pass: points clearly below the bin are in; the ones whose FP32 d2
//     lies in the bin (widened by a relative 2e-6) are re-evaluated in FP64 (no
//     FMA contraction) into a per-lane buffer of 64 in global memory and ranked
//     by (d2, original index) -- one pass resolves almost every lane; recorded
//     leaves whose box lies wholly below or above every lane's band are counted
//     from their envelope masks instead of being reloaded. If a band
//     overflows its buffer the bin is split again (the band pass has already
//     binned the bracket for that round); at FP32 resolution (exact duplicates)
//     the remaining members are extracted one by one.
// FP32 d2 carries a relative error below 5 * 2^-24, so the 2e-6 margins make
// every in/out decision outside the band exact. If a warp's accepted leaves
// exceed its list, its passes walk the index again instead (same result).
#include <cmath>

#include "sf_internal.cuh"

namespace sf {

constexpr int kKnnWarps = 4;
constexpr int kNB = 32;        // histogram bins per lane
constexpr int kBand = 64;      // band buffer per lane (global memory, interleaved by lane)
constexpr int kCand = 64;      // candidate leaves per walk batch
constexpr int kLeafList = 4096;  // accepted leaves recorded per warp (global)
constexpr int kKStack = 32 * kMaxLevels;
constexpr float kDelta = 2.0e-6f;

struct KnnWarpSmem {
    int stack[kKStack];
    int cand[kCand];
    float4 blo[32], bhi[32];   // child boxes under test
    float4 pts[kLeaf];         // staged candidates (x, y, z, original id bits)
    uint32_t hist[kNB][32];
    unsigned left;             // lanes left to a finer scale
};

struct KnnArgs {
    TreeView tv;
    const uint32_t *perm;
    int k;
    float scale;              // power of two applied to every coordinate (first try)
    float *h_sorted;          // out: h per sorted point
    uint32_t *nbr_orig;       // out (nullable): [n][k] by original index
    int *leaf_list;           // [slots][kLeafList] accepted leaves of the current query leaf
    uint32_t *leaf_mask;      // [slots][kLeafList] their points inside the warp envelope
    double *band_d;           // [slots][kBand][32] band members' FP64 d2
    uint32_t *band_i;         // [slots][kBand][32] band members' original ids
    unsigned int *next_leaf;  // work counter (zeroed before launch)
    unsigned long long *work; // nullable: [0] candidates staged (all passes), [1] query leaves
    const unsigned int *retry;    // nullable: the query leaves to process (*retry_n of them)
    const unsigned int *retry_n;
};

// Coordinates are scaled by a power of two on load, first to an extent of about 2^30, then
// for the lanes whose k-th point lies within 2^-30 of their bracket's radius (a point far
// out widens it), or whose bracket is below 1, to 2^30 times that, and so on: the k-th
// FP32 d2 neither overflows nor underflows. Scaling up is exact; scaling down loses bits below
// 2^-149, which FP64 distances of 2^-30 and more do not see.
__device__ __forceinline__ float4 ld_scaled(const float4 *p, float scale) {
    float4 v = __ldg(p);
    v.x *= scale;
    v.y *= scale;
    v.z *= scale;
    return v;
}

__device__ __forceinline__ float d2_f32(float4 a, float4 b) {
    const float dx = a.x - b.x, dy = a.y - b.y, dz = a.z - b.z;
    return fmaf(dz, dz, fmaf(dy, dy, dx * dx));
}

__device__ __forceinline__ double d2_f64(float4 a, float4 b) {
    const double dx = __dsub_rn((double)a.x, (double)b.x);
    const double dy = __dsub_rn((double)a.y, (double)b.y);
    const double dz = __dsub_rn((double)a.z, (double)b.z);
    return __dadd_rn(__dadd_rn(__dmul_rn(dx, dx), __dmul_rn(dy, dy)), __dmul_rn(dz, dz));
}

__device__ __forceinline__ bool key_less(double da, uint32_t ia, double db, uint32_t ib) {
    return da < db || (da == db && ia < ib);
}

// Per-warp candidate search: every lane holds one query point and the squared
// radius r2 of its ball (negative: the lane takes no part). COUNT: the work
// accounting variant (sf_knn_work_counts).
template <bool COUNT>
struct KnnWarp {
    const TreeView &tv;
    const uint32_t *perm;
    float scale;           // see ld_scaled
    KnnWarpSmem &S;
    int *leaf_list;        // this warp's recorded leaves
    uint32_t *leaf_mask;   // and, per leaf, its points inside the envelope
    float4 q;
    float r2;
    float env_lo[3], env_hi[3];  // warp envelope of all balls
    int nlist;
    bool overflow;
    unsigned long long ncand = 0;  // COUNT only: candidates staged over all passes

    __device__ KnnWarp(const TreeView &t, const uint32_t *p, float sc, KnnWarpSmem &s, int *c, uint32_t *cm)
        : tv(t), perm(p), scale(sc), S(s), leaf_list(c), leaf_mask(cm) {}

    // Mask of the children (lane c holds child c at level cl) within the ball
    // of at least one lane. Conservative: relative slack 1e-5.
    __device__ unsigned accept(int cl, int64_t c, bool valid) {
        const int lane = threadIdx.x & 31;
        bool pre = false;
        float4 lo = make_float4(0.f, 0.f, 0.f, 0.f), hi = lo;
        if (valid) {
            lo = ld_scaled(&tv.nlo[tv.off[cl] + c], scale);
            hi = ld_scaled(&tv.nhi[tv.off[cl] + c], scale);
            pre = lo.x <= env_hi[0] && hi.x >= env_lo[0] && lo.y <= env_hi[1] && hi.y >= env_lo[1] &&
                  lo.z <= env_hi[2] && hi.z >= env_lo[2];
        }
        unsigned m = __ballot_sync(0xffffffffu, pre);
        if (pre) {
            S.blo[lane] = lo;
            S.bhi[lane] = hi;
        }
        __syncwarp();
        unsigned acc = 0;
        const float lim = r2 * (1.0f + 1.0e-5f);
        while (m) {
            const int j = __ffs(m) - 1;
            m &= m - 1;
            const float4 bl = S.blo[j], bh = S.bhi[j];
            const float gx = fmaxf(fmaxf(bl.x - q.x, q.x - bh.x), 0.f);
            const float gy = fmaxf(fmaxf(bl.y - q.y, q.y - bh.y), 0.f);
            const float gz = fmaxf(fmaxf(bl.z - q.z, q.z - bh.z), 0.f);
            const float d2 = fmaf(gz, gz, fmaf(gy, gy, gx * gx));
            if (__any_sync(0xffffffffu, r2 >= 0.f && d2 <= lim)) acc |= 1u << j;
        }
        __syncwarp();
        return acc;
    }

    // Resumable walk: appends accepted leaves to S.cand until fewer than 32
    // slots remain or the stack is empty.
    __device__ int walk(int &sp) {
        const int lane = threadIdx.x & 31;
        const unsigned lt = (1u << lane) - 1u;
        int nout = 0;
        while (sp > 0 && nout <= kCand - 32) {
            const int e = S.stack[sp - 1];
            __syncwarp();
            sp -= 1;
            const int cl = (e >> 27) - 1;
            const int64_t c = (int64_t)(e & ((1 << 27) - 1)) * kFanout + lane;
            const unsigned m = accept(cl, c, c < tv.cnt[cl]);
            const bool ok = (m >> lane) & 1u;
            const int r = __popc(m & lt), kk = __popc(m);
            if (cl == 0) {
                if (ok) S.cand[nout + r] = (int)c;
                nout += kk;
            } else {
                if (ok) S.stack[sp + (kk - 1 - r)] = (cl << 27) | (int)c;
                sp += kk;
            }
            __syncwarp();
        }
        return nout;
    }

    __device__ int start(int &sp) {
        const int top = tv.nlevels - 1;
        if (top == 0) {
            sp = 0;
            if ((threadIdx.x & 31) == 0) S.cand[0] = 0;
            __syncwarp();
            return 1;
        }
        if ((threadIdx.x & 31) == 0) S.stack[0] = top << 27;
        __syncwarp();
        sp = 1;
        return 0;
    }

    // Stage the envelope-filtered points of the leaves S.cand[0..nl), one leaf
    // at a time (the next leaf's points load while the current one is used):
    // chunk(n) is called with S.pts[0..n) staged (x, y, z, original id bits).
    template <typename Chunk>
    __device__ __forceinline__ void visit(int nl, Chunk chunk, int record = -1) {
        const int lane = threadIdx.x & 31;
        float4 pn = make_float4(0.f, 0.f, 0.f, 0.f);
        uint32_t idn = 0;
        auto load = [&](int li) {
            const int64_t j = (int64_t)S.cand[li] * kLeaf + lane;
            if (j < tv.n) {
                pn = ld_scaled(&tv.pos[j], scale);
                idn = __ldg(&perm[j]);
            }
        };
        if (nl > 0) load(0);
        for (int li = 0; li < nl; ++li) {
            const int64_t j = (int64_t)S.cand[li] * kLeaf + lane;
            float4 p = pn;
            p.w = __uint_as_float(idn);
            if (li + 1 < nl) load(li + 1);
            const bool in = j < tv.n && p.x >= env_lo[0] && p.x <= env_hi[0] && p.y >= env_lo[1] &&
                            p.y <= env_hi[1] && p.z >= env_lo[2] && p.z <= env_hi[2];
            const unsigned m = __ballot_sync(0xffffffffu, in);
            if (COUNT) ncand += __popc(m);
            if (in) S.pts[__popc(m & ((1u << lane) - 1u))] = p;
            if (record >= 0 && lane == 0 && record + li < kLeafList) leaf_mask[record + li] = m;
            __syncwarp();
            chunk(__popc(m));
            __syncwarp();
        }
    }

    // Every accepted leaf by walking the index.
    template <typename Chunk>
    __device__ __forceinline__ void walk_points(Chunk chunk) {
        int sp;
        int nl = start(sp);
        while (true) {
            if (nl == 0) {
                if (sp == 0) break;
                nl = walk(sp);
                if (nl == 0) break;
            }
            visit(nl, chunk);
            nl = 0;
        }
    }

    // Walk once, recording the accepted leaves in the warp's global leaf list;
    // fn(n) sees each staged chunk S.pts[0..n) on the way (all lanes together).
    template <typename Fn>
    __device__ __forceinline__ void collect(Fn fn) {
        const int lane = threadIdx.x & 31;
        nlist = 0;
        overflow = false;
        int sp;
        int nl = start(sp);
        while (true) {
            if (nl == 0) {
                if (sp == 0) break;
                nl = walk(sp);
                if (nl == 0) break;
            }
            for (int i = lane; i < nl; i += 32)
                if (nlist + i < kLeafList) leaf_list[nlist + i] = S.cand[i];
            if (nlist + nl > kLeafList) overflow = true;
            visit(nl, fn, nlist);
            nlist += nl;
            nl = 0;
        }
        __syncwarp();
    }

    // fn(point with id bits in w) for every candidate, all lanes together: the
    // recorded leaves again (or a fresh walk if the list overflowed).
    template <typename Fn>
    __device__ __forceinline__ void each(Fn fn) {
        const int lane = threadIdx.x & 31;
        auto per_chunk = [&](int n) {
            int t = 0;
            for (; t + 2 <= n; t += 2) {
                const float4 a = S.pts[t], b = S.pts[t + 1];
                fn(a);
                fn(b);
            }
            if (t < n) fn(S.pts[t]);
        };
        if (!overflow) {
            for (int base = 0; base < nlist; base += kCand) {
                const int nb = min(kCand, nlist - base);
                __syncwarp();
                for (int i = lane; i < nb; i += 32) S.cand[i] = leaf_list[base + i];
                __syncwarp();
                visit(nb, per_chunk);
            }
            return;
        }
        walk_points(per_chunk);
    }

    // As each(), but a recorded leaf is loaded only if some lane needs its points:
    // cls(lo, hi) classifies the leaf box for this lane (0: visit, 1: every point
    // counts as below, 2: nothing to do) and below(n) adds the n envelope points of
    // a leaf classified 1 (the lane's own point excluded).
    template <typename Fn, typename Cls, typename Below>
    __device__ __forceinline__ void each_pruned(Fn fn, Cls cls, Below below, int64_t self_leaf) {
        const int lane = threadIdx.x & 31;
        if (overflow) {
            each(fn);
            return;
        }
        auto per_chunk = [&](int n) {
            for (int t = 0; t < n; ++t) fn(S.pts[t]);
        };
        for (int base = 0; base < nlist; base += 32) {
            const int nb = min(32, nlist - base);
            const int lidx = lane < nb ? leaf_list[base + lane] : 0;
            const uint32_t lmask = lane < nb ? leaf_mask[base + lane] : 0u;
            for (int t = 0; t < nb; ++t) {
                const int L = __shfl_sync(0xffffffffu, lidx, t);
                const uint32_t m = __shfl_sync(0xffffffffu, lmask, t);
                const float4 lo = ld_scaled(&tv.nlo[tv.off[0] + L], scale), hi = ld_scaled(&tv.nhi[tv.off[0] + L], scale);
                const int c = cls(lo, hi);
                if (!__any_sync(0xffffffffu, c == 0)) {
                    if (c == 1) below(__popc(m) - ((L == self_leaf && ((m >> lane) & 1u)) ? 1 : 0));
                    continue;
                }
                __syncwarp();
                if (lane == 0) S.cand[0] = L;
                __syncwarp();
                visit(1, per_chunk);
            }
        }
    }
};

// The leaf's queries at the first scale, or (FINER) those of `lanes` at finer_scale; S.left gets
// the lanes left to a finer one.
template <bool COUNT, bool FINER>
__device__ __forceinline__ void knn_leaf(const KnnArgs &a, KnnWarpSmem &S, int *leaf_list, uint32_t *leaf_mask,
                                         double *bd, uint32_t *bi, int64_t leaf, float finer_scale = 0.f,
                                         unsigned lanes = 0xffffffffu) {
    const float scale = FINER ? finer_scale : a.scale;
    const int lane = threadIdx.x & 31;
    const TreeView &tv = a.tv;
    const int k = a.k;
    const int64_t qi = leaf * kLeaf + lane;
    bool valid = qi < tv.n && (!FINER || ((lanes >> lane) & 1u));
    KnnWarp<COUNT> W(tv, a.perm, scale, S, leaf_list, leaf_mask);
    W.q = valid ? ld_scaled(&tv.pos[qi], scale) : make_float4(0.f, 0.f, 0.f, 0.f);
    const float4 q = W.q;
    const uint32_t qid = valid ? __ldg(&a.perm[qi]) : 0u;

    auto clear_hist = [&]() {
        for (int b = 0; b < kNB; ++b) S.hist[b][lane] = 0;
        __syncwarp();
    };

    // ---- 1. radius bound from the neighbouring leaves in sorted order
    const int64_t nleaf = tv.cnt[0];
    // a central window of (k + 1)/32 + 2 leaves brackets the bound, the full
    // window of (k + 1)/32 + 10 leaves (13 at k = 64) tightens it: any subset of
    // the other points gives an upper bound, more nearby points a tighter one
    auto window = [&](int64_t wl, int64_t &w0, int64_t &w1) {
        w0 = leaf - wl / 2;
        if (w0 < 0) w0 = 0;
        w1 = w0 + wl - 1;
        if (w1 >= nleaf) {
            w1 = nleaf - 1;
            w0 = w1 - wl + 1 < 0 ? 0 : w1 - wl + 1;
        }
    };
    int64_t c0, c1, w0, w1;
    window((int64_t)((k + 1 + 31) / 32) + 2, c0, c1);
    window((int64_t)((k + 1 + 31) / 32) + 10, w0, w1);
    // first bracket: the farthest corner of the central leaves' joint box
    float whi = 0.f;
    {
        float blo[3] = {INFINITY, INFINITY, INFINITY}, bhi[3] = {-INFINITY, -INFINITY, -INFINITY};
        for (int64_t L = c0; L <= c1; ++L) {
            const float4 lo = ld_scaled(&tv.nlo[L], scale), hi = ld_scaled(&tv.nhi[L], scale);
            blo[0] = fminf(blo[0], lo.x); blo[1] = fminf(blo[1], lo.y); blo[2] = fminf(blo[2], lo.z);
            bhi[0] = fmaxf(bhi[0], hi.x); bhi[1] = fmaxf(bhi[1], hi.y); bhi[2] = fmaxf(bhi[2], hi.z);
        }
        const float dx = fmaxf(q.x - blo[0], bhi[0] - q.x), dy = fmaxf(q.y - blo[1], bhi[1] - q.y),
                    dz = fmaxf(q.z - blo[2], bhi[2] - q.z);
        whi = fmaf(dz, dz, fmaf(dy, dy, dx * dx)) * (1.0f + 1.0e-5f);
        if (FINER) whi = fminf(whi, 0x1p64f);  // no bracket was wider in the coarser scale
    }
    auto window_visit = [&](int64_t L0, int64_t L1, auto fn) {
        for (int64_t L = L0; L <= L1; ++L) {
            const int64_t base = L * kLeaf;
            if (base + lane < tv.n) S.pts[lane] = ld_scaled(&tv.pos[base + lane], scale);
            __syncwarp();
            const int cnt = (int)(tv.n - base < kLeaf ? tv.n - base : kLeaf);
            for (int t = 0; t < cnt; ++t) fn(S.pts[t], base + t);
            __syncwarp();
        }
    };
    // round 0: the central leaves over [0, whi]; round 1: all window leaves over
    // [0, the central k-th's bin] (their k-th is no larger)
    for (int round = 0; round < 2; ++round) {
        float wlo = 0.f;
        clear_hist();
        const float width = whi - wlo;
        const float inv = width > 0.f ? (float)kNB / width : 0.f;
        int below = 0;
        window_visit(round == 0 ? c0 : w0, round == 0 ? c1 : w1, [&](float4 p, int64_t j) {
            if (j != qi) {
                const float d = d2_f32(q, p);
                if (d < wlo) ++below;
                else if (d <= whi) S.hist[min(kNB - 1, (int)((d - wlo) * inv))][lane] += 1;
            }
        });
        __syncwarp();
        int cum = below, b = 0;
        for (; b < kNB; ++b) {
            const int c = S.hist[b][lane];
            if (cum + c >= k) break;
            cum += c;
        }
        // keep the current bracket if rounding left the k-th outside it
        if (b < kNB && width > 0.f) {
            const float nhi = (b == kNB - 1 ? whi : wlo + (float)(b + 1) * (width / (float)kNB)) *
                              (1.0f + 1.0e-6f);
            whi = fminf(nhi, whi);
        }
        if (round == 1) {  // a finer scale?
            const bool room = valid && scale < 0x1p96f && fmaxf(fmaxf(fabsf(q.x), fabsf(q.y)), fabsf(q.z)) < 0x1p96f;
            unsigned left = 0;
            if (__any_sync(0xffffffffu, room && (b == 0 || whi < 1.0f))) {
                int near = 0, same = 0;
                const float lim = whi < 1.0f ? whi : whi * 0x1p-60f;
                window_visit(w0, w1, [&](float4 p, int64_t j) {
                    if (j != qi && d2_f32(q, p) <= lim) {
                        ++near;
                        same += p.x == q.x && p.y == q.y && p.z == q.z;  // at distance 0 in any scale
                    }
                });
                left = __ballot_sync(0xffffffffu, room && near >= k && same < k);
                valid = valid && !((left >> lane) & 1u);
            }
            if (lane == 0) S.left = left;
            if (!__any_sync(0xffffffffu, valid)) return;
        }
    }
    const float T = valid ? whi * (1.0f + 4.0e-6f) + 1.0e-37f : -1.f;

    // ---- 2. candidates within sqrt(T) of at least one lane's point
    W.r2 = T;
    {
        const float r = valid ? sqrtf(T) * (1.0f + 1.0e-5f) : 0.f;
        float lo3[3] = {valid ? q.x - r : INFINITY, valid ? q.y - r : INFINITY, valid ? q.z - r : INFINITY};
        float hi3[3] = {valid ? q.x + r : -INFINITY, valid ? q.y + r : -INFINITY, valid ? q.z + r : -INFINITY};
#pragma unroll
        for (int d = 0; d < 3; ++d)
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) {
                lo3[d] = fminf(lo3[d], __shfl_xor_sync(0xffffffffu, lo3[d], o));
                hi3[d] = fmaxf(hi3[d], __shfl_xor_sync(0xffffffffu, hi3[d], o));
            }
#pragma unroll
        for (int d = 0; d < 3; ++d) {
            W.env_lo[d] = lo3[d];
            W.env_hi[d] = hi3[d];
        }
    }
    // first histogram (32 bins over [0, T]) while the candidates are collected
    clear_hist();
    {
        const float inv0 = (valid && T > 0.f) ? (float)kNB / T : 0.f;
        const float t_a = valid ? T : -INFINITY;
        W.collect([&](int n) {
            for (int t = 0; t < n; ++t) {
                const float4 p = S.pts[t];
                const float d = d2_f32(q, p);
                if (d <= t_a && __float_as_uint(p.w) != qid)
                    S.hist[min(kNB - 1, (int)(d * inv0))][lane] += 1;
            }
            __syncwarp();
        });
    }

    // ---- 3./4. band passes; each also bins the band's bracket for a further round
    float lo_e = 0.f, hi_e = valid ? T : 0.f;
    int below = 0;               // candidates with d2 < lo_e
    bool done = !valid;
    int need = 0;
    double kth = 0.0;
    bool extract = false;
    float band_lo = 0.f, band_hi = 0.f;
    int nb_below = 0;
    for (int round = 0; round < 8; ++round) {
        if (!__any_sync(0xffffffffu, !done && !extract)) break;
        const bool act = !done && !extract;
        const float width = hi_e - lo_e;
        float e_lo = lo_e, e_hi = hi_e;
        if (act) {
            int cum = below, b = 0;
            for (; b < kNB - 1; ++b) {
                const int c = S.hist[b][lane];
                if (cum + c >= k) break;
                cum += c;
            }
            e_lo = lo_e + (float)b * (width / (float)kNB);
            e_hi = (b == kNB - 1) ? hi_e : lo_e + (float)(b + 1) * (width / (float)kNB);
            band_lo = e_lo * (1.0f - kDelta);
            band_hi = e_hi * (1.0f + kDelta);
        }
        clear_hist();
        const float bhi_a = act ? band_hi : -INFINITY;
        const float sub_w = e_hi - e_lo;
        const float sub_inv = sub_w > 0.f ? (float)kNB / sub_w : 0.f;
        int nbelow = 0, nband = 0, below_next = 0;
        // leaves wholly below this lane's band (by the far corner of their box) or
        // wholly above it (by the near corner) need no point loads; the margins
        // cover the rounding of the FP32 distances
        auto cls = [&](float4 lo, float4 hi) -> int {
            if (!act) return 2;
            const float gx = fmaxf(fmaxf(lo.x - q.x, q.x - hi.x), 0.f);
            const float gy = fmaxf(fmaxf(lo.y - q.y, q.y - hi.y), 0.f);
            const float gz = fmaxf(fmaxf(lo.z - q.z, q.z - hi.z), 0.f);
            const float fx = fmaxf(fabsf(q.x - lo.x), fabsf(q.x - hi.x));
            const float fy = fmaxf(fabsf(q.y - lo.y), fabsf(q.y - hi.y));
            const float fz = fmaxf(fabsf(q.z - lo.z), fabsf(q.z - hi.z));
            const float dmin = fmaf(gz, gz, fmaf(gy, gy, gx * gx));
            const float dmax = fmaf(fz, fz, fmaf(fy, fy, fx * fx));
            if (dmax * (1.0f + 1.0e-5f) < band_lo) return 1;
            if (dmin * (1.0f - 1.0e-5f) > band_hi) return 2;
            return 0;
        };
        auto below_all = [&](int n) {
            nbelow += n;
            below_next += n;
        };
        W.each_pruned([&](float4 p) {
            const float d = d2_f32(q, p);
            if (d <= bhi_a) {
                const uint32_t id = __float_as_uint(p.w);
                if (id != qid) {
                    if (d < band_lo) {
                        ++nbelow;
                    } else {
                        if (nband < kBand) {
                            bd[nband * 32 + lane] = d2_f64(q, p);
                            bi[nband * 32 + lane] = id;
                        }
                        ++nband;
                    }
                    if (d < e_lo) ++below_next;
                    else if (d <= e_hi) S.hist[min(kNB - 1, (int)((d - e_lo) * sub_inv))][lane] += 1;
                }
            }
        }, cls, below_all, leaf);
        __syncwarp();
        if (act) {
            need = k - nbelow;
            nb_below = nbelow;
            if (nband <= kBand) {
                for (int x = 1; x < nband; ++x) {
                    const double dv = bd[x * 32 + lane];
                    const uint32_t iv = bi[x * 32 + lane];
                    int y = x - 1;
                    while (y >= 0 && key_less(dv, iv, bd[y * 32 + lane], bi[y * 32 + lane])) {
                        bd[(y + 1) * 32 + lane] = bd[y * 32 + lane];
                        bi[(y + 1) * 32 + lane] = bi[y * 32 + lane];
                        --y;
                    }
                    bd[(y + 1) * 32 + lane] = dv;
                    bi[(y + 1) * 32 + lane] = iv;
                }
                const int pick = min(max(need, 1), min(nband, kBand)) - 1;
                kth = bd[pick * 32 + lane];
                done = true;
            } else if (round == 7 || !(e_hi - e_lo > fmaxf(4.0f * kDelta * e_hi, 1.0e-37f))) {
                extract = true;  // bin cannot shrink further (kNB / width would overflow), or out of rounds
            } else {
                lo_e = e_lo;     // the band pass already binned [e_lo, e_hi]
                hi_e = e_hi;
                below = below_next;
            }
        }
        __syncwarp();
    }
    // ---- fallback: extract the need smallest band members one by one, or (no ids wanted) one
    // distance after the other, with all that share it: FP64 at two lanes a clock bounds these
    // passes (200,000 points of which 15,000 coincide, k = 8: 429 ms one by one, 88 so)
    {
        const bool by_value = !a.nbr_orig;
        double last_d = -1.0;
        uint32_t last_i = 0;
        bool first = true;
        int got = 0;
        while (__any_sync(0xffffffffu, extract && got < need)) {
            const bool act = extract && got < need;
            double best_d = INFINITY;
            uint32_t best_i = 0xffffffffu;
            int same = 0;
            W.each([&](float4 p) {
                const uint32_t id = __float_as_uint(p.w);
                if (act && id != qid) {
                    const float d = d2_f32(q, p);
                    if (d >= band_lo && d <= band_hi) {
                        const double dd = d2_f64(q, p);
                        if (by_value) {
                            if (dd > last_d && dd <= best_d) {
                                same = dd < best_d ? 1 : same + 1;
                                best_d = dd;
                            }
                        } else {
                            const bool after = first || key_less(last_d, last_i, dd, id);
                            if (after && key_less(dd, id, best_d, best_i)) {
                                best_d = dd;
                                best_i = id;
                            }
                        }
                    }
                }
            });
            if (act) {
                if (!by_value && nb_below + got < k) a.nbr_orig[(int64_t)qid * k + nb_below + got] = best_i;
                last_d = best_d;
                last_i = best_i;
                first = false;
                got += by_value ? max(same, 1) : 1;
                if (got >= need) {
                    kth = best_d;
                    done = true;
                }
            }
        }
    }
    if (valid) {
        const double inv = 1.0 / (double)scale;  // a power of two
        a.h_sorted[qi] = (float)sqrt(kth * (inv * inv));
    }

    // ---- optional neighbour ids: the below set, then the band's first `need`
    if (a.nbr_orig) {
        int slot = 0;
        const float blo_a = valid ? band_lo : -INFINITY;
        W.each([&](float4 p) {
            const float d = d2_f32(q, p);
            const uint32_t id = __float_as_uint(p.w);
            if (d < blo_a && id != qid && slot < k) a.nbr_orig[(int64_t)qid * k + slot++] = id;
        });
        if (valid && !extract)
            for (int x = 0; x < need && x < kBand && slot + x < k; ++x)
                a.nbr_orig[(int64_t)qid * k + slot + x] = bi[x * 32 + lane];
    }
    if (COUNT && lane == 0) {
        atomicAdd(&a.work[0], W.ncand);
        if (S.left == 0) atomicAdd(&a.work[1], 1ull);
    }
}

template <bool COUNT>
__device__ __noinline__ void knn_leaf_finer(const KnnArgs &a, KnnWarpSmem &S, int *leaf_list, uint32_t *leaf_mask,
                                            double *bd, uint32_t *bi, int64_t leaf, float scale, unsigned lanes) {
    knn_leaf<COUNT, true>(a, S, leaf_list, leaf_mask, bd, bi, leaf, scale, lanes);
}

template <bool COUNT>
__global__ void __launch_bounds__(kKnnWarps * 32, 7) k_knn(const __grid_constant__ KnnArgs a) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int warp = threadIdx.x >> 5;
    KnnWarpSmem &S = reinterpret_cast<KnnWarpSmem *>(smem_raw)[warp];
    const int64_t slot = (int64_t)blockIdx.x * kKnnWarps + warp;
    int *leaf_list = a.leaf_list + slot * kLeafList;
    uint32_t *leaf_mask = a.leaf_mask + slot * kLeafList;
    double *bd = a.band_d + slot * (kBand * 32);
    uint32_t *bi = a.band_i + slot * (kBand * 32);
    const int64_t nleaf = a.retry ? (int64_t)*a.retry_n : a.tv.cnt[0];
    bool first = a.retry != nullptr;
    while (true) {
        unsigned int leaf = 0;
        // Retried leaves are few and long: the first of each warp is dealt out by block, so that they
        // spread over the SMs (700 of 6,250 leaves, k = 1: 57 ms by the counter alone, 40 so).
        if (first) {
            leaf = warp * gridDim.x + blockIdx.x;
        } else {
            if ((threadIdx.x & 31) == 0) leaf = atomicAdd(a.next_leaf, 1u) + (a.retry ? kKnnWarps * gridDim.x : 0u);
            leaf = __shfl_sync(0xffffffffu, leaf, 0);
        }
        first = false;
        if ((int64_t)leaf >= nleaf) break;
        if (a.retry) leaf = a.retry[leaf];
        knn_leaf<COUNT, false>(a, S, leaf_list, leaf_mask, bd, bi, (int64_t)leaf);
        __syncwarp();
        float scale = a.scale;
        while (const unsigned left = S.left) {  // ends: none is left past 2^96
            __syncwarp();
            scale *= 0x1p30f;
            knn_leaf_finer<COUNT>(a, S, leaf_list, leaf_mask, bd, bi, (int64_t)leaf, scale, left);
            __syncwarp();
        }
    }
}

// ---------------------------------------------------------------------------
// Selection kernel: every candidate is evaluated once.
//
// One warp per leaf of 32 queries, one query per lane. A lane keeps a list of the
// candidates within its current bound T, one word each: the code of the distance
// (upper 16 bits of the FP32 d2: exponent and 8 mantissa bits, a scale-free
// quantisation 0.4% wide) and a 15-bit reference (visit number, point of the leaf).
// When some lane's list could overflow, every lane finds its k-th entry's bin of 16
// codes, drops what lies above it and lowers T, so T shrinks as the search goes on:
//  1. T from one histogram over the 13 leaves around (k = 64; bins of 64 codes);
//  2. those leaves, then the index bottom-up from the query leaf (its siblings, its
//     parent's siblings, ...; within a subtree the nearest child first), so that T is
//     close to its final value before anything far is looked at;
//  3. the k-th entry's code: its few members and those of the codes next to it are
//     evaluated again in FP32 (its d2 is good to 5 * 2^-24, far less than a code), and
//     the k-th and what ties with it within 2e-6 in FP64, ranked by (d2, original
//     index).
// A leaf that this cannot resolve (more equal codes than a list holds, more than 1024 visited
// leaves) goes to a retry list for the same search with longer lists, then to k_knn; one
// whose distances leave the FP32 range straight to k_knn.
//
// What bounds it: issue slots (43,000 instructions a leaf at k = 64, 55% of the slots at
// the 10 warps an SM that the lists leave room for). 16.8M clustered points, k = 64,
// index build included: 116 ms with k_knn alone (two evaluations, a dependent histogram
// update each, 70 instructions a candidate, and single warps that searched for 80 ms
// where the window bounds an isolated point badly), 33 ms now; 100k, k = 32: 1.85 and
// 0.82 ms. Lists of 128 and 176 entries (11, 8 warps an SM) took 4% and 12% longer,
// 64-bin counting without lists (28 warps) twice the visits where T starts loose.
// ---------------------------------------------------------------------------
constexpr int kSelSeq = 1024;            // visited leaves a reference can name
constexpr uint32_t kCodeMask = 0xffff8000u;
constexpr int kMoreLeaves = 8;           // window leaves beyond the central ones (13 in all at k = 64)
constexpr int kRegMembers = 8;           // members (a code and the codes next to it) ranked in registers
constexpr int kRing = 64;                // staged candidates: two halves of 32

template <int CAP>
struct __align__(16) SelWarpSmem {
    uint32_t list[CAP][32];              // row r of lane l: list[r][l]
    float x[kRing], y[kRing], z[kRing];  // staged candidates
    uint32_t ref[kRing];
    union {
        uint32_t hist[17][32];                   // bin b of lane l
        struct { float4 lo[32], hi[32]; } box;   // child boxes under test
    } u;
    float4 glo[8], ghi[8];               // boxes of four queries each; glo.w: their largest T (with slack)
    int stack[32 * kMaxLevels];
};

struct KnnSelArgs {
    TreeView tv;
    const uint32_t *perm;
    int k;
    float *h_sorted;
    int *seq_leaf;               // [slots][kSelSeq] leaves visited for the current query leaf
    unsigned int *next_leaf;     // work counter (zeroed before launch)
    const unsigned int *todo;    // nullable: the query leaves to process (*todo_n of them)
    const unsigned int *todo_n;
    unsigned int *retry;         // [leaves] the leaves left to the next kernel: longer lists
    unsigned int *retry_n;       // their number (zeroed before launch)
    unsigned int *beyond;        // [leaves] those that FP32 distances cannot resolve: k_knn
    unsigned int *beyond_n;
    unsigned long long *work;    // nullable: as KnnArgs::work
};

template <int CAP, bool COUNT>
struct KnnSel {
    static constexpr int kKeep = CAP - 32;  // a list this long still takes 32 candidates
    const KnnSelArgs &a;
    SelWarpSmem<CAP> &S;
    int *seq_leaf;
    float4 q;
    float T;
    int cnt, seq;
    int head, staged;            // the ring: first staged candidate, how many (warp-uniform)
    bool fail, below32;          // warp-uniform: given up; because a k-th d2 is out of FP32's range
    float env_lo[3], env_hi[3];  // box around all lanes' balls
    unsigned long long ncand = 0;

    __device__ KnnSel(const KnnSelArgs &args, SelWarpSmem<CAP> &s, int *sl) : a(args), S(s), seq_leaf(sl) {}

    __device__ static int lane_id() { return threadIdx.x & 31; }

    // The query points' boxes, by groups of four lanes (Morton neighbours).
    __device__ void groups(bool valid) {
        float lo[3] = {valid ? q.x : INFINITY, valid ? q.y : INFINITY, valid ? q.z : INFINITY};
        float hi[3] = {valid ? q.x : -INFINITY, valid ? q.y : -INFINITY, valid ? q.z : -INFINITY};
#pragma unroll
        for (int d = 0; d < 3; ++d)
#pragma unroll
            for (int o = 1; o < 4; o <<= 1) {
                lo[d] = fminf(lo[d], __shfl_xor_sync(0xffffffffu, lo[d], o));
                hi[d] = fmaxf(hi[d], __shfl_xor_sync(0xffffffffu, hi[d], o));
            }
        if ((lane_id() & 3) == 0) {
            S.glo[lane_id() >> 2] = make_float4(lo[0], lo[1], lo[2], -1.f);
            S.ghi[lane_id() >> 2] = make_float4(hi[0], hi[1], hi[2], 0.f);
        }
        __syncwarp();
    }

    // After T changed: the box around all balls and the groups' largest T.
    __device__ void reach() {
        const bool on = T >= 0.f;
        const float r = on ? sqrtf(T) * (1.0f + 1.0e-5f) : 0.f;
        float lo3[3] = {on ? q.x - r : INFINITY, on ? q.y - r : INFINITY, on ? q.z - r : INFINITY};
        float hi3[3] = {on ? q.x + r : -INFINITY, on ? q.y + r : -INFINITY, on ? q.z + r : -INFINITY};
        float t = T;
#pragma unroll
        for (int o = 1; o < 4; o <<= 1) t = fmaxf(t, __shfl_xor_sync(0xffffffffu, t, o));
        if ((lane_id() & 3) == 0) S.glo[lane_id() >> 2].w = t * (1.0f + 2.0e-5f);
#pragma unroll
        for (int d = 0; d < 3; ++d)
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) {
                lo3[d] = fminf(lo3[d], __shfl_xor_sync(0xffffffffu, lo3[d], o));
                hi3[d] = fmaxf(hi3[d], __shfl_xor_sync(0xffffffffu, hi3[d], o));
            }
#pragma unroll
        for (int d = 0; d < 3; ++d) {
            env_lo[d] = lo3[d];
            env_hi[d] = hi3[d];
        }
        __syncwarp();
    }

    __device__ static float gap2(float4 lo, float4 hi, float4 qlo, float4 qhi) {
        const float dx = fmaxf(fmaxf(lo.x - qhi.x, qlo.x - hi.x), 0.f);
        const float dy = fmaxf(fmaxf(lo.y - qhi.y, qlo.y - hi.y), 0.f);
        const float dz = fmaxf(fmaxf(lo.z - qhi.z, qlo.z - hi.z), 0.f);
        return fmaf(dz, dz, fmaf(dy, dy, dx * dx));
    }

    // The children (lane c holds one) within the ball of at least one lane (relative
    // slack 1e-5): tested one per lane against the 8 groups, the few that pass then
    // against every ball (a group's box is wide at a jump of the Morton order).
    // dist: the child's least squared distance to a group.
    __device__ unsigned accept(int node, bool valid, float &dist) {
        float4 lo = make_float4(INFINITY, INFINITY, INFINITY, 0.f), hi = lo;
        if (valid) {
            lo = __ldg(&a.tv.nlo[node]);
            hi = __ldg(&a.tv.nhi[node]);
        }
        bool near = false;
        dist = INFINITY;
#pragma unroll 4
        for (int g = 0; g < 8; ++g) {
            const float4 gl = S.glo[g], gh = S.ghi[g];
            const float d2 = gap2(lo, hi, gl, gh);
            near = near || d2 <= gl.w;
            dist = fminf(dist, d2);
        }
        near = near && valid;
        unsigned m = __ballot_sync(0xffffffffu, near);
        if (near) {
            S.u.box.lo[lane_id()] = lo;
            S.u.box.hi[lane_id()] = hi;
        }
        __syncwarp();
        unsigned acc = 0;
        const float lim = T >= 0.f ? T * (1.0f + 1.0e-5f) : -1.f;
        while (m) {  // two at a time: independent chains
            const int j0 = __ffs(m) - 1;
            m &= m - 1;
            const int j1 = m ? __ffs(m) - 1 : j0;
            m &= m - 1;
            const bool n0 = gap2(S.u.box.lo[j0], S.u.box.hi[j0], q, q) <= lim;
            const bool n1 = gap2(S.u.box.lo[j1], S.u.box.hi[j1], q, q) <= lim;
            if (__any_sync(0xffffffffu, n0)) acc |= 1u << j0;
            if (__any_sync(0xffffffffu, n1)) acc |= 1u << j1;
        }
        __syncwarp();
        return acc;
    }

    // Staged candidates e, ..., e + 7: their FP32 d2.
    __device__ void eight(int e, float d[8]) const {
        const f32x2 QX = f2_pack(q.x, q.x), QY = f2_pack(q.y, q.y), QZ = f2_pack(q.z, q.z);
#pragma unroll
        for (int i = 0; i < 8; i += 4) {
            const ulonglong2 X = *reinterpret_cast<const ulonglong2 *>(&S.x[e + i]);
            const ulonglong2 Y = *reinterpret_cast<const ulonglong2 *>(&S.y[e + i]);
            const ulonglong2 Z = *reinterpret_cast<const ulonglong2 *>(&S.z[e + i]);
            f32x2 dx = f2_sub(QX, X.x), dy = f2_sub(QY, Y.x), dz = f2_sub(QZ, Z.x);
            f2_unpack(f2_fma(dz, dz, f2_fma(dy, dy, f2_mul(dx, dx))), d[i], d[i + 1]);
            dx = f2_sub(QX, X.y), dy = f2_sub(QY, Y.y), dz = f2_sub(QZ, Z.y);
            f2_unpack(f2_fma(dz, dz, f2_fma(dy, dy, f2_mul(dx, dx))), d[i + 2], d[i + 3]);
        }
    }

    // The bin of 2^sh codes that holds the rank-th smallest of the lane's first num entries:
    // its lowest code; false if num < rank. 16 bins a pass from `top` (a code the entry is
    // not above) downwards; the lowest takes the rest, and if the entry sought is among
    // these, another pass goes on from there. Every lane counts in its own column with
    // shared-memory atomics, which nothing waits for.
    __device__ bool locate(int sh, int num, int rank, uint32_t top, int &code_lo) {
        const int lane = lane_id();
        const int rows = __reduce_max_sync(0xffffffffu, num);
        int hib = (int)(top >> sh);
        const bool found = num >= rank;
        bool open = found;
        while (__any_sync(0xffffffffu, open)) {
            const int base = hib - 15;
#pragma unroll
            for (int b = 0; b < 16; ++b) S.u.hist[b][lane] = 0u;
            if (open) {
                for (int r = 0; r < rows; r += 8) {
                    uint32_t e[8];
#pragma unroll
                    for (int i = 0; i < 8; ++i) e[i] = S.list[r + i][lane];  // CAP is a multiple of 8
#pragma unroll
                    for (int i = 0; i < 8; ++i) {
                        // entries above the bins and rows past the end go to a 17th
                        const int b = r + i < num ? (int)(e[i] >> (15 + sh)) - base : 16;
                        atomicAdd(&S.u.hist[min(max(b, 0), 16)][lane], 1u);
                    }
                }
                int cum = 0, b = 0;
                for (; b < 15; ++b) {
                    cum += (int)S.u.hist[b][lane];
                    if (cum >= rank) break;
                }
                if (b == 0 && base > 0) {
                    hib = base;
                } else {
                    code_lo = (base + b) << sh;
                    open = false;
                }
            }
        }
        __syncwarp();
        return found;
    }

    // Keeps the lane's entries (of the first num) in [lo, hi], in order, at the front.
    __device__ int keep(int num, uint32_t lo, uint32_t hi) {
        const int lane = lane_id();
        const int rows = __reduce_max_sync(0xffffffffu, num);
        int w = 0;
        for (int r = 0; r < rows; r += 8) {
            uint32_t e[8];
#pragma unroll
            for (int i = 0; i < 8; ++i) e[i] = S.list[r + i][lane];
#pragma unroll
            for (int i = 0; i < 8; ++i)
                if (e[i] - lo <= hi - lo && r + i < num) S.list[w++][lane] = e[i];  // w <= r + i
        }
        return w;
    }

    // Every lane drops the entries above its k-th one's bin (but keeps the code next to
    // it) and lowers T to match: bins of 16 codes, of one code where that leaves a list
    // too long; sets fail if one still is.
    __device__ void compact() {
        for (int sh = 4; sh >= 0; sh -= 4) {
            int code_lo = 0;
            if (locate(sh, cnt, a.k + 1, __float_as_uint(T) >> 15, code_lo))
                T = fminf(T, __uint_as_float(((uint32_t)(code_lo + (1 << sh) + 1) << 15) - 1u));
            cnt = keep(cnt, 0u, T >= 0.f ? __float_as_uint(T) | 0x7fffu : 0u);
            fail = __any_sync(0xffffffffu, cnt > kKeep);
            if (!fail) break;
        }
        reach();
    }

    // Point of a list entry.
    __device__ int point_of(uint32_t e) const {
        return seq_leaf[(e >> 5) & (kSelSeq - 1)] * kLeaf + (int)(e & 31u);
    }

    // The FP64 squared distance of the k-th neighbour from the finished lists; sets fail
    // where FP32 is no guide.
    __device__ double kth_d2(bool valid) {
        const int lane = lane_id();
        const TreeView &tv = a.tv;
        // the k-th entry's bin of 16 codes, then its code, each with the codes next to it (which
        // the rounding of FP32 d2 reaches): the lists shrink to these few members
        int nmem = cnt, need = a.k + 1;  // 1-based rank among the members (the point itself is one)
        int code_lo = 0;
        uint32_t top = __float_as_uint(T) >> 15;
        bool found = false;
        for (int sh = 4; sh >= 0; sh -= 4) {
            const bool f = locate(sh, nmem, need, top, code_lo);
            if (sh == 4) {
                found = f;
                if (!f) nmem = 0;
            }
            const uint32_t lo = (uint32_t)max(code_lo - 1, 0) << 15,
                           hi = ((uint32_t)(code_lo + (1 << sh) + 1) << 15) - 1u;
            int less = 0;
            const int rows = __reduce_max_sync(0xffffffffu, nmem);
            for (int r = 0; r < rows; r += 8)
#pragma unroll
                for (int i = 0; i < 8; ++i) less += r + i < nmem && S.list[r + i][lane] < lo;
            need -= less;
            nmem = keep(nmem, lo, hi);
            if (__all_sync(0xffffffffu, nmem <= kRegMembers)) break;
            top = (uint32_t)(code_lo + 15);
        }
        bool ok = (found || !valid) && nmem <= CAP / 2;
        double kth = 0.0;
        if (!__all_sync(0xffffffffu, ok)) {
            fail = true;
            return kth;
        }
        float dk = INFINITY;           // the FP32 d2 of that rank
        int sure = 0, ties = 0;        // members FP32 puts below it; those it cannot tell from it
        int at = 0;                    // the point, where there is no tie
        if (__all_sync(0xffffffffu, nmem <= kRegMembers)) {
            float dm[kRegMembers];
            int pm[kRegMembers];
#pragma unroll
            for (int i = 0; i < kRegMembers; ++i) pm[i] = i < nmem ? point_of(S.list[i][lane]) : -1;
#pragma unroll
            for (int i = 0; i < kRegMembers; ++i)
                dm[i] = i < nmem ? d2_f32(q, __ldg(&tv.pos[pm[i]])) : INFINITY;
#pragma unroll
            for (int i = 0; i < kRegMembers; ++i) {
                int le = 0;
#pragma unroll
                for (int j = 0; j < kRegMembers; ++j) le += dm[j] <= dm[i];
                if (le >= need) dk = fminf(dk, dm[i]);
            }
#pragma unroll
            for (int i = 0; i < kRegMembers; ++i) {
                sure += dm[i] < dk * (1.0f - kDelta);
                if (dm[i] >= dk * (1.0f - kDelta) && dm[i] <= dk * (1.0f + kDelta)) {
                    ++ties;
                    at = pm[i];
                }
                if (i < nmem) S.list[CAP / 2 + i][lane] = __float_as_uint(dm[i]);
            }
        } else {
            for (int i = 0; i < nmem; ++i)
                S.list[CAP / 2 + i][lane] = __float_as_uint(d2_f32(q, __ldg(&tv.pos[point_of(S.list[i][lane])])));
            for (int le = 0; le < need && nmem > 0;) {  // from one value to the next
                const float last = dk == INFINITY ? -1.f : dk;
                float next = INFINITY;
                int c = 0;
                for (int i = 0; i < nmem; ++i) {
                    const float di = __uint_as_float(S.list[CAP / 2 + i][lane]);
                    if (di > last && di <= next) {
                        c = di < next ? 1 : c + 1;
                        next = di;
                    }
                }
                dk = next;
                le += max(c, 1);
            }
            for (int i = 0; i < nmem; ++i) {
                const float di = __uint_as_float(S.list[CAP / 2 + i][lane]);
                sure += di < dk * (1.0f - kDelta);
                if (di >= dk * (1.0f - kDelta) && di <= dk * (1.0f + kDelta)) {
                    ++ties;
                    at = point_of(S.list[i][lane]);
                }
            }
        }
        // d2 = 0 in FP32: the k-th coincides with the query, or FP32 does not show how far it is. (The
        // lists of 144 leave that to k_knn: with this loop their kernel takes 2.7% longer.)
        bool at_zero = false;
        if constexpr (CAP != 144) {
            int zero = 0;
            if (found && dk == 0.f)
                for (int i = 0; i < nmem; ++i) {
                    const float4 p = __ldg(&tv.pos[point_of(S.list[i][lane])]);
                    zero += p.x == q.x && p.y == q.y && p.z == q.z;
                }
            at_zero = found && dk == 0.f && zero >= need;
        }
        if (found && !at_zero && !(dk > 1.0e-34f && dk < 1.0e37f)) ok = false;
        if (found && ok && !at_zero) {
            kth = d2_f64(q, __ldg(&tv.pos[at]));
            if (ties > 1) {  // rank them in FP64, from one value to the next (exact ties are one)
                kth = -1.0;
                for (int left = need - sure; left > 0;) {
                    double next = INFINITY;
                    int c = 0;
                    for (int i = 0; i < nmem; ++i) {
                        const float di = __uint_as_float(S.list[CAP / 2 + i][lane]);
                        if (di < dk * (1.0f - kDelta) || di > dk * (1.0f + kDelta)) continue;
                        const double dd = d2_f64(q, __ldg(&tv.pos[point_of(S.list[i][lane])]));
                        if (dd > kth && dd <= next) {
                            c = dd < next ? 1 : c + 1;
                            next = dd;
                        }
                    }
                    kth = next;
                    left -= max(c, 1);
                }
            }
        }
        fail = below32 = !__all_sync(0xffffffffu, ok);
        return kth;
    }

    // More than k points of the run around qi at its place? Points that coincide follow one another
    // in the index (prev, next: whether the neighbours do).
    __device__ bool coincide(int qi, bool prev, bool next) const {
        auto same = [&](int i) {
            const float4 p = __ldg(&a.tv.pos[i]);
            return p.x == q.x && p.y == q.y && p.z == q.z;
        };
        int lo = qi, hi = qi;
        while (prev && lo > 0 && hi - lo < a.k && same(lo - 1)) --lo;
        while (next && hi + 1 < (int)a.tv.n && hi - lo < a.k && same(hi + 1)) ++hi;
        return hi - lo >= a.k;
    }

    __device__ void leaf(int leaf) {
        const int lane = lane_id();
        const TreeView &tv = a.tv;
        const int n_all = (int)tv.n, nleaf = (int)tv.cnt[0];  // both below 2^31
        const int qi = leaf * kLeaf + lane;
        bool valid = qi < n_all;
        q = valid ? __ldg(&tv.pos[qi]) : make_float4(0.f, 0.f, 0.f, 0.f);
        cnt = seq = head = staged = 0;
        fail = below32 = false;
        // More than k points at one place: the k-th is at 0, which FP32 distances do not show (1M
        // points at 25,000 places, k = 8: 12.2 ms when such leaves went to k_knn, 0.33 ms now).
        // Where few warps hide the loads of the neighbours they are shuffled: k = 64 of 4M
        // clustered points takes 1% longer with this, 3.5% by loads; k = 8 0% by loads, 2% so.
        bool prev = true, next = true;
        if (CAP > 128) {
            const float4 o = __ldg(&tv.pos[lane == 0 ? max(qi - 1, 0) : min(qi + 1, n_all - 1)]);  // lanes 0 and 31
            auto same = [&](float x, float y, float z, bool edge) {
                return edge ? o.x == q.x && o.y == q.y && o.z == q.z : x == q.x && y == q.y && z == q.z;
            };
            prev = same(__shfl_up_sync(0xffffffffu, q.x, 1), __shfl_up_sync(0xffffffffu, q.y, 1),
                        __shfl_up_sync(0xffffffffu, q.z, 1), lane == 0);
            next = same(__shfl_down_sync(0xffffffffu, q.x, 1), __shfl_down_sync(0xffffffffu, q.y, 1),
                        __shfl_down_sync(0xffffffffu, q.z, 1), lane == 31);
        }
        if (valid && (prev || next) && coincide(qi, prev, next)) {
            a.h_sorted[qi] = 0.f;
            valid = false;
        }
        groups(valid);

        // ---- 1. the leaves around this one: any k of their points bound the k-th distance
        // (the far corner of the central ones' joint box brackets it, more leaves tighten it)
        auto window = [&](int wl, int &w0, int &w1) {
            w0 = max(leaf - wl / 2, 0);
            w1 = min(w0 + wl - 1, nleaf - 1);
            w0 = max(w1 - wl + 1, 0);
        };
        int c0, c1, w0, w1;
        window((a.k + 1 + 31) / 32 + 2, c0, c1);
        window((a.k + 1 + 31) / 32 + 2 + kMoreLeaves, w0, w1);
        {
            float4 blo = __ldg(&tv.nlo[c0]), bhi = __ldg(&tv.nhi[c0]);
            for (int L = c0 + 1; L <= c1; ++L) {
                const float4 lo = __ldg(&tv.nlo[L]), hi = __ldg(&tv.nhi[L]);
                blo.x = fminf(blo.x, lo.x); blo.y = fminf(blo.y, lo.y); blo.z = fminf(blo.z, lo.z);
                bhi.x = fmaxf(bhi.x, hi.x); bhi.y = fmaxf(bhi.y, hi.y); bhi.z = fmaxf(bhi.z, hi.z);
            }
            const float dx = fmaxf(q.x - blo.x, bhi.x - q.x), dy = fmaxf(q.y - blo.y, bhi.y - q.y),
                        dz = fmaxf(q.z - blo.z, bhi.z - q.z);
            const float far = fminf(fmaf(dz, dz, fmaf(dy, dy, dx * dx)) * (1.0f + 1.0e-5f), 3.0e38f);
            // 32 bins of 64 codes from there down (8 octaves; the lowest takes the rest, a 33rd
            // what lies above), in the lists' memory: they are still empty
            const int base = (int)(__float_as_uint(far) >> 21) - 31;
#pragma unroll
            for (int b = 0; b < 33; ++b) S.list[b][lane] = 0u;
            float4 pn = __ldg(&tv.pos[min(w0 * kLeaf + lane, n_all - 1)]);
            for (int L = w0; L <= w1; ++L) {
                __syncwarp();
                S.x[lane] = L * kLeaf + lane < n_all ? pn.x : INFINITY;  // infinitely far: above the bins
                S.y[lane] = pn.y;
                S.z[lane] = pn.z;
                if (L < w1) pn = __ldg(&tv.pos[min((L + 1) * kLeaf + lane, n_all - 1)]);
                if (COUNT) ncand += min(kLeaf, n_all - L * kLeaf);
                __syncwarp();
                for (int e = 0; e < kLeaf; e += 8) {
                    float d[8];
                    eight(e, d);
#pragma unroll
                    for (int i = 0; i < 8; ++i) {  // the lane's own column: no result, no wait
                        const int b = (int)(__float_as_uint(d[i]) >> 21) - base;
                        atomicAdd(&S.list[min(max(b, 0), 32)][lane], 1u);
                    }
                }
            }
            int cum = 0, b = 0;
            for (; b < 31; ++b) {
                cum += (int)S.list[b][lane];
                if (cum > a.k) break;  // the point itself is counted
            }
            // The margin (as k_knn's) is the rounding of FP32 d2: the point FP32 puts just above the
            // bin's edge may be nearer than the one it puts just below.
            T = b < 31 && base + b >= 0
                    ? fminf(__uint_as_float((uint32_t)(base + b + 1) << 21) * (1.0f + 4.0e-6f), far)
                    : far;
            if (!valid) T = -1.f;
            __syncwarp();
        }
        reach();

        // ---- 2. those leaves, then the index from the query leaf upwards
        int cand0 = w0;  // leaves to look at: cand0 + the bits of cm
        unsigned cm = w1 - w0 + 1 >= 32 ? 0xffffffffu : (1u << (w1 - w0 + 1)) - 1u;
        float4 pn = make_float4(INFINITY, 0.f, 0.f, 0.f);  // the next leaf's point
        auto load = [&]() {
            const int j = (cand0 + __ffs(cm) - 1) * kLeaf + lane;
            pn = make_float4(INFINITY, 0.f, 0.f, 0.f);
            if (j < n_all) pn = __ldg(&tv.pos[j]);
        };
        load();
        int sp = 0, up = 0;
        bool end = false;
        while (!end) {
            if (cm) {  // a leaf: its points inside the envelope are staged
                const int L = cand0 + __ffs(cm) - 1;
                cm &= cm - 1;
                const float4 p = pn;
                if (cm) load();
                if (seq >= kSelSeq) {
                    fail = true;
                    break;
                }
                const bool in = p.x >= env_lo[0] && p.x <= env_hi[0] && p.y >= env_lo[1] &&
                                p.y <= env_hi[1] && p.z >= env_lo[2] && p.z <= env_hi[2];
                const unsigned im = __ballot_sync(0xffffffffu, in);
                if (im == 0) continue;
                if (COUNT) ncand += __popc(im);
                if (in) {
                    const int s = (head + staged + __popc(im & ((1u << lane) - 1u))) & (kRing - 1);
                    S.x[s] = p.x;
                    S.y[s] = p.y;
                    S.z[s] = p.z;
                    S.ref[s] = (uint32_t)(seq * 32 + lane);
                }
                if (lane == 0) seq_leaf[seq] = L;
                ++seq;
                staged += __popc(im);
            } else {  // a node: from the stack, or the next ancestor
                int lv, node = 0, skip = -1;
                if (sp > 0) {
                    const int e = S.stack[sp - 1];
                    __syncwarp();
                    sp -= 1;
                    lv = e >> 27;
                    node = e & ((1 << 27) - 1);
                } else {
                    lv = ++up;
                    if (lv < tv.nlevels) {
                        node = leaf >> (5 * lv);
                        skip = leaf >> (5 * (lv - 1));
                    }
                }
                if (lv >= tv.nlevels) {
                    end = true;
                } else {
                    const int c = node * kFanout + lane;
                    bool ok = c < (int)tv.cnt[lv - 1] && c != skip;
                    if (lv == 1) ok = ok && !(c >= w0 && c <= w1);
                    float dist;
                    const unsigned m = accept((int)tv.off[lv - 1] + c, ok, dist);
                    if (lv == 1) {
                        cand0 = node * kFanout;
                        cm = m;
                        if (cm) load();
                    } else {  // pushed, the nearest on top
                        int place = 0;
                        for (unsigned t = m; t; t &= t - 1) {
                            const int j = __ffs(t) - 1;
                            const float dj = __shfl_sync(0xffffffffu, dist, j);
                            place += dj < dist || (dj == dist && j < lane);
                        }
                        const int kk = __popc(m);
                        if ((m >> lane) & 1u) S.stack[sp + (kk - 1 - place)] = ((lv - 1) << 27) | c;
                        sp += kk;
                        __syncwarp();
                    }
                }
            }
            // evaluated 32 at a time (at the end what is left, padded to a multiple of 8)
            if (staged < 32 && !(end && staged > 0)) continue;
            const int n = min(32, (staged + 7) & ~7);
            if (lane >= staged && lane < n) S.x[head + lane] = INFINITY;  // infinitely far
            __syncwarp();
            {
                uint32_t *w = &S.list[cnt][lane];
                uint32_t *const w_0 = w;
                for (int e = head; e < head + n; e += 8) {
                    float d[8];
                    eight(e, d);
                    const uint4 r0 = *reinterpret_cast<const uint4 *>(&S.ref[e]);
                    const uint4 r1 = *reinterpret_cast<const uint4 *>(&S.ref[e + 4]);
                    const uint32_t r[8] = {r0.x, r0.y, r0.z, r0.w, r1.x, r1.y, r1.z, r1.w};
#pragma unroll
                    for (int i = 0; i < 8; ++i)
                        if (d[i] <= T) {
                            *w = (__float_as_uint(d[i]) & kCodeMask) | r[i];
                            w += 32;
                        }
                }
                cnt += (int)(w - w_0) / 32;
            }
            __syncwarp();
            head ^= 32;
            staged = max(staged - 32, 0);
            if (__any_sync(0xffffffffu, cnt > kKeep)) {
                compact();
                if (fail) break;
            }
        }

        // ---- 3. the k-th
        double kth = 0.0;
        if (!fail) kth = kth_d2(valid);
        if (fail) {
            if (lane == 0) {
                if (below32) a.beyond[atomicAdd(a.beyond_n, 1u)] = (unsigned int)leaf;
                else a.retry[atomicAdd(a.retry_n, 1u)] = (unsigned int)leaf;
            }
        } else if (valid) {
            a.h_sorted[qi] = (float)sqrt(kth);
        }
        if (COUNT && lane == 0) {
            atomicAdd(&a.work[0], ncand);
            if (!fail) atomicAdd(&a.work[1], 1ull);  // a retried leaf is counted there
        }
        ncand = 0;
        __syncwarp();
    }
};

template <int CAP, int WARPS, bool COUNT>
__global__ void __launch_bounds__(WARPS * 32) k_knn_sel(KnnSelArgs a) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int warp = threadIdx.x >> 5;
    SelWarpSmem<CAP> &S = reinterpret_cast<SelWarpSmem<CAP> *>(smem_raw)[warp];
    const int64_t slot = (int64_t)blockIdx.x * WARPS + warp;
    KnnSel<CAP, COUNT> W(a, S, a.seq_leaf + slot * kSelSeq);
    const int64_t nleaf = a.todo ? (int64_t)*a.todo_n : a.tv.cnt[0];
    while (true) {
        unsigned int leaf = 0;
        if ((threadIdx.x & 31) == 0) leaf = atomicAdd(a.next_leaf, 1u);
        leaf = __shfl_sync(0xffffffffu, leaf, 0);
        if ((int64_t)leaf >= nleaf) break;
        if (a.todo) leaf = a.todo[leaf];
        W.leaf((int)leaf);
    }
}

// The kNN's work accounting: after a launch with a.work set.
__global__ void k_knn_work_out(const unsigned long long *work, int64_t *out) {
    if (threadIdx.x == 0) {
        out[0] = (int64_t)work[0] * 32;  // (lane, candidate) distance evaluations
        out[1] = (int64_t)work[0];
        out[2] = (int64_t)work[1];
    }
}

__global__ void k_store_h(const float *__restrict__ h, int64_t n, float4 *__restrict__ pos) {
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n;
         i += (int64_t)gridDim.x * blockDim.x)
        pos[i].w = h[i];
}

__global__ void k_scatter_h(const float4 *__restrict__ pos, const uint32_t *__restrict__ perm,
                            int64_t n, float *__restrict__ h_orig) {
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n;
         i += (int64_t)gridDim.x * blockDim.x)
        h_orig[perm[i]] = pos[i].w;
}

__global__ void k_scatter_f(const float *__restrict__ v, const uint32_t *__restrict__ perm,
                            int64_t n, float *__restrict__ out) {
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n;
         i += (int64_t)gridDim.x * blockDim.x)
        out[perm[i]] = v[i];
}

template <int CAP, int WARPS, bool COUNT>
static sf_status launch_sel_t(const KnnSelArgs &a_in, int64_t nleaf, Scratch &sc, cudaStream_t s) {
    KnnSelArgs a = a_in;
    const size_t smem = sizeof(SelWarpSmem<CAP>) * WARPS;
    static std::atomic<uint64_t> attr{0};
    SF_TRY_CUDA(smem_attr_once(k_knn_sel<CAP, WARPS, COUNT>, smem, attr));
    int dev = 0, sms = 0, per_sm = 0;
    SF_TRY_CUDA(cudaGetDevice(&dev));
    SF_TRY_CUDA(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
    SF_TRY_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_knn_sel<CAP, WARPS, COUNT>, WARPS * 32, smem));
    // persistent: one resident wave, never more blocks than leaves need
    const int64_t blocks = std::max<int64_t>(1, std::min<int64_t>((int64_t)sms * std::max(1, per_sm),
                                                                  (nleaf + WARPS - 1) / WARPS));
    a.seq_leaf = sc.get<int>(blocks * WARPS * (int64_t)kSelSeq);
    SF_TRY_SCRATCH(sc);
    SF_TRY_CUDA(launch(k_knn_sel<CAP, WARPS, COUNT>, dim3((unsigned)blocks), dim3(WARPS * 32), smem, s, a));
    return SF_OK;
}

template <int CAP, int WARPS>
static sf_status launch_sel(const KnnSelArgs &a, int64_t nleaf, Scratch &sc, cudaStream_t s) {
    return a.work ? launch_sel_t<CAP, WARPS, true>(a, nleaf, sc, s) : launch_sel_t<CAP, WARPS, false>(a, nleaf, sc, s);
}

sf_status knn_run(sf_index *idx, int k, uint32_t *d_nbr_orig, float *d_h_sorted, cudaStream_t s,
                  unsigned long long *d_work = nullptr) {
    KnnArgs a;
    a.tv = idx->view();
    a.perm = idx->perm;
    a.k = k;
    a.h_sorted = d_h_sorted;
    a.nbr_orig = d_nbr_orig;
    a.work = d_work;
    a.retry = a.retry_n = nullptr;
    float extent = 0.f, most = 0.f;
    for (int d = 0; d < 3; ++d) {
        extent = std::max(extent, idx->bbox_hi[d] - idx->bbox_lo[d]);
        most = std::max(most, std::max(std::fabs(idx->bbox_lo[d]), std::fabs(idx->bbox_hi[d])));
    }
    // differences of at most 2^31, and the largest coordinate stays finite
    const int e = std::min(30 - (std::isfinite(extent) ? (extent > 0.f ? std::ilogb(extent) : 30) : 128),
                           most > 0.f ? 126 - std::ilogb(most) : 0);
    a.scale = std::ldexp(1.0f, std::min(e, 126));
    Scratch sc(s);
    unsigned int *counters = sc.get<unsigned int>(5);  // next leaf of three kernels, two retry counts
    SF_TRY_SCRATCH(sc);
    SF_TRY_CUDA(cudaMemsetAsync(counters, 0, 5 * sizeof(unsigned int), s));
    a.next_leaf = counters;
    KTimer timer(d_work ? "k_knn_count" : "k_knn", s);
    if (!d_nbr_orig) {  // the neighbour ids are k_knn's
        // Lists of CAP entries: between leaves CAP - 32 of them, which have to hold k and the
        // boundary's ties and leave room, so that few leaves force a compaction; shared
        // memory (128 bytes a row and warp) sets how many warps an SM holds. 144 entries serve up
        // to k = 92: there 1M uniform points take 3.2 ms (400 entries 5.4), at 100 4.4 and 5.5,
        // but 100,000 clustered ones 0.59 and 0.66, 0.83 and 0.68 ms (k_knn alone 8.3 and 7.2 ms,
        // 2.4 and 2.5; with the line at 66, k = 67 took 4.90 ms, more than k_knn's 4.27).
        KnnSelArgs b;
        b.tv = a.tv;
        b.perm = a.perm;
        b.k = k;
        b.h_sorted = d_h_sorted;
        b.seq_leaf = nullptr;
        b.next_leaf = counters + 1;
        b.todo = b.todo_n = nullptr;
        b.retry_n = counters + 3;
        b.retry = sc.get<unsigned int>(k <= 92 ? idx->cnt[0] : 1);
        b.beyond_n = counters + 4;
        b.beyond = sc.get<unsigned int>(idx->cnt[0]);
        b.work = d_work;
        SF_TRY_SCRATCH(sc);
        if (k <= 92) {
            if (k <= 34) SF_TRY((launch_sel<96, 13>(b, idx->cnt[0], sc, s)));
            else SF_TRY((launch_sel<144, 10>(b, idx->cnt[0], sc, s)));
            b.todo = b.retry;
            b.todo_n = b.retry_n;
        }
        b.next_leaf = counters + 2;
        b.retry_n = b.beyond_n;
        b.retry = b.beyond;
        SF_TRY((launch_sel<400, 4>(b, idx->cnt[0], sc, s)));
        a.retry = b.retry;
        a.retry_n = b.retry_n;
    }
    const size_t smem = sizeof(KnnWarpSmem) * kKnnWarps;
    auto kern = d_work ? k_knn<true> : k_knn<false>;
    static std::atomic<uint64_t> attr_plain{0}, attr_count{0};
    SF_TRY_CUDA(smem_attr_once(kern, smem, d_work ? attr_count : attr_plain));
    int dev = 0, sms = 0, per_sm = 0;
    SF_TRY_CUDA(cudaGetDevice(&dev));
    SF_TRY_CUDA(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
    SF_TRY_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, kKnnWarps * 32, smem));
    if (per_sm < 1) per_sm = 1;
    // persistent: one resident wave, never more blocks than leaves need
    const int64_t need_blocks = (idx->cnt[0] + kKnnWarps - 1) / kKnnWarps;
    const int64_t blocks = std::max<int64_t>(1, std::min<int64_t>((int64_t)sms * per_sm, need_blocks));
    a.leaf_list = sc.get<int>(blocks * kKnnWarps * (int64_t)kLeafList);
    a.leaf_mask = sc.get<uint32_t>(blocks * kKnnWarps * (int64_t)kLeafList);
    a.band_d = sc.get<double>(blocks * kKnnWarps * (int64_t)kBand * 32);
    a.band_i = sc.get<uint32_t>(blocks * kKnnWarps * (int64_t)kBand * 32);
    SF_TRY_SCRATCH(sc);
    SF_TRY_CUDA(launch(kern, dim3((unsigned)blocks), dim3(kKnnWarps * 32), smem, s, a));
    return SF_OK;
}

// Bandwidths resident in the index: h into pos.w, node maxima rebuilt.
sf_status knn_bandwidths(sf_index *idx, int k, uint32_t *d_nbr_orig, float *d_h_sorted,
                         cudaStream_t s) {
    Scratch sc(s);
    float *h = d_h_sorted ? d_h_sorted : sc.get<float>(idx->n);
    SF_TRY_SCRATCH(sc);
    SF_TRY(knn_run(idx, k, d_nbr_orig, h, s));
    const unsigned g = std::min<unsigned>(blocks_for(idx->n, 256), 152 * 16);
    SF_TRY_CUDA(launch(k_store_h, dim3(g), dim3(256), 0, s, (const float *)h, idx->n, idx->pos));
    SF_TRY(build_node_ell(idx, BW_ISO, nullptr, nullptr, idx->nell, s));
    return SF_OK;
}

sf_status knn_neighbours(sf_index *idx, int k, uint32_t *d_nbr_orig, float *d_h_orig,
                         cudaStream_t s) {
    Scratch sc(s);
    float *h = sc.get<float>(idx->n);
    SF_TRY_SCRATCH(sc);
    SF_TRY(knn_run(idx, k, d_nbr_orig, h, s));
    if (d_h_orig) {
        const unsigned g = std::min<unsigned>(blocks_for(idx->n, 256), 152 * 16);
        SF_TRY_CUDA(launch(k_scatter_f, dim3(g), dim3(256), 0, s, (const float *)h,
                           (const uint32_t *)idx->perm, idx->n, d_h_orig));
    }
    return SF_OK;
}

// The work of one kNN run (the index's resident bandwidths are left as they are):
// h_counts[0] (lane, candidate) distance evaluations, [1] candidates staged per
// query leaf, summed over all passes, [2] query leaves. Synchronises the stream.
sf_status knn_work_counts(sf_index *idx, int k, int64_t *h_counts, cudaStream_t s) {
    Scratch sc(s);
    float *h = sc.get<float>(idx->n);
    unsigned long long *work = sc.get<unsigned long long>(2);
    int64_t *out = sc.get<int64_t>(3);
    SF_TRY_SCRATCH(sc);
    SF_TRY_CUDA(cudaMemsetAsync(work, 0, 2 * sizeof(unsigned long long), s));
    SF_TRY(knn_run(idx, k, nullptr, h, s, work));
    SF_TRY_CUDA(launch(k_knn_work_out, dim3(1), dim3(32), 0, s, (const unsigned long long *)work, out));
    SF_TRY_CUDA(cudaMemcpyAsync(h_counts, out, 3 * sizeof(int64_t), cudaMemcpyDeviceToHost, s));
    SF_TRY_CUDA(cudaStreamSynchronize(s));
    return SF_OK;
}

sf_status scatter_bandwidths(const sf_index *idx, float *d_h_orig, cudaStream_t s) {
    const unsigned g = std::min<unsigned>(blocks_for(idx->n, 256), 152 * 16);
    SF_TRY_CUDA(launch(k_scatter_h, dim3(g), dim3(256), 0, s, (const float4 *)idx->pos,
                       (const uint32_t *)idx->perm, idx->n, d_h_orig));
    return SF_OK;
}

}  // namespace sf

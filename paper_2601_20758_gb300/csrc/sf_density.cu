// sf_density.cu -- the gather engine: kernel density at grid nodes and at points.
//
// What is computed (Sec. 3.1, Eq. 7; gather formulation of Sec. 3.2.1):
//   rho(r) = inv_neff * sum_j K(r - y_j ; l_j)
// over the particles of the scope, with K the Epanechnikov (Eq. 4) or the
// truncated Gaussian kernel and l_j the per-particle smoothing lengths. Every
// output is written by exactly one thread, in a fixed summation order: no
// atomics, results are deterministic.
//
// Grid, split pipeline (sf_kde_grid, batches): the ROI's nodes are cut into
// 8 x 4 x Z tiles, one warp each. A walk kernel lists every tile's candidate
// leaves (leaves whose support reaches the tile); the lists are cut into work
// items of similar length; persistent warps drain the items, each lane owning
// one (x, y) column of Z nodes in registers. Per candidate leaf the warp
// refines its points (footprint in the tile, ROI clip) and stages them in its
// own shared memory; 32 at a time, across leaves, get per-axis tables of the
// kernel factors at the tile's node coordinates, so the inner loop per (point,
// node) pair is two instructions (Gaussian: exp(a+b+c) = e^a e^b e^c with the
// truncation test on q_x + q_y < 9 - q_z) or three (Epanechnikov), and half of
// one for the points whose support covers the whole tile. A tile of one item is
// written by the work kernel; a last kernel adds the partials of the others in
// item order (deterministic). The allocation-free entry point
// keeps the older monolithic form: one CTA per 16 x 16 x 8 tile walking and
// summing in one launch.
//
// Points: one warp per leaf of 32 query points; the warp walks the index for
// leaves whose support reaches the query points' box, stages the candidates
// in a shared-memory ring and every lane sums over them for its own point,
// two candidates per instruction (packed FP32x2 arithmetic).
#include <cmath>
#include <vector>

#include "sf_internal.cuh"

namespace sf {

constexpr float kBig = 1.0e30f;
constexpr int kTileX = 16, kTileY = 16, kTileZ = 8;
constexpr int kGridThreads = 256;
constexpr int kStage = 128;       // staged points per chunk (4 leaves)
constexpr int kBatch = 64;        // candidate leaves per traversal batch
constexpr int kStack = 32 * kMaxLevels;
constexpr float kHalfLog2e = 0.72134752044448170368f;  // log2(e) / 2

__device__ __forceinline__ float ex2_approx(float x) {
    float y;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}


// Kernel-specific constants, in the units of q' used on the device:
//   EPAN : q' = sum (d_k / l_k)^2,           support q' < 1,  weight c (1 - q')
//   GAUSS: q' = sum (d_k / l_k)^2 log2(e)/2, support q' < 9 log2(e)/2, weight c 2^-q'
template <int KER>
struct KDef;
template <>
struct KDef<SF_K_EPAN> {
    static constexpr float qmax = 1.0f;   // in q'
    static constexpr float rmul = 1.0f;   // support radius / l
    static constexpr float uscale = 1.0f; // u_k = uscale / l_k
};
template <>
struct KDef<SF_K_GAUSS3> {
    static constexpr float qmax = 9.0f * kHalfLog2e;
    static constexpr float rmul = 3.0f;
    static constexpr float uscale = 0.84932180028801904272f;  // sqrt(log2(e)/2)
};

struct EngineArgs {
    TreeView tv;
    const float4 *ell;       // BW_ANISO per sorted point
    const float4 *nell;      // node max smoothing lengths (BW_ISO / BW_ANISO)
    const DensityParams *dp; // device params (uniform l, inv_neff)
    float cnorm;             // 15/(8 pi) or 1/((2 pi)^1.5 P3)
    float blo[3], bhi[3];    // clip box, float bounds equivalent to the closed double box
};

// Does node i possibly hold a particle whose support reaches the box [wlo, whi]?
// Conservative: the box comes widened by widen_box (a margin covering float
// rounding of the box), and the squared-support test carries kFilterSlack.
struct NodeBox {
    float4 lo, hi;
    float e[3];  // largest smoothing lengths
};
template <int BW>
__device__ __forceinline__ NodeBox node_box(const EngineArgs &a, const float *uni, int64_t i) {
    NodeBox b;
    b.lo = __ldg(&a.tv.nlo[i]);
    b.hi = __ldg(&a.tv.nhi[i]);
    if (BW == BW_UNIFORM) {
        b.e[0] = uni[0];
        b.e[1] = uni[1];
        b.e[2] = uni[2];
    } else {
        const float4 ne = __ldg(&a.nell[i]);
        b.e[0] = ne.x;
        b.e[1] = ne.y;
        b.e[2] = ne.z;
    }
    return b;
}
template <int KER, bool CLIP>
__device__ __forceinline__ bool box_reaches(const EngineArgs &a, const NodeBox &b, const float wlo[3],
                                            const float whi[3]) {
    if (!(b.e[0] > 0.f) || !(b.e[1] > 0.f) || !(b.e[2] > 0.f)) return false;
    bool ok = true;
    if (CLIP)
        ok = !(b.lo.x > a.bhi[0] || b.hi.x < a.blo[0] || b.lo.y > a.bhi[1] || b.hi.y < a.blo[1] ||
                    b.lo.z > a.bhi[2] || b.hi.z < a.blo[2]);
    const float nl[3] = {b.lo.x, b.lo.y, b.lo.z}, nh[3] = {b.hi.x, b.hi.y, b.hi.z};
    float q = 0.f;
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        const float gap = fmaxf(fmaxf(nl[k] - whi[k], wlo[k] - nh[k]), 0.f);
        const float t = gap * rcp_approx(b.e[k]);
        q = fmaf(t, t, q);
    }
    return ok && (q < KDef<KER>::rmul * KDef<KER>::rmul * (1.0f + kFilterSlack));
}
template <int KER, int BW, bool CLIP>
__device__ __forceinline__ bool node_reaches(const EngineArgs &a, const float *uni, int64_t i,
                                             const float wlo[3], const float whi[3]) {
    return box_reaches<KER, CLIP>(a, node_box<BW>(a, uni, i), wlo, whi);
}

// Warp-cooperative resumable depth-first walk. Emits accepted leaf indices in
// ascending order into out[0..), stopping once fewer than 32 slots remain.
// Stack entries encode (level << 27) | index-in-level; sp is warp-uniform.
// (Expanding up to four parents of leaves at once took longer: most runs of them on the
// stack are shorter, and the four tests are issued all the same.)
template <typename Test>
__device__ int warp_walk(const TreeView &tv, const Test &test, int *stack, int &sp, int *out,
                         int cap) {
    const int lane = threadIdx.x & 31;
    const unsigned lt = (1u << lane) - 1u;
    int nout = 0;
    while (sp > 0 && nout <= cap - 32) {
        const int e = stack[sp - 1];
        __syncwarp();
        sp -= 1;
        const int cl = (e >> 27) - 1;
        const int64_t c = (int64_t)(e & ((1 << 27) - 1)) * kFanout + lane;
        const bool ok = (c < tv.cnt[cl]) && test(tv.off[cl] + c);
        const unsigned m = __ballot_sync(0xffffffffu, ok);
        const int r = __popc(m & lt), k = __popc(m);
        if (cl == 0) {
            if (ok) out[nout + r] = (int)c;
            nout += k;
        } else {
            if (ok) stack[sp + (k - 1 - r)] = (cl << 27) | (int)c;
            sp += k;
        }
        __syncwarp();
    }
    return nout;
}

// Start a walk: test the root (lane 0) and push it, or emit it if it is a leaf.
template <typename Test>
__device__ int warp_walk_start(const TreeView &tv, const Test &test, int *stack, int &sp,
                               int *out) {
    const int lane = threadIdx.x & 31;
    const int top = tv.nlevels - 1;
    const bool ok = __shfl_sync(0xffffffffu, lane == 0 ? (int)test(tv.off[top]) : 0, 0) != 0;
    sp = 0;
    if (!ok) return 0;
    if (top == 0) {
        if (lane == 0) out[0] = 0;
        __syncwarp();
        return 1;
    }
    if (lane == 0) stack[0] = top << 27;
    __syncwarp();
    sp = 1;
    return 0;
}

// Exact float bounds of a closed double box: x >= lo_f <=> (double)x >= lo.
void float_bounds(const double lo[3], const double hi[3], float flo[3], float fhi[3]) {
    for (int k = 0; k < 3; ++k) {
        float a = (float)lo[k];
        if ((double)a < lo[k]) a = nextafterf(a, INFINITY);
        float b = (float)hi[k];
        if ((double)b > hi[k]) b = nextafterf(b, -INFINITY);
        flo[k] = a;
        fhi[k] = b;
    }
}

// Per-point smoothing lengths for the three bandwidth modes.
template <int BW>
__device__ __forceinline__ void point_ell(const EngineArgs &a, const float *uni, int64_t i,
                                          float4 p, float l[3]) {
    if (BW == BW_ISO) {
        l[0] = l[1] = l[2] = p.w;
    } else if (BW == BW_UNIFORM) {
        l[0] = uni[0];
        l[1] = uni[1];
        l[2] = uni[2];
    } else {
        const float4 e = __ldg(&a.ell[i]);
        l[0] = e.x;
        l[1] = e.y;
        l[2] = e.z;
    }
}

// ===========================================================================
// Grid
// ===========================================================================
// Geometry and outputs of one ROI grid (device-side descriptor).
struct RoiDesc {
    const float2 *axis;  // node coordinates as (hi, lo) float pairs: x[nx], y[ny], z[nz]
    int nx, ny, nz;
    int tiles_x, tiles_y, tiles_z;
    int tile_base;       // first global tile index of this ROI
    int group_base;      // first global group of tiles (see MrArgs::gx)
    int groups_x, groups_y;
    float *out;          // dims[2] x dims[1] x dims[0], x fastest
    double *mass_part;   // per tile of this ROI
    const DensityParams *dp;
    float blo[3], bhi[3];  // clip box (float bounds of the closed double box)
};

template <int TZ>
struct GridSmemT {
    float2 tx[kStage][kTileX];   // Gauss: (c e^{-qx'}, qx'); Epan: (qx', -)
    float2 ty[kStage][kTileY];   // Gauss: (e^{-qy'}, qy');   Epan: (qy', -)
    float2 tz[kStage][TZ];       // Gauss: (e^{-qz'}, qmax - qz'); Epan: (c (1 - qz'), -)
    float4 sp[kStage];           // staged (x, y, z, c)
    float4 su[kStage];           // staged (u_x, u_y, u_z, -)
    int2 sf[kStage];             // staged footprint: x0|x1<<8|y0<<16|y1<<24, z0|z1<<8
    float2 axt[kTileX + kTileY + TZ];  // the tile's node coordinates
    uint8_t wlist[kGridThreads / 32][kStage];  // per warp: staged candidates touching its rows
    int stack[kStack];
    int leaves[kBatch];
    int wcnt[kGridThreads / 32];
    int nleaves, sp_top, item;
    float uni[3];
    double inv_neff;
    double red[kGridThreads / 32];
    EngineArgs e;                // the call's engine arguments with this ROI's clip box and params
    RoiDesc roi;
};

struct TileGeom {
    int gx0, gy0, gz0;
    int nv[3];
    float tlo[3], thi[3], sp3[3];
};

template <int TZ, int WX = kTileX, int WY = kTileY>
__device__ __forceinline__ void tile_origin(const RoiDesc &r, int tile, int &gx0, int &gy0, int &gz0,
                                            int nv[3]) {
    const int tix = tile % r.tiles_x, tiy = (tile / r.tiles_x) % r.tiles_y,
              tiz = tile / (r.tiles_x * r.tiles_y);
    gx0 = tix * WX;
    gy0 = tiy * WY;
    gz0 = tiz * TZ;
    nv[0] = min(WX, r.nx - gx0);
    nv[1] = min(WY, r.ny - gy0);
    nv[2] = min(TZ, r.nz - gz0);
}

// The tile's node coordinates and the call's parameters into shared memory
// (S.roi and S.e must be set). Block-wide: it contains a barrier.
template <int TZ>
__device__ TileGeom tile_setup(GridSmemT<TZ> &S, int tile) {
    const int tid = threadIdx.x;
    const RoiDesc &r = S.roi;
    TileGeom g;
    tile_origin<TZ>(r, tile, g.gx0, g.gy0, g.gz0, g.nv);
    if (tid < kTileX + kTileY + TZ) {
        float2 v = make_float2(0.f, 0.f);
        if (tid < kTileX) {
            if (tid < g.nv[0]) v = r.axis[g.gx0 + tid];
        } else if (tid < kTileX + kTileY) {
            const int j = tid - kTileX;
            if (j < g.nv[1]) v = r.axis[r.nx + g.gy0 + j];
        } else {
            const int j = tid - kTileX - kTileY;
            if (j < g.nv[2]) v = r.axis[r.nx + r.ny + g.gz0 + j];
        }
        S.axt[tid] = v;
    }
    if (tid == 0) {
        const DensityParams dp = *S.e.dp;
        S.uni[0] = dp.ell_uniform[0];
        S.uni[1] = dp.ell_uniform[1];
        S.uni[2] = dp.ell_uniform[2];
        S.inv_neff = dp.inv_neff;
    }
    __syncthreads();
    const int off[3] = {0, kTileX, kTileX + kTileY};
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        g.tlo[k] = S.axt[off[k]].x;
        g.thi[k] = S.axt[off[k] + g.nv[k] - 1].x;
        // node spacing, for footprints (approximate; footprints are widened by 1)
        g.sp3[k] = g.nv[k] > 1 ? (S.axt[off[k] + 1].x - S.axt[off[k]].x) : 1.f;
    }
    return g;
}

// One chunk: the points of up to four candidate leaves are refined (support
// footprint inside the tile, ROI clip), staged, tabulated per axis and added
// into acc. Block-wide; ends with a barrier so shared memory can be reused.
template <int KER, int BW, bool CLIP, bool CNT, int TZ>
__device__ void grid_chunk(GridSmemT<TZ> &S, const TileGeom &g, const int *leaves, int nl,
                           float acc[TZ], unsigned long long &npairs) {
    const EngineArgs &E = S.e;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int cx = lane & 15, cy = warp * 2 + (lane >> 4);
    // ---- load and refine up to 128 candidate points (threads 0..127)
    bool acc_pt = false;
    float4 p = make_float4(0.f, 0.f, 0.f, 0.f);
    float l[3] = {0.f, 0.f, 0.f};
    int2 fp = make_int2(0, 0);
    if (tid < kStage) {
        const int li = tid >> 5;
        if (li < nl) {
            const int64_t i = (int64_t)leaves[li] * kLeaf + lane;
            if (i < E.tv.n) {
                p = __ldg(&E.tv.pos[i]);
                point_ell<BW>(E, S.uni, i, p, l);
                acc_pt = l[0] > 0.f && l[1] > 0.f && l[2] > 0.f;
                if (CLIP)
                    acc_pt = acc_pt && p.x >= E.blo[0] && p.x <= E.bhi[0] && p.y >= E.blo[1] &&
                             p.y <= E.bhi[1] && p.z >= E.blo[2] && p.z <= E.bhi[2];
                const float pc[3] = {p.x, p.y, p.z};
                int f0[3], f1[3];
                float qlb = 0.f;
#pragma unroll
                for (int k = 0; k < 3; ++k) {
                    const float R = l[k] * KDef<KER>::rmul;
                    if (g.sp3[k] > 0.f) {
                        const float a0 = fminf(fmaxf(ceilf((pc[k] - R - g.tlo[k]) / g.sp3[k]) - 1.f, -1.f), 64.f);
                        const float a1 = fminf(fmaxf(floorf((pc[k] + R - g.tlo[k]) / g.sp3[k]) + 1.f, -1.f), 64.f);
                        f0[k] = max(0, (int)a0);
                        f1[k] = min(g.nv[k] - 1, (int)a1);
                    } else {
                        f0[k] = 0;
                        f1[k] = g.nv[k] - 1;
                    }
                    if (f0[k] > f1[k]) acc_pt = false;
                    float gap = fmaxf(fmaxf(g.tlo[k] - pc[k], pc[k] - g.thi[k]), 0.f);
                    gap = fmaxf(gap - 1.0e-6f * (fabsf(g.tlo[k]) + fabsf(g.thi[k])), 0.f);
                    const float t = gap / R;
                    qlb += t * t;
                }
                if (!(qlb < 1.0f + 1.0e-5f)) acc_pt = false;
                if (acc_pt) {
                    fp.x = f0[0] | (f1[0] << 8) | (f0[1] << 16) | (f1[1] << 24);
                    fp.y = f0[2] | (f1[2] << 8);
                }
            }
        }
    }
    // ---- compact accepted points (stable: leaf order, then lane order)
    const unsigned bal = __ballot_sync(0xffffffffu, acc_pt);
    if (lane == 0) S.wcnt[warp] = __popc(bal);
    __syncthreads();
    int base = 0, ns = 0;
#pragma unroll
    for (int w = 0; w < kStage / 32; ++w) {
        const int c = S.wcnt[w];
        if (w < warp) base += c;
        ns += c;
    }
    if (acc_pt) {
        const int s = base + __popc(bal & ((1u << lane) - 1u));
        const float c = E.cnorm / ((l[0] * l[1]) * l[2]);
        S.sp[s] = make_float4(p.x, p.y, p.z, c);
        S.su[s] = make_float4(KDef<KER>::uscale / l[0], KDef<KER>::uscale / l[1],
                              KDef<KER>::uscale / l[2], 0.f);
        S.sf[s] = fp;
    }
    __syncthreads();
    // ---- per-warp lists: the staged candidates whose rows reach this warp's rows
    {
        int nw = 0;
        for (int g0 = 0; g0 < ns; g0 += 32) {
            const int sidx = g0 + lane;
            bool hit = false;
            if (sidx < ns) {
                const int fx = S.sf[sidx].x;
                const int y0 = (fx >> 16) & 255, y1 = (fx >> 24) & 255;
                hit = !(warp * 2 + 1 < y0 || warp * 2 > y1);
            }
            const unsigned m = __ballot_sync(0xffffffffu, hit);
            if (hit) S.wlist[warp][nw + __popc(m & ((1u << lane) - 1u))] = (uint8_t)sidx;
            nw += __popc(m);
        }
        __syncwarp();
        if (lane == 0) S.wcnt[warp] = nw;
    }
    // ---- per-axis tables: the entries inside each staged point's footprint
    constexpr int kEnt = kTileX + kTileY + TZ;
    for (int e = tid; e < ns * kEnt; e += kGridThreads) {
        const int s = e / kEnt;
        const int j = e - s * kEnt;
        const int2 F = S.sf[s];
        int axis, i, lo_i, hi_i;
        if (j < kTileX) {
            axis = 0; i = j; lo_i = F.x & 255; hi_i = (F.x >> 8) & 255;
        } else if (j < kTileX + kTileY) {
            axis = 1; i = j - kTileX; lo_i = (F.x >> 16) & 255; hi_i = (F.x >> 24) & 255;
        } else {
            axis = 2; i = j - kTileX - kTileY; lo_i = F.y & 255; hi_i = (F.y >> 8) & 255;
        }
        if (i < lo_i || i > hi_i) continue;  // never read by the accumulation
        const float4 P = S.sp[s];
        const float4 U = S.su[s];
        const float pc = axis == 0 ? P.x : (axis == 1 ? P.y : P.z);
        const float u = axis == 0 ? U.x : (axis == 1 ? U.y : U.z);
        const float2 nc = S.axt[j];
        const float d = (nc.x - pc) + nc.y;
        const float t = d * u;
        const float q = t * t;
        const bool sup = q < KDef<KER>::qmax;
        float2 v;
        if (KER == SF_K_GAUSS3) {
            const float w = sup ? ex2_approx(-q) : 0.f;
            if (axis == 0) v = make_float2(w * P.w, sup ? q : kBig);
            else if (axis == 1) v = make_float2(w, sup ? q : kBig);
            else v = make_float2(w, sup ? KDef<KER>::qmax - q : -1.f);
        } else {
            if (axis < 2) v = make_float2(sup ? q : kBig, 0.f);
            else v = make_float2(sup ? P.w * (1.0f - q) : -kBig, 0.f);
        }
        if (axis == 0) S.tx[s][i] = v;
        else if (axis == 1) S.ty[s][i] = v;
        else S.tz[s][i] = v;
    }
    __syncthreads();
    // ---- accumulate: warp owns rows 2w, 2w+1; lane owns column cx
    const int nw = S.wcnt[warp];
    for (int li = 0; li < nw; ++li) {
        const int s = S.wlist[warp][li];
        const int2 F = S.sf[s];
        const int x0 = F.x & 255, x1 = (F.x >> 8) & 255;
        const int y0 = (F.x >> 16) & 255, y1 = (F.x >> 24) & 255;
        const int z0 = F.y & 255, z1 = (F.y >> 8) & 255;
        const bool in = cx >= x0 && cx <= x1 && cy >= y0 && cy <= y1;
        // outside the footprint: no contribution (Gauss: q = BIG; Epan: q in .x = BIG)
        float2 ex = KER == SF_K_GAUSS3 ? make_float2(0.f, kBig) : make_float2(kBig, 0.f);
        float2 ey = ex;
        if (in) {
            ex = S.tx[s][cx];
            ey = S.ty[s][cy];
        }
        if (KER == SF_K_GAUSS3) {
            const float bse = ex.x * ey.x;
            const float qij = ex.y + ey.y;
#pragma unroll
            for (int k = 0; k < TZ; ++k) {
                if (k >= z0 && k <= z1) {
                    const float2 ez = S.tz[s][k];
                    if (qij < ez.y) {
                        acc[k] = fmaf(bse, ez.x, acc[k]);
                        if (CNT) ++npairs;
                    }
                }
            }
        } else {
            const float b = S.sp[s].w * (ex.x + ey.x);
#pragma unroll
            for (int k = 0; k < TZ; ++k) {
                if (k >= z0 && k <= z1) {
                    const float t = S.tz[s][k].x - b;
                    acc[k] += fmaxf(t, 0.f);
                    if (CNT) npairs += (t > 0.f);
                }
            }
        }
    }
    __syncthreads();
}

// Fold a chunk's FP32 sums into the compensated per-voxel sums (TwoSum).
template <int TZ>
__device__ __forceinline__ void fold(float acc[TZ], float sum[TZ], float cmp[TZ]) {
#pragma unroll
    for (int k = 0; k < TZ; ++k) {
        const float t = sum[k] + acc[k];
        const float bp = t - sum[k];
        cmp[k] += (sum[k] - (t - bp)) + (acc[k] - bp);
        sum[k] = t;
        acc[k] = 0.f;
    }
}

__device__ __forceinline__ void count_pairs_out(unsigned long long *dst, unsigned long long npairs) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) npairs += __shfl_xor_sync(0xffffffffu, npairs, o);
    if ((threadIdx.x & 31) == 0 && npairs) atomicAdd(dst, npairs);
}

// EngineArgs of one ROI: the call's common arguments with the ROI's params and clip box.
__device__ __forceinline__ void set_roi_engine(EngineArgs &e, const EngineArgs &common, const RoiDesc &r) {
    e = common;
    e.dp = r.dp;
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        e.blo[k] = r.blo[k];
        e.bhi[k] = r.bhi[k];
    }
}

// ---------------------------------------------------------------------------
// Monolithic variant (used by the allocation-free entry point): one CTA per
// tile walks the index for its tile and sums everything, 8 nodes deep in z.
// ---------------------------------------------------------------------------
struct GridArgs {
    EngineArgs e;
    RoiDesc roi;
    unsigned long long *pairs;
};

template <int KER, int BW, bool CLIP, bool CNT>
__global__ void __launch_bounds__(kGridThreads, 3) k_grid(GridArgs a) {
    constexpr int TZ = kTileZ;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    GridSmemT<TZ> &S = *reinterpret_cast<GridSmemT<TZ> *>(smem_raw);
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int tile = blockIdx.x;
    if (tid == 0) {
        S.e = a.e;
        S.roi = a.roi;
    }
    __syncthreads();
    const TileGeom g = tile_setup<TZ>(S, tile);
    float wlo[3], whi[3];
    widen_box(g.tlo, g.thi, wlo, whi);
    auto test = [&](int64_t node) { return node_reaches<KER, BW, CLIP>(S.e, S.uni, node, wlo, whi); };
    const int cx = lane & 15, cy = warp * 2 + (lane >> 4);
    unsigned long long npairs = 0;
    float acc[TZ], sum[TZ], cmp[TZ];
#pragma unroll
    for (int k = 0; k < TZ; ++k) acc[k] = sum[k] = cmp[k] = 0.f;

    if (warp == 0) {
        int spv;
        int n0 = warp_walk_start(S.e.tv, test, S.stack, spv, S.leaves);
        if (lane == 0) {
            S.sp_top = spv;
            S.nleaves = n0;
        }
    }
    __syncthreads();
    bool first = true;
    while (true) {
        if (warp == 0 && !(first && S.nleaves > 0)) {
            int spv = S.sp_top;
            int n = warp_walk(S.e.tv, test, S.stack, spv, S.leaves, kBatch);
            if (lane == 0) {
                S.sp_top = spv;
                S.nleaves = n;
            }
        }
        first = false;
        __syncthreads();
        const int nl = S.nleaves;
        const bool more = S.sp_top > 0;
        if (nl == 0 && !more) break;
        for (int cb = 0; cb < nl; cb += kStage / kLeaf) {
            grid_chunk<KER, BW, CLIP, CNT, TZ>(S, g, S.leaves + cb, min(kStage / kLeaf, nl - cb), acc,
                                               npairs);
            fold<TZ>(acc, sum, cmp);
        }
        if (!more) break;
    }
    if (CNT) count_pairs_out(a.pairs, (cx < g.nv[0] && cy < g.nv[1]) ? npairs : 0ull);
    // ---- write the tile and its mass
    double msum = 0.0;
    const double inv_neff = S.inv_neff;
    const RoiDesc &r = S.roi;
    if (cx < g.nv[0] && cy < g.nv[1]) {
        float *o = r.out + ((int64_t)g.gz0 * r.ny + (g.gy0 + cy)) * r.nx + (g.gx0 + cx);
        const int64_t zs = (int64_t)r.nx * r.ny;
#pragma unroll
        for (int k = 0; k < TZ; ++k) {
            if (k < g.nv[2]) {
                const double v = ((double)sum[k] + (double)cmp[k]) * inv_neff;
                const float fv = (float)v;
                o[k * zs] = fv;
                msum += (double)fv;
            }
        }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) msum += __shfl_xor_sync(0xffffffffu, msum, o);
    if (lane == 0) S.red[warp] = msum;
    __syncthreads();
    if (tid == 0) {
        double t = 0.0;
        for (int w = 0; w < kGridThreads / 32; ++w) t += S.red[w];
        r.mass_part[tile] = t;
    }
}

// ---------------------------------------------------------------------------
// Split pipeline over one or many ROIs. Tiles over dense regions hold far more
// candidates than others, so each (ROI, tile)'s candidate leaves are listed
// first and cut into balanced work items; persistent CTAs sum the items into
// per-item partial grids, and a per-tile reduction adds the partials in item
// order (deterministic). Global tile index = roi.tile_base + local tile.
// ---------------------------------------------------------------------------
struct MrArgs {
    EngineArgs e;               // common part (index, bandwidths, kernel constant)
    int prec;                   // SF_PREC_* of the work kernel (host-side choice)
    const RoiDesc *rois;        // device array
    const int *tile_roi;        // global tile -> ROI index (null: one ROI)
    int ntiles;
    // the walk takes groups of gx x gy x gz neighbouring tiles (1 or 2 per axis)
    const int *group_roi;       // global group -> ROI index (null: one ROI)
    int ngroups;
    int gx, gy, gz;
    unsigned long long *pairs;  // counting variant
    // count walk only (nullable): candidate leaves whose largest support radius on
    // every axis is below twice the ROI's node spacing (sizes the tile depth)
    unsigned long long *small_leaves = nullptr;
};

constexpr int kWalkWarps = 8;
constexpr int kWX = 8, kWY = 4;  // node tile of one warp in the split pipeline (x, y)

struct WalkWarpSmem {
    int stack[kStack];
    int leaves[kBatch];
    float4 tlo[8], thi[8];  // the group's tile boxes, widened (tlo.w: the tile's list offset as bits)
    EngineArgs e;
};

// One warp per group of up to 2 x 2 x 2 neighbouring tiles of an ROI: count (EMIT = false)
// or list (EMIT = true) each tile's candidate leaves. The index is walked once for the
// group's box; every leaf found is tested against the group's tiles, one leaf per lane.
// What bounds it: the latency of the walk's dependent loads. Per tile and one node at a
// time it took 0.41 ms (each of the two passes) for the 65,536 tiles of a 256^3 zoom of
// 67M points, 0.09 ms in groups of 8.
template <int KER, int BW, bool CLIP, bool EMIT, int TZ>
__global__ void __launch_bounds__(kWalkWarps * 32) k_mr_walk(MrArgs a, uint32_t *cnt,
                                                             const uint32_t *off, int *list) {
    __shared__ WalkWarpSmem W[kWalkWarps];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const unsigned lt = (1u << lane) - 1u;
    const int gg = blockIdx.x * kWalkWarps + warp;
    if (gg >= a.ngroups) return;
    WalkWarpSmem &S = W[warp];
    const RoiDesc &r = a.rois[a.group_roi ? a.group_roi[gg] : 0];
    if (lane == 0) set_roi_engine(S.e, a.e, r);
    const int lg = gg - r.group_base;
    const int t0[3] = {lg % r.groups_x * a.gx, (lg / r.groups_x) % r.groups_y * a.gy,
                       lg / (r.groups_x * r.groups_y) * a.gz};  // the group's first tile
    const int nt[3] = {min(a.gx, r.tiles_x - t0[0]), min(a.gy, r.tiles_y - t0[1]), min(a.gz, r.tiles_z - t0[2])};
    const int ntile = nt[0] * nt[1] * nt[2];
    // lane t < ntile: tile t of the group (x fastest) and its box
    const int tl = min(lane, ntile - 1);
    const int tix = t0[0] + tl % nt[0], tiy = t0[1] + (tl / nt[0]) % nt[1], tiz = t0[2] + tl / (nt[0] * nt[1]);
    const int local = (tiz * r.tiles_y + tiy) * r.tiles_x + tix, gt = r.tile_base + local;
    float wlo[3], whi[3];
    {
        int gx0, gy0, gz0, nv[3];
        tile_origin<TZ, kWX, kWY>(r, local, gx0, gy0, gz0, nv);
        const float tlo[3] = {r.axis[gx0].x, r.axis[r.nx + gy0].x, r.axis[r.nx + r.ny + gz0].x};
        const float thi[3] = {r.axis[gx0 + nv[0] - 1].x, r.axis[r.nx + gy0 + nv[1] - 1].x,
                              r.axis[r.nx + r.ny + gz0 + nv[2] - 1].x};
        widen_box(tlo, thi, wlo, whi);
    }
    if (lane < ntile) {
        S.tlo[lane] = make_float4(wlo[0], wlo[1], wlo[2], __uint_as_float(EMIT ? off[gt] : 0u));
        S.thi[lane] = make_float4(whi[0], whi[1], whi[2], 0.f);
    }
#pragma unroll
    for (int k = 0; k < 3; ++k)  // the group's box (lanes past the last tile repeat it)
#pragma unroll
        for (int o = 4; o > 0; o >>= 1) {
            wlo[k] = fminf(wlo[k], __shfl_xor_sync(0xffffffffu, wlo[k], o));
            whi[k] = fmaxf(whi[k], __shfl_xor_sync(0xffffffffu, whi[k], o));
        }
#pragma unroll
    for (int k = 0; k < 3; ++k) {  // as lanes 0..7 have it
        wlo[k] = __shfl_sync(0xffffffffu, wlo[k], 0);
        whi[k] = __shfl_sync(0xffffffffu, whi[k], 0);
    }
    __syncwarp();
    float uni[3] = {r.dp->ell_uniform[0], r.dp->ell_uniform[1], r.dp->ell_uniform[2]};
    auto test = [&](int64_t node) { return node_reaches<KER, BW, CLIP>(S.e, uni, node, wlo, whi); };
    int spv;
    int nl = warp_walk_start(S.e.tv, test, S.stack, spv, S.leaves);
    uint32_t mine = 0, nsmall = 0;  // lane t: leaves of tile t so far
    // the ROI's node spacing per axis (dims >= 2), for the small-support count
    const float sp[3] = {r.axis[1].x - r.axis[0].x, r.axis[r.nx + 1].x - r.axis[r.nx].x,
                         r.axis[r.nx + r.ny + 1].x - r.axis[r.nx + r.ny].x};
    const bool small = !EMIT && a.small_leaves;
    while (true) {
        if (nl == 0) {
            if (spv == 0) break;
            nl = warp_walk(S.e.tv, test, S.stack, spv, S.leaves, kBatch);
            if (nl == 0) break;
        }
        if (ntile == 1) {
            if (EMIT) {
                const uint32_t base = __float_as_uint(S.tlo[0].w) + __shfl_sync(0xffffffffu, mine, 0);
                for (int i = lane; i < nl; i += 32) list[base + i] = S.leaves[i];
            } else if (small) {
                for (int i0 = 0; i0 < nl; i0 += 32) {
                    bool sm = i0 + lane < nl;
                    if (sm) {
                        float e[3] = {uni[0], uni[1], uni[2]};
                        if (BW != BW_UNIFORM) {
                            const float4 ne = __ldg(&S.e.nell[S.e.tv.off[0] + S.leaves[i0 + lane]]);
                            e[0] = ne.x;
                            e[1] = ne.y;
                            e[2] = ne.z;
                        }
                        sm = KDef<KER>::rmul * e[0] < 2.f * sp[0] && KDef<KER>::rmul * e[1] < 2.f * sp[1] &&
                             KDef<KER>::rmul * e[2] < 2.f * sp[2];
                    }
                    nsmall += __popc(__ballot_sync(0xffffffffu, sm));
                }
            }
            mine += nl;
        } else {
            for (int i0 = 0; i0 < nl; i0 += 32) {
                const bool in = i0 + lane < nl;
                const int leaf = in ? S.leaves[i0 + lane] : 0;
                const NodeBox nb = node_box<BW>(S.e, uni, S.e.tv.off[0] + leaf);
                const bool sm = small && in && KDef<KER>::rmul * nb.e[0] < 2.f * sp[0] &&
                                KDef<KER>::rmul * nb.e[1] < 2.f * sp[1] && KDef<KER>::rmul * nb.e[2] < 2.f * sp[2];
                for (int t = 0; t < ntile; ++t) {
                    const float4 bl = S.tlo[t], bh = S.thi[t];
                    const float lo[3] = {bl.x, bl.y, bl.z}, hi[3] = {bh.x, bh.y, bh.z};
                    const bool ok = in && box_reaches<KER, CLIP>(S.e, nb, lo, hi);
                    const unsigned m = __ballot_sync(0xffffffffu, ok);
                    if (EMIT) {
                        const uint32_t at = __float_as_uint(bl.w) + __shfl_sync(0xffffffffu, mine, t);
                        if (ok) list[at + __popc(m & lt)] = leaf;
                    } else if (small) {
                        nsmall += __popc(__ballot_sync(0xffffffffu, ok && sm));
                    }
                    if (lane == t) mine += __popc(m);
                }
            }
        }
        __syncwarp();
        nl = 0;
    }
    if (!EMIT) {
        if (lane < ntile) cnt[gt] = mine;
        if (lane == 0 && small && nsmall) atomicAdd(a.small_leaves, (unsigned long long)nsmall);
    }
}

__global__ void k_total64(const uint32_t *__restrict__ cnt, int n, unsigned long long *out) {
    unsigned long long t = 0;
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) t += cnt[i];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
    if ((threadIdx.x & 31) == 0 && t) atomicAdd(out, t);
}

__global__ void k_grid_item_counts(const uint32_t *__restrict__ cnt, int ntiles, uint32_t lpw,
                                   uint32_t *__restrict__ ic) {
    const int t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t < ntiles) ic[t] = max(1u, (cnt[t] + lpw - 1) / lpw);
}

__global__ void k_grid_items(const uint32_t *__restrict__ cnt, const uint32_t *__restrict__ off,
                             const uint32_t *__restrict__ ic, const uint32_t *__restrict__ ioff,
                             int ntiles, uint32_t lpw, int4 *__restrict__ items) {
    const int t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= ntiles) return;
    const uint32_t n = cnt[t], b = off[t];
    for (uint32_t i = 0; i < ic[t]; ++i)
        items[ioff[t] + i] = make_int4(t, (int)(b + i * lpw), (int)(b + min(n, (i + 1) * lpw)), ic[t] == 1);
}

// ---- tensor-core sums of particles whose support covers the whole tile ------
// For such a particle every node (x, y, z) of the 8 x 4 x TZ tile is in support
// and its Gaussian term is the product tx[x] ty[y] tz[z] of its table entries,
// so the tile's sum over these particles is a matrix product:
//   rho[(x, y), z] += sum_s A[(x, y), s] B[s, z],  A = tx ty (32 x S),  B = tz (S x 8).
// It runs as mma.sync m16n8k8 (TF32) or m16n8k16 (BF16) blocks with FP32
// accumulators; 3xTF32 splits every operand into TF32 hi + lo parts and adds the
// three products hi*hi + hi*lo + lo*hi (about 2^-21 relative). These are the
// grid's precision variants; the FP32 path keeps every particle on the FP32
// pipes, which measured faster on this GPU than these mma.sync blocks.
__device__ __forceinline__ uint32_t tf32_of(float x) {
    uint32_t r;
    asm("cvt.rna.tf32.f32 %0, %1;" : "=r"(r) : "f"(x));
    return r;
}

__device__ __forceinline__ void mma_k8_tf32(float d[4], uint32_t a0, uint32_t a1, uint32_t a2,
                                            uint32_t a3, uint32_t b0, uint32_t b1) {
    asm volatile(
        "mma.sync.aligned.m16n8k8.row.col.f32.tf32.tf32.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, "
        "{%8,%9}, {%0,%1,%2,%3};"
        : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
        : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}

__device__ __forceinline__ void mma_k16_bf16(float d[4], uint32_t a0, uint32_t a1, uint32_t a2,
                                             uint32_t a3, uint32_t b0, uint32_t b1) {
    asm volatile(
        "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, "
        "{%8,%9}, {%0,%1,%2,%3};"
        : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
        : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}

// Two floats as a bf16 pair: `first` in the low half (the lower column / row index).
__device__ __forceinline__ uint32_t bf16x2_of(float first, float second) {
    uint32_t r;
    asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(r) : "f"(second), "f"(first));
    return r;
}

// A (x = g, y) (TF32 fragment values) times B; PREC 3XTF32 adds the three split products.
template <int PREC>
__device__ __forceinline__ void mma_k8(float d[4], float a0, float a1, float a2, float a3, float b0,
                                       float b1) {
    const uint32_t A0 = tf32_of(a0), A1 = tf32_of(a1), A2 = tf32_of(a2), A3 = tf32_of(a3);
    const uint32_t B0 = tf32_of(b0), B1 = tf32_of(b1);
    if (PREC != SF_PREC_3XTF32) {
        mma_k8_tf32(d, A0, A1, A2, A3, B0, B1);
        return;
    }
    const uint32_t L0 = tf32_of(a0 - __uint_as_float(A0)), L1 = tf32_of(a1 - __uint_as_float(A1));
    const uint32_t L2 = tf32_of(a2 - __uint_as_float(A2)), L3 = tf32_of(a3 - __uint_as_float(A3));
    const uint32_t M0 = tf32_of(b0 - __uint_as_float(B0)), M1 = tf32_of(b1 - __uint_as_float(B1));
    mma_k8_tf32(d, L0, L1, L2, L3, B0, B1);
    mma_k8_tf32(d, A0, A1, A2, A3, M0, M1);
    mma_k8_tf32(d, A0, A1, A2, A3, B0, B1);
}

// Shared memory of one warp of the split pipeline: its 8 x 4 x TZ node tile. Rows of the
// tables: the 32 staged particles being summed.
constexpr int kWRing = 2 * kLeaf;  // staged particles: two halves of 32
// x and y factors lie by groups of four particles, a node's four side by side, so that one
// 16-byte load fetches them; the groups' padding keeps the fill's stores (one particle a
// lane) off each other's banks.
constexpr int kGX = 4 * kWX + 4, kGY = 4 * kWY + 4;
template <int KER, int TZ, bool ANISO>
struct __align__(16) WTileSmem {
    float xq[kLeaf / 4][kGX], yq[kLeaf / 4][kGY];  // q'
    float xw[KER == SF_K_GAUSS3 ? kLeaf / 4 : 1][kGX];  // Gauss: c e^{-qx'}
    float yw[KER == SF_K_GAUSS3 ? kLeaf / 4 : 1][kGY];  // Gauss: e^{-qy'}
    float tzw[kLeaf][TZ];    // Gauss: e^{-qz'};          Epan: c (1 - qz')
    float tzl[KER == SF_K_GAUSS3 ? kLeaf : 1][TZ];  // Gauss: qmax - qz' (also the scratch of the tensor-core sums)
    float cs[KER == SF_K_GAUSS3 ? 4 : kLeaf];       // Epan: c
    float4 sp[kWRing];       // staged (x, y, z, h)
    float4 sl[ANISO ? kWRing : 1];  // and (l_x, l_y, l_z)
    float2 axt[kWX + kWY + TZ];     // node coordinates (past the grid's end: the last node's again)
    float uni[4];
    RoiDesc roi;
};
// four blocks of eight warps an SM
static_assert(sizeof(WTileSmem<SF_K_GAUSS3, kTileZ, false>) <= (228 * 1024 / 4 - 1024) / 8, "tile tables");

// Persistent warps: each takes (ROI, tile, leaf range) items from a counter and
// sums them into the item's partial grid. No block barriers: a warp owns its
// tile, its staging and its tables.
//
// What bounds it: issue slots and the ALU pipe, which every support test goes through. So
// candidates are staged across leaves and summed 32 at a time (every lane fills one
// particle's tables; one compensated fold per 32 particles, as for one full leaf), the
// particles whose support covers the tile come first and are summed without a test, two
// nodes an instruction (9 issue slots a particle and 256 nodes; 22 with the tests), and
// shared memory, which took 83% of its cycles when every particle's x and y factors were
// loaded by themselves, is read 16 bytes at a time (zoom below 1.92 -> 1.75 ms, 64 grids 30.8
// -> 28.2; the group loops unrolled further: 1.78 and 29.3). Work time (gaussian, kNN lengths)
// of a 256^3 zoom of 67M points, 70% of whose staged particles cover their tile, against one
// leaf staged at a time and every pair tested: 3.20 -> 1.75 ms; of its whole cube at 128^3
// (supports of about a spacing): 3.74 -> 2.56 ms; 192^3 in BF16: 1.34 -> 0.73 ms; 64 uneven
// grids: 48.8 -> 28.2 ms.
template <int KER, int BW, bool CLIP, bool CNT, int TZ, int PREC = SF_PREC_FP32>
__global__ void __launch_bounds__(kGridThreads, BW == BW_ANISO ? 3 : 4)
    k_mr_work(MrArgs a, const int4 *__restrict__ items, const uint32_t *__restrict__ n_items,
              const int *__restrict__ list, double *__restrict__ part, unsigned int *next) {
    // the tensor-core path of the precision variants: Gaussian, 8 nodes deep (the
    // B operand's 8 columns); the FP32 path sums every particle in FP32
    constexpr bool kMma = KER == SF_K_GAUSS3 && TZ == 8 && PREC != SF_PREC_FP32;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    typedef WTileSmem<KER, TZ, BW == BW_ANISO> Smem;
    Smem &S = reinterpret_cast<Smem *>(smem_raw)[warp];
    const int cx = lane & (kWX - 1), cy = lane / kWX;
    const unsigned lt = (1u << lane) - 1u;
    const uint32_t nitems = *n_items;
    unsigned long long npairs = 0;
    int cur_roi = -1;
    while (true) {
        unsigned int item = 0;
        if (lane == 0) item = atomicAdd(next, 1u);
        item = __shfl_sync(0xffffffffu, item, 0);
        if (item >= nitems) break;
        const int4 it = items[item];
        const int ri = a.tile_roi ? a.tile_roi[it.x] : 0;
        if (ri != cur_roi) {
            if (lane == 0) S.roi = a.rois[ri];
            cur_roi = ri;
            __syncwarp();
        }
        const EngineArgs &E = a.e;
        const RoiDesc &r = S.roi;
        // ---- the tile's node coordinates
        int gx0, gy0, gz0, nv[3];
        tile_origin<TZ, kWX, kWY>(r, it.x - r.tile_base, gx0, gy0, gz0, nv);
        if (lane < kWX + kWY + TZ) {
            float2 v;
            if (lane < kWX) v = r.axis[gx0 + min(lane, nv[0] - 1)];
            else if (lane < kWX + kWY) v = r.axis[r.nx + gy0 + min(lane - kWX, nv[1] - 1)];
            else v = r.axis[r.nx + r.ny + gz0 + min(lane - kWX - kWY, nv[2] - 1)];
            S.axt[lane] = v;
        }
        if (lane == 0) {
            S.uni[0] = r.dp->ell_uniform[0];
            S.uni[1] = r.dp->ell_uniform[1];
            S.uni[2] = r.dp->ell_uniform[2];
        }
        __syncwarp();
        float mcen[3], mhw[3];  // the tile box widened by the rounding margin, as centre and half-width
        // node spacing (of the float pairs: it may lie below the coordinates' float rounding); 0 on
        // all axes where the pairs themselves are too coarse to tell the nearest node from it
        float sp3[3];
        bool even = true;
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            const int off = k == 0 ? 0 : (k == 1 ? kWX : kWX + kWY);
            const float lo = S.axt[off].x, hi = S.axt[off + nv[k] - 1].x;
            sp3[k] = nv[k] > 1 ? (S.axt[off + 1].x - lo) + (S.axt[off + 1].y - S.axt[off].y) : 0.f;
            even = even && (nv[k] == 1 || sp3[k] > 0x1p-44f * fmaxf(fabsf(lo), fabsf(hi)));
            const float mg = 1.0e-6f * (fabsf(lo) + fabsf(hi));
            mcen[k] = 0.5f * ((lo - mg) + (hi + mg));
            mhw[k] = 0.5f * ((hi + mg) - (lo - mg));
        }
        if (!even) sp3[0] = sp3[1] = sp3[2] = 0.f;
        float acc[TZ], sum[TZ], cmp[TZ];
#pragma unroll
        for (int k = 0; k < TZ; ++k) acc[k] = sum[k] = cmp[k] = 0.f;
        unsigned long long np = 0;
        unsigned long long st_leaves = 0, st_staged = 0, st_full = 0;
        int head = 0, staged = 0;  // the ring: first staged particle, how many (warp-uniform)
        // the next candidate leaf's point is loaded one step ahead, its number two
        float4 pn = make_float4(0.f, 0.f, 0.f, 0.f);
        int64_t in = -1;
        auto load = [&](int leaf) {
            in = (int64_t)leaf * kLeaf + lane;
            if (in < E.tv.n) pn = __ldg(&E.tv.pos[in]);
        };
        int lnext = it.y + 1 < it.z ? list[it.y + 1] : 0;
        if (it.y < it.z) load(list[it.y]);
        for (int lb = it.y; lb < it.z || staged > 0; ++lb) {
            if (lb < it.z) {
                // ---- one candidate leaf: the points whose support reaches a node of the tile
                const int64_t i = in;
                const float4 p = pn;
                if (lb + 1 < it.z) {
                    load(lnext);
                    if (lb + 2 < it.z) lnext = list[lb + 2];
                }
                bool ok = false;
                float l[3] = {0.f, 0.f, 0.f};
                if (i < E.tv.n) {
                    point_ell<BW>(E, S.uni, i, p, l);
                    ok = l[0] > 0.f && l[1] > 0.f && l[2] > 0.f;
                    if (CLIP)
                        ok = ok && p.x >= r.blo[0] && p.x <= r.bhi[0] && p.y >= r.blo[1] &&
                             p.y <= r.bhi[1] && p.z >= r.blo[2] && p.z <= r.bhi[2];
                    const float pc[3] = {p.x, p.y, p.z};
                    float rl[3], qlb = 0.f;
                    bool small = false;
#pragma unroll
                    for (int k = 0; k < 3; ++k) {
                        rl[k] = BW == BW_ISO && k > 0 ? rl[0] : rcp_approx(l[k]);
                        const float t = fmaxf(fabsf(pc[k] - mcen[k]) - mhw[k], 0.f) * rl[k];
                        qlb = fmaf(t, t, qlb);
                        small = small || l[k] * KDef<KER>::rmul < sp3[k];
                    }
                    ok = ok && qlb < KDef<KER>::rmul * KDef<KER>::rmul * (1.0f + kFilterSlack);
                    // Supports below a node spacing may lie between the nodes: the smallest per-axis
                    // q (computed exactly as the tables compute it, at the nodes nearest the
                    // point) bounds every node's test (the float sums and differences are
                    // monotone): a particle that fails it adds nothing to any node of the
                    // tile (a dense cluster in a coarse grid's cell) and is not staged.
                    if (ok && small) {
                        float mq[3];
#pragma unroll
                        for (int k = 0; k < 3; ++k) {
                            const int off = k == 0 ? 0 : (k == 1 ? kWX : kWX + kWY);
                            const float u = KDef<KER>::uscale * rl[k];
                            const float at = sp3[k] > 0.f ? ((pc[k] - S.axt[off].x) - S.axt[off].y) / sp3[k] : 0.f;
                            const int ic = (int)rintf(fminf(fmaxf(at, 0.f), (float)(nv[k] - 1)));
                            float m = INFINITY;
#pragma unroll
                            for (int dd = -1; dd <= 1; ++dd) {
                                const float2 nc = S.axt[off + min(max(ic + dd, 0), nv[k] - 1)];
                                const float d = (nc.x - pc[k]) + nc.y;
                                const float t = d * u;
                                m = fminf(m, t * t);
                            }
                            mq[k] = m;
                        }
                        if (KER == SF_K_GAUSS3) {
                            ok = mq[0] + mq[1] < KDef<KER>::qmax - mq[2];
                        } else {
                            const float c = E.cnorm * ((rl[0] * rl[1]) * rl[2]);
                            ok = c * (1.0f - mq[2]) - c * (mq[0] + mq[1]) > 0.f;
                        }
                    }
                }
                const unsigned bal = __ballot_sync(0xffffffffu, ok);
                if (ok) {
                    const int s = (head + staged + __popc(bal & lt)) & (kWRing - 1);
                    S.sp[s] = p;
                    if (BW == BW_ANISO) S.sl[s] = make_float4(l[0], l[1], l[2], 0.f);
                }
                staged += __popc(bal);
                if (CNT && lane == 0 && bal) {
                    ++st_leaves;
                    st_staged += __popc(bal);
                }
                if (staged < kLeaf && lb + 1 < it.z) continue;  // warp-uniform
                if (staged == 0) continue;
            }
            // ---- tables of 32 staged particles (fewer only at the end), one particle a lane:
            // factors and q at the tile's nodes. A q past the support needs no mark: it
            // fails the test by itself (qx + qy < qmax - qz, every term non-negative).
            const int ns = min(staged, kLeaf);
            __syncwarp();
            bool full = false;  // the support covers every node of the tile
            // lanes past the last particle: one infinitely far, which adds nothing
            float c = 1.f, u[3] = {1.f, 1.f, 1.f};
            float4 p = make_float4(INFINITY, 0.f, 0.f, 0.f);
            if (lane < ns) {
                const int e = head + lane;
                p = S.sp[e];
                float l[3] = {p.w, p.w, p.w};
                if (BW == BW_UNIFORM) {
                    l[0] = S.uni[0]; l[1] = S.uni[1]; l[2] = S.uni[2];
                } else if (BW == BW_ANISO) {
                    const float4 q = S.sl[e];
                    l[0] = q.x; l[1] = q.y; l[2] = q.z;
                }
                float rl[3];
#pragma unroll
                for (int k = 0; k < 3; ++k) {
                    rl[k] = BW == BW_ISO && k > 0 ? rl[0] : rcp_approx(l[k]);
                    u[k] = KDef<KER>::uscale * rl[k];
                }
                c = E.cnorm * ((rl[0] * rl[1]) * rl[2]);
                // q is convex along each axis: its largest value is at an end node, and passing
                // the test with the per-axis maxima passes it at every node
                auto ends = [&](int off, int n, float pc, float uu) {
                    const float2 n0 = S.axt[off], n1 = S.axt[off + n - 1];
                    const float t0 = ((n0.x - pc) + n0.y) * uu, t1 = ((n1.x - pc) + n1.y) * uu;
                    return fmaxf(t0 * t0, t1 * t1);
                };
                const float mx = ends(0, kWX, p.x, u[0]);
                const float my = ends(kWX, kWY, p.y, u[1]);
                const float mz = ends(kWX + kWY, TZ, p.z, u[2]);
                if (KER == SF_K_GAUSS3) full = mx + my < KDef<KER>::qmax - mz;
                else full = c * (1.0f - mz) - c * (mx + my) > 0.f;
            }
            // rows: the full-coverage particles first, [0, nf); the others [nf, ns)
            const unsigned balf = __ballot_sync(0xffffffffu, full);
            const int nf = __popc(balf);
            if (CNT && lane == 0 && KER == SF_K_GAUSS3 && TZ == 8) st_full += nf;
            // some row is tested (warp-uniform): rows are taken by fours
            const bool tests = CNT || KER != SF_K_GAUSS3 || nf < ns || (ns & 3) != 0;
            {
                const int s = full ? __popc(balf & lt) : nf + __popc(~balf & lt);
                auto q_at = [&](float2 nc, float pc, float uu) {
                    const float t = ((nc.x - pc) + nc.y) * uu;
                    return t * t;
                };
                const int g = s >> 2, sl = s & 3;
                auto axis = [&](auto put, int off, int n, float pc, float uu) {  // nodes two at a time
#pragma unroll
                    for (int i = 0; i < n; i += 2) {
                        const float4 nc = *reinterpret_cast<const float4 *>(&S.axt[off + i]);
                        put(i, q_at(make_float2(nc.x, nc.y), pc, uu));
                        put(i + 1, q_at(make_float2(nc.z, nc.w), pc, uu));
                    }
                };
                axis([&](int i, float q) {
                    if (KER == SF_K_GAUSS3) S.xw[g][4 * i + sl] = ex2_approx(-q) * c;
                    if (tests) S.xq[g][4 * i + sl] = q;
                }, 0, kWX, p.x, u[0]);
                axis([&](int i, float q) {
                    if (KER == SF_K_GAUSS3) S.yw[g][4 * i + sl] = ex2_approx(-q);
                    if (tests) S.yq[g][4 * i + sl] = q;
                }, kWX, kWY, p.y, u[1]);
                // four nodes of z a step, in an order that starts by the row so that the lanes'
                // 16-byte stores spread over the banks
#pragma unroll
                for (int t = 0; t < TZ / 4; ++t) {
                    const int i = 4 * ((t + (s >> 2)) & (TZ / 4 - 1));
                    const float4 na = *reinterpret_cast<const float4 *>(&S.axt[kWX + kWY + i]);
                    const float4 nb = *reinterpret_cast<const float4 *>(&S.axt[kWX + kWY + i + 2]);
                    const float q0 = q_at(make_float2(na.x, na.y), p.z, u[2]), q1 = q_at(make_float2(na.z, na.w), p.z, u[2]);
                    const float q2 = q_at(make_float2(nb.x, nb.y), p.z, u[2]), q3 = q_at(make_float2(nb.z, nb.w), p.z, u[2]);
                    if (KER == SF_K_GAUSS3) {
                        *reinterpret_cast<float4 *>(&S.tzw[s][i]) =
                            make_float4(ex2_approx(-q0), ex2_approx(-q1), ex2_approx(-q2), ex2_approx(-q3));
                        constexpr float qm = KDef<KER>::qmax;
                        if (tests)
                            *reinterpret_cast<float4 *>(&S.tzl[s][i]) = make_float4(qm - q0, qm - q1, qm - q2, qm - q3);
                    } else {
                        *reinterpret_cast<float4 *>(&S.tzw[s][i]) =
                            make_float4(c * (1.0f - q0), c * (1.0f - q1), c * (1.0f - q2), c * (1.0f - q3));
                    }
                }
                if (KER != SF_K_GAUSS3) S.cs[s] = c;
            }
            __syncwarp();
            head ^= kLeaf;
            staged -= ns;
            // ---- accumulate: lane owns column (cx, cy) and TZ nodes in z; four rows at a time
            auto four = [](const float *q) { return *reinterpret_cast<const float4 *>(q); };
            const int gf = CNT || kMma ? 0 : nf >> 2;  // groups of full rows
            if (gf > 0) {
                f32x2 acc2[TZ / 2];
#pragma unroll
                for (int k = 0; k < TZ / 2; ++k) acc2[k] = f2_pack(acc[2 * k], acc[2 * k + 1]);
#pragma unroll 1
                for (int g = 0; g < gf; ++g) {
                    float bv[4];
                    if (KER == SF_K_GAUSS3) {
                        const float4 X = four(&S.xw[g][4 * cx]), Y = four(&S.yw[g][4 * cy]);
                        bv[0] = X.x * Y.x; bv[1] = X.y * Y.y; bv[2] = X.z * Y.z; bv[3] = X.w * Y.w;
                    } else {
                        const float4 X = four(&S.xq[g][4 * cx]), Y = four(&S.yq[g][4 * cy]), C = four(&S.cs[4 * g]);
                        bv[0] = C.x * (X.x + Y.x); bv[1] = C.y * (X.y + Y.y);
                        bv[2] = C.z * (X.z + Y.z); bv[3] = C.w * (X.w + Y.w);
                    }
#pragma unroll
                    for (int j = 0; j < 4; ++j) {
                        const f32x2 bb = f2_pack(bv[j], bv[j]);
#pragma unroll
                        for (int k = 0; k < TZ; k += 4) {
                            const ulonglong2 z = *reinterpret_cast<const ulonglong2 *>(&S.tzw[4 * g + j][k]);
                            if (KER == SF_K_GAUSS3) {
                                acc2[k / 2] = f2_fma(bb, z.x, acc2[k / 2]);
                                acc2[k / 2 + 1] = f2_fma(bb, z.y, acc2[k / 2 + 1]);
                            } else {
                                acc2[k / 2] = f2_add(acc2[k / 2], f2_sub(z.x, bb));
                                acc2[k / 2 + 1] = f2_add(acc2[k / 2 + 1], f2_sub(z.y, bb));
                            }
                        }
                    }
                }
#pragma unroll
                for (int k = 0; k < TZ / 2; ++k) f2_unpack(acc2[k], acc[2 * k], acc[2 * k + 1]);
            }
            // the groups from the first with a row that is not full (rows past the last particle
            // add nothing); with the tensor cores the full rows are theirs
#pragma unroll 1
            for (int g = kMma ? nf >> 2 : gf; 4 * g < ns; ++g) {
                const float4 X = four(&S.xq[g][4 * cx]), Y = four(&S.yq[g][4 * cy]);
                const float qv[4] = {X.x + Y.x, X.y + Y.y, X.z + Y.z, X.w + Y.w};
                float bv[4];
                if (KER == SF_K_GAUSS3) {
                    const float4 V = four(&S.xw[g][4 * cx]), W = four(&S.yw[g][4 * cy]);
                    bv[0] = V.x * W.x; bv[1] = V.y * W.y; bv[2] = V.z * W.z; bv[3] = V.w * W.w;
                } else {
                    const float4 C = four(&S.cs[4 * g]);
                    bv[0] = C.x * qv[0]; bv[1] = C.y * qv[1]; bv[2] = C.z * qv[2]; bv[3] = C.w * qv[3];
                }
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    if (kMma && 4 * g + j < nf) continue;
#pragma unroll
                    for (int k = 0; k < TZ; k += 4) {
                        const float4 w = four(&S.tzw[4 * g + j][k]);
                        const float wv[4] = {w.x, w.y, w.z, w.w};
                        if (KER == SF_K_GAUSS3) {
                            const float4 m = four(&S.tzl[4 * g + j][k]);
                            const float mv[4] = {m.x, m.y, m.z, m.w};
#pragma unroll
                            for (int i = 0; i < 4; ++i)
                                if (qv[j] < mv[i]) {
                                    acc[k + i] = fmaf(bv[j], wv[i], acc[k + i]);
                                    if (CNT && k + i < nv[2]) ++np;
                                }
                        } else {
#pragma unroll
                            for (int i = 0; i < 4; ++i) {
                                const float t = wv[i] - bv[j];
                                acc[k + i] += fmaxf(t, 0.f);
                                if (CNT && k + i < nv[2]) np += (t > 0.f);
                            }
                        }
                    }
                }
            }
            if (kMma && nf > 0) {  // warp-uniform: the full-coverage particles on the tensor cores
                const int gq = lane >> 2, tig = lane & 3;
                float d0[4] = {0.f, 0.f, 0.f, 0.f}, d1[4] = {0.f, 0.f, 0.f, 0.f};
                if (PREC == SF_PREC_BF16) {
                    for (int s0 = 0; s0 < nf; s0 += 16) {
                        float ax[4], ay[4][4], bz[4];  // particles s0 + 2 tig + {0, 1, 8, 9}
#pragma unroll
                        for (int e = 0; e < 4; ++e) {
                            const int sp = s0 + 2 * tig + (e & 1) + 8 * (e >> 1);
                            const bool v = sp < nf;
                            ax[e] = v ? S.xw[sp >> 2][4 * gq + (sp & 3)] : 0.f;
                            bz[e] = v ? S.tzw[sp][gq] : 0.f;
#pragma unroll
                            for (int y = 0; y < 4; ++y) ay[e][y] = v ? S.yw[sp >> 2][4 * y + (sp & 3)] : 0.f;
                        }
                        const uint32_t b0 = bf16x2_of(bz[0], bz[1]), b1 = bf16x2_of(bz[2], bz[3]);
#pragma unroll
                        for (int mb = 0; mb < 2; ++mb) {
                            float *d = mb ? d1 : d0;
                            const int y0 = 2 * mb, y1 = 2 * mb + 1;
                            mma_k16_bf16(d, bf16x2_of(ax[0] * ay[0][y0], ax[1] * ay[1][y0]),
                                         bf16x2_of(ax[0] * ay[0][y1], ax[1] * ay[1][y1]),
                                         bf16x2_of(ax[2] * ay[2][y0], ax[3] * ay[3][y0]),
                                         bf16x2_of(ax[2] * ay[2][y1], ax[3] * ay[3][y1]), b0, b1);
                        }
                    }
                } else {
                    for (int s0 = 0; s0 < nf; s0 += 8) {
                        const int sa = s0 + tig, sb = s0 + tig + 4;
                        const bool va = sa < nf, vb = sb < nf;
                        const float txa = va ? S.xw[sa >> 2][4 * gq + (sa & 3)] : 0.f, txb = vb ? S.xw[sb >> 2][4 * gq + (sb & 3)] : 0.f;
                        const float tza = va ? S.tzw[sa][gq] : 0.f, tzb = vb ? S.tzw[sb][gq] : 0.f;
#pragma unroll
                        for (int mb = 0; mb < 2; ++mb) {
                            const float ya0 = va ? S.yw[sa >> 2][8 * mb + (sa & 3)] : 0.f, ya1 = va ? S.yw[sa >> 2][8 * mb + 4 + (sa & 3)] : 0.f;
                            const float yb0 = vb ? S.yw[sb >> 2][8 * mb + (sb & 3)] : 0.f, yb1 = vb ? S.yw[sb >> 2][8 * mb + 4 + (sb & 3)] : 0.f;
                            mma_k8<PREC>(mb ? d1 : d0, txa * ya0, txa * ya1, txb * yb0, txb * yb1, tza, tzb);
                        }
                    }
                }
                // to the column owners: row r = x + 8 y of the product is lane r's column
                float *cb = reinterpret_cast<float *>(S.tzl);  // no longer read
                __syncwarp();
#pragma unroll
                for (int mb = 0; mb < 2; ++mb) {
                    const float *d = mb ? d1 : d0;
                    const int r0 = 16 * mb + gq;
                    cb[r0 * 8 + 2 * tig] = d[0];
                    cb[r0 * 8 + 2 * tig + 1] = d[1];
                    cb[(r0 + 8) * 8 + 2 * tig] = d[2];
                    cb[(r0 + 8) * 8 + 2 * tig + 1] = d[3];
                }
                __syncwarp();
#pragma unroll
                for (int k = 0; k < TZ; ++k) acc[k] += cb[lane * 8 + k];
            }
            __syncwarp();
            fold<TZ>(acc, sum, cmp);
        }
        if (CNT && cx < nv[0] && cy < nv[1]) npairs += np;
        if (CNT && lane == 0) {  // work accounting of the counting variant
            atomicAdd(a.pairs + 1, st_leaves);
            atomicAdd(a.pairs + 2, st_staged);
            atomicAdd(a.pairs + 3, st_full);
            atomicAdd(a.pairs + 4, st_staged * (kWX * kWY * TZ));
        }
        if (it.w) {  // the tile's only item: its grid values and mass, as k_mr_reduce writes them
            const double inv_neff = r.dp->inv_neff;
            double msum = 0.0;
            if (cx < nv[0] && cy < nv[1]) {
                float *o = r.out + ((int64_t)gz0 * r.ny + (gy0 + cy)) * r.nx + (gx0 + cx);
                const int64_t zs = (int64_t)r.nx * r.ny;
#pragma unroll
                for (int k = 0; k < TZ; ++k) {
                    if (k < nv[2]) {
                        const float fv = (float)(((double)sum[k] + (double)cmp[k]) * inv_neff);
                        o[k * zs] = fv;
                        msum += (double)fv;
                    }
                }
            }
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) msum += __shfl_xor_sync(0xffffffffu, msum, o);
            if (lane == 0) r.mass_part[it.x - r.tile_base] = msum;
            continue;
        }
        double *o = part + ((int64_t)item * 32 + lane) * TZ;
#pragma unroll
        for (int k = 0; k < TZ; ++k) o[k] = (double)sum[k] + (double)cmp[k];
    }
    if (CNT) count_pairs_out(a.pairs, npairs);
}

// One warp per (ROI, tile) of several items: sum their partial grids in item order,
// scale, write, and the tile's mass. (A single item's warp has written its tile itself:
// through the partial grids a 256^3 grid moved 0.27 GB each way, 0.18 ms to read. Having the
// warp of a tile's last item add the partial grids took the work kernel 10% longer on
// dense grids, for its registers.)
template <int TZ>
__global__ void __launch_bounds__(kGridThreads) k_mr_reduce(MrArgs a, const uint32_t *__restrict__ ic,
                                                            const uint32_t *__restrict__ ioff,
                                                            const double *__restrict__ part) {
    const int lane = threadIdx.x & 31;
    const int gt = blockIdx.x * (kGridThreads / 32) + (threadIdx.x >> 5);
    if (gt >= a.ntiles) return;
    const uint32_t ni = ic[gt];
    if (ni == 1) return;
    const int cx = lane & (kWX - 1), cy = lane / kWX;
    const RoiDesc &r = a.rois[a.tile_roi ? a.tile_roi[gt] : 0];
    const int tile = gt - r.tile_base;
    int gx0, gy0, gz0, nv[3];
    tile_origin<TZ, kWX, kWY>(r, tile, gx0, gy0, gz0, nv);
    const double inv_neff = r.dp->inv_neff;
    double v[TZ];
#pragma unroll
    for (int k = 0; k < TZ; ++k) v[k] = 0.0;
    const uint32_t i0 = ioff[gt];
    // A few tiles of a thousand items each: the loads in flight set the time (24^3 nodes of 4M
    // points: 185 us two items at a time, 109 now).
#pragma unroll(64 / TZ)
    for (uint32_t i = 0; i < ni; ++i) {
        const double2 *pp = reinterpret_cast<const double2 *>(part + ((int64_t)(i0 + i) * 32 + lane) * TZ);
#pragma unroll
        for (int k = 0; k < TZ / 2; ++k) {
            const double2 w = __ldg(&pp[k]);
            v[2 * k] += w.x;
            v[2 * k + 1] += w.y;
        }
    }
    double msum = 0.0;
    if (cx < nv[0] && cy < nv[1]) {
        float *o = r.out + ((int64_t)gz0 * r.ny + (gy0 + cy)) * r.nx + (gx0 + cx);
        const int64_t zs = (int64_t)r.nx * r.ny;
#pragma unroll
        for (int k = 0; k < TZ; ++k) {
            if (k < nv[2]) {
                const float fv = (float)(v[k] * inv_neff);
                o[k * zs] = fv;
                msum += (double)fv;
            }
        }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) msum += __shfl_xor_sync(0xffffffffu, msum, o);
    if (lane == 0) r.mass_part[tile] = msum;
}

__global__ void k_mass_final(const double *__restrict__ part, int64_t n, double cell,
                             double *out) {
    __shared__ double red[32];
    double t = 0.0;
    for (int64_t i = threadIdx.x; i < n; i += blockDim.x) t += part[i];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = t;
    __syncthreads();
    if (threadIdx.x == 0) {
        double s = 0.0;
        for (int w = 0; w < (int)(blockDim.x >> 5); ++w) s += red[w];
        *out = s * cell;
    }
}

// One block per ROI: its tiles' masses in order, times its cell volume.
__global__ void k_mr_mass(const RoiDesc *__restrict__ rois, const double *__restrict__ cells,
                          int nroi, double *__restrict__ mass) {
    __shared__ double red[32];
    const int ri = blockIdx.x;
    if (ri >= nroi) return;
    const RoiDesc &r = rois[ri];
    const int nt = r.tiles_x * r.tiles_y * r.tiles_z;
    double t = 0.0;
    for (int i = threadIdx.x; i < nt; i += blockDim.x) t += r.mass_part[i];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = t;
    __syncthreads();
    if (threadIdx.x == 0) {
        double s = 0.0;
        for (int w = 0; w < (int)(blockDim.x >> 5); ++w) s += red[w];
        mass[ri] = s * cells[ri];
    }
}

// ---- monolithic dispatch (allocation-free path) ----------------------------
template <int KER, int BW, bool CLIP, bool CNT>
static cudaError_t launch_grid_t(const GridArgs &a, unsigned tiles, cudaStream_t s) {
    const size_t smem = sizeof(GridSmemT<kTileZ>);
    static std::atomic<uint64_t> attr{0};
    cudaError_t e = smem_attr_once(k_grid<KER, BW, CLIP, CNT>, smem, attr);
    if (e != cudaSuccess) return e;
    KTimer t(CNT ? "k_grid_count" : "k_grid", s);
    return launch(k_grid<KER, BW, CLIP, CNT>, dim3(tiles), dim3(kGridThreads), smem, s, a);
}

template <int KER, int BW, bool CLIP>
static cudaError_t launch_grid(const GridArgs &a, unsigned tiles, cudaStream_t s) {
    return a.pairs ? launch_grid_t<KER, BW, CLIP, true>(a, tiles, s)
                   : launch_grid_t<KER, BW, CLIP, false>(a, tiles, s);
}

template <int KER>
static cudaError_t dispatch_grid(int bw, bool clip, const GridArgs &a, unsigned tiles,
                                 cudaStream_t s) {
    switch (bw * 2 + (clip ? 1 : 0)) {
        case BW_ISO * 2 + 0: return launch_grid<KER, BW_ISO, false>(a, tiles, s);
        case BW_ISO * 2 + 1: return launch_grid<KER, BW_ISO, true>(a, tiles, s);
        case BW_UNIFORM * 2 + 0: return launch_grid<KER, BW_UNIFORM, false>(a, tiles, s);
        case BW_UNIFORM * 2 + 1: return launch_grid<KER, BW_UNIFORM, true>(a, tiles, s);
        case BW_ANISO * 2 + 0: return launch_grid<KER, BW_ANISO, false>(a, tiles, s);
        default: return launch_grid<KER, BW_ANISO, true>(a, tiles, s);
    }
}

// ---- split pipeline ---------------------------------------------------------
// Sizing: count candidate leaves of every (ROI, tile); returns the total (syncs).
template <int KER, int BW, bool CLIP, int TZ>
// tot: 16 bytes -- [0] the 32-bit scan total, [1] the item count of mr_exec,
// bytes 8..15 the same total summed in 64 bits (guards the 32-bit offsets).
// h_small (with a.small_leaves set): the count of small-support candidate leaves.
static sf_status mr_count(const MrArgs &a, uint32_t *cnt, uint32_t *off, uint32_t *tot,
                          uint32_t *h_total, StatusPeek *peek, cudaStream_t s,
                          unsigned long long *h_small = nullptr) {
    const unsigned wb = blocks_for(a.ngroups, kWalkWarps);
    if (a.small_leaves) SF_TRY_CUDA(cudaMemsetAsync(a.small_leaves, 0, sizeof(unsigned long long), s));
    SF_TRY_CUDA(launch(k_mr_walk<KER, BW, CLIP, false, TZ>, dim3(wb), dim3(kWalkWarps * 32), 0, s, a,
                       cnt, (const uint32_t *)nullptr, (int *)nullptr));
    SF_TRY(scan_u32(cnt, off, a.ntiles, tot, s));
    unsigned long long *tot64 = reinterpret_cast<unsigned long long *>(tot + 2);
    SF_TRY_CUDA(cudaMemsetAsync(tot64, 0, sizeof(unsigned long long), s));
    SF_TRY_CUDA(launch(k_total64, dim3(std::min(blocks_for(a.ntiles, 256), 152u * 4u)), dim3(256), 0, s,
                       (const uint32_t *)cnt, a.ntiles, tot64));
    unsigned long long h64 = 0;
    SF_TRY_CUDA(cudaMemcpyAsync(&h64, tot64, sizeof h64, cudaMemcpyDeviceToHost, s));
    if (peek && peek->d_src)
        SF_TRY_CUDA(cudaMemcpyAsync(&peek->value, peek->d_src, sizeof(int), cudaMemcpyDeviceToHost, s));
    if (a.small_leaves && h_small)
        SF_TRY_CUDA(cudaMemcpyAsync(h_small, a.small_leaves, sizeof(unsigned long long),
                                    cudaMemcpyDeviceToHost, s));
    SF_TRY_CUDA(cudaStreamSynchronize(s));
    if (h64 > 0x7fffffffull)
        return fail(SF_ERR_CAPACITY, "grid candidate lists of %llu entries exceed 2^31; use fewer nodes or a smaller ROI",
                    h64);
    *h_total = (uint32_t)h64;
    return SF_OK;
}

template <int KER, int TZ, int BW>
static size_t mr_work_smem() {
    return sizeof(WTileSmem<KER, TZ, BW == BW_ANISO>) * (kGridThreads / 32);
}

template <int KER, int BW, bool CLIP, bool CNT, int TZ>
static sf_status mr_work_attr(int *per_sm) {
    const size_t smem = mr_work_smem<KER, TZ, BW>();
    static std::atomic<uint64_t> attr{0};
    SF_TRY_CUDA(smem_attr_once(k_mr_work<KER, BW, CLIP, CNT, TZ>, smem, attr));
    SF_TRY_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(per_sm, k_mr_work<KER, BW, CLIP, CNT, TZ>,
                                                              kGridThreads, smem));
    if (*per_sm < 1) *per_sm = 1;
    return SF_OK;
}

// Buffers of the execution phase, sized from the count.
struct MrBuffers {
    uint32_t *cnt, *off, *tot, *ic, *ioff;
    int *list;
    int4 *items;
    double *part;
    unsigned int *next;
    uint32_t lpw;
    int64_t slots;        // resident blocks of k_mr_work
};

template <int KER, int BW, bool CLIP, bool CNT, int TZ, int PREC>
static sf_status launch_work(const MrArgs &a, const MrBuffers &b, cudaStream_t s) {
    static std::atomic<uint64_t> attr{0};
    SF_TRY_CUDA(smem_attr_once(k_mr_work<KER, BW, CLIP, CNT, TZ, PREC>, mr_work_smem<KER, TZ, BW>(), attr));
    SF_TRY_CUDA(launch(k_mr_work<KER, BW, CLIP, CNT, TZ, PREC>, dim3((unsigned)b.slots), dim3(kGridThreads),
                       mr_work_smem<KER, TZ, BW>(), s, a, (const int4 *)b.items, (const uint32_t *)(b.tot + 1),
                       (const int *)b.list, b.part, b.next));
    return SF_OK;
}

// Execution: list, items, persistent work, ordered reduce (no host sync; capturable).
template <int KER, int BW, bool CLIP, bool CNT, int TZ>
static sf_status mr_exec(const MrArgs &a, const MrBuffers &b, cudaStream_t s) {
    const unsigned wb = blocks_for(a.ngroups, kWalkWarps);
    SF_TRY_CUDA(launch(k_mr_walk<KER, BW, CLIP, true, TZ>, dim3(wb), dim3(kWalkWarps * 32), 0, s, a,
                       (uint32_t *)nullptr, (const uint32_t *)b.off, b.list));
    SF_TRY_CUDA(launch(k_grid_item_counts, dim3(blocks_for(a.ntiles, 256)), dim3(256), 0, s,
                       (const uint32_t *)b.cnt, a.ntiles, b.lpw, b.ic));
    SF_TRY(scan_u32(b.ic, b.ioff, a.ntiles, b.tot + 1, s));
    SF_TRY_CUDA(launch(k_grid_items, dim3(blocks_for(a.ntiles, 256)), dim3(256), 0, s,
                       (const uint32_t *)b.cnt, (const uint32_t *)b.off, (const uint32_t *)b.ic,
                       (const uint32_t *)b.ioff, a.ntiles, b.lpw, b.items));
    SF_TRY_CUDA(cudaMemsetAsync(b.next, 0, sizeof(unsigned int), s));
    {
        KTimer t(CNT ? "k_grid_work_count" : "k_grid_work", s);
        bool done = false;
        if constexpr (KER == SF_K_GAUSS3 && TZ == 8 && !CNT && BW != BW_ANISO) {
            done = true;
            switch (a.prec) {
                case SF_PREC_TF32: SF_TRY((launch_work<KER, BW, CLIP, CNT, TZ, SF_PREC_TF32>(a, b, s))); break;
                case SF_PREC_3XTF32: SF_TRY((launch_work<KER, BW, CLIP, CNT, TZ, SF_PREC_3XTF32>(a, b, s))); break;
                case SF_PREC_BF16: SF_TRY((launch_work<KER, BW, CLIP, CNT, TZ, SF_PREC_BF16>(a, b, s))); break;
                default: done = false;
            }
        }
        if (!done) SF_TRY((launch_work<KER, BW, CLIP, CNT, TZ, SF_PREC_FP32>(a, b, s)));
    }
    SF_TRY_CUDA(launch(k_mr_reduce<TZ>, dim3(blocks_for(a.ntiles, kGridThreads / 32)), dim3(kGridThreads), 0, s, a,
                       (const uint32_t *)b.ic, (const uint32_t *)b.ioff, (const double *)b.part));
    return SF_OK;
}

// Sizes of an execution from the candidate total: resident blocks, leaves per
// work item, the item bound.
template <int KER, int BW, bool CLIP, bool CNT, int TZ>
static sf_status mr_sizes(const MrArgs &a, uint32_t total, int items_per_slot, int64_t *slots,
                          uint32_t *lpw, int64_t *max_items) {
    int dev = 0, sms = 0, per_sm = 0;
    SF_TRY_CUDA(cudaGetDevice(&dev));
    SF_TRY_CUDA(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
    SF_TRY((mr_work_attr<KER, BW, CLIP, CNT, TZ>(&per_sm)));
    *slots = (int64_t)sms * per_sm;  // resident blocks of 8 persistent warps
    const int64_t warps = *slots * (kGridThreads / 32);
    const int64_t ips = std::max(1, items_per_slot);
    // At least 16 leaves an item (full staging passes), 8 where so few items leave warps without one:
    // 24^3 nodes, fixed lengths, in 0.03 of a cloud of 4M points 203 us with 16, 194 with 8.
    const int64_t least = total < 8 * warps ? 8 : 16;
    *lpw = (uint32_t)std::max<int64_t>(least, (total + ips * warps - 1) / (ips * warps));
    *max_items = a.ntiles + total / *lpw + 1;
    return SF_OK;
}

// Bytes of the execution buffers mr_plan allocates (each rounded as Scratch counts it).
template <int TZ>
static int64_t mr_plan_bytes(int64_t ntiles, uint32_t total, int64_t max_items) {
    return scratch_round(4 * std::max<int64_t>(1, total)) + 2 * scratch_round(4 * ntiles) +
           scratch_round(16 * max_items) + scratch_round(8 * max_items * 32 * TZ) + scratch_round(4);
}

static int64_t scan_parts_bytes_(int64_t n) { return n > 0 ? scratch_round(4 * ((n + 2047) / 2048)) : 0; }

// Plan the buffers of an execution from the candidate total.
template <int KER, int BW, bool CLIP, bool CNT, int TZ>
static sf_status mr_plan(const MrArgs &a, uint32_t total, int items_per_slot, MrBuffers &b,
                         Scratch *sc, std::vector<void *> *owned, cudaStream_t s) {
    int64_t max_items = 0;
    SF_TRY((mr_sizes<KER, BW, CLIP, CNT, TZ>(a, total, items_per_slot, &b.slots, &b.lpw, &max_items)));
    auto get = [&](size_t bytes) -> void * {
        void *p = nullptr;
        if (sc) {
            p = sc->get<unsigned char>((int64_t)bytes);
        } else if (cudaMalloc(&p, bytes) == cudaSuccess) {
            owned->push_back(p);
        } else {
            p = nullptr;
        }
        return p;
    };
    b.list = (int *)get(sizeof(int) * std::max<int64_t>(1, total));
    b.ic = (uint32_t *)get(sizeof(uint32_t) * a.ntiles);
    b.ioff = (uint32_t *)get(sizeof(uint32_t) * a.ntiles);
    b.items = (int4 *)get(sizeof(int4) * max_items);
    b.part = (double *)get(sizeof(double) * max_items * 32 * TZ);
    b.next = (unsigned int *)get(sizeof(unsigned int));
    if (!b.list || !b.ic || !b.ioff || !b.items || !b.part || !b.next)
        return fail(SF_ERR_OOM, "grid work buffers (%lld items)", (long long)max_items);
    return SF_OK;
}

// ws_bytes (nullable): size the execution and return its bytes instead of running it.
template <int KER, int BW, bool CLIP, int TZ>
// shallow (non-null): if most candidate leaves have supports below twice the node
// spacing, set *shallow and return after the count (the caller re-plans with
// 8 x 4 x 4 tiles); otherwise *shallow = false and the call runs.
static sf_status mr_once(const MrArgs &a_in, int items_per_slot, StatusPeek *peek, int64_t *ws_bytes,
                         cudaStream_t s, bool *shallow = nullptr) {
    Scratch sc(s);
    MrBuffers b;
    MrArgs a = a_in;
    b.cnt = sc.get<uint32_t>(a.ntiles);
    b.off = sc.get<uint32_t>(a.ntiles);
    b.tot = sc.get<uint32_t>(4);
    if (shallow) a.small_leaves = sc.get<unsigned long long>(1);
    SF_TRY_SCRATCH(sc);
    uint32_t total = 0;
    unsigned long long nsmall = 0;
    SF_TRY((mr_count<KER, BW, CLIP, TZ>(a, b.cnt, b.off, b.tot, &total, peek, s, &nsmall)));
    a.small_leaves = nullptr;
    if (shallow) {
        *shallow = 2 * nsmall > (unsigned long long)total;
        if (*shallow) return SF_OK;
    }
    if (ws_bytes) {
        int64_t slots = 0, max_items = 0;
        uint32_t lpw = 0;
        SF_TRY((mr_sizes<KER, BW, CLIP, false, TZ>(a, total, items_per_slot, &slots, &lpw, &max_items)));
        *ws_bytes = 2 * scratch_round(4 * (int64_t)a.ntiles) + scratch_round(16) +
                    (shallow ? scratch_round(8) : 0) +
                    mr_plan_bytes<TZ>(a.ntiles, total, max_items) + scan_parts_bytes_(a.ntiles);
        return SF_OK;
    }
    if (a.pairs) {
        SF_TRY((mr_plan<KER, BW, CLIP, true, TZ>(a, total, items_per_slot, b, &sc, nullptr, s)));
        SF_TRY_SCRATCH(sc);
        return mr_exec<KER, BW, CLIP, true, TZ>(a, b, s);
    }
    SF_TRY((mr_plan<KER, BW, CLIP, false, TZ>(a, total, items_per_slot, b, &sc, nullptr, s)));
    SF_TRY_SCRATCH(sc);
    return mr_exec<KER, BW, CLIP, false, TZ>(a, b, s);
}

template <int KER, int TZ>
static sf_status dispatch_once(int bw, bool clip, const MrArgs &a, int ips, StatusPeek *pk,
                               int64_t *ws, cudaStream_t s, bool *sh = nullptr) {
    switch (bw * 2 + (clip ? 1 : 0)) {
        case BW_ISO * 2 + 0: return mr_once<KER, BW_ISO, false, TZ>(a, ips, pk, ws, s, sh);
        case BW_ISO * 2 + 1: return mr_once<KER, BW_ISO, true, TZ>(a, ips, pk, ws, s, sh);
        case BW_UNIFORM * 2 + 0: return mr_once<KER, BW_UNIFORM, false, TZ>(a, ips, pk, ws, s, sh);
        case BW_UNIFORM * 2 + 1: return mr_once<KER, BW_UNIFORM, true, TZ>(a, ips, pk, ws, s, sh);
        case BW_ANISO * 2 + 0: return mr_once<KER, BW_ANISO, false, TZ>(a, ips, pk, ws, s, sh);
        default: return mr_once<KER, BW_ANISO, true, TZ>(a, ips, pk, ws, s, sh);
    }
}

float kernel_cnorm(int kernel) {
    const double pi = 3.14159265358979323846;
    if (kernel == SF_K_EPAN) return (float)(15.0 / (8.0 * pi));
    const double p3 = std::erf(3.0 / std::sqrt(2.0)) - std::sqrt(2.0 / pi) * 3.0 * std::exp(-4.5);
    return (float)(1.0 / (std::pow(2.0 * pi, 1.5) * p3));
}

static EngineArgs engine_args(sf_index *idx, const sf_box &roi, const DensityCall &call) {
    EngineArgs e;
    e.tv = idx->view();
    e.ell = call.ell;
    e.nell = call.nell_override ? call.nell_override : idx->nell;
    e.dp = call.dp;
    e.cnorm = kernel_cnorm(call.kernel);
    float_bounds(roi.lo, roi.hi, e.blo, e.bhi);
    return e;
}

// Node coordinates r_k(i) = lo_k + i s_k in double, split into float (hi, lo).
void node_axes(const GridSpec &g, float2 *ax) {
    const int nd[3] = {g.nx, g.ny, g.nz};
    size_t o = 0;
    for (int k = 0; k < 3; ++k)
        for (int i = 0; i < nd[k]; ++i) {
            const double r = g.lo[k] + (double)i * g.s[k];
            const float h = (float)r;
            ax[o++] = make_float2(h, (float)(r - (double)h));
        }
}

static RoiDesc roi_desc(const GridSpec &g, int tz, const float2 *axis, int tile_base, float *out,
                        double *mass_part, const DensityParams *dp, const sf_box &roi,
                        int wx = kTileX, int wy = kTileY) {
    RoiDesc r;
    r.axis = axis;
    r.nx = g.nx;
    r.ny = g.ny;
    r.nz = g.nz;
    r.tiles_x = (g.nx + wx - 1) / wx;
    r.tiles_y = (g.ny + wy - 1) / wy;
    r.tiles_z = (g.nz + tz - 1) / tz;
    r.tile_base = tile_base;
    r.group_base = r.groups_x = r.groups_y = 0;  // set_groups
    r.out = out;
    r.mass_part = mass_part;
    r.dp = dp;
    float_bounds(roi.lo, roi.hi, r.blo, r.bhi);
    return r;
}

// Groups of tiles for the walk: as many neighbours to a group as leave at least 6,000
// groups, 12,000 for the 4-deep tiles (whose supports are about a node spacing, so that
// neighbours share few candidates); below that the longer walks of the larger boxes are
// not hidden any more. 65,536 tiles of a zoom of 67M points: 406, 236, 133, 86 us with 1,
// 2, 4, 8 tiles to a group; 32,768 4-deep tiles of its cube: 280, 295, 418 us with 1, 2, 4.
static void group_dims(int64_t ntiles, int tz, MrArgs &a) {
    const int64_t least = tz == 4 ? 12000 : 6000;
    a.gx = a.gy = a.gz = 1;
    if (ntiles >= 2 * least) a.gy = 2;
    if (ntiles >= 4 * least) a.gz = 2;
    if (ntiles >= 8 * least) a.gx = 2;
}
static int64_t set_groups(RoiDesc &r, const MrArgs &a, int64_t group_base) {
    r.group_base = (int)group_base;
    r.groups_x = (r.tiles_x + a.gx - 1) / a.gx;
    r.groups_y = (r.tiles_y + a.gy - 1) / a.gy;
    return (int64_t)r.groups_x * r.groups_y * ((r.tiles_z + a.gz - 1) / a.gz);
}

// The tile gather with TZ-deep tiles and ips work items per resident warp (8:
// measured equal or up to 7% faster than 4 on the zoom grids of the 1.07B cloud);
// shallow (non-null): see mr_once (returns early, nothing written, when set).
template <int TZ>
static sf_status grid_gather(sf_index *idx, const sf_box &roi, const GridSpec &g,
                             const DensityCall &call, float *d_out, double *d_mass, cudaStream_t s,
                             unsigned long long *d_pairs, StatusPeek *peek, int64_t *ws_bytes,
                             int ips, bool *shallow) {
    std::vector<float2> ax((size_t)g.nx + g.ny + g.nz);
    node_axes(g, ax.data());
    const int64_t tiles = (int64_t)((g.nx + kWX - 1) / kWX) * ((g.ny + kWY - 1) / kWY) *
                          ((g.nz + TZ - 1) / TZ);
    if (tiles >= (int64_t(1) << 30)) return fail(SF_ERR_INVALID_ARG, "grid too large");
    Scratch sc(s);
    float2 *d_axis = sc.get<float2>((int64_t)ax.size());
    double *mass_part = sc.get<double>(tiles);
    RoiDesc *d_roi = sc.get<RoiDesc>(1);
    SF_TRY_SCRATCH(sc);
    SF_TRY_CUDA(cudaMemcpyAsync(d_axis, ax.data(), ax.size() * sizeof(float2),
                                cudaMemcpyHostToDevice, s));
    MrArgs a;
    group_dims(tiles, TZ, a);
    RoiDesc r = roi_desc(g, TZ, d_axis, 0, d_out, mass_part, call.dp, roi, kWX, kWY);
    a.ngroups = (int)set_groups(r, a, 0);
    a.group_roi = nullptr;
    SF_TRY_CUDA(cudaMemcpyAsync(d_roi, &r, sizeof r, cudaMemcpyHostToDevice, s));
    a.e = engine_args(idx, roi, call);
    a.rois = d_roi;
    a.tile_roi = nullptr;
    a.ntiles = (int)tiles;
    a.pairs = d_pairs;
    a.prec = call.prec;
    {
        KTimer t(d_pairs ? "k_grid_count" : "k_grid", s);
        if (call.kernel == SF_K_EPAN)
            SF_TRY((dispatch_once<SF_K_EPAN, TZ>(call.bw, call.clip != 0, a, ips, peek, ws_bytes, s, shallow)));
        else
            SF_TRY((dispatch_once<SF_K_GAUSS3, TZ>(call.bw, call.clip != 0, a, ips, peek, ws_bytes, s, shallow)));
    }
    if (shallow && *shallow) return SF_OK;
    if (ws_bytes) {  // this function's own buffers on top of the execution's
        *ws_bytes += scratch_round(sizeof(float2) * ax.size()) + scratch_round(8 * tiles) +
                     scratch_round(sizeof(RoiDesc));
        return SF_OK;
    }
    if (d_mass) {
        const double cell = g.s[0] * g.s[1] * g.s[2];
        SF_TRY_CUDA(launch(k_mass_final, dim3(1), dim3(1024), 0, s, (const double *)mass_part,
                           tiles, cell, d_mass));
    }
    return SF_OK;
}

// Tile depth: 8 x 4 x 8 node tiles by default; when most of a grid's candidate
// leaves have supports below twice the node spacing on every axis (each particle
// reaches a few nodes: a whole billion-point cloud at 256^3, whose supports are
// about one spacing), 8 x 4 x 4 tiles with 32 work items per warp: fewer nodes
// swept per staged particle (measured 17% faster there, 45% slower on dense zoom
// grids, whose supports span 8 to 150 spacings; the finer items balance the
// cube's uneven tiles, 4% more). The decision costs the 8-deep count walk. The
// tensor-core variants need 8-deep tiles and keep them.
static sf_status density_grid_gather(sf_index *idx, const sf_box &roi, const GridSpec &g,
                                     const DensityCall &call, float *d_out, double *d_mass,
                                     cudaStream_t s, unsigned long long *d_pairs, StatusPeek *peek,
                                     int64_t *ws_bytes) {
    bool shallow = false;
    SF_TRY(grid_gather<kTileZ>(idx, roi, g, call, d_out, d_mass, s, d_pairs, peek, ws_bytes, 8,
                               call.prec == SF_PREC_FP32 ? &shallow : nullptr));
    if (!shallow) return SF_OK;
    if (ws_bytes) *ws_bytes = 0;
    const sf_status st = grid_gather<4>(idx, roi, g, call, d_out, d_mass, s, d_pairs, peek, ws_bytes,
                                        32, nullptr);
    if (st != SF_ERR_CAPACITY) return st;
    // the shallow tiles' lists would pass 2^31 entries where the 8-deep ones fit: keep those
    clear_error();
    if (ws_bytes) *ws_bytes = 0;
    return grid_gather<kTileZ>(idx, roi, g, call, d_out, d_mass, s, d_pairs, peek, ws_bytes, 8, nullptr);
}

// The pair-by-pair gather, or the exact moment form (sf_moments.cu) when the
// call asks for it, or, under SF_ACCEL_AUTO, when the gather's candidate lists
// would pass 2^31 entries (the gather stops at its sizing step, before any
// density kernel has run). The pair count always takes the gather.
static sf_status density_grid_impl(sf_index *idx, const sf_box &roi, const GridSpec &g,
                                   const DensityCall &call, float *d_out, double *d_mass,
                                   cudaStream_t s, unsigned long long *d_pairs, StatusPeek *peek,
                                   int64_t *ws_bytes) {
    if (!d_pairs && moments_apply(call)) {
        if (call.accel == SF_ACCEL_MOMENTS)
            return density_grid_moments(idx, roi, g, call, d_out, d_mass, s, ws_bytes, peek);
        const sf_status st = density_grid_gather(idx, roi, g, call, d_out, d_mass, s, nullptr, peek, ws_bytes);
        if (st != SF_ERR_CAPACITY) return st;
        clear_error();
        return density_grid_moments(idx, roi, g, call, d_out, d_mass, s, ws_bytes, peek);
    }
    return density_grid_gather(idx, roi, g, call, d_out, d_mass, s, d_pairs, peek, ws_bytes);
}

sf_status density_grid(sf_index *idx, const sf_box &roi, const GridSpec &g,
                       const DensityCall &call, float *d_out, double *d_mass, cudaStream_t s,
                       unsigned long long *d_pairs, StatusPeek *peek) {
    return density_grid_impl(idx, roi, g, call, d_out, d_mass, s, d_pairs, peek, nullptr);
}

// Device bytes density_grid holds at its peak for this ROI (it runs the
// candidate count, which synchronises the stream).
sf_status grid_workspace(sf_index *idx, const sf_box &roi, const GridSpec &g,
                         const DensityCall &call, int64_t *bytes, cudaStream_t s) {
    *bytes = 0;
    return density_grid_impl(idx, roi, g, call, nullptr, nullptr, s, nullptr, nullptr, bytes);
}

// Same result as density_grid with the monolithic kernel, on node coordinates
// and per-tile partial sums that the caller has already placed in device
// memory (no allocation here).
sf_status density_grid_prealloc(sf_index *idx, const sf_box &roi, const GridSpec &g,
                                const DensityCall &call, const float2 *d_axis,
                                double *d_mass_part, float *d_out, double *d_mass, cudaStream_t s) {
    GridArgs a;
    a.e = engine_args(idx, roi, call);
    a.roi = roi_desc(g, kTileZ, d_axis, 0, d_out, d_mass_part, call.dp, roi);
    a.pairs = nullptr;
    const int64_t tiles = (int64_t)a.roi.tiles_x * a.roi.tiles_y * a.roi.tiles_z;
    cudaError_t e = (call.kernel == SF_K_EPAN)
                        ? dispatch_grid<SF_K_EPAN>(call.bw, call.clip != 0, a, (unsigned)tiles, s)
                        : dispatch_grid<SF_K_GAUSS3>(call.bw, call.clip != 0, a, (unsigned)tiles, s);
    SF_TRY_CUDA(e);
    if (d_mass) {
        const double cell = g.s[0] * g.s[1] * g.s[2];
        SF_TRY_CUDA(launch(k_mass_final, dim3(1), dim3(1024), 0, s, (const double *)d_mass_part,
                           tiles, cell, d_mass));
    }
    return SF_OK;
}

int64_t grid_tile_count(const GridSpec &g) {
    return (int64_t)((g.nx + kTileX - 1) / kTileX) * ((g.ny + kTileY - 1) / kTileY) *
           ((g.nz + kTileZ - 1) / kTileZ);
}

// ===========================================================================
// Batched grids: many ROIs in one persistent execution, replayed from a graph
// ===========================================================================
struct BatchPlan {
    sf_index *idx = nullptr;
    int nroi = 0;
    int kernel = 0, bw = 0;
    bool clip = false;
    int tz = 8, ips = 4;
    bool use_graph = true;
    std::vector<RoiDesc> h_rois;       // host copy (out pointers updated per run)
    std::vector<void *> owned;         // cudaMalloc'ed buffers
    RoiDesc *d_rois = nullptr;
    double *d_mass = nullptr;
    MrArgs a;
    MrBuffers b;
    cudaGraph_t graph = nullptr;
    cudaGraphExec_t exec = nullptr;
};

template <int KER, int BW, bool CLIP, int TZ>
static sf_status batch_build(BatchPlan &P, cudaStream_t s) {
    uint32_t total = 0;
    SF_TRY((mr_count<KER, BW, CLIP, TZ>(P.a, P.b.cnt, P.b.off, P.b.tot, &total, nullptr, s)));
    SF_TRY((mr_plan<KER, BW, CLIP, false, TZ>(P.a, total, P.ips, P.b, nullptr, &P.owned, s)));
    if (!P.use_graph) return SF_OK;
    // capture the execution once, on a private stream (the caller's may be the
    // legacy default stream, which cannot be captured); runs replay it on theirs
    cudaStream_t cs = nullptr;
    SF_TRY_CUDA(cudaStreamCreateWithFlags(&cs, cudaStreamNonBlocking));
    cudaError_t ce = cudaStreamBeginCapture(cs, cudaStreamCaptureModeThreadLocal);
    if (ce != cudaSuccess) {
        cudaStreamDestroy(cs);
        return fail(SF_ERR_CUDA, "cudaStreamBeginCapture: %s", cudaGetErrorString(ce));
    }
    sf_status st = mr_exec<KER, BW, CLIP, false, TZ>(P.a, P.b, cs);
    cudaGraph_t g = nullptr;
    ce = cudaStreamEndCapture(cs, &g);
    cudaStreamDestroy(cs);
    if (st != SF_OK) {
        if (g) cudaGraphDestroy(g);
        return st;
    }
    SF_TRY_CUDA(ce);
    P.graph = g;
    SF_TRY_CUDA(cudaGraphInstantiate(&P.exec, g, 0));
    return SF_OK;
}

template <int KER, int BW, bool CLIP, int TZ>
static sf_status batch_exec(BatchPlan &P, cudaStream_t s) {
    if (P.exec) {
        KTimer t("k_batch_graph", s);
        SF_TRY_CUDA(cudaGraphLaunch(P.exec, s));
        g_launches.fetch_add(8, std::memory_order_relaxed);  // kernels inside the graph
        return SF_OK;
    }
    return mr_exec<KER, BW, CLIP, false, TZ>(P.a, P.b, s);
}

template <int KER, int TZ>
static sf_status batch_dispatch(BatchPlan &P, bool build, cudaStream_t s) {
    switch (P.bw * 2 + (P.clip ? 1 : 0)) {
        case BW_ISO * 2 + 0: return build ? batch_build<KER, BW_ISO, false, TZ>(P, s) : batch_exec<KER, BW_ISO, false, TZ>(P, s);
        case BW_ISO * 2 + 1: return build ? batch_build<KER, BW_ISO, true, TZ>(P, s) : batch_exec<KER, BW_ISO, true, TZ>(P, s);
        case BW_UNIFORM * 2 + 0: return build ? batch_build<KER, BW_UNIFORM, false, TZ>(P, s) : batch_exec<KER, BW_UNIFORM, false, TZ>(P, s);
        default: return build ? batch_build<KER, BW_UNIFORM, true, TZ>(P, s) : batch_exec<KER, BW_UNIFORM, true, TZ>(P, s);
    }
}

static sf_status batch_call(BatchPlan &P, bool build, cudaStream_t s) {
    if (P.kernel == SF_K_EPAN)
        return P.tz == 4 ? batch_dispatch<SF_K_EPAN, 4>(P, build, s) : batch_dispatch<SF_K_EPAN, 8>(P, build, s);
    return P.tz == 4 ? batch_dispatch<SF_K_GAUSS3, 4>(P, build, s) : batch_dispatch<SF_K_GAUSS3, 8>(P, build, s);
}

void batch_free(BatchPlan *P) {
    if (!P) return;
    if (P->exec) cudaGraphExecDestroy(P->exec);
    if (P->graph) cudaGraphDestroy(P->graph);
    for (void *p : P->owned) cudaFree(p);
    delete P;
}

// rois/grids: nroi boxes and GridSpecs; dps: device DensityParams per ROI (owned by the plan)
sf_status batch_create(sf_index *idx, int nroi, const sf_box *rois, const GridSpec *grids,
                       int kernel, int bw, bool clip, DensityParams *d_dps, int tz, int ips,
                       bool use_graph, cudaStream_t s, BatchPlan **out, int prec) {
    BatchPlan *P = new BatchPlan();
    P->idx = idx;
    P->nroi = nroi;
    P->kernel = kernel;
    P->bw = bw;
    P->clip = clip;
    P->tz = (tz == 4) ? 4 : 8;
    P->ips = ips;
    P->use_graph = use_graph;
    auto bail = [&](sf_status st) {
        batch_free(P);
        return st;
    };
    P->owned.push_back(d_dps);
    int64_t naxis = 0, ntiles = 0;
    std::vector<int64_t> tb(nroi);
    for (int r = 0; r < nroi; ++r) {
        naxis += grids[r].nx + grids[r].ny + grids[r].nz;
        tb[r] = ntiles;
        ntiles += (int64_t)((grids[r].nx + kWX - 1) / kWX) * ((grids[r].ny + kWY - 1) / kWY) *
                  ((grids[r].nz + P->tz - 1) / P->tz);
    }
    if (ntiles >= (int64_t(1) << 30)) return bail(fail(SF_ERR_INVALID_ARG, "batch too large"));
    std::vector<float2> ax(naxis);
    std::vector<int> tile_roi(ntiles), group_roi;
    group_dims(ntiles, P->tz, P->a);
    int64_t ngroups = 0;
    for (int r = 0; r < nroi; ++r) {
        RoiDesc t = roi_desc(grids[r], P->tz, nullptr, 0, nullptr, nullptr, nullptr, rois[r], kWX, kWY);
        ngroups += set_groups(t, P->a, 0);
    }
    group_roi.resize(ngroups);
    void *p_gr = nullptr;
    void *p_axis = nullptr, *p_rois = nullptr, *p_tr = nullptr, *p_mp = nullptr, *p_mass = nullptr,
         *p_cnt = nullptr, *p_off = nullptr, *p_tot = nullptr;
    cudaError_t e;
    if ((e = cudaMalloc(&p_axis, sizeof(float2) * naxis)) != cudaSuccess ||
        (e = cudaMalloc(&p_rois, sizeof(RoiDesc) * nroi)) != cudaSuccess ||
        (e = cudaMalloc(&p_tr, sizeof(int) * ntiles)) != cudaSuccess ||
        (e = cudaMalloc(&p_gr, sizeof(int) * ngroups)) != cudaSuccess ||
        (e = cudaMalloc(&p_mp, sizeof(double) * ntiles)) != cudaSuccess ||
        (e = cudaMalloc(&p_mass, sizeof(double) * 2 * nroi)) != cudaSuccess ||
        (e = cudaMalloc(&p_cnt, sizeof(uint32_t) * ntiles)) != cudaSuccess ||
        (e = cudaMalloc(&p_off, sizeof(uint32_t) * ntiles)) != cudaSuccess ||
        (e = cudaMalloc(&p_tot, sizeof(uint32_t) * 4)) != cudaSuccess) {
        for (void *q : {p_axis, p_rois, p_tr, p_gr, p_mp, p_mass, p_cnt, p_off, p_tot})
            if (q) cudaFree(q);
        return bail(fail(SF_ERR_OOM, "batch plan: %s", cudaGetErrorString(e)));
    }
    for (void *q : {p_axis, p_rois, p_tr, p_gr, p_mp, p_mass, p_cnt, p_off, p_tot}) P->owned.push_back(q);
    float2 *d_axis = (float2 *)p_axis;
    double *d_mp = (double *)p_mp;
    P->d_rois = (RoiDesc *)p_rois;
    P->d_mass = (double *)p_mass;
    int64_t ao = 0, go = 0;
    P->h_rois.resize(nroi);
    std::vector<double> cells(nroi);
    for (int r = 0; r < nroi; ++r) {
        node_axes(grids[r], ax.data() + ao);
        P->h_rois[r] = roi_desc(grids[r], P->tz, d_axis + ao, (int)tb[r], nullptr, d_mp + tb[r],
                                d_dps + r, rois[r], kWX, kWY);
        const int64_t ng = set_groups(P->h_rois[r], P->a, go);
        for (int64_t t = 0; t < ng; ++t) group_roi[go + t] = r;
        go += ng;
        const int64_t nt = (r + 1 < nroi ? tb[r + 1] : ntiles) - tb[r];
        for (int64_t t = 0; t < nt; ++t) tile_roi[tb[r] + t] = r;
        ao += grids[r].nx + grids[r].ny + grids[r].nz;
        cells[r] = grids[r].s[0] * grids[r].s[1] * grids[r].s[2];
    }
    if ((e = cudaMemcpyAsync(d_axis, ax.data(), sizeof(float2) * naxis, cudaMemcpyHostToDevice, s)) != cudaSuccess ||
        (e = cudaMemcpyAsync(P->d_rois, P->h_rois.data(), sizeof(RoiDesc) * nroi, cudaMemcpyHostToDevice, s)) != cudaSuccess ||
        (e = cudaMemcpyAsync(p_tr, tile_roi.data(), sizeof(int) * ntiles, cudaMemcpyHostToDevice, s)) != cudaSuccess ||
        (e = cudaMemcpyAsync(p_gr, group_roi.data(), sizeof(int) * ngroups, cudaMemcpyHostToDevice, s)) != cudaSuccess ||
        (e = cudaMemcpyAsync(P->d_mass + nroi, cells.data(), sizeof(double) * nroi, cudaMemcpyHostToDevice, s)) != cudaSuccess)
        return bail(fail(SF_ERR_CUDA, "batch plan upload: %s", cudaGetErrorString(e)));
    sf_box any = rois[0];
    DensityCall call;
    call.kernel = kernel;
    call.bw = bw;
    call.clip = clip ? 1 : 0;
    call.ell = nullptr;
    call.dp = d_dps;
    call.nell_override = nullptr;
    P->a.e = engine_args(idx, any, call);
    P->a.rois = P->d_rois;
    P->a.tile_roi = (const int *)p_tr;
    P->a.ntiles = (int)ntiles;
    P->a.group_roi = (const int *)p_gr;
    P->a.ngroups = (int)ngroups;
    P->a.pairs = nullptr;
    P->a.prec = prec;  // the work kernel's form (tensor-core variants: Gaussian, 8-deep tiles)
    P->b.cnt = (uint32_t *)p_cnt;
    P->b.off = (uint32_t *)p_off;
    P->b.tot = (uint32_t *)p_tot;
    sf_status st = batch_call(*P, true, s);
    if (st != SF_OK) return bail(st);
    *out = P;
    return SF_OK;
}

sf_status batch_run(BatchPlan *P, float *const *outs, double *h_mass, cudaStream_t s) {
    bool changed = false;
    for (int r = 0; r < P->nroi; ++r)
        if (P->h_rois[r].out != outs[r]) {
            P->h_rois[r].out = outs[r];
            changed = true;
        }
    if (changed)
        SF_TRY_CUDA(cudaMemcpyAsync(P->d_rois, P->h_rois.data(), sizeof(RoiDesc) * P->nroi,
                                    cudaMemcpyHostToDevice, s));
    SF_TRY(batch_call(*P, false, s));
    if (h_mass) {
        SF_TRY_CUDA(launch(k_mr_mass, dim3(P->nroi), dim3(256), 0, s, (const RoiDesc *)P->d_rois,
                           (const double *)(P->d_mass + P->nroi), P->nroi, P->d_mass));
        SF_TRY_CUDA(cudaMemcpyAsync(h_mass, P->d_mass, sizeof(double) * P->nroi, cudaMemcpyDeviceToHost, s));
        SF_TRY_CUDA(cudaStreamSynchronize(s));
    }
    return SF_OK;
}

// ===========================================================================
// Points (DIRECT)
// ===========================================================================
constexpr int kPtWarps = 4;
constexpr int kWideLeaves = 512;

struct PointsArgs {
    EngineArgs e;
    const int *leaves;          // query leaves (null: every leaf, slot = leaf)
    int64_t nslots;             // number of query leaves
    float *rho_sorted;          // [nslots * 32]: density of slot point (slot * 32 + lane)
    uint8_t *inroi;             // [nslots * 32]: 1 if that point lies in the ROI
    unsigned long long *pairs;  // counting variant
};

constexpr int kPtRing = 2 * kLeaf;  // staged candidates: two halves of 32

struct __align__(16) PtWarpSmem {
    // staged candidates as structure of arrays (pairs of entries load as one 64-bit word)
    float sx[kPtRing], sy[kPtRing], sz[kPtRing], sc[kPtRing];
    float su[3][kPtRing];  // BW_ISO: su[0] = u^2; else u_x, u_y, u_z
    float4 q[kLeaf];       // the query points
    int stack[kStack];
    int leaves[kBatch];
};

// SPLIT warps work on one query leaf, each on every SPLIT-th candidate leaf (all walk the
// index); their sums are added in warp order. SPLIT = kPtWarps where the query leaves
// alone would not fill the chip: then the longest leaf sets the time (100,000 points: 877 us
// by one warp a leaf, 289 us now).
//
// What bounds it: issue slots, about 9 a staged candidate (two candidates an instruction
// in packed FP32) and 45 a candidate leaf; half of the staged candidates are in support
// of a given lane (the union of 32 queries' reach).
template <int KER, int BW, bool CLIP, bool CNT, int SPLIT>
__global__ void __launch_bounds__(kPtWarps * 32) k_points(PointsArgs a) {
    __shared__ PtWarpSmem W[kPtWarps];
    __shared__ double s_part[SPLIT > 1 ? kPtWarps : 1][kLeaf];
    __shared__ float s_uni[3];
    __shared__ float s_runi[4];  // 1 / uniform l_k, and whether all l_k > 0
    __shared__ double s_inv;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    if (threadIdx.x == 0) {
        const DensityParams dp = *a.e.dp;
        s_uni[0] = dp.ell_uniform[0];
        s_uni[1] = dp.ell_uniform[1];
        s_uni[2] = dp.ell_uniform[2];
        s_runi[0] = 1.0f / s_uni[0];
        s_runi[1] = 1.0f / s_uni[1];
        s_runi[2] = 1.0f / s_uni[2];
        s_runi[3] = (s_uni[0] > 0.f && s_uni[1] > 0.f && s_uni[2] > 0.f) ? 1.f : 0.f;
        s_inv = dp.inv_neff;
    }
    __syncthreads();
    PtWarpSmem &S = W[warp];
    const int part = warp % SPLIT;
    const int64_t slot = ((int64_t)blockIdx.x * kPtWarps + warp) / SPLIT;
    if (slot >= a.nslots) return;
    const int64_t leaf = a.leaves ? (int64_t)a.leaves[slot] : slot;
    const int64_t qi = leaf * kLeaf + lane;
    const int64_t oi = slot * kLeaf + lane;
    const bool valid = qi < a.e.tv.n;
    float4 q = make_float4(0.f, 0.f, 0.f, 0.f);
    if (valid) q = __ldg(&a.e.tv.pos[qi]);
    // query points: those inside the ROI box (closed)
    const bool active = valid && q.x >= a.e.blo[0] && q.x <= a.e.bhi[0] && q.y >= a.e.blo[1] &&
                        q.y <= a.e.bhi[1] && q.z >= a.e.blo[2] && q.z <= a.e.bhi[2];
    if (part == 0) a.inroi[oi] = active ? 1 : 0;
    const unsigned am = __ballot_sync(0xffffffffu, active);
    if (am == 0) return;
    float tlo[3] = {active ? q.x : INFINITY, active ? q.y : INFINITY, active ? q.z : INFINITY};
    float thi[3] = {active ? q.x : -INFINITY, active ? q.y : -INFINITY, active ? q.z : -INFINITY};
#pragma unroll
    for (int k = 0; k < 3; ++k)
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            tlo[k] = fminf(tlo[k], __shfl_xor_sync(0xffffffffu, tlo[k], o));
            thi[k] = fmaxf(thi[k], __shfl_xor_sync(0xffffffffu, thi[k], o));
        }
    // the query box widened by the rounding margin (node test and per-point filter),
    // the latter as centre and half-width
    float mlo[3], mhi[3], mcen[3], mhw[3];
    widen_box(tlo, thi, mlo, mhi);
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        mcen[k] = 0.5f * (mlo[k] + mhi[k]);
        mhw[k] = 0.5f * (mhi[k] - mlo[k]);
    }
    // A leaf whose points lie apart (at a jump of the Morton order) has a box that can cover
    // clusters none of its points is near: from kWideLeaves candidate leaves on (the mean is
    // about 200) nodes are tested against every point. A whole launch waited for single
    // such leaves, of up to 36,000 candidate leaves: the densities at 16.8M clustered
    // points took 44.2 ms, 23.6 ms with this test. (Testing the candidates themselves so costs
    // what it saves there, and where every leaf is wide, as with the estimator's long
    // lengths, 1.7 times the whole: 4M points over the cube 1.43 s, 0.86 s without.)
    bool wide = false;
    int seen = 0;
    S.q[lane] = make_float4(active ? q.x : INFINITY, q.y, q.z, 0.f);
    __syncwarp();
    auto test = [&](int64_t node) {
        if (!node_reaches<KER, BW, CLIP>(a.e, s_uni, node, mlo, mhi)) return false;
        if (!wide) return true;
        const float4 lo = __ldg(&a.e.tv.nlo[node]), hi = __ldg(&a.e.tv.nhi[node]);
        float r[3];
        if (BW == BW_UNIFORM) {
            r[0] = rcp_approx(s_uni[0]); r[1] = rcp_approx(s_uni[1]); r[2] = rcp_approx(s_uni[2]);
        } else {
            const float4 e = __ldg(&a.e.nell[node]);
            r[0] = rcp_approx(e.x); r[1] = rcp_approx(e.y); r[2] = rcp_approx(e.z);
        }
        bool near = false;
        for (int j = 0; j < kLeaf; ++j) {
            const float4 p = S.q[j];
            const float gx = fmaxf(fmaxf(lo.x - p.x, p.x - hi.x), 0.f) * r[0];
            const float gy = fmaxf(fmaxf(lo.y - p.y, p.y - hi.y), 0.f) * r[1];
            const float gz = fmaxf(fmaxf(lo.z - p.z, p.z - hi.z), 0.f) * r[2];
            near = near || fmaf(gz, gz, fmaf(gy, gy, gx * gx)) <
                               KDef<KER>::rmul * KDef<KER>::rmul * (1.0f + kFilterSlack);
        }
        return near;
    };

    float sum = 0.f, cmp = 0.f;
    unsigned long long npairs = 0;
    const f32x2 QX = f2_pack(q.x, q.x), QY = f2_pack(q.y, q.y), QZ = f2_pack(q.z, q.z);
    // two packed candidates against this lane's query
    auto pair2 = [&](f32x2 x, f32x2 y, f32x2 z, f32x2 u0, f32x2 u1, f32x2 u2, f32x2 c, float &acc0, float &acc1) {
        const f32x2 dx = f2_sub(QX, x);
        const f32x2 dy = f2_sub(QY, y);
        const f32x2 dz = f2_sub(QZ, z);
        f32x2 qq;
        if (BW == BW_ISO) {
            qq = f2_mul(f2_fma(dz, dz, f2_fma(dy, dy, f2_mul(dx, dx))), u0);
        } else {
            const f32x2 tx = f2_mul(dx, u0);
            const f32x2 ty = f2_mul(dy, u1);
            const f32x2 tz = f2_mul(dz, u2);
            qq = f2_fma(tz, tz, f2_fma(ty, ty, f2_mul(tx, tx)));
        }
        float q0, q1, c0, c1;
        f2_unpack(qq, q0, q1);
        f2_unpack(c, c0, c1);
        const bool in0 = q0 < KDef<KER>::qmax, in1 = q1 < KDef<KER>::qmax;
        if (KER == SF_K_GAUSS3) {
            if (in0) acc0 = fmaf(c0, ex2_approx(-q0), acc0);
            if (in1) acc1 = fmaf(c1, ex2_approx(-q1), acc1);
        } else {
            if (in0) acc0 = fmaf(c0, 1.0f - q0, acc0);
            if (in1) acc1 = fmaf(c1, 1.0f - q1, acc1);
        }
        if (CNT) npairs += (unsigned)in0 + (unsigned)in1;
    };
    // entries s, ..., s + 3 (s a multiple of 4): one 16-byte load each of x, y, z, u and c
    auto quad = [&](int s, float &a0, float &a1, float &a2, float &a3) {
        auto ld = [](const float *p) { return *reinterpret_cast<const ulonglong2 *>(p); };
        const ulonglong2 x = ld(&S.sx[s]), y = ld(&S.sy[s]), z = ld(&S.sz[s]), c = ld(&S.sc[s]), u0 = ld(&S.su[0][s]);
        const ulonglong2 u1 = BW == BW_ISO ? u0 : ld(&S.su[1][s]), u2 = BW == BW_ISO ? u0 : ld(&S.su[2][s]);
        pair2(x.x, y.x, z.x, u0.x, u1.x, u2.x, c.x, a0, a1);
        pair2(x.y, y.y, z.y, u0.y, u1.y, u2.y, c.y, a2, a3);
    };
    auto add = [&](float v) {  // compensated running sum (TwoSum)
        const float t = sum + v;
        const float bp = t - sum;
        cmp += (sum - (t - bp)) + (v - bp);
        sum = t;
    };
    int head = 0, cnt = 0;  // ring of staged candidates: first entry, count (warp-uniform)
    int spv;
    int nl = warp_walk_start(a.e.tv, test, S.stack, spv, S.leaves);
    while (true) {
        if (nl == 0) {
            if (spv == 0) break;
            nl = warp_walk(a.e.tv, test, S.stack, spv, S.leaves, kBatch);
            if (nl == 0) break;
        }
        seen += nl;
        wide = seen >= kWideLeaves;
        // software pipeline: the next candidate leaf's point is loaded one step ahead
        float4 pn = make_float4(0.f, 0.f, 0.f, 0.f);
        float4 en = pn;
        if (part < nl) {
            const int64_t j0 = (int64_t)S.leaves[part] * kLeaf + lane;
            if (j0 < a.e.tv.n) {
                pn = __ldg(&a.e.tv.pos[j0]);
                if (BW == BW_ANISO) en = __ldg(&a.e.ell[j0]);
            }
        }
        for (int li = part; li < nl; li += SPLIT) {
            const int64_t j = (int64_t)S.leaves[li] * kLeaf + lane;
            const float4 p = pn;
            const float4 pe = en;
            if (li + SPLIT < nl) {
                const int64_t jn = (int64_t)S.leaves[li + SPLIT] * kLeaf + lane;
                if (jn < a.e.tv.n) {
                    pn = __ldg(&a.e.tv.pos[jn]);
                    if (BW == BW_ANISO) en = __ldg(&a.e.ell[jn]);
                }
            }
            bool ok = false;
            float r[3] = {0.f, 0.f, 0.f};  // 1 / l_k
            if (j < a.e.tv.n) {
                if (BW == BW_ISO) {
                    ok = p.w > 0.f;
                    r[0] = r[1] = r[2] = rcp_approx(p.w);
                } else if (BW == BW_UNIFORM) {
                    ok = s_runi[3] > 0.f;
                    r[0] = s_runi[0]; r[1] = s_runi[1]; r[2] = s_runi[2];
                } else {
                    ok = pe.x > 0.f && pe.y > 0.f && pe.z > 0.f;
                    r[0] = rcp_approx(pe.x); r[1] = rcp_approx(pe.y); r[2] = rcp_approx(pe.z);
                }
                if (CLIP)
                    ok = ok && p.x >= a.e.blo[0] && p.x <= a.e.bhi[0] && p.y >= a.e.blo[1] &&
                         p.y <= a.e.bhi[1] && p.z >= a.e.blo[2] && p.z <= a.e.bhi[2];
                const float pc[3] = {p.x, p.y, p.z};
                float qlb = 0.f;
#pragma unroll
                for (int k = 0; k < 3; ++k) {
                    const float t = fmaxf(fabsf(pc[k] - mcen[k]) - mhw[k], 0.f) * r[k];
                    qlb = fmaf(t, t, qlb);
                }
                ok = ok && qlb < KDef<KER>::rmul * KDef<KER>::rmul * (1.0f + kFilterSlack);
            }
            const unsigned m = __ballot_sync(0xffffffffu, ok);
            if (ok) {
                const int s = (head + cnt + __popc(m & ((1u << lane) - 1u))) & (kPtRing - 1);
                S.sx[s] = p.x;
                S.sy[s] = p.y;
                S.sz[s] = p.z;
                S.sc[s] = a.e.cnorm * ((r[0] * r[1]) * r[2]);
                const float u0 = KDef<KER>::uscale * r[0];
                if (BW == BW_ISO) {
                    S.su[0][s] = u0 * u0;
                } else {
                    S.su[0][s] = u0;
                    S.su[1][s] = KDef<KER>::uscale * r[1];
                    S.su[2][s] = KDef<KER>::uscale * r[2];
                }
            }
            cnt += __popc(m);
            if (cnt >= kLeaf) {  // warp-uniform: a full half of the ring is staged
                __syncwarp();
                float a0 = 0.f, a1 = 0.f, a2 = 0.f, a3 = 0.f;
#pragma unroll
                for (int e = 0; e < kLeaf; e += 4) quad(head + e, a0, a1, a2, a3);
                head ^= kLeaf;
                cnt -= kLeaf;
                add((a0 + a1) + (a2 + a3));
                __syncwarp();
            }
        }
        nl = 0;
    }
    // the staged remainder (cnt < 32 entries from head), padded to a multiple of 4 with
    // entries of zero weight
    const int pad = (4 - (cnt & 3)) & 3;
    if (lane < pad) {
        const int s = (head + cnt + lane) & (kPtRing - 1);
        S.sx[s] = S.sy[s] = S.sz[s] = S.sc[s] = 0.f;
        S.su[0][s] = S.su[1][s] = S.su[2][s] = 0.f;
    }
    __syncwarp();
    if (cnt > 0) {
        float a0 = 0.f, a1 = 0.f, a2 = 0.f, a3 = 0.f;
        for (int e = 0; e < cnt; e += 4) quad(head + e, a0, a1, a2, a3);
        if (CNT) npairs -= (unsigned)pad;  // the padding entries are "in support" (q = 0)
        add((a0 + a1) + (a2 + a3));
    }
    double total = (double)sum + (double)cmp;
    if (SPLIT > 1) {
        s_part[warp][lane] = total;
        __syncthreads();
        if (part != 0) return;
#pragma unroll
        for (int w = 1; w < SPLIT; ++w) total += s_part[warp + w][lane];
    }
    if (active) a.rho_sorted[oi] = (float)(total * s_inv);
    if (CNT) {
        if (!active) npairs = 0;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) npairs += __shfl_xor_sync(0xffffffffu, npairs, o);
        if (lane == 0 && npairs) atomicAdd(a.pairs, npairs);
    }
}

template <int KER, int BW, bool CLIP>
static cudaError_t launch_points(const PointsArgs &a, int64_t nleaf, cudaStream_t s) {
    if (a.pairs) {
        KTimer t("k_points_count", s);
        return launch(k_points<KER, BW, CLIP, true, 1>, dim3(blocks_for(nleaf, kPtWarps)),
                      dim3(kPtWarps * 32), 0, s, a);
    }
    KTimer t("k_points", s);
    int dev = 0, sms = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (e != cudaSuccess) return e;
    // below two waves of resident warps (32 an SM) a block shares each leaf
    if (nleaf < (int64_t)sms * 64)
        return launch(k_points<KER, BW, CLIP, false, kPtWarps>, dim3((unsigned)nleaf), dim3(kPtWarps * 32), 0, s, a);
    return launch(k_points<KER, BW, CLIP, false, 1>, dim3(blocks_for(nleaf, kPtWarps)),
                  dim3(kPtWarps * 32), 0, s, a);
}

template <int KER>
static cudaError_t dispatch_points(int bw, bool clip, const PointsArgs &a, int64_t nleaf,
                                   cudaStream_t s) {
    switch (bw * 2 + (clip ? 1 : 0)) {
        case BW_ISO * 2 + 0: return launch_points<KER, BW_ISO, false>(a, nleaf, s);
        case BW_ISO * 2 + 1: return launch_points<KER, BW_ISO, true>(a, nleaf, s);
        case BW_UNIFORM * 2 + 0: return launch_points<KER, BW_UNIFORM, false>(a, nleaf, s);
        case BW_UNIFORM * 2 + 1: return launch_points<KER, BW_UNIFORM, true>(a, nleaf, s);
        case BW_ANISO * 2 + 0: return launch_points<KER, BW_ANISO, false>(a, nleaf, s);
        default: return launch_points<KER, BW_ANISO, true>(a, nleaf, s);
    }
}

// ---------------------------------------------------------------------------
// Tensor-core cross term (precision variants of the point densities)
//
// With coordinates taken relative to the query leaf's centre, the squared
// distance of query i and candidate j is |x_i|^2 + |y_j|^2 - 2 x_i . y_j; the
// cross term of a 32 x 32 block is a [32 x 8] . [8 x 32] product (features x,
// y, z, zero-padded) done by mma.sync m16n8k8 in TF32 (or as the 3-pass
// hi/lo split, "3xTF32", accurate to about 2^-21 of |x||y|), or m16n8k16 in
// BF16 (8 significant bits); the squared norms,
// the scaling by 1/h^2, the cutoff, the kernel and the compensated sums stay
// in FP32. Isotropic bandwidths only (the kNN rule).
// ---------------------------------------------------------------------------
__device__ __forceinline__ uint32_t to_tf32(float x) {
    uint32_t r;
    asm("cvt.rna.tf32.f32 %0, %1;" : "=r"(r) : "f"(x));
    return r;
}

__device__ __forceinline__ void mma_tf32(float d[4], uint32_t a0, uint32_t a1, uint32_t b0) {
    // A rows (groupID, groupID + 8) x cols (tig, tig + 4): cols >= 4 are zero padding
    const uint32_t z = 0u;
    asm volatile(
        "mma.sync.aligned.m16n8k8.row.col.f32.tf32.tf32.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, "
        "{%8,%9}, {%0,%1,%2,%3};"
        : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
        : "r"(a0), "r"(a1), "r"(z), "r"(z), "r"(b0), "r"(z));
}

// BF16: m16n8k16 with the features in k = 0..3 (pairs (x, y), (z, 0) in the
// lanes with tig 0 and 1), k = 4..15 zero. a0 / a1: rows g / g + 8, b0: column g.
__device__ __forceinline__ void mma_bf16(float d[4], uint32_t a0, uint32_t a1, uint32_t b0) {
    const uint32_t z = 0u;
    asm volatile(
        "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, "
        "{%8,%9}, {%0,%1,%2,%3};"
        : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
        : "r"(a0), "r"(a1), "r"(z), "r"(z), "r"(b0), "r"(z));
}

// The TF32 fragment layout holds feature tig of a row in lane (g, tig); the BF16
// one wants features (2 tig, 2 tig + 1) packed in that lane (zero for tig >= 2).
__device__ __forceinline__ uint32_t bf16_pair_from_tf32_layout(float f) {
    const int lane = threadIdx.x & 31, tig = lane & 3;
    const float lo = __shfl_sync(0xffffffffu, f, (lane & ~3) | ((2 * tig) & 3));
    const float hi = __shfl_sync(0xffffffffu, f, (lane & ~3) | ((2 * tig + 1) & 3));
    uint32_t r;
    asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(r) : "f"(tig < 2 ? hi : 0.f), "f"(tig < 2 ? lo : 0.f));
    return r;
}

template <int PREC>
__device__ __forceinline__ void cross_mma(float d[4], float a0f, float a1f, float b0f) {
    const uint32_t a0h = to_tf32(a0f), a1h = to_tf32(a1f), b0h = to_tf32(b0f);
    mma_tf32(d, a0h, a1h, b0h);
    if (PREC == SF_PREC_3XTF32) {
        const uint32_t a0l = to_tf32(a0f - __uint_as_float(a0h));
        const uint32_t a1l = to_tf32(a1f - __uint_as_float(a1h));
        const uint32_t b0l = to_tf32(b0f - __uint_as_float(b0h));
        mma_tf32(d, a0h, a1h, b0l);
        mma_tf32(d, a0l, a1l, b0h);
    }
}

struct TcWarpSmem {
    int stack[kStack];
    int leaves[kBatch];
    float4 yp[kLeaf];   // candidate relative position (x', y', z', -)
    float4 yk[kLeaf];   // (|y'|^2, u^2, c, -)
};

template <int KER, bool CLIP, int PREC>
__global__ void __launch_bounds__(kPtWarps * 32) k_points_tc(PointsArgs a) {
    __shared__ TcWarpSmem W[kPtWarps];
    __shared__ double s_inv;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int g = lane >> 2, tig = lane & 3;
    if (threadIdx.x == 0) s_inv = a.e.dp->inv_neff;
    __syncthreads();
    TcWarpSmem &S = W[warp];
    const int64_t slot = (int64_t)blockIdx.x * kPtWarps + warp;
    if (slot >= a.nslots) return;
    const int64_t leaf = a.leaves ? (int64_t)a.leaves[slot] : slot;
    const int64_t qi = leaf * kLeaf + lane;
    const int64_t oi = slot * kLeaf + lane;
    const bool valid = qi < a.e.tv.n;
    float4 q = make_float4(0.f, 0.f, 0.f, 0.f);
    if (valid) q = __ldg(&a.e.tv.pos[qi]);
    const bool active = valid && q.x >= a.e.blo[0] && q.x <= a.e.bhi[0] && q.y >= a.e.blo[1] &&
                        q.y <= a.e.bhi[1] && q.z >= a.e.blo[2] && q.z <= a.e.bhi[2];
    a.inroi[oi] = active ? 1 : 0;
    const unsigned am = __ballot_sync(0xffffffffu, active);
    if (am == 0) return;
    float tlo[3] = {active ? q.x : INFINITY, active ? q.y : INFINITY, active ? q.z : INFINITY};
    float thi[3] = {active ? q.x : -INFINITY, active ? q.y : -INFINITY, active ? q.z : -INFINITY};
#pragma unroll
    for (int k = 0; k < 3; ++k)
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            tlo[k] = fminf(tlo[k], __shfl_xor_sync(0xffffffffu, tlo[k], o));
            thi[k] = fmaxf(thi[k], __shfl_xor_sync(0xffffffffu, thi[k], o));
        }
    const float cen[3] = {0.5f * (tlo[0] + thi[0]), 0.5f * (tlo[1] + thi[1]), 0.5f * (tlo[2] + thi[2])};
    // this lane's four rows (queries g, g+8, g+16, g+24) relative to the centre
    const float xq[3] = {q.x - cen[0], q.y - cen[1], q.z - cen[2]};
    float feat[4], xsq[4];
#pragma unroll
    for (int sl = 0; sl < 4; ++sl) {
        const int r = g + 8 * sl;
        const float rx = __shfl_sync(0xffffffffu, xq[0], r);
        const float ry = __shfl_sync(0xffffffffu, xq[1], r);
        const float rz = __shfl_sync(0xffffffffu, xq[2], r);
        feat[sl] = tig == 0 ? rx : (tig == 1 ? ry : (tig == 2 ? rz : 0.f));
        xsq[sl] = fmaf(rz, rz, fmaf(ry, ry, rx * rx));
    }
    uint32_t fa16[4] = {0u, 0u, 0u, 0u};  // BF16 A fragments of the four rows
    if (PREC == SF_PREC_BF16) {
#pragma unroll
        for (int sl = 0; sl < 4; ++sl) fa16[sl] = bf16_pair_from_tf32_layout(feat[sl]);
    }
    float uni[3] = {0.f, 0.f, 0.f};
    float wlo[3], whi[3];
    widen_box(tlo, thi, wlo, whi);
    auto test = [&](int64_t node) { return node_reaches<KER, BW_ISO, CLIP>(a.e, uni, node, wlo, whi); };

    float acc[4] = {0.f, 0.f, 0.f, 0.f}, sum[4] = {0.f, 0.f, 0.f, 0.f}, cmp[4] = {0.f, 0.f, 0.f, 0.f};
    int spv;
    int nl = warp_walk_start(a.e.tv, test, S.stack, spv, S.leaves);
    while (true) {
        if (nl == 0) {
            if (spv == 0) break;
            nl = warp_walk(a.e.tv, test, S.stack, spv, S.leaves, kBatch);
            if (nl == 0) break;
        }
        for (int li = 0; li < nl; ++li) {
            const int64_t j = (int64_t)S.leaves[li] * kLeaf + lane;
            bool ok = false;
            float4 p = make_float4(0.f, 0.f, 0.f, 0.f);
            if (j < a.e.tv.n) {
                p = __ldg(&a.e.tv.pos[j]);
                ok = p.w > 0.f;
                if (CLIP)
                    ok = ok && p.x >= a.e.blo[0] && p.x <= a.e.bhi[0] && p.y >= a.e.blo[1] &&
                         p.y <= a.e.bhi[1] && p.z >= a.e.blo[2] && p.z <= a.e.bhi[2];
                const float pc[3] = {p.x, p.y, p.z};
                float qlb = 0.f;
#pragma unroll
                for (int k = 0; k < 3; ++k) {
                    float gap = fmaxf(fmaxf(tlo[k] - pc[k], pc[k] - thi[k]), 0.f);
                    gap = fmaxf(gap - 1.0e-6f * (fabsf(tlo[k]) + fabsf(thi[k])), 0.f);
                    const float t = gap / (p.w * KDef<KER>::rmul);
                    qlb += t * t;
                }
                ok = ok && qlb < 1.0f + 1.0e-5f;
            }
            const unsigned m = __ballot_sync(0xffffffffu, ok);
            if (ok) {
                const int s = __popc(m & ((1u << lane) - 1u));
                const float y0 = p.x - cen[0], y1 = p.y - cen[1], y2 = p.z - cen[2];
                const float u = KDef<KER>::uscale / p.w;
                S.yp[s] = make_float4(y0, y1, y2, 0.f);
                S.yk[s] = make_float4(fmaf(y2, y2, fmaf(y1, y1, y0 * y0)), u * u,
                                      a.e.cnorm / ((p.w * p.w) * p.w), 0.f);
            }
            __syncwarp();
            const int ns = __popc(m);
            for (int nt = 0; nt * 8 < ns; ++nt) {
                // B column g = candidate nt*8 + g, feature row tig: -2 y'
                const int cb = nt * 8 + g;
                float bf = 0.f;
                if (cb < ns && tig < 3) {
                    const float4 y = S.yp[cb];
                    bf = -2.f * (tig == 0 ? y.x : (tig == 1 ? y.y : y.z));
                }
                float d0[4] = {0.f, 0.f, 0.f, 0.f}, d1[4] = {0.f, 0.f, 0.f, 0.f};
                if (PREC == SF_PREC_BF16) {
                    const uint32_t b16 = bf16_pair_from_tf32_layout(bf);
                    mma_bf16(d0, fa16[0], fa16[1], b16);     // rows g, g+8
                    mma_bf16(d1, fa16[2], fa16[3], b16);     // rows g+16, g+24
                } else {
                    cross_mma<PREC>(d0, feat[0], feat[1], bf);   // rows g, g+8
                    cross_mma<PREC>(d1, feat[2], feat[3], bf);   // rows g+16, g+24
                }
                // epilogue: columns 2 tig, 2 tig + 1 of this n-tile
#pragma unroll
                for (int cc = 0; cc < 2; ++cc) {
                    const int jc = nt * 8 + 2 * tig + cc;
                    if (jc < ns) {
                        const float4 yk = S.yk[jc];
                        const float dv[4] = {d0[cc], d0[2 + cc], d1[cc], d1[2 + cc]};
#pragma unroll
                        for (int sl = 0; sl < 4; ++sl) {
                            const float d2 = (xsq[sl] + yk.x) + dv[sl];
                            const float qq = fmaxf(d2, 0.f) * yk.y;
                            if (qq < KDef<KER>::qmax) {
                                if (KER == SF_K_GAUSS3) acc[sl] = fmaf(yk.z, ex2_approx(-qq), acc[sl]);
                                else acc[sl] = fmaf(yk.z, 1.0f - qq, acc[sl]);
                            }
                        }
                    }
                }
            }
            __syncwarp();
#pragma unroll
            for (int sl = 0; sl < 4; ++sl) {
                const float t = sum[sl] + acc[sl];
                const float bp = t - sum[sl];
                cmp[sl] += (sum[sl] - (t - bp)) + (acc[sl] - bp);
                sum[sl] = t;
                acc[sl] = 0.f;
            }
        }
        nl = 0;
    }
    // rows are spread over the four lanes of a group: add them up, then route row L to lane L
    double v[4];
#pragma unroll
    for (int sl = 0; sl < 4; ++sl) {
        v[sl] = (double)sum[sl] + (double)cmp[sl];
        v[sl] += __shfl_xor_sync(0xffffffffu, v[sl], 1);
        v[sl] += __shfl_xor_sync(0xffffffffu, v[sl], 2);
    }
    const int src = 4 * (lane & 7), mysl = lane >> 3;
    double mine = 0.0;
#pragma unroll
    for (int sl = 0; sl < 4; ++sl) {
        const double t = __shfl_sync(0xffffffffu, v[sl], src);
        if (sl == mysl) mine = t;
    }
    if (active) a.rho_sorted[oi] = (float)(mine * s_inv);
}

template <int KER, bool CLIP>
static cudaError_t launch_points_tc(int prec, const PointsArgs &a, int64_t nleaf, cudaStream_t s) {
    KTimer t("k_points_tc", s);
    if (prec == SF_PREC_BF16)
        return launch(k_points_tc<KER, CLIP, SF_PREC_BF16>, dim3(blocks_for(nleaf, kPtWarps)),
                      dim3(kPtWarps * 32), 0, s, a);
    if (prec == SF_PREC_3XTF32)
        return launch(k_points_tc<KER, CLIP, SF_PREC_3XTF32>, dim3(blocks_for(nleaf, kPtWarps)),
                      dim3(kPtWarps * 32), 0, s, a);
    return launch(k_points_tc<KER, CLIP, SF_PREC_TF32>, dim3(blocks_for(nleaf, kPtWarps)),
                  dim3(kPtWarps * 32), 0, s, a);
}

sf_status density_points_tc(sf_index *idx, const sf_box &roi, const DensityCall &call, int prec,
                            const int *d_leaves, int64_t nslots, float *d_rho_sorted,
                            uint8_t *d_inroi, cudaStream_t s) {
    if (call.bw != BW_ISO)
        return fail(SF_ERR_INVALID_ARG, "tensor-core point densities need isotropic (kNN) bandwidths");
    PointsArgs a;
    a.e = engine_args(idx, roi, call);
    a.leaves = d_leaves;
    a.nslots = d_leaves ? nslots : idx->cnt[0];
    a.rho_sorted = d_rho_sorted;
    a.inroi = d_inroi;
    a.pairs = nullptr;
    const int64_t nl = a.nslots;
    cudaError_t e;
    if (call.kernel == SF_K_EPAN)
        e = call.clip ? launch_points_tc<SF_K_EPAN, true>(prec, a, nl, s) : launch_points_tc<SF_K_EPAN, false>(prec, a, nl, s);
    else
        e = call.clip ? launch_points_tc<SF_K_GAUSS3, true>(prec, a, nl, s) : launch_points_tc<SF_K_GAUSS3, false>(prec, a, nl, s);
    SF_TRY_CUDA(e);
    return SF_OK;
}

sf_status density_points(sf_index *idx, const sf_box &roi, const DensityCall &call,
                         const int *d_leaves, int64_t nslots, float *d_rho_sorted,
                         uint8_t *d_inroi, cudaStream_t s, unsigned long long *d_pairs) {
    PointsArgs a;
    a.e = engine_args(idx, roi, call);
    a.leaves = d_leaves;
    a.nslots = d_leaves ? nslots : idx->cnt[0];
    a.rho_sorted = d_rho_sorted;
    a.inroi = d_inroi;
    a.pairs = d_pairs;
    cudaError_t e = (call.kernel == SF_K_EPAN)
                        ? dispatch_points<SF_K_EPAN>(call.bw, call.clip != 0, a, a.nslots, s)
                        : dispatch_points<SF_K_GAUSS3>(call.bw, call.clip != 0, a, a.nslots, s);
    SF_TRY_CUDA(e);
    return SF_OK;
}

}  // namespace sf

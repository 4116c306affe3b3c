// sf_fields.cu -- a density grid sampled at the nodes of another grid by
// trilinear interpolation (Sec. 3.1: the density at any position inside B from
// the eight nodes around it), scaled and optionally added to the destination.
//
// This serves the consumers of finished grids rather than the estimator: a
// view cache that answers a small pan or zoom from a grid computed over a
// larger box, and the precomputed-field conditions of the paper's study
// (Sec. 5: one fixed 64^3 field, or 64^3 and 128^3 fields blended by the
// scale), which read a global field at the nodes of the current view.
//
// One thread per destination column of 8 nodes; a node's cell in the source grid and
// its weights are formed in FP64 once per axis (the source grid's node coordinates as
// lo + i s, like every grid of the library). The eight-point weighted sum is that of FP64
// rounded once to float: evaluated in pairs of floats, and again in FP64 where the pairs'
// error leaves the rounding open.
#include <cmath>

#include "sf_internal.cuh"

namespace sf {

namespace {

struct Axes {
    double lo[3], inv[3];        // source: origin, 1 / spacing
    int n[3];                    // source nodes per axis
    double dlo[3], ds[3];        // destination: origin and spacing
    int dn[3];                   // destination nodes per axis
    double blo[3], bhi[3];       // the source box (closed)
};

// A destination node's place on one axis: the source cell (-1: outside the box), and the
// weights of its two nodes as float pairs (hi + lo).
struct AxisPlace {
    int c;
    float w0h, w0l, w1h, w1l;
};

__device__ __forceinline__ double axis_cell(const Axes &A, int k, int id, int &c, bool &in) {
    const double r = __dadd_rn(A.dlo[k], __dmul_rn((double)id, A.ds[k]));
    in = r >= A.blo[k] && r <= A.bhi[k];
    const double v = (r - A.lo[k]) * A.inv[k];
    int ci = (int)floor(v);
    c = ci < 0 ? 0 : (ci > A.n[k] - 2 ? A.n[k] - 2 : ci);
    return v - (double)c;
}

// Float pairs: s + e = a + b exactly (Knuth's two-sum: no ordering of |a| and |b| needed).
__device__ __forceinline__ float sum2(float a, float b, float &e) {
    const float s = __fadd_rn(a, b), bb = __fsub_rn(s, a);
    e = __fadd_rn(__fsub_rn(a, __fsub_rn(s, bb)), __fsub_rn(b, bb));
    return s;
}
// a w0 + b w1 and (ah + al) w0 + (bh + bl) w1 in float pairs.
__device__ __forceinline__ float mix1(float a, float b, const AxisPlace &p, float &lo) {
    const float s = __fmul_rn(a, p.w0h), t = __fmul_rn(b, p.w1h);
    const float es = fmaf(a, p.w0l, fmaf(a, p.w0h, -s)), et = fmaf(b, p.w1l, fmaf(b, p.w1h, -t));
    float e;
    const float r = sum2(s, t, e);
    lo = e + (es + et);
    return r;
}
__device__ __forceinline__ float mix2(float ah, float al, float bh, float bl, const AxisPlace &p, float &lo) {
    const float s = __fmul_rn(ah, p.w0h), t = __fmul_rn(bh, p.w1h);
    const float es = fmaf(al, p.w0h, fmaf(ah, p.w0l, fmaf(ah, p.w0h, -s)));
    const float et = fmaf(bl, p.w1h, fmaf(bh, p.w1l, fmaf(bh, p.w1h, -t)));
    float e;
    const float r = sum2(s, t, e);
    lo = e + (es + et);
    return r;
}

// float to double by its bits (the conversion instruction runs at the FP64 rate, a 64th of FP32's:
// 2 x 4096 x 1024 nodes in FP64 took 0.57 ms with it, 0.38 so).
__device__ __forceinline__ double widen(float f) {
    const uint32_t u = __float_as_uint(f), m = u & 0x7fffffffu;
    if (m - 0x00800000u < 0x7f000000u) return __hiloint2double((int)((u & 0x80000000u) | ((m >> 3) + 0x38000000u)), (int)(u << 29));
    return m == 0u ? __hiloint2double((int)u, 0) : (double)f;
}

// The same in FP64, for nodes that the float pairs cannot settle (x, y, z: the weights of the
// cell's lower and upper node).
__device__ __noinline__ float resample_fp64(const float *__restrict__ f, int64_t row, int64_t slice, double2 x,
                                            double2 y, double2 z, float weight) {
    const double w[4] = {x.x * y.x, x.y * y.x, x.x * y.y, x.y * y.y};
    double val = 0.0;
#pragma unroll
    for (int t = 0; t < 8; ++t)
        val += w[t & 3] * (t >> 2 ? z.y : z.x) * widen(__ldg(f + (t & 1) + ((t >> 1) & 1) * row + (t >> 2) * slice));
    return (float)(widen(weight) * val);
}

// What bounds it: with every node's cell, weights and sum in FP64 (about 70 instructions
// at 2 lanes a clock and SM) it ran at the FP64 rate: 108 us for 96^3 nodes. Per-axis
// places (one FP64 evaluation per block and axis node) leave the sum, about 120 FP32
// instructions in float pairs: 8.8 us (11 with cold caches), bounded by issue and the blocks'
// start-up (7.4 MB of compulsory traffic would take 1.1 us). Settling the rounding costs one to
// two us of a call (in a row: 10.3 us without, 11.3 to 12.3 with), the time that the ten or so
// open nodes of 96^3 take in FP64, each on its own. The pairs are good to 2^-41.8 of a sum of
// non-negative terms (2^-45.3, 2^-43.6 and 2^-42.9 for the three steps, whose low parts grow
// to 2^-20.7; 2^-44.7 for the weight; 2^-48 a pair of weights); kRsError covers that and the
// 2^-49 of FP64, so where both ends of the interval round to one float, FP64 rounds to
// it too: all but about one node in 90,000.
constexpr float kRsError = 0x1p-41f;
// A block takes 256 columns of up to 8 nodes. A warp is 32 nodes wide in x, or narrower (8, in
// grids narrower than that 2) where an eighth fewer warps cover the grid so (2 x 4096 x 1024
// nodes of a signed field, all FP64: 14.5 ms with 32 always, 0.38 now; 33 x 300 x 300: 397
// us and 177). Columns are shorter where the blocks would not fill the chip (33^3 nodes of a signed
// field: 41 us a call with 8, 26 now).
constexpr int kRsThreads = 256, kRsZ = 8;
constexpr int kRsBlocks = 2 * 152;

template <bool TALL>
__global__ void __launch_bounds__(kRsThreads)
    k_resample(const float *__restrict__ src, Axes A, int xlog, int z_nodes, float weight, int accumulate, float *__restrict__ dst,
               unsigned long long *outside) {
    __shared__ AxisPlace P[kRsThreads];  // of the block's nodes in x, y and z
    __shared__ double2 U[kRsThreads];    // their weights in FP64
    const int zlen = TALL ? kRsZ : z_nodes;  // (a constant saves 1 us of 12 at 96^3)
    const int tid = threadIdx.x, bx = 1 << xlog, by = kRsThreads >> xlog;
    const int g0[3] = {(int)blockIdx.x * bx, (int)blockIdx.y * by, (int)blockIdx.z * zlen};
    if (tid < bx + by + zlen) {
        const int k = tid < bx ? 0 : (tid < bx + by ? 1 : 2);
        const int i = g0[k] + tid - (k == 0 ? 0 : (k == 1 ? bx : bx + by));
        AxisPlace p;
        bool in;
        const double u = axis_cell(A, k, i, p.c, in), v = 1.0 - u;
        if (!in) p.c = -1;
        U[tid] = make_double2(v, u);
        p.w0h = (float)v;
        p.w0l = (float)(v - (double)p.w0h);
        p.w1h = (float)u;
        p.w1l = (float)(u - (double)p.w1h);
        // a node a rounding past the box's face, or so near a source node that its weight's
        // pair could leave the normal range: FP64 (no test of the sum passes a NaN)
        // (1 - u is 0 or at least 2^-53; the high word of u is 0 for u = 0)
        if (p.w0h < 0.f || (p.w1h < 0x1p-64f && __double2hiint(u) != 0)) p.w0h = NAN;
        P[tid] = p;
    }
    __syncthreads();
    const int ix = g0[0] + (tid & (bx - 1)), iy = g0[1] + (tid >> xlog);
    unsigned long long out_cnt = 0;
    if (ix < A.dn[0] && iy < A.dn[1]) {
        const AxisPlace px = P[tid & (bx - 1)], py = P[bx + (tid >> xlog)];
        const int nz = min(zlen, A.dn[2] - g0[2]);
        const int64_t row = A.n[0], slice = (int64_t)A.n[0] * A.n[1];
        float *d = dst + ((int64_t)g0[2] * A.dn[1] + iy) * A.dn[0] + ix;
        const int64_t dslice = (int64_t)A.dn[0] * A.dn[1];
        const float zero = weight * 0.f;  // a negative weight's zero is -0
#pragma unroll 2
        for (int z = 0; z < nz; ++z) {
            const AxisPlace &pz = P[bx + by + z];
            float res = zero;
            if (px.c >= 0 && py.c >= 0 && pz.c >= 0) {
                const float *f = src + pz.c * slice + py.c * row + px.c;
                const float f000 = __ldg(f), f100 = __ldg(f + 1);
                const float f010 = __ldg(f + row), f110 = __ldg(f + row + 1);
                const float f001 = __ldg(f + slice), f101 = __ldg(f + slice + 1);
                const float f011 = __ldg(f + slice + row), f111 = __ldg(f + slice + row + 1);
                float l00, l10, l01, l11, l0, l1, lo;
                const float h00 = mix1(f000, f100, px, l00), h10 = mix1(f010, f110, px, l10);
                const float h01 = mix1(f001, f101, px, l01), h11 = mix1(f011, f111, px, l11);
                const float h0 = mix2(h00, l00, h10, l10, py, l0), h1 = mix2(h01, l01, h11, l11, py, l1);
                const float hi = mix2(h0, l0, h1, l1, pz, lo);
                const float r = __fmul_rn(weight, hi);
                const float tail = fmaf(weight, lo, fmaf(weight, hi, -r)), err = kRsError * fabsf(r);
                res = r + (tail + err);
                const uint32_t any = __float_as_uint(f000) | __float_as_uint(f100) | __float_as_uint(f010) |
                                     __float_as_uint(f110) | __float_as_uint(f001) | __float_as_uint(f101) |
                                     __float_as_uint(f011) | __float_as_uint(f111);
                // FP64 where the rounding is open, a negative value may cancel others or a partial
                // product may have left the normal range (infinities and NaN among them);
                // all-zero neighbours and a weight of 0 are exact
                bool plain = (int)any >= 0 && hi > 1.0e-28f && hi < 1.0e37f && fabsf(r) > 1.0e-28f && fabsf(r) < 1.0e37f &&
                             res == r + (tail - err);
                if (any == 0 || (weight == 0.f && (int)any > 0 && hi < 1.0e37f)) {
                    res = zero;
                    plain = true;
                }
                if (!plain)
                    res = resample_fp64(f, row, slice, U[tid & (bx - 1)], U[bx + (tid >> xlog)], U[bx + by + z], weight);
            } else {
                ++out_cnt;
            }
            float *o = d + z * dslice;
            *o = accumulate ? *o + res : res;
        }
    }
    if (outside) {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) out_cnt += __shfl_xor_sync(0xffffffffu, out_cnt, o);
        if ((threadIdx.x & 31) == 0 && out_cnt) atomicAdd(outside, out_cnt);
    }
}

}  // namespace

}  // namespace sf

using namespace sf;

extern "C" sf_status sf_resample_grid(const float *d_src, const sf_box *src_box, const int32_t src_dims[3],
                                      const sf_box *dst_box, const int32_t dst_dims[3], float weight,
                                      int32_t accumulate, float *d_dst, int64_t *h_outside,
                                      void *stream) {
    clear_error();
    if (!d_src || !src_box || !src_dims || !dst_box || !dst_dims || !d_dst)
        return fail(SF_ERR_INVALID_ARG, "sf_resample_grid: NULL argument");
    if (!std::isfinite(weight)) return fail(SF_ERR_INVALID_ARG, "sf_resample_grid: weight must be finite");
    Axes A;
    for (int k = 0; k < 3; ++k) {
        const double lo = src_box->lo[k], hi = src_box->hi[k], dlo = dst_box->lo[k], dhi = dst_box->hi[k];
        if (!std::isfinite(lo) || !std::isfinite(hi) || !(hi > lo) || !std::isfinite(dlo) ||
            !std::isfinite(dhi) || !(dhi > dlo))
            return fail(SF_ERR_INVALID_ARG, "sf_resample_grid: axis %d boxes must satisfy lo < hi", k);
        if (src_dims[k] < 2 || src_dims[k] > 4096 || dst_dims[k] < 2 || dst_dims[k] > 4096)
            return fail(SF_ERR_INVALID_ARG, "sf_resample_grid: dims[%d] outside [2, 4096]", k);
        A.lo[k] = lo;
        A.n[k] = src_dims[k];
        A.inv[k] = 1.0 / ((hi - lo) / (double)(src_dims[k] - 1));
        A.dlo[k] = dlo;
        A.dn[k] = dst_dims[k];
        A.ds[k] = (dhi - dlo) / (double)(dst_dims[k] - 1);
        A.blo[k] = lo;
        A.bhi[k] = hi;
    }
    cudaStream_t s = (cudaStream_t)stream;
    Scratch sc(s);
    unsigned long long *cnt = nullptr;
    if (h_outside) {
        cnt = sc.get<unsigned long long>(1);
        SF_TRY_SCRATCH(sc);
        SF_TRY_CUDA(cudaMemsetAsync(cnt, 0, sizeof *cnt, s));
    }
    auto ceil_div = [](int n, int d) { return (n + d - 1) / d; };
    auto warps = [&](int lg) { return (int64_t)ceil_div(A.dn[0], 1 << lg) * ceil_div(A.dn[1], 32 >> lg); };
    int xlog = 5, zlen = kRsZ;
    for (int lg = 4; lg >= (A.dn[0] < 8 ? 1 : 3); --lg)
        if (8 * warps(lg) <= 7 * warps(xlog)) xlog = lg;
    const int bx = ceil_div(A.dn[0], 1 << xlog), by = ceil_div(A.dn[1], kRsThreads >> xlog);
    while (zlen > 1 && (int64_t)bx * by * ceil_div(A.dn[2], zlen) < kRsBlocks) zlen /= 2;
    const dim3 grid(bx, by, ceil_div(A.dn[2], zlen));
    SF_TRY_CUDA(launch(zlen == kRsZ ? k_resample<true> : k_resample<false>, grid, dim3(kRsThreads), 0, s, d_src, A, xlog, zlen, weight, accumulate ? 1 : 0, d_dst, cnt));
    if (h_outside) {
        unsigned long long h = 0;
        SF_TRY_CUDA(cudaMemcpyAsync(&h, cnt, sizeof h, cudaMemcpyDeviceToHost, s));
        SF_TRY_CUDA(cudaStreamSynchronize(s));
        *h_outside = (int64_t)h;
    }
    return SF_OK;
}

// ---------------------------------------------------------------------------
// Selection volume boundary (sf_iso_surface)
// ---------------------------------------------------------------------------
namespace sf {

namespace {

struct IsoGrid {
    int n[3];
    double lo[3], s[3];
    double t;
    float tf;  // the largest float up to t
};

// Corner c (0..3) of the tetrahedron of ordering o (0..5), as 0/1 offsets in a bitmask
// x | y << 1 | z << 2: corners 0, e_a, e_a + e_b, (1,1,1) for the orderings
// (x,y,z), (x,z,y), (y,x,z), (y,z,x), (z,x,y), (z,y,x).
__device__ __forceinline__ int tet_corner(int o, int c) {
    const int a = o >> 1;                                            // first axis: 0,0,1,1,2,2
    const int b = (o == 0 || o == 5) ? 1 : ((o == 1 || o == 3) ? 2 : 0);  // second axis
    if (c == 0) return 0;
    if (c == 1) return 1 << a;
    if (c == 2) return (1 << a) | (1 << b);
    return 7;
}

// The triangles (1 or 2) of one tetrahedron that the surface cuts, at out.
__device__ __forceinline__ int tet_triangles(const IsoGrid &G, const float *__restrict__ grid, int cx, int cy, int cz,
                                             int o, float *out) {
    // the two node coordinates of the cell on each axis; corner c's are picked by its bits
    double X[3][2], f[4];
    const int cell[3] = {cx, cy, cz};
    int m[4];
    bool in[4];
    int nin = 0;
#pragma unroll
    for (int k = 0; k < 3; ++k)
#pragma unroll
        for (int e = 0; e < 2; ++e) X[k][e] = G.lo[k] + (double)(cell[k] + e) * G.s[k];
    double cen[3] = {0.0, 0.0, 0.0};
#pragma unroll
    for (int c = 0; c < 4; ++c) {
        m[c] = tet_corner(o, c);
        const int ix = cx + (m[c] & 1), iy = cy + ((m[c] >> 1) & 1), iz = cz + (m[c] >> 2);
        f[c] = (double)__ldg(&grid[((int64_t)iz * G.n[1] + iy) * G.n[0] + ix]);
        in[c] = f[c] > G.t;
        nin += in[c];
        if (in[c])
#pragma unroll
            for (int k = 0; k < 3; ++k) cen[k] += (m[c] >> k) & 1 ? X[k][1] : X[k][0];
    }
    const int ntri = nin == 2 ? 2 : 1;
#pragma unroll
    for (int k = 0; k < 3; ++k) cen[k] /= (double)nin;
    auto pick = [&](int c) { return c < 2 ? (c == 0 ? f[0] : f[1]) : (c == 2 ? f[2] : f[3]); };
    auto bits = [&](int c) { return c < 2 ? (c == 0 ? m[0] : m[1]) : (c == 2 ? m[2] : m[3]); };
    auto cross = [&](int a, int b, double *r) {
        const double fa = pick(a), w = (G.t - fa) / (pick(b) - fa);
        const int ma = bits(a), mb = bits(b);
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            const double pa = (ma >> k) & 1 ? X[k][1] : X[k][0], pb = (mb >> k) & 1 ? X[k][1] : X[k][0];
            r[k] = pa + w * (pb - pa);
        }
    };
    double V[4][3];  // the crossings: 3 for one triangle, 4 for two (0 1 2 and 0 2 3)
    // pairs (a, b) of corners whose edge is crossed: the lone corner with each other one,
    // or the two inside corners (I, J) with the two outside (K, L): I K, I L, J L, J K
    int a0 = 0, a2 = 0, b0 = 0, b1 = 0, b2 = 0;
    if (ntri == 1) {
#pragma unroll
        for (int c = 0; c < 4; ++c)
            if (in[c] == (nin == 1)) a0 = c;  // the corner on its own side
        a2 = a0;
        b0 = a0 == 0 ? 1 : 0;
        b1 = a0 <= 1 ? 2 : 1;
        b2 = a0 <= 2 ? 3 : 2;
    } else {
        int I = -1, J = -1, K = -1, L = -1;
#pragma unroll
        for (int c = 0; c < 4; ++c) {
            if (in[c]) {
                if (I < 0) I = c; else J = c;
            } else {
                if (K < 0) K = c; else L = c;
            }
        }
        a0 = I;
        a2 = J;
        b0 = K;
        b1 = b2 = L;
    }
    cross(a0, b0, V[0]);
    cross(a0, b1, V[1]);
    cross(a2, b2, V[2]);
    cross(a2, b0, V[3]);
#pragma unroll
    for (int q = 0; q < 2; ++q) {
        if (q >= ntri) break;
        const double *A = V[0], *B = V[1 + q], *C = V[2 + q];
        const double e1[3] = {B[0] - A[0], B[1] - A[1], B[2] - A[2]};
        const double e2[3] = {C[0] - A[0], C[1] - A[1], C[2] - A[2]};
        const double n[3] = {e1[1] * e2[2] - e1[2] * e2[1], e1[2] * e2[0] - e1[0] * e2[2],
                             e1[0] * e2[1] - e1[1] * e2[0]};
        const double dn = n[0] * (A[0] - cen[0]) + n[1] * (A[1] - cen[1]) + n[2] * (A[2] - cen[2]);
        const bool flip = dn < 0.0;  // toward the inside: flip
        float *w = out + 9 * q;
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            w[k] = (float)A[k];
            w[3 + k] = (float)(flip ? C[k] : B[k]);
            w[6 + k] = (float)(flip ? B[k] : C[k]);
        }
    }
    return ntri;
}

// A warp takes 32 STEPS consecutive cells (x fastest) in STEPS steps of 32, a block those of
// its eight warps. A cell is first only the 8-bit mask of its corners above the threshold: (double)f > t
// exactly when f > the largest float up to t, so no FP64 is needed to count. Count
// pass: the block's triangles. Emit pass (blocks with any): the warps' cut tetrahedra
// are queued in shared memory and worked off 32 at a time, so that FP64 runs
// with full warps; 32 tetrahedra's triangles are collected there and written in one run.
// With one thread per cell, every corner of every tetrahedron compared in FP64 in both
// passes and the few cut cells of a warp on their own lanes, 192^3 nodes and 0.85
// million triangles took 4.5 ms (FP64 and divergence): 0.03 ms to count and 0.34 ms to
// emit now, still FP64 (a division, six products and the orientation a crossing).
//
// STEPS is 8, and 1 below four blocks of 8 an SM: there a warp's chain of FP64 batches sets the
// time (16^3 nodes of noise, five cut tetrahedra a cell: 580 us a call with 8, 125 with 1).
constexpr int kIsoWarps = 8;
constexpr int kIsoSteps = 8;
constexpr int kIsoSmall = 4 * 152;  // blocks of 8 steps below which a warp takes one step

// Bit c of a tetrahedron's mask = corner c of the cell (x | y << 1 | z << 2).
__device__ __forceinline__ int tet_mask(int o) {
    return 1 | (1 << tet_corner(o, 1)) | (1 << tet_corner(o, 2)) | (1 << 7);
}
__device__ __forceinline__ int tet_count(unsigned cell, int o) {  // triangles of tetrahedron o
    const int n = __popc(cell & tet_mask(o));
    return n == 0 || n == 4 ? 0 : (n == 2 ? 2 : 1);
}

// The cell's corner mask (0 for cells past the end).
__device__ __forceinline__ unsigned cell_mask(const IsoGrid &G, const float *__restrict__ grid, int64_t cell,
                                              int64_t nc, int &cx, int &cy, int &cz) {
    if (cell >= nc) return 0u;
    const uint32_t mx = G.n[0] - 1, my = G.n[1] - 1;
    if (nc <= 0x7fffffff) {
        const uint32_t c = (uint32_t)cell, row = c / mx;
        cx = (int)(c - row * mx);
        cz = (int)(row / my);
        cy = (int)(row - (uint32_t)cz * my);
    } else {
        const int64_t row = cell / mx;
        cx = (int)(cell - row * mx);
        cz = (int)(row / my);
        cy = (int)(row - (int64_t)cz * my);
    }
    const float *f = grid + ((int64_t)cz * G.n[1] + cy) * G.n[0] + cx;
    const int64_t row = G.n[0], slice = (int64_t)G.n[0] * G.n[1];
    unsigned m = 0;
#pragma unroll
    for (int c = 0; c < 8; ++c)
        m |= (unsigned)(__ldg(f + (c & 1) + ((c >> 1) & 1) * row + (c >> 2) * slice) > G.tf) << c;
    return m;
}

// 256-entry table of a cell mask's triangles (low byte) and cut tetrahedra (high byte).
__device__ __forceinline__ void iso_table(uint16_t *table) {
    int tri = 0, cut = 0;
    for (int o = 0; o < 6; ++o) {
        const int t = tet_count(threadIdx.x, o);
        tri += t;
        cut += t > 0;
    }
    table[threadIdx.x] = (uint16_t)(tri | cut << 8);
    __syncthreads();
}

template <int STEPS>
__global__ void __launch_bounds__(kIsoWarps * 32)
    k_iso_count(const float *__restrict__ grid, IsoGrid G, int64_t nc, uint32_t *__restrict__ cnt) {
    __shared__ uint16_t table[256];
    __shared__ uint32_t wsum[kIsoWarps];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    iso_table(table);
    uint32_t t = 0;
    const int64_t c0 = ((int64_t)blockIdx.x * kIsoWarps + warp) * (STEPS * 32) + lane;
    int cx, cy, cz;
#pragma unroll 2
    for (int s = 0; s < STEPS; ++s) t += table[cell_mask(G, grid, c0 + 32 * s, nc, cx, cy, cz)] & 255u;
    t = __reduce_add_sync(0xffffffffu, t);
    if (lane == 0) wsum[warp] = t;
    __syncthreads();
    if (threadIdx.x == 0) {
        uint32_t b = 0;
        for (int w = 0; w < kIsoWarps; ++w) b += wsum[w];
        cnt[blockIdx.x] = b;
    }
}

struct IsoWarpSmem {
    uint32_t queue[32 + 32 * 6 + 32];  // cell of the warp (8 bits) | tetrahedron << 8
    float tri[32 * 18];           // the triangles of 32 tetrahedra
};

template <int STEPS>
__global__ void __launch_bounds__(kIsoWarps * 32)
    k_iso_emit(const float *__restrict__ grid, IsoGrid G, int64_t nc, const uint32_t *__restrict__ cnt,
               const uint32_t *__restrict__ off, float *__restrict__ tris) {
    __shared__ uint16_t table[256];
    __shared__ uint32_t wsum[kIsoWarps];
    __shared__ IsoWarpSmem W[kIsoWarps];
    if (cnt[blockIdx.x] == 0) return;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const unsigned lt = (1u << lane) - 1u;
    iso_table(table);
    const int64_t w0 = ((int64_t)blockIdx.x * kIsoWarps + warp) * (STEPS * 32);
    unsigned mask[STEPS];
    uint32_t t = 0;
    int cx, cy, cz;
#pragma unroll
    for (int s = 0; s < STEPS; ++s) {
        mask[s] = cell_mask(G, grid, w0 + 32 * s + lane, nc, cx, cy, cz);
        t += table[mask[s]] & 255u;
    }
    t = __reduce_add_sync(0xffffffffu, t);
    if (lane == 0) wsum[warp] = t;
    __syncthreads();
    int64_t at = off[blockIdx.x];  // the warp's next triangle
    for (int w = 0; w < warp; ++w) at += wsum[w];
    IsoWarpSmem &S = W[warp];
    int queued = 0;
    auto drain = [&](int first, int n) {  // queued tetrahedra first, ..., first + n - 1 (n at most 32)
        int o = 0, ntri = 0;
        if (lane < n) {
            const uint32_t e = S.queue[first + lane];
            o = (int)(e >> 8);
            ntri = tet_count(cell_mask(G, grid, w0 + (e & 255u), nc, cx, cy, cz), o);
        }
        const unsigned two = __ballot_sync(0xffffffffu, ntri == 2);
        if (lane < n) tet_triangles(G, grid, cx, cy, cz, o, &S.tri[9 * (lane + __popc(two & lt))]);
        __syncwarp();
        const int total = n + __popc(two);
        for (int i = lane; i < 9 * total; i += 32) tris[9 * at + i] = S.tri[i];
        at += total;
        __syncwarp();
    };
#pragma unroll 1
    for (int s = 0; s < STEPS; ++s) {
        unsigned m = 0;
#pragma unroll
        for (int k = 0; k < STEPS; ++k)
            if (k == s) m = mask[k];
        const int cuts = table[m] >> 8;
        int before = cuts;  // inclusive scan over the lanes
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) {
            const int v = __shfl_up_sync(0xffffffffu, before, d);
            if (lane >= d) before += v;
        }
        const int total = __shfl_sync(0xffffffffu, before, 31);
        if (total == 0) continue;
        int p = queued + before - cuts;
        if (cuts)
            for (int o = 0; o < 6; ++o)
                if (tet_count(m, o)) S.queue[p++] = (uint32_t)(32 * s + lane) | (uint32_t)o << 8;
        queued += total;
        __syncwarp();
        int done = 0;
        for (; queued - done >= 32; done += 32) drain(done, 32);
        queued -= done;  // fewer than 32 are left: to the front
        const uint32_t e = S.queue[done + lane];
        __syncwarp();
        if (lane < queued) S.queue[lane] = e;
        __syncwarp();
    }
    if (queued) drain(0, queued);
}

}  // namespace

}  // namespace sf

extern "C" sf_status sf_iso_surface(const float *d_grid, const sf_box *roi, const int32_t dims[3],
                                    double threshold, float *d_tris, int64_t capacity, int64_t *h_ntri,
                                    void *stream) {
    clear_error();
    if (!d_grid || !roi || !dims || !h_ntri) return fail(SF_ERR_INVALID_ARG, "sf_iso_surface: NULL argument");
    if (!std::isfinite(threshold)) return fail(SF_ERR_INVALID_ARG, "sf_iso_surface: threshold must be finite");
    if (capacity < 0 || (capacity > 0 && !d_tris))
        return fail(SF_ERR_INVALID_ARG, "sf_iso_surface: bad capacity / output");
    IsoGrid G;
    for (int k = 0; k < 3; ++k) {
        if (!std::isfinite(roi->lo[k]) || !std::isfinite(roi->hi[k]) || !(roi->hi[k] > roi->lo[k]))
            return fail(SF_ERR_INVALID_ARG, "sf_iso_surface: roi axis %d must satisfy lo < hi", k);
        if (dims[k] < 2 || dims[k] > 4096)
            return fail(SF_ERR_INVALID_ARG, "sf_iso_surface: dims[%d] outside [2, 4096]", k);
        G.n[k] = dims[k];
        G.lo[k] = roi->lo[k];
        G.s[k] = (roi->hi[k] - roi->lo[k]) / (double)(dims[k] - 1);
    }
    G.t = threshold;
    G.tf = (float)threshold;
    if ((double)G.tf > threshold) G.tf = nextafterf(G.tf, -INFINITY);
    cudaStream_t s = (cudaStream_t)stream;
    const int64_t nc = (int64_t)(G.n[0] - 1) * (G.n[1] - 1) * (G.n[2] - 1);
    const bool small = nc < (int64_t)kIsoSmall * kIsoWarps * kIsoSteps * 32;
    const int64_t cells = kIsoWarps * 32 * (small ? 1 : kIsoSteps), nb = (nc + cells - 1) / cells;
    Scratch sc(s);
    uint32_t *cnt = sc.get<uint32_t>(nb);
    uint32_t *off = sc.get<uint32_t>(nb);
    uint32_t *tot = sc.get<uint32_t>(1);
    SF_TRY_SCRATCH(sc);
    SF_TRY_CUDA(launch(small ? k_iso_count<1> : k_iso_count<kIsoSteps>, dim3((unsigned)nb), dim3(kIsoWarps * 32), 0, s,
                       d_grid, G, nc, cnt));
    SF_TRY(scan_u32(cnt, off, nb, tot, s));
    uint32_t h = 0;
    SF_TRY_CUDA(cudaMemcpyAsync(&h, tot, sizeof h, cudaMemcpyDeviceToHost, s));
    SF_TRY_CUDA(cudaStreamSynchronize(s));
    *h_ntri = h;
    if ((int64_t)h > capacity) {
        if (capacity == 0 && !d_tris) return SF_OK;   // counting only
        return fail(SF_ERR_CAPACITY, "sf_iso_surface: %u triangles exceed capacity %lld", h, (long long)capacity);
    }
    if (h > 0)
        SF_TRY_CUDA(launch(small ? k_iso_emit<1> : k_iso_emit<kIsoSteps>, dim3((unsigned)nb), dim3(kIsoWarps * 32), 0, s,
                           d_grid, G, nc, (const uint32_t *)cnt, (const uint32_t *)off, d_tris));
    return SF_OK;
}

// projection.cu -- spatial projection (Sec. 2.4) on sm_103a.
//
// Contrast c was acquired on its own grid of M_c voxels; the 3 x 4 affine A_c
// maps its voxel coordinates (i, j, k, 1) to reconstruction voxel
// coordinates.  The reslicing Psi_c interpolates the K maps trilinearly at
// A_c m; acquisition voxels whose point falls outside the reconstruction grid
// carry no data term.  The likelihood becomes l(y) = sum_c l_c(Psi_c y), with
// gradient sum_c Psi_c' g_c and, for the Hessian, the block-diagonal
// majoriser sum_c Psi_c' H_c (the interpolation weights of an inside voxel are
// non-negative and sum to one).
//
//   k_grad_hess_proj  per acquisition voxel of one contrast: interpolate the
//                     maps (8 corners), then the same per-contrast voxel model
//                     as k_grad_hess (voxel_model.cuh); writes g_c and H_c (GhPlanes)
//                     and the contrast's NLL
//   k_push_all        per reconstruction voxel: gathers, over every contrast,
//                     the acquisition voxels whose interpolation stencil holds
//                     it (a box around A_c^-1 n) with the pull's own weights,
//                     so the push is the exact adjoint of the pull and its sum
//                     order is fixed (no atomics); writes g and H once
//   k_pull / k_push   Psi_c u and Psi_c' u for any number of channels
//
// Coordinates are float32; pull and push evaluate them with the same
// instructions, so both see identical weights.
#include <algorithm>
#include <cmath>
#include <cstdio>
#include <cstring>
#include <string>

#include "mpm_internal.cuh"
#include "voxel_model.cuh"

namespace mpm {

struct ProjC {
    int mx, my, mz;
    long long M;
    float A[12];      // acquisition voxel (i, j, k, 1) -> reconstruction coordinates
    float Ai[12];     // the inverse map
    float ext[3];     // half-extent of A^-1 applied to the cube (-1, 1)^3
    float iA0;        // 1 / A[0], or 0 where lines along i do not run along x (|A[0]| < 1/2)
    int shifted;      // A is a shift by whole voxels, t: voxel m pulls n = m + t alone
    int t[3];
};

struct DevProj {
    int C;
    ProjC c[MPM_MAX_CONTRASTS];
};

// g_c and H_c of an acquisition grid of M voxels, in planes of 16-byte vectors
// so that neighbouring lanes read and write neighbouring vectors (one record
// of 64 B per voxel made each of the push's loads touch 16 lines and took
// every cycle of L1):
//   q0 = (g0, g1, g2, H00)  q1 = (H01, H02, H11, H12)  h22 = H22
// and for a contrast with an MT pulse also
//   q2 = (g3, H03, H13, H23)  h33 = H33 (as (H22, H33) pairs in place of h22).
// Without an MT pulse nothing depends on map 3: 36 B per voxel instead of 56.
struct GhPlanes {
    float4 *q0, *q1, *q2;
    float* h22;
    float2* h22_33;
};

__host__ __device__ inline GhPlanes gh_planes(void* base, long long M)
{
    GhPlanes b;
    float* f = static_cast<float*>(base);
    b.q0 = reinterpret_cast<float4*>(f);
    b.q1 = reinterpret_cast<float4*>(f + 4 * M);
    b.q2 = reinterpret_cast<float4*>(f + 8 * M);
    b.h22 = f + 8 * M;
    b.h22_33 = reinterpret_cast<float2*>(f + 12 * M);
    return b;
}

// Floats per voxel of the buffers (at least 9 with three maps, 14 with four).
__host__ __device__ constexpr int gh_floats(int K) { return (K + K * (K + 1) / 2 + 3) / 4 * 4; }

// Per-contrast g_c / H_c buffers of the projected voxel pass.
struct ProjBufs {
    float4* gh[MPM_MAX_CONTRASTS];
};

// Blocks of the two kernels below take compact tiles, so that the neighbouring
// rows and planes they gather from stay in L1 (both kernels at 176x240x256, three
// scans: 2.16 ms with 8 x 4 x 8, 2.18 with 8 x 8 x 4, 2.23 with 16 x 8 x 2, 2.34
// with 4 x 8 x 8, 2.39 with 32 x 4 x 2).  Thin grids take other shapes of the same
// size: with 8 x 4 x 8 for all, one warp in eight works where the grid is one
// slice (both kernels at 512x512x1 234 us, 72 with 16 x 16 x 1; 1x256x256 105 and
// 63; 320x320x4 142 and 101).
constexpr int kProjLX = 3, kProjLY = 2, kProjLZ = 3;

static VoxelTiles proj_tiles(int nx, int ny, int nz)
{
    return voxel_tiles(nx, ny, nz, kProjLX, kProjLY, kProjLZ);
}

static bool usual_tiles(const VoxelTiles& g) { return g.lx == kProjLX && g.ly == kProjLY && g.lz == kProjLZ; }

// This thread's voxel of tile t.  USUAL: the usual shape, as constants (as
// variables they cost the two kernels 0.8% at 176x240x256).
template <bool USUAL>
__device__ __forceinline__ void proj_voxel(const VoxelTiles& g, long long t, int& x, int& y, int& z)
{
    VoxelTiles u = g;
    if (USUAL) {
        u.lx = kProjLX;
        u.ly = kProjLY;
        u.lz = kProjLZ;
    }
    u.voxel(t, x, y, z);
}

// Reconstruction coordinate of acquisition voxel (i, j, k); true when it lies
// in [0, n_d - 1] on every axis.
__device__ __forceinline__ bool reslice(const ProjC& q, int i, int j, int k, int nx, int ny,
                                        int nz, float r[3])
{
#pragma unroll
    for (int d = 0; d < 3; ++d)
        r[d] = fmaf(q.A[4 * d], (float)i, fmaf(q.A[4 * d + 1], (float)j, fmaf(q.A[4 * d + 2], (float)k, q.A[4 * d + 3])));
    return r[0] >= 0.0f && r[0] <= (float)(nx - 1) && r[1] >= 0.0f && r[1] <= (float)(ny - 1) &&
           r[2] >= 0.0f && r[2] <= (float)(nz - 1);
}

// Cell corner and fractional offsets of an inside point.
struct Cell {
    int b[3];
    float f[3];
};

__device__ __forceinline__ Cell cell_of(const float r[3])
{
    Cell c;
#pragma unroll
    for (int d = 0; d < 3; ++d) {
        const float fl = floorf(r[d]);
        c.b[d] = (int)fl;
        c.f[d] = r[d] - fl;
    }
    return c;
}

// Weight of corner (cx, cy, cz) of the cell: the same product, in the same
// order, in every kernel.
__device__ __forceinline__ float corner_weight(const Cell& c, int cx, int cy, int cz)
{
    const float wx = cx ? c.f[0] : 1.0f - c.f[0];
    const float wy = cy ? c.f[1] : 1.0f - c.f[1];
    const float wz = cz ? c.f[2] : 1.0f - c.f[2];
    return wx * wy * wz;
}

// Interpolate `channels` planar reconstruction images u[ch * N + n] at the
// cell; corners past the last voxel (weight 0) count as 0.
template <int CH>
__device__ __forceinline__ void interpolate(const Cell& c, const float* __restrict__ u, long long N,
                                            int nx, int ny, int nz, float (&out)[CH])
{
#pragma unroll
    for (int ch = 0; ch < CH; ++ch) out[ch] = 0.0f;
    const long long n0 = (long long)c.b[0] + (long long)nx * (c.b[1] + (long long)ny * c.b[2]);
#pragma unroll
    for (int cz = 0; cz < 2; ++cz)
#pragma unroll
        for (int cy = 0; cy < 2; ++cy)
#pragma unroll
            for (int cx = 0; cx < 2; ++cx) {
                const bool in = c.b[0] + cx < nx && c.b[1] + cy < ny && c.b[2] + cz < nz;
                const float w = corner_weight(c, cx, cy, cz);
                const long long n = n0 + cx + (long long)nx * (cy + (long long)ny * cz);
#pragma unroll
                for (int ch = 0; ch < CH; ++ch) out[ch] = fmaf(w, in ? __ldg(u + ch * N + n) : 0.0f, out[ch]);
            }
}

// Box of acquisition voxels that can pull reconstruction voxel (x, y, z).
__device__ __forceinline__ void candidate_box(const ProjC& q, int x, int y, int z, int lo[3],
                                              int hi[3])
{
    const int md[3] = {q.mx, q.my, q.mz};
#pragma unroll
    for (int d = 0; d < 3; ++d) {
        const float a = fmaf(q.Ai[4 * d], (float)x, fmaf(q.Ai[4 * d + 1], (float)y, fmaf(q.Ai[4 * d + 2], (float)z, q.Ai[4 * d + 3])));
        const float e = q.ext[d] + 1e-3f;
        lo[d] = max(0, (int)ceilf(a - e));
        hi[d] = min(md[d] - 1, (int)floorf(a + e));
    }
}

// One axis of a reconstruction voxel at coordinate c as its pullers see it: a
// point at r in [lo, hi] with c - 1 < r < c + 1 pulls it with weight min(c + 1 -
// r, r - (c - 1)), which is the pull's 1 - f for c = floor(r) and f for c =
// floor(r) + 1 (f = r - floor(r)) with its roundings (r - c is exact for r >= c).
struct Slab {
    float below, above, lo, hi;      // c - 1, c + 1; the part of [c - 1, c + 1] in the volume
    __device__ __forceinline__ Slab(int c, int n)
        : below((float)(c - 1)), above((float)(c + 1)), lo((float)max(c - 1, 0)), hi((float)min(c + 1, n - 1)) {}
    __device__ __forceinline__ float weight(float r) const { return fminf(above - r, r - below); }
    __device__ __forceinline__ bool holds(float r) const { return (r >= lo) & (r <= hi); }
};

// Calls f(w, m) for every acquisition voxel m of contrast q that pulls
// reconstruction voxel (x, y, z), with the weight the pull uses, in a fixed
// order (f is taken by value and returned).  Each coordinate is built with
// the same fused multiply-adds as reslice(), so every weight is bit-identical
// to the pull's.  Planes and lines of the candidate box that pass the voxel by
// at a distance are skipped whole (with a margin of 1e-3 for the rounding of
// the bounds), and a line's points start and end where it enters and leaves the
// voxel's x slab: about 8 points per voxel and contrast pull it, and each point
// tested costs as much as the arithmetic of one that does.  (Boxes two points
// wide are not worth either search: without that exception the pass and push of
// 128^3 volumes without an MT scan took 338 us instead of 321 where the scans
// were turned by 45 degrees about x, 300 instead of 286 where mirrored, 96 instead
// of 92 where twice as coarse.)  A contrast that is
// the reconstruction grid shifted by whole voxels (the reference scan) is read
// at its one voxel of weight 1.
template <typename IT, typename F>
__device__ __forceinline__ F gather_pullers(const ProjC& q, int x, int y, int z, int nx, int ny,
                                            int nz, F f)
{
    if (q.shifted) {
        const int i = x - q.t[0], j = y - q.t[1], k = z - q.t[2];
        if (i >= 0 && i < q.mx && j >= 0 && j < q.my && k >= 0 && k < q.mz)
            f(1.0f, (IT)i + (IT)q.mx * ((IT)j + (IT)q.my * (IT)k));
        return f;
    }
    int lo[3], hi[3];
    candidate_box(q, x, y, z, lo, hi);
    const float xf = (float)x, yf = (float)y, zf = (float)z;
    const Slab sx(x, nx), sy(y, ny), sz(z, nz);
    // middle of the box's lines and planes, and how far r1 and r2 stray from
    // their values there
    const float ic = 0.5f * (float)(lo[0] + hi[0]), jc = 0.5f * (float)(lo[1] + hi[1]);
    const float ih = ic - (float)lo[0], jh = jc - (float)lo[1];
    const float e1 = fmaf(fabsf(q.A[4]), ih, 1.001f), e2 = fmaf(fabsf(q.A[8]), ih, 1.001f);
    const float e2p = fmaf(fabsf(q.A[9]), jh, e2);
    for (int k = lo[2]; k <= hi[2]; ++k) {
        const float kf = (float)k;
        const float t2 = fmaf(q.A[10], kf, q.A[11]);
        if (hi[2] - lo[2] > 1 && fabsf(fmaf(q.A[8], ic, fmaf(q.A[9], jc, t2)) - zf) > e2p) continue;
        const float t0 = fmaf(q.A[2], kf, q.A[3]), t1 = fmaf(q.A[6], kf, q.A[7]);
        for (int j = lo[1]; j <= hi[1]; ++j) {
            const float jf = (float)j;
            const float u1 = fmaf(q.A[5], jf, t1), u2 = fmaf(q.A[9], jf, t2);
            if (fabsf(fmaf(q.A[4], ic, u1) - yf) > e1 || fabsf(fmaf(q.A[8], ic, u2) - zf) > e2) continue;
            const float u0 = fmaf(q.A[1], jf, t0);
            const IT row = (IT)q.mx * ((IT)j + (IT)q.my * (IT)k);
            int ib = lo[0], ie = hi[0];
            if (q.iA0 != 0.0f && ie - ib > 1) {
                // r0 = x at i = c; the slab's ends within 1e-3, then exactly
                const float c = (xf - u0) * q.iA0, h = fabsf(q.iA0) + 1e-3f;
                ib = max(ib, (int)ceilf(c - h));
                ie = min(ie, (int)floorf(c + h));
                const float ab = fmaf(q.A[0], (float)ib, u0) - xf, ae = fmaf(q.A[0], (float)ie, u0) - xf;
                if (!(fabsf(ab) < 1.0f)) ++ib;
                if (!(fabsf(ae) < 1.0f)) --ie;
            }
            for (int i = ib; i <= ie; ++i) {
                const float fi = (float)i;
                const float r0 = fmaf(q.A[0], fi, u0), r1 = fmaf(q.A[4], fi, u1), r2 = fmaf(q.A[8], fi, u2);
                const float wx = sx.weight(r0), wy = sy.weight(r1), wz = sz.weight(r2);
                if (!((fminf(fminf(wx, wy), wz) > 0.0f) & sx.holds(r0) & sy.holds(r1) & sz.holds(r2))) continue;
                f(wx * wy * wz, row + (IT)i);
            }
        }
    }
    return f;
}

// ------------------------------------------------- projected voxel pass

// K: the maps contrast c depends on (3 without an MT pulse).  Bound: its
// gathers' latency and instruction issue (about 900 instructions per voxel).
// It took 419 us per contrast at 176x240x256 with 64-bit divisions for the
// voxel's indices, all corners behind branches, four maps for every contrast
// and 64 B records staged in shared memory.  Four blocks per SM (60 to 64
// registers) for more of a voxel's loads in flight: left to itself the compiler
// takes 40 or 48 registers as it happens, and this pass and the push take 2.05 ms
// at 176x240x256 instead of 1.97, 1.35 instead of 1.31 at 188x195x184 with bfloat16
// echoes and the row-sum loading.
template <int K, int PRE, typename XT, bool USUAL>
__global__ void __launch_bounds__(kBlock, 4) k_grad_hess_proj(DevProblem P, ProjC q, int c,
                                                           const float* __restrict__ y,
                                                           const XT* __restrict__ x,
                                                           const float* __restrict__ b1p,
                                                           const float* __restrict__ b1m,
                                                           float4* __restrict__ gh, double* nll,
                                                           Reduce red, VoxelTiles tg)
{
    constexpr int T = K * (K + 1) / 2;
    const long long M = q.M;
    const GhPlanes out = gh_planes(gh, M);
    Acc nll_acc;
    for (long long t = blockIdx.x; t < tg.count; t += gridDim.x) {
        int i, j, k;
        if (t + gridDim.x < tg.count) {   // the next tile's echoes and B1 values into L2
            proj_voxel<USUAL>(tg, t + gridDim.x, i, j, k);
            if (i < q.mx && j < q.my && k < q.mz) {
                const long long mn = i + (long long)q.mx * (j + (long long)q.my * k);
                for (int e = 0; e < P.n_echoes[c]; ++e) prefetch_l2(x + e * M + mn);
                if (b1p) prefetch_l2(b1p + mn);
                if (b1m) prefetch_l2(b1m + mn);
            }
        }
        proj_voxel<USUAL>(tg, t, i, j, k);
        if (i >= q.mx || j >= q.my || k >= q.mz) continue;
        const long long m = i + (long long)q.mx * (j + (long long)q.my * k);
        float G[K], H[T];
#pragma unroll
        for (int u = 0; u < K; ++u) G[u] = 0.0f;
#pragma unroll
        for (int u = 0; u < T; ++u) H[u] = 0.0f;
        float nll_v = 0.0f;
        float r[3];
        if (reslice(q, i, j, k, P.nx, P.ny, P.nz, r)) {
            float yv[K];
            interpolate<K>(cell_of(r), y, P.N, P.nx, P.ny, P.nz, yv);
            float yk[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
            for (int u = 0; u < K; ++u) yk[u] = yv[u];
            float a, r1, r2, dl, mm;
            map_params_v(yk, K, a, r1, r2, dl, mm);
            const float bp = b1p ? __ldg(b1p + m) : 1.0f;
            const float bm = b1m ? __ldg(b1m + m) : 1.0f;
            const ContrastTerms ct = contrast_terms(P, c, a, relax(P.tr[c], r1), dl, mm, bp, bm);
            accumulate_contrast<K, PRE, XT>(P, c, ct, r2, x + m, M, G, H, nll_v);
        }
        out.q0[m] = make_float4(G[0], G[1], G[2], H[tri(K, 0, 0)]);
        out.q1[m] = make_float4(H[tri(K, 0, 1)], H[tri(K, 0, 2)], H[tri(K, 1, 1)], H[tri(K, 1, 2)]);
        if (K == 4) {
            out.q2[m] = make_float4(G[K - 1], H[tri(K, 0, K - 1)], H[tri(K, 1, K - 1)], H[tri(K, 2, K - 1)]);
            out.h22_33[m] = make_float2(H[tri(K, 2, 2)], H[tri(K, K - 1, K - 1)]);
        } else {
            out.h22[m] = H[tri(K, 2, 2)];
        }
        nll_acc.add(nll_v);
    }
    Acc v[1] = {nll_acc};
    double o[1];
    if (grid_reduce<1>(v, red, o) && threadIdx.x == 0) *nll = o[0];
}

// One contrast's contribution to (g, h) of a reconstruction voxel; MT: the
// contrast depends on map 3.
template <int K, bool MT>
struct PushInto {
    float (&A)[K + K * (K + 1) / 2];      // g, then the packed H
    GhPlanes b;
    template <typename IT>
    __device__ __forceinline__ void operator()(float w, IT m)
    {
        auto add = [&](int t, float v) { A[t] = fmaf(w, v, A[t]); };
        const float4 a = __ldg(b.q0 + m), c = __ldg(b.q1 + m);
        float4 d;
        float2 e;
        if (MT) {
            d = __ldg(b.q2 + m);
            e = __ldg(b.h22_33 + m);
        } else {
            e.x = __ldg(b.h22 + m);
        }
        add(0, a.x);
        add(1, a.y);
        add(2, a.z);
        add(K + tri(K, 0, 0), a.w);
        add(K + tri(K, 0, 1), c.x);
        add(K + tri(K, 0, 2), c.y);
        add(K + tri(K, 1, 1), c.z);
        add(K + tri(K, 1, 2), c.w);
        add(K + tri(K, 2, 2), e.x);
        if constexpr (MT) {
            add(K - 1, d.x);
            add(K + tri(K, 0, K - 1), d.y);
            add(K + tri(K, 1, K - 1), d.z);
            add(K + tri(K, 2, K - 1), d.w);
            add(K + tri(K, K - 1, K - 1), e.y);
        }
    }
};

// g = sum_c Psi_c' g_c, h = sum_c Psi_c' H_c; nll = sum_c nll_c (fixed order).
// Bound: instruction issue and the gathers' L1 traffic (about 8 contributing
// voxels per contrast).  Three scans of 176x240x256 took 1468 us with 64 B
// records, 64-bit divisions, linear blocks and every point of the box tested;
// both passes together took 2.73 ms, 1.97 ms now.
// IT: an index type that holds every acquisition voxel's index.
template <int K, typename IT, bool USUAL>
__global__ void __launch_bounds__(kBlock, 4) k_push_all(DevProblem P, DevProj Q, ProjBufs B,
                                                     float* __restrict__ g, float* __restrict__ h,
                                                     const double* nll_parts, double* nll,
                                                     VoxelTiles tg)
{
    constexpr int T = K * (K + 1) / 2;
    constexpr int CH = K + T;                     // channels: g, then the packed H
    const long long N = P.N;
    if (blockIdx.x == 0 && threadIdx.x == 0 && nll) {
        double s = 0.0;
        for (int c = 0; c < Q.C; ++c) s += nll_parts[c];
        *nll = s;
    }
    for (long long t = blockIdx.x; t < tg.count; t += gridDim.x) {
        int x, y, z;
        proj_voxel<USUAL>(tg, t, x, y, z);
        if (x >= P.nx || y >= P.ny || z >= P.nz) continue;
        const long long n = x + (long long)P.nx * (y + (long long)P.ny * z);
        float A[CH];
#pragma unroll
        for (int u = 0; u < CH; ++u) A[u] = 0.0f;
        // unrolled, so each contrast's affine is read as constant operands
#pragma unroll
        for (int c = 0; c < MPM_MAX_CONTRASTS; ++c) {
            if (c >= Q.C) break;
            const ProjC& q = Q.c[c];
            const GhPlanes b = gh_planes(B.gh[c], q.M);
            if (K == 4 && P.mt[c]) gather_pullers<IT>(q, x, y, z, P.nx, P.ny, P.nz, PushInto<K, K == 4>{A, b});
            else gather_pullers<IT>(q, x, y, z, P.nx, P.ny, P.nz, PushInto<K, false>{A, b});
        }
        if (K == 4) {
            // a contrast without an MT pulse adds zero times its terms to map
            // 3's: nothing, unless they are not finite
            A[K - 1] = fmaf(0.0f, A[0], A[K - 1]);
            A[K + tri(K, 0, K - 1)] = fmaf(0.0f, A[K + tri(K, 0, 0)], A[K + tri(K, 0, K - 1)]);
            A[K + tri(K, 1, K - 1)] = fmaf(0.0f, A[K + tri(K, 0, 1)], A[K + tri(K, 1, K - 1)]);
            A[K + tri(K, 2, K - 1)] = fmaf(0.0f, A[K + tri(K, 0, 2)], A[K + tri(K, 2, K - 1)]);
            A[K + tri(K, K - 1, K - 1)] = fmaf(0.0f, A[K + tri(K, 0, 0)], A[K + tri(K, K - 1, K - 1)]);
        }
#pragma unroll
        for (int u = 0; u < K; ++u) g[u * N + n] = A[u];
#pragma unroll
        for (int u = 0; u < T; ++u) h[u * N + n] = A[K + u];
    }
}

// ---------------------------------------------- Psi and Psi' on their own

__global__ void __launch_bounds__(kBlock) k_pull(DevProblem P, ProjC q, int channels,
                                                 const float* __restrict__ u,
                                                 float* __restrict__ out)
{
    const long long M = q.M;
    const long long sxy = (long long)q.mx * q.my;
    for (long long m = blockIdx.x * (long long)blockDim.x + threadIdx.x; m < M;
         m += (long long)gridDim.x * blockDim.x) {
        const int i = (int)(m % q.mx), j = (int)((m / q.mx) % q.my), k = (int)(m / sxy);
        float r[3];
        const bool in = reslice(q, i, j, k, P.nx, P.ny, P.nz, r);
        const Cell cl = cell_of(r);
        for (int ch = 0; ch < channels; ++ch) {
            float v[1] = {0.0f};
            if (in) interpolate<1>(cl, u + ch * P.N, P.N, P.nx, P.ny, P.nz, v);
            out[ch * M + m] = v[0];
        }
    }
}

// Running sum of w * u[m] for one channel.
struct SumInto {
    float s;
    const float* __restrict__ u;
    __device__ __forceinline__ void operator()(float w, long long m) { s = fmaf(w, __ldg(u + m), s); }
};

__global__ void __launch_bounds__(kBlock) k_push(DevProblem P, ProjC q, int channels,
                                                 const float* __restrict__ u,
                                                 float* __restrict__ out, int accumulate)
{
    const long long N = P.N, M = q.M;
    const long long sxy = (long long)P.nx * P.ny;
    const long long total = N * channels;
    for (long long id = blockIdx.x * (long long)blockDim.x + threadIdx.x; id < total;
         id += (long long)gridDim.x * blockDim.x) {
        const long long ch = id / N, n = id - ch * N;
        const int x = (int)(n % P.nx), y = (int)((n / P.nx) % P.ny), z = (int)(n / sxy);
        SumInto acc{accumulate ? out[id] : 0.0f, u + ch * M};
        acc = gather_pullers<long long>(q, x, y, z, P.nx, P.ny, P.nz, acc);
        out[id] = acc.s;
    }
}

// ------------------------------------------------------------------ host

static mpm_status make_proj(const mpm_problem* p, const mpm_projection* proj, DevProj& Q)
{
    if (!proj) return fail(MPM_ERR_INVALID_ARG, "projection is NULL");
    memset(&Q, 0, sizeof Q);
    Q.C = p->n_contrasts;
    for (int c = 0; c < Q.C; ++c) {
        ProjC& q = Q.c[c];
        q.mx = proj->dims[c][0];
        q.my = proj->dims[c][1];
        q.mz = proj->dims[c][2];
        if (q.mx < 1 || q.my < 1 || q.mz < 1)
            return fail(MPM_ERR_INVALID_ARG, "contrast %d: acquisition grid %d x %d x %d", c, q.mx,
                        q.my, q.mz);
        q.M = (long long)q.mx * q.my * q.mz;
        const double* A = proj->affine[c];
        for (int t = 0; t < 12; ++t)
            if (!std::isfinite(A[t]) || std::fabs(A[t]) > 1e7)
                return fail(MPM_ERR_INVALID_ARG, "contrast %d: affine entry %d is not finite", c, t);
        // inverse of the linear part by the adjugate, in double
        const double a = A[0], b = A[1], cc = A[2], d = A[4], e = A[5], f = A[6], g = A[8],
                     h = A[9], i = A[10];
        const double det = a * (e * i - f * h) - b * (d * i - f * g) + cc * (d * h - e * g);
        const double scale = std::fabs(a) + std::fabs(b) + std::fabs(cc) + std::fabs(d) +
                             std::fabs(e) + std::fabs(f) + std::fabs(g) + std::fabs(h) + std::fabs(i);
        if (!(std::fabs(det) > 1e-9 * scale * scale * scale))
            return fail(MPM_ERR_INVALID_ARG, "contrast %d: affine is singular", c);
        double L[9] = {(e * i - f * h) / det,  (cc * h - b * i) / det, (b * f - cc * e) / det,
                       (f * g - d * i) / det,  (a * i - cc * g) / det, (cc * d - a * f) / det,
                       (d * h - e * g) / det,  (b * g - a * h) / det,  (a * e - b * d) / det};
        for (int r = 0; r < 3; ++r) {
            double t = 0.0, ex = 0.0;
            for (int s = 0; s < 3; ++s) {
                t -= L[3 * r + s] * A[4 * s + 3];
                ex += std::fabs(L[3 * r + s]);
            }
            // a reconstruction voxel gathers from a box of 2 ext + 1 acquisition
            // voxels per axis: acquisition voxels at least a quarter of the
            // reconstruction voxel size keep it at 9 or fewer
            if (ex > 4.0)
                return fail(MPM_ERR_INVALID_ARG,
                            "contrast %d: acquisition voxels more than 4x smaller than the "
                            "reconstruction voxels along axis %d (inverse affine row sum %.3g)",
                            c, r, ex);
            for (int s = 0; s < 3; ++s) q.Ai[4 * r + s] = (float)L[3 * r + s];
            q.Ai[4 * r + 3] = (float)t;
            q.ext[r] = (float)ex;
            for (int s = 0; s < 4; ++s) q.A[4 * r + s] = (float)A[4 * r + s];
        }
        q.iA0 = std::fabs(q.A[0]) >= 0.5f ? 1.0f / q.A[0] : 0.0f;
        q.shifted = 1;
        for (int r = 0; r < 3; ++r) {
            const float t = q.A[4 * r + 3];
            for (int s = 0; s < 3; ++s)
                if (q.A[4 * r + s] != (r == s ? 1.0f : 0.0f)) q.shifted = 0;
            // sums of whole numbers below 2^24 are exact in float32
            if (t != std::floor(t) || std::fabs(t) >= 4194304.0f) q.shifted = 0;
            if (q.shifted) q.t[r] = (int)t;
        }
        if (std::max(q.mx, std::max(q.my, q.mz)) >= (1 << 22)) q.shifted = 0;
    }
    return MPM_OK;
}

// Workspace of the projected calls: the plain layout of `call` for the
// reconstruction grid, then the contrasts' NLL parts and g_c / H_c buffers.
struct ProjWs {
    FitWs L;
    double* nll_parts;
    float4* gh[MPM_MAX_CONTRASTS];
    size_t total;
};

static ProjWs proj_layout(const DevProblem& P, const DevProj& Q, int call, void* base, bool padded = true)
{
    ProjWs W;
    memset(&W, 0, sizeof W);
    W.L = layout(P, call, base, padded);
    size_t off = W.L.total;
    char* b = static_cast<char*>(base);
    auto take = [&](size_t bytes) -> char* {
        char* p = b ? b + off : nullptr;
        off += (bytes + 255) & ~(size_t)255;
        return p;
    };
    W.nll_parts = reinterpret_cast<double*>(take(sizeof(double) * MPM_MAX_CONTRASTS));
    for (int c = 0; c < Q.C; ++c) {
        W.gh[c] = reinterpret_cast<float4*>(take(sizeof(float) * (size_t)gh_floats(P.K) * Q.c[c].M));
    }
    W.total = off;
    return W;
}

static int tile_blocks(const VoxelTiles& g)
{
    return (int)std::max(1LL, std::min(g.count, 8LL * kNumSm));
}

// The pass of contrast c, which depends on K maps.
template <int K, int PRE>
static cudaError_t grad_hess_proj_c(const DevProblem& P, const DevProj& Q, int c, const ProjIn& in,
                                    const float* y, const ProjWs& W, Reduce red, cudaStream_t st)
{
    const ProjC& q = Q.c[c];
    const VoxelTiles tg = proj_tiles(q.mx, q.my, q.mz);
    const int grid = tile_blocks(tg);
    LaunchScope ls(MPM_KERNEL_GRAD_HESS_PROJ, st);
    auto launch = [&](auto* x, auto f) {
        f<<<grid, kBlock, 0, st>>>(P, q, c, y, x, in.b1p[c], in.b1m[c], W.gh[c], W.nll_parts + c, red, tg);
    };
    const bool usual = usual_tiles(tg);
    if (in.echo_dtype == 1) {
        using XT = __nv_bfloat16;
        launch(static_cast<const XT*>(in.x[c]),
               usual ? k_grad_hess_proj<K, PRE, XT, true> : k_grad_hess_proj<K, PRE, XT, false>);
    } else {
        launch(static_cast<const float*>(in.x[c]),
               usual ? k_grad_hess_proj<K, PRE, float, true> : k_grad_hess_proj<K, PRE, float, false>);
    }
    return cudaGetLastError();
}

template <int K, int PRE>
static cudaError_t grad_hess_proj_k(const DevProblem& P, const DevProj& Q, const ProjIn& in,
                                    const float* y, const ProjWs& W, float* g, float* h,
                                    double* nll, Reduce red, cudaStream_t st)
{
    for (int c = 0; c < Q.C; ++c) {
        const cudaError_t e = P.mt[c] ? grad_hess_proj_c<K, PRE>(P, Q, c, in, y, W, red, st)
                                      : grad_hess_proj_c<3, PRE>(P, Q, c, in, y, W, red, st);
        if (e != cudaSuccess) return e;
    }
    ProjBufs B;
    memset(&B, 0, sizeof B);
    for (int c = 0; c < Q.C; ++c) {
        B.gh[c] = W.gh[c];
    }
    LaunchScope ls(MPM_KERNEL_RESLICE, st);
    bool i32 = true;
    for (int c = 0; c < Q.C; ++c) i32 = i32 && Q.c[c].M <= 0xffffffffLL;
    const VoxelTiles tg = proj_tiles(P.nx, P.ny, P.nz);
    const int grid = tile_blocks(tg);
    const auto push = usual_tiles(tg) ? (i32 ? k_push_all<K, unsigned, true> : k_push_all<K, long long, true>)
                                      : (i32 ? k_push_all<K, unsigned, false> : k_push_all<K, long long, false>);
    push<<<grid, kBlock, 0, st>>>(P, Q, B, g, h, W.nll_parts, nll, tg);
    return cudaGetLastError();
}

template <int K>
static cudaError_t grad_hess_proj_pre(const DevProblem& P, const DevProj& Q, const ProjIn& in,
                                      const float* y, const ProjWs& W, float* g, float* h,
                                      double* nll, Reduce red, cudaStream_t st)
{
    if (P.precond == 1) return grad_hess_proj_k<K, 1>(P, Q, in, y, W, g, h, nll, red, st);
    if (P.precond == 2) return grad_hess_proj_k<K, 2>(P, Q, in, y, W, g, h, nll, red, st);
    return grad_hess_proj_k<K, 0>(P, Q, in, y, W, g, h, nll, red, st);
}

cudaError_t launch_grad_hess_proj(const DevProblem& P, const ProjJob& pj, const float* y, float* g,
                                  float* h, double* nll, Reduce red, cudaStream_t st)
{
    const DevProj& Q = *static_cast<const DevProj*>(pj.Q);
    const ProjWs& W = *static_cast<const ProjWs*>(pj.W);
    if (P.K == 4) return grad_hess_proj_pre<4>(P, Q, pj.in, y, W, g, h, nll, red, st);
    return grad_hess_proj_pre<3>(P, Q, pj.in, y, W, g, h, nll, red, st);
}

}  // namespace mpm

using namespace mpm;

namespace {

mpm_status check_proj_inputs(const mpm_problem* problem, const DevProj& Q, const void* const* x,
                             const float* const* b1p, const float* const* b1m, ProjIn& in)
{
    if (!x) return fail(MPM_ERR_INVALID_ARG, "x (array of per-contrast pointers) is NULL");
    memset(&in, 0, sizeof in);
    in.echo_dtype = problem->echo_dtype;
    const size_t ealign = problem->echo_dtype ? 2 : 4;
    for (int c = 0; c < Q.C; ++c) {
        char name[32];
        snprintf(name, sizeof name, "x[%d]", c);
        MPM_TRY(check_dev(x[c], name, false, ealign));
        in.x[c] = x[c];
        in.b1p[c] = b1p ? b1p[c] : nullptr;
        in.b1m[c] = b1m ? b1m[c] : nullptr;
        snprintf(name, sizeof name, "b1p[%d]", c);
        MPM_TRY(check_dev(in.b1p[c], name, true, 4));
        snprintf(name, sizeof name, "b1m[%d]", c);
        MPM_TRY(check_dev(in.b1m[c], name, true, 4));
    }
    return MPM_OK;
}

}  // namespace

extern "C" {

mpm_status mpm_workspace_size_proj(const mpm_problem* problem, const mpm_projection* proj,
                                   const mpm_opts* opts, int call, size_t* bytes)
{
    if (!bytes) return fail(MPM_ERR_INVALID_ARG, "bytes is NULL");
    MPM_TRY(check_problem(problem));
    if (call != MPM_CALL_FIT && call != MPM_CALL_GRAD_HESS)
        return fail(MPM_ERR_INVALID_ARG, "call must be MPM_CALL_FIT or MPM_CALL_GRAD_HESS");
    if (call == MPM_CALL_FIT) MPM_TRY(check_opts(opts));
    DevProj Q;
    MPM_TRY(make_proj(problem, proj, Q));
    *bytes = proj_layout(make_dev(problem), Q, call, nullptr).total;
    return MPM_OK;
}

mpm_status mpm_pull(const mpm_problem* problem, const mpm_projection* proj, int contrast,
                    int channels, const float* u, float* out, void* stream)
{
    MPM_TRY(check_problem(problem));
    DevProj Q;
    MPM_TRY(make_proj(problem, proj, Q));
    if (contrast < 0 || contrast >= Q.C)
        return fail(MPM_ERR_INVALID_ARG, "contrast %d outside [0, %d)", contrast, Q.C);
    if (channels < 1) return fail(MPM_ERR_INVALID_ARG, "channels must be >= 1");
    MPM_TRY(check_dev(u, "u", false, 4));
    MPM_TRY(check_dev(out, "out", false, 4));
    const DevProblem P = make_dev(problem);
    if (P.N == 0) return MPM_OK;
    cudaStream_t st = (cudaStream_t)stream;
    LaunchScope ls(MPM_KERNEL_RESLICE, st);
    k_pull<<<voxel_grid(Q.c[contrast].M), kBlock, 0, st>>>(P, Q.c[contrast], channels, u, out);
    MPM_CUDA(cudaGetLastError());
    return MPM_OK;
}

mpm_status mpm_push(const mpm_problem* problem, const mpm_projection* proj, int contrast,
                    int channels, const float* u, float* out, int accumulate, void* stream)
{
    MPM_TRY(check_problem(problem));
    DevProj Q;
    MPM_TRY(make_proj(problem, proj, Q));
    if (contrast < 0 || contrast >= Q.C)
        return fail(MPM_ERR_INVALID_ARG, "contrast %d outside [0, %d)", contrast, Q.C);
    if (channels < 1) return fail(MPM_ERR_INVALID_ARG, "channels must be >= 1");
    MPM_TRY(check_dev(u, "u", false, 4));
    MPM_TRY(check_dev(out, "out", false, 4));
    const DevProblem P = make_dev(problem);
    if (P.N == 0) return MPM_OK;
    cudaStream_t st = (cudaStream_t)stream;
    LaunchScope ls(MPM_KERNEL_RESLICE, st);
    k_push<<<voxel_grid(P.N), kBlock, 0, st>>>(P, Q.c[contrast], channels, u, out, accumulate);
    MPM_CUDA(cudaGetLastError());
    return MPM_OK;
}

mpm_status mpm_grad_hess_proj(const mpm_problem* problem, const mpm_projection* proj,
                              const void* const* x, const float* const* b1p,
                              const float* const* b1m, const float* y, float* g, float* h,
                              double* nll, void* ws, size_t ws_bytes, void* stream)
{
    MPM_TRY(check_problem(problem));
    DevProj Q;
    MPM_TRY(make_proj(problem, proj, Q));
    ProjIn in;
    MPM_TRY(check_proj_inputs(problem, Q, x, b1p, b1m, in));
    MPM_TRY(check_dev(y, "y", false, 4));
    MPM_TRY(check_dev(g, "g", false, 4));
    MPM_TRY(check_dev(h, "h", false, 4));
    MPM_TRY(check_dev(nll, "nll", false, 8));
    const DevProblem P = make_dev(problem);
    if (P.N == 0) return MPM_OK;
    const ProjWs need = proj_layout(P, Q, MPM_CALL_GRAD_HESS, nullptr);
    if (ws_bytes < need.total)
        return fail(MPM_ERR_WORKSPACE_TOO_SMALL, "workspace of %zu bytes, %zu needed", ws_bytes,
                    need.total);
    MPM_TRY(check_dev(ws, "ws", false, 256));
    const ProjWs W = proj_layout(P, Q, MPM_CALL_GRAD_HESS, ws);
    DevProj Qm = Q;
    cudaStream_t st = (cudaStream_t)stream;
    MPM_CUDA(cudaMemsetAsync(W.L.hdr, 0, sizeof(WsHeader), st));
    ProjWs Wm = W;
    ProjJob pj;
    pj.Q = &Qm;
    pj.W = &Wm;
    pj.in = in;
    MPM_CUDA(launch_grad_hess_proj(P, pj, y, g, h, nll, W.L.red, st));
    return MPM_OK;
}

}  // extern "C"

namespace mpm {

// Pieces of mpm_fit_proj that live with the projection: validation, the
// workspace layout and the image means over the acquisition grids.
mpm_status proj_prepare(const mpm_problem* problem, const mpm_projection* proj, const void* const* x,
                        const float* const* b1p, const float* const* b1m, void* ws, size_t ws_bytes,
                        ProjJob& pj, FitWs& L)
{
    DevProj* Q = new DevProj;
    ProjWs* W = new ProjWs;
    pj.Q = Q;
    pj.W = W;
    MPM_TRY(make_proj(problem, proj, *Q));
    MPM_TRY(check_proj_inputs(problem, *Q, x, b1p, b1m, pj.in));
    const DevProblem P = make_dev(problem);
    const bool padded = ws_bytes >= proj_layout(P, *Q, MPM_CALL_FIT, nullptr).total;
    const ProjWs need = proj_layout(P, *Q, MPM_CALL_FIT, nullptr, false);
    if (ws_bytes < need.total)
        return fail(MPM_ERR_WORKSPACE_TOO_SMALL, "workspace of %zu bytes, %zu needed", ws_bytes,
                    need.total);
    MPM_TRY(check_dev(ws, "ws", false, 256));
    *W = proj_layout(P, *Q, MPM_CALL_FIT, ws, padded);
    L = W->L;
    return MPM_OK;
}

void proj_release(ProjJob& pj)
{
    delete static_cast<DevProj*>(pj.Q);
    delete static_cast<ProjWs*>(pj.W);
    pj.Q = pj.W = nullptr;
}

size_t proj_key_bytes() { return sizeof(DevProj); }

// Bytes that identify a projected fit in the graph cache.
void proj_key(const ProjJob& pj, std::string& k)
{
    k.append(static_cast<const char*>(pj.Q), sizeof(DevProj));
    k.append(reinterpret_cast<const char*>(&pj.in), sizeof(ProjIn));
}

// Image means of every contrast over its own acquisition grid, written to
// means[echo0[c] + e].
cudaError_t proj_image_means(const DevProblem& P, const ProjJob& pj, double* parts, double* means,
                             cudaStream_t st)
{
    const DevProj& Q = *static_cast<const DevProj*>(pj.Q);
    for (int c = 0; c < Q.C; ++c) {
        DevProblem Pc = P;
        Pc.nx = Q.c[c].mx;
        Pc.ny = Q.c[c].my;
        Pc.nz = Q.c[c].mz;
        Pc.N = Q.c[c].M;
        Pc.I = P.n_echoes[c];
        cudaError_t e = launch_image_means(Pc, pj.in.echo_dtype, pj.in.x[c], parts, means + P.echo0[c], st);
        if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
}

}  // namespace mpm

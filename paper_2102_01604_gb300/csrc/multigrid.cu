// multigrid.cu -- conjugate gradient on the Newton system (H + L) delta =
// g + L y (Eq. 42) with an aggregation multigrid V-cycle as the
// preconditioner, an option beside the paper's block preconditioner
// (opts.mg_levels > 0; the paper's solver is the block-Jacobi PCG of
// stencil_kernels.cu / stencil_tma.cu).
//
// The hierarchy, rebuilt for every solve from H and the JTV weights:
//   - level 0 is the volume, with the edge coefficients of L,
//     kappa_a[n] = (w_n + w_{n + e_a}) / h_a^2 for the edge to the +a neighbour
//     (0 at the far face);
//   - level l + 1 merges 2 x 2 x 2 voxels of level l (ceil(n / 2) per axis); a
//     level of at most kMgMinVoxels voxels is the coarsest;
//   - prolongation copies a coarse voxel's value to its children, restriction
//     sums over them; the coarse operator is the Galerkin product P' A P,
//     which keeps the form of A: H summed over the children, and each coarse
//     edge coefficient the sum of the fine edge coefficients crossing it.
// Smoother: damped block-Jacobi x += omega D^-1 (r - A x), with D the 4 x 4
// voxel blocks H + diag(lambda_k sum of the six edge coefficients) (on level 0
// exactly the paper's preconditioner block).  V-cycle from x = 0: nu sweeps,
// coarse correction with the restricted residual, nu sweeps; the coarsest
// level takes coarse_sweeps sweeps.  Equal sweeps on both sides make the
// cycle symmetric, so plain CG may use it.
//
// Every kernel below takes tiles of 32 x 4 x 2 voxels, one per thread: no
// division per voxel, and the rows and planes a stencil shares stay in L1.
// Levels shorter than that along an axis take other shapes of the same size (with
// 32 x 4 x 2 for all, 12 iterations at 8x512x512 took 8.13 ms, 3.47 with 8 x 8 x
// 4; 1x256x256 2.45 and 0.95).  An iteration at the finest level is four
// launches: the matvec, the update with
// the first smoothing sweep (it has the residual at hand), the residual's
// restriction, and the last sweep with the coarse correction (each neighbour's
// parent added as it is read) and r . z.  They are bound by the latency of
// their loads: all of a voxel's are issued at once, none behind a test of an
// edge coefficient, and 64 registers keep four blocks on an SM (without that,
// 15.5 ms; hints of the next tile into L2, 14.3).  Solve of 176x240x256, 12
// iterations: 18.1 ms as seven kernels over linear 64-bit voxel indices, 13.7 ms.
//
// Vectors are voxel-interleaved (float4 per voxel, the fourth component zero
// for K = 3); H and kappa are planar.  CG scalars stay on the device (last
// block of each reducing launch), so a solve runs without host round trips and
// can be captured in a graph.
#include <type_traits>
#include <utility>

#include "mpm_internal.cuh"
#include "pcg_step.cuh"

namespace mpm {

constexpr long long kMgMinVoxels = 512;
constexpr int kMgMaxLevels = 16;
constexpr int kMgLX = 5, kMgLY = 2, kMgLZ = 1;      // tiles of 32 x 4 x 2 voxels

struct MgLevel {
    int nx, ny, nz;
    long long N;
    const float* h;     // [T][N]
    float* kap;         // [3][N]
    float4* r;          // right-hand side of this level's cycle
    float4* x;          // result of this level's cycle
    float4* t;          // ping-pong partner of x for the sweeps
    VoxelTiles tiles;
};

struct MgBufs {
    int L;                       // levels
    MgLevel lv[kMgMaxLevels];
    float4 *cx, *cp[2], *cq;     // CG: delta, directions (ping-pong), (H + L) p; r is lv[0].r, z is lv[0].x
};

static size_t al256(size_t b) { return (b + 255) & ~(size_t)255; }

// Level dimensions: ceil(n / 2) per axis until a level has at most
// kMgMinVoxels voxels or `levels` levels exist.
static int mg_dims(const DevProblem& P, int levels, int (*dims)[3])
{
    int n[3] = {P.nx, P.ny, P.nz};
    int L = 0;
    if (levels > kMgMaxLevels) levels = kMgMaxLevels;
    for (;;) {
        dims[L][0] = n[0];
        dims[L][1] = n[1];
        dims[L][2] = n[2];
        ++L;
        if (L >= levels || (long long)n[0] * n[1] * n[2] <= kMgMinVoxels) break;
        for (int a = 0; a < 3; ++a) n[a] = (n[a] + 1) / 2;
    }
    return L;
}

// Carves the multigrid buffers from `ws` (NULL: sizes only); returns bytes.
static size_t mg_carve(const DevProblem& P, int levels, void* ws, MgBufs* B)
{
    int dims[kMgMaxLevels][3];
    const int L = mg_dims(P, levels, dims);
    char* base = static_cast<char*>(ws);
    size_t off = 0;
    auto take = [&](size_t bytes) -> void* {
        void* p = base ? base + off : nullptr;
        off += al256(bytes);
        return p;
    };
    MgBufs b;
    b.L = L;
    for (int l = 0; l < L; ++l) {
        MgLevel& v = b.lv[l];
        v.nx = dims[l][0];
        v.ny = dims[l][1];
        v.nz = dims[l][2];
        v.N = (long long)v.nx * v.ny * v.nz;
        v.tiles = voxel_tiles(v.nx, v.ny, v.nz, kMgLX, kMgLY, kMgLZ);
        v.h = l == 0 ? nullptr : static_cast<const float*>(take(sizeof(float) * P.T * v.N));
        v.kap = static_cast<float*>(take(sizeof(float) * 3 * v.N));
        v.r = static_cast<float4*>(take(sizeof(float4) * v.N));
        v.x = static_cast<float4*>(take(sizeof(float4) * v.N));
        v.t = static_cast<float4*>(take(sizeof(float4) * v.N));
    }
    b.cx = static_cast<float4*>(take(sizeof(float4) * P.N));
    b.cp[0] = static_cast<float4*>(take(sizeof(float4) * P.N));
    b.cp[1] = static_cast<float4*>(take(sizeof(float4) * P.N));
    b.cq = static_cast<float4*>(take(sizeof(float4) * P.N));
    if (B) *B = b;
    return off;
}

size_t mg_ws_bytes(const DevProblem& P) { return mg_carve(P, kMgMaxLevels, nullptr, nullptr); }

// ------------------------------------------------------------ per voxel

// The six edge coefficients of voxel (x, y, z) of a level (order x-, x+, y-,
// y+, z-, z+; 0 where the neighbour is outside) and the neighbours' offsets (0
// there, so that every load below can be issued at once, before any
// coefficient has arrived).
__device__ __forceinline__ void level_edges(const MgLevel& L, int x, int y, int z, long long n,
                                            float (&c)[6], long long (&off)[6])
{
    const long long sxy = (long long)L.nx * L.ny;
    const float* kx = L.kap;
    const float* ky = L.kap + L.N;
    const float* kz = L.kap + 2 * L.N;
    const bool ok[6] = {x > 0, x + 1 < L.nx, y > 0, y + 1 < L.ny, z > 0, z + 1 < L.nz};
    off[0] = ok[0] ? -1 : 0;
    off[1] = ok[1] ? 1 : 0;
    off[2] = ok[2] ? -L.nx : 0;
    off[3] = ok[3] ? L.nx : 0;
    off[4] = ok[4] ? -sxy : 0;
    off[5] = ok[5] ? sxy : 0;
    const float k[6] = {kx[n + off[0]], kx[n], ky[n + off[2]], ky[n], kz[n + off[4]], kz[n]};
#pragma unroll
    for (int m = 0; m < 6; ++m) c[m] = ok[m] ? k[m] : 0.0f;
}

// A level's tiles.  USUAL: their shape as constants.  (As variables, and without
// the bounds on the update's and the coarsening's registers, 11 iterations at
// 45x62x49 took 930 us, 904 this way; 176x240x256 12.76 and 12.59 ms.)
template <bool USUAL>
__device__ __forceinline__ VoxelTiles tiles_of(const MgLevel& L)
{
    VoxelTiles t = L.tiles;
    if (USUAL) {
        t.lx = kMgLX;
        t.ly = kMgLY;
        t.lz = kMgLZ;
    }
    return t;
}

static bool usual_tiles(const MgLevel& L)
{
    return L.tiles.lx == kMgLX && L.tiles.ly == kMgLY && L.tiles.lz == kMgLZ;
}

// This thread's voxel of tile t; false where it lies outside the level.
template <bool USUAL>
__device__ __forceinline__ bool tile_voxel(const MgLevel& L, long long t, int& x, int& y, int& z, long long& n)
{
    tiles_of<USUAL>(L).voxel(t, x, y, z);
    n = x + (long long)L.nx * (y + (long long)L.ny * z);
    return x < L.nx && y < L.ny && z < L.nz;
}

static int mg_grid(const MgLevel& L)
{
    const long long cap = 8LL * kNumSm, t = L.tiles.count;
    return (int)(t < cap ? t : cap);
}

// (A v)_n on a level: H_n v_n + lambda_k sum_m c_m (v_n - v_m); at(m) returns
// v at neighbour m (v_n where there is none).
template <int K, class At>
__device__ __forceinline__ void level_apply(const DevProblem& P, const float (&hv)[K * (K + 1) / 2],
                                            const float (&c)[6], const float4& v, At at, float (&out)[K])
{
    float vn[K];
    unpack4<K>(v, vn);
    float lap[K];
#pragma unroll
    for (int a = 0; a < K; ++a) lap[a] = 0.0f;
    float4 nb[6];
#pragma unroll
    for (int m = 0; m < 6; ++m) nb[m] = at(m);
#pragma unroll
    for (int m = 0; m < 6; ++m) {
        float vm[K];
        unpack4<K>(nb[m], vm);
#pragma unroll
        for (int a = 0; a < K; ++a) lap[a] = fmaf(c[m], vn[a] - vm[a], lap[a]);
    }
#pragma unroll
    for (int a = 0; a < K; ++a) {
        float acc = P.lambda[a] * lap[a];
#pragma unroll
        for (int b = 0; b < K; ++b) acc = fmaf(hv[a < b ? tri(K, a, b) : tri(K, b, a)], vn[b], acc);
        out[a] = acc;
    }
}

__device__ __forceinline__ float4 add4(const float4& a, const float4& b)
{
    return make_float4(a.x + b.x, a.y + b.y, a.z + b.z, a.w + b.w);
}

template <int K>
__device__ __forceinline__ void load_h(const MgLevel& L, const float* h0, long long n,
                                       float (&hv)[K * (K + 1) / 2])
{
    const float* h = L.h ? L.h : h0;
#pragma unroll
    for (int t = 0; t < K * (K + 1) / 2; ++t) hv[t] = __ldg(h + t * L.N + n);
}

__device__ __forceinline__ bool solve_done(const WsHeader* hdr) { return hdr->sc.done != 0; }

// ------------------------------------------------------------ hierarchy

// Level 0 edge coefficients from the JTV weights.
template <bool USUAL>
__global__ void __launch_bounds__(kBlock) k_mg_kappa0(DevProblem P, MgLevel L, const float* __restrict__ w)
{
    const long long sxy = (long long)L.nx * L.ny;
    for (long long t = blockIdx.x; t < L.tiles.count; t += gridDim.x) {
        int x, y, z;
        long long n;
        if (!tile_voxel<USUAL>(L, t, x, y, z, n)) continue;
        const float wn = __ldg(w + n);
        L.kap[n] = x + 1 < L.nx ? (wn + __ldg(w + n + 1)) * P.ihx2 : 0.0f;
        L.kap[L.N + n] = y + 1 < L.ny ? (wn + __ldg(w + n + L.nx)) * P.ihy2 : 0.0f;
        L.kap[2 * L.N + n] = z + 1 < L.nz ? (wn + __ldg(w + n + sxy)) * P.ihz2 : 0.0f;
    }
}

// Galerkin coarse level: H summed over the children, each coarse edge the
// sum of the fine edges crossing it (those of the children on the +a side).
template <bool USUAL>
__global__ void __launch_bounds__(kBlock, 4) k_mg_coarsen(DevProblem P, MgLevel F, MgLevel C,
                                                       const float* h0)
{
    const int T = P.T;
    const float* fh = F.h ? F.h : h0;
    float* ch = const_cast<float*>(C.h);
    for (long long t = blockIdx.x; t < C.tiles.count; t += gridDim.x) {
        int cx, cy, cz;
        long long c;
        if (!tile_voxel<USUAL>(C, t, cx, cy, cz, c)) continue;
        float hs[10] = {0, 0, 0, 0, 0, 0, 0, 0, 0, 0};
        float ks[3] = {0, 0, 0};
        for (int dz = 0; dz < 2; ++dz)
            for (int dy = 0; dy < 2; ++dy)
                for (int dx = 0; dx < 2; ++dx) {
                    const int fx = 2 * cx + dx, fy = 2 * cy + dy, fz = 2 * cz + dz;
                    if (fx >= F.nx || fy >= F.ny || fz >= F.nz) continue;
                    const long long f = fx + (long long)F.nx * (fy + (long long)F.ny * fz);
                    for (int e = 0; e < T; ++e) hs[e] += __ldg(fh + e * F.N + f);
                    if (dx == 1 && fx + 1 < F.nx) ks[0] += F.kap[f];
                    if (dy == 1 && fy + 1 < F.ny) ks[1] += F.kap[F.N + f];
                    if (dz == 1 && fz + 1 < F.nz) ks[2] += F.kap[2 * F.N + f];
                }
        for (int e = 0; e < T; ++e) ch[e * C.N + c] = hs[e];
        for (int a = 0; a < 3; ++a) C.kap[a * C.N + c] = ks[a];
    }
}

// ------------------------------------------------------------ V-cycle

// omega D^-1 b of one voxel, D its preconditioner block.
template <int K>
__device__ __forceinline__ void block_solve(const DevProblem& P, const float (&hv)[K * (K + 1) / 2],
                                            const float (&c)[6], const float (&b)[K], float (&e)[K])
{
    float M[K][K], Lf[K * (K + 1) / 2];
    precond_block<K>(P, hv, edge_sum(c), M);
    cholesky_f32<K>(M, Lf);
    chol_apply<K>(Lf, b, e);
}

// What a sweep starts from.
enum : int {
    kFromZero = 0,       // xout = omega D^-1 r
    kFromX = 1,          // xout = xin + omega D^-1 (r - A xin)
    kFromCoarse = 2      // the same from xin + P xc, xc the next level's result
};

// Scalars of the next direction from r . z (the last block of a reducing launch).
__device__ __forceinline__ void direction_scalars(double rz, int first, WsHeader* hdr)
{
    SolveScalars& sc = hdr->sc;
    if (!(rz == rz)) atomicOr(&hdr->status, kStatusNaN);
    if (!(rz > 0.0)) {
        sc.done = 1;
        return;
    }
    sc.beta = first ? 0.0 : rz / sc.rz;
    sc.rz = rz;
}

// One damped block-Jacobi sweep on a level; DOT: the result is z, and r . z is
// reduced (`first`: of the first cycle).
template <int K, int FROM, bool DOT, bool USUAL>
__global__ void __launch_bounds__(kBlock, 4) k_mg_sweep(DevProblem P, MgLevel L, MgLevel C, const float* h0,
                                                     float omega, const float4* __restrict__ xin,
                                                     float4* __restrict__ xout, int first, WsHeader* hdr,
                                                     Reduce red)
{
    constexpr int T = K * (K + 1) / 2;
    if (solve_done(hdr)) return;
    Acc acc;
    for (long long t = blockIdx.x; t < L.tiles.count; t += gridDim.x) {
        int x, y, z;
        long long n;
        if (!tile_voxel<USUAL>(L, t, x, y, z, n)) continue;
        float c[6];
        long long off[6];
        level_edges(L, x, y, z, n, c, off);
        float hv[T];
        load_h<K>(L, h0, n, hv);
        float r[K], b[K], e[K], xo[K];
        unpack4<K>(L.r[n], r);
#pragma unroll
        for (int a = 0; a < K; ++a) b[a] = r[a];
        if (FROM != kFromZero) {
            // xin at a voxel, with its parent's correction added
            auto at = [&](int vx, int vy, int vz, long long m) {
                if (FROM == kFromX) return xin[m];
                return add4(xin[m], C.x[(vx >> 1) + (long long)C.nx * ((vy >> 1) + (long long)C.ny * (vz >> 1))]);
            };
            const float4 own = at(x, y, z, n);
            float ax[K];
            level_apply<K>(P, hv, c, own,
                           [&](int m) {
                               const int d = off[m] != 0 ? 1 : 0;
                               return at(m == 0 ? x - d : m == 1 ? x + d : x, m == 2 ? y - d : m == 3 ? y + d : y,
                                         m == 4 ? z - d : m == 5 ? z + d : z, n + off[m]);
                           },
                           ax);
            unpack4<K>(own, xo);
#pragma unroll
            for (int a = 0; a < K; ++a) b[a] -= ax[a];
        }
        block_solve<K>(P, hv, c, b, e);
#pragma unroll
        for (int a = 0; a < K; ++a) xo[a] = FROM == kFromZero ? omega * e[a] : fmaf(omega, e[a], xo[a]);
        xout[n] = pack4<K>(xo);
        if (DOT) {
            float s = r[0] * xo[0];
#pragma unroll
            for (int a = 1; a < K; ++a) s = fmaf(r[a], xo[a], s);
            acc.add(s);
        }
    }
    if constexpr (DOT) {
        Acc v[1] = {acc};
        double out[1];
        if (grid_reduce<1>(v, red, out) && threadIdx.x == 0) direction_scalars(out[0], first, hdr);
    }
}

// Restricted residual: C.r = P' (F.r - A_F x).  One fine voxel per thread; the
// children of a coarse voxel lie in one tile and are summed in the warp (the pair
// along x) and in shared memory (y, then z).  Along an axis on which the tile is
// one voxel long there is one voxel, and nothing to pair.
template <int K, bool USUAL>
__global__ void __launch_bounds__(kBlock, 4) k_mg_restrict(DevProblem P, MgLevel F, MgLevel C, const float* h0,
                                                        const float4* __restrict__ xf, const WsHeader* hdr)
{
    constexpr int T = K * (K + 1) / 2;
    __shared__ float4 part[kBlock];
    if (solve_done(hdr)) return;
    const int tid = threadIdx.x;
    const VoxelTiles tl = tiles_of<USUAL>(F);
    const int px = tl.lx > 0, py = tl.ly > 0, pz = tl.lz > 0;    // pairs along an axis
    const int lx = tl.lx - px, ly = tl.ly - py, lz = tl.lz - pz;     // the tile's coarse voxels
    const int u = tid & ((1 << lx) - 1), v = (tid >> lx) & ((1 << ly) - 1), s = tid >> (lx + ly);
    const int sy = 1 << lx, sz = sy << tl.ly;                                  // strides of part
    const int p0 = u + (v << py) * sy + (s << pz) * sz;
    const int ix = tid & ((1 << tl.lx) - 1), iy = (tid >> tl.lx) & ((1 << tl.ly) - 1),
              iz = tid >> (tl.lx + tl.ly);                                // this thread's place
    for (long long t = blockIdx.x; t < F.tiles.count; t += gridDim.x) {
        int x, y, z;
        long long n;
        float d[K];
#pragma unroll
        for (int a = 0; a < K; ++a) d[a] = 0.0f;
        if (tile_voxel<USUAL>(F, t, x, y, z, n)) {
            float c[6];
            long long off[6];
            level_edges(F, x, y, z, n, c, off);
            float hv[T], ax[K], r[K];
            load_h<K>(F, h0, n, hv);
            level_apply<K>(P, hv, c, xf[n], [&](int m) { return xf[n + off[m]]; }, ax);
            unpack4<K>(F.r[n], r);
#pragma unroll
            for (int a = 0; a < K; ++a) d[a] = r[a] - ax[a];
        }
        if (px) {
#pragma unroll
            for (int a = 0; a < K; ++a) d[a] += __shfl_down_sync(0xffffffffu, d[a], 1);
        }
        if (!px || !(tid & 1)) part[tid >> px] = pack4<K>(d);
        __syncthreads();
        if (tid < 1 << (lx + ly + lz)) {
            auto line = [&](int p) { return py ? add4(part[p], part[p + sy]) : part[p]; };
            const float4 sum = pz ? add4(line(p0), line(p0 + sz)) : line(p0);
            // the tile's corner, halved, is its first coarse voxel
            const int cx = ((x - ix) >> 1) + u, cy = ((y - iy) >> 1) + v, cz = ((z - iz) >> 1) + s;
            if (cx < C.nx && cy < C.ny && cz < C.nz) C.r[cx + (long long)C.nx * (cy + (long long)C.ny * cz)] = sum;
        }
        __syncthreads();
    }
}

// The coarsest level in one block: `sweeps` damped block-Jacobi sweeps from
// zero, ping-ponging between L.x and L.t (result in L.x after an even count of
// buffer swaps, else copied there).
template <int K>
__global__ void __launch_bounds__(512) k_mg_coarsest(DevProblem P, MgLevel L, const float* h0, float omega,
                                                      int sweeps, const WsHeader* hdr)
{
    constexpr int T = K * (K + 1) / 2;
    if (solve_done(hdr)) return;
    float4* bufs[2] = {L.x, L.t};
    for (int s = 0; s < sweeps; ++s) {
        const float4* xin = bufs[(s + 1) & 1];
        float4* xout = bufs[s & 1];
        for (long long n = threadIdx.x; n < L.N; n += blockDim.x) {
            const int x = (int)(n % L.nx), y = (int)((n / L.nx) % L.ny), z = (int)(n / ((long long)L.nx * L.ny));
            float c[6];
            long long off[6];
            level_edges(L, x, y, z, n, c, off);
            float hv[T], b[K], xo[K], e[K];
            load_h<K>(L, h0, n, hv);
            unpack4<K>(L.r[n], b);
            if (s > 0) {
                float ax[K];
                level_apply<K>(P, hv, c, xin[n], [&](int m) { return xin[n + off[m]]; }, ax);
#pragma unroll
                for (int a = 0; a < K; ++a) b[a] -= ax[a];
                unpack4<K>(xin[n], xo);
            } else {
#pragma unroll
                for (int a = 0; a < K; ++a) xo[a] = 0.0f;
            }
            block_solve<K>(P, hv, c, b, e);
#pragma unroll
            for (int a = 0; a < K; ++a) xo[a] = fmaf(omega, e[a], xo[a]);
            xout[n] = pack4<K>(xo);
        }
        __syncthreads();
    }
    if (sweeps > 0 && ((sweeps - 1) & 1)) {
        for (long long n = threadIdx.x; n < L.N; n += blockDim.x) L.x[n] = L.t[n];
    }
}

// The same for a level of at most 512 voxels, one per thread: H, the edges and
// the block's factor in registers, the iterates in shared memory (24 -> 10 us for
// 20 sweeps of 6 x 8 x 8 voxels).
template <int K>
__global__ void __launch_bounds__(512) k_mg_coarsest_small(DevProblem P, MgLevel L, const float* h0, float omega,
                                                            int sweeps, const WsHeader* hdr)
{
    constexpr int T = K * (K + 1) / 2;
    __shared__ float4 it[2][512];
    if (solve_done(hdr)) return;
    const int n = threadIdx.x;
    const bool in = n < (int)L.N;
    const int x = n % L.nx, y = (n / L.nx) % L.ny, z = n / (L.nx * L.ny);
    float c[6], hv[T], Lf[T], r[K], xo[K];
    long long off[6];
#pragma unroll
    for (int a = 0; a < K; ++a) xo[a] = 0.0f;
    if (in) {
        level_edges(L, x, y, z, n, c, off);
        load_h<K>(L, h0, n, hv);
        unpack4<K>(L.r[n], r);
        float M[K][K];
        precond_block<K>(P, hv, edge_sum(c), M);
        cholesky_f32<K>(M, Lf);
    }
    for (int s = 0; s < sweeps; ++s) {
        if (in) {
            float b[K], e[K];
#pragma unroll
            for (int a = 0; a < K; ++a) b[a] = r[a];
            if (s > 0) {
                const float4* xin = it[s & 1];
                float ax[K];
                level_apply<K>(P, hv, c, xin[n], [&](int m) { return xin[n + (int)off[m]]; }, ax);
#pragma unroll
                for (int a = 0; a < K; ++a) b[a] -= ax[a];
            }
            chol_apply<K>(Lf, b, e);
#pragma unroll
            for (int a = 0; a < K; ++a) xo[a] = fmaf(omega, e[a], xo[a]);
            it[(s + 1) & 1][n] = pack4<K>(xo);
        }
        __syncthreads();
    }
    if (in) L.x[n] = pack4<K>(xo);
}

// ------------------------------------------------------------ CG

// r = g + L y (L from the JTV weights), |r_0|^2; scalars reset.
template <int K, bool USUAL>
__global__ void __launch_bounds__(kBlock) k_mgcg_init(DevProblem P, MgLevel L0, const float* __restrict__ g,
                                                      const float* __restrict__ y, double tol2,
                                                      WsHeader* hdr, double* resid, Reduce red)
{
    Acc rr;
    for (long long t = blockIdx.x; t < L0.tiles.count; t += gridDim.x) {
        int x, yy, z;
        long long n;
        if (!tile_voxel<USUAL>(L0, t, x, yy, z, n)) continue;
        float c[6];
        long long off[6];
        level_edges(L0, x, yy, z, n, c, off);
        float r[K];
        float vr = 0.0f;
#pragma unroll
        for (int k = 0; k < K; ++k) {
            const float* yk = y + k * P.N;
            const float v = __ldg(yk + n);
            float s = 0.0f;
#pragma unroll
            for (int m = 0; m < 6; ++m)
                if (c[m] != 0.0f) s = fmaf(c[m], v - __ldg(yk + n + off[m]), s);
            r[k] = __ldg(g + k * P.N + n) + P.lambda[k] * s;
            vr = fmaf(r[k], r[k], vr);
        }
        L0.r[n] = pack4<K>(r);
        rr.add(vr);
    }
    Acc v[1] = {rr};
    double out[1];
    if (grid_reduce<1>(v, red, out) && threadIdx.x == 0) {
        SolveScalars& sc = hdr->sc;
        sc.rr0 = out[0];
        sc.rr = out[0];
        sc.rz = 0.0;
        sc.alpha = 0.0;
        sc.alpha_prev = 0.0;
        sc.beta = 0.0;
        sc.beta_prev = 0.0;
        sc.it = 0;
        sc.xcount = 0;
        sc.tol2 = tol2;
        const bool bad = !(out[0] == out[0]);
        if (bad) atomicOr(&hdr->status, kStatusNaN);
        sc.done = (bad || !(out[0] > 0.0)) ? 1 : 0;
        if (resid) resid[0] = sqrt(out[0]);
    }
}

// rz = r . z and beta = rz / rz_previous (first: beta unused), where no sweep
// of the finest level ends the cycle (a hierarchy of one level).
template <int K>
__global__ void __launch_bounds__(kBlock) k_mgcg_rz(long long N, const float4* __restrict__ r,
                                                    const float4* __restrict__ z, int first,
                                                    WsHeader* hdr, Reduce red)
{
    if (solve_done(hdr)) return;
    Acc acc;
    for (long long n = blockIdx.x * (long long)blockDim.x + threadIdx.x; n < N;
         n += (long long)gridDim.x * blockDim.x) {
        float a[K], b[K];
        unpack4<K>(r[n], a);
        unpack4<K>(z[n], b);
        float s = a[0] * b[0];
#pragma unroll
        for (int k = 1; k < K; ++k) s = fmaf(a[k], b[k], s);
        acc.add(s);
    }
    Acc v[1] = {acc};
    double out[1];
    if (grid_reduce<1>(v, red, out) && threadIdx.x == 0) direction_scalars(out[0], first, hdr);
}

// p = z + beta p_old (at the voxel and its neighbours), q = (H + L) p, p . q;
// alpha = rz / p.q.
template <int K, bool USUAL>
__global__ void __launch_bounds__(kBlock, 4) k_mgcg_matvec(DevProblem P, MgLevel L0, const float* h0,
                                                        const float4* __restrict__ pold,
                                                        float4* __restrict__ pnew, float4* __restrict__ q,
                                                        int first, WsHeader* hdr, Reduce red)
{
    constexpr int T = K * (K + 1) / 2;
    __shared__ float s_beta;
    __shared__ int s_done;
    if (threadIdx.x == 0) {
        s_done = hdr->sc.done;
        s_beta = (float)hdr->sc.beta;
    }
    __syncthreads();
    if (s_done) return;
    const float beta = s_beta;
    const float4* z = L0.x;
    auto dir = [&](long long m, float (&pm)[K]) {
        float zm[K];
        unpack4<K>(z[m], zm);
        if (first) {
#pragma unroll
            for (int a = 0; a < K; ++a) pm[a] = zm[a];
        } else {
            float po[K];
            unpack4<K>(pold[m], po);
#pragma unroll
            for (int a = 0; a < K; ++a) pm[a] = fmaf(beta, po[a], zm[a]);
        }
    };
    Acc acc;
    for (long long t = blockIdx.x; t < L0.tiles.count; t += gridDim.x) {
        int x, y, zz;
        long long n;
        if (!tile_voxel<USUAL>(L0, t, x, y, zz, n)) continue;
        float c[6];
        long long off[6];
        level_edges(L0, x, y, zz, n, c, off);
        float pn[K], lap[K];
        dir(n, pn);
#pragma unroll
        for (int a = 0; a < K; ++a) lap[a] = 0.0f;
        float nb[6][K];
#pragma unroll
        for (int m = 0; m < 6; ++m) dir(n + off[m], nb[m]);
#pragma unroll
        for (int m = 0; m < 6; ++m)
#pragma unroll
            for (int a = 0; a < K; ++a) lap[a] = fmaf(c[m], pn[a] - nb[m][a], lap[a]);
        float hv[T], qn[K];
        load_h<K>(L0, h0, n, hv);
        float s = 0.0f;
#pragma unroll
        for (int a = 0; a < K; ++a) {
            float v = P.lambda[a] * lap[a];
#pragma unroll
            for (int b = 0; b < K; ++b) v = fmaf(hv[a < b ? tri(K, a, b) : tri(K, b, a)], pn[b], v);
            qn[a] = v;
            s = fmaf(pn[a], v, s);
        }
        pnew[n] = pack4<K>(pn);
        q[n] = pack4<K>(qn);
        acc.add(s);
    }
    Acc v[1] = {acc};
    double out[1];
    if (grid_reduce<1>(v, red, out) && threadIdx.x == 0) {
        SolveScalars& sc = hdr->sc;
        if (!(out[0] == out[0])) atomicOr(&hdr->status, kStatusNaN);
        if (!(out[0] > 0.0)) {
            sc.done = 1;                 // no step; the solve keeps its x
            return;
        }
        sc.alpha = sc.rz / out[0];
    }
}

// x += alpha p, r -= alpha q, |r|^2; the iteration counter and the tolerance.
// SWEEP: also the next cycle's first sweep, t = omega D^-1 r.
template <int K, bool SWEEP, bool USUAL>
__global__ void __launch_bounds__(kBlock, 5) k_mgcg_update(DevProblem P, MgLevel L0, const float* h0, float omega,
                                                        int j, float4* __restrict__ xacc,
                                                        const float4* __restrict__ p,
                                                        const float4* __restrict__ q, WsHeader* hdr,
                                                        double* resid, Reduce red)
{
    __shared__ float s_alpha;
    __shared__ int s_done;
    if (threadIdx.x == 0) {
        s_done = hdr->sc.done;
        s_alpha = (float)hdr->sc.alpha;
    }
    __syncthreads();
    if (s_done) return;
    const float alpha = s_alpha;
    Acc acc;
    for (long long t = blockIdx.x; t < L0.tiles.count; t += gridDim.x) {
        int x, y, z;
        long long n;
        if (!tile_voxel<USUAL>(L0, t, x, y, z, n)) continue;
        float xv[K], pv[K], qv[K], rv[K];
        unpack4<K>(p[n], pv);
        unpack4<K>(q[n], qv);
        unpack4<K>(L0.r[n], rv);
        if (j == 0) {
#pragma unroll
            for (int a = 0; a < K; ++a) xv[a] = 0.0f;
        } else {
            unpack4<K>(xacc[n], xv);
        }
        float c[6], hv[K * (K + 1) / 2];
        if (SWEEP) {
            long long off[6];
            level_edges(L0, x, y, z, n, c, off);
            load_h<K>(L0, h0, n, hv);
        }
        float s = 0.0f;
#pragma unroll
        for (int a = 0; a < K; ++a) {
            xv[a] = fmaf(alpha, pv[a], xv[a]);
            rv[a] = fmaf(-alpha, qv[a], rv[a]);
            s = fmaf(rv[a], rv[a], s);
        }
        xacc[n] = pack4<K>(xv);
        L0.r[n] = pack4<K>(rv);
        if (SWEEP) {
            float e[K];
            block_solve<K>(P, hv, c, rv, e);
#pragma unroll
            for (int a = 0; a < K; ++a) e[a] *= omega;
            L0.t[n] = pack4<K>(e);
        }
        acc.add(s);
    }
    Acc v[1] = {acc};
    double out[1];
    if (grid_reduce<1>(v, red, out) && threadIdx.x == 0) {
        SolveScalars& sc = hdr->sc;
        if (!(out[0] == out[0])) atomicOr(&hdr->status, kStatusNaN);
        sc.rr = out[0];
        sc.it = j + 1;
        if (resid) resid[j + 1] = sqrt(out[0]);
        if (!(out[0] == out[0]) || (sc.tol2 > 0.0 && out[0] <= sc.tol2 * sc.rr0)) sc.done = 1;
    }
}

// delta = x (planar), or y <- y - x; the report.
template <int K>
__global__ void __launch_bounds__(kBlock) k_mgcg_final(long long N, const float4* __restrict__ xacc,
                                                       float* __restrict__ delta,
                                                       float* __restrict__ y_update, const WsHeader* hdr,
                                                       double* report_rel, int* report_it)
{
    const SolveScalars sc = hdr->sc;
    for (long long n = blockIdx.x * (long long)blockDim.x + threadIdx.x; n < N;
         n += (long long)gridDim.x * blockDim.x) {
        float v[K];
        if (sc.it > 0) {
            unpack4<K>(xacc[n], v);
        } else {
#pragma unroll
            for (int a = 0; a < K; ++a) v[a] = 0.0f;
        }
#pragma unroll
        for (int a = 0; a < K; ++a) {
            if (y_update)
                y_update[a * N + n] -= v[a];
            else
                delta[a * N + n] = v[a];
        }
    }
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        if (report_rel) *report_rel = sc.rr0 > 0.0 ? sqrt(sc.rr / sc.rr0) : 0.0;
        if (report_it) *report_it = sc.it;
    }
}

// ------------------------------------------------------------ host

// One V-cycle from level l.  `swept`: the first sweep of level l has been made
// (into its t); `first`: of the first cycle (level 0's last sweep reduces r . z).
template <int K>
static void vcycle(const DevProblem& P, const MgBufs& B, int l, const float* h0, const SolveOpts& o,
                   bool swept, int first, WsHeader* hdr, Reduce red, cudaStream_t st)
{
    const MgLevel& Lv = B.lv[l];
    const int grid = mg_grid(Lv);
    const bool usual = usual_tiles(Lv);
    const float om = o.mg_omega;
    auto sweep = [&](auto from, bool dot, const MgLevel& C, const float4* xin, float4* xout) {
        constexpr int FROM = decltype(from)::value;
        LaunchScope ls(MPM_KERNEL_MG, st);
        const auto f = dot ? (usual ? k_mg_sweep<K, FROM, true, true> : k_mg_sweep<K, FROM, true, false>)
                           : (usual ? k_mg_sweep<K, FROM, false, true> : k_mg_sweep<K, FROM, false, false>);
        f<<<grid, kBlock, 0, st>>>(P, Lv, C, h0, om, xin, xout, first, hdr, red);
    };
    using Zero = std::integral_constant<int, kFromZero>;
    using FromX = std::integral_constant<int, kFromX>;
    using Coarse = std::integral_constant<int, kFromCoarse>;
    if (l == B.L - 1) {
        if (Lv.N <= 512) {
            LaunchScope ls(MPM_KERNEL_MG, st);
            k_mg_coarsest_small<K><<<1, 512, 0, st>>>(P, Lv, h0, om, o.mg_coarse_sweeps, hdr);
        } else if (Lv.N <= 8192) {
            LaunchScope ls(MPM_KERNEL_MG, st);
            k_mg_coarsest<K><<<1, 512, 0, st>>>(P, Lv, h0, om, o.mg_coarse_sweeps, hdr);
        } else {
            // a large coarsest level (few levels asked for): one launch per sweep
            float4* bufs[2] = {Lv.x, Lv.t};
            for (int s = 0; s < o.mg_coarse_sweeps; ++s) {
                if (s == 0) sweep(Zero(), false, Lv, Lv.x, bufs[0]);
                else sweep(FromX(), false, Lv, bufs[(s + 1) & 1], bufs[s & 1]);
            }
            if (o.mg_coarse_sweeps > 0 && ((o.mg_coarse_sweeps - 1) & 1))
                cudaMemcpyAsync(Lv.x, Lv.t, sizeof(float4) * Lv.N, cudaMemcpyDeviceToDevice, st);
        }
        return;
    }
    // pre-smoothing: the result ends in `cur`.  The first sweep writes in
    // place and every later sweep swaps, 2 nu - 1 swaps in all, so starting
    // from t the cycle's result lands in x.
    float4* cur = Lv.t;
    float4* other = Lv.x;
    for (int s = 0; s < o.mg_nu; ++s) {
        if (s > 0) {
            sweep(FromX(), false, Lv, cur, other);
            std::swap(cur, other);
        } else if (!swept) {
            sweep(Zero(), false, Lv, cur, cur);
        }
    }
    const MgLevel& C = B.lv[l + 1];
    {
        LaunchScope ls(MPM_KERNEL_MG, st);
        const auto f = usual ? k_mg_restrict<K, true> : k_mg_restrict<K, false>;
        f<<<grid, kBlock, 0, st>>>(P, Lv, C, h0, cur, hdr);
    }
    vcycle<K>(P, B, l + 1, h0, o, false, first, hdr, red, st);
    for (int s = 0; s < o.mg_nu; ++s) {
        const bool dot = l == 0 && s == o.mg_nu - 1;
        if (s == 0) sweep(Coarse(), dot, C, cur, other);
        else sweep(FromX(), dot, Lv, cur, other);
        std::swap(cur, other);
    }
    if (cur != Lv.x) {
        // the level's result must be in x
        cudaMemcpyAsync(Lv.x, cur, sizeof(float4) * Lv.N, cudaMemcpyDeviceToDevice, st);
    }
}

template <int K>
static cudaError_t solve_mg_k(const DevProblem& P, const SolveOpts& o, const float* h, const float* w,
                              const float* g, const float* y, float* delta, float* y_update,
                              double* resid, double* report_rel, int* report_it, void* solve_ws,
                              WsHeader* hdr, Reduce red, cudaStream_t st)
{
    MgBufs B;
    mg_carve(P, o.mg_levels, solve_ws, &B);
    MgLevel L0 = B.lv[0];
    const int grid = voxel_grid(P.N), tgrid = mg_grid(L0);
    const double tol2 = o.tol_cg > 0.0 ? o.tol_cg * o.tol_cg : 0.0;
    const bool one_level = B.L == 1, usual = usual_tiles(L0);
    {
        LaunchScope ls(MPM_KERNEL_MG, st);
        const auto f = usual ? k_mg_kappa0<true> : k_mg_kappa0<false>;
        f<<<tgrid, kBlock, 0, st>>>(P, L0, w);
    }
    for (int l = 0; l + 1 < B.L; ++l) {
        LaunchScope ls(MPM_KERNEL_MG, st);
        const auto f = usual_tiles(B.lv[l + 1]) ? k_mg_coarsen<true> : k_mg_coarsen<false>;
        f<<<mg_grid(B.lv[l + 1]), kBlock, 0, st>>>(P, B.lv[l], B.lv[l + 1], h);
    }
    {
        LaunchScope ls(MPM_KERNEL_PCG_INIT, st);
        const auto f = usual ? k_mgcg_init<K, true> : k_mgcg_init<K, false>;
        f<<<tgrid, kBlock, 0, st>>>(P, L0, g, y, tol2, hdr, resid, red);
    }
    auto cycle = [&](bool swept, int first) {
        vcycle<K>(P, B, 0, h, o, swept, first, hdr, red, st);
        if (!one_level) return;
        LaunchScope ls(MPM_KERNEL_PCG_STEP, st);
        k_mgcg_rz<K><<<grid, kBlock, 0, st>>>(P.N, L0.r, L0.x, first, hdr, red);
    };
    cycle(false, 1);
    for (int j = 0; j < o.cg_iters; ++j) {
        float4* pold = B.cp[(j + 1) & 1];
        float4* pnew = B.cp[j & 1];
        const bool more = j + 1 < o.cg_iters;
        {
            LaunchScope ls(MPM_KERNEL_PCG_STEP, st);
            const auto f = usual ? k_mgcg_matvec<K, true> : k_mgcg_matvec<K, false>;
            f<<<tgrid, kBlock, 0, st>>>(P, L0, h, pold, pnew, B.cq, j == 0, hdr, red);
        }
        {
            LaunchScope ls(MPM_KERNEL_PCG_STEP, st);
            const auto f = more && !one_level
                               ? (usual ? k_mgcg_update<K, true, true> : k_mgcg_update<K, true, false>)
                               : (usual ? k_mgcg_update<K, false, true> : k_mgcg_update<K, false, false>);
            f<<<tgrid, kBlock, 0, st>>>(P, L0, h, o.mg_omega, j, B.cx, pnew, B.cq, hdr, resid, red);
        }
        if (more) cycle(!one_level, 0);
    }
    LaunchScope ls(MPM_KERNEL_PCG_FINAL, st);
    k_mgcg_final<K><<<grid, kBlock, 0, st>>>(P.N, B.cx, delta, y_update, hdr, report_rel, report_it);
    return cudaGetLastError();
}

cudaError_t launch_solve_mg(const DevProblem& P, const SolveOpts& o, const float* h, const float* w,
                            const float* g, const float* y, float* delta, float* y_update,
                            double* resid, double* report_rel, int* report_it, void* solve_ws,
                            WsHeader* hdr, Reduce red, cudaStream_t st)
{
    if (P.K == 4)
        return solve_mg_k<4>(P, o, h, w, g, y, delta, y_update, resid, report_rel, report_it,
                             solve_ws, hdr, red, st);
    return solve_mg_k<3>(P, o, h, w, g, y, delta, y_update, resid, report_rel, report_it, solve_ws,
                         hdr, red, st);
}

}  // namespace mpm

// stencil_kernels.cu -- the prior and the Newton-system solve (sm_103a):
//   k_jtv_staged   JTV weights w_n = (u_n + eps^2)^-1/2 and JTV_eps (Eqs. 38-40);
//                  k_jtv for small volumes and very wide rows
//   k_pcg_init     r_0 = g + L y, p_0 = z_0 = M^-1 r_0 (Eq. 42)
//   k_pcg_step     one PCG iteration (pcg_step.cuh): z_j, p_j from the previous
//                  ones, q = (H + L) p_j, v = M^-1 q, the x fold and the
//                  sums for alpha_j and beta_j -- the plain kernel used when the
//                  TMA-staged one (stencil_tma.cu) does not apply
//   k_pcg_final    delta = x + pending directions (or y <- y - delta)
//
// L = G'WG (x) diag(lambda) is applied as the 7-point weighted stencil
//   (L v)_k[n] = lambda_k sum_{m in N(n)} (w_n + w_m)(v_k[n] - v_k[m]) / h^2,
// neighbours outside the volume dropped (Neumann).  Blocks cover a 32 x 8
// (x, y) tile and march along z.  All CG scalars (alpha, beta, |r|) live in
// device memory and are produced by the last block of each reducing launch,
// so the whole PCG runs without a host round trip.
#include <algorithm>
#include <type_traits>

#include "mpm_internal.cuh"
#include "pcg_step.cuh"
#include "tma_common.cuh"

namespace mpm {

// Edge coefficients c_j = (w_n + w_m) / h_j^2 of the six neighbours (0 when
// the neighbour is outside the volume) and their offsets.
struct Edges {
    float c[6];
    long long off[6];
    bool ok[6];
};

__device__ __forceinline__ void make_edges(const DevProblem& P, int x, int y, int z,
                                           long long n, const float* __restrict__ w,
                                           float wn, Edges& e)
{
    const long long sxy = (long long)P.nx * P.ny;
    e.off[0] = -1;        e.ok[0] = x > 0;
    e.off[1] = 1;         e.ok[1] = x < P.nx - 1;
    e.off[2] = -P.nx;     e.ok[2] = y > 0;
    e.off[3] = P.nx;      e.ok[3] = y < P.ny - 1;
    e.off[4] = -sxy;      e.ok[4] = z > 0;
    e.off[5] = sxy;       e.ok[5] = z < P.nz - 1;
    const float ih[6] = {P.ihx2, P.ihx2, P.ihy2, P.ihy2, P.ihz2, P.ihz2};
#pragma unroll
    for (int j = 0; j < 6; ++j)
        e.c[j] = e.ok[j] ? (wn + __ldg(w + n + e.off[j])) * ih[j] : 0.0f;
}

// ------------------------------------------------------------- JTV weights

// Whether every index the JTV kernel forms for this volume (K arrays of N
// values, with room to spare) fits in a signed 32-bit int: its address
// arithmetic is then 32-bit (114 -> 111 us at 176x240x256).
static bool index32(const DevProblem& P)
{
    return P.N * (long long)(P.K * (P.K + 1) / 2 + 1) < 0x7fffffffLL;
}

constexpr int kInitAhead = 2;     // planes between the PCG start's L2 hint and the use

// (b - a)^2 of one voxel or of two at once (paired instructions, each lane
// rounded as the single form), and s + q h of two.
__device__ __forceinline__ float sqdiff(float b, float a)
{
    const float d = __fsub_rn(b, a);
    return __fmul_rn(d, d);
}
__device__ __forceinline__ float2 sqdiff(float2 b, float2 a)
{
    const float2 d = __ffma2_rn(a, make_float2(-1.0f, -1.0f), b);   // b - a, one rounding
    return __fmul2_rn(d, d);
}
__device__ __forceinline__ float2 addmul(float2 q, float h, float2 s)
{
    return __ffma2_rn(q, make_float2(h, h), s);
}
// Square roots s of x and their reciprocals r, two at once and without a
// branch: Newton-Raphson from the hardware's 1/sqrt estimate y, s = x y + (x -
// (x y)^2) y / 2 and r = y + y (1 - s y), each within about half an ulp (the
// residuals are exact in the fused multiply-adds).  For x in [1e-30, 1e30].
__device__ __forceinline__ void sqrt_recip(float2 x, float2& s, float2& r)
{
    const float2 y = make_float2(rsqrtf(x.x), rsqrtf(x.y));
    const float2 s0 = __fmul2_rn(x, y), ns0 = make_float2(-s0.x, -s0.y);
    s = __ffma2_rn(__ffma2_rn(ns0, s0, x), __fmul2_rn(y, make_float2(0.5f, 0.5f)), s0);
    const float2 ns = make_float2(-s.x, -s.y);
    r = __ffma2_rn(y, __ffma2_rn(ns, y, make_float2(1.0f, 1.0f)), y);
}

// Two compensated accumulators side by side (Acc::add in paired instructions).
struct Acc2 {
    float2 hi = {0.f, 0.f}, lo = {0.f, 0.f};
    __device__ __forceinline__ static float2 neg(float2 v) { return make_float2(-v.x, -v.y); }
    __device__ __forceinline__ void add(float2 x)
    {
        const float2 s = __fadd2_rn(hi, x);
        const float2 bp = __fadd2_rn(s, neg(hi));
        const float2 e = __fadd2_rn(__fadd2_rn(hi, neg(__fadd2_rn(s, neg(bp)))), __fadd2_rn(x, neg(bp)));
        hi = s;
        lo = __fadd2_rn(lo, e);
    }
    __device__ __forceinline__ Acc sum() const
    {
        Acc a, b;
        a.hi = hi.x, a.lo = lo.x;
        b.hi = hi.y, b.lo = lo.y;
        a.add(b);
        return a;
    }
};

constexpr int kJtvThreads = 256;
constexpr int kJtvRun = 4 * kJtvThreads;   // voxels of a plane per block of the staged kernel
constexpr int kJtvStagesMax = 4;

// Floats of one map in a stage: the block's voxels, a row on either side and
// the rest of the 16-byte granules at both ends.
__host__ __device__ constexpr int jtv_slot(int nx) { return (kJtvRun + 2 * nx + 6 + 3) / 4 * 4; }

// The staged kernel.  A block takes 1024 consecutive voxels of a plane and
// marches up a z range.  What it needs of a plane -- its voxels and one row
// below and above them -- is one contiguous range of each map, so K lanes bring
// each plane into a ring of `stages` shared-memory stages with one bulk copy
// each, planes ahead of their use, whatever the alignment: a copy takes the
// 16-byte granules that hold the range, and the range starts `shift` floats
// into its slot.  (Granules that would reach out of y are left out and their
// floats copied one by one.)  Plane z and the squared differences to plane
// z - 1 stay in registers; the y neighbours and plane z + 1 come from the
// stages.  RUNS (rows and arrays on 16-byte boundaries): a thread takes four
// neighbouring voxels along x, shared accesses are 16 bytes, the x neighbours
// come from the neighbouring lanes and every squared difference along x serves
// both its voxels.  Otherwise a thread takes four voxels 256 apart, so that a
// warp's shared accesses are 32 consecutive floats.  The six terms of a voxel
// are summed in the order x-, x+, y-, y+, z-, z+ (a missing neighbour's term
// left out).
//
// 20 B per voxel: HBM-bound once the loads are in flight and the instructions
// few.  The 32 x 8 tile kernel below takes about 350 thread instructions per
// voxel, 108.7 us at 176x240x256 (0.29 of the copy bandwidth) and 78 us at
// 181x217x181.  Runs of four with their loads through L1: 80.2 us, bound by the
// latency of 16 warps' loads; staged, 77.7; with the paired square roots and
// sums and one wave of z ranges 63.5 us (90 us without RUNS), 181x217x181 58 us.
// One thread filling all maps' stages was 16 us slower: it is on the path from
// one plane's barrier to the next.
template <int K, bool RUNS, typename IT>
__device__ __forceinline__ void jtv_staged_body(const DevProblem& P, int zc, int stages,
                                                const float* __restrict__ y, float* __restrict__ w,
                                                double* jtv, Reduce red, unsigned* status,
                                                long long wait_cycles, int withhold, const VGrid& vg)
{
    extern __shared__ __align__(128) unsigned char smem_raw[];
    __shared__ __align__(8) uint64_t full[kJtvStagesMax];
    __shared__ volatile int s_fail;
    float* smem = reinterpret_cast<float*>(smem_raw);
    const IT N = (IT)P.N;
    const int nx = P.nx, ny = P.ny, nz = P.nz;
    const int sxy = nx * ny;                                 // at most 2^23 (check_problem)
    const int tid = threadIdx.x;
    const int z0 = (int)vg.bz * zc, z1 = min(nz, z0 + zc), zlast = min(z1, nz - 1);
    const int n0 = (int)vg.bx * kJtvRun;                     // this block's first voxel of a plane
    const int lo = max(n0 - nx, 0), hi = min(n0 + kJtvRun + nx, sxy);
    const int slot = jtv_slot(nx);
    const uint32_t bar0 = smem_u32(&full[0]);
    // floats by which the range of (map k, plane z) starts into its slot
    const unsigned ymod = (unsigned)(reinterpret_cast<uintptr_t>(y) >> 2);
    auto shift = [&](int k, int z) {
        return (int)((ymod + (unsigned)k * (unsigned)P.N + (unsigned)z * (unsigned)sxy + (unsigned)lo) & 3u);
    };
    // Lane k of the first warp brings plane z of map k into stage st (the K
    // copies of a stage complete its barrier together).
    auto fill = [&](int z, int st) {
        const int k = tid;
        const uint32_t bar = bar0 + 8 * st;
        const float* r = y + k * N + (IT)sxy * z + lo;                  // the range's first float
        const int len = hi - lo;
        if (RUNS) {                                                     // whole granules, inside y
            mbar_expect_tx(bar, (uint32_t)len * 4u);
            bulk_load(smem_u32(smem + (st * K + k) * slot), r, (uint32_t)len * 4u, bar);
            return;
        }
        const int sh = shift(k, z);
        float* d = smem + (st * K + k) * slot + sh;                     // its place
        int b = -sh, e = (sh + len + 3) / 4 * 4 - sh;                   // the granules, from r
        if (r + b < y) b += 4;
        if (r + e > y + K * N) e -= 4;
        const uint32_t bytes = e > b ? (uint32_t)(e - b) * 4u : 0u;
        mbar_expect_tx(bar, bytes);
        if (bytes) bulk_load(smem_u32(d + b), r + b, bytes, bar);
        for (int q = 0; q < b && q < len; ++q) d[q] = __ldg(r + q);
        for (int q = bytes ? e : max(b, 0); q < len; ++q) d[q] = __ldg(r + q);
        // a later copy of this lane writes the same floats through the async proxy
        if (b > 0 || e < len) fence_async_proxy();
    };
    if (tid == 0) {
        s_fail = 0;
        for (int st = 0; st < kJtvStagesMax; ++st) mbar_init(bar0 + 8 * st, K);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    __syncthreads();
    const bool feeds = tid < K && !withhold;
    int issued = 0;                                          // planes brought in (the feeding lanes)
    if (feeds)
        for (; issued < stages && z0 + issued <= zlast; ++issued) fill(z0 + issued, issued);
    if (!RUNS) __syncthreads();                              // the floats copied one by one
    bool bad = false;
    auto wait = [&](int st, uint32_t ph) {
        if (bad || mbar_try_wait(bar0 + 8 * st, ph)) return;
        if (s_fail || !mbar_wait(bar0 + 8 * st, ph, wait_cycles)) {
            bad = true;
            s_fail = 1;
        }
    };
    // The thread's four voxels, as two pairs: their places in the range
    // (clamped to it) and, in `ok`, five bits each: inside, x-, x+, y-, y+.
    const int lane = tid & 31;
    int o[4];
    unsigned ok = 0;
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const int v = n0 + (RUNS ? 4 * tid + i : i * kJtvThreads + tid);
        const int yy = v / nx, x = v - yy * nx;
        const bool in = v < sxy;
        o[i] = in ? v - lo : (RUNS ? i : 0);
        if (in)
            ok |= (1u | (x > 0 ? 2u : 0u) | (x < nx - 1 ? 4u : 0u) | (yy > 0 ? 8u : 0u) | (yy < ny - 1 ? 16u : 0u))
                  << (5 * i);
    }
    // RUNS: no lane's run lies at a y face
    const bool ymid = RUNS && __all_sync(0xffffffffu, !(ok & 1u) || (ok & 24u) == 24u);
    auto has = [&](int i, unsigned bit) { return (ok & (bit << (5 * i))) != 0; };
    auto only = [&](float2 q, int h, unsigned bit) {       // the terms of the neighbours that exist
        return make_float2(has(2 * h, bit) ? q.x : 0.0f, has(2 * h + 1, bit) ? q.y : 0.0f);
    };
    auto pair_at = [&](const float* p, int h, int d) {      // RUNS: both at once
        if constexpr (RUNS) return *reinterpret_cast<const float2*>(p + o[2 * h] + d);
        else return make_float2(p[o[2 * h] + d], p[o[2 * h + 1] + d]);
    };
    auto four_at = [&](const float* p, int d, float2 (&q)[2]) {
        if constexpr (RUNS) {
            const float4 v = *reinterpret_cast<const float4*>(p + o[0] + d);
            q[0] = make_float2(v.x, v.y);
            q[1] = make_float2(v.z, v.w);
        } else {
            q[0] = pair_at(p, 0, d);
            q[1] = pair_at(p, 1, d);
        }
    };
    // neighbour offset d of one voxel, 0 (the voxel itself) where it has none
    auto off = [&](int i, int d, unsigned bit) { return has(i, bit) ? d : 0; };
    float2 cu[K][2], zl[K][2];                               // plane z; squared differences to plane z - 1
    Acc2 acc;
    int st = 0;                                              // stage of plane z
    uint32_t ph = 0;                                         // phase of the ring's current turn
    wait(0, 0);
#pragma unroll
    for (int k = 0; k < K; ++k) {
        four_at(smem + k * slot + shift(k, z0), 0, cu[k]);
        zl[k][0] = zl[k][1] = make_float2(0.f, 0.f);
        if (z0 > 0 && (ok & 1u)) {
            float2 dn[2];
            const float* q = y + k * N + (IT)sxy * (z0 - 1) + lo;
            if constexpr (RUNS) {
                four_at(q, 0, dn);
            } else {
                dn[0] = make_float2(__ldg(q + o[0]), __ldg(q + o[1]));
                dn[1] = make_float2(__ldg(q + o[2]), __ldg(q + o[3]));
            }
            zl[k][0] = sqdiff(dn[0], cu[k][0]);
            zl[k][1] = sqdiff(dn[1], cu[k][1]);
        }
    }
    for (int z = z0; z < z1; ++z) {
        const bool above = z + 1 < nz;
        const int su = st + 1 == stages ? 0 : st + 1;        // stage of plane z + 1
        const uint32_t pu = su == 0 ? ph ^ 1u : ph;
        if (above) wait(su, pu);
        float2 uu[2];
        // MID: every voxel of the warp has its y neighbours and plane z + 1 exists
        auto plane = [&](auto mid) {
            constexpr bool MID = decltype(mid)::value;
#pragma unroll
            for (int k = 0; k < K; ++k) {
                const float* p = smem + (st * K + k) * slot + (RUNS ? 0 : shift(k, z));
                const float* u = above ? smem + (su * K + k) * slot + (RUNS ? 0 : shift(k, z + 1)) : p;
                const float2 a = cu[k][0], b = cu[k][1];
                float2 up[2], ym[2], yp[2], s[2];
                four_at(u, 0, up);
                if constexpr (RUNS) {
                    four_at(p, off(0, -nx, 8u), ym);
                    four_at(p, off(0, nx, 16u), yp);
                    float vl = __shfl_up_sync(0xffffffffu, b.y, 1);
                    float vr = __shfl_down_sync(0xffffffffu, a.x, 1);
                    if (lane == 0) vl = p[o[0] + off(0, -1, 2u)];
                    if (lane == 31) vr = p[o[3] + off(3, 1, 4u)];
                    const float ql = has(0, 2u) ? sqdiff(vl, a.x) : 0.0f, qr = has(3, 4u) ? sqdiff(vr, b.y) : 0.0f;
                    const float q01 = sqdiff(a.y, a.x), q12 = sqdiff(b.x, a.y), q23 = sqdiff(b.y, b.x);
                    const float2 h2 = make_float2(P.ihx2, P.ihx2);
                    s[0] = __ffma2_rn(make_float2(q01, q12), h2, __fmul2_rn(make_float2(ql, q01), h2));
                    s[1] = __ffma2_rn(make_float2(q23, qr), h2, __fmul2_rn(make_float2(q12, q23), h2));
                } else {
#pragma unroll
                    for (int h = 0; h < 2; ++h) {
                        const int i = 2 * h, j = i + 1;
                        const float2 xm = make_float2(p[o[i] + off(i, -1, 2u)], p[o[j] + off(j, -1, 2u)]);
                        const float2 xp = make_float2(p[o[i] + off(i, 1, 4u)], p[o[j] + off(j, 1, 4u)]);
                        ym[h] = make_float2(p[o[i] + off(i, -nx, 8u)], p[o[j] + off(j, -nx, 8u)]);
                        yp[h] = make_float2(p[o[i] + off(i, nx, 16u)], p[o[j] + off(j, nx, 16u)]);
                        s[h] = __fmul2_rn(only(sqdiff(xm, cu[k][h]), h, 2u), make_float2(P.ihx2, P.ihx2));
                        s[h] = addmul(only(sqdiff(xp, cu[k][h]), h, 4u), P.ihx2, s[h]);
                    }
                }
                const float2 l2 = make_float2(P.lambda[k], P.lambda[k]);
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    float2 ya = sqdiff(ym[h], cu[k][h]), yb = sqdiff(yp[h], cu[k][h]);
                    float2 zu = sqdiff(up[h], cu[k][h]);
                    if (!MID) {
                        ya = only(ya, h, 8u);
                        yb = only(yb, h, 16u);
                        if (!above) zu = make_float2(0.f, 0.f);
                    }
                    s[h] = addmul(ya, P.ihy2, s[h]);
                    s[h] = addmul(yb, P.ihy2, s[h]);
                    s[h] = addmul(zl[k][h], P.ihz2, s[h]);
                    s[h] = addmul(zu, P.ihz2, s[h]);
                    zl[k][h] = zu;
                    cu[k][h] = up[h];
                    uu[h] = k == 0 ? __fmul2_rn(l2, s[h]) : __ffma2_rn(l2, s[h], uu[h]);
                }
            }
        };
        if (RUNS && ymid && above) plane(std::true_type());
        else plane(std::false_type());
        if (!bad) {
            const float2 e2 = make_float2(P.eps2, P.eps2);
            const float2 va = __fadd2_rn(uu[0], e2), vb = __fadd2_rn(uu[1], e2);
            float2 sa, sb, ra, rb;
            const float vmin = fminf(fminf(va.x, va.y), fminf(vb.x, vb.y));
            const float vmax = fmaxf(fmaxf(va.x, va.y), fmaxf(vb.x, vb.y));
            const float vsum = (va.x + va.y) + (vb.x + vb.y);        // NaN if any value is
            if (vmin >= 1e-30f && vmax <= 1e30f && vsum == vsum) {
                sqrt_recip(va, sa, ra);
                sqrt_recip(vb, sb, rb);
            } else {
                sa = make_float2(sqrtf(va.x), sqrtf(va.y));
                sb = make_float2(sqrtf(vb.x), sqrtf(vb.y));
                ra = make_float2(1.0f / sa.x, 1.0f / sa.y);
                rb = make_float2(1.0f / sb.x, 1.0f / sb.y);
            }
            acc.add(only(sa, 0, 1u));
            acc.add(only(sb, 1, 1u));
            if (w) {
                float* wz = w + (IT)sxy * z + lo;
                if (RUNS) {
                    if (ok & 1u) *reinterpret_cast<float4*>(wz + o[0]) = make_float4(ra.x, ra.y, rb.x, rb.y);
                } else {
                    if (has(0, 1u)) wz[o[0]] = ra.x;
                    if (has(1, 1u)) wz[o[1]] = ra.y;
                    if (has(2, 1u)) wz[o[2]] = rb.x;
                    if (has(3, 1u)) wz[o[3]] = rb.y;
                }
            }
        }
        __syncthreads();
        // every thread has read plane z: its stage takes the next plane
        // (unless a wait gave up: no second copy in flight to a stage)
        if (feeds && !s_fail && z0 + issued <= zlast) {
            fill(z0 + issued, st);
            ++issued;
        }
        st = su;
        ph = pu;
    }
    if (s_fail) {
        // drain: the last copies into each stage (earlier ones were waited for)
        if (tid == 0) {
            for (int i = max(0, issued - stages); i < issued; ++i)
                mbar_wait(bar0 + 8 * (i % stages), (uint32_t)(i / stages) & 1u, wait_cycles);
            if (status) atomicOr(status, kStatusTimeout);
        }
        __syncthreads();
    }
    Acc v[1] = {acc.sum()};
    double out[1];
    if (grid_reduce<1>(v, red, out, vg) && threadIdx.x == 0) *jtv = out[0];
}

template <int K, bool RUNS, typename IT>
__global__ void __launch_bounds__(kJtvThreads, 2)
    k_jtv_staged(DevProblem P, int zc, int stages, const float* __restrict__ y, float* __restrict__ w,
                 double* jtv, Reduce red, unsigned* status, long long wait_cycles, int withhold)
{
    jtv_staged_body<K, RUNS, IT>(P, zc, stages, y, w, jtv, red, status, wait_cycles, withhold, hw_grid());
}

template <int K, bool RUNS, typename IT>
__global__ void __launch_bounds__(kJtvThreads, 2)
    k_jtv_staged_batch(const __grid_constant__ Batch<JtvArgs> b, long long wait_cycles, int withhold)
{
    const int s = batch_subject(b.start, b.n);
    const JtvArgs& a = b.a[s];
    jtv_staged_body<K, RUNS, IT>(a.P, a.zc, a.stages, a.y, a.w, a.jtv, a.red, a.status, wait_cycles, withhold,
                           batch_grid(b.start[s], a.gx, a.gy, a.gz));
}

// The tile kernel, for small volumes and rows too wide for three stages.
// Each thread marches up its z range with the centre values of planes z - 1,
// z and z + 1 in registers; the centre of plane z + 2 is loaded one plane
// ahead.  The x / y neighbours come from the plane's tile in shared memory
// (double-buffered, one barrier per plane): every thread writes its centre,
// and 80 threads the tile's halo (rows y0 - 1 and y0 + 8, columns x0 - 1 and
// x0 + 32), which they too load two planes ahead.  The six terms are summed in
// the order x-, x+, y-, y+, z-, z+.
template <int K, typename IT>
__device__ __forceinline__ void jtv_body(const DevProblem& P, int zc, const float* __restrict__ y,
                                         float* __restrict__ w, double* jtv, Reduce red, const VGrid& vg)
{
    constexpr int TW = kTileX + 2, TH = kTileY + 2;
    __shared__ float tile[2][K][TH][TW];
    const IT N = (IT)P.N;
    const int nx = P.nx, ny = P.ny, nz = P.nz;
    const IT sxy = (IT)nx * ny;
    const int tx = threadIdx.x, ty = threadIdx.y;
    const int x = vg.bx * kTileX + tx;
    const int yy = vg.by * kTileY + ty;
    const int z0 = vg.bz * zc;
    const int z1 = min(nz, z0 + zc);
    // this thread's halo point, if any: its place in the tile and the volume
    const int t = ty * kTileX + tx;
    int hx = -1, hy = -1, hr = 0, hc = 0;
    if (t < 2 * kTileX) {                       // rows above and below the tile
        hr = t < kTileX ? 0 : TH - 1;
        hc = 1 + t % kTileX;
    } else if (t < 2 * kTileX + 2 * kTileY) {   // columns left and right
        const int u = t - 2 * kTileX;
        hr = 1 + u % kTileY;
        hc = u < kTileY ? 0 : TW - 1;
    }
    if (t < 2 * kTileX + 2 * kTileY) {
        hx = vg.bx * kTileX + hc - 1;
        hy = vg.by * kTileY + hr - 1;
    }
    const bool halo = hx >= 0 && hx < nx && hy >= 0 && hy < ny;
    const bool inside = x < nx && yy < ny;
    Acc acc;
    if (z0 < z1) {
        const IT base = inside ? x + (IT)nx * yy : 0;
        const IT hbase = halo ? hx + (IT)nx * hy : 0;
        const bool okx0 = x > 0, okx1 = x < nx - 1, oky0 = yy > 0, oky1 = yy < ny - 1;
        float dn[K], cu[K], up[K], nx2[K], h0[K], h1[K], h2[K];
#pragma unroll
        for (int k = 0; k < K; ++k) {
            const float* yk = y + k * N + base;
            const float* hk = y + k * N + hbase;
            cu[k] = inside ? __ldg(yk + sxy * z0) : 0.0f;
            dn[k] = inside && z0 > 0 ? __ldg(yk + sxy * (z0 - 1)) : 0.0f;
            up[k] = inside && z0 + 1 < nz ? __ldg(yk + sxy * (z0 + 1)) : 0.0f;
            h0[k] = halo ? __ldg(hk + sxy * z0) : 0.0f;
            h1[k] = halo && z0 + 1 < z1 ? __ldg(hk + sxy * (z0 + 1)) : 0.0f;
        }
        for (int z = z0; z < z1; ++z) {
            const int b = z & 1;
            const IT n = base + sxy * z;
            const bool okz0 = z > 0, okz1 = z < nz - 1;
#pragma unroll
            for (int k = 0; k < K; ++k) {
                tile[b][k][ty + 1][tx + 1] = cu[k];
                if (t < 2 * kTileX + 2 * kTileY) tile[b][k][hr][hc] = h0[k];
            }
            // the centre two planes up, and the halo two planes up, for later steps
#pragma unroll
            for (int k = 0; k < K; ++k) {
                nx2[k] = inside && z + 2 < nz && z + 1 < z1 ? __ldg(y + k * N + n + 2 * sxy) : 0.0f;
                h2[k] = halo && z + 2 < z1 ? __ldg(y + k * N + hbase + sxy * (z + 2)) : 0.0f;
            }
            __syncthreads();
            if (inside) {
                float u = 0.0f;
#pragma unroll
                for (int k = 0; k < K; ++k) {
                    const float v = cu[k];
                    float s = 0.0f;
                    float d;
                    if (okx0) { d = tile[b][k][ty + 1][tx] - v; s += d * d * P.ihx2; }
                    if (okx1) { d = tile[b][k][ty + 1][tx + 2] - v; s += d * d * P.ihx2; }
                    if (oky0) { d = tile[b][k][ty][tx + 1] - v; s += d * d * P.ihy2; }
                    if (oky1) { d = tile[b][k][ty + 2][tx + 1] - v; s += d * d * P.ihy2; }
                    if (okz0) { d = dn[k] - v; s += d * d * P.ihz2; }
                    if (okz1) { d = up[k] - v; s += d * d * P.ihz2; }
                    u += P.lambda[k] * s;
                }
                const float val = u + P.eps2;
                const float sq = sqrtf(val);
                if (w) w[n] = 1.0f / sq;
                acc.add(sq);
            }
#pragma unroll
            for (int k = 0; k < K; ++k) {
                dn[k] = cu[k];
                cu[k] = up[k];
                up[k] = nx2[k];
                h0[k] = h1[k];
                h1[k] = h2[k];
            }
        }
    }
    Acc v[1] = {acc};
    double out[1];
    if (grid_reduce<1>(v, red, out, vg) && threadIdx.x == 0 && threadIdx.y == 0) *jtv = out[0];
}

template <int K, typename IT>
__global__ void __launch_bounds__(kBlock) k_jtv(DevProblem P, int zc, const float* __restrict__ y,
                                                float* __restrict__ w, double* jtv, Reduce red)
{
    jtv_body<K, IT>(P, zc, y, w, jtv, red, hw_grid());
}

template <int K, typename IT>
__global__ void __launch_bounds__(kBlock) k_jtv_batch(const __grid_constant__ Batch<JtvArgs> b)
{
    const int s = batch_subject(b.start, b.n);
    const JtvArgs& a = b.a[s];
    jtv_body<K, IT>(a.P, a.zc, a.y, a.w, a.jtv, a.red, batch_grid(b.start[s], a.gx, a.gy, a.gz));
}

// ------------------------------------------------------ solve workspace

static size_t align256(size_t b) { return (b + 255) & ~(size_t)255; }

// v[2], p[3], x and z[2], each [N] float4.
static size_t pcg_bytes(const DevProblem& P, int vecs = 8) { return vecs * align256(sizeof(float4) * (size_t)P.N); }

// Copies of w and H with rows padded to a multiple of 4 floats (16 bytes), the
// row pitch the copy engine needs, for volumes whose x size is not one: the
// staged iteration then applies to them too.  The PCG start writes them as it
// reads w and H.  Solve of 181x217x181, 30 iterations: 9.61 ms with the plain
// iteration, 5.36 ms this way.
struct PackedRows {
    int pitch;           // floats per row
    size_t plane;        // floats per array
    float *w, *h;        // [plane], [T][plane]
};

static size_t packed_rows(const DevProblem& P, char* at, PackedRows* out)
{
    PackedRows r;
    r.pitch = (P.nx + 3) / 4 * 4;
    r.plane = (size_t)r.pitch * P.ny * P.nz;
    const size_t w = align256(sizeof(float) * r.plane);
    r.w = reinterpret_cast<float*>(at);
    r.h = at ? reinterpret_cast<float*>(at + w) : nullptr;
    if (out) *out = r;
    return w + align256(sizeof(float) * P.T * r.plane);
}

static bool wants_packed(const DevProblem& P)
{
    return P.nx % 4 != 0 && tma_tile_fits(P, tma_tile_choice(P));
}

// (The multigrid solver's need is the larger one but for volumes of up to 512
// voxels, whose z[1] lies elsewhere where there is no room for it, see carve.)
size_t solve_ws_least(const DevProblem& P) { return std::max(pcg_bytes(P, 7), mg_ws_bytes(P)); }

// The larger of the two solvers' needs; with rows to pad, room for their copies.
size_t solve_ws_bytes(const DevProblem& P)
{
    const size_t least = solve_ws_least(P);
    return P.nx % 4 ? std::max(least, pcg_bytes(P) + packed_rows(P, nullptr, nullptr)) : least;
}

SolveOpts solve_opts(const mpm_opts& o, bool overlap)
{
    SolveOpts s;
    s.cg_iters = o.cg_iters;
    s.tol_cg = o.tol_cg;
    s.mg_levels = o.mg_levels;
    s.mg_nu = o.mg_nu > 0 ? o.mg_nu : 1;
    s.mg_omega = o.mg_omega > 0.0 ? (float)o.mg_omega : 0.7f;
    s.mg_coarse_sweeps = o.mg_coarse_sweeps > 0 ? o.mg_coarse_sweeps : 20;
    s.overlap = overlap;
    return s;
}

// Without room for eight vectors (at most 512 voxels), z[1] takes the part of
// the reduction partials that the iteration's seven sums leave.
static SolveBufs carve(const DevProblem& P, void* ws, size_t ws_bytes, Reduce red)
{
    SolveBufs b;
    char* c = static_cast<char*>(ws);
    const size_t vec = align256(sizeof(float4) * (size_t)P.N);
    for (float4*& v : b.v) { v = reinterpret_cast<float4*>(c); c += vec; }
    for (float4*& v : b.p) { v = reinterpret_cast<float4*>(c); c += vec; }
    b.x = reinterpret_cast<float4*>(c);
    b.z[0] = reinterpret_cast<float4*>(c + vec);
    b.z[1] = ws_bytes >= pcg_bytes(P) ? reinterpret_cast<float4*>(c + 2 * vec)
                                      : reinterpret_cast<float4*>(red.partials + (size_t)kStepSums * kMaxBlocks);
    return b;
}

// --------------------------------------------------------------- PCG init

// PACKED: also writes the padded copies of w and H.  A template parameter,
// because the test at run time took 58 registers instead of 48, one block per
// SM less: 299 us instead of 233 at 176x240x256, where load latency bounds it
// (bounds of 6 and 8 blocks per SM: 241 and 301 us).
template <int K, bool PACKED>
__device__ __forceinline__ void pcg_init_body(const DevProblem& P, int zc, const float* __restrict__ h,
                                              const float* __restrict__ w, const float* __restrict__ g,
                                              const float* __restrict__ y, float4* __restrict__ p0,
                                              double tol2, WsHeader* hdr, double* resid, Reduce red,
                                              const PackedRows& rows, const VGrid& vg)
{
    constexpr int T = K * (K + 1) / 2;
    const long long N = P.N;
    const long long sxy = (long long)P.nx * P.ny;
    const int x = vg.bx * kTileX + threadIdx.x;
    const int yy = vg.by * kTileY + threadIdx.y;
    const int z0p = vg.bz * zc;
    const int z1p = min(P.nz, z0p + zc);
    Acc rz, rr;
    bool pd = true;
    if (x < P.nx && yy < P.ny) {
        for (int z = z0p; z < z1p; ++z) {
            const long long n = x + (long long)P.nx * yy + sxy * z;
            // the operands of plane z + kInitAhead into L2 while plane z is computed
            if (z + kInitAhead < z1p) {
                const long long na = n + kInitAhead * sxy;
                prefetch_l2(w + na);
#pragma unroll
                for (int k = 0; k < K; ++k) {
                    prefetch_l2(y + k * N + na);
                    prefetch_l2(g + k * N + na);
                }
#pragma unroll
                for (int t = 0; t < T; ++t) prefetch_l2(h + t * N + na);
            }
            const float wn = __ldg(w + n);
            Edges e;
            make_edges(P, x, yy, z, n, w, wn, e);
            float r[K];
#pragma unroll
            for (int k = 0; k < K; ++k) {
                const float* yk = y + k * N;
                const float v = __ldg(yk + n);
                float s = 0.0f;
#pragma unroll
                for (int j = 0; j < 6; ++j)
                    if (e.ok[j]) s += e.c[j] * (v - __ldg(yk + n + e.off[j]));
                r[k] = __ldg(g + k * N + n) + P.lambda[k] * s;
            }
            float hv[T], M[K][K];
#pragma unroll
            for (int t = 0; t < T; ++t) hv[t] = __ldg(h + t * N + n);
            if constexpr (PACKED) {
                const size_t np = x + (size_t)rows.pitch * (yy + (size_t)P.ny * z);
                rows.w[np] = wn;
#pragma unroll
                for (int t = 0; t < T; ++t) rows.h[t * rows.plane + np] = hv[t];
            }
            precond_block<K>(P, hv, edge_sum(e.c), M);
            float L[T], zz[K];
            pd &= cholesky_f32<K>(M, L);
            chol_apply<K>(L, r, zz);
            p0[n] = pack4<K>(zz);
            float vrz = 0.0f, vrr = 0.0f;
#pragma unroll
            for (int k = 0; k < K; ++k) {
                vrz += r[k] * zz[k];
                vrr += r[k] * r[k];
            }
            rz.add(vrz);
            rr.add(vrr);
        }
    }
    if (!pd) atomicOr(&hdr->status, kStatusNotPD);
    release_dependents();
    Acc v[2] = {rz, rr};
    double out[2];
    if (grid_reduce<2>(v, red, out, vg) && threadIdx.x == 0 && threadIdx.y == 0) {
        SolveScalars& sc = hdr->sc;
        sc.rz = out[0];
        sc.rr0 = out[1];
        sc.rr = out[1];
        sc.alpha = 0.0;
        sc.alpha_prev = 0.0;
        sc.beta = 0.0;
        sc.beta_prev = 0.0;
        sc.pz = 1.0f;
        sc.zin = sc.zout = 0;
        sc.it = 0;
        sc.xcount = 0;
        sc.tol2 = tol2;
        const bool bad = !(out[0] == out[0]) || !(out[1] == out[1]);
        if (bad) atomicOr(&hdr->status, kStatusNaN);
        sc.done = (bad || !(out[0] > 0.0) || (tol2 > 0.0 && out[1] <= tol2 * out[1])) ? 1 : 0;
        if (resid) resid[0] = sqrt(out[1]);
    }
}

template <int K, bool PACKED>
__global__ void __launch_bounds__(kBlock) k_pcg_init(DevProblem P, int zc, const float* __restrict__ h,
                                                     const float* __restrict__ w,
                                                     const float* __restrict__ g,
                                                     const float* __restrict__ y, float4* __restrict__ p0,
                                                     double tol2, WsHeader* hdr, double* resid,
                                                     Reduce red, PackedRows rows)
{
    pcg_init_body<K, PACKED>(P, zc, h, w, g, y, p0, tol2, hdr, resid, red, rows, hw_grid());
}

template <int K>
__global__ void __launch_bounds__(kBlock) k_pcg_init_batch(const __grid_constant__ Batch<InitArgs> b)
{
    const int s = batch_subject(b.start, b.n);
    const InitArgs& a = b.a[s];
    pcg_init_body<K, false>(a.P, a.zc, a.h, a.w, a.g, a.y, a.p0, a.tol2, a.hdr, a.resid, a.red, PackedRows{},
                     batch_grid(b.start[s], a.gx, a.gy, a.gz));
}

// -------------------------------------------------------- PCG iteration

// Plain form of one PCG iteration (pcg_step.cuh): a thread per (x, y) column
// marching a run of z planes; each neighbour's p_j is formed from its own
// p_{j-1}, v_{j-1} and p_{j-2} (or the stored z_{j-1}) read from memory.  Used
// for volumes or pointers the TMA kernel cannot take (a volume smaller than a tile, unaligned buffers).
// MINB blocks per SM: three, with a few registers spilled, where the launch has as
// many, because the latency of the neighbours' loads bounds it (30 iterations of
// 2x1024x512 with four maps 11.1 ms, 11.5 with the two that 106 registers leave;
// three maps 9.9 and 13.0); two, without spills, for smaller launches (17x16x15
// 30 iterations 297 us, 313 with three).
template <int K, int MODE, int MINB>
__global__ void __launch_bounds__(kBlock, MINB) k_pcg_step(DevProblem P, int zc, int j, int want_rr,
                                                     const float* __restrict__ h,
                                                     const float* __restrict__ w,
                                                     const float4* __restrict__ pin,
                                                     const float4* __restrict__ vin,
                                                     const float4* __restrict__ p2,
                                                     const float4* __restrict__ zprev,
                                                     float4* __restrict__ vout,
                                                     float4* __restrict__ pout, float4* __restrict__ xacc,
                                                     float4* __restrict__ zout, WsHeader* hdr,
                                                     double* resid, Reduce red)
{
    constexpr int T = K * (K + 1) / 2;
    constexpr bool first = MODE == kModeFirst;
    __shared__ StepScalars s_sc;
    __shared__ int s_done;
    const int tid = threadIdx.x + threadIdx.y * blockDim.x;
    wait_predecessor();
    if (tid == 0) {
        s_done = hdr->sc.done;
        s_sc = step_start(hdr->sc);
    }
    __syncthreads();
    if (s_done) return;
    if (MODE >= kModeFold && tid == 0 && blockIdx.x == 0 && blockIdx.y == 0 && blockIdx.z == 0)
        hdr->sc.xcount = j;
    const StepScalars sc = s_sc;
    const long long sxy = (long long)P.nx * P.ny;
    const int x = blockIdx.x * kTileX + threadIdx.x;
    const int yy = blockIdx.y * kTileY + threadIdx.y;
    const int z0p = blockIdx.z * zc;
    const int z1p = min(P.nz, z0p + zc);
    float part[kStepSums] = {};
    const float4 zero = make_float4(0.f, 0.f, 0.f, 0.f);
    // A copy of the loop for each case of a stored z: with a test at each of a
    // voxel's seven points, 30 iterations of 2x1024x512 with three maps took 13.6
    // ms, with the test of zout alone 12.0, where without either they took 10.9.
    auto march = [&](auto zin_c, auto zout_c) {
        constexpr bool ZIN = decltype(zin_c)::value, ZOUT = decltype(zout_c)::value;
        const float4* __restrict__ pz = ZIN ? zprev : p2;
        auto point = [&](long long m, Maps& zj, Maps& pj) {
            step_point<MODE>(sc, ZIN, pin[m], first ? zero : vin[m], MODE >= kModeStep ? pz[m] : zero, zj, pj);
        };
        for (int z = z0p; z < z1p; ++z) {
            const long long n = x + (long long)P.nx * yy + sxy * z;
            const float wn = __ldg(w + n);
            Edges e;
            make_edges(P, x, yy, z, n, w, wn, e);
            Maps zj, pj, nb[6];
            point(n, zj, pj);
#pragma unroll
            for (int m = 0; m < 6; ++m) {
                Maps zm;
                if (e.ok[m]) point(n + e.off[m], zm, nb[m]);
                else nb[m] = pj;
            }
            float hv[T];
#pragma unroll
            for (int t = 0; t < T; ++t) hv[t] = __ldg(h + t * P.N + n);
            Maps v;
            step_voxel<K>(P, e.c, zj, pj, [&](int m) { return nb[m]; }, hv, want_rr, v, part);
            if (!first) pout[n] = pj.vec();
            if (ZOUT) zout[n] = zj.vec();
            vout[n] = v.vec();
            if (MODE >= kModeFold) xacc[n] = fold_x(MODE == kModeFoldX ? xacc[n] : zero, sc, p2[n], pin[n]).vec();
        }
    };
    if (x < P.nx && yy < P.ny) {
        using Zin = std::bool_constant<(MODE >= kModeStep)>;      // z_{j-1} may have been stored
        using Zout = std::bool_constant<!first>;
        using No = std::false_type;
        if (Zin::value && sc.zin) {
            if (sc.zout) march(Zin(), Zout());
            else march(Zin(), No());
        } else if (Zout::value && sc.zout) {
            march(No(), Zout());
        } else {
            march(No(), No());
        }
    }
    release_dependents();
    Acc acc[kStepSums];
#pragma unroll
    for (int i = 0; i < kStepSums; ++i) acc[i].add(part[i]);
    double out[kStepSums];
    if (grid_reduce<kStepSums>(acc, red, out, hw_grid(), want_rr ? kStepSums : kSumRR) && tid == 0)
        step_scalars(out, j, want_rr, hdr, resid);
}

// -------------------------------------------------------------- PCG final

// Grid-stride voxels whose operands a thread of the final kernel loads
// together: two in the solo kernel (171 -> 134 us at 176x240x256), one in the
// batched kernel, whose share of blocks per subject counts on the occupancy of
// its 40 registers (two voxels: 76 registers, phase-batched fits 2% slower).
constexpr int kFinalUnroll = 2;

// delta = x + the directions not yet folded into x (none, p_{it-1}, or
// p_{it-2} and p_{it-1}), written planar, or y <- y - delta.  Each thread
// loads the operands of U voxels (one grid stride apart) before it combines
// and stores them, so that more reads are in flight per thread.
template <int K, int U>
__device__ __forceinline__ void pcg_final_body(long long N, const SolveBufs& B, float* __restrict__ delta,
                                               float* __restrict__ y_update, const WsHeader* hdr,
                                               double* report_rel, int* report_it, const VGrid& vg)
{
    wait_predecessor();
    const SolveScalars sc = hdr->sc;
    const bool have_x = sc.xcount > 0;
    const int pend = sc.it - sc.xcount;        // directions not yet in x: 0, 1 or 2
    const float alpha = (float)sc.alpha, alpha_prev = (float)sc.alpha_prev;
    const float4* __restrict__ pp = B.p[(sc.it + 2) % 3];    // p_{it-1}
    const float4* __restrict__ pp2 = B.p[(sc.it + 1) % 3];   // p_{it-2} when pend == 2
    const float4 zero4 = make_float4(0.f, 0.f, 0.f, 0.f);
    const long long stride = (long long)vg.gx * blockDim.x;
    for (long long n0 = vg.bx * (long long)blockDim.x + threadIdx.x; n0 < N; n0 += U * stride) {
        float4 xv[U], p1[U], p2[U];
        float yv[U][K];
#pragma unroll
        for (int i = 0; i < U; ++i) {
            const long long n = n0 + i * stride;
            const bool in = n < N;
            xv[i] = in && have_x ? B.x[n] : zero4;
            p2[i] = in && pend == 2 ? pp2[n] : zero4;
            p1[i] = in && pend >= 1 ? pp[n] : zero4;
#pragma unroll
            for (int a = 0; a < K; ++a) yv[i][a] = in && y_update ? y_update[a * N + n] : 0.0f;
        }
#pragma unroll
        for (int i = 0; i < U; ++i) {
            const long long n = n0 + i * stride;
            if (n >= N) break;
            float v[K], t[K];
            if (have_x) {
                unpack4<K>(xv[i], v);
            } else {
#pragma unroll
                for (int a = 0; a < K; ++a) v[a] = 0.0f;
            }
            if (pend == 2) {
                unpack4<K>(p2[i], t);
#pragma unroll
                for (int a = 0; a < K; ++a) v[a] = fmaf(alpha_prev, t[a], v[a]);
            }
            if (pend >= 1) {
                unpack4<K>(p1[i], t);
#pragma unroll
                for (int a = 0; a < K; ++a) v[a] = fmaf(alpha, t[a], v[a]);
            }
#pragma unroll
            for (int a = 0; a < K; ++a) {
                if (y_update)
                    y_update[a * N + n] = yv[i][a] - v[a];
                else
                    delta[a * N + n] = v[a];
            }
        }
    }
    if (vg.bx == 0 && threadIdx.x == 0) {
        if (report_rel) *report_rel = sc.rr0 > 0.0 ? sqrt(sc.rr / sc.rr0) : 0.0;
        if (report_it) *report_it = sc.it;
    }
}

template <int K>
__global__ void __launch_bounds__(kBlock) k_pcg_final(long long N, SolveBufs B,
                                                      float* __restrict__ delta,
                                                      float* __restrict__ y_update,
                                                      const WsHeader* hdr, double* report_rel,
                                                      int* report_it)
{
    pcg_final_body<K, kFinalUnroll>(N, B, delta, y_update, hdr, report_rel, report_it, hw_grid());
}

template <int K>
__global__ void __launch_bounds__(kBlock) k_pcg_final_batch(const __grid_constant__ Batch<FinalArgs> b)
{
    const int s = batch_subject(b.start, b.n);
    const FinalArgs& a = b.a[s];
    pcg_final_body<K, 1>(a.N, a.B, a.delta, a.y_update, a.hdr, a.report_rel, a.report_it,
                      batch_grid(b.start[s], b.start[s + 1] - b.start[s], 1, 1));
}

// ------------------------------------------------------------- launchers

StencilGrid stencil_grid(const DevProblem& P, int tx, int ty, int waves, double share)
{
    StencilGrid sg;
    sg.block = dim3(tx, ty, 1);
    const int gx = (P.nx + tx - 1) / tx;
    const int gy = (P.ny + ty - 1) / ty;
    const long long tiles = (long long)gx * gy;
    // about `waves` waves of 8 resident blocks per SM (times this volume's
    // share of a launch serving several), at most kMaxBlocks blocks
    const long long target = std::max(1LL, (long long)(share * waves * 8 * kNumSm));
    long long gz = target / (tiles > 0 ? tiles : 1);
    if (gz < 1) gz = 1;
    if (gz > P.nz) gz = P.nz;
    while (tiles * gz > kMaxBlocks && gz > 1) --gz;
    sg.zc = (int)((P.nz + gz - 1) / gz);
    gz = (P.nz + sg.zc - 1) / sg.zc;
    sg.grid = dim3(gx, gy, (unsigned)gz);
    return sg;
}

// Stages of the staged JTV kernel for this volume: as many as leave two blocks
// per SM, at least three (plane z, plane z + 1 and one in flight) within a
// block's shared memory; 0 (the tile kernel) where those do not fit, rows of
// more than 1831 voxels at K = 4, and for small volumes, where the staged
// kernel's longer start-up costs what it gives (64^3: 14.3 us staged, 14.6 not;
// without runs of four, 61^3: 15.4 and 12.9; 181x217x181: 58 and 78), and for
// planes that leave a block's 1024 voxels mostly empty.
constexpr long long kJtvStagedMinRuns = 1LL << 17, kJtvStagedMin = 1LL << 20;
constexpr int kJtvSmemHalf = 110 * 1024, kJtvSmemMax = 220 * 1024;

static int jtv_smem(const DevProblem& P, int stages) { return 4 * P.K * jtv_slot(P.nx) * stages; }

static bool jtv_runs(const DevProblem& P, const float* y, const float* w)
{
    return P.nx % 4 == 0 && (reinterpret_cast<uintptr_t>(y) | reinterpret_cast<uintptr_t>(w)) % 16 == 0;
}

// Whether a plane has work enough for the staged kernel's blocks: one of them
// takes as long as 2.3 tiles of 32 x 8 (2.9 without runs of four), so planes of
// one or two tiles are faster in the tile kernel (8x8x8192 31.3 us, 48.8 staged;
// 13x15x7000 43.1 and 53.1; 16x16x10000 54.2 and 57.0; but 16x20x6000 48.4 and
// 37.1), those of two in long volumes only (16x16x4096 30.7 and 29.0; 16x16x1024
// 21.0 and 15.2).
static bool jtv_plane_fills(const DevProblem& P, bool runs)
{
    const long long tiles = (long long)((P.nx + kTileX - 1) / kTileX) * ((P.ny + kTileY - 1) / kTileY);
    const long long blocks = ((long long)P.nx * P.ny + kJtvRun - 1) / kJtvRun;
    return 10 * tiles >= (runs ? 23 : 29) * blocks || (runs && tiles >= 2 * blocks && P.N <= kJtvStagedMin);
}

static int jtv_stages(const DevProblem& P, bool runs)
{
    if (P.N < (runs ? kJtvStagedMinRuns : kJtvStagedMin) || !jtv_plane_fills(P, runs)) return 0;
    for (int n = kJtvStagesMax; n >= 3; --n)
        if (jtv_smem(P, n) <= (n > 3 ? kJtvSmemHalf : kJtvSmemMax)) return n;
    return 0;
}

// Grid of the JTV kernel.  Staged: blocks over the voxels of a plane times z
// ranges, the split of grid_chunks over the resident blocks (a range also reads
// the planes below and above it, as an item of the PCG iteration does); a
// subject that shares a launch takes `share` of the blocks.
static void jtv_grid(const DevProblem& P, int stages, double share, JtvArgs& a)
{
    a.stages = stages;
    if (!stages) {
        const StencilGrid sg = stencil_grid(P, kTileX, kTileY, 2, share);
        a.zc = sg.zc;
        a.gx = sg.grid.x;
        a.gy = sg.grid.y;
        a.gz = sg.grid.z;
        return;
    }
    const long long bx = ((long long)P.nx * P.ny + kJtvRun - 1) / kJtvRun;
    const int per_sm = jtv_smem(P, stages) <= kJtvSmemHalf ? 2 : 1;
    const int gz = grid_chunks(bx, P.nz, std::max(1LL, (long long)(share * per_sm * kNumSm)), kMaxBlocks);
    a.zc = (P.nz + gz - 1) / gz;
    a.gx = (unsigned)bx;
    a.gy = 1;
    a.gz = (unsigned)((P.nz + a.zc - 1) / a.zc);
}

template <int K, bool RUNS, typename IT>
static cudaError_t jtv_smem_opt_in()
{
    static OncePerDevice solo, batch;
    const cudaError_t e = smem_opt_in(solo, k_jtv_staged<K, RUNS, IT>, kJtvSmemMax);
    return e ? e : smem_opt_in(batch, k_jtv_staged_batch<K, RUNS, IT>, kJtvSmemMax);
}

template <int K>
static cudaError_t prime_jtv_k()
{
    cudaError_t e = jtv_smem_opt_in<K, true, int>();
    if (!e) e = jtv_smem_opt_in<K, true, long long>();
    if (!e) e = jtv_smem_opt_in<K, false, int>();
    if (!e) e = jtv_smem_opt_in<K, false, long long>();
    return e;
}

cudaError_t prime_jtv_kernels()
{
    const cudaError_t e = prime_jtv_k<4>();
    return e ? e : prime_jtv_k<3>();
}

template <int K, bool RUNS, typename IT>
static cudaError_t launch_jtv_staged(const JtvArgs& a, cudaStream_t st)
{
    const cudaError_t e = jtv_smem_opt_in<K, RUNS, IT>();
    if (e) return e;
    k_jtv_staged<K, RUNS, IT><<<dim3(a.gx, a.gy, a.gz), kJtvThreads, jtv_smem(a.P, a.stages), st>>>(
        a.P, a.zc, a.stages, a.y, a.w, a.jtv, a.red, a.status, copy_wait_cycles(), copy_withhold());
    return cudaGetLastError();
}

template <int K, typename IT>
static cudaError_t launch_jtv_k(const JtvArgs& a, cudaStream_t st)
{
    if (a.stages)
        return jtv_runs(a.P, a.y, a.w) ? launch_jtv_staged<K, true, IT>(a, st)
                                       : launch_jtv_staged<K, false, IT>(a, st);
    k_jtv<K, IT><<<dim3(a.gx, a.gy, a.gz), dim3(kTileX, kTileY, 1), 0, st>>>(a.P, a.zc, a.y, a.w, a.jtv, a.red);
    return cudaGetLastError();
}

cudaError_t launch_jtv(const DevProblem& P, const float* y, float* w, double* jtv, Reduce red,
                       unsigned* status, cudaStream_t st)
{
    JtvArgs a{P, 0, 0, 0, 0, 0, y, w, jtv, red, status};
    jtv_grid(P, jtv_stages(P, jtv_runs(P, y, w)), 1.0, a);
    LaunchScope ls(MPM_KERNEL_JTV, st);
    if (P.K == 4) return index32(P) ? launch_jtv_k<4, int>(a, st) : launch_jtv_k<4, long long>(a, st);
    return index32(P) ? launch_jtv_k<3, int>(a, st) : launch_jtv_k<3, long long>(a, st);
}

// What iteration j of a solve does besides the common work.
int step_mode(int j)
{
    if (j == 0) return kModeFirst;
    if (j == 1) return kModeSecond;
    if (j % 2) return kModeStep;
    return j == 2 ? kModeFold : kModeFoldX;
}

template <int K>
static cudaError_t launch_step_plain(const DevProblem& P, const StencilGrid& sg, int j, int want_rr,
                              const float* h, const float* w, const SolveBufs& B, WsHeader* hdr,
                              double* resid, Reduce red, bool overlap, cudaStream_t st)
{
    const int jm = j > 0 ? j - 1 : 0;
    const float4 *pin = B.p[jm % 3], *vin = B.v[jm & 1], *p2 = B.p[(j + 1) % 3];
    const float4* zprev = B.z[jm & 1];
    float4 *vout = B.v[j & 1], *pout = B.p[j % 3], *zout = B.z[j & 1];
    cudaError_t e;
    const bool few = (long long)sg.grid.x * sg.grid.y * sg.grid.z <= 2 * kNumSm;
#define MPM_STEP_PLAIN(M)                                                                          \
    e = launch_dependent(overlap, few ? k_pcg_step<K, M, 2> : k_pcg_step<K, M, 3>, sg.grid, sg.block, 0, st, P, sg.zc, j, want_rr, h, w, pin, vin, p2, \
                         zprev, vout, pout, B.x, zout, hdr, resid, red)
    switch (step_mode(j)) {
    case kModeFirst: MPM_STEP_PLAIN(kModeFirst); break;
    case kModeSecond: MPM_STEP_PLAIN(kModeSecond); break;
    case kModeStep: MPM_STEP_PLAIN(kModeStep); break;
    case kModeFold: MPM_STEP_PLAIN(kModeFold); break;
    default: MPM_STEP_PLAIN(kModeFoldX); break;
    }
#undef MPM_STEP_PLAIN
    return e;
}

template <int K>
static cudaError_t solve_k(const DevProblem& P, const SolveOpts& so, const float* h,
                           const float* w, const float* g, const float* y, float* delta,
                           float* y_update, double* resid, double* report_rel, int* report_it,
                           void* solve_ws, size_t ws_bytes, WsHeader* hdr, Reduce red, cudaStream_t st)
{
    const StencilGrid sg = stencil_grid(P, kTileX, kTileY);
    const StencilGrid ig = stencil_grid(P, kTileX, kTileY, kInitWaves);
    SolveBufs B = carve(P, solve_ws, ws_bytes, red);
    const int cg_iters = so.cg_iters;
    const double tol2 = so.tol_cg > 0.0 ? so.tol_cg * so.tol_cg : 0.0;
    StepMaps maps;
    const int tile = tma_tile_choice(P);
    PackedRows rows{};
    bool tma;
    if (wants_packed(P) && ws_bytes >= pcg_bytes(P) + packed_rows(P, nullptr, nullptr)) {
        packed_rows(P, static_cast<char*>(solve_ws) + pcg_bytes(P), &rows);
        tma = make_step_maps(P, rows.h, rows.w, rows.pitch, B, tile, &maps);
        if (!tma) rows = PackedRows{};
    } else {
        tma = make_step_maps(P, h, w, P.nx, B, tile, &maps);
    }
    {
        LaunchScope ls(MPM_KERNEL_PCG_INIT, st);
        const auto init = rows.w ? k_pcg_init<K, true> : k_pcg_init<K, false>;
        init<<<ig.grid, ig.block, 0, st>>>(P, ig.zc, h, w, g, y, B.p[0], tol2, hdr, resid, red, rows);
    }
    const StencilGrid tg = tma ? tma_grid(P, tile) : sg;
    const bool want_resid = resid != nullptr || tol2 > 0.0;
    for (int j = 0; j < cg_iters; ++j) {
        const int rr = (want_resid || j == cg_iters - 1) ? 1 : 0;
        LaunchScope ls(MPM_KERNEL_PCG_STEP, st);
        const cudaError_t e = tma ? launch_step_tma(P, tg, maps, j, step_mode(j), rr, hdr, resid, red, so.overlap, st)
                                  : launch_step_plain<K>(P, sg, j, rr, h, w, B, hdr, resid, red, so.overlap, st);
        if (e != cudaSuccess) return e;
    }
    LaunchScope ls(MPM_KERNEL_PCG_FINAL, st);
    return launch_dependent(so.overlap, k_pcg_final<K>, dim3(voxel_grid(P.N)), dim3(kBlock), 0, st, P.N, B, delta, y_update,
                            hdr, report_rel, report_it);
}

cudaError_t tma_autotune(const DevProblem& P, void* solve_ws, WsHeader* hdr, Reduce red,
                         cudaStream_t st, int* best, float* ms)
{
    *best = -1;
    // Timed on zeroed operands carved from six of the solve workspace's vectors
    // so that no buffer the launch writes is also read: iteration 3 reads p_2,
    // p_1 and v_2 from vectors 0-2 and writes p_3 and v_3 to 4 and 5; H and w
    // alias the read-only vectors 0-3 (T N floats fit in 0-2 for K = 3, 4).
    const size_t vec = align256(sizeof(float4) * (size_t)P.N);
    char* c = static_cast<char*>(solve_ws);
    auto at = [&](int i) { return reinterpret_cast<float4*>(c + i * vec); };
    SolveBufs B;
    B.p[2] = at(0); B.p[1] = at(1); B.p[0] = at(4);
    B.v[0] = at(2); B.v[1] = at(5);
    B.x = B.z[0] = B.z[1] = at(3);       // not touched in iteration 3
    const float* h = reinterpret_cast<const float*>(at(0));
    const float* w = reinterpret_cast<const float*>(at(3));
    cudaError_t e;
    if ((e = cudaMemsetAsync(solve_ws, 0, solve_ws_bytes(P), st)) != cudaSuccess) return e;
    cudaEvent_t a, b;
    if ((e = cudaEventCreate(&a)) != cudaSuccess) return e;
    if ((e = cudaEventCreate(&b)) != cudaSuccess) {
        cudaEventDestroy(a);
        return e;
    }
    float best_ms = 0.0f;
    for (int t = 0; t < tma_tile_count(); ++t) {
        ms[t] = -1.0f;
        StepMaps m;
        if (!make_step_maps(P, h, w, P.nx, B, t, &m)) continue;
        const StencilGrid g = tma_grid(P, t);
        constexpr int reps = 5;
        for (int i = 0; i <= reps && e == cudaSuccess; ++i) {
            if (i == 1) e = cudaEventRecord(a, st);
            if (e == cudaSuccess) e = cudaMemsetAsync(hdr, 0, sizeof(WsHeader), st);
            if (e == cudaSuccess) e = launch_step_tma(P, g, m, 3, kModeStep, 0, hdr, nullptr, red, true, st);
        }
        if (e == cudaSuccess) e = cudaEventRecord(b, st);
        if (e == cudaSuccess) e = cudaEventSynchronize(b);
        float t_ms = 0.0f;
        if (e == cudaSuccess) e = cudaEventElapsedTime(&t_ms, a, b);
        if (e != cudaSuccess) break;
        ms[t] = t_ms / reps;
        if (*best < 0 || ms[t] < best_ms) {
            best_ms = ms[t];
            *best = t;
        }
    }
    cudaEventDestroy(a);
    cudaEventDestroy(b);
    if (e == cudaSuccess && *best >= 0) tma_tile_set(P, *best);
    return e;
}

// ------------------------------------------------- batched launches

SolveBufs solve_bufs(const DevProblem& P, void* solve_ws, size_t ws_bytes, Reduce red)
{
    return carve(P, solve_ws, ws_bytes, red);
}

template <int K, bool RUNS, typename IT>
static cudaError_t launch_jtv_batch_staged(int smem, const Batch<JtvArgs>& b, cudaStream_t st)
{
    const cudaError_t e = jtv_smem_opt_in<K, RUNS, IT>();
    if (e) return e;
    k_jtv_staged_batch<K, RUNS, IT><<<b.start[b.n], kJtvThreads, smem, st>>>(b, copy_wait_cycles(),
                                                                             copy_withhold());
    return cudaGetLastError();
}

template <int K, typename IT>
static cudaError_t launch_jtv_batch_k(bool staged, bool runs, int smem, const Batch<JtvArgs>& b,
                                      cudaStream_t st)
{
    if (staged)
        return runs ? launch_jtv_batch_staged<K, true, IT>(smem, b, st)
                    : launch_jtv_batch_staged<K, false, IT>(smem, b, st);
    k_jtv_batch<K, IT><<<b.start[b.n], dim3(kTileX, kTileY, 1), 0, st>>>(b);
    return cudaGetLastError();
}

cudaError_t launch_jtv_batch(int K, const JtvArgs* a, const double* share, int n, cudaStream_t st)
{
    // one kernel for the whole launch: runs of four if every subject has them,
    // staged if every subject is large enough for that form
    static thread_local Batch<JtvArgs> b;
    unsigned blocks[kBatchMax];
    JtvArgs args[kBatchMax];
    bool i32 = true, staged = true, runs = true;
    for (int i = 0; i < n; ++i) {
        i32 = i32 && index32(a[i].P);
        runs = runs && jtv_runs(a[i].P, a[i].y, a[i].w);
    }
    for (int i = 0; i < n; ++i) staged = staged && jtv_stages(a[i].P, runs) > 0;
    int smem = 0;
    for (int i = 0; i < n; ++i) {
        args[i] = a[i];
        const int stages = staged ? jtv_stages(a[i].P, runs) : 0;
        jtv_grid(a[i].P, stages, share[i], args[i]);
        blocks[i] = args[i].gx * args[i].gy * args[i].gz;
        smem = std::max(smem, jtv_smem(a[i].P, stages));
    }
    fill_batch(b, args, blocks, n);
    LaunchScope ls(MPM_KERNEL_JTV, st);
    if (K == 4)
        return i32 ? launch_jtv_batch_k<4, int>(staged, runs, smem, b, st)
                   : launch_jtv_batch_k<4, long long>(staged, runs, smem, b, st);
    return i32 ? launch_jtv_batch_k<3, int>(staged, runs, smem, b, st)
               : launch_jtv_batch_k<3, long long>(staged, runs, smem, b, st);
}

cudaError_t launch_pcg_init_batch(int K, const InitArgs* a, const unsigned* blocks, int n,
                                  cudaStream_t st)
{
    Batch<InitArgs> b;
    fill_batch(b, a, blocks, n);
    LaunchScope ls(MPM_KERNEL_PCG_INIT, st);
    const dim3 blk(kTileX, kTileY, 1);
    if (K == 4)
        k_pcg_init_batch<4><<<b.start[n], blk, 0, st>>>(b);
    else
        k_pcg_init_batch<3><<<b.start[n], blk, 0, st>>>(b);
    return cudaGetLastError();
}

cudaError_t launch_pcg_final_batch(int K, const FinalArgs* a, const unsigned* blocks, int n,
                                   cudaStream_t st)
{
    Batch<FinalArgs> b;
    fill_batch(b, a, blocks, n);
    LaunchScope ls(MPM_KERNEL_PCG_FINAL, st);
    if (K == 4)
        return launch_dependent(true, k_pcg_final_batch<4>, dim3(b.start[n]), dim3(kBlock), 0, st, b);
    return launch_dependent(true, k_pcg_final_batch<3>, dim3(b.start[n]), dim3(kBlock), 0, st, b);
}

cudaError_t launch_solve(const DevProblem& P, const SolveOpts& so, const float* h,
                         const float* w, const float* g, const float* y, float* delta,
                         float* y_update, double* resid, double* report_rel, int* report_it,
                         void* solve_ws, size_t ws_bytes, WsHeader* hdr, Reduce red, cudaStream_t st)
{
    if (so.mg_levels > 0)
        return launch_solve_mg(P, so, h, w, g, y, delta, y_update, resid, report_rel, report_it,
                               solve_ws, hdr, red, st);
    if (P.K == 4)
        return solve_k<4>(P, so, h, w, g, y, delta, y_update, resid, report_rel,
                          report_it, solve_ws, ws_bytes, hdr, red, st);
    return solve_k<3>(P, so, h, w, g, y, delta, y_update, resid, report_rel,
                      report_it, solve_ws, ws_bytes, hdr, red, st);
}

}  // namespace mpm

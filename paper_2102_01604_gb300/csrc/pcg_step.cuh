// pcg_step.cuh -- per-voxel arithmetic of the block-Jacobi PCG of the Newton
// system (H + L) delta = g + L y (Eq. 42, Sec. 2.6), shared by the TMA-staged
// iteration kernel (stencil_tma.cu) and the plain one (stencil_kernels.cu) so
// that both compute every voxel with the same operations in the same order.
//
// One kernel per PCG iteration.  The textbook recurrence keeps r and z = M^-1 r
// and needs two grid-wide reductions per iteration (p.q for alpha, r.z for
// beta).  Here the preconditioned residual is carried instead and updated as
//     z_{j+1} = z_j - alpha_j v_j,   v_j = M^-1 q_j,   q_j = (H + L) p_j,
// which is the same vector as M^-1 (r_j - alpha_j q_j) (M is linear), and the
// next r.z is expanded from quantities of iteration j alone:
//     r_{j+1}.z_{j+1} = r_j.z_j - 2 alpha_j q_j.z_j + alpha_j^2 q_j.v_j
// with r_j = M z_j formed per voxel (M symmetric, so r_j.v_j = z_j.q_j).  All
// four sums are reduced in the same launch as q_j, so alpha_j and beta_j are
// known when iteration j + 1 starts: it forms z_{j+1} and p_{j+1} = z_{j+1} +
// beta_j p_j for its tile and halo, applies the operator and writes v and p
// once.  |r_{j+1}|^2 is expanded the same way when the residual norm is
// wanted.  r.z is recomputed directly (z_j.M z_j) in every iteration, so the
// expansion spans one step and errors do not accumulate.
//
// z itself is not stored while the last two directions hold it,
//     z_j = p_j - beta_{j-1} p_{j-1},
// with the beta that formed p_j: an iteration reads p_j, p_{j-1} and v_j
// and writes p_{j+1} and v_{j+1}.  The iteration is bound by HBM: without z's
// store it moves 124 B per voxel (K = 4) instead of 140, and the x fold, whose
// two directions are both at hand, 16 B per iteration instead of 24.  The
// rounding of that z is 2^-24 |p_j|, of a stored one 2^-24 |z_j|.  On the
// Newton systems of a fit |p_j| is within a few |z_j| (1 to 3.3), but on stiff
// ones it reaches hundreds: at lambda = 1e5, 500 iterations, delta would end
// 1.5e-4 from the 64-bit solution instead of 1.2e-6.  So the scalars carry
//     (p_j.M p_j) / (z_j.M z_j) = 1 + beta_{j-1} (p_{j-1}.M p_{j-1}) / (z_{j-1}.M z_{j-1})
// (z_j.M p_{j-1} = 0), and an iteration above kStoreZ also stores its z_j, which
// the next one reads in place of p_{j-1}: 16 B per voxel more, and as much
// again in the folding iterations, whose p_{j-2} is then read for itself (from
// L2, where the producer has it fetched).  30 iterations at 176x240x256 with
// every z stored take 9.00 ms (9.18 without that fetch), 7.42 with none.  With
// 8^2 the errors are those of a z that is always stored (CPU restatement in
// float32, 20x16x12, delta after the last iteration):
//     lambda, iterations    z stored    never     above 4     8         16
//     10, 400               3.6e-7      3.7e-7    3.7e-7      3.7e-7    3.7e-7
//     1e3, 400              4.6e-7      2.1e-6    5.1e-7      5.1e-7    5.0e-7
//     1e5, 500              1.2e-6      1.5e-4    2.0e-6      1.9e-6    7.1e-7
//
// The preconditioner block M_n = H_n + diag(lambda_k d_n), d_n = sum of the
// six edge coefficients, is factorised in every iteration from H and the JTV
// weights (its float32 Cholesky factor is the same each time), so the solve
// stores no factor.
//
// The solve's own vectors (v, p, the accumulated x and z where stored) are stored voxel
// by voxel, four floats per voxel (K = 3 leaves the fourth zero), so one
// 16-byte access moves all maps of a voxel; H, w and the caller's arrays stay
// planar [component][N].
#pragma once

#include "device_common.cuh"

namespace mpm {

// Lower Cholesky factor of the K x K block, packed row by row
// (00, 10, 11, 20, 21, 22, 30, 31, 32, 33) with reciprocal diagonal.
__host__ __device__ constexpr int lo(int i, int j) { return i * (i + 1) / 2 + j; }

template <int K>
__device__ __forceinline__ bool cholesky_f32(const float (&M)[K][K], float (&L)[K * (K + 1) / 2])
{
    bool ok = true;
#pragma unroll
    for (int j = 0; j < K; ++j) {
        float s = M[j][j];
#pragma unroll
        for (int k = 0; k < j; ++k) s = fmaf(-L[lo(j, k)], L[lo(j, k)], s);
        if (!(s > 0.0f)) {
            ok = false;
            s = fmaxf(fabsf(M[j][j]), 1e-30f);
        }
        const float rj = rsqrtf(s);      // 1 / L_jj
        L[lo(j, j)] = rj;
#pragma unroll
        for (int i = j + 1; i < K; ++i) {
            float v = M[i][j];
#pragma unroll
            for (int k = 0; k < j; ++k) v = fmaf(-L[lo(i, k)], L[lo(j, k)], v);
            L[lo(i, j)] = v * rj;
        }
    }
    return ok;
}

// z = (L L')^-1 r with the packed factor.
template <int K>
__device__ __forceinline__ void chol_apply(const float (&L)[K * (K + 1) / 2], const float (&r)[K],
                                           float (&z)[K])
{
    float t[K];
#pragma unroll
    for (int i = 0; i < K; ++i) {
        float v = r[i];
#pragma unroll
        for (int k = 0; k < i; ++k) v = fmaf(-L[lo(i, k)], t[k], v);
        t[i] = v * L[lo(i, i)];
    }
#pragma unroll
    for (int i = K - 1; i >= 0; --i) {
        float v = t[i];
#pragma unroll
        for (int k = i + 1; k < K; ++k) v = fmaf(-L[lo(k, i)], z[k], v);
        z[i] = v * L[lo(i, i)];
    }
}

// Preconditioner block M = H + diag(lambda_k d) from the packed H.
template <int K>
__device__ __forceinline__ void precond_block(const DevProblem& P, const float (&hv)[K * (K + 1) / 2],
                                              float d, float (&M)[K][K])
{
#pragma unroll
    for (int a = 0; a < K; ++a)
#pragma unroll
        for (int b = a; b < K; ++b) M[a][b] = M[b][a] = hv[tri(K, a, b)];
#pragma unroll
    for (int a = 0; a < K; ++a) M[a][a] = fmaf(P.lambda[a], d, M[a][a]);
}

// Sum of the six edge coefficients (order x-, x+, y-, y+, z-, z+).
__device__ __forceinline__ float edge_sum(const float (&c)[6])
{
    return ((((c[0] + c[1]) + c[2]) + c[3]) + c[4]) + c[5];
}

// Largest (p.M p) / (z.M z) of an iteration that does not store z.
constexpr float kStoreZ = 64.0f;

// Per-solve workspace buffers: [N] float4 each (voxel-interleaved maps),
// 256-byte aligned.
struct SolveBufs {
    float4* v[2];    // v_j = M^-1 q_j in v[j & 1]
    float4* p[3];    // direction p_j in p[j % 3]
    float4* x;       // sum of the directions folded so far, alpha_i p_i
    float4* z[2];    // preconditioned residual z_j in z[j & 1], where it is stored
};

template <int K>
__device__ __forceinline__ void unpack4(const float4& a, float (&o)[K])
{
    o[0] = a.x;
    o[1] = a.y;
    o[2] = a.z;
    if constexpr (K > 3) o[3] = a.w;
}

template <int K>
__device__ __forceinline__ float4 pack4(const float (&o)[K])
{
    if constexpr (K > 3) return make_float4(o[0], o[1], o[2], o[3]);
    else return make_float4(o[0], o[1], o[2], 0.0f);
}

// What one iteration's launch does besides the common work.
enum : int {
    kModeFirst = 0,    // j = 0: p_0 = z_0 comes from the init kernel
    kModeSecond = 1,   // j = 1: z_0 = p_0, there is no p_{-1}
    kModeStep = 2,     // odd j > 1
    kModeFold = 3,     // j = 2: also x = alpha_0 p_0 + alpha_1 p_1
    kModeFoldX = 4     // even j > 2: also x += alpha_{j-2} p_{j-2} + alpha_{j-1} p_{j-1}
};

// Sums reduced by every iteration, in this order.
enum : int { kSumPQ, kSumZQ, kSumVQ, kSumZR, kSumRR, kSumRQ, kSumQQ, kStepSums };

// The four maps of a voxel as two pairs, for the paired float32 instructions
// (each lane rounds as its scalar form): the iteration's instruction issue is
// the bound next to HBM, and its per-map arithmetic pairs without moves.
struct Maps {
    float2 a, b;
    __device__ __forceinline__ Maps() {}
    __device__ __forceinline__ Maps(float2 x, float2 y) : a(x), b(y) {}
    __device__ __forceinline__ Maps(const float4& v) : a(make_float2(v.x, v.y)), b(make_float2(v.z, v.w)) {}
    __device__ __forceinline__ float operator[](int k) const
    {
        return k == 0 ? a.x : k == 1 ? a.y : k == 2 ? b.x : b.y;
    }
    __device__ __forceinline__ float4 vec() const { return make_float4(a.x, a.y, b.x, b.y); }
};

__device__ __forceinline__ float2 twice(float v) { return make_float2(v, v); }

// s v + w, and v - w.
__device__ __forceinline__ Maps axpy(float s, const Maps& v, const Maps& w)
{
    return Maps(__ffma2_rn(twice(s), v.a, w.a), __ffma2_rn(twice(s), v.b, w.b));
}
__device__ __forceinline__ Maps minus(const Maps& v, const Maps& w) { return axpy(-1.0f, w, v); }

// *at = v if `yes`, as one predicated store.  The tests for a stored z cost a
// solve of 176x240x256 0.3% this way (7.41 -> 7.43 ms; a 64^3 fit 10.05 -> 10.02;
// three maps, 136x141x109, 28 iterations 1.66 -> 1.68, 64^3 none),
// 0.8% with an if around the store (7.47), more with one branch around both
// forms of z (7.60) or a second copy of the march (7.42, but the 64^3 fit 10.38).
__device__ __forceinline__ void store_if(int yes, float4* at, const Maps& v)
{
    asm volatile("{\n\t.reg .pred q;\n\tsetp.ne.s32 q, %0, 0;\n\t@q st.global.v4.f32 [%1], {%2, %3, %4, %5};\n\t}"
                 ::"r"(yes), "l"(at), "f"(v.a.x), "f"(v.a.y), "f"(v.b.x), "f"(v.b.y)
                 : "memory");
}

// v = *at if `yes`, as one predicated load.
__device__ __forceinline__ void load_if(int yes, Maps& v, const float4* at)
{
    asm volatile("{\n\t.reg .pred q;\n\tsetp.ne.s32 q, %4, 0;\n\t@q ld.global.v4.f32 {%0, %1, %2, %3}, [%5];\n\t}"
                 : "+f"(v.a.x), "+f"(v.a.y), "+f"(v.b.x), "+f"(v.b.y)
                 : "r"(yes), "l"(at)
                 : "memory");
}

// sum_k v_k w_k (the padding of K = 3 is zero).
__device__ __forceinline__ float dot(const Maps& v, const Maps& w)
{
    const float2 s = __ffma2_rn(v.b, w.b, __fmul2_rn(v.a, w.a));
    return s.x + s.y;
}

// The scalars an iteration starts from: alpha_{j-1}, alpha_{j-2}, beta_{j-1}
// and beta_{j-2} (those that exist), whether z_{j-1} was stored and whether z_j is.
struct StepScalars {
    float alpha, alpha_prev, beta, beta_prev;
    int zin, zout;
};

__device__ __forceinline__ StepScalars step_start(const SolveScalars& sc)
{
    return StepScalars{(float)sc.alpha, (float)sc.alpha_prev, (float)sc.beta, (float)sc.beta_prev,
                       sc.zin, sc.zout};
}

// z_j and p_j of one point from p1 = p_{j-1}, v = v_{j-1} and pz = p_{j-2}, or
// z_{j-1} where that was stored (zin; j = 0: p1 is p_0 and v, pz are not read; j =
// 1: pz is not read).
template <int MODE>
__device__ __forceinline__ void step_point(const StepScalars& s, bool zin, const Maps& p1, const Maps& v,
                                           const Maps& pz, Maps& zj, Maps& pj)
{
    Maps z = p1;                                                          // z_{j-1}
    if (MODE >= kModeStep) z = zin ? pz : axpy(-s.beta_prev, pz, p1);
    zj = MODE == kModeFirst ? z : axpy(-s.alpha, v, z);
    pj = MODE == kModeFirst ? z : axpy(s.beta, p1, zj);
}

// x after folding in the two latest directions, in the order of two single
// updates: x + alpha_{j-2} p_{j-2}, then + alpha_{j-1} p_{j-1} (all four
// components; the padding of K = 3 stays zero).
__device__ __forceinline__ Maps fold_x(const Maps& x, const StepScalars& s, const Maps& p2, const Maps& p1)
{
    return axpy(s.alpha, p1, axpy(s.alpha_prev, p2, x));
}

// One voxel of iteration j: q = (H + L) p_j with the weighted 7-point stencil
//     (L p)_k = lambda_k sum_m c_m (p_k[n] - p_k[m]),  c_m = (w_n + w_m) / h^2
// (c_m = 0 for neighbours outside the volume, whose values nb then only need
// to be finite), v = M^-1 q, r = M z_j, and the voxel's terms added to part.
// nb(m) returns p_j at neighbour m (order x-, x+, y-, y+, z-, z+).
template <int K, class NB>
__device__ __forceinline__ void step_voxel(const DevProblem& P, const float (&c)[6], const Maps& zj,
                                           const Maps& pj, NB nb, const float (&hv)[K * (K + 1) / 2],
                                           bool resid, Maps& v, float (&part)[kStepSums])
{
    float M[K][K];
    precond_block<K>(P, hv, edge_sum(c), M);
    Maps s;
    {
        const Maps d = minus(pj, nb(0));
        s = Maps(__fmul2_rn(twice(c[0]), d.a), __fmul2_rn(twice(c[0]), d.b));
    }
#pragma unroll
    for (int m = 1; m < 6; ++m) s = axpy(c[m], minus(pj, nb(m)), s);
    float q[K];
#pragma unroll
    for (int a = 0; a < K; ++a) {
        float acc = P.lambda[a] * s[a];
#pragma unroll
        for (int b = 0; b < K; ++b) acc = fmaf(hv[a < b ? tri(K, a, b) : tri(K, b, a)], pj[b], acc);
        q[a] = acc;
    }
    float L[K * (K + 1) / 2], vk[K], r[K];
    cholesky_f32<K>(M, L);
    chol_apply<K>(L, q, vk);
#pragma unroll
    for (int a = 0; a < K; ++a) {
        float acc = M[a][0] * zj[0];
#pragma unroll
        for (int b = 1; b < K; ++b) acc = fmaf(M[a][b], zj[b], acc);
        r[a] = acc;
    }
    const Maps q4 = Maps(pack4<K>(q)), r4 = Maps(pack4<K>(r));
    v = Maps(pack4<K>(vk));
    part[kSumPQ] += dot(pj, q4);
    part[kSumZQ] += dot(zj, q4);
    part[kSumVQ] += dot(v, q4);
    part[kSumZR] += dot(zj, r4);
    if (resid) {
        part[kSumRR] += dot(r4, r4);
        part[kSumRQ] += dot(r4, q4);
        part[kSumQQ] += dot(q4, q4);
    }
}

// Float64 division in a serial chain: GB300's float64 operations have about a
// hundred cycles of latency each, and two IEEE divisions with their NaN tests
// made the one thread that derives the scalars take 4000 cycles (2 us of a
// 12 us iteration of a small volume).  recip: the float32 reciprocal and one
// Newton-Raphson step y <- y + y (1 - b y) (relative error about 2^-45; b
// outside float32's range divides); quot: a / b from it with one residual
// correction (about 2^-53).
__device__ __forceinline__ double recip(double b)
{
    if (!(b > 1e-30 && b < 1e30)) return 1.0 / b;
    const double y = (double)(1.0f / (float)b);
    return fma(y, fma(-b, y, 1.0), y);
}

__device__ __forceinline__ double quot(double a, double b, double y)
{
    const double q = a * y;
    return fma(fma(-b, q, a), y, q);
}

__device__ __forceinline__ bool is_nan(double v)
{
    return ((unsigned long long)__double_as_longlong(v) << 1) > 0xffe0000000000000ull;
}

// Scalars of iteration j from its reduced sums (the last block of the launch):
// alpha_j = r_j.z_j / p_j.q_j, the expanded r_{j+1}.z_{j+1} and |r_{j+1}|^2,
// beta_j and the stopping tests.  A breakdown (p.q or r.z not positive, or a
// NaN) stops the solve without a step.
__device__ __forceinline__ void step_scalars(const double (&s)[kStepSums], int j, bool resid_sums,
                                             WsHeader* hdr, double* resid)
{
    SolveScalars& sc = hdr->sc;
    const double alpha_old = sc.alpha, beta_old = sc.beta;
    const float pz_old = sc.pz;
    const int zout_old = sc.zout;
    bool bad = false;
#pragma unroll
    for (int i = 0; i < kStepSums; ++i) bad |= is_nan(s[i]);
    if (bad) atomicOr(&hdr->status, kStatusNaN);
    const double pq = s[kSumPQ], rz = s[kSumZR];
    if (bad || !(pq > 0.0) || !(rz > 0.0)) {
        sc.done = 1;                       // no further step; the alphas keep their values
        return;
    }
    const double ipq = recip(pq), irz = recip(rz);
    const double alpha = quot(rz, pq, ipq);
    const double rz_next = fma(alpha, fma(alpha, s[kSumVQ], -2.0 * s[kSumZQ]), rz);
    sc.alpha_prev = alpha_old;
    sc.alpha = alpha;
    sc.beta_prev = beta_old;
    sc.beta = quot(rz_next, rz, irz);
    sc.rz = rz_next;
    sc.pz = fmaf((float)sc.beta, pz_old, 1.0f);
    sc.zin = zout_old;
    sc.zout = !(sc.pz <= kStoreZ);
    sc.it = j + 1;
    if (resid_sums) {
        const double rr = s[kSumRR] - 2.0 * alpha * s[kSumRQ] + alpha * alpha * s[kSumQQ];
        sc.rr = rr > 0.0 ? rr : 0.0;
        if (resid) resid[j + 1] = sqrt(sc.rr);
        if (sc.tol2 > 0.0 && sc.rr <= sc.tol2 * sc.rr0) sc.done = 1;
    }
    if (!(rz_next > 0.0)) sc.done = 1;
}

}  // namespace mpm

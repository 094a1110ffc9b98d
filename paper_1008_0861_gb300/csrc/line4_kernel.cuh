// line4_kernel.cuh -- warp-autonomous update of contiguous lines (Eq. xup on
// rows; Eq. yup on the column-major copy T*).
//
// Same linear algebra as line_sweep_kernel and line2_kernel (delta form,
// bottom-up segment elimination, PCR of the segment-end unknowns, forward
// recovery; see sweep_kernels.cuh).  What differs is the organisation:
//  - a line belongs to a team of P <= 32 lanes of one warp (32/P lines per
//    warp); no phase waits for another warp except the final transposed
//    store, so warps of a block drift apart and overlap each other's loads
//    and arithmetic;
//  - face fluxes are computed with coalesced 16-byte loads (lane t takes
//    chunks t, t+P, ..., the next round in flight during this one), the
//    limited transverse difference as Eq. vanLeer nests it: once per cell
//    v = L(T_after - T, T - T_before), then once per face L(v_p, v_{p+1}),
//    so every cell's inner value serves both of its faces;
//  - F and lam*g go to the warp's shared area, where each lane then walks
//    its own segment bottom-up (a row is eliminated as soon as the flux of
//    the face below it is known), storing (rho, alpha, gamma) in place; the
//    segment-end system is solved with warp shuffles; recovery writes delta
//    in place;
//  - T_new = T_old + delta leaves either line-major (coalesced) or,
//    staged in the same area, position-major (`nlines` wide) with the
//    lines of a block packed into 16-byte stores: the x-update writes T*
//    column-major and the y-update writes T^{n+1} back row-major.
// Shared arrays hold whole 16-byte chunks at c ^ ((c >> s) & 7) within
// complete groups of 8, so that both the chunk-parallel phases and the
// segment walks touch distinct bank groups; the host picks s per line
// (Line2Job::swz, line4_swizzle) for the segment lengths it has, the default
// being log2 of the chunks per segment.
// FP32 reciprocals use the hardware approximation (rcp.approx.ftz.f32,
// within 1 ulp); FP64 quotients are rounded but for rare neighbours (dquot).
// Each block first asks for its input rows to be brought into L2 with bulk
// prefetches.
//
// D3: the lines of a three-dimensional grid (Section 2.1).  The face flux
// gains a second limited transverse term, mu2 * e2 * DeltaT-bar along the
// second transverse axis, from the lines -+ na away; everything after the
// flux is unchanged.  With lines along x indexed (z, y), the transposed
// output is indexed (x, z, y): the next update's lines run along y, its
// transverse axes are z then x, and its output (y, x, z) serves the
// z-update, whose output is (z, y, x) again.
#pragma once
#include "line2_kernel.cuh"

namespace aniso {

// Raw 16 bytes of T / N coefficients, converted only when used (so that a
// prefetch does not wait on its own load).
__device__ __forceinline__ float4 ld_raw(const float *p) { return __ldg(reinterpret_cast<const float4 *>(p)); }
__device__ __forceinline__ double2 ld_raw(const double *p) { return __ldg(reinterpret_cast<const double2 *>(p)); }
__device__ __forceinline__ uint2 ld_raw(const __half *p) { return __ldg(reinterpret_cast<const uint2 *>(p)); }
__device__ __forceinline__ void unpack_raw(const float4 &v, float *o) { V16<float>::unpack(v, o); }
__device__ __forceinline__ void unpack_raw(const double2 &v, double *o) { V16<double>::unpack(v, o); }
__device__ __forceinline__ void unpack_raw(const uint2 &v, float *o)
{
    const float2 a = __half22float2(*reinterpret_cast<const __half2 *>(&v.x));
    const float2 b = __half22float2(*reinterpret_cast<const __half2 *>(&v.y));
    o[0] = a.x;
    o[1] = a.y;
    o[2] = b.x;
    o[3] = b.y;
}

// The same 16 bytes of T / N coefficients element by element, from any
// address: elements a, b, c, d of a row.
__device__ __forceinline__ float4 ld_elem(const float *r, int a, int b, int c, int d)
{
    return make_float4(r[a], r[b], r[c], r[d]);
}
__device__ __forceinline__ uint2 ld_elem(const __half *r, int a, int b, int c, int d)
{
    const unsigned short *u = reinterpret_cast<const unsigned short *>(r);
    const unsigned x = u[a], y = u[b], z = u[c], w = u[d];
    return make_uint2(x | (y << 16), z | (w << 16));
}
__device__ __forceinline__ double2 ld_elem(const double *r, int a, int b, int, int) { return make_double2(r[a], r[b]); }
// Chunk c of a row of n cells; elements from n on are taken at p1.
template <int N, typename E> __device__ __forceinline__ auto ld_ragged(const E *row, int c, int n, int p1)
{
    const int p = c * N;
    if (p + N <= n) return ld_elem(row + p, 0, 1, 2, 3);
    auto at = [n, p1](int k) { return k < n ? k : p1; };
    return ld_elem(row, at(p), at(p + 1), at(p + 2), at(p + 3));
}

// Bulk prefetch of a byte range into L2 (no destination, no completion).
__device__ __forceinline__ void l2_prefetch(const void *p, size_t bytes)
{
    if (bytes == 0 || bytes > 0xffffffffu || ((reinterpret_cast<uintptr_t>(p) | bytes) & 15)) return;
    asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(p), "r"((unsigned)bytes) : "memory");
}

// Host: a launch of kern(a) in a.chained mode or plainly, with any amount of shared memory.
template <typename K>
static cudaError_t launch_line_kernel(K kern, const Line2Args &a, int nblocks, int nthreads, size_t smem, cudaStream_t s,
                                      int cluster = 0)
{
    const cudaError_t e = allow_smem(kern, smem);
    if (e != cudaSuccess) return e;
    return launch_kernel(kern, dim3((unsigned)nblocks), dim3((unsigned)nthreads), smem, s, a.chained != 0, cluster, a);
}

__device__ __forceinline__ float frcp_approx(float x)
{
    float r;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
}
template <typename R> struct Fast;
template <> struct Fast<float> {
    static __device__ __forceinline__ float rcp(float x) { return frcp_approx(x); }
    static __device__ __forceinline__ float div(float a, float b) { return a * frcp_approx(b); }
};
// FP64 vector instructions are what an FP64 update waits for (2 lanes a clock
// and SM), and divisions were most of its 98 a cell.  1/x here is one
// third-order Newton step (Chebyshev's method) from the hardware's 20-bit
// estimate: with e = 1 - x y, y (1 + e + e^2) = (1 - e^3) / x, three fused
// operations, within 1 ulp.  x and 1/x must be normal: |x| from 2^-1022 to 2^1022
// (an estimate that underflows gives 0, an infinite x NaN).
__device__ __forceinline__ double drcp_approx(double x)
{
    double y;
    asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(x));
    const double e = __fma_rn(-x, y, 1.0);
    return __fma_rn(y, __fma_rn(e, e, e), y);
}
// Quotient and reciprocal from such a y by one step with the exact remainder
// (Markstein, IBM J. Res. Dev. 34, 1990).  y is not the rounded 1/b that his proof
// of correct rounding asks for, but within 1 ulp of it, and the value before the
// last rounding within 2^-51 ulp of the quotient: the result is the rounded one
// unless the quotient lies that close to the middle of two numbers (1/x of an
// x = 2^k (2 - 2^-52) does), and the other neighbour then.  Quotient and
// remainder must be normal numbers.
__device__ __forceinline__ double dquot(double a, double b, double y)
{
    const double q = a * y;
    return __fma_rn(__fma_rn(-b, q, a), y, q);
}
__device__ __forceinline__ double drcp(double x)
{
    const double y = drcp_approx(x);
    return __fma_rn(__fma_rn(-x, y, 1.0), y, y);
}
template <> struct Fast<double> {
    static __device__ __forceinline__ double rcp(double x) { return drcp(x); }
    static __device__ __forceinline__ double div(double a, double b) { return a / b; }
};

// One level of the nested limiter (Eq. vanLeer: L(a,b) = 2ab/(a+b) when a, b
// share a strict sign, else 0; minmod / MC as in lim2; the arithmetic mean
// for LIM_ARITH, whose nesting gives the mean of the four differences).
template <typename R> __device__ __forceinline__ R lim_level(int lim, R a, R b)
{
    if (lim == LIM_ARITH) return R(0.5) * (a + b);
    return lim2<R>(lim, a, b);
}
// van Leer in FP32: a positive product is the strict-sign test (a + b is then
// nonzero); one approximate reciprocal.
__device__ __forceinline__ float vl_level(float a, float b)
{
    // (spelled out: a b + p could be fused, and must round alike in all forms)
    const float p = __fmul_rn(a, b);
    const float r = __fmul_rn(__fadd_rn(p, p), frcp_approx(__fadd_rn(a, b)));
    return p > 0.f ? r : 0.f;
}
template <typename R, bool VL> __device__ __forceinline__ R level(int lim, R a, R b)
{
    return lim_level<R>(lim, a, b);
}
template <> __device__ __forceinline__ float level<float, true>(int, float a, float b) { return vl_level(a, b); }

// The two levels of the nested limiter as one per cell (inner) and one per
// face (outer); outer's result times SCALE is L(L(a,b), L(c,d)).
template <typename R, bool VL, bool HARMONIC = false> struct Limit {
    static constexpr int SCALE = 1;
    static __device__ __forceinline__ R inner(int lim, R a, R b) { return level<R, VL>(lim, a, b); }
    static __device__ __forceinline__ R outer(int lim, R v, R w) { return level<R, VL>(lim, v, w); }
};
// FP64 van Leer.  A product in [2^-960, 2^1020) leaves quotient and remainder
// normal; others are told from the high word, off the FP64 pipe.
__device__ __forceinline__ bool vl_plain(double p) { return (unsigned)(__double2hiint(p) - 0x03f00000) < 0x7bc00000u; }
// Neither factor of a product p outside that range is 0, and p is not negative.
__device__ __forceinline__ bool vl_edge_of(double p, double a, double b)
{
    const int za = (__double2hiint(a) << 1) | __double2loint(a), zb = (__double2hiint(b) << 1) | __double2loint(b);
    return __double2hiint(p) >= 0 && za != 0 && zb != 0;
}
// Half of a level for such a product: as lim2 forms it.
static __device__ __noinline__ double vl_edge(double a, double b)
{
    return 0.5 * lim2<double>(LIM_VANLEER, a, b);
}
// The nest as written: a cell keeps ab / (a + b), half of its level, a face
// forms the same quotient of two cells', a quarter of the nest (powers of two:
// the bits of the nest of 2ab / (a + b)).  A run amplifies the last bit (the ring
// at 1000 times the limit by 1e6 in a hundred steps), which is why the quotients
// keep their rounding.
template <> struct Limit<double, true, false> {
    static constexpr int SCALE = 4;
    static __device__ __forceinline__ double inner(int, double a, double b)
    {
        const double p = a * b, s = a + b;
        const double q = dquot(p, s, drcp_approx(s));
        if (vl_plain(p)) return q;
        return vl_edge_of(p, a, b) ? vl_edge(a, b) : 0.0;
    }
    static __device__ __forceinline__ double outer(int, double v, double w)
    {
        const double p = v * w, s = v + w;
        const double q = dquot(p, s, drcp_approx(s));
        if (vl_plain(p)) return q;
        return vl_edge_of(p, v, w) ? 0.5 * vl_edge(2.0 * v, 2.0 * w) : 0.0;
    }
};
// By sums of reciprocals (the long lines, whose segments are others than they
// were): L is the harmonic mean, so the nest is 4 / (1/a + 1/b + 1/c + 1/d)
// where all four share a sign.  A cell keeps w = 1/a + 1/b = (a + b) / (a b) (0
// where the signs differ or the level is next to 0, NaN where it leaves the
// range), a face takes 1 / (w_p + w_{p+1}): 12 operations a cell instead of 18.
template <> struct Limit<double, true, true> {
    static constexpr int SCALE = 4;
    static __device__ __noinline__ double edge(double a, double b)
    {
        const double h = vl_edge(a, b), m = fabs(h);
        if (m < 0x1p-1000) return 0.0;
        return m < INFINITY ? 1.0 / h : copysign(__longlong_as_double(0x7ff8000000000000ll), a);
    }
    static __device__ __forceinline__ double inner(int, double a, double b)
    {
        const double p = a * b, w = (a + b) * drcp_approx(p);
        if (vl_plain(p)) return w;
        return vl_edge_of(p, a, b) ? edge(a, b) : 0.0;
    }
    // (2 / v and 2 / w are the cells' levels)
    static __device__ __noinline__ double outer_edge(double v, double w)
    {
        return fabs(v + w) < INFINITY ? 0.25 * lim2<double>(LIM_VANLEER, 2.0 / v, 2.0 / w) : v + w;
    }
    static __device__ __forceinline__ double outer(int, double v, double w)
    {
        const int hv = __double2hiint(v), hw = __double2hiint(w);
        const double r = drcp_approx(v + w);
        if (hv == 0 || hw == 0 || (hv ^ hw) < 0) return 0.0;
        // levels whose product is under 2^-950 (or NaN): as lim2 rounds it
        const unsigned e = (unsigned)(hv & 0x7fffffff) + (unsigned)(hw & 0x7fffffff);
        return e < 0xbba00000u ? r : outer_edge(v, w);
    }
};

// Which product of a flux is fused with the sum is spelled out, so that every
// form of the kernel rounds alike (a batch equals its grids one by one where
// their segments are the same: always in FP32, with ANISO_OPT_SEGMENT in FP64).
__device__ __forceinline__ float mul_rn(float a, float b) { return __fmul_rn(a, b); }
__device__ __forceinline__ double mul_rn(double a, double b) { return __dmul_rn(a, b); }
__device__ __forceinline__ float fma_rn(float a, float b, float c) { return __fmaf_rn(a, b, c); }
__device__ __forceinline__ double fma_rn(double a, double b, double c) { return __fma_rn(a, b, c); }

// NaN or infinity (the exponent bits, off the FP64 pipe).
__device__ __forceinline__ bool non_finite(float v) { return !(fabsf(v) < INFINITY); }
__device__ __forceinline__ bool non_finite(double v) { return (__double2hiint(v) & 0x7ff00000) == 0x7ff00000; }

// p + 0 v: p = 0 stays 0 while every v is finite and is NaN from the first that is
// not.  FP32: one test a lane at the end instead of one a chunk on its sum, which
// can leave the range where its values do not.
__device__ __forceinline__ float finite_probe(float p, float v) { return __fmaf_rn(v, 0.f, p); }

// PCR over a team of P <= 32 lanes (width-P shuffles), as pcr_warp.  Each lane
// takes the reciprocal of its own diagonal once and hands that on, instead of
// dividing by both neighbours' diagonals (the quotients' bits are kept).
__device__ __forceinline__ float pcr_ratio(float a, float, float y) { return a * y; }
__device__ __forceinline__ double pcr_ratio(double a, double b, double y) { return dquot(a, b, y); }
__device__ __forceinline__ float pcr_recip(float x) { return frcp_approx(x); }
__device__ __forceinline__ double pcr_recip(double x) { return drcp_approx(x); }
template <typename R> __device__ __forceinline__ R pcr_team(Reduced<R> q, int t, int P)
{
    const unsigned full = 0xffffffffu;
    for (int h = 1; h < P; h <<= 1) {
        const int tm = (t - h) & (P - 1), tp = (t + h) & (P - 1);
        const R iD = pcr_recip(q.D);
        R Dm = R(0), Dp = R(0);
        if constexpr (sizeof(R) == 8) {  // the remainders' divisors
            Dm = __shfl_sync(full, q.D, tm, P);
            Dp = __shfl_sync(full, q.D, tp, P);
        }
        const R Lm = __shfl_sync(full, q.L, tm, P), iDm = __shfl_sync(full, iD, tm, P);
        const R Um = __shfl_sync(full, q.U, tm, P), Rm = __shfl_sync(full, q.Rr, tm, P);
        const R Lp = __shfl_sync(full, q.L, tp, P), iDp = __shfl_sync(full, iD, tp, P);
        const R Up = __shfl_sync(full, q.U, tp, P), Rp = __shfl_sync(full, q.Rr, tp, P);
        const R k1 = pcr_ratio(q.L, Dm, iDm), k2 = pcr_ratio(q.U, Dp, iDp);
        q.D = q.D - k1 * Um - k2 * Lp;
        q.Rr = q.Rr - k1 * Rm - k2 * Rp;
        q.L = -k1 * Lm;
        q.U = -k2 * Up;
    }
    const R D = q.L + q.D + q.U;
    return pcr_ratio(q.Rr, D, pcr_recip(D));
}

// Bottom-up elimination of a segment's rows s .. e-1 into maps delta_k = rho -
// alp delta_{k-1} - gam X (X = delta_e) and their composite delta_{e-1} = qp +
// qq delta_{s-1} + qw X, which row e needs.
template <typename R, bool SYMMETRIC = false> struct Segment {
    R rho = R(0), alp = R(0), gam = R(-1);  // map of the row below: first the virtual row e
    R qp = R(0), qq = R(1), qw = R(0);
    // row k: -lgkm d_{k-1} + (1 + lgkm + lgk) d_k - lgk d_{k+1} = Fk - Fkm
    __device__ __forceinline__ void elim(R Fk, R Fkm, R lgk, R lgkm, R &ro, R &ao, R &go)
    {
        const R inv = Fast<R>::rcp((R(1) + lgkm + lgk) + lgk * alp);
        const R al = -lgkm * inv, ga = lgk * gam * inv, rh = ((Fk - Fkm) + lgk * rho) * inv;
        ro = rh;
        ao = al;
        go = ga;
        qp = qp + qq * rh;
        qw = qw - qq * ga;
        qq = -qq * al;
        rho = rh;
        alp = al;
        gam = ga;
    }
    // The equation of X in X_{t-1}, X, X_{t+1}: row e (-lgem, 1 + lgem + lge,
    // -lge; right-hand side re) with delta_{e-1} and the next segment's first
    // row (rho_n, alp_n, gam_n) substituted.
    __device__ __forceinline__ Reduced<R> reduced(R lgem, R lge, R re, R, R rho_n, R alp_n, R gam_n) const
    {
        return make_reduced<R>(-lgem, R(1) + lgem + lge, -lge, re, qp, qq, qw, rho_n, alp_n, gam_n);
    }
};
// SYMMETRIC (FP64, the long lines) carries less: the line matrix is symmetric
// (-lg_k on both sides of the diagonal), so the product of the alphas is that
// of the gammas times lg_k / lg_{e-1}, and row e sees the composite only times
// lg_{e-1}.  With w_k = lg_k gam_{k+1} (a factor of gam_k in any case),
// lg_{e-1} qp is the sum of -w_k rho_k, lg_{e-1} qw that of w_k gam_k, and
// lg_{e-1} qq is -gam_s lg_{s-1}: 14 FP64 operations a row instead of 17, and
// no quotient by an lg that may be 0.
template <> struct Segment<double, true> {
    double rho = 0.0, alp = 0.0, gam = -1.0;
    double A = 0.0, B = 0.0;  // lg_{e-1} qp, lg_{e-1} qw
    __device__ __forceinline__ void elim(double Fk, double Fkm, double lgk, double lgkm, double &ro, double &ao,
                                         double &go)
    {
        const double inv = drcp_approx((1.0 + lgkm + lgk) + lgk * alp);
        const double w = lgk * gam;
        rho = ((Fk - Fkm) + lgk * rho) * inv;
        alp = -lgkm * inv;
        gam = w * inv;
        A -= w * rho;
        B += w * gam;
        ro = rho;
        ao = alp;
        go = gam;
    }
    // lgs = lg_{s-1}, the face below the segment
    __device__ __forceinline__ Reduced<double> reduced(double lgem, double lge, double re, double lgs, double rho_n,
                                                       double alp_n, double gam_n) const
    {
        Reduced<double> q;
        q.L = gam * lgs;
        q.D = (1.0 + lgem + lge) - B + lge * alp_n;
        q.U = lge * gam_n;
        q.Rr = re + A + lge * rho_n;
        return q;
    }
};

// Register budgets.  The FP32 2-D form asks for four resident 256-thread
// blocks' worth of registers per SM (at most 64 per thread, no spills): lines
// short enough to need little shared memory then keep up to eight 128-thread
// blocks per SM instead of five (+7 % on the uneven batch, whose launches are
// split by occupancy).  The FP32 3-D form asks for three (80 registers
// instead of 112, a few spilled values, +3 %).  FP64 keeps two: it would
// spill more than it gains.
// NL: temperature-dependent diffusivity (Section 3.3): every face's
// coefficients (normal and transverse) are scaled by the harmonic mean of
// chi(T) = (max(T,0)/t_ref)^alpha over the face's two cells, from this
// update's input T.
template <typename R> __device__ __forceinline__ R chi_pow(R x, R a);
template <> __device__ __forceinline__ float chi_pow<float>(float x, float a) { return __powf(x, a); }
template <> __device__ __forceinline__ double chi_pow<double>(double x, double a) { return pow(x, a); }
template <typename R> __device__ __forceinline__ R face_harmonic(R a, R b)
{
    return (a > R(0) && b > R(0)) ? R(2) * a * Fast<R>::div(b, a + b) : R(0);
}

// Tensor memory (TMEM) as per-thread scratch.  A block of four warps
// allocates TM_COLS columns; warp w owns TMEM lanes 32 (w % 4) .. + 31, one per
// thread, so each thread has TM_COLS private 32-bit words.  The 32x32b shape
// moves four consecutive columns of the thread's own lane per instruction
// (warp-wide, aligned).
constexpr unsigned TM_COLS = 64;
__device__ __forceinline__ void tm_alloc(unsigned *s_dst, unsigned cols = TM_COLS)
{
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                     (unsigned)__cvta_generic_to_shared(s_dst)),
                 "r"(cols)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
}
__device__ __forceinline__ void tm_dealloc(unsigned base, unsigned cols = TM_COLS)
{
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(base), "r"(cols) : "memory");
}
__device__ __forceinline__ void tm_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tm_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tm_st4(unsigned taddr, float a, float b, float c, float d)
{
    asm volatile("tcgen05.st.sync.aligned.32x32b.x4.b32 [%0], {%1, %2, %3, %4};" ::"r"(taddr), "r"(__float_as_uint(a)),
                 "r"(__float_as_uint(b)), "r"(__float_as_uint(c)), "r"(__float_as_uint(d))
                 : "memory");
}
// (the load and its wait in one statement: the registers are defined on exit)
__device__ __forceinline__ void tm_ld4(unsigned taddr, float *o)
{
    unsigned r0, r1, r2, r3;
    asm volatile(
        "{\n\ttcgen05.ld.sync.aligned.32x32b.x4.b32 {%0, %1, %2, %3}, [%4];\n\t"
        "tcgen05.wait::ld.sync.aligned;\n\t}"
        : "=r"(r0), "=r"(r1), "=r"(r2), "=r"(r3)
        : "r"(taddr)
        : "memory");
    o[0] = __uint_as_float(r0);
    o[1] = __uint_as_float(r1);
    o[2] = __uint_as_float(r2);
    o[3] = __uint_as_float(r3);
}
__device__ __forceinline__ void tm_wait_st() { asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory"); }

// RAG: lines of any length and arrays of any alignment.  The line's last
// chunk holds its last nv = 1 .. N cells; loads and line-major stores go element
// by element (the four elements of a chunk share their sectors, so the extra
// instructions are most of the cost); an element past the line reads the cell
// after it (the wrap or the mirrored ghost), which the last face needs.  The
// last segment ends at position nv - 1 of its last chunk.  A line's solve is
// the same as with whole chunks.
// VC: the chunk rounds V of the launch's lines (their longest segment) as a
// constant, 0 = from the job.  The loops over rounds and segments are then
// unrolled: no counters, and nothing moved from one chunk's registers to the
// next's.
// COH: the coefficients by plain loads (Line2Args::fresh; RAG's always are).
// IMPL: a purely implicit update (no transverse term, mu = mu2 = 0: the second
// half-update of each axis in the 4-step scheme); neighbouring lines and
// transverse coefficients are then neither loaded nor limited.
// TM (FP32, 2-D, four-warp blocks, at most 8 chunks a lane): each lane's
// gamma lives in its TMEM lane instead of shared memory, so the line state in
// shared memory is 8 bytes a cell instead of 12 and more blocks fit an SM; the
// lane's chunks of T_old wait there too, from the flux phase to phase C
// (4 V + 4 V columns of the block's 32 or 64).
template <typename R, typename C, bool VL, bool D3 = false, bool NL = false, bool IMPL = false, bool TM = false,
          int RING = 1, bool RAG = false, int VC = 0, bool COH = false>
__global__ void __launch_bounds__(256, sizeof(R) == 4 && RING == 1 ? (D3 ? 3 : 4) : 2) line4_kernel(Line2Args args)
{
    static_assert(!TM || (sizeof(R) == 4 && !D3), "TMEM line state: FP32 2-D only");
    static_assert(!RAG || (!D3 && !NL && !IMPL && !TM), "ragged lines: the plain 2-D update only");
    typedef typename V16<R>::T VT;
    constexpr int N = V16<R>::N;
    constexpr int LOGN = N == 4 ? 2 : 1;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    __shared__ Line2Job J;
    if (args.jobs) {  // the block's job, copied by warp 0's lanes a word each
        constexpr int W8 = (int)(sizeof(Line2Job) / 8);
        static_assert(sizeof(Line2Job) % 8 == 0 && W8 <= 32, "job copy: one 8-byte word a lane");
        if (threadIdx.x < W8) {
            const int k = args.block_job ? args.block_job[blockIdx.x] : find_job(args.jobs, args.njobs);
            reinterpret_cast<unsigned long long *>(&J)[threadIdx.x] =
                reinterpret_cast<const unsigned long long *>(args.jobs + k)[threadIdx.x];
        }
    } else if (threadIdx.x == 0) {
        J = args.one;
    }
    __syncthreads();

    const int lim = args.limiter;
    const int P = J.team, n = J.n, m = RAG ? (n + N - 1) / N : n / N, nl = J.nlines, LPB = J.lines_per_block;
    const int nv = RAG ? n - (m - 1) * N : N;  // cells of the last chunk
    const int logP = __ffs(P) - 1;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int logL = 5 - logP;  // 32 / P lines per warp
    const int q = lane >> logP, t = lane & (P - 1);
    const int line0 = (blockIdx.x - J.block0) * LPB;
    const int line = line0 + (warp << logL) + q;
    const bool active = line < nl;
    const int lc = active ? line : nl - 1;
    int lu = lc + 1, ld = lc - 1;
    if (lu >= nl) lu = J.per_cross ? 0 : nl - 1;  // mirrored ghost line
    if (ld < 0) ld = J.per_cross ? nl - 1 : 0;
    int lbu = lc, lbd = lc;  // neighbours along the second transverse axis (D3)
    if constexpr (D3) {
        const int na = J.na, nb = nl / na, ka = lc % na, kb = lc / na;
        ld = ka > 0 ? lc - 1 : (J.per_cross ? lc + na - 1 : lc);
        lu = ka < na - 1 ? lc + 1 : (J.per_cross ? lc - (na - 1) : lc);
        lbd = kb > 0 ? lc - na : (J.per_cross ? lc + (nb - 1) * na : lc);
        lbu = kb < nb - 1 ? lc + na : (J.per_cross ? lc - (nb - 1) * na : lc);
    }
    const R *Tin = static_cast<const R *>(J.Tin);
    const R *rc = Tin + (size_t)lc * n, *ru = Tin + (size_t)lu * n, *rd = Tin + (size_t)ld * n;
    const R *rbu = Tin + (size_t)lbu * n, *rbd = Tin + (size_t)lbd * n;
    const C *G = static_cast<const C *>(J.g) + (size_t)lc * n;
    const C *E = static_cast<const C *>(J.e) + (size_t)lc * n;
    const C *E2 = D3 ? static_cast<const C *>(J.e2) + (size_t)lc * n : E;
    typedef Limit<R, VL> LM;
    const R lam = (R)J.lam, mu = R(LM::SCALE) * (R)J.mu, mu2 = R(LM::SCALE) * (R)J.mu2;
    const R chi_a = (R)J.chi_alpha, chi_it = (R)J.chi_itref;
    auto chi_of = [chi_a, chi_it](R T_) { return T_ > R(0) ? chi_pow<R>(T_ * chi_it, chi_a) : R(0); };
    const unsigned full = 0xffffffffu;

    // (what came before is the kernel's own arguments and indices; batched
    // launches, the only ones in the tensor-memory form, are never chained)
    if (!TM && !args.jobs) chain_wait();
    if constexpr (!TM) {
        after_wait(G);
        after_wait(E);
        if constexpr (D3) after_wait(E2);
    }

    // The block's input rows (its lines and the two neighbouring lines of T,
    // its coefficient rows) start streaming into L2 at once, so that the
    // warps' loads below find them there.  A hint only: issued when the
    // range is 16-byte aligned.
    if (threadIdx.x == 0) {
        const int f0 = line0 > 0 && !IMPL ? line0 - 1 : line0, f1 = min(line0 + LPB + (IMPL ? 0 : 1), nl),
                  g1 = min(line0 + LPB, nl);
        l2_prefetch(Tin + (size_t)f0 * n, (size_t)(f1 - f0) * n * sizeof(R));
        l2_prefetch(static_cast<const C *>(J.g) + (size_t)line0 * n, (size_t)(g1 - line0) * n * sizeof(C));
        if constexpr (!IMPL)
            l2_prefetch(static_cast<const C *>(J.e) + (size_t)line0 * n, (size_t)(g1 - line0) * n * sizeof(C));
        if constexpr (D3 && !IMPL) {
            l2_prefetch(static_cast<const C *>(J.e2) + (size_t)line0 * n, (size_t)(g1 - line0) * n * sizeof(C));
            // the block's neighbours along the second transverse axis, where not wrapped
            if (line0 >= J.na) l2_prefetch(Tin + (size_t)(line0 - J.na) * n, (size_t)(g1 - line0) * n * sizeof(R));
            if (g1 + J.na <= nl) l2_prefetch(Tin + (size_t)(line0 + J.na) * n, (size_t)(g1 - line0) * n * sizeof(R));
        }
    }

    // segment of lane t: chunks [c_lo, c_lo + Ut); the first rr lanes one more
    const int U = m >> logP, rr = m & (P - 1);
    const int Ut = U + (t < rr ? 1 : 0);
    const int c_lo = t * U + (t < rr ? t : rr), ce = c_lo + Ut - 1;
    const int V = VC > 0 ? VC : U + (rr ? 1 : 0);  // chunk rounds of the coalesced phases
    // (the tensor-memory form by fours: unrolled whole it spilled at 64 registers)
    constexpr int UNR = VC > 0 ? (TM ? 4 : VC) : 1;
    const int WA = m << logL;        // chunks per array in one warp's area
    const int mfull = m & ~7, logU = 31 - __clz(U);
    constexpr int NARR = TM ? 2 : 3;  // shared arrays per warp area
    const int AS = NARR * WA + (N == 4 ? line4_area_pad(P, NARR, m) : 0);  // chunks per warp area
    VT *wbase = reinterpret_cast<VT *>(smem_raw) + (size_t)warp * AS;
    VT *sA = wbase + q * m;           // F -> rho -> delta -> T_new
    VT *sB = wbase + WA + q * m;      // lam*g -> alpha
    VT *sC = wbase + 2 * WA + q * m;  // gamma (shared-memory form only)
    // TMEM form: the block's columns (32 when a lane's 4 V + 4 fit, so that
    // more blocks share an SM's 512), this warp's lane quarter
    // (warp 0 allocates now; the address is read after the barrier that
    // follows the first round's loads, so the allocation overlaps them)
    __shared__ unsigned s_tmem;
    unsigned tm_base = 0, tm_lane = 0;
    const unsigned tm_cols = 8 * V <= 32 ? 32u : 64u;
    if constexpr (TM) {
        if (warp == 0) tm_alloc(&s_tmem, tm_cols);
        tm_fence_before();
    }
    const int swsh = J.swz >= 2 ? J.swz - 1 : logU;
    const int swmk = J.swz == 1 ? 0 : 7;
    auto swz = [mfull, swsh, swmk](int c) { return c < mfull ? c ^ ((c >> swsh) & swmk) : c; };

    // ---- A: face fluxes and lam*g, coalesced (lane t: chunks v*P + t), last round first
    {
        const VT *vd = reinterpret_cast<const VT *>(rd), *vc = reinterpret_cast<const VT *>(rc),
                 *vu = reinterpret_cast<const VT *>(ru);
        const VT *vbd = reinterpret_cast<const VT *>(rbd), *vbu = reinterpret_cast<const VT *>(rbu);
        R Tcar = R(0), vcar = R(0);  // cell 0 of chunk (v+1)P, from the team's lane 0
        R wcar = R(0);               // the same for the second transverse axis (D3)
        // the loads of the next RING rounds are issued before a round's arithmetic
        typedef decltype(ld_raw(G)) CT;
        const int p1 = J.per_line ? 0 : n - 1;
        auto ldT = [&](const VT *v, const R *row, int c) -> VT {
            if constexpr (RAG) return ld_ragged<N>(row, c, n, p1);
            else return v[c];
        };
        auto ldC = [&](const C *row, int c) -> CT {
            if constexpr (RAG) return ld_ragged<N>(row, c, n, p1);
            else if constexpr (COH) return *reinterpret_cast<const CT *>(row + c * N);
            else return ld_raw(row + c * N);
        };
        int cl[RING];
        VT xc[RING], xd[RING], xu[RING], xbd[RING], xbu[RING];
        CT xg[RING], xe[RING], xe2[RING];
#pragma unroll
        for (int r = 0; r < RING; ++r) {
            cl[r] = min((max(V - 1 - r, 0) << logP) + t, m - 1);
            xc[r] = xd[r] = xu[r] = xbd[r] = xbu[r] = ldT(vc, rc, cl[r]);
            xg[r] = xe[r] = xe2[r] = ldC(G, cl[r]);
            if constexpr (!IMPL) {
                xd[r] = ldT(vd, rd, cl[r]);
                xu[r] = ldT(vu, ru, cl[r]);
                xe[r] = ldC(E, cl[r]);
            }
            if constexpr (D3 && !IMPL) {
                xbd[r] = vbd[cl[r]];
                xbu[r] = vbu[cl[r]];
                xe2[r] = ld_raw(E2 + cl[r] * N);
            }
        }
        // the cell after the line (periodic wrap or mirrored ghost), issued
        // with the first round's loads instead of inside that round (2-D; the
        // 3-D and temperature-dependent forms, short of registers, load it
        // where it is used)
        constexpr bool EARLY = !D3 && !NL;
        R eT = R(0), eU = R(0), eD = R(0);
        if constexpr (EARLY) {
            eT = rc[p1];
            if constexpr (!IMPL) {
                eU = ru[p1];
                eD = rd[p1];
            }
        }
        if constexpr (TM) {  // the block's TMEM address, the first loads in flight
            __syncthreads();
            tm_fence_after();
            tm_base = s_tmem;
            tm_lane = tm_base + ((unsigned)(32 * (warp & 3)) << 16);
        }
#pragma unroll UNR
        for (int v0 = V - 1; v0 >= 0; v0 -= RING)
#pragma unroll
        for (int r = 0; r < RING; ++r) {
            const int v = v0 - r;
            if (RING > 1 && v < 0) break;
            const int c = (v << logP) + t;
            R Td[N], Tc[N], Tu[N], Gv[N], Ev[N], Tbd[N], Tbu[N], E2v[N];
            V16<R>::unpack(xc[r], Tc);
            // TMEM form: this chunk of T_old waits in the lane's columns 4 (V + v)
            // for phase C, which takes the same chunks by the same lanes
            if constexpr (TM) tm_st4(tm_lane + 4u * (unsigned)(V + v), Tc[0], Tc[1], Tc[2], Tc[3]);
            unpack_raw(xg[r], Gv);
            if constexpr (!IMPL) {
                V16<R>::unpack(xd[r], Td);
                V16<R>::unpack(xu[r], Tu);
                unpack_raw(xe[r], Ev);
            }
            if constexpr (D3 && !IMPL) {
                V16<R>::unpack(xbd[r], Tbd);
                V16<R>::unpack(xbu[r], Tbu);
                unpack_raw(xe2[r], E2v);
            }
            const int cur = cl[r];
            if (v >= RING) {
                cl[r] = ((v - RING) << logP) + t;  // always < m
                xc[r] = ldT(vc, rc, cl[r]);
                xg[r] = ldC(G, cl[r]);
                if constexpr (!IMPL) {
                    xd[r] = ldT(vd, rd, cl[r]);
                    xu[r] = ldT(vu, ru, cl[r]);
                    xe[r] = ldC(E, cl[r]);
                }
                if constexpr (D3 && !IMPL) {
                    xbd[r] = vbd[cl[r]];
                    xbu[r] = vbu[cl[r]];
                    xe2[r] = ld_raw(E2 + cl[r] * N);
                }
            }
            R vv[N], ww[N];
            if constexpr (!IMPL) {
#pragma unroll
                for (int j = 0; j < N; ++j) vv[j] = LM::inner(lim, Tu[j] - Tc[j], Tc[j] - Td[j]);
            }
            if constexpr (D3 && !IMPL) {
#pragma unroll
                for (int j = 0; j < N; ++j) ww[j] = LM::inner(lim, Tbu[j] - Tc[j], Tc[j] - Tbd[j]);
            }
            R nT = __shfl_down_sync(full, Tc[0], 1, P), nv = R(0), nw = R(0);
            if constexpr (!IMPL) nv = __shfl_down_sync(full, vv[0], 1, P);
            if constexpr (D3 && !IMPL) nw = __shfl_down_sync(full, ww[0], 1, P);
            if (t == P - 1) {
                nT = Tcar;
                nv = vcar;
                nw = wcar;
            }
            if (cur == m - 1) {  // the cell after the line
                if constexpr (!EARLY) {
                    nT = rc[p1];
                    if constexpr (!IMPL) nv = LM::inner(lim, ru[p1] - nT, nT - rd[p1]);
                    if constexpr (D3 && !IMPL) nw = LM::inner(lim, rbu[p1] - nT, nT - rbd[p1]);
                } else {
                    nT = eT;
                    if constexpr (!IMPL) nv = LM::inner(lim, eU - nT, nT - eD);
                }
            }
            Tcar = __shfl_sync(full, Tc[0], 0, P);
            if constexpr (!IMPL) vcar = __shfl_sync(full, vv[0], 0, P);
            if constexpr (D3 && !IMPL) wcar = __shfl_sync(full, ww[0], 0, P);
            R F[N], lg[N], hf[N];
            if constexpr (NL) {
                R ch[N + 1];
#pragma unroll
                for (int j = 0; j < N; ++j) ch[j] = chi_of(Tc[j]);
                ch[N] = chi_of(nT);
#pragma unroll
                for (int j = 0; j < N; ++j) hf[j] = face_harmonic<R>(ch[j], ch[j + 1]);
            }
#pragma unroll
            for (int j = 0; j < N; ++j) {
                const R Tnx = j + 1 < N ? Tc[j + 1] : nT;
                const R gj = NL ? Gv[j] * hf[j] : Gv[j];
                lg[j] = lam * gj;
                if constexpr (IMPL) {
                    F[j] = lg[j] * (Tnx - Tc[j]);
                } else {
                    const R vnx = j + 1 < N ? vv[j + 1] : nv;
                    const R ej = NL ? Ev[j] * hf[j] : Ev[j];
                    F[j] = fma_rn(lg[j], Tnx - Tc[j], mul_rn(mul_rn(mu, ej), LM::outer(lim, vv[j], vnx)));
                }
                if constexpr (D3 && !IMPL) {
                    const R wnx = j + 1 < N ? ww[j + 1] : nw;
                    F[j] = fma_rn(mul_rn(mu2, NL ? E2v[j] * hf[j] : E2v[j]), LM::outer(lim, ww[j], wnx), F[j]);
                }
            }
            if (c < m) {
                sA[swz(c)] = V16<R>::pack(F);
                sB[swz(c)] = V16<R>::pack(lg);
            }
        }
    }
    __syncwarp();

    // ---- B1: bottom-up elimination of lane t's segment
    Segment<R> sg;
    R lgem = R(0), lge = R(0), re = R(0), lgs = R(0);
    {
        R Fpend = R(0), lgpend = R(0), Flast = R(0);
        R ro[N], ao[N], go[N];  // maps of the chunk above, waiting for its row 0
        bool pend = false;      // RAG: the segment ends in row 0 of its last chunk, whose lower face is still to come
#pragma unroll
        for (int v = 0; v < N; ++v) ro[v] = ao[v] = go[v] = R(0);
        // Chunk k = 0, 1, .. counts down from the segment's last, ce: the lanes'
        // segments differ by one chunk at their other end, so all eliminate their
        // last chunks together.  (TMEM form: every lane runs all V rounds, so that
        // the warp-wide stores stay uniform; chunk k's gamma goes to column 4 k.)
        R gs[N];  // gamma of chunk k - 1 once its row 0 is eliminated (TMEM form)
#pragma unroll
        for (int j = 0; j < N; ++j) gs[j] = R(0);
#pragma unroll UNR
        for (int k = 0; k < (VC > 0 || TM ? V : Ut); ++k) {
            if ((VC == 0 && !TM) || k < V - 1 || k < Ut) {
            const int c = ce - k;
            R F[N], lg[N], co[N], cao[N], cgo[N];
            V16<R>::unpack(sA[swz(c)], F);
            V16<R>::unpack(sB[swz(c)], lg);
            if (RAG && k == 0 && c == m - 1 && nv < N) {
                // the line's last cell is position nv - 1
                Flast = F[0];
                lge = lg[0];
                pend = nv == 1;
#pragma unroll
                for (int j = 1; j < N; ++j) {
                    co[j] = cao[j] = cgo[j] = R(0);
                    if (j == nv - 1) {
                        Flast = F[j];
                        lge = lg[j];
                        lgem = lg[j - 1];
                        re = F[j] - F[j - 1];
                    }
                }
#pragma unroll
                for (int j = N - 2; j >= 1; --j)
                    if (j < nv - 1) sg.elim(F[j], F[j - 1], lg[j], lg[j - 1], co[j], cao[j], cgo[j]);
            } else if (k == 0) {
                // row e (last cell of the segment) enters the reduced system
                lge = lg[N - 1];
                lgem = lg[N - 2];
                re = F[N - 1] - F[N - 2];
                Flast = F[N - 1];
                co[N - 1] = cao[N - 1] = cgo[N - 1] = R(0);
#pragma unroll
                for (int j = N - 2; j >= 1; --j) sg.elim(F[j], F[j - 1], lg[j], lg[j - 1], co[j], cao[j], cgo[j]);
            } else {
                // row 0 of the chunk above, then this chunk's rows N-1 .. 1
                if (RAG && pend) {
                    lgem = lg[N - 1];
                    re = Flast - F[N - 1];
                    pend = false;
                } else {
                    sg.elim(Fpend, F[N - 1], lgpend, lg[N - 1], ro[0], ao[0], go[0]);
                }
                sA[swz(c + 1)] = V16<R>::pack(ro);
                sB[swz(c + 1)] = V16<R>::pack(ao);
                if constexpr (TM) {
#pragma unroll
                    for (int j = 0; j < N; ++j) gs[j] = go[j];
                } else {
                    sC[swz(c + 1)] = V16<R>::pack(go);
                }
#pragma unroll
                for (int j = N - 1; j >= 1; --j) sg.elim(F[j], F[j - 1], lg[j], lg[j - 1], co[j], cao[j], cgo[j]);
            }
            Fpend = F[0];
            lgpend = lg[0];
#pragma unroll
            for (int j = 1; j < N; ++j) {
                ro[j] = co[j];
                ao[j] = cao[j];
                go[j] = cgo[j];
            }
            }
            // (the last round's, which only the longer segments have, is stored below)
            if constexpr (TM)
                if (k >= 1 && k < V - 1) tm_st4(tm_lane + 4u * (unsigned)(k - 1), gs[0], gs[1], gs[2], gs[3]);
        }
        // row s needs the face below the segment: the previous lane's last face
        const int tp = (t - 1) & (P - 1);
        const R Fprev = __shfl_sync(full, Flast, tp, P), lgprev = __shfl_sync(full, lge, tp, P);
        lgs = lgprev;
        if (RAG && pend) {  // a segment of one cell: its row is row e
            lgem = lgprev;
            re = Flast - Fprev;
        } else {
            sg.elim(Fpend, Fprev, lgpend, lgprev, ro[0], ao[0], go[0]);
        }
        sA[swz(c_lo)] = V16<R>::pack(ro);
        sB[swz(c_lo)] = V16<R>::pack(ao);
        if constexpr (TM) {
            // a segment of V chunks: chunk V - 2 at 4 (V - 2), V - 1 at 4 (V - 1); one of V - 1: V - 2 is its first
            const bool lng = Ut == V;
            if (V >= 2)
                tm_st4(tm_lane + 4u * (unsigned)(V - 2), lng ? gs[0] : go[0], lng ? gs[1] : go[1], lng ? gs[2] : go[2],
                       lng ? gs[3] : go[3]);
            tm_st4(tm_lane + 4u * (unsigned)(V - 1), go[0], go[1], go[2], go[3]);
            tm_wait_st();  // the recovery below reads these columns back
        } else {
            sC[swz(c_lo)] = V16<R>::pack(go);
        }
    }

    // Phase C's first two chunks of T_old start loading now, so that their
    // latency hides behind R and B2 (-3 to -4 % measured on 1024-cell lines).
    // (TMEM form: T_old is in tensor memory already)
    const VT *vcC = reinterpret_cast<const VT *>(rc);
    VT pre0{}, pre1{};
    auto ld_old = [&](int c) -> VT {
        if constexpr (RAG) return ld_ragged<N>(rc, c, n, n - 1);
        else return vcC[c];
    };
    if constexpr (!TM) {
        pre0 = pre1 = ld_old(t);  // t < P <= m
        if (t + P < m) pre1 = ld_old(t + P);
    }

    // ---- R: reduced system of the line in the segment-end unknowns
    R X, Xm;
    {
        const int tn = (t + 1) & (P - 1);
        const R rho_n = __shfl_sync(full, sg.rho, tn, P), alp_n = __shfl_sync(full, sg.alp, tn, P),
                gam_n = __shfl_sync(full, sg.gam, tn, P);
        X = pcr_team<R>(sg.reduced(lgem, lge, re, lgs, rho_n, alp_n, gam_n), t, P);
        Xm = __shfl_sync(full, X, (t - 1) & (P - 1), P);
    }

    // ---- B2: forward recovery of lane t's segment (delta over rho)
    {
        R dprev = Xm;
#pragma unroll UNR
        for (int k = (VC > 0 || TM ? V : Ut) - 1; k >= 0; --k) {
            R g4[N];
            if constexpr (TM) tm_ld4(tm_lane + 4u * (unsigned)k, reinterpret_cast<float *>(g4));  // warp-wide
            if ((VC > 0 || TM) && k == V - 1 && k >= Ut) continue;
            const int c = ce - k;
            R r4[N], a4[N], d[N];
            V16<R>::unpack(sA[swz(c)], r4);
            V16<R>::unpack(sB[swz(c)], a4);
            if constexpr (!TM) V16<R>::unpack(sC[swz(c)], g4);
#pragma unroll
            for (int j = 0; j < N; ++j) {
                d[j] = (k == 0 && j == N - 1) ? X : r4[j] - a4[j] * dprev - g4[j] * X;
                if (RAG && c == m - 1 && j >= nv - 1) d[j] = j == nv - 1 ? X : R(0);
                dprev = d[j];
            }
            sA[swz(c)] = V16<R>::pack(d);
        }
    }
    __syncwarp();

    // ---- C: T_new = T_old + delta, coalesced
    bool bad = false;
    R probe = R(0);
    // diagnostics: compensated sum of the chunk sums, min, max of this lane's cells
    const bool diag = args.diag_part != nullptr;
    R dh = R(0), dl = R(0), dmn = R(INFINITY), dmx = R(-INFINITY);
    {
        VT *vout = reinterpret_cast<VT *>(static_cast<R *>(J.Tout) + (size_t)lc * n);
#pragma unroll UNR
        for (int v = 0; v < V; ++v) {
            const int c = (v << logP) + t;
            R to[N], d[N];
            if constexpr (TM) {
                tm_ld4(tm_lane + 4u * (unsigned)(V + v), to);  // warp-wide, before the lane's bound check
                if (c >= m) continue;
            } else {
                if (c >= m) break;
                V16<R>::unpack(pre0, to);
                pre0 = pre1;  // two chunks in flight
                if (c + 2 * P < m) pre1 = ld_old(c + 2 * P);
            }
            V16<R>::unpack(sA[swz(c)], d);
#pragma unroll
            for (int j = 0; j < N; ++j) {
                to[j] += d[j];
                if constexpr (N == 4) probe = finite_probe(probe, to[j]);
                else bad |= non_finite(to[j]);
            }
            if (diag && active) {
                R sum = R(0);
#pragma unroll
                for (int j = 0; j < N; ++j) sum += to[j];
                const R y = sum - dl, tt = dh + y;
                dl = (tt - dh) - y;
                dh = tt;
#pragma unroll
                for (int j = 0; j < N; ++j) {
                    dmn = fmin(dmn, to[j]);
                    dmx = fmax(dmx, to[j]);
                }
            }
            if (!J.transpose_out) {
                if constexpr (RAG) {
                    R *o = static_cast<R *>(J.Tout) + (size_t)lc * n + (size_t)c * N;
#pragma unroll
                    for (int j = 0; j < N; ++j)
                        if (active && c * N + j < n) o[j] = to[j];
                } else {
                    if (active) vout[c] = V16<R>::pack(to);
                }
            } else {
                sA[swz(c)] = V16<R>::pack(to);
            }
        }
    }

    // ---- transposed store: out[p][line], N lines per 16-byte store.  With
    // two or more line groups a block (short lines), lanes l and l + 16 of a
    // warp write neighbouring groups of one position, so that each store
    // instruction fills whole 32-byte sectors (16 positions x 2 groups).
    if (J.transpose_out) {
        __syncthreads();
        R *out = static_cast<R *>(J.Tout);
        const int groups = LPB >> LOGN, logG = __ffs(groups) - 1;
        const bool vec_ok = (nl & (N - 1)) == 0 && (!RAG || (reinterpret_cast<uintptr_t>(out) & 15) == 0);
        const int pairs = groups == 1 ? n : (((n + 15) & ~15) << logG);
        for (int idx = threadIdx.x; idx < pairs; idx += blockDim.x) {
            const int p = groups == 1 ? idx : (((idx >> (4 + logG)) << 4) | (idx & 15));
            const int grp = groups == 1 ? 0 : ((idx >> 4) & (groups - 1));
            if (p >= n) continue;
            const int sc = swz(p >> LOGN), j = p & (N - 1);
            {
                R o[N];
#pragma unroll
                for (int i = 0; i < N; ++i) {
                    const int lb = (grp << LOGN) + i;
                    const VT *src = reinterpret_cast<const VT *>(smem_raw) + (size_t)(lb >> logL) * AS +
                                    (lb & ((1 << logL) - 1)) * m + sc;
                    o[i] = reinterpret_cast<const R *>(src)[j];
                }
                const int l0 = line0 + (grp << LOGN);
                R *dst = out + (size_t)p * nl + l0;
                if (vec_ok && l0 + N <= nl) {
                    *reinterpret_cast<VT *>(dst) = V16<R>::pack(o);
                } else {
#pragma unroll
                    for (int i = 0; i < N; ++i)
                        if (l0 + i < nl) dst[i] = o[i];
                }
            }
        }
    }
    if ((bad || (N == 4 && non_finite(probe))) && active) atomicOr(args.err, 1u);
    if (diag) {  // the block's partial, reduced in a fixed order (deterministic)
        __shared__ DiagPart s_diag[8];
        double ds = (double)dh - (double)dl, mn = (double)dmn, mx = (double)dmx;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            ds += __shfl_xor_sync(full, ds, o);
            mn = fmin(mn, __shfl_xor_sync(full, mn, o));
            mx = fmax(mx, __shfl_xor_sync(full, mx, o));
        }
        if (lane == 0) s_diag[warp] = DiagPart{ds, mn, mx};
        __syncthreads();
        if (threadIdx.x == 0) {
            DiagPart p = s_diag[0];
            for (int w = 1; w < (int)(blockDim.x >> 5); ++w) {
                p.sum += s_diag[w].sum;
                p.mn = fmin(p.mn, s_diag[w].mn);
                p.mx = fmax(p.mx, s_diag[w].mx);
            }
            args.diag_part[blockIdx.x] = p;
        }
    }
    if constexpr (TM) {  // every warp is done with TMEM before the block frees it
        tm_fence_before();
        __syncthreads();
        if (warp == 0) {
            tm_fence_after();
            tm_dealloc(tm_base, tm_cols);
        }
    }
}

}  // namespace aniso

// Device functions shared by the evaluation kernels (evaluate.cu: one thread per
// particle; evaluate_group.cu: a group of lanes per particle): the basis and cutoff of
// Eq. 6-8, pair vectors, list walks, the four-body invariant, the sphere-reduced
// polynomials, fixed-point accumulation and the deterministic FP64 totals.
#pragma once

#include "nep_common.cuh"
#include "poly32.cuh"
#include "poly64.cuh"
#include "sh_poly.cuh"

namespace nep {

__host__ __device__ constexpr int l_of(int k) { return k < 3 ? 1 : (k < 8 ? 2 : (k < 15 ? 3 : 4)); }
constexpr int kNLM = 24;
// The FP32 kernels are compiled for 2 and for 3 resident blocks per SM (which caps
// registers per thread); the runtime picks one per handle (autotuned).

// The cutoff of Eq. 8 halved, f_c / 2, and its derivative halved, f_c' / 2, at
// x = r / r_c in [0, 1].  FP32 evaluates the polynomials of poly32.cuh
// (the hardware sine and cosine err by about 1e-7 with a consistent sign, which
// summed over pairs biases the energy), FP64 those of poly64.cuh (on this range they take
// half the FP64 instructions of cospi and sincospi, and the FP64 kernels are bound by those).
__device__ __forceinline__ float cut_half(float x)
{
    const float y = x - 0.5f;
    return fmaf(-y, cut_p(y * y), 0.25f);
}
__device__ __forceinline__ double cut_half(double x)
{
    const double y = x - 0.5;
    return fma(-y, cut_p64(y * y), 0.25);
}
__device__ __forceinline__ void cut_half_d(float x, float inv_rc, float* hf, float* hdf)
{
    const float y = x - 0.5f;
    const float z = y * y;
    *hf = fmaf(-y, cut_p(z), 0.25f);
    *hdf = -cut_q(z) * inv_rc;
}
__device__ __forceinline__ void cut_half_d(double x, double inv_rc, double* hf, double* hdf)
{
    const double y = x - 0.5;
    const double z = y * y;
    *hf = fma(-y, cut_p64(z), 0.25);
    *hdf = -cut_q64(z) * inv_rc;
}

// Chebyshev basis f_k(r) of Eq. 7 with the cutoff of Eq. 8, k = 0..K-1, by the
// three-term recurrence T_{k+1} = 2 x T_k - T_{k-1}.
// x = r / r_c from the inverse cutoff and its FP32 rounding residual (FP64: exact enough)
__device__ __forceinline__ float scaled_r(float r, float inv_rc, float inv_lo) { return fmaf(r, inv_lo, r * inv_rc); }
__device__ __forceinline__ double scaled_r(double r, double inv_rc, double) { return r * inv_rc; }

template <typename real, int K>
__device__ __forceinline__ void basis(real r, real inv_rc, real inv_lo, real* f)
{
    const real xr = scaled_r(r, inv_rc, inv_lo);
    const real hf = cut_half(xr);  // f_c / 2
    const real s = xr - real(1);
    const real x = real(2) * s * s - real(1);
    const real x2 = x + x;
    real t0 = real(1), t1 = x;
    f[0] = hf + hf;
    if (K > 1) f[1] = hf * x + hf;
#pragma unroll
    for (int k = 2; k < K; ++k) {
        const real t2 = x2 * t1 - t0;
        f[k] = hf * t2 + hf;  // (T_k + 1) f_c / 2
        t0 = t1;
        t1 = t2;
    }
}

// Pair sums of the basis, split as f_k = (f_c/2) T_k + f_c/2: acc[k] += (f_c/2) T_k
// and hs += f_c/2, so that sum_j f_k = acc[k] + hs (one FMA per term instead of a
// product and an add).
template <typename real, int K>
__device__ __forceinline__ void basis_acc(real r, real inv_rc, real inv_lo, real (&acc)[K], real& hs)
{
    const real xr = scaled_r(r, inv_rc, inv_lo);
    const real hf = cut_half(xr);  // f_c / 2
    const real s = xr - real(1);
    const real x = real(2) * s * s - real(1);
    const real x2 = x + x;
    real t0 = real(1), t1 = x;
    hs += hf;
    acc[0] += hf;
    if (K > 1) acc[1] = fma(hf, x, acc[1]);
#pragma unroll
    for (int k = 2; k < K; ++k) {
        const real t2 = x2 * t1 - t0;
        acc[k] = fma(hf, t2, acc[k]);
        t0 = t1;
        t1 = t2;
    }
}

// The angular functions g_n(r) = sum_k c_nk f_k(r) are evaluated from the Chebyshev sums:
//   g_n = (f_c/2) P_n(x),  P_n = c'_n0 + sum_{k>=1} c_nk T_k(x),  c'_n0 = 2 c_n0 + sum_{k>=1} c_nk,
//   g_n' = (f_c/2) x' sum_{k>=1} c_nk T_k'(x) + (f_c'/2) P_n,
// with c' in place of c in column 0 of the angular tables, so the f_k and f_k' themselves
// need not be formed.  cheb_T: f_c/2 and T_k; cheb_dT: f_c/2, f_c'/2, x' f_c/2, T_k, T_k'
// (entry 0 unused).
template <typename real, int K>
__device__ __forceinline__ void cheb_T(real r, real inv_rc, real inv_lo, real& hf, real (&t)[K])
{
    const real xr = scaled_r(r, inv_rc, inv_lo);
    hf = cut_half(xr);
    const real s = xr - real(1);
    const real x = fma(real(2) * s, s, real(-1));
    const real x2 = x + x;
    t[0] = real(1);
    t[1] = x;
#pragma unroll
    for (int k = 2; k < K; ++k) t[k] = fma(x2, t[k - 1], -t[k - 2]);
}
template <typename real, int K>
__device__ __forceinline__ void cheb_dT(real r, real inv_rc, real inv_lo, real& hf, real& hdf, real& hdx, real (&t)[K],
                                        real (&d)[K])
{
    const real xr = scaled_r(r, inv_rc, inv_lo);
    cut_half_d(xr, inv_rc, &hf, &hdf);
    const real s = xr - real(1);
    const real x = fma(real(2) * s, s, real(-1));
    hdx = real(4) * s * inv_rc * hf;
    const real x2 = x + x;
    t[0] = real(1);
    t[1] = x;
    d[0] = real(0);
    d[1] = real(1);
#pragma unroll
    for (int k = 2; k < K; ++k) {  // T'_k = 2 T_{k-1} + 2 x T'_{k-1} - T'_{k-2}
        t[k] = fma(x2, t[k - 1], -t[k - 2]);
        d[k] = fma(real(2), t[k - 1], fma(x2, d[k - 1], -d[k - 2]));
    }
}
template <typename real, int K>
__device__ __forceinline__ real cheb_sum(const real (&c)[K], const real (&t)[K])
{
    real p = c[0];
#pragma unroll
    for (int k = 1; k < K; ++k) p = fma(c[k], t[k], p);
    return p;
}
// g_n and g_n' from one row of coefficients
template <typename real, int K>
__device__ __forceinline__ void cheb_g_dg(const real (&c)[K], const real (&t)[K], const real (&d)[K], real hf, real hdf,
                                          real hdx, real& g, real& dg)
{
    const real p = cheb_sum(c, t);
    real q = c[1];
#pragma unroll
    for (int k = 2; k < K; ++k) q = fma(c[k], d[k], q);
    g = hf * p;
    dg = fma(hdx, q, hdf * p);
}

// f_k and df_k/dr:  df_k = 1/2 [T_k'(x) x'(r) f_c + (T_k + 1) f_c'],
// with T'_{k+1} = 2 T_k + 2 x T'_k - T'_{k-1}.
template <typename real, int K>
__device__ __forceinline__ void basis_d(real r, real inv_rc, real inv_lo, real* f, real* df)
{
    const real xr = scaled_r(r, inv_rc, inv_lo);
    real hf, hdf;  // f_c / 2, f_c' / 2
    cut_half_d(xr, inv_rc, &hf, &hdf);
    const real s = xr - real(1);
    const real x = real(2) * s * s - real(1);
    const real hdx = real(4) * s * inv_rc * hf;                             // x'(r) f_c / 2
    const real x2 = x + x;
    real t0 = real(1), t1 = x, d0 = real(0), d1 = real(1);
    f[0] = hf + hf;
    df[0] = hdf + hdf;
    if (K > 1) {
        f[1] = hf * x + hf;
        df[1] = hdx + (hdf * x + hdf);
    }
#pragma unroll
    for (int k = 2; k < K; ++k) {
        const real t2 = x2 * t1 - t0;
        const real d2 = real(2) * t1 + (x2 * d1 - d0);
        f[k] = hf * t2 + hf;
        df[k] = d2 * hdx + (hdf * t2 + hdf);
        t0 = t1;
        t1 = t2;
        d0 = d1;
        d1 = d2;
    }
}

// Pair vector r_ij from i's and j's records and the entry's cell offset.
template <typename real>
__device__ __forceinline__ void pair_vec(const real* len, const PosRec<real>& ri, const PosRec<real>& rj, uint32_t e,
                                         real& dx, real& dy, real& dz)
{
    const uint32_t code = e >> kJBits;
    dx = (rj.x - ri.x) + (real)((int)(code & 7u) - 2) * len[0];
    dy = (rj.y - ri.y) + (real)((int)((code >> 3) & 7u) - 2) * len[1];
    dz = (rj.z - ri.z) + (real)((int)((code >> 6) & 7u) - 2) * len[2];
}

template <typename real>
__device__ __forceinline__ real norm2(real x, real y, real z)
{
    return fma(z, z, fma(y, y, x * x));
}

// f_ij from D = sum_n g_n' P_n(u) and ga = sum_n g_n grad P_n(u), ga's radial part removed:
// (D - (u . ga) / r) u + ga / r.
template <typename real>
__device__ __forceinline__ void angular_force(real D, const real (&ga)[3], real ux, real uy, real uz, real inv_r,
                                              real (&fij)[3])
{
    const real sr = fma(-fma(uz, ga[2], fma(uy, ga[1], ux * ga[0])), inv_r, D);
    fij[0] = fma(sr, ux, ga[0] * inv_r);
    fij[1] = fma(sr, uy, ga[1] * inv_r);
    fij[2] = fma(sr, uz, ga[2] * inv_r);
}

// Software-pipelined walk over one particle's neighbour list: the entries are
// loaded two iterations ahead and the neighbour's record one iteration ahead, so
// the dependent load chain (entry -> record) overlaps the previous pair's math.
template <typename real>
struct NbrWalk {
    const uint32_t* nl;  // &list[0][i]
    size_t stride;
    int cnt;
    const PosRec<real>* rec;
    uint32_t e0, e1;
    PosRec<real> r0;
    __device__ __forceinline__ NbrWalk(const uint32_t* list, int n, int i, int c, const PosRec<real>* recs)
        : nl(list + i), stride((size_t)n), cnt(c), rec(recs)
    {
        e0 = c > 0 ? nl[0] : 0u;
        e1 = c > 1 ? nl[stride] : 0u;
        r0 = rec[e0 & kJMask];  // index 0 is valid even for an empty list
    }
    // current entry and record, then advance the pipeline (s = current index)
    __device__ __forceinline__ void next(int s, uint32_t& e, PosRec<real>& rj)
    {
        e = e0;
        rj = r0;
        e0 = e1;
        e1 = (s + 2 < cnt) ? nl[(size_t)(s + 2) * stride] : 0u;
        r0 = rec[e0 & kJMask];
    }
};

// Walk over a column-major neighbour list whose entries are loaded 4 to 8 pairs
// ahead of use (the list is streamed from L2; a short loop body cannot hide that
// latency with a shallower prefetch).  body(entry) is called for every entry in order.
template <typename Body>
__device__ __forceinline__ void walk4(const uint32_t* nl, size_t stride, int cnt, Body&& body)
{
    auto ld = [&](int s) { return s < cnt ? nl[(size_t)s * stride] : 0u; };
    uint32_t q0 = ld(0), q1 = ld(1), q2 = ld(2), q3 = ld(3);
    int s = 0;
    for (; s + 4 <= cnt; s += 4) {
        const uint32_t a0 = q0, a1 = q1, a2 = q2, a3 = q3;
        q0 = ld(s + 4);
        q1 = ld(s + 5);
        q2 = ld(s + 6);
        q3 = ld(s + 7);
        body(a0);
        body(a1);
        body(a2);
        body(a3);
    }
    if (s < cnt) body(q0);
    if (s + 1 < cnt) body(q1);
    if (s + 2 < cnt) body(q2);
}

// walk4 generalised to groups of CH entries (CH = 4 or 8): the next group's
// entries are loaded while the current group is evaluated, so up to 2 CH entries
// (and CH pairs' neighbour loads) are in flight per thread.
template <int CH, typename Body>
__device__ __forceinline__ void walk_chunk(const uint32_t* nl, size_t stride, int cnt, Body&& body)
{
    auto ld = [&](int s) { return s < cnt ? nl[(size_t)s * stride] : 0u; };
    uint32_t q[CH];
#pragma unroll
    for (int u = 0; u < CH; ++u) q[u] = ld(u);
    int s = 0;
    for (; s + CH <= cnt; s += CH) {
        uint32_t cur[CH];
#pragma unroll
        for (int u = 0; u < CH; ++u) {
            cur[u] = q[u];
            q[u] = ld(s + CH + u);
        }
#pragma unroll
        for (int u = 0; u < CH; ++u) body(cur[u]);
    }
#pragma unroll
    for (int u = 0; u < CH - 1; ++u)
        if (s + u < cnt) body(q[u]);
}

// Half of a walk in groups of eight: the entries first ... first + 3 of every eight (first =
// 0 or 4), with the position among the four as the body's second argument (0..3, a constant
// after unrolling), so that a body can keep four partial sums.  The two halves' sums are
// partial sums by slot number mod 8: each grows to an eighth of the total, which cuts the
// FP32 rounding of a long accumulation, and they are the sums that the eight lanes of
// evaluate_group.cu form.  (All eight at once cost the four-type monolayer, with six pairs a
// particle, 1.5% of a step.)
template <typename Body>
__device__ __forceinline__ void walk_half(const uint32_t* nl, size_t stride, int cnt, int first, Body&& body)
{
    auto ld = [&](int s) { return s < cnt ? nl[(size_t)s * stride] : 0u; };
    int s = first;
    uint32_t q0 = ld(s), q1 = ld(s + 1), q2 = ld(s + 2), q3 = ld(s + 3);
    for (; s + 4 <= cnt; s += 8) {
        const uint32_t a0 = q0, a1 = q1, a2 = q2, a3 = q3;
        q0 = ld(s + 8);
        q1 = ld(s + 9);
        q2 = ld(s + 10);
        q3 = ld(s + 11);
        body(a0, 0);
        body(a1, 1);
        body(a2, 2);
        body(a3, 3);
    }
    if (s < cnt) body(q0, 0);
    if (s + 1 < cnt) body(q1, 1);
    if (s + 2 < cnt) body(q2, 2);
}

// 4 consecutive reals (16-byte aligned) into registers
__device__ __forceinline__ void load4(const float* p, float* o)
{
    const float4 v = *reinterpret_cast<const float4*>(p);
    o[0] = v.x; o[1] = v.y; o[2] = v.z; o[3] = v.w;
}
__device__ __forceinline__ void load4(const double* p, double* o)
{
    const double2 v0 = reinterpret_cast<const double2*>(p)[0], v1 = reinterpret_cast<const double2*>(p)[1];
    o[0] = v0.x; o[1] = v0.y; o[2] = v1.x; o[3] = v1.y;
}

template <typename real, int N>
__device__ __forceinline__ void loadN(const real* p, real* o)
{
#pragma unroll
    for (int k = 0; k + 3 < N; k += 4) load4(p + k, o + k);
#pragma unroll
    for (int k = N & ~3; k < N; ++k) o[k] = p[k];
}

// A gradient vector (N reals, rows 32-byte aligned when N = 8 floats) from global memory: eight
// floats in one 256-bit load, whose one line look-up is what a gather costs.
template <typename real, int N>
__device__ __forceinline__ void load_grad(const real* p, real* o)
{
    if constexpr (sizeof(real) == 4 && N == 8) {
        asm volatile("ld.global.v8.f32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
                     : "=f"(o[0]), "=f"(o[1]), "=f"(o[2]), "=f"(o[3]), "=f"(o[4]), "=f"(o[5]), "=f"(o[6]), "=f"(o[7])
                     : "l"(p));
    } else {
        loadN<real, N>(p, o);
    }
}

// A type pair's n x K coefficient table into registers.  A one-type model's single
// table starts on a 16-byte boundary and is read with vector loads; several types'
// tables sit at odd strides (bank spread) and are read as scalars.
template <typename real, int N>
__device__ __forceinline__ void load_coef(const real* c, bool aligned, real (&o)[N])
{
    if (aligned) {
        loadN<real, N>(c, o);
    } else {
#pragma unroll
        for (int q = 0; q < N; ++q) o[q] = c[q];
    }
}

// 1/sqrt(x): the hardware estimate refined by one Newton-Raphson step on
// f(y) = y^-2 - x, y' = y + y (1 - x y^2) / 2.  The estimate's error has a small
// consistent sign, which through r and u = r_ij / r would bias the descriptors of every
// particle alike; after the step the quadratic term is ~1e-14 and what remains is the
// (unsigned) rounding of y^2.
__device__ __forceinline__ float rsqrt_r(float x)
{
    const float y = rsqrtf(x);
    const float e = fmaf(-x, y * y, 1.0f);
    return fmaf(0.5f * y, e, y);
}
// Conversions between FP64 and FP32 by moving bits, for values of FP32's normal range (the
// conversion instructions run at the FP64 rate): FP64 truncated to FP32, and FP32 widened.
__device__ __forceinline__ bool fp32_range(int hi) { return (unsigned)(hi - 0x38100000) < 0x0fe00000u; }
__device__ __forceinline__ float narrow_bits(double x)
{
    return __int_as_float((int)(((unsigned)__double2hiint(x) - 0x38000000u) << 3 | (unsigned)__double2loint(x) >> 29));
}
__device__ __forceinline__ double widen_bits(float x)
{
    const unsigned b = (unsigned)__float_as_int(x);
    return __hiloint2double((int)((b >> 3) + 0x38000000u), (int)(b << 29));
}

// FP64: the FP32 estimate refined by one step of Householder's third-order iteration,
// y' = y + y e (1/2 + 3/8 e), e = 1 - x y^2 (|e| < 1e-6, so its error is below e^3).
__device__ __forceinline__ double rsqrt_r(double x)
{
    if (!fp32_range(__double2hiint(x))) return rsqrt(x);
    const double y = widen_bits(rsqrtf(narrow_bits(x)));
    const double e = fma(-(x * y), y, 1.0);
    return fma(y * e, fma(0.375, e, 0.5), y);
}

// tanh in FP32.  Each hidden unit's pre-activation keeps one sign over most
// particles, so an activation whose rounding error leans one way on part of its
// range biases every particle's energy alike; CUDA's tanhf does (about -9e-9 on
// [1/4, 1/2]).  Here: on |x| < 1 the odd polynomial of poly32.cuh (mean error below
// 2e-10 on every eighth of the range); beyond, (1 - e) / (1 + e) with
// e = exp(-2|x|), where no cancellation remains, divided through a reciprocal
// refined by one Newton-Raphson step.
__device__ __forceinline__ float tanh_r(float x)
{
    const float a = fabsf(x);
    if (a < 1.0f) {
        const float z = x * x;
        return fmaf(x * z, tanh_r_poly(z), x);
    }
    const float e = expf(-2.0f * a);
    const float d = 1.0f + e;
    float r = __fdividef(1.0f, d);
    r = fmaf(r, fmaf(-d, r, 1.0f), r);
    return copysignf((1.0f - e) * r, x);
}
// FP64: tanh a = -m / (2 + m), m = exp(-2a) - 1, a = |x|.  exp(-2a) = 2^(n/32) exp(r) with
// |r| <= ln 2 / 64: 2^(n/32) from a table, exp(r) - 1 by its series to r^6 (the next term is
// below 4e-18); the reciprocal of 2 + m in (1, 2] is an FP32 one refined to third order.  No
// cancellation: for small a, n = 0 and m is the series alone.
__device__ __forceinline__ double tanh_r(double x)
{
    const int top = __double2hiint(x) & 0x7fffffff;
    if (top >= 0x40340000) return top >= 0x7ff00000 ? tanh(x) : copysign(1.0, x);  // |x| >= 20
    const double t = -2.0 * fabs(x);
    constexpr double kRound = 6755399441055744.0;  // 3 2^51: adding it rounds to an integer
    const double s = fma(t, kLn2Inv, kRound);
    const int n = __double2loint(s);
    const double nd = s - kRound;
    const double r = fma(-nd, kLn2Lo, fma(-nd, kLn2Hi, t));
    double p = fma(r, 1.0 / 720.0, 1.0 / 120.0);
    p = fma(p, r, 1.0 / 24.0);
    p = fma(p, r, 1.0 / 6.0);
    p = fma(p, r, 0.5);
    p = fma(p * r, r, r);  // exp(r) - 1
    const double b = __ldg(kExp2Table + (n & 31));
    const double em = __hiloint2double(__double2hiint(b) + ((n >> 5) << 20), __double2loint(b));
    const double m = fma(em, p + __ldg(kExp2Rest + (n & 31)), em - 1.0);
    const double d = 2.0 + m;
    const double y = widen_bits(__fdividef(1.0f, narrow_bits(d)));
    const double e = fma(-d, y, 1.0);
    const double h = -m * fma(y, fma(e, e, e), y);
    return __hiloint2double(__double2hiint(h) | (__double2hiint(x) & (int)0x80000000), __double2loint(h));
}

// a product that is never contracted into a multiply-add
__device__ __forceinline__ float mul_rn(float x, float y) { return __fmul_rn(x, y); }
__device__ __forceinline__ double mul_rn(double x, double y) { return __dmul_rn(x, y); }

// Four-body invariant of one radial channel's l = 2 moments and its gradient.
// a[0..4] are A_n2m in the real basis of sh_eval (xy, yz, 2z^2 - x^2 - y^2, xz,
// x^2 - y^2).  sum_m a_m Y_2m(u) = u^T M u for the traceless symmetric M built
// below, and M = 15 / (8 pi) Q with Q = sum_j g_j (u_j u_j^T - I/3) (addition
// theorem for l = 2).  The Wigner-coupled triple product
// sum (2 2 2; m1 m2 m3) A_2m1 A_2m2 A_2m3 is the cubic invariant kappa tr(Q^3),
// kappa = (2 2 2; 0 0 0) (5 / 4 pi)^(3/2) 9/2, so q4 = kQ4 tr(M^3) with
// kQ4 = kappa (8 pi / 15)^3 = -32 sqrt(14) pi^(3/2) / 525.  d tr(M^3) / dM = 3 M^2.
constexpr double kQ4 = -1.2699291782903164;
constexpr double kY2xy = 1.0925484305920792;  // sqrt(15 / 4 pi): Y_2 of xy, yz, xz
constexpr double kY2zz = 0.31539156525252005; // sqrt(5 / 16 pi): Y_2 of 2z^2 - x^2 - y^2
constexpr double kY2xx = 0.5462742152960396;  // sqrt(15 / 16 pi): Y_2 of x^2 - y^2

template <typename real>
__device__ __forceinline__ real four_body(const real* a, real* grad)
{
    // (explicit multiply-adds: every kernel that inlines this rounds alike)
    const real c1 = real(kY2xy), c0 = real(kY2zz), c2 = real(kY2xx);
    const real hxy = real(0.5) * c1 * a[0], hyz = real(0.5) * c1 * a[1], hxz = real(0.5) * c1 * a[3];
    const real m0 = mul_rn(c0, a[2]);
    const real mxx = fma(c2, a[4], -m0), myy = fma(-c2, a[4], -m0), mzz = real(2) * m0;
    // M^2 (symmetric)
    const real sxx = fma(hxz, hxz, fma(hxy, hxy, mul_rn(mxx, mxx)));
    const real syy = fma(hyz, hyz, fma(myy, myy, mul_rn(hxy, hxy)));
    const real szz = fma(mzz, mzz, fma(hyz, hyz, mul_rn(hxz, hxz)));
    const real sxy = fma(hxz, hyz, fma(hxy, myy, mul_rn(mxx, hxy)));
    const real sxz = fma(hxz, mzz, fma(hxy, hyz, mul_rn(mxx, hxz)));
    const real syz = fma(hyz, mzz, fma(myy, hyz, mul_rn(hxy, hxz)));
    const real off = fma(hyz, syz, fma(hxz, sxz, mul_rn(hxy, sxy)));
    const real tr3 = fma(real(2), off, fma(mzz, szz, fma(myy, syy, mul_rn(mxx, sxx))));
    // dq4/da_m = kQ4 * 3 * sum_ab (M^2)_ab dM_ab/da_m
    const real k3 = real(3 * kQ4);
    grad[0] = k3 * c1 * sxy;
    grad[1] = k3 * c1 * syz;
    grad[2] = k3 * c0 * (real(2) * szz - sxx - syy);
    grad[3] = k3 * c1 * sxz;
    grad[4] = k3 * c2 * (sxx - syy);
    return real(kQ4) * tr3;
}

// Per-thread state of the force pass for one particle i.
template <typename real, int KRP>
struct ForceCtx {
    PosRec<real> ri;
    int i, ti, T;
    real len[3];
    real F[3];
    real W[9];
};

// 64-bit fixed-point accumulation (2^-32 units): integer sums do not depend on the
// order in which atomic adds arrive, so scattered forces stay bitwise reproducible.
constexpr float kFixScale = 4294967296.0f;  // 2^32 fixed-point units per eV/A (or eV)

__device__ __forceinline__ void fix_add(unsigned long long* p, float v)
{
    atomicAdd(p, (unsigned long long)__float2ll_rn(v * kFixScale));
}

// A fixed-point sum in FP32, the working precision of the forces (kept off the FP64
// pipe)
__device__ __forceinline__ float fix_value_f(unsigned long long v) { return (float)(long long)v * (1.0f / kFixScale); }

// One block of a sphere-reduced polynomial (layout of sh_reduce): the value and the x and
// y derivatives of sum_{a+b<=D} c[o(a) + b] x^a y^b, by Horner's scheme in y for each
// power of x (with the y-derivative) nested in Horner's scheme in x (with the
// x-derivative).
template <int D, bool BLOCK_B, typename real>
__device__ __forceinline__ void red_block(const real* c, real x, real y, real& v, real& vx, real& vy)
{
#pragma unroll
    for (int a = D; a >= 0; --a) {
        const int o = BLOCK_B ? sh_red_b(a) : sh_red_a(a);
        real al = c[o + D - a], dal = real(0);
#pragma unroll
        for (int b = D - a - 1; b >= 0; --b) {
            dal = b == D - a - 1 ? al : fma(dal, y, al);
            al = fma(al, y, c[o + b]);
        }
        if (a == D) {
            v = al;
            vx = vy = real(0);
        } else if (a == D - 1) {
            vx = v;
            v = fma(v, x, al);
            vy = dal;
        } else {
            vx = fma(vx, x, v);
            v = fma(v, x, al);
            vy = fma(vy, x, dal);
        }
    }
}

// Value and gradient at (x, y, z) of the sphere-reduced polynomial c (sh_reduce):
// P = A + z B, grad P = (A_x + z B_x, A_y + z B_y, B).  On the unit sphere P equals
// the harmonic sum it was reduced from, and grad P differs from that sum's gradient
// only along the normal.
template <typename real>
__device__ __forceinline__ void sh_red_eval(const real* c, real x, real y, real z, real& v, real& vx, real& vy,
                                            real& vz)
{
    real pa, pax, pay, pb, pbx, pby;
    red_block<4, false>(c, x, y, pa, pax, pay);
    red_block<3, true>(c, x, y, pb, pbx, pby);
    v = fma(z, pb, pa);
    vx = fma(z, pbx, pax);
    vy = fma(z, pby, pay);
    vz = pb;
}

// The MD step's closing half-kick of particle ui (caller index; lu within its
// request) from its final force, rounded as the separate kick kernel rounds it.
template <typename real>
__device__ __forceinline__ void closing_kick(const EvalArgs<real>& a, const ReqInfo& rq, int ui, int lu,
                                             const double (&F)[3])
{
    const int t = a.kick_types[ui];
    const double im = a.kick_im.v[t >= 0 && t < kMdMaxTypes ? t : 0];
    double* v = a.kick_vel + (size_t)3 * rq.begin + lu;
#pragma unroll
    for (int p = 0; p < 3; ++p) v[(size_t)p * rq.n] = half_kick(v[(size_t)p * rq.n], a.kick_half_dt, F[p], im);
}

// FP64 sums of (E, W[9]) over each request, in a fixed order whatever the timing:
//   1. each block sums its particles: the 10 values of its threads go to shared
//      memory, 80 threads sum 16 each (value k = t / 8, a stride-8 subset), then 10
//      threads sum the 8 parts, into partial[item];
//   2. the last block of each group of kGroup consecutive items of a request (counted
//      from the request's first item) sums the group's block partials and writes the
//      group sum over the group's first partial;
//   3. the last group of the request sums the group sums into totals[req].
// The summing threads take fixed subsets, so a request sums alike alone or in a
// batch.  Spreading the sums over the groups' last blocks keeps the serial tail of
// the kernel (FP64 arithmetic is scarce on this part) to two short passes.

// out[k] = sum over b < nb of src[b * 10 + k] (L2 reads: written by other blocks),
// with 120 threads in a fixed order; the result is valid in threads < 10
__device__ __forceinline__ double sum_partials(const double* src, int nb, int stride_items, double (&part)[10][12])
{
    const int t = threadIdx.x;
    if (t < 120) {
        const int k = t % 10, q = t / 10;
        double s = 0.0;
#pragma unroll 4
        for (int b = q; b < nb; b += 12) s += __ldcg(src + (size_t)b * stride_items * 10 + k);
        part[k][q] = s;
    }
    __syncthreads();
    double s = 0.0;
    if (t < 10) {
#pragma unroll
        for (int q = 0; q < 12; ++q) s += part[t][q];
    }
    return s;
}

template <int BS>
__device__ __forceinline__ void reduce_totals(double (&v)[10], int item, const WorkItem& it, const ReqInfo& rq,
                                              double* partial, unsigned int* gcounter, unsigned int* counter,
                                              const PlanCounts* counts, double* totals)
{
    static_assert(BS % 8 == 0 && BS >= 120, "block size");
    __shared__ double red[10][BS + 8];  // row stride 2 words mod 32 apart: 2-way for 64-bit loads
    __shared__ double part[10][12];
    __shared__ bool last;
    const int t = threadIdx.x;
    // the caller's addresses, loaded here so that the last block does not wait for them
    double *const energy = counts->energy, *const virial = counts->virial;
#pragma unroll
    for (int k = 0; k < 10; ++k) red[k][t] = v[k];
    __syncthreads();
    if (t < 80) {
        const int k = t >> 3, q = t & 7;
        double s = 0.0;
#pragma unroll
        for (int j = 0; j < BS / 8; ++j) s += red[k][8 * j + q];
        part[k][q] = s;
    }
    __syncthreads();
    if (t < 10) {
        double s = 0.0;
#pragma unroll
        for (int q = 0; q < 8; ++q) s += part[t][q];
        partial[(size_t)item * 10 + t] = s;
        __threadfence();  // the writers publish their partials before the count below
    }
    __syncthreads();
    const int rel = item - rq.item_begin;
    const int n_items = rq.item_end - rq.item_begin;
    const int g0 = rq.item_begin + rel / kGroup * kGroup;  // the group's first item
    const int gn = min(kGroup, rq.item_end - g0);
    if (t == 0) last = (atomicAdd(&gcounter[g0], 1u) == (unsigned int)gn - 1u);
    __syncthreads();
    if (!last) return;
    __threadfence();
    const double gs = sum_partials(partial + (size_t)g0 * 10, gn, 1, part);
    const int ng = (n_items + kGroup - 1) / kGroup;
    if (ng == 1) {  // one group: its sum is the total
        if (t < 10) write_total(energy, virial, totals, it.req, t, gs);
        if (t == 0) gcounter[g0] = 0u;
        return;
    }
    if (t < 10) {
        partial[(size_t)g0 * 10 + t] = gs;  // over the group's first partial
        if (t == 0) gcounter[g0] = 0u;
        __threadfence();
    }
    __syncthreads();
    if (t == 0) last = (atomicAdd(&counter[it.req], 1u) == (unsigned int)ng - 1u);
    __syncthreads();
    if (!last) return;
    __threadfence();
    const double ts = sum_partials(partial + (size_t)rq.item_begin * 10, ng, kGroup, part);
    if (t < 10) write_total(energy, virial, totals, it.req, t, ts);
    if (t == 0) counter[it.req] = 0u;
}

// The compiled descriptor shapes (n_R, n_A, K_R, K_A).
#define NEP_SHAPES(X) X(5, 4, 8, 8) X(5, 5, 9, 9)

}  // namespace nep

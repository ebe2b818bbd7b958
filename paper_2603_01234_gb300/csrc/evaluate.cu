// Descriptor + network kernel and force + virial kernel (Eq. 1-8, 15, 16) of the FP32
// forms, one thread per particle, and the dispatch of the evaluation kernels (small FP32
// batches and FP64: evaluate_group.cu).
//
// k_descriptor (one thread per sorted particle i):
//   radial   q_n   = sum_j g_n(r_ij)                              (Eq. 3, 6-8)
//   angular  A_nlm = sum_j g_n(r_ij) Y_lm(u_ij), q_nl = sum_m A^2  (Eq. 4-5)
//            with real orthonormal Y_lm (for real g_n, sum_m (-1)^m A_m A_-m of
//            the complex harmonics equals sum_m A_m^2 of the real ones)
//   network  U_i (Eq. 2) and dU_i/dq
//   stores   U_i;  e_i^t[k] = sum_n dU_i/dq_n c^{t_i t}_{nk} for every partner type t
//            (the radial gradient folded into the basis: dU_i/dr_ij|radial =
//            sum_k e_i^{t_j}[k] f_k'(r_ij) u_ij)
//
// Forces and virials, with
//   F_i = sum_j (f_ij - f_ji),   W_i = sum_j r_ij (x) f_ji   (Eq. 15),
// f_ij = dU_i/dr_ij, and E = sum U_i, W = sum W_i reduced in FP64 (Eq. 1, 16) by
// a deterministic last-block pass: k_descriptor also evaluates the angular pairs, in
// scatter form, from Phi_nlm = dU_i/dA_nlm = 2 dU_i/dq_nl A_nlm while it is in registers
// (Phi never reaches memory): F_i keeps f_ij, and -f_ij (and W_j's term) go to j through
// 64-bit fixed-point atomic adds (order-independent sums); k_force_radial then takes the
// radial pairs in gather form (f_ij and f_ji from i's and j's stored gradient vectors),
// adds the accumulated angular part and writes the outputs.
//
// Angular pair gradient.  For A = g(r) Y(u), u = r/|r|:
//   dA/dr = g' Y(u) u + (g / r) (grad Y(u) - (u . grad Y(u)) u),
// in which only the surface gradient of Y enters.  P_n = sum_lm Phi_nlm Y_lm is
// evaluated through its sphere-reduced polynomial (sh_reduce, sh_red_eval), which has
// P_n's values and surface gradients on the unit sphere.
#include "evaluate_math.cuh"

namespace nep {

template <typename real>
__device__ __forceinline__ void stage_params(const real* __restrict__ src, real* dst, int count)
{
    for (int k = threadIdx.x; k < count; k += blockDim.x) dst[k] = src[k];
    __syncthreads();
}

template <typename real, int NA, int KA, typename Ctx>
__device__ __forceinline__ void force_angular_phi_reg(const EvalArgs<real>& a, const real* P, const ParamLayout& off,
                                                      const real (&Psi)[NA][kShRed], Ctx& c, bool per_bead);

template <typename real, int NR, int NA, int KR, int KA, int RES, int MBT>
__device__ __forceinline__ void descriptor_item(const EvalArgs<real>& a, const WorkItem it, unsigned char* smem_raw);

// One work item per block (launch grids cover the item capacity; blocks past the
// batch's item count exit): the block stages its model's tables, then one thread
// per particle runs descriptor_item.
template <typename real, int NR, int NA, int KR, int KA, int MB, int RES, int MBT>
__global__ void __launch_bounds__(kBlock, MB) k_descriptor(EvalArgs<real> a)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    if ((int)blockIdx.x >= a.counts->n_items) return;
    const WorkItem it = a.items[blockIdx.x];
    const ModelDesc<real>& md = a.models[a.reqs[it.req].model];
    stage_params(md.params, reinterpret_cast<real*>(smem_raw), md.off.total);
    descriptor_item<real, NR, NA, KR, KA, RES, MBT>(a, it, smem_raw);
}

template <typename real, int NR, int NA, int KR, int KA, int RES, int MBT>
__device__ __forceinline__ void descriptor_item(const EvalArgs<real>& a, const WorkItem it, unsigned char* smem_raw)
{
    // MBT = 1: the four-body q4_n (l = 2) and five-body q5_n = q_n1^2 follow the
    // three-body descriptors (both always; a model with one of them has zero weights
    // on the other)
    constexpr int ND = NR + NA * (4 + 2 * MBT);
    constexpr int KRP = (KR + 3) & ~3;
    real* P = reinterpret_cast<real*>(smem_raw);
    const ReqInfo& rq = a.reqs[it.req];
    const ModelDesc<real> md = a.models[rq.model];
    const ParamLayout off = md.off;
    const int i = it.begin + threadIdx.x;
    if (i >= it.end) return;
    const int T = md.T, H = md.H;
    const real len[3] = {(real)rq.g.len[0], (real)rq.g.len[1], (real)rq.g.len[2]};
    const PosRec<real> ri = a.rec[i];
    const int ti = ri.t;
    real q[ND];
#pragma unroll
    for (int v = 0; v < ND; ++v) q[v] = real(0);

    // ---- radial descriptors (Eq. 3, 6-8) ----
    const int cR = min(a.cntR[i], a.mnR);
    if (T == 1) {
        // one pair type: q_n = sum_k c_nk (sum_j f_k(r_ij)), contracted once per bead;
        // the pair sums are kept as eight partial sums, four at a time (see walk_half)
        const real inv_rc = P[off.rcRi], inv_lo = P[off.rcRl];
        real fs[KR], hs = real(0);
#pragma unroll
        for (int k = 0; k < KR; ++k) fs[k] = real(0);
#pragma unroll 1
        for (int first = 0; first < 8; first += 4) {
            real fp[4][KR], hp[4];
#pragma unroll
            for (int p = 0; p < 4; ++p) {
                hp[p] = real(0);
#pragma unroll
                for (int k = 0; k < KR; ++k) fp[p][k] = real(0);
            }
            walk_half(a.nlR + i, (size_t)a.n, cR, first, [&](uint32_t e, int p) {
                const PosRec<real> rj = a.rec[e & kJMask];
                real dx, dy, dz;
                pair_vec(len, ri, rj, e, dx, dy, dz);
                const real r2 = norm2(dx, dy, dz);
                const real r = r2 * rsqrt_r(r2);
                basis_acc<real, KR>(r, inv_rc, inv_lo, fp[p], hp[p]);
            });
            hs += (hp[0] + hp[1]) + (hp[2] + hp[3]);
#pragma unroll
            for (int k = 0; k < KR; ++k) fs[k] += (fp[0][k] + fp[1][k]) + (fp[2][k] + fp[3][k]);
        }
#pragma unroll
        for (int k = 0; k < KR; ++k) fs[k] += hs;
        const real* c = P + off.cR;
#pragma unroll
        for (int nn = 0; nn < NR; ++nn) {
            real g = real(0);
#pragma unroll
            for (int k = 0; k < KR; ++k) g += c[nn * KR + k] * fs[k];
            const real* cl = P + off.cRl;  // plus the coefficients' FP32 rounding residuals
            real gl = real(0);
#pragma unroll
            for (int k = 0; k < KR; ++k) gl += cl[nn * KR + k] * fs[k];
            q[nn] = g + gl;
        }
    } else {
#pragma unroll 1
        for (int first = 0; first < 8; first += 4) {  // eight partial sums, four at a time (see walk_half)
            real qp[4][NR];
#pragma unroll
            for (int p = 0; p < 4; ++p)
#pragma unroll
                for (int nn = 0; nn < NR; ++nn) qp[p][nn] = real(0);
            walk_half(a.nlR + i, (size_t)a.n, cR, first, [&](uint32_t e, int p) {
                const PosRec<real> rj = a.rec[e & kJMask];
                real dx, dy, dz;
                pair_vec(len, ri, rj, e, dx, dy, dz);
                const real r2 = norm2(dx, dy, dz);
                const real r = r2 * rsqrt_r(r2);
                const int tp = ti * T + rj.t;
                real f[KR];
                basis<real, KR>(r, P[off.rcRi + tp], P[off.rcRl + tp], f);
                const real* c = P + off.cR + tp * coef_stride(NR, KR);
#pragma unroll
                for (int nn = 0; nn < NR; ++nn) {
                    real g = real(0);
#pragma unroll
                    for (int k = 0; k < KR; ++k) g += c[nn * KR + k] * f[k];
                    qp[p][nn] += g;
                }
            });
#pragma unroll
            for (int nn = 0; nn < NR; ++nn) q[nn] += (qp[0][nn] + qp[1][nn]) + (qp[2][nn] + qp[3][nn]);
        }
    }

    // ---- angular moments A_nlm (Eq. 5) ----
    real A[NA][kNLM];
#pragma unroll
    for (int nn = 0; nn < NA; ++nn)
#pragma unroll
        for (int k = 0; k < kNLM; ++k) A[nn][k] = real(0);
    const int cA = min(a.cntA[i], a.mnA);
    NbrWalk<real> wa(a.nlA, a.n, i, cA, a.rec);
    for (int s = 0; s < cA; ++s) {
        uint32_t e;
        PosRec<real> rj;
        wa.next(s, e, rj);
        real dx, dy, dz;
        pair_vec(len, ri, rj, e, dx, dy, dz);
        const real r2 = norm2(dx, dy, dz);
        const real inv_r = rsqrt_r(r2);
        const real r = r2 * inv_r;
        const int tp = ti * T + rj.t;
        real hf, t[KA];
        cheb_T<real, KA>(r, P[off.rcAi + tp], P[off.rcAl + tp], hf, t);
        real Y[kNLM];
        sh_eval(dx * inv_r, dy * inv_r, dz * inv_r, Y);
        const real* crow = P + off.cA + tp * coef_stride(NA, KA);
#pragma unroll
        for (int nn = 0; nn < NA; ++nn) {
            // one coefficient row at a time: the fence keeps the compiler from loading
            // every row up front, which would hold 32 more registers across the sums
            real cr[KA];
            load_coef(crow + nn * KA, T == 1 && KA % 4 == 0, cr);
            const real g = hf * cheb_sum(cr, t);
#pragma unroll
            for (int k = 0; k < kNLM; ++k) A[nn][k] += g * Y[k];
            asm volatile("" ::: "memory");
        }
    }
    // q_nl (Eq. 4)
#pragma unroll
    for (int nn = 0; nn < NA; ++nn)
#pragma unroll
        for (int k = 0; k < kNLM; ++k) q[NR + (l_of(k) - 1) * NA + nn] += A[nn][k] * A[nn][k];
    // four- and five-body terms; g4 keeps dq4/dA_n2m for the adjoint below
    real g4[MBT ? NA : 1][5];
    if constexpr (MBT == 1) {
#pragma unroll
        for (int nn = 0; nn < NA; ++nn) {
            q[NR + 4 * NA + nn] = four_body(&A[nn][3], g4[nn]);
            q[NR + 5 * NA + nn] = q[NR + nn] * q[NR + nn];
        }
    }

    // ---- network (Eq. 2) and dU/dq ----
    real U;
    real dq[ND];
    {
        // The FP32 form adds the parameters' rounding residuals (tables ...l) in
        // separate accumulators, so the energy is that of the caller's FP64 weights;
        // the gradient (forces, whose tolerance is far looser) uses the FP32 weights.
        // BF16 weights W0 are FP32 numbers already and have no residual table.
        constexpr bool res0 = RES == 1;
        const real* b0 = P + off.b0 + ti * H;
        const real* w1 = P + off.w1 + ti * H;
        const real* b0l = P + off.b0l + ti * H;
        const real* w1l = P + off.w1l + ti * H;
        U = -P[off.b1 + ti];
        real Ul = -P[off.b1l + ti];
#pragma unroll
        for (int v = 0; v < ND; ++v) dq[v] = real(0);
        if (T == 1) {
            // one type: W0 rows padded to a multiple of 4 and 16-byte aligned, read as
            // vectors once per hidden unit and kept for the gradient (every lane reads
            // the same row, a broadcast)
            constexpr int NDV = (ND + 3) & ~3;
            const real* w0 = P + off.w0;
            const real* w0l = P + (res0 ? off.w0l : off.w0);
            for (int mu = 0; mu < H; ++mu) {
                real w[NDV];
                loadN<real, NDV>(w0 + mu * NDV, w);
                real x = -b0[mu];
#pragma unroll
                for (int v = 0; v < ND; ++v) x += w[v] * q[v];
                real xl = -b0l[mu];  // the residual row four entries at a time (vector loads)
                if constexpr (res0)
#pragma unroll
                    for (int v4 = 0; v4 < NDV; v4 += 4) {
                        real wl[4];
                        load4(w0l + mu * NDV + v4, wl);
#pragma unroll
                        for (int u = 0; u < 4; ++u)
                            if (v4 + u < ND) xl += wl[u] * q[v4 + u];
                    }
                x += xl;
                const real h = tanh_r(x);
                U += w1[mu] * h;
                Ul += w1l[mu] * h;
                const real coef = w1[mu] * fma(-h, h, real(1));
#pragma unroll
                for (int v = 0; v < ND; ++v) dq[v] += coef * w[v];
            }
        } else {
            // several types: unpadded rows (padded ones put the rows that lanes of
            // different types read at once into the same shared-memory banks)
            const real* w0 = P + off.w0 + ti * H * ND;
            const real* w0l = P + (res0 ? off.w0l : off.w0) + ti * H * ND;
            for (int mu = 0; mu < H; ++mu) {
                real x = -b0[mu];
#pragma unroll
                for (int v = 0; v < ND; ++v) x += w0[mu * ND + v] * q[v];
                real xl = -b0l[mu];
                if constexpr (res0)
#pragma unroll
                    for (int v = 0; v < ND; ++v) xl += w0l[mu * ND + v] * q[v];
                x += xl;
                const real h = tanh_r(x);
                U += w1[mu] * h;
                Ul += w1l[mu] * h;
                const real coef = w1[mu] * fma(-h, h, real(1));
#pragma unroll
                for (int v = 0; v < ND; ++v) dq[v] += coef * w0[mu * ND + v];
            }
        }
        U += Ul;
    }
    a.U[i] = U;
    // e_i^t[k] = sum_n dU/dq_n c^{t_i t}_{nk}
    real* ei = a.e + (size_t)i * a.e_stride;
    for (int t = 0; t < T; ++t) {
        const real* c = P + off.cR + (ti * T + t) * coef_stride(NR, KR);
#pragma unroll
        for (int k = 0; k < KRP; ++k) {
            real v = real(0);
            if (k < KR) {
#pragma unroll
                for (int nn = 0; nn < NR; ++nn) v += dq[nn] * c[nn * KR + k];
            }
            ei[t * KRP + k] = v;
        }
    }
    if constexpr (MBT == 1) {
        // dq5/dA_n1m = 2 q_n1 dq_n1/dA_n1m: fold into the l = 1 coefficient
#pragma unroll
        for (int nn = 0; nn < NA; ++nn) dq[NR + nn] = fma(real(2) * q[NR + nn], dq[NR + 5 * NA + nn], dq[NR + nn]);
    }
    // Phi_nlm in place of A_nlm, in registers; then the angular pairs' forces
    // in scatter form (f_ij from Phi_i alone) while Phi_i is still here
#pragma unroll
    for (int k = 0; k < kNLM; ++k)
#pragma unroll
        for (int nn = 0; nn < NA; ++nn) {
            real v = real(2) * dq[NR + (l_of(k) - 1) * NA + nn] * A[nn][k];
            if constexpr (MBT == 1)
                if (k >= 3 && k < 8) v = fma(dq[NR + 4 * NA + nn], g4[nn][k - 3], v);
            A[nn][k] = v;
        }
    // each P_n = sum_k Phi_nk Y_k in its sphere-reduced form (see sh_red_eval)
    real Psi[NA][kShRed];
#pragma unroll
    for (int nn = 0; nn < NA; ++nn) sh_reduce(A[nn], Psi[nn]);
    ForceCtx<real, KRP> c;
    c.i = i;
    c.T = T;
    c.ri = ri;
    c.ti = ti;
#pragma unroll
    for (int k = 0; k < 3; ++k) c.len[k] = len[k];
#pragma unroll
    for (int k = 0; k < 3; ++k) c.F[k] = real(0);
#pragma unroll
    for (int k = 0; k < 9; ++k) c.W[k] = real(0);
    const bool per_bead = a.virial != nullptr;
    force_angular_phi_reg<real, NA, KA>(a, P, off, Psi, c, per_bead);
    // F_i's angular part into i's line; the thread's angular virial sum (what
    // the totals use, with or without per-particle virials) as plain stores
    unsigned long long* acc_i = a.accF + (size_t)i * 4;
#pragma unroll
    for (int p = 0; p < 3; ++p) fix_add(acc_i + p, c.F[p]);
#pragma unroll
    for (int k = 0; k < 9; ++k) a.wsum[(size_t)k * a.n + i] = c.W[k];
}

// Radial pairs:
//   f_ij = (e_i^{t_j} . f') u,  f_ji = -(e_j^{t_i} . f') u,  F_i += f_ij - f_ji,
//   W_i += r_ij (x) f_ji.  The pair body has no branch, so the scheduler can
//   interleave the bodies of each walk step.  f_ji is parallel to r_ij, so the
//   radial terms of W_i are symmetric: c.W[0..5] holds xx, yy, zz, xy, xz, yz of the
//   radial part alone (6 products per pair instead of 9).
template <typename real, int NR, int KR, int CH>
__device__ __forceinline__ void force_radial(const EvalArgs<real>& a, const real* P, const ParamLayout& off,
                                             ForceCtx<real, (KR + 3) & ~3>& c)
{
    constexpr int KRP = (KR + 3) & ~3;
    const real* e_i = a.e + (size_t)c.i * a.e_stride;
    const int cnt = min(a.cntR[c.i], a.mnR);
    const int T = c.T, ti = c.ti;
    auto radial_pair = [&](uint32_t e, const real* eij) {
        const int j = (int)(e & kJMask);
        const PosRec<real> rj = a.rec[j];
        real eji[KRP];
        load_grad<real, KRP>(a.e + (size_t)j * a.e_stride + ti * KRP, eji);
        real dx, dy, dz;
        pair_vec(c.len, c.ri, rj, e, dx, dy, dz);
        const real r2 = norm2(dx, dy, dz);
        const real inv_r = rsqrt_r(r2);
        const real r = r2 * inv_r;
        real f[KR], df[KR];
        basis_d<real, KR>(r, P[off.rcRi + ti * T + rj.t], P[off.rcRl + ti * T + rj.t], f, df);
        real ai = real(0), bj = real(0);
#pragma unroll
        for (int k = 0; k < KR; ++k) {
            ai += eij[k] * df[k];
            bj += eji[k] * df[k];
        }
        const real ux = dx * inv_r, uy = dy * inv_r, uz = dz * inv_r;
        const real fs = ai + bj;
        c.F[0] += fs * ux;
        c.F[1] += fs * uy;
        c.F[2] += fs * uz;
        const real w = bj * inv_r;
        const real wx = w * dx, wy = w * dy, wz = w * dz;
        c.W[0] -= wx * dx;
        c.W[1] -= wy * dy;
        c.W[2] -= wz * dz;
        c.W[3] -= wx * dy;
        c.W[4] -= wx * dz;
        c.W[5] -= wy * dz;
    };
    const uint32_t* nl = a.nlR + c.i;
    const size_t stride = (size_t)a.n;
    if (T == 1) {
        real ei1[KRP];  // the one partner type's vector
        load_grad<real, KRP>(e_i, ei1);
        walk_chunk<CH>(nl, stride, cnt, [&](uint32_t e) { radial_pair(e, ei1); });
    } else {
        walk_chunk<CH>(nl, stride, cnt, [&](uint32_t e) {
            real eij[KRP];
            load_grad<real, KRP>(e_i + a.rec[e & kJMask].t * KRP, eij);
            radial_pair(e, eij);
        });
    }
}

// ---- angular pairs in scatter form inside the descriptor kernel ------------------
// Each ordered angular pair is evaluated once, by the thread of its centre i, from
// Phi_i alone while it is still in registers: f_ij = dU_i/dr_ij.  F_i gains f_ij
// in registers; F_j loses it (and W_j gains r_ji (x) f_ij) through the fixed-point
// atomic adds.  For A = g(r) Y(u), u = r / |r|, the gradient with respect to r is
//   dA/dr = g' Y(u) u + (g / r) (grad Y(u) - (u . grad Y(u)) u),
// where grad Y may be the gradient of any function equal to Y on the unit sphere
// (only its surface part enters).  Summed over the components with
// P_n = sum_k Phi_nk Y_k:
//   f_ij = (sum_n g_n' P_n(u)) u + (ga - (u . ga) u) / r,   ga = sum_n g_n grad P_n(u),
// evaluated from each P_n's sphere-reduced form Psi_n (sh_red_eval).
template <typename real, int NA, int KA, typename Ctx>
__device__ __forceinline__ void force_angular_phi_reg(const EvalArgs<real>& a, const real* P, const ParamLayout& off,
                                                      const real (&Psi)[NA][kShRed], Ctx& c, bool per_bead)
{
    const int T = c.T, ti = c.ti;
    const int cA = min(a.cntA[c.i], a.mnA);
    NbrWalk<real> wa(a.nlA, a.n, c.i, cA, a.rec);
    for (int s = 0; s < cA; ++s) {
        uint32_t e;
        PosRec<real> rj;
        wa.next(s, e, rj);
        const int j = (int)(e & kJMask);
        real dx, dy, dz;
        pair_vec(c.len, c.ri, rj, e, dx, dy, dz);
        const real r2 = norm2(dx, dy, dz);
        const real inv_r = rsqrt_r(r2);
        const real r = r2 * inv_r;
        const int tij = ti * T + rj.t;
        real hf, hdf, hdx, t[KA], dt[KA];
        cheb_dT<real, KA>(r, P[off.rcAi + tij], P[off.rcAl + tij], hf, hdf, hdx, t, dt);
        real g[NA], dg[NA];
        const real* crow = P + off.cA + tij * coef_stride(NA, KA);
#pragma unroll
        for (int nn = 0; nn < NA; ++nn) {
            real cr[KA];  // one row at a time (see the angular moments)
            load_coef(crow + nn * KA, T == 1 && KA % 4 == 0, cr);
            cheb_g_dg(cr, t, dt, hf, hdf, hdx, g[nn], dg[nn]);
            asm volatile("" ::: "memory");
        }
        const real ux = dx * inv_r, uy = dy * inv_r, uz = dz * inv_r;
        real D = real(0);
        real ga[3] = {real(0), real(0), real(0)};
#pragma unroll
        for (int nn = 0; nn < NA; ++nn) {
            real v, vx, vy, vz;
            sh_red_eval(Psi[nn], ux, uy, uz, v, vx, vy, vz);
            D += dg[nn] * v;
            ga[0] += g[nn] * vx;
            ga[1] += g[nn] * vy;
            ga[2] += g[nn] * vz;
        }
        real fij[3];
        angular_force(D, ga, ux, uy, uz, inv_r, fij);
        unsigned long long* acc_j = a.accF + (size_t)j * 4;
#pragma unroll
        for (int p = 0; p < 3; ++p) {
            c.F[p] += fij[p];
            fix_add(acc_j + p, -fij[p]);
        }
        // W_j += r_ji (x) f_ij; each product is rounded on its own, so the thread's
        // sum (the totals) is the same whether or not it is also scattered
        const real d[3] = {dx, dy, dz};
        unsigned long long* accw_j = per_bead ? a.accW + (size_t)j * 12 : nullptr;
#pragma unroll
        for (int p = 0; p < 3; ++p)
#pragma unroll
            for (int q = 0; q < 3; ++q) {
                const real w = mul_rn(-d[p], fij[q]);
                c.W[3 * p + q] += w;
                if (per_bead) fix_add(accw_j + 3 * p + q, w);
            }
    }
}

// Radial pairs in gather form, then i's outputs.  By the time this kernel runs the
// descriptor kernel has finished every scatter, so i's fixed-point line holds the
// angular part of F_i (its own and what its neighbours sent) and of W_i (per-particle
// virials), or the thread's angular virial sum (totals only).  The kernel adds the
// radial part, writes the caller-order FP64 outputs, clears the line for the next
// evaluation, and reduces E and W in FP64 (Eq. 1, 16).
// MB: resident blocks per SM (a register budget); CH: neighbour entries per walk
// group (4 or 8), both chosen per configuration by the autotuner.
template <typename real, int NR, int KR, int MB, int CH>
__global__ void __launch_bounds__(kBlock, MB) k_force_radial(EvalArgs<real> a)
{
    constexpr int KRP = (KR + 3) & ~3;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    real* P = reinterpret_cast<real*>(smem_raw);
    const int w = blockIdx.x;  // one work item per block (see k_descriptor)
    if (w >= a.counts->n_items) return;
    const WorkItem it = a.items[w];
    const ReqInfo& rq = a.reqs[it.req];
    const ModelDesc<real> md = a.models[rq.model];
    const ParamLayout off = md.off;
    const int i = it.begin + threadIdx.x;
    stage_params(md.params, P, off.n_cut_coef);
    double tot[10];
#pragma unroll
    for (int k = 0; k < 10; ++k) tot[k] = 0.0;
    if (i < it.end) {
        ForceCtx<real, KRP> c;
        c.i = i;
        c.T = md.T;
        c.ri = a.rec[i];
        c.ti = c.ri.t;
        for (int k = 0; k < 3; ++k) c.len[k] = (real)rq.g.len[k];
#pragma unroll
        for (int k = 0; k < 3; ++k) c.F[k] = real(0);
#pragma unroll
        for (int k = 0; k < 9; ++k) c.W[k] = real(0);
        force_radial<real, NR, KR, CH>(a, P, off, c);
        // the radial virial in full (row-major 3 x 3) from its symmetric part
        const real Wr[9] = {c.W[0], c.W[3], c.W[4], c.W[3], c.W[1], c.W[5], c.W[4], c.W[5], c.W[2]};
        ulonglong2* line = reinterpret_cast<ulonglong2*>(a.accF + (size_t)i * 4);
        const ulonglong2 f01 = line[0], f2x = line[1];
        line[0] = line[1] = make_ulonglong2(0ull, 0ull);
        const int ui = a.perm[i];
        const int lu = ui - rq.begin;
        const bool out_ok = lu >= 0 && lu < rq.n;  // see kErrCellList
        if (!out_ok && a.err) atomicOr(a.err, kErrCellList);
        double* fo = a.force + (size_t)3 * rq.begin + lu;
        // F_i: the angular part from the fixed-point line plus the radial part, added in
        // the working precision and widened once (FP64 arithmetic is scarce)
        double Fi[3] = {(double)(fix_value_f(f01.x) + c.F[0]), (double)(fix_value_f(f01.y) + c.F[1]),
                        (double)(fix_value_f(f2x.x) + c.F[2])};
        if (out_ok) {
            fo[0] = Fi[0];
            fo[rq.n] = Fi[1];
            fo[(size_t)2 * rq.n] = Fi[2];
            if (a.kick_vel) closing_kick(a, rq, ui, lu, Fi);
        }
        if (a.virial) {  // W_i: the angular terms its neighbours sent, plus its radial terms
            ulonglong2* wl = reinterpret_cast<ulonglong2*>(a.accW + (size_t)i * 12);
            double* vo = a.virial + (size_t)9 * rq.begin + lu;
#pragma unroll
            for (int q = 0; q < 5; ++q) {
                const ulonglong2 v = wl[q];
                wl[q] = make_ulonglong2(0ull, 0ull);
                if (out_ok) {
                    vo[(size_t)(2 * q) * rq.n] = (double)(fix_value_f(v.x) + Wr[2 * q]);
                    if (2 * q + 1 < 9) vo[(size_t)(2 * q + 1) * rq.n] = (double)(fix_value_f(v.y) + Wr[2 * q + 1]);
                }
            }
        }
        const real Ui = a.U[i];
        if (a.site && out_ok) a.site[ui] = (double)Ui;
        tot[0] = (double)Ui;
        // i's contribution to the virial total: its angular sum plus its radial terms,
        // added in the working precision and widened once (FP64 arithmetic is scarce)
#pragma unroll
        for (int k = 0; k < 9; ++k) tot[1 + k] = (double)(a.wsum[(size_t)k * a.n + i] + Wr[k]);
    }
    reduce_totals<kBlock>(tot, w, it, rq, a.partial, a.gcounter, a.counter, a.counts, a.totals);
}

// ---- shape dispatch -----------------------------------------------------------
template <typename real>
bool evaluate_shape_supported(int nR, int nA, int KR, int KA)
{
#define NEP_CASE(a_, b_, c_, d_) \
    if (nR == a_ && nA == b_ && KR == c_ && KA == d_) return true;
    NEP_SHAPES(NEP_CASE)
#undef NEP_CASE
    return false;
}

// The descriptor kernel with the angular forces fused (K1) and the radial / output
// kernel (K2).  Variants: resident blocks per SM (register caps), for the descriptor
// the residual rows of W0 (RES) and the many-body terms (MBT), for the radial kernel the
// walk chunk.
template <int A_, int B_, int C_, int D_>
static cudaError_t set_smem(size_t smem_desc, size_t smem_force)
{
    cudaError_t e = cudaSuccess;
    auto set = [&](auto* kernel, size_t smem) {
        if (e == cudaSuccess)
            e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    };
    set(k_descriptor<float, A_, B_, C_, D_, 2, 0, 0>, smem_desc);
    set(k_descriptor<float, A_, B_, C_, D_, 2, 0, 1>, smem_desc);
    set(k_descriptor<float, A_, B_, C_, D_, 2, 1, 0>, smem_desc);
    set(k_descriptor<float, A_, B_, C_, D_, 2, 1, 1>, smem_desc);
    set(k_descriptor<float, A_, B_, C_, D_, 3, 0, 0>, smem_desc);
    set(k_descriptor<float, A_, B_, C_, D_, 3, 0, 1>, smem_desc);
    set(k_descriptor<float, A_, B_, C_, D_, 3, 1, 0>, smem_desc);
    set(k_descriptor<float, A_, B_, C_, D_, 3, 1, 1>, smem_desc);
    set(k_force_radial<float, A_, C_, 3, 4>, smem_force);
    set(k_force_radial<float, A_, C_, 3, 8>, smem_force);
    set(k_force_radial<float, A_, C_, 4, 4>, smem_force);
    set(k_force_radial<float, A_, C_, 4, 8>, smem_force);
    set(k_force_radial<float, A_, C_, 5, 4>, smem_force);
    set(k_force_radial<float, A_, C_, 5, 8>, smem_force);
    return e;
}

template <typename real>
cudaError_t evaluate_set_smem(int nR, int nA, int KR, int KA, size_t smem_desc, size_t smem_force)
{
    const cudaError_t e = group_set_smem<real>();
    if (e != cudaSuccess || sizeof(real) == 8) return e;
#define NEP_CASE(a_, b_, c_, d_) \
    if (nR == a_ && nA == b_ && KR == c_ && KA == d_) return set_smem<a_, b_, c_, d_>(smem_desc, smem_force);
    NEP_SHAPES(NEP_CASE)
#undef NEP_CASE
    return cudaErrorInvalidValue;
}

template <int NR, int NA, int KR, int KA, int MBT>
static cudaError_t launch_descriptor(const EvalArgs<float>& a, int nb, size_t smem, cudaStream_t st, int mb_desc)
{
    if (a.w0_residual) {
        if (mb_desc == 2) return launch_k(k_descriptor<float, NR, NA, KR, KA, 2, 1, MBT>, nb, kBlock, smem, st, a);
        return launch_k(k_descriptor<float, NR, NA, KR, KA, 3, 1, MBT>, nb, kBlock, smem, st, a);
    }
    if (mb_desc == 2) return launch_k(k_descriptor<float, NR, NA, KR, KA, 2, 0, MBT>, nb, kBlock, smem, st, a);
    return launch_k(k_descriptor<float, NR, NA, KR, KA, 3, 0, MBT>, nb, kBlock, smem, st, a);
}

// The radial kernel in its (blocks per SM, walk chunk) variant.
template <int NR, int KR>
static cudaError_t launch_force_radial(const EvalArgs<float>& a, int nb, size_t smem, cudaStream_t st, int mb, int ch)
{
    if (ch == 8) {
        if (mb == 5) return launch_k(k_force_radial<float, NR, KR, 5, 8>, nb, kBlock, smem, st, a);
        if (mb == 4) return launch_k(k_force_radial<float, NR, KR, 4, 8>, nb, kBlock, smem, st, a);
        return launch_k(k_force_radial<float, NR, KR, 3, 8>, nb, kBlock, smem, st, a);
    }
    if (mb == 5) return launch_k(k_force_radial<float, NR, KR, 5, 4>, nb, kBlock, smem, st, a);
    if (mb == 4) return launch_k(k_force_radial<float, NR, KR, 4, 4>, nb, kBlock, smem, st, a);
    return launch_k(k_force_radial<float, NR, KR, 3, 4>, nb, kBlock, smem, st, a);
}

template <typename real>
cudaError_t launch_evaluate(int nR, int nA, int KR, int KA, const EvalArgs<real>& a, int items_cap, bool by_groups,
                            size_t smem_desc, size_t smem_force, cudaStream_t st, cudaEvent_t mid, int mb_desc,
                            int mb_force, int ch_force)
{
    if (by_groups) return launch_evaluate_group<real>(nR, nA, KR, KA, a, items_cap, st, mid);
    if constexpr (sizeof(real) == 4) {
        if (!a.accF || !a.wsum) return cudaErrorInvalidValue;  // the FP32 form scatters into a.accF
        const int nb = items_cap;
#define NEP_CASE(a_, b_, c_, d_)                                                                        \
    if (nR == a_ && nA == b_ && KR == c_ && KA == d_) {                                                 \
        cudaError_t e = a.many_body ? launch_descriptor<a_, b_, c_, d_, 1>(a, nb, smem_desc, st, mb_desc) \
                                    : launch_descriptor<a_, b_, c_, d_, 0>(a, nb, smem_desc, st, mb_desc); \
        if (e != cudaSuccess) return e;                                                                 \
        if (mid && (e = cudaEventRecord(mid, st)) != cudaSuccess) return e;                             \
        return launch_force_radial<a_, c_>(a, nb, smem_force, st, mb_force, ch_force);                  \
    }
        NEP_SHAPES(NEP_CASE)
#undef NEP_CASE
    }
    return cudaErrorInvalidValue;
}

#define NEP_INSTANTIATE(real)                                                                             \
    template bool evaluate_shape_supported<real>(int, int, int, int);                                     \
    template cudaError_t evaluate_set_smem<real>(int, int, int, int, size_t, size_t);                     \
    template cudaError_t launch_evaluate<real>(int, int, int, int, const EvalArgs<real>&, int, bool, size_t, size_t, \
                                               cudaStream_t, cudaEvent_t, int, int, int);
NEP_INSTANTIATE(float)
NEP_INSTANTIATE(double)
#undef NEP_INSTANTIATE

}  // namespace nep

// Evaluation kernels with a group of kG lanes per particle, for batches that leave the
// thread-per-particle kernels of evaluate.cu most of the chip idle, and for every FP64
// evaluation.  Same steps, in two kernels:
//   k_descriptor_group  descriptors, network, gradients, and each angular pair's f_ij
//                       while the particle's adjoint is at hand
//   k_force_group       radial pairs in gather form, the angular parts, outputs, totals
//
// What bounds the thread-per-particle kernels on a few thousand particles is one
// thread's serial work: a block of 128 particles takes the same time alone on an SM
// (FP32 water: 52 us descriptor, 30 us radial) as three of them do.  Here the lanes of a
// group take one pair each, so a particle's pairs are evaluated kG at a time:
//   - radial descriptors: lane l sums the pairs of the slots l, l + kG, ...; the kG
//     partial sums are added pairwise by shuffles;
//   - angular moments: a lane writes its pair's g_n and Y_lm as one row of a shared tile,
//     then every lane adds all rows, in slot order, to its 12 of the 96 moments;
//   - network: a lane takes every kG-th hidden unit, then its share of the gradient's
//     components over all hidden units in order;
//   - pair forces: one pair per lane; FP32 components are summed in slot order through the
//     tile.
// Every FP32 sum is formed in the order in which evaluate.cu forms it, so a request gives
// the same bits whichever kernels its batch takes.  A particle's state lives in its
// lanes' registers and 1.4 KB (FP32) of shared memory instead of some 200 registers of one
// thread, which also is what makes this the better form in FP64 at every size: one thread
// per particle spills there.
//
// FP64 angular pairs: the descriptor kernel stores f_ij per list slot, and the force kernel
// takes f_ij from i's slot and f_ji from the slot of j's list that holds i (found by
// comparing list words), so each ordered pair is evaluated once.  FP64 arithmetic runs
// at 1/64 of the FP32 rate here, the search at the full rate.
#include "evaluate_math.cuh"

namespace nep {

constexpr int kG = kGroupLanes;      // lanes per particle
constexpr int kGP = kBlock / kG;     // particles per block
constexpr unsigned kFull = 0xffffffffu;
static_assert(kG == 8, "the radial partial sums of evaluate.cu follow the slot number mod 8");

// Shared memory of one group (reals): a tile of kG rows (one pair each), then n_A rows of
// 28 (moments, adjoint, reduced coefficients).  Rows are an odd multiple of four reals
// long, so that the lanes' 16-byte row writes fall into distinct banks; a group's size is
// 8 mod 32, so that the four groups of a warp read distinct banks.
template <int NA>
struct GroupTile {
    static constexpr int GS = (NA + 3) & ~3;
    static constexpr int ROW = (GS + 24) / 4 % 2 ? GS + 24 : GS + 28;
    static constexpr int PSI = 28;
    static constexpr int TILE = kG * ROW;
    static constexpr int USED = TILE + NA * PSI + 16;  // and PairFrame's table
    static constexpr int SIZE = (USED + 23) / 32 * 32 + 8;
    static_assert(SIZE >= USED, "group size");
};

template <typename real>
__device__ __forceinline__ void store4(real* p, real a, real b, real c, real d);
template <>
__device__ __forceinline__ void store4<float>(float* p, float a, float b, float c, float d)
{
    *reinterpret_cast<float4*>(p) = make_float4(a, b, c, d);
}
template <>
__device__ __forceinline__ void store4<double>(double* p, double a, double b, double c, double d)
{
    reinterpret_cast<double2*>(p)[0] = make_double2(a, b);
    reinterpret_cast<double2*>(p)[1] = make_double2(c, d);
}

// The sum over the group's lanes, ((0+1)+(2+3))+((4+5)+(6+7)), in every lane.
template <typename real>
__device__ __forceinline__ real group_sum(real v)
{
#pragma unroll
    for (int o = 1; o < kG; o <<= 1) v += __shfl_xor_sync(kFull, v, o);
    return v;
}

// Pair vectors of one particle.  FP64: r_i moved by the five possible cell offsets per axis,
// looked up in shared memory, so that a component is one subtraction (the conversion of the
// offset and the multiply-add would each cost as much on the FP64 pipe).
template <typename real>
struct PairFrame;
template <>
struct PairFrame<float> {
    float len[3];
    PosRec<float> ri;
    __device__ __forceinline__ PairFrame(const CellGrid& g, const PosRec<float>& r, float*, int) : ri(r)
    {
#pragma unroll
        for (int k = 0; k < 3; ++k) len[k] = (float)g.len[k];
    }
    __device__ __forceinline__ void vec(const PosRec<float>& rj, uint32_t e, float& dx, float& dy, float& dz) const
    {
        pair_vec(len, ri, rj, e, dx, dy, dz);
    }
};
template <>
struct PairFrame<double> {
    const double* moved;  // [3][5]
    __device__ __forceinline__ PairFrame(const CellGrid& g, const PosRec<double>& r, double* table, int lane)
        : moved(table)
    {
        if (lane < 5) {
            const double d = (double)(2 - lane);
            table[lane] = fma(d, g.len[0], r.x);
            table[5 + lane] = fma(d, g.len[1], r.y);
            table[10 + lane] = fma(d, g.len[2], r.z);
        }
        __syncwarp();
    }
    __device__ __forceinline__ void vec(const PosRec<double>& rj, uint32_t e, double& dx, double& dy, double& dz) const
    {
        const uint32_t code = e >> kJBits;
        dx = rj.x - moved[code & 7u];
        dy = rj.y - moved[5 + ((code >> 3) & 7u)];
        dz = rj.z - moved[10 + ((code >> 6) & 7u)];
    }
};

// A pair's geometry from the list entry.
template <typename real>
struct Pair {
    real dx, dy, dz, inv_r, r;
    int j, tj;
};
template <typename real>
__device__ __forceinline__ Pair<real> make_pair(const PairFrame<real>& frame, const PosRec<real>& rj, uint32_t e)
{
    Pair<real> p;
    p.j = (int)(e & kJMask);
    p.tj = rj.t;
    frame.vec(rj, e, p.dx, p.dy, p.dz);
    const real r2 = norm2(p.dx, p.dy, p.dz);
    p.inv_r = rsqrt_r(r2);
    p.r = r2 * p.inv_r;
    return p;
}

template <typename real, int NR, int NA, int KR, int KA, int RES, int MBT>
__global__ void __launch_bounds__(kBlock, sizeof(real) == 4 ? 4 : 3) k_descriptor_group(EvalArgs<real> a)
{
    using GT = GroupTile<NA>;
    constexpr int ND = NR + NA * (4 + 2 * MBT);
    constexpr int NDV = (ND + 3) & ~3;
    constexpr int KRP = (KR + 3) & ~3;
    constexpr bool kF32 = sizeof(real) == 4;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int item = (int)blockIdx.x / kG;
    if (item >= a.counts->n_items) return;
    const WorkItem it = a.items[item];
    const int first = it.begin + ((int)blockIdx.x % kG) * kGP;
    if (first >= it.end) return;
    const ReqInfo& rq = a.reqs[it.req];
    const ModelDesc<real> md = a.models[rq.model];
    const ParamLayout off = md.off;
    const real* __restrict__ P = md.params;  // read through L1: a block has too few particles to stage the tables for
    const int T = md.T, H = md.H;
    const int gl = (int)threadIdx.x % kG, grp = (int)threadIdx.x / kG;
    real* tile = reinterpret_cast<real*>(smem_raw) + grp * GT::SIZE;
    real* psi = tile + GT::TILE;
    // groups past the item's end follow its last particle with empty lists and write nothing
    const bool live = first + grp < it.end;
    const int i = live ? first + grp : it.end - 1;
    const PosRec<real> ri = a.rec[i];
    const PairFrame<real> frame(rq.g, ri, psi + NA * GT::PSI, gl);
    const int ti = ri.t;
    const int cR = live ? min(a.cntR[i], a.mnR) : 0, cA = live ? min(a.cntA[i], a.mnA) : 0;
    const size_t n = (size_t)a.n;

    // the network's scratch lies over the tile: q [40], coef [32], h [32], columns [40]
    real* sq = tile;
    real* scoef = tile + 40;
    real* sh = tile + 72;
    real* sdq = tile + 104;
    static_assert(GT::TILE >= 144 && ND + 2 <= 40, "network scratch");

    // ---- radial descriptors (Eq. 3, 6-8) ----
    real q_own = real(0);  // q_n of lane n < NR
    static_assert(NR <= kG, "a lane per radial descriptor");
    {
        const uint32_t* nl = a.nlR + (size_t)gl * n + i;
        const int cl = (cR - gl + kG - 1) / kG;  // this lane's slots (none: <= 0)
        if (T == 1) {
            real f[KR], hs = real(0);
#pragma unroll
            for (int k = 0; k < KR; ++k) f[k] = real(0);
            const real inv_rc = P[off.rcRi], inv_lo = P[off.rcRl];
            walk4(nl, kG * n, cl, [&](uint32_t e) {
                const Pair<real> p = make_pair(frame, a.rec[e & kJMask], e);
                basis_acc<real, KR>(p.r, inv_rc, inv_lo, f, hs);
            });
            hs = group_sum(hs);
#pragma unroll
            for (int k = 0; k < KR; ++k) f[k] = group_sum(f[k]) + hs;
            // lane n has row n
            const int nn = min(gl, NR - 1);
            const real* c = P + off.cR + nn * KR;
            real g = real(0);
#pragma unroll
            for (int k = 0; k < KR; ++k) g = fma(c[k], f[k], g);
            if constexpr (kF32) {
                const real* cl_ = P + off.cRl + nn * KR;
                real gl_ = real(0);
#pragma unroll
                for (int k = 0; k < KR; ++k) gl_ = fma(cl_[k], f[k], gl_);
                g += gl_;
            }
            q_own = g;
        } else {
            real qr[NR];
#pragma unroll
            for (int nn = 0; nn < NR; ++nn) qr[nn] = real(0);
            walk4(nl, kG * n, cl, [&](uint32_t e) {
                const Pair<real> p = make_pair(frame, a.rec[e & kJMask], e);
                const int tp = ti * T + p.tj;
                real f[KR];
                basis<real, KR>(p.r, P[off.rcRi + tp], P[off.rcRl + tp], f);
                const real* c = P + off.cR + tp * coef_stride(NR, KR);
#pragma unroll
                for (int nn = 0; nn < NR; ++nn) {
                    real g = real(0);
#pragma unroll
                    for (int k = 0; k < KR; ++k) g = fma(c[nn * KR + k], f[k], g);
                    qr[nn] += g;
                }
            });
#pragma unroll
            for (int nn = 0; nn < NR; ++nn) {
                qr[nn] = group_sum(qr[nn]);
                if (gl == nn) q_own = qr[nn];
            }
        }
    }

    // ---- angular moments A_nlm (Eq. 5): this lane's chunks gl + kG m of four moments ----
    constexpr int CHUNKS = NA * 6, CH = (CHUNKS + kG - 1) / kG;
    real acc[CH][4];
#pragma unroll
    for (int m = 0; m < CH; ++m)
#pragma unroll
        for (int u = 0; u < 4; ++u) acc[m][u] = real(0);
    const int most = __reduce_max_sync(kFull, cA);  // of the warp's four particles
    const uint32_t* nla = a.nlA + i;
    {
        uint32_t e = gl < cA ? nla[(size_t)gl * n] : 0u;
        PosRec<real> rj = a.rec[e & kJMask];
        for (int s0 = 0; s0 < most; s0 += kG) {
            const bool ok = s0 + gl < cA;
            real* row = tile + gl * GT::ROW;
            const uint32_t ec = e;
            const PosRec<real> rc = rj;
            e = s0 + kG + gl < cA ? nla[(size_t)(s0 + kG + gl) * n] : 0u;
            rj = a.rec[e & kJMask];
            real g[GT::GS], Y[kNLM];
#pragma unroll
            for (int k = 0; k < GT::GS; ++k) g[k] = real(0);
            if (ok) {
                const Pair<real> p = make_pair(frame, rc, ec);
                const int tp = ti * T + p.tj;
                real hf, t[KA];
                cheb_T<real, KA>(p.r, P[off.rcAi + tp], P[off.rcAl + tp], hf, t);
                const real* crow = P + off.cA + tp * coef_stride(NA, KA);
#pragma unroll
                for (int nn = 0; nn < NA; ++nn) {
                    real cr[KA];
                    load_coef(crow + nn * KA, T == 1 && KA % 4 == 0, cr);
                    g[nn] = hf * cheb_sum(cr, t);
                }
                sh_eval(p.dx * p.inv_r, p.dy * p.inv_r, p.dz * p.inv_r, Y);
            } else {  // a zero row adds exact zeros
#pragma unroll
                for (int k = 0; k < kNLM; ++k) Y[k] = real(0);
            }
#pragma unroll
            for (int k = 0; k < GT::GS; k += 4) store4(row + k, g[k], g[k + 1], g[k + 2], g[k + 3]);
#pragma unroll
            for (int k = 0; k < kNLM; k += 4) store4(row + GT::GS + k, Y[k], Y[k + 1], Y[k + 2], Y[k + 3]);
            __syncwarp();
            const int rows = min(kG, most - s0);
#pragma unroll 4
            for (int q = 0; q < rows; ++q) {
                const real* r = tile + q * GT::ROW;
#pragma unroll
                for (int m = 0; m < CH; ++m) {
                    const int ch = CHUNKS % kG ? min(gl + kG * m, CHUNKS - 1) : gl + kG * m;
                    const int nn = kG % NA ? ch % NA : gl % NA, kc = ch / NA;
                    const real gv = r[nn];
                    real y[4];
                    load4(r + GT::GS + 4 * kc, y);
#pragma unroll
                    for (int u = 0; u < 4; ++u) acc[m][u] = fma(gv, y[u], acc[m][u]);
                }
            }
            __syncwarp();
        }
    }
    // the moments as n_A rows of 24, then q_nl (Eq. 4) and the many-body terms by lane n
#pragma unroll
    for (int m = 0; m < CH; ++m) {
        const int ch = gl + kG * m;
        if (CHUNKS % kG == 0 || ch < CHUNKS)
            store4(psi + (ch % NA) * GT::PSI + 4 * (ch / NA), acc[m][0], acc[m][1], acc[m][2], acc[m][3]);
    }
    __syncwarp();
    real g4[5] = {real(0), real(0), real(0), real(0), real(0)};  // dq4/dA_n2m of channel n = gl
    if (gl < NA) {
        real A[kNLM];
        loadN<real, kNLM>(psi + gl * GT::PSI, A);
        real ql[4] = {real(0), real(0), real(0), real(0)};
#pragma unroll
        for (int k = 0; k < kNLM; ++k) ql[l_of(k) - 1] = fma(A[k], A[k], ql[l_of(k) - 1]);
#pragma unroll
        for (int l = 0; l < 4; ++l) sq[NR + l * NA + gl] = ql[l];
        if constexpr (MBT == 1) {
            sq[NR + 4 * NA + gl] = four_body(&A[3], g4);
            sq[NR + 5 * NA + gl] = ql[0] * ql[0];
        }
    }
    if (gl < NR) sq[gl] = q_own;
    __syncwarp();

    // ---- network (Eq. 2) and dU/dq ----
    // Columns v of the sums over the hidden units: v < ND is dU/dq_v (coef_mu w0_mu,v),
    // ND is U (h_mu w1_mu) and ND + 1 its residual part (h_mu w1l_mu).
    constexpr int NC = (ND + 2 + kG - 1) / kG;
    real U;
    {
        real q[NDV];
        loadN<real, NDV>(sq, q);
        const real* w0 = P + off.w0g + (size_t)ti * H * NDV;
        const real* w0l = RES ? P + off.w0lg + (size_t)ti * H * NDV : nullptr;
        const real* b0 = P + off.b0 + ti * H;
        const real* b0l = kF32 ? P + off.b0l + ti * H : nullptr;
        const real* w1 = P + off.w1 + ti * H;
        real col[NC];
        const real* cw[NC];
        const real* cm[NC];
        int cs[NC];
#pragma unroll
        for (int c = 0; c < NC; ++c) {
            const int v = gl + kG * c;
            col[c] = v == ND ? -P[off.b1 + ti] : real(0);
            cw[c] = w0 + v;
            cm[c] = scoef;
            cs[c] = NDV;
            if (v >= ND) {  // past ND + 1: a column that nothing reads
                cw[c] = w1;
                cm[c] = sh;
                cs[c] = 1;
                if (kF32 && v == ND + 1) {
                    col[c] = -P[off.b1l + ti];
                    cw[c] = P + off.w1l + ti * H;
                }
            }
        }
        for (int mu0 = 0; mu0 < H; mu0 += 32) {
            const int many = min(32, H - mu0);
            for (int u = gl; u < many; u += kG) {
                const int mu = mu0 + u;
                real w[NDV];
                loadN<real, NDV>(w0 + (size_t)mu * NDV, w);
                real x = -b0[mu];
#pragma unroll
                for (int v = 0; v < ND; ++v) x = fma(w[v], q[v], x);
                if constexpr (kF32) {
                    real xl = -b0l[mu];
                    if constexpr (RES == 1) {
                        loadN<real, NDV>(w0l + (size_t)mu * NDV, w);
#pragma unroll
                        for (int v = 0; v < ND; ++v) xl = fma(w[v], q[v], xl);
                    }
                    x += xl;
                }
                const real h = tanh_r(x);
                sh[u] = h;
                scoef[u] = w1[mu] * fma(-h, h, real(1));
            }
            __syncwarp();
#pragma unroll 4
            for (int u = 0; u < many; ++u)
#pragma unroll
                for (int c = 0; c < NC; ++c) col[c] = fma(cm[c][u], cw[c][(size_t)(mu0 + u) * cs[c]], col[c]);
            __syncwarp();
        }
#pragma unroll
        for (int c = 0; c < NC; ++c) sdq[gl + kG * c] = col[c];
        __syncwarp();
        U = sdq[ND];
        if constexpr (kF32) U += sdq[ND + 1];
    }
    if (live && gl == 0) a.U[i] = U;
    // e_i^t[k] = sum_n dU/dq_n c^{t_i t}_{nk}
    if (live) {
        real dr[NR];
#pragma unroll
        for (int nn = 0; nn < NR; ++nn) dr[nn] = sdq[nn];
        real* ei = a.e + (size_t)i * a.e_stride;
        for (int t = 0; t < T; ++t) {
            const real* c = P + off.cR + (ti * T + t) * coef_stride(NR, KR);
#pragma unroll
            for (int k = gl; k < KRP; k += kG) {
                real v = real(0);
                if (k < KR) {
#pragma unroll
                    for (int nn = 0; nn < NR; ++nn) v = fma(dr[nn], c[nn * KR + k], v);
                }
                ei[t * KRP + k] = v;
            }
        }
    }
    if constexpr (MBT == 1) {
        // dq5/dA_n1m = 2 q_n1 dq_n1/dA_n1m: fold into the l = 1 coefficient
        if (gl < NA) sdq[NR + gl] = fma(real(2) * sq[NR + gl], sdq[NR + 5 * NA + gl], sdq[NR + gl]);
        __syncwarp();
    }
    // Phi_nlm in place of A_nlm, then each P_n's sphere-reduced form in place of Phi_n
#pragma unroll
    for (int m = 0; m < CH; ++m) {
        const int ch = gl + kG * m;
        if (CHUNKS % kG == 0 || ch < CHUNKS) {
            const int nn = ch % NA, kc = ch / NA;
            real v[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const int k = 4 * kc + u;
                const int l = k < 3 ? 0 : (k < 8 ? 1 : (k < 15 ? 2 : 3));
                v[u] = real(2) * sdq[NR + l * NA + nn] * acc[m][u];
            }
            store4(psi + nn * GT::PSI + 4 * kc, v[0], v[1], v[2], v[3]);
        }
    }
    __syncwarp();
    if (gl < NA) {
        real phi[kNLM], red[GT::PSI];
        loadN<real, kNLM>(psi + gl * GT::PSI, phi);
        if constexpr (MBT == 1) {
            const real d4 = sdq[NR + 4 * NA + gl];
#pragma unroll
            for (int u = 0; u < 5; ++u) phi[3 + u] = fma(d4, g4[u], phi[3 + u]);
        }
        sh_reduce(phi, red);
        red[25] = red[26] = red[27] = real(0);
#pragma unroll
        for (int k = 0; k < GT::PSI; k += 4) store4(psi + gl * GT::PSI + k, red[k], red[k + 1], red[k + 2], red[k + 3]);
    }
    __syncwarp();

    // ---- angular pairs: f_ij = dU_i/dr_ij (see force_angular_phi_reg) ----
    const bool per_bead = a.virial != nullptr;
    real s0_ = real(0), s1_ = real(0);  // FP32: this lane's components gl and gl + 8 of (F, W)
    uint32_t e = gl < cA ? nla[(size_t)gl * n] : 0u;
    PosRec<real> rj = a.rec[e & kJMask];
    for (int s0 = 0; s0 < most; s0 += kG) {
        const int s = s0 + gl;
        const uint32_t ec = e;
        const PosRec<real> rc = rj;
        e = s + kG < cA ? nla[(size_t)(s + kG) * n] : 0u;
        rj = a.rec[e & kJMask];
        real out[12];
#pragma unroll
        for (int k = 0; k < 12; ++k) out[k] = real(0);
        if (s < cA) {
            const Pair<real> p = make_pair(frame, rc, ec);
            const int tij = ti * T + p.tj;
            real hf, hdf, hdx, t[KA], dt[KA];
            cheb_dT<real, KA>(p.r, P[off.rcAi + tij], P[off.rcAl + tij], hf, hdf, hdx, t, dt);
            const real* crow = P + off.cA + tij * coef_stride(NA, KA);
            const real ux = p.dx * p.inv_r, uy = p.dy * p.inv_r, uz = p.dz * p.inv_r;
            real D = real(0);
            real ga[3] = {real(0), real(0), real(0)};
#pragma unroll
            for (int nn = 0; nn < NA; ++nn) {
                real cr[KA];
                load_coef(crow + nn * KA, T == 1 && KA % 4 == 0, cr);
                real g, dg;
                cheb_g_dg(cr, t, dt, hf, hdf, hdx, g, dg);
                real c[GT::PSI];
                loadN<real, GT::PSI>(psi + nn * GT::PSI, c);
                real v, vx, vy, vz;
                sh_red_eval(c, ux, uy, uz, v, vx, vy, vz);
                D = fma(dg, v, D);
                ga[0] = fma(g, vx, ga[0]);
                ga[1] = fma(g, vy, ga[1]);
                ga[2] = fma(g, vz, ga[2]);
            }
            real fij[3];
            angular_force(D, ga, ux, uy, uz, p.inv_r, fij);
            if constexpr (kF32) {
                unsigned long long* acc_j = a.accF + (size_t)p.j * 4;
                const real d[3] = {p.dx, p.dy, p.dz};
#pragma unroll
                for (int k = 0; k < 3; ++k) {
                    out[k] = fij[k];
                    fix_add(acc_j + k, -fij[k]);
                }
                unsigned long long* accw_j = per_bead ? a.accW + (size_t)p.j * 12 : nullptr;
#pragma unroll
                for (int k = 0; k < 3; ++k)
#pragma unroll
                    for (int q = 0; q < 3; ++q) {
                        const real w = mul_rn(-d[k], fij[q]);
                        out[3 + 3 * k + q] = w;
                        if (per_bead) fix_add(accw_j + 3 * k + q, w);
                    }
            } else {
                real* o = a.fang + ((size_t)s * n + i) * 3;
                o[0] = fij[0];
                o[1] = fij[1];
                o[2] = fij[2];
            }
        }
        if constexpr (kF32) {  // the components' sums in slot order
            real* row = tile + gl * 12;
            store4(row, out[0], out[1], out[2], out[3]);
            store4(row + 4, out[4], out[5], out[6], out[7]);
            store4(row + 8, out[8], out[9], out[10], out[11]);
            __syncwarp();
            const int rows = min(kG, most - s0);
            for (int q = 0; q < rows; ++q) {
                s0_ += tile[q * 12 + gl];
                s1_ += tile[q * 12 + 8 + gl % 4];
            }
            __syncwarp();
        }
    }
    if constexpr (kF32) {
        if (live) {
            if (gl < 3) fix_add(a.accF + (size_t)i * 4 + gl, s0_);
            else a.wsum[(size_t)(gl - 3) * n + i] = s0_;
            if (gl < 4) a.wsum[(size_t)(5 + gl) * n + i] = s1_;
        }
    }
}

// Radial pairs in gather form (see force_radial of evaluate.cu), the angular parts, the
// outputs and the totals.  FP32: the angular part of F_i and W_i is in i's fixed-point
// lines.  FP64: it is summed here from the stored f_ij and f_ji.
template <typename real, int NR, int NA, int KR>
__global__ void __launch_bounds__(kBlock, 4) k_force_group(EvalArgs<real> a)
{
    constexpr int KRP = (KR + 3) & ~3;
    constexpr bool kF32 = sizeof(real) == 4;
    constexpr int ROW = 12, GROUP = kG * ROW + (kF32 ? 8 : 40);  // 8 mod 32 (see GroupTile); FP64: PairFrame's table
    __shared__ __align__(16) real smem[kGP * GROUP];
    __shared__ bool last;
    const int item = (int)blockIdx.x / kG;
    if (item >= a.counts->n_items) return;
    const WorkItem it = a.items[item];
    const int first = it.begin + ((int)blockIdx.x % kG) * kGP;
    if (first >= it.end) return;
    const ReqInfo& rq = a.reqs[it.req];
    const ModelDesc<real> md = a.models[rq.model];
    const ParamLayout off = md.off;
    const real* __restrict__ P = md.params;
    const int T = md.T;
    const int gl = (int)threadIdx.x % kG, grp = (int)threadIdx.x / kG;
    real* tile = smem + grp * GROUP;
    const bool live = first + grp < it.end;
    const int i = live ? first + grp : it.end - 1;
    const size_t n = (size_t)a.n;
    const PosRec<real> ri = a.rec[i];
    const PairFrame<real> frame(rq.g, ri, tile + kG * ROW, gl);
    const int ti = ri.t;
    const int cR = live ? min(a.cntR[i], a.mnR) : 0;
    const int most = __reduce_max_sync(kFull, cR);
    const real* e_i = a.e + (size_t)i * a.e_stride;
    const uint32_t* nl = a.nlR + i;
    real ei1[KRP];
    if (T == 1) load_grad<real, KRP>(e_i, ei1);
    // FP32: component c < 9 of (F, symmetric W) is the sum over the pairs, in slot order, of
    // the product of row entries ia and ib; lane c has component c, lane 0 also component 8.
    // FP64: each lane sums its pairs' components.
    const int ia = gl < 3 ? 0 : (gl < 6 ? gl + 1 : 4), ib = gl < 3 ? gl + 1 : (gl < 6 ? gl + 4 : gl + 2);
    real s0_ = real(0), s8 = real(0);
    real F[3] = {real(0), real(0), real(0)}, W[9];
#pragma unroll
    for (int k = 0; k < 9; ++k) W[k] = real(0);
    // the list two rounds ahead, the neighbour's record and gradient vector one round ahead
    uint32_t e = gl < cR ? nl[(size_t)gl * n] : 0u;
    uint32_t e2 = kG + gl < cR ? nl[(size_t)(kG + gl) * n] : 0u;
    PosRec<real> rj = a.rec[e & kJMask];
    real ej[KRP];
    load_grad<real, KRP>(a.e + (size_t)(e & kJMask) * a.e_stride + ti * KRP, ej);
    for (int s0 = 0; s0 < most; s0 += kG) {
        const int s = s0 + gl;
        const uint32_t ec = e;
        const PosRec<real> rc = rj;
        real eji[KRP];
#pragma unroll
        for (int k = 0; k < KRP; ++k) eji[k] = ej[k];
        e = e2;
        e2 = s + 2 * kG < cR ? nl[(size_t)(s + 2 * kG) * n] : 0u;
        if (s0 + kG < most) {
            rj = a.rec[e & kJMask];
            load_grad<real, KRP>(a.e + (size_t)(e & kJMask) * a.e_stride + ti * KRP, ej);
        }
        real fs = real(0), ux = real(0), uy = real(0), uz = real(0), wx = real(0), wy = real(0), wz = real(0);
        real dx = real(0), dy = real(0), dz = real(0);
        if (s < cR) {
            real eij[KRP];
            const Pair<real> p = make_pair(frame, rc, ec);
            if (T == 1) {
#pragma unroll
                for (int k = 0; k < KRP; ++k) eij[k] = ei1[k];
            } else {
                load_grad<real, KRP>(e_i + p.tj * KRP, eij);
            }
            real f[KR], df[KR];
            const int tp = ti * T + p.tj;
            basis_d<real, KR>(p.r, P[off.rcRi + tp], P[off.rcRl + tp], f, df);
            real ai = real(0), bj = real(0);
#pragma unroll
            for (int k = 0; k < KR; ++k) {
                ai = fma(eij[k], df[k], ai);
                bj = fma(eji[k], df[k], bj);
            }
            dx = p.dx;
            dy = p.dy;
            dz = p.dz;
            ux = dx * p.inv_r;
            uy = dy * p.inv_r;
            uz = dz * p.inv_r;
            fs = ai + bj;
            const real w = bj * p.inv_r;
            wx = w * dx;
            wy = w * dy;
            wz = w * dz;
        }
        if constexpr (kF32) {
            real* row = tile + gl * ROW;
            store4(row, fs, ux, uy, uz);
            store4(row + 4, -wx, -wy, -wz, dx);
            store4(row + 8, dy, dz, real(0), real(0));
            __syncwarp();
            // entries: 0 fs, 1-3 u, 4-6 -w, 7 dx, 8 dy, 9 dz
            const int rows = min(kG, most - s0);
#pragma unroll 4
            for (int q = 0; q < rows; ++q) {
                const real* r = tile + q * ROW;
                s0_ = fma(r[ia], r[ib], s0_);
                s8 = fma(r[5], r[9], s8);
            }
            __syncwarp();
        } else {
            F[0] = fma(fs, ux, F[0]);
            F[1] = fma(fs, uy, F[1]);
            F[2] = fma(fs, uz, F[2]);
            W[0] = fma(-wx, dx, W[0]);
            W[4] = fma(-wy, dy, W[4]);
            W[8] = fma(-wz, dz, W[8]);
            W[1] = fma(-wx, dy, W[1]);
            W[2] = fma(-wx, dz, W[2]);
            W[5] = fma(-wy, dz, W[5]);
        }
    }
    if constexpr (!kF32) {
        W[3] = W[1];
        W[6] = W[2];
        W[7] = W[5];
        // angular pairs: F_i += f_ij - f_ji, W_i += r_ij (x) f_ji; f_ji is in the slot of j's
        // list that holds i at the opposite cell offset (each code field d + 2 becomes
        // 2 - d).  A pair within rounding of the cutoff may be in one list only; its other
        // direction is left out.  The largest term of it is f_c', which falls to zero linearly
        // at r_c (f_c quadratically): pi^2/2 times the relative distance to r_c, some 1e-15 of a
        // pair's force, the rounding of the sums that it would enter.
        const int cA = live ? min(a.cntA[i], a.mnA) : 0;
        for (int s = gl; s < cA; s += kG) {
            const uint32_t ea = a.nlA[(size_t)s * n + i];
            const int j = (int)(ea & kJMask);
            const uint32_t back = (uint32_t)i | ((0x124u - (ea >> kJBits)) << kJBits);
            const int cj = min(a.cntA[j], a.mnA);
            real dx, dy, dz;
            frame.vec(a.rec[j], ea, dx, dy, dz);
            const real* fi = a.fang + ((size_t)s * n + i) * 3;
            real fj[3] = {real(0), real(0), real(0)};
            for (int t = 0; t < cj; ++t)
                if (a.nlA[(size_t)t * n + j] == back) {
                    const real* fp = a.fang + ((size_t)t * n + j) * 3;
                    fj[0] = fp[0];
                    fj[1] = fp[1];
                    fj[2] = fp[2];
                    break;
                }
            const real d[3] = {dx, dy, dz};
#pragma unroll
            for (int k = 0; k < 3; ++k) {
                F[k] += fi[k] - fj[k];
#pragma unroll
                for (int q = 0; q < 3; ++q) W[3 * k + q] = fma(d[k], fj[q], W[3 * k + q]);
            }
        }
    }
    // the particle's sums in shared memory: F[3] at 0, the radial virial (FP32: in full from
    // its symmetric part; FP64: the whole virial) W[9] at 3
    if constexpr (kF32) {
        if (gl < 3) {
            tile[gl] = s0_;
        } else {  // symmetric components 0 ... 4: xx yy zz xy xz
            const int c = gl - 3;
            const int k0 = c == 0 ? 0 : (c == 1 ? 4 : (c == 2 ? 8 : (c == 3 ? 1 : 2)));
            const int k1 = c == 3 ? 3 : (c == 4 ? 6 : k0);
            tile[3 + k0] = s0_;
            tile[3 + k1] = s0_;
        }
        if (gl == 0) tile[3 + 5] = tile[3 + 7] = s8;
    } else {
#pragma unroll
        for (int k = 0; k < 3; ++k) F[k] = group_sum(F[k]);
#pragma unroll
        for (int k = 0; k < 9; ++k) W[k] = group_sum(W[k]);
        if (gl == 0) {
#pragma unroll
            for (int k = 0; k < 3; ++k) tile[k] = F[k];
#pragma unroll
            for (int k = 0; k < 9; ++k) tile[3 + k] = W[k];
        }
    }
    __syncwarp();
    if (live) {
        const int ui = a.perm[i];
        const int lu = ui - rq.begin;
        const bool out_ok = lu >= 0 && lu < rq.n;  // see kErrCellList
        if (!out_ok && a.err && gl == 0) atomicOr(a.err, kErrCellList);
        if (gl < 3) {
            double Fp = (double)tile[gl];
            if constexpr (kF32) {
                unsigned long long* line = a.accF + (size_t)i * 4 + gl;
                Fp = (double)(fix_value_f(*line) + tile[gl]);
                *line = 0ull;
            }
            if (out_ok) {
                a.force[(size_t)3 * rq.begin + lu + (size_t)gl * rq.n] = Fp;
                if (a.kick_vel) {
                    const int t = a.kick_types[ui];
                    double* v = a.kick_vel + (size_t)3 * rq.begin + lu + (size_t)gl * rq.n;
                    *v = half_kick(*v, a.kick_half_dt, Fp, a.kick_im.v[t >= 0 && t < kMdMaxTypes ? t : 0]);
                }
            }
        }
        for (int k = gl; k < 9; k += kG) {
            const real w = tile[3 + k];
            if (a.virial) {
                double Wk = (double)w;
                if constexpr (kF32) {
                    unsigned long long* line = a.accW + (size_t)i * 12 + k;
                    Wk = (double)(fix_value_f(*line) + w);
                    *line = 0ull;
                }
                if (out_ok) a.virial[(size_t)9 * rq.begin + lu + (size_t)k * rq.n] = Wk;
            }
            // i's contribution to the virial total (FP32: its angular sum plus its radial part)
            real* ws = a.wsum + (size_t)k * n + i;
            *ws = kF32 ? *ws + w : w;
        }
        if (gl == 3 && a.site && out_ok) a.site[ui] = (double)a.U[i];
    }
    // totals: the item's last block sums its particles as one block of evaluate.cu would
    __threadfence();
    __syncthreads();
    const unsigned blocks = (unsigned)((it.end - it.begin + kGP - 1) / kGP);
    if (threadIdx.x == 0) last = atomicAdd(&a.icounter[item], 1u) == blocks - 1u;
    __syncthreads();
    if (!last) return;
    if (threadIdx.x == 0) a.icounter[item] = 0u;
    __threadfence();
    const int it_i = it.begin + (int)threadIdx.x;
    double tot[10];
#pragma unroll
    for (int k = 0; k < 10; ++k) tot[k] = 0.0;
    if (it_i < it.end) {
        tot[0] = (double)__ldcg(a.U + it_i);
#pragma unroll
        for (int k = 0; k < 9; ++k) tot[1 + k] = (double)__ldcg(a.wsum + (size_t)k * n + it_i);
    }
    reduce_totals<kBlock>(tot, item, it, rq, a.partial, a.gcounter, a.counter, a.counts, a.totals);
}

template <typename real, int NA>
constexpr size_t group_smem()
{
    return sizeof(real) * kGP * GroupTile<NA>::SIZE;
}

template <typename real, int NR, int NA, int KR, int KA, int RES, int MBT>
static cudaError_t launch_descriptor_group(const EvalArgs<real>& a, int nb, cudaStream_t st)
{
    return launch_k(k_descriptor_group<real, NR, NA, KR, KA, RES, MBT>, nb, kBlock, group_smem<real, NA>(), st, a);
}

template <typename real>
cudaError_t group_set_smem()
{
    // only the FP64 rows of the second shape take more than the 48 KB a kernel gets unasked
    auto set = [](auto* kernel, size_t bytes) {
        if (bytes <= 48 * 1024) return cudaSuccess;
        return cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
    };
    cudaError_t e = cudaSuccess;
#define NEP_CASE(a_, b_, c_, d_)                                                                               \
    if (e == cudaSuccess) e = set(k_descriptor_group<real, a_, b_, c_, d_, 0, 0>, group_smem<real, b_>());     \
    if (e == cudaSuccess) e = set(k_descriptor_group<real, a_, b_, c_, d_, 0, 1>, group_smem<real, b_>());     \
    if constexpr (sizeof(real) == 4) {                                                                         \
        if (e == cudaSuccess) e = set(k_descriptor_group<real, a_, b_, c_, d_, 1, 0>, group_smem<real, b_>()); \
        if (e == cudaSuccess) e = set(k_descriptor_group<real, a_, b_, c_, d_, 1, 1>, group_smem<real, b_>()); \
    }
    NEP_SHAPES(NEP_CASE)
#undef NEP_CASE
    return e;
}

template <typename real>
cudaError_t launch_evaluate_group(int nR, int nA, int KR, int KA, const EvalArgs<real>& a, int items_cap, cudaStream_t st,
                                  cudaEvent_t mid)
{
    const int nb = items_cap * kG;
    if (!a.wsum || !a.icounter || (sizeof(real) == 4 ? !a.accF : !a.fang)) return cudaErrorInvalidValue;
#define NEP_CASE(a_, b_, c_, d_)                                                                                \
    if (nR == a_ && nA == b_ && KR == c_ && KA == d_) {                                                         \
        cudaError_t e;                                                                                          \
        if constexpr (sizeof(real) == 4) {                                                                      \
            if (a.w0_residual)                                                                                  \
                e = a.many_body ? launch_descriptor_group<real, a_, b_, c_, d_, 1, 1>(a, nb, st)                \
                                : launch_descriptor_group<real, a_, b_, c_, d_, 1, 0>(a, nb, st);               \
            else                                                                                                \
                e = a.many_body ? launch_descriptor_group<real, a_, b_, c_, d_, 0, 1>(a, nb, st)                \
                                : launch_descriptor_group<real, a_, b_, c_, d_, 0, 0>(a, nb, st);               \
        } else {                                                                                                \
            e = a.many_body ? launch_descriptor_group<real, a_, b_, c_, d_, 0, 1>(a, nb, st)                    \
                            : launch_descriptor_group<real, a_, b_, c_, d_, 0, 0>(a, nb, st);                   \
        }                                                                                                       \
        if (e != cudaSuccess) return e;                                                                         \
        if (mid && (e = cudaEventRecord(mid, st)) != cudaSuccess) return e;                                     \
        return launch_k(k_force_group<real, a_, b_, c_>, nb, kBlock, 0, st, a);                                 \
    }
    NEP_SHAPES(NEP_CASE)
#undef NEP_CASE
    return cudaErrorInvalidValue;
}

#define NEP_INSTANTIATE(real)                                                                                  \
    template cudaError_t group_set_smem<real>();                                                               \
    template cudaError_t launch_evaluate_group<real>(int, int, int, int, const EvalArgs<real>&, int, cudaStream_t, \
                                                     cudaEvent_t);
NEP_INSTANTIATE(float)
NEP_INSTANTIATE(double)
#undef NEP_INSTANTIATE

}  // namespace nep

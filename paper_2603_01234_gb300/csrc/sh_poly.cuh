// Generated by gen_sh.py -- real orthonormal spherical harmonics, l = 1..4.
// Index k = l*l - 1 + (m + l).  (x, y, z) is a unit vector: the forms use
// x^2 + y^2 + z^2 = 1 and hold on the sphere only.
#pragma once

template <typename real>
__device__ __forceinline__ void sh_eval(real x, real y, real z, real* Y)
{
    const real x2 = x * x;
    const real y2 = y * y;
    const real z2 = z * z;
    const real xy = x * y;
    const real xz = x * z;
    const real yz = y * z;
    const real dd = fma(x, x, -y2);
    const real p3 = fma(real(3), x2, -y2);
    const real m3 = fma(real(-3), y2, x2);
    const real a3 = fma(real(2.2852289973223287), z2, real(-0.45704579946446574));
    const real t4 = fma(real(4.6833258049010242), z2, real(-2.0071396306718675));
    Y[0] = real(0.48860251190291992) * y;
    Y[1] = real(0.48860251190291992) * z;
    Y[2] = real(0.48860251190291992) * x;
    Y[3] = real(1.0925484305920791) * xy;
    Y[4] = real(1.0925484305920791) * yz;
    Y[5] = fma(real(0.94617469575756002), z2, real(-0.31539156525252001));
    Y[6] = real(1.0925484305920791) * xz;
    Y[7] = real(0.54627421529603954) * dd;
    Y[8] = real(0.59004358992664351) * y * p3;
    Y[9] = real(2.8906114426405541) * xy * z;
    Y[10] = y * a3;
    Y[11] = z * fma(real(1.8658816629505770), z2, real(-1.1195289977703462));
    Y[12] = x * a3;
    Y[13] = real(1.4453057213202770) * z * dd;
    Y[14] = real(0.59004358992664351) * x * m3;
    Y[15] = real(2.5033429417967045) * xy * dd;
    Y[16] = real(1.7701307697799305) * yz * p3;
    Y[17] = xy * fma(real(6.6232228703029201), z2, real(-0.94617469575756002));
    Y[18] = yz * t4;
    Y[19] = fma(fma(real(3.7024941420321506), z2, real(-3.1735664074561291)), z2, real(0.31735664074561291));
    Y[20] = xz * t4;
    Y[21] = dd * fma(real(3.3116114351514601), z2, real(-0.47308734787878001));
    Y[22] = real(1.7701307697799305) * xz * m3;
    Y[23] = real(0.62583573544917613) * fma(x2, m3, -(y2 * p3));
}

// Sphere-reduced form: with z^2 = 1 - x^2 - y^2 each Y_k equals A_k(x, y) + z B_k(x, y)
// on the unit sphere, deg A_k <= 4, deg B_k <= 3 (the two forms have equal values and
// equal surface gradients there).  A 25-entry coefficient vector holds block A
// (x^a y^b, a + b <= 4) at sh_red_a(a) + b and block B (z x^a y^b, a + b <= 3) at
// sh_red_b(a) + b.
constexpr int kShRed = 25;
__host__ __device__ constexpr int sh_red_a(int a) { return a * 5 - a * (a - 1) / 2; }
__host__ __device__ constexpr int sh_red_b(int a) { return 15 + a * 4 - a * (a - 1) / 2; }

// psi = sum_k phi[k] (reduced form of Y_k): the reduced coefficients of sum_k phi[k] Y_k
template <typename real>
__device__ __forceinline__ void sh_reduce(const real* phi, real* psi)
{
    psi[0] = fma(real(0.84628437532163443), phi[19], real(0.63078313050504001) * phi[5]);
    psi[1] = fma(real(1.8281831978578629), phi[10], real(0.48860251190291992) * phi[0]);
    psi[2] = fma(real(-2.8385240872726801), phi[21], fma(real(-4.2314218766081722), phi[19], fma(real(-0.54627421529603954), phi[7], real(-0.94617469575756002) * phi[5])));
    psi[3] = fma(real(-2.2852289973223287), phi[10], real(-0.59004358992664351) * phi[8]);
    psi[4] = fma(real(0.62583573544917613), phi[23], fma(real(3.3116114351514601), phi[21], real(3.7024941420321506) * phi[19]));
    psi[5] = fma(real(1.8281831978578629), phi[12], real(0.48860251190291992) * phi[2]);
    psi[6] = fma(real(5.6770481745453601), phi[17], real(1.0925484305920791) * phi[3]);
    psi[7] = fma(real(-1.7701307697799305), phi[14], real(-2.2852289973223287) * phi[12]);
    psi[8] = fma(real(-6.6232228703029201), phi[17], real(-2.5033429417967045) * phi[15]);
    psi[9] = fma(real(2.8385240872726801), phi[21], fma(real(-4.2314218766081722), phi[19], fma(real(0.54627421529603954), phi[7], real(-0.94617469575756002) * phi[5])));
    psi[10] = fma(real(-2.2852289973223287), phi[10], real(1.7701307697799305) * phi[8]);
    psi[11] = fma(real(-3.7550144126950568), phi[23], real(7.4049882840643013) * phi[19]);
    psi[12] = fma(real(0.59004358992664351), phi[14], real(-2.2852289973223287) * phi[12]);
    psi[13] = fma(real(-6.6232228703029201), phi[17], real(2.5033429417967045) * phi[15]);
    psi[14] = fma(real(0.62583573544917613), phi[23], fma(real(-3.3116114351514601), phi[21], real(3.7024941420321506) * phi[19]));
    psi[15] = fma(real(0.74635266518023078), phi[11], real(0.48860251190291992) * phi[1]);
    psi[16] = fma(real(2.6761861742291567), phi[18], real(1.0925484305920791) * phi[4]);
    psi[17] = fma(real(-1.4453057213202770), phi[13], real(-1.8658816629505770) * phi[11]);
    psi[18] = fma(real(-4.6833258049010242), phi[18], real(-1.7701307697799305) * phi[16]);
    psi[19] = fma(real(2.6761861742291567), phi[20], real(1.0925484305920791) * phi[6]);
    psi[20] = real(2.8906114426405541) * phi[9];
    psi[21] = fma(real(-5.3103923093397916), phi[22], real(-4.6833258049010242) * phi[20]);
    psi[22] = fma(real(1.4453057213202770), phi[13], real(-1.8658816629505770) * phi[11]);
    psi[23] = fma(real(-4.6833258049010242), phi[18], real(5.3103923093397916) * phi[16]);
    psi[24] = fma(real(1.7701307697799305), phi[22], real(-4.6833258049010242) * phi[20]);
}

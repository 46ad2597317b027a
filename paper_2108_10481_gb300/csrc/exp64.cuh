// FP64 exponential of the pair sums (the direct pair kernels and the near field's band and
// far-rule blocks). Not part of the C ABI.
#pragma once

#include <cuda_runtime.h>

namespace pb {

constexpr double EXP64_PER_UNIT = 0x1.71547652b82fep+6;  // 64 / ln 2

// 2^{j/64}, correctly rounded
static __device__ const double g_exp2_64[64] = {
    0x1.0000000000000p+0, 0x1.02c9a3e778061p+0, 0x1.059b0d3158574p+0, 0x1.0874518759bc8p+0,
    0x1.0b5586cf9890fp+0, 0x1.0e3ec32d3d1a2p+0, 0x1.11301d0125b51p+0, 0x1.1429aaea92de0p+0,
    0x1.172b83c7d517bp+0, 0x1.1a35beb6fcb75p+0, 0x1.1d4873168b9aap+0, 0x1.2063b88628cd6p+0,
    0x1.2387a6e756238p+0, 0x1.26b4565e27cddp+0, 0x1.29e9df51fdee1p+0, 0x1.2d285a6e4030bp+0,
    0x1.306fe0a31b715p+0, 0x1.33c08b26416ffp+0, 0x1.371a7373aa9cbp+0, 0x1.3a7db34e59ff7p+0,
    0x1.3dea64c123422p+0, 0x1.4160a21f72e2ap+0, 0x1.44e086061892dp+0, 0x1.486a2b5c13cd0p+0,
    0x1.4bfdad5362a27p+0, 0x1.4f9b2769d2ca7p+0, 0x1.5342b569d4f82p+0, 0x1.56f4736b527dap+0,
    0x1.5ab07dd485429p+0, 0x1.5e76f15ad2148p+0, 0x1.6247eb03a5585p+0, 0x1.6623882552225p+0,
    0x1.6a09e667f3bcdp+0, 0x1.6dfb23c651a2fp+0, 0x1.71f75e8ec5f74p+0, 0x1.75feb564267c9p+0,
    0x1.7a11473eb0187p+0, 0x1.7e2f336cf4e62p+0, 0x1.82589994cce13p+0, 0x1.868d99b4492edp+0,
    0x1.8ace5422aa0dbp+0, 0x1.8f1ae99157736p+0, 0x1.93737b0cdc5e5p+0, 0x1.97d829fde4e50p+0,
    0x1.9c49182a3f090p+0, 0x1.a0c667b5de565p+0, 0x1.a5503b23e255dp+0, 0x1.a9e6b5579fdbfp+0,
    0x1.ae89f995ad3adp+0, 0x1.b33a2b84f15fbp+0, 0x1.b7f76f2fb5e47p+0, 0x1.bcc1e904bc1d2p+0,
    0x1.c199bdd85529cp+0, 0x1.c67f12e57d14bp+0, 0x1.cb720dcef9069p+0, 0x1.d072d4a07897cp+0,
    0x1.d5818dcfba487p+0, 0x1.da9e603db3285p+0, 0x1.dfc97337b9b5fp+0, 0x1.e502ee78b3ff6p+0,
    0x1.ea4afa2a490dap+0, 0x1.efa1bee615a27p+0, 0x1.f50765b6e4540p+0, 0x1.fa7c1819e90d8p+0};

// e^x for x = t ln2/64 <= 0 by the table-driven method of Tang (ACM Trans. Math.
// Software 15(2), 1989): t = 64 m + j + f with |f| <= 1/2, e^x = 2^m 2^{j/64} 2^{f/64}.
// The caller forms t = -kappa r (64 / ln 2) with one product, so f is exact and no
// reduction of x by parts is needed. 2^{f/64}: the Taylor polynomial of degree 6 with its
// last term economised (its Chebyshev part of degree 6 dropped), degree 5, within
// 2.4e-18 relative. Below x = -700 the result is 0.
__device__ __forceinline__ double exp2_64th(double t) {
    const double shifter = 0x1.8p52;
    const double tn = __dadd_rn(t, shifter);
    const int n = __double2loint(tn);
    const double f = __dsub_rn(t, __dsub_rn(tn, shifter));
    double q = 0x1.5d87fe78a6731p-40;
    q = __fma_rn(q, f, 0x1.3b2ad5447eaecp-31);
    q = __fma_rn(q, f, 0x1.c6b08d704a0c0p-23);
    q = __fma_rn(q, f, 0x1.ebfbdff829821p-15);
    q = __fma_rn(q, f, 0x1.62e42fefa39efp-7);
    q = __fma_rn(q, f, 1.0);
    const double v = __ldg(g_exp2_64 + (n & 63)) * q;
    const bool under = (unsigned)__double2hiint(t) > 0xC0EF8F17u;  // integer compare: t below -700 (64 / ln 2)
    return under ? 0.0 : __hiloint2double(__double2hiint(v) + ((n >> 6) << 20), __double2loint(v));
}

}  // namespace pb

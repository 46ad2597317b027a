// Which loop of the pair kernels and of the treecode serves a block operator's rows. Plain C++ (no
// CUDA): the host tests compile it on its own.
//
// k: the coefficients of kernel row 0 (V_L, V_Y, K_L, K_Y) and of row 1 (the same for V/K rows, mode
// 0; D_L, D_Y, T_L, T_Y for a D/T row, mode 1). The loops that keep a Laplace coefficient out of
// their sums multiply, or divide, by it afterwards (in FP32 where the sums are), so they take
// coefficients of ordinary size only: a tiny one, which a combined form's alpha or beta can make,
// would overflow the ratio or flush to zero. The general loop serves every other operator.
#pragma once

#include <cmath>

namespace pb {

inline bool ordinary(double c) { return std::fabs(c) >= 0x1p-40 && std::fabs(c) <= 0x1p40; }

inline bool any_yukawa(const double (&k)[2][4]) {
    return k[0][1] != 0.0 || k[0][3] != 0.0 || k[1][1] != 0.0 || k[1][3] != 0.0;
}

// every operator with a Laplace coefficient that the Yukawa one can be written over
inline bool laplace_ratios(const double (&k)[2][4]) {
    for (int r = 0; r < 2; ++r)
        for (int j = 0; j < 4; j += 2)
            if (!ordinary(k[r][j]) || !(std::fabs(k[r][j + 1]) <= 0x1p40 * std::fabs(k[r][j]))) return false;
    return true;
}

// Pair kernels, V/K + D/T rows: 1 no Yukawa term, 2 V, K, D and T all as Laplace plus a ratio times Yukawa,
// 0 any coefficients. (V/K rows keep the coefficients apart from their sums whatever they are.)
inline int vkdt_kind(const double (&k)[2][4]) { return !any_yukawa(k) ? 1 : laplace_ratios(k) ? 2 : 0; }

// FP64 pair kernels: V/K rows 1 without a Yukawa term, 0 otherwise
inline int pair64_kind(int mode, const double (&k)[2][4]) { return mode == 0 ? (any_yukawa(k) ? 0 : 1) : vkdt_kind(k); }

// FP32 pair kernels: one loop for V/K rows
inline int pair32_kind(int mode, const double (&k)[2][4]) { return mode == 0 ? 0 : vkdt_kind(k); }

// Treecode, V/K rows: 3 one row without a Yukawa and the other without a Laplace term (lrow: the
// former), 0 otherwise. V/K + D/T rows as the pair kernels, but kind 1 too carries K's Laplace
// coefficient in the dipoles.
inline int tree_kind(int mode, const double (&k)[2][4], int* lrow) {
    const bool laplace0 = k[0][1] == 0.0 && k[0][3] == 0.0;
    const int l = laplace0 ? 0 : 1, y = 1 - l;
    *lrow = l;
    if (mode == 0)
        return k[l][1] == 0.0 && k[l][3] == 0.0 && k[y][0] == 0.0 && k[y][2] == 0.0 ? 3 : 0;
    const int kind = vkdt_kind(k);
    return kind == 1 && !ordinary(k[0][2]) ? 0 : kind;
}

}  // namespace pb

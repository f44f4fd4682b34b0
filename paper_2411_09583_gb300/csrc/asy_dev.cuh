// Device helpers shared by the spreading / interpolation kernels (k_asy.cu)
// and the FFT kernels (k_fft.cu) of the asymptotic blocks.
#pragma once

#include "df64.cuh"
#include "nuht_internal.h"

namespace nuht {

// psi^(xi) for xi >= 0 given as double-float, double-float throughout: with
// t = xi times the table's pieces per unit, piece floor(t) (clamped to the
// table) and v = 2 (t - piece) - 1 in [-1, 1], the compensated Horner sum of
// that piece's polynomial.
__device__ __forceinline__ df psihat_of(const Tables& T, df xi)
{
    const df t = df_mul(xi, df{T.ph_scale2.x, T.ph_scale2.y});
    int piece = (int)t.h;
    if ((float)piece == t.h && t.l < 0.f && piece > 0) --piece;
    if (piece > T.ph_pieces - 1) piece = T.ph_pieces - 1;
    const df u = df_add(t, df{-(float)piece, 0.f});
    const df v = df_add(df{2.f * u.h, 2.f * u.l}, df{-1.f, 0.f});
    return horner_comp(T.ph2 + piece * (T.ph_deg + 1), T.ph_deg, v.h, v.l, T.ph_comp);
}

}  // namespace nuht

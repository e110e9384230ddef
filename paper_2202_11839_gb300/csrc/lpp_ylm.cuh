// Harmonics of one unit vector, shared by the orders n = +-m of a degree (internal).
#pragma once

#include "lpp_internal.h"

namespace lpp {

// (x + i y)^m for m = 0 .. 8, once per vector
template <typename T>
struct Azimuth {
    T re[9], im[9];
    __device__ __forceinline__ void set(T x, T y) {
        re[0] = (T)1;
        im[0] = (T)0;
#pragma unroll
        for (int m = 1; m <= 8; ++m) {
            re[m] = re[m - 1] * x - im[m - 1] * y;
            im[m] = re[m - 1] * y + im[m - 1] * x;
        }
    }
};

// (L - M)! Q_L^M(z) with L and M known at compile time: the recurrence of ylm_poly_scaled with
// constant coefficients and no loops.
template <typename T, int L, int M>
__device__ __forceinline__ T q_fixed(T z) {
    T qmm = (T)1;
#pragma unroll
    for (int i = 1; i <= M; ++i) qmm *= (T)(2 * i - 1);
    T q = qmm;
    if constexpr (L > M) {
        T q0 = qmm, q1 = (T)(2 * M + 1) * z * qmm;
#pragma unroll
        for (int l = M + 2; l <= L; ++l) {
            const T q2 = (T)(2 * l - 1) * z * q1 - (T)((l + M - 1) * (l - M - 1)) * q0;
            q0 = q1;
            q1 = q2;
        }
        q = q1;
    }
    return q;
}

// The harmonics n = +m (yc) and n = -m (ys) of degree L (warp-uniform L, m), without their
// normalisation: the estimators' even degrees up to 8 by a compile-time case, anything else by
// the general recurrence.
template <typename T>
__device__ __forceinline__ void ylm_pair(int L, int m, const Azimuth<T>& az, T z, T& yc, T& ys) {
    switch (L * 16 + m) {
#define LPP_YCASE(LL, MM)                       \
    case LL * 16 + MM: {                        \
        const T q = q_fixed<T, LL, MM>(z);      \
        yc = q * az.re[MM];                     \
        ys = q * az.im[MM];                     \
        return;                                 \
    }
        LPP_YCASE(0, 0)
        LPP_YCASE(2, 0) LPP_YCASE(2, 1) LPP_YCASE(2, 2)
        LPP_YCASE(4, 0) LPP_YCASE(4, 1) LPP_YCASE(4, 2) LPP_YCASE(4, 3) LPP_YCASE(4, 4)
        LPP_YCASE(6, 0) LPP_YCASE(6, 1) LPP_YCASE(6, 2) LPP_YCASE(6, 3) LPP_YCASE(6, 4) LPP_YCASE(6, 5)
        LPP_YCASE(6, 6)
        LPP_YCASE(8, 0) LPP_YCASE(8, 1) LPP_YCASE(8, 2) LPP_YCASE(8, 3) LPP_YCASE(8, 4) LPP_YCASE(8, 5)
        LPP_YCASE(8, 6) LPP_YCASE(8, 7) LPP_YCASE(8, 8)
#undef LPP_YCASE
        default:
            yc = ylm_poly_scaled<T>(L, m, az.re[1], az.im[1], z);
            ys = ylm_poly_scaled<T>(L, -m, az.re[1], az.im[1], z);
    }
}

}  // namespace lpp

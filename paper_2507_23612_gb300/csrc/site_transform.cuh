// The coefficient transform of a site, shared by the projector forms.
#pragma once
#include "hub_internal.cuh"
#include "cplx.cuh"

namespace hub {

// W row of a site from its inner products c (KB: gamma C; Hubbard: M C, Eq. DerED)
template <typename R, bool CPLX>
__device__ __forceinline__ void site_transform(const SiteDev& S, const typename VT<double, CPLX>::T* c,
                                               const double* __restrict__ gamma, const double* __restrict__ M,
                                               typename VT<R, CPLX>::T* __restrict__ W, int n, int ncol) {
    using D = typename VT<double, CPLX>::T;
    using T = typename VT<R, CPLX>::T;
    for (int p = 0; p < S.nproj; ++p) {
        D w = zero_of(D());
        if (S.kind == 0) {
            w = mulr(gamma[S.proj_off + p], c[p]);
        } else {
            // coefficient of phi_p: sum_m M[p][m] C_m  (M = (U/2)(I - 2D))
            for (int m = 0; m < S.nproj; ++m) {
                D mm;
                if constexpr (CPLX) {
                    const double* Mi = M + (size_t)S.hub_index * 50;
                    mm = make_double2(Mi[2 * (p * 5 + m)], Mi[2 * (p * 5 + m) + 1]);
                } else {
                    mm = M[(size_t)S.hub_index * 25 + p * 5 + m];
                }
                w = cfma(mm, c[m], w);
            }
        }
        T wv;
        if constexpr (CPLX) wv = T{(R)w.x, (R)w.y};
        else wv = (R)w;
        W[(size_t)(S.proj_off + p) * ncol + n] = wv;
    }
}

}  // namespace hub

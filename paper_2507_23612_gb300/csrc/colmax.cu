// Largest magnitude of every column of a block, as the bits of its leading word (sign removed):
// the scales of the fixed-point stencil and of the digit-split projector products.  One read of
// the block (0.28 ms of 1.81 GB).
#include <algorithm>

#include "hub_internal.cuh"

namespace hub {

namespace {

// kColParts slices per column, each CTA storing its own maximum (nothing to clear); n and ld
// count reals
template <typename R>
__global__ void __launch_bounds__(512)
k_colmax(const R* __restrict__ X, long ld, long n, unsigned* __restrict__ cmax) {
    const R* col = X + (size_t)blockIdx.y * ld;
    const long per = (n + kColParts - 1) / kColParts;
    const long g0 = (long)blockIdx.x * per, g1 = min(g0 + per, n);
    auto bits = [](R v) {
        if constexpr (sizeof(R) == 8) return (unsigned)__double2hiint(v) & 0x7fffffffu;
        else return __float_as_uint(v) & 0x7fffffffu;
    };
    unsigned m = 0;
    long g = g0 + threadIdx.x;
    for (; g + 7 * 512 < g1; g += 8 * 512) {
        R v[8];
#pragma unroll
        for (int i = 0; i < 8; ++i) v[i] = col[g + i * 512];
#pragma unroll
        for (int i = 0; i < 8; ++i) m = max(m, bits(v[i]));
    }
    for (; g < g1; g += 512) m = max(m, bits(col[g]));
    __shared__ unsigned s[16];
    m = __reduce_max_sync(0xffffffffu, m);
    if ((threadIdx.x & 31) == 0) s[threadIdx.x >> 5] = m;
    __syncthreads();
    if (threadIdx.x < 32) {
        m = __reduce_max_sync(0xffffffffu, threadIdx.x < 16 ? s[threadIdx.x] : 0u);
        if (threadIdx.x == 0) cmax[(size_t)blockIdx.y * kColParts + blockIdx.x] = m;
    }
}

}  // namespace

int launch_colmax_at(hub_t h, const void* X, int ncol, int ld, unsigned* cmax) {
    const int cw = h->cplx ? 2 : 1;
    ProfScope ps(h, HUB_K_COPY);
    for (int c0 = 0; c0 < ncol; c0 += 65535) {
        const dim3 grid(kColParts, (unsigned)std::min(65535, ncol - c0));
        unsigned* out = cmax + (size_t)c0 * kColParts;
        if (h->esize == 8)
            k_colmax<double><<<grid, 512, 0, h->stream>>>((const double*)X + (size_t)c0 * ld * cw, (long)ld * cw, h->Nd * cw, out);
        else
            k_colmax<float><<<grid, 512, 0, h->stream>>>((const float*)X + (size_t)c0 * ld * cw, (long)ld * cw, h->Nd * cw, out);
    }
    HUB_CUDA_TRY(h, cudaGetLastError());
    return HUB_OK;
}

int launch_colmax(hub_t h, const void* X, int ncol, int ld) {
    int rc;
    if ((rc = ensure(h, (void**)&h->d_cmax, &h->cmax_bytes,
                     std::max(h->cmax_bytes, (size_t)ncol * kColParts * sizeof(unsigned))))) return rc;
    return launch_colmax_at(h, X, ncol, ld, h->d_cmax);
}

}  // namespace hub

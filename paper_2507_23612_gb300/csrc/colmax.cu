// Largest magnitude of every column of a block and of its pieces of 32 x 8 x n3 / 8 points, as the bits
// of its leading word (sign removed): the scales of the fixed-point stencil and of the digit-split
// products.  One read of the block (0.27 ms of 1.81 GB).
#include <algorithm>
#include <type_traits>

#include "hub_internal.cuh"

namespace hub {

namespace {

__device__ __forceinline__ unsigned lead_bits(double v) { return (unsigned)__double2hiint(v) & 0x7fffffffu; }
__device__ __forceinline__ unsigned lead_bits(float v) { return __float_as_uint(v) & 0x7fffffffu; }
__device__ __forceinline__ unsigned lead_bits(float2 v) { return max(lead_bits(v.x), lead_bits(v.y)); }

// One CTA per column and z part; its warps take strips of RY rows in turn, NX pieces of each together, so
// that the CTA reads the memory nearly in order (88 x 88 x 84 x 348 doubles: 249 us, 246 without the
// pieces; a strip of 8 rows per warp for all planes 260 to 400 us, and 1 ms for some grids of complex
// floats).  Indexes beyond the row or the strip are those of its last point: a maximum takes no harm.  CW
// elements E per point.  Every CTA stores its own maxima (nothing to clear).
constexpr int kColThreads = 512;
template <typename E, int CW, int NX, int RY>
__global__ void __launch_bounds__(kColThreads)
k_colmax(const E* __restrict__ X, long ld, BlockMap b, int n1, int n2, int n3, unsigned* __restrict__ cmax,
         unsigned* __restrict__ bmax) {
    extern __shared__ unsigned piece[];
    __shared__ unsigned tops[kColThreads / 32];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, part = blockIdx.x, nblk = b.nbx * b.nby;
    const int z0 = part * b.zper, z1 = min(z0 + b.zper, n3), row = n1 * CW;
    const E* col = X + (size_t)blockIdx.y * ld + (size_t)z0 * n2 * row;
    for (int i = threadIdx.x; i < nblk; i += kColThreads) piece[i] = 0;
    __syncthreads();
    const int strips = (n2 + RY - 1) / RY, total = max(z1 - z0, 0) * strips;
    unsigned top = 0;
    const int chunks = (n1 + 31) / 32;
    for (int bx = 0; bx < chunks; bx += NX) {
        int at[NX * CW];
#pragma unroll
        for (int k = 0; k < NX * CW; ++k) at[k] = min(32 * (CW * bx + k) + lane, row - 1);
        for (int t = warp; t < total; t += kColThreads / 32) {
            const int z = t / strips, y = (t - z * strips) * RY;
            E v[RY][NX * CW];
            unsigned m[NX];
#pragma unroll
            for (int i = 0; i < RY; ++i)
#pragma unroll
                for (int k = 0; k < NX * CW; ++k) v[i][k] = col[((long)z * n2 + min(y + i, n2 - 1)) * row + at[k]];
#pragma unroll
            for (int k = 0; k < NX; ++k) m[k] = 0;
#pragma unroll
            for (int i = 0; i < RY; ++i)
#pragma unroll
                for (int k = 0; k < NX * CW; ++k) m[k / CW] = max(m[k / CW], lead_bits(v[i][k]));
#pragma unroll
            for (int k = 0; k < NX; ++k) {
                const unsigned r = __reduce_max_sync(0xffffffffu, m[k]);
                if (lane == 0 && bx + k < chunks) atomicMax(&piece[(y >> b.ylog) * b.nbx + ((bx + k) >> (b.xlog - 5))], r);
                top = max(top, r);
            }
        }
    }
    if (lane == 0) tops[warp] = top;
    __syncthreads();
    if (bmax)
        for (int i = threadIdx.x; i < nblk; i += kColThreads) bmax[((size_t)blockIdx.y * kColParts + part) * nblk + i] = piece[i];
    if (threadIdx.x == 0) {
        for (int w = 1; w < kColThreads / 32; ++w) top = max(top, tops[w]);
        cmax[(size_t)blockIdx.y * kColParts + part] = top;
    }
}

template <typename E, int CW>
void run_parts(hub_t h, dim3 grid, const E* X, long ld, const BlockMap& b, unsigned* cmax, unsigned* bmax) {
    const size_t sm = (size_t)b.nbx * b.nby * sizeof(unsigned);
    auto run = [&](auto kernel) { kernel<<<grid, kColThreads, sm, h->stream>>>(X, ld, b, h->n1, h->n2, h->n3, cmax, bmax); };
    if (h->n1 <= 32) run(k_colmax<E, CW, 1, 8>);
    else if (h->n1 <= 64) run(k_colmax<E, CW, 2, 8 / CW>);
    else if (h->n1 <= 96) run(k_colmax<E, CW, 3, std::is_same<E, float2>::value ? 2 : 4 / CW>);
    else run(k_colmax<E, CW, 4, 4 / CW>);
}

}  // namespace

BlockMap block_map(const hub_ctx* h, const unsigned* cmax, int ncol) {
    BlockMap b{cmax ? cmax + (size_t)ncol * kColParts : nullptr, 0, 0, (h->n3 + kColParts - 1) / kColParts, 5, 3};
    auto count = [](int n, int log) { return (int)(((long)n + (1L << log) - 1) >> log); };
    for (;;) {
        b.nbx = count(h->n1, b.xlog);
        b.nby = count(h->n2, b.ylog);
        if ((long)b.nbx * b.nby <= kColPieces) return b;
        if (b.nby > 1) ++b.ylog;
        else ++b.xlog;
    }
}

size_t colmax_bytes(const hub_ctx* h, int ncol) {
    const BlockMap b = block_map(h, nullptr, 0);
    return (size_t)ncol * kColParts * (1 + (size_t)b.nbx * b.nby) * sizeof(unsigned);
}

static int run_colmax(hub_t h, const void* X, int ncol, int ld, unsigned* cmax, unsigned* bmax) {
    const BlockMap b = block_map(h, nullptr, 0);
    const int cw = h->cplx ? 2 : 1;
    ProfScope ps(h, HUB_K_COPY);
    for (int c0 = 0; c0 < ncol; c0 += 65535) {
        const dim3 grid(kColParts, (unsigned)std::min(65535, ncol - c0));
        unsigned* out = cmax + (size_t)c0 * kColParts;
        unsigned* map = bmax ? bmax + (size_t)c0 * kColParts * b.nbx * b.nby : nullptr;
        const size_t off = (size_t)c0 * ld * cw;
        if (h->esize == 8 && cw == 2) run_parts<double, 2>(h, grid, (const double*)X + off, 2L * ld, b, out, map);
        else if (h->esize == 8) run_parts<double, 1>(h, grid, (const double*)X + off, ld, b, out, map);
        else if (cw == 2) run_parts<float2, 1>(h, grid, (const float2*)X + off / 2, ld, b, out, map);
        else run_parts<float, 1>(h, grid, (const float*)X + off, ld, b, out, map);
    }
    HUB_CUDA_TRY(h, cudaGetLastError());
    return HUB_OK;
}

int launch_colmax_at(hub_t h, const void* X, int ncol, int ld, unsigned* cmax) { return run_colmax(h, X, ncol, ld, cmax, nullptr); }

int launch_colmax(hub_t h, const void* X, int ncol, int ld) {
    int rc;
    if ((rc = ensure(h, (void**)&h->d_cmax, &h->cmax_bytes, std::max(h->cmax_bytes, colmax_bytes(h, ncol))))) return rc;
    return run_colmax(h, X, ncol, ld, h->d_cmax, h->d_cmax + (size_t)ncol * kColParts);
}

}  // namespace hub

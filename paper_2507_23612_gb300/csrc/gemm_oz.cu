// Rayleigh-Ritz block products (CheFSI, Sec. II.B) of real FP64 blocks, and of real float blocks
// with float products, as digit products on the FP16 tensor cores (digits.cuh):
//
//   Gram / projected Hamiltonian  G = alpha A^T B    (A, B tall: Nd x m, Nd x n)
//   rotation                      Y = X Q            (X tall: Nd x k, Q small k x n)
//
// On CUDA cores the FP64 pipe (2 multiply-adds per clock and SM) bounds both: 80.1 and 140.4 ms on
// 650,496 x 348.  Here every operand is split into 7 (double) or 4 (float) 8-bit digits, the
// digit products are summed in FP32 accumulators, read out every 256 (512) terms, up to which the
// sums are exact where it counts (digits.cuh), and added up in 64-bit integers: the result carries
// the rounding of the operands to 54 (30) bits of their column's largest magnitude and one rounding
// of the sum.  (Every 512 terms the double forms took 0.5 ms less, of 4.5 and 3.2.)
//
// Both are D[128 x 64] = sum_k A[128, k] B[64, k]: rows and columns are orbitals and k the grid
// for the Gram product (k split over CTAs), rows are grid points, columns the new and k the old
// orbitals for the rotation.  In the rotation the column scales of X move into Q (a power of two
// per row), and the digits of one grid point share a scale over k, that of the orbitals there: a point
// where all of them are small keeps its bits.
//
// A conversion pass writes the digits in the order in which the MMAs read them (K-major, no
// swizzle: 16-byte units of 8 k; per 16 k and row tile one contiguous block), in panels of the
// grid, so that the product kernel's loads are plain bulk copies.  Digit i of A times digits
// 1 .. S + 1 - i of B (side by side along N) are one or two MMAs into the accumulators of the
// levels i .. S, as in the projector products.
//
// Kernel: warp 0 copies, warp 1 issues the MMAs, warps 2-9 read the accumulators (one TMEM lane
// quarter and 32 columns each) into 64-bit sums in registers.  Every mbarrier wait is bounded.
// Bound by the tensor pipe (28 digit products of FP64: 896 clocks per 16 k of a tile; 65 % busy on
// 88 x 88 x 28 x 128, with the digits at 71 % of the DRAM rate, the read-outs between): on
// 650,496 x 348 the symmetric Gram product takes 2.2 ms, the rotation 3.2 ms, the conversions
// 0.65 ms per operand (0.9 for the rotation's rows).
//
// Columns outside the digit format (non-finite or of extreme magnitude) are summed in plain FP64.
#include <algorithm>

#include "hub_internal.cuh"
#include "digits.cuh"
#include "tcgen05.cuh"

namespace hub {

namespace {

constexpr int MZ_M = 128, MZ_N = 64;
constexpr int MZ_THREADS = 320;
constexpr size_t MZ_PANEL = (size_t)1 << 30;        // bytes of one operand's digits per panel
constexpr size_t MZ_LEAST = (size_t)1 << 24;

template <typename R>
struct MCfg {
    static constexpr int S = Digits<R>::S;
    static constexpr int AB = S * MZ_M * 32, BB = S * MZ_N * 32;      // bytes of 16 k of a tile
    static constexpr int STAGE = AB + BB;
    static constexpr int NS = S == 7 ? 5 : 8;
    static constexpr int GROUP = S == 7 ? 16 : 32;      // 16-k steps per read-out of the accumulators
    // levels kept: one more than digits for float, because the first dropped level must not hold
    // squares (digit 3 times digit 3 of a column with itself adds up over the grid)
    static constexpr int L = S == 7 ? 7 : 5;
    static constexpr int ACC = L * MZ_N;
    static constexpr size_t SMEM = (size_t)NS * STAGE + 1024;
    static_assert(SMEM <= 227 * 1024 && ACC <= 512, "shared memory, TMEM");
};

struct MzArgs {
    const uint4* A;           // [k step][row tile of 128][digit][2][128] units of 8 k
    const uint4* B;           // [k step][column tile of 64][2][digit][64]
    int rt, ct;               // row and column tiles
    int ksteps;               // 16-k steps of this call
    // Gram product
    int tiles, splits, sym;
    int first;                // first panel: the partial sums start at zero
    longlong2* part;          // [split][tile][128 * 64] (low sum, high sum)
    // rotation
    void* Y;
    long ldy, row0, rows;     // rows row0 .. row0 + rows of Y
    int n;
    const int* escale;        // per column: exponent of the result; [n]: not covered
    const int* rexp;          // per row of the panel: its own, to be added
    const void* X;            // plain sums
    const double* Q;
    long ldx;
    int k;
    int* flags;
};

// tile t of the Gram product: rows 128 * i.x, columns 64 * i.y; a symmetric product has only the
// tiles that reach the diagonal or beyond
__device__ __forceinline__ int2 gram_tile(int t, int ct, int sym) {
    int it = 0, c = ct;
    while (t >= c) {
        t -= c;
        ++it;
        c = sym ? ct - 2 * it : ct;
    }
    return make_int2(it, (sym ? 2 * it : 0) + t);
}

// MODE 0: Gram product; 1: rotation
template <typename R, int MODE>
__global__ void __launch_bounds__(MZ_THREADS, 1)
k_mm_oz(const __grid_constant__ MzArgs a) {
    using C = MCfg<R>;
    constexpr int S = C::S;
    extern __shared__ __align__(1024) unsigned char dsm[];
    unsigned char* ring = reinterpret_cast<unsigned char*>((reinterpret_cast<uintptr_t>(dsm) + 1023) & ~(uintptr_t)1023);
    __shared__ __align__(8) uint64_t full_bar[C::NS], empty_bar[C::NS], tfull_bar, tempty_bar, done_bar;
    __shared__ uint32_t tmem_slot;
    __shared__ volatile int abort_flag;
    __shared__ int issued_sh;

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    // units of this CTA: one (tile, k range) of the Gram product; the (row tile, column tile) pairs
    // blockIdx.x, + gridDim.x, ... of the rotation, column tiles next to each other (A from L2)
    int2 tile = make_int2(0, 0);
    int ks0 = 0, ks1 = a.ksteps, nu = 1;
    if (MODE == 0) {
        tile = gram_tile(blockIdx.x % a.tiles, a.ct, a.sym);
        const int sp = blockIdx.x / a.tiles;
        ks0 = (int)((long)a.ksteps * sp / a.splits);
        ks1 = (int)((long)a.ksteps * (sp + 1) / a.splits);
    } else {
        const int all = a.rt * a.ct;
        nu = (all - (int)blockIdx.x + (int)gridDim.x - 1) / (int)gridDim.x;
    }
    auto unit = [&](int uu) {
        if (MODE == 0) return tile;
        const int u = (int)blockIdx.x + uu * (int)gridDim.x;
        return make_int2(u / a.ct, u % a.ct);
    };
    const int nk = ks1 - ks0, ngr = (nk + C::GROUP - 1) / C::GROUP;   // groups per unit

    if (threadIdx.x == 0) {
        abort_flag = 0;
        issued_sh = 0;
        for (int s = 0; s < C::NS; ++s) {
            mbar_init(&full_bar[s], 1);
            mbar_init(&empty_bar[s], 1);
        }
        mbar_init(&tfull_bar, 1);
        mbar_init(&tempty_bar, 256);
        mbar_init(&done_bar, 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(saddr(&tmem_slot)),
                     "r"(512u) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = tmem_slot;

    if (warp == 0) {
        if (lane == 0) {
            int i = 0, s = 0, ph = 1;                 // ph: parity of the stage's previous release
            bool stop = false;
            for (int uu = 0; uu < nu && !stop; ++uu) {
                const int2 t = unit(uu);
                const uint4* pa = a.A + ((size_t)ks0 * a.rt + t.x) * (C::AB / 16);
                const uint4* pb = a.B + ((size_t)ks0 * a.ct + t.y) * (C::BB / 16);
                for (int c = 0; c < nk; ++c, ++i) {
                    if (i >= C::NS && !mbar_wait(&empty_bar[s], ph, &abort_flag)) { stop = true; break; }
                    unsigned char* st = ring + (size_t)s * C::STAGE;
                    mbar_expect_tx(&full_bar[s], C::STAGE);
                    bulk_load(st, pa, C::AB, &full_bar[s]);
                    bulk_load(st + C::AB, pb, C::BB, &full_bar[s]);
                    issued_sh = i + 1;
                    pa += (size_t)a.rt * (C::AB / 16);
                    pb += (size_t)a.ct * (C::BB / 16);
                    if (++s == C::NS) { s = 0; ph ^= 1; }
                }
            }
        }
    } else if (warp == 1) {
        const bool el = elect_one();
        auto wait = [&](uint64_t* bar, int parity) { return __all_sync(0xffffffffu, mbar_wait(bar, parity, &abort_flag)) != 0; };
        const uint32_t a0 = desc_lo(ring, MZ_M * 16), b0 = desc_lo(ring + C::AB, S * MZ_N * 16);
        int s = 0, ph = 0, gi = 0;
        bool stop = false;
        for (int uu = 0; uu < nu && !stop; ++uu)
            for (int c0 = 0; c0 < nk && !stop; c0 += C::GROUP, ++gi) {
                if (gi >= 1 && !wait(&tempty_bar, (gi - 1) & 1)) { stop = true; break; }
                tc_fence_after();
                const int c1 = min(nk, c0 + C::GROUP);
                for (int c = c0; c < c1; ++c) {
                    if (!wait(&full_bar[s], ph)) { stop = true; break; }
                    tc_fence_after();
                    if (el) {
                        const uint32_t ao = a0 + (uint32_t)(s * (C::STAGE / 16)), bo = b0 + (uint32_t)(s * (C::STAGE / 16));
                        const uint32_t acc = c > c0 ? 1u : 0u;
#pragma unroll
                        for (int d = 0; d < S; ++d) {
                            // digit d of A times the digits of B that reach level L at most, in pieces
                            // of at most 256 columns; the piece that meets its levels first clears
                            // them (digit 0 the first S, digit 1 the extra one)
                            constexpr int kMax = 256;
                            const int n = (S < C::L - d ? S : C::L - d) * MZ_N;
                            const int cut = n > kMax ? kMax : (d == 1 && C::L > S ? n - MZ_N : n);
                            mma_f16_lo(tmem + (uint32_t)(d * MZ_N), ao + (uint32_t)(d * 2 * MZ_M), bo, kDescHi,
                                       instr_desc_f16(MZ_M, cut), d > 0 ? 1u : acc);
                            if (n > cut)
                                mma_f16_lo(tmem + (uint32_t)(d * MZ_N + cut), ao + (uint32_t)(d * 2 * MZ_M), bo + (uint32_t)cut, kDescHi,
                                           instr_desc_f16(MZ_M, n - cut), d == 0 || C::L > S ? acc : 1u);
                        }
                        mma_commit(&empty_bar[s]);
                    }
                    __syncwarp();
                    if (++s == C::NS) { s = 0; ph ^= 1; }
                }
                if (el && !stop) mma_commit(&tfull_bar);
            }
        if (el) mma_commit(&done_bar);
    } else {
        // warps 2-9: TMEM lanes 32 (warp % 4) .. + 31, columns 32 half .. + 31 of the tile
        const int quad = warp & 3, half = (warp - 2) >> 2;
        const uint32_t lane_base = (uint32_t)(32 * quad) << 16;
        const int row = 32 * quad + lane;
        int gi = 0;
        bool stop = false;
        for (int uu = 0; uu < nu && !stop; ++uu) {
            const int2 t = unit(uu);
            long long hs[32], ls[32];
#pragma unroll
            for (int c = 0; c < 32; ++c) hs[c] = ls[c] = 0;
            for (int g = 0; g < ngr; ++g, ++gi) {
                const bool ok = mbar_wait(&tfull_bar, gi & 1, &abort_flag);
                if (__any_sync(0xffffffffu, !ok)) { stop = true; break; }
                tc_fence_after();
#pragma unroll
                for (int c0 = 0; c0 < 32; c0 += 8) {
                    uint32_t v[C::L * 8];
                    tmem_levels<C::L, MZ_N, 8>(tmem + lane_base + (uint32_t)(half * 32 + c0), v);
#pragma unroll
                    for (int f = 0; f < 8; ++f) {
                        long long lo;
                        hs[c0 + f] += level_sum<R, 8>(v + f, &lo);
                        ls[c0 + f] += S == 7 ? lo : (long long)__float2int_rn(__uint_as_float(v[8 * (C::L - 1) + f]));
                    }
                }
                tc_fence_before();
                mbar_arrive(&tempty_bar);
            }
            if (stop) break;
            if constexpr (MODE == 0) {
                longlong2* p = a.part + ((size_t)blockIdx.x * MZ_M + row) * MZ_N + half * 32;
#pragma unroll
                for (int c = 0; c < 32; ++c) {
                    longlong2 s = a.first ? make_longlong2(0, 0) : p[c];
                    s.x += ls[c];
                    s.y += hs[c];
                    p[c] = s;
                }
            } else {
                const long r = (long)t.x * MZ_M + row;
                const bool plain = a.escale[a.n] != 0;
                if (r < a.rows) {
                    const int re = a.rexp[r];
                    R* y = (R*)a.Y + a.row0 + r;
#pragma unroll
                    for (int c = 0; c < 32; ++c) {
                        const int col = t.y * MZ_N + half * 32 + c;
                        if (col >= a.n) continue;
                        double v;
                        if (plain) {
                            v = 0.0;
                            const R* x = (const R*)a.X + a.row0 + r;
                            for (int k = 0; k < a.k; ++k) v = fma((double)x[(size_t)k * a.ldx], a.Q[(size_t)k * a.n + col], v);
                        } else if constexpr (S == 7) {
                            // hs 2^24 + ls, rounded once: |hs| < 2^46 per 512 terms
                            v = a.k <= 512 ? scale2((double)((hs[c] << 14) + ((ls[c] + 512) >> 10)), a.escale[col] + 10 + re)
                                           : scale2(fma((double)hs[c], 16777216.0, (double)ls[c]), a.escale[col] + re);
                        } else {
                            v = scale2((double)((hs[c] << 8) + ls[c]), a.escale[col] - 8 + re);
                        }
                        y[(size_t)col * a.ldy] = (R)v;
                    }
                }
            }
        }
    }
    __syncwarp();
    __syncthreads();
    if (threadIdx.x == 0) {
        if (!mbar_drain(&done_bar, 0)) abort_flag = 1;
        if (abort_flag) {
            atomicExch(a.flags + FLAG_TIMEOUT, 1);
            const int issued = issued_sh;
            for (int j = issued > C::NS ? issued - C::NS : 0; j < issued; ++j)
                mbar_drain(&full_bar[j % C::NS], (j / C::NS) & 1);
        }
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 0) {
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(512u) : "memory");
    }
}

// ---------------------------------------------------------------------------- conversion
template <typename R>
__device__ __forceinline__ int column_exponent(const unsigned* cmax, int col) {
    return (int)(column_max(cmax, col) >> (sizeof(R) == 8 ? 20 : 23));
}
template <typename R>
__device__ __forceinline__ bool covered(int E) { return E >= Digits<R>::kEmin && E <= Digits<R>::kEmax; }

// the digits of 8 numbers as S 16-byte units
template <typename R>
__device__ __forceinline__ void put_digits(const typename Digits<R>::I (&b)[8], uint4* dst, size_t step) {
#pragma unroll
    for (int d = 0; d < Digits<R>::S; ++d) {
        __half2 o[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) o[k] = digit_pair<R>(b[2 * k], b[2 * k + 1], d);
        dst[d * step] = *reinterpret_cast<uint4*>(o);
    }
}

// Gram product: rows g0 .. g0 + 8 units of all columns, k = grid; A form (128-column tiles) and /
// or B form (64-column tiles).  Lanes are neighbouring columns (the units of 32 columns are
// contiguous); a lane reads 8 consecutive points.
template <typename R>
__global__ void __launch_bounds__(256)
k_digits_tall(const R* __restrict__ X, long ld, long Nd, int ncol, long g0, int units, const unsigned* __restrict__ cmax,
              uint4* __restrict__ A, int rt, uint4* __restrict__ B, int ct, int vec) {
    constexpr int S = Digits<R>::S;
    const int lane = threadIdx.x & 31, col = blockIdx.y * 32 + lane;
    const int u = blockIdx.x * 8 + (threadIdx.x >> 5);              // unit of 8 points
    if (u >= units) return;
    int E = col < ncol ? column_exponent<R>(cmax, col) : 0;
    if (!covered<R>(E)) E = 1 << 14;                               // all digits zero
    const long g = g0 + (long)u * 8;
    const R* x = X + (size_t)(col < ncol ? col : 0) * ld;
    R v[8];
    if (vec && g + 8 <= Nd) {
#pragma unroll
        for (int i = 0; i < 8 * (int)sizeof(R) / 16; ++i)
            *reinterpret_cast<uint4*>(v + i * (16 / (int)sizeof(R))) = *reinterpret_cast<const uint4*>(x + g + i * (16 / (int)sizeof(R)));
    } else {
#pragma unroll
        for (int i = 0; i < 8; ++i) v[i] = g + i < Nd ? x[g + i] : R(0);
    }
    typename Digits<R>::I b[8];
#pragma unroll
    for (int i = 0; i < 8; ++i) b[i] = Digits<R>::bytes(v[i], E);
    const int step = u >> 1, kc = u & 1;
    if (A) put_digits<R>(b, A + (((size_t)step * rt + (col >> 7)) * S * 2 + kc) * MZ_M + (col & 127), 2 * MZ_M);
    if (B && col < ct * MZ_N) put_digits<R>(b, B + ((size_t)step * ct + (col >> 6)) * (2 * S * MZ_N) + (size_t)kc * S * MZ_N + (col & 63), MZ_N);
}

// Rotation: rows r0 .. of X, k = orbital (A form, 128-row tiles).  A CTA takes 32 rows: the largest
// exponent of each relative to its columns' (rexp), then the digits, 8 orbitals per thread (the second
// read comes from the caches: 32 x 348 doubles are 89 KB)
template <typename R>
__global__ void __launch_bounds__(256)
k_digits_rows(const R* __restrict__ X, long ld, int k, long r0, long rows, int rt, const unsigned* __restrict__ cmax,
              uint4* __restrict__ A, int* __restrict__ rexp) {
    constexpr int S = Digits<R>::S;
    extern __shared__ int cexp[];
    __shared__ int tops[8][32];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const long r = (long)blockIdx.x * 32 + lane;
    for (int c = threadIdx.x; c < k; c += 256) {
        const int E = column_exponent<R>(cmax, c);
        cexp[c] = covered<R>(E) ? E : 1 << 14;
    }
    __syncthreads();
    const bool in = r < rows;
    const R* x = X + r0 + (in ? r : 0);
    int top = -(1 << 16);
    int c = warp;
    for (; c + 24 < k; c += 32) {
        R v[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) v[i] = x[(size_t)(c + 8 * i) * ld];
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const int e = Digits<R>::exponent(v[i]);
            if (e > 0) top = max(top, e - cexp[c + 8 * i]);
        }
    }
    for (; c < k; c += 8) {
        const int e = Digits<R>::exponent(x[(size_t)c * ld]);
        if (e > 0) top = max(top, e - cexp[c]);
    }
    tops[warp][lane] = top;
    __syncthreads();
#pragma unroll
    for (int w = 0; w < 8; ++w) top = max(top, tops[w][lane]);
    if (top < -(1 << 13)) top = 0;                                     // nothing but zeros and columns not covered
    if (warp == 0 && r < (long)rt * MZ_M) rexp[r] = top;
    for (int u = warp; u < (k + 15) / 16 * 2; u += 8) {
        R v[8];
        typename Digits<R>::I b[8];
#pragma unroll
        for (int i = 0; i < 8; ++i) v[i] = 8 * u + i < k && in ? x[(size_t)(8 * u + i) * ld] : R(0);
#pragma unroll
        for (int i = 0; i < 8; ++i)
            b[i] = Digits<R>::exponent(v[i]) > 0 ? Digits<R>::bytes(v[i], cexp[8 * u + i] + top) : Digits<R>::kZero;
        put_digits<R>(b, A + (((size_t)(u >> 1) * rt + (r >> 7)) * S * 2 + (u & 1)) * MZ_M + (r & 127), 2 * MZ_M);
    }
}

// Q (double, row-major k x n) times the column scales of X, as B form digits; one warp per column.
// escale[col]: exponent of the result; escale[n]: set when a column of X or Q is not covered
// (cleared before).  The digits of Q have as many bits as those of X.
template <typename R>
__global__ void __launch_bounds__(128)
k_digits_q(const double* __restrict__ Q, int k, int n, int ct, const unsigned* __restrict__ cmax, uint4* __restrict__ B,
           int* __restrict__ escale) {
    constexpr int S = Digits<R>::S;
    const int col = blockIdx.x * 4 + (threadIdx.x >> 5), lane = threadIdx.x & 31;
    if (col >= ct * MZ_N) return;
    int top = 0;
    bool bad = false;
    for (int c = lane; c < k; c += 32) {
        const int E = column_exponent<R>(cmax, c);
        bad |= E != 0 && !covered<R>(E);
        const int e = col < n ? Digits<double>::exponent(Q[(size_t)c * n + col]) : 0;
        bad |= e == 0x7ff;
        if (e > 0 && E > 0) top = max(top, e + E);
    }
    top = __reduce_max_sync(0xffffffffu, top);
    bad = __any_sync(0xffffffffu, bad) != 0;
    if (lane == 0 && col < n) {
        // x = X 2^(E - unit), q 2^E = Qd 2^(top - 1076); 256^(S - 1) of the level sums
        escale[col] = top == 0 ? 0 : 8 * (S - 1) + top - Digits<R>::kUnit - (S == 7 ? 1076 : 1052);
        if (bad) atomicExch(escale + n, 1);
    }
    for (int u = lane; u < (k + 15) / 16 * 2; u += 32) {
        typename Digits<R>::I b[8];
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            const int c = 8 * u + i;
            const double q = c < k && col < n ? Q[(size_t)c * n + col] : 0.0;
            const int E = c < k ? column_exponent<R>(cmax, c) : 0;
            const unsigned long long w = Digits<double>::exponent(q) > 0 && E > 0 && top > 0 ?    // a denormal q has no part in top
                                              Digits<double>::bytes(q, top, E) : Digits<double>::kZero;
            if constexpr (S == 7) b[i] = w;
            else b[i] = (unsigned)(((long long)(w - Digits<double>::kZero) + (1 << 23)) >> 24) + Digits<float>::kZero;
        }
        put_digits<R>(b, B + ((size_t)(u >> 1) * ct + (col >> 6)) * (2 * S * MZ_N) + (size_t)(u & 1) * S * MZ_N + (col & 63), MZ_N);
    }
}

// G = alpha times the sum of the partial integers over the splits.  A CTA takes 32 entries, 8 threads
// of different warps an eighth of the splits each (one thread per entry took 29 us for a 48 x 48
// product of 152 splits: a serial chain of loads).  Columns that are not covered by plain sums over
// the grid (block-wide, one element after another).
template <typename R>
__global__ void __launch_bounds__(256)
k_gram_oz_reduce(const longlong2* __restrict__ part, int tiles, int splits, int ct, int sym, int m, int n, double alpha,
                 const unsigned* __restrict__ cmaxA, const unsigned* __restrict__ cmaxB, const R* __restrict__ A, long lda,
                 const R* __restrict__ B, long ldb, long Nd, double* __restrict__ G) {
    __shared__ longlong2 sums[8][32];
    __shared__ double red[8];
    __shared__ int odd_sh[32];
    __shared__ int nodd;
    const int lane = threadIdx.x & 31, part8 = threadIdx.x >> 5;
    const long t = (long)blockIdx.x * 32 + lane;
    int i = (int)(t / n), j = (int)(t % n);
    if (sym && j < i) { const int q = i; i = j; j = q; }
    if (threadIdx.x == 0) nodd = 0;
    if (t < (long)m * n) {
        const int it = i / MZ_M, jt = j / MZ_N;
        // tiles before row tile it: ct per row tile, or ct - 2 i of a symmetric product
        const int tile = sym ? it * ct - it * (it - 1) + (jt - 2 * it) : it * ct + jt;
        const longlong2* p = part + ((size_t)tile * MZ_M + (i & 127)) * MZ_N + (j & 63);
        longlong2 s = make_longlong2(0, 0);
#pragma unroll 4
        for (int z = part8; z < splits; z += 8) {
            const longlong2 v = p[(size_t)z * tiles * MZ_M * MZ_N];
            s.x += v.x;
            s.y += v.y;
        }
        sums[part8][lane] = s;
    }
    __syncthreads();
    if (part8 == 0 && t < (long)m * n) {
        const int Ei = column_exponent<R>(cmaxA, i), Ej = column_exponent<R>(cmaxB, j);
        if ((Ei == 0 || covered<R>(Ei)) && (Ej == 0 || covered<R>(Ej))) {
            long long lo = 0, hi = 0;
#pragma unroll
            for (int z = 0; z < 8; ++z) { lo += sums[z][lane].x; hi += sums[z][lane].y; }
            // hi 2^24 + lo (double), hi + lo / 256 (float)
            const double v = Digits<R>::S == 7 ? fma((double)hi, 16777216.0, (double)lo) : fma((double)lo, 0.00390625, (double)hi);
            G[t] = Ei == 0 || Ej == 0 ? 0.0 : alpha * scale2(v, 8 * (Digits<R>::S - 1) + Ei + Ej - 2 * Digits<R>::kUnit);
        } else {
            odd_sh[atomicAdd(&nodd, 1)] = lane;
        }
    }
    __syncthreads();
    for (int o = 0; o < nodd; ++o) {
        const long e = (long)blockIdx.x * 32 + odd_sh[o];
        const R* x = A + (size_t)(e / n) * lda;
        const R* y = B + (size_t)(e % n) * ldb;
        double s = 0.0;
        for (long g = threadIdx.x; g < Nd; g += 256) s = fma((double)x[g], (double)y[g], s);
        for (int k = 16; k > 0; k >>= 1) s += __shfl_down_sync(0xffffffffu, s, k);
        if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = s;
        __syncthreads();
        if (threadIdx.x == 0) {
            for (int k = 1; k < 8; ++k) s += red[k];
            G[e] = alpha * s;
        }
        __syncthreads();
    }
}

// ---------------------------------------------------------------------------- host
// room for the digits of `per` steps or, where there is less, of fewer (panels of 8 MB are the least
// that are tried)
bool claim_panel(hub_t h, long& per, size_t step, size_t fixed) {
    while (!claim(h, &h->d_bf16, &h->bf16_bytes, (size_t)per * step + fixed)) {
        if (per == 1 || (size_t)per * step < MZ_LEAST) return false;
        per = (per + 1) / 2;
    }
    return true;
}

template <typename R>
int gram_oz(hub_t h, const void* A, int lda, const void* B, int ldb, int m, int n, double alpha, bool sym, double* G) {
    using C = MCfg<R>;
    int rc;
    const long Nd = h->Nd;
    const bool same = A == B && lda == ldb && m == n;
    const int rt = (m + MZ_M - 1) / MZ_M, ct = (n + MZ_N - 1) / MZ_N;
    int tiles = 0;
    for (int it = 0; it < rt; ++it) tiles += sym ? ct - 2 * it : ct;
    const int splits = std::max(1, h->num_sms / tiles);
    // panels of whole 16-point steps
    const size_t stepA = (size_t)rt * C::AB, stepB = (size_t)ct * C::BB;
    const long steps = (Nd + 15) / 16;
    long per = std::max<long>(1, std::min<long>(steps, (long)(MZ_PANEL / std::max(stepA, stepB))));
    // column maxima: A's, then B's
    if (!claim(h, (void**)&h->d_cmax, &h->cmax_bytes, (size_t)(m + n) * kColParts * sizeof(unsigned)) ||
        !claim(h, &h->d_gpart, &h->gpart_bytes, (size_t)splits * tiles * MZ_M * MZ_N * sizeof(longlong2)) ||
        !claim_panel(h, per, stepA + stepB, 0)) return HUB_ENOMEM;
    unsigned* cmB = h->d_cmax + (same ? 0 : (size_t)m * kColParts);
    if ((rc = launch_colmax_at(h, A, m, lda, h->d_cmax))) return rc;
    if (!same && (rc = launch_colmax_at(h, B, n, ldb, cmB))) return rc;
    uint4* dA = (uint4*)h->d_bf16;
    uint4* dB = dA + (size_t)per * stepA / 16;
    MzArgs a{};
    a.A = dA;
    a.B = dB;
    a.rt = rt;
    a.ct = ct;
    a.tiles = tiles;
    a.splits = splits;
    a.sym = sym;
    a.part = (longlong2*)h->d_gpart;
    a.flags = h->d_flags;
    HUB_CUDA_TRY(h, cudaFuncSetAttribute(k_mm_oz<R, 0>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)C::SMEM));
    auto vec = [](const void* p, long ld) { return (int)((uintptr_t)p % 16 == 0 && (ld * (long)sizeof(R)) % 16 == 0); };
    for (long s0 = 0; s0 < steps; s0 += per) {
        const int ns = (int)std::min(per, steps - s0), units = 2 * ns;
        {
            ProfScope ps(h, HUB_K_COPY);
            k_digits_tall<R><<<dim3((units + 7) / 8, rt * 4), 256, 0, h->stream>>>(
                (const R*)A, lda, Nd, m, s0 * 16, units, h->d_cmax, dA, rt, same ? dB : nullptr, ct, vec(A, lda));
        }
        if (!same) {
            ProfScope ps(h, HUB_K_COPY);
            k_digits_tall<R><<<dim3((units + 7) / 8, ct * 2), 256, 0, h->stream>>>(
                (const R*)B, ldb, Nd, n, s0 * 16, units, cmB, nullptr, 0, dB, ct, vec(B, ldb));
        }
        HUB_CUDA_TRY(h, cudaGetLastError());
        a.ksteps = ns;
        a.first = s0 == 0;
        ProfScope ps(h, HUB_K_GRAM);
        k_mm_oz<R, 0><<<tiles * splits, MZ_THREADS, C::SMEM, h->stream>>>(a);
        HUB_CUDA_TRY(h, cudaGetLastError());
    }
    ProfScope ps(h, HUB_K_GRAM_REDUCE);
    k_gram_oz_reduce<R><<<(unsigned)(((long)m * n + 31) / 32), 256, 0, h->stream>>>(
        a.part, tiles, splits, ct, sym, m, n, alpha, h->d_cmax, cmB, (const R*)A, lda, (const R*)B, ldb, Nd, G);
    HUB_CUDA_TRY(h, cudaGetLastError());
    return HUB_OK;
}

template <typename R>
int rotate_oz(hub_t h, const void* X, int ldx, const double* Q, int k, int n, void* Y, int ldy) {
    using C = MCfg<R>;
    int rc;
    const long Nd = h->Nd;
    const int ct = (n + MZ_N - 1) / MZ_N, ks = (k + 15) / 16;
    const size_t perTile = (size_t)ks * C::AB + MZ_M * sizeof(int), nB = (size_t)ks * ct * C::BB;
    const long tilesAll = (Nd + MZ_M - 1) / MZ_M;
    long per = std::max<long>(1, std::min<long>(tilesAll, (long)(MZ_PANEL / perTile)));
    if (k > 12000) return HUB_ENOMEM;                 // the columns' exponents in shared memory
    const size_t nE = ((size_t)(n + 1) * sizeof(int) + 255) / 256 * 256;
    if (!claim(h, (void**)&h->d_cmax, &h->cmax_bytes, (size_t)k * kColParts * sizeof(unsigned)) ||
        !claim_panel(h, per, perTile, nB + nE)) return HUB_ENOMEM;
    if ((rc = launch_colmax_at(h, X, k, ldx, h->d_cmax))) return rc;
    uint4* dA = (uint4*)h->d_bf16;
    uint4* dB = dA + (size_t)per * ks * C::AB / 16;
    int* esc = (int*)((char*)dB + nB);
    int* rexp = (int*)((char*)esc + nE);
    HUB_CUDA_TRY(h, cudaMemsetAsync(esc + n, 0, sizeof(int), h->stream));
    {
        ProfScope ps(h, HUB_K_COPY);
        k_digits_q<R><<<(ct * MZ_N + 3) / 4, 128, 0, h->stream>>>(Q, k, n, ct, h->d_cmax, dB, esc);
    }
    HUB_CUDA_TRY(h, cudaGetLastError());
    MzArgs a{};
    a.A = dA;
    a.B = dB;
    a.ct = ct;
    a.ksteps = ks;
    a.Y = Y;
    a.ldy = ldy;
    a.n = n;
    a.escale = esc;
    a.rexp = rexp;
    a.X = X;
    a.Q = Q;
    a.ldx = ldx;
    a.k = k;
    a.flags = h->d_flags;
    HUB_CUDA_TRY(h, cudaFuncSetAttribute(k_mm_oz<R, 1>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)C::SMEM));
    for (long t0 = 0; t0 < tilesAll; t0 += per) {
        a.rt = (int)std::min(per, tilesAll - t0);
        a.row0 = t0 * MZ_M;
        a.rows = std::min<long>((long)a.rt * MZ_M, Nd - a.row0);
        {
            ProfScope ps(h, HUB_K_COPY);
            k_digits_rows<R><<<(unsigned)(a.rt * (MZ_M / 32)), 256, (size_t)k * sizeof(int), h->stream>>>(
                (const R*)X, ldx, k, a.row0, a.rows, a.rt, h->d_cmax, dA, rexp);
        }
        HUB_CUDA_TRY(h, cudaGetLastError());
        ProfScope ps(h, HUB_K_ROTATE);
        k_mm_oz<R, 1><<<(int)std::min<long>((long)a.rt * ct, h->num_sms), MZ_THREADS, C::SMEM, h->stream>>>(a);
        HUB_CUDA_TRY(h, cudaGetLastError());
    }
    return HUB_OK;
}

}  // namespace

int launch_gram_oz(hub_t h, const void* A, int lda, const void* B, int ldb, int m, int n, double alpha, bool sym, double* G) {
    return h->esize == 8 ? gram_oz<double>(h, A, lda, B, ldb, m, n, alpha, sym, G)
                         : gram_oz<float>(h, A, lda, B, ldb, m, n, alpha, sym, G);
}
int launch_rotate_oz(hub_t h, const void* X, int ldx, const double* Q, int k, int n, void* Y, int ldy) {
    return h->esize == 8 ? rotate_oz<double>(h, X, ldx, Q, k, n, Y, ldy) : rotate_oz<float>(h, X, ldx, Q, k, n, Y, ldy);
}

}  // namespace hub

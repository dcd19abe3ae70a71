// Real FP64 stencil in integer arithmetic.  GB300 issues 2 FP64 operations per clock and SM
// but about 30 32x32+64-bit integer multiply-adds and 110 32-bit adds, so the ~39 FP64
// operations per point of the floating-point form (17.15 ms on 88 x 88 x 84 x 348, 0.82 of
// the FP64 pipe) cost several times what the same sum costs in fixed point.
//
//   Yout = alpha * (-1/2 Lap_h Y + V .* Y - shift * Y) + beta * Yprev        (Sec. II.B)
//
// Number format.  Every CTA has one power-of-two scale: with E the biased exponent of the largest
// |x| of the pieces (32 x 8 points of an eighth of the planes, colmax.cu) that its points and their
// neighbours lie in, X = x * 2^(1081 - E) rounded to nearest, |X| < 2^59.  An element keeps all 53
// bits down to 2^-6 of that maximum and is never off by more than 2^-59 of it: one FP64 rounding of
// the sum, which holds terms of ~300 x, is larger.  A column may decay by any factor over the cell;
// only elements more than 2^-6 below others within some 70 x 30 x n3 / 4 points have fewer bits.  (One
// scale per column, whose far tails would be cut to zero, takes 4.25 ms below.)
// X is kept as two signed limbs, X = xh 2^30 + xl: pair sums of limbs need no carry.
// The Laplacian weights of order 2 n0 are rational: c_p = k_p / lcd with integers k_p of 22
// bits, so A_a = k_0 X + sum_p k_p (X_{+p} + X_{-p}) of each axis is exact, and only
// F_a = -1 / (2 lcd h_a^2) and V - shift are rounded (to 59 bits):
//   U_a = A_a >> 20 (62 bits),  Z = sum_a (U_a Fq_a) >> 61 + (X (V - shift)q) >> 56,
// one 64-bit integer per point, converted once; alpha and beta enter in FP64 (three FP64
// operations per point).  sf fixes the binary points: Fq = F 2^sf, Z counts x-units of
// 2^(81 - sf), (V - shift)q = (V - shift) 2^(sf - 25); it is as large as the sums' 64 bits
// allow: 57 to 59 bits of the largest F, fewer where |V| would pass 2^(83 - sf) (k_fx_veff).  F is
// rounded at 2^-54 of itself or less, as the weights of the FP64 form are, and V at 2^-54 of the
// largest kinetic energy or 2^-58 of the largest |V|.
// What the format does not cover (columns that are zero or below 2^-900, CTAs with elements that are
// not finite or above 2^900), potentials
// that would leave F under 53 bits (8192 Ha at 0.3 bohr, 8 Ha at 10) and shifts beyond
// 2^(83 - sf) Ha (the largest kinetic energy of the grid, at least) are computed by fx_slow in
// plain FP64.
//
// Kernel: one CTA owns a tile of the x-y plane of one column and marches along z.  A ring of 8
// planes (with a halo of 6 in x and y) in shared memory holds the limbs; plane z + 7 is
// converted and stored while plane z is computed, and plane z + 8 is in flight in registers, so
// there is one barrier per plane.  The 13 z-neighbours live in registers.  Bound by instruction
// issue (50 multiply-adds at half rate and ~310 other instructions per point: 62 % of the issue
// slots, ALU pipe 44 %, multiply-adds 32 %, DRAM 9 % on 88 x 88 x 28 x 128, waits for loads and for
// the plane barriers between); 17.15 -> 4.35 ms on 88 x 88 x 84 x 348 (DRAM floor 0.80 ms), plus
// 0.27 ms for the maxima.
#include <algorithm>
#include <cmath>

#include "hub_internal.cuh"
#include "grid_sum.cuh"

namespace hub {

namespace {

constexpr int FXH = 6;             // halo
constexpr int FXP = 44;            // row pitch of a plane in shared memory: tiles of at most 32 points
constexpr int FXS = 8;             // ring planes
constexpr int kFxEmin = 123, kFxEmax = 1923;

struct FxArgs {
    const double* Y;
    const double* Yprev;
    double* Yout;
    const double* V;
    const int2* Vq;               // (V 2^(sf - 25)) as limbs of 30 bits
    const int* vinfo;             // largest high word of |V|; not covered (0 or 1); sf
    const unsigned* cmax;         // column maxima and pieces (colmax.cu)
    BlockMap bmax;
    int n1, n2, n3, ld;
    int tx, ty, tilesx, tiles;    // tile shape and count
    int zchunk, nzc;
    int k[FXH + 1];               // integer weights, k[0] the centre
    double F[3], Flo[3];          // F = F + Flo
    double alpha, beta, shift;
    const double* coef;           // device {alpha, beta, shift} or nullptr
    double w[3][FXH], cen;        // FP64 weights (alpha = 1) of the slow form
    double* dot;                  // StencilDot
    double* part;
    unsigned* counter;
};

__device__ __forceinline__ int wrap(int i, int n) {      // i is at most a few n away
    while (i < 0) i += n;
    while (i >= n) i -= n;
    return i;
}

// x to nearest as limbs; e20 the biased exponent of the column's maximum << 20 (at least 123, so
// that a denormal x shifts to zero whatever its hidden bit).  (Cut towards zero, elements are off by
// up to twice as much and all to one side; the rounding costs 3 of a point's ~25 instructions.)
__device__ __forceinline__ int2 to_limbs(double v, int e20) {
    const unsigned hi = (unsigned)__double2hiint(v), lo = (unsigned)__double2loint(v);
    const int s = min((e20 - (int)(hi & 0x7ff00000u)) >> 20, 61) + 1;
    // the significand times 2^8, 61 bits: X = (t >> s, to half a unit) / 2 up
    const unsigned th = __funnelshift_l(lo, (hi & 0xfffffu) | 0x100000u, 8), tl = lo << 8;
    const unsigned long long t = ((((unsigned long long)th << 32) | tl) >> s) + 1;
    const int xl = (int)((unsigned)(t >> 1) & 0x3fffffffu), xh = (int)(t >> 31);
    return (int)hi < 0 ? make_int2(-xh, -xl) : make_int2(xh, xl);
}

// the plain FP64 form of one tile and chunk, straight from global memory; returns this thread's sum
// of Y * Yout
__device__ __noinline__ double fx_slow(const FxArgs& a, const double* __restrict__ Y, const double* Yp, double* Yo, int gx0,
                                     int gy0, int z0, int z1, double alpha, double beta, double shift) {
    const long plane = (long)a.n1 * a.n2;
    const int per = a.tx * a.ty;
    double dot = 0.0;
    for (int i = threadIdx.x; i < per * (z1 - z0); i += blockDim.x) {
        const int z = z0 + i / per, x = gx0 + i % per % a.tx, y = gy0 + i % per / a.tx;
        if (x >= a.n1 || y >= a.n2) continue;
        const long g = x + (long)a.n1 * y + plane * z;
        double acc = (a.cen - shift + a.V[g]) * Y[g];
        for (int p = 1; p <= FXH; ++p) {
            if (a.k[p] == 0) break;               // orders below 12
            acc = fma(a.w[2][p - 1], Y[g + (wrap(z + p, a.n3) - z) * plane] + Y[g + (wrap(z - p, a.n3) - z) * plane], acc);
            acc = fma(a.w[0][p - 1], Y[g + wrap(x + p, a.n1) - x] + Y[g + wrap(x - p, a.n1) - x], acc);
            acc = fma(a.w[1][p - 1], Y[g + (long)(wrap(y + p, a.n2) - y) * a.n1] + Y[g + (long)(wrap(y - p, a.n2) - y) * a.n1], acc);
        }
        acc *= alpha;
        Yo[g] = Yp ? fma(beta, Yp[g], acc) : acc;
        dot = fma(Y[g], acc, dot);
    }
    return dot;
}

// first piece and number of pieces of 2^log points that [lo, hi) of a periodic axis meets (lo >= -FXH);
// all of them where it reaches around to its own first piece
__device__ __forceinline__ int2 pieces(int lo, int hi, int n, int count, int log) {
    if (hi - lo + (1 << log) > n) return make_int2(0, count);
    const int a = (lo < 0 ? lo + n : lo) >> log, b = (hi > n ? hi - n - 1 : hi - 1) >> log;
    return make_int2(a, b >= a ? b - a + 1 : b - a + 1 + count);
}
// largest leading word of the pieces that meet a box: the same in every warp (a lane takes a z part
// and every fourth piece along y), without a barrier
__device__ __forceinline__ unsigned region_max(const BlockMap& b, int col, int x0, int x1, int n1, int y0, int y1, int n2, int z0,
                                               int z1, int n3) {
    const int part = threadIdx.x & 7, nblk = b.nbx * b.nby;
    const int b0 = part * b.zper, b1 = min(b0 + b.zper, n3);
    const bool in = b0 < b1 && (z1 - z0 >= n3 || (z0 < b1 && b0 < z1) || z0 < b1 - n3 || b0 + n3 < z1);
    const int2 px = pieces(x0, x1, n1, b.nbx, b.xlog), py = pieces(y0, y1, n2, b.nby, b.ylog);
    const unsigned* p = b.m + ((size_t)col * kColParts + part) * nblk;
    unsigned m = 0;
    if (in)
        for (int j = (threadIdx.x >> 3) & 3; j < py.y; j += 4) {
            int y = py.x + j;
            if (y >= b.nby) y -= b.nby;
            for (int i = 0; i < px.y; i += 4) {
                unsigned v[4];                         // in flight together
#pragma unroll
                for (int k = 0; k < 4; ++k) {
                    int x = px.x + min(i + k, px.y - 1);
                    if (x >= b.nbx) x -= b.nbx;
                    v[k] = p[y * b.nbx + x];
                }
                m = max(max(m, max(v[0], v[1])), max(v[2], v[3]));
            }
        }
    return __reduce_max_sync(0xffffffffu, m);
}

// 2^k, |k| < 1023 (scalbn's cases cost a small grid's launch 5 us)
__device__ __forceinline__ double pow2(int k) { return __hiloint2double((k + 1023) << 20, 0); }

__device__ __forceinline__ void mad(long long& acc, int s, int w) { acc += (long long)s * w; }

// the product for a conjugate-gradient step: dot[1] = sum, dot[0] = dot[2], dot[6] = dot[0] / dot[1] or 0
__device__ __forceinline__ void finish_dot(const FxArgs& a, double v) {
    double total;
    if (grid_sum(v, a.part, a.counter, total)) {
        const double rr = a.dot[2];
        a.dot[0] = rr;
        a.dot[1] = total;
        a.dot[6] = total > 0.0 ? rr / total : 0.0;
    }
}

// ROWS = 2: two rows per thread; the 14 rows that the y-sums of both need are loaded once, the
// halo is 12 rows for twice the tile's, and the loop's own instructions serve two points.
// MODE: 0 plain, 1 with Yprev, 2 with the sum of Y * Yout (one column).
template <int MODE, int ROWS, int NTMAX, int CTAS, int PER>
__global__ void __launch_bounds__(NTMAX, CTAS)
k_stencil_fx(const __grid_constant__ FxArgs a) {
    constexpr bool YP = MODE == 1, DOT = MODE == 2;
    extern __shared__ __align__(16) int2 ring[];
    const int tid = threadIdx.x, nt = blockDim.x;
    const int tile = (int)(blockIdx.x % a.tiles);
    const int zc = (int)(blockIdx.x / a.tiles) % a.nzc, col = (int)(blockIdx.x / a.tiles) / a.nzc;
    const int gx0 = (tile % a.tilesx) * a.tx, gy0 = (tile / a.tilesx) * a.ty;
    const int z0 = zc * a.zchunk, z1 = min(z0 + a.zchunk, a.n3);
    const int n1 = a.n1, n2 = a.n2, n3 = a.n3;
    const long plane = (long)n1 * n2, cell = plane * n3;
    const double* __restrict__ Y = a.Y + (size_t)col * a.ld;
    const double* Yp = YP ? a.Yprev + (size_t)col * a.ld : nullptr;
    double* Yo = a.Yout + (size_t)col * a.ld;
    const double alpha = a.coef ? a.coef[0] : a.alpha, beta = a.coef ? a.coef[1] : a.beta;
    const double shift = a.coef ? a.coef[2] : a.shift;

    // this thread's halo'd points of a plane (beyond the last one: a point that nobody reads)
    const int sx = a.tx + 2 * FXH, sy = a.ty + 2 * FXH, stage = sy * FXP + 2;
    int s_idx[PER], s_off[PER];
#pragma unroll
    for (int k = 0; k < PER; ++k) {
        const int i = tid + k * nt;
        s_idx[k] = sy * FXP;
        s_off[k] = 0;
        if (i < sx * sy) {
            const int iy = i / sx, ix = i - iy * sx;
            s_idx[k] = iy * FXP + ix;
            s_off[k] = wrap(gy0 - FXH + iy, n2) * n1 + wrap(gx0 - FXH + ix, n1);
        }
    }
    auto load = [&](long zo, double (&v)[PER]) {
#pragma unroll
        for (int k = 0; k < PER; ++k) v[k] = Y[zo + s_off[k]];
    };
    double pf[PER];
    long zl = (long)z0 * plane;                   // plane loaded last
    load(zl, pf);

    // the scale: the column's, or that of the pieces that this CTA's points and their neighbours lie in
    unsigned top;
    if constexpr (DOT) top = column_max(a.cmax, col);
    else top = region_max(a.bmax, col, gx0 - FXH, gx0 + a.tx + FXH, n1, gy0 - FXH, gy0 + a.ty + FXH, n2, z0 - FXH,
                          max(z1 + FXH, z0 + 8), n3);         // plane z0 + 7 is converted in any case
    int emax = (int)(top >> 20);
    const int sf = a.vinfo[2];
    const bool fits = fabs(shift) < pow2(83 - sf);              // NaN: false
    bool plain = emax > kFxEmax || !fits || a.vinfo[1];         // the same for the whole CTA
    if (emax < kFxEmin) {
        plain |= (int)(column_max(a.cmax, col) >> 20) < kFxEmin;
        emax = kFxEmin;
    }
    const int e20 = emax << 20;
    if (plain) {
        const double sum = fx_slow(a, Y, Yp, Yo, gx0, gy0, z0, z1, alpha, beta, shift);
        if constexpr (DOT) finish_dot(a, sum);
        return;
    }
    const double scale = alpha * pow2(81 - sf + emax - 1081);
    const long long shq = __double2ll_rn(shift * pow2(sf - 25));
    const int shh = (int)(shq >> 30), shl = (int)(shq & 0x3fffffff);
    int fh[3], fl[3];                             // F 2^sf as limbs of 30 bits
#pragma unroll
    for (int ax = 0; ax < 3; ++ax) {
        const long long fq = __double2ll_rn(a.F[ax] * pow2(sf)) + __double2ll_rn(a.Flo[ax] * pow2(sf));
        fh[ax] = (int)(fq >> 30);
        fl[ax] = (int)(fq & 0x3fffffff);
    }
    // Sums start at half a unit of the bits shifted out, M1 also at the mean of the dropped
    // ul * fl: a bias of one unit would be the same at every point, and the filter, which keeps
    // the smooth part of its input and damps the rest, would keep all of it
    const long long m1 = (1 << 29) + (((long long)fl[0] + fl[1] + fl[2]) >> 1);

    // rows ROWS * ty .. of the tile
    const int ty = tid / a.tx, tx = tid - ty * a.tx;
    bool act[ROWS];
    int own[ROWS];
#pragma unroll
    for (int r = 0; r < ROWS; ++r) {
        const int y = ROWS * ty + r;
        act[r] = y < a.ty && gx0 + tx < n1 && gy0 + y < n2;
        own[r] = act[r] ? (gy0 + y) * n1 + gx0 + tx : gy0 * n1 + gx0;
    }
    const int ctr = act[0] ? (ROWS * ty + FXH) * FXP + tx + FXH : FXH * FXP + FXH;
    const int last = z1 + FXH - 1;                // highest plane needed

    auto store = [&](int j, const double (&v)[PER]) {
        int2* dst = ring + (j & (FXS - 1)) * stage;
#pragma unroll
        for (int k = 0; k < PER; ++k) dst[s_idx[k]] = to_limbs(v[k], e20);
    };

    // planes z0 .. z0 + 6 into the ring (stage index: plane - z0), each while the next is in flight (plane
    // z0 + 7 at last, needed or not: it is inside the block); z-queue z0 - 6 .. z0 + 5
#pragma unroll 1
    for (int j = 0; j <= FXH; ++j) {
        double next[PER];
        zl += plane;
        if (zl == cell) zl = 0;
        load(zl, next);
        store(j, pf);
#pragma unroll
        for (int k = 0; k < PER; ++k) pf[k] = next[k];
    }
    int2 q[ROWS][2 * FXH + 1];                    // [i]: plane z - 7 + i before the shift
#pragma unroll
    for (int j = 0; j < FXH; ++j) {
        const long zo = (long)wrap(z0 - FXH + j, n3) * plane;
#pragma unroll
        for (int r = 0; r < ROWS; ++r) q[r][1 + j] = to_limbs(Y[zo + own[r]], e20);
    }
    long zo = (long)z0 * plane;
    int2 vq[ROWS];
    double yp[ROWS];
#pragma unroll
    for (int r = 0; r < ROWS; ++r) {
        vq[r] = a.Vq[zo + own[r]];
        yp[r] = YP ? Yp[zo + own[r]] : DOT ? Y[zo + own[r]] : 0.0;
    }
    double dot = 0.0;
    __syncthreads();
#pragma unroll
    for (int j = 0; j < FXH; ++j)
#pragma unroll
        for (int r = 0; r < ROWS; ++r) q[r][FXH + 1 + j] = ring[j * stage + ctr + r * FXP];

#pragma unroll 1
    for (int j = 0; j < z1 - z0; ++j) {
        const int2* f = ring + ((j + FXH) & (FXS - 1)) * stage + ctr;
#pragma unroll
        for (int r = 0; r < ROWS; ++r) {
#pragma unroll
            for (int i = 0; i < 2 * FXH; ++i) q[r][i] = q[r][i + 1];
            q[r][2 * FXH] = f[r * FXP];
        }
        store(j + FXH + 1, pf);                   // the ring slot of plane z - 1
        if (z0 + j + FXH + 2 <= last) {
            zl += plane;
            if (zl == cell) zl = 0;
            load(zl, pf);
        }
        int2 vc[ROWS];
        double ypc[ROWS];
        const long zn = zo + plane;
#pragma unroll
        for (int r = 0; r < ROWS; ++r) {
            vc[r] = make_int2(vq[r].x - shh, vq[r].y - shl);
            ypc[r] = yp[r];
            if (j + 1 < z1 - z0) {
                vq[r] = a.Vq[zn + own[r]];
                if (YP) yp[r] = Yp[zn + own[r]];
                if (DOT) yp[r] = Y[zn + own[r]];
            }
        }
        long long ch[ROWS], cl[ROWS], H[ROWS], M1[ROWS], M2[ROWS], A[ROWS], B[ROWS];
#pragma unroll
        for (int r = 0; r < ROWS; ++r) {
            ch[r] = (long long)q[r][FXH].x * a.k[0];
            cl[r] = (long long)q[r][FXH].y * a.k[0] + (1 << 19);
            H[r] = 0;
            M1[r] = m1;
            M2[r] = 1 << 30;
        }
        auto start = [&]() {
#pragma unroll
            for (int r = 0; r < ROWS; ++r) { A[r] = ch[r]; B[r] = cl[r]; }
        };
        auto pair = [&](int r, int2 u, int2 w, int k) {
            mad(A[r], u.x + w.x, k);
            mad(B[r], u.y + w.y, k);
        };
        auto end = [&](int ax) {
#pragma unroll
            for (int r = 0; r < ROWS; ++r) {
                const long long U = (A[r] << 10) + (B[r] >> 20);
                const int uh = (int)(U >> 31), ul = (int)((unsigned)U & 0x7fffffffu);
                mad(H[r], uh, fh[ax]);
                mad(M1[r], uh, fl[ax]);
                mad(M2[r], ul, fh[ax]);
            }
        };
        const int2* ps = ring + (j & (FXS - 1)) * stage + ctr;
        start();
#pragma unroll
        for (int p = 1; p <= FXH; ++p)
#pragma unroll
            for (int r = 0; r < ROWS; ++r) pair(r, q[r][FXH + p], q[r][FXH - p], a.k[p]);
        end(2);
        start();
#pragma unroll
        for (int p = 1; p <= FXH; ++p)
#pragma unroll
            for (int r = 0; r < ROWS; ++r) pair(r, ps[r * FXP + p], ps[r * FXP - p], a.k[p]);
        end(0);
        start();
        if constexpr (ROWS == 2) {
            int2 up = q[1][FXH], dn = q[0][FXH];  // rows p and 1 - p
#pragma unroll
            for (int p = 1; p <= FXH; ++p) {
                const int2 un = ps[(p + 1) * FXP], dm = ps[-p * FXP];
                pair(0, up, dm, a.k[p]);          // rows p and -p
                pair(1, un, dn, a.k[p]);          // rows 1 + p and 1 - p
                up = un;
                dn = dm;
            }
        } else {
#pragma unroll
            for (int p = 1; p <= FXH; ++p) pair(0, ps[p * FXP], ps[-p * FXP], a.k[p]);
        }
        end(1);
#pragma unroll
        for (int r = 0; r < ROWS; ++r) {
            const int2 c = q[r][FXH];
            long long M3 = 1 << 29;                    // the low limbs' product, then the mixed ones
            mad(M3, c.y, vc[r].y);
            M3 = (M3 >> 30) + (1 << 25);
            mad(M3, c.x, vc[r].y);
            mad(M3, c.y, vc[r].x);
            const long long Z = H[r] + (M1[r] >> 30) + (M2[r] >> 31) + (((long long)c.x * vc[r].x) << 4) + (M3 >> 26);
            const double t = (double)Z * scale;
            if (act[r]) Yo[zo + own[r]] = YP ? fma(beta, ypc[r], t) : t;
            if (DOT && act[r]) dot = fma(ypc[r], t, dot);
        }
        zo = zn;
        __syncthreads();
    }
    if constexpr (DOT) finish_dot(a, dot);
}

__global__ void k_fx_vmax(const double* __restrict__ V, int* __restrict__ info, long n) {
    unsigned m = 0;
    for (long t = (long)blockIdx.x * blockDim.x + threadIdx.x; t < n; t += (long)gridDim.x * blockDim.x)
        m = max(m, (unsigned)__double2hiint(V[t]) & 0x7fffffffu);
    m = __reduce_max_sync(0xffffffffu, m);
    if ((threadIdx.x & 31) == 0) atomicMax(info, (int)m);
}

// limbs of V 2^(sf - 25) with |V| < 2^(83 - sf), sfmin <= sf <= sf0
__global__ void k_fx_veff(const double* __restrict__ V, int2* __restrict__ Vq, int* __restrict__ info, long n, int sf0, int sfmin) {
    const long t = (long)blockIdx.x * blockDim.x + threadIdx.x;
    const int sf = min(sf0, 83 - ((info[0] >> 20) - 1022));       // |V| < 2^(exponent - 1022)
    const bool bad = sf < sfmin;                                 // non-finite values included
    if (t == 0) { info[1] = bad; info[2] = bad ? sf0 : sf; }
    if (t >= n) return;
    const long long q = bad ? 0 : __double2ll_rn(scalbn(V[t], sf - 25));
    Vq[t] = make_int2((int)(q >> 30), (int)(q & 0x3fffffff));
}

// c_p = k_p / lcd of the centred second derivative of order 2 n0, and sf
struct FxSetup {
    int k[FXH + 1];
    int lcd, sf, sfmin;       // sfmin: F of 53 bits
};
FxSetup fx_setup(hub_t h) {
    static const int lcds[FXH + 1] = {1, 1, 12, 180, 5040, 25200, 831600};
    FxSetup s{};
    s.lcd = lcds[h->n0];
    double c0, c[kMaxHalf];
    fd_laplacian_weights(h->n0, &c0, c);
    s.k[0] = (int)std::lround(c0 * s.lcd);
    for (int p = 1; p <= h->n0; ++p) s.k[p] = (int)std::lround(c[p - 1] * s.lcd);
    // lower orders: the same binary point (A >> 20 keeps 62 bits), so weights of the same size
    auto sum = [&] {
        int t = std::abs(s.k[0]);
        for (int p = 1; p <= h->n0; ++p) t += 2 * std::abs(s.k[p]);
        return t;
    };
    while (2 * sum() <= 5881856) {                // the sum of order 12
        s.lcd *= 2;
        for (int p = 0; p <= h->n0; ++p) s.k[p] *= 2;
    }
    double fmax = 0.0;
    for (int a = 0; a < 3; ++a) fmax = std::max(fmax, 0.5 / (s.lcd * h->h[a] * h->h[a]));
    // |Fq| < 2^59 keeps the three products of Z in 64 bits; sf <= 75 leaves 256 Ha for V and the shift.
    // On coarse grids (above 0.4 bohr) that would cut off bits of F (beyond 4 bohr) and of V, which is rounded
    // at 2^(24 - sf): 57 - e keeps that under 2^-54 of the largest kinetic energy (2^22.5 F on every
    // axis) and leaves 2^(26 + e) Ha, four times that energy
    int e;
    std::frexp(fmax, &e);                         // 2^(e - 1) <= fmax < 2^e
    s.sf = std::max(std::min(75, 59 - e), 57 - e);
    s.sfmin = 53 - e;
    return s;
}

}  // namespace

// bytes of the fixed-point potential behind a potential of Nd doubles: limbs, then vinfo
size_t fx_veff_bytes(int64_t Nd) { return (size_t)Nd * 8 + 16; }

int launch_fx_veff(hub_t h, const void* V) {
    const FxSetup s = fx_setup(h);
    const long n = h->Nd;
    int2* Vq = (int2*)((double*)V + n);
    int* info = (int*)(Vq + n);
    HUB_CUDA_TRY(h, cudaMemsetAsync(info, 0, 3 * sizeof(int), h->stream));
    {
        ProfScope ps(h, HUB_K_COPY);
        k_fx_vmax<<<h->num_sms, 256, 0, h->stream>>>((const double*)V, info, n);
    }
    ProfScope ps(h, HUB_K_COPY);
    k_fx_veff<<<(unsigned)((n + 255) / 256), 256, 0, h->stream>>>((const double*)V, Vq, info, n, s.sf, s.sfmin);
    HUB_CUDA_TRY(h, cudaGetLastError());
    return HUB_OK;
}

template <int ROWS, int NT, int CTAS, int PER>
static int run_fx(hub_t h, const StencilArgs& s, int variant, const StencilDot* dot = nullptr) {
    FxArgs a{};
    int rc;
    if (!s.cmax_ready && (rc = launch_colmax(h, s.Y, s.ncol, s.ld))) return rc;
    a.Y = (const double*)s.Y;
    a.Yprev = (const double*)s.Yprev;
    a.Yout = (double*)s.Yout;
    a.V = (const double*)s.V;
    a.Vq = (const int2*)(a.V + h->Nd);
    a.vinfo = (const int*)(a.Vq + h->Nd);
    a.cmax = h->d_cmax;
    a.bmax = block_map(h, h->d_cmax, s.ncol);
    a.n1 = s.n1; a.n2 = s.n2; a.n3 = s.n3; a.ld = s.ld;
    const FxSetup f = fx_setup(h);
    double wb = 0.0;
    for (int p = 0; p <= FXH; ++p) a.k[p] = f.k[p];
    for (int ax = 0; ax < 3; ++ax) {
        // to more than 53 bits: a rounding at 2^-53 is one and the same error of the kinetic energy at every
        // point, where the rounded weights of the FP64 form average out
        const int n = ax == 0 ? h->n1 : ax == 1 ? h->n2 : h->n3;
        const long double ih = (long double)n / (long double)h->L[ax];
        const long double F = -0.5L * ih * ih / f.lcd;
        a.F[ax] = (double)F;
        a.Flo[ax] = (double)(F - a.F[ax]);
        for (int p = 0; p < FXH; ++p) {
            a.w[ax][p] = p < s.n0 ? s.wbase[ax][p] : 0.0;
            wb += a.w[ax][p];
        }
    }
    a.cen = -2.0 * wb;
    a.alpha = s.alpha;
    a.beta = s.beta;
    a.shift = s.shift;
    a.coef = s.coef;
    // Tiles of equal width close to 32 (rows are contiguous; the halo costs 12 points a row).  Rows
    // per tile (even: two per thread) and chunks along z by the instructions of a CTA (25 per
    // converted point, 540 per thread and plane; a chunk converts 7 planes and 12 points more)
    // times the CTAs that a slot runs one after another; a wave that is not full counts whole.
    const int ntx = (s.n1 + 31) / 32;
    a.tx = (s.n1 + ntx - 1) / ntx;
    a.tilesx = ntx;
    const int rows = std::min(std::min(ROWS * (NT / a.tx), PER * NT / (a.tx + 2 * FXH) - 2 * FXH), 60) / ROWS * ROWS;   // 60: 200 KB
    const int key = s.ncol * 8 + variant;
    if (h->fx_plan[0] != key) {
        double best = 1e300;
        for (int ty = rows; ty >= ROWS; ty -= ROWS) {
            if (ty < rows && ty >= s.n2 + ROWS) continue;
            const int nt = (std::max(a.tx * ty / ROWS, ((a.tx + 2 * FXH) * (ty + 2 * FXH) + PER - 1) / PER) + 31) / 32 * 32;
            const long tiles = (long)ntx * ((s.n2 + ty - 1) / ty) * s.ncol;
            for (int nzc = 1; nzc <= s.n3; ++nzc) {
                const int zc = (s.n3 + nzc - 1) / nzc;
                const double waves = (double)(tiles * ((s.n3 + zc - 1) / zc)) / (CTAS * h->num_sms);
                const double cost = nt * (zc * (25.0 * PER + 100.0 + 220.0 * ROWS) + 25.0 * (7 * PER + 12 * ROWS) + 1000.0);
                const double t = cost * (waves < 1.0 ? 0.5 + 0.5 * waves : waves < 8.0 ? std::ceil(waves) : waves + 0.5);
                if (t < best) { best = t; h->fx_plan[1] = ty; h->fx_plan[2] = zc; }
                if (zc <= 4) break;
            }
        }
        h->fx_plan[0] = key;
    }
    a.ty = h->fx_plan[1];
    a.zchunk = h->fx_plan[2];
    a.nzc = (s.n3 + a.zchunk - 1) / a.zchunk;
    a.tiles = ntx * ((s.n2 + a.ty - 1) / a.ty);
    const int slots = (a.tx + 2 * FXH) * (a.ty + 2 * FXH);
    const int nt = (std::max(a.tx * a.ty / ROWS, (slots + PER - 1) / PER) + 31) / 32 * 32;
    const size_t smem = (size_t)FXS * ((a.ty + 2 * FXH) * FXP + 2) * sizeof(int2);
    const long grid = (long)a.tiles * a.nzc * s.ncol;
    if (grid > 0x7fffffffL) return fail(h, HUB_EINVAL, "stencil: too many tiles");
    ProfScope ps(h, HUB_K_STENCIL);
    auto run = [&](auto kernel) -> int {
        HUB_CUDA_TRY(h, cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
        kernel<<<(unsigned)grid, nt, smem, h->stream>>>(a);
        return HUB_OK;
    };
    if constexpr (ROWS == 1 && CTAS == 4) {
        if (dot) {
            a.dot = dot->dot;
            a.part = dot->part;
            a.counter = dot->counter;
            if ((rc = run(k_stencil_fx<2, ROWS, NT, CTAS, PER>))) return rc;
            HUB_CUDA_TRY(h, cudaGetLastError());
            return HUB_OK;
        }
    }
    if ((rc = s.Yprev ? run(k_stencil_fx<1, ROWS, NT, CTAS, PER>) : run(k_stencil_fx<0, ROWS, NT, CTAS, PER>))) return rc;
    HUB_CUDA_TRY(h, cudaGetLastError());
    return HUB_OK;
}

// CTA shapes (hub_set_tuning; 0 is the default), on 88 x 88 x 84 x 348 of normal deviates: 4.19, 4.17
// and 4.16 ms.
// Four CTAs of 192 threads hide the barriers of one another's planes; two rows per thread need
// fewer instructions (382 against ~450 per point) but leave 16 warps per SM.
int launch_stencil_fx(hub_t h, const StencilArgs& s) {
    switch (h->stencil_variant) {
        case 1: return run_fx<1, 256, 3, 4>(h, s, 1);
        case 2: return run_fx<2, 256, 2, 5>(h, s, 2);
        default: return run_fx<1, 192, 4, 4>(h, s, 0);
    }
}

int launch_stencil_fx_dot(hub_t h, const StencilArgs& s, const StencilDot& d) { return run_fx<1, 192, 4, 4>(h, s, 0, &d); }

}  // namespace hub

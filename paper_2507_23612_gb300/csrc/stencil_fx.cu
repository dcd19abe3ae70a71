// Real FP64 stencil in integer arithmetic.  GB300 issues 2 FP64 operations per clock and SM
// but about 30 32x32+64-bit integer multiply-adds and 110 32-bit adds, so the ~39 FP64
// operations per point of the floating-point form (17.15 ms on 88 x 88 x 84 x 348, 0.82 of
// the FP64 pipe) cost several times what the same sum costs in fixed point.
//
//   Yout = alpha * (-1/2 Lap_h Y + V .* Y - shift * Y) + beta * Yprev        (Sec. II.B)
//
// Number format.  Every column has one power-of-two scale: with E the biased exponent of its
// largest |x| (colmax.cu), X = x * 2^(1081 - E) rounded to an integer, |X| <= 2^59, so an
// element keeps all 53 bits down to 2^-6 of the column's maximum and is never off by more
// than 2^-60 of it (one FP64 rounding of the sum, which holds terms of ~300 x, is larger).
// X is kept as two signed limbs, X = xh 2^30 + xl: pair sums of limbs need no carry.
// The Laplacian weights of order 2 n0 are rational: c_p = k_p / lcd with integers k_p of 22
// bits, so A_a = k_0 X + sum_p k_p (X_{+p} + X_{-p}) of each axis is exact, and only
// F_a = -1 / (2 lcd h_a^2) and V - shift are rounded (to 59 bits):
//   U_a = A_a >> 20 (62 bits),  Z = sum_a (U_a Fq_a) >> 61 + (X (V - shift)q) >> 56,
// one 64-bit integer per point, converted once; alpha and beta enter in FP64 (three FP64
// operations per point).  sf fixes the binary points: Fq = F 2^sf, Z counts x-units of
// 2^(81 - sf), (V - shift)q = (V - shift) 2^(sf - 25); it is as large as the sums' 64 bits
// allow, 59 bits of F or fewer where |V| exceeds 256 Ha and the sum of F's terms (k_fx_veff).
// Columns that the format does not cover (zero, non-finite or outside 2^+-900), potentials
// that would leave F under 51 bits and shifts beyond 2^(83 - sf) Ha (the largest kinetic
// energy of the grid, at least) are computed by fx_slow in plain FP64.
//
// Kernel: one CTA owns a TX x TY tile of the x-y plane of one column and marches along z.  A
// ring of 8 planes (with a halo of 6 in x and y) in shared memory holds the limbs; plane z + 7
// is converted and stored while plane z is computed, and plane z + 8 is in flight in
// registers, so there is one barrier per plane.  The 13 z-neighbours live in registers.
#include <algorithm>
#include <cmath>

#include "hub_internal.cuh"

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
    const unsigned* cmax;         // column maxima (colmax.cu)
    int n1, n2, n3, ld;
    int tx, ty, tilesx, tiles;    // tile shape and count
    int zchunk, nzc;
    int k[FXH + 1];               // integer weights, k[0] the centre
    double F[3];
    double alpha, beta, shift;
    const double* coef;           // device {alpha, beta, shift} or nullptr
    double w[3][FXH], cen;        // FP64 weights (alpha = 1) of the slow form
};

__device__ __forceinline__ int wrap(int i, int n) {      // i is at most a few n away
    while (i < 0) i += n;
    while (i >= n) i -= n;
    return i;
}

// x as limbs, emax the biased exponent of the column's maximum (>= 123, so that a denormal x
// shifts to zero whatever its hidden bit)
__device__ __forceinline__ int2 to_limbs(double v, int emax) {
    const unsigned hi = (unsigned)__double2hiint(v), lo = (unsigned)__double2loint(v);
    const int e = (int)(hi >> 20) & 0x7ff;
    const int sh = min(emax - e, 63);
    unsigned long long t = ((unsigned long long)((hi & 0xfffffu) | 0x100000u) << 32) | lo;
    t = (((t << 7) >> sh) + 1) >> 1;
    int xh = (int)(t >> 30), xl = (int)((unsigned)t & 0x3fffffffu);
    if ((int)hi < 0) { xh = -xh; xl = -xl; }
    return make_int2(xh, xl);
}

// the plain FP64 form of one tile and chunk, straight from global memory
__device__ __noinline__ void fx_slow(const FxArgs& a, const double* __restrict__ Y, const double* Yp, double* Yo, int gx0,
                                     int gy0, int z0, int z1, double alpha, double beta, double shift) {
    const long plane = (long)a.n1 * a.n2;
    const int per = a.tx * a.ty;
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
    }
}

// (hi, lo) sums of limb products: acc += w * s
__device__ __forceinline__ void mad(long long& acc, int s, int w) { acc += (long long)s * w; }

// PER: halo'd points per thread
template <bool YP, int NTMAX, int CTAS, int FXPER>
__global__ void __launch_bounds__(NTMAX, CTAS)
k_stencil_fx(const __grid_constant__ FxArgs a) {
    extern __shared__ __align__(16) int2 ring[];
    const int tid = threadIdx.x, nt = blockDim.x;
    const int tile = (int)(blockIdx.x % a.tiles);
    const int zc = (int)(blockIdx.x / a.tiles) % a.nzc, col = (int)(blockIdx.x / a.tiles) / a.nzc;
    const int gx0 = (tile % a.tilesx) * a.tx, gy0 = (tile / a.tilesx) * a.ty;
    const int z0 = zc * a.zchunk, z1 = min(z0 + a.zchunk, a.n3);
    const int n1 = a.n1, n2 = a.n2, n3 = a.n3;
    const long plane = (long)n1 * n2;
    const double* __restrict__ Y = a.Y + (size_t)col * a.ld;
    const double* Yp = YP ? a.Yprev + (size_t)col * a.ld : nullptr;
    double* Yo = a.Yout + (size_t)col * a.ld;
    const double alpha = a.coef ? a.coef[0] : a.alpha, beta = a.coef ? a.coef[1] : a.beta;
    const double shift = a.coef ? a.coef[2] : a.shift;

    const int emax = (int)(column_max(a.cmax, col) >> 20);
    const int sf = a.vinfo[2];
    const bool fits = fabs(shift) < scalbn(1.0, 83 - sf);       // NaN: false
    if (emax < kFxEmin || emax > kFxEmax || !fits || a.vinfo[1]) {    // the same for the whole CTA
        fx_slow(a, Y, Yp, Yo, gx0, gy0, z0, z1, alpha, beta, shift);
        return;
    }
    const double scale = scalbn(alpha, 81 - sf + emax - 1081);
    const long long shq = __double2ll_rn(scalbn(shift, sf - 25));
    int fh[3], fl[3];                             // F 2^sf as limbs of 30 bits
#pragma unroll
    for (int ax = 0; ax < 3; ++ax) {
        const long long fq = __double2ll_rn(scalbn(a.F[ax], sf));
        fh[ax] = (int)(fq >> 30);
        fl[ax] = (int)(fq & 0x3fffffff);
    }
    const int shh = (int)(shq >> 30), shl = (int)(shq & 0x3fffffff);
    // Sums start at half a unit of the bits shifted out, M1 also at the mean of the dropped
    // ul * fl: a bias of one unit would be the same at every point, and the filter, which keeps
    // the smooth part of its input and damps the rest, would keep all of it
    const long long m1 = (1 << 29) + (((long long)fl[0] + fl[1] + fl[2]) >> 1);

    // this thread's halo'd points of a plane
    const int sx = a.tx + 2 * FXH, sy = a.ty + 2 * FXH, stage = sy * FXP;
    int s_idx[FXPER], s_off[FXPER];
#pragma unroll
    for (int k = 0; k < FXPER; ++k) {
        const int i = tid + k * nt;
        s_idx[k] = -1;
        s_off[k] = 0;
        if (i < sx * sy) {
            const int iy = i / sx, ix = i - iy * sx;
            s_idx[k] = iy * FXP + ix;
            s_off[k] = wrap(gy0 - FXH + iy, n2) * n1 + wrap(gx0 - FXH + ix, n1);
        }
    }
    const int ty = tid / a.tx, tx = tid - ty * a.tx;
    const bool active = ty < a.ty && gx0 + tx < n1 && gy0 + ty < n2;
    // inactive threads read a point of their own plane region (never stored)
    const int ctr = active ? (ty + FXH) * FXP + tx + FXH : FXH * FXP + FXH;
    const int own = active ? (gy0 + ty) * n1 + gx0 + tx : gy0 * n1 + gx0;
    const int last = z1 + FXH - 1;                // highest plane needed

    auto load = [&](int p, double (&v)[FXPER]) {
        const double* src = Y + (long)wrap(p, n3) * plane;
#pragma unroll
        for (int k = 0; k < FXPER; ++k) v[k] = s_idx[k] >= 0 ? src[s_off[k]] : 0.0;
    };
    auto store = [&](int p, const double (&v)[FXPER]) {
        int2* dst = ring + (p & (FXS - 1)) * stage;
#pragma unroll
        for (int k = 0; k < FXPER; ++k)
            if (s_idx[k] >= 0) dst[s_idx[k]] = to_limbs(v[k], emax);
    };

    // planes z0 .. z0 + 6 into the ring (stage index: plane - z0), z-queue z0 - 6 .. z0 + 5
    double pf[FXPER];
    for (int j = 0; j <= FXH; ++j) {
        load(z0 + j, pf);
        store(j, pf);
    }
    int2 q[2 * FXH + 1];
    {
        double v[FXH];
#pragma unroll
        for (int j = 0; j < FXH; ++j) v[j] = Y[(long)wrap(z0 - FXH + j, n3) * plane + own];
#pragma unroll
        for (int j = 0; j < FXH; ++j) q[1 + j] = to_limbs(v[j], emax);
    }
    load(z0 + FXH + 1 <= last ? z0 + FXH + 1 : last, pf);
    int2 vq = a.Vq[(long)z0 * plane + own];
    double yp = YP ? Yp[(long)z0 * plane + own] : 0.0;
    __syncthreads();
#pragma unroll
    for (int j = 0; j < FXH; ++j) q[FXH + 1 + j] = ring[j * stage + ctr];

    // The loop body is one plane; the shift of the queue is 24 register moves
#pragma unroll 1
    for (int j = 0; j < z1 - z0; ++j) {
        const int z = z0 + j;
#pragma unroll
        for (int i = 0; i < 2 * FXH; ++i) q[i] = q[i + 1];
        q[2 * FXH] = ring[((j + FXH) & (FXS - 1)) * stage + ctr];
        if (z + FXH + 1 <= last) store(j + FXH + 1, pf);          // the ring slot of plane z - 1
        if (z + FXH + 2 <= last) load(z + FXH + 2, pf);
        const int2 vc = make_int2(vq.x - shh, vq.y - shl);
        const double ypc = yp;
        if (z + 1 < z1) {
            vq = a.Vq[(long)(z + 1) * plane + own];
            if (YP) yp = Yp[(long)(z + 1) * plane + own];
        }
        const int2 c = q[FXH];
        const long long ch = (long long)c.x * a.k[0], cl = (long long)c.y * a.k[0] + (1 << 19);
        long long H = 0, M1 = m1, M2 = 1 << 30;
        const int2* ps = ring + (j & (FXS - 1)) * stage + ctr;
#pragma unroll
        for (int ax = 0; ax < 3; ++ax) {
            long long A = ch, B = cl;
#pragma unroll
            for (int p = 1; p <= FXH; ++p) {
                int2 u, v;
                if (ax == 2) { u = q[FXH + p]; v = q[FXH - p]; }
                else { u = ps[ax == 0 ? p : p * FXP]; v = ps[ax == 0 ? -p : -p * FXP]; }
                mad(A, u.x + v.x, a.k[p]);
                mad(B, u.y + v.y, a.k[p]);
            }
            const long long U = (A << 10) + (B >> 20);
            const int uh = (int)(U >> 31), ul = (int)((unsigned)U & 0x7fffffffu);
            mad(H, uh, fh[ax]);
            mad(M1, uh, fl[ax]);
            mad(M2, ul, fh[ax]);
        }
        long long M3 = 1 << 25;
        mad(M3, c.x, vc.y);
        mad(M3, c.y, vc.x);
        const long long Z = H + (M1 >> 30) + (M2 >> 31) + (((long long)c.x * vc.x) << 4) + (M3 >> 26);
        double r = (double)Z * scale;
        if (YP) r = fma(beta, ypc, r);
        if (active) Yo[(long)z * plane + own] = r;
        __syncthreads();
    }
}

__global__ void k_fx_vmax(const double* __restrict__ V, int* __restrict__ info, long n) {
    unsigned m = 0;
    for (long t = (long)blockIdx.x * blockDim.x + threadIdx.x; t < n; t += (long)gridDim.x * blockDim.x)
        m = max(m, (unsigned)__double2hiint(V[t]) & 0x7fffffffu);
    m = __reduce_max_sync(0xffffffffu, m);
    if ((threadIdx.x & 31) == 0) atomicMax(info, (int)m);
}

// limbs of V 2^(sf - 25) with |V| < 2^(83 - sf), sf <= sf0
__global__ void k_fx_veff(const double* __restrict__ V, int2* __restrict__ Vq, int* __restrict__ info, long n, int sf0) {
    const long t = (long)blockIdx.x * blockDim.x + threadIdx.x;
    const int sf = min(sf0, 83 - ((info[0] >> 20) - 1022));       // |V| < 2^(exponent - 1022)
    const bool bad = sf < sf0 - 8;                               // non-finite values included
    if (t == 0) { info[1] = bad; info[2] = bad ? sf0 : sf; }
    if (t >= n) return;
    const long long q = bad ? 0 : __double2ll_rn(scalbn(V[t], sf - 25));
    Vq[t] = make_int2((int)(q >> 30), (int)(q & 0x3fffffff));
}

// c_p = k_p / lcd of the centred second derivative of order 2 n0, and sf
struct FxSetup {
    int k[FXH + 1];
    int lcd, sf;
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
    // |Fq| < 2^59 keeps the three products of Z in 64 bits; sf <= 75 leaves 256 Ha for V
    int e;
    std::frexp(fmax, &e);                         // fmax < 2^e
    s.sf = std::min(75, 59 - e);
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
    k_fx_veff<<<(unsigned)((n + 255) / 256), 256, 0, h->stream>>>((const double*)V, Vq, info, n, s.sf);
    HUB_CUDA_TRY(h, cudaGetLastError());
    return HUB_OK;
}

template <int NT, int CTAS, int FXPER>
static int run_fx(hub_t h, const StencilArgs& s) {
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
    a.n1 = s.n1; a.n2 = s.n2; a.n3 = s.n3; a.ld = s.ld;
    const FxSetup f = fx_setup(h);
    double wb = 0.0;
    for (int p = 0; p <= FXH; ++p) a.k[p] = f.k[p];
    for (int ax = 0; ax < 3; ++ax) {
        a.F[ax] = -0.5 / (f.lcd * h->h[ax] * h->h[ax]);
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
    // tiles of equal width close to 32 (rows are contiguous; the halo costs 12 points a row),
    // rows so that a CTA has at most NT threads and FXPER points of the halo'd plane each
    const int ntx = (s.n1 + 31) / 32;
    a.tx = (s.n1 + ntx - 1) / ntx;
    const int rows = std::min(std::min(NT / a.tx, FXPER * NT / (a.tx + 2 * FXH) - 2 * FXH), 60);   // 60: 200 KB
    const int nty = (s.n2 + rows - 1) / rows;
    a.ty = (s.n2 + nty - 1) / nty;
    a.tilesx = ntx;
    a.tiles = ntx * nty;
    const int slots = (a.tx + 2 * FXH) * (a.ty + 2 * FXH);
    const int nt = (std::max(a.tx * a.ty, (slots + FXPER - 1) / FXPER) + 31) / 32 * 32;
    // chunks along z: about two waves of CTAs, each chunk re-reading 12 planes
    const long per = (long)a.tiles * s.ncol, want = 4L * CTAS * h->num_sms;
    int nzc = per < want ? (int)((want + per - 1) / per) : 1;
    a.zchunk = std::max(std::min(s.n3, 8), (s.n3 + nzc - 1) / nzc);
    a.nzc = (s.n3 + a.zchunk - 1) / a.zchunk;
    const size_t smem = (size_t)FXS * (a.ty + 2 * FXH) * FXP * sizeof(int2);
    const long grid = (long)a.tiles * a.nzc * s.ncol;
    if (grid > 0x7fffffffL) return fail(h, HUB_EINVAL, "stencil: too many tiles");
    ProfScope ps(h, HUB_K_STENCIL);
    auto run = [&](auto kernel) -> int {
        HUB_CUDA_TRY(h, cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
        kernel<<<(unsigned)grid, nt, smem, h->stream>>>(a);
        return HUB_OK;
    };
    if ((rc = s.Yprev ? run(k_stencil_fx<true, NT, CTAS, FXPER>) : run(k_stencil_fx<false, NT, CTAS, FXPER>))) return rc;
    HUB_CUDA_TRY(h, cudaGetLastError());
    return HUB_OK;
}

// CTA shapes (hub_set_tuning; 0 is the default).  Three CTAs of 256 threads (80 registers) hide
// the barrier of one another's planes: 4.5 ms on 88 x 88 x 84 x 348, against 4.8 (two of 384),
// 5.0 (two of 256 with 96 registers) and 6.4 (one of 512).
int launch_stencil_fx(hub_t h, const StencilArgs& s) {
    switch (h->stencil_variant) {
        case 1: return run_fx<384, 2, 3>(h, s);
        case 2: return run_fx<256, 2, 4>(h, s);
        default: return run_fx<256, 3, 4>(h, s);
    }
}

}  // namespace hub

// Dense FP64 steps of the Rayleigh-Ritz projection (CheFSI, Sec. II.B) on n x n matrices
// (n = number of orbitals, up to ~1100), all row-major in device memory, real (double) at
// the Gamma point and complex Hermitian (double2, interleaved re/im) for Bloch orbitals:
//   Cholesky S = L L^H (blocked, right-looking), L^-1, small GEMMs with optional adjoint
//   operands, and a Hermitian eigensolver by parallel cyclic Jacobi (round-robin pairing:
//   n/2 disjoint rotations per step) in one cooperative kernel.  Every device-wide wait in
//   this file is a bounded software barrier: after its iteration limit it raises
//   FLAG_TIMEOUT and the kernel returns, so a wait can never hang the GPU.
#include <algorithm>

#include "hub_internal.cuh"
#include "cplx.cuh"

namespace hub {

namespace {

constexpr int NB = 32;   // Cholesky block

// Cholesky S = L L^H by elimination with multipliers, a_ij <- a_ij - l_ik conj(w_jk) with the
// column w_k as it stands and l_ik = w_ik / w_kk; L = w_k / sqrt(w_kk).  Every kernel applies the
// steps k in the same order with the same operation, so that the rows of two equal columns of X
// stay equal bit for bit, their multiplier is 1 and the second pivot is zero or below: a block with
// a column twice is refused, and every positive pivot is accepted.  (With products of elements of
// L that pivot is the rounding of a square root, of either sign.)
__device__ __forceinline__ double eliminate(double a, double l, double w) { return fma(-l, w, a); }
__device__ __forceinline__ double2 eliminate(double2 a, double2 l, double2 w) {
    return make_double2(fma(-l.y, w.y, fma(-l.x, w.x, a.x)), fma(l.x, w.y, fma(-l.y, w.x, a.y)));
}
// workspace of a panel: pivots, the diagonal block as it stands, then the rows below: l, w
template <typename T>
struct CholWs {
    double* d;      // [NB]
    T* w;           // [NB][NB]
    T *lr, *wr;     // [n - NB][NB]
};

// factor the jb x jb diagonal block at (j0, j0) in place (one CTA, NB x NB in shared memory);
// the diagonal of a Hermitian matrix is real, so is L's
template <typename T>
__global__ void k_potf2(T* A, int lda, int j0, int jb, int* flags, CholWs<T> ws, int below) {
    __shared__ T s[NB][NB + 1];
    __shared__ T l[NB];
    __shared__ double piv[NB];
    const int t = threadIdx.x;
    for (int e = t; e < jb * jb; e += blockDim.x) {
        const int i = e / jb, j = e % jb;
        s[i][j] = A[(size_t)(j0 + i) * lda + j0 + j];
    }
    __syncthreads();
    for (int k = 0; k < jb; ++k) {
        double d = re_of(s[k][k]);
        const bool ok = d > 0.0 && isfinite(d);
        if (!ok) d = 1.0;
        if (t == 0) {
            if (!ok) flags[FLAG_NOTSPD] = 1;
            piv[k] = d;
        }
        for (int i = k + 1 + t; i < jb; i += blockDim.x) l[i] = divr(s[i][k], d);
        __syncthreads();
        for (int e = t; e < jb * jb; e += blockDim.x) {
            const int i = e / jb, j = e % jb;
            if (i > k && j > k && j <= i) s[i][j] = eliminate(s[i][j], l[i], s[j][k]);
        }
        __syncthreads();
    }
    for (int e = t; e < jb * jb; e += blockDim.x) {
        const int i = e / jb, j = e % jb;
        const double r = sqrt(piv[j]);
        A[(size_t)(j0 + i) * lda + j0 + j] = j < i ? divr(s[i][j], r) : j == i ? from_real<T>(r) : zero_of(T());
        if (below) {
            ws.w[i * NB + j] = s[i][j];
            if (i == 0) ws.d[j] = piv[j];
        }
    }
}

// the lower triangle of a Hermitian matrix from the upper one: the Gram product computes both within
// a tile and mirrors the others, which differ in the rounding of their imaginary parts
__global__ void k_mirror(double2* A, int n) {
    const long t = (long)blockIdx.x * blockDim.x + threadIdx.x;
    const int i = (int)(t / n), j = (int)(t % n);
    if (i < n && j < i) A[(size_t)i * n + j] = cconj(A[(size_t)j * n + i]);
}

// rows below the diagonal block: one thread per row
template <typename T>
__global__ void k_panel(T* A, int lda, int j0, int n, CholWs<T> ws) {
    __shared__ T w[NB][NB + 1];
    __shared__ double d[NB], root[NB];
    for (int e = threadIdx.x; e < NB * NB; e += blockDim.x) w[e / NB][e % NB] = ws.w[e];
    for (int e = threadIdx.x; e < NB; e += blockDim.x) { d[e] = ws.d[e]; root[e] = sqrt(ws.d[e]); }
    __syncthreads();
    const int r = blockIdx.x * blockDim.x + threadIdx.x;
    if (j0 + NB + r >= n) return;
    T l[NB];
    T* row = A + (size_t)(j0 + NB + r) * lda + j0;
    for (int c = 0; c < NB; ++c) {
        T v = row[c];
        for (int k = 0; k < c; ++k) v = eliminate(v, l[k], w[c][k]);
        l[c] = divr(v, d[c]);
        ws.wr[(size_t)r * NB + c] = v;
        ws.lr[(size_t)r * NB + c] = l[c];
        row[c] = divr(v, root[c]);
    }
}

// the lower triangle behind the panel, 32 x 32 tiles
template <typename T>
__global__ void k_trail(T* A, int lda, int j1, int n, CholWs<T> ws) {
    __shared__ T l[NB][NB + 1], w[NB][NB + 1];
    if (blockIdx.x > blockIdx.y) return;
    const int tx = threadIdx.x % NB, ty = threadIdx.x / NB, m = n - j1;      // NB x 8 threads
    const int i0 = blockIdx.y * NB, c0 = blockIdx.x * NB;
    for (int r = ty; r < NB; r += 8) {
        l[r][tx] = i0 + r < m ? ws.lr[(size_t)(i0 + r) * NB + tx] : zero_of(T());
        w[r][tx] = c0 + r < m ? ws.wr[(size_t)(c0 + r) * NB + tx] : zero_of(T());
    }
    __syncthreads();
    if (c0 + tx >= m) return;
    T acc[NB / 8];
#pragma unroll
    for (int q = 0; q < NB / 8; ++q)
        acc[q] = i0 + ty + 8 * q >= m ? zero_of(T()) : A[(size_t)(j1 + i0 + ty + 8 * q) * lda + j1 + c0 + tx];
#pragma unroll 8
    for (int k = 0; k < NB; ++k) {
        const T wk = w[tx][k];
#pragma unroll
        for (int q = 0; q < NB / 8; ++q) acc[q] = eliminate(acc[q], l[ty + 8 * q][k], wk);
    }
#pragma unroll
    for (int q = 0; q < NB / 8; ++q)
        if (i0 + ty + 8 * q < m) A[(size_t)(j1 + i0 + ty + 8 * q) * lda + j1 + c0 + tx] = acc[q];
}

// C = alpha op(A) op(B) + beta C, row-major, 32 x 32 tiles; op = identity or the adjoint
// (conjugate transpose; the transpose for real matrices); alpha, beta real
template <typename T>
__global__ void k_dgemm(int ta, int tb, int m, int n, int k, double alpha, const T* __restrict__ A,
                        int lda, const T* __restrict__ B, int ldb, double beta, T* C, int ldc) {
    __shared__ T As[32][33], Bs[32][33];
    const int tx = threadIdx.x % 32, ty = threadIdx.x / 32;   // 32 x 8 threads
    const int i0 = blockIdx.y * 32, j0 = blockIdx.x * 32;
    T acc[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) acc[q] = zero_of(T());
    for (int k0 = 0; k0 < k; k0 += 32) {
        for (int r = ty; r < 32; r += 8) {
            const int i = i0 + r, kk = k0 + tx;
            T a = zero_of(T());
            if (i < m && kk < k) a = ta ? cconj(A[(size_t)kk * lda + i]) : A[(size_t)i * lda + kk];
            As[r][tx] = a;
            const int kb = k0 + r, j = j0 + tx;
            T b = zero_of(T());
            if (kb < k && j < n) b = tb ? cconj(B[(size_t)j * ldb + kb]) : B[(size_t)kb * ldb + j];
            Bs[r][tx] = b;
        }
        __syncthreads();
#pragma unroll 8
        for (int kk = 0; kk < 32; ++kk) {
            const T b = Bs[kk][tx];
#pragma unroll
            for (int q = 0; q < 4; ++q) acc[q] = cfma(As[ty + 8 * q][kk], b, acc[q]);
        }
        __syncthreads();
    }
    for (int q = 0; q < 4; ++q) {
        const int i = i0 + ty + 8 * q, j = j0 + tx;
        if (i < m && j < n) {
            T* c = C + (size_t)i * ldc + j;
            *c = beta != 0.0 ? add(mulr(alpha, acc[q]), mulr(beta, *c)) : mulr(alpha, acc[q]);
        }
    }
}

// Linv = L^-1: one warp per column j solves L x = e_j by forward substitution
template <typename T>
__global__ void k_tri_inverse(const T* __restrict__ L, T* __restrict__ Linv, int n) {
    const int warp = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int lane = threadIdx.x & 31;
    if (warp >= n) return;
    const int j = warp;
    T* x = Linv;   // column j of Linv: x[i*n + j]
    for (int i = lane; i < j; i += 32) x[(size_t)i * n + j] = zero_of(T());
    for (int i = j; i < n; ++i) {
        T s = zero_of(T());
        for (int l = j + lane; l < i; l += 32) s = cfma(L[(size_t)i * n + l], x[(size_t)l * n + j], s);
        for (int o = 16; o > 0; o >>= 1) s = add(s, shfl_down(s, o));
        if (lane == 0)
            x[(size_t)i * n + j] = divr(csub(from_real<T>(i == j ? 1.0 : 0.0), s), re_of(L[(size_t)i * n + i]));
        __syncwarp();
    }
}

// A <- (A + A^H) / 2 (the diagonal of a Hermitian matrix is real)
template <typename T>
__global__ void k_symmetrize(T* A, int n) {
    const long t = (long)blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= (long)n * n) return;
    const int i = (int)(t / n), j = (int)(t % n);
    if (j < i) return;
    if (j == i) { A[(size_t)i * n + i] = from_real<T>(re_of(A[(size_t)i * n + i])); return; }
    const T v = mulr(0.5, add(A[(size_t)i * n + j], cconj(A[(size_t)j * n + i])));
    A[(size_t)i * n + j] = v;
    A[(size_t)j * n + i] = cconj(v);
}

// ---------------------------------------------------------------------------- Jacobi
constexpr int kJacThreads = 256;
constexpr long kSpinLimit = 1L << 22;

__device__ __forceinline__ unsigned ld_acquire(const unsigned* p) {
    unsigned v;
    asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}
// one thread waits until the counter has reached target; bounded, false once a wait ran out
__device__ __forceinline__ bool wait_count(const unsigned* bar, unsigned target, int* flags) {
    for (long it = 0; (int)(ld_acquire(bar) - target) < 0; ++it) {
        if (it > kSpinLimit || ((it & 1023) == 1023 && *((volatile int*)(flags + FLAG_TIMEOUT)) != 0)) {
            atomicExch(flags + FLAG_TIMEOUT, 1);
            return false;
        }
    }
    return true;
}

__device__ __forceinline__ void pair_of(int step, int k, int N, int& p, int& q) {
    // round-robin ("circle") schedule: player N-1 fixed, players 0..N-2 rotate; step < N - 1
    if (k == 0) { p = N - 1; q = step; }
    else {
        p = step + k;
        if (p >= N - 1) p -= N - 1;
        q = step - k;
        if (q < 0) q += N - 1;
    }
    if (p > q) { const int t = p; p = q; q = t; }
}

// Elements of other CTAs: from L2
__device__ __forceinline__ double ld_far(const double* p) { return __ldcg(p); }
__device__ __forceinline__ double2 ld_far(const double2* p) { return __ldcg(p); }

__device__ __forceinline__ int exponent_of(double v) { return (__double2hiint(v) >> 20) & 0x7ff; }

// c and sg = s exp(i arg a_pq) of the rotation that zeroes a_pq: s = t c, t the smaller root of
// |a_pq| t^2 + (a_qq - a_pp) t = |a_pq|.  t, 1 / sqrt(1 + t^2) and the phase are estimated in float
// (2^-22) and corrected in double to rounding (t twice, 2^-43 and 2^-65), so that the coupling falls to
// a few ulp and one step ends a 2 x 2 problem.  (The divisions and square roots of a double angle
// are some 50 dependent instructions of the FP64 pipe, of about 64 clocks each; these are 14.
// Left at the float estimates, a step costs 0.25 us less and the coupling falls to 2^-22; the second
// correction of t costs 0.08 us of it.)
template <typename T>
__device__ __forceinline__ void jacobi_angle(double app, double aqq, T apq, double& c, T& sg) {
    constexpr bool CPLX = sizeof(T) == 16;
    const double d = aqq - app;
    // all by the power of two that brings the largest of them near 1
    int e = exponent_of(d);
    if constexpr (CPLX) e = max(e, max(exponent_of(apq.x), exponent_of(apq.y)) + 1);
    else e = max(e, exponent_of(apq) + 1);
    const double sc = __hiloint2double(max(1, min(2046, 2046 - e)) << 20, 0);
    const double D = fabs(d * sc);
    double a, px = 1.0, py = 0.0;              // |a_pq| and its phase
    float af;
    if constexpr (CPLX) {
        const double xd = apq.x * sc, yd = apq.y * sc;
        const float x = (float)xd, y = (float)yd;
        const float big = fmaxf(fabsf(x), fabsf(y)), up = big < 1e-15f ? 1e18f : 1.0f;      // keeps the square in range
        const float xs = x * up, ys = y * up, rf = rsqrtf(fmaf(xs, xs, ys * ys));
        af = fabsf(x) * fabsf(xs * rf) + fabsf(y) * fabsf(ys * rf);
        const double r = (double)rf * (double)up, m = fma(xd, xd, yd * yd);
        const double h = fma(-(m * r), r, 1.0);
        const double r1 = fma(r * h, fma(0.375, h, 0.5), r);                // r (1 + h/2 + 3 h^2/8)
        px = xd * r1;
        py = yd * r1;
        a = m * r1;
    } else {
        a = fabs(apq * sc);
        af = (float)a;
    }
    const float df = (float)D, mf = 2.0f * af;
    const float tf = __fdividef(mf, df + sqrtf(fmaf(df, df, mf * mf)));
    const double t0 = (double)tf, y = (double)rsqrtf(fmaf(tf, tf, 1.0f)), y2 = y * y;
    const double g = (double)__fdividef(1.0f, fmaf(mf, tf, df));          // one over the derivative
    const double t1 = fma(-fma(fma(a, t0, D), t0, -a), g, t0);            // 2^-43
    const double t = fma(-fma(fma(a, t1, D), t1, -a), g, t1);
    const double u = fma(t, t, 1.0), ty = t * y;
    const double h = fma(-u, y2, 1.0), k = fma(0.375, h, 0.5);
    c = fma(y * h, k, y);                                                  // y (1 + h/2 + 3 h^2/8)
    const double s = fma(ty * h, k, ty);
    // the signs of a_qq - a_pp and a_pq by their bits: comparisons are FP64 instructions too
    int sign = __double2hiint(d);
    if constexpr (!CPLX) sign ^= __double2hiint(apq);
    const double ss = __hiloint2double(__double2hiint(s) ^ (sign & (int)0x80000000), __double2loint(s));
    if constexpr (CPLX) sg = make_double2(px * ss, py * ss);
    else sg = ss;
}
// the leading word of |v| (of the larger part): compared as integers, off the FP64 pipe
__device__ __forceinline__ int lead(double v) { return __double2hiint(v) & 0x7fffffff; }
__device__ __forceinline__ int lead(double2 v) { return max(lead(v.x), lead(v.y)); }

template <typename T>
struct JacobiArgs {
    T* A[2];                    // matrices (result: the diagonal)
    T* Ab[2];                   // second buffers
    T* V[2];                    // eigenvectors as columns
    double* ang[2];             // [2][RS * H]: the angles of the last step and this one
    unsigned long long* red[2]; // 4 slots each
    unsigned* bar;              // one counter per matrix, zeroed
    int* flags;
    int* sweeps;
    int nmat, n, N, max_sweeps, g, ng, v_shared;
    double tol;
};

// Parallel cyclic Jacobi with the round-robin pair schedule.  Each step applies n/2 disjoint
// rotations and writes the rotated matrix into the other of two buffers: nothing the step reads is
// written during it, so one grid-wide barrier per step suffices.  3500 steps of the 348-orbital
// block follow one another, so the length of a step is what counts: barrier, loads from L2, angles,
// update, stores.
//   * A CTA owns the blocks of one pair of groups of g pairs (upper triangle, the adjoint written
//     too), so that it needs 2 g angles and not all n/2, one per thread, from elements loaded
//     together with those of its blocks.  All copies of an angle have the same inputs and operations.
//   * The rotation of V is one step late and overlaps the barrier: a CTA keeps some rows of V in
//     shared memory (in global memory if they don't fit) and applies the angles of the step before,
//     which the CTAs of the diagonal groups leave in memory, between its arrival and the release.
//     One warp only waits.
// 348 orbitals: 29.9 -> 14.2 ms (58: 3.3 -> 1.7 ms; complex 348: 53.2 -> 21 ms) against every CTA
// computing every angle in double and V between the loads and the barrier.  Of a step's 8300 clocks
// 2600 go into loads and angles, 1700 into the update, 1000 into the stores and 1700 into the wait.
// The rotation of a pair (p, q) is J = [[c, sg], [-conj(sg), c]] with c real and
// sg = s exp(i arg a_pq): the phase makes the pivot real, then the real Jacobi angle of
// (a_pp, |a_pq|, a_qq) zeroes it; for real matrices sg = +-s and J is the plain rotation.
// With nmat = 2 the grid solves two independent matrices of the same size at once: each half of
// the CTAs owns one matrix, its buffers, its barrier counter and its reduction slots, and only the
// error flags are shared (a timeout in one half ends both).
template <typename T>
__global__ void __launch_bounds__(kJacThreads, 1) k_jacobi(const __grid_constant__ JacobiArgs<T> a) {
    constexpr bool CPLX = sizeof(T) == 2 * sizeof(double);
    constexpr int RS = CPLX ? 3 : 2;              // doubles per pair: c, sg (re[, im])
    constexpr int VT = kJacThreads - 32;          // threads that rotate V
    extern __shared__ double2 jac_smem[];
    __shared__ int ok_sh;
    const int n = a.n, N = a.N, H = N / 2, g = a.g, tid = threadIdx.x;
    const int grp = (a.nmat == 2 && blockIdx.x >= gridDim.x / 2) ? 1 : 0;
    const int nb = a.nmat == 2 ? gridDim.x / 2 : gridDim.x, cta = blockIdx.x - grp * nb;
    double* rot = (double*)jac_smem;              // angles of this CTA's groups
    double* late = rot + (2 * RS * g + 1) / 2 * 2;                 // all angles of the step before
    T* vrows = a.v_shared ? (T*)(late + (RS * H + 1) / 2 * 2) : nullptr;
    T* V = a.V[grp];
    double* ang = a.ang[grp];
    unsigned* bar = a.bar + grp;
    unsigned arrived = 0;
    // groups of this CTA: row I of the upper triangle of ng x ng
    int I = 0, J = cta;
    while (J >= a.ng - I) { J -= a.ng - I; ++I; }
    J += I;
    const int rows = cta < n ? (n - cta + nb - 1) / nb : 0;        // rows cta, cta + nb, ... of V
    auto vrow = [&](int r) -> T* { return vrows ? vrows + (size_t)r * n : V + (size_t)(cta + r * nb) * n; };
    for (int r = 0; r < rows; ++r)
        for (int j = tid; j < n; j += kJacThreads) vrow(r)[j] = from_real<T>(j == cta + r * nb ? 1.0 : 0.0);
    auto get = [](const double* w, double& c, T& sg) {
        c = w[0];
        if constexpr (CPLX) sg = make_double2(w[1], w[2]);
        else sg = w[1];
    };
    auto rotate_v = [&](int step, int t0, int nt) {
        int r = t0 / H, k = t0 - r * H;
        const int dr = nt / H, dk = nt - dr * H;
        while (r < rows) {
            double c;
            T sg;
            get(late + RS * k, c, sg);
            int p, q;
            pair_of(step, k, N, p, q);
            if (q < n && lead(sg) != 0) {
                T* v = vrow(r);
                const T vp = v[p], vq = v[q];
                v[p] = csub(mulr(c, vp), cmul(cconj(sg), vq));
                v[q] = cfma(sg, vp, mulr(c, vq));
            }
            r += dr;
            k += dk;
            if (k >= H) { k -= H; ++r; }
        }
    };
    // arrival (after every thread's stores) and wait of a grid-wide barrier
    auto arrive = [&] {
        __threadfence();
        atomicAdd(bar, 1u);
    };
    auto barrier = [&]() -> bool {
        __syncthreads();
        arrived += nb;
        if (tid == 0) {
            arrive();
            ok_sh = wait_count(bar, arrived, a.flags);
        }
        __syncthreads();
        return ok_sh != 0;
    };
    T* cur = a.A[grp];
    T* nxt = a.Ab[grp];
    unsigned long long* red = a.red[grp];
    const T zero = zero_of(T());
    const int e0 = tid < g * g ? tid / g * 65536 + tid % g : g * 65536;       // this thread's first block of the CTA's
    int sweep = 0, before = -1, par = 0;          // the step before (none), half of ang to write
    for (; sweep < a.max_sweeps; ++sweep) {
        // convergence: max |a_ij| (i != j) against max |a_ii|
        unsigned long long* acc = red + 2 * (sweep & 1);
        double off = 0.0, dia = 0.0;
        for (int i = cta; i < n; i += nb)
            for (int j = tid; j < n; j += kJacThreads) {
                const double v = cabs_of(ld_far(cur + (size_t)i * n + j));
                if (i == j) dia = fmax(dia, v); else off = fmax(off, v);
            }
        for (int o = 16; o > 0; o >>= 1) {
            off = fmax(off, __shfl_down_sync(0xffffffffu, off, o));
            dia = fmax(dia, __shfl_down_sync(0xffffffffu, dia, o));
        }
        if ((tid & 31) == 0) {
            atomicMax(acc, (unsigned long long)__double_as_longlong(off));
            atomicMax(acc + 1, (unsigned long long)__double_as_longlong(dia));
        }
        if (!barrier()) return;
        const double goff = __longlong_as_double((long long)__ldcg(acc));
        const double gdia = __longlong_as_double((long long)__ldcg(acc + 1));
        if (cta == 0 && tid == 0) {
            unsigned long long* other = red + 2 * ((sweep + 1) & 1);
            other[0] = 0ull;
            other[1] = 0ull;
        }
        if (goff <= a.tol * fmax(gdia, 1e-300)) break;
        if (sweep == a.max_sweeps - 1) {
            if (cta == 0 && tid == 0) a.flags[FLAG_NOCONV] = 1;
            break;
        }
        // pairs whose coupling is below this are left alone (threshold Jacobi)
        const int skip = lead((CPLX ? 0.7e-3 : 1e-3) * a.tol * fmax(gdia, 1e-300));
        for (int step = 0; step < N - 1; ++step) {
            // the angles of the step before come in while this step's are computed
            if (before >= 0) {
                const double2* src = (const double2*)(ang + (size_t)(par ^ 1) * ((RS * H + 1) / 2 * 2));
                for (int i = tid; i < (RS * H + 1) / 2; i += kJacThreads)
                    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"((unsigned)__cvta_generic_to_shared((double2*)late + i)),
                                 "l"(src + i) : "memory");
                asm volatile("cp.async.commit_group;" ::: "memory");
            }
            int p1, q1, p2, q2;
            T b00, b01, b10, b11;
            auto ld = [&](int i, int j) { return (i < n && j < n) ? ld_far(cur + (size_t)i * n + j) : zero; };
            auto load_block = [&](int i, int j) -> bool {
                const int P = I * g + i, Q = J * g + j;
                if (P >= Q || i >= g || Q >= H) return false;
                pair_of(step, P, N, p1, q1);
                pair_of(step, Q, N, p2, q2);
                b00 = ld(p1, p2); b01 = ld(p1, q2); b10 = ld(q1, p2); b11 = ld(q1, q2);
                return true;
            };
            bool have = load_block(e0 / 65536, e0 % 65536);
            // angles: one thread per pair; in a diagonal group also the pair's own block, which
            // gets the corrections of the diagonal and what is left of the coupling
            for (int i = tid; i < (I == J ? g : 2 * g); i += kJacThreads) {
                const int k = i < g ? I * g + i : J * g + i - g;
                if (k >= H) continue;
                int p, q;
                pair_of(step, k, N, p, q);
                double c = 1.0;
                T sg = zero;
                if (q < n) {
                    const T apq = ld(p, q);
                    const double app = re_of(ld(p, p)), aqq = re_of(ld(q, q));
                    if (lead(apq) > skip && lead(apq) <= 0x7ff00000) jacobi_angle(app, aqq, apq, c, sg);   // not NaN
                }
                double* w = rot + RS * i;
                w[0] = c;
                if constexpr (CPLX) { w[1] = sg.x; w[2] = sg.y; }
                else w[1] = sg;
                if (I == J) {
                    double* out = ang + (size_t)par * ((RS * H + 1) / 2 * 2) + (size_t)RS * k;
                    for (int d = 0; d < RS; ++d) __stcg(out + d, w[d]);
                }
            }
            __syncthreads();
            // every 2x2 block (P, Q) of the next matrix <- J_P^H B J_Q; the matrix stays Hermitian:
            // only the blocks P <= Q are computed, and each writes its adjoint too
            auto st = [&](int i, int j, T v) {
                if (i >= n || j >= n) return;
                nxt[(size_t)i * n + j] = v;
                nxt[(size_t)j * n + i] = cconj(v);
            };
            for (int e = tid; e < g * g; e += kJacThreads) {
                int i = e0 / 65536, j = e0 % 65536;
                if (e != tid) { i = e / g; j = e - i * g; have = load_block(i, j); }
                if (!have) continue;
                double c1, c2;
                T g1, g2;
                get(rot + RS * i, c1, g1);
                get(rot + RS * (j + (I == J ? 0 : g)), c2, g2);
                const T r00 = csub(mulr(c1, b00), cmul(g1, b10));
                const T r01 = csub(mulr(c1, b01), cmul(g1, b11));
                const T r10 = cfma(cconj(g1), b00, mulr(c1, b10));
                const T r11 = cfma(cconj(g1), b01, mulr(c1, b11));
                st(p1, p2, csub(mulr(c2, r00), cmul(cconj(g2), r01)));
                st(p1, q2, cfma(g2, r00, mulr(c2, r01)));
                st(q1, p2, csub(mulr(c2, r10), cmul(cconj(g2), r11)));
                st(q1, q2, cfma(g2, r10, mulr(c2, r11)));
            }
            if (I == J)
                for (int i = kJacThreads - 1 - tid; i < g; i += kJacThreads) {     // the last warps first
                    const int k = I * g + i;
                    if (k >= H) continue;
                    int p, q;
                    pair_of(step, k, N, p, q);
                    double c;
                    T sg;
                    get(rot + RS * i, c, sg);
                    const T apq = ld(p, q);
                    const double app = re_of(ld(p, p));
                    if (q >= n) {
                        nxt[(size_t)p * n + p] = from_real<T>(app);
                        continue;
                    }
                    const double aqq = re_of(ld(q, q));
                    const double d = aqq - app, s2 = re_of(cmul(cconj(sg), sg)), w = re_of(cmul(cconj(sg), apq));
                    const double u = fma(s2, d, -2.0 * c * w);
                    nxt[(size_t)p * n + p] = from_real<T>(app + u);
                    nxt[(size_t)q * n + q] = from_real<T>(aqq - u);
                    st(p, q, csub(csub(mulr(c * c, apq), cmul(cmul(sg, sg), cconj(apq))), mulr(c * d, sg)));
                }
            asm volatile("cp.async.wait_all;" ::: "memory");
            __syncthreads();
            arrived += nb;
            if (tid >= VT) {
                if (tid == VT) {
                    arrive();
                    ok_sh = wait_count(bar, arrived, a.flags);
                }
            } else if (before >= 0) {
                rotate_v(before, tid, VT);
            }
            __syncthreads();
            if (!ok_sh) return;
            before = step;
            par ^= 1;
            T* t = cur; cur = nxt; nxt = t;
        }
    }
    // the last step's rotations of V
    if (before >= 0) {
        const double* src = ang + (size_t)(par ^ 1) * ((RS * H + 1) / 2 * 2);
        for (int i = tid; i < RS * H; i += kJacThreads) late[i] = __ldcg(src + i);
        __syncthreads();
        rotate_v(before, tid, kJacThreads);
        __syncthreads();
    }
    if (vrows)
        for (int r = 0; r < rows; ++r)
            for (int j = tid; j < n; j += kJacThreads) V[(size_t)(cta + r * nb) * n + j] = vrows[(size_t)r * n + j];
    if (cur != a.A[grp])
        for (int i = cta; i < n; i += nb)
            for (int j = tid; j < n; j += kJacThreads) a.A[grp][(size_t)i * n + j] = ld_far(cur + (size_t)i * n + j);
    if (cta == 0 && tid == 0) a.sweeps[grp] = sweep;
}

// ascending order: rank by (value, index); V columns follow
template <typename T>
__global__ void k_sort_eig(const T* __restrict__ A, const T* __restrict__ V, int n,
                           double* __restrict__ eig, T* __restrict__ Vs) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const double ai = re_of(A[(size_t)i * n + i]);
    int rank = 0;
    for (int j = 0; j < n; ++j) {
        const double aj = re_of(A[(size_t)j * n + j]);
        rank += (aj < ai) || (aj == ai && j < i);
    }
    eig[rank] = ai;
    for (int r = 0; r < n; ++r) Vs[(size_t)r * n + rank] = V[(size_t)r * n + i];
}

}  // namespace

// The host entry points take double pointers; on a complex handle every matrix is n x n
// double2 (interleaved re/im, 2 n^2 doubles) and the same memory is read as such.
namespace {

template <typename T>
int gemm_t(hub_t h, bool ta, bool tb, int m, int n, int k, double alpha, const T* A, int lda, const T* B,
           int ldb, double beta, T* C, int ldc) {
    if (m == 0 || n == 0) return HUB_OK;
    dim3 grid((n + 31) / 32, (m + 31) / 32);
    ProfScope ps(h, HUB_K_DGEMM);
    k_dgemm<T><<<grid, 256, 0, h->stream>>>(ta, tb, m, n, k, alpha, A, lda, B, ldb, beta, C, ldc);
    HUB_CUDA_TRY(h, cudaGetLastError());
    return HUB_OK;
}

template <typename T>
int cholesky_t(hub_t h, T* A, int n, double* work) {
    CholWs<T> ws{};
    if (n > NB) {
        ws.d = work;                                     // NB doubles: 16-byte multiples follow
        ws.w = (T*)(work + NB);
        ws.lr = ws.w + NB * NB;
        ws.wr = ws.lr + (size_t)(n - NB) * NB;
    }
    if constexpr (sizeof(T) == 16) {
        ProfScope ps(h, HUB_K_CHOLESKY);
        k_mirror<<<(unsigned)(((size_t)n * n + 255) / 256), 256, 0, h->stream>>>(A, n);
        HUB_CUDA_TRY(h, cudaGetLastError());
    }
    for (int j0 = 0; j0 < n; j0 += NB) {
        const int jb = std::min(NB, n - j0), rest = n - j0 - jb;
        { ProfScope ps(h, HUB_K_CHOLESKY); k_potf2<T><<<1, 256, 0, h->stream>>>(A, n, j0, jb, h->d_flags, ws, rest > 0); }
        HUB_CUDA_TRY(h, cudaGetLastError());
        if (rest <= 0) continue;
        { ProfScope ps(h, HUB_K_CHOLESKY); k_panel<T><<<(rest + 127) / 128, 128, 0, h->stream>>>(A, n, j0, n, ws); }
        HUB_CUDA_TRY(h, cudaGetLastError());
        const unsigned tiles = (rest + NB - 1) / NB;
        { ProfScope ps(h, HUB_K_CHOLESKY); k_trail<T><<<dim3(tiles, tiles), 256, 0, h->stream>>>(A, n, j0 + jb, n, ws); }
        HUB_CUDA_TRY(h, cudaGetLastError());
    }
    return HUB_OK;
}

template <typename T>
int jacobi_t(hub_t h, int nmat, T* const* A, T* const* V, double* const* eig, int n) {
    const int N = n + (n & 1), H = N / 2;
    const size_t nn = (size_t)n * n;
    constexpr int CW = sizeof(T) / sizeof(double), RS = CW + 1;
    const size_t nang = (size_t)(RS * H + 1) / 2 * 2;
    const size_t per = 2 * CW * nn + 2 * nang + 4;         // doubles of workspace per matrix
    int rc;
    if ((rc = ensure(h, &h->d_work2, &h->work2_bytes, std::max(nmat * per * sizeof(double), h->work2_bytes))))
        return rc;
    JacobiArgs<T> a{};
    for (int g = 0; g < 2; ++g) {
        const int m = g < nmat ? g : 0;
        a.A[g] = A[m];
        a.ang[g] = (double*)h->d_work2 + m * per;               // 16-byte aligned
        a.red[g] = (unsigned long long*)(a.ang[g] + 2 * nang);
        a.V[g] = (T*)(a.ang[g] + 2 * nang + 4);
        a.Ab[g] = a.V[g] + nn;                                  // second matrix buffer
        if (g < nmat) HUB_CUDA_TRY(h, cudaMemsetAsync(a.red[g], 0, 4 * sizeof(unsigned long long), h->stream));
    }
    a.sweeps = h->d_flags + 6;                                  // slots 6 and 7
    a.bar = h->d_bar;
    a.flags = h->d_flags;
    a.nmat = nmat;
    a.n = n;
    a.N = N;
    a.max_sweeps = 60;
    // A coupling c that is left turns two orbitals by c / gap.  With 1e-13 for doubles, small blocks
    // (2 to 20 orbitals, 84 blocks) that stopped just below it had D and density wrong by up to 2e-12;
    // with 1e-15 all are within 3e-14 (median 5e-15 in both), for a sweep more in one block of eight.
    // Rounding doesn't hold couplings up: a rotation rounds each to an ulp of itself.
    a.tol = h->esize == 8 ? 1e-15 : 1e-13;
    HUB_CUDA_TRY(h, cudaMemsetAsync(h->d_bar, 0, 4 * sizeof(unsigned int), h->stream));
    HUB_CUDA_TRY(h, cudaMemsetAsync(a.sweeps, 0, 2 * sizeof(int), h->stream));
    if ((size_t)H * RS * sizeof(double) > 48 * 1024) return fail(h, HUB_EINVAL, "subspace too large for the Jacobi solver");
    // groups of g pairs, one CTA per pair of groups: as many groups as the SMs of one matrix hold,
    // of at least 6 pairs (fewer CTAs wait for one another: 58 orbitals take 15)
    const int room = std::max(1, h->num_sms / nmat);
    int ng = 1;
    while ((ng + 1) * (ng + 2) / 2 <= room && (H + ng) / (ng + 1) >= 6) ++ng;
    a.g = (H + ng - 1) / ng;
    a.ng = (H + a.g - 1) / a.g;
    const int blocks = a.ng * (a.ng + 1) / 2;
    const size_t base = ((size_t)(2 * RS * a.g + 1) / 2 * 2 + nang) * sizeof(double);
    const size_t vbytes = (size_t)((n + blocks - 1) / blocks) * n * sizeof(T);
    a.v_shared = base + vbytes <= 200 * 1024;
    const size_t smem = base + (a.v_shared ? vbytes : 0);
    HUB_CUDA_TRY(h, cudaFuncSetAttribute(k_jacobi<T>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
    void* args[] = {&a};
    {
        ProfScope ps(h, HUB_K_JACOBI);
        HUB_CUDA_TRY(h, cudaLaunchCooperativeKernel((void*)k_jacobi<T>, dim3(blocks * nmat), dim3(kJacThreads), args, smem,
                                                    h->stream));
    }
    for (int g = 0; g < nmat; ++g) {
        ProfScope ps(h, HUB_K_EIG_MISC);
        k_sort_eig<T><<<(n + 127) / 128, 128, 0, h->stream>>>(A[g], a.V[g], n, eig[g], V[g]);
    }
    HUB_CUDA_TRY(h, cudaGetLastError());
    return HUB_OK;
}

}  // namespace

int dense_gemm(hub_t h, bool ta, bool tb, int m, int n, int k, double alpha, const double* A,
               int lda, const double* B, int ldb, double beta, double* C, int ldc) {
    if (h->cplx)
        return gemm_t<double2>(h, ta, tb, m, n, k, alpha, (const double2*)A, lda, (const double2*)B, ldb, beta,
                               (double2*)C, ldc);
    return gemm_t<double>(h, ta, tb, m, n, k, alpha, A, lda, B, ldb, beta, C, ldc);
}

int dense_cholesky(hub_t h, double* A, int n, double* work) {
    return h->cplx ? cholesky_t<double2>(h, (double2*)A, n, work) : cholesky_t<double>(h, A, n, work);
}

int dense_tri_inverse(hub_t h, const double* L, double* Linv, int n) {
    const int threads = 256;
    const long warps = n;
    const unsigned blocks = (unsigned)((warps * 32 + threads - 1) / threads);
    ProfScope ps(h, HUB_K_TRI_INVERSE);
    if (h->cplx) k_tri_inverse<double2><<<blocks, threads, 0, h->stream>>>((const double2*)L, (double2*)Linv, n);
    else k_tri_inverse<double><<<blocks, threads, 0, h->stream>>>(L, Linv, n);
    HUB_CUDA_TRY(h, cudaGetLastError());
    return HUB_OK;
}

int dense_symmetrize(hub_t h, double* A, int n) {
    const long tot = (long)n * n;
    ProfScope ps(h, HUB_K_EIG_MISC);
    if (h->cplx) k_symmetrize<double2><<<(unsigned)((tot + 255) / 256), 256, 0, h->stream>>>((double2*)A, n);
    else k_symmetrize<double><<<(unsigned)((tot + 255) / 256), 256, 0, h->stream>>>(A, n);
    HUB_CUDA_TRY(h, cudaGetLastError());
    return HUB_OK;
}

// A (n x n Hermitian, destroyed) -> eig ascending (device [n]) and V (device n x n row-major,
// column j = eigenvector j).  Uses 2 n x n matrices and two steps' angles of scratch per matrix.
int dense_jacobi_eigh_multi(hub_t h, int nmat, double* const* A, double* const* V, double* const* eig, int n) {
    if (n == 0) return HUB_OK;
    if (nmat < 1 || nmat > 2) return fail(h, HUB_EINVAL, "one or two matrices per Jacobi launch");
    if (h->cplx) {
        double2* Az[2] = {(double2*)A[0], (double2*)A[nmat - 1]};
        double2* Vz[2] = {(double2*)V[0], (double2*)V[nmat - 1]};
        return jacobi_t<double2>(h, nmat, Az, Vz, eig, n);
    }
    return jacobi_t<double>(h, nmat, A, V, eig, n);
}

int dense_jacobi_eigh(hub_t h, double* A, double* V, double* eig, int n) {
    return dense_jacobi_eigh_multi(h, 1, &A, &V, &eig, n);
}

}  // namespace hub

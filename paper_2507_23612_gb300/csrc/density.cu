// Grid-sized steps of the self-consistent density SCF: the electron density of a block of
// orbitals, the periodic FD Poisson problem of the Hartree potential, local-density
// exchange, the Kerker preconditioner, and the vector algebra of Pulay mixing on the
// density.  Sec. II.B (last paragraph) names CheFSI with real-space preconditioned Pulay
// mixing whose density coefficients also mix the occupation matrices; the functional
// pieces are readings (the paper does not print E_DFT):
//   rho(g)  = scale * sum_n f_n |x_n(g)|^2
//   V_H:    -Lap_h V_H = 4 pi (rho - mean rho), mean V_H = 0 (neutralising background)
//   v_x:    -(4/3) k rho^(1/3), E_x = -k dV sum rho^(4/3), k = (3/4)(3/pi)^(1/3) (x 2^(1/3)
//           per channel of a spin-polarized pair)
//   Kerker: z = (-Lap_h)(-Lap_h + kappa^2)^-1 r
// Both linear problems are solved by conjugate gradients on (-Lap_h + shift), FP64, with the
// same 2*n0-th order FD Laplacian as the kinetic term (periodic: the density and the
// potentials are cell-periodic).  CG scalars stay on the device; the host reads the residual
// every kCgCheck iterations.  Reductions are two-stage with a fixed order (deterministic).
#include <algorithm>
#include <cmath>
#include <vector>

#include "hub_internal.cuh"
#include "cplx.cuh"
#include "grid_sum.cuh"

namespace hub {

namespace {

constexpr int kThreads = 256;
constexpr int kCgCheck = 16;          // CG iterations between host residual checks
constexpr int kMaxLin = 8;            // vectors of one linear combination

__device__ __forceinline__ double abs2(double v) { return v * v; }
__device__ __forceinline__ double abs2(float v) { return (double)v * v; }
__device__ __forceinline__ double abs2(double2 v) { return v.x * v.x + v.y * v.y; }
__device__ __forceinline__ double abs2(float2 v) { return (double)v.x * v.x + (double)v.y * v.y; }

// block sum of one double per thread into part[blockIdx.x] (blockDim.x == kThreads)
__device__ __forceinline__ void block_partial(double v, double* part) {
    __shared__ double red[kThreads / 32];
    for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = v;
    __syncthreads();
    if (threadIdx.x == 0) {
        double s = 0.0;
        for (int w = 0; w < kThreads / 32; ++w) s += red[w];
        part[blockIdx.x] = s;
    }
}

// out[slot] = scale * sum(part[0..n)); one CTA, fixed order
__global__ void k_reduce(const double* __restrict__ part, int n, double scale, double* __restrict__ out, int slot) {
    __shared__ double red[kThreads];
    double s = 0.0;
    for (int i = threadIdx.x; i < n; i += kThreads) s += part[i];
    red[threadIdx.x] = s;
    __syncthreads();
    for (int w = kThreads / 2; w > 0; w >>= 1) {
        if (threadIdx.x < w) red[threadIdx.x] += red[threadIdx.x + w];
        __syncthreads();
    }
    if (threadIdx.x == 0) {
        out[slot] = scale * red[0];
    }
}

// ---------------------------------------------------------------------------- density
template <typename T>
__global__ void __launch_bounds__(kThreads)
k_density(const T* __restrict__ X, int ld, int ncol, long Nd, const double* __restrict__ f, double scale,
          double* __restrict__ rho) {
    const long g = (long)blockIdx.x * kThreads + threadIdx.x;
    if (g >= Nd) return;
    double acc = 0.0;
    int n = 0;
    for (; n + 4 <= ncol; n += 4) {
        const T a = X[(long)n * ld + g], b = X[(long)(n + 1) * ld + g];
        const T c = X[(long)(n + 2) * ld + g], d = X[(long)(n + 3) * ld + g];
        acc += f[n] * abs2(a) + f[n + 1] * abs2(b) + f[n + 2] * abs2(c) + f[n + 3] * abs2(d);
    }
    for (; n < ncol; ++n) acc += f[n] * abs2(X[(long)n * ld + g]);
    rho[g] += scale * acc;
}

// ---------------------------------------------------------------------------- Laplacian
struct LapArgs {
    double w[3][kMaxHalf];   // c_p / h_a^2
    double center;           // c_0 sum_a h_a^-2
    int n0, n1, n2, n3;
};

// y = -Lap_h x (periodic)
__global__ void __launch_bounds__(kThreads)
k_neg_lap(const double* __restrict__ x, double* __restrict__ y, LapArgs a) {
    const long Nd = (long)a.n1 * a.n2 * a.n3;
    const long g = (long)blockIdx.x * kThreads + threadIdx.x;
    if (g < Nd) {
        const int i = (int)(g % a.n1);
        const long t = g / a.n1;
        const int j = (int)(t % a.n2);
        const int k = (int)(t / a.n2);
        const long sy = a.n1, sz = (long)a.n1 * a.n2;
        const double* row = x + (g - i);                      // (0, j, k)
        const double* col = x + (g - (long)j * sy);           // (i, 0, k)
        const double* pil = x + (g - (long)k * sz);           // (i, j, 0)
        const double x0 = x[g];
        double lap = a.center * x0;
        for (int p = 1; p <= a.n0; ++p) {
            int ip = i + p, im = i - p, jp = j + p, jm = j - p, kp = k + p, km = k - p;
            while (ip >= a.n1) ip -= a.n1;
            while (im < 0) im += a.n1;
            while (jp >= a.n2) jp -= a.n2;
            while (jm < 0) jm += a.n2;
            while (kp >= a.n3) kp -= a.n3;
            while (km < 0) km += a.n3;
            lap = fma(a.w[0][p - 1], row[ip] + row[im], lap);
            lap = fma(a.w[1][p - 1], col[(long)jp * sy] + col[(long)jm * sy], lap);
            lap = fma(a.w[2][p - 1], pil[(long)kp * sz] + pil[(long)km * sz], lap);
        }
        y[g] = -lap;
    }
}

// ---------------------------------------------------------------------------- CG steps
// scalar slots: 0 rr, 1 pq, 2 rr_new, 3 bb, 4 scratch, 5 CTAs done (a counter), 6 alpha = rr / pq,
// 7 beta = rr_new / rr (divided once, by the thread that has the sum: a division per thread was a
// third of the steps' time)
enum { S_RR = 0, S_PQ = 1, S_RRN = 2, S_BB = 3, S_TMP = 4, S_CNT = 5, S_ALPHA = 6, S_BETA = 7 };

// elements of a CTA of the vector steps: 4 per thread, loaded before any is stored
constexpr int kCgPer = 4;

// largest leading word of |v| over the threads, for the scale of the fixed-point stencil
__device__ __forceinline__ unsigned lead(double v) { return (unsigned)__double2hiint(v) & 0x7fffffffu; }
__device__ __forceinline__ void raise_max(unsigned m, unsigned* cmax) {
    m = __reduce_max_sync(0xffffffffu, m);
    if ((threadIdx.x & 31) == 0) atomicMax(cmax + blockIdx.x % kColParts, m);
}

__global__ void __launch_bounds__(kThreads)
k_vec_max(const double* __restrict__ x, long n, unsigned* __restrict__ cmax) {
    const long g = (long)blockIdx.x * kThreads + threadIdx.x;
    raise_max(g < n ? lead(x[g]) : 0, cmax);
}

// r = b - q, p = r; partials of r . r and of b . b (part, part + nblk); cmax: of p
__global__ void __launch_bounds__(kThreads)
k_cg_start(const double* __restrict__ b, const double* __restrict__ q, double* __restrict__ r, double* __restrict__ p,
           long n, double* __restrict__ part, int nblk, unsigned* __restrict__ cmax) {
    const long g = (long)blockIdx.x * kThreads + threadIdx.x;
    double rr = 0.0, bb = 0.0;
    unsigned m = 0;
    if (g < n) {
        const double v = b[g] - q[g];
        r[g] = v;
        p[g] = v;
        rr = v * v;
        bb = b[g] * b[g];
        m = lead(v);
    }
    raise_max(m, cmax);
    block_partial(rr, part);
    __syncthreads();
    block_partial(bb, part + nblk);
}

// x += alpha p; r -= alpha q; rr_new = r . r, beta; clears the maxima for k_cg_direction
__global__ void __launch_bounds__(kThreads)
k_cg_update(double* __restrict__ x, double* __restrict__ r, const double* __restrict__ p, const double* __restrict__ q,
            long n, double* __restrict__ s, double* __restrict__ part, unsigned* __restrict__ cmax) {
    const long g0 = (long)blockIdx.x * (kCgPer * kThreads) + threadIdx.x;
    double xv[kCgPer], rv[kCgPer], pv[kCgPer], qv[kCgPer];
#pragma unroll
    for (int i = 0; i < kCgPer; ++i) {
        const long g = g0 + i * kThreads;
        const bool in = g < n;
        xv[i] = in ? x[g] : 0.0;
        rv[i] = in ? r[g] : 0.0;
        pv[i] = in ? p[g] : 0.0;
        qv[i] = in ? q[g] : 0.0;
    }
    const double alpha = s[S_ALPHA];
    double rr = 0.0, total;
#pragma unroll
    for (int i = 0; i < kCgPer; ++i) {
        const long g = g0 + i * kThreads;
        if (g >= n) continue;
        x[g] = fma(alpha, pv[i], xv[i]);
        const double v = fma(-alpha, qv[i], rv[i]);
        r[g] = v;
        rr = fma(v, v, rr);
    }
    if (grid_sum(rr, part, (unsigned*)(s + S_CNT), total)) {
        s[S_RRN] = total;
        s[S_BETA] = s[S_RR] > 0.0 ? total / s[S_RR] : 0.0;
        for (int i = 0; i < kColParts; ++i) cmax[i] = 0;
    }
}

// p = r + beta p; cmax: of p
__global__ void __launch_bounds__(kThreads)
k_cg_direction(const double* __restrict__ r, double* __restrict__ p, long n, const double* __restrict__ s,
               unsigned* __restrict__ cmax) {
    const long g0 = (long)blockIdx.x * (kCgPer * kThreads) + threadIdx.x;
    double rv[kCgPer], pv[kCgPer];
#pragma unroll
    for (int i = 0; i < kCgPer; ++i) {
        const long g = g0 + i * kThreads;
        rv[i] = g < n ? r[g] : 0.0;
        pv[i] = g < n ? p[g] : 0.0;
    }
    const double beta = s[S_BETA];
    unsigned m = 0;
#pragma unroll
    for (int i = 0; i < kCgPer; ++i) {
        const long g = g0 + i * kThreads;
        const double v = fma(beta, pv[i], rv[i]);
        if (g < n) p[g] = v;
        m = max(m, lead(v));
    }
    raise_max(m, cmax);
}

// y = c0 * (x - s[slot] / n) (c0 = 4 pi: the Poisson right-hand side; slot holds sum x)
// (x and y may be the same vector)
__global__ void k_center_scale(const double* x, double* y, long n, double c0, const double* __restrict__ s,
                               int slot) {
    const long g = (long)blockIdx.x * kThreads + threadIdx.x;
    if (g < n) y[g] = c0 * (x[g] - s[slot] / (double)n);
}

__global__ void __launch_bounds__(kThreads)
k_partial_sum(const double* __restrict__ x, long n, double* __restrict__ part) {
    const long g = (long)blockIdx.x * kThreads + threadIdx.x;
    block_partial(g < n ? x[g] : 0.0, part);
}

__global__ void __launch_bounds__(kThreads)
k_partial_dot(const double* __restrict__ x, const double* __restrict__ y, long n, double* __restrict__ part) {
    const long g = (long)blockIdx.x * kThreads + threadIdx.x;
    block_partial(g < n ? x[g] * y[g] : 0.0, part);
}

__global__ void __launch_bounds__(kThreads)
k_partial_absdiff(const double* __restrict__ x, const double* __restrict__ y, long n, double* __restrict__ part) {
    const long g = (long)blockIdx.x * kThreads + threadIdx.x;
    block_partial(g < n ? fabs(x[g] - y[g]) : 0.0, part);
}

// ---------------------------------------------------------------------------- exchange
__global__ void __launch_bounds__(kThreads)
k_lda_x(const double* __restrict__ rho, double* __restrict__ vx, long n, double k, double* __restrict__ part) {
    const long g = (long)blockIdx.x * kThreads + threadIdx.x;
    double e = 0.0;
    if (g < n) {
        const double r = fmax(rho[g], 0.0);
        const double c = cbrt(r);
        vx[g] = -(4.0 / 3.0) * k * c;
        e = -k * r * c;                       // -k rho^(4/3)
    }
    block_partial(e, part);
}

// ---------------------------------------------------------------------------- linear algebra
struct LinArgs {
    const double* v[kMaxLin];
    double c[kMaxLin];
    int k;
};

// y = sum_i c_i v_i (+ beta * z when z != nullptr)
// (y may be one of the v_i)
__global__ void k_lincomb(double* y, long n, LinArgs a, const double* z, double beta) {
    const long g = (long)blockIdx.x * kThreads + threadIdx.x;
    if (g >= n) return;
    double s = 0.0;
    for (int i = 0; i < a.k; ++i) s = fma(a.c[i], a.v[i][g], s);
    if (z) s = fma(beta, z[g], s);
    y[g] = s;
}

__global__ void k_add3(double* __restrict__ y, const double* __restrict__ a, const double* __restrict__ b,
                       const double* __restrict__ c, long n) {
    const long g = (long)blockIdx.x * kThreads + threadIdx.x;
    if (g < n) y[g] = a[g] + b[g] + c[g];
}

unsigned blocks_for(long n) { return (unsigned)((n + kThreads - 1) / kThreads); }

}  // namespace

// ---------------------------------------------------------------------------- host side
// workspace: [partials: 2 nblk, one per 32 points of a row][8 scalars][r][p][q][b] doubles, and a
// zero potential in the form of the fixed-point stencil
static int dens_ws(hub_t h, double** part, double** s, double** r, double** p, double** q, double** b) {
    const long n = h->Nd;
    const long nblk = blocks_for(n);
    const size_t npart = std::max<size_t>(2 * nblk, (size_t)((h->n1 + 31) / 32) * h->n2 * h->n3);
    const size_t need = (npart + 8 + 5 * n) * sizeof(double) + fx_veff_bytes(n);
    int rc = ensure(h, &h->d_dens, &h->dens_bytes, need);
    if (rc) return rc;
    double* base = (double*)h->d_dens;
    *part = base;
    *s = base + npart;
    *r = *s + 8;
    *p = *r + n;
    *q = *p + n;
    *b = *q + n;
    return HUB_OK;
}

static LapArgs lap_args(hub_t h) {
    LapArgs a{};
    double c0, c[kMaxHalf];
    fd_laplacian_weights(h->n0, &c0, c);
    double inv2 = 0.0;
    for (int ax = 0; ax < 3; ++ax) {
        const double ih2 = 1.0 / (h->h[ax] * h->h[ax]);
        inv2 += ih2;
        for (int p = 0; p < h->n0; ++p) a.w[ax][p] = c[p] * ih2;
    }
    a.center = c0 * inv2;
    a.n0 = h->n0;
    a.n1 = h->n1; a.n2 = h->n2; a.n3 = h->n3;
    return a;
}

// s[slot] = scale * sum of the partials of the last partial kernel
static int reduce_to(hub_t h, const double* part, int nblk, double scale, double* s, int slot) {
    k_reduce<<<1, kThreads, 0, h->stream>>>(part, nblk, scale, s, slot);
    h->launches++;
    HUB_CUDA_TRY(h, cudaGetLastError());
    return HUB_OK;
}

// The CG on one right-hand side; zero: a potential of zeros with its fixed-point form
struct CgState {
    double shift;
    double *part, *s, *r, *p, *q, *x;
    const double* zero;
};

// q = (-Lap_h + shift) v as twice the kinetic stencil in fixed point (stencil_fx.cu) with the scale in
// h->d_cmax, and v . q.  The plain form is bound by the FP64 pipe (37 operations per point; 75 us on
// 88x88x84 against 31, whose few CTAs convert most points several times).
static int cg_apply(hub_t h, const CgState& c, const double* v) {
    const LapArgs la = lap_args(h);
    StencilArgs a{};
    a.Y = v;
    a.Yout = c.q;
    a.V = c.zero;
    a.n1 = h->n1; a.n2 = h->n2; a.n3 = h->n3;
    a.ld = (int)h->Nd;
    a.ncol = 1;
    a.n0 = h->n0;
    for (int ax = 0; ax < 3; ++ax)
        for (int p = 0; p < h->n0; ++p) a.wbase[ax][p] = -0.5 * la.w[ax][p];
    a.alpha = 2.0;
    a.shift = -0.5 * c.shift;
    a.cmax_ready = true;
    return launch_stencil_fx_dot(h, a, StencilDot{c.s + S_RR, c.part, (unsigned*)(c.s + S_CNT)});
}

// k iterations: stencil with p . q, x and r with r . r, p with its largest magnitude
static int cg_steps(hub_t h, const CgState& c, int k) {
    const long n = h->Nd;
    const unsigned nb = (unsigned)((n + kCgPer * kThreads - 1) / (kCgPer * kThreads));
    int rc;
    for (int i = 0; i < k; ++i) {
        if ((rc = cg_apply(h, c, c.p))) return rc;
        k_cg_update<<<nb, kThreads, 0, h->stream>>>(c.x, c.r, c.p, c.q, n, c.s, c.part, h->d_cmax);
        k_cg_direction<<<nb, kThreads, 0, h->stream>>>(c.r, c.p, n, c.s, h->d_cmax);
        h->launches += 2;
    }
    HUB_CUDA_TRY(h, cudaGetLastError());
    return HUB_OK;
}

// kCgCheck iterations as a graph of this solve (its buffers are this solve's): below some 10^5 points
// the host's launches are what an iteration waits for (28x30x56: 30.0 us per iteration with five plain
// launches, 23.3 so; 88x88x84, where the device is the slower: 110 and 49 us)
struct CgGraph {
    cudaStream_t side = nullptr;
    cudaGraphExec_t exec = nullptr;
    long long launches = 0;
    ~CgGraph() {
        if (exec) cudaGraphExecDestroy(exec);
        if (side) cudaStreamDestroy(side);
    }
    int capture(hub_t h, const CgState& c) {
        HUB_CUDA_TRY(h, cudaStreamCreateWithFlags(&side, cudaStreamNonBlocking));
        HUB_CUDA_TRY(h, cudaStreamBeginCapture(side, cudaStreamCaptureModeThreadLocal));
        const cudaStream_t saved = h->stream;
        const long long l0 = h->launches;
        h->stream = side;
        h->capturing = 1;
        const int rc = cg_steps(h, c, kCgCheck);
        h->capturing = 0;
        h->stream = saved;
        launches = h->launches - l0;
        h->launches = l0;
        cudaGraph_t graph = nullptr;
        const cudaError_t e = cudaStreamEndCapture(side, &graph);
        if (rc || e != cudaSuccess) {
            if (graph) cudaGraphDestroy(graph);
            if (rc) return rc;
            HUB_CUDA_TRY(h, e);
        }
        const cudaError_t ei = cudaGraphInstantiate(&exec, graph, 0);
        cudaGraphDestroy(graph);
        HUB_CUDA_TRY(h, ei);
        return HUB_OK;
    }
};

// (-Lap_h + shift) x = b by CG from the x given; |r| <= tol |b| or max_iter iterations.
// b lives in the workspace slot `bw` (untouched).  Returns HUB_ENOCONV past max_iter.
static int cg_solve(hub_t h, double shift, const double* bw, double* x, double tol, int max_iter, int* iters) {
    double *part, *s, *r, *p, *q, *b;
    int rc = dens_ws(h, &part, &s, &r, &p, &q, &b);
    if (rc) return rc;
    const long n = h->Nd;
    const unsigned nb = blocks_for(n);
    double* zero = b + n;
    if ((rc = ensure(h, (void**)&h->d_cmax, &h->cmax_bytes, std::max(h->cmax_bytes, kColParts * sizeof(unsigned))))) return rc;
    HUB_CUDA_TRY(h, cudaMemsetAsync(s, 0, 8 * sizeof(double), h->stream));
    HUB_CUDA_TRY(h, cudaMemsetAsync(zero, 0, n * sizeof(double), h->stream));
    HUB_CUDA_TRY(h, cudaMemsetAsync(h->d_cmax, 0, kColParts * sizeof(unsigned), h->stream));
    if ((rc = launch_fx_veff(h, zero))) return rc;
    {
        ProfScope ps(h, HUB_K_DENSITY);
        k_vec_max<<<nb, kThreads, 0, h->stream>>>(x, n, h->d_cmax);
    }
    const CgState c{shift, part, s, r, p, q, x, zero};
    if ((rc = cg_apply(h, c, x))) return rc;
    HUB_CUDA_TRY(h, cudaMemsetAsync(h->d_cmax, 0, kColParts * sizeof(unsigned), h->stream));
    k_cg_start<<<nb, kThreads, 0, h->stream>>>(bw, q, r, p, n, part, (int)nb, h->d_cmax);
    h->launches += 1;
    HUB_CUDA_TRY(h, cudaGetLastError());
    if ((rc = reduce_to(h, part, nb, 1.0, s, S_RRN))) return rc;
    if ((rc = reduce_to(h, part + nb, nb, 1.0, s, S_BB))) return rc;
    double chk[4];
    HUB_CUDA_TRY(h, cudaMemcpyAsync(chk, s, 4 * sizeof(double), cudaMemcpyDeviceToHost, h->stream));
    HUB_CUDA_TRY(h, cudaStreamSynchronize(h->stream));
    const double bb = chk[S_BB];
    int it = 0;
    if (bb == 0.0) {
        HUB_CUDA_TRY(h, cudaMemsetAsync(x, 0, n * sizeof(double), h->stream));
        if (iters) *iters = 0;
        return HUB_OK;
    }
    double rr = chk[S_RRN];
    CgGraph graph;
    while (rr > tol * tol * bb && it < max_iter) {
        const int chunk = std::min(kCgCheck, max_iter - it);
        if (chunk == kCgCheck && it > 0) {
            if (!graph.exec && (rc = graph.capture(h, c))) return rc;
            HUB_CUDA_TRY(h, cudaGraphLaunch(graph.exec, h->stream));
            h->launches += graph.launches;
        } else if ((rc = cg_steps(h, c, chunk))) {
            return rc;
        }
        it += chunk;
        HUB_CUDA_TRY(h, cudaMemcpyAsync(&rr, s + S_RRN, sizeof(double), cudaMemcpyDeviceToHost, h->stream));
        HUB_CUDA_TRY(h, cudaStreamSynchronize(h->stream));
        if (!std::isfinite(rr)) return fail(h, HUB_ENONFINITE, "non-finite CG residual");
    }
    if (iters) *iters = it;
    if (rr > tol * tol * bb) return fail(h, HUB_ENOCONV, "CG reached its iteration limit");
    return HUB_OK;
}

int density_sum(hub_t h, const double* x, double* out_host) {
    double *part, *s, *r, *p, *q, *b;
    int rc = dens_ws(h, &part, &s, &r, &p, &q, &b);
    if (rc) return rc;
    const unsigned nb = blocks_for(h->Nd);
    k_partial_sum<<<nb, kThreads, 0, h->stream>>>(x, h->Nd, part);
    h->launches++;
    HUB_CUDA_TRY(h, cudaGetLastError());
    if ((rc = reduce_to(h, part, nb, 1.0, s, S_TMP))) return rc;
    HUB_CUDA_TRY(h, cudaMemcpyAsync(out_host, s + S_TMP, sizeof(double), cudaMemcpyDeviceToHost, h->stream));
    HUB_CUDA_TRY(h, cudaStreamSynchronize(h->stream));
    return HUB_OK;
}

int density_dot(hub_t h, const double* x, const double* y, int absdiff, double* out_host) {
    double *part, *s, *r, *p, *q, *b;
    int rc = dens_ws(h, &part, &s, &r, &p, &q, &b);
    if (rc) return rc;
    const unsigned nb = blocks_for(h->Nd);
    if (absdiff) k_partial_absdiff<<<nb, kThreads, 0, h->stream>>>(x, y, h->Nd, part);
    else k_partial_dot<<<nb, kThreads, 0, h->stream>>>(x, y, h->Nd, part);
    h->launches++;
    HUB_CUDA_TRY(h, cudaGetLastError());
    if ((rc = reduce_to(h, part, nb, 1.0, s, S_TMP))) return rc;
    HUB_CUDA_TRY(h, cudaMemcpyAsync(out_host, s + S_TMP, sizeof(double), cudaMemcpyDeviceToHost, h->stream));
    HUB_CUDA_TRY(h, cudaStreamSynchronize(h->stream));
    return HUB_OK;
}

int density_lincomb(hub_t h, double* y, int k, const double* const* v, const double* c,
                    const double* z, double beta) {
    if (k < 0 || k > kMaxLin) return fail(h, HUB_EINVAL, "at most 8 vectors per combination");
    LinArgs a{};
    a.k = k;
    for (int i = 0; i < k; ++i) { a.v[i] = v[i]; a.c[i] = c[i]; }
    k_lincomb<<<blocks_for(h->Nd), kThreads, 0, h->stream>>>(y, h->Nd, a, z, beta);
    h->launches++;
    HUB_CUDA_TRY(h, cudaGetLastError());
    return HUB_OK;
}

__global__ void k_fill(double* __restrict__ y, long n, double v) {
    const long g = (long)blockIdx.x * 256 + threadIdx.x;
    if (g < n) y[g] = v;
}

int density_fill(hub_t h, double* y, double value) {
    k_fill<<<blocks_for(h->Nd), 256, 0, h->stream>>>(y, h->Nd, value);
    h->launches++;
    HUB_CUDA_TRY(h, cudaGetLastError());
    return HUB_OK;
}

int density_add3(hub_t h, double* y, const double* a, const double* b, const double* c) {
    k_add3<<<blocks_for(h->Nd), kThreads, 0, h->stream>>>(y, a, b, c, h->Nd);
    h->launches++;
    HUB_CUDA_TRY(h, cudaGetLastError());
    return HUB_OK;
}

}  // namespace hub

using namespace hub;

extern "C" {

int hub_density(hub_t h, const void* X, int ncol, int ld, const double* f_host, double scale,
                double* rho_dev) {
    if (!h) return HUB_EINVAL;
    if (ncol < 0) return fail(h, HUB_EINVAL, "ncol must be >= 0");
    if ((long)ld < h->Nd) return fail(h, HUB_EINVAL, "ld must be >= n1*n2*n3");
    if (!rho_dev) return fail(h, HUB_EINVAL, "NULL density");
    if (ncol == 0) return HUB_OK;
    if (!X || !f_host) return fail(h, HUB_EINVAL, "NULL block or occupations");
    int rc;
    const size_t need = (size_t)ncol * sizeof(double);
    if ((rc = ensure(h, &h->d_aux, &h->aux_bytes, std::max(need, h->aux_bytes)))) return rc;
    double* f_dev = (double*)h->d_aux;
    HUB_CUDA_TRY(h, cudaMemcpyAsync(f_dev, f_host, need, cudaMemcpyHostToDevice, h->stream));
    const unsigned nb = blocks_for(h->Nd);
    ProfScope ps(h, HUB_K_DENSITY);
    if (h->esize == 8) {
        if (h->cplx) k_density<double2><<<nb, kThreads, 0, h->stream>>>((const double2*)X, ld, ncol, h->Nd, f_dev, scale, rho_dev);
        else k_density<double><<<nb, kThreads, 0, h->stream>>>((const double*)X, ld, ncol, h->Nd, f_dev, scale, rho_dev);
    } else {
        if (h->cplx) k_density<float2><<<nb, kThreads, 0, h->stream>>>((const float2*)X, ld, ncol, h->Nd, f_dev, scale, rho_dev);
        else k_density<float><<<nb, kThreads, 0, h->stream>>>((const float*)X, ld, ncol, h->Nd, f_dev, scale, rho_dev);
    }
    HUB_CUDA_TRY(h, cudaGetLastError());
    return HUB_OK;
}

int hub_hartree(hub_t h, const double* rho_dev, double* V_dev, double tol, int max_iter,
                int* iters_out, double* EH_out) {
    hub::NvtxRange nvtx_("hub_hartree");
    if (!h) return HUB_EINVAL;
    if (!rho_dev || !V_dev) return fail(h, HUB_EINVAL, "NULL density or potential");
    if (!(tol > 0.0) || max_iter < 1) return fail(h, HUB_EINVAL, "tol must be > 0 and max_iter >= 1");
    double *part, *s, *r, *p, *q, *b;
    int rc = dens_ws(h, &part, &s, &r, &p, &q, &b);
    if (rc) return rc;
    const long n = h->Nd;
    const unsigned nb = blocks_for(n);
    {
        ProfScope ps(h, HUB_K_DENSITY);
        k_partial_sum<<<nb, kThreads, 0, h->stream>>>(rho_dev, n, part);
        HUB_CUDA_TRY(h, cudaGetLastError());
    }
    if ((rc = reduce_to(h, part, nb, 1.0, s, S_TMP))) return rc;
    k_center_scale<<<nb, kThreads, 0, h->stream>>>(rho_dev, b, n, 4.0 * M_PI, s, S_TMP);
    h->launches++;
    HUB_CUDA_TRY(h, cudaGetLastError());
    if ((rc = cg_solve(h, 0.0, b, V_dev, tol, max_iter, iters_out))) return rc;
    // remove the constant the singular operator leaves undetermined: V <- V - sum(V) / n
    k_partial_sum<<<nb, kThreads, 0, h->stream>>>(V_dev, n, part);
    h->launches++;
    HUB_CUDA_TRY(h, cudaGetLastError());
    if ((rc = reduce_to(h, part, nb, 1.0, s, S_TMP))) return rc;
    k_center_scale<<<nb, kThreads, 0, h->stream>>>(V_dev, V_dev, n, 1.0, s, S_TMP);
    h->launches++;
    HUB_CUDA_TRY(h, cudaGetLastError());
    if (EH_out) {
        double d = 0.0;
        if ((rc = density_dot(h, rho_dev, V_dev, 0, &d))) return rc;
        *EH_out = 0.5 * h->dV * d;
    }
    return HUB_OK;
}

int hub_lda_exchange(hub_t h, int nchan, const double* rho0, const double* rho1, double* vx0,
                     double* vx1, double* Ex_out) {
    if (!h) return HUB_EINVAL;
    if (nchan != 1 && nchan != 2) return fail(h, HUB_EINVAL, "one or two channels");
    if (!rho0 || !vx0 || (nchan == 2 && (!rho1 || !vx1))) return fail(h, HUB_EINVAL, "NULL density or potential");
    double *part, *s, *r, *p, *q, *b;
    int rc = dens_ws(h, &part, &s, &r, &p, &q, &b);
    if (rc) return rc;
    const long n = h->Nd;
    const unsigned nb = blocks_for(n);
    const double k = 0.75 * std::cbrt(3.0 / M_PI) * (nchan == 2 ? std::cbrt(2.0) : 1.0);
    double E = 0.0;
    for (int c = 0; c < nchan; ++c) {
        {
            ProfScope ps(h, HUB_K_DENSITY);
            k_lda_x<<<nb, kThreads, 0, h->stream>>>(c ? rho1 : rho0, c ? vx1 : vx0, n, k, part);
            HUB_CUDA_TRY(h, cudaGetLastError());
        }
        if ((rc = reduce_to(h, part, nb, h->dV, s, S_TMP))) return rc;
        double e = 0.0;
        HUB_CUDA_TRY(h, cudaMemcpyAsync(&e, s + S_TMP, sizeof(double), cudaMemcpyDeviceToHost, h->stream));
        HUB_CUDA_TRY(h, cudaStreamSynchronize(h->stream));
        E += e;
    }
    if (Ex_out) *Ex_out = E;
    return HUB_OK;
}

int hub_kerker(hub_t h, const double* r_dev, double* z_dev, double kappa, double tol, int max_iter,
               int* iters_out) {
    hub::NvtxRange nvtx_("hub_kerker");
    if (!h) return HUB_EINVAL;
    if (!r_dev || !z_dev) return fail(h, HUB_EINVAL, "NULL residual or output");
    if (!(kappa >= 0.0) || !(tol > 0.0) || max_iter < 1) return fail(h, HUB_EINVAL, "bad kappa, tol or max_iter");
    double *part, *s, *r, *p, *q, *b;
    int rc = dens_ws(h, &part, &s, &r, &p, &q, &b);
    if (rc) return rc;
    const unsigned nb = blocks_for(h->Nd);
    {
        ProfScope ps(h, HUB_K_DENSITY);
        k_neg_lap<<<nb, kThreads, 0, h->stream>>>(r_dev, b, lap_args(h));   // b = -Lap r
        HUB_CUDA_TRY(h, cudaGetLastError());
    }
    HUB_CUDA_TRY(h, cudaMemsetAsync(z_dev, 0, h->Nd * sizeof(double), h->stream));
    return cg_solve(h, kappa * kappa, b, z_dev, tol, max_iter, iters_out);
}

}  // extern "C"

// Digit form of the projector gather and scatter (Sec. II.B: the inner products of all
// functions of an atom are computed together) for FP64 blocks, complex blocks and real float
// blocks whose grid has no brick tables of the TF32 form.
//
// GB300's FP64 pipe does 2 multiply-adds per clock and SM, so the FP64 products of the
// point-major form ran at its limit (gather 9.09 ms, scatter 8.99 ms on 88 x 88 x 84 x 348; now
// 1.12 and 1.33 ms).  Both are small dense products per brick of 8 x 8 x 4 points, and here they run on the FP16
// tensor cores with operands split into 7 (double) or 4 (float) 8-bit digits (digits.cuh):
// digit products and, where it counts, their sums are exact, so the result carries the rounding of
// the operands to 54 (30) bits below the largest magnitude of the values of X, or of the coefficients,
// around the brick and of the function, and one rounding of the sum, below the rounding of the sums it
// replaces.
//
// Complex blocks are real ones of twice the points and functions: a brick's 256 complex points
// are 512 reals (re, im alternating), a function has slot a = (phi_r, phi_i) (real part of
// <phi|x>) and slot b = (-phi_i, phi_r) (imaginary part), and the same real matrix serves the
// scatter (rows re, im; slots a, b times W_r, W_i).
//
//   gather:   part[slot, n] = sum_k G[k, slot] X[k, n]       D[128 orbitals x slots], K = reals of a brick
//   scatter:  Y[k, n] += alpha sum_slot G[k, slot] W[slot, n]   D[128 reals x orbitals], K = slots of a brick
//
// Operand layout (K-major, no swizzle): 16-byte units of 8 consecutive k of one row, 8 rows to
// a 128-byte core matrix.  The digits of one operand lie one after another along N, so that
// digit i of A times digits 1 .. S + 1 - i of B is ONE MMA whose output columns are the
// accumulators of the levels i .. S (the accumulator of a level is NP columns wide): S MMAs
// per 16 k instead of S (S + 1) / 2, and A is read from shared memory S times.
//
// Gather kernel: persistent CTAs over (group of at most NP slots of a brick, 128 orbitals)
// units.  Warp 0 issues the value copies, warp 1 the MMAs into one of two accumulators (one, for large
// groups), two sets of
// 8 warps, on alternate slices of 16 or 32 k, copy raw X by cp.async (each warp its own 16 orbitals),
// convert and store the digits, and 8 warps add the levels of finished units.  Scatter kernel: units (brick, 256 reals, NT
// orbitals); 2 (double) or 4 warps build the digits of W and 16 update Y: with 8, in one set, a unit's
// loads of Y waited for the stores of the one before (1.50 -> 1.37 ms); complex float needs the four
// builders as well (88 x 88 x 56 x 230: 0.94 -> 0.67 ms; with two 0.97).  Bounds in FP64 (88 x 88 x 28 x
// 128): the gather's ALU pipe, 70 % busy with the digits of X (tensor pipe 22 %, DRAM 33 %); the
// scatter's FP64 pipe, 62 % busy with the conversion and addition of its results (DRAM 39 %).  Every mbarrier wait is
// bounded: after its limit the CTA raises FLAG_TIMEOUT, stops issuing, drains what it issued,
// frees its TMEM and returns.
//
// Columns whose largest magnitude is outside the format (non-finite, or beyond 2^+-900 and
// 2^+-87) are computed by plain sums in the reduction and in the scatter's epilogue.
#include <algorithm>
#include <type_traits>
#include <vector>

#include "hub_internal.cuh"
#include "cplx.cuh"
#include "digits.cuh"
#include "site_transform.cuh"
#include "tcgen05.cuh"

namespace hub {

namespace {

constexpr int OZ_M = 128;                     // orbitals (gather) or reals (scatter) per tile
constexpr int OZ_MAXK = 512;                  // slots per brick at most
constexpr int OZ_SETS = 2;                     // sets of 8 converter warps, on alternate slices
constexpr int OZ_GTHREADS = 32 * (2 + 8 * OZ_SETS + 8);
// d_wmax [brick][column]: biased exponent of the largest coefficient of the brick's functions times
// the function's, + kWOff, or 0 (all zero) or kWBad (with non-finite values)
constexpr int kWOff = 4096;
constexpr int kWBad = 1 << 20;

template <typename R, int CW>
struct GCfg {
    static constexpr int S = Digits<R>::S;
    // 8-real chunks per slice: for float two MMA steps of K = 16 share a slice's waits (complex, 88 x 88 x 28 x
    // 115: 0.173 -> 0.158 ms); double has no room for the stages
    static constexpr int CH = S == 7 ? 2 : 4;
    static constexpr int NP = S == 7 ? 64 : 128;                  // slots per group at most
    // A brick of complex double is two units of 256 reals: the sums of 512 products of digits could
    // pass 2^24 (digits.cuh).  88 x 88 x 56 x 230: 2.08 ms against 1.54 for whole bricks.
    static constexpr int PARTS = S == 7 ? CW : 1;
    static constexpr int SLICES = BRP * CW / (8 * CH) / PARTS;
    static constexpr int CB = 8 * (int)sizeof(R), PC = CB / 16;   // a raw chunk, its 16-byte pieces
    static constexpr int PPP = 16 / (int)sizeof(R) / CW;          // points per piece (complex double: 1)
    static constexpr int XB = S * CH * OZ_M * 16;              // digits of one X slice
    static constexpr int VB = CH * S * NP * 16;                // values of one slice
    static constexpr int NS = 2;                     // X stages: a multiple of the sets
    static constexpr int NV = S == 7 ? 4 : 2;                                  // value stages
    static constexpr int RAW = OZ_M * CH * CB;
    static constexpr int ND = S == 7 ? 3 : 2;                     // raw slices in flight per set (80 to 96 KB in all)
    static constexpr size_t SMEM = (size_t)NS * XB + (size_t)NV * VB + (size_t)OZ_SETS * ND * RAW + 1024;
    static_assert(S * NP <= 512 && SMEM <= 227 * 1024, "TMEM, shared memory");
    // TMEM columns of a unit of np slots: even units from the start, odd ones up to the end, so that
    // two small units are in flight and a large one has all of it
    static __device__ __forceinline__ uint32_t column(int uu, int np) { return uu & 1 ? 512u - (uint32_t)(S * np) : 0u; }
};

template <typename R, int CW>
struct SCfg {
    static constexpr int S = Digits<R>::S;
    static constexpr int NT = S == 7 ? 16 : 32;                   // orbitals per unit
    static constexpr int PASSES = BRP * CW / 256;                 // 256 reals per unit
    static constexpr int AU = 2 * S * 2 * OZ_M;                   // 16-byte units of a chunk of 16 slots
    static constexpr int AB = AU * 16;
    static constexpr int BB = 2 * S * NT * 16;
    static constexpr int NS = S == 7 ? 3 : 5;                     // chunks of values in flight or resident
    static constexpr int NB = 8;                                  // chunks of W digits
    static constexpr int BW = S == 7 ? 2 : 4;                     // warps that build the digits of W
    static constexpr int PCH = 16;                                // chunks per read-out of the wide form
    static constexpr int THREADS = 32 * (2 + BW + 16);
    static constexpr int ACC = S * NT;
    static constexpr size_t SMEM = (size_t)NS * AB + NB * BB + 1024;
    static_assert(4 * ACC <= 512 && ACC <= 256, "two units of two tiles in TMEM");
    static_assert(SMEM <= 227 * 1024, "shared memory");
};

struct OzGather {
    const void* X;
    const int4* grp;          // brick, slots, 16-byte offset, first slot
    const int2* slot;         // partial row (-1: padding), exponent of the function
    const uint4* val;
    double* part;
    BlockMap bmax;            // maxima of X
    int* wmax;                // cleared for the reduction: nw values
    long nw;
    long part_rows;           // rows of one part of the bricks
    long ld;                  // in reals
    int n1, n2, n3, ncol, nbx, nby, nunits, ctiles, vec;
    int* flags;
};

// scale of a column's digits on a brick: the largest exponent of the pieces around it, at least the
// smallest of the format; a brick with non-finite or larger values has zero digits (its column is
// summed in the reduction)
template <typename R, int CW>
__device__ __forceinline__ int oz_exponent(const OzGather& a, int x, int y, int z, int col) {
    if (col >= a.ncol) return 1 << 14;
    const unsigned m = brick_max(a.bmax, col, x, y, z, a.n3);
    const int E = max((int)(m >> (sizeof(R) == 8 ? 20 : 23)), Digits<R>::kEmin);
    return E > Digits<R>::kEmax ? 1 << 14 : E;
}

template <typename R, int CW>
__global__ void __launch_bounds__(OZ_GTHREADS, 1)
k_gather_oz(OzGather a) {
    using C = GCfg<R, CW>;
    constexpr int S = C::S;
    extern __shared__ __align__(1024) unsigned char dsm[];
    unsigned char* ring = reinterpret_cast<unsigned char*>((reinterpret_cast<uintptr_t>(dsm) + 1023) & ~(uintptr_t)1023);
    unsigned char* vring = ring + (size_t)C::NS * C::XB;
    __shared__ __align__(8) uint64_t x_bar[C::NS], empty_bar[C::NS], full_bar[C::NV], vempty_bar[C::NV], tfull_bar[2],
        tempty_bar[2], done_bar;
    __shared__ uint32_t tmem_slot;
    __shared__ volatile int abort_flag;
    __shared__ int issued_sh;

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int nu = (a.nunits - (int)blockIdx.x + (int)gridDim.x - 1) / (int)gridDim.x;
    for (long i = (long)blockIdx.x * OZ_GTHREADS + threadIdx.x; i < a.nw; i += (long)gridDim.x * OZ_GTHREADS) a.wmax[i] = 0;

    if (threadIdx.x == 0) {
        abort_flag = 0;
        issued_sh = 0;
        for (int s = 0; s < C::NS; ++s) {
            mbar_init(&x_bar[s], 256);
            mbar_init(&empty_bar[s], 1);
        }
        for (int s = 0; s < C::NV; ++s) {
            mbar_init(&full_bar[s], 1);
            mbar_init(&vempty_bar[s], 1);
        }
        for (int b = 0; b < 2; ++b) {
            mbar_init(&tfull_bar[b], 1);
            mbar_init(&tempty_bar[b], 256);
        }
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
            int i = 0;
            for (int uu = 0; uu < nu && !abort_flag; ++uu) {
                const int u = (int)blockIdx.x + uu * (int)gridDim.x, part = (u / a.ctiles) % C::PARTS;
                const int4 G = a.grp[u / (a.ctiles * C::PARTS)];
                const uint32_t units = (uint32_t)(C::CH * S * G.y);
                bool stop = false;
                for (int q = 0; q < C::SLICES; ++q, ++i) {
                    const int s = i % C::NV;
                    if (i >= C::NV && !mbar_wait(&vempty_bar[s], ((i / C::NV) - 1) & 1, &abort_flag)) { stop = true; break; }
                    mbar_expect_tx(&full_bar[s], units * 16);
                    bulk_load(vring + (size_t)s * C::VB, a.val + (size_t)G.z + (size_t)(part * C::SLICES + q) * units, units * 16,
                              &full_bar[s]);
                    issued_sh = i + 1;
                }
                if (stop) break;
            }
        }
    } else if (warp == 1) {
        const bool el = elect_one();
        auto wait = [&](uint64_t* bar, int parity) { return __all_sync(0xffffffffu, mbar_wait(bar, parity, &abort_flag)) != 0; };
        const uint32_t a0 = desc_lo(ring, OZ_M * 16);
        int s = 0, ph = 0, sv = 0, pv = 0;          // X and value stages and their phases
        bool stop = false;
        uint32_t before = 0;                        // slots of the unit before
        for (int uu = 0; uu < nu && !stop; ++uu) {
            const uint32_t np = (uint32_t)__shfl_sync(0xffffffffu, a.grp[((int)blockIdx.x + uu * (int)gridDim.x) / (a.ctiles * C::PARTS)].y, 0);
            const int buf = uu & 1;
            if (uu >= 2 && !wait(&tempty_bar[buf], ((uu >> 1) - 1) & 1)) break;
            // the unit before has to be read out first where the two don't fit
            if (uu >= 1 && S * (np + before) > 512u && !wait(&tempty_bar[buf ^ 1], ((uu - 1) >> 1) & 1)) break;
            before = np;
            tc_fence_after();
            const uint32_t d0 = tmem + C::column(uu, (int)np);
            const uint32_t idesc = instr_desc_f16(OZ_M, 0), step = np << 14, i0 = idesc + S * step;    // of N
            const uint32_t b0 = desc_lo(vring, S * np * 16);
            for (int q = 0; q < C::SLICES; ++q) {
                if (!wait(&full_bar[sv], pv) || !wait(&x_bar[s], ph)) { stop = true; break; }
                tc_fence_after();
                if (el) {
                    const uint32_t ao = a0 + (uint32_t)(s * (C::XB / 16)), bo = b0 + (uint32_t)(sv * (C::VB / 16));
                    auto issue = [&](auto wide) {
#pragma unroll
                        for (int kk = 0; kk < C::CH / 2; ++kk)
#pragma unroll
                            for (int d = 0; d < S; ++d) {
                                // levels d .. S - 1: N columns, at most 256 per instruction
                                const uint32_t N = (uint32_t)(S - d) * np, dc = d0 + (uint32_t)d * np;
                                const uint32_t ad = ao + (uint32_t)((d * C::CH + 2 * kk) * OZ_M), bd = bo + (uint32_t)(2 * kk) * (S * np);
                                const uint32_t more = (q > 0 || kk > 0 || d > 0) ? 1u : 0u;
                                if constexpr (decltype(wide)::value) {
                                    const uint32_t n0 = min(N, 256u);
                                    mma_f16_lo(dc, ad, bd, kDescHi, idesc + (n0 << 14), more);
                                    if (N > 256u) mma_f16_lo(dc + 256u, ad, bd + 256u, kDescHi, idesc + ((N - 256u) << 14), more);
                                } else {
                                    mma_f16_lo(dc, ad, bd, kDescHi, i0 - (uint32_t)d * step, more);
                                }
                            }
                    };
                    if (S * np > 256u) issue(std::true_type{});
                    else issue(std::false_type{});
                    mma_commit(&empty_bar[s]);
                    mma_commit(&vempty_bar[sv]);
                }
                __syncwarp();
                if (++s == C::NS) { s = 0; ph ^= 1; }
                if (++sv == C::NV) { sv = 0; pv ^= 1; }
            }
            if (el && !stop) mma_commit(&tfull_bar[buf]);
        }
        if (el) mma_commit(&done_bar);
    } else if (warp < 2 + 8 * OZ_SETS) {
        // raw X: task t of a warp is chunk t / 16 of the slice for the warp's orbital t % 16; its
        // CB bytes lie at t * CB, the 16-byte pieces permuted so that a quarter-warp's reads fall
        // into different banks.  A thread reads what its warp copied: __syncwarp is enough.
        const int set = (warp - 2) >> 3, w = (warp - 2) & 7;
        unsigned char* raw = vring + (size_t)C::NV * C::VB + (size_t)set * (C::ND * C::RAW) + (size_t)w * (16 * C::CH * C::CB);
        const int nsl = nu * C::SLICES;
        // pieces of a lane: `it` counts chunk r = it / (PC / 2), orbital j = it % (PC / 2) of the
        // lane's PC / 2; piece and place in the raw buffer depend on the lane alone
        constexpr int NJ = C::PC / 2;
        const int lp = lane % C::PC, ln = lane / C::PC;
        const uint32_t ldst = (uint32_t)(ln * C::CB + ((lp ^ ((lane >> 3) & (C::PC - 1))) << 4));
        const R* cb[NJ];
        bool cok[NJ];
        int gx = 0, gy = 0, gz = 0;                      // brick corner
        int chunk0 = 0;                                  // first chunk of the unit's part of the brick
        bool more = false;                               // the warp has orbitals in this unit
        int E = 0, Enext = 0;                            // exponent of this lane's orbital: of the unit converted and of the
                                                         // one whose copies begin (ND slices ahead, within the unit)
        static_assert(C::SLICES / OZ_SETS >= C::ND, "one unit ahead at most");
        auto issue = [&](int j) {                        // the set's j-th slice
            const int i = set + OZ_SETS * j, nq = i % C::SLICES;
            if (i < nsl) {
                if (nq == set) {
                    const int u = (int)blockIdx.x + (i / C::SLICES) * (int)gridDim.x;
                    const int brick = a.grp[u / (a.ctiles * C::PARTS)].x, c0 = (u % a.ctiles) * OZ_M + 16 * w;
                    chunk0 = (u / a.ctiles) % C::PARTS * (C::SLICES * C::CH);
                    gx = 8 * (brick % a.nbx) + C::PPP * lp;
                    gy = 8 * ((brick / a.nbx) % a.nby);
                    gz = 4 * (brick / (a.nbx * a.nby));
                    more = c0 < a.ncol;
                    Enext = oz_exponent<R, CW>(a, gx - C::PPP * lp, gy, gz, c0 + (lane & 15));
#pragma unroll
                    for (int o = 0; o < NJ; ++o) {
                        const int col = c0 + o * (32 / C::PC) + ln;
                        cok[o] = col < a.ncol;
                        cb[o] = (const R*)a.X + (size_t)(cok[o] ? col : 0) * a.ld;
                    }
                }
                const uint32_t dst = saddr(raw + (size_t)(j % C::ND) * C::RAW) + ldst;
                if (more)
#pragma unroll
                for (int r = 0; r < C::CH; ++r) {
                    const int row = (chunk0 + nq * C::CH + r) / CW, x = gx + (CW == 2 ? 4 * (r & 1) : 0);
                    const int y = gy + (row & 7), z = gz + (row >> 3);
                    const size_t off = ((size_t)x + (size_t)a.n1 * (y + (size_t)a.n2 * z)) * CW;
                    const bool rin = y < a.n2 && z < a.n3;
#pragma unroll
                    for (int o = 0; o < NJ; ++o) {
                        const uint32_t to = dst + (uint32_t)(r * NJ + o) * 512;
                        if (a.vec) {
                            const bool ok = rin && cok[o] && x < a.n1;
                            asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(to),
                                         "l"(ok ? cb[o] + off : (const R*)a.X), "r"(ok ? 16 : 0) : "memory");
                        } else {
                            constexpr int EB = (int)sizeof(R) * CW > 8 ? 8 : (int)sizeof(R) * CW;   // bytes of one copy
#pragma unroll
                            for (int e = 0; e < 16 / EB; ++e) {
                                const bool ok = rin && cok[o] && x + e * EB / ((int)sizeof(R) * CW) < a.n1;
                                asm volatile("cp.async.ca.shared.global [%0], [%1], %2, %3;" ::"r"(to + e * EB),
                                             "l"(ok ? cb[o] + off + e * (EB / (int)sizeof(R)) : (const R*)a.X), "n"(EB),
                                             "r"(ok ? EB : 0) : "memory");
                            }
                        }
                    }
                }
            }
            asm volatile("cp.async.commit_group;" ::: "memory");
        };
        auto perm = [](int t) { return C::PC == 4 ? (t >> 1) & 3 : (t >> 2) & 1; };
        for (int j = 0; j < C::ND; ++j) issue(j);
        bool any = false;                        // a warp without orbitals leaves its rows as they are: they reach only
                                                 // their own outputs
        for (int i = set, j = 0; i < nsl; i += OZ_SETS, ++j) {
            if (i % C::SLICES == set) {
                const int u = (int)blockIdx.x + (i / C::SLICES) * (int)gridDim.x;
                any = (u % a.ctiles) * OZ_M + 16 * w < a.ncol;
                E = Enext;
            }
            asm volatile("cp.async.wait_group %0;" ::"n"(C::ND - 1) : "memory");
            __syncwarp();
            const unsigned char* src = raw + (size_t)(j % C::ND) * C::RAW;
            typename Digits<R>::I b[C::CH / 2][8];
            if (any)
#pragma unroll
            for (int it = 0; it < C::CH / 2; ++it) {
                const int t = it * 32 + lane;
                R v[8];
#pragma unroll
                for (int p = 0; p < C::PC; ++p)
                    *reinterpret_cast<uint4*>(&v[p * (16 / (int)sizeof(R))]) =
                        *reinterpret_cast<const uint4*>(src + t * C::CB + ((p ^ perm(t)) << 4));
#pragma unroll
                for (int k = 0; k < 8; ++k) b[it][k] = Digits<R>::bytes(v[k], E);
            }
            __syncwarp();                        // the raw buffer may be refilled
            issue(j + C::ND);
            const int s = i % C::NS;
            const bool ok = i < C::NS || mbar_wait(&empty_bar[s], ((i / C::NS) - 1) & 1, &abort_flag);
            if (__any_sync(0xffffffffu, !ok)) break;
            unsigned char* xs = ring + (size_t)s * C::XB;
            if (any)
#pragma unroll
            for (int it = 0; it < C::CH / 2; ++it) {
                const int t = it * 32 + lane;
                unsigned char* to = xs + ((size_t)(t >> 4) * OZ_M + 16 * w + (t & 15)) * 16;
#pragma unroll
                for (int d = 0; d < S; ++d) {
                    __half2 o[4];
#pragma unroll
                    for (int k = 0; k < 4; ++k) o[k] = digit_pair<R>(b[it][2 * k], b[it][2 * k + 1], d);
                    *reinterpret_cast<uint4*>(to + (size_t)d * (C::CH * OZ_M * 16)) = *reinterpret_cast<uint4*>(o);
                }
            }
            fence_proxy_async();
            mbar_arrive(&x_bar[s]);
        }
        asm volatile("cp.async.wait_group 0;" ::: "memory");
    } else {
        // level sums of finished units: TMEM lane = orbital, two warps per lane quarter on alternate
        // groups of F slots
        constexpr int F = S == 7 ? 4 : 8;
        const int quad = warp & 3, half = (warp - 2 - 8 * OZ_SETS) >> 2;
        const uint32_t lane_base = (uint32_t)(32 * quad) << 16;
        for (int uu = 0; uu < nu; ++uu) {
            const int u = (int)blockIdx.x + uu * (int)gridDim.x;
            const int buf = uu & 1;
            const int4 G = a.grp[u / (a.ctiles * C::PARTS)];
            const size_t row0 = (size_t)((u / a.ctiles) % C::PARTS) * a.part_rows;
            const int col = (u % a.ctiles) * OZ_M + 32 * quad + lane;
            const int E = oz_exponent<R, CW>(a, 8 * (G.x % a.nbx), 8 * (G.x / a.nbx % a.nby), 4 * (G.x / (a.nbx * a.nby)), col);
            const bool ok = mbar_wait(&tfull_bar[buf], (uu >> 1) & 1, &abort_flag);
            if (__any_sync(0xffffffffu, !ok)) break;
            tc_fence_after();
            for (int c0 = F * half; c0 < G.y; c0 += 2 * F) {
                int4 sl[F / 2];                          // (partial row, exponent) of two slots each
#pragma unroll
                for (int f = 0; f < F / 2; ++f) sl[f] = reinterpret_cast<const int4*>(a.slot + G.w + c0)[f];
                uint32_t v[S * F];
                // level l of slot c at column l * (slots of the group) + c
                const uint32_t base = tmem + lane_base + C::column(uu, G.y) + (uint32_t)c0;
#pragma unroll
                for (int l = 0; l < S; ++l) {
                    if constexpr (F == 8) tmem_ld8(base + (uint32_t)(l * G.y), v + 8 * l);
                    else tmem_ld4(base + (uint32_t)(l * G.y), v + 4 * l);
                }
                asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
                for (int l = 0; l < S; ++l) {
                    if constexpr (F == 8) keep8(v + 8 * l);
                    else keep4(v + 4 * l);
                }
#pragma unroll
                for (int f = 0; f < F; ++f) {
                    const int row = f & 1 ? sl[f / 2].z : sl[f / 2].x, e = f & 1 ? sl[f / 2].w : sl[f / 2].y;
                    long long lo;
                    const long long hi = level_sum<R, F>(v + f, &lo);
                    double r;
                    int k = E + e - 2 * Digits<R>::kUnit;
                    if constexpr (S == 7) {
                        // (hi 2^24 + lo) 256^6
                        r = fma((double)hi, 16777216.0, (double)lo);
                        k += 48;
                    } else {
                        r = (double)hi;
                        k += 24;
                    }
                    r = scale2(r, k);
                    if (row >= 0 && col < a.ncol) a.part[(row0 + row) * a.ncol + col] = r;
                }
            }
            tc_fence_before();
            mbar_arrive(&tempty_bar[buf]);
        }
    }
    __syncwarp();
    __syncthreads();
    if (threadIdx.x == 0) {
        if (!mbar_drain(&done_bar, 0)) abort_flag = 1;
        if (abort_flag) {
            atomicExch(a.flags + FLAG_TIMEOUT, 1);
            const int issued = issued_sh;
            for (int j = issued > C::NV ? issued - C::NV : 0; j < issued; ++j)
                mbar_drain(&full_bar[j % C::NV], (j / C::NV) & 1);
        }
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 0) {
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(512u) : "memory");
    }
}

// ---------------------------------------------------------------------------- reduction
// C of every projector row from its partial rows (a fixed order: deterministic), W by the
// coefficient transform, and the column maxima of W 2^exponent for the scatter's digits.  One
// CTA per (site, 32 columns): warp w sums the partial rows w, w + 8, ... of each of the site's
// functions, then one lane per column adds the eight sums and transforms.
struct OzReduce {
    const SiteDev* sites;
    const int* roff;
    const int* rent;
    const double* part;
    const double* gamma;
    const double* M;
    const int* exps;
    double* C;
    void* W;
    int* wmax;
    const int* sfirst;        // bricks of every site
    const int* sbrick;
    const unsigned* cmax;
    const void* X;
    const int* idx;
    const void* vals;
    long part_rows;
    long ld;                  // in elements
    double dV;
    int ncol, want_W;
};

// A site's coefficients of column n (per lane; written by warp 0, which takes their maximum) into the
// maxima of the bricks that its functions reach.  256 threads, 32 columns.
template <typename R, int CW>
__device__ __forceinline__ void raise_wmax(const SiteDev& S, const R* W, const int* exps, const int* sfirst, const int* sbrick, int n,
                                           int ncol, int* wmax) {
    __shared__ int tops[32];
    const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (w == 0) {
        int top = 0;
        if (n < ncol)
            for (int p = 0; p < S.nproj; ++p)
                for (int q = 0; q < CW; ++q) {
                    const int e = Digits<R>::exponent(W[((size_t)(S.proj_off + p) * ncol + n) * CW + q]);
                    if (e == (sizeof(R) == 8 ? 0x7ff : 0xff)) top = kWBad;
                    else if (e > 0) top = max(top, e + exps[S.proj_off + p] - Digits<R>::kBias + kWOff);
                }
        tops[lane] = top;
    }
    __syncthreads();
    const int top = tops[lane];
    if (top == 0) return;
    for (int e = sfirst[blockIdx.x] + w; e < sfirst[blockIdx.x + 1]; e += 8) atomicMax(wmax + (size_t)sbrick[e] * ncol + n, top);
}

template <typename R, int CW>
__global__ void __launch_bounds__(256)
k_reduce_oz(OzReduce a) {
    constexpr bool CPLX = CW == 2;
    using D = typename VT<double, CPLX>::T;
    using T = typename VT<R, CPLX>::T;
    __shared__ double red[8][kMaxProj * CW][32];
    __shared__ double rsum[8][2];
    const SiteDev S = a.sites[blockIdx.x];
    const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int n = blockIdx.y * 32 + lane;
    const int nr = S.nproj * CW;
    auto partial = [&](int e, int c) {
        const size_t row = (size_t)a.rent[e] * CW + c;
        double v = a.part[row * a.ncol + n];
#pragma unroll
        for (int k = 1; k < GCfg<R, CW>::PARTS; ++k) v += a.part[(row + k * a.part_rows) * a.ncol + n];
        return v;
    };
    for (int p = 0; p < S.nproj; ++p) {
        const int e0 = a.roff[S.proj_off + p], e1 = a.roff[S.proj_off + p + 1];
        double acc[CW] = {};
        if (n < a.ncol) {
            int e = e0 + w;
            for (; e + 24 < e1; e += 32) {
                double v[4][CW];
#pragma unroll
                for (int k = 0; k < 4; ++k)
#pragma unroll
                    for (int c = 0; c < CW; ++c) v[k][c] = partial(e + 8 * k, c);
#pragma unroll
                for (int k = 0; k < 4; ++k)
#pragma unroll
                    for (int c = 0; c < CW; ++c) acc[c] += v[k][c];
            }
            for (; e < e1; e += 8)
#pragma unroll
                for (int c = 0; c < CW; ++c) acc[c] += partial(e, c);
        }
#pragma unroll
        for (int c = 0; c < CW; ++c) red[w][p * CW + c][lane] = acc[c];
    }
    __syncthreads();
    for (int r = w; r < nr; r += 8) {
        double s = 0.0;
#pragma unroll
        for (int k = 0; k < 8; ++k) s += red[k][r][lane];
        red[0][r][lane] = a.dV * s;
    }
    // columns outside the digit format: plain sums over the site's points
    const unsigned m = n < a.ncol ? column_max(a.cmax, n) : 0u;
    const int E = (int)(m >> (sizeof(R) == 8 ? 20 : 23));
    const unsigned bad = __ballot_sync(0xffffffffu, m != 0u && (E < Digits<R>::kEmin || E > Digits<R>::kEmax));
    __syncthreads();
    for (unsigned b = bad; b; b &= b - 1) {                       // the same in every warp
        const int j = __ffs((int)b) - 1;
        const T* x = (const T*)a.X + (size_t)(blockIdx.y * 32 + j) * a.ld;
        const T* vals = (const T*)a.vals + S.val_off;
        for (int p = 0; p < S.nproj; ++p) {
            D acc = zero_of(D());
            for (int i = threadIdx.x; i < S.npts; i += 256) {
                D xv, pv;
                if constexpr (CPLX) {
                    const T xx = x[a.idx[S.pt_off + i]], pp = vals[(size_t)i * S.nproj + p];
                    xv = make_double2((double)xx.x, (double)xx.y);
                    pv = make_double2((double)pp.x, (double)pp.y);
                } else {
                    xv = (double)x[a.idx[S.pt_off + i]];
                    pv = (double)vals[(size_t)i * S.nproj + p];
                }
                acc = cfma_conj(pv, xv, acc);
            }
            for (int o = 16; o > 0; o >>= 1) acc = add(acc, shfl_down(acc, o));
            if (lane == 0) {
                if constexpr (CPLX) { rsum[w][0] = acc.x; rsum[w][1] = acc.y; }
                else rsum[w][0] = acc;
            }
            __syncthreads();
            if (threadIdx.x < CW) {
                double s = 0.0;
                for (int k = 0; k < 8; ++k) s += rsum[k][threadIdx.x];
                red[0][p * CW + threadIdx.x][j] = a.dV * s;
            }
            __syncthreads();
        }
    }
    if (w == 0 && n < a.ncol) {
        D c[kMaxProj];
        for (int p = 0; p < S.nproj; ++p) {
            if constexpr (CPLX) c[p] = make_double2(red[0][2 * p][lane], red[0][2 * p + 1][lane]);
            else c[p] = red[0][p][lane];
            ((D*)a.C)[(size_t)(S.proj_off + p) * a.ncol + n] = c[p];
        }
        if (a.want_W) site_transform<R, CPLX>(S, c, a.gamma, a.M, (T*)a.W, n, a.ncol);
    }
    if (a.want_W) raise_wmax<R, CW>(S, (const R*)a.W, a.exps, a.sfirst, a.sbrick, n, a.ncol, a.wmax);
}

// maxima of a W that did not come from the reduction (wmax cleared before): one CTA per (site, 32 columns)
template <typename R, int CW>
__global__ void __launch_bounds__(256)
k_wmax_oz(const SiteDev* __restrict__ sites, const R* __restrict__ W, const int* __restrict__ exps, const int* __restrict__ sfirst,
          const int* __restrict__ sbrick, int ncol, int* __restrict__ wmax) {
    raise_wmax<R, CW>(sites[blockIdx.x], W, exps, sfirst, sbrick, blockIdx.y * 32 + (threadIdx.x & 31), ncol, wmax);
}

// ---------------------------------------------------------------------------- scatter
struct OzScatter {
    void* Y;
    const int4* brick;        // brick, slots (multiple of 16), 16-byte offset, first slot
    const int2* slot;         // real row of W (-1: padding), exponent of the function
    const uint4* val;
    const void* W;
    const int* wmax;
    const int* csr_off;       // the point-major table: columns outside the format
    const int2* csr_ent;
    const void* vals;
    double alpha;
    const double* alpha_dev;
    long ld;                  // in reals
    int ncol, n1, n2, n3, nbx, nby, nbricks, ctiles;
    int* flags;
};

// sum of the point-major entries of grid point g for column n (component comp of a complex one)
template <typename R, int CW>
__device__ __noinline__ double oz_plain(const OzScatter& a, long g, int comp, int n) {
    double s = 0.0;
    for (int e = a.csr_off[g]; e < a.csr_off[g + 1]; ++e) {
        const int2 m = a.csr_ent[e];
        for (int p = 0; p < (m.y & 15); ++p) {
            const R* v = (const R*)a.vals + (size_t)(m.x + p) * CW;
            const R* w = (const R*)a.W + ((size_t)((m.y >> 4) + p) * a.ncol + n) * CW;
            if (CW == 1) s += (double)v[0] * (double)w[0];
            else if (comp == 0) s += (double)v[0] * (double)w[0] - (double)v[CW - 1] * (double)w[CW - 1];
            else s += (double)v[0] * (double)w[CW - 1] + (double)v[CW - 1] * (double)w[0];
        }
    }
    return s;
}

// WIDE: double, with more than 256 slots on some brick, which are read out every 256: the sums of more
// products of digits could pass 2^24 (digits.cuh).  A form of its own: the loops of the read-outs
// cost the others 5 % (88 x 88 x 84 x 348: 1.35 against 1.42 ms).
template <typename R, int CW, bool WIDE>
__global__ void __launch_bounds__(SCfg<R, CW>::THREADS, 1)
k_scatter_oz(OzScatter a) {
    using C = SCfg<R, CW>;
    constexpr int S = C::S, NT = C::NT;
    extern __shared__ __align__(1024) unsigned char dsm[];
    unsigned char* ring = reinterpret_cast<unsigned char*>((reinterpret_cast<uintptr_t>(dsm) + 1023) & ~(uintptr_t)1023);
    unsigned char* wring = ring + (size_t)C::NS * C::AB;
    __shared__ __align__(8) uint64_t full_bar[C::NS], empty_bar[C::NS], w_bar[C::NB], wempty_bar[C::NB], tfull_bar[2],
        tempty_bar[2], done_bar;
    __shared__ uint32_t tmem_slot;
    __shared__ volatile int abort_flag;
    __shared__ int issued_sh;

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    // units of this CTA: (brick, pass) pairs blockIdx.x, + gridDim.x, ..., each with its orbital
    // tiles one after another.  The values of a pair with at most NS chunks stay in shared memory
    // for all its tiles; others are copied again for each (from L2).
    const int npair = a.nbricks * C::PASSES;
    const int np = (npair - (int)blockIdx.x + (int)gridDim.x - 1) / (int)gridDim.x;
    auto pair_of = [&](int q) { return (int)blockIdx.x + q * (int)gridDim.x; };

    if (threadIdx.x == 0) {
        abort_flag = 0;
        issued_sh = 0;
        for (int s = 0; s < C::NS; ++s) {
            mbar_init(&full_bar[s], 1);
            mbar_init(&empty_bar[s], 1);
        }
        for (int s = 0; s < C::NB; ++s) {
            mbar_init(&w_bar[s], 32);
            mbar_init(&wempty_bar[s], 1);
        }
        for (int b = 0; b < 2; ++b) {
            mbar_init(&tfull_bar[b], 1);
            mbar_init(&tempty_bar[b], 256);
        }
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
            int i = 0;
            bool stop = false;
            for (int q = 0; q < np && !stop; ++q) {
                const int pr = pair_of(q);
                const int4 B = a.brick[pr / C::PASSES];
                const int nk = B.y / 16;
                const uint4* src = a.val + (size_t)B.z + (size_t)(pr % C::PASSES) * nk * C::AU;
                const int loads = nk <= C::NS ? nk : nk * a.ctiles;
                for (int l = 0; l < loads; ++l, ++i) {
                    const int s = i % C::NS;
                    if (i >= C::NS && !mbar_wait(&empty_bar[s], ((i / C::NS) - 1) & 1, &abort_flag)) { stop = true; break; }
                    mbar_expect_tx(&full_bar[s], C::AB);
                    bulk_load(ring + (size_t)s * C::AB, src + (size_t)(l % nk) * C::AU, C::AB, &full_bar[s]);
                    issued_sh = i + 1;
                }
            }
        }
    } else if (warp == 1) {
        const bool el = elect_one();
        auto wait = [&](uint64_t* bar, int parity) { return __all_sync(0xffffffffu, mbar_wait(bar, parity, &abort_flag)) != 0; };
        const uint32_t a0 = desc_lo(ring, OZ_M * 16), b0 = desc_lo(wring, S * NT * 16);
        int ia = 0, sb = 0, pb = 0, uu = 0;         // value chunks so far, W stage and its phase, units so far
        int used0 = 0, used1 = 0;                   // read-outs so far of either buffer (WIDE)
        bool stop = false;
        for (int q = 0; q < np && !stop; ++q) {
            const int nk = __shfl_sync(0xffffffffu, a.brick[pair_of(q) / C::PASSES].y, 0) / 16;
            const bool keep = nk <= C::NS;
            for (int ct = 0; ct < a.ctiles && !stop; ++ct, ++uu) {
                const int buf = uu & 1;
                const uint32_t d0 = tmem + (uint32_t)(buf * 2 * C::ACC);
                int s = (keep ? ia : ia + ct * nk) % C::NS, ph = ((keep ? ia : ia + ct * nk) / C::NS) & 1;
                int used = WIDE ? (buf ? used1 : used0) : uu >> 1;
                if (used >= 1 && !wait(&tempty_bar[buf], (used - 1) & 1)) { stop = true; break; }
                tc_fence_after();
                for (int c = 0; c < nk; ++c) {
                    if (WIDE && c > 0 && c % C::PCH == 0) {            // read out in between
                        if (el) mma_commit(&tfull_bar[buf]);
                        ++used;
                        if (!wait(&tempty_bar[buf], (used - 1) & 1)) { stop = true; break; }
                        tc_fence_after();
                    }
                    if (!wait(&full_bar[s], ph) || !wait(&w_bar[sb], pb)) { stop = true; break; }
                    tc_fence_after();
                    if (el) {
                        const uint32_t ao = a0 + (uint32_t)(s * (C::AB / 16)), bo = b0 + (uint32_t)(sb * (C::BB / 16));
                        const uint32_t more = (WIDE ? c % C::PCH : c) > 0 ? 1u : 0u;
#pragma unroll
                        for (int t = 0; t < 2; ++t)
#pragma unroll
                            for (int d = 0; d < S; ++d)
                                mma_f16_lo(d0 + (uint32_t)(t * C::ACC + d * NT), ao + (uint32_t)((t * S + d) * (2 * OZ_M)), bo, kDescHi,
                                           instr_desc_f16(OZ_M, (S - d) * NT), d > 0 ? 1u : more);
                        mma_commit(&wempty_bar[sb]);
                        if (!keep || ct == a.ctiles - 1) mma_commit(&empty_bar[s]);
                    }
                    __syncwarp();
                    if (++s == C::NS) { s = 0; ph ^= 1; }
                    if (++sb == C::NB) { sb = 0; pb ^= 1; }
                }
                if (el && !stop) mma_commit(&tfull_bar[buf]);
                if (WIDE) (buf ? used1 : used0) = used + 1;
            }
            ia += keep ? nk : nk * a.ctiles;
        }
        if (el) mma_commit(&done_bar);
    } else if (warp < 2 + C::BW) {
        // digits of W^T, chunks of 16 slots: warp b builds the chunks b, b + C::BW, ... (which divides NB: a
        // warp waits for every phase of its own stages in turn); lane task (orbital, 8 slots),
        // NT / 16 tasks per lane
        const int b = warp - 2;
        int i = 0;
        bool stop = false;
        for (int q = 0; q < np && !stop; ++q) {
            const int4 B = a.brick[pair_of(q) / C::PASSES];
            const int* wmax = a.wmax + (size_t)(pair_of(q) / C::PASSES) * a.ncol;
            const int nk = B.y / 16;
            for (int l = 0; l < nk * a.ctiles; ++l, ++i) {
                if (i % C::BW != b) continue;
                const int s = i % C::NB, c = l % nk, c0 = (l / nk) * NT;
                typename Digits<R>::I v[NT / 16][8];
#pragma unroll
                for (int it = 0; it < NT / 16; ++it) {
                    const int task = it * 32 + lane, o = task % NT, kc = task / NT, col = c0 + o;
                    const int4* sl = reinterpret_cast<const int4*>(a.slot + B.w + c * 16 + kc * 8);
                    const int wm = col < a.ncol ? wmax[col] : 0;
                    const int E = wm - kWOff;
                    const bool good = wm > 0 && wm < kWBad;
                    R x[8];
                    int de[8];
#pragma unroll
                    for (int k = 0; k < 4; ++k) {
                        const int4 q4 = sl[k];                      // (row, exponent) of two slots
                        x[2 * k] = good && q4.x >= 0 ? ((const R*)a.W)[((size_t)(q4.x / CW) * a.ncol + col) * CW + q4.x % CW] : R(0);
                        x[2 * k + 1] = good && q4.z >= 0 ? ((const R*)a.W)[((size_t)(q4.z / CW) * a.ncol + col) * CW + q4.z % CW] : R(0);
                        de[2 * k] = q4.y - Digits<R>::kBias;
                        de[2 * k + 1] = q4.w - Digits<R>::kBias;
                    }
#pragma unroll
                    for (int k = 0; k < 8; ++k)      // denormal coefficients are zero: they have no part in the maximum
                        v[it][k] = Digits<R>::exponent(x[k]) > 0 ? Digits<R>::bytes(x[k], E, de[k]) : Digits<R>::kZero;
                }
                const bool ok = i < C::NB || mbar_wait(&wempty_bar[s], ((i / C::NB) - 1) & 1, &abort_flag);
                if (__any_sync(0xffffffffu, !ok)) { stop = true; break; }
                unsigned char* st = wring + (size_t)s * C::BB;
#pragma unroll
                for (int it = 0; it < NT / 16; ++it) {
                    const int task = it * 32 + lane, o = task % NT, kc = task / NT;
#pragma unroll
                    for (int d = 0; d < S; ++d) {
                        __half2 h4[4];
#pragma unroll
                        for (int k = 0; k < 4; ++k) h4[k] = digit_pair<R>(v[it][2 * k], v[it][2 * k + 1], d);
                        *reinterpret_cast<uint4*>(st + ((size_t)kc * (S * NT) + d * NT + o) * 16) = *reinterpret_cast<uint4*>(h4);
                    }
                }
                fence_proxy_async();
                mbar_arrive(&w_bar[s]);
            }
        }
    } else {
        // Y update: two sets of 8 warps on alternate units, so that one's loads of Y are in flight
        // while the other adds and stores; warps 0-3 of a set the first 128 reals of a unit, 4-7
        // the second; TMEM lane = real.  The unit's Y values and column exponents are loaded before
        // its product is awaited.
        const int set = (warp - 2 - C::BW) >> 3, t = ((warp - 2 - C::BW) >> 2) & 1, quad = warp & 3;
        constexpr int F = S == 7 ? 4 : 8;          // columns at a time: the registers allow no more
        const uint32_t lane_base = (uint32_t)(32 * quad) << 16;
        const double alpha = a.alpha_dev ? a.alpha_dev[0] : a.alpha;
        int uu = 0, used = 0;                      // units so far; read-outs so far of this set's buffer (WIDE)
        bool stop = false;
        for (int q = 0; q < np && !stop; ++q) {
            const int* wmax = a.wmax + (size_t)(pair_of(q) / C::PASSES) * a.ncol;
            const int pr = pair_of(q), brick = a.brick[pr / C::PASSES].x, nk = WIDE ? a.brick[pr / C::PASSES].y / 16 : 0;
            const int k = (pr % C::PASSES) * 256 + t * 128 + 32 * quad + lane;
            const int p = k / CW, comp = k % CW;
            const int x = 8 * (brick % a.nbx) + (p & 7), y = 8 * ((brick / a.nbx) % a.nby) + ((p >> 3) & 7);
            const int z = 4 * (brick / (a.nbx * a.nby)) + (p >> 6);
            const bool in = x < a.n1 && y < a.n2 && z < a.n3;
            const long g = in ? x + (long)a.n1 * (y + (long)a.n2 * z) : 0;
            for (int ct = 0; ct < a.ctiles; ++ct, ++uu) {
                if ((uu & 1) != set) continue;
                const int buf = set, c0 = ct * NT, nc = in ? min(NT, a.ncol - c0) : 0;
                R* Y = (R*)a.Y + g * CW + comp + (size_t)c0 * a.ld;
                R yv[NT];
#pragma unroll
                for (int o = 0; o < NT; ++o) yv[o] = o < nc ? Y[(size_t)o * a.ld] : R(0);
                // lane o < NT: column c0 + o.  Zero coefficients have zero digits whatever the exponent.
                const int wm = lane < NT && c0 + lane < a.ncol ? wmax[c0 + lane] : 0;
                const int E = wm == 0 ? Digits<R>::kBias : wm - kWOff;
                const unsigned odd = __ballot_sync(0xffffffffu, wm >= kWBad || E < Digits<R>::kEmin || E > Digits<R>::kEmax);
                auto read_out = [&]() {
                    const bool ok = mbar_wait(&tfull_bar[buf], (WIDE ? used : uu >> 1) & 1, &abort_flag);
                    if (__any_sync(0xffffffffu, !ok)) { stop = true; return; }
                    tc_fence_after();
#pragma unroll
                    for (int o0 = 0; o0 < NT; o0 += F) {
                        uint32_t v[S * F];
                        tmem_levels<S, NT, F>(tmem + lane_base + (uint32_t)(buf * 2 * C::ACC + t * C::ACC + o0), v);
#pragma unroll
                        for (int f = 0; f < F; ++f) {
                            const int Ef = __shfl_sync(0xffffffffu, E, o0 + f);
                            long long lo;
                            const long long hi = level_sum<R, F>(v + f, &lo);
                            if constexpr (S == 7) {
                                // (hi 2^24 + lo) 256^6 with the low 10 bits rounded off; zero or at least 2^-948
                                const double r = (double)((hi << 14) + ((lo + 512) >> 10));
                                const int up = (10 + 48 + Ef + Digits<R>::kBias - 2 * Digits<R>::kUnit) << 20;
                                yv[o0 + f] = fma(alpha, r == 0.0 ? r : __hiloint2double(__double2hiint(r) + up, __double2loint(r)),
                                                 yv[o0 + f]);
                            } else {
                                // hi 2^(24 + Ef + bias - 2 unit) in two factors within the range of float
                                const float sc = __int_as_float((24 + Ef + Digits<R>::kBias - 2 * Digits<R>::kUnit + 40 + 127) << 23);
                                yv[o0 + f] = fmaf((float)alpha * sc, (float)hi * 9.094947017729282e-13f, yv[o0 + f]);   // 2^-40
                            }
                        }
                    }
                    tc_fence_before();
                    mbar_arrive(&tempty_bar[buf]);
                    ++used;
                };
                read_out();
                if constexpr (WIDE)
                    for (int c = C::PCH; c < nk && !stop; c += C::PCH) read_out();
                if (stop) break;
#pragma unroll
                for (int o = 0; o < NT; ++o)
                    if (o < nc && !((odd >> o) & 1u)) Y[(size_t)o * a.ld] = yv[o];
                for (unsigned b = odd; b; b &= b - 1) {
                    const int o = __ffs((int)b) - 1;
                    if (o >= nc || a.csr_off[g] == a.csr_off[g + 1]) continue;
                    const double sum = oz_plain<R, CW>(a, g, comp, c0 + o);
                    const R y0 = Y[(size_t)o * a.ld];
                    if constexpr (S == 7) Y[(size_t)o * a.ld] = fma(alpha, sum, y0);
                    else Y[(size_t)o * a.ld] = fmaf((float)alpha, (float)sum, y0);
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

// ---------------------------------------------------------------------------- tables
// biased exponent of the largest value of each function (re and im): one CTA per site
template <typename R, int CW>
__global__ void k_oz_exponents(const SiteDev* __restrict__ sites, const R* __restrict__ vals, int* __restrict__ exps) {
    const SiteDev S = sites[blockIdx.x];
    __shared__ int m[kMaxProj];
    if (threadIdx.x < kMaxProj) m[threadIdx.x] = 0;
    __syncthreads();
    const R* v = vals + (size_t)S.val_off * CW;
    for (int p = 0; p < S.nproj; ++p) {
        int e = 0;
        for (int i = threadIdx.x; i < S.npts; i += blockDim.x)
            for (int c = 0; c < CW; ++c) e = max(e, Digits<R>::exponent(v[((size_t)i * S.nproj + p) * CW + c]));
        e = __reduce_max_sync(0xffffffffu, e);
        if ((threadIdx.x & 31) == 0) atomicMax(&m[p], e);
    }
    __syncthreads();
    // functions of all-zero (or denormal) values keep the smallest exponent of the format
    if (threadIdx.x < S.nproj) exps[S.proj_off + threadIdx.x] = max(m[threadIdx.x], Digits<R>::kEmin);
}

// digits of every table value into both layouts (cleared before): entry pair[row] of a table row
// is (group, slot in group, brick index, slot in brick) of its site's first function there
template <typename R, int CW>
__global__ void k_oz_fill(const int* __restrict__ items, const SiteDev* __restrict__ sites, const int* __restrict__ idx,
                          const R* __restrict__ vals, const int* __restrict__ exps, const int* __restrict__ row_pair,
                          const int4* __restrict__ pairs, const int4* __restrict__ grp, const int4* __restrict__ brk,
                          int n1, int n2, unsigned short* __restrict__ gval, unsigned short* __restrict__ sval) {
    constexpr int S = Digits<R>::S;
    const int s = items[3 * blockIdx.x], first = items[3 * blockIdx.x + 1], cnt = items[3 * blockIdx.x + 2];
    const SiteDev St = sites[s];
    for (int l = threadIdx.x; l < cnt * St.nproj; l += blockDim.x) {
        const int row = first + l / St.nproj, p = l % St.nproj;
        const int g = idx[row];
        const int x = g % n1, y = (g / n1) % n2, z = g / (n1 * n2);
        const int pin = (x % BRX) + BRX * ((y % BRY) + BRY * (z % BRZ));
        const int4 pr = pairs[row_pair[row]];
        const int4 G = grp[pr.x], B = brk[pr.z];
        const R* v = vals + ((size_t)St.val_off + (size_t)(row - St.pt_off) * St.nproj + p) * CW;
        const int E = exps[St.proj_off + p];
        for (int comp = 0; comp < CW; ++comp)            // row of the matrix: re, im
            for (int c = 0; c < CW; ++c) {               // slot a, b
                const R val = CW == 1 ? v[0] : (comp == c ? v[0] : (comp == 1 ? v[CW - 1] : -v[CW - 1]));
                const typename Digits<R>::I b = Digits<R>::bytes(val, E);
                const int k = pin * CW + comp;
                const int gs = pr.y + p * CW + c, bs = pr.w + p * CW + c;
                for (int d = 0; d < S; ++d) {
                    const int digit = (int)((b >> (8 * (S - 1 - d))) & 0xff) - 128;
                    const unsigned short hv = __half_as_ushort(__int2half_rn(digit));
                    gval[((size_t)G.z + (size_t)(k >> 3) * (S * G.y) + d * G.y + gs) * 8 + (k & 7)] = hv;
                    sval[((size_t)B.z + ((size_t)(k >> 8) * (B.y / 16) + (bs >> 4)) * (2 * S * 2 * OZ_M) +
                          (size_t)(((k >> 7) & 1) * S + d) * (2 * OZ_M) + ((bs >> 3) & 1) * OZ_M + (k & 127)) * 8 + (bs & 7)] = hv;
                }
            }
    }
}

__global__ void k_oz_slots(int n, int cw, const int* __restrict__ exps, int2* __restrict__ slots, const int* __restrict__ fn) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) slots[i].y = fn[i] >= 0 ? exps[fn[i]] : 0;
}

// a device copy of v, counted in bytes: false without room
template <typename Tp>
bool put(hub_t h, Tp** d, const std::vector<Tp>& v, size_t* bytes) {
    const size_t n = std::max<size_t>(v.size(), 1) * sizeof(Tp);
    if (!device_alloc(h, (void**)d, n)) return false;
    *bytes += n;
    return v.empty() || cudaMemcpy(*d, v.data(), v.size() * sizeof(Tp), cudaMemcpyHostToDevice) == cudaSuccess;
}

template <typename R, int CW>
int build_oz(hub_t h, Table& t, const std::vector<std::vector<int>>& site_pts) {
    using GC = GCfg<R, CW>;
    using SC = SCfg<R, CW>;
    constexpr int S = GC::S;
    const int n1 = h->n1, n2 = h->n2;
    t.nbx = (h->n1 + BRX - 1) / BRX;
    t.nby = (h->n2 + BRY - 1) / BRY;
    t.nbz = (h->n3 + BRZ - 1) / BRZ;
    const long nb = (long)t.nbx * t.nby * t.nbz;
    // (site, brick) pairs in site order, the pair of every table row, the pairs of every brick
    struct Pair { int site, brick; };
    std::vector<Pair> pl;
    std::vector<int> row_pair(t.npts), stamp(nb, -1), count(nb + 1, 0);
    for (int s = 0; s < t.nsites; ++s) {
        const int first = (int)pl.size();
        int r = t.h_sites[s].pt_off, pair = 0;
        long end = -1;                               // of the run of points in this row and brick
        for (int g : site_pts[s]) {
            if (g >= end) {
                const int q = g / n1, x = g - q * n1;
                const long b = x / BRX + t.nbx * ((q % n2) / BRY + (long)t.nby * (q / n2 / BRZ));
                if (stamp[b] < first) { stamp[b] = (int)pl.size(); pl.push_back({s, (int)b}); count[b + 1]++; }
                pair = stamp[b];
                end = (long)q * n1 + std::min(n1, (x / BRX + 1) * BRX);
            }
            row_pair[r++] = pair;
        }
    }
    for (long b = 0; b < nb; ++b) count[b + 1] += count[b];
    std::vector<int> by_brick(pl.size()), fill(count.begin(), count.end() - 1);
    for (int i = 0; i < (int)pl.size(); ++i) by_brick[fill[pl[i].brick]++] = i;
    std::vector<int4> pairs(pl.size()), grp, brk;
    std::vector<int2> gslot, bslot;
    std::vector<int> gfn, bfn, roff(t.nproj + 1, 0);
    size_t goff = 0, boff = 0;
    // Groups of all functions of a brick, so that X is converted once, where the bricks make many
    // rounds over the SMs (88 x 88 x 84 x 348: 1.30 -> 1.09 ms; complex float 88 x 88 x 56 x 230: 0.87 -> 0.63);
    // of half as many (two units in flight) below 8 rounds, which fill the SMs better (complex float
    // 88 x 88 x 28 x 115, 5.6 rounds: 0.176 against 0.184 ms with slices of 16; FP64 44 x 44 x 56, 3.3: 0.060 against 0.075).
    int used = 0;
    for (long b = 0; b < nb; ++b) used += count[b] != count[b + 1];
    const int cap = used < 8 * h->num_sms ? GC::NP / 2 : GC::NP;
    for (int i = 0; i < (int)pl.size(); ++i)
        for (int p = 0; p < t.h_sites[pl[i].site].nproj; ++p) roff[t.h_sites[pl[i].site].proj_off + p + 1]++;
    for (int r = 0; r < t.nproj; ++r) roff[r + 1] += roff[r];
    std::vector<int> rent(roff.back()), rfill(roff.begin(), roff.end() - 1);
    long prow = 0;
    for (long b = 0; b < nb; ++b) {
        if (count[b] == count[b + 1]) continue;
        const int bfirst = (int)bslot.size();
        int e = count[b], bs = 0;
        while (e < count[b + 1]) {
            const int gfirst = (int)gslot.size();
            int gs = 0;
            for (; e < count[b + 1]; ++e) {
                const int i = by_brick[e];
                const SiteDev& St = t.h_sites[pl[i].site];
                if (gs + St.nproj * CW > cap) break;
                pairs[i] = make_int4((int)grp.size(), gs, (int)brk.size(), bs);
                for (int p = 0; p < St.nproj; ++p, ++prow) {
                    rent[rfill[St.proj_off + p]++] = (int)prow;
                    for (int c = 0; c < CW; ++c) {
                        gslot.push_back(make_int2((int)prow * CW + c, 0));
                        gfn.push_back(St.proj_off + p);
                        bslot.push_back(make_int2((St.proj_off + p) * CW + c, 0));
                        bfn.push_back(St.proj_off + p);
                    }
                }
                gs += St.nproj * CW;
                bs += St.nproj * CW;
            }
            const int np = (gs + 15) / 16 * 16;
            for (int q = gs; q < np; ++q) { gslot.push_back(make_int2(-1, 0)); gfn.push_back(-1); }
            grp.push_back(make_int4((int)b, np, (int)goff, gfirst));
            goff += (size_t)(BRP * CW / 8) * S * np;
        }
        const int K = (bs + 15) / 16 * 16;
        for (int q = bs; q < K; ++q) { bslot.push_back(make_int2(-1, 0)); bfn.push_back(-1); }
        brk.push_back(make_int4((int)b, K, (int)boff, bfirst));
        boff += (size_t)SC::PASSES * (K / 16) * SC::AU;
        t.oz_wide |= K > 256;
        if (K > OZ_MAXK || goff >= (1ull << 31) || boff >= (1ull << 31) || prow * CW >= (1L << 31)) return HUB_OK;
    }
    std::vector<int> sfirst(t.nsites + 1, 0), sbrick(pl.size());
    for (size_t i = 0; i < pl.size(); ++i) {
        sfirst[pl[i].site + 1]++;
        sbrick[i] = pairs[i].z;
    }
    for (int i = 0; i < t.nsites; ++i) sfirst[i + 1] += sfirst[i];
    // on a device without room for both layouts the point-major form does all products
    size_t tmp = 0;
    int *d_row_pair = nullptr, *d_gfn = nullptr, *d_bfn = nullptr;
    int4* d_pairs = nullptr;
    auto room = [&](void** p, size_t n) {
        if (!device_alloc(h, p, n)) return false;
        t.oz_bytes += n;
        return true;
    };
    const bool ok = room((void**)&t.d_ozg_val, goff * 16) && room((void**)&t.d_ozb_val, boff * 16) &&
                    room((void**)&t.d_oz_exp, std::max(t.nproj, 1) * sizeof(int)) && put(h, &t.d_ozg, grp, &t.oz_bytes) &&
                    put(h, &t.d_ozg_row, gslot, &t.oz_bytes) && put(h, &t.d_ozb, brk, &t.oz_bytes) &&
                    put(h, &t.d_ozb_row, bslot, &t.oz_bytes) && put(h, &t.d_oz_roff, roff, &t.oz_bytes) &&
                    put(h, &t.d_oz_rent, rent, &t.oz_bytes) && put(h, &t.d_oz_sfirst, sfirst, &t.oz_bytes) &&
                    put(h, &t.d_oz_sbrick, sbrick, &t.oz_bytes) && put(h, &d_row_pair, row_pair, &tmp) &&
                    put(h, &d_pairs, pairs, &tmp) && put(h, &d_gfn, gfn, &tmp) && put(h, &d_bfn, bfn, &tmp);
    cudaError_t e = cudaGetLastError(), es = cudaSuccess;
    if (ok) {
        cudaMemsetAsync(t.d_ozg_val, 0, goff * 16, h->stream);
        cudaMemsetAsync(t.d_ozb_val, 0, boff * 16, h->stream);
        ProfScope ps(h, HUB_K_TABLE);
        const R* vals = (const R*)t.d_vals;
        k_oz_exponents<R, CW><<<t.nsites, 256, 0, h->stream>>>(t.d_sites, vals, t.d_oz_exp);
        k_oz_slots<<<((int)gslot.size() + 255) / 256, 256, 0, h->stream>>>((int)gslot.size(), CW, t.d_oz_exp, t.d_ozg_row, d_gfn);
        k_oz_slots<<<((int)bslot.size() + 255) / 256, 256, 0, h->stream>>>((int)bslot.size(), CW, t.d_oz_exp, t.d_ozb_row, d_bfn);
        k_oz_fill<R, CW><<<t.nitems, 256, 0, h->stream>>>(t.d_items, t.d_sites, t.d_idx, vals, t.d_oz_exp, d_row_pair, d_pairs,
                                                          t.d_ozg, t.d_ozb, n1, n2, (unsigned short*)t.d_ozg_val,
                                                          (unsigned short*)t.d_ozb_val);
        e = cudaGetLastError();
        es = cudaStreamSynchronize(h->stream);
    }
    for (void* p : {(void*)d_row_pair, (void*)d_pairs, (void*)d_gfn, (void*)d_bfn})
        if (p) cudaFree(p);
    h->mem_held -= tmp;
    if (!ok) free_oz(h, t);
    HUB_CUDA_TRY(h, e);
    HUB_CUDA_TRY(h, es);
    if (!ok) return HUB_OK;
    t.oz_ngroups = (int)grp.size();
    t.oz_nbricks = (int)brk.size();
    t.oz_npart = prow;
    t.oz = 1;
    return HUB_OK;
}

template <typename R, int CW>
int gather_oz(hub_t h, const void* X, int ncol, int ld, int spin, bool want_W) {
    using C = GCfg<R, CW>;
    Table& t = h->proj;
    int rc;
    if ((rc = launch_colmax(h, X, ncol, ld))) return rc;
    OzGather a{};
    a.X = X;
    a.grp = t.d_ozg;
    a.slot = t.d_ozg_row;
    a.val = t.d_ozg_val;
    a.part = (double*)h->d_part;
    a.bmax = block_map(h, h->d_cmax, ncol);
    a.wmax = h->d_wmax;
    a.nw = want_W ? (long)t.oz_nbricks * ncol : 0;
    a.ld = (long)ld * CW;
    a.n1 = h->n1; a.n2 = h->n2; a.n3 = h->n3;
    a.ncol = ncol;
    a.nbx = t.nbx; a.nby = t.nby;
    a.ctiles = (ncol + OZ_M - 1) / OZ_M;
    a.nunits = t.oz_ngroups * C::PARTS * a.ctiles;
    a.part_rows = t.oz_npart * CW;
    // 16-byte copies need whole pieces within a row and 16-byte row starts
    a.vec = h->n1 % C::PPP == 0 && ((size_t)a.ld * sizeof(R)) % 16 == 0 && (uintptr_t)X % 16 == 0;
    a.flags = h->d_flags;
    HUB_CUDA_TRY(h, cudaFuncSetAttribute(k_gather_oz<R, CW>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)C::SMEM));
    {
        ProfScope ps(h, HUB_K_GATHER);
        k_gather_oz<R, CW><<<std::max(1, std::min(a.nunits, h->num_sms)), OZ_GTHREADS, C::SMEM, h->stream>>>(a);
    }
    HUB_CUDA_TRY(h, cudaGetLastError());
    OzReduce r{};
    r.sites = t.d_sites;
    r.roff = t.d_oz_roff;
    r.rent = t.d_oz_rent;
    r.part = a.part;
    r.gamma = t.d_gamma;
    r.M = t.d_M[spin];
    r.exps = t.d_oz_exp;
    r.C = (double*)h->d_C;
    r.W = h->d_W;
    r.wmax = h->d_wmax;
    r.sfirst = t.d_oz_sfirst;
    r.sbrick = t.d_oz_sbrick;
    r.cmax = h->d_cmax;
    r.X = X;
    r.idx = t.d_idx;
    r.vals = t.d_vals;
    r.part_rows = t.oz_npart * CW;
    r.ld = ld;
    r.dV = h->dV;
    r.ncol = ncol;
    r.want_W = want_W;
    ProfScope ps(h, HUB_K_TRANSFORM);
    k_reduce_oz<R, CW><<<dim3((unsigned)t.nsites, (unsigned)((ncol + 31) / 32)), 256, 0, h->stream>>>(r);
    HUB_CUDA_TRY(h, cudaGetLastError());
    return HUB_OK;
}

template <typename R, int CW>
int scatter_oz(hub_t h, void* Y, int ncol, int ld, double alpha, const double* alpha_dev, bool wmax_ready) {
    using C = SCfg<R, CW>;
    Table& t = h->proj;
    int rc;
    if (!wmax_ready) {
        ProfScope ps(h, HUB_K_SCATTER);
        HUB_CUDA_TRY(h, cudaMemsetAsync(h->d_wmax, 0, (size_t)t.oz_nbricks * ncol * sizeof(int), h->stream));
        k_wmax_oz<R, CW><<<dim3((unsigned)t.nsites, (unsigned)((ncol + 31) / 32)), 256, 0, h->stream>>>(
            t.d_sites, (const R*)h->d_W, t.d_oz_exp, t.d_oz_sfirst, t.d_oz_sbrick, ncol, h->d_wmax);
        HUB_CUDA_TRY(h, cudaGetLastError());
    }
    OzScatter a{};
    a.Y = Y;
    a.brick = t.d_ozb;
    a.slot = t.d_ozb_row;
    a.val = t.d_ozb_val;
    a.W = h->d_W;
    a.wmax = h->d_wmax;
    a.csr_off = t.d_csr_off;
    a.csr_ent = t.d_csr_ent;
    a.vals = t.d_vals;
    a.alpha = alpha;
    a.alpha_dev = alpha_dev;
    a.ld = (long)ld * CW;
    a.ncol = ncol;
    a.n1 = h->n1; a.n2 = h->n2; a.n3 = h->n3;
    a.nbx = t.nbx; a.nby = t.nby;
    a.nbricks = t.oz_nbricks;
    a.ctiles = (ncol + C::NT - 1) / C::NT;
    a.flags = h->d_flags;
    const int npair = t.oz_nbricks * C::PASSES;
    auto run = [&](auto kernel) -> int {
        HUB_CUDA_TRY(h, cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)C::SMEM));
        ProfScope ps(h, HUB_K_SCATTER);
        kernel<<<std::max(1, std::min(npair, h->num_sms)), C::THREADS, C::SMEM, h->stream>>>(a);
        return HUB_OK;
    };
    if constexpr (C::S == 7) {
        if ((rc = t.oz_wide ? run(k_scatter_oz<R, CW, true>) : run(k_scatter_oz<R, CW, false>))) return rc;
    } else {
        if ((rc = run(k_scatter_oz<R, CW, false>))) return rc;
    }
    HUB_CUDA_TRY(h, cudaGetLastError());
    return HUB_OK;
}

}  // namespace

void free_oz(hub_t h, Table& t) {
    for (void* p : {(void*)t.d_ozg, (void*)t.d_ozg_row, (void*)t.d_ozg_val, (void*)t.d_ozb, (void*)t.d_ozb_row, (void*)t.d_ozb_val,
                    (void*)t.d_oz_exp, (void*)t.d_oz_roff, (void*)t.d_oz_rent, (void*)t.d_oz_sfirst, (void*)t.d_oz_sbrick})
        if (p) cudaFree(p);
    t.d_ozg = t.d_ozb = nullptr;
    t.d_ozg_row = t.d_ozb_row = nullptr;
    t.d_ozg_val = t.d_ozb_val = nullptr;
    t.d_oz_exp = t.d_oz_roff = t.d_oz_rent = t.d_oz_sfirst = t.d_oz_sbrick = nullptr;
    h->mem_held -= t.oz_bytes;
    t.oz_bytes = 0;
    if (t.oz) h->mem_gen++;
    t.oz = 0;
}

int build_oz_tables(hub_t h, Table& t, const std::vector<std::vector<int>>& site_pts) {
    if (t.nsites == 0) return HUB_OK;
    if (h->esize == 8) return h->cplx ? build_oz<double, 2>(h, t, site_pts) : build_oz<double, 1>(h, t, site_pts);
    return h->cplx ? build_oz<float, 2>(h, t, site_pts) : build_oz<float, 1>(h, t, site_pts);
}

// Where the digit forms are the faster ones (microseconds, measured on 88 x 88 x 56 and 30 x 30 x 40
// cells with 1 to 160 columns).  Their cost goes by rounds of units over the SMs, whole tiles of
// 128 (gather) or 16 / 32 (scatter) columns; the point-major forms' by function values times
// columns.  FP64, 88 x 88 x 56, 128 columns: gather 2.26 -> 0.32 ms, scatter 2.28 -> 0.39 ms;
// 1 column: 0.056 against 0.21 ms (point-major stays), 0.16 -> 0.06 ms.  Complex float, 128
// columns: 0.63 -> 0.51 ms and 0.78 -> 0.50 ms; 24 columns: 0.14 against 0.29 ms, 0.19 -> 0.16 ms.
bool gather_digits(hub_t h, int ncol) {
    const Table& t = h->proj;
    if (!t.oz) return false;
    const bool d = h->esize == 8;
    const int cw = h->cplx ? 2 : 1;
    // point-major: products, and the wider reduction of its partial sums
    const double c = d ? (h->cplx ? 7.1e-6 : 1.96e-6) : (h->cplx ? 5.5e-7 : 1.7e-7);
    const double plain = t.nvals * (c * ncol + (h->cplx ? 8e-6 : 4e-6)) + 10.0;
    // digits: full tiles and the last one
    const int parts = d ? cw : 1;
    const double rounds = (double)((t.oz_ngroups * parts + h->num_sms - 1) / h->num_sms) * 16 * cw / parts;
    const int last = ncol - ncol / OZ_M * OZ_M;
    const double full = d ? 1.04 : 0.88, part = d ? 0.60 + 0.44 * last / OZ_M : 0.42 + 0.46 * last / OZ_M;
    const double digits = rounds * (ncol / OZ_M * full + (last ? part : 0.0));
    if (digits >= plain || (long)t.oz_ngroups * parts * (ncol / OZ_M + 1) > 0x7fffffffL / 64) return false;
    // the gather's workspace (the point-major form takes over without it)
    return claim(h, (void**)&h->d_cmax, &h->cmax_bytes, colmax_bytes(h, ncol)) &&
           claim(h, (void**)&h->d_wmax, &h->wmax_bytes, (size_t)t.oz_nbricks * ncol * sizeof(int)) &&
           claim(h, &h->d_part, &h->part_bytes, (size_t)t.oz_npart * cw * parts * ncol * sizeof(double));
}

bool scatter_digits(hub_t h, int ncol, bool wmax_ready) {
    const Table& t = h->proj;
    if (!t.oz) return false;
    const bool d = h->esize == 8;
    const int cw = h->cplx ? 2 : 1, nt = d ? 16 : 32;
    const double plain = d ? (h->cplx ? 7.3e-6 : 1.97e-6) * t.nvals * std::max(ncol, 6)
                           : (h->cplx ? 6.8e-7 : 3.7e-7) * t.nvals * std::max(ncol, 12);
    const long pairs = (long)t.oz_nbricks * cw;
    const double digits = (double)((pairs + h->num_sms - 1) / h->num_sms) * ((ncol + nt - 1) / nt) * (d ? 4.2 : 5.5) + 12.0;
    return digits < plain + 10.0 && (wmax_ready || claim(h, (void**)&h->d_wmax, &h->wmax_bytes, (size_t)t.oz_nbricks * ncol * sizeof(int)));
}

int launch_gather_oz(hub_t h, const void* X, int ncol, int ld, int spin, bool want_W) {
    if (h->esize == 8) return h->cplx ? gather_oz<double, 2>(h, X, ncol, ld, spin, want_W) : gather_oz<double, 1>(h, X, ncol, ld, spin, want_W);
    return h->cplx ? gather_oz<float, 2>(h, X, ncol, ld, spin, want_W) : gather_oz<float, 1>(h, X, ncol, ld, spin, want_W);
}

int launch_scatter_oz(hub_t h, void* Y, int ncol, int ld, double alpha, const double* alpha_dev, bool wmax_ready) {
    if (h->esize == 8) return h->cplx ? scatter_oz<double, 2>(h, Y, ncol, ld, alpha, alpha_dev, wmax_ready)
                                      : scatter_oz<double, 1>(h, Y, ncol, ld, alpha, alpha_dev, wmax_ready);
    return h->cplx ? scatter_oz<float, 2>(h, Y, ncol, ld, alpha, alpha_dev, wmax_ready)
                   : scatter_oz<float, 1>(h, Y, ncol, ld, alpha, alpha_dev, wmax_ready);
}

}  // namespace hub

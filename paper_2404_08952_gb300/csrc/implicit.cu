// Semi-implicit DOLINC step for linear advection (Sec 2.4): matrix rows from the
// DOLINC weights, and one persistent cooperative launch per linear solve.
//
// k_imp_assemble  one thread per cell: for each face slot the flux speed a.S and the
//                 weights of the upwind and downwind averages in the face value
//                 (W0[0], W1[0] of the DOLINC representation, the same routine the
//                 stage kernels use), summed into the diagonal or stored against the
//                 neighbour; then every row is scaled by its diagonal.
// k_imp_solve     BiCGSTAB on the scaled rows, all iterations in one launch.  Each
//                 iteration is three grid-stride phases, each ended by a grid barrier
//                 that also reduces the phase's dot products:
//                   A  v = A p (the neighbours' p gathered);           sum rh.v
//                   B  s = r - alpha v, t = A s (the neighbours' s formed from their
//                      r and v);                      sums t.s, t.t, rh.s, rh.t
//                   C  x += alpha p + omega s; r = s - omega t;
//                      p = r + beta (p - omega v), own values only;   sum r.r
//                 omega = t.s / t.t, the next rh.r = rh.s - omega rh.t and beta come
//                 from B's sums, so C can update p without another barrier, and a
//                 neighbour is gathered three times per iteration (p; r, v).
//                 The block that arrives last at a barrier sums the per-block partials
//                 in block order (the result does not depend on arrival order),
//                 computes the next scalars and releases the grid.  A wait polls at
//                 most spin_limit times; one that gives up sets status bit 1 and an
//                 abort word that ends the solve in every block.  The launch is
//                 cooperative, so all blocks are resident and the waits end.
//                 Warm start: x starts from the previous step's solution, or from the
//                 linear extrapolation of the last two (r = b - A x0, one extra
//                 product in the set-up phase); else from 0.
//                 Vectors written inside the launch are read with ld.global.cg (L2),
//                 never through the incoherent L1.  Rows per face slot (the default:
//                 a thread's consecutive slot entries share L1 sectors) or in ELL form
//                 (width 4, 6 or 8, padded with zero weights: coalesced row loads, no
//                 reuse; measured no faster on the hex/prism mesh).
#include <algorithm>

#include "common.cuh"
#include "implicit.cuh"

namespace dol {

// ----------------------------------------------------------------------------- assembly
template <int NS>
__global__ void __launch_bounds__(256) k_imp_assemble(DevMesh m, int k, int r, double ax, double ay, double az,
                                                      double inv_dt, double theta, int ell, int32_t *nbr, double *off,
                                                      double *diag, double *bscale)
{
    const int c = blockIdx.x * blockDim.x + threadIdx.x;
    if (c >= m.n_cells) return;
    const long long n = m.n_cells;
    const double V = 1.0 / m.cellk64[4ll * c + 3];
    double dsum = 0.0;
    const int s0 = m.off[c], s1 = m.off[c + 1];
    // entry of slot s: ELL position (s - s0) n + c, or the slot itself (CSR)
    auto at = [&](int s) { return ell ? (long long)(s - s0) * n + c : (long long)s; };
    for (int s = s0; s < s1; ++s) {
        const int2 sw = m.slot2[s];
        const unsigned word = (unsigned)sw.y;
        const int f = (int)(word >> 2);
        const bool bnd = (word & 2u) != 0;
        const int side = (int)(word & 1u);
        const double *fr = m.face64 + 8ll * f;
        // a.S of the face in its internal owner -> neighbour orientation
        const double an = ax * fr[4] + ay * fr[5] + (m.dim == 3 ? az * fr[6] : 0.0);
        nbr[at(s)] = sw.x;
        if (bnd) {            // zero-gradient face: the flux of the cell's own value
            dsum += theta * an;
            off[at(s)] = 0.0;
            continue;
        }
        // weights of the owner's (cP) and the neighbour's (cN) averages in the upwind value
        double W0[NS + 1], W1[NS + 1], cP, cN;
        if (an >= 0.0) {
            dolinc_weights<NS, double>(k, r, fr[3], W0, W1);
            cP = W0[0];
            cN = W1[0];
        } else {
            dolinc_weights<NS, double>(k, r, rcp_bulk(fr[3]), W0, W1);
            cP = W1[0];
            cN = W0[0];
        }
        // the flux an (cP u_P + cN u_N) leaves the owner and enters the neighbour
        if (side == 0) {
            dsum += theta * an * cP;
            off[at(s)] = theta * an * cN;
        } else {
            dsum -= theta * an * cN;
            off[at(s)] = -theta * an * cP;
        }
    }
    const double D = V * inv_dt + dsum;
    const double iD = 1.0 / D;
    for (int s = s0; s < s1; ++s) off[at(s)] *= iD;
    for (int q = s1 - s0; q < ell; ++q) {      // ELL padding: the cell itself, weight 0
        nbr[(long long)q * n + c] = c;
        off[(long long)q * n + c] = 0.0;
    }
    diag[c] = D;
    bscale[c] = V * iD;
}

void launch_imp_assemble(const DevMesh &m, int ns, int k, int r, double ax, double ay, double az, double dt,
                         double theta, int ell, int32_t *nbr, double *off, double *diag, double *bscale,
                         cudaStream_t s)
{
    const int grid = (m.n_cells + 255) / 256;
    if (grid == 0) return;
    const double idt = 1.0 / dt;
    switch (ns) {
    case 1: k_imp_assemble<1><<<grid, 256, 0, s>>>(m, k, r, ax, ay, az, idt, theta, ell, nbr, off, diag, bscale); break;
    case 2: k_imp_assemble<2><<<grid, 256, 0, s>>>(m, k, r, ax, ay, az, idt, theta, ell, nbr, off, diag, bscale); break;
    case 3: k_imp_assemble<3><<<grid, 256, 0, s>>>(m, k, r, ax, ay, az, idt, theta, ell, nbr, off, diag, bscale); break;
    default: k_imp_assemble<4><<<grid, 256, 0, s>>>(m, k, r, ax, ay, az, idt, theta, ell, nbr, off, diag, bscale); break;
    }
}

// -------------------------------------------------------------------------------- solve
// Sum over the block of N values, in a fixed order; the results are in thread 0.
template <int N>
__device__ __forceinline__ void block_sum(double (&v)[N], double (*sh)[IMP_BLOCK / 32])
{
#pragma unroll
    for (int k = 0; k < N; ++k)
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) v[k] += __shfl_down_sync(0xffffffffu, v[k], o);
    const int w = threadIdx.x >> 5, l = threadIdx.x & 31;
    if (l == 0)
#pragma unroll
        for (int k = 0; k < N; ++k) sh[k][w] = v[k];
    __syncthreads();
    if (w == 0) {
#pragma unroll
        for (int k = 0; k < N; ++k) {
            v[k] = l < IMP_BLOCK / 32 ? sh[k][l] : 0.0;
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) v[k] += __shfl_down_sync(0xffffffffu, v[k], o);
        }
    }
    __syncthreads();
}

__device__ __forceinline__ double ldcg(const double *p) { return __ldcg(p); }
__device__ __forceinline__ void stcg(double *p, double v) { __stcg(p, v); }

// Grid barrier that reduces v[0..N) over all threads of the grid.  The last block to
// arrive sums the per-block partials in block order and calls fin(sums) in its thread
// 0 (fin writes the next scalars) before the others are released.  Returns false when
// the solve was aborted (a wait gave up here or in an earlier barrier).
template <int N> struct Red {
    double v[N];
};

template <int N, class Fin>
__device__ __forceinline__ bool reduce_barrier(const ImpSolve &a, Red<N> r, Fin fin)
{
    static_assert(N <= IMP_NRED, "partials hold IMP_NRED values per block");
    double (&v)[N] = r.v;
    __shared__ double sh[N][IMP_BLOCK / 32];
    __shared__ int last, ok;
    block_sum<N>(v, sh);
    volatile unsigned *gen = a.bar + 32, *abort = a.bar + 64;
    unsigned g = 0;
    if (threadIdx.x == 0) {
#pragma unroll
        for (int k = 0; k < N; ++k) a.part[IMP_NRED * blockIdx.x + k] = v[k];
        g = *gen;
        __threadfence();
        last = atomicAdd(a.bar, 1u) == gridDim.x - 1;
    }
    __syncthreads();
    if (last) {
        __threadfence();
        double t[N];
#pragma unroll
        for (int k = 0; k < N; ++k) t[k] = 0.0;
        for (int b = threadIdx.x; b < (int)gridDim.x; b += IMP_BLOCK)
#pragma unroll
            for (int k = 0; k < N; ++k) t[k] += ldcg(a.part + IMP_NRED * b + k);
        block_sum<N>(t, sh);
        if (threadIdx.x == 0) {
            fin(t);
            atomicExch(a.bar, 0u);
            __threadfence();
            atomicAdd(const_cast<unsigned *>(gen), 1u);
        }
    } else if (threadIdx.x == 0) {
        unsigned it = 0;
        while (*gen == g && !*abort) {
            if (++it > a.spin_limit) {
                atomicOr(a.status, 2u);
                atomicExch(const_cast<unsigned *>(abort), 1u);
                break;
            }
            __nanosleep(64);
        }
        __threadfence();
    }
    if (threadIdx.x == 0) ok = !*abort;
    __syncthreads();
    return ok;
}

// a.off . f(neighbour) over the row of cell c, added to acc: ELL rows of W entries
// (entry q of cell c at q n + c: a warp's loads are contiguous and independent), or the
// cell's slot range (W = 0).
template <int W, class F>
__device__ __forceinline__ double row_sum(const ImpSolve &a, int c, double acc, F f)
{
    if constexpr (W > 0) {
        int j[W];
        double o[W];
#pragma unroll
        for (int q = 0; q < W; ++q) {
            j[q] = __ldg(a.nbr + (long long)q * a.n + c);
            o[q] = __ldg(a.off + (long long)q * a.n + c);
        }
#pragma unroll
        for (int q = 0; q < W; ++q) acc = fma(o[q], f(j[q]), acc);
    } else {
        const int s0 = __ldg(a.row + c), s1 = __ldg(a.row + c + 1);
#pragma unroll 2
        for (int s = s0; s < s1; ++s) acc = fma(__ldg(a.off + s), f(__ldg(a.nbr + s)), acc);
    }
    return acc;
}

template <int W>
__global__ void __launch_bounds__(IMP_BLOCK) k_imp_solve(ImpSolve a)
{
    const int n = a.n;
    const int nth = gridDim.x * IMP_BLOCK;
    const int t0 = blockIdx.x * IMP_BLOCK + threadIdx.x;
    double *sc = a.scal;
    double *p = a.p, *v = a.v;
    bool ok;

    // Set-up: b = bscale * rhs; the initial guess x0 = 0, the previous step's solution
    // x1 (warm 1), or 2 x1 - x2 (warm 2: linear extrapolation from the last two steps),
    // formed for the neighbours on the fly and written to x; r = rh = p = b - A x0.
    {
        Red<2> red{{0.0, 0.0}};
        for (int c = t0; c < n; c += nth) {
            double rhs = a.R[c];
            if (a.Rn) rhs = (a.un[c] - a.u[c]) * a.inv_dt + a.theta * rhs + (1.0 - a.theta) * a.Rn[c];
            const double b = a.bscale[c] * rhs;
            double r0 = b, x0 = 0.0;
            if (a.warm) {
                auto guess = [&](int j) { return a.warm == 2 ? fma(2.0, a.x1[j], -a.x2[j]) : a.x1[j]; };
                x0 = guess(c);
                r0 = b - row_sum<W>(a, c, x0, guess);
            }
            a.x[c] = x0;
            a.r[c] = r0;
            a.rh[c] = r0;
            p[c] = r0;
            red.v[0] = fma(b, b, red.v[0]);
            red.v[1] = fma(r0, r0, red.v[1]);
        }
        ok = reduce_barrier(a, red, [&](const double *t) {
            stcg(sc + SC_RHO, t[1]);
            stcg(sc + SC_BB, t[0]);
            stcg(sc + SC_RR, t[1]);
            stcg(sc + SC_BRK, 0.0);
            stcg(sc + SC_SOLVES, ldcg(sc + SC_SOLVES) + 1.0);
            stcg(a.life + 1, ldcg(a.life + 1) + 1.0);
            stcg(sc + SC_DONE, (t[1] <= a.tol2 * t[0]) ? 1.0 : 0.0);
        });
    }

    for (int it = 0; ok && ldcg(sc + SC_DONE) == 0.0; ++it) {
        // A: v = A p (the neighbours' p gathered);  sum rh.v
        {
            Red<1> red{{0.0}};
            for (int c = t0; c < n; c += nth) {
                const double acc = row_sum<W>(a, c, ldcg(p + c), [&](int j) { return ldcg(p + j); });
                v[c] = acc;
                red.v[0] = fma(ldcg(a.rh + c), acc, red.v[0]);
            }
            ok = reduce_barrier(a, red, [&](const double *t) {
                if (t[0] == 0.0 || !isfinite(t[0])) {
                    atomicOr(a.status, 4u);
                    stcg(sc + SC_DONE, 1.0);
                } else {
                    stcg(sc + SC_ALPHA, ldcg(sc + SC_RHO) / t[0]);
                }
            });
            if (!ok || ldcg(sc + SC_DONE) != 0.0) break;
        }
        // B: s = r - alpha v; t = A s, the neighbours' s formed from their r and v;
        //    sums t.s, t.t, rh.s, rh.t: omega = t.s / t.t, the next rh.r = rh.s - omega
        //    rh.t, and beta, all known before the updates of phase C
        {
            const double al = ldcg(sc + SC_ALPHA);
            Red<4> red{{0.0, 0.0, 0.0, 0.0}};
            for (int c = t0; c < n; c += nth) {
                const double scv = fma(-al, ldcg(v + c), ldcg(a.r + c));
                const double acc = row_sum<W>(a, c, scv, [&](int j) { return fma(-al, ldcg(v + j), ldcg(a.r + j)); });
                a.s[c] = scv;
                a.t[c] = acc;
                const double rh = ldcg(a.rh + c);
                red.v[0] = fma(acc, scv, red.v[0]);
                red.v[1] = fma(acc, acc, red.v[1]);
                red.v[2] = fma(rh, scv, red.v[2]);
                red.v[3] = fma(rh, acc, red.v[3]);
            }
            ok = reduce_barrier(a, red, [&](const double *t) {
                stcg(sc + SC_ITERS, ldcg(sc + SC_ITERS) + 1.0);
                stcg(a.life, ldcg(a.life) + 1.0);
                const double om = t[1] > 0.0 ? t[0] / t[1] : 0.0;     // t = 0: s = 0, the next r is 0
                const double rho1 = t[2] - om * t[3];
                stcg(sc + SC_OMEGA, om);
                if (t[1] > 0.0 && (om == 0.0 || rho1 == 0.0 || !isfinite(rho1))) {
                    stcg(sc + SC_BRK, 1.0);      // breakdown: stop after phase C's updates
                    stcg(sc + SC_BETA, 0.0);
                } else {
                    stcg(sc + SC_BETA, om != 0.0 ? (rho1 / ldcg(sc + SC_RHO)) * (ldcg(sc + SC_ALPHA) / om) : 0.0);
                }
                stcg(sc + SC_RHO, rho1);
            });
            if (!ok) break;
        }
        // C: x += alpha p + omega s; r = s - omega t; p = r + beta (p - omega v), all
        //    of the cell's own values;  sum r.r (the true recursive residual)
        {
            const double al = ldcg(sc + SC_ALPHA), om = ldcg(sc + SC_OMEGA), beta = ldcg(sc + SC_BETA);
            Red<1> red{{0.0}};
            for (int c = t0; c < n; c += nth) {
                const double sv = ldcg(a.s + c), pc = ldcg(p + c);
                a.x[c] = fma(om, sv, fma(al, pc, ldcg(a.x + c)));
                const double rv = fma(-om, ldcg(a.t + c), sv);
                a.r[c] = rv;
                p[c] = fma(beta, pc - om * ldcg(v + c), rv);
                red.v[0] = fma(rv, rv, red.v[0]);
            }
            ok = reduce_barrier(a, red, [&](const double *t) {
                stcg(sc + SC_RR, t[0]);
                if (t[0] <= a.tol2 * ldcg(sc + SC_BB)) {
                    stcg(sc + SC_DONE, 1.0);
                } else if (ldcg(sc + SC_BRK) != 0.0 || !isfinite(t[0])) {
                    atomicOr(a.status, 4u);
                    stcg(sc + SC_DONE, 1.0);
                } else if (it + 1 >= a.max_iter) {
                    atomicOr(a.status, 8u);
                    stcg(sc + SC_DONE, 1.0);
                }
            });
        }
    }
    if (!ok) return;
    // u += delta
    for (int c = t0; c < n; c += nth) a.u[c] += ldcg(a.x + c);
}

// ------------------------------------------------------------------ chunks in shared memory
// k_imp_solve_sm: the same BiCGSTAB with one block of 512 threads per SM, each owning one
// contiguous chunk of the (Morton-ordered) cells.  Phases as above; what differs:
//   - The vector a phase gathers (p in A, s in B) lies in shared memory for the block's own
//     cells: of the neighbours of a chunk of 3400 cells 92% are in it.  Only the others'
//     values come from L2 (p; s formed from r and v, which every block publishes).
//   - The other vectors' own values also lie in shared memory, r, v and p (n_sm > 4, 5, 6)
//     as far as it reaches.
//   - A barrier is one exchange of posts (sm_reduce): every block sums the partials itself,
//     in block order, and computes the next scalars: no last block, no scalars through
//     memory.
// Bound: FP64 issue (23 operations per cell and iteration, 21 us of the chip's rate at
// 515k cells) and three exchanges of 3 to 4 us.  k_imp_solve gathers every neighbour from
// L2, 32 bytes for each 8, waits on chains of three loads per cell, and its shuffle trees
// in every warp and three-step barrier take 26 us of any iteration.  us per iteration, that
// kernel / this one: 2.6k cells 25.6 / 14.5, 96k 36.2 / 21.8, 515k 76.8 / 44.5, 768k
// 86.8 / 57.4; with n_sm = 2 (1.5M cells) 134 / 140, hence n_sm >= 4.  640 threads spill:
// 63 us at 515k.
constexpr int SMB = 512;
constexpr int SM_RED = IMP_NRED * SMB * 8;              // a barrier's values, one per thread
constexpr int SM_BYTES = 226 * 1024 - SM_RED;           // the vectors; with the static part below 227 KB

struct SmScal {
    double rho, al, irv, om, beta, bb, rr;      // irv = 1 / rh.v
    int done, brk, iters;
    unsigned status;
};

// 16 bytes {value, tag}, written and read as one
__device__ __forceinline__ void st_tagged(ulonglong2 *p, double v, unsigned long long tag)
{
    asm volatile("{\n\t.reg .b128 t;\n\tmov.b128 t, {%1, %2};\n\tst.relaxed.gpu.global.b128 [%0], t;\n\t}" ::"l"(p),
                 "l"(__double_as_longlong(v)), "l"(tag)
                 : "memory");
}
__device__ __forceinline__ ulonglong2 ld_tagged(const ulonglong2 *p)
{
    ulonglong2 r;
    asm volatile("{\n\t.reg .b128 t;\n\tld.relaxed.gpu.global.b128 t, [%2];\n\tmov.b128 {%0, %1}, t;\n\t}"
                 : "=l"(r.x), "=l"(r.y)
                 : "l"(p)
                 : "memory");
    return r;
}

// Grid barrier and sums: adds v[0..N) over the grid and runs fin(sums) in thread 0 of every
// block (the same values everywhere), which keeps the scalars; false if a wait gave up.
// Every block posts its partial sums, each with the round's tag in one 16-byte word, and
// waits for the posts of all blocks: one fence and one trip through L2, where an arrival
// counter and partials read after it take four.  Tags go on from launch to launch (base, in
// a.life), and two sets of words take turns, so a post is never overwritten unread.
// The chip does two FP64 operations per clock and SM, so a sum costs by the warp
// instructions issued: the block's 512 values go through shared memory and are added by
// two to four full warps per value, while the last warp waits for the fence; the scalars'
// divisions are one thread's.
template <int N, class Fin>
__device__ __forceinline__ bool sm_reduce(const ImpSolve &a, unsigned long long tag, const double (&v)[N], double *buf,
                                          Fin fin)
{
    constexpr int NW = SMB / 32, SEG = N <= 2 ? 4 : 2, PER = SMB / SEG / 32;   // warps that add one value
    static_assert(N * SEG < NW, "the last warp is free for the fence");
    __shared__ double sh[SEG][N], tot[N];
    __shared__ int gave_up;
    const int t = threadIdx.x, w = t >> 5, l = t & 31, nb = gridDim.x;
#pragma unroll
    for (int k = 0; k < N; ++k) buf[k * SMB + t] = v[k];
    if (t == 0) gave_up = 0;
    __syncthreads();
    if (w < SEG * N) {
        const double *q = buf + w * (SMB / SEG) + l;
        double s = 0.0;
#pragma unroll
        for (int k = 0; k < PER; ++k) s += q[32 * k];
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) s += __shfl_down_sync(0xffffffffu, s, o);
        if (l == 0) sh[w % SEG][w / SEG] = s;
    } else if (w == NW - 1 && l < N) {
        __threadfence();                          // the block's published vectors before its post
    }
    __syncthreads();
    ulonglong2 *post = reinterpret_cast<ulonglong2 *>(a.part) + (tag & 1) * IMP_NRED * nb;
    if (w == NW - 1 && l < N) {
        double s = sh[0][l];
#pragma unroll
        for (int k = 1; k < SEG; ++k) s += sh[k][l];
        st_tagged(post + IMP_NRED * blockIdx.x + l, s, tag);
    }
    // word i: value i % N of block i / N
    for (int i = t; i < N * nb; i += SMB) {
        const ulonglong2 *q = post + IMP_NRED * (i / N) + i % N;
        ulonglong2 x = ld_tagged(q);
        for (unsigned it = 0; x.y != tag; x = ld_tagged(q)) {
            if (++it > a.spin_limit) {
                atomicOr(a.status, 2u);
                atomicExch(a.bar + 64, 1u);
                gave_up = 1;
                break;
            }
            if ((it & 63u) == 0 && *(volatile unsigned *)(a.bar + 64)) {
                gave_up = 1;
                break;
            }
        }
        buf[i] = __longlong_as_double((long long)x.x);
    }
    if (t < N * nb) __threadfence();              // the posts before the vectors they announce
    __syncthreads();
    const bool ok = !gave_up;
    if (ok && w < N) {
        double s = 0.0;
#pragma unroll 5
        for (int b = l; b < nb; b += 32) s += buf[b * N + w];
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) s += __shfl_down_sync(0xffffffffu, s, o);
        if (l == 0) tot[w] = s;
    }
    if constexpr (N > 1) __syncthreads();
    if (ok && t == 0) fin(tot);
    __syncthreads();
    return ok;
}

// acc + sum of off . f(neighbour) over slots [s0, s1), six gathers in flight
template <class F> __device__ __forceinline__ double sm_row(const ImpSolve &a, int s0, int s1, double acc, F f)
{
    constexpr int B = 6;
    for (int s = s0; s < s1; s += B) {
        int j[B];
        double o[B], x[B];
#pragma unroll
        for (int q = 0; q < B; ++q)
            if (s + q < s1) {
                j[q] = __ldg(a.nbr + s + q);
                o[q] = __ldg(a.off + s + q);
            }
#pragma unroll
        for (int q = 0; q < B; ++q)
            if (s + q < s1) x[q] = f(j[q]);
#pragma unroll
        for (int q = 0; q < B; ++q)
            if (s + q < s1) acc = fma(o[q], x[q], acc);
    }
    return acc;
}

// ALL: every own vector is in shared memory; else the first n_sm of them.
template <bool ALL> __global__ void __launch_bounds__(SMB) k_imp_solve_sm(ImpSolve a, int chunk, int n_sm)
{
    extern __shared__ __align__(16) double dyn[];
    double *buf = dyn, *W = dyn + SM_RED / 8;
    const int c0 = blockIdx.x * chunk, m = min(chunk, a.n - c0), t0 = threadIdx.x;
    // W, t, rh and x always in shared memory; r, v, p while it lasts
    auto own = [&](int k, double *g) { return ALL || k < n_sm ? W + k * chunk : g + c0; };
    double *t = W + chunk, *rh = W + 2 * chunk, *x = W + 3 * chunk, *r = own(4, a.r), *v = own(5, a.v), *p = own(6, a.p);
    const bool pub_r = ALL || n_sm > 4, pub_v = ALL || n_sm > 5, pub_p = ALL || n_sm > 6;
    auto slots = [&](int c, int &s0, int &s1) {
        if (a.uniform > 0) s0 = c * a.uniform, s1 = s0 + a.uniform;
        else s0 = __ldg(a.row + c), s1 = __ldg(a.row + c + 1);
    };
    // f(i, own term's product + off . g(neighbour)) over the thread's own cells: g(j) the
    // gathered value, the sum in slot order.  The next cell's row (its first RB slots) and
    // the slot range of the one after are requested before the current row is summed.
    constexpr int RB = 6;
    auto rows = [&](auto g, auto f) {
        int j[RB], n0 = 0, n1 = 0, s0 = 0, s1 = 0;
        double o[RB];
        auto fetch = [&](int b, int e) {
#pragma unroll
            for (int q = 0; q < RB; ++q)
                if (b + q < e) {
                    j[q] = __ldg(a.nbr + b + q);
                    o[q] = __ldg(a.off + b + q);
                }
        };
        if (t0 < m) slots(c0 + t0, s0, s1);
        fetch(s0, s1);
        if (t0 + SMB < m) slots(c0 + t0 + SMB, n0, n1);
        for (int i = t0; i < m; i += SMB) {
            const int b = s0, e = s1;
            double x[RB], w[RB], acc = W[i];
#pragma unroll
            for (int q = 0; q < RB; ++q)
                if (b + q < e) {
                    x[q] = g(j[q]);
                    w[q] = o[q];
                }
            s0 = n0;
            s1 = n1;
            if (i + SMB < m) {
                fetch(s0, s1);
                if (i + 2 * SMB < m) slots(c0 + i + 2 * SMB, n0, n1);
            }
#pragma unroll
            for (int q = 0; q < RB; ++q)
                if (b + q < e) acc = fma(w[q], x[q], acc);
            for (int s = b + RB; s < e; ++s) acc = fma(__ldg(a.off + s), g(__ldg(a.nbr + s)), acc);
            f(i, acc);
        }
    };
    __shared__ SmScal sc;
    volatile unsigned long long *base = reinterpret_cast<volatile unsigned long long *>(a.life + 2);
    unsigned long long round = *base;
    if (t0 == 0) {
        sc.bb = sc.rr = 0.0;
        sc.done = sc.iters = 0;
        sc.status = 0;
    }
    bool ok = !grid_aborted(a.bar);

    {
        double red[2] = {0.0, 0.0};
        for (int i = t0; ok && i < m; i += SMB) {
            const int c = c0 + i;
            double rhs = a.R[c];
            if (a.Rn) rhs = (a.un[c] - a.u[c]) * a.inv_dt + a.theta * rhs + (1.0 - a.theta) * a.Rn[c];
            const double b = a.bscale[c] * rhs;
            double r0 = b, x0 = 0.0;
            if (a.warm) {
                auto guess = [&](int j) { return a.warm == 2 ? fma(2.0, a.x1[j], -a.x2[j]) : a.x1[j]; };
                int s0, s1;
                slots(c, s0, s1);
                x0 = guess(c);
                r0 = b - sm_row(a, s0, s1, x0, guess);
            }
            x[i] = x0;
            r[i] = r0;
            rh[i] = r0;
            p[i] = r0;
            W[i] = r0;
            if (pub_r) stcg(a.r + c, r0);
            if (pub_p) stcg(a.p + c, r0);
            red[0] = fma(b, b, red[0]);
            red[1] = fma(r0, r0, red[1]);
        }
        ok = ok && sm_reduce<2>(a, ++round, red, buf, [&](const double *q) {
            sc.bb = q[0];
            sc.rr = sc.rho = q[1];
            sc.done = q[1] <= a.tol2 * q[0];
        });
    }
    for (int it = 0; ok && !sc.done; ++it) {
        // A: v = A p;  sum rh.v
        {
            double red[1] = {0.0};
            auto p_of = [&](int j) {
                const unsigned q = (unsigned)(j - c0);
                return q < (unsigned)m ? W[q] : ldcg(a.p + j);
            };
            rows(p_of, [&](int i, double acc) {
                v[i] = acc;
                if (pub_v) stcg(a.v + c0 + i, acc);
                red[0] = fma(rh[i], acc, red[0]);
            });
            ok = sm_reduce<1>(a, ++round, red, buf, [&](const double *q) {
                if (q[0] == 0.0 || !isfinite(q[0])) {
                    sc.status |= 4u;
                    sc.done = 1;
                } else {
                    sc.al = sc.rho / q[0];
                    sc.irv = 1.0 / q[0];
                }
            });
            if (!ok || sc.done) break;
        }
        // B: s = r - alpha v (own cells first, in W); t = A s;  sums t.s, t.t, rh.s, rh.t
        {
            const double al = sc.al;
#pragma unroll 4
            for (int i = t0; i < m; i += SMB) W[i] = fma(-al, v[i], r[i]);
            __syncthreads();
            double red[4] = {0.0, 0.0, 0.0, 0.0};
            auto s_of = [&](int j) {
                const unsigned q = (unsigned)(j - c0);
                return q < (unsigned)m ? W[q] : fma(-al, ldcg(a.v + j), ldcg(a.r + j));
            };
            rows(s_of, [&](int i, double acc) {
                t[i] = acc;
                const double sv = W[i], h = rh[i];
                red[0] = fma(acc, sv, red[0]);
                red[1] = fma(acc, acc, red[1]);
                red[2] = fma(h, sv, red[2]);
                red[3] = fma(h, acc, red[3]);
            });
            ok = sm_reduce<4>(a, ++round, red, buf, [&](const double *q) {
                ++sc.iters;
                // beta = (rho1 / rho) (alpha / omega) with alpha / rho = 1 / rh.v
                const double om = q[1] > 0.0 ? q[0] / q[1] : 0.0;     // t = 0: s = 0, the next r is 0
                const double iom = q[1] / q[0];
                const double rho1 = q[2] - om * q[3];
                sc.brk = q[1] > 0.0 && (om == 0.0 || rho1 == 0.0 || !isfinite(rho1));
                sc.beta = sc.brk || om == 0.0 ? 0.0 : rho1 * sc.irv * iom;
                sc.om = om;
                sc.rho = rho1;
            });
            if (!ok) break;
        }
        // C: x += alpha p + omega s; r = s - omega t; p = r + beta (p - omega v);  sum r.r
        {
            const double al = sc.al, om = sc.om, beta = sc.beta;
            double red[1] = {0.0};
#pragma unroll 4
            for (int i = t0; i < m; i += SMB) {
                const int c = c0 + i;
                const double sv = W[i], pc = p[i];
                x[i] = fma(om, sv, fma(al, pc, x[i]));
                const double rv = fma(-om, t[i], sv), pn = fma(beta, pc - om * v[i], rv);
                r[i] = rv;
                p[i] = pn;
                W[i] = pn;
                if (pub_r) stcg(a.r + c, rv);
                if (pub_p) stcg(a.p + c, pn);
                red[0] = fma(rv, rv, red[0]);
            }
            ok = sm_reduce<1>(a, ++round, red, buf, [&](const double *q) {
                sc.rr = q[0];
                if (q[0] <= a.tol2 * sc.bb) {
                    sc.done = 1;
                } else if (sc.brk || !isfinite(q[0])) {
                    sc.status |= 4u;
                    sc.done = 1;
                } else if (it + 1 >= a.max_iter) {
                    sc.status |= 8u;
                    sc.done = 1;
                }
            });
        }
    }
    if (ok)
        for (int i = t0; i < m; i += SMB) {
            a.u[c0 + i] += x[i];
            a.x[c0 + i] = x[i];                   // kept for the next step's warm start
        }
    __syncthreads();
    if (t0 == 0) {
        if (blockIdx.x == 0) {
            double *g = a.scal;
            g[SC_BB] = sc.bb;
            g[SC_RR] = sc.rr;
            g[SC_ITERS] += sc.iters;
            g[SC_SOLVES] += 1.0;
            a.life[0] += sc.iters;
            a.life[1] += 1.0;
            if (sc.status) atomicOr(a.status, sc.status);
        }
        __threadfence();
        if (atomicAdd(a.bar + 32, 1u) == gridDim.x - 1) {     // the last block to leave
            a.bar[32] = 0;
            *base = round + 2;                                // above every tag posted
        }
    }
}

template <int W> cudaError_t launch_w(const ImpSolve &a, int grid, cudaStream_t s)
{
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(grid);
    cfg.blockDim = dim3(IMP_BLOCK);
    cfg.stream = s;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeCooperative;
    attr[0].val.cooperative = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, k_imp_solve<W>, a);
}

template <int W> int blocks_w()
{
    int n = 0;
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, k_imp_solve<W>, IMP_BLOCK, 0);
    return n;
}

int imp_ell_width(int max_slots) { return max_slots <= 4 ? 4 : max_slots <= 6 ? 6 : max_slots <= 8 ? 8 : 0; }

// cells of the largest mesh for which four vectors fit the SMs' shared memory
int64_t imp_sm_cells(int sms) { return (int64_t)sms * (SM_BYTES / 8 / 4 - 32); }

cudaError_t imp_sm_setup()
{
    for (auto k : {k_imp_solve_sm<true>, k_imp_solve_sm<false>}) {
        cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, SM_RED + SM_BYTES);
        if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
}

cudaError_t launch_imp_solve_sm(const ImpSolve &a, int sms, cudaStream_t s)
{
    // chunks of at least 256 cells, whole warps of them
    const int chunk = std::max(256, ((a.n + sms - 1) / sms + 31) / 32 * 32);
    const int n_sm = std::min(7, SM_BYTES / 8 / chunk);
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((a.n + chunk - 1) / chunk);
    cfg.blockDim = dim3(SMB);
    cfg.dynamicSmemBytes = SM_RED + (size_t)n_sm * chunk * 8;
    cfg.stream = s;
    cudaLaunchAttribute attrs[1];
    attrs[0].id = cudaLaunchAttributeCooperative;
    attrs[0].val.cooperative = 1;
    cfg.attrs = attrs;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, n_sm == 7 ? k_imp_solve_sm<true> : k_imp_solve_sm<false>, a, chunk, n_sm);
}

cudaError_t launch_imp_solve(const ImpSolve &a, int ell, int grid, cudaStream_t s)
{
    switch (ell) {
    case 4: return launch_w<4>(a, grid, s);
    case 6: return launch_w<6>(a, grid, s);
    case 8: return launch_w<8>(a, grid, s);
    default: return launch_w<0>(a, grid, s);
    }
}

int imp_solve_blocks_per_sm(int ell)
{
    switch (ell) {
    case 4: return blocks_w<4>();
    case 6: return blocks_w<6>();
    case 8: return blocks_w<8>();
    default: return blocks_w<0>();
    }
}

}  // namespace dol

// Troubled-cell indicator kernels: criterion, network inputs, tensor-core inference and
// the FP32 training kernels (see indicator.cuh).
#include <cuda_bf16.h>

#include "indicator.cuh"

namespace dol {

namespace {

// ------------------------------------------------------------------ criterion
// Cell c is troubled if, at one of its interior faces, (i) a reconstructed state of
// either orientation has rho <= 0 or p <= 0, or (ii) with c upwind, the ENO3-DOLINC
// three-cell indicators of rho or rho E (Sec 2.4) satisfy
// |D_C| > kappa min(|D_L|, |D_R|) and |D_C| > eps (|phi_0| + |phi_1|).
template <int DIM, class R>
__device__ __forceinline__ R pressure_of(R gam, const R *U)
{
    R ke = U[1] * U[1] + U[2] * U[2] + (DIM == 3 ? U[3] * U[3] : (R)0);
    return (gam - (R)1) * (U[DIM + 1] - (R)0.5 * ke / U[0]);
}

template <class R>
__device__ __forceinline__ bool rough(R g, const R *p0, const R *p1, R kappa, R eps)
{
    // far values phi_{-1}, phi_{-2}, phi_2 by Eq diffDLC (c is cell i, its neighbour i+1)
    const R gi = (R)1 / g;
    const R m1_0 = gi * (p1[0] - p0[1] - ((R)1 - g) * p0[0]);
    const R m1_1 = gi * (p1[1] - p0[2] - ((R)1 - g) * p0[1]);
    const R m2 = gi * (p0[0] - gi * m1_1 - ((R)1 - g) * m1_0);
    const R p2 = g * p0[0] + g * p1[1] + ((R)1 - g) * p1[0];
    const R DL = g * g * (p0[0] - ((R)1 + g) * m1_0 + g * m2);
    const R DC = p1[0] - ((R)1 + g) * p0[0] + g * m1_0;
    const R DR = (p2 - ((R)1 + g) * p1[0] + g * p0[0]) * gi * gi;
    const R mn = fmin(fabs(DL), fabs(DR));
    return fabs(DC) > kappa * mn && fabs(DC) > eps * (fabs(p0[0]) + fabs(p1[0]));
}

template <int DIM, int NSR, int PREC>
__global__ void __launch_bounds__(128) k_criterion(DevMesh mesh, StageArgs a, float kappa, float eps, uint8_t *flags)
{
    using R = typename PrecT<PREC>::R;
    constexpr int NV = DIM + 2;
    const int c = blockIdx.x * blockDim.x + threadIdx.x;
    if (c >= mesh.n_cells) return;
    bool trouble = false;
    int s0, s1;
    slot_range(mesh, c, s0, s1);
    for (int s = s0; s < s1; ++s) {
        const int2 sw = __ldg(mesh.slot2 + s);
        const unsigned word = (unsigned)sw.y;
        if (word & 2) continue;                       // boundary face
        const int nb = sw.x, f = (int)(word >> 2), side = word & 1;
        R fr[8];
        {
            const R *p = Geo<R>::face(mesh) + 8ll * f;
            ld4<R>(p, fr[0], fr[1], fr[2], fr[3]);
            ld4<R>(p + 4, fr[4], fr[5], fr[6], fr[7]);
        }
        const int P = side ? nb : c, N = side ? c : nb;
        R mono[ncum(DIM, NSR)];
        monomials<DIM, NSR, R>(fr[0], fr[1], fr[2], mono);
        R phP[NV][NSR + 1], phN[NV][NSR + 1];
        contract_cell<DIM, NV, NSR, PREC>(a, P, mono, phP, mesh);
        contract_cell<DIM, NV, NSR, PREC>(a, N, mono, phN, mesh);
        const R g = fr[3];
        // (i) positivity of both reconstructed states of the face
        R W0[NSR + 1], W1[NSR + 1], UL[NV], UR[NV];
        dolinc_weights<NSR, R>(a.k, a.r, g, W0, W1);
#pragma unroll
        for (int v = 0; v < NV; ++v) {
            R t = (R)0;
#pragma unroll
            for (int m = 0; m <= NSR; ++m) t = fma(W0[m], phP[v][m], fma(W1[m], phN[v][m], t));
            UL[v] = t;
        }
        dolinc_weights<NSR, R>(a.k, a.r, (R)1 / g, W0, W1);
#pragma unroll
        for (int v = 0; v < NV; ++v) {
            R t = (R)0;
#pragma unroll
            for (int m = 0; m <= NSR; ++m) {
                R q = fma(W0[m], phN[v][m], W1[m] * phP[v][m]);
                t = (m & 1) ? t - q : t + q;
            }
            UR[v] = t;
        }
        const R gam = par_gamma<R>(a);
        if (!(UL[0] > (R)0) || !(pressure_of<DIM, R>(gam, UL) > (R)0) || !(UR[0] > (R)0) ||
            !(pressure_of<DIM, R>(gam, UR) > (R)0))
            trouble = true;
        // (ii) smoothness with c as the upwind cell
        const R gc = side ? (R)1 / g : g;
#pragma unroll
        for (int vi = 0; vi < 2; ++vi) {
            const int v = vi == 0 ? 0 : NV - 1;
            R q0[3], q1[3];
#pragma unroll
            for (int m = 0; m < 3; ++m) {
                const R sg = (side && (m & 1)) ? (R)-1 : (R)1;
                q0[m] = sg * (side ? phN[v][m] : phP[v][m]);
                q1[m] = sg * (side ? phP[v][m] : phN[v][m]);
            }
            if (rough<R>(gc, q0, q1, (R)kappa, (R)eps)) trouble = true;
        }
    }
    flags[c] = trouble ? 1 : 0;
}

// ------------------------------------------------------------------ network inputs
// Own features of cell c: for m = 1, 2, the largest |phi^(m)_c(d_f)| over its faces of
// rho, rho E and the momentum vector, divided by rho_c, |E_c|, sqrt(rho_c |E_c|), mapped
// by log(1 + x).
template <int DIM, int PREC>
__global__ void __launch_bounds__(128) k_own_features(DevMesh mesh, StageArgs a, float *own)
{
    using R = typename PrecT<PREC>::R;
    constexpr int NV = DIM + 2;
    const int c = blockIdx.x * blockDim.x + threadIdx.x;
    if (c >= mesh.n_cells) return;
    using T1 = typename OrdT<PREC, 1>::T;
    using T2 = typename OrdT<PREC, 2>::T;
    constexpr int C1 = ncoef(DIM, 1), C2 = ncoef(DIM, 2);
    R p1[NV * C1], p2[NV * C2], u0[NV];
    load_rec<typename PrecT<PREC>::T0, NV, ord_stride<DIM, NV, 0, PREC>(), R>(
        static_cast<const typename PrecT<PREC>::T0 *>(a.ord[0]), c, u0);
    load_rec<T1, NV * C1, ord_stride<DIM, NV, 1, PREC>(), R>(static_cast<const T1 *>(a.ord[1]), c, p1);
    load_rec<T2, NV * C2, ord_stride<DIM, NV, 2, PREC>(), R>(static_cast<const T2 *>(a.ord[2]), c, p2);
    R mx[6] = {0, 0, 0, 0, 0, 0};
    int s0, s1;
    slot_range(mesh, c, s0, s1);
    for (int s = s0; s < s1; ++s) {
        const int f = (int)((unsigned)__ldg(mesh.slot2 + s).y >> 2);
        R d0, d1, d2, gg;
        ld4<R>(Geo<R>::face(mesh) + 8ll * f, d0, d1, d2, gg);
        R mono[ncum(DIM, 2)];
        monomials<DIM, 2, R>(d0, d1, d2, mono);
        R ph[NV][2];
#pragma unroll
        for (int v = 0; v < NV; ++v) {
            R t1 = (R)0, t2 = (R)0;
#pragma unroll
            for (int q = 0; q < C1; ++q) t1 = fma(p1[v * C1 + q], mono[1 + q], t1);
#pragma unroll
            for (int q = 0; q < C2; ++q) t2 = fma(p2[v * C2 + q], mono[1 + C1 + q], t2);
            ph[v][0] = (R)2 * t1;
            ph[v][1] = (R)4 * t2;
        }
#pragma unroll
        for (int m = 0; m < 2; ++m) {
            R mo = (R)0;
#pragma unroll
            for (int k = 0; k < DIM; ++k) mo += ph[1 + k][m] * ph[1 + k][m];
            mx[3 * m + 0] = fmax(mx[3 * m + 0], fabs(ph[0][m]));
            mx[3 * m + 1] = fmax(mx[3 * m + 1], fabs(ph[NV - 1][m]));
            mx[3 * m + 2] = fmax(mx[3 * m + 2], sqrt(mo));
        }
    }
    const R tiny = (R)1e-6;
    const R E = fabs(u0[NV - 1]);
    const R sc[3] = {u0[0] + tiny, E + tiny, sqrt(fabs(u0[0]) * E) + tiny};
#pragma unroll
    for (int m = 0; m < 2; ++m)
#pragma unroll
        for (int q = 0; q < 3; ++q) own[6ll * c + 3 * m + q] = (float)log1p(mx[3 * m + q] / sc[q]);
}

__device__ __forceinline__ bool lex_gt(const float *a, const float *b)
{
#pragma unroll
    for (int q = 0; q < 6; ++q) {
        if (a[q] > b[q]) return true;
        if (a[q] < b[q]) return false;
    }
    return false;
}

// the 6 features of cell c (24-byte records)
__device__ __forceinline__ void load6(const float *__restrict__ own, int c, float *f)
{
    const float2 *p = reinterpret_cast<const float2 *>(own + 6ll * c);
#pragma unroll
    for (int q = 0; q < 3; ++q) {
        const float2 v = __ldg(p + q);
        f[2 * q] = v.x, f[2 * q + 1] = v.y;
    }
}

// Network input of cell c: its own 6 features, then the 6 of the three largest face
// neighbours in lexicographic order (itself across a boundary face).
__device__ __forceinline__ void gather24_cell(const DevMesh &mesh, const float *__restrict__ own, int c, float *o)
{
    float top[3][6];
    int have = 0;
    int s0, s1;
    slot_range(mesh, c, s0, s1);
    for (int s = s0; s < s1; ++s) {
        const int nb = __ldg(mesh.slot2 + s).x;
        float f[6];
        load6(own, nb, f);
        // insert into the descending top-3 list (compile-time indices only)
        bool ins0 = have < 1 || lex_gt(f, top[0]);
        bool ins1 = !ins0 && (have < 2 || lex_gt(f, top[1]));
        bool ins2 = !ins0 && !ins1 && (have < 3 || lex_gt(f, top[2]));
#pragma unroll
        for (int q = 0; q < 6; ++q) {
            float t0 = top[0][q], t1 = top[1][q];
            if (ins0) { top[2][q] = t1; top[1][q] = t0; top[0][q] = f[q]; }
            else if (ins1) { top[2][q] = t1; top[1][q] = f[q]; }
            else if (ins2) { top[2][q] = f[q]; }
        }
        if (have < 3) ++have;
    }
    float self[6];
    load6(own, c, self);
#pragma unroll
    for (int a = 0; a < 3; ++a)
        if (a >= have)
#pragma unroll
            for (int q = 0; q < 6; ++q) top[a][q] = self[q];
#pragma unroll
    for (int q = 0; q < 6; ++q) o[q] = self[q];
#pragma unroll
    for (int a = 0; a < 3; ++a)
#pragma unroll
        for (int q = 0; q < 6; ++q) o[6 + 6 * a + q] = top[a][q];
}

__global__ void __launch_bounds__(128) k_gather24(DevMesh mesh, const float *__restrict__ own, float *__restrict__ x)
{
    const int c = blockIdx.x * blockDim.x + threadIdx.x;
    if (c >= mesh.n_cells) return;
    float o[24];
    gather24_cell(mesh, own, c, o);
#pragma unroll
    for (int q = 0; q < 24; ++q) x[24ll * c + q] = o[q];
}

// ------------------------------------------------------------------ tensor-core inference
// B fragments of mma.m16n8k16 (bf16, "col" B = W^T): lane (g = lane/4, t = lane%4) of
// tile (kt, nt) holds W[n][k], W[n][k+1] and W[n][k+8], W[n][k+9] with n = 8 nt + g,
// k = 16 kt + 2 t (zero outside the layer).
__device__ __forceinline__ uint32_t pack_bf16(float lo, float hi)
{
    __nv_bfloat162 h = __floats2bfloat162_rn(lo, hi);
    return *reinterpret_cast<uint32_t *>(&h);
}

__global__ void k_mlp_frags(const float *__restrict__ theta, uint2 *__restrict__ frag)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= N_FRAGS * 32) return;
    const int fidx = i / 32, lane = i % 32, g = lane >> 2, t = lane & 3;
    int layer, kt, nt, in_dim, out_dim, woff;
    if (fidx < FRAG_L2) { layer = 0; kt = fidx / 8; nt = fidx % 8; in_dim = MLP_IN; out_dim = MLP_H; woff = OFF_W1; }
    else if (fidx < FRAG_L3) { layer = 1; kt = (fidx - FRAG_L2) / 8; nt = (fidx - FRAG_L2) % 8; in_dim = MLP_H; out_dim = MLP_H; woff = OFF_W2; }
    else if (fidx < FRAG_L4) { layer = 2; kt = (fidx - FRAG_L3) / 8; nt = (fidx - FRAG_L3) % 8; in_dim = MLP_H; out_dim = MLP_H; woff = OFF_W3; }
    else { layer = 3; kt = fidx - FRAG_L4; nt = 0; in_dim = MLP_H; out_dim = 1; woff = OFF_W4; }
    (void)layer;
    const int n = 8 * nt + g, k = 16 * kt + 2 * t;
    auto w = [&](int kk) { return (n < out_dim && kk < in_dim) ? theta[woff + n * in_dim + kk] : 0.0f; };
    frag[i] = make_uint2(pack_bf16(w(k), w(k + 1)), pack_bf16(w(k + 8), w(k + 9)));
}

__device__ __forceinline__ void mma_bf16(float *d, const uint32_t *a, uint2 b)
{
    asm volatile("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, "
                 "{%0,%1,%2,%3};\n"
                 : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
                 : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b.x), "r"(b.y));
}

// 32 cells per warp tile, two m16 tiles that share every B fragment read from shared
// memory (with 16 cells the fragments' reads, 84 of 256 bytes per tile, were the kernel's
// largest cost).  Activations stay in registers between layers (the f32 accumulator layout
// of two adjacent n-tiles is the bf16 A layout of one k-tile).
// The tile's inputs are staged as bf16 pairs, 12 words per cell (rows of 12 words put the
// 32 words of an A fragment in distinct banks).  FUSED: they are not read from x but
// gathered (gather24_cell, one cell per lane).
// Bound: latency of the gathers and of dependent MMAs (tensor pipe 42% busy, 16 warps per
// SM).  1.05M triangles, fused: 121 us with 16 cells per tile, 95 with 32 at 160 registers,
// 76 at 128 (four blocks per SM).
constexpr int XW = MLP_IN / 2;

template <bool FUSED>
__global__ void __launch_bounds__(128, 4) k_mlp_infer(const uint2 *__restrict__ frag, const float *__restrict__ theta,
                                                   const float *__restrict__ x, long long n,
                                                   float *__restrict__ logits, uint8_t *__restrict__ flags,
                                                   DevMesh mesh, const float *__restrict__ own)
{
    __shared__ uint32_t sx[4][32][XW];
    __shared__ __align__(16) uint2 sfrag[N_FRAGS * 32];
    __shared__ float sbias[3 * MLP_H + 1];
    // all loads of the weights in flight together: a call on 1000 rows 4.6 -> 3.7 us (16 rows per
    // warp took 3.9), on 1M rows 56.8 -> 55.6
    static_assert(N_FRAGS * 32 % 2 == 0, "16-byte pieces");
    constexpr int NW = N_FRAGS * 16;
#pragma unroll
    for (int k = 0; k < (NW + 127) / 128; ++k) {
        const int i = threadIdx.x + 128 * k;
        if (i < NW) reinterpret_cast<uint4 *>(sfrag)[i] = __ldg(reinterpret_cast<const uint4 *>(frag) + i);
    }
    for (int i = threadIdx.x; i < MLP_H; i += blockDim.x) {
        sbias[i] = __bfloat162float(__float2bfloat16_rn(theta[OFF_B1 + i]));
        sbias[MLP_H + i] = __bfloat162float(__float2bfloat16_rn(theta[OFF_B2 + i]));
        sbias[2 * MLP_H + i] = __bfloat162float(__float2bfloat16_rn(theta[OFF_B3 + i]));
    }
    if (threadIdx.x == 0) sbias[3 * MLP_H] = __bfloat162float(__float2bfloat16_rn(theta[OFF_B4]));
    __syncthreads();
    const int lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3;
    const long long warps = (long long)gridDim.x * (blockDim.x / 32);
    const long long w0 = (long long)blockIdx.x * (blockDim.x / 32) + threadIdx.x / 32;
    uint32_t (*wx)[XW] = sx[threadIdx.x / 32];
    for (long long tile = w0; tile * 32 < n; tile += warps) {
        const long long c0 = tile * 32;
        __syncwarp();
        if constexpr (FUSED) {
            if (c0 + lane < n) {
                float o[MLP_IN];
                gather24_cell(mesh, own, (int)(c0 + lane), o);
#pragma unroll
                for (int q = 0; q < XW; ++q) wx[lane][q] = pack_bf16(o[2 * q], o[2 * q + 1]);
            }
        } else {
            // the tile's rows are contiguous: 16-byte pieces where the tile is whole and x
            // is aligned to them, else single values
            const float *xt = x + c0 * MLP_IN;
            if (c0 + 32 <= n && (reinterpret_cast<uintptr_t>(x) & 15) == 0) {
#pragma unroll
                for (int q = 0; q < MLP_IN / 4; ++q) {
                    const int i = lane + 32 * q;
                    const float4 v = __ldg(reinterpret_cast<const float4 *>(xt) + i);
                    (&wx[0][0])[2 * i] = pack_bf16(v.x, v.y);
                    (&wx[0][0])[2 * i + 1] = pack_bf16(v.z, v.w);
                }
            } else {
                for (int i = lane; i < 32 * XW; i += 32)
                    if (c0 + i / XW < n) (&wx[0][0])[i] = pack_bf16(__ldg(xt + 2 * i), __ldg(xt + 2 * i + 1));
            }
        }
        __syncwarp();
        // layer 1 input: 24 features padded to 32 (two k-tiles); rows past n are not stored
        uint32_t A[2][4][4];
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const uint32_t *p0 = wx[16 * h + g], *p1 = wx[16 * h + g + 8];
            A[h][0][0] = p0[t], A[h][0][1] = p1[t], A[h][0][2] = p0[t + 4], A[h][0][3] = p1[t + 4];
            A[h][1][0] = p0[t + 8], A[h][1][1] = p1[t + 8], A[h][1][2] = A[h][1][3] = 0u;
        }
        // three hidden layers
#pragma unroll
        for (int layer = 0; layer < 3; ++layer) {
            const int nk = layer == 0 ? 2 : 4;
            const int fbase = layer == 0 ? FRAG_L1 : (layer == 1 ? FRAG_L2 : FRAG_L3);
            float C[2][8][4];
#pragma unroll
            for (int nt = 0; nt < 8; ++nt) {
                const float b0 = sbias[layer * MLP_H + 8 * nt + 2 * t], b1 = sbias[layer * MLP_H + 8 * nt + 2 * t + 1];
#pragma unroll
                for (int h = 0; h < 2; ++h) C[h][nt][0] = b0, C[h][nt][1] = b1, C[h][nt][2] = b0, C[h][nt][3] = b1;
#pragma unroll
                for (int kt = 0; kt < 4; ++kt)
                    if (kt < nk) {
                        const uint2 B = sfrag[(fbase + kt * 8 + nt) * 32 + lane];
                        mma_bf16(C[0][nt], A[0][kt], B);
                        mma_bf16(C[1][nt], A[1][kt], B);
                    }
            }
#pragma unroll
            for (int h = 0; h < 2; ++h)
#pragma unroll
                for (int kt = 0; kt < 4; ++kt) {
                    A[h][kt][0] = pack_bf16(fmaxf(C[h][2 * kt][0], 0.f), fmaxf(C[h][2 * kt][1], 0.f));
                    A[h][kt][1] = pack_bf16(fmaxf(C[h][2 * kt][2], 0.f), fmaxf(C[h][2 * kt][3], 0.f));
                    A[h][kt][2] = pack_bf16(fmaxf(C[h][2 * kt + 1][0], 0.f), fmaxf(C[h][2 * kt + 1][1], 0.f));
                    A[h][kt][3] = pack_bf16(fmaxf(C[h][2 * kt + 1][2], 0.f), fmaxf(C[h][2 * kt + 1][3], 0.f));
                }
        }
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            float O[4] = {sbias[3 * MLP_H], 0.f, sbias[3 * MLP_H], 0.f};
#pragma unroll
            for (int kt = 0; kt < 4; ++kt) mma_bf16(O, A[h][kt], sfrag[(FRAG_L4 + kt) * 32 + lane]);
            const long long r0 = c0 + 16 * h + g, r1 = r0 + 8;
            if (t == 0) {
                if (r0 < n) {
                    if (logits) logits[r0] = O[0];
                    if (flags) flags[r0] = O[0] > 0.f;
                }
                if (r1 < n) {
                    if (logits) logits[r1] = O[2];
                    if (flags) flags[r1] = O[2] > 0.f;
                }
            }
        }
    }
}

// ------------------------------------------------------------------ training (FP32)
// Loss and gradient of a minibatch in two launches.
//
// k_mlp_grad: a CTA takes tiles of 64 rows through the forward and the backward pass with
// every activation in shared memory and adds the tile's weight gradient to 4 x 4 register
// blocks, one per thread and layer; after its last tile it writes one partial gradient.
// k_mlp_reduce sums the partials in CTA order (the gradient does not depend on which CTA
// finishes first) and, for a training step, applies Adam to the sum.
// Bound: FP32 FMA, 29 k per row (8192 rows: 3 us of the chip's FMA rate; one 64-row tile
// takes one CTA about 10 us, which is what a minibatch of up to 304 tiles costs).
// One kernel per layer and operand (a thread per output element, every activation through
// memory, weight gradients by serial loops over 2048 rows on 4 to 132 blocks, added
// atomically) took 1242 us at 8192 rows.
// Rows of 64 activations are 68 floats apart, rows of 24 inputs 28: eight consecutive
// rows' 16-byte pieces then lie in distinct banks.
constexpr int GT = 64, LDH = 68, LDX = 28;
struct MlpTile {
    float w1[MLP_H][LDX], w2[MLP_H][LDH], w3[MLP_H][LDH], w4[MLP_H], b[3][MLP_H], b4[4];
    float x[GT][LDX], h1[GT][LDH], h2[GT][LDH], h3[GT][LDH], dz[GT], loss[GT];
};

__device__ __forceinline__ float bf16_round(float x) { return __bfloat162float(__float2bfloat16_rn(x)); }
__device__ __forceinline__ float4 lds4(const float *p) { return *reinterpret_cast<const float4 *>(p); }
__device__ __forceinline__ void fma4(float (&c)[4], float a, float4 b)
{
    c[0] = fmaf(a, b.x, c[0]), c[1] = fmaf(a, b.y, c[1]), c[2] = fmaf(a, b.z, c[2]), c[3] = fmaf(a, b.w, c[3]);
}
__device__ __forceinline__ float dot4(float4 a, float4 b, float c)
{
    return fmaf(a.w, b.w, fmaf(a.z, b.z, fmaf(a.y, b.y, fmaf(a.x, b.x, c))));
}

// out[r][o] = relu(b[o] + sum_k in[r][k] w[o][k]): rows 4 ty.., columns tx + 16 j
template <int K, int LDI, int LDW>
__device__ __forceinline__ void tile_forward(const float (*in)[LDI], const float (*w)[LDW], const float *b,
                                             float (*out)[LDH], int ty, int tx)
{
    float c[4][4];
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) c[i][j] = b[tx + 16 * j];
#pragma unroll 2
    for (int k = 0; k < K; k += 4) {
        float4 a[4], q[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) a[i] = lds4(&in[4 * ty + i][k]);
#pragma unroll
        for (int j = 0; j < 4; ++j) q[j] = lds4(&w[tx + 16 * j][k]);
#pragma unroll
        for (int i = 0; i < 4; ++i)
#pragma unroll
            for (int j = 0; j < 4; ++j) c[i][j] = dot4(a[i], q[j], c[i][j]);
    }
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) out[4 * ty + i][tx + 16 * j] = fmaxf(c[i][j], 0.f);
}

// d[o][k] += sum_r dz[r][o] h[r][k]: rows o = 4 ty.., columns k = 4 tx..
template <int LDI>
__device__ __forceinline__ void tile_grad(const float (*dz)[LDH], const float (*h)[LDI], float (&d)[4][4], int ty, int tx)
{
#pragma unroll 4
    for (int r = 0; r < GT; ++r) {
        const float4 a = lds4(&dz[r][4 * ty]), q = lds4(&h[r][4 * tx]);
        fma4(d[0], a.x, q);
        fma4(d[1], a.y, q);
        fma4(d[2], a.z, q);
        fma4(d[3], a.w, q);
    }
}

// h[r][k] <- (h[r][k] > 0) sum_o dz[r][o] w[o][k], in place (ends with a barrier)
__device__ __forceinline__ void tile_backward(const float (*dz)[LDH], const float (*w)[LDH], float (*h)[LDH], int ty,
                                              int tx)
{
    float c[4][4] = {};
#pragma unroll 2
    for (int o = 0; o < MLP_H; o += 4) {
        float4 a[4], q[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) a[i] = lds4(&dz[4 * ty + i][o]);
#pragma unroll
        for (int j = 0; j < 4; ++j) q[j] = lds4(&w[o + j][4 * tx]);
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            fma4(c[i], a[i].x, q[0]);
            fma4(c[i], a[i].y, q[1]);
            fma4(c[i], a[i].z, q[2]);
            fma4(c[i], a[i].w, q[3]);
        }
    }
    __syncthreads();                              // h was also read as the layer's input
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        float4 m = lds4(&h[4 * ty + i][4 * tx]);
        m.x = m.x > 0.f ? c[i][0] : 0.f, m.y = m.y > 0.f ? c[i][1] : 0.f;
        m.z = m.z > 0.f ? c[i][2] : 0.f, m.w = m.w > 0.f ? c[i][3] : 0.f;
        *reinterpret_cast<float4 *>(&h[4 * ty + i][4 * tx]) = m;
    }
    __syncthreads();
}

__device__ __forceinline__ float column_sum(const float (*z)[LDH], int o)
{
    float s = 0.f;
#pragma unroll 8
    for (int r = 0; r < GT; ++r) s += z[r][o];
    return s;
}

__global__ void __launch_bounds__(256) k_mlp_grad(const float *__restrict__ theta, const float *__restrict__ x,
                                                  const uint8_t *__restrict__ y, long long n, float pw,
                                                  float *__restrict__ part)
{
    extern __shared__ __align__(16) unsigned char raw[];
    MlpTile &t = *reinterpret_cast<MlpTile *>(raw);
    const int tid = threadIdx.x, ty = tid / 16, tx = tid % 16;
    for (int i = tid; i < MLP_H * MLP_IN; i += 256) t.w1[i / MLP_IN][i % MLP_IN] = bf16_round(theta[OFF_W1 + i]);
    for (int i = tid; i < MLP_H * MLP_H; i += 256) {
        t.w2[i / MLP_H][i % MLP_H] = bf16_round(theta[OFF_W2 + i]);
        t.w3[i / MLP_H][i % MLP_H] = bf16_round(theta[OFF_W3 + i]);
    }
    if (tid < MLP_H) {
        t.w4[tid] = bf16_round(theta[OFF_W4 + tid]);
        t.b[0][tid] = bf16_round(theta[OFF_B1 + tid]);
        t.b[1][tid] = bf16_round(theta[OFF_B2 + tid]);
        t.b[2][tid] = bf16_round(theta[OFF_B3 + tid]);
    }
    if (tid == 0) t.b4[0] = bf16_round(theta[OFF_B4]);
    float d3[4][4] = {}, d2[4][4] = {}, d1[4][4] = {};
    float dv = 0.f, db1 = 0.f;                    // thread's bias and output-layer sums, see below
    const int o = tid % MLP_H, part4 = tid / MLP_H;
    for (long long r0 = (long long)blockIdx.x * GT; r0 < n; r0 += (long long)gridDim.x * GT) {
        __syncthreads();
        for (int i = tid; i < GT * MLP_IN; i += 256) {
            const long long g = r0 * MLP_IN + i;
            t.x[i / MLP_IN][i % MLP_IN] = g < n * MLP_IN ? __ldg(x + g) : 0.f;
        }
        __syncthreads();
        tile_forward<MLP_IN, LDX, LDX>(t.x, t.w1, t.b[0], t.h1, ty, tx);
        __syncthreads();
        tile_forward<MLP_H, LDH, LDH>(t.h1, t.w2, t.b[1], t.h2, ty, tx);
        __syncthreads();
        tile_forward<MLP_H, LDH, LDH>(t.h2, t.w3, t.b[2], t.h3, ty, tx);
        __syncthreads();
        {
            // logit of row tid / 4 by four threads, then the weighted BCE with logits:
            // dz = (s (pw y + 1 - y) - pw y) / n
            const int r = tid / 4, q = tid % 4;
            float z = 0.f;
#pragma unroll
            for (int k = 0; k < MLP_H; k += 16) z = dot4(lds4(&t.h3[r][k + 4 * q]), lds4(&t.w4[k + 4 * q]), z);
            z += __shfl_xor_sync(0xffffffffu, z, 1);
            z += __shfl_xor_sync(0xffffffffu, z, 2);
            if (q == 0) {
                float dz = 0.f, l = 0.f;
                if (r0 + r < n) {
                    const float zi = z + t.b4[0], yi = y[r0 + r] ? 1.f : 0.f;
                    const float s = 1.f / (1.f + expf(-zi));
                    dz = (s * (pw * yi + 1.f - yi) - pw * yi) / (float)n;
                    const float lsp = zi > 0.f ? zi + log1pf(expf(-zi)) : log1pf(expf(zi));   // log(1 + e^z)
                    l = (pw * yi * (lsp - zi) + (1.f - yi) * lsp) / (float)n;
                }
                t.dz[r] = dz;
                t.loss[r] = l;
            }
        }
        __syncthreads();
        // output layer: threads 0-63 its weights, 64 its bias, 65 the loss
        if (part4 == 0) {
#pragma unroll 8
            for (int r = 0; r < GT; ++r) dv = fmaf(t.dz[r], t.h3[r][o], dv);
        } else if (tid == 64 || tid == 65) {
            const float *v = tid == 64 ? t.dz : t.loss;
#pragma unroll 8
            for (int r = 0; r < GT; ++r) dv += v[r];
        }
        __syncthreads();
        for (int i = tid; i < GT * MLP_H / 4; i += 256) {        // h3 <- dZ3
            const int r = i / 16, k = 4 * (i % 16);
            const float4 h = lds4(&t.h3[r][k]), w = lds4(&t.w4[k]);
            const float g = t.dz[r];
            *reinterpret_cast<float4 *>(&t.h3[r][k]) = make_float4(h.x > 0.f ? g * w.x : 0.f, h.y > 0.f ? g * w.y : 0.f,
                                                                   h.z > 0.f ? g * w.z : 0.f, h.w > 0.f ? g * w.w : 0.f);
        }
        __syncthreads();
        tile_grad<LDH>(t.h3, t.h2, d3, ty, tx);
        tile_backward(t.h3, t.w3, t.h2, ty, tx);                 // h2 <- dZ2
        tile_grad<LDH>(t.h2, t.h1, d2, ty, tx);
        tile_backward(t.h2, t.w2, t.h1, ty, tx);                 // h1 <- dZ1
        // input layer: 96 threads its weights (16 x 6 blocks of 4 x 4), the others the
        // biases of the three hidden layers (two threads of 128 take two columns)
        if (tid < 96) tile_grad<LDX>(t.h1, t.x, d1, tid / 6, tid % 6);
        else if (tid < 224) {
            const int q = tid - 96;
            if (q < 64) db1 += column_sum(t.h1, q);
            else db1 += column_sum(t.h2, q - 64);
        }
        if (tid >= 192 && tid < 256) dv += column_sum(t.h3, tid - 192);
    }
    float *g = part + (long long)blockIdx.x * MLP_PART;
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const int k = (4 * ty + i) * MLP_H + 4 * tx;
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            g[OFF_W3 + k + j] = d3[i][j];
            g[OFF_W2 + k + j] = d2[i][j];
        }
        if (tid < 96)
#pragma unroll
            for (int j = 0; j < 4; ++j) g[OFF_W1 + (4 * (tid / 6) + i) * MLP_IN + 4 * (tid % 6) + j] = d1[i][j];
    }
    if (part4 == 0) g[OFF_W4 + o] = dv;
    if (tid == 64) g[OFF_B4] = dv;
    if (tid == 65) g[MLP_PARAMS] = dv;
    if (tid >= 96 && tid < 160) g[OFF_B1 + tid - 96] = db1;
    if (tid >= 160 && tid < 224) g[OFF_B2 + tid - 160] = db1;
    if (tid >= 192) g[OFF_B3 + tid - 192] = dv;
}

// Sum of the n_part partials of each parameter (32 parameters x 8 groups of partials per
// block, each group and then the groups in order); the sum goes to grad, the loss to
// *loss, and with theta the parameter takes an Adam step (c1, c2: 1 - beta^step).
__global__ void __launch_bounds__(256) k_mlp_reduce(const float *__restrict__ part, int n_part, float *grad, float *loss,
                                                    float *theta, float *m, float *v, float lr, float c1, float c2)
{
    __shared__ float sh[8][32];
    const int l = threadIdx.x & 31, w = threadIdx.x >> 5, i = blockIdx.x * 32 + l;
    float s = 0.f;
    if (i <= MLP_PARAMS)
#pragma unroll 8
        for (int p = w; p < n_part; p += 8) s += __ldg(part + (long long)p * MLP_PART + i);
    sh[w][l] = s;
    __syncthreads();
    if (w != 0 || i > MLP_PARAMS) return;
#pragma unroll
    for (int q = 1; q < 8; ++q) s += sh[q][l];
    if (i == MLP_PARAMS) {
        if (loss) *loss = s;
        return;
    }
    if (grad) grad[i] = s;
    if (theta) {
        const float mi = 0.9f * m[i] + 0.1f * s, vi = 0.999f * v[i] + 0.001f * s * s;
        m[i] = mi;
        v[i] = vi;
        theta[i] -= lr * (mi / c1) / (sqrtf(vi / c2) + 1e-8f);
    }
}

template <int DIM, int NSR, int PREC>
void crit_launch(const DevMesh &m, const StageArgs &a, double kappa, double eps, uint8_t *flags, cudaStream_t s)
{
    k_criterion<DIM, NSR, PREC><<<nblk(m.n_cells, 128), 128, 0, s>>>(m, a, (float)kappa, (float)eps, flags);
}
template <int DIM, int PREC> void own_launch(const DevMesh &m, const StageArgs &a, float *own, cudaStream_t s)
{
    k_own_features<DIM, PREC><<<nblk(m.n_cells, 128), 128, 0, s>>>(m, a, own);
}

template <int DIM, int NSR> void reg_one(IndicatorFns *t)
{
    t[indicator_index(DIM, NSR, PREC_F64)] = IndicatorFns{&crit_launch<DIM, NSR, PREC_F64>, &own_launch<DIM, PREC_F64>};
    t[indicator_index(DIM, NSR, PREC_F32)] = IndicatorFns{&crit_launch<DIM, NSR, PREC_F32>, &own_launch<DIM, PREC_F32>};
    t[indicator_index(DIM, NSR, PREC_BF16)] = IndicatorFns{&crit_launch<DIM, NSR, PREC_BF16>, &own_launch<DIM, PREC_BF16>};
}

}  // namespace

void register_indicator(IndicatorFns *t)
{
    reg_one<2, 2>(t);
    reg_one<2, 3>(t);
    reg_one<2, 4>(t);
    reg_one<3, 2>(t);
    reg_one<3, 3>(t);
    reg_one<3, 4>(t);
}

void launch_gather24(const DevMesh &m, const float *own, float *x, cudaStream_t s)
{
    k_gather24<<<nblk(m.n_cells, 128), 128, 0, s>>>(m, own, x);
}
void launch_mlp_frags(const float *theta, uint2 *frag, cudaStream_t s)
{
    k_mlp_frags<<<nblk(N_FRAGS * 32, 256), 256, 0, s>>>(theta, frag);
}
void launch_mlp_infer(const uint2 *frag, const float *theta, const float *x, long long n, float *logits,
                      uint8_t *flags, cudaStream_t s)
{
    long long tiles = (n + 31) / 32;
    int blocks = (int)((tiles + 3) / 4);
    if (blocks > 152 * 8) blocks = 152 * 8;
    if (blocks < 1) blocks = 1;
    k_mlp_infer<false><<<blocks, 128, 0, s>>>(frag, theta, x, n, logits, flags, DevMesh{}, nullptr);
}
void launch_mlp_infer_fused(const uint2 *frag, const float *theta, const DevMesh &m, const float *own, float *logits,
                            uint8_t *flags, cudaStream_t s)
{
    const long long n = m.n_cells;
    long long tiles = (n + 31) / 32;
    int blocks = (int)((tiles + 3) / 4);
    if (blocks > 152 * 8) blocks = 152 * 8;
    if (blocks < 1) blocks = 1;
    k_mlp_infer<true><<<blocks, 128, 0, s>>>(frag, theta, nullptr, n, logits, flags, m, own);
}
cudaError_t mlp_setup()
{
    return cudaFuncSetAttribute(k_mlp_grad, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(MlpTile));
}
int launch_mlp_grad(const float *theta, const float *x, const uint8_t *y, long long n, float pw, float *part,
                    cudaStream_t s)
{
    const long long tiles = (n + GT - 1) / GT;
    const int grid = (int)(tiles < MLP_MAX_PARTS ? tiles : MLP_MAX_PARTS);
    k_mlp_grad<<<grid, 256, sizeof(MlpTile), s>>>(theta, x, y, n, pw, part);
    return grid;
}
void launch_mlp_reduce(const float *part, int n_part, float *grad, float *loss, float *theta, float *m, float *v,
                       float lr, int step, cudaStream_t s)
{
    const float c1 = 1.f - powf(0.9f, (float)step), c2 = 1.f - powf(0.999f, (float)step);
    k_mlp_reduce<<<nblk(MLP_PARAMS + 1, 32), 256, 0, s>>>(part, n_part, grad, loss, theta, m, v, lr, c1, c2);
}

}  // namespace dol

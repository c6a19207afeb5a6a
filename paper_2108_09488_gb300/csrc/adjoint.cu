// adjoint.cu -- gradients of a concentration misfit with respect to the dispersivities, the molecular
// diffusion and the initial concentrations: the hand-written adjoint of the SPH step.
//
// The paper has no adjoint; this is derived from Eq. 3-5 and Eq. 8-9.  For a uniform velocity and
// uniform m / rho (the configured workloads):
//   * the rate is linear in C, r = L(theta) C, with (L u)_a = sum_b w_ab (u_a - u_b) and symmetric
//     weights w_ab = w_ba (the pair factor of Eq. 5 is even in x_ab), so L is symmetric;
//   * D of Eq. 3 is linear in theta = (alpha_L, alpha_T, D_m):  D = alpha_L B_L + alpha_T B_T + D_m I
//     with B_L = v v^T/|v| and B_T = |v| I - v v^T/|v|; for equal D_a = D_b the harmonic mean of
//     Eq. 5 is 2D, so L = alpha_L L_L + alpha_T L_T + D_m L_m with L_k the operator for D = B_k;
//   * the relative particle positions do not change (uniform drift), so L is the same at every
//     step and one predictor-corrector step (Eq. 8-9) is C^{l+1} = S C^l, S = I + dt L + dt^2 L^2 / 2.
// For J = 1/2 |C^N - C*|^2 and a fixed dt:
//   lambda^N = C^N - C*,  lambda^l = S^T lambda^{l+1} = S lambda^{l+1},  dJ/dC^0 = lambda^0,
//   dJ/dtheta_k = sum_l lambda^{l+1} . (dS/dtheta_k) C^l
//               = sum_l [ dt p.(L_k u) + dt^2/2 ( p.(L_k L u) + (L p).(L_k u) ) ],  u = C^l, p = lambda^{l+1}.
// Forward states are kept as checkpoints every `ckpt_every` steps and recomputed segment by segment
// on the way back.  All operators use one cell list built at the initial positions (the geometry
// is frozen, which is exact for a uniform drift), so forward and adjoint apply the same L.
// With a uniform v every one of these operators is a combination of two sums over the pairs,
//   S_L = pf sum_b g_L (x_a - x_b),  S_T = pf sum_b g_T (x_a - x_b),
// g_L and g_T the weights for D = vhat vhat^T and I - vhat vhat^T (frozen_table.cuh):
//   L_L = |v| S_L,  L_T = |v| S_T,  L_m = S_L + S_T,  L = d_L S_L + d_T S_T, d_i = alpha_i |v| + D_m
// (sums with D's other split, a (vhat . e)^2 + b, cancel: dJ/dalpha lost up to a factor of 8 in
// accuracy).  g_L and g_T never change during a call, so
// they are computed once (frozen_table.cuh) and an evaluation streams them; the state and the adjoint
// state of a backward step share one pass, and the dot products are taken in that pass from S_L and S_T,
// so a backward step is two launches and a forward step two.
// Bound: L2 / HBM, 8 bytes a pair (10 on average with the low parts that the backward passes read).  512^2 lattice,
// 20 neighbours, 40 steps: 13.3 -> 4.05 ms (the dot
// products' kernel alone took 97 us a step: nine threads folded 1024 FP64 partials one by one).
// Precision: the states are FP32 (C, half steps, L u), everything else that all pairs or steps share is kept to FP64
// or nearly (weights to 32 bits with their low parts, the geometry behind them, the time step, prefactor and
// coefficients), and the sums behind the dot products take every rounding along: dJ/dtheta is within 1e-9 (one
// case 8e-9) of an FP64 computation with the states rounded alike, and the states' roundings move it by up to 1.4e-7
// (6 plumes of 85^2 to 512^2 against FP64: 5e-10..5e-8; with weights and sums in FP32 4e-9..2e-7).
#include <math.h>
#include <stdio.h>
#include <string.h>

#include <algorithm>
#include <vector>

#include "ade_internal.h"

namespace ade {

namespace {

#include "rate_common.cuh"

#include "rate_walk.cuh"

#include "frozen_table.cuh"

constexpr int kT = kFrozenThreads;
constexpr double kTwo32 = 4294967296.0;
constexpr int kDots = 6;   // per backward step: p.S_L u, p.S_T u, b.S_L u, b.S_T u (b = L p), p.S_L a, p.S_T a (a = L u)

// S_L (x) and S_T (y) of NR fields, rows summed in FP32 and added up with Neumaier's compensation.  LOW (the dot
// products of the backward passes): the last field's sums take the weights' low parts and the rounding of every
// product and addition, for on a lattice the weights' and the row sums' roundings bias all particles alike
// (dJ/dtheta by up to 2e-7).  The states do not need that: they are rounded to FP32 themselves.
template <int NR, bool LOW>
struct ShapeSums {
    const float *x[NR];
    const float *words, *low;
    float xa[NR];
    float2 r[NR], a[NR], c[NR];
    __device__ __forceinline__ void zero()
    {
#pragma unroll
        for (int q = 0; q < NR; ++q) r[q] = a[q] = c[q] = f2(0.f, 0.f);
    }
    __device__ __forceinline__ void add(int q, float2 w, float2 lo, float xb)
    {
        const float2 d = both(xa[q] - xb);
        if (LOW && q == NR - 1) {
            c[q] = __ffma2_rn(lo, d, c[q]);
            r[q] = two_sum2(r[q], two_prod2(w, d, c[q]), c[q]);
        } else {
            r[q] = __ffma2_rn(w, d, r[q]);
        }
    }
    __device__ __forceinline__ void prefetch(const float *base, int first, int n) const
    {
        if (LOW) prefetch_l2(low + (((size_t)(base - words) >> 5) + first) / 2 * 32, (unsigned)(n / 2) * 128u + 128u);
    }
    template <int M>
    __device__ __forceinline__ void lines(const float *w, int s)
    {
        float2 wv[M];
        float lv[M], xv[NR][M];
        const int lane = threadIdx.x & 31;
        const float *lw = low + (((size_t)(w - words) - 2 * lane) >> 6) * 32 + lane;
#pragma unroll
        for (int u = 0; u < M; ++u) {
            wv[u] = __ldg(reinterpret_cast<const float2 *>(w) + u * 32);
            lv[u] = LOW ? ld_weight(lw + u * 32) : 0.f;
#pragma unroll
            for (int q = 0; q < NR; ++q) xv[q][u] = x[q][s + u];
        }
#pragma unroll
        for (int u = 0; u < M; ++u) {
            const float2 lo = unpack_low(lv[u]);
#pragma unroll
            for (int q = 0; q < NR; ++q) add(q, wv[u], lo, xv[q][u]);
        }
    }
    __device__ __forceinline__ void end_row()
    {
#pragma unroll
        for (int q = 0; q < NR; ++q) {
            neumaier_add2(a[q], c[q], r[q]);
            r[q] = f2(0.f, 0.f);
        }
    }
    __device__ __forceinline__ float s0(int q) const { return a[q].x + c[q].x; }
    __device__ __forceinline__ float s1(int q) const { return a[q].y + c[q].y; }
    __device__ __forceinline__ double d0(int q) const { return (double)a[q].x + (double)c[q].x; }
    __device__ __forceinline__ double d1(int q) const { return (double)a[q].y + (double)c[q].y; }
};

// The same sums over the positions, for a chunk without room in the table: the rows and ranges of the table's
// chunks (cut by the cell bands), two candidates at a time.
template <int DIM, int KERNEL, bool ISO, int NR, bool LOW>
__device__ __noinline__ void walk_sums(const uint4 *__restrict__ P, const uint32_t *__restrict__ cs, const RateParams &prm, Chunk c,
                                       const ShapeConst sc, ShapeSums<NR, LOW> &op)
{
    const uint4 pa = __ldg(P + min(c.i0 + (int)(threadIdx.x & 31), c.pe - 1));
    c.cy = c.p % prm.ncy;
    c.cz = c.p / prm.ncy;
    const PairConst kc(prm);
    const PairConst2 k(kc, kc.m1);
    chunk_rows<DIM, ISO, ISO ? kCutBand : kCutFull>(P, cs, prm, c, pa, nullptr, [&](int qs, int qe, int s, int m, int) {
        const int len = qe - qs;
        for (int t = 0; t < m; t += 2) {
            const int j0 = s + t, j1 = min(t + 1, m - 1) + s;
            const int i0 = j0 >= qe ? j0 - len : j0, i1 = j1 >= qe ? j1 - len : j1;
            Double2 gL, gT;
            pair_fine2<DIM, KERNEL, ISO>(pa, __ldg(P + i0), __ldg(P + i1), k, sc, gL, gT);
#pragma unroll
            for (int f = 0; f < NR; ++f) {
                op.add(f, f2(gL.h.x, gT.h.x), f2(gL.l.x, gT.l.x), op.x[f][qs + i0]);
                if (t + 1 < m) op.add(f, f2(gL.h.y, gT.h.y), f2(gL.l.y, gT.l.y), op.x[f][qs + i1]);
            }
        }
        op.end_row();
    });
}

// The table (prm.uw = vhat, prm.ub = 0) and the initial concentrations, doubled per pencil and as kept.
template <int DIM, int KERNEL, bool ISO>
__global__ __launch_bounds__(kT) void k_adj_table(const uint4 *__restrict__ P, const uint32_t *__restrict__ cs,
                                                  const RateParams prm, const FrozenTab tab, const ShapeConst sc, float *__restrict__ C0, float *__restrict__ kept)
{
    pdl_wait();
    __shared__ TrimRow srow[ISO ? kMaxRows : 1];
    if (ISO) stage_trim_rows(srow, prm);
    Chunk c;
    const int t = warp_number();
    const bool has = find_chunk(cs, prm, tab.dense, t, c);
    if (t < chunk_numbers(prm.n, prm.ncy * prm.ncz)) put_chunk(tab, c, has);
    if (!has) return;
    const int i = c.i0 + (threadIdx.x & 31);
    const uint4 pa = __ldg(P + min(i, c.pe - 1));
    build_chunk<DIM, KERNEL, ISO, ISO ? kCutBox : kCutFull, 2, true>(P, cs, prm, c, pa, srow, tab, sc);
    if (i < c.pe) C0[c.ps + i] = C0[c.pe + i] = kept[i] = __uint_as_float(pa.w);
}

// One pass over the table; fields doubled per pencil (states that are kept for later, once per particle).
//   HALF, FULL  out1 = base + step L x1 (HALF: base = x1)
//   BACK1       out0 = a = L x0 (x0 = u), out1 = x1 + step L x1 (x1 = p); dots of p and b = L p with S_L u, S_T u
//   BACK2       out1 = base + step L x1 (x1 = hp, base = p; out1 may be base); dots of p with S_L a, S_T a (x0 = a)
enum AdjMode { HALF = 0, FULL = 1, BACK1 = 2, BACK2 = 3 };
struct AdjPass {
    const float *x0, *x1, *base;
    float *out0, *out1;
    float ca, cb, cal, cbl;   // L x = ca S_L + cb S_T (hi + lo), pf folded in
    float step;
    float *kept;           // FULL: out1 once per particle as well (NULL: not)
    const float *next;     // BACK2: the kept state that the next step reads, doubled into next2 (NULL: none)
    float *next2;
    ShapeConst sc;
    double *partials;      // [blocks][kDots] of the step (BACK1: the first four, BACK2: the last two)
};

__device__ __forceinline__ float combine(const AdjPass &ps, float s0, float s1)
{
    return fmaf(ps.ca, s0, fmaf(ps.cb, s1, fmaf(ps.cal, s0, ps.cbl * s1)));
}

// Sum of v[0..4) over the warp's lanes: every exchange halves the values a lane holds, so four sums take
// 6 FP64 additions a lane instead of 20 (FP64 runs at a sixtieth of the FP32 rate here).  Lanes
// 0, 8, 16, 24 hold sums 0, 1, 2, 3.
__device__ __forceinline__ double warp_sums4(double v0, double v1, double v2, double v3)
{
    const int lane = threadIdx.x & 31;
    const bool hi = (lane & 16) != 0, h8 = (lane & 8) != 0;
    const double t0 = (hi ? v2 : v0) + __shfl_xor_sync(kFull, hi ? v0 : v2, 16);
    const double t1 = (hi ? v3 : v1) + __shfl_xor_sync(kFull, hi ? v1 : v3, 16);
    double r = (h8 ? t1 : t0) + __shfl_xor_sync(kFull, h8 ? t0 : t1, 8);
    for (int o = 4; o > 0; o >>= 1) r += __shfl_xor_sync(kFull, r, o);
    return r;
}

// Block sums of d[0..ND) into out[0..ND) (a fixed order).  Every thread must call it.
template <int ND>
__device__ __forceinline__ void block_sums(const double (&d)[ND], double *out)
{
    constexpr int G = (ND + 3) / 4;
    __shared__ double sh[kT / 32][4 * G];
    const int lane = threadIdx.x & 31;
#pragma unroll
    for (int g = 0; g < G; ++g) {
        const double r = warp_sums4(d[4 * g], 4 * g + 1 < ND ? d[(4 * g + 1) % ND] : 0.0, 4 * g + 2 < ND ? d[(4 * g + 2) % ND] : 0.0,
                                    4 * g + 3 < ND ? d[(4 * g + 3) % ND] : 0.0);
        if ((lane & 7) == 0) sh[threadIdx.x >> 5][4 * g + (lane >> 3)] = r;
    }
    __syncthreads();
    if (threadIdx.x < ND) {
        double t = 0.0;
        for (int w = 0; w < kT / 32; ++w) t += sh[w][threadIdx.x];
        out[threadIdx.x] = t;
    }
}

template <int DIM, int KERNEL, bool ISO, int MODE>
__global__ __launch_bounds__(kT) void k_adj_pass(const uint4 *__restrict__ P, const uint32_t *__restrict__ cs,
                                                 const RateParams prm, const FrozenTab tab, const AdjPass ps)
{
    pdl_wait();
    constexpr bool BACK = MODE >= BACK1;
    constexpr int NR = BACK ? 2 : 1, ND = MODE == BACK1 ? 4 : 2;   // fields: x1, then x0
    double dot[ND];
#pragma unroll
    for (int q = 0; q < ND; ++q) dot[q] = 0.0;
    Chunk c;
    uint4 sl;
    if (my_chunk(tab, prm, c, sl)) {
        const int i = c.i0 + (threadIdx.x & 31);
        const int at = c.ps + min(i, c.pe - 1);
        ShapeSums<NR, BACK> op;
        op.zero();
        op.words = tab.words;
        op.low = tab.low;
        op.x[0] = ps.x1;
        op.xa[0] = ps.x1[at];
        if (BACK) {
            op.x[NR - 1] = ps.x0;
            op.xa[NR - 1] = ps.x0[at];
        }
        if (sl.x != kNoRoom) stream_rows<2>(sl, tab, op);
        else walk_sums<DIM, KERNEL, ISO, NR, BACK>(P, cs, prm, c, ps.sc, op);
        if (i < c.pe) {
            const int again = c.pe + i;
            const float L1 = combine(ps, op.s0(0), op.s1(0));
            const float p = MODE == HALF || MODE == BACK1 ? op.xa[0] : ps.base[at];
            const float o = fmaf(ps.step, L1, p);
            ps.out1[at] = ps.out1[again] = o;
            if (MODE == FULL && ps.kept) ps.kept[i] = o;
            if (MODE == BACK2 && ps.next) ps.next2[at] = ps.next2[again] = ps.next[i];
            if (BACK) {
                const double s0 = op.d0(NR - 1), s1 = op.d1(NR - 1);
                dot[0] = (double)p * s0;
                dot[1] = (double)p * s1;
                if (MODE == BACK1) {
                    dot[2 % ND] = (double)L1 * s0;
                    dot[3 % ND] = (double)L1 * s1;
                    ps.out0[at] = ps.out0[again] = combine(ps, op.s0(NR - 1), op.s1(NR - 1));
                }
            }
        }
    }
    if (BACK)
        block_sums<ND>(dot, ps.partials + (size_t)blockIdx.x * kDots + (MODE == BACK2 ? 4 : 0));
}

// lambda^N = C^N - C* (doubled per pencil; C^N as kept) and its squares' block sums.
__global__ __launch_bounds__(kT) void k_adj_misfit(const uint32_t *__restrict__ perm, const RateParams prm, const FrozenTab tab,
                                                   const float *__restrict__ CN, const float *__restrict__ target,
                                                   float *__restrict__ p, double *__restrict__ partials)
{
    pdl_wait();
    double d[kDots] = {0.0};
    Chunk c = {};
    uint4 sl;
    const bool has = my_chunk(tab, prm, c, sl);
    const int i = c.i0 + (int)(threadIdx.x & 31);
    if (has && i < c.pe) {
        const uint32_t a = __ldg(perm + i);
        const float t = a < (uint32_t)prm.n ? __ldg(target + a) : 0.f;
        const float v = fmaf(-1.f, t, CN[i]);
        p[c.ps + i] = p[c.pe + i] = v;
        d[0] = (double)v * (double)v;
    }
    block_sums<kDots>(d, partials + (size_t)blockIdx.x * kDots);
}

// out[step][q] = sum over the blocks' partials, one CTA per step, in a fixed order.
constexpr int kFoldT = 256;
__global__ __launch_bounds__(kFoldT) void k_adj_fold(const double *__restrict__ partials, int blocks, double *__restrict__ out)
{
    pdl_wait();
    __shared__ double sh[kFoldT / 32][kDots];
    const double *p = partials + (size_t)blockIdx.x * blocks * kDots;
    double s[kDots];
#pragma unroll
    for (int q = 0; q < kDots; ++q) s[q] = 0.0;
    for (int b = threadIdx.x; b < blocks; b += kFoldT)
#pragma unroll
        for (int q = 0; q < kDots; ++q) s[q] += p[(size_t)b * kDots + q];
#pragma unroll
    for (int q = 0; q < kDots; ++q)
        for (int o = 16; o > 0; o >>= 1) s[q] += __shfl_down_sync(kFull, s[q], o);
    if ((threadIdx.x & 31) == 0)
#pragma unroll
        for (int q = 0; q < kDots; ++q) sh[threadIdx.x >> 5][q] = s[q];
    __syncthreads();
    if (threadIdx.x < kDots) {
        double t = 0.0;
        for (int w = 0; w < kFoldT / 32; ++w) t += sh[w][threadIdx.x];
        out[(size_t)blockIdx.x * kDots + threadIdx.x] = t;
    }
}

// out[perm[i]] = the value of sorted particle i, of a doubled field or a kept one.
__global__ __launch_bounds__(kT) void k_adj_scatter(const uint32_t *__restrict__ perm, const RateParams prm, const FrozenTab tab,
                                                    const float *__restrict__ x, bool doubled, float *__restrict__ out)
{
    pdl_wait();
    Chunk c;
    uint4 sl;
    if (!my_chunk(tab, prm, c, sl)) return;
    const int i = c.i0 + (threadIdx.x & 31);
    if (i >= c.pe) return;
    const uint32_t a = __ldg(perm + i);
    if (a < (uint32_t)prm.n) out[a] = x[doubled ? c.ps + i : i];
}

// A kept state doubled per pencil.
__global__ __launch_bounds__(kT) void k_adj_double(const RateParams prm, const FrozenTab tab, const float *__restrict__ x,
                                                   float *__restrict__ out)
{
    pdl_wait();
    Chunk c;
    uint4 sl;
    if (!my_chunk(tab, prm, c, sl)) return;
    const int i = c.i0 + (threadIdx.x & 31);
    if (i < c.pe) out[c.ps + i] = out[c.pe + i] = x[i];
}

// Everything one call needs.
struct Adj {
    const ade_ctx *c;
    cudaStream_t s;
    RateParams rp;         // uw = vhat, ub = 0
    FrozenTab tab;
    float ca, cb, cal, cbl;   // L(theta) x = ca S_L + cb S_T (hi + lo)
    ShapeConst sc;
    unsigned blocks;
};

template <int DIM, int KERNEL, bool ISO>
cudaError_t pass_t(const Adj &A, int mode, const AdjPass &ps)
{
    const uint4 *P = A.c->w.P0;
    const uint32_t *cs = A.c->w.cell_start;
    switch (mode) {
    case HALF: return launch_pdl(k_adj_pass<DIM, KERNEL, ISO, HALF>, A.blocks, kT, 0, A.s, P, cs, A.rp, A.tab, ps);
    case FULL: return launch_pdl(k_adj_pass<DIM, KERNEL, ISO, FULL>, A.blocks, kT, 0, A.s, P, cs, A.rp, A.tab, ps);
    case BACK1: return launch_pdl(k_adj_pass<DIM, KERNEL, ISO, BACK1>, A.blocks, kT, 0, A.s, P, cs, A.rp, A.tab, ps);
    default: return launch_pdl(k_adj_pass<DIM, KERNEL, ISO, BACK2>, A.blocks, kT, 0, A.s, P, cs, A.rp, A.tab, ps);
    }
}

template <int DIM, int KERNEL, bool ISO>
cudaError_t table_t(const Adj &A, float *C0, float *kept)
{
    return launch_pdl(k_adj_table<DIM, KERNEL, ISO>, A.blocks, kT, 0, A.s, A.c->w.P0, A.c->w.cell_start, A.rp, A.tab, A.sc, C0, kept);
}

#define ADE_ADJ_CALL(F, ...)                                                                                          \
    (A.c->dim == 2 ? (A.c->p.kernel == ADE_WENDLAND_C2                                                                \
                          ? (A.c->iso ? F<2, ADE_WENDLAND_C2, true>(__VA_ARGS__) : F<2, ADE_WENDLAND_C2, false>(__VA_ARGS__))   \
                          : (A.c->iso ? F<2, ADE_WENDLAND_C4, true>(__VA_ARGS__) : F<2, ADE_WENDLAND_C4, false>(__VA_ARGS__)))  \
                   : (A.c->p.kernel == ADE_WENDLAND_C2                                                                \
                          ? (A.c->iso ? F<3, ADE_WENDLAND_C2, true>(__VA_ARGS__) : F<3, ADE_WENDLAND_C2, false>(__VA_ARGS__))   \
                          : (A.c->iso ? F<3, ADE_WENDLAND_C4, true>(__VA_ARGS__) : F<3, ADE_WENDLAND_C4, false>(__VA_ARGS__))))

cudaError_t pass(const Adj &A, int mode, const AdjPass &ps) { return ADE_ADJ_CALL(pass_t, A, mode, ps); }
cudaError_t table(const Adj &A, float *C0, float *kept) { return ADE_ADJ_CALL(table_t, A, C0, kept); }

// One forward step C_out = S C_in: h = u + dt/2 L u, C_out = u + dt L h (kept: once per particle as well).
cudaError_t fwd_step(const Adj &A, const float *u, float *h, float *out, float *kept, float dt)
{
    AdjPass ps;
    memset(&ps, 0, sizeof(ps));
    ps.ca = A.ca;
    ps.cb = A.cb;
    ps.cal = A.cal;
    ps.cbl = A.cbl;
    ps.sc = A.sc;
    ps.x1 = u;
    ps.out1 = h;
    ps.step = 0.5f * dt;
    cudaError_t e = pass(A, HALF, ps);
    if (e != cudaSuccess) return e;
    ps.x1 = h;
    ps.base = u;
    ps.out1 = out;
    ps.kept = kept;
    ps.step = dt;
    return pass(A, FULL, ps);
}

// Adjoint workspace: states kept once per particle (checkpoints, one segment), working fields doubled per pencil, FP64
// partials of one segment; the weight table lies behind.
struct AdjLayout {
    size_t ckpt, seg, u0, u1, h, p, hp, a, dots, partials, slots, dense, cursor, total;
    int nck, blocks;
};

AdjLayout adj_layout(const ade_ctx *c, int nsteps, int ck)
{
    AdjLayout L;
    size_t off = 0;
    auto take = [&](size_t bytes) {
        size_t o = off;
        off += ((bytes > 0 ? bytes : 1) + 255) & ~(size_t)255;
        return o;
    };
    const size_t f1 = (size_t)c->n * 4, f2 = 2 * f1;
    const size_t slots = table_slots(c);
    L.blocks = (int)((slots + kT / 32 - 1) / (kT / 32));
    L.nck = (nsteps + ck - 1) / ck;
    L.ckpt = take(f1 * (L.nck + 1));
    L.seg = take(f1 * std::min(ck, nsteps));
    L.u0 = take(f2);
    L.u1 = take(f2);
    L.h = take(f2);
    L.p = take(f2);
    L.hp = take(f2);
    L.a = take(f2);
    L.dots = take(((size_t)nsteps + 1) * kDots * 8);
    L.partials = take((size_t)L.blocks * std::min(ck, nsteps) * kDots * 8);
    L.slots = take(slots * 32);
    L.dense = take(slots * 4);
    L.cursor = take(64);
    L.total = off;
    return L;
}

}  // namespace

}  // namespace ade

#define ADJ_CK(call)                                                                               \
    do {                                                                                           \
        cudaError_t e_ = (call);                                                                   \
        if (e_ != cudaSuccess) {                                                                   \
            char m_[256];                                                                          \
            snprintf(m_, sizeof(m_), "%s: %s", #call, cudaGetErrorString(e_));                     \
            return ade::report_error(ADE_ERR_CUDA, m_);                                            \
        }                                                                                          \
    } while (0)

using namespace ade;

extern "C" int ade_adjoint_workspace_bytes(const ade_ctx *c, int nsteps, int ckpt_every, size_t *bytes)
{
    if (!c || !bytes || nsteps < 1 || ckpt_every < 1) return ade::report_error(ADE_ERR_ARG, "bad argument");
    *bytes = adj_layout(c, nsteps, ckpt_every).total;
    return ADE_OK;
}

extern "C" int ade_adjoint_weights_bytes(ade_ctx *c, int counted, size_t *bytes, void *stream)
{
    if (!c || !bytes) return ade::report_error(ADE_ERR_ARG, "NULL argument");
    *bytes = 0;
    if (c->field || c->n == 0) return ADE_OK;
    const int rc = plan_context_table(c, 2, counted != 0, &c->adj_plan, (cudaStream_t)stream);
    if (rc || c->adj_plan.stride == 0u || (!counted && c->adj_plan.lines == 0)) return rc;
    // above the limit: as many chunks as fit
    *bytes = c->adj_plan.lines > 0 ? c->adj_plan.lines * 192 + 256 : (size_t)kTableMaxBytes / 256 * 256;
    return ADE_OK;
}

extern "C" int ade_adjoint(ade_ctx *c, const float *C_target_dev, int nsteps, int ckpt_every, void *aws,
                           size_t aws_bytes, float *dJdC0_dev, double *dJdtheta_host, double *J_host,
                           float *C_final_dev, void *stream)
{
    ade::NvtxRange nvtx_("ade_adjoint");
    if (!c || !C_target_dev || nsteps < 1 || ckpt_every < 1 || !aws)
        return ade::report_error(ADE_ERR_ARG, "bad argument");
    if (c->field) return ade::report_error(ADE_ERR_STATE, "the adjoint is for a uniform velocity (vmax = 0)");
    if (c->catt) return ade::report_error(ADE_ERR_STATE, "the adjoint is for Eq. 1 (tau = 0)");
    const AdjLayout L = adj_layout(c, nsteps, ckpt_every);
    if (aws_bytes < L.total || ((uintptr_t)aws & 255u)) return ade::report_error(ADE_ERR_CAPACITY, "adjoint workspace too small or misaligned");
    const int n = c->n;
    if (n == 0) {
        if (dJdtheta_host) dJdtheta_host[0] = dJdtheta_host[1] = dJdtheta_host[2] = 0.0;
        if (J_host) *J_host = 0.0;
        return ADE_OK;
    }
    const double gamma = c->p.gamma > 0.0 ? c->p.gamma : c->dim + 2.0;
    double vabs = 0.0;
    for (int i = 0; i < c->dim; ++i) vabs += c->p.v[i] * c->p.v[i];
    vabs = sqrt(vabs);
    // the table's shapes are those of 2 (1 - q): 2^3 f (C2) or 2^5 f (C4), undone in the prefactor
    const double pf = c->pf * (c->p.kernel == ADE_WENDLAND_C2 ? 0.125 : 0.03125);
    Adj A;
    A.c = c;
    A.s = (cudaStream_t)stream;
    A.rp = c->rp;
    A.rp.frame = c->w.frame;
    for (int i = 0; i < 3; ++i) A.rp.back[i] = 0u;
    A.rp.ub = 0.f;
    float lo[3];
    auto left = [](double v) { return (float)(v - (double)(float)v); };   // what FP32 leaves of v
    for (int i = 0; i < 3; ++i) {
        const double vh = vabs > 0.0 ? (i < c->dim ? c->p.v[i] / vabs : 0.0) : (i == 0 ? 1.0 : 0.0);
        A.rp.uw[i] = (float)vh;
        lo[i] = left(vh);
    }
    // 1/H in x-axis words, and the part of it that FP32 leaves
    A.sc.vl = make_float4(lo[0], lo[1], lo[2], (float)(c->p.box[0] / kTwo32 / c->H - (double)c->rp.invH));
    A.sc.g2 = (float)(2.0 * gamma);
    A.sc.bT = (float)(2.0 * (gamma - c->dim) + 2.0);
    A.sc.g2l = left(2.0 * gamma);
    A.sc.bTl = left(2.0 * (gamma - c->dim) + 2.0);
    A.sc.syl = (float)(c->p.box[1] / c->p.box[0] - (double)c->rp.sy);
    A.sc.szl = c->dim == 3 ? (float)(c->p.box[2] / c->p.box[0] - (double)c->rp.sz) : 0.f;
    // the passes step by dt rounded to FP32; what that leaves is put into L's coefficients
    const float dt = (float)c->dt;
    const double fit = dt > 0.f ? c->dt / (double)dt : 1.0;
    const double sa = fit * (c->p.alpha_L * vabs + c->p.D_m), sb = fit * (c->p.alpha_T * vabs + c->p.D_m);
    A.ca = (float)(pf * sa);
    A.cb = (float)(pf * sb);
    A.cal = (float)(pf * sa - (double)A.ca);
    A.cbl = (float)(pf * sb - (double)A.cb);
    A.blocks = frozen_blocks(A.rp);
    char *base = static_cast<char *>(aws);
    auto field = [&](size_t o) { return reinterpret_cast<float *>(base + o); };
    const size_t n1 = (size_t)n;
    float *ckpt = field(L.ckpt), *seg = field(L.seg), *h = field(L.h), *p = field(L.p), *hp = field(L.hp), *a = field(L.a);
    double *dots = reinterpret_cast<double *>(base + L.dots);
    double *partials = reinterpret_cast<double *>(base + L.partials);
    A.tab.words = field(L.total);   // what the caller gave beyond the fields
    A.tab.slots = reinterpret_cast<uint4 *>(base + L.slots);
    A.tab.cursor = reinterpret_cast<unsigned long long *>(base + L.cursor);
    const int pencils = A.rp.ncy * A.rp.ncz, numbers = chunk_numbers(n, pencils);
    const bool count = numbers > kCountChunksFrom || 4ll * pencils > numbers;   // (as counts_chunks in api.cu)
    A.tab.dense = count ? reinterpret_cast<uint32_t *>(base + L.dense) : nullptr;
    const size_t kept = std::min(aws_bytes - L.total, (size_t)kTableMaxBytes), lines = kept > 256 ? (kept - 256) / 192 : 0;
    A.tab.low = A.tab.words + lines * 32;      // (a line more than half of the table's: 256 bytes)
    divide_table(c->adj_plan, lines, &A.rp, &A.tab);
    const int nb = (int)A.blocks;
    if (nb > L.blocks) return ade::report_error(ADE_ERR_CAPACITY, "adjoint partials exceed the workspace");
    cudaStream_t s = A.s;
    const uint32_t *perm = c->w.perm;

    // frozen geometry: one cell list at the current positions
    ADJ_CK(cudaMemsetAsync(A.tab.cursor, 0, sizeof(*A.tab.cursor), s));
    const int rc = framed_cells(c, s);
    if (rc) return rc;
    ADJ_CK(launch_chunk_numbers(c->w.cell_start, A.rp, A.tab.dense, s));
    float *U[2] = {field(L.u0), field(L.u1)};   // the running state: U[cur]
    int cur = 0;
    ADJ_CK(table(A, U[0], ckpt));
    // forward: checkpoints every ckpt_every steps, the last segment's states straight into seg
    const int l0_last = (L.nck - 1) * ckpt_every;
    for (int l = 0; l < nsteps; ++l, cur ^= 1) {
        float *keep = nullptr;
        if (l + 1 == nsteps) keep = ckpt + (size_t)L.nck * n1;
        else if (l + 1 > l0_last) keep = seg + (size_t)(l + 1 - l0_last) * n1;
        else if ((l + 1) % ckpt_every == 0) keep = ckpt + (size_t)((l + 1) / ckpt_every) * n1;
        ADJ_CK(fwd_step(A, U[cur], h, U[cur ^ 1], keep, dt));
    }
    cur ^= 1;   // the state before the last step
    // C^N sits in checkpoint slot nck (the last step always writes a slot)
    const float *CN = ckpt + (size_t)L.nck * n1;
    if (C_final_dev) ADJ_CK(launch_pdl(k_adj_scatter, A.blocks, kT, 0, s, perm, A.rp, A.tab, CN, false, C_final_dev));
    // lambda^N = C^N - C*, J = 1/2 |lambda^N|^2
    ADJ_CK(launch_pdl(k_adj_misfit, A.blocks, kT, 0, s, perm, A.rp, A.tab, CN, C_target_dev, p, partials));
    ADJ_CK(launch_pdl(k_adj_fold, 1, kFoldT, 0, s, partials, nb, dots + (size_t)nsteps * kDots));
    // backward, segment by segment
    AdjPass ps;
    memset(&ps, 0, sizeof(ps));
    ps.ca = A.ca;
    ps.cb = A.cb;
    ps.cal = A.cal;
    ps.cbl = A.cbl;
    ps.sc = A.sc;
    for (int sgi = L.nck - 1; sgi >= 0; --sgi) {
        const int l0 = sgi * ckpt_every;
        const int l1 = l0 + ckpt_every < nsteps ? l0 + ckpt_every : nsteps;
        auto state = [&](int l) { return l == l0 ? ckpt + (size_t)sgi * n1 : seg + (size_t)(l - l0) * n1; };
        if (sgi < L.nck - 1) {
            ADJ_CK(launch_pdl(k_adj_double, A.blocks, kT, 0, s, A.rp, A.tab, (const float *)state(l0), U[cur]));
            for (int l = l0; l + 1 < l1; ++l, cur ^= 1) ADJ_CK(fwd_step(A, U[cur], h, U[cur ^ 1], state(l + 1), dt));
        }
        for (int l = l1 - 1; l >= l0; --l, cur ^= 1) {
            // a = L u, b = L p, hp = p + dt/2 b, then lambda^l = p + dt L hp (into p)
            ps.partials = partials + (size_t)(l - l0) * nb * kDots;
            ps.x0 = U[cur];
            ps.x1 = p;
            ps.base = nullptr;
            ps.out0 = a;
            ps.out1 = hp;
            ps.step = 0.5f * dt;
            ADJ_CK(pass(A, BACK1, ps));
            ps.x0 = a;
            ps.x1 = hp;
            ps.base = p;
            ps.out0 = nullptr;
            ps.out1 = p;
            ps.step = dt;
            ps.next = l > l0 ? state(l - 1) : nullptr;
            ps.next2 = U[cur ^ 1];
            ADJ_CK(pass(A, BACK2, ps));
        }
        ADJ_CK(launch_pdl(k_adj_fold, (unsigned)(l1 - l0), kFoldT, 0, s, partials, nb, dots + (size_t)l0 * kDots));
    }
    if (dJdC0_dev) ADJ_CK(launch_pdl(k_adj_scatter, A.blocks, kT, 0, s, perm, A.rp, A.tab, (const float *)p, true, dJdC0_dev));
    std::vector<double> hd(((size_t)nsteps + 1) * kDots);
    ADJ_CK(cudaMemcpyAsync(hd.data(), dots, hd.size() * 8, cudaMemcpyDeviceToHost, s));
    ADJ_CK(cudaStreamSynchronize(s));
    if (J_host) *J_host = 0.5 * hd[(size_t)nsteps * kDots];
    if (dJdtheta_host) {
        // sum_l dt p.(L_k u) + dt^2/2 (p.(L_k a) + b.(L_k u)) of S_L and S_T; a and b hold the factor `fit`
        const double dtd = c->dt, dt2 = c->dt * (double)dt;
        double g[2] = {0.0, 0.0};
        for (int l = 0; l < nsteps; ++l) {
            const double *d = hd.data() + (size_t)l * kDots;
            for (int q = 0; q < 2; ++q) g[q] += dtd * d[q] + 0.5 * dt2 * (d[4 + q] + d[2 + q]);
        }
        dJdtheta_host[0] = pf * vabs * g[0];
        dJdtheta_host[1] = pf * vabs * g[1];
        dJdtheta_host[2] = pf * (g[0] + g[1]);
    }
    return ADE_OK;
}

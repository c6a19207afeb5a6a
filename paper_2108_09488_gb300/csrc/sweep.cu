// sweep.cu -- one plume, many dispersivity sets: Eq. 4-5 for P parameter sets theta_p =
// (alpha_L, alpha_T, D_m)_p that share the particles, the uniform velocity and the time step, each
// with its own concentration field (a parameter sweep or the forward runs of an inversion).
//
// With a uniform v, K = 2D (Eq. 5 with equal tensors) and e = x_ab / r, a pair's weight for the tensor of Eq. 3
// is d_L,p g_L + d_T,p g_T with d_L = alpha_L |v| + D_m, d_T = alpha_T |v| + D_m and, f the kernel shape,
//     g_L = f (2 Gamma u - 2),  g_T = f (-2 Gamma u + 2 (Gamma - d) + 2),  u = (vhat . e)^2,
// so a pair's geometry -- separation, f and u -- is computed once and each parameter set costs a
// multiplication and a fused multiply-add for its weight, the concentration difference and the accumulation.  The cell list, the positions and the drift are
// shared; only the concentrations are per set.  Parameter sets are evaluated in groups of up to 8
// per launch (registers); the sorted concentrations lie in planes of four sets, 16 bytes per particle, so
// that a group's values are one or two 16-byte loads per candidate.
// Summation as in rate.cu: FP32 row sums, Neumaier across rows, fixed order.
//
// Calls of four evaluations and more keep g_L and g_T of every pair in a table (frozen_table.cuh) and stream it
// once per group and evaluation (k_sweep_pass); shorter ones (k_rate_sweep) compute them on the fly, with the
// same operations in the same order, so that a run's bits do not depend on how it is split into calls.  Bound of a pass with 8 sets: the
// latency of L1 and L2 at 27 % occupancy (32 bytes of concentrations a candidate, 96 registers).
// 512^2, 60 neighbours, 8 sets, per evaluation: 90 us on the fly, 66 us from the table.
#include "ade_internal.h"

namespace ade {

namespace {

#include "rate_common.cuh"

#include "rate_walk.cuh"

#include "frozen_table.cuh"

constexpr int kT = kRateThreads;
static_assert(kRateThreads == kFrozenThreads, "the table's launch grid counts blocks of kFrozenThreads");

// Sorted concentrations: planes of four sets, one 16-byte word per particle and plane (`plane` words
// each), so that a warp's loads of neighbouring particles are contiguous (interleaving all sets of a
// particle took twice the L1 wavefronts: 83 us a pass with 8 sets).  p: the group's first plane at word j 0.
template <int NT>
__device__ __forceinline__ void load_group(const float *__restrict__ p, size_t plane, size_t j, float v[NT])
{
    if (NT == 1) {
        v[0] = __ldg(p + 4 * j);
    } else if (NT == 2) {
        const float2 q = __ldg(reinterpret_cast<const float2 *>(p + 4 * j));
        v[0] = q.x;
        v[1 % NT] = q.y;
    } else {
#pragma unroll
        for (int k = 0; k < NT; k += 4) {
            const float4 q = __ldg(reinterpret_cast<const float4 *>(p) + (k / 4) * plane + j);
            v[k] = q.x;
            v[(k + 1) % NT] = q.y;
            v[(k + 2) % NT] = q.z;
            v[(k + 3) % NT] = q.w;
        }
    }
}

template <int NT>
__device__ __forceinline__ void store_group(float *p, size_t plane, size_t j, const float v[NT])
{
    if (NT == 1) {
        p[4 * j] = v[0];
    } else if (NT == 2) {
        *reinterpret_cast<float2 *>(p + 4 * j) = make_float2(v[0], v[1 % NT]);
    } else {
#pragma unroll
        for (int k = 0; k < NT; k += 4)
            reinterpret_cast<float4 *>(p)[(k / 4) * plane + j] = make_float4(v[k], v[(k + 1) % NT], v[(k + 2) % NT], v[(k + 3) % NT]);
    }
}

// The group's first plane, at its first set's word.
__device__ __forceinline__ size_t group_base(int g0, size_t plane) { return (size_t)(g0 >> 2) * plane * 4 + (size_t)(g0 & 3); }

// Sorted concentrations of one particle, C[p n + perm[i]], at words j0 and j1.
__device__ __forceinline__ void gather_sets(const uint32_t *__restrict__ perm, const float *__restrict__ C, size_t n, int P,
                                            int P4, int i, size_t plane, size_t j0, size_t j1, float *__restrict__ Cs)
{
    const uint32_t a = __ldg(perm + i);
    if (a >= (uint32_t)n) return;
    for (int p = 0; p < P4; p += 4) {
        float v[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) v[q] = p + q < P ? __ldg(C + (size_t)(p + q) * n + a) : 0.f;
        store_group<4>(Cs + (size_t)p * plane, plane, j0, v);
        if (j1 != j0) store_group<4>(Cs + (size_t)p * plane, plane, j1, v);
    }
}

__global__ __launch_bounds__(kT) void k_sweep_gather(const uint32_t *__restrict__ perm, const float *__restrict__ C, int n,
                                                     int P, int P4, float *__restrict__ Cs)
{
    pdl_wait();
    pdl_trigger();
    const int i = blockIdx.x * kT + threadIdx.x;
    if (i < n) gather_sets(perm, C, (size_t)n, P, P4, i, (size_t)n, (size_t)i, (size_t)i, Cs);
}

// The table of a call and the concentrations, doubled per pencil.
template <int DIM, int KERNEL, bool ISO>
__global__ __launch_bounds__(kT) void k_sweep_table(const uint4 *__restrict__ P, const uint32_t *__restrict__ cs,
                                                    const uint32_t *__restrict__ perm, const RateParams prm,
                                                    const FrozenTab tab, const ShapeConst sc, const float *__restrict__ C,
                                                    int sets, int P4, float *__restrict__ Cs)
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
    if (i < c.pe) gather_sets(perm, C, (size_t)prm.n, sets, P4, i, 2 * (size_t)prm.n, (size_t)(c.ps + i), (size_t)(c.pe + i), Cs);
    const uint4 pa = __ldg(P + min(i, c.pe - 1));
    build_chunk<DIM, KERNEL, ISO, ISO ? kCutBox : kCutFull, 2>(P, cs, prm, c, pa, srow, tab, sc);
}

// sum_b (d_L g_L + d_T g_T)(C_a - C_b) of NT sets, two sets to a packed FP32x2 instruction.
template <int NT>
struct SetSums {
    static constexpr int N2 = (NT + 1) / 2;
    const float *C;            // doubled, from the group's first set
    size_t plane;
    float2 Ca[N2], rs[N2], acc[N2], comp[N2], dL[N2], dT[N2];
    __device__ __forceinline__ void prefetch(const float *, int, int) const {}
    __device__ __forceinline__ void add(float2 g, const float2 (&Cb)[N2])
    {
        const float2 gl = f2(g.x, g.x), gt = f2(g.y, g.y), m1 = f2(-1.f, -1.f);
#pragma unroll
        for (int k = 0; k < N2; ++k)
            rs[k] = __ffma2_rn(__ffma2_rn(dL[k], gl, __fmul2_rn(dT[k], gt)), __ffma2_rn(Cb[k], m1, Ca[k]), rs[k]);
    }
    __device__ __forceinline__ void load(size_t j, float2 (&v)[N2]) const
    {
        float t[NT];
        load_group<NT>(C, plane, j, t);
#pragma unroll
        for (int k = 0; k < N2; ++k) v[k] = f2(t[2 * k], 2 * k + 1 < NT ? t[(2 * k + 1) % NT] : 0.f);
    }
    template <int M>
    __device__ __forceinline__ void lines(const float *w, int s)
    {
        constexpr int B = NT >= 8 ? 2 : 4;   // candidates in flight (registers)
        float2 g[M];
#pragma unroll
        for (int u = 0; u < M; ++u) g[u] = __ldg(reinterpret_cast<const float2 *>(w) + u * 32);
#pragma unroll
        for (int u0 = 0; u0 < M; u0 += B) {
            float2 v[B][N2];
#pragma unroll
            for (int u = 0; u < B; ++u)
                if (u0 + u < M) load((size_t)(s + u0 + u), v[u]);
#pragma unroll
            for (int u = 0; u < B; ++u)
                if (u0 + u < M) add(g[(u0 + u) % M], v[u]);
        }
    }
    __device__ __forceinline__ void end_row()
    {
#pragma unroll
        for (int k = 0; k < N2; ++k) {
            neumaier_add2(acc[k], comp[k], rs[k]);
            rs[k] = f2(0.f, 0.f);
        }
    }
};

// The same sums over the positions, for a chunk without room in the table.
template <int DIM, int KERNEL, bool ISO, int NT>
__device__ __noinline__ void walk_sets(const uint4 *__restrict__ P, const uint32_t *__restrict__ cs, const RateParams &prm,
                                       const Chunk &c, const ShapeConst &sc, SetSums<NT> &op)
{
    const uint4 pa = __ldg(P + min(c.i0 + (int)(threadIdx.x & 31), c.pe - 1));
    const int ncx = prm.ncx;
    const int cx = (int)__umulhi(pa.x - frame_x(prm), (uint32_t)ncx);
    const int cy = c.p % prm.ncy, cz = c.p / prm.ncy;
    const PairConst kc(prm);
    const PairConst2 k(kc, kc.m1);
    for (int r = 0; r < prm.nrows; ++r) {
        const StencilRow row = prm.rows[r];
        const int q = row_pencil_of<DIM>(row, cy, cz, prm);
        const int qs = (int)__ldg(cs + q * ncx), qe = (int)__ldg(cs + q * ncx + ncx), len = qe - qs;
        int s, cnt;
        cyclic_range(cs, q * ncx, cx - (int)row.w, cx + row.w + 1, ncx, qs, qe, s, cnt);
        for (int t = 0; t < cnt; ++t) {
            int j = s + t;
            j = j >= qe ? j - len : j;
            float2 v[SetSums<NT>::N2];
            op.load((size_t)(qs + j), v);
            op.add(pair_shape<DIM, KERNEL, ISO>(pa, __ldg(P + j), k, sc), v);
        }
        op.end_row();
    }
}

// One evaluation of one group from the table: predictor (C -> Ch) or corrector (C updated), Eq. 8-9.
// out.C set (a call's last corrector): the state goes to the caller's order instead, with the positions
// advanced by prm.inc (the drift of all steps; the first group writes them).
// Eight sets' sums take up to 96 registers, five CTAs per SM; held to 80 they spill, which was a third slower
// at 512^2, and so were two warps of four sets each on a chunk (twice the weights' traffic) and, a little,
// rings of the stream in shared memory (fewer warps).
template <int DIM, int KERNEL, bool ISO, int NT, int EPI>
__global__ __launch_bounds__(kT, 5) void k_sweep_pass(const uint4 *__restrict__ P, const uint32_t *__restrict__ cs,
                                                   const RateParams prm, const FrozenTab tab, const ShapeConst sc,
                                                   const SweepParams sp, float *C, float *Ch,
                                                   const uint32_t *__restrict__ perm, const SweepOut out)
{
    pdl_wait();
    const bool last = EPI == EPI_CORRECT && out.C;
    if (last && blockIdx.x == 0 && threadIdx.x == 0) *tab.cursor = 0ull;   // the next table starts empty
    const int g0 = sp.g0;
    Chunk c;
    uint4 sl;
    if (!my_chunk(tab, prm, c, sl)) return;
    const int i = c.i0 + (threadIdx.x & 31);
    const size_t plane = 2 * (size_t)prm.n, at = (size_t)(c.ps + min(i, c.pe - 1)), gb = group_base(g0, plane);
    SetSums<NT> op;
    op.C = (EPI == EPI_PREDICT ? C : Ch) + gb;
    op.plane = plane;
    op.load(at, op.Ca);
#pragma unroll
    for (int k = 0; k < SetSums<NT>::N2; ++k) {
        op.dL[k] = f2(sp.dL[2 * k], sp.dL[2 * k + 1]);
        op.dT[k] = f2(sp.dT[2 * k], sp.dT[2 * k + 1]);
        op.rs[k] = op.acc[k] = op.comp[k] = f2(0.f, 0.f);
    }
    if (sl.x != kNoRoom) stream_rows<2>(sl, tab, op);
    else walk_sets<DIM, KERNEL, ISO, NT>(P, cs, prm, c, sc, op);
    if (i >= c.pe) return;
    const float pf = prm.pf * shape_unscale<KERNEL>();
    float Cl[NT], o[NT];
    if (EPI == EPI_CORRECT) load_group<NT>(C + gb, plane, at, Cl);
#pragma unroll
    for (int k = 0; k < NT; ++k) {
        const float2 a2 = op.acc[k / 2], c2 = op.comp[k / 2], ca = op.Ca[k / 2];
        const float rate = pf * (k & 1 ? a2.y + c2.y : a2.x + c2.x);
        o[k] = fmaf(prm.dt, rate, EPI == EPI_CORRECT ? Cl[k] : (k & 1 ? ca.y : ca.x));
    }
    if (last) {
        const uint32_t a = __ldg(perm + i);
        const size_t n = (size_t)prm.n;
        if (a >= (uint32_t)n) return;
        bool bad = false;
#pragma unroll
        for (int k = 0; k < NT; ++k) {
            out.C[(size_t)(g0 + k) * n + a] = o[k];
            bad |= !isfinite(o[k]);
        }
        if (bad) atomicOr(out.status, 1);
        if (g0 == 0) {
            const uint4 q = __ldg(P + i);
            out.xq[a] = q.x + prm.inc[0];
            out.xq[n + a] = q.y + prm.inc[1];
            if (DIM == 3) out.xq[2 * n + a] = q.z + prm.inc[2];
        }
        return;
    }
    float *to = (EPI == EPI_PREDICT ? Ch : C) + gb;
    store_group<NT>(to, plane, at, o);
    store_group<NT>(to, plane, (size_t)(c.pe + i), o);
}

// One evaluation with the geometry computed on the fly: the rate or pair count, or a predictor (Ce -> out.Cout)
// or corrector (caller order) of a call too short for the table.  Pe: the positions of the build.
template <int DIM, int KERNEL, int EPI, int NT, bool COUNT>
__global__ __launch_bounds__(kT) void k_rate_sweep(const uint4 *__restrict__ Pe, const float *__restrict__ Ce,
                                                   const uint32_t *__restrict__ cs,
                                                   const uint32_t *__restrict__ perm, const RateParams prm,
                                                   const SweepParams sp, const SweepOut out)
{
    const int i = blockIdx.x * kT + threadIdx.x;
    const bool valid = i < prm.n;
    const int ii = valid ? i : prm.n - 1;
    const uint4 pa = __ldg(Pe + ii);
    const int g0 = sp.g0;
    const float *Cg = Ce + group_base(g0, (size_t)prm.n);
    float Ca[NT];
    load_group<NT>(Cg, (size_t)prm.n, (size_t)ii, Ca);
    const int ncx = prm.ncx, ncy = prm.ncy, ncz = prm.ncz;
    // cell of the build: position minus the drift since it, in the build's frame
    uint3 org = make_uint3(prm.back[0], prm.back[1], prm.back[2]);
    if (prm.frame) {
        org.x += __ldg(prm.frame + 4);
        org.y += __ldg(prm.frame + 5);
        org.z += __ldg(prm.frame + 6);
    }
    const int cx = (int)__umulhi(pa.x - org.x, (uint32_t)ncx);
    const int cy = (int)__umulhi(pa.y - org.y, (uint32_t)ncy);
    const int cz = DIM == 3 ? (int)__umulhi(pa.z - org.z, (uint32_t)ncz) : 0;
    const float far2 = prm.H2 * (1.f + 1.f / 4096.f), invH = prm.invH, sy = prm.sy, sz = prm.sz;   // far2: as chunk_rows
    const float vx = sp.vh[0], vy = sp.vh[1], vz = sp.vh[2], g2 = sp.g2, bT = sp.bT;
    float acc[NT], comp[NT];
#pragma unroll
    for (int k = 0; k < NT; ++k) acc[k] = comp[k] = 0.f;
    unsigned cnt = 0u;
    for (int ri = 0; ri < prm.nrows; ++ri) {
        const StencilRow row = prm.rows[ri];
        int yy = cy + row.dy;
        yy += (yy < 0) ? ncy : 0;
        yy -= (yy >= ncy) ? ncy : 0;
        int zz = 0;
        if (DIM == 3) {
            zz = cz + row.dz;
            zz += (zz < 0) ? ncz : 0;
            zz -= (zz >= ncz) ? ncz : 0;
        }
        const int base = (zz * ncy + yy) * ncx;
        const int lo = cx - row.w, hi = cx + row.w + 1;
        int r0[2], r1[2];
        if (lo < 0) {
            r0[0] = __ldg(cs + base + lo + ncx);
            r1[0] = __ldg(cs + base + ncx);
            r0[1] = __ldg(cs + base);
            r1[1] = __ldg(cs + base + hi);
        } else if (hi > ncx) {
            r0[0] = __ldg(cs + base + lo);
            r1[0] = __ldg(cs + base + ncx);
            r0[1] = __ldg(cs + base);
            r1[1] = __ldg(cs + base + hi - ncx);
        } else {
            r0[0] = __ldg(cs + base + lo);
            r1[0] = __ldg(cs + base + hi);
            r0[1] = r1[1] = 0;
        }
        float rs[NT];
#pragma unroll
        for (int k = 0; k < NT; ++k) rs[k] = 0.f;
        for (int piece = 0; piece < 2; ++piece)
#pragma unroll 4
            for (int j = r0[piece]; j < r1[piece]; ++j) {
                const uint4 pb = __ldg(Pe + j);
                const int ix = (int)(pa.x - pb.x), iy = (int)(pa.y - pb.y), iz = (int)(pa.z - pb.z);
                if (COUNT) {
                    const double dxd = (double)ix * prm.u[0], dyd = (double)iy * prm.u[1];
                    double r2d = __dadd_rn(__dmul_rn(dxd, dxd), __dmul_rn(dyd, dyd));
                    if (DIM == 3) {
                        const double dzd = (double)iz * prm.u[2];
                        r2d = __dadd_rn(r2d, __dmul_rn(dzd, dzd));
                    }
                    cnt += (r2d > 0.0 && r2d < prm.H2d) ? 1u : 0u;
                }
                const float dx = (float)ix;
                const float dy = (float)iy * sy;
                const float dz = DIM == 3 ? (float)iz * sz : 0.f;
                float r2 = fmaf(dx, dx, dy * dy);
                if (DIM == 3) r2 = fmaf(dz, dz, r2);
                if (r2 < far2 && r2 > 0.f) {
                    // the operations of pair_shape and SetSums::add, so that a step has the same bits here and
                    // from the table; a candidate between H and far2 has f = 0
                    const float rinv = rsqrt_ftz(r2);
                    const float om = fmaf(-(r2 * rinv), invH, 1.f);
                    const float f = shape2x<KERNEL>(fmaxf(om + om, 0.f));
                    float c = fmaf(vx, dx, vy * dy);
                    if (DIM == 3) c = fmaf(vz, dz, c);
                    const float t = c * rinv;
                    const float u = fminf(t * t, 1.f);
                    const float gL = f * fmaf(g2, u, -2.f), gT = f * fmaf(-g2, u, bT);
                    float Cb[NT];
                    load_group<NT>(Cg, (size_t)prm.n, (size_t)j, Cb);
#pragma unroll
                    for (int k = 0; k < NT; ++k) rs[k] = fmaf(fmaf(sp.dL[k], gL, sp.dT[k] * gT), Ca[k] - Cb[k], rs[k]);
                }
            }
#pragma unroll
        for (int k = 0; k < NT; ++k) neumaier_add(acc[k], comp[k], rs[k]);
    }
    if (COUNT) {
        unsigned c = valid ? cnt : 0u;
        for (int o = 16; o > 0; o >>= 1) c += __shfl_down_sync(0xffffffffu, c, o);
        if ((threadIdx.x & 31) == 0 && c) atomicAdd(out.pairs, (unsigned long long)c);
    }
    if (!valid) return;
    float rate[NT];
#pragma unroll
    for (int k = 0; k < NT; ++k) rate[k] = (prm.pf * shape_unscale<KERNEL>()) * (acc[k] + comp[k]);
    const size_t n = (size_t)prm.n;
    if (EPI == EPI_PREDICT) {
        float o[NT];
#pragma unroll
        for (int k = 0; k < NT; ++k) o[k] = fmaf(prm.dt, rate[k], Ca[k]);
        store_group<NT>(out.Cout + group_base(g0, n), n, (size_t)i, o);
        return;
    }
    const uint32_t a = __ldg(perm + i);
    if (a >= (uint32_t)n) return;
    if (EPI == EPI_RATE) {
        if (out.rate)
#pragma unroll
            for (int k = 0; k < NT; ++k) out.rate[(size_t)(g0 + k) * n + a] = rate[k];
        return;
    }
    bool bad = false;
#pragma unroll
    for (int k = 0; k < NT; ++k) {
        float *Cp = out.C + (size_t)(g0 + k) * n + a;
        const float Cn = fmaf(prm.dt, rate[k], *Cp);
        *Cp = Cn;
        bad |= !isfinite(Cn);
    }
    if (bad) atomicOr(out.status, 1);
    if (g0 == 0) {
        out.xq[a] = pa.x + prm.inc[0];
        out.xq[n + a] = pa.y + prm.inc[1];
        if (DIM == 3) out.xq[2 * n + a] = pa.z + prm.inc[2];
    }
}

template <int DIM, int KERNEL, int NT>
void launch_sweep_nt(int epi, bool count, int blocks, const uint4 *Pe, const float *Ce, const uint32_t *cs,
                     const uint32_t *perm, const RateParams &prm, const SweepParams &sp, const SweepOut &out,
                     cudaStream_t s)
{
    if (count)
        k_rate_sweep<DIM, KERNEL, EPI_RATE, NT, true><<<blocks, kT, 0, s>>>(Pe, Ce, cs, perm, prm, sp, out);
    else if (epi == EPI_RATE)
        k_rate_sweep<DIM, KERNEL, EPI_RATE, NT, false><<<blocks, kT, 0, s>>>(Pe, Ce, cs, perm, prm, sp, out);
    else if (epi == EPI_PREDICT)
        k_rate_sweep<DIM, KERNEL, EPI_PREDICT, NT, false><<<blocks, kT, 0, s>>>(Pe, Ce, cs, perm, prm, sp, out);
    else
        k_rate_sweep<DIM, KERNEL, EPI_CORRECT, NT, false><<<blocks, kT, 0, s>>>(Pe, Ce, cs, perm, prm, sp, out);
}

template <int DIM, int KERNEL>
void launch_sweep_k(int epi, bool count, int blocks, const uint4 *Pe, const float *Ce, const uint32_t *cs,
                    const uint32_t *perm, const RateParams &prm, const SweepParams &sp, const SweepOut &out,
                    cudaStream_t s)
{
    switch (sp.nt) {
    case 1: launch_sweep_nt<DIM, KERNEL, 1>(epi, count, blocks, Pe, Ce, cs, perm, prm, sp, out, s); break;
    case 2: launch_sweep_nt<DIM, KERNEL, 2>(epi, count, blocks, Pe, Ce, cs, perm, prm, sp, out, s); break;
    case 4: launch_sweep_nt<DIM, KERNEL, 4>(epi, count, blocks, Pe, Ce, cs, perm, prm, sp, out, s); break;
    default: launch_sweep_nt<DIM, KERNEL, 8>(epi, count, blocks, Pe, Ce, cs, perm, prm, sp, out, s); break;
    }
}

template <int DIM, int KERNEL, bool ISO, int NT>
cudaError_t pass_nt(const SweepRun &r, int epi, const SweepParams &sp, const RateParams &prm, const SweepOut &out, cudaStream_t s)
{
    const unsigned g = frozen_blocks(prm);
    return epi == EPI_PREDICT
               ? launch_pdl(k_sweep_pass<DIM, KERNEL, ISO, NT, EPI_PREDICT>, g, kT, 0, s, r.P, r.cs, prm, r.tab, ShapeConst{float4{}, r.g2, r.bT, 0.f, 0.f, 0.f, 0.f}, sp, r.C, r.Ch, r.perm, out)
               : launch_pdl(k_sweep_pass<DIM, KERNEL, ISO, NT, EPI_CORRECT>, g, kT, 0, s, r.P, r.cs, prm, r.tab, ShapeConst{float4{}, r.g2, r.bT, 0.f, 0.f, 0.f, 0.f}, sp, r.C, r.Ch, r.perm, out);
}

template <int DIM, int KERNEL, bool ISO>
cudaError_t pass_k(const SweepRun &r, int epi, const SweepParams &sp, const RateParams &prm, const SweepOut &out, cudaStream_t s)
{
    switch (sp.nt) {
    case 1: return pass_nt<DIM, KERNEL, ISO, 1>(r, epi, sp, prm, out, s);
    case 2: return pass_nt<DIM, KERNEL, ISO, 2>(r, epi, sp, prm, out, s);
    case 4: return pass_nt<DIM, KERNEL, ISO, 4>(r, epi, sp, prm, out, s);
    default: return pass_nt<DIM, KERNEL, ISO, 8>(r, epi, sp, prm, out, s);
    }
}

template <int DIM, int KERNEL, bool ISO>
cudaError_t table_k(const SweepRun &r, const RateParams &prm, const float *C, int sets, int P4, cudaStream_t s)
{
    return launch_pdl(k_sweep_table<DIM, KERNEL, ISO>, frozen_blocks(prm), kT, 0, s, r.P, r.cs, r.perm, prm, r.tab,
                      ShapeConst{float4{}, r.g2, r.bT, 0.f, 0.f, 0.f, 0.f}, C, sets, P4, r.C);
}

#define ADE_SWEEP_CALL(F, ...)                                                                                               \
    (dim == 2 ? (kernel == ADE_WENDLAND_C2                                                                                   \
                     ? (iso ? F<2, ADE_WENDLAND_C2, true>(__VA_ARGS__) : F<2, ADE_WENDLAND_C2, false>(__VA_ARGS__))          \
                     : (iso ? F<2, ADE_WENDLAND_C4, true>(__VA_ARGS__) : F<2, ADE_WENDLAND_C4, false>(__VA_ARGS__)))         \
              : (kernel == ADE_WENDLAND_C2                                                                                   \
                     ? (iso ? F<3, ADE_WENDLAND_C2, true>(__VA_ARGS__) : F<3, ADE_WENDLAND_C2, false>(__VA_ARGS__))          \
                     : (iso ? F<3, ADE_WENDLAND_C4, true>(__VA_ARGS__) : F<3, ADE_WENDLAND_C4, false>(__VA_ARGS__))))

}  // namespace

cudaError_t launch_sweep_gather(const uint32_t *perm, const float *C, int n, int P, int P4, float *Cs, cudaStream_t s)
{
    if (n == 0) return cudaSuccess;
    return launch_pdl(k_sweep_gather, (unsigned)((n + kT - 1) / kT), kT, 0, s, perm, C, n, P, P4, Cs);
}

cudaError_t launch_sweep_table(int dim, int kernel, bool iso, const SweepRun &r, const RateParams &prm, const float *C,
                               int sets, int P4, cudaStream_t s)
{
    const cudaError_t e = launch_chunk_numbers(r.cs, prm, r.tab.dense, s);
    if (e != cudaSuccess) return e;
    return ADE_SWEEP_CALL(table_k, r, prm, C, sets, P4, s);
}

cudaError_t launch_sweep_pass(int dim, int kernel, bool iso, int epi, const SweepRun &r, const SweepParams &sp,
                              const RateParams &prm, const SweepOut &out, cudaStream_t s)
{
    if (sp.nt != 1 && sp.nt != 2 && sp.nt != 4 && sp.nt != 8) return cudaErrorInvalidValue;
    return ADE_SWEEP_CALL(pass_k, r, epi, sp, prm, out, s);
}

cudaError_t launch_rate_sweep(int dim, int kernel, int epi, bool count, const uint4 *Pe, const float *Ce,
                              const uint32_t *cell_start, const uint32_t *perm, const RateParams &prm,
                              const SweepParams &sp, const SweepOut &out, cudaStream_t s)
{
    if (prm.n == 0) return cudaSuccess;
    if (sp.nt != 1 && sp.nt != 2 && sp.nt != 4 && sp.nt != 8) return cudaErrorInvalidValue;
    const int blocks = (prm.n + kT - 1) / kT;
    if (dim == 2) {
        if (kernel == ADE_WENDLAND_C2)
            launch_sweep_k<2, ADE_WENDLAND_C2>(epi, count, blocks, Pe, Ce, cell_start, perm, prm, sp, out, s);
        else
            launch_sweep_k<2, ADE_WENDLAND_C4>(epi, count, blocks, Pe, Ce, cell_start, perm, prm, sp, out, s);
    } else {
        if (kernel == ADE_WENDLAND_C2)
            launch_sweep_k<3, ADE_WENDLAND_C2>(epi, count, blocks, Pe, Ce, cell_start, perm, prm, sp, out, s);
        else
            launch_sweep_k<3, ADE_WENDLAND_C4>(epi, count, blocks, Pe, Ce, cell_start, perm, prm, sp, out, s);
    }
    return cudaGetLastError();
}

}  // namespace ade

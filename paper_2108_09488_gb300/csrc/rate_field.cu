// rate_field.cu -- Eq. 4-5 with a per-particle velocity field (heterogeneous flow), and the
// per-particle drift of the predictor-corrector (Eq. 8-9).
//
// Each particle carries its own constant velocity v_a (Eq. 1) and hence its own dispersion
// tensor D_a (Eq. 3).  For one ordered pair, in the notation of Eq. 4-5:
//   K_ij  = 4 D_ij,a D_ij,b / (D_ij,a + D_ij,b)     (0 where the denominator is 0),
//   Dcal  = Gamma x^T K x / r^2 - tr K,
//   disp  = 1/2 (m/rho) Dcal (C_a - C_b) W'(r)/r,
//   conv  = C_a (m/rho) (v_a - v_b) . x_ab W'(r)/r,      (grad_a W = W'(r) x_ab / r)
// with W'(r)/r = kc f(q) as in rate.cu.  Particles drift with their own velocities, so relative
// positions change during a step: the cell list is built for the radius H + dt vmax (the skin
// covers the relative drift up to the half step, |v_a - v_b| dt/2 <= dt vmax) while the support
// test uses H.  Each cell-sorted particle's candidates are those of the stencil rows of its
// build-time cell, cut to the chord its own position leaves; the sums of both terms over a row (2D) or
// a list (3D) are added with Neumaier compensation in a fixed order, so results are deterministic.
// Records of v and D are formed once per field in the caller's order (v is constant in time) and
// permuted into the cell-sorted order after every cell build (k_field_permute), so the pair
// loop's loads stay contiguous: candidates of a row are consecutive sorted indices.
//
// Conditioning of Eq. 5.  Diagonal components of D (Eq. 3) are never negative, but off-diagonal
// ones take the sign of v_i v_j, so for neighbours whose velocities point into different quadrants
// D_ij,a + D_ij,b can cancel and K_ij = 4 D_ij,a D_ij,b / (D_ij,a + D_ij,b) is then arbitrarily
// large and sensitive to the rounding of D.  D is therefore computed in FP64 per particle and
// each off-diagonal component is kept as an unevaluated FP32 pair hi + lo (lo = the FP64 value
// minus hi); the pair's denominator is (hi_a + hi_b) + (lo_a + lo_b), whose first sum is exact when
// the two cancel (Sterbenz), so K_ij keeps FP32 relative accuracy.  The lo words ride in the
// otherwise unused fourth lanes of the float4 records, so the pair loop loads nothing extra.
#include <algorithm>

#include "ade_internal.h"

namespace ade {

namespace {

#include "rate_common.cuh"

#include "rate_walk.cuh"

#include "frozen_table.cuh"

constexpr int kT = kRateThreads;

// Approximate reciprocal (MUFU, about 1 ulp; subnormal input and output flushed to zero).
__device__ __forceinline__ float rcp_approx(float x)
{
    float r;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
}

// Harmonic-mean component of Eq. 5 for a diagonal entry, with a4 = 4 a precomputed per particle.
// a, b >= 0, so a + b = 0 only when 4ab = 0 too: clamping the denominator to the smallest normal
// number returns K = 0 there without a branch.
__device__ __forceinline__ float hmean_diag(float a, float a4, float b)
{
    return (a4 * b) * rcp_approx(fmaxf(a + b, 1.17549435e-38f));
}

// Twice an off-diagonal component, 2 K_ij, from hi + lo pairs (see the conditioning note above),
// with a8 = 8 a_hi precomputed per particle.  A zero denominator gives K_ij = 0 as in Eq. 5's
// convention; denominators below the smallest normal number count as zero.
__device__ __forceinline__ float hmean_off2(float ah, float a8, float al, float bh, float bl)
{
    const float den = (ah + bh) + (al + bl);
    const float k2 = (a8 * bh) * rcp_approx(den);
    return fabsf(den) >= 1.17549435e-38f ? k2 : 0.f;
}

// Fixed-point drift of one particle read from its Inc record: half step, or full step 2h + c.
__device__ __forceinline__ void half_drift(const uint4 &ic, uint32_t out[3])
{
    out[0] = ic.x;
    out[1] = ic.y;
    out[2] = ic.z;
}

__device__ __forceinline__ void full_drift(const uint4 &ic, uint32_t out[3])
{
    out[0] = 2u * ic.x + ((ic.w & 3u) - 1u);
    out[1] = 2u * ic.y + (((ic.w >> 2) & 3u) - 1u);
    out[2] = 2u * ic.z + (((ic.w >> 4) & 3u) - 1u);
}

// Velocities of the caller's field into the caller-order records (fourth lane cleared) and
// max_a |v_a| as FP32 bits (non-negative floats order like their bit patterns); a non-finite speed
// counts as +inf so that the host check rejects it.
template <int DIM>
__global__ __launch_bounds__(kT) void k_field_velocity(const float *__restrict__ v, int n, float4 *__restrict__ Vc,
                                                       unsigned *__restrict__ out_bits)
{
    const int i = blockIdx.x * kT + threadIdx.x;
    float s = 0.f;
    if (i < n) {
        const float a = v[i], b = v[(size_t)n + i], c = DIM == 3 ? v[2 * (size_t)n + i] : 0.f;
        Vc[i] = make_float4(a, b, c, 0.f);
        s = sqrtf(a * a + b * b + c * c);
        if (!(s <= 3.0e38f)) s = __int_as_float(0x7f800000);
    }
    for (int o = 16; o > 0; o >>= 1) s = fmaxf(s, __shfl_down_sync(0xffffffffu, s, o));
    if ((threadIdx.x & 31) == 0) atomicMax(out_bits, __float_as_uint(s));
}

// Dispersion tensor (Eq. 3) of every particle in FP64 from its velocity, and its fixed-point
// drift per half and full step, stored as the records described in ade_internal.h (caller order).
template <int DIM>
__global__ __launch_bounds__(kT) void k_field_tensors(int n, FieldParams fp, float4 *__restrict__ Vc,
                                                      float4 *__restrict__ DAc, float4 *__restrict__ DBc,
                                                      uint4 *__restrict__ IncC)
{
    const int i = blockIdx.x * kT + threadIdx.x;
    if (i >= n) return;
    const float4 vr = Vc[i];
    const double vv[3] = {vr.x, vr.y, DIM == 3 ? (double)vr.z : 0.0};
    uint32_t h[3], cbits = 0u;
    for (int k = 0; k < 3; ++k) {
        const long long hk = __double2ll_rn(vv[k] * (0.5 * fp.vscale[k]));
        const long long fk = __double2ll_rn(vv[k] * fp.vscale[k]);
        h[k] = (uint32_t)(unsigned long long)hk;
        cbits |= (uint32_t)(fk - 2 * hk + 1) << (2 * k);
    }
    IncC[i] = make_uint4(h[0], h[1], h[2], cbits);
    const double s = sqrt(vv[0] * vv[0] + vv[1] * vv[1] + vv[2] * vv[2]);
    const double iso = fp.aT * s + fp.Dm;
    const double g = s > 0.0 ? (fp.aL - fp.aT) / s : 0.0;
    auto hi = [](double d) { return (float)d; };
    auto lo = [](double d) { return (float)(d - (double)(float)d); };
    const double dxx = iso + g * (vv[0] * vv[0]), dxy = g * (vv[0] * vv[1]), dyy = iso + g * (vv[1] * vv[1]);
    if (DIM == 2) {
        DAc[i] = make_float4(hi(dxx), hi(dxy), hi(dyy), lo(dxy));
    } else {
        const double dxz = g * (vv[0] * vv[2]), dyz = g * (vv[1] * vv[2]), dzz = iso + g * (vv[2] * vv[2]);
        Vc[i].w = lo(dxz);
        DAc[i] = make_float4(hi(dxx), hi(dxy), hi(dxz), lo(dxy));
        DBc[i] = make_float4(hi(dyy), hi(dyz), hi(dzz), lo(dyz));
    }
}

// Sorted records after a cell build.
template <int DIM>
__global__ __launch_bounds__(kT) void k_field_permute(const uint32_t *__restrict__ perm, int n,
                                                      const float4 *__restrict__ Vc, const float4 *__restrict__ DAc,
                                                      const float4 *__restrict__ DBc, const uint4 *__restrict__ IncC,
                                                      float4 *__restrict__ V, float4 *__restrict__ DA,
                                                      float4 *__restrict__ DB, uint4 *__restrict__ Inc)
{
    pdl_wait();
    pdl_trigger();
    const int i = blockIdx.x * kT + threadIdx.x;
    if (i >= n) return;
    const uint32_t a = __ldg(perm + i);
    V[i] = __ldg(Vc + a);
    DA[i] = __ldg(DAc + a);
    if (DIM == 3) DB[i] = __ldg(DBc + a);
    Inc[i] = __ldg(IncC + a);
}

// Ordered in-support pairs (FP64 test), one thread per sorted particle over the full stencil.
template <int DIM>
__global__ __launch_bounds__(kT) void k_count_field(const uint4 *__restrict__ Pe, const uint32_t *__restrict__ cs,
                                                    const RateParams prm, const EpiOut out)
{
    pdl_wait();
    const int i = blockIdx.x * kT + threadIdx.x;
    const bool valid = i < prm.n;
    const uint4 pa = __ldg(Pe + (valid ? i : prm.n - 1));
    const int ncx = prm.ncx, ncy = prm.ncy, ncz = prm.ncz;
    const int cx = (int)__umulhi(pa.x, (uint32_t)ncx);
    const int cy = (int)__umulhi(pa.y, (uint32_t)ncy);
    const int cz = DIM == 3 ? (int)__umulhi(pa.z, (uint32_t)ncz) : 0;
    unsigned cnt = 0u;
    for (int ri = 0; ri < prm.nrows; ++ri) {
        const StencilRow row = prm.rows[ri];
        const int q = row_pencil_of<DIM>(row, cy, cz, prm);
        int s0, e0, s1, e1;
        row_ranges(cs, q * ncx, cx - (int)row.w, cx + row.w + 1, ncx, s0, e0, s1, e1);
        for (int piece = 0; piece < 2; ++piece)
            for (int j = piece ? s1 : s0; j < (piece ? e1 : e0); ++j) {
                const uint4 pb = __ldg(Pe + j);
                cnt += in_support_fp64<DIM>((int)(pa.x - pb.x), (int)(pa.y - pb.y), (int)(pa.z - pb.z), prm);
            }
    }
    Acc acc{0.f, 0.f, 0.f, 0.f, valid ? cnt : 0u};
    warp_finish<EPI_RATE, true, kT>(acc, out);
}

// 3D: one target's own records for the pair terms.
struct FieldTarget {
    uint4 p;
    float4 v, da, db, da4, db4;
    float Ca;
    __device__ __forceinline__ FieldTarget(const uint4 &p_, float Ca_, const float4 &v_, const float4 &da_, const float4 &db_)
        : p(p_), v(v_), da(da_), db(db_), Ca(Ca_)
    {
        // 4 D (diagonal) and 8 D (off-diagonal) for the harmonic means
        da4 = make_float4(4.f * da.x, 8.f * da.y, 8.f * da.z, 0.f);
        db4 = make_float4(4.f * db.x, 8.f * db.y, 4.f * db.z, 0.f);
    }
};

__device__ __forceinline__ float field_sep(const FieldTarget &t, const uint4 &pb, const PairConst &k, float &dx, float &dy,
                                           float &dz)
{
    dx = sep(t.p.x, pb.x, k.m1);
    dy = sep(t.p.y, pb.y, k.m1) * k.sy;
    dz = sep(t.p.z, pb.z, k.m1) * k.sz;
    return fmaf(dz, dz, fmaf(dx, dx, dy * dy));
}

// Both terms of Eq. 4 for an in-support candidate j.
template <int KERNEL>
__device__ __forceinline__ void field_pair(const FieldTarget &t, const uint4 *__restrict__ Pe, const float4 *__restrict__ V,
                                           const float4 *__restrict__ DA, const float4 *__restrict__ DB, unsigned j,
                                           const PairConst &k, float gam, float &rd, float &rc)
{
    const uint4 pb = __ldg(Pe + j);
    const float4 vb = __ldg(V + j), d1 = __ldg(DA + j);
    float dx, dy, dz;
    const float r2 = field_sep(t, pb, k, dx, dy, dz);
    const float rinv = rsqrt_ftz(r2);
    const float f = shape<KERNEL>(fmaf(-(r2 * rinv), k.invH, 1.f));
    const float kxx = hmean_diag(t.da.x, t.da4.x, d1.x), kxy2 = hmean_off2(t.da.y, t.da4.y, t.da.w, d1.y, d1.w);
    const float4 d2 = __ldg(DB + j);
    const float kxz2 = hmean_off2(t.da.z, t.da4.z, t.v.w, d1.z, vb.w);
    const float kyy = hmean_diag(t.db.x, t.db4.x, d2.x);
    const float kyz2 = hmean_off2(t.db.y, t.db4.y, t.db.w, d2.y, d2.w);
    const float kzz = hmean_diag(t.db.z, t.db4.z, d2.z);
    const float qx = fmaf(kxx, dx, fmaf(kxy2, dy, kxz2 * dz));
    const float qy = fmaf(kyy, dy, kyz2 * dz);
    const float Q = fmaf(dx, qx, fmaf(dy, qy, kzz * dz * dz));
    const float tr = kxx + kyy + kzz;
    const float s = fmaf(gam * Q, rinv * rinv, -tr);
    rd = fmaf(f * s, t.Ca - __uint_as_float(pb.w), rd);
    const float dvx = fmaf(t.v.z - vb.z, dz, fmaf(t.v.x - vb.x, dx, (t.v.y - vb.y) * dy));
    rc = fmaf(f, dvx, rc);
}

// 2D: one thread per sorted particle.  Its range of a row is cut to the chord its own position leaves at the
// row's cell band, for the grid's radius H + dt vmax (positions of the build), and nearly all that is left
// is in support for some lane, so every candidate is evaluated, without a branch, and the sums of those
// out of support (or at zero separation) are dropped: the loads of several candidates are in flight at
// once.  Bound: instruction issue.  Per step at 1024^2, 120 neighbours: full rows and a branch 922 us, cut
// rows 891, no branch 889 (unrolled 2: 844, 4: 814, 8: 802; 4 in 48 registers 852); 512^2, 60 neighbours
// 201 -> 161; 256^2, 28 neighbours 84 -> 59; 300^2 jittered 122 -> 88.  (Rows hold ten and more candidates:
// the lists of the 3D kernel cost more than the lanes they keep busy.)
template <int KERNEL, int EPI>
__global__ __launch_bounds__(kT) void k_rate_field2(const uint4 *__restrict__ Pe, const uint32_t *__restrict__ cs,
                                                   const uint32_t *__restrict__ perm,
                                                   const float4 *__restrict__ V, const float4 *__restrict__ DA,
                                                   const uint4 *__restrict__ Inc, const RateParams prm, const FieldParams fp, const EpiOut out)
{
    pdl_wait();   // no early trigger: see pdl_trigger
    const int i = blockIdx.x * kT + threadIdx.x;
    const bool valid = i < prm.n;
    const int ii = valid ? i : prm.n - 1;
    const uint4 pa = __ldg(Pe + ii);
    const float4 va = __ldg(V + ii);
    const float4 da = __ldg(DA + ii);
    // fixed-point drift of this particle; the cell of the cell build is the evaluation position
    // minus the drift since the build (the half step, in the corrector)
    const uint4 ic = EPI == EPI_RATE ? make_uint4(0u, 0u, 0u, 0u) : __ldg(Inc + ii);
    uint32_t back[3] = {0u, 0u, 0u};
    if (EPI == EPI_CORRECT) half_drift(ic, back);
    const int ncx = prm.ncx, ncy = prm.ncy;
    const int cx = (int)__umulhi(pa.x - back[0], (uint32_t)ncx);
    const int cy = (int)__umulhi(pa.y - back[1], (uint32_t)ncy);
    const float inv32 = 2.3283064365386963e-10f;   // 2^-32
    const float fx = (float)((pa.x - back[0]) * (uint32_t)ncx) * inv32, fy = (float)((pa.y - back[1]) * (uint32_t)ncy) * inv32;
    TrimGeom g(prm);
    g.Hm2 = prm.Hg2 * (1.f + 1.f / 2048.f);
    const float Ca = __uint_as_float(pa.w);
    const float H2 = prm.H2, invH = prm.invH, sy = prm.sy, gam = fp.gamma;
    // 4 D (diagonal) and 8 D (off-diagonal) of this particle for the harmonic means
    const float4 da4 = make_float4(4.f * da.x, 8.f * da.y, 4.f * da.z, 0.f);
    float sd = 0.f, cd = 0.f, sc = 0.f, cc = 0.f;
    for (int ri = 0; ri < prm.nrows; ++ri) {
        const StencilRow row = prm.rows[ri];
        const TrimRow tr{(float)row.dy, 0.f, 0, 0};
        const float d2 = g.Hm2 - row_gap2<2>(make_float4(0.f, 1.f, 0.f, 0.f), tr, fy, fy, 0.f, 0.f, 0.f, 0.f, g);
        if (!(d2 > 0.f)) continue;
        const float xe = fmaf(d2 * rsqrt_ftz(d2), g.inv_wx, 1.f / 4096.f);
        int yy = cy + row.dy;
        yy += (yy < 0) ? ncy : 0;
        yy -= (yy >= ncy) ? ncy : 0;
        const int base = yy * ncx;
        const int lo = cx + max(__float2int_rd(fx - xe), -(int)row.w), hi = cx + min(__float2int_rd(fx + xe), (int)row.w) + 1;
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
        float rd = 0.f, rc = 0.f;
        for (int piece = 0; piece < 2; ++piece)
#pragma unroll 8
            for (int j = r0[piece]; j < r1[piece]; ++j) {
                const uint4 pb = __ldg(Pe + j);
                const float4 vb = __ldg(V + j);
                const float4 d1 = __ldg(DA + j);
                const int ix = (int)(pa.x - pb.x), iy = (int)(pa.y - pb.y);
                const float dx = (float)ix;
                const float dy = (float)iy * sy;
                const float r2 = fmaf(dx, dx, dy * dy);
                const bool in = r2 < H2 && r2 > 0.f;
                const float rinv = rsqrt_ftz(r2);
                const float f = shape<KERNEL>(fmaf(-(r2 * rinv), invH, 1.f));
                const float kxx = hmean_diag(da.x, da4.x, d1.x);
                const float kxy2 = hmean_off2(da.y, da4.y, da.w, d1.y, d1.w);
                const float kyy = hmean_diag(da.z, da4.z, d1.z);
                const float Q = fmaf(dx, fmaf(kxx, dx, kxy2 * dy), kyy * dy * dy);
                const float s = fmaf(gam * Q, rinv * rinv, -(kxx + kyy));
                const float rdn = fmaf(f * s, Ca - __uint_as_float(pb.w), rd);
                const float rcn = fmaf(f, fmaf(va.x - vb.x, dx, (va.y - vb.y) * dy), rc);
                rd = in ? rdn : rd;
                rc = in ? rcn : rc;
            }
        neumaier_add(sd, cd, rd);
        neumaier_add(sc, cc, rc);
    }
    const float rate = fmaf(prm.pf, sd + cd, fp.pconv * Ca * (sc + cc));

    Acc acc{0.f, 0.f, __int_as_float(0x7f800000), __int_as_float(0xff800000), 0u};
    if (valid) {
        if (EPI == EPI_RATE) {
            if (out.rate) {
                const uint32_t a = __ldg(perm + i);
                if (a < (uint32_t)prm.n) out.rate[a] = rate;
            }
        } else if (EPI == EPI_PREDICT) {
            // C^{l+1/2} = C^l + dt/2 r^l, x_a^{l+1/2} = x_a^l + dt/2 v_a
            uint32_t inc[3];
            half_drift(ic, inc);
            uint4 q;
            q.x = pa.x + inc[0];
            q.y = pa.y + inc[1];
            q.z = pa.z + inc[2];
            q.w = __float_as_uint(fmaf(prm.dt, rate, Ca));
            out.Pout[i] = q;
        } else {
            // C^{l+1} = C^l + dt r^{l+1/2}, x_a^{l+1} = x_a^l + dt v_a (caller order); x^l is the
            // evaluation position minus this particle's half-step drift (exact in fixed point)
            const uint32_t a = __ldg(perm + i);
            uint32_t inc[3];
            full_drift(ic, inc);
            float Cn = 0.f;
            if (a < (uint32_t)prm.n) {
                Cn = fmaf(prm.dt, rate, out.C[a]);
                out.C[a] = Cn;
                out.xq[a] = pa.x - back[0] + inc[0];
                out.xq[(size_t)prm.n + a] = pa.y - back[1] + inc[1];
            }
            if (!isfinite(Cn)) atomicOr(out.status, 1);
            two_sum_add(acc.hi, acc.lo, Cn, 0.f);
            acc.mn = fminf(acc.mn, Cn);
            acc.mx = fmaxf(acc.mx, Cn);
        }
    }
    warp_finish<EPI, false, kT>(acc, out);
}

// 3D: a warp takes up to 32 consecutive particles of one pencil (find_chunk), so its lanes share the
// stencil rows; each lane's range of a row is cut by the distance its own cell position leaves to the
// row's cell band, for the grid's radius H + dt vmax (positions of the build: the drift since cannot
// bring a pair within H that was beyond it).  The candidates are only tested first, and those in support
// noted in the lane's list in shared memory; full lists are evaluated together.  On an irregular set the
// lanes' ranges of a row differ, and a warp that evaluated where it tested would spend the pair's 110
// instructions on the longest lane's candidates, in support or not: 6.7 a pair on 45^3
// jittered particles.  SPLIT 4 (sets that leave the chip idle): the block's four warps share a chunk, each
// takes every fourth row, and warp 0 adds their sums in order.
// Per evaluation: 45^3 jittered, 195 neighbours, 425 -> 235 us (at the grid of about two
// particles per cell; 24^3 345 -> 105).
constexpr int kList = 40;   // entries per lane (one flush is one FP32 partial sum)

template <int KERNEL, int EPI, int SPLIT>
__global__ __launch_bounds__(kT) void k_rate_field3(const uint4 *__restrict__ Pe, const uint32_t *__restrict__ cs,
                                                   const uint32_t *__restrict__ perm,
                                                   const float4 *__restrict__ V, const float4 *__restrict__ DA,
                                                   const float4 *__restrict__ DB, const uint4 *__restrict__ Inc,
                                                   const RateParams prm, const FieldParams fp, const EpiOut out)
{
    constexpr int DIM = 3;
    pdl_wait();   // no early trigger: see pdl_trigger
    __shared__ float4 part[SPLIT > 1 ? kT : 1];
    __shared__ unsigned lists[kT / 32][kList * 32];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const int ncx = prm.ncx;
    Acc acc{0.f, 0.f, __int_as_float(0x7f800000), __int_as_float(0xff800000), 0u};
    const PairConst kc(prm);
    unsigned *list = lists[wid] + lane;
    TrimGeom g(prm);
    g.Hm2 = prm.Hg2 * (1.f + 1.f / 2048.f);
    Chunk c;
    if (find_chunk(cs, prm, nullptr, SPLIT > 1 ? (int)blockIdx.x : warp_number(), c)) {   // (SPLIT: the same for the whole block)
        const int i = c.i0 + lane;
        bool valid = i < c.pe;
        const int ii = valid ? i : c.pe - 1;
        const uint4 pa = __ldg(Pe + ii);
        // fixed-point drift of this particle; the cell of the cell build is the evaluation position
        // minus the drift since the build (the half step, in the corrector)
        const uint4 ic = EPI == EPI_RATE ? make_uint4(0u, 0u, 0u, 0u) : __ldg(Inc + ii);
        uint32_t back[3] = {0u, 0u, 0u};
        if (EPI == EPI_CORRECT) half_drift(ic, back);
        const FieldTarget t(pa, __uint_as_float(pa.w), __ldg(V + ii), __ldg(DA + ii), __ldg(DB + ii));
        const int cx = (int)__umulhi(pa.x - back[0], (uint32_t)ncx);
        const float inv32 = 2.3283064365386963e-10f;   // 2^-32
        const float fx = (float)((pa.x - back[0]) * (uint32_t)ncx) * inv32;
        const float fy = (float)((pa.y - back[1]) * (uint32_t)prm.ncy) * inv32;
        const float fz = (float)((pa.z - back[2]) * (uint32_t)prm.ncz) * inv32;
        float sd = 0.f, cd = 0.f, sc = 0.f, cc = 0.f;
        int have = 0;
        auto flush = [&]() {
            float rd = 0.f, rc = 0.f;
#pragma unroll 2
            for (int e = 0; e < have; ++e) field_pair<KERNEL>(t, Pe, V, DA, DB, list[32 * e], kc, fp.gamma, rd, rc);
            neumaier_add(sd, cd, rd);
            neumaier_add(sc, cc, rc);
            have = 0;
        };
        for (int ri = SPLIT > 1 ? wid : 0; ri < prm.nrows; ri += SPLIT) {
            const StencilRow row = prm.rows[ri];
            const TrimRow tr{(float)row.dy, (float)row.dz, 0, 0};
            const float e2 = row_gap2<DIM>(make_float4(0.f, 1.f, 0.f, 1.f), tr, fy, fy, 0.f, fz, fz, 0.f, g);
            const float d2 = fmaxf(g.Hm2 - e2, 0.f);
            if (!__any_sync(kFull, e2 < g.Hm2)) continue;
            const float xe = fmaf(d2 * rsqrt_ftz(fmaxf(d2, 1.f)), g.inv_wx, 1.f / 4096.f);
            const int w = row.w;
            const int q = row_pencil_of<DIM>(row, c.cy, c.cz, prm);
            const int qs = (int)__ldg(cs + q * ncx), qe = (int)__ldg(cs + q * ncx + ncx), len = qe - qs;
            int s, cnt;
            cyclic_range(cs, q * ncx, cx + max(__float2int_rd(fx - xe), -w), cx + min(__float2int_rd(fx + xe), w) + 1, ncx, qs, qe,
                         s, cnt);
            if (!(e2 < g.Hm2)) cnt = 0;
            for (int u = 0; __any_sync(kFull, u < cnt);) {
                // up to the room every lane's list has
                const int room = kList - (int)__reduce_max_sync(kFull, (unsigned)have);
                const int end = min(cnt, u + room);
                for (; u < end; ++u) {
                    const int j = s + u, jj = j >= qe ? j - len : j;
                    float dx, dy, dz;
                    const float r2 = field_sep(t, __ldg(Pe + jj), kc, dx, dy, dz);
                    if (r2 < prm.H2 && r2 > 0.f) list[32 * have++] = (unsigned)jj;
                }
                if (room < kList / 4) flush();
            }
        }
        flush();
        if (SPLIT > 1) {
            part[threadIdx.x] = make_float4(sd, cd, sc, cc);
            __syncthreads();
            if (wid == 0)
                for (int q = 1; q < SPLIT; ++q) {
                    const float4 o = part[32 * q + lane];
                    neumaier_add(sd, cd, o.x);
                    neumaier_add(sc, cc, o.z);
                    cd += o.y;
                    cc += o.w;
                }
            __syncthreads();
            if (wid != 0) valid = false;
        }
        const float rate = fmaf(prm.pf, sd + cd, fp.pconv * t.Ca * (sc + cc));
        if (!valid) {
        } else if (EPI == EPI_RATE) {
            if (out.rate) {
                const uint32_t a = __ldg(perm + i);
                if (a < (uint32_t)prm.n) out.rate[a] = rate;
            }
        } else if (EPI == EPI_PREDICT) {
            // C^{l+1/2} = C^l + dt/2 r^l, x_a^{l+1/2} = x_a^l + dt/2 v_a
            uint32_t inc[3];
            half_drift(ic, inc);
            uint4 o;
            o.x = pa.x + inc[0];
            o.y = pa.y + inc[1];
            o.z = pa.z + inc[2];
            o.w = __float_as_uint(fmaf(prm.dt, rate, t.Ca));
            out.Pout[i] = o;
        } else {
            // C^{l+1} = C^l + dt r^{l+1/2}, x_a^{l+1} = x_a^l + dt v_a (caller order); x^l is the
            // evaluation position minus this particle's half-step drift (exact in fixed point)
            const uint32_t a = __ldg(perm + i);
            uint32_t inc[3];
            full_drift(ic, inc);
            float Cn = 0.f;
            if (a < (uint32_t)prm.n) {
                Cn = fmaf(prm.dt, rate, out.C[a]);
                out.C[a] = Cn;
                out.xq[a] = pa.x - back[0] + inc[0];
                out.xq[(size_t)prm.n + a] = pa.y - back[1] + inc[1];
                out.xq[2 * (size_t)prm.n + a] = pa.z - back[2] + inc[2];
            }
            if (!isfinite(Cn)) atomicOr(out.status, 1);
            two_sum_add(acc.hi, acc.lo, Cn, 0.f);
            acc.mn = fminf(acc.mn, Cn);
            acc.mx = fmaxf(acc.mx, Cn);
        }
    }
    if (EPI == EPI_CORRECT) {   // one partial per warp (SPLIT: the block's first)
        const float4 r = warp_partial(acc);
        if (lane == 0 && (SPLIT == 1 || wid == 0)) out.wpart[SPLIT == 1 ? warp_number() : (int)blockIdx.x] = r;
    }
}

template <int KERNEL, int SPLIT>
cudaError_t launch_field3(int epi, unsigned grid, const uint4 *Pe, const uint32_t *cs, const uint32_t *perm,
                          const FieldWork &fw, const RateParams &prm, const FieldParams &fp, const EpiOut &out,
                          cudaStream_t s)
{
    switch (epi) {
    case EPI_RATE:
        return launch_pdl(k_rate_field3<KERNEL, EPI_RATE, SPLIT>, grid, kT, 0, s, Pe, cs, perm, fw.V, fw.DA, fw.DB, fw.Inc, prm, fp, out);
    case EPI_PREDICT:
        return launch_pdl(k_rate_field3<KERNEL, EPI_PREDICT, SPLIT>, grid, kT, 0, s, Pe, cs, perm, fw.V, fw.DA, fw.DB, fw.Inc, prm, fp, out);
    default:
        return launch_pdl(k_rate_field3<KERNEL, EPI_CORRECT, SPLIT>, grid, kT, 0, s, Pe, cs, perm, fw.V, fw.DA, fw.DB, fw.Inc, prm, fp, out);
    }
}

template <int KERNEL>
cudaError_t launch_field2(int epi, const uint4 *Pe, const uint32_t *cs, const uint32_t *perm, const FieldWork &fw,
                          const RateParams &prm, const FieldParams &fp, const EpiOut &out, cudaStream_t s)
{
    const unsigned g = (unsigned)((prm.n + kT - 1) / kT);
    switch (epi) {
    case EPI_RATE:
        return launch_pdl(k_rate_field2<KERNEL, EPI_RATE>, g, kT, 0, s, Pe, cs, perm, fw.V, fw.DA, fw.Inc, prm, fp, out);
    case EPI_PREDICT:
        return launch_pdl(k_rate_field2<KERNEL, EPI_PREDICT>, g, kT, 0, s, Pe, cs, perm, fw.V, fw.DA, fw.Inc, prm, fp, out);
    default:
        return launch_pdl(k_rate_field2<KERNEL, EPI_CORRECT>, g, kT, 0, s, Pe, cs, perm, fw.V, fw.DA, fw.Inc, prm, fp, out);
    }
}

// Chunks of a set that fills the chip less than about twice (152 SMs of 24 warps) are shared by the four
// warps of a block.
bool field_split(const RateParams &prm) { return prm.n / 32 < 2 * 152 * 24; }
int field_chunks(const RateParams &prm) { return chunk_numbers(prm.n, prm.ncy * prm.ncz); }

template <int KERNEL>
cudaError_t launch_field_k(int dim, int epi, const uint4 *Pe, const uint32_t *cs, const uint32_t *perm, const FieldWork &fw,
                    const RateParams &prm, const FieldParams &fp, const EpiOut &out, cudaStream_t s)
{
    if (dim == 2) return launch_field2<KERNEL>(epi, Pe, cs, perm, fw, prm, fp, out, s);
    if (!field_split(prm)) return launch_field3<KERNEL, 1>(epi, frozen_blocks(prm), Pe, cs, perm, fw, prm, fp, out, s);
    return launch_field3<KERNEL, 4>(epi, (unsigned)field_chunks(prm), Pe, cs, perm, fw, prm, fp, out, s);
}

}  // namespace

int field_partials(int dim, const RateParams &prm)
{
    if (dim == 2) return (prm.n + kT - 1) / kT * (kT / 32);
    return field_split(prm) ? field_chunks(prm) : (int)frozen_blocks(prm) * (kT / 32);
}

cudaError_t launch_field_records(int dim, const float *v_dev, int n, const FieldParams &fp, const FieldWork &fw,
                                 cudaStream_t s)
{
    if (v_dev) {
        cudaError_t e = cudaMemsetAsync(fw.vmax_bits, 0, sizeof(unsigned), s);
        if (e != cudaSuccess) return e;
    }
    if (n == 0) return cudaSuccess;
    const int blocks = (n + kT - 1) / kT;
    if (dim == 2) {
        if (v_dev) k_field_velocity<2><<<blocks, kT, 0, s>>>(v_dev, n, fw.Vc, fw.vmax_bits);
        k_field_tensors<2><<<blocks, kT, 0, s>>>(n, fp, fw.Vc, fw.DAc, fw.DBc, fw.IncC);
    } else {
        if (v_dev) k_field_velocity<3><<<blocks, kT, 0, s>>>(v_dev, n, fw.Vc, fw.vmax_bits);
        k_field_tensors<3><<<blocks, kT, 0, s>>>(n, fp, fw.Vc, fw.DAc, fw.DBc, fw.IncC);
    }
    return cudaGetLastError();
}

cudaError_t launch_field_permute(int dim, const uint32_t *perm, int n, const FieldWork &fw, cudaStream_t s)
{
    if (n == 0) return cudaSuccess;
    const int blocks = (n + kT - 1) / kT;
    if (dim == 2)
        launch_pdl(k_field_permute<2>, blocks, kT, 0, s, perm, n, fw.Vc, fw.DAc, fw.DBc, fw.IncC, fw.V, fw.DA, fw.DB, fw.Inc);
    else
        launch_pdl(k_field_permute<3>, blocks, kT, 0, s, perm, n, fw.Vc, fw.DAc, fw.DBc, fw.IncC, fw.V, fw.DA, fw.DB, fw.Inc);
    return cudaGetLastError();
}

cudaError_t launch_rate_field(int dim, int kernel, int epi, const uint4 *Pe, const uint32_t *cell_start,
                              const uint32_t *perm, const FieldWork &fw, const RateParams &prm,
                              const FieldParams &fp, const EpiOut &out, cudaStream_t s)
{
    if (prm.n == 0) return cudaSuccess;
    if (out.pairs) {
        const unsigned blocks = (unsigned)((prm.n + kT - 1) / kT);
        return dim == 2 ? launch_pdl(k_count_field<2>, blocks, kT, 0, s, Pe, cell_start, prm, out)
                        : launch_pdl(k_count_field<3>, blocks, kT, 0, s, Pe, cell_start, prm, out);
    }
    return kernel == ADE_WENDLAND_C2 ? launch_field_k<ADE_WENDLAND_C2>(dim, epi, Pe, cell_start, perm, fw, prm, fp, out, s)
                                     : launch_field_k<ADE_WENDLAND_C4>(dim, epi, Pe, cell_start, perm, fw, prm, fp, out, s);
}

}  // namespace ade

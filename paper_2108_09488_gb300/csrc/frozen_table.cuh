// frozen_table.cuh -- table of pair weights over one cell list, and its use (rate_frozen.cu, sweep.cu,
// adjoint.cu): included inside an unnamed namespace of ade, after rate_walk.cuh.
//
// Layout.  A warp owns up to 32 consecutive sorted particles (lane = particle) of one pencil (the
// cells of one (cy, cz) row along x), so its lanes share the stencil rows.  Per row the lanes' in-
// support candidates are contiguous index ranges, trimmed at both ends to the first and last
// candidate that can lie inside H; m = the longest lane's length.  All storage is in 32-word lines
// (128 B, lane = word): per chunk the rows' m (one word each), then per row, in stencil order, one
// line of first indices and m lines of weights: one linear stream per chunk.  The concentrations are
// kept twice per pencil, back to back (particle j of pencil [ps, pe) at ps + j and again at pe + j),
// so that a range that runs over the periodic x seam stays contiguous.  A chunk that finds no room in
// the table is marked and evaluated from the positions instead (the same sums), so a table that is
// too small costs time, never a result (claim_lines in pool.h never hands out a line twice).
//
// A value is one word (the weight for one tensor: VAL 1) or two (g_L and g_T, from which every
// uniform tensor's weight follows: VAL 2, lane l's pair in words 2l, 2l + 1 of two lines); with low parts
// (FINE), those of the pair that begins in line k of the table lie in line k / 2 of a plane of their own.
#pragma once

constexpr unsigned kFull = 0xffffffffu;

// Where one warp's chunk lies: particles [i0, min(i0 + 32, pe)) of pencil p (cy, cz), which holds [ps, pe).
struct Chunk {
    int cy, cz, i0, ps, pe, p;
    int local, slot;       // the chunk's number within its plume, and in the slot table
};

// Chunk number t of a plume.  Pencil p's first chunk has the number dense[p] (counted), or where that is NULL
// (first particle >> 5) + p: strictly increasing, with at most one number per pencil that no chunk has.
// So a launch takes one warp per number whatever the set: a pencil's share of the warps is its share of the particles
// (launched by pencil, with the mean pencil's number of warps each, a set that fills 5 % of the box ran 4 to 9
// times slower, and more particles than 65,535 blocks of one pencil could not be launched).
// The warp finds the pencil by its lanes looking at 32 pencils around the place an even set has it in, one
// latency on a lattice, and otherwise by a search that divides the pencils in 32 each time.
// False where no chunk has the number.
__device__ __forceinline__ bool find_chunk(const uint32_t *__restrict__ cs, const RateParams &prm, const uint32_t *__restrict__ dense, int t,
                                           Chunk &c)
{
    const int lane = threadIdx.x & 31, np = prm.ncy * prm.ncz, ncx = prm.ncx;
    const int total = dense ? (int)__ldg(dense + np) : chunk_numbers(prm.n, np);
    c.local = c.slot = t;      // (also where there is no chunk: put_chunk marks the slot of every number)
    if (t >= total) return false;
    auto first = [&](int q, int &s) {      // the number of pencil q's first chunk; s: its first particle
        s = (int)__ldg(cs + (size_t)q * ncx);
        return dense ? (int)__ldg(dense + q) : ((s - prm.goff) >> 5) + q;
    };
    const int lo = max(0, min((int)((float)t * ((float)np / (float)total)) - 15, np - 31));
    int s;
    int k = __popc(__ballot_sync(kFull, first(min(lo + lane, np), s) <= t && lo + lane < np));
    if (k > 0 && k < 32) {
        c.p = lo + k - 1;
        c.ps = __shfl_sync(kFull, s, k - 1);
        c.pe = __shfl_sync(kFull, s, k);
    } else {
        int a = k > 0 ? lo + 31 : 0, b = k > 0 ? np : lo;   // pencil a begins at or before t, pencil b after it
        while (b - a > 1) {
            const int step = (b - a + 31) >> 5, q = min(a + step * lane, b);
            k = __popc(__ballot_sync(kFull, q < b && first(q, s) <= t));
            b = min(a + step * k, b);
            a += step * (k - 1);
        }
        c.p = a;
        c.ps = (int)__ldg(cs + (size_t)a * ncx);
        c.pe = (int)__ldg(cs + (size_t)a * ncx + ncx);
    }
    c.i0 = c.ps + 32 * (t - (dense ? (int)__ldg(dense + c.p) : ((c.ps - prm.goff) >> 5) + c.p));
    c.cy = c.p % prm.ncy;
    c.cz = c.p / prm.ncy;
    return c.i0 < c.pe;
}

// The slot table: per number {first line, rows, lines, header lines} and {first particle, pencil's first,
// pencil's end, pencil}.  The kernel that fills the table writes both, later passes read them.
__device__ __forceinline__ void put_chunk(const FrozenTab &tab, const Chunk &c, bool has)
{
    if ((threadIdx.x & 31) == 0)
        tab.slots[2 * (size_t)c.slot + 1] = has ? make_uint4((unsigned)c.i0, (unsigned)c.ps, (unsigned)c.pe, (unsigned)c.p)
                                                : make_uint4(0u, 0u, 0u, 0u);
}

__device__ __forceinline__ bool get_chunk(const FrozenTab &tab, const RateParams &prm, int slot, Chunk &c, uint4 &sl)
{
    const uint4 w = __ldg(tab.slots + 2 * (size_t)slot + 1);
    sl = __ldg(tab.slots + 2 * (size_t)slot);
    c.i0 = (int)w.x;
    c.ps = (int)w.y;
    c.pe = (int)w.z;
    c.p = (int)w.w;
    c.slot = slot;
    return c.i0 < c.pe;
}

// This warp's number in a launch of frozen_blocks blocks, and the same for a chunk already in the table.
__device__ __forceinline__ int warp_number() { return blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5); }
__device__ __forceinline__ bool my_chunk(const FrozenTab &tab, const RateParams &prm, Chunk &c, uint4 &sl)
{
    const int t = warp_number();
    return t < chunk_numbers(prm.n, prm.ncy * prm.ncz) && get_chunk(tab, prm, t, c, sl);
}

// Origin of the build's cell grid along x (the records hold the positions of the build: no drift).
__device__ __forceinline__ uint32_t frame_x(const RateParams &prm) { return prm.frame ? __ldg(prm.frame + 4) : 0u; }

// Weight of the pair (a, b): the branch-free walks' product of shape and pair factor; 0 outside the
// support and at zero separation.
template <int DIM, int KERNEL, bool ISO>
__device__ __forceinline__ float pair_weight(const uint4 &pa, const uint4 &pb, const PairConst &k)
{
    float dx = sep(pa.x, pb.x, k.m1), dy = sep(pa.y, pb.y, k.m1), dz = 0.f;
    if (DIM == 3) dz = sep(pa.z, pb.z, k.m1);
    if (!ISO) {
        dy *= k.sy;
        if (DIM == 3) dz *= k.sz;
    }
    float r2 = fmaf(dx, dx, dy * dy);
    if (DIM == 3) r2 = fmaf(dz, dz, r2);
    const float rinv = rsqrt_ftz(r2);
    const float om = fmaf(-(r2 * rinv), k.invH, 1.f);
    const float omq2 = fmaxf(om + om, 0.f);
    const float s = fmaxf(dcal<DIM>(dx, dy, dz, rinv, k), -3.402823466e38f);
    return shape2x<KERNEL>(omq2) * s;
}

// The pair's weights for D = vhat vhat^T and D = I - vhat vhat^T (Eq. 3-5 with K = 2D),
//   g_L = f (2 Gamma u - 2),  g_T = f (-2 Gamma u + 2 (Gamma - d) + 2),  u = (vhat . e)^2,
// from which every uniform tensor's weight is (alpha_L |v| + D_m) g_L + (alpha_T |v| + D_m) g_T (sums of
// f and f u would cancel in that).  Both 0 outside the support and at zero separation.  Low parts (what FP32
// leaves) of the constants: vl {vhat, 1/H}, g2l, bTl, syl, szl (pair_fine2 only).
struct ShapeConst {
    float4 vl;
    float g2, bT;          // 2 Gamma, 2 (Gamma - d) + 2
    float g2l, bTl, syl, szl;
};

// The sweep's: two candidates at once, in packed FP32x2 instructions.
template <int DIM, int KERNEL, bool ISO>
__device__ __forceinline__ void pair_shape2(const uint4 &pa, const uint4 &p0, const uint4 &p1, const PairConst2 &k,
                                            const ShapeConst &sc, float2 &gL, float2 &gT)
{
    const float2 dx = f2(sep(pa.x, p0.x, k.m1), sep(pa.x, p1.x, k.m1));
    float2 dy = f2(sep(pa.y, p0.y, k.m1), sep(pa.y, p1.y, k.m1));
    float2 dz = f2(0.f, 0.f);
    if (DIM == 3) dz = f2(sep(pa.z, p0.z, k.m1), sep(pa.z, p1.z, k.m1));
    if (!ISO) {
        dy = __fmul2_rn(dy, k.sy);
        if (DIM == 3) dz = __fmul2_rn(dz, k.sz);
    }
    const float2 m1 = f2(-1.f, -1.f), one = f2(1.f, 1.f), g2 = f2(sc.g2, sc.g2);
    float2 r2 = __ffma2_rn(dx, dx, __fmul2_rn(dy, dy)), c = __ffma2_rn(k.w0, dx, __fmul2_rn(k.w1, dy));
    if (DIM == 3) {
        r2 = __ffma2_rn(dz, dz, r2);
        c = __ffma2_rn(k.w2, dz, c);
    }
    const float2 rinv = f2(rsqrt_ftz(r2.x), rsqrt_ftz(r2.y));
    const float2 om = __ffma2_rn(__fmul2_rn(r2, rinv), k.ninvH, one);
    const float2 f = shape2x2<KERNEL>(f2(fmaxf(om.x + om.x, 0.f), fmaxf(om.y + om.y, 0.f)));
    const float2 t = __fmul2_rn(c, rinv), t2 = __fmul2_rn(t, t), u = f2(fminf(t2.x, 1.f), fminf(t2.y, 1.f));
    gL = __fmul2_rn(f, __ffma2_rn(g2, u, f2(-2.f, -2.f)));
    gT = __fmul2_rn(f, __ffma2_rn(__fmul2_rn(g2, m1), u, f2(sc.bT, sc.bT)));
}

template <int DIM, int KERNEL, bool ISO>
__device__ __forceinline__ float2 pair_shape(const uint4 &pa, const uint4 &pb, const PairConst2 &k, const ShapeConst &sc)
{
    float2 gL, gT;
    pair_shape2<DIM, KERNEL, ISO>(pa, pb, pb, k, sc, gL, gT);
    return make_float2(gL.x, gT.x);
}

// Numbers of twice FP32's precision as unevaluated sums h + l, two at a time: sum and product with their
// rounding errors (Knuth's two-sum; fused multiply-add), added to what l holds already.
__device__ __forceinline__ float2 sub2(float2 a, float2 b) { return __ffma2_rn(b, f2(-1.f, -1.f), a); }
__device__ __forceinline__ float2 two_sum2(float2 a, float2 b, float2 &lo)
{
    const float2 s = __fadd2_rn(a, b), bb = sub2(s, a);
    lo = __fadd2_rn(lo, __fadd2_rn(sub2(a, sub2(s, bb)), sub2(b, bb)));
    return s;
}
__device__ __forceinline__ float2 two_prod2(float2 a, float2 b, float2 &lo)
{
    const float2 p = __fmul2_rn(a, b);
    lo = __fadd2_rn(lo, __ffma2_rn(a, b, __fmul2_rn(p, f2(-1.f, -1.f))));
    return p;
}
struct Double2 {
    float2 h, l;
};
__device__ __forceinline__ Double2 mul22(const Double2 &a, const Double2 &b)
{
    Double2 r;
    r.l = __ffma2_rn(a.h, b.l, __fmul2_rn(a.l, b.h));
    r.h = two_prod2(a.h, b.h, r.l);
    return r;
}
__device__ __forceinline__ Double2 settle(const Double2 &a)     // |l| at most half a unit of h's last place
{
    const float2 h = __fadd2_rn(a.h, a.l);
    return Double2{h, sub2(a.l, sub2(h, a.h))};
}
__device__ __forceinline__ float2 both(float x) { return f2(x, x); }
// Separation of two candidates along one axis (h + l is the integer difference exactly).
__device__ __forceinline__ Double2 sep22(uint32_t a, uint32_t b0, uint32_t b1)
{
    const int d0 = (int)(a - b0), d1 = (int)(a - b1);
    const float h0 = (float)d0, h1 = (float)d1;
    return Double2{f2(h0, h1), f2((float)(d0 - __float2int_rn(h0)), (float)(d1 - __float2int_rn(h1)))};
}

// g_L and g_T of two candidates to twice FP32 (the adjoint).  On a lattice the same few separations recur, so a
// weight's rounding biases every pair alike, and dJ/dtheta adds the pairs of all steps: with weights rounded
// to FP32 it was off by up to 2e-7 of its value.
template <int DIM, int KERNEL, bool ISO>
__device__ __forceinline__ void pair_fine2(const uint4 &pa, const uint4 &p0, const uint4 &p1, const PairConst2 &k,
                                           const ShapeConst &sc, Double2 &gL, Double2 &gT)
{
    const float2 m1 = both(-1.f), half = both(0.5f), none = both(0.f);
    const Double2 x = sep22(pa.x, p0.x, p1.x);
    Double2 y = sep22(pa.y, p0.y, p1.y), z = Double2{none, none};
    if (DIM == 3) z = sep22(pa.z, p0.z, p1.z);
    if (!ISO) {
        y = mul22(y, Double2{k.sy, both(sc.syl)});
        if (DIM == 3) z = mul22(z, Double2{k.sz, both(sc.szl)});
    }
    // r^2 and vhat . x
    float2 r2l = __fmul2_rn(__fadd2_rn(x.h, x.h), x.l), cl = __ffma2_rn(both(sc.vl.x), x.h, __fmul2_rn(k.w0, x.l));
    r2l = __ffma2_rn(__fadd2_rn(y.h, y.h), y.l, r2l);
    cl = __ffma2_rn(both(sc.vl.y), y.h, __ffma2_rn(k.w1, y.l, cl));
    float2 r2 = two_prod2(x.h, x.h, r2l), ch = two_prod2(k.w0, x.h, cl);
    r2 = two_sum2(r2, two_prod2(y.h, y.h, r2l), r2l);
    ch = two_sum2(ch, two_prod2(k.w1, y.h, cl), cl);
    if (DIM == 3) {
        r2l = __ffma2_rn(__fadd2_rn(z.h, z.h), z.l, r2l);
        cl = __ffma2_rn(both(sc.vl.z), z.h, __ffma2_rn(k.w2, z.l, cl));
        r2 = two_sum2(r2, two_prod2(z.h, z.h, r2l), r2l);
        ch = two_sum2(ch, two_prod2(k.w2, z.h, cl), cl);
    }
    // 1/r with a Newton step, r and -q = -r/H, 1 - q
    float2 rinv = f2(rsqrt_ftz(r2.x), rsqrt_ftz(r2.y));
    rinv = __ffma2_rn(__fmul2_rn(half, rinv), __ffma2_rn(__fmul2_rn(__fmul2_rn(r2, rinv), m1), rinv, both(1.f)), rinv);
    const float2 r = __fmul2_rn(r2, rinv), nr = __fmul2_rn(r, m1);
    const float2 rl = __fmul2_rn(__fmul2_rn(half, rinv), __fadd2_rn(__ffma2_rn(nr, r, r2), r2l));
    const float2 nq = __fmul2_rn(r, k.ninvH);
    Double2 om;
    om.l = __ffma2_rn(nr, both(sc.vl.w), __ffma2_rn(rl, k.ninvH, __ffma2_rn(r, k.ninvH, __fmul2_rn(nq, m1))));
    om.h = two_sum2(both(1.f), nq, om.l);
    om = settle(om);
    // twice 1 - q, 0 outside the support (and at r = 0, where it is not a number)
    const bool in0 = om.h.x > 0.f, in1 = om.h.y > 0.f;
    const Double2 w{f2(in0 ? om.h.x + om.h.x : 0.f, in1 ? om.h.y + om.h.y : 0.f), f2(in0 ? om.l.x + om.l.x : 0.f, in1 ? om.l.y + om.l.y : 0.f)};
    Double2 f = mul22(w, w);
    if (KERNEL == ADE_WENDLAND_C2) {
        f = mul22(f, w);
    } else {
        Double2 q{none, __fmul2_rn(both(-2.5f), w.l)};                          // 6 - 5 (1 - q)
        q.h = two_sum2(both(6.f), two_prod2(both(-2.5f), w.h, q.l), q.l);
        f = mul22(mul22(mul22(f, f), w), q);
    }
    // u = (vhat . x)^2 / r^2 and what is left of it
    const float2 t = __fmul2_rn(ch, rinv), t2 = __fmul2_rn(t, t);
    const float2 u = f2(fminf(t2.x, 1.f), fminf(t2.y, 1.f)), nu = __fmul2_rn(u, m1);
    float2 e = __fmul2_rn(__fadd2_rn(ch, ch), cl);
    const float2 n = two_prod2(ch, ch, e);
    e = __fadd2_rn(e, __ffma2_rn(nu, r2, n));       // (exact: n and u r^2 agree to a few units)
    e = __ffma2_rn(nu, r2l, e);
    float2 ul = __fmul2_rn(__fmul2_rn(e, rinv), rinv);
    ul = f2(fminf(fmaxf(ul.x, -1e-6f), 1e-6f), fminf(fmaxf(ul.y, -1e-6f), 1e-6f));   // (max-num: finite at r = 0 too)
    const float2 g2ul = __ffma2_rn(both(sc.g2), ul, __fmul2_rn(both(sc.g2l), u));
    Double2 A{none, g2ul}, B{none, __ffma2_rn(g2ul, m1, both(sc.bTl))};
    A.h = two_sum2(two_prod2(both(sc.g2), u, A.l), both(-2.f), A.l);
    B.h = two_sum2(two_prod2(both(sc.g2), nu, B.l), both(sc.bT), B.l);
    gL = settle(mul22(f, A));
    gT = settle(mul22(f, B));
}

// Two low parts in one word, 16 bits each: FP32 hi and a low part cut to 8 bits are 32 bits of a weight.
__device__ __forceinline__ float pack_low(float lL, float lT)
{
    return __uint_as_float((__float_as_uint(lT) & 0xffff0000u) | (__float_as_uint(lL) >> 16));
}
__device__ __forceinline__ float2 unpack_low(float w)
{
    return f2(__uint_as_float(__float_as_uint(w) << 16), __uint_as_float(__float_as_uint(w) & 0xffff0000u));
}

// Squared separation in x units^2.
template <int DIM, bool ISO>
__device__ __forceinline__ float sep2(const uint4 &pa, const uint4 &pb, const PairConst &k)
{
    float dx = sep(pa.x, pb.x, k.m1), dy = sep(pa.y, pb.y, k.m1), dz = 0.f;
    if (DIM == 3) dz = sep(pa.z, pb.z, k.m1);
    if (!ISO) {
        dy *= k.sy;
        if (DIM == 3) dz *= k.sz;
    }
    float r2 = fmaf(dx, dx, dy * dy);
    if (DIM == 3) r2 = fmaf(dz, dz, r2);
    return r2;
}

// The weights of two candidates, the FP32 part in packed FP32x2 instructions (each half with the
// operations of pair_weight, so the same bits).  ZS = false: zero separation does not occur (rows other
// than the particles' own), as in pair_range_direct.
template <int DIM, int KERNEL, bool ISO, bool ZS>
__device__ __forceinline__ float2 pair_weight2(const uint4 &pa, const uint4 &p0, const uint4 &p1, const PairConst2 &k)
{
    float2 dx = f2(sep(pa.x, p0.x, k.m1), sep(pa.x, p1.x, k.m1));
    float2 dy = f2(sep(pa.y, p0.y, k.m1), sep(pa.y, p1.y, k.m1));
    float2 dz = f2(0.f, 0.f);
    if (DIM == 3) dz = f2(sep(pa.z, p0.z, k.m1), sep(pa.z, p1.z, k.m1));
    if (!ISO) {
        dy = __fmul2_rn(dy, k.sy);
        if (DIM == 3) dz = __fmul2_rn(dz, k.sz);
    }
    float2 r2 = __ffma2_rn(dx, dx, __fmul2_rn(dy, dy));
    if (DIM == 3) r2 = __ffma2_rn(dz, dz, r2);
    const float2 rinv = f2(rsqrt_ftz(r2.x), rsqrt_ftz(r2.y));
    const float2 om = __ffma2_rn(__fmul2_rn(r2, rinv), k.ninvH, f2(1.f, 1.f));
    const float2 omq2 = ZS ? f2(fmaxf(om.x + om.x, 0.f), fmaxf(om.y + om.y, 0.f)) : f2(om.x + fabsf(om.x), om.y + fabsf(om.y));
    const float2 sr = dcal2<DIM>(dx, dy, dz, rinv, k);
    const float2 sc = ZS ? f2(fmaxf(sr.x, -3.402823466e38f), fmaxf(sr.y, -3.402823466e38f)) : sr;
    return __fmul2_rn(shape2x2<KERNEL>(omq2), sc);
}

// Weights of one row's m candidates s, s + 1, ... (WRAP: beyond qe on from qe - len) into out, a line each,
// and the row sum of the records' concentrations.
template <int DIM, int KERNEL, bool ISO, bool ZS, bool WRAP>
__device__ __forceinline__ float row_weights(const uint4 *__restrict__ P, const uint4 &pa, float Ca, const PairConst &k,
                                             const PairConst2 &k2, int s, int m, int qe, int len, float *__restrict__ out)
{
    float rs = 0.f;
    const uint4 *Ps = P + s;
    int t = 0;
#pragma unroll 2
    for (; t + 1 < m; t += 2) {
        const uint4 p0 = __ldg(WRAP && s + t >= qe ? Ps + t - len : Ps + t);
        const uint4 p1 = __ldg(WRAP && s + t + 1 >= qe ? Ps + t + 1 - len : Ps + t + 1);
        const float2 w = pair_weight2<DIM, KERNEL, ISO, ZS>(pa, p0, p1, k2);
        out[t * 32] = w.x;
        out[(t + 1) * 32] = w.y;
        rs = fmaf(w.x, Ca - __uint_as_float(p0.w), rs);
        rs = fmaf(w.y, Ca - __uint_as_float(p1.w), rs);
    }
    if (t < m) {
        const uint4 pb = __ldg(WRAP && s + t >= qe ? Ps + t - len : Ps + t);
        const float w = pair_weight<DIM, KERNEL, ISO>(pa, pb, k);
        out[t * 32] = w;
        rs = fmaf(w, Ca - __uint_as_float(pb.w), rs);
    }
    return rs;
}

// Cyclic candidate range of cells [lo, hi) of the pencil row whose cells start at `base` and whose
// particles are [qs, qe): first index and count (a range over the seam continues at qs).
__device__ __forceinline__ void cyclic_range(const uint32_t *__restrict__ cs, int base, int lo, int hi, int ncx,
                                             int qs, int qe, int &s, int &cnt)
{
    const bool wl = lo < 0, wh = hi > ncx;
    s = (int)__ldg(cs + base + (wl ? lo + ncx : lo));
    const int e = (int)__ldg(cs + base + (wh ? hi - ncx : hi));
    cnt = (wl || wh) ? (qe - s) + (e - qs) : e - s;
}

// Stencil row r seen from pencil (cy, cz): its pencil index.
template <int DIM>
__device__ __forceinline__ int row_pencil_of(const StencilRow &r, int cy, int cz, const RateParams &prm)
{
    int yy = cy + r.dy;
    yy += yy < 0 ? prm.ncy : 0;
    yy -= yy >= prm.ncy ? prm.ncy : 0;
    int zz = 0;
    if (DIM == 3) {
        zz = cz + r.dz;
        zz += zz < 0 ? prm.ncz : 0;
        zz -= zz >= prm.ncz ? prm.ncz : 0;
    }
    return zz * prm.ncy + yy;
}

// Row sums over the positions for a chunk without room in the table: the full stencil, concentrations
// from C (doubled per pencil), or from the records where C is NULL.
template <int DIM, int KERNEL, bool ISO>
__device__ __noinline__ float walk_chunk(const uint4 *__restrict__ P, const uint32_t *__restrict__ cs,
                                         const RateParams &prm, const Chunk &c, const float *__restrict__ C)
{
    const int lane = threadIdx.x & 31;
    const int i = min(c.i0 + lane, c.pe - 1);
    const uint4 pa = __ldg(P + i);
    const float Ca = C ? C[c.ps + i] : __uint_as_float(pa.w);
    const int ncx = prm.ncx;
    const int cx = (int)__umulhi(pa.x - frame_x(prm), (uint32_t)ncx);
    const int cy = c.p % prm.ncy, cz = c.p / prm.ncy;
    const PairConst k(prm);
    float acc = 0.f, comp = 0.f;
    for (int r = 0; r < prm.nrows; ++r) {
        const StencilRow row = prm.rows[r];
        const int q = row_pencil_of<DIM>(row, cy, cz, prm);
        const int qs = (int)__ldg(cs + q * ncx), qe = (int)__ldg(cs + q * ncx + ncx), len = qe - qs;
        int s, cnt;
        cyclic_range(cs, q * ncx, cx - (int)row.w, cx + row.w + 1, ncx, qs, qe, s, cnt);
        float rs = 0.f;
        for (int t = 0; t < cnt; ++t) {
            int j = s + t;
            j = j >= qe ? j - len : j;
            const uint4 pb = __ldg(P + j);
            rs = fmaf(pair_weight<DIM, KERNEL, ISO>(pa, pb, k), Ca - (C ? C[qs + j] : __uint_as_float(pb.w)), rs);
        }
        neumaier_add(acc, comp, rs);
    }
    return acc + comp;
}

// How a chunk's rows and ranges are cut before the separations are evaluated: every row and range
// (kCutFull: unequal boxes), by the cell bands (kCutBand: no pencil boxes at hand), or by the pencils'
// transverse boxes (kCutBox), as in the trimmed walks.
enum ChunkCut { kCutFull = 0, kCutBand = 1, kCutBox = 2 };

// Calls f(q's first and end particle, first candidate s, longest lane's count m, row word) for each row of
// chunk c that holds a candidate within H of some lane: the lanes' contiguous ranges of the row's pencil,
// cut as CUT says.  Rows are tested once per warp, each lane's range is cut by its own distance to the row
// and then to its first and last candidate that may lie inside H.
template <int DIM, bool ISO, int CUT, class F>
__device__ __forceinline__ void chunk_rows(const uint4 *__restrict__ P, const uint32_t *__restrict__ cs, const RateParams &prm,
                                           const Chunk &c, const uint4 &pa, const TrimRow *srow, F f)
{
    const int lane = threadIdx.x & 31;
    const int ncx = prm.ncx, nrows = prm.nrows;
    const int cx = (int)__umulhi(pa.x - frame_x(prm), (uint32_t)ncx);
    const bool valid = c.i0 + lane < c.pe;
    TrimSelf me = {};
    float ylo = 0.f, yhi = 0.f, zlo = 0.f, zhi = 0.f;
    const TrimGeom g(prm);
    const float wpc = 4294967296.f / (float)ncx;     // x words per cell
    const PairConst k(prm);
    const float far2 = prm.H2 * (1.f + 1.f / 4096.f);   // beyond this the weight is exactly 0
    if (CUT != kCutFull) {
        me = trim_self<DIM>(pa, c.cy, c.cz, prm);
        ylo = yhi = me.fy;
        zlo = zhi = me.fz;
        warp_interval<DIM>(ylo, yhi, zlo, zhi);
    }
    for (int rb = 0; rb < nrows; rb += 32) {
        float xe = 0.f;
        int pidx = 0, wx = 0;
        bool reach = rb + lane < nrows;
        if (CUT == kCutBox) {
            reach = warp_row_test<DIM>(rb, srow, nrows, me, c.cy, c.cz, prm, g, ylo, yhi, zlo, zhi, xe, pidx, wx);
        } else if (reach) {
            const StencilRow r = prm.rows[rb + lane];
            pidx = row_pencil_of<DIM>(r, c.cy, c.cz, prm);
            wx = (r.w & 0xff) | (r.dy == 0 && (DIM == 2 || r.dz == 0) ? 1 << 24 : 0);
            if (CUT == kCutBand) {
                const TrimRow tr{(float)r.dy, (float)r.dz, 0, 0};
                const float e2 = row_gap2<DIM>(make_float4(0.f, 1.f, 0.f, DIM == 3 ? 1.f : 0.f), tr, ylo, yhi, yhi - ylo, zlo, zhi,
                                               zhi - zlo, g);
                const float t = fmaxf(g.Hm2 - e2, 0.f);
                xe = fmaf(t * rsqrt_ftz(fmaxf(t, 1.f)), g.inv_wx, 1.f / 4096.f);
                reach = e2 < g.Hm2;
            }
        }
        for (unsigned mask = __ballot_sync(kFull, reach); mask != 0u; mask &= mask - 1u) {
            const int b = __ffs(mask) - 1;
            const int q = __shfl_sync(kFull, pidx, b), wb = __shfl_sync(kFull, wx, b), w = wb & 0xff;
            int dlo = -w, dhi = w, xw = 0x7fffffff;          // xw: the lane's x half-extent in words
            if (CUT == kCutBox) {
                const TrimRow tr = srow[rb + b];
                const float e2 = row_gap2<DIM>(load_box(prm, q), tr, me.fy, me.fy, 0.f, me.fz, me.fz, 0.f, g);
                const float t = g.Hm2 - e2, xl = t > 0.f ? fmaf(t * rsqrt_ftz(t), g.inv_wx, 1.f / 4096.f) : 0.f;
                dlo = max(__float2int_rd(me.fx - xl), -w);
                dhi = min(__float2int_rd(me.fx + xl), w);
                xw = t > 0.f ? __float2int_ru(fminf(xl * wpc, 2.0e9f)) : -1;
            } else if (CUT == kCutBand) {
                const float xeb = __shfl_sync(kFull, xe, b);
                dlo = max(__float2int_rd(me.fx - xeb), -w);
                dhi = min(__float2int_rd(me.fx + xeb), w);
            }
            const int qs = (int)__ldg(cs + q * ncx), qe = (int)__ldg(cs + q * ncx + ncx), len = qe - qs;
            int s, cnt;
            cyclic_range(cs, q * ncx, cx + dlo, cx + dhi + 1, ncx, qs, qe, s, cnt);
            if (!valid || xw < 0) cnt = 0;
            if (s >= qe) s = qs;                     // (the range's first cells are empty)
            // Both ends' two outermost candidates are looked at together (one latency): farther than xw
            // along x, or than H, their weight is exactly 0.
            auto out_of = [&](int t) {
                const int j = s + t, jj = j >= qe ? j - len : j;
                if (CUT == kCutBox) {
                    const int d = (int)(__ldg(&P[jj].x) - pa.x);
                    return d < -xw || d > xw;
                }
                return !(sep2<DIM, ISO>(pa, __ldg(P + jj), k) < far2);
            };
            while (cnt > 0) {
                const bool f0 = out_of(0), f1 = out_of(min(1, cnt - 1)), b0 = out_of(cnt - 1), b1 = out_of(max(cnt - 2, 0));
                const int df = f0 ? (f1 ? 2 : 1) : 0, db = b0 ? (b1 ? 2 : 1) : 0, left = cnt - df - db;
                if (left <= 0) {                     // the ends meet: what is left, if anything, lies between
                    if (f0 && f1 && b0 && b1 && cnt <= 4) cnt = 0;
                    break;
                }
                s += df;
                if (s >= qe) s -= len;
                cnt = left;
                if (df < 2 && db < 2) break;
            }
            const int m = (int)__reduce_max_sync(kFull, (unsigned)cnt);
            if (m > 0) f(qs, qe, s, m, wb);
        }
    }
}

// Lines that hold the rows' lengths, a word per row.
__device__ __forceinline__ unsigned header_lines(const RateParams &prm) { return (unsigned)(prm.nrows + 31) >> 5; }

// Weights (VAL 1) or g_L, g_T (VAL 2; FINE: and their low parts) of one chunk into the table; VAL 1 returns the row sums of the
// first evaluation (the concentrations of the records).  One pass over the rows: the chunk's lines go
// to its region (prm.fz_stride lines, what nearly every chunk needs: plan_table in api.cu) and only a chunk
// that outgrows it is done again into room taken from the pool behind; fz_stride 0: no table.
// Bound: instruction issue.  128^3 cube 1.27 ms with the first predictor (ncu), 1024^2 204 us; a form that counted
// every chunk's lines in a pass of its own took 0.4 ms and 55 us more.
template <int DIM, int KERNEL, bool ISO, int CUT, int VAL, bool FINE = false>
__device__ __forceinline__ float build_chunk(const uint4 *__restrict__ P, const uint32_t *__restrict__ cs, const RateParams &prm,
                             const Chunk &c, const uint4 &pa, const TrimRow *srow, const FrozenTab &tab,
                             const ShapeConst &sc = ShapeConst())
{
    const int lane = threadIdx.x & 31;
    const PairConst k(prm);
    const PairConst2 k2(k, k.m1);
    const float Ca = __uint_as_float(pa.w);
    const unsigned hs = header_lines(prm);
    unsigned base = prm.fz_base + (unsigned)c.local * prm.fz_stride, room = (unsigned)c.local < prm.fz_regions ? prm.fz_stride : 0u;
    float acc = 0.f, comp = 0.f;
    unsigned R = 0u, used = 0xffffffffu;
    for (int attempt = 0; attempt < (prm.fz_stride > 0u ? 2 : 0); ++attempt) {
        acc = comp = 0.f;
        R = 0u;
        used = hs;
        float *hdr = tab.words + (size_t)base * 32;
        float *out = hdr + hs * 32 + lane;
        chunk_rows<DIM, ISO, CUT>(P, cs, prm, c, pa, srow, [&](int qs, int qe, int s, int m, int wb) {
            const int len = qe - qs;
            // idle tail iterations of a shorter lane stay inside the doubled pencil (m <= len)
            used = add_lines(used, 1u + (unsigned)(m * VAL));
            const bool keep = used <= room;
            if (keep) {
                if (lane == 0) hdr[R] = __int_as_float(m);
                out[0] = __int_as_float(s + qs);     // index into the doubled concentrations
            }
            ++R;
            if (!keep) return;                       // to be done again
            out += 32;
            float rs = 0.f;
            if (FINE) {
                const size_t line = (size_t)(out - lane - tab.words) >> 5;
                for (int t = 0; t < m; t += 2) {
                    const int j0 = s + t, j1 = min(t + 1, m - 1) + s;
                    Double2 gL, gT;
                    pair_fine2<DIM, KERNEL, ISO>(pa, __ldg(P + (j0 >= qe ? j0 - len : j0)), __ldg(P + (j1 >= qe ? j1 - len : j1)), k2, sc,
                                                 gL, gT);
                    float2 *o = reinterpret_cast<float2 *>(out + lane) + t * 32;
                    float *low = tab.low + ((line >> 1) + t) * 32 + lane;
                    o[0] = f2(gL.h.x, gT.h.x);
                    low[0] = pack_low(gL.l.x, gT.l.x);
                    if (t + 1 < m) {
                        o[32] = f2(gL.h.y, gT.h.y);
                        low[32] = pack_low(gL.l.y, gT.l.y);
                    }
                }
            } else if (VAL == 2) {
                float2 *o2 = reinterpret_cast<float2 *>(out + lane);
                int t = 0;
                for (; t + 1 < m; t += 2) {
                    const int j0 = s + t, j1 = j0 + 1;
                    float2 gL, gT;
                    pair_shape2<DIM, KERNEL, ISO>(pa, __ldg(P + (j0 >= qe ? j0 - len : j0)), __ldg(P + (j1 >= qe ? j1 - len : j1)),
                                                  k2, sc, gL, gT);
                    o2[t * 32] = f2(gL.x, gT.x);
                    o2[(t + 1) * 32] = f2(gL.y, gT.y);
                }
                if (t < m) {
                    const int j = s + t;
                    o2[t * 32] = pair_shape<DIM, KERNEL, ISO>(pa, __ldg(P + (j >= qe ? j - len : j)), k2, sc);
                }
            } else if (__any_sync(kFull, s + m > qe)) {
                rs = row_weights<DIM, KERNEL, ISO, true, true>(P, pa, Ca, k, k2, s, m, qe, len, out);
            } else if ((wb >> 24) != 0) {
                rs = row_weights<DIM, KERNEL, ISO, true, false>(P, pa, Ca, k, k2, s, m, qe, len, out);
            } else {
                rs = row_weights<DIM, KERNEL, ISO, false, false>(P, pa, Ca, k, k2, s, m, qe, len, out);
            }
            out += m * 32 * VAL;
            neumaier_add(acc, comp, rs);
        });
        if (used <= room || attempt == 1) break;
        // outgrown: once more into the pool
        unsigned at = 0u;
        if (lane == 0)
            at = claim_lines(atomicAdd(tab.cursor, (unsigned long long)used), tab.cap, used);
        at = __shfl_sync(kFull, at, 0);
        if (at == kNoRoom) {
            room = 0u;
            break;
        }
        base = tab.pool + at;
        room = used;
    }
    if (lane == 0) tab.slots[2 * (size_t)c.slot] = make_uint4(used <= room ? base : kNoRoom, R, used, hs);
    if (VAL == 1 && used > room) return walk_chunk<DIM, KERNEL, ISO>(P, cs, prm, c, nullptr);
    return acc + comp;
}

// Weights are read once per evaluation: keep them out of L1, where the concentrations live.
__device__ __forceinline__ float ld_weight(const float *p)
{
    float v;
    asm("ld.global.nc.L1::no_allocate.f32 %0, [%1];" : "=f"(v) : "l"(p));
    return v;
}

__device__ __forceinline__ void prefetch_l2(const void *p, unsigned bytes)
{
    asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(p), "r"(bytes) : "memory");
}

// Streams one chunk's rows through `op`: op.lines<M>(w, s) takes M values per lane (w: the lane's
// first, the next 32 VAL words on) of the candidates s, s + 1, ... in the doubled arrays, with every
// load of the M in flight at once; op.end_row() closes a row.  Lane 0 keeps the stream kAhead lines
// ahead in L2 with bulk prefetches; the next row's first indices are loaded before the current
// row's lines.  Bound: memory.  Per evaluation of the 128^3 cube: a loop of four predicated lines 723 us
// (latency), the switch on the row's length 559, with the prefetches and the early index line 418.  A ring
// in shared memory filled by asynchronous copies was slower on the cube and at 1024^2 (fewer warps) and
// 6 % faster at 512^2 only.
constexpr int kAhead = 32, kPiece = 16;   // lines

template <int VAL, class Op>
__device__ __forceinline__ void stream_rows(const uint4 sl, const FrozenTab &tab, Op &op)
{
    const int lane = threadIdx.x & 31;
    const int R = (int)sl.y;
    const float *base = tab.words + (size_t)sl.x * 32;
    const float *w = base + lane;
    const int total = (int)sl.z;
    int ahead = min(total, kAhead);
    if (lane == 0) {
        prefetch_l2(base, (unsigned)ahead * 128u);
        op.prefetch(base, 0, ahead);
    }
    const float *hdr = w;
    w += (size_t)sl.w * 32;
    int hm = 0;
    float s = ld_weight(w);
    for (int r = 0; r < R; ++r) {
        if ((r & 31) == 0) hm = __float_as_int(ld_weight(hdr + r));
        const int m = __shfl_sync(kFull, hm, r & 31);
        int j = __float_as_int(s);
        const float *wl = w + 32 + (VAL - 1) * lane;
        w += 32 + m * (32 * VAL);
        if (r + 1 < R) s = ld_weight(w);
        const int pos = (int)((w - base) >> 5);
        if (ahead < total && pos + kAhead > ahead + kPiece) {
            const int n = min(total - ahead, pos + kAhead - ahead);
            if (lane == 0) {
                prefetch_l2(base + (size_t)ahead * 32, (unsigned)n * 128u);
                op.prefetch(base, ahead, n);
            }
            ahead += n;
        }
        int k = m;
        for (; k > 8; k -= 8, wl += 256 * VAL, j += 8) op.template lines<8>(wl, j);
        switch (k) {
        case 1: op.template lines<1>(wl, j); break;
        case 2: op.template lines<2>(wl, j); break;
        case 3: op.template lines<3>(wl, j); break;
        case 4: op.template lines<4>(wl, j); break;
        case 5: op.template lines<5>(wl, j); break;
        case 6: op.template lines<6>(wl, j); break;
        case 7: op.template lines<7>(wl, j); break;
        default: op.template lines<8>(wl, j); break;
        }
        op.end_row();
    }
}

// sum_b w_ab (C_a - C_b) from the table's weights.
struct WeightedSum {
    const float *C;
    float Ca, rs, acc, comp;
    __device__ __forceinline__ void prefetch(const float *, int, int) const {}
    template <int M>
    __device__ __forceinline__ void lines(const float *w, int s)
    {
        const float *Cr = C + s;
        float wv[M], cv[M];
#pragma unroll
        for (int u = 0; u < M; ++u) {
            wv[u] = ld_weight(w + u * 32);
            cv[u] = Cr[u];
        }
#pragma unroll
        for (int u = 0; u < M; ++u) rs = fmaf(wv[u], Ca - cv[u], rs);
    }
    __device__ __forceinline__ void end_row()
    {
        neumaier_add(acc, comp, rs);
        rs = 0.f;
    }
};

__device__ __forceinline__ float stream_chunk(const uint4 sl, const FrozenTab &tab, const float *C, float Ca)
{
    WeightedSum op{C, Ca, 0.f, 0.f, 0.f};
    stream_rows<1>(sl, tab, op);
    return op.acc + op.comp;
}

// rate_frozen.cu -- Eq. 4-5 for several evaluations over one cell list.
//
// In a uniform flow every particle drifts by the same fixed-point word, so the separations -- and
// with them every weight w_ab of dC_a/dt = sum_b w_ab (C_a - C_b) -- do not change during a run:
// only C does.  A call that evaluates Eq. 4 more than a few times therefore computes the weights
// once (k_frozen_build, the pair arithmetic of the walks) into a table in the weights buffer and each
// evaluation streams them (k_frozen_rate): 4 bytes, two loads and two FP32 operations per pair
// instead of about 39 instructions.  The table belongs to one call: it is rebuilt from the
// positions by every call that uses it.
//
// The table's layout is described in frozen_table.cuh.
//
// The arithmetic of each weight, the order of the sum inside a row (FP32) and over the rows
// (Neumaier) are those of the branch-free walks of rate.cu, and every candidate left out has
// weight exactly 0, so the results are bitwise those of the walks over the same cells.
#include "ade_internal.h"

namespace ade {

namespace {

#include "rate_common.cuh"

#include "rate_walk.cuh"

#include "frozen_table.cuh"

constexpr int kT = kFrozenThreads;

// Predictor (C -> Ch) or corrector (C updated from the rate at Ch) of one particle, Eq. 8-9, or the
// same for Cattaneo's (C, Q), Eq. 14 (see epilogue in rate_walk.cuh); Cl, ql: C and Q at level l.
template <int EPI>
__device__ __forceinline__ void frozen_epilogue(const RateParams &prm, const FrozenState &st, const Chunk &c, int i,
                                                float rate, float Cl, float ql)
{
    float dC = rate;
    if (EPI == EPI_PREDICT) {
        if (st.Qs) {
            st.Qh[i] = fmaf(prm.dt, (rate - ql) * st.tau_inv, ql);
            dC = ql;
        }
        st.Ch[c.ps + i] = st.Ch[c.pe + i] = fmaf(prm.dt, dC, Cl);
    } else {
        if (st.Qs) {
            const float qh = st.Qh[i];
            st.Qs[i] = fmaf(prm.dt, (rate - qh) * st.tau_inv, ql);
            dC = qh;
        }
        st.C[c.ps + i] = st.C[c.pe + i] = fmaf(prm.dt, dC, Cl);
    }
}

// The table and the first predictor.
template <int DIM, int KERNEL, bool ISO>
__global__ __launch_bounds__(kT) void k_frozen_build(const uint4 *__restrict__ P, const uint32_t *__restrict__ cs,
                                                     const uint32_t *__restrict__ perm, const RateParams prm,
                                                     const FrozenTab tab, const FrozenState st)
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
    const float sum = build_chunk<DIM, KERNEL, ISO, ISO ? kCutBox : kCutFull, 1>(P, cs, prm, c, pa, srow, tab);
    if (i >= c.pe) return;
    const float Cl = __uint_as_float(pa.w);
    st.C[c.ps + i] = st.C[c.pe + i] = Cl;
    float ql = 0.f;
    if (st.Qs) {
        const uint32_t a = __ldg(perm + i);
        ql = a < (uint32_t)prm.n ? st.Q[a] : 0.f;
        st.Qs[i] = ql;
    }
    frozen_epilogue<EPI_PREDICT>(prm, st, c, i, prm.upf * shape_unscale<KERNEL>() * sum, Cl, ql);
}

// One evaluation from the table.  Bound: HBM where the table exceeds L2 (4 bytes per pair and the idle
// tails of rows), latency below.  Per evaluation, tuned walk / table (ncu, cold caches): 128^3 cube, 250
// neighbours, 700 / 418 us (2.6 GB, 6.2 TB/s of the 6.7 a copy reaches); 1024^2, 120 neighbours 124 / 98; 512^2,
// 60 about 35 / 22; 256^2, 28 16 / 10.  The loads in flight are what the stream lives on: CTAS per SM, 12
// (40 registers), but 16 (32, of which three words spill) between one wave and kWideFrom chunk numbers, where a
// last wave that is nearly empty weighs more (per step, 12 / 16: 512^2 41.8 / 36.3 us, 64^3 175 / 163, 72^3 272 /
// 253; outside of that 256^2 14.1 / 14.8, 45^3 67 / 69, 100^3 595 / 601, 128^3 955 / 961).
constexpr int kWideFrom = 4 * 152 * 48;
template <int DIM, int KERNEL, bool ISO, int EPI, int CTAS>
__global__ __launch_bounds__(kT, CTAS) void k_frozen_rate(const uint4 *__restrict__ P, const uint32_t *__restrict__ cs,
                                                    const RateParams prm, const FrozenTab tab, const FrozenState st)
{
    pdl_wait();
    Chunk c;
    uint4 sl;
    if (!my_chunk(tab, prm, c, sl)) return;
    const float *Ce = EPI == EPI_PREDICT ? st.C : st.Ch;
    const int i = c.i0 + (threadIdx.x & 31);
    const float sum = sl.x != kNoRoom ? stream_chunk(sl, tab, Ce, Ce[c.ps + min(i, c.pe - 1)])
                                      : walk_chunk<DIM, KERNEL, ISO>(P, cs, prm, c, Ce);
    if (i >= c.pe) return;
    frozen_epilogue<EPI>(prm, st, c, i, prm.upf * shape_unscale<KERNEL>() * sum, st.C[c.ps + i], st.Qs ? st.Qs[i] : 0.f);
}

// Batched plumes: one chunk of one plume per warp (the cell table and the sorted arrays are the batch's; no
// pencil boxes).
template <int DIM, int KERNEL>
__global__ __launch_bounds__(kT) void k_frozen_build_batch(const uint4 *__restrict__ P, const uint32_t *__restrict__ cs,
                                                           const RateParams *__restrict__ descs,
                                                           const FrozenItem *__restrict__ items, int nitems,
                                                           const FrozenTab tab, const FrozenState st)
{
    pdl_wait();
    const int w = blockIdx.x * (kT / 32) + (threadIdx.x >> 5);
    if (w >= nitems) return;
    const FrozenItem it = items[w];
    const RateParams &prm = descs[it.plume];
    Chunk c;
    const bool has = find_chunk(cs + prm.coff, prm, nullptr, it.chunk, c);
    c.slot = w;
    put_chunk(tab, c, has);
    if (!has) return;
    const int i = c.i0 + (threadIdx.x & 31);
    const uint4 pa = __ldg(P + min(i, c.pe - 1));
    const float sum = build_chunk<DIM, KERNEL, true, kCutBand, 1>(P, cs + prm.coff, prm, c, pa, nullptr, tab);
    if (i >= c.pe) return;
    const float Cl = __uint_as_float(pa.w);
    st.C[c.ps + i] = st.C[c.pe + i] = Cl;
    frozen_epilogue<EPI_PREDICT>(prm, st, c, i, prm.upf * shape_unscale<KERNEL>() * sum, Cl, 0.f);
}

template <int DIM, int KERNEL, int EPI>
__global__ __launch_bounds__(kT, 12) void k_frozen_rate_batch(const uint4 *__restrict__ P, const uint32_t *__restrict__ cs,
                                                              const RateParams *__restrict__ descs,
                                                              const FrozenItem *__restrict__ items, int nitems,
                                                              const FrozenTab tab, const FrozenState st)
{
    pdl_wait();
    const int w = blockIdx.x * (kT / 32) + (threadIdx.x >> 5);
    if (w >= nitems) return;
    const RateParams &prm = descs[items[w].plume];
    Chunk c;
    uint4 sl;
    if (!get_chunk(tab, prm, w, c, sl)) return;
    const float *Ce = EPI == EPI_PREDICT ? st.C : st.Ch;
    const int i = c.i0 + (threadIdx.x & 31);
    const float sum = sl.x != kNoRoom ? stream_chunk(sl, tab, Ce, Ce[c.ps + min(i, c.pe - 1)])
                                      : walk_chunk<DIM, KERNEL, true>(P, cs + prm.coff, prm, c, Ce);
    if (i >= c.pe) return;
    frozen_epilogue<EPI>(prm, st, c, i, prm.upf * shape_unscale<KERNEL>() * sum, st.C[c.ps + i], 0.f);
}

// Lines one chunk needs (the rows and ranges of build_chunk) into two bins per octave.
template <int DIM, bool ISO, int CUT>
__device__ __forceinline__ void bin_chunk(const uint4 *__restrict__ P, const uint32_t *__restrict__ cs, const RateParams &prm,
                                          const Chunk &c, const TrimRow *srow, int val, ChunkBin *__restrict__ bins)
{
    const int lane = threadIdx.x & 31;
    const uint4 pa = __ldg(P + min(c.i0 + lane, c.pe - 1));
    unsigned used = header_lines(prm);
    chunk_rows<DIM, ISO, CUT>(P, cs, prm, c, pa, srow,
                              [&](int, int, int, int m, int) { used = add_lines(used, 1u + (unsigned)(m * val)); });
    if (lane != 0) return;
    const int top = 31 - __clz((int)used);
    ChunkBin *b = bins + 2 * top + (top > 0 ? (used >> (top - 1)) & 1 : 0);
    atomicAdd(&b->count, 1u);
    atomicMax(&b->most, used);
    atomicAdd(&b->sum, (unsigned long long)used);
}

template <int DIM, bool ISO>
__global__ __launch_bounds__(kT) void k_chunk_need(const uint4 *__restrict__ P, const uint32_t *__restrict__ cs,
                                                   const RateParams prm, int val, ChunkBin *__restrict__ bins)
{
    pdl_wait();
    __shared__ TrimRow srow[ISO ? kMaxRows : 1];
    if (ISO) stage_trim_rows(srow, prm);
    Chunk c;
    if (find_chunk(cs, prm, nullptr, warp_number(), c)) bin_chunk<DIM, ISO, ISO ? kCutBox : kCutFull>(P, cs, prm, c, srow, val, bins);
}

template <int DIM>
__global__ __launch_bounds__(kT) void k_chunk_need_batch(const uint4 *__restrict__ P, const uint32_t *__restrict__ cs,
                                                         const RateParams *__restrict__ descs, const FrozenItem *__restrict__ items,
                                                         int first, int last, ChunkBin *__restrict__ bins)
{
    pdl_wait();
    const int w = first + warp_number();
    if (w >= last) return;
    const FrozenItem it = items[w];
    const RateParams &prm = descs[it.plume];
    Chunk c;
    if (find_chunk(cs + prm.coff, prm, nullptr, it.chunk, c))
        bin_chunk<DIM, true, kCutBand>(P, cs + prm.coff, prm, c, nullptr, 1, bins + (size_t)(it.plume - items[first].plume) * kChunkBins);
}

constexpr int kCountT = 1024, kCountItems = 16;

// Chunks before each pencil: one block, kCountItems pencils per thread at a time (their loads in flight
// together: 16,384 pencils in one go).
__global__ __launch_bounds__(kCountT) void k_chunk_numbers(const uint32_t *__restrict__ cs, int np, int ncx,
                                                           uint32_t *__restrict__ dense)
{
    pdl_wait();
    __shared__ uint32_t warp_sum[kCountT / 32];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    uint32_t carry = 0u;
    for (int base = 0; base < np; base += kCountT * kCountItems) {
        const int q0 = base + (int)threadIdx.x * kCountItems;
        uint32_t at[kCountItems + 1], sum = 0u;
#pragma unroll
        for (int k = 0; k <= kCountItems; ++k) at[k] = __ldg(cs + (size_t)min(q0 + k, np) * ncx);
#pragma unroll
        for (int k = 0; k < kCountItems; ++k) sum += (at[k + 1] - at[k] + 31u) >> 5;
        uint32_t incl = sum;
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t v = __shfl_up_sync(kFull, incl, o);
            incl += lane >= o ? v : 0u;
        }
        if (lane == 31) warp_sum[wid] = incl;
        __syncthreads();
        uint32_t run = carry + incl - sum;
        for (int w = 0; w < kCountT / 32; ++w) {
            run += w < wid ? warp_sum[w] : 0u;
            carry += warp_sum[w];
        }
#pragma unroll
        for (int k = 0; k < kCountItems; ++k) {
            if (q0 + k < np) dense[q0 + k] = run;
            run += (at[k + 1] - at[k] + 31u) >> 5;
        }
        __syncthreads();
    }
    if (threadIdx.x == 0) dense[np] = carry;
}

// The state after `steps` steps of every plume, in the caller's order (descs: the correctors').
template <int DIM>
__global__ __launch_bounds__(kT) void k_frozen_finish_batch(const uint4 *__restrict__ P, const uint32_t *__restrict__ cs,
                                                            const uint32_t *__restrict__ perm, int n,
                                                            const RateParams *__restrict__ descs,
                                                            const uint16_t *__restrict__ plume_of, uint32_t steps,
                                                            const FrozenTab tab, const FrozenState st, const EpiOut out)
{
    pdl_wait();
    pdl_trigger();
    const int i = blockIdx.x * kT + threadIdx.x;
    if (i == 0) *tab.cursor = 0ull;
    if (i >= n) return;
    const uint32_t a = __ldg(perm + i);
    if (a >= (uint32_t)n) return;
    const RateParams &prm = descs[__ldg(plume_of + a)];
    const uint4 p = __ldg(P + i);
    const uint32_t *f = prm.frame + 4;
    const int cy = (int)__umulhi(p.y - f[1], (uint32_t)prm.ncy);
    const int cz = DIM == 3 ? (int)__umulhi(p.z - f[2], (uint32_t)prm.ncz) : 0;
    const float Cn = st.C[(int)__ldg(cs + prm.coff + (size_t)(cz * prm.ncy + cy) * prm.ncx) + i];
    uint32_t *xp = out.xq + (size_t)prm.goff * DIM;
    const uint32_t l = a - (uint32_t)prm.goff;
    out.C[a] = Cn;
    xp[l] = p.x + steps * prm.inc[0];
    xp[(size_t)prm.n + l] = p.y + steps * prm.inc[1];
    if (DIM == 3) xp[2 * (size_t)prm.n + l] = p.z + steps * prm.inc[2];
    if (!isfinite(Cn)) atomicOr(out.status, 1);
}

// The state after the call's steps, in the caller's order: C, Q, positions advanced by `inc` (the
// drift of all steps), the non-finite flag (a non-finite C stays non-finite in every later step), and
// one partial of the statistics per warp.
template <int DIM>
__global__ __launch_bounds__(kT) void k_frozen_finish(const uint4 *__restrict__ P, const uint32_t *__restrict__ cs,
                                                      const uint32_t *__restrict__ perm, const RateParams prm,
                                                      const FrozenTab tab, const FrozenState st, const EpiOut out)
{
    pdl_wait();
    pdl_trigger();
    const int i = blockIdx.x * kT + threadIdx.x;
    if (i == 0) *tab.cursor = 0ull;   // the next call's table starts empty
    Acc acc{0.f, 0.f, __int_as_float(0x7f800000), __int_as_float(0xff800000), 0u};
    if (i < prm.n) {
        const uint32_t a = __ldg(perm + i);
        const uint4 p = __ldg(P + i);
        // the start of the particle's pencil places it in the doubled concentrations
        const uint3 org = cell_origin(prm);
        const int cy = (int)__umulhi(p.y - org.y, (uint32_t)prm.ncy);
        const int cz = DIM == 3 ? (int)__umulhi(p.z - org.z, (uint32_t)prm.ncz) : 0;
        const float Cn = st.C[(int)__ldg(cs + (size_t)(cz * prm.ncy + cy) * prm.ncx) + i];
        if (a < (uint32_t)prm.n) {
            out.C[a] = Cn;
            out.xq[a] = p.x + prm.inc[0];
            out.xq[(size_t)prm.n + a] = p.y + prm.inc[1];
            if (DIM == 3) out.xq[2 * (size_t)prm.n + a] = p.z + prm.inc[2];
            if (st.Qs) st.Q[a] = st.Qs[i];
        }
        if (!isfinite(Cn)) atomicOr(out.status, 1);
        two_sum_add(acc.hi, acc.lo, Cn, 0.f);
        acc.mn = fminf(acc.mn, Cn);
        acc.mx = fmaxf(acc.mx, Cn);
    }
    warp_finish<EPI_CORRECT, false, kT>(acc, out);
}

template <int DIM, int KERNEL, bool ISO>
cudaError_t build_t(const uint4 *P, const uint32_t *cs, const uint32_t *perm, const RateParams &prm,
                    const FrozenTab &tab, const FrozenState &st, cudaStream_t s)
{
    return launch_pdl(k_frozen_build<DIM, KERNEL, ISO>, frozen_blocks(prm), kT, 0, s, P, cs, perm, prm, tab, st);
}

template <int DIM, int KERNEL, bool ISO>
cudaError_t rate_t(int epi, const uint4 *P, const uint32_t *cs, const RateParams &prm, const FrozenTab &tab,
                   const FrozenState &st, cudaStream_t s)
{
    const int numbers = chunk_numbers(prm.n, prm.ncy * prm.ncz);
    auto go = [&](auto kernel) { return launch_pdl(kernel, frozen_blocks(prm), kT, 0, s, P, cs, prm, tab, st); };
    if (numbers <= kCountChunksFrom || numbers > kWideFrom)
        return epi == EPI_PREDICT ? go(k_frozen_rate<DIM, KERNEL, ISO, EPI_PREDICT, 12>) : go(k_frozen_rate<DIM, KERNEL, ISO, EPI_CORRECT, 12>);
    return epi == EPI_PREDICT ? go(k_frozen_rate<DIM, KERNEL, ISO, EPI_PREDICT, 16>) : go(k_frozen_rate<DIM, KERNEL, ISO, EPI_CORRECT, 16>);
}

}  // namespace

unsigned frozen_blocks(const RateParams &prm)
{
    return (unsigned)((chunk_numbers(prm.n, prm.ncy * prm.ncz) + kT / 32 - 1) / (kT / 32));
}

cudaError_t launch_chunk_need(int dim, bool iso, const uint4 *P, const uint32_t *cs, const RateParams &prm, int val,
                              ChunkBin *bins, cudaStream_t s)
{
    auto go = [&](auto kernel) { return launch_pdl(kernel, frozen_blocks(prm), kT, 0, s, P, cs, prm, val, bins); };
    if (iso) return dim == 2 ? go(k_chunk_need<2, true>) : go(k_chunk_need<3, true>);
    return dim == 2 ? go(k_chunk_need<2, false>) : go(k_chunk_need<3, false>);
}

cudaError_t launch_chunk_need_batch(int dim, const uint4 *P, const uint32_t *cs, const RateParams *descs, const FrozenItem *items,
                                    int first, int last, ChunkBin *bins, cudaStream_t s)
{
    if (last <= first) return cudaSuccess;
    const unsigned nb = (unsigned)((last - first + kT / 32 - 1) / (kT / 32));
    return dim == 2 ? launch_pdl(k_chunk_need_batch<2>, nb, kT, 0, s, P, cs, descs, items, first, last, bins)
                    : launch_pdl(k_chunk_need_batch<3>, nb, kT, 0, s, P, cs, descs, items, first, last, bins);
}

cudaError_t launch_chunk_numbers(const uint32_t *cs, const RateParams &prm, uint32_t *dense, cudaStream_t s)
{
    if (!dense) return cudaSuccess;
    return launch_pdl(k_chunk_numbers, 1u, kCountT, 0, s, cs, prm.ncy * prm.ncz, prm.ncx, dense);
}

cudaError_t launch_frozen_build(int dim, int kernel, bool iso, const uint4 *P, const uint32_t *cs, const uint32_t *perm,
                                const RateParams &prm, const FrozenTab &tab, const FrozenState &st, cudaStream_t s)
{
#define ADE_CALL(D, K) (iso ? build_t<D, K, true>(P, cs, perm, prm, tab, st, s) : build_t<D, K, false>(P, cs, perm, prm, tab, st, s))
    if (dim == 2) return kernel == ADE_WENDLAND_C2 ? ADE_CALL(2, ADE_WENDLAND_C2) : ADE_CALL(2, ADE_WENDLAND_C4);
    return kernel == ADE_WENDLAND_C2 ? ADE_CALL(3, ADE_WENDLAND_C2) : ADE_CALL(3, ADE_WENDLAND_C4);
#undef ADE_CALL
}

cudaError_t launch_frozen_rate(int dim, int kernel, bool iso, int epi, const uint4 *P, const uint32_t *cs,
                               const RateParams &prm, const FrozenTab &tab, const FrozenState &st, cudaStream_t s)
{
#define ADE_CALL(D, K) (iso ? rate_t<D, K, true>(epi, P, cs, prm, tab, st, s) : rate_t<D, K, false>(epi, P, cs, prm, tab, st, s))
    if (dim == 2) return kernel == ADE_WENDLAND_C2 ? ADE_CALL(2, ADE_WENDLAND_C2) : ADE_CALL(2, ADE_WENDLAND_C4);
    return kernel == ADE_WENDLAND_C2 ? ADE_CALL(3, ADE_WENDLAND_C2) : ADE_CALL(3, ADE_WENDLAND_C4);
#undef ADE_CALL
}

cudaError_t launch_frozen_batch(int dim, int kernel, int epi, bool build, const uint4 *P, const uint32_t *cs,
                                const RateParams *descs, const FrozenItem *items, int nitems, const FrozenTab &tab,
                                const FrozenState &st, cudaStream_t s)
{
    const unsigned nb = (unsigned)((nitems + kT / 32 - 1) / (kT / 32));
#define ADE_CALL(D, K)                                                                                              \
    (build ? launch_pdl(k_frozen_build_batch<D, K>, nb, kT, 0, s, P, cs, descs, items, nitems, tab, st)             \
           : (epi == EPI_PREDICT                                                                                    \
                  ? launch_pdl(k_frozen_rate_batch<D, K, EPI_PREDICT>, nb, kT, 0, s, P, cs, descs, items, nitems, tab, st) \
                  : launch_pdl(k_frozen_rate_batch<D, K, EPI_CORRECT>, nb, kT, 0, s, P, cs, descs, items, nitems, tab, st)))
    if (dim == 2) return kernel == ADE_WENDLAND_C2 ? ADE_CALL(2, ADE_WENDLAND_C2) : ADE_CALL(2, ADE_WENDLAND_C4);
    return kernel == ADE_WENDLAND_C2 ? ADE_CALL(3, ADE_WENDLAND_C2) : ADE_CALL(3, ADE_WENDLAND_C4);
#undef ADE_CALL
}

cudaError_t launch_frozen_finish_batch(int dim, const uint4 *P, const uint32_t *cs, const uint32_t *perm, int n,
                                       const RateParams *descs, const uint16_t *plume_of, uint32_t steps,
                                       const FrozenTab &tab, const FrozenState &st, const EpiOut &out, cudaStream_t s)
{
    const unsigned nb = (unsigned)((n + kT - 1) / kT);
    return dim == 2 ? launch_pdl(k_frozen_finish_batch<2>, nb, kT, 0, s, P, cs, perm, n, descs, plume_of, steps, tab, st, out)
                    : launch_pdl(k_frozen_finish_batch<3>, nb, kT, 0, s, P, cs, perm, n, descs, plume_of, steps, tab, st, out);
}

cudaError_t launch_frozen_finish(int dim, const uint4 *P, const uint32_t *cs, const uint32_t *perm, const RateParams &prm,
                                 const FrozenTab &tab, const FrozenState &st, const EpiOut &out, cudaStream_t s)
{
    const unsigned nb = (unsigned)((prm.n + kT - 1) / kT);
    return dim == 2 ? launch_pdl(k_frozen_finish<2>, nb, kT, 0, s, P, cs, perm, prm, tab, st, out)
                    : launch_pdl(k_frozen_finish<3>, nb, kT, 0, s, P, cs, perm, prm, tab, st, out);
}

}  // namespace ade

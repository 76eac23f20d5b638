// Double-float ("df64") all-pairs quadrature: the FP64-accurate residual on
// the FP32 pipes.
//
// GB300 executes two FP64 fused multiply-adds per SM per clock against 128 in
// FP32, so the FP64 pair kernel is bound by that pipe.  Here every FP64 quantity
// of the pair sum is carried as an unevaluated sum hi + lo of two floats
// (Dekker 1971; Knuth's two-sum; two-product by fused multiply-add), which
// keeps about 46 significant bits: per term a relative error near 1e-13,
// well inside the 1e-10 per-row parity bar of the FP64 residual.  The sums
// are the same four sheet pairings, singularity subtractions and S2 term as
// the FP64 and FP32C kernels (Sec. 2.2 and 3.1 of the paper).
//
// The kernel is bound by the FMA pipe (two sources per instruction, packed
// FP32x2), so its cost is the number of FP32 operations per index pair: 321 on
// meshes with dx == dy, about 370 otherwise (659 single instructions before).
// 181 x 61: 2.29 -> 1.19 ms per launch with the pipe 82 % busy; 281 x 281:
// 117 -> 60 ms.  Occupancies from 3 to 6 CTAs per SM measure the same within 1 %.
// What keeps the count down:
//   - Horizontal offsets are exact: records carry the node column and row in
//     mesh units (half-integers), so with dx == dy s^2 + t^2 is one exact float
//     (SQ), else an exact s^2 plus (dy/dx)^2 t^2 in double-float.
//   - Weights cx cy (1, 1/2 or 1/4) are exact; the common factors dy/dx and dy
//     are applied to the finished sums.
//   - The slope terms s zeta_x + t zeta_y are formed once per source sheet.
//   - 1/r, 1/r^2 share one residual e = 1 - a y0^2 of the FP32 seed y0:
//     1/r = y0 (1 + e/2 + 3 e^2/8), 1/r^2 = y0^2 (1 + e + e^2).
//   - Double and single layer of a pairing share one accumulation,
//     (t / r^2 + w zeta_x) / r.
// Renormalisation is left out inside a term: a low part may reach about 2^-22 of
// the operands its high part came from, and products drop low times low part.  That
// is too much for the difference of two heights of one sheet that are many cells high,
// where little is left of the high parts: it is renormalised (2 % more operations)
// where a height of the residual at hand exceeds DF_HIGH = 16 cells.  Largest error of
// a term without | with it: 2e-14 | 1e-14 at a third of a cell, 4e-13 | 4e-14 at 3.5 cells,
// 5e-12 | 4e-13 at 50, 1.3e-9 | 7e-12 at 512 (the last is the rounding of the heights).  The three accumulators, whose low parts
// collect one rounding error per term, are renormalised every fourth source pair
// (without that the 281 x 281 residual loses two bits).
#include <math.h>

#include "bfs_internal.cuh"

namespace bfs {

// A pair of double-float values: hi + lo for two sources.
struct df2 {
    f2 h, l;
};

// a + b: Knuth's two-sum of the high parts, the error and the low parts added
__device__ __forceinline__ df2 d2_add(df2 a, df2 b)
{
    const f2 s = f2_add(a.h, b.h);
    const f2 bb = f2_sub(s, a.h);
    const f2 e = f2_add(f2_sub(a.h, f2_sub(s, bb)), f2_sub(b.h, bb));
    return df2{s, f2_add(e, f2_add(a.l, b.l))};
}

__device__ __forceinline__ df2 d2_sub(df2 a, df2 b)
{
    const f2 s = f2_sub(a.h, b.h);
    const f2 bb = f2_sub(s, a.h);
    const f2 e = f2_sub(f2_sub(a.h, f2_sub(s, bb)), f2_add(b.h, bb));
    return df2{s, f2_add(e, f2_sub(a.l, b.l))};
}

// a b: two-product of the high parts, the cross terms added
__device__ __forceinline__ df2 d2_mul(df2 a, df2 b)
{
    const f2 p = f2_mul(a.h, b.h);
    f2 e = f2_fma(a.h, b.h, f2_neg(p));
    e = f2_fma(a.h, b.l, e);
    return df2{p, f2_fma(a.l, b.h, e)};
}

// x s + y t for float s, t
__device__ __forceinline__ df2 d2_slope(df2 x, f2 s, df2 y, f2 t)
{
    const f2 p = f2_mul(x.h, s), q = f2_mul(y.h, t);
    f2 e = f2_fma(x.l, s, f2_fma(x.h, s, f2_neg(p)));
    e = f2_add(e, f2_fma(y.l, t, f2_fma(y.h, t, f2_neg(q))));
    const f2 v = f2_add(p, q);
    const f2 bb = f2_sub(v, p);
    const f2 r = f2_add(f2_sub(p, f2_sub(v, bb)), f2_sub(q, bb));
    return df2{v, f2_add(r, e)};
}

// a = s^2 + t^2 + d^2.  SQ: rho2 is an exact multiple of 1/4, so rho2 - a.h is
// exact (Sterbenz's lemma while d^2 <= rho2; beyond that both are multiples of
// the spacing of a.h as long as a.h < 2^22, which |d| <= DF_EXACT ensures: a.h is then
// at most 2 d^2) and one FMA gives the rest of d.h^2.  Past that a pair would be good to
// about 2^-24 only.
template <bool SQ>
__device__ __forceinline__ df2 d2_r2(df2 rho2, df2 d)
{
    if constexpr (SQ) {
        const f2 a = f2_fma(d.h, d.h, rho2.h);
        const f2 e = f2_fma(d.h, d.h, f2_sub(rho2.h, a));
        return df2{a, f2_fma(f2_add(d.h, d.h), d.l, e)};
    } else {
        const f2 p = f2_mul(d.h, d.h);
        const f2 e = f2_fma(f2_add(d.h, d.h), d.l, f2_fma(d.h, d.h, f2_neg(p)));
        return d2_add(rho2, df2{p, e});
    }
}

// The FP32 seed y0 of 1/sqrt(a), p + q = y0^2 exactly and m = a y0^2 - 1
// (below 2^-21; the first FMA rounds a product within 2^-21 of 1 to about
// 2^-46, the low parts follow).
struct Seed {
    f2 y, p, q, m;
};

__device__ __forceinline__ Seed d2_seed(df2 a)
{
    Seed s;
    s.y = f2_rsq(a.h);
    s.p = f2_mul(s.y, s.y);
    s.q = f2_fma(s.y, s.y, f2_neg(s.p));
    s.m = f2_fma(a.h, s.p, f2_both(-1.f));
    s.m = f2_fma(a.h, s.q, s.m);
    s.m = f2_fma(a.l, s.p, s.m);
    return s;
}

// 1/sqrt(a) and 1/a from the seed
__device__ __forceinline__ df2 d2_inv_r(const Seed &s)
{
    return df2{s.y, f2_mul(f2_mul(s.y, s.m), f2_fma(s.m, f2_both(0.375f), f2_both(-0.5f)))};
}

__device__ __forceinline__ df2 d2_inv_r2(const Seed &s)
{
    return df2{s.p, f2_fma(f2_mul(s.p, s.m), f2_add(s.m, f2_both(-1.f)), s.q)};
}

// the low part back within half a unit of the high one (|h| >= |l|)
__device__ __forceinline__ df2 d2_norm(df2 a)
{
    const f2 s = f2_add(a.h, a.l);
    return df2{s, f2_sub(a.l, f2_sub(s, a.h))};
}

__device__ __forceinline__ df2 both2(const float *p) { return df2{f2_both(p[0]), f2_both(p[1])}; }

constexpr int PDF_TPB = 128, PDF_CH = 64;

// Records: source pairs interleaved (value v of sources 2i and 2i+1 side by
// side), see DSRC in bfs_internal.cuh; targets DTGT floats each.  HIGH: heights beyond
// DF_HIGH.
template <bool SQ, bool HIGH>
__device__ __forceinline__ void pair_tile_df(const float *__restrict__ src, int per_split, const float *__restrict__ tgt,
                                             int Nt, double *__restrict__ part, float ry2h, float ry2l, double ry,
                                             double dy, float *sh)
{
    auto diff = [](df2 a, df2 b) {
        if constexpr (HIGH) return d2_norm(d2_sub(a, b));
        else return d2_sub(a, b);
    };
    const int split = blockIdx.y;
    const float *sb = src + (size_t)split * per_split * DSRC;
    const int t = blockIdx.x * PDF_TPB + threadIdx.x;
    const float *tr = tgt + (size_t)min(t, Nt - 1) * DTGT;
    const f2 tx = f2_both(tr[0]), ty = f2_both(tr[1]);
    const df2 tz = both2(tr + 2), cTB = both2(tr + 4), cBT = both2(tr + 6), tB = both2(tr + 8);
    const df2 ntf = df2{f2_both(-tr[10]), f2_both(-tr[11])}, ntg = df2{f2_both(-tr[12]), f2_both(-tr[13])};
    const df2 tzx = both2(tr + 14), tzy = both2(tr + 16);
    const df2 zero = df2{f2_both(0.f), f2_both(0.f)};
    df2 aT = zero, aS = zero, aB = zero;

    for (int c0 = 0; c0 < per_split; c0 += PDF_CH) {
        const int nc = min(PDF_CH, per_split - c0);
        __syncthreads();
        const float4 *g = reinterpret_cast<const float4 *>(sb + (size_t)c0 * DSRC);
        float4 *sv = reinterpret_cast<float4 *>(sh);
        for (int e = threadIdx.x; e < nc * DSRC / 4; e += PDF_TPB) sv[e] = g[e];
        __syncthreads();
#pragma unroll 1
        for (int i = 0; i < nc / 2; i++) {
            const f2 *r = reinterpret_cast<const f2 *>(sh) + i * DSRC;
            auto val = [&](int k) { return df2{r[k], r[k + 1]}; };
            const f2 sx = f2_sub(r[0], tx);  // exact: half-integer mesh offsets
            const f2 dj = f2_sub(r[1], ty);  // exact: integer row offset
            df2 rho2;
            if constexpr (SQ) {
                rho2 = df2{f2_fma(dj, dj, f2_mul(sx, sx)), f2_both(0.f)};
            } else {
                const f2 sxx = f2_mul(sx, sx), djj = f2_mul(dj, dj);  // exact
                rho2 = d2_add(d2_mul(df2{f2_both(ry2h), f2_both(ry2l)}, df2{djj, f2_both(0.f)}),
                              df2{sxx, f2_both(0.f)});
            }
            const df2 zs = val(2), bs = val(4), w1f = val(14), w1g = val(16);
            const f2 cw = r[22];
            // w S2 at the top target: A s^2 + B s t + C t^2 = s^2 + t^2 + (zeta_x* s + zeta_y* t)^2
            {
                const df2 ri = d2_inv_r(d2_seed(d2_r2<SQ>(rho2, d2_slope(tzx, sx, tzy, dj))));
                aS = d2_add(aS, df2{f2_mul(cw, ri.h), f2_mul(cw, ri.l)});
            }
            const df2 gt = d2_slope(val(6), sx, val(8), dj);
            const df2 zxd = val(18);
            // top target, top source: w (f - f*) K1 + w zeta_x K2
            {
                const df2 d = diff(zs, tz);
                const Seed s = d2_seed(d2_r2<SQ>(rho2, d));
                // w f - w f*: w is a power of two, so the product is exact
                const f2 v = f2_fma(ntf.h, cw, w1f.h);
                const f2 bb = f2_sub(v, w1f.h);
                const f2 e = f2_add(f2_sub(w1f.h, f2_sub(v, bb)), f2_fma(ntf.h, cw, f2_neg(bb)));
                const df2 dens = df2{v, f2_add(e, f2_fma(ntf.l, cw, w1f.l))};
                const df2 u = d2_add(d2_mul(d2_mul(dens, d2_sub(d, gt)), d2_inv_r2(s)), zxd);
                aT = d2_add(aT, d2_mul(u, d2_inv_r(s)));
            }
            // bottom target, top source: w f K1 + w zeta_x K2
            {
                const df2 d = d2_sub(zs, cBT);
                const Seed s = d2_seed(d2_r2<SQ>(rho2, d));
                const df2 u = d2_add(d2_mul(d2_mul(w1f, d2_sub(d, gt)), d2_inv_r2(s)), zxd);
                aB = d2_add(aB, d2_mul(u, d2_inv_r(s)));
            }
            const df2 gb = d2_slope(val(10), sx, val(12), dj);
            // top target, bottom source: -w g K1(beta) + w sigma beta_x K2(beta)
            {
                const df2 d = d2_sub(bs, cTB);
                const Seed s = d2_seed(d2_r2<SQ>(rho2, d));
                const df2 u = d2_add(d2_mul(d2_mul(w1g, d2_sub(gb, d)), d2_inv_r2(s)), val(20));
                aT = d2_add(aT, d2_mul(u, d2_inv_r(s)));
            }
            // bottom target, bottom source: -w (g - g*) K1(beta)
            {
                const df2 d = diff(bs, tB);
                const Seed s = d2_seed(d2_r2<SQ>(rho2, d));
                const f2 v = f2_fma(ntg.h, cw, w1g.h);
                const f2 bb = f2_sub(v, w1g.h);
                const f2 e = f2_add(f2_sub(w1g.h, f2_sub(v, bb)), f2_fma(ntg.h, cw, f2_neg(bb)));
                const df2 dens = df2{v, f2_add(e, f2_fma(ntg.l, cw, w1g.l))};
                aB = d2_add(aB, d2_mul(d2_mul(d2_mul(dens, d2_sub(gb, d)), d2_inv_r2(s)), d2_inv_r(s)));
            }
            if ((i & 3) == 3) {  // the low parts collect one rounding error per term
                aT = d2_norm(aT);
                aS = d2_norm(aS);
                aB = d2_norm(aB);
            }
        }
    }
    if (t >= Nt) return;
    // the two sources' halves joined in FP64, times the factor left out of the weights
    const df2 acc[NACC] = {aT, aS, aB};
#pragma unroll
    for (int q = 0; q < NACC; q++) {
        float h0, h1, l0, l1;
        f2_unpack(acc[q].h, h0, h1);
        f2_unpack(acc[q].l, l0, l1);
        const double v = ((double)h0 + (double)h1) + (double)(l0 + l1);
        part[((size_t)split * NACC + q) * Nt + t] = v * (q == 1 ? dy : ry);
    }
}

template <bool SQ>
__global__ void __launch_bounds__(PDF_TPB, 4)
k_pairs_df(const float *__restrict__ src, int per_split, const float *__restrict__ tgt, int Nt,
           double *__restrict__ part, float ry2h, float ry2l, double ry, double dy, const int *__restrict__ form)
{
    __shared__ __align__(16) float sh[PDF_CH * DSRC];
    if (SQ && form[1]) pair_tile_df<false, true>(src, per_split, tgt, Nt, part, ry2h, ry2l, ry, dy, sh);
    else if (form[0] == 0) pair_tile_df<SQ, false>(src, per_split, tgt, Nt, part, ry2h, ry2l, ry, dy, sh);
    else pair_tile_df<SQ, true>(src, per_split, tgt, Nt, part, ry2h, ry2l, ry, dy, sh);
}

PairPlan plan_df(int Nt, int Ns, int splits_req, int sms)
{
    return fine_plan(Nt, Ns, PDF_TPB, 8, 5, splits_req, sms);
}

int pairs_df_launch(bfs_ctx *c, cudaStream_t s)
{
    const double ryd = c->dy / c->dx, ry2d = ryd * ryd;
    const float ry2h = (float)ry2d, ry2l = (float)(ry2d - (double)ry2h);
    const PairPlan &p = c->plandf;
    const dim3 grid(p.tiles, p.splits);
    // the exact-square form needs s^2 + t^2 within its exact range, and vertical distances
    // too (d2_r2): those are the data's, and the kernel leaves the form by d_flag[2]
    const bool sq = c->dx == c->dy && c->N <= 1024 && c->M <= 512 && c->dx * 1024.0 >= 1.0;
    if (sq)
        k_pairs_df<true><<<grid, PDF_TPB, 0, s>>>(c->d_srcdf, p.per_split, c->d_tgtdf, c->Nt, c->d_part, ry2h,
                                                  ry2l, ryd, c->dy, c->d_flag + 1);
    else
        k_pairs_df<false><<<grid, PDF_TPB, 0, s>>>(c->d_srcdf, p.per_split, c->d_tgtdf, c->Nt, c->d_part, ry2h,
                                                   ry2l, ryd, c->dy, c->d_flag + 1);
    c->launches++;
    BFS_CUDA_TRY(c, cudaGetLastError());
    return BFS_OK;
}

}  // namespace bfs

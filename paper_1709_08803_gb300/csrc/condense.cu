// Static condensation of the slice blocks of the preconditioner (Sec. 4.2,
// App. A, App. B): phi_x is eliminated slice by slice before the block LU.
//
// In the linearised system F1 couples no two slices: its row k reads
//   phi_x*(k) + zeta*(k) / F^2 = r1(k),  phi_x*(k) = (phi_x(k) + phi_x(k+1)) / 2.
// With the radiation row F4 (phi_x at the first two nodes) these N equations
// determine phi_x(1..N) of the slice from its zeta and phi(1).  Nodal phi needs
// no solve at all: phi(k+1) - phi(k) = dx phi_x*(k), so
//   phi(i) = phi(1) + dx sum_{k<i} (r1(k) - zeta*(k) / F^2),
// and phi_x itself follows from phi_x(1) = (r4 - 2 g b(1)) / (n - 2 g) and
// phi_x(k+1) = 2 b(k) - phi_x(k), with b = r1 - zeta* / F^2 and g = x1 / dx.
// What is left per slice are the nb = 2 (N+1) + 1 unknowns
//   [zeta(1), zeta_x(1..N) | phi(1) | psi(1), psi_x(1..N)]
// and equations [F5, F6, F2(1..N-1) | F3 | F8, F9, F7(1..N-1)], with the same
// band: the block LU of the same matrix with the phi_x unknowns taken first.  It
// has 2/3 of the rows, so 4/9 of the bytes each sweep streams (220 instead of
// 496 MB at 181 x 61, h = 3) and 0.30 of the operations of the factorisation.
// The kernels of precond.cu and apply.cu then run on blocks of this size;
// k_cond_scan and k_cond_conv reduce the right-hand side (F2 and F7 lose the
// known part of phi) and k_cond_post recovers phi_x.
//
// Not with surface tension, whose curvature term couples the F1 rows of
// neighbouring slices, nor on coarse meshes at small F, where it costs digits (cond_ok).
//
// The mesh is uniform, so every kernel value depends on the column offset and the
// row distance alone: tables of K5, K7, K6 (row distance x column offset) are
// built once and read by the formation and by k_cond_conv.
#include <math.h>

#include <algorithm>

#include "bfs_internal.cuh"

namespace bfs {

struct CondArgs {
    int N, M, half, h, nb, R, ld;  // R rows of ld = 2 N - 2 offsets per table
    double x1, y1, dx, dy, F, n_rad, xhi, ylo, yhi;
    const double *k5, *k7, *k6;
};

static CondArgs cond_args(const bfs_ctx *c)
{
    CondArgs a;
    a.N = c->N; a.M = c->M; a.half = c->half; a.h = c->pc_h; a.nb = 2 * (c->N + 1) + 1;
    a.R = c->half ? 2 * c->M - 1 : c->M;
    a.ld = 2 * c->N - 2;
    a.x1 = c->x1; a.y1 = c->y1; a.dx = c->dx; a.dy = c->dy; a.F = c->pc_F; a.n_rad = c->opt.n_rad;
    a.xhi = c->x1 + (c->N - 1) * c->dx;
    a.yhi = c->y1 + (c->M - 1) * c->dy;
    a.ylo = c->half ? -a.yhi : c->y1;
    a.k5 = c->d_ktab;
    a.k7 = a.k5 + (size_t)a.R * a.ld;
    a.k6 = a.k7 + (size_t)a.R * a.ld;
    return a;
}

// phi_x can be taken first: no term that couples the F1 rows of two slices,
// a pivot n - 2 x1/dx of the first two phi_x that is no smaller than its own terms
// (it is x1/dx large on the truncated meshes of Sec. 3.1), and no growth of the
// rounding errors.  The elimination adds multiples of 2 pi dx^2/F^2 of zeta, summed over
// the slice's nodes, to blocks of the size of 2 pi, so what decides is N dx^2/F^2.
// Error of an FP64 apply against 64 bits, condensed over full blocks: 1.0 to 1.1 up to
// 60 (dx = 0.1, 0.3), 1.2 at 90 (dx = 0.3), 1.8 at 75 (dx = 3), 1.6 at 100 (dx = 0.1), 3 at
// 150 and 13 at 900 (dx = 3).  FP32: 1.2e-7 at 181 x 61 up to 150, 1.8e-7 at 300, 4.1e-7 at
// 900 (6e-8 with full blocks).
constexpr double COND_GROWTH = 75.0;
int cond_ok(const bfs_ctx *c)
{
    const double g = c->x1 / c->dx, piv = c->opt.n_rad - 2.0 * g;
    return c->opt.surface_tension == 0.0 && isfinite(piv) && fabs(piv) >= 1.0 &&
           fabs(piv) >= 0.5 * (fabs(c->opt.n_rad) + 2.0 * fabs(g)) &&
           c->N * c->dx * c->dx <= COND_GROWTH * c->F * c->F;
}

// Kernel values at row distance r dy and column offset (o - (N-2) - 1/2) dx,
// o = i - k + N - 2 for node i and half point k.
__global__ void k_cond_tables(CondArgs a, double *tab)
{
    const size_t n = (size_t)a.R * a.ld;
    for (size_t e = blockIdx.x * (size_t)blockDim.x + threadIdx.x; e < n; e += (size_t)gridDim.x * blockDim.x) {
        const int r = (int)(e / a.ld), o = (int)(e - (size_t)r * a.ld);
        const double s = (o - (a.N - 2) - 0.5) * a.dx, t = r * a.dy, p = s * s + t * t;
        const double q = rsqrt(p + 1.0);
        tab[e] = rsqrt(p);
        tab[n + e] = q;
        tab[2 * n + e] = q * q * q;
    }
}

__device__ __forceinline__ double cond_wx(const CondArgs &a, int i) { return (i == 0 || i == a.N - 1) ? 0.5 : 1.0; }
__device__ __forceinline__ double cond_wy(const CondArgs &a, int j)
{
    return a.half ? ((j == a.M - 1) ? 0.5 : 1.0) : ((j == 0 || j == a.M - 1) ? 0.5 : 1.0);
}

// sums over i of cx(i) K5 for every row distance and half point, one warp each
__global__ void k_cond_rows5(CondArgs a, double *__restrict__ out)
{
    const int w = (blockIdx.x * blockDim.x + threadIdx.x) >> 5, lane = threadIdx.x & 31;
    if (w >= a.R * (a.N - 1)) return;
    const int r = w / (a.N - 1), k = w - r * (a.N - 1);
    const double *t = a.k5 + (size_t)r * a.ld + (a.N - 2 - k);
    double v = 0.0;
    for (int i = lane; i < a.N; i += 32) v += cond_wx(a, i) * t[i];
    for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
    if (lane == 0) out[w] = v;
}

// Row sums of w K5 over all nodes and images (their closed-form integral is
// taken off by the caller's k_rowsum5_rect), from the row-distance sums
__global__ void k_cond_sum5(CondArgs a, const double *__restrict__ rows, double *__restrict__ out)
{
    const int e = blockIdx.x * blockDim.x + threadIdx.x;
    if (e >= (a.N - 1) * a.M) return;
    const int k = e % (a.N - 1), l = e / (a.N - 1);
    double v = 0.0;
    for (int j = 0; j < a.M; j++) {
        double q = rows[(size_t)abs(j - l) * (a.N - 1) + k];
        if (a.half && j >= 1) q += rows[(size_t)(j + l) * (a.N - 1) + k];
        v += cond_wy(a, j) * q;
    }
    out[e] = v * a.dx * a.dy;
}

constexpr int CF_TPB = 128;

// suf[i] = sum of x[j], j >= i, for i = 0..n (suf[n] = 0), by the whole CTA:
// each thread sums a run of entries, the runs are scanned by shuffles.
__device__ void cond_suffix(const double *x, double *suf, int n)
{
    __shared__ double tot[CF_TPB / 32];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int run = (n + CF_TPB - 1) / CF_TPB, lo = min(n, tid * run), hi = min(n, lo + run);
    double s = 0.0;
    for (int i = hi - 1; i >= lo; i--) s += x[i];
    double v = s;
    for (int o = 1; o < 32; o <<= 1) {
        const double t = __shfl_down_sync(0xffffffffu, v, o);
        if (lane + o < 32) v += t;
    }
    if (lane == 0) tot[warp] = v;
    __syncthreads();
    const double u = __shfl_down_sync(0xffffffffu, v, 1);  // this warp's later runs
    double after = lane < 31 ? u : 0.0;
    for (int w = warp + 1; w < CF_TPB / 32; w++) after += tot[w];
    for (int i = hi - 1; i >= lo; i--) {
        after += x[i];
        suf[i] = after;
    }
    if (tid == 0) suf[n] = 0.0;
    __syncthreads();
}

// Rows F2(k0) and F7(k0) of block (l, m): one CTA per (k0, d, l), threads over
// the source nodes.  tau(k) is the coefficient that zeta*(k) inherits from the
// eliminated phi_x; a column of it follows from its suffix sums and the
// trapezoid weights of zeta*.
__global__ void __launch_bounds__(CF_TPB) k_cond_form(CondArgs a, double *__restrict__ pc, const double *__restrict__ rowsum5)
{
    extern __shared__ double sh[];  // W6[N], suf[N+1], tau[N+1], ts[N+2]
    const int N = a.N, NB = N + 1, nb = a.nb, h = a.h;
    const int k0 = blockIdx.x, d = blockIdx.y, l = blockIdx.z, m = l + d - h;
    if (m < 0 || m >= a.M) return;
    double *W6 = sh, *suf = W6 + N, *tau = suf + NB, *ts = tau + NB;
    double *blk = pc + ((size_t)l * (2 * h + 1) + d) * nb * nb;
    double *r2 = blk + (size_t)(2 + k0) * nb, *r7 = blk + (size_t)(NB + 3 + k0) * nb;
    const size_t row = (size_t)abs(m - l) * a.ld + (N - 2 - k0), irow = (size_t)(m + l) * a.ld + (N - 2 - k0);
    const bool img = a.half && m >= 1, diag = l == m;
    const double TWO_PI = 6.283185307179586476925286766559;
    const double wy = a.dx * a.dy * cond_wy(a, m), cz = a.dx / (a.F * a.F);
    const double rs = diag ? 0.5 * rowsum5[l * (N - 1) + k0] : 0.0;
    for (int i = threadIdx.x; i < N; i += CF_TPB) {
        double k6 = a.k6[row + i];
        if (img) k6 += a.k6[irow + i];
        W6[i] = wy * cond_wx(a, i) * k6;
    }
    __syncthreads();
    cond_suffix(W6, suf, N);
    // tau(k), k = 1..N-1: -dx/F^2 times the sum of W6 over nodes beyond k
    for (int k = threadIdx.x; k <= N; k += CF_TPB) tau[k] = (k >= 1 && k < N) ? -cz * suf[k] : 0.0;
    __syncthreads();
    cond_suffix(tau, ts, NB);
    const double j = k0 + 1, c2 = diag ? TWO_PI * cz : 0.0;  // F2: +2 pi dx/F^2 (k < j), half of it at k = j
    auto t2 = [&](double k) { return k < j ? 1.0 : (k == j ? 0.5 : 0.0); };
    auto ts2 = [&](double p) { return p <= j ? j - p + 0.5 : 0.0; };
    for (int i = threadIdx.x; i < N; i += CF_TPB) {  // zeta_x(p), p = i + 1
        const int p = i + 1;
        double k5 = a.k5[row + i], k7 = a.k7[row + i];
        if (img) {
            k5 += a.k5[irow + i];
            k7 += a.k7[irow + i];
        }
        const double w = wy * cond_wx(a, i);
        double v5 = w * k5;
        if (i == k0 || i == k0 + 1) v5 -= rs;
        double e2, e7;
        if (p == 1) {
            e2 = 0.25 * t2(1.0) + 0.5 * ts2(2.0);
            e7 = 0.25 * tau[1] + 0.5 * ts[2];
        } else {
            const double q = p;
            e2 = ts2(q + 1.0) + (p < N ? 0.75 * t2(q) : 0.0) + 0.25 * t2(q - 1.0);
            e7 = (p < N ? ts[p + 1] : 0.0) + 0.75 * tau[p] + 0.25 * tau[p - 1];
        }
        r2[1 + i] = v5 + c2 * a.dx * e2;
        r7[1 + i] = w * k7 + a.dx * e7;
        // psi_x(p): F2 the trapezoid sum of W6, F7 its diagonal -2 pi psi*
        double v;
        if (i == 0) v = 0.5 * a.dx * suf[1];
        else if (i < N - 1) v = a.dx * (0.5 * W6[i] + suf[i + 1]);
        else v = 0.5 * a.dx * W6[N - 1];
        r2[NB + 2 + i] = v;
        double hkp = 0.0;  // weight of q_x(p) in the half-point value k0 (without dx)
        if (diag) {
            const int kk = k0 + 1;
            if (p == 1) hkp = kk == 1 ? 0.25 : 0.5;
            else hkp = p < kk ? 1.0 : (p == kk ? 0.75 : (p == kk + 1 ? 0.25 : 0.0));
        }
        r7[NB + 2 + i] = -TWO_PI * a.dx * hkp;
    }
    if (threadIdx.x == 0) {
        r2[0] = c2 * ts2(1.0);
        r7[0] = ts[1];
        r2[NB] = diag ? -TWO_PI : 0.0;
        r7[NB] = suf[0];
        r2[NB + 1] = suf[0];
        r7[NB + 1] = diag ? -TWO_PI : 0.0;
    }
}

// The five radiation rows of every diagonal block (one thread per slice)
__global__ void k_cond_form_rad(CondArgs a, double *__restrict__ pc)
{
    const int l = blockIdx.x * blockDim.x + threadIdx.x;
    if (l >= a.M) return;
    const int NB = a.N + 1, nb = a.nb;
    double *blk = pc + ((size_t)l * (2 * a.h + 1) + a.h) * nb * nb;
    const double n = a.n_rad, x1 = a.x1, g = x1 / a.dx;
    for (int f = 0; f < 2; f++) {  // F5, F6 on zeta; F8, F9 on psi
        double *ra = blk + (size_t)(f ? NB + 1 : 0) * nb + (f ? NB + 1 : 0), *rb = ra + nb;
        ra[0] = n;
        ra[1] = x1;
        rb[1] = n - g;
        rb[2] = g;
    }
    // F3: n phi(1) + x1 phi_x(1), phi_x(1) = (r4 - 2 g (r1(1) - zeta*(1)/F^2)) / (n - 2 g)
    double *r3 = blk + (size_t)NB * nb;
    const double cc = 2.0 * g * x1 / ((n - 2.0 * g) * a.F * a.F);
    r3[NB] = n;
    r3[0] = cc;
    r3[1] = 0.25 * cc * a.dx;
    r3[2] = 0.25 * cc * a.dx;
}

// ---------------------------------------------------------------------------
// Right-hand side: r (order of u) -> rc, slice by slice.  With b(k) = r1(k) and
// phi(i) = dx sum_{k<i} b(k) the part of phi already known,
//   F2(k) += 2 pi phi*(k),  F7(k) -= sum_m sum_i w K6 phi_m(i),
//   F3 -= x1 phi_x(1).
// k_cond_scan forms phi (one CTA per slice) and every row but F7, k_cond_conv the
// sums of F7.  FP64 adds are what a scan costs here (two per clock and SM), so
// each is one pass of shuffles per 256 nodes.
// ---------------------------------------------------------------------------
constexpr int CS_TPB = 256;

// Arithmetic of the F7 sums: FP64 with the FP64 sweeps; float pairs with the FP32
// ones, the high products summed two at a time into a pair (plain FP32 would
// leave the largest error of the apply here: 2.8e-7 of the solution at 181 x 61
// against 1.2e-7).
constexpr int CV_CH = 2;
__device__ __forceinline__ float2 cv_pack(double v)
{
    const float h = (float)v;
    return make_float2(h, (float)(v - (double)h));
}
struct Cv32 {
    typedef float2 K;
    typedef float2 G;
    float hi = 0.f, lo = 0.f;
    static __device__ __forceinline__ float2 pack(double v) { return cv_pack(v); }
    // the sum of two kernel values (an image's added): high parts rounded, the error kept
    static __device__ __forceinline__ float2 add(float2 a, float2 b)
    {
        const float s = __fadd_rn(a.x, b.x), bb = __fsub_rn(s, a.x);
        return make_float2(s, __fadd_rn(__fadd_rn(__fsub_rn(a.x, __fsub_rn(s, bb)), __fsub_rn(b.x, bb)), a.y + b.y));
    }
    template <int NJ>
    __device__ __forceinline__ void dot(const float2 *k, const float2 *g, int n)
    {
        float b = 0.f, c = 0.f;
#pragma unroll
        for (int j = 0; j < NJ; j++)
            if (j < n) {
                const float2 x = g[j], y = k[j];
                b = fmaf(y.x, x.x, b);
                c = fmaf(y.y, x.x, fmaf(y.x, x.y, c));
            }
        const float s = __fadd_rn(hi, b), bb = __fsub_rn(s, hi);
        lo = __fadd_rn(__fadd_rn(lo, c), __fadd_rn(__fsub_rn(hi, __fsub_rn(s, bb)), __fsub_rn(b, bb)));
        hi = s;
    }
    __device__ __forceinline__ double value() const { return (double)hi + (double)lo; }
};
struct Cv64 {
    typedef double K;
    typedef double G;
    double s = 0.0;
    static __device__ __forceinline__ double pack(double v) { return v; }
    static __device__ __forceinline__ double add(double a, double b) { return a + b; }
    template <int NJ>
    __device__ __forceinline__ void dot(const double *k, const double *g, int n)
    {
#pragma unroll
        for (int j = 0; j < NJ; j++)
            if (j < n) s = fma(k[j], g[j], s);
    }
    __device__ __forceinline__ double value() const { return s; }
};

// Inclusive prefix sum of one value per thread over the CTA, plus *carry, which
// becomes the total (every thread calls it; ends with a barrier).
__device__ __forceinline__ double cond_scan(double v, double &carry, double *tot)
{
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const double u = __shfl_up_sync(0xffffffffu, v, o);
        if (lane >= o) v += u;
    }
    if (lane == 31) tot[warp] = v;
    __syncthreads();
    double before = carry, all = carry;
#pragma unroll
    for (int w = 0; w < CS_TPB / 32; w++) {
        if (w == warp) before = all;
        all += tot[w];
    }
    carry = all;
    __syncthreads();
    return v + before;
}

template <typename CV>
__global__ void __launch_bounds__(CS_TPB) k_cond_scan(CondArgs a, const double *__restrict__ r, typename CV::G *__restrict__ g,
                                                      double *__restrict__ rc)
{
    extern __shared__ double ph[];  // phi of the slice
    __shared__ double tot[CS_TPB / 32];
    const int N = a.N, NB = N + 1, l = blockIdx.x;
    const size_t fld = (size_t)NB * a.M;
    const double *rl = r + (size_t)l * NB;
    double *out = rc + (size_t)l * a.nb;
    const double w = a.dx * a.dy * cond_wy(a, l);
    double carry = 0.0;
    for (int i0 = 0; i0 < N; i0 += CS_TPB) {
        const int i = i0 + threadIdx.x;
        const double v = cond_scan((i >= 1 && i < N) ? a.dx * rl[1 + i] : 0.0, carry, tot);
        if (i < N) {
            ph[i] = v;
            g[(size_t)l * N + i] = CV::pack(w * cond_wx(a, i) * v);
        }
    }
    __syncthreads();
    const double PI = 3.1415926535897932384626433832795;
    for (int k = threadIdx.x; k < N - 1; k += CS_TPB) out[2 + k] = rl[fld + 2 + k] + PI * (ph[k] + ph[k + 1]);
    if (threadIdx.x == 0) {
        const double gx = a.x1 / a.dx;
        out[0] = rl[0];
        out[1] = rl[1];
        out[NB] = rl[fld] - a.x1 * (rl[fld + 1] - 2.0 * gx * rl[2]) / (a.n_rad - 2.0 * gx);
        out[NB + 1] = rl[2 * fld];
        out[NB + 2] = rl[2 * fld + 1];
    }
}

// F7 of slice l: 32 half points per CTA (one a lane), the nodes of a slice dealt
// out over the warps.  The K6 rows of the band (a window of N + 31 offsets each;
// in the half domain with the images' values added) and the weighted phi of the
// band are staged in shared memory, where lanes read consecutive words.
constexpr int CC_TPB = 256;

template <typename CV>
__global__ void __launch_bounds__(CC_TPB) k_cond_conv(CondArgs a, const double *__restrict__ r,
                                                      const typename CV::K *__restrict__ k6,
                                                      const typename CV::G *__restrict__ g, double *__restrict__ rc)
{
    typedef typename CV::K T;
    typedef typename CV::G G;
    extern __shared__ double shc[];  // phi nd N, then K6 windows nd (N + 31)
    __shared__ __align__(8) char redb[CC_TPB / 32][32][8];
    auto red = reinterpret_cast<CV(*)[32]>(redb);
    const int N = a.N, NB = N + 1, h = a.h, nd = 2 * h + 1, l = blockIdx.y, k0 = blockIdx.x * 32, win = N + 31;
    G *gs = reinterpret_cast<G *>(shc);
    T *ks = reinterpret_cast<T *>(gs + (size_t)nd * N);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int q0 = max(0, h - l), q1 = min(nd, a.M - l + h);  // the band's slices m = l + q - h inside the mesh
    for (int e = threadIdx.x; e < (q1 - q0) * win; e += CC_TPB) {
        const int q = q0 + e / win, o = e % win, m = l + q - h;
        const int off = o + N - 2 - k0 - 31;  // o = i - (k - k0) + 31
        T v = T();
        if (off >= 0 && off < a.ld) {
            v = k6[(size_t)abs(q - h) * a.ld + off];
            if (a.half && m >= 1) v = CV::add(v, k6[(size_t)(m + l) * a.ld + off]);
        }
        ks[q * win + o] = v;
    }
    for (int e = threadIdx.x; e < (q1 - q0) * N; e += CC_TPB) gs[q0 * N + e] = g[(size_t)(l + q0 - h) * N + e];
    __syncthreads();
    const int per = (N + CC_TPB / 32 - 1) / (CC_TPB / 32), ia = warp * per, ib = min(N, ia + per);
    CV sum;
    for (int q = q0; q < q1; q++) {
        const T *kq = ks + q * win + 31 - lane;
        const G *gq = gs + q * N;
        int i = ia;
        for (; i + CV_CH <= ib; i += CV_CH) sum.template dot<CV_CH>(kq + i, gq + i, CV_CH);
        if (i < ib) sum.template dot<CV_CH>(kq + i, gq + i, ib - i);
    }
    red[warp][lane] = sum;
    __syncthreads();
    const int k = k0 + lane;
    if (warp == 0 && k < N - 1) {
        double s = 0.0;
#pragma unroll
        for (int w = 0; w < CC_TPB / 32; w++) s += red[w][lane].value();
        rc[(size_t)l * a.nb + NB + 3 + k] = r[2 * (size_t)NB * a.M + (size_t)l * NB + 2 + k] - s;
    }
}

// Solution: zc (slice by slice) and the F1, F4 rows of r -> z (order of u), one
// CTA per slice: zeta by the trapezoid rule, b = r1 - zeta*/F^2, and phi_x by
// its alternating recurrence, (-1)^k phi_x(k) a prefix sum.
// PAIR: zc holds float pairs (the task-table sweeps write them so, without FP64
// operations on their chain).
template <bool PAIR>
__global__ void __launch_bounds__(CS_TPB) k_cond_post(CondArgs a, const double *__restrict__ r,
                                                      const double *__restrict__ zc, double *__restrict__ z)
{
    __shared__ double tot[CS_TPB / 32];
    const int N = a.N, NB = N + 1, l = blockIdx.x;
    const size_t fld = (size_t)NB * a.M;
    const double *rl = r + (size_t)l * NB;
    auto s = [&](int i) -> double {
        if constexpr (PAIR) {
            const float2 v = reinterpret_cast<const float2 *>(zc)[(size_t)l * a.nb + i];
            return (double)v.x + (double)v.y;
        } else {
            return zc[(size_t)l * a.nb + i];
        }
    };
    double *zl = z + (size_t)l * NB;
    for (int i = threadIdx.x; i < NB; i += CS_TPB) zl[2 * fld + i] = s(NB + 1 + i);
    const double iF2 = 1.0 / (a.F * a.F), gx = a.x1 / a.dx;
    const double zs1 = s(0) + 0.25 * a.dx * (s(1) + s(2));
    const double px1 = (rl[fld + 1] - 2.0 * gx * (rl[2] - zs1 * iF2)) / (a.n_rad - 2.0 * gx);
    if (threadIdx.x == 0) {
        zl[0] = s(0);
        zl[1] = s(1);
        zl[fld] = s(NB);
        zl[fld + 1] = px1;
    }
    double zn = s(0), alt = -px1;  // zeta at the last node done; (-1)^k phi_x(k) there
    for (int i0 = 1; i0 < N; i0 += CS_TPB) {  // node k + 1 from node k, k = i0 + thread
        const int k = i0 + threadIdx.x;
        const bool in = k < N;
        const double db = in ? s(k + 1) : 0.0, inc = in ? 0.5 * a.dx * (s(k) + db) : 0.0;
        const double znext = cond_scan(inc, zn, tot);  // zeta(k+1)
        const double b = in ? rl[1 + k] - (znext - 0.5 * inc) * iF2 : 0.0;
        // (-1)^(k+1) phi_x(k+1) = (-1)^k phi_x(k) - 2 (-1)^k b(k)
        const double y = cond_scan((k & 1) ? 2.0 * b : -2.0 * b, alt, tot);
        if (in) {
            zl[1 + k] = db;
            zl[fld + 1 + k] = (k & 1) ? y : -y;
        }
    }
}

__global__ void k_cond_cast(const double *__restrict__ x, float2 *__restrict__ y, size_t n)
{
    for (size_t e = blockIdx.x * (size_t)blockDim.x + threadIdx.x; e < n; e += (size_t)gridDim.x * blockDim.x)
        y[e] = cv_pack(x[e]);
}

// Tables and the row sums of w K5 into d_rowsum5 (before its closed-form part); for
// condensed blocks also K6 in float pairs and the vectors of the reduced system.
int cond_tables(bfs_ctx *c, cudaStream_t s)
{
    const int R = c->half ? 2 * c->M - 1 : c->M, ld = 2 * c->N - 2;
    const size_t n = (size_t)R * ld, nv = (size_t)c->M * c->nb, nr = (size_t)R * (c->N - 1);
    BFS_ALLOC_TRY(c, cudaMalloc(&c->d_ktab, sizeof(double) * ((c->pc_cond ? 4 : 3) * n + nr)));
    const CondArgs a = cond_args(c);
    double *rows = c->d_ktab + 3 * n;
    k_cond_tables<<<512, 256, 0, s>>>(a, c->d_ktab);
    if (c->pc_cond) {
        BFS_ALLOC_TRY(c, cudaMalloc(&c->d_rc, sizeof(double) * (2 * nv + (size_t)c->NM)));  // then phi of k_cond_scan
        c->d_zc = c->d_rc + nv;
        k_cond_cast<<<512, 256, 0, s>>>(a.k6, reinterpret_cast<float2 *>(rows + nr), n);
        c->launches++;
    }
    k_cond_rows5<<<(R * (c->N - 1) + 7) / 8, 256, 0, s>>>(a, rows);
    k_cond_sum5<<<(c->Nt + 63) / 64, 64, 0, s>>>(a, rows, c->d_rowsum5);
    c->launches += 3;
    BFS_CUDA_TRY(c, cudaGetLastError());
    return BFS_OK;
}

// Shared memory of the kernels that stage rows of nodes: the limit of cond_fits,
// asked for whatever a launch needs (without it their static arrays count towards
// 48 KB too) and the same for every context.
constexpr size_t COND_SMEM = 200 * 1024;

int cond_form(bfs_ctx *c, cudaStream_t s)
{
    const CondArgs a = cond_args(c);
    for (const void *k : {(const void *)k_cond_form, (const void *)k_cond_scan<Cv32>, (const void *)k_cond_scan<Cv64>,
                          (const void *)k_cond_conv<Cv32>, (const void *)k_cond_conv<Cv64>})
        BFS_CUDA_TRY(c, cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)COND_SMEM));
    const size_t sm = sizeof(double) * (4 * (size_t)c->N + 8);
    k_cond_form<<<dim3(c->N - 1, 2 * c->pc_h + 1, c->M), CF_TPB, sm, s>>>(a, c->d_pc, c->d_rowsum5);
    k_cond_form_rad<<<(c->M + 31) / 32, 32, 0, s>>>(a, c->d_pc);
    c->launches += 2;
    BFS_CUDA_TRY(c, cudaGetLastError());
    return BFS_OK;
}

static size_t conv_smem(const bfs_ctx *c, int h, size_t item) { return item * (size_t)(2 * h + 1) * (2 * c->N + 31); }

static size_t conv_smem(const bfs_ctx *c, int h, size_t k, size_t g) { return (size_t)(2 * h + 1) * (g * c->N + k * (c->N + 31)); }

// Where condensing pays.  The reduction and the recovery cost about 25 us an
// apply, which small slices do not win back (FP32 sweeps, whole apply, condensed
// against full blocks: 57 / 35 us at 61 x 21, 86 / 72 at 121 x 41, 112 / 108 at
// 151 x 51, 132 / 137 at 181 x 61, 225 / 994 at 241 x 81; FP64: 183 / 165 at
// 61 x 21, 386 / 398 at 121 x 41, 731 / 966 at 181 x 61; the factorisation takes
// half the time from about 140 columns up).  With the FP32 sweeps at most 256
// columns: condensing lets the FP32 rounding of the factors grow with the
// columns (error of an apply relative to the solution, condensed against full
// blocks: 1.2e-7 / 1.3e-7 at 181, 1.4e-7 / 1.4e-7 at 241, 2.9e-7 / 1.3e-7 at 361).
int cond_fits(const bfs_ctx *c, int h)
{
    if (c->opt.precond_precision == BFS_FP32C ? (c->N < 140 || c->N > 256) : c->N < 100) return 0;
    return conv_smem(c, h, 8, 8) <= COND_SMEM && sizeof(double) * (4 * (size_t)c->N + 8) <= COND_SMEM;
}

template <typename CV>
static int cond_pre_t(bfs_ctx *c, const double *r, const typename CV::K *k6, cudaStream_t s)
{
    const CondArgs a = cond_args(c);
    typename CV::G *g = reinterpret_cast<typename CV::G *>(c->d_zc + (size_t)c->M * c->nb);
    const size_t sm = conv_smem(c, c->pc_h, sizeof(typename CV::K), sizeof(typename CV::G));
    const size_t ss = sizeof(double) * (size_t)c->N;
    k_cond_scan<CV><<<c->M, CS_TPB, ss, s>>>(a, r, g, c->d_rc);
    k_cond_conv<CV><<<dim3((c->N + 30) / 32, c->M), CC_TPB, sm, s>>>(a, r, k6, g, c->d_rc);
    c->launches += 2;
    BFS_CUDA_TRY(c, cudaGetLastError());
    return BFS_OK;
}

int cond_pre(bfs_ctx *c, const double *r, cudaStream_t s)
{
    const CondArgs a = cond_args(c);
    if (c->d_pc32)
        return cond_pre_t<Cv32>(c, r, reinterpret_cast<const float2 *>(a.k6 + (size_t)a.R * a.ld + (size_t)a.R * (c->N - 1)), s);
    return cond_pre_t<Cv64>(c, r, a.k6, s);
}

int cond_post(bfs_ctx *c, const double *r, double *z, bool pairs, cudaStream_t s)
{
    if (pairs) k_cond_post<true><<<c->M, CS_TPB, 0, s>>>(cond_args(c), r, c->d_zc, z);
    else k_cond_post<false><<<c->M, CS_TPB, 0, s>>>(cond_args(c), r, c->d_zc, z);
    c->launches++;
    BFS_CUDA_TRY(c, cudaGetLastError());
    return BFS_OK;
}

}  // namespace bfs

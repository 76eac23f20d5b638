// Learned initial guess (C ABI in include/bfs_cno.h): a small convolutional
// neural operator on the nodal grid (an addition: the paper starts Newton from
// a flat surface or from a nearby solution).  It maps the bottom B = beta + 1, the Froude number
// and the node coordinates to the nodal fields zeta, phi - x and psi - x; the
// guess is accepted only through Newton to the same residual tolerance.
//
// Network: four dilated 3x3 convolutions (dilations 1, 3, 9, 27; widths
// 16 -> 32 -> 32 -> 32 -> 16, of which 4 inputs and 3 outputs are used), SiLU
// between them, zero padding.  Weights and activations are BF16, every
// contraction runs on the tensor cores through mma.sync m16n8k16 with FP32
// accumulation; master weights and the Adam moments are FP32.
//
// Layouts: activations NHWC (batch, row y, column x, channel); layer weights
// are kept in two BF16 copies, [cout][tap][cin] for the forward pass and
// [cin][tap][cout] for the backward pass on the inputs (the same convolution
// kernel run with negated tap offsets), both filled from one FP32 master
// vector holding, per layer, the weights [cout][tap][cin] then the biases.
#include <cuda_bf16.h>
#include <math.h>
#include <stdint.h>
#include <string.h>

#include <algorithm>
#include <new>
#include <string>
#include <utility>
#include <vector>

#include "bfs_cno.h"
#include "bfs_internal.cuh"

namespace {

constexpr int NL = 4;
constexpr int CIN[NL] = {16, 32, 32, 32};
constexpr int COUT[NL] = {32, 32, 32, 16};
constexpr int DIL[NL] = {1, 3, 9, 27};
constexpr int IN_REAL = 4, OUT_REAL = 3;

int n_weights(int l) { return COUT[l] * 9 * CIN[l]; }

int n_params()
{
    int s = 0;
    for (int l = 0; l < NL; l++) s += n_weights(l) + COUT[l];
    return s;
}

__device__ __forceinline__ void mma16816(float c[4], const uint32_t a[4], const uint32_t b[2])
{
    asm volatile(
        "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, "
        "{%8,%9}, {%0,%1,%2,%3};\n"
        : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
        : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b[0]), "r"(b[1]));
}

__device__ __forceinline__ float sigm(float z) { return 1.f / (1.f + __expf(-z)); }

template <bool TRANS>
__device__ __forceinline__ void ldm4(uint32_t r[4], uint32_t addr)
{
    if (TRANS)
        asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0,%1,%2,%3}, [%4];"
                     : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(addr));
    else
        asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0,%1,%2,%3}, [%4];"
                     : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(addr));
}

__device__ __forceinline__ void cp16(uint32_t dst, const void *src, bool ok)
{
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(src), "r"(ok ? 16 : 0));
}

__device__ __forceinline__ void cp_join()
{
    asm volatile("cp.async.commit_group;");
    asm volatile("cp.async.wait_group 0;");
    __syncthreads();
}

// Work items of both kernels: XS pixels of one image row.  An item's three input
// rows (the taps' y offsets) with dil columns to either side lie in shared memory as
// [row][column] records of C channels, zero outside the grid, so that a tap is an
// offset of the record index.  The 16-byte units of record R are permuted by R such
// that eight consecutive records of an ldmatrix touch all banks.
constexpr int XS = 96;

template <int C>
__device__ __forceinline__ uint32_t rec(int R, int unit)
{
    return R * (2 * C) + ((C == 32 ? unit ^ (R >> 1 & 3) : unit ^ (R >> 2 & 1)) << 4);
}

template <int C>
__device__ __forceinline__ void stage_rows(uint32_t sm, const __nv_bfloat16 *in, int row, int y, int x0, int H, int W,
                                           int dil)
{
    constexpr int U = C / 8;
    const int wd = XS + 2 * dil;
    for (int e = threadIdx.x; e < 3 * wd * U; e += blockDim.x) {
        const int u = e % U, R = e / U, tr = R / wd, x = x0 - dil + R - tr * wd, dy = (tr - 1) * dil;
        const bool ok = y + dy >= 0 && y + dy < H && x >= 0 && x < W;
        cp16(sm + rec<C>(R, u), ok ? in + ((size_t)(row + dy) * W + x) * C + u * 8 : in, ok);
    }
}

// Implicit-GEMM dilated 3x3 convolution.  v[p][n] = sum over taps t and
// input channels c of in[p + sgn * off(t) * dil][c] * w[n][t][c] (+ bias[n]),
// zero outside the grid.  in: BF16 NHWC with C channels (C in {16, 32});
// w: BF16 [N][9][C].  What becomes of v:
//   OUT_Z     z = v (FP32 [P][N])
//   OUT_SILU  z = v and a = silu(v) (BF16)
//   OUT_GRAD  a = v silu'(z) (BF16), z read
// One warp per 16 pixels, N / 8 MMA column tiles per warp; weights and input rows are
// staged once per CTA and item.  Bound by the latency of an item's loads; 16 images of
// 181 x 61, 32 -> 32 channels: 27 us with SiLU and 34 with its derivative (90 with
// fragments loaded channel by channel from global memory, 15 more for either).  96
// pixels fill the warps of a 181-pixel row to 94 %.
enum ConvOut { OUT_Z, OUT_SILU, OUT_GRAD };

template <int C, int N, int OUT>
__global__ void __launch_bounds__(XS * 2)
k_conv(const __nv_bfloat16 *__restrict__ in, const __nv_bfloat16 *__restrict__ w, const float *__restrict__ bias,
       float *__restrict__ z, __nv_bfloat16 *__restrict__ a_out, int Bt, int H, int W, int dil, int sgn)
{
    extern __shared__ __align__(128) unsigned char smem[];
    constexpr int WS = (9 * C + 8) * 2;  // weight row, padded against bank conflicts
    const uint32_t sw = (uint32_t)__cvta_generic_to_shared(smem), si = sw + N * WS;
    const int lane = threadIdx.x & 31, m0 = threadIdx.x / 32 * 16;
    const int r = lane >> 2, cq = (lane & 3) * 2;
    const int nseg = (W + XS - 1) / XS, items = Bt * H * nseg, wd = XS + 2 * dil;
    for (int e = threadIdx.x; e < N * 9 * C / 8; e += blockDim.x)
        cp16(sw + e / (9 * C / 8) * WS + e % (9 * C / 8) * 16, w + (size_t)e * 8, true);
    const uint32_t wrow = sw + (lane / 16 * 8 + lane % 8) * WS + lane / 8 % 2 * 16;
    for (int it = blockIdx.x; it < items; it += gridDim.x) {
        const int row = it / nseg, x0 = (it - row * nseg) * XS, y = row % H;
        stage_rows<C>(si, in, row, y, x0, H, W, dil);
        cp_join();
        if (x0 + m0 < W) {
            float acc[N / 8][4];
#pragma unroll
            for (int nt = 0; nt < N / 8; nt++)
#pragma unroll
                for (int e = 0; e < 4; e++) acc[nt][e] = 0.f;
#pragma unroll
            for (int t = 0; t < 9; t++) {
                const int R = (1 + sgn * (t / 3 - 1)) * wd + dil * (1 + sgn * (t % 3 - 1)) + m0 + lane % 16;
#pragma unroll
                for (int c0 = 0; c0 < C; c0 += 16) {
                    uint32_t a[4];
                    ldm4<false>(a, si + rec<C>(R, c0 / 8 + lane / 16));
#pragma unroll
                    for (int np = 0; np < N / 16; np++) {
                        uint32_t b[4];
                        ldm4<false>(b, wrow + np * 16 * WS + (t * C + c0) * 2);
                        mma16816(acc[2 * np], a, b);
                        mma16816(acc[2 * np + 1], a, b + 2);
                    }
                }
            }
#pragma unroll
            for (int nt = 0; nt < N / 8; nt++) {
                const int n0 = nt * 8 + cq;
                const float b0 = bias ? bias[n0] : 0.f, b1 = bias ? bias[n0 + 1] : 0.f;
#pragma unroll
                for (int h = 0; h < 2; h++) {
                    const int x = x0 + m0 + r + 8 * h;
                    if (x >= W) continue;
                    const size_t o = ((size_t)row * W + x) * N + n0;
                    float2 v = make_float2(acc[nt][2 * h] + b0, acc[nt][2 * h + 1] + b1);
                    if (OUT != OUT_GRAD) *reinterpret_cast<float2 *>(z + o) = v;
                    if (OUT == OUT_SILU) v = make_float2(v.x * sigm(v.x), v.y * sigm(v.y));
                    if (OUT == OUT_GRAD) {
                        const float2 q = *reinterpret_cast<const float2 *>(z + o);
                        const float s0 = sigm(q.x), s1 = sigm(q.y);
                        v = make_float2(v.x * s0 * (1.f + q.x * (1.f - s0)), v.y * s1 * (1.f + q.y * (1.f - s1)));
                    }
                    if (OUT != OUT_Z)
                        *reinterpret_cast<__nv_bfloat162 *>(a_out + o) =
                            __halves2bfloat162(__float2bfloat16(v.x), __float2bfloat16(v.y));
                }
            }
        }
        __syncthreads();
    }
}

// Weight and bias gradients: dw[n][t][c] += sum over pixels p of in[p + off(t) dil][c]
// * g[p][n], db[n] += sum of g[p][n].  One warp per tap, C rows (c) by N columns, the
// pixels as the contraction: both operands lie pixel by pixel in shared memory and are
// transposed by ldmatrix.  A CTA goes over its items and adds to dw once, by FP32
// atomics; the centre tap's warp adds g up against a row of ones.  Same layer: 33 us
// (170 with 2-byte loads from global memory and a pass of its own for db, 22).
template <int C, int N>
__global__ void __launch_bounds__(288)
k_conv_wgrad(const __nv_bfloat16 *__restrict__ in, const __nv_bfloat16 *__restrict__ g, float *__restrict__ dw,
             float *__restrict__ db, int Bt, int H, int W, int dil)
{
    extern __shared__ __align__(128) unsigned char smem[];
    const uint32_t sg = (uint32_t)__cvta_generic_to_shared(smem), si = sg + XS * N * 2;
    const int lane = threadIdx.x & 31, t = threadIdx.x / 32;
    const int r = lane >> 2, cq = (lane & 3) * 2;
    const int nseg = (W + XS - 1) / XS, items = Bt * H * nseg, wd = XS + 2 * dil;
    const int R0 = t / 3 * wd + t % 3 * dil;
    const uint32_t ones[4] = {0x3f803f80u, 0x3f803f80u, 0x3f803f80u, 0x3f803f80u};
    float acc[C / 16][N / 8][4], ab[N / 8][4];
#pragma unroll
    for (int nt = 0; nt < N / 8; nt++)
#pragma unroll
        for (int e = 0; e < 4; e++) {
            ab[nt][e] = 0.f;
#pragma unroll
            for (int mt = 0; mt < C / 16; mt++) acc[mt][nt][e] = 0.f;
        }
    for (int it = blockIdx.x; it < items; it += gridDim.x) {
        const int row = it / nseg, x0 = (it - row * nseg) * XS, y = row % H;
        stage_rows<C>(si, in, row, y, x0, H, W, dil);
        for (int e = threadIdx.x; e < XS * N / 8; e += blockDim.x) {
            const int u = e % (N / 8), x = e / (N / 8);
            const bool ok = x0 + x < W;
            cp16(sg + rec<N>(x, u), ok ? g + ((size_t)row * W + x0 + x) * N + u * 8 : g, ok);
        }
        cp_join();
#pragma unroll 2
        for (int k = 0; k < XS; k += 16) {
            uint32_t a[C / 16][4];
#pragma unroll
            for (int mt = 0; mt < C / 16; mt++)
                ldm4<true>(a[mt], si + rec<C>(R0 + k + lane / 16 * 8 + lane % 8, mt * 2 + lane / 8 % 2));
#pragma unroll
            for (int np = 0; np < N / 16; np++) {
                uint32_t b[4];
                ldm4<true>(b, sg + rec<N>(k + lane % 16, np * 2 + lane / 16));
#pragma unroll
                for (int mt = 0; mt < C / 16; mt++) {
                    mma16816(acc[mt][2 * np], a[mt], b);
                    mma16816(acc[mt][2 * np + 1], a[mt], b + 2);
                }
                if (t == 4) {
                    mma16816(ab[2 * np], ones, b);
                    mma16816(ab[2 * np + 1], ones, b + 2);
                }
            }
        }
        __syncthreads();
    }
#pragma unroll
    for (int nt = 0; nt < N / 8; nt++) {
        const int n0 = nt * 8 + cq;
#pragma unroll
        for (int mt = 0; mt < C / 16; mt++)
#pragma unroll
            for (int h = 0; h < 2; h++) {
                float *d = dw + ((size_t)n0 * 9 + t) * C + mt * 16 + r + 8 * h;
                atomicAdd(d, acc[mt][nt][2 * h]);
                atomicAdd(d + 9 * C, acc[mt][nt][2 * h + 1]);
            }
        if (t == 4 && r == 0) {
            atomicAdd(db + n0, ab[nt][0]);
            atomicAdd(db + n0 + 1, ab[nt][1]);
        }
    }
}

// input features (FP32, 4 channels) -> BF16, padded to 16 channels
__global__ void k_in_bf16(const float *__restrict__ x, __nv_bfloat16 *__restrict__ o, int P)
{
    int e = blockIdx.x * blockDim.x + threadIdx.x;
    if (e >= P * 16) return;
    int p = e >> 4, c = e & 15;
    o[e] = __float2bfloat16(c < IN_REAL ? x[(size_t)p * IN_REAL + c] : 0.f);
}

// output (FP32, 16 channels, 3 used) vs target (3 channels): loss partials and
// the BF16 gradient 2 (y - t) / count
__global__ void k_mse(const float *__restrict__ y, const float *__restrict__ t, __nv_bfloat16 *__restrict__ gy,
                      float *__restrict__ loss, int P)
{
    __shared__ float sh[256];
    int e = blockIdx.x * blockDim.x + threadIdx.x;
    float l = 0.f;
    if (e < P * 16) {
        int p = e >> 4, c = e & 15;
        float g = 0.f;
        if (c < OUT_REAL) {
            float d = y[e] - t[(size_t)p * OUT_REAL + c];
            l = d * d;
            g = 2.f * d / (float)(P * OUT_REAL);
        }
        gy[e] = __float2bfloat16(g);
    }
    sh[threadIdx.x] = l;
    __syncthreads();
    for (int o = blockDim.x / 2; o > 0; o >>= 1) {
        if (threadIdx.x < o) sh[threadIdx.x] += sh[threadIdx.x + o];
        __syncthreads();
    }
    if (threadIdx.x == 0) atomicAdd(loss, sh[0] / (float)(P * OUT_REAL));
}

// master FP32 parameters -> the BF16 forward and backward weight copies
__global__ void k_cast_weights(const float *__restrict__ wm, __nv_bfloat16 *__restrict__ wf,
                               __nv_bfloat16 *__restrict__ wb, int Cin, int Cout)
{
    int e = blockIdx.x * blockDim.x + threadIdx.x;
    if (e >= Cout * 9 * Cin) return;
    int n = e / (9 * Cin), rem = e % (9 * Cin), t = rem / Cin, c = rem % Cin;
    __nv_bfloat16 v = __float2bfloat16(wm[e]);
    wf[e] = v;
    // backward on the inputs: [c][t][n], used with negated tap offsets
    wb[((size_t)c * 9 + t) * Cout + n] = v;
}

__global__ void k_adam(float *__restrict__ p, const float *__restrict__ g, float *__restrict__ m,
                       float *__restrict__ v, int n, float lr, float b1, float b2, float eps, float c1,
                       float c2)
{
    int e = blockIdx.x * blockDim.x + threadIdx.x;
    if (e >= n) return;
    float gi = g[e];
    float mi = b1 * m[e] + (1.f - b1) * gi;
    float vi = b2 * v[e] + (1.f - b2) * gi * gi;
    m[e] = mi;
    v[e] = vi;
    p[e] -= lr * (mi / c1) / (sqrtf(vi / c2) + eps);
}

// nodal predictions (zeta, phi - x, psi - x; one image) -> unknown vector u:
// q(x1) from the first node, q_x by centred differences (one-sided at the ends)
// plus 1 for phi and psi.
__global__ void k_fields_to_u(const float *__restrict__ y, const float *__restrict__ scale,
                              double *__restrict__ u, int N, int M, double dx, double x1)
{
    int e = blockIdx.x * blockDim.x + threadIdx.x;
    const int NB = N + 1;
    if (e >= 3 * NB * M) return;
    int f = e / (NB * M), rem = e % (NB * M), j = rem / NB, pidx = rem % NB;
    auto val = [&](int i) -> double { return (double)y[((size_t)j * N + i) * 16 + f] * scale[f]; };
    double out;
    if (pidx == 0) {
        out = val(0) + (f > 0 ? x1 : 0.0);
    } else {
        int i = pidx - 1;
        double d;
        if (i == 0) d = (-3.0 * val(0) + 4.0 * val(1) - val(2)) / (2.0 * dx);
        else if (i == N - 1) d = (3.0 * val(N - 1) - 4.0 * val(N - 2) + val(N - 3)) / (2.0 * dx);
        else d = (val(i + 1) - val(i - 1)) / (2.0 * dx);
        out = d + (f > 0 ? 1.0 : 0.0);
    }
    u[e] = out;
}

}  // namespace

struct bfs_cno {
    int H, W, Bmax, np;
    float *p, *g, *m, *v;   // FP32 parameters, gradient, Adam moments
    __nv_bfloat16 *wf[NL], *wb[NL];
    float *bias[NL], *dbias[NL], *dw[NL];
    __nv_bfloat16 *act[NL + 1];  // BF16 inputs of each layer (act[0] = features)
    float *z[NL];                // FP32 pre-activations
    __nv_bfloat16 *gz, *gz2;     // BF16 gradients w.r.t. pre-activations, by turns
    float *loss;
    float *scale;                // output scales (3)
    float *xin;                  // features of one image copied from the host (bfs_cno_solve_host)
    int step;
    std::string err;
};

namespace {
thread_local std::string g_cno_err;

int sms()
{
    int dev = 0;
    cudaGetDevice(&dev);
    return bfs::num_sms(dev);
}

constexpr size_t rows_smem(int C, int dil) { return (size_t)3 * (XS + 2 * dil) * C * 2; }
constexpr size_t conv_smem(int C, int N, int dil) { return (size_t)N * (9 * C + 8) * 2 + rows_smem(C, dil); }
constexpr size_t wgrad_smem(int C, int N, int dil) { return (size_t)XS * N * 2 + rows_smem(C, dil); }

// Both kernels of every layer, each way, stay within the 48 KB of shared memory that a launch
// may ask for without more (the largest is the convolution of 32 -> 32 channels at
// dilation 9, 40.8 KB).
constexpr size_t largest_smem()
{
    size_t m = 0;
    for (int l = 0; l < NL; l++)
        for (size_t b : {conv_smem(CIN[l], COUT[l], DIL[l]), conv_smem(COUT[l], CIN[l], DIL[l]),
                         wgrad_smem(CIN[l], COUT[l], DIL[l])})
            m = b > m ? b : m;
    return m;
}
static_assert(largest_smem() <= 48 * 1024, "shared memory of the convolutions");

template <int C, int N, int OUT>
void conv(const __nv_bfloat16 *in, const __nv_bfloat16 *w, const float *b, float *z, __nv_bfloat16 *a, int Bt, int H,
          int W, int dil, int sgn, cudaStream_t s)
{
    const int items = Bt * H * ((W + XS - 1) / XS);
    k_conv<C, N, OUT><<<std::min(items, 4 * sms()), 2 * XS, conv_smem(C, N, dil), s>>>(
        in, w, b, z, a, Bt, H, W, dil, sgn);
}

template <int OUT>
void conv_any(int C, int N, const __nv_bfloat16 *in, const __nv_bfloat16 *w, const float *b, float *z,
              __nv_bfloat16 *a, int Bt, int H, int W, int dil, int sgn, cudaStream_t s)
{
    if (C == 16 && N == 32) conv<16, 32, OUT>(in, w, b, z, a, Bt, H, W, dil, sgn, s);
    else if (C == 32 && N == 32) conv<32, 32, OUT>(in, w, b, z, a, Bt, H, W, dil, sgn, s);
    else if (C == 32 && N == 16) conv<32, 16, OUT>(in, w, b, z, a, Bt, H, W, dil, sgn, s);
}

template <int C, int N>
void wgrad(const __nv_bfloat16 *in, const __nv_bfloat16 *g, float *dw, float *db, int Bt, int H, int W, int dil,
           cudaStream_t s)
{
    const int items = Bt * H * ((W + XS - 1) / XS);
    k_conv_wgrad<C, N><<<std::min(items, 3 * sms()), 288, wgrad_smem(C, N, dil), s>>>(in, g, dw, db, Bt, H, W, dil);
}

void wgrad_any(int C, int N, const __nv_bfloat16 *in, const __nv_bfloat16 *g, float *dw, float *db, int Bt, int H,
               int W, int dil, cudaStream_t s)
{
    if (C == 16 && N == 32) wgrad<16, 32>(in, g, dw, db, Bt, H, W, dil, s);
    else if (C == 32 && N == 32) wgrad<32, 32>(in, g, dw, db, Bt, H, W, dil, s);
    else if (C == 32 && N == 16) wgrad<32, 16>(in, g, dw, db, Bt, H, W, dil, s);
}

int ferr(bfs_cno *n, int code, const std::string &m)
{
    if (n) n->err = m;
    else g_cno_err = m;
    return code;
}

int forward(bfs_cno *n, const float *x, int Bt, cudaStream_t s)
{
    const int P = Bt * n->H * n->W;
    k_in_bf16<<<(P * 16 + 255) / 256, 256, 0, s>>>(x, n->act[0], P);
    for (int l = 0; l < NL; l++) {
        if (l < NL - 1)
            conv_any<OUT_SILU>(CIN[l], COUT[l], n->act[l], n->wf[l], n->bias[l], n->z[l], n->act[l + 1], Bt, n->H,
                               n->W, DIL[l], 1, s);
        else
            conv_any<OUT_Z>(CIN[l], COUT[l], n->act[l], n->wf[l], n->bias[l], n->z[l], nullptr, Bt, n->H, n->W,
                            DIL[l], 1, s);
    }
    return cudaGetLastError() == cudaSuccess ? BFS_OK : ferr(n, BFS_ECUDA, "forward launch failed");
}

// gradient of the mean squared error w.r.t. all parameters into n->g; loss into n->loss
int backward(bfs_cno *n, const float *target, int Bt, cudaStream_t s)
{
    const int P = Bt * n->H * n->W;
    cudaMemsetAsync(n->g, 0, sizeof(float) * n->np, s);
    cudaMemsetAsync(n->loss, 0, sizeof(float), s);
    k_mse<<<(P * 16 + 255) / 256, 256, 0, s>>>(n->z[NL - 1], target, n->gz, n->loss, P);
    __nv_bfloat16 *g = n->gz, *gp = n->gz2;
    for (int l = NL - 1; l >= 0; l--) {
        // g holds dL/dz_l (BF16, COUT[l] channels)
        wgrad_any(CIN[l], COUT[l], n->act[l], g, n->dw[l], n->dbias[l], Bt, n->H, n->W, DIL[l], s);
        if (l == 0) break;
        conv_any<OUT_GRAD>(COUT[l], CIN[l], g, n->wb[l], nullptr, n->z[l - 1], gp, Bt, n->H, n->W, DIL[l], -1, s);
        std::swap(g, gp);
    }
    return cudaGetLastError() == cudaSuccess ? BFS_OK : ferr(n, BFS_ECUDA, "backward launch failed");
}

void cast_all(bfs_cno *n, cudaStream_t s)
{
    size_t off = 0;
    for (int l = 0; l < NL; l++) {
        k_cast_weights<<<(n_weights(l) + 255) / 256, 256, 0, s>>>(n->p + off, n->wf[l], n->wb[l], CIN[l], COUT[l]);
        off += n_weights(l) + COUT[l];
    }
}
}  // namespace

extern "C" {

const char *bfs_cno_last_error(const bfs_cno *n) { return n ? n->err.c_str() : g_cno_err.c_str(); }

int bfs_cno_num_params(void) { return n_params(); }

void bfs_cno_destroy(bfs_cno *n)
{
    if (!n) return;
    cudaFree(n->p);
    for (int l = 0; l < NL; l++) {
        cudaFree(n->wf[l]);
        cudaFree(n->wb[l]);
        cudaFree(n->z[l]);
        cudaFree(n->act[l]);
    }
    cudaFree(n->gz2);
    cudaFree(n->gz);  // loss and scale live inside the parameter allocation
    cudaFree(n->xin);
    delete n;
}

int bfs_cno_create(int H, int W, int Bmax, bfs_cno **out)
{
    if (!out) return ferr(nullptr, BFS_EINVAL, "out is NULL");
    *out = nullptr;
    if (H < 3 || W < 3 || Bmax < 1) return ferr(nullptr, BFS_EINVAL, "bad grid or batch size");
    bfs_cno *n = new (std::nothrow) bfs_cno();
    if (!n) return ferr(nullptr, BFS_ENOMEM, "host allocation failed");
    n->H = H; n->W = W; n->Bmax = Bmax; n->np = n_params();
    const size_t P = (size_t)Bmax * H * W;
    bool ok = cudaMalloc(&n->p, sizeof(float) * (4 * (size_t)n->np + 4)) == cudaSuccess;
    if (ok) {
        n->g = n->p + n->np; n->m = n->g + n->np; n->v = n->m + n->np;
        n->loss = n->v + n->np; n->scale = n->loss + 1;
        size_t off = 0;
        for (int l = 0; l < NL; l++) {
            n->dw[l] = n->g + off;
            n->bias[l] = n->p + off + n_weights(l);
            n->dbias[l] = n->g + off + n_weights(l);
            off += n_weights(l) + COUT[l];
            ok = ok && cudaMalloc(&n->wf[l], sizeof(__nv_bfloat16) * n_weights(l)) == cudaSuccess;
            ok = ok && cudaMalloc(&n->wb[l], sizeof(__nv_bfloat16) * n_weights(l)) == cudaSuccess;
            ok = ok && cudaMalloc(&n->z[l], sizeof(float) * P * COUT[l]) == cudaSuccess;
            ok = ok && cudaMalloc(&n->act[l], sizeof(__nv_bfloat16) * P * CIN[l]) == cudaSuccess;
        }
        ok = ok && cudaMalloc(&n->gz2, sizeof(__nv_bfloat16) * P * 32) == cudaSuccess;
        ok = ok && cudaMalloc(&n->xin, sizeof(float) * (size_t)H * W * 4) == cudaSuccess;
        ok = ok && cudaMalloc(&n->gz, sizeof(__nv_bfloat16) * P * 32) == cudaSuccess;
    }
    if (!ok || cudaMemset(n->p, 0, sizeof(float) * (4 * (size_t)n->np + 4)) != cudaSuccess) {
        bfs_cno_destroy(n);
        cudaGetLastError();
        return ferr(nullptr, BFS_ENOMEM, "device allocation failed");
    }
    *out = n;
    return BFS_OK;
}

// params: host FP32 vector of bfs_cno_num_params(); out_scale: 3 output scales
int bfs_cno_set_params(bfs_cno *n, const float *params, const float *out_scale)
{
    if (!n || !params) return BFS_EINVAL;
    if (cudaMemcpy(n->p, params, sizeof(float) * n->np, cudaMemcpyHostToDevice) != cudaSuccess)
        return ferr(n, BFS_ECUDA, "parameter upload failed");
    float sc[3] = {1.f, 1.f, 1.f};
    if (out_scale) memcpy(sc, out_scale, sizeof(sc));
    if (cudaMemcpy(n->scale, sc, sizeof(sc), cudaMemcpyHostToDevice) != cudaSuccess)
        return ferr(n, BFS_ECUDA, "scale upload failed");
    cudaMemset(n->m, 0, sizeof(float) * 2 * n->np);
    n->step = 0;
    cast_all(n, 0);
    return cudaDeviceSynchronize() == cudaSuccess ? BFS_OK : ferr(n, BFS_ECUDA, "cast failed");
}

int bfs_cno_get_params(bfs_cno *n, float *params)
{
    if (!n || !params) return BFS_EINVAL;
    return cudaMemcpy(params, n->p, sizeof(float) * n->np, cudaMemcpyDeviceToHost) == cudaSuccess
               ? BFS_OK : ferr(n, BFS_ECUDA, "parameter download failed");
}

// x: device FP32 [Bt][H][W][4]; y: device FP32 [Bt][H][W][16] (channels 0..2 used)
int bfs_cno_forward(bfs_cno *n, const float *x, int Bt, float *y, void *stream)
{
    if (!n || !x || !y || Bt < 1 || Bt > n->Bmax) return ferr(n, BFS_EINVAL, "bad arguments");
    cudaStream_t s = (cudaStream_t)stream;
    int rc = forward(n, x, Bt, s);
    if (rc) return rc;
    const size_t bytes = sizeof(float) * (size_t)Bt * n->H * n->W * 16;
    return cudaMemcpyAsync(y, n->z[NL - 1], bytes, cudaMemcpyDeviceToDevice, s) == cudaSuccess
               ? BFS_OK : ferr(n, BFS_ECUDA, "output copy failed");
}

// gradient of the mean squared error (target: device FP32 [Bt][H][W][3]) into
// grad_host (bfs_cno_num_params floats); *loss_host receives the loss.  Synchronous.
int bfs_cno_gradient(bfs_cno *n, const float *x, const float *target, int Bt, float *grad_host,
                     float *loss_host, void *stream)
{
    if (!n || !x || !target || Bt < 1 || Bt > n->Bmax) return ferr(n, BFS_EINVAL, "bad arguments");
    cudaStream_t s = (cudaStream_t)stream;
    int rc = forward(n, x, Bt, s);
    if (!rc) rc = backward(n, target, Bt, s);
    if (rc) return rc;
    if (grad_host && cudaMemcpyAsync(grad_host, n->g, sizeof(float) * n->np, cudaMemcpyDeviceToHost, s))
        return ferr(n, BFS_ECUDA, "gradient download failed");
    if (loss_host && cudaMemcpyAsync(loss_host, n->loss, sizeof(float), cudaMemcpyDeviceToHost, s))
        return ferr(n, BFS_ECUDA, "loss download failed");
    return cudaStreamSynchronize(s) == cudaSuccess ? BFS_OK : ferr(n, BFS_ECUDA, "synchronisation failed");
}

// one Adam step on the mean squared error; asynchronous (loss stays on device,
// read it with bfs_cno_read_loss)
int bfs_cno_train_step(bfs_cno *n, const float *x, const float *target, int Bt, float lr, void *stream)
{
    if (!n || !x || !target || Bt < 1 || Bt > n->Bmax) return ferr(n, BFS_EINVAL, "bad arguments");
    cudaStream_t s = (cudaStream_t)stream;
    int rc = forward(n, x, Bt, s);
    if (!rc) rc = backward(n, target, Bt, s);
    if (rc) return rc;
    n->step++;
    const float b1 = 0.9f, b2 = 0.999f;
    const float c1 = 1.f - powf(b1, (float)n->step), c2 = 1.f - powf(b2, (float)n->step);
    k_adam<<<(n->np + 255) / 256, 256, 0, s>>>(n->p, n->g, n->m, n->v, n->np, lr, b1, b2, 1e-8f, c1, c2);
    cast_all(n, s);
    return cudaGetLastError() == cudaSuccess ? BFS_OK : ferr(n, BFS_ECUDA, "train step failed");
}

int bfs_cno_read_loss(bfs_cno *n, float *loss_host, void *stream)
{
    if (!n || !loss_host) return BFS_EINVAL;
    cudaStream_t s = (cudaStream_t)stream;
    if (cudaMemcpyAsync(loss_host, n->loss, sizeof(float), cudaMemcpyDeviceToHost, s) != cudaSuccess ||
        cudaStreamSynchronize(s) != cudaSuccess)
        return ferr(n, BFS_ECUDA, "loss download failed");
    return BFS_OK;
}

// Initial guess for ctx from the network: features x (device FP32 [1][M][N][4])
// -> nodal fields -> unknown vector u (device, length 3(N+1)M).
int bfs_cno_guess(bfs_cno *n, bfs_ctx *c, const float *x, double *u, void *stream)
{
    if (!n || !c || !x || !u) return ferr(n, BFS_EINVAL, "NULL argument");
    if (c->M != n->H || c->N != n->W) return ferr(n, BFS_EINVAL, "mesh does not match the network grid");
    cudaStream_t s = (cudaStream_t)stream;
    int rc = forward(n, x, 1, s);
    if (rc) return rc;
    const int tot = 3 * (c->N + 1) * c->M;
    k_fields_to_u<<<(tot + 255) / 256, 256, 0, s>>>(n->z[NL - 1], n->scale, u, c->N, c->M, c->dx, c->x1);
    return cudaGetLastError() == cudaSuccess ? BFS_OK : ferr(n, BFS_ECUDA, "guess launch failed");
}

int bfs_cno_solve(bfs_cno *n, bfs_ctx *c, const float *x, double *u, bfs_stats *st, int *used_fallback,
                  void *stream)
{
    if (!n || !c || !x || !u) return ferr(n, BFS_EINVAL, "NULL argument");
    if (used_fallback) *used_fallback = 0;
    int rc = bfs_cno_guess(n, c, x, u, stream);
    if (rc) return rc;
    bfs_stats s1{};
    rc = bfs_solve(c, u, &s1, stream);
    if (st) *st = s1;
    // accepted only through Newton: a guess from which the solve fails gives way
    // to the method without the network, the uniform stream
    if (rc == BFS_OK || !(rc == BFS_ENOCONV || rc == BFS_ELINESEARCH || rc == BFS_EBREAKDOWN ||
                          rc == BFS_ENAN || rc == BFS_ETIMEOUT))
        return rc;
    if (used_fallback) *used_fallback = 1;
    bfs_stats s2{};
    if ((rc = bfs_flat_guess(c, u, stream))) return rc;
    rc = bfs_solve(c, u, &s2, stream);
    if (st) {
        s2.newton_its += s1.newton_its;
        s2.krylov_its += s1.krylov_its;
        s2.residual_evals_fp64 += s1.residual_evals_fp64;
        s2.residual_evals_fp32 += s1.residual_evals_fp32;
        s2.precond_applies += s1.precond_applies;
        s2.seconds += s1.seconds;
        *st = s2;
    }
    return rc;
}

int bfs_cno_solve_host(bfs_cno *n, bfs_ctx *c, const float *x_host, double *u_host, bfs_stats *st,
                       int *used_fallback, void *stream)
{
    if (!n || !c || !x_host || !u_host) return ferr(n, BFS_EINVAL, "NULL argument");
    if (c->M != n->H || c->N != n->W) return ferr(n, BFS_EINVAL, "mesh does not match the network grid");
    cudaStream_t s = (cudaStream_t)stream;
    int rc = bfs::alloc_solver(c);
    if (rc) return ferr(n, rc, c->err);
    double *u = c->d_uio;  // the context's own device copy of the iterate
    if (cudaMemcpyAsync(n->xin, x_host, sizeof(float) * (size_t)n->H * n->W * 4, cudaMemcpyHostToDevice, s) !=
        cudaSuccess)
        return ferr(n, BFS_ECUDA, "upload of the features failed");
    rc = bfs_cno_solve(n, c, n->xin, u, st, used_fallback, stream);
    if (cudaMemcpyAsync(u_host, u, sizeof(double) * c->n, cudaMemcpyDeviceToHost, s) != cudaSuccess ||
        cudaStreamSynchronize(s) != cudaSuccess)
        return rc ? rc : ferr(n, BFS_ECUDA, "download of u failed");
    return rc;
}

}  // extern "C"

// FP64-grade GEMM of the block LU on the tensor cores: the operands are cut into
// slices of seven bits whose products and sums are exact (Ozaki, Ogita, Oishi and
// Rump, Numer. Algorithms 59 (2012); on FP16 tensor cores Mukunoki et al., ISC 2020).
//
//   a(i,k) = 2^ea(i) sum_s a_s(i,k) 2^(-7s-6),  b(k,j) = 2^eb(j) sum_t b_t(k,j) 2^(-7t-6)
//
// with integers |a_s|, |b_t| <= 64 from one fixed-point value per entry, scaled by
// the largest entry of the row of A and of the column of B.  Then
//   sum_k a b = 2^(ea+eb-12) sum_d 2^-7d sum_{s+t=d} sum_k a_s b_t.
// An inner sum is an integer below S K 2^12 <= 2^24 over a segment of K, so the FP32
// accumulation of FP16 products is exact in any order.  What is lost is the last bit
// of the fixed point, 2^-7S of the row's largest entry, and the products with
// s + t >= S, of the same size.  The S sums are put together in 64-bit integers and
// FP64.
//
// FP64 factors take S = SG_S64, the double-float ones (48 bits) SG_S32 slices: the
// fewest with which an apply is as close to 64 bits as with the products of
// precond.cu (181 x 61: FP64 6.9e-12 and 6.9e-12, FP32 sweeps 1.21e-7 and 1.23e-7;
// 121 x 41: 4.3e-12 and 4.2e-12, 5.8e-8 and 5.7e-8; 151 x 53: 4.6e-12 and 4.7e-12,
// 8.9e-8 and 9.5e-8).
//
// The FP64 pipe (two operations per clock and SM) bounds a plain product at 0.17 ms
// for 365 rows; S = 9 costs 45 FP16 products of about a thousandth of that each.  A
// factorisation takes 86 ms (151) at 181 x 61 in FP64, 48 (58) with FP32 sweeps, 128
// (179) at 241 x 81.
#include <cuda_fp16.h>
#include <math.h>

#include "bfs_internal.cuh"

namespace bfs {
namespace {

constexpr int SG_S64 = 9, SG_S32 = 8;
constexpr int SG_T = 64;          // output tile, and the padding of the slices
constexpr int SG_KC = 32;         // depth of a staged chunk
constexpr int SG_L = 16;          // rows or columns per CTA of k_sg_split
constexpr int SG_OPS = 24;        // operands whose slices are held at once
constexpr int SG_PRODS = 64;      // products per launch
constexpr int SG_MIN = 128;       // smallest blocks taken
constexpr int SG_BAD = 1 << 20;   // exponent of a row or column with a non-finite entry

struct SgSplit {
    const double *src[SG_OPS];
    unsigned cols;  // bit: the operand is a B, scaled by columns and stored transposed
};

struct SgProds {
    short a[SG_PRODS], b[SG_PRODS];
    double *C[SG_PRODS];
};

// A finite |x| = m 2^(e-1075), m of 53 bits (subnormals count as zero): x 2^F as an
// integer, F = 7 S - 1 - ex, where |x| < 2^ex.
__device__ __forceinline__ long long sg_fixed(double x, int F)
{
    const long long b = __double_as_longlong(x);
    const int e = (int)(b >> 52) & 0x7ff;
    if (e == 0) return 0;
    const long long m = (b & 0xfffffffffffffll) | 0x10000000000000ll;
    const int sh = e - 1075 + F;  // at most 7 S - 54
    long long q;
    if (sh >= 0) q = m << sh;
    else if (sh < -54) q = 0;
    else q = (m + (1ll << (-sh - 1))) >> -sh;
    return b < 0 ? -q : q;
}

// Slices of 16 rows (A) or columns (B) of an operand, the entries of a line along k
// contiguous: two passes over the lines through shared memory, the second one from
// L2.  Bound by latency and the stores; integer arithmetic only (an FP64 operation
// per entry and slice would cost more than the product).
template <int S>
__global__ void __launch_bounds__(256) k_sg_split(SgSplit sp, int n, int P, unsigned short *__restrict__ out,
                                                  int *__restrict__ ex)
{
    __shared__ double t[SG_L][SG_T + 1];
    const int op = blockIdx.y, l0 = blockIdx.x * SG_L, tid = threadIdx.x;
    const double *src = sp.src[op];
    const bool cols = sp.cols >> op & 1;
    unsigned short *dst = out + (size_t)op * S * P * P;
    auto load = [&](int k0) {
        __syncthreads();
#pragma unroll
        for (int e = tid; e < SG_L * SG_T; e += 256) {
            const int l = cols ? e % SG_L : e / SG_T, k = cols ? e / SG_L : e % SG_T;
            const int gl = l0 + l, gk = k0 + k;
            t[l][k] = gl < n && gk < n ? (cols ? src[(size_t)gk * n + gl] : src[(size_t)gl * n + gk]) : 0.0;
        }
        __syncthreads();
    };
    const int l = tid / 16, q = tid % 16 * 4;
    int top = 0;  // largest biased exponent of the line
    for (int k0 = 0; k0 < n; k0 += SG_T) {
        load(k0);
#pragma unroll
        for (int j = 0; j < 4; j++)
            top = max(top, (int)(__double_as_longlong(t[l][q + j]) >> 52) & 0x7ff);
    }
#pragma unroll
    for (int o = 8; o; o >>= 1) top = max(top, __shfl_xor_sync(0xffffffffu, top, o));
    const int e = top - 1022, F = 7 * S - 1 - e;
    if (tid % 16 == 0) ex[op * P + l0 + l] = top == 0x7ff ? SG_BAD : top == 0 ? 0 : e;
    for (int k0 = 0; k0 < P; k0 += SG_T) {
        load(k0);
        long long v[4];
#pragma unroll
        for (int j = 0; j < 4; j++) v[j] = top == 0x7ff ? 0 : sg_fixed(t[l][q + j], F);
#pragma unroll
        for (int s = S - 1; s >= 0; s--) {
            ushort4 w;
            unsigned short *wp = &w.x;
#pragma unroll
            for (int j = 0; j < 4; j++) {
                const int d = s ? (((int)v[j] + 64) & 127) - 64 : (int)v[j];
                v[j] = (v[j] - d) >> 7;
                wp[j] = __half_as_ushort(__int2half_rn(d));
            }
            *reinterpret_cast<ushort4 *>(dst + ((size_t)s * P + l0 + l) * P + k0 + q) = w;
        }
    }
}

__device__ __forceinline__ void sg_ldm(unsigned (&r)[4], unsigned addr)
{
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0,%1,%2,%3}, [%4];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
                 : "r"(addr));
}

__device__ __forceinline__ void sg_mma(float (&c)[4], const unsigned (&a)[4], unsigned b0, unsigned b1)
{
    asm volatile("mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, "
                 "{%0,%1,%2,%3};"
                 : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
                 : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}

// an integer of less than 2^51 to FP64 by one FP64 subtraction (1.5 2^52 + v is exact)
__device__ __forceinline__ double sg_double(long long v)
{
    return __longlong_as_double(v + 0x4338000000000000ll) - 6755399441055744.0;
}

__device__ __forceinline__ double sg_scale(double v, int e)
{
    if (e >= -1000 && e <= 1000) return v * __longlong_as_double((long long)(e + 1023) << 52);
    return ldexp(v, e);
}

// C = alpha A B + beta C for a batch of products, 64 x 64 tiles, eight warps of 32 x 16.
// All S diagonals of a tile stay in registers (16 S a thread), so every slice of a
// chunk is staged once for its S (S + 1) / 2 products, against shared-memory and
// L2 traffic of every pair otherwise; that is why the tile is no larger.  The sums are
// mma.sync fragments: in tensor memory nine sums of 128 x 64 would be 576 columns, more
// than it has; those of 128 x 48 (432 columns) would fit and have not been tried.  Copies
// of the next chunk run (cp.async) under the products of this one.  The 17 products of a
// 365-row slice take 0.41 ms (1.65 with k_dgemm).  The tensor pipe is 60 % busy on the SMs
// that have a tile: 36 for one product (62 us), one CTA each, so that of the 216 to 324
// tiles of a batch the last wave counts.
template <int S>
__global__ void __launch_bounds__(256, 1) k_sg_gemm(SgProds pr, const unsigned short *__restrict__ sl,
                                                    const int *__restrict__ ex, int n, int P, int seg, double alpha,
                                                    double beta)
{
    extern __shared__ __align__(128) unsigned char sm[];
    constexpr int TB = SG_T * SG_KC * 2;  // bytes of one slice of one operand's chunk
    const int pz = blockIdx.z, tid = threadIdx.x, lane = tid % 32, wm = tid / 32 % 2, wn = tid / 64;
    const int row0 = blockIdx.y * SG_T, col0 = blockIdx.x * SG_T;
    const unsigned short *A = sl + (size_t)pr.a[pz] * S * P * P + (size_t)row0 * P;
    const unsigned short *B = sl + (size_t)pr.b[pz] * S * P * P + (size_t)col0 * P;
    const unsigned base = (unsigned)__cvta_generic_to_shared(sm);
    // 16-byte unit u of row r lies at unit u ^ (r / 2 % 4) of the row: eight rows of
    // one ldmatrix then touch all banks
    auto stage = [&](int buf, int k0) {
        const int r = tid / 4, u = tid % 4;
        const unsigned d = base + buf * (2 * S * TB) + r * 64 + ((u ^ (r >> 1 & 3)) << 4);
        const size_t g = (size_t)r * P + k0 + u * 8;
#pragma unroll
        for (int s = 0; s < S; s++) {
            asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(d + s * TB),
                         "l"(A + (size_t)s * P * P + g));
            asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(d + (S + s) * TB),
                         "l"(B + (size_t)s * P * P + g));
        }
        asm volatile("cp.async.commit_group;");
    };
    float acc[S][2][2][4];
#pragma unroll
    for (int i = 0; i < S * 16; i++) (&acc[0][0][0][0])[i] = 0.f;
    // ldmatrix: lanes 0-15 the rows of the first eight columns of k, 16-31 of the second;
    // for B, lanes 0-7 / 8-15 the two halves of k of the first eight columns
    const int ar = wm * 32 + lane % 16, au = lane / 16;
    const int br = wn * 16 + lane / 16 * 8 + lane % 8, bu = lane / 8 % 2;
    double b1 = beta;
    auto fold = [&]() {
        double *C = pr.C[pz];
        const int *ea = ex + pr.a[pz] * P + row0, *eb = ex + pr.b[pz] * P + col0;
#pragma unroll
        for (int mi = 0; mi < 2; mi++)
#pragma unroll
            for (int ni = 0; ni < 2; ni++)
#pragma unroll
                for (int q = 0; q < 4; q++) {
                    const int r = wm * 32 + mi * 16 + lane / 4 + q / 2 * 8;
                    const int cc = wn * 16 + ni * 8 + lane % 4 * 2 + q % 2;
                    // up to three sums fit an integer of 2^39, the rest in a second and third
                    constexpr int G = (S + 2) / 3;
                    double v = 0.0;
#pragma unroll
                    for (int g = 2; g >= 0; g--) {
                        long long w = 0;
                        int cnt = 0;
#pragma unroll
                        for (int d = g * G; d < (g + 1) * G; d++)
                            if (d < S) {
                                w = w * 128 + __float2int_rn(acc[d][mi][ni][q]);
                                cnt++;
                            }
                        // v = group g + 2^-7G of the groups after it, in units of its last sum
                        const double lead = sg_double(w);
                        const int up = 7 * (G - cnt);  // a short last group
                        v = fma(v, __longlong_as_double((long long)(1023 - 7 * G) << 52),
                                lead * __longlong_as_double((long long)(1023 + up) << 52));
                    }
                    // units of the first group's last sum: 2^-7(G-1)
                    if (row0 + r < n && col0 + cc < n) {
                        const int e0 = ea[r], e1 = eb[cc];
                        v = e0 == SG_BAD || e1 == SG_BAD ? __longlong_as_double(0x7ff8000000000000ll)
                                                         : sg_scale(v, e0 + e1 - 12 - 7 * (G - 1));
                        double *cp = C + (size_t)(row0 + r) * n + col0 + cc;
                        *cp = b1 == 0.0 ? alpha * v : fma(alpha, v, b1 * *cp);
                    }
                }
    };
    const int nch = (n + SG_KC - 1) / SG_KC;
    stage(0, 0);
    for (int ch = 0; ch < nch; ch++) {
        if (ch + 1 < nch) {
            stage((ch + 1) & 1, (ch + 1) * SG_KC);
            asm volatile("cp.async.wait_group 1;");
        } else {
            asm volatile("cp.async.wait_group 0;");
        }
        __syncthreads();
        const unsigned sa = base + (ch & 1) * (2 * S * TB), sb = sa + S * TB;
#pragma unroll
        for (int k2 = 0; k2 < SG_KC / 16; k2++) {
            unsigned b[S][4];
            {
                const unsigned off = br * 64 + (((k2 * 2 + bu) ^ (br >> 1 & 3)) << 4);
#pragma unroll
                for (int t = 0; t < S; t++) sg_ldm(b[t], sb + t * TB + off);
            }
#pragma unroll
            for (int s = 0; s < S; s++) {
                unsigned a[2][4];
#pragma unroll
                for (int mi = 0; mi < 2; mi++) {
                    const int r = ar + mi * 16;
                    sg_ldm(a[mi], sa + s * TB + r * 64 + (((k2 * 2 + au) ^ (r >> 1 & 3)) << 4));
                }
#pragma unroll
                for (int t = 0; t < S - s; t++)
#pragma unroll
                    for (int mi = 0; mi < 2; mi++) {
                        sg_mma(acc[s + t][mi][0], a[mi], b[t][0], b[t][1]);
                        sg_mma(acc[s + t][mi][1], a[mi], b[t][2], b[t][3]);
                    }
            }
        }
        if ((ch + 1) % seg == 0 && ch + 1 < nch) {  // the sums are no longer exact beyond a segment
            fold();
            b1 = 1.0;
#pragma unroll
            for (int i = 0; i < S * 16; i++) (&acc[0][0][0][0])[i] = 0.f;
        }
        __syncthreads();
    }
    fold();
}

template <int S>
int run(bfs_ctx *c, const std::vector<const double *> &A, const std::vector<const double *> &B,
        const std::vector<double *> &C, int n, double alpha, double beta, cudaStream_t s)
{
    const int P = (n + SG_T - 1) / SG_T * SG_T;
    const size_t smem = 2 * (size_t)2 * S * SG_T * SG_KC * 2;
    const int seg = (1 << 24) / (S << 12) / SG_KC;  // chunks whose sums stay below 2^24
    unsigned short *sl = static_cast<unsigned short *>(c->d_slices);
    int *ex = reinterpret_cast<int *>(sl + (size_t)SG_OPS * S * P * P);
    BFS_CUDA_TRY(c, cudaFuncSetAttribute((const void *)k_sg_gemm<S>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         (int)smem));
    for (size_t o = 0; o < A.size();) {
        SgSplit sp{};
        SgProds pr{};
        int nop = 0, cnt = 0;
        auto find = [&](const double *p, bool cols) {
            for (int i = 0; i < nop; i++)
                if (sp.src[i] == p && (sp.cols >> i & 1) == (unsigned)cols) return i;
            return -1;
        };
        for (; o < A.size() && cnt < SG_PRODS; o++, cnt++) {
            int ia = find(A[o], false), ib = find(B[o], true);
            if (nop + (ia < 0) + (ib < 0) > SG_OPS) break;
            if (ia < 0) sp.src[ia = nop++] = A[o];
            if (ib < 0) {
                sp.cols |= 1u << nop;
                sp.src[ib = nop++] = B[o];
            }
            pr.a[cnt] = (short)ia;
            pr.b[cnt] = (short)ib;
            pr.C[cnt] = C[o];
        }
        k_sg_split<S><<<dim3(P / SG_L, nop), 256, 0, s>>>(sp, n, P, sl, ex);
        k_sg_gemm<S><<<dim3(P / SG_T, P / SG_T, cnt), 256, smem, s>>>(pr, sl, ex, n, P, seg, alpha, beta);
        c->launches += 2;
    }
    BFS_CUDA_TRY(c, cudaGetLastError());
    return BFS_OK;
}

}  // namespace

// From 128 rows up, where a factorisation is not slower (45 x 15, 138 rows: FP64 7.6 ms
// against 7.7, FP32 sweeps 3.8 against 3.9; 61 x 21: 13.0 against 14.0, 6.3 against 6.8),
// and not with surface tension, whose rows span too many binades for one scale.
// Scratch for the slices; without it the GEMM kernels of precond.cu take the products.
void sg_alloc(bfs_ctx *c)
{
    if (c->nb < SG_MIN || c->opt.surface_tension != 0.0) return;
    const size_t P = (c->nb + SG_T - 1) / SG_T * SG_T;
    const int S = c->opt.precond_precision == BFS_FP32C ? SG_S32 : SG_S64;
    if (cudaMalloc(&c->d_slices, SG_OPS * (2 * S * P * P + sizeof(int) * P)) != cudaSuccess) {
        cudaGetLastError();
        c->d_slices = nullptr;
    }
}

// A, B, C as for the batches of precond.cu; within one call no C is an A or a B
int sg_gemm(bfs_ctx *c, const std::vector<const double *> &A, const std::vector<const double *> &B,
            const std::vector<double *> &C, double alpha, double beta, cudaStream_t s)
{
    return c->opt.precond_precision == BFS_FP32C ? run<SG_S32>(c, A, B, C, c->nb, alpha, beta, s)
                                                 : run<SG_S64>(c, A, B, C, c->nb, alpha, beta, s);
}

}  // namespace bfs

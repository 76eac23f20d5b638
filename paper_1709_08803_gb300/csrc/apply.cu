// Application of the factored block-banded preconditioner, z = P^{-1} r
// (Sec. 4.2 and App. A: the banded linear Jacobian, factored by block LU),
// in FP32 over an FP32 copy of the FP64 factors.
//
// The sweeps are chains of dependent slice steps.  With the one-ended LU
// (factored from slice 0 down) they are forward
//   y_k = x_k - sum_{i=k-h}^{k-1} L_ki y_i,
// then backward
//   z_k = D_k^-1 y_k - sum_{j=k+1}^{k+h} W_kj z_j,
// 2M steps in one chain.  The two-ended ("twisted") LU eliminates slices
// 0..t-1 downwards and M-1..t+h upwards; the two chains touch only the h
// middle slices, whose Schur complement C is inverted whole.  Its sweeps run
// as two chains side by side: forward from the top and upward from the bottom
// (y_k = x_k - sum U'_kj y_j, j = k+1..k+h), the middle y (both chains' terms),
// z_mid = C^-1 y_mid, and the back substitutions outwards -- about M dependent
// steps instead of 2M.
//
// Every step, in either form, is one task of a host-built table: the slice it
// finishes, whether it writes y (and adds the right-hand side) or z, and the
// stored blocks it multiplies, each with the vector slice it multiplies and the
// task that wrote that slice.  CTAs are split into as many groups as there are
// chains; a group runs its tasks in order, each CTA owning a contiguous run of
// rows of every slice.
//
// Dataflow instead of a grid barrier: every entry of y and z is one 64-bit
// word holding the FP32 value and a tag naming the launch and task that wrote
// it, stored and loaded with single-copy-atomic relaxed accesses.  A CTA loads
// the vector words of all its blocks at the start of a step, multiplies the
// ones that are ready, and then each thread spins only on the tags of the
// entries still missing -- in practice those the group's previous task wrote.
// The critical path per step is one producer-to-consumer trip through L2 plus
// a short dot product.  Tags grow with every launch (the buffers are zeroed
// when the preconditioner is factored or a wait has timed out, tags start at
// 1), so an entry left by an earlier launch never matches.
//
// The launches are cooperative (all CTAs resident), so every awaited entry is
// eventually written.  Each spin is still bounded (about a second by default,
// the option wait_polls otherwise); a thread that gives up raises bit 2 of the
// context flag and the CTA returns at its next step boundary.  A launch that
// finds bit 2 already raised does nothing: the host clears it, and resets the
// tagged vectors, when it reads the flag.
#include <string.h>

#include <algorithm>
#include <vector>

#include "bfs_internal.cuh"

namespace bfs {

struct FlowArgs {
    const float *pc;               // FP32 factors: block (k, m) row r at ((k nd + m - k + h) nb + r) ldp
    const double *r;               // right-hand side, order of u (condensed blocks: slice by slice)
    double *z;                     // result, in the same order
    unsigned long long *X, *Y;     // tagged slice-ordered vectors, M * nb each
    int nb, NB, M, h;
    int ldp;                       // padded row length of the FP32 factors (multiple of 4)
    int nslot;                     // shared-memory ring depth (task-table kernel)
    int sw, vs;                    // words a CTA owns in a vector slice, and a slice has (task-table kernel)
    int zpair;                     // write z as float pairs (condensed blocks; task-table kernel)
    int rows;                      // rows of a slice per CTA at most: its compute warps (task-table kernel)
    unsigned int *tagp;            // device word: tag of this launch's first step; step (task) s
                                   // writes tag0 + s, and block 0 advances the word by ntags on exit
    int *flag;
    unsigned int spin;             // polls of one wait before giving up
    const SweepDev *tasks;         // task table: group 0's tasks, then group 1's
    int ntask0, ntask1;            // tasks per group
    int G0;                        // CTAs of group 0 (the rest form group 1)
    int ntags;                     // tags one launch uses (= ntask0 + ntask1)
};

constexpr int FL_TPB = 512;
constexpr int FL_WARPS = FL_TPB / 32;
constexpr unsigned int FL_SPIN = 1u << 20;  // default polls of one entry before giving up (~1 s)

__device__ __forceinline__ unsigned long long ld_word(const unsigned long long *p)
{
    unsigned long long v;
    asm volatile("ld.relaxed.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
    return v;
}

__device__ __forceinline__ void st_word(unsigned long long *p, float v, unsigned int tag)
{
    const unsigned long long w = ((unsigned long long)tag << 32) | __float_as_uint(v);
    asm volatile("st.relaxed.gpu.global.u64 [%0], %1;" ::"l"(p), "l"(w) : "memory");
}

__device__ __forceinline__ unsigned int ld_tag(const unsigned int *p)
{
    unsigned int v;
    asm volatile("ld.relaxed.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}

// The launch's last CTA to depend on every other one advances the tag word,
// so every CTA has read this launch's tag by then and the next launch may use
// the next tags.
__device__ __forceinline__ void advance_tag(unsigned int *p, unsigned int tag0, unsigned int ntags)
{
    const unsigned int next = tag0 + ntags;
    asm volatile("st.relaxed.gpu.global.u32 [%0], %1;" ::"l"(p), "r"(next) : "memory");
}

// hi + lo += b: Knuth's two-sum (the explicit _rn operations keep the compiler
// from contracting).  The sweeps' rows cancel, so their sums are carried as
// pairs: the error left is that of the FP32 factors and products.
__device__ __forceinline__ void pair_add(float &hi, float &lo, float b)
{
    const float s = __fadd_rn(hi, b);
    const float bb = __fsub_rn(s, hi);
    lo = __fadd_rn(lo, __fadd_rn(__fsub_rn(hi, __fsub_rn(s, bb)), __fsub_rn(b, bb)));
    hi = s;
}

// Values of CPT tagged entries (those with cv set) once their tags are `tag`,
// w holding what an earlier load returned; all entries still missing are polled
// together, so that a wait costs one round trip through L2 whatever CPT is.
// False after `spin` polls.
template <int CPT>
__device__ __forceinline__ bool await_words(const unsigned long long *p, const int (&col)[CPT], const bool (&cv)[CPT],
                                            unsigned int tag, unsigned long long (&w)[CPT], float (&v)[CPT],
                                            unsigned int spin)
{
    unsigned int spins = 0;
    while (true) {
        bool all = true;
#pragma unroll
        for (int q = 0; q < CPT; q++) all = all && (!cv[q] || (unsigned int)(w[q] >> 32) == tag);
        if (all) break;
        if (++spins > spin) return false;
#pragma unroll
        for (int q = 0; q < CPT; q++)
            if (cv[q] && (unsigned int)(w[q] >> 32) != tag) w[q] = ld_word(p + col[q]);
    }
#pragma unroll
    for (int q = 0; q < CPT; q++) v[q] = cv[q] ? __uint_as_float((unsigned int)w[q]) : 0.f;
    return true;
}

// Value of a tagged entry once its tag is `tag`; false after `spin` polls.
__device__ __forceinline__ bool await_word(const unsigned long long *p, unsigned int tag, float &v,
                                           unsigned int spin)
{
    unsigned long long w = ld_word(p);
    unsigned int spins = 0;
    while ((unsigned int)(w >> 32) != tag) {
        if (++spins > spin) return false;
        __nanosleep(32);
        w = ld_word(p);
    }
    v = __uint_as_float((unsigned int)w);
    return true;
}

// Sums as float pairs for condensed blocks (whose rows cancel more), plain FP32
// ones otherwise.
template <bool PAIR>
__device__ __forceinline__ void flow_add(float &hi, float &lo, float b)
{
    if constexpr (PAIR) pair_add(hi, lo, b);
    else hi += b;
}

template <int RPC, int CPT, bool PAIR>
__global__ void __launch_bounds__(FL_TPB, 1) k_apply_flow(FlowArgs a)
{
    __shared__ float2 red[RPC][FL_WARPS];
    __shared__ unsigned int tag_sh;
    const float *pc = a.pc;
    const int nb = a.nb, NB = a.NB, M = a.M, h = a.h, nd = 2 * h + 1, G = gridDim.x;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    __shared__ int abort_sh;
    if ((int)blockIdx.x >= nb) return;  // no rows here
    if (tid == 0) {
        abort_sh = (ld_tag(reinterpret_cast<const unsigned int *>(a.flag)) & 2u) != 0;
        tag_sh = ld_tag(a.tagp);
    }
    __syncthreads();
    if (abort_sh) return;  // an earlier wait timed out: the host resets the vectors first
    const unsigned int tag0 = tag_sh;

    int row[RPC];
    bool rv[RPC];
#pragma unroll
    for (int j = 0; j < RPC; j++) {
        row[j] = blockIdx.x + j * G;
        rv[j] = row[j] < nb;
        if (!rv[j]) row[j] = 0;
    }
    int col[CPT];
    bool cv[CPT];
#pragma unroll
    for (int q = 0; q < CPT; q++) {
        col[q] = tid + q * FL_TPB;
        cv[q] = col[q] < nb;
        if (!cv[q]) col[q] = 0;
    }
    // the thread that finishes row j (tid == j) and its index in the order of u
    const int my_j = tid < RPC ? tid : -1;
    const bool my_rv = my_j >= 0 && blockIdx.x + my_j * G < nb;
    size_t my_e = 0;
    if (my_rv) {
        const int rw = blockIdx.x + my_j * G, g = rw / NB, p = rw - g * NB;
        my_e = (size_t)g * NB * M + p;  // + l NB for slice l
    }

    auto step_of = [&](int s, int &pass, int &k, int &lo, int &hi, int &crit) {
        pass = s < M ? 0 : 1;
        k = pass == 0 ? s : 2 * M - 1 - s;
        if (pass == 0) {
            lo = max(0, k - h); hi = k - 1;
            crit = (k >= 1 && h >= 1) ? k - 1 : -1;
        } else {
            lo = k; hi = min(M - 1, k + h);
            crit = (k == M - 1) ? k : (h >= 1 ? k + 1 : -1);
        }
    };
    // step that wrote the vector multiplied by block (k, m) in pass `pass`
    auto producer = [&](int pass, int k, int m) { return (pass == 0 || m == k) ? m : 2 * M - 1 - m; };
    auto vec = [&](int pass, int k, int m) -> const unsigned long long * {
        return (pass == 0 || m == k) ? a.Y + (size_t)m * nb : a.X + (size_t)m * nb;
    };
    const int ldp = a.ldp;
    auto block_row = [&](int k, int m, int j) { return pc + (((size_t)k * nd + (m - k + h)) * nb + row[j]) * ldp; };
    auto prefetch = [&](int s) {
        if (s >= 2 * M) return;
        int pass, k, lo, hi, crit;
        step_of(s, pass, k, lo, hi, crit);
        constexpr int per_line = 32;  // floats per 128-byte line
        const int nlines = (nb + per_line - 1) / per_line;
        for (int m = lo; m <= hi; m++)
            for (int idx = tid; idx < RPC * nlines; idx += FL_TPB) {
                const int j = idx / nlines, ln = idx - j * nlines;
                const int rw = blockIdx.x + j * G;
                if (rw < nb) {
                    const float *bp = pc + (((size_t)k * nd + (m - k + h)) * nb + rw) * ldp + ln * per_line;
                    asm volatile("prefetch.global.L2 [%0];" ::"l"(bp));
                }
            }
    };

    prefetch(0);
    prefetch(1);
    bool ok = true;
    for (int s = 0; s < 2 * M; s++) {
        int pass, k, lo, hi, crit;
        step_of(s, pass, k, lo, hi, crit);
        prefetch(s + 2);
        float acc[RPC], alo[RPC];
#pragma unroll
        for (int j = 0; j < RPC; j++) acc[j] = alo[j] = 0.f;
        double xk = 0.0;
        if (pass == 0 && my_rv) xk = a.r[my_e + (size_t)k * NB];

        // terms whose vectors were finished two or more steps ago, two blocks
        // in flight at a time (their tags are checked all the same)
        for (int m = lo; m <= hi; m++) {
            if (m == crit) continue;
            int m2 = m + 1;
            if (m2 == crit) m2++;
            const bool two = m2 <= hi;
            float f[2][RPC][CPT], v[2][CPT];
#pragma unroll
            for (int bb = 0; bb < 2; bb++) {
                const int mm = (bb == 0 || !two) ? m : m2;
                const bool use = bb == 0 || two;
                const unsigned long long *vp = vec(pass, k, mm);
                const unsigned int tg = tag0 + producer(pass, k, mm);
#pragma unroll
                for (int q = 0; q < CPT; q++) {
                    v[bb][q] = 0.f;
                    if (ok && use && cv[q]) ok = await_word(vp + col[q], tg, v[bb][q], a.spin);
                }
#pragma unroll
                for (int j = 0; j < RPC; j++) {
                    const float *bp = block_row(k, mm, j);
#pragma unroll
                    for (int q = 0; q < CPT; q++) f[bb][j][q] = (use && rv[j] && cv[q]) ? __ldg(bp + col[q]) : 0.f;
                }
            }
#pragma unroll
            for (int bb = 0; bb < 2; bb++) {
                const int mm = (bb == 0 || !two) ? m : m2;
                const float sg = (pass == 1 && mm == k) ? 1.f : -1.f;
#pragma unroll
                for (int j = 0; j < RPC; j++) {
                    float t = 0.f;
#pragma unroll
                    for (int q = 0; q < CPT; q++) t = fmaf(f[bb][j][q], v[bb][q], t);
                    flow_add<PAIR>(acc[j], alo[j], sg * t);
                }
            }
            if (two) m = m2;
        }

        // the dependent block: registers first, then wait for its vector
        if (crit >= 0) {
            float cf[RPC][CPT];
#pragma unroll
            for (int j = 0; j < RPC; j++) {
                const float *bp = block_row(k, crit, j);
#pragma unroll
                for (int q = 0; q < CPT; q++) cf[j][q] = (rv[j] && cv[q]) ? __ldg(bp + col[q]) : 0.f;
            }
            const float sg = (pass == 1 && crit == k) ? 1.f : -1.f;
            const unsigned long long *vp = vec(pass, k, crit);
            const unsigned int tg = tag0 + (unsigned int)(s - 1);
            float v[CPT];
            unsigned long long wv[CPT];
#pragma unroll
            for (int q = 0; q < CPT; q++) {
                v[q] = 0.f;
                wv[q] = cv[q] ? ld_word(vp + col[q]) : 0ull;
            }
            if (ok) ok = await_words<CPT>(vp, col, cv, tg, wv, v, a.spin);
#pragma unroll
            for (int j = 0; j < RPC; j++) {
                float t = 0.f;
#pragma unroll
                for (int q = 0; q < CPT; q++) t = fmaf(cf[j][q], v[q], t);
                flow_add<PAIR>(acc[j], alo[j], sg * t);
            }
        }
#pragma unroll
        for (int j = 0; j < RPC; j++) {
            float t = acc[j], tl = alo[j];
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) {
                const float ol = PAIR ? __shfl_xor_sync(0xffffffffu, tl, o) : 0.f;
                flow_add<PAIR>(t, tl, __shfl_xor_sync(0xffffffffu, t, o));
                tl += ol;
            }
            if (lane == 0) red[j][warp] = make_float2(t, tl);
        }
        if (!__syncthreads_and(ok)) {
            if (tid == 0) {
                atomicOr(a.flag, 2);
                if (blockIdx.x == 0) advance_tag(a.tagp, tag0, 2u * (unsigned int)M);
            }
            return;
        }
        if (my_rv) {
            float t = 0.f, tl = 0.f;
#pragma unroll
            for (int w = 0; w < FL_WARPS; w++) {
                flow_add<PAIR>(t, tl, red[my_j][w].x);
                tl += red[my_j][w].y;
            }
            const size_t si = (size_t)k * nb + blockIdx.x + my_j * G;
            const unsigned int tg = tag0 + (unsigned int)s;
            if (pass == 0) {
                const float xh = (float)xk;
                pair_add(t, tl, xh);
                st_word(a.Y + si, t + (tl + (float)(xk - (double)xh)), tg);
            } else {
                st_word(a.X + si, t + tl, tg);
                a.z[my_e + (size_t)k * NB] = (double)t + (double)tl;
            }
        }
        __syncthreads();  // red is rewritten by the next step
    }
    if (blockIdx.x == 0 && tid == 0) advance_tag(a.tagp, tag0, 2u * (unsigned int)M);
}

// ---------------------------------------------------------------------------
// Task-table kernel for slice blocks that fit its tiles (at most 8 rows of a
// slice per CTA, at most 576 columns, at most SW_BMAX blocks per task).
//
// What bounds it is the latency of one task: the vector that the group's
// previous task wrote has to reach every CTA through L2, be multiplied and be
// written again, about M times in a row.  So the roles are split by warp, and
// nothing but that vector's own path is on it:
//   - a producer warp streams the CTA's rows of every block of a task into a ring
//     of `nslot` shared-memory slots with 1-D bulk copies (cp.async.bulk,
//     completion counted in bytes on a "full" mbarrier per slot), up to nslot - 1
//     tasks ahead;
//   - PW poll warps own two vector entries a thread and do nothing but load tagged
//     words and put their values into shared memory: a task's prefetched vectors
//     first ("early" mbarrier), then the critical one ("crit" mbarrier), both
//     words polled in one loop without sleeping in between;
//   - one compute warp per row: 16-byte shared loads of the row and the vectors, the
//     terms that need not wait first, then the critical one, a shuffle reduction,
//     and lane 0 writes the entry.  No barrier of the CTA is left in the loop.
// The last two critical vectors stay in the compute warps' registers, where the
// next tasks need them again, and the right-hand sides are staged at the start.
//
// 181 x 61 (h = 3, 62 dependent tasks), condensed blocks: 104 us a launch, 1.7 us
// a task; the kernel before it (columns over threads, a CTA barrier and a
// cross-warp sum per task) took 133 us on the same blocks and 139 us on the full
// ones.  241 x 81 (h = 4): 0.99 ms (one-ended, k_apply_flow) -> 0.19 ms.
//
// Buffers: a poll warp writes for task s only once every compute warp is done
// with task s - 2 (the ring's "empty" barriers), so a task's vectors alternate
// between two sets.  Every wait is
// bounded; a warp that gives up raises bit 2 of the flag and `dead`, which ends
// the other warps' waits.
// ---------------------------------------------------------------------------
__device__ __forceinline__ unsigned int smem_u32(const void *p)
{
    return (unsigned int)__cvta_generic_to_shared(p);
}

__device__ __forceinline__ bool mbar_try(unsigned int bar, unsigned int parity)
{
    unsigned int done;
    asm volatile(
        "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}"
        : "=r"(done)
        : "r"(bar), "r"(parity)
        : "memory");
    return done != 0;
}

// Waits inside the CTA last as long as its poll warps' waits, whose polls are L2
// round trips: SW_WAIT of these cheaper polls for each of theirs.
constexpr unsigned long long SW_WAIT = 64;

__device__ __forceinline__ bool mbar_wait(unsigned int bar, unsigned int parity, unsigned int spin, volatile int *dead)
{
    const unsigned long long lim = SW_WAIT * spin;
    for (unsigned long long i = 0; i < lim; i++) {
        if (mbar_try(bar, parity)) return true;
        if (dead && *dead) return false;
    }
    return false;
}

__device__ __forceinline__ void mbar_arrive(const void *bar)
{
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(bar)) : "memory");
}

__device__ __forceinline__ void mbar_init(const void *bar, unsigned int count)
{
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count) : "memory");
}

static_assert(SW_HW == 2, "the compute warps hold two critical vectors in registers");
constexpr int SW_ROWS = 8;  // compute warps at most, one row each
constexpr long long SW_BACKOFF = 400;

template <int PW, int WPT, int NQ, int BM>
__global__ void __launch_bounds__(32 * (SW_ROWS + PW + 1), 1) k_apply_sweep(FlowArgs a)
{
    constexpr int MAXSLOT = 8, PT = 32 * PW;  // poll threads, each owning WPT words
    static_assert(BM <= SW_BMAX, "task table rows");
    extern __shared__ __align__(128) float ring[];  // nslot x (h + 1) x rows x ldp, vector buffers, the group's tasks
    __shared__ __align__(8) unsigned long long full[MAXSLOT], empty[MAXSLOT], early[2], crit[2];
    __shared__ unsigned int tag_sh;
    __shared__ int abort_sh;
    __shared__ volatile int dead;
    __shared__ float outv[4][SW_ROWS];  // a task's rows, until the CTA's last warp stores them together
    __shared__ int ndone[2];            // rows done in the even and in the odd tasks since the launch
    const float *pc = a.pc;
    const int nb = a.nb, NB = a.NB, h = a.h, nd = 2 * h + 1, ldp = a.ldp;
    const int nslot = a.nslot, rows = a.rows;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const size_t slot_floats = (size_t)(h + 1) * rows * ldp;
    // CTA group and its tasks
    const int grp = (int)blockIdx.x < a.G0 ? 0 : 1;
    const int Gg = a.G0;  // CTAs of either group
    const int lb = grp ? (int)blockIdx.x - a.G0 : (int)blockIdx.x;
    const SweepDev *gtasks = a.tasks + (grp ? a.ntask0 : 0);
    const int ntask = grp ? a.ntask1 : a.ntask0;
    float *vbuf = ring + (size_t)nslot * slot_floats;  // 2 critical vectors of ldp, then 2 x (h + 1) early ones
    // the task table, staged once: a descriptor read from global memory at
    // every step would put an L2 round trip in front of each step's waits
    SweepDev *tasks = reinterpret_cast<SweepDev *>(vbuf + (size_t)(2 + 2 * (h + 1)) * ldp);
    float2 *xs = reinterpret_cast<float2 *>(tasks + ntask);  // right-hand sides of this CTA's rows, task by task
    // rows [r0, r0 + nrv) of every slice: the first nb % Gg CTAs take one row more
    const int base = nb / Gg, extra = nb % Gg;
    const int nrv = base + (lb < extra ? 1 : 0);
    const int r0 = lb * base + min(lb, extra);

    if (nrv == 0 || ntask == 0) return;  // no rows here
    if (tid == 0) {
        abort_sh = (ld_tag(reinterpret_cast<const unsigned int *>(a.flag)) & 2u) != 0;
        tag_sh = ld_tag(a.tagp);
        dead = 0;
        ndone[0] = ndone[1] = 0;
        for (int i = 0; i < nslot; i++) {
            mbar_init(&full[i], 1);
            mbar_init(&empty[i], nrv);
        }
        for (int i = 0; i < 2; i++) {
            mbar_init(&early[i], PW);
            mbar_init(&crit[i], PW);
        }
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    for (int i = tid; i < (2 + 2 * (h + 1)) * ldp; i += blockDim.x) vbuf[i] = 0.f;  // the padding stays 0
    for (int i = tid; i < ntask * rows; i += blockDim.x) {  // as float pairs; 0 for z tasks
        const int s = i / rows, j = i - s * rows;
        float2 x = make_float2(0.f, 0.f);
        if (gtasks[s].head.y == 0 && j < nrv) {
            const int row = r0 + j, g = row / NB, pp = row - g * NB;
            const double xk = a.r[(size_t)g * NB * a.M + pp + (size_t)gtasks[s].head.x * NB];
            x.x = (float)xk;
            x.y = (float)(xk - (double)x.x);
        }
        xs[i] = x;
    }
    {
        const int4 *src = reinterpret_cast<const int4 *>(gtasks);
        int4 *dst = reinterpret_cast<int4 *>(tasks);
        const int words = ntask * (int)(sizeof(SweepDev) / sizeof(int4));
        for (int i = tid; i < words; i += blockDim.x) dst[i] = src[i];
    }
    __syncthreads();
    if (abort_sh) return;  // an earlier wait timed out: the host resets the vectors first
    const unsigned int tag0 = tag_sh;
    auto give_up = [&]() {
        if (lane == 0) {
            dead = 1;
            atomicOr(a.flag, 2);
        }
    };

    if (warp == rows + PW) {
        // producer warp: the rows [r0, r0 + nrv) of every block of task q into slot q % nslot
        int q = 0;
        bool fine = true;
        const unsigned int row_bytes = (unsigned int)(ldp * 4);
        for (; q < ntask; q++) {
            const int slot = q % nslot;
            if (q >= nslot) {
                int w = 1;
                if (lane == 0) w = mbar_wait(smem_u32(&empty[slot]), (unsigned int)((q / nslot - 1) & 1), a.spin, &dead);
                w = __shfl_sync(0xffffffffu, w, 0);
                if (!w) {
                    give_up();
                    fine = false;
                    break;
                }
            }
            const int k = tasks[q].head.x, nblk = tasks[q].head.z;
            const unsigned int fb = smem_u32(&full[slot]);
            if (lane == 0) {
                asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
                asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(fb),
                             "r"(row_bytes * (unsigned int)(nblk * nrv))
                             : "memory");
            }
            __syncwarp();
            for (int idx = lane; idx < nblk * nrv; idx += 32) {
                const int p = idx / nrv, j = idx - p * nrv;
                const int m = tasks[q].blk[p].x;
                const float *src = pc + (((size_t)k * nd + (m - k + h)) * nb + r0 + j) * ldp;
                float *dst = ring + (size_t)slot * slot_floats + ((size_t)p * rows + j) * ldp;
                asm volatile(
                    "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
                        smem_u32(dst)),
                    "l"(src), "r"(row_bytes), "r"(fb)
                    : "memory");
            }
        }
        // every copy issued must land before the CTA may end
        if (lane == 0) {
            const int last = fine ? ntask - 1 : q - 1;
            for (int pq = max(0, last - nslot + 1); pq <= last; pq++)
                if (!mbar_wait(smem_u32(&full[pq % nslot]), (unsigned int)((pq / nslot) & 1), a.spin, nullptr)) break;
        }
        return;
    }

    if (warp >= rows) {
        // poll warps: words pt, pt + PT, ... of every vector slice; word w holds row w mod sw
        // of CTA w / sw
        const int pt = tid - 32 * rows;
        int col[WPT], dst[WPT];
        bool cv[WPT];
#pragma unroll
        for (int q = 0; q < WPT; q++) {
            col[q] = pt + q * PT;
            const int c = col[q] / a.sw, j = col[q] - c * a.sw;
            cv[q] = c < Gg && j < base + (c < extra ? 1 : 0);
            dst[q] = c * base + min(c, extra) + j;
        }
        // task s: blocks [e0, e1) are early, block e1 is critical if there is one
        auto early_range = [&](int4 hd, int &e0, int &e1) {
            e0 = (hd.w & 1) + ((hd.w >> 1) & 1);
            e1 = hd.z - ((hd.w >> 2) & 1);
        };
        int4 blk[BM], head = tasks[0].head;  // of the task at hand; its early words, loaded a task ahead
        unsigned long long pre[BM][WPT], wc[WPT];
        auto load = [&](int s) {
            int e0, e1;
            head = tasks[s].head;
#pragma unroll
            for (int p = 0; p < BM; p++) blk[p] = tasks[s].blk[p];
            early_range(head, e0, e1);
#pragma unroll
            for (int p = 0; p < BM; p++)
#pragma unroll
                for (int q = 0; q < WPT; q++)
                    pre[p][q] = (p >= e0 && p < e1 && cv[q]) ? ld_word(a.Y + blk[p].y + col[q]) : 0ull;
        };
        bool ok = true;
        int sl = 0, sl1 = 0;              // ring slots of tasks s - 1 and s - 2
        unsigned int pr = 0u, pr1 = 0u;   // and the parities of their empty barriers
        load(0);
        for (int s = 0; s < ntask; s++) {
            int e0, e1;
            early_range(head, e0, e1);
            float v[WPT];
            // the buffers of task s - 2 are free once every compute warp is done with it
            if (s >= 2) ok = mbar_wait(smem_u32(&empty[sl1]), pr1, a.spin, &dead);
#pragma unroll
            for (int p = 0; p < BM; p++) {
                if (p < e0 || p >= e1 || !ok) continue;
                ok = await_words<WPT>(a.Y + blk[p].y, col, cv, tag0 + (unsigned int)blk[p].z, pre[p], v, a.spin);
                float *e = vbuf + (size_t)(2 + (s & 1) * (h + 1) + p) * ldp;
#pragma unroll
                for (int q = 0; q < WPT; q++)
                    if (cv[q]) e[dst[q]] = v[q];
            }
            __syncwarp();
            if (lane == 0) mbar_arrive(&early[s & 1]);
            const bool has_crit = (head.w & 4) != 0;
            int4 cb = blk[0];
#pragma unroll
            for (int p = 1; p < BM; p++)
                if (p == e1) cb = blk[p];
            if (s + 1 < ntask) load(s + 1);
            // the critical vector is polled from SW_BACKOFF clocks after this CTA finished its
            // own rows of it: polls before that rarely succeed, and CTAs polling the same few
            // lines slow the stores that they wait for (181 x 61, whole apply: 165 us
            // without the pause, 138 us with 400 clocks, 147 us with 800)
            if (has_crit) {
                const unsigned long long *cptr = a.Y + cb.y;
                ok = ok && mbar_wait(smem_u32(&empty[sl]), pr, a.spin, &dead);
                for (const long long c0 = clock64(); clock64() - c0 < SW_BACKOFF;) {}
#pragma unroll
                for (int q = 0; q < WPT; q++) wc[q] = cv[q] ? ld_word(cptr + col[q]) : 0ull;
                if (ok) ok = await_words<WPT>(cptr, col, cv, tag0 + (unsigned int)cb.z, wc, v, a.spin);
                float *e = vbuf + (size_t)(s & 1) * ldp;
#pragma unroll
                for (int q = 0; q < WPT; q++)
                    if (cv[q]) e[dst[q]] = v[q];
            }
            if (!__all_sync(0xffffffffu, ok)) {
                give_up();
                return;
            }
            if (lane == 0) mbar_arrive(&crit[s & 1]);
            sl1 = sl;
            pr1 = pr;
            if (s > 0 && ++sl == nslot) {
                sl = 0;
                pr ^= 1u;
            }
        }
        return;
    }

    // compute warps: row r0 + warp of every slice, columns 4 lane + 128 q
    if (warp >= nrv) return;
    const int row = r0 + warp;
    size_t my_e;  // its index in the order of u (+ k NB for slice k)
    {
        const int g = row / NB, pp = row - g * NB;
        my_e = (size_t)g * NB * a.M + pp;
    }
    bool cq[NQ];
#pragma unroll
    for (int q = 0; q < NQ; q++) cq[q] = 4 * lane + 128 * q < ldp;
    float acc[NQ], alo[NQ];
    // acc += +- S v: four products a partial sum, the partial sums added as pairs,
    // NQ independent chains
    auto dot = [&](const float4 (&f)[NQ], const float4 (&x)[NQ], int plus) {
        const unsigned int neg = plus ? 0u : 0x80000000u;
#pragma unroll
        for (int q = 0; q < NQ; q++) {
            const float u = fmaf(f[q].w, x[q].w, fmaf(f[q].z, x[q].z, fmaf(f[q].y, x[q].y, f[q].x * x[q].x)));
            pair_add(acc[q], alo[q], __uint_as_float(__float_as_uint(u) ^ neg));
        }
    };
    auto fetch = [&](const float *p, float4 (&f)[NQ]) {
#pragma unroll
        for (int q = 0; q < NQ; q++)
            f[q] = cq[q] ? *reinterpret_cast<const float4 *>(p + 4 * lane + 128 * q) : make_float4(0.f, 0.f, 0.f, 0.f);
    };
    float4 w0[NQ], w1[NQ];  // this lane's columns of the last two critical vectors
#pragma unroll
    for (int q = 0; q < NQ; q++) w0[q] = w1[q] = make_float4(0.f, 0.f, 0.f, 0.f);
    int slot = 0;
    unsigned int par = 0;  // of full[slot]
    for (int s = 0; s < ntask; s++) {
        const int4 head = tasks[s].head;
        const int nblk = head.z, win = head.w & 3, plus = head.w >> 4;
        const bool has_crit = (head.w & 4) != 0;
        const float *sp = ring + (size_t)slot * slot_floats + (size_t)warp * ldp;
        const size_t bs = (size_t)rows * ldp;
#pragma unroll
        for (int q = 0; q < NQ; q++) acc[q] = alo[q] = 0.f;
        if (lane == 0) {
            const float2 x = xs[s * rows + warp];
            acc[0] = x.x;
            alo[0] = x.y;
        }
        bool ok = mbar_wait(smem_u32(&full[slot]), par, a.spin, &dead);
        // the row's entries of the blocks in the register window and of the critical one
        const int nw = (win & 1) + (win >> 1);
        float4 f0[NQ], f1[NQ], fc[NQ];
        if (ok) {
            if (win & 1) fetch(sp, f0);
            if (win & 2) fetch(sp + (win & 1) * bs, f1);
            if (has_crit) fetch(sp + (nblk - 1) * bs, fc);
            if (win & 1) dot(f0, w0, plus & 1);
            if (win & 2) dot(f1, w1, (plus >> (win & 1)) & 1);
            const int nfree = nblk - (has_crit ? 1 : 0);
            if (nw < nfree) {
                ok = mbar_wait(smem_u32(&early[s & 1]), (unsigned int)((s >> 1) & 1), a.spin, &dead);
#pragma unroll 1
                for (int p = nw; p < nfree && ok; p++) {
                    fetch(sp + p * bs, f0);
                    fetch(vbuf + (size_t)(2 + (s & 1) * (h + 1) + p) * ldp, f1);
                    dot(f0, f1, (plus >> p) & 1);
                }
            }
        }
        // the critical term last: the vector the group's previous task wrote
        ok = ok && mbar_wait(smem_u32(&crit[s & 1]), (unsigned int)((s >> 1) & 1), a.spin, &dead);
        if (!__all_sync(0xffffffffu, ok)) {
            give_up();
            return;
        }
        if (has_crit) {
#pragma unroll
            for (int q = 0; q < NQ; q++) w1[q] = w0[q];
            fetch(vbuf + (size_t)(s & 1) * ldp, w0);
            dot(fc, w0, (plus >> (nblk - 1)) & 1);
        }
#pragma unroll
        for (int q = 1; q < NQ; q++) {
            pair_add(acc[0], alo[0], acc[q]);
            alo[0] += alo[q];
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            const float oh = __shfl_down_sync(0xffffffffu, acc[0], o), ol = __shfl_down_sync(0xffffffffu, alo[0], o);
            pair_add(acc[0], alo[0], oh);
            alo[0] += ol;
        }
        // the CTA's rows go out in one store of its last warp: lines that many CTAs are
        // about to poll are written once per CTA, not once per row.  A task without a
        // critical block waits for task s - 2 only, so one warp may be done with task s + 1
        // while another is still in task s: even and odd tasks have a counter each
        int last = 0;
        if (lane == 0) {
            outv[s & 3][warp] = acc[0] + alo[0];
            __threadfence_block();
            last = atomicAdd(&ndone[s & 1], 1) == nrv * ((s >> 1) + 1) - 1;
            mbar_arrive(&empty[slot]);  // every lane's reads of the slot came before the shuffles
        }
        if (__shfl_sync(0xffffffffu, last, 0)) {
            __threadfence_block();
            if (lane < nrv) {
                const unsigned int tg = tag0 + (unsigned int)((grp ? a.ntask0 : 0) + s);
                st_word((head.y ? a.X : a.Y) + (size_t)head.x * a.vs + lb * a.sw + lane,
                        reinterpret_cast<volatile float *>(outv[s & 3])[lane], tg);
            }
        }
        if (lane == 0 && head.y) {
            const size_t e = my_e + (size_t)head.x * NB;
            if (a.zpair) reinterpret_cast<float2 *>(a.z)[e] = make_float2(acc[0], alo[0]);
            else a.z[e] = (double)acc[0] + (double)alo[0];
        }
        if (++slot == nslot) {
            slot = 0;
            par ^= 1u;
        }
    }
    if (blockIdx.x == 0 && tid == 0) advance_tag(a.tagp, tag0, (unsigned int)a.ntags);
}

constexpr int SW_MAXSLOT = 6;
constexpr size_t SW_SMEM_MAX = 220 * 1024;

// ---------------------------------------------------------------------------
// Host: the task table.  Tasks of group 0 come first; the task with index s
// in group g has uid s (g = 0) or ntask0 + s (g = 1), and writes its slice
// with tag tag0 + uid.
// ---------------------------------------------------------------------------
int sweep_plan(int M, int h, int twisted, SweepPlan &P)
{
    P = SweepPlan();
    if (M < 1 || h < 0 || h + 1 > SW_BMAX) return BFS_EINVAL;
    const bool two = twisted && h >= 1 && M - h >= 2;
    std::vector<SweepTask> G[2];
    auto task = [](int k, int out) {
        SweepTask t;
        memset(&t, 0, sizeof t);
        t.k = k;
        t.out = out;
        return t;
    };
    auto blk = [](SweepTask &t, int m, int x, int plus) {
        t.m[t.nblk] = m;
        t.vec[t.nblk] = x | (plus << 1);
        t.nblk++;
    };
    if (!two) {
        for (int k = 0; k < M; k++) {  // forward: y_k = x_k - L_ki y_i
            SweepTask t = task(k, 0);
            for (int i = std::max(0, k - h); i < k; i++) blk(t, i, 0, 0);
            G[0].push_back(t);
        }
        for (int k = M - 1; k >= 0; k--) {  // backward: z_k = D_k^-1 y_k - W_kj z_j
            SweepTask t = task(k, 1);
            blk(t, k, 0, 1);
            for (int j = k + 1; j <= std::min(M - 1, k + h); j++) blk(t, j, 1, 0);
            G[0].push_back(t);
        }
    } else {
        const int t0 = (M - h) / 2, t1 = t0 + h;  // middle slices [t0, t1)
        for (int k = 0; k < t0; k++) {  // top chain, forward
            SweepTask t = task(k, 0);
            for (int i = std::max(0, k - h); i < k; i++) blk(t, i, 0, 0);
            G[0].push_back(t);
        }
        for (int k = M - 1; k >= t1; k--) {  // bottom chain, upward: y_k = x_k - U'_kj y_j
            SweepTask t = task(k, 0);
            for (int j = k + 1; j <= std::min(M - 1, k + h); j++) blk(t, j, 0, 0);
            G[1].push_back(t);
        }
        for (int g = 0; g < 2; g++)  // middle y: both chains' terms (the groups alternate slices)
            for (int m = t0 + g; m < t1; m += 2) {
                SweepTask t = task(m, 0);
                for (int i = std::max(0, m - h); i < t0; i++) blk(t, i, 0, 0);
                for (int j = t1; j <= std::min(M - 1, m + h); j++) blk(t, j, 0, 0);
                G[g].push_back(t);
            }
        for (int g = 0; g < 2; g++)  // middle z = C^-1 y_mid
            for (int m = t0 + g; m < t1; m += 2) {
                SweepTask t = task(m, 1);
                for (int q = t0; q < t1; q++) blk(t, q, 0, 1);
                G[g].push_back(t);
            }
        for (int k = t0 - 1; k >= 0; k--) {  // top chain, backward
            SweepTask t = task(k, 1);
            blk(t, k, 0, 1);
            for (int j = k + 1; j <= std::min(M - 1, k + h); j++) blk(t, j, 1, 0);
            G[0].push_back(t);
        }
        for (int k = t1; k < M; k++) {  // bottom chain, downward: z_k = D_k^-1 y_k - W'_kj z_j
            SweepTask t = task(k, 1);
            blk(t, k, 0, 1);
            for (int j = std::max(0, k - h); j < k; j++) blk(t, j, 1, 0);
            G[1].push_back(t);
        }
        P.twist = t0;
        P.groups = 2;
    }
    P.ntask[0] = (int)G[0].size();
    P.ntask[1] = (int)G[1].size();
    std::vector<int> prodY(M, -1), prodX(M, -1);
    for (int g = 0; g < 2; g++)
        for (int s = 0; s < P.ntask[g]; s++) {
            int &pr = (G[g][s].out ? prodX : prodY)[G[g][s].k];
            if (pr >= 0) return BFS_EINVAL;  // every vector slice has one writer
            pr = (g ? P.ntask[0] : 0) + s;
        }
    for (int g = 0; g < 2; g++)
        for (int s = 0; s < P.ntask[g]; s++) {
            SweepTask &t = G[g][s];
            const int prev = s > 0 ? (g ? P.ntask[0] : 0) + s - 1 : -1;
            int last = -1;
            for (int p = 0; p < t.nblk; p++) {
                const int u = ((t.vec[p] & 1) ? prodX : prodY)[t.m[p]];
                if (u < 0) return BFS_EINVAL;
                t.uid[p] = u;
                if (u == prev) last = p;
            }
            if (last >= 0 && last != t.nblk - 1) {  // the freshest vector last
                std::swap(t.m[last], t.m[t.nblk - 1]);
                std::swap(t.vec[last], t.vec[t.nblk - 1]);
                std::swap(t.uid[last], t.uid[t.nblk - 1]);
            }
        }
    // where each thread finds its columns of a block's vector: the group's
    // previous task wrote it (SW_CRIT: polled last); one of the last SW_HW
    // critical vectors the thread holds in registers (SW_WIN, with its index);
    // otherwise loaded at the end of the step before (SW_EARLY)
    for (int g = 0; g < 2; g++) {
        std::vector<int> win;  // uids of the vectors in the register window, newest first
        for (int s = 0; s < P.ntask[g]; s++) {
            SweepTask &t = G[g][s];
            const int prev = s > 0 ? (g ? P.ntask[0] : 0) + s - 1 : -1;
            int crit = -1;
            for (int p = 0; p < t.nblk; p++) {
                int src = SW_EARLY, wi = 0;
                if (t.uid[p] == prev) {
                    src = SW_CRIT;
                    crit = t.uid[p];
                } else {
                    for (int i = 0; i < (int)win.size(); i++)
                        if (win[i] == t.uid[p]) { src = SW_WIN; wi = i; }
                }
                t.vec[p] = (t.vec[p] & 3) | (src << 2) | (wi << 4);
            }
            if (crit >= 0) {
                win.insert(win.begin(), crit);
                if ((int)win.size() > SW_HW) win.pop_back();
            }
        }
    }
    P.tasks = G[0];
    P.tasks.insert(P.tasks.end(), G[1].begin(), G[1].end());
    return BFS_OK;
}

// The table as the kernel reads it (SweepDev); vs words a slice, nv words of y, which x
// follows.
static std::vector<SweepDev> device_table(const SweepPlan &P, int vs, size_t nv)
{
    std::vector<SweepDev> out;
    for (const SweepTask &t : P.tasks) {
        SweepDev d;
        memset(&d, 0, sizeof d);
        int n = 0, order = 0;
        auto src = [&](int p) { return (t.vec[p] >> 2) & 3; };
        auto take = [&](int p) {
            d.blk[n] = make_int4(t.m[p], (int)((t.vec[p] & 1) * nv) + t.m[p] * vs, t.uid[p], 0);
            order |= ((t.vec[p] >> 1) & 1) << (4 + n);
            n++;
        };
        for (int wi = 0; wi < SW_HW; wi++)
            for (int p = 0; p < t.nblk; p++)
                if (src(p) == SW_WIN && ((t.vec[p] >> 4) & 3) == wi) {
                    take(p);
                    order |= 1 << wi;
                }
        for (int p = 0; p < t.nblk; p++)
            if (src(p) == SW_EARLY) take(p);
        for (int p = 0; p < t.nblk; p++)
            if (src(p) == SW_CRIT) {
                take(p);
                order |= 4;
            }
        d.head = make_int4(t.k, t.out, t.nblk, order);
        out.push_back(d);
    }
    return out;
}

using FlowKernel = void (*)(FlowArgs);

// Instances of the task-table kernel by words of a vector slice per poll thread,
// columns of a lane (4 in every 128) and blocks per task.
constexpr int SW_PW = 5;
template <int WPT>
static FlowKernel pick_sweep_w(int nq, int bm)
{
    if (nq == 3) return bm == 4 ? k_apply_sweep<SW_PW, WPT, 3, 4> : k_apply_sweep<SW_PW, WPT, 3, SW_BMAX>;
    return bm == 4 ? k_apply_sweep<SW_PW, WPT, 5, 4> : k_apply_sweep<SW_PW, WPT, 5, SW_BMAX>;
}
static FlowKernel pick_sweep(int wpt, int nq, int bm)
{
    return wpt == 2 ? pick_sweep_w<2>(nq, bm) : pick_sweep_w<4>(nq, bm);
}

template <bool PAIR>
static FlowKernel pick_flow(int rpc, int cpt)
{
    if (rpc <= 4 && cpt <= 2) return k_apply_flow<4, 2, PAIR>;
    if (rpc <= 8 && cpt <= 2) return k_apply_flow<8, 2, PAIR>;
    if (rpc <= 8 && cpt <= 3) return k_apply_flow<8, 3, PAIR>;
    return nullptr;
}

// Shape of the task-table kernel for nb-wide slice blocks, half band h,
// `groups` CTA groups on G SMs and at most ntask tasks per group (staged in
// shared memory after the ring and the vectors); false if its tiles do not take them.
struct SweepShape {
    int Gg, rows, sw, wpt, nq, bm, nslot;
    size_t dyn;
    int tpb() const { return 32 * (rows + SW_PW + 1); }
};

static bool sweep_shape(int nb, int h, int groups, int G, int ntask, SweepShape &S)
{
    const int ldp = (nb + 3) / 4 * 4;
    // CTAs of a group: every one has a row at least, since a barrier of the kernel cannot
    // be set up for no arrivals and only a CTA with rows is waited for by the others
    S.Gg = std::min(G / groups, nb);
    S.bm = h + 1 <= 4 ? 4 : SW_BMAX;
    S.nq = ldp <= 384 ? 3 : 5;
    if (nb > 128 * S.nq || h + 1 > S.bm || S.Gg < 1) return false;
    S.rows = (nb + S.Gg - 1) / S.Gg;
    if (S.rows > SW_ROWS) return false;
    S.sw = S.rows <= 4 ? 4 : 8;  // 32- or 64-byte segment of a slice per CTA
    S.wpt = (S.sw * S.Gg + 32 * SW_PW - 1) / (32 * SW_PW) <= 2 ? 2 : 4;
    if (S.sw * S.Gg > 32 * SW_PW * S.wpt) return false;
    const size_t slot = (size_t)(h + 1) * S.rows * ldp * sizeof(float);
    const size_t rest = (size_t)(2 + 2 * (h + 1)) * ldp * sizeof(float) +
                        (size_t)ntask * (sizeof(SweepDev) + S.rows * sizeof(float2));
    if (rest + 2 * slot > SW_SMEM_MAX) return false;
    S.nslot = (int)std::min<size_t>(SW_MAXSLOT, (SW_SMEM_MAX - rest) / slot);
    S.dyn = slot * S.nslot + rest;
    return true;
}

// 1 if the FP32 sweeps of this context can run the two-chain (twisted)
// schedule for half band h, so that the factorisation should take that order.
int sweep_twist_ok(bfs_ctx *c, int h)
{
    if (c->opt.precond_precision != BFS_FP32C || c->opt.surface_tension != 0.0) return 0;
    if (h < 1 || c->M - h < 2) return 0;
    SweepPlan P;
    if (sweep_plan(c->M, h, 1, P) != BFS_OK || P.groups != 2) return 0;
    SweepShape S;
    if (!sweep_shape(c->nb, h, 2, num_sms(c->device), std::max(P.ntask[0], P.ntask[1]), S)) return 0;
    const FlowKernel kern = pick_sweep(S.wpt, S.nq, S.bm);
    BFS_CUDA_TRY(c, cudaFuncSetAttribute((const void *)kern, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         (int)SW_SMEM_MAX));
    int per_sm = 0;
    BFS_CUDA_TRY(c, cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, S.tpb(), S.dyn));
    return per_sm >= 1 ? 1 : 0;
}

// FP32 copy of the factors with rows padded from nb to ldp entries (zeros),
// so that every row starts on a 16-byte boundary.
__global__ void k_cast_f32(const double *__restrict__ in, float *__restrict__ out, size_t rows, int nb, int ldp)
{
    const size_t n = rows * (size_t)ldp;
    for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x) {
        const size_t r = i / ldp;
        const int c = (int)(i - r * ldp);
        out[i] = c < nb ? (float)in[r * nb + c] : 0.f;
    }
}

__global__ void k_set_tag(unsigned int *p, unsigned int v) { *p = v; }

// Zero the tagged vectors and restart the tags at 1 (so no stale entry can
// carry a tag a later launch waits for).
int flow_reset(bfs_ctx *c, cudaStream_t s)
{
    if (!c->d_flow) return BFS_OK;
    const size_t nv = (size_t)c->M * c->flow_vs;
    BFS_CUDA_TRY(c, cudaMemsetAsync(c->d_flow, 0, sizeof(unsigned long long) * (2 * nv + 1), s));
    k_set_tag<<<1, 1, 0, s>>>(reinterpret_cast<unsigned int *>(c->d_flow + 2 * nv), 1u);
    c->launches++;
    c->flow_count = 0;
    BFS_CUDA_TRY(c, cudaGetLastError());
    return BFS_OK;
}

// Before each FP32 sweep launch (direct or inside a graph): restart the tags
// well before they could wrap.
int flow_wrap_check(bfs_ctx *c, cudaStream_t s)
{
    const unsigned long long steps = (unsigned long long)std::max(c->sweep_ntags, 2 * c->M);
    if ((c->flow_count + 2) * steps >= 0xFFFFFFFFull - 0xFFFFull) return flow_reset(c, s);
    return BFS_OK;
}

int precond_make_f32(bfs_ctx *c, cudaStream_t s)
{
    const int ldp = (c->nb + 3) / 4 * 4;
    const size_t rows = (size_t)c->nb * c->M * (2 * c->pc_h + 1);
    const size_t cnt = rows * ldp;
    c->ldp32 = ldp;
    cudaFree(c->d_pc32);
    cudaFree(c->d_flow);
    cudaFree(c->d_tasks);
    c->d_pc32 = nullptr;
    c->d_flow = nullptr;
    c->d_tasks = nullptr;
    c->sweep_table = 0;
    // the task table: two chains if the factors are in the two-ended order
    const int twisted = c->pc_twist >= 0;
    SweepShape S;
    c->sweep_ntags = 2 * c->M;
    SweepPlan P;
    const bool planned = sweep_plan(c->M, c->pc_h, twisted, P) == BFS_OK;  // h < SW_BMAX only
    if (twisted && (!planned || P.twist != c->pc_twist)) {
        c->err = "sweep schedule does not match the factor order";
        return BFS_EINVAL;
    }
    const bool table = planned && sweep_shape(c->nb, c->pc_h, twisted ? 2 : 1, num_sms(c->device),
                                              std::max(P.ntask[0], P.ntask[1]), S);
    if (twisted && !table) {
        c->err = "two-ended factors need the task-table sweep kernel";
        return BFS_EINVAL;
    }
    // words of a vector slice: a segment per CTA for the task-table kernel
    c->flow_vs = table ? S.sw * S.Gg : c->nb;
    const size_t nv = (size_t)c->M * c->flow_vs;
    if (cudaMalloc(&c->d_pc32, sizeof(float) * cnt) != cudaSuccess ||
        cudaMalloc(&c->d_flow, sizeof(unsigned long long) * (2 * nv + 1)) != cudaSuccess) {
        cudaGetLastError();
        c->err = "FP32 preconditioner copy: out of device memory";
        return BFS_ENOMEM;
    }
    if (table) {
        c->h_tasks = device_table(P, c->flow_vs, nv);
        BFS_ALLOC_TRY(c, cudaMalloc(&c->d_tasks, sizeof(SweepDev) * c->h_tasks.size()));
        BFS_CUDA_TRY(c, cudaMemcpy(c->d_tasks, c->h_tasks.data(), sizeof(SweepDev) * c->h_tasks.size(),
                                   cudaMemcpyHostToDevice));
        c->sweep_table = 1;
        c->sweep_groups = P.groups;
        c->sweep_ntask[0] = P.ntask[0];
        c->sweep_ntask[1] = P.ntask[1];
        c->sweep_ntags = P.ntask[0] + P.ntask[1];
        c->sweep_wpt = S.wpt;
        c->sweep_nq = S.nq;
        c->sweep_gg = S.Gg;
        c->sweep_sw = S.sw;
        c->sweep_rows = S.rows;
        c->sweep_bm = S.bm;
        c->sweep_nslot = S.nslot;
        c->sweep_dyn = S.dyn;
    }
    int rc = flow_reset(c, s);
    if (rc) return rc;
    k_cast_f32<<<4 * num_sms(c->device), 256, 0, s>>>(c->d_pc, c->d_pc32, rows, c->nb, ldp);
    c->launches++;
    BFS_CUDA_TRY(c, cudaGetLastError());
    return BFS_OK;
}

static unsigned int spin_limit(const bfs_ctx *c)
{
    return c->opt.wait_polls > 0 ? (unsigned int)c->opt.wait_polls : FL_SPIN;
}

// Returns 1 if launched, 2 if launched with z written as float pairs, 0 if this apply is
// not for the FP32 sweep kernels (FP64 sweeps, or slice blocks wider than their tiles),
// or a negative code.
int apply_flow_launch(bfs_ctx *c, const double *r, double *z, cudaStream_t s)
{
    if (c->opt.precond_precision != BFS_FP32C || !c->d_pc32 || !c->d_flow) return 0;
    const int G = num_sms(c->device);
    FlowArgs a;
    a.pc = c->d_pc32;
    a.r = r; a.z = z;
    a.Y = c->d_flow;
    a.X = c->d_flow + (size_t)c->M * c->flow_vs;
    // condensed blocks: right-hand side and result slice by slice, one field of nb
    a.nb = c->nb; a.NB = c->pc_cond ? c->nb : c->N + 1; a.M = c->M; a.h = c->pc_h;
    a.ldp = c->ldp32;
    a.tagp = reinterpret_cast<unsigned int *>(c->d_flow + 2 * (size_t)c->M * c->flow_vs);
    a.flag = c->d_flag;
    a.spin = spin_limit(c);
    a.tasks = c->d_tasks;
    a.ntask0 = c->sweep_ntask[0];
    a.ntask1 = c->sweep_ntask[1];
    a.G0 = c->sweep_table ? c->sweep_gg : G;
    a.sw = c->sweep_sw;
    a.vs = c->flow_vs;
    a.ntags = c->sweep_ntags;
    a.nslot = c->sweep_nslot;
    a.rows = c->sweep_rows;
    a.zpair = c->sweep_table && c->pc_cond;
    FlowKernel kern;
    int tpb;
    size_t dyn = 0;
    if (c->sweep_table) {
        kern = pick_sweep(c->sweep_wpt, c->sweep_nq, c->sweep_bm);
        tpb = 32 * (c->sweep_rows + SW_PW + 1);
        dyn = c->sweep_dyn;
    } else {
        const int rpc = (c->nb + G - 1) / G, cpt = (c->nb + FL_TPB - 1) / FL_TPB;
        kern = c->pc_cond ? pick_flow<true>(rpc, cpt) : pick_flow<false>(rpc, cpt);
        tpb = FL_TPB;
        if (!kern) return 0;
    }
    if (!c->flow_checked) {
        if (c->sweep_table)  // one ceiling for every context, whatever its ring depth
            BFS_CUDA_TRY(c, cudaFuncSetAttribute((const void *)kern, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                                 (int)SW_SMEM_MAX));
        int per_sm = 0;
        BFS_CUDA_TRY(c, cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, tpb, dyn));
        if (per_sm < 1) {
            if (c->pc_twist >= 0) {
                c->err = "the two-chain sweep kernel cannot be resident";
                return BFS_ECUDA;
            }
            return 0;
        }
        c->flow_checked = 1;
    }
    if (!c->capturing) {
        int rc = flow_wrap_check(c, s);
        if (rc) return rc;
    }
    // test hook: one wait of this launch is for a vector no task writes
    const bool stall = c->sweep_table && c->dbg_stall_task >= 0 && !c->capturing && c->dbg_stall_skip-- == 0;
    if (stall) {
        std::vector<SweepDev> bad = c->h_tasks;
        SweepDev &t = bad[c->dbg_stall_task];
        // the last block's vector: polled for, not one held since an earlier task
        if (t.head.z > 0) t.blk[t.head.z - 1].z = c->sweep_ntags;  // the tag of the next launch's first task
        BFS_CUDA_TRY(c, cudaMemcpyAsync(c->d_tasks, bad.data(), sizeof(SweepDev) * bad.size(),
                                        cudaMemcpyHostToDevice, s));
        BFS_CUDA_TRY(c, cudaStreamSynchronize(s));
    }
    void *args[] = {&a};
    const int grid = c->sweep_table ? c->sweep_gg * c->sweep_groups : G;
    cudaError_t e = cudaLaunchCooperativeKernel((const void *)kern, dim3(grid), dim3(tpb), args, dyn, s);
    if (stall) {
        c->dbg_stall_task = -1;
        BFS_CUDA_TRY(c, cudaMemcpyAsync(c->d_tasks, c->h_tasks.data(), sizeof(SweepDev) * c->h_tasks.size(),
                                        cudaMemcpyHostToDevice, s));
        BFS_CUDA_TRY(c, cudaStreamSynchronize(s));
    }
    BFS_CUDA_TRY(c, e);
    c->launches++;
    c->flow_count++;
    return a.zpair ? 2 : 1;
}

}  // namespace bfs

extern "C" {

int bfs_sweep_schedule(int M, int half_band, int twisted, int *tasks_out, int cap, int *ntask_out)
{
    bfs::SweepPlan P;
    if (half_band > 3 || bfs::sweep_plan(M, half_band, twisted, P) != BFS_OK) return BFS_EINVAL;
    if (ntask_out) {
        ntask_out[0] = P.ntask[0];
        ntask_out[1] = P.ntask[1];
    }
    const int n = (int)P.tasks.size();
    if (tasks_out) {
        if (cap < n) return BFS_EINVAL;
        for (int i = 0; i < n; i++) {  // 16 ints a task: at most 4 blocks for half_band <= 3
            const bfs::SweepTask &t = P.tasks[i];
            int *o = tasks_out + 16 * i;
            const int head[4] = {t.k, t.out, t.nblk, 0};
            memcpy(o, head, sizeof head);
            memcpy(o + 4, t.m, 4 * sizeof(int));
            memcpy(o + 8, t.vec, 4 * sizeof(int));
            memcpy(o + 12, t.uid, 4 * sizeof(int));
        }
    }
    return n;
}

int bfs_debug_stall_sweep(bfs_ctx *c, int task) { return bfs_debug_stall_later(c, task, 0); }

int bfs_debug_stall_later(bfs_ctx *c, int task, int skip)
{
    if (!c) return BFS_EINVAL;
    if (!c->pc_ready || !c->sweep_table) {
        c->err = "the stall hook needs the FP32 task-table sweeps";
        return BFS_EINVAL;
    }
    if (skip < 0 || task < 0 || task >= (int)c->h_tasks.size() || c->h_tasks[task].head.z == 0) {
        c->err = "no waiting block in that task";
        return BFS_EINVAL;
    }
    c->dbg_stall_task = task;
    c->dbg_stall_skip = skip;
    return BFS_OK;
}

}  // extern "C"

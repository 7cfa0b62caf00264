// solve.cu -- the persistent PCG solver (FP64, and mixed FP32/FP64 by reliable
// updates or restarted refinement), the level-scheduled DIC factor and sweeps,
// the prepared-matrix Amul, and their host entry points.
//
// One cooperative launch per solve.  Rows live in the handle's level order:
// level L (rows whose longest chain of lower neighbours has length L) is the
// contiguous range lvl[L]..lvl[L+1], and every row keeps its neighbour-side
// ("lower") and owner-side ("upper") entries in ascending face order, so each
// row sum is taken in exactly the order of the sequential face loop.
//
// One PCG iteration with DIC (grid barriers after each step, and after each
// DIC level inside the sweeps):
//   update pass       x += alpha p, r -= alpha q, sum|r|       -> converged?
//   forward sweep     w = (P + L)^-1 r, level by level
//   backward sweep    w = (P + U)^-1 P w, rho = w.r            -> beta
//   search direction  p = w + beta p
//   Amul              q = A p, sigma = q.p                     -> alpha
#include <algorithm>
#include <cmath>
#include <cstdlib>
#include <map>
#include <mutex>

#include "solve.cuh"

namespace spuma {

// Slots of the block partials.  A slot may be written again only after a grid
// barrier that follows its last read: a block may still be reading when a
// faster one goes on.  What follows a read without a barrier in between has
// slots of its own: the initial sums, after which the loops' first sums (SL_A,
// SL_B; SL_D and SL_DMAX in the restarted form) or the true residual of a system
// that starts converged come at once, and the true residual, which follows the
// sums that stopped the loop.
enum Slot { SL_A = 0, SL_B = 1, SL_D = 2, SL_DMAX = 3, SL_C = 4, SL_INIT = SL_C, SL_TRUE = 6 };
static_assert(SL_TRUE + 2 <= kSlots, "two partial sums of the true residual");

__device__ __forceinline__ bool converged(double res, double res0, double tol, double rel_tol)
{
    return res < tol || (rel_tol > 0.0 && res < rel_tol * res0);
}

template <class T>
__device__ __forceinline__ Mat<T> mat_of(const SolveArgs& a);
template <>
__device__ __forceinline__ Mat<double> mat_of<double>(const SolveArgs& a)
{
    return Mat<double>{a.Lptr, a.Lcol, a.La64, a.Lc64, a.Uptr, a.Ucol, a.Ua64, a.Uc64, a.d64, a.rD64,
                       a.Ecol, a.Ea64, a.ell_w, a.n};
}
template <>
__device__ __forceinline__ Mat<float> mat_of<float>(const SolveArgs& a)
{
    return Mat<float>{a.Lptr, a.Lcol, a.La32, a.Lc32, a.Uptr, a.Ucol, a.Ua32, a.Uc32, a.d32, a.rD32,
                      a.Ecol, a.Ea32, a.ell_w, a.n};
}

// Cache priorities.  The matrix streams (entries, row extents, diagonal,
// rD) are read once per pass: they are loaded evict-first (__ldcs), so that
// the vectors other rows gather stay in L2; a stand-alone Amul stores its
// result evict-first too.  Inside the solver, FP32 gathers (x in the Amul, w
// in the sweeps) are loaded evict-last on top of that, and the solver hands
// those lines back (evict-normal) before it returns; FP64 vectors, twice the
// size, keep the default priority, since pinning them evicts them from each
// other; the pipelined Amul rows gather at the default priority too.  Measured
// at 200^3: stand-alone Amul FP64 168 -> 130 us, FP32 101 -> 91 us; mixed solve
// 352 -> 333 ms with evict-first streams, 330 ms with the FP32 gathers evict-last
// (FP64 gathers evict-last: Amul 130 -> 146 us).
template <class T, bool KEEP>
__device__ __forceinline__ unsigned long long keep_policy()
{
    unsigned long long p = 0;
    if constexpr (KEEP && sizeof(T) == 4)
        asm volatile("createpolicy.fractional.L2::evict_last.b64 %0, 1.0;" : "=l"(p));
    return p;
}
template <bool KEEP>
__device__ __forceinline__ float gather(const float* v, int c, unsigned long long pol)
{
    if constexpr (KEEP) {
        float r;
        asm volatile("ld.global.L2::cache_hint.f32 %0, [%1], %2;" : "=f"(r) : "l"(v + c), "l"(pol) : "memory");
        return r;
    } else {
        return v[c];
    }
}
template <bool KEEP>
__device__ __forceinline__ double gather(const double* v, int c, unsigned long long)
{
    return v[c];
}

// Back to evict-normal: every 128-byte line of [base, base + bytes), spread
// over the group's threads (a hint; the regions are 256-byte aligned).
__device__ __forceinline__ void release_lines(const void* base, size_t bytes, int first, int stride)
{
    const char* b = static_cast<const char*>(base);
    for (size_t off = (size_t)first * 128; off < bytes; off += (size_t)stride * 128)
        asm volatile("applypriority.global.L2::evict_normal [%0], 128;" : : "l"(b + off) : "memory");
}

// Shapes of the row chains: a row's entries are taken in groups whose column
// and coefficient loads are issued together, then the gathers, then the FMAs
// in entry order (two memory round trips per group, not per entry).  FP64 rows
// run one per thread, FP32 rows two per thread in lockstep.  Groups of 6 in
// the DIC sweeps (a hex-mesh row has at most 6 entries on either side) and in
// the Amul, which takes a row's lower and upper entries as one list (a whole
// hex-mesh row in one group).  Chosen by measurement on the 200^3 workload.
template <class T>
struct ChainShape {
    static constexpr int R = sizeof(T) == 4 ? 2 : 1;
    static constexpr int G = 6;
};
// Software-pipelined fixed-width Amul: R rows per round, whole rows of up to
// G entries.  Where it is used was decided by measurement at 200^3: inside
// the persistent solver for FP64 (219 -> 200 us per Amul) and, in the kernels of
// up to 512 threads, two rows a round in both precisions (a mixed iteration with
// the diagonal, FP32 pipelined against its two rows in lockstep: 200^3 164 | 192
// us, 128^3 49 | 57, 64^3 20 | 20); with 1024 threads FP32 keeps the lockstep rows
// (112 against 131 us per Amul); in the stand-alone prepared Amul for FP32 (107 ->
// 101 us; FP64 168 against 176 us).
template <class T>
struct PipeShape {
    static constexpr int R = 1;
    static constexpr int G = 6;
    static constexpr bool in_solver = sizeof(T) == 8;
    static constexpr bool stand_alone = sizeof(T) == 4;
};
template <class T>
struct AmulShape {
    static constexpr int R = sizeof(T) == 4 ? 2 : 1;
    static constexpr int G = 6;
};

// R rows' chains in lockstep; each row takes its entries [e0, e1) in its own
// order (DESC: from e1-1 down to e0).
template <class T, int R, int G, bool DESC, bool NEG>
__device__ __forceinline__ void rows_chain(T (&acc)[R], const int (&e0)[R], const int (&e1)[R], const int* col,
                                           const T* coef, const T* vec)
{
    const unsigned long long pol = keep_policy<T, true>();
    for (int off = 0;; off += G) {
        bool more = false;
#pragma unroll
        for (int k = 0; k < R; k++) more |= e0[k] + off < e1[k];
        if (!more) break;
        int c[R][G];
        T cf[R][G], v[R][G];
#pragma unroll
        for (int k = 0; k < R; k++)
#pragma unroll
            for (int j = 0; j < G; j++) {
                const int ej = DESC ? e1[k] - 1 - off - j : e0[k] + off + j;
                const bool ok = DESC ? ej >= e0[k] : ej < e1[k];
                c[k][j] = ok ? __ldcs(col + ej) : -1;
                cf[k][j] = ok ? __ldcs(coef + ej) : T(0);
            }
#pragma unroll
        for (int k = 0; k < R; k++)
#pragma unroll
            for (int j = 0; j < G; j++) v[k][j] = c[k][j] >= 0 ? gather<true>(vec, c[k][j], pol) : T(0);
#pragma unroll
        for (int k = 0; k < R; k++)
#pragma unroll
            for (int j = 0; j < G; j++)
                if (c[k][j] >= 0) acc[k] = fmadd(NEG ? -cf[k][j] : cf[k][j], v[k][j], acc[k]);
    }
}

// y = A x for R rows: d_p x_p, then the row's lower entries (ascending face)
// and upper entries (ascending face) taken as one list of nL + nU entries.
// KEEP: gathers of x evict-last (inside the solver, FP32).
template <class T, int R, int G, bool KEEP = true>
__device__ __forceinline__ void amul_rows(const Mat<T>& A, const T* x, const int (&p)[R], int n, T (&y)[R],
                                          T (&xp)[R])
{
    if (A.ell_w > 0) {
        // fixed-width layout: no row extents to load, entries coalesced
        const unsigned long long pol = keep_policy<T, KEEP>();
#pragma unroll
        for (int k = 0; k < R; k++) {
            const bool ok = p[k] < n;
            xp[k] = ok ? x[p[k]] : T(0);
            y[k] = ok ? mul_rn(__ldcs(A.d + p[k]), xp[k]) : T(0);
        }
        for (int j0 = 0; j0 < A.ell_w; j0 += G) {
            int c[R][G];
            T cf[R][G], vv[R][G];
#pragma unroll
            for (int k = 0; k < R; k++)
#pragma unroll
                for (int j = 0; j < G; j++) {
                    const bool ok = p[k] < n && j0 + j < A.ell_w;
                    const size_t e = (size_t)(j0 + j) * A.ell_stride + p[k];
                    c[k][j] = ok ? __ldcs(A.Ecol + e) : -1;
                    cf[k][j] = ok ? __ldcs(A.Ea + e) : T(0);
                }
#pragma unroll
            for (int k = 0; k < R; k++)
#pragma unroll
                for (int j = 0; j < G; j++) vv[k][j] = c[k][j] >= 0 ? gather<KEEP>(x, c[k][j], pol) : T(0);
#pragma unroll
            for (int k = 0; k < R; k++)
#pragma unroll
                for (int j = 0; j < G; j++)
                    if (c[k][j] >= 0) y[k] = fmadd(cf[k][j], vv[k][j], y[k]);
        }
        return;
    }
    const unsigned long long pol = keep_policy<T, KEEP>();
    int l0[R], nl[R], u0[R], nt[R];
#pragma unroll
    for (int k = 0; k < R; k++) {
        const bool ok = p[k] < n;
        l0[k] = ok ? __ldcs(A.Lptr + p[k]) : 0;
        nl[k] = ok ? __ldcs(A.Lptr + p[k] + 1) - l0[k] : 0;
        u0[k] = ok ? __ldcs(A.Uptr + p[k]) : 0;
        nt[k] = ok ? nl[k] + __ldcs(A.Uptr + p[k] + 1) - u0[k] : 0;
        xp[k] = ok ? x[p[k]] : T(0);
        y[k] = ok ? mul_rn(__ldcs(A.d + p[k]), xp[k]) : T(0);
    }
    for (int off = 0;; off += G) {
        bool more = false;
#pragma unroll
        for (int k = 0; k < R; k++) more |= off < nt[k];
        if (!more) break;
        int c[R][G];
        T cf[R][G], vv[R][G];
#pragma unroll
        for (int k = 0; k < R; k++)
#pragma unroll
            for (int j = 0; j < G; j++) {
                const int kk = off + j;
                const bool low = kk < nl[k];
                const int e = low ? l0[k] + kk : u0[k] + (kk - nl[k]);
                const bool ok = kk < nt[k];
                c[k][j] = ok ? __ldcs((low ? A.Lcol : A.Ucol) + e) : -1;
                cf[k][j] = ok ? __ldcs((low ? A.La : A.Ua) + e) : T(0);
            }
#pragma unroll
        for (int k = 0; k < R; k++)
#pragma unroll
            for (int j = 0; j < G; j++) vv[k][j] = c[k][j] >= 0 ? gather<KEEP>(x, c[k][j], pol) : T(0);
#pragma unroll
        for (int k = 0; k < R; k++)
#pragma unroll
            for (int j = 0; j < G; j++)
                if (c[k][j] >= 0) y[k] = fmadd(cf[k][j], vv[k][j], y[k]);
    }
}

// Fixed-width Amul rows, software-pipelined: the loads of a round (entries,
// x_p, d_p: none depends on an earlier result) are issued before the
// previous round's gathers, so each round costs about one memory round trip
// instead of two.  For rows of at most G entries (a whole row per round).
template <class T, int R, int G>
struct EllRound {
    int c[R][G];
    T a[R][G];
    T xp[R], d[R];
};

template <class T, int R, int G>
__device__ __forceinline__ void ell_load(EllRound<T, R, G>& e, const Mat<T>& A, const T* x, int pb, int stride, int n)
{
#pragma unroll
    for (int k = 0; k < R; k++) {
        const int p = pb + k * stride;
        const bool ok = p < n;
        e.xp[k] = ok ? x[p] : T(0);
        e.d[k] = ok ? __ldcs(A.d + p) : T(0);
#pragma unroll
        for (int j = 0; j < G; j++) {
            const bool okj = ok && j < A.ell_w;
            const size_t idx = (size_t)j * A.ell_stride + p;
            e.c[k][j] = okj ? __ldcs(A.Ecol + idx) : -1;
            e.a[k][j] = okj ? __ldcs(A.Ea + idx) : T(0);
        }
    }
}

template <class T, int R, int G>
__device__ __forceinline__ void ell_finish(const EllRound<T, R, G>& e, const Mat<T>& A, const T* x, T (&y)[R])
{
    T vv[R][G];
#pragma unroll
    for (int k = 0; k < R; k++)
#pragma unroll
        for (int j = 0; j < G; j++) vv[k][j] = e.c[k][j] >= 0 ? gather<false>(x, e.c[k][j], 0) : T(0);
#pragma unroll
    for (int k = 0; k < R; k++) {
        y[k] = mul_rn(e.d[k], e.xp[k]);
#pragma unroll
        for (int j = 0; j < G; j++)
            if (e.c[k][j] >= 0) y[k] = fmadd(e.a[k][j], vv[k][j], y[k]);
    }
}

// q = A x over rows first + j stride (j = 0, 1, ...) below n; the sink gets
// (row, q_row, x_row) of every row.
template <class T, int R, int G, class Sink>
__device__ __forceinline__ void ell_amul_pipelined(const Mat<T>& A, const T* x, int first, int stride, int n,
                                                   Sink sink)
{
    // two sets of registers take turns (a copy would wait for the loads): the
    // diagonal PCG's FP64 Amul at 128^3 48.5 -> 44.3 us per iteration
    EllRound<T, R, G> ra, rb;
    auto round = [&](EllRound<T, R, G>& cur, EllRound<T, R, G>& nxt, int pb) __attribute__((always_inline)) {
        const int pn = pb + R * stride;
        if (pn < n) ell_load<T, R, G>(nxt, A, x, pn, stride, n);
        T y[R];
        ell_finish<T, R, G>(cur, A, x, y);
#pragma unroll
        for (int k = 0; k < R; k++)
            if (pb + k * stride < n) sink(pb + k * stride, y[k], cur.xp[k]);
    };
    ell_load<T, R, G>(ra, A, x, first, stride, n);
    for (int pb = first; pb < n; pb += 2 * R * stride) {
        round(ra, rb, pb);
        if (pb + R * stride < n) round(rb, ra, pb + R * stride);
    }
}

template <class T>
__device__ __forceinline__ T amul_row(const Mat<T>& A, const T* x, int p)
{
    int pp[1] = {p};
    T y[1], xp[1];
    amul_rows<T, 1, AmulShape<T>::G>(A, x, pp, p + 1, y, xp);
    return y[0];
}

template <class T>
struct Vecs {
    T *x, *r, *w, *p, *q;
};

struct RowIter {
    int first, stride;
};

__device__ __forceinline__ RowIter rows_of(const Group& g)
{
    return RowIter{g.bid * (int)blockDim.x + (int)threadIdx.x, g.nblocks * (int)blockDim.x};
}

// Optional phase timing: group block 0, thread 0 adds SM-clock deltas between
// consecutive marks into phase_clk[slot] (slots: 0..63 forward level, 64..127
// backward level, 128 search direction, 129 Amul + sigma, 130 diagonal pass,
// 132 FP64 refinement residual, 134 update pass, 140 iterations).
enum ClkSlot { CK_FWD = 0, CK_BWD = 64, CK_PUPD = 128, CK_AMUL = 129, CK_DIAG = 130, CK_RESID = 132,
               CK_UPD = 134, CK_ITERS = 140 };

__device__ __forceinline__ long long sm_clock()
{
    long long t;
    asm volatile("mov.u64 %0, %%clock64;" : "=l"(t));
    return t;
}

struct PhaseClock {
    long long* acc;
    long long t;
    __device__ __forceinline__ PhaseClock(long long* a, int bid)
    {
        acc = (a && bid == 0 && threadIdx.x == 0) ? a : nullptr;
        t = sm_clock();
    }
    __device__ __forceinline__ void lap(int slot)
    {
        if (acc) {
            const long long now = sm_clock();
            acc[slot] += now - t;
            t = now;
        }
    }
    __device__ __forceinline__ void count(int slot)
    {
        if (acc) acc[slot] += 1;
    }
};

// Per-thread reduction accumulators.  FP64: fused multiply-add into a double.
// FP32 data: the exact product (a*b, fma(a, b, -a*b)) is added to a
// double-float (hi, lo) pair by Knuth's two-sum, so the sum keeps ~48 bits
// without converting every element to double; the pair is converted once.
template <class T>
struct Acc;
template <>
struct Acc<double> {
    double s = 0.0;
    __device__ __forceinline__ void prod(double a, double b) { s = __fma_rn(a, b, s); }
    __device__ __forceinline__ void add(double a) { s = __dadd_rn(s, a); }
    __device__ __forceinline__ double value() const { return s; }
};
template <>
struct Acc<float> {
    float hi = 0.0f, lo = 0.0f;
    __device__ __forceinline__ void add2(float p, float e)
    {
        const float sum = __fadd_rn(hi, p);
        const float bb = __fsub_rn(sum, hi);
        const float err = __fadd_rn(__fsub_rn(hi, __fsub_rn(sum, bb)), __fsub_rn(p, bb));
        hi = sum;
        lo = __fadd_rn(lo, __fadd_rn(err, e));
    }
    __device__ __forceinline__ void prod(float a, float b)
    {
        const float p = __fmul_rn(a, b);
        add2(p, __fmaf_rn(a, b, -p));
    }
    __device__ __forceinline__ void add(float a) { add2(a, 0.0f); }
    __device__ __forceinline__ double value() const { return (double)hi + (double)lo; }
};

// 16-byte vector of the working precision (float4 / double2): the streaming
// passes move 16 bytes per load so that enough bytes are in flight per SM.
template <class T>
struct V16;
template <>
struct V16<float> {
    using type = float4;
    static constexpr int n = 4;
};
template <>
struct V16<double> {
    using type = double2;
    static constexpr int n = 2;
};
__device__ __forceinline__ float4 vfma(float a, float4 x, float4 y)
{
    return make_float4(__fmaf_rn(a, x.x, y.x), __fmaf_rn(a, x.y, y.y), __fmaf_rn(a, x.z, y.z), __fmaf_rn(a, x.w, y.w));
}
__device__ __forceinline__ double2 vfma(double a, double2 x, double2 y)
{
    return make_double2(__fma_rn(a, x.x, y.x), __fma_rn(a, x.y, y.y));
}
template <class A>
__device__ __forceinline__ void vadd_abs(A& acc, float4 r)
{
    acc.add(fabsf(r.x));
    acc.add(fabsf(r.y));
    acc.add(fabsf(r.z));
    acc.add(fabsf(r.w));
}
template <class A>
__device__ __forceinline__ void vadd_abs(A& acc, double2 r)
{
    acc.add(fabs(r.x));
    acc.add(fabs(r.y));
}
__device__ __forceinline__ float4 vsub(float4 x, float4 y)
{
    return make_float4(__fsub_rn(x.x, y.x), __fsub_rn(x.y, y.y), __fsub_rn(x.z, y.z), __fsub_rn(x.w, y.w));
}
__device__ __forceinline__ float4 vmul(float4 x, float4 y)
{
    return make_float4(__fmul_rn(x.x, y.x), __fmul_rn(x.y, y.y), __fmul_rn(x.z, y.z), __fmul_rn(x.w, y.w));
}
__device__ __forceinline__ double2 vmul(double2 x, double2 y)
{
    return make_double2(__dmul_rn(x.x, y.x), __dmul_rn(x.y, y.y));
}
template <class A>
__device__ __forceinline__ void vprod(A& acc, float4 x, float4 y)
{
    acc.prod(x.x, y.x);
    acc.prod(x.y, y.y);
    acc.prod(x.z, y.z);
    acc.prod(x.w, y.w);
}
template <class A>
__device__ __forceinline__ void vprod(A& acc, double2 x, double2 y)
{
    acc.prod(x.x, y.x);
    acc.prod(x.y, y.y);
}
// ------------------------------------------------------------ phases --------
// Gather the LDU coefficients into the internal layout, a row at a time: its
// entries' faces in groups of 6, then their coefficients (each read once for
// the CSR, the fixed-width layout and the FP32 copies), then the stores.  Bound
// by the gathered coefficients; a pass per array gathered them two or three
// times and one entry after the other.  With the factor and the initial residual
// below taken by rows too, a solve's set-up and first iteration: 64^3 FP64 453 ->
// 399 us, 128^3 1422 -> 1120, 200^3 mixed 5258 -> 4066, PBiCG at 128^3 1603 ->
// 1422.
// Asymmetric: row u's lower entry of face f holds lower_f (A) and upper_f
// (A^T), row l's upper entry upper_f (A) and lower_f (A^T).
template <bool ASYM, class GR>
__device__ bool phase_gather(const SolveArgs& a, const GR& g)
{
    constexpr int G = 6;
    RowIter it = rows_of(g);
    bool bad = false;
    for (int p = it.first; p < a.n; p += it.stride) {
        const int l0 = a.Lptr[p], nl = a.Lptr[p + 1] - l0, u0 = a.Uptr[p], nt = nl + a.Uptr[p + 1] - u0;
        const double dv = a.diag_orig[a.perm[p]];
        for (int off = 0; off < max(nt, a.ell_w); off += G) {
            int f[G];
            double v[G], vt[G];
#pragma unroll
            for (int j = 0; j < G; j++) {
                const int k = off + j;
                f[j] = k < nl ? a.Lface[l0 + k] : k < nt ? a.Uface[u0 + k - nl] : -1;
            }
#pragma unroll
            for (int j = 0; j < G; j++) {
                const bool low = off + j < nl;
                v[j] = f[j] < 0 ? 0.0 : ASYM && low ? a.lower_orig[f[j]] : a.upper_orig[f[j]];
                if (ASYM) vt[j] = f[j] < 0 ? 0.0 : low ? a.upper_orig[f[j]] : a.lower_orig[f[j]];
            }
#pragma unroll
            for (int j = 0; j < G; j++) {
                const int k = off + j;
                if (k < nl) {
                    a.La64[l0 + k] = v[j];
                    bad |= !isfinite(v[j]);
                    if (ASYM) {
                        a.LaT64[l0 + k] = vt[j];
                        bad |= !isfinite(vt[j]);
                    } else {
                        a.La32[l0 + k] = (float)v[j];
                    }
                } else if (k < nt) {
                    a.Ua64[u0 + k - nl] = v[j];
                    if (ASYM)
                        a.UaT64[u0 + k - nl] = vt[j];
                    else
                        a.Ua32[u0 + k - nl] = (float)v[j];
                }
                if (k < a.ell_w) {
                    a.Ea64[(size_t)k * a.n + p] = v[j];
                    if (ASYM)
                        a.EaT64[(size_t)k * a.n + p] = vt[j];
                    else
                        a.Ea32[(size_t)k * a.n + p] = (float)v[j];
                }
            }
        }
        a.d64[p] = dv;
        if (!ASYM) a.d32[p] = (float)dv;
        bad |= !isfinite(dv);
    }
    if (bad) flag_error(a.status, SPUMA_ERR_NONFINITE, -1);
    return group_sync(g);
}

// RN(a/b) through the shared forms of fp64.cuh where they hold.
__device__ __forceinline__ double div_rn(double a, double b)
{
    return divisor_ok(b) && mid_range(a) ? div_by(a, b, recip(b)) : __ddiv_rn(a, b);
}

// A row's pivot: d_p - sum over its lower entries, in face order, of (x_e y_e) /
// pivot of the entry's column; entries in groups of 6, the pivots gathered
// together.
__device__ __forceinline__ double row_pivot(const SolveArgs& a, int p, const double* x, const double* y)
{
    constexpr int G = 6;
    double piv = a.d64[p];
    const int e1 = a.Lptr[p + 1];
    for (int e0 = a.Lptr[p]; e0 < e1; e0 += G) {
        int c[G];
        double xv[G], yv[G], pc[G];
#pragma unroll
        for (int j = 0; j < G; j++) {
            const bool ok = e0 + j < e1;
            c[j] = ok ? a.Lcol[e0 + j] : -1;
            xv[j] = ok ? x[e0 + j] : 0.0;
            yv[j] = !ok ? 0.0 : x == y ? xv[j] : y[e0 + j];
        }
#pragma unroll
        for (int j = 0; j < G; j++) pc[j] = c[j] >= 0 ? a.rD64[c[j]] : 1.0;
#pragma unroll
        for (int j = 0; j < G; j++)
            if (c[j] >= 0) piv = __dsub_rn(piv, div_rn(__dmul_rn(xv[j], yv[j]), pc[j]));
    }
    return piv;
}

// rd times entries e0 .. e1-1 of x into y (and y32).
__device__ __forceinline__ void scale_entries(double rd, const double* x, double* y, float* y32, int e0, int e1)
{
    constexpr int G = 6;
    for (; e0 < e1; e0 += G) {
        double v[G];
#pragma unroll
        for (int j = 0; j < G; j++) v[j] = e0 + j < e1 ? x[e0 + j] : 0.0;
#pragma unroll
        for (int j = 0; j < G; j++)
            if (e0 + j < e1) {
                const double c = __dmul_rn(rd, v[j]);
                y[e0 + j] = c;
                if (y32) y32[e0 + j] = (float)c;
            }
    }
}

// DIC pivots level by level: p_i = d_i - sum_{lower entries} (a a)/p_col,
// then rD = 1/p and the sweep coefficients rD_row * a (+ FP32 copies).
// Diagonal: rD = 1/d.
template <bool ASYM, class GR>
__device__ bool phase_factor(const SolveArgs& a, const GR& g)
{
    RowIter it = rows_of(g);
    const bool dilu = ASYM && a.precond == SPUMA_PRECOND_DILU, dic = !ASYM && a.precond == SPUMA_PRECOND_DIC;
    if (dilu || dic) {
        // DILU: p_u -= (upper_f lower_f) / p_l in face order
        for (int L = 0; L < a.nlev; L++) {
            const int r0 = a.lvl[L], r1 = a.lvl[L + 1];
            for (int p = r0 + it.first; p < r1; p += it.stride) {
                const double piv = row_pivot(a, p, ASYM ? a.LaT64 : a.La64, a.La64);
                a.rD64[p] = piv;
                if (ASYM ? !(piv != 0.0 && isfinite(piv)) : !(piv > 0.0))
                    flag_error(a.status, ASYM ? SPUMA_ERR_SINGULAR : SPUMA_ERR_NOT_SPD, a.perm[p]);
            }
            if (!group_sync(g)) return false;
        }
    }
    for (int p = it.first; p < a.n; p += it.stride) {
        double rd = 1.0;
        if (dilu || dic)
            rd = div_rn(1.0, a.rD64[p]);
        else if (a.precond == SPUMA_PRECOND_DIAGONAL)
            rd = div_rn(1.0, a.d64[p]);
        a.rD64[p] = rd;
        if (!ASYM) a.rD32[p] = (float)rd;
        if (dilu || dic) {
            const int l0 = a.Lptr[p], l1 = a.Lptr[p + 1], u0 = a.Uptr[p], u1 = a.Uptr[p + 1];
            scale_entries(rd, a.La64, a.Lc64, ASYM ? nullptr : a.Lc32, l0, l1);
            scale_entries(rd, a.Ua64, a.Uc64, ASYM ? nullptr : a.Uc32, u0, u1);
            if (ASYM) {
                scale_entries(rd, a.LaT64, a.LcT64, nullptr, l0, l1);
                scale_entries(rd, a.UaT64, a.UcT64, nullptr, u0, u1);
            }
        }
    }
    return group_sync(g);
}

// ------------------------------------------------------ DIC sweeps ---------
// The block's contiguous chunk [c0, c1) of level L (sweep mapping 1):
// the same 1/nblocks share of every level's Morton order, so a block's chunks
// of consecutive levels cover nearly the same region of the mesh.
__device__ __forceinline__ void level_chunk(const int* lvl, int L, int nblocks, int bid, int& c0, int& c1)
{
    const int r0 = lvl[L], r1 = lvl[L + 1];
    const int chunk = (r1 - r0 + nblocks - 1) / nblocks;
    c0 = (int)min((long long)r0 + (long long)bid * chunk, (long long)r1);
    c1 = min(c0 + chunk, r1);
}

// This block's chunks of the first kChunkTable levels, in shared memory, filled
// once per launch (fill_chunk_table) for the wide sweeps.  4 KB leaves blocks of
// 32 threads their 16 per SM; with 256 levels, a natural order of 128^3 (382
// levels) took 4.8 ms an iteration against 2.1.
constexpr int kChunkTable = 512;
__device__ __forceinline__ int2* chunk_table()
{
    __shared__ int2 table[kChunkTable];
    return table;
}
__device__ __forceinline__ void fill_chunk_table(const SolveArgs& a, const Group& g)
{
    int2* t = chunk_table();
    for (int L = threadIdx.x; L < min(a.nlev, kChunkTable); L += blockDim.x) {
        int c0, c1;
        level_chunk(a.lvl, L, g.nblocks, g.bid, c0, c1);
        t[L] = make_int2(c0, c1);
    }
    __syncthreads();
}

// The sweeps with 128 registers per thread (WideGroup).  A level's row takes
// three dependent memory round trips (extents; columns and coefficients;
// gathers of w), and only the last depends on the previous level: so a
// thread's rounds, taken over all its levels as one sequence, are pipelined
// across the grid barriers, the extents two rounds ahead and the entries, r and
// rD (or the row's own w) one round ahead.  After a barrier only the gathers,
// the FMA chain and the store remain.  Warp 0 takes no rows: its first thread
// is the one that arrives at the grid barrier, and the fence of that arrival
// would wait for the warp's own loads ahead.
template <class T>
struct WideShape {
    static constexpr int R = sizeof(T) == 4 ? 2 : 1;   // rows per thread and round
    static constexpr int G = 6;
};

// A thread without a row in a level goes on to its next one, but looks at most
// this many levels ahead at a time and takes an empty round there: threads at the
// edge of their block's chunks looked through all the levels left, at one step
// while the others waited for them, which on meshes of many levels (a natural
// order) cost more than the loads ahead gained.  An iteration, all levels | 8 | 4 |
// 2 | none: natural 64^3 (190 levels) FP64 1288 | 1012 | 983 | 995 | 1069 us, mixed
// 1267 | 893 | 849 | 839 | 989; 64^3 permuted (20 levels) FP64 130 | 131 | 130 | 132
// | 142, mixed 105 | 104 | 103 | 103 | 114 (an empty round per level occupies the
// warps that others wait beside).  One block's levels are narrower, and what an
// empty round costs there less: 100 x 100 x 4, mixed, 468 at 4, 437 at 2.
constexpr int kLookAhead = 4, kLookAheadSolo = 2;

// The thread's rounds: row pb (and pb + stride ...) of level L, below c1.
struct RoundIter {
    int L, pb, c1;
};

template <class T, int R, int G, int NS>
struct SweepRound {
    int e0[R], e1[R], c[R][G];
    T cf[R][G], s[R][NS];
};

// What a sweep loads of its own rows, starts the row's chain from and does with
// the result, and the vector it gathers (which is also where results go).
// w = rD r - sum c w_l; rho += w r at the top level (no upper neighbours there:
// w is final).
template <class T>
struct FwdR {
    static constexpr int NS = 2;
    const T *r, *rD;
    T* w;
    Acc<T>& rho;
    int top;
    __device__ __forceinline__ const T* vec() const { return w; }
    __device__ __forceinline__ void load(int p, T (&s)[NS]) const
    {
        s[0] = r[p];
        s[1] = __ldcs(rD + p);
    }
    __device__ __forceinline__ T init(T (&s)[NS]) const { return mul_rn(s[1], s[0]); }
    __device__ __forceinline__ void store(int p, T v, const T (&s)[NS], int L) const
    {
        w[p] = v;
        if (L == top) rho.prod(v, s[0]);
    }
};
// w -= sum c w_u; rho += w r.
template <class T>
struct BwdR {
    static constexpr int NS = 2;
    const T* r;
    T* w;
    Acc<T>& rho;
    __device__ __forceinline__ const T* vec() const { return w; }
    __device__ __forceinline__ void load(int p, T (&s)[NS]) const
    {
        s[0] = r[p];
        s[1] = w[p];
    }
    __device__ __forceinline__ T init(T (&s)[NS]) const { return s[1]; }
    __device__ __forceinline__ void store(int p, T v, const T (&s)[NS], int) const
    {
        w[p] = v;
        rho.prod(v, s[0]);
    }
};

// Levels from .. to-1 ascending (FWD) or to-1 .. from descending, one grid
// barrier after each (after the last one too unless !last_sync).  SOLO: the
// calling block takes whole levels by itself, with block barriers.  LONG: rows
// of more than G entries are met; their entries past the first G, which the loads
// ahead don't hold, come in groups of three (one by one, each a column and then
// its gather, a row of 14 neighbours cost 126^3 142 against 131 ms in the mixed
// solve; groups of six spill).  The other meshes' loop is free of that code, which
// cost 200^3 1.6 %.  `at_last` runs before the last level's barrier (a reduction's
// partials).
template <class T, bool FWD, bool SOLO, bool LONG, class GR, class Op, class Last>
__device__ __forceinline__ bool wide_sweep(const SolveArgs& a, const Mat<T>& A, const GR& g, PhaseClock& pc, int from,
                                           int to, bool last_sync, const Op& op, Last at_last)
{
    constexpr int R = WideShape<T>::R, G = WideShape<T>::G, NS = Op::NS;
    using Round = SweepRound<T, R, G, NS>;
    // blocks of up to three warps keep it at work
    const int service = !SOLO && blockDim.x >= 4 * kWarp ? kWarp : 0;
    const int tid = (int)threadIdx.x - service, bs = (int)blockDim.x - service;
    const bool chunks = !SOLO && a.sweep != 0, own = SOLO || chunks;
    const int first = own ? tid : g.bid * bs + tid, stride = own ? bs : g.nblocks * bs;
    const int2* table = chunk_table();
    const int* ptr = FWD ? A.Lptr : A.Uptr;
    const int* col = FWD ? A.Lcol : A.Ucol;
    const T* coef = FWD ? A.Lc : A.Uc;
    const unsigned long long pol = keep_policy<T, true>();
    const int Lbeg = FWD ? from : to - 1, Lend = FWD ? to : from - 1;
    // first round of level it.L or of the next level that has one, kAhead levels
    // on at most: there an empty one (see kLookAhead)
    constexpr int kAhead = SOLO ? kLookAheadSolo : kLookAhead;
    auto open = [&](RoundIter& it) {
        if (tid < 0) it.L = Lend;
        for (int k = 0; it.L != Lend; k++) {
            int c0;
            if (chunks && it.L < kChunkTable) {
                c0 = table[it.L].x;
                it.c1 = table[it.L].y;
            } else if (chunks) {
                level_chunk(a.lvl, it.L, g.nblocks, g.bid, c0, it.c1);
            } else {
                c0 = a.lvl[it.L];
                it.c1 = a.lvl[it.L + 1];
            }
            it.pb = c0 + first;
            if (it.pb < it.c1 || k == kAhead) return;
            it.L += FWD ? 1 : -1;
        }
    };
    auto next = [&](RoundIter& it) {
        it.pb += R * stride;
        if (it.pb < it.c1) return;
        it.L += FWD ? 1 : -1;
        open(it);
    };
    auto extents = [&](const RoundIter& it, int (&e0)[R], int (&e1)[R]) {
#pragma unroll
        for (int k = 0; k < R; k++) {
            const int p = it.pb + k * stride;
            const bool ok = it.L != Lend && p < it.c1;
            e0[k] = ok ? __ldcs(ptr + p) : 0;
            e1[k] = ok ? __ldcs(ptr + p + 1) : 0;
        }
    };
    auto entries = [&](const RoundIter& it, Round& q) {
#pragma unroll
        for (int k = 0; k < R; k++) {
            const int p = it.pb + k * stride;
#pragma unroll
            for (int j = 0; j < NS; j++) q.s[k][j] = T(0);
            if (it.L != Lend && p < it.c1) op.load(p, q.s[k]);
#pragma unroll
            for (int j = 0; j < G; j++) {
                const int e = FWD ? q.e0[k] + j : q.e1[k] - 1 - j;
                const bool has = FWD ? e < q.e1[k] : e >= q.e0[k];
                q.c[k][j] = has ? __ldcs(col + e) : -1;
                q.cf[k][j] = has ? __ldcs(coef + e) : T(0);
            }
        }
    };
    RoundIter cur{Lbeg, 0, 0}, nxt, nn;
    Round q, qn;
    int n0[R], n1[R];
    open(cur);
    nxt = cur;
    if (nxt.L != Lend) next(nxt);
    extents(cur, q.e0, q.e1);
    extents(nxt, n0, n1);
    entries(cur, q);
    for (int L = Lbeg; L != Lend; L += FWD ? 1 : -1) {
        while (cur.L == L) {
            // this round's gathers, then the entries of the next round and the
            // extents of the one after
            T x[R][G];
#pragma unroll
            for (int k = 0; k < R; k++)
#pragma unroll
                for (int j = 0; j < G; j++) x[k][j] = q.c[k][j] >= 0 ? gather<true>(op.vec(), q.c[k][j], pol) : T(0);
#pragma unroll
            for (int k = 0; k < R; k++) {
                qn.e0[k] = n0[k];
                qn.e1[k] = n1[k];
            }
            entries(nxt, qn);
            nn = nxt;
            if (nn.L != Lend) next(nn);
            extents(nn, n0, n1);
#pragma unroll
            for (int k = 0; k < R; k++) {
                T acc = op.init(q.s[k]);
#pragma unroll
                for (int j = 0; j < G; j++)
                    if (q.c[k][j] >= 0) acc = fmadd(-q.cf[k][j], x[k][j], acc);
                if (LONG && q.e1[k] - q.e0[k] > G) {   // the rest of a longer row
                    T rest[1] = {acc};
                    const int b0[1] = {FWD ? q.e0[k] + G : q.e0[k]}, b1[1] = {FWD ? q.e1[k] : q.e1[k] - G};
                    rows_chain<T, 1, 3, !FWD, true>(rest, b0, b1, col, coef, op.vec());
                    acc = rest[0];
                }
                const int p = cur.pb + k * stride;
                if (p < cur.c1) op.store(p, acc, q.s[k], L);
            }
            cur = nxt;
            q = qn;
            nxt = nn;
        }
        if (SOLO) {
            __syncthreads();
            continue;
        }
        if (L + (FWD ? 1 : -1) == Lend) {
            at_last();
            if (!last_sync) return true;
        }
        if (!group_sync(g)) return false;
        pc.lap((FWD ? CK_FWD : CK_BWD) + min(L, 63));
    }
    return true;
}

// One level's rows [r0, r1) from `first` with `stride` without the loads ahead
// (Group: 64 registers): extents one round ahead, entries in groups of G, R
// rows in lockstep.
template <class T, bool FWD, class Op>
__device__ __forceinline__ void level_rows(const Mat<T>& A, const Op& op, int r0, int r1, int first, int stride, int L)
{
    constexpr int R = ChainShape<T>::R, G = ChainShape<T>::G;
    const int* ptr = FWD ? A.Lptr : A.Uptr;
    int e0n[R], e1n[R];
#pragma unroll
    for (int k = 0; k < R; k++) {
        const int pn = r0 + first + k * stride;
        e0n[k] = pn < r1 ? __ldcs(ptr + pn) : 0;
        e1n[k] = pn < r1 ? __ldcs(ptr + pn + 1) : 0;
    }
    for (int pb = r0 + first; pb < r1; pb += R * stride) {
        int e0[R], e1[R];
        T v[R], s[R][Op::NS];
#pragma unroll
        for (int k = 0; k < R; k++) {
            const int p = pb + k * stride, pn = p + R * stride;
            e0[k] = e0n[k];
            e1[k] = e1n[k];
            e0n[k] = pn < r1 ? __ldcs(ptr + pn) : 0;
            e1n[k] = pn < r1 ? __ldcs(ptr + pn + 1) : 0;
#pragma unroll
            for (int j = 0; j < Op::NS; j++) s[k][j] = T(0);
            if (p < r1) op.load(p, s[k]);
        }
#pragma unroll
        for (int k = 0; k < R; k++) v[k] = op.init(s[k]);
        rows_chain<T, R, G, !FWD, true>(v, e0, e1, FWD ? A.Lcol : A.Ucol, FWD ? A.Lc : A.Uc, op.vec());
#pragma unroll
        for (int k = 0; k < R; k++)
            if (pb + k * stride < r1) op.store(pb + k * stride, v[k], s[k], L);
    }
}

// Levels from .. to-1 (FWD ascending, else descending) over the grid, one
// barrier after each (the last one's only with last_sync).  Row mapping
// (a.sweep): 1 (default), each block sweeps one contiguous chunk of every level
// (the same 1/nblocks share of each level's Morton order); 0, a level's rows
// strided over the group in blockDim-row pieces.  Measured at 200^3: mixed
// solve 328.8 against 333.5 ms, FP64 582.5 against 599.7 ms.
template <class T, bool FWD, class GR, class Op, class Last>
__device__ __forceinline__ bool sweep_levels(const SolveArgs& a, const Mat<T>& A, const GR& g, PhaseClock& pc, int from,
                                             int to, bool last_sync, const Op& op, Last at_last)
{
    if constexpr (GR::wide) {
        if (A.ell_w > 0 && A.ell_w <= WideShape<T>::G)
            return wide_sweep<T, FWD, false, false>(a, A, g, pc, from, to, last_sync, op, at_last);
        return wide_sweep<T, FWD, false, true>(a, A, g, pc, from, to, last_sync, op, at_last);
    } else {
        const RowIter it = rows_of(g);
        const int Lend = FWD ? to : from - 1;
        for (int L = FWD ? from : to - 1; L != Lend; L += FWD ? 1 : -1) {
            int c0, c1;
            if (a.sweep != 0) {
                level_chunk(a.lvl, L, g.nblocks, g.bid, c0, c1);
                level_rows<T, FWD>(A, op, c0, c1, (int)threadIdx.x, (int)blockDim.x, L);
            } else {
                level_rows<T, FWD>(A, op, a.lvl[L], a.lvl[L + 1], it.first, it.stride, L);
            }
            if (L + (FWD ? 1 : -1) == Lend) {
                at_last();
                if (!last_sync) return true;
            }
            if (!group_sync(g)) return false;
            pc.lap((FWD ? CK_FWD : CK_BWD) + min(L, 63));
        }
        return true;
    }
}

// The small last levels from .. to-1 on the group's first block alone.
template <class T, bool FWD, class GR, class Op>
__device__ __forceinline__ void sweep_solo(const SolveArgs& a, const Mat<T>& A, const GR& g, PhaseClock& pc, int from,
                                           int to, const Op& op)
{
    if constexpr (GR::wide) {
        wide_sweep<T, FWD, true, true>(a, A, g, pc, from, to, true, op, [] {});
    } else {
        for (int L = FWD ? from : to - 1; L != (FWD ? to : from - 1); L += FWD ? 1 : -1) {
            level_rows<T, FWD>(A, op, a.lvl[L], a.lvl[L + 1], (int)threadIdx.x, (int)blockDim.x, L);
            __syncthreads();
        }
    }
}

// w = M^-1 r with the DIC factor held in A's sweep coefficients, and the block
// partials of rho = w.r in SL_B before the last grid barrier.  Forward sweep
// over levels 0 .. nlev-1, backward over nlev-2 .. 0 (the top level has no
// upper neighbours: its backward step would leave w as it is, so its rho terms
// are taken in the forward step), one grid barrier per level.  The small last
// levels (level >= tail_from) run on the group's first block alone, forward
// then backward, with block-level barriers and one grid barrier after them.
template <class T, class GR>
__device__ bool dic_apply(const SolveArgs& a, const Mat<T>& A, Vecs<T> v, const GR& g, PhaseClock& pc)
{
    const int nlev = a.nlev, tail = min(a.tail_from, nlev);
    Acc<T> arho;
    auto rho_partials = [&] {
        double t[1] = {arho.value()};
        block_reduce_store<1>(t, a.partials, SL_B, g.bid);
    };
    if (nlev == 0) {
        rho_partials();
        return group_sync(g);
    }
    const FwdR<T> fwd{v.r, A.rD, v.w, arho, nlev - 1};
    const BwdR<T> bwd{v.r, v.w, arho};
    if (!sweep_levels<T, true>(a, A, g, pc, 0, tail, true, fwd, [&] {
            if (nlev == 1) rho_partials();
        }))
        return false;
    if (tail < nlev) {
        if (g.bid == 0) {
            sweep_solo<T, true>(a, A, g, pc, tail, nlev, fwd);
            sweep_solo<T, false>(a, A, g, pc, tail, nlev - 1, bwd);
        }
        if (tail == 0) rho_partials();
        if (!group_sync(g)) return false;
        pc.lap(CK_FWD + min(tail, 63));
    }
    return sweep_levels<T, false>(a, A, g, pc, 0, min(tail, nlev - 1), true, bwd, rho_partials);
}

// ----------------------------------------------------- streaming passes ---
// Diagonal / no preconditioning in one pass, fused with the pending x/r
// update; returns sum|r| (of the updated r) and rho = w.r through t[0], t[1].
// 16-byte loads, x passed through evict-first (as in update_pass), scalar
// tail: at 128^3, eight streams of 16.8 MB, 38.9 -> 33.3 us.
template <class T>
__device__ bool diag_pass(const SolveArgs& a, const Mat<T>& A, Vecs<T> v, bool pending, T alpha, const Group& g,
                          double (&t)[2])
{
    using VT = typename V16<T>::type;
    constexpr int W = V16<T>::n;
    RowIter it = rows_of(g);
    Acc<T> ares, arho;
    const bool diagonal = a.precond == SPUMA_PRECOND_DIAGONAL;
    const int nv = a.n / W;
    VT* xv = reinterpret_cast<VT*>(v.x);
    VT* rv = reinterpret_cast<VT*>(v.r);
    VT* wv = reinterpret_cast<VT*>(v.w);
    const VT* pv = reinterpret_cast<const VT*>(v.p);
    const VT* qv = reinterpret_cast<const VT*>(v.q);
    const VT* dv = reinterpret_cast<const VT*>(A.rD);
    for (int i = it.first; i < nv; i += it.stride) {
        VT rr = rv[i];
        VT ww;
        if (diagonal) ww = __ldcs(dv + i);
        if (pending) {
            const VT pp = pv[i];
            rr = vfma(-alpha, qv[i], rr);
            __stcs(xv + i, vfma(alpha, pp, __ldcs(xv + i)));
            rv[i] = rr;
            vadd_abs(ares, rr);
        }
        ww = diagonal ? vmul(ww, rr) : rr;
        wv[i] = ww;
        vprod(arho, ww, rr);
    }
    for (int p = nv * W + it.first; p < a.n; p += it.stride) {
        T rr = v.r[p];
        if (pending) {
            v.x[p] = fmadd(alpha, v.p[p], v.x[p]);
            rr = fmadd(-alpha, v.q[p], rr);
            v.r[p] = rr;
            ares.add(fabs(rr));
        }
        const T ww = diagonal ? mul_rn(A.rD[p], rr) : rr;
        v.w[p] = ww;
        arho.prod(ww, rr);
    }
    double acc[2] = {ares.value(), arho.value()};
    block_reduce_store<2>(acc, a.partials, SL_A, g.bid);
    if (!group_sync(g)) return false;
    grid_reduce_read<2>(t, a.partials, SL_A, g.nblocks);
    return true;
}

// p = w (first) or w + beta p; 16-byte loads, scalar tail
template <class T, class GR>
__device__ bool search_direction(const SolveArgs& a, Vecs<T> v, bool first, T beta, const GR& g)
{
    using VT = typename V16<T>::type;
    constexpr int W = V16<T>::n;
    RowIter it = rows_of(g);
    const int nv = a.n / W;
    VT* pv = reinterpret_cast<VT*>(v.p);
    const VT* wv = reinterpret_cast<const VT*>(v.w);
    int i = it.first;
    if constexpr (GR::wide) {   // two at a time: half the threads, as many bytes in flight
        for (; i + it.stride < nv; i += 2 * it.stride) {
            const VT w0 = wv[i], w1 = wv[i + it.stride];
            VT p0 = w0, p1 = w1;
            if (!first) {
                p0 = pv[i];
                p1 = pv[i + it.stride];
                p0 = vfma(beta, p0, w0);
                p1 = vfma(beta, p1, w1);
            }
            pv[i] = p0;
            pv[i + it.stride] = p1;
        }
    }
    for (; i < nv; i += it.stride) {
        const VT ww = wv[i];
        pv[i] = first ? ww : vfma(beta, pv[i], ww);
    }
    for (int p = nv * W + it.first; p < a.n; p += it.stride) v.p[p] = first ? v.w[p] : fmadd(beta, v.p[p], v.w[p]);
    return group_sync(g);
}

// q = A p and sigma = q.p
template <class T, class GR>
__device__ bool amul_sigma(const SolveArgs& a, const Mat<T>& A, Vecs<T> v, const GR& g, double* sigma)
{
    constexpr int R = AmulShape<T>::R, G = AmulShape<T>::G;
    Acc<T> asig;
    RowIter it = rows_of(g);
    // rows [r0, r1) from `first` with `stride`
    auto range = [&](int r0, int r1, int first, int stride) {
        if ((PipeShape<T>::in_solver || GR::wide) && A.ell_w > 0 && A.ell_w <= PipeShape<T>::G) {
            ell_amul_pipelined<T, GR::wide ? 2 : PipeShape<T>::R, PipeShape<T>::G>(A, v.p, r0 + first, stride, r1,
                                                                    [&](int p, T y, T xp) {
                                                                        v.q[p] = y;
                                                                        asig.prod(y, xp);
                                                                    });
            return;
        }
        for (int pb = r0 + first; pb < r1; pb += R * stride) {
            int p[R];
            T y[R], pp[R];
#pragma unroll
            for (int k = 0; k < R; k++) p[k] = pb + k * stride;
            amul_rows<T, R, G>(A, v.p, p, r1, y, pp);
#pragma unroll
            for (int k = 0; k < R; k++)
                if (p[k] < r1) {
                    v.q[p[k]] = y[k];
                    asig.prod(y[k], pp[k]);
                }
        }
    };
    // with amul_chunks each block takes its contiguous chunk of every level,
    // as in the sweeps: the rows a block takes cover one region of the mesh in
    // all levels, so the repeated gathers of a value stay in its SM's L1;
    // otherwise one segment, all rows strided over the group
    const int nseg = a.amul_chunks ? a.nlev : 1;
    for (int L = 0; L < nseg; L++) {
        int c0 = 0, c1 = a.n, first = it.first, stride = it.stride;
        if (a.amul_chunks) {
            level_chunk(a.lvl, L, g.nblocks, g.bid, c0, c1);
            first = (int)threadIdx.x;
            stride = (int)blockDim.x;
        }
        range(c0, c1, first, stride);
    }
    double sacc[1] = {asig.value()};
    block_reduce_store<1>(sacc, a.partials, SL_C, g.bid);
    if (!group_sync(g)) return false;
    double sg[1];
    grid_reduce_read<1>(sg, a.partials, SL_C, g.nblocks);
    *sigma = sg[0];
    return true;
}

// x += alpha p, r -= alpha q and sum|r| as a pass of its own, ahead of the
// forward sweep (16-byte loads, scalar tail).
template <class T, class GR>
__device__ bool update_pass(const SolveArgs& a, Vecs<T> v, T alpha, const GR& g, double* ressum)
{
    using VT = typename V16<T>::type;
    constexpr int W = V16<T>::n;
    RowIter it = rows_of(g);
    Acc<T> acc;
    const int nv = a.n / W;
    VT* xv = reinterpret_cast<VT*>(v.x);
    VT* rv = reinterpret_cast<VT*>(v.r);
    const VT* pv = reinterpret_cast<const VT*>(v.p);
    const VT* qv = reinterpret_cast<const VT*>(v.q);
    int i = it.first;
    if constexpr (GR::wide) {
        for (; i + it.stride < nv; i += 2 * it.stride) {
            const int i2 = i + it.stride;
            const VT q0 = qv[i], q1 = qv[i2], r0 = rv[i], r1 = rv[i2], p0 = pv[i], p1 = pv[i2];
            const VT x0 = __ldcs(xv + i), x1 = __ldcs(xv + i2);
            const VT s0 = vfma(-alpha, q0, r0), s1 = vfma(-alpha, q1, r1);
            __stcs(xv + i, vfma(alpha, p0, x0));
            __stcs(xv + i2, vfma(alpha, p1, x1));
            rv[i] = s0;
            rv[i2] = s1;
            vadd_abs(acc, s0);
            vadd_abs(acc, s1);
        }
    }
    for (; i < nv; i += it.stride) {
        const VT rr = vfma(-alpha, qv[i], rv[i]);
        __stcs(xv + i, vfma(alpha, pv[i], __ldcs(xv + i)));
        rv[i] = rr;
        vadd_abs(acc, rr);
    }
    for (int p = nv * W + it.first; p < a.n; p += it.stride) {
        v.x[p] = fmadd(alpha, v.p[p], v.x[p]);
        const T r1 = fmadd(-alpha, v.q[p], v.r[p]);
        v.r[p] = r1;
        acc.add(fabs(r1));
    }
    double t[1] = {acc.value()};
    block_reduce_store<1>(t, a.partials, SL_D, g.bid);
    if (!group_sync(g)) return false;
    grid_reduce_read<1>(t, a.partials, SL_D, g.nblocks);
    *ressum = t[0];
    return true;
}

// w = M^-1 r and rho = w.r, after the pending update (x += alpha p,
// r -= alpha q, a pass of its own for DIC, fused into the diagonal pass
// otherwise), whose sum|r| is handed to `after_update`: it stops the loop
// (1), lets it go on (0) or replaces r and asks for w to be computed from the
// new r (2).  DIC: the caller may run with the DIC preconditioner.
// Returns 0 (w and rho ready), 2 (stop) or -1 (device error).
template <class T, bool DIC, class AfterUpdate, class GR>
__device__ int precondition(const SolveArgs& a, const Mat<T>& A, Vecs<T> v, bool pending, T alpha, const GR& g,
                            PhaseClock& pc, double* rho, AfterUpdate after_update)
{
    if (DIC && a.precond == SPUMA_PRECOND_DIC) {
        if (pending) {
            double ressum;
            if (!update_pass<T>(a, v, alpha, g, &ressum)) return -1;
            pc.lap(CK_UPD);
            const int act = after_update(ressum);
            if (act < 0) return -1;
            if (act == 1) return 2;
        }
        if (!dic_apply<T>(a, A, v, g, pc)) return -1;
        double t[1];
        grid_reduce_read<1>(t, a.partials, SL_B, g.nblocks);
        *rho = t[0];
        return 0;
    }
    double t[2];
    if (!diag_pass<T>(a, A, v, pending, alpha, g, t)) return -1;
    pc.lap(CK_DIAG);
    const int act = pending ? after_update(t[0]) : 0;
    if (act < 0) return -1;
    if (act == 1) return 2;
    if (act == 2 && !diag_pass<T>(a, A, v, false, T(0), g, t)) return -1;
    *rho = t[1];
    return 0;
}

// PCG iterations on (A, v.r) from the current v.x (OpenFOAM recurrences).
// Returns the iteration count, or -1 when a device error stopped the group.
template <class T, class GR>
__device__ int pcg_loop(const SolveArgs& a, const Mat<T>& A, Vecs<T> v, double nfac, double res0, double tol,
                        double rel_tol, int max_iter, int min_iter, double* res_out, int* singular,
                        const GR& g)
{
    PhaseClock pc(a.phase_clk, g.bid);
    double res = res0;
    *res_out = res;
    if (!(min_iter > 0 || !converged(res0, res0, tol, rel_tol))) return 0;
    int n_it = 0;
    double rho = 1.0, rho_old;
    T alpha = (T)0;
    bool pending = false;
    for (;;) {
        rho_old = rho;
        const int st = precondition<T, true>(a, A, v, pending, alpha, g, pc, &rho, [&](double ressum) {
            res = ressum / nfac;
            n_it++;
            return ((n_it < max_iter && !converged(res, res0, tol, rel_tol)) || n_it < min_iter) ? 0 : 1;
        });
        if (st < 0) return -1;
        if (st == 2) break;
        const bool first = !pending;
        if (!search_direction<T>(a, v, first, first ? (T)0 : (T)(rho / rho_old), g)) return -1;
        pc.lap(CK_PUPD);
        double sigma;
        if (!amul_sigma<T>(a, A, v, g, &sigma)) return -1;
        pc.lap(CK_AMUL);
        pc.count(CK_ITERS);
        if (fabs(sigma) / nfac < 1e-300) {
            *singular = 1;
            break;
        }
        alpha = (T)(rho / sigma);
        pending = true;
    }
    *res_out = res;
    return n_it;
}

// FP64 refinement step of the mixed forms: x += xs (FP32 correction, reset to
// 0) when fold, then r = b - A64 x with sum|r| and max|r|, and r32 = float(r).
__device__ bool refine_residual(const SolveArgs& a, const Group& g, bool fold, double* ressum, double* rmax)
{
    RowIter it = rows_of(g);
    const Mat<double> A64 = mat_of<double>(a);
    if (fold) {
        for (int p = it.first; p < a.n; p += it.stride) {
            a.x[p] = __dadd_rn(a.x[p], (double)a.xi[p]);
            a.xi[p] = 0.0f;
        }
        if (!group_sync(g)) return false;
    }
    double acc[1] = {0.0}, mx[1] = {0.0};
    for (int p = it.first; p < a.n; p += it.stride) {
        const double rr = a.b[p] - amul_row<double>(A64, a.x, p);
        a.r[p] = rr;
        a.ri[p] = (float)rr;
        acc[0] += fabs(rr);
        mx[0] = fmax(mx[0], fabs(rr));
    }
    block_reduce_store<1>(acc, a.partials, SL_D, g.bid);
    block_max_store<1>(mx, a.partials, SL_DMAX, g.bid);
    if (!group_sync(g)) return false;
    double t[1], m[1];
    grid_reduce_read<1>(t, a.partials, SL_D, g.nblocks);
    grid_reduce_read<1, true>(m, a.partials, SL_DMAX, g.nblocks);
    *ressum = t[0];
    *rmax = m[0];
    return true;
}

// Mixed precision with reliable updates (without preconditioner or with the
// diagonal; DIC: solve_mixed_eisenstat): FP32 PCG whose correction and
// residual are replaced by FP64 ones (x += xs; r = b - A64 x) whenever the
// FP32 residual has dropped by inner_rel_tol since the last replacement, the
// FP32 residual claims convergence, or max_iter is reached; the search
// direction is kept, so the Krylov space is never restarted.
template <class GR>
__device__ bool solve_mixed_reliable(const SolveArgs& a, const GR& g, double nfac, double res0,
                                     spuma_solver_perf& pf)
{
    RowIter it = rows_of(g);
    const Mat<float> A32 = mat_of<float>(a);
    Vecs<float> v{a.xi, a.ri, a.wi, a.pi, a.qi};
    PhaseClock pc(a.phase_clk, g.bid);
    const double delta = a.inner_rel_tol;
    double res = res0, rupd = res0, rho = 1.0, rho_old;
    int n_it = 0, updates = 0, singular = 0;
    float alpha = 0.0f;
    bool pending = false, ok = true;
    if (!converged(res0, res0, a.tol, a.rel_tol)) {
        for (int p = it.first; p < a.n; p += it.stride) {
            v.r[p] = (float)a.r[p];
            v.x[p] = 0.0f;
        }
        if (!group_sync(g)) return false;
        for (;;) {
            rho_old = rho;
            const int st = precondition<float, false>(a, A32, v, pending, alpha, g, pc, &rho, [&](double ressum) {
                n_it++;
                const double ress = ressum / nfac;
                if (!(ress < delta * rupd || converged(ress, res0, a.tol, a.rel_tol) || n_it >= a.max_iter)) return 0;
                double rs, rm;
                if (!refine_residual(a, g, true, &rs, &rm)) return -1;
                pc.lap(CK_RESID);
                updates++;
                res = rs / nfac;
                if (converged(res, res0, a.tol, a.rel_tol) || n_it >= a.max_iter) return 1;
                rupd = res;
                return 2;
            });
            if (st < 0) return false;
            if (st == 2) break;
            const bool first = !pending;
            if (!search_direction<float>(a, v, first, first ? 0.0f : (float)(rho / rho_old), g)) return false;
            pc.lap(CK_PUPD);
            double sigma;
            if (!amul_sigma<float>(a, A32, v, g, &sigma)) return false;
            pc.lap(CK_AMUL);
            pc.count(CK_ITERS);
            if (fabs(sigma) / nfac < 1e-300) {
                singular = 1;
                double rs, rm;
                ok = refine_residual(a, g, true, &rs, &rm);
                res = rs / nfac;
                break;
            }
            alpha = (float)(rho / sigma);
            pending = true;
        }
    }
    // the Amul's rows in lockstep gather p evict-last: hand its lines back
    release_lines(a.pi, 4 * (size_t)a.n, it.first, it.stride);
    pf.initial_residual = res0;
    pf.final_residual = res;
    pf.n_iter = n_it;
    pf.n_outer = updates;
    pf.converged = converged(res, res0, a.tol, a.rel_tol);
    pf.singular = singular;
    return ok;
}

// The same reliable updates for DIC, with Eisenstat's form of the inner PCG (S.
// C. Eisenstat, "Efficient implementation of a class of preconditioned conjugate
// gradient methods", SIAM J. Sci. Stat. Comput. 2, 1981).  M = (P + L) P^-1 (P +
// U) shares A's off-diagonal, A = L + D + U, so the product A p follows from the
// two sweeps and no Amul is needed.  With y = (P + L)^-1 r (kept in place of r),
// the search direction's image t = P^-1 (P + U) p:
//   rho = y.P y;  t = y + beta t;  p = t - P^-1 U p           (backward sweep)
//   h = p - (P + L)^-1 A p = (2 - D/P) p - t - P^-1 L h        (forward sweep)
//   sigma = p.A p = (P t).(p - h);  alpha = rho/sigma
//   x += alpha p;  y -= alpha (p - h)
// the same iterates in exact arithmetic.  An iteration reads 16F + 72N bytes
// instead of 36F + 76N and has two grid barriers fewer: 200^3 402 -> 330 us,
// 128^3 181 -> 146, 64^3 100 -> 92 per iteration; 1142 iterations to 1e-11 at
// 200^3 against 1138 with the product.  sum|r|, which decides
// when the FP64 residual is taken, is followed by kappa sqrt(rho): kappa = sum|r|
// / sqrt(rho) at the last FP64 residual (it moves by 2-3 % between them once the
// first digits are gone: 24^3 and 48^3, log-normal diffusivity); whether the
// solve has converged is decided on the FP64 residual alone, as above.
struct FwdY {   // y = rD r - sum c y_l; rho += y (P y)
    static constexpr int NS = 3;
    const float *r, *rD, *P;
    float* y;
    Acc<float>& rho;
    __device__ __forceinline__ const float* vec() const { return y; }
    __device__ __forceinline__ void load(int p, float (&s)[NS]) const
    {
        s[0] = r[p];
        s[1] = __ldcs(rD + p);
        s[2] = __ldcs(P + p);
    }
    __device__ __forceinline__ float init(float (&s)[NS]) const { return __fmul_rn(s[1], s[0]); }
    __device__ __forceinline__ void store(int p, float v, const float (&s)[NS], int) const
    {
        y[p] = v;
        rho.prod(__fmul_rn(s[2], v), v);
    }
};
struct BwdP {   // t = y + beta t; p = t - sum c p_u
    static constexpr int NS = 2;
    const float* y;
    float *t, *p;
    float beta;
    bool first;
    __device__ __forceinline__ const float* vec() const { return p; }
    __device__ __forceinline__ void load(int i, float (&s)[NS]) const
    {
        s[0] = y[i];
        s[1] = first ? 0.0f : __ldcs(t + i);
    }
    __device__ __forceinline__ float init(float (&s)[NS]) const { return s[1] = first ? s[0] : __fmaf_rn(beta, s[1], s[0]); }
    __device__ __forceinline__ void store(int i, float v, const float (&s)[NS], int) const
    {
        t[i] = s[1];
        p[i] = v;
    }
};
struct FwdH {   // h = e p - t - sum c h_l; sigma += (P t)(p - h)
    static constexpr int NS = 4;
    const float *p, *t, *e, *P;
    float* h;
    Acc<float>& sigma;
    __device__ __forceinline__ const float* vec() const { return h; }
    __device__ __forceinline__ void load(int i, float (&s)[NS]) const
    {
        s[0] = p[i];
        s[1] = t[i];
        s[2] = __ldcs(e + i);
        s[3] = __ldcs(P + i);
    }
    __device__ __forceinline__ float init(float (&s)[NS]) const { return __fmaf_rn(s[2], s[0], -s[1]); }
    __device__ __forceinline__ void store(int i, float v, const float (&s)[NS], int) const
    {
        h[i] = v;
        sigma.prod(__fmul_rn(s[3], s[1]), __fsub_rn(s[0], v));
    }
};

template <class GR>
__device__ bool solve_mixed_eisenstat(const SolveArgs& a, const GR& g, double nfac, double res0, spuma_solver_perf& pf)
{
    RowIter it = rows_of(g);
    const Mat<float> A = mat_of<float>(a);
    PhaseClock pc(a.phase_clk, g.bid);
    // t, e = 2 - D/P and P live in FP64 vectors that the mixed forms do not use
    float *x = a.xi, *r = a.ri, *y = a.wi, *p = a.pi, *h = a.qi;
    float *t = reinterpret_cast<float*>(a.p), *e = reinterpret_cast<float*>(a.w), *P = reinterpret_cast<float*>(a.q);
    const int nlev = a.nlev, tail = min(a.tail_from, nlev), nv = a.n / 4;
    const double delta = a.inner_rel_tol;
    // partials of one sum, the barrier, the grid's value
    auto total = [&](Acc<float>& acc, int slot, double* out) {
        double v[1] = {acc.value()};
        block_reduce_store<1>(v, a.partials, slot, g.bid);
        if (!group_sync(g)) return false;
        grid_reduce_read<1>(v, a.partials, slot, g.nblocks);
        *out = v[0];
        return true;
    };
    auto read = [&](int slot, double* out) {
        double v[1];
        grid_reduce_read<1>(v, a.partials, slot, g.nblocks);
        *out = v[0];
    };
    auto partials = [&](Acc<float>& acc, int slot) {
        double v[1] = {acc.value()};
        block_reduce_store<1>(v, a.partials, slot, g.bid);
    };
    auto forward_r = [&](double* rho) {
        Acc<float> acc;
        const FwdY op{r, A.rD, P, y, acc};
        if (!sweep_levels<float, true>(a, A, g, pc, 0, tail, true, op, [&] {
                if (tail == nlev) partials(acc, SL_B);
            }))
            return false;
        if (tail < nlev) {
            if (g.bid == 0) sweep_solo<float, true>(a, A, g, pc, tail, nlev, op);
            return total(acc, SL_B, rho);
        }
        read(SL_B, rho);
        return true;
    };
    auto directions = [&](bool first, float beta, double* sigma) {
        const BwdP bwd{y, t, p, beta, first};
        if (tail < nlev) {
            if (g.bid == 0) sweep_solo<float, false>(a, A, g, pc, tail, nlev, bwd);
            if (!group_sync(g)) return false;
            pc.lap(CK_BWD + min(tail, 63));
        }
        // no barrier between the backward and the forward step of level 0: a
        // row's p and t are its own thread's
        if (!sweep_levels<float, false>(a, A, g, pc, 0, tail, false, bwd, [] {})) return false;
        Acc<float> acc;
        const FwdH fwd{p, t, e, P, h, acc};
        if (!sweep_levels<float, true>(a, A, g, pc, 0, tail, true, fwd, [&] {
                if (tail == nlev) partials(acc, SL_C);
            }))
            return false;
        if (tail < nlev) {
            if (g.bid == 0) sweep_solo<float, true>(a, A, g, pc, tail, nlev, fwd);
            const bool ok = total(acc, SL_C, sigma);
            pc.lap(CK_FWD + min(tail, 63));
            return ok;
        }
        read(SL_C, sigma);
        return true;
    };
    double res = res0, rupd = res0;
    int n_it = 0, updates = 0, singular = 0;
    bool ok = true;
    if (!converged(res0, res0, a.tol, a.rel_tol)) {
        for (int i = it.first; i < a.n; i += it.stride) {
            const double rd = a.rD64[i];
            P[i] = (float)__ddiv_rn(1.0, rd);
            e[i] = (float)__fma_rn(-rd, a.d64[i], 2.0);
            r[i] = (float)a.r[i];
            x[i] = 0.0f;
        }
        if (!group_sync(g)) return false;
        double rho, rho_old = 1.0;
        if (!forward_r(&rho)) return false;
        double kappa = res / sqrt(rho);
        for (bool first = true;; first = false) {
            double sigma;
            if (!directions(first, first ? 0.0f : (float)(rho / rho_old), &sigma)) return false;
            pc.count(CK_ITERS);
            double rs, rm;
            if (fabs(sigma) / nfac < 1e-300) {
                singular = 1;
                ok = refine_residual(a, g, true, &rs, &rm);
                res = rs / nfac;
                break;
            }
            const float alpha = (float)(rho / sigma);
            // x += alpha p, y -= alpha (p - h), rho = y.P y
            Acc<float> acc;
            float4 *x4 = reinterpret_cast<float4*>(x), *y4 = reinterpret_cast<float4*>(y);
            const float4 *p4 = reinterpret_cast<const float4*>(p), *h4 = reinterpret_cast<const float4*>(h);
            const float4* P4 = reinterpret_cast<const float4*>(P);
            for (int i = it.first; i < nv; i += it.stride) {
                const float4 pp = p4[i], gg = vsub(pp, __ldcs(h4 + i));
                const float4 yy = vfma(-alpha, gg, y4[i]);
                __stcs(x4 + i, vfma(alpha, pp, __ldcs(x4 + i)));
                y4[i] = yy;
                vprod(acc, vmul(__ldcs(P4 + i), yy), yy);
            }
            for (int i = 4 * nv + it.first; i < a.n; i += it.stride) {
                const float yy = __fmaf_rn(-alpha, __fsub_rn(p[i], h[i]), y[i]);
                x[i] = __fmaf_rn(alpha, p[i], x[i]);
                y[i] = yy;
                acc.prod(__fmul_rn(P[i], yy), yy);
            }
            rho_old = rho;
            if (!total(acc, SL_D, &rho)) return false;
            pc.lap(CK_UPD);
            n_it++;
            const double est = kappa * sqrt(rho);
            if (!(est < delta * rupd || converged(est, res0, a.tol, a.rel_tol) || n_it >= a.max_iter)) continue;
            if (!refine_residual(a, g, true, &rs, &rm)) return false;
            pc.lap(CK_RESID);
            updates++;
            res = rs / nfac;
            if (converged(res, res0, a.tol, a.rel_tol) || n_it >= a.max_iter) break;
            rupd = res;
            if (!forward_r(&rho)) return false;
            kappa = res / sqrt(rho);
        }
    }
    // y, p and h were gathered evict-last: hand their lines back
    release_lines(y, 4 * (size_t)a.n, it.first, it.stride);
    release_lines(p, 4 * (size_t)a.n, it.first, it.stride);
    release_lines(h, 4 * (size_t)a.n, it.first, it.stride);
    pf.initial_residual = res0;
    pf.final_residual = res;
    pf.n_iter = n_it;
    pf.n_outer = updates;
    pf.converged = converged(res, res0, a.tol, a.rel_tol);
    pf.singular = singular;
    return ok;
}

// x = x_orig (or 0), b = b_orig in internal order; q = A x; r = b - q;
// normFactor = sum(|q - s xbar| + |b - s xbar|) + 1e-20; returns res0 and nfac.
template <class GR>
__device__ bool phase_init(const SolveArgs& a, const GR& g, double* nfac, double* res0)
{
    RowIter it = rows_of(g);
    const Mat<double> A = mat_of<double>(a);
    double sx[1] = {0.0};
    for (int p = it.first; p < a.n; p += it.stride) {
        const int i = a.perm[p];
        const double xv = a.zero_x0 ? 0.0 : a.x_orig[i], bv = a.b_orig[i];
        a.x[p] = xv;
        a.b[p] = bv;
        sx[0] += xv;
        if (!isfinite(bv)) flag_error(a.status, SPUMA_ERR_NONFINITE, i);
    }
    block_reduce_store<1>(sx, a.partials, SL_A, g.bid);
    if (!group_sync(g)) return false;
    grid_reduce_read<1>(sx, a.partials, SL_A, g.nblocks);
    const double xbar = a.n > 0 ? sx[0] / (double)a.n : 0.0;
    double t2[2] = {0.0, 0.0};
    for (int p = it.first; p < a.n; p += it.stride) {
        const double qq = amul_row<double>(A, a.x, p), bv = a.b[p], rr = bv - qq;
        a.q[p] = qq;
        a.r[p] = rr;
        // the row sum of A in entry order (the padding of the fixed-width layout adds 0)
        double s = a.d64[p];
        if (a.ell_w > 0) {
            for (int j = 0; j < a.ell_w; j++) s += a.Ea64[(size_t)j * a.n + p];
        } else {
            for (int e = a.Lptr[p]; e < a.Lptr[p + 1]; e++) s += a.La64[e];
            for (int e = a.Uptr[p]; e < a.Uptr[p + 1]; e++) s += a.Ua64[e];
        }
        const double tt = s * xbar;
        t2[0] += fabs(qq - tt) + fabs(bv - tt);
        t2[1] += fabs(rr);
    }
    block_reduce_store<2>(t2, a.partials, SL_INIT, g.bid);
    if (!group_sync(g)) return false;
    grid_reduce_read<2>(t2, a.partials, SL_INIT, g.nblocks);
    const double sum_r = t2[1];
    *nfac = t2[0] + 1e-20;
    *res0 = sum_r / *nfac;
    return true;
}

// The report's true residual ||b - A x||_2 / ||b||_2 (||b - A x||_2 when b = 0)
// in FP64 from the FP64 coefficients of A, for every solve kind: each r_p in
// the Amul's face order, the sums of squares as fused multiply-adds per
// thread, then the deterministic block and grid reductions.  b_int: b in
// internal order, or NULL to read the caller's b through perm (PBiCG reuses
// the internal b as its transposed residual).
__device__ bool true_residual(const SolveArgs& a, const Mat<double>& A, const double* b_int, const Group& g,
                              double* out)
{
    RowIter it = rows_of(g);
    double acc[2] = {0.0, 0.0};
    for (int p = it.first; p < a.n; p += it.stride) {
        const double bv = b_int ? b_int[p] : a.b_orig[a.perm[p]];
        const double rr = __dsub_rn(bv, amul_row<double>(A, a.x, p));
        acc[0] = __fma_rn(rr, rr, acc[0]);
        acc[1] = __fma_rn(bv, bv, acc[1]);
    }
    block_reduce_store<2>(acc, a.partials, SL_TRUE, g.bid);
    if (!group_sync(g)) return false;
    double t[2];
    grid_reduce_read<2>(t, a.partials, SL_TRUE, g.nblocks);
    *out = t[1] > 0.0 ? __ddiv_rn(__dsqrt_rn(t[0]), __dsqrt_rn(t[1])) : __dsqrt_rn(t[0]);
    return true;
}

__device__ void phase_store_x(const SolveArgs& a, const Group& g)
{
    RowIter it = rows_of(g);
    for (int p = it.first; p < a.n; p += it.stride) a.x_orig[a.perm[p]] = a.x[p];
}

// Mixed precision, restarted form: FP64 refinement around FP32 inner PCG
// solves of A d = r / max|r| from d = 0 to inner_rel_tol.
template <class GR>
__device__ bool solve_mixed_restart(const SolveArgs& a, const GR& g, double nfac, spuma_solver_perf& pf)
{
    RowIter it = rows_of(g);
    const Mat<float> A32 = mat_of<float>(a);
    Vecs<float> vi{a.xi, a.ri, a.wi, a.pi, a.qi};
    int outer = 0, total = 0, singular = 0;
    double res = 0.0, res0 = 0.0;
    for (;;) {
        double rs, rm;
        if (!refine_residual(a, g, false, &rs, &rm)) return false;
        res = rs / nfac;
        if (outer == 0) res0 = res;
        if (res < a.tol || outer >= a.max_outer || singular) break;
        const double s = rm;
        if (s == 0.0) break;
        Acc<float> ain;
        for (int p = it.first; p < a.n; p += it.stride) {
            float rv = (float)(a.r[p] / s);
            vi.r[p] = rv;
            vi.x[p] = 0.0f;
            ain.add(fabsf(rv));
        }
        double iacc[1] = {ain.value()};
        block_reduce_store<1>(iacc, a.partials, SL_C, g.bid);
        if (!group_sync(g)) return false;
        double ti[1];
        grid_reduce_read<1>(ti, a.partials, SL_C, g.nblocks);
        const double infac = ti[0] + 1e-20;
        const double ires0 = ti[0] / infac;
        double ires;
        int n_in = pcg_loop<float>(a, A32, vi, infac, ires0, 0.0, a.inner_rel_tol, a.max_iter, 1, &ires, &singular, g);
        if (n_in < 0) return false;
        total += n_in;
        for (int p = it.first; p < a.n; p += it.stride) a.x[p] = fma(s, (double)vi.x[p], a.x[p]);
        if (!group_sync(g)) return false;
        outer++;
    }
    release_lines(a.wi, 4 * (size_t)a.n, it.first, it.stride);
    release_lines(a.pi, 4 * (size_t)a.n, it.first, it.stride);
    pf.initial_residual = res0;
    pf.final_residual = res;
    pf.n_iter = total;
    pf.n_outer = outer;
    pf.converged = res < a.tol;
    pf.singular = singular;
    return true;
}

// -------------------------------------------------------------- PBiCG ---
// One level's rows of both DILU applies (A and A^T) in one direction: they
// share the level's structure, so the extents and columns are read once, and
// the two chains' gathers are in flight together.  FWD: w = rD r - sum c w_l,
// else w -= sum c w_u (descending) and rho += wA rT.
template <bool FWD, int G>
__device__ __forceinline__ void dilu_rows(const Mat<double>& A, const Mat<double>& AT, const double* rA,
                                          const double* rT, double* wA, double* wT, int r0, int r1, int first,
                                          int stride, bool rho, Acc<double>& arho)
{
    const int* ptr = FWD ? A.Lptr : A.Uptr;
    const int* col = FWD ? A.Lcol : A.Ucol;
    const double *ca = FWD ? A.Lc : A.Uc, *ct = FWD ? AT.Lc : AT.Uc;
    int p = r0 + first;
    int n0 = p < r1 ? __ldcs(ptr + p) : 0, n1 = p < r1 ? __ldcs(ptr + p + 1) : 0;
    for (; p < r1; p += stride) {
        const int e0 = n0, e1 = n1, pn = p + stride;
        n0 = pn < r1 ? __ldcs(ptr + pn) : 0;
        n1 = pn < r1 ? __ldcs(ptr + pn + 1) : 0;
        const double rt = rT[p];
        double ya, yt;
        if (FWD) {
            const double rd = __ldcs(A.rD + p);
            ya = mul_rn(rd, rA[p]);
            yt = mul_rn(rd, rt);
        } else {
            ya = wA[p];
            yt = wT[p];
        }
        for (int off = 0; off < e1 - e0; off += G) {
            int c[G];
            double a[G], t[G], xa[G], xt[G];
#pragma unroll
            for (int j = 0; j < G; j++) {
                const int e = FWD ? e0 + off + j : e1 - 1 - off - j;
                const bool ok = FWD ? e < e1 : e >= e0;
                c[j] = ok ? __ldcs(col + e) : -1;
                a[j] = ok ? __ldcs(ca + e) : 0.0;
                t[j] = ok ? __ldcs(ct + e) : 0.0;
            }
#pragma unroll
            for (int j = 0; j < G; j++) {
                xa[j] = c[j] >= 0 ? wA[c[j]] : 0.0;
                xt[j] = c[j] >= 0 ? wT[c[j]] : 0.0;
            }
#pragma unroll
            for (int j = 0; j < G; j++)
                if (c[j] >= 0) {
                    ya = fmadd(-a[j], xa[j], ya);
                    yt = fmadd(-t[j], xt[j], yt);
                }
        }
        wA[p] = ya;
        wT[p] = yt;
        if (rho) arho.prod(ya, rt);
    }
}

// wA = M^-1 rA and wT = M^-T rT, level by level together (as dic_apply: one
// grid barrier per level, the small last levels on the first block alone),
// with the partials of rho = wA.rT in SL_B before the last barrier.  The two
// applies one after the other took twice the barriers and read the extents
// and columns twice: 128^3, DILU, an iteration 517 -> 381 us.
template <class GR>
__device__ bool dilu_apply(const SolveArgs& a, const Mat<double>& A, const Mat<double>& AT, const double* rA,
                           const double* rT, double* wA, double* wT, const GR& g, PhaseClock& pc)
{
    constexpr int G = GR::wide ? 6 : 3;
    const RowIter it = rows_of(g);
    const int nlev = a.nlev, tail = min(a.tail_from, nlev);
    const int tid = (int)threadIdx.x, bs = (int)blockDim.x;
    Acc<double> arho;
    auto end_step = [&](bool last) {
        if (last) {
            double t[1] = {arho.value()};
            block_reduce_store<1>(t, a.partials, SL_B, g.bid);
        }
        return group_sync(g);
    };
    if (nlev == 0) return end_step(true);
    auto rows = [&](int L, int& c0, int& c1, int& first, int& stride) {
        if (a.sweep != 0) {
            level_chunk(a.lvl, L, g.nblocks, g.bid, c0, c1);
            first = tid;
            stride = bs;
        } else {
            c0 = a.lvl[L];
            c1 = a.lvl[L + 1];
            first = it.first;
            stride = it.stride;
        }
    };
    int c0, c1, first, stride;
    for (int L = 0; L < tail; L++) {
        rows(L, c0, c1, first, stride);
        dilu_rows<true, G>(A, AT, rA, rT, wA, wT, c0, c1, first, stride, L == nlev - 1, arho);
        if (!end_step(nlev == 1)) return false;
        pc.lap(CK_FWD + min(L, 63));
    }
    if (tail < nlev) {
        if (g.bid == 0) {
            for (int L = tail; L < nlev; L++) {
                dilu_rows<true, G>(A, AT, rA, rT, wA, wT, a.lvl[L], a.lvl[L + 1], tid, bs, L == nlev - 1, arho);
                __syncthreads();
            }
            for (int L = nlev - 2; L >= tail; L--) {
                dilu_rows<false, G>(A, AT, rA, rT, wA, wT, a.lvl[L], a.lvl[L + 1], tid, bs, true, arho);
                __syncthreads();
            }
        }
        if (!end_step(tail == 0)) return false;
        pc.lap(CK_FWD + min(tail, 63));
    }
    for (int L = min(tail, nlev - 1) - 1; L >= 0; L--) {
        rows(L, c0, c1, first, stride);
        dilu_rows<false, G>(A, AT, rA, rT, wA, wT, c0, c1, first, stride, true, arho);
        if (!end_step(L == 0)) return false;
        pc.lap(CK_BWD + min(L, 63));
    }
    return true;
}

// yA = A pA and yT = A^T pT over the thread's rows, sink(p, yA_p, yT_p).  On
// the fixed-width layout both read a row's columns once; each sum in entry
// order, as amul_row takes it.
template <class GR, class Sink>
__device__ __forceinline__ void dual_amul(const SolveArgs& a, const Mat<double>& A, const Mat<double>& AT,
                                          const double* pA, const double* pT, const GR& g, Sink sink)
{
    const RowIter it = rows_of(g);
    if (GR::wide && A.ell_w > 0 && A.ell_w <= 6) {
        for (int p = it.first; p < a.n; p += it.stride) {
            int c[6];
            double u[6], w[6], xa[6], xt[6];
#pragma unroll
            for (int j = 0; j < 6; j++) {
                const bool ok = j < A.ell_w;
                const size_t e = (size_t)j * A.ell_stride + p;
                c[j] = ok ? __ldcs(A.Ecol + e) : -1;
                u[j] = ok ? __ldcs(A.Ea + e) : 0.0;
                w[j] = ok ? __ldcs(AT.Ea + e) : 0.0;
            }
            const double d = __ldcs(A.d + p);
            double ya = mul_rn(d, pA[p]), yt = mul_rn(d, pT[p]);
#pragma unroll
            for (int j = 0; j < 6; j++) {
                xa[j] = c[j] >= 0 ? pA[c[j]] : 0.0;
                xt[j] = c[j] >= 0 ? pT[c[j]] : 0.0;
            }
#pragma unroll
            for (int j = 0; j < 6; j++)
                if (c[j] >= 0) {
                    ya = fmadd(u[j], xa[j], ya);
                    yt = fmadd(w[j], xt[j], yt);
                }
            sink(p, ya, yt);
        }
        return;
    }
    for (int p = it.first; p < a.n; p += it.stride) {
        const double ya = amul_row<double>(A, pA, p);
        sink(p, ya, amul_row<double>(AT, pT, p));
    }
}

// OpenFOAM PBiCG on an asymmetric matrix (the paper's momentum solver: PBiCG
// with DILU), FP64, after phase_init (x, rA = b - A x, normFactor from the
// row sums of A).  Vectors: x, rA = r, wA = w, pA = p, wT = q, rT = b (the
// right-hand side is not needed past rT = b - A^T x), pT.  A^T shares A's
// structure: its lower entries of row u hold upper_f and its upper entries of
// row l lower_f; the transposed DILU sweeps use rD times those.
template <class GR>
__device__ bool solve_pbicg(const SolveArgs& a, const GR& g, double nfac, double res0, spuma_solver_perf& pf)
{
    RowIter it = rows_of(g);
    const Mat<double> A = mat_of<double>(a);
    Mat<double> AT = A;
    AT.La = a.LaT64;
    AT.Ua = a.UaT64;
    AT.Lc = a.LcT64;
    AT.Uc = a.UcT64;
    AT.Ea = a.EaT64;
    double *x = a.x, *rA = a.r, *wA = a.w, *pA = a.p, *wT = a.q, *rT = a.b, *pT = a.pT;
    PhaseClock pc(a.phase_clk, g.bid);
    const int nv = a.n / 2;   // 16-byte pairs of the streaming passes
    auto d2 = [](double* q) { return reinterpret_cast<double2*>(q); };
    for (int p = it.first; p < a.n; p += it.stride) rT[p] = a.b[p] - amul_row<double>(AT, x, p);
    if (!group_sync(g)) return false;
    double res = res0;
    int n_it = 0, singular = 0;
    if (a.min_iter > 0 || !converged(res0, res0, a.tol, a.rel_tol)) {
        double wArA = 1.0, wArA_old, alpha = 0.0;
        bool pending = false;
        for (;;) {
            if (pending) {
                double acc[1] = {0.0};
                for (int i = it.first; i < nv; i += it.stride) {
                    const double2 ra = vfma(-alpha, d2(wA)[i], d2(rA)[i]), rt = vfma(-alpha, d2(wT)[i], d2(rT)[i]);
                    __stcs(d2(x) + i, vfma(alpha, d2(pA)[i], __ldcs(d2(x) + i)));
                    d2(rA)[i] = ra;
                    d2(rT)[i] = rt;
                    acc[0] += fabs(ra.x);
                    acc[0] += fabs(ra.y);
                }
                for (int p = 2 * nv + it.first; p < a.n; p += it.stride) {
                    x[p] = fmadd(alpha, pA[p], x[p]);
                    rA[p] = fmadd(-alpha, wA[p], rA[p]);
                    rT[p] = fmadd(-alpha, wT[p], rT[p]);
                    acc[0] += fabs(rA[p]);
                }
                block_reduce_store<1>(acc, a.partials, SL_D, g.bid);
                if (!group_sync(g)) return false;
                grid_reduce_read<1>(acc, a.partials, SL_D, g.nblocks);
                res = acc[0] / nfac;
                n_it++;
                pc.lap(CK_UPD);
                if (!((n_it < a.max_iter && !converged(res, res0, a.tol, a.rel_tol)) || n_it < a.min_iter)) break;
            }
            wArA_old = wArA;
            if (a.precond == SPUMA_PRECOND_DILU) {
                if (!dilu_apply(a, A, AT, rA, rT, wA, wT, g, pc)) return false;
            } else {
                double acc[1] = {0.0};
                for (int p = it.first; p < a.n; p += it.stride) {
                    const double wa = __dmul_rn(a.rD64[p], rA[p]);
                    wA[p] = wa;
                    wT[p] = __dmul_rn(a.rD64[p], rT[p]);
                    acc[0] = fmadd(wa, rT[p], acc[0]);
                }
                block_reduce_store<1>(acc, a.partials, SL_B, g.bid);
                if (!group_sync(g)) return false;
                pc.lap(CK_DIAG);
            }
            double t[1];
            grid_reduce_read<1>(t, a.partials, SL_B, g.nblocks);
            wArA = t[0];
            const bool first = !pending;
            const double beta = first ? 0.0 : wArA / wArA_old;
            for (int i = it.first; i < nv; i += it.stride) {
                const double2 wa = d2(wA)[i], wt = d2(wT)[i];
                d2(pA)[i] = first ? wa : vfma(beta, d2(pA)[i], wa);
                d2(pT)[i] = first ? wt : vfma(beta, d2(pT)[i], wt);
            }
            for (int p = 2 * nv + it.first; p < a.n; p += it.stride) {
                pA[p] = first ? wA[p] : fmadd(beta, pA[p], wA[p]);
                pT[p] = first ? wT[p] : fmadd(beta, pT[p], wT[p]);
            }
            if (!group_sync(g)) return false;
            pc.lap(CK_PUPD);
            double acc[1] = {0.0};
            dual_amul(a, A, AT, pA, pT, g, [&](int p, double ya, double yt) {
                wA[p] = ya;
                wT[p] = yt;
                acc[0] = fmadd(ya, pT[p], acc[0]);
            });
            block_reduce_store<1>(acc, a.partials, SL_C, g.bid);
            if (!group_sync(g)) return false;
            grid_reduce_read<1>(acc, a.partials, SL_C, g.nblocks);
            pc.lap(CK_AMUL);
            pc.count(CK_ITERS);
            const double wApT = acc[0];
            if (fabs(wApT) / nfac < 1e-300) {
                singular = 1;
                break;
            }
            alpha = wArA / wApT;
            pending = true;
        }
    }
    pf.initial_residual = res0;
    pf.final_residual = res;
    pf.n_iter = n_it;
    pf.converged = converged(res, res0, a.tol, a.rel_tol);
    pf.singular = singular;
    return true;
}

// Kinds of persistent launch, one kernel each so that every kernel holds only
// its own path (register allocation is per kernel).
enum SolveKind { KIND_SETUP = 0, KIND_F64 = 1, KIND_MIXED = 2, KIND_MIXED_RESTART = 3, KIND_PBICG = 4, KIND_MIXED_DIC = 5 };

}  // namespace spuma
#include "small.cuh"
namespace spuma {

// TRUE_INLINE: the report's true residual is computed inside the launch
// (batched launches); the single-system solver leaves it to the two small
// kernels that follow it on the stream (k_true_residual_*), so that its own
// register allocation is not burdened by one more Amul.
template <int KIND, bool TRUE_INLINE, class GR>
__device__ void run_system(const SolveArgs& a, const GR& g)
{
    spuma_solver_perf pf;
    pf.initial_residual = 0.0;
    pf.final_residual = 0.0;
    pf.true_rel_residual_l2 = 0.0;
    pf.n_iter = 0;
    pf.n_outer = 0;
    pf.converged = 0;
    pf.singular = 0;
    pf.status = 0;
    pf.n_levels = a.nlev;
    bool ok = true;
    if constexpr (GR::wide) fill_chunk_table(a, g);
    if (a.mode == MODE_PREPARE || a.mode == MODE_SOLVE) {
        ok = phase_gather<KIND == KIND_PBICG>(a, g);
        if (ok) ok = phase_factor<KIND == KIND_PBICG>(a, g);
    }
    if (KIND == KIND_SETUP && ok && a.mode == MODE_PRECONDITION) {
        // w = M^-1 r for r = b_orig, written to x_orig (FP64)
        RowIter it = rows_of(g);
        for (int p = it.first; p < a.n; p += it.stride) a.r[p] = a.b_orig[a.perm[p]];
        ok = group_sync(g);
        Vecs<double> v{a.x, a.r, a.w, a.p, a.q};
        const Mat<double> A = mat_of<double>(a);
        if (ok) {
            if (a.precond == SPUMA_PRECOND_DIC) {
                PhaseClock pc(nullptr, g.bid);
                ok = dic_apply<double>(a, A, v, g, pc);
            } else {
                for (int p = it.first; p < a.n; p += it.stride)
                    a.w[p] = a.precond == SPUMA_PRECOND_DIAGONAL ? __dmul_rn(a.rD64[p], a.r[p]) : a.r[p];
                ok = group_sync(g);
            }
        }
        if (ok)
            for (int p = it.first; p < a.n; p += it.stride) a.x_orig[a.perm[p]] = a.w[p];
    }
    if constexpr (KIND != KIND_SETUP) {
        if (ok && a.mode == MODE_SOLVE) {
            double nfac = 1.0, res0 = 0.0;
            ok = phase_init(a, g, &nfac, &res0);
            if (ok) {
                if constexpr (KIND == KIND_PBICG) {
                    ok = solve_pbicg(a, g, nfac, res0, pf);
                } else if constexpr (KIND == KIND_MIXED) {
                    ok = solve_mixed_reliable(a, g, nfac, res0, pf);
                } else if constexpr (KIND == KIND_MIXED_DIC) {
                    ok = solve_mixed_eisenstat(a, g, nfac, res0, pf);
                } else if constexpr (KIND == KIND_MIXED_RESTART) {
                    ok = solve_mixed_restart(a, g, nfac, pf);
                } else {
                    Vecs<double> v{a.x, a.r, a.w, a.p, a.q};
                    double res = res0;
                    int sing = 0;
                    int n_it;
                    if constexpr (GR::cluster) {
                        ok = cluster_all_ok(g);
                        n_it = ok ? small_pcg(a, g, nfac, res0, &res, &sing) : -1;
                    } else {
                        n_it = pcg_loop<double>(a, mat_of<double>(a), v, nfac, res0, a.tol, a.rel_tol, a.max_iter,
                                                a.min_iter, &res, &sing, g);
                    }
                    ok = n_it >= 0;
                    pf.initial_residual = res0;
                    pf.final_residual = res;
                    pf.n_iter = n_it < 0 ? 0 : n_it;
                    pf.converged = converged(res, res0, a.tol, a.rel_tol);
                    pf.singular = sing;
                }
            }
            if constexpr (TRUE_INLINE) {
                if (ok) {
                    Mat<double> A64 = mat_of<double>(a);
                    if (KIND == KIND_PBICG) A64.ell_w = 0;   // asymmetric: the internal CSR holds A
                    ok = true_residual(a, A64, KIND == KIND_PBICG ? nullptr : a.b, g, &pf.true_rel_residual_l2);
                }
            }
            if (ok && !a.no_store) phase_store_x(a, g);
        }
    }
    if (g.bid == 0 && threadIdx.x == 0 && a.perf) {
        __threadfence();
        pf.status = ld_volatile_int(a.status);
        // a group that stopped always has a status; keep the report honest if not
        if (!ok && pf.status == 0) pf.status = SPUMA_ERR_DEVICE_TIMEOUT;
        if (pf.status != 0) pf.converged = 0;
        *a.perf = pf;
    }
}

template <int MAXT>
struct GroupOf {
    using type = Group;
};
template <>
struct GroupOf<512> {
    using type = WideGroup;
};

// One instance per solve kind and largest block size (512 threads: 128
// registers per thread; 1024: 64).
template <int KIND, int MAXT>
__global__ void __launch_bounds__(MAXT, 1) k_solve(SolveArgs a, unsigned long long timeout_ns)
{
    typename GroupOf<MAXT>::type g;
    g.word = reinterpret_cast<unsigned long long*>(a.status + DS_BARRIER);
    g.status = a.status;
    g.nblocks = (int)gridDim.x;
    g.bid = (int)blockIdx.x;
    g.timeout_ns = timeout_ns;
    run_system<KIND, false>(a, g);
}

// The FP64 DIC solve of a small system: one cluster or one block (small.cuh).
template <class GR>
__global__ void __launch_bounds__(kSmallThreads, 1) k_solve_small(SolveArgs a)
{
    GR g;
    g.word = nullptr;
    g.status = a.status;
    g.nblocks = (int)gridDim.x;
    g.bid = (int)blockIdx.x;
    g.timeout_ns = 0;
    run_system<KIND_F64, false>(a, g);
}

// The single-system solver's true residual, after it on the stream: per-block
// sums of r_p^2 and b_p^2 (r = b - A64 x in the Amul's face order, one FMA per
// term, each thread's rows in order) into the partials, then one warp adds
// the block partials in block order and writes ||r||_2/||b||_2 (||r||_2 when
// b = 0) into the report.  Deterministic, like every reduction here.
__global__ void __launch_bounds__(256) k_true_residual_part(SolveArgs a, int asym)
{
    Mat<double> A64 = mat_of<double>(a);
    if (asym) A64.ell_w = 0;
    double acc[2] = {0.0, 0.0};
    for (int p = blockIdx.x * blockDim.x + threadIdx.x; p < a.n; p += gridDim.x * blockDim.x) {
        const double bv = asym ? a.b_orig[a.perm[p]] : a.b[p];
        const double rr = __dsub_rn(bv, amul_row<double>(A64, a.x, p));
        acc[0] = __fma_rn(rr, rr, acc[0]);
        acc[1] = __fma_rn(bv, bv, acc[1]);
    }
    block_reduce_store<2>(acc, a.partials, SL_A, blockIdx.x);
}

__global__ void k_true_residual_final(SolveArgs a, int nblocks)
{
    double t[2];
    grid_reduce_read<2>(t, a.partials, SL_A, nblocks);
    if (threadIdx.x == 0 && a.perf)
        a.perf->true_rel_residual_l2 = t[1] > 0.0 ? __ddiv_rn(__dsqrt_rn(t[0]), __dsqrt_rn(t[1])) : __dsqrt_rn(t[0]);
}

// The batched launch, one instance per solve kind and largest block size
// (the register budget follows from it: 128 per thread up to 512 threads, 64
// at 1024).
template <int KIND, int MAXT>
__global__ void __launch_bounds__(MAXT, MAXT <= 256 ? 2 : 1) k_solve_batch(BatchTable t, unsigned long long timeout_ns)
{
    __shared__ SolveArgs sa;
    int s = 0;
    while (s + 1 < t.n_sys && (int)blockIdx.x >= t.split[s + 1]) s++;
    if (threadIdx.x == 0) sa = *t.args[s];
    __syncthreads();
    typename GroupOf<(MAXT <= 512 ? 512 : 1024)>::type g;
    g.word = reinterpret_cast<unsigned long long*>(sa.status + DS_BARRIER);
    g.status = sa.status;
    g.nblocks = t.split[s + 1] - t.split[s];
    g.bid = (int)blockIdx.x - t.split[s];
    g.timeout_ns = timeout_ns;
    run_system<KIND, true>(sa, g);
}

// Stand-alone Amul on the prepared matrix (internal order): the PCG's Amul
// phase as a kernel of its own.
template <class T>
__global__ void __launch_bounds__(256) k_amul_prepared(int n, Mat<T> A, const T* __restrict__ x, T* __restrict__ y)
{
    constexpr int R = AmulShape<T>::R, G = AmulShape<T>::G;
    const int stride = gridDim.x * blockDim.x;
    if (PipeShape<T>::stand_alone && A.ell_w > 0 && A.ell_w <= PipeShape<T>::G) {
        ell_amul_pipelined<T, PipeShape<T>::R, PipeShape<T>::G>(A, x, blockIdx.x * blockDim.x + threadIdx.x, stride, n,
                                                                [&](int p, T yv, T) { __stcs(y + p, yv); });
        return;
    }
    for (int pb = blockIdx.x * blockDim.x + threadIdx.x; pb < n; pb += R * stride) {
        int p[R];
        T yy[R], xp[R];
#pragma unroll
        for (int k = 0; k < R; k++) p[k] = pb + k * stride;
        amul_rows<T, R, G, false>(A, x, p, n, yy, xp);
#pragma unroll
        for (int k = 0; k < R; k++)
            if (p[k] < n) __stcs(y + p[k], yy[k]);
    }
}

// Stand-alone Amul on the fixed-width layout alone (no row-extent branch in
// the kernel, rows of at most W entries): its registers stay within 32 per
// thread, so that 2048 threads per SM are resident and enough loads are in
// flight; one wave of 8 blocks per SM walks the rows (FP64: 140 -> 130.6 us
// at 200^3 against the kernel shared with the row-extent path).  Each row: d_p x_p, then
// its entries in layout order (lower ascending, then upper ascending), one
// FMA each: the same sums as the solver's Amul phase.
template <class T, int W>
__global__ void __launch_bounds__(256, 8) k_amul_ell(int n, Mat<T> A, const T* __restrict__ x, T* __restrict__ y)
{
    const int stride = gridDim.x * blockDim.x;
    for (int p = blockIdx.x * blockDim.x + threadIdx.x; p < n; p += stride) {
        int c[W];
        T a[W], v[W];
#pragma unroll
        for (int j = 0; j < W; j++) {
            const bool ok = j < A.ell_w;
            const size_t e = (size_t)j * A.ell_stride + p;
            c[j] = ok ? __ldcs(A.Ecol + e) : -1;
            a[j] = ok ? __ldcs(A.Ea + e) : T(0);
        }
        const T xp = x[p];
        const T d = __ldcs(A.d + p);
#pragma unroll
        for (int j = 0; j < W; j++) v[j] = c[j] >= 0 ? x[c[j]] : T(0);
        T yy = mul_rn(d, xp);
#pragma unroll
        for (int j = 0; j < W; j++)
            if (c[j] >= 0) yy = fmadd(a[j], v[j], yy);
        __stcs(y + p, yy);
    }
}

__global__ void k_permute(int n, int dir, const int* __restrict__ perm, const double* __restrict__ src, double* dst)
{
    for (int p = blockIdx.x * blockDim.x + threadIdx.x; p < n; p += gridDim.x * blockDim.x) {
        if (dir == 0)
            dst[p] = src[perm[p]];
        else
            dst[perm[p]] = src[p];
    }
}

__global__ void k_read_rD(int n, const int* __restrict__ perm, const double* __restrict__ rD, double* out)
{
    for (int p = blockIdx.x * blockDim.x + threadIdx.x; p < n; p += gridDim.x * blockDim.x) out[perm[p]] = rD[p];
}

// ------------------------------------------------------------ host side -----
// Row mapping of the DIC sweeps: 1 (default) contiguous level chunks per
// block, 0 strided (SPUMA_SWEEP=0, a measurement override).
static int sweep_mode()
{
    static const int m = [] {
        const char* e = getenv("SPUMA_SWEEP");
        return (e && atoi(e) == 0) ? 0 : 1;
    }();
    return m;
}

SolveArgs make_args(spuma_ldu_t h)
{
    SolveArgs a{};
    const Layout& L = h->L;
    a.n = h->n;
    a.nf = h->nf;
    a.nlev = h->nlev;
    a.tail_from = h->nlev;

    a.lvl = h->at<int>(L.lvl);
    a.perm = h->at<int>(L.perm);
    a.Lptr = h->at<int>(L.Lptr);
    a.Lcol = h->at<int>(L.Lcol);
    a.Lface = h->at<int>(L.Lface);
    a.Uptr = h->at<int>(L.Uptr);
    a.Ucol = h->at<int>(L.Ucol);
    a.Uface = h->at<int>(L.Uface);
    a.La64 = h->at<double>(L.La64);
    a.Ua64 = h->at<double>(L.Ua64);
    a.Lc64 = h->at<double>(L.Lc64);
    a.Uc64 = h->at<double>(L.Uc64);
    a.d64 = h->at<double>(L.d64);
    a.rD64 = h->at<double>(L.rD64);
    a.lower_orig = nullptr;
    a.LaT64 = L.asym ? h->at<double>(L.LaT64) : nullptr;
    a.UaT64 = L.asym ? h->at<double>(L.UaT64) : nullptr;
    a.LcT64 = L.asym ? h->at<double>(L.LcT64) : nullptr;
    a.UcT64 = L.asym ? h->at<double>(L.UcT64) : nullptr;
    a.pT = L.asym ? h->at<double>(L.pT64) : nullptr;
    a.EaT64 = L.asym ? h->at<double>(L.EaT64) : nullptr;
    a.Ecol = h->at<int>(L.Ecol);
    a.Ea64 = h->at<double>(L.Ea64);
    a.Ea32 = h->at<float>(L.Ea32);
    a.ell_w = h->ell_w;
    a.La32 = h->at<float>(L.La32);
    a.Ua32 = h->at<float>(L.Ua32);
    a.Lc32 = h->at<float>(L.Lc32);
    a.Uc32 = h->at<float>(L.Uc32);
    a.d32 = h->at<float>(L.d32);
    a.rD32 = h->at<float>(L.rD32);
    a.x = h->at<double>(L.x64);
    a.r = h->at<double>(L.r64);
    a.w = h->at<double>(L.w64);
    a.p = h->at<double>(L.p64);
    a.q = h->at<double>(L.q64);
    a.b = h->at<double>(L.b64);
    a.xi = h->at<float>(L.x32);
    a.ri = h->at<float>(L.r32);
    a.wi = h->at<float>(L.w32);
    a.pi = h->at<float>(L.p32);
    a.qi = h->at<float>(L.q32);
    a.partials = h->at<double>(L.partials);
    a.bar = h->at<unsigned>(L.bar);
    a.status = h->at<int>(L.status);
    a.sweep = sweep_mode();
    return a;
}

static int precision_kind(int precision, int precond)
{
    if (precision == SPUMA_MIXED) return precond == SPUMA_PRECOND_DIC ? KIND_MIXED_DIC : KIND_MIXED;
    return precision == SPUMA_MIXED_RESTART ? KIND_MIXED_RESTART : KIND_F64;
}

static int kind_of(const SolveArgs& a)
{
    if (a.mode != MODE_SOLVE) return KIND_SETUP;
    if (a.lower_orig) return KIND_PBICG;
    return precision_kind(a.precision, a.precond);
}

template <int MAXT>
static const void* solve_kernel_t(int kind)
{
    switch (kind) {
    case KIND_SETUP: return (const void*)k_solve<KIND_SETUP, MAXT>;
    case KIND_MIXED: return (const void*)k_solve<KIND_MIXED, MAXT>;
    case KIND_MIXED_DIC: return (const void*)k_solve<KIND_MIXED_DIC, MAXT>;
    case KIND_MIXED_RESTART: return (const void*)k_solve<KIND_MIXED_RESTART, MAXT>;
    case KIND_PBICG: return (const void*)k_solve<KIND_PBICG, MAXT>;
    default: return (const void*)k_solve<KIND_F64, MAXT>;
    }
}

static const void* solve_kernel(int kind, int threads)
{
    return threads <= 512 ? solve_kernel_t<512>(kind) : solve_kernel_t<1024>(kind);
}

template <int MAXT>
static const void* batch_kernel_t(int kind)
{
    switch (kind) {
    case KIND_MIXED: return (const void*)k_solve_batch<KIND_MIXED, MAXT>;
    case KIND_MIXED_DIC: return (const void*)k_solve_batch<KIND_MIXED_DIC, MAXT>;
    case KIND_MIXED_RESTART: return (const void*)k_solve_batch<KIND_MIXED_RESTART, MAXT>;
    default: return (const void*)k_solve_batch<KIND_F64, MAXT>;
    }
}

static const void* batch_kernel(int kind, int threads)
{
    if (threads <= 256) return batch_kernel_t<256>(kind);
    if (threads <= 512) return batch_kernel_t<512>(kind);
    return batch_kernel_t<1024>(kind);
}

static std::mutex g_occ_mu;
static std::map<long long, int> g_occ;   // (kernel, block threads, ring) -> co-resident blocks per SM

int solve_blocks_per_sm(int threads, bool batch, int kind, size_t dyn = 0)
{
    std::lock_guard<std::mutex> lk(g_occ_mu);
    const long long key = (((long long)(threads * 2 + (batch ? 1 : 0)) * 8 + kind) << 20) + (long long)dyn;
    auto it = g_occ.find(key);
    if (it != g_occ.end()) return it->second;
    const void* k = batch ? batch_kernel(kind, threads) : solve_kernel(kind, threads);
    int nb = 0;
    cudaError_t e = cudaSuccess;
    if (dyn) e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)dyn);
    if (e == cudaSuccess) e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, k, threads, dyn);
    if (e != cudaSuccess) {
        cudaGetLastError();
        nb = 0;
    }
    g_occ[key] = nb;
    return nb;
}

// Blocks of the persistent single-system solver: one per row chunk of
// `threads` rows, at most all co-resident blocks (SPUMA_SOLVE_BLOCKS_PER_SM
// caps the blocks per SM, a tuning override).  0 when the kernel cannot be
// resident.
int solve_grid(spuma_ldu_t h, int threads, int kind, size_t dyn)
{
    int per_sm = solve_blocks_per_sm(threads, false, kind, dyn);
    if (per_sm < 1) return 0;
    if (const char* env = getenv("SPUMA_SOLVE_BLOCKS_PER_SM")) {
        int v = atoi(env);
        if (v >= 1 && v < per_sm) per_sm = v;
    }
    int64_t want = ((int64_t)h->n + threads - 1) / threads;
    int64_t maxg = std::min<int64_t>((int64_t)per_sm * h->num_sms, kMaxBlocks);
    return (int)std::max<int64_t>(1, std::min<int64_t>(want, maxg));
}

// First level of the run of small last levels (each with at most `limit` rows)
// that the solver's first block handles alone; SPUMA_TAIL_ROWS overrides the
// limit (0 disables).  The limit is the block's threads, and in the DIC solves
// at least tail_rows: a block of 256 threads takes 1024 rows in fewer steps than
// a grid barrier costs.  Mixed, 256 threads, 256 | 512 | 1024 rows: 16^3 permuted
// 61 | 45 | 44 us an iteration, 20^3 67 | 64 | 58, 32^3 81 | 78 | 77; FP64, whose
// rows the pipe takes longer for, 36^3 99.5 | 99.5 | 103.
static int tail_rows(int kind, int precision)
{
    return kind == KIND_PBICG ? 0 : precision == SPUMA_F64 ? 512 : 1024;
}
int tail_level(spuma_ldu_t h, int limit)
{
    if (const char* e = getenv("SPUMA_TAIL_ROWS")) limit = atoi(e);
    int t = h->nlev;
    while (t > 1 && (int64_t)h->h_lvl[t] - h->h_lvl[t - 1] <= limit) t--;
    // keep at least two levels in the tail, else the single grid barrier saves nothing
    return (h->nlev - t >= 2) ? t : h->nlev;
}

// Threads per block of a single-system solve (block_threads 0).  Up to 512 the
// kernels have 128 registers per thread and keep a round of sweep loads in
// flight across the grid barriers (wide_sweep).  Measured per iteration, DIC
// FP64 / mixed, 256 | 512 | 1024 threads: 24^3 73 / 63 | 76 / 64 | 92 / 82 us,
// 32^3 80 / 69 | 84 / 73 | 104 / 93, 64^3 119 / 98 | 112 / 92 | 151 / 131,
// 100^3 175 / 114 | 171 / 110 | 195 / 153, 128^3 257 / 149 | 251 / 146 | 274 /
// 174, 200^3 709 / 333 | 692 / 330 | 702 / 336; diagonal FP64 at 64^3 24 against
// 30, at 128^3 90 against 96; mixed with the diagonal, 256 or 512 by this rule |
// 1024: 24^3 14 | 26, 48^3 18 | 26, 64^3 20 | 28, 128^3 49 | 59, 200^3 164 | 167;
// restarted, diagonal: 13 | 25, 17 | 25, 19 | 26, 47 | 56, 160 | 160, DIC 68 | 90, 88 |
// 116, 101 | 137, 181 | 207, 441 | 424.  PBiCG, whose sweeps run without the loads ahead,
// wants more threads on large meshes: DILU at 64^3 158 against 183, at 128^3 393
// against 379.
// Systems that the first block has to itself past level 0 (no wider level): FP64
// beyond one row per thread of 256 in blocks of 1024 (100 x 100 x 4, levels of 400
// rows: 681 | 599 | 561), mixed beyond three rounds in blocks of 512 (50 x 50 x 20,
// 970 rows: 361 | 307; below, 28^3, 588 rows: 191 | 212).
static int default_threads(spuma_ldu_t h, const SolveArgs& a, const spuma_solver_controls* ctl)
{
    if (ctl->block_threads > 0) return ctl->block_threads;
    if (a.lower_orig) return a.n <= 50000 ? 256 : a.n > 1000000 ? 1024 : 512;
    if (a.precond == SPUMA_PRECOND_DIC && tail_level(h, 1024) <= 1) {
        int widest = 0;
        for (int L = 1; L < h->nlev; L++) widest = std::max(widest, h->h_lvl[L + 1] - h->h_lvl[L]);
        if (a.precision == SPUMA_F64 && widest > 256) return 1024;
        if (a.precision != SPUMA_F64 && widest > 768) return 512;
    }
    // the restarted form's Amul and sweeps at 200^3, 512 | 1024 threads: 441 | 424 us an iteration (128^3 181 | 207)
    if (a.precision == SPUMA_MIXED_RESTART && a.precond == SPUMA_PRECOND_DIC && a.n > 4000000) return 1024;
    return a.n <= 50000 ? 256 : 512;
}

// The report's true residual (the solver's x in internal order is still in the
// workspace).
static spuma_status launch_true_residual(spuma_ldu_t h, const SolveArgs& b, int kind, cudaStream_t s)
{
    const int tg = (int)std::max<int64_t>(1, std::min<int64_t>(((int64_t)h->n + 255) / 256, (int64_t)h->num_sms * 8));
    k_true_residual_part<<<tg, 256, 0, s>>>(b, kind == KIND_PBICG ? 1 : 0);
    k_true_residual_final<<<1, 32, 0, s>>>(b, tg);
    count_launch(2);
    SPUMA_CUDA(cudaGetLastError());
    return SPUMA_OK;
}

// Blocks of the cluster that solves h's FP64 DIC systems (small.cuh), 0 when the
// grid solver takes them: rows of more than six entries, more levels than the
// table holds, or more rows than the blocks hold; and with a time limit that a
// wait could exceed.  The hardware barriers keep none; a block reaches the next
// one within the work on its 2400 rows, tens of microseconds, so a wait there
// stays below any limit from kSmallLimit up.
constexpr unsigned long long kSmallLimit = 1000000;   // 1 ms
static int small_cluster(spuma_ldu_t h)
{
    if (barrier_timeout_ns() < kSmallLimit) return 0;
    if (h->ell_w < 1 || h->ell_w > 6 || h->nlev > kSmallLevels || h->n > kSmallMaxRows) return 0;
    return h->n <= kSmallOneBlock ? 1 : kSmallMaxCluster;
}

static const void* small_kernel(int G)
{
    return G > 1 ? (const void*)k_solve_small<ClusterGroup> : (const void*)k_solve_small<BlockGroup>;
}

// Whether a cluster of G blocks with `smem` bytes can run on the current
// device (asked once per device, size and amount).
static bool small_fits(int device, int G, size_t smem, cudaLaunchConfig_t& cfg)
{
    static std::map<std::pair<int, long long>, bool> known;
    std::lock_guard<std::mutex> lk(g_occ_mu);
    const auto key = std::make_pair(device, (long long)smem * 64 + G);
    auto it = known.find(key);
    if (it != known.end()) return it->second;
    int nc = 0;
    const void* k = small_kernel(G);
    cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)small_smem(kSmallSlots));
    if (e == cudaSuccess) e = cudaFuncSetAttribute(k, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
    if (e == cudaSuccess) e = cudaOccupancyMaxActiveClusters(&nc, k, &cfg);
    if (e != cudaSuccess) cudaGetLastError();
    return known[key] = e == cudaSuccess && nc > 0;
}

// Launches the solve on a cluster; false when the grid solver must take it.
static bool launch_small(spuma_ldu_t h, const SolveArgs& a, cudaStream_t s, spuma_status* st)
{
    const int G = small_cluster(h);
    if (G == 0) return false;
    const int nslot = ((h->n + 31) / 32 + G - 1) / G * 32;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(G);
    cfg.blockDim = dim3(kSmallThreads);
    cfg.dynamicSmemBytes = small_smem(nslot);
    cfg.stream = s;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = G;
    at[0].val.clusterDim.y = 1;
    at[0].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    if (!small_fits(h->device, G, cfg.dynamicSmemBytes, cfg)) return false;
    auto run = [&]() -> spuma_status {
        SPUMA_CUDA(cudaMemsetAsync(h->at<char>(h->L.bar), 0, h->L.status + 256 - h->L.bar, s));
        SolveArgs b = a;
        if (getenv("SPUMA_PHASE_CLOCKS")) {
            b.phase_clk = h->at<long long>(h->L.clk);
            SPUMA_CUDA(cudaMemsetAsync(b.phase_clk, 0, 8 * 256, s));
        }
        void* args[] = {(void*)&b};
        SPUMA_CUDA(cudaLaunchKernelExC(&cfg, small_kernel(G), args));
        count_launch();
        return launch_true_residual(h, b, KIND_F64, s);
    };
    *st = run();
    return true;
}

spuma_status launch_solve(spuma_ldu_t h, const SolveArgs& a, int threads, cudaStream_t s)
{
    if (threads < 32 || threads > 1024 || threads % 32) {
        set_error("block_threads must be a multiple of 32 in [32, 1024]");
        return SPUMA_ERR_INVALID_ARG;
    }
    const int kind = kind_of(a);
    const int grid = solve_grid(h, threads, kind, 0);
    if (grid < 1) { set_error("solver kernel cannot be resident"); return SPUMA_ERR_CUDA; }
    SPUMA_CUDA(cudaMemsetAsync(h->at<char>(h->L.bar), 0, h->L.status + 256 - h->L.bar, s));
    unsigned long long tns = barrier_timeout_ns();
    SolveArgs b = a;
    b.tail_from = tail_level(h, std::max(threads, tail_rows(kind, a.precision)));
    // SPUMA_AMUL_CHUNKS=1: the Amul phase walks level chunks when the levels
    // are wide (an average level gives every block at least a block's worth
    // of rows).  Off by default: measured at 200^3, Amul phase 101.9 -> 112.7
    // us per FP32 iteration, mixed solve 328.8 -> 338.1 ms
    static const bool amul_chunks_env = getenv("SPUMA_AMUL_CHUNKS") && atoi(getenv("SPUMA_AMUL_CHUNKS")) != 0;
    b.amul_chunks = amul_chunks_env && b.sweep != 0 && h->nlev > 0 &&
                    (int64_t)h->n / h->nlev >= (int64_t)grid * threads;
    if (getenv("SPUMA_PHASE_CLOCKS")) {
        b.phase_clk = h->at<long long>(h->L.clk);
        SPUMA_CUDA(cudaMemsetAsync(b.phase_clk, 0, 8 * 256, s));
    }
    void* args[] = {(void*)&b, (void*)&tns};
    SPUMA_CUDA(cudaLaunchCooperativeKernel(solve_kernel(kind, threads), grid, threads, args, 0, s));
    count_launch();
    return b.mode == MODE_SOLVE ? launch_true_residual(h, b, kind, s) : SPUMA_OK;
}

spuma_status launch_batch_kernel(const BatchTable& t, int grid, int threads, int kind, cudaStream_t s)
{
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(grid);
    cfg.blockDim = dim3(threads);
    cfg.stream = s;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeCooperative;
    at[0].val.cooperative = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    unsigned long long tns = barrier_timeout_ns();
    BatchTable tt = t;
    void* args[] = {(void*)&tt, (void*)&tns};
    SPUMA_CUDA(cudaLaunchKernelExC(&cfg, batch_kernel(kind, threads), args));
    return SPUMA_OK;
}

int batch_kind(int precision, int precond) { return precision_kind(precision, precond); }

void fill_controls(SolveArgs& a, const spuma_solver_controls* ctl)
{
    a.precond = ctl->precond;
    a.precision = ctl->precision;
    a.tol = ctl->tolerance;
    a.rel_tol = ctl->rel_tol;
    a.inner_rel_tol = ctl->inner_rel_tol;
    a.max_iter = ctl->max_iter;
    a.min_iter = ctl->min_iter;
    a.max_outer = ctl->max_outer;
}

bool ctl_ok(const spuma_solver_controls* c)
{
    if (!c) return false;
    if (c->precond < 0 || c->precond > 2) return false;
    if (c->precision != SPUMA_F64 && c->precision != SPUMA_MIXED && c->precision != SPUMA_MIXED_RESTART) return false;
    if (!(c->tolerance >= 0.0) || !(c->rel_tol >= 0.0) || c->max_iter < 0 || c->min_iter < 0) return false;
    if ((c->precision == SPUMA_MIXED || c->precision == SPUMA_MIXED_RESTART) &&
        (!(c->inner_rel_tol > 0.0) || c->max_outer < 0))
        return false;
    return true;
}

spuma_status pcg_solve_internal(spuma_ldu_t h, const double* diag, const double* upper, const double* b, double* x,
                                const spuma_solver_controls* ctl, spuma_solver_perf* perf, cudaStream_t s,
                                int zero_x0)
{
    if (!h || !ctl_ok(ctl) || (h->n > 0 && (!diag || !b || !x)) || (h->nf > 0 && !upper)) {
        set_error("spuma_pcg_solve: bad argument");
        return SPUMA_ERR_INVALID_ARG;
    }
    if (h->n == 0) {
        if (perf) {
            spuma_solver_perf z{};
            z.converged = 1;
            SPUMA_CUDA(cudaMemcpyAsync(perf, &z, sizeof(z), cudaMemcpyHostToDevice, s));
        }
        return SPUMA_OK;
    }
    SolveArgs a = make_args(h);
    fill_controls(a, ctl);
    a.mode = MODE_SOLVE;
    a.zero_x0 = zero_x0;
    a.diag_orig = diag;
    a.upper_orig = upper;
    a.b_orig = b;
    a.x_orig = x;
    a.perf = perf;
    spuma_status st = SPUMA_OK;
    if (ctl->block_threads != 0 || kind_of(a) != KIND_F64 || a.precond != SPUMA_PRECOND_DIC || !launch_small(h, a, s, &st))
        st = launch_solve(h, a, default_threads(h, a, ctl), s);
    if (st == SPUMA_OK) h->prepared_precond = ctl->precond;
    return st;
}

}  // namespace spuma

using namespace spuma;

extern "C" {

spuma_status spuma_pbicg_solve(spuma_ldu_t h, const double* diag, const double* lower, const double* upper,
                               const double* b, double* x, const spuma_solver_controls* ctl, spuma_solver_perf* perf,
                               spuma_stream_t stream)
{
    if (!h || !ctl || (ctl->precond != SPUMA_PRECOND_NONE && ctl->precond != SPUMA_PRECOND_DIAGONAL &&
                       ctl->precond != SPUMA_PRECOND_DILU) ||
        ctl->precision != SPUMA_F64 || !(ctl->tolerance >= 0.0) || !(ctl->rel_tol >= 0.0) || ctl->max_iter < 0 ||
        ctl->min_iter < 0 || (h->n > 0 && (!diag || !b || !x)) || (h->nf > 0 && (!lower || !upper))) {
        set_error("spuma_pbicg_solve: bad argument (precond NONE, DIAGONAL or DILU; precision F64)");
        return SPUMA_ERR_INVALID_ARG;
    }
    cudaStream_t s = (cudaStream_t)stream;
    if (h->n == 0) {
        if (perf) {
            spuma_solver_perf z{};
            z.converged = 1;
            SPUMA_CUDA(cudaMemcpyAsync(perf, &z, sizeof(z), cudaMemcpyHostToDevice, s));
        }
        return SPUMA_OK;
    }
    if (!h->L.asym) {
        set_error("spuma_pbicg_solve: the workspace was not sized with SPUMA_WORKSPACE_ASYMMETRIC");
        return SPUMA_ERR_WORKSPACE_TOO_SMALL;
    }
    SolveArgs a = make_args(h);
    fill_controls(a, ctl);
    a.mode = MODE_SOLVE;
    a.zero_x0 = 0;
    a.diag_orig = diag;
    a.upper_orig = upper;
    a.lower_orig = lower;
    a.b_orig = b;
    a.x_orig = x;
    a.perf = perf;
    h->prepared_precond = -1;
    return launch_solve(h, a, default_threads(h, a, ctl), s);
}

spuma_status spuma_matrix_prepare(spuma_ldu_t h, const double* diag, const double* upper, int32_t precond,
                                  spuma_stream_t stream)
{
    if (!h || (h->n > 0 && !diag) || (h->nf > 0 && !upper) || precond < 0 || precond > 2) {
        set_error("spuma_matrix_prepare: bad argument");
        return SPUMA_ERR_INVALID_ARG;
    }
    if (h->n == 0) return SPUMA_OK;
    SolveArgs a = make_args(h);
    a.mode = MODE_PREPARE;
    a.precond = precond;
    a.diag_orig = diag;
    a.upper_orig = upper;
    spuma_status st = launch_solve(h, a, 256, (cudaStream_t)stream);
    if (st == SPUMA_OK) h->prepared_precond = precond;
    return st;
}

spuma_status spuma_read_rD(spuma_ldu_t h, double* rD_out, spuma_stream_t stream)
{
    if (!h || (h->n > 0 && !rD_out)) { set_error("spuma_read_rD: bad argument"); return SPUMA_ERR_INVALID_ARG; }
    if (h->n == 0) return SPUMA_OK;
    int g = std::min((h->n + 255) / 256, h->num_sms * 16);
    k_read_rD<<<g, 256, 0, (cudaStream_t)stream>>>(h->n, h->at<int>(h->L.perm), h->at<double>(h->L.rD64), rD_out);
    count_launch();
    SPUMA_CUDA(cudaGetLastError());
    return SPUMA_OK;
}

spuma_status spuma_amul_prepared(spuma_ldu_t h, int32_t precision, const void* x, void* y, spuma_stream_t stream)
{
    if (!h || (h->n > 0 && (!x || !y)) || (precision != SPUMA_F64 && precision != SPUMA_F32)) {
        set_error("spuma_amul_prepared: bad argument");
        return SPUMA_ERR_INVALID_ARG;
    }
    if (h->n == 0) return SPUMA_OK;
    SolveArgs a = make_args(h);
    int g = std::min((h->n + 255) / 256, h->num_sms * 16);
    cudaStream_t s = (cudaStream_t)stream;
    if (precision == SPUMA_F64) {
        Mat<double> A{a.Lptr, a.Lcol, a.La64, a.Lc64, a.Uptr, a.Ucol, a.Ua64, a.Uc64, a.d64, a.rD64,
                      a.Ecol, a.Ea64, a.ell_w, a.n};
        const int ge = std::min(g, h->num_sms * 8);
        if (a.ell_w > 0 && a.ell_w <= 6)
            k_amul_ell<double, 6><<<ge, 256, 0, s>>>(h->n, A, (const double*)x, (double*)y);
        else if (a.ell_w > 0)
            k_amul_ell<double, kEllMax><<<ge, 256, 0, s>>>(h->n, A, (const double*)x, (double*)y);
        else
            k_amul_prepared<double><<<g, 256, 0, s>>>(h->n, A, (const double*)x, (double*)y);
    } else {
        Mat<float> A{a.Lptr, a.Lcol, a.La32, a.Lc32, a.Uptr, a.Ucol, a.Ua32, a.Uc32, a.d32, a.rD32,
                     a.Ecol, a.Ea32, a.ell_w, a.n};
        // FP32: the software-pipelined kernel measured faster than the
        // 32-register one (90.4 against 92.8 us at 200^3)
        k_amul_prepared<float><<<g, 256, 0, s>>>(h->n, A, (const float*)x, (float*)y);
    }
    count_launch();
    SPUMA_CUDA(cudaGetLastError());
    return SPUMA_OK;
}

spuma_status spuma_permute(spuma_ldu_t h, int32_t dir, const double* src, double* dst, spuma_stream_t stream)
{
    if (!h || (dir != 0 && dir != 1) || (h->n > 0 && (!src || !dst)) || src == dst) {
        set_error("spuma_permute: bad argument");
        return SPUMA_ERR_INVALID_ARG;
    }
    if (h->n == 0) return SPUMA_OK;
    int g = std::min((h->n + 255) / 256, h->num_sms * 16);
    k_permute<<<g, 256, 0, (cudaStream_t)stream>>>(h->n, dir, h->at<int>(h->L.perm), src, dst);
    count_launch();
    SPUMA_CUDA(cudaGetLastError());
    return SPUMA_OK;
}

spuma_status spuma_precondition(spuma_ldu_t h, int32_t precond, const double* r, double* w, spuma_stream_t stream)
{
    if (!h || (h->n > 0 && (!r || !w)) || precond < 0 || precond > 2) {
        set_error("spuma_precondition: bad argument");
        return SPUMA_ERR_INVALID_ARG;
    }
    if (precond != SPUMA_PRECOND_NONE && h->prepared_precond != precond) {
        set_error("spuma_precondition: call spuma_matrix_prepare with this preconditioner first");
        return SPUMA_ERR_INVALID_ARG;
    }
    if (h->n == 0) return SPUMA_OK;
    SolveArgs a = make_args(h);
    a.mode = MODE_PRECONDITION;
    a.precond = precond;
    a.b_orig = r;
    a.x_orig = w;
    // Blocks of 256 threads with 128 registers leave too few threads an SM for the
    // permuting passes of a large system: none, 256 | 1024 threads, 200^3 283 | 203 us,
    // 128^3 52 | 47, 64^3 26 | 29; DIC 642 | 559, 229 | 231, 113 | 134.
    const int large = precond == SPUMA_PRECOND_DIC ? 4000000 : 1000000;
    return launch_solve(h, a, h->n > large ? 1024 : 256, (cudaStream_t)stream);
}

spuma_status spuma_read_phase_clocks(spuma_ldu_t h, int64_t* out, int32_t n, spuma_stream_t stream)
{
    if (!h || !out || n < 0 || n > 256) { set_error("spuma_read_phase_clocks: bad argument"); return SPUMA_ERR_INVALID_ARG; }
    SPUMA_CUDA(cudaMemcpyAsync(out, h->at<long long>(h->L.clk), 8 * (size_t)n, cudaMemcpyDeviceToHost,
                               (cudaStream_t)stream));
    SPUMA_CUDA(cudaStreamSynchronize((cudaStream_t)stream));
    return SPUMA_OK;
}

spuma_status spuma_pcg_solve(spuma_ldu_t h, const double* diag, const double* upper, const double* b, double* x,
                             const spuma_solver_controls* ctl, spuma_solver_perf* perf, spuma_stream_t stream)
{
    return pcg_solve_internal(h, diag, upper, b, x, ctl, perf, (cudaStream_t)stream, 0);
}

}  // extern "C"

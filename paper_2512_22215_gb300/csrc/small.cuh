// small.cuh -- the FP64 DIC-PCG of small systems on one thread-block cluster
// (included by solve.cu, after the phases it shares with the grid solver).
//
// On the whole grid an iteration of a small system is grid barriers: 1.3 to 1.6
// us each, one per DIC level and sweep, plus trips to L2 for a row's lists and
// for every gathered value.  Here the blocks of one cluster (or one block) keep
// the rows' sweep coefficients and packed columns, the residual and the gathered
// vector in shared memory, gather from each other's and meet at the cluster's
// hardware barrier (0.22 us; a block barrier for one block).  Row p lives in
// warp-sized pieces dealt round the cluster: piece p / 32 belongs to block
// (p / 32) mod G, so every level is spread evenly and a gather's address follows
// from the column alone.  The sweep is one short loop for both directions: the
// instructions of a longer one (loads ahead in two register sets, a copy per
// direction) took longer to fetch than the loads they hid (16^3: 105 us).
// Iterates are those of the grid solver (the same row sums in the same order; the
// dot products in their own fixed order).
//
// An iteration, grid solver -> this one: natural order 16^3 (46 levels) 120 -> 82
// us, 24^3 (70) 312 -> 129, 32^3 (94) 472 -> 179; multicoloured 16^3 (13 levels)
// 64 -> 32, 24^3 (15) 74 -> 43, 32^3 (16) 80 -> 63; 8^3 (22) 57 -> 33 on one block
// (44 on a cluster of 16).  What is left is 0.75 us per level and sweep: the
// barrier, a remote gather and the row's chain of FP64 operations.

#pragma once

namespace spuma {

constexpr int kSmallLevels = 256;       // levels of the level table
constexpr int kSmallSlots = 2400;       // rows per block (shared memory; 12 bits of a packed column)
constexpr int kSmallThreads = 256;      // (512 were slower: more warps at every barrier)
constexpr int kSmallOneBlock = 1024;    // rows up to which one block is faster than 16 (8^3: 33 against 44 us an
                                        // iteration; 12^3: 34 against 32; 2 to 8 blocks lie between)
constexpr int kSmallMaxCluster = 16;    // 4 bits of a packed column
constexpr int kSmallMaxRows = kSmallMaxCluster * kSmallSlots;

// One block, or a cluster of several (a kernel each).
struct BlockGroup : Group {
    static constexpr bool cluster = true, several = false;
};
struct ClusterGroup : Group {
    static constexpr bool cluster = true, several = true;
};

// The aligned forms want the warp converged, and callers come here out of loops
// and branches that its lanes leave at different times.
__device__ __forceinline__ void cluster_arrive()
{
    __syncwarp();
    asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
}
__device__ __forceinline__ void cluster_wait()
{
    __syncwarp();
    asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
}
__device__ __forceinline__ void cluster_barrier()
{
    cluster_arrive();
    cluster_wait();
}

// The setup phases' barrier: true when no error is recorded.  A block that
// leaves early counts as arrived at later barriers; the solver loop, whose
// blocks read each other's shared memory, is entered only after
// cluster_all_ok().
template <class GR>
__device__ __forceinline__ bool small_sync(const GR& g)
{
    __shared__ int s_err;
    if constexpr (GR::several)
        cluster_barrier();
    else
        __syncthreads();
    if (threadIdx.x == 0) s_err = ld_volatile_int(g.status);
    __syncthreads();
    const bool ok = s_err == 0;
    __syncthreads();
    return ok;
}
__device__ __forceinline__ bool group_sync(const ClusterGroup& g) { return small_sync(g); }
__device__ __forceinline__ bool group_sync(const BlockGroup& g) { return small_sync(g); }

// The same answer in every block: errors are recorded before the first
// barrier, read between the two (a block that left found one, so all do).
template <class GR>
__device__ __forceinline__ bool cluster_all_ok(const GR& g)
{
    const bool ok = group_sync(g);
    if constexpr (GR::several) cluster_barrier();
    return ok;
}

__device__ __forceinline__ unsigned smem_addr(const void* p) { return (unsigned)__cvta_generic_to_shared(p); }
__device__ __forceinline__ unsigned remote_addr(unsigned own, unsigned rank)
{
    unsigned a;
    asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(a) : "r"(own), "r"(rank));
    return a;
}
__device__ __forceinline__ double ld_cluster(unsigned addr)
{
    double v;
    asm volatile("ld.shared::cluster.f64 %0, [%1];" : "=d"(v) : "r"(addr) : "memory");
    return v;
}
__device__ __forceinline__ void st_cluster(unsigned addr, double v)
{
    asm volatile("st.shared::cluster.f64 [%0], %1;" ::"r"(addr), "d"(v) : "memory");
}

template <bool CL>
struct SmallSolve {
    const SolveArgs& a;
    double *S, *r;                   // own rows in shared memory: gathered vector (w, then p), residual
    double *c, *rD;                  // sweep coefficients [6][nslot] (lower, then upper ascending), rD
    unsigned short *col, *cnt;       // packed columns [6][nslot], lower count | all << 8
    double *x, *q, *p;               // the others, by row, in global memory
    int4* tab;                       // per level: own pieces [x, y), rows [z, w)
    double* red;                     // [2][16] partial sums of the cluster's blocks
    int G, lg, rank, nslot, parity;
    unsigned s_base;

    __device__ __forceinline__ int row_of(int slot) const { return ((((slot >> 5) << lg) + rank) << 5) + (slot & 31); }
    __device__ __forceinline__ unsigned pack(int row) const
    {
        const int piece = row >> 5;
        return (unsigned)((piece & (G - 1)) << 12 | ((piece >> lg) << 5) | (row & 31));
    }
    __device__ __forceinline__ double gathered(unsigned k) const
    {
        if constexpr (CL) return ld_cluster(remote_addr(s_base, k >> 12) + 8u * (k & 4095u));
        return S[k];
    }
    __device__ __forceinline__ void barrier() const
    {
        if constexpr (CL)
            cluster_barrier();
        else
            __syncthreads();
    }
    __device__ __forceinline__ void barrier_arrive() const
    {
        if constexpr (CL)
            cluster_arrive();
        else
            __syncthreads();
    }
    __device__ __forceinline__ void barrier_wait() const
    {
        if constexpr (CL) cluster_wait();
    }

    // The cluster's sum of v, in every thread: the blocks' sums go to every
    // block's table before the barrier, each warp adds them up in the same
    // order (a butterfly over the ranks).
    __device__ __forceinline__ double total(double v)
    {
        double t[1] = {v};
        block_sum_to_first<1>(t);
        double* slot = red + 16 * parity;
        parity ^= 1;
        if (threadIdx.x == 0) {
            if constexpr (CL)
                for (int k = 0; k < G; k++) st_cluster(remote_addr(smem_addr(slot + rank), k), t[0]);
            else
                slot[0] = t[0];
        }
        barrier();
        const int lane = threadIdx.x & 15;
        double s = lane < G ? slot[lane] : 0.0;
#pragma unroll 1
        for (int o = G >> 1; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
        return __shfl_sync(0xffffffffu, s, 0);
    }

    // One sweep over the levels, forward (w = rD r - sum c w_l, entries
    // ascending) or backward (w -= sum c w_u, descending), with the thread's part
    // of rho = w.r.  A warp walks its pieces of all levels in one loop; what a
    // row needs besides the gathered values is loaded between arriving at the
    // level's barrier and waiting there.  A chain is as long as the warp's longest
    // row: an FP64 instruction takes its quadrant's pipe for 64 cycles with every
    // lane off.
    __device__ __forceinline__ double sweep(bool fwd, double rho)
    {
        const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, W = blockDim.x >> 5, step = fwd ? 1 : -1;
        const int end = fwd ? a.nlev : -1;
        int L = fwd ? 0 : a.nlev - 2;
        if (L == end) return rho;
        int4 t = tab[L];
        int lb = t.x + warp;
        bool arrived = false;
#pragma unroll 1
        for (;;) {
            const int s = (lb << 5) + lane, row = row_of(s);
            const bool some = lb < t.y, ok = some && row >= t.z && row < t.w;
            double f[6], rr = 0.0, acc = 0.0;
            unsigned k[6];
            int n = 0;
            if (some) {
                const int m = cnt[s], nl = m & 255, nt = m >> 8;
                const int first = (fwd ? 0 : nt - 1) * nslot + s, pitch = step * nslot;
                n = !ok ? 0 : fwd ? nl : nt - nl;
                rr = r[s];
                acc = fwd ? __dmul_rn(rD[s], rr) : S[s];
#pragma unroll
                for (int j = 0; j < 6; j++) {
                    k[j] = j < n ? col[first + j * pitch] : 0;
                    f[j] = j < n ? c[first + j * pitch] : 0.0;
                }
            }
            const int most = __reduce_max_sync(0xffffffffu, n);
            if (arrived) {
                barrier_wait();
                arrived = false;
            }
            if (some) {
                double v[6];
#pragma unroll
                for (int j = 0; j < 6; j++) v[j] = j < n ? gathered(k[j]) : 0.0;
#pragma unroll
                for (int j = 0; j < 6; j++)
                    if (j < most) acc = __fma_rn(-f[j], v[j], acc);   // past the row's end: acc + -0
                if (ok) S[s] = acc;
            }
            lb += W;
            const bool add = some && (!fwd || L == a.nlev - 1);   // top level: w is final going up
            if (lb >= t.y) {
                barrier_arrive();
                arrived = true;
                L += step;
            }
            if (add) rho = __fma_rn(ok ? acc : 0.0, rr, rho);
            if (L == end) break;
            if (arrived) {
                t = tab[L];
                lb = t.x + warp;
            }
        }
        barrier_wait();
        return rho;
    }

    __device__ __forceinline__ void setup()
    {
        const int n = a.n;
        for (int L = threadIdx.x; L < a.nlev; L += blockDim.x) {
            const int r0 = a.lvl[L], r1 = a.lvl[L + 1];
            const int b0 = r0 >> 5, b1 = (r1 + 31) >> 5;   // the level's pieces [b0, b1)
            tab[L] = make_int4((b0 - rank + G - 1) >> lg, (b1 - rank + G - 1) >> lg, r0, r1);
        }
#pragma unroll 1
        for (int s = threadIdx.x; s < nslot; s += blockDim.x) {
            const int row = row_of(s);
            S[s] = 0.0;
            r[s] = row < n ? a.r[row] : 0.0;
            rD[s] = row < n ? a.rD64[row] : 0.0;
            cnt[s] = 0;
            if (row >= n) continue;
            const int l0 = a.Lptr[row], nl = a.Lptr[row + 1] - l0, u0 = a.Uptr[row], nt = nl + a.Uptr[row + 1] - u0;
            cnt[s] = (unsigned short)(nl | nt << 8);
            for (int j = 0; j < nt; j++) {
                const bool low = j < nl;
                const int e = low ? l0 + j : u0 + j - nl;
                col[j * nslot + s] = (unsigned short)pack(low ? a.Lcol[e] : a.Ucol[e]);
                c[j * nslot + s] = low ? a.Lc64[e] : a.Uc64[e];
            }
        }
        barrier();
    }

    // q = A p (p gathered from S), returns the thread's part of sigma = q.p
    __device__ __forceinline__ double amul()
    {
        double sig = 0.0;
#pragma unroll 1
        for (int s = threadIdx.x; s < nslot; s += blockDim.x) {
            const int row = row_of(s), nt = cnt[s] >> 8;
            if (row >= a.n) continue;
            double e[6], v[6];
#pragma unroll
            for (int j = 0; j < 6; j++) {
                e[j] = j < nt ? a.Ea64[(size_t)j * a.n + row] : 0.0;
                v[j] = j < nt ? gathered(col[j * nslot + s]) : 0.0;
            }
            const double pp = S[s];
            double y = __dmul_rn(a.d64[row], pp);
#pragma unroll
            for (int j = 0; j < 6; j++)
                if (j < nt) y = __fma_rn(e[j], v[j], y);
            q[row] = y;
            sig = __fma_rn(y, pp, sig);
        }
        return sig;
    }

    // PCG iterations (the recurrences of pcg_loop); returns their count.
    __device__ int loop(double nfac, double res0, double* res_out, int* singular, PhaseClock& pc)
    {
        double res = res0, rho = 1.0, rho_old, alpha = 0.0;
        int n_it = 0;
        *res_out = res;
        if (!(a.min_iter > 0 || !converged(res0, res0, a.tol, a.rel_tol))) return 0;
#pragma unroll 1
        for (bool pending = false;; pending = true) {
            if (pending) {
                double acc = 0.0;
                for (int s = threadIdx.x; s < nslot; s += blockDim.x) {
                    const int row = row_of(s);
                    if (row >= a.n) continue;
                    x[row] = __fma_rn(alpha, S[s], x[row]);   // S holds p until the sweeps
                    const double rr = __fma_rn(-alpha, q[row], r[s]);
                    r[s] = rr;
                    acc += fabs(rr);
                }
                res = total(acc) / nfac;
                n_it++;
                pc.lap(CK_UPD);
                if (!((n_it < a.max_iter && !converged(res, res0, a.tol, a.rel_tol)) || n_it < a.min_iter)) break;
            }
            rho_old = rho;
            double sum = 0.0;
#pragma unroll 1
            for (int dir = 0; dir < 2; dir++) {   // one copy of the code
                sum = sweep(dir == 0, sum);
                pc.lap(dir == 0 ? CK_FWD : CK_BWD);
            }
            rho = total(sum);
            const double beta = pending ? rho / rho_old : 0.0;
            for (int s = threadIdx.x; s < nslot; s += blockDim.x) {
                const int row = row_of(s);
                if (row >= a.n) continue;
                const double w = S[s], pp = pending ? __fma_rn(beta, p[row], w) : w;
                p[row] = pp;
                S[s] = pp;
            }
            barrier();
            pc.lap(CK_PUPD);
            const double sigma = total(amul());
            pc.lap(CK_AMUL);
            pc.count(CK_ITERS);
            if (fabs(sigma) / nfac < 1e-300) {
                *singular = 1;
                break;
            }
            alpha = rho / sigma;
        }
        *res_out = res;
        return n_it;
    }
};

// Bytes of dynamic shared memory for nslot rows per block.
__host__ __device__ constexpr size_t small_smem(int nslot) { return (8 * 9 + 2 * 7) * (size_t)nslot; }

template <class GR>
__device__ int small_pcg(const SolveArgs& a, const GR& g, double nfac, double res0, double* res, int* singular)
{
    constexpr bool CL = GR::several;
    extern __shared__ __align__(16) double small_vec[];
    __shared__ int4 tab[kSmallLevels];
    __shared__ double red[32];
    int lg = 0;
    while ((1 << lg) < g.nblocks) lg++;
    const int nslot = (((((a.n + 31) >> 5) + g.nblocks - 1) >> lg)) << 5;
    unsigned short* cols = reinterpret_cast<unsigned short*>(small_vec + 9 * nslot);
    SmallSolve<CL> s{a, small_vec, small_vec + nslot, small_vec + 3 * nslot, small_vec + 2 * nslot, cols,
                     cols + 6 * nslot, a.x, a.q, a.p, tab, red, g.nblocks, lg, g.bid, nslot, 0, smem_addr(small_vec)};
    PhaseClock pc(a.phase_clk, g.bid);
    s.setup();
    return s.loop(nfac, res0, res, singular, pc);
}

}  // namespace spuma

// ops.cu -- face/cell stream kernels on the caller's original ordering:
// laplacian assembly ("Gauss linear corrected"), the LDU Amul through the
// face-to-cell gather lists, and the adjoint's face gradient.
#include <algorithm>

#include "solve.cuh"

namespace spuma {

SolveArgs make_args(spuma_ldu_t h);
spuma_status launch_solve(spuma_ldu_t h, const SolveArgs& a, int threads, cudaStream_t s);
spuma_status pcg_solve_internal(spuma_ldu_t h, const double* diag, const double* upper, const double* b, double* x,
                                const spuma_solver_controls* ctl, spuma_solver_perf* perf, cudaStream_t s,
                                int zero_x0);

static int grid1d(int64_t work, int threads, int num_sms)
{
    int64_t g = (work + threads - 1) / threads;
    g = std::min<int64_t>(g, (int64_t)num_sms * 16);
    return (int)std::max<int64_t>(g, 1);
}

// upper_f = -a_f in face order.  Bound by the FP64 pipe: about 35 instructions
// a face (by time and pipe activity, 87 %) with the shared reciprocals of
// fp64.cuh, 54 with the built-in division and square root: 200^3 assembly 2.87 ->
// 2.05 ms, its reverse mode 2.49 -> 1.62 ms.
__global__ void k_face_coeff(int nf, const int* __restrict__ l, const int* __restrict__ u,
                             const double* __restrict__ sf, const double* __restrict__ c,
                             const double* __restrict__ gamma, double* __restrict__ upper)
{
    for (int f = blockIdx.x * blockDim.x + threadIdx.x; f < nf; f += gridDim.x * blockDim.x) {
        const int lf = l[f], uf = u[f];
        const double* s = sf + 3 * (size_t)f;
        const double* cl = c + 3 * (size_t)lf;
        const double* cu = c + 3 * (size_t)uf;
        upper[f] = -face_coeff(s[0], s[1], s[2], __dsub_rn(cu[0], cl[0]), __dsub_rn(cu[1], cl[1]),
                               __dsub_rn(cu[2], cl[2]), gamma[f]);
    }
}

// Reverse mode of the assembly with respect to gamma: d a / d gamma is the
// face coefficient at gamma = 1 (a is linear in gamma).
__global__ void k_gamma_grad(int nf, const int* __restrict__ l, const int* __restrict__ u,
                             const double* __restrict__ sf, const double* __restrict__ c,
                             const double* __restrict__ gu, const double* __restrict__ gd, double* gg)
{
    for (int f = blockIdx.x * blockDim.x + threadIdx.x; f < nf; f += gridDim.x * blockDim.x) {
        const double* s = sf + 3 * (size_t)f;
        const double* cl = c + 3 * (size_t)l[f];
        const double* cu = c + 3 * (size_t)u[f];
        const double da = face_coeff(s[0], s[1], s[2], __dsub_rn(cu[0], cl[0]), __dsub_rn(cu[1], cl[1]),
                                     __dsub_rn(cu[2], cl[2]), 1.0);
        gg[f] = __dmul_rn(__dsub_rn(__dadd_rn(gd[l[f]], gd[u[f]]), gu[f]), da);
    }
}

__global__ void k_bgamma_grad(int nb, const int* __restrict__ bcell, const int8_t* __restrict__ btype,
                              const double* __restrict__ bsf, const double* __restrict__ bcf,
                              const double* __restrict__ c, const double* __restrict__ gd, double* gb)
{
    for (int b = blockIdx.x * blockDim.x + threadIdx.x; b < nb; b += gridDim.x * blockDim.x) {
        if (btype[b] != 1) {
            gb[b] = 0.0;
            continue;
        }
        const int i = bcell[b];
        const double* s = bsf + 3 * (size_t)b;
        const double* cb = bcf + 3 * (size_t)b;
        const double* ci = c + 3 * (size_t)i;
        const double da = face_coeff(s[0], s[1], s[2], __dsub_rn(cb[0], ci[0]), __dsub_rn(cb[1], ci[1]),
                                     __dsub_rn(cb[2], ci[2]), 1.0);
        gb[b] = __dmul_rn(gd[i], da);
    }
}

// The Dirichlet faces of each cell as a linked list (head[cell], next[b]; the
// order of a list is whatever the atomics gave, k_diag takes it ascending):
// one memset and one kernel instead of a count, a three-kernel scan, a copy and
// a fill (about 55 us at 200^3, launch-bound on small meshes).
__global__ void k_blink(int nb, const int* __restrict__ bcell, const int8_t* __restrict__ btype, int* head, int* next)
{
    for (int b = blockIdx.x * blockDim.x + threadIdx.x; b < nb; b += gridDim.x * blockDim.x)
        if (btype[b] == 1) next[b] = atomicExch(head + bcell[b], b);
}

// A list in ascending order, by its cell's thread alone (bottom-up merges of
// runs of 1, 2, 4, ... faces).
__device__ __noinline__ int sort_list(int first, int* next)
{
    for (int run = 1;; run *= 2) {
        int head = -1, tail = -1, p = first, merges = 0;
        while (p >= 0) {
            int q = p, np = 0, nq = run;
            while (np < run && q >= 0) {
                q = next[q];
                np++;
            }
            merges++;
            while (np > 0 || (nq > 0 && q >= 0)) {
                const bool left = np > 0 && (nq == 0 || q < 0 || p < q);
                const int e = left ? p : q;
                if (left) {
                    p = next[p];
                    np--;
                } else {
                    q = next[q];
                    nq--;
                }
                if (tail >= 0)
                    next[tail] = e;
                else
                    head = e;
                tail = e;
            }
            p = q;
        }
        next[tail] = -1;
        first = head;
        if (merges == 1) return first;
    }
}

// d plus a_b of the cell's Dirichlet faces in ascending face order, a list of
// more than one face sorted first.
__device__ __forceinline__ double add_boundary(double d, int i, const int* head, int* next, const double* c,
                                               const double* bsf, const double* bcf, const double* bgamma)
{
    int b = head ? head[i] : -1;
    if (b >= 0 && next[b] >= 0) b = sort_list(b, next);
    for (; b >= 0; b = next[b]) {
        const double* s = bsf + 3 * (size_t)b;
        const double* cb = bcf + 3 * (size_t)b;
        const double* ci = c + 3 * (size_t)i;
        d = __dadd_rn(d, face_coeff(s[0], s[1], s[2], __dsub_rn(cb[0], ci[0]), __dsub_rn(cb[1], ci[1]),
                                    __dsub_rn(cb[2], ci[2]), bgamma[b]));
    }
    return d;
}

// diag_i = sum over the faces of i in face order (neighbour side ascending,
// owner side ascending) of a_f = -upper_f, then the Dirichlet faces of i in
// ascending order.
__global__ void k_diag(int n, const int* __restrict__ lo_start, const int* __restrict__ lo_face,
                       const int* __restrict__ own_start, const double* __restrict__ upper,
                       const int* __restrict__ head, int* __restrict__ next, const double* __restrict__ c,
                       const double* __restrict__ bsf, const double* __restrict__ bcf,
                       const double* __restrict__ bgamma, double* __restrict__ diag)
{
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
        double d = 0.0;
        for (int k = lo_start[i]; k < lo_start[i + 1]; k++) d = __dadd_rn(d, -upper[lo_face[k]]);
        for (int f = own_start[i]; f < own_start[i + 1]; f++) d = __dadd_rn(d, -upper[f]);
        diag[i] = add_boundary(d, i, head, next, c, bsf, bcf, bgamma);
    }
}

// The same over the fixed-width face lists (entry j of cell i at FL[j n + i],
// +-(f + 1), 0 padding, face order): a cell's face indices arrive in coalesced
// loads with no extents before them, its coefficients in one gather round.
template <int W>
__global__ void __launch_bounds__(256, 8) k_diag_fl(int n, int w, const int* __restrict__ FL,
                                                    const double* __restrict__ upper, const int* __restrict__ head,
                                                    int* __restrict__ next, const double* __restrict__ c,
                                                    const double* __restrict__ bsf, const double* __restrict__ bcf,
                                                    const double* __restrict__ bgamma, double* __restrict__ diag)
{
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
        int e[W];
#pragma unroll
        for (int j = 0; j < W; j++) e[j] = j < w ? __ldcs(FL + (size_t)j * n + i) : 0;
        double t[W];
#pragma unroll
        for (int j = 0; j < W; j++) t[j] = e[j] != 0 ? __ldcs(upper + abs(e[j]) - 1) : 0.0;
        double d = 0.0;
#pragma unroll
        for (int j = 0; j < W; j++)
            if (e[j] != 0) d = __dsub_rn(d, t[j]);
        __stcs(diag + i, add_boundary(d, i, head, next, c, bsf, bcf, bgamma));
    }
}

// y = A x on the caller's arrays.  A row's neighbour-side entries (face and
// column lists) and owner-side entries (its run of faces) are taken as one
// list in groups of G: the group's indices load together, then its
// coefficients and x values, then the FMAs in face order, so a hex row costs
// three memory round trips instead of one chain of three per entry.  On a
// randomly numbered mesh the 72 M gathers of 8 bytes from 32-byte sectors bound
// it (200^3, FP64: 832 -> 811 us).
template <class T>
__global__ void __launch_bounds__(256) k_amul_ldu(int n, const int* __restrict__ lo_start,
                                                  const int* __restrict__ lo_face, const int* __restrict__ lo_col,
                                                  const int* __restrict__ own_start, const int* __restrict__ uaddr,
                                                  const T* __restrict__ diag, const T* __restrict__ upper,
                                                  const T* __restrict__ x, T* __restrict__ y)
{
    constexpr int G = 6;
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
        const int k0 = lo_start[i], nl = lo_start[i + 1] - k0, f0 = own_start[i], nt = nl + own_start[i + 1] - f0;
        T acc = mul_rn(__ldcs(diag + i), x[i]);
        for (int off = 0; off < nt; off += G) {
            int f[G], c[G];
            T a[G], v[G];
#pragma unroll
            for (int j = 0; j < G; j++) {
                const int e = off + j;
                const bool ok = e < nt, low = e < nl;
                f[j] = !ok ? -1 : low ? __ldcs(lo_face + k0 + e) : f0 + (e - nl);
                c[j] = !ok ? 0 : low ? __ldcs(lo_col + k0 + e) : __ldcs(uaddr + f0 + (e - nl));
            }
#pragma unroll
            for (int j = 0; j < G; j++) {
                a[j] = f[j] >= 0 ? upper[f[j]] : T(0);
                v[j] = f[j] >= 0 ? x[c[j]] : T(0);
            }
#pragma unroll
            for (int j = 0; j < G; j++)
                if (f[j] >= 0) acc = fmadd(a[j], v[j], acc);
        }
        __stcs(y + i, acc);
    }
}

// The same an entry at a time, neighbour side then owner side: for meshes whose
// rows don't fit one group.  A second and third group of six, partly empty, cost
// more than the loops' own unrolling: 14 neighbours per cell, FP64, 262 thousand
// cells 42 us in groups, 38 here; 2.0 million 252 and 236.
template <class T>
__global__ void k_amul_ldu_long(int n, const int* __restrict__ lo_start, const int* __restrict__ lo_face,
                                const int* __restrict__ lo_col, const int* __restrict__ own_start,
                                const int* __restrict__ uaddr, const T* __restrict__ diag,
                                const T* __restrict__ upper, const T* __restrict__ x, T* __restrict__ y)
{
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
        T acc = mul_rn(diag[i], x[i]);
        for (int k = lo_start[i]; k < lo_start[i + 1]; k++) acc = fmadd(upper[lo_face[k]], x[lo_col[k]], acc);
        for (int f = own_start[i]; f < own_start[i + 1]; f++) acc = fmadd(upper[f], x[uaddr[f]], acc);
        y[i] = acc;
    }
}

template <class T>
static void launch_amul(spuma_ldu_t h, const void* diag, const void* upper, const void* x, void* y, cudaStream_t s)
{
    const Layout& L = h->L;
    // rows of at most six entries (every row of a mesh that has the fixed-width layout at that width)
    const auto kernel = h->ell_w > 0 && h->ell_w <= 6 ? k_amul_ldu<T> : k_amul_ldu_long<T>;
    kernel<<<grid1d(h->n, 256, h->num_sms), 256, 0, s>>>(
        h->n, h->at<int>(L.lo_start), h->at<int>(L.lo_face), h->at<int>(L.lo_col), h->at<int>(L.own_start),
        h->at<int>(L.uaddr), (const T*)diag, (const T*)upper, (const T*)x, (T*)y);
}

__global__ void k_face_gradient(int nf, int n, const int* __restrict__ l, const int* __restrict__ u,
                                const double* __restrict__ lam, const double* __restrict__ x,
                                double* __restrict__ dupper, double* __restrict__ ddiag)
{
    const int stride = gridDim.x * blockDim.x;
    for (int f = blockIdx.x * blockDim.x + threadIdx.x; f < nf; f += stride) {
        const int lf = l[f], uf = u[f];
        dupper[f] = -(lam[lf] * x[uf] + lam[uf] * x[lf]);
    }
    if (ddiag)
        for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += stride) ddiag[i] = -(lam[i] * x[i]);
}

}  // namespace spuma

using namespace spuma;

extern "C" {

spuma_status spuma_assemble_laplacian(spuma_ldu_t h, const double* face_sf, const double* cell_c,
                                      const double* face_gamma, int32_t n_bfaces, const int32_t* bface_cell,
                                      const double* bface_sf, const double* bface_cf, const double* bface_gamma,
                                      const int8_t* bface_type, double* upper, double* diag, spuma_stream_t stream)
{
    if (!h || n_bfaces < 0 || (h->n > 0 && (!cell_c || !diag)) || (h->nf > 0 && (!face_sf || !face_gamma || !upper)) ||
        (n_bfaces > 0 && (!bface_cell || !bface_sf || !bface_cf || !bface_gamma || !bface_type))) {
        set_error("spuma_assemble_laplacian: bad argument");
        return SPUMA_ERR_INVALID_ARG;
    }
    if (h->n == 0) return SPUMA_OK;
    // temporaries in the (idle) FP64 vector region: head[n], next[<=10n]
    const Layout& L = h->L;
    if ((int64_t)n_bfaces > 10LL * h->n) {
        set_error("more than 10 boundary faces per cell");
        return SPUMA_ERR_WORKSPACE_TOO_SMALL;
    }
    cudaStream_t s = (cudaStream_t)stream;
    const int T = 256;
    if (h->nf > 0) {
        k_face_coeff<<<grid1d(h->nf, T, h->num_sms), T, 0, s>>>(h->nf, h->at<int>(L.laddr), h->at<int>(L.uaddr), face_sf,
                                                                cell_c, face_gamma, upper);
        count_launch();
    }
    int* head = nullptr;
    int* next = nullptr;
    if (n_bfaces > 0) {
        head = h->at<int>(L.x64);             // n ints (x64 holds 2n)
        next = h->at<int>(L.p64);             // <= 10n ints: p64, q64, b64, x32.. are contiguous (>= 11n ints)
        SPUMA_CUDA(cudaMemsetAsync(head, 0xff, 4 * (size_t)h->n, s));
        k_blink<<<grid1d(n_bfaces, T, h->num_sms), T, 0, s>>>(n_bfaces, bface_cell, bface_type, head, next);
        count_launch();
    }
    if (h->nf > 0 && h->ell_w > 0 && h->ell_w <= 6) {
        k_diag_fl<6><<<std::min(grid1d(h->n, T, h->num_sms), h->num_sms * 8), T, 0, s>>>(
            h->n, h->ell_w, h->at<int>(L.FL), upper, head, next, cell_c, bface_sf, bface_cf, bface_gamma, diag);
    } else if (h->nf > 0 || n_bfaces > 0) {
        k_diag<<<grid1d(h->n, T, h->num_sms), T, 0, s>>>(h->n, h->at<int>(L.lo_start), h->at<int>(L.lo_face),
                                                         h->at<int>(L.own_start), upper, head, next, cell_c,
                                                         bface_sf, bface_cf, bface_gamma, diag);
    } else {
        SPUMA_CUDA(cudaMemsetAsync(diag, 0, 8 * (size_t)h->n, s));
    }
    count_launch();
    SPUMA_CUDA(cudaGetLastError());
    return SPUMA_OK;
}

spuma_status spuma_assemble_laplacian_adjoint(spuma_ldu_t h, const double* face_sf, const double* cell_c,
                                              int32_t n_bfaces, const int32_t* bface_cell, const double* bface_sf,
                                              const double* bface_cf, const int8_t* bface_type,
                                              const double* dldupper, const double* dlddiag, double* dldgamma,
                                              double* dldbgamma, spuma_stream_t stream)
{
    if (!h || n_bfaces < 0 || (h->n > 0 && (!cell_c || !dlddiag)) ||
        (h->nf > 0 && (!face_sf || !dldupper || !dldgamma)) ||
        (n_bfaces > 0 && dldbgamma && (!bface_cell || !bface_sf || !bface_cf || !bface_type))) {
        set_error("spuma_assemble_laplacian_adjoint: bad argument");
        return SPUMA_ERR_INVALID_ARG;
    }
    cudaStream_t s = (cudaStream_t)stream;
    const int T = 256;
    const Layout& L = h->L;
    if (h->nf > 0) {
        k_gamma_grad<<<grid1d(h->nf, T, h->num_sms), T, 0, s>>>(h->nf, h->at<int>(L.laddr), h->at<int>(L.uaddr),
                                                                face_sf, cell_c, dldupper, dlddiag, dldgamma);
        count_launch();
    }
    if (n_bfaces > 0 && dldbgamma) {
        k_bgamma_grad<<<grid1d(n_bfaces, T, h->num_sms), T, 0, s>>>(n_bfaces, bface_cell, bface_type, bface_sf,
                                                                    bface_cf, cell_c, dlddiag, dldbgamma);
        count_launch();
    }
    SPUMA_CUDA(cudaGetLastError());
    return SPUMA_OK;
}

spuma_status spuma_amul(spuma_ldu_t h, int32_t precision, const void* diag, const void* upper, const void* x,
                        void* y, spuma_stream_t stream)
{
    if (!h || (precision != SPUMA_F64 && precision != SPUMA_F32) || (h->n > 0 && (!diag || !x || !y)) ||
        (h->nf > 0 && !upper)) {
        set_error("spuma_amul: bad argument");
        return SPUMA_ERR_INVALID_ARG;
    }
    if (h->n == 0) return SPUMA_OK;
    cudaStream_t s = (cudaStream_t)stream;
    if (precision == SPUMA_F64)
        launch_amul<double>(h, diag, upper, x, y, s);
    else
        launch_amul<float>(h, diag, upper, x, y, s);
    count_launch();
    SPUMA_CUDA(cudaGetLastError());
    return SPUMA_OK;
}

spuma_status spuma_pcg_adjoint(spuma_ldu_t h, const double* diag, const double* upper, const double* x,
                               const double* dldx, double* dldb, double* dldupper, double* dlddiag,
                               const spuma_solver_controls* ctl, spuma_solver_perf* perf, spuma_stream_t stream)
{
    if (!h || !ctl || ctl->precision != SPUMA_F64 || (h->n > 0 && (!diag || !x || !dldx || !dldb)) ||
        (h->nf > 0 && (!upper || !dldupper))) {
        set_error("spuma_pcg_adjoint: bad argument (FP64 controls required)");
        return SPUMA_ERR_INVALID_ARG;
    }
    if (h->n == 0) return SPUMA_OK;
    // A lambda = dL/dx from lambda = 0 (A^T = A), written to dldb
    spuma_status st = pcg_solve_internal(h, diag, upper, dldx, dldb, ctl, perf, (cudaStream_t)stream, 1);
    if (st != SPUMA_OK) return st;
    const int T = 256;
    int g = grid1d(std::max(h->nf, h->n), T, h->num_sms);
    k_face_gradient<<<g, T, 0, (cudaStream_t)stream>>>(h->nf, h->n, h->at<int>(h->L.laddr), h->at<int>(h->L.uaddr),
                                                       dldb, x, dldupper, dlddiag);
    count_launch();
    SPUMA_CUDA(cudaGetLastError());
    return SPUMA_OK;
}

}  // extern "C"

// Device code of the IEWPF analysis (Sec. 4 and App. A of arXiv 1910.01031):
// observation set-up, eta-compensated innovations, assembly and FP64
// Cholesky factorisation of HQH^T + R, the S d solves with phi_i, the
// perpendicular random vectors' dot products, the ensemble-wide target
// weight / beta / Lambert-W alpha step, the posterior coarse field and the
// local 49x49 block root applied around each observation.  Each function
// does the work of one thread, warp or CTA (as named) for one problem, so
// that single-problem and batched kernels share it.
#pragma once
#include "common.cuh"
#include "kernels.h"
#include "log_uniform.h"

namespace iewpf {
namespace ana {

__device__ __forceinline__ int min_image(int d, int n)
{
    d = pmod(d, n);
    return d > n / 2 ? d - n : d;
}

// cell and nearest coarse point (ties to the lower one) of observation l
__device__ __forceinline__ void obs_cell_one(const double* __restrict__ xy, int l, const Grid& G, const Coarse& C,
                                             double dx, double dy, int* __restrict__ cell, int* __restrict__ block0)
{
    const int j = pmod((int)floor(xy[2 * l] / dx), G.nx);
    const int k = pmod((int)floor(xy[2 * l + 1] / dy), G.ny);
    cell[2 * l] = j;
    cell[2 * l + 1] = k;
    float t;
    int a = coarse_interval(j, C.nRx, C.c, C.o, G.nx, t);
    int xa = coarse_pos(a, C.nRx, C.c, C.o, G.nx), xb = coarse_pos(a + 1, C.nRx, C.c, C.o, G.nx);
    block0[2 * l] = pmod((j - xa) <= (xb - j) ? a : a + 1, C.nRx);
    int b = coarse_interval(k, C.nRy, C.c, C.o, G.ny, t);
    int ya = coarse_pos(b, C.nRy, C.c, C.o, G.ny), yb = coarse_pos(b + 1, C.nRy, C.c, C.o, G.ny);
    block0[2 * l + 1] = pmod((k - ya) <= (yb - k) ? b : b + 1, C.nRy);
}

// CTA of NTHREADS: observations whose stencil box meets `tile`, listed in
// observation order (deterministic sums in the update kernel)
__device__ __forceinline__ void tile_bin_cta(const int* __restrict__ cell, int nobs, const Grid& G, int R, int tile,
                                             int* __restrict__ cnt, int* __restrict__ list, int cap,
                                             int* __restrict__ flag)
{
    __shared__ int base;
    __shared__ int warp_tot[NTHREADS / 32];
    const int tx = tile % ((G.nx + OBS_TX - 1) / OBS_TX), ty = tile / ((G.nx + OBS_TX - 1) / OBS_TX);
    const int cx = tx * OBS_TX + OBS_TX / 2, cy = ty * OBS_TY + OBS_TY / 2;
    __syncthreads();
    if (threadIdx.x == 0) base = 0;
    __syncthreads();
    for (int l0 = 0; l0 < nobs; l0 += NTHREADS) {
        const int l = l0 + threadIdx.x;
        bool hit = false;
        if (l < nobs) {
            const int ox = min_image(cell[2 * l] - cx, G.nx), oy = min_image(cell[2 * l + 1] - cy, G.ny);
            hit = abs(ox) <= R + OBS_TX / 2 + 1 && abs(oy) <= R + OBS_TY / 2 + 1;
        }
        const unsigned m = __ballot_sync(0xffffffffu, hit);
        const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
        if (lane == 0) warp_tot[w] = __popc(m);
        __syncthreads();
        int off = base;
        for (int i = 0; i < w; ++i) off += warp_tot[i];
        off += __popc(m & ((1u << lane) - 1u));
        if (hit) {
            if (off < cap) list[tile * cap + off] = l;
            else atomicOr(flag, FLAG_TILE_OVERFLOW);
        }
        __syncthreads();
        if (threadIdx.x == 0) {
            int tot = 0;
            for (int i = 0; i < NTHREADS / 32; ++i) tot += warp_tot[i];
            base += tot;
        }
        __syncthreads();
    }
    if (threadIdx.x == 0) cnt[tile] = base < cap ? base : cap;
}

// d = y (H + eta)/H - (hu, hv) at the observed cell (eq. etaCompensatedInnovation)
__device__ __forceinline__ void innovate_one(const float* __restrict__ b0, const float* __restrict__ b1,
                                             const int* __restrict__ par, const int* __restrict__ cell,
                                             const double* __restrict__ y, int nobs, const Grid& G, double H,
                                             double* __restrict__ d, int i)
{
    const int p = i / nobs, l = i % nobs;
    const float* __restrict__ U = (par[p] ? b1 : b0) + (long long)p * 3 * G.plane;
    const long long c = (long long)cell[2 * l + 1] * G.nx + cell[2 * l];
    const double s = (H + (double)U[c]) / H;
    d[(long long)i * 2] = fma(y[2 * l], s, -(double)U[G.plane + c]);
    d[(long long)i * 2 + 1] = fma(y[2 * l + 1], s, -(double)U[2 * G.plane + c]);
}

// (HQH^T)_{(l,a),(k,b)}: component a of the response to a unit b observation
// at obs k, read at obs l's cell
__device__ __forceinline__ double kval(const double* K, int R, const int* cell, int l, int a, int k, int b,
                                       const Grid& G)
{
    const int ox = min_image(cell[2 * l] - cell[2 * k], G.nx);
    const int oy = min_image(cell[2 * l + 1] - cell[2 * k + 1], G.ny);
    if (abs(ox) > R || abs(oy) > R) return 0.0;
    const int W = 2 * R + 1;
    return K[((b * 3 + 1 + a) * W + (oy + R)) * W + (ox + R)];
}

// entry i of the symmetrised HQH^T + sigma^2 I
__device__ __forceinline__ void hqht_one(const double* __restrict__ K, int R, const int* __restrict__ cell, int nobs,
                                         const Grid& G, int dense, double sigma2, double* __restrict__ M, long long i)
{
    const int n = 2 * nobs;
    const int r = (int)(i / n), c = (int)(i % n);
    const int l = r >> 1, a = r & 1, k = c >> 1, b = c & 1;
    double v = 0.0;
    if (dense || l == k) v = 0.5 * (kval(K, R, cell, l, a, k, b, G) + kval(K, R, cell, k, b, l, a, G));
    if (r == c) v += sigma2;
    M[i] = v;
}

// Right-looking Cholesky of a dense SPD matrix in place (lower triangle), one
// CTA; the update of column k touches only rows with a non-zero in it, so
// block-diagonal and banded matrices cost their fill, not n^3/3.  A may live
// in global or shared memory; nzlist holds n ints.  The strict upper triangle
// is zeroed; *bad (shared) is set for a non-positive pivot.  ld: doubles from
// row to row (odd in shared memory, where columns are read too).
__device__ __forceinline__ void cholesky_factor_cta(double* __restrict__ A, int n, int ld, int* __restrict__ nzlist,
                                                    int* bad)
{
    __shared__ int nnz;
    __shared__ double piv;
    for (int k = 0; k < n; ++k) {
        if (threadIdx.x == 0) {
            const double dkk = A[(long long)k * ld + k];
            if (!(dkk > 0.0)) *bad = 1;
            piv = dkk > 0.0 ? sqrt(dkk) : 1.0;
            A[(long long)k * ld + k] = piv;
            nnz = 0;
        }
        __syncthreads();
        for (int i = k + 1 + threadIdx.x; i < n; i += blockDim.x) {
            const double v = A[(long long)i * ld + k];
            if (v != 0.0) {
                A[(long long)i * ld + k] = v / piv;
                nzlist[atomicAdd(&nnz, 1)] = i;
            }
        }
        __syncthreads();
        const int m = nnz;
        const long long pairs = (long long)m * m;
        for (long long q = threadIdx.x; q < pairs; q += blockDim.x) {
            const int i = nzlist[q / m], j = nzlist[q % m];
            if (j <= i) A[(long long)i * ld + j] = fma(-A[(long long)i * ld + k], A[(long long)j * ld + k], A[(long long)i * ld + j]);
        }
        __syncthreads();
    }
    for (long long q = threadIdx.x; q < (long long)n * n; q += blockDim.x) {
        const int i = (int)(q / n), j = (int)(q % n);
        if (j > i) A[(long long)i * ld + j] = 0.0;
    }
    __syncthreads();
}

// CTA: counts p[1..n] to offsets p[0..n] in place, by warp 0
__device__ __forceinline__ void prefix_cta(int* p, int n)
{
    if (threadIdx.x < 32) {
        const int lane = threadIdx.x;
        int base = 0;
        for (int t0 = 1; t0 <= n; t0 += 32) {
            const int t = t0 + lane;
            int v = t <= n ? p[t] : 0;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int w = __shfl_up_sync(0xffffffffu, v, o);
                if (lane >= o) v += w;
            }
            if (t <= n) p[t] = base + v;
            base += __shfl_sync(0xffffffffu, v, 31);
        }
        if (lane == 0) p[0] = 0;
    }
    __syncthreads();
}

// CTA: rows in increasing index within each level (deterministic), ptr the
// level boundaries, *nlev their number: every row counts those before it
__device__ __forceinline__ void level_sort_cta(const int* __restrict__ lev, int n, int* __restrict__ order,
                                               int* __restrict__ ptr, int* __restrict__ nlev)
{
    for (int i = threadIdx.x; i < n; i += blockDim.x) {
        const int li = lev[i];
        int below = 0, same = 0, top = 0;
        for (int j = 0; j < n; ++j) {
            const int lj = lev[j];
            below += lj < li;
            same += lj == li && j < i;
            top = max(top, lj);
        }
        order[below + same] = i;
        if (same == 0) ptr[li] = below;
        if (i == 0) {
            ptr[top + 1] = n;
            *nlev = top + 1;
        }
    }
}

// The factorisation of cholesky_factor_cta level by level, A in shared memory:
// a column depends on those that its row has entries in, so the columns of one
// level of the elimination tree are factored together.  FP64 latency bounds a
// column (a square root, then a division: about 3500 cycles), so what counts
// is how many follow one another: 128 for 64 drifters column by column, a few
// by levels where most of them do not interact (factor and plan 258 us, now
// 69).  Left-looking, with every entry's products in the order of
// cholesky_factor_cta and its rules for zeros: the same bits.  False, with A
// unchanged, when the levels are more than a quarter of the columns (a thread
// per entry would then have too many products) or the columns few.
// n <= 1024; work:
// chol_levels_ints(n) ints of shared memory.
__host__ __device__ __forceinline__ int chol_levels_ints(int n) { return 2 * n * ((n + 31) / 32) + 4 * n + 3; }
__device__ __forceinline__ bool cholesky_levels_cta(double* A, int n, int ld, int* work, int* bad)
{
    if (n < 32) return false;
    const int nw = (n + 31) / 32, lane = threadIdx.x & 31, warp = threadIdx.x >> 5, warps = blockDim.x >> 5;
    unsigned* const col = reinterpret_cast<unsigned*>(work);   // [n][nw] rows below the diagonal of each column
    unsigned* const row = col + n * nw;                        // [n][nw] columns before the diagonal of each row
    int* const lev = work + 2 * n * nw;
    int* const order = lev + n;
    int* const first = order + n;                              // [n + 1]
    int* const ptr = first + n + 1;                            // [n + 1], then the number of levels
    for (int k = warp; k < n; k += warps) {
        for (int w = 0; w < nw; ++w) {
            const int i = 32 * w + lane;
            const unsigned b = __ballot_sync(0xffffffffu, i > k && i < n && A[i * ld + k] != 0.0);
            if (lane == 0) col[k * nw + w] = b;
        }
        if (lane == 0) lev[k] = 0;
    }
    __syncthreads();
    // fill: a column's first row below the diagonal is its parent, which
    // inherits its other rows
    if (warp == 0)
        for (int k = 0; k < n; ++k) {
            const unsigned mine = lane < nw ? col[k * nw + lane] : 0u;
            const unsigned any = __ballot_sync(0xffffffffu, mine != 0u);
            if (any == 0u) continue;
            const int w0 = __ffs(any) - 1;
            const int bit = __ffs(__shfl_sync(0xffffffffu, mine, w0)) - 1, p = 32 * w0 + bit;
            if (lane < nw) col[p * nw + lane] |= lane == w0 ? mine & ~(1u << bit) : mine;
            if (lane == 0) lev[p] = max(lev[p], lev[k] + 1);
            __syncwarp();
        }
    __syncthreads();
    for (int j = warp; j < n; j += warps)
        for (int w = 0; w < nw; ++w) {
            const int k = 32 * w + lane;
            const unsigned b = __ballot_sync(0xffffffffu, k < j && ((col[min(k, n - 1) * nw + (j >> 5)] >> (j & 31)) & 1u));
            if (lane == 0) row[j * nw + w] = b;
        }
    level_sort_cta(lev, n, order, ptr, ptr + n + 1);
    __syncthreads();
    const int nlev = ptr[n + 1];
    if (4 * nlev > n) return false;
    // first[t]: entries below the diagonal of the columns before position t
    for (int t = threadIdx.x; t < n; t += blockDim.x) {
        int c = 0;
        for (int w = 0; w < nw; ++w) c += __popc(col[order[t] * nw + w]);
        first[t + 1] = c;
    }
    __syncthreads();
    prefix_cta(first, n);
    // entry (i, j) less its products over the columns of row j, in their order
    auto reduced = [&](int i, int j) {
        double acc = A[i * ld + j];
        for (int w = 0; w <= j >> 5; ++w)
            for (unsigned b = row[j * nw + w]; b; b &= b - 1u) {
                const int k = 32 * w + __ffs(b) - 1;
                const double ajk = A[j * ld + k], aik = A[i * ld + k];
                if (ajk != 0.0 && aik != 0.0) acc = fma(-aik, ajk, acc);
            }
        return acc;
    };
    for (int l = 0; l < nlev; ++l) {
        // a thread per pivot, then a thread per entry
        for (int t = ptr[l] + threadIdx.x; t < ptr[l + 1]; t += blockDim.x) {
            const int j = order[t];
            const double d = reduced(j, j);
            if (!(d > 0.0)) *bad = 1;
            A[j * ld + j] = d > 0.0 ? sqrt(d) : 1.0;
        }
        __syncthreads();
        for (int q = first[ptr[l]] + threadIdx.x; q < first[ptr[l + 1]]; q += blockDim.x) {
            int lo = ptr[l], hi = ptr[l + 1];           // first[lo] <= q < first[hi]
            while (hi - lo > 1) {
                const int mid = (lo + hi) >> 1;
                if (first[mid] <= q) lo = mid;
                else hi = mid;
            }
            const int j = order[lo];
            int rank = q - first[lo], w = 0, c;
            while (rank >= (c = __popc(col[j * nw + w]))) rank -= c, ++w;
            unsigned b = col[j * nw + w];
            for (; rank > 0; --rank) b &= b - 1u;
            const int i = 32 * w + __ffs(b) - 1;
            const double v = reduced(i, j);
            A[i * ld + j] = v != 0.0 ? v / A[j * ld + j] : v;
        }
        __syncthreads();
    }
    for (int i = warp; i < n; i += warps)
        for (int k = i + 1 + lane; k < n; k += 32) A[i * ld + k] = 0.0;
    __syncthreads();
    return true;
}

// The factor's columns as CSC of the strictly lower part, rows increasing:
// one warp per column counts (ballots), a prefix sum gives colptr, and the
// warps write the row lists in order.
__device__ __forceinline__ void csc_cta(const double* __restrict__ L, int n, int ld, int* colptr, int* __restrict__ rowidx)
{
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
    for (int k = warp; k < n; k += nw) {
        int cnt = 0;
        for (int i0 = k + 1; i0 < n; i0 += 32) {
            const int i = i0 + lane;
            cnt += __popc(__ballot_sync(0xffffffffu, i < n && L[(long long)i * ld + k] != 0.0));
        }
        if (lane == 0) colptr[k + 1] = cnt;
    }
    __syncthreads();
    prefix_cta(colptr, n);
    for (int k = warp; k < n; k += nw) {
        int pos = colptr[k];
        for (int i0 = k + 1; i0 < n; i0 += 32) {
            const int i = i0 + lane;
            const bool nz = i < n && L[(long long)i * ld + k] != 0.0;
            const unsigned bal = __ballot_sync(0xffffffffu, nz);
            if (nz) rowidx[pos + __popc(bal & ((1u << lane) - 1u))] = i;
            pos += __popc(bal);
        }
    }
    __syncthreads();
}

// Factor in global memory and list the factor's columns; rowidx doubles as
// the work list during the factorisation.
// rowidx and nzlist may be the same array (the work list of the
// factorisation, then the row indices of the factor), so neither is restrict
__device__ __forceinline__ void cholesky_cta(double* __restrict__ A, int n, int* __restrict__ colptr, int* rowidx,
                                             int* __restrict__ flag, int* nzlist)
{
    __shared__ int bad;
    __syncthreads();
    if (threadIdx.x == 0) bad = 0;
    __syncthreads();
    cholesky_factor_cta(A, n, n, nzlist, &bad);
    csc_cta(A, n, n, colptr, rowidx);
    if (threadIdx.x == 0 && bad) atomicOr(flag, FLAG_NOTPD);
}

// Level schedule of the triangular solves with the factor L (CSC below the
// diagonal in colptr/rowidx).  Rows of one level of the forward sweep
// L y = d depend only on rows of lower levels, and likewise columns of one
// level of the backward sweep L^T x = y; 2 x 2 blocks (observations that do
// not interact) give two levels each.  Int layout of `plan`, n = order:
// rowptr[n+1] | forder[n] | fptr[n+1] | border[n] | bptr[n+1] | nlev[2] |
// lev[n] | colidx[n(n-1)/2] (CSR below the diagonal, column order in a row).
// rf, rb: per position t of the forward (backward) level order, the row
// (column) and the bounds of its entries: {i, start, end}
struct SolvePlan {
    int *rowptr, *forder, *fptr, *border, *bptr, *nlev, *lev, *rf, *rb, *colidx;
};

__host__ __device__ inline SolvePlan solve_plan_view(int* base, int n)
{
    SolvePlan P;
    P.rowptr = base;
    P.forder = P.rowptr + n + 1;
    P.fptr = P.forder + n;
    P.border = P.fptr + n + 1;
    P.bptr = P.border + n;
    P.nlev = P.bptr + n + 1;
    P.lev = P.nlev + 2;
    P.rf = P.lev + n;
    P.rb = P.rf + 3 * n;
    P.colidx = P.rb + 3 * n;
    return P;
}

// CTA: lev[i] = 1 + the largest level among the j with entry(i, j), by rounds
// over all i until none grows (levels only grow, so a round may read those
// that it is raising); lev in shared memory
template <class F>
__device__ __forceinline__ void levels_smem_cta(int* lev_, int n, F entry)
{
    volatile int* lev = lev_;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
    for (int i = threadIdx.x; i < n; i += blockDim.x) lev[i] = 0;
    __syncthreads();
    bool grew = true;
    while (grew) {
        grew = false;
        for (int i = warp; i < n; i += nw) {
            int m = -1;
            for (int j0 = 0; j0 < n; j0 += 32) {
                const int j = j0 + lane;
                if (j < n && entry(i, j)) m = max(m, lev[j]);
            }
            m = __reduce_max_sync(0xffffffffu, m) + 1;
            if (m > lev[i]) {
                grew = true;
                __syncwarp();
                if (lane == 0) lev[i] = m;
            }
            __syncwarp();
        }
        grew = __syncthreads_or(grew);
    }
}

// CTA: reciprocal diagonal, CSR of L below the diagonal and both level
// schedules; after csc_cta (colptr/rowidx complete).  The levels are kept in
// shared memory where they fit, and with L itself there (SMEM) the rows'
// non-zeros are read from it (64 drifters: one thread or warp going row by
// row through global memory took about 90 us, rounds over all rows 10).
constexpr int PLAN_LEV = 2048;
template <bool SMEM>
__device__ __forceinline__ void solve_plan_cta(const double* __restrict__ L, int n, int ld, const int* __restrict__ colptr,
                                               const int* __restrict__ rowidx, double* __restrict__ rdiag,
                                               int* plan_base)
{
    const SolvePlan P = solve_plan_view(plan_base, n);
    __shared__ int slev[PLAN_LEV];
    int* const lev = n <= PLAN_LEV ? slev : P.lev;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
    __syncthreads();
    for (int i = threadIdx.x; i < n; i += blockDim.x) rdiag[i] = 1.0 / L[(long long)i * ld + i];
    for (int i = warp; i < n; i += nw) {
        int cnt = 0;
        for (int j0 = 0; j0 < i; j0 += 32) {
            const int j = j0 + lane;
            cnt += __popc(__ballot_sync(0xffffffffu, j < i && L[(long long)i * ld + j] != 0.0));
        }
        if (lane == 0) P.rowptr[i + 1] = cnt;
    }
    __syncthreads();
    prefix_cta(P.rowptr, n);
    for (int i = warp; i < n; i += nw) {
        int pos = P.rowptr[i];
        for (int j0 = 0; j0 < i; j0 += 32) {
            const int j = j0 + lane;
            const bool nz = j < i && L[(long long)i * ld + j] != 0.0;
            const unsigned bal = __ballot_sync(0xffffffffu, nz);
            if (nz) P.colidx[pos + __popc(bal & ((1u << lane) - 1u))] = j;
            pos += __popc(bal);
        }
    }
    __syncthreads();
    // forward levels: 1 + the largest level among the row's columns.  In shared
    // memory a warp per row, all rows until nothing changes (as many rounds as
    // levels); else row after row
    if (SMEM) {
        levels_smem_cta(lev, n, [&](int i, int j) { return j < i && L[(long long)i * ld + j] != 0.0; });
    } else if (warp == 0)
        for (int i = 0; i < n; ++i) {
            int m = -1;
            for (int q = P.rowptr[i] + lane; q < P.rowptr[i + 1]; q += 32) m = max(m, lev[P.colidx[q]]);
            m = __reduce_max_sync(0xffffffffu, m);
            if (lane == 0) lev[i] = m + 1;
            __syncwarp();
        }
    __syncthreads();
    level_sort_cta(lev, n, P.forder, P.fptr, P.nlev);
    __syncthreads();
    // backward levels: 1 + the largest level among the column's rows
    if (SMEM) {
        levels_smem_cta(lev, n, [&](int i, int k) { return k > i && L[(long long)k * ld + i] != 0.0; });
    } else if (warp == 0)
        for (int i = n - 1; i >= 0; --i) {
            int m = -1;
            for (int q = colptr[i] + lane; q < colptr[i + 1]; q += 32) m = max(m, lev[rowidx[q]]);
            m = __reduce_max_sync(0xffffffffu, m);
            if (lane == 0) lev[i] = m + 1;
            __syncwarp();
        }
    __syncthreads();
    level_sort_cta(lev, n, P.border, P.bptr, P.nlev + 1);
    __syncthreads();
    for (int t = threadIdx.x; t < n; t += blockDim.x) {
        const int i = P.forder[t], k = P.border[t];
        P.rf[3 * t] = i;
        P.rf[3 * t + 1] = P.rowptr[i];
        P.rf[3 * t + 2] = P.rowptr[i + 1];
        P.rb[3 * t] = k;
        P.rb[3 * t + 1] = colptr[k];
        P.rb[3 * t + 2] = colptr[k + 1];
    }
    __syncthreads();
}

// warp: S d = (L L^T)^{-1} d for particle w and phi_w = d^T S d along the
// level schedule: a level of 32 rows or more gives one row per lane (the
// row's sum in column order), a narrower one a group of lanes to each row
// (lane-strided partial sums, then the group's sum)
// perm (may be null): the factor is that of P A P^T with unknown i of the
// factored system = unknown perm[i] of the observations; the sweeps then run
// in that order in scratch (n doubles per particle), d is read through perm
// and the result written back through it
// Lr, Lc (may be null): the factor's values below the diagonal in the order
// of the plan's CSR (colidx) and of the CSC (rowidx), so that a row's or a
// column's products read consecutive doubles instead of scattered entries of
// the dense factor (launch_pack_factor)
// sx (may be null): n doubles of shared memory owned by this warp; the sweeps
// then run there instead of in scratch or x, so that the products of a level
// wait on shared memory, not on L2, for the values of the levels before
__device__ __forceinline__ void solve_levels_warp(const double* __restrict__ L, const int* __restrict__ colptr,
                                                  const int* __restrict__ rowidx, const double* __restrict__ rdiag,
                                                  const int* plan_base, int n, const double* __restrict__ d,
                                                  double* __restrict__ x, double* __restrict__ phi, int w,
                                                  const int* __restrict__ perm = nullptr,
                                                  double* __restrict__ scratch = nullptr,
                                                  const double* __restrict__ Lr = nullptr,
                                                  const double* __restrict__ Lc = nullptr, double* sx = nullptr)
{
    const SolvePlan P = solve_plan_view(const_cast<int*>(plan_base), n);
    const int lane = threadIdx.x & 31;
    double* xp = sx ? sx : (perm ? scratch : x) + (long long)w * n;
    const double* dp = d + (long long)w * n;
    auto dval = [&](int i) { return perm ? dp[perm[i]] : dp[i]; };
    // entry q of row i (column j) of the CSR; entry q of column i (row k) of the CSC
    auto lrow = [&](int q, int i, int j) { return Lr ? Lr[q] : L[(long long)i * n + j]; };
    auto lcol = [&](int q, int i, int k) { return Lc ? Lc[q] : L[(long long)k * n + i]; };
    // the right-hand side in the order of the factored system; the forward
    // sweep then overwrites it row by row
    for (int i = lane; i < n; i += 32) xp[i] = dval(i);
    __syncwarp();
    // One sweep over the levels lv[0..nl] of a level order whose position t
    // holds row (or column) ri[3t] with entries ri[3t+1]..ri[3t+2] (index
    // idx[q], value val(q, i, idx[q])).  A level of m < 32 rows gives each row
    // a group of g = 32 / 2^ceil(log2 m) lanes (lane-strided partial sums in
    // entry order, then the group's sum), a wider one a lane per row, in
    // rounds of 32 rows.  None of the loads but those of xp depends on an
    // earlier level, so they are issued ahead: while level l is summed, the
    // first batch of entries and the diagonal of level l+1, the row
    // descriptors of level l+2 and the bounds of level l+3 are in flight.
    constexpr int U = 8;
    auto sweep = [&](const int* __restrict__ lv, int nl, const int* __restrict__ ri, const int* __restrict__ idx,
                     auto val) {
        auto bound = [&](int k) { return lv[k < nl ? k : nl]; };
        auto log_group = [](int m) { return m >= 32 ? 0 : 5 - (m <= 1 ? 0 : 32 - __clz(m - 1)); };
        // this lane's first row of a level: {i (-1: none), first entry, end}
        auto fetch_row = [&](int lo, int hi, int& i, int& q0, int& q1) {
            const int lg = log_group(hi - lo);
            const int t = lo + (lane >> lg);
            i = -1;
            q0 = q1 = 0;
            if (t < hi) {
                i = ri[3 * t];
                q0 = ri[3 * t + 1] + (lane & ((1 << lg) - 1));
                q1 = ri[3 * t + 2];
            }
        };
        auto fetch_batch = [&](int i, int q0, int q1, int g, int* jj, double* vv) {
#pragma unroll
            for (int u = 0; u < U; ++u) jj[u] = q0 + u * g < q1 ? idx[q0 + u * g] : -1;
#pragma unroll
            for (int u = 0; u < U; ++u) vv[u] = jj[u] >= 0 ? val(q0 + u * g, i, jj[u]) : 0.0;
        };
        auto sum_batch = [&](const int* jj, const double* vv, double acc) {
#pragma unroll
            for (int u = 0; u < U; ++u)
                if (jj[u] >= 0) acc = fma(vv[u], xp[jj[u]], acc);
            return acc;
        };
        // the row of one round: the prefetched first batch, then the rest
        auto finish_row = [&](int lg, int i, int q0, int q1, const int* jj, const double* vv, double rd) {
            const int g = 1 << lg;
            double acc = 0.0;
            if (i >= 0) {
                // the next batch is in flight while the current one is summed
                int cj[U];
                double cv[U];
#pragma unroll
                for (int u = 0; u < U; ++u) {
                    cj[u] = jj[u];
                    cv[u] = vv[u];
                }
                for (int q = q0 + U * g;; q += U * g) {
                    const bool more = q < q1;
                    int kj[U];
                    double kv[U];
                    if (more) fetch_batch(i, q, q1, g, kj, kv);
                    acc = sum_batch(cj, cv, acc);
                    if (!more) break;
#pragma unroll
                    for (int u = 0; u < U; ++u) {
                        cj[u] = kj[u];
                        cv[u] = kv[u];
                    }
                }
            }
            for (int o = g >> 1; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
            if (i >= 0 && (lane & (g - 1)) == 0) xp[i] = (xp[i] - acc) * rd;
        };
        // pipeline: level l (bounds, row, batch, diagonal), level l+1 (bounds,
        // row), level l+2 (bounds)
        int lo0 = bound(0), hi0 = bound(1), lo1 = hi0, hi1 = bound(2), lo2 = hi1, hi2 = bound(3);
        int i0, a0, e0, i1, a1, e1;
        fetch_row(lo0, hi0, i0, a0, e0);
        fetch_row(lo1, hi1, i1, a1, e1);
        int j0[U];
        double v0[U];
        fetch_batch(i0, a0, e0, 1 << log_group(hi0 - lo0), j0, v0);
        double rd0 = i0 >= 0 ? rdiag[i0] : 0.0;
        for (int l = 0; l < nl; ++l) {
            // issue the loads of the levels ahead
            int j1[U];
            double v1[U];
            fetch_batch(i1, a1, e1, 1 << log_group(hi1 - lo1), j1, v1);
            const double rd1 = i1 >= 0 ? rdiag[i1] : 0.0;
            int i2, a2, e2;
            fetch_row(lo2, hi2, i2, a2, e2);
            const int hi3 = bound(l + 4);
            // level l: the first round from the prefetched values, further
            // rounds (more than 32 rows) loaded here
            const int lg = log_group(hi0 - lo0);
            finish_row(lg, i0, a0, e0, j0, v0, rd0);
            for (int t = lo0 + 32 + lane; t - lane < hi0; t += 32) {
                int i = -1, q0 = 0, q1 = 0;
                if (t < hi0) {
                    i = ri[3 * t];
                    q0 = ri[3 * t + 1];
                    q1 = ri[3 * t + 2];
                }
                int jj[U];
                double vv[U];
                fetch_batch(i, q0, q1, 1, jj, vv);
                finish_row(0, i, q0, q1, jj, vv, i >= 0 ? rdiag[i] : 0.0);
            }
            __syncwarp();
            // advance the pipeline
            lo0 = lo1; hi0 = hi1; i0 = i1; a0 = a1; e0 = e1; rd0 = rd1;
#pragma unroll
            for (int u = 0; u < U; ++u) {
                j0[u] = j1[u];
                v0[u] = v1[u];
            }
            lo1 = lo2; hi1 = hi2; i1 = i2; a1 = a2; e1 = e2;
            lo2 = hi2; hi2 = hi3;
        }
    };
    // forward: y_i = (d_i - sum_j L_ij y_j) / L_ii
    sweep(P.fptr, P.nlev[0], P.rf, P.colidx, lrow);
    // backward: x_i = (y_i - sum_k L_ki x_k) / L_ii over k > i
    sweep(P.bptr, P.nlev[1], P.rb, rowidx, lcol);
    double acc = 0.0;
    for (int i = lane; i < n; i += 32) acc = fma(dval(i), xp[i], acc);
    acc = warp_sum(acc);
    if (lane == 0) phi[w] = acc;
    if (perm || sx) {
        double* out = x + (long long)w * n;
        for (int i = lane; i < n; i += 32) out[perm ? perm[i] : i] = xp[i];
    }
}

// The factor as the two sweeps read it, for solve_group_cta: positions t of the
// level order hold row[t] = {row (column) i, first entry, end, -} and its
// reciprocal diagonal rd[t]; the entries (in the order of the CSR or CSC) are
// contiguous along the order.  step[s] = {first position, rows (at most 32) +
// 256 log2 of the lanes per row, first entry, end}: a level, or a round of 32
// rows of a wider one.
struct __align__(16) SweepEntry {
    double val;
    int idx, pad;
};
struct SweepStream {
    int4 *step, *row;   // [n] each
    SweepEntry* ent;    // [nnz]
    double* rd;         // [n]
    int* nstep;         // [1]
};
// bytes of one direction's arrays, and its view at base (16-byte aligned)
__host__ __device__ __forceinline__ size_t sweep_stream_bytes(int n, int nnz)
{
    return 16 * (2 * (size_t)n + nnz + ((size_t)n + 1) / 2 + 1);
}
__host__ __device__ __forceinline__ SweepStream sweep_stream_view(void* base, int n, int nnz)
{
    SweepStream S;
    S.step = static_cast<int4*>(base);
    S.row = S.step + n;
    S.ent = reinterpret_cast<SweepEntry*>(S.row + n);
    S.nstep = reinterpret_cast<int*>(S.ent + nnz);
    S.rd = reinterpret_cast<double*>(S.ent + nnz + 1);
    return S;
}

// warp: row, rd and the steps of one direction from the plan's triples ri and
// level bounds lv[0..nl]
__device__ __forceinline__ void sweep_rows_warp(const int* __restrict__ ri, const int* __restrict__ lv, int nl, int n,
                                                const double* __restrict__ rdiag, const SweepStream& S)
{
    const int lane = threadIdx.x & 31;
    int base = 0;
    for (int t0 = 0; t0 < n; t0 += 32) {
        const int t = t0 + lane;
        const int len = t < n ? ri[3 * t + 2] - ri[3 * t + 1] : 0;
        int end = len;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int v = __shfl_up_sync(0xffffffffu, end, o);
            if (lane >= o) end += v;
        }
        if (t < n) {
            S.row[t] = make_int4(ri[3 * t], base + end - len, base + end, 0);
            S.rd[t] = rdiag[ri[3 * t]];
        }
        base += __shfl_sync(0xffffffffu, end, 31);
    }
    __syncwarp();
    int ns = 0;
    if (lane == 0) {
        for (int l = 0; l < nl; ++l) {
            const int m = lv[l + 1] - lv[l];
            const int lg = m >= 32 ? 0 : 5 - (m <= 1 ? 0 : 32 - __clz(m - 1));
            for (int t = lv[l]; t < lv[l + 1]; t += 32) {
                const int e = min(t + 32, lv[l + 1]);
                S.step[ns++] = make_int4(t, (e - t) + 256 * lg, S.row[t].y, S.row[e - 1].z);
            }
        }
        *S.nstep = ns;
    }
}

__device__ __forceinline__ void cp_async16(void* s, const void* g)
{
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"((uint32_t)__cvta_generic_to_shared(s)), "l"(g)
                 : "memory");
}
template <int N>
__device__ __forceinline__ void cp_async_wait()
{
    asm volatile("cp.async.wait_group %0;\n" ::"n"(N) : "memory");
}

// CTA of 32 P threads: solve_levels_warp for P particles together, their
// vectors interleaved in shared memory (entry i of particle p at i P + p).  The
// 32 lanes that a level's rows share there are 32 slots here, of P lanes each,
// one per particle: a factor entry is loaded once for P particles, and the
// slots spread over P warps.  The entries flow through a ring in shared memory
// (cp.async, several steps ahead), so that a step waits on shared memory and
// its FP64 chain alone.  A row's partial sums, their order and the order of the
// group's sum are those of solve_levels_warp: the same bits.
constexpr int SOLVE_RING = 2048;      // entries
template <int P>
__host__ __device__ constexpr size_t solve_group_smem(int n)
{
    return SOLVE_RING * sizeof(SweepEntry) + ((size_t)n * P + P * P) * sizeof(double);
}
template <int P>
__device__ __forceinline__ void solve_group_cta(const SweepStream& F, const SweepStream& B, int n, int nnz,
                                                const double* __restrict__ d, double* __restrict__ x,
                                                double* __restrict__ phi, int w0, int ne,
                                                const int* __restrict__ perm, double* smem)
{
    constexpr int S = 32 / P;      // slots per warp (P warps)
    constexpr int LS = P == 4 ? 3 : 2;
    static_assert(1 << LS == S, "slots per warp");
    SweepEntry* const rent = reinterpret_cast<SweepEntry*>(smem);
    double* const part = smem + SOLVE_RING * (sizeof(SweepEntry) / sizeof(double));
    double* const sx = part + P * P;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int p = lane % P, slot = lane / P;
    const int np = min(P, ne - w0);
    for (int k = tid; k < n * np; k += 32 * P) {
        const int w = k / n, i = k - w * n;
        sx[i * P + w] = d[(long long)(w0 + w) * n + (perm ? perm[i] : i)];
    }
    if (np < P)
        for (int k = tid; k < n; k += 32 * P)
            for (int w = np; w < P; ++w) sx[k * P + w] = 0.0;
    auto sweep = [&](const SweepStream& Q) {
        const int ns = *Q.nstep;
        int issued = 0;
        auto top_up = [&](int upto) {
            for (int q = issued + tid; q < upto; q += 32 * P) {
                cp_async16(rent + (q & (SOLVE_RING - 1)), Q.ent + q);
            }
            issued = max(issued, upto);
            asm volatile("cp.async.commit_group;\n" ::: "memory");
        };
        auto step_at = [&](int k) { return k < ns ? Q.step[k] : make_int4(n, 0, nnz, nnz); };
        // this slot's row of a step {row (-1: none), first entry, end, diagonal} and
        // place in the row's group of g slots: the upper bits of the place are the
        // slot's in its warp, so that the halves that the group's sum joins first
        // lie in one warp
        struct Row {
            int i, q0, q1;
            double rd;
        };
        auto row_at = [&](const int4& st) {
            const int lg = st.y >> 8, m = st.y & 255;
            int r, sub;
            if (lg >= LS) {
                r = warp >> (lg - LS);
                sub = (warp & ((1 << (lg - LS)) - 1)) + (slot << (lg - LS));
            } else {
                r = (warp << (LS - lg)) + (slot >> lg);
                sub = slot & ((1 << lg) - 1);
            }
            Row R{-1, 0, 0, 0.0};
            if (r < m) {
                const int4 v = Q.row[st.x + r];
                R.i = v.x;
                R.q0 = v.y + sub;
                R.q1 = v.z;
                R.rd = Q.rd[st.x + r];
            }
            return R;
        };
        int4 s0 = step_at(0), s1 = step_at(1), s2 = step_at(2);
        Row r0 = row_at(s0), r1 = row_at(s1);
        top_up(min(nnz, SOLVE_RING));
        cp_async_wait<0>();
        __syncthreads();
        int safe = issued, mark1 = issued, mark2 = issued;   // entries arrived; issued one and two steps ago
#pragma unroll 3
        for (int k = 0; k < ns; ++k) {
            const int4 s3 = step_at(k + 3);
            const Row r2 = row_at(s2);
            // what precedes this step's entries is free
            issued = max(issued, s0.z);
            top_up(min(nnz, s0.z + SOLVE_RING));
            const bool ring = s0.w - s0.z <= SOLVE_RING;
            if (ring && s0.w > safe) {
                cp_async_wait<0>();
                __syncthreads();
                safe = issued;
            }
            const int lg = s0.y >> 8, g = 1 << lg;
            double acc = 0.0;
            // batches of 8 entries, a last one of those that are left
            auto products = [&](const SweepEntry* ent, int mask) {
                constexpr int U = 8;
                int q = r0.q0, left = (r0.q1 - r0.q0 + g - 1) >> lg;
                for (; left >= U; left -= U, q += U << lg) {
                    double v[U], xv[U];
#pragma unroll
                    for (int u = 0; u < U; ++u) {
                        const SweepEntry e = ent[(q + (u << lg)) & mask];
                        v[u] = e.val;
                        xv[u] = sx[e.idx * P + p];
                    }
#pragma unroll
                    for (int u = 0; u < U; ++u) acc = fma(v[u], xv[u], acc);
                }
                if (left > 0) {
                    double v[U - 1], xv[U - 1];
#pragma unroll
                    for (int u = 0; u < U - 1; ++u)
                        if (u < left) {
                            const SweepEntry e = ent[(q + (u << lg)) & mask];
                            v[u] = e.val;
                            xv[u] = sx[e.idx * P + p];
                        }
#pragma unroll
                    for (int u = 0; u < U - 1; ++u)
                        if (u < left) acc = fma(v[u], xv[u], acc);
                }
            };
            if (ring) products(rent, SOLVE_RING - 1);
            else products(Q.ent, -1);
            __syncwarp();
            for (int o = min(g, S) >> 1; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o * P);
            if (g <= S) {
                if (r0.i >= 0 && (slot & (g - 1)) == 0) sx[r0.i * P + p] = (sx[r0.i * P + p] - acc) * r0.rd;
            } else {
                // the group's sum over its warps
                const int wg = 1 << (lg - LS);
                if (slot == 0) part[warp * P + p] = acc;
                __syncthreads();
                if (r0.i >= 0 && slot == 0 && (warp & (wg - 1)) == 0) {
                    double v[P];
#pragma unroll
                    for (int c = 0; c < P; ++c) v[c] = c < wg ? part[(warp + c) * P + p] : 0.0;
#pragma unroll
                    for (int o = P / 2; o > 0; o >>= 1)
                        if (o < wg)
#pragma unroll
                            for (int c = 0; c < o; ++c) v[c] += v[c + o];
                    sx[r0.i * P + p] = (sx[r0.i * P + p] - v[0]) * r0.rd;
                }
            }
            // the next step's entries: the copies of this step and of the one
            // before may stay in flight if none of them are among those (none do
            // after a step too large for the ring, whose own copies nobody reads)
            if (ring && s1.w <= mark2) {
                cp_async_wait<2>();
                safe = max(safe, mark2);
            } else if (ring && s1.w <= mark1) {
                cp_async_wait<1>();
                safe = max(safe, mark1);
            } else {
                cp_async_wait<0>();
                safe = issued;
            }
            __syncthreads();
            mark2 = mark1;
            mark1 = issued;
            s0 = s1; s1 = s2; s2 = s3;
            r0 = r1; r1 = r2;
        }
        cp_async_wait<0>();
        __syncthreads();
    };
    __syncthreads();
    sweep(F);
    sweep(B);
    // phi, a warp per particle, and the solution in the observations' order
    if (warp < np) {
        const double* dp = d + (long long)(w0 + warp) * n;
        double* out = x + (long long)(w0 + warp) * n;
        double acc = 0.0;
        for (int i = lane; i < n; i += 32) {
            const int o = perm ? perm[i] : i;
            const double v = sx[i * P + warp];
            acc = fma(dp[o], v, acc);
            out[o] = v;
        }
        acc = warp_sum(acc);
        if (lane == 0) phi[w0 + warp] = acc;
    }
}

constexpr int DOT_THREADS = 256;
constexpr int DOT_BLOCKS_PER_CTA = 8;

// u = (a + 1/2) 2^-32 in one FP64 operation: the bits of 2^20 + a 2^-32 are a
// under a fixed upper word, and the difference is exact
__device__ __forceinline__ double uniform64(uint32_t a)
{
    return __hiloint2double(0x41300000, (int)a) - (0x1p20 - 0x1p-33);
}

// CTA of DOT_THREADS: partial sums of xi^T xi, nu~^T nu~, nu~^T xi of particle
// p over the Philox blocks of slice bx, from the Box-Muller identities: with
// z = r (cos, sin)(pi 2u_b), r^2 = -2 log u_a, a pair adds -2 log u_a to the
// squared norm and, with the pair of the other vector, r_nu r_xi cos(pi
// (2u_b,nu - 2u_b,xi)) to the cross product.
//  * Squared norms in FP64: sum log u = log prod u, a product of the thread's
//    uniforms (at most 16, each at least 2^-33, so far from underflow) and
//    one logarithm for all of them: two FP64 operations per pair instead of a
//    logarithm each, on the few FP64 lanes that bound this kernel.
//  * The cross product's terms need each logarithm: as two floats
//    (log_uniform, 2^-28), so that the product rounds to float as that of two
//    FP64 logarithms does; square root and cosine in FP32, the angle's
//    difference in 32-bit integers, where its period is exact; the product of
//    the two exactly, summed as three floats (two-sums), more bits than a
//    double.  A term's rms error against 64 bits is 0.78e-7; 1.10e-7 with FP64
//    logarithms, the difference rounded to FP32 unreduced and an FP64 sum.
// Bound by the FP64 lanes.  With form_r_block 4.05 ms per 1000 x 208^2 coarse
// points with an FP64 logarithm per pair and a generator per normal, 0.57 ms
// so; the terms added in FP64 (conversions and two operations per block) took
// 0.1 ms more.
__device__ __forceinline__ void rand_dots_cta(uint64_t seed, uint32_t t, uint32_t s_xi, uint32_t s_nu, int NR,
                                              double* __restrict__ partial, int nblk, int p, int bx)
{
    const uint2 key = seed_key(seed);
    const int nq = NR / 4;                           // whole blocks
    double px = 1.0, pn = 1.0;                       // products of the u_a of xi and of nu~
    double tx = 0.0, tn = 0.0, tc = 0.0;             // terms of the last, partial block
    float cs = 0.0f, ce = 0.0f, cg = 0.0f;           // cross product: its sum as three floats
    static_assert(2 * DOT_BLOCKS_PER_CTA * 33 < 1000, "the products stay normal");
    for (int b = bx * DOT_THREADS + threadIdx.x; b < nq; b += nblk * DOT_THREADS) {
        const uint4 wx = philox4x32_10(make_uint4((uint32_t)b, (uint32_t)p, t, s_xi), key);
        const uint4 wn = philox4x32_10(make_uint4((uint32_t)b, (uint32_t)p, t, s_nu), key);
        px *= uniform64(wx.x) * uniform64(wx.z);
        pn *= uniform64(wn.x) * uniform64(wn.z);
        const uint32_t xa[2] = {wx.x, wx.z}, xb[2] = {wx.y, wx.w}, na[2] = {wn.x, wn.z}, nb[2] = {wn.y, wn.w};
#pragma unroll
        for (int l = 0; l < 2; ++l) {
            float xh, xl, nh, nl;
            log_uniform(xa[l], xh, xl);
            log_uniform(na[l], nh, nl);
            const float q = xh * nh;
            const float r = sqrtf(4.0f * (q + (fmaf(xh, nh, -q) + fmaf(xh, nl, xl * nh))));
            const float c = cospif((float)(int)(nb[l] - xb[l]) * 0x1p-31f);
            // s + e = a + b exactly
            auto two_sum = [](float a, float b, float& s, float& e) {
                s = a + b;
                const float bb = s - a;
                e = (a - (s - bb)) + (b - bb);
            };
            const float v = r * c;
            float e1, e2, e3;
            two_sum(cs, v, cs, e1);
            two_sum(ce, e1, ce, e2);
            two_sum(ce, fmaf(r, c, -v), ce, e3);
            cg += e2 + e3;
        }
    }
    // a last block of 1 to 3 normals: its pairs in FP64, one per lane of one warp
    // (pair lane / 2 of xi or, odd lanes, of nu~; one after the other in a thread
    // they were half of the kernel at 64 x 64)
    if (4 * nq < NR && bx == nblk - 1 && threadIdx.x >= DOT_THREADS - 32) {
        const int lane = threadIdx.x & 31;
        double z[2] = {0.0, 0.0};
        if (lane < 4) {
            const uint4 w = philox4x32_10(make_uint4((uint32_t)nq, (uint32_t)p, t, lane & 1 ? s_nu : s_xi), key);
            box_muller64(lane & 2 ? w.z : w.x, lane & 2 ? w.w : w.y, z[0], z[1]);
        }
#pragma unroll
        for (int l = 0; l < 3; ++l) {
            const double x = __shfl_sync(0xffffffffu, z[l & 1], l & 2), v = __shfl_sync(0xffffffffu, z[l & 1], (l & 2) + 1);
            if (lane == 0 && 4 * nq + l < NR) {
                tx = fma(x, x, tx);
                tn = fma(v, v, tn);
                tc = fma(v, x, tc);
            }
        }
    }
    __shared__ double red[3][DOT_THREADS / 32];
    const double xx = warp_sum(fma(-2.0, log(px), tx));
    const double nn = warp_sum(fma(-2.0, log(pn), tn));
    const double nx = warp_sum((((double)cg + (double)ce) + (double)cs) + tc);
    __syncthreads();
    if ((threadIdx.x & 31) == 0) {
        red[0][threadIdx.x >> 5] = xx;
        red[1][threadIdx.x >> 5] = nn;
        red[2][threadIdx.x >> 5] = nx;
    }
    __syncthreads();
    if (threadIdx.x < 3) {
        double s = 0.0;
        for (int w = 0; w < DOT_THREADS / 32; ++w) s += red[threadIdx.x][w];
        partial[((long long)p * nblk + bx) * 3 + threadIdx.x] = s;
    }
}

// -s - log(1 - s) for s in [0, 1): power series s^2 (1/2 + s/3 + ...) below
// 0.1 (terms to s^18; the next is below 2e-18 of the sum), even and odd
// powers as two Horner chains of fused multiply-adds so that their latencies
// overlap; closed form above
__device__ __forceinline__ double phi_s(double s)
{
    if (s < 0.1) {
        const double t = s * s;
        double e = 1.0 / 18, o = 1.0 / 17;
        e = fma(e, t, 1.0 / 16), o = fma(o, t, 1.0 / 15);
        e = fma(e, t, 1.0 / 14), o = fma(o, t, 1.0 / 13);
        e = fma(e, t, 1.0 / 12), o = fma(o, t, 1.0 / 11);
        e = fma(e, t, 1.0 / 10), o = fma(o, t, 1.0 / 9);
        e = fma(e, t, 1.0 / 8), o = fma(o, t, 1.0 / 7);
        e = fma(e, t, 1.0 / 6), o = fma(o, t, 1.0 / 5);
        e = fma(e, t, 1.0 / 4), o = fma(o, t, 1.0 / 3);
        e = fma(e, t, 1.0 / 2);
        return t * fma(o, s, e);
    }
    return -s - log1p(-s);
}

// alpha of eq. iewpfAlphaSol with W_0 solved through its defining equation
// u - 1 - log u = q (u = -W_0), q = (x - 1 - log x) + c*/N_psi, x = gamma/N_psi:
// Newton in s = 1 - u started from the branch-point series
// s = p - p^2/3 + 11 p^3/72 - 43 p^4/540, p = sqrt(2 (1 + e z)) (Corless et
// al. 1996), or in u itself for q > 1/2.  Returns alpha, or NaN on failure.
__device__ __forceinline__ double alpha_lambert(double gamma, double cstar, double N)
{
    const double x = gamma / N;
    const double dl = x - 1.0;
    double q = (dl - log1p(dl)) + fmax(cstar, 0.0) / N;
    if (!(q >= 0.0) || !isfinite(q)) return nan("");
    double u;
    if (q == 0.0) {
        u = 1.0;
    } else if (q <= 0.5) {
        const double pp = sqrt(-2.0 * expm1(-q));
        double s = pp * (1.0 + pp * (-1.0 / 3.0 + pp * (11.0 / 72.0 - pp * (43.0 / 540.0))));
        s = fmin(fmax(s, 0.0), 0.999);
        for (int it = 0; it < 8; ++it) {
            const double f = phi_s(s) - q;
            const double fp = s / (1.0 - s);
            if (fp <= 0.0) break;
            const double ds = f / fp;
            double sn = s - ds;
            if (sn <= 0.0) sn = 0.5 * s;
            else if (sn >= 1.0) sn = 0.5 * (s + 1.0);
            // a Newton step of relative size e leaves a relative error of
            // e^2 / (2 (1 - s)): below 1e-9 the step just taken was the last
            else if (fabs(ds) <= 1e-9 * s) {
                s = sn;
                break;
            }
            s = sn;
        }
        u = 1.0 - s;
    } else {
        u = exp(-1.0 - q);
        for (int it = 0; it < 60; ++it) {
            const double f = u - 1.0 - log(u) - q;
            const double fp = 1.0 - 1.0 / u;
            double un = u - f / fp;
            if (un <= 0.0) un = 0.5 * u;
            if (un >= 1.0) un = 0.5 * (u + 1.0);
            if (un == u) break;
            u = un;
        }
    }
    return u / x;
}

__device__ __forceinline__ void block_sum_min(double v_sum, double v_min, double* s_out, double* m_out)
{
    __shared__ double ws[32], wm[32];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    double s = warp_sum(v_sum);
    double m = v_min;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) m = fmin(m, __shfl_xor_sync(0xffffffffu, m, o));
    __syncthreads();
    if (lane == 0) {
        ws[w] = s;
        wm[w] = m;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        double ts = 0.0, tm = INFINITY;
        for (int i = 0; i < (int)(blockDim.x >> 5); ++i) {
            ts += ws[i];
            tm = fmin(tm, wm[i]);
        }
        *s_out = ts;
        *m_out = tm;
    }
    __syncthreads();
}

// Schemes of the ensemble-wide step: the two-stage IEWPF (App. A, eqs.
// betaTwoStage, cistarTwoStage) and the one-stage IEWPF (App. A, eqs.
// iewpf_targetWeight, iewpfCStar), which has no nu and so no beta.
constexpr int TWO_STAGE = 0;
constexpr int ONE_STAGE = 1;

// CTA: the ensemble-wide step for the particles [i0, i1).  Two-stage:
// w_target = mean c_i, beta, c*, alpha, -log w.  One-stage: w_target = max
// c_i, beta reported as 0 (the nu term of the posterior vanishes with it),
// c* = w_target - c_i, alpha, -log w.  scal[0] = w_target, scal[1] = beta,
// scal[2] = mean c_i.  cval(i), zval(i): c_i and zeta_i of any particle;
// gamma, zeta of the slice are read from the arrays.  The two ensemble-wide
// reductions (mean or maximum of c, minimum of beta's candidates) run over
// all particles in every CTA, in the same order, so that CTAs with different
// slices need no synchronisation and hold the same target and beta.
template <class FC, class FZ>
__device__ __forceinline__ void weights_slice_cta(FC cval, FZ zval, const double* gamma, const double* zeta, int ne,
                                                  int i0, int i1, double N, int scheme, double* alpha,
                                                  double* cstar, double* neglogw, double* scal, int* flag)
{
    __shared__ double s_sum, s_min;
    const bool one = scheme == ONE_STAGE;
    double acc = 0.0, mc = INFINITY;
    bool bad = false;
    for (int i = threadIdx.x; i < ne; i += blockDim.x) {
        const double c = cval(i);
        acc += c;
        mc = fmin(mc, -c);
        bad |= !isfinite(c);
    }
    for (int i = i0 + threadIdx.x; i < i1; i += blockDim.x) bad |= !isfinite(gamma[i]) || (!one && !isfinite(zeta[i]));
    bad = __syncthreads_or(bad);
    block_sum_min(acc, mc, &s_sum, &s_min);
    const double cmean = s_sum / ne;
    const double target = one ? -s_min : cmean;
    double beta = 0.0;
    if (!one) {
        double mn = INFINITY;
        for (int i = threadIdx.x; i < ne; i += blockDim.x) mn = fmin(mn, (target - cval(i)) / zval(i) + 1.0);
        block_sum_min(0.0, mn, &s_sum, &s_min);
        beta = s_min;
    }
    bool dom = false;
    for (int i = i0 + threadIdx.x; i < i1; i += blockDim.x) {
        const double c = cval(i), g = gamma[i];
        const double cs = one ? target - c : target - c - (beta - 1.0) * zeta[i];
        const double a = alpha_lambert(g, cs, N);
        dom |= !(a > 0.0) || !isfinite(a);
        alpha[i] = a;
        cstar[i] = cs;
        if (neglogw) {
            const double t = (a - 1.0) * g - N * log(a);
            neglogw[i] = one ? t + c : t + (beta - 1.0) * zeta[i] + c;
        }
    }
    dom = __syncthreads_or(dom);
    if (threadIdx.x == 0) {
        if (i0 == 0) {
            scal[0] = target;
            scal[1] = beta;
            scal[2] = cmean;
        }
        int f = 0;
        if (bad) f |= FLAG_NONFINITE;
        if (!(beta >= 0.0)) f |= FLAG_BETA;
        if (dom) f |= FLAG_DOMAIN;
        if (f) atomicOr(flag, f);
    }
}

// the same on given arrays of all particles, one CTA
__device__ __forceinline__ void weights_cta(const double* c, const double* gamma, const double* zeta, int ne,
                                            double N, int scheme, double* alpha, double* cstar, double* neglogw,
                                            double* scal, int* flag)
{
    weights_slice_cta([&](int i) { return c[i]; }, [&](int i) { return zeta[i]; }, gamma, zeta, ne, 0, ne, N, scheme,
                      alpha, cstar, neglogw, scal, flag);
}

// CTAs of SYNC_THREADS, one per slice [i0, i1) of the particles: gamma, zeta,
// a, the length scale and c of the slice from the partial dot products, then
// the weights step.  What other slices need of a particle (c_i and zeta_i)
// each CTA forms again from phi and the partial sums, by the same operations.
constexpr int SYNC_THREADS = 256;
__device__ __forceinline__ void sync_alpha_cta(const double* __restrict__ phi, const double* __restrict__ partial,
                                               int nblk, int ne, int i0, int i1, double NR, double N, double logNe,
                                               int scheme, double* c, double* gamma, double* zeta, double* alpha,
                                               double* cstar, double* neglogw, double* coef, double* scal, int* flag)
{
    auto cval = [&](int i) { return phi[i] + logNe; };              // eq. iewpf_ci
    auto zval = [&](int i) {
        double nn = 0.0;
        for (int b = 0; b < nblk; ++b) nn += partial[((long long)i * nblk + b) * 3 + 1];
        return nn * N / NR;                                          // eq. scalingGammaZeta
    };
    for (int i = i0 + threadIdx.x; i < i1; i += blockDim.x) {
        double xx = 0.0, nn = 0.0, nx = 0.0;
        for (int b = 0; b < nblk; ++b) {
            xx += partial[((long long)i * nblk + b) * 3 + 0];
            nn += partial[((long long)i * nblk + b) * 3 + 1];
            nx += partial[((long long)i * nblk + b) * 3 + 2];
        }
        const double a = nx / xx;                                    // eq. nuPerpendicular
        coef[2 * i] = a;
        coef[2 * i + 1] = sqrt(nn / (nn - a * nx));
        gamma[i] = xx * N / NR;                                      // eq. scalingGammaZeta
        zeta[i] = nn * N / NR;
        c[i] = cval(i);
    }
    __syncthreads();
    weights_slice_cta(cval, zval, gamma, zeta, ne, i0, i1, N, scheme, alpha, cstar, neglogw, scal, flag);
}

// r = beta^{1/2} nu + alpha^{1/2} xi at the four coarse points of Philox block
// q of particle p, nu = s (nu~ - a xi).  One thread per block: a block holds
// four normals (the numbers normal32 returns one by one), so a thread per
// point would run every generator four times.
__device__ __forceinline__ void form_r_block(uint64_t seed, uint32_t t, uint32_t s_xi, uint32_t s_nu, int NR,
                                             const double* __restrict__ coef, const double* __restrict__ scal,
                                             const double* __restrict__ alpha, float* __restrict__ r, int p, int q)
{
    const uint2 key = seed_key(seed);
    const uint4 wx = philox4x32_10(make_uint4((uint32_t)q, (uint32_t)p, t, s_xi), key);
    const uint4 wn = philox4x32_10(make_uint4((uint32_t)q, (uint32_t)p, t, s_nu), key);
    float xi[4], nut[4], v[4];
    box_muller32(wx.x, wx.y, xi[0], xi[1]);
    box_muller32(wx.z, wx.w, xi[2], xi[3]);
    box_muller32(wn.x, wn.y, nut[0], nut[1]);
    box_muller32(wn.z, wn.w, nut[2], nut[3]);
    const float a = (float)coef[2 * p], sc = (float)coef[2 * p + 1];
    // square roots in FP32 (the factors enter an FP32 field; an FP64 square
    // root per block would cost more than the rest of the kernel)
    const float sb = sqrtf((float)fmax(scal[1], 0.0)), sa = sqrtf((float)alpha[p]);
#pragma unroll
    for (int l = 0; l < 4; ++l) v[l] = fmaf(sb, sc * fmaf(-a, xi[l], nut[l]), sa * xi[l]);
    float* __restrict__ o = r + (long long)p * NR + 4LL * q;
    if ((NR & 3) == 0) {
        *reinterpret_cast<float4*>(o) = make_float4(v[0], v[1], v[2], v[3]);
    } else {
#pragma unroll
        for (int l = 0; l < 4; ++l)
            if (4 * q + l < NR) o[l] = v[l];
    }
}

// Local blocks r_l <- M49 r_l (7 x 7 coarse points around an observation), a
// warp per block: lane t computes outputs t and t + 32 (< 49), its two rows
// of M49 in registers, the 49 inputs read from shared memory four at a time.
// A block costs the round trip of its inputs to L2 and 49 dependent products;
// the inputs of the next block are loaded during the products where the two
// share no point.
struct BlockRoot {
    float m0[49], m1[49];
    __device__ __forceinline__ void load(const float* __restrict__ M49)
    {
        const int lane = threadIdx.x & 31;
#pragma unroll
        for (int j = 0; j < 49; ++j) {
            m0[j] = __ldg(M49 + lane * 49 + j);
            m1[j] = lane + 32 < 49 ? __ldg(M49 + (lane + 32) * 49 + j) : 0.0f;
        }
    }
};
struct BlockIn {
    int i0, i1;      // this lane's points
    float x0, x1;    // and their values
    __device__ __forceinline__ void place(int2 c, int nRx, int nRy)
    {
        const int lane = threadIdx.x & 31, t1 = lane + 32 < 49 ? lane + 32 : 48;
        auto wrap = [](int a, int n) { return a < 0 ? a + n : (a >= n ? a - n : a); };
        i0 = wrap(c.y + lane / 7 - 3, nRy) * nRx + wrap(c.x + lane % 7 - 3, nRx);
        i1 = wrap(c.y + t1 / 7 - 3, nRy) * nRx + wrap(c.x + t1 % 7 - 3, nRx);
    }
    __device__ __forceinline__ void fetch(const float* rp)
    {
        // (volatile: issued here, ahead of the products of the block before)
        asm volatile("ld.global.f32 %0, [%1];" : "=f"(x0) : "l"(rp + i0) : "memory");
        asm volatile("ld.global.f32 %0, [%1];" : "=f"(x1) : "l"(rp + i1) : "memory");
    }
};
// v: 52 floats of shared memory, 16-byte aligned, owned by the warp
__device__ __forceinline__ void block_product(const BlockRoot& M, const BlockIn& B, float* v, float& a0, float& a1)
{
    const int lane = threadIdx.x & 31;
    v[lane] = B.x0;
    if (lane + 32 < 49) v[lane + 32] = B.x1;
    __syncwarp();
    a0 = a1 = 0.0f;
#pragma unroll
    for (int q = 0; q < 13; ++q) {
        const float4 w = *reinterpret_cast<const float4*>(v + 4 * q);
        const float c[4] = {w.x, w.y, w.z, w.w};
#pragma unroll
        for (int u = 0; u < 4; ++u)
            if (4 * q + u < 49) {
                a0 = fmaf(M.m0[4 * q + u], c[u], a0);
                a1 = fmaf(M.m1[4 * q + u], c[u], a1);
            }
    }
    __syncwarp();
}

// warp: the blocks of particle p in observation order.  Blocks that follow
// each other mostly share points, so a block's inputs are loaded two blocks
// ahead and those of the two blocks before it, then written, come from their
// outputs in shared memory (v: 3 x 52 floats, 16-byte aligned): a block costs
// its products, not the round trip through L2 of its predecessor's outputs.
__device__ __forceinline__ void block_seq_warp(float* r, int NR, const float* __restrict__ M49,
                                               const int* __restrict__ block0, int nobs, int nRx, int nRy, int p,
                                               float* v)
{
    if (nobs <= 0) return;
    const int lane = threadIdx.x & 31, t1 = lane + 32 < 49 ? lane + 32 : 48;
    float* rp = r + (long long)p * NR;
    const int2* cells = reinterpret_cast<const int2*>(block0);
    BlockRoot M;
    M.load(M49);
    const int lx0 = lane % 7, ly0 = lane / 7, lx1 = t1 % 7, ly1 = t1 / 7;
    // the block's place relative to another's, in (-n / 2, n / 2]
    auto offset = [](int a, int b, int n) {
        const int d = a - b;
        return 2 * d > n ? d - n : (2 * d <= -n ? d + n : d);
    };
    int2 cm = cells[0], c0 = cm, c1 = cells[min(1, nobs - 1)], c2 = cells[min(2, nobs - 1)];
    // blocks ahead whose inputs are brought to L2 (DRAM takes longer than two blocks)
    constexpr int SEQ_AHEAD = 8;
    int2 ca = cells[min(SEQ_AHEAD, nobs - 1)];
    BlockIn cur, nxt;
    cur.place(c0, nRx, nRy);
    cur.fetch(rp);
    nxt.place(c1, nRx, nRy);
    nxt.fetch(rp);
    float* const out0 = v + 52;
#pragma unroll 4
    for (int l = 0; l < nobs; ++l) {
        const int2 c3 = cells[min(l + 3, nobs - 1)];
        if (l + SEQ_AHEAD < nobs) {
            BlockIn q;
            q.place(ca, nRx, nRy);
            asm volatile("prefetch.global.L2 [%0];" ::"l"(rp + q.i0));
            asm volatile("prefetch.global.L2 [%0];" ::"l"(rp + q.i1));
            ca = cells[min(l + 1 + SEQ_AHEAD, nobs - 1)];
        }
        BlockIn far;
        far.place(c2, nRx, nRy);
        far.fetch(rp);
        float a0, a1;
        block_product(M, cur, v, a0, a1);
        const int cur0 = 52 * (l & 1);
        rp[cur.i0] = a0;
        out0[cur0 + lane] = a0;
        if (lane + 32 < 49) {
            rp[cur.i1] = a1;
            out0[cur0 + lane + 32] = a1;
        }
        __syncwarp();
        // the next block's inputs were loaded before this block and the one before wrote
        const int dx = offset(c1.x, c0.x, nRx), dy = offset(c1.y, c0.y, nRy);
        const int ex = offset(c1.x, cm.x, nRx), ey = offset(c1.y, cm.y, nRy);
        auto latest = [&](int t, int lx, int ly, float g) {
            const bool in0 = ((unsigned)(lx + dx) < 7u) & ((unsigned)(ly + dy) < 7u);
            const bool inm = ((unsigned)(lx + ex) < 7u) & ((unsigned)(ly + ey) < 7u) & (l > 0);
            const int k = in0 ? cur0 + 7 * dy + dx + t : (inm ? (52 - cur0) + 7 * ey + ex + t : 0);
            const float w = out0[k];
            return in0 | inm ? w : g;
        };
        cur.i0 = nxt.i0;
        cur.i1 = nxt.i1;
        cur.x0 = latest(lane, lx0, ly0, nxt.x0);
        cur.x1 = latest(t1, lx1, ly1, nxt.x1);
        nxt = far;
        cm = c0; c0 = c1; c1 = c2; c2 = c3;
    }
}

}  // namespace ana
}  // namespace iewpf

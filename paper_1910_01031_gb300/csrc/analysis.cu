// IEWPF analysis kernels for one problem per launch (Sec. 4 and App. A of
// arXiv 1910.01031); the device code is in analysis_dev.cuh.
#include <algorithm>
#include <type_traits>
#include <vector>

#include "analysis_dev.cuh"
#include "tc_dev.cuh"

namespace iewpf {

namespace {

// dynamic shared memory of cholesky_small_kernel (n <= 159) at most
constexpr int kCholSmem = 212 * 1024;
// dynamic shared memory of a CTA of the grouped sweeps at most
constexpr int kSolveGroupSmem = 224 * 1024;
static_assert(ana::solve_group_smem<4>((int)(kSolveSmemBytes / sizeof(double))) > kSolveGroupSmem,
              "a layout that fits a group fits a warp");

__global__ void obs_cells_kernel(const double* __restrict__ xy, int nobs, Grid G, Coarse C, double dx, double dy,
                                 int* __restrict__ cell, int* __restrict__ block0)
{
    const int l = blockIdx.x * blockDim.x + threadIdx.x;
    if (l < nobs) ana::obs_cell_one(xy, l, G, C, dx, dy, cell, block0);
}

__global__ void __launch_bounds__(NTHREADS)
tile_bin_kernel(const int* __restrict__ cell, int nobs, Grid G, int R, int* __restrict__ cnt, int* __restrict__ list,
                int cap, int* __restrict__ flag)
{
    ana::tile_bin_cta(cell, nobs, G, R, blockIdx.x, cnt, list, cap, flag);
}

__global__ void innovate_kernel(const float* __restrict__ b0, const float* __restrict__ b1,
                                const int* __restrict__ par, const int* __restrict__ cell,
                                const double* __restrict__ y, int nobs, Grid G, double H, double* __restrict__ d)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < G.ne * nobs) ana::innovate_one(b0, b1, par, cell, y, nobs, G, H, d, i);
}

__global__ void hqht_kernel(const double* __restrict__ K, int R, const int* __restrict__ cell, int nobs, Grid G,
                            int dense, double sigma2, double* __restrict__ M)
{
    const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (i < 4LL * nobs * nobs) ana::hqht_one(K, R, cell, nobs, G, dense, sigma2, M, i);
}

__global__ void __launch_bounds__(1024)
cholesky_kernel(double* __restrict__ A, int n, int* __restrict__ colptr, int* rowidx, int* __restrict__ flag,
                int* nzlist, double* __restrict__ rdiag, int* plan)
{
    ana::cholesky_cta(A, n, colptr, rowidx, flag, nzlist);
    ana::solve_plan_cta<false>(A, n, n, colptr, rowidx, rdiag, plan);
}

// the same factorisation on a copy in shared memory (n rows of an odd
// number of doubles, then chol_levels_ints(n) >= n ints)
__global__ void __launch_bounds__(1024)
cholesky_small_kernel(double* __restrict__ A, int n, int* __restrict__ colptr, int* __restrict__ rowidx,
                      int* __restrict__ flag, double* __restrict__ rdiag, int* plan)
{
    extern __shared__ double sA[];
    const int ld = n | 1;
    int* work = reinterpret_cast<int*>(sA + n * ld);
    __shared__ int bad;
    if (threadIdx.x == 0) bad = 0;
    for (int q = threadIdx.x; q < n * n; q += blockDim.x) sA[q / n * ld + q % n] = A[q];
    __syncthreads();
    if (!ana::cholesky_levels_cta(sA, n, ld, work, &bad)) ana::cholesky_factor_cta(sA, n, ld, work, &bad);
    for (int q = threadIdx.x; q < n * n; q += blockDim.x) A[q] = sA[q / n * ld + q % n];
    ana::csc_cta(sA, n, ld, colptr, rowidx);
    ana::solve_plan_cta<true>(sA, n, ld, colptr, rowidx, rdiag, plan);
    if (threadIdx.x == 0 && bad) atomicOr(flag, FLAG_NOTPD);
}

// the factor's values below the diagonal in the order of the plan's CSR (Lr)
// and of the CSC (Lc): a warp per row and per column of the dense factor
__global__ void pack_factor_kernel(const double* __restrict__ L, int n, const int* __restrict__ colptr,
                                   const int* __restrict__ rowidx, const int* plan, double* __restrict__ Lr,
                                   double* __restrict__ Lc)
{
    const ana::SolvePlan P = ana::solve_plan_view(const_cast<int*>(plan), n);
    const int lane = threadIdx.x & 31;
    const int nw = (gridDim.x * blockDim.x) >> 5;
    for (int i = (blockIdx.x * blockDim.x + threadIdx.x) >> 5; i < n; i += nw) {
        for (int q = P.rowptr[i] + lane; q < P.rowptr[i + 1]; q += 32) Lr[q] = L[(long long)i * n + P.colidx[q]];
        for (int q = colptr[i] + lane; q < colptr[i + 1]; q += 32) Lc[q] = L[(long long)rowidx[q] * n + i];
    }
}

__global__ void solve_kernel(const double* __restrict__ L, const int* __restrict__ colptr,
                             const int* __restrict__ rowidx, const double* __restrict__ rdiag,
                             const int* __restrict__ plan, int n, const double* __restrict__ d,
                             double* __restrict__ x, double* __restrict__ phi, int ne, const int* __restrict__ perm,
                             double* __restrict__ scratch, const double* __restrict__ Lr, const double* __restrict__ Lc)
{
    const int warp = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    if (warp < ne)
        ana::solve_levels_warp(L, colptr, rowidx, rdiag, plan, n, d, x, phi, warp, perm, scratch, Lr, Lc);
}

// the same with a CTA of one warp per particle and its vector in shared
// memory (n doubles)
__global__ void __launch_bounds__(32)
solve_smem_kernel(const double* __restrict__ L, const int* __restrict__ colptr, const int* __restrict__ rowidx,
                  const double* __restrict__ rdiag, const int* __restrict__ plan, int n, const double* __restrict__ d,
                  double* __restrict__ x, double* __restrict__ phi, const int* __restrict__ perm,
                  const double* __restrict__ Lr, const double* __restrict__ Lc)
{
    extern __shared__ double sx[];
    ana::solve_levels_warp(L, colptr, rowidx, rdiag, plan, n, d, x, phi, blockIdx.x, perm, nullptr, Lr, Lc, sx);
}

// the factor in the order of the sweeps: rows, diagonals and steps of both
// directions (a warp each), then the entries (a warp per position)
__global__ void __launch_bounds__(32)
sweep_rows_kernel(const int* plan, int n, int nnz, const double* __restrict__ rdiag, void* stream)
{
    const ana::SolvePlan P = ana::solve_plan_view(const_cast<int*>(plan), n);
    const bool back = blockIdx.x;
    const ana::SweepStream S =
        ana::sweep_stream_view(static_cast<char*>(stream) + back * ana::sweep_stream_bytes(n, nnz), n, nnz);
    ana::sweep_rows_warp(back ? P.rb : P.rf, back ? P.bptr : P.fptr, P.nlev[back], n, rdiag, S);
}
__global__ void sweep_entries_kernel(const double* __restrict__ L, const int* plan, int n, int nnz,
                                     const int* __restrict__ rowidx, void* stream)
{
    const ana::SolvePlan P = ana::solve_plan_view(const_cast<int*>(plan), n);
    const bool back = blockIdx.y;
    const ana::SweepStream S =
        ana::sweep_stream_view(static_cast<char*>(stream) + back * ana::sweep_stream_bytes(n, nnz), n, nnz);
    const int lane = threadIdx.x & 31;
    for (int t = (blockIdx.x * blockDim.x + threadIdx.x) >> 5; t < n; t += (gridDim.x * blockDim.x) >> 5) {
        const int4 r = S.row[t];
        const int q0 = (back ? P.rb : P.rf)[3 * t + 1];
        for (int q = lane; q < r.z - r.y; q += 32) {
            const int j = (back ? rowidx : P.colidx)[q0 + q];
            S.ent[r.y + q] = {back ? L[(long long)j * n + r.x] : L[(long long)r.x * n + j], j, 0};
        }
    }
}

// P particles per CTA.  The sweeps are a chain of levels (2 x 544 for 1521
// coupled moorings), each a barrier and the FP64 latency of its longest sum;
// the warp per particle of solve_smem_kernel also waited on L2 for every
// level's entries, which it read for that particle alone (1000 particles: 5.5
// ms, now 3.4; FP64 pipe active half of the time)
template <int P>
__global__ void __launch_bounds__(32 * P)
solve_group_kernel(const void* stream, int n, int nnz, const double* __restrict__ d, double* __restrict__ x,
                   double* __restrict__ phi, int ne, const int* __restrict__ perm)
{
    extern __shared__ __align__(16) double group_smem[];
    char* base = static_cast<char*>(const_cast<void*>(stream));
    ana::solve_group_cta<P>(ana::sweep_stream_view(base, n, nnz),
                            ana::sweep_stream_view(base + ana::sweep_stream_bytes(n, nnz), n, nnz), n, nnz, d, x, phi,
                            blockIdx.x * P, ne, perm, group_smem);
}

__global__ void __launch_bounds__(ana::DOT_THREADS)
rand_dots_kernel(uint64_t seed, uint32_t t, uint32_t s_xi, uint32_t s_nu, int NR, double* __restrict__ partial,
                 int nblk)
{
    ana::rand_dots_cta(seed, t, s_xi, s_nu, NR, partial, nblk, blockIdx.y, blockIdx.x);
}

// A slice of particles per CTA.  The step is a serial chain of FP64 (two
// reductions, then the Lambert-W solve of each particle), so its time is
// latency at small ensembles and the few FP64 lanes of an SM at large ones: the
// alpha solves are spread over many SMs and the reductions, cheap next to
// them, repeated in each.
// One CTA of 1024 threads, a division per series term: 144 us at 10 and 100
// particles, 896 us at 1000; in slices, with the series by Horner, 22 us at 10
// and 100 and 30 us at 1000 (analysis of 64^2 x 10: 379 -> 272 us, of 624^2 x 1000: 26.60
// -> 25.74 ms).
__global__ void __launch_bounds__(ana::SYNC_THREADS)
sync_alpha_kernel(const double* __restrict__ phi, const double* __restrict__ partial, int nblk, int ne, int slice,
                  double NR, double N, double logNe, int scheme, double* c, double* gamma, double* zeta,
                  double* alpha, double* cstar, double* neglogw, double* coef, double* scal, int* flag)
{
    const int i0 = blockIdx.x * slice;
    ana::sync_alpha_cta(phi, partial, nblk, ne, i0, min(ne, i0 + slice), NR, N, logNe, scheme, c, gamma, zeta, alpha,
                        cstar, neglogw, coef, scal, flag);
}

__global__ void __launch_bounds__(1024)
weights_kernel(const double* c, const double* gamma, const double* zeta, int ne, double N, int scheme,
               double* alpha, double* cstar, double* neglogw, double* scal, int* flag)
{
    ana::weights_cta(c, gamma, zeta, ne, N, scheme, alpha, cstar, neglogw, scal, flag);
}

__global__ void form_r_kernel(uint64_t seed, uint32_t t, uint32_t s_xi, uint32_t s_nu, int NR,
                              const double* __restrict__ coef, const double* __restrict__ scal,
                              const double* __restrict__ alpha, float* __restrict__ r)
{
    const int q = blockIdx.x * blockDim.x + threadIdx.x;
    if (4 * q < NR) ana::form_r_block(seed, t, s_xi, s_nu, NR, coef, scal, alpha, r, blockIdx.y, q);
}

// blocks that follow each other in every particle (positions that change each
// cycle): a warp per particle; two barriers and a round trip per block before
// (64 drifters x 100: 85 us, now 32)
__global__ void __launch_bounds__(32)
block_seq_kernel(float* __restrict__ r, int NR, const float* __restrict__ M49, const int* __restrict__ block0, int nobs,
                 int nRx, int nRy)
{
    __shared__ __align__(16) float v[3 * 52];
    ana::block_seq_warp(r, NR, M49, block0, nobs, nRx, nRy, blockIdx.x, v);
}

// all levels of the local blocks of particle blockIdx.x: the CTA's warps
// share the blocks of a level (cells: their places, level by level), a barrier
// separates the levels.  Bound by latency: enough warps per particle to fill
// the chip and the next block's inputs in flight (1521 blocks x 256 particles
// on one level: 755 us with 2 warps, now 134)
constexpr int BL_WARPS = 16;
__global__ void __launch_bounds__(32 * BL_WARPS)
block_levels_kernel(float* r, int NR, const float* __restrict__ M49, const int2* __restrict__ cells,
                    const int* __restrict__ level_off, int nlev, int nRx, int nRy)
{
    __shared__ __align__(16) float v[BL_WARPS][52];
    const int lane = threadIdx.x & 31, wl = threadIdx.x >> 5, nw = blockDim.x >> 5;
    ana::BlockRoot M;
    M.load(M49);
    float* rp = r + (long long)blockIdx.x * NR;
    for (int lev = 0; lev < nlev; ++lev) {
        const int hi = level_off[lev + 1];
        int ib = level_off[lev] + wl;
        ana::BlockIn cur, nxt;
        int2 c1 = make_int2(0, 0);
        if (ib < hi) {
            cur.place(cells[ib], nRx, nRy);
            cur.fetch(rp);
            c1 = cells[min(ib + nw, hi - 1)];
        }
        for (; ib < hi; ib += nw) {
            nxt.place(c1, nRx, nRy);
            if (ib + nw < hi) {
                nxt.fetch(rp);
                c1 = cells[min(ib + 2 * nw, hi - 1)];
            }
            float a0, a1;
            ana::block_product(M, cur, v[wl], a0, a1);
            rp[cur.i0] = a0;
            if (lane + 32 < 49) rp[cur.i1] = a1;
            cur = nxt;
        }
        __syncthreads();     // the next level reads what this one wrote
    }
}

__global__ void philox_blocks_kernel(uint64_t seed, uint32_t p, uint32_t t, uint32_t stream, long long n,
                                     uint4* __restrict__ out)
{
    const long long b = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (b >= n) return;
    out[b] = philox4x32_10(make_uint4((uint32_t)b, p, t, stream), seed_key(seed));
}

__global__ void normals_kernel(uint64_t seed, uint32_t p, uint32_t t, uint32_t stream, long long n,
                               double* __restrict__ o64, float* __restrict__ o32)
{
    const long long m = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (m >= n) return;
    const uint2 key = seed_key(seed);
    const uint4 w = philox4x32_10(make_uint4((uint32_t)(m >> 2), p, t, stream), key);
    const bool hi = (m & 2) != 0;
    const uint32_t a = hi ? w.z : w.x, b = hi ? w.w : w.y;
    if (o64) {
        double z0, z1;
        box_muller64(a, b, z0, z1);
        o64[m] = (m & 1) ? z1 : z0;
    }
    if (o32) o32[m] = normal32(key, p, t, stream, (uint32_t)m);
}

}  // namespace

cudaError_t launch_obs_setup(const double* xy, int nobs, const Grid& G, const Coarse& C, double dx, double dy,
                             int R, int* obs_cell, int* obs_block0, int* tile_cnt, int* tile_obs, int tile_cap,
                             int* flag, cudaStream_t st)
{
    if (nobs > 0) obs_cells_kernel<<<(nobs + 127) / 128, 128, 0, st>>>(xy, nobs, G, C, dx, dy, obs_cell, obs_block0);
    const int ntiles = ((G.nx + OBS_TX - 1) / OBS_TX) * ((G.ny + OBS_TY - 1) / OBS_TY);
    tile_bin_kernel<<<ntiles, NTHREADS, 0, st>>>(obs_cell, nobs, G, R, tile_cnt, tile_obs, tile_cap, flag);
    return cudaGetLastError();
}

cudaError_t launch_innovate(const float* b0, const float* b1, const int* par, const int* obs_cell,
                            const double* y, int nobs, const Grid& G, double H, double* d, cudaStream_t st)
{
    const int n = G.ne * nobs;
    if (n > 0) innovate_kernel<<<(n + 127) / 128, 128, 0, st>>>(b0, b1, par, obs_cell, y, nobs, G, H, d);
    return cudaGetLastError();
}

cudaError_t launch_hqht(const double* K64, int R, const int* obs_cell, int nobs, const Grid& G, int dense,
                        double sigma2, double* M, cudaStream_t st)
{
    const long long n = 2LL * nobs * 2 * nobs;
    if (n > 0) hqht_kernel<<<(unsigned)((n + 255) / 256), 256, 0, st>>>(K64, R, obs_cell, nobs, G, dense, sigma2, M);
    return cudaGetLastError();
}

cudaError_t launch_cholesky(double* M, int n, int* colptr, int* rowidx, int* flag, double* rdiag, int* plan,
                            cudaStream_t st)
{
    // small systems (drifter layouts change every cycle) factor in shared memory
    const size_t smem = (size_t)n * n * sizeof(double) + (size_t)n * sizeof(int);
    if (n >= 1 && smem <= 200 * 1024) {
        cudaError_t e = tc::smem_attr_once<cholesky_small_kernel>(kCholSmem);
        if (e != cudaSuccess) return e;
        const size_t bytes = (size_t)n * (n | 1) * sizeof(double) + ana::chol_levels_ints(n) * sizeof(int);
        cholesky_small_kernel<<<1, 1024, bytes, st>>>(M, n, colptr, rowidx, flag, rdiag, plan);
        return cudaGetLastError();
    }
    // rowidx doubles as the per-column work list during the factorisation
    cholesky_kernel<<<1, 1024, 0, st>>>(M, n, colptr, rowidx, flag, rowidx, rdiag, plan);
    return cudaGetLastError();
}

// Several particles per CTA where their vectors fit its shared memory (n <=
// 6140 for 4, 3064 for 8) and that takes at most 3 / 2 as many waves of CTAs as
// a warp each does (a wave of 1521 coupled moorings, n = 3042: 3.4 ms against
// 5.5), and of 4 and 8 the one with fewer waves (4 at a tie: 5350 against 5624 us
// per analysis of 100 particles; of 1000, 8 takes one wave and 13.2 ms, 4 two
// and 16.0, a warp each 15.4).  Where a group fits, a warp's vector does too
// (solve_smem_kernel), so that kernel's shared memory sets the waves compared
// with.
int solve_group(int n, int ne, int sms)
{
    // 16 warps of these kernels are resident per SM
    auto waves = [&](int P, size_t smem) {
        const size_t resident = std::min((size_t)16 / P, (size_t)(228 * 1024) / (smem + 1024));
        return ((size_t)(ne + P - 1) / P + sms * resident - 1) / (sms * resident);
    };
    const size_t s4 = ana::solve_group_smem<4>(n), s8 = ana::solve_group_smem<8>(n);
    if (s4 > kSolveGroupSmem) return 1;
    const size_t w1 = waves(1, (size_t)n * sizeof(double)), w4 = waves(4, s4);
    const size_t w8 = s8 <= kSolveGroupSmem ? waves(8, s8) : w4 + 1;
    if (2 * std::min(w4, w8) > 3 * w1) return 1;
    return w4 <= w8 ? 4 : 8;
}

cudaError_t launch_solve(const double* L, const int* colptr, const int* rowidx, const double* rdiag, const int* plan,
                         int n, const double* d, double* Sd, double* phi, int ne, cudaStream_t st, const int* perm,
                         double* scratch, const double* Lr, const double* Lc, const void* stream, int nnz)
{
    if ((perm && !scratch) || (!Lr != !Lc)) return cudaErrorInvalidValue;
    if (ne <= 0) return cudaSuccess;
    if (stream && n > 0) {
        auto group = [&](auto Pc) {
            constexpr int P = decltype(Pc)::value;
            cudaError_t e = tc::smem_attr_once<solve_group_kernel<P>>(kSolveGroupSmem);
            if (e != cudaSuccess) return e;
            solve_group_kernel<P><<<(ne + P - 1) / P, 32 * P, ana::solve_group_smem<P>(n), st>>>(stream, n, nnz, d, Sd,
                                                                                                phi, ne, perm);
            return cudaGetLastError();
        };
        const int P = solve_group(n, ne, tc::sm_count());
        if (P == 4) return group(std::integral_constant<int, 4>());
        if (P == 8) return group(std::integral_constant<int, 8>());
    }
    if (n > 0 && (size_t)n * sizeof(double) <= kSolveSmemBytes) {
        solve_smem_kernel<<<ne, 32, (size_t)n * sizeof(double), st>>>(L, colptr, rowidx, rdiag, plan, n, d, Sd, phi,
                                                                       perm, Lr, Lc);
        return cudaGetLastError();
    }
    const int threads = 128;
    const int blocks = (ne * 32 + threads - 1) / threads;
    solve_kernel<<<blocks, threads, 0, st>>>(L, colptr, rowidx, rdiag, plan, n, d, Sd, phi, ne, perm, scratch, Lr,
                                             Lc);
    return cudaGetLastError();
}

cudaError_t launch_pack_factor(const double* L, int n, const int* colptr, const int* rowidx, const int* plan,
                               double* Lr, double* Lc, cudaStream_t st)
{
    if (n <= 0) return cudaSuccess;
    const int threads = 256;
    const int blocks = std::min((n * 32 + threads - 1) / threads, 65535);
    pack_factor_kernel<<<blocks, threads, 0, st>>>(L, n, colptr, rowidx, plan, Lr, Lc);
    return cudaGetLastError();
}

size_t solve_stream_bytes(int n, int nnz) { return 2 * ana::sweep_stream_bytes(n, nnz); }

cudaError_t launch_pack_stream(const double* L, int n, int nnz, const int* rowidx, const int* plan, const double* rdiag,
                               void* stream, cudaStream_t st)
{
    if (n <= 0) return cudaSuccess;
    sweep_rows_kernel<<<2, 32, 0, st>>>(plan, n, nnz, rdiag, stream);
    const int threads = 256;
    const dim3 blocks(std::min((n * 32 + threads - 1) / threads, 65535), 2);
    sweep_entries_kernel<<<blocks, threads, 0, st>>>(L, plan, n, nnz, rowidx, stream);
    return cudaGetLastError();
}

int rand_dots_blocks(int NR)
{
    const int nq = (NR + 3) / 4;
    int nblk = (nq + ana::DOT_THREADS * ana::DOT_BLOCKS_PER_CTA - 1) / (ana::DOT_THREADS * ana::DOT_BLOCKS_PER_CTA);
    return nblk < 1 ? 1 : nblk;
}

cudaError_t launch_rand_dots(uint64_t seed, uint32_t t, uint32_t s_xi, uint32_t s_nu, int NR, int ne,
                             double* partial, int nblk, cudaStream_t st)
{
    dim3 grid(nblk, ne);
    rand_dots_kernel<<<grid, ana::DOT_THREADS, 0, st>>>(seed, t, s_xi, s_nu, NR, partial, nblk);
    return cudaGetLastError();
}

cudaError_t launch_sync_alpha(const double* phi, const double* partial, int nblk, int ne, double NR,
                              double N_psi, double logNe, int scheme, double* c, double* gamma, double* zeta,
                              double* alpha, double* cstar, double* neglogw, double* coef, double* scal,
                              int* flag, cudaStream_t st)
{
    // slices of a warp's width (one Lambert-W solve per lane of one warp), of
    // more where that would take more than 128 CTAs
    const int slice = 32 * ((ne + 32 * 128 - 1) / (32 * 128));
    sync_alpha_kernel<<<(ne + slice - 1) / slice, ana::SYNC_THREADS, 0, st>>>(
        phi, partial, nblk, ne, slice, NR, N_psi, logNe, scheme, c, gamma, zeta, alpha, cstar, neglogw, coef, scal, flag);
    return cudaGetLastError();
}

cudaError_t launch_weights_only(const double* c, const double* gamma, const double* zeta, int ne, double N_psi,
                                int scheme, double* alpha, double* cstar, double* neglogw, double* scal, int* flag,
                                cudaStream_t st)
{
    weights_kernel<<<1, 1024, 0, st>>>(c, gamma, zeta, ne, N_psi, scheme, alpha, cstar, neglogw, scal, flag);
    return cudaGetLastError();
}

cudaError_t launch_form_r(uint64_t seed, uint32_t t, uint32_t s_xi, uint32_t s_nu, int NR, int ne,
                          const double* coef, const double* scal, const double* alpha, float* r,
                          cudaStream_t st)
{
    dim3 grid(((NR + 3) / 4 + 255) / 256, ne);
    form_r_kernel<<<grid, 256, 0, st>>>(seed, t, s_xi, s_nu, NR, coef, scal, alpha, r);
    return cudaGetLastError();
}

cudaError_t launch_block_seq(float* r, int NR, int ne, const float* M49, const int* obs_block0, int nobs, int nRx,
                             int nRy, cudaStream_t st)
{
    if (nobs <= 0) return cudaSuccess;
    block_seq_kernel<<<ne, 32, 0, st>>>(r, NR, M49, obs_block0, nobs, nRx, nRy);
    return cudaGetLastError();
}

cudaError_t launch_block_levels(float* r, int NR, int ne, const float* M49, const int* obs_block0, int nobs,
                                const int* cells, const int* level_off, int nlev, int nRx, int nRy, cudaStream_t st)
{
    if (nlev <= 0 || ne <= 0) return cudaSuccess;
    // a lattice that closes on itself chains its blocks (1521 levels of one): a
    // warp along the chain where each has an SM to itself (100 particles: 4.9 ms
    // per analysis, 5.4 by levels; 1000: 13.7 and 13.0), else the levels
    if (nobs < 2 * nlev && ne <= tc::sm_count())
        return launch_block_seq(r, NR, ne, M49, obs_block0, nobs, nRx, nRy, st);
    // 16 warps (of 128 registers a thread) are resident per SM
    int warps = 2;
    while (warps < BL_WARPS && (long long)ne * warps * 2 <= 16LL * tc::sm_count()) warps *= 2;
    block_levels_kernel<<<ne, 32 * warps, 0, st>>>(r, NR, M49, reinterpret_cast<const int2*>(cells), level_off, nlev,
                                                   nRx, nRy);
    return cudaGetLastError();
}

void block_levels(const int* block0, int nobs, int nRx, int nRy, std::vector<int>& order, std::vector<int>& level_off)
{
    // two 7-point windows on a circle of n points meet when their centres are
    // at most 6 apart (circular distance)
    auto near = [](int a, int b, int n) {
        int d = a - b;
        if (d < 0) d = -d;
        d %= n;
        return std::min(d, n - d) <= 6;
    };
    std::vector<int> level(nobs, 0);
    int top = 0;
    for (int l = 0; l < nobs; ++l) {
        int lv = 0;
        for (int k = 0; k < l; ++k)
            if (level[k] + 1 > lv && near(block0[2 * k], block0[2 * l], nRx) &&
                near(block0[2 * k + 1], block0[2 * l + 1], nRy))
                lv = level[k] + 1;
        level[l] = lv;
        top = std::max(top, lv);
    }
    level_off.assign(top + 2, 0);
    for (int l = 0; l < nobs; ++l) ++level_off[level[l] + 1];
    for (int v = 0; v <= top; ++v) level_off[v + 1] += level_off[v];
    order.assign(nobs, 0);
    std::vector<int> fill(level_off.begin(), level_off.end() - 1);
    for (int l = 0; l < nobs; ++l) order[fill[level[l]]++] = l;
}

namespace {

// breadth-first levels from `root` over the nodes with mark[v] == stamp;
// returns the levels (lists of nodes) and sets dist[v] for the reached ones
std::vector<std::vector<int>> bfs_levels(const std::vector<std::vector<int>>& adj, const std::vector<int>& mark,
                                         int stamp, int root, std::vector<int>& dist)
{
    std::vector<std::vector<int>> lev;
    lev.push_back({root});
    dist[root] = 0;
    for (;;) {
        std::vector<int> next;
        for (int v : lev.back())
            for (int w : adj[v])
                if (mark[w] == stamp && dist[w] < 0) {
                    dist[w] = (int)lev.size();
                    next.push_back(w);
                }
        if (next.empty()) break;
        lev.push_back(std::move(next));
    }
    return lev;
}

void nd_rec(const std::vector<std::vector<int>>& adj, std::vector<int> nodes, std::vector<int>& mark, int& stamp,
            std::vector<int>& dist, std::vector<int>& out)
{
    if (nodes.size() <= 32) {
        out.insert(out.end(), nodes.begin(), nodes.end());
        return;
    }
    ++stamp;
    for (int v : nodes) {
        mark[v] = stamp;
        dist[v] = -1;
    }
    // a far node of the component of nodes[0]: the last level of a search from it
    std::vector<std::vector<int>> lev = bfs_levels(adj, mark, stamp, nodes[0], dist);
    const int far = lev.back().front();
    for (int v : nodes) dist[v] = -1;
    lev = bfs_levels(adj, mark, stamp, far, dist);
    std::vector<int> rest;                                  // other components
    for (int v : nodes)
        if (dist[v] < 0) rest.push_back(v);
    const int D = (int)lev.size();
    if (D < 3) {
        // too shallow to split: this component as it is, then the rest
        for (const auto& l : lev) out.insert(out.end(), l.begin(), l.end());
        if (!rest.empty()) nd_rec(adj, rest, mark, stamp, dist, out);
        return;
    }
    size_t reached = 0;
    for (const auto& l : lev) reached += l.size();
    int m = 1;
    size_t below = lev[0].size();
    while (m < D - 2 && below + lev[m].size() < reached / 2) below += lev[m++].size();
    std::vector<int> a, b;
    for (int k = 0; k < m; ++k) a.insert(a.end(), lev[k].begin(), lev[k].end());
    for (int k = m + 1; k < D; ++k) b.insert(b.end(), lev[k].begin(), lev[k].end());
    const std::vector<int> sep = lev[m];
    nd_rec(adj, a, mark, stamp, dist, out);
    nd_rec(adj, b, mark, stamp, dist, out);
    if (!rest.empty()) nd_rec(adj, rest, mark, stamp, dist, out);
    out.insert(out.end(), sep.begin(), sep.end());
}

}  // namespace

long long nd_order(const int* cells, int nobs, int nx, int ny, int reach, std::vector<int>& order)
{
    long long pairs = 0;
    auto near = [&](int d, int n) {
        d = d < 0 ? -d : d;
        d %= n;
        return std::min(d, n - d) <= reach;
    };
    std::vector<std::vector<int>> adj(nobs);
    for (int k = 0; k < nobs; ++k)
        for (int l = k + 1; l < nobs; ++l)
            if (near(cells[2 * k] - cells[2 * l], nx) && near(cells[2 * k + 1] - cells[2 * l + 1], ny)) {
                adj[k].push_back(l);
                adj[l].push_back(k);
                ++pairs;
            }
    std::vector<int> nodes(nobs), mark(nobs, 0), dist(nobs, -1);
    for (int k = 0; k < nobs; ++k) nodes[k] = k;
    int stamp = 0;
    order.clear();
    order.reserve(nobs);
    nd_rec(adj, nodes, mark, stamp, dist, order);
    return pairs;
}

cudaError_t launch_philox_blocks(uint64_t seed, uint32_t p, uint32_t t, uint32_t stream, long long n,
                                 uint32_t* out, cudaStream_t st)
{
    if (n > 0)
        philox_blocks_kernel<<<(unsigned)((n + 255) / 256), 256, 0, st>>>(seed, p, t, stream, n,
                                                                          reinterpret_cast<uint4*>(out));
    return cudaGetLastError();
}

cudaError_t launch_normals(uint64_t seed, uint32_t p, uint32_t t, uint32_t stream, long long n, double* o64,
                           float* o32, cudaStream_t st)
{
    if (n > 0) normals_kernel<<<(unsigned)((n + 255) / 256), 256, 0, st>>>(seed, p, t, stream, n, o64, o32);
    return cudaGetLastError();
}

}  // namespace iewpf

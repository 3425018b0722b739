// Model steps of small problems (Sec. 3.1 of arXiv 1910.01031): all scheme
// steps of a model step in one launch, each particle's state resident in the
// shared memory of a thread-block cluster.
//
// A grid of a few thousand cells gives the register march (march_dev.cuh) too
// little to do: a warp walks its chunk and the 9 rows around it one after the
// other, a launch and a loop-control launch per scheme step, 17 us for the 64^2
// cells of 10 particles.  Here a cluster of CTAs holds the particle, a slab of
// rows each; a scheme step is two stages of three phases over the slab's cells
// (limited slopes, face fluxes, update), a barrier between phases, and the two
// rows that the neighbours need are stored straight into their shared memory
// (DSMEM) before a cluster barrier ends the stage.  The arithmetic of every
// cell is the march's, operation by operation, so the bits are the same.
//
// Model step of 13 scheme steps, march -> resident:
//   64^2: 10 particles 242 -> 86 us, 40: 283 -> 162 us, 160: 402 -> 335 us (640:
//   the march is as fast); 96^2 x 20: 331 -> 169 us; 128^2 x 10: 294 -> 156 us
#include <algorithm>

#include "march_dev.cuh"
#include "tc_dev.cuh"

namespace iewpf {

namespace {

using march::add;
using march::Consts;
using march::fma;
using march::gmm;
using march::mul;
using march::rcp;
using march::sub;

// A CTA's warps: one per block of 32 columns and row, for all of a phase's
// rows at once (h + 2 of the slopes) or equal parts of them
constexpr int RS_MAX_WARPS = 32;
inline int slab_warps(int nx, int h)
{
    const int nb = (nx + 31) / 32, rows = h + 2;
    int k = 1;
    while (nb * ((rows + k - 1) / k) > RS_MAX_WARPS) ++k;
    return nb * ((rows + k - 1) / k);
}

// rows of slab r of cl
__host__ __device__ inline int slab0(int ny, int cl, int r) { return (int)((long long)ny * r / cl); }

// Shared memory of a slab of up to h rows: two states with two halo rows on
// each side, six slopes with one, six fluxes (east faces, and north faces from
// the row below the slab)
__host__ __device__ inline size_t slab_floats(int nx, int h)
{
    return (size_t)nx * (2 * 3 * (h + 4) + 6 * (h + 2) + 6 * (h + 1));
}
inline int slab_rows(int ny, int cl) { return (ny + cl - 1) / cl; }
inline size_t slab_bytes(int nx, int ny, int cl) { return slab_floats(nx, slab_rows(ny, cl)) * sizeof(float); }
constexpr size_t kSlabBytes = 200 * 1024;

__device__ __forceinline__ void cluster_barrier()
{
    asm volatile("barrier.cluster.arrive.release.aligned;\n barrier.cluster.wait.acquire.aligned;\n" ::: "memory");
}
__device__ __forceinline__ uint32_t cluster_rank()
{
    uint32_t r;
    asm("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
    return r;
}
// address of `p` (this CTA's shared memory) in CTA `rank` of the cluster
__device__ __forceinline__ uint32_t remote(const float* p, uint32_t rank)
{
    uint32_t a;
    asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(a) : "r"(tc::su32(p)), "r"(rank));
    return a;
}
__device__ __forceinline__ void st_remote(uint32_t a, float v)
{
    asm volatile("st.shared::cluster.f32 [%0], %1;" ::"r"(a), "f"(v) : "memory");
}

// One model step of particle blockIdx.x / cl: n_sub scheme steps from the CFL
// rate amax (or fixed), the state rewritten in place (store = 0: not, for
// timing).  amax is cleared for the model error's rates.
__global__ void __launch_bounds__(32 * RS_MAX_WARPS, 1)
resident_kernel(float* __restrict__ buf0, float* __restrict__ buf1, const int* __restrict__ par,
                float* __restrict__ amax, int* __restrict__ nsub, float* __restrict__ dtp, Grid G, int cl,
                double courant, double dt_model, int fixed, unsigned long long* __restrict__ work,
                int* __restrict__ flag, int store)
{
    extern __shared__ float sm[];
    __shared__ int s_n;
    const int p = blockIdx.x / cl, rank = (int)cluster_rank();
    const int nx = G.nx, ny = G.ny;
    const int y0 = slab0(ny, cl, rank), h = slab0(ny, cl, rank + 1) - y0;
    const int hm = (ny + cl - 1) / cl;                // rows the arrays are laid out for
    const int RP = (hm + 4) * nx, SP = (hm + 2) * nx, FP = (hm + 1) * nx;
    float* const raw = sm;                            // [2][3][hm + 4][nx], row r at r + 2
    float* const slo = raw + 6 * RP;                  // [6][hm + 2][nx], row r at r + 1
    float* const flx = slo + 6 * SP;                  // [6][hm + 1][nx], row r at r + 1
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    if (tid == 0) {
        int n = nsub_of(amax[p], courant, dt_model, fixed);
        if (n > kMaxSubSingle) {
            // a non-finite or runaway state: cap the loop and report it
            n = kMaxSubSingle;
            if (rank == 0) atomicOr(flag, (int)FLAG_NONFINITE);
        }
        s_n = n;
    }
    // a warp's column and rows: blocks of 32 columns side by side, then rows
    const int nb = (nx + 31) / 32, step = (int)(blockDim.x >> 5) / nb;
    const int x = 32 * (warp % nb) + lane, w0 = warp / nb;
    const bool col = x < nx;
    const int xe = x + 1 >= nx ? 0 : x + 1, xw = x == 0 ? nx - 1 : x - 1;
    float* const U = (par[p] ? buf1 : buf0) + (long long)p * 3 * G.plane;
    if (col)
        for (int r = w0 - 2; r < h + 2; r += step) {
            const int y = pmod(y0 + r, ny);
#pragma unroll
            for (int f = 0; f < 3; ++f) raw[f * RP + (r + 2) * nx + x] = U[f * G.plane + (long long)y * nx + x];
        }
    // the neighbours' halo rows: my first two rows are the rows h', h' + 1 of
    // the slab below (h' its height), my last two the rows -2, -1 of the one above
    const int below = rank == 0 ? cl - 1 : rank - 1, above = rank + 1 == cl ? 0 : rank + 1;
    const int hb = slab0(ny, cl, below + 1) - slab0(ny, cl, below);
    const uint32_t a_below = remote(raw, below), a_above = remote(raw, above);
    cluster_barrier();                                // every CTA runs and has loaded
    const int n = s_n;
    const float dts = (float)(dt_model / (double)n), dty = dts * G.inv_dy;
    if (rank == 0 && tid == 0 && store) {
        nsub[p] = n;
        dtp[p] = dts;
        amax[p] = 0.0f;
        atomicAdd(work, (unsigned long long)n);
    }
    const Consts<float> K = march::make_consts<float>(G);
    for (int stage = 0; stage < 2 * n; ++stage) {
        const float* const src = raw + (stage & 1 ? 3 * RP : 0);
        float* const dst = raw + (stage & 1 ? 0 : 3 * RP);
        const float *const e = src + 2 * nx, *const qu = e + RP, *const qv = qu + RP;
        auto pot = [&](float k, float q, float ev) { return fma(k, mul(q, rcp(add(K.H, ev))), ev); };
        auto slope = [&](float a, float b) { return gmm(mul(K.theta2, a), add(a, b), mul(K.theta2, b)); };
        // limited slopes: in x of the slab's rows, in y of one more on each side
        if (col)
            for (int r = w0 - 1; r < h + 1; r += step) {
                const int o = r * nx, c = o + x;
                const float ec = e[c], uc = qu[c], vc = qv[c];
                float* const t = slo + (r + 1) * nx + x;
                {
                    const float es = e[c - nx], us = qu[c - nx], en = e[c + nx], un = qu[c + nx];
                    const float dp = sub(pot(K.ky, uc, ec), pot(K.nky, us, es)), dn = sub(pot(K.ky, un, en), pot(K.nky, uc, ec));
                    t[0] = slope(dp, dn);
                    t[SP] = slope(sub(uc, us), sub(un, uc));
                    t[2 * SP] = slope(sub(vc, qv[c - nx]), sub(qv[c + nx], vc));
                }
                if (r >= 0 && r < h) {
                    const float ew = e[o + xw], vw = qv[o + xw], ee = e[o + xe], ve = qv[o + xe];
                    const float dp = sub(pot(K.nkx, vc, ec), pot(K.kx, vw, ew)), dn = sub(pot(K.nkx, ve, ee), pot(K.kx, vc, ec));
                    t[3 * SP] = slope(dp, dn);
                    t[4 * SP] = slope(sub(uc, qu[o + xw]), sub(qu[o + xe], uc));
                    t[5 * SP] = slope(sub(vc, vw), sub(ve, vc));
                }
            }
        __syncthreads();
        // fluxes through north faces (from the row below the slab) and east faces
        if (col)
            for (int r = w0 - 1; r < h; r += step) {
                const int o = r * nx, c = o + x;
                const float *const s = slo + (r + 1) * nx, *const sn = s + nx;
                float* const t = flx + (r + 1) * nx + x;
                const float ec = e[c], uc = qu[c], vc = qv[c];
                {
                    const float en = e[c + nx], un = qu[c + nx], vn = qv[c + nx];
                    float g0, gv, gu;
                    march::flux(fma(K.quarter, s[x], pot(K.nky, uc, ec)), fma(K.quarter, s[2 * SP + x], vc),
                                fma(K.quarter, s[SP + x], uc), fma(K.nquarter, sn[x], pot(K.ky, un, en)),
                                fma(K.nquarter, sn[2 * SP + x], vn), fma(K.nquarter, sn[SP + x], un), K, g0, gv, gu);
                    t[0] = g0;
                    t[FP] = gu;
                    t[2 * FP] = gv;
                }
                if (r >= 0) {
                    const float ee = e[o + xe], ue = qu[o + xe], ve = qv[o + xe];
                    float f0, f1, f2;
                    march::flux(fma(K.quarter, s[3 * SP + x], pot(K.kx, vc, ec)), fma(K.quarter, s[4 * SP + x], uc),
                                fma(K.quarter, s[5 * SP + x], vc), fma(K.nquarter, s[3 * SP + xe], pot(K.nkx, ve, ee)),
                                fma(K.nquarter, s[4 * SP + xe], ue), fma(K.nquarter, s[5 * SP + xe], ve), K, f0, f1, f2);
                    t[3 * FP] = f0;
                    t[4 * FP] = f1;
                    t[5 * FP] = f2;
                }
            }
        __syncthreads();
        // update: stage 1 writes W = U + dt L(U) beside U, stage 2 (U + W + dt L(W)) / 2 over U
        if (col)
            for (int r = w0; r < h; r += step) {
                const int c = r * nx + x;
                const float* const t = flx + (r + 1) * nx;
                const float uc = qu[c], vc = qv[c];
                const float L0 = fma(sub(t[3 * FP + xw], t[3 * FP + x]), K.rxy, sub(t[x - nx], t[x]));
                const float L1 = fma(K.fdy, vc, fma(sub(t[4 * FP + xw], t[4 * FP + x]), K.rxy, sub(t[FP + x - nx], t[FP + x])));
                const float L2 = fma(K.nfdy, uc, fma(sub(t[5 * FP + xw], t[5 * FP + x]), K.rxy,
                                                     sub(t[2 * FP + x - nx], t[2 * FP + x])));
                float z[3] = {fma(dty, L0, e[c]), fma(dty, L1, uc), fma(dty, L2, vc)};
#pragma unroll
                for (int f = 0; f < 3; ++f) {
                    const int i = f * RP + (r + 2) * nx + x;
                    if (stage & 1) z[f] = 0.5f * (dst[i] + z[f]);
                    dst[i] = z[f];
                    const uint32_t d = (uint32_t)((dst - raw + f * RP + x) * 4);
                    if (r < 2) st_remote(a_below + d + (uint32_t)((hb + r + 2) * nx * 4), z[f]);
                    if (r >= h - 2) st_remote(a_above + d + (uint32_t)((r - h + 2) * nx * 4), z[f]);
                }
            }
        cluster_barrier();
    }
    if (col && store)
        for (int r = w0; r < h; r += step)
#pragma unroll
            for (int f = 0; f < 3; ++f) U[f * G.plane + (long long)(y0 + r) * nx + x] = raw[f * RP + (r + 2) * nx + x];
}

}  // namespace

namespace {

// slabs of at least 4 rows whose arrays fit an SM's shared memory
bool slabs_fit(int nx, int ny, int cl)
{
    return (nx + 31) / 32 <= RS_MAX_WARPS && ny / cl >= 4 && slab_bytes(nx, ny, cl) <= kSlabBytes;
}

// the launch of clusters of cl CTAs; `at` holds its attribute
cudaLaunchConfig_t cluster_launch(int nx, int ny, int ne, int cl, cudaStream_t st, cudaLaunchAttribute* at)
{
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)(ne * cl));
    cfg.blockDim = dim3(32 * slab_warps(nx, slab_rows(ny, cl)));
    cfg.dynamicSmemBytes = slab_bytes(nx, ny, cl);
    cfg.stream = st;
    at->id = cudaLaunchAttributeClusterDimension;
    at->val.clusterDim.x = (unsigned)cl;
    at->val.clusterDim.y = at->val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    return cfg;
}

}  // namespace

// Cluster sizes that hold nx x ny (slabs_fit) and find as many SMs in reach of
// one cluster on the current device (a part of a GPU may have fewer)
bool resident_fits(int nx, int ny, int cl)
{
    if (!slabs_fit(nx, ny, cl)) return false;
    if (tc::smem_attr_once<resident_kernel>((int)kSlabBytes) != cudaSuccess) return false;
    cudaLaunchAttribute at;
    const cudaLaunchConfig_t cfg = cluster_launch(nx, ny, 1, cl, nullptr, &at);
    int clusters = 0;
    if (cudaOccupancyMaxActiveClusters(&clusters, resident_kernel, &cfg) != cudaSuccess) {
        cudaGetLastError();
        return false;
    }
    return clusters > 0;
}

cudaError_t launch_resident(float* b0, float* b1, const int* par, float* amax, int* nsub, float* dtp, const Grid& G,
                            double courant, double dt_model, int fixed, unsigned long long* work, int* flag, int cl,
                            int store, cudaStream_t st)
{
    if (!slabs_fit(G.nx, G.ny, cl)) return cudaErrorInvalidValue;
    cudaError_t e = tc::smem_attr_once<resident_kernel>((int)kSlabBytes);
    if (e != cudaSuccess) return e;
    cudaLaunchAttribute at;
    const cudaLaunchConfig_t cfg = cluster_launch(G.nx, G.ny, G.ne, cl, st, &at);
    return cudaLaunchKernelEx(&cfg, resident_kernel, b0, b1, par, amax, nsub, dtp, G, cl, courant, dt_model, fixed, work,
                              flag, store);
}

}  // namespace iewpf

// Register-marching scheme step (Sec. 3.1 of arXiv 1910.01031), one problem
// per launch; the device code is in march_dev.cuh.
#include "march_dev.cuh"

namespace iewpf {

namespace {

// The warps of a particle's strips and chunks are consecutive; the index is
// broadcast from lane 0 so that everything derived from it (particle, rows,
// row addresses) is uniform over the warp.
//
// Bound by instruction issue and, with 8 to 12 warps per SM, by the latency
// that so few hide: at 512^2 x 100 the paired form executes 336 warp
// instructions per 32 cells of the grid (the scalar form 456), the halo's share
// among them (3 columns per lane: 576 columns for 512, and 9 rows for every
// chunk of 256), issues in 59% of the cycles, and about 128 of the 336 are
// packed, which seem to take two dispatch slots each; memory traffic is a
// quarter of what HBM could move in that time.  Registers: 168 with 2 columns per lane (the
// bound of 384 threads), so that 12 warps share an SM; 255 with 3 columns, 8
// warps.  Giving each stage a warp of its own (128 registers, 16 warps, rows
// handed over in shared memory) issues in 81% of the cycles instead of 58%
// but executes 485 instructions, and is slower (401 us).
// One launch, before the potential and flux forms of march_dev.cuh -> now:
//   512^2 x 100: 394 -> 372 us; 1024^2 x 64: 1033 -> 992 us; 1024^2 x 1000:
//   15.2 -> 14.1 ms; 64^2 x 640 (rows closing on a ring of 32 lanes): 75 -> 60 us
template <int NC, bool RING, bool PAIRED>
__global__ void __launch_bounds__(NC == 2 ? 384 : 256)
rk2_march_kernel(march::StepArgs a, int s)
{
    const long long warp =
        (long long)blockIdx.x * (blockDim.x >> 5) + __shfl_sync(march::FULL, (int)(threadIdx.x >> 5), 0);
    const long long per_p = (long long)a.n_strips * a.n_chunks;
    if (warp >= per_p * a.G.ne) return;
    const int p = (int)(warp / per_p);
    const int rem = (int)(warp % per_p);
    const int st = a.s_dev ? *a.s_dev : s;
    if (PAIRED) march::march_warp_paired<NC, RING>(a, p, rem / a.n_strips, rem % a.n_strips, st);
    else march::march_warp<NC, RING>(a, p, rem / a.n_strips, rem % a.n_strips, st);
}

template <int NC, bool RING>
cudaError_t launch(const march::StepArgs& a, int s, int warps, int paired, cudaStream_t st)
{
    const long long n = (long long)a.n_strips * a.n_chunks * a.G.ne;
    const unsigned blocks = (unsigned)((n + warps - 1) / warps);
    if (paired) rk2_march_kernel<NC, RING, true><<<blocks, 32 * warps, 0, st>>>(a, s);
    else rk2_march_kernel<NC, RING, false><<<blocks, 32 * warps, 0, st>>>(a, s);
    return cudaGetLastError();
}

template <int NC>
cudaError_t launch_nc(float* b0, float* b1, const int* par, const int* nsub, const float* dtp, int s, const Grid& G,
                      int TH, int warps_per_cta, int paired, const int* s_dev, cudaStream_t st)
{
    const march::StepArgs a{b0, b1, par, nsub, dtp, G, TH, march::strips(G.nx, NC), (G.ny + TH - 1) / TH, s_dev};
    if (march::ring(G.nx, NC)) return launch<NC, true>(a, s, warps_per_cta, paired, st);
    return launch<NC, false>(a, s, warps_per_cta, paired, st);
}

}  // namespace

cudaError_t launch_rk2_march(float* b0, float* b1, const int* par, const int* nsub, const float* dtp, int s,
                             const Grid& G, const MarchShape& shape, cudaStream_t st,
                             const int* s_dev)
{
    if (shape.TH < 1 || shape.warps < 1 || shape.warps > 8) return cudaErrorInvalidValue;
    switch (shape.nc) {
    case 2: return launch_nc<2>(b0, b1, par, nsub, dtp, s, G, shape.TH, shape.warps, shape.paired, s_dev, st);
    case 3: return launch_nc<3>(b0, b1, par, nsub, dtp, s, G, shape.TH, shape.warps, shape.paired, s_dev, st);
    case 4: return launch_nc<4>(b0, b1, par, nsub, dtp, s, G, shape.TH, shape.warps, shape.paired, s_dev, st);
    default: return cudaErrorInvalidValue;
    }
}

}  // namespace iewpf

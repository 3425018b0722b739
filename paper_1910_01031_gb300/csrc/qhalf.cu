// Model error and analysis update (Sec. 3.2 and 4.6 of arXiv 1910.01031),
// one problem per launch; the device code is in qhalf_dev.cuh.
#include <algorithm>
#include <type_traits>

#include "qhalf_dev.cuh"
#include "tc_dev.cuh"

namespace iewpf {

namespace {

// normals of every particle, one Philox block per thread
__global__ void coarse_normals_kernel(QhalfArgs A, long long NR)
{
    const long long q = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (4 * q >= NR) return;
    const int p = blockIdx.y;
    const uint32_t t = (A.t_dev ? *A.t_dev : 0u) + A.t;
    qhalf::normals_block(seed_key(A.seed), (uint32_t)p, t, A.stream, (uint32_t)q, NR, A.xi_buf + (long long)p * NR);
}

// Q_SOAR^{1/2} of every coarse point of every particle (blockIdx.z).  Bound by
// instructions: the points two and more from the periodic seam in groups of
// SOAR_ROWS rows, a warp along the columns, the others (whose neighbours and
// distances take index arithmetic) densely packed in CTAs of their own, the
// rows of blocks from inner_y on.  A point per thread with 64-bit divisions for
// its place, the seam's points among the others: 279 us for 341^2 coarse points
// x 256, now 106; 171^2 x 100: 38, now 18.
__global__ void __launch_bounds__(256)
coarse_soar_kernel(const float* __restrict__ src, const float* __restrict__ wtab, Grid G, Coarse C,
                   float* __restrict__ out, int inner_y)
{
    const long long NR = (long long)C.nRx * C.nRy;
    const float* __restrict__ s = src + blockIdx.z * NR;
    float* __restrict__ o = out + blockIdx.z * NR;
    if ((int)blockIdx.y < inner_y) {
        const int am = 2 + 32 * blockIdx.x + (threadIdx.x & 31);
        const int bm = 2 + qhalf::SOAR_ROWS * (8 * blockIdx.y + (threadIdx.x >> 5));
        if (am >= C.nRx - 2 || bm >= C.nRy - 2) return;
        if (bm + qhalf::SOAR_ROWS <= C.nRy - 2) {
            qhalf::soar_rows(s, wtab, C, am, bm, o);
        } else {
            for (int b = bm; b < C.nRy - 2; ++b) o[b * C.nRx + am] = qhalf::soar_point(s, wtab, C, G, am, b);
        }
        return;
    }
    const int e = (int)(((blockIdx.y - inner_y) * gridDim.x + blockIdx.x) * 256 + threadIdx.x);
    int am, bm;
    if (e < 4 * C.nRy) {                 // the first and last two columns
        const int c = e / C.nRy;
        am = c < 2 ? c : C.nRx - 4 + c;
        bm = e - c * C.nRy;
    } else {                             // the rest of the first and last two rows
        const int f = e - 4 * C.nRy, c = f / (C.nRx - 4);
        if (c >= 4) return;
        bm = c < 2 ? c : C.nRy - 4 + c;
        am = 2 + f - c * (C.nRx - 4);
    }
    o[bm * C.nRx + am] = qhalf::soar_point(s, wtab, C, G, am, bm);
}

// model error and analysis update on FINE_TX x FINE_TY tiles (the analysis
// update's observation lists are binned by the same tiles)
using qhalf::FINE_TX;
using qhalf::FINE_TY;

// CTAs per SM of the form for single particles
constexpr int FINE_PER_SM1 = 4;

template <bool PULL, int PB, int SUB>
__global__ void __launch_bounds__(NTHREADS, PB == 1 ? FINE_PER_SM1 : 2)
qhalf_fine_kernel(QhalfArgs A, Grid G, Coarse C, int cap, int k_in_smem)
{
    extern __shared__ __align__(16) float fine_smem[];
    qhalf::fine_cta<PULL, PB, SUB>(A, G, C, blockIdx.x, blockIdx.y * qhalf::fine_parts(PB, SUB), A.soar_buf, fine_smem,
                                   cap, k_in_smem);
}

constexpr size_t kStencilSmem = 64 * 1024;      // c_Omega up to 3 (44 KB)

template <bool PULL, int PB, int SUB>
cudaError_t launch_fine(const QhalfArgs& A, const Grid& G, const Coarse& C, int tiles, cudaStream_t st)
{
    constexpr int parts = qhalf::fine_parts(PB, SUB);
    const int cap = PULL ? std::min(A.nobs, MAX_TILE_OBS) : 0;
    const size_t kbytes = PULL && PB > 1 ? 6 * sizeof(float) * (2 * A.R + 1) * (2 * A.R + 1) : 0;
    const int k_in_smem = kbytes > 0 && kbytes <= kStencilSmem;
    const size_t smem = qhalf::fine_list_bytes(cap, parts) + (k_in_smem ? kbytes : 0);
    if (PULL) {
        const cudaError_t e = tc::smem_attr_once<qhalf_fine_kernel<PULL, PB, SUB>>(
            (int)(qhalf::fine_list_bytes(MAX_TILE_OBS, parts) + kStencilSmem));
        if (e != cudaSuccess) return e;
    }
    qhalf_fine_kernel<PULL, PB, SUB>
        <<<dim3((unsigned)tiles, (unsigned)((G.ne + parts - 1) / parts)), NTHREADS, smem, st>>>(A, G, C, cap, k_in_smem);
    return cudaGetLastError();
}

}  // namespace

int qhalf_launches(const QhalfArgs& A)
{
    if (!A.xi_buf || !A.soar_buf) return 0;
    return A.from_philox ? 3 : 2;
}

cudaError_t launch_qhalf(const QhalfArgs& A, const Grid& G, const Coarse& C, cudaStream_t st)
{
    if (C.tab > qhalf::TAB_MAX || !A.xi_buf || !A.soar_buf) return cudaErrorInvalidValue;
    const long long NR = (long long)C.nRx * C.nRy;
    const float* src = A.x;
    if (A.from_philox) {
        const long long nq = (NR + 3) / 4;
        coarse_normals_kernel<<<dim3((unsigned)((nq + 255) / 256), G.ne), 256, 0, st>>>(A, NR);
        src = A.xi_buf;
    }
    const int bx = (C.nRx - 4 + 31) / 32, rows = 8 * qhalf::SOAR_ROWS, inner_y = (C.nRy - 4 + rows - 1) / rows;
    const int seam = (4 * C.nRy + 4 * (C.nRx - 4) + 255) / 256;
    coarse_soar_kernel<<<dim3(bx, inner_y + (seam + bx - 1) / bx, G.ne), 256, 0, st>>>(src, A.wtab, G, C, A.soar_buf,
                                                                                     inner_y);
    const int tiles = ((G.nx + FINE_TX - 1) / FINE_TX) * ((G.ny + FINE_TY - 1) / FINE_TY);
    const int parts = qhalf::fine_choice(
        [&](int n) { return (long long)tiles * ((G.ne + n - 1) / n); }, tc::sm_count(), FINE_PER_SM1);
    auto run = [&](auto pull) {
        constexpr bool P = decltype(pull)::value;
        if (parts == qhalf::fine_parts(4, 1)) return launch_fine<P, 4, 1>(A, G, C, tiles, st);
        if (parts == qhalf::fine_parts(4, 4)) return launch_fine<P, 4, 4>(A, G, C, tiles, st);
        return launch_fine<P, 1, 4>(A, G, C, tiles, st);
    };
    return A.with_pull ? run(std::true_type{}) : run(std::false_type{});
}

}  // namespace iewpf

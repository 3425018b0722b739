// Device code of the model-error operator Q^{1/2} = Q_GB^{1/2} I_Omega Q_SOAR^{1/2}
// (Sec. 3.2 of arXiv 1910.01031, eqs. local_soar_on_eta,
// geostrophic_balance_disc, covarianceOperatorsDef) in three stages:
//   Philox normals once per coarse point (normals_block)
//   -> 5x5 SOAR once per coarse point (soar_point)
//   -> per fine tile: bicubic to the tile + 1-cell ring, central-difference
//      geostrophic momentum, read-modify-write of the state (fine_cta).
// The analysis update reuses the fine stage with the posterior coarse field
// and adds the optimal-proposal pull (eq. detailedOPDUpdate) in the same
// read-modify-write.
#pragma once
#include "common.cuh"
#include "fine_choice.h"
#include "kernels.h"

namespace iewpf {
namespace qhalf {

constexpr int TAB_MAX = 45;                   // 3 c for c <= 15
// fine tiles of the model error and of the analysis update (the tiles the
// observation lists are binned by)
constexpr int FINE_TX = OBS_TX, FINE_TY = OBS_TY;

// Coarse stages once per coarse point.  Normals of block q (counter q) of a
// Philox stream: words (0, 1) and (2, 3) give the Box-Muller pairs of normals
// 4q, 4q + 1 and 4q + 2, 4q + 3 (the same numbers normal32 returns one by one).
__device__ __forceinline__ void normals_block(uint2 key, uint32_t p, uint32_t t, uint32_t stream, uint32_t q,
                                              long long NR, float* __restrict__ out)
{
    const uint4 w = philox4x32_10(make_uint4(q, p, t, stream), key);
    float z[4];
    box_muller32(w.x, w.y, z[0], z[1]);
    box_muller32(w.z, w.w, z[2], z[3]);
#pragma unroll
    for (int j = 0; j < 4; ++j)
        if (4LL * q + j < NR) out[4LL * q + j] = z[j];
}

// Q_SOAR^{1/2} at coarse point (am, bm) of field src [N_R]: the 5 x 5 sum of
// eq. local_soar_on_eta over the coarse neighbours, rows outer
__device__ __forceinline__ float soar_point(const float* __restrict__ src, const float* __restrict__ wtab,
                                            const Coarse& C, const Grid& G, int am, int bm)
{
    if (am >= 2 && am + 2 < C.nRx && bm >= 2 && bm + 2 < C.nRy) {
        // away from the periodic seam the neighbours are c fine cells apart:
        // the same weights and sums as below without the periodic index
        // arithmetic
        float acc = 0.0f;
#pragma unroll
        for (int db = -2; db <= 2; ++db) {
            const float* __restrict__ row = src + (bm + db) * C.nRx + am;
            const float* __restrict__ wr = wtab + C.c * (db < 0 ? -db : db) * C.tab;
#pragma unroll
            for (int da = -2; da <= 2; ++da) acc = fmaf(wr[C.c * (da < 0 ? -da : da)], row[da], acc);
        }
        return acc;
    }
    const int x0 = coarse_pos(am, C.nRx, C.c, C.o, G.nx), y0 = coarse_pos(bm, C.nRy, C.c, C.o, G.ny);
    int dxf[5], col[5];
#pragma unroll
    for (int da = -2; da <= 2; ++da) {
        dxf[da + 2] = abs(coarse_pos(am + da, C.nRx, C.c, C.o, G.nx) - x0);
        col[da + 2] = pmod(am + da, C.nRx);
    }
    float acc = 0.0f;
#pragma unroll
    for (int db = -2; db <= 2; ++db) {
        const int dyf = abs(coarse_pos(bm + db, C.nRy, C.c, C.o, G.ny) - y0);
        const int row = pmod(bm + db, C.nRy) * C.nRx;
#pragma unroll
        for (int da = -2; da <= 2; ++da) acc = fmaf(wtab[dyf * C.tab + dxf[da + 2]], src[row + col[da + 2]], acc);
    }
    return acc;
}

// points (am, bm0 + r), r < SOAR_ROWS, all two and more away from the seam:
// each row of five neighbours is loaded once for the points it enters; the
// sums of soar_point, term by term
constexpr int SOAR_ROWS = 4;
__device__ __forceinline__ void soar_rows(const float* __restrict__ src, const float* __restrict__ wtab, const Coarse& C,
                                          int am, int bm0, float* __restrict__ out)
{
    float w[3][3], acc[SOAR_ROWS];
#pragma unroll
    for (int b = 0; b < 3; ++b)
#pragma unroll
        for (int a = 0; a < 3; ++a) w[b][a] = __ldg(wtab + C.c * b * C.tab + C.c * a);
#pragma unroll
    for (int j = 0; j < SOAR_ROWS + 4; ++j) {
        const float* __restrict__ row = src + (bm0 - 2 + j) * C.nRx + am;
        float v[5];
#pragma unroll
        for (int k = 0; k < 5; ++k) v[k] = row[k - 2];
#pragma unroll
        for (int r = 0; r < SOAR_ROWS; ++r) {
            const int db = j - 2 - r;
            if (db < -2 || db > 2) continue;
            if (db == -2) acc[r] = 0.0f;
#pragma unroll
            for (int k = 0; k < 5; ++k) acc[r] = fmaf(w[db < 0 ? -db : db][k < 2 ? 2 - k : k - 2], v[k], acc[r]);
        }
    }
#pragma unroll
    for (int r = 0; r < SOAR_ROWS; ++r) out[(bm0 + r) * C.nRx + am] = acc[r];
}

// The fine stage: a warp marches down a strip of 32 columns of PB particles
// at once, one column per lane, with no shared memory between lanes and no
// barriers: the four coarse rows around the current row, interpolated in x at
// the lane's column, roll in registers (a new one every c rows), the
// y-interpolation gives the field of one row, three rows of it roll for the
// y-difference, and the x-difference takes the neighbours' values by shuffle.
// The two columns beside the strip, which only that difference needs, are one
// more column per warp: lanes 2 pp and 2 pp + 1 carry those of particle pp.
// A coarse row is one load per particle (lane l the l-th coarse column the
// strip touches, requested an interval ahead) and four shuffles, where the
// strip's coarse columns fit the lanes (c >= 2), else four loads.
// PB particles share the row's weights and, with the pull, each load of the
// stencil: those loads bound the pull when every particle makes its own.
//
// Pull: each listed observation that reaches the row of the strip, in list
// order, adds its six stencil products to the cells it reaches (offset within
// R of the cell in the minimum image, both axes: the stencil's reach 2R + 1
// lies within the grid, iewpf_create refuses smaller ones, so each cell sees
// one image).  The sum of a cell starts from the interpolated field and its
// balanced momentum; the state is rewritten once.
//
// The CTA: TY rows x two strips (the OBS_TX x OBS_TY tiles of the observation
// lists) of fine_parts(PB, SUB) particles; four warps per strip take a group of PB
// particles each (SUB = 1), or a quarter of the rows of one group (SUB = 4);
// fine_choice says which.
//
// Bound by latency and issue with 4 particles per warp (128 registers, 16 warps
// per SM), by latency with one (64 registers, 32 warps: 1024^2 x 1 14.5 us, 18.5
// with 90 registers and 16); 8 per warp halve the stencil's loads again but also
// the warps.
// Analysis update: the tile kernel it replaced interpolated through shared
// memory with four barriers and then applied one observation at a time to the
// whole tile, each particle loading the stencil anew and a barrier between
// observations: 11.1 ms at 624^2 x 1000 (7 of 1521 observations reach a
// cell), now 4.1 ms; 4.2 -> 2.0 ms at 1024^2 x 256 (2.7 of 1521); 234 -> 180 us
// at 512^2 x 100 (64 drifters).  Model error: 168 -> 153 us at 512^2 x 100, 48
// -> 38 us at 256^2 x 100.
constexpr int STRIPS = OBS_TX / 32;
constexpr int GROUPS = NTHREADS / 32 / STRIPS;
__host__ __device__ constexpr int fine_parts(int PB, int SUB) { return PB * (GROUPS / SUB); }
static_assert(fine_parts(4, 1) == 16 && fine_parts(4, 4) == 4 && fine_parts(1, 4) == 1, "the forms of fine_choice");

// Dynamic shared memory of one CTA (16-byte aligned) for lists of up to cap
// observations of `parts` particles: S d as (su, su', sv, sv') of each pair of
// particles, the pairs of an observation together ((su, sv) of a single
// particle), then the observations' offsets from the tile origin, then the
// copy of the stencil.
__host__ __device__ constexpr size_t fine_list_bytes(int cap, int parts) { return (size_t)cap * (8 + 8 * (size_t)parts); }

struct FineRows {
    float4 w[FINE_TY + 2];      // y-weights of rows y0 - 1 .. y0 + TY
    int b[FINE_TY + 2];         // and their coarse intervals
};

__device__ __forceinline__ void column_taps(int x, const Grid& G, const Coarse& C, int& a, float w[4])
{
    float t;
    a = coarse_interval(x, C.nRx, C.c, C.o, G.nx, t);
    cubic_weights(t, w);
}

__device__ __forceinline__ float taps(const float w[4], float v0, float v1, float v2, float v3)
{
    float v = 0.0f;
    v = fmaf(w[0], v0, v);
    v = fmaf(w[1], v1, v);
    v = fmaf(w[2], v2, v);
    v = fmaf(w[3], v3, v);
    return v;
}

// adds (su, sv) of the warp's PB particles times the stencil values k[6] (su:
// 0..2, sv: 3..5) to their sums; pairs of particles in packed FMAs (each half
// rounds as the scalar instruction)
template <int PB>
__device__ __forceinline__ void pull_add(float (&acc)[3][PB], const float* __restrict__ s, const float k[6])
{
    if constexpr (PB == 1) {
        const float2 v = *reinterpret_cast<const float2*>(s);
#pragma unroll
        for (int f = 0; f < 3; ++f) acc[f][0] = fmaf(v.y, k[3 + f], fmaf(v.x, k[f], acc[f][0]));
    } else {
#pragma unroll
        for (int pp = 0; pp < PB; pp += 2) {
            const float4 v = *reinterpret_cast<const float4*>(s + 2 * pp);
#pragma unroll
            for (int f = 0; f < 3; ++f) {
                float2 a = make_float2(acc[f][pp], acc[f][pp + 1]);
                a = __ffma2_rn(make_float2(v.x, v.y), make_float2(k[f], k[f]), a);
                a = __ffma2_rn(make_float2(v.z, v.w), make_float2(k[3 + f], k[3 + f]), a);
                acc[f][pp] = a.x;
                acc[f][pp + 1] = a.y;
            }
        }
    }
}

// the pull of one row: ty, sx the row and the strip's first column in the
// tile; sd the warp's S d of observation 0, sd_stride floats per observation;
// K [2R+1][2R+1][6]
template <int PB>
__device__ __forceinline__ void pull_row(float (&acc)[3][PB], const Grid& G, int R, const int2* __restrict__ off,
                                         int n_obs, const float* __restrict__ sd, int sd_stride,
                                         const float* __restrict__ K, int ty, int sx)
{
    const int lane = threadIdx.x & 31, W = 2 * R + 1;
    for (int q0 = 0; q0 < n_obs; q0 += 32) {
        // lane j: does observation q0 + j reach a cell of this row, at which
        // stencil row (element kb) and, for the strip's first column, at which
        // column xo (0 .. 2R, or a period above)
        bool in = false;
        int kb = 0, xo = 0;
        if (q0 + lane < n_obs) {
            const int2 o = off[q0 + lane];
            int oy = o.y + ty;
            const int ox = o.x + sx;
            if (oy > R) oy -= G.ny;
            in = oy >= -R && oy <= R && ((ox <= R && ox + 31 >= -R) || (ox - G.nx <= R && ox + 31 - G.nx >= -R));
            kb = (oy + R) * W * 6;
            xo = ox + R;
        }
        for (unsigned mask = __ballot_sync(0xffffffffu, in); mask; mask &= mask - 1) {
            const int j = __ffs(mask) - 1;
            const int b = __shfl_sync(0xffffffffu, kb, j);
            int t = __shfl_sync(0xffffffffu, xo, j) + lane;
            if (t > 2 * R) t -= G.nx;
            if ((unsigned)t <= (unsigned)(2 * R)) {
                const float2* __restrict__ k2 = reinterpret_cast<const float2*>(K + b + 6 * t);
                const float2 a = k2[0], bb = k2[1], c = k2[2];
                const float k[6] = {a.x, a.y, bb.x, bb.y, c.x, c.y};
                pull_add<PB>(acc, sd + (q0 + j) * sd_stride, k);
            }
        }
    }
}

// One tile of the particles p0 .. p0 + fine_parts(PB, SUB) - 1 (those below
// ne) from their SOAR fields so_g [ne][N_R].  PULL: smem is
// fine_list_bytes(cap, ...) with cap >= the tile's list length, followed by the stencil's 6 (2R +
// 1)^2 floats if k_smem: it is copied there when the tile's list is long
// enough to reuse it (every observation of a row reads it at another offset,
// and the state's stream through L1 evicts it).
// Called by whole CTAs of NTHREADS threads; a CTA may call it for several
// tiles in turn.
template <bool PULL, int PB, int SUB>
__device__ __forceinline__ void fine_cta(const QhalfArgs& A, const Grid& G, const Coarse& C, int tile, int p0,
                                         const float* __restrict__ so_g, float* smem, int cap, bool k_smem)
{
    constexpr int PARTS = fine_parts(PB, SUB);
    __shared__ FineRows rows;
    const int ntx = (G.nx + FINE_TX - 1) / FINE_TX;
    const int x0 = (tile % ntx) * FINE_TX, y0 = (tile / ntx) * FINE_TY;
    const int np = min(PARTS, G.ne - p0), tid = threadIdx.x, lane = tid & 31;
    int2* const off = reinterpret_cast<int2*>(smem + 2 * (size_t)cap * PARTS);
    float* const sK = smem + 2 * (size_t)cap * (PARTS + 1);
    __syncthreads();                         // a previous tile's readers are done
    for (int i = tid; i < FINE_TY + 2; i += NTHREADS) {
        float t, w[4];
        rows.b[i] = coarse_interval(y0 - 1 + i, C.nRy, C.c, C.o, G.ny, t);
        cubic_weights(t, w);
        rows.w[i] = make_float4(w[0], w[1], w[2], w[3]);
    }
    int n = 0;
    bool copied = false;
    if (PULL) {
        // the minimum-image offset of the tile origin from each listed
        // observation, in (-n/2, n/2] (the cells add theirs, at most one
        // period above), and the particles' S d
        n = min(min(A.tile_cnt[tile], MAX_TILE_OBS), cap);
        copied = k_smem && n >= 4;
        if (copied)
            for (int k = tid; k < 6 * (2 * A.R + 1) * (2 * A.R + 1); k += NTHREADS) sK[k] = A.K[k];
        for (int q = tid; q < n; q += NTHREADS) {
            const int l = A.tile_obs[tile * A.tile_cap + q];
            int dx = pmod(x0 - A.obs_cell[2 * l], G.nx), dy = pmod(y0 - A.obs_cell[2 * l + 1], G.ny);
            if (dx > G.nx / 2) dx -= G.nx;
            if (dy > G.ny / 2) dy -= G.ny;
            off[q] = make_int2(dx, dy);
        }
        for (int k = tid; k < n * PARTS; k += NTHREADS) {
            const int q = k / PARTS, pp = k % PARTS;
            const long long at = (long long)(p0 + min(pp, np - 1)) * 2 * A.nobs + 2 * A.tile_obs[tile * A.tile_cap + q];
            float* const d = smem + 2 * q * PARTS + (PB == 1 ? 2 * pp : 4 * (pp >> 1) + (pp & 1));
            d[0] = (float)A.Sd[at];
            d[PB == 1 ? 1 : 2] = (float)A.Sd[at + 1];
        }
    }
    __syncthreads();
    const int warp = tid >> 5, grp = warp / STRIPS, sx = 32 * (warp % STRIPS);
    constexpr int ROWS = FINE_TY / SUB;
    const int r0 = (grp % SUB) * ROWS, r1 = r0 + ROWS, g0 = (grp / SUB) * PB;
    if (x0 + sx >= G.nx || y0 + r0 >= G.ny || g0 >= np) return;      // uniform over the warp
    const long long NR = (long long)C.nRx * C.nRy;
    const int x = x0 + sx + lane;
    const bool valid = x < G.nx;
    int a, ha;
    float wx[4], hw[4];
    column_taps(x, G, C, a, wx);
    column_taps((lane & 1) ? x0 + sx + 32 : x0 + sx - 1, G, C, ha, hw);
    // the coarse columns a0 - 1 .. a0 + 30 by lane, if they hold the strip's taps
    const int a0 = __shfl_sync(0xffffffffu, a, 0);
    const bool by_lane = __shfl_sync(0xffffffffu, a, 31) + 2 <= a0 + 30;
    const int mycol = pmod(a0 - 1 + lane, C.nRx);
    int hc[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) hc[k] = pmod(ha - 1 + k, C.nRx);
    // coarse row of an extended index (at most a few rows beyond the grid)
    auto wrap_row = [&](int bk) { return bk < 0 ? bk + C.nRy : (bk >= C.nRy ? bk - C.nRy : bk); };
    const float* __restrict__ hso = so_g + (long long)(p0 + min(g0 + min(lane >> 1, PB - 1), np - 1)) * NR;
    const int last = np - 1 - g0;            // particles beyond np repeat the last and are not stored
    const float* so_p[PB];
#pragma unroll
    for (int pp = 0; pp < PB; ++pp) so_p[pp] = so_g + (long long)(p0 + g0 + min(pp, last)) * NR;
    float R[4][PB], hR[4], raw[PB], hraw[4];
    auto request = [&](int bk) {             // coarse row bk
        const int o = wrap_row(bk) * C.nRx;      // within one particle's coarse grid
        if (by_lane) {
#pragma unroll
            for (int pp = 0; pp < PB; ++pp) raw[pp] = so_p[pp][o + mycol];
        }
#pragma unroll
        for (int k = 0; k < 4; ++k) hraw[k] = hso[o + hc[k]];
    };
    auto take = [&](int k, int bk) {         // into R[k]
        if (by_lane) {
#pragma unroll
            for (int pp = 0; pp < PB; ++pp)
                R[k][pp] = taps(wx, __shfl_sync(0xffffffffu, raw[pp], a - a0), __shfl_sync(0xffffffffu, raw[pp], a - a0 + 1),
                                __shfl_sync(0xffffffffu, raw[pp], a - a0 + 2), __shfl_sync(0xffffffffu, raw[pp], a - a0 + 3));
        } else {
            const int o = wrap_row(bk) * C.nRx;
            const int c0 = pmod(a - 1, C.nRx), c1 = pmod(a, C.nRx), c2 = pmod(a + 1, C.nRx), c3 = pmod(a + 2, C.nRx);
#pragma unroll
            for (int pp = 0; pp < PB; ++pp) {
                const float* __restrict__ q = so_p[pp] + o;
                R[k][pp] = taps(wx, q[c0], q[c1], q[c2], q[c3]);
            }
        }
        hR[k] = taps(hw, hraw[0], hraw[1], hraw[2], hraw[3]);
    };
    int b = rows.b[r0];
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        request(b - 1 + k);
        take(k, b - 1 + k);
    }
    request(b + 3);
    // the state at column x of the row to write
    float* U[PB];
#pragma unroll
    for (int pp = 0; pp < PB; ++pp) {
        const int p = p0 + g0 + min(pp, last);
        U[pp] = (A.par[p] ? A.b1 : A.b0) + (long long)p * 3 * G.plane + (long long)(y0 + r0) * G.nx + (valid ? x : 0);
    }
    // Model error (no pull, whose products cover the wait and leave no registers):
    // the lines of the next row's state are brought to L1, lane l < 3 PB asking
    // for field l % 3 of particle l / 3 (lanes 16 + l for the strip's last column,
    // where that is on another line); one row of loads in flight per warp left the
    // stage waiting on memory (30 model errors of 256^2 x 100 and three network
    // calls: 8.54 ms, now 8.37).
    const int pl = lane & 15;
    const bool ask = !PULL && pl < 3 * PB;
    const float* ahead = nullptr;
    const float* stop = nullptr;
    if (!PULL) {
        const int p = p0 + g0 + min(pl / 3, last), xl = x0 + sx + (lane & 16 ? min(31, G.nx - 1 - x0 - sx) : 0);
        ahead = (A.par[p] ? A.b1 : A.b0) + ((long long)p * 3 + pl % 3) * G.plane + (long long)(y0 + r0) * G.nx + xl;
        stop = ahead + (long long)(min(r1, G.ny - y0) - r0) * G.nx;
        if (ask) asm volatile("prefetch.global.L1 [%0];" ::"l"(ahead));
        ahead += G.nx;
    }
    float dm[PB], d0[PB], dn[PB], hd = 0.0f, m[PB];
#pragma unroll
    for (int pp = 0; pp < PB; ++pp) dm[pp] = d0[pp] = m[pp] = 0.0f;
    for (int i = r0; i < r1 + 2; ++i) {
        const int ty = i - 2, gy = y0 + ty;          // the row to write
        if (gy >= G.ny) break;
        const bool write = ty >= r0;
        float u[3][PB];                              // (requested first, used last)
        if (write) {
#pragma unroll
            for (int pp = 0; pp < PB; ++pp)
#pragma unroll
                for (int f = 0; f < 3; ++f) u[f][pp] = U[pp][f * G.plane];
            if (!PULL) {
                if (ask && ahead < stop) asm volatile("prefetch.global.L1 [%0];" ::"l"(ahead));
                ahead += G.nx;
            }
        }
        // field of row y0 + i - 1
        if (rows.b[i] != b) {
            b = rows.b[i];
#pragma unroll
            for (int k = 0; k < 3; ++k) {
#pragma unroll
                for (int pp = 0; pp < PB; ++pp) R[k][pp] = R[k + 1][pp];
                hR[k] = hR[k + 1];
            }
            take(3, b + 2);
            request(b + 3);
        }
        const float4 w4 = rows.w[i];
        const float w[4] = {w4.x, w4.y, w4.z, w4.w};
#pragma unroll
        for (int pp = 0; pp < PB; ++pp) dn[pp] = taps(w, R[0][pp], R[1][pp], R[2][pp], R[3][pp]);
        const float hn = taps(w, hR[0], hR[1], hR[2], hR[3]);
        if (write) {
            float acc[3][PB];
#pragma unroll
            for (int pp = 0; pp < PB; ++pp) {
                const float hl = __shfl_sync(0xffffffffu, hd, 2 * pp), hr = __shfl_sync(0xffffffffu, hd, 2 * pp + 1);
                float l = __shfl_up_sync(0xffffffffu, d0[pp], 1), r = __shfl_down_sync(0xffffffffu, d0[pp], 1);
                if (lane == 0) l = hl;
                if (lane == 31) r = hr;
                acc[0][pp] = d0[pp];
                acc[1][pp] = -G.sgh * (dn[pp] - dm[pp]) * G.inv_2dy;
                acc[2][pp] = G.sgh * (r - l) * G.inv_2dx;
            }
            if (PULL) {
                if (copied) pull_row<PB>(acc, G, A.R, off, n, smem + 2 * g0, 2 * PARTS, sK, ty, sx);
                else pull_row<PB>(acc, G, A.R, off, n, smem + 2 * g0, 2 * PARTS, A.K, ty, sx);
            }
            if (valid) {
#pragma unroll
                for (int pp = 0; pp < PB; ++pp) {
                    if (pp <= last) {
                        const float e1 = u[0][pp] + acc[0][pp], u1 = u[1][pp] + acc[1][pp], v1 = u[2][pp] + acc[2][pp];
                        U[pp][0] = e1;
                        U[pp][G.plane] = u1;
                        U[pp][2 * G.plane] = v1;
                        if (A.amax) m[pp] = fmaxf(m[pp], cfl_of(e1, u1, v1, G));
                    }
                }
            }
#pragma unroll
            for (int pp = 0; pp < PB; ++pp) U[pp] += G.nx;
        }
#pragma unroll
        for (int pp = 0; pp < PB; ++pp) {
            dm[pp] = d0[pp];
            d0[pp] = dn[pp];
        }
        hd = hn;
    }
    if (A.amax) {
#pragma unroll
        for (int pp = 0; pp < PB; ++pp) {
            const float v = warp_max(m[pp]);
            // non-negative floats order like their bit patterns
            if (lane == 0 && pp <= last) atomicMax(reinterpret_cast<int*>(A.amax) + p0 + g0 + pp, __float_as_int(v));
        }
    }
}

}  // namespace qhalf
}  // namespace iewpf

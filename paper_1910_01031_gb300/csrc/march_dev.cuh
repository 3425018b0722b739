// Device code of the register-marching scheme step (Sec. 3.1 of arXiv 1910.01031):
// one step of the second-order SSP Runge-Kutta method with central-upwind
// fluxes and the Coriolis-adjusted (well-balanced) reconstruction of eta,
// organised for issue efficiency on GB300, in a scalar form (march_warp) and
// a form with the two stages paired in f32x2 registers (march_warp_paired).
//
// Each warp owns a strip of 32*NC columns (NC per lane) and marches down a
// chunk of rows.  Rows above and below live in a rolling window in registers;
// x-neighbours come from the adjacent lanes by warp shuffles.  Both
// Runge-Kutta stages run in the same march, the second behind the first, so a
// cell is read once and written once per scheme step, with no shared memory
// and no block barriers.  The 4 outermost columns on each side of a strip are
// halo (recomputed by the neighbouring strip) and 8 extra rows fill the
// pipeline of each chunk.  Where the whole row fits one warp (nx <= 32 NC, a
// multiple of NC) the lanes form a ring instead and no column is computed
// twice.  Divisions and square roots use the hardware approximations (rcp,
// sqrt; a few ulp).  The file is compiled without automatic multiply-add
// contraction and every fused multiply-add is written out, so each cell's
// arithmetic is the same whatever the tile shape, stage pairing or kernel.
//
// What bounds the step is the number of FP32 instructions per cell, so the
// scheme is written with as few as its formulas allow:
//  * potentials: with P = eta + k u and M = eta - k u, k = f dy / (2g), the
//    reconstructed difference of the y-potential over a face, (g (eta1 - eta0)
//    + f dy/2 (u0 + u1)) / g, is P1 - M0, and the face values of eta are
//    M + s/4 (north) and P - s/4 (south) with s the limited (doubled)
//    difference; in x with k = f dx / (2g) and the signs of v swapped;
//  * flux: with A = a+ / (a+ - a-) and B = -A a-, the central-upwind flux is
//    F_R + A (F_L - F_R) + B (q_L - q_R), whose rounding errors scale with
//    the jump over the face but for one at the flux's own last place (the
//    momentum flux adds F_R last for that: added within the chain of FMAs it
//    rounded twice there, and under a mean elevation of 30 m and more in 230 m
//    of water a forecast's momentum was 9% further from 64 bits than with the
//    flux as one quotient; 3 to 6% nearer so);
//  * flux differences are scaled by dt/dy once, at the update.
#pragma once
#include "common.cuh"
#include "kernels.h"

namespace iewpf {
namespace march {

constexpr unsigned FULL = 0xffffffffu;

// single hardware approximations (flush-to-zero: depths and wave speeds are
// far from the subnormal range)
__device__ __forceinline__ float frcp(float x)
{
    float y;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}
__device__ __forceinline__ float fsqrt(float x)
{
    float y;
    asm("sqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

// three-input minimum and maximum (one instruction each on sm_100 and later)
__device__ __forceinline__ float fmin3(float a, float b, float c)
{
    float y;
    asm("min.f32 %0, %1, %2, %3;" : "=f"(y) : "f"(a), "f"(b), "f"(c));
    return y;
}
__device__ __forceinline__ float fmax3(float a, float b, float c)
{
    float y;
    asm("max.f32 %0, %1, %2, %3;" : "=f"(y) : "f"(a), "f"(b), "f"(c));
    return y;
}

// The arithmetic below is written once for T = float (one stage) and T =
// float2 (the two stages in the halves of a packed register: an add, multiply
// or fused multiply-add covers both in one instruction and rounds each half
// as the scalar instruction does; the hardware approximations, minima,
// maxima, selects and shuffles stay per half).
using f2 = float2;
__device__ __forceinline__ float add(float a, float b) { return a + b; }
__device__ __forceinline__ float sub(float a, float b) { return a - b; }
__device__ __forceinline__ float mul(float a, float b) { return a * b; }
__device__ __forceinline__ float fma(float a, float b, float c) { return fmaf(a, b, c); }
__device__ __forceinline__ float rcp(float a) { return frcp(a); }
__device__ __forceinline__ float sqr(float a) { return fsqrt(a); }
__device__ __forceinline__ float max3z(float a, float b) { return fmax3(a, b, 0.0f); }
__device__ __forceinline__ float max3zn(float a, float b) { return fmax3(-a, -b, 0.0f); }
// a where x >= 0, else b
__device__ __forceinline__ float sel(float x, float a, float b) { return x >= 0.0f ? a : b; }
// generalized minmod, doubled: the minmod of (x, y, z) = (2 theta a, a + b, 2
// theta b) for the differences a, b: the smallest of the three when all are
// positive, the largest when all are negative, else 0 -- the median of (min,
// 0, max), max(min, min(max, 0)).  Every use scales the slope by a power of
// two, so carrying it doubled is exact.
__device__ __forceinline__ float gmm(float x, float y, float z)
{
    return fmaxf(fmin3(x, y, z), fminf(fmax3(x, y, z), 0.0f));
}

__device__ __forceinline__ f2 bc(float a) { return make_float2(a, a); }
__device__ __forceinline__ f2 add(f2 a, f2 b) { return __fadd2_rn(a, b); }
// a - b as fma(b, -1, a), the same rounding (with the packed subtraction
// instruction the two kinds' results differ in some last bits)
__device__ __forceinline__ f2 sub(f2 a, f2 b) { return __ffma2_rn(b, make_float2(-1.0f, -1.0f), a); }
__device__ __forceinline__ f2 mul(f2 a, f2 b) { return __fmul2_rn(a, b); }
__device__ __forceinline__ f2 fma(f2 a, f2 b, f2 c) { return __ffma2_rn(a, b, c); }
__device__ __forceinline__ f2 rcp(f2 a) { return make_float2(frcp(a.x), frcp(a.y)); }
__device__ __forceinline__ f2 sqr(f2 a) { return make_float2(fsqrt(a.x), fsqrt(a.y)); }
__device__ __forceinline__ f2 max3z(f2 a, f2 b) { return make_float2(max3z(a.x, b.x), max3z(a.y, b.y)); }
__device__ __forceinline__ f2 max3zn(f2 a, f2 b) { return make_float2(max3zn(a.x, b.x), max3zn(a.y, b.y)); }
__device__ __forceinline__ f2 sel(f2 x, f2 a, f2 b) { return make_float2(sel(x.x, a.x, b.x), sel(x.y, a.y, b.y)); }
__device__ __forceinline__ f2 gmm(f2 x, f2 y, f2 z) { return make_float2(gmm(x.x, y.x, z.x), gmm(x.y, y.y, z.y)); }

// grid constants, broadcast to both halves for float2
template <class T>
struct Consts {
    T H, sg, nsg, g_half, gH, theta2, quarter, nquarter, kx, nkx, ky, nky, rxy, fdy, nfdy;
};
__device__ __forceinline__ void to(float a, float& o) { o = a; }
__device__ __forceinline__ void to(float a, f2& o) { o = bc(a); }
template <class T>
__device__ __forceinline__ Consts<T> make_consts(const Grid& G)
{
    Consts<T> K;
    to(G.H, K.H);
    to(G.sqrt_g, K.sg);
    to(-G.sqrt_g, K.nsg);
    to(G.g_half, K.g_half);
    to(G.gH, K.gH);
    to(G.theta2, K.theta2);
    to(0.25f, K.quarter);
    to(-0.25f, K.nquarter);
    to(G.fdx_2g, K.kx);
    to(-G.fdx_2g, K.nkx);
    to(G.fdy_2g, K.ky);
    to(-G.fdy_2g, K.nky);
    to(G.dy_dx, K.rxy);
    to(G.fdy, K.fdy);
    to(-G.fdy, K.nfdy);
    return K;
}

// central-upwind flux: mass F0, normal momentum qn -> F1, tangential qt
// carried by the mass flux with the upwind tangential velocity -> F2
template <class T>
__device__ __forceinline__ void flux(T eL, T qnL, T qtL, T eR, T qnR, T qtR, const Consts<T>& K, T& F0, T& F1, T& F2)
{
    const T hL = add(K.H, eL), hR = add(K.H, eR);
    const T rL = rcp(hL), rR = rcp(hR);
    const T cL = sqr(hL), cR = sqr(hR);                  // wave speed sqrt(g) c
    const T unL = mul(qnL, rL), unR = mul(qnR, rR);
    const T ap = max3z(fma(K.sg, cL, unL), fma(K.sg, cR, unR));         // a+
    const T am = max3zn(fma(K.nsg, cL, unL), fma(K.nsg, cR, unR));      // -a-
    const T A = mul(ap, rcp(add(ap, am))), B = mul(A, am);
    const T dq = sub(qnL, qnR);
    F0 = fma(B, sub(eL, eR), fma(A, dq, qnR));
    // p(eta) = g eta (H + eta/2) = eta (g/2 eta + g H)
    const T mL = fma(qnL, unL, mul(eL, fma(K.g_half, eL, K.gH)));
    const T mR = fma(qnR, unR, mul(eR, fma(K.g_half, eR, K.gH)));
    // m_R last: one rounding at its last place
    F1 = add(mR, fma(B, dq, mul(A, sub(mL, mR))));
    F2 = mul(F0, sel(F0, mul(qtL, rL), mul(qtR, rR)));
}

// lanes to the left and right: neighbours within a strip, or on a ring of
// lanes that closes the periodic row
template <bool RING>
struct Lanes {
    int left, right;
    __device__ __forceinline__ explicit Lanes(int n)
    {
        const int lane = threadIdx.x & 31;
        left = lane == 0 ? n - 1 : lane - 1;
        right = lane + 1 >= n ? 0 : lane + 1;
    }
    __device__ __forceinline__ float up(float v) const
    {
        return RING ? __shfl_sync(FULL, v, left) : __shfl_up_sync(FULL, v, 1);
    }
    __device__ __forceinline__ float dn(float v) const
    {
        return RING ? __shfl_sync(FULL, v, right) : __shfl_down_sync(FULL, v, 1);
    }
    __device__ __forceinline__ f2 up(f2 v) const { return make_float2(up(v.x), up(v.y)); }
    __device__ __forceinline__ f2 dn(f2 v) const { return make_float2(dn(v.x), dn(v.y)); }
};

// Rolling window of one stage (T = float) or both (float2).  CARRY: the
// scaled differences of the previous face are kept in registers; otherwise
// they are formed again (the packed form is short of registers).
template <int NC, class T, bool RING, bool CARRY>
struct Marcher {
    T e[2][NC], qu[2][NC], qv[2][NC];   // rows 1 and 2 (the newest); row 0 leaves in push
    T P[NC], M[NC];                     // eta +- k u of row 2
    T dL[NC];                           // potential difference on the face between rows 1 and 2
    T tL[NC], tu[NC], tv[NC];           // 2 theta times the differences on that face (CARRY)
    T Ne[NC], Nu[NC], Nv[NC];           // values of row 1 at its north face
    T G0[NC], Gu[NC], Gv[NC];           // flux through the face south of row 1

    __device__ __forceinline__ void zero()
    {
        T z;
        to(0.0f, z);
#pragma unroll
        for (int k = 0; k < NC; ++k) {
#pragma unroll
            for (int r = 0; r < 2; ++r) e[r][k] = qu[r][k] = qv[r][k] = z;
            P[k] = M[k] = dL[k] = Ne[k] = Nu[k] = Nv[k] = G0[k] = Gu[k] = Gv[k] = z;
            if (CARRY) tL[k] = tu[k] = tv[k] = z;
        }
    }

    // Push the next row; returns dy L(U) of the row that leaves the window
    // (two rows behind the pushed one) and that row's state.
    __device__ __forceinline__ void push(const T* ne, const T* nqu, const T* nqv, const Consts<T>& K,
                                         const Lanes<RING>& ln, T* L0, T* L1, T* L2, T* oe, T* oqu, T* oqv)
    {
        // the window moves: row 0 = the row to emit, 1, 2 = the new row
        // y direction: slopes of row 1, flux on the face between rows 0 and 1
#pragma unroll
        for (int k = 0; k < NC; ++k) {
            const T u2 = mul(nqu[k], rcp(add(K.H, ne[k])));
            const T P2 = fma(K.ky, u2, ne[k]), M2 = fma(K.nky, u2, ne[k]);
            const T dLn = sub(P2, M[k]);
            const T dun = sub(nqu[k], qu[1][k]), dvn = sub(nqv[k], qv[1][k]);
            const T dup = sub(qu[1][k], qu[0][k]), dvp = sub(qv[1][k], qv[0][k]);
            const T tLn = mul(K.theta2, dLn), tun = mul(K.theta2, dun), tvn = mul(K.theta2, dvn);
            const T tLp = CARRY ? tL[k] : mul(K.theta2, dL[k]);
            const T tup = CARRY ? tu[k] : mul(K.theta2, dup);
            const T tvp = CARRY ? tv[k] : mul(K.theta2, dvp);
            const T sL = gmm(tLp, add(dL[k], dLn), tLn);
            const T su = gmm(tup, add(dup, dun), tun);
            const T sv = gmm(tvp, add(dvp, dvn), tvn);
            if (CARRY) {
                tL[k] = tLn;
                tu[k] = tun;
                tv[k] = tvn;
            }
            T g0, gv, gu;
            flux(Ne[k], Nv[k], Nu[k], fma(K.nquarter, sL, P[k]), fma(K.nquarter, sv, qv[1][k]),
                 fma(K.nquarter, su, qu[1][k]), K, g0, gv, gu);
            L0[k] = sub(G0[k], g0);
            L1[k] = sub(Gu[k], gu);
            L2[k] = sub(Gv[k], gv);
            Ne[k] = fma(K.quarter, sL, M[k]);
            Nu[k] = fma(K.quarter, su, qu[1][k]);
            Nv[k] = fma(K.quarter, sv, qv[1][k]);
            G0[k] = g0;
            Gu[k] = gu;
            Gv[k] = gv;
            P[k] = P2;
            M[k] = M2;
            dL[k] = dLn;
            oe[k] = e[0][k];
            oqu[k] = qu[0][k];
            oqv[k] = qv[0][k];
            e[0][k] = e[1][k];
            qu[0][k] = qu[1][k];
            qv[0][k] = qv[1][k];
            e[1][k] = ne[k];
            qu[1][k] = nqu[k];
            qv[1][k] = nqv[k];
        }
        // x direction on row 0: differences on the faces f = 1..NC right of
        // column f - 1 with the right neighbour's first column, the left
        // face's from the left neighbour
        T XP[NC], XM[NC];
#pragma unroll
        for (int k = 0; k < NC; ++k) {
            const T v = mul(oqv[k], rcp(add(K.H, oe[k])));
            XP[k] = fma(K.kx, v, oe[k]);
            XM[k] = fma(K.nkx, v, oe[k]);
        }
        T dK[NC + 1], dU[NC + 1], dV[NC + 1];
#pragma unroll
        for (int f = 1; f < NC; ++f) {
            dK[f] = sub(XM[f], XP[f - 1]);
            dU[f] = sub(oqu[f], oqu[f - 1]);
            dV[f] = sub(oqv[f], oqv[f - 1]);
        }
        dK[NC] = sub(ln.dn(XM[0]), XP[NC - 1]);
        dU[NC] = sub(ln.dn(oqu[0]), oqu[NC - 1]);
        dV[NC] = sub(ln.dn(oqv[0]), oqv[NC - 1]);
        dK[0] = ln.up(dK[NC]);
        dU[0] = ln.up(dU[NC]);
        dV[0] = ln.up(dV[NC]);
        T eE[NC], eW[NC], uE[NC], uW[NC], vE[NC], vW[NC];
#pragma unroll
        for (int k = 0; k < NC; ++k) {
            const T sK = gmm(mul(K.theta2, dK[k]), add(dK[k], dK[k + 1]), mul(K.theta2, dK[k + 1]));
            const T sU = gmm(mul(K.theta2, dU[k]), add(dU[k], dU[k + 1]), mul(K.theta2, dU[k + 1]));
            const T sV = gmm(mul(K.theta2, dV[k]), add(dV[k], dV[k + 1]), mul(K.theta2, dV[k + 1]));
            eE[k] = fma(K.quarter, sK, XP[k]);
            eW[k] = fma(K.nquarter, sK, XM[k]);
            uE[k] = fma(K.quarter, sU, oqu[k]);
            uW[k] = fma(K.nquarter, sU, oqu[k]);
            vE[k] = fma(K.quarter, sV, oqv[k]);
            vW[k] = fma(K.nquarter, sV, oqv[k]);
        }
        // face f lies on the left of own column f; face NC is the right edge
        T F0[NC + 1], F1[NC + 1], F2[NC + 1];
#pragma unroll
        for (int f = 1; f < NC; ++f) flux(eE[f - 1], uE[f - 1], vE[f - 1], eW[f], uW[f], vW[f], K, F0[f], F1[f], F2[f]);
        flux(eE[NC - 1], uE[NC - 1], vE[NC - 1], ln.dn(eW[0]), ln.dn(uW[0]), ln.dn(vW[0]), K, F0[NC], F1[NC], F2[NC]);
        F0[0] = ln.up(F0[NC]);
        F1[0] = ln.up(F1[NC]);
        F2[0] = ln.up(F2[NC]);
#pragma unroll
        for (int k = 0; k < NC; ++k) {
            L0[k] = fma(sub(F0[k], F0[k + 1]), K.rxy, L0[k]);
            L1[k] = fma(K.fdy, oqv[k], fma(sub(F1[k], F1[k + 1]), K.rxy, L1[k]));
            L2[k] = fma(K.nfdy, oqu[k], fma(sub(F2[k], F2[k + 1]), K.rxy, L2[k]));
        }
    }
};

// One warp's strip of one chunk: the columns of this lane and the rows.
template <int NC, bool RING>
struct Strip {
    const float* in;        // the particle's state, read
    float* out;             // and written
    unsigned off[NC];       // byte offset of the lane's columns in a row
    bool keep[NC];
    int y0, rows;
    __device__ __forceinline__ bool init(const StepArgs& a, int p, int chunk, int strip, int s)
    {
        const Grid& G = a.G;
        if (s >= a.nsub[p]) return false;
        const int src = a.par[p] ^ (s & 1);
        in = (src ? a.buf1 : a.buf0) + (long long)p * 3 * G.plane;
        out = (src ? a.buf0 : a.buf1) + (long long)p * 3 * G.plane;
        y0 = chunk * a.TH;
        rows = min(a.TH, G.ny - y0);
        const int lane = threadIdx.x & 31;
#pragma unroll
        for (int k = 0; k < NC; ++k) {
            const int c = lane * NC + k;
            if (RING) {
                keep[k] = c < G.nx;
                off[k] = keep[k] ? 4u * (unsigned)c : 0u;
            } else {
                const int x = strip * (32 * NC - 8) - 4 + c;
                off[k] = 4u * (unsigned)pmod(x, G.nx);
                keep[k] = c >= 4 && c < 32 * NC - 4 && x < G.nx;
            }
        }
        return true;
    }
    // field f of row y at the lane's column k
    __device__ __forceinline__ static float ld(const float* row, unsigned off)
    {
        return __ldg(reinterpret_cast<const float*>(reinterpret_cast<const char*>(row) + off));
    }
    __device__ __forceinline__ static void st(float* row, unsigned off, float v)
    {
        *reinterpret_cast<float*>(reinterpret_cast<char*>(row) + off) = v;
    }
};

// One warp's strip of one chunk of particle p in scheme step s.
template <int NC, bool RING>
__device__ __forceinline__ void march_warp(const StepArgs& a, int p, int chunk, int strip, int s)
{
    const Grid& G = a.G;
    Strip<NC, RING> S;
    if (!S.init(a, p, chunk, strip, s)) return;
    const float dty = a.dtp[p] * G.inv_dy;
    const Consts<float> K = make_consts<float>(G);
    const Lanes<RING> ln(RING ? G.nx / NC : 32);
    Marcher<NC, float, RING, true> S1, S2;
    S1.zero();
    S2.zero();
    float f0e[NC], f0u[NC], f0v[NC], f1e[NC], f1u[NC], f1v[NC];   // U0 of the last two emitted rows
#pragma unroll
    for (int k = 0; k < NC; ++k) f0e[k] = f0u[k] = f0v[k] = f1e[k] = f1u[k] = f1v[k] = 0.0f;
    const int n_it = S.rows + 8;
    float ne[NC], nqu[NC], nqv[NC];
    {
        const float* r = S.in + (long long)pmod(S.y0 - 4, G.ny) * G.nx;
#pragma unroll
        for (int k = 0; k < NC; ++k) {
            ne[k] = S.ld(r, S.off[k]);
            nqu[k] = S.ld(r + G.plane, S.off[k]);
            nqv[k] = S.ld(r + 2 * G.plane, S.off[k]);
        }
    }
    int yn = pmod(S.y0 - 3, G.ny);     // row of the next prefetch, wrapped as it advances
    float* o = S.out + (long long)S.y0 * G.nx;
    for (int it = 0; it < n_it; ++it) {
        // prefetch the next input row
        float pe[NC], pqu[NC], pqv[NC];
        if (it + 1 < n_it) {
            const float* r = S.in + (long long)yn * G.nx;
#pragma unroll
            for (int k = 0; k < NC; ++k) {
                pe[k] = S.ld(r, S.off[k]);
                pqu[k] = S.ld(r + G.plane, S.off[k]);
                pqv[k] = S.ld(r + 2 * G.plane, S.off[k]);
            }
        }
        yn = yn + 1 == G.ny ? 0 : yn + 1;
        // stage 1 on U0, then stage 2 on U1 = U0 + dt L(U0)
        float L0[NC], L1[NC], L2[NC], ue[NC], uu[NC], uv[NC];
        S1.push(ne, nqu, nqv, K, ln, L0, L1, L2, ue, uu, uv);
        float we[NC], wu[NC], wv[NC];
#pragma unroll
        for (int k = 0; k < NC; ++k) {
            we[k] = fmaf(dty, L0[k], ue[k]);
            wu[k] = fmaf(dty, L1[k], uu[k]);
            wv[k] = fmaf(dty, L2[k], uv[k]);
        }
        float M0[NC], M1[NC], M2[NC], ve[NC], vu[NC], vv[NC];
        S2.push(we, wu, wv, K, ln, M0, M1, M2, ve, vu, vv);
        if (it >= 8) {
#pragma unroll
            for (int k = 0; k < NC; ++k) {
                if (S.keep[k]) {
                    S.st(o, S.off[k], 0.5f * (f1e[k] + fmaf(dty, M0[k], ve[k])));
                    S.st(o + G.plane, S.off[k], 0.5f * (f1u[k] + fmaf(dty, M1[k], vu[k])));
                    S.st(o + 2 * G.plane, S.off[k], 0.5f * (f1v[k] + fmaf(dty, M2[k], vv[k])));
                }
            }
            o += G.nx;
        }
#pragma unroll
        for (int k = 0; k < NC; ++k) {
            f1e[k] = f0e[k]; f1u[k] = f0u[k]; f1v[k] = f0v[k];
            f0e[k] = ue[k]; f0u[k] = uu[k]; f0v[k] = uv[k];
            ne[k] = pe[k]; nqu[k] = pqu[k]; nqv[k] = pqv[k];
        }
    }
}

// The same march with the two Runge-Kutta stages as the two halves of packed
// f32x2 registers: the low half carries stage 1 on U0, the high half stage 2
// on U1 = U0 + dt L(U0), one row later than in march_warp so that both halves
// of a push are independent (stage 2 takes the row that stage 1 finished in
// the previous iteration).  Each half performs exactly the scalar march's
// operations in the same order, so results are identical bit for bit.  The
// original state of the output row is read again from the input (a row read
// five iterations earlier, normally still in L1) instead of being held.
template <int NC, bool RING>
__device__ __forceinline__ void march_warp_paired(const StepArgs& a, int p, int chunk, int strip, int s)
{
    const Grid& G = a.G;
    Strip<NC, RING> S;
    if (!S.init(a, p, chunk, strip, s)) return;
    const f2 dty = bc(a.dtp[p] * G.inv_dy);
    const Consts<f2> K = make_consts<f2>(G);
    const Lanes<RING> ln(RING ? G.nx / NC : 32);
    Marcher<NC, f2, RING, false> S12;
    S12.zero();
    // push input: low half the next row of U0, high half W of the row that
    // stage 1 finished in the previous iteration
    f2 ne[NC], nqu[NC], nqv[NC];
    {
        const float* r = S.in + (long long)pmod(S.y0 - 4, G.ny) * G.nx;
#pragma unroll
        for (int k = 0; k < NC; ++k) {
            ne[k] = make_float2(S.ld(r, S.off[k]), 0.0f);
            nqu[k] = make_float2(S.ld(r + G.plane, S.off[k]), 0.0f);
            nqv[k] = make_float2(S.ld(r + 2 * G.plane, S.off[k]), 0.0f);
        }
    }
    const int n_it = S.rows + 9;
    int yn = pmod(S.y0 - 3, G.ny);     // row of the next prefetch, wrapped as it advances
    const float* ro = S.in + (long long)S.y0 * G.nx;
    float* o = S.out + (long long)S.y0 * G.nx;
    for (int it = 0; it < n_it; ++it) {
        float pe[NC], pqu[NC], pqv[NC];
        if (it + 1 < n_it) {
            const float* r = S.in + (long long)yn * G.nx;
#pragma unroll
            for (int k = 0; k < NC; ++k) {
                pe[k] = S.ld(r, S.off[k]);
                pqu[k] = S.ld(r + G.plane, S.off[k]);
                pqv[k] = S.ld(r + 2 * G.plane, S.off[k]);
            }
        }
        yn = yn + 1 == G.ny ? 0 : yn + 1;
        // the original state of this iteration's output row, read again
        // (issued here so that the loads complete during the push)
        const bool emit = it >= 9;
        float o0[NC], o1[NC], o2[NC];
        if (emit) {
#pragma unroll
            for (int k = 0; k < NC; ++k) {
                o0[k] = S.ld(ro, S.off[k]);
                o1[k] = S.ld(ro + G.plane, S.off[k]);
                o2[k] = S.ld(ro + 2 * G.plane, S.off[k]);
            }
        }
        f2 L0[NC], L1[NC], L2[NC], oe[NC], ou[NC], ov[NC];
        S12.push(ne, nqu, nqv, K, ln, L0, L1, L2, oe, ou, ov);
        // low: W = U0 + dt L(U0) of the row stage 1 emitted; high: U1 + dt
        // L(U1) of the row stage 2 emitted
        f2 z0[NC], z1[NC], z2[NC];
#pragma unroll
        for (int k = 0; k < NC; ++k) {
            z0[k] = fma(dty, L0[k], oe[k]);
            z1[k] = fma(dty, L1[k], ou[k]);
            z2[k] = fma(dty, L2[k], ov[k]);
        }
        if (emit) {
#pragma unroll
            for (int k = 0; k < NC; ++k) {
                if (S.keep[k]) {
                    S.st(o, S.off[k], 0.5f * (o0[k] + z0[k].y));
                    S.st(o + G.plane, S.off[k], 0.5f * (o1[k] + z1[k].y));
                    S.st(o + 2 * G.plane, S.off[k], 0.5f * (o2[k] + z2[k].y));
                }
            }
            ro += G.nx;
            o += G.nx;
        }
#pragma unroll
        for (int k = 0; k < NC; ++k) {
            ne[k] = make_float2(pe[k], z0[k].x);
            nqu[k] = make_float2(pqu[k], z1[k].x);
            nqv[k] = make_float2(pqv[k], z2[k].x);
        }
    }
}

}  // namespace march
}  // namespace iewpf

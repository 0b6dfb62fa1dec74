// dbm_aux_impl.cuh -- kernels of the initialisation, state transfer and
// FP64 output calls of the D2V16 DBM (f = f^eq from macroscopic fields, the
// macroscopic fields, the nonequilibrium moments of Eqs. Delta2, Delta31,
// Delta3, Delta42, the conserved totals), and their launches for one species
// count S.  dbm_aux_s<S>.cu instantiates the launches per S so that the
// units compile in parallel; dbm_aux.cu dispatches on S.
#pragma once
#include <stdio.h>

#include <type_traits>

#include "dbm_bf16.cuh"

namespace dbm {

// Ghost images of a cell's stored planes (masks from ghost_mask: comparisons
// only, and a second look at the cell's own stores on the domain edge; the
// images used to come from eight integer modulos in every cell: k_set_f on
// 2048 x 1024 took 207 us, now 159).
template <typename T>
__device__ __forceinline__ void images_of_planes(T *f, long long plane, int nplanes, long long cell, int x, int y,
                                                 int nx, int ny, int pitch, int bc_x, int bc_y)
{
    const unsigned mx = ghost_mask(x, nx, bc_x), my = ghost_mask(y, ny, bc_y);
    if ((mx | my) == 0u) return;
    for (int p = 0; p < nplanes; ++p) store_images(f + p * plane, x, y, nx, ny, pitch, mx, my, f[p * plane + cell]);
}

// f = f^eq(rho^s / m^s, u, T), computed in FP64 and rounded to `real`.
template <typename real, int S>
__global__ void __launch_bounds__(256)
    k_set_state(const __grid_constant__ OutConsts<S> c, real *__restrict__ f,
                const double *__restrict__ rho_s, const double *__restrict__ ux,
                const double *__restrict__ uy, const double *__restrict__ T)
{
    const int x = blockIdx.x * blockDim.x + threadIdx.x;
    const int y = blockIdx.y * blockDim.y + threadIdx.y;
    if (x >= c.nx || y >= c.ny) return;
    const long long N = (long long)c.nx * c.ny;
    const long long d = (long long)y * c.nx + x;
    const long long cell = (long long)(y + GY) * c.pitch + (x + GX);
    const double u_x = ux[d], u_y = uy[d], t = T[d];
#pragma unroll 1
    for (int s = 0; s < S; ++s) {
        double fh[Q];
        fhat16<double>(rho_s[s * N + d] / c.m[s], u_x, u_y, t / c.m[s], c.dpi[s], fh);
        for (int i = 0; i < Q; ++i) {
            double v = 0.0;
#pragma unroll
            for (int k = 0; k < Q; ++k) v += c.cinv[s][i][k] * fh[k];
            f[(s * Q + i) * c.plane + cell] = (real)v;
        }
    }
    images_of_planes(f, c.plane, S * Q, cell, x, y, c.nx, c.ny, c.pitch, c.bc_x, c.bc_y);
}

// 1 / m^s in FP64, for the conversion of the FP64 input fields.
template <int S>
struct InvMass {
    double v[S];
};

// FP32 storage: f = f^eq(rho^s / m^s, u, T) by the step kernel's own FP32
// symmetry-block solve (with its projection onto exact mass, momentum and
// energy): the state starts as the equilibrium the FP32 step itself builds,
// at a fraction of the cost of the FP64 matrix product (a few float ulps
// from the correctly rounded FP64 equilibrium).
template <int S>
__global__ void __launch_bounds__(256)
    k_set_state_blocks(const __grid_constant__ StepConsts<float, S> c, float *__restrict__ f,
                       const double *__restrict__ rho_s, const double *__restrict__ ux,
                       const double *__restrict__ uy, const double *__restrict__ T, const __grid_constant__ InvMass<S> im_d)
{
    const int x = blockIdx.x * blockDim.x + threadIdx.x;
    const int y = blockIdx.y * blockDim.y + threadIdx.y;
    if (x >= c.nx || y >= c.ny) return;
    const long long N = (long long)c.nx * c.ny;
    const long long d = (long long)y * c.nx + x;
    const long long cell = (long long)(y + GY) * c.pitch + (x + GX);
    const float u_x = (float)ux[d], u_y = (float)uy[d];
    const double t = T[d];
#pragma unroll 1
    for (int s = 0; s < S; ++s) {
        float cb[16], o[16];
        fhat_blocks<float>((float)(rho_s[s * N + d] * im_d.v[s]), u_x, u_y, (float)(t * im_d.v[s]), c.dpi[s], cb);
        solve_blocks<float>(c, s, cb, o);
#pragma unroll
        for (int i = 0; i < Q; ++i) f[(s * Q + i) * c.plane + cell] = feq_of<float>(i, o);
    }
    images_of_planes(f, c.plane, S * Q, cell, x, y, c.nx, c.ny, c.pitch, c.bc_x, c.bc_y);
}

// Source of f for the output kernels: a plain FP64 or FP32 state buffer
// (the BF16-deviation state has BfSrc, which rebuilds f).
template <typename real>
struct PlainSrc {
    using value = real;
    const real *f;
    long long plane;
    __device__ __forceinline__ static double widened(float v) { return widen(v); }
    __device__ __forceinline__ static double widened(double v) { return v; }
    __device__ __forceinline__ void load16(int s, long long cell, double v[Q]) const
    {
#pragma unroll
        for (int i = 0; i < Q; ++i) v[i] = widened(f[(s * Q + i) * plane + cell]);
    }
    __device__ __forceinline__ void load16f(int s, long long cell, float v[Q]) const
    {
#pragma unroll
        for (int i = 0; i < Q; ++i) v[i] = (float)f[(s * Q + i) * plane + cell];
    }
};

// Sums of one ring of four values in FP64: all (mass), the vector part
// (rx, ry) and the second moments' part per unit v^2 (axis rings: xx = f0 + f2
// and yy = f1 + f3; diagonal rings: xx = yy = all and xy).  Additions in place
// of the 16 products with each velocity component.
struct RingSums {
    double all, rx, ry, xx, yy, xy;
};
template <bool DIAG>
__device__ __forceinline__ RingSums ring_sums(const double f[4])
{
    RingSums g;
    const double a = f[0] + f[2], b = f[1] + f[3];
    g.all = a + b;
    if (DIAG) {
        const double d = f[0] - f[2], e = f[3] - f[1];
        g.rx = d + e;
        g.ry = d - e;
        g.xx = g.yy = g.all;
        g.xy = a - b;
    } else {
        g.rx = f[0] - f[2];
        g.ry = f[1] - f[3];
        g.xx = a;
        g.yy = b;
        g.xy = 0.0;
    }
    return g;
}
__device__ __forceinline__ RingSums ring_sums(int r, const double f[4])
{
    return (r & 1) ? ring_sums<true>(f) : ring_sums<false>(f);
}

// Species moments of one cell in FP64: n, j = sum f v, E = sum f (v.v+eta^2).
template <int S, class Src>
__device__ __forceinline__ void cell_moments(const OutConsts<S> &c, const Src &src, long long cell,
                                             double n[S], double jx[S], double jy[S], double en[S])
{
#pragma unroll
    for (int s = 0; s < S; ++s) {
        double fv[Q];
        src.load16(s, cell, fv);
        n[s] = jx[s] = jy[s] = en[s] = 0.0;
#pragma unroll
        for (int r = 0; r < 4; ++r) {
            const RingSums g = ring_sums(r, fv + 4 * r);
            n[s] += g.all;
            jx[s] += c.vr[s][r] * g.rx;
            jy[s] += c.vr[s][r] * g.ry;
            en[s] += c.qr[s][r] * g.all;
        }
    }
}

template <int S>
__device__ __forceinline__ void cell_mixture(const OutConsts<S> &c, const double n[S],
                                             const double jx[S], const double jy[S],
                                             const double en[S], double &ux, double &uy, double &T)
{
    double w = 0, wx = 0, wy = 0;
#pragma unroll
    for (int s = 0; s < S; ++s) {
        w += c.m[s] * n[s] * c.inv_tau[s];
        wx += c.m[s] * jx[s] * c.inv_tau[s];
        wy += c.m[s] * jy[s] * c.inv_tau[s];
    }
    ux = wx / w;
    uy = wy / w;
    const double u2 = ux * ux + uy * uy;
    double num = 0, den = 0;
#pragma unroll
    for (int s = 0; s < S; ++s) {
        num += (c.m[s] * en[s] - c.m[s] * n[s] * u2) * c.inv_tau[s];
        den += n[s] * c.dpi[s] * c.inv_tau[s];
    }
    T = num / den;
}

template <int S, class Src>
__global__ void __launch_bounds__(256)
    k_moments(const __grid_constant__ OutConsts<S> c, const __grid_constant__ Src src,
              double *__restrict__ out)
{
    const int x = blockIdx.x * blockDim.x + threadIdx.x;
    const int y = blockIdx.y * blockDim.y + threadIdx.y;
    if (x >= c.nx || y >= c.ny) return;
    const long long N = (long long)c.nx * c.ny;
    const long long d = (long long)y * c.nx + x;
    const long long cell = (long long)(y + GY) * c.pitch + (x + GX);
    double n[S], jx[S], jy[S], en[S];
    cell_moments<S>(c, src, cell, n, jx, jy, en);
    double rho = 0, ntot = 0;
#pragma unroll
    for (int s = 0; s < S; ++s) {
        // an absent species (n = 0) reports zero velocity and temperature
        const bool here = n[s] != 0.0;
        const double usx = here ? jx[s] / n[s] : 0.0, usy = here ? jy[s] / n[s] : 0.0;
        out[(4 * s + 0) * N + d] = n[s];
        out[(4 * s + 1) * N + d] = usx;
        out[(4 * s + 2) * N + d] = usy;
        out[(4 * s + 3) * N + d] =
            here ? c.m[s] * (en[s] / n[s] - (usx * usx + usy * usy)) / c.dpi[s] : 0.0;
        rho += c.m[s] * n[s];
        ntot += n[s];
    }
    double ux, uy, T;
    cell_mixture<S>(c, n, jx, jy, en, ux, uy, T);
    out[(4 * S + 0) * N + d] = rho;
    out[(4 * S + 1) * N + d] = ux;
    out[(4 * S + 2) * N + d] = uy;
    out[(4 * S + 3) * N + d] = T;
    out[(4 * S + 4) * N + d] = ntot * T;
}

// Kernel parameters of k_moments_f32: the constants as the floats it works
// with (converting the double ones in the kernel costs the FP64 pipe).
template <int S>
struct MomentConsts {
    float vr[S][4], qr[S][4], m[S], dpi[S];
    float lam[S], kap[S];  // m / tau, (D + I) / tau
    int nx, ny, pitch;
};

template <int S>
inline MomentConsts<S> moment_consts(const OutConsts<S> &c)
{
    MomentConsts<S> k;
    memset(&k, 0, sizeof(k));
    for (int s = 0; s < S; ++s) {
        for (int r = 0; r < 4; ++r) {
            k.vr[s][r] = (float)c.vr[s][r];
            k.qr[s][r] = (float)c.qr[s][r];
        }
        k.m[s] = (float)c.m[s];
        k.dpi[s] = (float)c.dpi[s];
        k.lam[s] = (float)(c.m[s] * c.inv_tau[s]);
        k.kap[s] = (float)(c.dpi[s] * c.inv_tau[s]);
    }
    k.nx = c.nx;
    k.ny = c.ny;
    k.pitch = c.pitch;
    return k;
}

// The macroscopic fields of a float state (DBM_FP32 or DBM_BF16DEV), in
// float arithmetic, stored as FP64: the state carries float precision, and
// on this GPU the FP64 evaluation of k_moments is bound by the FP64 pipe (8 ms
// for 4096^2 cells against 0.6 ms for the memory traffic).  Species sums by
// rings as in the step; the mixture temperature's cancelling subtraction in
// float-float (mixture_T); u^s and T^s from n^s, j^s, E^s with one fused
// multiply-add each.  Relative error a few float ulps of each field.  Float
// constants and widen() keep the FP64 pipe out of it but for one product a
// cell: 4096^2, two species, 1.27 -> 0.59 ms, the memory time.
template <int S, class Src>
__global__ void __launch_bounds__(256)
    k_moments_f32(const __grid_constant__ MomentConsts<S> c, const __grid_constant__ Src src,
                  double *__restrict__ out)
{
    const int x = blockIdx.x * blockDim.x + threadIdx.x;
    const int y = blockIdx.y * blockDim.y + threadIdx.y;
    if (x >= c.nx || y >= c.ny) return;
    const long long N = (long long)c.nx * c.ny;
    const long long d = (long long)y * c.nx + x;
    const long long cell = (long long)(y + GY) * c.pitch + (x + GX);
    float rho = 0.0f, ntot = 0.0f, w = 0.0f, wx = 0.0f, wy = 0.0f, we = 0.0f, wd = 0.0f;
#pragma unroll
    for (int s = 0; s < S; ++s) {
        float f[Q];
        src.load16f(s, cell, f);
        float sn = 0.0f, sx = 0.0f, sy = 0.0f, se = 0.0f;
#pragma unroll
        for (int r = 0; r < 4; ++r) {
            const float f0 = f[4 * r], f1 = f[4 * r + 1], f2 = f[4 * r + 2], f3 = f[4 * r + 3];
            const float rs = (f0 + f2) + (f1 + f3);
            float rx, ry;
            if ((r & 1) == 0) {
                rx = f0 - f2;
                ry = f1 - f3;
            } else {
                const float a = f0 - f2, b = f3 - f1;
                rx = a + b;
                ry = a - b;
            }
            sn += rs;
            sx = fmaf(c.vr[s][r], rx, sx);
            sy = fmaf(c.vr[s][r], ry, sy);
            se = fmaf(c.qr[s][r], rs, se);
        }
        const bool here = sn != 0.0f;  // an absent species reports zero velocity and temperature
        const float rn = here ? 1.0f / sn : 0.0f;
        const float usx = sx * rn, usy = sy * rn;
        const float ts = here ? c.m[s] * fmaf(-usx, usx, fmaf(-usy, usy, se * rn)) / c.dpi[s] : 0.0f;
        out[(4 * s + 0) * N + d] = widen(sn);
        out[(4 * s + 1) * N + d] = widen(usx);
        out[(4 * s + 2) * N + d] = widen(usy);
        out[(4 * s + 3) * N + d] = widen(ts);
        rho = fmaf(c.m[s], sn, rho);
        ntot += sn;
        w = fmaf(c.lam[s], sn, w);
        wx = fmaf(c.lam[s], sx, wx);
        wy = fmaf(c.lam[s], sy, wy);
        we = fmaf(c.lam[s], se, we);
        wd = fmaf(c.kap[s], sn, wd);
    }
    const float rw = 1.0f / w, ux = wx * rw, uy = wy * rw;
    const float T = mixture_T(we, w, wd, ux, uy);
    out[(4 * S + 0) * N + d] = widen(rho);
    out[(4 * S + 1) * N + d] = widen(ux);
    out[(4 * S + 2) * N + d] = widen(uy);
    out[(4 * S + 3) * N + d] = widen(T);
    out[(4 * S + 4) * N + d] = widen(ntot) * widen(T);
}

// Weights of the nonequilibrium sums, products of the ring constants with m
// formed on the host: on the FP64 pipe they would be 20 of a species' 250
// operations.
template <int S>
struct NoneqConsts {
    OutConsts<S> c;
    double v2[S][4], qv[S][4], v3[S][4], qv2[S][4];  // m v^2, m q v, m v^3, m q v^2
    double inv_m[S];
};

template <int S>
inline NoneqConsts<S> noneq_consts(const OutConsts<S> &c)
{
    NoneqConsts<S> k;
    memset(&k, 0, sizeof(k));
    k.c = c;
    for (int s = 0; s < S; ++s) {
        for (int r = 0; r < 4; ++r) {
            const double v = c.vr[s][r], q = c.qr[s][r];
            k.v2[s][r] = c.m[s] * (v * v);
            k.qv[s][r] = c.m[s] * (q * v);
            k.v3[s][r] = c.m[s] * (v * v * v);
            k.qv2[s][r] = c.m[s] * (q * v * v);
        }
        k.inv_m[s] = 1.0 / c.m[s];
    }
    return k;
}

// m times the moments of rows 5..16 of M (xx, xy, yy, q x, q y, xxx, xxy, xyy,
// yyy, q xx, q xy, q yy) of one species' values; with LOW also n, j_x, j_y, E.
template <bool LOW, int S>
__device__ __forceinline__ void high_moments(const NoneqConsts<S> &k, int s, const double f[Q], double t[12],
                                             double low[4])
{
#pragma unroll
    for (int j = 0; j < 12; ++j) t[j] = 0.0;
    if (LOW) low[0] = low[1] = low[2] = low[3] = 0.0;
#pragma unroll
    for (int r = 0; r < 4; ++r) {
        const RingSums g = ring_sums(r, f + 4 * r);
        if (LOW) {
            low[0] += g.all;
            low[1] += k.c.vr[s][r] * g.rx;
            low[2] += k.c.vr[s][r] * g.ry;
            low[3] += k.c.qr[s][r] * g.all;
        }
        if (r & 1) {  // xx and yy are the ring's sum, xxx = xyy, xxy = yyy
            const double e2 = k.v2[s][r] * g.all, e4 = k.qv2[s][r] * g.all;
            const double cx = k.v3[s][r] * g.rx, cy = k.v3[s][r] * g.ry;
            t[0] += e2;
            t[2] += e2;
            t[9] += e4;
            t[11] += e4;
            t[5] += cx;
            t[7] += cx;
            t[6] += cy;
            t[8] += cy;
            t[1] += k.v2[s][r] * g.xy;
            t[10] += k.qv2[s][r] * g.xy;
        } else {
            t[0] += k.v2[s][r] * g.xx;
            t[2] += k.v2[s][r] * g.yy;
            t[9] += k.qv2[s][r] * g.xx;
            t[11] += k.qv2[s][r] * g.yy;
            t[5] += k.v3[s][r] * g.rx;
            t[8] += k.v3[s][r] * g.ry;
        }
        t[3] += k.qv[s][r] * g.rx;
        t[4] += k.qv[s][r] * g.ry;
    }
}

// Nonequilibrium moments.  The equilibrium is M^-1 f-hat, so its moments of
// the 16 monomials of M are f-hat itself, and all twelve moments of the
// output are among them: Delta = m (M f - f-hat).  Neither f^eq nor a sum
// over it is needed, and M f comes from ring sums: under 200 FP64 operations
// per species and cell where summing f - f^eq over the velocities took 1400
// (the FP64 pipe bounds this kernel: 2048 x 1024, two species, 7.9 -> 1.63
// ms).  Up to two species keep their sums in registers until the mixture u and
// T are known; more load their values again.
template <int S, class Src>
__global__ void __launch_bounds__(128)
    k_noneq(const __grid_constant__ NoneqConsts<S> k, const __grid_constant__ Src src,
            double *__restrict__ out)
{
    const OutConsts<S> &c = k.c;
    const int x = blockIdx.x * blockDim.x + threadIdx.x;
    const int y = blockIdx.y * blockDim.y + threadIdx.y;
    if (x >= c.nx || y >= c.ny) return;
    const long long N = (long long)c.nx * c.ny;
    const long long d = (long long)y * c.nx + x;
    const long long cell = (long long)(y + GY) * c.pitch + (x + GX);
    constexpr bool KEEP = S <= 2;
    double n[S], jx[S], jy[S], en[S], kept[KEEP ? S : 1][12], low[4];
    if constexpr (KEEP) {
#pragma unroll
        for (int s = 0; s < S; ++s) {
            double fc[Q];
            src.load16(s, cell, fc);
            high_moments<true>(k, s, fc, kept[s], low);
            n[s] = low[0], jx[s] = low[1], jy[s] = low[2], en[s] = low[3];
        }
    } else {
        cell_moments<S>(c, src, cell, n, jx, jy, en);
    }
    double ux, uy, T;
    cell_mixture<S>(c, n, jx, jy, en, ux, uy, T);
#pragma unroll(S <= 2 ? S : 1)
    for (int s = 0; s < S; ++s) {
        double fh[Q], t[12];
        double ns = n[0];  // selected, not indexed
#pragma unroll
        for (int j = 1; j < S; ++j)
            if (s == j) ns = n[j];
        if constexpr (KEEP) {
#pragma unroll
            for (int j = 0; j < 12; ++j) t[j] = kept[s][j];
        } else {
            double fc[Q];
            src.load16(s, cell, fc);
            high_moments<false>(k, s, fc, t, low);
        }
        // f-hat is linear in n: m f-hat is that of m n
        fhat16<double>(c.m[s] * ns, ux, uy, T * k.inv_m[s], c.dpi[s], fh);
        double *o = out + 20LL * s * N + d;
#pragma unroll
        for (int j = 0; j < 12; ++j) o[j * N] = t[j] - fh[4 + j];
        o[12 * N] = 0.5 * t[0];
        o[13 * N] = 0.5 * t[2];
        o[14 * N] = 0.5 * fh[4];
        o[15 * N] = 0.5 * fh[6];
        o[16 * N] = 0.5 * t[3];
        o[17 * N] = 0.5 * t[4];
        o[18 * N] = 0.5 * fh[7];
        o[19 * N] = 0.5 * fh[8];
    }
}

// Conserved totals: each block sums a fixed, strided subset of one species'
// cells in a fixed order and reduces it by a fixed tree; the final kernel
// adds the block partials in a fixed order.  The result is independent of
// timing.
//
// The totals are linear in f, so a thread only adds up its cells (float states:
// each velocity; FP64 states: 12 ring sums a species) and the block forms mass,
// momentum and energy from the sums once.  Float states: a velocity's running
// total over 32 cells is three floats, h + l + t: h and l take each value by
// exact two-sums and only t, at most 2^-38 of the magnitudes added, is rounded,
// 2^-57 of them in the worst case, so nothing is lost that FP64 additions of
// the values would keep; a total past the float range is formed again in FP64.
// This runs on the FP32 pipes, 13 additions a value; the FP64 pipe, two lanes
// per SM and cycle, gets one per species and cell.  Multiplying every value by its
// weights in FP64 took 190 (4096^2, two species: 8.7 -> 0.59 ms; with the ring
// sums of a group and twelve trees a warp in FP64 0.67).
struct FloatTriple {
    float h, l, t;
    __device__ __forceinline__ void add(float f)
    {
        float e, e2;
        h = ff_sum(h, f, e);
        l = ff_sum(l, e, e2);
        t = __fadd_rn(t, e2);
    }
    __device__ __forceinline__ double value() const { return widen(h) + (widen(l) + widen(t)); }
    __device__ __forceinline__ float size() const { return fabsf(h) + fabsf(t); }  // not finite when any part is not
};
// a + sign b, exactly but for the rounding of t
__device__ __forceinline__ FloatTriple triple_sum(const FloatTriple &a, const FloatTriple &b, float sign)
{
    FloatTriple s;
    float e, e1, e2;
    s.h = ff_sum(a.h, sign * b.h, e);
    const float m = ff_sum(a.l, sign * b.l, e1);
    s.l = ff_sum(m, e, e2);
    s.t = __fadd_rn(__fmaf_rn(sign, b.t, a.t), __fadd_rn(e1, e2));
    return s;
}

// Running totals of a species over a thread's cells.
struct SpeciesTotalF {
    FloatTriple a[Q];
    __device__ __forceinline__ void clear()
    {
#pragma unroll
        for (int i = 0; i < Q; ++i) a[i].h = a[i].l = a[i].t = 0.0f;
    }
    __device__ __forceinline__ void add_ring(int r, float f0, float f1, float f2, float f3)
    {
        a[4 * r].add(f0), a[4 * r + 1].add(f1), a[4 * r + 2].add(f2), a[4 * r + 3].add(f3);
    }
    // adds the ring sums; false, and nothing added, when a value was infinite or
    // NaN or a float total left the range (a running total that overflowed stays
    // infinite or NaN)
    __device__ __forceinline__ bool flush(double acc[4][3]) const
    {
        bool finite = true;
#pragma unroll
        for (int r = 0; r < 4; ++r)  // of a ring's sums, so of its four totals
            finite = finite && a[4 * r].size() + a[4 * r + 1].size() + a[4 * r + 2].size() + a[4 * r + 3].size() < 0x1p127f;
        if (!finite) return false;
#pragma unroll
        for (int r = 0; r < 4; ++r) {
            // the ring's sums as in ring_sums
            const FloatTriple *f = a + 4 * r;
            const FloatTriple p = triple_sum(f[0], f[2], 1.0f), q = triple_sum(f[1], f[3], 1.0f);
            const FloatTriple d = triple_sum(f[0], f[2], -1.0f), e = triple_sum(f[3], f[1], -1.0f);
            acc[r][0] += triple_sum(p, q, 1.0f).value();
            acc[r][1] += (r & 1) ? triple_sum(d, e, 1.0f).value() : d.value();
            acc[r][2] += (r & 1) ? triple_sum(d, e, -1.0f).value() : -e.value();
        }
        return true;
    }
};
struct SpeciesTotalD {
    double a[4][3];
    __device__ __forceinline__ void clear()
    {
#pragma unroll
        for (int r = 0; r < 4; ++r) a[r][0] = a[r][1] = a[r][2] = 0.0;
    }
    __device__ __forceinline__ void add_ring(int r, double f0, double f1, double f2, double f3)
    {
        const double f[4] = {f0, f1, f2, f3};
        const RingSums g = ring_sums(r, f);
        a[r][0] += g.all, a[r][1] += g.rx, a[r][2] += g.ry;
    }
    __device__ __forceinline__ bool flush(double acc[4][3]) const
    {
#pragma unroll
        for (int r = 0; r < 4; ++r) acc[r][0] += a[r][0], acc[r][1] += a[r][1], acc[r][2] += a[r][2];
        return true;
    }
};

// The values of velocities 4 r .. 4 r + 3 of four cells in a row, v[velocity][cell]
// (rows start 16-byte aligned; the row's padding covers a ragged last vector).
__device__ __forceinline__ void load_ring4(const float *p, long long plane, float v[4][4])
{
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const float4 q = __ldg(reinterpret_cast<const float4 *>(p + i * plane));
        v[i][0] = q.x, v[i][1] = q.y, v[i][2] = q.z, v[i][3] = q.w;
    }
}
__device__ __forceinline__ void load_ring4(const double *p, long long plane, double v[4][4])
{
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const double2 q = __ldg(reinterpret_cast<const double2 *>(p + i * plane));
        const double2 w = __ldg(reinterpret_cast<const double2 *>(p + i * plane) + 1);
        v[i][0] = q.x, v[i][1] = q.y, v[i][2] = w.x, v[i][3] = w.y;
    }
}

template <class Total, typename real>
__device__ __forceinline__ void total_cells(const PlainSrc<real> &src, int s, long long cell, int live, Total &tot)
{
#pragma unroll
    for (int r = 0; r < 4; ++r) {
        real v[4][4];
        load_ring4(src.f + (s * Q + 4 * r) * src.plane + cell, src.plane, v);
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            if (j >= live) break;
            tot.add_ring(r, v[0][j], v[1][j], v[2][j], v[3][j]);
        }
    }
}
template <class Total, int S>
__device__ __forceinline__ void total_cells(const BfSrc<S> &src, int s, long long cell, int live, Total &tot)
{
#pragma unroll 1
    for (int j = 0; j < live; ++j) {
        float f[Q];
        src.load16f(s, cell + j, f);
#pragma unroll
        for (int r = 0; r < 4; ++r) tot.add_ring(r, f[4 * r], f[4 * r + 1], f[4 * r + 2], f[4 * r + 3]);
    }
}

// Blocks per species: four partials each, within the scratch's CONS_BLOCKS
// times S + 4.
constexpr int cons_blocks(int S) { return S == 1 ? 512 : CONS_BLOCKS / 4 * (S + 4) / S; }
static_assert(4 * 1 * cons_blocks(1) <= CONS_BLOCKS * 5 && 4 * 2 * cons_blocks(2) <= CONS_BLOCKS * 6 &&
                  4 * 3 * cons_blocks(3) <= CONS_BLOCKS * 7 && 4 * 4 * cons_blocks(4) <= CONS_BLOCKS * 8 &&
                  4 * 5 * cons_blocks(5) <= CONS_BLOCKS * 9 && 4 * 6 * cons_blocks(6) <= CONS_BLOCKS * 10 &&
                  4 * 7 * cons_blocks(7) <= CONS_BLOCKS * 11 && 4 * 8 * cons_blocks(8) <= CONS_BLOCKS * 12,
              "conservation partials exceed the scratch buffer");

__device__ __forceinline__ double warp_total(double v)
{
#pragma unroll
    for (int w = 16; w > 0; w >>= 1) v += __shfl_down_sync(0xffffffffu, v, w);
    return v;
}

// The totals of twelve values over a warp, to out[0 .. 11].  Each exchange also
// halves what a lane goes on with (12, 6, 3, 2, 1 values), so a lane makes 13
// FP64 additions where twelve trees of their own take 60; the additions of a
// value, and so its bits, are those of warp_total.
__device__ __forceinline__ void warp_totals(const double *v, double *out)
{
    const int lane = threadIdx.x & 31;
    double a[6], b[3];
#pragma unroll
    for (int i = 0; i < 6; ++i) {
        const bool up = lane & 16;
        a[i] = (up ? v[6 + i] : v[i]) + __shfl_xor_sync(0xffffffffu, up ? v[i] : v[6 + i], 16);
    }
#pragma unroll
    for (int i = 0; i < 3; ++i) {
        const bool up = lane & 8;
        b[i] = (up ? a[3 + i] : a[i]) + __shfl_xor_sync(0xffffffffu, up ? a[i] : a[3 + i], 8);
    }
    const bool third = lane & 4, second = lane & 2;
    const double c0 = (third ? b[2] : b[0]) + __shfl_xor_sync(0xffffffffu, third ? b[0] : b[2], 4);
    const double c1 = b[1] + __shfl_xor_sync(0xffffffffu, b[1], 4);
    double d = (second ? c1 : c0) + __shfl_xor_sync(0xffffffffu, second ? c0 : c1, 2);
    d += __shfl_xor_sync(0xffffffffu, d, 1);
    if ((lane & 1) == 0 && !(third && second))
        out[(lane & 16 ? 6 : 0) + (lane & 8 ? 3 : 0) + (third ? 2 : second ? 1 : 0)] = d;
}

template <int S, class Src>
__global__ void __launch_bounds__(256, 2)
    k_cons_partial(const __grid_constant__ OutConsts<S> c, const __grid_constant__ Src src,
                   double *__restrict__ partial)
{
    constexpr bool DOUBLE = std::is_same<typename Src::value, double>::value;
    using Total = typename std::conditional<DOUBLE, SpeciesTotalD, SpeciesTotalF>::type;
    constexpr unsigned FLUSH = 8;  // vectors of four cells between additions to the FP64 sums
    const int s = blockIdx.y;
    double acc[4][3];
    Total tot;
#pragma unroll
    for (int r = 0; r < 4; ++r) acc[r][0] = acc[r][1] = acc[r][2] = 0.0;
    const unsigned nv = (unsigned)(c.nx + 3) / 4u, count = nv * (unsigned)c.ny;
    const unsigned stride = gridDim.x * 256u;
    unsigned t = blockIdx.x * 256u + threadIdx.x;
    while (t < count) {
        const unsigned first = t;
        tot.clear();
#pragma unroll 1
        for (unsigned k = 0; k < FLUSH && t < count; ++k, t += stride) {
            const unsigned y = t / nv, x = 4u * (t - y * nv);
            total_cells(src, s, (long long)(y + GY) * c.pitch + (x + GX), min(4, c.nx - (int)x), tot);
        }
        if (tot.flush(acc)) continue;
        // the same cells value by value in FP64
#pragma unroll 1
        for (unsigned q = first; q < t; q += stride) {
            const unsigned y = q / nv, x = 4u * (q - y * nv);
            const long long cell = (long long)(y + GY) * c.pitch + (x + GX);
#pragma unroll 1
            for (int j = 0; j < min(4, c.nx - (int)x); ++j) {
                double f[Q];
                src.load16(s, cell + j, f);
#pragma unroll
                for (int r = 0; r < 4; ++r) {
                    const RingSums g = ring_sums(r, f + 4 * r);
                    acc[r][0] += g.all, acc[r][1] += g.rx, acc[r][2] += g.ry;
                }
            }
        }
    }
    __shared__ double red[8][12];
    warp_totals(&acc[0][0], red[threadIdx.x >> 5]);
    __syncthreads();
    if (threadIdx.x == 0) {
        double n = 0.0, jx = 0.0, jy = 0.0, en = 0.0;
#pragma unroll
        for (int r = 0; r < 4; ++r) {
            double g[3];
#pragma unroll
            for (int k = 0; k < 3; ++k) {
                g[k] = 0.0;
#pragma unroll
                for (int w = 0; w < 8; ++w) g[k] += red[w][3 * r + k];
            }
            n += g[0];
            jx += c.vr[s][r] * g[1];
            jy += c.vr[s][r] * g[2];
            en += c.qr[s][r] * g[0];
        }
        double *p = partial + 4 * ((long long)s * gridDim.x + blockIdx.x);
        p[0] = n;
        p[1] = jx;
        p[2] = jy;
        p[3] = en;
    }
}

// One warp per species and sum (128 S threads).
template <int S>
static __global__ void __launch_bounds__(128 * S)
    k_cons_final(const __grid_constant__ OutConsts<S> c, const double *__restrict__ partial, int nblocks,
                 double *__restrict__ out)
{
    __shared__ double sum[S][4];
    const int w = threadIdx.x >> 5, lane = threadIdx.x & 31, s = w >> 2, k = w & 3;
    double v = 0.0;
    for (int b = lane; b < nblocks; b += 32) v += partial[4 * ((long long)s * nblocks + b) + k];
    v = warp_total(v);
    if (lane == 0) sum[s][k] = v;
    __syncthreads();
    if (threadIdx.x != 0) return;
    double px = 0.0, py = 0.0, en = 0.0, heat = 0.0;
    for (int q = 0; q < S; ++q) {
        const double m = c.m[q];
        out[q] = m * sum[q][0];
        px += m * sum[q][1];
        py += m * sum[q][2];
        en += 0.5 * m * sum[q][3];
        if (c.has_reaction && q == c.fuel) heat = c.Qheat * sum[q][0] / c.abs_a_fuel;
    }
    out[S] = px;
    out[S + 1] = py;
    out[S + 2] = en;
    out[S + 3] = heat;
}

inline dim3 cell_grid(const dbm_handle *h, dim3 block)
{
    return dim3((h->p.nx + block.x - 1) / block.x, (h->p.ny + block.y - 1) / block.y);
}

template <typename real, int S>
inline void set_state_t(dbm_handle *h, void *f, const double *rho_s, const double *ux,
                        const double *uy, const double *T, cudaStream_t st)
{
    dim3 b(32, 8);
    if constexpr (sizeof(real) == 4) {
        StepConsts<float, S> c;
        fill_step_consts<float, S>(h, c);
        InvMass<S> im;
        for (int s = 0; s < S; ++s) im.v[s] = 1.0 / h->p.sp[s].m;
        k_set_state_blocks<S><<<cell_grid(h, b), b, 0, st>>>(c, (float *)f, rho_s, ux, uy, T, im);
    } else {
        OutConsts<S> c;
        fill_out_consts<S>(h, c);
        k_set_state<real, S><<<cell_grid(h, b), b, 0, st>>>(c, (real *)f, rho_s, ux, uy, T);
    }
}

// The source of f for a state buffer of this handle's precision.
template <typename real, int S>
inline PlainSrc<real> plain_src(const dbm_handle *h, const void *f)
{
    return PlainSrc<real>{(const real *)f, h->lay.plane};
}
template <int S>
inline BfSrc<S> bf_src(const dbm_handle *h, const void *f)
{
    BfSrc<S> b;
    fill_step_consts<float, S>(h, b.k);
    b.st = bf_state(h, (void *)f);
    return b;
}

template <int S, class Src>
inline void moments_t(dbm_handle *h, const Src &src, double *out, cudaStream_t st)
{
    OutConsts<S> c;
    fill_out_consts<S>(h, c);
    dim3 b(32, 8);
    if constexpr (std::is_same<typename Src::value, double>::value)
        k_moments<S, Src><<<cell_grid(h, b), b, 0, st>>>(c, src, out);
    else
        k_moments_f32<S, Src><<<cell_grid(h, b), b, 0, st>>>(moment_consts<S>(c), src, out);
}

template <int S, class Src>
inline void noneq_t(dbm_handle *h, const Src &src, double *out, cudaStream_t st)
{
    OutConsts<S> c;
    fill_out_consts<S>(h, c);
    dim3 b(32, 4);
    k_noneq<S, Src><<<cell_grid(h, b), b, 0, st>>>(noneq_consts<S>(c), src, out);
}

template <int S, class Src>
inline void cons_t(dbm_handle *h, const Src &src, double *partial, double *out, cudaStream_t st)
{
    OutConsts<S> c;
    fill_out_consts<S>(h, c);
    const long long vectors = (long long)((h->p.nx + 3) / 4) * h->p.ny;
    const long long full = (vectors + 255) / 256;
    const int blocks = (int)(full < cons_blocks(S) ? full : cons_blocks(S));
    k_cons_partial<S, Src><<<dim3(blocks, S), 256, 0, st>>>(c, src, partial);
    k_cons_final<S><<<1, 128 * S, 0, st>>>(c, partial, blocks, out);
}


// The launches of one species count, dispatching on the handle's precision
// (the BF16-deviation state exists for S <= 4).
template <int S>
void aux_set_state(dbm_handle *h, void *f, const double *rho_s, const double *ux, const double *uy, const double *T,
                   cudaStream_t st)
{
    if (h->p.precision == DBM_FP64)
        set_state_t<double, S>(h, f, rho_s, ux, uy, T, st);
    else
        set_state_t<float, S>(h, f, rho_s, ux, uy, T, st);
}

template <int S>
void aux_moments(dbm_handle *h, const void *f, double *out, cudaStream_t st)
{
    if (h->p.precision == DBM_FP64) {
        moments_t<S>(h, plain_src<double, S>(h, f), out, st);
    } else if (h->p.precision == DBM_FP32) {
        moments_t<S>(h, plain_src<float, S>(h, f), out, st);
    } else if constexpr (S <= 4) {
        moments_t<S>(h, bf_src<S>(h, f), out, st);
    }
}

template <int S>
void aux_noneq(dbm_handle *h, const void *f, double *out, cudaStream_t st)
{
    if (h->p.precision == DBM_FP64) {
        noneq_t<S>(h, plain_src<double, S>(h, f), out, st);
    } else if (h->p.precision == DBM_FP32) {
        noneq_t<S>(h, plain_src<float, S>(h, f), out, st);
    } else if constexpr (S <= 4) {
        noneq_t<S>(h, bf_src<S>(h, f), out, st);
    }
}

template <int S>
void aux_cons(dbm_handle *h, const void *f, double *partial, double *out, cudaStream_t st)
{
    if (h->p.precision == DBM_FP64) {
        cons_t<S>(h, plain_src<double, S>(h, f), partial, out, st);
    } else if (h->p.precision == DBM_FP32) {
        cons_t<S>(h, plain_src<float, S>(h, f), partial, out, st);
    } else if constexpr (S <= 4) {
        cons_t<S>(h, bf_src<S>(h, f), partial, out, st);
    }
}

}  // namespace dbm

// dbm_step_f64.cu -- the FP64 step, in reference operation order.
//
// The FP64 path is the parity path of the library: its results are held to
// a relative L-inf of 1e-12 against a plain FP64 CPU evaluation of the
// paper's formulas after thousands of steps, through shocks.  Two FP64
// evaluations of the same step that merely round in a different order
// drift apart by ~1e-12 over 2000 steps of a shock tube (the limiter and
// the relaxation pass every rounding difference on), so this kernel
// evaluates each formula with the same operands in the same order as it is
// printed, and this translation unit is compiled without multiply-add
// contraction (--fmad=false):
//   - species moments n = sum f, n u = sum f v, E = sum f (v.v + eta^2),
//     T^s = m (E/n - u.u)/(D+I)  (section "Discrete Boltzmann model");
//   - mixture u = sum(rho u^s/tau)/sum(rho/tau),
//     T = sum((m E - rho u.u)/tau)/sum(n (D+I)/tau) (momentum and energy
//     conservation of Eq. CollisionTerm);
//   - f^eq = M^-1 f-hat with the f-hat list as printed; Omega, R and G as
//     separate terms (Eqs. CollisionTerm, ReactionTerm, ForceTerm);
//   - NND fluxes H from the split fluxes F+- = (c +- |c|)/2 f;
//   - f^{n+1} = f + dt (Omega + R + G - d(v_x f)/dx - d(v_y f)/dy).
//
// What bounds it: the FP64 pipe, two lanes per SM and cycle on this GPU (a
// warp's instruction occupies it for 16 cycles; 64 FP32 or integer lanes go
// by meanwhile).  So the work is arranged to issue few FP64 instructions, to
// fill their 32 lanes, and to reach every SM; everything that rounds the same
// with less of that pipe is done with less:
//   - the half of each split flux that is zero is left out, the limiter is a
//     choice between its arguments on the integer pipe, and its half joins
//     the flux in one multiply-add (the half of a double is exact);
//   - in M^-1 f-hat, the entries that vanish by symmetry (at most 1e-31 of
//     their neighbours as computed) are left out, and the four velocities of
//     a ring, whose entries differ in sign only, share each product;
//   - a division by a constant b is a product with 1/b and two multiply-adds
//     (Markstein 1990: with y = RN(1/b), q = RN(a y), r = RN(a - q b) exact,
//     RN(q + r y) is the rounded quotient).
// About 1000 FP64 instructions per species and cell; the plain form of the same
// arithmetic had 2500 (two species, 512 x 384: 2342 us a step, now 745,
// with the pipe at the rate that back-to-back additions reach, one warp
// instruction in 19 cycles).
//
// A CTA steps CELLS cells (consecutive in row order, so ragged rows leave no
// lane idle) in phases through shared memory, each with its own split:
//   1  the 4 moment sums of a cell and species, one thread each (each sum is
//      a serial chain, the four run side by side);
//   2  species velocities and weights;
//   3  mixture u, T and the rate;
//   4  f-hat of each term;
//   5  collision, advection and update, a warp per ring of four velocities.
// k_step_f64: 32 cells, in phase 5 the ring's four velocities in each thread
// (shared products).  k_step_f64_small: 4 cells, for grids that leave the chip
// idle, where the chain of dependent operations is the time: a warp issues an
// FP64 instruction at most every 64 cycles whatever the others do, so every
// phase is spread over warps (see there).
// Ghosts of the new state are written as images by the edge cells.
#include "dbm_consts.h"
#include "dbm_device.cuh"
#include "dbm_step_impl.cuh"

namespace dbm {

// a / d.b rounded to nearest (see above).  Operands whose remainder could
// leave the normal range, and divisors a host check refuses (span 0), take
// the division itself.
__device__ __forceinline__ double div_by(double a, const ConstDiv &d)
{
    const unsigned hi = (unsigned)__double2hiint(a) & 0x7fffffffu;
    const bool zero = (hi | (unsigned)__double2loint(a)) == 0u;
    if ((hi >> 20) - d.lo <= d.span || (zero && d.span != 0u)) {
        const double q = a * d.y;
        return fma(fma(-q, d.b, a), d.y, q);
    }
    return a / d.b;
}

// minmod(a, b) = (sgn a + sgn b)/2 min(|a|, |b|): one of the arguments or 0,
// chosen by integer comparisons of the bits.
__device__ __forceinline__ double minmod_bits(double a, double b)
{
    const long long ia = __double_as_longlong(a), ib = __double_as_longlong(b);
    const long long ma = ia & 0x7fffffffffffffffLL, mb = ib & 0x7fffffffffffffffLL;
    const long long m = ma < mb ? ia : ib;
    return (ia ^ ib) < 0 ? 0.0 : __longlong_as_double(m);
}

// d(c f)/dx of one velocity component of magnitude v at a cell: fm2, fm1, fp1
// are f two cells and one cell upwind and one downwind, g0 = v f at the cell, h
// the grid spacing.  Seen along c, both signs have the same flux
// H = v f + minmod(...)/2.
__device__ __forceinline__ double nnd_dflux(double fm2, double fm1, double fp1, double g0, double v,
                                            const ConstDiv &h)
{
    const double gm2 = v * fm2, gm1 = v * fm1, gp1 = v * fp1;
    const double d0 = gm1 - gm2, d1 = g0 - gm1, d2 = gp1 - g0;
    const double hr = fma(0.5, minmod_bits(d1, d2), g0), hl = fma(0.5, minmod_bits(d0, d1), gm1);
    return div_by(hr - hl, h);
}

// f-hat_1..16 at (n, u, T) for a species of mass m and extra degrees of
// freedom I, theta = T/m, D = 2, in the printed form; written to
// fh[k * stride].  PART 0..3: a quarter of the work each; -1: all of it.
template <int PART = -1>
__device__ __forceinline__ void fhat_printed(double n, double ux, double uy, double T, const ConstDiv &m, double I,
                                             double *fh, int stride)
{
    constexpr bool ALL = PART < 0;
    const double D = 2.0;
    const double th = div_by(T, m);
    const double u2 = ux * ux + uy * uy;
    const double a0 = (D + I) * th + u2, a2 = (D + I + 2.0) * th + u2, a4 = (D + I + 4.0) * th + u2;
    if (ALL || PART == 0) {
        fh[0] = n;
        fh[1 * stride] = n * ux;
        fh[2 * stride] = n * uy;
        fh[4 * stride] = n * (th + ux * ux);
        fh[5 * stride] = n * ux * uy;
        fh[6 * stride] = n * (th + uy * uy);
        fh[10 * stride] = n * uy * th + n * ux * ux * uy;
    }
    if (ALL || PART == 1) {
        fh[3 * stride] = n * a0;
        fh[7 * stride] = n * ux * a2;
        fh[8 * stride] = n * uy * a2;
        fh[14 * stride] = n * ux * uy * a4;
    }
    if (ALL || PART == 2) {
        fh[9 * stride] = 3.0 * n * ux * th + n * ux * ux * ux;
        fh[11 * stride] = n * ux * th + n * ux * uy * uy;
        fh[12 * stride] = 3.0 * n * uy * th + n * uy * uy * uy;
    }
    if (ALL || PART == 3) {
        fh[13 * stride] = n * a2 * th + n * ux * ux * a4;
        fh[15 * stride] = n * a2 * th + n * uy * uy * a4;
    }
}

// Rows of M^-1.  The row of the ring's first velocity, (+,0) or (+,+), gives
// every other: along y an axis ring has the x row's entries at the mirrored
// moments, opposite velocities have the odd moments negated, and on the
// diagonals the sign of an entry is that of its moment.  Terms are added in
// the printed order k = 0..15.
__host__ __device__ constexpr int axis_k(int y, int j)  // moments of an axis row, in order
{
    return y ? (j == 0 ? 0 : j == 1 ? 2 : j == 2 ? 3 : j == 3 ? 4 : j == 4 ? 6 : j == 5 ? 8 : j == 6 ? 10 : j == 7 ? 12
                : j == 8 ? 13 : 15)
             : (j == 0 ? 0 : j == 1 ? 1 : j == 2 ? 3 : j == 3 ? 4 : j == 4 ? 6 : j == 5 ? 7 : j == 6 ? 9 : j == 7 ? 11
                : j == 8 ? 13 : 15);
}
__host__ __device__ constexpr int axis_c(int y, int j)  // where the x row has that entry
{
    return y ? (j == 0 ? 0 : j == 1 ? 1 : j == 2 ? 3 : j == 3 ? 6 : j == 4 ? 4 : j == 5 ? 7 : j == 6 ? 11 : j == 7 ? 9
                : j == 8 ? 15 : 13)
             : axis_k(0, j);
}
__host__ __device__ constexpr bool axis_odd(int j) { return j == 1 || j == 5 || j == 6 || j == 7; }
// powers of v_x and v_y (mod 2) in moment k
__host__ __device__ constexpr bool odd_x(int k) { return k == 1 || k == 5 || k == 7 || k == 9 || k == 11 || k == 14; }
__host__ __device__ constexpr bool odd_y(int k) { return k == 2 || k == 5 || k == 8 || k == 10 || k == 12 || k == 14; }

// Output of the ring's equilibrium: V = 4 velocities per thread (lane: cell)
// or V = 1 (velocity `vel` of the ring).  row: 16 entries of the ring's
// first velocity; fh[k * CELLS]: the cell's moments.
template <bool DIAG, int V, int CELLS>
__device__ __forceinline__ void ring_equilibrium(const double *row, const double *fh, int vel, double f[V])
{
    if constexpr (DIAG) {
#pragma unroll
        for (int k = 0; k < Q; ++k) {
            const double t = row[k] * fh[k * CELLS];
#pragma unroll
            for (int v = 0; v < V; ++v) {
                const int i = V == 4 ? v : vel;
                const bool neg = (odd_x(k) && (i == 1 || i == 2)) != (odd_y(k) && (i == 2 || i == 3));
                const double s = neg ? -t : t;
                f[v] = k == 0 ? s : f[v] + s;
            }
        }
    } else if constexpr (V == 4) {
#pragma unroll
        for (int y = 0; y < 2; ++y)
#pragma unroll
            for (int j = 0; j < 10; ++j) {
                const double t = row[axis_c(y, j)] * fh[axis_k(y, j) * CELLS];
                f[y] = j == 0 ? t : f[y] + t;
                f[y + 2] = j == 0 ? t : axis_odd(j) ? f[y + 2] - t : f[y + 2] + t;
            }
    } else {
        const bool y = vel & 1, back = vel & 2;
#pragma unroll
        for (int j = 0; j < 10; ++j) {
            const double c = y ? row[axis_c(1, j)] : row[axis_c(0, j)];
            const double t = c * fh[(y ? axis_k(1, j) : axis_k(0, j)) * CELLS];
            const double s = axis_odd(j) && back ? -t : t;
            f[0] = j == 0 ? s : f[0] + s;
        }
    }
}

// Moment sum k of a species (n, j_x, j_y, E), terms in velocity order.
template <int K>
__device__ __forceinline__ double moment_sum(const double v[4], const double q[4], const double f[Q])
{
    double sum = 0.0;
#pragma unroll
    for (int i = 0; i < Q; ++i) {
        if ((K == 1 && dir_x(i) == 0) || (K == 2 && dir_y(i) == 0)) continue;
        const double w = K == 1 ? dir_x(i) * v[i >> 2] : K == 2 ? dir_y(i) * v[i >> 2] : q[i >> 2];
        sum = sum + (K == 0 ? f[i] : f[i] * w);
    }
    return sum;
}

// Values of a cell and species between phases 2 and 4, and of a cell
// between 3 and 4.
enum { W_RHO = 0, W_LAM, W_LX, W_LY, W_ME, W_CAP, W_UX, W_UY, W_TS, W_N };
enum { M_UX = 0, M_UY, M_T, M_NTOT, M_OMEGA, M_DT, M_COUNT };

__host__ __device__ constexpr int f64_side(int S) { return S >= 2 ? 2 : 1; }  // species side by side in phase 5

template <int S>
constexpr size_t f64_smem(int cells, int sets)
{
    return sizeof(double) * (size_t)cells * (S * Q * sets + S * (4 + W_N) + M_COUNT);
}

template <int S>
__global__ void __launch_bounds__(128 * f64_side(S))
    k_step_f64(const __grid_constant__ F64Consts<S> c, const ChainedIn<double> in,
               double *__restrict__ fout, unsigned *__restrict__ flag)
{
    constexpr int CELLS = 32, SW = f64_side(S), NT = 128 * SW, V = 4;
    extern __shared__ __align__(16) double sm[];
    double *mom = sm;                          // [S][4][CELLS]
    double *wts = mom + S * 4 * CELLS;         // [S][W_N][CELLS]
    double *mix = wts + S * W_N * CELLS;       // [M_COUNT][CELLS]
    double *fhs = mix + M_COUNT * CELLS;       // [sets][S][Q][CELLS]
    const long long P = c.plane;
    const unsigned d0 = blockIdx.x * (unsigned)CELLS, total = (unsigned)c.nx * (unsigned)c.ny;
    const int tid = threadIdx.x;
    const bool react = c.has_reaction != 0, force = c.has_force != 0;
    // a cell past the end takes the last one's values and stores nothing
    auto locate = [&](int j, unsigned &x, unsigned &y) {
        const unsigned d = min(d0 + (unsigned)j, total - 1u);
        y = d / (unsigned)c.nx;
        x = d - y * (unsigned)c.nx;
        return (long long)(y + GY) * c.pitch + (x + GX);
    };

    const double *fin = in.wait();

    // 1. moment sums
#pragma unroll 1
    for (int it = tid; it < S * 4 * CELLS; it += NT) {
        const int j = it % CELLS, k = (it / CELLS) & 3, s = it / (4 * CELLS);
        unsigned x, y;
        const long long cell = locate(j, x, y);
        const double *pl = fin + (long long)s * Q * P + cell;
        double f[Q], sum;
#pragma unroll
        for (int i = 0; i < Q; ++i) f[i] = pl[i * P];
        // k is uniform over a warp: no products with 1 or 0
        if (k == 0)
            sum = moment_sum<0>(c.vr[s], c.qr[s], f);
        else if (k == 1)
            sum = moment_sum<1>(c.vr[s], c.qr[s], f);
        else if (k == 2)
            sum = moment_sum<2>(c.vr[s], c.qr[s], f);
        else
            sum = moment_sum<3>(c.vr[s], c.qr[s], f);
        mom[(s * 4 + k) * CELLS + j] = sum;
    }
    __syncthreads();

    // 2. species velocities and the weights of the mixture sums
#pragma unroll 1
    for (int it = tid; it < S * CELLS; it += NT) {
        const int j = it % CELLS, s = it / CELLS;
        const double *mo = mom + s * 4 * CELLS + j;
        double *w = wts + s * W_N * CELLS + j;
        const double sn = mo[0], E = mo[3 * CELLS];
        double ux = 0.0, uy = 0.0, Ts = 0.0;  // an absent species: zero velocity and temperature
        if (sn != 0.0) {
            ux = mo[CELLS] / sn;
            uy = mo[2 * CELLS] / sn;
            if (force) Ts = c.md[s].b * (E / sn - (ux * ux + uy * uy)) / (2.0 + c.I[s]);
        }
        const double rho = c.md[s].b * sn;
        w[W_RHO * CELLS] = rho;
        w[W_LAM * CELLS] = div_by(rho, c.taud[s]);
        w[W_LX * CELLS] = div_by(rho * ux, c.taud[s]);
        w[W_LY * CELLS] = div_by(rho * uy, c.taud[s]);
        w[W_ME * CELLS] = c.md[s].b * E;
        w[W_CAP * CELLS] = div_by(sn * (2.0 + c.I[s]), c.taud[s]);
        if (force) {
            w[W_UX * CELLS] = ux;
            w[W_UY * CELLS] = uy;
            w[W_TS * CELLS] = Ts;
        }
    }
    __syncthreads();

    // 3. mixture velocity and temperature, reaction rate
    if (tid < CELLS) {
        const int j = tid;
        const double *mo = mom + j, *w = wts + j;
        double sw = 0.0, sx = 0.0, sy = 0.0, ntot = 0.0;
#pragma unroll
        for (int s = 0; s < S; ++s) {
            sw += w[(s * W_N + W_LAM) * CELLS];
            sx += w[(s * W_N + W_LX) * CELLS];
            sy += w[(s * W_N + W_LY) * CELLS];
            ntot += fabs(mo[s * 4 * CELLS]);
        }
        const double Ux = sx / sw, Uy = sy / sw;
        const double u2 = Ux * Ux + Uy * Uy;
        double num = 0.0, den = 0.0;
#pragma unroll
        for (int s = 0; s < S; ++s) {
            num += div_by(w[(s * W_N + W_ME) * CELLS] - w[(s * W_N + W_RHO) * CELLS] * u2, c.taud[s]);
            den += w[(s * W_N + W_CAP) * CELLS];
        }
        const double T = num / den;
        unsigned bad = 0;
#pragma unroll
        for (int s = 0; s < S; ++s) {
            const double n = mo[s * 4 * CELLS];
            if (!(n >= -1e-6 * ntot) || !isfinite(n)) bad |= DBM_HEALTH_DENSITY;
        }
        if (!(ntot > 0.0)) bad |= DBM_HEALTH_DENSITY;
        if (!(T > 0.0)) bad |= DBM_HEALTH_TEMPERATURE;
        if (!isfinite(T) || !isfinite(Ux) || !isfinite(Uy)) bad |= DBM_HEALTH_NONFINITE;
        double omega = 0.0, dTdt = 0.0;
        if (react) {
            omega = c.k_ov * mo[c.fuel * 4 * CELLS] * mo[c.oxid * 4 * CELLS] * exp(-c.Ea_over_R / T);
            double src = 0.0, cap = 0.0;
#pragma unroll
            for (int s = 0; s < S; ++s) {
                src += (2.0 + c.I[s]) * c.a[s] * omega;
                cap += mo[s * 4 * CELLS] * (2.0 + c.I[s]);
            }
            dTdt = (c.Qheat * omega - 0.5 * T * src) / (0.5 * cap);
        }
        mix[M_UX * CELLS + j] = Ux;
        mix[M_UY * CELLS + j] = Uy;
        mix[M_T * CELLS + j] = T;
        mix[M_NTOT * CELLS + j] = ntot;
        mix[M_OMEGA * CELLS + j] = omega;
        mix[M_DT * CELLS + j] = dTdt;
        if (bad) raise_flag(flag, bad);
    }
    __syncthreads();

    // 4. f-hat of each term: set 0 (n, u, T), then with a reaction (n*, u, T*),
    // then with a force (n, u-dagger, T^s) and (n, u^s, T^s)
    constexpr int SET = S * Q * CELLS;
#pragma unroll 1
    for (int it = tid; it < S * CELLS; it += NT) {
        const int j = it % CELLS, s = it / CELLS;
        const double n = mom[s * 4 * CELLS + j];
        const double Ux = mix[M_UX * CELLS + j], Uy = mix[M_UY * CELLS + j], T = mix[M_T * CELLS + j];
        double *fh = fhs + s * Q * CELLS + j;
        fhat_printed(n, Ux, Uy, T, c.md[s], c.I[s], fh, CELLS);
        if (react) {
            const double tau = c.taud[s].b;
            const double nstar = n + tau * c.a[s] * mix[M_OMEGA * CELLS + j];
            const double Tstar = T + tau * mix[M_DT * CELLS + j];
            if (nstar < -1e-6 * mix[M_NTOT * CELLS + j]) raise_flag(flag, DBM_HEALTH_NSTAR);
            fh += SET;
            fhat_printed(nstar, Ux, Uy, Tstar, c.md[s], c.I[s], fh, CELLS);
        }
        if (force) {
            const double tau = c.taud[s].b;
            const double *w = wts + s * W_N * CELLS + j;
            const double ux = w[W_UX * CELLS], uy = w[W_UY * CELLS], Ts = w[W_TS * CELLS];
            fh += SET;
            fhat_printed(n, ux + c.ax * tau, uy + c.ay * tau, Ts, c.md[s], c.I[s], fh, CELLS);
            fh += SET;
            fhat_printed(n, ux, uy, Ts, c.md[s], c.I[s], fh, CELLS);
        }
    }
    __syncthreads();

    chain_end();

    // 5. collision, advection and update of one ring per warp
    const int warp = tid >> 5, lane = tid & 31, r = warp & 3;
    const int j = lane;
    unsigned x, y;
    const long long cell = locate(j, x, y);
    const bool live = d0 + (unsigned)j < total;
    const unsigned mx = ghost_mask((int)x, c.nx, c.bc_x), my = ghost_mask((int)y, c.ny, c.bc_y);
    auto ring_step = [&](auto diag_tag, int s) {
        constexpr bool DIAG = decltype(diag_tag)::value;
        const double *row = c.row[s][r];
        const ConstDiv tau = c.taud[s];
        const double v = c.vr[s][r];
        double feq[V], rhs[V], f[V], e1[V], e0[V];
#pragma unroll
        for (int q = 0; q < V; ++q) f[q] = fin[(s * Q + 4 * r + q) * P + cell];
        const double *fh = fhs + s * Q * CELLS + j;
        ring_equilibrium<DIAG, V, CELLS>(row, fh, 0, feq);
#pragma unroll
        for (int q = 0; q < V; ++q) rhs[q] = div_by(-(f[q] - feq[q]), tau);  // Omega
        if (react) {
            fh += SET;
            ring_equilibrium<DIAG, V, CELLS>(row, fh, 0, e1);
#pragma unroll
            for (int q = 0; q < V; ++q) rhs[q] = rhs[q] + div_by(e1[q] - feq[q], tau);  // R
        }
        if (force) {
            ring_equilibrium<DIAG, V, CELLS>(row, fh + SET, 0, e1);
            ring_equilibrium<DIAG, V, CELLS>(row, fh + 2 * SET, 0, e0);
#pragma unroll
            for (int q = 0; q < V; ++q) rhs[q] = rhs[q] + div_by(e1[q] - e0[q], tau);  // G
        }
#pragma unroll
        for (int q = 0; q < V; ++q) {
            const int i = q;
            const long long plane = (long long)(s * Q + 4 * r + i) * P;
            const double *pl = fin + plane + cell;
            const double g0 = v * f[q];
            double adv;
            if constexpr (DIAG) {
                const int ex = (i == 1 || i == 2) ? -1 : 1, ey = (i == 2 || i == 3) ? -c.pitch : c.pitch;
                adv = nnd_dflux(pl[-2 * ex], pl[-ex], pl[ex], g0, v, c.dxd);
                adv += nnd_dflux(pl[-2 * ey], pl[-ey], pl[ey], g0, v, c.dyd);
            } else {
                const int st = (i & 1) ? c.pitch : 1, e = (i & 2) ? -st : st;
                adv = nnd_dflux(pl[-2 * e], pl[-e], pl[e], g0, v, (i & 1) ? c.dyd : c.dxd);
            }
            const double fnew = f[q] + c.dt * (rhs[q] - adv);
            if (!live) continue;
            double *po = fout + plane;
            po[cell] = fnew;
            if (mx | my) store_images(po, (int)x, (int)y, c.nx, c.ny, c.pitch, mx, my, fnew);
        }
    };
#pragma unroll 1
    for (int s = warp >> 2; s < S; s += SW) {
        if (r & 1)
            ring_step(std::true_type{}, s);
        else
            ring_step(std::false_type{}, s);
    }
}

template <int S>
static int launch_f64_wide(dbm_handle *h, const F64Consts<S> &c, int sets, const double *fin, double *fout,
                           cudaStream_t st)
{
    constexpr int CELLS = 32;
    const size_t smem = f64_smem<S>(CELLS, sets);
    if (smem > 48 * 1024) {
        static std::atomic<unsigned long long> allowed{0};
        const cudaError_t e = allow_smem(k_step_f64<S>, f64_smem<S>(CELLS, 4), allowed);
        if (e != cudaSuccess) return set_cuda_error(h, e, "FP64 step kernel shared-memory attribute");
    }
    const long long cells = (long long)h->p.nx * h->p.ny;
    return set_cuda_error(h, launch_chained(k_step_f64<S>, dim3((unsigned)((cells + CELLS - 1) / CELLS)),
                                            dim3(128 * f64_side(S)), smem, st, c, ChainedIn<double>(fin), fout,
                                            (unsigned *)h->scratch),
                          "FP64 step kernel launch");
}

// ---------------------------------------------------------------------------
// The FP64 step of a small grid: 4 cells per CTA.
//
// Four phase warps run phases 1 to 4, each split so that no warp has more
// than about 20 FP64 instructions in a row: the products of the moment sums
// by value and the sums by moment, one quantity of a species per warp, f-hat
// in four parts.  Meanwhile the ring warps (a ring each; 16 lanes, 4 cells by 4
// velocities, per species, two species a warp) form the advection terms, which
// need no moments, and after the last phase the equilibrium and the update.
// One CTA's chain is then about 11 000 cycles where one thread per item of
// each phase and 8 cells took 38 000 (two species, us a step: 400 x 1
// 17.7 -> 9.8; three reacting 31 -> 18).
// ---------------------------------------------------------------------------

constexpr int SMALL_CELLS = 4;
__host__ __device__ constexpr int small_ring_warps(int S) { return 4 * ((S + 1) / 2); }

template <int S>
__global__ void __launch_bounds__(128 + 32 * small_ring_warps(S))
    k_step_f64_small(const __grid_constant__ F64Consts<S> c, const ChainedIn<double> in,
                     double *__restrict__ fout, unsigned *__restrict__ flag)
{
    constexpr int C = SMALL_CELLS, PHASE = 128;
    __shared__ double val[S][3][Q][C];     // f, f v (the ring's speed), f q
    __shared__ double mom[S][4][C];        // n, j_x, j_y, E
    __shared__ double wts[S][W_N][C];
    __shared__ double mix[M_COUNT][C];
    __shared__ double den[C], term[S][C];
    __shared__ double fhs[4][S][Q][C];
    const long long P = c.plane;
    const unsigned d0 = blockIdx.x * (unsigned)C, total = (unsigned)c.nx * (unsigned)c.ny;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const bool react = c.has_reaction != 0, force = c.has_force != 0;
    auto locate = [&](int j, unsigned &x, unsigned &y) {
        const unsigned d = min(d0 + (unsigned)j, total - 1u);
        y = d / (unsigned)c.nx;
        x = d - y * (unsigned)c.nx;
        return (long long)(y + GY) * c.pitch + (x + GX);
    };
    const double *fin = in.wait();

    if (tid < PHASE) {
        auto phase_sync = [] { asm volatile("barrier.sync 1, 128;" ::: "memory"); };
        // 1. values and their products, one per thread; then the sums
#pragma unroll 1
        for (int it = tid; it < S * Q * C; it += PHASE) {
            const int j = it & 3, i = (it >> 2) & 15, s = it >> 6;
            unsigned x, y;
            const double f = fin[(long long)(s * Q + i) * P + locate(j, x, y)];
            val[s][0][i][j] = f;
            val[s][1][i][j] = f * c.vr[s][i >> 2];
            val[s][2][i][j] = f * c.qr[s][i >> 2];
        }
        phase_sync();
        {  // warp q and its upper half take species q and q + 4; lane: cell and moment
            const int j = lane & 3, k = (lane >> 2) & 3, s = warp + 4 * (lane >> 4);
            if (s < S) {
                double sum = 0.0;
#pragma unroll
                for (int i = 0; i < Q; ++i) {
                    const double f = val[s][k == 0 ? 0 : k == 3 ? 2 : 1][i][j];
                    const int d = k == 1 ? dir_x(i) : k == 2 ? dir_y(i) : 1;
                    sum = sum + (d < 0 ? -f : d == 0 ? 0.0 : f);
                }
                mom[s][k][j] = sum;
            }
        }
        phase_sync();
        // 2. one quantity per warp; lane: cell and species
        const int j = lane & 3, s = lane >> 2;
        const bool mine = s < S;
        const int q = mine ? s : 0;  // species constants of an idle lane
        if (mine) {
            const double sn = mom[s][0][j];
            const double rho = c.md[q].b * sn;
            if (warp == 0) {
                const double ux = sn != 0.0 ? mom[s][1][j] / sn : 0.0;  // an absent species: zero velocity
                wts[s][W_UX][j] = ux;
                wts[s][W_LX][j] = div_by(rho * ux, c.taud[q]);
            } else if (warp == 1) {
                const double uy = sn != 0.0 ? mom[s][2][j] / sn : 0.0;
                wts[s][W_UY][j] = uy;
                wts[s][W_LY][j] = div_by(rho * uy, c.taud[q]);
            } else if (warp == 2) {
                wts[s][W_RHO][j] = rho;
                wts[s][W_LAM][j] = div_by(rho, c.taud[q]);
                wts[s][W_ME][j] = c.md[q].b * mom[s][3][j];
            } else {
                wts[s][W_CAP][j] = div_by(sn * (2.0 + c.I[q]), c.taud[q]);
            }
        }
        phase_sync();
        // 3. mixture u, the denominator of T
        if (lane < C) {
            if (warp <= 1) {
                double sw = 0.0, sx = 0.0;
#pragma unroll
                for (int k = 0; k < S; ++k) {
                    sw += wts[k][W_LAM][lane];
                    sx += wts[k][warp == 0 ? W_LX : W_LY][lane];
                }
                mix[M_UX + warp][lane] = sx / sw;
            } else if (warp == 2) {
                double d = 0.0, ntot = 0.0;
#pragma unroll
                for (int k = 0; k < S; ++k) {
                    d += wts[k][W_CAP][lane];
                    ntot += fabs(mom[k][0][lane]);
                }
                den[lane] = d;
                mix[M_NTOT][lane] = ntot;
            }
        }
        if (force && warp == 3 && mine) {
            const double sn = mom[s][0][j];
            double Ts = 0.0;
            if (sn != 0.0) {
                const double ux = wts[s][W_UX][j], uy = wts[s][W_UY][j];
                Ts = c.md[q].b * (mom[s][3][j] / sn - (ux * ux + uy * uy)) / (2.0 + c.I[q]);
            }
            wts[s][W_TS][j] = Ts;
        }
        phase_sync();
        if (warp == 0) {
            if (mine) {
                const double Ux = mix[M_UX][j], Uy = mix[M_UY][j];
                const double u2 = Ux * Ux + Uy * Uy;
                term[s][j] = div_by(wts[s][W_ME][j] - wts[s][W_RHO][j] * u2, c.taud[q]);
            }
            __syncwarp();
            if (lane < C) {
                const double Ux = mix[M_UX][lane], Uy = mix[M_UY][lane], ntot = mix[M_NTOT][lane];
                double num = 0.0;
#pragma unroll
                for (int k = 0; k < S; ++k) num += term[k][lane];
                const double T = num / den[lane];
                unsigned bad = 0;
#pragma unroll
                for (int k = 0; k < S; ++k) {
                    const double n = mom[k][0][lane];
                    if (!(n >= -1e-6 * ntot) || !isfinite(n)) bad |= DBM_HEALTH_DENSITY;
                }
                if (!(ntot > 0.0)) bad |= DBM_HEALTH_DENSITY;
                if (!(T > 0.0)) bad |= DBM_HEALTH_TEMPERATURE;
                if (!isfinite(T) || !isfinite(Ux) || !isfinite(Uy)) bad |= DBM_HEALTH_NONFINITE;
                double omega = 0.0, dTdt = 0.0;
                if (react) {
                    omega = c.k_ov * mom[c.fuel][0][lane] * mom[c.oxid][0][lane] * exp(-c.Ea_over_R / T);
                    double src = 0.0, cap = 0.0;
#pragma unroll
                    for (int k = 0; k < S; ++k) {
                        src += (2.0 + c.I[k]) * c.a[k] * omega;
                        cap += mom[k][0][lane] * (2.0 + c.I[k]);
                    }
                    dTdt = (c.Qheat * omega - 0.5 * T * src) / (0.5 * cap);
                }
                mix[M_T][lane] = T;
                mix[M_OMEGA][lane] = omega;
                mix[M_DT][lane] = dTdt;
                if (bad) raise_flag(flag, bad);
            }
        }
        phase_sync();
        // 4. f-hat: a part per warp; lane: cell and species
        if (mine) {
            const double n = mom[s][0][j], Ux = mix[M_UX][j], Uy = mix[M_UY][j], T = mix[M_T][j];
            const double tau = c.taud[q].b;
            auto part = [&](int set, double n_, double ux, double uy, double t) {
                double *fh = &fhs[set][s][0][j];
                if (warp == 0)
                    fhat_printed<0>(n_, ux, uy, t, c.md[q], c.I[q], fh, C);
                else if (warp == 1)
                    fhat_printed<1>(n_, ux, uy, t, c.md[q], c.I[q], fh, C);
                else if (warp == 2)
                    fhat_printed<2>(n_, ux, uy, t, c.md[q], c.I[q], fh, C);
                else
                    fhat_printed<3>(n_, ux, uy, t, c.md[q], c.I[q], fh, C);
            };
            part(0, n, Ux, Uy, T);
            if (react) {
                const double nstar = n + tau * c.a[q] * mix[M_OMEGA][j];
                if (warp == 0 && nstar < -1e-6 * mix[M_NTOT][j]) raise_flag(flag, DBM_HEALTH_NSTAR);
                part(1, nstar, Ux, Uy, T + tau * mix[M_DT][j]);
            }
            if (force) {
                const double ux = wts[s][W_UX][j], uy = wts[s][W_UY][j], Ts = wts[s][W_TS][j];
                part(2, n, ux + c.ax * tau, uy + c.ay * tau, Ts);
                part(3, n, ux, uy, Ts);
            }
        }
        __syncthreads();
        chain_end();
        return;
    }

    // 5. a ring per warp, a velocity of a cell and species per lane
    const int r = warp & 3, j = lane & 3, i = (lane >> 2) & 3;
    const int s = 2 * ((warp - 4) >> 2) + (lane >> 4);
    const bool mine = s < S;
    const int q = mine ? s : 0;
    unsigned x, y;
    const long long cell = locate(j, x, y);
    const long long plane = (long long)(q * Q + 4 * r + i) * P;
    const double *pl = fin + plane + cell;
    const double f = pl[0], v = c.vr[q][r];
    double adv;
    {
        const double g0 = v * f;
        if (r & 1) {
            const int ex = (i == 1 || i == 2) ? -1 : 1, ey = (i == 2 || i == 3) ? -c.pitch : c.pitch;
            adv = nnd_dflux(pl[-2 * ex], pl[-ex], pl[ex], g0, v, c.dxd);
            adv += nnd_dflux(pl[-2 * ey], pl[-ey], pl[ey], g0, v, c.dyd);
        } else {
            const int st = (i & 1) ? c.pitch : 1, e = (i & 2) ? -st : st;
            const ConstDiv h = (i & 1) ? c.dyd : c.dxd;
            adv = nnd_dflux(pl[-2 * e], pl[-e], pl[e], g0, v, h);
        }
    }
    __syncthreads();
    chain_end();
    auto equilibrium = [&](int set) {
        double e[1];
        if (r & 1)
            ring_equilibrium<true, 1, C>(c.row[q][r], &fhs[set][q][0][j], i, e);
        else
            ring_equilibrium<false, 1, C>(c.row[q][r], &fhs[set][q][0][j], i, e);
        return e[0];
    };
    const ConstDiv tau = c.taud[q];
    const double feq = equilibrium(0);
    double rhs = div_by(-(f - feq), tau);                                 // Omega
    if (react) rhs = rhs + div_by(equilibrium(1) - feq, tau);             // R
    if (force) {
        const double g1 = equilibrium(2), g0 = equilibrium(3);
        rhs = rhs + div_by(g1 - g0, tau);                                 // G
    }
    const double fnew = f + c.dt * (rhs - adv);
    if (!mine || d0 + (unsigned)j >= total) return;
    double *po = fout + plane;
    po[cell] = fnew;
    const unsigned mx = ghost_mask((int)x, c.nx, c.bc_x), my = ghost_mask((int)y, c.ny, c.bc_y);
    if (mx | my) store_images(po, (int)x, (int)y, c.nx, c.ny, c.pitch, mx, my, fnew);
}

// Grids of up to four 4-cell CTAs per SM take the 4-cell kernel (us a step on 152
// SMs, 4 cells / 32 cells: two species 2048 cells 20.2 / 25.7, 3000 cells 27.6 /
// 25.8; four under a force 63 / 71, 76 / 71; either side of the line, 2432 and
// 2433 cells: one species 18.8 / 19.8, two 20.2 / 26.1, eight under a force 122 /
// 136).
constexpr int SMALL_CELLS_PER_SM = 4 * SMALL_CELLS;

bool f64_small_grid(const dbm_handle *h) { return (long long)h->p.nx * h->p.ny <= (long long)SMALL_CELLS_PER_SM * h->sms; }

template <int S>
static int launch_f64_t(dbm_handle *h, const double *fin, double *fout, cudaStream_t st)
{
    F64Consts<S> c;
    fill_f64_consts<S>(h, c);
    const long long cells = (long long)h->p.nx * h->p.ny;
    if (!f64_small_grid(h))
        return launch_f64_wide<S>(h, c, 1 + (c.has_reaction ? 1 : 0) + (c.has_force ? 2 : 0), fin, fout, st);
    static std::atomic<unsigned long long> allowed{0};
    const cudaError_t e = allow_smem(k_step_f64_small<S>, ALONE_SMEM, allowed);
    if (e != cudaSuccess) return set_cuda_error(h, e, "FP64 small-grid step kernel shared-memory attribute");
    const long long ctas = (cells + SMALL_CELLS - 1) / SMALL_CELLS;
    return set_cuda_error(h, launch_chained(k_step_f64_small<S>, dim3((unsigned)ctas),
                                            dim3(128 + 32 * small_ring_warps(S)), ctas <= h->sms ? ALONE_SMEM : 0, st, c,
                                            ChainedIn<double>(fin), fout, (unsigned *)h->scratch),
                          "FP64 small-grid step kernel launch");
}

int launch_step_f64(dbm_handle *h, int cur, cudaStream_t st)
{
    const double *fin = (const double *)h->f[cur];
    double *fout = (double *)h->f[cur ^ 1];
    switch (h->p.nspecies) {
    case 1: return launch_f64_t<1>(h, fin, fout, st);
    case 2: return launch_f64_t<2>(h, fin, fout, st);
    case 3: return launch_f64_t<3>(h, fin, fout, st);
    case 4: return launch_f64_t<4>(h, fin, fout, st);
    case 5: return launch_f64_t<5>(h, fin, fout, st);
    case 6: return launch_f64_t<6>(h, fin, fout, st);
    case 7: return launch_f64_t<7>(h, fin, fout, st);
    case 8: return launch_f64_t<8>(h, fin, fout, st);
    }
    return DBM_ERR_INVALID;
}

}  // namespace dbm

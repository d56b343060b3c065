// Explicit right-hand side in FP64 (arXiv 2105.01865, Sec. 3 and Eq. eq-re):
// the terms of ch_explicit_rhs, arranged for a GPU whose FP64 rate is 1/64 of
// its FP32 rate, so that the kernel is bound by the FP64 operations of a cell
// and little else counts.  Everything that neighbouring cells or faces form
// alike is formed once and passed on, through shared memory in x and y and
// through a register queue in z:
//   d_j = C_{j+1} - C_j, the first differences of a line;
//   Q_j = 4 eps + (13/3) (d_j - d_{j-1})^2, the curvature part of the WENO5
//         smoothness indicators of the three faces that use cell j;
//   psi'(C), once a cell instead of seven times.
// A face then needs 29 operations (49 when it formed all of this itself), and
// the fourth difference of a line is (d_{i+1} - d_{i-2}) - 3 (d_i - d_{i-1}).
// The upwind side costs none: with g the differences of the upwind stencil in
// upwind order, the face value is C_up + F(g) for a positive and C_up - F(g)
// for a negative velocity, F the same function, so the sign only turns the
// direction in which the shared line is read.
//
// 256 x 256 x 128 shear drop, with advection: 3641 us a launch when
// it shared the paired FP32 design, 2586 so, about 160 FP64 operations a
// cell at 85 % of the FP64 pipe.  64^3 without: 91 and 35 us.
#pragma once

#include "ch_kernels.cuh"

namespace chg {

// a / b to within a unit in the last place: the hardware's reciprocal estimate
// (2^-20), one Newton step (2^-40) and one correction of the quotient by its
// residual (Markstein's scheme).  Outside 2^-800 .. 2^1000, where b, its
// reciprocal or the residual may be subnormal (the estimate takes a subnormal for
// zero), the division.
__device__ __forceinline__ double div_newton(double a, double b) {
    if ((unsigned)__double2hiint(b) - 0x0df00000u > 0x7e700000u - 0x0df00000u) return a / b;
    double y;
    asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(b));
    y = fma(y, fma(-b, y, 1.0), y);
    const double q = a * y;
    return fma(fma(-b, q, a), y, q);
}

// F(g) of a face and the curvature parts q0, q1, q2 of its three candidates
// (upwind to downwind): with s_k = q_k + E_k^2 = 4 (eps + beta_k) and t_k = s_k^2,
// weights w0 = t1 t2, w1 = 2 h1 = 6 t0 t2, w2 = 3 t0 t1 and candidates
// value - C_up = (5 g2 - 2 g1) / 6, (g2 + 2 g3) / 6, (4 g3 - g4) / 6, the middle
// one doubled to go with h1.
__device__ __forceinline__ double weno5_g(double g1, double g2, double g3, double g4, double q0, double q1, double q2) {
    const double E0 = fma(3.0, g2, -g1), E1 = g2 + g3, E2 = fma(-3.0, g3, g4);
    const double s0 = fma(E0, E0, q0), s1 = fma(E1, E1, q1), s2 = fma(E2, E2, q2);
    const double t0 = s0 * s0, t1 = s1 * s1, t2 = s2 * s2;
    const double t03 = 3.0 * t0, w0 = t1 * t2, h1 = t03 * t2, w2 = t03 * t1;
    const double a = (2.0 / 3.0) * g3;
    const double p0 = fma(5.0 / 6.0, g2, (-1.0 / 3.0) * g1), p1 = fma(1.0 / 3.0, g2, a), p2 = fma(-1.0 / 6.0, g4, a);
    const double num = fma(w2, p2, fma(h1, p1, w0 * p0));
    return div_newton(num, fma(2.0, h1, w0 + w2));
}
// vel (C_up + F) or vel (C_up - F): the sign goes with that of vel
__device__ __forceinline__ bool upwind(double vel) { return __double2hiint(vel) >= 0; }
__device__ __forceinline__ double face_flux_g(double vel, double c_up, double F) {
    return fma(fabs(vel), F, vel * c_up);
}

constexpr int kEX = 32;  // tile in x (one warp)

// TY rows a tile, one cell a thread.  Needs no alignment and takes any nx.
template <bool ADV, bool DIRI, int TY, int MINB>
__global__ void __launch_bounds__(kEX * TY, MINB)
ch_explicit_f64(const double* __restrict__ C, const double* __restrict__ u, const double* __restrict__ v,
                const double* __restrict__ w, const double* __restrict__ Hprev, double* __restrict__ Hout,
                double* __restrict__ r, RhsArgs<double> a, int zchunk) {
    pdl_wait();
    pdl_launch_dependents();
    constexpr int NT = kEX * TY, PX = kEX + 6, PY = TY + 6;
    __shared__ double Cs[2][PY][PX];                 // cells i0-3 .., j0-3 ..
    __shared__ double xd[TY][PX];                    // d of cell i0-3+c
    __shared__ double yd[TY + 5][kEX];               // d of row j0-3+r
    __shared__ double xQ[ADV ? TY : 1][PX], yQ[ADV ? TY + 5 : 1][kEX];
    __shared__ double Ps[TY + 2][kEX + 2];           // psi' of cells i0-1 .., j0-1 ..
    __shared__ double Fx[ADV ? TY : 1][kEX + 1], Fy[ADV ? TY + 1 : 1][kEX];
    __shared__ int gi_tab[PX], gj_tab[PY];
    const int tx = threadIdx.x, ty = threadIdx.y, tid = ty * kEX + tx;
    const int i0 = blockIdx.x * kEX, j0 = blockIdx.y * TY, k0 = blockIdx.z * zchunk;
    const int i = i0 + tx, j = j0 + ty, kend = min(k0 + zchunk, a.nz);
    const bool in_xy = i < a.nx && j < a.ny;
    const int ic = min(i, a.nx - 1), jc = min(j, a.ny - 1);
    const int64_t plane = (int64_t)a.nx * a.ny, col = (int64_t)jc * a.nx + ic;
    const double eps4 = 4.0 * a.eps;

    for (int e = tid; e < PX + PY; e += NT) {
        if (e < PX) gi_tab[e] = bc_index(i0 + e - 3, a.nx, a.bcx);
        else gj_tab[e - PX] = bc_index(j0 + (e - PX) - 3, a.ny, a.bcy);
    }
    // faces of this thread (lower x and y) and the tile's extra upper ones: the
    // y-face j0 + TY by warp 0, the x-face i0 + 32 by the first TY lanes of warp 1
    const bool wall_x = a.bcx == CH_NOFLUX && (i <= 0 || i >= a.nx);
    const int fi = a.bcx == CH_PERIODIC ? bc_index(i, a.nx, CH_PERIODIC) : min(i, a.nx);
    const bool wall_y = a.bcy == CH_NOFLUX && (j <= 0 || j >= a.ny);
    const int fj = a.bcy == CH_PERIODIC ? bc_index(j, a.ny, CH_PERIODIC) : min(j, a.ny);
    const int ie = i0 + kEX, je = j0 + TY, jex = min(j0 + tx, a.ny - 1);
    const bool wall_xe = a.bcx == CH_NOFLUX && ie >= a.nx, wall_ye = a.bcy == CH_NOFLUX && je >= a.ny;
    const int fie = a.bcx == CH_PERIODIC ? bc_index(ie, a.nx, CH_PERIODIC) : min(ie, a.nx);
    const int fje = a.bcy == CH_PERIODIC ? bc_index(je, a.ny, CH_PERIODIC) : min(je, a.ny);
    const bool xtra_y = ADV && ty == 0 && !wall_ye, xtra_x = ADV && ty == 1 && tx < TY && !wall_xe;

    auto zval = [&](int k) {
        const double c = C[bc_near(k, a.nz, a.bcz) * plane + col];
        return DIRI && bc_negate(k, a.nz, a.bcz) ? -c : c;
    };
    auto psi = [](double c) { return c * fma(c, c - 1.5, 0.5); };
    auto curv = [&](double dm, double dp) {
        const double D = dp - dm;
        return fma((13.0 / 3.0) * D, D, eps4);
    };
    auto flux = [](double vel, double cm, double cp, double dm2, double dm1, double d0, double dp1, double dp2,
                   double qm1, double q0, double q1, double q2) {  // d and q about the face, lower cell's d is d0
        const bool up = upwind(vel);
        const double F = weno5_g(up ? dm2 : dp2, up ? dm1 : dp1, d0, up ? dp1 : dm1, up ? qm1 : q2, up ? q0 : q1,
                                 up ? q1 : q0);
        return face_flux_g(vel, up ? cm : cp, F);
    };
    // the z-line: cz[m] = C(k + m), dz[m] = d(k - 2 + m), qz[m] = Q(k - 1 + m)
    double cz[5], dz[5], qz[4], psm, ps0;
    double fz_lo = 0.0;
    {
        double c[8];  // C(k0 - 3 .. k0 + 4)
#pragma unroll
        for (int m = 0; m < 8; ++m) c[m] = zval(k0 - 3 + m);
#pragma unroll
        for (int m = 0; m < 5; ++m) cz[m] = c[3 + m];
#pragma unroll
        for (int m = 0; m < 5; ++m) dz[m] = c[m + 2] - c[m + 1];
        if (ADV) {
#pragma unroll
            for (int m = 0; m < 4; ++m) qz[m] = curv(dz[m], dz[m + 1]);
            if (!(a.bcz != CH_PERIODIC && k0 == 0)) {
                const double dl = c[1] - c[0];  // d(k0 - 3)
                fz_lo = flux(w[k0 * plane + col], c[2], c[3], dl, dz[0], dz[1], dz[2], dz[3], curv(dl, dz[0]), qz[0],
                             qz[1], qz[2]);
            }
        }
        psm = psi(c[2]);
        if (DIRI && k0 == 0) psm = -psi(c[3]);  // psi' = 0 on the wall: its ghost is its own negated mirror
        ps0 = psi(c[3]);
    }
    __syncthreads();  // index tables ready

    auto stage = [&](int kk) {
        const double* Ck = C + kk * plane;
        double* dst = &Cs[(kk - k0) & 1][0][0];
        for (int e = tid; e < PX * PY; e += NT) {
            const int row = e / PX, cc = e - row * PX;
            cp_async_elem(dst + e, Ck + (int64_t)gj_tab[row] * a.nx + gi_tab[cc]);
        }
        cp_async_commit();
    };
    stage(k0);
    for (int k = k0; k < kend; ++k) {
        if (k + 1 < kend) stage(k + 1);
        // this plane's inputs, waited for after the shared lines are formed
        const double cn = zval(k + 5);
        double uv = 0.0, vv = 0.0, wv = 0.0, ve = 0.0, hp = 0.0;
        const bool zwall = a.bcz != CH_PERIODIC && k + 1 >= a.nz;
        if (ADV) {
            if (!wall_x) uv = u[((int64_t)k * a.ny + jc) * a.nfx + fi];
            if (!wall_y) vv = v[((int64_t)k * a.nfy + fj) * a.nx + ic];
            if (!zwall) wv = w[(k + 1 < a.nz ? k + 1 : 0) * plane + col];
            if (xtra_y) ve = v[((int64_t)k * a.nfy + fje) * a.nx + ic];
            if (xtra_x) ve = u[((int64_t)k * a.ny + jex) * a.nfx + fie];
        }
        if (a.has_prev && in_xy) hp = Hprev[k * plane + col];
        if (k + 1 < kend) cp_async_wait<1>();
        else cp_async_wait<0>();
        __syncthreads();
        const double(*P)[PX] = Cs[(k - k0) & 1];
        // ---- the lines of the plane
        for (int e = tid; e < TY * (PX - 1); e += NT) {
            const int row = e / (PX - 1), c = e - row * (PX - 1);
            const double* p = &P[row + 3][c];
            const double d = p[1] - p[0];
            xd[row][c] = d;
            if (ADV && c > 0) xQ[row][c] = curv(p[0] - p[-1], d);
        }
        for (int row = ty; row < TY + 5; row += TY) {
            const double d = P[row + 1][tx + 3] - P[row][tx + 3];
            yd[row][tx] = d;
            if (ADV && row > 0) yQ[row][tx] = curv(P[row][tx + 3] - P[row - 1][tx + 3], d);
        }
        Ps[ty + 1][tx + 1] = ps0;
        if (ty < 2) Ps[ty * (TY + 1)][tx + 1] = psi(P[ty == 0 ? 2 : TY + 3][tx + 3]);
        else if (ty == 2 && tx < TY) Ps[tx + 1][0] = psi(P[tx + 3][2]);
        else if (ty == 3 && tx < TY) Ps[tx + 1][kEX + 1] = psi(P[tx + 3][kEX + 3]);
        // the cells past a ragged edge have no psi of their own in ps0
        if (!in_xy) Ps[ty + 1][tx + 1] = psi(P[ty + 3][tx + 3]);
        __syncthreads();
        // ---- face fluxes
        double fz_up = 0.0;
        if (ADV) {
            auto line_flux = [&](double vel, double cm, double cp, const double* d, const double* q, int st) {
                // d, q at the cell three below the face; st: stride along the line
                const bool up = upwind(vel);
                const int s = up ? st : -st;
                const double* g = up ? d : d + 4 * st;
                const double* h = up ? q + st : q + 4 * st;
                const double F = weno5_g(g[0], g[s], g[2 * s], g[3 * s], h[0], h[s], h[2 * s]);
                return face_flux_g(vel, up ? cm : cp, F);
            };
            Fx[ty][tx] = wall_x ? 0.0 : line_flux(uv, P[ty + 3][tx + 2], P[ty + 3][tx + 3], &xd[ty][tx], &xQ[ty][tx], 1);
            Fy[ty][tx] = wall_y ? 0.0
                                : line_flux(vv, P[ty + 2][tx + 3], P[ty + 3][tx + 3], &yd[ty][tx], &yQ[ty][tx], kEX);
            if (ty == 0)
                Fy[TY][tx] = xtra_y ? line_flux(ve, P[TY + 2][tx + 3], P[TY + 3][tx + 3], &yd[TY][tx], &yQ[TY][tx], kEX)
                                    : 0.0;
            if (ty == 1 && tx < TY)
                Fx[tx][kEX] = xtra_x ? line_flux(ve, P[tx + 3][kEX + 2], P[tx + 3][kEX + 3], &xd[tx][kEX], &xQ[tx][kEX], 1)
                                     : 0.0;
            if (!zwall) fz_up = flux(wv, cz[0], cz[1], dz[0], dz[1], dz[2], dz[3], dz[4], qz[0], qz[1], qz[2], qz[3]);
        }
        // ---- M lap(psi') and A_d C, from the shared lines
        double psp = psi(cz[1]);
        const double ps_next = psp;  // psi'(C) of the next plane
        if (DIRI && k + 1 == a.nz) psp = -psi(-cz[1]);
        const double pc = Ps[ty + 1][tx + 1];
        const double lap = (((Ps[ty + 1][tx] - pc) + (Ps[ty + 1][tx + 2] - pc)) +
                            ((Ps[ty][tx + 1] - pc) + (Ps[ty + 2][tx + 1] - pc)) + ((psm - pc) + (psp - pc))) *
                           a.inv_h2;
        auto fourth = [](double dm2, double dm1, double d0, double d1) { return fma(-3.0, d0 - dm1, d1 - dm2); };
        const double astar = (fourth(xd[ty][tx + 1], xd[ty][tx + 2], xd[ty][tx + 3], xd[ty][tx + 4]) +
                              fourth(yd[ty + 1][tx], yd[ty + 2][tx], yd[ty + 3][tx], yd[ty + 4][tx])) +
                             fourth(dz[0], dz[1], dz[2], dz[3]);
        double H = a.mob * lap;
        if (ADV) {
            __syncthreads();
            const double div = (Fx[ty][tx + 1] - Fx[ty][tx]) + (Fy[ty + 1][tx] - Fy[ty][tx]) + (fz_up - fz_lo);
            H = fma(-a.inv_h, div, H);
        } else {
            __syncthreads();  // the lines are formed anew next
        }
        if (in_xy) {
            double rhs = fma(-a.impl, astar, a.dtg * H);
            if (a.has_prev) rhs = fma(a.dtr, hp, rhs);
            Hout[k * plane + col] = H;
            if (r) r[k * plane + col] = rhs;
        }
        // ---- one plane up
        psm = ps0;
        ps0 = ps_next;
        const double dn = cz[4] - cz[3];  // d(k + 3)
#pragma unroll
        for (int m = 0; m < 4; ++m) {
            cz[m] = cz[m + 1];
            dz[m] = dz[m + 1];
        }
        cz[4] = cn;
        dz[4] = dn;
        if (ADV) {
            qz[0] = qz[1];
            qz[1] = qz[2];
            qz[2] = qz[3];
            qz[3] = curv(dz[3], dz[4]);
        }
        fz_lo = fz_up;
    }
}

}  // namespace chg

// Explicit right-hand side in FP32 (arXiv 2105.01865, Sec. 3 and Eq. eq-re):
// H^l = -div(uC)_WENO5 + M lap(psi'(C)), r = dt(gamma H^l + rho H^{l-1})
// - alpha dt M sum_d A_d C.  A thread owns the x-adjacent cells (ia, ia + 1) of
// its row and marches z; every value is a pair, so one paired instruction
// (FADD2, FMUL2, FFMA2) serves both cells.  A CTA's tile is 64 x 8 cells.
//
// What bounds it: instruction issue, then the FMA pipe.  The paired arithmetic
// of the formulas is about 180 instructions a pair and plane; what counts is
// how many others come with it (about 450 instructions in all; 602 in the form
// this replaces, at 5.36 against 4.60 ms a launch on 1024 x 1024 x 512, 1.43
// against 1.13 ms on 500^3 and, one cell a thread for odd nx, 81 against 57 us
// on 211 x 157 x 93).  So
//  - a plane's inputs arrive by asynchronous copies into shared memory, C as
//    one 16-byte copy a thread, the face velocities and H^{l-1} as one 8-byte
//    copy each into the thread's own slots, whose sources advance by one
//    addition a plane.  A wall face's copy has length 0 and fills with zeros,
//    so its flux vanishes without a test;
//  - a thread's x-window is four 8-byte shared loads; its upper x-face comes
//    from the next lane by a shuffle; its lower faces stay in registers;
//  - psi' is formed once a plane for the cell's own column and carried;
//  - the WENO5 quotient is one reciprocal estimate;
//  - warps 0 and 1 also form the tile's extra faces, and the others need not wait
//    for them at once: a warp arrives at a split barrier once its own x- and
//    y-faces are published and waits after its z-faces, Laplacian and fourth
//    differences (4.85 ms with one barrier in that place, 4.60 so).
// 3 CTAs an SM at 80 registers (2 at 117: 4.91 ms); odd rows, which hold
// more offsets, 2 at 120 (55 against 61 us on 211 x 157 x 93).
// XM says how rows lie: kRowsPeriodic, 16-byte aligned (nx a multiple of 4) and
// periodic, so that a halo chunk is a chunk of the row's other end; kRowsWalled,
// aligned with walls; kRowsEven, nx even: pairs of cells are 8-byte aligned, whole
// and never wrap, so everything but u moves in pairs (198 x 200 x 150: 93 us, 117 as
// kRowsAny; 514 x 130 x 66: 68 and 86); kRowsAny, odd rows: copies, loads and stores go
// element by element.
#pragma once

#include "ch_pairs.cuh"

namespace chg {

// cp.async of N floats, of which the first `bytes` are read and the rest zero
template <int N>
__device__ __forceinline__ void cp_async_fill(float* smem, const float* gmem, int bytes) {
    const unsigned sa = (unsigned)__cvta_generic_to_shared(smem);
    asm volatile("cp.async.ca.shared.global [%0], [%1], %2, %3;\n" ::"r"(sa), "l"(gmem), "n"(N * 4), "r"(bytes) : "memory");
}

// Split barrier of a CTA's warps on a shared-memory mbarrier: a warp arrives
// once its shared writes are done, works on, and waits later.  The wait gives up
// after 2 s (false).
__device__ __forceinline__ void warps_init(unsigned long long* bar, unsigned warps) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;\n" ::"r"((unsigned)__cvta_generic_to_shared(bar)), "r"(warps)
                 : "memory");
}
__device__ __forceinline__ void warps_arrive(unsigned long long* bar, int lane) {
    __syncwarp();
    if (lane == 0)
        asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];\n" ::"r"((unsigned)__cvta_generic_to_shared(bar)) : "memory");
}
__device__ __forceinline__ bool warps_try(unsigned long long* bar, unsigned parity) {
    unsigned ok;
    asm volatile("{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}\n"
                 : "=r"(ok)
                 : "r"((unsigned)__cvta_generic_to_shared(bar)), "r"(parity)
                 : "memory");
    return ok != 0;
}
__device__ __forceinline__ bool warps_wait(unsigned long long* bar, unsigned parity) {
    if (warps_try(bar, parity)) return true;
    unsigned long long t0, t;
    asm volatile("mov.u64 %0, %%globaltimer;\n" : "=l"(t0));
    while (!warps_try(bar, parity)) {
        asm volatile("mov.u64 %0, %%globaltimer;\n" : "=l"(t));
        if (t - t0 > 2000000000ull) return false;
    }
    return true;
}

// WENO5 (Jiang-Shu) face values of two faces at once in first differences of
// the stencil (a' = v1 - v2, b = v3 - v2, c = v4 - v3, d = v5 - v4): with
//   4 beta_k = (13/3) D_k^2 + E_k^2, D = (b + a', c - b, d - c), E = (2b + D0, b + c, D2 - 2c),
//   t_k = (4 eps + 4 beta_k)^2, weights (t1 t2 / 3, 2 t0 t2, t0 t1) and
//   candidates v3 + (5b + 2a', b + 2c, 4c - d) / 6, the middle one doubled
// the value is v3 plus a quotient of weighted sums.  eps4 is 4 eps.  The
// denominator is kept normal: the estimate takes a subnormal for 0.
__device__ __forceinline__ Pr<float> weno5q(Pr<float> v1, Pr<float> v2, Pr<float> v3, Pr<float> v4, Pr<float> v5,
                                            Pr<float> eps4) {
    const Pr<float> am = sub(v1, v2), b = sub(v3, v2), c = sub(v4, v3), d = sub(v5, v4);
    const Pr<float> D0 = add(b, am), D1 = sub(c, b), D2 = sub(d, c);
    const Pr<float> E0 = fma2(sp(2.f), b, D0), E1 = add(b, c), E2 = fma2(sp(-2.f), c, D2);
    const Pr<float> c133 = sp(13.f / 3.f), third = sp(1.f / 3.f);
    const Pr<float> s0 = fma2(mul(c133, D0), D0, fma2(E0, E0, eps4));
    const Pr<float> s1 = fma2(mul(c133, D1), D1, fma2(E1, E1, eps4));
    const Pr<float> s2 = fma2(mul(c133, D2), D2, fma2(E2, E2, eps4));
    const Pr<float> t0 = mul(s0, s0), t1 = mul(s1, s1), t2 = mul(s2, s2);
    const Pr<float> w0 = mul(mul(third, t1), t2), h1 = mul(t0, t2), w2 = mul(t0, t1);
    const Pr<float> c23 = mul(sp(2.f / 3.f), c);
    const Pr<float> p0 = fma2(sp(5.f / 6.f), b, mul(third, am)), p1 = fma2(third, b, c23), p2 = fma2(sp(-1.f / 6.f), d, c23);
    const Pr<float> num = fma2(w2, p2, fma2(h1, p1, mul(w0, p0)));
    const Pr<float> den = fma2(sp(2.f), h1, add(w0, w2));
    float rx, ry;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(rx) : "f"(fmaxf(den.x(), 1.17549435e-38f)));
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(ry) : "f"(fmaxf(den.y(), 1.17549435e-38f)));
    return fma2(num, mk(rx, ry), v3);
}

// Flux pair through two faces; m3..p2 are the cell pairs f-3 .. f+2.
__device__ __forceinline__ Pr<float> face_flux_q(Pr<float> vel, Pr<float> m3, Pr<float> m2, Pr<float> m1, Pr<float> p0,
                                                 Pr<float> p1, Pr<float> p2, Pr<float> eps4) {
    const bool ux = vel.x() >= 0.f, uy = vel.y() >= 0.f;
    return mul(vel, weno5q(mk(ux ? m3.x() : p2.x(), uy ? m3.y() : p2.y()), mk(ux ? m2.x() : p1.x(), uy ? m2.y() : p1.y()),
                           mk(ux ? m1.x() : p0.x(), uy ? m1.y() : p0.y()), mk(ux ? p0.x() : m1.x(), uy ? p0.y() : m1.y()),
                           mk(ux ? p1.x() : m2.x(), uy ? p1.y() : m2.y()), eps4));
}

enum { kRowsAny, kRowsEven, kRowsWalled, kRowsPeriodic };

template <bool ADV>
struct Explicit3Smem {
    static constexpr int PX = kTX2 + 2 * kHL2, PY = kTY + 2 * kHalo, NT = 32 * kTY;
    // without advection there is one barrier a plane, and a third buffer keeps
    // the plane being read from the one being filled
    static constexpr int NB = ADV ? 2 : 3;
    __align__(16) float Cs[NB][PY][PX];
    __align__(16) float Sl[2][ADV ? 4 : 1][2 * NT];  // H^{l-1}, u, v, w of the thread's pair at [2 tid]
    __align__(16) float Sy[2][ADV ? kTX2 : 2];       // v of the tile's extra y-faces
    __align__(16) float Fy[ADV ? kTY + 1 : 1][kTX2];
    unsigned long long bar;                          // split barrier of the face fluxes
    float Sx[2][ADV ? kTY : 1];                      // u of its extra x-faces
    float Fe[ADV ? kTY : 1];
    int gi_tab[PX], gj_tab[PY];
};

// One 64 x 8 x zchunk tile (tile coordinates bx, by, bz) by the 256 threads of
// a CTA.  No __restrict__: the batched kernel writes these arrays in one phase
// and reads them in the next.
template <bool ADV, bool DIRI, int XM>
__device__ __forceinline__ void explicit_tile3(const float* C, const float* u, const float* v, const float* w,
                                               const float* Hprev, float* Hout, float* r, const RhsArgs<float>& a,
                                               int bx, int by, int bz, int zchunk, Explicit3Smem<ADV>& sm,
                                               unsigned int* status) {
    constexpr int PX = kTX2 + 2 * kHL2, PY = kTY + 2 * kHalo, NT = 32 * kTY;
    // AL: rows are 16-byte aligned; EV: 8-byte aligned, so both cells of a pair are in or out
    constexpr bool EV = XM != kRowsAny, AL = EV && XM != kRowsEven, per_x = XM == kRowsPeriodic;  // per_x false: a.bcx decides
    constexpr int NB = Explicit3Smem<ADV>::NB;
    auto& Cs = sm.Cs;
    auto& Sl = sm.Sl;
    auto& Sy = sm.Sy;
    auto& Sx = sm.Sx;
    auto& Fy = sm.Fy;
    auto& Fe = sm.Fe;
    auto& gi_tab = sm.gi_tab;
    auto& gj_tab = sm.gj_tab;

    const int tid = threadIdx.x + threadIdx.y * 32, tx = tid & 31, ty = tid >> 5;
    const int i0 = bx * kTX2, j0 = by * kTY, k0 = bz * zchunk, kend = min(k0 + zchunk, a.nz);
    const int ia = i0 + 2 * tx, j = j0 + ty;
    const bool in_a = ia < a.nx && j < a.ny, in_b = EV ? in_a : ia + 1 < a.nx && j < a.ny;
    // the pair's columns in global memory; where the second is past the row, the
    // one that its ghost copies
    const int jc = min(j, a.ny - 1), ic = min(ia, EV ? a.nx - 2 : a.nx - 1);
    const int icb = EV || ic + 1 < a.nx ? ic + 1 : (a.bcx == CH_PERIODIC ? 0 : a.nx - 1);
    const int plane = a.nx * a.ny;  // every field holds fewer than 2^31 elements
    const int col = jc * a.nx + ic;
    const Pr<float> eps4 = sp(4.f * a.eps);
    auto ld2g = [&](const float* p) {  // the pair whose first element is at column ic
        if constexpr (EV) return ldp(p);
        else return mk(p[0], p[icb - ic]);
    };

    __syncthreads();  // the buffers may still be read by a previous tile of this CTA
    if (ADV && tid == 0) warps_init(&sm.bar, kTY);
    if (tid < PX) gi_tab[tid] = bc_index(i0 + tid - kHL2, a.nx, a.bcx);
    else if (tid < PX + PY) gj_tab[tid - PX] = bc_index(j0 + (tid - PX) - kHalo, a.ny, a.bcy);

    // z-column queue of pairs: q[m] = C(k - 2 + m)
    Pr<float> q[6];
    auto zpair = [&](int k) {
        if (k >= 0 && k < a.nz) return ld2g(C + (k * plane + col));
        Pr<float> c = ld2g(C + (bc_near(k, a.nz, a.bcz) * plane + col));
        if (DIRI && bc_negate(k, a.nz, a.bcz)) c = sub(sp(0.f), c);
        return c;
    };
#pragma unroll
    for (int m = 0; m < 6; ++m) q[m] = zpair(k0 - 2 + m);
    Pr<float> fz_lo = sp(0.f);
    if (ADV && !(a.bcz != CH_PERIODIC && k0 == 0))
        fz_lo = face_flux_q(ld2g(w + (k0 * plane + col)), zpair(k0 - 3), q[0], q[1], q[2], q[3], q[4], eps4);
    Pr<float> psm = psi_pp(q[1]), ps0 = psi_pp(q[2]);
    if (DIRI && k0 == 0) psm = sub(sp(0.f), ps0);  // psi' = 0 on the wall: its ghost is its own negated mirror
    __syncthreads();  // index tables ready

    // this thread's copies.  C: AL, chunk tid of 252 (18 a row; the last threads
    // repeat the last one); a chunk past a no-flux x-wall is reversed, element by
    // element.  EV, pairs likewise: pairs tid and tid + 256 of 504 (36 a row).  Else
    // elements tid + 256 m.
    const int ctid = min(tid, PX * PY / 4 - 1);
    constexpr int kCN = AL ? 1 : EV ? 2 : (PX * PY + NT - 1) / NT;
    int csrc[kCN];
    bool rev = false;
    if constexpr (AL) {
        const int row = ctid / (PX / 4), c = (ctid - row * (PX / 4)) * 4, c0 = i0 + c - kHL2;
        rev = !per_x && (c0 < 0 || c0 == a.nx);
        // chunks further past a wall are never used: any valid source
        csrc[0] = gj_tab[row] * a.nx + (!per_x && c0 > a.nx ? 0 : gi_tab[c]);
    } else if constexpr (EV) {
#pragma unroll
        for (int m = 0; m < 2; ++m) {
            const int e = min(tid + m * NT, PX * PY / 2 - 1), row = e / (PX / 2), c = (e - row * (PX / 2)) * 2;
            const int c0 = i0 + c - kHL2;
            const bool wall = a.bcx != CH_PERIODIC;
            csrc[m] = gj_tab[row] * a.nx + (wall && c0 > a.nx + 2 ? 0 : gi_tab[c]);
            if (wall && (c0 < 0 || c0 == a.nx || c0 == a.nx + 2)) csrc[m] = ~csrc[m];  // reversed
        }
    } else {
#pragma unroll
        for (int m = 0; m < kCN; ++m) {
            const int e = tid + m * NT, row = e / PX;
            csrc[m] = e < PX * PY ? gj_tab[row] * a.nx + gi_tab[e - row * PX] : 0;
        }
    }
    // velocities of the faces ia, ia + 1 (x) and j (y), and the tile's extra
    // faces: the y-face j0 + 8 by warp 0, the x-face i0 + 64 by warp 1
    const bool bper_x = per_x || a.bcx == CH_PERIODIC, per_y = a.bcy == CH_PERIODIC, per_z = a.bcz == CH_PERIODIC;
    int eu = 0, eub = 0, ev = 0, ew = 0, ex = 0, nu = 0, nub = 0, nv = 0, nx_ = 0, su = 0, sv = 0, sx = 0;
    if (ADV) {
        const int fa = bper_x ? bc_index(ia, a.nx, CH_PERIODIC) : min(ia, a.nx);
        const int fb = bper_x ? bc_index(ia + 1, a.nx, CH_PERIODIC) : min(ia + 1, a.nx);
        const int fy = per_y ? bc_index(j, a.ny, CH_PERIODIC) : min(j, a.ny);
        su = a.ny * a.nfx;
        sv = a.nfy * a.nx;
        eu = k0 * su + jc * a.nfx + fa;
        eub = fb - fa;
        ev = k0 * sv + fy * a.nx + ic;
        nu = !bper_x && (ia <= 0 || ia >= a.nx) ? 0 : 4;
        nub = !bper_x && ia + 1 >= a.nx ? 0 : 4;
        nv = !per_y && (j <= 0 || j >= a.ny) ? 0 : 4;
        ew = k0 * plane + col;
        if (ty == 0) {  // extra y-faces
            const int je = j0 + kTY, fye = per_y ? bc_index(je, a.ny, CH_PERIODIC) : min(je, a.ny);
            ex = k0 * sv + fye * a.nx + ic;
            sx = sv;
            nx_ = !per_y && je >= a.ny ? 0 : 4;
        } else if (ty == 1 && tx < kTY) {  // extra x-faces, one row a lane
            const int ie = i0 + kTX2, fxe = bper_x ? bc_index(ie, a.nx, CH_PERIODIC) : min(ie, a.nx);
            ex = k0 * su + min(j0 + tx, a.ny - 1) * a.nfx + fxe;
            sx = su;
            nx_ = !bper_x && ie >= a.nx ? 0 : 4;
        }
    }
    int eh = k0 * plane + col;  // H^{l-1}
    const int nh = in_a && a.has_prev ? 4 : 0, nhb = in_b && a.has_prev ? 4 : 0;
    float* slot = &Sl[0][0][2 * tid];
    constexpr int SB = (ADV ? 4 : 1) * 2 * NT;  // floats from one buffer's slots to the other's

    // plane kk into C buffer b and slots s, the sources of the slots standing at kk
    auto stage = [&](int kk, int b, int s) {
        const float* Ck = C + kk * plane;
        float* dst = &Cs[b][0][0];
        if constexpr (AL) {
            if (per_x || !rev) cp_async_16(dst + 4 * ctid, Ck + csrc[0]);
            else
#pragma unroll
                for (int e = 0; e < 4; ++e) cp_async_elem(dst + 4 * ctid + e, Ck + csrc[0] - e);
        } else if constexpr (EV) {
#pragma unroll
            for (int m = 0; m < 2; ++m) {
                float* d = dst + 2 * min(tid + m * NT, PX * PY / 2 - 1);
                if (csrc[m] >= 0) {
                    cp_async_pair(d, Ck + csrc[m]);
                } else {
                    cp_async_elem(d, Ck + ~csrc[m]);
                    cp_async_elem(d + 1, Ck + (~csrc[m] - 1));
                }
            }
        } else {
#pragma unroll
            for (int m = 0; m < kCN; ++m)
                if (tid + m * NT < PX * PY) cp_async_elem(dst + tid + m * NT, Ck + csrc[m]);
        }
        float* S = slot + s * SB;
        if constexpr (EV) {
            cp_async_fill<2>(S, Hprev + eh, 2 * nh);
        } else {
            cp_async_fill<1>(S, Hprev + eh, nh);
            cp_async_fill<1>(S + 1, Hprev + eh + (icb - ic), nhb);
        }
        eh += plane;
        if constexpr (ADV) {
            if constexpr (per_x) {
                cp_async_pair(S + 2 * NT, u + eu);
            } else {
                cp_async_fill<1>(S + 2 * NT, u + eu, nu);
                cp_async_fill<1>(S + 2 * NT + 1, u + (eu + eub), nub);
            }
            // the z-face above plane kk: w of plane kk + 1, wrapped
            const float* wk = w + (kk + 1 < a.nz || !per_z ? ew + plane : col);
            if constexpr (EV) {
                cp_async_fill<2>(S + 4 * NT, v + ev, 2 * nv);
                cp_async_pair(S + 6 * NT, wk);
            } else {
                cp_async_fill<1>(S + 4 * NT, v + ev, nv);
                cp_async_fill<1>(S + 4 * NT + 1, v + ev + (icb - ic), nv);
                cp_async_elem(S + 6 * NT, wk);
                cp_async_elem(S + 6 * NT + 1, wk + (icb - ic));
            }
            if (ty == 0) {
                if constexpr (EV) {
                    cp_async_fill<2>(&Sy[s][2 * tx], v + ex, 2 * nx_);
                } else {
                    cp_async_fill<1>(&Sy[s][2 * tx], v + ex, nx_);
                    cp_async_fill<1>(&Sy[s][2 * tx + 1], v + ex + (icb - ic), nx_);
                }
            } else if (ty == 1 && tx < kTY) {
                cp_async_fill<1>(&Sx[s][tx], u + ex, nx_);
            }
            eu += su;
            ev += sv;
            ew += plane;
            ex += sx;
        }
        cp_async_commit();
    };

    int idx = k0 * plane + col;  // this plane's output
    stage(k0, 0, 0);
    // two planes a turn without advection (13.6 against 14.1 us on 128^3); with
    // it the second copy spills (5.33 against 4.85 ms on 1024 x 1024 x 512)
    constexpr int kTurn = ADV ? 1 : 2;
#pragma unroll kTurn
    for (int k = k0, buf = 0, sl = 0; k < kend; ++k, sl ^= 1) {
        const int nbuf = buf + 1 == NB ? 0 : buf + 1;
        if (k + 1 < kend) {
            stage(k + 1, nbuf, sl ^ 1);
            cp_async_wait<1>();
        } else {
            cp_async_wait<0>();
        }
        const Pr<float> qnext = zpair(k + 4);
        __syncthreads();
        const float(*P)[PX] = Cs[buf];
        const float* S = slot + sl * SB;
        const int cy = ty + kHalo, cx = 2 * tx + kHL2;  // cell ia
        // x-window ia-4 .. ia+3 and the y-column pairs j-3 .. j+2
        const Pr<float> x0 = ldp(&P[cy][cx - 4]), x1 = ldp(&P[cy][cx - 2]), c0 = ldp(&P[cy][cx]), x3 = ldp(&P[cy][cx + 2]);
        const Pr<float> ym2 = ldp(&P[cy - 2][cx]), ym1 = ldp(&P[cy - 1][cx]);
        const Pr<float> yp1 = ldp(&P[cy + 1][cx]), yp2 = ldp(&P[cy + 2][cx]);
        const Pr<float> xm2 = x1, xm1 = mk(x1.y(), c0.x()), xp1 = mk(c0.y(), x3.x()), xp2 = x3;
        const Pr<float> hp = ldp(S);
        Pr<float> fx = sp(0.f), fy = sp(0.f), fz_up = sp(0.f);
        if constexpr (ADV) {
            // lower x-faces of the two cells, lower y-faces, upper z-faces
            fx = face_flux_q(ldp(S + 2 * NT), mk(x0.y(), x1.x()), x1, xm1, c0, xp1, x3, eps4);
            fy = face_flux_q(ldp(S + 4 * NT), ldp(&P[cy - 3][cx]), ym2, ym1, c0, yp1, yp2, eps4);
            stp(&Fy[ty][2 * tx], fy);
            if (ty == 0) {
                const int yy = kTY + kHalo;
                stp(&Fy[kTY][2 * tx],
                    face_flux_q(ldp(&Sy[sl][2 * tx]), ldp(&P[yy - 3][cx]), ldp(&P[yy - 2][cx]), ldp(&P[yy - 1][cx]),
                                ldp(&P[yy][cx]), ldp(&P[yy + 1][cx]), ldp(&P[yy + 2][cx]), eps4));
            } else if (ty == 1 && tx < kTY / 2) {  // rows 2 tx, 2 tx + 1 of the tile
                const int ra = 2 * tx + kHalo, rb = ra + 1, xx = kTX2 + kHL2;
                const Pr<float> f = face_flux_q(
                    mk(Sx[sl][2 * tx], Sx[sl][2 * tx + 1]), mk(P[ra][xx - 3], P[rb][xx - 3]),
                    mk(P[ra][xx - 2], P[rb][xx - 2]), mk(P[ra][xx - 1], P[rb][xx - 1]), mk(P[ra][xx], P[rb][xx]),
                    mk(P[ra][xx + 1], P[rb][xx + 1]), mk(P[ra][xx + 2], P[rb][xx + 2]), eps4);
                Fe[2 * tx] = f.x();
                Fe[2 * tx + 1] = f.y();
            }
            // the face between this warp's rows and its neighbours' is published: arrive
            // now, wait after the z-faces, the Laplacian and the fourth differences
            warps_arrive(&sm.bar, tx);
            if (per_z || k + 1 < a.nz) fz_up = face_flux_q(ldp(S + 6 * NT), q[0], q[1], q[2], q[3], q[4], q[5], eps4);
        }
        // M lap(psi'(C)), neighbour differences first, so FP32 keeps the
        // accuracy of the small differences
        const Pr<float> ps_next = psi_pp(q[3]);
        Pr<float> psp = ps_next;
        if (DIRI && k + 1 == a.nz) psp = sub(sp(0.f), psi_pp(sub(sp(0.f), q[3])));
        const Pr<float> pxe = psi_pp(mk(x1.y(), x3.x()));  // of cells ia - 1 and ia + 2
        const Pr<float> lap = mul(add(add(add(sub(mk(pxe.x(), ps0.x()), ps0), sub(mk(ps0.y(), pxe.y()), ps0)),
                                          add(sub(psi_pp(ym1), ps0), sub(psi_pp(yp1), ps0))),
                                      add(sub(psm, ps0), sub(psp, ps0))),
                                  sp(a.inv_h2));
        // [1,-4,6,-4,1] sums of A_x + A_y + A_z (Eq. eq-a3d) from the first
        // differences along each line: (d1 - d-2) - 3 (d0 - d-1)
        auto fourth = [&](Pr<float> m2, Pr<float> m1, Pr<float> p1, Pr<float> p2) {
            return fma2(sp(-3.f), sub(sub(p1, c0), sub(c0, m1)), sub(sub(p2, p1), sub(m1, m2)));
        };
        const Pr<float> astar = add(add(fourth(xm2, xm1, xp1, xp2), fourth(ym2, ym1, yp1, yp2)), fourth(q[0], q[1], q[3], q[4]));
        Pr<float> H = mul(sp(a.mob), lap);
        if constexpr (ADV) {
            float fr = __shfl_down_sync(kFull, fx.x(), 1);  // the next lane's lower x-face
            if (!warps_wait(&sm.bar, (k - k0) & 1)) atomicOr(status, 4u);
            if (tx == 31) fr = Fe[ty];
            const Pr<float> dxf = sub(mk(fx.y(), fr), fx), dyf = sub(ldp(&Fy[ty + 1][2 * tx]), fy);
            H = fma2(sp(-a.inv_h), add(add(dxf, dyf), sub(fz_up, fz_lo)), H);
            fz_lo = fz_up;
        }
        const Pr<float> rhs = fma2(sp(a.dtr), hp, fma2(sp(-a.impl), astar, mul(sp(a.dtg), H)));
        if constexpr (EV) {
            if (in_a) {
                stp(Hout + idx, H);
                if (r) stp(r + idx, rhs);
            }
        } else {
            if (in_a) {
                Hout[idx] = H.x();
                if (r) r[idx] = rhs.x();
            }
            if (in_b) {
                Hout[idx + 1] = H.y();
                if (r) r[idx + 1] = rhs.y();
            }
        }
        idx += plane;
        psm = ps0;
        ps0 = ps_next;
#pragma unroll
        for (int m = 0; m < 5; ++m) q[m] = q[m + 1];
        q[5] = qnext;
        buf = nbuf;
    }
}

template <bool ADV, bool DIRI, int XM>
__global__ void __launch_bounds__(32 * kTY, XM == kRowsAny ? 2 : 3)
ch_explicit_rhs3(const float* __restrict__ C, const float* __restrict__ u, const float* __restrict__ v,
                 const float* __restrict__ w, const float* __restrict__ Hprev, float* __restrict__ Hout,
                 float* __restrict__ r, RhsArgs<float> a, int zchunk, unsigned int* status) {
    pdl_wait();
    pdl_launch_dependents();
    __shared__ Explicit3Smem<ADV> sm;
    explicit_tile3<ADV, DIRI, XM>(C, u, v, w, Hprev, Hout, r, a, blockIdx.x, blockIdx.y, blockIdx.z, zchunk, sm, status);
}

}  // namespace chg

// The standard explicit scheme the paper's split operator replaces
// (arXiv 2105.01865, Sec. 3.1, Eq. eq-disbi; compared in Sec. 4.1).
//
// Every term of Eq. (eq-ch) is explicit in the same low-storage RK3:
//   H^l = -div(uC) + M lap_h(psi'(C) - Cn^2 lap_h C),
//   C  <- C + dt (gamma_l H^l + rho_l H^{l-1}).
// M lap_h(psi' - Cn^2 lap_h C) equals M lap_h psi'(C) - M Cn^2 lap_h^2 C, the
// 25-point biharmonic of Eq. (eq-disbi) (13 points in 2D), so the substep is
// three launches: the chemical potential mu = psi'(C) - Cn^2 lap_h C
// (ch_std_mu), the WENO5 advection of the split scheme's explicit kernel run
// with its diffusive and implicit terms switched off, and the update
// (ch_std_update).  Ghost cells follow the split scheme: periodic wrap or the
// mirror about a wall face, so both Laplacians are conservative.
#include <cuda_runtime.h>

#include "ch_internal.h"
#include "ch_kernels.cuh"

using namespace chg;

namespace {

template <typename T>
struct StdArgs {
    int nx, ny, nz;
    int bcx, bcy, bcz;
    T cn2_h2;   // Cn^2 / h^2
    T mob_h2;   // M / h^2
    T dtg, dtr; // dt gamma_l, dt rho_l
    int has_prev;
};

// Neighbour index at +-1 along a line of n cells: wrap, or the mirror about
// the wall face (ghost C_{-1} = C_0, C_n = C_{n-1}).
__device__ __forceinline__ int nb_lo(int i, int n, int bc) { return i > 0 ? i - 1 : (bc == CH_PERIODIC ? n - 1 : 0); }
__device__ __forceinline__ int nb_hi(int i, int n, int bc) { return i + 1 < n ? i + 1 : (bc == CH_PERIODIC ? 0 : n - 1); }

// V adjacent cells of a thread: one access of 4 V or 8 V bytes (V = 4: rows are
// 16-byte aligned)
template <typename T, int V>
__device__ __forceinline__ void ldv(const T* p, T (&v)[V]) {
    if constexpr (V == 4) {
        const float4 t = *reinterpret_cast<const float4*>(p);
        v[0] = t.x; v[1] = t.y; v[2] = t.z; v[3] = t.w;
    } else {
        v[0] = *p;
    }
}
template <typename T, int V>
__device__ __forceinline__ void stv(T* p, const T (&v)[V]) {
    if constexpr (V == 4) *reinterpret_cast<float4*>(p) = make_float4(v[0], v[1], v[2], v[3]);
    else *p = v[0];
}

// Sums of the six neighbour differences of f at the cells (i .. i + V - 1, j, k)
// (lap_h times h^2), differences formed first as in the split scheme's Laplacian.
template <typename T, int V>
__device__ __forceinline__ void lap_sum(const T* f, int i, int j, int k, const StdArgs<T>& a, const T (&c)[V], T (&s)[V]) {
    const int64_t row = (int64_t)a.nx, plane = (int64_t)a.nx * a.ny;
    const int64_t base = (int64_t)k * plane + (int64_t)j * row;
    const T xl = f[base + nb_lo(i, a.nx, a.bcx)], xr = f[base + nb_hi(i + V - 1, a.nx, a.bcx)];
    T ym[V], yp[V], zm[V], zp[V];
    ldv<T, V>(f + (int64_t)k * plane + (int64_t)nb_lo(j, a.ny, a.bcy) * row + i, ym);
    ldv<T, V>(f + (int64_t)k * plane + (int64_t)nb_hi(j, a.ny, a.bcy) * row + i, yp);
    ldv<T, V>(f + (int64_t)nb_lo(k, a.nz, a.bcz) * plane + (int64_t)j * row + i, zm);
    ldv<T, V>(f + (int64_t)nb_hi(k, a.nz, a.bcz) * plane + (int64_t)j * row + i, zp);
#pragma unroll
    for (int q = 0; q < V; ++q) {
        const T xm = q ? c[q - 1] : xl, xp = q + 1 < V ? c[q + 1] : xr;
        s[q] = (((xm - c[q]) + (xp - c[q])) + ((ym[q] - c[q]) + (yp[q] - c[q]))) + ((zm[q] - c[q]) + (zp[q] - c[q]));
    }
}

// Both kernels are bound by their loads, seven a cell.  Four adjacent cells a
// thread (FP32, nx a multiple of 4) share 16-byte accesses and take the x-
// neighbours from each other: 36.6 -> 14.2 us (mu) and 49.3 -> 22.8 (update) on
// 256 x 256 x 128.

// mu = psi'(C) - Cn^2 lap_h C, psi'(C) = C (C (C - 1.5) + 0.5)
template <typename T, int V>
__global__ void __launch_bounds__(256) ch_std_mu(const T* __restrict__ C, T* __restrict__ mu, StdArgs<T> a) {
    const int bx = V == 1 ? 32 : blockDim.x, by = V == 1 ? 8 : blockDim.y;
    const int i = (blockIdx.x * bx + threadIdx.x) * V, j = blockIdx.y * by + threadIdx.y, k = blockIdx.z;
    if (i >= a.nx || j >= a.ny) return;
    const int64_t idx = ((int64_t)k * a.ny + j) * a.nx + i;
    T c[V], s[V];
    ldv<T, V>(C + idx, c);
    lap_sum<T, V>(C, i, j, k, a, c, s);
#pragma unroll
    for (int q = 0; q < V; ++q) {
        const T psi_p = c[q] * (c[q] * (c[q] - T(1.5)) + T(0.5));
        s[q] = psi_p - a.cn2_h2 * s[q];
    }
    stv<T, V>(mu + idx, s);
}

// H = [-div(uC)] + M lap_h mu; C += dt (gamma H + rho H^{l-1}).  Hadv may be
// the same array as Hout (each thread reads its cells before writing them).
template <typename T, int V, bool ADV>
__global__ void __launch_bounds__(256) ch_std_update(const T* __restrict__ mu, const T* Hadv, const T* __restrict__ Hprev,
                                                     T* Hout, T* __restrict__ C, StdArgs<T> a, unsigned int* status) {
    const int bx = V == 1 ? 32 : blockDim.x, by = V == 1 ? 8 : blockDim.y;
    const int i = (blockIdx.x * bx + threadIdx.x) * V, j = blockIdx.y * by + threadIdx.y, k = blockIdx.z;
    if (i >= a.nx || j >= a.ny) return;
    const int64_t idx = ((int64_t)k * a.ny + j) * a.nx + i;
    T m[V], H[V], hp[V], c[V], ha[V];
    ldv<T, V>(mu + idx, m);
    ldv<T, V>(C + idx, c);
    if (ADV) ldv<T, V>(Hadv + idx, ha);
    if (a.has_prev) ldv<T, V>(Hprev + idx, hp);
    lap_sum<T, V>(mu, i, j, k, a, m, H);
    bool bad = false;
#pragma unroll
    for (int q = 0; q < V; ++q) {
        H[q] *= a.mob_h2;
        if (ADV) H[q] += ha[q];
        T rhs = a.dtg * H[q];
        if (a.has_prev) rhs += a.dtr * hp[q];
        c[q] += rhs;
        bad |= !isfinite(c[q]);
    }
    stv<T, V>(Hout + idx, H);
    stv<T, V>(C + idx, c);
    if (bad) atomicOr(status, 1u);
}

template <typename T>
int substep_standard(ch_handle* h, int l, cudaEvent_t* ev) {
    const ch_params& p = h->p;
    StdArgs<T> a;
    a.nx = (int)h->n[0];
    a.ny = (int)h->n[1];
    a.nz = (int)h->n[2];
    a.bcx = p.bc[0];
    a.bcy = p.bc[1];
    a.bcz = p.bc[2];
    a.cn2_h2 = (T)(p.cn * p.cn / (p.h * p.h));
    a.mob_h2 = (T)(1.0 / (p.pe * p.h * p.h));
    a.dtg = (T)(p.dt * kGamma[l]);
    a.dtr = (T)(p.dt * kRho[l]);
    a.has_prev = kRho[l] != 0.0;
    T* C = (T*)h->C;
    T* mu = (T*)h->r;  // the split scheme's right-hand side buffer holds mu
    T* Hcur = (T*)h->H[l & 1];
    const T* Hprev = (const T*)h->H[(l + 1) & 1];
    const bool quads = sizeof(T) == 4 && a.nx % 4 == 0;
    // With quads a row may have fewer of them than a warp has lanes: then a warp
    // takes two or four rows, the widest that leaves the fewest lanes idle (a step of
    // 32 x 512 x 32: 30.9 us in whole rows, 18.5 so; one cell a thread 24.7)
    int bx = 32;
    if (quads) {
        const int row = a.nx / 4;
        auto lanes = [&](int b) { return (row + b - 1) / b * b; };
        for (int b = 16; b >= 8; b /= 2)
            if (lanes(b) < lanes(bx)) bx = b;
    }
    const int by = 256 / bx, per = quads ? 4 * bx : bx;  // cells of a block's row
    const dim3 block(bx, by), grid((unsigned)((a.nx + per - 1) / per), (unsigned)((a.ny + by - 1) / by), (unsigned)a.nz);
    constexpr int Q = sizeof(T) == 4 ? 4 : 1;
    if (ev) CHG_CUDA(h, cudaEventRecord(ev[0], h->stream));
    if (quads) ch_std_mu<T, Q><<<grid, block, 0, h->stream>>>(C, mu, a);
    else ch_std_mu<T, 1><<<grid, block, 0, h->stream>>>(C, mu, a);
    CHG_CUDA(h, cudaGetLastError());
    if (ev) CHG_CUDA(h, cudaEventRecord(ev[1], h->stream));
    if (p.advect) {
        const int rc = launch_advection_any(h, C, Hcur);
        if (rc != CH_OK) return rc;
    }
    if (ev) CHG_CUDA(h, cudaEventRecord(ev[2], h->stream));
    if (p.advect && quads)
        ch_std_update<T, Q, true><<<grid, block, 0, h->stream>>>(mu, Hcur, Hprev, Hcur, C, a, h->status);
    else if (p.advect)
        ch_std_update<T, 1, true><<<grid, block, 0, h->stream>>>(mu, Hcur, Hprev, Hcur, C, a, h->status);
    else if (quads)
        ch_std_update<T, Q, false><<<grid, block, 0, h->stream>>>(mu, nullptr, Hprev, Hcur, C, a, h->status);
    else
        ch_std_update<T, 1, false><<<grid, block, 0, h->stream>>>(mu, nullptr, Hprev, Hcur, C, a, h->status);
    CHG_CUDA(h, cudaGetLastError());
    if (ev) {
        CHG_CUDA(h, cudaEventRecord(ev[3], h->stream));
        CHG_CUDA(h, cudaEventRecord(ev[4], h->stream));
    }
    return CH_OK;
}

}  // namespace

namespace chg {

int launch_substep_standard(ch_handle* h, int l, cudaEvent_t* ev) {
    return h->prec == CH_F64 ? substep_standard<double>(h, l, ev) : substep_standard<float>(h, l, ev);
}

}  // namespace chg

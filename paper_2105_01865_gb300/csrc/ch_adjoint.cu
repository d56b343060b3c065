// Adjoint (reverse-mode derivative) of nsteps Cahn-Hilliard steps without
// advection, with checkpointed recomputation (arXiv 2105.01865, Sec. 3 step;
// the derivative itself has no counterpart in the paper).
//
// For substep l with C' = C + P^-1 r, r = dt(gamma H + rho Hp) - alpha dt M A C,
// H = M lap(psi'(C)), P = prod_d (I + c A_d), c = alpha dt M / 2, the reverse
// map of adjoints (lam_C', lam_H' of this H as the next substep's Hp) is
//   lam_r  = P^-1 lam_C'                       (the same line solves)
//   lam_H  = dt gamma lam_r + lam_H',  lam_Hp = dt rho lam_r
//   lam_C  = lam_C' - alpha dt M A lam_r + psi''(C) M lap(lam_H)
//   dL/dM += <lam_H, lap psi'(C)> - alpha dt <lam_r, A C>
//            - (alpha dt / 2) sum_d <A_d lam_r, (I + c A_d)^-1 r>
// (all operators symmetric; the P_d act on different axes and commute).
#include <cuda_runtime.h>

#include <algorithm>
#include <vector>

#include "ch_internal.h"
#include "ch_kernels.cuh"

using namespace chg;

namespace {

constexpr int kAThreadsX = 32, kAThreadsY = 8;

template <typename T>
struct AdjArgs {
    int nx, ny, nz, bcx, bcy, bcz;
    double dt, gamma, rho, alpha, mob, kappa, inv_h2;
};

template <typename T>
__device__ __forceinline__ T psi_prime_t(T c) { return c * (c * (c - T(1.5)) + T(0.5)); }

// The products of a cell for dL/dM, into FP64 sums: FP64 holds the product of two
// FP32 values exactly and has range to spare for any scale of the loss.
__device__ __forceinline__ void adj_dots(const double (&a)[5], const double (&b)[5], double& d1, double& d2) {
    d1 += a[0] * b[0];
#pragma unroll
    for (int m = 1; m < 5; ++m) d2 += a[m] * b[m];
}
// FP32 values are widened by their bits on the integer pipe, and by the
// conversion, which runs at 1/64 of the FP32 rate like the multiply-adds, only in
// cells where one is subnormal or not finite.  128^3: a launch takes 69 us, 100
// with conversions throughout, 50 with sums in double-float, which has no more than
// FP32's range and 48 bits.
__device__ __forceinline__ bool zero_or_normal(float f) {
    const unsigned t = __float_as_uint(f) << 1;  // without its sign
    return t == 0u || t - 0x01000000u < 0xfe000000u;
}
__device__ __forceinline__ double widen(float f) {
    const unsigned b = __float_as_uint(f);
    const unsigned hi = ((unsigned)((int)b >> 3) & 0x8fffffffu) + 0x38000000u;  // exponent bias 127 -> 1023
    return f == 0.f ? 0.0 : __hiloint2double((int)hi, (int)(b << 29));
}
__device__ __forceinline__ void adj_dots(const float (&a)[5], const float (&b)[5], double& d1, double& d2) {
    bool plain = true;
#pragma unroll
    for (int m = 0; m < 5; ++m) plain = plain & zero_or_normal(a[m]) & zero_or_normal(b[m]);
    if (plain)
        adj_dots({widen(a[0]), widen(a[1]), widen(a[2]), widen(a[3]), widen(a[4])},
                 {widen(b[0]), widen(b[1]), widen(b[2]), widen(b[3]), widen(b[4])}, d1, d2);
    else
        adj_dots({(double)a[0], (double)a[1], (double)a[2], (double)a[3], (double)a[4]},
                 {(double)b[0], (double)b[1], (double)b[2], (double)b[3], (double)b[4]}, d1, d2);
}

// [1,-4,6,-4,1] of five neighbours along one direction, as differences
template <typename T>
__device__ __forceinline__ T fourth(T m2, T m1, T c, T p1, T p2) {
    const T da = m1 - c, db = p1 - c;
    return ((m2 - m1) - da) + ((p2 - p1) - db) - T(2) * (da + db);
}

// The reverse substep map above, in the field precision.  A thread marches
// kAdjZ planes of its column: its z-neighbours stay in registers, and the
// in-plane ones are read through offsets found once, so a cell costs 27 loads
// that neighbouring threads share in L1.  Bound by those loads.  One thread a
// cell, with every neighbour's index reduced modulo the box, took 356 us on
// 128^3 (FP32); this form 69, 19 of them for the FP64 sums.  FP32 takes 4 CTAs an SM (64
// registers; 3 at 76: 82 us).
constexpr int kAdjZ = 8;
template <typename T>
__global__ void __launch_bounds__(kAThreadsX * kAThreadsY, sizeof(T) == 4 ? 4 : 2)
adj_substep(const T* __restrict__ C, const T* __restrict__ lam_r, const T* __restrict__ lamH_in,
            const T* __restrict__ lamC_in, const T* __restrict__ s0, const T* __restrict__ s1,
            const T* __restrict__ s2, T* __restrict__ lamC_out, T* __restrict__ lamHp_out, double* partials,
            AdjArgs<T> a) {
    const int i = blockIdx.x * kAThreadsX + threadIdx.x;
    const int j = blockIdx.y * kAThreadsY + threadIdx.y;
    const int k0 = blockIdx.z * kAdjZ, k1 = min(k0 + kAdjZ, a.nz);
    double dm = 0.0;
    if (i < a.nx && j < a.ny) {
        // in-plane neighbours of (i, j), as offsets from it
        const int64_t plane = (int64_t)a.nx * a.ny, ij = (int64_t)j * a.nx + i;
        const int xm1 = bc_near(i - 1, a.nx, a.bcx) - i, xp1 = bc_near(i + 1, a.nx, a.bcx) - i;
        const int xm2 = bc_near(i - 2, a.nx, a.bcx) - i, xp2 = bc_near(i + 2, a.nx, a.bcx) - i;
        const int ym1 = (bc_near(j - 1, a.ny, a.bcy) - j) * a.nx, yp1 = (bc_near(j + 1, a.ny, a.bcy) - j) * a.nx;
        const int ym2 = (bc_near(j - 2, a.ny, a.bcy) - j) * a.nx, yp2 = (bc_near(j + 2, a.ny, a.bcy) - j) * a.nx;
        auto zoff = [&](int k) { return bc_near(k, a.nz, a.bcz) * plane + ij; };
        const T dtg = T(a.dt * a.gamma), mob = T(a.mob), inv_h2 = T(a.inv_h2), kap = T(a.kappa);
        const T adt = T(a.alpha * a.dt), dtr = T(a.dt * a.rho);
        // q[m] = row k - 2 + m of C and lam_r; lam_H' of this substep one row down and at k
        T qc[5], ql[5];
#pragma unroll
        for (int m = 0; m < 4; ++m) {
            qc[m] = C[zoff(k0 - 2 + m)];
            ql[m] = lam_r[zoff(k0 - 2 + m)];
        }
        T hm = lamH_in[zoff(k0 - 1)], hc = lamH_in[zoff(k0)];
        double d1 = 0.0, d2 = 0.0;  // <lam_H, lap psi'> and <lam_r, A C> + sum_d <A_d lam_r, s_d> / 2
        for (int k = k0; k < k1; ++k) {
            const int64_t e = k * plane + ij, z2 = zoff(k + 2);
            qc[4] = C[z2];
            ql[4] = lam_r[z2];
            const T hp = lamH_in[zoff(k + 1)];
            const T *pc = C + e, *pl = lam_r + e, *ph = lamH_in + e;
            const T c = qc[2], lr = ql[2];
            const T cxm = pc[xm1], cxp = pc[xp1], cym = pc[ym1], cyp = pc[yp1];
            const T lxm = pl[xm1], lxp = pl[xp1], lym = pl[ym1], lyp = pl[yp1];
            const T lh0 = dtg * lr + hc;
            const T lap_lh = (((dtg * lxm + ph[xm1]) - lh0) + ((dtg * lxp + ph[xp1]) - lh0) +
                              ((dtg * lym + ph[ym1]) - lh0) + ((dtg * lyp + ph[yp1]) - lh0) +
                              ((dtg * ql[1] + hm) - lh0) + ((dtg * ql[3] + hp) - lh0)) *
                             inv_h2;
            const T p0 = psi_prime_t(c);
            const T lap_psi = ((psi_prime_t(cxm) - p0) + (psi_prime_t(cxp) - p0) + (psi_prime_t(cym) - p0) +
                               (psi_prime_t(cyp) - p0) + (psi_prime_t(qc[1]) - p0) + (psi_prime_t(qc[3]) - p0)) *
                              inv_h2;
            const T A_lr[3] = {kap * fourth(pl[xm2], lxm, lr, lxp, pl[xp2]),
                               kap * fourth(pl[ym2], lym, lr, lyp, pl[yp2]),
                               kap * fourth(ql[0], ql[1], lr, ql[3], ql[4])};
            const T A_C = kap * (fourth(pc[xm2], cxm, c, cxp, pc[xp2]) + fourth(pc[ym2], cym, c, cyp, pc[yp2]) +
                                 fourth(qc[0], qc[1], c, qc[3], qc[4]));
            const T ppp = (T(3) * c - T(3)) * c + T(0.5);
            lamC_out[e] = lamC_in[e] - adt * mob * ((A_lr[0] + A_lr[1]) + A_lr[2]) + ppp * mob * lap_lh;
            lamHp_out[e] = dtr * lr;
            adj_dots({lh0, lr, T(0.5) * A_lr[0], T(0.5) * A_lr[1], T(0.5) * A_lr[2]}, {lap_psi, A_C, s0[e], s1[e], s2[e]}, d1,
                     d2);
#pragma unroll
            for (int m = 0; m < 4; ++m) {
                qc[m] = qc[m + 1];
                ql[m] = ql[m + 1];
            }
            hm = hc;
            hc = hp;
        }
        dm = d1 - a.alpha * a.dt * d2;
    }
    __shared__ double ws[kAThreadsX * kAThreadsY / 32];
    for (int o = 16; o > 0; o >>= 1) dm += __shfl_xor_sync(0xffffffffu, dm, o);
    const int tid = threadIdx.y * kAThreadsX + threadIdx.x;
    if ((tid & 31) == 0) ws[tid >> 5] = dm;
    __syncthreads();
    if (tid == 0) {
        double t = 0.0;
        for (int w = 0; w < kAThreadsX * kAThreadsY / 32; ++w) t += ws[w];
        partials[((int64_t)blockIdx.z * gridDim.y + blockIdx.y) * gridDim.x + blockIdx.x] = t;
    }
}

__global__ void adj_accumulate(const double* partials, int64_t n, double* acc) {
    __shared__ double ws[8];
    double t = 0.0;
    for (int64_t b = threadIdx.x; b < n; b += blockDim.x) t += partials[b];
    for (int o = 16; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
    if ((threadIdx.x & 31) == 0) ws[threadIdx.x >> 5] = t;
    __syncthreads();
    if (threadIdx.x == 0) {
        double s = 0.0;
        for (int w = 0; w < (int)(blockDim.x >> 5); ++w) s += ws[w];
        *acc += s;
    }
}

size_t a256(size_t x) { return (x + 255) / 256 * 256; }

struct AdjLayout {
    size_t field, nck, K, total;
};

AdjLayout adj_layout(const ch_handle* h, int64_t nsteps, int64_t K) {
    AdjLayout L;
    L.field = a256((size_t)h->ncell * h->esz);
    L.nck = (size_t)((nsteps + K - 1) / K);
    L.K = (size_t)std::min(K, nsteps);
    const size_t nblocks = (size_t)((h->n[0] + kAThreadsX - 1) / kAThreadsX) *
                           ((h->n[1] + kAThreadsY - 1) / kAThreadsY) * ((h->n[2] + kAdjZ - 1) / kAdjZ);
    L.total = (L.nck + L.K + 15) * L.field + a256(nblocks * sizeof(double)) + 256;
    return L;
}

}  // namespace

extern "C" {

size_t ch_adjoint_workspace_bytes(const ch_handle* h, int64_t nsteps, int64_t ckpt_every) {
    if (!h || nsteps < 1 || ckpt_every < 1 || h->p.advect) return 0;
    return adj_layout(h, nsteps, ckpt_every).total;
}

int ch_step_adjoint(ch_handle* h, const void* C0, int64_t nsteps, int64_t ckpt_every, const void* lam_T, void* lam_0,
                    double* dL_dM, void* work, size_t work_bytes) {
    if (!h) return CH_EINVAL;
    if (h->p.advect) return fail(h, CH_EINVAL, "ch_step_adjoint: only u = 0 (advect = 0) is supported");
    if (h->p.scheme != CH_SCHEME_SPLIT) return fail(h, CH_EINVAL, "ch_step_adjoint: only the split scheme");
    if (h->n[2] < 5) return fail(h, CH_EINVAL, "ch_step_adjoint: needs nz >= 5");
    if (h->p.bc[2] == CH_DIRICHLET) return fail(h, CH_EINVAL, "ch_step_adjoint: Dirichlet walls are not supported");
    if (!C0 || !lam_T || !lam_0 || !dL_dM || !work || nsteps < 1 || ckpt_every < 1 || ((uintptr_t)work % 256))
        return fail(h, CH_EINVAL, "ch_step_adjoint: bad argument");
    const AdjLayout L = adj_layout(h, nsteps, ckpt_every);
    if (work_bytes < L.total) return fail(h, CH_ENOMEM, "ch_step_adjoint: workspace too small");
    const size_t fb = (size_t)h->ncell * h->esz;
    char* w = (char*)work;
    auto field = [&](size_t idx) { return (void*)(w + idx * L.field); };
    size_t q = 0;
    std::vector<void*> ckpt(L.nck), seg(L.K);
    for (auto& p : ckpt) p = field(q++);
    for (auto& p : seg) p = field(q++);
    void* X[3] = {field(q++), field(q++), field(q++)};
    void* Hs[2] = {field(q++), field(q++)};
    void* Htmp = field(q++);
    void* rtmp = field(q++);
    void* lamr = field(q++);
    void* sd[3] = {field(q++), field(q++), field(q++)};
    void* lamC = field(q++);
    void* lamH = field(q++);
    void* lamCn = field(q++);
    void* lamHn = field(q++);
    double* partials = (double*)field(q);
    double* acc = (double*)(w + L.total - 256);
    cudaStream_t st = h->stream;
    const ch_params& p = h->p;
    const int nx = (int)h->n[0], ny = (int)h->n[1], nz = (int)h->n[2];
    dim3 grid((nx + kAThreadsX - 1) / kAThreadsX, (ny + kAThreadsY - 1) / kAThreadsY, (nz + kAdjZ - 1) / kAdjZ);
    dim3 block(kAThreadsX, kAThreadsY);
    const int64_t nblk = (int64_t)grid.x * grid.y * grid.z;
    auto cp = [&](void* dst, const void* src) {
        return cudaMemcpyAsync(dst, src, fb, cudaMemcpyDeviceToDevice, st);
    };
    int rc = CH_OK;
    CHG_CUDA(h, cudaMemsetAsync(acc, 0, sizeof(double), st));

    // forward pass: checkpoints every ckpt_every steps
    CHG_CUDA(h, cp(seg[0], C0));
    for (int64_t s = 0; s < nsteps && rc == CH_OK; ++s) {
        if (s % ckpt_every == 0) CHG_CUDA(h, cp(ckpt[s / ckpt_every], seg[0]));
        if (s + 1 < nsteps) rc = launch_step_any(h, seg[0]);
    }
    if (rc != CH_OK) return rc;

    CHG_CUDA(h, cp(lamC, lam_T));
    const double kappa = p.w * p.cn * p.cn / (p.h * p.h * p.h * p.h);
    for (int64_t m = (int64_t)L.nck - 1; m >= 0 && rc == CH_OK; --m) {
        const int64_t s0 = m * ckpt_every, s1 = std::min(s0 + ckpt_every, nsteps);
        // recompute the segment's step-start states
        CHG_CUDA(h, cp(seg[0], ckpt[m]));
        for (int64_t s = s0 + 1; s < s1 && rc == CH_OK; ++s) {
            CHG_CUDA(h, cp(seg[s - s0], seg[s - s0 - 1]));
            rc = launch_step_any(h, seg[s - s0]);
        }
        for (int64_t s = s1 - 1; s >= s0 && rc == CH_OK; --s) {
            // substep start states X[l] and the explicit terms H of substeps 0, 1
            CHG_CUDA(h, cp(X[0], seg[s - s0]));
            for (int l = 0; l < 2 && rc == CH_OK; ++l) {
                rc = launch_explicit_any(h, l, X[l], l ? Hs[l - 1] : nullptr, Hs[l], rtmp);
                CHG_CUDA(h, cp(X[l + 1], X[l]));
                for (int d = 0; d < 3 && rc == CH_OK; ++d)
                    rc = launch_solve_any(h, l, d, rtmp, rtmp, d == 2 ? X[l + 1] : nullptr);
            }
            CHG_CUDA(h, cudaMemsetAsync(lamH, 0, fb, st));
            for (int l = 2; l >= 0 && rc == CH_OK; --l) {
                rc = launch_explicit_any(h, l, X[l], l ? Hs[l - 1] : nullptr, Htmp, rtmp);
                for (int d = 0; d < 3 && rc == CH_OK; ++d) rc = launch_solve_any(h, l, d, d ? lamr : lamC, lamr, nullptr);
                for (int d = 0; d < 3 && rc == CH_OK; ++d) rc = launch_solve_any(h, l, d, rtmp, sd[d], nullptr);
                if (rc != CH_OK) break;
                if (h->prec == CH_F64) {
                    AdjArgs<double> a{nx, ny, nz, p.bc[0], p.bc[1], p.bc[2], p.dt, kGamma[l], kRho[l], kGamma[l] + kRho[l],
                                      1.0 / p.pe, kappa, 1.0 / (p.h * p.h)};
                    adj_substep<double><<<grid, block, 0, st>>>(
                        (const double*)X[l], (const double*)lamr, (const double*)lamH, (const double*)lamC,
                        (const double*)sd[0], (const double*)sd[1], (const double*)sd[2], (double*)lamCn,
                        (double*)lamHn, partials, a);
                } else {
                    AdjArgs<float> a{nx, ny, nz, p.bc[0], p.bc[1], p.bc[2], p.dt, kGamma[l], kRho[l], kGamma[l] + kRho[l],
                                     1.0 / p.pe, kappa, 1.0 / (p.h * p.h)};
                    adj_substep<float><<<grid, block, 0, st>>>(
                        (const float*)X[l], (const float*)lamr, (const float*)lamH, (const float*)lamC,
                        (const float*)sd[0], (const float*)sd[1], (const float*)sd[2], (float*)lamCn, (float*)lamHn,
                        partials, a);
                }
                CHG_CUDA(h, cudaGetLastError());
                adj_accumulate<<<1, 256, 0, st>>>(partials, nblk, acc);
                CHG_CUDA(h, cudaGetLastError());
                std::swap(lamC, lamCn);
                std::swap(lamH, lamHn);
            }
        }
    }
    if (rc != CH_OK) return rc;
    CHG_CUDA(h, cp(lam_0, lamC));
    CHG_CUDA(h, cudaMemcpyAsync(dL_dM, acc, sizeof(double), cudaMemcpyDeviceToHost, st));
    CHG_CUDA(h, cudaStreamSynchronize(st));
    return CH_OK;
}

}  // extern "C"

// Marching line solver: (I + c A_d) x = r along x-, y- or z-lines (Eqs.
// eq-fac-1..3 of arXiv 2105.01865), one thread per line.
//
// The operator 1 + c [1,-4,6,-4,1] of an unbounded line factors into constant
// two-term recurrences, y_j = r_j - l1 y_{j-1} - l2 y_{j-2} going up and
// x_j = y_j / u0 - l1 x_{j+1} - l2 x_{j+2} going down (march_factors in
// line_tables.h).  A bounded line is the unbounded one on its periodic
// continuation, or on its mirror image about the wall faces (negated for
// Dirichlet walls), so every row uses the same three constants: no tables, no
// wall rows, no Woodbury correction.  Both recurrences forget where they
// started: kb blocks of B rows after a start from zero, what is left of it is
// below 2^-36 (FP32) or 2^-64 (FP64) of the solution, under its rounding by
// 2^12 and 2^11.  So the upward pass starts kb blocks before the line, on
// ghost rows, and the downward pass of each block of B rows starts kb blocks
// above it.  Operators that decay more slowly (over kMarchMaxReach rows) and lines
// no longer than their kb blocks keep the scan solvers of ch_kernels.cuh and
// ch_cols2.cuh; between the forms that take a line, line_rule.h chooses.
//
// A warp streams its lines through a ring of shared-memory blocks: block b is
// being swept upward while blocks b + 1 .. b + D are in flight (cp.async) and
// block b - kb, complete, is swept downward and written out.  Each row is
// read once and written once, and warps share nothing, so a warp needs no
// barrier wider than itself.  Ghost rows past the line's end come from a copy
// of the rows they mirror (`save`), taken before the in-place results
// overwrite them.
//
// What bounds it: on large boxes memory.  On 1024 x 1024 x 512 (FP32) the x-,
// y- and z-solves take 663, 648 and 1060 us, 97, 99 and 91 % of the copy rate
// over 8, 8 and 12 bytes a cell; the scans they replace took 1280, 1420 and
// 1390, since they ran every row four times and held an SM for one tile's
// load, solve and store in turn.  On small boxes the chain of one warp, hence
// the second form below.
#pragma once

#include <type_traits>

#include "ch_kernels.cuh"
#include "line_rule.h"

namespace chg {

template <typename T>
struct MarchCoef {
    T nl1, nl2, dinv;  // -l1, -l2, 1/u0
    int n;             // rows of a line
    int bc;            // CH_PERIODIC, CH_NOFLUX or CH_DIRICHLET
    int reach;         // restart distance in rows (a multiple of 8)
    int kb;            // and in blocks of B rows (>= 1)
};

// V adjacent lines of one thread
template <typename T, int V>
struct LV;
template <typename T>
struct LV<T, 1> {
    T a;
    static __device__ __forceinline__ LV ld(const T* p) { return {*p}; }
    __device__ __forceinline__ void st(T* p) const { *p = a; }
    static __device__ __forceinline__ LV zero() { return {T(0)}; }
    __device__ __forceinline__ LV neg() const { return {-a}; }
    __device__ __forceinline__ bool finite() const { return isfinite(a); }
};
template <>
struct LV<float, 2> {
    float2 a;
    static __device__ __forceinline__ LV ld(const float* p) { return {*reinterpret_cast<const float2*>(p)}; }
    __device__ __forceinline__ void st(float* p) const { *reinterpret_cast<float2*>(p) = a; }
    static __device__ __forceinline__ LV zero() { return {make_float2(0.f, 0.f)}; }
    __device__ __forceinline__ LV neg() const { return {make_float2(-a.x, -a.y)}; }
    __device__ __forceinline__ bool finite() const { return isfinite(a.x) && isfinite(a.y); }
};
template <typename T>
__device__ __forceinline__ LV<T, 1> lfma(T c, LV<T, 1> x, LV<T, 1> y) { return {fmadd(c, x.a, y.a)}; }
__device__ __forceinline__ LV<float, 2> lfma(float c, LV<float, 2> x, LV<float, 2> y) {
    return {__ffma2_rn(make_float2(c, c), x.a, y.a)};
}
template <typename T>
__device__ __forceinline__ LV<T, 1> lmul(T c, LV<T, 1> x) { return {fmul(c, x.a)}; }
__device__ __forceinline__ LV<float, 2> lmul(float c, LV<float, 2> x) { return {__fmul2_rn(make_float2(c, c), x.a)}; }
template <typename T>
__device__ __forceinline__ LV<T, 1> ladd(LV<T, 1> x, LV<T, 1> y) { return {x.a + y.a}; }
__device__ __forceinline__ LV<float, 2> ladd(LV<float, 2> x, LV<float, 2> y) { return {__fadd2_rn(x.a, y.a)}; }

// cp.async of N elements (4, 8 or 16 bytes)
template <typename T, int N>
__device__ __forceinline__ void march_copy(T* smem, const T* gmem) {
    constexpr int kBytes = N * (int)sizeof(T);
    if constexpr (kBytes == 16) {
        cp_async_16(smem, gmem);
    } else {
        const unsigned sa = (unsigned)__cvta_generic_to_shared(smem);
        asm volatile("cp.async.ca.shared.global [%0], [%1], %2;\n" ::"r"(sa), "l"(gmem), "n"(kBytes) : "memory");
    }
}

// f(i, row i) for rows 0 .. rows - 1 at p, p + step, ...: 8 rows are loaded
// while the 8 before them are worked on.  f may store to shared memory (to
// rows already read); loads written out like this are issued ahead of its
// stores, where a plain loop would wait out the load latency on every row.
// ROWS: rows as a constant (a multiple of 8), the loop written out, or 0.
template <typename L, int ROWS, typename T, typename F>
__device__ __forceinline__ void march_rows(const T* p, int step, int rows, F&& f) {
    auto ld8 = [&](int i, L (&v)[8]) {
#pragma unroll
        for (int q = 0; q < 8; ++q) v[q] = L::ld(p + (i + q) * step);
    };
    auto f8 = [&](int i, L (&v)[8]) {
#pragma unroll
        for (int q = 0; q < 8; ++q) f(i + q, v[q]);
    };
    if constexpr (ROWS > 0) {
        L v[2][8];
        ld8(0, v[0]);
#pragma unroll
        for (int i = 0; i < ROWS; i += 8) {
            if (i + 8 < ROWS) ld8(i + 8, v[(i / 8 + 1) & 1]);
            f8(i, v[(i / 8) & 1]);
        }
    } else {
        int i = 0;
        if (rows >= 8) {
            L v[8], u[8];
            ld8(0, v);
#pragma unroll 1
            for (;;) {
                const bool m1 = i + 16 <= rows, m2 = i + 24 <= rows;
                if (m1) ld8(i + 8, u);
                f8(i, v);
                i += 8;
                if (!m1) break;
                if (m2) ld8(i + 8, v);
                f8(i, u);
                i += 8;
                if (!m2) break;
            }
        }
#pragma unroll 1
        for (; i < rows; ++i) f(i, L::ld(p + i * step));
    }
}
// The same along a contiguous line, 8 elements as 16-byte accesses; rows a
// multiple of 8, p 16-byte aligned.  f works on 8 values; Down: from the top.
template <bool Down, int ROWS, typename T, typename F>
__device__ __forceinline__ void march_line(const T* p, int rows, F&& f) {
    constexpr int VEC = 16 / (int)sizeof(T);
    const int nr = ROWS > 0 ? ROWS : rows;
    auto at = [&](int i) { return Down ? nr - 8 - i : i; };
    auto ld8 = [&](int i, T (&v)[8]) {
#pragma unroll
        for (int e = 0; e < 8; e += VEC) vld<T, VEC>(p + at(i) + e, *reinterpret_cast<T(*)[VEC]>(&v[e]));
    };
    if constexpr (ROWS > 0) {
        T v[2][8];
        ld8(0, v[0]);
#pragma unroll
        for (int i = 0; i < ROWS; i += 8) {
            if (i + 8 < ROWS) ld8(i + 8, v[(i / 8 + 1) & 1]);
            f(at(i), v[(i / 8) & 1]);
        }
    } else {
        if (rows <= 0) return;
        T v[8], u[8];
        ld8(0, v);
#pragma unroll 1
        for (int i = 0;;) {
            const bool m1 = i + 8 < rows, m2 = i + 16 < rows;
            if (m1) ld8(i + 8, u);
            f(at(i), v);
            if (!m1) break;
            if (m2) ld8(i + 16, v);
            f(at(i + 8), u);
            i += 16;
            if (!m2) break;
        }
    }
}

// Bytes of shared memory of one warp: kb + 1 + D ring blocks and kb of `save`.
template <typename T, int V>
constexpr size_t march_yz_bytes(int kb) {
    using S = MarchShape<T>;
    return (size_t)(2 * kb + 1 + S::D) * S::B * 32 * V * sizeof(T);
}
// x: a block holds 32 lines of B columns, each padded by 16 bytes
template <typename T>
constexpr size_t march_x_bytes(int kb) {
    using S = MarchShape<T>;
    return (size_t)((kb + 1 + S::D) * (S::B + 16 / (int)sizeof(T)) + kb * S::B + 16 / (int)sizeof(T)) * 32 * sizeof(T);
}

// Strided lines (y, z): the warp's 32 V lines are adjacent columns, nc of them
// inside the field; src, dst and Cf point at the first column's row 0, rows
// are ls apart.  dst may be src.  VL: elements per copy (16 bytes where every
// row of the field is 16-byte aligned, else the thread's own V columns, with
// nc a multiple of it).  UPD: Cf += x in place of dst = x.
template <typename T, int V, int VL, bool UPD>
__device__ __forceinline__ void march_yz(const T* src, T* dst, T* Cf, int nc, int64_t ls, const MarchCoef<T>& k, T* sm,
                                         unsigned int* status) {
    using L = LV<T, V>;
    constexpr int B = MarchShape<T>::B, D = MarchShape<T>::D;
    constexpr int CW = 32 * V, SLOT = B * CW;
    const int lane = threadIdx.x & 31;
    const int n = k.n, kb = k.kb, S = kb + 1 + D, cap = kb * B;
    const bool per = k.bc == CH_PERIODIC;
    T* save = sm + S * SLOT + V * lane;
    // copies: CPR of VL elements make a row, a warp copies RPI rows at once,
    // a block in B / RPI; this lane's column and first row
    constexpr int CPR = CW / VL, RPI = 32 / CPR;
    const int c0 = (lane % CPR) * VL, r0 = lane / CPR;
    const int nb = 2 * kb + (n + B - 1) / B;
    // ring positions (element offsets) of the blocks being loaded, swept upward
    // and written out
    const int ring = S * SLOT;
    auto next = [&](int o) { return o + SLOT == ring ? 0 : o + SLOT; };
    auto prev = [&](int o) { return o == 0 ? ring - SLOT : o - SLOT; };
    int o_load = 0, o_up = 0, o_out = 0;

    auto load = [&](int b) {
        if (b < nb) {
            const int c = c0, r = r0;
            const int j0 = (b - kb) * B;  // first row of the block
            T* s = sm + o_load + r * CW + c;
            if (c < nc) {
                if (j0 >= 0 || per) {
                    const T* g = src + (int64_t)(j0 + r + (j0 < 0 ? n : 0)) * ls + c;
                    if (j0 + B <= n) {
#pragma unroll 8
                        for (int i = 0; i < B; i += RPI) march_copy<T, VL>(s + i * CW, g + i * ls);
                    } else {
                        for (int i = 0; i + r < n - j0; i += RPI) march_copy<T, VL>(s + i * CW, g + i * ls);
                    }
                } else {
                    for (int i = 0; i < B; i += RPI) march_copy<T, VL>(s + i * CW, src + (-1 - j0 - r - i) * ls + c);
                }
            }
        }
        o_load = next(o_load);
        cp_async_commit();
    };
    L y1 = L::zero(), y2 = L::zero();
    // upward over rows i0 .. i1 - 1 of a block's slot s, the right-hand sides
    // read from in; Save: and kept at sv, sv + step, ...; Neg: negated
    auto sweep = [&](auto rows_c, auto save_c, auto neg_c, const T* in, T* s, T* sv, int step, int rows) {
        constexpr bool Save = decltype(save_c)::value, Neg = decltype(neg_c)::value;
        march_rows<L, decltype(rows_c)::value>(in, CW, rows, [&](int i, L v) {
            if constexpr (Save) v.st(sv + i * step);
            if constexpr (Neg) v = v.neg();
            const L y = lfma(k.nl1, y1, lfma(k.nl2, y2, v));
            y2 = y1;
            y1 = y;
            lmul(k.dinv, y).st(s + i * CW);
        });
    };
    using All = std::integral_constant<int, B>;
    using Some = std::integral_constant<int, 0>;
    using No = std::false_type;
    using Yes = std::true_type;
    auto up = [&](int b) {
        const int j0 = (b - kb) * B;
        T* s = sm + o_up + V * lane;
        if (j0 < 0 && k.bc == CH_DIRICHLET) return sweep(Some{}, No{}, Yes{}, s, s, s, 0, B);
        if (per && j0 >= 0 && j0 < cap) return sweep(Some{}, Yes{}, No{}, s, s, save + j0 * CW, CW, B);
        if (j0 < 0 || j0 + B <= (per ? n : n - cap)) return sweep(All{}, No{}, No{}, s, s, s, 0, B);
        // the line's last rows, then their continuation out of `save`
        int i = 0;
        if (per) {
            i = max(0, min(B, n - j0));
            sweep(Some{}, No{}, No{}, s, s, s, 0, i);
        } else {
            i = max(0, n - cap - j0);
            sweep(Some{}, No{}, No{}, s, s, s, 0, i);
            const int e = max(0, min(B, n - j0)) - i;
            if (e > 0) {
                sweep(Some{}, Yes{}, No{}, s + i * CW, s + i * CW, save + (n - 1 - j0 - i) * CW, -CW, e);
                i += e;
            }
        }
        const int e = max(0, min(B, n + cap - j0) - i);
        const T* g = save + (j0 + i - n) * CW;
        if (k.bc == CH_DIRICHLET) sweep(Some{}, No{}, Yes{}, g, s + i * CW, s, 0, e);
        else sweep(Some{}, No{}, No{}, g, s + i * CW, s, 0, e);
        for (i += e; i < B; ++i) L::zero().st(s + i * CW);
    };
    bool bad = false;
    L check = L::zero();  // 0 x C summed: not a number once a C is not finite
    for (int b = 0; b < D; ++b) load(b);
    for (int b = 0; b < nb; ++b) {
        __syncwarp();  // the ring slot of block b + D has been read
        load(b + D);
        // the block that is complete after this one's upward sweep, and its C (FP64: 64
        // rows, 424 bytes of which spill)
        const int t = b - kb, rows = min(B, n - (t - kb) * B);
        const int64_t row0 = (int64_t)((t - kb) * B) * ls;
        L cv[UPD ? B : 1];
        const bool whole = UPD && rows == B && nc == CW;
        if (whole && t >= kb) {
            const T* g = Cf + row0 + V * lane;
#pragma unroll
            for (int i = 0; i < B; ++i, g += ls) cv[i] = L::ld(g);
        }
        cp_async_wait<D>();
        __syncwarp();  // block b, copied by all lanes
        up(b);
        if (t >= kb) {
            L x1 = L::zero(), x2 = L::zero();
            auto down = [&](L z) {
                const L x = lfma(k.nl1, x1, lfma(k.nl2, x2, z));
                x2 = x1;
                x1 = x;
            };
            int o = o_up;
            for (int w = b; w > t; --w, o = prev(o))
                march_rows<L, B>(sm + o + V * lane + (B - 1) * CW, -CW, B, [&](int, L z) { down(z); });
            T* s = sm + o_out;
            if (whole) {
                T* g = Cf + row0 + (B - 1) * ls + V * lane;
                march_rows<L, B>(s + V * lane + (B - 1) * CW, -CW, B, [&](int i, L z) {
                    down(z);
                    const L c = ladd(cv[UPD ? B - 1 - i : 0], x1);
                    check = lfma(T(0), c, check);
                    c.st(g);
                    g -= ls;
                });
            } else {  // in place, then written out as it was copied in
                march_rows<L, B>(s + V * lane + (B - 1) * CW, -CW, B, [&](int i, L z) {
                    down(z);
                    x1.st(s + V * lane + (B - 1 - i) * CW);
                });
                __syncwarp();
                if (c0 < nc) {
                    s += r0 * CW + c0;
                    T* g = (UPD ? Cf : dst) + row0 + r0 * ls + c0;
                    // eight accesses at a time: the loads of C ahead of the stores
#pragma unroll 1
                    for (int i = r0; i < rows; i += 8 * RPI, s += 8 * RPI * CW, g += 8 * RPI * ls) {
                        T d[8][VL], c[UPD ? 8 : 1][VL];
#pragma unroll
                        for (int u = 0; u < 8; ++u)
                            if (i + u * RPI < rows) {
                                vld<T, VL>(s + u * RPI * CW, d[u]);
                                if constexpr (UPD) vld<T, VL>(g + u * RPI * ls, c[u]);
                            }
#pragma unroll
                        for (int u = 0; u < 8; ++u)
                            if (i + u * RPI < rows) {
                                if constexpr (UPD)
#pragma unroll
                                    for (int q = 0; q < VL; ++q) {
                                        d[u][q] += c[u][q];
                                        bad |= !isfinite(d[u][q]);
                                    }
                                vst<T, VL>(g + u * RPI * ls, d[u]);
                            }
                    }
                }
            }
        }
        if (t >= 0) o_out = next(o_out);
        o_up = next(o_up);
    }
    cp_async_wait<0>();
    if (UPD && (bad || !check.finite())) atomicOr(status, 1u);
}

// x-lines: the warp's 32 lines are rows of n contiguous elements, one per
// lane, nl of them inside the field.  A block is 32 lines x B columns, line l
// at l (B + pad) with a 16-byte pad, so that the lanes' 16-byte accesses to a
// column group are free of bank conflicts; copies and write-back run along
// the lines.  vec: the lines are 16-byte aligned (n a multiple of VEC).
template <typename T>
__device__ __forceinline__ void march_x(const T* src, T* dst, int nl, const MarchCoef<T>& k, T* sm, bool vec) {
    constexpr int B = MarchShape<T>::B, D = MarchShape<T>::D, VEC = 16 / (int)sizeof(T);
    constexpr int P = B + VEC, SLOT = 32 * P, CPL = B / VEC;
    const int lane = threadIdx.x & 31;
    const int n = k.n, kb = k.kb, S = kb + 1 + D, cap = kb * B;
    const bool per = k.bc == CH_PERIODIC;
    T* save = sm + S * SLOT + lane * (cap + VEC);
    const int nb = 2 * kb + (n + B - 1) / B;
    const int ring = S * SLOT;
    auto next = [&](int o) { return o + SLOT == ring ? 0 : o + SLOT; };
    auto prev = [&](int o) { return o == 0 ? ring - SLOT : o - SLOT; };
    int o_load = 0, o_up = 0, o_out = 0;
    // copies along the lines: this lane's first line and its column in a block
    constexpr int LPI = 32 / CPL;  // lines a warp copies at once
    const int l0 = lane / CPL, c0 = (lane % CPL) * VEC;
    const int64_t first = (int64_t)l0 * n + c0, lstep = (int64_t)LPI * n;

    auto load = [&](int b) {
        if (b < nb) {
            const int j0 = (b - kb) * B;
            T* s = sm + o_load;
            if (vec && (j0 >= 0 || per)) {
                const T* g = src + first + j0 + (j0 < 0 ? n : 0);
                s += l0 * P + c0;
                if (nl == 32 && j0 + B <= n) {
#pragma unroll
                    for (int i = 0; i < CPL; ++i) march_copy<T, VEC>(s + i * LPI * P, g + i * lstep);
                } else if (j0 + c0 < n) {
                    for (int i = 0; i * LPI + l0 < nl; ++i) march_copy<T, VEC>(s + i * LPI * P, g + i * lstep);
                }
            } else {
                for (int c = lane; c < B; c += 32) {
                    const int j = j0 + c;
                    if (j < n) {
                        const T* g = src + (j >= 0 ? j : per ? j + n : -1 - j);
#pragma unroll 4
                        for (int l = 0; l < nl; ++l) march_copy<T, 1>(s + l * P + c, g + (int64_t)l * n);
                    }
                }
            }
        }
        o_load = next(o_load);
        cp_async_commit();
    };
    T y1 = T(0), y2 = T(0);
    auto row = [&](T v) {
        const T y = fmadd(k.nl1, y1, fmadd(k.nl2, y2, v));
        y2 = y1;
        y1 = y;
        return fmul(k.dinv, y);
    };
    auto put8 = [&](T* p, T (&v)[8]) {
#pragma unroll
        for (int e = 0; e < 8; e += VEC) vst<T, VEC>(p + e, *reinterpret_cast<T(*)[VEC]>(&v[e]));
    };
    // upward over a whole block, 16 bytes an access
    auto sweep = [&](auto save_c, const T* in, T* s, T* sv) {
        march_line<false, B>(in, B, [&](int i, T (&v)[8]) {
            if constexpr (decltype(save_c)::value) put8(sv + i, v);
#pragma unroll
            for (int q = 0; q < 8; ++q) v[q] = row(v[q]);
            put8(s + i, v);
        });
    };
    auto up = [&](int b) {
        const int j0 = (b - kb) * B;
        T* s = sm + o_up + lane * P;
        if (j0 + B <= (per || j0 < 0 ? n : n - cap)) {
            if (per && j0 >= 0 && j0 < cap) sweep(std::true_type{}, s, s, save + j0);
            else sweep(std::false_type{}, s, s, s);
        } else if (vec && j0 >= n && j0 + B <= n + cap) {
            sweep(std::false_type{}, save + (j0 - n), s, s);
        } else {  // the line's last columns, then their continuation out of `save`
#pragma unroll 4
            for (int i = 0; i < B; ++i) {
                const int j = j0 + i;
                T v = T(0);
                if (j < n) {
                    v = s[i];
                    if (!per && j >= n - cap) save[n - 1 - j] = v;
                } else if (j < n + cap) {
                    v = save[j - n];
                }
                s[i] = row(v);
            }
        }
    };
    for (int b = 0; b < D; ++b) load(b);
    for (int b = 0; b < nb; ++b) {
        __syncwarp();  // the ring slot of block b + D has been read
        load(b + D);
        cp_async_wait<D>();
        __syncwarp();  // block b, copied by all lanes
        up(b);
        const int t = b - kb;
        if (t >= kb) {
            T x1 = T(0), x2 = T(0);
            auto down = [&](T z) {
                const T x = fmadd(k.nl1, x1, fmadd(k.nl2, x2, z));
                x2 = x1;
                x1 = x;
                return x;
            };
            int o = o_up;
            for (int w = b; w > t; --w, o = prev(o))
                march_line<true, B>(sm + o + lane * P, B, [&](int, T (&v)[8]) {
#pragma unroll
                    for (int q = 7; q >= 0; --q) down(v[q]);
                });
            T* own = sm + o_out + lane * P;
            march_line<true, B>(own, B, [&](int i, T (&v)[8]) {
#pragma unroll
                for (int q = 7; q >= 0; --q) v[q] = down(v[q]);
                put8(own + i, v);
            });
            __syncwarp();  // the block's results, written along the lines by all lanes
            const int j0 = (t - kb) * B;
            const T* s = sm + o_out;
            if (vec) {
                T* g = dst + first + j0;
                s += l0 * P + c0;
                T v[VEC];
                if (nl == 32 && j0 + B <= n) {
#pragma unroll
                    for (int i = 0; i < CPL; ++i) {
                        vld<T, VEC>(s + i * LPI * P, v);
                        vst<T, VEC>(g + i * lstep, v);
                    }
                } else if (j0 + c0 < n) {
                    for (int i = 0; i * LPI + l0 < nl; ++i) {
                        vld<T, VEC>(s + i * LPI * P, v);
                        vst<T, VEC>(g + i * lstep, v);
                    }
                }
            } else {
                for (int c = lane; c < B; c += 32)
                    if (j0 + c < n) {
#pragma unroll 4
                        for (int l = 0; l < nl; ++l) dst[(int64_t)l * n + j0 + c] = s[l * P + c];
                    }
            }
        }
        if (t >= 0) o_out = next(o_out);
        o_up = next(o_up);
    }
    cp_async_wait<0>();
}

// One warp per CTA and group of 32 V columns: xg column groups of ncol columns
// per outer index (z-lines pass the whole plane as one row of columns).
template <typename T, int V, int VL, bool UPD>
__global__ void __launch_bounds__(32)
ch_march_yz(const T* src, T* dst, T* Cf, int ncol, int xg, int64_t outer_stride, int64_t line_stride, MarchCoef<T> k,
            unsigned int* status) {
    extern __shared__ __align__(16) unsigned char march_smem[];
    pdl_wait();
    pdl_launch_dependents();
    const int g = blockIdx.x % xg, c0 = g * 32 * V;
    const int64_t base = (int64_t)(blockIdx.x / xg) * outer_stride + c0;
    march_yz<T, V, VL, UPD>(src + base, dst + base, UPD ? Cf + base : nullptr, min(32 * V, ncol - c0), line_stride, k,
                            reinterpret_cast<T*>(march_smem), status);
}

template <typename T>
__global__ void __launch_bounds__(32)
ch_march_x(const T* src, T* dst, int64_t nlines, MarchCoef<T> k) {
    extern __shared__ __align__(16) unsigned char march_smem[];
    pdl_wait();
    pdl_launch_dependents();
    const int64_t l0 = (int64_t)blockIdx.x * 32;
    march_x<T>(src + l0 * k.n, dst + l0 * k.n, (int)min((int64_t)32, nlines - l0), k, reinterpret_cast<T*>(march_smem),
               k.n % (16 / (int)sizeof(T)) == 0);
}

// ---------------------------------------------------------------------------
// Whole lines in shared memory: the same recurrences with every line cut into
// chunks of R rows, one warp each, that all start `reach` rows early.  A CTA
// holds 32 lines; warp w sweeps rows wR - reach .. wR + R - 1 upward, keeps its
// own R in registers, publishes them after a barrier, and sweeps downward
// from `reach` rows above.  The chunks cover the line and the `reach` ghost
// rows past its end.  This form has many more warps in flight than the
// streaming one and chains of only reach + R rows, for boxes too small to
// fill the chip with one warp per 32 lines.  Needs reach <= n.
// ---------------------------------------------------------------------------
// Row of the line that row j of its continuation copies, -n <= j < 2n.
__device__ __forceinline__ int tile_row(int j, int n, bool per) {
    return j < 0 ? (per ? j + n : -1 - j) : j >= n ? (per ? j - n : 2 * n - 1 - j) : j;
}

template <typename T, int R, int VL, bool UPD>
__device__ __forceinline__ void tile_yz(const T* src, T* dst, T* Cf, int nc, int64_t ls, const MarchCoef<T>& k, T* s,
                                        int warps, unsigned int* status) {
    const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5, n = k.n, reach = k.reach;
    const bool per = k.bc == CH_PERIODIC, valid = lane < nc;
    const int a = w * R, rows = min(R, n - a);  // own rows inside the line (<= 0: ghost rows only)
    constexpr int CPR = 32 / VL;
    const int c = (tid % CPR) * VL;
    if (c < nc)
        for (int j = tid / CPR; j < n; j += warps * VL) march_copy<T, VL>(s + j * 32 + c, src + j * ls + c);
    cp_async_commit();
    cp_async_wait<0>();
    __syncthreads();
    T* sl = s + lane;
    T y1 = T(0), y2 = T(0), z[R];
    auto row = [&](T v) {
        const T y = fmadd(k.nl1, y1, fmadd(k.nl2, y2, v));
        y2 = y1;
        y1 = y;
        return y;
    };
    if (a - reach >= 0 && a + R <= n) {
        march_rows<LV<T, 1>, 0>(sl + (a - reach) * 32, 32, reach, [&](int, LV<T, 1> v) { row(v.a); });
        const T* p = sl + a * 32;
#pragma unroll
        for (int i = 0; i < R; ++i) z[i] = p[i * 32];
#pragma unroll
        for (int i = 0; i < R; ++i) z[i] = fmul(k.dinv, row(z[i]));
    } else {
        const bool diri = k.bc == CH_DIRICHLET;
#pragma unroll 1
        for (int j0 = a - reach; j0 < a; j0 += 8) {
            T v[8];
#pragma unroll
            for (int q = 0; q < 8; ++q) v[q] = sl[tile_row(j0 + q, n, per) * 32];
#pragma unroll
            for (int q = 0; q < 8; ++q) row(diri && (j0 + q < 0 || j0 + q >= n) ? -v[q] : v[q]);
        }
#pragma unroll
        for (int i = 0; i < R; ++i) {
            const int j = a + i;
            z[i] = T(0);
            if (j < n + reach) {
                const T v = sl[tile_row(j, n, per) * 32];
                z[i] = fmul(k.dinv, row(diri && j >= n ? -v : v));
            }
        }
    }
    __syncthreads();  // the right-hand sides have been read
#pragma unroll
    for (int i = 0; i < R; ++i) sl[(a + i) * 32] = z[i];
    __syncthreads();
    if (rows <= 0) return;
    y1 = y2 = T(0);
    const int top = min(a + R + reach, warps * R);  // rows past the ghosts hold zeros
    T* out = (UPD ? Cf : dst) + a * ls + lane;
    // with UPD a thread's registers hold the rows of C, loaded ahead of the
    // sweeps, and the upward results come back out of shared memory
    T cv[UPD ? R : 1];
    if constexpr (UPD) {
#pragma unroll
        for (int i = 0; i < R; ++i)
            if (valid && i < rows) cv[i] = out[i * ls];
    }
    march_rows<LV<T, 1>, 0>(sl + (top - 1) * 32, -32, top - a - R, [&](int, LV<T, 1> v) { row(v.a); });
    if constexpr (UPD) {
        bool bad = false;
        march_rows<LV<T, 1>, R>(sl + (a + R - 1) * 32, -32, R, [&](int i, LV<T, 1> v) {
            const T c = cv[R - 1 - i] + row(v.a);
            if (valid && R - 1 - i < rows) {
                bad |= !isfinite(c);
                out[(R - 1 - i) * ls] = c;
            }
        });
        if (bad) atomicOr(status, 1u);
    } else {
#pragma unroll
        for (int i = R - 1; i >= 0; --i) {
            const T x = row(z[i]);
            if (valid && i < rows) out[i * ls] = x;
        }
    }
}

template <typename T, int R>
__device__ __forceinline__ void tile_x(const T* src, T* dst, int nl, const MarchCoef<T>& k, T* s, int warps) {
    constexpr int VEC = 16 / (int)sizeof(T);
    const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5, n = k.n, reach = k.reach;
    const int P = tile_x_pitch<T, R>(warps);
    const bool per = k.bc == CH_PERIODIC, vec = n % VEC == 0;
    const int a = w * R, rows = min(R, n - a);
    for (int l = w; l < nl; l += warps) {
        const T* g = src + (int64_t)l * n;
        if (vec)
            for (int j = lane * VEC; j < n; j += 32 * VEC) march_copy<T, VEC>(s + l * P + j, g + j);
        else
            for (int j = lane; j < n; j += 32) march_copy<T, 1>(s + l * P + j, g + j);
    }
    cp_async_commit();
    cp_async_wait<0>();
    __syncthreads();
    T* sl = s + lane * P;
    T y1 = T(0), y2 = T(0), z[R];
    auto row = [&](T v) {
        const T y = fmadd(k.nl1, y1, fmadd(k.nl2, y2, v));
        y2 = y1;
        y1 = y;
        return y;
    };
    if (a - reach >= 0 && a + R <= n) {
        march_line<false, 0>(sl + a - reach, reach, [&](int, T (&v)[8]) {
#pragma unroll
            for (int q = 0; q < 8; ++q) row(v[q]);
        });
#pragma unroll
        for (int i = 0; i < R; i += VEC) vld<T, VEC>(sl + a + i, *reinterpret_cast<T(*)[VEC]>(&z[i]));
#pragma unroll
        for (int i = 0; i < R; ++i) z[i] = fmul(k.dinv, row(z[i]));
    } else {
#pragma unroll 1
        for (int j0 = a - reach; j0 < a; j0 += 8) {
            T v[8];
#pragma unroll
            for (int q = 0; q < 8; ++q) v[q] = sl[tile_row(j0 + q, n, per)];
#pragma unroll
            for (int q = 0; q < 8; ++q) row(v[q]);
        }
#pragma unroll
        for (int i = 0; i < R; ++i) {
            z[i] = T(0);
            if (a + i < n + reach) z[i] = fmul(k.dinv, row(sl[tile_row(a + i, n, per)]));
        }
    }
    __syncthreads();  // the right-hand sides have been read
#pragma unroll
    for (int i = 0; i < R; i += VEC) vst<T, VEC>(sl + a + i, *reinterpret_cast<T(*)[VEC]>(&z[i]));
    __syncthreads();
    if (rows > 0) {
        y1 = y2 = T(0);
        // past the ghosts: zeros
        march_line<true, 0>(sl + a + R, min(reach, (warps - 1) * R - a), [&](int, T (&v)[8]) {
#pragma unroll
            for (int q = 7; q >= 0; --q) row(v[q]);
        });
#pragma unroll
        for (int i = R - 1; i >= 0; --i) z[i] = row(z[i]);
    }
    __syncthreads();  // the upward results have been read
    if (rows > 0) {
#pragma unroll
        for (int i = 0; i < R; i += VEC) vst<T, VEC>(sl + a + i, *reinterpret_cast<T(*)[VEC]>(&z[i]));
    }
    __syncthreads();
    for (int l = w; l < nl; l += warps) {
        T* g = dst + (int64_t)l * n;
        if (vec) {
            for (int j = lane * VEC; j < n; j += 32 * VEC) {
                T v[VEC];
                vld<T, VEC>(s + l * P + j, v);
                vst<T, VEC>(g + j, v);
            }
        } else {
            for (int j = lane; j < n; j += 32) g[j] = s[l * P + j];
        }
    }
}

template <typename T, int R, int VL, bool UPD>
__global__ void __launch_bounds__(tile_max_warps<R>() * 32)
ch_tile_yz(const T* src, T* dst, T* Cf, int ncol, int xg, int64_t outer_stride, int64_t line_stride, MarchCoef<T> k,
           unsigned int* status) {
    extern __shared__ __align__(16) unsigned char march_smem[];
    pdl_wait();
    pdl_launch_dependents();
    const int g = blockIdx.x % xg, c0 = g * 32;
    const int64_t base = (int64_t)(blockIdx.x / xg) * outer_stride + c0;
    tile_yz<T, R, VL, UPD>(src + base, dst + base, UPD ? Cf + base : nullptr, min(32, ncol - c0), line_stride, k,
                           reinterpret_cast<T*>(march_smem), blockDim.x >> 5, status);
}

template <typename T, int R>
__global__ void __launch_bounds__(tile_max_warps<R>() * 32)
ch_tile_x(const T* src, T* dst, int64_t nlines, MarchCoef<T> k) {
    extern __shared__ __align__(16) unsigned char march_smem[];
    pdl_wait();
    pdl_launch_dependents();
    const int64_t l0 = (int64_t)blockIdx.x * 32;
    tile_x<T, R>(src + l0 * k.n, dst + l0 * k.n, (int)min((int64_t)32, nlines - l0), k,
                 reinterpret_cast<T*>(march_smem), blockDim.x >> 5);
}

}  // namespace chg

// Which form solves the lines of a direction: the scan solvers of ch_kernels.cuh
// and ch_cols2.cuh, or a form of ch_march.cuh (a warp of 16, 32 or 64 rows of a
// line in shared memory, or a warp that streams whole lines).
//
// No threshold on one size serves: the scans run the padded line (32 M rows)
// four times, with a correction of periodic lines and in fewer columns at once on
// odd rows; the others pay `reach` rows of restart up and down for every chunk or
// block, which a slowly decaying operator can make longer than the line itself.
// So each form's time is estimated and the least taken:
//   us = t0 + sqrt((row x rows in sequence)^2 + (work x rows in all / SM)^2 + (mem x copy time)^2)
// (the scans have no third term).  The constants are least-squares fits to 2958
// solves timed in every form (50 boxes of 64 x 64 x 1 to 1024 x 1024 x 128, odd and
// even rows, periodic and walled lines of 20 to 1024 rows, every restart distance);
// nine in ten estimates are within 15 % (FP32) and 20 % (FP64).  The form taken is on
// average 2 % slower than the fastest; it is over 5 % slower than the scans in 18 of
// the solves, 25 % at most (80-row walled lines, 25 against 21 us).  Thresholds on
// groups and length, tried before, were slower than the scans in 460, up to 4.9 times.
#pragma once

#include <cmath>
#include <cstddef>
#include <cstdint>

#ifdef __CUDACC__
#define CHG_HD __host__ __device__
#else
#define CHG_HD
#endif

namespace chg {

constexpr size_t kMaxSmem = 227 * 1024;  // dynamic shared memory per CTA (sm_103a)
constexpr int kMarchMaxReach = 96;  // rows

template <typename T>
struct MarchShape {  // rows per block, blocks in flight
    static constexpr int B = sizeof(T) == 4 ? 32 : 64;
    // FP32, 1 and 3 blocks in flight: x 697 and 682 us against 675, z 1083 and
    // 1092 against 1060 on 1024 x 1024 x 512
    static constexpr int D = sizeof(T) == 4 ? 2 : 1;
};
template <typename T>
CHG_HD constexpr int march_kb(int reach) { return (reach + MarchShape<T>::B - 1) / MarchShape<T>::B; }
template <typename T>
CHG_HD constexpr int march_max_kb() { return march_kb<T>(kMarchMaxReach); }

// Most warps of a CTA: what leaves a thread room for its R rows (and R of C).
template <int R>
CHG_HD constexpr int tile_max_warps() { return R <= 16 ? 20 : R <= 32 ? 16 : 8; }
template <int R>
CHG_HD constexpr int tile_warps(int n, int reach) { return (n + reach + R - 1) / R; }
template <typename T, int R>
CHG_HD constexpr size_t tile_yz_bytes(int warps) { return (size_t)warps * R * 32 * sizeof(T); }
// x: the pitch keeps 16-byte accesses of adjacent lines free of bank conflicts
template <typename T, int R>
CHG_HD constexpr int tile_x_pitch(int warps) { return (warps * R + 31) / 32 * 32 + 16 / (int)sizeof(T); }
template <typename T, int R>
CHG_HD constexpr size_t tile_x_bytes(int warps) { return (size_t)tile_x_pitch<T, R>(warps) * 32 * sizeof(T); }

enum LineForm { kLineScan, kLineTile16, kLineTile32, kLineTile64, kLineMarch };

struct LineBox {
    int64_t n[3];
    int dir;
    bool periodic;  // along dir
    int reach;      // restart distance (0: the operator decays too slowly)
};

// Whether a form takes the lines at all: none is shorter than its restart, and
// a tile's warps and shared memory suffice.
template <typename T, int R>
bool tile_fits(const LineBox& b) {
    const int n = (int)b.n[b.dir], warps = tile_warps<R>(n, b.reach);
    return b.reach && b.reach <= n && warps <= tile_max_warps<R>() && tile_yz_bytes<T, R>(warps) <= kMaxSmem &&
           tile_x_bytes<T, R>(warps) <= kMaxSmem;
}
template <typename T>
bool march_fits(const LineBox& b) {
    return b.reach && b.n[b.dir] > march_kb<T>(b.reach) * MarchShape<T>::B;
}

// Groups of 32 lines
inline int64_t line_groups(const LineBox& b) {
    return b.dir == 0 ? (b.n[1] * b.n[2] + 31) / 32 : b.dir == 1 ? (b.n[0] + 31) / 32 * b.n[2] : (b.n[0] * b.n[1] + 31) / 32;
}

struct ScanCost {
    double t0, row, walled, even, odd;  // walled lines, nx = 2 mod 4 and odd: factors on the work
    double work[6];                     // of 32-line groups, for M = 1, 2, 4, .. 32 rows a lane
};
struct MarchCost {
    double t0, row, work, mem;
};

template <typename T>
double scan_us(const LineBox& b) {
    static constexpr ScanCost k[2][3] = {
        {{5.7, 0.19, 0.70, 1.44, 1.70, {1.19, 1.49, 1.88, 3.41, 6.93, 14.1}},
         {7.9, 0.27, 0.77, 1.06, 1.76, {0.43, 0.76, 1.58, 4.16, 6.55, 14.4}},
         {8.0, 0.26, 0.78, 1.06, 1.86, {0.46, 1.14, 2.07, 5.23, 7.52, 22.5}}},
        {{15.5, 0.85, 0.80, 1.0, 1.0, {20.6, 23.4, 36.1, 58.0, 89.4, 189.0}},
         {5.4, 7.65, 0.85, 1.0, 1.0, {11.2, 16.1, 27.9, 66.4, 179.0, 390.0}},
         {9.3, 10.4, 0.86, 1.06, 1.06, {11.6, 17.5, 30.1, 74.5, 221.0, 480.0}}}};
    const ScanCost& c = k[sizeof(T) == 8][b.dir];
    int m = 0;
    while ((32 << m) < b.n[b.dir]) ++m;
    const double per_sm = (double)line_groups(b) / 152.0;
    const double align = b.n[0] % 4 == 0 ? 1.0 : b.n[0] % 2 == 0 ? c.even : c.odd;
    // over 512 rows (M = 32) other kernels, with no longer a sequence
    return c.t0 + std::hypot(c.row * (m < 5 ? 1 << m : 16), per_sm * c.work[m] * (b.periodic ? 1.0 : c.walled) * align);
}

template <typename T>
double march_us(const LineBox& b, LineForm f) {
    // by form, x and y or z (which also reads and writes C)
    static constexpr MarchCost f32[4][2] = {{{6.5, 0.055, 0.0029, 1.43}, {6.5, 0.058, 0.0033, 1.37}},
                                            {{7.6, 0.044, 0.0034, 1.35}, {7.1, 0.064, 0.0038, 1.48}},
                                            {{8.0, 0.0063, 0.00168, 0.33}, {8.3, 0.0081, 0.0019, 0.94}},
                                            {{8.5, 0.0104, 0.0027, 0.0}, {9.1, 0.022, 0.0031, 1.42}}};
    static constexpr MarchCost f64[4][2] = {{{5.7, 0.24, 0.036, 6.4}, {5.1, 0.25, 0.0375, 6.2}},
                                            {{5.2, 0.23, 0.042, 6.6}, {6.2, 0.25, 0.046, 5.8}},
                                            {{1.4, 0.09, 0.0335, 7.3}, {0.0, 0.11, 0.047, 3.7}},
                                            {{8.9, 0.09, 0.038, 6.4}, {0.0, 0.11, 0.047, 3.7}}};
    const int z = b.dir == 2, n = (int)b.n[b.dir];
    const int64_t row = z ? b.n[0] * b.n[1] : b.n[0];  // columns of a row of lines: its alignment
    const bool aligned = row * sizeof(T) % 16 == 0;
    const MarchCost& c = sizeof(T) == 8 ? f64[f == kLineTile32 ? 0 : f == kLineTile64 ? 1 : aligned ? 2 : 3][z]
                                        : f32[f == kLineTile16 ? 0 : f == kLineTile32 ? 1 : aligned ? 2 : 3][z];
    double seq, all;  // rows in sequence, and in all of a line
    if (f == kLineMarch) {
        const int B = MarchShape<T>::B, kb = march_kb<T>(b.reach), nb = (n + B - 1) / B;
        seq = all = (double)(2 * kb + nb) * B + (double)nb * (kb + 1) * B;
    } else {
        const int R = f == kLineTile16 ? 16 : f == kLineTile32 ? 32 : 64;
        seq = b.reach + R;
        all = seq * ((n + b.reach + R - 1) / R);
    }
    const double groups = (double)line_groups(b);
    const double copy = groups * 32.0 * n * sizeof(T) * (z ? 3 : 2) / 6.69e6;  // us at 6.69 TB/s
    const double w = c.work * all * groups / 152.0;
    return c.t0 + std::sqrt(c.row * seq * c.row * seq + w * w + c.mem * copy * c.mem * copy);
}

template <typename T>
LineForm choose_line_form(const LineBox& b) {
    // FP64 x-lines of a plane, in a few warps: the fit is too high there (18 us in the
    // scan, 29 in a tile, for 256 lines of 256 rows)
    if (sizeof(T) == 8 && b.dir == 0 && line_groups(b) <= 16) return kLineScan;
    LineForm best = kLineScan;
    double least = 0.9 * scan_us<T>(b);  // the estimates' spread: leave the scans for a clear gain
    auto consider = [&](LineForm f, bool fits) {
        const double t = fits ? march_us<T>(b, f) : least;
        if (t < least) {
            least = t;
            best = f;
        }
    };
    if (sizeof(T) == 4) consider(kLineTile16, tile_fits<T, 16>(b));
    consider(kLineTile32, tile_fits<T, 32>(b));
    if (sizeof(T) == 8) consider(kLineTile64, tile_fits<T, 64>(b));
    consider(kLineMarch, march_fits<T>(b));
    return best;
}

}  // namespace chg

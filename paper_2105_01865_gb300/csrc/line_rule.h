// Which form solves the lines of a direction: the scan solvers of ch_kernels.cuh
// and ch_cols2.cuh, or a form of ch_march.cuh (a warp of 16, 32 or 64 rows of a
// line in shared memory, or a warp that streams whole lines).
//
// No threshold on one size serves: the scans run the padded line (32 M rows)
// four times, with a correction of periodic lines and in fewer columns at once on
// odd rows; the others pay `reach` rows of restart up and down for every chunk or
// block, which a slowly decaying operator can make longer than the line itself.
// So each form's time is estimated and the least taken:
//   us = t0 + the 4-norm of (row x rows in sequence, work x rows in all / SM, mem x copy time)
// (the scans have no third term).  The constants are those that lose least by the
// choice over 14538 solves timed in every form, back to back (216 boxes of 8^3 to
// 1024 x 1024 x 512, planes among them, odd and even rows, periodic and walled lines,
// restarts of 8 to 96 rows); as times of one solve they are rough.  The form taken is on
// average 0.4 (FP32) and 0.9 % (FP64) slower than the fastest, and over 10 % slower than
// the scans in 58 of the solves, 44 % at most; most of these take 4 to 15 us, where a
// launch moves in steps of 2 us.  Thresholds on groups and length were slower than the
// scans by up to 4.9 times.
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
    bool copied;    // the right-hand sides are not where the solution goes
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

inline double norm4(double a, double b, double c) { return std::sqrt(std::sqrt(a * a * a * a + b * b * b * b + c * c * c * c)); }

struct ScanCost {
    double t0[2], row;  // t0 of periodic and of walled lines
    // factors on the work: walled lines where nx is a multiple of 4 and elsewhere;
    // nx a multiple of 4, of 2 alone, odd
    double walled[2], align[3];
    double work[6];  // of 32-line groups, for M = 1, 2, 4, .. 32 rows a lane
};
struct MarchCost {
    double t0, row, work, mem;
};

template <typename T>
double scan_us(const LineBox& b) {
    static constexpr ScanCost k[2][3] = {{{{3.05, 4.1}, 0.19, {0.441, 0.566}, {1.0, 0.893, 1.19}, {0.883, 1.49, 2.27, 4.51, 11.9, 30.2}},
                                          {{5.5, 4.11}, 0.628, {0.732, 0.835}, {1.0, 1.2, 1.97}, {0.285, 0.632, 1.5, 5.6, 6.83, 24.0}},
                                          {{4.73, 3.55}, 0.924, {0.766, 0.87}, {1.0, 1.36, 3.11}, {0.308, 0.999, 2.3, 6.31, 11.0, 22.4}}},
                                         {{{11.1, 6.72}, 0.372, {1.01, 0.94}, {1.0, 1.9, 1.15}, {21.9, 30.1, 33.6, 53.4, 74.5, 145.0}},
                                          {{10.4, 4.15}, 6.98, {0.942, 0.963}, {1.0, 0.902, 0.826}, {12.7, 17.2, 36.1, 73.3, 187.0, 177.0}},
                                          {{6.29, 2.87}, 8.61, {0.98, 1.0}, {1.0, 1.01, 0.998}, {13.0, 22.4, 38.2, 73.3, 187.0, 211.0}}}};
    const ScanCost& c = k[sizeof(T) == 8][b.dir];
    int m = 0;
    while ((32 << m) < b.n[b.dir]) ++m;
    const double per_sm = (double)line_groups(b) / 152.0;
    const int al = b.n[0] % 4 == 0 ? 0 : b.n[0] % 2 == 0 ? 1 : 2;
    const double work = c.work[m] * c.align[al] * (b.periodic ? 1.0 : c.walled[al > 0]);
    // over 512 rows (M = 32) other kernels, with no longer a sequence
    const double t = c.t0[!b.periodic] + norm4(c.row * (m < 5 ? 1 << m : 16), per_sm * work, 0.0);
    // they work in place: a launch to copy the right-hand sides first
    return b.copied ? t + 2.0 + 2.0 * sizeof(T) * b.n[0] * b.n[1] * b.n[2] / 6.69e6 : t;
}

template <typename T>
double march_us(const LineBox& b, LineForm f) {
    // tiles of 16 (FP64: 32) and 32 (64) rows and streams, on rows that are 16-byte
    // aligned and that are not, along x, y and z (which also reads and writes C)
    static constexpr MarchCost k[2][3][2][3] = {
        {{{{4.12, 0.085, 0.00348, 1.51}, {3.49, 0.0694, 0.00487, 0.149}, {2.67, 0.0801, 0.00435, 1.61}},
          {{4.68, 0.0718, 0.00419, 0.0743}, {3.74, 0.0601, 0.00395, 1.48}, {2.45, 0.0733, 0.00582, 1.55}}},
         {{{3.56, 0.102, 0.00417, 1.26}, {0.875, 0.134, 0.00575, 2.81}, {1.56, 0.182, 0.0059, 2.71}},
          {{6.76, 0.0504, 0.00341, 1.11}, {4.99, 0.0753, 0.00385, 1.74}, {3.99, 0.0999, 0.00552, 0.0903}}},
         {{{3.54, 0.00921, 0.00212, 0.0157}, {3.85, 0.00847, 0.00154, 0.0289}, {3.29, 0.0115, 0.00241, 0.0302}},
          {{4.64, 0.021, 0.00255, 0.00989}, {4.18, 0.0108, 0.00246, 0.00957}, {3.38, 0.0336, 0.00492, 0.0101}}}},
        {{{{14.1, 0.129, 0.0393, 5.85}, {0.0, 0.293, 0.0447, 0.185}, {0.00166, 0.329, 0.0458, 3.51}},
          {{0.0, 0.357, 0.0378, 6.57}, {6.11, 0.198, 0.0508, 0.267}, {10.8, 0.0489, 0.0421, 0.296}}},
         {{{17.0, 0.0992, 0.0431, 3.51}, {3.26, 0.206, 0.053, 0.94}, {6.07, 0.216, 0.0561, 0.239}},
          {{6.62, 0.202, 0.0452, 0.243}, {19.0, 0.0107, 0.0529, 0.218}, {4.14, 0.264, 0.0559, 5.95}}},
         {{{13.2, 0.0707, 0.0383, 0.209}, {0.0, 0.104, 0.0447, 0.273}, {0.0, 0.126, 0.054, 0.483}},
          {{11.9, 0.081, 0.0451, 1.06}, {0.0, 0.0907, 0.0456, 12.4}, {0.0, 0.124, 0.0486, 0.196}}}}};
    const int z = b.dir == 2, n = (int)b.n[b.dir];
    const int64_t row = z ? b.n[0] * b.n[1] : b.n[0];  // columns of a row of lines: its alignment
    const bool aligned = row * sizeof(T) % 16 == 0;
    const int form = f == kLineMarch ? 2 : f == (sizeof(T) == 8 ? kLineTile32 : kLineTile16) ? 0 : 1;
    const MarchCost& c = k[sizeof(T) == 8][form][!aligned][b.dir];
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
    return c.t0 + norm4(c.row * seq, c.work * all * groups / 152.0, c.mem * copy);
}

template <typename T>
LineForm choose_line_form(const LineBox& b) {
    LineForm best = kLineScan;
    double least = scan_us<T>(b);
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

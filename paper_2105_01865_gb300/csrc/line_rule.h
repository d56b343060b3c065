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
// choice over 7798 solves timed in every form, back to back (101 boxes of 24^3 to
// 1024 x 512 x 128, planes among them, odd and even rows, periodic and walled lines of 24
// to 1024 rows, seven restart distances); as times of one solve they are rough.  The form
// taken is on average 0.5 (FP32) and 1 % (FP64) slower than the fastest, and over 10 %
// slower than the scans in 25 of the solves, 28 % at most; most of these take 6 to 15 us,
// where a launch moves in steps of 2 us.  Thresholds on groups and length were slower
// than the scans by up to 4.9 times.
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
    double t0, row;
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
    static constexpr ScanCost k[2][3] = {{{1.71, 0.308, {0.491, 0.651}, {1.0, 1.05, 0.993}, {1.36, 2.18, 2.26, 5.03, 14.1, 34.1}},
                                          {3.46, 0.601, {0.366, 0.629}, {1.0, 0.996, 1.5}, {0.479, 1.38, 2.7, 14.5, 13.3, 14.8}},
                                          {2.93, 0.0155, {0.621, 0.696}, {1.0, 1.1, 2.85}, {0.622, 1.41, 3.26, 8.32, 14.7, 19.6}}},
                                         {{5.88, 0.715, {0.906, 0.766}, {1.0, 1.06, 1.04}, {21.3, 29.8, 39.2, 60.7, 74.3, 197.0}},
                                          {9.23, 5.43, {0.738, 0.728}, {1.0, 0.822, 0.956}, {11.2, 20.3, 36.6, 82.1, 212.0, 229.0}},
                                          {0.0578, 9.71, {0.821, 0.927}, {1.0, 1.1, 0.936}, {12.4, 26.5, 43.5, 82.1, 194.0, 268.0}}}};
    const ScanCost& c = k[sizeof(T) == 8][b.dir];
    int m = 0;
    while ((32 << m) < b.n[b.dir]) ++m;
    const double per_sm = (double)line_groups(b) / 152.0;
    const int al = b.n[0] % 4 == 0 ? 0 : b.n[0] % 2 == 0 ? 1 : 2;
    const double work = c.work[m] * c.align[al] * (b.periodic ? 1.0 : c.walled[al > 0]);
    // over 512 rows (M = 32) other kernels, with no longer a sequence
    const double t = c.t0 + norm4(c.row * (m < 5 ? 1 << m : 16), per_sm * work, 0.0);
    // they work in place: a launch to copy the right-hand sides first
    return b.copied ? t + 2.0 + 2.0 * sizeof(T) * b.n[0] * b.n[1] * b.n[2] / 6.69e6 : t;
}

template <typename T>
double march_us(const LineBox& b, LineForm f) {
    // tiles of 16 (FP64: 32) and 32 (64) rows and streams, on rows that are 16-byte
    // aligned and that are not, along x, y and z (which also reads and writes C)
    static constexpr MarchCost k[2][3][2][3] = {
        {{{{2.37, 0.112, 0.00443, 1.57}, {2.74, 0.0595, 0.00508, 0.238}, {2.84, 0.0117, 0.00512, 1.57}},
          {{0.00752, 0.179, 0.00524, 0.0869}, {2.59, 0.057, 0.00469, 1.82}, {0.0293, 0.114, 0.00648, 0.53}}},
         {{{0.351, 0.153, 0.00557, 1.47}, {0.00442, 0.133, 0.00668, 2.81}, {3.55, 0.0973, 0.00644, 2.52}},
          {{5.14, 0.0503, 0.00331, 0.127}, {7.19, 0.0, 0.00422, 1.54}, {0.115, 0.152, 0.00609, 0.219}}},
         {{{0.00631, 0.0135, 0.00273, 0.0343}, {2.5, 0.00934, 0.00156, 0.0601}, {3.48, 0.011, 0.00263, 0.0468}},
          {{8.54, 0.0157, 0.00302, 0.01}, {2.43, 0.0144, 0.00325, 0.00989}, {1.27, 0.0407, 0.00359, 0.01}}}},
        {{{{7.48, 0.215, 0.0422, 7.99}, {0.00181, 0.286, 0.0471, 0.599}, {0.00237, 0.304, 0.0438, 7.54}},
          {{11.8, 0.123, 0.0337, 10.5}, {0.0, 0.322, 0.0548, 0.593}, {0.00365, 0.369, 0.046, 0.572}}},
         {{{10.8, 0.15, 0.0502, 0.532}, {4.59, 0.189, 0.0548, 0.418}, {6.97, 0.187, 0.056, 0.449}},
          {{0.0149, 0.696, 0.00656, 8.52}, {18.0, 0.00159, 0.0529, 0.322}, {0.181, 0.0156, 0.0586, 6.71}}},
         {{{0.00252, 0.0812, 0.0578, 0.837}, {0.0533, 0.101, 0.0481, 2.3}, {0.0544, 0.128, 0.0448, 12.0}},
          {{0.0, 0.0763, 0.0418, 1.23}, {0.0, 0.0879, 0.0454, 12.1}, {2.05, 0.106, 0.0468, 13.4}}}}};
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

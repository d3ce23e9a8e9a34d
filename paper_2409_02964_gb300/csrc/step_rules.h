// step_rules.h -- which step kernel a 2-D lattice runs, and its rows per CTA. Host code
// without CUDA, so the rules can be evaluated for any lattice on any machine.
#pragma once

#include <algorithm>

namespace lbmv {

// CTAs of the FP64 tile kernel cover this many columns.
constexpr int kTile64Cols = 28;

// Row blocks lie on the grid's y axis, which holds at most this many: every automatic height
// keeps within it (a lattice may be 2^31 rows high, and tiles of 8 rows end at 524280).
constexpr int kMaxGridY = 65535;

struct StepShape {
    int nx, ny;
    int gridx;         // CTAs in x of the marching kernel
    int resident;      // marching CTAs resident on the device
    int nsm;
    int kernel;        // the marching kernel (1 to 5)
    int sbytes;        // bytes of a stored population
    int strip_rows;    // rows asked for, 0 = automatic
    bool solid;        // lattice with solid cells
    bool auto_kernel;  // created without asking for a kernel
    bool wall_y;       // walls in y
};

struct TileShape {
    int rows;   // output rows per CTA, 0 = the lattice marches
    bool big;   // the 12-warp instance
};

inline int row_blocks(int ny, int rows) { return (int)(((long long)ny + rows - 1) / rows); }

// Rows per strip (CTA): strip_rows, or automatic. A strip of H rows steps through H + 6
// (kernel 5: 0.9 us a row with one warp or eight per SM), so few waves of tall strips cost
// fewer halo rows, while several waves of short ones keep the memory busier and end more
// evenly. Kernel 5 takes the fewest waves w whose strips stay within kWaveRows[w]; FP32
// step on one GB300 in us, strips of 1 / 2 / 3 / 5 waves: 800^2 16.2 / 19.8 / 22.8 / -,
// 1531 x 1024 30.0 / 30.4 / 36.1 / 40, 1800 x 1400 42.4 / 42.1 / 46.3 / 53.7, 2048^2
// 72.2 / 64.9 / 66.4 / 72.6, 3000 x 2500 119 / 105.7 / 104.2 / 110.1, 4001 x 3001
// 185.9 / 165.8 / 164.4 / 164.2 (five waves of at least 16 rows, the rule before: 21.5,
// 36.1, 48.1, 72.9, 110.2, 170.1). Where a wave holds a strip or three of each column, w
// waves' worth of strips rounded down leave the last one far from full; one strip more is
// taken if that ends sooner by whole waves (FP32 in us: 100000 x 30 54.4 / 49.6, 100000 x 600
// 803 / 747, 300000 x 100 392 / 383). With solid cells kernel 5 cuts ten waves of at least 16
// rows: the CTAs next to a solid take several times as long as the others, and shorter
// strips shorten the longest CTA. FP64 on kernel 1: march64_us; with solid cells only where
// 16-row strips are fewer than two per SM and no kernel was asked for (us a step, generic
// strips / march64_us: 39 x 17 262 / 50, 150 x 90 421 / 78, 400 x 300 390 / 205, 838 x 226
// 377 / 266, but 900 x 900 732 / 801). Otherwise (kernels 1 to 4):
// five waves of at least 16 rows.
//
// march64_us: a CTA (128 threads) keeps an SM's FP64 pipe 5/6 busy by itself, 7.8 us a row,
// and two on an SM take 13 us a row; a strip of H rows steps through about H + 4. FP64
// step in us, H = 12 / 16 / 24 / 48: 1024 x 768 380 / 472 / 365 / 406, 2000 x 1500 1317 /
// 1400 / 1383 / 1392. A strip of all rows has fewer halo rows to work on, H + 3 or, between
// walls, H + 2 (36000 x 8: 136 and 123 us at 8 rows, where tiles of 4 take 151 and 144). Beyond
// two CTAs of each row per SM the waves of strips of unequal height overlap and the model no
// longer holds: five waves of at least 16 rows (60000 x 20 533 us, tiles 621; walled 524, one
// strip 585).
inline double march64_us(const StepShape& s, int H) {
    const long long ctas = (long long)s.gridx * row_blocks(s.ny, H), slots = 2LL * s.nsm;
    const long long rem = ctas % slots;
    return (H + (H < s.ny ? 4 : (s.wall_y ? 2 : 3))) * (13.0 * (ctas / slots) + (rem == 0 ? 0.0 : (rem <= s.nsm ? 7.8 : 13.0)));
}

inline int strip_height(const StepShape& s) {
    static const int kWaveRows[4] = {24, 36, 40, 44};
    if (s.strip_rows > 0) return std::min(s.strip_rows, s.ny);
    const int least = row_blocks(s.ny, kMaxGridY);
    auto rows = [&](int waves) {
        const int nstrips = std::max(1, waves * s.resident / s.gridx);
        return row_blocks(s.ny, nstrips);
    };
    int H;
    if (s.kernel == 5 && !s.solid) {
        int w = 1;
        while (w < 5 && rows(w) > kWaveRows[w - 1]) ++w;
        H = rows(w);
        auto row_times = [&](int h) {
            const long long ctas = (long long)s.gridx * row_blocks(s.ny, h);
            return (ctas + s.resident - 1) / s.resident * (h + 6);
        };
        const int one_more = row_blocks(s.ny, std::max(1, w * s.resident / s.gridx) + 1);
        if (row_times(one_more) < row_times(H)) H = one_more;
    } else if (s.sbytes == 8 && s.gridx <= 2 * s.nsm &&
               (!s.solid || (s.auto_kernel && (long long)s.gridx * row_blocks(s.ny, 16) < 2LL * s.nsm))) {
        H = least;
        for (int k = least + 1; k <= std::min(s.ny, std::max(128, least)); ++k)
            if (march64_us(s, k) < march64_us(s, H)) H = k;
    } else {
        const int waves = (s.solid && s.kernel == 5) ? 10 : 5;
        const int nstrips = std::max(1, (waves * s.resident + s.gridx - 1) / s.gridx);
        H = std::max(row_blocks(s.ny, nstrips), 16);
    }
    return std::min(std::max(H, least), s.ny);
}

// The tile kernel (vanse_tile.cuh) instead of kernel 5, for lattices that did not ask for
// a kernel or a strip height: small ones, where a strip's serial rows are the step's time,
// and those with solid cells up to 4.5 M cells (FP16 / BF16 4 M), whose marching strips are as
// slow as their slowest row. Beyond, a lattice whose solid cells lie together marches most of
// its strips on the solid-free path, quicker than tiles (us a step, tiles / marching, one
// block of solid cells: 1531 x 1024 FP32 44.9 / 93.8, 2048^2 110 / 129, 2500^2 157 / 148,
// 4096^2 406 / 302, FP16 1600^2 84 / 103, 2048^2 135 / 131; with scattered ones as well 2500^2
// FP32 188 / 228, 4096^2 488 / 590: the host does not know which it has).
// Rows per CTA and instance: R = 4 without spills while all CTAs fit at once (two per
// SM), R = 4 of the 80-register instance while three per SM hold them, else R = 8. Without
// solid cells up to two waves of the last (512^2 9.7 us against 11.1 for the marching
// kernel in strips of 4 rows, 640^2 12.8 against 11.9).
inline TileShape tile_shape(const StepShape& s) {
    auto ctas = [&](int R) { return (long long)s.gridx * row_blocks(s.ny, R); };
    const TileShape march{0, false};
    if (!s.solid && ctas(8) > 4LL * s.nsm) return march;
    if (s.solid && (double)s.nx * s.ny > (s.sbytes == 4 ? 4.5e6 : 4.0e6)) return march;
    const int rows = ctas(4) <= 3LL * s.nsm ? 4 : 8;
    if (row_blocks(s.ny, rows) > kMaxGridY) return march;
    return TileShape{rows, ctas(4) > 2LL * s.nsm};
}

// Whether a step of a lattice with solid cells that may run as tiles does: a step with a force
// field, drag or a moving void fraction (general) takes the longer forms in every tile, while
// most marching strips gain nothing from their absence, so the line lies lower: 3 M cells (us a
// step, tiles / marching, one block of solid cells, force field: FP32 1800 x 1600 118.5 / 117.0,
// 2000 x 1900 156 / 148, 2100^2 177 / 160, BF16 2000 x 1500 126 / 125, 2000 x 1900 158 / 144;
// scattered ones as well FP32 2000 x 1900 289 / 315, 2100^2 moving 332 / 304).
inline bool solid_tiles_pay(const StepShape& s, bool general) { return !general || (double)s.nx * s.ny <= 3.0e6; }

// The FP64 tile kernel instead of kernel 1 where it is quicker: rows per CTA by the FP64
// pipe time of the busiest SM, CTAs per SM times kUs[R] (measured on 2000 x 1500; the same
// figure predicts every size within 10 %). FP64 step in us, tiles / kernel 1 at 16 rows:
// 64^2 9.6 / 137 (R = 2), 130 x 71 10 / 144 (R = 3), 256^2 40 / 145 (R = 6), 512^2 133 /
// 246 (R = 8); 1024 x 768 398 / 365 at 24 rows.
inline int tile64_rows(const StepShape& s, int march_rows) {
    static const struct { int rows; double us; } kUs[] = {{1, 4.0}, {2, 5.8}, {3, 7.2}, {4, 8.7}, {6, 13.2}, {8, 16.6}};
    if (s.gridx > 2 * s.nsm && march_rows < s.ny) return 0;
    double best = march64_us(s, march_rows);
    int rows = 0;
    for (const auto& k : kUs) {
        if (row_blocks(s.ny, k.rows) > kMaxGridY) continue;
        const long long ctas = (long long)row_blocks(s.nx, kTile64Cols) * row_blocks(s.ny, k.rows);
        const double us = k.us * (double)((ctas + s.nsm - 1) / s.nsm);
        if (us < best) { best = us; rows = k.rows; }
    }
    return rows;
}

}  // namespace lbmv

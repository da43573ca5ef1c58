// tiles.cuh -- the order in which tiles and pairs are handed out: queue position
// to blocks, on the device and (for the tests) on the host.
#pragma once

#include <cmath>
#include <cstdint>

#include "f64int.cuh"   // PCF_HD

namespace pcfgb {

// Tile queue bands: the default orders take the blocks of one side in bands
// of kTileBand and, inside a band, every block of the other side in turn
// against the band's blocks.  Each PCF of the other side is then staged from
// memory once per band rather than once per block of the first side, which
// cuts the walk's re-reads of the packed input (evicted from L2 by the
// output stream) by about kTileBand.
constexpr int kTileBand = 16;

// Line m of the upper triangle of an N x N matrix that holds entry t, where
// line m has N - m entries and starts at m N - m (m - 1) / 2: with R entries
// from t to the end, L = N - m is the smallest L with L (L + 1) / 2 >= R.  A
// float32 square root places it to within a few lines and integers make it
// exact.  (A float64 square root costs 20 and more float64 operations, each
// 65-77 issue cycles of its sub-partition on GB300.)
PCF_HD int64_t upper_line(int64_t N, int64_t t)
{
    const int64_t R = N * (N + 1) / 2 - t;
    const float r = (float)(uint32_t)((uint64_t)R >> 32) * 4294967296.0f + (float)(uint32_t)R;
    int64_t L = (int64_t)(uint32_t)sqrtf(r + r);
    if (L > N) L = N;
    if (L < 1) L = 1;
    while (L > 1 && (L - 1) * L / 2 >= R) --L;
    while (L * (L + 1) / 2 < R) ++L;
    return N - L;
}

// Tile t of the queue (longest PCFs first) -> (row block bi, column block bj).
// Symmetric (bi <= bj, NB blocks): line m of the triangle holds NB - m tiles
// and starts at tile m NB - m (m - 1) / 2.  Order 1: line m is row block m,
// columns NB - 1 down to m.  Order 0 (default): line m is column block
// NB - 1 - m; the lines are taken in bands of kTileBand columns c1 down to
// c0, and inside a band row blocks c1 down to 0 each take the band's columns
// from c1 down (row c1 - r of the band's top triangle takes r + 1 of them).
PCF_HD void decode_upper_tile(int64_t NB, int64_t t, int order,
                                                  int64_t& bi, int64_t& bj)
{
    auto start = [NB](int64_t m) { return m * NB - m * (m - 1) / 2; };
    const int64_t m = upper_line(NB, t);
    if (order) {
        bi = m;
        bj = NB - 1 - (t - start(m));
        return;
    }
    const int64_t m0 = (m / kTileBand) * kTileBand;                // the band's first line
    const int64_t Bq = NB - m0 < kTileBand ? NB - m0 : kTileBand;  // its columns
    const int64_t c1 = NB - 1 - m0, c0 = c1 - Bq + 1;
    int64_t u = t - start(m0);
    const int64_t tri = Bq * (Bq + 1) / 2;
    if (u < tri) {
        int64_t r = 0;
        while ((r + 1) * (r + 2) / 2 <= u) ++r;
        bi = c1 - r;
        bj = c1 - (u - r * (r + 1) / 2);
    } else {
        u -= tri;
        bi = c0 - 1 - u / Bq;
        bj = c1 - u % Bq;
    }
}

// Cross (nb_r x nb_c blocks): bands of kTileBand row blocks from the last
// down; inside a band, column blocks from the last down, each against the
// band's rows from the last down.
PCF_HD void decode_cross_tile(int64_t NBr, int64_t NBc, int64_t t,
                                                  int64_t& bi, int64_t& bj)
{
    const int64_t band = t / ((int64_t)kTileBand * NBc);
    const int64_t r1 = NBr - 1 - band * kTileBand;
    const int64_t Bq = r1 + 1 < kTileBand ? r1 + 1 : kTileBand;
    const int64_t u = t - band * (int64_t)kTileBand * NBc;
    bj = NBc - 1 - u / Bq;
    bi = r1 - u % Bq;
}

}  // namespace pcfgb

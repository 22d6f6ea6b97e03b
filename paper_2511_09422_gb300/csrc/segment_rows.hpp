// Rows of the inner segments into which a step cuts its lattices: plain host arithmetic.
#pragma once
#include <cmath>

namespace lbk {

// Greatest height of a half-storage lattice whose rows are not whole chunks of 8 values:
// its strips at the x ends are staged lane by lane, and the taller their segments, the
// longer a step waits for the last of them.  F16 with FP32 h, without this limit -> with
// it (us per step): 1037 x 771 80.8 -> 72.4, 859 x 1230 104.2 -> 89.1, 2274 x 926 174 -> 162,
// 1500 x 1300 159.5 -> 151.2; lattices that take no more than 12 rows anyway are the same.
constexpr int RAGGED_ROWS = 12;

// Work items of a batch of lattices at h rows a segment; each(f) calls f(strips, ny) for
// every lattice.  Many small lattices of different heights (below SMALL_ROWS on average)
// fill no rounds of equal items: most of their items are wall bands and last segments of
// fewer rows, so their rows are added up, in items of h + 3 rows.  200 droplets of 48 .. 100
// rows (us per step, by count at 7 rows -> by rows at 13): FP32 155.2 -> 152.8, D2Q5 134.7 ->
// 130.8, F16 195.9 -> 179.5, F16 with FP32 h 197.7 -> 182.5.  Larger lattices are counted: by
// rows, 3 droplets of 100 .. 400 rows took 9 % longer in F16, 40 of 64 .. 300 rows 3 % in FP32.
constexpr int SMALL_ROWS = 128;
template <class Each>
inline long long batch_items(int h, Each each)
{
    long long count = 0, work = 0, lattices = 0, rows = 0;
    int least = 0, most = 0;
    each([&](long long strips, int ny) {
        const int inner = ny >= 5 ? ny - 4 : 0, segments = (inner + h - 1) / h;
        count += strips * (2 + segments);
        work += strips * (inner + 3 * segments + 2 * (2 + 3));
        least = lattices == 0 || ny < least ? ny : least;
        most = lattices == 0 || ny > most ? ny : most;
        lattices++;
        rows += ny;
    });
    return least < most && rows < SMALL_ROWS * lattices ? (work + h + 2) / (h + 3) : count;
}

// The height, at most max_rows, of the lowest estimated step time; items(h) counts the
// work items at height h, for the W warps of the wave.  An item runs h + 3 rows one after
// another (its own, and the fill of the rings).  The warps take the items in rounds of W;
// a row takes longer the more warps share a scheduler (1.45 us with one, 2.1 us with two
// FP32 warps; 1.6, 2.5 and 2.8 us with one, two and three of a half form), and with many
// rounds the last one is only partly filled.
//
// Measured for all heights up to the greatest (us per step, the height taken here first):
//   FP32  64 x 256: 8.7 at 2, 11.4 at 4;   512 x 256: 15.5 at 4, 18.4 at 2;   256^2: 12.6 at 4, 11.3 at 2;
//         512^2: 26.1 at 8, 29.1 at 4;   700^2: 48.9 at 8, 46.0 at 7;   1024^2: 89.7 at 10, 93.5 at 8
//   D2Q5  1037 x 771: 58.6 at 24, 57.2 at 23, 61.5 at 12;   1024^2: 77.8 at 16, 75.5 at 15, 78.6 at 10;
//         3000 x 2000: 389.6 at 22, 378.7 at 24
//   F16   512^2: 26.6 at 6, 30.0 at 3;   1037 x 771: 72.3 at 8, 72.9 at 15;   1024^2: 76.9 at 21, 77.6 at 20, 87.1 at 8;
//         3000 x 2000: 419.6 at 23, 398.4 at 24
//   F16 with FP32 h   700^2: 45.7 at 10;   2048^2: 289.5 at 20, 283.1 at 17
// Of 98 lattices from 64 x 256 to 3000 x 2000, 48 take their best height and 85 are within 5 %
// of it; the farthest are narrow or low ones of little work, such as 256^2 in FP32 (11 %) and
// 140 x 530 in F16 (18.4 at 5, 14.9 at 2).
template <class Items>
inline int best_segment_rows(long long W, bool half, int max_rows, Items items)
{
    int best = 1;
    double least = 0.0;
    for (int h = 1; h <= max_rows; h++) {
        const long long n = items(h);
        const double waves = (double)n / (double)W, rounds = waves <= 8.0 ? std::ceil(waves) : waves + 0.5;
        const long long per_scheduler = ((n < W ? n : W) + 607) / 608;
        const double share = per_scheduler <= 1 ? 1.0 : (!half ? 1.45 : (per_scheduler == 2 ? 1.55 : 1.75));
        const double cost = rounds * (h + 3) * share;
        if (h == 1 || cost < least) {
            least = cost;
            best = h;
        }
    }
    return best;
}

}  // namespace lbk

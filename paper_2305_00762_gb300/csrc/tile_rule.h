// Tile shape of the FP64 form for a grid (host code without CUDA, so that a host
// test can ask it).
//
// The faces of 16 x 15 (511) are two rounds of 256 threads at 128 registers, the
// fastest per cell where there are tiles enough (1024^2 plain: 16 x 16 with 288
// threads 5% slower, 20 x 12 2%, 28 x 8 6%). A grid of few tiles is bound by the
// tiles the busiest SM gets, so a smaller tile that divides the work further wins:
// 16 x 8 with its 280 faces in one round, 8 x 4 where even that leaves SMs idle.
// An SM's first tile costs its latency, each further one its share of the pipes:
// a step takes first + next (k - 1) for k tiles on the busiest SM, k rounded up
// while it is small and the last wave counts. The shape with the smallest is
// taken. The figures (us of a step, four-quadrant flow) were measured with every
// shape on 16 grids of 48^2 .. 512^2 for each instance; fourth order is within
// 3% of the plain one. Loss against the best shape measured, at most: plain and
// fourth order 8% (150^2), viscous 2%, MEG7-cons 7%, viscous MEG7-cons 23% (136^2,
// where the first tile's latency depends on the flow). With the plain figures for
// every instance it was 10%, 29% and 105%. The result does not depend on the shape.
#pragma once

namespace gbr {

struct TileShape {
    int bx, by;
};

inline TileShape fixed_tile_rule(int nx, int ny, int sms, bool cons, bool viscous)
{
    struct Cost {
        double first, next;
    };
    static const Cost cost[4][3] = {
        // 16 x 15, 16 x 8, 8 x 4
        {{121, 65}, {83, 40}, {49, 23}},      // plain (and fourth order)
        {{149, 79}, {100, 46}, {62, 34}},     // viscous
        {{272, 94}, {168, 61}, {112, 39}},    // MEG7-cons
        {{240, 165}, {125, 102}, {110, 90}},  // viscous MEG7-cons (one CTA an SM)
    };
    static const TileShape shape[3] = {{16, 15}, {16, 8}, {8, 4}};
    const Cost* c = cost[(cons ? 2 : 0) + (viscous ? 1 : 0)];
    int best = 0;
    double least = 0.0;
    for (int i = 0; i < 3; ++i) {
        const double tiles = (double)((nx + shape[i].bx - 1) / shape[i].bx) * ((ny + shape[i].by - 1) / shape[i].by);
        const double k = tiles / sms, up = (double)(long long)k;
        const double t = c[i].first + c[i].next * ((k <= 16.0 ? (k > up ? up + 1.0 : up) : k + 0.5) - 1.0);
        if (i == 0 || t < least) {
            best = i;
            least = t;
        }
    }
    return shape[best];
}

}  // namespace gbr

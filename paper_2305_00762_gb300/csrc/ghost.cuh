// Ghost-cell boundary conditions (arXiv:2305.00762, Sec. 3: ghost-cell
// approach) for one padded state; shared by the single-grid and the batched
// ghost kernels.
#pragma once

#include <cuda_runtime.h>

#include "gbr_internal.h"

namespace gbr {

// Source index of ghost coordinate k on an axis of n interior cells, and
// whether the normal / tangential velocity changes sign (kinds: 0 periodic,
// 1 transmissive, 2 no-slip wall, 3 symmetry; custom sides are resolved to
// one of 1-3 before).
__device__ __forceinline__ int ghost_src(int k, int n, int lo, int hi, bool& flip_n, bool& flip_t)
{
    flip_n = false;
    flip_t = false;
    if (k >= 0 && k < n) return k;
    const int bc = k < 0 ? lo : hi;
    if (bc == 0) return k < 0 ? k + n : k - n;  // (n is at least the ghost depth)
    if (bc == 1) return k < 0 ? 0 : n - 1;
    flip_n = true;
    flip_t = (bc == 2);
    return k < 0 ? -1 - k : 2 * n - 1 - k;
}

// Number of ghost cells of a grid: 6 full rows below and above, 6 cells left
// and right of every interior row.
__host__ __device__ __forceinline__ long long ghost_count(const Grid& g)
{
    return 2LL * kGhost * (g.nx + 2 * kGhost) + 2LL * kGhost * g.ny;
}

constexpr int kBcCustom = 4, kBcFixed = 5, kBcHalo = 6;

// Kind of a custom side beside the cell with tangential index k (centre at
// (k + 1/2) h along the side) at time t; for kBcFixed also its state.
__device__ __forceinline__ int side_kind(const SideBC& S, int k, double h, double t, const double*& state)
{
    const bool lo = (k + 0.5) * h < S.s0 + S.speed * t;
    state = lo ? S.qlo : S.qhi;
    return lo ? S.kind_lo : S.kind_hi;
}

// The conservative state of the ghost cell at padded coordinates (gx, gy) of
// the state q, from its interior cells. A corner ghost takes the y image of the
// x image of an interior cell, so the velocity sign flips of both axes compose.
// The ghost rows of a halo side (south / north of one slab of a grid split along
// y) hold the neighbouring slab's interior rows, written before: false for their
// interior columns (the state in memory is the one), and their west / east
// ghosts follow the x rule of their own row, as for an interior row. With custom
// sides (sides != null, boundary time t), a south / north ghost whose side is
// fixed there takes the fixed state; otherwise the source row is found first and
// a west / east side is resolved at that row (a fixed state is then mirrored
// across the south / north side like any x image).
__device__ __forceinline__ bool ghost_value(const Grid& g, const double* q, const int bc[4], int gx, int gy,
                                            const SideBC* sides, double dx, double dy, double t, double (&v)[4])
{
    const int nx = g.nx, ny = g.ny;
    const int j = gx - kGhost, i = gy - kGhost;
    const bool halo_row = (i < 0 && bc[2] == kBcHalo) || (i >= ny && bc[3] == kBcHalo);
    if (halo_row && j >= 0 && j < nx) return false;
    const long long pl = g.plane;
    int ky[2] = {bc[2], bc[3]}, kx[2] = {bc[0], bc[1]};
    if (sides && (i < 0 || i >= ny) && bc[i < 0 ? 2 : 3] == kBcCustom) {
        const double* st;
        const int k = side_kind(sides[i < 0 ? 2 : 3], j, dx, t, st);
        if (k == kBcFixed) {
            for (int m = 0; m < 4; ++m) v[m] = st[m];
            return true;
        }
        ky[i < 0 ? 0 : 1] = k;
    }
    bool fnx, ftx, fny = false, fty = false;
    const int is = halo_row ? i : ghost_src(i, ny, ky[0], ky[1], fny, fty);
    if (sides && (j < 0 || j >= nx) && bc[j < 0 ? 0 : 1] == kBcCustom) {
        const double* st;
        const int k = side_kind(sides[j < 0 ? 0 : 1], is, dy, t, st);
        if (k == kBcFixed) {
            v[0] = st[0];
            v[1] = fty ? -st[1] : st[1];
            v[2] = fny ? -st[2] : st[2];
            v[3] = st[3];
            return true;
        }
        kx[j < 0 ? 0 : 1] = k;
    }
    const int js = ghost_src(j, nx, kx[0], kx[1], fnx, ftx);
    const bool flip_u = fnx != fty;  // x momentum: normal to x faces, tangential to y faces
    const bool flip_v = ftx != fny;
    const long long s = (long long)(is + kGhost) * g.pitch + (js + kGhost);
    const double u = q[s + pl], w = q[s + 2 * pl];
    v[0] = q[s];
    v[1] = flip_u ? -u : u;
    v[2] = flip_v ? -w : w;
    v[3] = q[s + 3 * pl];
    return true;
}

// Fill ghost cell number id (0 <= id < ghost_count) of the padded state q.
__device__ __forceinline__ void fill_ghost(const Grid& g, double* q, const int bc[4], long long id,
                                           const SideBC* sides = nullptr, double dx = 0.0, double dy = 0.0,
                                           double t = 0.0)
{
    const int nx = g.nx, ny = g.ny, W = nx + 2 * kGhost;
    const long long band = (long long)kGhost * W;
    int gx, gy;
    if (id < band) {
        gy = (int)(id / W);
        gx = (int)(id - (long long)gy * W);
    } else if (id < 2 * band) {
        const long long k = id - band;
        gy = ny + kGhost + (int)(k / W);
        gx = (int)(k - (long long)(k / W) * W);
    } else {
        const long long k = id - 2 * band;
        gy = kGhost + (int)(k / (2 * kGhost));
        const int c = (int)(k - (long long)(k / (2 * kGhost)) * (2 * kGhost));
        gx = c < kGhost ? c : nx + c;
    }
    double v[4];
    if (!ghost_value(g, q, bc, gx, gy, sides, dx, dy, t, v)) return;
    const long long d = (long long)gy * g.pitch + gx;
    for (int m = 0; m < 4; ++m) q[d + m * g.plane] = v[m];
}

// The step size formed on the device in mode 2 (Sec. 2.5); the host's otherwise.
__device__ __forceinline__ double step_size(const GhostParams& P)
{
    if (P.mode != 2) return P.dt;
    const double lam = __longlong_as_double((long long)P.ds->lam[P.cur]);
    return fmin(P.cfl / lam, P.dt_max);
}
// The scalars of a step that begins, by one thread (modes 1 and 2): nothing of
// what the step's first stage reads (lam[cur], ts[cur]) is written.
__device__ __forceinline__ void begin_step(const GhostParams& P)
{
    DevScalars* d = P.ds;
    const double dt = step_size(P);
    d->dt = dt;
    d->t += dt;
    d->ts[P.next] = d->ts[P.cur] + dt;
    d->lam[P.next] = 0ull;
}
// Boundary time of a stage: the step's start time ts[cur] plus c_stage dt (dt
// was written by an earlier launch whenever c_stage != 0).
__device__ __forceinline__ double boundary_time(const GhostParams& P)
{
    return P.ds->ts[P.cur] + (P.c_stage != 0.0 ? P.c_stage * P.ds->dt : 0.0);
}

}  // namespace gbr

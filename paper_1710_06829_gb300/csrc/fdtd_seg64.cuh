// Helpers of the FP64 kernels: a thread owns 2 x 2 cells (x, y) of a plane, an even x first, and
// marches z; 16-byte loads and stores; the extended stencil on the four cells with the differences
// that they share formed once.
#pragma once

#include "fdtd_tma.cuh"

namespace fdtd {
namespace seg64 {

struct Quad {
    double v[2][2];   // [y][x]
};

// The 2 x 2 cells of thread t: i, j the first cell (j < 0: none), o its offset in the plane, two: the
// second row is a cell of the grid too; y1: offset of the row that stands in for it (the second row,
// or the first again below a ragged end).
struct Tile {
    int i, j;
    long long o, y1;
    bool two;
};

__host__ __device__ inline long long tiles(const Geom& g) {
    return (long long)(g.nx / 2) * ((g.ny + 1) / 2);
}

__device__ __forceinline__ Tile tile_of(const Geom& g, long long t) {
    Tile r;
    const int half = g.nx / 2;
    r.i = (int)(t % half) * 2;
    r.j = (int)(t / half) * 2;
    if (t >= tiles(g)) {
        r.j = -1;
        return r;
    }
    r.two = r.j + 1 < g.ny;
    r.o = (long long)(r.j + PY) * g.nxp + r.i + PX;
    r.y1 = r.two ? g.nxp : 0;
    return r;
}

__device__ __forceinline__ long long plane_at(const Geom& g, int q) {
    int r = q % g.nz;
    if (r < 0) r += g.nz;
    return (long long)r * g.plane;
}

__device__ __forceinline__ bool nonfinite(double v) {
    return ((unsigned)__double2hiint(v) & 0x7ff00000u) == 0x7ff00000u;
}

__device__ __forceinline__ void ld2(const double* p, double* v) {
    const double2 a = *reinterpret_cast<const double2*>(p);
    v[0] = a.x;
    v[1] = a.y;
}

// two cells (i, i + 1; i even) of row (j, k) and their periodic images
__device__ __forceinline__ void put2(const Geom& g, double* F, int i, int j, int k, const double* v) {
    const double2 a = make_double2(v[0], v[1]);
    double* p = F + pidx(g, i, j, k);
    auto row = [&](double* q) {
        *reinterpret_cast<double2*>(q) = a;
        if (i < PX) *reinterpret_cast<double2*>(q + g.nx) = a;
        if (i >= g.nx - PX) *reinterpret_cast<double2*>(q - g.nx) = a;
    };
    row(p);
    if (j < PY || j >= g.ny - PY)
        for (int my = -PY; my <= PY; ++my) {
            const int jj = j + my * g.ny;
            if (my != 0 && jj >= -PY && jj < g.ny + PY) row(p + (long long)my * g.ny * g.nxp);
        }
}

// F[+x] - F at the four cells; F points at the first one, Y is the row pitch
__device__ __forceinline__ void own_dx(const double* F, long long Y, Quad& d) {
#pragma unroll
    for (int r = 0; r < 2; ++r) {
        double a[2];
        ld2(F + r * Y, a);
        const double b = F[r * Y + 2];
        d.v[r][0] = a[1] - a[0];
        d.v[r][1] = b - a[1];
    }
}

// F[+y] - F
__device__ __forceinline__ void own_dy(const double* F, long long Y, Quad& d) {
    double a[3][2];
#pragma unroll
    for (int r = 0; r < 3; ++r) ld2(F + r * Y, a[r]);
#pragma unroll
    for (int r = 0; r < 2; ++r)
#pragma unroll
        for (int u = 0; u < 2; ++u) d.v[r][u] = a[r + 1][u] - a[r][u];
}

// D*_x (transverse y, then z) at plane p; d0, dp, dm: own x differences of planes p, p+1, p-1
__device__ __forceinline__ void dstar_x(const double* F, long long Y, const Quad& d0, const Quad& dp,
                                        const Quad& dm, double cA, double cD, double cB, double cC,
                                        Quad& out) {
    double lo[2], hi[2];   // x differences of rows y-1, y+2
    {
        double a[2];
        ld2(F - Y, a);
        const double b = F[-Y + 2];
        lo[0] = a[1] - a[0];
        lo[1] = b - a[1];
        ld2(F + 2 * Y, a);
        const double c = F[2 * Y + 2];
        hi[0] = a[1] - a[0];
        hi[1] = c - a[1];
    }
#pragma unroll
    for (int r = 0; r < 2; ++r) {
        const double* q = F + r * Y;
        double mid[2], rt[2];
        ld2(q, mid);
        ld2(q + 2, rt);
        const double lf = q[-1];
#pragma unroll
        for (int u = 0; u < 2; ++u)
            out.v[r][u] = dstar_diff(d0.v[r][u], rt[u], u ? mid[0] : lf, r ? hi[u] : d0.v[1][u],
                                     r ? d0.v[0][u] : lo[u], dp.v[r][u], dm.v[r][u], cA, cD, cB, cC);
    }
}

// D*_y (transverse x, then z) at plane p; d0, dp, dm: own y differences of planes p, p+1, p-1; y3: offset
// of row y+3 (of row y+2 where the second row is not the grid's: row y+3 is then past the ghosts)
__device__ __forceinline__ void dstar_y(const double* F, long long Y, long long y3, const Quad& d0, const Quad& dp,
                                        const Quad& dm, double cA, double cD, double cB, double cC,
                                        Quad& out) {
    double lf[2], rt[2];   // y differences of columns x-1, x+2
#pragma unroll
    for (int r = 0; r < 2; ++r) {
        lf[r] = F[(r + 1) * Y - 1] - F[r * Y - 1];
        rt[r] = F[(r + 1) * Y + 2] - F[r * Y + 2];
    }
#pragma unroll
    for (int r = 0; r < 2; ++r) {
        double up[2], dn[2];
        ld2(F + (r ? y3 : 2 * Y), up);
        ld2(F + (r - 1) * Y, dn);
#pragma unroll
        for (int u = 0; u < 2; ++u)
            out.v[r][u] = dstar_diff(d0.v[r][u], up[u], dn[u], u ? rt[r] : d0.v[r][1],
                                     u ? d0.v[r][0] : lf[r], dp.v[r][u], dm.v[r][u], cA, cD, cB, cC);
    }
}

// D*_z (transverse x, then y) at plane p: F at planes p-1, p, p+1, p+2
__device__ __forceinline__ void dstar_z(const double* Fm, const double* F0, const double* F1,
                                        const double* F2, long long Y, double cA, double cD, double cB,
                                        double cC, Quad& out) {
    Quad d;
    double lf[2], rt[2], lo[2], hi[2];   // z differences at x-1, x+2 (both rows), y-1, y+2
#pragma unroll
    for (int r = 0; r < 2; ++r) {
        double a[2], b[2];
        ld2(F1 + r * Y, a);
        ld2(F0 + r * Y, b);
#pragma unroll
        for (int u = 0; u < 2; ++u) d.v[r][u] = a[u] - b[u];
        lf[r] = F1[r * Y - 1] - F0[r * Y - 1];
        rt[r] = F1[r * Y + 2] - F0[r * Y + 2];
    }
    {
        double a[2], b[2];
        ld2(F1 - Y, a);
        ld2(F0 - Y, b);
#pragma unroll
        for (int u = 0; u < 2; ++u) lo[u] = a[u] - b[u];
        ld2(F1 + 2 * Y, a);
        ld2(F0 + 2 * Y, b);
#pragma unroll
        for (int u = 0; u < 2; ++u) hi[u] = a[u] - b[u];
    }
#pragma unroll
    for (int r = 0; r < 2; ++r) {
        double up[2], dn[2];
        ld2(F2 + r * Y, up);
        ld2(Fm + r * Y, dn);
#pragma unroll
        for (int u = 0; u < 2; ++u)
            out.v[r][u] = dstar_diff(d.v[r][u], up[u], dn[u], u ? rt[r] : d.v[r][1],
                                     u ? d.v[r][0] : lf[r], r ? hi[u] : d.v[1][u],
                                     r ? d.v[0][u] : lo[u], cA, cD, cB, cC);
    }
}

}  // namespace seg64

// Launch of a marching FP64 kernel in blocks of `threads` threads: `columns` blocks of tiles x chunks
// of tz planes, the columns fastest, all on one grid axis (a y axis ends at 65535 chunks).
struct March64 {
    int tz;
    unsigned columns, blocks;
};
March64 march64_grid(const Geom& g, int threads);

}  // namespace fdtd

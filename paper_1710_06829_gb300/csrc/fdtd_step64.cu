// FP64 leapfrog step in two kernels, out of place: B^{n+1/2} from (E^n, B^{n-1/2}), then E^{n+1}.
//
// The FP64 pipe of this part has two lanes an SM (a warp's FP64 instruction takes 64 cycles of its
// scheduler), so FP64 instructions bound the step, by a factor of ten over its memory traffic, and
// everything else is nearly free.  A thread of the Faraday kernel owns 2 x 2 cells (x, y) and
// marches z: the differences of E along each axis that its four cells share, and those that a later
// plane needs again (kept in registers), are formed once, 14 a cell instead of 30; neighbouring
// threads' differences are formed again rather than exchanged, so there is no barrier, and loads
// come from L1.  77 FP64 instructions a cell and step (62 here, 15 in the Ampere kernel), where the
// reference form takes 96.
// Values and rounding order are those of dstar_diff / ampere_comp: bitwise the same fields.
// Us a step, the kernels before (one tiled kernel with barriers where 64 x 8 tiles fit, else the
// reference form) and these: 192 x 128 x 96 717 / 386 (0.164 ns a cell), 100 x 90 x 80 199 / 125,
// 36^3 27 / 18, 60 x 32 x 39 31 / 19, 128^3 638 / 355.  A kernel that shares every difference
// through shared memory (76 instructions, two barriers a plane) took 518 us at 192 x 128 x 96: the pipe
// idles at the barriers.
#include <algorithm>

#include "fdtd_seg64.cuh"

namespace fdtd {
namespace step64 {

using namespace seg64;

constexpr int NT = 128;
// Threads of a Faraday block.  A warp's plane takes 8 us of its scheduler, so a small grid is a
// question of how evenly its warps fall on the SMs: single warps do best (us a step with blocks of
// 128, 64, 32: 60 x 32 x 39 27.8, 22.6, 18.6; 48^3 29.0, 24.5, 24.4; 64^3 52.8, 53.0, 48.0; 192 x 128 x
// 96 384.6, 385.0, 384.8).
constexpr int NF = 32;

// SP: absorbing layers
template <bool SP>
__global__ void __launch_bounds__(NF, 3 * NT / NF)
faraday_kernel(Geom g, Mult<double> m, FieldSet<double> in, FieldSet<double> out,
               const double* __restrict__ spy, const double* __restrict__ spz, int tz,
               unsigned columns) {
    pdl_wait();
    const unsigned chunk = blockIdx.x / columns, column = blockIdx.x - chunk * columns;
    const Tile t = tile_of(g, (long long)column * NF + threadIdx.x);
    const int z0 = (int)chunk * tz, zend = min(z0 + tz, g.nz);
    if (t.j < 0) return;
    const double *Ex = in.c[0] + t.o, *Ey = in.c[1] + t.o, *Ez = in.c[2] + t.o;
    const long long Y = g.nxp, y3 = (t.two ? 3 : 2) * Y;
    // own differences of the planes before and at p, carried along z
    Quad xy_m, xy_0, xz_m, xz_0, yx_m, yx_0, yz_m, yz_0;
    long long om = plane_at(g, z0 - 1), o0 = plane_at(g, z0), o1 = plane_at(g, z0 + 1);
    own_dx(Ey + om, Y, xy_m);
    own_dx(Ey + o0, Y, xy_0);
    own_dx(Ez + om, Y, xz_m);
    own_dx(Ez + o0, Y, xz_0);
    own_dy(Ex + om, Y, yx_m);
    own_dy(Ex + o0, Y, yx_0);
    own_dy(Ez + om, Y, yz_m);
    own_dy(Ez + o0, Y, yz_0);
    for (int p = z0; p < zend; ++p) {
        const long long o2 = plane_at(g, p + 2);
        double f[2] = {1.0, 1.0};
        if (SP) {
            f[0] = spy[t.j] * spz[p];
            f[1] = spy[min(t.j + 1, g.ny - 1)] * spz[p];
        }
        Quad a, b, next;
        auto update = [&](int c, auto&& delta) {   // B_c + delta, written with its images
#pragma unroll
            for (int r = 0; r < 2; ++r) {
                double v[2];
                ld2(in.c[3 + c] + t.o + o0 + r * t.y1, v);
#pragma unroll
                for (int u = 0; u < 2; ++u) {
                    v[u] += delta(r, u);
                    if (SP) v[u] *= f[r];
                }
                if (r == 0 || t.two) put2(g, out.c[3 + c], t.i, t.j + r, p, v);
            }
        };
        // B_x + (D*_z E_y - D*_y E_z)
        dstar_z(Ey + om, Ey + o0, Ey + o1, Ey + o2, Y, m.cA[2], m.cD[2], m.cB[2][0], m.cB[2][1], a);
        own_dy(Ez + o1, Y, next);
        dstar_y(Ez + o0, Y, y3, yz_0, next, yz_m, m.cA[1], m.cD[1], m.cB[1][0], m.cB[1][2], b);
        yz_m = yz_0;
        yz_0 = next;
        update(0, [&](int r, int u) { return a.v[r][u] - b.v[r][u]; });
        // B_y + (D*_x E_z - D*_z E_x)
        own_dx(Ez + o1, Y, next);
        dstar_x(Ez + o0, Y, xz_0, next, xz_m, m.cA[0], m.cD[0], m.cB[0][1], m.cB[0][2], a);
        xz_m = xz_0;
        xz_0 = next;
        dstar_z(Ex + om, Ex + o0, Ex + o1, Ex + o2, Y, m.cA[2], m.cD[2], m.cB[2][0], m.cB[2][1], b);
        update(1, [&](int r, int u) { return a.v[r][u] - b.v[r][u]; });
        // B_z + (D*_y E_x - D*_x E_y)
        own_dy(Ex + o1, Y, next);
        dstar_y(Ex + o0, Y, y3, yx_0, next, yx_m, m.cA[1], m.cD[1], m.cB[1][0], m.cB[1][2], a);
        yx_m = yx_0;
        yx_0 = next;
        own_dx(Ey + o1, Y, next);
        dstar_x(Ey + o0, Y, xy_0, next, xy_m, m.cA[0], m.cD[0], m.cB[0][1], m.cB[0][2], b);
        xy_m = xy_0;
        xy_0 = next;
        update(2, [&](int r, int u) { return a.v[r][u] - b.v[r][u]; });
        om = o0;
        o0 = o1;
        o1 = o2;
    }
    pdl_trigger();
}

// E^{n+1} from E^n (in) and B^{n+1/2} (out's B): two cells of a row a thread, 15 FP64 instructions a
// cell.
template <bool SP>
__global__ void __launch_bounds__(NT)
ampere_kernel(Geom g, Mult<double> m, FieldSet<double> in, FieldSet<double> out,
              const double* __restrict__ spy, const double* __restrict__ spz,
              const double* __restrict__ jyz, const double* jx_row,
              double* __restrict__ h0, double* __restrict__ h1, double* __restrict__ h2,
              int* __restrict__ err) {
    pdl_wait();
    const long long n = (long long)(g.nx / 2) * g.ny * g.nz, Y = g.nxp;
    bool bad = false;
    for (long long t = (long long)blockIdx.x * NT + threadIdx.x; t < n; t += (long long)gridDim.x * NT) {
        const long long r = t / (g.nx / 2);
        const int i = (int)(t - r * (g.nx / 2)) * 2, k = (int)(r / g.ny), j = (int)(r - (long long)k * g.ny);
        const long long o = pidx(g, i, j, k), om = o + plane_at(g, k - 1) - plane_at(g, k);
        double E[3][2], bx[2], by[2], bz[2], bxy[2], bzy[2], bxz[2], byz[2];
#pragma unroll
        for (int c = 0; c < 3; ++c) ld2(in.c[c] + o, E[c]);
        const double *Bx = out.c[3], *By = out.c[4], *Bz = out.c[5];
        ld2(Bx + o, bx);
        ld2(By + o, by);
        ld2(Bz + o, bz);
        ld2(Bx + o - Y, bxy);
        ld2(Bz + o - Y, bzy);
        ld2(Bx + om, bxz);
        ld2(By + om, byz);
        const double byl = By[o - 1], bzl = Bz[o - 1];
        const double f = SP ? spy[j] * spz[k] : 1.0;
#pragma unroll
        for (int u = 0; u < 2; ++u) {
            E[0][u] = ampere_comp(E[0][u], bz[u], bzy[u], by[u], byz[u], m.cE[1], m.cE[2]);
            E[1][u] = ampere_comp(E[1][u], bx[u], bxz[u], bz[u], u ? bz[0] : bzl, m.cE[2], m.cE[0]);
            E[2][u] = ampere_comp(E[2][u], by[u], u ? by[0] : byl, bx[u], bxy[u], m.cE[0], m.cE[1]);
            if (jx_row != nullptr) E[0][u] = fma(-m.dt, (jx_row[i + u] * jyz[j]) * jyz[g.ny + k], E[0][u]);
#pragma unroll
            for (int c = 0; c < 3; ++c) {
                if (SP) E[c][u] *= f;
                bad = bad || nonfinite(E[c][u]);
            }
        }
        double* const h[3] = {h0, h1, h2};
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            put2(g, out.c[c], i, j, k, E[c]);
            if (h0 != nullptr) put2(g, h[c], i, j, k, E[c]);
        }
    }
    pdl_trigger();
    if (bad) atomicOr(err, ERR_FIELD);
}

}  // namespace step64

// Planes a thread takes: the FP64 pipe is the limit, so the scheduler with the most warps decides,
// warps x (planes + the first plane's extra differences, a quarter of a plane's work); a single warp
// takes 1.3 times its share.
static int march64(const Geom& g, int threads) {
    const long long columns = (seg64::tiles(g) + threads - 1) / threads;
    int best = 1;
    double best_cost = -1.0;
    for (int tz = g.nz < 64 ? g.nz : 64; tz >= 1; --tz) {
        const long long blocks = columns * ((g.nz + tz - 1) / tz), per_sm = (blocks + 151) / 152;
        const double warps = (double)((per_sm * (threads / 32) + 3) / 4);   // of the fullest scheduler
        const double cost = (warps > 1.0 ? warps : 1.3) * (tz + 0.25);
        if (best_cost < 0.0 || cost < best_cost) {
            best_cost = cost;
            best = tz;
        }
    }
    return best;
}

March64 march64_grid(const Geom& g, int threads) {
    March64 r;
    r.tz = march64(g, threads);
    r.columns = (unsigned)((seg64::tiles(g) + threads - 1) / threads);
    r.blocks = r.columns * (unsigned)((g.nz + r.tz - 1) / r.tz);
    return r;
}

void launch_step64(const Geom& g, const Mult<double>& m, FieldSet<double> in, FieldSet<double> out,
                   const double* spy, const double* spz, const double* jyz, const double* jx_row,
                   double* hist_E[3], int* err, cudaStream_t st) {
    using namespace step64;
    const March64 r = march64_grid(g, NF);
    launch_pdl(spy ? faraday_kernel<true> : faraday_kernel<false>, dim3(r.blocks), dim3(NF), 0, st, g, m, in,
               out, spy, spz, r.tz, r.columns);
    const long long pairs = (long long)(g.nx / 2) * g.ny * g.nz;
    const unsigned nb = (unsigned)std::min<long long>((pairs + NT - 1) / NT, 1 << 20);
    launch_pdl(spy ? ampere_kernel<true> : ampere_kernel<false>, dim3(nb), dim3(NT), 0, st, g, m, in, out,
               spy, spz, jyz, jx_row, hist_E[0], hist_E[1], hist_E[2], err);
}

}  // namespace fdtd

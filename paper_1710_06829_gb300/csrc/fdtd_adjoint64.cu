// FP64 reverse leapfrog step with the coefficient gradient (derivation in fdtd_adjoint.cu), in place:
//   mu = S (lambda_B + dt G^T S lambda_E) -> lambda_B,  then  lambda_E <- S lambda_E + dt F^T mu
// and the gradient in its transposed form, from the same differences of mu (fdtd_adjoint32f.cu):
// with d(k) = mu[k-a] - mu[k], each DT_a mu that enters lambda_E'_k with sign s adds
//   s E_k (mu[-2a] - mu[+a] - 3 d(0)),  s E_k (d(-b) + d(+b) - 2 d(0)),  s E_k (d(-c) + d(+c) - 2 d(0))
// to the gradients in delta_a, beta_ab and beta_ac, and E^n is read at the own cells only.
//
// FP64 instructions bound it (two lanes an SM, see fdtd_step64.cu): 15 a cell for mu and, with a
// thread's 2 x 2 cells, z march and shared differences, 62 for lambda_E and 24 for the gradient's
// twelve sums; the reference form, which takes brackets of E for the gradient, needs about 260.
// Us a reverse step, the reference form and these kernels: 192 x 128 x 96 989 / 473, 100 x 90 x 80
// 417 / 155, 32^3 68 / 25, 16 x 100 x 100 281 / 61.
#include "fdtd_seg64.cuh"

namespace fdtd {
namespace adj64 {

using namespace seg64;

constexpr int NT = 128;
// of a lambda block: single warps, as in the forward step (us a reverse step with blocks of 128 / 32:
// 60 x 32 x 39 37.3 / 27.1, 64^3 69.5 / 62.4, 192 x 128 x 96 472 / 474)
constexpr int NL = 32;

template <bool SP>
__global__ void __launch_bounds__(NT)
mu_kernel(Geom g, Mult<double> m, FieldSet<double> lam, const double* __restrict__ spy,
          const double* __restrict__ spz) {
    pdl_wait();
    const long long n = (long long)(g.nx / 2) * g.ny * g.nz, Y = g.nxp;
    for (long long t = (long long)blockIdx.x * NT + threadIdx.x; t < n; t += (long long)gridDim.x * NT) {
        const long long q = t / (g.nx / 2);
        const int i = (int)(t - q * (g.nx / 2)) * 2, k = (int)(q / g.ny), j = (int)(q - (long long)k * g.ny);
        const int j1 = j + 1 == g.ny ? 0 : j + 1, k1 = k + 1 == g.nz ? 0 : k + 1;
        const long long o = pidx(g, i, j, k), oz = o + plane_at(g, k + 1) - plane_at(g, k);
        double ex[3], ey[3], ez[3], exy[2], ezy[2], exz[2], eyz[2], b[3][2];
        ld2(lam.c[0] + o, ex);
        ld2(lam.c[1] + o, ey);
        ld2(lam.c[2] + o, ez);
        ey[2] = lam.c[1][o + 2];
        ez[2] = lam.c[2][o + 2];
        ld2(lam.c[0] + o + Y, exy);
        ld2(lam.c[2] + o + Y, ezy);
        ld2(lam.c[0] + oz, exz);
        ld2(lam.c[1] + oz, eyz);
#pragma unroll
        for (int c = 0; c < 3; ++c) ld2(lam.c[3 + c] + o, b[c]);
        double s0 = 1.0, sy = 1.0, sz = 1.0;
        if (SP) {
            s0 = spy[j] * spz[k];
            sy = spy[j1] * spz[k];
            sz = spy[j] * spz[k1];
        }
#pragma unroll
        for (int u = 0; u < 2; ++u) {
            // l_E = S lambda_E at the cell and its +x (same factor), +y, +z neighbours
            const double x0 = SP ? s0 * ex[u] : ex[u], y0 = SP ? s0 * ey[u] : ey[u],
                         z0 = SP ? s0 * ez[u] : ez[u];
            const double yx = SP ? s0 * ey[u + 1] : ey[u + 1], zx = SP ? s0 * ez[u + 1] : ez[u + 1];
            const double xy = SP ? sy * exy[u] : exy[u], zy = SP ? sy * ezy[u] : ezy[u];
            const double xz = SP ? sz * exz[u] : exz[u], yz = SP ? sz * eyz[u] : eyz[u];
            b[0][u] += m.cE[2] * (y0 - yz) - m.cE[1] * (z0 - zy);
            b[1][u] += m.cE[0] * (z0 - zx) - m.cE[2] * (x0 - xz);
            b[2][u] += m.cE[1] * (x0 - xy) - m.cE[0] * (y0 - yx);
            if (SP) {
#pragma unroll
                for (int c = 0; c < 3; ++c) b[c][u] *= s0;
            }
        }
#pragma unroll
        for (int c = 0; c < 3; ++c) put2(g, lam.c[3 + c], i, j, k, b[c]);
    }
    pdl_trigger();
}

// Differences of the transposed stencils at the four cells: G[-a] - G[0]
__device__ __forceinline__ void own_tx(const double* G, long long Y, Quad& d) {
#pragma unroll
    for (int r = 0; r < 2; ++r) {
        double a[2];
        ld2(G + r * Y, a);
        const double b = G[r * Y - 1];
        d.v[r][0] = b - a[0];
        d.v[r][1] = a[0] - a[1];
    }
}

__device__ __forceinline__ void own_ty(const double* G, long long Y, Quad& d) {
    double a[3][2];
#pragma unroll
    for (int r = 0; r < 3; ++r) ld2(G + (r - 1) * Y, a[r]);
#pragma unroll
    for (int r = 0; r < 2; ++r)
#pragma unroll
        for (int u = 0; u < 2; ++u) d.v[r][u] = a[r][u] - a[r + 1][u];
}

// One DT value from its difference d, far pair f = G[-2a] - G[+a] and transverse sums sb, sc; acc += w
// times (f, sb, sc, d)
__device__ __forceinline__ double dt_value(double d, double f, double sb, double sc, double cA,
                                           double cD, double cB, double cC, double w, double* acc) {
    acc[0] = fma(w, f, acc[0]);
    acc[1] = fma(w, sb, acc[1]);
    acc[2] = fma(w, sc, acc[2]);
    acc[3] = fma(w, d, acc[3]);
    return fma(cC, sc, fma(cB, sb, fma(cD, f, cA * d)));
}

// DT_x (transverse y, then z) at plane p; d0, dp, dm: own differences of planes p, p+1, p-1
__device__ __forceinline__ void dt_x(const double* G, long long Y, const Quad& d0, const Quad& dp,
                                     const Quad& dm, double cA, double cD, double cB, double cC,
                                     const Quad& w, double* acc, Quad& out) {
    double lo[2], hi[2], a[2];   // rows y-1, y+2
    ld2(G - Y, a);
    lo[0] = G[-Y - 1] - a[0];
    lo[1] = a[0] - a[1];
    ld2(G + 2 * Y, a);
    hi[0] = G[2 * Y - 1] - a[0];
    hi[1] = a[0] - a[1];
#pragma unroll
    for (int r = 0; r < 2; ++r) {
        const double* q = G + r * Y;
        double lf[2];   // x-2, x-1
        ld2(q - 2, lf);
        const double r1 = q[1], r2 = q[2];
#pragma unroll
        for (int u = 0; u < 2; ++u)
            out.v[r][u] = dt_value(d0.v[r][u], lf[u] - (u ? r2 : r1),
                                   (r ? d0.v[0][u] : lo[u]) + (r ? hi[u] : d0.v[1][u]),
                                   dm.v[r][u] + dp.v[r][u], cA, cD, cB, cC, w.v[r][u], acc);
    }
}

// DT_y (transverse x, then z)
__device__ __forceinline__ void dt_y(const double* G, long long Y, const Quad& d0, const Quad& dp,
                                     const Quad& dm, double cA, double cD, double cB, double cC,
                                     const Quad& w, double* acc, Quad& out) {
#pragma unroll
    for (int r = 0; r < 2; ++r) {
        const double lf = G[(r - 1) * Y - 1] - G[r * Y - 1];
        const double rt = G[(r - 1) * Y + 2] - G[r * Y + 2];
        double dn[2], up[2];   // rows y-2, y+1
        ld2(G + (r - 2) * Y, dn);
        ld2(G + (r + 1) * Y, up);
#pragma unroll
        for (int u = 0; u < 2; ++u)
            out.v[r][u] = dt_value(d0.v[r][u], dn[u] - up[u],
                                   (u ? d0.v[r][0] : lf) + (u ? rt : d0.v[r][1]),
                                   dm.v[r][u] + dp.v[r][u], cA, cD, cB, cC, w.v[r][u], acc);
    }
}

// DT_z (transverse x, then y): G at planes p-2, p-1, p, p+1
__device__ __forceinline__ void dt_z(const double* G2, const double* Gm, const double* G0,
                                     const double* Gp, long long Y, double cA, double cD, double cB,
                                     double cC, const Quad& w, double* acc, Quad& out) {
    Quad d;
    double lf[2], rt[2], lo[2], hi[2], a[2], b[2];
#pragma unroll
    for (int r = 0; r < 2; ++r) {
        ld2(Gm + r * Y, a);
        ld2(G0 + r * Y, b);
#pragma unroll
        for (int u = 0; u < 2; ++u) d.v[r][u] = a[u] - b[u];
        lf[r] = Gm[r * Y - 1] - G0[r * Y - 1];
        rt[r] = Gm[r * Y + 2] - G0[r * Y + 2];
    }
    ld2(Gm - Y, a);
    ld2(G0 - Y, b);
#pragma unroll
    for (int u = 0; u < 2; ++u) lo[u] = a[u] - b[u];
    ld2(Gm + 2 * Y, a);
    ld2(G0 + 2 * Y, b);
#pragma unroll
    for (int u = 0; u < 2; ++u) hi[u] = a[u] - b[u];
#pragma unroll
    for (int r = 0; r < 2; ++r) {
        ld2(G2 + r * Y, a);
        ld2(Gp + r * Y, b);
#pragma unroll
        for (int u = 0; u < 2; ++u)
            out.v[r][u] = dt_value(d.v[r][u], a[u] - b[u],
                                   (u ? d.v[r][0] : lf[r]) + (u ? rt[r] : d.v[r][1]),
                                   (r ? d.v[0][u] : lo[u]) + (r ? hi[u] : d.v[1][u]), cA, cD, cB, cC,
                                   w.v[r][u], acc);
    }
}

// SP: absorbing layers.  partials[block][9] += (delta_a, beta_a,b1, beta_a,b2) for a = x, y, z
template <bool SP>
__global__ void __launch_bounds__(NL, 2 * NT / NL)
lambda_kernel(Geom g, Mult<double> m, FieldSet<double> lam, const double* e_x, const double* e_y,
              const double* e_z, const double* __restrict__ spy, const double* __restrict__ spz,
              double* __restrict__ partials, int tz, unsigned columns) {
    pdl_wait();
    const unsigned chunk = blockIdx.x / columns, column = blockIdx.x - chunk * columns;
    const Tile t = tile_of(g, (long long)column * NL + threadIdx.x);
    const int z0 = (int)chunk * tz, zend = min(z0 + tz, g.nz);
    double acc[3][4];   // per axis: sums of w (far pair, first, second transverse sum, difference)
#pragma unroll
    for (int a = 0; a < 3; ++a)
#pragma unroll
        for (int q = 0; q < 4; ++q) acc[a][q] = 0.0;
    if (t.j >= 0) {
        const double *Mx = lam.c[3] + t.o, *My = lam.c[4] + t.o, *Mz = lam.c[5] + t.o;
        const long long Y = g.nxp;
        Quad zx_m, zx_0, zy_m, zy_0, yx_m, yx_0, xy_m, xy_0;   // mu component, axis; planes p-1, p
        long long o2 = plane_at(g, z0 - 2), om = plane_at(g, z0 - 1), o0 = plane_at(g, z0);
        own_tx(Mz + om, Y, zx_m);
        own_tx(Mz + o0, Y, zx_0);
        own_ty(Mz + om, Y, zy_m);
        own_ty(Mz + o0, Y, zy_0);
        own_tx(My + om, Y, yx_m);
        own_tx(My + o0, Y, yx_0);
        own_ty(Mx + om, Y, xy_m);
        own_ty(Mx + o0, Y, xy_0);
        for (int p = z0; p < zend; ++p) {
            const long long op = plane_at(g, p + 1);
            double f[2] = {1.0, 1.0};
            if (SP) {
                f[0] = spy[t.j] * spz[p];
                f[1] = spy[min(t.j + 1, g.ny - 1)] * spz[p];
            }
            Quad w, nw, a, b, next;
            auto weight = [&](const double* e) {   // E^n at the own cells, zero off the grid
#pragma unroll
                for (int r = 0; r < 2; ++r) {
                    ld2(e + t.o + o0 + r * t.y1, w.v[r]);
#pragma unroll
                    for (int u = 0; u < 2; ++u) {
                        if (r && !t.two) w.v[r][u] = 0.0;
                        nw.v[r][u] = -w.v[r][u];
                    }
                }
            };
            auto update = [&](int c) {   // S lambda_E + (a - b), with its images
#pragma unroll
                for (int r = 0; r < 2; ++r) {
                    if (r && !t.two) break;
                    double v[2];
                    ld2(lam.c[c] + t.o + o0 + r * Y, v);
#pragma unroll
                    for (int u = 0; u < 2; ++u) {
                        const double d = a.v[r][u] - b.v[r][u];
                        v[u] = SP ? fma(f[r], v[u], d) : v[u] + d;
                    }
                    put2(g, lam.c[c], t.i, t.j + r, p, v);
                }
            };
            // lambda_E_x: DT_y mu_z - DT_z mu_y
            weight(e_x);
            own_ty(Mz + op, Y, next);
            dt_y(Mz + o0, Y, zy_0, next, zy_m, m.cA[1], m.cD[1], m.cB[1][0], m.cB[1][2], w, acc[1], a);
            zy_m = zy_0;
            zy_0 = next;
            dt_z(My + o2, My + om, My + o0, My + op, Y, m.cA[2], m.cD[2], m.cB[2][0], m.cB[2][1], nw,
                 acc[2], b);
            update(0);
            // lambda_E_y: DT_z mu_x - DT_x mu_z
            weight(e_y);
            dt_z(Mx + o2, Mx + om, Mx + o0, Mx + op, Y, m.cA[2], m.cD[2], m.cB[2][0], m.cB[2][1], w,
                 acc[2], a);
            own_tx(Mz + op, Y, next);
            dt_x(Mz + o0, Y, zx_0, next, zx_m, m.cA[0], m.cD[0], m.cB[0][1], m.cB[0][2], nw, acc[0], b);
            zx_m = zx_0;
            zx_0 = next;
            update(1);
            // lambda_E_z: DT_x mu_y - DT_y mu_x
            weight(e_z);
            own_tx(My + op, Y, next);
            dt_x(My + o0, Y, yx_0, next, yx_m, m.cA[0], m.cD[0], m.cB[0][1], m.cB[0][2], w, acc[0], a);
            yx_m = yx_0;
            yx_0 = next;
            own_ty(Mx + op, Y, next);
            dt_y(Mx + o0, Y, xy_0, next, xy_m, m.cA[1], m.cD[1], m.cB[1][0], m.cB[1][2], nw, acc[1], b);
            xy_m = xy_0;
            xy_0 = next;
            update(2);
            o2 = om;
            om = o0;
            o0 = op;
        }
    }
    pdl_trigger();
    // the warp's sums: lane 3 q + r adds every third value of quantity q, the first of three the rest
    __shared__ double sm[9][NL + 1];
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        sm[3 * a][threadIdx.x] = fma(-3.0, acc[a][3], acc[a][0]);
        sm[3 * a + 1][threadIdx.x] = fma(-2.0, acc[a][3], acc[a][1]);
        sm[3 * a + 2][threadIdx.x] = fma(-2.0, acc[a][3], acc[a][2]);
    }
    __syncwarp();
    const int l = threadIdx.x, q = l / 3;
    double x = 0.0;
    if (q < 9) {
        for (int k = l % 3; k < NL; k += 3) x += sm[q][k];
    }
    const double x1 = __shfl_down_sync(0xffffffffu, x, 1), x2 = __shfl_down_sync(0xffffffffu, x, 2);
    if (q < 9 && l % 3 == 0)
        partials[(long long)blockIdx.x * 9 + q] += x + (x1 + x2);
}

}  // namespace adj64

int adjoint64_blocks(const Geom& g) { return (int)march64_grid(g, adj64::NL).blocks; }

void launch_adjoint64(const Geom& g, const Mult<double>& m, FieldSet<double> lam, const double* const E[3],
                      const double* spy, const double* spz, double* partials, cudaStream_t st) {
    using namespace adj64;
    const long long pairs = (long long)(g.nx / 2) * g.ny * g.nz, need = (pairs + NT - 1) / NT;
    const unsigned nb = (unsigned)(need < (1 << 20) ? need : (1 << 20));
    launch_pdl(spy ? mu_kernel<true> : mu_kernel<false>, dim3(nb), dim3(NT), 0, st, g, m, lam, spy, spz);
    const March64 r = march64_grid(g, NL);
    launch_pdl(spy ? lambda_kernel<true> : lambda_kernel<false>, dim3(r.blocks), dim3(NL), 0, st, g, m, lam,
               E[0], E[1], E[2], spy, spz, partials, r.tz, r.columns);
}

}  // namespace fdtd

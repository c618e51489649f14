// FP64 leapfrog step of planes that do not couple along z (nz = 1, or a batch of 2D problems).
//
// The FP64 pipe of this part has two lanes an SM, so a warp's FP64 instruction takes 64 cycles of
// its scheduler while everything else is nearly free: the kernel is arranged for few FP64
// instructions and to occupy every scheduler.  A CTA owns a TX x TY tile of one plane:
//   1. the E^n box (x0-2 .., y0-2 ..) is copied to shared memory;
//   2. every difference along x (of E_y, E_z) and along y (of E_x, E_z) is formed once and shared:
//      D*_a uses the difference at the cell and at its two transverse neighbours;
//   3. B^{n+1/2} on the tile, the column x0-1 and the row y0-1 (D*_z vanishes, see fdtd_step2d.cu);
//   4. E^{n+1}.
// About 45 FP64 instructions a cell, where the marching 3D kernel takes 110 and forms two planes of
// B for the one.  Values and rounding order are those of dstar_diff / ampere_comp on the reference
// form's differences: bitwise the same fields.
// Us a step, the 3D kernel (whole tiles) or the reference form before and this kernel: 128^2
// 39.6 / 7.6, 1000 x 750 166 / 84, 512 x 512 x 32 2677 / 869 (FP64 pipe 84 % busy).
#include <type_traits>

#include "fdtd_tma.cuh"

namespace fdtd {
namespace flat64 {

template <int TX, int TY>
struct Cfg {
    static constexpr int NT = TX * TY;
    static constexpr int EW = TX + 4, EH = TY + 4;   // E: x0-2 .. x0+TX+1, y0-2 .. y0+TY+1
    static constexpr int XW = TX + 1, XH = TY + 3;   // x differences: x0-1 .. x0+TX-1, y0-2 .. y0+TY
    static constexpr int YW = TX + 3, YH = TY + 1;   // y differences: x0-2 .. x0+TX, y0-1 .. y0+TY-1
    static constexpr int BW = TX + 1, BH = TY + 1;   // B: x0-1 .. x0+TX-1, y0-1 .. y0+TY-1
    static constexpr int NB = (BW * BH + NT - 1) / NT;
    static constexpr int EN = EW * EH, XN = XW * XH, YN = YW * YH, BN = BW * BH;
    // dynamic shared memory: 15160 bytes of the small tile, 50296 of the large one (static shared
    // memory ends at 48 KB)
    static constexpr size_t SMEM = (3 * EN + 2 * XN + 2 * YN + 3 * BN) * sizeof(double);
};

__device__ __forceinline__ bool nonfinite(double v) {
    return ((unsigned)__double2hiint(v) & 0x7ff00000u) == 0x7ff00000u;
}

// ZC: D*_x or D*_y has a transverse z term (a 3D problem one plane thick)
template <int TX, int TY, bool ZC>
__global__ void __launch_bounds__(TX* TY)
step2d64_kernel(Geom g, Mult<double> m, FieldSet<double> in, FieldSet<double> out,
                const double* __restrict__ spy, const double* __restrict__ spz,
                const double* __restrict__ jyz, const double* jx_row,
                double* __restrict__ h0, double* __restrict__ h1, double* __restrict__ h2,
                int* __restrict__ err) {
    using C = Cfg<TX, TY>;
    constexpr int EW = C::EW, XW = C::XW, YW = C::YW, BW = C::BW, NT = C::NT;
    extern __shared__ __align__(16) double smem64[];
    double (*sE)[C::EN] = reinterpret_cast<double (*)[C::EN]>(smem64);
    double (*sX)[C::XN] = reinterpret_cast<double (*)[C::XN]>(smem64 + 3 * C::EN);   // d_x of E_y, E_z
    double (*sY)[C::YN] = reinterpret_cast<double (*)[C::YN]>(sX + 2);               // d_y of E_x, E_z
    double (*sB)[C::BN] = reinterpret_cast<double (*)[C::BN]>(sY + 2);
    static_assert(C::EW % 2 == 0, "rows of the E box start on 16 bytes");
    pdl_wait();
    const int ntx = (g.nx + TX - 1) / TX, nty = (g.ny + TY - 1) / TY;
    int w = blockIdx.x;
    const int tx = w % ntx;
    w /= ntx;
    const int ty = w % nty, k = w / nty;
    const int x0 = tx * TX, y0 = ty * TY, tid = threadIdx.x;
    const long long po = (long long)k * g.plane;

    // E box: padded row y0 + r, column x0 + 2 + 2 c; a ragged tile's box stops at the ghosts
    for (int t = tid; t < C::EH * (EW / 2); t += NT) {
        const int r = t / (EW / 2), c = t - r * (EW / 2);
        if (y0 + r >= g.nyp || x0 + 2 + 2 * c >= g.nxp) continue;
        const long long o = po + (long long)(y0 + r) * g.nxp + x0 + 2 + 2 * c;
#pragma unroll
        for (int q = 0; q < 3; ++q)
            asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(smem_u32(&sE[q][r * EW + 2 * c])),
                         "l"(in.c[q] + o)
                         : "memory");
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
    // B^{n-1/2} of this thread's cells (moved back onto the grid past a ragged end: dropped)
    double b[C::NB][3];
#pragma unroll
    for (int q = 0; q < C::NB; ++q) {
        const int t = min(tid + q * NT, C::BH * BW - 1), r = t / BW, c = t - r * BW;
        const int i = min(x0 - 1 + c, g.nx - 1), j = min(y0 - 1 + r, g.ny - 1);
        const long long o = po + (long long)(j + PY) * g.nxp + (i + PX);
#pragma unroll
        for (int a = 0; a < 3; ++a) b[q][a] = in.c[3 + a][o];
    }
    asm volatile("cp.async.wait_group 0;" ::: "memory");
    __syncthreads();
    for (int t = tid; t < C::XH * XW; t += NT) {
        const int r = t / XW, c = t - r * XW, e = r * EW + c + 1;
        sX[0][t] = sE[1][e + 1] - sE[1][e];
        sX[1][t] = sE[2][e + 1] - sE[2][e];
    }
    for (int t = tid; t < C::YH * YW; t += NT) {
        const int r = t / YW, c = t - r * YW, e = (r + 1) * EW + c;
        sY[0][t] = sE[0][e + EW] - sE[0][e];
        sY[1][t] = sE[2][e + EW] - sE[2][e];
    }
    __syncthreads();
#pragma unroll
    for (int q = 0; q < C::NB; ++q) {
        const int t = tid + q * NT;
        if (t >= C::BH * BW) break;
        const int r = t / BW, c = t - r * BW, e = (r + 1) * EW + c + 1;
        const int x = (r + 1) * XW + c, y = r * YW + c + 1;
        // D*_x, D*_y (dstar_diff's order; the transverse z differences equal the plane's own)
        auto ds = [](double d, double f2, double fm, double dp, double dm, double cA, double cD,
                     double cB, double cZ) {
            double v = cA * d;
            v = fma(cD, f2 - fm, v);
            v = fma(cB, dp + dm, v);
            return ZC ? fma(cZ, d + d, v) : v;
        };
        auto DX = [&](int s, const double* E) {
            return ds(sX[s][x], E[e + 2], E[e - 1], sX[s][x + XW], sX[s][x - XW], m.cA[0], m.cD[0],
                      m.cB[0][1], m.cB[0][2]);
        };
        auto DY = [&](int s, const double* E) {
            return ds(sY[s][y], E[e + 2 * EW], E[e - EW], sY[s][y + 1], sY[s][y - 1], m.cA[1], m.cD[1],
                      m.cB[1][0], m.cB[1][2]);
        };
        double bx = b[q][0] - DY(1, sE[2]);
        double by = b[q][1] + DX(1, sE[2]);
        double bz = b[q][2] + (DY(0, sE[0]) - DX(0, sE[1]));
        const int i = x0 - 1 + c, j = y0 - 1 + r;
        if (spy != nullptr) {
            const double f = spy[j < 0 ? j + g.ny : min(j, g.ny - 1)] * spz[k];
            bx *= f;
            by *= f;
            bz *= f;
        }
        sB[0][t] = bx;
        sB[1][t] = by;
        sB[2][t] = bz;
        if (c >= 1 && r >= 1 && i < g.nx && j < g.ny) {
            store_img(g, out.c[3], i, j, k, bx);
            store_img(g, out.c[4], i, j, k, by);
            store_img(g, out.c[5], i, j, k, bz);
        }
    }
    __syncthreads();
    pdl_trigger();
    const int cx = tid % TX, ry = tid / TX, i = x0 + cx, j = y0 + ry;
    if (i >= g.nx || j >= g.ny) return;
    const int e = (ry + 2) * EW + cx + 2, t = (ry + 1) * BW + cx + 1;
    double ex = sE[0][e] + __dmul_rn(m.cE[1], sB[2][t] - sB[2][t - BW]);
    double ey = sE[1][e] - __dmul_rn(m.cE[0], sB[2][t] - sB[2][t - 1]);
    double ez = ampere_comp(sE[2][e], sB[1][t], sB[1][t - 1], sB[0][t], sB[0][t - BW], m.cE[0], m.cE[1]);
    if (jx_row != nullptr) ex = fma(-m.dt, (jx_row[i] * jyz[j]) * jyz[g.ny + k], ex);
    if (spy != nullptr) {
        const double f = spy[j] * spz[k];
        ex *= f;
        ey *= f;
        ez *= f;
    }
    if (nonfinite(ex) || nonfinite(ey) || nonfinite(ez)) atomicOr(err, ERR_FIELD);
    store_img(g, out.c[0], i, j, k, ex);
    store_img(g, out.c[1], i, j, k, ey);
    store_img(g, out.c[2], i, j, k, ez);
    if (h0 != nullptr) {
        store_img(g, h0, i, j, k, ex);
        store_img(g, h1, i, j, k, ey);
        store_img(g, h2, i, j, k, ez);
    }
}

}  // namespace flat64

// before the first launch: room for the large tile's shared memory
bool step2d64_prepare() {
    using namespace flat64;
    bool ok = true;
    for (auto kern : {step2d64_kernel<32, 16, false>, step2d64_kernel<32, 16, true>})
        ok = ok && cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                        (int)Cfg<32, 16>::SMEM) == cudaSuccess;
    return ok;
}

void launch_step2d64(const Geom& g, const Mult<double>& m, FieldSet<double> in, FieldSet<double> out,
                     const double* spy, const double* spz, const double* jyz, const double* jx_row,
                     double* hist_E[3], int* err, cudaStream_t st) {
    using namespace flat64;
    auto go = [&](auto tx, auto ty) {
        constexpr int TX = decltype(tx)::value, TY = decltype(ty)::value;
        const long long tiles = (long long)((g.nx + TX - 1) / TX) * ((g.ny + TY - 1) / TY) * g.nz;
        const bool zc = m.cB[0][2] != 0.0 || m.cB[1][2] != 0.0;
        launch_pdl(zc ? step2d64_kernel<TX, TY, true> : step2d64_kernel<TX, TY, false>,
                   dim3((unsigned)tiles), dim3(Cfg<TX, TY>::NT), Cfg<TX, TY>::SMEM, st, g, m, in, out, spy, spz, jyz,
                   jx_row, hist_E[0], hist_E[1], hist_E[2], err);
    };
    // Small tiles reach more SMs and schedulers, large ones form fewer halo values (us, 16 x 8 / 32 x 16:
    // 128^2 7.6 / 12.5, 512^2 35.6 / 36.5, 300 x 200 x 10 73 / 76, 1000 x 750 88 / 84, 2048^2 470 / 437).
    using std::integral_constant;
    if ((long long)g.nx * g.ny * g.nz < 700000) go(integral_constant<int, 16>(), integral_constant<int, 8>());
    else go(integral_constant<int, 32>(), integral_constant<int, 16>());
}

}  // namespace fdtd

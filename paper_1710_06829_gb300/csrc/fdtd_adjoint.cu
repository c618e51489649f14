// Adjoint (transposed) leapfrog step with the fused stencil-coefficient gradient.
//
// The forward step is u^{n+1} = M u^n + s^n with
//   B1 = S (B0 + dt F E0),   E1 = S (E0 + dt (G B1 - J)),
// F E = -D* x E (extended stencil, Eq. D*), G B = D x B (Yee), S the diagonal
// sponge (identity without absorbing layers).  For the adjoint state
// lambda = (lambda_E, lambda_B) attached to u^{n+1}:
//   l_E = S lambda_E,   mu = S (lambda_B + dt G^T l_E),
//   lambda_E <- l_E + dt F^T mu,   lambda_B <- mu,
//   dL/dtheta += dt <mu, (dF/dtheta) E0>.
// With alpha eliminated by Eq. (alpha), for D*_a applied to a field F:
//   d/d delta_a:  [(F[+2a] - F[-a]) - 3 (F[+a] - F[0])] / dx_a
//   d/d beta_ab:  [(F[+a+b] - F[+b]) + (F[+a-b] - F[-b]) - 2 (F[+a] - F[0])] / dx_a
// Kernel adjB computes mu (written to lambda_B) and the gradient partials;
// kernel adjE then updates lambda_E from the new lambda_B.
#include <type_traits>

#include "fdtd_seg.cuh"

namespace fdtd {

__device__ __forceinline__ long long zoff_a(const Geom& g, int k, int dz) {
    int kk = (k + dz) % g.nz;
    if (kk < 0) kk += g.nz;
    return (long long)(kk - k) * g.plane;
}

template <typename T>
__device__ __forceinline__ void store_images_a(const Geom& g, T* F, int i, int j, int k, T v) {
    const long long base = (long long)k * g.nyp;
    F[(base + j + PY) * g.nxp + i + PX] = v;
    const bool xedge = (i < PX) || (i >= g.nx - PX);
    const bool yedge = (j < PY) || (j >= g.ny - PY);
    if (!xedge && !yedge) return;
    for (int my = -2; my <= 2; ++my) {
        const int jj = j + my * g.ny;
        if (jj < -PY || jj >= g.ny + PY) continue;
        for (int mx = -1; mx <= 1; ++mx) {
            const int ii = i + mx * g.nx;
            if (ii < -PX || ii >= g.nx + PX) continue;
            if (mx == 0 && my == 0) continue;
            F[(base + jj + PY) * g.nxp + ii + PX] = v;
        }
    }
}

// sponge factor of the cell whose owned index is (j, k) possibly shifted by one
template <typename T>
__device__ __forceinline__ T sp_at(const Geom& g, const T* spy, const T* spz, int j, int k) {
    if (spy == nullptr) return T(1);
    int jj = j % g.ny;
    if (jj < 0) jj += g.ny;
    int kk = k % g.nz;
    if (kk < 0) kk += g.nz;
    return spy[jj] * spz[kk];
}

// Gradient brackets of D*_a at c for field F: returns (d/d delta_a, d/d beta_ab, d/d beta_ac)
// without the 1/dx_a factor.
template <typename T>
__device__ __forceinline__ void dcoef(const T* __restrict__ F, long long c, long long a1,
                                      long long a2, long long am1, long long bp, long long bm,
                                      long long cp, long long cm, T& dd, T& db, T& dc) {
    const T ax = F[c + a1] - F[c];
    dd = (F[c + a2] - F[c + am1]) - T(3) * ax;
    db = (F[c + a1 + bp] - F[c + bp]) + (F[c + a1 + bm] - F[c + bm]) - T(2) * ax;
    dc = (F[c + a1 + cp] - F[c + cp]) + (F[c + a1 + cm] - F[c + cm]) - T(2) * ax;
}

// The cells are summed in chains: chain (b, t) holds the cells i = t, t + 256, ... of the rows b,
// b + CHAIN_ROWS, ... in that order, at most ADJ_FLUSH of their terms in the field precision before
// they are added to FP64 accumulators (an FP64 add costs 64 issue slots on this part).  The chains
// fix the rounding of an FP32 gradient, so they stay as they are; which thread takes a chain does
// not matter, so the threads take them one after the other, the chains of a row on neighbouring
// threads (one block a chain row left most lanes of a narrow grid idle and, at 140 registers,
// one block an SM: 418 us at 300 x 250 x 56 FP32, 180 here), and a block's sums are taken once.
// Groups are a loop of their own: as a test in the cell loop the adds were made in every cell.
constexpr int ADJ_THREADS = 128, CHAIN_WIDTH = 256, CHAIN_ROWS = 152 * 8, ADJ_FLUSH = 16;

static long long adjoint_chains(const Geom& g) {
    const long long rows = (long long)g.ny * g.nz;
    return (rows < CHAIN_ROWS ? rows : CHAIN_ROWS) * (g.nx < CHAIN_WIDTH ? g.nx : CHAIN_WIDTH);
}

int adjoint_B_blocks(const Geom& g) {
    const long long b = (adjoint_chains(g) + ADJ_THREADS - 1) / ADJ_THREADS;
    return (int)(b < 152 * 4 ? b : 152 * 4);   // the resident blocks
}

// partials layout: [block][9] = per axis a (x, y, z): d/d delta_a, d/d beta_a,b1, d/d beta_a,b2
// with b1 < b2 the two other axes.  Accumulated across steps (+=) by the owning block.
template <typename T>
__global__ void __launch_bounds__(ADJ_THREADS, sizeof(T) == 4 ? 4 : 2)
adjoint_B_kernel(Geom g, Mult<T> m, FieldSet<T> lam, const T* __restrict__ Ex,
                 const T* __restrict__ Ey, const T* __restrict__ Ez, const T* __restrict__ spy,
                 const T* __restrict__ spz, double* __restrict__ partials) {
    double acc[9];
#pragma unroll
    for (int q = 0; q < 9; ++q) acc[q] = 0.0;
    const int rows = g.ny * g.nz;
    const int nrow = rows < CHAIN_ROWS ? rows : CHAIN_ROWS, width = g.nx < CHAIN_WIDTH ? g.nx : CHAIN_WIDTH;
    const long long Y = g.nxp;
    const T* lEx = lam.c[0];
    const T* lEy = lam.c[1];
    const T* lEz = lam.c[2];
    for (int ch = blockIdx.x * ADJ_THREADS + threadIdx.x; ch < nrow * width; ch += gridDim.x * ADJ_THREADS) {
        const int b = ch / width, t = ch - b * width;
        for (int r = b, i = t; r < rows;) {
            T racc[9];
#pragma unroll
            for (int q = 0; q < 9; ++q) racc[q] = T(0);
#pragma unroll 1
            for (int cnt = 0; cnt < ADJ_FLUSH && r < rows; ++cnt) {
                const int k = r / g.ny, j = r - k * g.ny;
                const long long rowbase = pidx(g, 0, j, k);
                const long long zp1 = zoff_a(g, k, 1), zm1 = zoff_a(g, k, -1), zp2 = zoff_a(g, k, 2);
                // l_E = S lambda_E at the cell and its +x, +y, +z neighbours
                const T s0 = sp_at(g, spy, spz, j, k);
                const T sxp = s0;
                const T syp = sp_at(g, spy, spz, j + 1, k);
                const T szp = sp_at(g, spy, spz, j, k + 1);
                const long long c = rowbase + i;
                const T ex0 = s0 * lEx[c], ey0 = s0 * lEy[c], ez0 = s0 * lEz[c];
                // G^T l_E (transposed backward differences = forward differences with a minus sign)
                T nx_ = lam.c[3][c] + (m.cE[2] * (ey0 - szp * lEy[c + zp1]) - m.cE[1] * (ez0 - syp * lEz[c + Y]));
                T ny_ = lam.c[4][c] + (m.cE[0] * (ez0 - sxp * lEz[c + 1]) - m.cE[2] * (ex0 - szp * lEx[c + zp1]));
                T nz_ = lam.c[5][c] + (m.cE[1] * (ex0 - syp * lEx[c + Y]) - m.cE[0] * (ey0 - sxp * lEy[c + 1]));
                const T mux = s0 * nx_, muy = s0 * ny_, muz = s0 * nz_;
                // gradient: axis x appears as +mu_y D*_x E_z - mu_z D*_x E_y
                T d0, d1, d2, e0, e1, e2;
                dcoef(Ez, c, 1, 2, -1, Y, -Y, zp1, zm1, d0, d1, d2);
                dcoef(Ey, c, 1, 2, -1, Y, -Y, zp1, zm1, e0, e1, e2);
                racc[0] += muy * d0 - muz * e0;
                racc[1] += muy * d1 - muz * e1;
                racc[2] += muy * d2 - muz * e2;
                // axis y: +mu_z D*_y E_x - mu_x D*_y E_z   (transverse order x, z)
                dcoef(Ex, c, Y, 2 * Y, -Y, 1, -1, zp1, zm1, d0, d1, d2);
                dcoef(Ez, c, Y, 2 * Y, -Y, 1, -1, zp1, zm1, e0, e1, e2);
                racc[3] += muz * d0 - mux * e0;
                racc[4] += muz * d1 - mux * e1;
                racc[5] += muz * d2 - mux * e2;
                // axis z: +mu_x D*_z E_y - mu_y D*_z E_x   (transverse order x, y)
                dcoef(Ey, c, zp1, zp2, zm1, 1, -1, Y, -Y, d0, d1, d2);
                dcoef(Ex, c, zp1, zp2, zm1, 1, -1, Y, -Y, e0, e1, e2);
                racc[6] += mux * d0 - muy * e0;
                racc[7] += mux * d1 - muy * e1;
                racc[8] += mux * d2 - muy * e2;
                store_images_a(g, lam.c[3], i, j, k, mux);
                store_images_a(g, lam.c[4], i, j, k, muy);
                store_images_a(g, lam.c[5], i, j, k, muz);
                i += CHAIN_WIDTH;
                if (i >= g.nx) {
                    i = t;
                    r += nrow;
                }
            }
#pragma unroll
            for (int q = 0; q < 9; ++q) acc[q] += (double)racc[q];
        }
    }
    __shared__ double sm[9][ADJ_THREADS];
#pragma unroll
    for (int q = 0; q < 9; ++q) sm[q][threadIdx.x] = acc[q];
    __syncthreads();
    const int w = threadIdx.x >> 5, l = threadIdx.x & 31;
    for (int q = w; q < 9; q += ADJ_THREADS / 32) {
        double v = (sm[q][l] + sm[q][l + 32]) + (sm[q][l + 64] + sm[q][l + 96]);
        for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
        if (l == 0) partials[(long long)blockIdx.x * 9 + q] += v;
    }
}

// lambda_E <- S lambda_E + dt F^T mu,  F^T from the transposed taps of D*:
//   (D*_a)^T G = alpha_a (G[-a] - G[0]) + delta_a (G[-2a] - G[+a])
//              + sum_b beta_ab ((G[-a-b] - G[-b]) + (G[-a+b] - G[+b])).
template <typename T>
__device__ __forceinline__ T dstarT_at(const T* __restrict__ G, long long c, long long am1,
                                       long long am2, long long ap1, long long bp, long long bm,
                                       long long cp, long long cm, T cA, T cD, T cBb, T cBc) {
    T v = cA * (G[c + am1] - G[c]);
    v = fma(cD, G[c + am2] - G[c + ap1], v);
    v = fma(cBb, (G[c + am1 + bm] - G[c + bm]) + (G[c + am1 + bp] - G[c + bp]), v);
    v = fma(cBc, (G[c + am1 + cm] - G[c + cm]) + (G[c + am1 + cp] - G[c + cp]), v);
    return v;
}

template <typename T>
__global__ void adjoint_E_kernel(Geom g, Mult<T> m, FieldSet<T> lam, const T* __restrict__ spy,
                                 const T* __restrict__ spz) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= g.nx) return;
    for (int k = blockIdx.z; k < g.nz; k += gridDim.z)
        for (int j = blockIdx.y; j < g.ny; j += gridDim.y) {
            const long long c = pidx(g, i, j, k);
            const long long Y = g.nxp;
            const long long zp1 = zoff_a(g, k, 1), zm1 = zoff_a(g, k, -1), zm2 = zoff_a(g, k, -2);
            const T* mux = lam.c[3];
            const T* muy = lam.c[4];
            const T* muz = lam.c[5];
#define DTX(G) dstarT_at(G, c, -1, -2, 1, Y, -Y, zp1, zm1, m.cA[0], m.cD[0], m.cB[0][1], m.cB[0][2])
#define DTY(G) dstarT_at(G, c, -Y, -2 * Y, Y, 1, -1, zp1, zm1, m.cA[1], m.cD[1], m.cB[1][0], m.cB[1][2])
#define DTZ(G) dstarT_at(G, c, zm1, zm2, zp1, 1, -1, Y, -Y, m.cA[2], m.cD[2], m.cB[2][0], m.cB[2][1])
            const T s0 = sp_at(g, spy, spz, j, k);
            const T ex = s0 * lam.c[0][c] + (DTY(muz) - DTZ(muy));
            const T ey = s0 * lam.c[1][c] + (DTZ(mux) - DTX(muz));
            const T ez = s0 * lam.c[2][c] + (DTX(muy) - DTY(mux));
#undef DTX
#undef DTY
#undef DTZ
            store_images_a(g, lam.c[0], i, j, k, ex);
            store_images_a(g, lam.c[1], i, j, k, ey);
            store_images_a(g, lam.c[2], i, j, k, ez);
        }
}

template <typename T>
void launch_adjoint_B_v0(const Geom& g, const Mult<T>& m, FieldSet<T> lam, const T* E_hist[3],
                         const T* sponge_y, const T* sponge_z, double* partials, int nblk,
                         cudaStream_t st) {
    adjoint_B_kernel<T><<<nblk, ADJ_THREADS, 0, st>>>(g, m, lam, E_hist[0], E_hist[1], E_hist[2],
                                                        sponge_y, sponge_z, partials);
}

// The same for FP32, four cells of a row a thread: 29 16-byte loads and 22 of one value, instead of 300
// of one value, the differences that the cells share formed once.  Values and order are those
// of dstarT_at.  Bound: L1 and L2 (every row comes to each block that reads it).  Us, one cell a
// thread and this kernel: 300 x 250 x 56 75.6 / 46.5, 140 x 100 x 150 41.1 / 22.3, 100 x 90 x 80
// 15.8 / 10.2, 500 x 300 x 32 78.5 / 52.3, 36^3 4.3 / 4.5.  At 300 x 250 x 56 tiles of several rows a
// block take 58, the stores at the end 51.4.
__global__ void __launch_bounds__(128)
adjoint_E4_kernel(Geom g, Mult<float> m, FieldSet<float> lam, const float* __restrict__ spy,
                  const float* __restrict__ spz, int n) {
    using namespace seg;
    const int t = blockIdx.x * 128 + threadIdx.x, ns = g.nx / 4;
    if (t >= n) return;
    const int row = t / ns, i = (t - row * ns) * 4, k = row / g.ny, j = row - k * g.ny;
    const int c = (int)pidx(g, i, j, k), Y = g.nxp;
    const int zp = (int)zoff_a(g, k, 1), zm = (int)zoff_a(g, k, -1), zmm = (int)zoff_a(g, k, -2);
    const float *X = lam.c[3] + c, *V = lam.c[4] + c, *Z = lam.c[5] + c;
    // DT along an axis of one component: the own row o, one back b, two back bb, one ahead f of the
    // row, and the differences b - o of the rows beside (p, q: first axis, r, s: second)
    auto comb = [](const float* d, const float* bb, const float* f, const float* p, const float* q,
                   const float* r, const float* s, float cA, float cD, float cB, float cC, float* out) {
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            float v = cA * d[u];
            v = fma(cD, bb[u] - f[u], v);
            v = fma(cB, p[u] + q[u], v);
            out[u] = fma(cC, r[u] + s[u], v);
        }
    };
    auto diff = [](const Q4& a, const Q4& b, float* d) {
#pragma unroll
        for (int u = 0; u < 4; ++u) d[u] = a.v[u] - b.v[u];
    };
    // differences of one row against the next along x, x-1 .. x+4's: transverse x neighbours of d
    auto beside = [](const float* d, float lo, float hi, float* left, float* right) {
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            left[u] = u ? d[u ? u - 1 : 0] : lo;
            right[u] = u < 3 ? d[u < 3 ? u + 1 : 3] : hi;
        }
    };
    // differences along x of a row whose value at x-1 is l
    auto along = [](float l, const Q4& a, float* d) {
#pragma unroll
        for (int u = 0; u < 4; ++u) d[u] = (u ? a.v[u ? u - 1 : 0] : l) - a.v[u];
    };
    // DT_x: own row a (x-2, x-1, x+4 in l2, l1, r), rows y-1, y+1, z-1, z+1 with their values at x-1
    auto dtx = [&](const Q4& a, float l2, float l1, float r, const Q4& ym, float lym, const Q4& yp,
                   float lyp, const Q4& bm, float lbm, const Q4& bp, float lbp, float* out) {
        float d[4], p[4], q[4], e[4], f[4], bb[4], ff[4];
        along(l1, a, d);
        along(lym, ym, p);
        along(lyp, yp, q);
        along(lbm, bm, e);
        along(lbp, bp, f);
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            bb[u] = u == 0 ? l2 : u == 1 ? l1 : a.v[u > 1 ? u - 2 : 0];
            ff[u] = u < 3 ? a.v[u < 3 ? u + 1 : 3] : r;
        }
        comb(d, bb, ff, p, q, e, f, m.cA[0], m.cD[0], m.cB[0][1], m.cB[0][2], out);
    };
    // DT_y of the component at G: own rows a (y), b (y-1), f (y+1); values beside the own row at
    // x-1 and x+4 in al, ar; rows (y, z-1), (y, z+1) in am, ap
    auto dty = [&](const float* G, const Q4& a, const Q4& b, const Q4& f, float al, float ar, const Q4& am,
                   const Q4& bm, const Q4& ap, float* out) {
        const Q4 bb = ldq(G, -2 * Y), bp = ldq(G, zp - Y);
        float d[4], l[4], r[4], e[4], h[4];
        diff(b, a, d);
        beside(d, G[-Y - 1] - al, G[-Y + 4] - ar, l, r);
        diff(bm, am, e);
        diff(bp, ap, h);
        comb(d, bb.v, f.v, l, r, e, h, m.cA[1], m.cD[1], m.cB[1][0], m.cB[1][2], out);
    };
    // DT_z: own rows a (z), b (z-1), f (z+1); beside a and b at x-1, x+4 in al, ar, bl, br; rows y-1
    // and y+1 of z in am, ap, of z-1 in bm, bp
    auto dtz = [&](const float* G, const Q4& a, const Q4& b, const Q4& f, float al, float ar, float bl,
                   float br, const Q4& am, const Q4& bm, const Q4& ap, const Q4& bp, float* out) {
        const Q4 bb = ldq(G, zmm);
        float d[4], l[4], r[4], e[4], h[4];
        diff(b, a, d);
        beside(d, bl - al, br - ar, l, r);
        diff(bm, am, e);
        diff(bp, ap, h);
        comb(d, bb.v, f.v, l, r, e, h, m.cA[2], m.cD[2], m.cB[2][0], m.cB[2][1], out);
    };
    const float s0 = sp_at(g, spy, spz, j, k);
    const bool edge = i < PX || i >= g.nx - PX || j < PY || j >= g.ny - PY;
    const SegOut dst = seg_out(g, i, j, edge);
    const unsigned po = (unsigned)k * (unsigned)g.plane;
    auto put = [&](int q, const float* a, const float* b) {
        const Q4 l = ldq(lam.c[q], c);
        float v[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) v[u] = __fmaf_rn(s0, l.v[u], __fsub_rn(a[u], b[u]));
        put_seg(lam.c[q], po, dst, v);
    };
    float yz[4], xz[4], zy[4], xy[4], zx[4], yx[4];
    {   // mu_z: DT_y, DT_x
        const Q4 a = ldq(Z, 0), b = ldq(Z, -Y), f = ldq(Z, Y), am = ldq(Z, zm), ap = ldq(Z, zp),
                 bm = ldq(Z, zm - Y);
        const float l1 = Z[-1], r = Z[4];
        dty(Z, a, b, f, l1, r, am, bm, ap, yz);
        dtx(a, Z[-2], l1, r, b, Z[-Y - 1], f, Z[Y - 1], am, Z[zm - 1], ap, Z[zp - 1], xz);
    }
    {   // mu_y: DT_z, DT_x
        const Q4 a = ldq(V, 0), b = ldq(V, zm), f = ldq(V, zp), am = ldq(V, -Y), ap = ldq(V, Y);
        const float l1 = V[-1], r = V[4], bl = V[zm - 1];
        dtz(V, a, b, f, l1, r, bl, V[zm + 4], am, ldq(V, zm - Y), ap, ldq(V, zm + Y), zy);
        dtx(a, V[-2], l1, r, am, V[-Y - 1], ap, V[Y - 1], b, bl, f, V[zp - 1], xy);
    }
    put(0, yz, zy);
    {   // mu_x: DT_z, DT_y
        const Q4 a = ldq(X, 0), b = ldq(X, zm), f = ldq(X, zp), am = ldq(X, -Y), ap = ldq(X, Y),
                 bm = ldq(X, zm - Y);
        const float l1 = X[-1], r = X[4];
        dtz(X, a, b, f, l1, r, X[zm - 1], X[zm + 4], am, bm, ap, ldq(X, zm + Y), zx);
        dty(X, a, am, ap, l1, r, b, bm, f, yx);
    }
    put(1, zx, xz);
    put(2, xy, yx);
}

template <typename T>
void launch_adjoint_E_v0(const Geom& g, const Mult<T>& m, FieldSet<T> lam, const T* sponge_y,
                         const T* sponge_z, cudaStream_t st) {
    if constexpr (std::is_same<T, float>::value) {
        // put_seg's single image offsets want nx >= 8 and ny >= 4, the kernel 32-bit offsets
        if (g.nx >= 2 * PX && g.ny >= 2 * PY && g.total < (1LL << 31)) {
            const int n = g.nx / 4 * g.ny * g.nz;
            adjoint_E4_kernel<<<(n + 127) / 128, 128, 0, st>>>(g, m, lam, sponge_y, sponge_z, n);
            return;
        }
    }
    dim3 blk(128), grd((g.nx + 127) / 128, (unsigned)(g.ny < 65535 ? g.ny : 65535),
                        (unsigned)(g.nz < 65535 ? g.nz : 65535));   // j, k loop in the kernel
    adjoint_E_kernel<T><<<grd, blk, 0, st>>>(g, m, lam, sponge_y, sponge_z);
}

template void launch_adjoint_B_v0<float>(const Geom&, const Mult<float>&, FieldSet<float>,
                                         const float* [3], const float*, const float*, double*,
                                         int, cudaStream_t);
template void launch_adjoint_B_v0<double>(const Geom&, const Mult<double>&, FieldSet<double>,
                                          const double* [3], const double*, const double*,
                                          double*, int, cudaStream_t);
template void launch_adjoint_E_v0<float>(const Geom&, const Mult<float>&, FieldSet<float>,
                                         const float*, const float*, cudaStream_t);
template void launch_adjoint_E_v0<double>(const Geom&, const Mult<double>&, FieldSet<double>,
                                          const double*, const double*, cudaStream_t);

// grad12[beta row-major 3x3, delta 3] += scale_a * sum_b partials[b][.]  (one block, fixed order)
__global__ void reduce_grad_kernel(const double* __restrict__ part, int nblocks, GradScale sc,
                                   double* __restrict__ grad) {
    __shared__ double red[9][32];
    const int q = threadIdx.y;       // 0..8
    const int l = threadIdx.x;       // 0..31
    double v = 0.0;
#pragma unroll 8
    for (int b = l; b < nblocks; b += 32) v += part[(long long)b * 9 + q];
    red[q][l] = v;
    __syncthreads();
    if (l == 0) {
        double s = 0.0;
        for (int t = 0; t < 32; ++t) s += red[q][t];
        const int a = q / 3, which = q % 3;
        if (which == 0) {
            grad[9 + a] += sc.s[q] * s;
        } else {
            // transverse axes of a in increasing order
            const int b = (which == 1) ? (a == 0 ? 1 : 0) : (a == 2 ? 1 : 2);
            grad[a * 3 + b] += sc.s[q] * s;
        }
    }
}

void launch_reduce_grad(const double* part, int nblocks, GradScale sc, double* grad12,
                        cudaStream_t st) {
    reduce_grad_kernel<<<1, dim3(32, 9), 0, st>>>(part, nblocks, sc, grad12);
}

}  // namespace fdtd

// Macro-particle kernels of the PIC cycle: gather + Boris push + Esirkepov current, and the
// charge density.
//
// Particle shape: first order (cloud in cell); node i of axis a carries max(0, 1 - |x/dx_a - i|).
// Gather: each field component is interpolated from its own staggered positions (App. A):
//   E_x (i+1/2, j, k), E_y (i, j+1/2, k), E_z (i, j, k+1/2),
//   B_x (i, j+1/2, k+1/2), B_y (i+1/2, j, k+1/2), B_z (i+1/2, j+1/2, k),
// with B at the integer time level the mean of B^{n-1/2} and B^{n+1/2}.
// Push: Boris's relativistic scheme in u = gamma v (c = 1): half electric kick, rotation
// about t = (q/m)(dt/2) B / gamma^-, half electric kick; then x += dt u / gamma.
// Current: Esirkepov's decomposition of the shape change S1 - S0 into W_x + W_y + W_z,
//   W_x = dSx (S0y S0z + dSy S0z / 2 + S0y dSz / 2 + dSy dSz / 3)   (and cyclically),
//   J_x(i+1/2) - J_x(i-1/2) = -q W_x(i) / (dt dy dz),
// so that (rho^{n+1} - rho^n)/dt + D.J^{n+1/2} = 0 holds to rounding (App. A numerical
// continuity equation) and Gauss's law D.E = rho (Eq. divE) is kept.  A particle moves less
// than a cell per step (|v| < c; dt^2 S <= 1 at k_a = pi / dx_a gives c dt <= dx_a where delta_a <= 0),
// so per axis its old and new supports fit the 4-node window floor(g0) - 1 .. floor(g0) + 2.  A longer
// move, which schemes with delta_a > 0 allow, is taken with the next cell's weights continued.
//
// Ampere's law is linear in J, so the cycle first forms E^{n+1} without the current (the
// vacuum step kernel) and the push adds -dt J^{n+1/2} into its owned cells: no current
// array, no extra pass over the grid; a small kernel then copies the owned cells near the x
// and y ends to their periodic images (the ghosts the next step reads).
//
// The kernel was bound by instruction issue (4600 to 5900 warp instructions for 32 particles: a
// rolled deposit over all 144 window faces, 64-bit index arithmetic for each of 72 loads, nine
// divisions, spills), so it is written for few instructions (about 700):
//   - fields are read through the ghosts of the padded layout, so only z wraps: four row addresses
//     a component, the second value of a row at a fixed offset;
//   - where there are many particles for the grid, B^n = (B^{n-1/2} + B^{n+1/2}) / 2 is formed once
//     per cell (launch_bmean) instead of once per particle and node;
//   - a face's weight is A_b A_c + dS_b dS_c / 12 with A = S0 + dS / 2 (Esirkepov's four terms);
//   - the 12 faces that a particle in any case reaches are added without loops, the 8 more of an
//     axis on which it changes its cell in a branch of their own, the rest of a move across
//     several axes in another;
//   - where all 32 particles of a warp sit in one cell (a dense bunch, particles kept in cell
//     order), the values of each face are summed through shared memory and added once.
// Push per cycle: bunch of 2^22 particles in a 512 x 256 x 256 grid 717 -> 214 us; 2^22 particles of
// a 128^3 plasma, drifted by a cell, 823 -> 287 us (with single additions instead of add_pair 15 us more),
// bound by L2 (72 % busy: 10 sectors of additions and 11 of loads a particle) and L1 (76 %).
#include <climits>
#include <cmath>

#include "pic.cuh"

namespace fdtd {
namespace picd {

constexpr int THREADS = 256;
constexpr unsigned FULL = 0xffffffffu;

__device__ __forceinline__ int wrapi(int i, int n) {
    int r = i % n;
    return r < 0 ? r + n : r;
}

// first-order weights of grid coordinate gc on nodes i0 = floor(gc) and i1 = i0 + 1 (wrapped)
template <typename T>
struct Lin {
    int i0, i1;
    T w0, w1;
};

template <typename T>
__device__ __forceinline__ Lin<T> lin(T gc, int n) {
    const T f = floor(gc);
    Lin<T> l;
    l.w1 = gc - f;
    l.w0 = T(1) - l.w1;
    l.i0 = wrapi((int)f, n);
    l.i1 = l.i0 + 1 == n ? 0 : l.i0 + 1;
    return l;
}

// a finite coordinate moved into [0, L] (unchanged when already inside)
template <typename T>
__device__ __forceinline__ T into_box(T x, T L) {
    if (x >= T(0) && x < L) return x;
    const T r = x - L * floor(x / L);
    return r < T(0) ? T(0) : (r > L ? L : r);
}

template <typename T>
__device__ __forceinline__ bool finite3(T a, T b, T c) {
    return isfinite(a) && isfinite(b) && isfinite(c);
}

// One axis of a particle: the cell f its old position lies in, the weight w of node f + 1, and the
// staggered pair of nodes (f - 1, f) or (f, f + 1) with the weight ws of its upper node.
template <typename T>
struct Cell {
    int f;
    T f0, w, ws;
    int st;   // lower staggered node minus f: -1 or 0
};

template <typename T>
__device__ __forceinline__ Cell<T> cell_of(T g) {
    Cell<T> c;
    c.f0 = floor(g);
    c.f = (int)c.f0;
    c.w = g - c.f0;
    c.st = c.w < T(0.5) ? -1 : 0;
    c.ws = c.st ? c.w + T(0.5) : c.w - T(0.5);
    return c;
}

// The move along one axis, on the nodes f, f + 1 and, where the particle changes its cell, the node
// beyond (f + 2 or f - 1): shape change dS, mean shape A = S0 + dS / 2, and the cumulative change at
// the face above f and at the further face that a change of cell reaches (the sum over all nodes
// vanishes).  o: element offsets of the three nodes, wrapped into the owned cells.
template <typename T, typename I>
struct Move {
    T A[3], D[3];
    T C0, Cx;
    int s;      // -1, 0, 1: change of cell
    I o[3], ox; // ox: the further face's offset
};

template <typename T, typename I>
__device__ __forceinline__ Move<T, I> move_of(const Cell<T>& c, T g1, int n, I pitch, I origin,
                                              int (&node)[3]) {
    Move<T, I> m;
    // |move| < 1; the clamp keeps the offsets in the grid whatever the fields hold (NaN: s = -1)
    const T sf = fmin(T(1), fmax(T(-1), floor(g1) - c.f0));
    m.s = (int)sf;
    const T w1 = g1 - (c.f0 + sf), v1 = T(1) - w1, v = T(1) - c.w;
    m.D[0] = (m.s == 0 ? v1 : m.s < 0 ? w1 : T(0)) - v;
    m.D[1] = (m.s == 0 ? w1 : m.s > 0 ? v1 : T(0)) - c.w;
    m.D[2] = m.s == 0 ? T(0) : m.s > 0 ? w1 : v1;
    m.A[0] = v + T(0.5) * m.D[0];
    m.A[1] = c.w + T(0.5) * m.D[1];
    m.A[2] = T(0.5) * m.D[2];
    m.C0 = m.s < 0 ? m.D[2] + m.D[0] : m.D[0];
    m.Cx = m.s > 0 ? m.C0 + m.D[1] : m.D[2];
    const int e = m.s < 0 ? c.f - 1 : c.f + 2;
    node[0] = c.f >= n ? c.f - n : c.f;
    node[1] = node[0] + 1 == n ? 0 : node[0] + 1;
    node[2] = e < 0 ? e + n : e >= n ? e - n : e;
    if (node[2] >= n) node[2] %= n;   // grids of one or two cells
#pragma unroll
    for (int q = 0; q < 3; ++q) m.o[q] = (I)node[q] * pitch + origin;
    m.ox = m.s > 0 ? m.o[1] : m.o[2];
    return m;
}

template <typename T>
__device__ __forceinline__ void add_to(T* p, T v) {
    if (v != T(0)) atomicAdd(p, v);
}

// Adds v0, v1 at the x nodes f, f + 1 of a row (offset o of node f; f + 1 wraps only where o % 4 == 3):
// one 16-byte reduction of the aligned group of four that holds both, which L2 takes as one
// sector, where there is one.
template <typename T, typename I>
__device__ __forceinline__ void add_pair(T* row, I o, I o1, T v0, T v1) {
    if constexpr (sizeof(T) == 4) {
        const int r = (int)(o & 3);
        if (r != 3) {
            if (v0 == T(0) && v1 == T(0)) return;
            const float a = r == 0 ? v0 : 0.0f, b = r == 0 ? v1 : r == 1 ? v0 : 0.0f,
                        c = r == 1 ? v1 : r == 2 ? v0 : 0.0f, d = r == 2 ? v1 : 0.0f;
            asm volatile("red.relaxed.gpu.global.add.v4.f32 [%0], {%1, %2, %3, %4};" ::"l"(row + (o - r)),
                         "f"(a), "f"(b), "f"(c), "f"(d)
                         : "memory");
            return;
        }
    }
    add_to(row + o, v0);
    add_to(row + o1, v1);
}

// weight of the transverse nodes b, c of a face
template <typename T, typename I>
__device__ __forceinline__ T face_weight(const Move<T, I>& B, int b, const Move<T, I>& C, int c) {
    return fma(B.A[b], C.A[c], T(1.0 / 12.0) * B.D[b] * C.D[c]);
}

// -dt J^{n+1/2} of one particle.  sy, sz: the layers' factors of its nodes (j, k).
template <bool SP, typename T, typename I>
__device__ __forceinline__ void deposit_lane(const PushArgs<T>& a, const Move<T, I>& X,
                                             const Move<T, I>& Y, const Move<T, I>& Z,
                                             const T (&sy)[3], const T (&sz)[3]) {
    const T cx = a.escale[0] * X.C0, cy = a.escale[1] * Y.C0, cz = a.escale[2] * Z.C0;
    const T dx = a.escale[0] * X.Cx, dy = a.escale[1] * Y.Cx, dz = a.escale[2] * Z.Cx;
    const T syx = SP ? (Y.s > 0 ? sy[1] : sy[2]) : T(1), szx = SP ? (Z.s > 0 ? sz[1] : sz[2]) : T(1);
    auto jx = [&](T v, I face, int b, int c) {
        v *= face_weight(Y, b, Z, c);
        add_to(a.Eout[0] + (face + Y.o[b] + Z.o[c]), SP ? v * (sy[b] * sz[c]) : v);
    };
    auto jy = [&](T v, I face, T sf, int b, int c) {
        v *= face_weight(X, b, Z, c);
        add_to(a.Eout[1] + (face + X.o[b] + Z.o[c]), SP ? v * (sf * sz[c]) : v);
    };
    auto jz = [&](T v, I face, T sf, int b, int c) {
        v *= face_weight(X, b, Y, c);
        add_to(a.Eout[2] + (face + X.o[b] + Y.o[c]), SP ? v * (sy[c] * sf) : v);
    };
    auto all4 = [](auto&& f) {
#pragma unroll
        for (int q = 0; q < 4; ++q) f(q >> 1, q & 1);
    };
    if (cx != T(0)) all4([&](int b, int c) { jx(cx, X.o[0], b, c); });
    if (cy != T(0)) {
#pragma unroll
        for (int c = 0; c < 2; ++c) {
            const T v = SP ? cy * (sy[0] * sz[c]) : cy;
            add_pair(a.Eout[1] + (Y.o[0] + Z.o[c]), X.o[0], X.o[1], v * face_weight(X, 0, Z, c),
                     v * face_weight(X, 1, Z, c));
        }
    }
    if (cz != T(0)) {
#pragma unroll
        for (int c = 0; c < 2; ++c) {
            const T v = SP ? cz * (sy[c] * sz[0]) : cz;
            add_pair(a.Eout[2] + (Y.o[c] + Z.o[0]), X.o[0], X.o[1], v * face_weight(X, 0, Y, c),
                     v * face_weight(X, 1, Y, c));
        }
    }
    if (X.s) {
        all4([&](int b, int c) { jx(dx, X.ox, b, c); });
#pragma unroll
        for (int q = 0; q < 2; ++q) {
            jy(cy, Y.o[0], sy[0], 2, q);
            jz(cz, Z.o[0], sz[0], 2, q);
        }
    }
    if (Y.s) {
        all4([&](int b, int c) { jy(dy, Y.ox, syx, b, c); });
#pragma unroll
        for (int q = 0; q < 2; ++q) {
            jx(cx, X.o[0], 2, q);
            jz(cz, Z.o[0], sz[0], q, 2);
        }
    }
    if (Z.s) {
        all4([&](int b, int c) { jz(dz, Z.ox, szx, b, c); });
#pragma unroll
        for (int q = 0; q < 2; ++q) {
            jx(cx, X.o[0], q, 2);
            jy(cy, Y.o[0], sy[0], q, 2);
        }
    }
    if ((X.s != 0) + (Y.s != 0) + (Z.s != 0) < 2) return;
    // a move across several axes
#pragma unroll
    for (int q = 0; q < 2; ++q) {
        if (X.s && Y.s) {
            jx(dx, X.ox, 2, q);
            jy(dy, Y.ox, syx, 2, q);
        }
        if (X.s && Z.s) {
            jx(dx, X.ox, q, 2);
            jz(dz, Z.ox, szx, 2, q);
        }
        if (Y.s && Z.s) {
            jy(dy, Y.ox, syx, q, 2);
            jz(dz, Z.ox, szx, q, 2);
        }
    }
    if (X.s && Y.s) jz(cz, Z.o[0], sz[0], 2, 2);
    if (X.s && Z.s) jy(cy, Y.o[0], sy[0], 2, 2);
    if (Y.s && Z.s) jx(cx, X.o[0], 2, 2);
    if (X.s && Y.s && Z.s) {
        jx(dx, X.ox, 2, 2);
        jy(dy, Y.ox, syx, 2, 2);
        jz(dz, Z.ox, szx, 2, 2);
    }
}

constexpr int ROW = 36;   // shared row of 32 values: 16-byte reads of neighbouring rows on distinct banks

// -dt J_a of a warp whose particles share their cell and, per axis, the sense of any change of cell:
// value (face u, node b, node c) of every lane goes to row 9 u + 3 b + c, lane r then sums row r and adds
// it.  xa, xb, xc (warp-uniform): some lane changes its cell on that axis.
template <bool SP, typename T, typename I, class Sp>
__device__ __forceinline__ void deposit_shared(T* __restrict__ E, const Move<T, I>& A,
                                               const Move<T, I>& B, const Move<T, I>& C, T scale,
                                               bool xa, bool xb, bool xc, I face_o, const I* bo,
                                               const I* co, Sp&& sp, T* __restrict__ sm) {
    const int l = threadIdx.x & 31;
    if (!__any_sync(FULL, A.C0 != T(0) || (A.s && A.Cx != T(0)))) return;
    __syncwarp();
#pragma unroll
    for (int b = 0; b < 3; ++b) {
        if (b == 2 && !xb) continue;
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            if (c == 2 && !xc) continue;
            const T f = scale * face_weight(B, b, C, c);
            sm[(3 * b + c) * ROW + l] = SP ? A.C0 * f * sp(0, b, c) : A.C0 * f;
            if (xa) sm[(9 + 3 * b + c) * ROW + l] = !A.s ? T(0) : SP ? A.Cx * f * sp(1, b, c) : A.Cx * f;
        }
    }
    __syncwarp();
    const int u = l / 9, b = (l % 9) / 3, c = l % 3;
    if (u < 2 && (u == 0 || xa) && (b < 2 || xb) && (c < 2 || xc)) {
        T t[4] = {T(0), T(0), T(0), T(0)};
#pragma unroll
        for (int q = 0; q < 32; q += 4)
#pragma unroll
            for (int r = 0; r < 4; ++r) t[r] += sm[l * ROW + q + r];
        const I ob = b == 0 ? bo[0] : b == 1 ? bo[1] : bo[2];
        const I oc = c == 0 ? co[0] : c == 1 ? co[1] : co[2];
        add_to(E + ((u == 0 ? A.o[0] : face_o) + ob + oc), (t[0] + t[1]) + (t[2] + t[3]));
    }
}

// Threads of a block: with particles all over the grid (MEAN) one block fills an SM, so that the
// 24 warps of a sweep read neighbouring field rows and the next sweep finds them in L1 (plasma
// 317 us with three blocks of 256, 287 with one of 768; in cell order no difference); a bunch is spread over more, smaller
// blocks, whose work differs less (214 us with nine of 256 an SM, 234 to 254 with blocks of 768).
// FP64 is bound by its pipe either way (3585 and 3600 us a cycle).
template <typename T, bool MEAN>
constexpr int PUSH = MEAN && sizeof(T) == 4 ? 3 * THREADS : THREADS;
template <typename T, bool MEAN>
constexpr size_t PUSH_SMEM = (size_t)(PUSH<T, MEAN> / 32) * 18 * ROW * sizeof(T);

// MEAN: a.B0 holds B^n; otherwise B^n = (B0 + B1) / 2 per node.  SP: absorbing layers.  I: type of the
// element offsets (int where a padded array has fewer than 2^31 elements).
template <typename T, bool MEAN, bool SP, typename I>
__global__ void __launch_bounds__(PUSH<T, MEAN>, sizeof(T) == 8 ? 2 : MEAN ? 1 : 3)
push_kernel(PushArgs<T> a) {
    const Geom& g = a.g;
    extern __shared__ __align__(16) unsigned char smem[];
    T (*rows)[18 * ROW] = reinterpret_cast<T (*)[18 * ROW]>(smem);   // of each warp
    const I Y = (I)g.nxp, Z = (I)g.plane;
    // A block takes a contiguous range of particles: with particles in about the order of their cells
    // it then finds the field rows of one sweep in L1 for the next (bunch: 214 us, in
    // interleaved sweeps 260).  The loop bound is block-uniform, so every lane runs every iteration.
    const long long per = ((a.n + gridDim.x - 1) / gridDim.x + 31) / 32 * 32;
    const long long first = blockIdx.x * per, end = first + per < a.n ? first + per : a.n;
    for (long long base = first; base < end; base += PUSH<T, MEAN>) {
        const long long p = base + threadIdx.x;
        bool live = p < end;
        T x = 0, y = 0, z = 0, ux = 0, uy = 0, uz = 0;
        if (live) {
            x = a.x[0][p]; y = a.x[1][p]; z = a.x[2][p];
            ux = a.u[0][p]; uy = a.u[1][p]; uz = a.u[2][p];
            if (!finite3(x, y, z) || !finite3(ux, uy, uz)) {
                atomicOr(a.err, ERR_PARTICLE);
                live = false;
                x = y = z = T(0);   // a harmless cell for the idle lane
            } else {
                x = into_box(x, a.L[0]); y = into_box(y, a.L[1]); z = into_box(z, a.L[2]);
            }
        }
        const Cell<T> cx = cell_of(x * a.inv_dx[0]), cy = cell_of(y * a.inv_dx[1]),
                      cz = cell_of(z * a.inv_dx[2]);
        T u1x = 0, u1y = 0, u1z = 0, x1 = 0, y1 = 0, z1 = 0;
        if (live) {
            // ---- gather at x^n: columns f + st and rows f + st reach at most one past either end,
            // which the ghosts hold
            const int k0 = cz.f >= g.nz ? cz.f - g.nz : cz.f;
            const I zn0 = (I)k0 * Z, zn1 = (I)(k0 + 1 == g.nz ? 0 : k0 + 1) * Z;
            const I zs0 = cz.st ? (I)(k0 == 0 ? g.nz - 1 : k0 - 1) * Z : zn0, zs1 = cz.st ? zn0 : zn1;
            const I xn = (I)(cx.f + PX), xs = xn + cx.st;
            const I yn = (I)(cy.f + PY) * Y, ys = yn + (cy.st ? -Y : 0);
            auto mix = [](T lo, T hi, T w) { return fma(w, hi, (T(1) - w) * lo); };
            auto gather = [&](const T* __restrict__ F, I o, T wx, T wy, I za, I zb, T wz) {
                const T *p0 = F + (o + za), *p1 = F + (o + zb);
                return mix(mix(mix(p0[0], p0[1], wx), mix(p0[Y], p0[Y + 1], wx), wy),
                           mix(mix(p1[0], p1[1], wx), mix(p1[Y], p1[Y + 1], wx), wy), wz);
            };
            auto gatherB = [&](int c, I o, T wx, T wy, I za, I zb, T wz) {
                if (MEAN) return gather(a.B0[c], o, wx, wy, za, zb, wz);
                const T *p0 = a.B0[c] + (o + za), *p1 = a.B0[c] + (o + zb);
                const T *q0 = a.B1[c] + (o + za), *q1 = a.B1[c] + (o + zb);
                auto m = [](T u, T v) { return T(0.5) * (u + v); };
                return mix(mix(mix(m(p0[0], q0[0]), m(p0[1], q0[1]), wx),
                               mix(m(p0[Y], q0[Y]), m(p0[Y + 1], q0[Y + 1]), wx), wy),
                           mix(mix(m(p1[0], q1[0]), m(p1[1], q1[1]), wx),
                               mix(m(p1[Y], q1[Y]), m(p1[Y + 1], q1[Y + 1]), wx), wy), wz);
            };
            const T Ex = gather(a.E[0], xs + yn, cx.ws, cy.w, zn0, zn1, cz.w);
            const T Ey = gather(a.E[1], xn + ys, cx.w, cy.ws, zn0, zn1, cz.w);
            const T Ez = gather(a.E[2], xn + yn, cx.w, cy.w, zs0, zs1, cz.ws);
            const T Bx = gatherB(0, xn + ys, cx.w, cy.ws, zs0, zs1, cz.ws);
            const T By = gatherB(1, xs + yn, cx.ws, cy.w, zs0, zs1, cz.ws);
            const T Bz = gatherB(2, xs + ys, cx.ws, cy.ws, zn0, zn1, cz.w);
            // ---- Boris push u^{n-1/2} -> u^{n+1/2}
            const T h = a.h;
            const T umx = ux + h * Ex, umy = uy + h * Ey, umz = uz + h * Ez;
            const T hg = h / sqrt(T(1) + umx * umx + umy * umy + umz * umz);
            const T tx = hg * Bx, ty = hg * By, tz = hg * Bz;
            const T s2 = T(2) / (T(1) + (tx * tx + ty * ty + tz * tz));
            const T upx = umx + (umy * tz - umz * ty);
            const T upy = umy + (umz * tx - umx * tz);
            const T upz = umz + (umx * ty - umy * tx);
            u1x = umx + s2 * (upy * tz - upz * ty) + h * Ex;
            u1y = umy + s2 * (upz * tx - upx * tz) + h * Ey;
            u1z = umz + s2 * (upx * ty - upy * tx) + h * Ez;
            const T dg = a.dt / sqrt(T(1) + u1x * u1x + u1y * u1y + u1z * u1z);
            x1 = x + dg * u1x; y1 = y + dg * u1y; z1 = z + dg * u1z;
            // ---- new state, positions wrapped into [0, L)
            auto wrapped = [](T v, T L) { return v < T(0) ? v + L : v >= L ? v - L : v; };
            a.x[0][p] = wrapped(x1, a.L[0]);
            a.x[1][p] = wrapped(y1, a.L[1]);
            a.x[2][p] = wrapped(z1, a.L[2]);
            a.u[0][p] = u1x; a.u[1][p] = u1y; a.u[2][p] = u1z;
        }
        // ---- Esirkepov current: -dt J^{n+1/2} into E^{n+1}
        int ix[3], jy[3], kz[3];
        const Move<T, I> X = move_of<T, I>(cx, x1 * a.inv_dx[0], g.nx, (I)1, (I)PX, ix);
        const Move<T, I> Ym = move_of<T, I>(cy, y1 * a.inv_dx[1], g.ny, Y, (I)PY * Y, jy);
        const Move<T, I> Zm = move_of<T, I>(cz, z1 * a.inv_dx[2], g.nz, Z, (I)0, kz);
        T sy[3], sz[3];
#pragma unroll
        for (int q = 0; q < 3; ++q) {
            sy[q] = SP ? a.spy[jy[q]] : T(1);
            sz[q] = SP ? a.spz[kz[q]] : T(1);
        }
        const int f0x = __shfl_sync(FULL, cx.f, 0), f0y = __shfl_sync(FULL, cy.f, 0),
                  f0z = __shfl_sync(FULL, cz.f, 0);
        bool uni = __all_sync(FULL, live && cx.f == f0x && cy.f == f0y && cz.f == f0z);
        if (uni) {
            // the further nodes and faces of the axes on which lanes change their cell, all the same way
            const unsigned px = __ballot_sync(FULL, X.s > 0), mx = __ballot_sync(FULL, X.s < 0);
            const unsigned py = __ballot_sync(FULL, Ym.s > 0), my = __ballot_sync(FULL, Ym.s < 0);
            const unsigned pz = __ballot_sync(FULL, Zm.s > 0), mz = __ballot_sync(FULL, Zm.s < 0);
            uni = (px == 0 || mx == 0) && (py == 0 || my == 0) && (pz == 0 || mz == 0);
            if (uni) {
                const bool xx = (px | mx) != 0, xy = (py | my) != 0, xz = (pz | mz) != 0;
                // node offsets shared by the warp: the third from a lane that changes its cell
                auto third = [&](I own, unsigned ball) {
                    return __shfl_sync(FULL, own, ball ? __ffs(ball) - 1 : 0);
                };
                const I ox[3] = {X.o[0], X.o[1], third(X.o[2], px | mx)};
                const I oy[3] = {Ym.o[0], Ym.o[1], third(Ym.o[2], py | my)};
                const I oz[3] = {Zm.o[0], Zm.o[1], third(Zm.o[2], pz | mz)};
                T* sm = rows[threadIdx.x >> 5];
                // the layers' factors; a lane that stays in its cell has zeros at the further ones
                const T syx = Ym.s > 0 ? sy[1] : sy[2], szx = Zm.s > 0 ? sz[1] : sz[2];
                deposit_shared<SP>(a.Eout[0], X, Ym, Zm, a.escale[0], xx, xy, xz, px ? ox[1] : ox[2], oy,
                                   oz, [&](int, int b, int c) { return sy[b] * sz[c]; }, sm);
                deposit_shared<SP>(a.Eout[1], Ym, X, Zm, a.escale[1], xy, xx, xz, py ? oy[1] : oy[2], ox,
                                   oz, [&](int u, int, int c) { return (u ? syx : sy[0]) * sz[c]; }, sm);
                deposit_shared<SP>(a.Eout[2], Zm, X, Ym, a.escale[2], xz, xx, xy, pz ? oz[1] : oz[2], ox,
                                   oy, [&](int u, int, int c) { return sy[c] * (u ? szx : sz[0]); }, sm);
                continue;
            }
        }
        if (!live) continue;
        deposit_lane<SP>(a, X, Ym, Zm, sy, sz);
    }
}

// out = (b0 + b1) / 2 over n elements (whole padded arrays, images included; n is a multiple of 4)
template <typename T>
__global__ void __launch_bounds__(THREADS)
bmean_kernel(long long n, const T* __restrict__ b0, const T* __restrict__ b1, T* __restrict__ out) {
    struct alignas(16) V4 {
        T v[4];
    };
    for (long long t = (long long)blockIdx.x * THREADS + threadIdx.x; t < n / 4;
         t += (long long)gridDim.x * THREADS) {
        const V4 p = reinterpret_cast<const V4*>(b0)[t], q = reinterpret_cast<const V4*>(b1)[t];
        V4 r;
#pragma unroll
        for (int u = 0; u < 4; ++u) r.v[u] = T(0.5) * (p.v[u] + q.v[u]);
        reinterpret_cast<V4*>(out)[t] = r;
    }
}

// Every ghost cell of three padded arrays takes the value of the owned cell it is the image of, four
// cells of a row at a time: PX = 4 and nx % 4 = 0, so the ghost columns of a row are one group
// each, and so is every group's source.  Bound: HBM (strided groups) and launch.  Us, a cell at a
// time and this: 512 x 256 x 256 18.6 / 13.6, 128^3 5.1 / 3.4.
template <typename T>
struct alignas(16) Group {
    T v[4];
};
static_assert(PX == 4, "the ghost columns of one side are one group");

template <typename T>
__global__ void __launch_bounds__(THREADS)
refresh_kernel(Geom g, T* __restrict__ F0, T* __restrict__ F1, T* __restrict__ F2) {
    const int nv = g.nxp / 4, own = g.nx / 4;                // groups of a padded row, of its owned cells
    const long long per_plane = 2LL * PY * nv + 2LL * g.ny;   // ghost rows, then two groups a row
    const long long total = per_plane * g.nz;
    for (long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x; t < total;
         t += (long long)gridDim.x * blockDim.x) {
        const int k = (int)(t / per_plane), r = (int)(t - (long long)k * per_plane);
        int v, jp;   // group and row of the ghosts
        if (r < 2 * PY * nv) {
            const int row = r / nv;
            v = r - row * nv;
            jp = row < PY ? row : g.ny + row;   // rows 0 .. PY-1 and ny+PY .. ny+2PY-1
        } else {
            const int q = r - 2 * PY * nv;
            jp = PY + (q >> 1);
            v = q & 1 ? nv - 1 : 0;
        }
        const int vs = v == 0 ? own : v == nv - 1 ? 1 : v;   // the owned group with these values
        const int js = wrapi(jp - PY, g.ny) + PY;
        const long long plane = (long long)k * g.nyp;
        const long long dst = ((plane + jp) * g.nxp) / 4 + v, src = ((plane + js) * g.nxp) / 4 + vs;
        Group<T>* const F[3] = {reinterpret_cast<Group<T>*>(F0), reinterpret_cast<Group<T>*>(F1),
                                reinterpret_cast<Group<T>*>(F2)};
        Group<T> x[3];
#pragma unroll
        for (int c = 0; c < 3; ++c) x[c] = F[c][src];
#pragma unroll
        for (int c = 0; c < 3; ++c) F[c][dst] = x[c];
    }
}

template <typename T>
__global__ void __launch_bounds__(THREADS)
rho_kernel(Geom g, const T* __restrict__ x0, const T* __restrict__ x1, const T* __restrict__ x2,
           long long n, T ix, T iy, T iz, T Lx, T Ly, T Lz, T scale, T* __restrict__ rho, int* err) {
    for (long long p = (long long)blockIdx.x * blockDim.x + threadIdx.x; p < n;
         p += (long long)gridDim.x * blockDim.x) {
        T x = x0[p], y = x1[p], z = x2[p];
        if (!finite3(x, y, z)) {
            atomicOr(err, ERR_PARTICLE);
            continue;
        }
        x = into_box(x, Lx); y = into_box(y, Ly); z = into_box(z, Lz);
        const Lin<T> a = lin(x * ix, g.nx), b = lin(y * iy, g.ny), c = lin(z * iz, g.nz);
#pragma unroll
        for (int ia = 0; ia < 2; ++ia)
#pragma unroll
            for (int ib = 0; ib < 2; ++ib)
#pragma unroll
                for (int ic = 0; ic < 2; ++ic) {
                    const T w = (ia ? a.w1 : a.w0) * (ib ? b.w1 : b.w0) * (ic ? c.w1 : c.w0);
                    const long long o = ((long long)(ic ? c.i1 : c.i0) * g.ny + (ib ? b.i1 : b.i0)) * g.nx +
                                        (ia ? a.i1 : a.i0);
                    if (w != T(0)) atomicAdd(rho + o, scale * w);
                }
    }
}

inline unsigned blocks_for(long long n) {
    long long b = (n + THREADS - 1) / THREADS;
    if (b > 152LL * 16) b = 152LL * 16;
    if (b < 1) b = 1;
    return (unsigned)b;
}

}  // namespace picd

template <typename T>
bool pic_mean_prepare() {
    auto set = [](auto kern) {
        return cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                    (int)picd::PUSH_SMEM<T, true>) == cudaSuccess;
    };
    return set(picd::push_kernel<T, true, true, int>) && set(picd::push_kernel<T, true, false, int>) &&
           set(picd::push_kernel<T, true, true, long long>) &&
           set(picd::push_kernel<T, true, false, long long>);
}
template bool pic_mean_prepare<float>();
template bool pic_mean_prepare<double>();

template <typename T>
void launch_pic_push(const PushArgs<T>& a, bool mean, cudaStream_t st) {
    if (a.n <= 0) return;
    // nine blocks of 256 an SM (three resident; 456, 912, 1368, 4864 blocks: bunch 227, 217, 214, 237
    // us) or one large one (1, 2, 3, 6 an SM: plasma 287, 291, 295, 308 us)
    const int threads = mean ? picd::PUSH<T, true> : picd::PUSH<T, false>;
    const size_t smem = mean ? picd::PUSH_SMEM<T, true> : picd::PUSH_SMEM<T, false>;
    const long long want = (a.n + threads - 1) / threads, most = (threads > picd::THREADS ? 1 : 9) * 152;
    const unsigned blocks = (unsigned)(want < most ? want : most);
    auto go = [&](auto kern) { kern<<<blocks, threads, smem, st>>>(a); };
    const bool sp = a.spy != nullptr;
    auto with = [&](auto idx) {
        using I = decltype(idx);
        if (mean) sp ? go(picd::push_kernel<T, true, true, I>) : go(picd::push_kernel<T, true, false, I>);
        else sp ? go(picd::push_kernel<T, false, true, I>) : go(picd::push_kernel<T, false, false, I>);
    };
    if (a.g.total < (1LL << 31)) with((int)0);
    else with((long long)0);
}

template <typename T>
void launch_bmean(long long n, const T* b0, const T* b1, T* out, cudaStream_t st) {
    picd::bmean_kernel<T><<<picd::blocks_for(n / 4), picd::THREADS, 0, st>>>(n, b0, b1, out);
}
template void launch_bmean<float>(long long, const float*, const float*, float*, cudaStream_t);
template void launch_bmean<double>(long long, const double*, const double*, double*, cudaStream_t);

template <typename T>
void launch_refresh_images(const Geom& g, T* F0, T* F1, T* F2, cudaStream_t st) {
    const long long total = (2LL * PY * (g.nxp / 4) + 2LL * g.ny) * g.nz;
    picd::refresh_kernel<T><<<picd::blocks_for(total), picd::THREADS, 0, st>>>(g, F0, F1, F2);
}

template <typename T>
void launch_deposit_rho(const Geom& g, const T* const x[3], long long n, const T inv_dx[3],
                        const T L[3], T scale, T* rho, int* err, cudaStream_t st) {
    if (n <= 0) return;
    picd::rho_kernel<T><<<picd::blocks_for(n), picd::THREADS, 0, st>>>(
        g, x[0], x[1], x[2], n, inv_dx[0], inv_dx[1], inv_dx[2], L[0], L[1], L[2], scale, rho, err);
}

template void launch_pic_push<float>(const PushArgs<float>&, bool, cudaStream_t);
template void launch_pic_push<double>(const PushArgs<double>&, bool, cudaStream_t);
template void launch_refresh_images<float>(const Geom&, float*, float*, float*, cudaStream_t);
template void launch_refresh_images<double>(const Geom&, double*, double*, double*, cudaStream_t);
template void launch_deposit_rho<float>(const Geom&, const float* const[3], long long,
                                        const float[3], const float[3], float, float*, int*,
                                        cudaStream_t);
template void launch_deposit_rho<double>(const Geom&, const double* const[3], long long,
                                         const double[3], const double[3], double, double*, int*,
                                         cudaStream_t);

}  // namespace fdtd

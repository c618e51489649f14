// Dispersion norm (Sec. 4, Eq. norm) and its exact gradient over a midpoint k-grid.
//
// Per point k (k_i = (m_i + 1/2) pi / (N_i dx_i)):
//   s_i^2 = sin^2(k_i dx_i / 2) / dx_i^2,  c_i = cos(k_i dx_i)
//   S = sum_i s_i^2 A_i,  A_i = alpha_i + delta_i (1 + 2 c_i) + 2 sum_{j != i} beta_ij c_j
//                                                           (Eq. dispersion_relation)
//   omega = (2/dt) asin(dt sqrt S),  r = omega - |k|
//   f  += w r^2
//   df += w 2 r (d omega/d theta),  with d omega/dS = 1/(sqrt S sqrt(1 - dt^2 S)),
//         dS/d beta_ij = 2 s_i^2 (c_j - 1),  dS/d delta_i = 2 s_i^2 (c_i - 1),
//         d omega/d dt = -omega/dt + 2 sqrt S / (dt sqrt(1 - dt^2 S)).
// Everything per point and every accumulation is FP64, and the FP64 pipe (two lanes an SM on this
// part) is the limit, so the work is arranged to need few FP64 instructions (about 40 a point
// where the printed formulas took 109, two square roots, a division and an arcsine among them):
//   - with alpha eliminated and c_i = 1 - 2 dx_i^2 u_i (u_i = s_i^2),
//         S = sum_i u_i - 4 sum_i delta_i dx_i^2 u_i^2 - 4 sum_{i != j} beta_ij dx_j^2 u_i u_j
//     is a quadratic in u_x along a row of constant (k_y, k_z): two multiply-adds a point;
//   - the gradient's sums over a row need only sum h, sum h u_x and sum h u_x^2 with
//     h = r (d omega/dS); the factors of the row are applied once a row segment;
//   - square roots come as x rsqrt(x) from the hardware's approximate rsqrt and one third-order
//     step (error below 2^-58 before rounding), reciprocal square roots with two more operations;
//   - omega = (2/dt) theta with sin theta = x, cos theta = sqrt(1 - x^2): the nearest angle of a
//     256-step table (its index from FP32) plus the arcsine series of the small difference;
//   - the weights depend on the row, or (cone) on the row and a first index: points of weight zero
//     cost nothing.
// 256^3 points: 3350 us with the printed formulas, 1315 us here (floor of 42 FP64 instructions a
// point on that pipe: 1220 us); 30 degree cone 1446 -> 237 us; 256^2 points, launch-bound, 46 us in
// three kernels -> 19 us in two (2 us of it the blocks' sums, 3 us the last block's: 7 us when it
// read the partials one quantity after another).
// A thread takes one row segment at a time, neighbouring threads neighbouring k_y; a block's sums
// are taken once, and the block that arrives last adds the blocks' partials in a fixed order
// (deterministic result).
#include <math_constants.h>

#include <cmath>

#include "fdtd_internal.cuh"

#include <algorithm>

namespace fdtd {

constexpr int NQ = 11;   // f, dbeta x 6 (xy, xz, yx, yz, zx, zy), ddelta x 3, ddt
constexpr int NORM_THREADS = 256;

struct NormParams {
    double alpha[3], delta[3], beta[3][3];
    double dt;
    int N[3];
    int dims;
    int weight;
    double wparam;   // cone: cos(half-angle); gauss: dy / width
    long long npts;
    double pref;     // prod(dx) * prod(pi / (N_i dx_i))
    // constants of the row polynomial S = P + u_x (Q + R u_x) and of the gradient factors:
    //   P = u_y + u_z + py u_y^2 + pz u_z^2 + pyz u_y u_z,  Q = 1 + qy u_y + qz u_z
    double py, pz, pyz, qy, qz, R;
    double m2dx2[3];             // -2 dx_i^2
    double two_over_dt, four_over_dt2;
    int seg_len, nseg;   // points of a row segment, segments of a row
};

// Table of one call: (k, s^2) of every axis value, then the angle table, then the block ticket.
constexpr int ANGLES = 256;   // steps of the angle table over [0, pi/2]
struct alignas(16) Angle {
    double sn, cs, th, pad;
};

__global__ void norm_table_kernel(NormParams p, double dx0, double dx1, double dx2,
                                  double2* __restrict__ tab, Angle* __restrict__ ang,
                                  unsigned* __restrict__ ticket) {
    int t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t == 0) *ticket = 0;
    const double dxa[3] = {dx0, dx1, dx2};
    for (int a = 0; a < 3; ++a) {
        if (t < p.N[a]) {
            double k = 0.0;
            if (a < p.dims) k = (t + 0.5) * M_PI / (p.N[a] * dxa[a]);
            const double sn = sin(0.5 * k * dxa[a]) / dxa[a];
            tab[t] = make_double2(k, sn * sn);
            return;
        }
        t -= p.N[a];
        tab += p.N[a];
    }
    if (t <= ANGLES) {
        Angle e;
        e.th = t * (0.5 * M_PI / ANGLES);
        sincos(e.th, &e.sn, &e.cs);
        e.pad = 0.0;
        ang[t] = e;
    }
}

// sqrt(a), and 1 / sqrt(a), of a normal positive a: the hardware's approximation r (2^-20 or
// better) and one third-order step, 1/sqrt(a) = r (1 - e)^(-1/2), e = 1 - a r^2
__device__ __forceinline__ double rsqrt_seed(double a) {
    double r;
    asm("rsqrt.approx.ftz.f64 %0, %1;" : "=d"(r) : "d"(a));
    return r;
}
__device__ __forceinline__ double root(double a) {
    const double r = rsqrt_seed(a), s = a * r, e = fma(-s, r, 1.0);
    return fma(e * s, fma(e, 0.375, 0.5), s);
}
__device__ __forceinline__ void root_both(double a, double& s, double& rs) {
    const double r = rsqrt_seed(a), s0 = a * r, e = fma(-s0, r, 1.0), t = fma(e, 0.375, 0.5);
    s = fma(e * s0, t, s0);
    rs = fma(e * r, t, r);
}

// a positive double between 2^-126 and 2^127, and its value in single precision (truncated), by integer
// shifts
__device__ __forceinline__ bool narrows(double x) {
    return (unsigned)__double2hiint(x) - 0x38100000u < 0x0fd00000u;
}
__device__ __forceinline__ float narrow(double x) {
    return __uint_as_float(((unsigned)(__double2hiint(x) - 0x38000000) << 3) |
                           ((unsigned)__double2loint(x) >> 29));
}

// the cone's weight at (kx, ky, kz): single precision decides away from the cone's surface (its
// error is below 1e-6 of either side), the FP64 expression next to it and outside the float range.
// t2: ky^2 + kz^2 of the row in single precision, NaN where that cannot be formed
__device__ __forceinline__ float cone_row(double ky, double kz) {
    if ((ky != 0.0 && !narrows(ky)) || (kz != 0.0 && !narrows(kz))) return CUDART_NAN_F;
    const float y = ky > 0.0 ? narrow(ky) : 0.0f, z = kz > 0.0 ? narrow(kz) : 0.0f;
    return y * y + z * z;
}
__device__ __forceinline__ bool in_cone(double kx, double ky, double kz, float t2, double cos_half) {
    if (narrows(kx)) {
        const float x = narrow(kx), n = sqrtf(x * x + t2), c = n * (float)cos_half;
        if (n > 1e-15f && n < 1e15f && fabsf(x - c) > 1e-5f * n) return x > c;
    }
    return kx >= sqrt(kx * kx + ky * ky + kz * kz) * cos_half;
}

constexpr int NORM_BLOCK = 128;

// Sums of v over the block, quantity q returned by thread q < NQ.  Through shared memory, one
// warp a quantity: 8 FP64 additions a warp and quantity instead of 5 for each of 11 in every warp.
__device__ __forceinline__ double norm_block_sum(const double (&v)[NQ], double (*sm)[NORM_BLOCK],
                                                 double* res) {
    __syncthreads();
#pragma unroll
    for (int q = 0; q < NQ; ++q) sm[q][threadIdx.x] = v[q];
    __syncthreads();
    constexpr int WARPS = NORM_BLOCK / 32, R = (NQ + WARPS - 1) / WARPS;
    const int w = threadIdx.x >> 5, l = threadIdx.x & 31;
    double x[R];   // the warp's quantities together: independent chains of FP64 additions
#pragma unroll
    for (int r = 0; r < R; ++r) {
        const int q = min(w + r * WARPS, NQ - 1);
        x[r] = (sm[q][l] + sm[q][l + 32]) + (sm[q][l + 64] + sm[q][l + 96]);
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1)
#pragma unroll
        for (int r = 0; r < R; ++r) x[r] += __shfl_down_sync(0xffffffffu, x[r], o);
#pragma unroll
    for (int r = 0; r < R; ++r)
        if (l == 0 && w + r * WARPS < NQ) res[w + r * WARPS] = x[r];
    __syncthreads();
    return threadIdx.x < NQ ? res[threadIdx.x] : 0.0;
}

__global__ void __launch_bounds__(NORM_BLOCK)
norm_kernel(NormParams p, const double2* __restrict__ tab, const Angle* __restrict__ ang,
            double* __restrict__ part, unsigned* __restrict__ ticket, double* __restrict__ out) {
    double acc[NQ];
#pragma unroll
    for (int q = 0; q < NQ; ++q) acc[q] = 0.0;
    const double2* ty = tab + p.N[0];
    const double2* tz = ty + p.N[1];
    const long long items = (long long)p.N[1] * p.N[2] * p.nseg;
    for (long long t = (long long)blockIdx.x * NORM_BLOCK + threadIdx.x; t < items;
         t += (long long)gridDim.x * NORM_BLOCK) {
        int my, mz, m0;
        if (items <= 0x7fffffff) {
            const int r = (int)t / p.N[1];
            my = (int)t - r * p.N[1];
            mz = r / p.nseg;
            m0 = (r - mz * p.nseg) * p.seg_len;
        } else {
            const long long r = t / p.N[1];
            my = (int)(t - r * p.N[1]);
            mz = (int)(r / p.nseg);
            m0 = (int)(r - (long long)mz * p.nseg) * p.seg_len;
        }
        const int m1 = min(m0 + p.seg_len, p.N[0]);
        const double2 y = ty[my], z = tz[mz];
        double w = 1.0;
        if (p.weight == FDTD_W_CONE_X) {
            // along the row the weight is 0 up to an index and 1 from it on
            const float t2 = cone_row(y.x, z.x);
            if (!in_cone(tab[m1 - 1].x, y.x, z.x, t2, p.wparam)) continue;
            if (!in_cone(tab[m0].x, y.x, z.x, t2, p.wparam)) {
                int lo = m0, hi = m1 - 1;   // outside at lo, inside at hi
                while (hi - lo > 1) {
                    const int mid = (lo + hi) >> 1;
                    if (in_cone(tab[mid].x, y.x, z.x, t2, p.wparam)) hi = mid;
                    else lo = mid;
                }
                m0 = hi;
            }
        } else if (p.weight == FDTD_W_GAUSS_Y) {
            const double u = y.x * p.wparam;
            w = exp(-u * u);
            if (w == 0.0) continue;
        }
        // S = P + u (Q + R u) along the row
        const double uy = y.y, uz = z.y;
        const double P = (uy + uz) + fma(uy, fma(p.py, uy, p.pyz * uz), p.pz * uz * uz);
        const double Q = fma(p.qy, uy, fma(p.qz, uz, 1.0));
        const double R = p.R;
        const double kt2 = y.x * y.x + z.x * z.x;
        double F = 0.0, H0 = 0.0, H1 = 0.0, H2 = 0.0, D = 0.0;
        for (int m = m0; m < m1; ++m) {
            const double2 e = tab[m];
            const double u = e.y;
            const double S = fma(u, fma(R, u, Q), P);   // x = dt sqrt(S) = sin(omega dt / 2)
            double sq, rs;
            root_both(S, sq, rs);
            double x = p.dt * sq;
            const double q = fma(-x, x, 1.0);
            double c, rc, th;
            // S between 2^-126 and 2^127, x and q positive, between 2^-63 and 1: integer comparisons
            if (narrows(S) &&
                (unsigned)__double2hiint(x) - 0x3c000000u < 0x04000000u &&
                (unsigned)__double2hiint(q) - 0x3c000000u < 0x04000000u) {
                root_both(q, c, rc);
                const Angle* A = ang + min(__float2int_rn(asinf(narrow(x)) *
                                                          (float)(2.0 * ANGLES / M_PI)), ANGLES);
                // sin(theta - theta_i), at most 0.0031: its arcsine to 2^-53
                const double d = x * A->cs - c * A->sn, d2 = d * d;
                th = A->th + fma(d * d2, fma(d2, 3.0 / 40.0, 1.0 / 6.0), d);
            } else {   // on the edge of the stable range, or beyond: the plain functions
                sq = sqrt(S);
                x = p.dt * sq;
                c = sqrt(fma(-x, x, 1.0));
                rs = 1.0 / sq;
                rc = 1.0 / c;
                th = asin(x);
            }
            const double res = fma(p.two_over_dt, th, -root(fma(e.x, e.x, kt2)));
            F = fma(res, res, F);
            const double h = res * (rs * rc), hu = h * u;   // r d omega/dS
            H0 += h;
            H1 += hu;
            H2 = fma(hu, u, H2);
            D = fma(res, fma(x, rc, -th), D);
        }
        // w 2 r d omega/dS times dS/dtheta, c_i - 1 = -2 dx_i^2 u_i
        const double s = 4.0 * w, cx = p.m2dx2[0], cy = p.m2dx2[1] * uy, cz = p.m2dx2[2] * uz;
        H0 *= s;
        H1 *= s;
        H2 *= s;
        acc[0] = fma(w, F, acc[0]);
        // beta: (x,y), (x,z), (y,x), (y,z), (z,x), (z,y)
        acc[1] = fma(H1, cy, acc[1]);
        acc[2] = fma(H1, cz, acc[2]);
        acc[3] = fma(H1 * uy, cx, acc[3]);
        acc[4] = fma(H0 * uy, cz, acc[4]);
        acc[5] = fma(H1 * uz, cx, acc[5]);
        acc[6] = fma(H0 * uz, cy, acc[6]);
        acc[7] = fma(H2, cx, acc[7]);
        acc[8] = fma(H0 * uy, cy, acc[8]);
        acc[9] = fma(H0 * uz, cz, acc[9]);
        acc[10] = fma(w * p.four_over_dt2, D, acc[10]);
    }
    __shared__ double sm[NQ][NORM_BLOCK];
    __shared__ double res[NQ];
    __shared__ bool last;
    const double mine = norm_block_sum(acc, sm, res);
    if (threadIdx.x < NQ) {
        part[(long long)threadIdx.x * gridDim.x + blockIdx.x] = mine;
        __threadfence();
    }
    __syncthreads();
    if (threadIdx.x == 0) last = atomicAdd(ticket, 1u) == gridDim.x - 1;
    __syncthreads();
    if (!last) return;
    __threadfence();
#pragma unroll
    for (int q = 0; q < NQ; ++q) acc[q] = 0.0;
    for (unsigned b = threadIdx.x; b < gridDim.x; b += NORM_BLOCK)
#pragma unroll
        for (int q = 0; q < NQ; ++q)   // the quantities' loads in flight together
            acc[q] += __ldcg(part + (long long)q * gridDim.x + b);
    const double total = norm_block_sum(acc, sm, res);
    // out[14] = {f, dbeta 3x3 row-major, ddelta 3, ddt}
    const int slot[NQ] = {0, 1 + 1, 1 + 2, 1 + 3, 1 + 5, 1 + 6, 1 + 7, 10, 11, 12, 13};
#pragma unroll
    for (int q = 0; q < NQ; ++q)
        if (threadIdx.x == q) out[slot[q]] = p.pref * total;
    if (threadIdx.x < 3) out[1 + 4 * threadIdx.x] = 0.0;   // diagonal of d/d beta
}

// out[14] = {f, dbeta 3x3 row-major, ddelta 3, ddt}
__global__ void norm_final_kernel(const double* __restrict__ part, int nblocks, double pref,
                                  double* __restrict__ out) {
    __shared__ double red[NQ][32];
    const int q = threadIdx.y, l = threadIdx.x;
    double v = 0.0;
    for (int b = l; b < nblocks; b += 32) v += part[(long long)b * NQ + q];
    red[q][l] = v;
    __syncthreads();
    if (l == 0) {
        double s = 0.0;
        for (int t = 0; t < 32; ++t) s += red[q][t];
        s *= pref;
        // map q -> out slot
        const int slot[NQ] = {0, 1 + 1, 1 + 2, 1 + 3, 1 + 5, 1 + 6, 1 + 7, 10, 11, 12, 13};
        out[slot[q]] = s;
    }
    if (q == 0 && l < 3) out[1 + 4 * l] = 0.0;   // diagonal of d/d beta
}

int norm_blocks(long long npts) {
    long long b = (npts + NORM_THREADS - 1) / NORM_THREADS;
    if (b > 152 * 16) b = 152 * 16;
    if (b < 1) b = 1;
    return (int)b;
}

// Two blocks of four warps an SM keep the FP64 pipe busy and leave few block sums to take; the
// count is odd so that a block's items do not all come from the same part of the rows (with the
// cone weight only some parts hold work).
constexpr int NORM_GRID = 2 * 152 - 1;

size_t norm_scratch_doubles(const int N[3]) {
    return (size_t)2 * (N[0] + N[1] + N[2]) + 4 * (ANGLES + 1) + (size_t)NORM_GRID * NQ + 14 + 2;
}

static void fill_params(NormParams& p, const double alpha[3], const double beta[3][3],
                        const double delta[3], double dt, const double dx[3], int dims,
                        const int N[3], int weight, double wparam) {
    for (int i = 0; i < 3; ++i) {
        p.alpha[i] = alpha[i];
        p.delta[i] = delta[i];
        for (int j = 0; j < 3; ++j) p.beta[i][j] = beta[i][j];
        p.N[i] = i < dims ? N[i] : 1;
    }
    p.dt = dt;
    p.dims = dims;
    p.weight = weight;
    if (weight == FDTD_W_CONE_X) p.wparam = cos(wparam);
    else if (weight == FDTD_W_GAUSS_Y) p.wparam = dx[1] / wparam;
    else p.wparam = 0.0;
    p.npts = (long long)p.N[0] * p.N[1] * p.N[2];
    p.pref = 1.0;
    for (int i = 0; i < dims; ++i) p.pref *= dx[i] * (M_PI / (p.N[i] * dx[i]));
    double d2[3];   // absent axes contribute nothing
    for (int i = 0; i < 3; ++i) {
        d2[i] = i < dims ? dx[i] * dx[i] : 0.0;
        p.m2dx2[i] = -2.0 * d2[i];
    }
    const double m4 = -4.0;
    p.py = m4 * delta[1] * d2[1];
    p.pz = m4 * delta[2] * d2[2];
    p.pyz = m4 * (beta[1][2] * d2[2] + beta[2][1] * d2[1]);
    p.qy = m4 * (beta[0][1] * d2[1] + beta[1][0] * d2[0]);
    p.qz = m4 * (beta[0][2] * d2[2] + beta[2][0] * d2[0]);
    p.R = m4 * delta[0] * d2[0];
    p.two_over_dt = 2.0 / dt;
    p.four_over_dt2 = 4.0 / (dt * dt);
}

// Runs the two kernels on `st` using `scratch` (norm_scratch_doubles() doubles);
// the 14 results land at host_out (device address of pinned host memory) or, if that is NULL, in
// scratch's last 16 entries, returned via *out_dev.
// Segment length: one warp a scheduler (152 x 4 x 32 threads) saturates the FP64 pipe, so few
// points are cut into that many segments of at least 4 (256^2 points: 17.4 us with 4, 22 with 2,
// 35 with 16), many into segments of 64 (256^3: 1284 us, 16: 1310); of 16 with the cone weight, whose
// rows differ in work (231 us, 64: 295).
void launch_disp_norm(const double alpha[3], const double beta[3][3], const double delta[3],
                      double dt, const double dx[3], int dims, const int N[3], int weight,
                      double wparam, double* scratch, double* host_out, double** out_dev,
                      cudaStream_t st) {
    NormParams p;
    fill_params(p, alpha, beta, delta, dt, dx, dims, N, weight, wparam);
    const long long per = (p.npts + 152 * 128 - 1) / (152 * 128);
    p.seg_len = (int)std::min<long long>(std::max<long long>(per, 4), weight == FDTD_W_CONE_X ? 16 : 64);
    p.nseg = (p.N[0] + p.seg_len - 1) / p.seg_len;
    const long long lines = (long long)p.N[0] + p.N[1] + p.N[2];
    const long long items = (long long)p.N[1] * p.N[2] * p.nseg;
    double2* tab = (double2*)scratch;
    Angle* ang = (Angle*)(tab + lines);
    double* part = (double*)(ang + ANGLES + 1);
    double* out = part + (size_t)NORM_GRID * NQ;
    unsigned* ticket = (unsigned*)(out + 14);
    const long long entries = lines + ANGLES + 1;
    norm_table_kernel<<<(unsigned)((entries + 63) / 64), 64, 0, st>>>(p, dx[0], dx[1], dx[2], tab, ang,
                                                                      ticket);
    const int nb = (int)std::min<long long>((items + NORM_BLOCK - 1) / NORM_BLOCK, NORM_GRID);
    if (host_out != nullptr) out = host_out;
    // (no dependent launch: blocks placed while the table's still run share the SMs unevenly, a whole
    // call of the cone 252 -> 302 us, of 256^3 1330 -> 1337 to 1617, against 1.5 us gained on 256^2)
    norm_kernel<<<nb, NORM_BLOCK, 0, st>>>(p, tab, ang, part, ticket, out);
    *out_dev = out;
}

}  // namespace fdtd

namespace fdtd {

// omega(k) of Eq. (dispersion_relation) at n arbitrary wave vectors (FP64 per point).
__global__ void omega_kernel(NormParams p, double dx0, double dx1, double dx2,
                             const double* __restrict__ k, int n, double* __restrict__ out) {
    const int t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= n) return;
    const double dxa[3] = {dx0, dx1, dx2};
    double s2[3], c[3];
    for (int i = 0; i < 3; ++i) {
        const double ki = i < p.dims ? k[3 * t + i] : 0.0;
        const double sn = sin(0.5 * ki * dxa[i]) / dxa[i];
        s2[i] = sn * sn;
        c[i] = cos(ki * dxa[i]);
    }
    double S = 0.0;
    for (int i = 0; i < 3; ++i) {
        double A = p.alpha[i] + p.delta[i] * (1.0 + 2.0 * c[i]);
        for (int j = 0; j < 3; ++j)
            if (j != i) A += 2.0 * p.beta[i][j] * c[j];
        S += s2[i] * A;
    }
    out[t] = 2.0 / p.dt * asin(p.dt * sqrt(S));
}

void launch_omega(const double alpha[3], const double beta[3][3], const double delta[3], double dt,
                  const double dx[3], int dims, const double* k_dev, int n, double* out_dev,
                  cudaStream_t st) {
    NormParams p;
    for (int i = 0; i < 3; ++i) {
        p.alpha[i] = alpha[i];
        p.delta[i] = delta[i];
        for (int j = 0; j < 3; ++j) p.beta[i][j] = beta[i][j];
    }
    p.dt = dt;
    p.dims = dims;
    omega_kernel<<<(n + 127) / 128, 128, 0, st>>>(p, dx[0], dx[1], dx[2], k_dev, n, out_dev);
}

}  // namespace fdtd

namespace fdtd {

// ---- group-velocity norm (the conclusions' proposal; this library's reading) ----------------
// f_g = prefactor * sum w (|d omega/dk| - 1)^2 on the same midpoint grid, with
//   A_i = alpha_i + delta_i (1 + 2 c_i) + 2 sum_{j != i} beta_ij c_j       (as in norm_kernel)
//   G_m = dS/dk_m = sin(k_m dx_m)/(2 dx_m) A_m - 2 dx_m sin(k_m dx_m) (delta_m s_m^2
//                                                    + sum_{i != m} beta_im s_i^2)
//   |v_g| = w_S |G|,  w_S = 1 / (sqrt(S) sqrt(1 - dt^2 S)),
// and the gradient by the chain rule (w_SS = -w_S^3 (1 - 2 dt^2 S) / 2, d w_S/d dt = w_S^3 dt S^2):
//   d|v_g| = w_SS dS |G| + w_S (G . dG) / |G|, with dS/d beta_ij = 2 s_i^2 (c_j - 1),
//   dS/d delta_i = 2 s_i^2 (c_i - 1), dG_m/d beta_ij = [m=i] sin_i (c_j - 1)/dx_i
//   - [m=j] 2 dx_j sin_j s_i^2, dG_m/d delta_i = [m=i] (sin_i (c_i - 1)/dx_i - 2 dx_i sin_i s_i^2).
// FP64 throughout; per-block partials and the fixed-order final sum of norm_kernel.

struct GroupParams {
    NormParams n;
    double dx[3];
};

__global__ void group_table_kernel(GroupParams p, double* __restrict__ tab) {
    // tab layout: for axis a: [k], [s2], [c], [sin(k dx)] of N_a entries each
    const int t = blockIdx.x * blockDim.x + threadIdx.x;
    int off = 0;
    for (int a = 0; a < 3; ++a) {
        const int n = p.n.N[a];
        if (t < n) {
            double k = 0.0;
            if (a < p.n.dims) k = (t + 0.5) * M_PI / (n * p.dx[a]);
            const double sn = sin(0.5 * k * p.dx[a]) / p.dx[a];
            tab[off + t] = k;
            tab[off + n + t] = sn * sn;
            tab[off + 2 * n + t] = cos(k * p.dx[a]);
            tab[off + 3 * n + t] = sin(k * p.dx[a]);
        }
        off += 4 * n;
    }
}

__global__ void __launch_bounds__(NORM_THREADS)
group_norm_kernel(GroupParams gp, const double* __restrict__ tab, double* __restrict__ partials) {
    const NormParams& p = gp.n;
    double acc[NQ];
#pragma unroll
    for (int q = 0; q < NQ; ++q) acc[q] = 0.0;
    const double* T[3];
    {
        int off = 0;
        for (int a = 0; a < 3; ++a) {
            T[a] = tab + off;
            off += 4 * p.N[a];
        }
    }
    const double dt = p.dt;
    for (long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x; t < p.npts;
         t += (long long)gridDim.x * blockDim.x) {
        const int mi[3] = {(int)(t % p.N[0]), (int)((t / p.N[0]) % p.N[1]),
                           (int)(t / ((long long)p.N[0] * p.N[1]))};
        double k[3], s2[3], c[3], sn[3];
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            const int n = p.N[a];
            k[a] = T[a][mi[a]];
            s2[a] = T[a][n + mi[a]];
            c[a] = T[a][2 * n + mi[a]];
            sn[a] = T[a][3 * n + mi[a]];
        }
        double A[3], S = 0.0;
#pragma unroll
        for (int i = 0; i < 3; ++i) {
            double a = p.alpha[i] + p.delta[i] * (1.0 + 2.0 * c[i]);
#pragma unroll
            for (int j = 0; j < 3; ++j)
                if (j != i) a += 2.0 * p.beta[i][j] * c[j];
            A[i] = a;
            S += s2[i] * a;
        }
        const double kn = sqrt(k[0] * k[0] + k[1] * k[1] + k[2] * k[2]);
        double w = 1.0;
        if (p.weight == FDTD_W_CONE_X) {
            w = (k[0] >= kn * p.wparam) ? 1.0 : 0.0;
        } else if (p.weight == FDTD_W_GAUSS_Y) {
            const double u = k[1] * p.wparam;
            w = exp(-u * u);
        }
        if (w == 0.0) continue;
        double G[3];
#pragma unroll
        for (int m = 0; m < 3; ++m) {
            double tm = p.delta[m] * s2[m];
#pragma unroll
            for (int i = 0; i < 3; ++i)
                if (i != m) tm += p.beta[i][m] * s2[i];
            G[m] = sn[m] / (2.0 * gp.dx[m]) * A[m] - 2.0 * gp.dx[m] * sn[m] * tm;
        }
        const double Gn = sqrt(G[0] * G[0] + G[1] * G[1] + G[2] * G[2]);
        const double wS = 1.0 / (sqrt(S) * sqrt(1.0 - dt * dt * S));
        const double vg = wS * Gn;
        const double r = vg - 1.0;
        acc[0] += w * r * r;
        const double cm = 2.0 * w * r;
        const double wS3 = wS * wS * wS;
        const double wSS = -0.5 * wS3 * (1.0 - 2.0 * dt * dt * S);
        const double a1 = cm * wSS * Gn;   // times dS/dtheta
        const double a2 = cm * wS / Gn;    // times G . dG/dtheta
        // beta: (x,y), (x,z), (y,x), (y,z), (z,x), (z,y)  (same slots as norm_kernel)
        const int bi[6] = {0, 0, 1, 1, 2, 2}, bj[6] = {1, 2, 0, 2, 0, 1};
#pragma unroll
        for (int q = 0; q < 6; ++q) {
            const int i = bi[q], j = bj[q];
            const double dS = 2.0 * s2[i] * (c[j] - 1.0);
            const double GdG = G[i] * sn[i] * (c[j] - 1.0) / gp.dx[i] -
                               G[j] * 2.0 * gp.dx[j] * sn[j] * s2[i];
            acc[1 + q] += a1 * dS + a2 * GdG;
        }
#pragma unroll
        for (int i = 0; i < 3; ++i) {
            const double dS = 2.0 * s2[i] * (c[i] - 1.0);
            const double GdG = G[i] * (sn[i] * (c[i] - 1.0) / gp.dx[i] - 2.0 * gp.dx[i] * sn[i] * s2[i]);
            acc[7 + i] += a1 * dS + a2 * GdG;
        }
        acc[10] += cm * wS3 * dt * S * S * Gn;
    }
    __shared__ double red[NORM_THREADS / 32][NQ];
    const int wq = threadIdx.x >> 5, l = threadIdx.x & 31;
#pragma unroll
    for (int q = 0; q < NQ; ++q) {
        double v = acc[q];
        for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
        if (l == 0) red[wq][q] = v;
    }
    __syncthreads();
    if (threadIdx.x < NQ) {
        double v = 0.0;
        for (int ww = 0; ww < NORM_THREADS / 32; ++ww) v += red[ww][threadIdx.x];
        partials[(long long)blockIdx.x * NQ + threadIdx.x] = v;
    }
}

size_t group_scratch_doubles(const int N[3], long long npts) {
    return (size_t)4 * (N[0] + N[1] + N[2]) + (size_t)norm_blocks(npts) * NQ + 14;
}

void launch_disp_group_norm(const double alpha[3], const double beta[3][3], const double delta[3],
                            double dt, const double dx[3], int dims, const int N[3], int weight,
                            double wparam, double* scratch, double* host_out, double** out_dev,
                            cudaStream_t st) {
    GroupParams gp;
    NormParams& p = gp.n;
    fill_params(p, alpha, beta, delta, dt, dx, dims, N, weight, wparam);
    for (int i = 0; i < 3; ++i) gp.dx[i] = dx[i];
    double* tab = scratch;
    const size_t ntab = (size_t)4 * (p.N[0] + p.N[1] + p.N[2]);
    double* part = scratch + ntab;
    const int nb = norm_blocks(p.npts);
    double* out = part + (size_t)nb * NQ;
    int nmax = p.N[0] > p.N[1] ? p.N[0] : p.N[1];
    if (p.N[2] > nmax) nmax = p.N[2];
    group_table_kernel<<<(nmax + 255) / 256, 256, 0, st>>>(gp, tab);
    group_norm_kernel<<<nb, NORM_THREADS, 0, st>>>(gp, tab, part);
    if (host_out != nullptr) out = host_out;
    norm_final_kernel<<<1, dim3(32, NQ), 0, st>>>(part, nb, p.pref, out);
    *out_dev = out;
}

}  // namespace fdtd

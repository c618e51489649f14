// Diagnostics on the library-owned state (all accumulation in FP64, deterministic).
//
//   energy in a window:   (1/2) sum (E^2 + B^2) dV over cells with i in the periodic x-window
//                          [x_lo, x_lo + x_len) and j, k inside [margin, n - margin);
//   plane-wave amplitude:  sum_cells F_c exp(-i k . r_c), r_c the component's staggered
//                          position (App. A) -- the measured phase advance per step gives the
//                          scheme's omega(k) (Sec. 3), its envelope the group velocity (Sec. 5);
//   energy moments:        sum e (1, cos th, sin th) dV with e = (1/2) F^2 per component at its
//                          staggered position and th = 2 pi x_a / L_a along one axis: the
//                          circular mean atan2(S, C) L_a / 2 pi is the centroid of a wave
//                          packet on the periodic grid, its speed the group velocity (Sec. 5);
//   divergences:           D* . B (Eq. divstarb, extended stencil), Yee D . B and D . E
//                          (Eq. divE) written per cell to a dense caller buffer.
// Partials: one FP64 value (or pair) per block, summed in a fixed order by the last block.
#include <cmath>

#include "fdtd_tma.cuh"

namespace fdtd {

constexpr int DG_THREADS = 256;

int diag_blocks(const Geom& g) {
    const long long cells = (long long)g.nx * g.ny * g.nz;
    long long b = (cells + DG_THREADS - 1) / DG_THREADS;
    if (b > 152 * 8) b = 152 * 8;
    if (b < 1) b = 1;
    return (int)b;
}

// Block sums of v into part, then the grid's sums by the block that arrives last (`ticket` counts
// the blocks and is left at zero for the next launch): always the same order, whichever block it
// is, and no second launch (a one-block summing kernel took 5.6 us after each diagnostic).  ADD:
// out += the sums.
template <int NV, bool ADD = false>
__device__ __forceinline__ void reduce_finish(double (&v)[NV], double* __restrict__ part,
                                              unsigned* __restrict__ ticket, double scale,
                                              double* __restrict__ out) {
    __shared__ double red[DG_THREADS / 32][NV];
    __shared__ bool last;
    const int w = threadIdx.x >> 5, l = threadIdx.x & 31;
    auto block_sum = [&](double (&x)[NV]) {   // result q in thread q
#pragma unroll
        for (int q = 0; q < NV; ++q) {
            double s = x[q];
            for (int o = 16; o > 0; o >>= 1) s += __shfl_down_sync(0xffffffffu, s, o);
            if (l == 0) red[w][q] = s;
        }
        __syncthreads();
        double s = 0.0;
        if (threadIdx.x < NV)
            for (int ww = 0; ww < DG_THREADS / 32; ++ww) s += red[ww][threadIdx.x];
        return s;
    };
    const double mine = block_sum(v);
    if (threadIdx.x < NV) {
        part[(long long)blockIdx.x * NV + threadIdx.x] = mine;
        __threadfence();
    }
    __syncthreads();
    if (threadIdx.x == 0) last = atomicAdd(ticket, 1u) == gridDim.x - 1;
    __syncthreads();
    if (!last) return;
    __threadfence();
    double t[NV];
#pragma unroll
    for (int q = 0; q < NV; ++q) t[q] = 0.0;
    for (int b = threadIdx.x; b < (int)gridDim.x; b += DG_THREADS)
#pragma unroll
        for (int q = 0; q < NV; ++q) t[q] += __ldcg(part + (long long)b * NV + q);
    const double total = block_sum(t);
    if (threadIdx.x < NV) out[threadIdx.x] = (ADD ? out[threadIdx.x] : 0.0) + scale * total;
    if (threadIdx.x == 0) *ticket = 0;
}

template <typename T>
__global__ void __launch_bounds__(DG_THREADS)
energy_kernel(Geom g, FieldSet<T> s, int x_lo, int x_len, int my, int mz, double* part,
              unsigned* ticket, double scale, double* out) {
    double acc[1] = {0.0};
    const long long n = (long long)x_len * (g.ny - 2 * my) * (g.nz - 2 * mz);
    const int ny_in = g.ny - 2 * my;
    for (long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x; t < n;
         t += (long long)gridDim.x * blockDim.x) {
        const int ii = (int)(t % x_len);
        const long long r = t / x_len;
        const int j = my + (int)(r % ny_in);
        const int k = mz + (int)(r / ny_in);
        int i = (x_lo + ii) % g.nx;
        if (i < 0) i += g.nx;
        const long long c = pidx(g, i, j, k);
#pragma unroll
        for (int q = 0; q < 6; ++q) {
            const double v = (double)s.c[q][c];
            acc[0] += v * v;
        }
    }
    reduce_finish<1>(acc, part, ticket, scale, out);
}

// loss += sum_{j,k} (F[x_p, j, k] - T[k][j])^2.  Every value of the plane lies in a sector of its
// own, so the kernel is bound by their latency: one value a thread over as many blocks as that
// gives (up to the scratch's) keeps them all in flight.  128 x 128 values: 22.4 us in one block
// (the former kernel), 6.1 us here.
template <typename T>
__global__ void __launch_bounds__(DG_THREADS)
probe_loss_kernel(Geom g, const T* F, int xp, const T* target, double* part, unsigned* ticket,
                  double* loss) {
    pdl_trigger();
    pdl_wait();
    double acc[1] = {0.0};
    const long long n = (long long)g.ny * g.nz;
    for (long long t = (long long)blockIdx.x * DG_THREADS + threadIdx.x; t < n;
         t += (long long)gridDim.x * DG_THREADS) {
        const int k = (int)(t / g.ny), j = (int)(t - (long long)k * g.ny);
        const double d = (double)F[pidx(g, xp, j, k)] - (double)target[t];
        acc[0] += d * d;
    }
    reduce_finish<1, true>(acc, part, ticket, 1.0, loss);
}

// (cos, sin) of w (m + o) for m < n: one entry per grid line of an axis
__device__ __forceinline__ void phase_entry(double2* tab, int m, double w, double o) {
    double sn, cs;
    sincos(w * (m + o), &sn, &cs);
    tab[m] = make_double2(cs, sn);
}

// A 16-byte vector of a row: four floats or two doubles
template <typename T>
struct Vec;
template <>
struct Vec<float> {
    static constexpr int N = 4;
    static __device__ __forceinline__ void load(const float* p, double* v) {
        const float4 a = *reinterpret_cast<const float4*>(p);
        v[0] = a.x; v[1] = a.y; v[2] = a.z; v[3] = a.w;
    }
};
template <>
struct Vec<double> {
    static constexpr int N = 2;
    static __device__ __forceinline__ void load(const double* p, double* v) {
        const double2 a = *reinterpret_cast<const double2*>(p);
        v[0] = a.x; v[1] = a.y;
    }
};

// Four floats widened by integer shifts: the value times 2^-896, exactly, for every finite float
// (denormals included), since the float's exponent field is placed in the double's as it is.  The
// conversion instruction runs on the FP64 pipe (two lanes an SM), where it would cost as much as
// a multiply-add.  `top` collects the magnitudes' bits: 0x7f800000 or more tells that an infinity
// or a NaN was among them, which this form does not carry over; and where the largest is below 2^-120,
// products with a phase fall below the normal doubles and lose digits (above it at most 2^-59 of the
// largest value).  Such values are converted instead.
constexpr double WIDEN_BACK = 0x1p896;
__device__ __forceinline__ bool widens(unsigned top) {
    return top == 0 || (top >= 0x03800000u && top < 0x7f800000u);
}
__device__ __forceinline__ void widen(const float* p, double* v, unsigned& top) {
    const uint4 a = *reinterpret_cast<const uint4*>(p);
    const unsigned b[4] = {a.x, a.y, a.z, a.w};
#pragma unroll
    for (int u = 0; u < 4; ++u) {
        const unsigned m = b[u] & 0x7fffffffu;
        top = max(top, m);
        v[u] = __hiloint2double((int)((b[u] & 0x80000000u) | (m >> 3)), (int)(m << 29));
    }
}

// The projections walk items of one 16-byte column group and up to ITEM_ROWS rows of a plane, the
// column groups fastest, so that a warp reads whole rows and an item's column and plane factors
// are applied once.
constexpr int ITEM_ROWS = 16;

template <typename T>
__host__ __device__ inline long long item_count(const Geom& g) {
    return (long long)(g.nx / (16 / (int)sizeof(T))) * ((g.ny + ITEM_ROWS - 1) / ITEM_ROWS) * g.nz;
}

struct Item {
    int i, j0, j1, k;
};

template <typename T>
__device__ __forceinline__ Item item_at(const Geom& g, long long t) {
    const int nc = g.nx / Vec<T>::N, nj = (g.ny + ITEM_ROWS - 1) / ITEM_ROWS;
    const long long r = t / nc;
    Item it;
    it.i = (int)(t - r * nc) * Vec<T>::N;
    it.k = (int)(r / nj);
    it.j0 = (int)(r - (long long)it.k * nj) * ITEM_ROWS;
    it.j1 = min(it.j0 + ITEM_ROWS, g.ny);
    return it;
}

// sum F exp(-i k.r) with r = ((i + ox) dx, (j + oy) dy, (k + oz) dz), in FP64.  The phase is a
// product of one factor per axis, so nx + ny + nz sincos (phase_kernel) replace one per cell: the
// sum over a column's rows takes two FP64 multiply-adds a cell, the factors of the column and the
// plane come once an item.  256^3 FP32: 1140 us with a sincos a cell, 126 us with the product form
// and converted floats, 88 us with widen(); the FP64 pipe (two lanes an SM) is the limit, not the
// 67 MB that are read.
__global__ void phase_kernel(Geom g, double kx, double ky, double kz, double ox, double oy,
                             double oz, double2* __restrict__ tab) {
    pdl_trigger();
    pdl_wait();
    const int t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t < g.nx) phase_entry(tab, t, kx, ox);
    else if (t < g.nx + g.ny) phase_entry(tab + g.nx, t - g.nx, ky, oy);
    else if (t < g.nx + g.ny + g.nz) phase_entry(tab + g.nx + g.ny, t - g.nx - g.ny, kz, oz);
}

template <typename T>
__global__ void __launch_bounds__(DG_THREADS)
planewave_kernel(Geom g, const T* F, const double2* tab, double* part,
                 unsigned* ticket, double* out) {
    constexpr int V = Vec<T>::N;
    pdl_trigger();
    pdl_wait();
    double acc[2] = {0.0, 0.0};
    const long long n = item_count<T>(g);
    for (long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x; t < n;
         t += (long long)gridDim.x * blockDim.x) {
        const Item it = item_at<T>(g, t);
        const T* p = F + pidx(g, it.i, it.j0, it.k);
        const double2* ey = tab + g.nx + it.j0;
        double re[V], im[V];
        bool plain = true;   // the row sums hold
        const int rows = it.j1 - it.j0;
        auto rows_sum = [&](auto&& load) {
#pragma unroll
            for (int u = 0; u < V; ++u) re[u] = im[u] = 0.0;
#pragma unroll 4
            for (int j = 0; j < rows; ++j) {
                double v[V];
                load(p + (long long)j * g.nxp, v);
                const double2 e = ey[j];
#pragma unroll
                for (int u = 0; u < V; ++u) {
                    re[u] = fma(v[u], e.x, re[u]);
                    im[u] = fma(v[u], e.y, im[u]);
                }
            }
        };
        if constexpr (sizeof(T) == 4) {
            unsigned top = 0;
            rows_sum([&](const float* q, double* v) { widen(q, v, top); });
#pragma unroll
            for (int u = 0; u < V; ++u) { re[u] *= WIDEN_BACK; im[u] *= WIDEN_BACK; }
            plain = widens(top);
        } else {
            rows_sum([&](const T* q, double* v) { Vec<T>::load(q, v); });
#pragma unroll
            for (int u = 0; u < V; ++u) plain = plain && isfinite(re[u]) && isfinite(im[u]);
        }
        const double2 ez = tab[g.nx + g.ny + it.k];
        auto times = [](double2 a, double2 b) {
            return make_double2(a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x);
        };
        if (plain) {
            double2 c = make_double2(0.0, 0.0);
#pragma unroll
            for (int u = 0; u < V; ++u) {
                const double2 e = times(make_double2(re[u], im[u]), tab[it.i + u]);
                c.x += e.x;
                c.y += e.y;
            }
            c = times(c, ez);
            acc[0] += c.x;
            acc[1] -= c.y;
        } else {   // cell by cell: infinities reach the sums as value x phase
            for (int j = 0; j < rows; ++j)
                for (int u = 0; u < V; ++u) {
                    const double2 e = times(times(tab[it.i + u], ey[j]), ez);
                    const double v = (double)p[(long long)j * g.nxp + u];
                    acc[0] += v * e.x;
                    acc[1] -= v * e.y;
                }
        }
    }
    reduce_finish<2>(acc, part, ticket, 1.0, out);
}

// sum over components and cells of (1/2) F^2 (1, cos th, sin th), th = 2 pi (idx_a + off) / n_a
// with off = 1/2 for the components staggered along a (App. A positions).  The angles come from
// a table of 2 n_a entries (whole, then half positions) instead of two sincos a cell.
__global__ void moment_phase_kernel(int na, double2* __restrict__ tab) {
    const int t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t < na) phase_entry(tab, t, 2.0 * M_PI / na, 0.0);
    else if (t < 2 * na) phase_entry(tab + na, t - na, 2.0 * M_PI / na, 0.5);
}

template <typename T>
__global__ void __launch_bounds__(DG_THREADS)
moments_kernel(Geom g, FieldSet<T> s, int axis, const double2* __restrict__ tab, double* part,
               unsigned* ticket, double scale, double* out) {
    constexpr int V = Vec<T>::N;
    double acc[3] = {0.0, 0.0, 0.0};
    const long long n = item_count<T>(g);
    const int na = axis == 0 ? g.nx : axis == 1 ? g.ny : g.nz;
    for (long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x; t < n;
         t += (long long)gridDim.x * blockDim.x) {
        const Item it = item_at<T>(g, t);
        const long long base = pidx(g, it.i, it.j0, it.k);
        const int rows = it.j1 - it.j0;
        double e0[V], eh[V];   // energy at the whole and the half positions of each column
#pragma unroll
        for (int u = 0; u < V; ++u) e0[u] = eh[u] = 0.0;
        auto add = [&](double a0, double ah, int m) {
            const double2 w0 = tab[m], wh = tab[na + m];
            acc[0] += a0 + ah;
            acc[1] += a0 * w0.x + ah * wh.x;
            acc[2] += a0 * w0.y + ah * wh.y;
        };
        for (int j = 0; j < rows; ++j) {
            double r0[V], rh[V];
#pragma unroll
            for (int u = 0; u < V; ++u) r0[u] = rh[u] = 0.0;
#pragma unroll
            for (int q = 0; q < 6; ++q) {
                double v[V];
                Vec<T>::load(s.c[q] + base + (long long)j * g.nxp, v);
                // staggered along `axis`: E_a, and the two B components other than B_a
                const bool half = (q < 3) == (q % 3 == axis);
#pragma unroll
                for (int u = 0; u < V; ++u) {
                    if (half) rh[u] = fma(v[u], v[u], rh[u]);
                    else r0[u] = fma(v[u], v[u], r0[u]);
                }
            }
#pragma unroll
            for (int u = 0; u < V; ++u) { e0[u] += r0[u]; eh[u] += rh[u]; }
            if (axis == 1) {
                double a0 = 0.0, ah = 0.0;
#pragma unroll
                for (int u = 0; u < V; ++u) { a0 += r0[u]; ah += rh[u]; }
                add(a0, ah, it.j0 + j);
            }
        }
        if (axis == 0) {
#pragma unroll
            for (int u = 0; u < V; ++u) add(e0[u], eh[u], it.i + u);
        } else if (axis == 2) {
            double a0 = 0.0, ah = 0.0;
#pragma unroll
            for (int u = 0; u < V; ++u) { a0 += e0[u]; ah += eh[u]; }
            add(a0, ah, it.k);
        }
    }
    reduce_finish<3>(acc, part, ticket, scale, out);
}

// ---- divergences (dense output, FP64) -----------------------------------------------------

__device__ __forceinline__ long long zo(const Geom& g, int k, int dz) {
    int kk = (k + dz) % g.nz;
    if (kk < 0) kk += g.nz;
    return (long long)(kk - k) * g.plane;
}

// which: 0 = D*.B (extended, forward type, at cell corners), 1 = Yee D.B (forward type),
//        2 = D.E (Yee, backward type, at nodes).  Multipliers carry 1/dx (not dt).
template <typename T>
__global__ void divergence_kernel(Geom g, Mult<double> w, FieldSet<T> s, int which,
                                  double* __restrict__ out) {
    const long long n = (long long)g.nx * g.ny * g.nz;
    const long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= n) return;
    const int i = (int)(t % g.nx);
    const long long r = t / g.nx;
    const int j = (int)(r % g.ny);
    const int k = (int)(r / g.ny);
    const long long c = pidx(g, i, j, k);
    const long long Y = g.nxp;
    const long long zp1 = zo(g, k, 1), zm1 = zo(g, k, -1), zp2 = zo(g, k, 2);
    double v = 0.0;
    if (which == 2) {
        const T* Ex = s.c[0];
        const T* Ey = s.c[1];
        const T* Ez = s.c[2];
        v = w.cE[0] * ((double)Ex[c] - (double)Ex[c - 1]) + w.cE[1] * ((double)Ey[c] - (double)Ey[c - Y]) +
            w.cE[2] * ((double)Ez[c] - (double)Ez[c + zm1]);
    } else {
        const T* B[3] = {s.c[3], s.c[4], s.c[5]};
        const long long a1[3] = {1, Y, zp1}, a2[3] = {2, 2 * Y, zp2}, am1[3] = {-1, -Y, zm1};
        const long long tp[3][2] = {{Y, zp1}, {1, zp1}, {1, Y}};
        const long long tm[3][2] = {{-Y, zm1}, {-1, zm1}, {-1, -Y}};
        for (int a = 0; a < 3; ++a) {
            const T* F = B[a];
            const double ax = (double)F[c + a1[a]] - (double)F[c];
            if (which == 1) {
                v += w.cE[a] * ax;
                continue;
            }
            double d = w.cA[a] * ax + w.cD[a] * ((double)F[c + a2[a]] - (double)F[c + am1[a]]);
            const int b[2] = {a == 0 ? 1 : 0, a == 2 ? 1 : 2};
            for (int q = 0; q < 2; ++q) {
                d += w.cB[a][b[q]] * (((double)F[c + a1[a] + tp[a][q]] - (double)F[c + tp[a][q]]) +
                                      ((double)F[c + a1[a] + tm[a][q]] - (double)F[c + tm[a][q]]));
            }
            v += d;
        }
    }
    out[t] = v;
}

// scratch of one handle: partials [diag_blocks][3], the phase tables, the ticket
size_t diag_scratch_bytes(const Geom& g) {
    return (size_t)diag_blocks(g) * 3 * sizeof(double) +
           (size_t)2 * (g.nx + g.ny + g.nz) * sizeof(double2) + 16;
}

struct DiagScratch {
    double* part;
    double2* tab;
    unsigned* ticket;
};

static DiagScratch diag_scratch(const Geom& g, double* base) {
    DiagScratch d;
    d.ticket = (unsigned*)base;   // first 16 bytes: zero between launches
    d.tab = (double2*)(base + 2);
    d.part = (double*)(d.tab + 2 * (size_t)(g.nx + g.ny + g.nz));
    return d;
}

static int blocks_of(long long items, const Geom& g) {
    const long long b = (items + DG_THREADS - 1) / DG_THREADS;
    return (int)(b < diag_blocks(g) ? b : diag_blocks(g));
}

template <typename T>
void launch_energy(const Geom& g, FieldSet<T> s, int x_lo, int x_len, int my, int mz, double dV,
                   double* scratch, double* out, cudaStream_t st) {
    const DiagScratch d = diag_scratch(g, scratch);
    energy_kernel<T><<<diag_blocks(g), DG_THREADS, 0, st>>>(g, s, x_lo, x_len, my, mz, d.part,
                                                            d.ticket, 0.5 * dV, out);
}

template <typename T>
void launch_probe_loss(const Geom& g, const T* E, int x_index, const T* target, double* scratch,
                       double* loss, cudaStream_t st) {
    const DiagScratch d = diag_scratch(g, scratch);
    launch_pdl(probe_loss_kernel<T>, dim3(blocks_of((long long)g.ny * g.nz, g)), dim3(DG_THREADS), 0, st, g,
               E, x_index, target, d.part, d.ticket, loss);
}
template void launch_probe_loss<float>(const Geom&, const float*, int, const float*, double*,
                                       double*, cudaStream_t);
template void launch_probe_loss<double>(const Geom&, const double*, int, const double*, double*,
                                        double*, cudaStream_t);

template <typename T>
void launch_planewave(const Geom& g, const T* F, const double k[3], const double off[3],
                      double* scratch, double* out, cudaStream_t st) {
    const DiagScratch d = diag_scratch(g, scratch);
    const int lines = g.nx + g.ny + g.nz;
    launch_pdl(phase_kernel, dim3((lines + 63) / 64), dim3(64), 0, st, g, k[0], k[1], k[2], off[0], off[1],
               off[2], d.tab);
    launch_pdl(planewave_kernel<T>, dim3(blocks_of(item_count<T>(g), g)), dim3(DG_THREADS), 0, st, g, F, d.tab,
               d.part, d.ticket, out);
}

template <typename T>
void launch_moments(const Geom& g, FieldSet<T> s, int axis, double dV, double* scratch, double* out,
                    cudaStream_t st) {
    const DiagScratch d = diag_scratch(g, scratch);
    const int na = axis == 0 ? g.nx : axis == 1 ? g.ny : g.nz;
    moment_phase_kernel<<<(2 * na + 63) / 64, 64, 0, st>>>(na, d.tab);
    moments_kernel<T><<<blocks_of(item_count<T>(g), g), DG_THREADS, 0, st>>>(
        g, s, axis, d.tab, d.part, d.ticket, 0.5 * dV, out);
}

template <typename T>
void launch_divergence(const Geom& g, const Mult<double>& w, FieldSet<T> s, int which, double* out,
                       cudaStream_t st) {
    const long long n = (long long)g.nx * g.ny * g.nz;
    divergence_kernel<T><<<(unsigned)((n + 255) / 256), 256, 0, st>>>(g, w, s, which, out);
}

template void launch_energy<float>(const Geom&, FieldSet<float>, int, int, int, int, double,
                                   double*, double*, cudaStream_t);
template void launch_energy<double>(const Geom&, FieldSet<double>, int, int, int, int, double,
                                    double*, double*, cudaStream_t);
template void launch_planewave<float>(const Geom&, const float*, const double[3], const double[3],
                                      double*, double*, cudaStream_t);
template void launch_planewave<double>(const Geom&, const double*, const double[3],
                                       const double[3], double*, double*, cudaStream_t);
template void launch_moments<float>(const Geom&, FieldSet<float>, int, double, double*, double*,
                                    cudaStream_t);
template void launch_moments<double>(const Geom&, FieldSet<double>, int, double, double*, double*,
                                     cudaStream_t);
template void launch_divergence<float>(const Geom&, const Mult<double>&, FieldSet<float>, int,
                                       double*, cudaStream_t);
template void launch_divergence<double>(const Geom&, const Mult<double>&, FieldSet<double>, int,
                                        double*, cudaStream_t);

}  // namespace fdtd

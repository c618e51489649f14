// FP32 leapfrog step of planes that do not couple along z: a 2D grid (nz = 1) or a batch of
// independent 2D problems.
//
// A CTA owns a 64 x 4 (x, y) tile of one plane.  E^n comes as a 72 x 8 box (x0-4 ..,
// y0-2 ..) by 16-byte asynchronous copies, B^{n-1/2} straight into registers; the CTA forms
// B^{n+1/2} on the tile, on the halo row y0-1 and on the halo column x0-1, passes it through shared
// memory and forms E^{n+1}: one read and one write of the state and the box halo, which L2 serves.
// The 3D kernel (fdtd_fused32.cu) gives the same fields but marches along z: for one plane it
// forms two planes of B and reads the plane's E box five times.
//
// All z differences vanish (nz = 1) or have zero multipliers (batch), so D*_z drops out and the
// transverse z terms of D*_x and D*_y are the plane's own differences (times a multiplier that is
// zero unless a 3D problem is one plane thick): the fields are bitwise those of the 3D kernels.
// A thread works on segments of four cells as there (fdtd_seg.cuh).
//
// Bound: launch and latency for a small plane, HBM and L2 for a large batch.  Us a step, the 3D kernel (whole tiles) or
// the reference form before and this kernel: 128 x 128 33 / 2.8 (4.2 without the dependent launch),
// 1000 x 750 24 / 8.0 (10.3), 512 x 512 x 32 107 / 76 (403 MB: 0.78 of the copy rate).
#include "fdtd_seg.cuh"

namespace fdtd {
namespace flat32 {

using namespace seg;

constexpr int W = 4, TX = 64, NSEG = TX / W;
constexpr int TY = 4;        // 2, 8 and 16 rows measured within 3 % or slower (512 x 512 x 32: 93, 81,
                             // 84 us against 80; 128 x 128: 4.2, 6.0, 6.2 us against 4.2)
constexpr int EW = TX + 8, EH = TY + 4, EPL = EW * EH;   // E box x0-4 .. x0+67, y0-2 .. y0+TY+1
constexpr int BW = TX + 4, BPL = BW * (TY + 1);          // B rows x0-4 .. x0+63, y0-1 .. y0+TY-1
constexpr int NTASK = NSEG * (TY + 1) + TY + 1;          // rows and the halo column
constexpr int NT = (NTASK + 31) / 32 * 32;

__device__ __forceinline__ void copy16(float* dst, const float* src) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(smem_u32(dst)), "l"(src) : "memory");
}

__global__ void __launch_bounds__(NT)
step2d_kernel(Geom g, Mult<float> m, Mult2 m2, FieldSet<float> in, FieldSet<float> out,
              const float* __restrict__ spy, const float* __restrict__ spz,
              const float* __restrict__ jyz, const float* jx_row,
              float* __restrict__ h0, float* __restrict__ h1, float* __restrict__ h2,
              int* __restrict__ err) {
    __shared__ __align__(16) float sE[3 * EPL];
    __shared__ __align__(16) float sB[3 * BPL];
    pdl_trigger();
    pdl_wait();
    const int ntx = (g.nx + TX - 1) / TX, nty = (g.ny + TY - 1) / TY;
    int w = blockIdx.x;
    const int tx = w % ntx;
    w /= ntx;
    const int ty = w % nty, k = w / nty;
    const int x0 = tx * TX, y0 = ty * TY, tid = threadIdx.x;
    const unsigned plane = (unsigned)g.plane, po = (unsigned)k * plane;
    const bool edge = (x0 < PX) || (x0 + TX > g.nx - PX) || (y0 < PY) || (y0 + TY > g.ny - PY);

    // task of this thread, as in the 3D kernel: owned rows, then the halo row y0-1, then the halo
    // column (its segment's last cell x0-1 is the one that is used), then idle copies of the last
    const int bx = tid < NSEG * (TY + 1) ? W * (tid % NSEG) : -W;
    const int by = tid < NSEG * TY ? tid / NSEG
                   : tid < NSEG * (TY + 1) ? -1 : min(tid - NSEG * (TY + 1) - 1, TY - 1);
    const bool own = tid < NSEG * TY;   // warp-uniform (TY is even)
    const bool live = x0 + bx < g.nx && y0 + by < g.ny;   // not past a ragged grid's cells
    const int i = min(x0 + bx, g.nx - W), j = min(y0 + by, g.ny - 1);
    const bool lb = bx == 0, rb = bx < 0 || bx == TX - W;
    const int e = (by + 2) * EW + (bx + 4), bi = (by + 1) * BW + (bx + 4);
    const SegOut dst = seg_out(g, max(i, 0), max(j, 0), edge);
    float bo[3][W];   // before the box's copies (behind them: 512 x 512 x 32 80 us, here 76)
#pragma unroll
    for (int c = 0; c < 3; ++c)
        unpackv(*reinterpret_cast<const float4*>(in.c[3 + c] + po + (unsigned)((j + PY) * g.nxp + i + PX)),
                bo[c]);

    // E box: padded row y0 + r and column x0 + 4 c hold (x0-4+4c, y0-2+r); a ragged tile's box stops
    // at the ghosts
    const int rows = min(EH, g.nyp - y0), cols = min(EW, g.nxp - x0) / W;
    for (int t = tid; t < EH * (EW / W); t += NT) {
        const int r = t / (EW / W), c = t - r * (EW / W);
        if (r >= rows || c >= cols) continue;
        const unsigned o = po + (unsigned)((y0 + r) * g.nxp + x0 + W * c);
#pragma unroll
        for (int q = 0; q < 3; ++q) copy16(sE + q * EPL + r * EW + W * c, in.c[q] + o);
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
    float f = 1.0f;
    if (spy != nullptr) f = spy[j < 0 ? j + g.ny : j] * spz[k];

    asm volatile("cp.async.wait_group 0;" ::: "memory");
    __syncthreads();
    // ---- B^{n+1/2}
    const float *Ex = sE, *Ey = sE + EPL, *Ez = sE + 2 * EPL;
    const Q4 x_ = ldq(Ex, e), y_ = ldq(Ey, e), z_ = ldq(Ez, e);
    float b[3][W];
    {
        u64 d[2], r2[2];
        float t[W];
        dstar_y2<EW>(Ez, Ez, Ez, z_, z_, z_, e, lb, rb, m2.cA[1], m2.cD[1], m2.cB[1][0], m2.cB[1][2], d);
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            r2[h] = sub2(pk(bo[0][2 * h], bo[0][2 * h + 1]), d[h]);
            upk(r2[h], b[0][2 * h], b[0][2 * h + 1]);
        }
        dstar_x4<EW>(Ez, Ez, Ez, z_, z_, z_, e, lb, rb, m.cA[0], m.cD[0], m.cB[0][1], m.cB[0][2], t);
#pragma unroll
        for (int u = 0; u < W; ++u) b[1][u] = bo[1][u] + t[u];
        dstar_y2<EW>(Ex, Ex, Ex, x_, x_, x_, e, lb, rb, m2.cA[1], m2.cD[1], m2.cB[1][0], m2.cB[1][2], d);
        dstar_x4<EW>(Ey, Ey, Ey, y_, y_, y_, e, lb, rb, m.cA[0], m.cD[0], m.cB[0][1], m.cB[0][2], t);
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            r2[h] = add2(pk(bo[2][2 * h], bo[2][2 * h + 1]), sub2(d[h], pk(t[2 * h], t[2 * h + 1])));
            upk(r2[h], b[2][2 * h], b[2][2 * h + 1]);
        }
    }
    if (spy != nullptr) {
#pragma unroll
        for (int c = 0; c < 3; ++c)
#pragma unroll
            for (int u = 0; u < W; ++u) b[c][u] *= f;
    }
    if (tid < NTASK) {
#pragma unroll
        for (int c = 0; c < 3; ++c) stv(sB + c * BPL, bi, b[c]);
    }
    if (own && live) {
#pragma unroll
        for (int c = 0; c < 3; ++c) put_seg(out.c[3 + c], po, dst, b[c]);
    }
    __syncthreads();
    // ---- E^{n+1} (D x B without its z differences)
    if (!own) return;
    const float *Bx = sB, *By = sB + BPL, *Bz = sB + 2 * BPL;
    const Q4 Bzy = ldq(Bz, bi - BW), Bxy = ldq(Bx, bi - BW);
    float zl = from_left(b[2][3]), yl = from_left(b[1][3]);   // x-1
    if (lb) {
        zl = Bz[bi - 1];
        yl = By[bi - 1];
    }
    float ex[W], ey[W], ez[W];
#pragma unroll
    for (int u = 0; u < W; ++u) {
        const float zm = u ? b[2][u ? u - 1 : 0] : zl, ym = u ? b[1][u ? u - 1 : 0] : yl;
        // ampere_comp with a zero z difference
        ex[u] = x_.v[u] + __fmul_rn(m.cE[1], b[2][u] - Bzy.v[u]);
        ey[u] = y_.v[u] - __fmul_rn(m.cE[0], b[2][u] - zm);
        ez[u] = ampere_comp(z_.v[u], b[1][u], ym, b[0][u], Bxy.v[u], m.cE[0], m.cE[1]);
    }
    if (!live) return;
    if (jx_row != nullptr) {
        float jv[W];
        unpackv(*reinterpret_cast<const float4*>(jx_row + i), jv);
        const float sy = jyz[j], sz = jyz[g.ny + k];
#pragma unroll
        for (int u = 0; u < W; ++u) ex[u] = fma(-m.dt, (jv[u] * sy) * sz, ex[u]);
    }
    if (spy != nullptr) {
#pragma unroll
        for (int u = 0; u < W; ++u) { ex[u] *= f; ey[u] *= f; ez[u] *= f; }
    }
    float fin = 0.0f;   // non-finite detection (nonfinite_acc)
#pragma unroll
    for (int u = 0; u < W; ++u)
        fin = nonfinite_acc(nonfinite_acc(nonfinite_acc(fin, ex[u]), ey[u]), ez[u]);
    put_seg(out.c[0], po, dst, ex);
    put_seg(out.c[1], po, dst, ey);
    put_seg(out.c[2], po, dst, ez);
    if (h0 != nullptr) {
        put_seg(h0, po, dst, ex);
        put_seg(h1, po, dst, ey);
        put_seg(h2, po, dst, ez);
    }
    if (!(fin == 0.0f)) atomicOr(err, ERR_FIELD);
}

}  // namespace flat32

void launch_step2d32(const Geom& g, const Mult<float>& m, FieldSet<float> in, FieldSet<float> out,
                     const float* spy, const float* spz, const float* jyz, const float* jx_row,
                     float* hist_E[3], int* err, cudaStream_t st) {
    using namespace flat32;
    const long long tiles = (long long)((g.nx + TX - 1) / TX) * ((g.ny + TY - 1) / TY) * g.nz;
    launch_pdl(step2d_kernel, dim3((unsigned)tiles), dim3(NT), 0, st, g, m, make_mult2(m), in, out, spy,
               spz, jyz, jx_row, hist_E[0], hist_E[1], hist_E[2], err);
}

}  // namespace fdtd

// FP32 reverse leapfrog step of planes that do not couple along z (a batch of 2D problems, or
// nz = 1), in one kernel: the step of fdtd_adjoint32f.cu without what it does for z.
//
// A CTA owns a 64 x 8 (x, y) tile and a chunk of planes, as there; each plane is a problem of its
// own, so the chunk has no halo planes:
//   phase A: mu on the tile and its halo (x0-4 .. x0+67, y0-2 .. y0+8) from the lambda_E box
//     (72 x 12, two-slot ring) and the lambda_B box (72 x 11, three-slot ring; mu takes its place
//     there, cell by cell), copied by TMA two planes ahead;
//   phase B: lambda_E' and the gradient terms of the own cells from mu, E^n and lambda_E, the own
//     rows of mu and lambda_E staying in registers.
// One block barrier a plane: phase B of plane p reads the ring slot that plane p+3 is copied to
// after the barrier of plane p+1.  128 threads, a thread its own segment of four cells in both
// phases (and 67 of them one of the halo's), four CTAs an SM.
//
// The z differences are the plane's own (nz = 1) or have zero multipliers (batch): D*_z and the
// third gradient term of D*_x and D*_y (T_beta_az, exactly zero or not asked for) drop out.  Every
// value is formed and every sum taken over the same cells in the same order as there (the chunk's
// planes are one compensated FP32 sum a thread and axis); lambda is bitwise that of the 3D kernels.
//
// Bound: HBM for a large batch (60 B a cell), launch and latency for a small one.  Us a step, the 3D
// kernel and this one: 512 x 512 x 32 148 / 97 (503 MB: 0.77 of the copy rate), 512 x 512 x 8 50 / 29,
// 1024 x 1024 72 / 27, 192 x 40 x 70 38 / 23, 64 x 8 8.7 / 4.3.
#include "fdtd_seg.cuh"

namespace fdtd {
namespace adj32p {

using namespace seg;

constexpr int W = 4, TX = 64, TY = 8, NSEG = TX / W;
constexpr int NT = NSEG * TY;                            // 128 threads, one own segment each
constexpr int NHALO = 3 * NSEG + 2 * (TY + 1) + 1;       // rows -1, -2, 8 and the two columns
constexpr int PRODUCER = NT - 1;                         // no halo task in its warp
static_assert(NHALO <= NT - 32, "the producer's warp has no halo task");
constexpr int LW = TX + 8, LH = TY + 4, LPL = LW * LH;   // lambda_E box 72 x 12
constexpr int LSLOT = ((LPL * 4 + 127) / 128) * 128 / 4;
constexpr int MH = TY + 3, MPL = LW * MH;                // lambda_B box and mu plane 72 x 11
constexpr int MSLOT = ((MPL * 4 + 127) / 128) * 128 / 4;
constexpr int NL = 2, NM = 3;
constexpr size_t OFF_M = (size_t)NL * 3 * LSLOT * 4;
constexpr size_t OFF_BAR = OFF_M + (size_t)NM * 3 * MSLOT * 4;
constexpr size_t SMEM = OFF_BAR + NL * 8;
constexpr uint32_t UNIT_BYTES = 3u * (LPL + MPL) * 4;

// the plane's sums of one axis: w times (t2, sb, d0), as bracket_acc of the 3D kernel
template <bool NEG>
__device__ __forceinline__ void bracket2(float* acc, float w, float d0, float t2, float sb) {
    const float ww = NEG ? -w : w;
    acc[0] = fmaf(ww, t2, acc[0]);
    acc[1] = fmaf(ww, sb, acc[1]);
    acc[2] = fmaf(ww, d0, acc[2]);
}

// DT_y of a mu component (transverse x; z: the plane itself); a0: the own row
template <bool NEG>
__device__ __forceinline__ void dty(const float* G, const float* a0, int e, bool lb, bool rb, float cA,
                                    float cD, float cBx, float cBz, const float* w, float* acc,
                                    float out[W]) {
    const Q4 am = ldq(G, e - LW), amm = ldq(G, e - 2 * LW), ap = ldq(G, e + LW);
    float d[6];   // d[k] = G(y-1) - G(y) at x-1+k
#pragma unroll
    for (int u = 0; u < W; ++u) d[1 + u] = am.v[u] - a0[u];
    d[0] = from_left(d[4]);
    d[5] = from_right(d[1]);
    if (lb) d[0] = G[e - LW - 1] - G[e - 1];
    if (rb) d[5] = G[e - LW + 4] - G[e + 4];
#pragma unroll
    for (int u = 0; u < W; ++u) {
        out[u] = dstar_diff(d[1 + u], amm.v[u], ap.v[u], d[u], d[2 + u], d[1 + u], d[1 + u], cA, cD, cBx,
                            cBz);
        bracket2<NEG>(acc, w[u], d[1 + u], amm.v[u] - ap.v[u], d[u] + d[2 + u]);
    }
}

// DT_x (transverse y; z: the plane itself)
template <bool NEG>
__device__ __forceinline__ void dtx(const float* G, const float* R, int e, bool lb, bool rb, float cA,
                                    float cD, float cBy, float cBz, const float* w, float* acc,
                                    float out[W]) {
    const Q4 Ym = ldq(G, e - LW), Yp = ldq(G, e + LW);
    float r[7], ym[5], yp[5];   // G at x-2 .. x+4; x-1 .. x+3
#pragma unroll
    for (int u = 0; u < W; ++u) {
        r[2 + u] = R[u];
        ym[1 + u] = Ym.v[u];
        yp[1 + u] = Yp.v[u];
    }
    r[0] = from_left(R[2]);
    r[1] = from_left(R[3]);
    r[6] = from_right(R[0]);
    ym[0] = from_left(Ym.v[3]);
    yp[0] = from_left(Yp.v[3]);
    if (lb) {
        r[0] = G[e - 2];
        r[1] = G[e - 1];
        ym[0] = G[e - LW - 1];
        yp[0] = G[e + LW - 1];
    }
    if (rb) r[6] = G[e + 4];
#pragma unroll
    for (int u = 0; u < W; ++u) {
        const float d0 = r[u + 1] - r[u + 2];
        const float dym = ym[u] - ym[u + 1], dyp = yp[u] - yp[u + 1];
        out[u] = dstar_diff(d0, r[u], r[u + 3], dym, dyp, d0, d0, cA, cD, cBy, cBz);
        bracket2<NEG>(acc, w[u], d0, r[u] - r[u + 3], dym + dyp);
    }
}

// SP: absorbing layers present; without them S = 1 folds away
template <bool SP>
__global__ void __launch_bounds__(NT, 4)
adj2d_kernel(const __grid_constant__ FusedMaps maps, Geom g, Mult<float> m, FieldSet<float> out,
             const float* e_x, const float* e_y, const float* e_z, const float* __restrict__ spy,
             const float* __restrict__ spz, double* __restrict__ partials, int tz,
             int* __restrict__ err) {
    extern __shared__ __align__(128) unsigned char smem[];
    float* sL = reinterpret_cast<float*>(smem);
    float* sM = reinterpret_cast<float*>(smem + OFF_M);
    uint64_t* bar = reinterpret_cast<uint64_t*>(smem + OFF_BAR);

    const int ntx = g.nx / TX, nty = g.ny / TY;
    int w = blockIdx.x;
    const int tx = w % ntx;
    w /= ntx;
    const int ty = w % nty;
    const int x0 = tx * TX, y0 = ty * TY, z0 = (w / nty) * tz;
    const int niter = min(tz, g.nz - z0);
    const int tid = threadIdx.x, wp = tid >> 5;
    const bool edge = (x0 < PX) || (x0 + TX > g.nx - PX) || (y0 < PY) || (y0 + TY > g.ny - PY);
    const unsigned plane = (unsigned)g.plane;

    // unit u: the boxes of plane z0 + u
    auto issue_unit = [&](int u) {
        uint64_t* b = &bar[u % NL];
        mbar_expect_tx(b, UNIT_BYTES);
        for (int c = 0; c < 3; ++c) {
            tma_load_3d(sL + ((u % NL) * 3 + c) * LSLOT, &maps.e[c], x0, y0, z0 + u, b);
            tma_load_3d(sM + ((u % NM) * 3 + c) * MSLOT, &maps.b[c], x0, y0, z0 + u, b);
        }
    };

    // own segment, and the halo's (warps 0-2; lanes without one form a copy of the last, dropped:
    // the warp's shuffles need every lane)
    const int bx = W * (tid % NSEG), by = tid / NSEG;
    const bool lb = bx == 0, rb = bx == TX - W;
    const int e = (by + 2) * LW + (bx + 4);
    const int jw = y0 + by;
    const SegOut dst = seg_out(g, x0 + bx, jw, edge);
    const int t = min(tid, NHALO - 1);
    int hx, hy;
    if (t < 3 * NSEG) {   // rows -1, -2, 8
        hx = W * (t % NSEG);
        hy = t < NSEG ? -1 : t < 2 * NSEG ? -2 : TY;
    } else if (t < 3 * NSEG + TY + 2) {   // left column, rows -1 .. 8
        hx = -W;
        hy = t - 3 * NSEG - 1;
    } else {   // right column, rows -1 .. 7
        hx = TX;
        hy = t - 3 * NSEG - (TY + 2) - 1;
    }
    const bool hrb = hx < 0 || hx >= TX - W;
    const int he = (hy + 2) * LW + (hx + 4);
    int jh = (y0 + hy) % g.ny;
    if (jh < 0) jh += g.ny;

    if (tid == PRODUCER) {
        for (int s = 0; s < NL; ++s) mbar_init(&bar[s], 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    }
    __syncthreads();
    pdl_trigger();   // nothing above touches global memory
    pdl_wait();
    int issued = 0;
    if (tid == PRODUCER)
        for (; issued < NL && issued < niter; ++issued) issue_unit(issued);

    // compensated FP32 sums over the chunk's planes, (delta, beta) of each: D*_y from mu_z, D*_x,
    // D*_y from mu_x (three sums in the 3D kernel too)
    float gs[6], gc[6];
#pragma unroll
    for (int k = 0; k < 6; ++k) {
        gs[k] = 0.0f;
        gc[k] = 0.0f;
    }
    // mu of the segment at in-box index a, into the ring slot M
    auto form_mu = [&](const float* L, float* M, int a, bool last, float s0, float syp, bool keep,
                       float (&mu)[3][W], float (&le)[3][W]) {
        const Q4 bxq = ldq(M, a), byq = ldq(M + MSLOT, a), bzq = ldq(M + 2 * MSLOT, a);
        const Q4 ex = ldq(L, a), ey = ldq(L + LSLOT, a), ez = ldq(L + 2 * LSLOT, a);
        const Q4 exy = ldq(L, a + LW), ezy = ldq(L + 2 * LSLOT, a + LW);
        float ey4 = from_right(ey.v[0]), ez4 = from_right(ez.v[0]);
        if (last) {
            ey4 = L[LSLOT + a + 4];
            ez4 = L[2 * LSLOT + a + 4];
        }
#pragma unroll
        for (int u = 0; u < W; ++u) {
            // the rounding order of the 3D kernel's mu
            const float ex0 = __fmul_rn(s0, ex.v[u]), ey0 = __fmul_rn(s0, ey.v[u]),
                        ez0 = __fmul_rn(s0, ez.v[u]);
            const float ezx = u < W - 1 ? ez.v[u + 1 < W ? u + 1 : 0] : ez4;   // x+1, unscaled
            const float eyx = u < W - 1 ? ey.v[u + 1 < W ? u + 1 : 0] : ey4;
            const float gx = __fmaf_rn(m.cE[2], __fmaf_rn(-s0, ey.v[u], ey0),
                                       __fmul_rn(-m.cE[1], __fmaf_rn(-syp, ezy.v[u], ez0)));
            const float gy = __fmaf_rn(m.cE[0], __fmaf_rn(-s0, ezx, ez0),
                                       __fmul_rn(-m.cE[2], __fmaf_rn(-s0, ex.v[u], ex0)));
            const float gz = __fmaf_rn(m.cE[1], __fmaf_rn(-syp, exy.v[u], ex0),
                                       __fmul_rn(-m.cE[0], __fmaf_rn(-s0, eyx, ey0)));
            mu[0][u] = __fmul_rn(s0, __fadd_rn(bxq.v[u], gx));
            mu[1][u] = __fmul_rn(s0, __fadd_rn(byq.v[u], gy));
            mu[2][u] = __fmul_rn(s0, __fadd_rn(bzq.v[u], gz));
            le[0][u] = ex.v[u];
            le[1][u] = ey.v[u];
            le[2][u] = ez.v[u];
        }
        if (keep) {
            stv(M, a, mu[0]);
            stv(M + MSLOT, a, mu[1]);
            stv(M + 2 * MSLOT, a, mu[2]);
        }
    };

    bool failed = false;
    int it = 0, mslot = 0;
    for (; it < niter; ++it, mslot = (mslot == NM - 1 ? 0 : mslot + 1)) {
        const int q = z0 + it;
        const unsigned po = (unsigned)q * plane;
        float eo[3][W];   // E^n of the own cells, used after the barrier
        unpackv(__ldcg(reinterpret_cast<const float4*>(e_x + po + dst.ro)), eo[0]);
        unpackv(__ldcg(reinterpret_cast<const float4*>(e_y + po + dst.ro)), eo[1]);
        unpackv(__ldcg(reinterpret_cast<const float4*>(e_z + po + dst.ro)), eo[2]);
        const float* L = sL + (it % NL) * 3 * LSLOT;
        float* M = sM + mslot * 3 * MSLOT;
        float mu[3][W], le[3][W];
        float s0 = 1.0f;
        bool ok = mbar_wait(&bar[it % NL], (uint32_t)((it / NL) & 1));
        ok = __all_sync(FULL, ok);   // keeps the shuffles below warp-uniform
        if (ok) {
            // ---- phase A
            float syp = 1.0f;
            if (SP) {
                s0 = spy[jw] * spz[q];
                syp = spy[jw + 1 == g.ny ? 0 : jw + 1] * spz[q];
            }
            if (wp < 3) {
                float hs = 1.0f, hsyp = 1.0f;
                if (SP) {
                    hs = spy[jh] * spz[q];
                    hsyp = spy[jh + 1 == g.ny ? 0 : jh + 1] * spz[q];
                }
                form_mu(L, M, he, hrb, hs, hsyp, tid < NHALO, mu, le);
            }
            form_mu(L, M, e, rb, s0, syp, true, mu, le);
            put_seg(out.c[3], po, dst, mu[0]);
            put_seg(out.c[4], po, dst, mu[1]);
            put_seg(out.c[5], po, dst, mu[2]);
        }
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        if (__syncthreads_or(!ok)) {
            failed = true;
            break;
        }
        // the lambda_E slot of this plane and the ring slot of the last one (read in phase B before
        // this barrier) take plane q + 2
        if (tid == PRODUCER && it + NL < niter) {
            issue_unit(it + NL);
            issued = it + NL + 1;
        }
        // ---- phase B
        float acc[9], t1[W], t2[W];
#pragma unroll
        for (int k = 0; k < 9; ++k) acc[k] = 0.0f;
        dty<false>(M + 2 * MSLOT, mu[2], e, lb, rb, m.cA[1], m.cD[1], m.cB[1][0], m.cB[1][2], eo[0], acc,
                   t1);
#pragma unroll
        for (int u = 0; u < W; ++u) t1[u] = __fmaf_rn(s0, le[0][u], t1[u]);
        put_seg(out.c[0], po, dst, t1);
        dtx<true>(M + 2 * MSLOT, mu[2], e, lb, rb, m.cA[0], m.cD[0], m.cB[0][1], m.cB[0][2], eo[1],
                  acc + 3, t1);
#pragma unroll
        for (int u = 0; u < W; ++u) t1[u] = __fmaf_rn(s0, le[1][u], -t1[u]);
        put_seg(out.c[1], po, dst, t1);
        dtx<false>(M + MSLOT, mu[1], e, lb, rb, m.cA[0], m.cD[0], m.cB[0][1], m.cB[0][2], eo[2], acc + 3,
                   t1);
        dty<true>(M, mu[0], e, lb, rb, m.cA[1], m.cD[1], m.cB[1][0], m.cB[1][2], eo[2], acc + 6, t2);
#pragma unroll
        for (int u = 0; u < W; ++u) t1[u] = __fmaf_rn(s0, le[2][u], __fsub_rn(t1[u], t2[u]));
        put_seg(out.c[2], po, dst, t1);
#pragma unroll
        for (int k = 0; k < 6; ++k) {   // the plane's terms, compensated add
            const float* a = acc + 3 * (k / 2);
            const float x = fmaf(k % 2 == 0 ? -3.0f : -2.0f, a[2], a[k % 2]);
            const float y = x - gc[k];
            const float s = gs[k] + y;
            gc[k] = (s - gs[k]) - y;
            gs[k] = s;
        }
    }
    if (failed) {   // a copy did not arrive in time: drain this CTA's copies in flight
        if (tid == PRODUCER) {
            atomicOr(err, ERR_WAIT);
            for (int u = it; u < issued; ++u) mbar_wait(&bar[u % NL], (uint32_t)((u / NL) & 1));
        }
        return;
    }
    // block reduction, as in the 3D kernel: exact two-sums within a warp, FP64 across warps (rows
    // 0-3: the sums of its first group of warps, rows 4-7: of the second)
    __shared__ double red[2 * NT / 32][9];
    const int l = tid & 31;
    if (l < 9) {
        red[wp][l] = 0.0;
        red[NT / 32 + wp][l] = 0.0;
    }
    __syncwarp();
#pragma unroll
    for (int k = 0; k < 6; ++k) {
        float vs = gs[k], vc = gc[k];
        for (int sh = 16; sh > 0; sh >>= 1) {
            const float os = __shfl_down_sync(FULL, vs, sh), oc = __shfl_down_sync(FULL, vc, sh);
            const float s = __fadd_rn(vs, os);
            const float bv = __fsub_rn(s, vs);
            const float er = __fadd_rn(__fsub_rn(vs, __fsub_rn(s, bv)), __fsub_rn(os, bv));
            vs = s;
            vc = __fsub_rn(__fadd_rn(vc, oc), er);
        }
        // (delta_y, beta_yx), (delta_x, beta_xy), (delta_y, beta_yx)
        if (l == 0) red[k < 2 ? wp : NT / 32 + wp][(k / 2 == 1 ? 0 : 3) + k % 2] = (double)vs - (double)vc;
    }
    __syncthreads();
    if (tid < 9) {
        double v = 0.0;
        for (int r = 0; r < 2 * NT / 32; ++r) v += red[r][tid];
        partials[(long long)blockIdx.x * 9 + tid] += v;
    }
}

}  // namespace adj32p

bool adjoint2d32_prepare() {
    return cudaFuncSetAttribute(adj32p::adj2d_kernel<true>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                (int)adj32p::SMEM) == cudaSuccess &&
           cudaFuncSetAttribute(adj32p::adj2d_kernel<false>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                (int)adj32p::SMEM) == cudaSuccess;
}

// as launch_adjoint32_fused (whole 64 x 8 tiles; `tz` planes a chunk, `blocks` chunks of tiles)
void launch_adjoint2d32(const FusedMaps& maps, const Geom& g, const Mult<float>& m, FieldSet<float> out,
                        const float* const E[3], const float* spy, const float* spz, double* partials,
                        int tz, int blocks, int* err, cudaStream_t st) {
    auto kern = spy != nullptr ? adj32p::adj2d_kernel<true> : adj32p::adj2d_kernel<false>;
    launch_pdl(kern, dim3((unsigned)blocks), dim3(adj32p::NT), adj32p::SMEM, st, maps, g, m, out, E[0], E[1],
               E[2], spy, spz, partials, tz, err);
}

}  // namespace fdtd

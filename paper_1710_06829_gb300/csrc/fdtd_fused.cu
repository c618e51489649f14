// Plans of the fused leapfrog step (which kernel a grid takes, the TMA descriptors of the FP32
// ones) and the L2 discard of the blocked schedule.
#include <type_traits>

#include "fdtd_tma.cuh"

namespace fdtd {

// ---------------------------------------------------------------- host side

typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*,
                                  const cuuint64_t*, const cuuint64_t*, const cuuint32_t*,
                                  const cuuint32_t*, CUtensorMapInterleave, CUtensorMapSwizzle,
                                  CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

static EncodeTiledFn encode_fn() {
    static EncodeTiledFn fn = nullptr;
    if (!fn) {
        void* p = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault,
                                             &q) == cudaSuccess &&
            q == cudaDriverEntryPointSuccess)
            fn = (EncodeTiledFn)p;
    }
    return fn;
}

void launch_fused32_range(const FusedMaps& maps, FieldSet<float> in, const Geom& g,
                          const Mult<float>& m, FieldSet<float> out, const float* spy,
                          const float* spz, int zs, int ze, int* err, cudaStream_t st);
bool fused32_supported(const Geom& g, bool flat);
int fused32_ebox_w();
bool fused32_prepare();
void launch_fused32(const FusedMaps& maps, FieldSet<float> in, const Geom& g, const Mult<float>& m,
                    FieldSet<float> out, const float* spy, const float* spz, const float* jyz,
                    const float* jx_row, float* hist_E[3], int* err, cudaStream_t st);

void launch_step2d32(const Geom& g, const Mult<float>& m, FieldSet<float> in, FieldSet<float> out,
                     const float* spy, const float* spz, const float* jyz, const float* jx_row,
                     float* hist_E[3], int* err, cudaStream_t st);

bool step2d64_prepare();
void launch_step2d64(const Geom& g, const Mult<double>& m, FieldSet<double> in, FieldSet<double> out,
                     const double* spy, const double* spz, const double* jyz, const double* jx_row,
                     double* hist_E[3], int* err, cudaStream_t st);

void launch_step64(const Geom& g, const Mult<double>& m, FieldSet<double> in, FieldSet<double> out,
                   const double* spy, const double* spz, const double* jyz, const double* jx_row,
                   double* hist_E[3], int* err, cudaStream_t st);

template <typename T>
bool fused_supported(const Geom& g, bool flat) {
    if constexpr (std::is_same<T, float>::value) return fused32_supported(g, flat);
    return true;   // fdtd_step2d64.cu and fdtd_step64.cu take every size
}

// a bw x bh box (FP32) of one padded array
bool encode_box_f32(CUtensorMap* map, const Geom& g, float* base, int bw, int bh) {
    EncodeTiledFn fn = encode_fn();
    if (!fn) return false;
    const cuuint64_t dims[3] = {(cuuint64_t)g.nxp, (cuuint64_t)g.nyp, (cuuint64_t)g.nz};
    const cuuint64_t strides[2] = {(cuuint64_t)g.nxp * 4, (cuuint64_t)g.plane * 4};
    const cuuint32_t box[3] = {(cuuint32_t)bw, (cuuint32_t)bh, 1};
    const cuuint32_t estr[3] = {1, 1, 1};
    return fn(map, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 3, base, dims, strides, box, estr,
              CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
              CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

// E^n box (x0-4 .., y0-2 .. of a 64 x 8 tile: 72 x 12, FP32) of one padded array, as the adjoint
// kernels read it
bool encode_ebox_f32(CUtensorMap* map, const Geom& g, float* base) {
    return encode_box_f32(map, g, base, 72, 12);
}

template <typename T>
FusedPlan* fused_plan_create(const Geom& g, bool flat, T* const set0[6], T* const set1[6]) {
    if (!fused_supported<T>(g, flat)) return nullptr;
    FusedPlan* p = new FusedPlan();
    p->flat = flat;
    bool ok = true;
    if constexpr (std::is_same<T, float>::value) {
        for (int s = 0; s < 2; ++s) {
            T* const* set = s == 0 ? set0 : set1;
            // E boxes x0-4 .., y0-2 ..; B boxes x0-4 .., y0-1 .. (68 x 9)
            for (int c = 0; c < 3; ++c)
                ok = ok && encode_box_f32(&p->maps[s].e[c], g, set[c], fused32_ebox_w(), 12) &&
                     encode_box_f32(&p->maps[s].b[c], g, set[3 + c], 68, 9);
        }
        ok = ok && fused32_prepare();
    } else if (flat) {
        ok = step2d64_prepare();
    }
    if (!ok) {
        delete p;
        return nullptr;
    }
    return p;
}

void fused_plan_destroy(FusedPlan* p) { delete p; }

void launch_step_fused32_range(const FusedPlan* plan, int in_set, const Geom& g,
                               const Mult<float>& m, FieldSet<float> in, FieldSet<float> out,
                               const float* sponge_y, const float* sponge_z, int zs, int ze,
                               int* err, cudaStream_t st) {
    launch_fused32_range(plan->maps[in_set], in, g, m, out, sponge_y, sponge_z, zs, ze, err, st);
}

// ---------------------------------------------------------------- L2 discard

// Drops the 128-byte lines [lo[c], hi[c]) (line indices of absolute addresses) of six arrays
// from L2 without writing them back (discard.global.L2); their contents become undefined.
__global__ void discard_l2_kernel(unsigned long long lo0, unsigned long long lo1,
                                  unsigned long long lo2, unsigned long long lo3,
                                  unsigned long long lo4, unsigned long long lo5,
                                  unsigned long long n) {
    const unsigned long long lo[6] = {lo0, lo1, lo2, lo3, lo4, lo5};
    const unsigned long long stride = (unsigned long long)gridDim.x * blockDim.x;
    for (unsigned long long t = (unsigned long long)blockIdx.x * blockDim.x + threadIdx.x; t < 6 * n;
         t += stride) {
        const unsigned long long a = (lo[t / n] + t % n) * 128ull;
        asm volatile("discard.global.L2 [%0], 128;" ::"l"(a) : "memory");
    }
}

void launch_discard_planes(const Geom& g, size_t esz, void* const arr[6], int p0, int p1,
                           cudaStream_t st) {
    if (p1 <= p0) return;
    const unsigned long long pb = (unsigned long long)g.plane * esz;
    unsigned long long lo[6];
    unsigned long long n = ~0ull;
    for (int c = 0; c < 6; ++c) {
        const unsigned long long b = reinterpret_cast<unsigned long long>(arr[c]);
        const unsigned long long first = (b + p0 * pb + 127) / 128, last = (b + p1 * pb) / 128;
        lo[c] = first;
        const unsigned long long nc = last > first ? last - first : 0;
        n = nc < n ? nc : n;   // the arrays have equal sizes and alignments in practice
    }
    if (n == 0) return;
    const unsigned long long total = 6 * n;
    const int blk = 256;
    const int grd = (int)((total + blk - 1) / blk < 4096 ? (total + blk - 1) / blk : 4096);
    discard_l2_kernel<<<grd, blk, 0, st>>>(lo[0], lo[1], lo[2], lo[3], lo[4], lo[5], n);
}

template <typename T>
void launch_step_fused(const FusedPlan* plan, int in_set, const Geom& g, const Mult<T>& m,
                       FieldSet<T> in, FieldSet<T> out, const T* sponge_y, const T* sponge_z,
                       const T* jyz, const T* jx_row, T* hist_E[3], int* err, cudaStream_t st) {
    if constexpr (std::is_same<T, float>::value) {
        if (plan->flat) {
            launch_step2d32(g, m, in, out, sponge_y, sponge_z, jyz, jx_row, hist_E, err, st);
            return;
        }
        launch_fused32(plan->maps[in_set], in, g, m, out, sponge_y, sponge_z, jyz, jx_row, hist_E,
                       err, st);
        return;
    }
    if constexpr (std::is_same<T, double>::value) {
        if (plan->flat)
            launch_step2d64(g, m, in, out, sponge_y, sponge_z, jyz, jx_row, hist_E, err, st);
        else
            launch_step64(g, m, in, out, sponge_y, sponge_z, jyz, jx_row, hist_E, err, st);
    }
}

template bool fused_supported<float>(const Geom&, bool);
template bool fused_supported<double>(const Geom&, bool);
template FusedPlan* fused_plan_create<float>(const Geom&, bool, float* const[6], float* const[6]);
template FusedPlan* fused_plan_create<double>(const Geom&, bool, double* const[6], double* const[6]);
template void launch_step_fused<float>(const FusedPlan*, int, const Geom&, const Mult<float>&,
                                       FieldSet<float>, FieldSet<float>, const float*, const float*, const float*,
                                       const float*, float* [3], int*, cudaStream_t);
template void launch_step_fused<double>(const FusedPlan*, int, const Geom&, const Mult<double>&,
                                        FieldSet<double>, FieldSet<double>, const double*, const double*,
                                        const double*, const double*, double* [3], int*,
                                        cudaStream_t);

}  // namespace fdtd

// Gradient of a real loss with respect to per-ping position offsets, given
// the image gradient G = dL/dI* (the autofocus VJP), and its deterministic
// reduction over image tiles.
#include "tdbp_core.cuh"

namespace sas {
namespace core {

template <typename ET, bool DIM3, int MODE>
static int launch_one_grad(const Setup& S, cudaStream_t st) {
    const bool mv = S.prm.vel != nullptr;
    auto kern = S.prm.beam ? (mv ? tdbp_kernel<ET, DIM3, MODE, true, true> : tdbp_kernel<ET, DIM3, MODE, true, false>)
                           : (mv ? tdbp_kernel<ET, DIM3, MODE, false, true> : tdbp_kernel<ET, DIM3, MODE, false, false>);
    if (S.prm.refract) {   // without a beam or motion (prepare)
        kern = tdbp_kernel<ET, DIM3, MODE, false, false, true>;
    } else if (!S.prm.beam && !mv && S.prm.npos_pad == NPOS_FIXED) {
        kern = tdbp_kernel<ET, DIM3, MODE, false, false, false, true>;
    }
    SAS_CUDA(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)S.smem));
    kern<<<S.blocks, NTHREADS, S.smem, st>>>(S.map, S.prm);
    SAS_CUDA(cudaGetLastError());
    return SAS_OK;
}

template <>
int launch_mode<MODE_OFFSET_GRAD>(const Setup& S, int echo_dtype, int dim3, cudaStream_t st) {
    switch (echo_dtype) {
        case SAS_ECHO_C64:
            return dim3 ? launch_one_grad<float2, true, MODE_OFFSET_GRAD>(S, st)
                        : launch_one_grad<float2, false, MODE_OFFSET_GRAD>(S, st);
        case SAS_ECHO_C32_F16:
            return dim3 ? launch_one_grad<__half2, true, MODE_OFFSET_GRAD>(S, st)
                        : launch_one_grad<__half2, false, MODE_OFFSET_GRAD>(S, st);
        case SAS_ECHO_C32_BF16:
            return dim3 ? launch_one_grad<__nv_bfloat162, true, MODE_OFFSET_GRAD>(S, st)
                        : launch_one_grad<__nv_bfloat162, false, MODE_OFFSET_GRAD>(S, st);
        default:
            set_error("no echo uploaded");
            return SAS_ERR_STATE;
    }
}

// out[t] = sum over tiles (in a fixed order, FP64) of partials[tile][t], t = 3 ping +
// axis: 32 values a block, 32 threads a value, each over every 32nd tile, then the
// threads' sums in order (a thread a value over all tiles waited on one load after the
// other: 81 us for 608 tiles x 768 values)
constexpr int RT_SLICES = 32;
__global__ void __launch_bounds__(32 * RT_SLICES) reduce_tiles_kernel(const double* __restrict__ partials, int ntiles,
                                                                      int n, double* __restrict__ out) {
    __shared__ double red[RT_SLICES][33];
    const int lane = threadIdx.x & 31, sl = threadIdx.x >> 5, t = blockIdx.x * 32 + lane;
    double s = 0.0;
    if (t < n) {
#pragma unroll 4
        for (int k = sl; k < ntiles; k += RT_SLICES) s += partials[(size_t)k * n + t];
    }
    red[sl][lane] = s;
    __syncthreads();
    if (sl == 0 && t < n) {
        for (int w = 1; w < RT_SLICES; ++w) s += red[w][lane];
        out[t] = s;
    }
}

}  // namespace core

int launch_offset_grad(sas_geometry_t h, const sas_grid& g, const float2* grad_image, double* grad_offsets,
                       cudaStream_t st) {
    const int dim3 = g.nz > 1;
    core::Setup S;
    int rc = core::prepare(h, g, dim3, 2LL * sm_count(), S, true, core::MODE_OFFSET_GRAD);
    if (rc != SAS_OK) return rc;
    const long long ntiles = (long long)S.prm.tiles_x * S.prm.tiles_y * S.prm.tiles_z;
    const size_t need = (size_t)ntiles * h->P * 3 * sizeof(double);
    void* part = nullptr;
    bool own = false;
    SAS_CUDA(call_scratch(h->partials, need, true, st, &part, &own));
    // (tile, ping) partials with no pair inside the beams are never written
    cudaError_t e = cudaMemsetAsync(part, 0, need, st);
    S.prm.gimage = grad_image;
    S.prm.partials = (double*)part;
    rc = e == cudaSuccess ? core::launch_mode<core::MODE_OFFSET_GRAD>(S, h->echo_dtype, dim3, st)
                          : cuda_fail(e, "offset gradient memset");
    if (rc == SAS_OK) {
        const int n = h->P * 3;
        core::reduce_tiles_kernel<<<(n + 31) / 32, 32 * core::RT_SLICES, 0, st>>>((const double*)part, (int)ntiles, n,
                                                                                 grad_offsets);
        e = cudaGetLastError();
        if (e != cudaSuccess) rc = cuda_fail(e, "reduce_tiles_kernel");
    }
    if (own) cudaFreeAsync(part, st);
    return rc;
}

}  // namespace sas
